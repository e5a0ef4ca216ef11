"""A first allocation that fails: FP64 calls whose Fourier slices are a good part of it run without them.

Simulated on the host (kubo_debug_fail_allocations); a second failure is KUBO_ERR_OOM with the outputs untouched, as is
the first one where there is nothing to drop (small models, mixed modes).  The FP64-pipe sum differs by its
rounding, amplified by the smallest gaps: within 1e-9 of the largest value.
"""
import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


def _calls(kubo, torch):
    m = tbgen.random_tb(32, 4, 1.5, 3)
    H, ef = torch.from_numpy(m.H_R).cuda(), torch.tensor([0.0, 0.2], dtype=torch.float64, device="cuda")
    mesh, k_range = (24, 24, 24), (1000, 7000)
    g = torch.ones(1, 2, dtype=torch.float64, device="cuda")
    kidx = torch.arange(6000, dtype=torch.int64).cuda()
    return {
        "ahc": lambda: kubo.ahc(H, m.R, mesh, ef, etas=[0.05], k_range=k_range),
        "ahc_host": lambda: kubo.ahc_host(m.H_R, m.R, mesh, ef.cpu().numpy(), etas=[0.05], k_range=k_range),
        "ahc_k": lambda: kubo.ahc_k(H, m.R, mesh, kidx, etas=[0.05]),
        "bloch": lambda: kubo.bloch(H, m.R, mesh, kidx),
        "grad": lambda: kubo.ahc_grad(H, m.R, mesh, ef, g, etas=[0.05], kT=0.05, k_range=k_range),
        "batched": lambda: kubo.ahc_batched([(H, m.R, (20, 20, 16), ef, 0.05)])[0],
    }


def _flat(r):
    return [np.asarray(x.cpu() if hasattr(x, "cpu") else x) for x in (r if isinstance(r, (tuple, list)) else [r])]


@pytest.mark.parametrize("name", ["ahc", "ahc_host", "ahc_k", "bloch", "grad", "batched"])
def test_retry_without_slices(name):
    import torch
    import paper_2309_06675_gb300 as kubo
    call = _calls(kubo, torch)[name]
    ref = _flat(call())
    try:
        kubo.debug_fail_allocations(1)
        got = _flat(call())
        for a, b in zip(got, ref):
            assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()
        kubo.debug_fail_allocations(2)
        with pytest.raises(kubo.KuboError) as ei:
            call()
        assert ei.value.name == "KUBO_ERR_OOM"
    finally:
        kubo.debug_fail_allocations(0)
    for a, b in zip(_flat(call()), ref):
        assert np.array_equal(a, b)
