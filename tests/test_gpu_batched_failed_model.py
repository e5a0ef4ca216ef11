"""A batch in which one model fails the device check: the others keep the layout the buffer was sized for.

26^3 k-points at W = 64 are more than a stream's share of the batch memory on four streams (13,793) and
less than on three, so a layout of the three valid models alone would be 2.6 GB larger than the buffer.
"""
import ctypes

import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


def test_failed_model_among_large_ones():
    import torch
    import paper_2309_06675_gb300 as kubo
    mesh = (26, 26, 26)
    models = [tbgen.random_tb(8, 1, 1.0, 0)] + [tbgen.random_tb(64, 1, 1.0, s) for s in (1, 2, 3)]
    H = [torch.from_numpy(m.H_R).cuda() for m in models]
    H[0][0, 0, 0] = float("nan")
    R = [np.ascontiguousarray(m.R, dtype=np.int32) for m in models]
    ef = torch.zeros(1, dtype=torch.float64, device="cuda")
    outs = [torch.full((1, 1), 7.0, dtype=torch.float64, device="cuda") for _ in models]
    arr = (kubo.Problem * 4)()
    for a, h, r, out in zip(arr, H, R, outs):
        a.H_R, a.R_vecs, a.W, a.N_R = h.data_ptr(), r.ctypes.data, h.shape[1], h.shape[0]
        for q in range(3):
            a.kmesh[q] = mesh[q]
        a.E_F, a.n_EF, a.eta, a.out = ef.data_ptr(), 1, 1e-3, out.data_ptr()
    o = kubo.Options()
    kubo.lib().kubo_options_init(ctypes.byref(o))
    o.stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert kubo.lib().kubo_ahc_batched(arr, 4, ctypes.byref(o), None) == 2
    assert [a.status for a in arr] == [2, 0, 0, 0]
    assert float(outs[0]) == 7.0
    for h, m, out in list(zip(H, models, outs))[1:]:
        one = float(kubo.ahc(h, m.R, mesh, ef, eta=1e-3))
        assert abs(float(out) - one) <= 1e-13 * max(abs(one), 1e-3)
