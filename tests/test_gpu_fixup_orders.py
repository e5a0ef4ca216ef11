"""The FP64 redo of the mixed modes (mixed_fixup_rel) at orders around its kernels' limits.

With every k-point flagged the sum is that of the FP64 kernels (mixed_df keeps its double-float eigenvectors,
~1e-12, above W = 64); without the redo it is off by the FP32 rotations' ~1e-6.
"""
import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W", [16, 25, 64, 65, 97, 128])
@pytest.mark.parametrize("precision,tol", [("mixed", 1e-9), ("mixed_fourier", 1e-9), ("mixed_df", 1e-7)])
def test_redo_of_every_k_point(W, precision, tol):
    import torch
    import paper_2309_06675_gb300 as kubo
    m = tbgen.random_tb(W, 1, 1.5, seed=W)
    H, ef = torch.from_numpy(m.H_R).cuda(), torch.linspace(-1, 1, 5, dtype=torch.float64).cuda()
    kw = dict(etas=[0.05, 0.2], chunk_k=50)
    prof = kubo.Profile()
    ref = kubo.ahc(H, m.R, (5, 4, 4), ef, **kw).cpu().numpy()
    got = kubo.ahc(H, m.R, (5, 4, 4), ef, precision=precision, fixup_rel=10.0, profile=prof, **kw).cpu().numpy()
    assert prof.fixup_k == 80
    assert np.abs(got - ref).max() <= tol * np.abs(ref).max()
