"""The autotuner of kubo_ahc_batched times only what a precision's kernels take: schedules alone in FP64 (streams 1 and 2
by two batch sizes for three models), the reduction's partitions and the mixed kernels' parameters as well in MIXED."""
import numpy as np
import pytest
import tbgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,candidates", [("fp64", 4), ("mixed", 4 + 2 + 2 + 2)])
def test_candidates(precision, candidates):
    import torch
    import paper_2309_06675_gb300 as kubo
    P = []
    for W, seed in ((7, 1), (19, 2), (33, 3)):
        m = tbgen.random_tb(W, 1, 1.0, seed)
        P.append((torch.from_numpy(m.H_R).cuda(), m.R, (5, 3, 2), torch.from_numpy(np.array([0.1])).cuda()))
    _, sched, status = kubo.ahc_batched(P, precision=precision, tune=True)
    assert status == ["KUBO_OK"] * 3
    assert sched["tuned_candidates"] == candidates
    assert sched["symv_parts"] == 4 or precision != "fp64"
