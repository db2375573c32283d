"""The FP32 low-rank kernel at ranks above 20, which works on one compartment at a time above
40. Against the oracle; bar: 1e-5 after a fixed iteration count.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _compare(precision, dims, batch, P, Q, rank, iters=8):
    import torch
    from oracle import ladmm as L
    from paper_2401_12890_gb300 import ssm, synth
    n = int(np.prod(dims))
    K, M, _ = synth.random_problem(P, Q, (n * (batch or 1),), seed=Q + n, snr=50.0)
    M = M.astype(np.float32)
    plan = ssm.Plan(K, dims, 0.02, 0.3, form="lowrank", precision=precision, rank=rank,
                    max_iter=iters, check_every=3, tol_primal=1e-12, tol_change=1e-12, batch=batch)
    Md = torch.from_numpy(M).cuda()
    plan.solve(Md * 1e12)
    F, info = plan.solve(Md)
    plan.close()
    F = F.cpu().numpy()
    assert info["iterations"] == iters
    for b in sorted({0, (batch or 1) // 2, (batch or 1) - 1}):
        c = slice(b * n, (b + 1) * n)
        ref = L.ladmm(K, np.ascontiguousarray(M[:, c]).astype(np.float64), dims, 0.02, 0.3,
                      rank=rank, iters=iters, check_every=0)["z"]
        assert np.linalg.norm(F[:, c] - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("rank", [24, 40, 41, 48, 56, 64])
@pytest.mark.parametrize("dims", [(23, 18), (9, 8, 7)])
def test_large_ranks_fp32(dims, rank):
    _compare("fp32", dims, None, 70, 99, rank)
