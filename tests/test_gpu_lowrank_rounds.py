"""The low-rank forms' launch layouts where the tiles are just past whole rounds of CTAs: whole
tiles (or few segments) first, the rest in more segments, each tile's partial u' in as many
slots; and the FP32 kernel at ranks 33 to 64, which works on one compartment at a time above 40.
Against the oracle; bar: 1e-5 after a fixed iteration count. The launch-shape override makes
the rounds small, so that small grids reach every branch.
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


# CTAs, grid, slices, Q: one tile, a few and all but one past whole rounds; rounds of one CTA
@pytest.mark.parametrize("ctas,dims,batch,Q", [
    (1, (20, 19), None, 100), (3, (32, 32), None, 130), (3, (33, 32), None, 260),
    (5, (16, 8), 6, 161), (5, (16, 8), 9, 225), (7, (24, 10, 6), None, 97),
    (4, (40, 33), None, 31), (9, (37, 29), 4, 64)])
@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
def test_rounds(monkeypatch, precision, ctas, dims, batch, Q):
    monkeypatch.setenv("SSM_LOWRANK_GRID", str(ctas))
    monkeypatch.setenv("SSM_LRTC_GRID", str(ctas))
    _compare(precision, dims, batch, 30, Q, 20)


@pytest.mark.parametrize("dims,batch,Q", [((24, 30), 27, 100), ((39, 26), 56, 70),
                                          ((33, 27, 19), None, 60)])
@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
def test_rounds_of_the_device(precision, dims, batch, Q):
    _compare(precision, dims, batch, 30, Q, 20, iters=4)


@pytest.mark.parametrize("rank", [24, 40, 41, 48, 56, 64])
@pytest.mark.parametrize("dims", [(23, 18), (9, 8, 7)])
def test_large_ranks_fp32(dims, rank):
    _compare("fp32", dims, None, 70, 99, rank)


@pytest.mark.parametrize("rank", [40, 64])
@pytest.mark.parametrize("ctas", [2, 5])
def test_large_ranks_tf32x3(monkeypatch, ctas, rank):
    monkeypatch.setenv("SSM_LRTC_GRID", str(ctas))
    _compare("tf32x3", (31, 28), None, 70, 150, rank)
