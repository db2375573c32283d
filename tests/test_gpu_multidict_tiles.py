"""Spatially varying dictionaries at the edges of the two iteration kernels' ranges: grids
below and above 1600 voxels (work table of 32-voxel tiles, voxel patches), padded ranks up to
and past 16, ragged patches in 1D, 2D and 3D, compartments around a half chunk, random
labels. Bar: the FP32 low-rank forms' 1e-5 against the oracle after a fixed iteration count.

A solve of much larger data runs first (the next one takes z = 0 without reading memory), and
replayed blocks, residual tests and a continued solve give the same bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [
    # dims, P, Q, rank, dictionaries
    ((39, 41), 12, 16, 4, 3),            # 1599 voxels
    ((40, 40), 12, 17, 4, 3),
    ((1601,), 20, 31, 7, 5),
    ((57, 29), 20, 33, 8, 1),
    ((131, 13), 24, 48, 9, 16),
    ((12, 13, 11), 24, 50, 12, 4),
    ((53, 37), 40, 65, 16, 7),
    ((53, 37), 40, 65, 17, 7),
    ((7, 5, 47), 40, 34, 32, 2),
]


@pytest.mark.parametrize("dims,P,Q,rank,ndict", CASES)
def test_edges_match_oracle(dims, P, Q, rank, ndict):
    import torch
    from oracle import multidict as MD
    from paper_2401_12890_gb300 import ssm
    rng = np.random.default_rng(P * 31 + Q + rank)
    N = int(np.prod(dims))
    Ks = rng.random((ndict, P, Q))
    labels = rng.integers(0, ndict, N).astype(np.int32)
    F0 = rng.random((Q, N)) * (rng.random((Q, N)) < 0.2)
    M = np.empty((P, N), np.float32)
    for c in range(ndict):
        M[:, labels == c] = Ks[c] @ F0[:, labels == c]
    Md = torch.from_numpy(M).cuda()
    plan = ssm.MultiPlan(Ks, labels, dims, 0.05, 0.5, rank=rank, max_iter=12, check_every=0)
    plan.solve(Md * 1e12)
    F = plan.solve(Md)[0].cpu().numpy()
    ref = MD.ladmm_multi(Ks, labels, M.astype(np.float64), dims, 0.05, 0.5, rank=rank, iters=12,
                         check_every=0)["z"]
    assert np.linalg.norm(F - ref) <= 1e-5 * np.linalg.norm(ref)
    plan.solve(Md * 1e12)
    plan.set_max_iter(0)
    assert np.all(plan.solve(Md)[0].cpu().numpy() == 0.0)
    plan.set_max_iter(12)
    assert np.array_equal(plan.resume(Md)[0].cpu().numpy(), F)
    plan.set_graphs(True)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    out = torch.empty(F.shape, device="cuda")
    with torch.cuda.stream(s):
        for _ in range(2):
            plan.solve_async(Md, out, stream=s)
    s.synchronize()
    assert np.array_equal(out.cpu().numpy(), F)
    plan.close()
    plan = ssm.MultiPlan(Ks, labels, dims, 0.05, 0.5, rank=rank, max_iter=12, check_every=3,
                         tol_change=1e-30)
    assert np.array_equal(plan.solve(Md)[0].cpu().numpy(), F)
    plan.close()
