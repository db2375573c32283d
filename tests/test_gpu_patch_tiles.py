"""The low-rank forms' voxel patches and blocked state at their edges, against the oracle:
axes of one voxel, grids thinner than a patch, ragged patches in every axis, compartments
around a half chunk (16) and a chunk (32), unlinked stacks, masks, few and many units per
block. Bar: the low-rank forms' 1e-5 after a fixed iteration count.

Every plan first solves much larger data, so that a state left over from one solve (the
first iteration of the next takes z = 0 without reading memory) would show; the same solve
replayed from captured blocks, and continued from a solve of no iterations, gives the same
bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [
    # dims, P, Q, rank, mask, waves
    ((1, 1), 6, 1, 1, False, 1),
    ((1, 9), 20, 16, 4, False, 1),
    ((131, 1), 20, 17, 5, False, 1),
    ((1, 1, 37), 24, 31, 3, False, 1),
    ((3, 129), 24, 32, 8, False, 1),
    ((129, 2), 24, 33, 20, True, 1),
    ((17, 1, 9), 24, 47, 12, False, 1),
    ((5, 11, 7), 40, 65, 32, False, 1),
    ((9, 10, 6), 48, 96, 13, True, 1),
    ((19, 23), 60, 70, 40, False, 1),
    ((150, 131), 30, 40, 20, True, 8),
    ((41, 38, 9), 30, 48, 30, False, 1),
]


@pytest.mark.parametrize("precision", ["fp32", "tf32x3"])
@pytest.mark.parametrize("dims,P,Q,rank,masked,waves", CASES)
def test_patch_edges(dims, P, Q, rank, masked, waves, precision):
    import torch
    from oracle import ladmm as L
    from paper_2401_12890_gb300 import ssm, synth
    K, M, _ = synth.random_problem(P, Q, dims, seed=P * 11 + Q, snr=50.0)
    M = M.astype(np.float32)
    mask = None
    if masked:
        mask = np.random.default_rng(2).uniform(size=int(np.prod(dims))) < 0.7
    Md = torch.from_numpy(M).cuda()
    plan = ssm.Plan(K, dims, 0.02, 0.3, form="lowrank", precision=precision, rank=rank,
                    max_iter=12, check_every=0, launch_waves=waves)
    if masked:
        plan.set_mask(mask)
    plan.solve(Md * 1e12)
    F = plan.solve(Md)[0].cpu().numpy()
    ref = L.ladmm(K, M.astype(np.float64), dims, 0.02, 0.3, rank=rank, iters=12, check_every=0,
                  mask=mask)["z"]
    assert np.linalg.norm(F - ref) <= 1e-5 * np.linalg.norm(ref)
    if masked:
        assert np.all(F[:, ~mask] == 0.0)
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
