"""The TF32x3 form at ranks 33 to 64 on narrow grids and stacks of small slices, whose patches
have the most halo rows for their voxels: every variant of the iteration (plain, storing d,
testing, both) finds room for its stages. Bar: 1e-5 against the oracle after a fixed
iteration count; the stopping rule's stop and residual as the oracle's.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# dims, slices of a stack (None: one grid)
GRIDS = [((63, 2), None), ((2, 61), None), ((124, 2), None), ((185, 2), None), ((2, 301), None),
         ((300,), None), ((1, 260), None), ((30, 2), 4), ((11, 2), 64), ((5, 4), 64), ((4, 4), 64),
         ((3, 3), 64), ((6,), 64), ((2, 2), 40), ((1, 1), 130)]


@pytest.mark.parametrize("rank", [33, 64])
@pytest.mark.parametrize("dims,batch", GRIDS)
def test_every_variant_runs(dims, batch, rank):
    import torch
    from oracle import ladmm as L
    from paper_2401_12890_gb300 import ssm, synth
    n = int(np.prod(dims))
    K, M, _ = synth.random_problem(70, 75, (n * (batch or 1),), seed=rank + n, snr=50.0)
    M = M.astype(np.float32)
    Md = torch.from_numpy(M).cuda()
    # max_iter, check_every, tolerance: a test at the end only, every 3 (plain, storing and
    # testing iterations), at every iteration (testing and storing at once)
    for iters, every, tol in ((4, 0, 0.0), (7, 3, 1e-12), (4, 1, 1e-12)):
        plan = ssm.Plan(K, dims, 0.02, 0.3, form="lowrank", precision="tf32x3", rank=rank,
                        max_iter=iters, check_every=every, tol_primal=tol, tol_change=tol,
                        batch=batch)
        F, info = plan.solve(Md)
        plan.close()
        F = F.cpu().numpy()
        assert info["iterations"] == iters
        for b in sorted({0, (batch or 1) - 1}):
            c = slice(b * n, (b + 1) * n)
            ref = L.ladmm(K, np.ascontiguousarray(M[:, c]).astype(np.float64), dims, 0.02, 0.3,
                          rank=rank, iters=iters, check_every=0)["z"]
            assert np.linalg.norm(F[:, c] - ref) <= 1e-5 * np.linalg.norm(ref)
