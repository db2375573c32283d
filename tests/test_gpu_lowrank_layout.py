"""The TF32x3 form's launch layouts around the point where a few spare CTAs take the tails of
many tiles (no tails there) and where they take few (main and tail units): stacks of slices
of 130 to 150 tiles, against the oracle's slices. Bar: 1e-5 after a fixed iteration count.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,batch,Q", [((36, 29), 13, 225), ((36, 29), 13, 40),
                                          ((32, 32), 10, 225), ((36, 29), 15, 130)])
def test_layouts_match_oracle(dims, batch, Q):
    import torch
    from oracle import ladmm as L
    from paper_2401_12890_gb300 import ssm, synth
    n = dims[0] * dims[1]
    K, M, _ = synth.random_problem(30, Q, (n * batch,), seed=Q + batch, snr=50.0)
    M = M.astype(np.float32)
    plan = ssm.Plan(K, dims, 0.02, 0.3, form="lowrank", precision="tf32x3", rank=20, max_iter=8,
                    check_every=0, batch=batch)
    F = plan.solve(torch.from_numpy(M).cuda())[0].cpu().numpy()
    plan.close()
    for b in (0, batch - 1):
        c = slice(b * n, (b + 1) * n)
        ref = L.ladmm(K, np.ascontiguousarray(M[:, c]).astype(np.float64), dims, 0.02, 0.3, rank=20,
                      iters=8, check_every=0)["z"]
        assert np.linalg.norm(F[:, c] - ref) <= 1e-5 * np.linalg.norm(ref)
