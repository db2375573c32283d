"""The FP32 product's tile shapes and epilogues (full-rank FP32 form, objective) at the
edges of their tiles, against FP64.

Full-rank form: the FP32 parity bar of the other tests (1e-5 against the oracle's z after a
fixed iteration count). Objective: each residual m - k f is an FP32 chain of Q products, so
its error is at most (Q + 1) 2^-24 sum |k f| (a first-order bound); the sums are FP64.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,P,Q,masked", [
    ((1, 1), 3, 2, False), ((5, 13), 20, 63, False), ((64, 1), 20, 64, False),
    ((13, 5, 3), 10, 65, False), ((67, 9), 40, 130, True), ((9, 7, 6), 12, 40, True),
    ((150, 140), 24, 260, False)])
def test_full_rank_fp32(dims, P, Q, masked):
    import torch
    from oracle import ladmm as L
    from paper_2401_12890_gb300 import ssm, synth
    K, M, _ = synth.random_problem(P, Q, dims, seed=P * 7 + Q, snr=50.0)
    M = M.astype(np.float32)
    mask = None
    if masked:
        mask = np.random.default_rng(1).uniform(size=int(np.prod(dims))) < 0.7
    plan = ssm.Plan(K, dims, 0.02, 0.3, form="dense", max_iter=12, check_every=0)
    if masked:
        plan.set_mask(mask)
    F, _ = plan.solve(torch.from_numpy(M).cuda())
    F = F.cpu().numpy()
    plan.close()
    ref = L.ladmm(K, M.astype(np.float64), dims, 0.02, 0.3, dense=True, iters=12, check_every=0,
                  mask=mask)["z"]
    assert np.linalg.norm(F - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("dims,P,Q,pad", [
    ((1, 1), 1, 1, 0), ((7, 9), 5, 31, 1), ((16, 8), 64, 32, 0), ((33, 4), 65, 33, 0),
    ((10, 9, 8), 129, 70, 3), ((260, 200), 128, 40, 0), ((211, 191), 70, 65, 2)])
@pytest.mark.parametrize("masked", [False, True])
def test_objective(dims, P, Q, pad, masked):
    """pad: extra columns of F's and M's rows (rows that are not 16-byte aligned)."""
    import torch
    from oracle import ladmm as L
    from paper_2401_12890_gb300 import ssm
    rng = np.random.default_rng(P + Q)
    N = int(np.prod(dims))
    K = rng.uniform(0, 1, (P, Q))
    F = rng.uniform(0, 1, (Q, N)).astype(np.float32)
    M = (K @ F + 0.1 * rng.standard_normal((P, N))).astype(np.float32)
    mask = rng.uniform(size=N) < 0.8 if masked else None
    plan = ssm.Plan(K, dims, 0.02, 0.3, form="lowrank", rank=1)
    if masked:
        plan.set_mask(mask)
    Fp = torch.zeros((Q, N + pad), dtype=torch.float32, device="cuda")
    Mp = torch.zeros((P, N + pad), dtype=torch.float32, device="cuda")
    Fp[:, :N], Mp[:, :N] = torch.from_numpy(F), torch.from_numpy(M)
    J = plan.objective(Mp[:, :N], Fp[:, :N], use_full_k=True)
    plan.close()
    K32 = K.astype(np.float32).astype(np.float64)
    ref = L.objective(K32, M, F, dims, 0.02, mask=mask)
    inside = slice(None) if mask is None else np.flatnonzero(mask)
    R = (M.astype(np.float64) - K32 @ F)[:, inside]
    eps = ((Q + 1) * 2.0 ** -24) * (K32 @ F)[:, inside]
    # FP32 squares of the neighbour differences: a few roundings of a sum of positive terms
    rough = 4 * 2.0 ** -24 * (ref - 0.5 * np.sum(R * R))
    bound = np.sum(np.abs(R) * eps + 0.5 * eps ** 2) + abs(rough) + 1e-12 * abs(ref)
    assert abs(J - ref) <= bound, (J, ref, bound)
