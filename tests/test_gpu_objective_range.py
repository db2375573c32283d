"""The objective at the ends of the FP32 range: the sum over neighbour pairs is an FP64 sum of
FP32 squares, so it overflows only where a square does, and an infinite or NaN estimate
gives what IEEE arithmetic gives. Bar for finite values: the squares' FP32 roundings
(4 * 2^-24) and the residuals' (Q + 1) 2^-24 each, as in the objective's other tests.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GRIDS = [((13, 9), 7), ((13, 9), 200), ((40, 1), 33), ((6, 5, 4), 64), ((1, 1), 9)]


def _plan(dims, Q, seed=1):
    from paper_2401_12890_gb300 import ssm
    K = np.random.default_rng(seed).uniform(0.1, 1, (3, Q))
    return K, ssm.Plan(K, dims, 0.02, 0.3, form="lowrank", rank=1)


def _J(plan, F, M):
    import torch
    return plan.objective(torch.from_numpy(M).cuda(), torch.from_numpy(F).cuda(), use_full_k=True)


@pytest.mark.parametrize("scale", [1e-18, 1.0, 1e18, 4e18])
@pytest.mark.parametrize("dims,Q", GRIDS)
def test_finite_sums_stay_finite(dims, Q, scale):
    from oracle import ladmm as L
    N = int(np.prod(dims))
    rng = np.random.default_rng(Q)
    # large differences in a few maps only, so that the terms of a sum differ in size
    F = (rng.uniform(0, 1, (Q, N)) * np.where(np.arange(Q) % 5 == 0, 1, 1e-3)[:, None] * scale)
    F = F.astype(np.float32)
    K, plan = _plan(dims, Q)
    M = np.zeros((3, N), np.float32)
    J = _J(plan, F, M)
    plan.close()
    K32 = K.astype(np.float32).astype(np.float64)
    ref = L.objective(K32, M, F, dims, 0.02)
    assert np.isfinite(ref)
    assert abs(J - ref) <= (2 * (Q + 1) + 8) * 2.0 ** -24 * ref


@pytest.mark.parametrize("dims,Q", GRIDS)
@pytest.mark.parametrize("value", [np.inf, -np.inf, 1e20, np.nan])
def test_infinite_and_nan(dims, Q, value):
    N = int(np.prod(dims))
    K, plan = _plan(dims, Q)
    F = np.random.default_rng(3).uniform(0, 1, (Q, N)).astype(np.float32)
    M = np.zeros((3, N), np.float32)
    for n in sorted({0, N // 2, N - 1}):
        for q in sorted({0, Q // 2, Q - 1}):
            G = F.copy()
            G[q, n] = value
            J = _J(plan, G, M)
            if np.isnan(value):
                assert np.isnan(J)
            elif np.isinf(value) or N > 1:     # 1e20: a neighbour difference's square
                assert J == np.inf, (n, q, J)
            else:                              # one voxel has no neighbours: finite
                assert np.isfinite(J)
    plan.close()
