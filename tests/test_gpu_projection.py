"""The data projections (step 4) against FP64, at the edges of their tiles.

One iteration from zero of the full-rank FP32 form with lambda = 0 returns
F = max(0, h) beta / (beta + 1e-10), h = (K^T K + beta I)^{-1} K^T m, so F shows h. The
bound: h is one FP32 rounding of a sum whose slicing drops less than 6 * 2^-40 of the
(power-of-two) row and column scales per term, each at most twice the largest entry
(P 2^-35 amax mmax), and the element-wise step adds a handful of roundings
(8 * 2^-24 |h|).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _plan(K, n, **kw):
    from paper_2401_12890_gb300 import ssm
    return ssm.Plan(K, (n, 1), 0.0, kw.pop("beta", 0.5), max_iter=1, check_every=0, **kw)


@pytest.mark.parametrize("P,Q,N", [(1, 5, 1), (31, 32, 127), (32, 33, 128), (33, 64, 129),
                                   (70, 65, 9), (64, 96, 300), (200, 97, 130), (130, 200, 257),
                                   (1000, 100, 140), (1024, 96, 129), (1025, 70, 129),
                                   (2100, 20, 65)])
def test_full_rank_projection(P, Q, N):
    import torch
    rng = np.random.default_rng(P * 1000 + Q)
    K = rng.standard_normal((P, Q)) * np.exp(rng.uniform(-3, 3, (P, 1)))
    M = rng.standard_normal((P, N)) * 10.0 ** rng.integers(-12, 12, (1, N))
    M[:, 0] = 0.0
    M = M.astype(np.float32)
    beta = 0.5
    plan = _plan(K, N, beta=beta, form="dense")
    F, info = plan.solve(torch.from_numpy(M).cuda())
    plan.close()
    A = np.linalg.solve(K.T @ K + beta * np.eye(Q), K.T)
    h = np.maximum(A @ M.astype(np.float64), 0.0) * (beta / (beta + 1e-10))
    amax, mmax = np.abs(A).max(axis=1)[:, None], np.abs(M.astype(np.float64)).max(axis=0)[None, :]
    bound = 8 * 2.0 ** -24 * h + P * 2.0 ** -35 * amax * mmax + 1e-300
    err = np.abs(F.cpu().numpy().astype(np.float64) - h)
    assert (err <= bound).all(), float((err / bound).max())


@pytest.mark.parametrize("r,P,N", [(1, 4, 3), (32, 40, 129), (33, 60, 130), (64, 70, 257)])
def test_low_rank_projection(r, P, N):
    """One iteration of the low-rank form: F = max(0, V_r a) beta / (beta + 1e-10),
    a_i = sigma_i u_i^T m / (beta + sigma_i^2); the FP32 product over r terms adds up to
    (r + 8) roundings of its absolute sum."""
    import torch
    rng = np.random.default_rng(r)
    Q = 80
    K = rng.standard_normal((P, Q))
    M = rng.standard_normal((P, N)).astype(np.float32)
    beta = 2.0
    plan = _plan(K, N, beta=beta, form="lowrank", rank=r)
    F, _ = plan.solve(torch.from_numpy(M).cuda())
    plan.close()
    U, s, Vt = np.linalg.svd(K, full_matrices=False)
    a = (s[:r] / (beta + s[:r] ** 2))[:, None] * (U[:, :r].T @ M.astype(np.float64))
    ref = np.maximum(Vt[:r].T @ a, 0.0) * (beta / (beta + 1e-10))
    bound = (r + 8) * 2.0 ** -24 * (np.abs(Vt[:r]).T @ np.abs(a))
    err = np.abs(F.cpu().numpy().astype(np.float64) - ref)
    assert (err <= bound).all(), float((err / bound).max())


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("form", ["dense", "lowrank"])
def test_non_finite_data_is_reported(bad, form):
    import torch
    from paper_2401_12890_gb300 import ssm
    rng = np.random.default_rng(3)
    K = rng.standard_normal((20, 30))
    M = rng.standard_normal((20, 200)).astype(np.float32)
    M[7, 130] = bad
    plan = _plan(K, 200, form=form)
    with pytest.raises(ssm.SsmError) as e:
        plan.solve(torch.from_numpy(M).cuda())
    plan.close()
    assert e.value.status == ssm.SSM_ENAN


def test_extreme_scales():
    """Columns near the small end of the FP32 range keep their accuracy."""
    import torch
    rng = np.random.default_rng(5)
    K = rng.standard_normal((40, 24))
    M = (rng.standard_normal((40, 4)) * np.array([1e-36, 1e-25, 1.0, 1e15])).astype(np.float32)
    beta = 0.5
    plan = _plan(K, 4, beta=beta, form="dense")
    F, _ = plan.solve(torch.from_numpy(M).cuda())
    plan.close()
    A = np.linalg.solve(K.T @ K + beta * np.eye(24), K.T)
    h = np.maximum(A @ M.astype(np.float64), 0.0)
    err = np.abs(F.cpu().numpy().astype(np.float64) - h)
    # (beta / (beta + 1e-10) and the step's roundings: 1e-6; subnormals: spacing 2^-149)
    assert (err <= 1e-6 * h + 1e-8 * h.max(axis=0) + 2.0 ** -147).all()
