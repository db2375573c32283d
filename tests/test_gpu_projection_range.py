"""The data projections where the entries of a row of the operand or of a voxel's data differ
by orders of magnitude, and where the sum cancels: in the low-rank forms as accurate as an
FP64 accumulation.

S_1 = sigma_1 u_1^T m is seen through one iteration of the low-rank form at rank 1 from
zero with lambda = 0: F = max(0, v_1 S_1 / (beta + sigma_1^2)) beta / (beta + 1e-10). Bound:
the 9 FP32 roundings of that (as in the projections' other tests) and an FP64 accumulation's
P 2^-52 sum |a| |m|, the sum of the absolute terms and not the largest ones' product.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _first_component(u, M):
    """(F, reference, sum of absolute terms) for K = u v^T, v >= 0, and data M (P x N)."""
    import torch
    from paper_2401_12890_gb300 import ssm
    P, N = M.shape
    Q = 40
    v = np.random.default_rng(1).uniform(0.5, 1, Q)
    v /= np.linalg.norm(v)
    K = np.outer(u, v)
    beta = 0.5
    plan = ssm.Plan(K, (N, 1), 0.0, beta, form="lowrank", rank=1, max_iter=1, check_every=0)
    F, _ = plan.solve(torch.from_numpy(M).cuda())
    plan.close()
    s2 = float(u @ u)
    terms = u[:, None].astype(np.longdouble) * M.astype(np.longdouble)
    scale = (v / (beta + s2) * (beta / (beta + 1e-10)))[:, None]
    total = terms.sum(axis=0)[None, :]
    return (F.cpu().numpy().astype(np.float64), np.maximum(scale * total, 0).astype(np.float64),
            (scale * np.abs(terms).sum(axis=0)[None, :]).astype(np.float64))


def _check(u, M):
    F, ref, absolute = _first_component(u, M)
    bound = 9 * 2.0 ** -24 * ref + len(u) * 2.0 ** -52 * absolute + 2.0 ** -140
    err = np.abs(F - ref)
    assert (err <= bound).all(), float((err / bound).max())


@pytest.mark.parametrize("P", [2, 40, 120, 600, 1100])
@pytest.mark.parametrize("row,column", [(1e3, 1e3), (1e4, 1e4), (1e6, 1e4), (1.0, 1e10),
                                        (1e10, 1e10)])
def test_spikes_at_different_samples(P, row, column):
    """One large entry in the row of the operand, one in the voxel's data, at different p;
    all terms positive."""
    rng = np.random.default_rng(P)
    u = rng.uniform(0.5, 1, P)
    u[0] *= row
    u /= np.linalg.norm(u)
    M = rng.uniform(0.5, 1, (P, 150)).astype(np.float32)
    M[P - 1] *= np.float32(column)
    M[:, 7] = 0.0                              # and ordinary, empty and tiny columns among them
    M[:, 9] *= np.float32(1e-30)
    M[P - 1, 40:90] /= np.float32(column)
    _check(u, M)


@pytest.mark.parametrize("P", [32, 120, 513, 1000])
@pytest.mark.parametrize("level", [1e-2, 1e-5, 1e-8, 0.0])
def test_cancelling_sums(P, level):
    """Data nearly orthogonal to the row: the sum is `level` of its terms."""
    rng = np.random.default_rng(P)
    u = np.where(np.arange(P) % 2 == 0, 1.0, -1.0) * np.repeat(rng.uniform(0.5, 1, (P + 1) // 2), 2)[:P]
    u /= np.linalg.norm(u)
    M = np.repeat(rng.uniform(0.5, 1, ((P + 1) // 2, 140)), 2, axis=0)[:P]
    M = (M + level * rng.uniform(0, 1, M.shape) * np.sign(u)[:, None]).astype(np.float32)
    _check(u, M)


@pytest.mark.parametrize("P", [128, 512, 1024, 1500])
def test_constant_signals(P):
    """Every entry the same: every slice's products have one sign, and the sums of the slices'
    products are as large as they get."""
    for x in (0.8242, 0.99609, 0.5 + 2.0 ** -20, 0.66666):
        u = np.full(P, x) / np.sqrt(P)
        M = np.full((P, 130), x, np.float32)
        M[:, 1::2] = np.float32(1.0 - 2.0 ** -24)
        M[P // 2:, ::3] *= -1
        _check(u, M)


def test_zero_rows_and_columns():
    """A dictionary with an atom of zeros (a zero row of the full-rank operand) and data of
    zeros: exact zeros, and no others disturbed."""
    import torch
    from paper_2401_12890_gb300 import ssm
    rng = np.random.default_rng(2)
    K = rng.uniform(0, 1, (20, 70))
    K[:, 5] = 0.0
    M = rng.uniform(0, 1, (20, 200)).astype(np.float32)
    M[:, 100:] = 0.0
    plan = ssm.Plan(K, (200, 1), 0.0, 0.5, form="dense", max_iter=1, check_every=0)
    F = plan.solve(torch.from_numpy(M).cuda())[0].cpu().numpy()
    plan.close()
    h = np.linalg.solve(K.T @ K + 0.5 * np.eye(70), K.T @ M.astype(np.float64))
    assert np.all(F[5] == 0.0) and np.all(F[:, 100:] == 0.0)
    assert np.abs(F - np.maximum(h, 0)).max() <= 1e-6 * np.abs(h).max()


def test_full_rank_spikes():
    """(K^T K + beta I)^{-1} K^T with samples of very different gain, spiked voxels and ordinary
    ones. The full-rank forms drop less than 6 * 2^-40 of the row's and the column's
    power-of-two scales per term. A itself is formed in FP64 from the eigenpairs: its error,
    100 n 2^-53 ||K||^2 / beta relative (n = 90, ||K||^2 about 400: 4e-7), is on the absolute
    terms; 8 roundings of the result."""
    import torch
    from paper_2401_12890_gb300 import ssm
    rng = np.random.default_rng(4)
    P, Q, beta = 100, 90, 1e-3
    K = rng.standard_normal((P, Q))
    K[3] *= 1e-4                                # its weight in the inverse: large and small rows
    K[:, 11] *= 1e-3
    M = rng.standard_normal((P, 140)).astype(np.float32)
    M[3, ::2] *= np.float32(1e7)
    M[50, 1::3] *= np.float32(1e6)
    plan = ssm.Plan(K, (140, 1), 0.0, beta, form="dense", max_iter=1, check_every=0)
    F = plan.solve(torch.from_numpy(M).cuda())[0].cpu().numpy().astype(np.float64)
    plan.close()
    A = np.linalg.solve(K.T @ K + beta * np.eye(Q), K.T)
    M = M.astype(np.float64)
    h = np.maximum(A @ M, 0.0) * (beta / (beta + 1e-10))
    scales = 2.0 ** (np.ceil(np.log2(np.abs(A).max(axis=1)))[:, None] +
                     np.ceil(np.log2(np.abs(M).max(axis=0)))[None, :])
    bound = 8 * 2.0 ** -24 * h + 6 * P * 2.0 ** -40 * scales + 4e-7 * (np.abs(A) @ np.abs(M))
    err = np.abs(F - h)
    assert (err <= bound).all(), float((err / bound).max())
