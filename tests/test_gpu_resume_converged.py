"""A solve that stops on its tolerance and is continued: the first residual test of the
continuation belongs to the iteration it stands on, whatever the plan solved before.

The low-rank forms store d only around tests, so the iteration that stops a solve early
leaves none, and the continuation has to form it. Bars: the iterates of an uninterrupted
solve, bit for bit, and its residuals; the oracle's primal residual ||z - f|| / ||z|| to 2e-5,
as z and f are each held to 1e-5 of their norm (another d moves it by ||d|| / beta, 0.4 of
the norm here).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FORMS = [("lowrank", "fp32"), ("lowrank", "tf32x3"), ("dense", "fp32"), ("dense", "bf16x3"),
         ("admm", "fp32"), ("multi", "patches"), ("multi", "table")]


def _plans(form, prec, dims, labels):
    """(make plan, K per dictionary)"""
    from paper_2401_12890_gb300 import ssm, synth
    K, M, _ = synth.random_problem(20, 70, dims, seed=11, snr=50.0)
    if form != "multi":
        return lambda **kw: ssm.Plan(K, dims, 0.05, 0.8, form=form, precision=prec, **kw), K, M
    Ks = np.stack([K, K])             # both labels' dictionary: the oracle of one holds
    rank = 8 if prec == "patches" else 20
    return lambda **kw: ssm.MultiPlan(Ks, labels, dims, 0.05, 0.8, rank=rank, **kw), K, M


@pytest.mark.parametrize("graphs", [False, True])
@pytest.mark.parametrize("first,every", [(1, 0), (3, 1)])
@pytest.mark.parametrize("form,prec", FORMS, ids=[f"{a}_{b}" for a, b in FORMS])
def test_first_test_after_early_stop(form, prec, first, every, graphs):
    import torch
    from oracle import ladmm as L
    dims = (50, 41)
    n = dims[0] * dims[1]
    labels = (np.arange(n) % 2).astype(np.int32)
    make, K, M = _plans(form, prec, dims, labels)
    Md = torch.from_numpy(np.ascontiguousarray(M, np.float32)).cuda()
    # stops at iteration 10 (a loose tolerance), with no test due at iteration 11
    plan = make(max_iter=40, check_every=10, tol_primal=0.9, tol_change=0.9)
    if graphs:
        plan.set_graphs(True)
    plan.solve(Md * 1e15)             # leaves d of another scale, if any, behind
    _, info = plan.solve(Md)
    assert info["iterations"] == 10 and info["status"] == 0
    plan.params.check_every, plan.params.tol_change = every, 0.0
    plan.params.tol_primal = 1e-12 if every else 0.0
    plan.set_max_iter(first)
    F, info = plan.resume(Md)
    F2, _ = plan.resume(Md)           # and on from there
    plan.close()
    whole = make(max_iter=10 + first, check_every=0)
    Fw, iw = whole.solve(Md)
    whole.set_max_iter(10 + 2 * first)
    Fw2, _ = whole.solve(Md)
    whole.close()
    assert torch.equal(F, Fw) and torch.equal(F2, Fw2)
    assert info["res_change"] == pytest.approx(iw["res_change"], rel=1e-6)
    assert info["res_primal"] == pytest.approx(iw["res_primal"], rel=1e-6)
    if form in ("lowrank", "dense"):
        ref = L.ladmm(K, M.astype(np.float32).astype(np.float64), dims, 0.05, 0.8,
                      dense=form == "dense", iters=10 + first, check_every=1,
                      return_history=True)
        assert info["res_primal"] == pytest.approx(ref["history"][-1][1], abs=2e-5)
