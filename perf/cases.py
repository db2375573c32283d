"""Solves a user of the library runs, each through its public entry points (paper_2401_12890_gb300.ssm).

A case is a dict of plain values. `listed()` holds twelve; `draw(rng)` makes another one of
the same ranges. `prepare` plans once per dictionary and grid, as a program that
reconstructs many images of one protocol does, and puts an image's data on the GPU; `run`
is one call on it. `exact` is the same estimate in FP64 (torch only), `work` the bytes and
floating-point operations the iteration needs.

Kinds:
  solve      Plan.solve: one grid, one dictionary (optionally an object mask)
  batch      Plan(batch=B).solve: B slices of one protocol at once
  multi      MultiPlan.solve: a dictionary per voxel label (quantised transmit field)
  group      Group.solve: independent small problems of differing sizes together
  objective  Plan.objective: the value of Eq. 7 at an estimate
"""
import math

import numpy as np
import torch

from paper_2401_12890_gb300 import ssm, synth

LAM = 1e-2
SPARE_TOL = 1e-6      # tight enough that the iteration budget ends every solve

# Protocols: the encodings (e0 x e1) and compartments (a0 x a1) of the configurations in
# synth.WORKLOADS, the beta tuned for each and its K's ||K||_F^2 scale (P Q entries, or Q
# for normalised columns), and the rank the truncation rule gives there.
FAMILIES = {
    "dr_small": ("dr2d_tiny", 6, 5, 15, 15, 20),
    "dr": ("dr2d_slice", 15, 8, 50, 50, 20),
    "ir": ("rr3d_t1t2", 8, 8, 40, 40, 30),
    "spgr": ("mrf2d", 1000, 1, 30, 30, 8),
    "t2": ("mse_t2", 32, 1, 300, 1, 13),
}
# sizes of the group's problems: dims, P, Q (the shapes of the batching benchmark)
GROUP_SHAPES = [((32, 32), 30, 225), ((24, 20), 16, 100), ((48, 16), 24, 64),
                ((64,), 12, 50), ((12, 10, 6), 20, 80), ((40, 40), 30, 144)]


def _case(name, kind, family, dims, form="lowrank", precision="fp32", iters=100, check=0,
          mask=False, count=1, enc=None, atoms=None):
    w, e0, e1, a0, a1, rank = FAMILIES[family]
    if enc:
        e0, e1 = enc
    if atoms:
        a0, a1 = atoms
    base = FAMILIES[family]
    scale = a0 * a1 / (base[3] * base[4])
    if family != "spgr":
        scale *= e0 * e1 / (base[1] * base[2])
    dims = tuple(dims) + (1,) * (3 - len(dims))
    case = {"kind": kind, "family": family, "nx": dims[0], "ny": dims[1], "nz": dims[2],
            "e0": e0, "e1": e1, "a0": a0, "a1": a1, "form": form, "precision": precision,
            "iters": iters, "check": check, "mask": mask, "count": count,
            "beta": synth.WORKLOADS[w].beta * scale, "rank": min(rank, e0 * e1)}
    return {"name": name, **case} if name else case


def listed():
    return [
        # a 32 x 32 region of interest: a few microseconds of GPU work per iteration, so
        # launches and latency count
        _case("roi_lowrank_tf32x3", "solve", "dr_small", (32, 32), "lowrank", "tf32x3", iters=300),
        # the usual call: one slice in the tensor-core low-rank form, with the stopping
        # rule tested every 10 iterations
        _case("slice_lowrank_tf32x3", "solve", "dr", (128, 128), "lowrank", "tf32x3", check=10),
        # the same slice in the default form (plain FP32)
        _case("slice_lowrank_fp32", "solve", "dr", (128, 128), "lowrank", "fp32"),
        # a volume: the largest state (3.8 GB per map set), six neighbours per voxel
        _case("volume_lowrank_tf32x3", "solve", "ir", (96, 96, 64), "lowrank", "tf32x3", iters=20),
        # fingerprinting: a tall dictionary (1000 time points) of small rank
        _case("fingerprint_lowrank_fp32", "solve", "spgr", (192, 192), "lowrank", "fp32"),
        # full-rank f-step on the tensor cores, no truncation of the dictionary
        _case("slice_dense_bf16x3", "solve", "dr", (128, 128), "dense", "bf16x3", iters=30),
        # the same on an odd-sized fingerprinting slice: ragged tiles, projections on every
        # one of 900 directions
        _case("fingerprint_dense_bf16x3", "solve", "spgr", (157, 131), "dense", "bf16x3", iters=30),
        # multicomponent T2 in an object mask, full-rank in plain FP32
        _case("masked_t2_dense_fp32", "solve", "t2", (84, 72), "dense", "fp32", mask=True),
        # a stack of odd-sized small slices of one protocol solved at once
        _case("batched_slices_tf32x3", "batch", "dr_small", (37, 29), "lowrank", "tf32x3", count=40),
        # a dictionary per transmit-field level (61 levels)
        _case("b1_levels_lowrank_fp32", "multi", "spgr", (156, 156), "lowrank", "fp32", count=61,
              enc=(120, 1)),
        # small requests of differing sizes solved together, as the server groups them
        _case("group_lowrank_fp32", "group", "dr_small", (32, 32), "lowrank", "fp32", count=24),
        # the objective of an estimate (convergence reports, choice of beta)
        _case("slice_objective", "objective", "dr", (128, 128), "lowrank", "fp32"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def iters_for(per_iter, most):     # no draw costs more than the listed volume
        return max(5, min(log(20, 300), int(most / per_iter)))

    kind = rng.choice(["solve"] * 7 + ["batch", "multi", "group", "objective"])
    form, precision = rng.choice([("lowrank", "tf32x3")] * 3 + [("lowrank", "fp32")] * 2 +
                                 [("dense", "bf16x3")] * 2 + [("dense", "fp32")])
    if kind == "group":
        return _case(None, kind, "dr_small", (32, 32), iters=log(20, 150), count=rng.randint(4, 32))
    if kind == "multi":
        dims, levels = (log(40, 156), log(40, 156)), rng.randint(5, 61)
        return _case(None, kind, "spgr", dims, iters=log(20, 100), count=levels,
                     enc=(rng.randint(60, 120), 1))
    if kind == "batch":
        if form == "dense":
            form, precision = "lowrank", "tf32x3"
        return _case(None, kind, "dr_small", (log(20, 48), log(20, 48)), form, precision,
                     iters=log(20, 150), count=rng.randint(2, 64))
    family = rng.choice(["dr", "ir", "spgr", "t2", "dr_small"])
    enc = atoms = None
    if family in ("dr", "ir"):
        enc = (rng.randint(5, 15 if family == "dr" else 7), rng.randint(4, 8))
        side = 50 if family == "dr" else 40
        atoms = (log(12, side), log(12, side))
    elif family == "spgr":
        enc = (log(120, 1000), 1)
    if family == "ir" and form == "lowrank" and kind == "solve":
        dims = (log(16, 96), log(16, 96), log(8, 64))
    else:
        dims = (log(24, 192), log(24, 192))
    case = _case(None, kind, family, dims, form, precision, check=rng.choice([0, 10]),
                 mask=kind == "solve" and len(dims) == 2 and rng.random() < 0.2, enc=enc, atoms=atoms)
    n, q = math.prod(dims), case["a0"] * case["a1"]
    if kind == "objective":
        case.update(form="lowrank", precision="fp32", check=0)
    elif form == "lowrank":
        case["iters"] = iters_for(n * q, 1.5e10)
    else:
        case["iters"] = iters_for(2.0 * q * q * n, 6e12 if precision == "bf16x3" else 1e12)
    return case


# --------------------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------------------

def _dims(case):
    if case["nz"] > 1:
        return (case["nx"], case["ny"], case["nz"])
    return (case["nx"], case["ny"])


def _dictionary(case, b1=1.0):
    e0, e1, a0, a1 = case["e0"], case["e1"], case["a0"], case["a1"]
    family = case["family"]
    if family in ("dr", "dr_small"):
        return synth.diffusion_relaxation_dictionary(
            np.linspace(0, 3000, e0), np.linspace(60, 200, e1),
            np.geomspace(1e-4, 3e-3, a0), np.geomspace(10, 300, a1))
    if family == "ir":
        return synth.inversion_recovery_dictionary(
            np.geomspace(50, 3000, e0), np.linspace(10, 300, e1),
            np.geomspace(200, 4000, a0), np.geomspace(10, 300, a1))
    if family == "spgr":
        return synth.spgr_fingerprint_dictionary(
            e0, np.geomspace(200, 4000, a0), np.geomspace(10, 300, a1), seed=1045, b1=b1)
    return synth.multi_echo_t2_dictionary(np.arange(1, e0 + 1) * 10.0, np.geomspace(10, 2000, a0))


def _maps(dims, seed, count):
    """count smooth maps over the grid (a few low-frequency cosines each), voxel order."""
    rng = np.random.default_rng(seed)
    axes = [torch.arange(d, dtype=torch.float64, device="cuda") / d for d in reversed(dims)]
    mesh = torch.meshgrid(*axes, indexing="ij")
    out = []
    for _ in range(count):
        field = torch.zeros(tuple(reversed(dims)), dtype=torch.float64, device="cuda")
        for _ in range(4):
            k, ph = rng.uniform(0.3, 2.0, len(dims)) * 2 * np.pi, rng.uniform(0, 2 * np.pi)
            field += torch.cos(sum(float(a) * m for a, m in zip(k, mesh)) + float(ph))
        out.append(field.reshape(-1) / 4)
    return torch.stack(out)


def _truth(case, dims, seed):
    """Spectra (Q x 3, Gaussian peaks) and amplitudes (3 x N): two peaks everywhere, the
    third in a part of the image."""
    S = synth.spectral_peaks((case["a0"], case["a1"]),
                             [(0.25, 0.30), (0.60, 0.65), (0.80, 0.25)],
                             [(0.07, 0.09), (0.08, 0.06), (0.06, 0.07)])
    A = _maps(dims, seed, 3)
    A[:2] = 1.0 + 0.5 * A[:2]
    A[2] = 1.5 * A[2].clamp(min=0.0)
    return torch.from_numpy(S).cuda(), A


def _mask(case):
    return synth.ellipse_mask(_dims(case), 0.9695) if case["mask"] else None


def _noisy(clean, snr, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    noise = torch.randn(clean.shape, generator=gen, device="cuda", dtype=torch.float32)
    return (clean + noise * (clean[0].abs().max() / snr)).float().contiguous()


def _data(case, K, seed):
    """An image's data (P x N float32 on the GPU): K times the truth, plus noise."""
    dims = _dims(case)
    if case["kind"] == "batch":
        dims = dims + (case["count"],)
    S, A = _truth(case, dims, seed)
    mask = _mask(case)
    if mask is not None:
        A = A * torch.from_numpy(mask).cuda()
    return _noisy((torch.from_numpy(K).cuda() @ S) @ A, 50.0 if case["family"] == "spgr" else 100.0,
                  seed)


def _levels(case):
    return [_dictionary(case, b1) for b1 in np.linspace(0.8, 1.2, case["count"])]


def _multi_data(case, Ks, seed):
    """(labels, data): a smooth transmit field quantised to the levels, data per level."""
    dims = _dims(case)
    field = _maps(dims, seed + 1, 1)[0]
    u = (field - field.min()) / (field.max() - field.min())
    labels = (u * len(Ks)).long().clamp(max=len(Ks) - 1)
    S, A = _truth(case, dims, seed)
    KS = torch.stack([torch.from_numpy(K).cuda() @ S for K in Ks])       # level x P x 3
    clean = torch.empty((case["e0"], labels.numel()), dtype=torch.float64, device="cuda")
    for c in range(len(Ks)):
        sel = (labels == c).nonzero()[:, 0]
        clean[:, sel] = KS[c] @ A[:, sel]
    return labels, _noisy(clean, 50.0, seed)


def _group_problems(case, seed):
    """(dims, K, M) of each problem: the shapes in turn, a random dictionary each."""
    out = []
    for i in range(case["count"]):
        dims, P, Q = GROUP_SHAPES[i % len(GROUP_SHAPES)]
        K, M, _ = synth.random_problem(P, Q, dims, seed=1000 * (seed % 100000) + i, snr=60.0)
        out.append((dims, K, torch.from_numpy(M.astype(np.float32)).cuda()))
    return out


def _estimate(case, seed):
    """An estimate to evaluate: the truth with a smooth error, nonnegative (Q x N float32)."""
    S, A = _truth(case, _dims(case), seed)
    B = _maps(_dims(case), seed + 7, 3)
    return ((S @ (A * (1.0 + 0.05 * B))).clamp(min=0.0)).float().contiguous()


# --------------------------------------------------------------------------------------
# the calls
# --------------------------------------------------------------------------------------

def _stopping(case):
    tol = SPARE_TOL if case["check"] else 0.0
    return dict(max_iter=case["iters"], check_every=case["check"], tol_primal=tol, tol_change=tol)


def prepare(case, seed):
    kind, dims = case["kind"], _dims(case)
    if kind == "group":
        problems = _group_problems(case, seed)
        plans = [ssm.Plan(K, d, 0.02, 0.3, **_stopping(case)) for d, K, _ in problems]
        return {"kind": kind, "group": ssm.Group(plans), "plans": plans,
                "Ms": [M for _, _, M in problems]}
    if kind == "multi":
        Ks = _levels(case)
        labels, M = _multi_data(case, Ks, seed)
        plan = ssm.MultiPlan(Ks, labels.cpu().numpy(), dims, LAM, case["beta"], **_stopping(case))
        return {"kind": kind, "plan": plan, "M": M}
    K = _dictionary(case)
    plan = ssm.Plan(K, dims, LAM, case["beta"], form=case["form"], precision=case["precision"],
                    batch=case["count"] if kind == "batch" else None, **_stopping(case))
    if case["mask"]:
        plan.set_mask(_mask(case))
    state = {"kind": kind, "plan": plan, "M": _data(case, K, seed)}
    if kind == "objective":
        state["F"] = _estimate(case, seed)
    return state


def run(state):
    if state["kind"] == "group":
        Fs, _, _ = state["group"].solve(state["Ms"])
        return Fs
    if state["kind"] == "objective":
        return state["plan"].objective(state["M"], state["F"], use_full_k=True)
    F, info = state["plan"].solve(state["M"])
    return {"F": F, "iterations": info["iterations"]}


def work(case):
    """The data read and the maps written once; per iteration the rank-r products cost 4 r
    per element, the full-rank one 2 Q, the z-step and dual step about 12; the projections
    2 P per direction and voxel. (An iterate that on-chip memory cannot hold also moves
    8 bytes per element and iteration; those are not counted.)"""
    if case["kind"] == "group":
        sizes = [(math.prod(d), p, q, p) for d, p, q in
                 (GROUP_SHAPES[i % len(GROUP_SHAPES)] for i in range(case["count"]))]
    else:
        n = case["nx"] * case["ny"] * case["nz"] * (case["count"] if case["kind"] == "batch" else 1)
        sizes = [(n, case["e0"] * case["e1"], case["a0"] * case["a1"], case["rank"])]
    total = {"bytes": 0, "flops": 0}
    for n, p, q, r in sizes:
        if case["kind"] == "objective":
            total["bytes"] += 4 * (n * (p + q) + p * q)
            total["flops"] += 2 * p * q * n
            continue
        dense = case["form"] == "dense"
        total["bytes"] += 4 * n * (p + q)
        total["flops"] += case["iters"] * n * q * ((2 * q if dense else 4 * r) + 12)
        total["flops"] += 2 * n * p * (min(p, q) if dense else r)
    return total


# --------------------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------------------

def _neighbours(z, dims):
    """Sum of every voxel's grid neighbours for each map (Q x N)."""
    g = z.view((z.shape[0],) + tuple(reversed(dims)))
    out = torch.zeros_like(g)
    for ax in range(1, g.dim()):
        n = g.shape[ax]
        if n > 1:
            out.narrow(ax, 0, n - 1).add_(g.narrow(ax, 1, n - 1))
            out.narrow(ax, 1, n - 1).add_(g.narrow(ax, 0, n - 1))
    return out.view_as(z)


def _factors(K):
    """Singular values, left and right vectors, and the truncation rank (error below 5e-5
    of ||K||_F)."""
    U, s, Vt = np.linalg.svd(K, full_matrices=False)
    tail = np.sqrt(np.append(np.cumsum((s ** 2)[::-1])[::-1], 0.0) / np.sum(s ** 2))
    return U, s, Vt.T, int(np.argmax(tail < 5e-5))


def _iterate(G, f_step, dims, lam, beta, iters, mask=None):
    """The linearized ADMM iteration from zero."""
    inside = torch.ones(G.shape[1], dtype=torch.float64, device="cuda") if mask is None else mask
    deg = _neighbours(inside[None], dims) * inside
    xi = 0.75 * lam * 2.0 * sum(2.0 - 2.0 * math.cos(math.pi * (n - 1) / n) for n in dims if n > 1) + 1e-10
    z, d = torch.zeros_like(G), torch.zeros_like(G)
    for _ in range(iters):
        f = f_step(torch.add(G, z, alpha=beta).sub_(d))
        lap = _neighbours(z, dims).neg_().addcmul_(deg, z)
        zn = lap.mul_(-2.0 * lam).add_(z, alpha=xi).add_(f, alpha=beta).add_(d)
        zn = zn.div_(xi + beta).clamp_(min=0.0).mul_(inside)
        d = d.sub_(zn, alpha=beta).add_(f, alpha=beta).mul_(inside)
        z = zn
    return z


def _solve_exact(K, M, dims, lam, beta, iters, dense, mask=None):
    U, s, V, r = _factors(K)
    n = s.size
    r = n if dense else r
    U, s, V = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (U[:, :r], s[:r], V[:, :r]))
    G = V @ (s[:, None] * (U.T @ M.double()))
    W = (s ** 2 / (beta * beta + beta * s ** 2))[:, None]
    if dense and K.shape[0] >= K.shape[1]:
        # the right vectors are complete: one Q x Q product
        inverse = (V / (s ** 2 + beta)) @ V.T
        return _iterate(G, lambda c: inverse @ c, dims, lam, beta, iters, mask)
    return _iterate(G, lambda c: torch.addmm(c / beta, V, W * (V.T @ c), alpha=-1.0), dims, lam,
                    beta, iters, mask)


def _multi_exact(case, seed):
    Ks = _levels(case)
    labels, M = _multi_data(case, Ks, seed)
    M = M.double()
    beta, G, steps = case["beta"], None, []
    for c, K in enumerate(Ks):
        sel = (labels == c).nonzero()[:, 0]
        if not sel.numel():
            continue
        U, s, V, r = _factors(K)
        U, s, V = (torch.from_numpy(np.ascontiguousarray(x)).cuda()
                   for x in (U[:, :r], s[:r], V[:, :r]))
        if G is None:
            G = torch.empty((K.shape[1], labels.numel()), dtype=torch.float64, device="cuda")
        G[:, sel] = V @ (s[:, None] * (U.T @ M[:, sel]))
        steps.append((sel, V, (s ** 2 / (beta * beta + beta * s ** 2))[:, None]))

    def f_step(c):
        f = c / beta
        for sel, V, W in steps:
            f[:, sel] -= V @ (W * (V.T @ c[:, sel]))
        return f

    return _iterate(G, f_step, _dims(case), LAM, beta, case["iters"])


def exact(case, seed):
    kind, dims = case["kind"], _dims(case)
    if kind == "group":
        return [_solve_exact(K, M, d, 0.02, 0.3, case["iters"], False)
                for d, K, M in _group_problems(case, seed)]
    if kind == "multi":
        return {"F": _multi_exact(case, seed), "iterations": None}
    K = _dictionary(case)
    M = _data(case, K, seed)
    if kind == "objective":
        F = _estimate(case, seed).double()
        grid = F.view((F.shape[0],) + tuple(reversed(dims)))
        rough = sum(float((grid.diff(dim=ax) ** 2).sum()) for ax in range(1, grid.dim()))
        return 0.5 * float(((M.double() - torch.from_numpy(K).cuda() @ F) ** 2).sum()) + LAM * rough
    mask = _mask(case)
    if mask is not None:
        mask = torch.from_numpy(mask).cuda().double()
    if kind == "batch":
        # slices are independent: the maps of all slices are maps of one slice's grid
        B, n = case["count"], math.prod(dims)
        z = [_solve_exact(K, M[:, b * n:(b + 1) * n], dims, LAM, case["beta"], case["iters"], False)
             for b in range(B)]
        return {"F": torch.cat(z, dim=1), "iterations": None}
    return {"F": _solve_exact(K, M, dims, LAM, case["beta"], case["iters"], case["form"] == "dense",
                              mask), "iterations": None}
