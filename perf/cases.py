"""Performance cases of the separated-operator library: what a user's program has it do.

Every function is a sum of unit-charge Gaussians in the cell [-L, L]^3 (exponents log-uniform,
centres uniform in [-20, 20]^3), every operator 1/r or exp(-mu r)/r as a sum of M Gaussians, as in
the repository's workloads.  A case names a `kind` (which entry points run), the order k, the
sizes and a function of the family; the seed turns and mirrors that function in its cell (one of the
cube's 48 symmetries) and gives its sign, so that every seed has other values on other boxes but as
many of them.  `exact` recomputes a case in plain 64-bit torch, with its own fit, blocks, screen,
two-scale filters and tree logic.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1507_01888_gb300 import mra, solvers

L_CELL = 32.0


# ------------------------------------------------------------------------------------ the cases

def listed():
    bsh10 = {"kernel": "bsh", "mu": 1.0, "M": 60, "k": 10, "thresh": 1e-6, "a_lo": 1.0, "a_hi": 1e4}
    return [
        # The smallest call: a 64-box tree through the default (FP64) apply; launches and
        # synchronisations count.
        {"name": "fp64_uniform_k6_l2", "kind": "apply", "precision": "fp64", "kernel": "poisson", "M": 20, "k": 6,
         "function": 1, "level": 2, "gaussians": 3, "a_lo": 10.0, "a_hi": 1e3},
        # An ordinary small tree (the plain Poisson workload: 512 boxes) in split precision.
        {"name": "split_uniform_k6_l3", "kind": "apply", "precision": "split", "kernel": "poisson", "M": 20, "k": 6,
         "function": 1, "level": 3, "gaussians": 3, "a_lo": 10.0, "a_hi": 1e3},
        # The bound-state Helmholtz apply on an adaptive k = 10 tree with the norm screen, in the
        # default precision: what thresholds below 1e-7 need, and the reference of every accuracy check.
        {"name": "fp64_bsh_k10", "function": 2, "kind": "apply", "precision": "fp64", "gaussians": 8, **bsh10},
        # The same apply in split precision as the benchmark runs it: recorded once, replayed with one
        # graph launch per step, four terms joined per flush (what the tuner settles on).
        {"name": "split_bsh_k10_graph", "function": 2, "kind": "graph", "precision": "split", "gaussians": 8, "join": 4,
         **bsh10},
        # Several functions in one pass (a batch of orbitals or densities), k = 8.
        {"name": "split_batched_k8", "kind": "batched", "precision": "split", "functions": 16, "kernel": "poisson",
         "function": 3, "M": 40, "k": 8, "thresh": 1e-5, "a_lo": 1.0, "a_hi": 1e3, "gaussians": 8},
        # High order, low threshold (k = 14, M = 100): the other tensor-core kernel, in the tile shape the
        # tuner settles on.
        {"name": "split_poisson_k14", "kind": "apply", "precision": "split", "kernel": "poisson", "M": 100, "k": 14,
         "function": 5, "thresh": 1e-8, "gaussians": 2, "a_lo": 1.0, "a_hi": 1e6, "tile_variant": 1},
        # The operator's long range: non-standard form on a uniform tree, split precision (k and 2k = 12).
        {"name": "split_ns_uniform_k6_l4", "kind": "ns_uniform", "precision": "split", "kernel": "poisson", "M": 40,
         "function": 6, "k": 6, "level": 4, "gaussians": 16, "a_lo": 0.05, "a_hi": 2.0, "tile_variant": 1},
        # Non-standard form on an adaptive tree at the bound-state workload's own k = 10 (2k = 20), FP64.
        {"name": "fp64_ns_tree_k10", "function": 2, "kind": "ns_tree", "precision": "fp64", "gaussians": 1, **bsh10,
         "thresh": 1e-4},
        # One iteration of the bound-state solver, as the solver calls it: product, refit, non-standard
        # apply with the norm screen, truncation, inner products.
        {"name": "bsh_step_k6", "kind": "bsh_step", "precision": "split", "k": 6, "thresh": 1e-4, "M": 60,
         "function": 7},
        # After an apply: the multi-level result summed down to leaves and coarsened.
        {"name": "reconstruct_truncate_k10", "function": 2, "kind": "post", "precision": "split", "gaussians": 8,
         **bsh10},
        # Where every function comes from: adaptive projection of a Gaussian sum.
        {"name": "project_k10", "function": 2, "kind": "project", "k": 10, "thresh": 1e-6, "gaussians": 8, "a_lo": 1.0,
         "a_hi": 1e4},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _thresh(rng, k):
    """A tree's threshold within the decade that its order is used for: low orders would need far deeper trees."""
    hi = 1e-3 if k <= 5 else 1e-4 if k <= 7 else 1e-5
    return _log(rng, 0.1 * hi, hi)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "graph", "batched", "ns_uniform", "ns_tree", "bsh_step", "post",
                       "project"])
    prec = rng.choice(["fp64", "split"])
    kernel = rng.choice(["poisson", "bsh"])
    c = {"kind": kind, "precision": prec, "kernel": kernel, "M": rng.randint(12, 80), "a_lo": 1.0,
         "a_hi": _log(rng, 1e2, 1e4), "function": rng.randint(10, 10 ** 6)}
    if kernel == "bsh":
        c["mu"] = _log(rng, 0.4, 3.0)
    if kind == "apply" and rng.random() < 0.5:  # a whole level
        c.update(k=rng.choice([3, 4, 5, 6, 7, 8, 9, 10]) if prec == "fp64" else rng.choice([4, 6, 8, 10]),
                 level=rng.randint(1, 3), gaussians=rng.randint(1, 8))
        return c
    if kind == "apply":  # an adaptive tree; odd orders run in FP64 only, 12 and more in their own kernels
        c.update(k=rng.choice([4, 5, 6, 7, 8, 9, 10]) if prec == "fp64" else rng.choice([6, 8, 10, 12, 14]),
                 gaussians=rng.randint(1, 3))
    elif kind == "graph":
        c.update(precision="split", k=rng.choice([6, 8, 10]), gaussians=rng.randint(1, 8), join=rng.choice([0, 4]))
    elif kind == "batched":
        c.update(precision="split", k=rng.choice([6, 8]), functions=rng.randint(2, 16), gaussians=rng.randint(1, 4),
                 a_hi=1e3)
    elif kind == "ns_uniform":
        c.update(k=rng.choice([4, 6]), level=rng.randint(2, 4), gaussians=rng.randint(4, 16), a_lo=0.05, a_hi=2.0)
        return c
    elif kind == "ns_tree":
        c.update(k=rng.choice([4, 6, 8]), gaussians=1, thresh=_log(rng, 1e-4, 1e-3))
        return c
    elif kind == "bsh_step":
        return {"kind": kind, "precision": "split", "k": rng.choice([4, 6]), "thresh": _log(rng, 1e-4, 1e-3),
                "M": rng.randint(40, 80), "function": c["function"]}
    elif kind == "post":
        c.update(precision="split", k=rng.choice([4, 6, 8, 10]), gaussians=rng.randint(1, 8))
    else:
        c = {"kind": kind, "k": rng.choice([4, 5, 6, 7, 8, 10, 12]), "gaussians": rng.randint(1, 8), "a_lo": 1.0,
             "a_hi": c["a_hi"], "function": c["function"]}
    c["thresh"] = _thresh(rng, c["k"])
    return c


def _turned(a, coef, c, seed):
    """The Gaussian sum with its centres turned and mirrored, and its sign, by the seed."""
    q = seed % 96
    c = c[:, list(itertools.permutations(range(3)))[q % 6]] * [1 - 2 * (q // 6 & 1), 1 - 2 * (q // 12 & 1),
                                                                1 - 2 * (q // 24 & 1)]
    return {"coef": coef * (1 - 2 * (q // 48)), "expnt": a, "cx": c[:, 0].copy(), "cy": c[:, 1].copy(),
            "cz": c[:, 2].copy()}


def _gaussian_sum(n, a_lo, a_hi, function, seed):
    rng = np.random.default_rng(function)
    a = np.exp(rng.uniform(np.log(a_lo), np.log(a_hi), size=n))
    return _turned(a, (a / np.pi) ** 1.5, rng.uniform(-20.0, 20.0, size=(n, 3)), seed)


def _functions(case, seed):
    """The Gaussian sums of a case; a batch has 1 .. gaussians of them in each function."""
    if case["kind"] != "batched":
        return [_gaussian_sum(case["gaussians"], case["a_lo"], case["a_hi"], case["function"], seed)]
    counts = np.random.default_rng(case["function"]).integers(1, case["gaussians"] + 1, size=case["functions"])
    return [_gaussian_sum(int(n), case["a_lo"], case["a_hi"], 1000 * case["function"] + i, seed + 7 * i)
            for i, n in enumerate(counts)]


def _tau(case):
    """The norm screen's threshold: 0.01 times the tree's; whole levels are applied unscreened."""
    return 0.01 * case["thresh"] if "thresh" in case and case["kind"] != "ns_tree" else 0.0


def _opts(case):
    kw = {"precision": mra.PREC_SPLIT_BF16 if case["precision"] == "split" else mra.PREC_FP64,
          "tile_variant": case.get("tile_variant", 0), "join": case.get("join", 0)}
    if case["kind"] in ("ns_uniform", "ns_tree"):
        return mra.make_opts(stencil=mra.STENCIL_SHELLS, max_disp=1, **kw)
    if "level" in case:
        return mra.make_opts(stencil=mra.STENCIL_NEAREST, **kw)
    return mra.make_opts(stencil=mra.STENCIL_SHELLS, max_disp=1, screen=mra.SCREEN_NORM, tau=_tau(case), **kw)


def _trees(case, seed):
    kw = {"uniform_level": case["level"]} if "level" in case else {"thresh": case["thresh"]}
    return [mra.project(f, case["k"], L_CELL, **kw) for f in _functions(case, seed)]


def _operator(case, lo, hi, max_disp):
    kern = mra.BSH if case["kernel"] == "bsh" else mra.POISSON
    return mra.Operator(kern, case["M"], case["k"], L_CELL, lo, hi, max_disp=max_disp, mu=case.get("mu", 0.0),
                        fit_eps=case.get("thresh", 1e-5))


def _levels(tree):
    lev = tree.keys[: tree.n] >> 57
    return int(lev.min()), int(lev.max())


def _bsh_inputs(case, seed):
    """-1/r at the origin, an orbital near e^-r (three Gaussians, slightly off the centre) and an energy near -1/2."""
    rng = np.random.default_rng(case["function"])
    k, thresh = case["k"], case["thresh"]
    V, _ = solvers.project_potential(1.0, k, 20.0, thresh)
    a = np.array([0.11, 0.41, 2.2])
    g = _turned(a, np.array([0.44, 0.54, 0.15]) * (2 * a / math.pi) ** 0.75, rng.uniform(-0.2, 0.2, size=(3, 3)), seed)
    return V, mra.project(g, k, 20.0, thresh=thresh), float(rng.uniform(-0.55, -0.45))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "project":
        return {"case": case, "function": _functions(case, seed)[0]}
    if kind == "bsh_step":
        V, psi, E = _bsh_inputs(case, seed)
        return {"case": case, "V": V, "psi": psi, "E": E, "cache": {}}
    trees = _trees(case, seed)
    tree, offsets = mra.concat_trees(trees) if kind == "batched" else (trees[0], None)
    s = {"case": case, "tree": tree, "offsets": offsets}
    lo, hi = _levels(tree)
    if kind in ("ns_uniform", "ns_tree"):
        s["op"] = _operator(case, 0, hi, 3)
        s["ns"] = mra.NSOperator(s["op"], max_disp=1)
        if kind == "ns_uniform":
            s["apply"] = mra.NSApplier(s["op"], s["ns"], tree, 1, _opts(case))
        else:
            s["apply"] = mra.NSTreeApplier(s["op"], s["ns"], 1, _opts(case), out_cap=8 * tree.n)
        return s
    s["op"] = _operator(case, lo, hi, 1)
    if kind == "apply":
        s["apply"] = mra.Applier(s["op"], tree, _opts(case))
    elif kind in ("graph", "batched"):
        s["graph"] = mra.ApplyGraph(s["op"], tree, _opts(case), offsets=offsets)
    else:  # post: the result of an apply is in hand
        s["result"], _ = mra.apply(s["op"], tree, _opts(case))
    return s


def _out(t):
    return {"keys": t.keys[: t.n], "coeffs": t.coeffs[: t.n]}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "project":
        return _out(mra.project(state["function"], case["k"], L_CELL, thresh=case["thresh"]))
    if kind == "bsh_step":
        E, psi, dE = solvers.bsh_step(state["V"], state["psi"], state["E"], case["thresh"], M_bsh=case["M"],
                                      cache=state["cache"])
        return {"E": E, "dE": dE, "psi": _out(psi)}
    if kind in ("graph", "batched"):
        return _out(state["graph"].launch())
    if kind == "post":
        leaves = mra.reconstruct(state["result"])
        small, err2 = mra.truncate(leaves, case["thresh"])
        return {"leaves": _out(leaves), "truncated": _out(small), "err2": err2}
    return _out(state["apply"](state["tree"]))


def work(case):
    """Nominal bytes and operations: trees in and out once; a mode product (2 k^4 operations) for each kept
    (source, displacement, Gaussian) term, the first two products of a term being shared with its neighbours.
    Sizes of adaptive trees are the mean of their family."""
    k, kind = case["k"], case["kind"]
    box = 8.0 * (k ** 3 + 1)
    if kind == "bsh_step":
        n = 10000 * (1e-4 / case["thresh"]) ** 0.3
        return {"bytes": n * box, "flops": n / 7 * 8 * case["M"] * 2 * ((2 * k) ** 4 + k ** 4)}
    if "level" in case:
        n = 8.0 ** case["level"]
    else:
        # leaves per Gaussian: about 500 (ten octaves of exponent) for each factor of ten in the threshold below 1e-2,
        # fewer at higher order
        per = 500 * math.log10(1e-2 / case["thresh"]) * (10.0 / k) * math.log10(10 * case["a_hi"] / case["a_lo"]) / 5
        fn = case["functions"] * (case["gaussians"] + 1) / 2 if kind == "batched" else case["gaussians"]
        n = max(64.0, per * fn)
    if kind == "project":
        return {"bytes": n * box, "flops": n * case["gaussians"] * 2 * k ** 3}
    if kind == "post":
        return {"bytes": 4 * n * box, "flops": n * 2 * 3 * 2 * 2 * k ** 4}
    if kind in ("ns_uniform", "ns_tree"):
        terms = n / 7 * 20 * case["M"]
        return {"bytes": 3 * n * box, "flops": terms * 2 * ((2 * k) ** 4 + k ** 4)}
    terms = n * case["M"] * (20 if "level" in case else 6)
    return {"bytes": 2 * n * box, "flops": terms * 2 * k ** 4}


# ------------------------------------------------------------ the same results in plain 64 bits

def _gl(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.tensor(0.5 * (x + 1), device="cuda"), torch.tensor(0.5 * w, device="cuda")


def _phi(k, x):
    """phi_i(x) = sqrt(2i+1) P_i(2x-1), i < k, in a new last dimension."""
    t = 2 * x - 1
    p = [torch.ones_like(t), t]
    for i in range(2, k):
        p.append(((2 * i - 1) * t * p[i - 1] - (i - 1) * p[i - 2]) / i)
    return torch.stack([math.sqrt(2 * i + 1) * p[i] for i in range(k)], dim=-1)


def _two_scale(k):
    """Ub[(c, i)][j] = 2^{-1/2} int_0^1 phi_i(y) phi_j((y+c)/2) dy."""
    x, w = _gl(k + 2)
    return torch.cat([torch.einsum("q,qi,qj->ij", w, _phi(k, x), _phi(k, 0.5 * (x + c))) / math.sqrt(2)
                      for c in (0, 1)])


def _key(n, x, y, z):
    return (n << 57) | (x << 38) | (y << 19) | z


def _xyz(keys):
    return (keys >> 38) & 0x7FFFF, (keys >> 19) & 0x7FFFF, keys & 0x7FFFF


def _find(sorted_keys, keys):
    """Positions of keys in sorted_keys, and which are there."""
    if len(sorted_keys) == 0:
        return torch.zeros_like(keys), torch.zeros_like(keys, dtype=torch.bool)
    p = torch.searchsorted(sorted_keys, keys).clamp(max=len(sorted_keys) - 1)
    return p, sorted_keys[p] == keys


def _children(keys):
    n = keys >> 57
    x, y, z = _xyz(keys)
    return torch.stack([_key(n + 1, 2 * x + (c >> 2), 2 * y + ((c >> 1) & 1), 2 * z + (c & 1)) for c in range(8)], 1)


def _parents(keys, up=1):
    x, y, z = _xyz(keys)
    return _key((keys >> 57) - up, x >> up, y >> up, z >> up)


def _down(Ub, s):
    """Coefficients on the eight children, [n, 8, k, k, k]."""
    k = Ub.shape[1]
    S = torch.einsum("ai,nijl->najl", Ub, s)
    S = torch.einsum("bj,najl->nabl", Ub, S)
    S = torch.einsum("cl,nabl->nabc", Ub, S)
    return S.reshape(-1, 2, k, 2, k, 2, k).permute(0, 1, 3, 5, 2, 4, 6).reshape(-1, 8, k, k, k)


def _up(Ub, ch):
    """(children's coefficients as one (2k)^3 tensor, their filter)."""
    k = Ub.shape[1]
    S = ch.reshape(-1, 2, 2, 2, k, k, k).permute(0, 1, 4, 2, 5, 3, 6).reshape(-1, 2 * k, 2 * k, 2 * k)
    s = torch.einsum("ai,nabc->nibc", Ub, S)
    s = torch.einsum("bj,nibc->nijc", Ub, s)
    return S, torch.einsum("cl,nijc->nijl", Ub, s)


def _fit(mu, M, r_lo, r_hi):
    """Trapezoid terms c_m, t_m of the kernel: the first (h, s_lo) of the grid with the least maximum
    relative error on 3000 log-spaced points."""
    p = torch.arange(3000, dtype=torch.float64, device="cuda")
    r = r_lo * (r_hi / r_lo) ** (p / 2999)
    K = torch.exp(-mu * r) / r
    m = torch.arange(M, dtype=torch.float64, device="cuda")

    def terms(h, s_lo):
        s = s_lo[..., None] + m * h
        return 2 / math.sqrt(math.pi) * h * torch.exp(s - mu * mu * torch.exp(-2 * s) / 4), torch.exp(2 * s)

    s_lo = (torch.arange(113, dtype=torch.float64, device="cuda") - 100) / 4
    best = (math.inf, 0.0, 0.0)
    for i in range(116):
        c, t = terms((5.0 + i) / 100.0, s_lo)
        tot = torch.zeros((113, 3000), dtype=torch.float64, device="cuda")
        for q in range(M):
            tot += c[:, q, None] * torch.exp(-t[:, q, None] * (r * r))
        err, j = ((tot - K).abs() / K).amax(1).min(0)
        if float(err) < best[0]:
            best = (float(err), (5.0 + i) / 100.0, float(s_lo[int(j)]))
    c, t = terms(best[1], torch.tensor(best[2], dtype=torch.float64, device="cuda"))
    return c, t


def _blocks(k, h, t, D):
    """R[m][l + D][i][j] = h int int phi_i(u) exp(-t_m h^2 (u-v+l)^2) phi_j(v) du dv: 24 panels of 20 points on
    each side of z = u - v = 0, over the part of it where the Gaussian is above e^-46 of its maximum."""
    gx, gw = _gl(20)
    kx, kw = _gl(k + 1)
    out = []
    for l in range(-D, D + 1):
        tot = 0.0
        T = t * h * h
        for wa, wb in ((l - 1.0, float(l)), (float(l), l + 1.0)):
            near = max(wa, -wb, 0.0)
            W = torch.sqrt(near * near + 46.0 / T)
            lo, hi = torch.clamp(-W, min=wa), torch.clamp(W, max=wb)
            pw = (hi - lo) / 24
            w = lo[:, None, None] + pw[:, None, None] * (torch.arange(24, device="cuda")[:, None] + gx)
            wt = (pw[:, None, None] * gw * torch.exp(-T[:, None, None] * w * w)).reshape(len(t), -1)
            z = (w - l).reshape(len(t), -1)
            a, b = z.clamp(min=0.0), (1.0 + z).clamp(max=1.0)
            u = a[..., None] + (b - a)[..., None] * kx
            tot = tot + torch.einsum("mz,mzq,mzqi,mzqj->mij", wt, (b - a)[..., None] * kw, _phi(k, u),
                                     _phi(k, u - z[..., None]))
        out.append(h * tot)
    return torch.stack(out, 1)


class _Op:
    """Blocks of one operator by level, made when first asked for; doubled(): of its 2k form."""

    def __init__(self, case_kernel, mu, M, k, L, fit_eps, max_disp):
        r_hi = min(2 * L, math.log(1 / fit_eps) / mu) if case_kernel == "bsh" else 2 * L
        self.c, self.t = _fit(mu if case_kernel == "bsh" else 0.0, M, 1e-4, r_hi)
        self.k, self.L, self.max_disp, self.have = k, L, max_disp, {}

    def level(self, n):
        if n not in self.have:
            self.have[n] = _blocks(self.k, 2 * self.L / 2 ** n, self.t, min(self.max_disp, 2 ** n - 1))
        return self.have[n]

    def doubled(self, n, D):
        R, k = self.level(n + 1), self.k
        D = min(D, 2 ** n - 1)
        mid = R.shape[1] // 2
        return torch.stack([torch.cat([torch.cat([R[:, 2 * l + ci - cj + mid] for cj in (0, 1)], -1)
                                       for ci in (0, 1)], -2) for l in range(-D, D + 1)], 1)


def _apply_level(n, keys, coeffs, c, R, D, shells, tau, f=None):
    """One level's boxes: every kept term's contribution, summed by destination key; of several functions f
    (under 64), by the key with f in the place of the level."""
    x, y, z = _xyz(keys)
    nb, mid = 1 << n, R.shape[1] // 2
    D = min(D, mid, nb - 1)
    N = R.flatten(2).norm(dim=2)
    sn = coeffs.flatten(1).norm(dim=1)
    ls = [(a, b, d) for a in range(-D, D + 1) for b in range(-D, D + 1) for d in range(-D, D + 1)]
    inside, keep = {}, {}
    for l in ls:
        ok = ((x + l[0]) >= 0) & ((x + l[0]) < nb) & ((y + l[1]) >= 0) & ((y + l[1]) < nb) & ((z + l[2]) >= 0) & \
            ((z + l[2]) < nb)
        B = (((c.abs() * N[:, l[0] + mid]) * N[:, l[1] + mid]) * N[:, l[2] + mid])[None] * sn[:, None]
        keep[l] = (B >= tau) & ok[:, None] if tau > 0 else ok[:, None].expand(len(keys), len(c))
        inside[l] = ok
    if shells and tau > 0:
        going = torch.ones(len(keys), dtype=torch.bool, device="cuda")
        for d in range(D + 1):
            shell = [l for l in ls if max(map(abs, l)) == d]
            for l in shell:
                keep[l] = keep[l] & going[:, None]
            going = going & torch.stack([keep[l].any(1) for l in shell]).any(0)
    first = torch.full_like(x, n) if f is None else f
    dest = {l: _key(first, x + l[0], y + l[1], z + l[2])[keep[l].any(1)] for l in ls}
    okeys = torch.unique(torch.cat(list(dest.values())))
    out = torch.zeros((len(okeys),) + coeffs.shape[1:], dtype=torch.float64, device="cuda")
    kept = {l: keep[l].any(0).tolist() for l in ls}
    for m in range(len(c)):
        for lx in range(-D, D + 1):
            t1 = None
            for ly in range(-D, D + 1):
                t2 = None
                for lz in range(-D, D + 1):
                    l = (lx, ly, lz)
                    if not kept[l][m]:
                        continue
                    if t1 is None:
                        t1 = torch.einsum("ai,nijl->najl", R[m, lx + mid], coeffs)
                    if t2 is None:
                        t2 = torch.einsum("bj,najl->nabl", R[m, ly + mid], t1)
                    b = keep[l][:, m].nonzero()[:, 0]
                    t3 = c[m] * torch.einsum("cl,nabl->nabc", R[m, lz + mid], t2[b])
                    out.index_add_(0, _find(okeys, _key(first[b], x[b] + lx, y[b] + ly, z[b] + lz))[0], t3)
    return okeys, out


def _apply(op, keys, coeffs, D, shells, tau):
    ks, cs = [], []
    lev = keys >> 57
    for n in torch.unique(lev).tolist():
        at = lev == n
        k1, c1 = _apply_level(n, keys[at], coeffs[at], op.c, op.level(n), D, shells, tau)
        ks.append(k1)
        cs.append(c1)
    return torch.cat(ks), torch.cat(cs)  # keys order by level first


def _apply_batch(op, trees, D, shells, tau):
    """Several functions at once; the results back to back, each in key order."""
    keys, coeffs = torch.cat([t.keys[: t.n] for t in trees]), torch.cat([t.coeffs[: t.n] for t in trees])
    func = torch.cat([torch.full_like(t.keys[: t.n], i) for i, t in enumerate(trees)])
    fs, ks, cs = [], [], []
    lev = keys >> 57
    for n in torch.unique(lev).tolist():
        at = lev == n
        k1, c1 = _apply_level(n, keys[at], coeffs[at], op.c, op.level(n), D, shells, tau, func[at])
        fs.append(k1 >> 57)
        ks.append(_key(torch.full_like(k1, n), *_xyz(k1)))
        cs.append(c1)
    order = torch.sort(torch.cat(fs), stable=True)[1]
    return torch.cat(ks)[order], torch.cat(cs)[order]


def _rows(keys, rows, want, shape):
    """rows of `want` keys, zero where absent."""
    p, hit = _find(keys, want)
    out = torch.zeros((len(want),) + shape, dtype=torch.float64, device="cuda")
    out[hit] = rows[p[hit]]
    return out


def _ns(op, keys, coeffs, n0, D, tau):
    """Non-standard form apply on the leaves of a complete octree."""
    k = op.k
    Ub = _two_scale(k)
    lev = keys >> 57
    top = int(lev.max())
    inner, S, s = {}, {}, {}
    for n in range(top - 1, n0 - 1, -1):
        deep = keys[lev > n]
        inner[n] = torch.unique(_key(n, *[v >> ((deep >> 57) - n) for v in _xyz(deep)]))
        ch = _children(inner[n]).reshape(-1)
        rows = _rows(keys, coeffs, ch, (k, k, k))
        if n + 1 in s:
            rows += _rows(inner[n + 1], s[n + 1], ch, (k, k, k))
        S[n], s[n] = _up(Ub, rows.reshape(-1, 8, k, k, k))
    rk = inner[n0]
    a, b = _apply_level(n0, rk, s[n0], op.c, op.level(n0), 2 ** n0 - 1, True, tau)
    r = _rows(a, b, rk, (k, k, k))
    okeys, orows = [], []
    for n in range(n0, top):
        yk, Y = _apply_level(n, inner[n], S[n], op.c, op.doubled(n, D), D, True, tau)
        zk, Z = _apply_level(n, inner[n], s[n], op.c, op.level(n), D, True, tau)
        x, y, z = _xyz(inner[n])
        halo = []
        for lx in range(-D, D + 1):
            for ly in range(-D, D + 1):
                for lz in range(-D, D + 1):
                    ok = torch.ones_like(x, dtype=torch.bool)
                    for v in (x + lx, y + ly, z + lz):
                        ok &= (v >= 0) & (v < 1 << n)
                    halo.append(_key(n, x + lx, y + ly, z + lz)[ok])
        ref = _find(torch.unique(torch.cat(halo)), rk)[1]
        okeys.append(rk[~ref])
        orows.append(r[~ref])
        p = rk[ref]
        ch = _down(Ub, r[ref] - _rows(zk, Z, p, (k, k, k)))
        Yc = _rows(yk, Y, p, (2 * k,) * 3).reshape(-1, 2, k, 2, k, 2, k).permute(0, 1, 3, 5, 2, 4, 6)
        ck, order = torch.sort(_children(p).reshape(-1))
        rk, r = ck, (ch + Yc.reshape(-1, 8, k, k, k)).reshape(-1, k, k, k)[order]
    return torch.cat(okeys + [rk]), torch.cat(orows + [r])


def _reconstruct(keys, coeffs):
    """Boxes of several levels summed down to disjoint leaves."""
    k = coeffs.shape[1]
    Ub = _two_scale(k)
    lev = keys >> 57
    lo, top = int(lev.min()), int(lev.max())
    covered = torch.zeros_like(keys, dtype=torch.bool)  # an input box lies strictly above
    above, inner = {}, {}
    for n in range(lo, top):
        deep = lev > n
        anc = _key(n, *[v >> (lev[deep] - n) for v in _xyz(keys[deep])])
        covered[deep] |= _find(keys, anc)[1]
        above[n] = (deep, anc)
    for n in range(lo, top):
        # interior boxes: below (or at) an input box and above another
        deep, anc = above[n]
        own = _find(keys, anc)[1]
        for m in range(lo, n):
            own |= _find(keys, _parents(anc, n - m))[1]
        inner[n] = torch.unique(anc[own])
    nk = torch.empty(0, dtype=torch.int64, device="cuda")
    nv = torch.empty((0, k, k, k), dtype=torch.float64, device="cuda")
    okeys, orows = [], []
    for n in range(lo, top + 1):
        at = (lev == n) & ~covered
        rk, order = torch.sort(torch.cat([nk, keys[at]]))
        r = torch.cat([nv, coeffs[at]])[order]
        at = (lev == n) & covered
        r.index_add_(0, _find(rk, keys[at])[0], coeffs[at])
        inn = _find(inner[n], rk)[1] if n < top else torch.zeros_like(rk, dtype=torch.bool)
        okeys.append(rk[~inn])
        orows.append(r[~inn])
        nk, nv = _children(rk[inn]).reshape(-1), _down(Ub, r[inn]).reshape(-1, k, k, k)
    return torch.cat(okeys), torch.cat(orows)


def _truncate(keys, coeffs, thresh):
    k = coeffs.shape[1]
    Ub = _two_scale(k)
    lev = keys >> 57
    out, err2 = [], 0.0
    mk = torch.empty(0, dtype=torch.int64, device="cuda")
    mv = torch.empty((0, k, k, k), dtype=torch.float64, device="cuda")
    for n in range(int(lev.max()), -1, -1):
        rk, order = torch.sort(torch.cat([keys[lev == n], mk]))
        r = torch.cat([coeffs[lev == n], mv])[order]
        mk, mv = mk[:0], mv[:0]
        if n > 0 and len(rk):
            p, count = torch.unique(_parents(rk), return_counts=True)
            p = p[count == 8]
            at = _find(rk, _children(p).reshape(-1))[0]
            ch = r[at].reshape(-1, 8, k, k, k)
            if len(p):
                s = _up(Ub, ch)[1]
                d2 = (ch - _down(Ub, s)).flatten(1).square().sum(1)
                go = d2.sqrt() <= thresh
                err2 += float(d2[go].sum())
                mk, mv = p[go], s[go]
                stay = torch.ones_like(rk, dtype=torch.bool)
                stay[at.reshape(-1, 8)[go].reshape(-1)] = False
                rk, r = rk[stay], r[stay]
        out.append((rk, r))
    return torch.cat([a for a, _ in out[::-1]]), torch.cat([b for _, b in out[::-1]]), err2


def _common(ka, a, kb, b):
    """Two functions' coefficients on their common leaves."""
    u = torch.unique(torch.cat([ka, kb]))
    shape = a.shape[1:]
    keys, ra = _reconstruct(u, _rows(ka, a, u, shape))
    return keys, ra, _reconstruct(u, _rows(kb, b, u, shape))[1]


def _multiply(ka, a, kb, b, L):
    keys, ca, cb = _common(ka, a, kb, b)
    k = a.shape[1]
    x, w = _gl(k)
    V = _phi(k, x)
    VtW = (V * w[:, None]).T.contiguous()

    def modes(A, s):
        s = torch.einsum("ai,nijl->najl", A, s)
        s = torch.einsum("bj,najl->nabl", A, s)
        return torch.einsum("cl,nabl->nabc", A, s)

    h = 2 * L / 2.0 ** (keys >> 57).double()
    return keys, modes(VtW, modes(V, ca) * modes(V, cb)) * (h ** -1.5)[:, None, None, None]


def _inner(ka, a, kb, b):
    if len(ka) == len(kb) and bool((ka == kb).all()):
        return float((a * b).sum())
    _, ca, cb = _common(ka, a, kb, b)
    return float((ca * cb).sum())


def _project_boxes(g, k, L, keys):
    """Exact 1-D integrals of every Gaussian over every box: 32 panels of 20 points over the part of the box
    where the Gaussian is above e^-46 of its maximum there."""
    gx, gw = _gl(20)
    h = 2 * L / 2.0 ** (keys >> 57).double()
    coef, ex = (torch.tensor(g[f], device="cuda") for f in ("coef", "expnt"))
    T = ex[None] * (h * h)[:, None]
    F = []
    for name, b in zip(("cx", "cy", "cz"), _xyz(keys)):
        x = (torch.tensor(g[name], device="cuda")[None] + L) / h[:, None]
        wa = b[:, None].double() - x
        wb = wa + 1.0
        near = torch.maximum(torch.maximum(wa, -wb), torch.zeros_like(wa))
        W = torch.sqrt(near * near + 46.0 / T)
        lo, hi = torch.maximum(wa, -W), torch.minimum(wb, W)
        pw = ((hi - lo) / 32).clamp(min=0.0)
        tot = 0.0
        for p in range(32):
            w = lo[..., None] + pw[..., None] * (p + gx)
            tot = tot + torch.einsum("bgq,bgqi->bgi", pw[..., None] * gw * torch.exp(-T[..., None] * w * w),
                                     _phi(k, w - wa[..., None]))
        F.append(tot)
    return torch.einsum("bg,bgi,bgj,bgl->bijl", coef[None] * (h ** 1.5)[:, None], *F)


def _project(g, k, L, thresh, init_level=2, max_level=19):
    Ub = _two_scale(k)
    nb = 1 << (init_level - 1)
    i = torch.arange(nb ** 3, device="cuda")
    par = _key(torch.full_like(i, init_level - 1), i // (nb * nb), (i // nb) % nb, i % nb)
    out = []
    while len(par):
        ck = _children(par)
        ch = _project_boxes(g, k, L, ck.reshape(-1)).reshape(-1, 8, k, k, k)
        d = (ch - _down(Ub, _project_boxes(g, k, L, par))).flatten(1).norm(dim=1)
        leaf = (d <= thresh) | ((ck[:, 0] >> 57) >= max_level)
        out.append((ck[leaf].reshape(-1), ch[leaf].reshape(-1, k, k, k)))
        par = ck[~leaf].reshape(-1)
    keys, order = torch.sort(torch.cat([a for a, _ in out]))
    return keys, torch.cat([b for _, b in out])[order]


def exact(case, seed):
    kind, k = case["kind"], case["k"]

    def out(keys, coeffs):
        return {"keys": keys, "coeffs": coeffs}

    if kind == "project":
        return out(*_project(_functions(case, seed)[0], k, L_CELL, case["thresh"]))
    if kind == "bsh_step":
        V, psi, E = _bsh_inputs(case, seed)
        v, p = ((t.keys[: t.n], t.coeffs[: t.n]) for t in (V, psi))
        vk, vp = _multiply(*v, *p, 20.0)
        op = _Op("bsh", math.sqrt(-2 * E), case["M"], k, 20.0, 1e-6, 3)
        rk, r = _ns(op, vk, vp, 1, 1, 0.01 * case["thresh"])
        nk, new, _ = _truncate(rk, r * (-1 / (2 * math.pi)), case["thresh"])
        nn = _inner(nk, new, nk, new)
        dE = -(_inner(vk, vp, *p) - _inner(vk, vp, nk, new)) / nn
        return {"E": E + dE, "dE": dE, "psi": out(nk, new / math.sqrt(nn))}
    if kind == "post":
        s = prepare(case, seed)["result"]
        lk, lv = _reconstruct(s.keys[: s.n], s.coeffs[: s.n])
        tk, tv, err2 = _truncate(lk, lv, case["thresh"])
        return {"leaves": out(lk, lv), "truncated": out(tk, tv), "err2": err2}
    trees = _trees(case, seed)
    ns = kind in ("ns_uniform", "ns_tree")
    op = _Op(case["kernel"], case.get("mu", 0.0), case["M"], k, L_CELL, case.get("thresh", 1e-5), 3 if ns else 1)
    if kind == "batched":
        return out(*_apply_batch(op, trees, 1, True, _tau(case)))
    keys, coeffs = trees[0].keys[: trees[0].n], trees[0].coeffs[: trees[0].n]
    return out(*(_ns(op, keys, coeffs, 1, 1, 0.0) if ns else
                 _apply(op, keys, coeffs, 1, "level" not in case, _tau(case))))
