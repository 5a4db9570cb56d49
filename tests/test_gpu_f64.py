"""The FP64 source-stationary apply in parity components (|l|_inf <= 1) against the CPU oracle, over the
orders and shapes where its slices, odd halves and record ranges have edges.

Tolerance: the per-box bar of test_gpu_parity (1e-12 of the larger of the box and the sum of its
terms' bounds): a coefficient is a sum of at most 27 M terms of three k-long products, rounded
to 2^-53 each, so its error is below (27 * 64 + 3 * 20) 2^-53 < 2e-13 of that sum.
"""
import numpy as np
import pytest

import oracle as O
import workloads as W
from oracle_inputs import oracle_fit
from test_gpu_parity import fp64_box_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mra():
    import torch
    assert torch.cuda.is_available()
    from paper_1507_01888_gb300 import mra as m
    m.load()
    return m


@pytest.mark.parametrize("k,n_boxes", [(1, 64), (2, 30), (3, 1), (5, 200), (7, 64), (9, 40), (11, 20), (12, 30), (13, 9),
                                       (14, 300), (15, 5), (16, 40)])
@pytest.mark.parametrize("screened", [False, True])
def test_orders_and_sizes_match_oracle(mra, k, n_boxes, screened):
    keys, coeffs = W.random_tree_coeffs(n_boxes, k, 3, seed=31 * k + n_boxes)
    op = mra.Operator(1, 12, k, 32.0, 3, 3, max_disp=1, mu=0.7, fit_eps=1e-4)
    f = oracle_fit(op)
    tau = 1e-2 if screened else 0.0
    opts = mra.make_opts(stencil=mra.STENCIL_SHELLS, max_disp=1, screen=mra.SCREEN_NORM if screened else mra.SCREEN_NONE,
                         tau=tau)
    ref = O.apply(keys, coeffs, f["c"], f["t"], 32.0, stencil=0, max_disp=1, tau=tau)
    out, st = mra.apply(op, mra.Tree.from_host(keys, coeffs, 32.0), opts)
    fp64_box_check(*out.host(), ref)
    assert st["terms_kept"] == ref.terms


def test_ranges_of_records_equal_one_range(mra):
    """More partial sums than one range of the scratch holds (6.8 GB against 4): bit for bit the result of
    destination partitions, each of which fits one range."""
    import torch
    keys, coeffs = W.random_tree_coeffs(8192, 16, 5, seed=3)
    op = mra.Operator(0, 2, 16, 32.0, 5, 5, max_disp=1, fit_eps=1e-4)
    tree = mra.Tree.from_host(keys, coeffs, 32.0)
    whole, st = mra.apply(op, tree, mra.make_opts())
    assert st["pairs"] * 16 ** 3 * 8 > 4 << 30
    ks = whole.keys[: whole.n].cpu().numpy().view("uint64")
    cuts = [0, int(ks[len(ks) // 3]), int(ks[2 * len(ks) // 3]), 1 << 63]
    parts = []
    for lo, hi in zip(cuts, cuts[1:]):
        p, _ = mra.apply(op, tree, mra.make_opts(dest_range=(lo, hi)))
        parts.append((p.keys[: p.n].clone(), p.coeffs[: p.n].clone()))
    assert torch.equal(torch.cat([p[0] for p in parts]), whole.keys[: whole.n])
    assert torch.equal(torch.cat([p[1] for p in parts]), whole.coeffs[: whole.n])


@pytest.mark.parametrize("k", [4, 5])
def test_term_kept_for_one_sign_only(mra, k):
    """The two blocks of +-1 can differ in the last bit of their norms; with the threshold between the two
    bounds the screen keeps a term for one displacement and not for its mirror image."""
    op = mra.Operator(0, 60, k, 32.0, 2, 6, max_disp=1, fit_eps=1e-6)
    f = op.fit()
    rng = np.random.default_rng(k)
    done = 0
    for level in range(2, 7):
        s = rng.standard_normal((k, k, k))
        key = W.random_tree_coeffs(1, k, level, 0)[0][:1].copy()
        key[0] = (np.uint64(level) << np.uint64(57)) | (np.uint64(1) << np.uint64(38)) | \
            (np.uint64(1) << np.uint64(19)) | np.uint64(1)
        tree = mra.Tree.from_host(key, s[None], 32.0)
        sn = float(mra.norm(tree)[0][0])
        for m in range(60):
            N = {l: op.block(level, m, l)[1] for l in (-1, 0, 1)}
            bound = {l: abs(f["c"][m]) * N[l] * N[0] * N[0] * sn for l in (-1, 0, 1)}
            if bound[1] == bound[-1] or bound[0] < max(bound[1], bound[-1]):
                continue
            out, st = mra.apply(op, tree, mra.make_opts(stencil=mra.STENCIL_SHELLS, max_disp=1, screen=mra.SCREEN_NORM,
                                                        tau=max(bound[1], bound[-1])))
            gk, gc = out.host()
            fit = oracle_fit(op)
            ref = O.apply(key, s[None], fit["c"], fit["t"], 32.0, stencil=0, max_disp=1, tau=0.0)
            assert set(gk.tolist()) <= set(ref.keys.tolist())
            # the reference result from the blocks themselves, term by term, with the library's decisions
            want = {}
            n_terms = 0
            for l in np.ndindex(3, 3, 3):
                l = tuple(v - 1 for v in l)
                for q in range(60):
                    R = {v: op.block(level, q, v) for v in set(l)}
                    B = abs(f["c"][q]) * R[l[0]][1] * R[l[1]][1] * R[l[2]][1] * sn
                    if not B >= max(bound[1], bound[-1]):
                        continue
                    n_terms += 1
                    d = int(key[0]) + (l[0] << 38) + (l[1] << 19) + l[2]
                    v = f["c"][q] * np.einsum("ai,bj,cl,ijl->abc", R[l[0]][0], R[l[1]][0], R[l[2]][0], s)
                    want.setdefault(d, [np.zeros_like(s), 0.0])
                    want[d][0] += v
                    want[d][1] += B
            assert st["terms_kept"] == n_terms
            assert sorted(want) == [int(v) for v in gk]
            for d, got in zip(gk, gc):
                r, scale = want[int(d)]
                assert np.linalg.norm(got - r) <= 1e-12 * max(np.linalg.norm(r), scale)
            done += 1
            break
        if done == 2:
            break
    if done == 0:
        pytest.skip("every pair of blocks has equal norms here")


@pytest.mark.parametrize("k,n_boxes", [(6, 200), (9, 60)])
def test_without_room_for_partial_sums(mra, k, n_boxes):
    """The apply and a recorded one give the result when not even the smallest partial buffer is to be had, and a
    batch of functions gives each function's."""
    import torch
    keys, coeffs = W.random_tree_coeffs(n_boxes, k, 3, seed=k)
    op = mra.Operator(1, 12, k, 32.0, 3, 3, max_disp=1, mu=0.7, fit_eps=1e-4)
    f = oracle_fit(op)
    ref = O.apply(keys, coeffs, f["c"], f["t"], 32.0, stencil=0, max_disp=1, tau=1e-2)
    o = mra.make_opts(stencil=mra.STENCIL_SHELLS, max_disp=1, screen=mra.SCREEN_NORM, tau=1e-2)
    tree = mra.Tree.from_host(keys, coeffs, 32.0)
    cat, offs = mra.concat_trees([tree, tree])
    free, _ = mra.apply(op, tree, o)
    mra.debug_limit_memory(1 << 19)  # bytes; the partial sums take more than 1 MB
    try:
        out, st = mra.apply(op, tree, o)
        assert st["pairs"] * k ** 3 * 8 > 1 << 20
        g = mra.ApplyGraph(op, tree, o)
        g.out.coeffs.zero_()
        g.launch()
        g.status()
        both, _ = mra.BatchedApplier(op, cat, offs, o)(cat)
    finally:
        mra.debug_limit_memory(0)
    fp64_box_check(*free.host(), ref)
    fp64_box_check(*out.host(), ref)
    n = out.n
    assert g.out.n == n and torch.equal(g.out.coeffs[:n], out.coeffs[:n])
    assert both.n == 2 * n and all(torch.equal(both.coeffs[i * n: (i + 1) * n], out.coeffs[:n]) for i in (0, 1))


def test_ranges_of_records_in_the_doubled_basis(mra):
    """The non-standard operator's apply in several ranges of records, where the sums are turned back into the
    children's coefficients after the last one only: bit for bit the result of one range."""
    import torch
    k, level = 12, 3
    keys, coeffs = W.random_tree_coeffs(400, k, level, seed=12)
    base = mra.Operator(0, 3, k // 2, 32.0, level, level + 1, max_disp=3, fit_eps=1e-4)
    op = mra.NSOperator(base, max_disp=1)
    tree = mra.Tree.from_host(keys, coeffs, 32.0)
    whole, st = mra.apply(op, tree, mra.make_opts())
    total = st["pairs"] * k ** 3 * 8
    assert 65 << 20 < total < 4 << 30
    mra.debug_limit_memory(65 << 20)  # the smallest partial buffer (64 MB) fits; below that the gather would run
    try:
        parts, _ = mra.apply(op, tree, mra.make_opts())
    finally:
        mra.debug_limit_memory(0)
    assert parts.n == whole.n and torch.equal(parts.keys[: parts.n], whole.keys[: whole.n])
    assert torch.equal(parts.coeffs[: parts.n], whole.coeffs[: whole.n])


@pytest.mark.parametrize("k", [2, 3])
def test_term_kept_for_one_sign_only_in_the_doubled_basis(mra, k):
    """As test_term_kept_for_one_sign_only, with the non-standard operator's blocks."""
    lo, hi = 1, 6
    op = mra.NSOperator(mra.Operator(0, 20, k, 32.0, lo, hi + 1, max_disp=3, fit_eps=1e-4), max_disp=1)
    c, kk = op.base.fit()["c"], 2 * k
    s = np.random.default_rng(k).standard_normal((kk, kk, kk))
    done = 0
    for level in range(lo + 1, hi + 1):
        key = np.array([(level << 57) | (1 << 38) | (1 << 19) | 1], dtype=np.uint64)
        tree = mra.Tree.from_host(key, s[None], 32.0)
        sn = float(mra.norm(tree)[0][0])
        R = [{l: op.block(level, m, l) for l in (-1, 0, 1)} for m in range(20)]
        for m in range(20):
            up, down, mid = (abs(c[m]) * R[m][l][1] * R[m][0][1] * R[m][0][1] * sn for l in (1, -1, 0))
            tau = max(up, down)
            if up == down or mid < tau:
                continue
            out, st = mra.apply(op, tree, mra.make_opts(stencil=mra.STENCIL_SHELLS, max_disp=1, screen=mra.SCREEN_NORM, tau=tau))
            want, n_terms, lone = {}, 0, 0
            for l in np.ndindex(3, 3, 3):
                l = tuple(v - 1 for v in l)
                for q in range(20):
                    def bound(*d):
                        return abs(c[q]) * R[q][d[0]][1] * R[q][d[1]][1] * R[q][d[2]][1] * sn
                    if not bound(*l) >= tau:
                        continue
                    n_terms += 1
                    lone += not bound(-l[0], l[1], l[2]) >= tau
                    d = int(key[0]) + (l[0] << 38) + (l[1] << 19) + l[2]
                    r = want.setdefault(d, [np.zeros_like(s), 0.0])
                    r[0] += c[q] * np.einsum("ai,bj,cl,ijl->abc", R[q][l[0]][0], R[q][l[1]][0], R[q][l[2]][0], s)
                    r[1] += bound(*l)
            assert lone > 0 and st["terms_kept"] == n_terms
            gk, gc = out.host()
            assert sorted(want) == [int(v) for v in gk]
            for d, got in zip(gk, gc):
                r, scale = want[int(d)]
                assert np.linalg.norm(got - r) <= 1e-12 * max(np.linalg.norm(r), scale)
            done += 1
            break
    assert done > 0, "no pair of blocks with unequal norms"
