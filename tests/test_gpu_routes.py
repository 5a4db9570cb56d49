"""Shapes and launch forms that are chosen by rules on the order give the sums of the general form."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mra():
    import torch
    assert torch.cuda.is_available()
    from paper_1507_01888_gb300 import mra as m
    m.load()
    return m


@pytest.mark.parametrize("k", [12, 14, 16])
@pytest.mark.parametrize("n_boxes", [1, 7, 90])
def test_split_wide_shape_is_independent_of_its_neighbours(mra, k, n_boxes):
    """tile_variant 0 from k = 12 on: a destination's result does not depend on the destinations beside it
    (every term is flushed alone), and it lies within the split error of the joined shape."""
    import torch
    keys, coeffs = W.random_tree_coeffs(n_boxes, k, 3, seed=k + n_boxes)
    op = mra.Operator(0, 6, k, 32.0, 3, 3, max_disp=1, fit_eps=1e-4)
    tree = mra.Tree.from_host(keys, coeffs, 32.0)
    kw = dict(precision=mra.PREC_SPLIT_BF16, stencil=mra.STENCIL_NEAREST)
    whole, _ = mra.apply(op, tree, mra.make_opts(**kw))
    ks = whole.keys[: whole.n].cpu().numpy().view("uint64")
    cut = int(ks[whole.n // 2 + 1])
    parts = [mra.apply(op, tree, mra.make_opts(dest_range=r, **kw))[0] for r in ((0, cut), (cut, 1 << 63))]
    assert torch.equal(torch.cat([p.coeffs[: p.n] for p in parts]), whole.coeffs[: whole.n])
    joined, _ = mra.apply(op, tree, mra.make_opts(tile_variant=1, **kw))
    assert mra.compare(joined, whole)["rel_l2"] <= 4e-7
    exact, _ = mra.apply(op, tree, mra.make_opts(stencil=mra.STENCIL_NEAREST))
    assert mra.compare(whole, exact)["rel_l2"] <= 2e-7


@pytest.mark.parametrize("k", [4, 6, 8, 10])
def test_split_parts_of_a_tile_equal_whole_tiles(mra, k):
    """With few tiles the source-stationary kernel gives a tile's groups to several CTAs; many copies of the
    same function in one batch run whole tiles, and each copy has the single function's result bit for bit."""
    import torch
    keys, coeffs = W.random_tree_coeffs(20, k, 3, seed=k)
    op = mra.Operator(0, 3, k, 32.0, 3, 3, max_disp=1, fit_eps=1e-4)
    tree = mra.Tree.from_host(keys, coeffs, 32.0)
    o = mra.make_opts(precision=mra.PREC_SPLIT_BF16, stencil=mra.STENCIL_NEAREST)
    single, st = mra.apply(op, tree, o)
    copies = 8 * 304 * {4: 8, 6: 3, 8: 2, 10: 1}[k] // 20 + 40
    cat, offs = mra.concat_trees([tree] * copies)
    out, out_offs = mra.BatchedApplier(op, cat, offs, o)(cat)
    assert out.n == copies * single.n
    want = single.coeffs[: single.n]
    assert bool((out.coeffs[: out.n].reshape(copies, *want.shape) == want).all())
    assert torch.equal(out.keys[: single.n], single.keys[: single.n])


@pytest.mark.parametrize("k", [4, 6, 8, 10])
def test_split_three_parts_of_a_tile_equal_nine(mra, k):
    """Between one and eight tiles for every CTA slot a tile's groups go to three CTAs: each copy of a batch of that
    size has the single function's result (nine CTAs a tile) bit for bit."""
    import torch
    keys, coeffs = W.random_tree_coeffs(20, k, 3, seed=k)
    op = mra.Operator(0, 3, k, 32.0, 3, 3, max_disp=1, fit_eps=1e-4)
    tree = mra.Tree.from_host(keys, coeffs, 32.0)
    o = mra.make_opts(precision=mra.PREC_SPLIT_BF16, stencil=mra.STENCIL_NEAREST)
    single, _ = mra.apply(op, tree, o)
    slots, G = 2 * torch.cuda.get_device_properties(0).multi_processor_count, {4: 8, 6: 3, 8: 2, 10: 1}[k]
    copies = 2 * slots * G // 20 + 1
    assert slots <= 20 * copies // G and 20 * copies // G + 20 < 8 * slots
    cat, offs = mra.concat_trees([tree] * copies)
    out, _ = mra.BatchedApplier(op, cat, offs, o)(cat)
    want = single.coeffs[: single.n]
    assert out.n == copies * single.n
    assert bool((out.coeffs[: out.n].reshape(copies, *want.shape) == want).all())


def test_truncate_into_its_own_buffers(mra):
    """mra_truncate with the result in the input's buffers, and with too little room (which leaves them as they are)."""
    import ctypes
    f = W.gaussian_sum(2, 1.0, 50.0, seed=5, centre_box=5.0)
    t = mra.project(f, 5, 16.0, thresh=1e-6)
    ref, err2 = mra.truncate(t, 1e-3)
    assert ref.n < t.n
    keys, coeffs = t.keys.clone(), t.coeffs.clone()
    vin, vout, e2 = t.view(), t.view(), ctypes.c_double()
    vout.cap = ref.n - 1
    assert mra.load().mra_truncate(ctypes.byref(vin), 1e-3, ctypes.byref(vout), ctypes.byref(e2),
                                   mra._stream(None)) == mra.MRA_ERR_CAPACITY
    assert vout.n == ref.n and bool((t.keys == keys).all()) and bool((t.coeffs == coeffs).all())
    vout = t.view()
    assert mra.load().mra_truncate(ctypes.byref(vin), 1e-3, ctypes.byref(vout), ctypes.byref(e2), mra._stream(None)) == 0
    assert vout.n == ref.n and e2.value == err2
    assert bool((t.keys[: ref.n] == ref.keys[: ref.n]).all()) and bool((t.coeffs[: ref.n] == ref.coeffs[: ref.n]).all())


@pytest.mark.parametrize("k", [3, 10])
def test_fp64_graph_replay_equals_plain_apply(mra, k):
    import torch
    keys, coeffs = W.random_tree_coeffs(60, k, 3, seed=k)
    op = mra.Operator(0, 5, k, 32.0, 3, 3, max_disp=1, fit_eps=1e-4)
    tree = mra.Tree.from_host(keys, coeffs, 32.0)
    o = mra.make_opts()
    plain, _ = mra.apply(op, tree, o)
    g = mra.ApplyGraph(op, tree, o)
    for scale in (1.0, -0.5):
        tree.coeffs.mul_(scale)
        got = g.launch()
        g.status()
        want, _ = mra.apply(op, tree, o)
        assert torch.equal(got.coeffs[: got.n], want.coeffs[: want.n])
        assert torch.equal(got.keys[: got.n], plain.keys[: plain.n])


def _leaves(rng, k, depth, keep):
    """Random disjoint boxes of levels 1 to `depth` (a box is divided, kept with probability `keep`, or left out)."""
    def key(n, x, y, z):
        return (n << 57) | (x << 38) | (y << 19) | z
    todo, out = [(1, x, y, z) for x in (0, 1) for y in (0, 1) for z in (0, 1)], []
    while todo:
        n, x, y, z = todo.pop()
        if n < depth and rng.random() < 0.3:
            todo += [(n + 1, 2 * x + i, 2 * y + j, 2 * z + m) for i in (0, 1) for j in (0, 1) for m in (0, 1)]
        elif rng.random() < keep:
            out.append(key(n, x, y, z))
    keys = np.array(sorted(out) or [key(1, 0, 1, 0)], dtype=np.uint64)
    return keys, rng.standard_normal((len(keys), k, k, k))


@pytest.mark.parametrize("k", [1, 5, 10])
@pytest.mark.parametrize("form", ["any", "second finer", "first finer", "apart", "nested"])
def test_products_use_the_sums_of_each_tree_by_itself(mra, k, form):
    """Product and inner product on the common leaves, against each tree with zero boxes at the other's keys summed
    down by itself: leaves at different levels on either side, one tree at or below the other's leaves, trees
    without a common box, and a tree with boxes below one another."""
    import torch
    rng = np.random.default_rng(7 * k + len(form))
    (ka, ca), (kb, cb) = _leaves(rng, k, 4, 0.8), _leaves(rng, k, 5, 0.7)
    if form in ("second finer", "first finer"):
        t = mra.reconstruct(mra.Tree.from_host(*_union(ka, ca, kb, cb), 8.0))
        kb = t.keys[: t.n].cpu().numpy().view("uint64")
        cb = rng.standard_normal((t.n, k, k, k))
        if form == "first finer":
            (ka, ca), (kb, cb) = (kb, cb), (ka, ca)
    elif form == "apart":
        left = (ka >> np.uint64(38)) & np.uint64(0x7ffff) < (np.uint64(1) << ((ka >> np.uint64(57)) - np.uint64(1)))
        right = (kb >> np.uint64(38)) & np.uint64(0x7ffff) >= (np.uint64(1) << ((kb >> np.uint64(57)) - np.uint64(1)))
        ka, ca, kb, cb = ka[left], ca[left], kb[right], cb[right]
        assert len(ka) and len(kb)
    elif form == "nested":
        ka, ca = _union(ka, ca, *_leaves(rng, k, 4, 0.8))
    ta, tb = mra.Tree.from_host(ka, ca, 8.0), mra.Tree.from_host(kb, cb, 8.0)
    sa = mra.reconstruct(mra.Tree.from_host(*_union(ka, ca, kb, 0 * cb), 8.0))
    sb = mra.reconstruct(mra.Tree.from_host(*_union(kb, cb, ka, 0 * ca), 8.0))
    assert torch.equal(sa.keys[: sa.n], sb.keys[: sb.n])
    got, want = mra.multiply(ta, tb), mra.multiply(sa, sb)
    assert torch.equal(got.keys[: got.n], want.keys[: want.n])
    assert torch.equal(got.coeffs[: got.n], want.coeffs[: want.n])
    assert mra.inner(ta, tb) == mra.inner(sa, sb)
    if len(ka) > 1:
        wrong = mra.Tree.from_host(ka[::-1].copy(), ca, 8.0)
        for pair in ((wrong, tb), (tb, wrong)):
            with pytest.raises(mra.MraError):
                mra.inner(*pair)


def _union(ka, ca, kb, cb):
    """Boxes of both, coefficients added where both have the box."""
    keys = np.union1d(ka, kb)
    c = np.zeros((len(keys),) + ca.shape[1:])
    c[np.searchsorted(keys, ka)] += ca
    c[np.searchsorted(keys, kb)] += cb
    return keys, c
