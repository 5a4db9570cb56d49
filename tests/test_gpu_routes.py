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
