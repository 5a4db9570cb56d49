"""Projection from shared 1-D factors against the CPU oracle: several batches of staged Gaussians, the
orders at the ends of the range, odd orders and exponents whose Gaussians vanish on most boxes.

Tolerance: the bar of test_gpu_parity's projection tests (1e-12 of the box's norm, or of 1e-6 of the whole
norm for boxes that hold almost nothing).
"""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mra():
    import torch
    assert torch.cuda.is_available()
    from paper_1507_01888_gb300 import mra as m
    m.load()
    return m


def check(got, ok, oc):
    keys, coeffs = got.host()
    assert (keys == ok).all()
    d = np.sqrt(((coeffs - oc) ** 2).reshape(len(ok), -1).sum(1))
    n = np.sqrt((oc ** 2).reshape(len(ok), -1).sum(1))
    assert np.all(d <= 1e-12 * np.maximum(n, 1e-6 * np.sqrt((oc ** 2).sum())))


@pytest.mark.parametrize("k,ng,a_hi,thresh", [(2, 3, 20.0, 1e-1), (3, 40, 50.0, 3e-2), (5, 16, 1e3, 1e-3), (7, 17, 1e4, 1e-4),
                                              (11, 33, 1e3, 1e-5), (16, 2, 1e6, 1e-8)])
def test_adaptive_orders_and_counts(mra, k, ng, a_hi, thresh):
    f = W.gaussian_sum(ng, 0.5, a_hi, seed=k + ng)
    ok, oc, margin = O.project(f, k, 32.0, thresh=thresh, init_level=2, max_level=14)
    assert margin > 1e-8, "refinement decision too close to the threshold for a unique tree"
    check(mra.project(f, k, 32.0, thresh=thresh, init_level=2, max_level=14), ok, oc)


@pytest.mark.parametrize("k,ng,level", [(1, 5, 2), (4, 1, 0), (9, 100, 1), (13, 20, 2), (16, 3, 3)])
def test_uniform_orders_and_counts(mra, k, ng, level):
    f = W.gaussian_sum(ng, 0.01, 1e3, seed=k * ng)
    ok, oc, _ = O.project(f, k, 32.0, uniform_level=level)
    check(mra.project(f, k, 32.0, uniform_level=level), ok, oc)


def test_no_gaussians(mra):
    f = {name: np.zeros(0) for name in ("coef", "expnt", "cx", "cy", "cz")}
    t = mra.project(f, 4, 32.0, uniform_level=1)
    assert t.n == 8 and float(t.coeffs[:8].abs().max()) == 0.0
    assert mra.project(f, 4, 32.0, thresh=1e-3).n == 64


@pytest.mark.parametrize("k,level", [(6, 2), (8, 1), (10, 2), (12, 1), (14, 2)])
@pytest.mark.parametrize("a_lo,a_hi", [(1e-4, 1e-1), (1e-1, 1e3), (1e3, 1e7)])
def test_flat_to_narrow_gaussians(mra, k, level, a_lo, a_hi):
    """From one panel for the whole box to panels of a small part of it, and each split of a box over the threads."""
    f = W.gaussian_sum(6, a_lo, a_hi, seed=k)
    ok, oc, _ = O.project(f, k, 32.0, uniform_level=level)
    check(mra.project(f, k, 32.0, uniform_level=level), ok, oc)


def _mixed(ng, real, a_lo, a_hi, seed):
    """`real` Gaussians spread over ng, the others with coefficient zero: the tables have room for all, the sums are those
    of the real ones."""
    f, rng = W.gaussian_sum(real, a_lo, a_hi, seed=seed, centre_box=31.0), np.random.default_rng(seed)
    at = np.sort(rng.choice(ng, real, replace=False))
    full = {"coef": np.zeros(ng), "expnt": np.full(ng, 1e3), "cx": np.zeros(ng), "cy": np.zeros(ng), "cz": np.zeros(ng)}
    for name in full:
        full[name][at] = f[name]
    return f, full


def test_many_gaussians_in_bounded_tables(mra):
    """Factor tables of all parents of a level would take over 1 GB: the parents are taken in parts, in 256 MB of tables, and
    the tree is that of the Gaussians that count."""
    import torch
    f, full = _mixed(4000, 800, 1e6, 1e7, 3)
    few = mra.project(f, 2, 32.0, thresh=1e-2, max_level=13)
    torch.cuda.synchronize()
    mra.release_memory()
    free0 = torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved()
    many = mra.project(full, 2, 32.0, thresh=1e-2, max_level=13)
    used = free0 - (torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved())
    keys = many.keys[: many.n].cpu().numpy().view("uint64")
    lv = (keys >> np.uint64(57)).astype(int)
    coords = max(sum(len(np.unique((keys[lv == n] >> np.uint64(s)) & np.uint64(0x7ffff) >> np.uint64(1)))
                     for s in (38, 19, 0)) for n in np.unique(lv))
    assert coords * 4000 * (40 * 2 + 3) > 1 << 30
    assert used < 800 << 20, f"{used >> 20} MB"
    assert many.n == few.n and torch.equal(many.keys[: many.n], few.keys[: few.n])
    assert torch.equal(many.coeffs[: many.n], few.coeffs[: few.n])


def test_short_memory_takes_smaller_batches(mra):
    """With little memory for the tables the parents of a level, or the Gaussians of a uniform level, are taken in
    smaller parts: the same sums."""
    import torch
    f, full = _mixed(500, 30, 1e3, 1e5, 9)
    whole = mra.project(full, 2, 32.0, thresh=1e-2, max_level=9)
    g = W.gaussian_sum(60, 0.1, 1e3, seed=4)
    level = mra.project(g, 5, 32.0, uniform_level=3)
    assert whole.n * 64 * 2 < 3 << 20
    mra.debug_limit_memory(3 << 20)
    try:
        parts = mra.project(full, 2, 32.0, thresh=1e-2, max_level=9)
        mra.debug_limit_memory(16 << 10)
        batches = mra.project(g, 5, 32.0, uniform_level=3)
    finally:
        mra.debug_limit_memory(0)
    for a, b in ((whole, parts), (level, batches)):
        assert a.n == b.n and torch.equal(a.keys[: a.n], b.keys[: b.n]) and torch.equal(a.coeffs[: a.n], b.coeffs[: b.n])
