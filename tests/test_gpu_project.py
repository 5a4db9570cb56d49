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
