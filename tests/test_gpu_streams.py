"""Calls on a stream that is not torch's current one: what they return is complete for every stream."""
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


@pytest.mark.parametrize("busy", ["current", "side"])
def test_projected_tree_is_complete_on_another_stream(mra, busy):
    """The tree that project returns is read at once on the other stream while the stream that ran the projection, or
    torch's current one, has a long kernel queued before the call."""
    import torch
    f = W.gaussian_sum(2, 1.0, 50.0, seed=5, centre_box=5.0)
    ref = mra.project(f, 6, 16.0, thresh=1e-4)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    if busy == "current":
        torch.cuda._sleep(400_000_000)  # about 0.2 s of SM clock
        got, reader = mra.project(f, 6, 16.0, thresh=1e-4, stream=side), side
    else:
        with torch.cuda.stream(side):
            torch.cuda._sleep(400_000_000)
            got, reader = mra.project(f, 6, 16.0, thresh=1e-4), torch.cuda.default_stream()
    with torch.cuda.stream(reader):
        keys, coeffs = got.keys[: got.n].clone(), got.coeffs[: got.n].clone()
    torch.cuda.synchronize()
    assert got.n == ref.n
    assert torch.equal(keys, ref.keys[: ref.n]) and torch.equal(coeffs, ref.coeffs[: ref.n])
