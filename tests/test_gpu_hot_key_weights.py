"""Weights of a one-attribute relation's equal keys, added before the keys are hashed: sums at
the limits of int64, and no dearer than unit weights of the same keys."""
import pytest
import torch

import paper_2402_15953_gb300 as sk
from _timing import best_times

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [1, 1 << 31, 1 << 32, (1 << 63) - 1])
@pytest.mark.parametrize("keys", [1, 3, 20_000])
def test_sums_wrap(top, keys):
    """All lanes alike, a few groups, mostly single lanes: the sketch of the batch equals the sum of
    the sketches of its tuples taken apart (one per warp), modulo 2^64."""
    g = torch.Generator(device="cuda").manual_seed(keys)
    n = 3001
    k = torch.randint(0, keys, (1, n), generator=g, device="cuda") * 3_000_000_019
    w = torch.randint(-top, top, (n,), generator=g, device="cuda")
    w[::7] = -(1 << 63)
    w[3::7] = 0
    spaced = torch.zeros(n * 32, dtype=torch.int64, device="cuda")
    spaced[::32] = w
    other = torch.arange(n * 32, device="cuda").view(1, -1) + (1 << 40)
    other[0, ::32] = k[0]   # the filler keys have weight 0
    got = []
    for cols, weights in ((k, w), (other, spaced)):
        s = sk.SketchSet([1, 1], [(0, 0, 1, 0)], 1 << 16, 5, 3)
        s.update(0, cols, weights)
        got.append(s.counters.clone())
        s.close()
    assert torch.equal(*got)


@pytest.mark.parametrize("top,distinct,took", [(1, True, 1.43), (1 << 40, False, 2.06)])
def test_no_dearer_than_unit_weights(top, distinct, took):
    """Weights add eight bytes to a tuple's eight and, with equal keys in a warp, a ballot per bit of
    the largest (merging by a reduction per group took `took` times the unit-weight update for distinct
    keys, and so did weights beyond 2^25, which were not merged): less than half of the excess is left."""
    g = torch.Generator(device="cuda").manual_seed(1)
    n, m, d = 4_000_000, 1_000_000, 5
    if distinct:
        keys = torch.randint(0, 1 << 60, (1, n), generator=g, device="cuda")
    else:
        keys = (torch.rand((1, n), generator=g, device="cuda", dtype=torch.float64) ** 6 * 1_000_000).long()
    w = torch.randint(1, top + 1, (n,), generator=g, device="cuda")
    s = sk.SketchSet([1, 1], [(0, 0, 1, 0)], m, d, 3)
    with_w, unit = best_times([lambda: s.update(0, keys, w), lambda: s.update(0, keys)])
    s.close()
    assert with_w <= (1 + took) / 2 * unit, (with_w, unit)
