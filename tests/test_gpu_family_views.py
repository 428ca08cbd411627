"""All views of a family's relation through one first phase (batches of 2^21 tuples and more):
every sub-query's sketches equal to the per-tuple view update's, bit for bit."""
import itertools

import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,logm,d,n,window,subs", [
    (4, 16, 9, (1 << 21) + 5, 0, "all"), (2, 13, 9, (1 << 21), 0, "all"), (5, 16, 4, 2_500_001, 900_000, "all"),
    (3, 16, 7, 2_200_003, 0, "some"), (1, 16, 9, (1 << 21) + 31, 0, "all")])
def test_equals_per_tuple_views(k, logm, d, n, window, subs, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(k)
    dom = [2003 + 1009 * u for u in range(k)]
    cols = torch.stack([torch.randint(0, x, (n,), generator=g, device="cuda") for x in dom])
    cols[:, ::3] = 5                       # a heavy bin in every view
    cols[k - 1, 77::60013] = dom[k - 1]    # outside one attribute's domain: left out of every view
    cols[0, 99::70001] = -1
    queries = [list(c) for r in range(1, k + 1) for c in itertools.combinations(range(k), r)]
    if subs == "some":
        queries = queries[2:5]
    if window:
        monkeypatch.setenv("SK_PART_WINDOW", str(window))
    got = []
    for part in ("1", "0"):
        monkeypatch.setenv("SK_PART_UPDATE", part)
        f = sk.SketchFamily([k] + [1] * k, [(0, u, 1 + u, 0) for u in range(k)], queries, 1 << logm, d, 5)
        f.update(0, cols, domain=dom)
        with pytest.raises(sk.SketchError):
            f.sync()
        got.append([f.sketch(i, 0) for i in range(len(queries))])
        f.close()
    assert all((x == y).all() for x, y in zip(*got))


@pytest.mark.parametrize("k,logm,d,n,window", [
    (3, 15, 9, 3 << 19, 0), (2, 16, 1, (3 << 19) + 1, 0), (4, 16, 8, 1_600_001, 8193), (5, 14, 9, 1_599_999, 500_000)])
def test_tile_edges(k, logm, d, n, window, monkeypatch):
    """One part and two, one row, 45 planes, windows that end inside a tile of 8192 tuples."""
    test_equals_per_tuple_views(k, logm, d, n, window, "all", monkeypatch)
