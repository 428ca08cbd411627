"""A family's relation takes the planes of all its views, or one view at a time, as its views and its
batch make the cheaper; either way with the same sketches."""
import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,n,subs,planes", [
    (5, 20_000_000, [[0, 1], [0, 1, 2, 3, 4]], False), (4, 50_000_000, [[0], [1, 2]], False),
    (5, 8_000_000, [[0], [1]], True), (5, 20_000_000, [[0], [1], [0, 1]], True), (2, 20_000_000, [[0], [0, 1]], True)])
def test_choice(k, n, subs, planes, monkeypatch):
    """Two views of many attributes gather and write for all of them: one view at a time is up to 1.2
    times as fast for long batches.  The launches tell: a table, then two kernels for all views, or a
    validity pass and two kernels per view."""
    g = torch.Generator(device="cuda").manual_seed(k)
    dom = [50_000] * k
    cols = torch.randint(0, 50_000, (k, n), generator=g, device="cuda")
    got = []
    for part in ("1", "0"):
        monkeypatch.setenv("SK_PART_UPDATE", part)
        f = sk.SketchFamily([k] + [1] * k, [(0, u, 1 + u, 0) for u in range(k)], subs, 1 << 16, 9, 5)
        launches = sk.sk_launch_count()
        f.update(0, cols, domain=dom)
        launches = sk.sk_launch_count() - launches
        if part == "1":
            assert launches == (3 if planes else 2 + 2 * len(subs))
        got.append([f.sketch(i, 0) for i in range(len(subs))])
        f.close()
    assert all((x == y).all() for x, y in zip(*got))
