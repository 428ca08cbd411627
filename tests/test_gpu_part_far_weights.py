"""Weighted batches through the two-phase update when weights exceed what an item holds: tiles of
few and of only such weights, batches just below and above the share that sends every tuple to the
counters, and what such a batch costs."""
import pytest
import torch

import paper_2402_15953_gb300 as sk
from _timing import best_times

pytestmark = pytest.mark.gpu


def _set(a, m, d):
    return sk.SketchSet([a] + [1] * a, [(0, k, 1 + k, 0) for k in range(a)], m, d, 3)


@pytest.mark.parametrize("far", [0, 1, 22, 23, 32])
@pytest.mark.parametrize("a,logm,d,n,window,record", [
    (5, 16, 9, 1_048_613, 0, "24"), (2, 13, 7, 131_107, 0, "24"), (1, 13, 9, 140_033, 33_000, "24"),
    (3, 16, 9, 1_048_577, 400_000, "32"), (2, 14, 14, 262_145, 0, "24"), (4, 15, 11, 8_000_001, 0, "24")])
def test_equals_single_phase(far, a, logm, d, n, window, record, monkeypatch):
    """`far` of each 32 consecutive tuples beyond any item, some keys outside their domains; claims of
    32 to 512 tuples, windows that claim anew."""
    g = torch.Generator(device="cuda").manual_seed(far)
    dom = [3001 + 977 * u for u in range(a)]
    cols = torch.stack([torch.randint(0, x, (n,), generator=g, device="cuda") for x in dom])
    cols[a - 1, 17::911] = -1
    w = torch.randint(-9, 10, (n,), generator=g, device="cuda")
    w[torch.arange(n, device="cuda") % 32 < far] = (1 << 45) + 3
    monkeypatch.setenv("SK_KEY_TABLE", "1")
    monkeypatch.setenv("SK_PART_RECORD", record)
    if window:
        monkeypatch.setenv("SK_PART_WINDOW", str(window))
    got = []
    for part in ("1", "0"):
        monkeypatch.setenv("SK_PART_UPDATE", part)
        s = _set(a, 1 << logm, d)
        s.update(0, cols, w, dom)
        with pytest.raises(sk.SketchError):
            s.sync()
        got.append(s.counters.clone())
        s.close()
    assert torch.equal(*got)


@pytest.mark.parametrize("a,logm,d,n,took", [(1, 14, 5, 2_000_000, 1.34), (5, 16, 9, 20_000_000, 1.2)])
def test_no_dearer_than_single_phase(a, logm, d, n, took, monkeypatch):
    """Amounts up to 10^6, uniform keys: the single-phase update's reductions and little more (with items
    and reductions both paid for, `took` times as much): less than half of the excess is left."""
    g = torch.Generator(device="cuda").manual_seed(4)
    cols = torch.randint(0, 100_000, (a, n), generator=g, device="cuda")
    w = torch.randint(1, 1_000_001, (n,), generator=g, device="cuda")
    s = _set(a, 1 << logm, d)

    def update(part):
        monkeypatch.setenv("SK_PART_UPDATE", part)
        s.update(0, cols, w, [100_000] * a)

    two, one = best_times([lambda: update("1"), lambda: update("0")])
    s.close()
    assert two <= (1 + took) / 2 * one, (two, one)
