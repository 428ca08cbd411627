"""Weighted batches through the two-phase partitioned update: counters equal to the
single-phase key-table update's, bit for bit."""
import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


def _weights(kind, n, g):
    if kind == "turnstile":
        return 1 - 2 * (torch.rand(n, generator=g, device="cuda") < 0.1).to(torch.int64)
    w = torch.randint(-3, 4, (n,), generator=g, device="cuda")
    if kind == "edges":   # at and beyond the largest weight an item can hold, and at int64's limits
        edge = torch.tensor([65535, -65535, 65536, -65536, 65537, 1 << 40, -(1 << 40), (1 << 63) - 1, -(1 << 63), 0],
                            device="cuda")
        w[::3] = edge[torch.randint(0, len(edge), (w[::3].numel(),), generator=g, device="cuda")]
    return w


@pytest.mark.parametrize("kind", ["turnstile", "small", "edges"])
@pytest.mark.parametrize("a,logm,d,n,window,record", [
    (5, 16, 9, 1_048_613, 0, "24"), (1, 13, 9, 131_107, 0, "24"), (3, 16, 7, 1_100_003, 300_000, "24"),
    (2, 16, 1, 1_048_576, 0, "24"), (4, 16, 9, 1_048_609, 0, "32"), (5, 13, 14, 140_001, 0, "24"),
    (2, 12, 13, 70_001, 0, "24")])
def test_equals_single_phase(kind, a, logm, d, n, window, record, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(a * 100 + d)
    dom = [3001 + 977 * u for u in range(a)]
    cols = torch.stack([torch.randint(0, x, (n,), generator=g, device="cuda") for x in dom])
    cols[:, torch.rand(n, generator=g, device="cuda") < 0.3] = 11   # a heavy bin per row
    cols[0, 100::5003] = dom[0]                                     # outside: left out
    w = _weights(kind, n, g)
    monkeypatch.setenv("SK_KEY_TABLE", "1")
    monkeypatch.setenv("SK_PART_RECORD", record)
    if window:
        monkeypatch.setenv("SK_PART_WINDOW", str(window))
    got = []
    for part in ("1", "0"):
        monkeypatch.setenv("SK_PART_UPDATE", part)
        s = sk.SketchSet([a] + [1] * a, [(0, k, 1 + k, 0) for k in range(a)], 1 << logm, d, 3)
        launches = sk.sk_launch_count()
        s.update(0, cols, w, dom)
        launches = sk.sk_launch_count() - launches
        with pytest.raises(sk.SketchError):
            s.sync()
        assert launches == (1 + 2 * (-(-n // (window or n))) if part == "1" else 2)
        got.append(s.counters.clone())
        s.close()
    assert torch.equal(*got)
