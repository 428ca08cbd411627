"""One-attribute relations into global counters: equal keys of a warp are added as one, with the
same counters as the key-table update, bit for bit (single batches and batched plans)."""
import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 33, 100_003])
@pytest.mark.parametrize("m", [1 << 16, 60_001])
@pytest.mark.parametrize("weights", ["none", "small", "edge", "huge"])
def test_equal_keys(n, m, weights, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(n)
    keys = torch.randint(0, 40, (1, n), generator=g, device="cuda")
    keys[0, ::5] = 7
    w = None
    if weights != "none":
        top = {"small": 3, "edge": (1 << 25) - 1, "huge": (1 << 62)}[weights]
        w = torch.randint(-top, top + 1, (n,), generator=g, device="cuda")
        if weights == "edge":
            w[::3] = 1 << 25 if n > 32 else top   # some warps beyond the merged range
    d, got = 9, []
    for domain in ([50], None):
        monkeypatch.setenv("SK_KEY_TABLE", "1")
        s = sk.SketchSet([1, 1], [(0, 0, 1, 0)], m, d, 3)
        s.update(0, keys, w, domain)
        got.append(s.counters.clone())
        s.close()
    s = sk.SketchSet([1, 1], [(0, 0, 1, 0)], m, d, 3)
    plan = sk.UpdatePlan([(s, 0, keys, w)])
    plan.run()
    got.append(s.counters.clone())
    plan.close()
    s.close()
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
