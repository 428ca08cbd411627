"""The wide partitioned update of widths 2^17 .. 2^20 (chunks sorted by part in shared memory):
counters equal to per-tuple hashing, bit for bit."""
import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


def _both(monkeypatch, a, m, d, cols, domain, window=None):
    got = []
    for tables in ("1", "0"):
        monkeypatch.setenv("SK_KEY_TABLE", tables)
        monkeypatch.setenv("SK_PART_UPDATE", "2")
        if window:
            monkeypatch.setenv("SK_PART_WINDOW", str(window))
        s = sk.SketchSet([a] + [1] * a, [(0, k, 1 + k, 0) for k in range(a)], m, d, 3)
        s.update(0, cols, domain=domain)
        try:
            s.sync()
        except sk.SketchError as e:
            assert e.status == sk.SK_ERR_KEY_OUT_OF_DOMAIN
        got.append(s.counters.clone())
        s.close()
    assert torch.equal(*got)


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 70_001])
@pytest.mark.parametrize("a,logm,d", [(1, 20, 16), (2, 17, 9), (3, 18, 4), (5, 20, 5), (2, 19, 13), (4, 17, 1)])
def test_equals_per_tuple(n, a, logm, d, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(n + a)
    dom = [1 + 97 * (u + 1) ** 4 for u in range(a)]
    cols = torch.stack([torch.randint(0, x, (n,), generator=g, device="cuda") for x in dom])
    _both(monkeypatch, a, 1 << logm, d, cols, dom)


@pytest.mark.parametrize("window", [None, 5000, 4096])
def test_heavy_key_and_windows(window, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(9)
    n = 300_007
    cols = torch.randint(0, 5000, (2, n), generator=g, device="cuda")
    cols[:, torch.rand(n, generator=g, device="cuda") < 0.7] = 17   # one bin holds most items of a row
    _both(monkeypatch, 2, 1 << 20, 16, cols, [5000, 5000], window)


def test_keys_outside_their_domain_are_left_out(monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(4)
    cols = torch.randint(-3, 1010, (2, 20_011), generator=g, device="cuda")
    cols[1, ::7] = (1 << 40) + 5
    _both(monkeypatch, 2, 1 << 18, 9, cols, [1000, 1000])
