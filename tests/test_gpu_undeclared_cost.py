"""Batches without declared domains take the tables only where these gain: never much dearer than
per-tuple hashing, and with the same counters."""
import pytest
import torch

import paper_2402_15953_gb300 as sk
from _timing import best_times

pytestmark = pytest.mark.gpu


def _set(a, m, d):
    return sk.SketchSet([a] + [1] * a, [(0, k, 1 + k, 0) for k in range(a)], m, d, 3)


def _compare(a, d, cols, w, bound, monkeypatch):
    s = _set(a, 1 << 16, d)

    def update(part):
        monkeypatch.setenv("SK_PART_UPDATE", part)
        s.update(0, cols, w)

    got = []
    for part in ("1", "0"):
        s.reset()
        update(part)
        got.append(s.counters[0].clone())
    assert torch.equal(*got)
    tables, hashing = best_times([lambda: update("1"), lambda: update("0")])
    s.close()
    assert tables <= bound * hashing, (tables, hashing)


@pytest.mark.parametrize("a,d,n,domain,took", [(5, 5, 10_000_019, 2_000_000, 1.98), (5, 9, 30_000_001, 5_000_000, 1.65)])
def test_uniform_keys_of_wide_domains(a, d, n, domain, took, monkeypatch):
    """Uniform keys over a fifth to a sixth as many values as tuples: building the tables and
    fetching their records from memory costs more than hashing (`took` times that when every dense
    batch took them): less than half of the excess is left."""
    g = torch.Generator(device="cuda").manual_seed(2)
    cols = torch.randint(0, domain, (a, n), generator=g, device="cuda")
    _compare(a, d, cols, None, (1 + took) / 2, monkeypatch)


def test_skewed_keys_of_a_wide_domain(monkeypatch):
    """The same domain with most tuples on few keys gains from the tables."""
    g = torch.Generator(device="cuda").manual_seed(2)
    cols = (torch.rand((5, 10_000_019), generator=g, device="cuda", dtype=torch.float64) ** 8 * 1_000_000).long()
    _compare(5, 9, cols, None, 0.8, monkeypatch)


@pytest.mark.parametrize("a,d,n,took", [(2, 9, 4_194_304, 1.53), (2, 5, 10_000_019, 1.44)])
def test_large_weights_of_two_columns(a, d, n, took, monkeypatch):
    """Amounts that no item of the tables' path holds: their reductions bind either way, and with two
    columns the tables only add to them (`took` times hashing): less than half of that is left."""
    g = torch.Generator(device="cuda").manual_seed(2)
    cols = torch.randint(0, 50_000, (a, n), generator=g, device="cuda")
    w = torch.randint(1, 1_000_001, (n,), generator=g, device="cuda")
    _compare(a, d, cols, w, (1 + took) / 2, monkeypatch)
