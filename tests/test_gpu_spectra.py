"""Product-of-spectra estimates at every transform length: equal, as integers, to the exact
inner product (two relations) and to the stepwise GF(2^64 - 2^32 + 1) estimate (more)."""
import numpy as np
import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


def _chain(r):
    return ([1] + [2] * (r - 2) + [1], [(k, 0 if k == 0 else 1, k + 1, 0) for k in range(r - 1)])


def _star(r):
    return [r - 1] + [1] * (r - 1), [(0, k, 1 + k, 0) for k in range(r - 1)]


def _fill(s, seed, bits):
    """Counters of mixed magnitude: mostly small, some of up to `bits` bits, with both signs."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = s.counters
    small = torch.randint(-50, 51, c.shape, generator=g, device="cuda")
    big = torch.randint(-(1 << bits) + 1, 1 << bits, c.shape, generator=g, device="cuda")
    pick = torch.rand(c.shape, generator=g, device="cuda") < 0.05
    c.copy_(torch.where(pick, big, small))


@pytest.mark.parametrize("logm", range(10, 23))
def test_two_relations_exact_inner_product(logm, monkeypatch):
    monkeypatch.setenv("SK_FUSED_SMALL", "0")
    d = 3 if logm < 20 else 2
    s = sk.SketchSet(*_chain(2), 1 << logm, d, 5)
    _fill(s, logm, 62)
    a, b = (x.numpy().astype(object) for x in s.counters.cpu())
    assert s.estimate()["rows"] == [int((a[i] * b[i]).sum()) for i in range(d)]
    s.close()


@pytest.mark.parametrize("logm", range(10, 23))
@pytest.mark.parametrize("shape,r", [(_chain, 3), (_star, 4), (_chain, 6)])
def test_rows_equal_stepwise(logm, shape, r, monkeypatch):
    monkeypatch.setenv("SK_FUSED_SMALL", "0")
    d = 5 if logm < 17 else 2
    s = sk.SketchSet(*shape(r), 1 << logm, d, 7)
    _fill(s, 100 + logm, 20)
    got = s.estimate()
    s.set_estimator("ntt")
    want = s.estimate()
    assert got["rows"] == want["rows"] and got["median"] == want["median"]
    s.close()


@pytest.mark.parametrize("logms", [(10, 10, 11, 12), (13, 9, 16, 13, 17, 5), (18, 14)])
def test_many_sets_equal_single(logms):
    sets = []
    for i, logm in enumerate(logms):
        s = sk.SketchSet(*(_chain(3 + i % 4) if i % 2 else _star(2 + i % 4)), 1 << logm, 3 + i % 3, 11 + i)
        _fill(s, 200 + i, 8 + 9 * i)
        sets.append(s)
    many = sk.estimate_many(sets)
    for s, e in zip(sets, many):
        s.set_estimator("ntt")
        assert s.estimate()["rows"] == e["rows"]
    assert np.all([e["retries"] == 0 for e in many])


_SHARED = ([1, 2, 1, 1], [(0, 0, 1, 0), (2, 0, 1, 0), (3, 0, 1, 1)])   # three relations share an attribute


@pytest.mark.parametrize("m", [2, 3, 127, 512, 513, 1000, 1024, 1025, 2048, 5000, 16384, 20_001, 65_536, 100_000,
                               131_073, 524_288, 1_000_000, 1 << 22])
@pytest.mark.parametrize("query", [_SHARED, _chain(2), _chain(3), _chain(5), _star(4)])
def test_schedule_equals_stepwise(m, query, monkeypatch):
    """Widths that are no power of two and shared attributes: the schedule modulo the primes."""
    if query is not _SHARED and (m & (m - 1)) == 0:
        pytest.skip("a product of spectra")
    d = 5 if m < 100_000 else 2
    s = sk.SketchSet(*query, m, d, 7)
    _fill(s, m % 1000 + len(query[0]), 20)
    got = s.estimate()
    assert got["max_limbs"] < 9 and got["limb_bits"] == 0   # CRT primes, not limbs
    s.set_estimator("ntt")
    assert s.estimate()["rows"] == got["rows"]
    s.close()
