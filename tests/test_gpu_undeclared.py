"""Batches without declared domains: found dense, they take the tables and the partitioned
update, else per-tuple hashing; the counters are the same, bit for bit."""
import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


def _run(a, logm, d, cols, w):
    s = sk.SketchSet([a] + [1] * a, [(0, k, 1 + k, 0) for k in range(a)], 1 << logm, d, 3)
    s.update(0, cols, w)
    s.sync()   # no domain was declared: no key is outside one
    c = s.counters.clone()
    s.close()
    return c


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("keys", ["dense", "one far", "negative", "sparse", "at the limit"])
@pytest.mark.parametrize("a,logm,d,n", [(2, 16, 9, 1_048_579), (5, 16, 9, 1_500_001), (3, 13, 9, 262_151),
                                        (4, 16, 1, 1_048_576)])
def test_equals_per_tuple(a, logm, d, n, keys, weighted, monkeypatch):
    g = torch.Generator(device="cuda").manual_seed(a + d)
    cols = torch.randint(0, 50_000, (a, n), generator=g, device="cuda")
    if keys == "one far":
        cols[a - 1, n - 2] = (1 << 60) + 3
    elif keys == "negative":
        cols[0, n // 2 + 1] = -1
    elif keys == "sparse":
        cols = torch.randint(-(1 << 62), 1 << 62, (a, n), generator=g, device="cuda")
    elif keys == "at the limit":   # the tables hold n / 4 keys per attribute
        cols[0, 12345] = n // 4 - 1
        cols[1, 54321] = n // 4
    w = torch.randint(-3, 4, (n,), generator=g, device="cuda") if weighted else None
    monkeypatch.setenv("SK_UNDECLARED_LEAST", "1")
    found = _run(a, logm, d, cols, w)
    monkeypatch.setenv("SK_PART_UPDATE", "0")
    assert torch.equal(found, _run(a, logm, d, cols, w))


def test_captured_update(monkeypatch):
    """Under capture the update allocates nothing and reads the buffer's contents at replay."""
    monkeypatch.setenv("SK_UNDECLARED_LEAST", "1")
    n = 1_048_576
    cols = torch.randint(0, 1000, (2, n), device="cuda")
    s = sk.SketchSet([2, 1, 1], [(0, 0, 1, 0), (0, 1, 2, 0)], 1 << 16, 9, 3)
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        s.update(0, cols)
    cols.copy_(torch.randint(-(1 << 62), 1 << 62, (2, n), device="cuda"))
    s.reset()
    graph.replay()
    torch.cuda.synchronize()
    got = s.counters.clone()
    s.reset()
    s.update(0, cols)
    assert torch.equal(got, s.counters)
    s.close()
