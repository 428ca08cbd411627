"""Key columns in page-locked host memory: read across the link once, same counters."""
import pytest
import torch

import paper_2402_15953_gb300 as sk

pytestmark = pytest.mark.gpu


def _counters(cols, m, d, domain):
    s = sk.SketchSet([2, 1, 1], [(0, 0, 1, 0), (0, 1, 2, 0)], m, d, 3)
    before = sk.sk_launch_count()
    sk.sk_sketch_update_batch(s.handle, 0, cols.shape[1], cols.data_ptr(), cols.stride(0), None, domain,
                              torch.cuda.current_stream().cuda_stream)
    launches = sk.sk_launch_count() - before
    s.sync()
    c = s.counters.clone()
    s.close()
    return c, launches


@pytest.mark.parametrize("logm,d,declared", [(16, 9, False), (17, 9, True), (17, 8, True)])
def test_equal_to_device_columns(logm, d, declared, monkeypatch):
    monkeypatch.setenv("SK_UNDECLARED_LEAST", "1")
    monkeypatch.setenv("SK_PART_UPDATE", "2")
    n = 1_048_601
    host = torch.randint(0, 1000, (2, n), generator=torch.Generator().manual_seed(d)).pin_memory()
    domain = [1000, 1000] if declared else None
    there, launches = _counters(host, 1 << logm, d, domain)
    here, _ = _counters(host.cuda(), 1 << logm, d, domain)
    assert torch.equal(there, here)
    if not declared:   # the per-tuple update alone: no pass that looks for dense keys first
        assert launches == 1
