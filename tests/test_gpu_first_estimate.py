"""The first estimates of a process, on streams that do not wait for the default one: the
constants that they upload must be in place before anything reads them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys, torch
import paper_2402_15953_gb300 as sk
many = sys.argv[1] == "many"
with torch.cuda.stream(torch.cuda.Stream()):   # non-blocking
    sets = []
    for m in (256, 1 << 10, 1000, 1 << 14):    # one launch; columns and rows; stepwise; both
        s = sk.SketchSet([1, 2, 1], [(0, 0, 1, 0), (1, 1, 2, 0)], m, 5, 7)
        for k, a in enumerate((1, 2, 1)):
            s.update(k, torch.randint(0, 50, (a, 2000), device="cuda"))
        s.sync()
        sets.append(s)
    first = [e["rows"] for e in sk.estimate_many(sets)] if many else [s.estimate()["rows"] for s in reversed(sets)][::-1]
    for s in sets:
        s.set_estimator("ntt")                 # the GF(q) steps read none of these constants
    assert first == [s.estimate()["rows"] for s in sets]
"""


@pytest.mark.parametrize("form", ["one", "many"])
def test_first_estimates_on_a_side_stream(form):
    subprocess.run([sys.executable, "-c", CHILD, form], cwd=ROOT, check=True, timeout=300)
