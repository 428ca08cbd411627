"""Times of calls on the GPU, for tests that hold one path of a call against another."""
from __future__ import annotations

from typing import Callable, List

import torch


def best_times(calls: List[Callable[[], None]], rounds: int = 25) -> List[float]:
    """The shortest time of each call in milliseconds, the calls taken in turn."""
    best = [float("inf")] * len(calls)
    for r in range(rounds + 2):
        for i, call in enumerate(calls):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            call()
            b.record()
            b.synchronize()
            if r >= 2:   # two rounds of warm-up
                best[i] = min(best[i], a.elapsed_time(b))
    return best
