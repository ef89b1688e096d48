"""Batches in AA order run the persistent kernel with one lattice instead of two; a step of it moves the
same bytes and does the same arithmetic, so it takes about the same time."""
from __future__ import annotations

import pytest

import scenarios as S

pytestmark = pytest.mark.gpu

AB, AA = 0, 1


def test_a_batch_in_aa_order_costs_what_the_persistent_kernel_costs_on_two_lattices():
    """At most 1.12 times (measured 1.00 to 1.01; 1.22 when the collide phase addressed every slot for
    itself).  Timed in turn, the best of five, so that clocks and neighbours do not decide."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2203_04508_gb300 as G
    scs = S.c4_batch(n=96)
    batches = {}
    for layout in (AB, AA):
        b = G.Batch([sc.physics() for sc in scs], layout=layout)
        b.init([sc.droplets() for sc in scs])
        b.set_kernel(1)
        b.set_tile(5)
        b.set_schedule(1)
        b.step(10)
        b.synchronize()
        batches[layout] = b
    best = {AB: float("inf"), AA: float("inf")}
    for _ in range(5):
        for layout, b in batches.items():
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(b.stream)
            b.step(10)
            e1.record(b.stream)
            b.synchronize()
            best[layout] = min(best[layout], e0.elapsed_time(e1))
    for b in batches.values():
        b.check()
    print(best, best[AA] / best[AB])
    assert best[AA] <= 1.12 * best[AB]
