"""A step in two graph branches is not slower than in one.

The k-space chain runs beside the real-space pass. Where it took the SMs first, a pass that fills
the GPU about once crowded on those left over and ran up to 2.3 times as long. A handle that
records its phase times steps in one branch; two branches may take a tenth longer at most (they
exist to take less; the tenth is for the clock and the events).
"""
import pytest
import torch

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def step_us(h, n=10):
    h.step(4)
    best = float("inf")
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        h.step(n)
        b.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * a.elapsed_time(b) / n)
    return best


@pytest.mark.parametrize("precision,traversal,N,frac", [("fp64", "rbl", 5000, 1.0),
                                                        ("fp64", "rbl", 30001, 0.1),
                                                        ("fp32_comp", "rbl", 10001, 1.0),
                                                        ("fp32_comp", "rbl", 45000, 1.0),
                                                        ("fp64", "pair", 1701, 1.0),
                                                        ("fp32", "pair", 90000, 1.0),
                                                        ("fp64", "list", 30001, 1.0),
                                                        ("fp32_comp", "list", 64003, 1.0),
                                                        ("fp32_comp", "cells", 30001, 0.1)])
def test_two_branches_are_not_slower(precision, traversal, N, frac):
    sy = synth.make_system(N, density=0.1, seed=11, frac_charged=frac)
    kw = dict(r_core=5.0, p_rbl=10) if traversal == "rbl" else {}
    with binding.from_system(sy, P=100, alpha=synth.ALPHA, r_c=10.0 if N > 2000 else 8.0,
                             precision=precision, **kw) as h:
        if traversal == "pair":
            h.set_tuning("pair_cluster", 0)
        if traversal == "list":
            h.set_neighbor_list(1.0)
        two = step_us(h)
        h.set_profiling(True)
        one = step_us(h)
    assert two < 1.1 * one, (two, one)
