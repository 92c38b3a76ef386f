"""The cluster kernel's fixed-point sums become forces a block of 512 to 4,096 at a time: sizes at and
around the block's steps, odd numbers of sums, against the per-particle kernel (two FP32 forms of
1e-5 each against the oracle; 2e-12 in FP64, two of 1e-12)."""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision", [(1023, "fp32_comp"), (4001, "fp64"), (103765, "fp32"),
                                         (207531, "fp32_comp"), (415061, "fp32_comp"),
                                         (830127, "fp32")])
def test_finish_matches_per_particle(N, precision):
    build.build()
    sy = synth.make_system(N, density=0.03, frac_charged=0.1, seed=23)
    F = []
    for on in (1, 0):
        with binding.from_system(sy, P=4, alpha=0.09, r_c=6.0, precision=precision) as h:
            h.set_tuning("pair_cluster", on)
            F.append([h.forces_f64(0)[0], h.forces_f64(0)[0]])
    a, b = F[0][0], F[1][0]
    assert np.array_equal(F[0][0], F[0][1])  # (the sums are cleared for the next evaluation)
    assert np.linalg.norm(a - b) < (2e-12 if precision == "fp64" else 2e-5) * np.linalg.norm(b)
