"""The FP32 cluster kernel's work split and its erfc fit against the FP64 oracle.

A super-cluster's visits are shared by several warps, and in small boxes by several blocks; the
split follows the box's size. The Coulomb terms come from a polynomial for erfcx up to
sqrt(alpha) r_c of about 3.7 and from erfcf past it. Neighbour counts are exact; forces hold
the 1e-5 of the other FP32 parity tests, which covers the frame coordinates' rounding.
"""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

import sampled

pytestmark = pytest.mark.gpu

C, ALPHA, RC = synth.COULOMB_C, synth.ALPHA, synth.R_CUT


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


# 32 warps a super-cluster in the smallest boxes, 4 in the middle, 2 in the largest; ragged sizes
@pytest.mark.parametrize("N,kw", [(2300, dict(L=30.0, all_charged=True)),
                                  (9001, dict(density=0.09, all_charged=True)),
                                  (9002, dict(density=0.1, frac_charged=0.1)),
                                  (60003, dict(density=0.1, frac_charged=0.1)),
                                  (60003, dict(density=0.09, all_charged=True)),
                                  (400001, dict(density=0.1, frac_charged=0.1))])
def test_split_shapes_match_oracle(orc, N, kw):
    sy = synth.make_system(N, seed=31, **kw)
    idx = np.sort(np.random.default_rng(5).choice(N, 48, replace=False))
    with binding.from_system(sy, P=60, alpha=ALPHA, r_c=RC) as h:
        F, _, _ = h.forces_f64(4)
        nbr, _ = h.neighbor_counts()
        m, S = sampled.oracle_modes(orc, h, sy, 60, 4)
    Fo, no = sampled.total_forces_sampled(orc, sy, idx, m, S)
    assert np.array_equal(nbr[idx], no)
    assert rel_l2(F[idx], Fo) < 1e-5


@pytest.mark.parametrize("alpha", [0.01, 0.09, 0.13, 0.2, 0.6])
def test_erfc_fit_and_fallback_match_oracle(orc, alpha):
    sy = synth.make_system(2000, density=0.02, seed=8, all_charged=True)
    with binding.from_system(sy, P=40, alpha=alpha, r_c=RC) as h:
        F, E, _ = h.forces_f64(1)
        m, S = sampled.oracle_modes(orc, h, sy, 40, 1, alpha=alpha)
    ref = orc.total_forces(sy.s, sy.q, sy.types, sy.box, alpha, RC, C, sy.eps, sy.sig, m, S)
    assert rel_l2(F, ref["F"]) < 1e-5
    assert E["real"] == pytest.approx(ref["U_real"], rel=1e-5)


@pytest.mark.parametrize("box,n", [((27.2, 27.2, 27.2), 2001), ((25.7, 25.6, 25.8), 1701),
                                   ((60.0, 27.0, 26.0), 4201), ((34.2, 31.0, 28.2), 3000)])
@pytest.mark.parametrize("all_charged", [False, True])
def test_five_cell_boxes_match_oracle(orc, box, n, all_charged):
    """Boxes of five cells of r_c / 2 in y or z: stencil rows reach past the frame's edge, and
    clusters lie across it."""
    sy = synth.make_system(n, L=box[0], seed=12, all_charged=all_charged)
    sy.box = np.array(box)
    with binding.from_system(sy, P=40, alpha=ALPHA, r_c=RC) as h:
        F, E, _ = h.forces_f64(2)
        nbr, _ = h.neighbor_counts()
        m, S = sampled.oracle_modes(orc, h, sy, 40, 2)
    ref = orc.total_forces(sy.s, sy.q, sy.types, sy.box, ALPHA, RC, C, sy.eps, sy.sig, m, S)
    assert np.array_equal(nbr, ref["nbr"])
    assert rel_l2(F, ref["F"]) < 1e-5
    assert E["lj"] == pytest.approx(ref["U_lj"], rel=2e-6)
