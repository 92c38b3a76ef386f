"""The per-particle pair kernel where its tiles are shared by several blocks, and the FP64 form's
evaluation in grid units, against the oracle: a handful of particles, ragged sizes on both sides
of a split's end, wrapping boxes, cubic and orthorhombic edges, two LJ types, every particle
charged and none. Neighbour counts are exact; forces hold the forms' 1e-5 and 1e-10."""
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


@pytest.mark.parametrize("precision,tol", [("fp32_comp", 1e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("N,L,frac,ortho,two", [(41, 25.2, 1.0, False, False),
                                                (2001, 27.2, 0.1, False, True),
                                                (5003, 36.9, 1.0, True, True),
                                                (8001, 60.0, 0.0, True, False),
                                                (70001, 88.8, 0.1, False, False),
                                                (140001, 112.0, 0.1, True, True)])
def test_split_pair_pass_matches_oracle(orc, precision, tol, N, L, frac, ortho, two):
    sy = synth.make_system(N, L=L, frac_charged=frac, seed=19)
    if ortho:
        sy.box = sy.box * np.array([1.05, 1.0, 0.97])
    if two:
        sy.types = (np.arange(N) % 2).astype(np.int32)
        sy.eps, sy.sig = np.array([0.1, 0.15, 0.15, 0.2]), np.array([3.0, 2.8, 2.8, 2.6])
    idx = np.arange(N) if N < 6000 else np.sort(np.random.default_rng(3).choice(N, 40, replace=False))
    with binding.from_system(sy, P=24, alpha=ALPHA, r_c=RC, precision=precision) as h:
        h.set_tuning("pair_cluster", 0)
        F, E, W = h.forces_f64(5)
        nbr, _ = h.neighbor_counts()
        h.forces(5, energies=False)
        e2, _ = h.energies()
        m, S = sampled.oracle_modes(orc, h, sy, 24, 5)
    Fo, no = sampled.total_forces_sampled(orc, sy, idx, m, S)
    assert np.array_equal(nbr[idx], no)
    assert rel_l2(F[idx], Fo) < tol
    assert e2 == E  # the counting and the plain pass, bit for bit
    if N < 6000:
        ref = orc.total_forces(sy.s, sy.q, sy.types, sy.box, ALPHA, RC, C, sy.eps, sy.sig, m, S)
        scale = abs(ref["U_lj"]) + abs(ref["U_real"])
        assert abs(E["lj"] - ref["U_lj"]) < tol * scale
        assert abs(E["real"] - ref["U_real"]) < tol * scale
