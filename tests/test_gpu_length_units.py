"""The FP32 forms in other units of length: the same system in Angstrom and rescaled.

Forces and energies are those of the oracle in the same units, within the bounds that hold in
Angstrom: 1e-5 for the forces, 2e-6 for the energies. The scales: 30 and 60 (r_c^-14 leaves the
normal FP32 numbers in between) and 100 (picometres; 2^32 times 48 eps sigma^12 is no FP32 number).
"""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def scaled(N, u, eps, density=0.1):
    sy = synth.make_system(N, density=density, seed=14, frac_charged=0.1, eps=eps)
    sy.box, sy.sig = sy.box * u, sy.sig * u
    return sy, synth.ALPHA / u ** 2, synth.COULOMB_C * u * (eps / 0.1)


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("precision", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("u", [1.0, 30.0, 60.0, 100.0])
@pytest.mark.parametrize("cluster", [0, 1])
def test_cells(orc, precision, u, cluster):
    sy, alpha, C = scaled(4202, u, 0.1)
    rc = 10.0 * u
    with binding.from_system(sy, P=40, alpha=alpha, r_c=rc, coulomb_C=C, precision=precision) as h:
        h.set_tuning("pair_cluster", cluster)
        F, E, W = h.forces_f64(1)
        nbr, _ = h.neighbor_counts()
        m, S = h.sample_k(1)
    ref = orc.total_forces(sy.s, sy.q, sy.types, sy.box, alpha, rc, C, sy.eps, sy.sig, m, S)
    assert np.array_equal(nbr, ref["nbr"])
    assert rel_l2(F, ref["F"]) < 1e-5
    assert E["lj"] == pytest.approx(ref["U_lj"], rel=2e-6)
