"""The FP32 forms in other units of length: the same system in Angstrom and rescaled.

Forces and energies are those of the oracle in the same units, within the bounds that hold in
Angstrom: 1e-5 for the forces, 2e-6 for the energies. The scales: 30 and 60 (r_c^-14 leaves the
normal FP32 numbers in between), 100 (picometres; 2^32 times 48 eps sigma^12 is no FP32 number)
and, for the random batch list, whose forces are no fixed-point sums, 7 / 30000 (r^-12 of close
pairs is no FP32 number; eps is raised so that 48 eps sigma^12 is a normal one).
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


@pytest.mark.parametrize("precision", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("u,eps", [(1.0, 0.1), (30.0, 0.1), (100.0, 0.1), (7.0 / 30000, 1e5)])
@pytest.mark.parametrize("eager", [0, 1])
def test_random_batch_list(orc, precision, u, eps, eager):
    sy, alpha, C = scaled(6001, u, eps)
    r_core, r_s, p, seed, step = 4.0 * u, 8.0 * u, 10, 3, 6
    with binding.from_system(sy, P=8, alpha=alpha, r_c=r_s, r_core=r_core, p_rbl=p, seed=seed,
                             coulomb_C=C, precision=precision) as h:
        h.set_tuning("rbl_eager", eager)
        F, E, W = h.forces_f64(step)
        pa = h.rbl_partners()
        m, S = h.sample_k(step)
    ref = orc.rbl(sy.s, sy.q, sy.types, sy.box, alpha, r_core, r_s, p, seed, step, 0, C, sy.eps,
                  sy.sig)
    assert np.array_equal(pa, ref["partners"])
    Fk, _, _ = orc.rbe_kspace(sy.s, sy.q, sy.box, alpha, C, m, S)
    assert rel_l2(F, ref["F"] + Fk) < 1e-5
    assert abs(E["lj"] - ref["U_lj"]) < 2e-6 * (abs(ref["U_lj"]) + abs(ref["U_real"]))
    assert E["lj"] == pytest.approx(ref["U_lj"], rel=2e-5)
    assert W["lj"] == pytest.approx(ref["W_lj"], rel=2e-5)


@pytest.mark.parametrize("precision", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("frac", [0.1, 1.0])
@pytest.mark.parametrize("eager", [0, 1])
def test_random_batch_list_idle_halves(orc, precision, frac, eager):
    """r_s far below 1 (8e-4): a lane's odd pair leaves half of a packed pair idle, and what that
    half computes must not reach the sums."""
    u, eps, N = 1e-4, 1e5, 4202
    sy = synth.make_system(N, density=0.1, seed=14, frac_charged=frac, eps=eps)
    sy.box, sy.sig = sy.box * u, sy.sig * u
    alpha, C = synth.ALPHA / u ** 2, synth.COULOMB_C * u * (eps / 0.1)
    r_core, r_s, p, seed, step = 4.0 * u, 8.0 * u, 7, 3, 6
    with binding.from_system(sy, P=8, alpha=alpha, r_c=r_s, r_core=r_core, p_rbl=p, seed=seed,
                             coulomb_C=C, precision=precision) as h:
        h.set_tuning("rbl_eager", eager)
        F, E, W = h.forces_f64(step)
        m, S = h.sample_k(step)
    ref = orc.rbl(sy.s, sy.q, sy.types, sy.box, alpha, r_core, r_s, p, seed, step, 0, C, sy.eps,
                  sy.sig)
    Fk, _, _ = orc.rbe_kspace(sy.s, sy.q, sy.box, alpha, C, m, S)
    assert rel_l2(F, ref["F"] + Fk) < 1e-5
    scale = abs(ref["U_lj"]) + abs(ref["U_real"])
    assert abs(E["lj"] - ref["U_lj"]) < 2e-6 * scale
    assert abs(E["real"] - ref["U_real"]) < 2e-6 * scale


@pytest.mark.parametrize("precision", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("traversal,two", [("rbl", 0), ("rbl", 1), ("cells", 1)])
def test_charges_alone(orc, precision, traversal, two):
    """No Lennard-Jones part (eps 0), neighbours some 4e-6 apart: r^-6 is an FP32 number, r^-8 is
    not, and neither may reach the forces."""
    u, N, seed, step = 2e-6, 4202, 3, 6
    sy = synth.make_system(N, density=0.1, seed=14, all_charged=True, eps=0.0)
    sy.box, sy.sig = sy.box * u, sy.sig * u
    if two:
        sy.types = (np.arange(N) % 3 == 0).astype(np.int32)
        sy.eps, sy.sig = np.zeros(4), np.array([3.0, 2.8, 2.8, 2.6]) * u
    alpha, C, r_s, r_core = synth.ALPHA / u ** 2, synth.COULOMB_C * u ** 2, 8.0 * u, 4.0 * u
    kw = dict(r_core=r_core, p_rbl=7) if traversal == "rbl" else {}
    with binding.from_system(sy, P=8, alpha=alpha, r_c=r_s, seed=seed, coulomb_C=C,
                             precision=precision, **kw) as h:
        F, E, W = h.forces_f64(step)
        m, S = h.sample_k(step)
    if traversal == "rbl":
        ref = orc.rbl(sy.s, sy.q, sy.types, sy.box, alpha, r_core, r_s, 7, seed, step, 0, C, sy.eps,
                      sy.sig)
        F0 = ref["F"] + orc.rbe_kspace(sy.s, sy.q, sy.box, alpha, C, m, S)[0]
    else:
        ref = orc.total_forces(sy.s, sy.q, sy.types, sy.box, alpha, r_s, C, sy.eps, sy.sig, m, S)
        F0 = ref["F"]
    assert rel_l2(F, F0) < 1e-5
    assert E["lj"] == 0.0 and E["real"] == pytest.approx(ref["U_real"], rel=1e-5)
