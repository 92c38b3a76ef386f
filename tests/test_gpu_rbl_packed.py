"""The FP32 random batch list kernel (packed pairs, 64 candidates a window) against the oracle.

Sizes where its windows, halves and draws can go wrong: a stencil of a few candidates, one
particle past a warp, windows cut short, draw counts that leave half a packed pair idle, every
particle charged and none, two LJ types in an orthorhombic box. Set sizes and drawn partners
are exact; forces hold the FP32 forms' 1e-5, energies their 2e-6 of the sums' scale.
"""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu

C, ALPHA = synth.COULOMB_C, synth.ALPHA


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


@pytest.mark.parametrize("precision", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("N,density,frac,p,two", [(33, 0.008, 1.0, 3, False),
                                                  (1025, 0.05, 0.0, 1, False),
                                                  (4099, 0.1, 0.3, 32, True),
                                                  (9001, 0.1, 1.0, 7, False),
                                                  (20001, 0.03, 1.0, 30, True)])
@pytest.mark.parametrize("eager", [0, 1])
def test_packed_kernel_matches_oracle(orc, precision, N, density, frac, p, two, eager):
    r_core, r_s, seed, step = 2.7, 5.0, 3, 6
    sy = synth.make_system(N, density=density, seed=21, frac_charged=frac)
    if two:
        sy.box = sy.box * np.array([1.15, 1.0, 0.95])
        sy.types = (np.arange(N) % 3 == 0).astype(np.int32)
        sy.eps, sy.sig = np.array([0.1, 0.15, 0.15, 0.2]), np.array([2.4, 2.2, 2.2, 2.0])
    with binding.from_system(sy, P=8, alpha=ALPHA, r_c=r_s, r_core=r_core, p_rbl=p, seed=seed,
                             precision=precision) as h:
        h.set_tuning("rbl_eager", eager)
        F, E, W = h.forces_f64(step)
        nc, ns = h.neighbor_counts()
        pa = h.rbl_partners()
        m, S = h.sample_k(step)
    ref = orc.rbl(sy.s, sy.q, sy.types, sy.box, ALPHA, r_core, r_s, p, seed, step, 0, C, sy.eps,
                  sy.sig)
    assert np.array_equal(nc, ref["n_core"]) and np.array_equal(ns, ref["n_shell"])
    assert np.array_equal(pa, ref["partners"])
    Fk, _, _ = orc.rbe_kspace(sy.s, sy.q, sy.box, ALPHA, C, m, S)
    assert rel_l2(F, ref["F"] + Fk) < 1e-5
    scale = abs(ref["U_lj"]) + abs(ref["U_real"])
    assert abs(E["lj"] - ref["U_lj"]) < 2e-6 * scale
    assert abs(E["real"] - ref["U_real"]) < 2e-6 * scale + 1e-6
