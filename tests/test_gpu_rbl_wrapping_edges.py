"""Random batch list in wrapping boxes whose edges divide the kernel's padding coordinate.

The FP32 kernel takes candidates 64 at a time and pads the last 64 with a far coordinate. A box
of three cells on some axis folds every difference into [-L/2, L/2), and folding a far coordinate
gives any value: exactly 0 where L divides it (24, 28, 32, 34, 37, ...). A padded slot must not
count, whatever it folds to. Set sizes and drawn partners are exact; forces hold the FP32 forms'
1e-5, energies their 2e-6 of the sums' scale.
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


@pytest.mark.parametrize("precision", ["fp32_comp", "fp32"])
@pytest.mark.parametrize("eager", [0, 1])
@pytest.mark.parametrize("box,r_s,N", [((24.0, 24.0, 24.0), 8.0, 1301),
                                       ((32.0, 32.0, 32.0), 10.0, 3000),
                                       ((32.0, 32.0, 32.0), 10.0, 3001),
                                       ((34.0, 34.0, 34.0), 10.0, 3600),
                                       ((37.0, 37.0, 37.0), 10.0, 4601),
                                       ((28.0, 32.0, 34.0), 8.5, 2800)])
def test_padding_never_counts(orc, precision, eager, box, r_s, N):
    r_core, p, seed, step = 5.0, 10, 3, 6
    sy = synth.make_system(N, L=box[0], seed=5, frac_charged=0.3)
    sy.box = np.array(box)
    with binding.from_system(sy, P=8, alpha=ALPHA, r_c=r_s, r_core=r_core, p_rbl=p, seed=seed,
                             precision=precision) as h:
        h.set_tuning("rbl_eager", eager)
        F, E, W = h.forces_f64(step)
        nc, ns = h.neighbor_counts()
        pa = h.rbl_partners()
        n, _, _ = h.cells()
        m, S = h.sample_k(step)
    assert min(n) == 3 and r_s + min(box) / 3 >= min(box) / 2  # (the wrapping variant)
    ref = orc.rbl(sy.s, sy.q, sy.types, sy.box, ALPHA, r_core, r_s, p, seed, step, 0, C, sy.eps,
                  sy.sig)
    assert np.array_equal(nc, ref["n_core"]) and np.array_equal(ns, ref["n_shell"])
    assert np.array_equal(pa, ref["partners"])
    Fk, _, _ = orc.rbe_kspace(sy.s, sy.q, sy.box, ALPHA, C, m, S)
    F0 = ref["F"] + Fk
    assert float(np.linalg.norm(F - F0) / np.linalg.norm(F0)) < 1e-5
    scale = abs(ref["U_lj"]) + abs(ref["U_real"])
    assert abs(E["lj"] - ref["U_lj"]) < 2e-6 * scale
    assert abs(E["real"] - ref["U_real"]) < 2e-6 * scale + 1e-6
