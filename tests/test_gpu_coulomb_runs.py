"""The charged subset's Coulomb pass finds its candidates in runs of cells: more runs than a warp has
lanes (cells of r_c / 3), none or hardly any charges, rows that wrap in x and rows that cover the
whole box, strong splitting (no erfc fit) against the oracle. 1e-5 of the forces, as elsewhere."""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu

C = synth.COULOMB_C


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


@pytest.mark.parametrize("precision", ["fp32_comp", "fp32", "fp64"])
@pytest.mark.parametrize("N,box,frac,sub,alpha", [(9001, (60., 50., 55.), 0.4, 3, 0.09),
                                                  (9001, (30., 70., 70.), 0.45, 3, 0.09),
                                                  (5003, (25., 60., 60.), 0.3, 2, 0.09),
                                                  (5003, (90., 40., 40.), 0.002, 1, 0.09),
                                                  (4001, (45., 45., 45.), 0.2, 2, 0.6)])
def test_candidate_runs_match_oracle(orc, precision, N, box, frac, sub, alpha):
    build.build()
    sy = synth.make_system(N, L=40.0, frac_charged=frac, seed=17)
    sy.box = np.array(box)
    rc = 10.0
    with binding.from_system(sy, P=20, alpha=alpha, r_c=rc, precision=precision, coulomb_C=C,
                             cell_sub=sub) as h:
        F, E, _ = h.forces_f64(0)
        m, S = h.sample_k(0)
    ref = orc.total_forces(sy.s, sy.q, sy.types, sy.box, alpha, rc, C, sy.eps, sy.sig, m, S)
    assert rel_l2(F, ref["F"]) < (1e-12 if precision == "fp64" else 1e-5)
