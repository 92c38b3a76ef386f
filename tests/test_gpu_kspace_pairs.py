"""The FP32 k-space passes take their particles and their modes two at a time: odd numbers of
both, one of each, tiles and mode chunks that end on an odd one, few and many threads a particle.

rho holds the bounds of the forms (2e-6 compensated, 2e-5 plain), forces 1e-5, against the oracle.
"""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu

C, ALPHA = synth.COULOMB_C, synth.ALPHA


def rel_l2(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b))


@pytest.mark.parametrize("precision,tol", [("fp32_comp", 2e-6), ("fp32", 2e-5)])
@pytest.mark.parametrize("N,nq,P", [(500, 3, 1), (500, 5, 2), (2000, 65, 255), (2000, 97, 257),
                                    (30001, 30001, 131)])
def test_odd_particles_and_modes(orc, precision, tol, N, nq, P):
    run(orc, precision, tol, N, nq, P, None)


@pytest.mark.parametrize("precision,tol", [("fp32_comp", 2e-6), ("fp32", 2e-5)])
@pytest.mark.parametrize("N,P,tile", [(170001, 200, 256), (160003, 57, 256), (312001, 33, 512)])
def test_tiles_shared_by_a_block(orc, precision, tol, N, P, tile):
    """Long tiles in numbers that do not fill the last block's."""
    run(orc, precision, tol, N, N, P, tile)


def run(orc, precision, tol, N, nq, P, tile):
    build.build()
    sy = synth.make_system(N, density=0.02, frac_charged=0.0, seed=31)
    rng = np.random.default_rng(7)
    q = np.where(np.arange(nq) % 2, 1.0, -1.0)  # neutral, of an odd number: -1, 1, ..., 2, -1
    q[1] = 2.0
    sy.q[rng.permutation(N)[:nq]] = q
    r_core, r_s, p, seed, step = 2.7, 5.0, 4, 3, 2
    with binding.from_system(sy, P=P, alpha=ALPHA, r_c=r_s, r_core=r_core, p_rbl=p, seed=seed,
                             precision=precision) as h:
        if tile:
            h.set_tuning("sf_tile", tile)
        F, _, _ = h.forces_f64(step)
        rho, m = h.rho()
        _, S = h.sample_k(step)
    assert rel_l2(rho, orc.rho(sy.s, sy.q, sy.box, m)) < tol
    if tile:
        return
    ref = orc.rbl(sy.s, sy.q, sy.types, sy.box, ALPHA, r_core, r_s, p, seed, step, 0, C, sy.eps,
                  sy.sig)
    Fk, _, _ = orc.rbe_kspace(sy.s, sy.q, sy.box, ALPHA, C, m, S)
    assert rel_l2(F, ref["F"] + Fk) < 1e-5
