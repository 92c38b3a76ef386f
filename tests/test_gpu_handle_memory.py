"""Device memory a charged particle costs a handle: its arrays, and nothing beside them.

Coordinates 12 bytes, charge 4 (and 8 in FP64), slot 4, the structure factor's partials 16 P / 32;
over cells also the Coulomb pass's record 16 and partials 32 / 4.
"""
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.lib()


@pytest.mark.parametrize("kw,per", [(dict(precision="fp32_comp"), 48), (dict(precision="fp64"), 56),
                                    (dict(precision="fp32", r_core=5.0), 24),
                                    (dict(precision="fp64", r_core=5.0), 32)])
def test_bytes_a_charged_particle(kw, per):
    N, used = 64000, []
    for frac in (0.0, 1.0):
        sy = synth.make_system(N, density=0.1, seed=2, frac_charged=frac)
        with binding.from_system(sy, P=8, alpha=synth.ALPHA, r_c=synth.R_CUT, **kw) as h:
            used.append(h.memory_bytes())
    assert (used[1] - used[0]) / N == pytest.approx(per, rel=0.01)
