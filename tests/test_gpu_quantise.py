"""rbe_set_positions stores s = rint(fl(r / L) 2^32) mod 2^32 for every position, whichever way the
kernel forms it: inside the box, on the grid, at halves of the grid (the rounding's ties), at and
past the edges, negative, tiny. Edges of the box with all kinds of significands."""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box", [(32.0, 64.0, 33.3), (27.1, 218.87756, 271.0), (1000.1, 25.7, 90.0)])
def test_positions_quantise_as_the_definition(box):
    build.build()
    n = 6000
    sy = synth.make_system(n, L=30.0, seed=1)
    sy.box = np.array(box)
    rng = np.random.default_rng(2)
    s = rng.integers(0, 2 ** 32, (n, 3)).astype(np.float64)
    frac = np.where(rng.random((n, 3)) < 0.4, s / 2 ** 32, rng.random((n, 3)))
    frac[: n // 8] = (s[: n // 8] + 0.5) / 2 ** 32
    pos = frac * sy.box
    pos[n // 2:] += rng.integers(-2, 3, (n - n // 2, 1)) * sy.box
    edge = np.array([0.0, -0.0, 1e-300, -1e-12, 0.5, 1.0, 1.5, -1.0])
    pos[: edge.size] = edge[:, None] * sy.box
    pos[edge.size] = np.nextafter(sy.box, 0)
    with binding.from_system(sy, P=4, alpha=0.09, r_c=10.0) as h:
        h.set_positions(pos)
        _, _, got = h.state()
    f = (pos / sy.box) * 4294967296.0
    fm = f - 4294967296.0 * np.floor(f / 4294967296.0)
    assert np.array_equal(got, (np.rint(fm).astype(np.uint64) & 0xFFFFFFFF).astype(np.uint32))
