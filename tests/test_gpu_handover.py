"""Positions in and results out, through every kind of memory, on both sides of the size up to which
kernels write host memory themselves: the same numbers, whichever way they travel."""
import numpy as np
import pytest

from paper_2609_02694_gb300 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32_comp", "fp64"])
@pytest.mark.parametrize("N", [501, 8192, 8193, 60000])
def test_every_memory_gives_the_same(N, precision):
    import torch
    build.build()
    sy = synth.make_system(N, density=0.02, seed=5)
    with binding.from_system(sy, P=8, alpha=0.09, r_c=10.0, precision=precision) as h:
        pos = sy.positions()
        pos[0] += sy.box  # (a wrapped one)
        wide = torch.from_numpy(np.concatenate([np.zeros(3), pos.ravel()]))
        kinds = [pos, torch.from_numpy(pos), torch.from_numpy(pos).pin_memory(),
                 wide.pin_memory()[3:], torch.from_numpy(pos).cuda(), wide.cuda()[3:]]
        outs = [np.zeros((N, 3), np.float32), torch.zeros(N, 3), torch.zeros(N, 3).pin_memory(),
                torch.zeros(3 * N + 1).pin_memory()[1:], torch.zeros(N, 3, device="cuda"),
                torch.zeros(3 * N + 1, device="cuda")[1:]]
        ref = None
        for p, out in zip(kinds, outs):
            h.set_positions(np.zeros((N, 3)) + 1.0)  # (elsewhere first)
            h.set_positions(p)
            x, v, s = h.state()
            assert np.array_equal(s, sy.s)
            assert np.array_equal(x, sy.s.astype(np.float64) * (sy.box / synth.TWO32))
            assert np.array_equal(v, sy.v if precision == "fp64" else sy.v.astype(np.float32))
            for energies in (False, True):
                F = h.forces(3, out=out, energies=energies)
                e = None
                if energies:
                    F, e, w = F
                torch.cuda.synchronize()
                F = np.array(F if isinstance(F, np.ndarray) else F.cpu().numpy()).reshape(N, 3)
                if ref is None:
                    ref = F
                    assert np.abs(F).max() > 0
                assert np.array_equal(F, ref)
                if energies:
                    last = e if p is pos else last
                    assert e == last
