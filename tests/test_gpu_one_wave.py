"""FP64 plates of 32 to 36 warps per SM at one or two warps per slice, which the pass kernels take in one wave with 56 registers:
bitwise the other mappings' states on both sides of the range, with breaking, uneven volumes, both forms of pass 1 and
reads between steps (GPU only)."""
import numpy as np
import pytest

from paper_2309_11273_gb300 import Simulation
from paper_2309_11273_gb300 import _binding as B
from paper_2309_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _plate(nx, ny, uneven=False):
    w = W.cracked_plate(nx=nx, ny=ny, crack_cells=nx // 2 + 0.125)
    w.u0 = np.random.default_rng(3).normal(0.0, 2e-9, (2, w.n))
    w.u0[1] += 4e-4 * (w.y - 0.5 * w.y.max())  # near the critical stretch: bonds break from the first steps
    if uneven:
        w.vol = w.vol * (1.0 + 0.2 * (np.arange(w.n) % 3))
    return w


def _run(w, options, **kw):
    sim = Simulation(w, **kw)
    for opt, value in options:
        sim.set_option(opt, value)
    out = []
    for k in (1, 2, 30, 7):
        sim.step(k)
        if k != 2:
            out += list(sim.state())
    path = sim.get_option(B.PD_OPT_RESIDENT)
    out += [sim.damage(), sim.neighbors()[2]]
    sim.close()
    return path, out


# 2,416 slices (the last resident plate), 2,433, 2,736 (the last of the range) and 2,757
@pytest.mark.parametrize("nx,ny,resident", [(278, 278, 1), (279, 279, 0), (288, 304, 0), (297, 297, 1)])
@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("pairs", [1, 0])
def test_plates_of_one_tight_wave(nx, ny, resident, uneven, pairs):
    w = _plate(nx, ny, uneven)
    path, want = _run(w, [], pairs=pairs)
    assert path == (resident if pairs else 0)
    assert (want[-1] == 0).any()  # bonds broke
    for options in ([(B.PD_OPT_RESIDENT, 0)], [(B.PD_OPT_BLOCK, 64), (B.PD_OPT_SPLIT, 2)],
                    [(B.PD_OPT_BLOCK, 128), (B.PD_OPT_SPLIT, 2)], [(B.PD_OPT_BLOCK, 256)],
                    [(B.PD_OPT_BLOCK, 512), (B.PD_OPT_SPLIT, 2)]):
        path, got = _run(w, options, pairs=pairs)
        assert path == 0
        for x, y in zip(got, want):
            assert np.array_equal(x, y), options


# the same with one warp per slice: 4,864 slices (the last with 64 registers in one wave), 4,901, 5,472 and 5,487
@pytest.mark.parametrize("nx,ny", [(304, 512), (396, 396), (342, 512), (419, 419)])
@pytest.mark.parametrize("uneven", [False, True])
def test_plates_of_one_tight_wave_with_one_warp_per_slice(nx, ny, uneven):
    w = _plate(nx, ny, uneven)
    _, want = _run(w, [])
    assert (want[-1] == 0).any()
    for options in ([(B.PD_OPT_BLOCK, 64)], [(B.PD_OPT_BLOCK, 128)], [(B.PD_OPT_BLOCK, 256)]):
        _, got = _run(w, options)
        for x, y in zip(got, want):
            assert np.array_equal(x, y), options
