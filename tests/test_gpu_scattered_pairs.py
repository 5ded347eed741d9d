"""Pass 1a of the linearized FP64 pair form on points off the lattice (GPU only): warps whose lanes start their owned
entries at many different slots walk them slot by slot, others lane by lane.  From a lattice, where few starts differ,
over jitters of the points that change ever more families, to scattered points: bitwise the single pass, with bonds
breaking and reads between steps, at every split and through the check before a read."""
import numpy as np
import pytest

from paper_2309_11273_gb300 import Simulation
from paper_2309_11273_gb300 import _binding as B
from paper_2309_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _body(dim, jitter):
    rng = np.random.default_rng(17)
    if dim == 3:
        w = W.notched_block(23, 14, 11, nsteps=100, seed=5, amp=2e-8)
        axes = (w.x, w.y, w.z)
    else:
        w = W.cracked_plate(nx=61, ny=43, crack_cells=30.125)
        w.u0 = rng.normal(0.0, 2e-9, (2, w.n))
        w.u0[1] += 4e-4 * (w.y - 0.5 * w.y.max())
        axes = (w.x, w.y)
    for a in axes:
        a += rng.uniform(-jitter, jitter, a.size) * w.dx
    return w


def _run(w, pairs, split):
    sim = Simulation(w, pairs=pairs)
    sim.set_option(B.PD_OPT_BLOCK, 128)
    sim.set_option(B.PD_OPT_SPLIT, split)
    out = []
    for k in (1, 2, 25, 40):
        sim.step(k)
        if k != 2:
            out += list(sim.state())
    out += [sim.damage(), sim.neighbors()[2]]
    sim.close()
    return out


@pytest.mark.parametrize("jitter", [0.0, 1e-3, 0.02, 0.1, 0.3])
@pytest.mark.parametrize("dim", [2, 3])
def test_scattered_points_are_bitwise_the_single_pass(dim, jitter):
    w = _body(dim, jitter)
    want = _run(w, 0, 1)
    assert (want[-1] == 0).any()  # bonds broke
    for split in (1, 2, 4):
        for x, y in zip(_run(w, 1, split), want):
            assert np.array_equal(x, y), split
