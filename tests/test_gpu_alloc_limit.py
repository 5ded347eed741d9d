"""A step whose device allocations fail (PD_OPT_DEVICE_LIMIT stands for a full device): it reports PD_ERR_OOM, so
does the next one, the state stays as it was, and once there is room the run is bitwise that of a context that
always had it (GPU only)."""
import numpy as np
import pytest

from paper_2309_11273_gb300 import PD_FP64, PD_LINEARIZED, PD_MIXED, PD_NONLINEAR, PDError, Simulation
from paper_2309_11273_gb300 import _binding as B
from paper_2309_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _sim(dim, kinematics, solver):
    if dim == 3:
        w = W.notched_block(12, 8, 7, nsteps=100, seed=5, amp=2e-8)
        w.flag = w.axis_point = w.axis_dir = None
    else:
        w = W.cracked_plate(nx=40, ny=30, crack_cells=20.125)
        w.u0 = np.random.default_rng(3).normal(0.0, 2e-9, (2, w.n))
    sim = Simulation(w, kinematics=kinematics, s0=0.0 if solver else None)
    sim.set_option(B.PD_OPT_SOLVER, solver)
    return sim


def _bytes(sim):
    return B.pd_get_info(sim.h)[2]


def _full_run(make):
    """(device bytes before the first step, after six steps and a read, the state)."""
    ref = make()
    b0 = _bytes(ref)
    ref.step(6)
    want = ref.state()
    b1 = _bytes(ref)
    ref.close()
    return b0, b1, want


@pytest.mark.parametrize("solver", [B.PD_SOLVER_EXPLICIT, B.PD_SOLVER_ADR])
@pytest.mark.parametrize("dim,kinematics", [(2, PD_LINEARIZED), (3, PD_LINEARIZED), (2, PD_NONLINEAR), (3, PD_NONLINEAR)])
def test_a_failed_allocation_leaves_nothing_half_built(dim, kinematics, solver):
    def make():
        return _sim(dim, kinematics, solver)
    b0, b1, want = _full_run(make)
    refused = 0
    for part in np.linspace(0.0, 1.0, 13)[:-1]:
        sim = make()
        u0 = sim.state()[0]
        sim.set_option(B.PD_OPT_DEVICE_LIMIT, int(b0 + part * (b1 - b0)))
        try:
            sim.step(6)
        except PDError as e:
            assert e.status == B.PD_ERR_OOM
            refused += 1
            with pytest.raises(PDError) as again:
                sim.step(6)
            assert again.value.status == B.PD_ERR_OOM
            assert np.array_equal(sim.state()[0], u0)
            sim.set_option(B.PD_OPT_DEVICE_LIMIT, 0)
            sim.step(6)
            for x, y in zip(sim.state(), want):
                assert np.array_equal(x, y)
        sim.close()
    assert refused > 0


@pytest.mark.parametrize("dim", [2, 3])
def test_nonlinear_bodies_take_the_single_pass_where_the_pair_tables_do_not_fit(dim):
    b0, b_pair, _ = _full_run(lambda: _sim(dim, PD_NONLINEAR, B.PD_SOLVER_EXPLICIT))

    def single():
        sim = _sim(dim, PD_NONLINEAR, B.PD_SOLVER_EXPLICIT)
        sim.set_option(B.PD_OPT_PAIRS, 0)
        return sim
    _, b_single, want = _full_run(single)
    # 120 and 48 bytes per slot: neither form holds the other's tables
    assert 2.4 * (b_single - b0) < b_pair - b0 < 2.6 * (b_single - b0)
    for limit in (b_single, (b_single + b_pair) // 2, b_pair - 1):
        sim = _sim(dim, PD_NONLINEAR, B.PD_SOLVER_EXPLICIT)
        sim.set_option(B.PD_OPT_DEVICE_LIMIT, limit)
        sim.step(6)
        for x, y in zip(sim.state(), want):
            assert np.array_equal(x, y)
        assert sim.get_option(B.PD_OPT_PAIRS) == 0
        sim.close()


@pytest.mark.parametrize("read", [False, True])
def test_switching_the_nonlinear_form_when_only_one_fits(read):
    _, b_pair, _ = _full_run(lambda: _sim(3, PD_NONLINEAR, B.PD_SOLVER_EXPLICIT))
    out = []
    for limit in (0, b_pair):
        sim = _sim(3, PD_NONLINEAR, B.PD_SOLVER_EXPLICIT)
        sim.set_option(B.PD_OPT_DEVICE_LIMIT, limit)
        for pairs in (1, 0, 1, 0):
            sim.step(3)
            sim.set_option(B.PD_OPT_PAIRS, pairs)
            if read:
                sim.damage()  # the pending check, in the form just chosen
            sim.step(2)
            assert sim.get_option(B.PD_OPT_PAIRS) == pairs
        out.append(list(sim.state()) + [sim.damage()])
        sim.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("precision", [PD_FP64, PD_MIXED])
def test_no_room_for_the_resident_kernels_barrier(precision):
    def make():
        w = W.cracked_plate(nx=40, ny=30, crack_cells=20.125)
        return Simulation(w, precision=precision)
    ref = make()
    ref.step(6)
    want = ref.state()
    sim = make()
    sim.set_option(B.PD_OPT_PROFILE, 1)  # the pass kernels: every table, no barrier yet
    sim.step(1)
    sim.set_option(B.PD_OPT_PROFILE, 0)
    sim.set_option(B.PD_OPT_DEVICE_LIMIT, _bytes(sim))
    sim.step(5)
    for x, y in zip(sim.state(), want):
        assert np.array_equal(x, y)


def test_a_switched_nonlinear_form_may_be_captured_at_once():
    import torch
    stream = torch.cuda.Stream()

    def make(**kw):
        w = W.notched_block(12, 8, 7, nsteps=100, seed=5, amp=2e-8)
        w.flag = w.axis_point = w.axis_dir = None
        return Simulation(w, kinematics=PD_NONLINEAR, **kw)
    ref, sim = make(), make(stream=stream.cuda_stream)
    for s in (ref, sim):
        s.step(2)
        s.set_option(B.PD_OPT_PAIRS, 0)
    ref.step(4)
    sim.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        sim.step(4)
    with torch.cuda.stream(stream):
        g.replay()
    for x, y in zip(sim.state(), ref.state()):
        assert np.array_equal(x, y)
