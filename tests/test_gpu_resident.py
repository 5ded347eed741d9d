"""The resident step kernel (bodies that fit the chip in one wave) against the pass kernels, which a
chosen launch mapping selects: bitwise the same states, damage and bond status at the edges of its sizes
and forms, with breaking, reads between steps, constraints, uneven volumes and batches; its bounded
barrier wait (GPU only)."""
import numpy as np
import pytest

from paper_2309_11273_gb300 import PD_MIXED, PD_NONLINEAR, PD_W_INV, BatchSimulation, PDError, Simulation
from paper_2309_11273_gb300 import _binding as B
from paper_2309_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pass_kernels(sim):
    sim.set_option(B.PD_OPT_BLOCK, 128)
    return sim


def _run(sim, chunks):
    out = []
    for k in chunks:
        sim.step(k)
        out += list(sim.state())
    out += [sim.damage(), sim.neighbors()[2]]
    sim.close()
    return out


def _same(make, chunks):
    for x, y in zip(_run(make(), chunks), _run(_pass_kernels(make()), chunks)):
        assert np.array_equal(x, y)


def _plate(nx, ny, ratio=3.015):
    w = W.cracked_plate(nx=nx, ny=ny, ratio=ratio, crack_cells=nx // 2 + 0.125)
    w.u0 = np.random.default_rng(3).normal(0.0, 2e-9, (2, w.n))
    w.u0[1] += 4e-4 * (w.y - 0.5 * w.y.max())  # near the critical stretch: bonds break from the first steps
    return w


# particles: one slice, a ragged one, each side of four and of two warps per slice, the largest resident
# bodies (768-thread blocks) and the first beyond them
@pytest.mark.parametrize("nx,ny", [(5, 4), (11, 8), (40, 40), (139, 140), (180, 110), (221, 220), (250, 256), (341, 340),
                                   (350, 340)])
def test_plates_are_bitwise_the_pass_kernels(nx, ny):
    _same(lambda: Simulation(_plate(nx, ny)), [1, 2, 30, 17])


@pytest.mark.parametrize("shape", [(9, 7, 5), (24, 12, 10), (40, 25, 20), (61, 30, 25), (40, 38, 32), (40, 38, 33)])
def test_blocks_are_bitwise_the_pass_kernels(shape):
    def make():
        w = W.notched_block(*shape, nsteps=300, seed=5, amp=2e-8)
        return Simulation(w)
    _same(make, [1, 25, 24])


def test_uneven_volumes_and_impact():
    def cloud():
        rng = np.random.default_rng(11)
        x, y, z = W.grid_3d(30, 20, 18, 1e-3)
        x, y, z = (a + rng.uniform(-2e-4, 2e-4, a.size) for a in (x, y, z))
        w = W.Workload("cloud", W.MODEL_3D, dx=1e-3, delta=3.015e-3, dt=2e-7, nsteps=50, x=x, y=y, z=z,
                       vol=1e-9 * rng.uniform(0.5, 1.5, x.size), Gc=50.0, u0=rng.normal(0.0, 3e-7, (3, x.size)), **W.CONCRETE)
        return Simulation(w)
    _same(cloud, [3, 40])
    _same(lambda: Simulation(W.kalthoff(nx=120, ny=61, notch_cells=30.125, gap_cells=30)), [50, 51])


def test_batches_and_relaxation():
    _same(lambda: BatchSimulation(W.plate_batch(nplates=9, side_hi=90)), [60, 40])

    def static():
        x, y, z = W.grid_3d(30, 12, 10, 1e-3)
        flag = np.where(x < 3e-3, 1, 0).astype(np.uint8)
        b = np.zeros((3, x.size))
        b[2] = -2e6
        w = W.Workload("static", W.MODEL_3D, dx=1e-3, delta=3.015e-3, dt=1.0, nsteps=0, x=x, y=y, z=z,
                       vol=np.full(x.size, 1e-9), flag=flag, b=b, **W.CONCRETE)
        sim = Simulation(w, s0=0.0)
        sim.set_option(B.PD_OPT_SOLVER, B.PD_SOLVER_ADR)
        return sim
    _same(static, [1, 40, 59])


# the mixed form on the lattice layout: one slice, ragged ones, rows in shared memory and through L2 (48- and
# 124-slot rows on many slices), 512- and 768-thread blocks, the largest resident body and the first beyond
@pytest.mark.parametrize("lo", [0, 1])
@pytest.mark.parametrize("nx,ny,ratio", [(5, 5, 3.015), (11, 8, 3.015), (40, 40, 4.015), (279, 278, 3.015),
                                         (290, 280, 3.015), (341, 340, 4.015), (350, 340, 3.015)])
def test_mixed_plates_are_bitwise_the_pass_kernels(nx, ny, ratio, lo):
    def make():
        sim = Simulation(_plate(nx, ny, ratio), precision=PD_MIXED, shadow_lo=lo)
        assert sim.get_option(B.PD_OPT_LATTICE) == 1
        return sim
    _same(make, [1, 2, 30, 17])


@pytest.mark.parametrize("influence", [0, PD_W_INV])
@pytest.mark.parametrize("shape", [(9, 7, 5), (33, 12, 10), (61, 30, 35), (64, 45, 40)])
def test_mixed_blocks_are_bitwise_the_pass_kernels(shape, influence):
    def make():
        w = W.notched_block(*shape, nsteps=300, seed=5, amp=2e-8, dt=2.5e-7)
        return Simulation(w, precision=PD_MIXED, influence=influence)
    _same(make, [1, 25, 24])


@pytest.mark.parametrize("lo", [0, 1])
@pytest.mark.parametrize("shape", [(7, 5), (40, 40), (279, 278), (341, 340), (350, 340), (9, 7, 5), (33, 12, 10), (61, 30, 35),
                                   (64, 45, 40)])
def test_mixed_nonlinear_bodies_are_bitwise_the_pass_kernels(shape, lo):
    def make():
        w = _plate(*shape) if len(shape) == 2 else W.notched_block(*shape, nsteps=300, seed=5, amp=2e-8)
        return Simulation(w, precision=PD_MIXED, kinematics=PD_NONLINEAR, shadow_lo=lo)
    _same(make, [1, 25, 24])


def test_mixed_impact_and_batch():
    _same(lambda: Simulation(W.kalthoff(nx=120, ny=61, notch_cells=30.125, gap_cells=30), precision=PD_MIXED), [50, 51])
    _same(lambda: BatchSimulation(W.plate_batch(nplates=9, side_hi=90), precision=PD_MIXED), [60, 40])


def test_contexts_on_their_own_streams_and_threads():
    """Two FP64 and one mixed context, each with its own stream, step from three threads at once (every grid
    wants the whole chip): all end with the state of a run alone."""
    import threading
    makes = [lambda: Simulation(_plate(200, 120)), lambda: Simulation(_plate(90, 60)),
             lambda: Simulation(_plate(230, 160), precision=PD_MIXED)]
    alone = []
    for mk in makes:
        sim = mk()
        sim.step(400)
        alone.append(sim.state()[0])
        sim.close()
    sims, got = [mk() for mk in makes], [None] * 3

    def work(k):
        for _ in range(8):
            sims[k].step(50)
        got[k] = sims[k].state()[0]
    threads = [threading.Thread(target=work, args=(k,)) for k in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, g in zip(alone, got):
        assert g is not None and np.array_equal(a, g)


def test_switching_between_the_kernels_keeps_the_run():
    ref = Simulation(_plate(90, 60))
    ref.step(120)
    sim = Simulation(_plate(90, 60))
    sim.step(40)
    _pass_kernels(sim).step(40)
    assert B.pd_autotune(sim.h, 2)[0] > 0
    sim.step(40)
    for x, y in zip(list(sim.state()) + [sim.damage()], list(ref.state()) + [ref.damage()]):
        assert np.array_equal(x, y)


def test_expired_barrier_reports_timeout_and_the_context_recovers():
    w = _plate(60, 40)
    sim = Simulation(w)
    sim.set_option(B.PD_OPT_EXPIRE_WAITS, 1)  # block 0 never arrives: every wait runs out
    sim.step(3)
    with pytest.raises(PDError) as e:
        sim.sync()
    assert e.value.status == B.PD_ERR_TIMEOUT
    sim.set_option(B.PD_OPT_EXPIRE_WAITS, 0)
    B.pd_build_neighbors(sim.h, w.cracks)
    B.pd_set_bc(sim.h, 2, w.n, None, w.b)
    sim.set_state(w.u0)
    sim.step(50)
    ref = Simulation(w)
    ref.step(50)
    assert np.array_equal(sim.state()[0], ref.state()[0])


def _run_unread(sim, calls):
    for k in calls:
        sim.step(k)
    out = list(sim.state()) + [sim.damage(), sim.neighbors()[2]]
    sim.close()
    return out


def _same_unread(make, calls):
    res, ref = _run_unread(make(), calls), _run_unread(_pass_kernels(make()), calls)
    assert (ref[-1] == 0).any()  # bonds broke
    for x, y in zip(res, ref):
        assert np.array_equal(x, y)


# The first step of a call that follows an unread one checks its bonds, and so does each launch of a call longer
# than one launch (1000 steps): the intact sums a call starts from and the marks of its first check must not mix.
# (40, 40): without the pair form; the others with it, at four, two and one warps per slice
@pytest.mark.parametrize("nx,ny,ratio", [(40, 40, 3.015), (138, 140, 4.015), (200, 200, 3.015), (341, 340, 3.015)])
@pytest.mark.parametrize("calls", [[1, 1, 1, 2, 3, 12], [1, 1100]])
def test_unread_calls_on_breaking_plates(nx, ny, ratio, calls):
    _same_unread(lambda: Simulation(_plate(nx, ny, ratio)), calls)


@pytest.mark.parametrize("shape", [(9, 7, 5), (30, 25, 24), (40, 38, 32)])
def test_unread_calls_on_breaking_blocks(shape):
    _same_unread(lambda: Simulation(W.notched_block(*shape, nsteps=100, seed=5, amp=2e-8)), [1, 1, 2, 1, 40, 55])


@pytest.mark.parametrize("kinematics", [0, PD_NONLINEAR])
@pytest.mark.parametrize("nx,ny", [(40, 40), (341, 340)])
def test_unread_calls_on_breaking_mixed_plates(nx, ny, kinematics):
    _same_unread(lambda: Simulation(_plate(nx, ny), precision=PD_MIXED, kinematics=kinematics), [1, 1, 1, 2, 3, 12, 30])


@pytest.mark.parametrize("first", ["sync", "state", "damage", "stats", "neighbors", "check_state", "autotune", "save"])
def test_an_expired_barrier_loses_the_state(first, tmp_path):
    """The first call that meets it reports the timeout; then nothing reads or steps the state until there is a new
    one (a checkpoint brings back the bond status too)."""
    w = _plate(60, 40)
    ckpt = str(tmp_path / "before")
    ref = Simulation(w, precision=PD_MIXED if first == "state" else 0)
    ref.step(30)
    ref.save_state(ckpt)
    ref.step(20)
    sim = Simulation(w, precision=PD_MIXED if first == "state" else 0)
    sim.set_option(B.PD_OPT_EXPIRE_WAITS, 1)
    sim.step(3)
    calls = {"sync": sim.sync, "state": sim.state, "damage": sim.damage, "stats": sim.stats, "neighbors": sim.neighbors,
             "check_state": lambda: B._check(B.pd_check_state(sim.h, 1.0)), "autotune": lambda: B.pd_autotune(sim.h, 1),
             "save": lambda: sim.save_state(str(tmp_path / "lost")), "step": lambda: sim.step(1)}
    with pytest.raises(PDError) as e:
        calls[first]()
    assert e.value.status == B.PD_ERR_TIMEOUT
    sim.set_option(B.PD_OPT_EXPIRE_WAITS, 0)
    for name, call in calls.items():
        if name == "sync":
            call()
            continue
        with pytest.raises(PDError) as e:
            call()
        assert e.value.status == B.PD_ERR_STATE, name
    sim.load_state(ckpt)
    sim.step(20)
    for x, y in zip(list(sim.state()) + [sim.damage()], list(ref.state()) + [ref.damage()]):
        assert np.array_equal(x, y)


def test_a_state_set_before_the_timeout_is_read_steps_all_the_same():
    w = W.plate_vibration(nx=40, ny=20, nsteps=20)
    sim = Simulation(w, s0=0.0)
    sim.set_option(B.PD_OPT_EXPIRE_WAITS, 1)
    sim.step(3)
    sim.set_option(B.PD_OPT_EXPIRE_WAITS, 0)
    sim.set_state(w.initial_u())
    sim.step(20)
    with pytest.raises(PDError) as e:
        sim.sync()
    assert e.value.status == B.PD_ERR_TIMEOUT
    ref = Simulation(w, s0=0.0)
    ref.step(20)
    for x, y in zip(sim.state(), ref.state()):
        assert np.array_equal(x, y)


def _last_path(sim, steps=2):
    sim.step(steps)
    return sim.get_option(B.PD_OPT_RESIDENT)


# which bodies run resident on the 152 SMs of a GB300: both sides of every limit of the plans (24, 20 and 16 warps per SM)
@pytest.mark.parametrize("nx,ny,want", [(5, 4, 1), (139, 140, 1), (221, 220, 1), (341, 340, 1), (350, 340, 0)])
def test_plates_take_the_kernel_that_the_plan_names(nx, ny, want):
    for kw in ({}, {"precision": PD_MIXED}, {"precision": PD_MIXED, "kinematics": PD_NONLINEAR}):
        sim = Simulation(_plate(nx, ny), **kw)
        assert sim.get_option(B.PD_OPT_RESIDENT) == 1  # the setting, before the first step
        assert _last_path(sim) == want, kw
        assert _last_path(_pass_kernels(sim)) == 0
        sim.close()


@pytest.mark.parametrize("shape,fp64,mixed", [((9, 7, 5), 1, 1), ((40, 38, 32), 1, 1), ((40, 38, 33), 0, 1), ((64, 45, 40), 0, 1),
                                              ((64, 48, 40), 0, 0)])
def test_blocks_take_the_kernel_that_the_plan_names(shape, fp64, mixed):
    for kw, want in (({}, fp64), ({"precision": PD_MIXED}, mixed), ({"kinematics": PD_NONLINEAR}, 0),
                     ({"precision": PD_MIXED, "kinematics": PD_NONLINEAR}, mixed)):
        sim = Simulation(W.notched_block(*shape), **kw)
        assert _last_path(sim) == want, kw
        sim.close()


@pytest.mark.parametrize("precision", [0, PD_MIXED])
def test_the_resident_option(precision):
    ref = Simulation(_plate(90, 60), precision=precision)
    assert _last_path(ref, 40) == 1
    sim = Simulation(_plate(90, 60), precision=precision)
    sim.set_option(B.PD_OPT_RESIDENT, 0)
    assert sim.get_option(B.PD_OPT_RESIDENT) == 0
    assert _last_path(sim, 20) == 0
    sim.set_option(B.PD_OPT_RESIDENT, 1)
    assert _last_path(sim, 20) == 1
    for x, y in zip(list(sim.state()) + [sim.damage()], list(ref.state()) + [ref.damage()]):
        assert np.array_equal(x, y)
    for opt in (B.PD_OPT_PROFILE, B.PD_OPT_SOLVER):
        sim.set_option(opt, 1)
        assert _last_path(sim) == 0
        sim.set_option(opt, 0)
        assert _last_path(sim) == 1


@pytest.mark.parametrize("precision", [0, PD_MIXED])
def test_a_callers_capture_takes_the_pass_kernels(precision):
    import torch
    stream = torch.cuda.Stream()
    ref = Simulation(_plate(90, 60), precision=precision)
    ref.step(10)
    sim = Simulation(_plate(90, 60), precision=precision, stream=stream.cuda_stream)
    assert _last_path(sim, 2) == 1
    sim.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        sim.step(8)
    assert sim.get_option(B.PD_OPT_RESIDENT) == 0
    with torch.cuda.stream(stream):
        g.replay()
    for x, y in zip(list(sim.state()) + [sim.damage()], list(ref.state()) + [ref.damage()]):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("offset", [1, 511])
def test_a_read_into_arrays_that_share_their_pages(offset):
    """pd_get_state brings the pages of large output arrays in while the GPU still steps: what else lies on the first
    and last page stays as it was."""
    w = W.notched_block(60, 60, 60)
    ref = Simulation(w, precision=PD_MIXED)
    ref.step(40)
    want = ref.state()[0]
    sim = Simulation(w, precision=PD_MIXED)
    buf = np.full(3 * w.n + 1024, -7.5)
    u = buf[offset:offset + 3 * w.n].reshape(3, w.n)
    sim.step(40)
    B.pd_get_state(sim.h, 3, w.n, u=u, v=False, theta=False)
    assert np.array_equal(u, want)
    assert (buf[:offset] == -7.5).all() and (buf[offset + 3 * w.n:] == -7.5).all()
