"""Pass 1a of the nonlinear FP64 pair form on both sides of its series' range (|Y|^2 - |xi|^2 = 2^-8 |xi|^2),
against the oracle (GPU only).

One step from rest leaves v = dt F / rho, the force itself.  Every bond's term is within a few units of
2^-53 of its exact value on either side of the range, and a force sums at most 122 of them, so v is held to
the parity bar of 1e-12 of its largest value (tests/parity.py), and theta likewise."""
import numpy as np
import pytest

import oracle as O
from paper_2309_11273_gb300 import PD_NONLINEAR, PDError, Simulation
from paper_2309_11273_gb300._binding import PD_ERR_NUMERIC
from paper_2309_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _body(dim, uniform, rng):
    dx = 1e-3
    if dim == 2:
        x, y = W.grid_2d(37, 9, dx)
        z, model = None, W.MODEL_PLANE_STRESS
    else:
        x, y, z = W.grid_3d(35, 7, 6, dx)
        model = W.MODEL_3D
    vol = np.full(x.size, dx ** dim)
    if not uniform:
        vol = vol * rng.uniform(0.7, 1.3, x.size)
    return W.Workload("body", model, E=30e9, nu=0.2, rho=2400.0, dx=dx, delta=3.015 * dx, dt=1e-7, nsteps=1, x=x,
                      y=y, z=z, vol=vol)


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("stretch", [0.0, 1e-9, 1.9e-3, 1.95e-3, 2.0e-3, -1.97e-3, 0.3, -0.4])
def test_extension_series_and_its_range(dim, uniform, stretch):
    rng = np.random.default_rng(7)
    w = _body(dim, uniform, rng)
    X = np.stack([w.x, w.y] if dim == 2 else [w.x, w.y, w.z])
    # a uniform stretch (every bond at t = 2 s + s^2) with a part that spreads the bonds around it
    w.u0 = stretch * X + rng.normal(0.0, 1e-9 + 2e-2 * abs(stretch) * w.dx, X.shape)
    sim = Simulation(w, s0=0.0, kinematics=PD_NONLINEAR)
    ref = O.OracleSim(w.model, w.E, w.nu, w.rho, w.delta, 0.0, w.dt, w.x, w.y, w.z, w.vol, w.cracks, kin=O.NONLINEAR)
    ref.set_state(w.u0, w.initial_v())
    ref.step(1)
    sim.step(1)
    u, v, theta = sim.state()
    sim.close()
    assert np.abs(v - ref.v).max() <= 1e-12 * np.abs(ref.v).max()
    assert np.abs(u - ref.u).max() <= 1e-12 * np.abs(ref.u).max()
    assert np.abs(theta - ref.theta).max() <= 1e-12 * np.abs(ref.theta).max()


@pytest.mark.parametrize("uniform", [True, False])
@pytest.mark.parametrize("dim", [2, 3])
def test_two_particles_at_one_place(dim, uniform):
    """A bond of no length: once its ends have moved apart its extension is |Y| and it pulls along Y, as the single
    pass (PD_OPT_PAIRS 0), which tables no 1/|xi|, has it; at rest the state has no direction for it and the run is
    reported as non-finite in both forms.  The same bars as above."""
    rng = np.random.default_rng(5)
    w = _body(dim, uniform, rng)
    for k, j in ((3, 4), (40, 39), (100, 137)):  # in one slice and across two
        w.x[k], w.y[k] = w.x[j], w.y[j]
        if dim == 3:
            w.z[k] = w.z[j]
    w.u0 = rng.normal(0.0, 1e-6, (dim, w.n))
    got = []
    for pairs in (1, 0):
        sim = Simulation(w, s0=0.0, kinematics=PD_NONLINEAR, pairs=pairs)
        sim.step(1)
        got.append(sim.state())
        sim.set_state(np.zeros((dim, w.n)))
        sim.step(1)
        with pytest.raises(PDError) as e:
            sim.sync()
        assert e.value.status == PD_ERR_NUMERIC
        sim.close()
    for x, y in zip(*got):
        assert np.abs(x - y).max() <= 1e-12 * np.abs(y).max()
