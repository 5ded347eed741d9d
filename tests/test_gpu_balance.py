"""Body force against bond force in the FP64 forms (GPU only): where b = -F / V exactly, the sum is formed before it
meets dt / rho, so a body at rest stays at rest, bit for bit, whatever dt / rho rounds to.

With dt = rho = 1 one step from rest leaves v = F / V itself, the value that the second run then balances."""
import numpy as np
import pytest

from paper_2309_11273_gb300 import PD_NONLINEAR, Simulation
from paper_2309_11273_gb300 import _binding as B
from paper_2309_11273_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _body(dim, rho, dt, b):
    dx = 1e-3
    if dim == 2:
        x, y = W.grid_2d(23, 15, dx)
        z, model = None, W.MODEL_PLANE_STRESS
    else:
        x, y, z = W.grid_3d(11, 7, 6, dx)
        model = W.MODEL_3D
    u0 = np.random.default_rng(9).normal(0.0, 1e-6, (dim, x.size))
    return W.Workload("body", model, E=30e9, nu=0.2, rho=rho, dx=dx, delta=3.015 * dx, dt=dt, nsteps=1, x=x, y=y, z=z,
                      vol=np.full(x.size, dx ** dim), u0=u0, b=b)


@pytest.mark.parametrize("options", [{}, {"bond_cache": 0}, {"kinematics": PD_NONLINEAR},
                                     {"kinematics": PD_NONLINEAR, "pairs": 0}, {"kinematics": PD_NONLINEAR, "bond_cache": 0}])
@pytest.mark.parametrize("resident", [1, 0])
@pytest.mark.parametrize("dim", [2, 3])
def test_a_balanced_body_stays_at_rest(dim, resident, options):
    sim = Simulation(_body(dim, 1.0, 1.0, None), s0=0.0, **options)
    sim.set_option(B.PD_OPT_RESIDENT, resident)
    sim.step(1)
    f = sim.state()[1]
    sim.close()
    assert np.abs(f).min() > 0.0
    w = _body(dim, 2411.7, 1.3e-7, -f)
    sim = Simulation(w, s0=0.0, **options)
    sim.set_option(B.PD_OPT_RESIDENT, resident)
    sim.step(1)
    u, v, _ = sim.state()
    sim.close()
    assert np.array_equal(v, np.zeros_like(v))
    assert np.array_equal(u, w.u0)
