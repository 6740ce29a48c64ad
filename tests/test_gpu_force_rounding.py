"""A weak body force in FP32 over many steps: the force is added with its own precision, not with that
of the momentum it is added to. u against the FP64 oracle.

The bound: each population's update rounds about three times at no more than its size, 3 w |u| <
3.4e-4 / 2 for |u| < 1e-3 .. 2e-3, so by 1e-11; the 18 moving ones leave a node's momentum with noise of
about sqrt(54) 1e-11 = 7e-11 a step, 500 independent steps with 1.6e-9, against |u| of about 1e-3: 1.6e-6
with no step undone. The collisions and the viscosity undo most of it; half of that is allowed. (A force
rounded into the momentum errs the same way every step: 500 times a few 1e-11.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,tau,g", [((24, 20, 18), 0.9, (2e-6, 0.0, 0.0)),
                                         ((36, 28, 31), 0.73, (1e-6, -1.5e-6, 0.0))])
def test_force_in_float_over_many_steps(shape, tau, g):
    import oracle
    from paper_2305_18919_gb300 import binding
    nx, ny, nz = shape
    x, y = (2 * np.pi * np.arange(n) / n for n in (nx, ny))
    z = np.pi * (np.arange(nz) - 0.5) / (nz - 2)
    env = np.sin(z)[:, None, None]
    u = np.zeros((nz, ny, nx, 3))
    u[..., 0] = 1e-3 * env * np.sin(y + 0.3)[None, :, None] * np.cos(2 * z + 0.5)[:, None, None]
    u[..., 1] = 1e-3 * env * np.sin(x + 1.3)[None, None, :]
    u[..., 2] = 1e-3 * env * np.sin(x + 0.9)[None, None, :] * np.cos(y + 0.2)[None, :, None]
    rho = 1 + 1e-4 * np.sin(x + 0.5)[None, None, :] * np.cos(y)[None, :, None] * env
    ref = oracle.Simulation(nx, ny, nz, tau, 1.0, (0, 0, 0), (0, 0, 0), g, False)
    lat = binding.Lattice(nx, ny, nz, tau, 1.0, (0, 0, 0), (0, 0, 0), g, "fp32")
    for s in (ref, lat):
        s.init_equilibrium(rho, u)
        s.step(500)
    want, got = ref.fields()[1][1:-1], lat.fields()[1][1:-1]
    assert np.linalg.norm(got - want) / np.linalg.norm(want) < 8e-7
    lat.close()
