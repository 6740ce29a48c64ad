"""Relaxation times so long that 1 - 1/tau rounds to 1 in the arithmetic type: the state stays finite,
and a body force still accelerates the fluid by g per step (walls far from the middle layer)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tau", [("fp64", 1e17), ("fp32", 1e9), ("fp16", 1e9), ("bf16", 1e9)])
def test_force_without_relaxation(precision, tau):
    from paper_2305_18919_gb300 import binding
    nx, ny, nz = 8, 8, 24
    g = 2.0 ** -12  # exact in every type
    lat = binding.Lattice(nx, ny, nz, tau, 1.0, (0, 0, 0), (0, 0, 0), (g, 0, 0), precision, True)
    lat.step(4)
    rho, u = lat.fields()
    # with periodic z the flow is uniform: u = n g + g / 2 after n steps, to the storage's rounding of
    # four updates, half a last place of the momentum each
    eps = {"fp64": 2.0 ** -52, "fp32": 2.0 ** -23, "fp16": 2.0 ** -10, "bf16": 2.0 ** -7}[precision]
    assert np.isfinite(rho).all()
    assert np.abs(u[..., 0] - 4.5 * g).max() <= 4 * eps * 4.5 * g
    lat.close()
