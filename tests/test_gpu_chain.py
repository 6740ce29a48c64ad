"""The interface passes at the edges of their shapes: source tiles with about as many vertices as a
bucket holds (128), below and above, and positions many periods outside the box or negative."""
import numpy as np
import pytest

from pairs import make_pair, rel_l2
from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu

# as in the spill tests: fine meshes sum hundreds of vertex forces per node
TOL = {"fp64": 1e-11, "fp32": 2e-6}


def _bases_per_tile(q):
    _, counts = np.unique((np.floor(q).astype(int) - 1) // 4, axis=0, return_counts=True)
    return counts


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("sub,radius,lo,hi", [(2, 4.0, 1, 64), (4, 6.5, 64, 128),
                                              (4, 5.5, 129, 160), (4, 3.4, 300, 400)])
def test_force_field_across_bucket_sizes(sub, radius, lo, hi, precision):
    a = tuple(0.01 * x for x in inputs.ALPHA_CLASSES["softly_coated"])
    wl = inputs.scaled_wetting(24, 20, sub, radius, a, 0.5 * 0.01, precision=precision, lift=2.0)
    ref, gpu = make_pair(wl, precision)
    v, _ = wl.mesh()
    c = v.mean(0)
    q = c + 1.005 * (inputs.perturb(v, 0.02, seed=3) - c)
    assert lo <= _bases_per_tile(q).max() <= hi
    ref.set_vertices(q)
    gpu.set_vertices(q)
    assert rel_l2(gpu.force_field(), ref.force_field()) < TOL[precision]
    for s in (ref, gpu):
        s.step(2)
    assert rel_l2(gpu.vertex_velocities(), ref.vertex_velocities()) < (
        1e-11 if precision == "fp64" else 1e-5)
    gpu.close()


@pytest.mark.parametrize("shift", [(-1, 0), (3, -2), (-1000, 4096), (2 ** 27, -2 ** 27)])
def test_unwrapped_positions(shift):
    """A mesh moved by whole periods in x and y moves with the flow in the same way."""
    a = tuple(0.01 * x for x in inputs.ALPHA_CLASSES["softly_coated"])
    wl = inputs.scaled_wetting(24, 20, 2, 4.0, a, 0.005, precision="fp64", lift=1.0)
    _, here = make_pair(wl, "fp64")
    d = np.array([shift[0] * wl.nx, shift[1] * wl.ny, 0.0])
    v, f = wl.mesh()
    from paper_2305_18919_gb300 import binding
    there = binding.Lattice.from_workload(wl, precision="fp64")
    q = inputs.perturb(v, 0.05, seed=8)
    q[:, :2] = np.round(q[:, :2] * 2 ** 16) / 2 ** 16  # exact after the shift as well
    here.set_vertices(q)
    there.set_vertices(q + d)
    # the interface forces see q - reference, which differs: off, so that only the flow moves them
    for lat in (here, there):
        lat.set_interface((0.0, 0.0, 0.0), volume_force_on=0)
        rho = np.ones((wl.nz, wl.ny, wl.nx))
        y = np.arange(wl.ny)[None, :, None] * (2 * np.pi / wl.ny)
        x = np.arange(wl.nx)[None, None, :] * (2 * np.pi / wl.nx)
        u = np.zeros((wl.nz, wl.ny, wl.nx, 3))
        u[..., 0] = 0.01 * np.sin(y)
        u[..., 1] = 0.01 * np.sin(x)
        lat.init_equilibrium(rho, u)
        lat.step(1)
    tol = 1e-15 + 2.0 ** -52 * np.abs(d).max() * 1e-2
    assert np.abs(there.vertex_velocities() - here.vertex_velocities()).max() <= tol
    here.close()
    there.close()
