"""Spreading from source tiles that hold more vertices than a bucket (128): all of a mesh in one tile,
meshes whose last bitmap word is partial, more vertices of a tile in one round of the scan than the
stage holds, and many spilled tiles. The force field is the sum of the nodal forces over the stencils,
within the rounding of that sum; steps give the same bits through the one-kernel step and through the
separate kernels."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (24, 20, 19)


def _weights(q):
    """Base nodes [nv][3] and one-dimensional Peskin weights [nv][3][4], in extended precision."""
    q = q.astype(np.longdouble)
    r = q - np.floor(q)
    s = np.sqrt(1 + 4 * r - 4 * r * r)
    w = np.stack([3 - 2 * r - s, 3 - 2 * r + s, 1 + 2 * r + s, 1 + 2 * r - s], -1) / 8
    return np.floor(q).astype(int) - 1, w


def _spread(q, phi, u):
    """The force field and a bound of its rounding error for arithmetic of unit roundoff u. A node sums
    n terms phi w in any order: (n + 6) u |phi w| each, six for the products. A one-dimensional weight,
    at most a half, is off by at most 2 u absolutely (four roundings of values up to 3, over 8, and its
    argument's), so a product of three by 2 u (1/4 + 1/4 + 1/4) = 1.5 u."""
    nx, ny, nz = SHAPE
    base, w = _weights(q)
    F = np.zeros((nz, ny, nx, 3), np.longdouble)
    A = np.zeros((nz, ny, nx, 3), np.longdouble)  # sum of |phi w|
    B = np.zeros((nz, ny, nx, 3), np.longdouble)  # sum of |phi|
    n = np.zeros((nz, ny, nx, 1))
    for dz in range(4):
        for dy in range(4):
            for dx in range(4):
                at = (base[:, 2] + dz, (base[:, 1] + dy) % ny, (base[:, 0] + dx) % nx)
                t = phi * (w[:, 0, dx] * w[:, 1, dy] * w[:, 2, dz])[:, None]
                np.add.at(F, at, t)
                np.add.at(A, at, np.abs(t))
                np.add.at(B, at, np.abs(phi))
                np.add.at(n, at, 1)
    return F, u * ((n + 6) * A + 1.5 * B)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("sub,radius,centre,most", [
    (2, 0.95, (11.0, 11.0, 11.0), 162), (3, 0.95, (11.0, 11.0, 11.0), 642),
    (4, 0.95, (11.0, 11.0, 11.0), 2562), (4, 2.6, (12.3, 9.7, 9.1), None),
    (5, 6.0, (0.4, 19.6, 9.2), None)])
def test_spilled_tiles(sub, radius, centre, most, precision):
    from paper_2305_18919_gb300 import binding
    v, f = inputs.icosphere(sub, radius, centre)
    q = inputs.perturb(v, 0.002, seed=6)
    tiles = np.stack([((np.floor(q[:, k]).astype(int) - 1) % SHAPE[k]) // 4 for k in range(3)], -1)
    held = np.unique(tiles, axis=0, return_counts=True)[1].max()
    assert held == most if most else held > 128
    lats = [binding.Lattice(*SHAPE, 0.9, precision=precision) for _ in range(2)]
    for lat in lats:
        lat.add_mesh(v, f)
        lat.set_interface((1e-4, 1e-4, 1e-4), volume_force_on=0)
        lat.set_vertices(q)
    lat = lats[0]
    F, bound = _spread(q, lat.forces(), 2.0 ** (-53 if precision == "fp64" else -24))
    assert (np.abs(lat.force_field() - F) <= bound).all()
    lats[1].set_profiling(True)  # the separate kernels
    for lat in lats:
        lat.step(4)
    for call in ("vertices", "vertex_velocities", "populations", "force_field"):
        assert np.array_equal(*(getattr(lat, call)() for lat in lats))
    for lat in lats:
        lat.close()
