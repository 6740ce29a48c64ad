"""The fused step kernel (one launch for many steps) against the separate kernels, which profiling
selects: the same populations, vertices and vertex velocities bit for bit, for meshes below and
above one round of the grid, ragged rows, walls and periodic z, a body force, every storage type,
step counts around the steps of one launch, and lattices without a mesh."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu


def _run(lat, counts):
    out = []
    for n in counts:
        lat.step(n)
        out += [lat.populations(), *lat.fields()]
        if lat.nv:
            out += [lat.vertices(), lat.vertex_velocities()]
    return out


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape,sub,radius,z_periodic", [((24, 28, 18), 2, 5.0, False),
                                                         ((20, 24, 20), 3, 5.5, True),
                                                         ((52, 44, 41), 5, 12.0, False)])
def test_fused_steps_are_the_separate_ones(shape, sub, radius, z_periodic, precision):
    from paper_2305_18919_gb300 import binding
    nx, ny, nz = shape
    v, f = inputs.icosphere(sub, radius, (nx / 2 + 0.3, ny / 2 - 0.2, (nz - 1) / 2 + 0.1))
    rng = np.random.default_rng(3)
    rho = 1 + rng.uniform(-1e-3, 1e-3, (nz, ny, nx))
    u = rng.uniform(-0.01, 0.01, (nz, ny, nx, 3))
    got = []
    for separate in (False, True):
        lat = binding.Lattice(nx, ny, nz, 0.8, 1.0, (-0.01, 0, 0), (0.01, 0, 0), (1e-6, 2e-6, 0),
                              precision, z_periodic)
        lat.add_mesh(v, f)
        lat.set_interface((0.01, 0.01, 0.01), 1.0, 1e-4, 0.5, 1, 1)
        lat.set_vertices(inputs.perturb(v, 0.01, seed=2))
        lat.init_equilibrium(rho, u)
        lat.set_profiling(separate)
        got.append(_run(lat, (1, 1, 2, 5)) + _run(lat, (65, 130) if shape[0] == 24 else (3,)))
        lat.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("precision", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape,z_periodic", [((4, 4, 3), False), ((4, 8, 4), True),
                                              ((36, 20, 17), False), ((100, 36, 12), True)])
def test_fused_lattice_steps(shape, z_periodic, precision):
    from paper_2305_18919_gb300 import binding
    nx, ny, nz = shape
    rng = np.random.default_rng(7)
    rho = 1 + rng.uniform(-1e-3, 1e-3, (nz, ny, nx))
    u = rng.uniform(-0.01, 0.01, (nz, ny, nx, 3))
    got = []
    for separate in (False, True):
        lat = binding.Lattice(nx, ny, nz, 0.9, 1.0, (0.01, 0, 0), (0, 0.01, 0), (1e-6, 0, 0), precision,
                              z_periodic)
        lat.init_equilibrium(rho, u)
        lat.set_profiling(separate)
        got.append(_run(lat, (1, 1, 2, 64, 131)))
        lat.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)


def test_asynchronous_steps_and_failure():
    """Queued fused steps report a failed health check at the next read-back, as separate ones."""
    from paper_2305_18919_gb300 import binding
    a = tuple(0.01 * x for x in inputs.ALPHA_CLASSES["softly_coated"])
    wl = inputs.scaled_wetting(24, 20, 2, 5.0, a, 0.005, precision="fp32", lift=0.5)
    one, two = (binding.Lattice.from_workload(wl) for _ in range(2))
    two.set_profiling(True)
    for lat in (one, two):
        lat.step(1)
        for n in (1, 3, 70):
            lat.step_async(n)
    assert np.array_equal(one.vertices(), two.vertices())
    v, _ = wl.mesh()
    for lat in (one, two):
        lat.set_vertices(v.mean(0) + 0.9 * (v - v.mean(0)))  # beyond the volume check
        lat.step_async(2)
        with pytest.raises(binding.IBLBError) as e:
            lat.vertices()
        assert e.value.code == binding.IBLB_EUNSTABLE
        lat.close()
