"""A grid barrier of the one-kernel step that gives up (a limit of 0 lets the first block to arrive
give up) ends every block, is reported as a timeout, also by steps queued behind it, and leaves the
context usable: with a state restored it repeats a fresh context's run bit for bit."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (36, 32, 27)


def _context(precision, mesh):
    from paper_2305_18919_gb300 import binding
    lat = binding.Lattice(*SHAPE, 0.8, 1.0, (-0.01, 0, 0), (0.01, 0, 0), (1e-6, 0, 0), precision)
    v, f = inputs.icosphere(3, 7.0, (17.6, 16.3, 13.1))
    if mesh:
        lat.add_mesh(v, f)
        lat.set_interface((0.01, 0.01, 0.01), 1.0, 0.0, 0.5, 0, 1)
    rng = np.random.default_rng(3)
    nx, ny, nz = SHAPE
    rho = 1 + rng.uniform(-1e-3, 1e-3, (nz, ny, nx))
    u = rng.uniform(-0.01, 0.01, (nz, ny, nx, 3))
    q = inputs.perturb(v, 0.02, seed=2)

    def start():
        lat.init_equilibrium(rho, u)
        if mesh:
            lat.set_vertices(q)
    return lat, start


def _result(lat, steps=6):
    lat.step(steps)
    out = [lat.populations(), *lat.fields()]
    return out + ([lat.vertices(), lat.vertex_velocities(), lat.force_field()] if lat.nv else [])


def _same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("precision,mesh", [("fp64", True), ("fp32", True), ("fp16", True),
                                            ("bf16", True), ("fp32", False), ("fp16", False)])
def test_barrier_limit_runs_out_and_context_recovers(precision, mesh, tmp_path):
    from paper_2305_18919_gb300 import binding
    ref, start = _context(precision, mesh)
    start()
    want = _result(ref)
    ref.step(3)
    ref.save_state(tmp_path / "s")
    later = _result(ref, 5)
    ref.close()
    lat, start = _context(precision, mesh)
    start()
    lat.step(1)  # the first step runs as separate kernels
    for k, lost in enumerate((3, 2, 70, 131)):  # both maps, several launches queued
        lat.step(4 + k % 2)
        lat.set_barrier_wait_limit(0)
        if k < 2:  # reported by the call itself, or by the next read
            with pytest.raises(binding.IBLBError) as e:
                lat.step(lost)
        else:
            lat.step_async(lost)
            lat.step_async(2)
            with pytest.raises(binding.IBLBError) as e:
                lat.fields()
        assert e.value.code == binding.IBLB_ETIMEOUT
        lat.set_barrier_wait_limit(2 * 10 ** 9)
        start()
        _same(_result(lat), want)
    # an unread timeout, discarded with the state it left
    lat.set_barrier_wait_limit(0)
    lat.step_async(5)
    lat.set_barrier_wait_limit(2 * 10 ** 9)
    start()
    _same(_result(lat), want)
    lat.set_barrier_wait_limit(0)
    lat.step_async(2)
    lat.set_barrier_wait_limit(2 * 10 ** 9)
    lat.load_state(tmp_path / "s")
    _same(_result(lat, 5), later)
    for ns in (-1, 60 * 10 ** 9 + 1):
        with pytest.raises(binding.IBLBError) as e:
            lat.set_barrier_wait_limit(ns)
        assert e.value.code == binding.IBLB_EINVAL
    lat.close()
