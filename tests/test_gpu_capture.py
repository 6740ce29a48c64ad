"""Steps captured into a CUDA graph and replayed between the host's own calls: they continue from the
context's current state, as steps taken by the calls themselves."""
import ctypes

import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu
SHAPE = (32, 28, 25)


class Case:
    """A context on a stream of its own with two steps captured, and one that takes plain steps."""

    def __init__(self, precision, mesh=True, force_field_first=False):
        import torch
        from paper_2305_18919_gb300 import binding
        self.stream = torch.cuda.Stream()
        self.v, f = inputs.icosphere(3, 6.5, (15.8, 14.2, 12.1))
        nx, ny, nz = SHAPE
        rng = np.random.default_rng(5)
        self.rho = 1 + rng.uniform(-1e-3, 1e-3, (nz, ny, nx))
        self.u = rng.uniform(-0.01, 0.01, (nz, ny, nx, 3))
        self.lats = []
        for s in (ctypes.c_void_p(self.stream.cuda_stream), None):
            lat = binding.Lattice(*SHAPE, 0.8, 1.0, (-0.01, 0, 0), (0.01, 0, 0), (1e-6, 0, 0),
                                  precision, stream=s, ib_sms=-1)
            if mesh:
                lat.add_mesh(self.v, f)
                lat.set_interface((0.01, 0.01, 0.01))
            lat.init_equilibrium(self.rho, self.u)
            lat.step(3)
            self.lats.append(lat)
        if force_field_first:
            self.lats[0].force_field()
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph, stream=self.stream):
            self.lats[0].step_async(2)

    def replay(self, n=1):
        import torch
        with torch.cuda.stream(self.stream):
            for _ in range(n):
                self.graph.replay()
        torch.cuda.synchronize()
        self.lats[1].step(2 * n)

    def both(self, call):
        return [call(lat) for lat in self.lats]

    def close(self):
        for lat in self.lats:
            lat.close()


def _same(pair):
    assert np.array_equal(pair[0], pair[1])


@pytest.mark.parametrize("force_field_first", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
def test_replayed_steps_and_the_force_field(precision, force_field_first):
    c = Case(precision, force_field_first=force_field_first)
    # positions set between the capture and its first run
    c.both(lambda lat: lat.set_vertices(inputs.perturb(c.v, 0.02, seed=1)))
    for n in (1, 3):
        c.replay(n)
        for _ in range(2):  # read twice: the first read leaves nothing behind
            _same(c.both(lambda lat: lat.force_field()))
        _same(c.both(lambda lat: lat.vertices()))
        _same(c.both(lambda lat: lat.populations()))
    c.replay()
    c.both(lambda lat: lat.set_vertices(inputs.perturb(c.v, 0.02, seed=2)))
    _same(c.both(lambda lat: lat.force_field()))
    c.replay()
    _same(c.both(lambda lat: lat.vertex_velocities()))
    c.close()


def test_failure_of_replayed_steps_is_not_that_of_later_ones():
    import torch
    c = Case("fp32")
    lat, ref = c.lats
    for x in c.lats:
        x.step_async(2)
        x.vertices()  # reads the health word: clear
    lat.set_vertices(c.v.mean(0) + 0.9 * (c.v - c.v.mean(0)))  # beyond the volume check
    with torch.cuda.stream(c.stream):
        c.graph.replay()
    torch.cuda.synchronize()
    for x in c.lats:
        x.init_equilibrium(c.rho, c.u)
        x.set_vertices(inputs.perturb(c.v, 0.02, seed=3))
        x.step_async(2)
    _same(c.both(lambda x: x.vertices()))
    c.close()
