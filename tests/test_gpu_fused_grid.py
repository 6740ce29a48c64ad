"""The one-kernel step on either side of the sizes from which its grid takes all SMs, and several
contexts stepped at once from threads of their own: the bits of the separate kernels and of a context
stepped alone."""
import ctypes
import threading

import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu


def _context(shape, sub, precision, seed=1, stream=None):
    from paper_2305_18919_gb300 import binding
    lat = binding.Lattice(*shape, 0.8, 1.0, (-0.01, 0, 0), (0.01, 0, 0), (1e-6, 0, 0), precision,
                          stream=stream)
    v, f = inputs.icosphere(sub, 0.2 * min(shape), tuple(n / 2 + 0.1 for n in shape))
    lat.add_mesh(v, f)
    lat.set_interface((0.01, 0.01, 0.01))
    lat.set_vertices(inputs.perturb(v, 0.01, seed=seed))
    return lat


def _state(lat):
    return [lat.populations(), lat.vertices(), lat.vertex_velocities()]


@pytest.mark.parametrize("shape,sub,precision", [
    ((64, 64, 64), 4, "fp32"), ((68, 64, 64), 4, "fp32"), ((64, 64, 64), 3, "bf16"),
    ((48, 48, 48), 5, "fp16"), ((48, 48, 48), 4, "fp16"), ((40, 40, 40), 3, "fp64"),
    ((44, 40, 40), 3, "fp64"), ((20, 20, 20), 2, "fp64")])
def test_grid_sizes(shape, sub, precision):
    got = []
    for separate in (False, True):
        lat = _context(shape, sub, precision)
        lat.set_profiling(separate)
        for n in (3, 12):
            lat.step(n)
        got.append(_state(lat))
        lat.close()
    for x, y in zip(*got):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("shape,sub,precision", [((24, 24, 24), 2, "fp32"), ((32, 32, 32), 2, "fp64"),
                                                 ((72, 72, 72), 4, "fp16")])
def test_contexts_at_once(shape, sub, precision):
    import torch
    streams = [torch.cuda.Stream() for _ in range(4)]
    at_once = [_context(shape, sub, precision, seed, ctypes.c_void_p(s.cuda_stream))
               for seed, s in enumerate(streams)]
    errors = []

    def run(lat):
        try:
            for n in (1, 70, 40):
                lat.step(n)
        except Exception as e:  # reported below, with the thread's context
            errors.append(e)
    threads = [threading.Thread(target=run, args=(lat,)) for lat in at_once]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for seed, lat in enumerate(at_once):
        alone = _context(shape, sub, precision, seed)
        alone.step(111)
        for x, y in zip(_state(lat), _state(alone)):
            assert np.array_equal(x, y)
        alone.close()
        lat.close()
