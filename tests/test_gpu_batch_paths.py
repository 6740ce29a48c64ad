"""Batched steps on each of the paths they take: the lattice pass beside the interface chain on an SM
partition and in FP64, the pass that takes the interface force in otherwise, with a body force, on one
lane and on three, with one precision and several. Every box ends bit for bit as when stepped alone."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu


def _box(shape, sub, radius, seed):
    v, f = inputs.icosphere(sub, radius, tuple(n / 2 + 0.2 for n in shape))
    return shape, v, f, inputs.perturb(v, 0.01, seed=seed)


def _configure(lat, box, start):
    shape, v, f, q = box
    lat.add_mesh(v, f)
    lat.set_interface((0.01, 0.005, 0.01), 1.0, 1e-4, 0.5, 1, 1)
    lat.set_vertices(q)
    if start is not None:
        rho, u = start
        lat.init_equilibrium(rho, u)


def _check(boxes, precisions, steps, ib_sms=0, force=(0.0, 0.0, 0.0), z_periodic=False, initial=True):
    from paper_2305_18919_gb300 import binding
    args = (0.8, 1.0, (-0.01, 0, 0), (0.01, 0, 0), force)
    rng = np.random.default_rng(9)
    starts = [(1 + rng.uniform(-1e-3, 1e-3, b[0][::-1]), rng.uniform(-0.01, 0.01, b[0][::-1] + (3,)))
              if initial else None for b in boxes]
    batch = binding.Batch([binding.lattice_desc(*b[0], *args, p, z_periodic, ib_sms)
                           for b, p in zip(boxes, precisions)])
    for lat, box, start in zip(batch.contexts, boxes, starts):
        _configure(lat, box, start)
    for n in steps:
        batch.step(n)
    assert not batch.status().any()
    for lat, box, start, p in zip(batch.contexts, boxes, starts, precisions):
        ref = binding.Lattice(*box[0], *args, p, z_periodic, ib_sms=-1)
        _configure(ref, box, start)
        ref.step(sum(steps))
        for call in ("vertices", "vertex_velocities", "populations"):
            assert np.array_equal(getattr(lat, call)(), getattr(ref, call)())
        ref.close()
    batch.close()


BOXES = [_box((32, 28, 25), 3, 6.5, 1), _box((24, 36, 21), 2, 5.0, 2), _box((44, 20, 30), 3, 5.5, 3)]


@pytest.mark.parametrize("ib_sms", [0, 32])
@pytest.mark.parametrize("force,z_periodic", [((0.0, 0.0, 0.0), False), ((2e-6, -1e-6, 0.0), False),
                                              ((1e-6, 0.0, 2e-6), True)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
def test_one_precision(precision, force, z_periodic, ib_sms):
    boxes = BOXES if not z_periodic else [_box((32, 28, 24), 3, 6.5, 1), _box((24, 36, 20), 2, 5.0, 2)]
    _check(boxes, [precision] * len(boxes), (7, 4), ib_sms, force, z_periodic)


@pytest.mark.parametrize("ib_sms", [0, 32])
def test_precisions_side_by_side(ib_sms):
    _check(BOXES + [_box((28, 28, 28), 3, 6.0, 4)], ["fp16", "fp64", "bf16", "fp32"], (5, 6), ib_sms,
           (1e-6, 0.0, 0.0))


def test_three_lanes_of_several_precisions():
    """4 Mi nodes and more: three lanes, some of which hold boxes of both kinds."""
    shapes = [(96, 96, 96), (128, 128, 96), (96, 128, 100), (100, 96, 96), (92, 96, 80), (64, 64, 64)]
    assert sum(a * b * c for a, b, c in shapes) >= 4 << 20
    boxes = [_box(s, 4, 0.18 * min(s), k) for k, s in enumerate(shapes)]
    _check(boxes, ["fp64", "fp32", "fp16", "fp32", "bf16", "fp64"], (5,), initial=False)
