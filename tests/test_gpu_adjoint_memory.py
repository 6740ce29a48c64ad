"""Adjoint calls that run out of device memory: the gradient frees what it had allocated, the context
goes on, and with room again gives the gradient of a fresh context; a recording that does not fit
beside the last gradient's arrays takes their room. Most of the device's memory is held meanwhile."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def _workload():
    a = tuple(0.01 * x for x in inputs.ALPHA_CLASSES["softly_coated"])
    return inputs.scaled_wetting(64, 64, 3, 12.0, a, 0.005, precision="fp64", lift=0.5)


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _hold(leave):
    """All of the free device memory but about `leave` bytes."""
    import torch
    torch.cuda.empty_cache()
    return torch.empty(_free() - leave, dtype=torch.uint8, device="cuda")


def _release(*held):
    import torch
    del held
    torch.cuda.empty_cache()


def test_gradient_without_room_leaks_nothing():
    from paper_2305_18919_gb300 import binding
    wl = _workload()
    v, _ = wl.mesh()
    q = inputs.perturb(v, 0.02, seed=4)
    w = np.cos(np.arange(v.size).reshape(v.shape) * 0.7)
    ref = binding.Lattice.from_workload(wl, precision="fp64")
    ref.set_vertices(q)
    ref.adjoint_record(4, 2)
    want = ref.adjoint_gradient(w)
    ref.close()
    lat = binding.Lattice.from_workload(wl, precision="fp64")
    lat.set_vertices(q)
    lat.adjoint_record(4, 2)
    state = 19 * 64 ** 3 * 8  # bytes of one population array: 38 MiB; a gradient's two come first
    held = _hold(state + state // 2)
    before = _free()
    assert state < before < 2 * state
    for _ in range(3):
        with pytest.raises(binding.IBLBError) as e:
            lat.adjoint_gradient(w)
        assert e.value.code == binding.IBLB_ENOMEM
        assert before - _free() <= 4 * MIB
    lat.set_vertices(lat.vertices())  # the failed allocation is no later call's error
    del held
    _release()
    np.testing.assert_allclose(lat.adjoint_gradient(w), want, rtol=1e-12, atol=1e-14 * np.abs(want).max())
    lat.close()


def test_recording_takes_the_room_of_the_last_gradient():
    from paper_2305_18919_gb300 import binding
    wl = _workload()
    v, _ = wl.mesh()
    w = np.cos(np.arange(v.size).reshape(v.shape) * 0.7)
    lat = binding.Lattice.from_workload(wl, precision="fp64")
    lat.adjoint_record(4, 2)
    lat.adjoint_gradient(w)
    state = 19 * 64 ** 3 * 8
    held = _hold(state // 2)
    lat.adjoint_record(8, 2)  # two more states than before: only the work arrays leave room
    assert lat.steps_done >= 12
    del held
    _release()
    assert np.isfinite(lat.adjoint_gradient(w)).all()
    lat.close()
