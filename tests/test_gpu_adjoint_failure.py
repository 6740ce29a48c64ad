"""A gradient whose recomputation fails a health check (parameters changed after the recording) leaves
the context at the end of the recorded run, and the recording serves again."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("nsteps,every", [(5, 2), (4, 4), (7, 3)])
def test_failed_gradient_returns_to_the_end(precision, nsteps, every):
    from paper_2305_18919_gb300 import binding
    a = tuple(0.01 * x for x in inputs.ALPHA_CLASSES["softly_coated"])
    wl = inputs.scaled_wetting(24, 20, 2, 5.0, a, 0.005, precision=precision, lift=0.5)
    v, _ = wl.mesh()
    w = np.cos(np.arange(v.size).reshape(v.shape) * 0.7)
    lat = binding.Lattice.from_workload(wl, precision=precision)
    lat.set_vertices(inputs.perturb(v, 0.02, seed=4))
    lat.step(2)
    lat.adjoint_record(nsteps, every)
    want = lat.adjoint_gradient(w)
    q, f = lat.vertices(), lat.populations()
    args = (wl.kV, wl.eps, wl.xi, wl.wall_force_on, wl.volume_force_on)
    lat.set_interface((5.0, 5.0, 5.0), *args)
    with pytest.raises(binding.IBLBError) as e:
        lat.adjoint_gradient(w)
    assert e.value.code == binding.IBLB_EUNSTABLE and "health" in str(e.value)
    assert np.array_equal(lat.vertices(), q) and np.array_equal(lat.populations(), f)
    lat.set_interface(wl.alpha, *args)
    got = lat.adjoint_gradient(w)
    np.testing.assert_allclose(got, want, rtol=1e-12, atol=1e-14 * np.abs(want).max())
    assert np.array_equal(lat.vertices(), q) and np.array_equal(lat.populations(), f)
    lat.close()
