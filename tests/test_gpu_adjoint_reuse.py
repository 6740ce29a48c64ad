"""A context's adjoint arrays serve several recordings: longer, shorter, other copy spacings, a
release in between. Each gradient is that of a fresh context (to the order of the FP64 atomic
additions of the force field, 1e-12), and a failed or missing recording is refused."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_recordings_of_other_lengths(precision):
    from paper_2305_18919_gb300 import binding
    a = tuple(0.01 * x for x in inputs.ALPHA_CLASSES["softly_coated"])
    wl = inputs.scaled_wetting(24, 20, 2, 5.0, a, 0.005, precision=precision, lift=0.5)
    v, _ = wl.mesh()
    q = inputs.perturb(v, 0.02, seed=4)
    rho = np.ones((wl.nz, wl.ny, wl.nx))
    u = np.full((wl.nz, wl.ny, wl.nx, 3), 1e-3)
    w = np.cos(np.arange(v.size).reshape(v.shape) * 0.7)

    def gradient(lat, nsteps, every, lead):
        lat.init_equilibrium(rho, u)
        lat.set_vertices(q)
        if lead:
            lat.step(lead)
        lat.adjoint_record(nsteps, every)
        return lat.adjoint_gradient(w), lat.vertices()

    kept = binding.Lattice.from_workload(wl, precision=precision)
    for k, (nsteps, every, lead) in enumerate([(7, 3, 0), (12, 5, 2), (5, 9, 0), (1, 1, 1), (9, 2, 0)]):
        fresh = binding.Lattice.from_workload(wl, precision=precision)
        g0, q0 = gradient(fresh, nsteps, every, lead)
        fresh.close()
        g1, q1 = gradient(kept, nsteps, every, lead)
        assert np.array_equal(q1, q0)
        np.testing.assert_allclose(g1, g0, rtol=1e-12, atol=1e-14 * np.abs(g0).max())
        if k == 2:
            kept.adjoint_release()
            with pytest.raises(binding.IBLBError):
                kept.adjoint_gradient(w)
    # a recording that fails leaves none: the mesh is compressed beyond the volume check
    kept.set_vertices(v.mean(0) + 0.9 * (v - v.mean(0)))
    with pytest.raises(binding.IBLBError):
        kept.adjoint_record(4, 2)
    with pytest.raises(binding.IBLBError):
        kept.adjoint_gradient(w)
    kept.close()
