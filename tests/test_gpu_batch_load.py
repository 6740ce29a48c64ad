"""A box of a batch that loads a state between two batched steps goes on with that state's
parameters (relaxation time, walls, body force), with and without a mesh."""
import numpy as np
import pytest

from paper_2305_18919_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
def test_loaded_parameters_reach_the_batched_steps(precision, mesh, tmp_path):
    from paper_2305_18919_gb300 import binding
    shape = (24, 20, 18)
    v, f = inputs.icosphere(2, 4.0, (12.2, 10.1, 8.7))
    rng = np.random.default_rng(2)
    rho = 1 + rng.uniform(-1e-3, 1e-3, shape[::-1])
    u = rng.uniform(-0.01, 0.01, shape[::-1] + (3,))

    def configure(lat):
        if mesh:
            lat.add_mesh(v, f)
            lat.set_interface((0.01, 0.01, 0.01))
        lat.init_equilibrium(rho, u)

    # the state of a run with other parameters
    other = binding.Lattice(*shape, 0.7, 1.0, (0, 0.02, 0), (0.01, 0, 0), (2e-5, -1e-5, 0), precision)
    configure(other)
    other.step(3)
    other.save_state(tmp_path / "s")
    b = binding.Batch([binding.lattice_desc(*shape, 1.1, 1.0, (-0.01, 0, 0), (0, 0, 0), (0, 0, 0),
                                            precision) for _ in range(2)])
    for lat in b.contexts:
        configure(lat)
    b.step(5)
    b.contexts[1].load_state(tmp_path / "s")
    b.step(4)
    other.step(4)
    assert np.array_equal(b.contexts[1].populations(), other.populations())
    alone = binding.Lattice(*shape, 1.1, 1.0, (-0.01, 0, 0), (0, 0, 0), (0, 0, 0), precision)
    configure(alone)
    alone.step(9)
    assert np.array_equal(b.contexts[0].populations(), alone.populations())
    if mesh:
        assert np.array_equal(b.contexts[1].vertices(), other.vertices())
    for lat in (other, alone):
        lat.close()
    b.close()
