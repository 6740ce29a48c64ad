"""Read-back of rho and u against the same sums over the populations in double: smallest lattices,
rows that are no whole number of warps, walls and periodic z, a body force, every storage type,
before and after the first step, and buffers that are only 8-byte aligned."""
import ctypes

import numpy as np
import pytest

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
              (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)], dtype=float)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape,z_periodic,rho0", [((4, 4, 3), False, 1.0), ((4, 8, 4), True, 1.0),
                                                   ((12, 4, 5), False, 0.7),
                                                   ((132, 4, 7), False, 1.3)])
def test_fields_are_the_moments(shape, z_periodic, rho0, precision):
    import torch
    from paper_2305_18919_gb300 import binding
    nx, ny, nz = shape
    g = np.array((1e-4, -2e-4, 3e-4 if z_periodic else 0.0))
    lat = binding.Lattice(nx, ny, nz, 0.8, rho0, (0.01, 0, 0), (-0.02, 0, 0), g, precision, z_periodic)
    rng = np.random.default_rng(5)
    rho_in = rho0 * (1 + rng.uniform(-0.01, 0.01, (nz, ny, nx)))
    lat.init_equilibrium(rho_in, rng.uniform(-0.03, 0.03, (nz, ny, nx, 3)))
    fluid = slice(None) if z_periodic else slice(1, nz - 1)
    for steps in (0, 1, 2):
        if steps:
            lat.step(1)
        f = lat.populations()[:, fluid]
        rho = f.sum(0)
        # the force is carried in the arithmetic type of the context
        gf = g if precision == "fp64" else g.astype(np.float32).astype(float)
        u = (np.einsum("ik,izyx->zyxk", C, f) + 0.5 * gf) / rho[..., None]
        r1, u1 = lat.fields()
        # 19 terms rounded at 2^-53 of about 1 on the way out of populations(), and 2^-45 of
        # deviations up to 0.04 in the float contexts' pairs
        tol = 19 * 2.0 ** -53 + 60 * 2.0 ** -45 * 0.04
        assert np.abs(r1[fluid] - rho).max() < tol
        assert np.abs(u1[fluid] - u).max() < 4 * tol / rho0
        buf = torch.full((4 * nx * ny * nz + 1,), float("nan"), dtype=torch.float64, device="cuda")
        n = nx * ny * nz
        lat._check(lat._L.iblb_read_fields_device(lat.h, ctypes.c_void_p(buf.data_ptr() + 8),
                                                  ctypes.c_void_p(buf.data_ptr() + 8 * (1 + n))))
        torch.cuda.synchronize()
        out = buf[1:].cpu().numpy()
        assert np.array_equal(out[:n].reshape(r1.shape), r1)
        assert np.array_equal(out[n:].reshape(u1.shape), u1)
    lat.close()
