"""Density and velocity read-outs (lb_read_fields) against the moments of the
stored populations, formed in FP64 from the LB_FIELD_DEV read-out of the same
state: every storage format, velocity and periodic axes, edges from one group
of sites per row up, destinations that are and are not 16-byte aligned."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    assert torch.cuda.is_available()
    lbt.load()
    return lbt, torch


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("periodic", [(False, False, False), (True, False, False), (False, True, True), (True, True, True)])
@pytest.mark.parametrize("E", [8, 24, 40])
@pytest.mark.parametrize("storage", [0, 1, 2, 3])
def test_fields_are_the_moments_of_the_populations(gpu, storage, E, periodic, offset):
    lbt, torch = gpu
    accel = (1e-4, -2e-4, 3e-4)
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, periodic=periodic, accel=accel)], storage)
    rng = np.random.default_rng(E)
    u0 = np.ascontiguousarray(0.05 * rng.standard_normal((3, E, E, E)), tr.np_real)
    tr.lb_init(0, u0)
    d = tr.deviations(0).astype(np.float64)
    n3 = E ** 3
    rho = torch.zeros(n3 + 4, dtype=tr.real, device="cuda")
    u = torch.zeros(3 * n3 + 4, dtype=tr.real, device="cuda")
    torch.cuda.synchronize()
    tr.lb_read_fields(0, lbt.LB_FIELD_RHO, rho.data_ptr() + offset * rho.element_size())
    tr.lb_read_fields(0, lbt.LB_FIELD_U, u.data_ptr() + offset * u.element_size())
    c, _ = oracle.lattice()
    bnd = np.zeros((E, E, E), bool)  # axes z, y, x
    for a in range(3):
        if not periodic[a]:
            np.moveaxis(bnd, 2 - a, 0)[[0, -1]] = True
    pulled = np.stack([np.where(bnd, d[i], np.roll(d[i], (c[i, 2], c[i, 1], c[i, 0]), (0, 1, 2))) for i in range(19)])
    r = 1.0 + pulled.sum(0)
    j = np.einsum("ia,izyx->azyx", c.astype(np.float64), pulled)
    j += np.where(bnd, 0.0, 0.5 * r) * np.array(accel)[:, None, None, None]
    # sums of at most 20 terms of order 0.1 in the arithmetic type, one division
    tol = 40 * 0.1 * (2.0 ** -53 if storage == 0 else 2.0 ** -24)
    got_r = rho[offset:offset + n3].cpu().numpy().astype(np.float64).reshape(E, E, E)
    got_u = u[offset:offset + 3 * n3].cpu().numpy().astype(np.float64).reshape(3, E, E, E)
    assert np.abs(got_r - r).max() <= tol + (2.0 ** -53 if storage == 0 else 2.0 ** -24)
    assert np.abs(got_u - j / r).max() <= tol
    guard = torch.cat([rho[:offset], rho[offset + n3:], u[:offset], u[offset + 3 * n3:]])
    assert float(guard.abs().max()) == 0.0  # nothing written past the field
    tr.close()
