"""Velocity read-out where the density is near the top of the storage type's
range, so that its reciprocal is below the smallest normal number: u = j / rho
all the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,rho_b", [(0, 1e308), (1, 1e38), (1, 2e38), (1, 1e30)])
def test_velocity_of_a_dense_boundary(storage, rho_b):
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    E = 16
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, rho_b=rho_b)], storage)
    face = 0.05 * np.random.default_rng(1).standard_normal((6, 3, E, E))
    tr.lb_init(0, np.zeros((3, E, E, E), tr.np_real))
    for j in range(2):
        tr.lb_set_boundary(0, j, np.ascontiguousarray(face, tr.np_real))
    tr.lb_step(1)  # the boundary layer of t = 1; the interior still pulls from rho = 1
    u = torch.empty((3, E, E, E), dtype=tr.real, device="cuda")
    torch.cuda.synchronize()
    tr.lb_read_fields(0, lbt.LB_FIELD_U, u)
    got = u.cpu().numpy().astype(np.float64)
    # x- face: populations with some ten roundings each, j a difference of ten of them, all of the density's size
    tol = 10 * 10 * (2.0 ** -53 if storage == 0 else 2.0 ** -24)
    assert np.abs(got[:, :, :, 0] - face[0]).max() <= tol
    assert np.abs(got[:, :, :, -1] - face[1])[:, 1:-1, 1:-1].max() <= tol
    tr.close()
