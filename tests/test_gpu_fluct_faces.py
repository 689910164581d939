"""The fluctuating collision of boxes with velocity faces, in the formats that
work on pairs of sites: the boundary layer is the equilibrium of the boundary
velocity whatever the boundary sites pulled, and all sites agree with the body
that takes one site a thread (the same noise words and FP32 arithmetic in
another order)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

ULP = {1: 2.0 ** -24, 2: 2.0 ** -11, 3: 2.0 ** -8}  # relative rounding of a stored population


def gammas(tau=0.8):
    g = np.full(19, 1.0 - 1.0 / tau)
    g[4], g[10:16], g[16:19] = 0.2, -0.3, 0.1
    return g


def run(lbt, torch, E, storage, periodic, u0, faces, kT, steps, sites):
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, periodic=periodic)], storage)
    tr.lb_set_launch(lbt.LB_KERNEL_STAGED, 0, 0, sites)
    tr.lb_init(0, np.ascontiguousarray(u0, tr.np_real))
    tr.lb_set_fluctuation(0, kT, 99, gammas())
    for n in range(steps):
        if not all(periodic):
            for j in ((0, 1) if n == 0 else (n + 1,)):
                tr.lb_set_boundary(0, j, np.ascontiguousarray(faces[j], tr.np_real))
        tr.lb_step(1)
    d = tr.deviations(0).astype(np.float64)
    tr.lb_sync()
    tr.close()
    return d


@pytest.fixture(scope="module")
def gpu():
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    assert torch.cuda.is_available()
    lbt.load()
    return lbt, torch


@pytest.mark.parametrize("sites", [1, 2])
@pytest.mark.parametrize("storage", [1, 2, 3])
def test_boundary_sites_do_not_depend_on_what_they_pull(gpu, storage, sites):
    """A fast inflow on the x- face: the sum of what its sites pull is below
    -1 (the populations along the face, 1 - u^2 of them, without those from
    the interior), a density that has no square root."""
    lbt, torch = gpu
    E, ux = 16, 1.25
    u0 = np.zeros((3, E, E, E))
    u0[0, :, :, 0] = ux
    face = np.zeros((6, 3, E, E))
    face[0, 0] = ux
    d = run(lbt, torch, E, storage, (False,) * 3, u0, [face, face], 1e-6, 1, sites)
    c, w = oracle.lattice()
    cu = c[:, 0] * ux
    want = w * (3.0 * cu + 4.5 * cu * cu - 1.5 * ux * ux)
    # a population of the boundary equilibrium: some ten roundings in FP32 of terms up to 12 w, one of storage
    tol = 12 * w.max() * 10 * 2.0 ** -24 + np.abs(want).max() * ULP[storage]
    assert np.abs(d[:, :, :, 0] - want[:, None, None]).max() <= tol
    assert np.isfinite(d).all()


@pytest.mark.parametrize("periodic", [(False, False, False), (True, False, False), (False, True, False), (False, False, True),
                                      (True, True, True)])
@pytest.mark.parametrize("E", [8, 24, 40])
@pytest.mark.parametrize("storage", [1, 2, 3])
def test_pairs_of_sites_agree_with_single_sites(gpu, storage, E, periodic):
    lbt, torch = gpu
    steps, kT = 3, 1e-4
    rng = np.random.default_rng(E)
    u0 = 0.03 * rng.standard_normal((3, E, E, E))
    faces = 0.03 * rng.standard_normal((steps + 1, 6, 3, E, E))
    a = run(lbt, torch, E, storage, periodic, u0, faces, kT, steps, 2)
    b = run(lbt, torch, E, storage, periodic, u0, faces, kT, steps, 1)
    top = np.abs(b).max()
    assert top < 0.3
    # FP32: 100 roundings of values of that size a step.  16 bits: a stored value may round to its neighbour (two units of
    # ULP), and the collision passes the four largest of what a site pulled on with a factor of at most one each
    tol = steps * 100 * 2.0 ** -24 * top + (0 if storage == 1 else steps * 4 * 2 * ULP[storage] * top)
    assert np.abs(a - b).max() <= tol
