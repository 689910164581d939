"""A fluctuating box whose boundary comes from the learned upsampler: its
boundary layer is the one of the same box without fluctuations -- Hermite plus
the network's residual -- in every storage format and in both bodies of the
stream-collide (one and two sites a thread)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("E", [16, 64])
@pytest.mark.parametrize("storage,sites", [(0, 1), (1, 1), (1, 2), (2, 1), (2, 2), (3, 1), (3, 2)])
def test_boundary_layer_carries_the_residual(storage, sites, E):
    import torch

    from paper_0809_4958_gb300 import inputs, lbtracer as lbt
    lbt.load()
    K, u_max = 8, 0.05
    rng = np.random.default_rng(2)
    master = inputs.mlp_init(5, K)
    nout = 3 * K
    master[-nout:] = 40.0 * rng.standard_normal(nout)  # a residual of some 0.02 on every face
    params = lbt.Upsampler(K=K, batch_rows=128, master=master.astype(np.float32)).export()
    smp = [0.03 * rng.standard_normal((6, 3, E, E)) for _ in range(3)]
    u0 = 0.03 * rng.standard_normal((3, E, E, E))
    out = {}
    for interp, noise in ((lbt.LB_TIME_HERMITE, False), (lbt.LB_TIME_MLP, False), (lbt.LB_TIME_MLP, True)):
        tr = lbt.Tracers([lbt.box_desc(E, 0.8, time_interp=interp, K=K)], storage)
        tr.lb_set_launch(lbt.LB_KERNEL_STAGED, 0, 0, sites)
        if interp == lbt.LB_TIME_MLP:
            tr.lb_mlp_bind(params, u_max)
        tr.lb_init(0, np.ascontiguousarray(u0, tr.np_real))
        if noise:
            tr.lb_set_fluctuation(0, 1e-5, 3, np.full(19, -0.25))
        for j in range(3):
            tr.lb_set_boundary(0, j, np.ascontiguousarray(smp[j], tr.np_real))
        tr.lb_step(2)
        out[interp, noise] = tr.deviations(0).astype(np.float64)
        tr.lb_sync()
        tr.close()
    bnd = np.ones((E, E, E), bool)
    bnd[1:-1, 1:-1, 1:-1] = False
    herm, plain, noisy = (out[k][:, bnd] for k in ((1, False), (2, False), (2, True)))
    assert np.abs(plain - herm).max() > 1e-3  # the residual matters
    # the boundary equilibrium in the arithmetic type (some twenty roundings of terms of at most 0.5), then storage
    eps = (2.0 ** -53, 2.0 ** -24, 2.0 ** -24, 2.0 ** -24)[storage]
    store = (0.0, 0.0, 2.0 ** -10, 2.0 ** -7)[storage]
    assert np.abs(noisy - plain).max() <= 20 * 0.5 * eps + store * np.abs(plain).max()
