"""Upsampler boxes whose x-face samples come staged with the tiles and boxes
whose samples do not fit a stage (in FP32 four samples with a weight and the
residual fit from an edge of 64 on), alone and together in one launch, with
and without chains: against the register kernel, which loads every sample and
residual from global memory."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def run(lbt, torch, kernel, edges, storage, nbeads, periodic, steps):
    from paper_0809_4958_gb300 import inputs
    K, u_max = 8, 0.05
    rng = np.random.default_rng(7)
    master = inputs.mlp_init(5, K)
    master[-3 * K:] = 40.0 * rng.standard_normal(3 * K)  # a residual of some 0.03
    params = lbt.Upsampler(K=K, batch_rows=128, master=master.astype(np.float32)).export()
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, periodic=periodic, time_interp=lbt.LB_TIME_MLP, K=K, nbeads=nbeads)
                      for E in edges], storage)
    if kernel is not None:
        tr.lb_set_launch(kernel, 128, 0, 0)
    tr.lb_mlp_bind(params, u_max)
    for b, E in enumerate(edges):
        tr.lb_init(b, np.ascontiguousarray(0.03 * rng.standard_normal((3, E, E, E)), tr.np_real))
        if nbeads:
            tr.chain_couple(b, lbt.chain_desc(nbeads), inputs.chain_start(b, nbeads, E))
    faces = sum(18 * E * E for E in edges)
    smp = [torch.from_numpy(0.03 * rng.standard_normal(faces)).to("cuda", tr.real) for _ in range(4)]
    torch.cuda.synchronize()
    pushed = -1
    for n in range(steps):
        while pushed < n // K + 2:
            pushed += 1
            tr.lb_set_boundary(lbt.LB_ALL_BOXES, pushed, smp[pushed])
        tr.lb_step(1)
    out = [tr.deviations(b).astype(np.float64) for b in range(len(edges))]
    tr.lb_sync()
    tr.close()
    return out


@pytest.mark.parametrize("nbeads", [0, 8])
@pytest.mark.parametrize("edges", [(24,), (56,), (64,), (72,), (128,), (64, 24, 40, 88)])
@pytest.mark.parametrize("storage", [1, 2, 3])
def test_staged_residuals_match_the_register_kernel(edges, storage, nbeads):
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    steps = 3
    for periodic in ((False, False, False), (False, True, False)):
        a = run(lbt, torch, None, edges, storage, nbeads, periodic, steps)
        b = run(lbt, torch, lbt.LB_KERNEL_REGISTER, edges, storage, nbeads, periodic, steps)
        # values of order 0.1: 40 FP32 roundings a step; 16 bits: those may flip the last bit of what is stored
        ulp = (None, 2.0 ** -24, 2.0 ** -10, 2.0 ** -7)[storage]
        tol = 0.3 * steps * (40 * ulp if storage == 1 else ulp)
        for x, y in zip(a, b):
            assert np.abs(x - y).max() <= tol
