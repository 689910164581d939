"""Ensembles in which a producer claims runs of two and of four neighbouring
tiles (from 4 and from 16 tiles to an SM on, smaller boxes than that leave
single tiles), runs that cross box borders and a last run that is cut: against
the register kernel, which deals tiles by block index."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def run(lbt, torch, kernel, edges, storage, nbeads, steps):
    from paper_0809_4958_gb300 import inputs
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, nbeads=nbeads) for E in edges], storage)
    if kernel is not None:
        tr.lb_set_launch(kernel, 128, 0, 0)
    rng = np.random.default_rng(11)
    for b, E in enumerate(edges):
        tr.lb_init(b, np.ascontiguousarray(0.03 * rng.standard_normal((3, E, E, E)), tr.np_real))
        if nbeads:
            tr.chain_couple(b, lbt.chain_desc(nbeads), inputs.chain_start(b, nbeads, E))
    faces = sum(18 * E * E for E in edges)
    smp = [torch.from_numpy(0.03 * rng.standard_normal(faces)).to("cuda", tr.real) for _ in range(steps + 2)]
    torch.cuda.synchronize()
    for n in range(steps):
        for j in ((0, 1) if n == 0 else (n + 1,)):
            tr.lb_set_boundary(lbt.LB_ALL_BOXES, j, smp[j])
        tr.lb_step(1)
    out = [tr.deviations(b).astype(np.float64) for b in range(len(edges))]
    tr.lb_sync()
    tr.close()
    return out


@pytest.mark.parametrize("nbeads", [0, 4])
@pytest.mark.parametrize("boxes", [3, 31, 100])
@pytest.mark.parametrize("storage", [1, 2, 3])
def test_runs_of_tiles_match_the_register_kernel(storage, boxes, nbeads):
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    edges = tuple(int(e) for e in np.random.default_rng(boxes).choice([16, 24, 32, 40], boxes))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    per_sm = sum((e ** 3 + 959) // 960 for e in edges) // sms
    assert (per_sm < 4, 4 <= per_sm < 16, per_sm >= 16) == (boxes == 3, boxes == 31, boxes == 100)
    steps = 3
    a = run(lbt, torch, None, edges, storage, nbeads, steps)
    b = run(lbt, torch, lbt.LB_KERNEL_REGISTER, edges, storage, nbeads, steps)
    # values of order 0.1: 40 FP32 roundings a step; 16 bits: those may flip the last bit of what is stored
    ulp = (None, 2.0 ** -24, 2.0 ** -10, 2.0 ** -7)[storage]
    tol = 0.3 * steps * (40 * ulp if storage == 1 else ulp)
    for x, y in zip(a, b):
        assert np.abs(x - y).max() <= tol
