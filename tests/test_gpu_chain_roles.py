"""The default FP64 bead layout (work split by warp role) against one lane per
bead (lb_set_bead_launch(1, 1)) at the chain lengths where the split can go
wrong: one to three beads, a warp's 32 and its neighbours, 128 (the most the
four roles cover) and beyond.  Both add the same pair forces in another order:
50 substeps of some 30 roundings a step, forces of order 30 against masses of 1
on positions of order 40, growing by less than 10 a step."""
import numpy as np
import pytest

from test_gpu_chain_order import serpentine

pytestmark = pytest.mark.gpu


def run(lbt, torch, lanes, N, kT, steps):
    E = 40 if N <= 33 else 64
    from paper_0809_4958_gb300 import inputs
    tr = lbt.Tracers([lbt.box_desc(E, 0.8, nbeads=N)], lbt.LB_STORE_F64)
    if lanes:
        tr.lb_set_bead_launch(lanes, 1)
    rng = np.random.default_rng(N)
    tr.lb_init(0, 0.02 * rng.standard_normal((3, E, E, E)))
    # folded, rows touching: lists and contacts of every kind occur, bonds near their rest length
    pos = serpentine(N, E, max(4, int(N ** 0.5)))
    tr.chain_couple(0, lbt.chain_desc(N, kT=kT, seed=11), pos, np.array([0.3, 0.0, 0.0]) + 0.03 * rng.standard_normal((N, 3)))
    face = torch.zeros((18, E, E), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    tr.lb_set_boundary(0, 0, face)
    out = []
    for n in range(steps):
        tr.lb_set_boundary(0, n + 1, face)
        tr.lb_step(1)
        out.append(np.concatenate(tr.chain(0, N)))
    tr.close()
    return out


@pytest.mark.parametrize("kT", [0.0, 1e-3])
@pytest.mark.parametrize("N", [1, 2, 3, 31, 32, 33, 64, 97, 128, 129, 200])
def test_roles_match_one_lane_per_bead(N, kT):
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    a, b = run(lbt, torch, 0, N, kT, 3), run(lbt, torch, 1, N, kT, 3)
    for n, (x, y) in enumerate(zip(a, b)):
        assert np.abs(x - y).max() <= 50 * 30 * 30 * 40 * 2.0 ** -53 * 10.0 ** n
