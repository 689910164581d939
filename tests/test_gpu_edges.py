"""The staged x-face samples of the stream-collide at the sizes where they can
go wrong: edges whose sample runs just fit and just do not fit the room of a
stage, one to four samples with a weight, several boxes of different edges in
one launch with and without chains -- against the register kernel, which loads
every boundary sample from global memory (same FP32 collision up to its order
of additions: velocities of order 0.05 over six steps of about 40 roundings)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def run(lbt, torch, kernel, edges, interp, K, storage, periodic, steps=6):
    descs = [lbt.box_desc(E, 0.8, periodic=periodic, time_interp=interp, K=K) for E in edges]
    tr = lbt.Tracers(descs, storage)
    if kernel is not None:
        tr.lb_set_launch(kernel, 128 if kernel == lbt.LB_KERNEL_REGISTER else 0, 0, 0)
    rng = np.random.default_rng(5)
    for b, E in enumerate(edges):
        tr.lb_init(b, np.ascontiguousarray(0.05 * rng.standard_normal((3, E, E, E)), tr.np_real))
    faces = sum(18 * E * E for E in edges)
    smp = [torch.from_numpy(0.05 * rng.standard_normal(faces)).to("cuda", tr.real) for _ in range(steps + 3)]
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


@pytest.mark.parametrize("interp,K", [(0, 1), (0, 3), (1, 2)])
@pytest.mark.parametrize("edges", [(8,), (16,), (24,), (40,), (48,), (56,), (72,), (24, 64, 8, 48)])
@pytest.mark.parametrize("storage", [1, 2])
def test_staged_faces_match_the_register_kernel(edges, interp, K, storage):
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    for periodic in ((False, False, False), (False, True, False)):
        a = run(lbt, torch, None, edges, interp, K, storage, periodic)
        b = run(lbt, torch, lbt.LB_KERNEL_REGISTER, edges, interp, K, storage, periodic)
        # FP32: values of order 0.05, 6 steps x 40 roundings; 16 bits: those may flip the last bit of what is stored
        tol = 0.3 * 6 * 40 * 2.0 ** -24 if storage == 1 else 0.3 * 6 * 2.0 ** -10
        for x, y in zip(a, b):
            assert np.abs(x - y).max() <= tol


def test_many_boxes_claimed_in_runs():
    """More than 64 tiles to an SM in boxes of many sizes: the runs of tiles a
    producer claims cross box borders."""
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    edges = tuple(int(e) for e in np.random.default_rng(1).choice([8, 24, 40, 64], 120))
    assert sum((e ** 3 + 959) // 960 for e in edges) > 64 * 152
    a = run(lbt, torch, None, edges, 0, 1, 1, (False,) * 3, steps=3)
    b = run(lbt, torch, lbt.LB_KERNEL_REGISTER, edges, 0, 1, 1, (False,) * 3, steps=3)
    for x, y in zip(a, b):
        assert np.abs(x - y).max() <= 0.3 * 3 * 40 * 2.0 ** -24
