"""A training step whose tensor-core work was late in some block (its bounded
wait ran out): gradient and loss are NaN, and the master weights, the moments
and the inference copy stay as they were."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_0809_4958_gb300 import build
    so = str(tmp_path_factory.mktemp("late") / "train_late.so")
    srcs = [os.path.join(HERE, "train_late.cu")] + [os.path.join(build.CSRC, f) for f in ("lbt_mlp.cu", "lbt_mlp_tc.cu")]
    subprocess.run([build.NVCC] + build.FLAGS + ["-shared", "-o", so] + srcs, check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("nparts,late_at", [(1, None), (1, 0), (152, None), (152, 0), (152, 151), (160, 159)])
@pytest.mark.parametrize("K", [8, 16])
def test_a_late_block_changes_no_weight(lib, K, nparts, late_at):
    import torch

    n = 32 * 128 + 128 + 128 * 128 + 128 + 128 * 3 * K + 3 * K
    g = torch.Generator(device="cuda").manual_seed(1)
    partial = torch.randn((nparts, n), device="cuda", generator=g)
    loss_part = torch.rand(nparts, dtype=torch.float64, device="cuda", generator=g)
    late = torch.zeros(nparts, dtype=torch.int32, device="cuda")
    if late_at is not None:
        late[late_at] = 1
    master, m = torch.randn(n, device="cuda", generator=g), torch.randn(n, device="cuda", generator=g)
    v = torch.rand(n, device="cuda", generator=g)
    params = torch.zeros(1 << 17, dtype=torch.uint8, device="cuda")
    grad, loss = torch.zeros(n, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    before = [t.clone() for t in (master, m, v, params)]
    torch.cuda.synchronize()
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert lib.t_reduce(p(partial), p(loss_part), p(late), nparts, K, p(grad), p(loss), p(master), p(m), p(v), p(params)) == 0
    after = (master, m, v, params)
    if late_at is None:
        want = partial.double().sum(0)
        # a sum of nparts terms in FP32
        assert float((grad.double() - want).abs().max()) <= nparts * 2.0 ** -24 * float(partial.abs().sum(0).max())
        assert abs(float(loss) - float(loss_part.sum())) <= nparts * 2.0 ** -53 * float(loss_part.sum())
        assert all(not torch.equal(a, b) for a, b in zip(after, before))
    else:
        assert bool(torch.isnan(grad).all()) and bool(torch.isnan(loss).all())
        assert all(torch.equal(a, b) for a, b in zip(after, before))


def test_the_training_step_uses_the_flags():
    """An ordinary step writes its blocks' flags before the reduction reads
    them, also into a workspace that held anything before."""
    import torch

    from paper_0809_4958_gb300 import inputs, lbtracer as lbt
    lbt.load()
    K, rows = 16, 1000
    up = lbt.Upsampler(K=K, batch_rows=rows, master=inputs.mlp_init(3, K))
    grads = up.nmaster() * 4
    start = 4 * ((grads + 255) // 256 * 256)  # behind master, moments and gradient
    end = up.ws.numel() - up.params.numel()
    up.ws[start:end] = 0xFF
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn((rows, 32), device="cuda", generator=g).to(torch.bfloat16)
    X[:, 24:] = 0
    T = torch.randn((rows, 3 * K), device="cuda", generator=g)
    got, loss = up.grad(X, T)
    assert bool(torch.isfinite(got).all()) and np.isfinite(float(loss))
