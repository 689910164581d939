"""The training loss as a sum: a network whose last layer is zero predicts its
output bias, chosen with 16 significant bits so that the two bf16 parts the
tensor cores add hold it exactly.  The loss is then the sum of the squares of
FP32 differences, known on the CPU; it was an FP64 sum of exact squares from
the beginning, and has to be as good over the whole range of the targets.

Tolerance: squares are exact in FP64 (24-bit differences); a sum of positive
terms in FP64 loses at most 2^-53 per addition on the path of a term: the
columns of a thread over its tiles (24 x 4 here), five shuffles, eight warps,
at most 160 blocks in five strides and five shuffles, and the scale."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-12, 1e-21, 1e25])
@pytest.mark.parametrize("K,rows", [(8, 1), (16, 129), (16, 16384), (8, 3 * 152 * 128 + 77)])
def test_loss_is_the_sum_of_squares(K, rows, size):
    import torch

    from paper_0809_4958_gb300 import inputs, lbtracer as lbt
    lbt.load()
    nout = 3 * K
    master = inputs.mlp_init(3, K)
    master[-nout - 128 * nout:] = 0.0
    rng = np.random.default_rng(rows)
    bias = np.zeros(nout, np.float32)
    if size >= 1e-12:
        bias = np.float32(min(size, 1.0)) * (rng.integers(2 ** 15, 2 ** 16, nout) * 2.0 ** -16).astype(np.float32)
        bias = (bias.view(np.uint32) & np.uint32(0xFFFFFF00)).view(np.float32)  # 16 significant bits
    master[-nout:] = bias
    up = lbt.Upsampler(K=K, batch_rows=rows, master=master)
    T = (size * rng.standard_normal((rows, nout))).astype(np.float32)
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn((rows, 32), device="cuda", generator=g).to(torch.bfloat16)
    X[:, 24:] = 0
    _, loss = up.grad(X, torch.from_numpy(T).cuda())
    d = (bias[None, :] - T).astype(np.float64)  # an FP32 subtraction
    scale = float(np.float32(1.0) / np.float32(rows * nout))
    want = float(np.sum((d * d).astype(np.longdouble))) * scale
    got = float(loss)
    assert abs(got - want) <= (24 * 4 + 5 + 8 + 5 + 5 + 2) * 2.0 ** -53 * want, (got, want)
