"""Training kernel of the upsampler (lb_mlp_grad, lb_mlp_train_step) at the row
counts where its tiling can go wrong -- one row, one tile less and more than a
row, fewer and more tiles than SMs -- with targets that are and are not
16-byte aligned, against the gradient in FP64 through the bf16 weights the
network runs with.

Tolerance: activations and their gradients are rounded to bf16 (2^-9 relative)
five times along the longest path and enter products of independent roundings,
so the gradient lies within 5 x 2^-8 = 2e-2 of the FP64 one (relative L2); the
loss within the forward's three roundings, 3 x 2^-8."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def reference(torch, master, K, X, T):
    w, o = [], 0
    for shape in ((32, 128), (128,), (128, 128), (128,), (128, 3 * K), (3 * K,)):
        n = int(np.prod(shape))
        t = torch.from_numpy(master[o:o + n].reshape(shape)).cuda()
        w.append((t.to(torch.bfloat16) if len(shape) == 2 else t).double().requires_grad_())
        o += n
    h = torch.relu(torch.relu(X.double() @ w[0] + w[1]) @ w[2] + w[3]) @ w[4] + w[5]
    loss = ((h - T.double()) ** 2).mean()
    return torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, w)]), float(loss)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("rows", [1, 127, 128, 129, 1000, 152 * 128 + 1, 3 * 152 * 128 + 77])
@pytest.mark.parametrize("K", [8, 16])
def test_gradient_at_tile_edges(K, rows, offset):
    import torch

    from paper_0809_4958_gb300 import inputs, lbtracer as lbt
    lbt.load()
    master = inputs.mlp_init(3, K)
    rng = np.random.default_rng(4)
    master = (master + 0.05 * rng.standard_normal(master.size)).astype(np.float32)  # biases and all
    master[24 * 128:32 * 128] = 0.0  # rows of the padding features
    g = torch.Generator(device="cuda").manual_seed(rows)
    X = torch.randn((rows, 32), device="cuda", generator=g).to(torch.bfloat16)
    X[:, 24:] = 0
    buf = torch.randn(rows * 3 * K + 1, device="cuda", generator=g)
    T = buf[offset:offset + rows * 3 * K].view(rows, 3 * K)
    up = lbt.Upsampler(K=K, batch_rows=rows, master=master)
    got, loss = up.grad(X, T)
    ref, ref_loss = reference(torch, master, K, X, T)
    assert float((got.double() - ref).norm() / ref.norm()) <= 2e-2
    assert abs(float(loss) - ref_loss) <= 3 * 2.0 ** -8 * ref_loss
    again, _ = up.grad(X, T)
    assert torch.equal(got, again)  # fixed summation order
    # one Adam step from zero moments moves every parameter by lr g / (|g| + eps)
    up.step(X, T, 1e-3)
    p = up.export()
    w2 = p[128 * 32 * 2:128 * 32 * 2 + 128 * 128 * 2].view(torch.bfloat16).view(128, 128)
    m2 = torch.from_numpy(master[32 * 128 + 128:32 * 128 + 128 + 128 * 128].reshape(128, 128)).cuda()
    g2 = got[32 * 128 + 128:32 * 128 + 128 + 128 * 128].view(128, 128)
    new = (m2 - 1e-3 * g2 / (g2.abs() + 1e-8)).T
    assert float((w2.float() - new).abs().max()) <= 2.0 ** -8 * float(new.abs().max()) + 1e-5


def test_loss_on_a_four_byte_boundary():
    """The loss (8 bytes) may go anywhere in device memory, between floats too."""
    import torch

    from paper_0809_4958_gb300 import inputs, lbtracer as lbt
    lib = lbt.load()
    K, rows = 8, 300
    up = lbt.Upsampler(K=K, batch_rows=rows, master=inputs.mlp_init(3, K))
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn((rows, 32), device="cuda", generator=g).to(torch.bfloat16)
    X[:, 24:] = 0
    T = torch.randn((rows, 3 * K), device="cuda", generator=g)
    _, loss = up.grad(X, T)
    want = float(loss)
    buf = torch.zeros(4, dtype=torch.float32, device="cuda")
    out = torch.zeros(up.nmaster(), dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    rc = lib.lb_mlp_grad(up.ws.data_ptr(), K, rows, X.data_ptr(), T.data_ptr(), rows, out.data_ptr(),
                         buf.data_ptr() + 4, up.stream.cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    assert float(np.frombuffer(buf.cpu().numpy()[1:3].tobytes())[0]) == want
    assert float(buf[0]) == 0.0 and float(buf[3]) == 0.0
