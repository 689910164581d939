"""Upsampler targets (lb_mlp_targets) at the block edges of its kernel -- face
sets that are and are not whole blocks of 32 rows, substep counts below, at and
above one round of 16 -- against the Hermite residual in FP64.

Tolerance: the residual (of order 64 here) is a difference of values of order
64 / u_max x 0.05 = 64 in FP32 with some ten roundings: 64 x 10 x 2^-24."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("E,K", [(2, 1), (3, 16), (8, 8), (9, 17), (24, 16), (10, 40)])
@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_targets_are_the_hermite_residual(E, K, first, dtype):
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    u_max = 0.05
    rng = np.random.default_rng(E * 100 + K)
    smp = [torch.from_numpy(rng.uniform(-u_max, u_max, (6, 3, E, E))).to("cuda", getattr(torch, dtype)) for _ in range(4)]
    fine = torch.from_numpy(rng.uniform(-u_max, u_max, (K + 1, 6, 3, E, E))).to("cuda", getattr(torch, dtype))
    T = lbt.mlp_targets(*smp, fine, E, K, first, u_max).double()
    sp, s0, s1, s2 = (s.double() for s in smp)
    m0, m1 = (s1 - s0 if first else 0.5 * (s1 - sp)), 0.5 * (s2 - s0)
    ref = []
    for s in range(1, K + 1):
        th = s / K
        herm = ((2 * th ** 3 - 3 * th ** 2 + 1) * s0 + (th ** 3 - 2 * th ** 2 + th) * m0 + (-2 * th ** 3 + 3 * th ** 2) * s1
                + (th ** 3 - th ** 2) * m1)
        ref.append((fine[s].double() - herm).permute(0, 2, 3, 1).reshape(-1, 3) * (64.0 / u_max))
    assert float((T - torch.cat(ref, 1)).abs().max()) <= 64 * 10 * 2.0 ** -24
