"""Targets of a face set whose rows do not fit 32-bit indexes (E = 18920, one
substep, 6 E^2 = 2.1 G rows): constant samples give the same target in every
row, the last ones among them.  Holds some 103 GB; skipped where they are not
free."""
import pytest

pytestmark = pytest.mark.gpu


def test_rows_beyond_32_bits():
    import torch

    from paper_0809_4958_gb300 import lbtracer as lbt
    lbt.load()
    E, K, u_max = 18920, 1, 0.5
    rows = 6 * E * E
    assert rows > 2 ** 31
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 130 * 10 ** 9:
        pytest.skip("needs 130 GB of free device memory")
    s = torch.empty(18 * E * E, dtype=torch.float32, device="cuda").fill_(0.25)
    fine = torch.empty(2 * 18 * E * E, dtype=torch.float32, device="cuda").fill_(0.5)
    T = torch.empty((rows, 3 * K), dtype=torch.float32, device="cuda").fill_(float("nan"))
    lbt.mlp_targets(s, s, s, s, fine, E, K, 0, u_max, out=T)
    want = (0.5 - 0.25) * 64.0 / u_max  # exact: constants of two bits, Hermite of a constant record
    flat = T.view(-1)
    step = 1 << 28
    for a in range(0, flat.numel(), step):
        assert bool((flat[a:a + step] == want).all()), a
    del s, fine, T, flat
    torch.cuda.empty_cache()
