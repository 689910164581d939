"""The kernels' own reciprocal, quotient and square root over random mantissas
and the whole exponent range, zeros, infinities and NaN among them, against the
correctly rounded operations of the CPU (which CUDA's division and square root
give too).  Bounds: the reciprocal and the square root within one ulp where
they are used (normal argument and result), the quotient within one ulp, two
where the numerator is within 2^26 of the smallest normal number, and equal
where it falls back to the division."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    import torch

    from paper_0809_4958_gb300 import build
    assert torch.cuda.is_available()
    so = str(tmp_path_factory.mktemp("devmath") / "device_math.so")
    subprocess.run([build.NVCC] + build.FLAGS + ["-shared", "-o", so, os.path.join(HERE, "device_math.cu")], check=True)
    lib = ctypes.CDLL(so)

    def call(name, out_dtype, *arrays):
        ts = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]
        n = len(arrays[-1])
        y = torch.zeros(n, dtype=torch.float64 if out_dtype == np.float64 else torch.float32, device="cuda")
        torch.cuda.synchronize()
        args = [ctypes.c_void_p(t.data_ptr()) for t in ts] + [ctypes.c_void_p(y.data_ptr()), n]
        assert getattr(lib, name)(*args) == 0
        return y.cpu().numpy()

    return call


def draw(rng, n, dtype):
    """Random bit patterns: every exponent, both signs, subnormals, zeros, infinities, NaN."""
    if dtype == np.float64:
        x = rng.integers(0, 2 ** 64, n, dtype=np.uint64).view(np.float64)
    else:
        x = rng.integers(0, 2 ** 32, n, dtype=np.uint32).view(np.float32)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, np.finfo(dtype).max, np.finfo(dtype).tiny,
                        np.finfo(dtype).smallest_subnormal, 1.0, -1.0], dtype)
    x[:len(special)] = special
    return x


def ulps(got, want):
    with np.errstate(all="ignore"):
        unit = np.spacing(np.abs(want)).astype(np.longdouble)
    return np.abs(got.astype(np.longdouble) - want.astype(np.longdouble)) / unit


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_reciprocal(dev, dtype):
    rng = np.random.default_rng(1)
    x = draw(rng, 1 << 20, dtype)
    tiny = np.finfo(dtype).tiny
    with np.errstate(all="ignore"):
        want = (dtype(1) / x).astype(dtype)
    got = dev("t_inverse_f64" if dtype == np.float64 else "t_inverse_f32", dtype, x)
    ok = np.isfinite(x) & (np.abs(x) >= tiny) & np.isfinite(want) & (np.abs(want) >= tiny)
    assert ok.sum() > 1 << 19
    assert ulps(got[ok], want[ok]).max() <= 1


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_quotient(dev, dtype):
    rng = np.random.default_rng(2)
    n = 1 << 20
    rho, j = draw(rng, n, dtype), draw(rng, n, dtype)
    j[:100], rho[:100] = np.repeat(j[:10], 10), np.tile(rho[:10], 10)  # all pairs of the special values
    half = slice(n // 2, 3 * n // 4)  # numerators of the denominator's size
    with np.errstate(all="ignore"):
        j[half] = (rho[half] * rng.uniform(-1, 1, n // 4)).astype(dtype)
    quarter = slice(3 * n // 4, n)  # densities beyond the reciprocal's range
    rho[quarter] = (np.finfo(dtype).max * rng.uniform(0.25, 1, n // 4)).astype(dtype)
    with np.errstate(all="ignore"):
        want = (j / rho).astype(dtype)
    got = dev("t_ratio_f64" if dtype == np.float64 else "t_ratio_f32", dtype, j, rho)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    inf = np.isinf(want) | np.isinf(j) | np.isinf(rho) | (rho == 0)
    nan = np.isnan(want)
    assert np.array_equal(got[inf & ~nan], want[inf & ~nan])
    ok = ~(inf | nan)
    off = ulps(got[ok], want[ok])
    near = np.abs(j[ok]) < np.finfo(dtype).tiny * dtype(2.0) ** 26
    assert off[~near].max() <= 1
    assert off.max() <= 2
    beyond = np.zeros(n, bool)
    beyond[quarter] = True
    assert off[beyond[ok]].max() <= 1


def test_square_root(dev):
    rng = np.random.default_rng(3)
    x = draw(rng, 1 << 20, np.float64)
    x[1 << 18:] = np.exp(rng.uniform(np.log(1e-32), np.log(1e32), x.size - (1 << 18)))
    with np.errstate(all="ignore"):
        want = np.sqrt(x)
    got = dev("t_sqrt", np.float64, x)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    edge = ~np.isfinite(want) | (x == 0)
    assert np.array_equal(got[edge & ~np.isnan(want)], want[edge & ~np.isnan(want)])
    assert ulps(got[~edge], want[~edge]).max() <= 1


def test_widening_is_exact(dev):
    x = draw(np.random.default_rng(4), 1 << 20, np.float32)
    got = dev("t_widen", np.float64, x)
    with np.errstate(all="ignore"):
        want = x.astype(np.float64)
    nan = np.isnan(want)
    assert np.isnan(got[nan]).all()
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))


@pytest.mark.parametrize("rl", [0.36, 1.4224, 4.0])
@pytest.mark.parametrize("span", [1.0, 60.0, 200.0, 5000.0])
def test_neighbour_lists_hold_every_pair_within_their_radius(dev, rl, span):
    """The FP32 lists of FP64 chains: a pair just inside the FP64 radius is
    listed however far from bead 0 it lies (a margin of 1e-5 of the radius
    alone misses pairs from some 128 units on), one clearly outside is not."""
    rng = np.random.default_rng(5)
    n = 1 << 18
    a = rng.uniform(-span, span, (n, 3))
    e = rng.standard_normal((n, 3))
    e /= np.linalg.norm(e, axis=1)[:, None]
    inside = a + rl * (1 - 1e-9) * e
    far = a + (rl * (1 + 2e-5) + 2e-6 * span) * e
    r2 = np.full(n, rl * rl)
    keep = ((inside - a) ** 2).sum(1) < r2
    assert keep.mean() > 0.9
    got = dev("t_listed", np.float32, a, inside, r2)
    f = lambda x: x.astype(np.float32)  # noqa: E731
    d = f(a) - f(inside)
    former = (d * d).sum(1) < np.float32(rl * rl) * np.float32(1 + 2e-5)
    print("span %g, radius %g: %d of %d pairs missed by a relative margin alone" % (span, rl, (~former[keep]).sum(), keep.sum()))
    assert (got[keep] == 1).all()
    assert (dev("t_listed", np.float32, a, far, r2) == 0).all()
