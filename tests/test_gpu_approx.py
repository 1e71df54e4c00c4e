"""The square roots, exponential and reciprocal that the kernels take in place of
the exact ones, over the ranges of their arguments, against numpy in more bits and,
for the 32-bit ones, against CUDA's own sqrtf and expf (through torch).

Bars, relative: 2^-24 and a twentieth for the square root (a Newton step squares the
estimate's error, 2^-22 at most, so the last rounding is what is left); for exp(-a) the
2^-22 that PTX states for ex2.approx and 2^-24 for each of its three roundings here;
for the 64-bit ones one rounding, 2^-53 (reciprocal; the same twentieth) and 2^-52 (reciprocal
square root: its last step rounds a product first)."""
import numpy as np
import pytest

from test_gpu_gp_device import S, ctx, torch  # noqa: F401
from workloads import Stream

pytestmark = pytest.mark.gpu


def apply(S, ctx, which, x):  # noqa: F811
    x = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    y = torch.full_like(x, 7.0)
    S.scoot_probe_math(ctx, which, x, y)
    ctx.check()
    return y.cpu().numpy()


def spread(n, lo, hi, name):
    """n values, their logarithm uniform from 2^lo to 2^hi, and the powers of two between."""
    e = lo + (hi - lo) * Stream(n, name).uniform(n)
    return np.concatenate([np.exp2(np.floor(e)) * (1 + (e - np.floor(e))), np.exp2(np.arange(int(lo), int(hi)))])


def test_square_root(S, ctx):  # noqa: F811
    x = spread(1 << 20, -99.0, 127.0, "sqrt").astype(np.float32)
    got, want = apply(S, ctx, 0, x).astype(np.float64), np.sqrt(x.astype(np.float64))
    worst = np.abs(got / want - 1).max()
    ours = np.abs(torch.sqrt(torch.from_numpy(x).cuda()).cpu().numpy().astype(np.float64) / want - 1).max()
    print(f"sqrt_acc {worst * 2 ** 24:.3f}, sqrtf {ours * 2 ** 24:.3f} of 2^-24")
    assert worst <= 1.05 * 2.0 ** -24
    small = np.concatenate([[0.0], spread(1 << 10, -126.0, -99.0, "small")]).astype(np.float32)
    assert np.abs(apply(S, ctx, 0, small) - np.sqrt(small.astype(np.float64))).max() <= 2e-15
    bad = apply(S, ctx, 0, np.array([np.nan, np.inf], np.float32))
    assert np.isnan(bad).all()  # what the covariance makes of infinity in the end: inf times exp(-inf)


def test_exponential(S, ctx):  # noqa: F811
    a = np.concatenate([[0.0], 86.0 * Stream(3, "exp").uniform(1 << 20), spread(1 << 18, -40.0, 6.0, "exp small")]).astype(np.float32)
    got, want = apply(S, ctx, 1, a).astype(np.float64), np.exp(-a.astype(np.float64))
    worst = np.abs(got / want - 1).max()
    ours = np.abs(torch.exp(-torch.from_numpy(a).cuda()).cpu().numpy().astype(np.float64) / want - 1).max()
    print(f"exp_acc {worst * 2 ** 24:.3f}, expf {ours * 2 ** 24:.3f} of 2^-24")
    assert worst <= 2.0 ** -22 + 3 * 2.0 ** -24
    far = apply(S, ctx, 1, np.array([88.0, 104.0, 1e4, 1e19], np.float32))
    assert (far >= 0).all() and (far <= np.exp(-87.9)).all() and (far[1:] == 0).all()
    assert np.isnan(apply(S, ctx, 1, np.array([np.nan], np.float32))).all()


@pytest.mark.parametrize("which,lo,hi,bar", [(2, -1000.0, 1000.0, 1.05 * 2.0 ** -53), (3, -99.0, 99.0, 2.0 ** -52),
                                             (3, -1000.0, 1000.0, 2.0 ** -52)])
def test_reciprocals(S, ctx, which, lo, hi, bar):  # noqa: F811
    v = spread(1 << 18, lo, hi, "reciprocal")
    long = v.astype(np.longdouble)
    want = 1 / long if which == 2 else 1 / np.sqrt(long)
    worst = float(np.abs(apply(S, ctx, which, v).astype(np.longdouble) / want - 1).max())
    print(f"which={which} 2^{lo:.0f}..2^{hi:.0f}: {worst * 2 ** 53:.3f} of 2^-53")
    assert worst <= bar
