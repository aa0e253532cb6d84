"""The device sums against exact arithmetic.

With e the exponent of the largest value and u = 2^(e - 63), a warp's integer sum of 32 M values truncates each value by
less than u and drops less than 2^SH u at its end (SH = 6 for M = 1, else 9); a block's sum truncates each warp's by less
than 2^SH u more, and its one rounding is 2^-53 of the sum (with the six bits a large sum drops, 2^-56 more). Values next
to the subnormals or to overflow take a floating-point tree of M - 1 + 5 + 5 additions, each 2^-53 of the sum of
magnitudes. These bounds are the tolerances.
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    from paper_2005_01275_gb300 import build
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_math.cu")
    so = str(tmp_path_factory.mktemp("device_math") / "device_math.so")
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", src, "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def block_sums(dev, v):
    """v: [blocks, NV, M, threads] -> [blocks, NV]"""
    v = np.ascontiguousarray(v, dtype=np.float64)
    out = np.full(v.shape[:2], 7.0)
    assert dev.block_sums_host(ptr(v), ptr(out), v.shape[0], v.shape[3], v.shape[1], v.shape[2]) == 0
    return out


def grid_sums(dev, v, cluster=0):
    """v: [2, blocks, threads] -> [blocks, 2]"""
    v = np.ascontiguousarray(v, dtype=np.float64)
    out = np.full((v.shape[1], 2), 7.0)
    assert dev.grid_sums_host(ptr(v), ptr(out), v.shape[1], v.shape[2], cluster) == 0
    return out


def exact(v, f=lambda x: x):
    t = 0
    for x in np.asarray(v, dtype=np.float64).reshape(-1).tolist():
        n, d = f(x).as_integer_ratio()
        t += n << (1075 - d.bit_length())
    return Fraction(t, 2 ** 1074)


def magnitude(v):
    return exact(v, abs)


def bound(v):
    """Of a block's sum of v [M, threads]."""
    m, nw = v.shape[0], v.shape[1] // 32
    top = float(np.abs(v).max())
    e = int(np.frexp(top)[1]) - 1
    tree = any(0 < np.abs(w).max() < 2.0 ** -950 or np.abs(w).max() > 2.0 ** 1000
               for w in v.reshape(m, nw, 32).transpose(1, 0, 2))
    if tree:
        return (m + 9) * Fraction(1, 2 ** 53) * magnitude(v) * Fraction(101, 100)
    sh = 6 if m == 1 else 9
    return nw * (32 * m + 2 * 2 ** sh) * Fraction(2) ** (e - 63) + Fraction(9, 8) * abs(exact(v)) / 2 ** 53


def draws(rng, m, threads):
    """[M, threads] arrays of the kinds the solvers sum, and of what they must not lose."""
    shape = (m, threads)
    u = rng.uniform(-1, 1, shape)
    wide = u * 2.0 ** rng.integers(-60, 60, shape)
    idle = u ** 2
    idle[:, threads - 32:] = 0.0                      # a warp that holds nothing
    lone = np.zeros(shape)
    lone[m - 1, threads // 2] = -0.3
    cancel = wide.copy()
    cancel[:, threads // 2:] = -cancel[:, :threads // 2]
    mixed = u ** 2 * np.repeat(2.0 ** rng.integers(-200, 200, threads // 32), 32)   # a scale for each warp
    apart = np.zeros(shape)
    apart[:, 0], apart[:, threads - 1] = 1.0, 2.0 ** -1030   # a subnormal in a warp of its own
    return dict(signed=u, squares=u ** 2, wide=wide, idle=idle, zero=np.zeros(shape), lone=lone, cancel=cancel,
                mixed=mixed, small=u * 2.0 ** -1030, tiny=u * 2.0 ** -960, large=u * 2.0 ** 1013, apart=apart)


@pytest.mark.parametrize("nv,m", [(1, 1), (3, 1), (1, 4), (2, 5)])
@pytest.mark.parametrize("threads", [64, 256, 512, 1024])
def test_block_sums_stay_within_their_bound(dev, nv, m, threads):
    rng = np.random.default_rng(11 * m + threads)
    for _ in range(4):
        cases = [draws(rng, m, threads) for _ in range(nv)]
        for name in cases[0]:
            v = np.stack([c[name] for c in cases])
            s = block_sums(dev, v[None])[0]
            for k in range(nv):
                assert abs(Fraction(float(s[k])) - exact(v[k])) <= bound(v[k]), (name, k)


@pytest.mark.parametrize("nw", [4, 6, 16])
def test_an_idle_warp_leaves_the_sum_exact(dev, nw):
    """One warp's values add up to 2^53, an even number of others hold a one each and one holds nothing (the solvers'
    server warp): every value is a multiple of the window's last bit, so the integer sum is exact, where additions in
    double lose the ones."""
    for idle in (0, 1, nw - 1):
        v = np.zeros(32 * nw)
        busy = [w for w in range(nw) if w != idle]
        busy = busy[:1 + (len(busy) - 1) // 2 * 2]
        for w in busy:
            v[32 * w + 3] = 1.0
        v[32 * busy[0] + 5] = 2.0 ** 53 - 1
        want = 2.0 ** 53 + (len(busy) - 1)
        assert block_sums(dev, v[None, None, None])[0, 0] == want
        for blocks, cluster in ((3, 0), (4, 1)):
            g = np.zeros((2, blocks, 32 * nw))
            g[0, 1], g[1, 2] = v, -v
            assert (grid_sums(dev, g, cluster) == [want, -want]).all()


@pytest.mark.parametrize("value,want", [(np.inf, np.inf), (-np.inf, -np.inf), (np.nan, np.nan)])
def test_infinities_and_nan_pass_through(dev, value, want):
    rng = np.random.default_rng(5)
    for m in (1, 4):
        for lane in (0, 45, 255):
            v = rng.uniform(-1, 1, (1, 1, m, 256))
            v[0, 0, m - 1, lane] = value
            np.testing.assert_equal(block_sums(dev, v)[0, 0], want)
            v[0, 0, 0, (lane + 77) % 256] = -np.inf if value == np.inf else np.nan
            if value != -np.inf:
                assert np.isnan(block_sums(dev, v)[0, 0])
    g = rng.uniform(-1, 1, (2, 5, 128))
    g[1, 3, 64] = value
    out = grid_sums(dev, g)
    np.testing.assert_equal(out[:, 1], np.full(5, want))
    assert np.isfinite(out[:, 0]).all()


@pytest.mark.parametrize("blocks,cluster", [(1, 0), (3, 0), (152, 0), (160, 0), (161, 0), (304, 0), (1, 1), (2, 1), (8, 1)])
def test_grid_sums_stay_within_their_bound(dev, blocks, cluster):
    """Every block gets the same bits. Block sums as above, then one warp's sum of up to 160 of them (M = 5); the blocks
    beyond are added to those first, one rounding each."""
    rng = np.random.default_rng(blocks)
    threads = 128
    for name in ("signed", "squares", "wide", "cancel", "mixed", "zero", "lone"):
        v = np.stack([np.stack([draws(rng, 1, threads)[name][0] for _ in range(blocks)]) for _ in range(2)])
        v[:, blocks // 2, 64:96] = 0.0
        got = grid_sums(dev, v, cluster)
        assert (got == got[0]).all(), name
        for k in range(2):
            err = sum(bound(b[None]) for b in v[k])
            parts = [exact(b) for b in v[k]]
            top = float(max(abs(p) for p in parts))
            e = int(np.frexp(top)[1])
            err += (32 * 5 + 2 ** 9) * Fraction(2) ** (e - 63) + Fraction(9, 8) * abs(sum(parts)) / 2 ** 53
            err += max(0, -(-(blocks - 160) // 32)) * sum(abs(p) for p in parts) / 2 ** 53
            assert abs(Fraction(float(got[0, k])) - sum(parts)) <= err * Fraction(101, 100), name


def scalar(dev, op, a, b=None):
    a = np.ascontiguousarray(a, dtype=np.float64)
    v = np.concatenate([a, a if b is None else np.asarray(b, dtype=np.float64)])
    out = np.empty(a.size)
    assert dev.scalar_host(ptr(v), ptr(out), a.size, op) == 0
    return out


def over_the_range(rng, n):
    """Signed values of every exponent, and those next to the bounds of the short forms and of the format."""
    x = rng.uniform(1, 2, n) * 2.0 ** rng.integers(-1022, 1024, n)
    edges = [2.0 ** e for k in (-1022, -961, -960, -959, -481, -480, -1, 0, 1, 480, 481, 959, 960, 961, 1023)
             for e in (k - 1, k) if e >= -1074]
    x = np.concatenate([x, edges, np.nextafter(edges, 0), np.nextafter(edges, np.inf), [5e-324, 1e-310, np.inf, np.nan, 0.0]])
    return np.where(rng.uniform(size=x.size) < 0.5, -x, x)


def relative_error(got, num, den):
    return abs(Fraction(float(got)) * Fraction(float(den)) - Fraction(float(num))) / abs(Fraction(float(num)))


def test_reciprocal_and_quotient(dev):
    """Within the short forms' ranges (2^-960 .. 2^960; both operands in 2^-480 .. 2^480): half a unit of the last place and
    what the truncated series leaves, 2^-60, or the quotient's second-order terms. Outside them the plain operation."""
    rng = np.random.default_rng(2)
    a = over_the_range(rng, 4000)
    with np.errstate(all="ignore"):
        for got, num, den, top in ((scalar(dev, 0, a), np.ones_like(a), a, 961),):
            for g, x, y in zip(got, num, den):
                if 2.0 ** -960 <= abs(y) < 2.0 ** top:
                    assert relative_error(g, x, y) <= Fraction(1, 2 ** 53) + Fraction(1, 2 ** 59), y
                else:
                    np.testing.assert_equal(g, x / y)
        b = rng.permutation(over_the_range(rng, 4000))
        a[:1000], b[:1000] = a[:1000] % 7 + 0.1, b[:1000] % 5 + 0.3
        a, b = np.concatenate([a, [2.0 ** 900, 2.0 ** -900, 1.5 * 2.0 ** 700]]), np.concatenate([b, [2.0 ** -900, 2.0 ** 900, 2.0 ** -400]])
        got = scalar(dev, 1, a, b)
        short = (np.abs(a) >= 2.0 ** -480) & (np.abs(a) < 2.0 ** 481) & (np.abs(b) >= 2.0 ** -480) & (np.abs(b) < 2.0 ** 481)
        np.testing.assert_array_equal(got[~short], (a / b)[~short])
        assert short.sum() > 1000
        for g, x, y in zip(got[short], a[short], b[short]):
            assert relative_error(g, x, y) <= Fraction(1, 2 ** 53) + Fraction(1, 2 ** 80), (x, y)


def test_conversions_by_bits(dev):
    rng = np.random.default_rng(3)
    a = np.concatenate([over_the_range(rng, 4000), rng.standard_normal(4000) * 2.0 ** rng.integers(-155, 130, 4000),
                        np.float32(1.5) + np.arange(-4, 5) * 2.0 ** -25, [2.0 ** 128 - 2.0 ** 103, 2.0 ** 128 - 2.0 ** 104]])
    with np.errstate(all="ignore"):
        f = a.astype(np.float32)
    np.testing.assert_array_equal(scalar(dev, 2, a), f.astype(np.float64))
    np.testing.assert_array_equal(scalar(dev, 3, f.astype(np.float64)), f.astype(np.float64))
