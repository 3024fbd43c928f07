"""The arithmetic helpers under the pair sums, one by one: reciprocals from
the hardware's estimate, the quintic's polynomial pieces, conversions on the
integer pipe, anchor separations.  tests/pair_numerics.cu runs them on
arrays; it is compiled here against the library's headers."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2107_01276_gb300 import build as B
from tests.helpers import cuda_ok

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def num(tmp_path_factory):
    if not cuda_ok():
        pytest.skip("no CUDA device")
    import os
    so = tmp_path_factory.mktemp("numerics") / "pair_numerics.so"
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "pair_numerics.cu")
    r = subprocess.run([B._nvcc()] + B.NVCC_FLAGS + ["-shared", "-I", B.CSRC, "-o", str(so), src],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(str(so))

    def call(name, arrays, outs, *more):
        import torch
        dev = [torch.from_numpy(a).cuda() for a in arrays]
        res = [torch.zeros(o[0], dtype=o[1], device="cuda") for o in outs]
        torch.cuda.synchronize()
        args = [ctypes.c_void_p(t.data_ptr()) for t in dev]
        post = [ctypes.c_void_p(t.data_ptr()) for t in res]
        st = getattr(L, name)(ctypes.c_int(len(arrays[0])), *args, *more, *post)
        assert st == 0, st
        return [t.cpu().numpy() for t in res]
    return call


def _f64():
    import torch
    return torch.float64


def _f32():
    import torch
    return torch.float32


def _normals(lo, hi, n=200000, seed=1):
    """Normal doubles with binary exponents lo .. hi - 1, random and edge
    mantissas."""
    rng = np.random.default_rng(seed)
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    m[:n // 8] = rng.choice([0, 1, 2, (1 << 52) - 1, (1 << 52) - 2, 1 << 51], n // 8)
    e = rng.integers(lo + 1023, hi + 1023, n).astype(np.uint64)
    return ((e << np.uint64(52)) | m).view(np.float64)


@pytest.mark.parametrize("lo,hi", [(-8, 8), (-1022, 1022)])
@pytest.mark.parametrize("name", ["num_frcp", "num_frsqrt"])
def test_reciprocals_within_one_and_a_half_ulp(num, name, lo, hi):
    """Relative to the spacing at the result (at most 2^-52 of it), against
    extended precision (whose own error is below 2^-60)."""
    x = _normals(lo, hi)
    (got,) = num(name, [x], [(len(x), _f64())])
    big = np.longdouble(x)
    ref = 1 / big if name == "num_frcp" else 1 / np.sqrt(big)
    ulp = np.longdouble(np.spacing(np.float64(ref)))
    assert np.finfo(np.longdouble).nmant >= 63
    assert (np.abs(np.longdouble(got) - ref) / ulp).max() <= 1.5


def test_is_normal(num):
    import torch
    t = np.float64(2.0) ** -1022
    x = np.array([0.0, 5e-324, np.nextafter(t, 0), t, 1.0, np.inf, np.nan, -np.nan])
    (got,) = num("num_is_normal", [x], [(len(x), torch.int32)])
    assert got.tolist() == [0, 0, 0, 1, 1, 1, 1, 1]


def test_quintic_pieces(num):
    """w = a^5 - 6 b^5 + 15 c^5 and s = a^4 - 6 b^4 + 15 c^4 of the clipped
    a = 3 - q, b = 2 - q, c = 1 - q.  Horner's rule with 0 <= t <= 1: ten
    roundings of partial sums below 146 (w) and 56 (s)."""
    rng = np.random.default_rng(2)
    q = np.concatenate([rng.uniform(0, 3.2, 100000), [0.0, 1.0, 2.0, 3.0, np.inf],
                        np.nextafter([1.0, 2.0, 3.0], 0), np.nextafter([1.0, 2.0, 3.0], 9)])
    w, s = num("num_qs", [q], [(len(q), _f64())] * 2)
    a, b, c = (np.longdouble(np.clip(k - np.longdouble(q), 0, None)) for k in (3, 2, 1))
    assert np.abs(w - (a ** 5 - 6 * b ** 5 + 15 * c ** 5)).max() <= 10 * 146 * 2.0 ** -53
    assert np.abs(s - (a ** 4 - 6 * b ** 4 + 15 * c ** 4)).max() <= 10 * 56 * 2.0 ** -53
    outer = q >= 2
    assert (np.abs(w - a ** 5) <= 6 * 2.0 ** -53 * a ** 5)[outer].all()
    assert (w[q >= 3] == 0).all() and (s[q >= 3] == 0).all()


def _bits(a):
    return a.view(np.uint64 if a.dtype.itemsize == 8 else np.uint32)


def _same_or_both_nan(a, b):
    return ((_bits(a) == _bits(b)) | (np.isnan(a) & np.isnan(b))).all()


@np.errstate(invalid="ignore", over="ignore")
def _doubles_around_floats():
    """Random bit patterns, every float exponent, ties between floats, one
    bit to either side of them, carries into the next exponent, the ends of
    the normal floats, infinities and NaN; both signs."""
    rng = np.random.default_rng(3)
    f = rng.integers(0, 1 << 31, 60000, dtype=np.uint32)
    f[:512] = (np.arange(512, dtype=np.uint32) % 256) << 23
    f[512:1024] = f[:512] | 0x7fffff
    d = f.view(np.float32).astype(np.float64)
    d = d[np.isfinite(d)]
    half = np.float64(0.5) * np.spacing(d.astype(np.float32)).astype(np.float64)
    tie = d + half
    edge = np.array([0.0, 2.0 ** -126, 2.0 ** -127, 2.0 ** -149, 2.0 ** -150, 2.0 ** -151,
                     2.0 ** 127, 3.4028234663852886e38, 3.4028235677973366e38, 2.0 ** 128, 1e300,
                     5e-324, np.inf, np.nan])
    x = np.concatenate([rng.integers(0, 1 << 64, 60000, dtype=np.uint64).view(np.float64), d, tie,
                        np.nextafter(tie, 0), np.nextafter(tie, np.inf), edge,
                        np.nextafter(edge[1:-2], 0), np.nextafter(edge[1:-2], np.inf)])
    return np.concatenate([x, -x])


def test_double_to_float_is_the_conversion(num):
    x = _doubles_around_floats()
    got, ref = num("num_d2f", [x], [(len(x), _f32())] * 2)
    assert _same_or_both_nan(got, ref)
    x = np.abs(x[x != 0])
    got, ref = num("num_d2f_up", [x], [(len(x), _f32())] * 2)
    assert _same_or_both_nan(got, ref)


def test_float_to_double_is_the_conversion_but_for_subnormals(num):
    """A subnormal gives a zero of its sign, as the conversion does where
    subnormals are flushed (the file of the pair passes)."""
    rng = np.random.default_rng(4)
    b = rng.integers(0, 1 << 32, 200000, dtype=np.uint32)
    b[:8] = [0, 0x80000000, 0x007fffff, 0x00800000, 0x7f7fffff, 0x7f800000, 0xff800000, 0x7fc00001]
    x = b.view(np.float32)
    got, ref = num("num_f2d", [x], [(len(x), _f64())] * 2)
    sub = (b & 0x7f800000) == 0
    ref[sub] = np.copysign(0.0, ref[sub])
    assert sub.any() and _same_or_both_nan(got, ref)


def test_unsigned_to_double_is_exact(num):
    rng = np.random.default_rng(5)
    x = np.concatenate([np.arange(70000), 2 ** np.arange(31), 2 ** np.arange(1, 32) - 1,
                        rng.integers(0, 1 << 31, 100000)]).astype(np.uint32)
    got, ref = num("num_u2d", [x], [(len(x), _f64())] * 2)
    assert (_bits(got) == _bits(ref)).all() and (got == x).all()


@pytest.mark.parametrize("periodic", [(1, 1), (1, 0), (0, 0)])
@pytest.mark.parametrize("n", [(1, 2), (3, 4), (5, 16), (255, 256), (1000, 4097), (32767, 32768),
                               (65534, 65535)])
def test_anchor_separations_by_the_integer_rule(num, n, periodic):
    """anchor_sep and its paired form on the lattice's own constants: the
    values of the wrapped integer index, bit for bit, index differences at
    half the period among them."""
    rng = np.random.default_rng(n[0] + n[1])
    A = (0.37 / n[0], 1.9 / n[1])
    N = 40000
    rec = []
    for r in range(2):
        f = np.empty((N, 4), np.float32)
        g = [rng.integers(0, n[a], N) for a in (0, 1)]
        if r == 1:   # differences around zero and half the period
            for a in (0, 1):
                k = rng.integers(-2, 3, N // 2) + rng.choice([0, n[a] // 2, n[a] - n[a] // 2], N // 2)
                g[a][:N // 2] = (rec[0][1][a][:N // 2] + k) % n[a]
        for a in (0, 1):
            f[:, a] = rng.uniform(-0.01, 1.01, N) * A[a]
        f[:, 2] = 1.0
        f[:, 3] = (g[0] | (g[1] << 16)).astype(np.uint32).view(np.float32)
        rec.append((f, g))
    more = [ctypes.c_double(A[0]), ctypes.c_double(A[1])] + \
        [ctypes.c_int(v) for v in n + periodic]
    (o,) = num("num_sep", [rec[0][0], rec[1][0]], [((N, 6), _f32())], *more)
    assert (_bits(o[:, 2:4].copy()) == _bits(o[:, 0:2].copy())).all()
    assert (_bits(o[:, 4:6].copy()) == _bits(o[:, 0:2].copy())).all()
