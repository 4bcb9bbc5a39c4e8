"""The kernels' integer and FP32 routes of FP64 arithmetic, compiled for the host from their
sources and compared with the plain operations: conversions, reciprocals, operand splits and
the distance test of the greedy selection. No GPU."""
import os
import re
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2601_19957_gb300", "csrc")

# (file, function) in the order they need one another
FUNCTIONS = [("sb_internal.cuh", "cvt_f32_slow"), ("sb_internal.cuh", "cvt_f64_slow"),
             ("sb_internal.cuh", "f64_to_f32"), ("sb_internal.cuh", "f32_to_f64"),
             ("laplace.cu", "dd_far_exact"), ("laplace.cu", "dd_far"), ("laplace.cu", "recip"),
             ("laplace.cu", "recip_as"), ("tc.cu", "split24"), ("tc.cu", "round_op_slow"), ("tc.cu", "round_op"),
             ("tc.cu", "split_lo_slow"), ("tc.cu", "split_op")]

SHIMS = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
#define __noinline__
enum { SB_PREC_FP64 = 0, SB_PREC_TF32 = 1, SB_PREC_BF16 = 2 };
template <typename A, typename B> static A bits(B b) { A a; static_assert(sizeof(A) == sizeof(B), ""); std::memcpy(&a, &b, sizeof a); return a; }
static int __double2hiint(double v) { return (int)(bits<uint64_t>(v) >> 32); }
static int __double2loint(double v) { return (int)(uint32_t)bits<uint64_t>(v); }
static double __hiloint2double(int h, int l) { return bits<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static float __uint_as_float(uint32_t u) { return bits<float>(u); }
static uint32_t __float_as_uint(float f) { return bits<uint32_t>(f); }
static float __frcp_rn(float f) { return 1.0f / f; }
static float __uint2float_rn(uint32_t u) { return (float)u; }
using std::fma; using std::fabs;
static float fabsf_(float f) { return std::fabs(f); }
// a bf16 as the float of its value
struct bf16 { float v; };
static float __bfloat162float(bf16 b) { return b.v; }
static bf16 __float2bfloat16_rn(float f) {
    uint32_t u = bits<uint32_t>(f);
    if ((u & 0x7fffffffu) > 0x7f800000u) return {f};
    return {bits<float>((u + 0x7fffu + ((u >> 16) & 1u)) & 0xffff0000u)};
}
// one rounding from double: round to odd in float, then to bf16
static bf16 __double2bfloat16(double x) {
    float f = (float)x;
    if (std::isfinite(f) && (double)f != x) {
        if (std::fabs((double)f) > std::fabs(x)) f = std::nextafterf(f, 0.0f);
        f = bits<float>(bits<uint32_t>(f) | 1u);
    }
    return __float2bfloat16_rn(f);
}
// to nearest, ties away, 10 fraction bits
static float to_tf32(float f) {
    uint32_t u = bits<uint32_t>(f);
    if ((u & 0x7f800000u) == 0x7f800000u) return f;
    return bits<float>((u + 0x1000u) & 0xffffe000u);
}
"""

ENTRY = r"""
extern "C" {
void t_f32(int64_t n, const double *x, float *y) { for (int64_t i = 0; i < n; ++i) y[i] = f64_to_f32(x[i]); }
void t_f64(int64_t n, const float *x, double *y) { for (int64_t i = 0; i < n; ++i) y[i] = f32_to_f64(x[i]); }
void t_far(int64_t n, const double *x, const double *b, const double *tau, int8_t *y) {
    for (int64_t i = 0; i < n; ++i) y[i] = dd_far(x[i], b[i], f64_to_f32(b[i]), tau[i], f64_to_f32(tau[i]));
}
void t_recip(int64_t n, const double *x, double *y, double *z) {
    for (int64_t i = 0; i < n; ++i) { y[i] = recip(x[i]); z[i] = recip_as<true>(x[i]); }
}
void t_split24(int64_t n, const double *x, float *t, float *r, int8_t *ok) {
    for (int64_t i = 0; i < n; ++i) ok[i] = split24(x[i], t[i], r[i]);
}
void t_split(int64_t n, int prec, const double *x, float *h, float *l, float *h0, float *l0) {
    for (int64_t i = 0; i < n; ++i) {
        if (prec == 2) {
            split_op<2>(x[i], h[i], l[i]);
            h0[i] = __double2bfloat16(x[i]).v;
            l0[i] = __double2bfloat16(x[i] - (double)h0[i]).v;
        } else {
            split_op<1>(x[i], h[i], l[i]);
            h0[i] = to_tf32((float)x[i]);
            l0[i] = to_tf32((float)(x[i] - (double)h0[i]));
        }
    }
}
}
"""


def _function(text, name):
    """The definition of a function: its template line, if any, to its closing brace."""
    m = re.search(r"^((?:template[^\n]*\n)?[^\n;]*__device__[^\n;]*\b" + name + r"\([^;{]*\)\s*\{)", text, re.M)
    assert m, name
    depth, i = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[m.start():i]


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    import ctypes as C

    out = tmp_path_factory.mktemp("dev")
    src = SHIMS + "#define fabsf fabsf_\n"
    for name, fn in FUNCTIONS:
        src += _function(open(os.path.join(CSRC, name)).read(), fn) + "\n"
    (out / "dev.cpp").write_text(src + ENTRY)
    so = str(out / "dev.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", str(out / "dev.cpp"), "-o", so],
                   check=True)
    lib = C.CDLL(so)
    p = lambda a: a.ctypes.data_as(C.c_void_p)

    def call(name, n, *args):
        getattr(lib, name)(C.c_int64(n), *[p(a) if isinstance(a, np.ndarray) else C.c_int(a) for a in args])

    return call


def _far(dev, x, b, tau):
    x, b, tau = (np.ascontiguousarray(np.broadcast_to(v, x.shape), dtype=np.float64) for v in (x, b, tau))
    y = np.empty(x.shape, dtype=np.int8)
    dev("t_far", x.size, x, b, tau, y)
    return y.astype(bool), np.abs(x - b) > tau


@pytest.mark.parametrize("exp", [0, -60, -100, -125, -130, -140, -148, -400, -1000, 60, 120, 126, 500])
def test_distance_test_is_the_exact_one_at_every_scale(dev, exp):
    """Points of a box of size 2^exp, distances at, near and away from tau = 1e-3 of it."""
    rng = np.random.default_rng(exp + 2000)
    n = 20000
    tau = 1e-3 * rng.uniform(0.5, 2.0, n)
    b = rng.uniform(-1, 1, n)
    rel = rng.choice([0.0, 1e-16, 1e-9, 1e-7, 1e-6, 1e-5, 0.1, 0.5, 0.9, 10.0], n)
    x = b + tau * (1.0 + rel * rng.choice([-1.0, 1.0], n)) * rng.choice([-1.0, 1.0], n)
    s = 2.0 ** exp
    got, want = _far(dev, x * s, b * s, tau * s)
    assert np.array_equal(got, want), np.count_nonzero(got != want)


def test_distance_test_at_the_ends(dev):
    x = np.array([np.nan, np.inf, -np.inf, 1e300, 0.0, 5e-324, 1e39, -1e39, 3.4e38, 0.0])
    for b in (0.0, 1e300, -1e39, 5e-324, np.inf):
        for tau in (0.0, 5e-324, 1e-310, 1e-40, 1e-3, 1e38, 1e39, 1e300):
            with np.errstate(invalid="ignore"):
                got, want = _far(dev, x, np.full(x.shape, b), np.full(x.shape, tau))
            assert np.array_equal(got, want), (b, tau)


def _doubles(seed, n=200000):
    """Random bit patterns over all exponents, with ties, ends of the ranges and specials."""
    rng = np.random.default_rng(seed)
    bits = rng.integers(0, 1 << 63, n, dtype=np.uint64) | (rng.integers(0, 2, n, dtype=np.uint64) << np.uint64(63))
    near = (rng.integers(860, 1160, n, dtype=np.uint64) << np.uint64(52)) | (bits & np.uint64((1 << 52) - 1))
    # halfway between neighbours of FP32, bf16 and tf32, and a unit beside it
    tie = []
    for keep in (23, 10, 7):
        b = near & ~np.uint64((1 << (52 - keep)) - 1) | np.uint64(1 << (51 - keep))
        tie += [b, b + np.uint64(1), b - np.uint64(1)]
    sign = rng.integers(0, 2, n, dtype=np.uint64) << np.uint64(63)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -126, 2.0 ** -149, 2.0 ** -150,
                        2.0 ** -151, np.nextafter(2.0 ** -126, 0), 2.0 ** 128, np.nextafter(2.0 ** 128, 0),
                        (2 - 2.0 ** -24) * 2.0 ** 127, np.finfo(np.float32).max, np.finfo(np.float64).max, 1.0, -1.0])
    return np.concatenate([bits.view(np.float64), (near | sign).view(np.float64)] +
                          [t.view(np.float64) for t in tie] + [special])


def _same(a, b):
    """Equal bits, or both NaN."""
    u = np.uint32 if a.dtype == np.float32 else np.uint64
    return (a.view(u) == b.view(u)) | (np.isnan(a) & np.isnan(b))


def test_double_to_float_is_the_conversion(dev):
    x = _doubles(1)
    y = np.empty(x.shape, np.float32)
    dev("t_f32", x.size, x, y)
    with np.errstate(over="ignore", invalid="ignore", under="ignore"):
        assert _same(y, x.astype(np.float32)).all()


def test_float_to_double_is_the_conversion(dev):
    rng = np.random.default_rng(2)
    x = np.concatenate([rng.integers(0, 1 << 32, 400000, dtype=np.uint64).astype(np.uint32).view(np.float32),
                        np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e-45, -1e-45, 2.0 ** -126, 3.4028235e38], np.float32)])
    y = np.empty(x.shape, np.float64)
    dev("t_f64", x.size, x, y)
    with np.errstate(invalid="ignore"):
        assert _same(y, x.astype(np.float64)).all()


def test_reciprocal_is_within_a_unit_and_the_corrected_one_rounds(dev):
    """recip: one unit in the last place. recip_as<true>: a division's rounding, where the
    correction step's products do not underflow (a third-order step then one of Newton)."""
    x = _doubles(3)
    x = x[np.isfinite(x) & (x != 0)]
    x = np.concatenate([x, 1.0 + np.arange(2000) * 2.0 ** -52, 2.0 - np.arange(1, 2000) * 2.0 ** -52])
    y, z = np.empty_like(x), np.empty_like(x)
    dev("t_recip", x.size, x, y, z)
    with np.errstate(over="ignore"):
        want = 1.0 / x
    ok = np.isfinite(want)
    with np.errstate(invalid="ignore"):
        assert np.all(np.abs(y - want)[ok] <= np.spacing(np.abs(want))[ok])
        assert _same(y, want)[~ok].all()
    e = (x.view(np.uint64) >> np.uint64(52)) & np.uint64(0x7ff)
    mid = (e >= 64) & (e <= 1982)
    assert np.array_equal(z[mid], want[mid])
    normal = ok & (np.abs(want) >= 2.0 ** -1022)
    assert np.all(np.abs(z - want)[normal] <= np.spacing(np.abs(want))[normal])


def test_truncation_and_rest_add_up(dev):
    x = _doubles(4)
    t, r = np.empty(x.shape, np.float32), np.empty(x.shape, np.float32)
    ok = np.empty(x.shape, np.int8)
    dev("t_split24", x.size, x, t, r, ok)
    a = np.abs(x)
    inside = (a >= 2.0 ** -63) & (a < 2.0 ** 64)
    assert np.array_equal(ok.astype(bool), inside | (x == 0))
    x, t, r = x[inside], t[inside], r[inside]
    rest = x - t.astype(np.float64)  # exact: x's last 29 bits
    assert np.all(np.abs(t) <= np.abs(x)) and np.all(np.abs(rest) < np.abs(t) * 2.0 ** -22)
    assert np.array_equal(r, rest.astype(np.float32))


@pytest.mark.parametrize("prec", [1, 2])
def test_operand_split_is_the_fp64_one(dev, prec):
    """hi always; lo wherever the remainder is above FP32's resolution of x (below it, where the
    truncation and the rest cancel, within 2^-48 of x)."""
    x = _doubles(5 + prec)
    x = x[np.isfinite(x) & (np.abs(x) < 1e38)]
    h, l, h0, l0 = (np.empty(x.shape, np.float32) for _ in range(4))
    dev("t_split", x.size, prec, x, h, l, h0, l0)
    assert np.array_equal(h, h0)  # (a zero may lose its sign)
    rem = np.abs(x - h0.astype(np.float64))
    far = rem > np.abs(x) * 2.0 ** -24
    assert np.array_equal(l[far], l0[far]), np.count_nonzero(l[far] != l0[far])
    assert np.all(np.abs(l.astype(np.float64) - l0) <= np.abs(x) * 2.0 ** -48)
