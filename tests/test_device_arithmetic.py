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
