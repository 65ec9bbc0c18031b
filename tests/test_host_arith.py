"""The device arithmetic of csrc/common.cuh, compiled for the host (its intrinsics spelled as plain IEEE operations) and compared with
FP64 sums where it can go wrong: six neighbours of any mixture of zeros, subnormals and normal values; the residual of FP32 states over
spans, signs and cancelling neighbours of all kinds."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2102_12416_gb300", "csrc")

# What common.cuh takes from CUDA, for a host compiler (the memory and wait helpers are declared only).
SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
using std::max; using std::min; using std::fabs;
template <class A, class B> static inline A bits(B b) { A a; static_assert(sizeof(a) == sizeof(b), ""); memcpy(&a, &b, sizeof a); return a; }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline long long __double_as_longlong(double a) { return bits<long long>(a); }
static inline double __longlong_as_double(long long a) { return bits<double>(a); }
static inline uint32_t __float_as_uint(float a) { return bits<uint32_t>(a); }
static inline float __uint_as_float(uint32_t a) { return bits<float>(a); }
static inline int __double2hiint(double a) { return (int)(bits<uint64_t>(a) >> 32); }
static inline int __double2loint(double a) { return (int)bits<uint64_t>(a); }
static inline double __hiloint2double(int h, int l) { return bits<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
static inline uint32_t __funnelshift_l(uint32_t l, uint32_t h, uint32_t s) { s &= 31; return s ? h << s | l >> (32 - s) : h; }
static inline uint32_t __funnelshift_r(uint32_t l, uint32_t h, uint32_t s) { s &= 31; return s ? l >> s | h << (32 - s) : l; }
struct dim3_ { unsigned x, y, z; };
extern dim3_ threadIdx, blockDim;
uint32_t atomicCAS(uint32_t*, uint32_t, uint32_t);
void __nanosleep(unsigned);
void __syncthreads();
double __shfl_down_sync(unsigned, double, int);
"""

# r = s - 6u of n points by the routes of the kernels; v holds the six neighbours (xm xp ym yp zm zp) and u of each.
CODE = r"""
#include "common.cuh"
using namespace jgb;
extern "C" {
// The three pair sums and xy by the short adder; the other routine where sum_far says so (both forms that the kernels use).
void near_sums(const double* v, int64_t n, double* out) {
  for (int64_t i = 0; i < n; ++i, v += 7) {
    int f = 0;
    const double x = dadd_near(v[0], v[1], f), y = dadd_near(v[2], v[3], f), z = dadd_near(v[4], v[5], f);
    double s = dadd_near(x, y, f);
    if (f < 0 && sum_far(v[0], v[1], v[2], v[3], v[4], v[5], true) < 0) s = v[0] + v[1] + (v[2] + v[3]), out[i] = s + (v[4] + v[5]);
    else out[i] = s + z;
  }
}
// The residual of FP32 values; counts the points that the split form takes.
int64_t resid32(const float* v, int64_t n, double* out) {
  int64_t split = 0;
  for (int64_t i = 0; i < n; ++i, v += 7) {
    float d, e;
    const bool ok = resid_split(v[0], v[1], v[2], v[3], v[4], v[5], v[6], d, e) && point_exact(v[0], v[1], v[2], v[3], v[4], v[5], v[6]);
    split += ok;
    out[i] = ok ? widen_f32(d) + widen_f32(e) : resid_f64(v[0], v[1], v[2], v[3], v[4], v[5], v[6]);
  }
  return split;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    (d / "cuda_runtime.h").write_text(SHIM)
    (d / "arith.cpp").write_text(CODE)
    so = str(d / "arith.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-w", f"-I{d}", f"-I{CSRC}", str(d / "arith.cpp"),
                    "-o", so], check=True)
    return ctypes.CDLL(so)


def _call(fn, v, out):
    fn.restype = ctypes.c_int64
    return fn(ctypes.c_void_p(v.ctypes.data), ctypes.c_int64(len(v)), *(ctypes.c_void_p(o.ctypes.data) for o in out))


def _mixed64(n, seed):
    """Rows of seven values: zeros, subnormals below and above 2^-1042 (high word zero or not), normals of all sizes, close ones."""
    r = np.random.default_rng(seed)
    kind = r.integers(0, 6, (n, 7))
    exp = np.select([kind <= 2, kind == 3], [np.zeros((n, 7), np.int64), r.integers(1, 2039, (n, 7))], 1023 - r.integers(0, 25, (n, 7)))
    mant = r.integers(0, 1 << 52, (n, 7))
    mant = np.select([kind == 0, kind == 1], [np.zeros((n, 7), np.int64), mant >> r.integers(20, 52, (n, 7))], mant)
    return ((exp << 52) | mant).view(np.float64)


def test_short_adder_far_operands(lib):
    """Every point whose operands are out of the short adder's reach is found, a pair of a zero and the smallest subnormals
    included: the sums are the FP64 sums, bit for bit."""
    tiny = [0.0, 5e-324, 2.0 ** -1043, 2.0 ** -1042, 2.1e-314, 2.0 ** -1022]
    rows = [(a, b, c, d, 0.5, 0.25, 0.0) for a in tiny for b in tiny for c in (0.0, 1.0, 2.0 ** -20, 1e100, 5e-324) for d in (0.0, 1.0, 1e100)]
    rows += [(c, d, a, b, e, f, 0.0) for a, b, c, d, e, f, _ in rows]
    for v in [np.array(rows)] + [_mixed64(1 << 20, s) for s in (1, 2)]:
        v = np.ascontiguousarray(v)
        got = np.empty(len(v))
        _call(lib.near_sums, v, [got])
        want = ((v[:, 0] + v[:, 1]) + (v[:, 2] + v[:, 3])) + (v[:, 4] + v[:, 5])
        bad = np.nonzero(got.view(np.int64) != want.view(np.int64))[0]
        assert len(bad) == 0, (len(bad), [float(x).hex() for x in v[bad[0]]])


def _states32(n):
    """(what, rows of six neighbours and u, share that the split form must take)"""
    r = np.random.default_rng(5)
    one = r.uniform(0.5, 1.0, (n, 7))
    sign = r.choice([-1.0, 1.0], (n, 7))
    wide = 2.0 ** r.integers(-26, 1, (n, 7))  # spans around 2^19, where the split form ends
    cancel = one * 2.0 ** r.integers(-40, -20, (n, 7))
    k = r.integers(0, 3, n) * 2
    cancel[np.arange(n), k] = one[:, 0]
    cancel[np.arange(n), k + 1] = -one[:, 0]
    u = one[:, :6].sum(1) / 6.0
    near = one.copy()
    near[:, 6] = np.float32(u) * (1 + 2.0 ** -23 * r.integers(-3, 4, n))  # near convergence: |r| far below the sums
    sparse = np.where(r.uniform(size=(n, 7)) < 0.4, 0.0, one * sign)
    return [("plain", one, 1.0), ("signed", one * sign, 1.0), ("near", near, 1.0), ("zeros", sparse, 1.0), ("wide", one * wide, 0.05),
            ("wide signed", one * wide * sign, 0.05), ("cancel", cancel, 0.0), ("smooth", 3.0 + 1e-3 * one, 1.0),
            ("exponents", one * sign * 2.0 ** r.integers(-149, 128, (n, 7)), 0.0), ("subnormal", one * sign * 2.0 ** -135, 1.0),
            ("overflow", np.where(r.uniform(size=(n, 7)) < 0.3, 3.0e38, one) * sign, 0.0),
            ("inf", np.where(r.uniform(size=(n, 7)) < 0.1, np.inf, one), 0.0), ("nan", np.where(r.uniform(size=(n, 7)) < 0.1, np.nan, one), 0.0)]


def test_fp32_residual_is_that_of_fp64_sums(lib):
    """r of every point equals the FP64 sums of the widened values: where the split form is taken every term is exact, elsewhere the
    FP64 sums themselves are.  The split form takes all points of ordinary states."""
    for what, rows, share in _states32(1 << 18):
        with np.errstate(over="ignore"):
            v = np.ascontiguousarray(rows.astype(np.float32))
        got = np.empty(len(v))
        split = _call(lib.resid32, v, [got])
        w = v.astype(np.float64)
        with np.errstate(invalid="ignore"):
            want = (((w[:, 0] + w[:, 1]) + (w[:, 2] + w[:, 3])) + (w[:, 4] + w[:, 5])) - 6.0 * w[:, 6]
        bad = np.nonzero((got != want) & ~(np.isnan(got) & np.isnan(want)))[0]
        assert len(bad) == 0, (what, len(bad), [float(x).hex() for x in v[bad[0]]], got[bad[0]], want[bad[0]])
        assert split >= share * len(v), (what, split)
