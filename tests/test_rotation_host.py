"""The FP64 rotation choice of the device header (csrc/jacobi_core.cuh), compiled
for the host: the header's own code with the device intrinsics written out and the
two approximate seeds (reciprocal, reciprocal square root) exact but for a
relative error of up to 2^-22, the hardware's documented bound."""
from __future__ import annotations

import ctypes as C
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

CORE = os.path.join(os.path.dirname(__file__), "..", "paper_2608_28952_gb300", "csrc", "jacobi_core.cuh")
U = 2.0 ** -53

PRELUDE = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>
using std::max; using std::min; using std::fabs;
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
struct double2 { double x, y; };
struct dim { int x = 0, y = 0, z = 0; };
static dim threadIdx, blockDim;
static void __syncthreads() {}
static int atomicAdd(int* p, int v) { int o = *p; *p += v; return o; }
template <class A, class B> static A bits(B b) { A a; static_assert(sizeof a == sizeof b); memcpy(&a, &b, sizeof a); return a; }
#define OP(T, n, e) static T n(T a, T b) { return e; }
OP(double, __dadd_rn, a + b) OP(double, __dsub_rn, a - b) OP(double, __dmul_rn, a * b) OP(double, __ddiv_rn, a / b)
OP(float, __fadd_rn, a + b) OP(float, __fsub_rn, a - b) OP(float, __fmul_rn, a * b) OP(float, __fdiv_rn, a / b)
OP(float, __fdividef, a / b)
static double __dsqrt_rn(double a) { return std::sqrt(a); }
static float __fsqrt_rn(float a) { return std::sqrt(a); }
static int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
static int __double2loint(double x) { return (int)bits<uint64_t>(x); }
static double __hiloint2double(int h, int l) { return bits<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
static float __int_as_float(int x) { return bits<float>(x); }
static int __float_as_int(float x) { return bits<int>(x); }
static long long __double_as_longlong(double x) { return bits<long long>(x); }
static double __longlong_as_double(long long x) { return bits<double>(x); }
static double g_off = 0.0;   // relative error of the seeds
static float seed(float x, bool root) { return (float)((1.0 + g_off) / (root ? std::sqrt((double)x) : (double)x)); }
static float rsqrtf(float x) { return seed(x, true); }
"""

TAIL = r"""
extern "C" void wanted(int n, const double* p, const double* q, const double* x, double tol, int* out)
{
    for (int i = 0; i < n; ++i) out[i] = jac::rotation_wanted(p[i], q[i], x[i], tol);
}
extern "C" void params(int n, const double* p, const double* q, const double* x, int pivot, double off, double* t, double* s, double* tau)
{
    g_off = off;
    for (int i = 0; i < n; ++i)
        if (pivot) jac::schur2_pivot(p[i], q[i], x[i], s[i], t[i], tau[i]);
        else jac::schur2(p[i], q[i], x[i], s[i], t[i], tau[i]);
}
extern "C" int paired(double d, double x) { return jac::schur2_paired(jac::f64_biased_exp(d), jac::f64_biased_exp(x)); }
"""


@pytest.fixture(scope="module")
def core(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    src = open(CORE).read().replace("#include <cuda_runtime.h>", "").replace("#pragma once", "")
    src, n = re.subn(r'asm\("(rsqrt|rcp)\.approx[^;]*;" : "=f"\(y\) : "f"\(x\)\);',
                     lambda m: f"y = seed(x, {'true' if m[1] == 'rsqrt' else 'false'});", src)
    assert n == 2
    d = tmp_path_factory.mktemp("core")
    (d / "core.cpp").write_text(PRELUDE + src + TAIL)
    lib = d / "core.so"
    # no contraction: the header's fused operations are fma(), the rest round one by one
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-o", str(lib),
                    str(d / "core.cpp")], check=True)
    return C.CDLL(str(lib))


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


@pytest.mark.parametrize("tol", [0.0, 4 * U, 1e-3])
def test_rotation_test_on_special_values(core, tol):
    """|a_pq| > tol sqrt|a_pp| sqrt|a_qq| over zeros, subnormals, the ends of the
    range, infinities and NaN, as the formula gives it in FP64: a comparison
    with NaN is false, so nothing is rotated for one."""
    v = np.array([0.0, -0.0, 5e-324, 1e-310, 2.3e-308, 1e-160, 1e-3, 1.0, -3.0, 1e160, 1.7e308, np.inf, -np.inf, np.nan])
    p, q, x = (np.ascontiguousarray(a.ravel()) for a in np.meshgrid(v, v, v, indexing="ij"))
    out = np.zeros(p.size, np.int32)
    core.wanted(p.size, _p(p), _p(q), _p(x), C.c_double(tol), _p(out))
    with np.errstate(all="ignore"):
        rhs = (tol * np.sqrt(np.abs(p))) * np.sqrt(np.abs(q))
        want = np.abs(x) > rhs
        near = np.abs(np.abs(x) - rhs) <= 1e-12 * rhs     # (the form without square roots rounds elsewhere)
    bad = (out != want) & ~(near & np.isfinite(rhs))
    assert not bad.any(), list(zip(p[bad], q[bad], x[bad], out[bad]))[:8]


def _triples(seed):
    """Magnitudes 1e-280 to 1e280; within a triple close together, or up to 1e20 and
    1e60 apart; equal and negative diagonals."""
    r = np.random.default_rng(seed)
    n = 40000
    base = 10.0 ** r.uniform(-280, 280, n)
    p, q = (base * r.standard_normal(n) * 10.0 ** r.uniform(-3, 3, n) for _ in range(2))
    x = base * r.standard_normal(n) * 10.0 ** r.choice([0.0, -5.0, -12.0, -17.0, -20.0, -60.0, 4.0], n)
    q[: n // 8] = p[: n // 8]
    p[n // 8: n // 4] *= -1
    ok = (np.abs(x) > 1e-290) & np.isfinite(p) & np.isfinite(q)
    return [np.ascontiguousarray(a[ok]) for a in (p, q, x)]


@pytest.mark.parametrize("off", [0.0, 2.0 ** -22, -2.0 ** -22])
@pytest.mark.parametrize("pivot", [1, 0])
def test_rotation_parameters(core, pivot, off):
    """t, s and tau of the pivot solves' choice (the halves that two lanes share,
    joined) and of the batched solves', with the seeds off by their bound, against
    the textbook formulas in long double: within 6 units of 2^-53, and (1 - s tau)^2 +
    s^2 = 1 within 8, the bounds that the kernels' results are held to."""
    p, q, x = _triples(11 + pivot)
    t, s, tau = (np.zeros(p.size) for _ in range(3))
    core.params(p.size, _p(p), _p(q), _p(x), pivot, C.c_double(off), _p(t), _p(s), _p(tau))
    d = q - p
    if pivot:      # both kinds of triple are among them
        kind = {core.paired(C.c_double(a), C.c_double(b)) for a, b in zip(d[:4000], x[:4000])}
        assert kind == {0, 1}
    L = np.longdouble
    with np.errstate(all="ignore"):
        zeta = L(d) / (L(2) * L(x))
        tt = np.where(zeta >= 0, L(1), L(-1)) / (np.abs(zeta) + np.sqrt(L(1) + zeta * zeta))
    cc = L(1) / np.sqrt(L(1) + tt * tt)
    for name, got, want in (("t", t, tt), ("s", s, tt * cc), ("tau", tau, tt * cc / (L(1) + cc))):
        err = np.abs((L(got) - want) / want).astype(np.float64)
        err = err[np.abs(want) > 1e-290]
        assert err.max() <= 6 * U, (name, err.max() / U)
    c = 1.0 - s * tau
    assert np.abs(c * c + s * s - 1.0).max() <= 8 * U
