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
