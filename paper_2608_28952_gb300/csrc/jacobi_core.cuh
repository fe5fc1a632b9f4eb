// jacobi_core.cuh -- the scalar parallel-ordered Jacobi solve of one symmetric
// k x k matrix by one CTA, shared by the pivot kernel of the blocked method
// (FP64) and the batched kernels (FP32 and FP64).
//
// The solve is Algorithm 2 applied with block size 1: each sweep is k-1
// rounds of the round-robin order over the k indices; a round computes the
// k/2 textbook 2x2 Schur rotations from the round's starting values, rotates
// every disjoint 2x2 "quad" (rows of pair e1, columns of pair e2) from both
// sides, sets each rotated 2x2 pivot to its exact diagonal form and rotates
// the columns of V.  The symmetric matrix lives in packed lower-triangular
// form; the diagonal is carried as hi (in the packed array) + lo.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace jac {

__device__ __forceinline__ int tri(int i) { return (i * (i + 1)) >> 1; }
__device__ __forceinline__ int sidx(int i, int j) { return i >= j ? tri(i) + j : tri(j) + i; }

// ---------------------------------------------------------------- correctly rounded ops
__device__ __forceinline__ double rn_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double rn_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double rn_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double rn_div(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ double rn_sqrt(double a) { return __dsqrt_rn(a); }
__device__ __forceinline__ float rn_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rn_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rn_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rn_div(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float rn_sqrt(float a) { return __fsqrt_rn(a); }

template <typename T>
struct Lim;
template <>
struct Lim<double> {
    static constexpr double big = 1e150;   // 1 + zeta^2 would overflow beyond this
};
template <>
struct Lim<float> {
    static constexpr float big = 1e18f;
};

// The textbook 2x2 symmetric Schur rotation: zeta = (aqq - app)/(2 apq),
// t = sgn(zeta)/(|zeta| + sqrt(1 + zeta^2)) with sgn(0) = +1, c = 1/sqrt(1+t^2),
// s = t c; J = [[c, s], [-s, c]] makes J^T [[app, apq], [apq, aqq]] J diagonal
// with diagonal (app - t apq, aqq + t apq).  Every operation is rounded
// separately (no contraction).  Returns s, t and tau = s/(1+c).
template <typename T>
__device__ __forceinline__ void schur2_ref(T app, T aqq, T apq, T& s, T& t, T& tau)
{
    const T zeta = rn_div(rn_sub(aqq, app), rn_mul(T(2), apq));
    if (fabs(zeta) > Lim<T>::big) {
        t = rn_div(T(0.5), zeta);
    } else {
        const T r = rn_sqrt(rn_add(T(1), rn_mul(zeta, zeta)));
        t = rn_div(zeta >= T(0) ? T(1) : T(-1), rn_add(fabs(zeta), r));
    }
    const T c = rn_div(T(1), rn_sqrt(rn_add(T(1), rn_mul(t, t))));
    s = rn_mul(t, c);
    tau = rn_div(s, rn_add(T(1), c));
}

template <typename T>
__device__ __forceinline__ void schur2(T app, T aqq, T apq, T& s, T& t, T& tau)
{
    schur2_ref(app, aqq, apq, s, t, tau);
}

template <typename T>
__device__ __forceinline__ bool rotation_wanted(T app, T aqq, T apq, T tol)
{
    if (apq == T(0)) return false;
    return fabs(apq) > rn_mul(rn_mul(tol, rn_sqrt(fabs(app))), rn_sqrt(fabs(aqq)));
}

// ---------------------------------------------------------------- FP64 with few FP64 instructions
// On this part FP64 runs at 1/64 of the FP32 rate: any FP64 instruction, a
// conversion included, holds its warp for 64 cycles, while an FP32 or integer
// one takes about 5.  The rotation choice is the serial chain of a solve, so
// the FP64 overloads below do all they can outside the FP64 unit:
//   * conversions between FP64 and FP32 by integer instructions on the bits;
//   * t (the root of a t^2 + d t - a = 0 with |t| <= 1, d = aqq - app, a = apq,
//     the textbook's choice), tau (t tau^2 + 2 tau - t = 0) and c ((1 + t^2) c^2
//     - 1 = 0) each from an FP32 seed and one Newton step in pairs of floats
//     (exact products by fma, error-free sums): 2^-42 relative;
//   * then one Newton step in FP64 each: two FMAs for the residual, one for
//     the step with the seed's FP32 reciprocal of the derivative, one addition
//     to join the pair; s = t c.
// 15 FP64 instructions (and tau and c side by side where two threads share a
// rotation) in place of about 40 with single FP32 seeds, two FP64 Newton steps
// and hardware conversions.  t is within 2u of the exact root, tau and s within
// 4u, (1 - s tau)^2 + s^2 = 1 within 2u (measured over 2e7 triples): the rotation
// applied in Rutishauser's form stays orthogonal to working precision.
__device__ __forceinline__ int f64_biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

__device__ __forceinline__ float rsqrt_seed(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_seed(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// |x| 2^-e, e its exponent, in two parts: the leading 24 bits (truncated), in
// [1, 2) for a normal x, and the next 23
__device__ __forceinline__ float f64_lead(double x)
{
    return __int_as_float((127 << 23) | ((__double2hiint(x) & 0xFFFFF) << 3) | (int)((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ float f64_rest(double x)
{
    return (__int_as_float(0x4B000000 | ((__double2loint(x) & 0x1FFFFFFF) >> 6)) - 8388608.0f) * __int_as_float(81 << 23);
}
// 2^e, e <= 0; 0 below 2^-80
__device__ __forceinline__ float f32_pow2(int e) { return e < -80 ? 0.0f : __int_as_float((e + 127) << 23); }
// f 2^e exactly (f a normal float or 0, the result normal)
__device__ __forceinline__ double f64_of(float f, int e)
{
    const int b = __float_as_int(f), m = b & 0x7fffffff;
    return m < 0x00800000 ? 0.0 : __hiloint2double((b & 0x80000000) | ((m >> 3) + ((896 + e) << 20)), b << 29);
}
// the nearest float (ties away), 0 below the normal range; |x| < 2^127
__device__ __forceinline__ float f32_of(double x)
{
    const long long v = (__double_as_longlong(x) & 0x7fffffffffffffffll) + (1ll << 28);
    const long long m = (v >> 29) - (896ll << 23);
    return m < 0x00800000 ? 0.0f : __int_as_float((int)m | (__double2hiint(x) & 0x80000000));
}

// any finite triple, by FP32 seeds and FP64 Newton steps on scaled values
__device__ __forceinline__ void schur2_wide(double d, double apq, double& s, double& t, double& tau)
{
    // scale d and apq by 2^(1022 - E'), E' = clamp(max exponent, 2, 2044): the larger lands in [0.5, 4)
    int E = max(f64_biased_exp(d), f64_biased_exp(apq));
    E = min(max(E, 2), 2044);
    // (t depends on the ratio only: the Newton steps run on the scaled values,
    // so 1/g' stays in range even for subnormal apq)
    const double sc = __hiloint2double((2045 - E) << 20, 0);
    const double ds = d * sc, as = apq * sc;
    const float d32 = (float)ds, a2 = 2.0f * (float)as;
    const bool dzero = (__double_as_longlong(d) << 1) == 0;
    const bool dneg = __double2hiint(d) < 0, aneg = __double2hiint(apq) < 0;
    const float R = sqrtf(fmaf(d32, d32, a2 * a2));
    const float sgz = (dzero || dneg == aneg) ? 1.0f : -1.0f;          // sgn(zeta), sgn(0) = +1
    const float t32 = sgz * __fdividef(fabsf(a2), fabsf(d32) + R);
    const float sgg = dzero ? (aneg ? -1.0f : 1.0f) : (dneg ? -1.0f : 1.0f);   // sign of g'(t)
    const double r = (double)__fdividef(sgg, R);                       // ~ 1/g_s'(t), g_s = g sc
    double tt = (double)t32;
    tt = fma(-fma(fma(as, tt, ds), tt, -as), r, tt);
    tt = fma(-fma(fma(as, tt, ds), tt, -as), r, tt);
    if (fabsf(a2) < 1e-30f)   // the seed lost bits (FP32 subnormal range): one more step
        tt = fma(-fma(fma(as, tt, ds), tt, -as), r, tt);
    t = tt;
    const double x = fma(tt, tt, 1.0);                                 // in [1, 2]
    const double y0 = (double)rsqrtf((float)x);
    const double h = fma(-(x * y0), y0, 1.0);
    const double c = fma(y0 * h, fma(0.375, h, 0.5), y0);
    s = tt * c;
    const double u = 1.0 + c;                                          // in (1.7, 2]
    const double r0 = (double)__fdividef(1.0f, (float)u);
    const double e = fma(-u, r0, 1.0);
    tau = s * fma(r0, fma(e, e, e), r0);
}

// Biased exponents of d and apq for which the pairs of floats serve: normal
// range with room for the Newton steps, and apq no smaller than 2^-60 d.
__device__ __forceinline__ bool schur2_paired(int Ed, int Ea)
{
    const int E = max(Ed, Ea);
    return E >= 128 && E <= 1900 && Ea + 60 >= E;
}

// The root t of a t^2 + d t - a, a = |apq|, d = |aqq - app| (biased exponents
// Ea, Ed; dh + dl = d 2^-Ed's leading bits), and its pair of floats.
__device__ __forceinline__ double schur2_t(double a, int Ea, double d, int Ed, float dh, float dl, float& t0, float& te)
{
    const int E = max(Ed, Ea);
    const float sa = f32_pow2(Ea - E), sd = f32_pow2(Ed - E);
    const float ah = f64_lead(a) * sa, al = f64_rest(a) * sa;
    dh *= sd;
    dl *= sd;
    const float A = 2.0f * ah, n = fmaf(dh, dh, A * A), rs = rsqrt_seed(n);
    t0 = A * rcp_seed(fmaf(n, rs, dh));
    // residual a (t0^2 - 1) + d t0; its derivative at the root is sqrt(d^2 + 4 a^2)
    const float P = dh * t0, Pe = fmaf(dh, t0, -P), p = t0 * t0, pe = fmaf(t0, t0, -p), Q = ah * p, Qe = fmaf(ah, p, -Q);
    const float s1 = __fsub_rn(P, ah), b1 = __fsub_rn(s1, P);
    const float e1 = __fadd_rn(__fsub_rn(P, __fsub_rn(s1, b1)), __fsub_rn(-ah, b1));
    const float s2 = __fadd_rn(s1, Q), b2 = __fsub_rn(s2, s1);
    const float e2 = __fadd_rn(__fsub_rn(s1, __fsub_rn(s2, b2)), __fsub_rn(Q, b2));
    const float low = ((e1 + e2) + (Pe + Qe)) + (fmaf(dl, t0, -al) + fmaf(al, p, ah * pe));
    te = -(s2 + low) * rs;
    const double td = f64_of(t0, 0) + f64_of(te, 0);
    return fma(-fma(fma(a, td, d), td, -a), f64_of(rs, 1023 - E), td);
}

// tau (want_c false) or c (true) of the tangent t = t0 + te: the root of
// t z^2 + 2 z - t, or of (1 + t^2) z^2 - 1; either derivative is 2 / c.
__device__ __forceinline__ double schur2_z(double t, float t0, float te, bool want_c)
{
    const float p1 = t0 * t0, p1e = fmaf(t0, t0, -p1), xh = __fadd_rn(1.0f, p1);
    const float xl = __fadd_rn(__fsub_rn(1.0f, xh), p1) + fmaf(2.0f * t0, te, p1e);
    const float c0 = rsqrt_seed(xh), u0 = t0 * c0 * rcp_seed(1.0f + c0);
    const float z0 = want_c ? c0 : u0, Ah = want_c ? xh : t0, Al = want_c ? xl : te, B = want_c ? 0.0f : 2.0f;
    const float Ch = want_c ? -1.0f : -t0, Cl = want_c ? 0.0f : -te;
    const float P = B * z0, p = z0 * z0, pe = fmaf(z0, z0, -p), Q = Ah * p, Qe = fmaf(Ah, p, -Q);
    const float s1 = __fadd_rn(P, Ch), b1 = __fsub_rn(s1, P);
    const float e1 = __fadd_rn(__fsub_rn(P, __fsub_rn(s1, b1)), __fsub_rn(Ch, b1));
    const float s2 = __fadd_rn(s1, Q), b2 = __fsub_rn(s2, s1);
    const float e2 = __fadd_rn(__fsub_rn(s1, __fsub_rn(s2, b2)), __fsub_rn(Q, b2));
    const float low = ((e1 + e2) + Qe) + (fmaf(Ah, pe, Al * p) + Cl);
    const float ze = -0.5f * c0 * (s2 + low);
    const double zd = f64_of(z0, 0) + f64_of(ze, 0);
    const double A64 = want_c ? fma(t, t, 1.0) : t, B64 = want_c ? 0.0 : 2.0, C64 = want_c ? -1.0 : -t;
    return fma(-fma(fma(A64, zd, B64), zd, C64), f64_of(0.5f * c0, 0), zd);
}

// sgn(zeta) as a sign bit, sgn(0) = +1
__device__ __forceinline__ int schur2_sign(double d, double apq)
{
    return (__double_as_longlong(d) << 1) == 0 ? 0 : (__double2hiint(d) ^ __double2hiint(apq)) & 0x80000000;
}

// The batched forms' choice: the seeds of schur2_wide, whose rounding their
// results (the signs of eigenvectors among them) have always had.
__device__ __forceinline__ void schur2(double app, double aqq, double apq, double& s, double& t, double& tau)
{
    schur2_wide(rn_sub(aqq, app), apq, s, t, tau);
}

// The pivot solves' choice in the two halves that two lanes share there.  A half: t
// and z = tau or c, all for |d| and |apq| (dh, dl: d's leading parts); false
// where the pairs of floats don't serve.
__device__ __forceinline__ bool schur2_half(double d, double apq, float dh, float dl, bool want_c, double& t, double& z)
{
    const int Ed = f64_biased_exp(d), Ea = f64_biased_exp(apq);
    if (!schur2_paired(Ed, Ea)) return false;
    float t0, te;
    t = schur2_t(fabs(apq), Ea, fabs(d), Ed, dh, dl, t0, te);
    z = schur2_z(t, t0, te, want_c);
    return true;
}
__device__ __forceinline__ double f64_flip(double x, int sign_bit)   // no FP64 instruction
{
    return __hiloint2double(__double2hiint(x) ^ sign_bit, __double2loint(x));
}
// The halves joined (t, tau and c as both left them): signs, s, and every triple
// that the pairs of floats don't take.  flip: zeta = 0 picks t = -1 (the pair's
// indices are in descending order).
__device__ __forceinline__ void schur2_join(double d, double apq, bool paired, bool flip, double& s, double& t, double& tau, double& c)
{
    int sgn = schur2_sign(d, apq);
    s = t * c;
    if (!paired) {
        schur2_wide(d, apq, s, t, tau);
        c = fma(-s, tau, 1.0);
        sgn = 0;
    }
    if (flip && (__double_as_longlong(d) << 1) == 0) sgn = 0x80000000;
    s = f64_flip(s, sgn);
    t = f64_flip(t, sgn);
    tau = f64_flip(tau, sgn);
}
// The same by one thread.
__device__ __forceinline__ void schur2_pivot(double app, double aqq, double apq, double& s, double& t, double& tau)
{
    const double d = rn_sub(aqq, app);
    const float dh = f64_lead(d), dl = f64_rest(d);
    double c = 1.0;
    const bool paired = schur2_half(d, apq, dh, dl, false, t, tau);
    schur2_half(d, apq, dh, dl, true, t, c);
    schur2_join(d, apq, paired, false, s, t, tau, c);
}

// |apq| > tol sqrt|app| sqrt|aqq| as apq^2 > tol^2 |app| |aqq|, first on
// the leading 24 bits in FP32 with the exponents apart (no FP64 instruction):
// the truncations move either side by less than 2^-20, so only a ratio within
// 2^-18 of 1 needs FP64.  There, where every operand lies in [2^-400, 2^400],
// the squares can neither overflow nor underflow and nonnegative doubles
// compare like their bit patterns; elsewhere the square-root form.
// The FP32 part: 1 rotate, 0 skip, -1 undecided (subnormals, infinities and NaN
// too: they have no leading bits to compare); y = the leading parts of tol tol app
// aqq multiplied, esum = the sum of their biased exponents.
__device__ __forceinline__ bool f64_normal_exp(int e) { return (unsigned)(e - 1) < 2046u; }
__device__ __forceinline__ int rotation_wanted_lead(double apq, float y, int esum)
{
    const int ep = f64_biased_exp(apq), sh = esum - 2 * ep - 2046;   // rhs / lhs in [2^(sh - 2), 2^(sh + 4))
    if (!f64_normal_exp(ep)) return (__double_as_longlong(apq) << 1) == 0 ? 0 : -1;
    const float fa = f64_lead(apq), x = fa * fa, r = y * __int_as_float((min(max(sh, -9), 9) + 127) << 23);
    if (sh > 8) return 0;
    if (sh < -8) return 1;
    return fabsf(x - r) > 3.8e-6f * x ? x > r : -1;
}
__device__ __forceinline__ bool rotation_wanted_exact(double app, double aqq, double apq, double tol)
{
    const int ep = f64_biased_exp(apq), e1 = f64_biased_exp(app), e2 = f64_biased_exp(aqq);
    const bool safe = ep >= 623 && ep <= 1423 && e1 >= 623 && e1 <= 1423 && e2 >= 623 && e2 <= 1423;
    if (safe) {
        const double lhs = apq * apq, rhs = (tol * tol) * (fabs(app) * fabs(aqq));
        return __double_as_longlong(lhs) > __double_as_longlong(rhs);
    }
    return fabs(apq) > rn_mul(rn_mul(tol, rn_sqrt(fabs(app))), rn_sqrt(fabs(aqq)));
}
__device__ __forceinline__ bool rotation_wanted(double app, double aqq, double apq, double tol)
{
    if ((__double_as_longlong(apq) << 1) == 0) return false;
    const int e1 = f64_biased_exp(app), e2 = f64_biased_exp(aqq), et = f64_biased_exp(tol);
    if (f64_normal_exp(e1) && f64_normal_exp(e2) && f64_normal_exp(et)) {
        const float ft = f64_lead(tol);
        const int w = rotation_wanted_lead(apq, (ft * ft) * (f64_lead(app) * f64_lead(aqq)), e1 + e2 + 2 * et);
        if (w >= 0) return w;
    }
    return rotation_wanted_exact(app, aqq, apq, tol);
}

// (x, y) <- (c x - s y, s x + c y) in Rutishauser's form with tau = s/(1+c):
// x - s (y + tau x), y + s (x - tau y).  Rounding is relative to the
// correction, so vectors keep their length for the small angles of late
// sweeps (where the computed (c, s) have c^2 + s^2 = 1 + u on average).
template <typename T>
__device__ __forceinline__ void rot2(T s, T tau, T& x, T& y)
{
    const T a = x, b = y;
    x = fma(-s, fma(tau, a, b), a);
    y = fma(s, fma(-tau, b, a), b);
}

// (hi, lo) += sgn * t * apq with the product formed exactly (fma) and added
// by an error-free two-sum: the diagonal is carried as hi + lo so that
// rotations whose diagonal change is below half an ulp still move the energy
// of the zeroed entry into the diagonal.
template <typename T>
__device__ __forceinline__ void dd_add_prod(T& hi, T& lo, T t, T apq, T sgn)
{
    T dh = rn_mul(t, apq);
    T dl = fma(t, apq, -dh);
    dh *= sgn;
    dl *= sgn;
    const T a = hi, sum = rn_add(a, dh);
    const T bb = rn_sub(sum, a);
    T err = rn_add(rn_sub(a, rn_sub(sum, bb)), rn_sub(dh, bb));
    err = rn_add(err, rn_add(lo, dl));
    const T h2 = rn_add(sum, err);
    lo = rn_sub(err, rn_sub(h2, sum));
    hi = h2;
}

// Shared scratch of one solve.
template <typename T>
struct CoreSmem {
    T* st;         // two rounds x k/2 pairs x (s, tau), 16-byte aligned
    T* dlo;        // k entries
    int* pk;       // two rounds x k/2: p | q << 10 | (rotate ? 1 << 20 : 0)
    int* cnt;      // one int: rotations of the current sweep
};

template <typename T> struct Pair2;
template <> struct Pair2<float> { using type = float2; };
template <> struct Pair2<double> { using type = double2; };

// Solve the packed symmetric k x k matrix Ap (k even) in place by blockDim.x
// threads.  V (k x k, column-major, ld k) accumulates the rotations when not
// null, in its own type TV (FP32 for a transform that only feeds the split
// low-precision products: the rotation parameters are rounded to TV once per
// use).  Returns the rotations applied; *sweeps_out = sweeps run.  On return
// the diagonal of Ap holds hi + lo rounded once.  Caller: all threads, after
// Ap, V (= I) and sm.dlo (= 0) are initialised and synchronised.
//
// A round has two phases: all threads rotate the round's quads; then the first
// warps choose the next round's rotations (a serial chain that would leave
// the others idle) while the others rotate V by this round, so the
// parameters of two rounds are kept.  The thread that chooses a rotation
// also sets its 2 x 2 block to the exact diagonal form at once: no quad holds
// those entries.  What a round costs is instructions, not arithmetic, so a
// pair's indices and flag are one word and its parameters one load, a thread
// keeps its first quads' pairs in registers, and V is rotated by one warp per
// pair.  2048 FP32 SVDs of 1024 x 64: 14.27 -> 9.60 ms with the same bits.
template <typename T, typename TV = T>
__device__ int jacobi_solve(T* Ap, TV* V, int k, T tol, int max_sweeps, const unsigned* qtab,
                            const CoreSmem<T>& sm, int* sweeps_out)
{
    using T2 = typename Pair2<T>::type;
    constexpr int QC = 4;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int half = k >> 1, nq = half * (half - 1) / 2;
    T2* st = reinterpret_cast<T2*>(sm.st);
    int* pk = sm.pk;
    // choosing threads (whole warps); the rest rotate V meanwhile
    const bool split = V && nt >= 64;
    const int cw = split ? max(32, min((half + 31) & ~31, (nt / 2) & ~31)) : nt;
    unsigned qc[QC];
#pragma unroll
    for (int i = 0; i < QC; ++i) qc[i] = tid + i * nt < nq ? qtab[tid + i * nt] : 0u;
    auto choose = [&](int r, int first, int step) {
        for (int ee = first; ee < half; ee += step) {
            const int pa = ee, pb = k - 1 - ee;
            int va = pa - 1 + r, vb = pb - 1 + r;
            if (va >= k - 1) va -= k - 1;
            if (vb >= k - 1) vb -= k - 1;
            const int ia = pa == 0 ? 0 : 1 + va, ib = 1 + vb;
            const int p = min(ia, ib), q = max(ia, ib), ip = tri(p) + p, iq = tri(q) + q;
            const T app = Ap[ip], aqq = Ap[iq], apq = Ap[iq - q + p];
            const bool on = rotation_wanted(app, aqq, apq, tol);
            const int o = (r & 1) * half + ee;
            pk[o] = p | (q << 10) | (on ? 1 << 20 : 0);
            if (on) {
                T s, t, tau;
                schur2(app, aqq, apq, s, t, tau);
                T2 v;
                v.x = s;
                v.y = tau;
                st[o] = v;
                // the rotated 2 x 2 block: exact diagonal form
                T hp = app, hq = aqq;
                dd_add_prod(hp, sm.dlo[p], t, apq, T(-1));
                dd_add_prod(hq, sm.dlo[q], t, apq, T(1));
                Ap[ip] = hp;
                Ap[iq] = hq;
                Ap[iq - q + p] = T(0);
                atomicAdd(sm.cnt, 1);
            }
        }
    };
    auto rotate_quad = [&](unsigned qq, int so) {   // both-sided rotation of one quad
        const int e1 = qq & 0xffff, e2 = qq >> 16;
        const int w1 = pk[so + e1], w2 = pk[so + e2];
        if (!((w1 | w2) >> 20)) return;
        const int p1 = w1 & 0x3ff, q1 = (w1 >> 10) & 0x3ff, p2 = w2 & 0x3ff, q2 = (w2 >> 10) & 0x3ff;
        const int tp1 = tri(p1), tq1 = tri(q1), tp2 = tri(p2), tq2 = tri(q2);
        const int i00 = p1 >= p2 ? tp1 + p2 : tp2 + p1, i01 = p1 >= q2 ? tp1 + q2 : tq2 + p1;
        const int i10 = q1 >= p2 ? tq1 + p2 : tp2 + q1, i11 = q1 >= q2 ? tq1 + q2 : tq2 + q1;
        T x00 = Ap[i00], x01 = Ap[i01], x10 = Ap[i10], x11 = Ap[i11];
        if (w1 >> 20) {  // rows: J1^T X
            const T2 v = st[so + e1];
            rot2(v.x, v.y, x00, x10);
            rot2(v.x, v.y, x01, x11);
        }
        if (w2 >> 20) {  // columns: X J2
            const T2 v = st[so + e2];
            rot2(v.x, v.y, x00, x01);
            rot2(v.x, v.y, x10, x11);
        }
        Ap[i00] = x00;
        Ap[i01] = x01;
        Ap[i10] = x10;
        Ap[i11] = x11;
    };
    auto rotate_v = [&](int so, int w, int nw) {   // V <- V J, warp w of nw
        for (int ee = w; ee < half; ee += nw) {
            const int word = pk[so + ee];
            if (!(word >> 20)) continue;
            const T2 v = st[so + ee];
            const TV s = (TV)v.x, tau = (TV)v.y;
            TV* vp = V + (size_t)(word & 0x3ff) * k;
            TV* vq = V + (size_t)((word >> 10) & 0x3ff) * k;
            for (int row = tid & 31; row < k; row += 32) {
                TV a = vp[row], b = vq[row];
                rot2(s, tau, a, b);
                vp[row] = a;
                vq[row] = b;
            }
        }
    };
    int total_rot = 0, sweeps = 0;
    for (int sw = 0; sw < max_sweeps; ++sw) {
        if (tid == 0) *sm.cnt = 0;
        __syncthreads();
        choose(0, tid, nt);
        __syncthreads();
        for (int r = 0; r < k - 1; ++r) {
            const int so = (r & 1) * half;
#pragma unroll
            for (int i = 0; i < QC; ++i)
                if (tid + i * nt < nq) rotate_quad(qc[i], so);
            for (int qi = tid + QC * nt; qi < nq; qi += nt) rotate_quad(qtab[qi], so);
            __syncthreads();
            const bool more = r + 1 < k - 1;
            if (!split) {
                if (more) choose(r + 1, tid, nt);
                if (V) rotate_v(so, 0, 1);
            } else if (!more) {
                rotate_v(so, tid >> 5, nt >> 5);
            } else if (tid < cw) {
                choose(r + 1, tid, cw);
            } else {
                rotate_v(so, (tid - cw) >> 5, (nt - cw) >> 5);
            }
            __syncthreads();
        }
        const int cnt = *sm.cnt;
        total_rot += cnt;
        sweeps = sw + 1;
        __syncthreads();
        if (cnt == 0) break;
    }
    for (int x = tid; x < k; x += nt) Ap[tri(x) + x] += sm.dlo[x];  // hi + lo, rounded once
    __syncthreads();
    *sweeps_out = sweeps;
    return total_rot;
}

// Flat quad table for half-size h: entries e1 | e2 << 16 for e1 < e2 < h,
// ordered by e2 then e1 (so a table for h serves every smaller size too).
__device__ __forceinline__ void build_quad_table(unsigned* qtab, int h)
{
    for (int e2 = 1 + threadIdx.x; e2 < h; e2 += blockDim.x)
        for (int e1 = 0; e1 < e2; ++e1) qtab[(e2 * (e2 - 1) >> 1) + e1] = (unsigned)e1 | ((unsigned)e2 << 16);
}

}  // namespace jac
