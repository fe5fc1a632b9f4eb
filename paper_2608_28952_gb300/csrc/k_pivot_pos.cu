// k_pivot_pos.cu -- the pivot solves of one step, C = 1 .. 16 CTAs per
// pair (a thread-block cluster when C > 1): Algorithm 2 applied with b = 1 to
// each 2b x 2b pivot in the round-robin order, the diagonal carried as
// hi + lo.
//
// Layout: by position, not by index.  Round r of the round-robin order pairs
// position e ("top", T_e) with position k - 1 - e ("bottom", B_e); from one
// round to the next every index but the first moves on by one position.  The
// pivot's entries are kept as 2 x 2 quads (i, j), i < j, rows {T_i, B_i} and
// columns {T_j, B_j}, and it is the entries that move: the rotated TT entry of
// quad (i, j) goes to quad (i - 1, j - 1), BB to (i + 1, j + 1), TB to
// (i - 1, j + 1), BT to (i + 1, j - 1), with fixed exceptions at the ends.
// So which thread rotates which quad, and where its four results go, are the
// same in every round: no index table, no address arithmetic and no bank
// conflict in the rounds, and with the quads numbered along i + j a CTA of a
// cluster sends only 2-8 % of its entries to another CTA (an index layout:
// three quarters of them at C = 4).
//
// Roles in a CTA (what bounds a round is the FP64 unit: one warp instruction
// per ~18 cycles for the whole SM, and one per 64 cycles for any one warp, so
// four warps with independent work fill it and more only queue in front of
// the serial chain below):
//   * 4 bulk warps (8 for the largest pivots): each thread owns up to QPT quads:
//     loads them all, rotates them in registers by round g, stores the results
//     at their next positions;
//   * auxiliary warps: this CTA's rows of V, and the diagonal (hi + lo) by the
//     rotations already chosen (where V's rotation would only get in the way
//     of the choice, or has no warps of its own, the bulk warps do it after
//     their quads);
//   * chain warps, two lanes per pair of round g + 1: that pair's entry is one
//     entry of one quad of round g (BT of quad (e - 1, e + 1); TT of (0, 1)
//     and BB of (k/2 - 2, k/2 - 1) at the ends), so a pair of lanes forms that
//     entry (two multiplications and two FMAs), chooses round g + 1's rotation
//     (the top's lane finds tau while the bottom's finds c), sends the
//     parameters to every CTA and (t, a_pq) to whoever carries the two diagonal
//     entries next.  Where auxiliary warps carry the diagonal they also hand
//     over d = aqq - app and its leading bits, ready before the entry is:
//     14 FP64 instructions are left in the chain (k = 32, with shears for
//     rotations: 77.5 -> 69.7 us a launch; 72 with rot2).
// What ends a round (clock stamps, cycles from its start; FP64 V but where said):
//   k, CTAs        quads stored   V done   entry formed   choice sent   round
//   32, 1          1665           3360     925            3310          3550
//   64, 4          1630           3380     920            3490          4240
//   128, 6         6270           7340     2410           6730          8790
//   128, 6, FP32   4020           3730     790            4270          5050
// So at k <= 64 the bulk warps (quads, then V) and the chain (its choice takes
// 2300 to 2600 cycles beside them, 14 x 64 of them FP64 issue) end together; above,
// the FP64 unit, and the slowest CTA's share of it, decides.
// One cluster barrier per round ("round g is stored, round g + 1's parameters
// are there") with two buffers of the quads; where shared memory holds only
// one, a second one ("every quad of round g is in registers") whose wait is
// hidden behind the rotations.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <algorithm>

#include "internal.h"
#include "jacobi_core.cuh"
#include "cluster_common.cuh"
#include "qrcp.cuh"

namespace cg = cooperative_groups;

namespace jac {

namespace {

constexpr size_t PP_STATIC = 4608;              // bound of the static shared arrays
constexpr size_t PP_SMEM_MAX = 227 * 1024 - PP_STATIC;
constexpr int PP_QMAX = 8;      // quads per bulk thread, at most
constexpr int PP_MAXC = 16;     // (clusters above 8 are not portable; GB300 takes 16)

__host__ __device__ inline int pp_quads(int k) { return (k / 2) * (k / 2 - 1) / 2; }
__host__ __device__ inline int pp_chunk(int k, int C) { return (pp_quads(k) + C - 1) / C; }

// Number of the quad (i, j), i < j < h: along m = i + j, then j - i.
__host__ __device__ inline int pp_qid(int i, int j, int h)
{
    const int m = i + j, K = 2 * (h - 1);
    const int off = m <= h - 1 ? (m * m) >> 2 : ((h * (h - 1)) >> 1) - (((K - m + 1) * (K - m + 1)) >> 2);
    return off + ((j - i - 1) >> 1);
}

// The quad that holds the entry of the next round's pair e (h >= 2).
__host__ __device__ inline void pp_lead(int e, int h, int& i, int& j)
{
    i = e == 0 ? 0 : e - 1;
    j = e == 0 ? 1 : (e == h - 1 ? h - 1 : e + 1);
}

__host__ __device__ inline int pp_lead_rank(int e, int h, int chunk)
{
    if (h < 2) return 0;
    int i, j;
    pp_lead(e, h, i, j);
    return pp_qid(i, j, h) / chunk;
}

// Where the index at side t (0 top, 1 bottom) of pair e is in the next round.
__device__ __forceinline__ void pp_next(int& t, int& e, int h)
{
    if (h == 1) return;
    int p = t == 0 ? e : 2 * h - 1 - e;
    if (p > 0) p = p == 1 ? 2 * h - 1 : p - 1;
    t = p >= h;
    e = t ? 2 * h - 1 - p : p;
}

// The index at position pos in a round (rd = round mod (k - 1)).
__device__ __forceinline__ int pp_index(int pos, int rd, int nr)
{
    if (pos == 0) return 0;
    int v = pos - 1 + rd;
    if (v >= nr) v -= nr;
    return 1 + v;
}

__device__ __forceinline__ int pp_pair_map(int I, int J, int b, int x) { return x < b ? I * b + x : J * b + (x - b); }

__device__ __forceinline__ uint32_t pp_mapa(uint32_t a, int rank)
{
    uint32_t o;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(rank));
    return o;
}
__device__ __forceinline__ void pp_st2(uint32_t a, double x, double y)
{
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(x), "d"(y) : "memory");
}
__device__ __forceinline__ void pp_block_barrier(int threads) { asm volatile("barrier.sync 2, %0;" ::"r"(threads) : "memory"); }
__device__ __forceinline__ void pp_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void pp_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// The rotation of a quad.  Rutishauser's form (rot2: four FMAs for two entries)
// rounds each entry once at full size.  Three shears, x1 = x - tau y, y' = y + s x1,
// x' = x1 - tau y', take three FMAs but round x twice: V's loss of orthogonality
// over a solve is 1.25 times rot2's and the errors of singular values and
// residuals 1.15 to 1.25 times (measured, svd 300 x 60 to 2000 x 300).  So an FP64
// result takes rot2 throughout; the shears rotate the FP64 quads of the
// low-precision sweeps alone, which leave as FP32 (the same error against 64 bits
// to two digits, n = 8192, b = 128: one step 4.43 ms, 4.95 with rot2 there; FP64
// solves pay 1.5 % for theirs at n = 64 to 1000, svd 1000 x 200 5 %).
template <bool V32>
__device__ __forceinline__ void quad_rot(double s, double tau, double& x, double& y)
{
    if constexpr (V32) {
        const double u = fma(-tau, y, x);
        y = fma(s, u, y);
        x = fma(-tau, y, u);
    } else {
        rot2(s, tau, x, y);
    }
}

template <bool V32> struct PpV { using T = double; };
template <> struct PpV<true> { using T = float; };

// order-preserving map of doubles to integers (no FP64 comparisons in the sort)
__device__ __forceinline__ long long pp_key(double x)
{
    const long long v = __double_as_longlong(x + 0.0);   // -0 and +0 alike
    return v < 0 ? (long long)0x8000000000000000ull - v : v;
}

struct PpSmem {   // offsets in doubles
    int buf, v, par, dg, prep, cs, fin, par32, ints;
    bool two;     // two buffers of the quads: stores need not wait for the loads
    size_t bytes;
};

__host__ __device__ inline PpSmem pp_smem(int k, int C, bool v32)
{
    const int h = k / 2;
    PpSmem s;
    s.buf = 4 * pp_chunk(k, C) + ((h + 1) & ~1);   // the quads' entries, then the pairs' own
    const int vel = (k + C - 1) / C * k;
    const int vd = ((v32 ? (vel + 1) / 2 : vel) + 1) / 2 * 2;
    const int prep = pp_chunk(k, C) <= 128 * PP_QMAX ? 5 * h : 0;   // (128 bulk threads: with auxiliary warps)
    const int rest = vd + 22 * h + prep + k + (v32 ? 2 * h : 0);
    s.two = (size_t)(2 * s.buf + rest) * 8 + (size_t)(2 * k + 2 * h) * sizeof(int) <= PP_SMEM_MAX;
    s.v = (s.two ? 2 : 1) * s.buf;
    s.par = s.v + vd;                       // params: 2 rounds x h pairs x (s, tau)
    s.dg = s.par + 4 * h;
    s.prep = s.dg + 16 * h;                 // diagonal: (hi, lo) and (t, a_pq), each 2 rounds x 2 sides x h
    s.cs = s.prep + prep;                     // per pair of this CTA's: the next choice's part of the diagonal
    s.fin = s.cs + 2 * h;                   // cosines: 2 rounds x h
    s.par32 = s.fin + k;
    s.ints = s.par32 + (v32 ? 2 * h : 0);   // float2 x 2 rounds x h
    s.bytes = (size_t)s.ints * 8 + (size_t)(2 * k + 2 * h) * sizeof(int);
    return s;
}

// NB bulk threads with QPT quads each, up to CH chain threads and AT auxiliary
// threads; V32: V in FP32, rotated by the auxiliary threads.
template <int NB, int QPT, int CH, int AT, bool V32>
__global__ void __launch_bounds__(NB + CH + AT, 1) k_pivot_pos(PivotArgs a, int C)
{
    // The auxiliary threads rotate V: an FP32 one always; an FP64 one (as much work as the quads)
    // where the FP64 unit bounds the round, not where the rotation choice does
    // and would wait behind four more FP64 warps (one quad per bulk thread;
    // measured: k = 32 72 us with V after the quads, 85 us beside them; k = 128
    // with 16 pairs 695 and 602 us)
    constexpr bool kAuxV = AT > 0 && (V32 || QPT > 1);
    // and carry the diagonal, unless an FP64 V keeps them busy (then the first
    // bulk threads do, and the chain reads its part of the diagonal itself)
    constexpr bool kAuxDiag = AT >= CH && (V32 || !kAuxV);
    using VT = typename PpV<V32>::T;
    extern __shared__ __align__(16) double psm[];
    cg::cluster_group cluster = cg::this_cluster();
    const int r = C > 1 ? (int)cluster.block_rank() : 0;
    const int e0 = blockIdx.x / C, tid = threadIdx.x, nt = blockDim.x;
    const int k = a.k, b = a.b, h = k >> 1, nr = k - 1, NQ = pp_quads(k), chunk = pp_chunk(k, C);
    const int q_lo = min(NQ, r * chunk), nq = min(NQ, q_lo + chunk) - q_lo;
    const int r_lo = r * k / C, rows = (r + 1) * k / C - r_lo;   // of V
    const PpSmem L = pp_smem(k, C, V32);
    // quads by entry [TT TB BT BB][chunk], then the pairs' own entries [h]; round
    // g reads buffer g & 1 and writes the other (or both are one)
    const int flip = L.two ? L.buf : 0, pv0 = 4 * chunk;
    VT* Vl = reinterpret_cast<VT*>(psm + L.v);            // rows x k (ld rows): V(r_lo + i, index j)
    double2* par = reinterpret_cast<double2*>(psm + L.par);   // [round parity][pair] (s, tau); no rotation: (0, 0)
    // the diagonal by position, [round parity][side][pair]: (hi, lo) before the
    // round's rotation, and that rotation's (+-t, a_pq) to apply to it
    double2* dg = reinterpret_cast<double2*>(psm + L.dg);
    double2* dt = dg + 4 * h;
    // what the next choice needs of a pair's diagonal: (app, aqq), the leading
    // parts of d = aqq - app, the right-hand side of the rotation test, d
    double2* pr_ad = reinterpret_cast<double2*>(psm + L.prep);
    float4* pr_f = reinterpret_cast<float4*>(pr_ad + h);
    double* pr_d = reinterpret_cast<double*>(pr_f + h);
    double* cs = psm + L.cs;
    double* fin = psm + L.fin;                            // the diagonal by index: at the start, and at the end
    float2* par32 = reinterpret_cast<float2*>(psm + L.par32);
    int* s_dest = reinterpret_cast<int*>(psm + L.ints);
    int* s_pos = s_dest + k;
    int* s_own = s_pos + k;                               // rank whose chain lanes serve the pair
    int* s_ce = s_own + h;                                // this CTA's chain pairs
    __shared__ int s_nce, s_cntg[4], s_nr, s_r1;
    __shared__ double s_red[(NB + CH + AT) / 32], s_part[PP_MAXC];
    // (the roles run rounds of their own, so they meet at a barrier with a thread
    // count: a __syncthreads() has to be one and the same for the whole block)
    auto sync_all = [&] {
        if (C == 1) {
            pp_block_barrier(nt);
        } else {
            pp_arrive();
            pp_wait();
        }
    };
    // "every quad of the round is in registers": only with one buffer
    auto loaded = [&] {
        if (L.two) return;
        if (C == 1) pp_block_barrier(nt);
        else pp_arrive();
    };
    auto may_store = [&] {
        if (!L.two && C > 1) pp_wait();
    };
    int I, J;
    bool frozen;
    {
        const int2 pr = a.pairs[e0];
        frozen = pr.x < 0;
        I = frozen ? -1 - pr.x : pr.x;
        J = frozen ? -1 - pr.y : pr.y;
    }
    // entry (x, y) of the pivot by index in the first round's arrangement
    auto pivot_in = [&](int x, int y) -> double {   // x >= y
        if (a.gram) {
            const double* g = a.gram + (size_t)e0 * a.npanels * k * k + x + (size_t)k * y;
            double s = 0.0;
            for (int p = 0; p < a.npanels; ++p) s += g[(size_t)p * k * k];   // fixed order
            return s;
        }
        const size_t gi = pp_pair_map(I, J, b, x) + (size_t)a.ld * pp_pair_map(I, J, b, y);
        return a.Ain32 ? (double)a.Ain32[gi] : a.Ain[gi];
    };
    // local slot of the off-diagonal entry (x, y) by index (first round's
    // arrangement), or -1 when another CTA holds it
    auto slot_of = [&](int x, int y) -> int {
        const int ex = x < h ? x : k - 1 - x, ey = y < h ? y : k - 1 - y;
        if (ex == ey) return s_own[ex] == r ? pv0 + ex : -1;
        const int sx = x >= h, sy = y >= h;
        const int i = min(ex, ey), j = max(ex, ey), si = ex < ey ? sx : sy, sj = ex < ey ? sy : sx;
        const int q = pp_qid(i, j, h) - q_lo;
        return q >= 0 && q < nq ? (2 * si + sj) * chunk + q : -1;
    };

    for (int e = tid; e < h; e += nt) s_own[e] = pp_lead_rank(e, h, chunk);
    __syncthreads();
    if (tid == 0) {
        int c = 0;
        for (int e = 0; e < h; ++e)
            if (s_own[e] == r) s_ce[c++] = e;
        s_nce = c;
        for (int u = 0; u < 4; ++u) s_cntg[u] = 0;
    }
    // ---- load: this CTA's entries, the whole diagonal, V rows = identity rows
    for (int idx = tid; idx < k * k; idx += nt) {
        const int x = idx % k, y = idx / k;
        if (x < y) continue;
        if (x == y) {
            fin[x] = pivot_in(x, x);
            continue;
        }
        const int o = slot_of(x, y);
        if (o >= 0) psm[o] = pivot_in(x, y);
    }
    for (int idx = tid; idx < rows * k; idx += nt) {
        const int i = idx % rows, j = idx / rows;
        Vl[idx] = (r_lo + i == j) ? VT(1) : VT(0);
    }
    __syncthreads();

    // ---- one-sided stop statistic (Gram pivots): max |a_xy| / sqrt(a_xx a_yy)
    // over the cluster, from one reciprocal square root per index
    if (a.relmax) {
        double* rs = reinterpret_cast<double*>(dg);   // k doubles; dg is written later
        for (int x = tid; x < k; x += nt) rs[x] = fin[x] > 0.0 ? 1.0 / sqrt(fin[x]) : 0.0;
        __syncthreads();
        double mx = 0.0;
        if (!frozen)
            for (int idx = tid; idx < k * k; idx += nt) {
                const int x = idx % k, y = idx / k;
                if (x <= y) continue;
                const int o = slot_of(x, y);
                if (o >= 0) mx = fmax(mx, (fabs(psm[o]) * rs[x]) * rs[y]);
            }
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((tid & 31) == 0) s_red[tid >> 5] = mx;
        __syncthreads();
        if (tid == 0) {
            double m = 0.0;
            for (int w = 0; w < nt / 32; ++w) m = fmax(m, s_red[w]);
            if (C > 1) *cluster.map_shared_rank(&s_part[r], 0) = m;
            else s_part[0] = m;
        }
        sync_all();
        if (r == 0 && tid == 0) {
            double m = 0.0;
            for (int u = 0; u < C; ++u) m = fmax(m, s_part[u]);
            a.relmax[e0] = m;
        }
    }
    // every CTA of the cluster runs and has its tables before the first remote store
    sync_all();

    const double tol = a.tol_rel;
    const int max_sweeps = frozen ? 0 : a.max_sweeps;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(psm);
    int total_rot = 0, sweeps = 0, G = 0;
    const int role = tid < NB ? 0 : (tid >= nt - AT ? 2 : 1);

    // where a rotated entry goes: rank << sh | slot, the same in every round
    const int sh = C > 8 ? 12 : (C > 4 ? 13 : 14);
    const uint32_t smask = (1u << sh) - 1u;
    auto put = [&](int to, uint32_t d, double v) {
        const int rk = (int)(d >> sh);
        const uint32_t sl = to + (d & smask);
        if (rk == r) psm[sl] = v;
        else dsm_st(pp_mapa(sbase + 8u * sl, rk), v);
    };
    auto place = [&](int si, int i, int sj, int j) -> uint32_t {   // next place of the entry (side si of pair i, sj of j)
        pp_next(si, i, h);
        pp_next(sj, j, h);
        if (i == j) return (uint32_t)((s_own[i] << sh) | (pv0 + i));   // a pair's own entry (kept for the end)
        const int id = i < j ? pp_qid(i, j, h) : pp_qid(j, i, h), rk = id / chunk;
        return (uint32_t)((rk << sh) | ((i < j ? 2 * si + sj : 2 * sj + si) * chunk + (id - rk * chunk)));
    };
    int* cnt0 = C > 1 ? cluster.map_shared_rank(s_cntg, 0) : s_cntg;
    // every role runs the same rounds; body(g, sw, rd, last) passes loaded() and
    // may_store() once each
    auto rounds = [&](auto body) {
        if (max_sweeps > 0) {   // round 0 is chosen
            sync_all();
        }
        for (int sw = 0; sw < max_sweeps; ++sw) {
            // the counter of sweep sw + 2 was last read after sweep sw - 2
            if (r == 0 && tid == 0) s_cntg[(sw + 2) & 3] = 0;
            for (int rd = 0; rd < nr; ++rd) {
                body(sw * nr + rd, sw, rd, rd == nr - 1 && sw + 1 == max_sweeps);
                sync_all();
            }
            G += nr;
            const int cnt = cnt0[sw & 3];
            total_rot += cnt;
            sweeps = sw + 1;
            if (cnt == 0) break;
        }
    };
    // this CTA's rows of V by the round, by thread vt of VN.  Whole warps of
    // rows: a warp takes pairs, a lane a row; else the (pair, row) items dealt
    // to the threads in order.
    const int vt = role == 2 ? tid - (nt - AT) : tid;
    constexpr int VN = kAuxV ? AT : NB;
    const bool vwarp = rows % 32 == 0;
    const int ve0 = vwarp ? vt >> 5 : vt / rows, vi0 = vwarp ? vt & 31 : vt - ve0 * rows;
    const int vde = vwarp ? VN / 32 : VN / rows, vdi = vwarp ? 0 : VN - vde * rows;
    auto rotate_v = [&](int so, int rd) {
        constexpr int U = NB > 128 && !kAuxV ? 2 : 4;   // items in flight: 4 (256 bulk threads and more: 2 of each row
        constexpr int UO = NB > 128 && !kAuxV ? 4 : 1;  // group, which costs fewer registers)
        int e = ve0, i = vi0;
        while (e < h) {
            int ot[U], ob[U];
            VT ps[U], pu[U];
            bool on[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                on[u] = e < h;
                const int f = min(e, h - 1);
                ot[u] = rows * pp_index(f, rd, nr) + i;
                ob[u] = rows * pp_index(k - 1 - f, rd, nr) + i;
                if constexpr (V32) {
                    const float2 p = par32[so + f];
                    ps[u] = p.x;
                    pu[u] = p.y;
                } else {
                    const double2 p = par[so + f];
                    ps[u] = p.x;
                    pu[u] = p.y;
                }
                e += vde;
                i += vdi;
                if (i >= rows) {
                    i -= rows;
                    ++e;
                }
            }
#pragma unroll UO
            for (int o = 0; o < (vwarp ? rows : 1); o += 32) {
                VT xt[U], xb[U];
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (on[u]) {
                        xt[u] = Vl[ot[u] + o];
                        xb[u] = Vl[ob[u] + o];
                    }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (on[u]) {
                        rot2(ps[u], pu[u], xt[u], xb[u]);
                        Vl[ot[u] + o] = xt[u];
                        Vl[ob[u] + o] = xb[u];
                    }
            }
        }
    };
    // the diagonal, carried as hi + lo by one thread per entry (ld: its number
    // among this CTA's): the round's rotation applied, sent to the next position
    const bool dcar = role == (kAuxDiag ? 2 : 0) && (vt >> 1) < s_nce;
    const int dside = vt & 1, de = dcar ? s_ce[vt >> 1] : 0;
    int dg_to = 0, dg_rank = 0;
    if (dcar) {
        int t1 = dside, e1 = de;
        pp_next(t1, e1, h);
        dg_to = t1 * h + e1;
        dg_rank = s_own[e1];
    }
    auto put_diag = [&](int g, double hi, double lo) {
        double2* d = dg + (g & 1) * 2 * h + dg_to;
        if (dg_rank == r) *d = make_double2(hi, lo);
        else pp_st2(pp_mapa((uint32_t)__cvta_generic_to_shared(d), dg_rank), hi, lo);
    };
    const int tol_e = f64_biased_exp(tol);
    const float tol_f = f64_lead(tol) * f64_lead(tol);
    // leading parts of a pair's diagonal for the next choice
    auto prepare = [&](double app, double aqq, double d) {
        const int e1 = f64_biased_exp(app), e2 = f64_biased_exp(aqq);
        const bool ok = f64_normal_exp(e1) && f64_normal_exp(e2) && f64_normal_exp(tol_e);
        return make_float4(f64_lead(d), f64_rest(d), tol_f * (f64_lead(app) * f64_lead(aqq)),
                           __int_as_float(ok ? e1 + e2 + 2 * tol_e : -1));
    };
    auto rotated_diag = [&](int g, double& hi, double& lo) {
        const int o = (2 * (g & 1) + dside) * h + de;
        const double2 d = dg[o], c = dt[o];
        hi = d.x;
        lo = d.y;
        dd_add_prod(hi, lo, c.x, c.y, 1.0);
    };
    auto carry_diag = [&](int g) {
        if (!dcar) return;
        double hi, lo;
        rotated_diag(g, hi, lo);
        put_diag(g + 1, hi, lo);
    };
    // the same by auxiliary warps, which first hand the chain its part of it
    const int pair_threads = nt - NB;   // chain and auxiliary threads
    auto carry_diag_for_chain = [&](int g, bool last) {
        double2 d = make_double2(0.0, 0.0), c = d;
        if (dcar) {
            const int o = (2 * (g & 1) + dside) * h + de;
            d = dg[o];
            c = dt[o];
        }
        if (!last) {
            const double dv = d.x + fma(c.x, c.y, d.y), other = __shfl_xor_sync(0xffffffffu, dv, 1);
            if (dcar && dside == 0) {
                const double df = rn_sub(other, dv);
                pr_ad[de] = make_double2(dv, other);
                pr_f[de] = prepare(dv, other, df);
                pr_d[de] = df;
            }
            asm volatile("barrier.arrive 1, %0;" ::"r"(pair_threads) : "memory");
        }
        if (!dcar) return;
        dd_add_prod(d.x, d.y, c.x, c.y, 1.0);
        put_diag(g + 1, d.x, d.y);
    };
    if (dcar && max_sweeps > 0) put_diag(0, fin[dside ? k - 1 - de : de], 0.0);
    if (role == 0) {
        int ij[QPT];
        uint32_t dst[2 * QPT];
#pragma unroll
        for (int u = 0; u < QPT; ++u) {
            ij[u] = 0;
            dst[2 * u] = dst[2 * u + 1] = 0;
            const int q = q_lo + tid + u * NB;
            if (q >= q_lo + nq) continue;
            int m = 1;                        // the diagonal i + j = m that holds quad q; its first is (i0, m - i0)
            for (int step = 128; step > 0; step >>= 1) {
                const int mm = m + step, i0 = (mm - 1) >> 1;
                if (mm <= 2 * h - 3 && pp_qid(i0, mm - i0, h) <= q) m = mm;
            }
            const int i0 = (m - 1) >> 1, off = q - pp_qid(i0, m - i0, h);
            const int i = i0 - off, j = m - i0 + off;
            ij[u] = i | (j << 8);
            dst[2 * u] = place(0, i, 0, j) | (place(0, i, 1, j) << 16);
            dst[2 * u + 1] = place(1, i, 0, j) | (place(1, i, 1, j) << 16);
        }
        unsigned local = 0;   // bit u: all of quad u's entries stay in this CTA
#pragma unroll
        for (int u = 0; u < QPT; ++u) {
            bool l = true;
#pragma unroll
            for (int t = 0; t < 4; ++t) l &= (int)(((dst[2 * u + (t >> 1)] >> (16 * (t & 1))) & 0xffffu) >> sh) == r;
            if (l) {              // (and then without the rank)
                local |= 1u << u;
                dst[2 * u] &= smask | (smask << 16);
                dst[2 * u + 1] &= smask | (smask << 16);
            }
        }
        rounds([&](int g, int, int rd, bool) {
            const int so = (g & 1) * h, from = (g & 1) * flip, to = flip - from;
            const double* st = psm + from;
            double x[QPT][4];
#pragma unroll
            for (int u = 0; u < QPT; ++u) {
                const int q = tid + u * NB;
                if (q < nq) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) x[u][t] = st[t * chunk + q];
                }
            }
            loaded();
#pragma unroll
            for (int u = 0; u < QPT; ++u) {
                if (tid + u * NB < nq) {
                    const double2 pi = par[so + (ij[u] & 0xff)], pj = par[so + (ij[u] >> 8)];
                    quad_rot<V32>(pi.x, pi.y, x[u][0], x[u][2]);
                    quad_rot<V32>(pi.x, pi.y, x[u][1], x[u][3]);
                    quad_rot<V32>(pj.x, pj.y, x[u][0], x[u][1]);
                    quad_rot<V32>(pj.x, pj.y, x[u][2], x[u][3]);
                }
            }
            may_store();
            double* sn = psm + to;
#pragma unroll
            for (int u = 0; u < QPT; ++u) {
                if (tid + u * NB < nq) {
                    const uint32_t d0 = dst[2 * u] & 0xffffu, d1 = dst[2 * u] >> 16;
                    const uint32_t d2 = dst[2 * u + 1] & 0xffffu, d3 = dst[2 * u + 1] >> 16;
                    if ((local >> u) & 1) {
                        sn[d0] = x[u][0];
                        sn[d1] = x[u][1];
                        sn[d2] = x[u][2];
                        sn[d3] = x[u][3];
                    } else {
                        put(to, d0, x[u][0]);
                        put(to, d1, x[u][1]);
                        put(to, d2, x[u][2]);
                        put(to, d3, x[u][3]);
                    }
                }
            }
            if constexpr (!kAuxDiag) carry_diag(g);
            if constexpr (!kAuxV) rotate_v(so, rd);
        });
    } else if (role == 1) {
        const int cl = tid - NB, lead = cl & 1;            // lead: 0 the top's lane, 1 the bottom's
        const bool mine = (cl >> 1) < s_nce;
        const int ce = mine ? s_ce[cl >> 1] : 0;           // the pair
        double pv = 0.0;                                   // its entry after its rotation
        int ci = 0, cj = 0, cslot = 0;
        uint32_t pvd = 0;
        if (mine && h >= 2) {
            pp_lead(ce, h, ci, cj);
            cslot = pp_qid(ci, cj, h) - q_lo + lead * chunk;
            pvd = place(0, ce, 1, ce);
        }
        int nrot = 0;                                      // rotations this lane chose for the sweep
        auto flush = [&](int sw) {
            const int n = __reduce_add_sync(0xffffffffu, nrot);
            if (n && (tid & 31) == 0) atomicAdd(&cnt0[sw & 3], n);
            nrot = 0;
        };
        int t1 = lead, e1 = ce;                            // where this lane's index goes
        pp_next(t1, e1, h);
        const int dgd = t1 * h + e1, dgr = s_own[e1];
        // The rotation of round g for the pair's entry av, (app, aqq) = ad, their
        // difference d and its leading parts f: parameters to every CTA, and the
        // change of the diagonal to the lanes that hold its next position.  The
        // top's lane finds tau, the bottom's the cosine.
        auto choose = [&](int g, int rd, double av, double2 ad, double d, float4 f) {
            const int es = __float_as_int(f.w);
            int want = es >= 0 ? rotation_wanted_lead(av, f.z, es) : -1;
            if (want < 0) want = (__double_as_longlong(av) << 1) != 0 && rotation_wanted_exact(ad.x, ad.y, av, tol);
            const bool on = mine && want;
            double s, t = 0.0, z = 0.0;
            const bool paired = on && schur2_half(d, av, f.x, f.y, lead, t, z);
            const double zo = __shfl_xor_sync(0xffffffffu, z, 1);
            double tau = lead ? zo : z, c = lead ? z : zo;
            if (on) {   // zeta = 0: t = +1 with the smaller index as p
                schur2_join(d, av, paired, pp_index(ce, rd, nr) > pp_index(k - 1 - ce, rd, nr), s, t, tau, c);
            } else {
                s = t = tau = 0.0;
                c = 1.0;
            }
            if (mine) {
                const int sl = (g & 1) * h + ce;
                for (int u = lead; u < C; u += 2) {
                    if (u == r) {
                        par[sl] = make_double2(s, tau);
                        cs[sl] = c;
                        if (V32) par32[sl] = make_float2(f32_of(s), f32_of(tau));
                    } else {
                        pp_st2(pp_mapa((uint32_t)__cvta_generic_to_shared(par + sl), u), s, tau);
                        dsm_st(pp_mapa((uint32_t)__cvta_generic_to_shared(cs + sl), u), c);
                        if (V32) {
                            const uint32_t ad32 = pp_mapa((uint32_t)__cvta_generic_to_shared(par32 + sl), u);
                            dsm_st(ad32, f32_of(s));
                            dsm_st(ad32 + 4, f32_of(tau));
                        }
                    }
                }
                const double tl = lead ? t : f64_flip(t, 0x80000000), al = on ? av : 0.0;
                double2* dd = dt + (g & 1) * 2 * h + dgd;
                if (dgr == r) *dd = make_double2(tl, al);
                else pp_st2(pp_mapa((uint32_t)__cvta_generic_to_shared(dd), dgr), tl, al);
                pv = on ? 0.0 : av;
            }
            nrot += on && lead == 0;
        };
        if (max_sweeps > 0) {
            const double2 ad = make_double2(fin[ce], fin[k - 1 - ce]);
            const double d = rn_sub(ad.y, ad.x);
            choose(0, 0, mine ? psm[pv0 + ce] : 0.0, ad, d, prepare(ad.x, ad.y, d));
        }
        rounds([&](int g, int sw, int rd, bool last) {
            const int so = (g & 1) * h, from = (g & 1) * flip, to = flip - from;
            const double* st = psm + from;
            double av = pv, x0 = 0.0, x2 = 0.0, si = 0.0, cci = 1.0, sj = 0.0, ccj = 1.0;
            const double pv_old = pv;
            if (mine && h >= 2) {   // this lane's column of the quad: the top's or the bottom's of pair cj
                x0 = st[cslot];
                x2 = st[cslot + 2 * chunk];
                si = par[so + ci].x;
                cci = cs[so + ci];
                sj = par[so + cj].x;
                ccj = cs[so + cj];
            }
            double2 ad = make_double2(0.0, 0.0);
            double d = 0.0;
            float4 f = make_float4(1.0f, 0.0f, 1.0f, 0.0f);
            if constexpr (!kAuxDiag) {   // no auxiliary warps: the diagonal after round g from its own change
                double dv = 0.0;
                if (mine) {
                    const int o = (2 * (g & 1) + lead) * h + ce;
                    const double2 x = dg[o], y = dt[o];
                    dv = x.x + fma(y.x, y.y, x.y);
                }
                const double other = __shfl_xor_sync(0xffffffffu, dv, 1);
                ad = lead ? make_double2(other, dv) : make_double2(dv, other);
                d = rn_sub(ad.y, ad.x);
                f = prepare(ad.x, ad.y, d);
            }
            loaded();
            if (!last) {
                if (h >= 2) {
                    // row of the entry: pair ci's bottom s T + c B, or for pair 0 its top c T - s B
                    const bool top = ce == 0, bot = ce == h - 1;
                    const double y = fma(top ? f64_flip(si, 0x80000000) : si, top ? x2 : x0, cci * (top ? x0 : x2));
                    const double yo = __shfl_xor_sync(0xffffffffu, y, 1);
                    const double yt = lead ? yo : y, yb = lead ? y : yo;
                    // column: pair cj's top, or its bottom for the last pair
                    av = fma(bot ? sj : f64_flip(sj, 0x80000000), bot ? yt : yb, ccj * (bot ? yb : yt));
                }
                if constexpr (kAuxDiag) {
                    asm volatile("barrier.sync 1, %0;" ::"r"(pair_threads) : "memory");
                    if (mine) {
                        ad = pr_ad[ce];
                        d = pr_d[ce];
                        f = pr_f[ce];
                    }
                }
                if (rd + 1 == nr) flush(sw);
                choose(g + 1, rd + 1 == nr ? 0 : rd + 1, av, ad, d, f);
            } else {
                flush(sw);
            }
            may_store();
            if (mine && lead == 0) {
                if (h >= 2) put(to, pvd, pv_old);
                else psm[to + pv0] = pv_old;
            }
        });
    } else {
        rounds([&](int g, int, int rd, bool last) {
            loaded();
            if constexpr (kAuxDiag) carry_diag_for_chain(g, last);
            if constexpr (kAuxV) rotate_v((g & 1) * h, rd);
            may_store();
        });
    }
    // ---- the final diagonal, hi + lo rounded once, by index, in every CTA
    // (after whole sweeps the positions are the first round's again)
    if (dcar && G > 0) {
        double hi, lo;
        rotated_diag(G - 1, hi, lo);
        const double v = hi + lo;
        const int x = dside ? k - 1 - de : de;
        for (int u = 0; u < C; ++u) {
            if (u == r) fin[x] = v;
            else dsm_st(pp_mapa((uint32_t)__cvta_generic_to_shared(fin + x), u), v);
        }
    }
    sync_all();

    // ---- permutation (identical in every CTA: same diagonal; the QRCP order
    // of Sec. 2.1's pivoting step is computed by rank 0 on the leading rows of
    // Vhat, gathered from the CTAs that own them, and sent to every CTA)
    if (tid == 0) {
        int n = 0, r1 = 0;
        for (int x = 0; x < k; ++x)
            if (pp_pair_map(I, J, b, x) < a.n_real) {
                r1 += x < b;
                s_pos[n++] = x;
            }
        s_nr = n;
        s_r1 = r1;
    }
    __syncthreads();
    if (a.order == 2 && total_rot > 0) {
        __shared__ int s_perm[256];
        __shared__ double s_cn[256], s_vh[128];
        const int n = s_nr, r1 = s_r1;
        double* M = a.qrws + (size_t)e0 * b * k;
        for (int idx = tid; idx < r1 * n; idx += nt) {   // this CTA's leading rows of Vhat
            const int i = idx % r1, j = idx / r1, row = s_pos[i];
            if (row >= r_lo && row < r_lo + rows) M[idx] = Vl[(row - r_lo) + (size_t)rows * s_pos[j]];
        }
        __threadfence();
        sync_all();
        if (r == 0) {
            qrcp_order(r1, n, M, s_perm, s_cn, s_vh);
            for (int x = tid; x < k; x += nt) s_dest[x] = x;
            __syncthreads();
            for (int t = tid; t < n; t += nt) s_dest[s_pos[s_perm[t]]] = s_pos[t];
            __syncthreads();
            for (int u = 1; u < C; ++u) {
                int* rdst = cluster.map_shared_rank(s_dest, u);
                for (int x = tid; x < k; x += nt) rdst[x] = s_dest[x];
            }
        }
        sync_all();
    } else {
        for (int x = tid; x < k; x += nt) {
            int dest = x;
            if (a.order == 1 && total_rot > 0 && pp_pair_map(I, J, b, x) < a.n_real) {
                const long long dx = pp_key(fin[x]);
                int rr = 0;
                for (int t = 0; t < s_nr; ++t) {
                    const int y = s_pos[t];
                    const long long dy = pp_key(fin[y]);
                    rr += (dy > dx) || (dy == dx && y < x);
                }
                dest = s_pos[rr];
            }
            s_dest[x] = dest;
        }
        __syncthreads();
    }

    // ---- outputs: this CTA's rows of V (and the matching columns of V^T), its entries of D
    double* Vo = a.V + (size_t)e0 * 2 * k * k;
    for (int idx = tid; idx < rows * k; idx += nt) {
        const int i = idx % rows, j = idx / rows;
        const double v = Vl[idx];  // V(r_lo + i, j) -> column s_dest[j]
        Vo[(r_lo + i) + (size_t)k * s_dest[j]] = v;
        Vo[(size_t)k * k + s_dest[j] + (size_t)k * (r_lo + i)] = v;
    }
    if (a.Aout || a.Aout32) {
        for (int idx = tid; idx < k * k; idx += nt) {
            const int x = idx % k, y = idx / k;
            const int o = x == y ? (x >= r_lo && x < r_lo + rows ? 0 : -1) : slot_of(x, y);
            if (o < 0) continue;
            const double v = x == y ? fin[x] : psm[o + (G & 1) * flip];
            const size_t g = pp_pair_map(I, J, b, s_dest[x]) + (size_t)a.ld * pp_pair_map(I, J, b, s_dest[y]);
            if (a.Aout32) a.Aout32[g] = (float)v;
            else a.Aout[g] = v;
        }
    }
    if (r == 0 && tid == 0) {
        a.rot[e0] = total_rot;
        atomicAdd(&a.cnt->rotations, (unsigned long long)total_rot);
        atomicAdd(&a.cnt->inner_sweeps, (unsigned long long)sweeps);
        if (!frozen) atomicAdd(&a.cnt->pair_solves, 1ull);
        atomicAdd(&a.cnt->flops_fp64, (unsigned long long)total_rot * (unsigned long long)((a.v32 ? 12 : 18) * k));
    }
    // no CTA may leave while others can still read or write its shared memory
    sync_all();
}

using PpKernel = void (*)(PivotArgs, int);

// 128 bulk threads while they hold a CTA's quads in registers (four warps fill
// the FP64 unit), else 256, or 288 for the few largest shares that shared
// memory still takes (2b = 184 and 186 with C = 2, 224 with 3; one step of 76 pairs,
// b = 92, low precision: 8.8 ms, 14.8 with one CTA per pair).  A block's warps
// per SM quarter set the registers a thread may use: with 128 bulk threads, 4
// auxiliary warps fit; with 256 the diagonal goes to bulk threads and an FP32 V
// to one warp, with 288 both go to bulk threads.  Null where no instance holds
// the share.
template <bool V32>
PpKernel pp_kernel(int chunk, int chain, int& nb, int& at)
{
    nb = chunk > 256 * PP_QMAX ? 288 : (chunk > 128 * PP_QMAX ? 256 : 128);
    const int qpt = (chunk + nb - 1) / nb;
    if (nb == 288) {
        at = 0;
        return qpt <= PP_QMAX && chain <= 96 ? k_pivot_pos<288, PP_QMAX, 96, 0, V32> : nullptr;
    }
    if (nb == 256) {
        at = V32 ? 32 : 0;
        if (chain > 128) return nullptr;
        return chain <= 96 ? k_pivot_pos<256, PP_QMAX, 96, V32 ? 32 : 0, V32> : k_pivot_pos<256, PP_QMAX, 128, V32 ? 32 : 0, V32>;
    }
    at = 128;
    if (chain > 96) return nullptr;
    if (qpt <= 1) return k_pivot_pos<128, 1, 96, 128, V32>;
    if (qpt <= 2) return k_pivot_pos<128, 2, 96, 128, V32>;
    if (qpt <= 4) return k_pivot_pos<128, 4, 96, 128, V32>;
    return k_pivot_pos<128, PP_QMAX, 96, 128, V32>;
}

}  // namespace

namespace {

// Kernel, block and shared memory of the pivot solves of order k with C CTAs
// per pair.
struct PpLaunch {
    PpKernel kern;
    int threads;
    size_t smem;
};

PpLaunch pp_launch(int k, int C, bool v32)
{
    const int h = k / 2, chunk = pp_chunk(k, C);
    int cnt[PP_MAXC] = {}, most = 1;
    for (int e = 0; e < h; ++e) most = std::max(most, ++cnt[pp_lead_rank(e, h, chunk)]);
    const int chain = (2 * most + 31) / 32 * 32;
    int nb, at;
    PpLaunch l;
    l.kern = v32 ? pp_kernel<true>(chunk, chain, nb, at) : pp_kernel<false>(chunk, chain, nb, at);
    l.threads = nb + chain + at;
    l.smem = pp_smem(k, C, v32).bytes;
    return l;
}

cudaError_t pp_config(const PpLaunch& l, int C, int npairs, cudaLaunchAttribute* attr, cudaLaunchConfig_t* cfg)
{
    if (!l.kern) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(l.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)std::max(l.smem, PP_SMEM_MAX));
    if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(l.kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = C;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->gridDim = dim3(npairs * C);
    cfg->blockDim = dim3(l.threads);
    cfg->dynamicSmemBytes = l.smem;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    return cudaSuccess;
}

}  // namespace

bool pivot_pos_fits(int k, int C, size_t smem_cap)
{
    return C <= PP_MAXC && (C == 1 || k / C >= 8) && pp_smem(k, C, false).bytes + PP_STATIC <= smem_cap &&
           pp_launch(k, C, false).kern && pp_launch(k, C, true).kern;
}

// Cluster size for a step with npairs pairs: the largest C whose
// clusters can all run at once (asked of the runtime: a GPU part holds whole
// clusters only, so npairs * C <= SMs is not enough) and that still pays, or 1.
// A round's FP64 work per CTA shrinks with C while the rotation choice and the
// cluster barrier do not.  Measured on GB300, us per launch with C = 1 / 2 / 4
// / 8: k = 32 (8 pairs) 72 / 78 / 79 / -; k = 40 132 / 99 / 96 / -; k = 64 369 / 218 /
// 158 / 150; k = 96 (5 pairs) 1135 / 660 / 426 / 291; k = 128 (4 pairs) 2490 / 1317 /
// 763 / 447, with 6 CTAs 600, 12 422, 16 338.  Two waves of larger clusters lose:
// 16 pairs at k = 64 291 with 8 CTAs, at k = 128 888 with 8 and 602 with 6; 32
// pairs at k = 256 8112 with 8 and 5138 with 4.
int pivot_cluster_size(int k, int npairs, size_t smem_cap)
{
    const int cmax = k <= 32 ? 1 : (k <= 64 ? 4 : (k <= 96 ? 8 : PP_MAXC));
    int least = 2;   // above k = 128, several waves of the smallest clusters beat one CTA on global scratch
    while (least <= PP_MAXC && !pivot_pos_fits(k, least, smem_cap)) ++least;
    for (int C = cmax; C > 1; --C) {
        if (!pivot_pos_fits(k, C, smem_cap)) continue;
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = {};
        const PpLaunch l = pp_launch(k, C, false);
        int n = 0;
        if (pp_config(l, C, npairs, attr, &cfg) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, l.kern, &cfg) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        if (n >= npairs || (k > 128 && C == least && n > 0)) return C;
    }
    return 1;
}

cudaError_t launch_pivot_pos(const PivotArgs& a, int C, cudaStream_t s)
{
    if (a.npairs <= 0) return cudaSuccess;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = {};
    const PpLaunch l = pp_launch(a.k, C, a.v32 != 0);
    const cudaError_t e = pp_config(l, C, a.npairs, attr, &cfg);
    if (e != cudaSuccess) return e;
    cfg.stream = s;
    // with all of an SM's shared memory no CTA of a kernel that runs beside this
    // one shares the SM's FP64 unit with the rotation choice
    if (a.alone) cfg.dynamicSmemBytes = PP_SMEM_MAX;
    return cudaLaunchKernelEx(&cfg, l.kern, a, C);
}

}  // namespace jac
