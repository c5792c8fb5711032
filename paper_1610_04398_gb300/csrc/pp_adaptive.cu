// Pressure at every cell of an adaptive (multiresolution) grid, Eq. greenSum with each source
// cell clamped at its own rho_h: the fast multipole method on the tree and the interaction
// lists of pp_atree (dual-tree walk), in FP64 and in mixed precision.  Leaves are blocks of
// 8 x 8 cells; a box of level l has side s = 2^-l of the unit domain and centre
// ((ix + 1/2) s, (iy + 1/2) s).  Expansions are kept in units of their own box side (multipole
// M_k = alpha_k / s^k, local L_l = b_l s^l, Appendix A.2's series and their standard local
// shifts, for 2 pi P), every translation factored as diagonal * real matrix * diagonal:
//   P2M   S = sum q, M_k = sum q w^k / k, w = (z - c) / s (table of w^k / k)
//   M2M   parent M_k = zeta^k [S / k + sum_{j<=k} C(k-1, j-1) (2 zeta)^-j M_j], zeta = (+-1 +- i) / 4
//   M2L   with tau = (c_src - c_tgt) / s_tgt, rho = s_src / s_tgt, x_k = -M_k (-rho/tau)^k:
//         L_0 += S (log|tau| + log s_tgt) + Re sum_k x_k,
//         L_l += tau^-l (-S / l + sum_k x_k C(l+k-1, k-1))
//   L2L   child L_l += (2 zeta)^-l sum_{k>=l} C(k, l) zeta^k L_k
//   L2P   P = Re sum_l L_l w^l / (2 pi); near field over the near-field leaf pairs from tables
//         of log|D| over the integer cell offsets D of the pair (below).
// A solve is three launches: the upward pass (k_aup), the translations (k_am2l) and, per
// leaf, the shifts down its path, the local evaluation and the near field (k_aleaf).  Every
// sum runs in a fixed order, so results repeat bitwise.  The first solve on a tree uploads
// the tree, the lists and the tables and allocates the expansions; they stay with the tree.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <new>
#include <vector>

#include "../../include/pp.h"
#include "pp_atree_state.h"
#include "pp_common.h"
#include "pp_fixed.cuh"
#include "pp_log.cuh"

namespace {

using pp::cplx_of;
using pp::df_add;
using pp::df_fma;
using pp::df_to;
using pp::mad_wide;

constexpr int kMaxOrderA = 30;
constexpr int kTP = 32;  // stride (coefficients) of the expansion arrays and of the tables
constexpr double kInv2PiA = 0.15915494309189533576888376337251;
constexpr double kC0A = 0.78539816339744830962 - 1.5 - 0.34657359027997265471;  // pi/4 - 3/2 - ln2/2
constexpr double kLn2A = 0.69314718055994530941723212145818;
constexpr double kLn2Lo = 2.319046813846299558417771e-17;  // log 2 - kLn2A

struct AGeo {
    double cx, cy, s;     // centre and side
    int level, ix, iy;    // the box's position in the tree
};

__host__ __device__ __forceinline__ double2 zmul(double2 a, double2 b) {
    return double2{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
__host__ __device__ __forceinline__ double2 zscale(double2 a, double f) { return double2{a.x * f, a.y * f}; }

// Cell (cx, cy) of a leaf block, index cy * 8 + cx, in units of the block side about its centre.
__host__ __device__ __forceinline__ double2 cell_w(int c) {
    return double2{((c & 7) + 0.5) / 8.0 - 0.5, ((c >> 3) + 0.5) / 8.0 - 0.5};
}

template <typename T>
__device__ __forceinline__ typename cplx_of<T>::type cx(T x, T y) {
    typename cplx_of<T>::type r;
    r.x = x;
    r.y = y;
    return r;
}
template <typename T, typename C>
__device__ __forceinline__ C cmulT(C a, C b) {
    return cx<T>(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// Constant tables of the factored steps, built on the host in FP64, stored in the precision of
// the expansions.  Rows of 32: lane l of a warp reads column l.
template <typename T>
struct AConst {
    typedef typename cplx_of<T>::type C;
    T m2l[kTP][kTP];  // [k][l]: C(l+k-1, k-1) for l >= 1, 1 for l = 0
    T m2m[kTP][kTP];  // [j][k]: C(k-1, j-1) for 1 <= j <= k; [0][k] = 1/k
    T l2l[kTP][kTP];  // [k][l]: C(k, l) for l <= k
    C W[64][kTP];     // [cell][k]: w^k / k
    C V[kTP][64];     // [l][cell]: w^l
    C Z[4][kTP];      // [child quadrant][k]: zeta^k
    C ZI[4][kTP];     // [child quadrant][k]: (2 zeta)^-k
};

// Near-field leaf pair of a target leaf: the source leaf, how the levels relate (kind 0: the
// same level; kappa > 0: the source is kappa levels finer; kappa < 0: coarser; kDirect: summed
// directly) and the offsets of the pair's cells (see k_aleaf).
struct APair {
    int src, kind, ox, oy;
};
constexpr int kDirect = 64;
constexpr int kMaxKappa = 3;     // level differences served from the table
constexpr int kMaxOddSide = 192;  // its largest side

// ------------------------------------------------------------------------------------
// Upward pass, one warp per leaf: the leaf's multipole from the table of w^k / k (lane k
// forms M_k), then up the tree: the warp that arrives last at a parent (an arrival counter, cleared by
// k_am2l for the next solve; no warp waits) shifts the four children, whichever warp that is: the arithmetic and
// its order do not depend on it.  One launch in place of one per level: 0.24 ms (FP64) and 21 us
// (mixed) a level for 1629 boxes before, most of it latency and powers formed per lane.
// The children's zeta are 90 degree rotations of each other, zeta_q = i^m(q) zeta_3, so with
// G_r[j] = sum_q i^(m(q) r) M_j of child q the four shifts are one real product,
//   M_k = zeta_3^k [G_k[0] / k + sum_j C(k-1, j-1) (2 zeta_3)^-j G_(k-j)[j]]
// (indices of G mod 4, G[0] from the monopoles): 76 FP64 instructions a parent instead of 192.
// FP64 solves also write each leaf's weights in fixed point for the near field: v = q 2^(kNearBitsA - e)
// rounded, e the leaf's exponent (|q| < 2^e), kBadExp for a leaf with a non-finite weight.
// ------------------------------------------------------------------------------------
// Mixed solves copy theirs (q need not be aligned for the near field's 16-byte reads).
constexpr int kBadExp = INT_MAX;
constexpr int kNearBitsA = 56, kNearLogBitsA = 53;

template <typename T>
struct NearSrc {
    typedef T type;
};
template <>
struct NearSrc<double> {
    typedef long long type;
};

template <typename T>
__global__ void __launch_bounds__(128) k_aup(int nleaf, const int* __restrict__ leafbox,
                                             const int* __restrict__ parent, const int* __restrict__ first_child,
                                             const T* __restrict__ q, int p, const AConst<T>* __restrict__ ct,
                                             double* __restrict__ S, float2* __restrict__ Sf,
                                             typename cplx_of<T>::type* __restrict__ M, unsigned* __restrict__ cnt,
                                             typename NearSrc<T>::type* __restrict__ qfix, int* __restrict__ qexp) {
    typedef typename cplx_of<T>::type C;
    __shared__ T Rm[kTP][kTP];
    __shared__ C G[4][kTP][4];
    __shared__ T qs[4][64];
    const int w = threadIdx.x >> 5, k = threadIdx.x & 31;
    for (int i = threadIdx.x; i < kTP * kTP; i += 128) (&Rm[0][0])[i] = (&ct->m2m[0][0])[i];
    __syncthreads();
    const int leaf = blockIdx.x * 4 + w;
    if (leaf >= nleaf) return;  // warp-uniform; no block barrier follows
    const T q0 = q[int64_t(leaf) * 64 + k], q1 = q[int64_t(leaf) * 64 + 32 + k];
    qs[w][k] = q0;
    qs[w][k + 32] = q1;
    T s = q0 + q1;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    int b = leafbox[leaf];
    if constexpr (sizeof(T) == 8) {
        const bool bad = __any_sync(0xffffffffu, !(isfinite(q0) && isfinite(q1)));
        double m = fmax(fabs(q0), fabs(q1));
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        int e = -900;
        if (!bad && m > 0.0) e = max(ilogb(m) + 1, -900);
        const double f = __hiloint2double((1023 + kNearBitsA - (bad ? 0 : e)) << 20, 0);  // 2^(kNearBitsA - e)
        qfix[int64_t(leaf) * 64 + k] = bad ? 0 : __double2ll_rn(q0 * f);
        qfix[int64_t(leaf) * 64 + 32 + k] = bad ? 0 : __double2ll_rn(q1 * f);
        if (k == 0) qexp[leaf] = bad ? kBadExp : e;
    } else {
        qfix[int64_t(leaf) * 64 + k] = q0;
        qfix[int64_t(leaf) * 64 + 32 + k] = q1;
    }
    __syncwarp();
    C acc = cx<T>(T(0), T(0));
    if (k >= 1 && k <= p) {
#pragma unroll 8
        for (int c = 0; c < 64; ++c) {
            const C wk = ct->W[c][k];
            acc.x = fma(qs[w][c], wk.x, acc.x);
            acc.y = fma(qs[w][c], wk.y, acc.y);
        }
    }
    if (k <= p) M[int64_t(b) * kTP + k] = acc;
    if (k == 0) {
        S[b] = double(s);
        if (sizeof(T) == 4) Sf[b] = make_float2(float(s), 0.f);
    }
    const C zk = ct->Z[3][k], zik = ct->ZI[3][k];
    for (;;) {
        const int pa = parent[b];
        if (pa < 0) return;
        __threadfence();  // this warp's expansion before its arrival
        __syncwarp();
        unsigned arrived = 0;
        if (k == 0) arrived = atomicAdd(cnt + pa, 1u);
        if (__shfl_sync(0xffffffffu, arrived, 0) != 3u) return;
        __threadfence();  // the other children's after it
        b = pa;
        const int fc = first_child[b];
        C m[4];
        double sq[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            sq[c] = __ldcg(S + fc + c);
            m[c] = k >= 1 && k <= p ? __ldcg(M + int64_t(fc + c) * kTP + k) : cx<T>(T(0), T(0));
            if (k == 0) m[c] = cx<T>(T(sq[c]), T(0));
        }
        // i^m(q): m(3) = 0, m(2) = 1, m(0) = 2, m(1) = 3
        const C e = cx<T>(m[3].x + m[0].x, m[3].y + m[0].y), f = cx<T>(m[2].x + m[1].x, m[2].y + m[1].y);
        const C g = cx<T>(m[3].x - m[0].x, m[3].y - m[0].y), h = cx<T>(m[2].x - m[1].x, m[2].y - m[1].y);
        __syncwarp();  // the last level's reads of G are done
        G[w][k][0] = cmulT<T>(cx<T>(e.x + f.x, e.y + f.y), zik);
        G[w][k][1] = cmulT<T>(cx<T>(g.x - h.y, g.y + h.x), zik);
        G[w][k][2] = cmulT<T>(cx<T>(e.x - f.x, e.y - f.y), zik);
        G[w][k][3] = cmulT<T>(cx<T>(g.x + h.y, g.y - h.x), zik);
        __syncwarp();
        C y = cx<T>(T(0), T(0));
#pragma unroll 4
        for (int j = 0; j <= p; ++j) {
            const T r = Rm[j][k];
            const C v = G[w][j][(k - j) & 3];
            y.x = fma(r, v.x, y.x);
            y.y = fma(r, v.y, y.y);
        }
        const double ssum = sq[0] + sq[1] + sq[2] + sq[3];
        if (k >= 1 && k <= p) M[int64_t(b) * kTP + k] = cmulT<T>(y, zk);
        if (k == 0) {
            M[int64_t(b) * kTP] = cx<T>(T(0), T(0));
            S[b] = ssum;
            if (sizeof(T) == 4) Sf[b] = pp::df_from(ssum);
        }
    }
}

template <typename T>
struct OpLog {  // log|tau| of an operator: FP64, or a double-float pair
    typedef double type;
};
template <>
struct OpLog<float> {
    typedef float2 type;
};

// ------------------------------------------------------------------------------------
// M2L: one CTA of 64-thread units (two; mixed four) per target box, its entries dealt to the units in turn, as
// many entries at once as rows of p + 1 coefficients fit a unit (3 at p = 20, 4 at p = 12; one a
// warp left a third to a half of the lanes idle: 198 against 130 us at p = 20 in FP64, whose
// pipe bounds the kernel).  The diagonals (rho/tau)^k and tau^-l come from a table per distinct
// operator (a few hundred for the tens of thousands of pairs).  Thread k of an entry forms x_k
// in shared memory, thread l sums its row of the real product.  Mixed precision: the constant
// term S log|tau| and the sums of S in double-float.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void unit_sync(int unit) {  // literal barrier numbers: five reserved, not sixteen
    switch (unit) {
        case 0: asm volatile("bar.sync 1, 64;" ::: "memory"); break;
        case 1: asm volatile("bar.sync 2, 64;" ::: "memory"); break;
        case 2: asm volatile("bar.sync 3, 64;" ::: "memory"); break;
        default: asm volatile("bar.sync 4, 64;" ::: "memory"); break;
    }
}

// Units a target: the mixed kernel is bound by the latency of an entry's loads, so four.
template <typename T>
struct M2LUnits {
    static constexpr int value = sizeof(T) == 8 ? 2 : 4;
};

template <typename T>
__global__ void __launch_bounds__(64 * M2LUnits<T>::value) k_am2l(const int* __restrict__ ptr, const int2* __restrict__ pair,
                                              const AGeo* __restrict__ geo, const typename OpLog<T>::type* __restrict__ oplog,
                                              const typename cplx_of<T>::type* __restrict__ op, int p,
                                              const AConst<T>* __restrict__ ct, const double* __restrict__ S,
                                              const float2* __restrict__ Sf,
                                              const typename cplx_of<T>::type* __restrict__ M,
                                              typename cplx_of<T>::type* __restrict__ L, double* __restrict__ L0,
                                              unsigned* __restrict__ cnt) {
    typedef typename cplx_of<T>::type C;
    constexpr int kUnits = M2LUnits<T>::value, kThreads = 64 * kUnits;
    __shared__ T R[kTP][kTP];
    __shared__ C xs[kUnits][2][64];
    __shared__ C red[kThreads];
    __shared__ float4 red0[sizeof(T) == 4 ? kThreads : 1];  // mixed: constant term and sum of S, pairs
    const int a = blockIdx.x, tid = threadIdx.x, unit = tid >> 6;
    const int e0 = ptr[a], e1 = ptr[a + 1];
    if (tid == 0) cnt[a] = 0u;  // the upward pass's arrivals
    if (e0 == e1) {  // no sources (block-uniform)
        if (tid <= p) L[int64_t(a) * kTP + tid] = cx<T>(T(0), T(0));
        if (tid == 0) L0[a] = 0.0;
        return;
    }
    const int P1 = p + 1, slots = 64 / P1;              // entries a unit takes at once (2 at p = 30)
    const int slot = (tid & 63) / P1, t = (tid & 63) - slot * P1;  // slot == slots: an idle thread
    for (int i = tid; i < kTP * kTP; i += kThreads) (&R[0][0])[i] = (&ct->m2l[0][0])[i];
    __syncthreads();
    C acc = cx<T>(T(0), T(0));
    const double lns = -kLn2A * geo[a].level;  // log of the target's side
    const T cl = t == 0 ? T(0) : T(-1) / T(t);
    float ah = 0.f, al = 0.f, sh = 0.f, sl = 0.f;  // mixed: constant term, sum of S
    int buf = 0;
    int2 ahead = make_int2(0, 0);  // mixed: the pair of the next round, read a round early
    if (sizeof(T) == 4 && slot < slots && e0 + unit * slots + slot < e1) ahead = pair[e0 + unit * slots + slot];
    for (int base = e0 + unit * slots; base < e1; base += kUnits * slots, buf ^= 1) {  // uniform over the unit
        const int e = base + slot;
        const bool act = slot < slots && e < e1;
        C tl = cx<T>(T(0), T(0));
        const int2 pr = sizeof(T) == 4 ? ahead : act ? pair[e] : ahead;
        if (sizeof(T) == 4 && slot < slots && e + kUnits * slots < e1) ahead = pair[e + kUnits * slots];
        if (act) {
            const C* o = op + int64_t(pr.y) * (2 * kTP);
            tl = o[kTP + t];
            xs[unit][buf][tid & 63] = cmulT<T>(M[int64_t(pr.x) * kTP + t], o[t]);
        }
        unit_sync(unit);  // two buffers: one barrier an entry
        if (act) {
            const C* x = &xs[unit][buf][slot * P1];
            C y = cx<T>(T(0), T(0));
            if constexpr (sizeof(T) == 8) {
                y.x = S[pr.x] * (t == 0 ? oplog[pr.y] + lns : cl);
            } else {
                const float2 Sb = Sf[pr.x], lt = oplog[pr.y];
                y.x = Sb.x * cl;
                df_fma(ah, al, Sb.x, Sb.y, lt.x, lt.y);
                df_add(sh, sl, Sb.x, Sb.y);
            }
#pragma unroll 4
            for (int k = 1; k <= p; ++k) {
                const T r = R[k][t];
                const C v = x[k];
                y.x = fma(r, v.x, y.x);
                y.y = fma(r, v.y, y.y);
            }
            if constexpr (sizeof(T) == 4) df_add(ah, al, y.x, 0.f);  // thread 0: Re sum x_k
            acc.x = fma(tl.x, y.x, fma(-tl.y, y.y, acc.x));
            acc.y = fma(tl.x, y.y, fma(tl.y, y.x, acc.y));
        }
    }
    red[tid] = acc;
    if constexpr (sizeof(T) == 4) red0[tid] = make_float4(ah, al, sh, sl);
    __syncthreads();
    if (tid <= p) {
        C s = cx<T>(T(0), T(0));
        float rh = 0.f, rl = 0.f, qh = 0.f, ql = 0.f;
        for (int u = 0; u < kUnits; ++u)
            for (int i = 0; i < slots; ++i) {
                const C v = red[u * 64 + i * P1 + tid];
                s.x += v.x;
                s.y += v.y;
                if constexpr (sizeof(T) == 4) {
                    const float4 r = red0[u * 64 + i * P1];
                    df_add(rh, rl, r.x, r.y);
                    df_add(qh, ql, r.z, r.w);
                }
            }
        L[int64_t(a) * kTP + tid] = s;
        if (tid == 0) L0[a] = sizeof(T) == 4 ? df_to(rh, rl) + lns * df_to(qh, ql) : double(s.x);
    }
}

// ------------------------------------------------------------------------------------
// Leaves: one CTA per leaf.  All its warps but one sum the near field, the last shifts the locals down
// the leaf's path from the root (each leaf repeats its ancestors' shifts: no launch per level)
// and forms the constant terms; then one thread per cell evaluates the local expansion.
//
// Near field.  Cell centres of two leaves differ by integer multiples of half the finer cell's
// side, so log|x - x'| is log(unit) plus a table over integers.  Same level: offset m =
// ox + rx - tx in cells (source cell column rx, target column tx), table `te` of log|(mx, my)|,
// its [0][0] the self term c0.  Levels kappa apart: the offset is 2 m + 1 half cells of the finer
// side with m = ox + 2^kappa rx - tx (source coarser) or ox + rx - 2^kappa tx (source finer), table
// `to` over (|2 m_x + 1|, |2 m_y + 1|); the source's clamp never acts between different cells.
// log(unit) times the source leaf's S is added once per leaf (FP64).  Pairs beyond the table
// (kDirect) and, in FP64, leaves with non-finite weights are summed cell by cell.
// A thread owns one row of 8 target cells and one row of 8 source cells of its share of the pairs: its 64
// cell pairs need 15 (same level) or 22 (kappa 1) kernel values, kept in registers.  Before, each
// pair took its own table read, and pairs of different levels a square root and a logarithm.
//
// FP64 runs the cell pairs in fixed point on the integer pipe (pp_fixed.cuh), each product exact.  Source
// weights are 57-bit integers (relative to the largest exponent et of the target's sources), kernel
// values 57-bit integers (2^-53 units, |log| < 6.3); 16 source leaves a thread are summed before they
// are added to the FP64 sum.
// ------------------------------------------------------------------------------------
template <typename T>
struct NearAcc;

template <>
struct NearAcc<float> {
    typedef float Kv;  // kernel value
    float part[8], acc[8], comp[8];
    float q[8];
    __device__ void init() {
#pragma unroll
        for (int j = 0; j < 8; ++j) part[j] = acc[j] = comp[j] = 0.f;
    }
    __device__ void load(const float* src, int) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(src)), b = __ldg(reinterpret_cast<const float4*>(src) + 1);
        q[0] = a.x, q[1] = a.y, q[2] = a.z, q[3] = a.w, q[4] = b.x, q[5] = b.y, q[6] = b.z, q[7] = b.w;
    }
    __device__ __forceinline__ void add(int j, int r, float k) { part[j] = fmaf(q[r], k, part[j]); }
    __device__ void leaf_done(int, int) {  // Kahan sum of the leaves' partial sums
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float y = part[j] - comp[j];
            const float s = acc[j] + y;
            comp[j] = (s - acc[j]) - y;
            acc[j] = s;
            part[j] = 0.f;
        }
    }
    __device__ void finish(int) {}
    typedef float2 Out;  // a double-float pair
    __device__ __forceinline__ Out out(int j) const { return make_float2(acc[j], -comp[j]); }
    __device__ static __forceinline__ Out add(Out a, Out b) {
        df_add(a.x, a.y, b.x, b.y);
        return a;
    }
    __device__ static __forceinline__ Out shfl(Out a, int o) {
        return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
    }
    __device__ static __forceinline__ double value(Out a) { return df_to(a.x, a.y); }
};

template <>
struct NearAcc<double> {
    typedef int2 Kv;  // (high, low) halves
    pp::FixedSum sum[8];
    double acc[8];
    int2 q[8];
    __device__ void init() {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            sum[j].clear();
            acc[j] = 0.0;
        }
    }
    // the row's fixed-point weights, shifted right (rounded) to the common exponent
    __device__ void load(const long long* src, int sh) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const longlong2 v2 = __ldg(reinterpret_cast<const longlong2*>(src) + i);
            long long v[2] = {v2.x, v2.y};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (sh > 0) v[u] = sh > 60 ? 0 : (v[u] + (1ll << (sh - 1))) >> sh;
                q[2 * i + u] = pp::split28(v[u]);
            }
        }
    }
    __device__ __forceinline__ void add(int j, int r, int2 k) { sum[j].add(q[r], q[r].x + q[r].y, k, k.x + k.y); }
    // units: 2^(et - kNearBitsA - kNearLogBitsA)
    __device__ void drain(int et) {
        const double f1 = __hiloint2double((1023 + et + 56 - kNearBitsA - kNearLogBitsA) << 20, 0);
        const double f2 = f1 * 3.7252902984619140625e-09;  // 2^-28
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            long long hi;
            int lo;
            sum[j].digits(hi, lo);
            acc[j] = fma(double(hi), f1, fma(double(lo), f2, acc[j]));
            sum[j].clear();
        }
    }
    __device__ void leaf_done(int n, int et) {
        if ((n & 15) == 15) drain(et);  // 128 terms, |log| < 6.3: sum hh below 2^62.7, cross terms below 2^62.9
    }
    __device__ void finish(int et) { drain(et); }
    typedef double Out;
    __device__ __forceinline__ Out out(int j) const { return acc[j]; }
    __device__ static __forceinline__ Out add(Out a, Out b) { return a + b; }
    __device__ static __forceinline__ Out shfl(Out a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
    __device__ static __forceinline__ double value(Out a) { return a; }
};

// Mixed solves take the table's offsets in units of 2^same cells (2^odd half cells), so that its values are
// small and their FP32 sums do not cancel against log(unit) S (noise on cells of five sizes, p = 20, theta =
// 0.5: relative l2 error 2.7e-7, in cells 3.8e-7).
template <typename T>
struct NearUnit {
    static constexpr int same = sizeof(T) == 4 ? 3 : 0, odd = sizeof(T) == 4 ? 5 : 0;
};

// Pairs of near-field warps per CTA, and the path's warp: FP64 needs 128 registers a thread, and
// three CTAs of five warps fit an SM.
template <typename T>
struct LeafCta {
    static constexpr int groups = sizeof(T) == 8 ? 2 : 4;
    static constexpr int threads = 64 * groups + 32;
};

template <typename T>
__global__ void __launch_bounds__(LeafCta<T>::threads, 3)
k_aleaf(const int* __restrict__ leafbox, const int* __restrict__ anc, int nlev, const int* __restrict__ ptr,
        const APair* __restrict__ pairs, const AGeo* __restrict__ geo, int p, const AConst<T>* __restrict__ ct,
        const typename cplx_of<T>::type* __restrict__ L, const double* __restrict__ L0,
        const typename NearAcc<T>::Kv* __restrict__ te, int R, const typename NearAcc<T>::Kv* __restrict__ to, int Wo,
        const double* __restrict__ S, const T* __restrict__ q, const typename NearSrc<T>::type* __restrict__ qfix,
        const int* __restrict__ qexp, T* __restrict__ p_out) {
    typedef typename cplx_of<T>::type C;
    typedef typename NearAcc<T>::Kv Kv;
    extern __shared__ __align__(16) unsigned char smem_leaf[];
    Kv* tab = reinterpret_cast<Kv*>(smem_leaf);  // (R + 1) rows of stride R + 2
    constexpr int kGroups = LeafCta<T>::groups;
    __shared__ typename NearAcc<T>::Out near[kGroups][64];
    __shared__ C Ls[kTP];
    __shared__ double c0s;
    const int i = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int b = leafbox[i];
    const int e0 = ptr[i], e1 = ptr[i + 1];
    const int W = R + 2;
    for (int m = tid; m < (R + 1) * W; m += LeafCta<T>::threads) tab[m] = te[m];
    __syncthreads();
    if (warp < 2 * kGroups) {
        const int g = warp >> 1, sy = lane & 7, ty = (lane >> 3) + 4 * (warp & 1);
        int et = -900;
        if constexpr (sizeof(T) == 8) {  // the largest exponent of the target's sources
            for (int e = e0 + lane; e < e1; e += 32) {
                const int x = qexp[pairs[e].src];
                if (x != kBadExp) et = max(et, x);
            }
            et = __reduce_max_sync(0xffffffffu, et);
        }
        NearAcc<T> A;
        A.init();
        int n = 0;
        for (int e = e0 + g; e < e1; e += kGroups) {
            const APair pr = pairs[e];
            int sh = 0;
            bool direct = pr.kind == kDirect;
            if constexpr (sizeof(T) == 8) {
                const int x = qexp[pr.src];
                direct = direct || x == kBadExp;
                sh = et - x;
            }
            if (!direct) {
                A.load(qfix + int64_t(pr.src) * 64 + sy * 8, sh);
                if (pr.kind == 0) {
                    const Kv* kr = tab + abs(pr.oy + sy - ty) * W;
                    Kv kc[15];
#pragma unroll
                    for (int m = 0; m < 7; ++m) kc[m] = kr[abs(pr.ox - 7 + m)];
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        kc[r + 7] = kr[abs(pr.ox + r)];
#pragma unroll
                        for (int j = 0; j < 8; ++j) A.add(j, r, kc[r - j + 7]);
                    }
                } else {
                    const int kap = abs(pr.kind);
                    const int my = pr.kind < 0 ? pr.oy + (sy << kap) - ty : pr.oy + sy - (ty << kap);
                    const Kv* kr = to + (my ^ (my >> 31)) * Wo;
                    const auto kernel = [&](int m) { return __ldg(kr + (m ^ (m >> 31))); };
                    if (kap == 1 && pr.kind < 0) {  // source column r, target column j: kc[2 r - j + 7]
                        Kv kc[22];
#pragma unroll
                        for (int m = 0; m < 6; ++m) kc[m] = kernel(pr.ox - 7 + m);
#pragma unroll
                        for (int r = 0; r < 8; ++r) {
                            kc[2 * r + 6] = kernel(pr.ox - 1 + 2 * r);
                            kc[2 * r + 7] = kernel(pr.ox + 2 * r);
#pragma unroll
                            for (int j = 0; j < 8; ++j) A.add(j, r, kc[2 * r - j + 7]);
                        }
                    } else if (kap == 1) {  // kc[r - 2 j + 14]
                        if constexpr (sizeof(T) == 8) {  // even columns, then odd ones: half the values at once
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                Kv kc[11];
#pragma unroll
                                for (int m = 0; m < 7; ++m) kc[m] = kernel(pr.ox - 14 + u + 2 * m);
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    kc[i + 7] = kernel(pr.ox + u + 2 * i);
#pragma unroll
                                    for (int j = 0; j < 8; ++j) A.add(j, 2 * i + u, kc[i - j + 7]);
                                }
                            }
                        } else {
                            Kv kc[22];
#pragma unroll
                            for (int m = 0; m < 22; ++m) kc[m] = kernel(pr.ox - 14 + m);
#pragma unroll
                            for (int r = 0; r < 8; ++r)
#pragma unroll
                                for (int j = 0; j < 8; ++j) A.add(j, r, kc[r - 2 * j + 14]);
                        }
                    } else {
                        const int sr = pr.kind < 0 ? kap : 0, sj = pr.kind < 0 ? 0 : kap;
#pragma unroll
                        for (int r = 0; r < 8; ++r)
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const int m = pr.ox + (r << sr) - (j << sj);
                                A.add(j, r, __ldg(kr + (m ^ (m >> 31))));
                            }
                    }
                }
            } else if constexpr (sizeof(T) == 8) {
                const AGeo gt = geo[b], gs = geo[leafbox[pr.src]];
                const double rho = gs.s / 8.0 * exp(kC0A);
                const double yt = gt.cy + gt.s * ((ty + 0.5) / 8.0 - 0.5), ys = gs.cy + gs.s * ((sy + 0.5) / 8.0 - 0.5);
                for (int r = 0; r < 8; ++r) {
                    const double xs = gs.cx + gs.s * ((r + 0.5) / 8.0 - 0.5), qv = q[int64_t(pr.src) * 64 + sy * 8 + r];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const double dx = gt.cx + gt.s * ((j + 0.5) / 8.0 - 0.5) - xs, dy = yt - ys;
                        A.acc[j] += qv * log(fmax(sqrt(dx * dx + dy * dy), rho));
                    }
                }
            } else {
                // source cell centres relative to the target cell, in units of the target's cell side
                const AGeo gt = geo[b], gs = geo[leafbox[pr.src]];
                const double hc = gt.s / 8.0;
                const float ox = float((gs.cx - 0.5 * gs.s - (gt.cx - 0.5 * gt.s)) / hc) - 0.5f;
                const float oy = float((gs.cy - 0.5 * gs.s - (gt.cy - 0.5 * gt.s)) / hc) - (ty + 0.5f);
                const float step = float(gs.s / 8.0 / hc);      // source cell side / target cell side
                const float rho = step * 0.34604881609982794f;  // rho_h of the source cell: exp(pi/4 - 3/2 - ln2/2) h
                const float lhc = float(log(hc));
                const float dy = oy + (sy + 0.5f) * step;
                for (int r = 0; r < 8; ++r) {
                    const float qv = q[int64_t(pr.src) * 64 + sy * 8 + r];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float dx = ox + (r + 0.5f) * step - float(j);
                        A.part[j] = fmaf(qv, logf(fmaxf(sqrtf(dx * dx + dy * dy), rho)) + lhc, A.part[j]);
                    }
                }
            }
            A.leaf_done(n++, et);
        }
        A.finish(et);
        // the eight source rows are lanes of one target row: a lane ends with one target's sum
        typename NearAcc<T>::Out v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = A.out(j);
#pragma unroll
        for (int o = 4; o >= 1; o >>= 1)
#pragma unroll
            for (int j = 0; j < o; ++j) {
                const bool up = (sy & o) != 0;
                v[j] = NearAcc<T>::add(up ? v[j + o] : v[j], NearAcc<T>::shfl(up ? v[j] : v[j + o], o));
            }
        near[g][ty * 8 + sy] = v[0];
    } else {
        // the path's locals: cur is this lane's coefficient of the box above
        const int lev = geo[b].level;
        double c0 = 0.0;
        C cur = cx<T>(T(0), T(0));
        for (int l = 0; l <= lev; ++l) {
            const int bx = anc[int64_t(i) * nlev + l];
            const C m = lane <= p ? L[int64_t(bx) * kTP + lane] : cx<T>(T(0), T(0));
            const double m0 = L0[bx];
            if (l > 0) {
                const AGeo gb = geo[bx];
                const int qd = (gb.ix & 1) + 2 * (gb.iy & 1);
                __syncwarp();
                Ls[lane] = cmulT<T>(cur, ct->Z[qd][lane]);
                __syncwarp();
                C y = cx<T>(T(0), T(0));
#pragma unroll 4
                for (int k = 1; k <= p; ++k) {
                    const T r = ct->l2l[k][lane];
                    const C v = Ls[k];
                    y.x = fma(r, v.x, y.x);
                    y.y = fma(r, v.y, y.y);
                }
                c0 += double(y.x);  // lane 0: Re sum_k zeta^k L_k
                cur = cmulT<T>(y, ct->ZI[qd][lane]);
            }
            cur.x += m.x;
            cur.y += m.y;
            c0 += m0;
        }
        // log(unit) S over the near sources served from a table, unit = 2^-u: log 2 enters once, to more than
        // FP64's digits (the sums it multiplies cancel much of the table's)
        double sl = 0.0;
        for (int e = e0 + lane; e < e1; e += 32) {
            const APair pr = pairs[e];
            bool direct = pr.kind == kDirect;
            if constexpr (sizeof(T) == 8) direct = direct || qexp[pr.src] == kBadExp;
            const int unit = pr.kind == 0 ? lev + 3 - NearUnit<T>::same : lev + 4 + max(pr.kind, 0) - NearUnit<T>::odd;
            if (!direct) sl = fma(S[leafbox[pr.src]], double(unit), sl);
        }
        for (int o = 16; o > 0; o >>= 1) sl += __shfl_xor_sync(0xffffffffu, sl, o);
        __syncwarp();
        Ls[lane] = cur;
        if (lane == 0) c0s = fma(-kLn2A, sl, fma(-kLn2Lo, sl, c0));
    }
    __syncthreads();
    if (tid < 64) {
        T ser = T(0);
#pragma unroll 4
        for (int l = 1; l <= p; ++l) {
            const C v = ct->V[l][tid], m = Ls[l];
            ser = fma(m.x, v.x, fma(-m.y, v.y, ser));
        }
        typename NearAcc<T>::Out nr = NearAcc<T>::add(near[0][tid], near[1][tid]);
        if constexpr (kGroups == 4) nr = NearAcc<T>::add(nr, NearAcc<T>::add(near[2][tid], near[3][tid]));
        p_out[int64_t(i) * 64 + tid] = T((c0s + double(ser) + NearAcc<T>::value(nr)) * kInv2PiA);
    }
}

// Surface pressure at off-grid points by the tree-code over the adaptive tree (Sec. 2.3.1's
// targets; Appendix A.2's group acceptance), one warp per point: level by level from the root, a
// box is accepted for the point when its half-diagonal r is below theta d (d the distance from
// its centre) and its multipole is evaluated there, S log|w| - Re sum_k M_k (s / w)^k with w = z - c
// (Eq. pressTruncated about the box centre); a leaf that is not accepted is summed directly over
// its 64 cells, each clamped at its own rho_h; any other box opens its four children.  Accepted
// boxes are collected and evaluated 32 at a time, a lane each, so the FP64 pipe, which bounds
// the walk, works on full warps; logarithms come from the table method.  A level's open boxes lie
// within s / (sqrt 2 theta) of the point: at most 37 for theta >= 0.25, 148 children.
constexpr int kSurfCand = 256;

__global__ void __launch_bounds__(128) k_asurf(int npts, int nb, const double* __restrict__ pts, const AGeo* __restrict__ geo,
                                               const int* __restrict__ fchild, const int* __restrict__ boxleaf, int p,
                                               const double* __restrict__ S, const double2* __restrict__ M,
                                               const double* __restrict__ q, double theta, double* __restrict__ P_out,
                                               int* __restrict__ err) {
    __shared__ int cand[4][2][kSurfCand];
    __shared__ int acc_list[4][64];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * 4 + w;
    if (i >= npts) return;  // warp-uniform, no block barriers
    const double zx = pts[2 * i], zy = pts[2 * i + 1];
    const double th2 = theta * theta, rho8 = exp(kC0A) / 8.0;
    const unsigned below = (1u << lane) - 1u;
    double acc = 0.0;
    bool overflow = false;
    const auto evaluate = [&](int b) {  // an accepted box: u = s / w, Horner for sum_k M_k u^k
        const AGeo g = geo[b];
        const double dx = zx - g.cx, dy = zy - g.cy;
        const double d2 = dx * dx + dy * dy, sd = g.s / d2;
        const double2 u{dx * sd, -dy * sd};
        const double2* Mb = M + int64_t(b) * kTP;
        double2 h = Mb[p];
#pragma unroll 4
        for (int k = p - 1; k >= 1; --k) {
            const double2 m = Mb[k];
            h = double2{fma(h.x, u.x, fma(-h.y, u.y, m.x)), fma(h.x, u.y, fma(h.y, u.x, m.y))};
        }
        acc = fma(S[b], 0.5 * pp::log_table(d2), acc) - (h.x * u.x - h.y * u.y);
    };
    const auto direct = [&](int lb) {  // a leaf's 64 cells, two a lane
        const AGeo g = geo[lb];
        const double* qs = q + int64_t(boxleaf[lb]) * 64;
        const double rho = g.s * rho8, rho2 = rho * rho;
        const double2 c0 = cell_w(lane);
        const double ex = zx - fma(g.s, c0.x, g.cx), ey = zy - fma(g.s, c0.y, g.cy), ey1 = ey - 0.5 * g.s;
        const double x2 = ex * ex;  // cells `lane` and `lane + 32`, four rows on
        acc = fma(qs[lane], 0.5 * pp::log_table(fmax(fma(ey, ey, x2), rho2)), acc);
        acc = fma(qs[lane + 32], 0.5 * pp::log_table(fmax(fma(ey1, ey1, x2), rho2)), acc);
    };
    if (lane == 0) cand[w][0][0] = 0;
    __syncwarp();
    int cur = 0, n = 1, na = 0;
    if (isnan(zx) || isnan(zy)) {  // accepts no box and is within every clamp (fmax): every leaf, beyond what a list holds
        for (int b = 0; b < nb; ++b)
            if (fchild[b] < 0) direct(b);
        n = 0;
    }
    while (n > 0) {
        int next = 0;
        for (int base = 0; base < n; base += 32) {
            const bool act = base + lane < n;
            const int b = act ? cand[w][cur][base + lane] : 0;
            bool take = false, leaf = false, inner = false;
            int fc = -1;
            if (act) {
                const AGeo g = geo[b];
                const double dx = zx - g.cx, dy = zy - g.cy;
                take = 0.5 * g.s * g.s < th2 * (dx * dx + dy * dy);
                fc = fchild[b];
                leaf = !take && fc < 0;
                inner = !take && fc >= 0;
            }
            const unsigned tm = __ballot_sync(0xffffffffu, take);
            if (take) acc_list[w][na + __popc(tm & below)] = b;
            na += __popc(tm);
            __syncwarp();
            if (na >= 32) {
                evaluate(acc_list[w][lane]);
                na -= 32;
                const int v = acc_list[w][32 + lane];
                __syncwarp();
                acc_list[w][lane] = v;
                __syncwarp();
            }
            for (unsigned lm = __ballot_sync(0xffffffffu, leaf); lm; lm &= lm - 1)
                direct(__shfl_sync(0xffffffffu, b, __ffs(lm) - 1));
            const unsigned im = __ballot_sync(0xffffffffu, inner);
            if (inner) {
                const int at = next + 4 * __popc(im & below);
                if (at + 4 <= kSurfCand) {
#pragma unroll
                    for (int c = 0; c < 4; ++c) cand[w][cur ^ 1][at + c] = fc + c;
                } else {
                    overflow = true;
                }
            }
            next += 4 * __popc(im);
        }
        __syncwarp();
        cur ^= 1;
        n = min(next, kSurfCand);
    }
    if (lane < na) evaluate(acc_list[w][lane]);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) P_out[i] = acc * kInv2PiA;
    if (overflow) atomicExch(err, 1);
}

template <typename T>
cudaError_t upload(std::vector<void*>& bufs, T** dst, const std::vector<T>& src, cudaStream_t st) {
    const size_t bytes = sizeof(T) * (src.empty() ? 1 : src.size());
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(dst), bytes);
    if (e != cudaSuccess) return e;
    bufs.push_back(*dst);
    if (!src.empty()) e = cudaMemcpyAsync(*dst, src.data(), sizeof(T) * src.size(), cudaMemcpyHostToDevice, st);
    return e;
}

template <typename T>
cudaError_t dev_alloc(std::vector<void*>& bufs, T** dst, size_t n) {
    const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(dst), sizeof(T) * std::max<size_t>(n, 1));
    if (e == cudaSuccess) bufs.push_back(*dst);
    return e;
}

// Host arrays of one solve: box geometry, leaf -> box, each leaf's path, and both interaction
// lists as CSR by target.
struct AdaptivePrep {
    int nb = 0, nleaf = 0, L = 0, R = 0, Wo = 1;
    std::vector<AGeo> geo;
    std::vector<int> fchild, parent, leafbox, boxleaf, anc, m2l_ptr, p2p_ptr;
    std::vector<int2> m2l;     // source box, operator
    std::vector<APair> p2p;
    std::vector<double> op;    // tau_x, tau_y, rho per distinct operator
};

// Index of the operator (level difference, offset in units of the deepest box's half side) in a
// table that grows by insertion: open addressing over the integer key.
struct OpTable {
    struct Key {
        int64_t x, y;
        int dl;
    };
    std::vector<Key> keys;
    std::vector<int> slot;
    OpTable() : slot(1024, -1) {}
    static size_t hash(const Key& k) {
        uint64_t h = uint64_t(k.x) * 0x9E3779B97F4A7C15ull ^ uint64_t(k.y) * 0xC2B2AE3D27D4EB4Full ^
                     uint64_t(k.dl + 64) * 0x165667B19E3779F9ull;
        return size_t(h ^ (h >> 29));
    }
    int find(const Key& k, bool* fresh) {
        *fresh = false;
        for (size_t i = hash(k);; ++i) {
            int& s = slot[i & (slot.size() - 1)];
            if (s < 0) {
                *fresh = true;
                s = int(keys.size());
                keys.push_back(k);
                const int id = s;
                if (2 * keys.size() > slot.size()) grow();
                return id;
            }
            const Key& o = keys[s];
            if (o.x == k.x && o.y == k.y && o.dl == k.dl) return s;
        }
    }
    void grow() {
        slot.assign(2 * slot.size(), -1);
        for (size_t n = 0; n < keys.size(); ++n)
            for (size_t i = hash(keys[n]);; ++i) {
                int& s = slot[i & (slot.size() - 1)];
                if (s < 0) {
                    s = int(n);
                    break;
                }
            }
    }
};

int prepare_adaptive(pp_atree tree, AdaptivePrep& a) {
    int64_t sz[4];
    if (pp_atree_sizes(tree, sz) != PP_OK) return PP_ERR_ARG;
    const int nb = int(sz[0]), nm = int(sz[1]), np2 = int(sz[2]), L = int(sz[3]);
    try {
        std::vector<int> level(nb), ix(nb), iy(nb), leaf(nb), m2l(2 * size_t(nm)), p2p(2 * size_t(np2));
        a.parent.resize(nb);
        a.fchild.resize(nb);
        pp_atree_boxes(tree, level.data(), ix.data(), iy.data(), a.parent.data(), a.fchild.data(), leaf.data());
        pp_atree_lists(tree, m2l.data(), p2p.data());
        a.nb = nb;
        a.L = L;
        a.nleaf = 0;
        for (int b = 0; b < nb; ++b) a.nleaf += leaf[b] >= 0;
        a.geo.resize(nb);
        a.leafbox.assign(a.nleaf, -1);
        a.boxleaf = leaf;
        for (int b = 0; b < nb; ++b) {
            const double s = std::ldexp(1.0, -level[b]);
            a.geo[b] = AGeo{(ix[b] + 0.5) * s, (iy[b] + 0.5) * s, s, level[b], ix[b], iy[b]};
            if (leaf[b] >= 0) a.leafbox[leaf[b]] = b;
        }
        a.anc.assign(size_t(a.nleaf) * (L + 1), 0);
        for (int i = 0; i < a.nleaf; ++i)
            for (int b = a.leafbox[i]; b >= 0; b = a.parent[b]) a.anc[size_t(i) * (L + 1) + level[b]] = b;
        // translations: pairs are sorted by target; the operator depends on the level difference
        // and the offset in target sides
        a.m2l_ptr.assign(nb + 1, 0);
        a.m2l.resize(nm);
        OpTable ops;
        for (int e = 0; e < nm; ++e) {
            const int t = m2l[2 * e], s = m2l[2 * e + 1];
            ++a.m2l_ptr[t + 1];
            const int f = std::max(level[t], level[s]);
            const auto at = [&](int i, int l) { return (2 * int64_t(i) + 1) << (f - l); };
            const OpTable::Key k{at(ix[s], level[s]) - at(ix[t], level[t]), at(iy[s], level[s]) - at(iy[t], level[t]),
                                 level[s] - level[t]};
            bool fresh;
            const int id = ops.find(k, &fresh);
            if (fresh) {
                const double unit = std::ldexp(0.5, level[t] - f);  // half the finer side, in target sides
                a.op.push_back(double(k.x) * unit);
                a.op.push_back(double(k.y) * unit);
                a.op.push_back(std::ldexp(1.0, -k.dl));
            }
            a.m2l[e] = make_int2(s, id);
        }
        for (int b = 0; b < nb; ++b) a.m2l_ptr[b + 1] += a.m2l_ptr[b];
        // near-field pairs with their table offsets, and the sides of the two tables
        a.p2p_ptr.assign(a.nleaf + 1, 0);
        a.p2p.resize(np2);
        int dmax = 0, odd = -1;
        const auto fold = [](int64_t m) { return m >= 0 ? m : ~m; };
        for (int e = 0; e < np2; ++e) {
            ++a.p2p_ptr[p2p[2 * e] + 1];
            const AGeo &gt = a.geo[a.leafbox[p2p[2 * e]]], &gs = a.geo[a.leafbox[p2p[2 * e + 1]]];
            const int kind = gs.level - gt.level, k = std::abs(kind);
            APair pr{p2p[2 * e + 1], kind, 0, 0};
            if (kind == 0) {
                pr.ox = 8 * (gs.ix - gt.ix);
                pr.oy = 8 * (gs.iy - gt.iy);
                dmax = std::max(dmax, std::max(std::abs(gs.ix - gt.ix), std::abs(gs.iy - gt.iy)));
            } else if (k <= kMaxKappa) {
                const auto off = [&](int64_t is, int64_t it) {
                    return kind < 0 ? ((8 * is) << k) + (int64_t(1) << (k - 1)) - 1 - 8 * it
                                    : 8 * is - ((8 * it) << k) - (int64_t(1) << (k - 1));
                };
                const int64_t lo = kind < 0 ? 7 : 7 << k, hi = kind < 0 ? 7 << k : 7;
                const int64_t ox = off(gs.ix, gt.ix), oy = off(gs.iy, gt.iy);
                const int64_t big = std::max(std::max(fold(ox - lo), fold(ox + hi)), std::max(fold(oy - lo), fold(oy + hi)));
                if (big < kMaxOddSide) {
                    pr.ox = int(ox);
                    pr.oy = int(oy);
                    odd = std::max(odd, int(big));
                } else {
                    pr.kind = kDirect;
                }
            } else {
                pr.kind = kDirect;
            }
            a.p2p[e] = pr;
        }
        for (int i = 0; i < a.nleaf; ++i) a.p2p_ptr[i + 1] += a.p2p_ptr[i];
        a.R = 8 * dmax + 7;
        a.Wo = (odd + 1) | 1;
    } catch (const std::bad_alloc&) {
        return PP_ERR_OOM;
    }
    return PP_OK;
}

// What a tree keeps between solves: the prepared arrays on the device and, per precision (set up
// on its first solve), the constant tables, the operators' diagonals, the near-field tables and
// the expansions.
template <typename T>
struct AdaptiveSide {
    typedef typename cplx_of<T>::type C;
    bool ready = false;
    AConst<T>* ct = nullptr;
    C *op = nullptr, *M = nullptr, *L = nullptr;
    typename OpLog<T>::type* oplog = nullptr;
    typename NearAcc<T>::Kv *te = nullptr, *to = nullptr;
};

struct AdaptiveState {
    AdaptivePrep a;
    std::vector<void*> bufs;
    int *d_leafbox = nullptr, *d_fchild = nullptr, *d_parent = nullptr, *d_mptr = nullptr, *d_pptr = nullptr,
        *d_anc = nullptr, *d_boxleaf = nullptr, *d_err = nullptr, *d_qexp = nullptr;
    int2* d_mpair = nullptr;
    APair* d_ppair = nullptr;
    unsigned* d_cnt = nullptr;  // arrivals per box, zero when a solve starts
    AGeo* d_geo = nullptr;
    double *d_S = nullptr, *d_L0 = nullptr;
    float2* d_Sf = nullptr;
    long long* d_qfix = nullptr;
    AdaptiveSide<double> f64;
    AdaptiveSide<float> mixed;
    int last_p = 0;  // order of the last FP64 solve: the multipoles the surface tree-code reads
};

void release_state(void* v) {
    AdaptiveState* s = static_cast<AdaptiveState*>(v);
    for (void* b : s->bufs) cudaFree(b);
    delete s;
}

template <typename T>
AConst<T>* fill_const() {
    AConst<T>* c = new (std::nothrow) AConst<T>();
    if (!c) return nullptr;
    const auto put = [](typename cplx_of<T>::type& d, double2 z) {
        d.x = T(z.x);
        d.y = T(z.y);
    };
    const auto binom = [](int n, int r) {
        if (r < 0 || r > n) return 0.0;
        double v = 1.0;
        for (int i = 1; i <= r; ++i) v = v * double(n - r + i) / double(i);
        return v;
    };
    for (int k = 0; k < kTP; ++k)
        for (int l = 0; l < kTP; ++l) {
            c->m2l[k][l] = T(k < 1 ? 0.0 : l == 0 ? 1.0 : binom(l + k - 1, k - 1));
            c->m2m[k][l] = T(l < 1 ? 0.0 : k == 0 ? 1.0 / l : binom(l - 1, k - 1));
            c->l2l[k][l] = T(binom(k, l));
        }
    for (int n = 0; n < 64; ++n) {
        double2 w{1.0, 0.0};
        for (int k = 0; k < kTP; ++k) {
            put(c->V[k][n], w);
            put(c->W[n][k], k ? zscale(w, 1.0 / k) : double2{0.0, 0.0});
            w = zmul(w, cell_w(n));
        }
    }
    for (int n = 0; n < 4; ++n) {
        const double2 z{((n & 1) - 0.5) * 0.5, ((n >> 1) - 0.5) * 0.5};
        const double2 i2{z.x * 4.0, -z.y * 4.0};  // 1 / (2 zeta), |2 zeta|^2 = 1/2
        double2 a{1.0, 0.0}, b{1.0, 0.0};
        for (int k = 0; k < kTP; ++k) {
            put(c->Z[n][k], a);
            put(c->ZI[n][k], b);
            a = zmul(a, z);
            b = zmul(b, i2);
        }
    }
    return c;
}

void put_log(double& d, double v) { d = v; }
void put_log(float2& d, double v) { d = make_float2(float(v), float(v - double(float(v)))); }
void put_kernel(float& d, double v) { d = float(v); }
void put_kernel(int2& d, double v) { d = pp::split28(std::llrint(std::ldexp(v, kNearLogBitsA))); }

template <typename T>
cudaError_t setup_side(AdaptiveState* s, AdaptiveSide<T>& d, cudaStream_t st) {
    typedef typename cplx_of<T>::type C;
    const AdaptivePrep& a = s->a;
    const size_t nop = a.op.size() / 3;
    AConst<T>* hc = fill_const<T>();
    if (!hc) return cudaErrorMemoryAllocation;
    cudaError_t e;
    try {
        std::vector<C> op(nop * 2 * kTP);
        std::vector<typename OpLog<T>::type> lg(nop);
        for (size_t i = 0; i < nop; ++i) {
            const double tx = a.op[3 * i], ty = a.op[3 * i + 1], rho = a.op[3 * i + 2], r2 = tx * tx + ty * ty;
            put_log(lg[i], 0.5 * std::log(r2));
            const double2 ti{tx / r2, -ty / r2}, x{-rho * ti.x, -rho * ti.y};  // 1 / tau, -rho / tau
            double2 px{-1.0, 0.0}, pt{1.0, 0.0};                              // -(-rho / tau)^k, tau^-l
            for (int k = 0; k < kTP; ++k) {
                C& u = op[(2 * i) * kTP + k];
                C& v = op[(2 * i + 1) * kTP + k];
                u.x = T(px.x), u.y = T(px.y), v.x = T(pt.x), v.y = T(pt.y);
                px = zmul(px, x);
                pt = zmul(pt, ti);
            }
        }
        std::vector<typename NearAcc<T>::Kv> te(size_t(a.R + 1) * (a.R + 2)), to(size_t(a.Wo) * a.Wo);
        for (int y = 0; y <= a.R; ++y)
            for (int x = 0; x <= a.R; ++x)
                put_kernel(te[size_t(y) * (a.R + 2) + x],
                           (x + y == 0 ? kC0A : 0.5 * std::log(double(x * x + y * y))) - NearUnit<T>::same * kLn2A);
        for (int y = 0; y < a.Wo; ++y)
            for (int x = 0; x <= y; ++x) {
                const double v = 0.5 * std::log(double((2 * x + 1) * (2 * x + 1) + (2 * y + 1) * (2 * y + 1))) -
                                 NearUnit<T>::odd * kLn2A;
                put_kernel(to[size_t(y) * a.Wo + x], v);
                put_kernel(to[size_t(x) * a.Wo + y], v);
            }
        const size_t ne = size_t(a.nb) * kTP;
        if ((e = upload(s->bufs, &d.op, op, st)) || (e = upload(s->bufs, &d.oplog, lg, st)) ||
            (e = upload(s->bufs, &d.te, te, st)) || (e = upload(s->bufs, &d.to, to, st)) ||
            (e = dev_alloc(s->bufs, &d.ct, 1)) || (e = dev_alloc(s->bufs, &d.M, ne)) ||
            (e = dev_alloc(s->bufs, &d.L, ne)) ||
            (e = cudaMemcpyAsync(d.ct, hc, sizeof(AConst<T>), cudaMemcpyHostToDevice, st))) {
            delete hc;
            return e;
        }
        e = cudaStreamSynchronize(st);  // uploads done before the host arrays go
    } catch (const std::bad_alloc&) {
        e = cudaErrorMemoryAllocation;
    }
    delete hc;
    d.ready = e == cudaSuccess;
    return e;
}

cudaError_t setup_state(AdaptiveState* s, cudaStream_t st) {
    const AdaptivePrep& a = s->a;
    cudaError_t e;
    if ((e = upload(s->bufs, &s->d_leafbox, a.leafbox, st)) || (e = upload(s->bufs, &s->d_fchild, a.fchild, st)) ||
        (e = upload(s->bufs, &s->d_parent, a.parent, st)) || (e = upload(s->bufs, &s->d_mptr, a.m2l_ptr, st)) ||
        (e = upload(s->bufs, &s->d_mpair, a.m2l, st)) || (e = upload(s->bufs, &s->d_pptr, a.p2p_ptr, st)) ||
        (e = upload(s->bufs, &s->d_ppair, a.p2p, st)) || (e = upload(s->bufs, &s->d_geo, a.geo, st)) ||
        (e = upload(s->bufs, &s->d_anc, a.anc, st)) || (e = upload(s->bufs, &s->d_boxleaf, a.boxleaf, st)) ||
        (e = dev_alloc(s->bufs, &s->d_err, 1)) || (e = dev_alloc(s->bufs, &s->d_S, a.nb)) ||
        (e = dev_alloc(s->bufs, &s->d_L0, a.nb)) || (e = dev_alloc(s->bufs, &s->d_Sf, a.nb)) ||
        (e = dev_alloc(s->bufs, &s->d_cnt, a.nb)) || (e = dev_alloc(s->bufs, &s->d_qexp, a.nleaf)) ||
        (e = dev_alloc(s->bufs, &s->d_qfix, size_t(a.nleaf) * 64)))
        return e;
    return cudaMemsetAsync(s->d_cnt, 0, sizeof(unsigned) * a.nb, st);
}

// The tree's state and one precision's side of it, made on first use.
template <typename T>
int ensure_side(pp_atree tree, AdaptiveSide<T> AdaptiveState::* side, cudaStream_t st, AdaptiveState** out) {
    AdaptiveState* s = static_cast<AdaptiveState*>(pp::atree_state(tree));
    if (!s) {
        s = new (std::nothrow) AdaptiveState();
        if (!s) return PP_ERR_OOM;
        const int pst = prepare_adaptive(tree, s->a);
        cudaError_t e = pst == PP_OK ? setup_state(s, st) : cudaSuccess;
        if (pst == PP_OK && e == cudaSuccess) e = cudaStreamSynchronize(st);  // uploads done before reuse
        if (pst != PP_OK || e != cudaSuccess) {
            release_state(s);
            cudaGetLastError();
            return pst != PP_OK ? pst : e == cudaErrorMemoryAllocation ? PP_ERR_OOM : PP_ERR_CUDA;
        }
        pp::atree_set_state(tree, s, release_state);
    }
    if (!(s->*side).ready) {
        const cudaError_t e = setup_side<T>(s, s->*side, st);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return e == cudaErrorMemoryAllocation ? PP_ERR_OOM : PP_ERR_CUDA;
        }
    }
    *out = s;
    return PP_OK;
}

template <typename T>
int solve_adaptive(AdaptiveState* s, const AdaptiveSide<T>& d, int p, const T* q, T* p_out, cudaStream_t st) {
    const AdaptivePrep& a = s->a;
    typename NearSrc<T>::type* qs = reinterpret_cast<typename NearSrc<T>::type*>(s->d_qfix);
    k_aup<T><<<(a.nleaf + 3) / 4, 128, 0, st>>>(a.nleaf, s->d_leafbox, s->d_parent, s->d_fchild, q, p, d.ct, s->d_S,
                                               s->d_Sf, d.M, s->d_cnt, qs, s->d_qexp);
    k_am2l<T><<<a.nb, 64 * M2LUnits<T>::value, 0, st>>>(s->d_mptr, s->d_mpair, s->d_geo, d.oplog, d.op, p, d.ct, s->d_S, s->d_Sf, d.M,
                                    d.L, s->d_L0, s->d_cnt);
    const size_t smem = sizeof(typename NearAcc<T>::Kv) * size_t(a.R + 1) * (a.R + 2);
    k_aleaf<T><<<a.nleaf, LeafCta<T>::threads, smem, st>>>(s->d_leafbox, s->d_anc, a.L + 1, s->d_pptr, s->d_ppair, s->d_geo,
                                                    p, d.ct, d.L, s->d_L0, d.te, a.R, d.to, a.Wo, s->d_S, q,
                                                    qs, s->d_qexp, p_out);
    return cudaGetLastError() == cudaSuccess ? PP_OK : PP_ERR_CUDA;
}

}  // namespace

extern "C" int pp_atree_solve(pp_atree tree, int order, const double* q, double* p_out, void* stream) {
    if (!tree || !q || !p_out || order < 2 || order > kMaxOrderA) return PP_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    AdaptiveState* s = nullptr;
    int r = ensure_side<double>(tree, &AdaptiveState::f64, st, &s);
    if (r == PP_OK) r = solve_adaptive<double>(s, s->f64, order, q, p_out, st);
    if (r == PP_OK) s->last_p = order;
    return r;
}

extern "C" int pp_atree_solve_mixed(pp_atree tree, int order, const float* q, float* p_out, void* stream) {
    if (!tree || !q || !p_out || order < 2 || order > kMaxOrderA) return PP_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    AdaptiveState* s = nullptr;
    int r = ensure_side<float>(tree, &AdaptiveState::mixed, st, &s);
    if (r == PP_OK) r = solve_adaptive<float>(s, s->mixed, order, q, p_out, st);
    if (r == PP_OK) s->last_p = 0;  // S is the mixed solve's now: the surface tree-code needs an FP64 solve
    return r;
}

extern "C" int pp_atree_surface_pressure(pp_atree tree, const double* q, int npts, const double* points, double theta,
                                         double* P_out, void* stream) {
    if (!tree || !q || !points || !P_out || npts < 1 || npts > (1 << 24) || !(theta >= 0.25 && theta <= 0.95))
        return PP_ERR_ARG;
    AdaptiveState* s = static_cast<AdaptiveState*>(pp::atree_state(tree));
    if (!s || s->last_p < 1) return PP_ERR_STATE;  // the multipoles come from a solve
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaMemsetAsync(s->d_err, 0, sizeof(int), st) != cudaSuccess) return PP_ERR_CUDA;
    k_asurf<<<(npts + 3) / 4, 128, 0, st>>>(npts, s->a.nb, points, s->d_geo, s->d_fchild, s->d_boxleaf, s->last_p, s->d_S,
                                               s->f64.M, q, theta, P_out, s->d_err);
    if (cudaGetLastError() != cudaSuccess) return PP_ERR_CUDA;
    int err = 0;
    if (cudaMemcpyAsync(&err, s->d_err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return PP_ERR_CUDA;
    return err ? PP_ERR_STATE : PP_OK;
}
