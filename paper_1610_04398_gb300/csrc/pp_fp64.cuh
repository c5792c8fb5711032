// The FP64 path's kernels (orders up to 23, leaf level >= 2; other orders keep the generic
// kernels).  GB300's FP64 pipe issues 1.67 lanes a clock and SM (one warp instruction in about 19
// cycles), so the design counts FP64 instructions: the two long sums, the near field and the
// multipole-to-local translations, run in fixed point on the integer pipe (pp_fixed.cuh), and
// the remaining steps use the symmetry of their geometry to share products:
//   source: constant factors of the stencils folded into the last three multiply-adds;
//   leaf multipoles and evaluation: the 64 cells of a leaf are six orbits of eight and four of
//     four under the square's symmetries, and powers of an orbit's cells differ by i^k and
//     conjugation only: 3 multiply-adds a coefficient and orbit in place of 2 or 4 per cell;
//   shifts: the four children of a box sit at 90 degree rotations, so one real product serves
//     all four children in place of four.
// Times at the kernels: one GB300, 1024^2, p = 20, theta = 0.5.
#pragma once

#include <vector>

#include "pp_fixed.cuh"
#include "pp_kernels.cuh"

namespace pp {
namespace f64 {

constexpr int kMaxP = 24;  // coefficients

static __device__ const RealOps<double> g_ops = RealOps<double>();

// Level exponents of the multipoles (|M_k| 2^floor(k/2) < 2^e over a level's boxes), then the
// arrival counters of the upward pass, in the plan's counter array.
__device__ __forceinline__ int* level_exp(const Tree<double>& t) { return reinterpret_cast<int*>(t.up_counter); }
__device__ __forceinline__ unsigned* arrivals(const Tree<double>& t) { return t.up_counter + 32; }

__device__ __forceinline__ int coef_exp(double2 m, int k) {
    const int e = exp_of(max(__double2hiint(m.x) & 0x7fffffff, __double2hiint(m.y) & 0x7fffffff));
    return e == kExpBad || e == kExpZero ? e : e + (k >> 1);
}

// ------------------------------------------------------------------------------------
// (a1) Source, one warp per strip of 32 columns and kSrcRows rows (fewer on small grids), marching down with the rows above,
// at and below in registers; x neighbours by shuffles (the strip's outer columns read by lanes
// 0 and 31).  About 21 FP64 instructions a cell, which bound it (42 us at 1024^2 at the pipe's
// rate; 129 us before, 72 now).  Also clears the level exponents.
// ------------------------------------------------------------------------------------
template <int kSrcRows>
__global__ void __launch_bounds__(128) k_rhs64(Tree<double> t, const double* __restrict__ u, const double* __restrict__ v,
                                               const double* __restrict__ chi, const double* __restrict__ usx,
                                               const double* __restrict__ usy, double rho, double lam,
                                               double* __restrict__ f_out) {
    if (blockIdx.x == 0 && threadIdx.x < 32) level_exp(t)[threadIdx.x] = kExpZero;
    if (blockIdx.x == 0 && threadIdx.x == 0) *t.surf_counter = 0u;
    const int n = t.n, lane = threadIdx.x & 31;
    const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int strips = n >> 5;
    const int x = int(w % strips) * 32 + lane, y0 = int(w / strips) * kSrcRows;
    if (y0 >= n) return;  // warp-uniform
    const int xe = lane == 0 ? x - 1 : x + 1;  // the outer column of lanes 0 and 31
    const bool edge_lane = (lane == 0 && x > 0) || (lane == 31 && x < n - 1);
    const bool edge_strip = __any_sync(0xffffffffu, x == 0 || x == n - 1);
    const double inv2h = 0.5 / t.h, hh = t.h * t.h;
    const double c1 = -rho * inv2h * inv2h, c2 = 2.0 * c1, c3 = rho * lam * inv2h;
    // rows y - 1, y, y + 1: u, v, b = chi (us_y - v); of row y also a = chi (us_x - u) and the outer
    // column's u, v, a
    double um = 0.0, vm = 0.0, bm = 0.0, uc = 0.0, vc = 0.0, bc = 0.0, ac = 0.0, eu = 0.0, ev = 0.0, ea = 0.0;
    const auto load3 = [&](int y, double& a, double& b, double& c) {
        const int64_t g = int64_t(y) * n + x;
        a = u[g];
        b = v[g];
        c = chi[g] * (usy[g] - b);
    };
    const auto load_row = [&](int y, double& a, double& b, double& cb, double& ca, double& oa, double& ob, double& oc) {
        const int64_t g = int64_t(y) * n + x;
        const double c = chi[g];
        a = u[g];
        b = v[g];
        ca = c * (usx[g] - a);
        cb = c * (usy[g] - b);
        if (edge_lane) {
            const int64_t o = int64_t(y) * n + xe;
            oa = u[o];
            ob = v[o];
            oc = chi[o] * (usx[o] - oa);
        }
    };
    if (y0 > 0) load3(y0 - 1, um, vm, bm);
    load_row(y0, uc, vc, bc, ac, eu, ev, ea);
    const auto ddx = [&](double e, double outer) {  // 2h d/dx
        double l = __shfl_up_sync(0xffffffffu, e, 1), r = __shfl_down_sync(0xffffffffu, e, 1);
        if (lane == 0) l = outer;
        if (lane == 31) r = outer;
        double d = r - l;
        if (edge_strip) {
            const double l2 = __shfl_up_sync(0xffffffffu, e, 2), r2 = __shfl_down_sync(0xffffffffu, e, 2);
            if (x == 0) d = -3.0 * e + 4.0 * r - r2;
            if (x == n - 1) d = 3.0 * e - 4.0 * l + l2;
        }
        return d;
    };
#pragma unroll 2
    for (int y = y0; y < y0 + kSrcRows; ++y) {
        double un = 0.0, vn = 0.0, bn = 0.0, an = 0.0, nu = 0.0, nv = 0.0, na = 0.0;
        if (y + 1 < n) load_row(y + 1, un, vn, bn, an, nu, nv, na);
        const double dux = ddx(uc, eu), dvx = ddx(vc, ev), dax = ddx(ac, ea);
        double duy = un - um, dvy = vn - vm, dby = bn - bm;
        if (y == 0 || y == n - 1) {  // one-sided: the third row from memory
            double u3, v3, b3;
            load3(y == 0 ? 2 : n - 3, u3, v3, b3);
            if (y == 0) {
                duy = -3.0 * uc + 4.0 * un - u3;
                dvy = -3.0 * vc + 4.0 * vn - v3;
                dby = -3.0 * bc + 4.0 * bn - b3;
            } else {
                duy = 3.0 * uc - 4.0 * um + u3;
                dvy = 3.0 * vc - 4.0 * vm + v3;
                dby = 3.0 * bc - 4.0 * bm + b3;
            }
        }
        const double f = fma(c3, dax + dby, fma(c2, duy * dvx, c1 * fma(dvy, dvy, dux * dux)));
        if (f_out) f_out[int64_t(y) * n + x] = f;
        t.q[(int64_t(y >> 3) * t.nL + (x >> 3)) * 64 + (y & 7) * 8 + (x & 7)] = f * hh;
        um = uc, vm = vc, bm = bc;
        uc = un, vc = vn, bc = bn, ac = an, eu = nu, ev = nv, ea = na;
    }
}

// ------------------------------------------------------------------------------------
// Leaf multipoles.  One CTA per 32 leaves, lane = leaf, warp r forms the coefficients k = r mod 4.
// Orbit of w = (a + i b) / 8 (a >= b): with q_m at i^m w and q'_m at i^m conj(w),
//   M_k k = w^k Q_r + conj(w)^k Q'_r,  Q_0 = q0+q1+q2+q3, Q_2 = q0-q1+q2-q3,
//   Q_1 = (q0-q2) + i (q1-q3), Q_3 = conj Q_1.
// 832 FP64 instructions for the 64 cells and 20 coefficients in place of 2560 and more: 384 us
// before at 1024^2, 46 now.
// ------------------------------------------------------------------------------------
__host__ __device__ constexpr int cell_at(int x2, int y2) { return ((y2 + 7) >> 1) * 8 + ((x2 + 7) >> 1); }  // (x2, y2) / 2

// Representative (a, b) of orbit `orb`: (1,1), (3,1), (3,3), (5,1), ... (7,7).
__device__ __forceinline__ int2 orbit_of(int orb) {
    int a = 1, b = orb;
    while (b > (a - 1) / 2) b -= (a + 1) / 2, a += 2;
    return make_int2(a, 2 * b + 1);
}
// The rows of a cell table (64 x P1) at the ten representatives.
__device__ __forceinline__ void stage_orbits(double2* dst, const double2* __restrict__ tab, int P1) {
    for (int i = threadIdx.x; i < 10 * P1; i += blockDim.x) {
        const int2 o = orbit_of(i / P1);
        dst[i] = tab[cell_at(o.x, o.y) * P1 + i % P1];
    }
}

template <int R, int KN>
__device__ __forceinline__ void p2m_class(const double* qs, const double2* W, int P1,
                                          double2 (&M)[KN], double& S) {
#pragma unroll
    for (int i = 0; i < KN; ++i) M[i] = double2{0.0, 0.0};
    S = 0.0;
#pragma unroll 1
    for (int a = 1; a <= 7; a += 2) {
        double Sa = 0.0;  // the sum in blocks: fewer roundings at its full size
#pragma unroll 1
        for (int b = 1; b <= a; b += 2, W += P1) {
            const double q0 = qs[cell_at(a, b)], q1 = qs[cell_at(-b, a)], q2 = qs[cell_at(-a, -b)], q3 = qs[cell_at(b, -a)];
            double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;
            if (a != b) p0 = qs[cell_at(a, -b)], p1 = qs[cell_at(b, a)], p2 = qs[cell_at(-a, b)], p3 = qs[cell_at(-b, -a)];
            const double2* w = W;  // w^k / k (entry 0: 1)
            if (R == 0 || R == 2) {
                const double s = R == 0 ? 1.0 : -1.0;
                const double Q = (q0 + q2) + s * (q1 + q3), P = (p0 + p2) + s * (p1 + p3);
                const double A = Q + P, B = Q - P;
#pragma unroll
                for (int i = 0; i < KN; ++i) {
                    const int k = 4 * i + R;
                    if (k == 0) {
                        Sa += A;
                    } else if (k < P1) {
                        const double2 z = w[k];
                        M[i].x = fma(A, z.x, M[i].x);
                        M[i].y = fma(B, z.y, M[i].y);
                    }
                }
            } else {
                const double s = R == 1 ? 1.0 : -1.0;
                const double X = q0 - q2, Y = s * (q1 - q3), Xp = p0 - p2, Yp = s * (p1 - p3);
                const double xs = X + Xp, xd = X - Xp, ys = Y + Yp, yd = Y - Yp;
#pragma unroll
                for (int i = 0; i < KN; ++i) {
                    const int k = 4 * i + R;
                    if (k < P1) {
                        const double2 z = w[k];
                        M[i].x = fma(xs, z.x, fma(-yd, z.y, M[i].x));
                        M[i].y = fma(ys, z.x, fma(xd, z.y, M[i].y));
                    }
                }
            }
        }
        S += Sa;
    }
}

template <int R, int KN>
__device__ __forceinline__ int p2m_store(const Tree<double>& t, const double* qs, const double2* W, int64_t box,
                                         bool act) {
    double2 M[KN];
    double S;
    p2m_class<R, KN>(qs, W, t.P1, M, S);
    int e = kExpZero;
#pragma unroll
    for (int i = 0; i < KN; ++i) {
        const int k = 4 * i + R;
        if (k >= t.P1) continue;
        const double2 m = k == 0 ? double2{S, 0.0} : M[i];
        if (act) t.mp[box * t.P1 + k] = m;
        e = max(e, coef_exp(m, k));
    }
    if (R == 0 && act) t.S[box] = S;
    return act ? e : kExpZero;
}

template <int KN>
__global__ void __launch_bounds__(128) k_p2m64(Tree<double> t) {
    __shared__ double qs[32 * 65];  // stride 65: lanes (leaves) on distinct banks
    __shared__ double2 Ws[10 * kMaxP];
    const int64_t leaf0 = int64_t(blockIdx.x) * 32, nleaf = int64_t(t.nL) * t.nL;
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5;
    const int64_t box0 = int64_t(blockIdx.x) * 128 + threadIdx.x;  // four threads a leaf: one a box above
    if (box0 < level_offset(t.Lleaf - 1)) arrivals(t)[box0] = 0u;
    for (int i = threadIdx.x; i < 32 * 64; i += 128)
        qs[(i >> 6) * 65 + (i & 63)] = leaf0 + (i >> 6) < nleaf ? t.q[leaf0 * 64 + i] : 0.0;
    stage_orbits(Ws, t.Wp2m, t.P1);
    __syncthreads();
    const bool act = leaf0 + lane < nleaf;
    const int64_t box = level_offset(t.Lleaf) + leaf0 + lane;
    const double* q = qs + lane * 65;
    int e;
    switch (r) {
        case 0: e = p2m_store<0, KN>(t, q, Ws, box, act); break;
        case 1: e = p2m_store<1, KN>(t, q, Ws, box, act); break;
        case 2: e = p2m_store<2, KN>(t, q, Ws, box, act); break;
        default: e = p2m_store<3, KN>(t, q, Ws, box, act); break;
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) atomicMax(level_exp(t) + t.Lleaf, e);
}

// ------------------------------------------------------------------------------------
// Upward pass in one launch: a warp per box of level L - 1 shifts its four leaves' multipoles;
// the warp that arrives last at a parent (arrival counters, cleared by k_p2m64; no warp waits) goes on
// with it.  With zeta_q = i^m(q) zeta_3 the four shifts are one real product over
// G_r[j] = sum_q i^(m(q) r) M_j (child q), lane k forming coefficient k:
//   M_k = zeta_3^k [G_k[0] / k + sum_j C(k-1, j-1) (2 zeta_3)^-j G_(k-j)[j]].
// 235 us in four launches before at 1024^2 (the top four levels, in one CTA, 135 of them), 64 now.
// ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) k_up64(Tree<double> t) {
    __shared__ double Rm[kMaxP][kMaxP];  // [j][k]
    __shared__ double2 G[4][kMaxP][4];
    const int w = threadIdx.x >> 5, k = threadIdx.x & 31, P1 = t.P1;
    for (int i = threadIdx.x; i < P1 * P1; i += 128) Rm[i / P1][i % P1] = g_ops.m2m[i % P1][i / P1];
    __syncthreads();
    int l = t.Lleaf - 1;
    int64_t b = int64_t(blockIdx.x) * 4 + w;
    if (b >= (int64_t(1) << (2 * l))) return;  // warp-uniform; no block barrier follows
    const int kc = k < P1 ? k : 0;
    const double2 zk = t.Zq[3 * P1 + kc], zik = t.Ziq[3 * P1 + kc];
    for (;;) {
        const int side = 1 << l, bx = int(b & (side - 1)), by = int(b >> l);
        const int64_t child = level_offset(l + 1) + int64_t(2 * by) * (2 * side) + 2 * bx;
        double2 m[4];
        double sq[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t c = child + int64_t(q >> 1) * (2 * side) + (q & 1);
            sq[q] = __ldcg(t.S + c);
            m[q] = k < P1 ? __ldcg(t.mp + c * P1 + k) : double2{0.0, 0.0};  // entry 0: (S, 0)
        }
        // i^m(q): m(3) = 0, m(2) = 1, m(0) = 2, m(1) = 3
        const double2 e{m[3].x + m[0].x, m[3].y + m[0].y}, f{m[2].x + m[1].x, m[2].y + m[1].y};
        const double2 g{m[3].x - m[0].x, m[3].y - m[0].y}, h{m[2].x - m[1].x, m[2].y - m[1].y};
        const auto mul = [](double2 a, double2 c) {
            return double2{fma(a.x, c.x, -a.y * c.y), fma(a.x, c.y, a.y * c.x)};
        };
        __syncwarp();  // the last level's reads of G are done
        if (k < P1) {
            G[w][k][0] = mul(double2{e.x + f.x, e.y + f.y}, zik);
            G[w][k][1] = mul(double2{g.x - h.y, g.y + h.x}, zik);
            G[w][k][2] = mul(double2{e.x - f.x, e.y - f.y}, zik);
            G[w][k][3] = mul(double2{g.x + h.y, g.y - h.x}, zik);
        }
        __syncwarp();
        double2 y{0.0, 0.0}, y1{0.0, 0.0};
#pragma unroll 4
        for (int j = 0; j < P1; j += 2) {  // two chains
            const double r = Rm[j][kc];
            const double2 v = G[w][j][(k - j) & 3];
            y.x = fma(r, v.x, y.x);
            y.y = fma(r, v.y, y.y);
            if (j + 1 < P1) {
                const double r1 = Rm[j + 1][kc];
                const double2 v1 = G[w][j + 1][(k - j - 1) & 3];
                y1.x = fma(r1, v1.x, y1.x);
                y1.y = fma(r1, v1.y, y1.y);
            }
        }
        y.x += y1.x;
        y.y += y1.y;
        const double S = sq[0] + sq[1] + sq[2] + sq[3];
        const double2 M = k == 0 ? double2{S, 0.0} : mul(y, zk);
        const int64_t box = level_offset(l) + b;
        if (k < P1) t.mp[box * P1 + k] = M;
        if (k == 0) t.S[box] = S;
        const int ex = __reduce_max_sync(0xffffffffu, k < P1 ? coef_exp(M, k) : kExpZero);
        if (k == 0) atomicMax(level_exp(t) + l, ex);
        if (l == 0) return;
        const int64_t pa = int64_t(by >> 1) * (side >> 1) + (bx >> 1);
        unsigned* cnt = arrivals(t) + level_offset(l - 1) + pa;
        __threadfence();  // this warp's expansion before its arrival
        __syncwarp();
        unsigned arrived = 0;
        if (k == 0) arrived = atomicAdd(cnt, 1u);
        if (__shfl_sync(0xffffffffu, arrived, 0) != 3u) return;
        __threadfence();  // the other children's after it
        b = pa;
        --l;
    }
}

// ------------------------------------------------------------------------------------
// Near field in fixed point.  One CTA of 256 threads per 2 x 2 leaves: the source weights of the
// (2 + 2D)^2 leaves around them, 55 or 56 bits relative to their largest exponent (what FP64 holds of
// weights within two or three bits of it), and a quadrant of the kernel table log(h max(|(mx, my)|, rho_h /
// h)) (2^-52 or 2^-53 units; h clamped to e^-11 .. e^11, what is left of log h entering through the near
// leaves' monopoles in k_down64) sit in shared memory.  A thread owns a row of 8 target cells and one
// source row of every near leaf: 15 kernel values and 8 weights for 64 cell pairs, an exact product each
// (FixedSum).  The eight source rows (lanes of a target row) are added in integers, one lane a target.
// Before, with 53 bits, the products' low digits dropped and all of log h in the monopoles, whose product
// cancels most of the table's sum, the near field's error was 1.5 to 20 times that of FP64
// multiply-adds; now 0.4 to 1.1 times (64^2, p = 20, theta = 0.5: relative l2 of the field 3.5 and 6.0e-16).
// Bound by the integer multiply-adds: 1600 pairs a cell at theta = 0.5, 570 us at 1024^2 at the
// measured rate; 2818 us on the FP64 pipe (evaluation included), 713 with the low digits dropped, 770 now.
// ------------------------------------------------------------------------------------
constexpr double kNearLn = 11.0;  // |log h| in the table: with log 66 below 16
constexpr int kNearRow = 10;  // int2 per source row (8 used): rows on distinct banks

__host__ __device__ constexpr int near64_halo(int D) { return (2 + 2 * D) * (2 + 2 * D); }
inline size_t near64_smem(int D) {
    const int R = 8 * D + 7;
    return sizeof(int2) * (size_t(near64_halo(D)) * 8 * kNearRow + size_t(R + 1) * (R + 2));
}

__global__ void __launch_bounds__(256, 2) k_near64(Tree<double> t, double* __restrict__ p_out) {
    extern __shared__ __align__(16) int2 sm64[];
    __shared__ int wexp[8];
    const int D = t.Dmax, H = 2 + 2 * D, R = t.Rk, W = R + 2, nL = t.nL;
    int2* qs = sm64;                         // [halo leaf][row][kNearRow]
    int2* tab = qs + H * H * 8 * kNearRow;   // [|my|][|mx|], rows of stride R + 2
    const int LX0 = blockIdx.x * 2, LY0 = blockIdx.y * 2;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int2* ktab = reinterpret_cast<const int2*>(t.Krel);
    for (int i = tid; i < (R + 1) * W; i += 256) tab[i] = ktab[i];
    const auto weight = [&](int i) {  // halo cell i: leaf i / 64
        const int lf = i >> 6, LX = LX0 - D + lf % H, LY = LY0 - D + lf / H;
        return LX >= 0 && LY >= 0 && LX < nL && LY < nL ? t.q[(int64_t(LY) * nL + LX) * 64 + (i & 63)] : 0.0;
    };
    int e = kExpZero;
    for (int i = tid; i < H * H * 64; i += 256) e = max(e, exp_of(__double2hiint(weight(i)) & 0x7fffffff));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) wexp[warp] = e;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) e = max(e, wexp[i]);
    const bool bad = e == kExpBad;
    e = max(e, -900);
    for (int i = tid; i < H * H * 64; i += 256)
        qs[(i >> 3) * kNearRow + (i & 7)] = bad ? int2{0, 0} : split28(to_fixed(weight(i), e, t.near_q));
    __syncthreads();

    const int lx = (warp >> 1) & 1, ly = warp >> 2, ty = (lane >> 3) + 4 * (warp & 1), sy = lane & 7;
    const int LX = LX0 + lx, LY = LY0 + ly;
    double acc = 0.0;  // this lane's target, column sy of row ty
    FixedSum sum[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j].clear();
    // the eight lanes of a row: lane sy ends with target sy's sum (butterfly, in integers), as v1 2^68 + v0 2^28
    const auto drain = [&]() {
        long long v1[8], v0[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            long long hi;
            int lo;
            sum[j].digits(hi, lo);
            v1[j] = hi >> 12;
            v0[j] = (hi & 4095) << 28 | lo;
            sum[j].clear();
        }
#pragma unroll
        for (int o = 4; o >= 1; o >>= 1)
#pragma unroll
            for (int j = 0; j < o; ++j) {
                const bool up = (sy & o) != 0;
                const long long s1 = up ? v1[j] : v1[j + o], s0 = up ? v0[j] : v0[j + o];
                v1[j] = (up ? v1[j + o] : v1[j]) + __shfl_xor_sync(0xffffffffu, s1, o);
                v0[j] = (up ? v0[j + o] : v0[j]) + __shfl_xor_sync(0xffffffffu, s0, o);
            }
        const int unit = e - t.near_q - t.near_k;
        acc += fma(double(v1[0]), pow2(68 + unit), double(v0[0]) * pow2(28 + unit));
    };
    int n = 0;
    for (int i = 0; i < t.n_near; ++i) {
        const int2 o = t.near[i];
        if (LX + o.x < 0 || LY + o.y < 0 || LX + o.x >= nL || LY + o.y >= nL) continue;  // warp-uniform
        const int4* q4 = reinterpret_cast<const int4*>(qs + (((ly + D + o.y) * H + lx + D + o.x) * 8 + sy) * kNearRow);
        const int2* kr = tab + abs(8 * o.y + sy - ty) * W;
        int2 kc[15];  // source column r and target column j: kc[r - j + 7]
        int ks[15];
        const auto kernel = [&](int m) {
            kc[m] = kr[abs(8 * o.x - 7 + m)];
            ks[m] = kc[m].x + kc[m].y;
        };
#pragma unroll
        for (int m = 0; m < 7; ++m) kernel(m);
#pragma unroll
        for (int r2 = 0; r2 < 4; ++r2) {
            const int4 a = q4[r2];
            const int2 q[2] = {int2{a.x, a.y}, int2{a.z, a.w}};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                kernel(2 * r2 + u + 7);
                const int qsum = q[u].x + q[u].y;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int m = 2 * r2 + u - j + 7;
                    sum[j].add(q[u], qsum, kc[m], ks[m]);
                }
            }
        }
        // 16 leaves, 128 terms a thread: the sums stay below 2^63 (f64_pack_near), v1 then adds eight lanes
        if ((++n & 15) == 0) drain();
    }
    drain();
    const double out = bad ? __longlong_as_double(0x7ff8000000000000ll) : acc;
    p_out[int64_t(LY * 8 + ty) * t.n + LX * 8 + sy] = out;
}

// ------------------------------------------------------------------------------------
// Multipole-to-local translations of every level in fixed point.  Per list entry the operator is
// one complex P1 x P1 matrix B (the same for all targets of a child position); a row l of B is
// scaled by a power of two that makes its largest entry below 1 (with column k carrying the
// 2^-floor(k/2) the multipoles are scaled by), wbits fixed-point bits; the multipoles have kM2LBits
// relative to the largest of the two levels involved.  Complex products by three real ones,
// (a + i b)(c + i d): ac, bd and (a + b)(c + d) accumulate separately over all entries, modulo 2^64:
// only their differences have to fit, and those are bounded by the sum of a row's entries over an entry
// group's part of the list, 4 to 45 times the largest, not by their number (f64_pack_m2l).  So 56 + 57 bits
// fit; with 52 + 54 the dropped low products were 2^-52 of the largest term and the far field's error up
// to 20 times that of FP64 multiply-adds; now 0.5 to 1.1 times.
// A CTA takes 32 targets of one child position (lane = target): warp = entry group x rows; four
// entry groups of four warps, each staging its entries' sources (converted from FP64) and operator
// in shared memory, one entry ahead.  Small grids split the entries further over a cluster of CTAs
// that add their integer sums through distributed shared memory.  The S log(|tau| side) terms stay FP64, a
// logarithm each (log|tau| and log side apart cancel).
// Bound by the integer multiply-adds, 9 per complex product: 390 us at 1024^2, p = 20, theta = 0.5
// at the measured rate; 2665 us before on the FP64 pipe in one launch per level, 922 now.
// ------------------------------------------------------------------------------------
constexpr int kM2LPad = 33;
constexpr int kM2LBits = 56;

__host__ __device__ constexpr size_t m2l64_group_bytes(int P1) {  // one buffer of one entry group
    return sizeof(int4) * (size_t(P1) * kM2LPad + size_t(P1) * P1);
}
inline size_t m2l64_smem(int P1) {  // the staging buffers, later the groups' sums and S terms
    const size_t stage = 8 * m2l64_group_bytes(P1), rows = P1 <= 16 ? 16 : P1 <= 20 ? 20 : 24;
    const size_t sums = 4 * rows * 4 * 32 * 8 + 4 * 32 * 8;
    return stage > sums ? stage : sums;
}

__device__ __forceinline__ void group_sync(int g) {
    switch (g) {
        case 0: asm volatile("bar.sync 1, 128;" ::: "memory"); break;
        case 1: asm volatile("bar.sync 2, 128;" ::: "memory"); break;
        case 2: asm volatile("bar.sync 3, 128;" ::: "memory"); break;
        default: asm volatile("bar.sync 4, 128;" ::: "memory"); break;
    }
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// 8 bytes of another cluster CTA's shared memory, at the address `own` has in this CTA's.
__device__ __forceinline__ long long ld_peer64(const void* own, uint32_t rank) {
    uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(own)), pa;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(pa) : "r"(a), "r"(rank));
    long long v;
    asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(pa) : "memory");
    return v;
}

template <int NL>
__global__ void __launch_bounds__(512, 1) k_m2l64(Tree<double> t, F64Scales sc, int cs) {
    extern __shared__ __align__(16) int4 smm[];
    const int P1 = t.P1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int eg = warp >> 2, lg = warp & 3, gt = tid & 127;
    const uint32_t rank = cs > 1 ? cluster_rank() : 0;
    // the CTA's level, child position and chunk of 32 targets (finest level first)
    int64_t c = blockIdx.x / cs;
    int l = t.Lleaf;
    int64_t chunks;
    for (;; --l) {
        chunks = ((int64_t(1) << (2 * (l - 1))) + 31) >> 5;
        if (c < 4 * chunks) break;
        c -= 4 * chunks;
    }
    const int side = 1 << l, half = side >> 1;
    const int par = int(c & 3);
    const int64_t idx = (c >> 2) * 32 + lane;
    const bool act = idx < int64_t(half) * half;
    const int px = act ? int(idx % half) : 0, py = act ? int(idx / half) : 0;  // the target's parent
    const int64_t off = level_offset(l), offp = level_offset(l - 1);
    const int* le = level_exp(t);
    int E = max(le[l], le[l - 1]);
    const bool bad = E == kExpBad;
    E = max(E, -840);  // so that every unit below is a normal number
    const M2LEntry* lst = t.il + int64_t(par) * t.il_stride;
    const int cnt = t.il_count[par];
    int4* const buf0 = smm + size_t(eg) * 2 * (P1 * kM2LPad + P1 * P1);
    const int bufn = P1 * kM2LPad + P1 * P1;
    const int4* ops = reinterpret_cast<const int4*>(t.Bm2l);  // [op][k][l] fixed point

    // the source box of target lane j for entry en (-1: outside the grid)
    const auto source = [&](const M2LEntry& en, int jx, int jy, bool ja) -> int64_t {
        if (!ja) return -1;
        if (en.pad == 0) {
            const int sx = 2 * jx + (par & 1) + en.dx, sy = 2 * jy + (par >> 1) + en.dy;
            return sx >= 0 && sy >= 0 && sx < side && sy < side ? off + int64_t(sy) * side + sx : -1;
        }
        const int sx = jx + en.dx, sy = jy + en.dy;
        return sx >= 0 && sy >= 0 && sx < half && sy < half ? offp + int64_t(sy) * half + sx : -1;
    };
    const auto stage = [&](int e, int b) {  // by the 128 threads of the group
        const M2LEntry en = lst[e];
        int4* xs = buf0 + b * bufn;
        int4* ws = xs + P1 * kM2LPad;
        const int4* wop = ops + int64_t(en.op) * P1 * P1;
        for (int i = gt; i < P1 * P1; i += 128) cp_async16(ws + i, wop + i);
        cp_async_commit();
        const int64_t mine = source(en, px, py, act);
#pragma unroll
        for (int i = 0; i < 8; ++i) {  // box of lane 8 lg + i, one coefficient a thread
            const int j = 8 * lg + i;
            const int64_t s = __shfl_sync(0xffffffffu, mine, j);
            if (lane < P1) {
                int4 x = make_int4(0, 0, 0, 0);
                if (s >= 0 && !bad) {
                    const double2 m = t.mp[s * P1 + lane];
                    const int2 re = split28(to_fixed(m.x, E - (lane >> 1), kM2LBits)),
                               im = split28(to_fixed(m.y, E - (lane >> 1), kM2LBits));
                    x = make_int4(re.x, re.y, im.x, im.y);
                }
                xs[lane * kM2LPad + j] = x;
            }
        }
    };
    long long h1[NL], m1[NL], h2[NL], m2[NL], h3[NL], m3[NL];
#pragma unroll
    for (int i = 0; i < NL; ++i) h1[i] = m1[i] = h2[i] = m2[i] = h3[i] = m3[i] = 0;
    const double lnS = fma(double(-l), 0.69314718055994530941723212145818, sc.ln_root);  // log of the box side
    double a0 = 0.0;
    const int l0 = lg * NL;  // this warp's rows l0 .. l0 + NL - 1 (those below P1)
    const int step = 4 * cs, first = int(rank) * 4 + eg;
    const auto fold = [&]() {  // mid's upper part into hh, 28 bits left
#pragma unroll
        for (int i = 0; i < NL; ++i) {
            h1[i] += m1[i] >> 28, m1[i] &= 0x0fffffff;
            h2[i] += m2[i] >> 28, m2[i] &= 0x0fffffff;
            h3[i] += m3[i] >> 28, m3[i] &= 0x0fffffff;
        }
    };
    if (first < cnt) stage(first, 0);
    int b = 0, done = 0;
    for (int e = first; e < cnt; e += step, b ^= 1) {
        cp_async_wait<0>();
        group_sync(eg);  // buffer b is staged, buffer b ^ 1 is free
        if (e + step < cnt) stage(e + step, b ^ 1);
        const int4* xs = buf0 + b * bufn + lane;
        const int4* ws = buf0 + b * bufn + P1 * kM2LPad + l0;
        if (l0 < P1) {
#pragma unroll 1
            for (int k = 0; k < P1; ++k) {
                const int4 x = xs[k * kM2LPad];
                const int xh = x.x + x.z, xl = x.y + x.w;
#pragma unroll
                for (int i = 0; i < NL; ++i) {
                    if (l0 + i < P1) {  // warp-uniform
                        const int4 w = ws[k * P1 + i];
                        const int wh = w.x + w.z, wl = w.y + w.w;
                        mad_wide(h1[i], x.x, w.x);
                        mad_wide(m1[i], x.x, w.y);
                        mad_wide(m1[i], x.y, w.x);
                        mad_wide(h2[i], x.z, w.z);
                        mad_wide(m2[i], x.z, w.w);
                        mad_wide(m2[i], x.w, w.z);
                        mad_wide(h3[i], xh, wh);
                        mad_wide(m3[i], xh, wl);
                        mad_wide(m3[i], xl, wh);
                    }
                }
            }
        }
        if ((++done & sc.fold_mask) == 0) fold();  // that many entries of the cross terms stay below 2^63
        if (lg == 0) {
            const M2LEntry en = lst[e];
            const int64_t s = source(en, px, py, act);
            if (s >= 0) {
                a0 = fma(t.S[s], t.lnTau[en.op] + lnS, a0);
            }
        }
    }
    fold();
    // the groups' and the cluster's sums: real part 1 - 2, imaginary part 3 - 1 - 2, per row; the rows
    // are dealt to the cluster's CTAs and their warps
    __syncthreads();  // the staging buffers are free
    long long* red = reinterpret_cast<long long*>(smm);  // [group][row][re hh, re mid, im hh, im mid][32]
    double* redS = reinterpret_cast<double*>(red + size_t(4) * 4 * NL * 4 * 32);
#pragma unroll
    for (int i = 0; i < NL; ++i) {
        long long* o = red + ((size_t(eg) * 4 * NL + l0 + i) * 4) * 32 + lane;
        o[0] = h1[i] - h2[i];
        o[32] = m1[i] - m2[i];
        o[64] = h3[i] - h1[i] - h2[i];
        o[96] = m3[i] - m1[i] - m2[i];
    }
    if (lg == 0) redS[eg * 32 + lane] = a0;
    if (cs > 1) cluster_sync_all();
    else __syncthreads();
    for (int ll = int(rank) + cs * warp; ll < P1; ll += 16 * cs) {
        long long v[4] = {0, 0, 0, 0}, w[2] = {0, 0};  // w: the upper sums' low 16 bits (a group's may fill 64)
        for (int r = 0; r < cs; ++r) {
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const long long* o = red + ((size_t(g) * 4 * NL + ll) * 4) * 32 + lane;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const long long x = r == int(rank) ? o[32 * u] : ld_peer64(o + 32 * u, r);
                    v[u] += u & 1 ? x : x >> 16;
                    if (!(u & 1)) w[u >> 1] += x & 0xffff;
                }
            }
        }
        // units: 2^(E - kM2LBits) 2^-wbits 2^el(l)
        const int s = E - kM2LBits - sc.wbits + sc.el[ll];
        double re = fma(double(v[0]), pow2(72 + s), double((w[0] << 28) + v[1]) * pow2(28 + s));
        double im = fma(double(v[2]), pow2(72 + s), double((w[1] << 28) + v[3]) * pow2(28 + s));
        if (bad) re = im = __longlong_as_double(0x7ff8000000000000ll);
        if (ll == 0) {
            double A = 0.0;
            for (int r = 0; r < cs; ++r)
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const double* o = redS + g * 32 + lane;
                    A += r == int(rank) ? *o : __longlong_as_double(ld_peer64(o, r));
                }
            re += A;
            im = 0.0;
        }
        if (act) {
            const int64_t box = off + int64_t(2 * py + (par >> 1)) * side + 2 * px + (par & 1);
            t.loc[box * P1 + ll] = double2{re, im};
            if (ll == 0) t.L0[box] = re;
        }
    }
    if (cs > 1) cluster_sync_all();  // no CTA leaves while its sums are being read
}

// ------------------------------------------------------------------------------------
// Local-to-local.  With zeta_q = i^m(q) zeta_3, the four children of a box share the partial sums
// over k = r mod 4, Y_r[l] = sum C(k, l) zeta_3^k b_k:
//   c_l = (2 zeta_3)^-l sum_r i^(m(q) (r - l)) Y_r[l],  constant: Re sum_r i^(m(q) r) Y_r[0].
// A warp per parent, lane l forms coefficient l of all four children.
// ------------------------------------------------------------------------------------
// Children's locals (the multipole-to-local part in cl, updated in place: this lane's coefficient l
// and, in lane 0, the constant c0) from the parent's local b (lane l's coefficient) and constant p0.
__device__ __forceinline__ void l2l_children(double2* Y, const double (*Rl)[kMaxP], int P1, int l, double2 b, double p0,
                                             double2 zl, double2 zil, double2 (&cl)[4], double (&c0)[4]) {
    const auto mul = [](double2 a, double2 c) { return double2{fma(a.x, c.x, -a.y * c.y), fma(a.x, c.y, a.y * c.x)}; };
    __syncwarp();
    if (l < P1) Y[l] = l == 0 ? double2{0.0, 0.0} : mul(b, zl);
    __syncwarp();
    double2 y[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) y[r] = double2{0.0, 0.0};
    const int lc = l < P1 ? l : 0;
    for (int k0 = 0; k0 < P1; k0 += 4)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int k = k0 + r;
            if (k < P1) {
                const double c = Rl[k][lc];
                const double2 w = Y[k];
                y[r].x = fma(c, w.x, y[r].x);
                y[r].y = fma(c, w.y, y[r].y);
            }
        }
    // u_s = sum_r i^(s (r - l)) y_r for s = m(q): rotate y so that index 0 is r = l mod 4
    double2 z[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int s = (r + lc) & 3;
        z[r] = s == 0 ? y[0] : s == 1 ? y[1] : s == 2 ? y[2] : y[3];
    }
    const double2 e{z[0].x + z[2].x, z[0].y + z[2].y}, f{z[1].x + z[3].x, z[1].y + z[3].y};
    const double2 g{z[0].x - z[2].x, z[0].y - z[2].y}, h{z[1].x - z[3].x, z[1].y - z[3].y};
    const double2 s[4] = {double2{e.x + f.x, e.y + f.y}, double2{g.x - h.y, g.y + h.x}, double2{e.x - f.x, e.y - f.y},
                          double2{g.x + h.y, g.y - h.x}};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const double2 v = s[q == 3 ? 0 : q == 2 ? 1 : q == 0 ? 2 : 3];
        if (l == 0) c0[q] += p0 + v.x;
        const double2 d = mul(v, zil);
        cl[q].x += d.x;
        cl[q].y += d.y;
    }
}

__device__ __forceinline__ void stage_l2l(double (*Rl)[kMaxP], int P1) {
    for (int i = threadIdx.x; i < P1 * P1; i += blockDim.x) Rl[i / P1][i % P1] = g_ops.l2l[i % P1][i / P1];
}

// One level: the boxes of level l (their complete locals) into their children, in place.
__global__ void __launch_bounds__(128) k_l2l64(Tree<double> t, int l) {
    __shared__ double Rl[kMaxP][kMaxP];  // [k][l] = C(k, l)
    __shared__ double2 Ys[4][kMaxP];
    const int P1 = t.P1, w = threadIdx.x >> 5, k = threadIdx.x & 31;
    stage_l2l(Rl, P1);
    __syncthreads();
    const int64_t b = int64_t(blockIdx.x) * 4 + w;
    if (b >= (int64_t(1) << (2 * l))) return;
    const int side = 1 << l, kc = k < P1 ? k : 0;
    const int64_t box = level_offset(l) + b;
    const int64_t child = level_offset(l + 1) + 2 * (b >> l) * (2 * side) + 2 * (b & (side - 1));
    double2 cl[4];
    double c0[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t c = child + int64_t(q >> 1) * (2 * side) + (q & 1);
        cl[q] = t.loc[c * P1 + kc];
        c0[q] = t.L0[c];
    }
    l2l_children(Ys[w], Rl, P1, k, t.loc[box * P1 + kc], t.L0[box], t.Zq[3 * P1 + kc], t.Ziq[3 * P1 + kc], cl, c0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t c = child + int64_t(q >> 1) * (2 * side) + (q & 1);
        if (k < P1) t.loc[c * P1 + k] = k == 0 ? double2{c0[q], 0.0} : cl[q];
        if (k == 0) t.L0[c] = c0[q];
    }
}

// ------------------------------------------------------------------------------------
// The last levels of shifts and the evaluation, one CTA per box of level lr = L - depth (depth 2, or
// 3 where that still gives every SM a CTA): the subtree's locals pass through shared memory, a
// warp per parent; then lane = leaf, a warp per orbit of cells (see k_p2m64): with G, H the sums over
// l = 0, 2 mod 4 of Re(L_l w^l) and E, F the sums over odd l of Re(L_l w^l) and +-Im(L_l w^l), the
// values at w, iw, -w, -iw are G + H + E, G - H - F, G + H - E, G - H + F, and those at conj(w)
// share the four products: 80 FP64 instructions for 8 cells at p = 20 in place of 640.
// ------------------------------------------------------------------------------------
constexpr int kDown64Warps = 10;  // one per orbit of cells

template <int depth>
__global__ void __launch_bounds__(32 * kDown64Warps) k_down64(Tree<double> t, double* __restrict__ p_out) {
    constexpr int kLeaves = 1 << (2 * depth), TL = 1 << depth;
    extern __shared__ __align__(16) double2 smd[];
    __shared__ double Rl[kMaxP][kMaxP];
    constexpr int kThreads = 32 * kDown64Warps;
    __shared__ double2 Ys[kDown64Warps][kMaxP];
    __shared__ double2 Vs[10 * kMaxP];
    const int P1 = t.P1, tid = threadIdx.x, w = tid >> 5, k = tid & 31;
    const int lr = t.Lleaf - depth, X = blockIdx.x, Y = blockIdx.y;
    double2* Ls = smd;                                                   // levels lr .. L: [box][P1]
    constexpr int kBoxes = depth == 3 ? 85 : 21;
    double* L0s = reinterpret_cast<double*>(Ls + kBoxes * P1);           // [box]
    double* Lt = L0s + kBoxes;                                           // leaves: [2 P1][kLeaves + 1]
    stage_l2l(Rl, P1);
    stage_orbits(Vs, t.Vl2p, P1);
    for (int j = 0, sb = 0; j <= depth; sb += 1 << (2 * j), ++j) {
        const int wd = 1 << j, lev = lr + j;
        const int64_t row0 = level_offset(lev) + int64_t(Y * wd) * (1 << lev) + X * wd;
        for (int i = tid; i < wd * wd * P1; i += kThreads) {
            const int bx = i / P1;
            Ls[sb * P1 + i] = t.loc[(row0 + int64_t(bx >> j) * (1 << lev) + (bx & (wd - 1))) * P1 + i - bx * P1];
        }
        for (int i = tid; i < wd * wd; i += kThreads) L0s[sb + i] = t.L0[row0 + int64_t(i >> j) * (1 << lev) + (i & (wd - 1))];
    }
    __syncthreads();
    const int kc = k < P1 ? k : 0;
    const double2 zl = t.Zq[3 * P1 + kc], zil = t.Ziq[3 * P1 + kc];
    for (int j = 0, sb = 0; j < depth; sb += 1 << (2 * j), ++j) {
        const int wd = 1 << j, cb = sb + wd * wd;
        for (int b = w; b < wd * wd; b += kDown64Warps) {
            const int ch = cb + 2 * (b >> j) * (2 * wd) + 2 * (b & (wd - 1));
            double2 cl[4];
            double c0[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int c = ch + (q >> 1) * 2 * wd + (q & 1);
                cl[q] = Ls[c * P1 + kc];
                c0[q] = L0s[c];
            }
            l2l_children(Ys[w], Rl, P1, k, Ls[(sb + b) * P1 + kc], L0s[sb + b], zl, zil, cl, c0);
            const int64_t row0 = level_offset(lr + j + 1) + int64_t(Y * 2 * wd) * (1 << (lr + j + 1)) + X * 2 * wd;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int cy = 2 * (b >> j) + (q >> 1), cxx = 2 * (b & (wd - 1)) + (q & 1);
                const int c = cb + cy * 2 * wd + cxx;
                const int64_t gb = row0 + int64_t(cy) * (1 << (lr + j + 1)) + cxx;
                const double2 v = k == 0 ? double2{c0[q], 0.0} : cl[q];
                if (k < P1) {
                    Ls[c * P1 + k] = v;
                    t.loc[gb * P1 + k] = v;
                }
                if (k == 0) {
                    L0s[c] = c0[q];
                    t.L0[gb] = c0[q];
                }
            }
        }
        __syncthreads();
    }
    if (!p_out) return;
    // leaves transposed (lane = leaf), and their constants: Re b_0 plus near_ln times the near monopoles
    constexpr int lb = kBoxes - kLeaves, LS = kLeaves + 1;
    for (int i = tid; i < kLeaves * P1; i += kThreads) {
        const int lf = i / P1, kk = i - lf * P1;
        const double2 v = Ls[(lb + lf) * P1 + kk];
        Lt[2 * kk * LS + lf] = v.x;
        Lt[(2 * kk + 1) * LS + lf] = v.y;
    }
    __syncthreads();
    const int side = 1 << t.Lleaf;
    for (int lf = tid; lf < kLeaves; lf += kThreads) {
        const int LX = X * TL + (lf & (TL - 1)), LY = Y * TL + lf / TL;
        double s = 0.0;
        for (int e = 0; t.near_ln != 0.0 && e < t.n_near; ++e) {
            const int2 o = t.near[e];
            const int sx = LX + o.x, sy = LY + o.y;
            if (sx >= 0 && sy >= 0 && sx < side && sy < side) s += t.S[level_offset(t.Lleaf) + int64_t(sy) * side + sx];
        }
        Lt[lf] = fma(t.near_ln, s, L0s[lb + lf]);
    }
    __syncthreads();
    constexpr int kGroups = (kLeaves + 31) / 32;
    for (int item = w; item < 10 * kGroups; item += kDown64Warps) {
        const int orb = item / kGroups, lf = (item % kGroups) * 32 + k;
        const bool act = lf < kLeaves;
        const int a = orbit_of(orb).x, b = orbit_of(orb).y;
        const double* L = Lt + (act ? lf : 0);
        const double2* V = Vs + orb * P1;  // w^l
        double g1 = 0.0, g2 = 0.0, h1 = 0.0, h2 = 0.0, e1 = 0.0, e2 = 0.0, f1 = 0.0, f2 = 0.0;
#pragma unroll 1
        for (int l = 1; l < P1; l += 4) {
            const double2 v1 = V[l];
            const double* x = L + 2 * l * LS;
            e1 = fma(x[0], v1.x, e1);
            e2 = fma(x[LS], v1.y, e2);
            f1 = fma(x[0], v1.y, f1);
            f2 = fma(x[LS], v1.x, f2);
            if (l + 1 < P1) {
                const double2 v = V[l + 1];
                h1 = fma(x[2 * LS], v.x, h1);
                h2 = fma(x[3 * LS], v.y, h2);
            }
            if (l + 2 < P1) {
                const double2 v = V[l + 2];
                e1 = fma(x[4 * LS], v.x, e1);
                e2 = fma(x[5 * LS], v.y, e2);
                f1 = fma(-x[4 * LS], v.y, f1);
                f2 = fma(-x[5 * LS], v.x, f2);
            }
            if (l + 3 < P1) {
                const double2 v = V[l + 3];
                g1 = fma(x[6 * LS], v.x, g1);
                g2 = fma(x[7 * LS], v.y, g2);
            }
        }
        if (!act) continue;
        double* P = p_out + int64_t((Y * TL + lf / TL) * 8) * t.n + (X * TL + (lf & (TL - 1))) * 8;
        // the constant meets the near field, which it mostly cancels, before the series does
        const auto put = [&](int x2, int y2, double v) {
            double* d = P + int64_t((y2 + 7) >> 1) * t.n + ((x2 + 7) >> 1);
            *d = ((*d + L[0]) + v) * kInv2Pi;
        };
        {
            const double s = (g1 - g2) + (h1 - h2), d = (g1 - g2) - (h1 - h2), E = e1 - e2, F = f1 + f2;
            put(a, b, s + E), put(-b, a, d - F), put(-a, -b, s - E), put(b, -a, d + F);
        }
        if (a != b) {
            const double s = (g1 + g2) + (h1 + h2), d = (g1 + g2) - (h1 + h2), E = e1 + e2, F = f2 - f1;
            put(a, -b, s + E), put(b, a, d - F), put(-a, b, s - E), put(-b, -a, d + F);
        }
    }
}

}  // namespace f64

// ------------------------------------------------------------------------------------
// Launchers
// ------------------------------------------------------------------------------------
bool f64_ok(int P1, int Lleaf) { return P1 <= f64::kMaxP && Lleaf >= 2; }

size_t f64_counter_words(int Lleaf) { return 32 + size_t(level_offset(Lleaf - 1)); }

// The multipole-to-local operators [op][k][l] (FP64 complex, row scaling as in k_m2l64) as fixed
// point, in place of the FP64 values (16 bytes each either way).  wbits: the largest for which a row's sum
// over an entry group (every fourth of the list, or fewer), sum (|Re| + |Im|) of its entries, times the
// multipoles' 2^kM2LBits stays below 2^63 in units of 2^56, and the halves' sums below 2^31.  An entry's
// cross terms are below P1 2^(kM2LBits + 1) + 2^wbits sum (|Re| + |Im|); fold_mask + 1 entries of them stay
// below 2^63.
void f64_pack_m2l(double2* B, int n_ops, int P1, const M2LEntry* il, const int* il_count, int il_stride, F64Scales* sc) {
    const auto size = [](double2 b) { return std::fabs(b.x) + std::fabs(b.y); };
    double big[32] = {};  // largest scaled entry of each row
    for (int op = 0; op < n_ops; ++op)
        for (int k = 0; k < P1; ++k) {
            const double f = pow2(-(k >> 1));
            const double2* b = B + (size_t(op) * P1 + k) * P1;
            for (int l = 0; l < P1; ++l) big[l] = std::max(big[l], f * std::max(std::fabs(b[l].x), std::fabs(b[l].y)));
        }
    for (int l = 0; l < 32; ++l) sc->el[l] = l < P1 && big[l] > 0.0 ? std::ilogb(big[l]) + 1 : 0;
    std::vector<double> row(size_t(n_ops) * P1, 0.0);  // an entry's sums, in units of the row's scale
    double one = 0.0, all = 1.0;
    for (int op = 0; op < n_ops; ++op)
        for (int l = 0; l < P1; ++l) {
            double& r = row[size_t(op) * P1 + l];
            for (int k = 0; k < P1; ++k) r += size(B[(size_t(op) * P1 + k) * P1 + l]) * pow2(-(k >> 1) - sc->el[l]);
            one = std::max(one, r);
        }
    for (int c = 0; c < 16; ++c)
        for (int l = 0; l < P1; ++l) {
            double s = 0.0;
            for (int e = c >> 2; e < il_count[c & 3]; e += 4)
                s += row[size_t(il[size_t(c & 3) * il_stride + e].op) * P1 + l];
            all = std::max(all, s);
        }
    sc->wbits = 57;
    while (std::ldexp(all, f64::kM2LBits + sc->wbits - 56) > 9.2e18) --sc->wbits;
    const double cross = std::ldexp(double(P1), f64::kM2LBits + 1) + std::ldexp(one, sc->wbits);
    sc->fold_mask = 3;
    while (sc->fold_mask > 0 && cross * (sc->fold_mask + 1) > 9.2e18) sc->fold_mask >>= 1;
    for (int k = 0; k < P1; ++k)
        for (int l = 0; l < P1; ++l) {
            const double f = pow2(sc->wbits - (k >> 1) - sc->el[l]);
            for (int op = 0; op < n_ops; ++op) {
                double2& b = B[(size_t(op) * P1 + k) * P1 + l];
                const int2 re = split28(std::llrint(b.x * f)), im = split28(std::llrint(b.y * f));
                const int4 v = make_int4(re.x, re.y, im.x, im.y);
                std::memcpy(static_cast<void*>(&b), &v, sizeof(v));
            }
        }
}

// The near field's kernel table as a quadrant of fixed-point values: [|my|][|mx|], rows of R + 2; near_ln,
// the part of log h that is not in it.  Log h in long double: its error would be the same in every entry.
// The bits of weights (q) and values (k) by the table's largest value K: 128 terms of sum hh are below
// 2^(q + k + 7 - 56) K and of the cross terms below 2^(q + 6) + 2^(k + 6) K; with 56 + 53 bits and K < 6 (h
// above 1 / 140 where h < 1), 56 + 52 and K < 8, 55 + 52 and K < 16, both stay below 2^62.9.
void f64_pack_near(double* K, int R, double h, double* near_ln, int* near_q, int* near_k) {
    const long double lnh = std::log((long double)h);
    const long double in = std::min(std::max(lnh, (long double)-f64::kNearLn), (long double)f64::kNearLn);
    const auto value = [in](int x, int y) {
        return in + (x + y == 0 ? 0.78539816339744830962L - 1.5L - 0.34657359027997265471L
                                : (long double)(0.5 * std::log(double(x * x + y * y))));
    };
    const long double big = std::max(std::fabs(value(0, 0)), std::fabs(value(R + 1, R + 1)));
    *near_ln = double(lnh - in);
    *near_q = big < 8.0L ? 56 : 55;
    *near_k = big < 6.0L ? 53 : 52;
    int2* o = reinterpret_cast<int2*>(K);
    for (int y = 0; y <= R; ++y)
        for (int x = 0; x <= R + 1; ++x) o[size_t(y) * (R + 2) + x] = split28(std::llrint(std::ldexp(value(x, y), *near_k)));
}

cudaError_t launch_rhs64(const Tree<double>& t, const double* u, const double* v, const double* chi, const double* usx,
                         const double* usy, double rho, double lam, double* f_out, cudaStream_t st) {
    // rows a warp: as many as leave eight warps an SM (the two halo rows cost the fewer, the more rows)
    int rows = 8;
    while (rows > 2 && int64_t(t.n / 32) * (t.n / rows) < t.resident_threads / 256 * 8) rows >>= 1;
    const unsigned blocks = unsigned((int64_t(t.n / 32) * (t.n / rows) + 3) / 4);
    switch (rows) {
        case 2: f64::k_rhs64<2><<<blocks, 128, 0, st>>>(t, u, v, chi, usx, usy, rho, lam, f_out); break;
        case 4: f64::k_rhs64<4><<<blocks, 128, 0, st>>>(t, u, v, chi, usx, usy, rho, lam, f_out); break;
        default: f64::k_rhs64<8><<<blocks, 128, 0, st>>>(t, u, v, chi, usx, usy, rho, lam, f_out); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const unsigned nb = unsigned((int64_t(t.nL) * t.nL + 31) / 32);
    switch ((t.P1 + 3) / 4) {
        case 1: case 2: case 3: f64::k_p2m64<3><<<nb, 128, 0, st>>>(t); break;
        case 4: f64::k_p2m64<4><<<nb, 128, 0, st>>>(t); break;
        case 5: f64::k_p2m64<5><<<nb, 128, 0, st>>>(t); break;
        default: f64::k_p2m64<6><<<nb, 128, 0, st>>>(t); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_up64(const Tree<double>& t, cudaStream_t st) {
    const int64_t warps = int64_t(1) << (2 * (t.Lleaf - 1));
    f64::k_up64<<<unsigned((warps + 3) / 4), 128, 0, st>>>(t);
    return cudaGetLastError();
}

cudaError_t launch_near64(const Tree<double>& t, double* p_out, cudaStream_t st) {
    f64::k_near64<<<dim3(t.nL / 2, t.nL / 2), 256, f64::near64_smem(t.Dmax), st>>>(t, p_out);
    return cudaGetLastError();
}

// CTAs that share a chunk of targets (a cluster): enough for four CTAs an SM, at most 8.
static int m2l64_cluster(const Tree<double>& t, unsigned* chunks) {
    int64_t c = 0;
    for (int l = 2; l <= t.Lleaf; ++l) c += 4 * (((int64_t(1) << (2 * (l - 1))) + 31) >> 5);
    *chunks = unsigned(c);
    const int64_t want = t.resident_threads / 256 * 4;
    int cs = 1;
    while (cs < 8 && c * cs < want) cs <<= 1;
    return cs;
}

cudaError_t launch_m2l64(const Tree<double>& t, const F64Scales& sc, cudaStream_t st) {
    unsigned chunks;
    const int cs = m2l64_cluster(t, &chunks);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(cs);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(chunks * unsigned(cs));
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = f64::m2l64_smem(t.P1);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    switch ((t.P1 + 3) / 4) {
        case 1: case 2: case 3: case 4: return cudaLaunchKernelEx(&cfg, f64::k_m2l64<4>, t, sc, cs);
        case 5: return cudaLaunchKernelEx(&cfg, f64::k_m2l64<5>, t, sc, cs);
        default: return cudaLaunchKernelEx(&cfg, f64::k_m2l64<6>, t, sc, cs);
    }
}

static int down64_depth(int Lleaf, int64_t resident) {
    return Lleaf >= 3 && (int64_t(1) << (2 * (Lleaf - 3))) >= resident / 256 ? 3 : 2;
}

int f64_down_launches(const Tree<double>& t) {
    const int lr = t.Lleaf - down64_depth(t.Lleaf, t.resident_threads);
    return 1 + (lr > 2 ? lr - 2 : 0);
}

cudaError_t launch_down64(const Tree<double>& t, double* p_out, cudaStream_t st) {
    const int depth = down64_depth(t.Lleaf, t.resident_threads), lr = t.Lleaf - depth;
    for (int l = 2; l < lr; ++l) {
        f64::k_l2l64<<<unsigned(((int64_t(1) << (2 * l)) + 3) / 4), 128, 0, st>>>(t, l);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const int boxes = depth == 3 ? 85 : 21, leaves = 1 << (2 * depth);
    const size_t smem = sizeof(double2) * boxes * t.P1 + sizeof(double) * (boxes + size_t(2) * t.P1 * (leaves + 1));
    const dim3 grid(1u << lr, 1u << lr);
    if (depth == 3) f64::k_down64<3><<<grid, 32 * f64::kDown64Warps, smem, st>>>(t, p_out);
    else f64::k_down64<2><<<grid, 32 * f64::kDown64Warps, smem, st>>>(t, p_out);
    return cudaGetLastError();
}

cudaError_t prepare_f64() {
    const void* fns[] = {(const void*)f64::k_near64, (const void*)f64::k_m2l64<4>, (const void*)f64::k_m2l64<5>,
                         (const void*)f64::k_m2l64<6>, (const void*)f64::k_down64<2>, (const void*)f64::k_down64<3>};
    for (const void* f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace pp
