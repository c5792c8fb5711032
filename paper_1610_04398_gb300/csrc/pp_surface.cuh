// (a7) + (a8) Surface pressure by the tree-code (Sec. A.2, Fig. "multipole"), the tractions of Sec.
// 2.3 and their integrals in one launch, for both precisions.
#pragma once

#include "pp_common.h"
#include "pp_fixed.cuh"
#include "pp_log.cuh"

namespace pp {

// Points a CTA walks at once, a warp each; one more warp forms their tractions, a lane each.  The
// FP64 walk is bound by its SM's FP64 pipe: few points a CTA, so that few points still spread over
// the SMs.  The mixed walk has no FP64: as many points as fill the traction warp's instructions.
// kMany (mixed, more points than one wave of the other form holds, 24 an SM): 64 registers instead
// of 72, so that an SM holds 28 points.  The 4096 points of a 256^2 step were 1.12 waves and every
// warp's chain ran twice: 25.9 us, now 22.7 (in the step, 51.1 to 47.2).  Up to one wave the 72 registers
// are better: 2048 points at 2048^2 take 21.0 against 22.0 us (146.0 against 147.4 in the step).
template <typename T, bool kMany = false>
struct SurfCta {
    static constexpr int warps = sizeof(T) == 8 ? 4 : kMany ? 7 : 8;
    static constexpr int ctas = kMany ? 4 : 3;  // per SM
    static constexpr int threads = 32 * (warps + 1);
};
constexpr int kSurfCap = 256;         // candidates of a level; accepted boxes a warp holds at once (FP64)
constexpr int kSurfLane = 16;         // accepted boxes a lane holds at once (mixed)
constexpr int kSurfLeaves = 64;       // leaves summed directly, per point

struct SurfWalk {  // a warp's lists
    int cand[2][kSurfCap];
    int taken[kSurfLane * 32];  // level << 24 | box: [slot][lane] (mixed), or kSurfCap in order (FP64)
    int leaves[kSurfLeaves];
};

__device__ __forceinline__ float surf_log(float x) { return logf(x); }
__device__ __forceinline__ double surf_log(double x) { return log_table(x); }

// A point and, for mixed plans and points inside the domain, its cell and the fraction in it.
struct SurfPoint {
    double zx, zy;
    int inside, ix, iy;
    float fx, fy;
};

// The walk's result: 2 pi P, as a double-float pair without the log h part (pair), or in FP64.
struct SurfPhi {
    double phi;
    float hi, lo;
    int pair;
};

// 2 pi P at a point, one warp.  From the root down a box is accepted when r_box < theta d; the
// accepted boxes are only listed, so a level costs its tests and no memory latency, and then
// evaluated (Eq. pressTruncated about each centre), a lane each: in FP64, whose pipe bounds the walk, 32
// at a time whatever lane listed them; in mixed plans by the lane that listed them, in order, so a
// lane's FP32 sum has the terms and the order of a walk that evaluates each level as it goes.
// Leaves that are never accepted are summed directly, two cells a lane.  A level's open boxes lie within
// side / (sqrt 2 theta) of the point: at most 37 for theta >= 0.25.
//
// Mixed plans, points inside the domain: offsets in cell units, an exact integer difference plus
// the point's fraction of a cell (split by the traction warp), and the monopole sums as double-float
// pairs, so the walk has no FP64 (an FP64 instruction holds its SM's pipe for 19 cycles, and sixty
// of them a point were 13 of the walk's 25 us).  The log h parts of every accepted box and near cell add up to log h times
// the root monopole (they partition the domain) and enter once at the end.
// kCell: the cell-unit walk, without FP64 even in code that is predicated off.
template <typename T, int P1T, bool kCell>
__device__ __forceinline__ void surf_walk(const Tree<T>& t, const SurfaceArgs& a, const SurfPoint& pt, SurfWalk& sm,
                                          int lane, bool& overflow, SurfPhi& out) {
    typedef typename cplx_of<T>::type C;
    const int P1 = P1T > 0 ? P1T : t.P1;
    const double zx = pt.zx, zy = pt.zy, L = double(t.n) * t.h;
    // the root is never accepted for a point inside the domain: such points start from level 1
    const bool inside = kCell || pt.inside != 0;
    const int ix = pt.ix, iy = pt.iy;
    const float fx = pt.fx, fy = pt.fy;
    const auto offset = [&](int l, int bx, int by, T& dx, T& dy, T& s) {  // point minus centre, box side
        if constexpr (kCell) {
            const int sc = 8 << (t.Lleaf - l);
            dx = T(float(ix - (bx * sc + (sc >> 1))) + fx);
            dy = T(float(iy - (by * sc + (sc >> 1))) + fy);
            s = T(sc);
        } else {
            const double sd = L * pow2(-l);
            dx = T(zx - (t.x0 + (bx + 0.5) * sd));
            dy = T(zy - (t.y0 + (by + 0.5) * sd));
            s = T(sd);
        }
    };
    double mono = 0.0;
    float mh = 0.f, ml = 0.f;  // cell units: the monopole sum as a double-float pair
    T ser = T(0);
    const auto evaluate = [&](int lb) {
        const int l = lb >> 24, b = lb & 0xffffff, side = 1 << l;
        T dx, dy, s;
        offset(l, b & (side - 1), b >> l, dx, dy, s);
        const int64_t box = level_offset(l) + b;
        const Multipole<T> M = multipole(t, l, b);
        const T d2 = fma(dx, dx, dy * dy), sd = s / d2;
        const T ux = sd * dx, uy = -sd * dy;
        C h;
        if constexpr (P1T > 0 && sizeof(T) == 4) {
            static_assert(P1T % 2 == 1, "columns 1 .. P1 - 1 in pairs");
#pragma unroll
            for (int k = P1T - 2; k >= 1; k -= 2) {
                const float4 m = *M.pair(k);  // coefficients k and k + 1
                if (k == P1T - 2) {
                    h.x = m.z;
                    h.y = m.w;
                } else {
                    const T hr = fma(h.x, ux, fma(-h.y, uy, T(m.z)));
                    h.y = fma(h.x, uy, fma(h.y, ux, T(m.w)));
                    h.x = hr;
                }
                const T hr = fma(h.x, ux, fma(-h.y, uy, T(m.x)));
                h.y = fma(h.x, uy, fma(h.y, ux, T(m.y)));
                h.x = hr;
            }
        } else {
            h = M[P1 - 1];
#pragma unroll 4
            for (int k = P1 - 2; k >= 1; --k) {
                const C m = M[k];
                const T hr = fma(h.x, ux, fma(-h.y, uy, m.x));
                h.y = fma(h.x, uy, fma(h.y, ux, m.y));
                h.x = hr;
            }
        }
        const T lg = T(0.5) * surf_log(d2);
        if constexpr (kCell) {
            const float2 sp = t.Sf[box];
            df_fma(mh, ml, sp.x, sp.y, float(lg), 0.f);
        } else {
            mono = fma(t.S[box], double(lg), mono);
        }
        ser -= h.x * ux - h.y * uy;
    };
    const unsigned below = (1u << lane) - 1u;
    const T th2 = sizeof(T) == 8 ? T(a.theta * a.theta) : T(a.theta2f);
    int n = 1, cur = 0, na = 0, nleaf = 0;
    if (inside) {
        n = 4;
        if (lane < 4) sm.cand[0][lane] = lane;
    } else if (lane == 0) {
        sm.cand[0][0] = 0;
    }
    __syncwarp();
    for (int l = inside ? 1 : 0; l <= t.Lleaf; ++l) {
        const int side = 1 << l;
        int next = 0;
        for (int base = 0; base < n; base += 32) {
            const bool in = base + lane < n;
            const int b = in ? sm.cand[cur][base + lane] : 0;
            const int bx = b & (side - 1), by = b >> l;
            T dx, dy, s;
            offset(l, bx, by, dx, dy, s);
            const bool take = in && T(0.5) * s * s < th2 * fma(dx, dx, dy * dy), open = in && !take;
            const unsigned om = __ballot_sync(0xffffffffu, open);
            if constexpr (sizeof(T) == 4) {
                if (__any_sync(0xffffffffu, na == kSurfLane)) {  // make room
                    for (int i = 0; i < na; ++i) evaluate(sm.taken[i * 32 + lane]);
                    na = 0;
                }
                if (take) sm.taken[32 * na++ + lane] = l << 24 | b;
            } else {
                const unsigned tm = __ballot_sync(0xffffffffu, take);
                if (na > kSurfCap - 32) {
                    __syncwarp();  // the entries come from all lanes (a vote does not order memory)
                    for (int i = lane; i < na; i += 32) evaluate(sm.taken[i]);
                    na = 0;
                    __syncwarp();
                }
                if (take) sm.taken[na + __popc(tm & below)] = l << 24 | b;
                na += __popc(tm);
            }
            const int pos = __popc(om & below);
            if (l < t.Lleaf) {
                if (open) {
                    const int at = next + 4 * pos;
                    if (at + 4 <= kSurfCap) {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            sm.cand[cur ^ 1][at + q] = (2 * by + (q >> 1)) * (2 * side) + 2 * bx + (q & 1);
                    } else {
                        overflow = true;
                    }
                }
                next += 4 * __popc(om);
            } else {
                if (open) {
                    if (nleaf + pos < kSurfLeaves) sm.leaves[nleaf + pos] = b;
                    else overflow = true;
                }
                nleaf += __popc(om);
            }
        }
        __syncwarp();
        cur ^= 1;
        n = min(next, kSurfCap);
    }
    nleaf = min(nleaf, kSurfLeaves);
    if constexpr (sizeof(T) == 4) {
        for (int i = 0; i < na; ++i) evaluate(sm.taken[i * 32 + lane]);  // this lane's own
        __syncwarp();
    } else {
        for (int i = lane; i < na; i += 32) evaluate(sm.taken[i]);
    }
    T rh2, hT;
    if constexpr (kCell) rh2 = T(a.rho2_cell), hT = T(1);
    else rh2 = T(a.rho_h * a.rho_h), hT = T(t.h);
    T nearf = T(0);
    const T cxl = (T(lane & 7) + T(0.5)) * hT, cyl = (T(lane >> 3) + T(0.5)) * hT;  // cells lane, lane + 32
    const T cyh = (T((lane >> 3) + 4) + T(0.5)) * hT;
#pragma unroll 4
    for (int e = 0; e < nleaf; ++e) {
        const int b = sm.leaves[e];
        const int LX = b & (t.nL - 1), LY = b >> t.Lleaf;
        const T q0 = t.q[int64_t(b) * 64 + lane], q1 = t.q[int64_t(b) * 64 + 32 + lane];
        // point relative to the leaf corner (FP64, or exact cell units), cells relative to that in T
        T ox, oy;
        if constexpr (kCell) {
            ox = T(float(ix - 8 * LX) + fx);
            oy = T(float(iy - 8 * LY) + fy);
        } else {
            ox = T(zx - (t.x0 + 8.0 * LX * t.h));
            oy = T(zy - (t.y0 + 8.0 * LY * t.h));
        }
        const T dx = ox - cxl, dy = oy - cyl, dy1 = oy - cyh;
        const T x2 = dx * dx, r0 = fma(dy, dy, x2), r1 = fma(dy1, dy1, x2);
        T part = q0 * (T(0.5) * surf_log(r0 > rh2 ? r0 : rh2));
        part = fma(q1, T(0.5) * surf_log(r1 > rh2 ? r1 : rh2), part);
        if constexpr (kCell || sizeof(T) == 8) nearf += part;
        else mono += double(part);
    }
    if constexpr (kCell) {  // warp-uniform: the lanes' sums as double-float pairs, reduced on the FP32 pipe
        df_add(mh, ml, float(ser), 0.f);
        df_add(mh, ml, float(nearf), 0.f);
        for (int o = 16; o > 0; o >>= 1) {
            const float oh = __shfl_xor_sync(0xffffffffu, mh, o), ol = __shfl_xor_sync(0xffffffffu, ml, o);
            df_add(mh, ml, oh, ol);
        }
        if (lane == 0) out.hi = mh, out.lo = ml, out.pair = 1;
        return;
    }
    double tot = mono + double(ser) + double(nearf);
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) out.phi = tot, out.pair = 0;
}

__device__ __forceinline__ int clampi(double x, int lo, int hi) {
    if (!(x == x)) return lo;  // NaN
    if (x < double(lo)) return lo;
    if (x > double(hi)) return hi;
    return int(x);
}

// Velocity gradient at a cell by central differences.
template <typename T>
__device__ __forceinline__ void cell_grad(const T* u, const T* v, int n, double inv2h, int i, int j, double g[4]) {
    const int64_t c = int64_t(j) * n + i;
    g[0] = (double(u[c + 1]) - double(u[c - 1])) * inv2h;
    g[1] = (double(u[c + n]) - double(u[c - n])) * inv2h;
    g[2] = (double(v[c + 1]) - double(v[c - 1])) * inv2h;
    g[3] = (double(v[c + n]) - double(v[c - n])) * inv2h;
}

// "P is there", a barrier that the walking warps and the traction warp reach in different code:
// a named one, since __syncthreads() has to be the same for all threads of a block (bar.sync wants
// whole warps: the lanes join first).
template <int kThreads>
__device__ __forceinline__ void surf_barrier() {
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
}

// The walks, the tractions and the force sums in one launch.  The traction warp splits the CTA's points,
// then, while they are walked, forms what the tractions need besides P (the velocity gradient at the
// lifted point, the dS), then the tractions and their sums.  The CTA that finishes last (a counter it
// resets; no CTA waits) adds the CTAs' sums in a fixed order and forms drag and lift.  Before, the
// walk, the tractions (8.5 us, a chain of FP64 latencies) and the final sum (4.8 us) ran one after the
// other: 39 us for 2048 points at 2048^2, p = 12, theta 0.5, 19 now (4096 points at 256^2: 37, 21 now).
template <typename T, int P1T, bool kMany>
__global__ void __launch_bounds__((SurfCta<T, kMany>::threads), (SurfCta<T, kMany>::ctas))
k_surface(Tree<T> t, const T* __restrict__ u, const T* __restrict__ v, SurfaceArgs a) {
    constexpr int kWarps = SurfCta<T, kMany>::warps, kThreads = SurfCta<T, kMany>::threads;
    extern __shared__ __align__(16) unsigned char surf_smem[];
    SurfWalk* walk = reinterpret_cast<SurfWalk*>(surf_smem);  // [kWarps]
    __shared__ SurfPoint pts[kWarps];
    __shared__ SurfPhi phi[kWarps];
    __shared__ double red[4][kWarps + 1];
    __shared__ bool last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int chunks = (a.npts + kWarps - 1) / kWarps;
    double sum[4] = {0.0, 0.0, 0.0, 0.0};  // the traction warp's: F_P, F_nu
    for (int c = blockIdx.x; c < chunks; c += int(gridDim.x)) {
        const int p0 = c * kWarps;
        const int i = p0 + lane;
        const bool act = warp == kWarps && lane < kWarps && i < a.npts;
        double px = 0.0, py = 0.0;
        if (act) {
            px = a.pts[2 * i];
            py = a.pts[2 * i + 1];
            SurfPoint s;
            s.zx = px;
            s.zy = py;
            const double L = double(t.n) * t.h;
            s.inside = px >= t.x0 && px <= t.x0 + L && py >= t.y0 && py <= t.y0 + L && t.Lleaf >= 1;
            s.ix = s.iy = 0;
            s.fx = s.fy = 0.f;
            if (sizeof(T) == 4 && s.inside) {
                const double cxd = (px - t.x0) * t.inv_h, cyd = (py - t.y0) * t.inv_h;
                s.ix = int(floor(cxd));
                s.iy = int(floor(cyd));
                s.fx = float(cxd - s.ix);
                s.fy = float(cyd - s.iy);
            }
            pts[lane] = s;
        }
        __syncthreads();
        if (warp < kWarps) {
            if (p0 + warp < a.npts) {  // warp-uniform
                bool overflow = false;
                if (sizeof(T) == 4 && pts[warp].inside && t.Sf)  // (FP64 plans: the other walk)
                    surf_walk<T, P1T, sizeof(T) == 4>(t, a, pts[warp], walk[warp], lane, overflow, phi[warp]);
                else
                    surf_walk<T, P1T, false>(t, a, pts[warp], walk[warp], lane, overflow, phi[warp]);
                if (__any_sync(0xffffffffu, overflow) && lane == 0) atomicExch(a.err, 1);
            }
            surf_barrier<kThreads>();  // P is there
        } else {
            double nx = 0.0, ny = 0.0, dS = 0.0, tnx = 0.0, tny = 0.0, s0 = 0.0;
            if (act) {
                const int n = t.n;
                s0 = sizeof(T) == 4 ? t.lnh * t.S[0] : 0.0;  // log h times the root monopole
                nx = a.nrm[2 * i], ny = a.nrm[2 * i + 1];
                if (a.dS) {
                    dS = a.dS[i];
                } else {  // trapezoid weights on the closed polygon
                    const int ip = (i + 1 == a.npts) ? 0 : i + 1, im = (i == 0) ? a.npts - 1 : i - 1;
                    const double x1 = a.pts[2 * ip] - px, y1 = a.pts[2 * ip + 1] - py;
                    const double x0 = px - a.pts[2 * im], y0 = py - a.pts[2 * im + 1];
                    dS = 0.5 * (sqrt(x0 * x0 + y0 * y0) + sqrt(x1 * x1 + y1 * y1));
                }
                const double yx = px + a.lift * nx, yy = py + a.lift * ny;
                const double inv2h = 0.5 * t.inv_h;
                double g[4];
                if (a.interp == 0) {
                    const int ci = clampi(floor((yx - t.x0) / t.h), 1, n - 2);
                    const int cj = clampi(floor((yy - t.y0) / t.h), 1, n - 2);
                    cell_grad(u, v, n, inv2h, ci, cj, g);
                } else {
                    const double fxx = (yx - t.x0) / t.h - 0.5, fyy = (yy - t.y0) / t.h - 0.5;
                    const int i0 = clampi(floor(fxx), 1, n - 3), j0 = clampi(floor(fyy), 1, n - 3);
                    const double ax = fmin(fmax(fxx - i0, 0.0), 1.0), ay = fmin(fmax(fyy - j0, 0.0), 1.0);
                    const double wts[4] = {(1 - ax) * (1 - ay), ax * (1 - ay), (1 - ax) * ay, ax * ay};
                    for (int k = 0; k < 4; ++k) g[k] = 0.0;
                    for (int q = 0; q < 4; ++q) {
                        double gq[4];
                        cell_grad(u, v, n, inv2h, i0 + (q & 1), j0 + (q >> 1), gq);
                        for (int k = 0; k < 4; ++k) g[k] += wts[q] * gq[k];
                    }
                }
                const double dxy = 0.5 * (g[1] + g[2]);
                tnx = a.mu2 * (g[0] * nx + dxy * ny);
                tny = a.mu2 * (dxy * nx + g[3] * ny);
            }
            surf_barrier<kThreads>();  // P is there
            if (act) {
                const SurfPhi f = phi[lane];
                const double P = (f.pair ? df_to(f.hi, f.lo) + s0 : f.phi) * 0.15915494309189533576888376337251;
                const double tpx = -P * nx, tpy = -P * ny;
                if (a.per_point) {
                    double* o = a.per_point + int64_t(5) * i;
                    o[0] = P;
                    o[1] = tpx;
                    o[2] = tpy;
                    o[3] = tnx;
                    o[4] = tny;
                }
                sum[0] += tpx * dS;
                sum[1] += tpy * dS;
                sum[2] += tnx * dS;
                sum[3] += tny * dS;
            }
        }
        // the next chunk's points are written by the warp that has read this chunk's results
    }
    // the CTA's partial sums (the traction warp's lanes), kept in the plan's surface scratch
    if (warp == kWarps) {
        static_assert(kWarps <= 8, "points of a CTA in lanes 0 .. 7");
#pragma unroll
        for (int k = 0; k < 4; ++k)
            for (int o = 4; o > 0; o >>= 1) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], o);
        if (lane == 0) {
            for (int k = 0; k < 4; ++k) a.Psurf[4 * int64_t(blockIdx.x) + k] = sum[k];
            __threadfence();
            last = atomicAdd(t.surf_counter, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (unsigned b = threadIdx.x; b < gridDim.x; b += kThreads)
        for (int k = 0; k < 4; ++k) acc[k] += __ldcg(a.Psurf + 4 * int64_t(b) + k);
    if (warp * 32u < gridDim.x)  // the other warps hold zeros
        for (int k = 0; k < 4; ++k)
            for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
    if (lane == 0)
        for (int k = 0; k < 4; ++k) red[k][warp] = acc[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = min(kWarps + 1, int((gridDim.x + 31) / 32));
        double F[4];
        for (int k = 0; k < 4; ++k) {
            F[k] = red[k][0];
            for (int w = 1; w < nw; ++w) F[k] += red[k][w];
        }
        const double Fx = F[0] + F[2], Fy = F[1] + F[3];
        for (int k = 0; k < 4; ++k) a.forces[k] = F[k];
        a.forces[4] = Fx * a.uhat_x + Fy * a.uhat_y;
        a.forces[5] = -Fx * a.uhat_y + Fy * a.uhat_x;
        *t.surf_counter = 0u;
    }
}

}  // namespace pp
