// Density pass (steps O4, O3): the support radius H of every particle, its
// number density and its neighbour list.
//
// A group of lanes shares one particle (launches that fill the chip: one
// thread a particle, k_density_one).  The lanes take the cells of
// the search window in rounds, test their cell's candidates into a bit mask,
// place the hits by a prefix sum over the group (so the cache holds them in
// scan order: cells in row order, ascending index within a cell) and keep
// their share of the cached distances in registers for the iteration.  What
// bounds the pass is the chain of dependent loads (cell range, then
// candidates) and the instructions per candidate; a group shortens the chain
// by its lanes, keeps 4 to 8 times fewer particles' caches per block in
// shared memory, and loses less to lanes whose cells hold more particles
// than their neighbours' (an evolved state).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "gz_device.cuh"
#include "gz_launch.cuh"

namespace gz {

namespace {

inline int blocks(int n, int t) { return (n + t - 1) / t; }

constexpr int kDensBlock = 128;
constexpr int kDensCache = 64;  // candidates within 1.05 H a group can hold
constexpr int kLanes = 4;       // lanes of a group ...
constexpr int kWideLanes = 16;  // ... and in FP32 launches too small for those

// FP32 launches: below kWideMax particles sixteen lanes each, below kThreadMin
// four, and from there on one thread each (k_density_one), which fills the
// chip with fewer instructions a particle.  Measured, us a launch on the first
// steps (late in the run): Sod 16^3 sixteen lanes 24 (27), eight 28 (35), four
// 40 (53); Sod 32^3 sixteen 69 (81), eight 58 (68), four 50 (67), one 42 (81);
// KH 41^3 four 105 (99), one 66 (66); Sedov 64^3 one 100 (369); 128^3 one 806
// (1160).  FP64 keeps four: its sums are the lanes' sums.
constexpr int kWideMax = 12000;
constexpr int kThreadMin = 45000;
// Cells per axis from which k_density_one looks for warps whose windows lie
// inside the box (scan_inside): most warps of a large box (128^3: 865 us
// without, 803 with), few of an ensemble's small ones (703 without, 705 with).
constexpr int kInsideMin = 24;

// Radius of the candidate cache for a support Ht: 5% headroom so that small
// growth of H during the iteration needs no rescan, never past h_lim.
template <typename T>
__device__ __forceinline__ T dens_cache_radius(T Ht, const KParams& p) {
    T R = Ht * T(1.05);
    if (!(R < (T)p.h_lim)) R = max(Ht, (T)p.h_lim);
    return R;
}

// The two terms of the density sum at q = r/H: W(q) and -q W'(q) = x y.  One
// cubic in q (q <= 1/2) or 1 - q (beyond) with selected coefficients,
// W = 1 - 6x^2 + 6x^3 | 2x^3, -q W' = (12 - 18x) x^2 | (6 - 6x) x^2.  FP32: the
// second as two factors, summed by explicit multiply-adds, so that every form
// of the pass rounds its sums alike; callers add the entries with r < H.  FP64
// (halved and divided by 6; the pieces decided on the high word, no FP64
// comparison) vanishes beyond the support.
__device__ __forceinline__ void dens_terms2(float q, float& w, float& x, float& y) {
    const bool in = q <= 0.5f;
    const float t = in ? q : 1.f - q;
    x = t * t;
    w = fmaf(fmaf(in ? 6.f : 2.f, t, in ? -6.f : 0.f), x, in ? 1.f : 0.f);
    y = fmaf(in ? -18.f : -6.f, t, in ? 12.f : 6.f);
}
__device__ __forceinline__ void dens_terms2(double q, double& w, double& d) {
    const bool in = __double2hiint(q) < 0x3FE00000;
    const bool out = __double2hiint(q) >= 0x3FF00000;
    const double x = in ? q : 1.0 - q;
    const double x2 = x * x;
    const double a = fma(fma(in ? 3.0 : 1.0, x, in ? -3.0 : 0.0), x2, in ? 0.5 : 0.0);
    const double b = fma(in ? -3.0 : -1.0, x, in ? 2.0 : 1.0) * x2;
    w = out ? 0.0 : a;
    d = out ? 0.0 : b;
}

// r from r^2 for the iteration.
__device__ __forceinline__ float dist(float r2) {
    const float m = fmaxf(r2, 1e-37f);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(m));
    return m * y;
}
__device__ __forceinline__ double dist(double r2) { return sqrt(r2); }

template <int G, typename T>
__device__ __forceinline__ T group_add(unsigned gm, T v) {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) v += __shfl_xor_sync(gm, v, o);
    return v;
}

// One evaluation of the sums S = sum W and sd = sum -q W' over the entries with
// r < H among the n cached ones (scan order; lane l of a group of G holds
// entries l, l + G, ...: distance r[u] and r^2 at r2[u G + l]).
// FP32: a compensated sum over the entries in scan order, whichever form of
// the pass holds them (the support's last bits, and with them which pairs just
// reach each other, then do not depend on the form): the lanes form the terms
// of G entries and every lane adds all of them in order.
template <int G, int E>
__device__ __forceinline__ void group_eval(unsigned gm, int gl, int n, const float (&r)[E], const float* r2, float H,
                                           float& S, float& sd) {
    const float H2 = H * H, iH = 1.f / H;
    Acc sw;
    sd = 0.f;
#pragma unroll
    for (int u = 0; u < E; ++u) {
        if (u * G >= n) break;
        const int k = u * G + gl;
        const bool in = k < n && r2[k] < H2;
        float w, x, y;
        dens_terms2(r[u] * iH, w, x, y);
        const unsigned m = __ballot_sync(gm, in) >> (threadIdx.x & 31 & ~(G - 1));
#pragma unroll
        for (int s = 0; s < G; ++s) {
            const float ws = __shfl_sync(gm, w, s, G), xs = __shfl_sync(gm, x, s, G), ys = __shfl_sync(gm, y, s, G);
            if (m >> s & 1u) {
                sw.add(ws);
                sd = fmaf(ys, xs, sd);
            }
        }
    }
    S = sw.fvalue();
}
// FP64: the lanes' sums added up.
template <int G, int E>
__device__ __forceinline__ void group_eval(unsigned gm, int, int n, const double (&r)[E], const double*, double H,
                                           double& S, double& sd) {
    const double iH = 1.0 / H;
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int u = 0; u < E; ++u) {
        if (u * G >= n) break;
        double w, d;
        dens_terms2(r[u] * iH, w, d);
        a += w;
        b += d;
    }
    S = 2.0 * group_add<G>(gm, a);
    sd = 6.0 * group_add<G>(gm, b);
}

// Result of one evaluation: f's sign decides the bracket, and the next H.
template <typename T>
struct HIter {
    T lo = T(0), hi = T(0);
    bool has_lo = false, has_hi = false, clamped = false;
};

// One step of the bracketed Newton iteration on
// f(H) = (32/3)(1 + S) - N_ngb, f' = (32/3) sd / H, S = sum w, sd = sum -w' q.
// Returns true when |f| is within the tolerance, else sets H to the next
// trial.  FP32: f, the quotient and the bracket are FP32 numbers, the update
// H - f/f' is an FP64 one, whose results FP32 operations give exactly: the FP64
// difference of two FP32 numbers rounded to FP32 is their FP32 difference, and
// where that falls on an end of the bracket the sign of its rounding error
// tells which side the FP64 number lies on.  (The FP64 operations themselves,
// at 1/64 of the FP32 rate, would be a tenth of the pass.)
__device__ __forceinline__ bool h_step(HIter<float>& b, float& H, float S, float sd, const KParams& p, bool last) {
    const float C = 32.f / 3.f;
    const float f = C * __fadd_rn(1.f, S) - (float)p.ngb;
    if (fabsf(f) <= p.ftol) return true;
    if (last) return false;
    if (f < 0.f) {
        b.lo = H;
        b.has_lo = true;
    } else {
        b.hi = H;
        b.has_hi = true;
    }
    const float lo = b.has_lo ? b.lo : 0.5f * H, hi = b.has_hi ? b.hi : 2.f * H;
    const float fp = C * sd / H;
    float Hn = 0.f;
    bool ok = false;
    if (fp > 0.f) {
        const float q = f / fp;
        Hn = __fsub_rn(H, q);
        ok = Hn > lo && Hn < hi;
        if (Hn == lo || Hn == hi) {
            const float t = __fsub_rn(Hn, H);
            const float err = __fsub_rn(__fsub_rn(H, __fsub_rn(Hn, t)), __fadd_rn(q, t));  // (H - q) - Hn
            ok = Hn == lo ? err > 0.f : err < 0.f;
        }
    }
    if (!ok) Hn = (b.has_lo && b.has_hi) ? 0.5f * __fadd_rn(b.lo, b.hi) : (f < 0.f ? 2.f * H : 0.5f * H);
    if (Hn >= p.hlimf) {
        Hn = (float)(0.5 * ((double)H + p.h_lim));
        b.clamped = true;
    }
    H = Hn;
    return false;
}
__device__ __forceinline__ bool h_step(HIter<double>& b, double& H, double S, double sd, const KParams& p, bool last) {
    const double C = 32.0 / 3.0;
    const double f = C * (1.0 + S) - p.ngb;
    if (fabs(f) <= p.dtol) return true;
    if (last) return false;
    if (f < 0.0) {
        b.lo = H;
        b.has_lo = true;
    } else {
        b.hi = H;
        b.has_hi = true;
    }
    const double lo = b.has_lo ? b.lo : 0.5 * H, hi = b.has_hi ? b.hi : 2.0 * H;
    const double fp = C * sd / H;
    double Hn = 0.0;
    bool ok = false;
    if (fp > 0.0) {
        Hn = H - f / fp;
        ok = Hn > lo && Hn < hi;
    }
    if (!ok) Hn = (b.has_lo && b.has_hi) ? 0.5 * (b.lo + b.hi) : (f < 0.0 ? 2.0 * H : 0.5 * H);
    if (Hn >= p.h_lim) {
        Hn = 0.5 * (H + p.h_lim);
        b.clamped = true;
    }
    H = Hn;
    return false;
}

// Whether a support is wide (wide_cells).
template <typename T>
__device__ __forceinline__ bool wide(T R, const BoxInfo& bx) {
    return (float)R * (float)bx.nc > bx.wide;
}
template <typename T>
__device__ __forceinline__ bool in_box(const P4<T>& p) {
    return p.x >= T(0) && p.x <= T(1) && p.y >= T(0) && p.y <= T(1) && p.z >= T(0) && p.z <= T(1);
}
// Whether a particle's scan is left to a warp from the start.  A position outside
// the box (or none) sees no candidates: nothing to share.
template <typename T>
__device__ __forceinline__ bool to_warp(T R, const BoxInfo& bx, const P4<T>& me) {
    return wide(R, bx) && in_box(me);
}

// Cell coordinate of a position (as the binning forms it).
__device__ __forceinline__ int cell_at(float v, int nc) { return min(max((int)floorf(v * (float)nc), 0), nc - 1); }

// Starting H of particle i: its guess, or (flagged by the caller) the box's
// mean when the guess is unusable.
template <typename T>
__device__ __forceinline__ T h_start(T h, const BoxInfo& bx, const KParams& p, bool& bad) {
    bad = !((double)h > 0.0) || !((double)h < p.h_lim);
    if (!bad) return h;
    double H = cbrt(3.0 * p.ngb / (4.0 * kPi * (double)bx.count));
    if (!(H < p.h_lim)) H = 0.5 * p.h_lim;
    return (T)H;
}

__device__ __forceinline__ float n_of(float S, float H) {
    return 8.f * __fadd_rn(1.f, S) / ((float)kPi * H * H * H);
}
__device__ __forceinline__ double n_of(double S, double H) { return 8.0 * (1.0 + S) / (kPi * H * H * H); }

template <typename T, int G>
__global__ void __launch_bounds__(kDensBlock, sizeof(T) == 4 ? 7 : 1)
    k_density(int N, Sorted<T> s, Grid g, KParams p, unsigned* nbr, int* ncount,
              int* iters, DevStatus* st, const int* list,
              const int* nlist, int* defer, int* ndefer, int ccap) {
    after_previous();
    constexpr int P = kDensBlock / G, E = kDensCache / G;
    constexpr int S = kDensCache + G;  // (the groups of a warp start on different banks)
    __shared__ T c_r2[P][S];
    __shared__ unsigned c_j[P][S];
    const int gl = threadIdx.x % G, gp = threadIdx.x / G;
    const unsigned gm = group_mask<G>();
    int i = blockIdx.x * P + gp;
    if (list) {  // the particles of an index list only (hierarchical steps)
        if (i >= *nlist) return;
        i = list[i];
    } else if (i >= N) {
        return;
    }
    const BoxInfo bx = g.boxes[s.box[i]];
    const P4<T> me = s.pos[i];
    bool bad;
    T H = h_start<T>(s.h[i], bx, p, bad);
    if (bad && gl == 0) set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, s.id[i]);
    T Rc = T(-1), Hev = H, Sv = T(0), sdv = T(0);
    T r[E];
    int ncache = 0, it;
    HIter<T> b;
    bool conv = false;
    for (it = 1; it <= p.max_iter; ++it) {
        if (!(H <= Rc)) {  // first evaluation, or grown past the cache radius
            Rc = dens_cache_radius<T>(H, p);
            __syncwarp(gm);
            ncache = to_warp(Rc, bx, me) ? ccap + 1 : group_scan<T, G>(g, bx, s.pos, i, me.x, me.y, me.z, Rc, gl, gm, ccap,
                                            [&](int k, int j) {
                                                if (k < kDensCache) c_j[gp][k] = (unsigned)j;
                                            });
            if (ncache > ccap) {
                // more candidates than the cache holds (a support spanning
                // many cells): left to k_density_warp
                if (gl == 0) defer[atomicAdd(ndefer, 1)] = i;
                return;
            }
            __syncwarp(gm);
            bool outside = false;  // (FP64: the prefilter lets candidates just outside through)
            const T Rc2 = Rc * Rc;
#pragma unroll
            for (int u = 0; u < E; ++u) {
                const int k = u * G + gl;
                r[u] = T(8);  // (past every support)
                if (k < ncache) {
                    const P4<T> q = s.pos[c_j[gp][k]];
                    const T r2 = sep2(mi_diff(q.x, me.x, me.x - T(1)), mi_diff(q.y, me.y, me.y - T(1)),
                                      mi_diff(q.z, me.z, me.z - T(1)));
                    c_r2[gp][k] = r2;
                    r[u] = dist(r2);
                    if constexpr (sizeof(T) == 8) outside |= !(r2 < Rc2);
                }
            }
            if constexpr (sizeof(T) == 8) {
                // taken out (one particle in a thousand), so that every entry's
                // place, and with it the order of the sums, is the warp form's
                if (__any_sync(gm, outside)) {
                    __syncwarp(gm);
                    if (gl == 0) {
                        int kept = 0;
                        for (int k = 0; k < ncache; ++k) {
                            const T r2 = c_r2[gp][k];
                            if (!(r2 < Rc2)) continue;
                            c_r2[gp][kept] = r2;
                            c_j[gp][kept++] = c_j[gp][k];
                        }
                        ncache = kept;
                    }
                    ncache = __shfl_sync(gm, ncache, 0, G);
                    __syncwarp(gm);
#pragma unroll
                    for (int u = 0; u < E; ++u) r[u] = u * G + gl < ncache ? dist(c_r2[gp][u * G + gl]) : T(8);
                }
            }
        }
        group_eval<G>(gm, gl, ncache, r, c_r2[gp], H, Sv, sdv);
        Hev = H;
        if (h_step(b, H, Sv, sdv, p, it == p.max_iter)) {
            conv = true;
            break;
        }
    }
    if (it > p.max_iter) it = p.max_iter;
    const T H2 = Hev * Hev;
    int cnt = 0;
    for (int k0 = 0; k0 < ncache; k0 += G) {  // list of the returned H, in scan order
        const int k = k0 + gl;
        const bool in = k < ncache && c_r2[gp][k] < H2;
        const unsigned m = (__ballot_sync(gm, in) & gm) >> (threadIdx.x & 31 & ~(G - 1));
        const int slot = cnt + __popc(m & ((1u << gl) - 1u));
        if (in && slot < p.cap) store_slot(nbr + lslot(slot, i, N), c_j[gp][k]);
        cnt += __popc(m);
    }
    if (gl != 0) return;
    s.h[i] = Hev;
    s.n[i] = n_of(Sv, Hev);
    if (s.sd) s.sd[i] = sdv;  // (absent in the allocation-free density call)
    iters[i] = it;
    ncount[i] = cnt;
    if (!conv) {
        set_status(st, GZ_S_HCONV, GZ_C_HCONV, s.id[i]);
        if (b.clamped) atomicOr(&st->bits, GZ_S_HLIM);
    }
    if (cnt > p.cap) set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, s.id[i]);
}

// FP32, one thread per particle: the form for launches that fill the chip
// (k_density is faster below kThreadMin particles).  The first scan keeps
// (r^2, j) of the candidates within 1.05 H in the thread's column of shared
// memory.  Held to 96 registers (10 blocks of 64 per SM).
constexpr int kOneBlock = 64;
template <int kCache>
__device__ __noinline__ int dens_fill(const Grid& g, const BoxInfo& bx, const P4<float>* pos, int i,
                                      float xi, float yi, float zi, float R, float (*c_r2)[kOneBlock],
                                      unsigned (*c_j)[kOneBlock], int t) {
    const float R2 = R * R;
    int n = 0;
    for_candidates<float>(g, bx, pos, i, xi, yi, zi, R, [&](int j, float r2, bool ok) {
        const int k = min(n, kCache);
        c_r2[k][t] = r2;
        c_j[k][t] = (unsigned)j;
        n += ok && r2 < R2;
    });
    return n;
}

// The same scan for a window that does not reach the box's faces (lo..hi the
// cells of [x - R, x + R]): the same candidates, distances and order without
// any periodic shift, and the particle itself told apart once per four
// candidates.  pos is readable up to three records past its last.
template <typename E>
__device__ __forceinline__ void scan_inside(const int2* cells, int nc, const int (&lo)[3],
                                            const int (&hi)[3], const P4<float>* pos, int self,
                                            float xi, float yi, float zi, float R, E&& hit) {
    const float R2 = R * R, cl = 1.f / (float)nc, R2m = R2 * 1.0001f;
    for (int cz = lo[2]; cz <= hi[2]; ++cz) {
        const float gz = fmaxf(fmaxf((float)cz * cl - zi, zi - (float)(cz + 1) * cl), 0.f);
        const float gz2 = gz * gz;
        if (gz2 > R2m) continue;
        for (int cy = lo[1]; cy <= hi[1]; ++cy) {
            const float gy = fmaxf(fmaxf((float)cy * cl - yi, yi - (float)(cy + 1) * cl), 0.f);
            const float gzy2 = gz2 + gy * gy;
            if (gzy2 > R2m) continue;
            const int2* row = cells + (cz * nc + cy) * nc;
            // the ranges of up to three cells of the row in flight together
            for (int x0 = lo[0]; x0 <= hi[0]; x0 += 3) {
                int2 ses[3];
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                    const int cx = x0 + u;
                    const float gx = fmaxf(fmaxf((float)cx * cl - xi, xi - (float)(cx + 1) * cl), 0.f);
                    ses[u] = make_int2(0, 0);
                    if (cx <= hi[0] && !(gzy2 + gx * gx > R2m)) ses[u] = row[cx];
                }
#pragma unroll 1
                for (int c = 0; c < 3; ++c) {
                    const int2 se = c == 0 ? ses[0] : (c == 1 ? ses[1] : ses[2]);
                    for (int j0 = se.x; j0 < se.y; j0 += 4) {
                        P4<float> q[4];
                        float r2[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) q[u] = pos[j0 + u];
#pragma unroll
                        for (int u = 0; u < 4; ++u) r2[u] = sep2(q[u].x - xi, q[u].y - yi, q[u].z - zi);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            hit(j0 + u, r2[u], r2[u] < R2 && j0 + u < se.y && j0 + u != self);
                        }
                    }
                }
            }
        }
    }
}

// Cells lo..hi of the window [x - R, x + R]; true when every lane's lies
// inside its box (what scan_inside asks for).
__device__ __forceinline__ bool warp_inside(const BoxInfo& bx, const P4<float>& me, float R, int (&lo)[3],
                                            int (&hi)[3]) {
    bool in = R >= 0.f && !wide(R, bx) && 2.f * R + 2.f / (float)bx.nc < 0.5f;
    const float c3[3] = {me.x, me.y, me.z};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = (int)floorf((c3[a] - R) * (float)bx.nc - 1e-3f);
        hi[a] = (int)floorf((c3[a] + R) * (float)bx.nc + 1e-3f);
        in = in && c3[a] >= 0.f && c3[a] <= 1.f && lo[a] >= 0 && hi[a] < bx.nc;
    }
    return __all_sync(__activemask(), in);
}

// The loops have no branch a candidate, an entry or a neighbour: a candidate
// is written at the cache's end and overwritten by the next unless it counts,
// and the sums advance by selection.  Some lane of a warp takes nearly every
// such branch, so it saved nothing and cost its reconvergence: 128^3 919 us
// with the branches, 871 without those of the scan, 855 of the list, 820 of
// the sums, 803 with the last group's unused entries filled up.  Neither
// fewer steps (two neighbouring cells as one range: 853) nor the next
// candidates loaded ahead (925 against 919) gave anything.
template <int kCache, bool kInside>
__global__ void __launch_bounds__(kOneBlock, 10)
    k_density_one(int N, Sorted<float> s, Grid g, KParams p, unsigned* nbr,
                  int* ncount, int* iters, DevStatus* st,
                  const int* list, const int* nlist, int* defer,
                  int* ndefer) {
    after_previous();
    __shared__ float c_r2[kCache + 1][kOneBlock];
    __shared__ unsigned c_j[kCache + 1][kOneBlock];
    const int t = threadIdx.x;
    int i = blockIdx.x * kOneBlock + t;
    if (list) {  // the particles of an index list only (hierarchical steps)
        if (i >= *nlist) return;
        i = list[i];
    } else if (i >= N) {
        return;
    }
    const BoxInfo bx = g.boxes[s.box[i]];
    const P4<float> me = s.pos[i];
    bool bad;
    float H = h_start<float>(s.h[i], bx, p, bad);
    if (bad) set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, s.id[i]);
    float Rc = dens_cache_radius<float>(H, p);
    int ncache = 0;
    // the cache of the starting H, scanned before the iteration (few live values
    // here).  kInside: a warp with every window inside the box takes the plain
    // scan.
    int lo[3], hi[3];
    bool in = false;
    if constexpr (kInside) in = warp_inside(bx, me, Rc, lo, hi);
    // a cell so full that one thread would walk it while its warp waits: its
    // particles are left to k_density_warp, whose lanes share it (64^3 with 4096
    // particles in one cell: 6.2 ms one thread each, 1.3 so; 32768 in one: 558 and
    // 55).  Looking at every cell of the window as well costs 1 to 2 % of the pass.
    const int2 own = g.cells[bx.cell_off + (cell_at(me.z, bx.nc) * bx.nc + cell_at(me.y, bx.nc)) * bx.nc + cell_at(me.x, bx.nc)];
    if (own.y - own.x > kCrowdCell && in_box(me)) {
        ncache = kCache + 1;
    } else if (in) {
        scan_inside(g.cells + bx.cell_off, bx.nc, lo, hi, s.pos, i, me.x, me.y, me.z, Rc,
                                    [&](int j, float r2, bool h) {
                                        const int k = min(ncache, kCache);
                                        c_r2[k][t] = r2;
                                        c_j[k][t] = (unsigned)j;
                                        ncache += h;
                                    });
    } else if (to_warp(Rc, bx, me)) {
        ncache = kCache + 1;
    } else if constexpr (kInside) {
        ncache = dens_fill<kCache>(g, bx, s.pos, i, me.x, me.y, me.z, Rc, c_r2, c_j, t);
    } else {
        const float R2 = Rc * Rc;
        for_candidates<float>(g, bx, s.pos, i, me.x, me.y, me.z, Rc, [&](int j, float r2, bool ok) {
            const int k = min(ncache, kCache);
            c_r2[k][t] = r2;
            c_j[k][t] = (unsigned)j;
            ncache += ok && r2 < R2;
        });
    }
    float Hev = H, Sv = 0.f, sdv = 0.f;
    HIter<float> b;
    bool conv = false;
    int it;
    for (it = 1; it <= p.max_iter; ++it) {
        if (H > Rc) {  // grown past the cache radius: rescan
            Rc = dens_cache_radius<float>(H, p);
            ncache = to_warp(Rc, bx, me) ? kCache + 1 : dens_fill<kCache>(g, bx, s.pos, i, me.x, me.y, me.z, Rc, c_r2, c_j, t);
        }
        if (ncache > kCache) {  // left to k_density_warp
            defer[atomicAdd(ndefer, 1)] = i;
            return;
        }
        const float H2 = H * H, iH = 1.f / H;
        Acc sw;
        sdv = 0.f;
#pragma unroll
        for (int u = 0; u < 3; ++u) c_r2[min(ncache + u, kCache)][t] = 1e30f;  // (fills up the last four)
        for (int k0 = 0; k0 < ncache; k0 += 4) {  // four entries' terms at a time, added in order
            float r2[4], w[4], x[4], y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                r2[u] = c_r2[k0 + u][t];
                dens_terms2(dist(r2[u]) * iH, w[u], x[u], y[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool h = r2[u] < H2;
                Acc a = sw;
                a.add(w[u]);
                const float d = fmaf(y[u], x[u], sdv);
                sw.s = h ? a.s : sw.s;
                sw.c = h ? a.c : sw.c;
                sdv = h ? d : sdv;
            }
        }
        Sv = sw.fvalue();
        Hev = H;
        if (h_step(b, H, Sv, sdv, p, it == p.max_iter)) {
            conv = true;
            break;
        }
    }
    if (it > p.max_iter) it = p.max_iter;
    const float H2 = Hev * Hev;
    int cnt = 0;
    // list of the returned H, in scan order, gathered at the cache's front and
    // written four slots at a time (512 contiguous bytes a warp; slot by slot
    // the pass took 30 us more at 128^3)
    for (int k = 0; k < ncache; ++k) {
        c_j[cnt][t] = c_j[k][t];  // (overwritten unless it counts)
        cnt += c_r2[k][t] < H2;
    }
    for (int k = 0; k < min(cnt, p.cap); k += 4)
        *reinterpret_cast<uint4*>(nbr + lslot(k, i, N)) =
            make_uint4(c_j[k][t], c_j[k + 1][t], c_j[k + 2][t], c_j[k + 3][t]);
    s.h[i] = Hev;
    s.n[i] = n_of(Sv, Hev);
    if (s.sd) s.sd[i] = sdv;
    iters[i] = it;
    ncount[i] = cnt;
    if (!conv) {
        set_status(st, GZ_S_HCONV, GZ_C_HCONV, s.id[i]);
        if (b.clamped) atomicOr(&st->bits, GZ_S_HLIM);
    }
    if (cnt > p.cap) set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, s.id[i]);
}

// The particles k_density deferred (more candidates within 1.05 H than its
// cache holds): one warp per particle, the same iteration.  The candidates
// within 1.05 H are gathered once into a warp's cache of kWarpCache entries
// (in scan order); later evaluations and the list read only that.  A particle
// with more of them scans the cells at every evaluation.  Grid-stride over
// the deferred list, whose length only the device knows.
// FP32: up to kDensCache entries, which another form could hold, the sums run as
// in group_eval (the lanes form the terms of 32 entries, then every lane adds
// those with r < H in order), so which form iterates a particle does not change
// its H and n; the derivative sum kept for the adjoint is a compensated one.
// More entries are nobody else's: each lane sums its own and the lanes' sums are
// added up in FP64 (one chain of 400 terms leaves 2.6e-7 of the derivative sum,
// the lanes 3e-8).  FP64: the lanes' sums of group_eval.
constexpr int kWarpDensBlock = 64;
constexpr int kWarpCache = 512;

// sd: for the iteration; sdk: to keep.
__device__ __forceinline__ void warp_eval(int lane, int n, const float* r2, float* tw, float* tx, float* ty, float H,
                                          float& S, float& sd, float& sdk) {
    const float H2 = H * H, iH = 1.f / H;
    if (n > kDensCache) {
        Acc w;
        float d = 0.f;
        for (int k = lane; k < n; k += 32)
            if (r2[k] < H2) {
                float t, x, y;
                dens_terms2(dist(r2[k]) * iH, t, x, y);
                w.add(t);
                d = fmaf(y, x, d);
            }
        S = (float)group_add<32>(0xffffffffu, (double)w.s - (double)w.c);
        sd = sdk = (float)group_add<32>(0xffffffffu, (double)d);
        return;
    }
    Acc sw, sk;
    sd = 0.f;
    for (int k0 = 0; k0 < n; k0 += 32) {
        const int k = k0 + lane;
        const float q = k < n ? r2[k] : 1e30f;
        const bool in = q < H2;
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (in) {  // the hits of these 32, close together in order
            const int at = __popc(m & ((1u << lane) - 1u));
            dens_terms2(dist(q) * iH, tw[at], tx[at], ty[at]);
        }
        __syncwarp();
        const int hits = __popc(m);
#pragma unroll 4
        for (int s = 0; s < hits; ++s) {
            sw.add(tw[s]);
            sd = fmaf(ty[s], tx[s], sd);
            sk.add(__fmul_rn(ty[s], tx[s]));
        }
        __syncwarp();
    }
    S = sw.fvalue();
    sdk = sk.fvalue();
}
__device__ __forceinline__ void warp_eval(int lane, int n, const double* r2, double*, double*, double*, double H,
                                          double& S, double& sd, double& sdk) {
    // (lane l's four-entry stride as in group_eval: lanes 4 m + c add class c)
    const double iH = 1.0 / H;
    double a = 0.0, b = 0.0;
    if (lane < kLanes) {
        for (int k = lane; k < n; k += kLanes) {
            double w, d;
            dens_terms2(sqrt(r2[k]) * iH, w, d);
            a += w;
            b += d;
        }
    }
    a = group_add<kLanes>(0xffffffffu, a);
    b = group_add<kLanes>(0xffffffffu, b);
    S = 2.0 * __shfl_sync(0xffffffffu, a, 0);
    sd = sdk = 6.0 * __shfl_sync(0xffffffffu, b, 0);
}

// An evaluation straight from the cells (more candidates than the warp's cache
// holds), the lanes' sums added up.
template <typename T>
__device__ __noinline__ void warp_eval_cells(const Grid& g, const BoxInfo& bx, const P4<T>* pos, int i,
                                             const P4<T>& me, int lane, T H, T& S, T& sd) {
    const T H2 = H * H, iH = T(1) / H;
    double a = 0.0, b = 0.0;
    for_candidates_lanes<T>(g, bx, pos, i, me.x, me.y, me.z, H, lane, [&](int, T, T, T, T r2) {
        if (r2 < H2) {
            if constexpr (sizeof(T) == 4) {
                float w, x, y;
                dens_terms2(dist(r2) * iH, w, x, y);
                a += (double)w;
                b += (double)(x * y);
            } else {
                double w, d;
                dens_terms2(sqrt(r2) * iH, w, d);
                a += 2.0 * w;
                b += 6.0 * d;
            }
        }
    });
    S = (T)group_add<32>(0xffffffffu, a);
    sd = (T)group_add<32>(0xffffffffu, b);
}

template <typename T>
__global__ void __launch_bounds__(kWarpDensBlock)
    k_density_warp(int N, Sorted<T> s, Grid g, KParams p, unsigned* nbr,
                   int* ncount, int* iters, DevStatus* st,
                   const int* defer, const int* ndefer) {
    after_previous();
    constexpr unsigned full = 0xffffffffu;
    __shared__ T w_r2[kWarpDensBlock / 32][kWarpCache];
    __shared__ unsigned w_j[kWarpDensBlock / 32][kWarpCache];
    __shared__ T w_t[kWarpDensBlock / 32][3][32];
    const int lane = threadIdx.x & 31;
    T *t_w = w_t[threadIdx.x >> 5][0], *t_x = w_t[threadIdx.x >> 5][1], *t_y = w_t[threadIdx.x >> 5][2];
    T* c_r2 = w_r2[threadIdx.x >> 5];
    unsigned* c_j = w_j[threadIdx.x >> 5];
    const int warps = gridDim.x * (kWarpDensBlock / 32);
    const int nd = *ndefer;
    for (int w = blockIdx.x * (kWarpDensBlock / 32) + (threadIdx.x >> 5); w < nd; w += warps) {
        const int i = defer[w];
        const BoxInfo bx = g.boxes[s.box[i]];
        const P4<T> me = s.pos[i];
        bool bad;  // (flagged by k_density)
        T H = h_start<T>(s.h[i], bx, p, bad);
        T Rc = T(-1), Hev = H, Sv = T(0), sdv = T(0), sdk = T(0);
        int ncache = 0, it;
        HIter<T> b;
        bool conv = false;
        for (it = 1; it <= p.max_iter; ++it) {
            if (!(H <= Rc)) {
                Rc = dens_cache_radius<T>(H, p);
                __syncwarp();
                ncache = for_hits_lanes_ordered<T>(g, bx, s.pos, i, me.x, me.y, me.z, Rc, Rc * Rc, lane,
                                                   [&](int k, int j, T r2) {
                                                       if (k < kWarpCache) {
                                                           c_r2[k] = r2;
                                                           c_j[k] = (unsigned)j;
                                                       }
                                                   });
                __syncwarp();
            }
            if (ncache <= kWarpCache)
                warp_eval(lane, ncache, c_r2, t_w, t_x, t_y, H, Sv, sdv, sdk);
            else {
                warp_eval_cells(g, bx, s.pos, i, me, lane, H, Sv, sdv);
                sdk = sdv;
            }
            Hev = H;
            if (h_step(b, H, Sv, sdv, p, it == p.max_iter)) {
                conv = true;
                break;
            }
        }
        if (it > p.max_iter) it = p.max_iter;
        // list of the returned H, in the order a thread's scan writes it
        const T H2 = Hev * Hev;
        int cnt = 0;
        if (ncache <= kWarpCache) {
            for (int k0 = 0; k0 < ncache; k0 += 32) {
                const int k = k0 + lane;
                const bool in = k < ncache && c_r2[k] < H2;
                const unsigned m = __ballot_sync(full, in);
                const int slot = cnt + __popc(m & ((1u << lane) - 1u));
                if (in && slot < p.cap) store_slot(nbr + lslot(slot, i, N), c_j[k]);
                cnt += __popc(m);
            }
        } else {
            cnt = for_hits_lanes_ordered<T>(g, bx, s.pos, i, me.x, me.y, me.z, Hev, H2, lane, [&](int k, int j, T) {
                if (k < p.cap) store_slot(nbr + lslot(k, i, N), (unsigned)j);
            });
        }
        if (lane == 0) {
            s.h[i] = Hev;
            s.n[i] = n_of(Sv, Hev);
            if (s.sd) s.sd[i] = sdk;
            iters[i] = it;
            ncount[i] = cnt;
            if (!conv) {
                set_status(st, GZ_S_HCONV, GZ_C_HCONV, s.id[i]);
                if (b.clamped) atomicOr(&st->bits, GZ_S_HLIM);
            }
            if (cnt > p.cap) set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, s.id[i]);
        }
        __syncwarp();
    }
}

// Neighbour lists N_i = {j : r_ij < H_i} for given H (O3).  only_over > 0:
// only the particles whose count exceeds it (lists a checkpoint kept up to
// that many slots; the others are restored from it).
// FP32, large launches: one thread per particle with the density pass's scan.
// Bound like it by the chain range -> candidates through L1 and L2, and by its
// own scattered stores: the first kStage neighbours are gathered in shared
// memory and written four slots at a time.  75^3 particles: 124 us (slot by
// slot 138, and 150 with the periodic shifts in every window); kStage = 40
// leaves less of L1 (127), 16 and 24 send more to the slow stores (130..137).
// Four lanes a particle take 201 there, so the line to the form below is the
// density pass's.
constexpr int kGivenBlock = 128, kStage = 32;
template <bool kInside>
__global__ void __launch_bounds__(kGivenBlock, 8)
    k_lists_one(int N, Sorted<float> s, Grid g, KParams p, unsigned* nbr, int* ncount,
                DevStatus* st, int only_over) {
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    if (only_over > 0 && ncount[i] <= only_over) return;
    const BoxInfo bx = g.boxes[s.box[i]];
    const float H = s.h[i], H2 = H * H;
    const P4<float> me = s.pos[i];
    unsigned* L = nbr + lslot(0, i, N);
    int c = 0;
    const int t = threadIdx.x;
    __shared__ unsigned c_j[kStage][kGivenBlock];
    auto hit = [&](int j, float, bool h) {
        if (!h) return;
        if (c < kStage)
            c_j[c][t] = (unsigned)j;
        else if (c < p.cap)
            store_slot(L + lcol(c, N), (unsigned)j);
        ++c;
    };
    int lo[3], hi[3];
    bool in = false;
    if constexpr (kInside) in = warp_inside(bx, me, H, lo, hi);
    if (in)
        scan_inside(g.cells + bx.cell_off, bx.nc, lo, hi, s.pos, i, me.x, me.y, me.z, H, hit);
    else
        for_candidates<float>(g, bx, s.pos, i, me.x, me.y, me.z, H, [&](int j, float r2, bool ok) {
            hit(j, r2, ok && r2 < H2);
        });
    const int most = min(min(c, kStage), p.cap);
    for (int k = 0; k < most; k += 4)
        *reinterpret_cast<uint4*>(L + lcol(k, N)) = make_uint4(c_j[k][t], c_j[k + 1][t], c_j[k + 2][t], c_j[k + 3][t]);
    ncount[i] = c;
    if (c > p.cap) set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, s.id[i]);
}

// Small launches and FP64: four lanes per particle.
template <typename T>
__global__ void __launch_bounds__(kDensBlock)
    k_lists(int N, Sorted<T> s, Grid g, KParams p, unsigned* nbr, int* ncount,
            DevStatus* st, int only_over) {
    after_previous();
    const int gl = threadIdx.x % kLanes, i = (blockIdx.x * kDensBlock + threadIdx.x) / kLanes;
    const unsigned gm = group_mask<kLanes>();
    if (i >= N) return;
    if (only_over > 0 && ncount[i] <= only_over) return;
    const P4<T> me = s.pos[i];
    unsigned* L = nbr + lslot(0, i, N);
    const int c = group_scan<T, kLanes, true>(g, g.boxes[s.box[i]], s.pos, i, me.x, me.y, me.z, s.h[i], gl, gm, 1 << 30,
                                              [&](int k, int j) {
                                                  if (k < p.cap) store_slot(L + lcol(k, N), (unsigned)j);
                                              });
    if (gl != 0) return;
    ncount[i] = c;
    if (c > p.cap) set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, s.id[i]);
}

// Work of the cell scan at the converged H: per particle, the candidates a
// scan of radius 1.05 H (the density cache's) tests, those inside 1.05 H and
// those inside H; summed over the particles (out[0..2]).
template <typename T>
__global__ void __launch_bounds__(128)
    k_scan_stats(int N, Sorted<T> s, Grid g, KParams p, unsigned long long* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long v[3] = {0, 0, 0};
    if (i < N) {
        const BoxInfo bx = g.boxes[s.box[i]];
        const P4<T> me = s.pos[i];
        const T Ht = s.h[i];
        const T R = dens_cache_radius<T>(Ht, p);
        const T R2 = R * R, H2 = Ht * Ht;
        for_candidates<T>(g, bx, s.pos, i, me.x, me.y, me.z, R, [&](int, T r2, bool ok) {
            v[0] += ok;
            v[1] += ok && r2 < R2;
            v[2] += ok && r2 < H2;
        });
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        unsigned long long x = v[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(out + k, x);
    }
}

}  // namespace

static Grid grid_of(const Ctx& c) {
    Grid g;
    g.boxes = c.boxes;
    g.cells = c.cells;
    return g;
}

template <typename T>
cudaError_t run_density(Ctx& c, const int* list, const int* nlist, int n) {
    if (!list) n = c.N;
    if (n < 1) return cudaSuccess;
    const Sorted<T> sv = sorted_view<T>(c);
    // particles with more candidates within 1.05 H than their cache holds are
    // iterated by a warp each.  k_density_one: 40 entries (the largest count
    // seen on the workloads with N_ngb = 32) for boxes of 32^3 particles or
    // more, 48 for smaller ones, whose strong contrasts overflow 40 more often
    long long min_count = c.N;
    int min_nc = 1 << 30;
    for (const BoxInfo& b : c.hboxes) {
        min_count = std::min(min_count, (long long)b.count);
        min_nc = std::min(min_nc, b.nc);
    }
    if (c.grid_count > 0) min_count = c.grid_count;  // a subdomain: as the whole box
    const int asked = c.params.density_cache, ccap = asked > 0 ? asked : kDensCache;
    const int tcap = asked > 0 ? asked : (min_count >= 32 * 32 * 32 ? 40 : 48);
    c.launches += 2;
    auto one = [&](auto kernel) {
        launch_next(c, kernel, blocks(n, kOneBlock), kOneBlock, c.N, sv, grid_of(c), kparams(c), c.nbr, c.ncount,
                    c.iters, c.status, list, nlist, c.defer,
                    c.ndefer);
    };
    bool done = false;
    if constexpr (std::is_same<T, float>::value) {
        if (n >= kThreadMin) {
            const bool inside = min_nc >= kInsideMin;
            if (tcap == 40)
                inside ? one(k_density_one<40, true>) : one(k_density_one<40, false>);
            else
                inside ? one(k_density_one<48, true>) : one(k_density_one<48, false>);
            done = true;
        }
    }
    auto group = [&](auto kernel, int lanes) {
        launch_next(c, kernel, blocks(n, kDensBlock / lanes), kDensBlock, c.N, sv, grid_of(c), kparams(c), c.nbr,
                    c.ncount, c.iters, c.status, list, nlist,
                    c.defer, c.ndefer, ccap);
    };
    if constexpr (std::is_same<T, float>::value) {
        if (!done && n < kWideMax) {
            group(k_density<T, kWideLanes>, kWideLanes);
            done = true;
        }
    }
    if (!done) group(k_density<T, kLanes>, kLanes);
    // as many warps as fit: each waits on its own loads (Sedov 64^3 late in the
    // run, the whole pass: 4 blocks an SM 509 us, 8 409, 24 395)
    const int wb = std::max(1, std::min(blocks(n, kWarpDensBlock / 32), 152 * 24));
    launch_next(c, k_density_warp<T>, wb, kWarpDensBlock, c.N, sv, grid_of(c), kparams(c), c.nbr, c.ncount,
                c.iters, c.status, c.defer, c.ndefer);
    return cudaGetLastError();
}

// kept > 0: only the lists longer than that (their first slots are there already).
template <typename T>
cudaError_t run_build_lists(Ctx& c, int kept) {
    c.launches += 1;
    const Sorted<T> sv = sorted_view<T>(c);
    if constexpr (std::is_same<T, float>::value) {
        if (c.N >= kThreadMin) {
            int min_nc = 1 << 30;
            for (const BoxInfo& b : c.hboxes) min_nc = std::min(min_nc, b.nc);
            auto one = [&](auto kernel) {
                launch_next(c, kernel, blocks(c.N, kGivenBlock), kGivenBlock, c.N, sv, grid_of(c), kparams(c), c.nbr,
                            c.ncount, c.status, kept);
            };
            min_nc >= kInsideMin ? one(k_lists_one<true>) : one(k_lists_one<false>);
            return cudaGetLastError();
        }
    }
    launch_next(c, k_lists<T>, blocks(c.N, kDensBlock / kLanes), kDensBlock, c.N, sv, grid_of(c), kparams(c), c.nbr,
                c.ncount, c.status, kept);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_scan_stats(Ctx& c, long long* out_dev) {
    c.launches += 1;
    cudaError_t e = cudaMemsetAsync(out_dev, 0, 3 * sizeof(long long), c.stream);
    if (e != cudaSuccess) return e;
    k_scan_stats<T><<<blocks(c.N, 128), 128, 0, c.stream>>>(c.N, sorted_view<T>(c), grid_of(c), kparams(c),
                                                             (unsigned long long*)out_dev);
    return cudaGetLastError();
}
template cudaError_t run_scan_stats<float>(Ctx&, long long*);
template cudaError_t run_scan_stats<double>(Ctx&, long long*);


#define GZ_INST(T)                                                            \
    template cudaError_t run_density<T>(Ctx&, const int*, const int*, int);   \
    template cudaError_t run_build_lists<T>(Ctx&, int);
GZ_INST(float)
GZ_INST(double)
#undef GZ_INST

}  // namespace gz
