// Hydro passes of the MFM step in sorted particle order (steps S2-S6).
// One thread per particle; neighbour lists are stored in groups of four
// slots across the particles (lslot), so a warp reads one group of its lists
// as contiguous bytes.  Every pair quantity that mixes both particles of a
// pair is either symmetric in its operands or evaluated in one fixed order of
// the pair (pair_order), so both particles get bitwise-opposite
// contributions (no atomics on rates).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "gz_device.cuh"
#include "gz_launch.cuh"

namespace gz {

namespace {

inline int blocks(int n, int t) { return (n + t - 1) / t; }

// Reverse pairs (O10): j in N_i with r_ij >= H_j is appended to j's list.
// Reads the packed positions, whose w component is the converged H.  Launches
// under kRevSplit particles have eight threads a particle (k_reverse_split),
// larger ones one (k_reverse, 32 registers: with the four positions of a group
// in flight it takes 55, and 178 us at 128^3 instead of 132).  Reverse lists
// with their sort, eight threads / one, us: Sod 16^3 13 / 28, Sod 32^3 15 / 29,
// KH 41^3 19 / 27, Sedov 64^3 39 / 35, turbulence 128^3 252 / 132.
constexpr int kRevGroups = 8, kRevSplit = 150000;
template <typename T>
__device__ __forceinline__ void append_reverse(int i, int j, int N, int rcap, int* rcount,
                                               unsigned* rnbr, const long long* id,
                                               DevStatus* st) {
    const int slot = atomicAdd(&rcount[j], 1);
    if (slot < rcap)
        rnbr[lslot(slot, j, N)] = (unsigned)i;
    else
        set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, id[j]);
}

template <typename T>
__global__ void k_reverse(int N, Sorted<T> s, KParams p, const unsigned* nbr,
                          const int* ncount, int* rcount,
                          unsigned* rnbr, DevStatus* st) {
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const P4<T> me = s.pos[i];
    const T xim1 = me.x - T(1), yim1 = me.y - T(1), zim1 = me.z - T(1);
    const int cnt = min(ncount[i], p.cap);
    const unsigned* L = nbr + 4 * (size_t)i;
    for (int k0 = 0; k0 < cnt; k0 += 4) {
        const uint4 jj = col4_once(L, k0, N);
        const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (k0 + u >= cnt) break;
            const int j = (int)js[u];
            const P4<T> q = s.pos[j];
            const T dx = mi_diff(q.x, me.x, xim1), dy = mi_diff(q.y, me.y, yim1),
                    dz = mi_diff(q.z, me.z, zim1);
            if (!less_(sep2(dx, dy, dz), q.w * q.w)) append_reverse<T>(i, j, N, p.rcap, rcount, rnbr, s.id, st);
        }
    }
}

// Thread (i, y) takes list groups y, y + kRevGroups, ... of particle i, the four
// partners' positions in flight together; most threads do one group.
template <typename T>
__global__ void __launch_bounds__(32 * kRevGroups)
    k_reverse_split(int N, Sorted<T> s, KParams p, const unsigned* nbr,
                    const int* ncount, int* rcount, unsigned* rnbr,
                    DevStatus* st) {
    after_previous();
    const int i = blockIdx.x * 32 + threadIdx.x;
    if (i >= N) return;
    const int cnt = min(ncount[i], p.cap);
    if (4 * (int)threadIdx.y >= cnt) return;
    const P4<T> me = s.pos[i];
    const unsigned* L = nbr + 4 * (size_t)i;
    for (int k0 = 4 * threadIdx.y; k0 < cnt; k0 += 4 * kRevGroups) {
        const uint4 jj = col4_once(L, k0, N);
        const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
        P4<T> q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            q[u] = me;
            if (k0 + u < cnt) q[u] = s.pos[js[u]];
        }
        T dx[4], dy[4], dz[4];
        offsets4(q, me.x, me.y, me.z, me.x - T(1), me.y - T(1), me.z - T(1), dx, dy, dz);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k0 + u < cnt && !less_(sep2(dx[u], dy[u], dz[u]), q[u].w * q[u].w))
                append_reverse<T>(i, (int)js[u], N, p.rcap, rcount, rnbr, s.id, st);
    }
}

// Orders each reverse list by sorted index so the flux sums are deterministic:
// up to eight entries (most lists) in registers, each placed by the number of
// smaller ones; longer ones by insertion.
__global__ void k_sort_rev(int N, const int* rcount, unsigned* rnbr,
                           int rcap) {
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int n = min(rcount[i], rcap);
    if (n < 2) return;
    unsigned* L = rnbr + 4 * (size_t)i;
    if (n <= 8) {
        const uint4 a = *reinterpret_cast<const uint4*>(L);
        uint4 b = make_uint4(0, 0, 0, 0);
        if (n > 4) b = *reinterpret_cast<const uint4*>(L + lcol(4, N));
        const unsigned v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k >= n) break;
            int at = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) at += q < n && v[q] < v[k];
            L[lcol(at, N)] = v[k];
        }
        return;
    }
    insert_sort(L, n, N);
}
// The same with eight lanes a list, for launches under kRevSplit particles (Sod
// 16^3, late in the run: one thread a list took 11 us, half of it waiting on
// the few lists of more than eight).
__global__ void __launch_bounds__(kListBlock) k_sort_rev_lanes(int N, const int* rcount,
                                                               unsigned* rnbr, int rcap) {
    after_previous();
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) / kListLanes;
    if (i < N) sort_list(rnbr + 4 * (size_t)i, min(rcount[i], rcap), N);
}

// O5 primitives: rho = m n, P = (gamma - 1) rho u, c = sqrt(gamma P / rho); and
// what the passes after it count from zero (every one of them follows a
// k_prim): reverse-list counts, CFL minima, u-floor hits.
template <typename T>
__global__ void k_prim(int N, Sorted<T> s, KParams p, DevStatus* st, int* rcount, int nb,
                       unsigned long long* dtmin, int* box_hits) {
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    for (int b = i; b < nb; b += gridDim.x * blockDim.x) {
        dtmin[b] = dbits(INFINITY);
        box_hits[b] = 0;
    }
    if (i >= N) return;
    rcount[i] = 0;
    const T g = (T)p.gamma;
    const T rho = s.m[i] * s.n[i];
    const T P = (g - T(1)) * rho * s.u[i];
    const T c = sqrt(g * P / rho);
    s.rho[i] = rho;
    s.P[i] = P;
    s.c[i] = c;
    s.pos[i].w = s.h[i];
    s.prim[i] = P4<T>{rho, s.vx[i], s.vy[i], s.vz[i]};
    s.prim2[i] = P2<T>{P, c};
    if (!(rho > T(0)) || !(P > T(0)) || !finite_(c) || !finite_(s.vx[i]) || !finite_(s.vy[i]) ||
        !finite_(s.vz[i]))
        set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, s.id[i]);
}

// ---------------------------------------------------------- O6-O9, O13
// Gradients, limiter and packed flux record; optionally the per-particle
// signal-speed step (over N_i and the reverse list) and its per-box minimum.
// Record (32 values): x y z H | 1/H knorm rho P | vx vy vz g0 | g1..g14 | B0..B5
// with knorm = 8/(pi H^3 n^2) so that V_i psi_j(x_i) = knorm * w(r/H).
// Neighbours are read four at a time (one 16-byte load of indices, a group
// ahead, then the packed records of all four) so their loads are in flight
// together.  The pass waits on them half the time and issues the other half;
// instructions a neighbour (one boundary test for four offsets, the kernel
// without its two pieces, min/max as such) took it from 624 to 494 us at 128^3, FP64 at 48^3 894 to
// 627.  Held to 128 registers (4 blocks per SM); at 5 blocks it spills (570 us),
// and with the next group's records loaded ahead (162 registers) it took 598.
// kInfo: also track which particles the limiter's bounds came from and write
// what the adjoint reads (ginfo, lim); without it (a plain forward step) that
// bookkeeping takes no registers or instructions.
// kDt: also the signal-speed step.
template <typename T, bool kInfo, bool kDt>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? (kInfo ? 3 : 4) : 1)
    k_gradients(int N, Sorted<T> s, const unsigned* nbr, const int* ncount,
                const unsigned* rnbr, const int* rcount, KParams p,
                T* rec, double* dti, unsigned long long* dtmin,
                DevStatus* st, T* ginfo, int* lim,
                const int* list, const int* nlist,
                const unsigned char* owned) {
    after_previous();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    bool active;
    if (list) {  // the particles of an index list only (hierarchical steps)
        active = i < *nlist;
        i = active ? list[i] : 0;
    } else {
        active = i < N;
    }
    double dt_i = INFINITY;
    int mybox = 0;
    if (active) {
        mybox = s.box[i];
        const P4<T> me = s.pos[i];
        const T xi = me.x, yi = me.y, zi = me.z, Hi = me.w;
        const T xim1 = xi - T(1), yim1 = yi - T(1), zim1 = zi - T(1);
        const T ni = s.n[i];
        const P4<T> pm = s.prim[i];
        const P2<T> pm2 = s.prim2[i];
        const T Wi[5] = {pm.x, pm.y, pm.z, pm.w, pm2.x};
        const T ci = pm2.y;
        const T iH = T(1) / Hi;
        const T norm = T(8.0 / kPi) * iH * iH * iH / ni, norm2 = T(2) * norm;
        // FP32 steps: the spare slots of a list's last group run through with no
        // weight instead of a branch a slot, 494 -> 473 us at 128^3 (late in
        // the run 549 -> 519); gradients alone (90 us at 75^3) and
        // FP64, bound by its arithmetic (48^3 625 against 645), skip them
        constexpr bool kFlat = sizeof(T) == 4 && kDt && !kInfo;
        T E[6] = {0, 0, 0, 0, 0, 0};
        T Sg[15];
        T fmax[5], fmin[5];
        int kmax[5], kmin[5];  // particles holding the extremes (for the adjoint)
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            fmax[f] = fmin[f] = Wi[f];
            kmax[f] = kmin[f] = i;
            Sg[3 * f] = Sg[3 * f + 1] = Sg[3 * f + 2] = T(0);
        }
        T vmax = T(0);
        bool any = false;
        const int cnt = min(ncount[i], p.cap);
        const unsigned* L = nbr + 4 * (size_t)i;
        uint4 jj = make_uint4(0, 0, 0, 0);
        if (cnt > 0) jj = col4(L, 0, N);
        for (int k0 = 0; k0 < cnt; k0 += 4) {
            const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
            if (k0 + 4 < cnt) jj = col4(L, k0 + 4, N);
            P4<T> q[4], w[4];
            P2<T> w2[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                // (a spare slot reads the particle itself: no weight, no extreme)
                const unsigned j = k0 + u < cnt ? js[u] : (unsigned)i;
                q[u] = s.pos[j];
                w[u] = s.prim[j];
                w2[u] = s.prim2[j];
            }
            T dx4[4], dy4[4], dz4[4];
            offsets4(q, xi, yi, zi, xim1, yim1, zim1, dx4, dy4, dz4);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!kFlat && k0 + u >= cnt) break;
                const T dx = dx4[u], dy = dy4[u], dz = dz4[u];
                const T r2 = max_(sep2(dx, dy, dz), Tiny<T>::sq);
                T r, ir;
                roots_(r2, r, ir);
                // psi (norm applied per pair: applied to the sums, its rounding stays whole
                // in each of them, up to 3 % of the error of B and the gradients, and
                // nothing is faster)
                const T kh = kern_half(r, iH) * norm2;
                const T pdx = kh * dx, pdy = kh * dy, pdz = kh * dz;
                E[0] += pdx * dx;
                E[1] += pdx * dy;
                E[2] += pdx * dz;
                E[3] += pdy * dy;
                E[4] += pdy * dz;
                E[5] += pdz * dz;
                const T Wj[5] = {w[u].x, w[u].y, w[u].z, w[u].w, w2[u].x};
                T df[5];
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    df[f] = Wj[f] - Wi[f];
                    Sg[3 * f] += df[f] * pdx;
                    Sg[3 * f + 1] += df[f] * pdy;
                    Sg[3 * f + 2] += df[f] * pdz;
                    if constexpr (kInfo) {
                        if (Wj[f] > fmax[f]) {
                            fmax[f] = Wj[f];
                            kmax[f] = (int)js[u];
                        }
                        if (Wj[f] < fmin[f]) {
                            fmin[f] = Wj[f];
                            kmin[f] = (int)js[u];
                        }
                    } else {
                        fmax[f] = max_(fmax[f], Wj[f]);
                        fmin[f] = min_(fmin[f], Wj[f]);
                    }
                }
                if constexpr (kDt) {
                    const T vd = dot3(df[1], df[2], df[3], dx, dy, dz);
                    const T vs = ci + w2[u].y - min_(vd * ir, T(0));
                    vmax = k0 + u == 0 ? vs : (k0 + u < cnt ? max_(vmax, vs) : vmax);
                }
            }
        }
        any = cnt > 0;
        // O7: B = E^-1; FP64 re-do of E and its inverse when kappa > kappa_max
        T B[6], det, kap;
        invert_sym<T>(E, B, det, kap);
        T gt[15];
        bool singular;
        if (sizeof(T) == 4 && !(kap <= (T)p.kappa_max)) {
            double E64[6] = {0, 0, 0, 0, 0, 0};
            const double xd = (double)xi, yd = (double)yi, zd = (double)zi;
            const double iHd = 1.0 / (double)Hi;
            const double normd = 8.0 / kPi * iHd * iHd * iHd / (double)ni;
            for (int k = 0; k < cnt; ++k) {
                const P4<T> q = s.pos[L[lcol(k, N)]];
                const double dx = mi_diff((double)q.x, xd, 0.0), dy = mi_diff((double)q.y, yd, 0.0),
                             dz = mi_diff((double)q.z, zd, 0.0);
                const double r = sqrt(sep2(dx, dy, dz));
                const double psi = normd * kern_w(r * iHd);
                E64[0] += psi * dx * dx;
                E64[1] += psi * dx * dy;
                E64[2] += psi * dx * dz;
                E64[3] += psi * dy * dy;
                E64[4] += psi * dy * dz;
                E64[5] += psi * dz * dz;
            }
            double B64[6], det64, kap64;
            invert_sym<double>(E64, B64, det64, kap64);
            atomicOr(&st->bits, GZ_S_KAPPA_FP64);
            atomicAdd(&st->counters[GZ_C_KAPPA_FP64], 1ull);
            singular = !(det64 > 0.0) || !(kap64 <= 1e8);
#pragma unroll
            for (int q = 0; q < 6; ++q) B[q] = (T)B64[q];
#pragma unroll
            for (int f = 0; f < 5; ++f) {
                const double s0 = Sg[3 * f], s1 = Sg[3 * f + 1], s2 = Sg[3 * f + 2];
                gt[3 * f] = (T)(B64[0] * s0 + B64[1] * s1 + B64[2] * s2);
                gt[3 * f + 1] = (T)(B64[1] * s0 + B64[3] * s1 + B64[4] * s2);
                gt[3 * f + 2] = (T)(B64[2] * s0 + B64[4] * s1 + B64[5] * s2);
            }
        } else {
            singular = !(det > T(0)) || !(kap <= T(1e8));
#pragma unroll
            for (int f = 0; f < 5; ++f) {
                const T s0 = Sg[3 * f], s1 = Sg[3 * f + 1], s2 = Sg[3 * f + 2];
                gt[3 * f] = B[0] * s0 + B[1] * s1 + B[2] * s2;
                gt[3 * f + 1] = B[1] * s0 + B[3] * s1 + B[4] * s2;
                gt[3 * f + 2] = B[2] * s0 + B[4] * s1 + B[5] * s2;
            }
        }
        if (singular) {
            set_status(st, GZ_S_SINGULAR, GZ_C_SINGULAR, s.id[i]);
#pragma unroll
            for (int q = 0; q < 6; ++q) B[q] = T(0);
#pragma unroll
            for (int q = 0; q < 15; ++q) gt[q] = T(0);
        }
        // O9 limiter: alpha_f = min_j min(1, beta (f_ext - f_i) / D_j), D_j = g . s_ij d.
        // The numerator is fixed per field and the quotient decreases as D
        // moves away from 0 on its side, so the minimum is taken by the
        // largest positive and the most negative D_j: one division per field
        // and side after the loop instead of one per neighbour
        T Dpos[5] = {T(0), T(0), T(0), T(0), T(0)}, Dneg[5] = {T(0), T(0), T(0), T(0), T(0)};
        int jpos[5] = {-1, -1, -1, -1, -1}, jneg[5] = {-1, -1, -1, -1, -1};
        const T beta = (T)p.beta;
        if (cnt > 0) jj = col4(L, 0, N);
        for (int k0 = 0; k0 < cnt; k0 += 4) {
            const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
            if (k0 + 4 < cnt) jj = col4(L, k0 + 4, N);
            P4<T> q[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                q[u] = s.pos[k0 + u < cnt ? js[u] : (unsigned)i];  // (a spare slot: D = 0, no constraint)
            }
            T dx4[4], dy4[4], dz4[4];
            offsets4(q, xi, yi, zi, xim1, yim1, zim1, dx4, dy4, dz4);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const T Hs = Hi + q[u].w, sij = quot_(Hi, Hs, rcp_(Hs));
                const T ox = sij * dx4[u], oy = sij * dy4[u], oz = sij * dz4[u];
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    const T D = dot3(gt[3 * f], gt[3 * f + 1], gt[3 * f + 2], ox, oy, oz);
                    if constexpr (kInfo) {
                        if (D > Dpos[f]) {
                            Dpos[f] = D;
                            jpos[f] = (int)js[u];
                        }
                        if (D < Dneg[f]) {
                            Dneg[f] = D;
                            jneg[f] = (int)js[u];
                        }
                    } else {
                        Dpos[f] = max_(Dpos[f], D);
                        Dneg[f] = min_(Dneg[f], D);
                    }
                }
            }
        }
        T al[5];
        int jact[5], kact[5];
        T Dact[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            T a = T(1);
            jact[f] = -1;
            kact[f] = i;
            Dact[f] = T(0);
            if (Dpos[f] > T(0)) {
                const T ap = min(T(1), pdiv(beta * (fmax[f] - Wi[f]), Dpos[f]));
                if (ap < a) {
                    a = ap;
                    jact[f] = jpos[f];
                    kact[f] = kmax[f];
                    Dact[f] = Dpos[f];
                }
            }
            if (Dneg[f] < T(0)) {
                const T am = min(T(1), pdiv(beta * (fmin[f] - Wi[f]), Dneg[f]));
                if (am < a) {
                    a = am;
                    jact[f] = jneg[f];
                    kact[f] = kmin[f];
                    Dact[f] = Dneg[f];
                }
            }
            al[f] = a;
        }
        if constexpr (kDt) {
            const int rc = min(rcount[i], p.rcap);
            const unsigned* RL = rnbr + 4 * (size_t)i;
            for (int k0 = 0; k0 < rc; k0 += 4) {
                const uint4 rr = col4(RL, k0, N);
                const unsigned js[4] = {rr.x, rr.y, rr.z, rr.w};
                P4<T> q[4], w[4];
                P2<T> w2[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned j = k0 + u < rc ? js[u] : js[0];
                    q[u] = s.pos[j];
                    w[u] = s.prim[j];
                    w2[u] = s.prim2[j];
                }
                T dx4[4], dy4[4], dz4[4];
                offsets4(q, xi, yi, zi, xim1, yim1, zim1, dx4, dy4, dz4);
#pragma unroll
                for (int u = 0; u < 4; ++u) {  // (a spare slot repeats the first)
                    if (!kFlat && k0 + u >= rc) break;
                    const T ir = rsq_(max_(sep2(dx4[u], dy4[u], dz4[u]), Tiny<T>::sq));
                    const T vd = dot3(w[u].y - Wi[1], w[u].z - Wi[2], w[u].w - Wi[3], dx4[u], dy4[u], dz4[u]);
                    const T vs = ci + w2[u].y - min_(vd * ir, T(0));
                    vmax = any ? max_(vmax, vs) : vs;
                    any = true;
                }
            }
            if (std::is_same<T, float>::value)  // FP32 path: no FP64 cbrt / division per particle
                dt_i = (any && vmax > T(0)) ? (double)(2.f * cbrtf(1.f / (float)ni) / (float)vmax) : INFINITY;
            else
                dt_i = (any && vmax > T(0)) ? 2.0 * cbrt(1.0 / (double)ni) / (double)vmax : INFINITY;
            dti[i] = dt_i;
        }
        if (kInfo && ginfo) {  // what the adjoint of this pass needs (rows 32-byte aligned)
            T G[kGInfo];
#pragma unroll
            for (int q = 0; q < 15; ++q) {
                G[q] = gt[q];
                G[15 + q] = Sg[q];
            }
#pragma unroll
            for (int f = 0; f < 5; ++f) {
                G[30 + f] = al[f];
                G[35 + f] = Dact[f];
            }
            store_row32<kGInfo>(ginfo + (size_t)i * kGInfo, G);
            // the limiting particles: jact[0..4] then kact[0..4], a 40-byte row
            // (8-byte aligned) written as five 8-byte stores
            const int Lv[10] = {jact[0], jact[1], jact[2], jact[3], jact[4],
                                kact[0], kact[1], kact[2], kact[3], kact[4]};
            int2* Lm = reinterpret_cast<int2*>(lim + (size_t)i * 10);
#pragma unroll
            for (int m = 0; m < 5; ++m) Lm[m] = make_int2(Lv[2 * m], Lv[2 * m + 1]);
        }
        // the flux record: one 128-byte (FP32) row, written with 32-byte stores
        T R[kRecord];
        R[0] = xi;
        R[1] = yi;
        R[2] = zi;
        R[3] = Hi;
        R[4] = iH;
        R[5] = norm / ni;
        R[6] = Wi[0];
        R[7] = Wi[4];
        R[8] = Wi[1];
        R[9] = Wi[2];
        R[10] = Wi[3];
#pragma unroll
        for (int q = 0; q < 15; ++q) R[11 + q] = al[q / 3] * gt[q];
#pragma unroll
        for (int q = 0; q < 6; ++q) R[26 + q] = B[q];
        store_rec(rec, i, R);
    }
    if constexpr (kDt) {
        // warp-level minimum per box, one atomic per warp when the warp is in one box;
        // in a subdomain only its owned particles take part
        const unsigned full = 0xffffffffu;
        const bool counts = active && (!owned || owned[s.orig[i]]);
        unsigned long long v = counts ? dbits(dt_i) : dbits(INFINITY);
        const int b0 = __shfl_sync(full, mybox, 0);
        const bool same = __all_sync(full, !active || mybox == b0);
        if (same) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                unsigned long long w = __shfl_xor_sync(full, v, o);
                v = w < v ? w : v;
            }
            if ((threadIdx.x & 31) == 0) atomicMin(&dtmin[b0], v);
        } else if (counts) {
            atomicMin(&dtmin[mybox], v);
        }
    }
}

// Builds flux records from caller-supplied gradients and B (caller order).
// With a list: its particles only, skipping those flagged in skip (the
// inactive partners of a hierarchical substep, whose gradients and B are
// those of their last active time).
template <typename T>
__global__ void k_pack_given(int N, Sorted<T> s, const T* grad, const T* B,
                             T* rec, const int* list,
                             const int* nlist, const unsigned char* skip) {
    after_previous();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (list) {
        if (i >= *nlist) return;
        i = list[i];
        if (skip && skip[i]) return;
    } else if (i >= N) {
        return;
    }
    const unsigned o = s.orig[i];
    const T Hi = s.h[i], ni = s.n[i];
    const T iH = T(1) / Hi;
    T R[kRecord];
    R[0] = s.x[i];
    R[1] = s.y[i];
    R[2] = s.z[i];
    R[3] = Hi;
    R[4] = iH;
    R[5] = T(8.0 / kPi) * iH * iH * iH / ni / ni;
    R[6] = s.rho[i];
    R[7] = s.P[i];
    R[8] = s.vx[i];
    R[9] = s.vy[i];
    R[10] = s.vz[i];
#pragma unroll
    for (int q = 0; q < 15; ++q) R[11 + q] = grad[(size_t)q * N + o];
#pragma unroll
    for (int q = 0; q < 6; ++q) R[26 + q] = B[(size_t)q * N + o];
    store_rec(rec, i, R);
}

template <typename T>
__global__ void k_grad_out(int N, const unsigned* orig, const T* rec,
                           T* grad, T* B) {
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    T R[kRecord];
    load_rec(rec, i, R);
    if (grad)
#pragma unroll
        for (int q = 0; q < 15; ++q) grad[(size_t)q * N + o] = R[11 + q];
    if (B)
#pragma unroll
        for (int q = 0; q < 6; ++q) B[(size_t)q * N + o] = R[26 + q];
}

// Rates of a particle over its pairs N_i then R_i (sum_runs: one thread, or
// kSplit four warps per 32 particles; either reads one list group of adjacent
// particles at a time, so that a warp's partners lie close together).  kMFV:
// the MFV fluxes (O15), which add dm/dt.  kRiem: the MFM face's Riemann solver
// (pair_rates).
constexpr int kFluxBlock = 128;

template <typename T, bool kMFV, int kRiem, bool kSplit>
__global__ void __launch_bounds__(kFluxBlock, kLoadAhead<T, kMFV, kRiem> ? 3 : 1)
    k_fluxes(int N, const T* rec, const long long* sid,
             const int* sbox, const unsigned* nbr,
             const int* ncount, const unsigned* rnbr,
             const int* rcount, KParams p, const double* dt_use,
             double* dpdt, double* dEdt, double* dmdt,
             DevStatus* st) {
    after_previous();
    constexpr int nq = kMFV ? 5 : 4;
    const int it = flux_item<kSplit>();
    if (!kSplit && it >= N) return;
    const int i = min(it, N - 1);  // (kSplit: the last block's spare threads repeat a particle, with no pairs)
    T a[kRecord];
    load_rec(rec, i, a);
    const long long idi = kMFV ? sid[i] : 0;  // (MFV pairs are oriented by id)
    const T hdt = p.hancock ? (T)(0.5 * dt_use[sbox[i]]) : T(0);
    const T gam = (T)p.gamma;
    T ia[5];
    half_inc(a, hdt, gam, ia);
    const int cnt = it < N ? min(ncount[i], p.cap) : 0, rcnt = it < N ? min(rcount[i], p.rcap) : 0;
    int nfall = 0, nneg = 0;
    auto pair = [&](const T(&b)[kRecord], int j, T(&run)[nq]) {
        T dp[3], dE, dm;
        int fl = 0;
        if (pair_rates<T, kMFV, kRiem>(a, b, ia, pair_order<kMFV>(i, j, idi, sid), hdt, gam, dp, dE, dm, fl)) {
            run[0] += dp[0];
            run[1] += dp[1];
            run[2] += dp[2];
            run[3] += dE;
            if constexpr (kMFV) run[4] += dm;
        }
        nfall += fl & 1;
        nneg += (fl >> 1) & 1;
    };
    if constexpr (kSplit) {
        const Totals<2> t = sum_runs_split<T, nq, kPairUnroll<kRiem>>(i, N, rec, nbr, cnt, rnbr, rcnt, pair);
        if (it < N) store_rates_split<nq>(t.v, i, N, dpdt, dEdt, dmdt);
    } else {
        const Totals<nq> t = sum_runs<T, nq, kLoadAhead<T, kMFV, kRiem>, kPairUnroll<kRiem>>(i, N, rec, nbr, cnt, rnbr, rcnt, pair);
        store_rates<nq>(t.v, i, N, dpdt, dEdt, dmdt);
    }
    count_flags(st, nfall, nneg);
}

// dmdt (MFV, O15) non-null: the mass advances too and is written back.
template <typename T>
__global__ void k_update(int N, Sorted<T> s, const double* dpdt,
                         const double* dEdt, const double* dmdt,
                         const double* dt_use, gz_particles out,
                         int* box_hits, DevStatus* st, double* rates_out) {
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = s.orig[i];
    const int b = s.box[i];
    if (rates_out) {  // the step's conserved-variable rates, caller order
        rates_out[o] = dpdt[i];
        rates_out[(size_t)N + o] = dpdt[(size_t)N + i];
        rates_out[2 * (size_t)N + o] = dpdt[2 * (size_t)N + i];
        rates_out[3 * (size_t)N + o] = dEdt[i];
    }
    T x = s.x[i], y = s.y[i], z = s.z[i], vx = s.vx[i], vy = s.vy[i], vz = s.vz[i], u = s.u[i];
    bool mass_ok = true;
    if (dmdt) {
        T m = s.m[i];
        update_one_mfv(m, x, y, z, vx, vy, vz, u, dpdt[i], dpdt[(size_t)N + i],
                       dpdt[2 * (size_t)N + i], dEdt[i], dmdt[i], dt_use[b]);
        ((T*)out.m)[o] = m;
        mass_ok = m > T(0);
    } else {
        update_one(s.m[i], x, y, z, vx, vy, vz, u, dpdt[i], dpdt[(size_t)N + i],
                   dpdt[2 * (size_t)N + i], dEdt[i], dt_use[b]);
    }
    ((T*)out.x)[o] = x;
    ((T*)out.y)[o] = y;
    ((T*)out.z)[o] = z;
    ((T*)out.vx)[o] = vx;
    ((T*)out.vy)[o] = vy;
    ((T*)out.vz)[o] = vz;
    ((T*)out.u)[o] = u;
    ((T*)out.h)[o] = s.h[i];
    if (!(u > T(0))) {
        atomicAdd(&box_hits[b], 1);
        set_status(st, GZ_S_UFLOOR, GZ_C_UFLOOR, -1);
    }
    if (!(mass_ok && finite_(x) && finite_(y) && finite_(z) && finite_(vx) && finite_(vy) &&
          finite_(vz) && finite_(u)))
        set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, s.id[i]);
}

template <typename T>
struct Bits;
template <>
struct Bits<float> {
    typedef unsigned U;
    static constexpr int nbits = 32;
    __device__ static U get(float v) { return __float_as_uint(v); }
    __device__ static float put(U b) { return __uint_as_float(b); }
};
template <>
struct Bits<double> {
    typedef unsigned long long U;
    static constexpr int nbits = 64;
    __device__ static U get(double v) { return (U)__double_as_longlong(v); }
    __device__ static double put(U b) { return __longlong_as_double((long long)b); }
};

// O14 floor: for each box with a hit, the lower median of u at step start
// (radix select on the bit patterns of positive values), then every
// non-positive updated u of the box is set to u_floor_frac * median.
template <typename T>
__global__ void k_ufloor(Sorted<T> s, const BoxInfo* boxes,
                         const int* box_hits, gz_particles out, double frac,
                         const unsigned char* owned, int nown) {
    after_previous();
    typedef typename Bits<T>::U U;
    const int b = blockIdx.x;
    if (box_hits[b] == 0) return;
    const int first = boxes[b].first, count = boxes[b].count;
    // in a subdomain (owned non-null, one box) the median of its owned particles
    __shared__ unsigned hist[256];
    __shared__ U prefix_s;
    __shared__ int k_s;
    U prefix = 0, mask = 0;
    int k = ((owned ? nown : count) - 1) / 2;
    if (k < 0) return;
    for (int shift = Bits<T>::nbits - 8; shift >= 0; shift -= 8) {
        for (int t = threadIdx.x; t < 256; t += blockDim.x) hist[t] = 0;
        __syncthreads();
        for (int e = threadIdx.x; e < count; e += blockDim.x) {
            if (owned && !owned[s.orig[first + e]]) continue;
            const U v = Bits<T>::get(s.u[first + e]);
            if ((v & mask) == prefix) atomicAdd(&hist[(unsigned)((v >> shift) & 255u)], 1u);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int d = 0;
            for (; d < 255; ++d) {
                if (k < (int)hist[d]) break;
                k -= (int)hist[d];
            }
            prefix_s = prefix | ((U)d << shift);
            k_s = k;
        }
        __syncthreads();
        prefix = prefix_s;
        k = k_s;
        mask |= ((U)255u << shift);
        __syncthreads();
    }
    const T fl = (T)(frac * (double)Bits<T>::put(prefix));
    T* u = (T*)out.u;
    for (int e = threadIdx.x; e < count; e += blockDim.x) {
        const int o = first + e;  // caller order and sorted order share box ranges
        if (!(u[o] > T(0))) u[o] = fl;
    }
}

__global__ void k_dt_final(int nb, const unsigned long long* dtmin, double cfl,
                           double dt_fixed, double* dt_use, double* out) {
    after_previous();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const double raw = __longlong_as_double((long long)dtmin[b]);
    const double dt = dt_fixed > 0.0 ? dt_fixed : cfl * raw;
    dt_use[b] = dt;
    if (out) out[b] = dt;
}
__global__ void k_dt_set(int nb, double dt, double* dt_use) {
    after_previous();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nb) dt_use[b] = dt;
}
__global__ void k_dt_out(int nb, const unsigned long long* __restrict__ dtmin, double cfl,
                         double* __restrict__ out) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nb) out[b] = cfl * __longlong_as_double((long long)dtmin[b]);
}

__global__ void k_get_nbrs(int N, const unsigned* __restrict__ orig, const long long* __restrict__ sid,
                           const unsigned* __restrict__ nbr, const int* __restrict__ ncount, int cap_in,
                           int32_t* __restrict__ count_out, int64_t* __restrict__ ids_out, int cap) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    const int c = ncount[i];
    count_out[o] = c;
    if (!ids_out) return;
    const int m = min(min(c, cap_in), cap);
    for (int k = 0; k < cap; ++k)
        ids_out[(size_t)k * N + o] = k < m ? (int64_t)sid[nbr[lslot(k, i, N)]] : (int64_t)-1;
}

// The limiter's choices per particle (sorted-order indices, 10 per particle)
// as particle ids in caller order: rows 0-4 the neighbour whose face bound
// set alpha_f (-1: alpha_f = 1), rows 5-9 the particle holding the extreme.
__global__ void k_get_limiters(int N, const unsigned* __restrict__ orig, const long long* __restrict__ sid,
                               const int* __restrict__ lim, int64_t* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    for (int f = 0; f < 10; ++f) {
        const int j = lim[(size_t)i * 10 + f];
        out[(size_t)f * N + o] = j >= 0 ? (int64_t)sid[j] : (int64_t)-1;
    }
}

__global__ void k_pairs(int N, const int* __restrict__ ncount, const int* __restrict__ rcount,
                        int cap, int rcap, long long* __restrict__ out) {
    long long v = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
        v += min(ncount[i], cap) + min(rcount[i], rcap);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) atomicAdd((unsigned long long*)out, (unsigned long long)v);
}

}  // namespace

cudaError_t run_pair_count(Ctx& c, long long* out_dev) {
    c.launches += 1;
    cudaMemsetAsync(out_dev, 0, sizeof(long long), c.stream);
    k_pairs<<<304, 256, 0, c.stream>>>(c.N, c.ncount, c.rcount, c.cap, c.rcap, out_dev);
    return cudaGetLastError();
}

KParams kparams(const Ctx& c) {
    KParams k;
    k.gamma = c.params.gamma;
    k.ngb = c.params.ngb;
    k.cfl = c.params.cfl;
    k.kappa_max = c.params.kappa_max;
    k.beta = c.params.beta;
    k.u_floor_frac = c.params.u_floor_frac;
    k.h_lim = c.params.h_lim;
    k.hancock = c.params.hancock;
    k.scheme = c.params.scheme;
    k.max_iter = c.params.max_iter;
    const double tn = c.params.tol * c.params.ngb;
    k.dtol = tn;
    k.ftol = (float)tn;
    if ((double)k.ftol > tn) k.ftol = nextafterf(k.ftol, 0.f);
    k.hlimf = (float)c.params.h_lim;
    if ((double)k.hlimf < c.params.h_lim) k.hlimf = nextafterf(k.hlimf, 1.f);
    k.cap = c.cap;
    k.rcap = c.rcap;
    return k;
}

template <typename T>
cudaError_t run_reverse(Ctx& c) {
    c.launches += 2;
    if (c.N < kRevSplit)
        launch_next(c, k_reverse_split<T>, blocks(c.N, 32), dim3(32, kRevGroups), c.N, sorted_view<T>(c), kparams(c),
                    c.nbr, c.ncount, c.rcount, c.rnbr, c.status);
    else
        launch_next(c, k_reverse<T>, blocks(c.N, 256), 256, c.N, sorted_view<T>(c), kparams(c), c.nbr, c.ncount,
                    c.rcount, c.rnbr, c.status);
    if (c.N < kRevSplit)
        launch_next(c, k_sort_rev_lanes, blocks(c.N, kListBlock / kListLanes), kListBlock, c.N, c.rcount, c.rnbr,
                    c.rcap);
    else
        launch_next(c, k_sort_rev, blocks(c.N, 256), 256, c.N, c.rcount, c.rnbr, c.rcap);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_prim(Ctx& c) {
    c.launches += 1;
    launch_next(c, k_prim<T>, blocks(c.N, 256), 256, c.N, sorted_view<T>(c), kparams(c), c.status, c.rcount,
                c.nboxes, (unsigned long long*)c.dt_box, c.box_hits);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_gradients(Ctx& c, bool want_dt, bool with_info, const int* list, const int* nlist, int n) {
    c.launches += 1;
    if (!list) n = c.N;
    if (n < 1) return cudaGetLastError();
    auto go = [&](auto kernel) {
        launch_next(c, kernel, blocks(n, 128), 128, c.N, sorted_view<T>(c), c.nbr, c.ncount, c.rnbr, c.rcount,
                    kparams(c), (T*)c.rec, c.dti, (unsigned long long*)c.dt_box,
                    c.status, with_info ? (T*)c.ginfo : nullptr,
                    with_info ? c.lim : nullptr, list, nlist, c.owned);
    };
    if (with_info)
        want_dt ? go(k_gradients<T, true, true>) : go(k_gradients<T, true, false>);
    else
        want_dt ? go(k_gradients<T, false, true>) : go(k_gradients<T, false, false>);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_pack_given(Ctx& c, const T* grad, const T* B, const int* list, const int* nlist, int n,
                           const unsigned char* skip) {
    c.launches += 1;
    if (list && n < 1) return cudaSuccess;
    launch_next(c, k_pack_given<T>, blocks(list ? n : c.N, 256), 256, c.N, sorted_view<T>(c), grad, B,
                (T*)c.rec, list, nlist, skip);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_grad_out(Ctx& c, T* grad, T* B) {
    c.launches += 1;
    launch_next(c, k_grad_out<T>, blocks(c.N, 256), 256, c.N, c.vals, (const T*)c.rec, grad, B);
    return cudaGetLastError();
}

template <typename T, bool kMFV, int kRiem>
static void launch_fluxes(Ctx& c) {
    auto go = [&](auto kernel, int items) {
        launch_next(c, kernel, blocks(c.N, items), kFluxBlock, c.N, (const T*)c.rec, c.sid, c.sbox, c.nbr, c.ncount,
                    c.rnbr, c.rcount, kparams(c), c.dt_use, c.dpdt,
                    c.dEdt, kMFV ? c.dmdt : nullptr, c.status);
    };
    if (c.N < kFluxSplit)
        go(k_fluxes<T, kMFV, kRiem, true>, 32);
    else
        go(k_fluxes<T, kMFV, kRiem, false>, kFluxBlock);
}

template <typename T>
cudaError_t run_fluxes(Ctx& c) {
    c.launches += 1;
    if (c.params.scheme == GZ_MFV)
        launch_fluxes<T, true, GZ_RIEMANN_HLLC>(c);
    else if (c.params.riemann == GZ_RIEMANN_EXACT)
        launch_fluxes<T, false, GZ_RIEMANN_EXACT>(c);
    else if (c.params.riemann == GZ_RIEMANN_FALLBACK)
        launch_fluxes<T, false, GZ_RIEMANN_FALLBACK>(c);
    else
        launch_fluxes<T, false, GZ_RIEMANN_HLLC>(c);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_update(Ctx& c, gz_particles& p, double* rates_out) {
    c.launches += 2;
    int* hits = c.box_hits;
    launch_next(c, k_update<T>, blocks(c.N, 256), 256, c.N, sorted_view<T>(c), c.dpdt, c.dEdt,
                c.params.scheme == GZ_MFV ? c.dmdt : nullptr, c.dt_use, p,
                hits, c.status, rates_out);
    launch_next(c, k_ufloor<T>, c.nboxes, 1024, sorted_view<T>(c), c.boxes, hits, p,
                c.params.u_floor_frac, c.owned, c.n_owned);
    return cudaGetLastError();
}

// The u floor of O14 alone (after a kick that flagged box_hits).
template <typename T>
cudaError_t run_ufloor(Ctx& c, gz_particles& p) {
    c.launches += 1;
    launch_next(c, k_ufloor<T>, c.nboxes, 1024, sorted_view<T>(c), c.boxes, c.box_hits, p,
                c.params.u_floor_frac, c.owned, c.n_owned);
    return cudaGetLastError();
}

// Rates saved by a forward step (caller order) into the sorted rate arrays.
__global__ void k_rates_in(int N, const unsigned* __restrict__ orig, const double* __restrict__ rates,
                           double* __restrict__ dpdt, double* __restrict__ dEdt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    dpdt[i] = rates[o];
    dpdt[(size_t)N + i] = rates[(size_t)N + o];
    dpdt[2 * (size_t)N + i] = rates[2 * (size_t)N + o];
    dEdt[i] = rates[3 * (size_t)N + o];
}

cudaError_t run_rates_in(Ctx& c, const double* rates) {
    c.launches += 1;
    k_rates_in<<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, c.vals, rates, c.dpdt, c.dEdt);
    return cudaGetLastError();
}

cudaError_t run_dt_finalize(Ctx& c, double dt_fixed, double* dt_used_dev) {
    c.launches += 1;
    launch_next(c, k_dt_final, blocks(c.nboxes, 256), 256, c.nboxes, (const unsigned long long*)c.dt_box, c.params.cfl,
                dt_fixed, c.dt_use, dt_used_dev);
    return cudaGetLastError();
}

cudaError_t run_dt_set(Ctx& c, double dt) {
    c.launches += 1;
    launch_next(c, k_dt_set, blocks(c.nboxes, 256), 256, c.nboxes, dt, c.dt_use);
    return cudaGetLastError();
}

__global__ void k_dt_copy(int nb, const double* __restrict__ dt, double* __restrict__ dt_use) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < nb) dt_use[b] = dt[b];
}

cudaError_t run_dt_copy(Ctx& c, const double* dt) {
    c.launches += 1;
    k_dt_copy<<<blocks(c.nboxes, 256), 256, 0, c.stream>>>(c.nboxes, dt, c.dt_use);
    return cudaGetLastError();
}

// One-box table of a subdomain, written from values passed by value.
__global__ void k_set_box(BoxInfo* boxes, BoxInfo b) {
    if (threadIdx.x == 0 && blockIdx.x == 0) boxes[0] = b;
}

cudaError_t run_set_box(Ctx& c) {
    c.launches += 1;
    k_set_box<<<1, 32, 0, c.stream>>>(c.boxes, c.hboxes[0]);
    return cudaGetLastError();
}

cudaError_t run_dt_out(Ctx& c, double* out) {
    c.launches += 1;
    k_dt_out<<<blocks(c.nboxes, 256), 256, 0, c.stream>>>(c.nboxes, (const unsigned long long*)c.dt_box,
                                                          c.params.cfl, out);
    return cudaGetLastError();
}

cudaError_t run_get_limiters(Ctx& c, const int* lim, int64_t* out) {
    c.launches += 1;
    k_get_limiters<<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, c.vals, c.sid, lim, out);
    return cudaGetLastError();
}

cudaError_t run_get_neighbours(Ctx& c, int32_t* count_out, int64_t* ids_out, int cap) {
    c.launches += 1;
    k_get_nbrs<<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, c.vals, c.sid, c.nbr, c.ncount, c.cap,
                                                       count_out, ids_out, cap);
    return cudaGetLastError();
}

#define GZ_INST(T)                                                   \
    template cudaError_t run_reverse<T>(Ctx&);                                                  \
    template cudaError_t run_prim<T>(Ctx&);                                                     \
    template cudaError_t run_gradients<T>(Ctx&, bool, bool, const int*, const int*, int);      \
    template cudaError_t run_pack_given<T>(Ctx&, const T*, const T*, const int*, const int*, int, \
                                           const unsigned char*);                               \
    template cudaError_t run_grad_out<T>(Ctx&, T*, T*);                                         \
    template cudaError_t run_fluxes<T>(Ctx&);                                                   \
    template cudaError_t run_update<T>(Ctx&, gz_particles&, double*);                          \
    template cudaError_t run_ufloor<T>(Ctx&, gz_particles&);
GZ_INST(float)
GZ_INST(double)
#undef GZ_INST

}  // namespace gz
