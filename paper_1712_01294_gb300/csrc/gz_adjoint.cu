// Adjoint (reverse mode) of the MFM step, hand-written pass by pass.
//
// Conventions, identical to the derivative oracle: neighbour sets and the
// flux pair set are frozen at their forward values; dt is a constant; H is
// the root of f(H; x) = 0 and is differentiated implicitly; the u floor is a
// constant; min / max / clamp pass the adjoint to the branch the forward
// took.  Every pass re-evaluates its forward quantities (nothing per pair is
// stored) and accumulates adjoints by gathering: the thread of particle i
// visits i's pairs and adds only the terms that belong to i, so there are no
// atomics and the result is deterministic.
//
// Adjoint record per particle (working precision, sorted order), kAdj values:
//   0-2 x   3-5 v   6 u   7 m   8 H   9 n   10 rho   11 P   12-26 g (limited)
//   27-32 B (xx xy xz yy yz zz)
#include <algorithm>

#include "gz_device.cuh"
#include "gz_launch.cuh"

namespace gz {

namespace {

inline int blocks(int n, int t) { return (n + t - 1) / t; }

enum : int { AX = 0, AV = 3, AU = 6, AM = 7, AH = 8, AN = 9, ARHO = 10, AP = 11, AG = 12, AB = 27 };

// What the pairs of particle a add up to (pair_adjoint); flux_adj_row turns it
// into a's adjoint row after the last pair, so that nothing that depends on a
// alone is formed per pair.
template <typename T>
struct AdjSums {
    T x[3];   // -dJ/dx_a
    T F[5];   // face value F_a (to the half-step primitives)
    T W[5];   // primitives of a as clamp bounds or in the first-order fallback
    T g[15];  // F_a's gradients
    T B[6];
    T k;      // knorm_a
    T q;      // sum of dJ/dln(1/H_a) through knorm_a w(r/H_a), over knorm_a
    T h;      // H_a through the face position
};

// Adjoint of particle a's share of the pair (a, b).  wp = dpbar_a - dpbar_b
// and wE = dEbar_a - dEbar_b weight the pair's rate contributions.  The
// forward is re-evaluated as pair_rates forms it (its symmetric star state,
// in which v_f drops out), so every branch matches; ia: half_inc of a.
// Divisions are products with the reciprocals the forward takes anyway: FP64
// is bound by its pipe (977 operations a pair where the canonical L/R order,
// v_f and a's own terms were carried through each pair, 3.88 ms at 40^3; a good
// half of that here, 2.20 ms, of which 0.27 ms keep terms from cancelling).
template <typename T>
__device__ __forceinline__ void pair_adjoint(const T (&a)[kRecord], const T (&b)[kRecord], const T (&ia)[5], bool aL,
                                             T hdt, T gam, const T* wp, T wE, AdjSums<T>& s) {
    // ---- forward (same operations as pair_rates)
    const T dx = mi_diff(b[0], a[0], a[0] - T(1));
    const T dy = mi_diff(b[1], a[1], a[1] - T(1));
    const T dz = mi_diff(b[2], a[2], a[2] - T(1));
    const T r2 = max_(sep2(dx, dy, dz), Tiny<T>::sq);
    T r, ir;
    roots_(r2, r, ir);
    T wa, wb, da, db;
    kern_half_d(r, a[4], wa, da);
    kern_half_d(r, b[4], wb, db);
    const T ca = a[5] * wa, cb = b[5] * wb;
    const T* Ba = a + 26;
    const T* Bb = b + 26;
    const T ua[3] = {dot3(Ba[0], Ba[1], Ba[2], dx, dy, dz), dot3(Ba[1], Ba[3], Ba[4], dx, dy, dz),
                     dot3(Ba[2], Ba[4], Ba[5], dx, dy, dz)};
    const T ub[3] = {dot3(Bb[0], Bb[1], Bb[2], dx, dy, dz), dot3(Bb[1], Bb[3], Bb[4], dx, dy, dz),
                     dot3(Bb[2], Bb[4], Bb[5], dx, dy, dz)};
    T A[3];  // (half of the face area vector)
#pragma unroll
    for (int k = 0; k < 3; ++k) A[k] = add_rn(mul_rn(ca, ua[k]), mul_rn(cb, ub[k]));
    const T Aq = sep2(A[0], A[1], A[2]);
    if (!pos_(Aq - Tiny<T>::sq)) return;
    T Ah, iA;
    roots_(Aq, Ah, iA);
    const T n[3] = {A[0] * iA, A[1] * iA, A[2] * iA};
    const T iHs = rcp_(a[3] + b[3]);
    const T sa = a[3] * iHs, sb = b[3] * iHs;
    T Ga[5], Gb[5], Da[5], Db[5], ib[5];
    int ka[5], kb[5];  // clamp sides: 0 inside, -1 at the lower bound, +1 at the upper
    half_inc(b, hdt, gam, ib);
    const T Wa0[5] = {a[6], a[8], a[9], a[10], a[7]};
    const T Wb0[5] = {b[6], b[8], b[9], b[10], b[7]};
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        Da[f] = dot3(a[11 + 3 * f], a[12 + 3 * f], a[13 + 3 * f], dx, dy, dz);
        Db[f] = dot3(b[11 + 3 * f], b[12 + 3 * f], b[13 + 3 * f], dx, dy, dz);
        const T lo = min_(Wa0[f], Wb0[f]), hi = max_(Wa0[f], Wb0[f]);
        const T Fa = face_value(Wa0[f], sa, Da[f], ia[f]), Fb = face_value(Wb0[f], -sb, Db[f], ib[f]);
        ka[f] = less_(Fa, lo) ? -1 : (less_(hi, Fa) ? 1 : 0);
        kb[f] = less_(Fb, lo) ? -1 : (less_(hi, Fb) ? 1 : 0);
        Ga[f] = ka[f] < 0 ? lo : (ka[f] > 0 ? hi : Fa);
        Gb[f] = kb[f] < 0 ? lo : (kb[f] > 0 ? hi : Fb);
    }
    const bool fallback = !(pos_(Ga[0]) && pos_(Ga[4]) && pos_(Gb[0]) && pos_(Gb[4]));
    if (fallback) {
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            Ga[f] = Wa0[f];
            Gb[f] = Wb0[f];
        }
    }
    const T ira = rcp_(Ga[0]), irb = rcp_(Gb[0]);
    const T qa = gam * Ga[4] * ira, qb = gam * Gb[4] * irb;
    const T ica = rsq_(max_(qa, Tiny<T>::sq)), icb = rsq_(max_(qb, Tiny<T>::sq));
    const T cca = mul_rn(qa, ica), ccb = mul_rn(qb, icb);
    const T dv[3] = {Gb[1] - Ga[1], Gb[2] - Ga[2], Gb[3] - Ga[3]};
    const T sv[3] = {Ga[1] + Gb[1], Ga[2] + Gb[2], Ga[3] + Gb[3]};
    const T du = dot3(dv[0], dv[1], dv[2], n[0], n[1], n[2]);
    const T us = dot3(sv[0], sv[1], sv[2], n[0], n[1], n[2]);
    const T e1 = du - ccb, e2 = cca - du;
    const T al = min_(-cca, e1), be = max_(ccb, e2);
    const T ma = mul_rn(Ga[0], al), mb = mul_rn(Gb[0], be);
    const T den = ma - mb, iden = rcp_(den), msum = ma + mb;
    T sc, isc;  // (the scaling of pair_rates)
    pow2_near(den, sc, isc);
    const T mas = ma * sc, mbs = mb * sc, idens = iden * isc;
    const T dP = Gb[4] - Ga[4];
    T num;
    const T psr = star_pressure(Ga[4], Gb[4], dP, du, mas, mbs, mb, idens, num);
    // P_a - P*, P_b - P* without the rounding of P*
    const T cor = num * idens;
    const bool lower = less_(Ga[4], Gb[4]);
    const T Pas = lower ? -cor : -(dP + cor), Pbs = lower ? dP - cor : -cor;
    const T X = fma(-msum, du, T(2) * dP) * iden;
    const T S = T(0.5) * (us + X);
    const bool neg = psr < T(0);
    const T ps = neg ? T(0) : psr;
    const T Am = T(2) * Ah;
    // ---- reverse: J = -ps (wp . A + wE S |A|)
    const T wA = T(2) * dot3(wp[0], wp[1], wp[2], A[0], A[1], A[2]);
    const T wS = wE * S;
    const T b_psr = neg ? T(0) : -fma(wS, Am, wA);
    const T b_h = T(-0.5) * (ps * wE) * Am;  // of us and of X
    // X = num2 iden, psr = num1 idens with num1 = sc (ma Pb - mb Pa - ma mb du),
    // iden = 1 / (ma - mb); b_1 the adjoint of num1, of order b_psr like every
    // product formed with it.  The pressures enter as differences from psr.
    const T b_2 = b_h * iden, b_1 = b_psr * idens;
    T b_Pa = -fma(b_1, mbs, T(2) * b_2), b_Pb = fma(b_1, mas, T(2) * b_2);
    const T b_ma = fma(b_1, fma(-mbs, du, sc * Pbs), -(b_2 * (du + X)));
    const T b_mb = -fma(b_1, fma(mas, du, sc * Pas), b_2 * (du - X));
    T b_du = -fma(msum, b_2, b_1 * (mas * mb));
    // ma = rho_a min(-c_a, du - c_b), mb = rho_b max(c_b, c_a - du); a tie goes to
    // the particle that is L (the derivative oracle's rule).  rho c is
    // sqrt(gamma P rho): half of its logarithm's derivative to each
    T b_ra = b_ma * al, b_rb = b_mb * be;
    T b_ca = T(0), b_cb = T(0);
    const bool own_a = aL ? !less_(e1, -cca) : less_(-cca, e1);
    const bool own_b = aL ? less_(e2, ccb) : !less_(ccb, e2);
    if (own_a) {
        b_ra *= T(0.5);
        b_Pa = fma(T(-0.5) * gam * ica, b_ma, b_Pa);
    } else {
        const T b_al = b_ma * Ga[0];
        b_du += b_al;
        b_cb -= b_al;
    }
    if (own_b) {
        b_rb *= T(0.5);
        b_Pb = fma(T(0.5) * gam * icb, b_mb, b_Pb);
    } else {
        const T b_be = b_mb * Gb[0];
        b_ca += b_be;
        b_du -= b_be;
    }
    // c = sqrt(gamma P / rho), where the other side bounds
    const T ha = T(0.5) * ira * b_ca, hb = T(0.5) * irb * b_cb;
    b_Pa = fma(ha * gam, ica, b_Pa);
    b_ra = fma(-ha, cca, b_ra);
    b_Pb = fma(hb * gam, icb, b_Pb);
    b_rb = fma(-hb, ccb, b_rb);
    const T ea = b_h - b_du, eb = b_h + b_du;
    const T bGa[5] = {b_ra, ea * n[0], ea * n[1], ea * n[2], b_Pa};
    const T bGb[5] = {b_rb, eb * n[0], eb * n[1], eb * n[2], b_Pb};
    // A: n = A/|A| and |A| (A here half the area: the factors of 2 cancel in n)
    const T nn = fma(b_h, us, b_du * du);
    const T b_Am = -(ps * wS);
    const T kA = T(-2) * ps, kN = T(2) * b_Am - nn * iA;
    T bA[3];  // (of the half area vector)
#pragma unroll
    for (int k = 0; k < 3; ++k)
        bA[k] = fma(kA, wp[k], fma(kN, n[k], iA * fma(b_h, sv[k], b_du * dv[k])));
    // fallback and clamps; a bound min / max(W_L, W_R) passes its adjoint to
    // L on a tie (the rule the derivative oracle's where() takes), so the two
    // sides of a pair never both claim it
    T bFa[5], bFb[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        bFa[f] = T(0);
        bFb[f] = T(0);
        if (fallback) {
            s.W[f] += bGa[f];
        } else {
            if (ka[f] == 0) bFa[f] = bGa[f];
            if (kb[f] == 0) bFb[f] = bGb[f];
            if (ka[f] != 0 || kb[f] != 0) {
                const bool lt = less_(Wa0[f], Wb0[f]), gt = less_(Wb0[f], Wa0[f]);
                const bool loA = lt || (aL && !gt), hiA = gt || (aL && !lt);
                if (ka[f] != 0 && (ka[f] < 0 ? loA : hiA)) s.W[f] += bGa[f];
                if (kb[f] != 0 && (kb[f] < 0 ? loA : hiA)) s.W[f] += bGb[f];
            }
        }
    }
    // face states: F_a = W_a + s_a g_a . d + inc_a ; F_b = W_b - s_b g_b . d + inc_b
    T bd[3] = {T(0), T(0), T(0)}, b_sa = T(0), b_sb = T(0);
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        s.F[f] += bFa[f];
        const T ta = bFa[f] * sa, tb = bFb[f] * sb;
        s.g[3 * f] = fma(ta, dx, s.g[3 * f]);
        s.g[3 * f + 1] = fma(ta, dy, s.g[3 * f + 1]);
        s.g[3 * f + 2] = fma(ta, dz, s.g[3 * f + 2]);
        b_sa = fma(bFa[f], Da[f], b_sa);
        b_sb = fma(bFb[f], Db[f], b_sb);  // (its negative)
#pragma unroll
        for (int k = 0; k < 3; ++k) bd[k] = fma(ta, a[11 + 3 * f + k], fma(-tb, b[11 + 3 * f + k], bd[k]));
    }
    // s_a = Ha / Hs, s_b = Hb / Hs
    s.h = fma(b_sa + b_sb, b[3] * (iHs * iHs), s.h);
    // A = ca B_a d + cb B_b d
    const T b_cka = dot3(bA[0], bA[1], bA[2], ua[0], ua[1], ua[2]);
    const T b_ckb = dot3(bA[0], bA[1], bA[2], ub[0], ub[1], ub[2]);
    const T va[3] = {ca * bA[0], ca * bA[1], ca * bA[2]};
    const T vb[3] = {cb * bA[0], cb * bA[1], cb * bA[2]};
    s.B[0] = fma(va[0], dx, s.B[0]);
    s.B[1] = fma(va[0], dy, fma(va[1], dx, s.B[1]));
    s.B[2] = fma(va[0], dz, fma(va[2], dx, s.B[2]));
    s.B[3] = fma(va[1], dy, s.B[3]);
    s.B[4] = fma(va[1], dz, fma(va[2], dy, s.B[4]));
    s.B[5] = fma(va[2], dz, s.B[5]);
    bd[0] += dot3(Ba[0], Ba[1], Ba[2], va[0], va[1], va[2]) + dot3(Bb[0], Bb[1], Bb[2], vb[0], vb[1], vb[2]);
    bd[1] += dot3(Ba[1], Ba[3], Ba[4], va[0], va[1], va[2]) + dot3(Bb[1], Bb[3], Bb[4], vb[0], vb[1], vb[2]);
    bd[2] += dot3(Ba[2], Ba[4], Ba[5], va[0], va[1], va[2]) + dot3(Bb[2], Bb[4], Bb[5], vb[0], vb[1], vb[2]);
    // ca = knorm_a w(r / Ha), cb likewise
    s.k = fma(b_cka, wa, s.k);
    s.q = fma(b_cka, fma(da, r * a[4], T(3) * wa), s.q);  // (the two parts of dJ/dH_a cancel in part)
    const T b_qa = b_cka * a[5] * da;
    const T br = fma(b_qa, a[4], (b_ckb * b[5] * db) * b[4]) * ir;
    // d = x_b - x_a
    s.x[0] += fma(br, dx, bd[0]);
    s.x[1] += fma(br, dy, bd[1]);
    s.x[2] += fma(br, dz, bd[2]);
}

// Adjoint of the flux pass: per particle over its pairs (N_i then R_i).
template <typename T>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 3 : 1)
    k_flux_adj(int N, const T* __restrict__ rec, const T* __restrict__ sn, const long long* __restrict__ sid,
               const int* __restrict__ sbox, const unsigned* __restrict__ nbr, const int* __restrict__ ncount,
               const unsigned* __restrict__ rnbr, const int* __restrict__ rcount, KParams p,
               const double* __restrict__ dt_use, const T* __restrict__ wgt, T* __restrict__ adj) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    T a[kRecord];
    load_rec(rec, i, a);
    const long long idi = sid[i];
    const T hdt = p.hancock ? (T)(0.5 * dt_use[sbox[i]]) : T(0);
    const T gam = (T)p.gamma;
    T ia[5];
    half_inc(a, hdt, gam, ia);
    T wi[4];
    load4(wgt + 4 * (size_t)i, wi);
    AdjSums<T> s;
    for (int q = 0; q < 3; ++q) s.x[q] = T(0);
    for (int q = 0; q < 5; ++q) s.F[q] = s.W[q] = T(0);
    for (int q = 0; q < 15; ++q) s.g[q] = T(0);
    for (int q = 0; q < 6; ++q) s.B[q] = T(0);
    s.k = s.q = s.h = T(0);
#pragma unroll 1
    for (int list = 0; list < 2; ++list) {
        const unsigned* L = list == 0 ? nbr + 4 * (size_t)i : rnbr + 4 * (size_t)i;
        const int cnt = list == 0 ? min(ncount[i], p.cap) : min(rcount[i], p.rcap);
#pragma unroll 1
        for (int k = 0; k < cnt; ++k) {
            const int j = (int)L[lcol(k, N)];
            T b[kRecord];
            load_rec(rec, j, b);
            T wj[4];
            load4(wgt + 4 * (size_t)j, wj);
            const T wp[3] = {wi[0] - wj[0], wi[1] - wj[1], wi[2] - wj[2]};
            pair_adjoint(a, b, ia, idi < sid[j], hdt, gam, wp, wi[3] - wj[3], s);
        }
    }
    // the half-step primitives: W + (dt/2)(-rho div v, -grad P/rho, -gamma P div v)
    const T div = (a[11 + 3] + a[11 + 7]) + a[11 + 11];
    const T irho = pdiv(T(1), a[6]);
    const T e = -hdt * div, k = -hdt * irho;
    T bW[5], bg[15];
#pragma unroll
    for (int f = 0; f < 5; ++f) bW[f] = s.F[f] + s.W[f];
    bW[0] += e * s.F[0];
    bW[4] += gam * e * s.F[4];
#pragma unroll
    for (int q = 0; q < 15; ++q) bg[q] = s.g[q];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        bW[0] -= (k * s.F[1 + q]) * (irho * a[11 + 12 + q]);  // (1/rho^2 alone could leave the range)
        bg[12 + q] += k * s.F[1 + q];
    }
    const T b_div = -hdt * (a[6] * s.F[0] + gam * a[7] * s.F[4]);
    bg[3] += b_div;
    bg[7] += b_div;
    bg[11] += b_div;
    // knorm = 8 / (pi H^3 n^2); q = r / H
    const T bH = s.h - s.q * a[5] * a[4];
    const T bn = T(-2) * s.k * a[5] * pdiv(T(1), sn[i]);
    T* o = adj + (size_t)i * kAdj;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        o[AX + q] -= s.x[q];
        o[AV + q] += bW[1 + q];
    }
    o[AH] += bH;
    o[AN] += bn;
    o[ARHO] += bW[0];
    o[AP] += bW[4];
#pragma unroll
    for (int q = 0; q < 15; ++q) o[AG + q] += bg[q];
#pragma unroll
    for (int q = 0; q < 6; ++q) o[AB + q] += s.B[q];
}

// Caller-order adjoint weights of the rates -> sorted [N][4].
template <typename T>
__global__ void k_gather_wgt(int N, const unsigned* __restrict__ orig, const double* __restrict__ dpbar,
                             const double* __restrict__ dEbar, T* __restrict__ wgt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    store4(wgt + 4 * (size_t)i, (T)dpbar[o], (T)dpbar[(size_t)N + o], (T)dpbar[2 * (size_t)N + o], (T)dEbar[o]);
}

// Sorted adjoint records -> caller-order outputs (any pointer may be null).
template <typename T>
__global__ void k_adj_out_flux(int N, const unsigned* __restrict__ orig, const T* __restrict__ adj,
                               double* __restrict__ xbar, double* __restrict__ hbar,
                               double* __restrict__ nbar, double* __restrict__ Wbar,
                               double* __restrict__ gbar, double* __restrict__ Bbar) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    const T* a = adj + (size_t)i * kAdj;
    if (xbar)
        for (int k = 0; k < 3; ++k) xbar[(size_t)k * N + o] = a[AX + k];
    if (hbar) hbar[o] = a[AH];
    if (nbar) nbar[o] = a[AN];
    if (Wbar) {
        Wbar[o] = a[ARHO];
        for (int k = 0; k < 3; ++k) Wbar[(size_t)(1 + k) * N + o] = a[AV + k];
        Wbar[4 * (size_t)N + o] = a[AP];
    }
    if (gbar)
        for (int q = 0; q < 15; ++q) gbar[(size_t)q * N + o] = a[AG + q];
    if (Bbar)
        for (int q = 0; q < 6; ++q) Bbar[(size_t)q * N + o] = a[AB + q];
}

// ------------------------------------------------------------- update
// O14 reversed.  v' = v + dt dp/m, x' = x + dt (v + v')/2,
// u' = u + |v|^2/2 + dt dE/m - |v'|^2/2 (a floored u' is a constant).
template <typename T>
__global__ void k_update_adj(int N, Sorted<T> s, const double* __restrict__ dpdt,
                             const double* __restrict__ dEdt, const double* __restrict__ dt_use,
                             gz_particles gend, T* __restrict__ adj, T* __restrict__ wgt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = s.orig[i];
    const T dt = (T)dt_use[s.box[i]];
    const T m = s.m[i];
    const T v[3] = {s.vx[i], s.vy[i], s.vz[i]};
    const T dp[3] = {(T)dpdt[i], (T)dpdt[(size_t)N + i], (T)dpdt[2 * (size_t)N + i]};
    const T dE = (T)dEdt[i];
    // forward update in the working precision, for the floor decision
    T X = s.x[i], Y = s.y[i], Z = s.z[i], VX = v[0], VY = v[1], VZ = v[2], U = s.u[i];
    update_one(m, X, Y, Z, VX, VY, VZ, U, dpdt[i], dpdt[(size_t)N + i], dpdt[2 * (size_t)N + i],
               dEdt[i], dt_use[s.box[i]]);
    const bool floored = !(U > T(0));
    const T im = T(1) / m;
    T vn[3];
    for (int k = 0; k < 3; ++k) vn[k] = v[k] + dt * dp[k] * im;
    const T xb[3] = {gend.x ? ((const T*)gend.x)[o] : T(0), gend.y ? ((const T*)gend.y)[o] : T(0),
                     gend.z ? ((const T*)gend.z)[o] : T(0)};
    const T vb[3] = {gend.vx ? ((const T*)gend.vx)[o] : T(0), gend.vy ? ((const T*)gend.vy)[o] : T(0),
                     gend.vz ? ((const T*)gend.vz)[o] : T(0)};
    const T ub = (gend.u && !floored) ? ((const T*)gend.u)[o] : T(0);
    T* a = adj + (size_t)i * kAdj;
    T mb = -ub * dt * dE * im * im;
    T wv[3];
    for (int k = 0; k < 3; ++k) {
        a[AX + k] += xb[k];
        a[AV + k] += vb[k] + dt * xb[k] + ub * (v[k] - vn[k]);
        const T w = vb[k] + T(0.5) * dt * xb[k];
        wv[k] = dt * im * (w - ub * vn[k]);
        mb += -(vn[k] - v[k]) * im * w + ub * vn[k] * (vn[k] - v[k]) * im;
    }
    store4(wgt + 4 * (size_t)i, wv[0], wv[1], wv[2], ub * dt * im);
    a[AU] += ub;
    a[AM] += mb;
}

// ---------------------------------------------------------- gradients
// One pair (i, j) of particle i's sums E = sum psi d d^T and
// S_f = sum psi (f_j - f_i) d, reversed: with psi = 2 norm w (w half the
// kernel, dw half its derivative, ir = 1/r, iH = 1/H_i), Sb and Eb the sums'
// adjoints and df the field differences, t[f] = Sb_f . d, and
//   psib = d^T Eb d + sum_f df_f t_f,   db = psi (2 Eb d + sum_f df_f Sb_f) + psib psi'(r) d / r.
template <typename T>
__device__ __forceinline__ void pair_grad_adj(const T* Sb, const T* Eb, T norm2, T w, T dw, T ir, T iH, T dx, T dy,
                                              T dz, const T (&df)[5], T& psi, T (&t)[5], T& psib, T (&db)[3]) {
    psi = norm2 * w;
    const T E0 = T(2) * Eb[0], E3 = T(2) * Eb[3], E5 = T(2) * Eb[5];
    T v0 = dot3(E0, Eb[1], Eb[2], dx, dy, dz);
    T v1 = dot3(Eb[1], E3, Eb[4], dx, dy, dz);
    T v2 = dot3(Eb[2], Eb[4], E5, dx, dy, dz);
    psib = T(0.5) * dot3(v0, v1, v2, dx, dy, dz);
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        t[f] = dot3(Sb[3 * f], Sb[3 * f + 1], Sb[3 * f + 2], dx, dy, dz);
        psib = fma(df[f], t[f], psib);
        v0 = fma(df[f], Sb[3 * f], v0);
        v1 = fma(df[f], Sb[3 * f + 1], v1);
        v2 = fma(df[f], Sb[3 * f + 2], v2);
    }
    const T rb = psib * norm2 * dw * iH * ir;
    db[0] = fma(psi, v0, rb * dx);
    db[1] = fma(psi, v1, rb * dy);
    db[2] = fma(psi, v2, rb * dz);
}

// Seeds of particle i's gradient pass: from the adjoints of its limited
// gradients and of B, through the limiter (active constraint only), g = B S
// and B = E^-1.  Adds i's own terms; stores what i's neighbours gather.
// seeds: [0,15) Sbar, [15,21) Ebar (xx xy xz yy yz zz), then per field f
// at 21 + 5 f: xbar (3) and Hbar of the active neighbour, fbar of the
// extreme particle.
template <typename T>
__global__ void __launch_bounds__(128)
    k_grad_seeds(int N, Sorted<T> s, const T* __restrict__ rec, const T* __restrict__ ginfo,
                 const int* __restrict__ lim, const unsigned* __restrict__ nbr,
                 const int* __restrict__ ncount, KParams p, T* __restrict__ adj,
                 T* __restrict__ seeds, unsigned long long* __restrict__ lbloom) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    T* a = adj + (size_t)i * kAdj;
    T* sd = seeds + (size_t)i * kSeed;
    unsigned long long bloom = 0ull;
    const T* G = ginfo + (size_t)i * kGInfo;
    const P4<T> me = s.pos[i];
    const T xi = me.x, yi = me.y, zi = me.z, Hi = me.w;
    const T xim1 = xi - T(1), yim1 = yi - T(1), zim1 = zi - T(1);
    const P4<T> pm = s.prim[i];
    const T Wi[5] = {pm.x, pm.y, pm.z, pm.w, s.prim2[i].x};
    const T Bs[6] = {rec[rec_at<T>(i, 26)], rec[rec_at<T>(i, 27)], rec[rec_at<T>(i, 28)],
                     rec[rec_at<T>(i, 29)], rec[rec_at<T>(i, 30)], rec[rec_at<T>(i, 31)]};
    T fbi[5] = {0, 0, 0, 0, 0};
    T xbi[3] = {0, 0, 0};
    T Hbi = T(0.0), nbi = T(0.0);
    T gb[15];
    T Bb[6];
    for (int q = 0; q < 6; ++q) Bb[q] = (T)a[AB + q];
    // the limiter part of the record (28-55) starts at zero: 16-byte stores
    // (rows are 32-byte aligned, 56 values a row)
#pragma unroll
    for (int q = 28; q < kSeed; q += 4) store4(sd + q, T(0), T(0), T(0), T(0));
    const T beta = p.beta;
    for (int f = 0; f < 5; ++f) {
        const T al = G[30 + f];
        const T g[3] = {G[3 * f], G[3 * f + 1], G[3 * f + 2]};
        const T ghb[3] = {(T)a[AG + 3 * f], (T)a[AG + 3 * f + 1], (T)a[AG + 3 * f + 2]};
        for (int k = 0; k < 3; ++k) gb[3 * f + k] = al * ghb[k];
        const T alb = (ghb[0] * g[0] + ghb[1] * g[1]) + ghb[2] * g[2];
        const int j = lim[(size_t)i * 10 + f];
        if (j >= 0 && alb != T(0.0)) {
            const int k = lim[(size_t)i * 10 + 5 + f];
            const T D = G[35 + f];
            const T c1 = alb * beta / D;
            if (k == i) {
                fbi[f] += c1;
            } else {
                sd[28 + 5 * f + 4] = c1;
                bloom |= 1ull << (k & 63);
            }
            fbi[f] -= c1;
            bloom |= 1ull << (j & 63);
            const T Db = -alb * al / D;
            const P4<T> qj = s.pos[j];
            const T dx = mi_diff(qj.x, xi, xim1), dy = mi_diff(qj.y, yi, yim1),
                         dz = mi_diff(qj.z, zi, zim1);
            const T Hj = qj.w, Hs = (T)Hi + Hj;
            const T sij = (T)Hi / Hs;
            const T o[3] = {sij * dx, sij * dy, sij * dz};
            for (int kk = 0; kk < 3; ++kk) gb[3 * f + kk] += Db * o[kk];
            const T ob[3] = {Db * g[0], Db * g[1], Db * g[2]};
            const T sb = (ob[0] * dx + ob[1] * dy) + ob[2] * dz;
            Hbi += sb * Hj / (Hs * Hs);
            sd[28 + 5 * f + 3] = -sb * (T)Hi / (Hs * Hs);
            for (int kk = 0; kk < 3; ++kk) {
                sd[28 + 5 * f + kk] = ob[kk] * sij;
                xbi[kk] -= ob[kk] * sij;
            }
        }
    }
    // g = B S
    const bool singular = Bs[0] == T(0.0) && Bs[1] == T(0.0) && Bs[2] == T(0.0) && Bs[3] == T(0.0) &&
                          Bs[4] == T(0.0) && Bs[5] == T(0.0);
    T Sb[15];
    for (int f = 0; f < 5; ++f) {
        const T S0 = G[15 + 3 * f], S1 = G[16 + 3 * f], S2 = G[17 + 3 * f];
        const T g0 = gb[3 * f], g1 = gb[3 * f + 1], g2 = gb[3 * f + 2];
        Bb[0] += g0 * S0;
        Bb[1] += g0 * S1 + g1 * S0;
        Bb[2] += g0 * S2 + g2 * S0;
        Bb[3] += g1 * S1;
        Bb[4] += g1 * S2 + g2 * S1;
        Bb[5] += g2 * S2;
        Sb[3 * f] = Bs[0] * g0 + Bs[1] * g1 + Bs[2] * g2;
        Sb[3 * f + 1] = Bs[1] * g0 + Bs[3] * g1 + Bs[4] * g2;
        Sb[3 * f + 2] = Bs[2] * g0 + Bs[4] * g1 + Bs[5] * g2;
    }
    // B = E^-1: Ebar = -B Bbar B (full symmetric matrices)
    const T Bm[3][3] = {{Bs[0], Bs[1], Bs[2]}, {Bs[1], Bs[3], Bs[4]}, {Bs[2], Bs[4], Bs[5]}};
    const T Pm[3][3] = {{Bb[0], T(0.5) * Bb[1], T(0.5) * Bb[2]},
                             {T(0.5) * Bb[1], Bb[3], T(0.5) * Bb[4]},
                             {T(0.5) * Bb[2], T(0.5) * Bb[4], Bb[5]}};
    T T1[3][3], Em[3][3];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) T1[r][c] = (Pm[r][0] * Bm[0][c] + Pm[r][1] * Bm[1][c]) + Pm[r][2] * Bm[2][c];
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) Em[r][c] = -((Bm[r][0] * T1[0][c] + Bm[r][1] * T1[1][c]) + Bm[r][2] * T1[2][c]);
    T Eb[6] = {Em[0][0], Em[0][1] + Em[1][0], Em[0][2] + Em[2][0], Em[1][1], Em[1][2] + Em[2][1], Em[2][2]};
    if (singular) {
        for (int q = 0; q < 6; ++q) Eb[q] = T(0.0);
        for (int q = 0; q < 15; ++q) Sb[q] = T(0.0);
    }
    // own terms of E = sum psi d d^T and S_f = sum (f_j - f_i) psi d
    const T ni = s.n[i];
    const T iH = T(1) / Hi;
    const T norm = T(8.0 / kPi) * iH * iH * iH / ni;
    // record read by every j with j in N_i (k_grad_gather)
    {  // (16-byte stores)
        const T r0[28] = {Sb[0], Sb[1], Sb[2], Sb[3], Sb[4], Sb[5], Sb[6], Sb[7], Sb[8], Sb[9],
                          Sb[10], Sb[11], Sb[12], Sb[13], Sb[14], Eb[0], Eb[1], Eb[2], Eb[3], Eb[4],
                          Eb[5], norm, Wi[0], Wi[1], Wi[2], Wi[3], Wi[4], T(0)};
#pragma unroll
        for (int q = 0; q < 28; q += 4) store4(sd + q, r0[q], r0[q + 1], r0[q + 2], r0[q + 3]);
    }
    lbloom[i] = bloom;
    T normb = T(0.0), Hq = T(0);  // sums of psib w and of psib w' r (w half the kernel)
    const T norm2 = T(2) * norm;
    const int cnt = min(ncount[i], p.cap);
    const unsigned* L = nbr + 4 * (size_t)i;
    for (int k0 = 0; k0 < cnt; k0 += 4) {  // four neighbours' loads in flight at a time
      const uint4 jj = col4(L, k0, N);
      const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
      P4<T> qv[4], pv[4];
      T Pv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
          qv[u] = me;
          if (k0 + u < cnt) {
              qv[u] = s.pos[js[u]];
              pv[u] = s.prim[js[u]];
              Pv[u] = s.prim2[js[u]].x;
          }
      }
      T dx4[4], dy4[4], dz4[4];
      offsets4(qv, xi, yi, zi, xim1, yim1, zim1, dx4, dy4, dz4);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (k0 + u >= cnt) break;
        const T dx = dx4[u], dy = dy4[u], dz = dz4[u];
        const T r2 = max_(sep2(dx, dy, dz), Tiny<T>::sq);
        T r, ir, w, dw;
        roots_(r2, r, ir);
        kern_half_d(r, iH, w, dw);
        const P4<T> pj = pv[u];
        const T df[5] = {pj.x - Wi[0], pj.y - Wi[1], pj.z - Wi[2], pj.w - Wi[3], Pv[u] - Wi[4]};
        T psi, t[5], psib, db[3];
        pair_grad_adj(Sb, Eb, norm2, w, dw, ir, iH, dx, dy, dz, df, psi, t, psib, db);
#pragma unroll
        for (int f = 0; f < 5; ++f) fbi[f] = fma(-psi, t[f], fbi[f]);
        normb = fma(psib, w, normb);
        Hq = fma(psib * dw, r, Hq);
        xbi[0] -= db[0];
        xbi[1] -= db[1];
        xbi[2] -= db[2];
      }
    }
    normb *= T(2);
    Hbi -= Hq * norm2 * iH * iH;
    Hbi += normb * (-T(3.0) * (T)norm / (T)Hi);
    nbi += normb * (-(T)norm / (T)ni);
    a[AX] += xbi[0];
    a[AX + 1] += xbi[1];
    a[AX + 2] += xbi[2];
    a[AH] += Hbi;
    a[AN] += nbi;
    a[ARHO] += fbi[0];
    a[AV] += fbi[1];
    a[AV + 1] += fbi[2];
    a[AV + 2] += fbi[3];
    a[AP] += fbi[4];
}

// Gradient-pass terms of particle j in the sums of every i with j in N_i
// (all such i are in j's pair lists).  Per candidate i the thread reads i's
// packed position and its 28-value record (S_bar, E_bar, psi norm, W_i) as
// 128-bit loads; the limiter rows are read only when i's bloom mask has the
// bit of j.
template <typename T>
__global__ void __launch_bounds__(128)
    k_grad_gather(int N, Sorted<T> s, const int* __restrict__ lim, const unsigned* __restrict__ nbr,
                  const int* __restrict__ ncount, const unsigned* __restrict__ rnbr,
                  const int* __restrict__ rcount, KParams p, const T* __restrict__ seeds,
                  const unsigned long long* __restrict__ lbloom, T* __restrict__ adj) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const P4<T> mj = s.pos[j];
    const P4<T> pj = s.prim[j];
    const T Wj[5] = {pj.x, pj.y, pj.z, pj.w, s.prim2[j].x};
    const unsigned long long jbit = 1ull << (j & 63);
    T fb[5] = {0, 0, 0, 0, 0}, xb[3] = {0, 0, 0}, Hb = T(0.0);
    for (int list = 0; list < 2; ++list) {
        const unsigned* Lj = list == 0 ? nbr + 4 * (size_t)j : rnbr + 4 * (size_t)j;
        const int cnt = list == 0 ? min(ncount[j], p.cap) : min(rcount[j], p.rcap);
        for (int k0 = 0; k0 < cnt; k0 += 4) {  // four candidates' loads in flight at a time
          const uint4 ii = col4(Lj, k0, N);
          const unsigned is[4] = {ii.x, ii.y, ii.z, ii.w};
          P4<T> mv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u)
              if (k0 + u < cnt) mv[u] = s.pos[is[u]];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (k0 + u >= cnt) break;
            const int i = (int)is[u];
            const P4<T> mi = mv[u];
            const T Hi = mi.w;
            // offset as seen by i (x_j - x_i), exactly as i's gradient pass computed it
            const T dx = mi_diff(mj.x, mi.x, mi.x - T(1)), dy = mi_diff(mj.y, mi.y, mi.y - T(1)),
                    dz = mi_diff(mj.z, mi.z, mi.z - T(1));
            const T r2 = sep2(dx, dy, dz);
            if (!less_(r2, Hi * Hi)) continue;  // j is not in N_i
            const T* R = seeds + (size_t)i * kSeed;
            T sd[32];  // record 0-27 (and 4 limiter values, unused here)
            load_row32<32>(R, sd);
            const T r2m = max_(r2, Tiny<T>::sq);
            const T iH = rcp_(Hi);
            T r, ir, w, dw;
            roots_(r2m, r, ir);
            kern_half_d(r, iH, w, dw);
            const T df[5] = {Wj[0] - sd[22], Wj[1] - sd[23], Wj[2] - sd[24], Wj[3] - sd[25], Wj[4] - sd[26]};
            T psi, t[5], psib, db[3];
            pair_grad_adj(sd, sd + 15, T(2) * sd[21], w, dw, ir, iH, dx, dy, dz, df, psi, t, psib, db);
#pragma unroll
            for (int f = 0; f < 5; ++f) fb[f] = fma(psi, t[f], fb[f]);
            xb[0] += db[0];
            xb[1] += db[1];
            xb[2] += db[2];
            // limiter terms where j is i's active neighbour or extreme particle
            if (__ldg(lbloom + i) & jbit) {
                const int* li = lim + (size_t)i * 10;
                for (int f = 0; f < 5; ++f) {
                    const int ja = li[f];
                    if (ja == j) {
                        xb[0] += R[28 + 5 * f];
                        xb[1] += R[28 + 5 * f + 1];
                        xb[2] += R[28 + 5 * f + 2];
                        Hb += R[28 + 5 * f + 3];
                    }
                    if (ja >= 0 && li[5 + f] == j) fb[f] += R[28 + 5 * f + 4];
                }
            }
          }
        }
    }
    T* a = adj + (size_t)j * kAdj;
    a[AX] += xb[0];
    a[AX + 1] += xb[1];
    a[AX + 2] += xb[2];
    a[AH] += Hb;
    a[ARHO] += fb[0];
    a[AV] += fb[1];
    a[AV + 1] += fb[2];
    a[AV + 2] += fb[3];
    a[AP] += fb[4];
}

// ------------------------------------------------------------ density
// rho = m n, P = (gamma - 1) m n u; n = 8 (1 + sum w) / (pi H^3) with H the
// root of f = (32/3)(1 + sum w) - N_ngb: Hbar_tot = Hbar + nbar dn/dH,
// lambda = -Hbar_tot / f_H, and every r_ij in N_i receives
// (w'(q)/H)(nbar 8/(pi H^3) + lambda 32/3) = kappa_i w'(q_ij).
template <typename T>
__global__ void __launch_bounds__(128)
    k_dens_seeds(int N, Sorted<T> s, const unsigned* __restrict__ nbr, const int* __restrict__ ncount,
                 KParams p, T* __restrict__ adj, T* __restrict__ kap) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    T* a = adj + (size_t)i * kAdj;
    const T m = s.m[i], n = s.n[i], u = s.u[i], g1 = T(p.gamma) - T(1.0);
    const T rhob = a[ARHO], Pb = a[AP];
    const T nb = a[AN] + rhob * m + Pb * g1 * m * u;
    a[AM] += rhob * n + Pb * g1 * n * u;
    a[AU] += Pb * g1 * m * n;
    const P4<T> me = s.pos[i];
    const T xi = me.x, yi = me.y, zi = me.z, Hi = me.w;
    const T xim1 = xi - T(1), yim1 = yi - T(1), zim1 = zi - T(1);
    const T iH = T(1) / Hi;
    const int cnt = min(ncount[i], p.cap);
    const unsigned* L = nbr + 4 * (size_t)i;
    // sum over N_i of w'(q) q: the density pass kept its negative (same
    // terms, same order), so no loop over N_i is needed for it here
    const T dsum = -s.sd[i];
    const T H = Hi;
    const T c8 = T(8.0) / (T(kPi) * H * H * H);
    const T dndH = -T(3.0) * n / H - c8 * dsum / H;
    const T fH = -(T(32.0) / T(3.0)) * dsum / H;
    const T Hbt = a[AH] + nb * dndH;
    const T lam = fH != T(0.0) ? -Hbt / fH : T(0.0);
    const T kappa = (nb * c8 + lam * T(32.0) / T(3.0)) / H;
    kap[i] = kappa;
    const T kappa2 = T(2) * kappa;  // (kern_half_d: half the kernel's derivative)
    T xb[3] = {0, 0, 0};
    for (int k0 = 0; k0 < cnt; k0 += 4) {  // four neighbours' loads in flight at a time
        const uint4 jj = col4(L, k0, N);
        const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
        P4<T> qv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (k0 + u < cnt) qv[u] = s.pos[js[u]];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (k0 + u >= cnt) break;
            const P4<T> qj = qv[u];
            const T dx = mi_diff(qj.x, xi, xim1), dy = mi_diff(qj.y, yi, yim1), dz = mi_diff(qj.z, zi, zim1);
            const T r2 = max_(sep2(dx, dy, dz), Tiny<T>::sq);
            T r, ir, w, dw;
            roots_(r2, r, ir);
            kern_half_d(r, iH, w, dw);
            const T c = kappa2 * dw * ir;
            xb[0] -= c * dx;
            xb[1] -= c * dy;
            xb[2] -= c * dz;
        }
    }
    a[AX] += xb[0];
    a[AX + 1] += xb[1];
    a[AX + 2] += xb[2];
}

template <typename T>
__global__ void __launch_bounds__(128)
    k_dens_gather(int N, Sorted<T> s, const unsigned* __restrict__ nbr, const int* __restrict__ ncount,
                  const unsigned* __restrict__ rnbr, const int* __restrict__ rcount, KParams p,
                  const T* __restrict__ kap, T* __restrict__ adj) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    const P4<T> mj = s.pos[j];
    T xb[3] = {0, 0, 0};
    for (int list = 0; list < 2; ++list) {
        const unsigned* Lj = list == 0 ? nbr + 4 * (size_t)j : rnbr + 4 * (size_t)j;
        const int cnt = list == 0 ? min(ncount[j], p.cap) : min(rcount[j], p.rcap);
        for (int k0 = 0; k0 < cnt; k0 += 4) {  // four candidates' loads in flight at a time
            const uint4 ii = col4(Lj, k0, N);
            const unsigned is[4] = {ii.x, ii.y, ii.z, ii.w};
            P4<T> mv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u < cnt) mv[u] = s.pos[is[u]];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (k0 + u >= cnt) break;
                const int i = (int)is[u];
                const P4<T> mi = mv[u];
                const T dx = mi_diff(mj.x, mi.x, mi.x - T(1)), dy = mi_diff(mj.y, mi.y, mi.y - T(1)),
                        dz = mi_diff(mj.z, mi.z, mi.z - T(1));
                T r2 = sep2(dx, dy, dz);
                if (!less_(r2, mi.w * mi.w)) continue;
                r2 = max_(r2, Tiny<T>::sq);
                T r, ir, w, dw;
                roots_(r2, r, ir);
                kern_half_d(r, rcp_(mi.w), w, dw);
                const T c = T(2) * kap[i] * dw * ir;
                xb[0] += c * dx;
                xb[1] += c * dy;
                xb[2] += c * dz;
            }
        }
    }
    T* a = adj + (size_t)j * kAdj;
    a[AX] += xb[0];
    a[AX + 1] += xb[1];
    a[AX + 2] += xb[2];
}

template <typename T>
__global__ void k_adj_out_step(int N, const unsigned* __restrict__ orig, const T* __restrict__ adj,
                               gz_particles gs) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    const T* a = adj + (size_t)i * kAdj;
    if (gs.x) ((T*)gs.x)[o] = (T)a[AX];
    if (gs.y) ((T*)gs.y)[o] = (T)a[AX + 1];
    if (gs.z) ((T*)gs.z)[o] = (T)a[AX + 2];
    if (gs.vx) ((T*)gs.vx)[o] = (T)a[AV];
    if (gs.vy) ((T*)gs.vy)[o] = (T)a[AV + 1];
    if (gs.vz) ((T*)gs.vz)[o] = (T)a[AV + 2];
    if (gs.u) ((T*)gs.u)[o] = (T)a[AU];
    if (gs.m) ((T*)gs.m)[o] = (T)a[AM];
}

}  // namespace

template <typename T>
cudaError_t run_step_adjoint(Ctx& c, const gz_particles& gend, gz_particles& gstart) {
    const int N = c.N;
    const KParams kp = kparams(c);
    Sorted<T> s = sorted_view<T>(c);
    c.launches += 8;
    cudaMemsetAsync(c.adj, 0, sizeof(T) * (size_t)N * kAdj, c.stream);
    k_update_adj<T><<<blocks(N, 256), 256, 0, c.stream>>>(N, s, c.dpdt, c.dEdt, c.dt_use, gend, (T*)c.adj, (T*)c.wgt);
    k_flux_adj<T><<<blocks(N, 128), 128, 0, c.stream>>>(N, (const T*)c.rec, (const T*)c.sn, c.sid, c.sbox,
                                                         c.nbr, c.ncount, c.rnbr, c.rcount, kp, c.dt_use,
                                                         (const T*)c.wgt, (T*)c.adj);
    k_grad_seeds<T><<<blocks(N, 128), 128, 0, c.stream>>>(N, s, (const T*)c.rec, (const T*)c.ginfo, c.lim,
                                                           c.nbr, c.ncount, kp, (T*)c.adj, (T*)c.seeds,
                                                           c.lbloom);
    k_grad_gather<T><<<blocks(N, 128), 128, 0, c.stream>>>(N, s, c.lim, c.nbr, c.ncount, c.rnbr, c.rcount,
                                                            kp, (const T*)c.seeds, c.lbloom, (T*)c.adj);
    k_dens_seeds<T><<<blocks(N, 128), 128, 0, c.stream>>>(N, s, c.nbr, c.ncount, kp, (T*)c.adj, (T*)c.wgt);
    k_dens_gather<T><<<blocks(N, 128), 128, 0, c.stream>>>(N, s, c.nbr, c.ncount, c.rnbr, c.rcount, kp,
                                                            (const T*)c.wgt, (T*)c.adj);
    k_adj_out_step<T><<<blocks(N, 256), 256, 0, c.stream>>>(N, c.vals, (const T*)c.adj, gstart);
    return cudaGetLastError();
}
template cudaError_t run_step_adjoint<float>(Ctx&, const gz_particles&, gz_particles&);
template cudaError_t run_step_adjoint<double>(Ctx&, const gz_particles&, gz_particles&);

cudaError_t ensure_adjoint_scratch(Ctx& c) {
    if (c.adj) return cudaSuccess;
    const size_t Nz = (size_t)c.capacity;  // (a subdomain context's N changes)
    const size_t tsz = c.precision == GZ_FP64 ? 8 : 4;
    auto up = [](size_t b) { return (b + 255) & ~(size_t)255; };  // 256-byte aligned slices
    const size_t sz[6] = {up(sizeof(double) * Nz * kAdj), up(sizeof(double) * Nz * 4), up(tsz * Nz * kSeed),
                          up(sizeof(unsigned long long) * Nz), up(sizeof(int) * Nz * 10),
                          up(tsz * Nz * kGInfo)};
    size_t bytes = 0;
    for (size_t b : sz) bytes += b;
    char* base = nullptr;
    cudaError_t e = cudaMalloc((void**)&base, bytes);
    if (e != cudaSuccess) return e;
    c.adj_arena = base;
    c.adj = base;
    base += sz[0];
    c.wgt = base;
    base += sz[1];
    c.seeds = base;
    base += sz[2];
    c.lbloom = (unsigned long long*)base;
    base += sz[3];
    c.lim = (int*)base;
    base += sz[4];
    c.ginfo = base;
    return cudaSuccess;
}

template <typename T>
cudaError_t run_flux_adjoint(Ctx& c, const double* dpbar, const double* dEbar) {
    c.launches += 2;
    cudaMemsetAsync(c.adj, 0, sizeof(T) * (size_t)c.N * kAdj, c.stream);
    k_gather_wgt<T><<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, c.vals, dpbar, dEbar, (T*)c.wgt);
    k_flux_adj<T><<<blocks(c.N, 128), 128, 0, c.stream>>>(c.N, (const T*)c.rec, (const T*)c.sn, c.sid,
                                                           c.sbox, c.nbr, c.ncount, c.rnbr, c.rcount,
                                                           kparams(c), c.dt_use, (const T*)c.wgt, (T*)c.adj);
    return cudaGetLastError();
}

cudaError_t run_adj_out_flux(Ctx& c, double* xbar, double* hbar, double* nbar, double* Wbar, double* gbar,
                             double* Bbar) {
    c.launches += 1;
    if (c.precision == GZ_FP64)
        k_adj_out_flux<double><<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, c.vals, (const double*)c.adj, xbar,
                                                                       hbar, nbar, Wbar, gbar, Bbar);
    else
        k_adj_out_flux<float><<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, c.vals, (const float*)c.adj, xbar,
                                                                      hbar, nbar, Wbar, gbar, Bbar);
    return cudaGetLastError();
}

template cudaError_t run_flux_adjoint<float>(Ctx&, const double*, const double*);
template cudaError_t run_flux_adjoint<double>(Ctx&, const double*, const double*);

}  // namespace gz
