// Device functions shared by the forward passes and their adjoints.
#pragma once

#include "gz_internal.cuh"

namespace gz {

// Kahan-compensated FP32 sum.
struct Acc {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v) {
        float y = __fsub_rn(v, c);
        float t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
    __device__ __forceinline__ float fvalue() const { return __fsub_rn(s, c); }
};

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

// Division of the gradient limiter and the adjoint: the FP32 path uses the
// hardware reciprocal (about 2 ulp, deterministic); FP64 stays IEEE.
__device__ __forceinline__ float pdiv(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double pdiv(double a, double b) { return a / b; }

// Reciprocal, reciprocal square root and both roots for the pair passes.
// FP32: the hardware approximations (2 ulp), without the range scaling the
// library forms add around them; normal arguments.  FP64: the hardware's 20-bit
// start and one step of third order, y (1 + e + e^2) with e = 1 - x y, and
// y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2 (the binomial series of 1/(1 - e) and
// (1 - e)^(-1/2)), e formed to more than 53 bits: within 0.51 ulp, for |x| in
// [2^-1000, 2^1000], negative x too for the reciprocal.  The square root is
// x y with one correction (x - s^2) y / 2, as accurate: pairs' distances enter
// every face, and x y alone (1 ulp) made FP64 rates 10 % less accurate than
// CUDA's sqrt does.  (CUDA's division and square root in their places would be
// some 50 more of the 290 FP64 operations a pair.)
__device__ __forceinline__ float rcp_(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsq_(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ double rcp_(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rsq_(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = __dmul_rn(x, y);
    const double e = fma(-fma(x, y, -h), y, fma(-h, y, 1.0));
    return fma(y * e, fma(e, 0.375, 0.5), y);
}
// s = sqrt(x), y = 1/s.
__device__ __forceinline__ void roots_(float x, float& s, float& y) {
    y = rsq_(x);
    s = __fmul_rn(x, y);
}
__device__ __forceinline__ void roots_(double x, double& s, double& y) {
    y = rsq_(x);
    const double r = __dmul_rn(x, y);
    s = fma(fma(-r, r, x), 0.5 * y, r);
}
// a / b with y = rcp_(b).  FP64: one correction, so that the quotient rounds
// about once, like a division.
__device__ __forceinline__ float quot_(float a, float, float y) { return __fmul_rn(a, y); }
__device__ __forceinline__ double quot_(double a, double b, double y) {
    const double q = __dmul_rn(a, y);
    return fma(fma(-q, b, a), y, q);
}
// min and max of two numbers.  FP64: compared as integers, which leaves the FP64
// pipe alone; a negative number's integer is mirrored, so that -0 and +0 are one
// number.
__device__ __forceinline__ float min_(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float max_(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ long long order_(double a) {
    const long long i = __double_as_longlong(a);
    return i < 0 ? (long long)(0x8000000000000000ull - (unsigned long long)i) : i;
}
__device__ __forceinline__ double min_(double a, double b) { return order_(a) < order_(b) ? a : b; }
__device__ __forceinline__ double max_(double a, double b) { return order_(a) < order_(b) ? b : a; }
__device__ __forceinline__ bool pos_(float a) { return a > 0.f; }
__device__ __forceinline__ bool pos_(double a) {  // a > 0 (false for NaN)
    const long long i = __double_as_longlong(a);
    return i > 0 && i <= 0x7ff0000000000000ll;
}
// s, a power of two near 1/|D|, and is = 1/s (D normal; clamped where one of the
// two would not be): scaling by them is exact.
__device__ __forceinline__ void pow2_near(float D, float& s, float& is) {
    const unsigned e = min(max(__float_as_uint(D) & 0x7f800000u, 0x00800000u), 0x7e800000u);
    s = __uint_as_float(0x7f000000u - e);
    is = __uint_as_float(e);
}
__device__ __forceinline__ void pow2_near(double D, double& s, double& is) {
    const int e = min(max(__double2hiint(D) & 0x7ff00000, 0x00100000), 0x7fd00000);
    s = __hiloint2double(0x7fe00000 - e, 0);
    is = __hiloint2double(e, 0);
}
// Smallest squares the pair geometry takes (below them rsq_ has no normal
// argument): a face this small (area 3e-19) carries nothing.
template <typename T>
struct Tiny;
template <>
struct Tiny<float> {
    static constexpr float sq = 1e-37f;
};
template <>
struct Tiny<double> {
    static constexpr double sq = 1e-300;
};
// W(q)/2 = t^3 - 4 v^3, t = max(1 - q, 0), v = max(1/2 - q, 0): the kernel
// shape of both pieces without a test (0 beyond the support).
__device__ __forceinline__ float kern_half(float r, float iH) {
    const float t = __saturatef(fmaf(-r, iH, 1.f)), v = __saturatef(fmaf(-r, iH, 0.5f));
    return fmaf(-4.f * (v * v), v, t * t * t);
}
__device__ __forceinline__ double kern_half(double r, double iH) {
    const double q = __dmul_rn(r, iH);
    const int h = __double2hiint(q);
    const bool in = h < 0x3FE00000;
    const double x = in ? q : 1.0 - q;
    const double w = fma(fma(in ? 3.0 : 1.0, x, in ? -3.0 : 0.0), x * x, in ? 0.5 : 0.0);
    return h >= 0x3FF00000 ? 0.0 : w;
}

// W(q)/2 and W'(q)/2 at q = r/H.
__device__ __forceinline__ void kern_half_d(float r, float iH, float& w, float& d) {
    const float t = __saturatef(fmaf(-r, iH, 1.f)), v = __saturatef(fmaf(-r, iH, 0.5f));
    const float t2 = t * t, v2 = v * v;
    w = fmaf(-4.f * v2, v, t2 * t);
    d = fmaf(12.f, v2, -3.f * t2);
}
__device__ __forceinline__ void kern_half_d(double r, double iH, double& w, double& d) {
    const double q = __dmul_rn(r, iH);
    const int h = __double2hiint(q);
    const bool in = h < 0x3FE00000, out = h >= 0x3FF00000;
    const double x = in ? q : 1.0 - q;
    const double ww = fma(fma(in ? 3.0 : 1.0, x, in ? -3.0 : 0.0), x * x, in ? 0.5 : 0.0);
    const double dd = x * fma(in ? 9.0 : -3.0, x, in ? -6.0 : 0.0);
    w = out ? 0.0 : ww;
    d = out ? 0.0 : dd;
}
// a < b (of numbers, not NaN), FP64 compared as integers.
__device__ __forceinline__ bool less_(float a, float b) { return a < b; }
__device__ __forceinline__ bool less_(double a, double b) { return order_(a) < order_(b); }

// x . y, fused the same way wherever it is formed.
template <typename T>
__device__ __forceinline__ T dot3(T x0, T x1, T x2, T y0, T y1, T y2) {
    return fma(x2, y2, fma(x1, y1, mul_rn(x0, y0)));
}

// Minimum-image offsets of four positions from (x, y, z) (xm1 = x - 1, ...).
// FP32: plain differences, which are mi_diff's wherever no |d| reaches 1/2, and
// one test for the four; FP64: mi_diff (its test is on words).
__device__ __forceinline__ void offsets4(const P4<float> (&q)[4], float x, float y, float z, float xm1, float ym1,
                                         float zm1, float (&dx)[4], float (&dy)[4], float (&dz)[4]) {
    float m = 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        dx[u] = q[u].x - x;
        dy[u] = q[u].y - y;
        dz[u] = q[u].z - z;
        m = fmaxf(fmaxf(m, fabsf(dx[u])), fmaxf(fabsf(dy[u]), fabsf(dz[u])));
    }
    if (m >= 0.5f) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            dx[u] = mi_diff(q[u].x, x, xm1);
            dy[u] = mi_diff(q[u].y, y, ym1);
            dz[u] = mi_diff(q[u].z, z, zm1);
        }
    }
}
__device__ __forceinline__ void offsets4(const P4<double> (&q)[4], double x, double y, double z, double, double,
                                         double, double (&dx)[4], double (&dy)[4], double (&dz)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        dx[u] = mi_diff(q[u].x, x, 0.0);
        dy[u] = mi_diff(q[u].y, y, 0.0);
        dz[u] = mi_diff(q[u].z, z, 0.0);
    }
}

// Symmetric 3x3 inverse by adjugate; kappa = |E|_F |B|_F / 3.
template <typename A>
__device__ __forceinline__ void invert_sym(const A E[6], A B[6], A& det, A& kap) {
    const A a = E[0], b = E[1], c = E[2], d = E[3], e = E[4], f = E[5];
    const A Cxx = d * f - e * e, Cxy = c * e - b * f, Cxz = b * e - c * d;
    const A Cyy = a * f - c * c, Cyz = b * c - a * e, Czz = a * d - b * b;
    det = a * Cxx + b * Cxy + c * Cxz;
    const A id = A(1) / det;
    B[0] = Cxx * id;
    B[1] = Cxy * id;
    B[2] = Cxz * id;
    B[3] = Cyy * id;
    B[4] = Cyz * id;
    B[5] = Czz * id;
    const A nE = sqrt(a * a + d * d + f * f + A(2) * (b * b + c * c + e * e));
    const A nB = sqrt(B[0] * B[0] + B[3] * B[3] + B[5] * B[5] +
                      A(2) * (B[1] * B[1] + B[2] * B[2] + B[4] * B[4]));
    kap = nE * nB / A(3);
}

// ---------------------------------------------------------- O10-O12
// A flux record is one 128-byte line (FP32) or two (FP64), read with 32-byte
// vector loads (sm_100+ ld.global.v8.f32 / v4.f64).  Its 32-byte sectors are
// stored rotated by the record's index: a warp gathering one sector of 32
// records would otherwise find them all in the same quarter of the L1 data
// banks (records start on 128-byte lines) and take one pass a lane (31
// measured for 28 lanes); rotated, adjacent records' sectors lie in different
// quarters.
template <typename T>
__device__ __forceinline__ size_t rec_at(int i, int q) {  // place of value q of record i
    constexpr int per = 32 / sizeof(T), ns = kRecord / per;
    return (size_t)i * kRecord + (((q / per + i) & (ns - 1)) * per + q % per);
}
// The record passes may be set up while the pass that writes the records still
// runs (launch_next), so the loads are coherent ones, not of the read-only path
// (.nc: memory nobody writes while the kernel lives), and volatile with a
// memory clobber: they stay behind after_previous.  They take the same time
// (128^3: 2.90 ms a step with the read-only loads, 2.89 with these).
__device__ __forceinline__ void load_rec(const float* rec, int i, float (&v)[kRecord]) {
#pragma unroll
    for (int k = 0; k < kRecord / 8; ++k)
        asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(v[8 * k]), "=f"(v[8 * k + 1]), "=f"(v[8 * k + 2]), "=f"(v[8 * k + 3]), "=f"(v[8 * k + 4]),
              "=f"(v[8 * k + 5]), "=f"(v[8 * k + 6]), "=f"(v[8 * k + 7])
            : "l"(rec + rec_at<float>(i, 8 * k))
            : "memory");
}
__device__ __forceinline__ void load_rec(const double* rec, int i, double (&v)[kRecord]) {
#pragma unroll
    for (int k = 0; k < kRecord / 4; ++k)
        asm volatile("ld.global.v4.f64 {%0,%1,%2,%3}, [%4];"
            : "=d"(v[4 * k]), "=d"(v[4 * k + 1]), "=d"(v[4 * k + 2]), "=d"(v[4 * k + 3])
            : "l"(rec + rec_at<double>(i, 4 * k))
            : "memory");
}

// n values (a multiple of 32 bytes) from 32-byte-aligned global memory with
// 32-byte vector loads, for per-particle rows read by other particles'
// threads (scattered rows: whole sectors per L1 wavefront).  Read-only path: for
// kernels launched the ordinary way (the adjoint passes) only.
template <int n>
__device__ __forceinline__ void load_row32(const float* __restrict__ p, float* v) {
    static_assert(n % 8 == 0, "rows of whole 32-byte vectors");
#pragma unroll
    for (int k = 0; k < n / 8; ++k)
        asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(v[8 * k]), "=f"(v[8 * k + 1]), "=f"(v[8 * k + 2]), "=f"(v[8 * k + 3]), "=f"(v[8 * k + 4]),
              "=f"(v[8 * k + 5]), "=f"(v[8 * k + 6]), "=f"(v[8 * k + 7])
            : "l"(p + 8 * k));
}
template <int n>
__device__ __forceinline__ void load_row32(const double* __restrict__ p, double* v) {
    static_assert(n % 4 == 0, "rows of whole 32-byte vectors");
#pragma unroll
    for (int k = 0; k < n / 4; ++k)
        asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
            : "=d"(v[4 * k]), "=d"(v[4 * k + 1]), "=d"(v[4 * k + 2]), "=d"(v[4 * k + 3])
            : "l"(p + 4 * k));
}

// n values (a multiple of 32 bytes) to 32-byte-aligned global memory with
// 32-byte vector stores: a per-particle row written by its thread fills
// whole sectors instead of one 4-byte piece per store.  The rows are read
// by later passes, not by the writing one: not allocated in L1.
template <int n>
__device__ __forceinline__ void store_row32(float* p, const float* v) {
    static_assert(n % 8 == 0, "rows of whole 32-byte vectors");
#pragma unroll
    for (int k = 0; k < n / 8; ++k)
        asm volatile("st.global.L1::no_allocate.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                     :
                     : "l"(p + 8 * k), "f"(v[8 * k]), "f"(v[8 * k + 1]), "f"(v[8 * k + 2]), "f"(v[8 * k + 3]),
                       "f"(v[8 * k + 4]), "f"(v[8 * k + 5]), "f"(v[8 * k + 6]), "f"(v[8 * k + 7])
                     : "memory");
}
template <int n>
__device__ __forceinline__ void store_row32(double* p, const double* v) {
    static_assert(n % 4 == 0, "rows of whole 32-byte vectors");
#pragma unroll
    for (int k = 0; k < n / 4; ++k)
        asm volatile("st.global.L1::no_allocate.v4.f64 [%0], {%1,%2,%3,%4};"
                     :
                     : "l"(p + 4 * k), "d"(v[4 * k]), "d"(v[4 * k + 1]), "d"(v[4 * k + 2]), "d"(v[4 * k + 3])
                     : "memory");
}

template <typename T>
__device__ __forceinline__ void store_rec(T* rec, int i, const T (&v)[kRecord]) {
    constexpr int per = 32 / sizeof(T);
#pragma unroll
    for (int k = 0; k < kRecord; k += per) store_row32<per>(rec + rec_at<T>(i, k), v + k);
}

// Four values to / from 16-byte-aligned memory.
__device__ __forceinline__ void store4(float* dst, float a, float b, float c, float d) {
    *reinterpret_cast<float4*>(dst) = make_float4(a, b, c, d);
}
__device__ __forceinline__ void store4(double* dst, double a, double b, double c, double d) {
    reinterpret_cast<double2*>(dst)[0] = make_double2(a, b);
    reinterpret_cast<double2*>(dst)[1] = make_double2(c, d);
}
__device__ __forceinline__ void load4(const float* src, float (&v)[4]) {
    const float4 w = __ldg(reinterpret_cast<const float4*>(src));
    v[0] = w.x;
    v[1] = w.y;
    v[2] = w.z;
    v[3] = w.w;
}
__device__ __forceinline__ void load4(const double* src, double (&v)[4]) {
    const double2 w0 = __ldg(reinterpret_cast<const double2*>(src));
    const double2 w1 = __ldg(reinterpret_cast<const double2*>(src) + 1);
    v[0] = w0.x;
    v[1] = w0.y;
    v[2] = w1.x;
    v[3] = w1.y;
}

// O15: HLLC flux of mass, momentum and total energy through a face that
// moves with vf (unit normal n from L to R), from the face states FL, FR
// (rho, v, P) and the wave speeds the caller already formed in the face
// frame (u_K = (v_K - vf) . n, S_L, S_R, S*).  In that frame w = v - vf,
// U = (rho, rho w, E) with E = P/(gamma-1) + rho |w|^2/2 and the flux along n
// is F(U) = (rho u, rho u w + P n, u (E + P)).  The flux at the face (xi = 0)
// is F_K or F_K + S_K (U*_K - U_K) for the side K the waves leave it on, with
// the star state U*_K = rho_K (S_K - u_K)/(S_K - S*) (1, w_K + (S* - u_K) n,
// E_K/rho_K + (S* - u_K)(S* + P_K/(rho_K (S_K - u_K)))).  With q = 1/(S_K - S*),
// g = rho_K q, f = g (S_K - u_K) and dS = S* - u_K the jump S_K (U*_K - U_K)
// is S_K dS (g, g w_K + f n, q (E_K + P_K) + f S*), the same quantity without
// the cancellation of U*_K - U_K for weak waves.  Back in the lab frame the
// fluxes are F_m, F_w + vf F_m and F_E + vf . F_w + |vf|^2 F_m / 2.
template <typename T>
__device__ __forceinline__ void mfv_flux(const T (&FL)[5], const T (&FR)[5], T uL, T uR, T SL, T SR,
                                         T ss, T vfx, T vfy, T vfz, T nx, T ny, T nz, T gam, T& Fm,
                                         T (&Fp)[3], T& FE) {
    // side: L when S_L >= 0 or S* >= 0; the star jump unless S_L >= 0 (L) or
    // S_R <= 0 (R); a NaN speed takes R without the jump, like the oracle
    const bool left = SL >= T(0) || ss >= T(0);
    const bool star = left ? !(SL >= T(0)) : SR > T(0);
    const T rho = left ? FL[0] : FR[0];
    const T P = left ? FL[4] : FR[4];
    const T un = left ? uL : uR;
    const T wx = (left ? FL[1] : FR[1]) - vfx;
    const T wy = (left ? FL[2] : FR[2]) - vfy;
    const T wz = (left ? FL[3] : FR[3]) - vfz;
    const T E = fma(T(0.5) * rho, dot3(wx, wy, wz, wx, wy, wz), pdiv(P, gam - T(1)));
    const T ru = mul_rn(rho, un);
    T fr = ru;
    T fx = fma(ru, wx, mul_rn(P, nx)), fy = fma(ru, wy, mul_rn(P, ny)), fz = fma(ru, wz, mul_rn(P, nz));
    T fe = mul_rn(un, E + P);
    if (star) {
        const T SK = left ? SL : SR;
        const T q = pdiv(T(1), SK - ss);
        const T g = mul_rn(rho, q), f = mul_rn(g, SK - un);
        const T k = mul_rn(SK, ss - un);
        fr = fma(k, g, fr);
        fx = fma(k, fma(g, wx, mul_rn(f, nx)), fx);
        fy = fma(k, fma(g, wy, mul_rn(f, ny)), fy);
        fz = fma(k, fma(g, wz, mul_rn(f, nz)), fz);
        fe = fma(k, fma(q, E + P, mul_rn(f, ss)), fe);
    }
    // (explicit multiply-adds: every kernel that forms the flux gets the same bits)
    Fm = fr;
    Fp[0] = fma(vfx, fr, fx);
    Fp[1] = fma(vfy, fr, fy);
    Fp[2] = fma(vfz, fr, fz);
    FE = fma(T(0.5) * dot3(vfx, vfy, vfz, vfx, vfy, vfz), fr, fe + dot3(vfx, vfy, vfz, fx, fy, fz));
}

// x^y for x > 0 in FP32, 2^(y log2 x) from the hardware base-2 logarithm
// (relative error about 1e-7 (1 + |y log2 x|)).
__device__ __forceinline__ float ppow(float x, float y) { return exp2f(y * __log2f(x)); }

// Exact Riemann problem of the face (option of O12).  Pressure function of one
// side at the trial star pressure p: shock branch (p > P_K)
// (p - P_K) sqrt(A_K/(p + B_K)) with A_K = 2/((gamma+1) rho_K),
// B_K = (gamma-1)/(gamma+1) P_K; rarefaction branch
// 2 c_K/(gamma-1) ((p/P_K)^e - 1), e = (gamma-1)/(2 gamma), whose derivative
// (p/P_K)^(e-1)/(rho_K c_K) is formed from the same power.  f and df/dp.
__device__ __forceinline__ void pres_side(double p, double rho, double P, double c, double gam, double& f,
                                          double& fd) {
    if (p > P) {
        const double A = 2.0 / ((gam + 1.0) * rho), Bk = (gam - 1.0) / (gam + 1.0) * P;
        const double q = sqrt(A / (p + Bk));
        f = (p - P) * q;
        fd = q * (1.0 - 0.5 * ((p - P) / (p + Bk)));
    } else {
        const double r = p / P;
        const double pe = pow(r, (gam - 1.0) / (2.0 * gam));
        f = 2.0 * c / (gam - 1.0) * (pe - 1.0);
        fd = pe / (r * rho * c);
    }
}

// Star pressure and contact speed of the exact solution: the root of
// F(p) = f_L(p) + f_R(p) + u_R - u_L, an increasing concave function.
// Starting point (Toro's adaptive choice): the primitive-variable estimate
// p_PV = (P_L + P_R)/2 - (u_R - u_L)(rho_L + rho_R)(c_L + c_R)/8 when the
// pressures differ by at most 2x and p_PV lies between them; below them the
// two-rarefaction solution [(c_L + c_R - (gamma-1)(u_R - u_L)/2) /
// (c_L P_L^-e + c_R P_R^-e)]^(1/e) (the root itself when both waves are
// rarefactions); above them the two-shock estimate
// (g_L P_L + g_R P_R - (u_R - u_L))/(g_L + g_R), g_K = sqrt(A_K/(p_PV + B_K));
// at least 1e-12 (P_L + P_R).  Newton steps kept inside the bracket the signs
// of F have established (bisection, or doubling while no upper end is known)
// until two iterates agree to 1e-15 (FP64) or 1e-6 (FP32) relative, or (FP32)
// F is at the rounding level of its terms, 4e-7 of |f_L| + |f_R| + |u_R - u_L|,
// where a strong rarefaction's F cannot resolve p to 1e-6; at most 200 (FP64)
// or 20 (FP32) steps.  u* = (u_L + u_R)/2 + (f_R - f_L)/2.  Returns false when
// the two fans open a vacuum (2 (c_L + c_R)/(gamma-1) <= u_R - u_L).
__device__ __forceinline__ bool exact_star(double rL, double uL, double PL, double rR, double uR, double PR, double gam,
                                           double& ps, double& us) {
    const double cL = sqrt(gam * PL / rL), cR = sqrt(gam * PR / rR);
    const double du = uR - uL;
    if (2.0 * (cL + cR) / (gam - 1.0) <= du) return false;
    const double plo = min(PL, PR), phi = max(PL, PR);
    double p = 0.5 * (PL + PR) - 0.125 * du * (rL + rR) * (cL + cR);
    if (!(phi <= 2.0 * plo && p >= plo && p <= phi)) {
        if (p < plo) {
            const double e = (gam - 1.0) / (2.0 * gam);
            const double num = (cL + cR) - 0.5 * (gam - 1.0) * du;
            const double den = cL * pow(PL, -e) + cR * pow(PR, -e);
            p = pow(num / den, 1.0 / e);
        } else {
            const double p0 = max(p, 0.0);
            const double gp1 = gam + 1.0, gm1 = gam - 1.0;
            const double gL = sqrt(2.0 / (gp1 * rL) / (p0 + gm1 / gp1 * PL));
            const double gR = sqrt(2.0 / (gp1 * rR) / (p0 + gm1 / gp1 * PR));
            p = ((gL * PL + gR * PR) - du) / (gL + gR);
        }
    }
    const double pmin = 1e-12 * (PL + PR);
    if (!(p >= pmin)) p = pmin;
    double lo = 0.0, hi = 0.0;
    bool has_hi = false;
    for (int it = 0; it < 200; ++it) {
        double fL, dL, fR, dR;
        pres_side(p, rL, PL, cL, gam, fL, dL);
        pres_side(p, rR, PR, cR, gam, fR, dR);
        const double F = (fL + fR) + du;
        if (F > 0.0) {
            hi = p;
            has_hi = true;
        } else {
            lo = p;
        }
        double pn = p - F / (dL + dR);
        if (!(pn > lo) || (has_hi && !(pn < hi))) pn = has_hi ? 0.5 * (lo + hi) : 2.0 * p;
        const bool done = fabs(pn - p) <= 1e-15 * (pn + p);
        p = pn;
        if (done) break;
    }
    double fL, dL, fR, dR;
    pres_side(p, rL, PL, cL, gam, fL, dL);
    pres_side(p, rR, PR, cR, gam, fR, dR);
    ps = p;
    us = 0.5 * (uL + uR) + 0.5 * (fR - fL);
    return true;
}

// The same in FP32, written for warps whose lanes hold different waves: both
// branches of the two pressure functions are formed and selected (three
// special-function results a side, against four divergent combinations of
// branches: the form above ran 8 of 32 lanes, 616 us for Sod 50^3's flux pass,
// this one 282), and the primitive-variable
// estimate starts the iteration wherever the pressures are within 2x and it is
// not below half the lower one, where Newton's step from it needs one or two
// rounds.  Elsewhere the same two-rarefaction and two-shock estimates.  Stops
// as above; u* takes the two functions at the last pressure, carried there by
// their derivatives.
__device__ __forceinline__ bool exact_star(float rL, float uL, float PL, float rR, float uR, float PR, float gam,
                                           float& ps, float& us) {
    const float qL = gam * PL * rcp_(rL), qR = gam * PR * rcp_(rR);
    const float cL = qL * rsq_(fmaxf(qL, 1e-37f)), cR = qR * rsq_(fmaxf(qR, 1e-37f));
    const float gm1 = gam - 1.f, gp1 = gam + 1.f, i1 = rcp_(gm1), e = 0.5f * gm1 * rcp_(gam);
    const float du = uR - uL;
    if (2.f * (cL + cR) * i1 <= du) return false;
    const float plo = fminf(PL, PR), phi = fmaxf(PL, PR);
    const float iAL = 0.5f * gp1 * rL, iAR = 0.5f * gp1 * rR;  // 1/A_K
    const float mu = gm1 * rcp_(gp1), BL = mu * PL, BR = mu * PR;
    float p = 0.5f * (PL + PR) - 0.125f * du * (rL + rR) * (cL + cR);
    if (!(phi <= 2.f * plo && p >= 0.5f * plo && p <= phi)) {
        if (p < plo) {
            const float num = (cL + cR) - 0.5f * gm1 * du;
            const float den = cL * ppow(PL, -e) + cR * ppow(PR, -e);
            p = ppow(num * rcp_(den), rcp_(e));
        } else {
            const float p0 = fmaxf(p, 0.f);
            const float gL = rsq_((p0 + BL) * iAL), gR = rsq_((p0 + BR) * iAR);
            p = ((gL * PL + gR * PR) - du) * rcp_(gL + gR);
        }
    }
    const float pmin = 1e-12f * (PL + PR);
    if (!(p >= pmin)) p = pmin;
    const float iPL = rcp_(PL), iPR = rcp_(PR), kL = 2.f * cL * i1, kR = 2.f * cR * i1;
    const float jL = PL * rcp_(rL * cL), jR = PR * rcp_(rR * cR);  // P/(rho c)
    float lo = 0.f, hi = 0.f, fL = 0.f, fR = 0.f, dL = 0.f, dR = 0.f, dp = 0.f;
    bool has_hi = false;
    auto side = [&](float P, float iP, float B, float iA, float k, float j, float ip, float& f, float& d) {
        const float q = rsq_((p + B) * iA), dP = p - P;
        const float pe = ppow(p * iP, e);
        const bool shock = p > P;
        f = shock ? dP * q : k * (pe - 1.f);
        // (iA q q = 1/(p + B): q^3 would overflow at rho P below 1e-26)
        d = shock ? fmaf(-0.5f * dP * (iA * q * q), q, q) : pe * j * ip;
    };
#pragma unroll 1
    for (int it = 0; it < 20; ++it) {
        const float ip = rcp_(p);
        side(PL, iPL, BL, iAL, kL, jL, ip, fL, dL);
        side(PR, iPR, BR, iAR, kR, jR, ip, fR, dR);
        const float F = (fL + fR) + du;
        dp = 0.f;
        if (fabsf(F) <= 4e-7f * ((fabsf(fL) + fabsf(fR)) + fabsf(du))) break;
        if (F > 0.f) {
            hi = p;
            has_hi = true;
        } else {
            lo = p;
        }
        float pn = p - F * rcp_(dL + dR);
        if (!(pn > lo) || (has_hi && !(pn < hi))) pn = has_hi ? 0.5f * (lo + hi) : 2.f * p;
        dp = pn - p;
        const bool done = fabsf(dp) <= 1e-6f * (pn + p);
        p = pn;
        if (done) break;
        dp = 0.f;
    }
    ps = p;
    us = 0.5f * (uL + uR) + 0.5f * ((fR - fL) + (dR - dL) * dp);
    return true;
}

// Orientation of a pair (sorted indices i, j; ids idi = id of i, sid[]) in
// the forward flux passes: whether i is L.  MFM: the lower sorted index,
// which both particles of the pair know, so no id is gathered.  MFV: the
// lower id.  Either is a fixed order of the pair, so its two particles
// compute the same canonical flux and get bitwise-opposite contributions
// (the adjoint orients by id: its tie rule at the clamp names L).
template <bool kById>
__device__ __forceinline__ bool pair_order(int i, int j, long long idi, const long long* sid) {
    if constexpr (kById)
        return idi < sid[j];
    else
        return i < j;
}

// Hancock increments of a record's primitives (rho, v, P) to the half step (O11),
// (dt/2)(-rho div v, -grad P / rho, -gamma P div v); hdt = 0 without them.  Both
// particles of a pair form a particle's values with these same operations.
template <typename T>
__device__ __forceinline__ void half_inc(const T (&a)[kRecord], T hdt, T gam, T (&inc)[5]) {
    const T div = (a[11 + 3] + a[11 + 7]) + a[11 + 11];
    const T e = -hdt * div;
    const T k = -hdt * rcp_(a[6]);
    inc[0] = e * a[6];
    inc[1] = k * a[11 + 12];
    inc[2] = k * a[11 + 13];
    inc[3] = k * a[11 + 14];
    inc[4] = gam * e * a[7];
}
// Face value of a field: w + (s g.d + inc), the small terms first, so that it is
// rounded once at the field's size.  (With w + inc formed before: one operation
// a field less, FP64 at 48^3 3 % of the step, FP32 nothing measurable, and energy
// and mass fluxes of quiet gas 3 to 6 % less accurate.)
template <typename T>
__device__ __forceinline__ T face_value(T w, T s, T gd, T inc) {
    return add_rn(w, fma(s, gd, inc));
}

// HLLC star pressure from the face pressures, dP = P_b - P_a, du and the
// impedances (mas, mbs scaled to order one, idens 1/(m_a - m_b) scaled back):
// the lower pressure plus (m dP - m_a m_b du)/(m_a - m_b), m its side's impedance.
// One rounding at the pressure's size where waves are weak (the quotient of
// pressure terms has three, and rates are differences of pressures over the
// neighbours), and no cancellation where they are strong.
template <typename T>
__device__ __forceinline__ T star_pressure(T Pa, T Pb, T dP, T du, T mas, T mbs, T mb, T idens, T& num) {
    const bool lower = less_(Pa, Pb);
    num = fma(-(mas * mb), du, mul_rn(lower ? mas : mbs, dP));
    return fma(num, idens, lower ? Pa : Pb);
}

// Contribution of the pair (a, b) to particle a's rates: dp (3), dE and,
// under MFV (O15), dm.  ia: half_inc of a.  kRiem: the MFM face's star from
// HLLC (0), the exact solver (1), or HLLC with the exact star where HLLC's
// P* < 0 (2).  Returns false when the face area vanishes.  flags: 1 fallback,
// 2 P* < 0 (or vacuum).
//
// Every quantity is symmetric or changes sign under a <-> b, d -> -d, down to
// the bits, so the two particles of a pair get opposite contributions.  For
// the HLLC star that holds by the form it is written in: with
// du = (v_b - v_a).n of the face states, m_a = rho_a min(-c_a, du - c_b) and
// m_b = rho_b max(c_b, c_a - du) (the Davis speeds relative to the face
// states; their exchange is -m_b, -m_a),
//   P* = (m_a P_b - m_b P_a - m_a m_b du) / (m_a - m_b) (star_pressure),
//   S* = ((v_a + v_b).n + (2 (P_b - P_a) - (m_a + m_b) du) / (m_a - m_b)) / 2,
// the contact speed in the lab frame, S*_face + v_f.n whatever v_f is.  Only
// velocity differences enter P*, so nothing cancels at high Mach number.  P*'s
// products of an impedance with a pressure or another impedance would leave the
// range long before the states do (FP32: rho c below 1e-19 or above 1e19), so
// one of the two impedances is scaled to about 1 by an exact power of two, and
// 1/(m_a - m_b) back by it: the same bits, and P* has the states' own range.
template <typename T, bool kMFV, int kRiem>
__device__ __forceinline__ bool pair_rates(const T (&a)[kRecord], const T (&b)[kRecord], const T (&ia)[5], bool aL,
                                           T hdt, T gam, T (&dp)[3], T& dE, T& dm, int& fl) {
    const T dx = mi_diff(b[0], a[0], a[0] - T(1));
    const T dy = mi_diff(b[1], a[1], a[1] - T(1));
    const T dz = mi_diff(b[2], a[2], a[2] - T(1));
    const T r2 = max_(sep2(dx, dy, dz), Tiny<T>::sq);
    T r, ir;
    roots_(r2, r, ir);
    // (the approximate root is most of the FP32 rates' error; MFV pays for a correction)
    if constexpr (kMFV && sizeof(T) == 4) r = fma(fma(-r, r, r2), T(0.5) * ir, r);
    const T ca = a[5] * kern_half(r, a[4]);  // (half of V psi; doubled in A)
    const T cb = b[5] * kern_half(r, b[4]);
    const T Bax = dot3(a[26], a[27], a[28], dx, dy, dz), Bay = dot3(a[27], a[29], a[30], dx, dy, dz),
            Baz = dot3(a[28], a[30], a[31], dx, dy, dz);
    const T Bbx = dot3(b[26], b[27], b[28], dx, dy, dz), Bby = dot3(b[27], b[29], b[30], dx, dy, dz),
            Bbz = dot3(b[28], b[30], b[31], dx, dy, dz);
    const T A0 = add_rn(mul_rn(ca, Bax), mul_rn(cb, Bbx));
    const T A1 = add_rn(mul_rn(ca, Bay), mul_rn(cb, Bby));
    const T A2 = add_rn(mul_rn(ca, Baz), mul_rn(cb, Bbz));
    const T Aq = sep2(A0, A1, A2);
    if (!pos_(Aq - Tiny<T>::sq)) return false;
    T Ah, iA;
    roots_(Aq, Ah, iA);
    const T n0 = A0 * iA, n1 = A1 * iA, n2 = A2 * iA;
    const T Hs = a[3] + b[3], iH = rcp_(Hs);
    // (MFV: the face's velocity, which the mass flux is measured from, hangs on them)
    const T sa = kMFV ? quot_(a[3], Hs, iH) : a[3] * iH, sb = kMFV ? quot_(b[3], Hs, iH) : b[3] * iH;
    // face states: primitives + g . (s d) + Hancock increments, clamped between the
    // particles' primitives
    T Fa[5], Fb[5], ib[5];
    half_inc(b, hdt, gam, ib);
    const T Wa0[5] = {a[6], a[8], a[9], a[10], a[7]};
    const T Wb0[5] = {b[6], b[8], b[9], b[10], b[7]};
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        const T ga = dot3(a[11 + 3 * f], a[12 + 3 * f], a[13 + 3 * f], dx, dy, dz);
        const T gb = dot3(b[11 + 3 * f], b[12 + 3 * f], b[13 + 3 * f], dx, dy, dz);
        const T lo = min_(Wa0[f], Wb0[f]), hi = max_(Wa0[f], Wb0[f]);
        Fa[f] = min_(max_(face_value(Wa0[f], sa, ga, ia[f]), lo), hi);
        Fb[f] = min_(max_(face_value(Wb0[f], -sb, gb, ib[f]), lo), hi);
    }
    if (!(pos_(Fa[0]) && pos_(Fa[4]) && pos_(Fb[0]) && pos_(Fb[4]))) {
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            Fa[f] = Wa0[f];
            Fb[f] = Wb0[f];
        }
        fl |= 1;
    }
    // O12 star state from the face states
    const T qa = gam * Fa[4] * rcp_(Fa[0]), qb = gam * Fb[4] * rcp_(Fb[0]);
    const T cca = mul_rn(qa, rsq_(max_(qa, Tiny<T>::sq))), ccb = mul_rn(qb, rsq_(max_(qb, Tiny<T>::sq)));
    const T du = dot3(Fb[1] - Fa[1], Fb[2] - Fa[2], Fb[3] - Fa[3], n0, n1, n2);
    const T ma = mul_rn(Fa[0], min_(-cca, du - ccb)), mb = mul_rn(Fb[0], max_(ccb, cca - du));
    const T den = ma - mb, iden = rcp_(den);
    T sc, isc;
    pow2_near(den, sc, isc);
    const T mas = ma * sc, mbs = mb * sc;  // (of order one)
    const T dP = Fb[4] - Fa[4];
    T num, ps = star_pressure(Fa[4], Fb[4], dP, du, mas, mbs, mb, iden * isc, num);
    bool neg = ps < T(0);
    if constexpr (!kMFV && kRiem == 0) {
        if (neg) {
            fl |= 2;
            ps = T(0);
        }
        const T X = quot_(fma(-(ma + mb), du, T(2) * dP), den, iden);
        const T p2 = T(-2) * ps;
        dp[0] = mul_rn(p2, A0);  // (rounded here: every caller adds the same bits)
        dp[1] = mul_rn(p2, A1);
        dp[2] = mul_rn(p2, A2);
        // S* |A|, the velocities' part straight from the area vector (A0.. are half of it)
        dE = mul_rn(-ps, fma(X, Ah, dot3(Fa[1] + Fb[1], Fa[2] + Fb[2], Fa[3] + Fb[3], A0, A1, A2)));
        dm = T(0);
        return true;
    } else {
        const T Am = T(2) * Ah;
        // canonical order: L = a when aL (pair_order); face frame v_f
        T FL[5], FR[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            FL[f] = aL ? Fa[f] : Fb[f];
            FR[f] = aL ? Fb[f] : Fa[f];
        }
        const T vLx = aL ? a[8] : b[8], vLy = aL ? a[9] : b[9], vLz = aL ? a[10] : b[10];
        const T vRx = aL ? b[8] : a[8], vRy = aL ? b[9] : a[9], vRz = aL ? b[10] : a[10];
        const T sL = aL ? sa : sb;
        const T nx = aL ? n0 : -n0, ny = aL ? n1 : -n1, nz = aL ? n2 : -n2;
        const T vfx = fma(sL, vRx - vLx, vLx), vfy = fma(sL, vRy - vLy, vLy), vfz = fma(sL, vRz - vLz, vLz);
        const T uL = dot3(FL[1] - vfx, FL[2] - vfy, FL[3] - vfz, nx, ny, nz);
        const T uR = dot3(FR[1] - vfx, FR[2] - vfy, FR[3] - vfz, nx, ny, nz);
        const T mL = aL ? ma : -mb, mR = aL ? mb : -ma;
        const T s0 = quot_(fma(-mR, uR, fma(mL, uL, FR[4] - FL[4])), den, iden);  // S* in the face frame
        if constexpr (kMFV) {
            // both particles of the pair form the same canonical flux bits; L
            // loses what R gains
            if (neg) fl |= 2;
            const T cL = aL ? cca : ccb, cR = aL ? ccb : cca;
            const T SL = min(uL - cL, uR - cR), SR = max(uL + cL, uR + cR);
            T Fm, Fp[3], FE;
            mfv_flux(FL, FR, uL, uR, SL, SR, s0, vfx, vfy, vfz, nx, ny, nz, gam, Fm, Fp, FE);
            const T m = mul_rn(Fm, Am), px = mul_rn(Fp[0], Am), py = mul_rn(Fp[1], Am),
                    pz = mul_rn(Fp[2], Am), e = mul_rn(FE, Am);
            dm = aL ? -m : m;
            dp[0] = aL ? -px : px;
            dp[1] = aL ? -py : py;
            dp[2] = aL ? -pz : pz;
            dE = aL ? -e : e;
            return true;
        } else {
            const T vfn = dot3(vfx, vfy, vfz, nx, ny, nz);
            T sm = s0;  // contact speed of the energy rate
            if (kRiem == 1 || neg) {
                T pe, ue;
                if (exact_star(FL[0], uL, FL[4], FR[0], uR, FR[4], gam, pe, ue)) {
                    ps = pe;
                    sm = ue;
                    if (kRiem == 1) neg = false;
                } else {
                    ps = T(0);
                    sm = T(0);
                    neg = true;
                }
            }
            if (neg) fl |= 2;
            if (ps < T(0)) ps = T(0);
            dm = T(0);
            const T p2 = T(-2) * ps;
            dp[0] = mul_rn(p2, A0);
            dp[1] = mul_rn(p2, A1);
            dp[2] = mul_rn(p2, A2);
            const T ef = mul_rn(ps * (sm + vfn), Am);
            dE = aL ? -ef : ef;
            return true;
        }
    }
}

// Sums of one particle's pair contributions, shared by the flux pass and the
// hierarchical exchange: over N_i then R_i, in the working precision over runs
// of 8 list slots, the runs added up in list order.  One thread forms
// the runs one after another (sum_runs), or the block's four warps, which then
// hold the same 32 particles, form four of them at a time (sum_runs_split):
// the same bits.
// Totals are FP64 in both precisions (the FP32 mode's rates are accumulated in
// double).  Two FP32 words instead (48 bits) took 5 % less of the pass, 128^3 797
// -> 758 us, but are not what the mode promises, and one infinite term turns
// such a total into NaN.
template <int nq>
struct Totals {
    double v[nq];
};
template <typename T, bool kMFV, int kRiem>
constexpr bool kLoadAhead = sizeof(T) == 4 && !kMFV && kRiem == 0;
template <int kRiem>
constexpr int kPairUnroll = kRiem == 0 ? 4 : 1;

// f(j) for the first min(n, 4) slots of a list group, in kUnroll copies.
template <int kUnroll, typename F>
__device__ __forceinline__ void for_slots(const uint4& jj, int n, F&& f) {
    if constexpr (kUnroll == 4) {
        const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (u >= n) break;
            f((int)js[u]);
        }
    } else {
#pragma unroll 1
        for (int u = 0; u < min(n, 4); ++u) f((int)(u == 0 ? jj.x : (u == 1 ? jj.y : (u == 2 ? jj.z : jj.w))));
    }
}

// pair(rec, j, dst) adds the pair with record rec of partner j to dst[nq].
// kAhead: the next partner's record is loaded while the current pair is
// evaluated (two record buffers, so the loop is written for two pairs at a
// time; 164 registers, 12 warps an SM).  The pass waits on its gathers: FP32
// MFM at 128^3 856 us without, 803 with (821 now, with face values and star
// pressure rounded once).  The forms with more arithmetic a
// pair (MFV, the exact solver, FP64) need the registers themselves.  kUnroll:
// copies of the pair's code (the exact solver's is long: one).
template <typename T, int nq, bool kAhead, int kUnroll, typename P>
__device__ __forceinline__ Totals<nq> sum_runs(int i, int N, const T* rec,
                                               const unsigned* nbr, int cnt,
                                               const unsigned* rnbr, int rcnt, P&& pair) {
    double sum[nq];
#pragma unroll
    for (int q = 0; q < nq; ++q) sum[q] = 0.0;
    T A[kRecord], B[kRecord];
#pragma unroll 1
    for (int list = 0; list < 2; ++list) {
        const unsigned* L = (list == 0 ? nbr : rnbr) + 4 * (size_t)i;
        const int n = list == 0 ? cnt : rcnt;
        if (n < 1) continue;
        uint4 jj = col4_once(L, 0, N);
        if constexpr (kAhead) load_rec(rec, (int)jj.x, A);
        T run[nq];
#pragma unroll 1
        for (int k0 = 0; k0 < n; k0 += 4) {
            if (!(k0 & 4)) {
#pragma unroll
                for (int q = 0; q < nq; ++q) run[q] = T(0);
            }
            uint4 nn = jj;
            if (k0 + 4 < n) nn = col4_once(L, k0 + 4, N);
            if constexpr (kAhead) {
                if (k0 + 1 < n) load_rec(rec, (int)jj.y, B);
                pair(A, (int)jj.x, run);
                if (k0 + 1 < n) {
                    if (k0 + 2 < n) load_rec(rec, (int)jj.z, A);
                    pair(B, (int)jj.y, run);
                    if (k0 + 2 < n) {
                        if (k0 + 3 < n) load_rec(rec, (int)jj.w, B);
                        pair(A, (int)jj.z, run);
                        if (k0 + 3 < n) {
                            if (k0 + 4 < n) load_rec(rec, (int)nn.x, A);
                            pair(B, (int)jj.w, run);
                        }
                    }
                }
            } else {
                for_slots<kUnroll>(jj, n - k0, [&](int j) {
                    load_rec(rec, j, A);
                    pair(A, j, run);
                });
            }
            jj = nn;
            if ((k0 & 4) || k0 + 4 >= n) {
#pragma unroll
                for (int q = 0; q < nq; ++q) sum[q] += (double)run[q];
            }
        }
    }
    Totals<nq> t;
#pragma unroll
    for (int q = 0; q < nq; ++q) t.v[q] = sum[q];
    return t;
}

// Four warps: warp c forms runs c, c + 4, ...; v[0] becomes quantity c's total
// (v[1], in warp 0, the fifth's).  Every thread of the block must get here.
template <typename T, int nq, int kUnroll, typename P>
__device__ __forceinline__ Totals<2> sum_runs_split(int i, int N, const T* rec,
                                                    const unsigned* nbr, int cnt,
                                                    const unsigned* rnbr, int rcnt, P&& pair) {
    __shared__ T sh[4][nq][32];
    const int c = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int runs = (cnt + 7) / 8, all = runs + (rcnt + 7) / 8;
    double sum[2] = {0.0, 0.0};
    for (int r0 = 0; __syncthreads_or(r0 < all); r0 += 4) {
        const int r = r0 + c;
        T run[nq];
#pragma unroll
        for (int q = 0; q < nq; ++q) run[q] = T(0);
        if (r < all) {
            const unsigned* L = (r < runs ? nbr : rnbr) + 4 * (size_t)i;
            const int n = r < runs ? cnt : rcnt, k1 = 8 * (r < runs ? r : r - runs);
#pragma unroll 1
            for (int k0 = k1; k0 < min(n, k1 + 8); k0 += 4) {
                const uint4 jj = col4_once(L, k0, N);
                for_slots<kUnroll>(jj, n - k0, [&](int j) {
                    T b[kRecord];
                    load_rec(rec, j, b);
                    pair(b, j, run);
                });
            }
        }
#pragma unroll
        for (int q = 0; q < nq; ++q) sh[c][q][l] = run[q];
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            if (r0 + w >= all) break;
            sum[0] += (double)sh[w][c][l];
            if constexpr (nq == 5) sum[1] += (double)sh[w][4][l];
        }
    }
    Totals<2> t;
    t.v[0] = sum[0];
    t.v[1] = sum[1];
    return t;
}

// Particle of a flux thread (or its position in an index list).
template <bool kSplit>
__device__ __forceinline__ int flux_item() {
    return kSplit ? blockIdx.x * 32 + (threadIdx.x & 31) : blockIdx.x * blockDim.x + threadIdx.x;
}
// The rates of a thread's particle: all of them, or (four warps) quantity c.
template <int nq>
__device__ __forceinline__ void store_rates(const double (&v)[nq], int i, int N, double* dpdt,
                                            double* dEdt, double* dmdt) {
    dpdt[i] = v[0];
    dpdt[(size_t)N + i] = v[1];
    dpdt[2 * (size_t)N + i] = v[2];
    dEdt[i] = v[3];
    if constexpr (nq == 5) dmdt[i] = v[4];
}
template <int nq>
__device__ __forceinline__ void store_rates_split(const double (&v)[2], int i, int N, double* dpdt,
                                                  double* dEdt, double* dmdt) {
    const int c = threadIdx.x >> 5;
    if (c < 3)
        dpdt[(size_t)c * N + i] = v[0];
    else
        dEdt[i] = v[0];
    if constexpr (nq == 5)
        if (c == 0) dmdt[i] = v[1];
}
__device__ __forceinline__ void count_flags(DevStatus* st, int nfall, int nneg) {
    if (nfall) {
        atomicOr(&st->bits, GZ_S_FALLBACK);
        atomicAdd(&st->counters[GZ_C_FALLBACK], (unsigned long long)nfall);
    }
    if (nneg) {
        atomicOr(&st->bits, GZ_S_PSTAR_NEG);
        atomicAdd(&st->counters[GZ_C_PSTAR_NEG], (unsigned long long)nneg);
    }
}

// ----------------------------------------------------------------- O14
__device__ __forceinline__ double wrap1(double v) {
    if (v < 0.0) v += 1.0;
    if (v >= 1.0) v -= 1.0;
    return v;
}

// FP64 state: the literal conserved update, like the oracle, every operation
// rounded explicitly (no contraction), so that each kernel that kicks or
// drifts a particle (the step's update, the hierarchical kick and drift)
// produces the same bits.  Kick: p += dt dp/dt, E += dt dE/dt, v = p/m,
// u = E/m - v^2/2.
__device__ __forceinline__ void kick_one(double m, double& vx, double& vy, double& vz, double& u, double dpx,
                                         double dpy, double dpz, double dE, double dt) {
    const double v2 = __dadd_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz));
    const double E = __dadd_rn(__dmul_rn(m, __dadd_rn(u, __dmul_rn(0.5, v2))), __dmul_rn(dt, dE));
    const double nx = __ddiv_rn(__dadd_rn(__dmul_rn(m, vx), __dmul_rn(dt, dpx)), m);
    const double ny = __ddiv_rn(__dadd_rn(__dmul_rn(m, vy), __dmul_rn(dt, dpy)), m);
    const double nz = __ddiv_rn(__dadd_rn(__dmul_rn(m, vz), __dmul_rn(dt, dpz)), m);
    const double n2 = __dadd_rn(__dadd_rn(__dmul_rn(nx, nx), __dmul_rn(ny, ny)), __dmul_rn(nz, nz));
    u = __dsub_rn(__ddiv_rn(E, m), __dmul_rn(0.5, n2));
    vx = nx;
    vy = ny;
    vz = nz;
}
// Trapezoid drift of one coordinate: wrap(x + dt (v_old + v_new)/2).
__device__ __forceinline__ double drift_one(double x, double v_old, double v_new, double dt) {
    return wrap1(__dadd_rn(x, __dmul_rn(dt, __dmul_rn(0.5, __dadd_rn(v_old, v_new)))));
}
__device__ __forceinline__ void update_one(double m, double& x, double& y, double& z, double& vx,
                                           double& vy, double& vz, double& u, double dpx, double dpy,
                                           double dpz, double dE, double dt) {
    const double ox = vx, oy = vy, oz = vz;
    kick_one(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dt);
    x = drift_one(x, ox, vx, dt);
    y = drift_one(y, oy, vy, dt);
    z = drift_one(z, oz, vz, dt);
}
// FP32 state: the same update written with the increments dv = dt (dp/dt)/m
// and du = dt (dE/dt)/m - dv . (v + dv/2), which is E/m - v_new^2/2 - u
// without the cancellation of the literal form; the drift is
// x + dt (v_old + dv/2).  Explicit rounding as above.
__device__ __forceinline__ float wrapf(float v) {
    if (v < 0.f) v += 1.f;
    if (v >= 1.f) v -= 1.f;
    return v;
}
__device__ __forceinline__ void kick_one(float m, float& vx, float& vy, float& vz, float& u, double dpx,
                                         double dpy, double dpz, double dE, double dt, float& dvx,
                                         float& dvy, float& dvz) {
    const float dtf = (float)dt, im = __fdiv_rn(1.f, m);
    dvx = __fmul_rn(__fmul_rn(dtf, (float)dpx), im);
    dvy = __fmul_rn(__fmul_rn(dtf, (float)dpy), im);
    dvz = __fmul_rn(__fmul_rn(dtf, (float)dpz), im);
    const float hx = __fadd_rn(vx, __fmul_rn(0.5f, dvx)), hy = __fadd_rn(vy, __fmul_rn(0.5f, dvy)),
                hz = __fadd_rn(vz, __fmul_rn(0.5f, dvz));
    const float w = __fadd_rn(__fadd_rn(__fmul_rn(dvx, hx), __fmul_rn(dvy, hy)), __fmul_rn(dvz, hz));
    const float du = __fsub_rn(__fmul_rn(__fmul_rn(dtf, (float)dE), im), w);
    u = __fadd_rn(u, du);
    vx = __fadd_rn(vx, dvx);
    vy = __fadd_rn(vy, dvy);
    vz = __fadd_rn(vz, dvz);
}
__device__ __forceinline__ float drift_onef(float x, float v_old, float dv, double dt) {
    return wrapf(__fadd_rn(x, __fmul_rn((float)dt, __fadd_rn(v_old, __fmul_rn(0.5f, dv)))));
}
__device__ __forceinline__ void update_one(float m, float& x, float& y, float& z, float& vx,
                                           float& vy, float& vz, float& u, double dpx, double dpy,
                                           double dpz, double dE, double dt) {
    const float ox = vx, oy = vy, oz = vz;
    float dvx, dvy, dvz;
    kick_one(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dt, dvx, dvy, dvz);
    x = drift_onef(x, ox, dvx, dt);
    y = drift_onef(y, oy, dvy, dt);
    z = drift_onef(z, oz, dvz, dt);
}

// MFV (O15): the mass advances too, m' = m + dt dm/dt, and momentum and
// total energy are divided by m'.  FP64 state: the literal form, like the
// oracle, explicitly rounded like kick_one.
__device__ __forceinline__ void kick_one_mfv(double& m, double& vx, double& vy, double& vz, double& u,
                                             double dpx, double dpy, double dpz, double dE, double dm,
                                             double dt) {
    const double mn = __dadd_rn(m, __dmul_rn(dt, dm));
    const double v2 = __dadd_rn(__dadd_rn(__dmul_rn(vx, vx), __dmul_rn(vy, vy)), __dmul_rn(vz, vz));
    const double E = __dadd_rn(__dmul_rn(m, __dadd_rn(u, __dmul_rn(0.5, v2))), __dmul_rn(dt, dE));
    const double nx = __ddiv_rn(__dadd_rn(__dmul_rn(m, vx), __dmul_rn(dt, dpx)), mn);
    const double ny = __ddiv_rn(__dadd_rn(__dmul_rn(m, vy), __dmul_rn(dt, dpy)), mn);
    const double nz = __ddiv_rn(__dadd_rn(__dmul_rn(m, vz), __dmul_rn(dt, dpz)), mn);
    const double n2 = __dadd_rn(__dadd_rn(__dmul_rn(nx, nx), __dmul_rn(ny, ny)), __dmul_rn(nz, nz));
    u = __dsub_rn(__ddiv_rn(E, mn), __dmul_rn(0.5, n2));
    vx = nx;
    vy = ny;
    vz = nz;
    m = mn;
}
__device__ __forceinline__ void update_one_mfv(double& m, double& x, double& y, double& z, double& vx,
                                               double& vy, double& vz, double& u, double dpx, double dpy,
                                               double dpz, double dE, double dm, double dt) {
    const double ox = vx, oy = vy, oz = vz;
    kick_one_mfv(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dm, dt);
    x = drift_one(x, ox, vx, dt);
    y = drift_one(y, oy, vy, dt);
    z = drift_one(z, oz, vz, dt);
}
// FP32 state: with dM = dt dm/dt, m' = m + dM (formed in FP64) and the
// increments dv = (dt dp/dt - dM v)/m' and
// du = (dt dE/dt - dM (u + v^2/2))/m' - dv . (v + dv/2), which equal
// p'/m' - v and E'/m' - v'^2/2 - u without the cancellation of the literal
// form; explicitly rounded like kick_one.
__device__ __forceinline__ void kick_one_mfv(float& m, float& vx, float& vy, float& vz, float& u, double dpx,
                                             double dpy, double dpz, double dE, double dm, double dt,
                                             float& dvx, float& dvy, float& dvz) {
    const float mn = (float)__dadd_rn((double)m, __dmul_rn(dt, dm));
    const float dtf = (float)dt, im = __fdiv_rn(1.f, mn), dM = __fmul_rn(dtf, (float)dm);
    dvx = __fmul_rn(__fsub_rn(__fmul_rn(dtf, (float)dpx), __fmul_rn(dM, vx)), im);
    dvy = __fmul_rn(__fsub_rn(__fmul_rn(dtf, (float)dpy), __fmul_rn(dM, vy)), im);
    dvz = __fmul_rn(__fsub_rn(__fmul_rn(dtf, (float)dpz), __fmul_rn(dM, vz)), im);
    const float hx = __fadd_rn(vx, __fmul_rn(0.5f, dvx)), hy = __fadd_rn(vy, __fmul_rn(0.5f, dvy)),
                hz = __fadd_rn(vz, __fmul_rn(0.5f, dvz));
    const float v2 = __fadd_rn(__fadd_rn(__fmul_rn(vx, vx), __fmul_rn(vy, vy)), __fmul_rn(vz, vz));
    const float ek = __fadd_rn(u, __fmul_rn(0.5f, v2));
    const float w = __fadd_rn(__fadd_rn(__fmul_rn(dvx, hx), __fmul_rn(dvy, hy)), __fmul_rn(dvz, hz));
    const float du = __fsub_rn(__fmul_rn(__fsub_rn(__fmul_rn(dtf, (float)dE), __fmul_rn(dM, ek)), im), w);
    u = __fadd_rn(u, du);
    vx = __fadd_rn(vx, dvx);
    vy = __fadd_rn(vy, dvy);
    vz = __fadd_rn(vz, dvz);
    m = mn;
}
__device__ __forceinline__ void update_one_mfv(float& m, float& x, float& y, float& z, float& vx,
                                               float& vy, float& vz, float& u, double dpx, double dpy,
                                               double dpz, double dE, double dm, double dt) {
    const float ox = vx, oy = vy, oz = vz;
    float dvx, dvy, dvz;
    kick_one_mfv(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dm, dt, dvx, dvy, dvz);
    x = drift_onef(x, ox, dvx, dt);
    y = drift_onef(y, oy, dvy, dt);
    z = drift_onef(z, oz, dvz, dt);
}

}  // namespace gz
