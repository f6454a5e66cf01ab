// Internal declarations of the GB300 MFM library: context layout, device
// status, kernel-side helpers.  Nothing here is part of the C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "gz.h"

namespace gz {

constexpr double kPi = 3.14159265358979323846;
constexpr int kRecord = 32;  // values per packed particle record (flux pass)
constexpr int kAdj = 33;     // adjoint values per particle (see gz_adjoint.cu)
constexpr int kSeed = 56;    // gradient-pass adjoint record per particle (working precision):
                             // [0,15) S_bar, [15,21) E_bar, 21 psi norm, [22,27) W, 27 pad,
                             // [28,53) limiter seeds (5 per field), [53,56) pad
constexpr int kGInfo = 40;   // raw gradients, S sums, limiter factors, active limiter Delta

// Device status word (one per context).
struct DevStatus {
    unsigned int bits;
    unsigned int pad;
    unsigned long long first_bad_id;  // smallest id with an error bit (~0 = none)
    unsigned long long counters[GZ_NCOUNTERS];
};

// Per-box cell grid description (device table).
struct BoxInfo {
    int nc;          // cells per axis
    int cell_off;    // first cell of this box in the cell array
    int first;       // first particle (sorted order == caller order per box)
    int count;       // particles in the box
    unsigned key_off;  // first sort key of this box (keys: Morton index of the cell + key_off)
    float wide;        // cells from which a support counts as wide (wide_cells)
};

// A support spanning more cells than this is left to a warp by the density
// pass: its scan is mostly of empty cells (a blast's emptied centre: up to
// thousands, which one thread or a group of four would walk while the rest of
// the block waits).  In cells of the mean support radius H0 or larger: 1.7 (2.1:
// ensemble late in the run 1318 us instead of 1292, Sedov 64^3 370 instead of
// 364; 1.4: 1304 and 387).  Finer cells hold fewer particles each, and a support
// of H0 then spans H0 nc of them: 1.7 H0 (1.7 cells sent every particle there
// once cells were under 0.6 H0, 64^3 at 0.5: 946 us instead of 296).
inline float wide_cells(double H0, int nc) { return (float)(1.7 * (H0 * nc > 1.0 ? H0 * nc : 1.0)); }

// Scalar parameters passed by value to kernels.
struct KParams {
    double gamma, ngb, cfl, kappa_max, beta, u_floor_frac, h_lim;
    double dtol;        // tol * ngb
    float ftol, hlimf;  // tol * ngb rounded down, h_lim rounded up (the same tests on FP32 numbers)
    int hancock, max_iter, cap, rcap, scheme;
};

// Packed per-particle records (one 16-byte-aligned vector load each).
template <typename T>
struct alignas(16) P4 {
    T x, y, z, w;
};
template <typename T>
struct alignas(2 * sizeof(T)) P2 {
    T x, y;
};

// Sorted-order views the kernels share.
template <typename T>
struct Sorted {
    T *x, *y, *z, *vx, *vy, *vz, *m, *u, *h;
    long long* id;      // original ids, sorted order
    unsigned* orig;     // caller index of sorted particle
    int* box;           // box of sorted particle
    T *n, *rho, *P, *c;
    T* sd;              // sum over N_i of -w'(q) q at the converged H (density pass)
    P4<T>* pos;         // (x, y, z, H)
    P4<T>* prim;        // (rho, vx, vy, vz)
    P2<T>* prim2;       // (P, c)
};

struct Grid {
    const BoxInfo* boxes;  // device
    const int2* cells;     // (start, end) per cell, all boxes
};

struct Ctx {
    gz_params params;
    int precision;
    int N;
    int nboxes;
    std::vector<int64_t> counts;
    std::vector<BoxInfo> hboxes;
    int total_cells;
    long long total_keys;  // sort keys of all boxes (per box 8^b, 2^b >= cells per axis)
    cudaStream_t stream;
    // a second stream for the step checkpoint's list copies, which overlap
    // the pair passes (created on the first checkpointing step)
    cudaStream_t side = nullptr;
    cudaEvent_t side_fork = nullptr, side_join = nullptr;
    std::string err;

    // device buffers
    void* arena;
    size_t arena_bytes;
    BoxInfo* boxes;
    int2* cells;
    unsigned *keys, *keys_alt, *vals, *vals_alt;
    unsigned *kcount, *kstart;  // particles per key and their first sorted index (counting sort), else null
    unsigned* hist;             // partial sums of the sort
    int* box_of;  // caller order
    // sorted state (working precision) and derived per-particle data
    void *sx, *sy, *sz, *svx, *svy, *svz, *sm, *su, *sh, *sn, *srho, *sP, *sc, *ssd;
    void *spos, *sprim, *sprim2;  // packed records P4 (x y z H), P4 (rho v), P2 (P c)
    long long* sid;
    int* sbox;
    int* iters;
    int* ncount;
    unsigned* nbr;  // cap slots a particle, in groups of four across the particles (lslot)
    int* rcount;
    unsigned* rnbr;  // rcap slots a particle, laid out like nbr
    void* rec;       // [N][kRecord] working precision
    int* defer = nullptr;   // [N] particles the density pass leaves to its warp-per-particle kernel
    int* ndefer = nullptr;  // [1] their number
    double* dpdt;    // [3][N] sorted
    double* dEdt;    // [N] sorted
    double* dmdt;    // [N] sorted (GZ_MFV only, else null)
    double* dti;     // [N] sorted
    double* dt_box;  // [nboxes] CFL minimum (before the cfl factor is applied: raw min)
    double* dt_use;  // [nboxes] step used
    int* box_hits;   // [nboxes] u-floor hits of the current step
    DevStatus* status;
    int cap, rcap;
    int nbr_valid;  // neighbour lists of the last density pass are current
    long long launches;  // kernel launches issued
    // per-pass CUDA-event profile
    int prof;
    std::vector<cudaEvent_t> ev_pool;
    struct Pending {
        int pass;
        cudaEvent_t a, b;
    };
    std::vector<Pending> pending;
    cudaEvent_t open_ev[GZ_NPASSES] = {};  // PassTimer::begin events awaiting their end
    double prof_ms[GZ_NPASSES];
    long long prof_calls[GZ_NPASSES];
    long long* pairs_dev;  // scratch for gz_pair_count
    // captured multi-step graph
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t graph_exec = nullptr;
    long long graph_kernels = 0;
    // adjoint scratch, allocated on the first backward call
    void* adj_arena = nullptr;
    void* adj = nullptr;      // [N][kAdj] working precision
    void* wgt = nullptr;      // [N][4] rate adjoints (working precision); then kappa [N]
    void* seeds = nullptr;    // [N][kSeed] working precision
    unsigned long long* lbloom = nullptr;  // [N] bit (j & 63) set for each limiter target j
    int* lim = nullptr;       // [N][10] limiter: active neighbour, extreme particle per field
    void* ginfo = nullptr;    // [N][kGInfo] working precision
    // hierarchical-step scratch, allocated on the first gz_step_hier call
    void* hier_arena = nullptr;
    void* hxp = nullptr;      // [3][N] predicted positions (caller order)
    void* hva = nullptr;      // [3][N] velocity at the start of each particle's step
    void* hdvs = nullptr;     // [3][N] velocity change since then
    void* hn = nullptr;       // [N] n of each particle's last active time
    void* hgrad = nullptr;    // [15][N] limited gradients of that time
    void* hB = nullptr;       // [6][N] E^-1 of that time
    int* hsa = nullptr;       // [N] substep its current step started at
    int* hbin = nullptr;      // [N] bin (caller order)
    int* sbin = nullptr;      // [N] bin (sorted order)
    int* alist = nullptr;     // [N] active particles (sorted indices)
    int* tlist = nullptr;     // [N] particles with an exchange this substep
    int* hcount = nullptr;    // [4] device counters (1: |alist|, 2: |tlist|, 3: next substep's actives)
    int* bcount = nullptr;    // per-block counts of the list compaction
    unsigned char* aflag = nullptr;  // [N] active (sorted order)
    unsigned char* tflag = nullptr;  // [N] touched (sorted order)
    float* cellmin = nullptr;             // [cells] smallest H of the cell's active particles
    unsigned char* cellnear = nullptr;    // [cells] an active cell lies within two cells
    unsigned long long* dtmax = nullptr;  // [nboxes] largest finite criterion (bits)
    int* hcount_host = nullptr;           // pinned: active particles of the next substep (two slots)
    cudaEvent_t hier_counted = nullptr;   // its copy done
    // subdomain of a decomposed box (gz_create_subdomain): the particles held
    // are the owned ones and ghost copies completing their neighbourhoods
    unsigned char* owned = nullptr;  // [capacity] 1 = owned (caller order); null: all owned
    int n_owned = 0;                 // owned particles held
    long long grid_count = 0;        // particle count the cell grid is built for (0: the box's own)
    int capacity = 0;                // particles the arrays hold (the context's creation count)
    int step_open = 0;               // gz_step_begin done, gz_step_finish pending
    const int* last_lim = nullptr;   // limiter indices of the last step checkpoint, in this sort
};

// ------------------------------------------------------------------ status
__device__ __forceinline__ void set_status(DevStatus* st, unsigned bit, int counter,
                                           long long id) {
    atomicOr(&st->bits, bit);
    atomicAdd(&st->counters[counter], 1ull);
    if ((bit & GZ_S_ERROR_MASK) && id >= 0)
        atomicMin(&st->first_bad_id, (unsigned long long)id);
}

// --------------------------------------------------------- O1 min image
// FP64: exactly the oracle's expression (difference, then shift by one where
// d >= 1/2 or d < -1/2).  The two comparisons are made on d's words: the FP64
// pipe runs at 1/64 of the FP32 rate and is what bounds every FP64 pass, and
// most pairs then cost it the one subtraction.
__device__ __forceinline__ double mi_diff(double xj, double xi, double /*xim1*/) {
    double d = xj - xi;
    const unsigned h = (unsigned)__double2hiint(d);
    if ((h & 0x7fffffffu) >= 0x3FE00000u) {  // |d| >= 1/2 (or NaN)
        if ((int)h >= 0)
            d = d - 1.0;
        else if (h > 0xBFE00000u || __double2loint(d) != 0)
            d = d + 1.0;
    }
    return d;
}
// FP32: shift the operand near 1 first (x - 1 is exact for x in [1/2, 1)),
// so the wrapped offset is correctly rounded like an unwrapped one.
__device__ __forceinline__ float mi_diff(float xj, float xi, float xim1) {
    float d = xj - xi;
    float dl = __fsub_rn(__fsub_rn(xj, 1.0f), xi);
    float dh = __fsub_rn(xj, xim1);
    return d >= 0.5f ? dl : (d < -0.5f ? dh : d);
}

// --------------------------------------------------------- O2 kernel
template <typename T>
__device__ __forceinline__ T kern_w(T q) {
    T t = T(1) - q;
    T a = T(1) + q * q * (T(-6) + T(6) * q);
    T b = T(2) * t * t * t;
    return q <= T(0.5) ? a : (q < T(1) ? b : T(0));
}

__device__ __forceinline__ bool finite_(float v) { return isfinite(v); }
__device__ __forceinline__ bool finite_(double v) { return isfinite(v); }

// r^2 = (dx dx + dy dy) + dz dz.  FP64 rounds after every operation (no FMA
// contraction), exactly like the oracle, so neighbour decisions agree bitwise.
__device__ __forceinline__ double sep2(double dx, double dy, double dz) {
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}
// FP32: written with explicit fused multiply-adds so that every kernel forms
// r^2 of a pair with the same bits, whatever the compiler contracts elsewhere.
__device__ __forceinline__ float sep2(float dx, float dy, float dz) {
    return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// Neighbour lists (N_i and the reverse lists) are stored in groups of four
// slots: slots 4g..4g+3 of sorted particle i are the 16 bytes at (g N + i) 4,
// N the context's particle count.  A warp, whose threads hold consecutive
// particles, reads one group of their lists as 512 contiguous bytes, one
// 16-byte load a thread.  A particle's list is the column nbr + 4 i; slot k
// of a column lies at lcol(k, N).  (Capacities are multiples of four.)
__device__ __forceinline__ size_t lcol(int k, int N) { return (size_t)(k >> 2) * 4 * (size_t)N + (size_t)(k & 3); }
__device__ __forceinline__ size_t lslot(int k, int i, int N) { return 4 * (size_t)i + lcol(k, N); }
// Slots k0..k0+3 (k0 a multiple of four) of the list column L; those at or
// past the list's count hold no particle.
__device__ __forceinline__ uint4 col4(const unsigned* L, int k0, int N) {
    return *reinterpret_cast<const uint4*>(L + lcol(k0, N));
}
// The same slots for a pass that reads each list once: not kept in L1, which
// stays for the records and positions the pass gathers (a pass that reads
// its lists twice, like the gradient pass, keeps col4).  A coherent load that
// stays behind after_previous.
__device__ __forceinline__ uint4 col4_once(const unsigned* L, int k0, int N) {
    uint4 r;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(L + lcol(k0, N))
                 : "memory");
    return r;
}

// A list slot written by the pass that builds the list: not allocated in
// L1, which stays for the candidates' positions the pass is scanning.
__device__ __forceinline__ void store_slot(unsigned* p, unsigned v) {
    asm volatile("st.global.L1::no_allocate.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// First statement of every kernel that launch_next starts: waits until the
// kernel before it (and so everything before that) has completed and its writes
// are visible.  Without effect in a kernel launched the ordinary way.  What the
// kernel before it writes must not be read through the read-only path: such a
// kernel and what it calls take no __restrict__ pointers (the compiler may then
// use that path, or move a load above the wait) and no .nc loads.
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ordered-integer image of a non-negative double (for atomicMin)
__device__ __forceinline__ unsigned long long dbits(double v) {
    return (unsigned long long)__double_as_longlong(v);
}

// Loop over all candidates in the cells that overlap the cube [x - R, x + R]
// of particle self's box, calling fn(j, r2, ok): ok is false for the particle
// itself and for the slots of a cell's last group of four that lie past its
// range (j and r2 then mean nothing).  The callers act on ok and r2 by
// selection: a branch a candidate, which some lane of the warp nearly always
// takes, costs more than the two stores it would save.
// FP32 with a range well inside half the box: the periodic shift is chosen
// per cell row instead of per candidate, d = (x_j + a) - b with
// (a, b) = (0, x_i), (-1, x_i) for cells wrapped below 0 (x_j - 1 is exact
// there) or (0, x_i - 1) for cells wrapped above 1 (x_i - 1 is exact): the
// same correctly rounded offsets mi_diff gives, at a third of the cost.
// Candidates arrive in ascending j within each cell.
template <typename T, typename F>
__device__ __forceinline__ void for_candidates(const Grid& g, const BoxInfo& bx,
                                               const P4<T>* pos, int self, T xi, T yi,
                                               T zi, T R, F&& fn) {
    const int nc = bx.nc;
    const int2* cells = g.cells + bx.cell_off;
    // positions outside [0, 1] (flagged by the binning pass) see no candidates
    if (!(xi >= T(0) && xi <= T(1) && yi >= T(0) && yi <= T(1) && zi >= T(0) && zi <= T(1) &&
          R >= T(0)))
        return;
    const bool full = !(R < T(0.5));  // (also catches non-finite R)
    const T c3[3] = {xi, yi, zi};
    int lo[3], hi[3];
    bool wraps_all = full;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = full ? 0 : (int)floor((c3[a] - R) * (T)nc - T(1e-3));
        hi[a] = full ? nc - 1 : (int)floor((c3[a] + R) * (T)nc + T(1e-3));
        if (hi[a] - lo[a] + 1 >= nc) {
            lo[a] = 0;
            hi[a] = nc - 1;
            wraps_all = true;
        }
    }
    const T xim1 = xi - T(1), yim1 = yi - T(1), zim1 = zi - T(1);
    const bool percell = sizeof(T) == 4 && !wraps_all && (T(2) * R + T(2) / (T)nc < T(0.5));
    // cells whose nearest point lies beyond R hold no candidate: skipped (the
    // gap of each axis from the cell's unwrapped extent; the margin covers the
    // rounding of the cell bounds; no pruning when the range wraps the box)
    const T cl = T(1) / (T)nc, R2m = R * R * T(1.0001);
    for (int cz = lo[2]; cz <= hi[2]; ++cz) {
        const int wz = cz < 0 ? cz + nc : (cz >= nc ? cz - nc : cz);
        const T az = cz < 0 ? T(-1) : T(0), bz = cz >= nc ? zim1 : zi;
        const T gz = wraps_all ? T(0) : max(max((T)cz * cl - zi, zi - (T)(cz + 1) * cl), T(0));
        const T gz2 = gz * gz;
        if (gz2 > R2m) continue;
        for (int cy = lo[1]; cy <= hi[1]; ++cy) {
            const int wy = cy < 0 ? cy + nc : (cy >= nc ? cy - nc : cy);
            const T ay = cy < 0 ? T(-1) : T(0), by = cy >= nc ? yim1 : yi;
            const T gy = wraps_all ? T(0) : max(max((T)cy * cl - yi, yi - (T)(cy + 1) * cl), T(0));
            const T gzy2 = gz2 + gy * gy;
            if (gzy2 > R2m) continue;
            const int row = (wz * nc + wy) * nc;
            for (int cx = lo[0]; cx <= hi[0]; ++cx) {
                const int wx = cx < 0 ? cx + nc : (cx >= nc ? cx - nc : cx);
                const T ax = cx < 0 ? T(-1) : T(0), bxx = cx >= nc ? xim1 : xi;
                const T gx = wraps_all ? T(0) : max(max((T)cx * cl - xi, xi - (T)(cx + 1) * cl), T(0));
                if (gzy2 + gx * gx > R2m) continue;
                const int2 se = cells[row + wx];
                // four candidates at a time, their distances formed together
                // (pos is readable up to three records past its last), and
                // handed over without a branch
                for (int j0 = se.x; j0 < se.y; j0 += 4) {
                    P4<T> q[4];
                    T r2s[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) q[u] = pos[j0 + u];
                    if (percell) {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            r2s[u] = sep2((q[u].x + ax) - bxx, (q[u].y + ay) - by, (q[u].z + az) - bz);
                    } else {
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            r2s[u] = sep2(mi_diff(q[u].x, xi, xim1), mi_diff(q[u].y, yi, yim1), mi_diff(q[u].z, zi, zim1));
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) fn(j0 + u, r2s[u], j0 + u < se.y && j0 + u != self);
                }
            }
        }
    }
}

constexpr int kLaneCells = 16;
constexpr int kCrowdCell = 128;  // particles from which a cell is shared by lanes instead of walked by one thread

// Warp-cooperative candidate scan for one particle per warp (every lane
// passes the same particle): each lane calls fn(j, dx, dy, dz, r2) for its
// share of the candidates j != self in the cells overlapping [x - R, x + R]
// (cells whose nearest point lies beyond R skipped, as in for_candidates).
// Ranges of under kLaneCells cells are shared candidate by candidate (the
// lanes take start + lane, start + 32 + lane, ... of every cell); larger ones
// cell by cell (lane l takes cells l, l + 32, ... of the range, in row
// order), which keeps lanes busy where a support holds many cells and puts
// the cells' range and candidate loads in flight together instead of one
// cell after another.  Which lane
// sees which candidate depends only on the particle, so per-lane sums
// combined in a fixed order are deterministic.  Offsets from mi_diff.
template <typename T, typename F>
__device__ __forceinline__ void for_candidates_lanes(const Grid& g, const BoxInfo& bx,
                                                     const P4<T>* pos, int self, T xi, T yi,
                                                     T zi, T R, int lane, F&& fn) {
    const int nc = bx.nc;
    const int2* cells = g.cells + bx.cell_off;
    if (!(xi >= T(0) && xi <= T(1) && yi >= T(0) && yi <= T(1) && zi >= T(0) && zi <= T(1) &&
          R >= T(0)))
        return;
    const bool full = !(R < T(0.5));
    const T c3[3] = {xi, yi, zi};
    int lo[3], hi[3];
    bool wraps_all = full;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        lo[a] = full ? 0 : (int)floor((c3[a] - R) * (T)nc - T(1e-3));
        hi[a] = full ? nc - 1 : (int)floor((c3[a] + R) * (T)nc + T(1e-3));
        if (hi[a] - lo[a] + 1 >= nc) {
            lo[a] = 0;
            hi[a] = nc - 1;
            wraps_all = true;
        }
    }
    const T xim1 = xi - T(1), yim1 = yi - T(1), zim1 = zi - T(1);
    const T cl = T(1) / (T)nc, R2m = R * R * T(1.0001);
    auto gap = [&](int c, T v) { return wraps_all ? T(0) : max(max((T)c * cl - v, v - (T)(c + 1) * cl), T(0)); };
    auto cell_range = [&](int cx, int cy, int cz, int2& se) {
        const T gx = gap(cx, xi), gy = gap(cy, yi), gz = gap(cz, zi);
        if (gx * gx + gy * gy + gz * gz > R2m) return false;
        const int wx = cx < 0 ? cx + nc : (cx >= nc ? cx - nc : cx);
        const int wy = cy < 0 ? cy + nc : (cy >= nc ? cy - nc : cy);
        const int wz = cz < 0 ? cz + nc : (cz >= nc ? cz - nc : cz);
        se = cells[(wz * nc + wy) * nc + wx];
        return true;
    };
    auto visit = [&](int j) {
        const P4<T> q = pos[j];
        const T dx = mi_diff(q.x, xi, xim1), dy = mi_diff(q.y, yi, yim1), dz = mi_diff(q.z, zi, zim1);
        fn(j, dx, dy, dz, sep2(dx, dy, dz));
    };
    const int ex = hi[0] - lo[0] + 1, ey = hi[1] - lo[1] + 1, ez = hi[2] - lo[2] + 1;
    const int ncube = ex * ey * ez;
    if (ncube >= kLaneCells) {
        for (int f0 = 0; f0 < ncube; f0 += 32) {
            const int f = f0 + lane;
            const int cx = lo[0] + f % ex, cy = lo[1] + (f / ex) % ey, cz = lo[2] + f / (ex * ey);
            int2 se = make_int2(0, 0);
            if (f < ncube && !cell_range(cx, cy, cz, se)) se = make_int2(0, 0);
            // (a crowded cell is shared by the lanes)
            for (unsigned big = __ballot_sync(0xffffffffu, se.y - se.x > kCrowdCell); big; big &= big - 1) {
                const int l = __ffs(big) - 1;
                const int a = __shfl_sync(0xffffffffu, se.x, l), e = __shfl_sync(0xffffffffu, se.y, l);
                for (int j = a + lane; j < e; j += 32)
                    if (j != self) visit(j);
                if (lane == l) se.y = se.x;
            }
            for (int j = se.x; j < se.y; ++j)
                if (j != self) visit(j);
        }
    } else {
        for (int cz = lo[2]; cz <= hi[2]; ++cz)
            for (int cy = lo[1]; cy <= hi[1]; ++cy)
                for (int cx = lo[0]; cx <= hi[0]; ++cx) {
                    int2 se;
                    if (!cell_range(cx, cy, cz, se)) continue;
                    for (int j = se.x + lane; j < se.y; j += 32)
                        if (j != self) visit(j);
                }
    }
}

// The FP32 number next to a position x towards 0 (its leading 24 bits), formed
// from its words: a conversion would go through the FP64 pipe, whose rate is
// 1/64 of FP32's.  (Numbers below 2^-126 give 0 or a denormal.)  Positions that
// are no numbers, or out of FP32's range, give an infinity or NaN, whose
// distance to anything is no number, so they are near nothing; those outside
// [0, 1] keep their sign.
__device__ __forceinline__ float chop(double x) {
    const int h = __double2hiint(x);
    const int m = min(max(h & 0x7fffffff, 0x38000000) - 0x38000000, 0x0ff00000);
    return __int_as_float((h & 0x80000000) | (m << 3) | (int)((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ float chop(float x) { return x; }

// Search window of a particle: the cells overlapping [x - R, x + R] (periodic),
// their offsets and the tests for_candidates applies to them, with the cells
// numbered in its loop order.
template <typename T>
struct Window {
    int lo[3], ex, exy, ncube, nc;
    float R2m, cl, rex, rexy;
    bool wraps_all, percell;
    __device__ __forceinline__ Window(int nc_, T xi, T yi, T zi, T R) : nc(nc_) {
        ncube = 0;
        // positions outside [0, 1] (flagged by the binning pass) see no candidates
        if (!(xi >= T(0) && xi <= T(1) && yi >= T(0) && yi <= T(1) && zi >= T(0) && zi <= T(1) && R >= T(0))) return;
        const bool full = !(R < T(0.5));  // (also catches non-finite R)
        const T c3[3] = {xi, yi, zi};
        int n[3];
        wraps_all = full;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            lo[a] = full ? 0 : (int)floor((c3[a] - R) * (T)nc - T(1e-3));
            int hi = full ? nc - 1 : (int)floor((c3[a] + R) * (T)nc + T(1e-3));
            if (hi - lo[a] + 1 >= nc) {
                lo[a] = 0;
                hi = nc - 1;
                wraps_all = true;
            }
            n[a] = hi - lo[a] + 1;
        }
        ex = n[0];
        exy = n[0] * n[1];
        ncube = exy * n[2];
        rex = __frcp_rn((float)ex);
        rexy = __frcp_rn((float)exy);
        cl = 1.f / (float)nc;
        const float Rf = (float)R + (sizeof(T) == 8 ? 4e-7f : 0.f);
        R2m = Rf * Rf * 1.0001f;
        percell = sizeof(T) == 4 && !wraps_all && (2.f * Rf + 2.f * cl < 0.5f);
    }
    // Coordinates of cell f of the window (x fastest), unwrapped.  The float
    // quotients are off by at most one, corrected after.
    __device__ __forceinline__ void coords(int f, int& cx, int& cy, int& cz) const {
        int z = (int)(((float)f + 0.5f) * rexy);
        int rem = f - z * exy;
        if (rem < 0) {
            --z;
            rem += exy;
        } else if (rem >= exy) {
            ++z;
            rem -= exy;
        }
        int y = (int)(((float)rem + 0.5f) * rex);
        int x = rem - y * ex;
        if (x < 0) {
            --y;
            x += ex;
        } else if (x >= ex) {
            ++y;
            x -= ex;
        }
        cx = lo[0] + x;
        cy = lo[1] + y;
        cz = lo[2] + z;
    }
    // Candidates of cell (cx, cy, cz): none when its nearest point lies beyond R.
    // In FP32 for both precisions: the margin on R^2 covers the rounding of the
    // cell bounds and of the FP32 copies of x and R.
    __device__ __forceinline__ int2 range(const int2* cells, int cx, int cy, int cz, float xi, float yi,
                                          float zi) const {
        auto gap = [&](int c, float v) {
            return wraps_all ? 0.f : max(max((float)c * cl - v, v - (float)(c + 1) * cl), 0.f);
        };
        const float gx = gap(cx, xi), gy = gap(cy, yi), gz = gap(cz, zi);
        if ((gz * gz + gy * gy) + gx * gx > R2m) return make_int2(0, 0);
        return cells[wrapped(cx, cy, cz)];
    }
    // Index of cell (cx, cy, cz) within its box.
    __device__ __forceinline__ int wrapped(int cx, int cy, int cz) const {
        const int wx = cx < 0 ? cx + nc : (cx >= nc ? cx - nc : cx);
        const int wy = cy < 0 ? cy + nc : (cy >= nc ? cy - nc : cy);
        const int wz = cz < 0 ? cz + nc : (cz >= nc ? cz - nc : cz);
        return (wz * nc + wy) * nc + wx;
    }
};

template <int G>
__device__ __forceinline__ unsigned group_mask() {
    static_assert(G >= 2 && G <= 32 && (G & (G - 1)) == 0, "a group is a power of two of lanes");
    return (0xffffffffu >> (32 - G)) << (threadIdx.x & 31 & ~(G - 1));
}

// Squared distance of two chopped positions in FP32 and the bound below which
// every pair with r < R falls: chop and the subtraction put at most 1.8e-7 on
// an axis (3.2e-7 on r), the squares and sums 3 rounding errors.
__device__ __forceinline__ float r2_chop(double xj, double yj, double zj, float xi, float yi, float zi) {
    float dx = chop(xj) - xi, dy = chop(yj) - yi, dz = chop(zj) - zi;
    dx -= rintf(dx);
    dy -= rintf(dy);
    dz -= rintf(dz);
    return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}
__device__ __forceinline__ float r2_chop_bound(double R) {
    const float r = ((float)R + 4e-7f) * (1.f + 1e-6f);
    return r * r;
}

// The n entries of the list column L put in increasing order by insertion.
__device__ __forceinline__ void insert_sort(unsigned* L, int n, int N) {
    for (int a = 1; a < n; ++a) {
        const unsigned x = L[lcol(a, N)];
        int b = a - 1;
        while (b >= 0 && L[lcol(b, N)] > x) {
            L[lcol(b + 1, N)] = L[lcol(b, N)];
            --b;
        }
        L[lcol(b + 1, N)] = x;
    }
}

// The same by kListLanes lanes (the entries are distinct; blocks of kListBlock
// threads): each lane places its entries by the number of smaller ones; lists
// longer than kListMax by insertion.  For lists of a few dozen entries: one
// thread's insertion through global memory is a chain of dependent accesses
// (hierarchical Sedov 64^3: 26 us a substep, 15 so).
constexpr int kListLanes = 8, kListBlock = 128, kListMax = 64;
__device__ __forceinline__ void sort_list(unsigned* L, int n, int N) {
    __shared__ unsigned sh[kListBlock / kListLanes][kListMax + kListLanes];
    if (n < 2) return;
    const int gl = threadIdx.x % kListLanes;
    const unsigned gm = group_mask<kListLanes>();
    unsigned* v = sh[threadIdx.x / kListLanes];
    if (n <= kListMax) {
        for (int k = gl; k < n; k += kListLanes) v[k] = L[lcol(k, N)];
        __syncwarp(gm);
        for (int k = gl; k < n; k += kListLanes) {
            const unsigned x = v[k];
            int at = 0;
            for (int q = 0; q < n; ++q) at += v[q] < x;
            L[lcol(at, N)] = x;
        }
    } else if (gl == 0) {
        insert_sort(L, n, N);
    }
}

// Scan of one particle's search window by the G lanes of its group (all of
// them pass the same particle): the candidates j != self with r^2 < R^2,
// handed to emit(k, j) with k = 0, 1, ... in for_candidates' order (cells in
// its loop order, j ascending within a cell), each by one lane of the group.
// A round takes G cells, one a lane (cells of more than 32 candidates one after
// another, 32 candidates a lane): the lane tests its candidates into a bit mask, a prefix sum over the group numbers the hits, and the lane
// hands its set bits over (a few instructions each: lanes have unequal hits,
// so what is done per hit is left to the caller's pass over the numbered
// hits, where every lane is busy).  Returns the number of hits (the same for
// every lane); stops early once there are more than `most`.
// FP64: the mask comes from FP32 distances with a margin, so the FP64 pipe
// sees only the hits; candidates up to 5e-7 outside R are handed over
// too, unless kExact asks for the FP64 test of each.
template <typename T, int G, bool kExact = false, typename E>
__device__ __forceinline__ int group_scan(const Grid& g, const BoxInfo& bx, const P4<T>* pos,
                                          int self, T xi, T yi, T zi, T R, int gl, unsigned gm, int most,
                                          E&& emit) {
    const Window<T> w(bx.nc, xi, yi, zi, R);
    const int2* cells = g.cells + bx.cell_off;
    const T xim1 = xi - T(1), yim1 = yi - T(1), zim1 = zi - T(1);
    const T R2 = R * R;
    const float xf = chop(xi), yf = chop(yi), zf = chop(zi);
    const float R2f = sizeof(T) == 8 ? r2_chop_bound((double)R) : 0.f;
    int base = 0;
    for (int f0 = 0; f0 < w.ncube; f0 += G) {
        int2 se = make_int2(0, 0);
        // FP32 well inside half the box: the periodic shift of the cell,
        // (x_j + a) - b, the same correctly rounded offsets mi_diff gives
        T ax = T(0), ay = T(0), az = T(0), bxx = xi, byy = yi, bzz = zi;
        if (f0 + gl < w.ncube) {
            int cx, cy, cz;
            w.coords(f0 + gl, cx, cy, cz);
            se = w.range(cells, cx, cy, cz, xf, yf, zf);
            if (sizeof(T) == 4 && w.percell) {
                ax = cx < 0 ? T(-1) : T(0);
                ay = cy < 0 ? T(-1) : T(0);
                az = cz < 0 ? T(-1) : T(0);
                bxx = cx >= w.nc ? xim1 : xi;
                byy = cy >= w.nc ? yim1 : yi;
                bzz = cz >= w.nc ? zim1 : zi;
            }
        }
        auto within = [&](const P4<T>& q) {
            return sep2(mi_diff(q.x, xi, xim1), mi_diff(q.y, yi, yim1), mi_diff(q.z, zi, zim1)) < R2;
        };
        auto near = [&](const P4<T>& q) {
            if constexpr (sizeof(T) == 8) return r2_chop(q.x, q.y, q.z, xf, yf, zf) < R2f;
            return within(q);
        };
        // the hits among each lane's candidates a..e-1 (32 at most), numbered and
        // handed over
        auto take = [&](int a, int e, auto hit) {
            unsigned m = 0;
            for (int j0 = a; j0 < e; j0 += 4) {
                P4<T> q[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) q[u] = pos[min(j0 + u, e - 1)];
                unsigned n4 = 0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (hit(q[u])) n4 |= 1u << u;
                m |= n4 << (j0 - a);
            }
            const int nj = max(e - a, 0);
            if (nj < 32) m &= (1u << nj) - 1u;  // (the last group of four repeats the last candidate)
            if (self >= a && self < e) m &= ~(1u << (self - a));
            if constexpr (sizeof(T) == 8 && kExact)
                for (unsigned b = m; b; b &= b - 1)
                    if (!within(pos[a + __ffs(b) - 1])) m &= ~(b & (0u - b));
            const int cnt = __popc(m);
            int pre = cnt;
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
                const int y = __shfl_up_sync(gm, pre, o, G);
                if (gl >= o) pre += y;
            }
            const int total = __shfl_sync(gm, pre, G - 1, G);
            int k = base + pre - cnt;
            for (; m; m &= m - 1) emit(k++, a + __ffs(m) - 1);
            base += total;
        };
        if (__any_sync(gm, se.y - se.x > 32)) {
            // a cell of more than 32 candidates: these G cells one after
            // another, 32 candidates a lane at a time
            for (int l = 0; l < G && base <= most; ++l) {
                const int a = __shfl_sync(gm, se.x, l, G), e = __shfl_sync(gm, se.y, l, G);
                for (int j0 = a; j0 < e && base <= most; j0 += 32 * G) take(j0 + 32 * gl, min(e, j0 + 32 * gl + 32), near);
            }
        } else if constexpr (sizeof(T) == 8) {
            take(se.x, se.y, near);
        } else if (w.percell) {
            take(se.x, se.y,
                 [&](const P4<T>& q) { return sep2((q.x + ax) - bxx, (q.y + ay) - byy, (q.z + az) - bzz) < R2; });
        } else {
            take(se.x, se.y, near);
        }
        if (base > most) break;
    }
    return base;
}

// The candidates j != self with r^2 < R2 in the cells overlapping
// [x - R, x + R] (every lane passes the same particle), handed to
// emit(k, j, r2) with k = 0, 1, ... in the order for_candidates visits them
// (cells in its loop order, j ascending within a cell), so a list written
// by a warp equals the one a thread's scan writes.  Cells are taken as
// for_candidates_lanes takes them: small ranges candidate by candidate (a
// ballot per 32 candidates places the hits), large ones 32 cells at a time
// (each lane tests its cell's candidates four at a time into a bit mask, an
// exclusive prefix across the warp places the hits, the lane writes them: the
// density pass of Sedov 64^3 late in the run 395 -> 370 us over counting them
// one by one), with the ranges of four such rounds loaded together: a wide
// support's cells are mostly empty, and the scan waits on those loads.
// Returns the number of hits.
constexpr int kAhead = 4;
template <typename T, typename E>
__device__ __forceinline__ int for_hits_lanes_ordered(const Grid& g, const BoxInfo& bx,
                                                      const P4<T>* pos, int self, T xi, T yi,
                                                      T zi, T R, T R2, int lane, E&& emit) {
    const Window<T> w(bx.nc, xi, yi, zi, R);
    const int2* cells = g.cells + bx.cell_off;
    const T xim1 = xi - T(1), yim1 = yi - T(1), zim1 = zi - T(1);
    const float xf = chop(xi), yf = chop(yi), zf = chop(zi);
    auto r2_of = [&](int j) {
        const P4<T> q = pos[j];
        return sep2(mi_diff(q.x, xi, xim1), mi_diff(q.y, yi, yim1), mi_diff(q.z, zi, zim1));
    };
    const unsigned full_mask = 0xffffffffu;
    int base = 0;
    auto one_cell = [&](int a, int e) {  // the cell's candidates by all lanes, a ballot per 32
        for (int j0 = a; j0 < e; j0 += 32) {
            const int j = j0 + lane;
            const T r2 = j < e ? r2_of(j) : T(0);
            const bool h = j < e && j != self && r2 < R2;
            const unsigned m = __ballot_sync(full_mask, h);
            if (h) emit(base + __popc(m & ((1u << lane) - 1u)), j, r2);
            base += __popc(m);
        }
    };
    if (w.ncube >= kLaneCells) {
        for (int f0 = 0; f0 < w.ncube; f0 += 32 * kAhead) {
            int2 ses[kAhead];
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int f = f0 + 32 * u + lane;
                ses[u] = make_int2(0, 0);
                if (f < w.ncube) {
                    int cx, cy, cz;
                    w.coords(f, cx, cy, cz);
                    ses[u] = w.range(cells, cx, cy, cz, xf, yf, zf);
                }
            }
#pragma unroll 1
            for (int u = 0; u < kAhead; ++u) {
                const int2 se = u == 0 ? ses[0] : (u == 1 ? ses[1] : (u == 2 ? ses[2] : ses[3]));
                if (!__any_sync(full_mask, se.y > se.x)) continue;
                if (__any_sync(full_mask, se.y - se.x > 32)) {  // crowded cells: one after another
                    for (int l = 0; l < 32; ++l)
                        one_cell(__shfl_sync(full_mask, se.x, l), __shfl_sync(full_mask, se.y, l));
                    continue;
                }
                // the cell's hits, four candidates tested at a time
                unsigned m = 0;
                const int nj = se.y - se.x;
                for (int j0 = se.x; j0 < se.y; j0 += 4) {
                    T r2[4];
#pragma unroll
                    for (int v = 0; v < 4; ++v) r2[v] = r2_of(min(j0 + v, se.y - 1));
                    unsigned n4 = 0;
#pragma unroll
                    for (int v = 0; v < 4; ++v) n4 |= (unsigned)(r2[v] < R2) << v;
                    m |= n4 << (j0 - se.x);
                }
                if (nj < 32) m &= (1u << nj) - 1u;  // (the last four repeat the last candidate)
                if (self >= se.x && self < se.y) m &= ~(1u << (self - se.x));
                const int cnt = __popc(m);
                int pre = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(full_mask, pre, o);
                    if (lane >= o) pre += y;
                }
                const int total = __shfl_sync(full_mask, pre, 31);
                int k = base + pre - cnt;
                for (; m; m &= m - 1) {
                    const int j = se.x + __ffs(m) - 1;
                    emit(k++, j, r2_of(j));
                }
                base += total;
            }
        }
    } else {
        for (int f = 0; f < w.ncube; ++f) {
            int cx, cy, cz;
            w.coords(f, cx, cy, cz);
            const int2 se = w.range(cells, cx, cy, cz, xf, yf, zf);  // (the same for every lane)
            one_cell(se.x, se.y);
        }
    }
    return base;
}

}  // namespace gz
