// Hierarchical (power-of-two) timesteps: one sync interval of 2^K substeps
// built on the step's passes.  Reading of the method's hierarchical adaptive
// timesteps (the paper gives no formula):
//   - particle i sits in bin k_i in [0, K], step dt_i = D/2^k_i, and is active
//     at substep s when s is a multiple of 2^(K - k_i);
//   - substep 0: every particle is active; D = dt_fixed, or
//     min(cfl max_i dtc_i, 2^K cfl min_i dtc_i) per box (dtc the O13 criterion);
//     k_i = smallest k with D/2^k <= cfl dtc_i (K at most).  Later active
//     times may only deepen a bin;
//   - the caller's x holds each particle's position at the start of its
//     current step; at substep s every particle is placed at
//     x + (s - s_a) D/2^K * v_bar, v_bar = (v_start + v)/2, and a step that
//     ends moves x by dt_i v_bar (the trapezoid drift of O14);
//   - active particles run O4-O9 and O13; the others keep H, n, gradients and
//     B of their last active time.  Every flux pair with an active particle
//     exchanges the O11/O12 face fluxes over dt_ij = D/2^max(k_i, k_j)
//     (Hancock with dt_ij/2): each side accumulates rate * 2^(k_a - k_ij)
//     (exact power-of-two scaling, so the two shares stay equal and opposite)
//     and kicks momentum and energy by dt_a times that sum.
// Any Riemann option of the MFM face, and MFV (the exchange uses pair_rates
// with them; under MFV the mass shares ride along and the kick advances m).
// K = 0 is gz_step bitwise.  Pair lists of an active particle: N_i from the
// density pass and the pairs with r >= H_i (r < H_j), written by the partner
// j from a scan of its own support; an inactive particle's list holds its
// active partners, written by them (atomic slot counters, then every such
// list sorted by index, so every sum runs in a fixed order).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "gz_device.cuh"
#include "gz_launch.cuh"

namespace gz {

namespace {

inline int nblk(int n, int t) { return (n + t - 1) / t; }

constexpr int kCmpBlock = 1024;

template <typename T>
__device__ __forceinline__ T wrap_pos(T v) {
    if (v < T(0)) v += T(1);
    if (v >= T(1)) v -= T(1);
    return v;
}

// ------------------------------------------------------ interval start
template <typename T>
__global__ void k_h_init(int N, gz_particles p, T* hva, T* hdvs,
                         int* hsa, int* hbin) {
    after_previous();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= N) return;
    hva[o] = ((const T*)p.vx)[o];
    hva[(size_t)N + o] = ((const T*)p.vy)[o];
    hva[2 * (size_t)N + o] = ((const T*)p.vz)[o];
    hdvs[o] = hdvs[(size_t)N + o] = hdvs[2 * (size_t)N + o] = T(0);
    hsa[o] = 0;
    hbin[o] = 0;
}

// Mean velocity of the current step so far: (v_start + v)/2 (FP64), or
// v_start + dv/2 with the accumulated change dv (FP32, the increment form).
template <typename T>
__device__ __forceinline__ T vbar(T va, T v, T dvs) {
    if constexpr (std::is_same<T, float>::value)
        return va + 0.5f * dvs;
    else
        return 0.5 * (va + v);
}

// Predicted positions of every particle at substep s (caller order).
template <typename T>
__global__ void k_h_predict(int N, int s, int K, gz_particles p, const T* hva,
                            const T* hdvs, const int* hsa,
                            const int* box_of, const double* D, T* xp) {
    after_previous();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o < N) {
        const int steps = s - hsa[o];
        const T* X[3] = {(const T*)p.x, (const T*)p.y, (const T*)p.z};
        const T* V[3] = {(const T*)p.vx, (const T*)p.vy, (const T*)p.vz};
        if (steps == 0) {
#pragma unroll
            for (int r = 0; r < 3; ++r) xp[(size_t)r * N + o] = X[r][o];
        } else {
            const double tau = ldexp(D[box_of[o]], -K) * (double)steps;
#pragma unroll
            for (int r = 0; r < 3; ++r) {
                const size_t q = (size_t)r * N + o;
                xp[q] = wrap_pos<T>(X[r][o] + (T)tau * vbar<T>(hva[q], V[r][o], hdvs[q]));
            }
        }
    }
}

// Number of particles active at substep s, once the bins up to it are final.
__global__ void k_h_count(int N, int s, int K, const int* hbin, int* count) {
    after_previous();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    const int c = __syncthreads_count(o < N && s % (1 << (K - hbin[o])) == 0);
    if (threadIdx.x == 0 && c) atomicAdd(count, c);
}

// Sorted bins and active flags, and the flags' counts per compaction block.
__global__ void __launch_bounds__(kCmpBlock)
    k_h_flags(int N, int s, int K, const unsigned* orig, const int* hbin,
              int* sbin, unsigned char* aflag, int* bcount) {
    after_previous();
    const int i = blockIdx.x * kCmpBlock + threadIdx.x;
    bool act = false;
    if (i < N) {
        const int b = hbin[orig[i]];
        sbin[i] = b;
        act = s % (1 << (K - b)) == 0;
        aflag[i] = (unsigned char)act;
    }
    const int c = __syncthreads_count(act);
    if (threadIdx.x == 0) bcount[blockIdx.x] = c;
}

// ------------------------------------------- ordered stream compaction
// flag -> list of the flagged indices in increasing order: per-block counts
// (by the kernel that sets the flags), their scan (by every writing block for
// itself up to kCmpDirect blocks, else by one block), per-block writes (warp
// ballots within a block).
constexpr int kCmpDirect = 4096;

__global__ void __launch_bounds__(kCmpBlock) k_cmp_scan(int nb, int* bcount, int* total) {
    after_previous();
    __shared__ int part[kCmpBlock];
    const int t = threadIdx.x;
    const int chunk = (nb + kCmpBlock - 1) / kCmpBlock;
    const int b0 = min(nb, t * chunk), b1 = min(nb, b0 + chunk);
    int sum = 0;
    for (int b = b0; b < b1; ++b) sum += bcount[b];
    part[t] = sum;
    __syncthreads();
    for (int off = 1; off < kCmpBlock; off <<= 1) {  // inclusive scan (Hillis-Steele)
        const int v = t >= off ? part[t - off] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    int run = part[t] - sum;  // exclusive prefix of this thread's chunk
    for (int b = b0; b < b1; ++b) {
        const int c = bcount[b];
        bcount[b] = run;
        run += c;
    }
    if (t == kCmpBlock - 1) *total = part[t];
}

// total non-null: boff holds the counts, and the last block writes their sum.
__global__ void __launch_bounds__(kCmpBlock)
    k_cmp_write(int N, const unsigned char* flag, const int* boff,
                int* list, int* total) {
    after_previous();
    __shared__ int wsum[kCmpBlock / 32];
    int base = 0;
    if (total) {
        int v = 0;
        for (int b = threadIdx.x; b < (int)blockIdx.x; b += kCmpBlock) v += boff[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
        __syncthreads();
        for (int w2 = 0; w2 < kCmpBlock / 32; ++w2) base += wsum[w2];
        __syncthreads();
        if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = base + boff[blockIdx.x];
    } else {
        base = boff[blockIdx.x];
    }
    const int i = blockIdx.x * kCmpBlock + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool f = i < N && flag[i];
    const unsigned ball = __ballot_sync(0xffffffffu, f);
    if (lane == 0) wsum[w] = __popc(ball);
    __syncthreads();
    if (w == 0) {  // exclusive scan of the warp counts
        const int v = wsum[lane];
        int x = v;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, off);
            if (lane >= off) x += y;
        }
        wsum[lane] = x - v;
    }
    __syncthreads();
    if (f) list[base + wsum[w] + __popc(ball & ((1u << lane) - 1u))] = i;
}

// --------------------------------------------------------- pair lists
// Smallest support radius among every cell's active particles (+inf without
// any), rounded down; 0 for a crowded cell with one, whose particles one thread
// would walk (a state that went to NaN, 64^3: 12 ms).
template <typename T>
__global__ void k_h_cellmin(int ncells, const int2* cells, const unsigned char* aflag,
                            const P4<T>* pos, float* cellmin) {
    after_previous();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncells) return;
    const int2 se = cells[c];
    float h = INFINITY;
    if (se.y - se.x > kCrowdCell) {  // (0: the cell is only never skipped)
        for (int i = se.x; i < se.y && h > 0.f; ++i)
            if (aflag[i]) h = 0.f;
    } else {
        for (int i = se.x; i < se.y; ++i)
            if (aflag[i]) {
                if constexpr (sizeof(T) == 8)
                    h = fminf(h, __double2float_rd(pos[i].w));
                else
                    h = fminf(h, pos[i].w);
            }
    }
    cellmin[c] = h;
}

// Cells within two cells (per axis, periodic) of a cell holding an active
// particle, marked by the active cells themselves (near must start zeroed).
__global__ void k_h_dilate(int ncells, const BoxInfo* boxes, int nboxes,
                           const float* cellmin, unsigned char* near) {
    after_previous();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncells || cellmin[c] == INFINITY) return;
    int lo = 0, hi = nboxes - 1;  // box of the cell: last box with cell_off <= c
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (boxes[mid].cell_off <= c)
            lo = mid;
        else
            hi = mid - 1;
    }
    const BoxInfo bx = boxes[lo];
    const int nc = bx.nc, l = c - bx.cell_off;
    const int cx = l % nc, cy = (l / nc) % nc, cz = l / (nc * nc);
    for (int dz = -2; dz <= 2; ++dz) {
        const int wz = ((cz + dz) % nc + nc) % nc;
        for (int dy = -2; dy <= 2; ++dy) {
            const int wy = ((cy + dy) % nc + nc) % nc;
            for (int dx = -2; dx <= 2; ++dx) {
                const int wx = ((cx + dx) % nc + nc) % nc;
                near[bx.cell_off + (wz * nc + wy) * nc + wx] = 1;
            }
        }
    }
}

template <typename T>
__device__ __forceinline__ int cell_of(T v, int nc) {
    T f = floor(v * (T)nc);
    if (!(f >= T(0))) return 0;
    if (f > (T)(nc - 1)) return nc - 1;
    return (int)f;
}

// The flux pairs of active i with r >= H_i (so r < H_j, O10), found from the
// partner's side: every particle j scans its own support and appends itself to
// the list of each active i there with r >= H_i; the lists are put in index
// order by k_h_sort.  r^2 is the bit pattern the density pass forms for the
// pair, so these lists and N_i split the flux pairs exactly.  Cells whose
// active particles all have H >= H_j hold no such pair and are skipped.  An
// active j needs no scan: its N_j, which the density pass has just listed,
// holds every such i.  Sixteen lanes share a particle's cells, or its list: a
// blast's emptied centre spans up to thousands of cells, and with one thread
// each the launch waited for those (Sedov 64^3, an interval's lists of 16
// substeps, late in the run: one thread 9.6 ms, 4 lanes 6.2, 8 lanes 5.1, 16
// lanes 4.7; active particles by their lists 2.75).
constexpr int kScatterLanes = 16;
template <typename T>
__global__ void __launch_bounds__(128)
    k_h_rscatter(int N, Sorted<T> s, Grid g, KParams p, const unsigned* nbr,
                 const int* ncount, const unsigned char* aflag,
                 const float* cellmin, const unsigned char* near,
                 unsigned* rnbr, int* rcount, DevStatus* st) {
    after_previous();
    const int gl = threadIdx.x % kScatterLanes;
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) / kScatterLanes;
    if (j >= N) return;
    const P4<T> me = s.pos[j];
    const T xm1 = me.x - T(1), ym1 = me.y - T(1), zm1 = me.z - T(1);
    auto append = [&](int i) {
        const int slot = atomicAdd(&rcount[i], 1);
        if (slot < p.rcap)
            rnbr[lslot(slot, i, N)] = (unsigned)j;
        else
            set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, s.id[i]);
    };
    if (aflag[j]) {  // its N_j holds every such i
        const int cnt = min(ncount[j], p.cap);
        const unsigned* L = nbr + 4 * (size_t)j;
        for (int k0 = 4 * gl; k0 < cnt; k0 += 4 * kScatterLanes) {
            const uint4 jj = col4(L, k0, N);
            const unsigned is[4] = {jj.x, jj.y, jj.z, jj.w};
            P4<T> q[4];
            bool in[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const unsigned i = k0 + u < cnt ? is[u] : (unsigned)j;
                q[u] = s.pos[i];
                in[u] = k0 + u < cnt && aflag[i];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const T r2 = sep2(mi_diff(q[u].x, me.x, xm1), mi_diff(q[u].y, me.y, ym1), mi_diff(q[u].z, me.z, zm1));
                if (in[u] && !(r2 < q[u].w * q[u].w)) append((int)is[u]);
            }
        }
        return;
    }
    const BoxInfo bx = g.boxes[s.box[j]];
    const T Hj = me.w;
    // a support spanning under two cells lies within two cells of its own
    // (the scan's range floor((x -+ H) nc -+ 1e-3)): without an active cell
    // there, nothing to append
    if (Hj * (T)bx.nc < T(1.99)) {
        const int nc = bx.nc;
        if (!near[bx.cell_off + (cell_of(me.z, nc) * nc + cell_of(me.y, nc)) * nc + cell_of(me.x, nc)]) return;
    }
    const T H2 = Hj * Hj;
    const float Hf = (float)Hj * (1.f + 1e-6f);  // (not below H_j)
    const float xf = chop(me.x), yf = chop(me.y), zf = chop(me.z);
    const Window<T> w(bx.nc, me.x, me.y, me.z, Hj);
    for (int f = gl; f < w.ncube; f += kScatterLanes) {
        int cx, cy, cz;
        w.coords(f, cx, cy, cz);
        const int lc = w.wrapped(cx, cy, cz);
        if (!(cellmin[bx.cell_off + lc] < Hf)) continue;
        const int2 se = w.range(g.cells + bx.cell_off, cx, cy, cz, xf, yf, zf);
        for (int i0 = se.x; i0 < se.y; i0 += 4) {  // four candidates' loads in flight at a time
            P4<T> q[4];
            unsigned char act[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = min(i0 + u, se.y - 1);
                q[u] = s.pos[i];
                act[u] = aflag[i];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u;
                const T r2 = sep2(mi_diff(q[u].x, me.x, xm1), mi_diff(q[u].y, me.y, ym1), mi_diff(q[u].z, me.z, zm1));
                if (i >= se.y || i == j || !act[u] || !(r2 < H2) || r2 < q[u].w * q[u].w) continue;
                append(i);
            }
        }
    }
}

// Active i appends itself to the list of each inactive partner: thread (t, y)
// takes list groups y, y + kInGroups, ... (four slots each) of active particle t.
constexpr int kInGroups = 8;
__global__ void k_h_inlist(const int* alist, const int* nA,
                           const unsigned char* aflag, unsigned* nbr,
                           int* ncount, const unsigned* rnbr,
                           const int* rcount, int cap, int rcap,
                           const long long* sid, int N, DevStatus* st) {
    after_previous();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= *nA) return;
    const int i = alist[t];
    for (int list = 0; list < 2; ++list) {
        const unsigned* L = list == 0 ? nbr + 4 * (size_t)i : rnbr + 4 * (size_t)i;
        const int n = list == 0 ? min(ncount[i], cap) : min(rcount[i], rcap);
        for (int k0 = 4 * threadIdx.y; k0 < n; k0 += 4 * kInGroups) {
            const uint4 jj = col4(L, k0, N);
            const unsigned js[4] = {jj.x, jj.y, jj.z, jj.w};
            bool in[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) in[u] = k0 + u < n && !aflag[js[u]];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!in[u]) continue;
                const int j = (int)js[u];
                const int slot = atomicAdd(&ncount[j], 1);
                if (slot < cap)
                    nbr[lslot(slot, j, N)] = (unsigned)i;
                else
                    set_status(st, GZ_S_NBR_OVERFLOW, GZ_C_NBR_OVERFLOW, sid[j]);
            }
        }
    }
}

// Index order for the lists written by other threads: the inactive
// particles' partner lists and the active particles' r >= H_i pairs.
__global__ void __launch_bounds__(kListBlock)
    k_h_sort(int N, const unsigned char* aflag, int* ncount,
             unsigned* nbr, int cap, const int* rcount,
             unsigned* rnbr, int rcap) {
    after_previous();
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) / kListLanes;
    if (i >= N) return;
    unsigned* L;
    int n;
    if (aflag[i]) {
        L = rnbr + 4 * (size_t)i;
        n = min(rcount[i], rcap);
    } else {
        n = min(ncount[i], cap);
        L = nbr + 4 * (size_t)i;
    }
    sort_list(L, n, N);
    if (!aflag[i] && threadIdx.x % kListLanes == 0) ncount[i] = n;
}

// Touched particles (active, or with an active partner), and their counts per
// compaction block.
__global__ void __launch_bounds__(kCmpBlock)
    k_h_tflags(int N, const unsigned char* aflag, const int* ncount,
               unsigned char* tflag, int* bcount) {
    after_previous();
    const int i = blockIdx.x * kCmpBlock + threadIdx.x;
    const bool t = i < N && (aflag[i] || ncount[i] > 0);
    if (i < N) tflag[i] = (unsigned char)t;
    const int c = __syncthreads_count(t);
    if (threadIdx.x == 0) bcount[blockIdx.x] = c;
}

// ----------------------------------------------- per-particle bookkeeping
// Active particles keep what the inactive ones will read later: H (into the
// caller's h), n, the limited gradients and B (from the flux record).
template <typename T>
__global__ void k_h_persist(int N, const int* alist, const int* nA,
                            Sorted<T> s, const T* rec, gz_particles p, T* hn,
                            T* hgrad, T* hB) {
    after_previous();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= *nA) return;
    const int i = alist[t];
    const unsigned o = s.orig[i];
    T R[kRecord];
    load_rec(rec, i, R);
#pragma unroll
    for (int q = 0; q < 15; ++q) hgrad[(size_t)q * N + o] = R[11 + q];
#pragma unroll
    for (int q = 0; q < 6; ++q) hB[(size_t)q * N + o] = R[26 + q];
    hn[o] = s.n[i];
    ((T*)p.h)[o] = s.h[i];
}

// Largest finite criterion of every box (substep 0): a warp's maximum in one
// atomic when the warp lies in one box (positive doubles order like their
// bit patterns).
__global__ void k_h_dtmax(const int* alist, const int* nA,
                          const int* box, const double* dti,
                          unsigned long long* dtmax) {
    after_previous();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const bool in = t < *nA;
    const int i = in ? alist[t] : 0;
    const double v = in ? dti[i] : 0.0;
    unsigned long long bits = (in && isfinite(v) && v > 0.0) ? (unsigned long long)__double_as_longlong(v) : 0ull;
    const int b = in ? box[i] : -1;
    const unsigned full = 0xffffffffu;
    const int b0 = __shfl_sync(full, b, 0);
    if (__all_sync(full, !in || b == b0)) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long w = __shfl_xor_sync(full, bits, o);
            bits = w > bits ? w : bits;
        }
        if ((threadIdx.x & 31) == 0 && b0 >= 0 && bits) atomicMax(&dtmax[b0], bits);
    } else if (in && bits) {
        atomicMax(&dtmax[b], bits);
    }
}

// Interval per box: min(cfl max dtc, 2^K cfl min dtc).
__global__ void k_h_interval(int nb, const unsigned long long* dtmin,
                             const unsigned long long* dtmax, double cfl, int K,
                             double* D) {
    after_previous();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    const double lo = __longlong_as_double((long long)dtmin[b]);
    const double hi = dtmax[b] ? __longlong_as_double((long long)dtmax[b]) : 0.0;
    const double a = cfl * hi, c = ldexp(cfl * lo, K);
    D[b] = a < c ? a : c;
}

__device__ __forceinline__ int bin_for(double D, double cfl_dtc, int K) {
    for (int k = 0; k <= K; ++k)
        if (ldexp(D, -k) <= cfl_dtc) return k;
    return K;
}

// Bins of the active particles: assigned at substep 0, deepened later.
__global__ void k_h_bins(const int* alist, const int* nA,
                         const unsigned* orig, const int* box,
                         const double* dti, const double* D, double cfl, int K,
                         int first, int* hbin, int* sbin) {
    after_previous();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= *nA) return;
    const int i = alist[t];
    int k = bin_for(D[box[i]], cfl * dti[i], K);
    if (!first) k = max(k, sbin[i]);
    sbin[i] = k;
    hbin[orig[i]] = k;
}

// ------------------------------------------------------------ exchange
constexpr int kXBlock = 128;

// 2^e for the levels' small e, without FP64 arithmetic in the FP32 passes.
template <typename T>
__device__ __forceinline__ T pow2_(int e) {
    if constexpr (sizeof(T) == 4)
        return __int_as_float((127 + e) << 23);
    else
        return __hiloint2double((1023 + e) << 20, 0);
}

// Touched particle i over its pair lists (an active particle: N_i then its
// r >= H_i pairs; an inactive one: its active partners): the pair's face
// fluxes with the Hancock half step of dt_ij, scaled by 2^(k_i - k_ij),
// summed like the flux pass (sum_runs).  kRiem: the MFM face's Riemann solver;
// kMFV: the MFV fluxes, whose mass share is summed too (pair_rates).  The
// powers of two are built from their exponents in the working precision (the
// same values): two FP64 scalings and conversions a pair, at 1/64 of the FP32
// rate, were half of the FP32 pass (Sedov 64^3, 16 substeps late in the run:
// 2.86 ms with them, 1.61 without, 1.59 with the next record ahead).
template <typename T, int kRiem, bool kMFV, bool kSplit>
__global__ void __launch_bounds__(kXBlock, kLoadAhead<T, kMFV, kRiem> ? 3 : 1)
    k_h_exchange(const int* tlist, const int* nT, const T* rec,
                 const long long* sid, const int* sbox,
                 const int* sbin, const unsigned* nbr,
                 const int* ncount, const unsigned* rnbr,
                 const int* rcount, KParams p, const double* D,
                 double* dpdt, double* dEdt, double* dmdt, int N,
                 DevStatus* st) {
    after_previous();
    constexpr int nq = kMFV ? 5 : 4;
    const int t = flux_item<kSplit>(), n = *nT;
    if (kSplit ? (int)blockIdx.x * 32 >= n : t >= n) return;
    const int i = tlist[min(t, n - 1)];  // (kSplit: spare threads repeat a particle, with no pairs)
    T a[kRecord];
    load_rec(rec, i, a);
    const long long idi = kMFV ? sid[i] : 0;  // (MFV pairs are oriented by id)
    const int ka = sbin[i];
    const T hD = p.hancock ? (T)(0.5 * D[sbox[i]]) : T(0);
    const T gam = (T)p.gamma;
    const int cnt = t < n ? min(ncount[i], p.cap) : 0, rcnt = t < n ? min(rcount[i], p.rcap) : 0;
    int nfall = 0, nneg = 0;
    auto pair = [&](const T(&b)[kRecord], int j, T(&run)[nq]) {
        const int kab = max(ka, sbin[j]);
        const T hdt = hD * pow2_<T>(-kab);
        T ia[5];
        half_inc(a, hdt, gam, ia);
        T dp[3], dE, dm;
        int fl = 0;
        const bool aL = pair_order<kMFV>(i, j, idi, sid);
        if (pair_rates<T, kMFV, kRiem>(a, b, ia, aL, hdt, gam, dp, dE, dm, fl)) {
            const T sc = pow2_<T>(ka - kab);
            run[0] += dp[0] * sc;
            run[1] += dp[1] * sc;
            run[2] += dp[2] * sc;
            run[3] += dE * sc;
            if constexpr (kMFV) run[4] += dm * sc;
        }
        nfall += fl & 1;
        nneg += (fl >> 1) & 1;
    };
    if constexpr (kSplit) {
        const Totals<2> s = sum_runs_split<T, nq, kPairUnroll<kRiem>>(i, N, rec, nbr, cnt, rnbr, rcnt, pair);
        if (t < n) store_rates_split<nq>(s.v, i, N, dpdt, dEdt, dmdt);
    } else {
        const Totals<nq> s = sum_runs<T, nq, kLoadAhead<T, kMFV, kRiem>, kPairUnroll<kRiem>>(i, N, rec, nbr, cnt, rnbr, rcnt, pair);
        store_rates<nq>(s.v, i, N, dpdt, dEdt, dmdt);
    }
    count_flags(st, nfall, nneg);
}

// Kick of a touched particle by dt_i times its scaled sums: the O14 momentum
// and energy update without the drift (FP64 literal form; FP32 increments,
// which also accumulate the step's velocity change for the drift).
template <typename T>
__global__ void k_h_kick(const int* tlist, const int* nT, int N, Sorted<T> s,
                         const int* sbin, const double* dpdt,
                         const double* dEdt, const double* dmdt,
                         const double* D, gz_particles out, T* hdvs,
                         int* box_hits, DevStatus* st) {
    after_previous();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= *nT) return;
    const int i = tlist[t];
    const unsigned o = s.orig[i];
    const int b = s.box[i];
    const double dt = ldexp(D[b], -sbin[i]);
    const double dpx = dpdt[i], dpy = dpdt[(size_t)N + i], dpz = dpdt[2 * (size_t)N + i], dE = dEdt[i];
    T vx = s.vx[i], vy = s.vy[i], vz = s.vz[i], u = s.u[i];
    T m = s.m[i];
    if constexpr (std::is_same<T, float>::value) {
        float dvx, dvy, dvz;
        if (dmdt)
            kick_one_mfv(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dmdt[i], dt, dvx, dvy, dvz);
        else
            kick_one(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dt, dvx, dvy, dvz);
        hdvs[o] = __fadd_rn(hdvs[o], dvx);
        hdvs[(size_t)N + o] = __fadd_rn(hdvs[(size_t)N + o], dvy);
        hdvs[2 * (size_t)N + o] = __fadd_rn(hdvs[2 * (size_t)N + o], dvz);
    } else {
        if (dmdt)
            kick_one_mfv(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dmdt[i], dt);
        else
            kick_one(m, vx, vy, vz, u, dpx, dpy, dpz, dE, dt);
    }
    if (dmdt) ((T*)out.m)[o] = m;
    ((T*)out.vx)[o] = vx;
    ((T*)out.vy)[o] = vy;
    ((T*)out.vz)[o] = vz;
    ((T*)out.u)[o] = u;
    if (!(u > T(0))) {
        atomicAdd(&box_hits[b], 1);
        set_status(st, GZ_S_UFLOOR, GZ_C_UFLOOR, -1);
    }
    if (!(m > T(0) && finite_(vx) && finite_(vy) && finite_(vz) && finite_(u)))
        set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, s.id[i]);
}

// End of the steps that finish after substep s: drift by dt_i v_bar, new
// step start (caller order).
template <typename T>
__global__ void k_h_finalize(int N, int s, int K, gz_particles p, T* hva, T* hdvs,
                             int* hsa, const int* hbin,
                             const int* box_of, const double* D, DevStatus* st) {
    after_previous();
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= N) return;
    const int k = hbin[o];
    if ((s + 1) % (1 << (K - k)) != 0) return;
    const double dt = ldexp(D[box_of[o]], -k);
    T* X[3] = {(T*)p.x, (T*)p.y, (T*)p.z};
    const T* V[3] = {(const T*)p.vx, (const T*)p.vy, (const T*)p.vz};
    bool ok = true;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        const size_t q = (size_t)r * N + o;
        T x;
        if constexpr (std::is_same<T, float>::value)
            x = drift_onef(X[r][o], hva[q], hdvs[q], dt);
        else
            x = drift_one(X[r][o], hva[q], V[r][o], dt);
        X[r][o] = x;
        ok = ok && finite_(x);
        hva[q] = V[r][o];
        hdvs[q] = T(0);
    }
    hsa[o] = s + 1;
    if (!ok) set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, (long long)p.id[o]);
}

template <typename T>
void launch_exchange(Ctx& c, const KParams& kp, int N, int nA) {
    const int r = c.params.riemann;
    const bool split = nA < kFluxSplit;
    auto go = [&](auto one, auto four) {
        auto kernel = split ? four : one;
        launch_next(c, kernel, nblk(N, split ? 32 : kXBlock), kXBlock, c.tlist, c.hcount + 2, (const T*)c.rec, c.sid, c.sbox,
                    c.sbin, c.nbr, c.ncount, c.rnbr, c.rcount, kp, c.dt_use,
                    c.dpdt, c.dEdt, c.dmdt, N, c.status);
    };
    if (c.params.scheme == GZ_MFV)
        go(k_h_exchange<T, GZ_RIEMANN_HLLC, true, false>, k_h_exchange<T, GZ_RIEMANN_HLLC, true, true>);
    else if (r == GZ_RIEMANN_EXACT)
        go(k_h_exchange<T, GZ_RIEMANN_EXACT, false, false>, k_h_exchange<T, GZ_RIEMANN_EXACT, false, true>);
    else if (r == GZ_RIEMANN_FALLBACK)
        go(k_h_exchange<T, GZ_RIEMANN_FALLBACK, false, false>, k_h_exchange<T, GZ_RIEMANN_FALLBACK, false, true>);
    else
        go(k_h_exchange<T, GZ_RIEMANN_HLLC, false, false>, k_h_exchange<T, GZ_RIEMANN_HLLC, false, true>);
}

}  // namespace

cudaError_t ensure_hier_scratch(Ctx& c) {
    if (c.hier_arena) return cudaSuccess;
    // sized for the context's capacity (a subdomain context's N changes)
    const size_t Nz = (size_t)c.capacity, sz = c.precision == GZ_FP64 ? 8 : 4;
    const size_t nb = (size_t)nblk(c.capacity, kCmpBlock);
    struct Item {
        void** ptr;
        size_t bytes;
    } items[] = {
        {&c.hxp, 3 * sz * Nz},         {&c.hva, 3 * sz * Nz},        {&c.hdvs, 3 * sz * Nz},
        {&c.hn, sz * Nz},              {&c.hgrad, 15 * sz * Nz},     {&c.hB, 6 * sz * Nz},
        {(void**)&c.hsa, 4 * Nz},      {(void**)&c.hbin, 4 * Nz},    {(void**)&c.sbin, 4 * Nz},
        {(void**)&c.alist, 4 * Nz},    {(void**)&c.tlist, 4 * Nz},   {(void**)&c.hcount, 4 * 4},
        {(void**)&c.bcount, 4 * nb},   {(void**)&c.aflag, Nz},       {(void**)&c.tflag, Nz},
        {(void**)&c.cellmin, 4 * (size_t)c.total_cells}, {(void**)&c.cellnear, (size_t)c.total_cells},
        {(void**)&c.dtmax, 8 * (size_t)c.nboxes},
    };
    size_t total = 0;
    for (auto& it : items) total += (it.bytes + 255) & ~(size_t)255;
    void* base = nullptr;
    cudaError_t e = cudaMalloc(&base, total);
    if (e != cudaSuccess) return e;
    e = cudaMallocHost((void**)&c.hcount_host, 4 * sizeof(int));
    if (e == cudaSuccess && !c.hier_counted) {
        e = cudaEventCreateWithFlags(&c.hier_counted, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            cudaFreeHost(c.hcount_host);
            c.hcount_host = nullptr;
        }
    }
    if (e != cudaSuccess) {
        cudaFree(base);
        return e;
    }
    char* q = (char*)base;
    for (auto& it : items) {
        *it.ptr = q;
        q += (it.bytes + 255) & ~(size_t)255;
    }
    c.hier_arena = base;
    return cudaSuccess;
}

// The list of the flagged particles, from the flags' block counts in c.bcount.
static cudaError_t compact(Ctx& c, const unsigned char* flag, int* list, int* count) {
    const int nb = nblk(c.N, kCmpBlock);
    const bool direct = nb <= kCmpDirect;
    c.launches += direct ? 1 : 2;
    if (!direct) launch_next(c, k_cmp_scan, 1, kCmpBlock, nb, c.bcount, count);
    launch_next(c, k_cmp_write, nb, kCmpBlock, c.N, flag, c.bcount, list, direct ? count : nullptr);
    return cudaGetLastError();
}

template <typename T>
cudaError_t run_step_hier(Ctx& c, gz_particles& p, int K, double dt_fixed, double* dt_used_dev,
                          int32_t* bins_out, long long* active_out, const PassTimer& timer) {
    cudaError_t e = ensure_hier_scratch(c);
    if (e != cudaSuccess) return e;
    const int N = c.N;
    cudaStream_t st = c.stream;
    const KParams kp = kparams(c);
    Grid g;
    g.boxes = c.boxes;
    g.cells = c.cells;
    T* hxp = (T*)c.hxp;
    gz_particles pp = p;  // predicted positions, everything else the caller's arrays
    pp.x = hxp;
    pp.y = hxp + N;
    pp.z = hxp + 2 * (size_t)N;
    c.launches += 1;
    launch_next(c, k_h_init<T>, nblk(N, 256), 256, N, p, (T*)c.hva, (T*)c.hdvs, c.hsa, c.hbin);
    long long active = 0;
    const int S = 1 << K;
    int nA = N;  // (substep 0: every particle)
    for (int s = 0; s < S && e == cudaSuccess; ++s) {
        if (s > 0) {  // the count of this substep's active particles, formed after the last one's bins
            e = cudaEventSynchronize(c.hier_counted);
            if (e != cudaSuccess) break;
            nA = c.hcount_host[s & 1];
        }
        c.launches += 1;
        launch_next(c, k_h_predict<T>, nblk(N, 256), 256, N, s, K, p, (const T*)c.hva, (const T*)c.hdvs, c.hsa,
                    c.box_of, c.dt_use, hxp);
        active += nA;
        if (nA > 0) {
            Sorted<T> sv = sorted_view<T>(c);
            timer.begin(GZ_PASS_SORT);
            e = sort_and_bin<T>(c, pp, c.hn);
            c.launches += 1;
            launch_next(c, k_h_flags, nblk(N, kCmpBlock), kCmpBlock, N, s, K, c.vals, c.hbin, c.sbin, c.aflag, c.bcount);
            if (e == cudaSuccess) e = compact(c, c.aflag, c.alist, c.hcount + 1);
            timer.end(GZ_PASS_SORT);
            cudaMemsetAsync(c.ncount, 0, sizeof(int) * (size_t)N, st);
            timer.begin(GZ_PASS_DENSITY);
            if (e == cudaSuccess) e = run_density<T>(c, c.alist, c.hcount + 1, nA);
            timer.end(GZ_PASS_DENSITY);
            timer.begin(GZ_PASS_PRIM);
            if (e == cudaSuccess) e = run_prim<T>(c);
            timer.end(GZ_PASS_PRIM);
            timer.begin(GZ_PASS_REVERSE);
            c.launches += 6;
            c.launches += 1;
            launch_next(c, k_h_cellmin<T>, nblk(c.total_cells, 256), 256, c.total_cells, c.cells, c.aflag, sv.pos,
                        c.cellmin);
            cudaMemsetAsync(c.cellnear, 0, (size_t)c.total_cells, st);
            launch_next(c, k_h_dilate, nblk(c.total_cells, 256), 256, c.total_cells, c.boxes, c.nboxes, c.cellmin,
                        c.cellnear);
            launch_next(c, k_h_rscatter<T>, nblk(N, 128 / kScatterLanes), 128, N, sv, g, kp, c.nbr, c.ncount, c.aflag,
                        c.cellmin, c.cellnear, c.rnbr, c.rcount, c.status);
            launch_next(c, k_h_inlist, nblk(nA, 32), dim3(32, kInGroups), c.alist, c.hcount + 1, c.aflag, c.nbr, c.ncount,
                        c.rnbr, c.rcount, c.cap, c.rcap, c.sid, c.N, c.status);
            launch_next(c, k_h_sort, nblk(N, kListBlock / kListLanes), kListBlock, N, c.aflag, c.ncount, c.nbr, c.cap,
                        c.rcount, c.rnbr, c.rcap);
            launch_next(c, k_h_tflags, nblk(N, kCmpBlock), kCmpBlock, N, c.aflag, c.ncount, c.tflag, c.bcount);
            if (e == cudaSuccess) e = compact(c, c.tflag, c.tlist, c.hcount + 2);
            timer.end(GZ_PASS_REVERSE);
            timer.begin(GZ_PASS_GRAD);
            if (e == cudaSuccess) e = run_gradients<T>(c, true, false, c.alist, c.hcount + 1, nA);
            if (e == cudaSuccess)
                e = run_pack_given<T>(c, (const T*)c.hgrad, (const T*)c.hB, c.tlist, c.hcount + 2, N, c.aflag);
            c.launches += 1;
            launch_next(c, k_h_persist<T>, nblk(nA, 256), 256, N, c.alist, c.hcount + 1, sv, (const T*)c.rec, p,
                        (T*)c.hn, (T*)c.hgrad, (T*)c.hB);
            if (s == 0) {
                if (dt_fixed > 0.0) {
                    if (e == cudaSuccess) e = run_dt_set(c, dt_fixed);
                } else {
                    cudaMemsetAsync(c.dtmax, 0, 8 * (size_t)c.nboxes, st);
                    c.launches += 2;
                    launch_next(c, k_h_dtmax, nblk(nA, 256), 256, c.alist, c.hcount + 1, c.sbox, c.dti, c.dtmax);
                    launch_next(c, k_h_interval, nblk(c.nboxes, 256), 256, c.nboxes,
                                (const unsigned long long*)c.dt_box, c.dtmax, c.params.cfl, K, c.dt_use);
                }
            }
            c.launches += 1;
            launch_next(c, k_h_bins, nblk(nA, 256), 256, c.alist, c.hcount + 1, c.vals, c.sbox, c.dti, c.dt_use,
                        c.params.cfl, K, s == 0 ? 1 : 0, c.hbin, c.sbin);
            timer.end(GZ_PASS_GRAD);
        }
        if (s + 1 < S) {
            // the bins are final: the next substep's count goes to the host
            // while the exchange runs
            c.launches += 1;
            cudaMemsetAsync(c.hcount + 3, 0, sizeof(int), st);
            launch_next(c, k_h_count, nblk(N, 256), 256, N, s + 1, K, c.hbin, c.hcount + 3);
            cudaMemcpyAsync(c.hcount_host + ((s + 1) & 1), c.hcount + 3, sizeof(int), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaEventRecord(c.hier_counted, st);
        }
        if (nA > 0) {
            Sorted<T> sv = sorted_view<T>(c);
            timer.begin(GZ_PASS_FLUX);
            c.launches += 1;
            launch_exchange<T>(c, kp, N, nA);
            timer.end(GZ_PASS_FLUX);
            timer.begin(GZ_PASS_UPDATE);
            c.launches += 1;
            launch_next(c, k_h_kick<T>, nblk(N, 256), 256, c.tlist, c.hcount + 2, N, sv, c.sbin, c.dpdt, c.dEdt,
                        c.params.scheme == GZ_MFV ? c.dmdt : nullptr, c.dt_use,
                        p, (T*)c.hdvs, c.box_hits, c.status);
            if (e == cudaSuccess) e = run_ufloor<T>(c, p);
            timer.end(GZ_PASS_UPDATE);
        }
        c.launches += 1;
        launch_next(c, k_h_finalize<T>, nblk(N, 256), 256, N, s, K, p, (T*)c.hva, (T*)c.hdvs, c.hsa, c.hbin,
                    c.box_of, c.dt_use, c.status);
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (e == cudaSuccess && dt_used_dev)
        e = cudaMemcpyAsync(dt_used_dev, c.dt_use, sizeof(double) * (size_t)c.nboxes, cudaMemcpyDeviceToDevice,
                            st);
    if (e == cudaSuccess && bins_out)
        e = cudaMemcpyAsync(bins_out, c.hbin, sizeof(int) * (size_t)N, cudaMemcpyDeviceToDevice, st);
    c.nbr_valid = 0;  // the lists now mix active lists with partner lists
    if (active_out) *active_out = active;
    return e;
}

template cudaError_t run_step_hier<float>(Ctx&, gz_particles&, int, double, double*, int32_t*, long long*,
                                          const PassTimer&);
template cudaError_t run_step_hier<double>(Ctx&, gz_particles&, int, double, double*, int32_t*, long long*,
                                           const PassTimer&);

void free_hier_scratch(Ctx& c) {
    if (c.hier_arena) cudaFree(c.hier_arena);
    if (c.hcount_host) cudaFreeHost(c.hcount_host);
    if (c.hier_counted) cudaEventDestroy(c.hier_counted);
    c.hier_counted = nullptr;
    c.hier_arena = nullptr;
    c.hcount_host = nullptr;
}

}  // namespace gz
