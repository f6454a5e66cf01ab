// Binning, sort and permutation (step S1: particles are Morton-sorted into a
// uniform cell grid per box, in caller order within a cell, and the cells'
// ranges formed).  A counting sort over the keys where there are at most
// kKeysPerParticle keys a particle (every grid of about one support radius a
// cell), else a device LSD radix sort; both are stable and give one order.
#include <algorithm>

#include "gz_launch.cuh"

namespace gz {

namespace {

inline int blocks(int n, int t) { return (n + t - 1) / t; }

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kMaxDigitBits = 10;  // digits of up to 10 bits: 1024 buckets a pass
constexpr int kMaxDigits = 1 << kMaxDigitBits;
constexpr int kDigitsPerThread = kMaxDigits / kSortThreads;
constexpr int kSortTile = 4096;
constexpr int kSortPerWarp = kSortTile / kSortWarps;

// Spread the low 10 bits of v so that bit k lands on bit 3k.
__device__ __forceinline__ unsigned spread3(unsigned v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}
// Inverse of spread3.
__device__ __forceinline__ unsigned compact3(unsigned v) {
    v &= 0x09249249u;
    v = (v ^ (v >> 2)) & 0x030C30C3u;
    v = (v ^ (v >> 4)) & 0x0300F00Fu;
    v = (v ^ (v >> 8)) & 0x030000FFu;
    v = (v ^ (v >> 16)) & 0x000003FFu;
    return v;
}

template <typename T>
__device__ __forceinline__ int cell_coord(T v, int nc) {
    T s = floor(v * (T)nc);
    if (!(s >= T(0))) return 0;  // also NaN
    if (s > (T)(nc - 1)) return nc - 1;
    return (int)s;
}

// Sort key of a particle: its box's first key + the Morton index of its cell.
template <typename T>
__device__ __forceinline__ unsigned key_of(const BoxInfo& bx, T x, T y, T z) {
    return bx.key_off + (spread3(cell_coord(x, bx.nc)) | (spread3(cell_coord(y, bx.nc)) << 1) |
                         (spread3(cell_coord(z, bx.nc)) << 2));
}
template <typename T>
__device__ __forceinline__ bool inside(T x, T y, T z) {
    return x >= T(0) && x < T(1) && y >= T(0) && y < T(1) && z >= T(0) && z < T(1);
}

template <typename T>
__global__ void k_keys(int N, const T* __restrict__ x, const T* __restrict__ y,
                       const T* __restrict__ z, const int64_t* __restrict__ id,
                       const int* __restrict__ box_of, const BoxInfo* __restrict__ boxes,
                       unsigned* __restrict__ keys, unsigned* __restrict__ vals, DevStatus* st) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const T xv = x[i], yv = y[i], zv = z[i];
    if (!inside(xv, yv, zv)) set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, id[i]);
    keys[i] = key_of(boxes[box_of[i]], xv, yv, zv);
    vals[i] = (unsigned)i;
}

// ------------------------------------------------------- counting sort
// Key of every particle and its arrival number in its key's count (any order:
// k_permute puts the particles of a cell in caller order).  Behind the keys'
// counts: the number of crowded keys and of k_cs_place's finished blocks.
template <typename T>
__global__ void k_cs_count(int N, const T* __restrict__ x, const T* __restrict__ y, const T* __restrict__ z,
                           const int64_t* __restrict__ id, const int* __restrict__ box_of,
                           const BoxInfo* __restrict__ boxes, unsigned* __restrict__ count,
                           unsigned* __restrict__ key, unsigned* __restrict__ slot, DevStatus* st) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const T xv = x[i], yv = y[i], zv = z[i];
    if (!inside(xv, yv, zv)) set_status(st, GZ_S_NONFINITE, GZ_C_NONFINITE, id[i]);
    const unsigned k = key_of(boxes[box_of[i]], xv, yv, zv);
    key[i] = k;
    slot[i] = atomicAdd(&count[k], 1u);
}

constexpr int kScanThreads = 1024;
constexpr int kScanTile = 4 * kScanThreads;
constexpr int kScanDirect = 8;  // up to this many tiles, a block sums the counts before its own itself

__device__ __forceinline__ uint4 count4(const unsigned* count, long long k, long long K) {
    if (k + 3 < K) return *reinterpret_cast<const uint4*>(count + k);
    uint4 v = make_uint4(0, 0, 0, 0);
    if (k < K) v.x = count[k];
    if (k + 1 < K) v.y = count[k + 1];
    if (k + 2 < K) v.z = count[k + 2];
    return v;
}
// Sum over the block (every thread gets it).
__device__ __forceinline__ unsigned block_sum(unsigned v, unsigned* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned t = 0;
#pragma unroll
    for (int w = 0; w < kScanThreads / 32; ++w) t += sh[w];
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(kScanThreads)
    k_cs_sums(long long K, const unsigned* count, unsigned* sums) {
    after_previous();
    __shared__ unsigned sh[kScanThreads / 32];
    const uint4 v = count4(count, (long long)blockIdx.x * kScanTile + 4 * threadIdx.x, K);
    const unsigned t = block_sum(v.x + v.y + v.z + v.w, sh);
    if (threadIdx.x == 0) sums[blockIdx.x] = t;
}

// Particles of one key beyond which k_permute's walk of the cell (its number of
// steps squared) costs more than k_cs_place's last block sorting the cell.  The
// whole sort with every particle in one cell, walked / sorted: 32^3 584 / 113 us,
// 64^3 10314 / 513, 128^3 - / 3869 (a lattice: 19, 26 and 103).
constexpr int kCrowd = 16384;

// First sorted index of every key, the range of every cell (empty ones
// included) and the list of the crowded keys.  sums: the tiles' sums, or null
// when every block adds the counts before its tile itself.
__global__ void __launch_bounds__(kScanThreads)
    k_cs_scan(long long K, unsigned* count, const unsigned* sums, const BoxInfo* boxes, int nboxes,
              unsigned* start, int2* cells, unsigned* crowd) {
    after_previous();
    __shared__ unsigned sh[kScanThreads / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned before = 0;
    if (sums) {
        for (int b = t; b < (int)blockIdx.x; b += kScanThreads) before += sums[b];
    } else {
        for (int b = 0; b < (int)blockIdx.x; ++b) {
            const uint4 v = *reinterpret_cast<const uint4*>(count + (size_t)b * kScanTile + 4 * t);
            before += v.x + v.y + v.z + v.w;
        }
    }
    unsigned base = blockIdx.x ? block_sum(before, sh) : 0u;
    const long long k0 = (long long)blockIdx.x * kScanTile + 4 * t;
    const uint4 v = count4(count, k0, K);
    const unsigned c[4] = {v.x, v.y, v.z, v.w};
    const unsigned mine = (c[0] + c[1]) + (c[2] + c[3]);
    unsigned x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    for (int w = 0; w < warp; ++w) base += sh[w];
    unsigned s = base + x - mine;
    if (k0 >= K) return;
    int b = 0;  // box of the key: the last with key_off <= k0
    for (int hi = nboxes - 1; b < hi;) {
        const int mid = (b + hi + 1) >> 1;
        if (boxes[mid].key_off <= (unsigned)k0)
            b = mid;
        else
            hi = mid - 1;
    }
    BoxInfo bx = boxes[b];
    unsigned next = b + 1 < nboxes ? boxes[b + 1].key_off : 0xffffffffu;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const long long k = k0 + u;
        if (k >= K) break;
        while (b + 1 < nboxes && (unsigned)k >= next) {
            bx = boxes[++b];
            next = b + 1 < nboxes ? boxes[b + 1].key_off : 0xffffffffu;
        }
        start[k] = s;
        if (c[u] > kCrowd) crowd[atomicAdd(count + K, 1u)] = (unsigned)k;
        const unsigned mort = (unsigned)k - bx.key_off;
        const int cx = compact3(mort), cy = compact3(mort >> 1), cz = compact3(mort >> 2);
        if (cx < bx.nc && cy < bx.nc && cz < bx.nc)
            cells[bx.cell_off + (cz * bx.nc + cy) * bx.nc + cx] = make_int2((int)s, (int)(s + c[u]));
        s += c[u];
    }
}

// The n distinct caller indices (below N) of a crowded cell in increasing order,
// by one block: a bitmap of the N indices, whose set bits come out in order.
// (Written and read past L1, which does not see the atomics.)
__device__ __forceinline__ void sort_crowd(unsigned* seg, unsigned* bits, int n, int N) {
    __shared__ int wsum[32];
    const int t = threadIdx.x, T = blockDim.x, lane = t & 31, warp = t >> 5;
    const int words = (N - 1) / 32 + 1;
    for (int w = t; w < words; w += T) __stcg(bits + w, 0u);
    __syncthreads();
    for (int e = t; e < n; e += T) {
        const unsigned v = __ldcg(seg + e);  // (written by other blocks)
        atomicOr(bits + (v >> 5), 1u << (v & 31));
    }
    __syncthreads();
    int done = 0;
    for (int w0 = 0; w0 < words; w0 += T) {
        unsigned b = w0 + t < words ? __ldcg(bits + w0 + t) : 0u;
        const int mine = __popc(b);
        int x = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        int at = done + x - mine;
        for (int w = 0; w < T / 32; ++w) {
            if (w < warp) at += wsum[w];
            done += wsum[w];
        }
        for (; b; b &= b - 1) seg[at++] = 32u * (unsigned)(w0 + t) + (unsigned)(__ffs(b) - 1);
        __syncthreads();
    }
}

// Particles by key, in any order within a cell, except in crowded cells (a
// state that went to NaN is binned in one): once every block has placed its
// particles, the last one puts those in caller order.  crowd (N words): the
// crowded keys, then room for a bitmap of the particles.  Without crowded cells
// a block reads one word more.
__global__ void k_cs_place(int N, const unsigned* key, const unsigned* slot, const unsigned* start, unsigned* order,
                           unsigned* count, long long K, unsigned* crowd) {
    after_previous();
    __shared__ bool last;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int crowds = (int)count[K];
    if (i < N) order[start[key[i]] + slot[i]] = (unsigned)i;
    if (crowds == 0) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(count + K + 1, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int c = 0; c < crowds; ++c) {
        const unsigned k = crowd[c], a = start[k];
        sort_crowd(order + a, crowd + crowds, (int)count[k], N);
    }
}

// ----------------------------------------------------------- radix sort
// Digit counts of one tile (nd = 2^bits digits, mask = nd - 1).
__global__ void k_rs_hist(const unsigned* __restrict__ keys, int N, int shift, unsigned mask, int nd,
                          unsigned* __restrict__ hist, int nblk) {
    __shared__ unsigned h[kMaxDigits];
    for (int t = threadIdx.x; t < nd; t += blockDim.x) h[t] = 0;
    __syncthreads();
    const int base = blockIdx.x * kSortTile;
    for (int k = threadIdx.x; k < kSortTile; k += blockDim.x) {
        int e = base + k;
        if (e < N) atomicAdd(&h[(keys[e] >> shift) & mask], 1u);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nd; t += blockDim.x) hist[t * nblk + blockIdx.x] = h[t];
}

// Exclusive scan of one digit's row hist[d][0..nblk) (block d), and the row
// total into totals[d].
__global__ void k_rs_rows(unsigned* __restrict__ hist, int nblk, unsigned* __restrict__ totals) {
    __shared__ unsigned wsum[kSortWarps];
    __shared__ unsigned base_s;
    unsigned* row = hist + (size_t)blockIdx.x * nblk;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    unsigned running = 0;
    for (int b0 = 0; b0 < nblk; b0 += kSortThreads) {
        const int b = b0 + t;
        const unsigned v = b < nblk ? row[b] : 0u;
        unsigned x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        if (t == 0) {
            unsigned acc = 0;
            for (int w = 0; w < kSortWarps; ++w) {
                const unsigned ws = wsum[w];
                wsum[w] = acc;
                acc += ws;
            }
            base_s = acc;
        }
        __syncthreads();
        if (b < nblk) row[b] = running + wsum[warp] + x - v;
        running += base_s;
        __syncthreads();
    }
    if (t == 0) totals[blockIdx.x] = running;
}

// Stable scatter: each warp owns a contiguous sub-tile and walks it in order;
// lanes with equal digits are ranked with __match_any_sync.
__global__ void k_rs_scatter(const unsigned* __restrict__ kin, const unsigned* __restrict__ vin,
                             int N, int shift, unsigned mask, int nd, const unsigned* __restrict__ hist,
                             int nblk, const unsigned* __restrict__ totals, unsigned* __restrict__ kout,
                             unsigned* __restrict__ vout) {
    static_assert(kDigitsPerThread * kSortThreads == kMaxDigits, "whole digits per thread");
    __shared__ unsigned cnt[kSortWarps][kMaxDigits];
    __shared__ unsigned dbase[kMaxDigits];
    __shared__ unsigned wsum[kSortWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    {  // the nd digits of this pass (nd a power of 2)
        const int lg = __ffs(nd) - 1;
        for (int t = threadIdx.x; t < kSortWarps * nd; t += blockDim.x) cnt[t >> lg][t & (nd - 1)] = 0;
    }
    {  // exclusive scan of the nd digit totals, kDigitsPerThread consecutive digits a thread
        const int d0 = kDigitsPerThread * threadIdx.x;
        unsigned v[kDigitsPerThread];
        unsigned tv = 0;
#pragma unroll
        for (int u = 0; u < kDigitsPerThread; ++u) {
            v[u] = d0 + u < nd ? totals[d0 + u] : 0u;
            tv += v[u];
        }
        unsigned incl = tv;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        unsigned before = 0;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        unsigned run = before + incl - tv;
#pragma unroll
        for (int u = 0; u < kDigitsPerThread; ++u) {
            dbase[d0 + u] = run;
            run += v[u];
        }
    }
    __syncthreads();
    const int wbase = blockIdx.x * kSortTile + warp * kSortPerWarp;
    for (int c = 0; c < kSortPerWarp; c += 32) {
        int e = wbase + c + lane;
        if (e < N) atomicAdd(&cnt[warp][(kin[e] >> shift) & mask], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < nd; d += blockDim.x) {
        unsigned run = dbase[d] + hist[d * nblk + blockIdx.x];
        for (int w = 0; w < kSortWarps; ++w) {
            unsigned v = cnt[w][d];
            cnt[w][d] = run;
            run += v;
        }
    }
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    for (int c = 0; c < kSortPerWarp; c += 32) {
        const int e = wbase + c + lane;
        const bool valid = e < N;
        const unsigned vmask = __ballot_sync(0xffffffffu, valid);
        unsigned peers = 0, d = 0;
        if (valid) {
            const unsigned k = kin[e];
            d = (k >> shift) & mask;
            peers = __match_any_sync(vmask, d);
            const unsigned pos = cnt[warp][d] + __popc(peers & lt);
            kout[pos] = k;
            vout[pos] = vin[e];
        }
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) cnt[warp][d] += __popc(peers);
        __syncwarp();
    }
}

// The state in sorted order.  kCounted: p walks k_cs_place's order, a cell's
// particles in any order; a particle's place is its cell's start plus the
// number of the cell's particles before it in caller order (a loop over the
// cell; a crowded one is in order already), and the sorted keys
// and indices are written.  Else they are given, and the cells' ranges
// are written from the keys' boundaries (cells zeroed before).
template <typename T, bool kCounted>
__global__ void k_permute(int N, unsigned* skeys, unsigned* svals,
                          const unsigned* order, const unsigned* key_in,
                          const unsigned* count, const unsigned* start, gz_particles p,
                          const void* n_in, const int* box_of,
                          const BoxInfo* boxes, Sorted<T> s, int2* cells,
                          int* ndefer) {
    after_previous();
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= N) return;
    if (q == 0) *ndefer = 0;  // (the density pass after it counts from zero)
    unsigned src, key;
    int i = q;
    if constexpr (kCounted) {
        src = order[q];
        key = key_in[src];
        const int n = (int)count[key], a = (int)start[key], e = a + n;
        if (n <= kCrowd) {
            i = a;
            for (int k = a; k < e; ++k) i += order[k] < src;
        }
        skeys[i] = key;
        svals[i] = src;
    } else {
        src = svals[q];
        key = skeys[q];
    }
    const T x = ((const T*)p.x)[src], y = ((const T*)p.y)[src], z = ((const T*)p.z)[src], h = ((const T*)p.h)[src];
    s.x[i] = x;
    s.y[i] = y;
    s.z[i] = z;
    // velocities, mass and energy are optional (the density pass reads none)
    if (p.vx) s.vx[i] = ((const T*)p.vx)[src];
    if (p.vy) s.vy[i] = ((const T*)p.vy)[src];
    if (p.vz) s.vz[i] = ((const T*)p.vz)[src];
    if (p.m) s.m[i] = ((const T*)p.m)[src];
    if (p.u) s.u[i] = ((const T*)p.u)[src];
    s.h[i] = h;
    s.pos[i] = P4<T>{x, y, z, h};
    s.id[i] = (long long)p.id[src];
    if (n_in) s.n[i] = ((const T*)n_in)[src];
    s.orig[i] = src;
    const int b = box_of[src];
    s.box[i] = b;
    if constexpr (!kCounted) {
        const BoxInfo bx = boxes[b];
        const unsigned mort = key - bx.key_off;
        const int cx = compact3(mort), cy = compact3(mort >> 1), cz = compact3(mort >> 2);
        const int lin = bx.cell_off + (cz * bx.nc + cy) * bx.nc + cx;
        if (i == 0 || skeys[i - 1] != key) cells[lin].x = i;
        if (i == N - 1 || skeys[i + 1] != key) cells[lin].y = i + 1;
    }
}

template <typename T>
__global__ void k_unpermute(int N, int rows, const unsigned* __restrict__ orig,
                            const T* __restrict__ src, T* __restrict__ dst) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const unsigned o = orig[i];
    for (int r = 0; r < rows; ++r) dst[(size_t)r * N + o] = src[(size_t)r * N + i];
}

}  // namespace

template <typename T>
Sorted<T> sorted_view(Ctx& c) {
    Sorted<T> s;
    s.x = (T*)c.sx;
    s.y = (T*)c.sy;
    s.z = (T*)c.sz;
    s.vx = (T*)c.svx;
    s.vy = (T*)c.svy;
    s.vz = (T*)c.svz;
    s.m = (T*)c.sm;
    s.u = (T*)c.su;
    s.h = (T*)c.sh;
    s.id = c.sid;
    s.orig = c.vals;  // filled by sort_and_bin
    s.box = c.sbox;
    s.n = (T*)c.sn;
    s.rho = (T*)c.srho;
    s.P = (T*)c.sP;
    s.c = (T*)c.sc;
    s.sd = (T*)c.ssd;
    s.pos = (P4<T>*)c.spos;
    s.prim = (P4<T>*)c.sprim;
    s.prim2 = (P2<T>*)c.sprim2;
    return s;
}
template Sorted<float> sorted_view<float>(Ctx&);
template Sorted<double> sorted_view<double>(Ctx&);

size_t sort_sums_len(long long N, long long keys, bool counted) {
    if (counted) return (size_t)((keys + kScanTile - 1) / kScanTile);
    const size_t nblk = (size_t)((N + kSortTile - 1) / kSortTile);
    return kMaxDigits * nblk + kMaxDigits;  // per-block counts of up to 1024 digits, then the digit totals
}

template <typename T>
static cudaError_t counting_sort(Ctx& c, const gz_particles& p, const void* n_in) {
    const int N = c.N;
    const long long K = c.total_keys;
    cudaStream_t st = c.stream;
    unsigned* order = (unsigned*)c.defer;  // (free until the density pass)
    cudaMemsetAsync(c.kcount, 0, 4 * (size_t)(K + kCountExtra), st);
    k_cs_count<T><<<blocks(N, 256), 256, 0, st>>>(N, (const T*)p.x, (const T*)p.y, (const T*)p.z, p.id, c.box_of,
                                                   c.boxes, c.kcount, c.keys_alt, c.vals_alt, c.status);
    const int tiles = (int)((K + kScanTile - 1) / kScanTile);
    const bool direct = tiles <= kScanDirect;
    if (!direct) launch_next(c, k_cs_sums, tiles, kScanThreads, K, c.kcount, c.hist);
    launch_next(c, k_cs_scan, tiles, kScanThreads, K, c.kcount, direct ? nullptr : c.hist, c.boxes, c.nboxes, c.kstart,
                c.cells, c.keys);
    // (c.keys is k_permute's to write: room for the crowded keys, at most one in
    // kCrowd particles, and a bit a particle; large launches have blocks that
    // sort faster)
    const int pt = N < (1 << 17) ? 256 : 1024;
    launch_next(c, k_cs_place, blocks(N, pt), pt, N, c.keys_alt, c.vals_alt, c.kstart, order, c.kcount, K, c.keys);
    launch_next(c, k_permute<T, true>, blocks(N, 256), 256, N, c.keys, c.vals, order, c.keys_alt, c.kcount, c.kstart, p,
                n_in, c.box_of, c.boxes, sorted_view<T>(c), c.cells, c.ndefer);
    c.launches += direct ? 4 : 5;
    return cudaGetLastError();
}

template <typename T>
cudaError_t sort_and_bin(Ctx& c, const gz_particles& p, const void* n_in) {
    c.last_lim = nullptr;  // a new sort: earlier sorted-order indices no longer apply
    if (c.kcount) return counting_sort<T>(c, p, n_in);
    const int N = c.N;
    cudaStream_t st = c.stream;
    k_keys<T><<<blocks(N, 256), 256, 0, st>>>(N, (const T*)p.x, (const T*)p.y, (const T*)p.z, p.id,
                                               c.box_of, c.boxes, c.keys, c.vals, c.status);
    const int nblk = blocks(N, kSortTile);
    int total_bits = 0;
    while ((1ll << total_bits) < c.total_keys) ++total_bits;
    // the fewest passes of at most kMaxDigitBits bits, the bits spread evenly
    const int npass = (total_bits + kMaxDigitBits - 1) / kMaxDigitBits;
    const int bits = npass ? (total_bits + npass - 1) / npass : 0;
    c.launches += 1 + 3 * npass;  // (and k_permute, counted by permute_and_bin)
    unsigned *ki = c.keys, *vi = c.vals, *ko = c.keys_alt, *vo = c.vals_alt;
    for (int shift = 0; shift < total_bits; shift += bits) {
        const int pb = std::min(bits, total_bits - shift);
        const int nd = 1 << pb;
        const unsigned mask = (unsigned)nd - 1u;
        unsigned* totals = c.hist + (size_t)nd * nblk;
        k_rs_hist<<<nblk, kSortThreads, 0, st>>>(ki, N, shift, mask, nd, c.hist, nblk);
        k_rs_rows<<<nd, kSortThreads, 0, st>>>(c.hist, nblk, totals);
        k_rs_scatter<<<nblk, kSortThreads, 0, st>>>(ki, vi, N, shift, mask, nd, c.hist, nblk, totals, ko, vo);
        unsigned* t = ki;
        ki = ko;
        ko = t;
        t = vi;
        vi = vo;
        vo = t;
    }
    if (ki != c.keys) {  // odd number of passes: keep the result in the primary buffers
        cudaMemcpyAsync(c.keys, ki, sizeof(unsigned) * N, cudaMemcpyDeviceToDevice, st);
        cudaMemcpyAsync(c.vals, vi, sizeof(unsigned) * N, cudaMemcpyDeviceToDevice, st);
    }
    return permute_and_bin<T>(c, p, n_in);
}

template <typename T>
cudaError_t permute_and_bin(Ctx& c, const gz_particles& p, const void* n_in) {
    c.last_lim = nullptr;
    const int N = c.N;
    cudaStream_t st = c.stream;
    c.launches += 1;
    cudaMemsetAsync(c.cells, 0, sizeof(int2) * (size_t)c.total_cells, st);
    k_permute<T, false><<<blocks(N, 256), 256, 0, st>>>(N, c.keys, c.vals, nullptr, nullptr, nullptr, nullptr, p,
                                                         n_in, c.box_of, c.boxes, sorted_view<T>(c), c.cells, c.ndefer);
    return cudaGetLastError();
}
template cudaError_t sort_and_bin<float>(Ctx&, const gz_particles&, const void*);
template cudaError_t sort_and_bin<double>(Ctx&, const gz_particles&, const void*);
template cudaError_t permute_and_bin<float>(Ctx&, const gz_particles&, const void*);
template cudaError_t permute_and_bin<double>(Ctx&, const gz_particles&, const void*);

template <typename T>
cudaError_t unpermute_T(Ctx& c, const T* src, T* dst, int rows) {
    c.launches += 1;
    k_unpermute<T><<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, rows, c.vals, src, dst);
    return cudaGetLastError();
}
template cudaError_t unpermute_T<float>(Ctx&, const float*, float*, int);
template cudaError_t unpermute_T<double>(Ctx&, const double*, double*, int);

cudaError_t unpermute_d(Ctx& c, const double* src, double* dst, int rows) {
    return unpermute_T<double>(c, src, dst, rows);
}
cudaError_t unpermute_i(Ctx& c, const int* src, int* dst) {
    c.launches += 1;
    k_unpermute<int><<<blocks(c.N, 256), 256, 0, c.stream>>>(c.N, 1, c.vals, src, dst);
    return cudaGetLastError();
}

}  // namespace gz
