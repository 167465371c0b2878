// Periodic neighbour list with a skin and the ghost (periodic-image) map.
//
// Sec. 2.2: one neighbour list of radius r_c serves every message-passing
// layer; Sec. 1 motivates the skin (rebuild only after atoms moved skin/2).
// On one GPU the paper's ghost atoms (Fig. 3a, Fig. 4a) become ghost slots
// N..N+G-1: every periodic image that lies within r_c + skin of the cell,
// pointing at its owner atom and carrying an integer image shift.
//
// Build (all deterministic):
//   1. wrap positions into the cell in FP64 and key every atom by
//      (element, cell bin) -- on the first build and every 8th rebuild; the
//      rebuilds in between keep the previous internal order;
//   2. counting sort by key -> internal order (element-major so the atomic
//      networks see contiguous per-element tiles, spatially sorted inside an
//      element so neighbour gathers stay local);
//   3. enumerate ghost images (count while gathering, scan, fill while keying, a
//      warp's lanes sharing its 32 atoms' images);
//   4. bin owned + used ghost slots into an extended cell grid (counting sort);
//   5. warp per owned atom: scan the stencil bins (in a rectangular cell each
//      column trimmed to the sphere), FP32 pre-test with a margin, FP64 exact
//      test for pairs near r_c + skin, ballot-compacted writes into a
//      fixed-stride row.
// The first build sizes the ghost and row capacities (one host round trip);
// every later rebuild re-runs the same kernels into the resident buffers
// without allocating or synchronising, so it can sit inside a CUDA graph.
// The FP64 test follows one fixed arithmetic order (no FMA contraction):
//   r = (x_w,o - x_w,i) + S(n), S(n)_d = (n0 H0d + n1 H1d) + n2 H2d,
//   d^2 = (r0 r0 + r1 r1) + r2 r2 < (r_c + skin)^2.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"

namespace reann {
namespace {

constexpr int kScanThreads = 256;
// Per-slot kernels whose time goes to FP64 arithmetic (wrapping, image shifts, halo tests) run
// in 64-thread blocks: 24,576 atoms then spread over all SMs' FP64 units (256-thread blocks
// left a third of the SMs without work)
constexpr int kFp64Threads = 64;

__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }

// n h rounded as the FP64 product, without the FP64 multiply for the image shifts -1, 0, 1
// (0 h is a zero with the sign of h): GB300's FP64 pipe is narrow, and the rebuild's
// per-slot kernels are bound by it
__device__ __forceinline__ double smul(int n, double h) {
    if (n == 0) return copysign(0.0, h);
    if (n == 1) return h;
    if (n == -1) return -h;
    return dmul((double)n, h);
}

// In a rectangular cell only the diagonal counts: the other terms are zeros, and adding them
// changes at most the sign of a zero
__device__ __forceinline__ void shift_vec(const CellGeom& g, int n0, int n1, int n2, double s[3]) {
    if (g.ortho) {
        s[0] = smul(n0, g.h[0]);
        s[1] = smul(n1, g.h[4]);
        s[2] = smul(n2, g.h[8]);
        return;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) s[d] = dadd(dadd(smul(n0, g.h[d]), smul(n1, g.h[3 + d])), smul(n2, g.h[6 + d]));
}
// the same vector with plain FP64 products (bitwise equal): for the neighbour search's
// boundary test, where the lanes of a warp hold different shifts and branches diverge
__device__ __forceinline__ void shift_vec_mul(const CellGeom& g, int n0, int n1, int n2, double s[3]) {
#pragma unroll
    for (int d = 0; d < 3; ++d)
        s[d] = dadd(dadd(dmul((double)n0, g.h[d]), dmul((double)n1, g.h[3 + d])), dmul((double)n2, g.h[6 + d]));
}

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ int pack_shift(int a, int b, int c) { return (a + 128) | ((b + 128) << 8) | ((c + 128) << 16); }
__device__ __forceinline__ void unpack_shift(int p, int& a, int& b, int& c) {
    a = (p & 255) - 128;
    b = ((p >> 8) & 255) - 128;
    c = ((p >> 16) & 255) - 128;
}

// ghosts in use: the device count clamped to the capacity
__device__ __forceinline__ int64_t ghosts_in_use(const int32_t* g_count, int64_t g_cap) {
    const int64_t g = *g_count;
    return g < g_cap ? g : g_cap;
}

// 1. wrap + key (caller order)
// Wrap one position into the cell in FP64 (fixed operation order): fractional
// coordinates f = x . hinv, integer shift m = floor(f), wrapped Cartesian
// x - m.H and fractional f - m; `bad` for a non-finite or absurd position.
__device__ __forceinline__ void wrap_one(const CellGeom& g, const double x_in[3], double xw[3], double fw[3], int m[3],
                                         bool& bad) {
    double x[3] = {x_in[0], x_in[1], x_in[2]};
    double fr[3];
    bad = !(isfinite(x[0]) && isfinite(x[1]) && isfinite(x[2]));
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        fr[k] = g.ortho ? dmul(x[k], g.hinv[4 * k])  // (the other terms are zeros)
                        : dadd(dadd(dmul(x[0], g.hinv[k]), dmul(x[1], g.hinv[3 + k])), dmul(x[2], g.hinv[6 + k]));
        if (!isfinite(fr[k]) || fabs(fr[k]) > 1e9) bad = true;
    }
    if (bad) {
#pragma unroll
        for (int k = 0; k < 3; ++k) fr[k] = 0.0, x[k] = 0.0;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) m[k] = (int)floor(fr[k]);
    double s[3];
    shift_vec(g, m[0], m[1], m[2], s);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        xw[k] = dsub(x[k], s[k]);
        fw[k] = dsub(fr[k], (double)m[k]);
    }
}

// ---- deterministic counting sort ------------------------------------------

// Exclusive scan of `in` (n entries, int32) into out[0..n], one launch over
// tiles of kScanTile entries, one block per tile, joined by decoupled look-back
// (D. Merrill and M. Garland, Single-pass Parallel Prefix Scan with Decoupled
// Look-back, NVIDIA technical report NVR-2016-002): a block takes its tile
// number from a ticket counter (so every lower tile's block has started),
// publishes its tile's sum, walks back over the published words of the tiles
// before it (one warp, 32 words per read) until one carries an inclusive
// prefix, and publishes its own inclusive prefix.  A tile is loaded and stored
// coalesced through shared memory (padded one word per 32 against bank
// conflicts), each thread scans kScanPer consecutive entries, and a two-level
// warp scan joins the threads.
// The status words (scan_tiles(n) + 2: one per tile, the ticket, the count of
// finished blocks) start at zero; the last block to finish sets them back to
// zero.  A wait on a lower tile is bounded (kScanSpin polls, seconds): when it
// runs out the block sets FLAG_TIMEOUT and goes on with a wrong carry.
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;
constexpr int32_t kScanAgg = 1 << 30, kScanIncl = (int32_t)0x80000000u, kScanVal = (1 << 30) - 1;
constexpr long long kScanSpin = 1ll << 22;

__global__ void __launch_bounds__(kScanThreads) k_scan(const int* __restrict__ gate, int64_t n,
                                                       const int32_t* __restrict__ in, int32_t* __restrict__ out,
                                                       int32_t* __restrict__ status, int* __restrict__ flags) {
    pdl_enter();
    if (gate && *gate == 0) return;  // rebuild not needed this step
    __shared__ int32_t buf[kScanTile + kScanTile / 32];
    __shared__ int32_t warp_sums[kScanThreads / 32];
    __shared__ int32_t s_tile, s_carry;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int nb = (int)gridDim.x;
    if (tid == 0) s_tile = atomicAdd(&status[nb], 1);
    __syncthreads();
    const int tile = s_tile;
    const int64_t base = (int64_t)tile * kScanTile;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const int x = k * kScanThreads + tid;
        buf[x + x / 32] = base + x < n ? in[base + x] : 0;
    }
    __syncthreads();
    int32_t v[kScanPer];
    int32_t local = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const int x = tid * kScanPer + k;
        v[k] = buf[x + x / 32];
        local += v[k];
    }
    int32_t incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[w] = incl;
    __syncthreads();
    if (w == 0) {
        int32_t t = lane < kScanThreads / 32 ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        if (lane < kScanThreads / 32) warp_sums[lane] = t;  // inclusive
    }
    __syncthreads();
    const int32_t total = warp_sums[kScanThreads / 32 - 1];
    if (w == 0) {  // look-back by one warp: lane l reads the word of tile top - l
        int32_t carry = 0;
        if (tile == 0) {
            if (lane == 0) atomicExch(&status[0], kScanIncl | total);
        } else {
            if (lane == 0) atomicExch(&status[tile], kScanAgg | total);
            bool late = false;
            for (int top = tile - 1; top >= 0; top -= 32) {
                const int q = top - lane;
                int32_t word = kScanIncl;  // below tile 0: an inclusive zero
                if (q >= 0) {
                    long long spins = 0;
                    do {
                        word = *reinterpret_cast<volatile int32_t*>(status + q);
                    } while (word == 0 && ++spins <= kScanSpin);
                    if (word == 0) {
                        late = true;
                        word = kScanIncl;
                    }
                }
                // the nearest tile with an inclusive prefix ends the walk
                const unsigned inc = __ballot_sync(0xffffffffu, (word & kScanIncl) != 0);
                const int stop = inc ? __ffs(inc) - 1 : 31;
                int32_t val = lane <= stop ? (word & kScanVal) : 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
                carry += val;
                if (inc) break;
            }
            if (__any_sync(0xffffffffu, late) && lane == 0) atomicOr(&flags[FLAG_TIMEOUT], 1);
            if (lane == 0) atomicExch(&status[tile], kScanIncl | (carry + total));
        }
        if (lane == 0) s_carry = carry;
    }
    __syncthreads();
    int32_t run = s_carry + (w > 0 ? warp_sums[w - 1] : 0) + incl - local;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const int x = tid * kScanPer + k;
        buf[x + x / 32] = run;
        run += v[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const int x = k * kScanThreads + tid;
        if (base + x < n) out[base + x] = buf[x + x / 32];
    }
    if (tid == 0) {
        if (tile == nb - 1) out[n] = s_carry + total;
        __threadfence();
        if (atomicAdd(&status[nb + 1], 1) == nb - 1) {  // every block is past its look-back
            for (int q = 0; q < nb + 2; ++q) status[q] = 0;
        }
    }
}

// The same scan of up to kDirectMax entries without communication: every block adds up
// all entries before its tile itself (at most 256 KB from L2), so no block waits for
// another.  24,576 entries, traced within the chain: 7.7 -> 6.1 us, 192: 7.1 -> 5.6 us (the
// look-back's ticket, polls and reset); past 64 Ki entries the re-reading grows quadratically.
constexpr int kDirectThreads = 1024, kDirectTile = 4 * kDirectThreads;
constexpr int64_t kDirectMax = 1 << 16;
__global__ void __launch_bounds__(kDirectThreads) k_scan_direct(const int* __restrict__ gate, int64_t n,
                                                                const int32_t* __restrict__ in,
                                                                int32_t* __restrict__ out) {
    pdl_enter();
    if (gate && *gate == 0) return;  // rebuild not needed this step
    __shared__ int32_t warp_sums[32], warp_before[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * kDirectTile, i0 = base + 4 * tid;
    int4 v = make_int4(0, 0, 0, 0);
    if (i0 + 3 < n) {
        v = *reinterpret_cast<const int4*>(in + i0);
    } else {
        if (i0 < n) v.x = in[i0];
        if (i0 + 1 < n) v.y = in[i0 + 1];
        if (i0 + 2 < n) v.z = in[i0 + 2];
    }
    int32_t before = 0;  // this thread's share of the entries before the tile
    const int4* p = reinterpret_cast<const int4*>(in);
#pragma unroll 4
    for (int64_t q = tid; q < base / 4; q += kDirectThreads) {
        const int4 x = p[q];
        before += (x.x + x.y) + (x.z + x.w);
    }
    const int32_t local = (v.x + v.y) + (v.z + v.w);
    int32_t incl = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 31) warp_sums[w] = incl;
    if (lane == 0) warp_before[w] = before;
    __syncthreads();
    if (w == 0) {
        int32_t t = warp_sums[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        const int32_t all = __reduce_add_sync(0xffffffffu, warp_before[lane]);
        warp_sums[lane] = t + all;  // entries up to the end of this warp
        if (lane == 0) warp_before[0] = all;
    }
    __syncthreads();
    const int32_t run = (w > 0 ? warp_sums[w - 1] : warp_before[0]) + incl - local;
    const int4 e = make_int4(run, run + v.x, run + v.x + v.y, run + v.x + v.y + v.z);
    if (i0 + 3 < n) {
        *reinterpret_cast<int4*>(out + i0) = e;
    } else {
        if (i0 < n) out[i0] = e.x;
        if (i0 + 1 < n) out[i0 + 1] = e.y;
        if (i0 + 2 < n) out[i0 + 2] = e.z;
    }
    if (blockIdx.x == gridDim.x - 1 && tid == kDirectThreads - 1) out[n] = run + local;
}

// out = exclusive scan of in, out[n] = the sum, by one block of kDirectThreads threads
__device__ __forceinline__ void block_scan(int n, const int32_t* in, int32_t* out, int32_t* warp_sums) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int32_t carry = 0;
    for (int base = 0; base < n; base += kDirectTile) {
        int32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = base + 4 * tid + k < n ? in[base + 4 * tid + k] : 0;
        const int32_t local = (v[0] + v[1]) + (v[2] + v[3]);
        int32_t incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_sums[w] = incl;
        __syncthreads();
        const int32_t s = warp_sums[lane];
        const int32_t before = __reduce_add_sync(0xffffffffu, lane < w ? s : 0);
        int32_t run = carry + before + incl - local;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (base + 4 * tid + k < n) out[base + 4 * tid + k] = run;
            run += v[k];
        }
        carry += __reduce_add_sync(0xffffffffu, s);
        __syncthreads();  // warp_sums is written again
    }
    if (tid == 0) out[n] = carry;
    __syncthreads();
}

inline int64_t scan_tiles(int64_t n) { return n > 0 ? (n + kScanTile - 1) / kScanTile : 1; }
inline int64_t scan_status_words(int64_t n) { return scan_tiles(n) + 2; }

// out[0..n] = exclusive scan of in[0..n), out[n] the total; status: scan_status_words(n)
// zeroed words
static void scan_exclusive(cudaStream_t s, const int* gate, int64_t n, const int32_t* in, int32_t* out,
                           int32_t* status, int* flags) {
    if (n <= kDirectMax) {
        launch_pdl(k_scan_direct, (unsigned)std::max<int64_t>(1, (n + kDirectTile - 1) / kDirectTile), kDirectThreads, 0,
                   s, gate, n, in, out);
        return;
    }
    launch_pdl(k_scan, (unsigned)scan_tiles(n), kScanThreads, 0, s, gate, n, in, out, status, flags);
}

// The sorts cover n entries, of which the last g_cap are ghost slots that are in use up to
// *g_count (null: all n).  Unused slots take no part (counted like the others, all of them
// would queue at one address).
__device__ __forceinline__ int64_t entries_in_use(int64_t n, const int32_t* g_count, int64_t g_cap) {
    return g_count ? n - g_cap + (*g_count < g_cap ? *g_count : g_cap) : n;
}

__global__ void k_scatter(const int* __restrict__ gate, int64_t n, const int32_t* __restrict__ g_count, int64_t g_cap,
                          const int32_t* __restrict__ key, const int32_t* __restrict__ start,
                          int32_t* __restrict__ counts, int32_t* __restrict__ order) {
    pdl_enter();
    if (gate && *gate == 0) return;  // rebuild not needed this step
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= entries_in_use(n, g_count, g_cap)) return;
    int k = key[i];
    // counting the histogram back down: the bucket's entries take its slots from the top,
    // and the counts end at zero, ready for the next sort's histogram
    int p = start[k] + atomicSub(&counts[k], 1) - 1;
    order[p] = (int32_t)i;
}

// Deterministic placement inside each bucket: the entry at position p of the
// atomic-order scatter moves to start[b] + (number of entries of its bucket with
// a smaller index).  One thread per entry, each scanning its own bucket (buckets
// hold tens of entries).  With `order` its index is stored there; with `pin` its
// FP32 position follows it into sorted order, the index carried in .w (bit
// pattern), so that the search reads candidates contiguously.
__global__ void k_bucket_rank(const int* __restrict__ gate, int64_t n, const int32_t* __restrict__ g_count,
                              int64_t g_cap, const int32_t* __restrict__ key, const int32_t* __restrict__ start,
                              const int32_t* __restrict__ scattered, int32_t* __restrict__ order,
                              const float4* __restrict__ pin, float4* __restrict__ pout) {
    pdl_enter();
    if (gate && *gate == 0) return;  // rebuild not needed this step
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= entries_in_use(n, g_count, g_cap)) return;
    const int32_t v = scattered[p];
    const int32_t b = key[v];
    const int lo = start[b], hi = start[b + 1];
    int rank = 0;
    for (int q = lo; q < hi; ++q) rank += scattered[q] < v;
    if (order) order[lo + rank] = v;
    if (pin) {
        const float4 x = pin[v];
        pout[lo + rank] = make_float4(x.x, x.y, x.z, __int_as_float(v));
    }
}

// an axis's image interval [lo, hi] in one word (|lo|, |hi| < 128)
__device__ __forceinline__ int32_t pack_halo(int lo, int hi) { return (lo + 128) | ((hi + 128) << 8); }
__device__ __forceinline__ void unpack_halo(int32_t p, int& lo, int& hi) {
    lo = (p & 255) - 128;
    hi = ((p >> 8) & 255) - 128;
}

// admissible image shifts of one axis: those keeping f + a within (-reach, 1 + reach),
// an interval because the test is monotone in a
__device__ __forceinline__ void halo_interval(const CellGeom& g, int k, double f, int& lo, int& hi) {
    // Away from the faces (most atoms of a large cell) no other image: decided in FP32, whose rounding
    // the margin covers.  The FP64 pipe bounds the wrap (1,048,576 atoms: 144 -> 97 us).
    const float ff = (float)f, reach = (float)g.reach[k] + 1e-4f;
    if (reach < 0.5f && ff > reach && ff < 1.f - reach) {
        lo = hi = 0;
        return;
    }
    lo = 1;
    hi = 0;
    for (int a = -g.nmax[k]; a <= g.nmax[k]; ++a) {
        const double v = f + a;
        if (v > -g.reach[k] && v < 1.0 + g.reach[k]) {
            if (lo > hi) lo = a;
            hi = a;
        }
    }
}

// an atom's wrapped coordinates, the integer shifts and its image intervals (pack_halo)
struct WrappedAtoms {
    double *xw, *fw;
    int32_t *mw, *halo;
};

// Rebuilds between sorts: every kResortPeriod-th rebuild sorts the owned atoms
// again; the others keep the internal order of the last sort, and only wrap the
// new positions (straight into internal order) and count their ghost images.
// The list itself (ghosts, extended bins, search) is rebuilt in full either way.
// state[0] counts rebuilds since the last sort (k_ghosts_ext counts on);
// state[1] gates the sort's kernels, 0 when the rebuild is gated off.
constexpr int kResortPeriod = 8;

// 1. wrap: caller-order atom i with its sort key and the sort's histogram when this
// rebuild sorts (first: always), else the caller's position of internal atom i
__global__ void k_wrap(const int* __restrict__ gate, int* __restrict__ state, bool first, int64_t n, CellGeom g,
                       const double* __restrict__ pos, const int32_t* __restrict__ species, int n_elem,
                       WrappedAtoms caller, int32_t* __restrict__ key, int32_t* __restrict__ counts,
                       WrappedAtoms internal, const int32_t* __restrict__ perm, int32_t* __restrict__ gcnt,
                       int* __restrict__ flags, double* __restrict__ ref) {
    pdl_enter();
    const bool run = !gate || *gate != 0;
    const bool sort = run && (first || state[0] >= kResortPeriod);
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) state[1] = sort ? 1 : 0;
    if (!run || i >= n) return;
    const int64_t c = sort ? i : perm[i];
    const double x[3] = {pos[3 * c], pos[3 * c + 1], pos[3 * c + 2]};
    // the positions of this build, for the moved-by-more-than-skin/2 test
    ref[3 * c] = x[0];
    ref[3 * c + 1] = x[1];
    ref[3 * c + 2] = x[2];
    double xwi[3], f[3];
    int m[3];
    bool bad;
    wrap_one(g, x, xwi, f, m, bad);
    if (bad) atomicOr(&flags[FLAG_GEOM], 1);
    const WrappedAtoms& o = sort ? caller : internal;
    int cnt = 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o.xw[3 * i + k] = xwi[k];
        o.fw[3 * i + k] = f[k];
        o.mw[3 * i + k] = m[k];
        int lo, hi;
        halo_interval(g, k, f[k], lo, hi);
        o.halo[3 * i + k] = pack_halo(lo, hi);
        cnt *= hi - lo + 1;
    }
    if (!sort) {
        // ghost images: the product of the intervals minus the zero shift, which wrapped coordinates
        // in [0, 1) always admit
        gcnt[i] = cnt - 1;
        return;
    }
    int sp = species[i];
    if (sp < 0 || sp >= n_elem) {
        atomicOr(&flags[FLAG_SPECIES], 1);
        sp = 0;
    }
    int b[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) b[k] = clampi((int)floor(f[k] * g.nb[k]), 0, g.nb[k] - 1);
    const int nbins = g.nb[0] * g.nb[1] * g.nb[2];
    const int k = sp * nbins + (b[0] * g.nb[1] + b[1]) * g.nb[2] + b[2];
    key[i] = k;
    atomicAdd(&counts[k], 1);  // the counting sort's histogram
}

// 2. per-atom arrays into internal order, with each atom's number of ghost images
struct GatherAtoms {
    WrappedAtoms caller, internal;
    const int32_t* species_c;
    int32_t *species, *gcnt;
};
__device__ __forceinline__ void gather_atom(const GatherAtoms& a, int64_t i, int64_t c) {
    int cnt = 1;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a.internal.xw[3 * i + k] = a.caller.xw[3 * c + k];
        a.internal.fw[3 * i + k] = a.caller.fw[3 * c + k];
        a.internal.mw[3 * i + k] = a.caller.mw[3 * c + k];
        const int32_t h = a.caller.halo[3 * c + k];
        a.internal.halo[3 * i + k] = h;
        int lo, hi;
        unpack_halo(h, lo, hi);
        cnt *= hi - lo + 1;
    }
    a.species[i] = a.species_c[c];
    a.gcnt[i] = cnt - 1;
}
__global__ void k_gather_internal(const int* __restrict__ gate, int64_t n, const int32_t* __restrict__ perm,
                                  GatherAtoms a) {
    pdl_enter();
    if (*gate == 0) return;  // the order is kept
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) gather_atom(a, i, perm[i]);
}

// Sort (if state[1] says so), gather and ghost-count scan of a small system by one block:
// one launch instead of five, which return at once on most rebuilds, and on the steps of a
// trajectory that need none, at 0.85 us each.  Step with rebuild before and with it, us: 192
// atoms 108.0 -> 103.0, 1,536 115.0 -> 112.7, 3,069 131.0 -> 131.3, 4,095 133.0 -> 137.9 (one
// block's sort grows past what the launches cost); with k_wrap's merge alone 4,098 atoms
// 139.9 -> 136.4.  20 trajectory steps of 1,536 atoms 2,050 -> 1,967.
constexpr int64_t kSmallOrder = 2048, kSmallKeys = 1 << 15;
__global__ void __launch_bounds__(kDirectThreads) k_order_small(const int* gate, const int* state, int n, int nkeys,
                                                                const int32_t* key, int32_t* counts, int32_t* start,
                                                                int32_t* scattered, int32_t* perm, GatherAtoms a,
                                                                int32_t* goff) {
    pdl_enter();
    if (gate && *gate == 0) return;  // rebuild not needed this step
    __shared__ int32_t warp_sums[32];
    const int tid = threadIdx.x;
    if (state[1] != 0) {
        block_scan(nkeys, counts, start, warp_sums);
        for (int i = tid; i < n; i += kDirectThreads) {
            const int k = key[i];
            scattered[start[k] + atomicSub(&counts[k], 1) - 1] = i;
        }
        __syncthreads();
        for (int p = tid; p < n; p += kDirectThreads) {
            const int v = scattered[p], b = key[v], lo = start[b], hi = start[b + 1];
            int rank = 0;
            for (int q = lo; q < hi; ++q) rank += scattered[q] < v;
            perm[lo + rank] = v;
        }
        __syncthreads();
        for (int i = tid; i < n; i += kDirectThreads) gather_atom(a, i, perm[i]);
        __syncthreads();
    }
    block_scan(n, a.gcnt, goff, warp_sums);
}

// 3-4. ghost images (fractional coordinate within (-reach, 1 + reach) on every
// axis) and the extended binning of owned + ghost slots.
// Extended key and FP32 position of slot (owner o, image shift (a, b, c)):
__device__ __forceinline__ void ext_slot(const CellGeom& g, const double* __restrict__ xw, const double* __restrict__ fw,
                                         int64_t o, int a, int b, int c, int32_t* __restrict__ key,
                                         int32_t* __restrict__ counts, float4* __restrict__ p32, int64_t s) {
    double f[3] = {fw[3 * o] + a, fw[3 * o + 1] + b, fw[3 * o + 2] + c};
    int bx[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) bx[k] = clampi((int)floor(f[k] * g.ns[k]) + g.pad[k], 0, g.nbx[k] - 1);
    const int k = (bx[0] * g.nbx[1] + bx[1]) * g.nbx[2] + bx[2];
    key[s] = k;
    atomicAdd(&counts[k], 1);  // the extended sort's histogram
    double sv[3];
    shift_vec(g, a, b, c, sv);
    p32[s] = make_float4((float)(xw[3 * o] + sv[0]), (float)(xw[3 * o + 1] + sv[1]), (float)(xw[3 * o + 2] + sv[2]), 0.f);
}

// ext_slot for the atom itself (shift 0): f + 0 and x + 0 without the FP64 adds (they
// differ at most in the sign of a zero, which no bin or distance sees)
__device__ __forceinline__ void ext_slot_self(const CellGeom& g, const double* __restrict__ xw,
                                              const double* __restrict__ fw, int64_t o, int32_t* __restrict__ key,
                                              int32_t* __restrict__ counts, float4* __restrict__ p32) {
    int bx[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) bx[k] = clampi((int)floor(fw[3 * o + k] * g.ns[k]) + g.pad[k], 0, g.nbx[k] - 1);
    const int k = (bx[0] * g.nbx[1] + bx[1]) * g.nbx[2] + bx[2];
    key[o] = k;
    atomicAdd(&counts[k], 1);
    p32[o] = make_float4((float)xw[3 * o], (float)xw[3 * o + 1], (float)xw[3 * o + 2], 0.f);
}

// 3-4. ghost images and the extended binning.  A warp takes apw atoms: each lane keys its
// own atom, then the warp walks its atoms' images 32 at a time (slots goff[first] ..
// goff[last + 1], in order; the order of an atom's images is a, b, c over the per-axis
// intervals without the zero shift), so that the images of the few atoms near the
// cell's faces, up to 7 in a large cell and 26 or more in a small one, are shared
// by all lanes instead of keyed one after another by their owner's.  Bound by the FP64
// pipe and the histogram's atomics; 24,576 atoms: 15.7 -> 9.6 us, 1,048,576: 74 -> 49 us
// against one thread per slot with the unused ones keyed to a bucket of their own (whose
// sort took another 28 us there).
__global__ void k_ghosts_ext(const int* __restrict__ gate, int64_t n, CellGeom g, const double* __restrict__ xw,
                             const double* __restrict__ fw, const int32_t* __restrict__ goff, int64_t g_cap,
                             int32_t* __restrict__ owner, int32_t* __restrict__ shift, int32_t* __restrict__ key,
                             int32_t* __restrict__ counts, float4* __restrict__ p32, const int32_t* __restrict__ halo,
                             int apw, int* __restrict__ state, int* __restrict__ flags) {
    pdl_enter();
    if (gate && *gate == 0) return;  // rebuild not needed this step
    if (state && blockIdx.x == 0 && threadIdx.x == 0) state[0] = state[1] ? 1 : state[0] + 1;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t s0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * apw, s = s0 + lane;
    if (s0 >= n) return;  // whole warps
    // this lane's atom: where its images end (lanes without one have none), its intervals
    int32_t end = INT32_MAX, low = 0, extent = 0;
    if (lane < apw && s < n) {
        ext_slot_self(g, xw, fw, s, key, counts, p32);
        int lo[3], hi[3];  // as the wrap computed them
#pragma unroll
        for (int k = 0; k < 3; ++k) unpack_halo(halo[3 * s + k], lo[k], hi[k]);
        low = pack_shift(lo[0], lo[1], lo[2]);
        extent = (hi[0] - lo[0] + 1) | ((hi[1] - lo[1] + 1) << 8) | ((hi[2] - lo[2] + 1) << 16);
        end = goff[s + 1];
    }
    const int32_t first = goff[s0], last = goff[s0 + apw < n ? s0 + apw : n];
    if (last > g_cap && lane == 0) atomicOr(&flags[FLAG_GHOST_OVERFLOW], 1);
    for (int32_t q0 = first; q0 < last; q0 += 32) {
        const int32_t q = q0 + lane;
        // the image's atom: the first lane whose images end beyond q
        int lo = 0, hi = 31;
#pragma unroll
        for (int step = 0; step < 5; ++step) {
            const int mid = (lo + hi) >> 1;
            if (__shfl_sync(FULL, end, mid) > q) hi = mid;
            else lo = mid + 1;
        }
        const int r = min(lo, 31);
        const int32_t prev = __shfl_sync(FULL, end, max(r - 1, 0));
        const int32_t low_r = __shfl_sync(FULL, low, r), ext_r = __shfl_sync(FULL, extent, r);
        if (q < last && q < g_cap) {
            int l0, l1, l2;
            unpack_shift(low_r, l0, l1, l2);
            const int d1 = (ext_r >> 8) & 255, d2 = (ext_r >> 16) & 255;
            int e = q - (r > 0 ? prev : first);           // its number among the atom's images
            e += e >= (-l0 * d1 - l1) * d2 - l2 ? 1 : 0;  // and among all shifts, the zero shift included
            const int ab = e / d2, a = ab / d1, b = ab - a * d1, c = e - ab * d2;
            const int64_t o = s0 + r;
            owner[q] = (int32_t)o;
            shift[q] = pack_shift(l0 + a, l1 + b, l2 + c);
            ext_slot(g, xw, fw, o, l0 + a, l1 + b, l2 + c, key, counts, p32, n + q);
        }
    }
}

// 5. neighbour search: one warp per owned atom.  For each (x, y) column of the
// stencil the z-run of bins is one contiguous range of the bin-sorted slots;
// lane l takes column l of a batch of 32, a warp scan of the run lengths
// concatenates them, and the warp walks the concatenation 32 candidates at a
// time, reading the sorted FP32 positions with their slot index in .w.  The
// columns that start among the 32 candidates are gathered as a bit mask (one
// warp-wide OR); counting the mask's bits up to a candidate gives its column.
// Candidates come in the same order as a bin-by-bin walk (x, then y, then z).
// Bound by latency and issue (57 % of the slots before the next batch's positions were
// fetched ahead; 722 warp instructions per atom).  24,576 atoms: 34.1 -> 27.2 us, 1,048,576: 1,128 ->
// 830 us against a binary search by shuffles for the column, integer divisions for
// the bins, one atomic per atom for the longest row, the atom's FP64 position held
// in registers (rarely needed, read there) and each batch fetched when its turn came.
// Two batches ahead take 971 us, 128-thread blocks 853, five blocks per SM 910.
__global__ void __launch_bounds__(256) k_nbr_search(const int* __restrict__ gate, int64_t n, CellGeom g,
                                                   const double* __restrict__ xw, const int32_t* __restrict__ owner,
                                                   const int32_t* __restrict__ shift, const float4* __restrict__ p32,
                                                   const float4* __restrict__ p32s, const int32_t* __restrict__ bstart,
                                                   const int32_t* __restrict__ ekey,
                                                   int stride, int32_t* __restrict__ nbr, int32_t* __restrict__ cnt_out,
                                                   int* __restrict__ flags) {
    pdl_enter();
    if (gate && *gate == 0) return;  // rebuild not needed this step
    const unsigned FULL = 0xffffffffu;
    __shared__ int s_bases[8][32];
    const int lane = threadIdx.x & 31;
    int* s_base = s_bases[threadIdx.x >> 5];
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (i >= n) return;
    const float4 pi = p32[i];
    // the atom's own bin, as the extended keying computed it (its FP64 floor, evaluated by
    // every lane here, kept a third of GB300's narrow FP64 pipe busy)
    int b[3];
    {
        // FP32 quotients, put right where they are off (by one, below 2^20 bins an axis)
        const int key = ekey[i], plane = g.nbx[1] * g.nbx[2];
        b[0] = (int)(__fdividef((float)key, (float)plane));
        int rem = key - b[0] * plane;
        while (rem < 0) --b[0], rem += plane;
        while (rem >= plane) ++b[0], rem -= plane;
        b[1] = (int)(__fdividef((float)rem, (float)g.nbx[2]));
        b[2] = rem - b[1] * g.nbx[2];
        while (b[2] < 0) --b[1], b[2] += g.nbx[2];
        while (b[2] >= g.nbx[2]) ++b[1], b[2] -= g.nbx[2];
    }
    const int x0 = max(0, b[0] - g.sw[0]), x1 = min(g.nbx[0] - 1, b[0] + g.sw[0]);
    const int y0 = max(0, b[1] - g.sw[1]), y1 = min(g.nbx[1] - 1, b[1] + g.sw[1]);
    const int z0 = max(0, b[2] - g.sw[2]), z1 = min(g.nbx[2] - 1, b[2] + g.sw[2]);
    const int ny = y1 - y0 + 1, ncol = (x1 - x0 + 1) * ny;
    const float inv_ny = __fdividef(1.f, (float)ny);
    const float lo2 = g.rcut2_f - g.margin, hi2 = g.rcut2_f + g.margin;
    int count = 0;
    int32_t* row = nbr + (size_t)i * stride;
    for (int cb = 0; cb < ncol; cb += 32) {
        int st = 0, len = 0;
        if (cb + lane < ncol) {
            const int col = cb + lane, cx = (int)((col + 0.5f) * inv_ny);  // col / ny: half a step from any integer
            const int bx = x0 + cx, by = y0 + col - cx * ny;
            const int bin0 = (bx * g.nbx[1] + by) * g.nbx[2];
            int za = z0, zb = z1;
            if (g.ortho) {
                // rectangular cell: bin b of axis k spans [(b - pad) w, (b - pad + 1) w) in Cartesian
                // coordinates; keep the z-bins within sqrt(r^2 - rho^2) of the atom, rho being the
                // atom's distance to the column.  FP32 (the FP64 units are slow) with 2e-3 A of slack,
                // far above the rounding of coordinates and bin edges.
                constexpr float kSlack = 2e-3f;
                const float lx = (bx - g.pad[0]) * g.binw[0], ly = (by - g.pad[1]) * g.binw[1];
                const float dx = fmaxf(0.f, fmaxf(lx - pi.x, pi.x - (lx + g.binw[0])) - kSlack);
                const float dy = fmaxf(0.f, fmaxf(ly - pi.y, pi.y - (ly + g.binw[1])) - kSlack);
                const float rho2 = dx * dx + dy * dy;
                if (rho2 >= g.rcut2_f) {
                    zb = za - 1;
                } else {
                    const float hz = sqrtf(g.rcut2_f - rho2) + kSlack;
                    za = max(z0, (int)floorf((pi.z - hz) * g.binw_inv[2]) + g.pad[2]);
                    zb = min(z1, (int)floorf((pi.z + hz) * g.binw_inv[2]) + g.pad[2]);
                }
            }
            if (za <= zb) {
                st = bstart[bin0 + za];
                len = bstart[bin0 + zb + 1] - st;
            }
        }
        int pref = len;  // inclusive scan of the run lengths
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(FULL, pref, o);
            if (lane >= o) pref += y;
        }
        const int total = __shfl_sync(FULL, pref, 31);
        const int excl = pref - len;
        const unsigned filled = __ballot_sync(FULL, len > 0), upto = (2u << lane) - 1u;
        if (len > 0) s_base[__popc(filled & (upto >> 1))] = st - excl;  // of the non-empty columns, in order
        __syncwarp();
        int before = 0;  // non-empty columns that start before t0
        auto fetch = [&](int t0) {  // candidate t0 + lane
            const int rel = excl - t0;
            const unsigned starts = __reduce_or_sync(FULL, len > 0 && rel >= 0 && rel < 32 ? 1u << rel : 0u);
            const int c = s_base[before + __popc(starts & upto) - 1] + t0 + lane;
            before += __popc(starts);
            return t0 + lane < total ? p32s[c] : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 next = make_float4(0.f, 0.f, 0.f, 0.f);
        if (total > 0) next = fetch(0);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            const float4 pj = next;
            if (t0 + 32 < total) next = fetch(t0 + 32);  // on its way while this batch is decided
            bool hit = false;
            int j = -1;
            if (t < total) {
                j = __float_as_int(pj.w);
                if (j != (int)i) {
                    const float dx = pj.x - pi.x, dy = pj.y - pi.y, dz = pj.z - pi.z;
                    const float d2 = dx * dx + dy * dy + dz * dz;
                    if (d2 < lo2 && d2 > 1e-4f) {
                        hit = true;
                    } else if (d2 <= hi2) {
                        // exact FP64 decision (and the coincident-atom check)
                        int64_t o = j;
                        int a0 = 0, a1 = 0, a2 = 0;
                        if (j >= n) {
                            o = owner[j - n];
                            unpack_shift(shift[j - n], a0, a1, a2);
                        }
                        double sv[3];
                        shift_vec_mul(g, a0, a1, a2, sv);
                        double rr[3];
#pragma unroll
                        for (int k = 0; k < 3; ++k) rr[k] = dadd(dsub(xw[3 * o + k], xw[3 * i + k]), sv[k]);
                        const double dd = dadd(dadd(dmul(rr[0], rr[0]), dmul(rr[1], rr[1])), dmul(rr[2], rr[2]));
                        hit = dd < g.rcut2;
                        if (dd < 1e-16) atomicOr(&flags[FLAG_GEOM], 2);
                    }
                }
            }
            const unsigned m = __ballot_sync(FULL, hit);
            if (hit) {
                const int p = count + __popc(m & ((1u << lane) - 1u));
                if (p < stride) row[p] = j;
            }
            count += __popc(m);
        }
        __syncwarp();  // s_base is rewritten for the next 32 columns
    }
    if (lane == 0) {
        cnt_out[i] = min(count, stride);
        if (count > stride) atomicOr(&flags[FLAG_NBR_OVERFLOW], 1);
        // (every atom's atomic at one address would serialise the kernel's end)
        if (count > __ldcg(&flags[FLAG_MAXNBR])) atomicMax(&flags[FLAG_MAXNBR], count);
    }
}

// per evaluation: refresh owned + ghost positions (FP64 -> hi/lo FP32 pair)
// (with c0, also the first layer's coefficients c0[species] of every slot)
__global__ void k_refresh(int64_t n, const int32_t* __restrict__ g_count, int64_t g_cap, CellGeom g,
                          const double* __restrict__ pos, const int32_t* __restrict__ perm,
                          const int32_t* __restrict__ wrapm, const int32_t* __restrict__ owner,
                          const int32_t* __restrict__ shift, float4* __restrict__ out,
                          const int32_t* __restrict__ species, const float* __restrict__ c0,
                          float* __restrict__ coef) {
    pdl_enter();
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n + ghosts_in_use(g_count, g_cap)) return;
    int64_t o = s;
    int a = 0, b = 0, c = 0;
    if (s >= n) {
        o = owner[s - n];
        unpack_shift(shift[s - n], a, b, c);
    }
    const int64_t cidx = perm[o];
    double sm[3], sv[3];
    shift_vec(g, wrapm[3 * o], wrapm[3 * o + 1], wrapm[3 * o + 2], sm);
    shift_vec(g, a, b, c, sv);
    double x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] = (pos[3 * cidx + k] - sm[k]) + sv[k];
    float h[3], l[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        h[k] = (float)x[k];
        l[k] = (float)(x[k] - (double)h[k]);
    }
    out[2 * s] = make_float4(h[0], h[1], h[2], 0.f);
    out[2 * s + 1] = make_float4(l[0], l[1], l[2], 0.f);
    if (c0) {
        const float4* src = reinterpret_cast<const float4*>(c0 + species[o] * NPHI);
        float4* dst = reinterpret_cast<float4*>(coef + (size_t)s * NPHI);
        dst[0] = src[0];
        dst[1] = src[1];
    }
}

// largest displacement since the build: flag when any atom moved more than half the skin
__global__ void k_moved(int64_t n, const double* __restrict__ pos, const double* __restrict__ ref, double thr2,
                        int* __restrict__ moved) {
    pdl_enter();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double dx = pos[3 * i] - ref[3 * i], dy = pos[3 * i + 1] - ref[3 * i + 1], dz = pos[3 * i + 2] - ref[3 * i + 2];
    if (!(dx * dx + dy * dy + dz * dz <= thr2)) atomicOr(moved, 1);
}


inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// What a stage of the first build finds ready: zeroed histogram, scan words and flags, the
// caller's species and the rebuild state.  One launch; as separate memsets and copies (one of them
// from pageable memory), and with the sizes below copied back one by one, a 4,000-atom structure's
// build, evaluation and release took 539 us instead of 492.
struct BuildBegin {
    int64_t n;  // 0: no species
    const int32_t* species;
    int32_t* species_c;
    int64_t n_counts;
    int32_t* counts;
    int64_t n_status;
    int32_t* status;
    int* flags;
    int32_t* rb_state;  // nullable
};
__global__ void k_build_begin(BuildBegin b) {
    pdl_enter();
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < b.n; i += step) b.species_c[i] = b.species[i];
    for (int64_t i = i0; i < b.n_counts; i += step) b.counts[i] = 0;
    for (int64_t i = i0; i < b.n_status; i += step) b.status[i] = 0;
    if (i0 < NFLAGS) b.flags[i0] = 0;
    if (b.rb_state && i0 < 4) b.rb_state[i0] = i0 == 0 ? 1 : 0;
}

// the flags, the element ranges of the internal order and the ghost count, into pinned host
// memory: [flags | starts of the elements .. end | (at MAX_ELEM + 1) ghosts]
__global__ void k_read_sizes(int n_elem, int64_t nbins, const int32_t* __restrict__ start,
                             const int32_t* __restrict__ ghosts, const int* __restrict__ flags, int* host) {
    pdl_enter();
    const int t = threadIdx.x;
    if (t < NFLAGS) host[t] = flags[t];
    if (t <= n_elem) host[NFLAGS + t] = start[t * nbins];
    if (t == 0) host[NFLAGS + MAX_ELEM + 1] = *ghosts;
}

// the flags into pinned host memory, zeroed for the next calls; with energy (nullable) it follows them
__global__ void k_take_flags(int* __restrict__ flags, const double* __restrict__ energy, int* host) {
    pdl_enter();
    const int t = threadIdx.x;
    if (t < NFLAGS) {
        host[t] = flags[t];
        flags[t] = 0;
    }
    if (t == 0 && energy) *reinterpret_cast<double*>(host + NFLAGS) = *energy;
}

}  // namespace

// Counting sort of n entries (the ghost slots among them in use up to *g_count, null: all;
// see entries_in_use) with keys in [0, nkeys) whose histogram `counts` the kernel that
// produced the keys has filled: order (nullable) = indices sorted by (key, index), pout =
// their FP32 positions pin; start = bucket offsets.  The scatter counts the histogram back
// down to zero for the next sort.
static cudaError_t counting_sort(cudaStream_t s, const int* gate, int64_t n, const int32_t* g_count, int64_t g_cap,
                                 int64_t nkeys, const int32_t* key, int32_t* counts, int32_t* start,
                                 int32_t* scattered, int32_t* order, int32_t* tsum, int* flags,
                                 const float4* pin = nullptr, float4* pout = nullptr) {
    scan_exclusive(s, gate, nkeys, counts, start, tsum, flags);
    if (n > 0) {
        launch_pdl(k_scatter, blocks_for(n, 256), 256, 0, s, gate, n, g_count, g_cap, key, start, counts, scattered);
        launch_pdl(k_bucket_rank, blocks_for(n, 256), 256, 0, s, gate, n, g_count, g_cap, key, start, scattered, order,
                   pin, pout);
    }
    return cudaGetLastError();
}

void* nlist_alloc_bytes(reann_nlist* nl, size_t bytes) {
    void* p = nullptr;
    bytes = std::max<size_t>(bytes, 1);
    // (a block taken from the pool under capture would belong to the graph)
    const bool big = nl->list_pool && (bytes >= ListPool::kBig || nl->alloc_capturing);
    auto take = [&] {
        return nl->mem_pool && !big ? cudaMallocFromPoolAsync(&p, bytes, nl->mem_pool, nl->alloc_stream) : cudaMalloc(&p, bytes);
    };
    cudaError_t e = take();
    if (e != cudaSuccess && nl->list_pool) {  // give the pool's unused blocks back and try again
        (void)cudaGetLastError();
        cudaStreamSynchronize(nl->list_pool->stream);  // (what is on its way back)
        cudaMemPoolTrimTo(nl->mem_pool, 0);
        e = take();
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    (big ? nl->big_allocs : nl->allocs).push_back(p);
    return p;
}

void nlist_free_block(reann_nlist* nl, void* p) {
    for (auto* list : {&nl->allocs, &nl->big_allocs}) {
        const auto it = std::find(list->begin(), list->end(), p);
        if (it == list->end()) continue;
        list->erase(it);
        if (nl->mem_pool && list == &nl->allocs)
            cudaFreeAsync(p, nl->alloc_stream);
        else
            cudaFree(p);
        return;
    }
}

template <typename T>
static T* dalloc(reann_nlist* nl, size_t count) {
    return nlist_alloc<T>(nl, count);
}

static int64_t owned_keys(const reann_nlist* nl) {
    const CellGeom& g = nl->geom;
    return (int64_t)g.nb[0] * g.nb[1] * g.nb[2] * nl->n_elem;
}
static int64_t ext_bins(const reann_nlist* nl) {
    const CellGeom& g = nl->geom;
    return (int64_t)g.nbx[0] * g.nbx[1] * g.nbx[2];
}

// steps 1-3a: wrap, sort, gather, ghost count + scan (goff[n] = ghost count on the device)
// gate: nothing is done where it is zero (nullptr: always run)
// first: the list's first build, which sorts
static cudaError_t stage_sort_and_count(cudaStream_t s, reann_nlist* nl, const double* pos, int* flags,
                                        const int* gate, bool first) {
    const int64_t n = nl->n, nkeys = owned_keys(nl);
    NlistScratch& w = nl->w;
    const WrappedAtoms caller{w.xw_c, w.fw_c, w.mw_c, w.halo_c}, internal{w.xw, w.fw, nl->wrapm, w.halo};
    const GatherAtoms gather{caller, internal, w.species_c, nl->species, w.gcnt};
    launch_pdl(k_wrap, blocks_for(n, kFp64Threads), kFp64Threads, 0, s, gate, w.rb_state, first, n, nl->geom, pos,
               w.species_c, nl->n_elem, caller, w.key, w.counts, internal, nl->perm, w.gcnt, flags, nl->pos_ref);
    if (n <= kSmallOrder && nkeys <= kSmallKeys) {
        launch_pdl(k_order_small, 1, kDirectThreads, 0, s, gate, w.rb_state, (int)n, (int)nkeys, w.key, w.counts,
                   w.start, w.scat, nl->perm, gather, w.goff);
        return cudaGetLastError();
    }
    const int* sort_gate = w.rb_state + 1;
    counting_sort(s, sort_gate, n, nullptr, 0, nkeys, w.key, w.counts, w.start, w.scat, nl->perm, w.tsum, flags);
    launch_pdl(k_gather_internal, blocks_for(n, kFp64Threads), kFp64Threads, 0, s, sort_gate, n, nl->perm, gather);
    scan_exclusive(s, gate, n, w.gcnt, w.goff, w.tsum, flags);
    return cudaGetLastError();
}

static cudaError_t stage_ghosts_and_bins(cudaStream_t s, reann_nlist* nl, int* flags, const int* gate, bool first) {
    const int64_t n = nl->n, next = n + nl->g_cap;
    NlistScratch& w = nl->w;
    const int64_t nx = ext_bins(nl);
    // Atoms per warp: in a small cell most atoms have several images, and a warp's chain of 32-image
    // batches is what the launch lasts.  us with 4 / 8 / 16 / 32: 192 atoms 4.2 / 5.2 / 7.7 / 11.5,
    // 3,069 4.7 / 5.7 / 7.8 / 9.2, 8,100 7.0 / 6.4 / 8.2 / 10.6, 24,576 14.6 / 11.5 / 9.8 / 10.0.
    const int apw = n <= 8192 ? 4 : 32;
    launch_pdl(k_ghosts_ext, blocks_for((n + apw - 1) / apw * 32, kFp64Threads), kFp64Threads, 0, s, gate, n, nl->geom,
               w.xw, w.fw, w.goff, nl->g_cap, nl->g_owner, nl->g_shift, w.ekey, w.ecounts, w.p32, w.halo, apw,
               first ? nullptr : w.rb_state, flags);
    counting_sort(s, gate, next, w.goff + n, nl->g_cap, nx, w.ekey, w.ecounts, w.estart, w.escat, nullptr, w.etsum,
                  flags, w.p32, w.p32s);
    return cudaGetLastError();
}

static cudaError_t stage_search(cudaStream_t s, reann_nlist* nl, int* flags, const int* gate) {
    const int64_t n = nl->n;
    NlistScratch& w = nl->w;
    launch_pdl(k_nbr_search, blocks_for(n * 32, 256), 256, 0, s, gate, n, nl->geom, w.xw, nl->g_owner,
               nl->g_shift, w.p32, w.p32s, w.estart, w.ekey, nl->stride, nl->nbr, nl->nbr_cnt, flags);
    return cudaGetLastError();
}

static void launch_begin(cudaStream_t s, const BuildBegin& b) {
    const int64_t most = std::max(std::max(b.n, b.n_counts), std::max<int64_t>(b.n_status, NFLAGS));
    launch_pdl(k_build_begin, (unsigned)std::min<int64_t>(1024, blocks_for(most, 256)), 256, 0, s, b);
}

int build_nlist_device(reann_ctx* ctx, reann_nlist* nl, const double* pos, const int32_t* species) {
    cudaStream_t s = ctx->stream;
    const int64_t n = nl->n;
    NlistScratch& w = nl->w;
    const int64_t nkeys = owned_keys(nl);
    if (n >= (int64_t(1) << 28))  // the scans' status words carry sums below 2^30 (atoms + ghost capacity)
        return set_error(ctx, REANN_E_ARG, "more than 2^28 atoms in one list");
    w.xw_c = dalloc<double>(nl, 3 * n);
    w.fw_c = dalloc<double>(nl, 3 * n);
    w.mw_c = dalloc<int32_t>(nl, 3 * n);
    w.key = dalloc<int32_t>(nl, n);
    w.counts = dalloc<int32_t>(nl, nkeys);
    w.start = dalloc<int32_t>(nl, nkeys + 1);
    w.xw = dalloc<double>(nl, 3 * n);
    w.fw = dalloc<double>(nl, 3 * n);
    w.gcnt = dalloc<int32_t>(nl, n);
    w.halo_c = dalloc<int32_t>(nl, 3 * n);
    w.halo = dalloc<int32_t>(nl, 3 * n);
    w.goff = dalloc<int32_t>(nl, n + 1);
    w.species_c = dalloc<int32_t>(nl, n);
    w.scat = dalloc<int32_t>(nl, n);
    w.rb_state = dalloc<int32_t>(nl, 4);
    w.tsum = dalloc<int32_t>(nl, std::max(scan_status_words(nkeys), scan_status_words(n)));
    nl->perm = dalloc<int32_t>(nl, n);
    nl->species = dalloc<int32_t>(nl, n);
    nl->wrapm = dalloc<int32_t>(nl, 3 * n);
    nl->pos_ref = dalloc<double>(nl, 3 * n);
    if (!w.xw_c || !w.fw_c || !w.mw_c || !w.key || !w.counts || !w.start || !w.xw || !w.fw || !w.gcnt || !w.goff ||
        !w.halo_c || !w.halo ||
        !w.species_c || !w.scat || !nl->perm || !nl->species || !nl->wrapm || !nl->pos_ref || !w.rb_state ||
        !w.tsum)
        return set_error(ctx, REANN_E_NOMEM, "neighbour-list allocation failed");
    // counts and tsum are kept zero between sorts; this build sorts, rebuilds count from 1
    launch_begin(s, {n, species, w.species_c, nkeys, w.counts, std::max(scan_status_words(nkeys), scan_status_words(n)),
                     w.tsum, ctx->d_flags, w.rb_state});
    REANN_CUDA_TRY(ctx, stage_sort_and_count(s, nl, pos, ctx->d_flags, nullptr, true));
    // sizes: element ranges of the internal order and the ghost count, read back with the flags
    const int32_t* es = ctx->h_flags + NFLAGS;
    launch_pdl(k_read_sizes, 1, 64, 0, s, nl->n_elem, nkeys / nl->n_elem, w.start, w.goff + n, ctx->d_flags,
               ctx->h_flags);
    REANN_CUDA_TRY(ctx, cudaGetLastError());
    REANN_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    const int32_t G = es[MAX_ELEM + 1];
    if (ctx->h_flags[FLAG_SPECIES]) return set_error(ctx, REANN_E_ARG, "species index out of range");
    if (ctx->h_flags[FLAG_GEOM]) return set_error(ctx, REANN_E_GEOM, "non-finite atom position");
    for (int e = 0; e <= nl->n_elem; ++e) nl->elem_start[e] = es[e];
    for (int e = 0; e < nl->n_elem; ++e)
        if (es[e + 1] > es[e]) nl->elem_end = e + 1;
    nl->g = G;
    nl->ghosts_by_owner = true;  // k_ghosts_ext enumerates each atom's images contiguously at goff[i]
    // capacity with headroom so that rebuilds after atom motion fit
    nl->g_cap = G + G / 4 + 64;
    const int64_t next = n + nl->g_cap;
    const int64_t nx = ext_bins(nl);
    nl->g_owner = dalloc<int32_t>(nl, nl->g_cap);
    nl->g_shift = dalloc<int32_t>(nl, nl->g_cap);
    w.ekey = dalloc<int32_t>(nl, next);
    w.p32 = dalloc<float4>(nl, next);
    w.p32s = dalloc<float4>(nl, next);
    w.ecounts = dalloc<int32_t>(nl, nx);
    w.estart = dalloc<int32_t>(nl, nx + 1);
    w.escat = dalloc<int32_t>(nl, next);
    w.etsum = dalloc<int32_t>(nl, scan_status_words(nx));
    if (!nl->g_owner || !nl->g_shift || !w.ekey || !w.p32 || !w.p32s || !w.ecounts || !w.estart ||
        !w.escat || !w.etsum)
        return set_error(ctx, REANN_E_NOMEM, "ghost allocation failed");
    launch_begin(s, {0, nullptr, nullptr, nx, w.ecounts, scan_status_words(nx), w.etsum, ctx->d_flags, nullptr});
    REANN_CUDA_TRY(ctx, stage_ghosts_and_bins(s, nl, ctx->d_flags, nullptr, true));
    // row capacity: expected neighbours from the number density, with headroom
    const CellGeom& g = nl->geom;
    const double vol = std::fabs(g.h[0] * (g.h[4] * g.h[8] - g.h[5] * g.h[7]) -
                                 g.h[1] * (g.h[3] * g.h[8] - g.h[5] * g.h[6]) +
                                 g.h[2] * (g.h[3] * g.h[7] - g.h[4] * g.h[6]));
    const double expect = (double)n / vol * 4.18879020478639 * std::pow(g.rcut2, 1.5);
    int stride = (int)std::min<double>(1 << 20, std::ceil((1.5 * expect + 32) / 8.0) * 8);
    for (int attempt = 0; attempt < 2; ++attempt) {
        nl->stride = stride;
        nl->nbr = dalloc<int32_t>(nl, (size_t)n * stride);
        nl->nbr_cnt = dalloc<int32_t>(nl, n);
        if (!nl->nbr || !nl->nbr_cnt) return set_error(ctx, REANN_E_NOMEM, "neighbour-list allocation failed");
        if (attempt > 0) REANN_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_flags, 0, sizeof(int) * NFLAGS, s));
        REANN_CUDA_TRY(ctx, stage_search(s, nl, ctx->d_flags, nullptr));
        REANN_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->h_flags, ctx->d_flags, sizeof(int) * NFLAGS, cudaMemcpyDeviceToHost, s));
        REANN_CUDA_TRY(ctx, cudaStreamSynchronize(s));
        if (ctx->h_flags[FLAG_GEOM]) return set_error(ctx, REANN_E_GEOM, "coincident atoms (distance < 1e-8 A)");
        if (ctx->h_flags[FLAG_GHOST_OVERFLOW]) return set_error(ctx, REANN_E_CAPACITY, "ghost capacity exceeded");
        nl->max_count = ctx->h_flags[FLAG_MAXNBR];
        if (!ctx->h_flags[FLAG_NBR_OVERFLOW]) break;
        if (attempt == 1) return set_error(ctx, REANN_E_CAPACITY, "neighbour capacity exceeded");
        // grow to the observed maximum (plus headroom for later motion) and search again
        stride = ((ctx->h_flags[FLAG_MAXNBR] + ctx->h_flags[FLAG_MAXNBR] / 8 + 16 + 7) / 8) * 8;
    }
    return REANN_OK;
}

// one launch for what were a copy of the flags, their reset and a copy of the energy (host callback
// of 24,576 atoms 414.7 -> 411.3 us)
cudaError_t launch_take_flags(cudaStream_t s, int* flags, const double* energy, int* host) {
    static_assert(NFLAGS % 2 == 0 && reann_ctx::kHostInts >= 2, "the energy follows the flags, 8 B aligned");
    launch_pdl(k_take_flags, 1, 32, 0, s, flags, energy, host);
    return cudaGetLastError();
}

// gate == nullptr: always rebuild; otherwise every kernel returns at once unless *gate != 0
cudaError_t launch_rebuild(cudaStream_t s, reann_nlist* nl, const double* pos, int* flags, const int* gate) {
    cudaError_t e = stage_sort_and_count(s, nl, pos, flags, gate, false);
    if (e == cudaSuccess) e = stage_ghosts_and_bins(s, nl, flags, gate, false);
    if (e == cudaSuccess) e = stage_search(s, nl, flags, gate);
    return e;
}

cudaError_t launch_moved(cudaStream_t s, const reann_nlist* nl, const double* pos, int* moved) {
    const double half = 0.5 * nl->skin;
    launch_pdl(k_moved, blocks_for(nl->n, kFp64Threads), kFp64Threads, 0, s, nl->n, pos, nl->pos_ref, half * half,
               moved);
    return cudaGetLastError();
}

const int32_t* ghost_count_ptr(const reann_nlist* nl) { return nl->w.goff + nl->n; }

cudaError_t launch_refresh_positions(cudaStream_t s, const reann_nlist* nl, const double* pos, const float* c0) {
    const int64_t total = nl->n + nl->g_cap;
    launch_with(true, eval_launch(nl).carve(), k_refresh, blocks_for(total, kFp64Threads), kFp64Threads, 0, s, nl->n, ghost_count_ptr(nl), nl->g_cap,
               nl->geom, pos, nl->perm, nl->wrapm, nl->g_owner, nl->g_shift, nl->pos, nl->species, c0,
               nl->coef);
    return cudaGetLastError();
}

int export_nlist(reann_ctx* ctx, const reann_nlist* nl, int64_t cap, int32_t* oi, int32_t* oj, int32_t* on,
                 int64_t* count) {
    cudaStream_t s = ctx->stream;
    const int64_t n = nl->n;
    int32_t G = 0;
    REANN_CUDA_TRY(ctx, cudaMemcpyAsync(&G, ghost_count_ptr(nl), sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    REANN_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    const int64_t g = std::min<int64_t>(G, nl->g_cap);
    std::vector<int32_t> nbr((size_t)n * nl->stride), cnt(n), perm(n), wm(3 * n), own(g), sh(g);
    REANN_CUDA_TRY(ctx, cudaMemcpyAsync(nbr.data(), nl->nbr, sizeof(int32_t) * nbr.size(), cudaMemcpyDeviceToHost, s));
    REANN_CUDA_TRY(ctx, cudaMemcpyAsync(cnt.data(), nl->nbr_cnt, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, s));
    REANN_CUDA_TRY(ctx, cudaMemcpyAsync(perm.data(), nl->perm, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, s));
    REANN_CUDA_TRY(ctx, cudaMemcpyAsync(wm.data(), nl->wrapm, sizeof(int32_t) * 3 * n, cudaMemcpyDeviceToHost, s));
    if (g > 0) {
        REANN_CUDA_TRY(ctx, cudaMemcpyAsync(own.data(), nl->g_owner, sizeof(int32_t) * g, cudaMemcpyDeviceToHost, s));
        REANN_CUDA_TRY(ctx, cudaMemcpyAsync(sh.data(), nl->g_shift, sizeof(int32_t) * g, cudaMemcpyDeviceToHost, s));
    }
    REANN_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    int64_t q = 0;
    for (int64_t i = 0; i < n; ++i) {
        for (int e = 0; e < cnt[i]; ++e) {
            int64_t slot = nbr[(size_t)i * nl->stride + e];
            int64_t o = slot;
            int a[3] = {0, 0, 0};
            if (slot >= n) {
                o = own[slot - n];
                int p = sh[slot - n];
                a[0] = (p & 255) - 128;
                a[1] = ((p >> 8) & 255) - 128;
                a[2] = ((p >> 16) & 255) - 128;
            }
            if (q < cap) {
                oi[q] = perm[i];
                oj[q] = perm[o];
                for (int k = 0; k < 3; ++k) on[3 * q + k] = a[k] - wm[3 * o + k] + wm[3 * i + k];
            }
            ++q;
        }
    }
    *count = q;
    return REANN_OK;
}

}  // namespace reann
