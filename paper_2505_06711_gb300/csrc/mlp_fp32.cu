// Per-element atomic networks in plain FP32 (SIMT FMA), forward and
// input-gradient backward.
//
// Sec. 2.1, Eq. 2: c^{t+1}_i = M^t_{Z_i}(rho^t_i) (48 -> 64 -> 64 -> 8), and the
// energy network eps_i = M^{T-1}_{Z_i}(rho^{T-1}_i) (48 -> 64 -> 64 -> 1), SiLU
// between layers.  The reverse pass (Eqs. 4-5) needs only the input gradient
// rhobar = J^T ybar (a vector-Jacobian product, Sec. 2.2), never weight
// gradients.
//
// Atoms are stored element-major, so a tile of 64 consecutive rows uses one
// element's weights.  A block of NT threads takes NT / 16 x RPT rows of a tile: the whole
// tile (256 threads, RPT = 4), or, so that the few tiles of a small system occupy two or
// four times the SMs and each thread's chain is shorter, half of it (256 threads, RPT = 2;
// backward 128, RPT = 4) or a quarter (128 threads, RPT = 2), and
// computes a 64-wide layer output as NT / 16 x 16 threads x (RPT rows x 4 columns),
// reading float4 fragments of the row-major activations and weights from shared
// memory.  A row's arithmetic is the same for every split.  The forward keeps one
// activation buffer (48 KB of shared memory: four blocks per SM) and writes
// SiLU'(z1), SiLU'(z2) of every row; the backward reads them instead of
// recomputing the forward, and with the 48-feature networks also takes the
// bbar step of Eq. 1's squares and writes the adjoint records (69 KB: three
// blocks per SM).  The energy network (48 features) is one kernel, forward and
// backward: its output adjoint is 1, so nothing waits for another layer, the SiLU'
// values stay in registers and the tile's weights are staged by one launch (24,576
// atoms: 15.3 + 23.8 us in two launches, 34.6 us in one; 1,048,576: 407 + 712, 1,071).
// Before pdl_enter() the networks read only what no kernel of the stream writes after the
// previous kernel began: the tile list and the weights, whose copies are then under way
// while the previous kernel ends.
//   Bound by L1, the float4 fragments (a 16 B load writes 512 B of registers per warp whatever it
// broadcasts), and issue: 7,680 FMAs per row forward and 10,240 with the bbar step
// backward, beside a quarter as many instructions for SiLU.  1,048,576 atoms: 451 us forward (L1
// 80 %, issue 77 %) and 735 us backward (89 %, 58 %); fma.rn.f32x2 was measured at 0.8 x the FMA
// rate of single fmas.
#include <cuda_runtime.h>

#include <mutex>

#include "bulk.cuh"
#include "common.cuh"

namespace reann {
namespace {

constexpr int LDH = H1 + 4;  // 68
static_assert(MLP_TILE == 64, "a block takes 16, 32 or 64 rows of a tile");
// input rows of FIN features are held with stride FIN (one bulk copy of the
// tile's contiguous rows) in the buffer that later holds h1 (stride LDH)
template <int FIN>
__host__ __device__ constexpr int ldx() { return FIN; }
template <int FIN, int RPT, int NT>
__host__ __device__ constexpr int abuf() { return NT / 16 * RPT * (ldx<FIN>() > LDH ? ldx<FIN>() : LDH); }

// the 16 RPT rows of a tile that this block takes (nrows <= 0: none)
template <int RPT, int NT>
__device__ __forceinline__ Tile block_rows(const Tile* __restrict__ tiles) {
    constexpr int PARTS = MLP_TILE / (NT / 16 * RPT);
    Tile t = tiles[blockIdx.x / PARTS];
    const int skip = NT / 16 * RPT * (int)(blockIdx.x % PARTS);
    t.row0 += skip;
    t.nrows = min(t.nrows - skip, NT / 16 * RPT);
    return t;
}

struct NetsOfLayer {
    NetDev e[MAX_ELEM];
};

// SiLU(z) = z s and SiLU'(z) = s (1 + z (1 - s)) from one correctly rounded
// reciprocal s = 1 / (1 + exp(-z)); h receives SiLU, the result is SiLU'
__device__ __forceinline__ float silu_d(float z, float& h) {
    const float s = __frcp_rn(1.f + expf(-z));
    h = z * s;
    return s * fmaf(z, 1.f - s, 1.f);
}

// Wait (bounded) for the tile's bulk copies on `bar`; all threads agree.  Thread 0
// initialised `bar` and issued the copies before it reaches the first barrier
// here, so no thread polls the mbarrier before its initialisation.  When the
// wait runs out: record FLAG_TIMEOUT, wait once more for the copies in flight
// (FLAG_TIMEOUT_DRAIN if they still have not landed) and return false.
__device__ __forceinline__ bool staged(uint64_t* bar, int* flags) {
    __syncthreads();
    if (__syncthreads_and(bulk::mbar_wait(bar, 0))) return true;
    if (threadIdx.x == 0) atomicOr(&flags[FLAG_TIMEOUT], 1);
    const bool drained = __syncthreads_and(bulk::mbar_wait(bar, 0));
    if (!drained && threadIdx.x == 0) atomicOr(&flags[FLAG_TIMEOUT_DRAIN], 1);
    return false;
}

// acc[i][j] += sum_k A[(RPT ty+i)*LDA + k] * B[k*LDB + 4tx + j], K multiple of 4
template <int K, int LDA, int LDB, int RPT>
__device__ __forceinline__ void mma_rx4(const float* A, const float* B, int ty, int tx, float acc[RPT][4]) {
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        float4 a[RPT], b[4];
#pragma unroll
        for (int i = 0; i < RPT; ++i) a[i] = *reinterpret_cast<const float4*>(A + (RPT * ty + i) * LDA + k);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) b[kk] = *reinterpret_cast<const float4*>(B + (k + kk) * LDB + 4 * tx);
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const float av[4] = {a[i].x, a[i].y, a[i].z, a[i].w};
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                acc[i][0] = fmaf(av[kk], b[kk].x, acc[i][0]);
                acc[i][1] = fmaf(av[kk], b[kk].y, acc[i][1]);
                acc[i][2] = fmaf(av[kk], b[kk].z, acc[i][2]);
                acc[i][3] = fmaf(av[kk], b[kk].w, acc[i][3]);
            }
        }
    }
}

template <int RPT>
__device__ __forceinline__ void set_bias(const float* b, int tx, float acc[RPT][4]) {
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = b ? b[4 * tx + j] : 0.f;
}
// a thread's RPT x 4 values to rows of shared memory (stride LDH)
template <int RPT>
__device__ __forceinline__ void put_rows(float* S, int ty, int tx, const float v[RPT][4]) {
#pragma unroll
    for (int i = 0; i < RPT; ++i)
        *reinterpret_cast<float4*>(S + (RPT * ty + i) * LDH + 4 * tx) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
}

// Sum of NV partial values over the 16 lanes of a half-warp (the tx of one ty), as
// a butterfly reduce-scatter: with NV = 32 lane tx ends with values 2 tx and
// 2 tx + 1, with fewer every lane ends with value tx / (16 / NV).  The order of a
// value's additions does not depend on NV.
template <int NV>
__device__ __forceinline__ void reduce16(float v[NV], int tx) {
    int cnt = NV;
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) {
        if (cnt > 1) {
            const bool upper = tx & off;
            const int half = cnt / 2;
#pragma unroll
            for (int k = 0; k < NV / 2; ++k) {
                if (k < half) {
                    const float send = upper ? v[k] : v[k + half];
                    const float keep = upper ? v[k + half] : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
                }
            }
            cnt = half;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
        }
    }
}

// W3 (64 x OUT) in shared memory with row k = 4 tx + j stored at (j * 16 + tx):
// the 16 lanes of a half-warp read 16 different rows without bank conflicts
template <int OUT>
__device__ __forceinline__ int w3_row(int k) {
    return (k & 3) * 16 + (k >> 2);
}

// The tile part's atomic energies (rows r, lanes with `own`) summed in FP64 in a
// fixed order into *out; sE: ROWS doubles of shared memory.
template <int ROWS>
__device__ __forceinline__ void sum_energies(double* sE, int r, bool own, double e, double* out) {
    __syncthreads();  // every thread is done with the buffer
    if (own) sE[r] = e;
    __syncthreads();
    if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        double x = ROWS == 64 ? sE[l] + sE[l + 32] : (ROWS == 32 || l < 16 ? sE[l] : 0.0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (l == 0) *out = x;
    }
}

// ----------------------------------------------------------- forward ---
// Shared memory: weights (31 KB) and one activation buffer that holds the input
// rows, then h1 (64 x 68 floats at RPT = 4); h2 stays in registers and the output
// layer is a half-warp reduction, so four blocks fit on an SM.  With dsave, the
// row's SiLU derivatives are kept for the reverse pass: dsave[row][0..63] =
// SiLU'(z1), dsave[row][64..127] = SiLU'(z2).
constexpr int kSave = H1 + H2;
template <int OUT, int FIN, int RPT, int NT>
__global__ void __launch_bounds__(NT) k_mlp_fwd(NetsOfLayer nets, const Tile* __restrict__ tiles,
                                               const float* __restrict__ rho, float* __restrict__ out,
                                               int out_stride, GhostOut gh, float* __restrict__ dsave,
                                               double* __restrict__ epart, int* __restrict__ flags) {
    constexpr int R = NT / 16 * RPT;
    __shared__ __align__(8) uint64_t bar;
    extern __shared__ __align__(16) float sm[];
    float* sW1 = sm;                 // FIN x 64
    float* sW2 = sW1 + FIN * H1;     // 64 x 64
    float* sW3 = sW2 + H1 * H2;      // 64 x OUT (8 reserved), rows permuted (w3_row)
    float* sb1 = sW3 + H2 * 8;       // 64
    float* sb2 = sb1 + H1;           // 64
    float* sb3 = sb2 + H2;           // 8
    float* sA = sb3 + 8;             // input rows (stride FIN), then h1 (stride LDH)
    const int tid = threadIdx.x;
    const Tile tl = block_rows<RPT, NT>(tiles);
    if (tl.nrows <= 0) {  // padding entry of a fixed-size tile list, or nothing left of the tile
        pdl_enter();
        if (OUT == 1 && epart && tid == 0) epart[blockIdx.x] = 0.0;
        return;
    }
    const NetDev& w = nets.e[tl.elem];
    const uint32_t xb = (uint32_t)tl.nrows * FIN * 4;
    if (tid == 0) {  // W1, W2 and the input rows by bulk copies (TMA engine)
        bulk::mbar_init(&bar, 1);
        bulk::mbar_init_fence();
        bulk::mbar_expect_tx(&bar, (FIN * H1 + H1 * H2) * 4 + xb);
        bulk::bulk_g2s(sW1, w.W1, FIN * H1 * 4, &bar);
        bulk::bulk_g2s(sW2, w.W2, H1 * H2 * 4, &bar);
    }
    for (int i = tid; i < H2 * OUT; i += NT) sW3[w3_row<OUT>(i / OUT) * OUT + i % OUT] = w.W3[i];
    for (int i = tid; i < H1; i += NT) sb1[i] = w.b1[i];
    for (int i = tid; i < H2; i += NT) sb2[i] = w.b2[i];
    if (tid < OUT) sb3[tid] = w.b3[tid];
    for (int i = tl.nrows * FIN + tid; i < R * FIN; i += NT) sA[i] = 0.f;  // rows past the end
    pdl_enter();
    if (tid == 0) bulk::bulk_g2s(sA, rho + (size_t)tl.row0 * FIN, xb, &bar);
    if (!staged(&bar, flags)) return;
    const int ty = tid >> 4, tx = tid & 15;
    float acc[RPT][4];
    // layer 1
    set_bias<RPT>(sb1, tx, acc);
    mma_rx4<FIN, ldx<FIN>(), H1, RPT>(sA, sW1, ty, tx, acc);
    float ds[RPT][4];  // SiLU'(z1) (acc becomes h1)
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) ds[i][j] = silu_d(acc[i][j], acc[i][j]);
    if (dsave)
#pragma unroll
        for (int i = 0; i < RPT; ++i)
            if (RPT * ty + i < tl.nrows)
                *reinterpret_cast<float4*>(dsave + (size_t)(tl.row0 + RPT * ty + i) * kSave + 4 * tx) =
                    make_float4(ds[i][0], ds[i][1], ds[i][2], ds[i][3]);
    __syncthreads();  // every thread is done reading the input rows
    put_rows<RPT>(sA, ty, tx, acc);
    __syncthreads();
    // layer 2 (h2 stays in registers)
    set_bias<RPT>(sb2, tx, acc);
    mma_rx4<H1, LDH, H2, RPT>(sA, sW2, ty, tx, acc);
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) ds[i][j] = silu_d(acc[i][j], acc[i][j]);  // acc becomes h2
    if (dsave)
#pragma unroll
        for (int i = 0; i < RPT; ++i)
            if (RPT * ty + i < tl.nrows)
                *reinterpret_cast<float4*>(dsave + (size_t)(tl.row0 + RPT * ty + i) * kSave + H1 + 4 * tx) =
                    make_float4(ds[i][0], ds[i][1], ds[i][2], ds[i][3]);
    // layer 3: per-thread partial dot products over its 4 columns, reduced over tx
    constexpr int NV = RPT * OUT, PER = NV > 16 ? NV / 16 : 1, DUP = NV < 16 ? 16 / NV : 1;
    float v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float* w3 = sW3 + (j * 16 + tx) * OUT;
#pragma unroll
        for (int o = 0; o < OUT; ++o) {
            const float wv = w3[o];
#pragma unroll
            for (int i = 0; i < RPT; ++i) v[i * OUT + o] = fmaf(acc[i][j], wv, v[i * OUT + o]);
        }
    }
    reduce16<NV>(v, tx);
    const int q0 = tx / DUP * PER, r = RPT * ty + q0 / OUT, o = q0 % OUT;  // this lane's value(s): row r, outputs o ..
    const bool own = tx % DUP == 0;
    if (OUT == 1) {
        const float e = v[0] + sb3[0];
        if (own && r < tl.nrows) out[(size_t)(tl.row0 + r) * out_stride] = e;
        if (epart)
            sum_energies<R>(reinterpret_cast<double*>(sA), r, own, r < tl.nrows ? (double)e : 0.0, epart + blockIdx.x);
    } else if (own && r < tl.nrows) {
        const int64_t i = tl.row0 + r;
        float y[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            y[k] = v[k] + sb3[o + k];
            out[(size_t)i * out_stride + o + k] = y[k];
        }
        if (gh.goff)  // the row's ghost images get the same coefficients (Fig. 4a)
            for (int64_t g = gh.goff[i]; g < gh.goff[i + 1] && g < gh.gcap; ++g)
#pragma unroll
                for (int k = 0; k < PER; ++k) out[(size_t)(gh.base + g) * out_stride + o + k] = y[k];
    }
}

// ---------------------------------------------------------- backward ---
// rhobar = W1 (s1 * (W2 (s2 * (W3 ybar))))   per row, with s1 = SiLU'(z1) and
// s2 = SiLU'(z2) kept by the forward (dsave), so nothing is recomputed.
// Shared memory: the transposed weights, ybar, one activation buffer (z2bar, then
// z1bar) and, with BBAR, the rhobar rows and the contraction weights.
//
// BBAR (Eq. 1's squares only): instead of writing rhobar, go on to the density
// adjoint's first step for the rows (bbar_records).
__device__ __forceinline__ float4 ld_save(const float* dsave, const Tile& tl, int r, int col) {
    if (r >= tl.nrows) return make_float4(0.f, 0.f, 0.f, 0.f);
    return __ldg(reinterpret_cast<const float4*>(dsave + (size_t)(tl.row0 + r) * kSave + col));
}

// rhobar = z1bar W1^T for the block's rows (z1bar in sG): into sR (stride LDH) with BBAR, else to memory
template <int FIN, bool BBAR, int RPT>
__device__ __forceinline__ void rhobar_rows(const float* sG, const float* sW1t, float* sR, float* __restrict__ rhobar,
                                            const Tile& tl, int ty, int tx) {
    for (int cg = tx; cg < FIN / 4; cg += 16) {  // FIN / 4 column groups of 4 over the 16 tx
        float acc[RPT][4];
        set_bias<RPT>(nullptr, tx, acc);
        mma_rx4<H1, LDH, FIN, RPT>(sG, sW1t, ty, cg, acc);
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = RPT * ty + i;
            if (BBAR) {
                *reinterpret_cast<float4*>(sR + r * LDH + 4 * cg) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            } else if (r < tl.nrows) {
                *reinterpret_cast<float4*>(rhobar + (size_t)(tl.row0 + r) * FIN + 4 * cg) =
                    make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
            }
        }
    }
}

// contraction weights transposed per l: sWc[(l N_orb + k) N_phi + m] = W_{l,m,k}
template <int NT>
__device__ __forceinline__ void stage_wc(float* sWc, const float* __restrict__ Wt, int tid) {
    for (int i = tid; i < (LMAX + 1) * NPHI * NORB; i += NT) {
        const int l = i / (NPHI * NORB), m = (i / NORB) % NPHI, k = i % NORB;
        sWc[(l * NORB + k) * NPHI + m] = Wt[i];
    }
}

// The bbar step of the block's rows, written as their adjoint records (bbar with the layer's c, ghost
// images too) through sRec.  Four threads per row, up to three terms of one l each, or eight, up to two.
template <int RPT, int NT>
__device__ __forceinline__ void bbar_records(const float* sR, const float* sWc, float* sRec, const Tile& tl,
                                             const float* __restrict__ bck, const float* __restrict__ coef,
                                             float* __restrict__ rec, const GhostOut& gh, int tid) {
    constexpr int TPR = 16 / RPT;
    const int r = tid / TPR, q = tid % TPR;
    if (r < tl.nrows) {
        const size_t row = (size_t)(tl.row0 + r);
        const float* rb = sR + r * LDH;
        const float* b = bck + row * NB;
        if constexpr (TPR == 4) {
            // q = 0: term 0 (and two that are not kept, in step with its neighbours), c and 0;
            // q = 1, 2, 3: terms 1-3, 4-6, 7-9
            const int l = q == 0 ? 0 : (q == 1 ? 1 : 2);
            bbar_terms<3>(b, sWc + l * NORB * NPHI, rb + l * NORB, q == 0 ? 0 : 3 * q - 2, q == 0 ? 1 : 3, sRec, r);
            if (q == 0) {
                float o[NPHI];
                rec_tail(coef, row, NANG, o);
                stage_rec(sRec, r, NANG, o);
                rec_tail(coef, row, NANG + 1, o);
                stage_rec(sRec, r, NANG + 1, o);
            }
        } else {
            // q = 0: term 0 (and one that is not kept); 1, 2: terms 1 and 2, 3; 3, 4, 5: two terms each; 6, 7: c and 0
            static_assert(TPR == 8, "four or eight threads per row");
            if (q >= 6) {
                float o[NPHI];
                rec_tail(coef, row, NANG + q - 6, o);
                stage_rec(sRec, r, NANG + q - 6, o);
            } else {
                const int l = q == 0 ? 0 : (q <= 2 ? 1 : 2), a0 = q == 0 ? 0 : (q <= 2 ? 2 * q - 1 : 2 * q - 2);
                bbar_terms<2>(b, sWc + l * NORB * NPHI, rb + l * NORB, a0, q == 0 || q == 2 ? 1 : 2, sRec, r);
            }
        }
    }
    __syncthreads();
    flush_rec(sRec, tl.nrows, tl.row0, rec, gh, tid, NT);  // ghost images get the rows' records too (reverse exchange)
}

template <int OUT, int FIN, bool BBAR, int RPT, int NT>
__global__ void __launch_bounds__(NT, 3) k_mlp_bwd(NetsOfLayer nets, const Tile* __restrict__ tiles,
                                               const float* __restrict__ dsave, const float* __restrict__ ybar,
                                               float* __restrict__ rhobar, const float* __restrict__ Wt,
                                               const float* __restrict__ bck, const float* __restrict__ coef,
                                               float* __restrict__ rec, GhostOut gh, int* __restrict__ flags) {
    constexpr int R = NT / 16 * RPT;
    __shared__ __align__(8) uint64_t bar;
    extern __shared__ __align__(16) float sm[];
    float* sW1t = sm;                 // W1^T: 64 x FIN
    float* sW2t = sW1t + H1 * FIN;    // W2^T: 64 x 64
    float* sW3t = sW2t + H1 * H2;     // W3^T: OUT x 64 (8 rows reserved)
    float* sY = sW3t + 8 * H2;        // R x 8
    float* sG = sY + R * 8;           // z2bar, then z1bar (stride LDH)
    float* sR = sG + R * LDH;         // rhobar rows (BBAR, stride LDH)
    float* sWc = sR + R * LDH;        // (L+1) x N_orb x N_phi contraction W^t, transposed per l (BBAR)
    const int tid = threadIdx.x;
    const Tile tl = block_rows<RPT, NT>(tiles);
    if (tl.nrows <= 0) {  // padding entry of a fixed-size tile list, or nothing left of the tile
        pdl_enter();
        return;
    }
    const int ty = tid >> 4, tx = tid & 15;
    const NetDev& w = nets.e[tl.elem];
    if (tid == 0) {  // W1^T, W2^T, W3^T by bulk copies (TMA engine)
        bulk::mbar_init(&bar, 1);
        bulk::mbar_init_fence();
        bulk::mbar_expect_tx(&bar, (H1 * FIN + H1 * H2 + OUT * H2) * 4);
        bulk::bulk_g2s(sW1t, w.W1t, H1 * FIN * 4, &bar);
        bulk::bulk_g2s(sW2t, w.W2t, H1 * H2 * 4, &bar);
        bulk::bulk_g2s(sW3t, w.W3t, OUT * H2 * 4, &bar);
    }
    if (BBAR) stage_wc<NT>(sWc, Wt, tid);
    pdl_enter();
    // the thread's SiLU'(z2), in flight while ybar and the weights arrive
    float4 s2[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) s2[i] = ld_save(dsave, tl, RPT * ty + i, H1 + 4 * tx);
    for (int i = tid; i < R * OUT; i += NT) {
        const int r = i / OUT, o = i % OUT;
        sY[r * 8 + o] = (OUT == 1) ? 1.f : (r < tl.nrows ? ybar[(size_t)(tl.row0 + r) * OUT + o] : 0.f);
    }
    if (!staged(&bar, flags)) return;
    // z2bar = (ybar W3^T) * s2 -> sG
    float acc[RPT][4];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int o = 0; o < OUT; ++o) {
            const float y = sY[(RPT * ty + i) * 8 + o];
            const float4 wv = *reinterpret_cast<const float4*>(sW3t + o * H2 + 4 * tx);
            v[0] = fmaf(y, wv.x, v[0]);
            v[1] = fmaf(y, wv.y, v[1]);
            v[2] = fmaf(y, wv.z, v[2]);
            v[3] = fmaf(y, wv.w, v[3]);
        }
        acc[i][0] = v[0] * s2[i].x, acc[i][1] = v[1] * s2[i].y, acc[i][2] = v[2] * s2[i].z, acc[i][3] = v[3] * s2[i].w;
    }
    put_rows<RPT>(sG, ty, tx, acc);
    float4 s1[RPT];  // SiLU'(z1), in flight during the z1bar product
#pragma unroll
    for (int i = 0; i < RPT; ++i) s1[i] = ld_save(dsave, tl, RPT * ty + i, 4 * tx);
    __syncthreads();
    // z1bar = (z2bar W2^T) * s1
    set_bias<RPT>(nullptr, tx, acc);
    mma_rx4<H2, LDH, H1, RPT>(sG, sW2t, ty, tx, acc);
    __syncthreads();  // everyone is done reading z2bar
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        acc[i][0] *= s1[i].x, acc[i][1] *= s1[i].y, acc[i][2] *= s1[i].z, acc[i][3] *= s1[i].w;
    }
    put_rows<RPT>(sG, ty, tx, acc);
    __syncthreads();
    rhobar_rows<FIN, BBAR, RPT>(sG, sW1t, sR, rhobar, tl, ty, tx);
    if (!BBAR) return;
    __syncthreads();
    // records staged where W1^T, W2^T, no longer needed, were
    bbar_records<RPT, NT>(sR, sWc, sW1t, tl, bck, coef, rec, gh, tid);
}

static_assert(NFEAT * H1 + H1 * H2 >= MLP_TILE * kRecLd, "record staging must fit in the W1, W2 region");

// ------------------------------------------------------ energy network ---
// Forward and backward of the energy network (48 -> 64 -> 64 -> 1) of the block's
// rows, then the bbar step: eps, the tile's FP64 energy and the adjoint records.
// ybar = 1, so z2bar = W3 * SiLU'(z2) and nothing but rho is read.  Shared memory: W1,
// W2 (later rhobar) and W1^T, W2^T (later the records), one activation buffer, the
// contraction weights: 76 KB, three blocks per SM.
template <int RPT, int NT>
__global__ void __launch_bounds__(NT, 3) k_mlp_energy(NetsOfLayer nets, const Tile* __restrict__ tiles,
                                                      const float* __restrict__ rho, float* __restrict__ eps,
                                                      double* __restrict__ epart, const float* __restrict__ Wt,
                                                      const float* __restrict__ bck, const float* __restrict__ coef,
                                                      float* __restrict__ rec, GhostOut gh, int* __restrict__ flags) {
    constexpr int R = NT / 16 * RPT, F = NFEAT;
    static_assert(F * H1 + H1 * H2 >= R * LDH, "rhobar rows must fit in the W1, W2 region");
    __shared__ __align__(8) uint64_t bar;
    extern __shared__ __align__(16) float sm[];
    float* sW1 = sm;                // 48 x 64
    float* sW2 = sW1 + F * H1;      // 64 x 64
    float* sW1t = sW2 + H1 * H2;    // 64 x 48
    float* sW2t = sW1t + H1 * F;    // 64 x 64
    float* sA = sW2t + H1 * H2;     // input rows (stride 48), then h1, z2bar, z1bar (stride LDH)
    float* sWc = sA + R * LDH;      // contraction weights, transposed per l
    const int tid = threadIdx.x;
    const Tile tl = block_rows<RPT, NT>(tiles);
    if (tl.nrows <= 0) {  // padding entry of a fixed-size tile list, or nothing left of the tile
        pdl_enter();
        if (epart && tid == 0) epart[blockIdx.x] = 0.0;
        return;
    }
    const NetDev& w = nets.e[tl.elem];
    const uint32_t xb = (uint32_t)tl.nrows * F * 4;
    if (tid == 0) {
        bulk::mbar_init(&bar, 1);
        bulk::mbar_init_fence();
        bulk::mbar_expect_tx(&bar, 2 * (F * H1 + H1 * H2) * 4 + xb);
        bulk::bulk_g2s(sW1, w.W1, F * H1 * 4, &bar);
        bulk::bulk_g2s(sW2, w.W2, H1 * H2 * 4, &bar);
        bulk::bulk_g2s(sW1t, w.W1t, F * H1 * 4, &bar);
        bulk::bulk_g2s(sW2t, w.W2t, H1 * H2 * 4, &bar);
    }
    stage_wc<NT>(sWc, Wt, tid);
    for (int i = tl.nrows * F + tid; i < R * F; i += NT) sA[i] = 0.f;  // rows past the end
    const int ty = tid >> 4, tx = tid & 15;
    const float4 b1 = __ldg(reinterpret_cast<const float4*>(w.b1) + tx), b2 = __ldg(reinterpret_cast<const float4*>(w.b2) + tx);
    const float4 w3 = __ldg(reinterpret_cast<const float4*>(w.W3) + tx);
    const float b3 = __ldg(w.b3);
    pdl_enter();
    if (tid == 0) bulk::bulk_g2s(sA, rho + (size_t)tl.row0 * F, xb, &bar);
    if (!staged(&bar, flags)) return;
    float acc[RPT][4], s1[RPT][4];
#pragma unroll
    for (int i = 0; i < RPT; ++i) acc[i][0] = b1.x, acc[i][1] = b1.y, acc[i][2] = b1.z, acc[i][3] = b1.w;
    mma_rx4<F, F, H1, RPT>(sA, sW1, ty, tx, acc);
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s1[i][j] = silu_d(acc[i][j], acc[i][j]);  // acc becomes h1
    __syncthreads();  // every thread is done reading the input rows
    put_rows<RPT>(sA, ty, tx, acc);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RPT; ++i) acc[i][0] = b2.x, acc[i][1] = b2.y, acc[i][2] = b2.z, acc[i][3] = b2.w;
    mma_rx4<H1, LDH, H2, RPT>(sA, sW2, ty, tx, acc);
    float v[RPT];  // this thread's share of eps (the sum's order is k_mlp_fwd's)
    const float wv[4] = {w3.x, w3.y, w3.z, w3.w};
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        v[i] = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float h;
            const float d = silu_d(acc[i][j], h);
            v[i] = fmaf(h, wv[j], v[i]);
            acc[i][j] = wv[j] * d;  // z2bar
        }
    }
    reduce16<RPT>(v, tx);
    constexpr int DUP = 16 / RPT;
    const int r = RPT * ty + tx / DUP;
    const bool own = tx % DUP == 0;
    const float e = v[0] + b3;
    if (own && r < tl.nrows) eps[tl.row0 + r] = e;
    if (epart)
        sum_energies<R>(reinterpret_cast<double*>(sA), r, own, r < tl.nrows ? (double)e : 0.0, epart + blockIdx.x);
    __syncthreads();  // h1 and the energies have been read
    put_rows<RPT>(sA, ty, tx, acc);
    __syncthreads();
    set_bias<RPT>(nullptr, tx, acc);
    mma_rx4<H2, LDH, H1, RPT>(sA, sW2t, ty, tx, acc);
#pragma unroll
    for (int i = 0; i < RPT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] *= s1[i][j];  // z1bar
    __syncthreads();
    put_rows<RPT>(sA, ty, tx, acc);
    __syncthreads();
    rhobar_rows<F, true, RPT>(sA, sW1t, sW1, nullptr, tl, ty, tx);
    __syncthreads();
    bbar_records<RPT, NT>(sW1, sWc, sW1t, tl, bck, coef, rec, gh, tid);
}

template <int FIN, int RPT, int NT>
constexpr size_t fwd_smem() { return sizeof(float) * (FIN * H1 + H1 * H2 + H2 * 8 + H1 + H2 + 8 + abuf<FIN, RPT, NT>()); }
template <int FIN, bool BBAR, int RPT, int NT>
constexpr size_t bwd_smem() {
    return sizeof(float) * (H1 * FIN + H1 * H2 + 8 * H2 + NT / 16 * RPT * 8 + NT / 16 * RPT * LDH +
                            (BBAR ? NT / 16 * RPT * LDH + (LMAX + 1) * NPHI * NORB : 0));
}
template <int RPT, int NT>
constexpr size_t energy_smem() {
    return sizeof(float) * (2 * (NFEAT * H1 + H1 * H2) + NT / 16 * RPT * LDH + (LMAX + 1) * NPHI * NORB);
}
static_assert(3 * (energy_smem<4, 256>() + 16 + 1024) <= 228 * 1024, "three blocks of the energy network per SM");

template <typename K>
void allow_smem(K* k, size_t bytes) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <int RPT, int NT>
void set_fwd_attrs() {
    allow_smem(k_mlp_fwd<NPHI, NFEAT, RPT, NT>, fwd_smem<NFEAT, RPT, NT>());
    allow_smem(k_mlp_fwd<1, NFEAT_P, RPT, NT>, fwd_smem<NFEAT_P, RPT, NT>());
    allow_smem(k_mlp_fwd<NPHI, NFEAT_P, RPT, NT>, fwd_smem<NFEAT_P, RPT, NT>());
    allow_smem(k_mlp_energy<RPT, NT>, energy_smem<RPT, NT>());
}
template <int RPT, int NT>
void set_bwd_attrs() {
    allow_smem(k_mlp_bwd<NPHI, NFEAT, true, RPT, NT>, bwd_smem<NFEAT, true, RPT, NT>());
    allow_smem(k_mlp_bwd<1, NFEAT_P, false, RPT, NT>, bwd_smem<NFEAT_P, false, RPT, NT>());
    allow_smem(k_mlp_bwd<NPHI, NFEAT_P, false, RPT, NT>, bwd_smem<NFEAT_P, false, RPT, NT>());
}
void ensure_attrs() {
    // once per device, safe under concurrent first calls
    static std::mutex mu;
    static uint64_t done = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 64 && ((done >> dev) & 1)) return;
    set_fwd_attrs<2, 128>();
    set_fwd_attrs<2, 256>();
    set_fwd_attrs<4, 256>();
    set_bwd_attrs<2, 128>();
    set_bwd_attrs<4, 128>();
    set_bwd_attrs<4, 256>();
    if (dev < 64) done |= (uint64_t)1 << dev;
}

NetsOfLayer layer_nets(const NetTable& t, int layer) {
    NetsOfLayer n;
    for (int e = 0; e < MAX_ELEM; ++e) n.e[e] = t.net[layer][e];
    return n;
}

}  // namespace

// Parts while they still fit the 152 SMs in one wave.  us per launch of the coefficient
// network's forward / energy network / backward with 1, 2 and 4 parts of 256 threads: 4 tiles (192
// atoms) 8.7 / 18.5 / 13.5, 6.3 / 13.6 / 9.8, 5.4 / 10.4 / 7.5; 63 tiles 8.4 / 17.7 / 12.6, 6.3 / 13.6 / 9.9,
// 7.8 / 15.8 / 11.4; 96 tiles 8.5 / 17.5 / 12.2, 9.3 / 19.8 / 14.5, 10.2 / 21.7 / 15.2.  A part's time is that of its
// shared-memory fragments, of which two rows per thread need 40 % less per row than one: quarters with 128
// threads instead of 256 took an evaluation of 192 atoms from 70.7 to 66.8 us, of 1,536 from 77.7 to 74.4
// (with 64 threads and four rows each 74.0 and 82.2); halves with 128 threads in the backward
// one of 4,500 from 108.5 to 105.4 (in the forward networks 108.6).
int mlp_parts_f32(const reann_nlist* nl) {
    const int64_t nt = tiles_of(nl);
    return nt <= 38 ? 4 : (nt <= 76 ? 2 : 1);
}

cudaError_t launch_mlp_fwd_f32(cudaStream_t s, const reann_nlist* nl, const NetTable& nets, int t, bool energy,
                               const float* rho, float* out, int out_stride, bool pairs, GhostOut gh, float* dsave,
                               double* epart, int* flags) {
    const int nt = (int)tiles_of(nl), parts = mlp_parts_f32(nl);
    if (nt == 0) return cudaSuccess;
    if (energy && !pairs) return cudaErrorInvalidValue;  // launch_mlp_energy_f32
    ensure_attrs();
    const NetsOfLayer ln = layer_nets(nets, t);
    const EvalLaunch how = eval_launch(nl);
#define REANN_FWD(O, F, RPT, NT)                                                                                         \
    launch_with(how.chain, how.carve(), k_mlp_fwd<O, F, RPT, NT>, nt * parts, NT, fwd_smem<F, RPT, NT>(), s, ln, nl->tiles, \
                rho, out, out_stride, gh, dsave, epart, flags)
#define REANN_FWD_R(O, F)        \
    do {                         \
        if (parts == 4)          \
            REANN_FWD(O, F, 2, 128);  \
        else if (parts == 2)     \
            REANN_FWD(O, F, 2, 256);  \
        else                     \
            REANN_FWD(O, F, 4, 256);  \
    } while (0)
    if (!pairs)
        REANN_FWD_R(NPHI, NFEAT);
    else if (energy)
        REANN_FWD_R(1, NFEAT_P);
    else
        REANN_FWD_R(NPHI, NFEAT_P);
#undef REANN_FWD_R
#undef REANN_FWD
    return cudaGetLastError();
}

cudaError_t launch_mlp_bwd_f32(cudaStream_t s, const reann_nlist* nl, const NetTable& nets, int t, bool energy,
                               const float* dsave, const float* ybar, float* rhobar, int* flags, bool pairs,
                               const float* Wt, const float* bck, const float* coef, float* rec, GhostOut gh) {
    const int nt = (int)tiles_of(nl), parts = mlp_parts_f32(nl);
    if (nt == 0) return cudaSuccess;
    if (energy && !pairs) return cudaErrorInvalidValue;  // launch_mlp_energy_f32
    ensure_attrs();
    const NetsOfLayer ln = layer_nets(nets, t);
    const EvalLaunch how = eval_launch(nl);
#define REANN_BWD(O, F, B, RPT, NT)                                                                                    \
    launch_with(how.chain, how.carve(), k_mlp_bwd<O, F, B, RPT, NT>, nt * parts, NT, bwd_smem<F, B, RPT, NT>(), s, ln,  \
                nl->tiles, dsave, ybar, rhobar, B ? Wt : nullptr, B ? bck : nullptr, B ? coef : nullptr,           \
                B ? rec : nullptr, B ? gh : GhostOut{}, flags)
#define REANN_BWD_R(O, F, B)        \
    do {                            \
        if (parts == 4)             \
            REANN_BWD(O, F, B, 2, 128);  \
        else if (parts == 2)        \
            REANN_BWD(O, F, B, 4, 128);  \
        else                        \
            REANN_BWD(O, F, B, 4, 256);  \
    } while (0)
    if (!pairs)
        REANN_BWD_R(NPHI, NFEAT, true);
    else if (energy)
        REANN_BWD_R(1, NFEAT_P, false);
    else
        REANN_BWD_R(NPHI, NFEAT_P, false);
#undef REANN_BWD_R
#undef REANN_BWD
    return cudaGetLastError();
}

cudaError_t launch_mlp_energy_f32(cudaStream_t s, const reann_nlist* nl, const NetTable& nets, int t, const float* rho,
                                  float* eps, double* epart, const float* Wt, const float* bck, const float* coef,
                                  float* rec, GhostOut gh, int* flags) {
    const int nt = (int)tiles_of(nl), parts = mlp_parts_f32(nl);
    if (nt == 0) return cudaSuccess;
    ensure_attrs();
    const NetsOfLayer ln = layer_nets(nets, t);
    const EvalLaunch how = eval_launch(nl);
#define REANN_EN(RPT, NT)                                                                                            \
    launch_with(how.chain, how.carve(), k_mlp_energy<RPT, NT>, nt * parts, NT, energy_smem<RPT, NT>(), s, ln, nl->tiles, \
                rho, eps, epart, Wt, bck, coef, rec, gh, flags)
    if (parts == 4)
        REANN_EN(2, 128);
    else if (parts == 2)
        REANN_EN(2, 256);
    else
        REANN_EN(4, 256);
#undef REANN_EN
    return cudaGetLastError();
}

}  // namespace reann
