// Edge kernels of the REANN message-passing layer and its adjoint.
//
// Forward (Sec. 2.1, Eq. 1), per owned atom i and layer t:
//   b_{i,a,m} = sum_{j live} c^t_{j,m} phi_m(d_ij) A_a(r_ij)
//   g_{i,a,k} = sum_m b_{i,a,m} W^t_{l(a),m,k}
//   rho_{i,l,k} = sum_{a in l} w_a g_{i,a,k}^2
// Reverse (Sec. 2.2, Eqs. 3-5), per layer, given rhobar:
//   gbar = 2 w_a g rhobar,  bbar_{a,m} = sum_k gbar_{a,k} W_{l(a),m,k}
//   and, gathering over atom k's own (symmetric, full) list with r = r_j - r_k:
//     dE/dr_k = -sum_j sum_{a,m} [bbar_{k,a,m} c_{j,m} + (-1)^l bbar_{j,a,m} c_{k,m}] grad_r(phi_m A_a)(r)
//     cbar_{k,m} = sum_j phi_m(d) sum_a (-1)^l bbar_{j,a,m} A_a(r)
//   (the second term of each line is the reverse edge j -> k, written with
//   A_a(-r) = (-1)^l A_a(r); ghost slots j carry their owner's bbar, which is
//   the paper's ghost-gradient exchange as a vector-Jacobian product, Sec. 2.2).
// No atomics: every output row is written by the lanes of its own centre atom.
//
// Edge records.  The list of live (d < r_c) edges and everything about an edge
// that is the same in all 2T edge passes of an evaluation is computed once per
// evaluation (k_edges): r = r_j - r_i and j, the first Gaussian times the cutoff
// and the factor of the Gaussian recurrence, d and the cutoff's logarithmic
// derivative (32 B per live edge, in the row order of the list).  The passes
// stream the records of their atom (coalesced) and gather only what belongs to
// the neighbour: its coefficients (forward) or its adjoint record (reverse).
// Both passes give 4 to 32 lanes to a centre atom, more where there are few atoms.
// The order in which an atom's edges are summed follows the size of its structure
// and never how many rows a launch has (see the passes).
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"

namespace reann {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kEdgeWarps = 8;  // warps (centre atoms) per block of the edge kernels

// exp(a + b) for |a| < 80 and a small correction b (the rounding error of a) by
// Cody-Waite range reduction (W. J. Cody and W. Waite, Software Manual for the
// Elementary Functions, 1980): a = k ln2 + r with ln2 split into a short high part
// (k ln2_hi exact) and a correction, |r| <= ln2/2, then the degree-7 Taylor
// polynomial of exp(r + b) (truncation < 6e-9 relative) in Horner form and an exact
// scaling by 2^k.  Measured on the GPU against FP64 its mean relative error is
// ~1e-9 (unbiased), so the m-fold Gaussian recurrence below does not turn a
// one-sided rounding habit into a shift of every phi_m.
__device__ __forceinline__ float exp_cw(float a, float b) {
    a = fminf(fmaxf(a, -87.f), 88.f);  // keeps 2^k a normal float
    const float k = rintf(a * 1.44269504f);
    float r = fmaf(-k, 0.693145751953125f, a);
    r = fmaf(-k, 1.428606820309417e-06f, r) + b;
    float p = 1.f / 5040.f;
    p = fmaf(p, r, 1.f / 720.f);
    p = fmaf(p, r, 1.f / 120.f);
    p = fmaf(p, r, 1.f / 24.f);
    p = fmaf(p, r, 1.f / 6.f);
    p = fmaf(p, r, 0.5f);
    p = fmaf(p, r, 1.f);
    p = fmaf(p, r, 1.f);
    return p * __int_as_float(((int)k + 127) << 23);
}

// exp(sign (x + x_lo) (c_hi + c_lo)) with the product's rounding error carried along
__device__ __forceinline__ float exp_prod(float sign, float x, float x_lo, float c_hi, float c_lo) {
    const float a = x * c_hi;
    return exp_cw(sign * a, sign * (fmaf(x, c_hi, -a) + fmaf(x, c_lo, x_lo * c_hi)));
}

// All Gaussians from the first one by the equal-spacing recurrence
//   exp(-a(d-mu_{m+1})^2) = exp(-a(d-mu_m)^2) q kappa_m,  q = exp(2 a Delta d),
// kappa_m a float pair (see Radial).  The first value carries f_c and the power of
// two R.scale, which keeps it normal near r_c for every a r_c^2 <= 80; the passes
// multiply their sums by R.unscale.
__device__ __forceinline__ void phi_chain(const Radial& R, float phi_first, float q, float phi[NPHI]) {
    phi[0] = phi_first;
#pragma unroll
    for (int m = 0; m + 1 < NPHI; ++m) {
        const float p = phi[m] * q;
        phi[m + 1] = fmaf(p, R.kap_hi[m], p * R.kap_lo[m]);
    }
}

// f_c(d) = (cos(pi d/r_c)/2 + 1/2)^2 evaluated as cos^4(pi x / 2), x = d / r_c
// taken with 1/r_c as a float pair (d inv_hi + d inv_lo: within an ulp of the
// correctly rounded quotient and without the one-sided error of a rounded 1/r_c,
// which near r_c, where the cutoff's logarithmic derivative is large, would
// bias every atom), no rounded pi constant, and no cancellation of 1/2 + cos/2
// near d = r_c.  f_c' / f_c = -(2 pi / r_c) tan(pi x / 2), finite also where the
// cosine rounds to zero (f_c is zero there).
__device__ __forceinline__ void cutoff(const Radial& R, float d, float& fc, float& dlog) {
    float s, c;
    const float x = fmaf(d, R.inv_rc_hi, d * R.inv_rc_lo);
    sincospif(0.5f * x, &s, &c);
    const float c2 = c * c;
    fc = c2 * c2;
    const float u = -6.28318530717959f * s / (c == 0.f ? 1e-20f : c);
    dlog = fmaf(u, R.inv_rc_hi, u * R.inv_rc_lo);
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }

// 32 consecutive bytes (32 B aligned) in one load: one instruction and one tag lookup for a
// neighbour's coefficients or position.  Volatile with a memory clobber, like every load written in
// assembly here: kernels read what the one before wrote, and nothing else keeps such a load behind pdl_enter().
__device__ __forceinline__ void ldg8(const void* p, float4& a, float4& b) {
    asm volatile("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                 : "l"(p)
                 : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p) : "memory"); }

// K = 1, 2 or 4 consecutive floats (aligned to their size)
template <int K>
__device__ __forceinline__ void ldk(const float* p, float* v) {
    if constexpr (K == 4) {
        const float4 x = ld4(p);
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    } else if constexpr (K == 2) {
        const float2 x = *reinterpret_cast<const float2*>(p);
        v[0] = x.x, v[1] = x.y;
    } else {
        v[0] = p[0];
    }
}
template <int K>
__device__ __forceinline__ void stk(float* p, const float* v) {
    if constexpr (K == 4)
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (K == 2)
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    else
        p[0] = v[0];
}

// Orbital pair (k, k'), k <= k', of pair feature p = 0..35 (row-major over k)
__constant__ unsigned char c_pair_k[NORB_P * (NORB_P + 1) / 2];
__constant__ unsigned char c_pair_k2[NORB_P * (NORB_P + 1) / 2];

// -------------------------------------------------------------- edges ----
// Live (d < r_c) entries of the list rows [row0, row0 + rows) and their records,
// one warp per row; row row0 + k's records go to record row k.  A batch of 32
// entries is tested, one per lane; the kept ones are queued in shared memory and
// their records computed 32 at a time, so that the transcendental functions run
// with full warps and the records are stored as whole lines.  (Queues that run on
// over 2, 4 or 8 rows of a warp, to fill the last batch of a row as well, were
// measured at 1.13 x, 1.08 x and 1.05 x the time for 24,576 to 32,000 atoms and
// 0.91 x for 1,048,576.)  Bound by the latency of the position gathers; with the next batch's
// positions fetched ahead 192 atoms take 3.6 instead of 4.2 us, 24,576 20.4 instead of 21.9,
// 1,048,576 720 instead of 787 (writing 2.8 GB of records there takes 410).
//   xyzj = (r, j as bits); phi = (phi_0 R.scale, q) of phi_chain; der = (d, f_c' / f_c)
__global__ void __launch_bounds__(kEdgeWarps * 32) k_edges(int64_t row0, int64_t rows, int stride, Radial R,
                                                           const int32_t* __restrict__ nbr,
                                                           const int32_t* __restrict__ cnt,
                                                           const float4* __restrict__ pos, float4* __restrict__ xyzj,
                                                           float2* __restrict__ phi, float2* __restrict__ der,
                                                           int32_t* __restrict__ live_cnt, int* __restrict__ flags) {
    pdl_enter();
    __shared__ float4 queue[kEdgeWarps][64];
    const int lane = threadIdx.x & 31;
    const int64_t k = (int64_t)blockIdx.x * kEdgeWarps + (threadIdx.x >> 5);
    if (k >= rows) return;
    const int64_t i = row0 + k;
    float4* q = queue[threadIdx.x >> 5];
    float4 hi_i, lo_i;
    ldg8(pos + 2 * i, hi_i, lo_i);
    const int c = cnt[i];
    const int32_t* row = nbr + (size_t)i * stride;
    const size_t out = (size_t)k * stride;
    int done = 0, tail = 0;  // records written, entries ever queued (queue index mod 64)
    auto emit = [&]() {      // the record of queue entry done + lane
        const float4 e = q[(done + lane) & 63];
        const float d = sqrtf(e.x * e.x + e.y * e.y + e.z * e.z);
        float fc, dlog;
        cutoff(R, d, fc, dlog);
        // every radial function is that of the same rounded d (its rounding then acts like a
        // displacement of 1e-7 A, to which all of them respond together)
        const float dd = d * d;
        const float g0 = exp_prod(-1.f, dd, fmaf(d, d, -dd), R.alpha_hi, R.alpha_lo);
        const float qf = exp_prod(1.f, d, 0.f, R.tad_hi, R.tad_lo);
        xyzj[out + done + lane] = e;
        phi[out + done + lane] = make_float2(g0 * R.scale * fc, qf);
        der[out + done + lane] = make_float2(d, dlog);
    };
    // the next batch's positions and the indices of the one after it are on their way meanwhile
    int j = lane < c ? row[lane] : 0, j1 = lane + 32 < c ? row[lane + 32] : 0;
    float4 hj, lj;
    if (lane < c) ldg8(pos + 2 * (int64_t)j, hj, lj);
    for (int base = 0; base < c; base += 32) {
        const bool in = base + lane < c;
        const int j2 = base + 64 + lane < c ? row[base + 64 + lane] : 0;
        float4 h1, l1;
        if (base + 32 + lane < c) ldg8(pos + 2 * (int64_t)j1, h1, l1);
        bool keep = false;
        float x = 0.f, y = 0.f, z = 0.f;
        if (in) {
            x = (hj.x - hi_i.x) + (lj.x - lo_i.x);
            y = (hj.y - hi_i.y) + (lj.y - lo_i.y);
            z = (hj.z - hi_i.z) + (lj.z - lo_i.z);
            const float d2 = x * x + y * y + z * z;
            keep = d2 < R.rc2;
            if (!(d2 > 1e-16f)) {
                keep = false;
                atomicOr(&flags[FLAG_GEOM], 4);
            }
        }
        const unsigned m = __ballot_sync(FULL, keep);
        if (keep) q[(tail + __popc(m & ((1u << lane) - 1u))) & 63] = make_float4(x, y, z, __int_as_float(j));
        tail += __popc(m);
        j = j1, j1 = j2, hj = h1, lj = l1;
        __syncwarp();
        if (tail - done >= 32) {
            emit();
            done += 32;
            __syncwarp();  // the emitted entries are read before their places are queued again
        }
    }
    if (lane < tail - done) emit();
    if (lane == 0) live_cnt[i] = tail;
}

// ------------------------------------------------------------- forward ---
// LPA lanes per centre atom (32 / LPA atoms per warp), by the atoms of its structure (fwd_lanes), never
// by how many rows a launch has: the lanes decide the order in which a row's edges are summed, and a
// structure's results are the same alone and among others.  Lane q walks the edges
// q, q + LPA, ... of its atom and accumulates the 80 products t_m A_a,
// t_m = c_{j,m} phi_m, in registers; the record two edges ahead and the
// coefficients one edge ahead are in flight meanwhile.  A butterfly
// reduce-scatter over the LPA lanes leaves 80 / LPA of the sums in each lane
// (stored as the b checkpoint), and lane q contracts its 16 / LPA orbitals.
// Bound by the latency of the record stream and the coefficient gathers at 16
// warps per SM (126 registers, 80 of them sums; issue slots 55 % busy).  Reading
// records instead of recomputing the edge's geometry took a launch from 29.7 to
// 19.9 us (24,576 atoms) and from 692 to 541 us (1,048,576 atoms).  Eight lanes per
// edge with the sums of one channel each (48 registers, 37 warps) were slower, 39
// against 21 us for 32,000 atoms: 5 shared-memory wavefronts per edge.
// PAIRS = false: Eq. 1, rho_{l,k} = sum_{a in l} w_a g_{a,k}^2 over 16 orbitals.
// PAIRS = true: the orbital-pair products rho_{l,(k,k')} = sum_{a in l} w_a g_{a,k} g_{a,k'},
// k <= k' over 8 orbitals (108 features).
constexpr int kFwdWarps = 4;
constexpr int kBStride = 84;  // padded b row of an atom in shared memory (16 B aligned)

// one butterfly stage over CNT values: lanes with bit O set keep the upper half
template <int CNT, int O>
__device__ __forceinline__ void rs_half(float* v, int q) {
    const bool upper = q & O;
#pragma unroll
    for (int k = 0; k < CNT / 2; ++k) {
        const float send = upper ? v[k] : v[CNT / 2 + k];
        const float keep = upper ? v[CNT / 2 + k] : v[k];
        v[k] = keep + __shfl_xor_sync(FULL, send, O);
    }
}

// POOL: the rows are a serving pool's (structure: the atoms of each row's structure).
template <bool PAIRS, int LPA, bool POOL>
__global__ void __launch_bounds__(kFwdWarps * 32, 4) k_density_fwd(int64_t row0, int64_t rows, int stride, Radial R,
                                                            const int32_t* __restrict__ live_cnt,
                                                            const float4* __restrict__ xyzj,
                                                            const float2* __restrict__ phi,
                                                            const float* __restrict__ coef,
                                                            const float* __restrict__ Wt, float* __restrict__ rho,
                                                            float* __restrict__ bck, bool far,
                                                            const int32_t* __restrict__ structure) {
    constexpr int KO = PAIRS ? NORB_P : NORB, APW = 32 / LPA;
    static_assert(LPA == 4 || LPA == 8 || LPA == 16, "80 sums split evenly");
    __shared__ __align__(16) float sW[(LMAX + 1) * NPHI * KO];
    __shared__ __align__(16) float sB[kFwdWarps * APW][kBStride];
    for (int i = threadIdx.x; i < (LMAX + 1) * NPHI * KO; i += blockDim.x) sW[i] = Wt[i];
    pdl_enter();  // so far only the weights were read
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane & (LPA - 1), slot = lane / LPA;
    const int64_t kr = ((int64_t)blockIdx.x * kFwdWarps + warp) * APW + slot;
    const int64_t atom = row0 + kr;
    // (of a serving pool's rows only those whose structure takes this many lanes)
    const bool valid = kr < rows && (!POOL || fwd_lanes(structure[atom]) == LPA);
    float acc[NB];
#pragma unroll
    for (int v = 0; v < NB; ++v) acc[v] = 0.f;
    if (valid) {
        const int cnt = live_cnt[atom];
        const float4* ex = xyzj + (size_t)kr * stride;
        const float2* ep = phi + (size_t)kr * stride;
        // the row's records start on their way to L2 at once (large systems stream them from HBM)
        if (far) {
            for (int e = 8 * q; e < cnt; e += 8 * LPA) prefetch_l2(ex + e);
            for (int e = 16 * q; e < cnt; e += 16 * LPA) prefetch_l2(ep + e);
        }
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 e1 = zero, c0 = zero, c1 = zero;
        float2 p1 = make_float2(0.f, 0.f);
        if (q < cnt) {
            e1 = ex[q];
            p1 = ep[q];
            ldg8(coef + (size_t)__float_as_int(e1.w) * NPHI, c0, c1);
        }
        float4 e2 = zero;
        float2 p2 = make_float2(0.f, 0.f);
        if (q + LPA < cnt) e2 = ex[q + LPA], p2 = ep[q + LPA];
        for (int e = q; e < cnt; e += LPA) {
            const float x = e1.x, y = e1.y, z = e1.z;
            float ph[NPHI];
            phi_chain(R, p1.x, p1.y, ph);
            const float t[NPHI] = {c0.x * ph[0], c0.y * ph[1], c0.z * ph[2], c0.w * ph[3],
                                   c1.x * ph[4], c1.y * ph[5], c1.z * ph[6], c1.w * ph[7]};
            e1 = e2;
            p1 = p2;
            if (e + LPA < cnt) ldg8(coef + (size_t)__float_as_int(e2.w) * NPHI, c0, c1);
            if (e + 2 * LPA < cnt) e2 = ex[e + 2 * LPA], p2 = ep[e + 2 * LPA];
            const float A[NANG] = {1.f, x, y, z, x * x, y * y, z * z, x * y, x * z, y * z};
#pragma unroll
            for (int a = 0; a < NANG; ++a)
#pragma unroll
                for (int m = 0; m < NPHI; ++m) acc[a * NPHI + m] = fmaf(t[m], A[a], acc[a * NPHI + m]);
        }
    }
    // reduce-scatter: lane q keeps b[80 / LPA * rev(q) ..), rev the order the halves were taken in
    constexpr int NL = NB / LPA;
    if constexpr (LPA == 16) rs_half<NB, 8>(acc, q);
    if constexpr (LPA >= 8) rs_half<(LPA == 16 ? NB / 2 : NB), 4>(acc, q);
    rs_half<NL * 4, 2>(acc, q);
    rs_half<NL * 2, 1>(acc, q);
    float* sb = sB[warp * APW + slot];
#pragma unroll
    for (int v = 0; v < NL; ++v) acc[v] *= R.unscale;
    if constexpr (LPA == 16) {
#pragma unroll
        for (int v = 0; v < NL; ++v) sb[NL * q + v] = acc[v];
    } else {
#pragma unroll
        for (int v = 0; v < NL; v += 2) *reinterpret_cast<float2*>(sb + NL * q + v) = make_float2(acc[v], acc[v + 1]);
    }
    __syncwarp();
    if (valid)
#pragma unroll
        for (int v = 4 * q; v < NB; v += 4 * LPA) *reinterpret_cast<float4*>(bck + (size_t)atom * NB + v) = ld4(sb + v);
    if constexpr (PAIRS) {
        // g_{a,k} = sum_m b_{a,m} W_{l,m,k} into the b row's place: lane q the orbitals k = q, q + LPA, ...
        constexpr int KL = LPA >= NORB_P ? 1 : NORB_P / LPA;
        float g[NANG][KL];
#pragma unroll
        for (int a = 0; a < NANG; ++a) {
            const int l = ang_l(a);
            const float4 b0 = ld4(sb + a * NPHI), b1 = ld4(sb + a * NPHI + 4);
            const float bm[NPHI] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < KL; ++i) {
                g[a][i] = 0.f;
#pragma unroll
                for (int m = 0; m < NPHI; ++m)
                    g[a][i] = fmaf(bm[m], sW[(l * NPHI + m) * KO + ((q + i * LPA) & (NORB_P - 1))], g[a][i]);
            }
        }
        __syncwarp();
#pragma unroll
        for (int a = 0; a < NANG; ++a)
#pragma unroll
            for (int i = 0; i < KL; ++i)
                if (q + i * LPA < NORB_P) sb[a * NORB_P + q + i * LPA] = g[a][i];
        __syncwarp();
        if (!valid) return;
        constexpr int KP = NORB_P * (NORB_P + 1) / 2;
        for (int f = q; f < NFEAT_P; f += LPA) {
            const int l = f / KP, p = f - l * KP;
            const int k = c_pair_k[p], k2 = c_pair_k2[p];
            const int a0 = l == 0 ? 0 : (l == 1 ? 1 : 4), a1 = l == 0 ? 1 : (l == 1 ? 4 : NANG);
            float acc_f = 0.f;
            for (int a = a0; a < a1; ++a) acc_f = fmaf(ang_w(a) * sb[a * NORB_P + k], sb[a * NORB_P + k2], acc_f);
            rho[(size_t)atom * NFEAT_P + f] = acc_f;
        }
        return;
    }
    if (!valid) return;
    // contraction over m and the squared multinomial sum; lane q owns KL consecutive orbitals
    constexpr int KL = NORB / LPA;
    float racc[LMAX + 1][KL];
#pragma unroll
    for (int l = 0; l <= LMAX; ++l)
#pragma unroll
        for (int k = 0; k < KL; ++k) racc[l][k] = 0.f;
#pragma unroll
    for (int a = 0; a < NANG; ++a) {
        const int l = ang_l(a);
        const float4 b0 = ld4(sb + a * NPHI), b1 = ld4(sb + a * NPHI + 4);
        const float bm[NPHI] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        float g[KL];
#pragma unroll
        for (int k = 0; k < KL; ++k) g[k] = 0.f;
#pragma unroll
        for (int m = 0; m < NPHI; ++m) {
            float w[KL];
            ldk<KL>(sW + (l * NPHI + m) * NORB + KL * q, w);
#pragma unroll
            for (int k = 0; k < KL; ++k) g[k] = fmaf(bm[m], w[k], g[k]);
        }
        const float wa = ang_w(a);
#pragma unroll
        for (int k = 0; k < KL; ++k) racc[l][k] = fmaf(wa * g[k], g[k], racc[l][k]);
    }
#pragma unroll
    for (int l = 0; l <= LMAX; ++l) stk<KL>(rho + (size_t)atom * NFEAT + l * NORB + KL * q, racc[l]);
}

// -------------------------------------------------------------- bbar -----
// bbar_{a,m} = sum_k gbar_{a,k} W_{l(a),m,k}, g recomputed from the b checkpoint, for the orbital-pair
// features (Eq. 1's squares are taken by the backward networks):
//   gbar_{a,k} = w_a sum_k' R_{kk'} g_{a,k'},  R_{kk'} = rhobar_{l,(min,max)} (x 2 on the diagonal)
// written into the atom's adjoint record with the layer's c (values 10, 11 of
// the record).  TPA = 12 threads per atom take a value each, 4 take values q, q + 4, q + 8: a chain
// a third as long against fewer registers.  us per launch with 12 / 4: 192 atoms 6.2 / 8.8, 3,069 8.3 /
// 11.7, 10,976 21.7 / 22.2, 16,200 24.7 / 22.9, 256,000 181 / 130.  The block's
// kBbarAtoms records are staged in shared memory and stored as whole lines.
constexpr int kBbarAtoms = 16;  // small blocks (192 or 64 threads) balance better over the SMs than 64 atoms each
template <int TPA>
__global__ void __launch_bounds__(TPA * kBbarAtoms) k_bbar(int64_t n, const float* __restrict__ Wt,
                                                                const float* __restrict__ bck,
                                                                const float* __restrict__ rhobar,
                                                                const float* __restrict__ coef,
                                                                float* __restrict__ rec, GhostOut gh) {
    constexpr int KO = NORB_P, KP = NORB_P * (NORB_P + 1) / 2;
    __shared__ __align__(16) float sW[(LMAX + 1) * NPHI * KO];
    __shared__ __align__(16) float sRec[kBbarAtoms * kRecLd];
    for (int i = threadIdx.x; i < (LMAX + 1) * NPHI * KO; i += blockDim.x) sW[i] = Wt[i];
    pdl_enter();  // so far only the weights were read
    __syncthreads();
    const int64_t atom0 = (int64_t)blockIdx.x * kBbarAtoms;
    const int r = threadIdx.x / TPA;
    const int64_t atom = atom0 + r;
    const int nrows = n - atom0 < kBbarAtoms ? (int)(n - atom0) : kBbarAtoms;
#pragma unroll 1
    for (int v = threadIdx.x % TPA; v < NREC / NPHI && r < nrows; v += TPA) {
        float out[NPHI];
        if (v >= NANG) {
            rec_tail(coef, atom, v, out);
        } else {
            const int a = v, l = ang_l(a);
            const float4 b0 = ldg4(bck + (size_t)atom * NB + a * NPHI), b1 = ldg4(bck + (size_t)atom * NB + a * NPHI + 4);
            const float* rb = rhobar + (size_t)atom * NFEAT_P + l * KP;
            float pre[KP];  // few atoms: all in flight at once (many: the registers cost more warps)
            if (TPA == 12)
#pragma unroll
                for (int p = 0; p < KP / 4; ++p) {
                    const float4 x = ldg4(rb + 4 * p);
                    pre[4 * p] = x.x, pre[4 * p + 1] = x.y, pre[4 * p + 2] = x.z, pre[4 * p + 3] = x.w;
                }
            const float bm[NPHI] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
            float g[NORB_P], gb[NORB_P];
#pragma unroll
            for (int k = 0; k < NORB_P; ++k) {
                g[k] = 0.f;
                gb[k] = 0.f;
#pragma unroll
                for (int m = 0; m < NPHI; ++m) g[k] = fmaf(bm[m], sW[(l * NPHI + m) * KO + k], g[k]);
            }
            int p = 0;
#pragma unroll
            for (int k = 0; k < NORB_P; ++k)
#pragma unroll
                for (int k2 = k; k2 < NORB_P; ++k2, ++p) {
                    const float rv = TPA == 12 ? pre[p] : __ldg(rb + p);
                    gb[k] = fmaf(rv, g[k2], gb[k]);
                    gb[k2] = fmaf(rv, g[k], gb[k2]);
                }
            const float wa = rec_scale(a) * ang_w(a);
#pragma unroll
            for (int m = 0; m < NPHI; ++m) {
                out[m] = 0.f;
#pragma unroll
                for (int k = 0; k < NORB_P; ++k) out[m] = fmaf(wa * gb[k], sW[(l * NPHI + m) * KO + k], out[m]);
            }
        }
        stage_rec(sRec, r, v, out);
    }
    __syncthreads();
    flush_rec(sRec, nrows, atom0, rec, gh, threadIdx.x, blockDim.x);
}

// ---------------------------------------------------------- adjoint ------

// Reverse pass (header formulas), LPA lanes per centre atom k (32 / LPA atoms per
// warp), lane (g, m) owning radial channel m of every (LPA / 8)th edge, g the lane's group of 8.  Per
// batch of LPA edges each lane expands one edge's record into shared memory (the
// next batch's record is on its way meanwhile).  Then, for its edges, lane (g, m)
// gathers channel m of the neighbour's adjoint record (3 float4 loads; per load the
// 8 lanes of a group read one full 128 B line) and accumulates its share of
// dE/dr_k and of cbar_{k,m}.
//   The shares are summed by NC LPA / 8 classes of edges, e mod (NC LPA / 8), edge after edge,
// and the classes' sums added as (0 + 2) + (1 + 3).  How many classes is decided by the
// atoms of the structure (adj_classes), never by how many rows a launch has, so that a structure's results
// are the same alone and among others; a group keeps the sums of NC classes: four as (LPA, NC)
// = (32, 1) or, in launches of many rows, (16, 2); two as (16, 1); one as (8, 1).
//   Bound by the L2 latency and the L1 wavefronts of the record gathers (384 B per
// edge; the L1 data stage is 70 % busy while blocks are resident, issue slots 56 %).
// 59 -> 41 us per launch (24,576 atoms), 1,408 -> 1,166 us (1,048,576 atoms), 28 -> 7 us
// (192 atoms, where the number of edges that follow one another decides).  Records
// gathered one edge ahead in a second register set gained nothing.
//   With Q_k(r) = sum_a bbar_{k,a} A_a and Q_j(r) = sum_a (-1)^l bbar_{j,a} A_a (both
// quadratics per channel) the edge's share of -dE/dr_k is, per channel,
//   c_j (psi Q_k r + phi grad Q_k) + c_k (psi Q_j r + phi grad Q_j).
// Summed over the edges, the term c_j phi grad Q_k needs only the moments sum_j
// c_j phi A_a = b_{k,a} that the forward pass kept (grad Q_k is linear in r), so
// it is added once per atom from the checkpoint b instead of once per edge.
// Preferred shared memory of the reverse pass: 75 % holds the blocks its registers allow;
// the driver's choice was 2 % slower (1,048,576 atoms 1,160 -> 1,138 us, 24,576 40.8 -> 39.8),
// 25 % and 100 % 14 to 38 %.
constexpr int kAdjCarveout = 75;
// Small blocks: the block scheduler balances the SMs at fine grain.
constexpr int kAdjWarps = 4;
// With forces set (the last reverse layer), the kernel also writes F = -dE/dr
// and the atomic energies in caller order (perm: internal -> caller index);
// with first set (the first reverse layer), grad and vir are written, not
// accumulated.
struct Outputs {
    const int32_t* perm;
    const float* eps;
    float* forces;
    float* atom_energy;
    bool first;
};

// 8 values of a lane's edge to shared memory at f = base + 8 lane; lanes 4-7 of every 8 store the halves the
// other way round: no bank conflicts
__device__ __forceinline__ void store8(float* f, const float v[NPHI], int lane) {
    const bool sw = lane & 4;
    const int h0 = sw ? 4 : 0, h1 = 4 - h0;
    *reinterpret_cast<float4*>(f + h0) = make_float4(sw ? v[4] : v[0], sw ? v[5] : v[1], sw ? v[6] : v[2], sw ? v[7] : v[3]);
    *reinterpret_cast<float4*>(f + h1) = make_float4(sw ? v[0] : v[4], sw ? v[1] : v[5], sw ? v[2] : v[6], sw ? v[3] : v[7]);
}

// WANT_VIR: also W -= (dE/dr_e) r_e^T over the atom's own edges (their
// bbar_k c_j terms: every directed edge once) into vir (N x 9, accumulated
// over the layers like grad); the part with grad Q_k again comes from b.
// POOL: the rows are a serving pool's (structure: the atoms of each row's structure).
// Seven blocks per SM with the virial: 32,000 atoms 50 us a launch, 56 with eight (64 registers).
template <bool WANT_CBAR, bool WANT_VIR, int LPA, int NC, bool POOL>
__global__ void __launch_bounds__(kAdjWarps * 32, LPA == 32 || WANT_VIR ? 7 : 8) k_density_adj(int64_t row0, int64_t rows, int stride, Radial R,
                                                                const int32_t* __restrict__ live_cnt,
                                                                const float4* __restrict__ xyzj,
                                                                const float2* __restrict__ phi,
                                                                const float2* __restrict__ der,
                                                                const float* __restrict__ rec,
                                                                const float* __restrict__ bck,
                                                                float* __restrict__ cbar, float* __restrict__ grad,
                                                                float* __restrict__ vir,
                                                                const int32_t* __restrict__ structure, Outputs out) {
    pdl_enter();
    constexpr int APW = 32 / LPA, G = LPA / 8;  // atoms per warp, groups of 8 lanes per atom
    // Per atom, for its batch of LPA edges: (r, j) [LPA][4], phi [LPA][8] and phi' / d [LPA][8], or, with 32 lanes,
    // (r, d) [LPA][4], phi [LPA][8] and (j, f_c' / f_c, 1/d) [LPA][4], so that seven blocks fit beside the carveout of
    // small systems (4,000 atoms: 16.9 us a launch instead of 20.0; with 16 and 8 lanes the first form takes 41.0
    // instead of 44.4 for 24,576 atoms, 1,162 instead of 1,406 for 1,048,576).  An
    // atom's blocks are padded so that the words its groups and the other atoms of the warp read
    // together lie in different banks.
    constexpr bool kPsi = LPA < 32;
    constexpr int PAD = LPA == 32 ? 0 : (LPA == 16 ? 16 : 8), LE = 4 * LPA + PAD, LP = 8 * LPA + PAD;
    __shared__ __align__(16) float sE[kAdjWarps * APW][kPsi ? LE + 2 * LP : 2 * LE + LP];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, m = lane & 7, sub = lane & (LPA - 1), g = sub >> 3;
    const int64_t kr = ((int64_t)blockIdx.x * kAdjWarps + warp) * APW + lane / LPA;
    const int64_t atom = row0 + kr;
    // (of a serving pool's rows only those whose structure takes this many classes)
    const bool valid = kr < rows && (!POOL || adj_classes(structure[atom]) == NC * G);
    float* s_e = sE[warp * APW + lane / LPA];
    float *s_phi = s_e + LE, *s_psi = s_phi + LP, *s_j = s_phi + LP;
    const float m_two_a = -2.f * R.alpha_hi, mu_hi = R.mu_hi[m], mu_lo = R.mu_lo[m];
    // the 12 values of channel m in an atom's record: bbar_{0..9,m} (the squares' doubled), c_m, 0
    auto load_rec = [&](int r, float* v) {
        const float* p = rec + (size_t)r * NREC + 4 * m;
        if constexpr (LPA < 32) {
            asm volatile(
                "ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%12];\n\t"
                "ld.global.nc.v4.f32 {%4, %5, %6, %7}, [%12 + 128];\n\t"
                "ld.global.nc.v4.f32 {%8, %9, %10, %11}, [%12 + 256];"
                : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                  "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11])
                : "l"(p)
                : "memory");
        } else {
#pragma unroll
            for (int line = 0; line < 3; ++line) {
                const float4 x = ldg4(p + line * 4 * NPHI);
                v[4 * line] = x.x, v[4 * line + 1] = x.y, v[4 * line + 2] = x.z, v[4 * line + 3] = x.w;
            }
        }
    };
    int cnt = 0;
    float bk[12];
#pragma unroll
    for (int v = 0; v < 12; ++v) bk[v] = 0.f;
    if (valid) {
        cnt = live_cnt[atom];
        load_rec((int)atom, bk);
    }
    int cmax = cnt;  // longest row of the warp's atoms
#pragma unroll
    for (int o = LPA; o < 32; o <<= 1) cmax = max(cmax, __shfl_xor_sync(FULL, cmax, o));
    const float ck = bk[NANG];
    bk[4] *= 0.5f, bk[5] *= 0.5f, bk[6] *= 0.5f;
    const float4* ex = xyzj + (size_t)kr * stride;
    const float2* ep = phi + (size_t)kr * stride;
    const float2* ed = der + (size_t)kr * stride;
    float gx[NC], gy[NC], gz[NC], cb[NC];
    float w6[NC][6];  // sum c_j psi Q_k r r^T: xx, yy, zz, xy, xz, yz
#pragma unroll
    for (int i = 0; i < NC; ++i) {
        gx[i] = gy[i] = gz[i] = cb[i] = 0.f;
#pragma unroll
        for (int q = 0; q < 6; ++q) w6[i][q] = 0.f;
    }
    float w9[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) w9[q] = 0.f;
    float4 e_nx = make_float4(0.f, 0.f, 0.f, 0.f);  // the next batch's record of this lane
    float2 p_nx = make_float2(0.f, 0.f), d_nx = p_nx;
    if (sub < cnt) e_nx = ex[sub], p_nx = ep[sub], d_nx = ed[sub];
    // one edge's shares: vx, vy, vz of -dE/dr_k, phi and Q_j (cbar += phi Q_j), a = c_j psi Q_k (virial)
    struct Share {
        float vx, vy, vz, ph, Qj, a;
        float4 e;
    };
    auto share = [&](int s) {
        const float4 e = ld4(s_e + 4 * s);
        float bj[12];
        float ph, ps;
        if constexpr (kPsi) {
            load_rec(__float_as_int(e.w), bj);
            ph = s_phi[8 * s + m], ps = s_psi[8 * s + m];  // phi, phi' / d
        } else {
            const float4 r = ld4(s_j + 4 * s);  // j, f_c' / f_c, 1 / d
            load_rec(__float_as_int(r.x), bj);
            ph = s_phi[8 * s + m];
            ps = ph * (fmaf(m_two_a, (e.w - mu_hi) - mu_lo, r.y) * r.z);
        }
        const float x = e.x, y = e.y, z = e.z, cj = bj[NANG];
        // grad Q_j; Q_j = q0 + (r . (l + grad Q_j)) / 2 for a quadratic with linear part l
        const float gjx = fmaf(z, bj[8], fmaf(y, bj[7], fmaf(x, bj[4], -bj[1])));
        const float gjy = fmaf(z, bj[9], fmaf(x, bj[7], fmaf(y, bj[5], -bj[2])));
        const float gjz = fmaf(y, bj[9], fmaf(x, bj[8], fmaf(z, bj[6], -bj[3])));
        const float Qj = fmaf(0.5f, fmaf(z, gjz - bj[3], fmaf(y, gjy - bj[2], x * (gjx - bj[1]))), bj[0]);
        // Q_k by Horner's rule (bk's squares halved below)
        const float Qk = fmaf(x, fmaf(z, bk[8], fmaf(y, bk[7], fmaf(x, bk[4], bk[1]))),
                              fmaf(y, fmaf(z, bk[9], fmaf(y, bk[5], bk[2])), fmaf(z, fmaf(z, bk[6], bk[3]), bk[0])));
        const float sk = cj * Qk;
        const float sc = ps * fmaf(ck, Qj, sk);
        const float qt = ck * ph;
        return Share{fmaf(sc, x, qt * gjx), fmaf(sc, y, qt * gjy), fmaf(sc, z, qt * gjz), ph, Qj, ps * sk, e};
    };
    auto add_w6 = [](float* w, float a, const float4& e) {
        const float ax = a * e.x, ay = a * e.y, az = a * e.z;
        w[0] = fmaf(ax, e.x, w[0]);
        w[1] = fmaf(ay, e.y, w[1]);
        w[2] = fmaf(az, e.z, w[2]);
        w[3] = fmaf(ax, e.y, w[3]);
        w[4] = fmaf(ax, e.z, w[4]);
        w[5] = fmaf(ay, e.z, w[5]);
    };
    auto add = [&](int i, const Share& v) {  // to class i's sums
        gx[i] -= v.vx;
        gy[i] -= v.vy;
        gz[i] -= v.vz;
        if (WANT_CBAR) cb[i] = fmaf(v.ph, v.Qj, cb[i]);
        if (WANT_VIR) add_w6(w6[i], v.a, v.e);
    };
    for (int e0 = 0; e0 < cmax; e0 += LPA) {
        const int ne = min(cnt - e0, LPA);
        if (sub < ne) {
            float ph[NPHI];
            phi_chain(R, p_nx.x, p_nx.y, ph);
            const float d = d_nx.x, inv_d = __frcp_rn(d);
            *reinterpret_cast<float4*>(s_e + 4 * sub) = make_float4(e_nx.x, e_nx.y, e_nx.z, kPsi ? e_nx.w : d);
            store8(s_phi + 8 * sub, ph, sub);
            // phi_m' / d = phi_m (f_c' / f_c - 2 a (d - mu_m)) / d with mu_m a float pair: phi_m is largest where the
            // difference is small (as 2 a mu_m / d - 2 a, rounded term by term, it had up to six times the error)
            if constexpr (kPsi) {
#pragma unroll
                for (int k = 0; k < NPHI; ++k) ph[k] *= fmaf(m_two_a, (d - R.mu_hi[k]) - R.mu_lo[k], d_nx.y) * inv_d;
                store8(s_psi + 8 * sub, ph, sub);
            } else {
                *reinterpret_cast<float4*>(s_j + 4 * sub) = make_float4(e_nx.w, d_nx.y, inv_d, 0.f);
            }
            if (e0 + LPA + sub < cnt) e_nx = ex[e0 + LPA + sub], p_nx = ep[e0 + LPA + sub], d_nx = ed[e0 + LPA + sub];
        }
        __syncwarp();
        // the group's classes, one after the other
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll 1
            for (int s = g + G * i; s < ne; s += G * NC) add(i, share(s));
        __syncwarp();
    }
    // the row's sums, in every group
    auto total = [](const float* p) {
        float v = NC == 2 ? p[0] + p[NC - 1] : p[0];
        if (LPA == 32) v += __shfl_xor_sync(FULL, v, 16);
        if (LPA >= 16) v += __shfl_xor_sync(FULL, v, 8);
        return v;
    };
    gx[0] = total(gx), gy[0] = total(gy), gz[0] = total(gz), cb[0] = total(cb);
    if (WANT_VIR)
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            float p[NC];
#pragma unroll
            for (int i = 0; i < NC; ++i) p[i] = w6[i][q];
            w6[0][q] = total(p);
        }
    float sx = gx[0] * R.unscale, sy = gy[0] * R.unscale, sz = gz[0] * R.unscale;
    if (WANT_CBAR && g == 0 && valid) cbar[(size_t)atom * NPHI + m] = cb[0] * R.unscale;
    if (WANT_VIR)
#pragma unroll
        for (int q = 0; q < 6; ++q) w6[0][q] *= R.unscale;
    if (g == 0 && valid) {
        // sum_j c_j phi grad Q_k (and, for the virial, times r) from the forward's moments b_{k,a,m}
        const float* b = bck + (size_t)atom * NB + m;
        const float h4 = 2.f * bk[4], h5 = 2.f * bk[5], h6 = 2.f * bk[6];
        const float b0 = __ldg(b), b1 = __ldg(b + NPHI), b2 = __ldg(b + 2 * NPHI), b3 = __ldg(b + 3 * NPHI);
        sx -= fmaf(bk[1], b0, fmaf(h4, b1, fmaf(bk[7], b2, bk[8] * b3)));
        sy -= fmaf(bk[2], b0, fmaf(bk[7], b1, fmaf(h5, b2, bk[9] * b3)));
        sz -= fmaf(bk[3], b0, fmaf(bk[8], b1, fmaf(bk[9], b2, h6 * b3)));
        if (WANT_VIR) {
            const float b4 = __ldg(b + 4 * NPHI), b5 = __ldg(b + 5 * NPHI), b6 = __ldg(b + 6 * NPHI);
            const float b7 = __ldg(b + 7 * NPHI), b8 = __ldg(b + 8 * NPHI), b9 = __ldg(b + 9 * NPHI);
            w9[0] = fmaf(bk[1], b1, fmaf(h4, b4, fmaf(bk[7], b7, bk[8] * b8)));
            w9[1] = fmaf(bk[1], b2, fmaf(h4, b7, fmaf(bk[7], b5, bk[8] * b9)));
            w9[2] = fmaf(bk[1], b3, fmaf(h4, b8, fmaf(bk[7], b9, bk[8] * b6)));
            w9[3] = fmaf(bk[2], b1, fmaf(bk[7], b4, fmaf(h5, b7, bk[9] * b8)));
            w9[4] = fmaf(bk[2], b2, fmaf(bk[7], b7, fmaf(h5, b5, bk[9] * b9)));
            w9[5] = fmaf(bk[2], b3, fmaf(bk[7], b8, fmaf(h5, b9, bk[9] * b6)));
            w9[6] = fmaf(bk[3], b1, fmaf(bk[8], b4, fmaf(bk[9], b7, h6 * b8)));
            w9[7] = fmaf(bk[3], b2, fmaf(bk[8], b7, fmaf(bk[9], b5, h6 * b9)));
            w9[8] = fmaf(bk[3], b3, fmaf(bk[8], b8, fmaf(bk[9], b9, h6 * b6)));
        }
    }
#pragma unroll
    for (int o = 1; o < NPHI; o <<= 1) {
        sx += __shfl_xor_sync(FULL, sx, o);
        sy += __shfl_xor_sync(FULL, sy, o);
        sz += __shfl_xor_sync(FULL, sz, o);
    }
    if (WANT_VIR) {
        const float* w = w6[0];
        w9[0] += w[0], w9[4] += w[1], w9[8] += w[2];
        w9[1] += w[3], w9[3] += w[3], w9[2] += w[4], w9[6] += w[4], w9[5] += w[5], w9[7] += w[5];
#pragma unroll
        for (int o = 1; o < NPHI; o <<= 1)
#pragma unroll
            for (int q = 0; q < 9; ++q) w9[q] += __shfl_xor_sync(FULL, w9[q], o);
    }
    if (sub == 0 && valid) {
        float* gr = grad + (size_t)atom * 3;
        if (!out.first) {  // the first reverse layer starts the sums (no memset)
            sx += gr[0];
            sy += gr[1];
            sz += gr[2];
        }
        if (out.forces) {  // the last layer: F = -dE/dr and eps_i in caller order
            const int64_t c = out.perm[atom];
            out.forces[3 * c] = -sx;
            out.forces[3 * c + 1] = -sy;
            out.forces[3 * c + 2] = -sz;
            if (out.atom_energy) out.atom_energy[c] = out.eps[atom];
        } else {
            gr[0] = sx;
            gr[1] = sy;
            gr[2] = sz;
        }
        if (WANT_VIR) {
            float* vr = vir + (size_t)atom * 9;
#pragma unroll
            for (int q = 0; q < 9; ++q) vr[q] = out.first ? -w9[q] : vr[q] - w9[q];
        }
    }
}

// ------------------------------------------------------- small kernels ---
__device__ __forceinline__ int64_t ghosts_in_use(const int32_t* g_count, int64_t g_cap) {
    const int64_t g = *g_count;
    return g < g_cap ? g : g_cap;
}

// first-layer coefficients c0 of owned rows [0, n_rows) and ghost slots n + [0, g_rows)
__global__ void k_init_coef(int64_t n, int64_t n_rows, int64_t g_rows, const int32_t* __restrict__ g_count,
                            int64_t g_cap, const int32_t* __restrict__ species, const int32_t* __restrict__ owner,
                            const float* __restrict__ c0, float* __restrict__ coef) {
    pdl_enter();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int64_t s, o;
    if (t < n_rows) {
        s = o = t;
    } else {
        const int64_t gi = t - n_rows;
        if (gi >= g_rows || gi >= ghosts_in_use(g_count, g_cap)) return;
        s = n + gi;
        o = owner[gi];
    }
    const int e = species[o];
    const float4* src = reinterpret_cast<const float4*>(c0 + e * NPHI);
    float4* dst = reinterpret_cast<float4*>(coef + (size_t)s * NPHI);
    dst[0] = src[0];
    dst[1] = src[1];
}

// ghost rows <- owner rows (the per-layer ghost refresh of Fig. 4a), width in floats, multiple of 4
__global__ void k_gather_rows(int64_t n, const int32_t* __restrict__ g_count, int64_t g_cap, int w4,
                              const int32_t* __restrict__ owner, float* __restrict__ base) {
    pdl_enter();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ghosts_in_use(g_count, g_cap) * w4) return;
    const int64_t gi = t / w4;
    const int c = (int)(t - gi * w4);
    float4* b = reinterpret_cast<float4*>(base);
    b[(n + gi) * w4 + c] = b[(int64_t)owner[gi] * w4 + c];
}

constexpr int kSumThreads = 256;

// Total energy from the np tile sums of the energy network, in a fixed order.  It is launched after the
// last reverse pass and runs beside it: when it starts, every block of the preceding kernel has passed
// its own griddepcontrol.wait, so the energy network, several kernels back, has completed (the sums are
// read from L2).  Waiting only before it exits keeps completion transitive.  Between the energy
// network and the reverse passes, where it waited for the one and held up the other, it
// cost an evaluation 1.7 us (192 atoms 71.8 -> 70.1 us; 20 trajectory steps of 1,536 atoms 1,985 -> 1,947).
__global__ void __launch_bounds__(kSumThreads) k_energy_final(int np, const double* __restrict__ partial,
                                                             double* __restrict__ energy) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ double sm[kSumThreads];
    double s = 0.0;
    for (int i = threadIdx.x; i < np; i += kSumThreads) s += __ldcg(partial + i);
    sm[threadIdx.x] = s;
    __syncthreads();
    for (int o = kSumThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) energy[0] = sm[0];
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// FP64 sum of the per-atom virials (N x 9): partial sums per kVirRows atoms, then one block.
// Thread t of a block walks the rows' values 288 apart, always the same component t % 9, so the
// loads are whole lines and one barrier does; with atom_virial the values go out in caller order on
// the way.  Bound by latency.  32,000 atoms, evaluation with both outputs: 450 -> 418 us against a
// pass over strided rows per component, with 8 barriers each, and a third launch for the output.
constexpr int kVirThreads = 288, kVirRows = 256;
__global__ void __launch_bounds__(kVirThreads) k_virial_partial(int64_t n, const float* __restrict__ vir,
                                                               double* __restrict__ partial,
                                                               const int32_t* __restrict__ perm,
                                                               float* __restrict__ atom_virial) {
    pdl_enter();
    __shared__ double sm[kVirThreads];
    const int t = threadIdx.x, c = t % 9, lane = t & 31, w = t >> 5;
    const int64_t row0 = (int64_t)blockIdx.x * kVirRows + t / 9;
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kVirRows / 32; ++k) {
        const int64_t i = row0 + 32 * k;
        if (i < n) {
            const float v = vir[9 * i + c];
            s += (double)v;
            if (atom_virial) atom_virial[9 * (int64_t)perm[i] + c] = v;
        }
    }
    sm[t] = s;
    __syncthreads();
    s = sm[9 * lane + w];  // warp w: component w of the 32 row classes
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) partial[(int64_t)w * gridDim.x + blockIdx.x] = s;
}

// warp w: component w
__global__ void __launch_bounds__(kVirThreads) k_virial_final(int np, const double* __restrict__ partial,
                                                             double* __restrict__ out) {
    pdl_enter();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double* p = partial + (int64_t)w * np;
    double s = 0.0;
#pragma unroll 4
    for (int i = lane; i < np; i += 32) s += p[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[w] = s;
}

__global__ void k_unpermute_rows(int64_t n, int width, const int32_t* __restrict__ perm, const float* __restrict__ src,
                                 int src_stride, float* __restrict__ dst) {
    pdl_enter();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * width) return;
    const int64_t i = t / width;
    const int c = (int)(t - i * width);
    dst[(int64_t)perm[i] * width + c] = src[i * src_stride + c];
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_init_coef(cudaStream_t s, const reann_nlist* nl, const float* c0) {
    const int64_t nr = rows_of(nl), gr = ghost_rows_of(nl);
    if (nr + gr == 0) return cudaSuccess;
    launch_with(true, eval_launch(nl).carve(), k_init_coef, blocks_for(nr + gr, 256), 256, 0, s, nl->n, nr, gr, ghost_count_ptr(nl), nl->g_cap,
               nl->species, nl->g_owner, c0, nl->coef);
    return cudaGetLastError();
}

cudaError_t launch_gather_ghost_rows(cudaStream_t s, const reann_nlist* nl, float* base, int width) {
    const int64_t gr = ghost_rows_of(nl);
    if (gr == 0) return cudaSuccess;
    const int w4 = width / 4;
    launch_with(true, eval_launch(nl).carve(), k_gather_rows, blocks_for(gr * w4, 256), 256, 0, s, nl->n, ghost_count_ptr(nl), gr, w4, nl->g_owner,
               base);
    return cudaGetLastError();
}

cudaError_t launch_edges(cudaStream_t s, const reann_nlist* nl, const Radial& r, int64_t row0, int64_t rows,
                         int* flags) {
    if (rows == 0) return cudaSuccess;
    launch_with(true, eval_launch(nl).carve(), k_edges, blocks_for(rows, kEdgeWarps), kEdgeWarps * 32, 0, s, row0, rows, nl->stride, r, nl->nbr,
               nl->nbr_cnt, nl->pos, nl->edge_xyzj, nl->edge_phi, nl->edge_der, nl->live_cnt, flags);
    return cudaGetLastError();
}

cudaError_t launch_density_fwd(cudaStream_t s, const reann_nlist* nl, const Radial& r, int64_t row0, int64_t rows,
                               const float* W, const float* coef, float* rho, float* bck, bool pairs) {
    if (rows == 0) return cudaSuccess;
    // Lanes per atom: more lanes shorten an atom's chain of edges (few atoms: latency), fewer need
    // less reduction work per atom (many).  us per launch with 16 / 8 / 4 lanes: 192 atoms 4.5 / 5.6 /
    // 7.9, 4,000 5.5 / 5.8 / 7.1, 10,976 11.8 / 10.8 / 9.1, 24,576 25 / 20 / 20, 1,048,576 914 / 670 / 536.
    const EvalLaunch how = eval_launch(nl);
    // records of more rows than this outgrow L2 between the passes: prefetch each atom's when it
    // starts (1,048,576 atoms: 580 -> 541 us; 24,576 atoms: 19.9 -> 20.2 us, so not there)
    const bool far = rows > (int64_t)1 << 16;
#define REANN_FWD(P, L, POOL)                                                                                        \
    launch_with(how.chain, how.carve(), k_density_fwd<P, L, POOL>, blocks_for(rows, kFwdWarps * (32 / L)), kFwdWarps * 32, 0, s, \
                row0, rows, nl->stride, r, nl->live_cnt, nl->edge_xyzj, nl->edge_phi, coef, W, rho, bck, far, nl->structure)
#define REANN_FWD_P(L)                      \
    do {                                    \
        if (pairs && nl->structure)         \
            REANN_FWD(true, L, true);       \
        else if (pairs)                     \
            REANN_FWD(true, L, false);      \
        else if (nl->structure)             \
            REANN_FWD(false, L, true);      \
        else                                \
            REANN_FWD(false, L, false);     \
    } while (0)
    // a serving pool's rows belong to structures of their own: a launch for each number of lanes they take
    const int lanes = nl->structure ? nl->fwd_passes : fwd_lanes(nl->n);
    if (lanes & 16) REANN_FWD_P(16);
    if (lanes & 8) REANN_FWD_P(8);
    if (lanes & 4) REANN_FWD_P(4);
#undef REANN_FWD_P
#undef REANN_FWD
    return cudaGetLastError();
}

cudaError_t launch_bbar(cudaStream_t s, const reann_nlist* nl, const float* W, const float* bck, const float* rhobar,
                        const float* coef, float* rec, GhostOut gh) {
    const int64_t nr = rows_of(nl);
    if (nr == 0) return cudaSuccess;
    const int tpa = nr <= kChainRows ? 12 : 4;
    launch_with(true, eval_launch(nl).carve(), tpa == 12 ? k_bbar<12> : k_bbar<4>, blocks_for(nr, kBbarAtoms), tpa * kBbarAtoms, 0,
                s, nr, W, bck, rhobar, coef, rec, gh);
    return cudaGetLastError();
}

cudaError_t upload_pair_table() {
    unsigned char k1[NORB_P * (NORB_P + 1) / 2], k2[NORB_P * (NORB_P + 1) / 2];
    int p = 0;
    for (int a = 0; a < NORB_P; ++a)
        for (int b = a; b < NORB_P; ++b, ++p) {
            k1[p] = (unsigned char)a;
            k2[p] = (unsigned char)b;
        }
    cudaError_t e = cudaMemcpyToSymbol(c_pair_k, k1, sizeof(k1));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_pair_k2, k2, sizeof(k2));
    return e;
}

cudaError_t launch_density_adj(cudaStream_t s, const reann_nlist* nl, const Radial& r, int64_t row0, int64_t rows,
                               const float* rec, const float* bck, float* cbar, float* grad, bool want_cbar,
                               float* vir, float* forces, float* atom_energy, bool first) {
    const Outputs out{forces ? nl->perm : nullptr, forces ? nl->eps : nullptr, forces, atom_energy, first};
    if (rows == 0) return cudaSuccess;
    // Lanes per atom, as in the forward pass.  us per launch with 32 / 16 / 8 lanes: 192 atoms 7.2 /
    // 10.6 / 18.3, 4,000 8.6 / 11.1 / 16.1, 24,576 43.5 / 41.1 / 49, 32,000 53 / 47.0 / 45.6,
    // 1,048,576 1,644 / 1,242 / 1,161.  The sums' classes follow: four with 32 lanes, two with 16, one with 8.
    const EvalLaunch how = eval_launch(nl);
#define REANN_ADJ_L(C, V, L, N, P)                                                                                    \
    launch_with(how.chain, how.carve(kAdjCarveout), k_density_adj<C, V, L, N, P>, blocks_for(rows, kAdjWarps * (32 / L)), \
                kAdjWarps * 32, 0, s, row0, rows, nl->stride, r, nl->live_cnt, nl->edge_xyzj, nl->edge_phi, nl->edge_der, rec, bck, cbar, grad, vir, nl->structure, out)
#define REANN_ADJ(C, V)                  \
    do {                                 \
        if (classes == 4)                \
            REANN_ADJ_L(C, V, 32, 1, false); \
        else if (classes == 2)           \
            REANN_ADJ_L(C, V, 16, 1, false); \
        else                             \
            REANN_ADJ_L(C, V, 8, 1, false);  \
    } while (0)
    if (!nl->structure) {
        const int classes = adj_classes(nl->n);
        if (want_cbar && vir)
            REANN_ADJ(true, true);
        else if (want_cbar)
            REANN_ADJ(true, false);
        else if (vir)
            REANN_ADJ(false, true);
        else
            REANN_ADJ(false, false);
    }
#undef REANN_ADJ
#define REANN_ADJ(L, N)                            \
    do {                                           \
        if (want_cbar)                             \
            REANN_ADJ_L(true, false, L, N, true);  \
        else                                       \
            REANN_ADJ_L(false, false, L, N, true); \
    } while (0)
    // A serving pool's rows belong to structures of their own: a launch for each number of classes that
    // the evaluated structures take.  Many rows of four classes go with 16 lanes (24,576 rows: 41.8 us, with 32 51).
    if (nl->structure) {
        if (nl->adj_passes & 4) {
            if (rows_of(nl) <= 16384)
                REANN_ADJ(32, 1);
            else
                REANN_ADJ(16, 2);
        }
        if (nl->adj_passes & 2) REANN_ADJ(16, 1);
        if (nl->adj_passes & 1) REANN_ADJ(8, 1);
    }
#undef REANN_ADJ
#undef REANN_ADJ_L
    return cudaGetLastError();
}

int64_t virial_partials(int64_t n) { return 9 * (int64_t)std::max(1u, blocks_for(n, kVirRows)); }

cudaError_t launch_virial_sum(cudaStream_t s, const reann_nlist* nl, const float* vir, double* partial, double* out,
                              float* atom_virial) {
    const int np = (int)blocks_for(nl->n, kVirRows);
    launch_pdl(k_virial_partial, np, kVirThreads, 0, s, nl->n, vir, partial, nl->perm, atom_virial);
    launch_pdl(k_virial_final, 1, kVirThreads, 0, s, np, partial, out);
    return cudaGetLastError();
}

cudaError_t launch_energy_final(cudaStream_t s, const double* partial, int np, double* energy, int carve) {
    launch_with(true, carve, k_energy_final, 1, kSumThreads, 0, s, np, partial, energy);
    return cudaGetLastError();
}

cudaError_t launch_unpermute_rows(cudaStream_t s, const reann_nlist* nl, const float* src, int src_stride, float* dst,
                                  int width) {
    launch_pdl(k_unpermute_rows, blocks_for(nl->n * width, 256), 256, 0, s, nl->n, width, nl->perm, src, src_stride,
               dst);
    return cudaGetLastError();
}

}  // namespace reann
