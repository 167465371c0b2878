// Velocity-Verlet integration in FP64 around the REANN force evaluation, NVE
// or NVT with one Nose-Hoover thermostat.
//
// One MD step (captured once as a CUDA graph and replayed):
//   [NVT: thermostat half step, v *= s]
//   v += (dt/2) F/m;  x += dt v;  rebuild the neighbour list if any atom moved
//   more than skin/2 since the last build (gated kernels, no host round trip);
//   E, F = REANN(x);  v += (dt/2) F/m;  K = sum m v^2 / 2 (FP64);
//   [NVT: thermostat half step, v *= s];  record E, K (and the bath energy).
// Thermostat half step of length dt/2 (time-reversible Trotter splitting of
// the Nose-Hoover equations xi' = (2K - g kT)/Q, eta' = xi, v' = -xi v):
//   xi += (dt/4) G(K);  eta += (dt/2) xi;  s = exp(-(dt/2) xi);  K *= s^2;
//   xi += (dt/4) G(K),  with G(K) = (2K - g kT)/Q, Q = g kT tau^2, g = 3N - 3.
// The conserved quantity is E + K + Q xi^2 / 2 + g kT eta.
// The integration around the rebuild and the forces is two kernels (a small system's
// step is a chain of launches of about 2 us each): k_first_half also makes the
// skin/2 test, k_second_half also sums K, takes the thermostat's half step and
// records (NVT scales the velocities afterwards).  The recording kernel finds the
// call's output arrays in device memory (MdOut, written once per call), so the
// captured step serves calls with other output arrays and step counts.
// Units: A, fs, amu, eV; 1 eV/(A amu) = 9.648533212e-3 A/fs^2.
#include <cuda_runtime.h>

#include "common.cuh"

namespace reann {
namespace {

constexpr double kAccel = 9.648533212e-3;  // (eV/A)/amu -> A/fs^2
constexpr int kThreads = 256, kPer = 8;

// once per call: the output arrays, and the step counter and rebuild gate at zero
__global__ void k_md_begin(MdOut* __restrict__ dst, MdOut out, int* __restrict__ ints) {
    pdl_enter();
    *dst = out;
    ints[0] = ints[1] = 0;
}

// v = s v + (dt/2) F/m (s read from the device; 1 without a thermostat), x += dt v, and
// the gate of the rebuild: set when the atom is more than skin/2 from where it was at
// the last build
__global__ void __launch_bounds__(64) k_first_half(int64_t n, double* __restrict__ pos, double* __restrict__ vel,
                                                   const float* __restrict__ forces, const double* __restrict__ mass,
                                                   double half_dt, double dt, const double* __restrict__ scale,
                                                   const double* __restrict__ ref, double thr2, int* __restrict__ gate) {
    pdl_enter();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double m = mass[i];
    double d2 = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int64_t t = 3 * i + k;
        const double v0 = scale ? vel[t] * *scale : vel[t];
        const double v = v0 + half_dt * kAccel * (double)forces[t] / m;
        const double x = pos[t] + dt * v;
        vel[t] = v;
        pos[t] = x;
        const double d = x - ref[t];
        d2 += d * d;
    }
    if (!(d2 <= thr2)) atomicOr(gate, 1);
}

__global__ void k_scale(int64_t n, double* __restrict__ vel, const double* __restrict__ scale) {
    pdl_enter();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 3 * n) vel[t] *= *scale;
}

// thermostat half step on the device scalars: sc[1] K, sc[2] xi, sc[3] eta, sc[4] s
__device__ __forceinline__ void nh_half(double* sc, double dt, double gkt, double q) {
    double K = sc[1], xi = sc[2], eta = sc[3];
    xi += 0.25 * dt * (2.0 * K - gkt) / q;
    eta += 0.5 * dt * xi;
    const double s = exp(-0.5 * dt * xi);
    K *= s * s;
    xi += 0.25 * dt * (2.0 * K - gkt) / q;
    sc[1] = K;
    sc[2] = xi;
    sc[3] = eta;
    sc[4] = s;
}

__global__ void k_nh_half(double* __restrict__ sc, double dt, double gkt, double q) {
    pdl_enter();
    nh_half(sc, dt, gkt, q);
}

// kinetic energy in eV, two-level FP64 tree (fixed order, deterministic)
__global__ void __launch_bounds__(kThreads) k_ekin_partial(int64_t n, const double* __restrict__ vel,
                                                           const double* __restrict__ mass,
                                                           double* __restrict__ partial) {
    pdl_enter();
    __shared__ double sm[kThreads];
    const int64_t base = (int64_t)blockIdx.x * kThreads * kPer;
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int64_t i = base + k * kThreads + threadIdx.x;
        if (i < n) {
            const double vx = vel[3 * i], vy = vel[3 * i + 1], vz = vel[3 * i + 2];
            s += 0.5 * mass[i] * (vx * vx + vy * vy + vz * vz) / kAccel;
        }
    }
    sm[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sm[0];
}

__global__ void __launch_bounds__(kThreads) k_ekin_final(int np, const double* __restrict__ partial,
                                                         double* __restrict__ out) {
    pdl_enter();
    __shared__ double sm[kThreads];
    double s = 0.0;
    for (int i = threadIdx.x; i < np; i += kThreads) s += partial[i];
    sm[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = sm[0];
}

// v += (dt/2) F/m and the step's end: the kinetic energy (FP64, per block of
// kHalfThreads atoms in a fixed tree, then the blocks' sums by the block that finishes
// last, in a fixed order), with tau > 0 the thermostat's half step, the step's energies
// and the bath energy Q xi^2 / 2 + g kT eta into the call's arrays at the step counter,
// and the count of rebuilds.  ints: rebuild gate (left at zero), step counter, rebuild
// count, ticket (atomicInc wraps it to zero).
constexpr int kHalfThreads = 128;
__global__ void __launch_bounds__(kHalfThreads) k_second_half(int64_t n, double* __restrict__ vel,
                                                              const float* __restrict__ forces,
                                                              const double* __restrict__ mass, double half_dt,
                                                              double* __restrict__ partial, double* __restrict__ sc,
                                                              const MdOut* __restrict__ outp, int* __restrict__ ints,
                                                              double dt, double tau, double gkt, double q) {
    pdl_enter();
    __shared__ double sm[kHalfThreads];
    __shared__ bool last;
    const int tid = threadIdx.x;
    const int64_t i = (int64_t)blockIdx.x * kHalfThreads + tid;
    double s = 0.0;
    if (i < n) {
        const double m = mass[i];
        double v2 = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int64_t t = 3 * i + k;
            const double v = vel[t] + half_dt * kAccel * (double)forces[t] / m;
            vel[t] = v;
            v2 += v * v;
        }
        s = 0.5 * m * v2 / kAccel;
    }
    auto tree = [&] {
        sm[tid] = s;
        __syncthreads();
        for (int o = kHalfThreads / 2; o > 0; o >>= 1) {
            if (tid < o) sm[tid] += sm[tid + o];
            __syncthreads();
        }
    };
    tree();
    if (tid == 0) {
        partial[blockIdx.x] = sm[0];
        __threadfence();
        last = atomicInc(reinterpret_cast<unsigned*>(ints + 3), gridDim.x - 1) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    s = 0.0;
    for (int b = tid; b < (int)gridDim.x; b += kHalfThreads) s += __ldcg(partial + b);
    tree();
    if (tid != 0) return;
    sc[1] = sm[0];
    if (tau > 0.0) nh_half(sc, dt, gkt, q);
    const MdOut out = *outp;
    const int k = ints[1];
    if (k < out.n_steps) {
        if (out.e_pot) out.e_pot[k] = sc[0];
        if (out.e_kin) out.e_kin[k] = sc[1];
        if (out.e_bath) out.e_bath[k] = 0.5 * q * sc[2] * sc[2] + gkt * sc[3];
    }
    ints[1] = k + 1;
    if (ints[0]) ints[2] += 1;
    ints[0] = 0;
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

int64_t md_partials(int64_t n) { return blocks_for(n, kHalfThreads); }

cudaError_t launch_md_begin(cudaStream_t s, MdOut* dst, const MdOut& out, int* ints) {
    launch_pdl(k_md_begin, 1, 1, 0, s, dst, out, ints);
    return cudaGetLastError();
}

cudaError_t launch_first_half(cudaStream_t s, int64_t n, double* pos, double* vel, const float* forces,
                              const double* mass, double dt, const double* scale, const double* ref, double skin,
                              int* gate) {
    const double half = 0.5 * skin;
    launch_pdl(k_first_half, blocks_for(n, 64), 64, 0, s, n, pos, vel, forces, mass, 0.5 * dt, dt, scale, ref,
               half * half, gate);
    return cudaGetLastError();
}

cudaError_t launch_second_half(cudaStream_t s, int64_t n, double* vel, const float* forces, const double* mass,
                               double dt, double* partial, double* scalars, const MdOut* out, int* ints, double tau,
                               double gkt, double q) {
    launch_pdl(k_second_half, blocks_for(n, kHalfThreads), kHalfThreads, 0, s, n, vel, forces, mass, 0.5 * dt, partial,
               scalars, out, ints, dt, tau, gkt, q);
    return cudaGetLastError();
}

cudaError_t launch_scale(cudaStream_t s, int64_t n, double* vel, const double* scale) {
    launch_pdl(k_scale, blocks_for(3 * n, 256), 256, 0, s, n, vel, scale);
    return cudaGetLastError();
}

cudaError_t launch_nh_half(cudaStream_t s, double* scalars, double dt, double gkt, double q) {
    launch_pdl(k_nh_half, 1, 1, 0, s, scalars, dt, gkt, q);
    return cudaGetLastError();
}

cudaError_t launch_ekin(cudaStream_t s, int64_t n, const double* vel, const double* mass, double* partial,
                        double* out) {
    const int np = (int)blocks_for(n, kThreads * kPer);
    launch_pdl(k_ekin_partial, np, kThreads, 0, s, n, vel, mass, partial);
    launch_pdl(k_ekin_final, 1, kThreads, 0, s, np, partial, out);
    return cudaGetLastError();
}

}  // namespace reann
