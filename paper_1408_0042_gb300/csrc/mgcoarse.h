// Coarsest multigrid solve on a 3D grid, out = S diag(1 / |mu_i + mu_j + mu_k -
// sig|) S^T in (signed: 1 / (mu - sig)) with S = Sx (x) Sy (x) Sz, in the three
// arithmetic forms of the V-cycle.
//
// One CTA per column (as for 2D grids) keeps 16 or so SMs busy with six
// transforms one after the other: 143 us in FP64 on 16^3 points and 16
// columns, 189 us in double-word arithmetic on 24 x 20 x 16 points and 11
// columns.  Three kernels spread the same sums over the chip: the x and y
// transforms of a z-plane and column, then per (x, y) the transform along z,
// the division and the inverse transform, then the inverse y and x
// transforms.  Every value is summed by one thread in the order of the
// one-CTA form, so the results are the same bits.  Now 31 and 36 us (FP32, 16^3
// points and 32 columns: 40 -> 22 us).
#pragma once

#include "plhr_internal.h"

#ifdef __CUDACC__
namespace plhr {

// Arithmetic of a form: V values, Vs the basis and eigenvalue entries
struct CoarseF64 {
    using V = double;
    static constexpr int kLeast = 0;   // points from which the three kernels win
    static __device__ __forceinline__ V zero() { return 0.0; }
    static __device__ __forceinline__ void madd(V& s, V a, V b) { s += a * b; }
    static __device__ __forceinline__ V scale(V x, V mx, V my, V mz, V sig, int signed_inv) {
        const V mu = mx + my + mz;
        return x / (signed_inv ? mu - sig : fabs(mu - sig));
    }
};
struct CoarseF32 {
    using V = float;
    static constexpr int kLeast = 600;   // V-cycles with 8^3 points 34 us against 36, with 14 x 10 x 6 equal
    static __device__ __forceinline__ V zero() { return 0.0f; }
    static __device__ __forceinline__ void madd(V& s, V a, V b) { s += a * b; }
    static __device__ __forceinline__ V scale(V x, V mx, V my, V mz, V sig, int) {
        const V mu = mx + my + mz;
        return x / fabsf(mu - sig);
    }
};

constexpr int kCoarseThreads = 256;
constexpr int kCoarseLine = 32;       // (x, y, column) elements per CTA of the z kernel
constexpr size_t kCoarseSmem = 160 * 1024;

// FWD: out = (Sx (x) Sy)^T in per z-plane (in: leading dimension ldi, input type
// Tin); else out = (Sx (x) Sy) out.  CTA = column blockIdx.x % nc, plane
// blockIdx.x / nc.
template <class A, bool FWD, typename Tin>
__global__ void __launch_bounds__(kCoarseThreads) k_coarse_plane(int nx, int ny, int nc,
                                                                 const typename A::V* __restrict__ Sx,
                                                                 const typename A::V* __restrict__ Sy, const Tin* in,
                                                                 int64_t ldi, typename A::V* out) {
    using V = typename A::V;
    extern __shared__ __align__(16) unsigned char coarse_sh[];
    const int np = nx * ny;
    V* a = reinterpret_cast<V*>(coarse_sh);
    V* b = a + np;
    V* bx = b + np;
    V* by = bx + nx * nx;
    const int c = blockIdx.x % nc;
    const int64_t p0 = (int64_t)(blockIdx.x / nc) * np;
    for (int i = threadIdx.x; i < nx * nx; i += kCoarseThreads) bx[i] = Sx[i];
    for (int i = threadIdx.x; i < ny * ny; i += kCoarseThreads) by[i] = Sy[i];
    for (int i = threadIdx.x; i < np; i += kCoarseThreads) a[i] = (V)in[(p0 + i) * ldi + c];
    __syncthreads();
    for (int i = threadIdx.x; i < np; i += kCoarseThreads) {
        const int y = i / nx, x = i - y * nx;
        V s = A::zero();
        if (FWD)
            for (int q = 0; q < nx; ++q) A::madd(s, bx[q * nx + x], a[y * nx + q]);
        else
            for (int q = 0; q < ny; ++q) A::madd(s, by[y * ny + q], a[q * nx + x]);
        b[i] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < np; i += kCoarseThreads) {
        const int y = i / nx, x = i - y * nx;
        V s = A::zero();
        if (FWD)
            for (int q = 0; q < ny; ++q) A::madd(s, by[q * ny + y], b[q * nx + x]);
        else
            for (int q = 0; q < nx; ++q) A::madd(s, bx[x * nx + q], b[y * nx + q]);
        out[(p0 + i) * nc + c] = s;
    }
}

// out = Sz diag(1 / |mu - sig|) Sz^T out along z, for 32 consecutive (x, y,
// column) elements per CTA
template <class A>
__global__ void __launch_bounds__(kCoarseThreads) k_coarse_line(int nx, int ny, int nz, int nc,
                                                                const typename A::V* __restrict__ Sz,
                                                                const typename A::V* __restrict__ mx,
                                                                const typename A::V* __restrict__ my,
                                                                const typename A::V* __restrict__ mz,
                                                                typename A::V sig, int signed_inv,
                                                                typename A::V* out) {
    using V = typename A::V;
    extern __shared__ __align__(16) unsigned char coarse_sh[];
    V* a = reinterpret_cast<V*>(coarse_sh);
    V* b = a + nz * kCoarseLine;
    V* bz = b + nz * kCoarseLine;
    const int64_t plane = (int64_t)nx * ny * nc;
    const int64_t e0 = (int64_t)blockIdx.x * kCoarseLine;
    const int lane = threadIdx.x % kCoarseLine, part = threadIdx.x / kCoarseLine;
    constexpr int kParts = kCoarseThreads / kCoarseLine;
    const bool in = e0 + lane < plane;
    for (int i = threadIdx.x; i < nz * nz; i += kCoarseThreads) bz[i] = Sz[i];
    for (int z = part; z < nz; z += kParts) a[z * kCoarseLine + lane] = in ? out[z * plane + e0 + lane] : A::zero();
    __syncthreads();
    const int64_t xy = (e0 + lane) / nc;
    const int iy = in ? (int)(xy / nx) : 0, ix = in ? (int)(xy - (int64_t)iy * nx) : 0;
    for (int m = part; m < nz; m += kParts) {
        V s = A::zero();
        for (int q = 0; q < nz; ++q) A::madd(s, bz[q * nz + m], a[q * kCoarseLine + lane]);
        b[m * kCoarseLine + lane] = A::scale(s, mx[ix], my[iy], mz[m], sig, signed_inv);
    }
    __syncthreads();
    if (!in) return;
    for (int z = part; z < nz; z += kParts) {
        V s = A::zero();
        for (int m = 0; m < nz; ++m) A::madd(s, bz[z * nz + m], b[m * kCoarseLine + lane]);
        out[z * plane + e0 + lane] = s;
    }
}

template <class A>
size_t coarse_plane_smem(const Grid& g) {
    return sizeof(typename A::V) * (size_t)(2 * g.nx * g.ny + g.nx * g.nx + g.ny * g.ny);
}
template <class A>
size_t coarse_line_smem(const Grid& g) {
    return sizeof(typename A::V) * (size_t)(2 * g.nz * kCoarseLine + g.nz * g.nz);
}
// whether the three kernels take this grid: 3D, large enough that three launches pay, a plane and a bundle of z-lines
// fit shared memory, 32-bit launch sizes
template <class A>
bool coarse_split(const Grid& g, int nc) {
    return g.d == 3 && g.n() >= A::kLeast && g.nx <= 1024 && g.ny <= 1024 && g.nz <= 1024 && coarse_plane_smem<A>(g) <= kCoarseSmem &&
           coarse_line_smem<A>(g) <= kCoarseSmem && g.nz * (int64_t)nc < (1 << 30) &&
           g.nx * g.ny * (int64_t)nc < ((int64_t)1 << 35);
}

// out (n0 x nc, dense) = T_0 in; in must not overlap out
template <class A, typename Tin>
cudaError_t coarse_solve_split(const Grid& g, int nc, const typename A::V* const* S, const typename A::V* const* mu,
                               typename A::V sig, int signed_inv, const Tin* in, int64_t ldi, typename A::V* out,
                               cudaStream_t s) {
    using V = typename A::V;
    const int nx = (int)g.nx, ny = (int)g.ny, nz = (int)g.nz;
    const size_t sp = coarse_plane_smem<A>(g), sl = coarse_line_smem<A>(g);
    cudaError_t e = cudaSuccess;
    if (sp > 48 * 1024) {
        e = cudaFuncSetAttribute(k_coarse_plane<A, true, Tin>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_coarse_plane<A, false, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp);
    }
    if (e == cudaSuccess && sl > 48 * 1024)
        e = cudaFuncSetAttribute(k_coarse_line<A>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sl);
    if (e != cudaSuccess) return e;
    const int lines = (int)(((int64_t)nx * ny * nc + kCoarseLine - 1) / kCoarseLine);
    k_coarse_plane<A, true, Tin><<<nz * nc, kCoarseThreads, sp, s>>>(nx, ny, nc, S[0], S[1], in, ldi, out);
    k_coarse_line<A><<<lines, kCoarseThreads, sl, s>>>(nx, ny, nz, nc, S[2], mu[0], mu[1], mu[2], sig, signed_inv, out);
    k_coarse_plane<A, false, V><<<nz * nc, kCoarseThreads, sp, s>>>(nx, ny, nc, S[0], S[1], out, nc, out);
    count_launches(3);
    return cudaGetLastError();
}

}  // namespace plhr
#endif
