// Absolute-value multigrid V-cycle (Appendix A, Algorithm 4) on blocks of
// vectors [grid point][column], FP64.
//
// Per smoothing level l (finest first):
//   step 2  pre-smoothing  w <- w + omega_l (r - B_l w), nu times from w = 0
//   step 3  r_c = R (r - B_l w), w_c = AV-MG(r_c) (or the exact coarsest
//           solve), w <- w + P w_c
//   step 4  post-smoothing, nu times (M_l = omega_l^{-1} I is symmetric, so
//           M_l^{-*} = M_l^{-1})
// B_l is the level Laplacian L_l or p_2(L_l - sigma I) = ((L_l - sigma)^2 +
// c_l^2)/(2 c_l).  Transfers are cell-centred: the restriction is R = P^T / 2^d
// for the prolongation P (piecewise constant, or the tensor product of the 1D
// weights 3/4, 1/4 to the two nearest coarse cells).  The coarsest solve
// applies |L_0 - sigma I|^{-1} = S diag(1 / |mu - sigma|) S^T with a separable
// orthonormal basis S = Sx (x) Sy (x) Sz and per-axis eigenvalues mu.
//
// INV-MG (Appendix A, Algorithm 5; H.indefinite): the same cycle with
// B_l = L_l - sigma I_l on every level (the shift enters the sweeps and the
// residual) and the signed coarsest solve S diag(1 / (mu - sigma)) S^T.
#include "fxsum.h"
#include "mgcoarse.h"
#include "plhr_internal.h"

namespace plhr {
namespace {

constexpr int kT = 256;

struct G3 {
    int64_t nx, ny, nz;
};

__device__ __forceinline__ void unflat(int64_t row, const G3& g, int64_t& ix, int64_t& iy, int64_t& iz) {
    if ((uint64_t)row <= 0xffffffffull) {   // 32-bit divisions (the grid fits: nx, ny < 2^32)
        const unsigned r = (unsigned)row, nx = (unsigned)g.nx, ny = (unsigned)g.ny;
        const unsigned t = r / nx;
        ix = r - t * nx;
        const unsigned z = t / ny;
        iy = t - z * ny;
        iz = z;
        return;
    }
    ix = row % g.nx;
    int64_t t = row / g.nx;
    iy = t % g.ny;
    iz = t / g.ny;
}

// Sum of the neighbours of x at xp, zero outside the grid
template <bool D3>
__device__ __forceinline__ double nb_sum(const double* __restrict__ xp, int64_t ld, int64_t ix, int64_t iy,
                                         int64_t iz, const G3& g) {
    const int64_t sy = ld * g.nx, sz = sy * g.ny;
    const double x0 = ix > 0 ? xp[-ld] : 0.0, x1 = ix < g.nx - 1 ? xp[ld] : 0.0;
    const double y0 = iy > 0 ? xp[-sy] : 0.0, y1 = iy < g.ny - 1 ? xp[sy] : 0.0;
    double s = (x0 + x1) + (y0 + y1);
    if (D3) {
        const double z0 = iz > 0 ? xp[-sz] : 0.0, z1 = iz < g.nz - 1 ? xp[sz] : 0.0;
        s += z0 + z1;
    }
    return s;
}

#define GRID_LOOP(total)                                                                 \
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (total);        \
         e += (int64_t)gridDim.x * blockDim.x)

// The FP64 pipe (1/64 of the FP32 rate) binds these kernels, so each is written
// in as few FP64 operations as its stencil allows: five additions for the
// neighbours and one multiply(-add) per coefficient, the coefficients formed on
// the host.  (64^3 x 16: a sweep 77 -> 69 us; the first two sweeps, one kernel
// now, 95 -> 61 us.)

// out = cx x + cn sum of x's neighbours (+ cr r when r is given): the sweeps
// w + om (r - (ih2 L - shift) w), 2 om r - om^2 (ih2 L - shift) r (the first two
// sweeps from zero in one), the residual r - (ih2 L - shift) w and (ih2 L - sig) x
template <bool D3, bool R>
__global__ void __launch_bounds__(kT) k_stencil(G3 g, int nc, double cx, double cn, double cr,
                                                const double* __restrict__ x, int64_t ldx,
                                                const double* __restrict__ r, int64_t ldr, double* __restrict__ out,
                                                int64_t total) {
    GRID_LOOP(total) {
        int64_t row;
        int c;
        split_index(e, nc, row, c);
        int64_t ix, iy, iz;
        unflat(row, g, ix, iy, iz);
        const double* xp = x + row * ldx + c;
        const double s = nb_sum<D3>(xp, ldx, ix, iy, iz, g);
        double v = cn * s;
        if (R) v = fma(cr, r[row * ldr + c], v);
        out[row * nc + c] = fma(cx, xp[0], v);
    }
}

// The two for blocks on which the FP64 pipe binds: the neighbours are summed on the
// integer pipes, which leaves five FP64 operations of eight in a sweep (64^3 x 16: a
// sweep 69 -> 51 us, the first two 61 -> 41, FP64 pipe 71-75 % and integer ALU 45-59 %
// busy).
template <bool D3, bool R>
__global__ void __launch_bounds__(kFxThreads) k_stencil_fx(FxBox g, int nc, int planes, double cx, double cn, double cr,
                                                           const double* __restrict__ x, int64_t ldx,
                                                           const double* __restrict__ r, int64_t ldr,
                                                           double* __restrict__ out) {
    fx_walk<D3, false>(g, nc, planes, cn, x, ldx, [&](int64_t row, int c, double xc, double v) {
        if (R) v = fma(cr, r[row * ldr + c], v);
        out[row * nc + c] = fma(cx, xc, v);
    });
}
template <bool D3>
__global__ void __launch_bounds__(kFxThreads) k_poly_fx(FxBox g, int nc, int planes, double cw, double cr, double ct,
                                                        double cn, const double* __restrict__ w,
                                                        const double* __restrict__ t, const double* __restrict__ r,
                                                        int64_t ldr, double* __restrict__ out) {
    fx_walk<D3, false>(g, nc, planes, cn, t, nc, [&](int64_t row, int c, double tc, double v) {
        v = fma(ct, tc, v);
        v = fma(cw, w[row * nc + c], v);
        out[row * nc + c] = fma(cr, r[row * ldr + c], v);
    });
}

// w = om r (one sweep from zero)
__global__ void __launch_bounds__(kT) k_scale(int nc, double om, const double* __restrict__ r, int64_t ldr,
                                              double* __restrict__ w, int64_t total) {
    GRID_LOOP(total) {
        int64_t row;
        int c;
        split_index(e, nc, row, c);
        w[e] = om * r[row * ldr + c];
    }
}

// polynomial level, t = (L - sig) w, B w = ((L - sig) t + c^2 w) / (2 c):
// out = cw w + cr r + ct t + cn sum of t's neighbours is the sweep w + om (r - B w)
// or the residual r - B w
template <bool D3>
__global__ void __launch_bounds__(kT) k_poly_step(G3 g, int nc, double cw, double cr, double ct, double cn,
                                                  const double* __restrict__ w, const double* __restrict__ t,
                                                  const double* __restrict__ r, int64_t ldr, double* __restrict__ out,
                                                  int64_t total) {
    GRID_LOOP(total) {
        int64_t row;
        int c;
        split_index(e, nc, row, c);
        int64_t ix, iy, iz;
        unflat(row, g, ix, iy, iz);
        const double* tp = t + row * nc + c;
        double v = fma(ct, tp[0], cn * nb_sum<D3>(tp, nc, ix, iy, iz, g));
        v = fma(cw, w[row * nc + c], v);
        out[row * nc + c] = fma(cr, r[row * ldr + c], v);
    }
}

// Transfers, one segment of a grid line per CTA, separably, with the
// weights' common power of two taken out: linear prolongation is (3 a + b) / 4
// per axis (a the coarse cell of the fine point, b the next nearest, zero
// outside), linear restriction (3 (a + b) + (c + d)) / 8 (a, b the children of
// the coarse cell, c, d the fine points beside them); constant ones are a and
// (a + b) / 2.  The y-z part of a segment goes to shared memory, then x.  4.5 and 3.5
// FP64 operations per fine value instead of the 24 and 25 of a tensor product of
// weights per point.  (64^3 x 16: restriction 116 -> 58 us, prolongation 174 -> 35 us.)

struct LineCut {
    int cols;   // columns per CTA (blockIdx.y: first one / cols)
    int seg;    // coarse points per CTA (blockIdx.z: first one / seg)
};

// w_fine += P w_coarse on fine line blockIdx.x = (y, z)
template <bool D3>
__global__ void __launch_bounds__(kT) k_prolong_line(G3 gf, G3 gc, int nc, LineCut k, int lin,
                                                     const double* __restrict__ wc, double* __restrict__ wf) {
    extern __shared__ double line_sh[];   // [coarse x0 - 1 ..][column]
    const int64_t line = blockIdx.x;
    const int64_t iz = line / gf.ny, iy = line - iz * gf.ny;
    const int c0 = blockIdx.y * k.cols, cols = min(k.cols, nc - c0);
    const int x0 = blockIdx.z * k.seg, seg = min(k.seg, (int)gc.nx - x0);
    const int64_t ya = iy >> 1, yb = (iy & 1) ? ya + 1 : ya - 1;
    const int64_t za = D3 ? iz >> 1 : 0, zb = (iz & 1) ? za + 1 : za - 1;
    const bool hy = lin && yb >= 0 && yb < gc.ny, hz = D3 && lin && zb >= 0 && zb < gc.nz;
    const double* paa = wc + (za * gc.ny + ya) * gc.nx * nc + c0;
    const double* pab = wc + (za * gc.ny + yb) * gc.nx * nc + c0;
    const double* pba = wc + (zb * gc.ny + ya) * gc.nx * nc + c0;
    const double* pbb = wc + (zb * gc.ny + yb) * gc.nx * nc + c0;
    for (int t = threadIdx.x; t < (seg + 2) * cols; t += kT) {
        const int q = t / cols, c = t - q * cols;
        const int x = x0 - 1 + q;
        double v = 0.0;
        if (x >= 0 && x < (int)gc.nx) {
            const int64_t o = (int64_t)x * nc + c;
            v = paa[o];
            if (lin) {
                const double vb = hy ? pab[o] : 0.0;
                v = fma(3.0, v, vb);
                if (D3) {
                    const double wa = hz ? pba[o] : 0.0, wb = hz && hy ? pbb[o] : 0.0;
                    v = fma(3.0, v, fma(3.0, wa, wb));
                }
            }
        }
        line_sh[t] = v;
    }
    __syncthreads();
    const double scale = lin ? (D3 ? 0x1p-6 : 0x1p-4) : 1.0;
    for (int t = threadIdx.x; t < 2 * seg * cols; t += kT) {
        const int x = t / cols, c = t - x * cols;   // fine point 2 x0 + x
        const double* u = line_sh + ((x >> 1) + 1) * cols + c;
        double v = u[0];
        if (lin) v = fma(3.0, v, (x & 1) ? u[cols] : u[-cols]);
        double* w = wf + (line * gf.nx + 2 * x0 + x) * nc + c0 + c;
        *w = fma(scale, v, *w);
    }
}

// rc = R f on coarse line blockIdx.x = (y, z)
template <bool D3>
__global__ void __launch_bounds__(kT) k_restrict_line(G3 gf, G3 gc, int nc, LineCut k, int lin,
                                                      const double* __restrict__ f, double* __restrict__ rc) {
    extern __shared__ double line_sh[];   // [fine 2 x0 - 1 ..][column]
    const int64_t line = blockIdx.x;
    const int64_t iz = line / gc.ny, iy = line - iz * gc.ny;
    const int c0 = blockIdx.y * k.cols, cols = min(k.cols, nc - c0);
    const int x0 = blockIdx.z * k.seg, seg = min(k.seg, (int)gc.nx - x0);
    const int64_t ys = gf.nx * nc, zs = ys * gf.ny;
    const bool y0 = lin && 2 * iy - 1 >= 0, y3 = lin && 2 * iy + 2 < gf.ny;
    const bool z0 = D3 && lin && 2 * iz - 1 >= 0, z3 = D3 && lin && 2 * iz + 2 < gf.nz;
    const double* p0 = f + 2 * iy * ys + (D3 ? 2 * iz * zs : 0) + c0;
    // the y sum of a fine plane, in eighths (halves when constant)
    auto ysum = [&](const double* p) {
        const double a = p[0], b = p[ys];
        if (!lin) return a + b;
        const double c = y0 ? p[-ys] : 0.0, d = y3 ? p[2 * ys] : 0.0;
        return fma(3.0, a + b, c + d);
    };
    for (int t = threadIdx.x; t < (2 * seg + 2) * cols; t += kT) {
        const int q = t / cols, c = t - q * cols;
        const int x = 2 * x0 - 1 + q;
        double v = 0.0;
        if (x >= 0 && x < (int)gf.nx) {
            const double* p = p0 + (int64_t)x * nc + c;
            v = ysum(p);
            if (D3) {
                const double b = ysum(p + zs);
                if (!lin) {
                    v += b;
                } else {
                    const double cz = z0 ? ysum(p - zs) : 0.0, d = z3 ? ysum(p + 2 * zs) : 0.0;
                    v = fma(3.0, v + b, cz + d);
                }
            }
        }
        line_sh[t] = v;
    }
    __syncthreads();
    const double scale = lin ? (D3 ? 0x1p-9 : 0x1p-6) : (D3 ? 0x1p-3 : 0x1p-2);
    for (int t = threadIdx.x; t < seg * cols; t += kT) {
        const int x = t / cols, c = t - x * cols;
        const double* p = line_sh + (2 * x + 1) * cols + c;
        double v = p[0] + p[cols];
        if (lin) v = fma(3.0, v, p[-cols] + p[2 * cols]);
        rc[(line * gc.nx + x0 + x) * nc + c0 + c] = scale * v;
    }
}

// Coarsest solve, one CTA per column: out = S diag(1/|mu_i + mu_j + mu_k - sig|) S^T in
// (signed: 1 / (mu - sig)); the two work vectors of the column live in shared
// memory, or in global scratch (gwork, 2 n0 doubles per column) when the
// coarsest grid is too large for it
// (S[point][mode] per axis, orthonormal).
// coarsest level: 1024 threads per column (each output is still one thread's
// sum in a fixed order); the transforms of one column are latency-bound
constexpr int kTC = 1024;
__global__ void __launch_bounds__(kTC) k_coarse_sep(int d, int64_t nx, int64_t ny, int64_t nz, int nc,
                                                   const double* __restrict__ Sx, const double* __restrict__ Sy,
                                                   const double* __restrict__ Sz, const double* __restrict__ mx,
                                                   const double* __restrict__ my, const double* __restrict__ mz,
                                                   double sig, int signed_inv, const double* __restrict__ in,
                                                   int64_t ldi, double* __restrict__ out, int64_t ldo,
                                                   double* __restrict__ gwork) {
    extern __shared__ double sh[];
    const int64_t n0 = nx * ny * nz;
    const int c = blockIdx.x;
    double* a = gwork ? gwork + (int64_t)c * 2 * n0 : sh;
    double* b = a + n0;
    for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) a[i] = in[i * ldi + c];
    __syncthreads();
    // forward: coefficient(mode) = sum_point S[point][mode] x[point], axis by axis
    // x axis
    for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) {
        int64_t m = i % nx, rest = i / nx;
        double s = 0.0;
        for (int64_t p = 0; p < nx; ++p) s += Sx[p * nx + m] * a[rest * nx + p];
        b[i] = s;
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) {
        int64_t x = i % nx, m = (i / nx) % ny, z = i / (nx * ny);
        double s = 0.0;
        for (int64_t p = 0; p < ny; ++p) s += Sy[p * ny + m] * b[(z * ny + p) * nx + x];
        a[i] = s;
    }
    __syncthreads();
    if (d == 3) {
        for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) {
            int64_t xy = i % (nx * ny), m = i / (nx * ny);
            double s = 0.0;
            for (int64_t p = 0; p < nz; ++p) s += Sz[p * nz + m] * a[p * nx * ny + xy];
            b[i] = s;
        }
        __syncthreads();
    } else {
        for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) b[i] = a[i];
        __syncthreads();
    }
    // scale
    for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) {
        int64_t ix = i % nx, iy = (i / nx) % ny, iz = i / (nx * ny);
        double mu = mx[ix] + my[iy] + (d == 3 ? mz[iz] : 0.0);
        b[i] = b[i] / (signed_inv ? mu - sig : fabs(mu - sig));
    }
    __syncthreads();
    // inverse: x[point] = sum_mode S[point][mode] coef[mode]
    if (d == 3) {
        for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) {
            int64_t xy = i % (nx * ny), p = i / (nx * ny);
            double s = 0.0;
            for (int64_t m = 0; m < nz; ++m) s += Sz[p * nz + m] * b[m * nx * ny + xy];
            a[i] = s;
        }
        __syncthreads();
    } else {
        for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) a[i] = b[i];
        __syncthreads();
    }
    for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) {
        int64_t x = i % nx, p = (i / nx) % ny, z = i / (nx * ny);
        double s = 0.0;
        for (int64_t m = 0; m < ny; ++m) s += Sy[p * ny + m] * a[(z * ny + m) * nx + x];
        b[i] = s;
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n0; i += blockDim.x) {
        int64_t p = i % nx, rest = i / nx;
        double s = 0.0;
        for (int64_t m = 0; m < nx; ++m) s += Sx[p * nx + m] * b[rest * nx + m];
        out[i * ldo + c] = s;
    }
}

G3 g3(const Grid& g) { return G3{g.nx, g.ny, g.nz}; }

int nblk(int64_t total) { return grid_size_for(total, kT, sm_count() * 16); }

struct LevelBufs {
    double* cw;    // coarsest level only: global scratch of a large coarsest solve
    double* w0;    // ping
    double* w1;    // pong
    double* tmp;   // residual / polynomial intermediate
    double* rc;    // restricted residual for the next coarser level
    double* wc;    // coarse correction from the next coarser level
};

// out = cx x + cn sum of neighbours (+ cr r)
void launch_stencil(const Grid& g, int nc, double cx, double cn, double cr, const double* x, int64_t ldx,
                    const double* r, int64_t ldr, double* out, cudaStream_t s) {
    const int64_t total = g.n() * nc;
    const G3 G = g3(g);
    const int nb = nblk(total);
    const FxBox box{g.nx, g.ny, g.nz, 0};
    if (const int planes = fx_planes(g.d, box, nc, cn)) {
        auto go = [&](auto kern) {
            kern<<<fx_grid(g.d, box, nc, planes), kFxThreads, 0, s>>>(box, nc, planes, cx, cn, cr, x, ldx, r, ldr, out);
        };
        if (g.d == 3) go(r ? k_stencil_fx<true, true> : k_stencil_fx<true, false>);
        else go(r ? k_stencil_fx<false, true> : k_stencil_fx<false, false>);
    } else if (g.d == 3) {
        if (r) k_stencil<true, true><<<nb, kT, 0, s>>>(G, nc, cx, cn, cr, x, ldx, r, ldr, out, total);
        else k_stencil<true, false><<<nb, kT, 0, s>>>(G, nc, cx, cn, cr, x, ldx, r, ldr, out, total);
    } else {
        if (r) k_stencil<false, true><<<nb, kT, 0, s>>>(G, nc, cx, cn, cr, x, ldx, r, ldr, out, total);
        else k_stencil<false, false><<<nb, kT, 0, s>>>(G, nc, cx, cn, cr, x, ldx, r, ldr, out, total);
    }
    count_launches(1);
}

// out = cw w + cr (r - B w), B the level's operator (tmp: scratch of a polynomial level)
cudaError_t level_step(const MGLevel& L, double sigma, int nc, double cw, double cr, const double* w, const double* r,
                       int64_t ldr, double* tmp, double* out, cudaStream_t s) {
    const Grid& g = L.g;
    const double ih2 = g.inv_h2(), diag = 2.0 * g.d * ih2;
    if (!L.poly) {
        const double shift = L.shifted ? sigma : 0.0;
        launch_stencil(g, nc, cw - cr * (diag - shift), cr * ih2, cr, w, nc, r, ldr, out, s);
        return cudaGetLastError();
    }
    launch_stencil(g, nc, diag - sigma, -ih2, 0.0, w, nc, nullptr, 0, tmp, s);
    const double cb = cr / (2.0 * L.c);   // weight of (L - sig) t + c^2 w
    const int64_t total = g.n() * nc;
    const FxBox box{g.nx, g.ny, g.nz, 0};
    if (const int planes = fx_planes(g.d, box, nc, cb * ih2)) {
        auto kern = g.d == 3 ? k_poly_fx<true> : k_poly_fx<false>;
        kern<<<fx_grid(g.d, box, nc, planes), kFxThreads, 0, s>>>(box, nc, planes, cw - cb * L.c * L.c, cr,
                                                                  -cb * (diag - sigma), cb * ih2, w, tmp, r, ldr, out);
    } else if (g.d == 3)
        k_poly_step<true><<<nblk(total), kT, 0, s>>>(g3(g), nc, cw - cb * L.c * L.c, cr, -cb * (diag - sigma), cb * ih2,
                                                     w, tmp, r, ldr, out, total);
    else
        k_poly_step<false><<<nblk(total), kT, 0, s>>>(g3(g), nc, cw - cb * L.c * L.c, cr, -cb * (diag - sigma), cb * ih2,
                                                      w, tmp, r, ldr, out, total);
    count_launches(1);
    return cudaGetLastError();
}

// CTAs of the line transfers: up to 32 columns, segments whose fine points fit
// 32 KB (64 points of 32 columns, whole lines at the usual sizes)
LineCut line_cut(const Grid& gc, int nc) {
    LineCut k;
    k.cols = nc < 32 ? nc : 32;
    const int64_t fit = 32 * 1024 / (int64_t)sizeof(double) / k.cols / 2 - 1;
    k.seg = (int)(fit < gc.nx ? fit : gc.nx);
    return k;
}
dim3 line_grid(int64_t lines, const Grid& gc, int nc, const LineCut& k) {
    return dim3((unsigned)lines, (unsigned)((nc + k.cols - 1) / k.cols), (unsigned)((gc.nx + k.seg - 1) / k.seg));
}

// largest coarsest grid whose two work vectors are staged in shared memory
constexpr int64_t kCoarseShmPoints = kMaxSmemCoarse;

cudaError_t coarse_solve(const MGHierarchy& H, int nc, const double* in, int64_t ldi, double* out, int64_t ldo,
                         double* gwork, cudaStream_t s) {
    const Grid& g = H.lev[0].g;
    if (ldo == nc && coarse_split<CoarseF64>(g, nc))
        return coarse_solve_split<CoarseF64>(g, nc, H.d_basis, H.d_mu, H.sigma, H.indefinite, in, ldi, out, s);
    int64_t n0 = g.n();
    const bool global = n0 > kCoarseShmPoints;
    size_t shm = global ? 0 : sizeof(double) * 2 * n0;
    if (shm > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_coarse_sep, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
        if (e != cudaSuccess) return e;
    }
    k_coarse_sep<<<nc, kTC, shm, s>>>(g.d, g.nx, g.ny, g.nz, nc, H.d_basis[0], H.d_basis[1],
                                     g.d == 3 ? H.d_basis[2] : H.d_basis[1], H.d_mu[0], H.d_mu[1],
                                     g.d == 3 ? H.d_mu[2] : H.d_mu[1], H.sigma, H.indefinite, in, ldi, out, ldo,
                                     global ? gwork : nullptr);
    count_launches(1);
    return cudaGetLastError();
}

// Recursive V-cycle on level l; r has leading dimension ldr (level nc otherwise);
// the result is written to out with leading dimension nc.
cudaError_t vcycle(const MGHierarchy& H, int l, int nc, const double* r, int64_t ldr, double* out,
                   std::vector<LevelBufs>& B, cudaStream_t s) {
    if (l == 0) return coarse_solve(H, nc, r, ldr, out, nc, B[0].cw, s);
    const MGLevel& L = H.lev[l];
    const MGLevel& Lc = H.lev[l - 1];
    LevelBufs& b = B[l];
    cudaError_t e;
    const Grid& g = L.g;
    const double ih2 = g.inv_h2(), om = L.omega;
    // pre-smoothing from zero; on a level without the polynomial the first two
    // sweeps are one: 2 om r - om^2 B r
    double* cur = b.w0;
    double* nxt = b.w1;
    int done = 1;
    if (!L.poly && H.nu >= 2) {
        const double diag = 2.0 * g.d * ih2 - (L.shifted ? H.sigma : 0.0);
        launch_stencil(g, nc, 2.0 * om - om * om * diag, om * om * ih2, 0.0, r, ldr, nullptr, 0, cur, s);
        done = 2;
    } else {
        k_scale<<<nblk(g.n() * nc), kT, 0, s>>>(nc, om, r, ldr, cur, g.n() * nc);
        count_launches(1);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    for (int i = done; i < H.nu; ++i) {
        e = level_step(L, H.sigma, nc, 1.0, om, cur, r, ldr, b.tmp, nxt, s);
        if (e != cudaSuccess) return e;
        double* t = cur; cur = nxt; nxt = t;
    }
    // coarse-grid correction
    e = level_step(L, H.sigma, nc, 0.0, 1.0, cur, r, ldr, b.tmp, nxt, s);
    if (e != cudaSuccess) return e;
    const LineCut cut = line_cut(Lc.g, nc);
    const size_t sm = sizeof(double) * 2 * (cut.seg + 1) * cut.cols;
    const dim3 gr = line_grid(Lc.g.ny * Lc.g.nz, Lc.g, nc, cut), gp = line_grid(g.ny * g.nz, Lc.g, nc, cut);
    if (g.d == 3) k_restrict_line<true><<<gr, kT, sm, s>>>(g3(g), g3(Lc.g), nc, cut, H.linear, nxt, b.rc);
    else k_restrict_line<false><<<gr, kT, sm, s>>>(g3(g), g3(Lc.g), nc, cut, H.linear, nxt, b.rc);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = vcycle(H, l - 1, nc, b.rc, nc, b.wc, B, s);
    if (e != cudaSuccess) return e;
    if (g.d == 3) k_prolong_line<true><<<gp, kT, sm, s>>>(g3(g), g3(Lc.g), nc, cut, H.linear, b.wc, cur);
    else k_prolong_line<false><<<gp, kT, sm, s>>>(g3(g), g3(Lc.g), nc, cut, H.linear, b.wc, cur);
    count_launches(1);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // post-smoothing; the last step writes to out
    for (int i = 0; i < H.nu; ++i) {
        double* dst = (i == H.nu - 1) ? out : nxt;
        e = level_step(L, H.sigma, nc, 1.0, om, cur, r, ldr, b.tmp, dst, s);
        if (e != cudaSuccess) return e;
        nxt = cur;
        cur = dst;
    }
    return cudaSuccess;
}

}  // namespace

int64_t mg_workspace_doubles(const MGHierarchy& H, int nc) {
    int64_t tot = 0;
    for (size_t l = 1; l < H.lev.size(); ++l) {
        tot += 3 * H.lev[l].g.n() * nc;            // w0, w1, tmp
        tot += 2 * H.lev[l - 1].g.n() * nc;        // rc, wc
    }
    if (H.lev[0].g.n() > kCoarseShmPoints) tot += 2 * H.lev[0].g.n() * nc;   // large coarsest solve
    return tot;
}

cudaError_t mg_vcycle(const MGHierarchy& H, int nc, const double* r, int64_t ldr, double* w, int64_t ldw,
                      double* work, cudaStream_t s) {
    if (nc <= 0) return cudaSuccess;
    const int top = (int)H.lev.size() - 1;
    std::vector<LevelBufs> B(H.lev.size());
    double* p = work;
    B[0].cw = nullptr;
    for (int l = 1; l <= top; ++l) {
        int64_t nf = H.lev[l].g.n() * nc, ncc = H.lev[l - 1].g.n() * nc;
        B[l].w0 = p; p += nf;
        B[l].w1 = p; p += nf;
        B[l].tmp = p; p += nf;
        B[l].rc = p; p += ncc;
        B[l].wc = p; p += ncc;
    }
    if (H.lev[0].g.n() > kCoarseShmPoints) B[0].cw = p;
    // the kernels use leading dimension nc for level buffers; the caller's
    // output must be dense (ldw == nc) or is staged through the ping buffer
    if (ldw == nc) return vcycle(H, top, nc, r, ldr, w, B, s);
    return cudaErrorInvalidValue;
}

}  // namespace plhr
