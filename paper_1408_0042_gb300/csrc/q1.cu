// 27-point trilinear (Q1) finite-element stiffness and mass products, and the
// complex Bloch Hamiltonian product, on blocks stored row-major
// [grid point][column].
//
// Q1 (Section 5.1's bilinear elements, in 3D).  The unknowns are the interior
// nodes of a tensor mesh of E_a = n_a + 1 elements per axis with width h;
// interior node i (0-based) sits at mesh point i + 1 and belongs to the cells
// i (as their upper corner) and i + 1 (as their lower corner) along each axis.
// With the 1D linear-element matrices k = [[1, -1], [-1, 1]] / h and
// m = [[2, 1], [1, 2]] h / 6, the element stiffness entry between local
// corners a and b depends only on which axes differ (d_a = [a_a != b_a]):
//     K_e(a, b) = c_e (k(d_x) m(d_y) m(d_z) + m(d_x) k(d_y) m(d_z) + m(d_x) m(d_y) k(d_z)),
//     k(0) = 1/h, k(1) = -1/h, m(0) = 2h/6, m(1) = h/6,
// and the assembled mass matrix is the tensor product of the 1D rows [1, 4, 1]
// h / 6 (coefficient-free).  Nodes on the boundary carry the homogeneous
// Dirichlet value 0.
//
// The FP64 pipe (1/64 of the FP32 rate) binds these products, so the stiffness
// is applied in the basis that diagonalises every element matrix: sums and
// differences of the corner values along each axis.  k has the eigenvalues 0
// and 2 / h there and m has h / 2 and h / 6, so an element's combination with n
// differences is multiplied by c_e h (4 - n) / 48 (0 for n = 0).  The sums and
// differences of a face are formed once and used for the elements above and
// below it (a thread walks up the z axis with its face), and an element's
// products leave through the same butterflies: about 36 FP64 operations per
// node instead of the 72 multiply-adds of 8 cells times 8 corners, with the mass
// product 47 instead of 130 (64^3 elements, 9 columns: 499 -> 271 us; the tiles'
// repeated faces, partly filled warps and the SMs without a CTA make the pipe's
// 188 us 245).
//
// Bloch Hamiltonian (Section 5.3, complex Hermitian): periodic 7-point
// stencil with the phase e^{i kappa_d h} on the link j -> j + e_d and the
// potential on the diagonal, on complex128 blocks (re, im interleaved).
#include "plhr_internal.h"

namespace plhr {
namespace {

struct Q1Geo {
    int64_t nx, ny, nz;   // interior nodes per axis
    double h;
    const double* cell;   // element coefficients ((nx+1)(ny+1)(nz+1), x fastest) or null (c = 1)
};

enum { Q1_AXPBY = 0, Q1_SHIFTS = 1, Q1_PAIR = 2 };

// Tile of a CTA: faces (fx, fy), fx <= tx, fy <= ty, for cols columns; face
// (fx, fy) has its lower corner at node (x0 + fx - 1, y0 + fy - 1), and the
// nodes with fx, fy >= 1 are the tile's outputs; tz node planes.
struct Q1Tile {
    int cols, chunks, tx, ty, tz, ntx;
};

// MODE Q1_AXPBY: y = alpha (op x) + beta x; Q1_SHIFTS: y = op x, o1 = y - lam_c x,
// o2 = y - sig x (each optional), op = stiffness (A) or mass (B);
// Q1_PAIR: y = stiffness x, o1 = mass x.  The stiffness carries ca = scale h / 48,
// the mass cb = scale (h / 6)^3.
template <int MODE, bool A, bool B>
__global__ void __launch_bounds__(1024) k_q1(Q1Geo g, Q1Tile k, int nc, double ca, double cb,
                                             const double* __restrict__ x, int64_t ldx, double* __restrict__ y,
                                             int64_t ldy, double* __restrict__ o1, int64_t ld1,
                                             const double* __restrict__ lam, double* __restrict__ o2, int64_t ld2,
                                             double alpha, double beta, double sig) {
    extern __shared__ double corner[];   // [plane parity][corner][fy][fx][column]
    const int fxn = k.tx + 1, fyn = k.ty + 1;
    const int cells = fxn * fyn * k.cols;
    const int c0 = (int)(blockIdx.x % k.chunks) * k.cols;
    const int64_t tile = blockIdx.x / k.chunks;
    const int t = threadIdx.x, c = t % k.cols, f = t / k.cols;
    const int fx = f % fxn, fy = f / fxn;
    const int64_t gx = (tile % k.ntx) * k.tx + fx - 1, gy = (tile / k.ntx) * k.ty + fy - 1;
    const int col = c0 + c;
    const bool face = t < cells && col < nc && gx < g.nx && gy < g.ny;
    const bool node = face && fx >= 1 && fy >= 1;
    const int64_t z0 = (int64_t)blockIdx.y * k.tz, z1 = z0 + k.tz < g.nz ? z0 + k.tz : g.nz;
    const bool xl = gx >= 0, xr = gx + 1 < g.nx, yl = gy >= 0, yr = gy + 1 < g.ny;
    const bool xm = gx >= 1, ym = gy >= 1;
    const int64_t sy = g.nx * ldx, ex = g.nx + 1;
    double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;   // face sums of the plane below: SS, SD, DS, DD (x first)
    double u0 = 0.0, u1 = 0.0, u2 = 0.0, u3 = 0.0;   // what the element below gives its upper face
    double m1 = 0.0, m2 = 0.0;                        // [1 4 1] x [1 4 1] sums of the two planes below
    double vprev = 0.0;                               // the node's value on the plane below
    for (int64_t p = z0 - 1; p <= z1; ++p) {
        // corner values of the face: v(x, y) with x, y in {0, 1}; zero on the boundary
        double v00 = 0.0, v10 = 0.0, v01 = 0.0, v11 = 0.0;
        double mass = 0.0;
        if (face && p >= 0 && p < g.nz) {
            const double* q = x + ((p * g.ny + gy) * g.nx + gx) * ldx + col;
            if (yl) {
                if (xl) v00 = q[0];
                if (xr) v10 = q[ldx];
            }
            if (yr) {
                if (xl) v01 = q[sy];
                if (xr) v11 = q[sy + ldx];
            }
            if (B && node) {
                const double a0 = xm && ym ? q[-sy - ldx] : 0.0, a1 = ym ? q[-sy] : 0.0, a2 = xr && ym ? q[-sy + ldx] : 0.0;
                const double b0 = xm ? q[-ldx] : 0.0, d0 = xm && yr ? q[sy - ldx] : 0.0;
                const double below = fma(4.0, a1, a0 + a2), mid = fma(4.0, v00, b0 + v10), above = fma(4.0, v01, d0 + v11);
                mass = fma(4.0, mid, below + above);
            }
        }
        double f0, f1, f2, f3;
        const int buf = (int)(p & 1) * 4 * cells;
        if (A) {
            const double s0 = v00 + v10, d0 = v10 - v00, s1 = v01 + v11, d1 = v11 - v01;
            f0 = s0 + s1; f1 = s1 - s0; f2 = d0 + d1; f3 = d1 - d0;
            if (p >= z0) {
                // The element between planes p - 1 and p: sum and difference of
                // (lower, upper) times (4 - n) c_e h / 48 and (3 - n) c_e h / 48,
                // back to (lower, upper), e.g. n = 1: 3 (f + p) -+ 2 (f - p) = f + 5 p, 5 f + p
                const double c1 = face && g.cell ? ca * g.cell[(p * (g.ny + 1) + gy + 1) * ex + gx + 1] : ca;
                const double t0 = 3.0 * c1 * (f0 - p0);
                // plane p - 1 from the elements below and above it
                const double w0 = u0 - t0, w1 = fma(c1, fma(5.0, p1, f1), u1), w2 = fma(c1, fma(5.0, p2, f2), u2),
                             w3 = fma(c1, fma(3.0, p3, f3), u3);
                u0 = t0;
                u1 = c1 * fma(5.0, f1, p1);
                u2 = c1 * fma(5.0, f2, p2);
                u3 = c1 * fma(3.0, f3, p3);
                if (p > z0) {
                    // the face's share of its corners' rows: S -> both, D -> - at 0, + at 1
                    const double lo = w0 - w1, hi = w0 + w1, dl = w2 - w3, dh = w2 + w3;
                    if (t < cells) {
                        double* o = corner + buf + t;
                        o[0] = lo - dl;
                        o[cells] = lo + dl;
                        o[2 * cells] = hi - dh;
                        o[3 * cells] = hi + dh;
                    }
                }
            }
        }
        if (p > z0) {   // output plane p - 1 (z0 .. z1 - 1)
            if (A) __syncthreads();
            if (node) {
                const int64_t row = ((p - 1) * g.ny + gy) * g.nx + gx;
                double ya = 0.0, yb = 0.0;
                if (A) {
                    // as corner 00 of its own face, 10 of the one at x - 1, 01 at y - 1, 11 at both
                    const double* o = corner + buf + t;
                    const int ox = k.cols, oy = fxn * k.cols;
                    ya = (o[0] + o[cells - ox]) + (o[2 * cells - oy] + o[3 * cells - oy - ox]);
                }
                if (B) yb = cb * fma(4.0, m1, m2 + mass);
                if (MODE == Q1_PAIR) {
                    y[row * ldy + col] = ya;
                    o1[row * ld1 + col] = yb;
                } else {
                    const double a = A ? ya : yb;
                    if (MODE == Q1_AXPBY) {
                        y[row * ldy + col] = alpha * a + beta * vprev;
                    } else {
                        if (y) y[row * ldy + col] = a;
                        if (o1) o1[row * ld1 + col] = a - lam[col] * vprev;
                        if (o2) o2[row * ld2 + col] = a - sig * vprev;
                    }
                }
            }
        }
        if (A) { p0 = f0; p1 = f1; p2 = f2; p3 = f3; }
        m2 = m1;
        m1 = mass;
        vprev = v00;
    }
}

Q1Geo q1geo(const Grid& g) { return {g.nx, g.ny, g.nz, g.h, g.cell}; }

// The tile, columns and z segments with the least FP64 time: the warps of a CTA
// times the planes it passes (one more than it puts out) times the rounds of
// CTAs over the SMs.  A face row and column and an element plane are repeated
// per tile, partly filled warps and last rounds cost as much as full ones.
// Candidates: edges whose faces fill whole warps or nearly (16^2, 13^2, 11^2, 9^2,
// 18^2 faces) at 1 to 4 columns.  With edge 15 alone 40^3 x 2 takes 33 us against 25,
// without 17 64^3 x 9 takes 277 against 271; edges 6, 20, 24, 31 win nothing.  Wide
// blocks take 3 or 4 columns (longer runs of memory), few columns make more CTAs
// on small grids: 48 x 40 x 56 x 5 84 us with 3 or 4 only, 68 with 1 to 4; up to 8
// columns win nothing.
Q1Tile q1_tile(const Grid& g, int nc, dim3& grid, int& threads, size_t& smem) {
    auto even = [](int64_t n, int64_t most) {
        const int64_t parts = (n + most - 1) / most;
        return (int)((n + parts - 1) / parts);
    };
    const int64_t sms = sm_count();
    Q1Tile best{};
    double least = 0.0;
    int64_t ctas = 0, segs = 0;
    for (int cmax = nc < 4 ? nc : 4, last = 0; cmax >= 1; --cmax) {
        const int cols = even(nc, cmax);
        if (cols == last) continue;
        last = cols;
        for (int edge : {15, 12, 10, 8, 17}) {
            Q1Tile k;
            k.cols = cols;
            k.chunks = (nc + k.cols - 1) / k.cols;
            k.tx = even(g.nx, edge);
            k.ty = even(g.ny, edge);
            k.ntx = (int)((g.nx + k.tx - 1) / k.tx);
            const int t = (k.tx + 1) * (k.ty + 1) * k.cols;
            if (t > 1024) continue;
            const int64_t n = (int64_t)k.ntx * ((g.ny + k.ty - 1) / k.ty) * k.chunks;
            for (int64_t parts = 1; parts <= 16; ++parts) {
                k.tz = even(g.nz, (g.nz + parts - 1) / parts);
                const int64_t s = (g.nz + k.tz - 1) / k.tz;
                const double cost = (double)((t + 31) / 32) * (k.tz + 1) * (double)((n * s + sms - 1) / sms);
                if (ctas == 0 || cost < least) {
                    least = cost;
                    best = k;
                    ctas = n;
                    segs = s;
                }
                if (k.tz <= 4) break;
            }
        }
    }
    grid = dim3((unsigned)ctas, (unsigned)segs);
    const int cells = (best.tx + 1) * (best.ty + 1) * best.cols;
    threads = (cells + 31) / 32 * 32;
    smem = sizeof(double) * 8 * (size_t)cells;
    return best;
}

template <int MODE, bool A, bool B>
cudaError_t q1_launch(const Grid& g, int nc, double sa, double sb, const double* x, int64_t ldx, double* y, int64_t ldy,
                      double* o1, int64_t ld1, const double* lam, double* o2, int64_t ld2, double alpha, double beta,
                      double sig, cudaStream_t s) {
    if (g.n() * nc == 0) return cudaSuccess;
    dim3 grid;
    int threads;
    size_t smem;
    const Q1Tile k = q1_tile(g, nc, grid, threads, smem);
    if (!A) smem = 0;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k_q1<MODE, A, B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)smem);
        if (e != cudaSuccess) return e;
    }
    // rounded once: they scale every entry of the result
    const long double h = g.h;
    const double ca = (double)(sa * h / 48), cb = (double)(sb * h * h * h / 216);
    k_q1<MODE, A, B><<<grid, threads, smem, s>>>(q1geo(g), k, nc, ca, cb, x, ldx, y, ldy, o1, ld1, lam, o2, ld2, alpha,
                                                 beta, sig);
    count_launches(1);
    return cudaGetLastError();
}

// Bloch Hamiltonian on complex128 blocks: y = 1/2 sum_d (2 x - ph_d x_{+d} - conj(ph_d) x_{-d}) / h^2 + V x
struct BlochGeo {
    int64_t nx, ny, nz;
    double ih2;                 // 1 / h^2
    double cr[3], ci[3];        // e^{i kappa_d h}
    const double* pot;
};

__global__ void __launch_bounds__(256) k_bloch(BlochGeo g, int nc, const double2* __restrict__ x, int64_t ldx,
                                               double2* __restrict__ y, int64_t ldy, int64_t total) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        int64_t row;
        int c;
        split_index(e, nc, row, c);
        const int64_t ix = row % g.nx, t = row / g.nx, iy = t % g.ny, iz = t / g.ny;
        const int64_t n[3] = {g.nx, g.ny, g.nz}, i[3] = {ix, iy, iz}, st[3] = {1, g.nx, g.nx * g.ny};
        const double2 xc = x[row * ldx + c];
        double sr = 0.0, si = 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int64_t up = i[d] < n[d] - 1 ? st[d] : -(n[d] - 1) * st[d];
            const int64_t dn = i[d] > 0 ? -st[d] : (n[d] - 1) * st[d];
            const double2 xp = x[(row + up) * ldx + c], xm = x[(row + dn) * ldx + c];
            // 2 x - ph x_+ - conj(ph) x_-
            sr += 2.0 * xc.x - (g.cr[d] * xp.x - g.ci[d] * xp.y) - (g.cr[d] * xm.x + g.ci[d] * xm.y);
            si += 2.0 * xc.y - (g.cr[d] * xp.y + g.ci[d] * xp.x) - (g.cr[d] * xm.y - g.ci[d] * xm.x);
        }
        const double v = g.pot ? g.pot[row] : 0.0;
        y[row * ldy + c] = make_double2(0.5 * g.ih2 * sr + v * xc.x, 0.5 * g.ih2 * si + v * xc.y);
    }
}

}  // namespace

cudaError_t q1_axpby(const Grid& g, int nc, const double* x, int64_t ldx, double* y, int64_t ldy, double alpha,
                     double beta, cudaStream_t s) {
    return g.q1 == 1 ? q1_launch<Q1_AXPBY, true, false>(g, nc, g.scale, 0.0, x, ldx, y, ldy, nullptr, 0, nullptr,
                                                        nullptr, 0, alpha, beta, 0.0, s)
                     : q1_launch<Q1_AXPBY, false, true>(g, nc, 0.0, g.scale, x, ldx, y, ldy, nullptr, 0, nullptr,
                                                        nullptr, 0, alpha, beta, 0.0, s);
}

cudaError_t q1_apply_shifts(const Grid& g, int nc, const double* x, int64_t ldx, double* ax, int64_t ldax,
                            double* o1, int64_t ld1, const double* lam, double* o2, int64_t ld2, double sig,
                            cudaStream_t s) {
    return g.q1 == 1 ? q1_launch<Q1_SHIFTS, true, false>(g, nc, g.scale, 0.0, x, ldx, ax, ldax, o1, ld1, lam, o2, ld2,
                                                         1.0, 0.0, sig, s)
                     : q1_launch<Q1_SHIFTS, false, true>(g, nc, 0.0, g.scale, x, ldx, ax, ldax, o1, ld1, lam, o2, ld2,
                                                         1.0, 0.0, sig, s);
}

cudaError_t q1_pair(const Grid& A, const Grid& B, int nc, const double* x, int64_t ldx, double* ax, int64_t ldax,
                    double* bx, int64_t ldbx, cudaStream_t s) {
    return q1_launch<Q1_PAIR, true, true>(A, nc, A.scale, B.scale, x, ldx, ax, ldax, bx, ldbx, nullptr, nullptr, 0, 1.0,
                                          0.0, 0.0, s);
}

bool q1_same_mesh(const Grid& A, const Grid& B) {
    return A.q1 == 1 && B.q1 == 2 && A.nx == B.nx && A.ny == B.ny && A.nz == B.nz && A.h == B.h;
}

cudaError_t bloch_apply(const Grid& g, int nc, const double* x, int64_t ldx, double* y, int64_t ldy,
                        cudaStream_t s) {
    const int64_t total = g.n() * nc;
    if (total == 0) return cudaSuccess;
    BlochGeo b;
    b.nx = g.nx; b.ny = g.ny; b.nz = g.nz;
    b.ih2 = 1.0 / (g.h * g.h);
    for (int d = 0; d < 3; ++d) {
        b.cr[d] = std::cos(g.kappa[d] * g.h);
        b.ci[d] = std::sin(g.kappa[d] * g.h);
    }
    b.pot = g.pot;
    const int blocks = grid_size_for(total, 256, sm_count() * 16);
    k_bloch<<<blocks, 256, 0, s>>>(b, nc, reinterpret_cast<const double2*>(x), ldx, reinterpret_cast<double2*>(y),
                                   ldy, total);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace plhr
