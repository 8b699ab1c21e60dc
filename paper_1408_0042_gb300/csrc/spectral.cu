// Teter-Payne-Allan preconditioner (Section 5.3: a positive diagonal matrix
// in the plane-wave basis) on a tensor grid, FP64:
//     T = S diag(K(mu / E)) S^T,
//     K(x) = (27 + 18x + 12x^2 + 8x^3) / (27 + 18x + 12x^2 + 8x^3 + 16x^4),
// with S = Sx (x) Sy (x) Sz the orthonormal eigenvectors of the grid's kinetic
// operator -1/2 Lap_h (real Fourier modes on a periodic axis, sine modes on a
// Dirichlet axis), mu = mu_x + mu_y + mu_z their kinetic energies and E one
// fixed reference energy.  T is symmetric positive definite and commutes with
// -1/2 Lap_h.
//
// Application: forward transforms along x and y, then along z forward, the
// factor (a precomputed per-mode table) and back in one kernel, then the inverse
// transforms along y and x; double-word values (hi + lo FP32 pairs, ~48-bit
// significands) between the passes, FP64 at both ends.  GB300 issues FP64 at
// 1/64 of the FP32 rate, so a double-word multiply-add (13 FP32 instructions)
// costs about a fifth of an FP64 one.
//
// Every mode of an axis is even or odd under a reflection of the points (p to
// N - p of a periodic axis, p to N - 1 - p of a Dirichlet one), and on a
// periodic axis of even N also under p to N / 2 - p.  Folding the points by
// these reflections (sums and differences) leaves a dense product per parity
// class: two of about (N / 2)^2, or four of (N / 4)^2, multiply-adds per line
// instead of N^2.  N = 64 periodic: 1026 instead of 4096.  The multiply-adds
// bound the passes before (116-128 us each at 64^3 x 10, six passes and a
// conversion: 715 us); now 38-46 us, 77 us for the fused pass along z: 240 us.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "dword.h"
#include "plhr_internal.h"

namespace plhr {
namespace {

constexpr int kT = 256;
constexpr int kMaxAxis = 144;

// One axis: parity classes c of np[c] folded points and as many modes.  Folded
// point i of class c sits at position base[c] + step[c] i of the folded line;
// its modes at first[c] .. of the coefficient line.  Class matrices [np][ld]
// (ld = np rounded up to 4, zero padding) start at entry mat[c].
struct AxisPlan {
    int N, classes, two;   // two: second reflection used
    int periodic;
    int nE;                // folded positions 0 .. nE - 1: even under the first reflection
    int np[4], base[4], step[4], first[4], mat[4];
    int mat_size;          // entries of all class matrices
    int groups;            // groups of 4 outputs over all classes
    int group0[4];         // first group of a class
};

struct AxisPass {
    AxisPlan pl;
    int64_t nx, ny;        // grid (lines of axis x, y, z)
    int axis;
    int64_t stride;        // point stride along the axis
    int nc;
    int64_t elems;         // lines x columns
};

double tpa(double x) {
    const double num = 27.0 + x * (18.0 + x * (12.0 + 8.0 * x));
    const double x2 = x * x;
    return num / (num + 16.0 * x2 * x2);
}

// first point of line l along the axis (lines of axis x: (y, z) rows; of
// axis y: (x, z) with x fastest; of axis z: (x, y) with x fastest, so that
// consecutive lines are neighbours in memory)
__device__ __forceinline__ int64_t line_base(const AxisPass& a, int64_t l) {
    if (a.axis == 0) return l * a.nx;
    if (a.axis == 1) return (l / a.nx) * a.nx * a.ny + l % a.nx;
    return l;
}

// partner of point p under the first reflection (p itself when fixed)
__device__ __forceinline__ int mirror(const AxisPlan& pl, int p) {
    if (!pl.periodic) return pl.N - 1 - p;
    return p == 0 ? 0 : pl.N - p;
}
// folded position of the odd combination of p and its partner
__device__ __forceinline__ int odd_pos(const AxisPlan& pl, int p) { return pl.nE + (pl.periodic ? p - 1 : p); }

__device__ __forceinline__ int class_of_group(const AxisPlan& pl, int g) {
    int c = 0;
    while (c + 1 < pl.classes && g >= pl.group0[c + 1]) ++c;
    return c;
}

constexpr int kQ = 4;   // outputs per thread (register block)
// (line, column) elements per tile: one warp wide, so that the matrix reads are
// broadcasts; small tiles keep five CTAs on an SM (64 elements: 285 us per
// application at 64^3 x 10, 32: 240 us)
constexpr int kTile = 32;

// out[q] (q < 4) = sum_j M[j][q] in[(base + step j) kTile], j < n (M rows ld apart)
__device__ __forceinline__ void dot4(dw* v, const dw* M, int ld, const dw* in, int base, int step, int n) {
    float hi[kQ], lo[kQ];
#pragma unroll
    for (int u = 0; u < kQ; ++u) { hi[u] = 0.0f; lo[u] = 0.0f; }
    const dw* x = in + base * kTile;
    for (int j = 0; j < n; ++j, x += step * kTile, M += ld) {
        const dw xv = *x;
        const float4 m01 = *reinterpret_cast<const float4*>(M), m23 = *reinterpret_cast<const float4*>(M + 2);
        dw_fma_acc(hi[0], lo[0], dw{m01.x, m01.y}, xv);
        dw_fma_acc(hi[1], lo[1], dw{m01.z, m01.w}, xv);
        dw_fma_acc(hi[2], lo[2], dw{m23.x, m23.y}, xv);
        dw_fma_acc(hi[3], lo[3], dw{m23.z, m23.w}, xv);
    }
#pragma unroll
    for (int u = 0; u < kQ; ++u) v[u] = dw_fast_two_sum(hi[u], lo[u]);
}

enum { AX_FWD = 0, AX_INV = 1, AX_BOTH = 2 };

// One pass along an axis.  AX_FWD: coefficients of the lines (times the factor K
// of the mode when given); AX_INV: the lines of coefficients; AX_BOTH: forward,
// times K, inverse.
// A tile is 32 (line, column) elements, all N points; Tin / Tout: FP64 (leading
// dimensions ldi, ldo) or double-word (dense, leading dimension nc).  M:
// class matrices [point][mode] for the forward product, Mt: [mode][point] for
// the inverse.
template <int MODE, typename Tin, typename Tout>
__global__ void __launch_bounds__(kT) k_axis(const __grid_constant__ AxisPass a, const dw* __restrict__ M,
                                             const dw* __restrict__ Mt, const Tin* in, int64_t ldi, Tout* out,
                                             int64_t ldo, const dw* __restrict__ K) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const AxisPlan& pl = a.pl;
    const int N = pl.N, nE = pl.nE;
    constexpr int W = kTile;
    dw* sm = reinterpret_cast<dw*>(smraw);                         // matrices of the products this pass takes
    dw* A = sm + (MODE == AX_BOTH ? 2 : 1) * pl.mat_size;          // [N][W]
    dw* B = A + N * W;                                             // [N][W], unless AX_FWD
    int64_t* pin = reinterpret_cast<int64_t*>(MODE == AX_FWD ? B : B + N * W);   // [W] input offsets of point 0
    int64_t* pout = pin + W;
    int64_t* ppt = pout + W;
    for (int i = threadIdx.x; i < pl.mat_size; i += kT) {
        sm[i] = MODE == AX_INV ? Mt[i] : M[i];
        if (MODE == AX_BOTH) sm[pl.mat_size + i] = Mt[i];
    }
    auto load = [&](int64_t at) -> dw {
        if constexpr (std::is_same_v<Tin, double>) return dw_from_double_fast(in[at]);
        else return in[at];
    };
    auto store = [&](int64_t at, dw v) {
        if constexpr (std::is_same_v<Tout, double>) out[at] = dw_to_double_fast(v);
        else out[at] = v;
    };
    const int64_t si = a.stride * ldi, so = a.stride * ldo;
    for (int64_t e0 = (int64_t)blockIdx.x * W; e0 < a.elems; e0 += (int64_t)gridDim.x * W) {
        const int we = (int)(a.elems - e0 < W ? a.elems - e0 : W);
        __syncthreads();   // the previous tile is consumed (and the matrices are staged)
        for (int e = threadIdx.x; e < we; e += kT) {
            const int64_t l = (e0 + e) / a.nc;
            const int c = (int)((e0 + e) - l * a.nc);
            const int64_t pt = line_base(a, l);
            pin[e] = pt * ldi + c;
            pout[e] = pt * ldo + c;
            ppt[e] = pt;
        }
        __syncthreads();
        if (MODE == AX_INV) {
            for (int t = threadIdx.x; t < N * W; t += kT) {
                const int p = t / W, e = t % W;
                if (e < we) A[t] = load(pin[e] + p * si);
            }
            __syncthreads();
        } else {
            // load and fold by the first reflection: the even part at p, the odd part behind
            // (p = 0 .. nE - 1 are the points not past their partners)
            for (int t = threadIdx.x; t < nE * W; t += kT) {
                const int p = t / W, e = t % W;
                if (e >= we) continue;
                const int m = mirror(pl, p);
                const dw x = load(pin[e] + p * si);
                if (m == p) {
                    A[t] = x;
                } else {
                    const dw y = load(pin[e] + m * si);
                    A[t] = dw_add(x, y);
                    A[odd_pos(pl, p) * W + e] = dw_sub(x, y);
                }
            }
            __syncthreads();
            if (pl.two) {
                // by the second one, in both parts: sums at the front, differences at the back
                const int nO = N - nE, hE = nE / 2, hO = nO / 2;
                for (int t = threadIdx.x; t < (hE + hO) * W; t += kT) {
                    const int i = t / W, e = t % W;
                    const int p = i < hE ? i : nE + i - hE, m = i < hE ? nE - 1 - i : N - 1 - (i - hE);
                    const dw x = A[p * W + e], y = A[m * W + e];
                    A[p * W + e] = dw_add(x, y);
                    A[m * W + e] = dw_sub(x, y);
                }
                __syncthreads();
            }
        }
        // the class products: 4 outputs per thread
        dw v[kQ];
        if (MODE != AX_INV) {
            for (int t = threadIdx.x; t < pl.groups * W; t += kT) {
                const int g = t / W, e = t % W;
                if (e >= we) continue;
                const int c = class_of_group(pl, g), q0 = (g - pl.group0[c]) * kQ;
                const int n = pl.np[c], ld = (n + 3) & ~3;
                dot4(v, sm + pl.mat[c] + q0, ld, A + e, pl.base[c], pl.step[c], n);
#pragma unroll
                for (int u = 0; u < kQ; ++u) {
                    if (q0 + u >= n) break;
                    const int m = pl.first[c] + q0 + u;
                    const dw f = K ? dw_mul(v[u], K[ppt[e] + m * a.stride]) : v[u];
                    if (MODE == AX_BOTH) B[m * W + e] = f;
                    else store(pout[e] + m * so, f);
                }
            }
            if (MODE == AX_FWD) continue;
            __syncthreads();
        }
        // inverse: coefficients in src, folded points to dst, unfolded on the way out
        const dw* src = MODE == AX_BOTH ? B : A;
        dw* dst = MODE == AX_BOTH ? A : B;
        const dw* mt = MODE == AX_BOTH ? sm + pl.mat_size : sm;
        for (int t = threadIdx.x; t < pl.groups * W; t += kT) {
            const int g = t / W, e = t % W;
            if (e >= we) continue;
            const int c = class_of_group(pl, g), q0 = (g - pl.group0[c]) * kQ;
            const int n = pl.np[c], ld = (n + 3) & ~3;
            dot4(v, mt + pl.mat[c] + q0, ld, src + e, pl.first[c], 1, n);
#pragma unroll
            for (int u = 0; u < kQ; ++u)
                if (q0 + u < n) dst[(pl.base[c] + pl.step[c] * (q0 + u)) * W + e] = v[u];
        }
        __syncthreads();
        if (pl.two) {
            const int nO = N - nE, hE = nE / 2, hO = nO / 2;
            for (int t = threadIdx.x; t < (hE + hO) * W; t += kT) {
                const int i = t / W, e = t % W;
                const int p = i < hE ? i : nE + i - hE, m = i < hE ? nE - 1 - i : N - 1 - (i - hE);
                const dw x = dst[p * W + e], y = dst[m * W + e];
                dst[p * W + e] = dw_add(x, y);
                dst[m * W + e] = dw_sub(x, y);
            }
            __syncthreads();
        }
        for (int t = threadIdx.x; t < nE * W; t += kT) {
            const int p = t / W, e = t % W;
            if (e >= we) continue;
            const int m = mirror(pl, p);
            const dw x = dst[t];
            if (m == p) {
                store(pout[e] + p * so, x);
            } else {
                const dw y = dst[odd_pos(pl, p) * W + e];
                store(pout[e] + p * so, dw_add(x, y));
                store(pout[e] + m * so, dw_sub(x, y));
            }
        }
    }
}

constexpr int kAxisShm = 200 * 1024;

// shared memory of one pass
size_t axis_smem(const AxisPlan& pl, int mode) {
    return sizeof(dw) * ((mode == AX_BOTH ? 2 : 1) * (size_t)pl.mat_size +
                         (mode == AX_FWD ? 1 : 2) * (size_t)pl.N * kTile) + 3 * sizeof(int64_t) * (size_t)kTile;
}

// orthonormal eigenvectors S[p][m] and eigenvalues mu (times 1/2 scale of the
// kinetic operator folded in by the caller) of the 1D second difference
void axis_basis(int64_t N, bool periodic, std::vector<double>& S, std::vector<double>& mu) {
    S.assign(N * N, 0.0);
    mu.assign(N, 0.0);
    if (!periodic) {
        for (int64_t m = 0; m < N; ++m) {
            const double th = (m + 1) * M_PI / (N + 1);
            mu[m] = 2.0 - 2.0 * std::cos(th);
            for (int64_t p = 0; p < N; ++p) S[p * N + m] = std::sqrt(2.0 / (N + 1)) * std::sin((p + 1) * th);
        }
        return;
    }
    // real Fourier modes: constant; cos and sin of frequency f = 1 .. (N-1)/2;
    // the alternating mode when N is even
    int64_t col = 0;
    for (int64_t p = 0; p < N; ++p) S[p * N + col] = 1.0 / std::sqrt((double)N);
    mu[col++] = 0.0;
    for (int64_t f = 1; 2 * f < N; ++f) {
        const double th = 2.0 * M_PI * f / N;
        for (int64_t p = 0; p < N; ++p) {
            S[p * N + col] = std::sqrt(2.0 / N) * std::cos(th * p);
            S[p * N + col + 1] = std::sqrt(2.0 / N) * std::sin(th * p);
        }
        mu[col] = mu[col + 1] = 2.0 - 2.0 * std::cos(th);
        col += 2;
    }
    if (N % 2 == 0) {
        for (int64_t p = 0; p < N; ++p) S[p * N + col] = (p % 2 ? -1.0 : 1.0) / std::sqrt((double)N);
        mu[col++] = 4.0;
    }
}

// The plan of an axis, and the mode order of its coefficient lines: order[m] is
// the column of axis_basis's S.
AxisPlan axis_plan(int64_t N, bool periodic, std::vector<int>& order) {
    AxisPlan pl{};
    pl.N = (int)N;
    pl.periodic = periodic ? 1 : 0;
    pl.nE = periodic ? (int)(N / 2 + 1) : (int)((N + 1) / 2);
    pl.two = periodic && N % 2 == 0 && N >= 4;
    const int nO = pl.N - pl.nE;
    std::vector<int> modes[4];
    if (!periodic) {
        for (int m = 0; m < N; ++m) modes[m & 1].push_back(m);       // even m: symmetric about the middle
    } else {
        // columns of S: constant, then cos f, sin f for f = 1 .. (N - 1) / 2, then the alternating one
        auto even = [&](int f) { return f == 0 ? 0 : 2 * f == N ? (int)N - 1 : 2 * f - 1; };
        for (int f = 0; f < pl.nE; ++f) modes[pl.two ? (f & 1) : 0].push_back(even(f));
        for (int f = 1; f <= nO; ++f) modes[pl.two ? 2 + !(f & 1) : 1].push_back(2 * f);
    }
    const int ends[4][3] = {   // base, step, points of the two-reflection classes
        {0, 1, (pl.nE + 1) / 2}, {pl.nE - 1, -1, pl.nE / 2}, {pl.nE, 1, (nO + 1) / 2}, {pl.N - 1, -1, nO / 2}};
    order.clear();
    int mat = 0, group = 0;
    for (int c = 0; c < (pl.two ? 4 : 2); ++c) {
        const int n = (int)modes[c].size();
        if (n == 0) continue;
        const int k = pl.classes++;
        pl.np[k] = n;
        pl.base[k] = pl.two ? ends[c][0] : c == 0 ? 0 : pl.nE;
        pl.step[k] = pl.two ? ends[c][1] : 1;
        pl.first[k] = (int)order.size();
        pl.mat[k] = mat;
        pl.group0[k] = group;
        mat += n * ((n + 3) & ~3);
        group += (n + 3) / 4;
        order.insert(order.end(), modes[c].begin(), modes[c].end());
    }
    pl.mat_size = mat;
    pl.groups = group;
    return pl;
}

// point of the line that folded point i of class k stands for
int plan_point(const AxisPlan& pl, int k, int i) {
    const int pos = pl.base[k] + pl.step[k] * i;
    // differences of the second reflection are kept at the partner's position
    const int at = pl.step[k] > 0 ? pos : pos < pl.nE ? pl.nE - 1 - pos : pl.nE + pl.N - 1 - pos;
    return at < pl.nE ? at : at - pl.nE + pl.periodic;
}

}  // namespace

int64_t spectral_workspace_doubles(const SpecPrec& P, int nc) { return 2 * P.n() * nc; }

cudaError_t spectral_apply(const SpecPrec& P, int nc, const double* r, int64_t ldr, double* w, double* work,
                           cudaStream_t s) {
    if (nc <= 0) return cudaSuccess;
    const int64_t n = P.n();
    dw* t0 = reinterpret_cast<dw*>(work);
    dw* t1 = t0 + n * nc;
    const int64_t Ns[3] = {P.nx, P.ny, P.nz};
    const int64_t strides[3] = {1, P.nx, P.nx * P.ny};
    const dw* K = reinterpret_cast<const dw*>(P.d_K);
    for (int ax = 0; ax < P.d; ++ax)   // the documented limit of axis size and columns
        if ((int64_t)sizeof(dw) * (Ns[ax] * Ns[ax] + Ns[ax] * nc) > kAxisShm) return cudaErrorInvalidValue;
    auto pass = [&](auto mode, int ax, const auto* in, int64_t ldi, auto* out, int64_t ldo,
                    const dw* K) -> cudaError_t {
        constexpr int MODE = decltype(mode)::value;
        using Tin = std::remove_const_t<std::remove_pointer_t<decltype(in)>>;
        using Tout = std::remove_pointer_t<decltype(out)>;
        std::vector<int> order;
        AxisPass a;
        a.pl = axis_plan(Ns[ax], P.periodic, order);
        a.nx = P.nx;
        a.ny = P.ny;
        a.axis = ax;
        a.stride = strides[ax];
        a.nc = nc;
        a.elems = n / Ns[ax] * nc;
        const size_t shm = axis_smem(a.pl, MODE);
        cudaError_t e = cudaFuncSetAttribute(k_axis<MODE, Tin, Tout>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kAxisShm);
        if (e != cudaSuccess) return e;
        const int blocks = (int)std::min<int64_t>((a.elems + kTile - 1) / kTile, (int64_t)sm_count() * 16);
        k_axis<MODE, Tin, Tout><<<blocks, kT, shm, s>>>(a, reinterpret_cast<const dw*>(P.d_S[ax]),
                                                        reinterpret_cast<const dw*>(P.d_St[ax]), in, ldi, out, ldo, K);
        count_launches(1);
        return cudaGetLastError();
    };
    const std::integral_constant<int, AX_FWD> fwd;
    const std::integral_constant<int, AX_INV> inv;
    const std::integral_constant<int, AX_BOTH> both;
    const int last = P.d - 1;
    cudaError_t e = pass(fwd, 0, r, ldr, t0, nc, nullptr);
    if (e == cudaSuccess && P.d == 3) {
        e = pass(fwd, 1, (const dw*)t0, nc, t1, nc, nullptr);
        std::swap(t0, t1);
    }
    // the last axis forward, factor, inverse, in place (a CTA owns its tile's
    // lines); in two passes where the matrices of both directions do not fit
    // (Dirichlet axes from 130 points)
    std::vector<int> order;
    if (e == cudaSuccess && axis_smem(axis_plan(Ns[last], P.periodic, order), AX_BOTH) <= (size_t)kAxisShm) {
        e = pass(both, last, (const dw*)t0, nc, t0, nc, K);
    } else if (e == cudaSuccess) {
        e = pass(fwd, last, (const dw*)t0, nc, t0, nc, K);
        if (e == cudaSuccess) e = pass(inv, last, (const dw*)t0, nc, t0, nc, nullptr);
    }
    if (e == cudaSuccess && P.d == 3) {
        e = pass(inv, 1, (const dw*)t0, nc, t1, nc, nullptr);
        std::swap(t0, t1);
    }
    if (e == cudaSuccess) e = pass(inv, 0, (const dw*)t0, nc, w, nc, nullptr);
    return e;
}

}  // namespace plhr

using namespace plhr;

extern "C" plhr_status plhr_prec_tpa(plhr_prec** out, const plhr_op* A, double sigma, double energy) {
    clear_error();
    if (!out || !A || !std::isfinite(sigma) || !std::isfinite(energy)) {
        set_error("plhr_prec_tpa: invalid argument");
        return PLHR_EINVAL;
    }
    const Grid& g = A->g;
    if (g.csr) {
        set_error("plhr_prec_tpa: A must be a stencil or Hamiltonian operator (not CSR)");
        return PLHR_EINVAL;
    }
    const int64_t Ns[3] = {g.nx, g.ny, g.d == 3 ? g.nz : 1};
    for (int a = 0; a < g.d; ++a)
        if (Ns[a] > kMaxAxis) {
            set_error("plhr_prec_tpa: axis size %lld exceeds %d", (long long)Ns[a], kMaxAxis);
            return PLHR_EINVAL;
        }
    if (!(energy > 0)) {
        // sigma - min V, or the mean kinetic energy of the grid's modes d / h^2
        double vmin = 0.0;
        if (g.pot) {
            std::vector<double> hv(g.n());
            if (cudaMemcpy(hv.data(), g.pot, sizeof(double) * g.n(), cudaMemcpyDeviceToHost) != cudaSuccess) {
                set_error("plhr_prec_tpa: reading the potential failed");
                return PLHR_ECUDA;
            }
            vmin = hv[0];
            for (double v : hv) vmin = std::fmin(vmin, v);
        }
        energy = sigma - vmin;
        if (!(energy > 0)) energy = g.d * 2.0 * g.inv_h2();   // d / h^2 for the scale 1/2
    }
    plhr_prec* T = new plhr_prec;
    T->kind = PREC_TPA;
    SpecPrec& P = T->sp;
    P.d = g.d;
    P.nx = Ns[0]; P.ny = Ns[1]; P.nz = Ns[2];
    P.energy = energy;
    // double-word (hi, lo) pairs of FP64 values
    auto pairs = [](const std::vector<double>& v) {
        std::vector<float> w(2 * v.size());
        for (size_t i = 0; i < v.size(); ++i) {
            w[2 * i] = (float)v[i];
            w[2 * i + 1] = (float)(v[i] - (double)w[2 * i]);
        }
        return w;
    };
    auto upload = [&](float** dst, const std::vector<float>& src) {
        return cudaMalloc(dst, sizeof(float) * src.size()) == cudaSuccess &&
               cudaMemcpy(*dst, src.data(), sizeof(float) * src.size(), cudaMemcpyHostToDevice) == cudaSuccess;
    };
    P.periodic = g.periodic != 0;
    std::vector<double> mus[3];   // in the order of the coefficient lines
    for (int a = 0; a < 3; ++a) mus[a].assign(1, 0.0);
    for (int a = 0; a < g.d; ++a) {
        const int64_t N = Ns[a];
        std::vector<double> S, mu;
        std::vector<int> order;
        axis_basis(N, P.periodic, S, mu);
        const AxisPlan pl = axis_plan(N, P.periodic, order);
        mus[a].resize(N);
        for (int64_t m = 0; m < N; ++m) mus[a][m] = mu[order[m]] * g.inv_h2();   // the kinetic operator's eigenvalues
        std::vector<double> M(pl.mat_size, 0.0), Mt(pl.mat_size, 0.0);
        for (int c = 0; c < pl.classes; ++c) {
            const int n = pl.np[c], ld = (n + 3) & ~3;
            for (int i = 0; i < n; ++i)
                for (int q = 0; q < n; ++q) {
                    const double v = S[plan_point(pl, c, i) * N + order[pl.first[c] + q]];
                    M[pl.mat[c] + i * ld + q] = v;
                    Mt[pl.mat[c] + q * ld + i] = v;
                }
        }
        if (!upload(&P.d_S[a], pairs(M)) || !upload(&P.d_St[a], pairs(Mt))) {
            set_error("plhr_prec_tpa: device allocation or upload failed");
            plhr_prec_destroy(T);
            return PLHR_ENOMEM;
        }
    }
    // the factor per 3D mode, x fastest
    std::vector<double> Kf(P.n());
    for (int64_t iz = 0; iz < P.nz; ++iz)
        for (int64_t iy = 0; iy < P.ny; ++iy)
            for (int64_t ix = 0; ix < P.nx; ++ix)
                Kf[(iz * P.ny + iy) * P.nx + ix] =
                    tpa((mus[0][ix] + mus[1][iy] + (g.d == 3 ? mus[2][iz] : 0.0)) / energy);
    if (!upload(&P.d_K, pairs(Kf))) {
        set_error("plhr_prec_tpa: device allocation or upload failed");
        plhr_prec_destroy(T);
        return PLHR_ENOMEM;
    }
    *out = T;
    return PLHR_OK;
}

extern "C" double plhr_prec_tpa_energy(const plhr_prec* T) {
    return (T && T->kind == PREC_TPA) ? T->sp.energy : 0.0;
}
