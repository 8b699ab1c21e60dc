// Small dense stage of one PLHR iteration on the device (no host round trip).  Input: the raw Grams of the trial basis
// Z = [V W S P] (Z*Z, U*Q with U = AZ - sigma Z, Q*Z, Q = T U) and the column
// scales of Z.  Steps:
//  1. B-orthonormalisation of Z (Alg. 2 step 6) done implicitly: with the
//     column-scaled Gram D Z*Z D = R^T R (Cholesky, columns whose pivot^2 falls
//     below 1e-12 are dropped), Z-hat = Z D R^{-1} is B-orthonormal and spans
//     [V], [V W], [V W S], [V W S P] blockwise, as the paper's blockwise
//     procedure does.
//  2. Projected T-harmonic problem (Eq. THarm_evp) in the Z-hat basis:
//     G_L = sym(R^-T D U*Q D R^-1), G_R = R^-T D Q*Z D R^-1; through tau = 1/xi
//     (Eq. THarm_evp_sinv): G_L = L L^T, C = L^-1 G_R L^-T, eigenpairs (tau, z)
//     of C, y = L^-T z.
//  3. Eigenvalues of C: Householder reduction to Hessenberg form and the
//     Francis double-shift QR iteration, eigenvalues only (Golub & Van Loan,
//     "Matrix Computations", Sec. 7.4-7.5); eigenvectors of the selected ones by
//     inverse iteration on the Hessenberg form.
//  4. Order by |xi| with each complex xi followed by its conjugate, select k'
//     (Alg. 3 steps 7-10), rotate complex y so Re(y) is orthogonal to Im(y)
//     and the longer of the two, build the real Y' = [Y0 YR yR~ YI].
//  5. Coefficients on the raw basis: P_new = Z C_P, V_new = V C_VV + P_new.
#include "dense.h"
#include "dword.h"

#include <cooperative_groups.h>

#include <cfloat>
#include <mutex>

namespace plhr {
namespace {

constexpr int MAXM = kDenseMaxM;
constexpr int LDS = MAXM + 1;     // shared row stride: column accesses hit distinct banks
constexpr int NT = 512;           // threads of a k_pencil CTA

__device__ __forceinline__ void wsync() { __syncwarp(); }
__device__ __forceinline__ void bsync() { __syncthreads(); }

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// ---------------------------------------------------------------- warp Cholesky (final Rayleigh-Ritz)
// plain Cholesky A = L L^T by one warp (lower stored in A's lower triangle)
__device__ bool chol_lower(double* A, int n, int ld) {
    const int lane = threadIdx.x & 31;
    bool ok = true;
    for (int j = 0; j < n; ++j) {
        double p = A[j * ld + j];
        if (!(p > 0.0) || !isfinite(p)) { ok = false; break; }
        double r = sqrt(p);
        wsync();
        for (int l = j + 1 + lane; l < n; l += 32) A[l * ld + j] /= r;
        wsync();
        if (lane == 0) A[j * ld + j] = r;
        for (int idx = lane; idx < (n - j - 1) * (n - j - 1); idx += 32) {
            int a = j + 1 + idx / (n - j - 1), b = j + 1 + idx % (n - j - 1);
            if (b <= a) A[a * ld + b] -= A[a * ld + j] * A[b * ld + j];
        }
        wsync();
    }
    wsync();
    return ok;
}

// ---------------------------------------------------------------- block-wide dense kernels
// r = sqrt(p) and ri = 1 / r, p > 0: an FP32 estimate and two Goldschmidt
// iterations on p scaled by an even power of two, one Newton correction of the
// root (P. Markstein, "Software division and square root using Goldschmidt's
// algorithms", RNC 2004).  Eight dependent FP64 operations for both, where an FP64
// warp instruction takes 64 cycles of its pipe.
__device__ __forceinline__ void sqrt_and_inverse(double p, double& r, double& ri) {
    const int hi = __double2hiint(p);
    if (hi < 0x00100000) {   // subnormal
        r = sqrt(p);
        ri = 1.0 / r;
        return;
    }
    const int e = ((hi >> 20) - 1023) & ~1;
    const double m = __hiloint2double(hi - (e << 20), __double2loint(p));   // in [1, 4)
    const float y = rsqrtf((float)m);
    double g = m * (double)y, h = (double)(0.5f * y);
    for (int i = 0; i < 2; ++i) {
        const double d = fma(-g, h, 0.5);
        g = fma(g, d, g);
        h = fma(h, d, h);
    }
    g = fma(fma(-g, g, m), h, g);
    r = __hiloint2double(__double2hiint(g) + ((e / 2) << 20), __double2loint(g));
    ri = __hiloint2double(__double2hiint(h) + ((1 - e / 2) << 20), __double2loint(h));
}

// Cholesky A = R^T R of a symmetric n x n (upper triangle used and replaced).
// With keep, column j is dropped when its pivot is below tol (the matrix is
// column-normalised, so the test is relative); without, a pivot that is not
// above tol ends it (false).  Warps 0 and 1, on two sub-partitions, bring row
// j + 1 up to date, form its pivot's root and scale it (a product and a correction
// with the remainder instead of a division an entry) while the warps of the other
// two sub-partitions update the rows below with row j: a column is the longer of a
// chain of about 14 FP64 operations and the update, and one barrier (64 columns
// with the Gram's normalisation: 291,000 -> 133,000 cycles).
__device__ bool bchol(double* A, int n, int* keep, double tol) {
    __shared__ int stop[2];   // by parity: a thread may read its entry while the next is written
    const int tid = threadIdx.x, warp = tid >> 5;
    const int ut = (warp >> 2) * 64 + (warp & 1) * 32 + (tid & 31);   // of warps 2, 3 mod 4
    if (tid < 2) stop[tid] = 0;
    bsync();
    double root = 0.0;   // thread 0: the last row's diagonal entry, written one barrier later
    for (int j = -1; j < n; ++j) {
        if (tid < 64) {
            if (tid == 0 && j >= 0) A[j * LDS + j] = root;
            const int i = j + 1, l = i + tid;
            if (i < n) {
                const double f = j >= 0 ? A[j * LDS + i] : 0.0;
                const double p = fma(-f, f, A[i * LDS + i]);
                const bool ok = (p > tol) && isfinite(p);
                double v = 0.0;
                if (l < n) v = fma(-f, j >= 0 ? A[j * LDS + l] : 0.0, A[i * LDS + l]);
                root = 0.0;
                if (ok) {
                    double ri;
                    sqrt_and_inverse(p, root, ri);
                    const double q = v * ri;
                    v = fma(fma(-q, root, v), ri, q);
                } else {
                    v = 0.0;
                }
                if (tid > 0 && l < n) A[i * LDS + l] = v;
                if (tid == 0) {
                    if (keep) keep[i] = ok ? 1 : 0;
                    else if (!ok) stop[i & 1] = 1;
                }
            }
        } else if ((warp & 3) >= 2 && j >= 0) {
            for (int a = j + 2 + (ut >> 4); a < n; a += NT / 32) {
                const double f = A[j * LDS + a];
                for (int b = a + (ut & 15); b < n; b += 16) A[a * LDS + b] = fma(-f, A[j * LDS + b], A[a * LDS + b]);
            }
        }
        bsync();
        if (stop[(j + 1) & 1]) return false;
    }
    return true;
}

// Solves T x = b for a lower triangular T by one warp: b0, b1 are rows lane and
// lane + 32 of b, then of x.  Tc[l * LDS + i] = T_il / T_ll (i > l), rinv_l = 1 / T_ll:
// each unknown, unscaled, is subtracted from the rows below at once, one FP64
// operation deep, and the scaling comes last.
__device__ __forceinline__ void warp_solve(const double* Tc, const double* rinv, int n, double& b0, double& b1) {
    const int lane = threadIdx.x & 31;
    const int n0 = n < 32 ? n : 32;
    for (int l = 0; l < n0; ++l) {
        const double x = __shfl_sync(0xffffffffu, b0, l);
        const double* t = Tc + l * LDS;
        if (lane > l && lane < n) b0 = fma(-t[lane], x, b0);
        if (lane + 32 < n) b1 = fma(-t[lane + 32], x, b1);
    }
    for (int l = 32; l < n; ++l) {
        const double x = __shfl_sync(0xffffffffu, b1, l - 32);
        if (lane + 32 > l && lane + 32 < n) b1 = fma(-Tc[l * LDS + lane + 32], x, b1);
    }
    if (lane < n) b0 *= rinv[lane];
    if (lane + 32 < n) b1 *= rinv[lane + 32];
}

// Householder reduction of H (n x n) to upper Hessenberg form.  The reflector
// of step k, I - beta_k v v^T with v = (0,..,0, v_{k+1}, .., v_{n-1}), is kept
// in row k of Vh and beta[k] (beta = 0: identity).
//
// The reduction runs in double-word arithmetic on H scaled by a power of two
// to unit norm: its transformations are orthogonal, so it is as accurate as
// the double-word QR iteration that follows it, and the FP64 form (one
// dependent FP64 chain per column, each warp instruction holding the FP64 pipe
// for 64 cycles) cost about a million cycles at n = 64.  Every column and row
// belongs to eight threads that split its sum over i (lazily normalised
// double-word sums, combined by three shuffles); columns c and c + 8 share a half
// warp, so that its 16 accesses (odd stride) fall into distinct banks.  One warp
// forms the reflector's scalars.  Four warps a scheduler hide each other's
// dependent operations (two threads a column, one warp a scheduler: 522,000 ->
// 378,000 cycles at n = 64).  v and beta describe the same reflector at any
// scale, so only H is scaled back; H, Vh and beta are FP64 again on return.
__device__ void bhessenberg(double* Hd, double* Vhd, double* betad, int n, double* red) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const dw zero = dw_make(0.0f);
    double an = 0.0;
    for (int i = tid; i < n * n; i += NT) an = fmax(an, fabs(Hd[(i / n) * LDS + i % n]));
    an = warp_max(an);
    if (lane == 0) red[warp] = an;
    bsync();
    for (int w = 0; w < NT / 32; ++w) an = fmax(an, red[w]);
    bsync();
    const int ex = an > 0.0 ? ilogb(an) : 0;
    const double down = ldexp(1.0, -ex), up = ldexp(1.0, ex);
    dw* H = reinterpret_cast<dw*>(Hd);
    dw* V = reinterpret_cast<dw*>(Vhd);
    dw* B = reinterpret_cast<dw*>(betad);
    for (int i = tid; i < n * n; i += NT) {
        const int r = i / n, c = i % n;
        H[r * LDS + c] = dw_from_double_fast(Hd[r * LDS + c] * down);
    }
    bsync();
    float* redf = reinterpret_cast<float*>(red);
    const int part = lane & 7, own = (warp & 7) + 8 * (lane >> 3) + 32 * (warp >> 3);
    auto sum8 = [](dw v) {
        for (int o = 1; o < 8; o <<= 1)
            v = dw_add(v, dw{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
        return v;
    };
    for (int k = 0; k < n - 2; ++k) {
        // warp 0: ||x||^2 for x = H[k+1:n, k], beta and v_{k+1}
        if (warp == 0) {
            dwacc acc = {0.0f, 0.0f};
            for (int i = k + 1 + lane; i < n; i += 32) {
                const dw x = H[i * LDS + k];
                dwacc_add_mul(acc, x, x);
            }
            dw ss = dwacc_result(acc);
            for (int o = 16; o > 0; o >>= 1)
                ss = dw_add(ss, dw{__shfl_xor_sync(0xffffffffu, ss.hi, o), __shfl_xor_sync(0xffffffffu, ss.lo, o)});
            const dw x0 = H[(k + 1) * LDS + k];
            dw alpha = dw_sqrt(ss);
            if (x0.hi > 0.0f) alpha = dw_neg(alpha);
            // v_{k+1} = x0 - alpha, v^T v = 2 (ss - x0 alpha) (alpha^2 = ss, no
            // cancellation: -x0 alpha >= 0), beta = 2 / v^T v
            const dw den = dw_sub(ss, dw_mul(x0, alpha));
            const bool none = dw_is_zero(alpha) || !(den.hi > 0.0f);
            if (lane == 0) {
                const dw b = none ? zero : dw_div(dw_make(1.0f), den), v0 = dw_sub(x0, alpha);
                redf[0] = b.hi; redf[1] = b.lo;
                redf[2] = v0.hi; redf[3] = v0.lo;
                redf[4] = none ? 1.0f : 0.0f;
                B[k] = b;
            }
        }
        bsync();
        const dw b = {redf[0], redf[1]};
        const bool skip = redf[4] != 0.0f;
        if (tid < n)
            V[k * LDS + tid] = (tid <= k || skip) ? zero : (tid == k + 1 ? dw{redf[2], redf[3]} : H[tid * LDS + k]);
        bsync();
        if (!skip) {
            const dw* v = V + k * LDS;
            // H <- (I - b v v^T) H : column c = own (columns below k are zero in rows > k)
            {
                const int c = own;
                const bool act = c < n && c >= k;
                dwacc acc = {0.0f, 0.0f};
                if (act)
                    for (int i = k + 1 + part; i < n; i += 8) dwacc_add_mul(acc, v[i], H[i * LDS + c]);
                const dw sv = dw_neg(dw_mul(sum8(dwacc_result(acc)), b));
                if (act)
                    for (int i = k + 1 + part; i < n; i += 8) {
                        dwacc h = dwacc_of(H[i * LDS + c]);
                        dwacc_add_mul(h, sv, v[i]);
                        H[i * LDS + c] = dwacc_result(h);
                    }
            }
            bsync();
            // H <- H (I - b v v^T) : row r = own
            {
                const int r = own;
                const bool act = r < n;
                dwacc acc = {0.0f, 0.0f};
                if (act)
                    for (int i = k + 1 + part; i < n; i += 8) dwacc_add_mul(acc, H[r * LDS + i], v[i]);
                const dw sv = dw_neg(dw_mul(sum8(dwacc_result(acc)), b));
                if (act)
                    for (int i = k + 1 + part; i < n; i += 8) {
                        dwacc h = dwacc_of(H[r * LDS + i]);
                        dwacc_add_mul(h, sv, v[i]);
                        H[r * LDS + i] = dwacc_result(h);
                    }
            }
            // column k below its subdiagonal entry is zero now; no row update reads it
            for (int i = k + 2 + tid; i < n; i += NT) H[i * LDS + k] = zero;
        }
        bsync();
    }
    // back to FP64 (each entry converted in place by the thread that reads it)
    for (int i = tid; i < n * n; i += NT) {
        const int r = i / n, c = i % n;
        Hd[r * LDS + c] = dw_to_double(H[r * LDS + c]) * up;
    }
    for (int i = tid; i < (n - 2) * n; i += NT) {
        const int r = i / n, c = i % n;
        Vhd[r * LDS + c] = dw_to_double(V[r * LDS + c]);
    }
    for (int i = tid; i < n - 2; i += NT) betad[i] = dw_to_double(B[i]);
    bsync();
}

// ---------------------------------------------------------------- eigenvalues (three warps)
// Householder vector for (x, y, z) in double-word arithmetic: u = (1, u1, u2),
// tau and beta with (I - tau u u^T)(x, y, z)^T = (beta, 0, 0)^T.
//
// This is the longest part of a bulge step's dependent chain (double-word sums
// are ten FP32 operations deep), so it is written with as few of them as the
// accuracy allows: the squares are summed unnormalised, the square root and
// the two reciprocals take one correction from FP32 and one from the
// double-word remainder (their leading parts are correctly rounded after the
// first, so the differences in the second are exact), and the reciprocal of
// |x| + ||.|| starts from the FP32 norm, beside the norm's own corrections.
// Relative errors stay below 2^-44 as with the general operations.
__device__ __forceinline__ dw recip_refine(dw w, float r) {   // 1 / w, r its FP32 approximation
    const float e = __fmaf_rn(-w.lo, r, __fmaf_rn(-w.hi, r, 1.0f));
    dw q = dw_fast_two_sum(r, __fmul_rn(e, r));
    const float p = __fmul_rn(w.hi, q.hi), pe = __fmaf_rn(w.hi, q.hi, -p);
    const float t = __fmaf_rn(-w.lo, q.hi, __fmaf_rn(-w.hi, q.lo, -pe));
    return dw_fast_two_sum(q.hi, __fmaf_rn(__fadd_rn(__fsub_rn(1.0f, p), t), r, q.lo));
}
__device__ __forceinline__ void house3(dw x, dw y, dw z, dw& u1, dw& u2, dw& tau, dw& beta) {
    const dw zero = dw_make(0.0f);
    if (dw_is_zero(y) && dw_is_zero(z)) {
        u1 = zero; u2 = zero; tau = zero; beta = x;
        return;
    }
    // u and tau do not depend on the scale of (x, y, z): bring the largest to
    // about 1 by a power of two (exact) so that the squares stay inside FP32's
    // exponent range
    const float mx = fmaxf(fabsf(x.hi), fmaxf(fabsf(y.hi), fabsf(z.hi)));
    const float sc = pow2_inverse_of(mx);
    const float sg = x.hi > 0.0f ? 1.0f : -1.0f;
    x = dw_mul_pow2(x, __fmul_rn(sc, sg));   // |x|
    y = dw_mul_pow2(y, sc);
    z = dw_mul_pow2(z, sc);
    const dw px = dw_two_prod(x.hi, x.hi), py = dw_two_prod(y.hi, y.hi), pz = dw_two_prod(z.hi, z.hi);
    const float lx = __fmaf_rn(2.0f * x.hi, x.lo, px.lo), ly = __fmaf_rn(2.0f * y.hi, y.lo, py.lo),
                lz = __fmaf_rn(2.0f * z.hi, z.lo, pz.lo);
    const dw s1 = dw_two_sum(px.hi, py.hi), s2 = dw_two_sum(s1.hi, pz.hi);
    const dw ss = dw_fast_two_sum(s2.hi, __fadd_rn(__fadd_rn(lx, ly), __fadd_rn(__fadd_rn(s1.lo, lz), s2.lo)));
    // norm
    const float rs = rsqrtf(ss.hi), hr = 0.5f * rs;
    const float f = __fmul_rn(ss.hi, rs);
    const float rw = __fdividef(1.0f, __fadd_rn(x.hi, f));
    dw nrm = dw_fast_two_sum(f, __fmul_rn(__fadd_rn(__fmaf_rn(-f, f, ss.hi), ss.lo), hr));
    {
        const float p = __fmul_rn(nrm.hi, nrm.hi), pe = __fmaf_rn(nrm.hi, nrm.hi, -p);
        const float t = __fsub_rn(__fmaf_rn(-2.0f * nrm.hi, nrm.lo, ss.lo), pe);
        nrm = dw_fast_two_sum(nrm.hi, __fmaf_rn(__fadd_rn(__fsub_rn(ss.hi, p), t), hr, nrm.lo));
    }
    // w = |x| + norm; u = sg (y, z) / w, tau = w / norm, beta = -sg norm
    const dw h = dw_fast_two_sum(nrm.hi, x.hi);
    const dw w = dw_fast_two_sum(h.hi, __fadd_rn(__fadd_rn(nrm.lo, x.lo), h.lo));
    const dw rv = recip_refine(w, rw);
    const dw rn = recip_refine(nrm, rs);
    const dw srv = dw_mul_pow2(rv, sg);
    u1 = dw_mul(y, srv);
    u2 = dw_mul(z, srv);
    // w / norm = 1 + |x| / norm: the error of the quotient counts half at most, and the
    // product w (1 / norm) cost a tenth of the eigenvalues' accuracy (mean error at m = 64
    // 9.1e-14, 7.2e-14 now, 8.4e-14 with general operations; the same time)
    const dw q = dw_two_prod(x.hi, rn.hi), t = dw_fast_two_sum(1.0f, q.hi);
    tau = dw_fast_two_sum(t.hi, __fadd_rn(t.lo, __fadd_rn(q.lo, __fmaf_rn(x.hi, rn.lo, __fmul_rn(x.lo, rn.hi)))));
    beta = dw_mul_pow2(nrm, __fmul_rn(-sg, pow2_inverse_of(sc)));   // sc is a power of two
}

// (a0 + u1 a1 + u2 a2) tau: the leading parts by error-free sums and products,
// everything below them in FP32, not normalised (its use, reflected, is a lazily
// normalised sum)
__device__ __forceinline__ dw house_dot(dw a0, dw a1, dw a2, dw u1, dw u2, dw tau) {
    const dw p = dw_two_prod(u1.hi, a1.hi), q = dw_two_prod(u2.hi, a2.hi);
    const float lp = __fmaf_rn(u1.hi, a1.lo, __fmaf_rn(u1.lo, a1.hi, p.lo));
    const float lq = __fmaf_rn(u2.hi, a2.lo, __fmaf_rn(u2.lo, a2.hi, q.lo));
    const dw s = dw_two_sum(p.hi, q.hi), v = dw_two_sum(s.hi, a0.hi);
    const float lo = __fadd_rn(__fadd_rn(__fadd_rn(lp, lq), __fadd_rn(s.lo, a0.lo)), v.lo);
    const dw r = dw_two_prod(v.hi, tau.hi);
    return {r.hi, __fadd_rn(r.lo, __fmaf_rn(lo, tau.hi, __fmul_rn(v.hi, tau.lo)))};
}
// a - s u
__device__ __forceinline__ dw reflected(dw a, dw u, dw s) {
    dwacc v = dwacc_of(a);
    dwacc_add_mul(v, dw_neg(s), u);
    return dwacc_result(v);
}
// which ? a : b as two select instructions: a ternary on a value that differs from
// lane to lane became a branch, with what follows it once per side
__device__ __forceinline__ dw dw_select(bool which, dw a, dw b) {
    dw r;
    asm("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %6, 0;\n\tselp.f32 %0, %2, %4, p;\n\tselp.f32 %1, %3, %5, p;\n\t}"
        : "=f"(r.hi), "=f"(r.lo)
        : "f"(a.hi), "f"(a.lo), "f"(b.hi), "f"(b.lo), "r"((int)which));
    return r;
}
// named barriers between the two roles of the iteration: a side that only
// announces arrives, the other waits
template <int ID>
__device__ __forceinline__ void role_arrive() { asm volatile("bar.arrive %0, 96;" ::"n"(ID) : "memory"); }
template <int ID>
__device__ __forceinline__ void role_wait() { asm volatile("bar.sync %0, 96;" ::"n"(ID) : "memory"); }

// Francis double-shift QR (Golub & Van Loan Sec. 7.5) on the upper Hessenberg
// H, eigenvalues only: every transformation is applied to the active window
// rows/columns l..hi alone (no Schur vectors, no full Schur form), which is
// all the eigenvalues need.  Deflated 1x1 and 2x2 diagonal blocks remain.
//
// A step's reflector depends on the one before through the 4 x 4 block at the
// bulge only, so warp 0 chases the bulge alone: it forms the reflector, applies
// it to the block's columns, then to its rows and to the column that enters the
// block next (an entry per lane, warp barriers), and reads the next reflector's
// column.  Two more warps apply the reflector to the remaining columns (left) and
// rows (right, disjoint from them) while warp 0 forms the next one.  A step costs
// the chain reflector - left - right on one entry: 980 cycles against 1370
// with all threads in step, a column and then a row each.
//
// The iteration runs in double-word arithmetic on H scaled by a power of two to
// unit norm (H is converted in place: a double and a double-word value take the
// same 8 bytes) and is converted back at the end.  Returns false if the iteration
// does not converge; sweeps (optional) gets the number of QR sweeps and of bulge
// steps.
constexpr int kFrancisThreads = 96;   // the named barriers' count
enum { BAR_REFLECTOR = 1, BAR_APPLIED = 2 };
constexpr int kFrancisRows = MAXM + 4;   // rows of H in shared memory
static_assert(kFrancisThreads >= MAXM, "one column / row per thread");

__device__ __forceinline__ bool francis_eigenvalues(double* Hd, int n, long long* sweeps) {
    __shared__ double red[kFrancisThreads / 32];
    __shared__ int last[kFrancisThreads / 32];
    __shared__ dw refl[2][3];
    const int t = threadIdx.x;
    double anorm = 0.0;
    for (int i = t; i < n * n; i += kFrancisThreads) {
        int r = i / n, c = i % n;
        if (c >= r - 1) anorm = fmax(anorm, fabs(Hd[r * LDS + c]));
    }
    anorm = warp_max(anorm);
    if ((t & 31) == 0) red[t >> 5] = anorm;
    __syncthreads();
    for (int w = 0; w < kFrancisThreads / 32; ++w) anorm = fmax(anorm, red[w]);
    const int ex = anorm > 0.0 ? ilogb(anorm) : 0;
    const double down = ldexp(1.0, -ex), up = ldexp(1.0, ex);
    dw* H = reinterpret_cast<dw*>(Hd);
    for (int i = t; i < n * n; i += kFrancisThreads) {
        int r = i / n, c = i % n;
        double v = (c >= r - 1) ? Hd[r * LDS + c] * down : 0.0;
        H[r * LDS + c] = dw_from_double(v);
    }
    // what the bulge's loads reach beyond the matrix
    for (int i = t; i < kFrancisRows * LDS; i += kFrancisThreads)
        if (i >= n * LDS || i % LDS >= n) H[i] = dw_make(0.0f);
    __syncthreads();
    // negligible subdiagonal: relative to the neighbouring diagonal, or to
    // ||H|| (= 1 to 2 after scaling; normwise backward stable).  Only the
    // eigenvalues of largest modulus are used, and they keep full relative
    // accuracy; the normwise test lets the many eigenvalues near zero deflate
    // quickly.  eps is a few units of the double-word precision.
    const float eps = 0x1p-46f;
    const float hnorm = 1.0f;
    const dw zero = dw_make(0.0f), one = dw_make(1.0f);
    bool ok = true;
    int hi = n - 1;
    int its = 0, total_its = 0, total_steps = 0;
    while (hi >= 0) {
        // l = the last row at or above hi whose subdiagonal entry is negligible
        // (row 0 always is), found by all threads at once
        {
            bool small = t == 0;
            if (t > 0 && t <= hi) {
                float s = fabsf(H[(t - 1) * LDS + t - 1].hi) + fabsf(H[t * LDS + t].hi);
                if (s < hnorm) s = hnorm;
                small = fabsf(H[t * LDS + t - 1].hi) <= eps * s;
            }
            const unsigned b = __ballot_sync(0xffffffffu, small);
            if ((t & 31) == 0) last[t >> 5] = b ? (t & ~31) + 31 - __clz(b) : 0;
        }
        __syncthreads();
        int l = 0;
        for (int w = 0; w < kFrancisThreads / 32; ++w) l = max(l, last[w]);
        if (l > 0 && t == 0) H[l * LDS + l - 1] = zero;
        __syncthreads();
        if (l >= hi - 1) {          // 1x1 or 2x2 block converged
            hi = l - 1;
            its = 0;
            continue;
        }
        if (its >= 40) {
            // a stalled window holds a (near-)defective cluster of numerically
            // equal eigenvalues, which converges only linearly; deflate at the
            // smallest subdiagonal when it is below 1e-7 ||H|| (the eigenvalues
            // move by about that much; only a basis of the cluster is needed)
            int jm = l + 1;
            float vm = fabsf(H[(l + 1) * LDS + l].hi);
            for (int j = l + 2; j <= hi; ++j) {
                float v = fabsf(H[j * LDS + j - 1].hi);
                if (v < vm) { vm = v; jm = j; }
            }
            if (vm <= 1e-7f * hnorm) {
                __syncthreads();
                if (t == 0) H[jm * LDS + jm - 1] = zero;
                __syncthreads();
                its = 0;
                continue;
            }
        }
        if (++total_its > 100 * n) { ok = false; break; }
        ++its;
        total_steps += hi - l;
        dw s, tt;
        if (its % 10 == 0) {
            dw w = dw_add(dw_make(fabsf(H[hi * LDS + hi - 1].hi)), dw_make(fabsf(H[(hi - 1) * LDS + hi - 2].hi)));
            s = dw_mul_f(w, 1.5f);
            tt = dw_mul(w, w);
        } else {
            dw a = H[(hi - 1) * LDS + hi - 1], b = H[(hi - 1) * LDS + hi], c = H[hi * LDS + hi - 1],
               d = H[hi * LDS + hi];
            s = dw_add(a, d);
            tt = dw_sub(dw_mul(a, d), dw_mul(b, c));
        }
        dw h00 = H[l * LDS + l], h01 = H[l * LDS + l + 1], h10 = H[(l + 1) * LDS + l],
           h11 = H[(l + 1) * LDS + l + 1], h21 = H[(l + 2) * LDS + l + 1];
        // first column of (H - s1 I)(H - s2 I)
        dw x = dw_add(dw_add(dw_mul(h00, dw_sub(h00, s)), dw_mul(h01, h10)), tt);
        dw y = dw_mul(h10, dw_sub(dw_add(h00, h11), s));
        dw z = dw_mul(h10, h21);
        // every thread has read the shift and the first bulge column before
        // any thread writes
        __syncthreads();
        if (t >= 32) {
            // reflector k: columns k + 5.. (left), rows ..k - 1 (right); thread q has
            // column hi - q, then row l + 63 - q (never both: hi - l <= 63)
            const int q = t - 32, col = hi - q, row = l + 63 - q;
            for (int k = l; k < hi; ++k) {
                role_wait<BAR_REFLECTOR>();
                const bool left = col >= k + 5;
                if (left || row < k) {
                    dw* h = H + (left ? k * LDS + col : row * LDS + k);
                    const int step = left ? LDS : 1;
                    const dw u1 = refl[k & 1][0], u2 = refl[k & 1][1], tau = refl[k & 1][2];
                    const dw a0 = h[0], a1 = h[step], a2 = h[2 * step];
                    const dw sa = house_dot(a0, a1, a2, u1, u2, tau);
                    h[0] = reflected(a0, one, sa);
                    h[step] = reflected(a1, u1, sa);
                    if (k < hi - 1) h[2 * step] = reflected(a2, u2, sa);
                }
                if (k < hi - 1) role_arrive<BAR_APPLIED>();
            }
        } else {
            // lanes 0..11: entry e of column, then row k + c of the block; lanes 12..14
            // store column k - 1, (beta, 0, 0), then take row k + e of column k + 4;
            // lanes 16..18 store the reflector.  Every lane loads (the rest of the
            // last rows is zero or finite, and is not stored), so that nothing but the
            // stores is conditional.
            const int c = t & 3, e = t < 12 ? t >> 2 : c;
            const bool block = t < 12, edge = t >= 12 && t < 15;
            const dw* from = H + l * LDS + l + c;
            dw* to = H + (block ? (l + e) * LDS + l + c : (l + e) * LDS + l - 1);
            dw* rows = H + (block ? (l + c) * LDS + l : l * LDS + l + 4);
            const int step = block ? 1 : LDS;
            for (int k = l; k < hi; ++k) {
                // rows (columns) k..k+2, the last step's k and k+1 with u2 = 0
                const bool three = k < hi - 1, entry = e < 2 || (e == 2 && three), in = k + c <= hi;
                const dw a0 = from[0], a1 = from[LDS], a2 = from[2 * LDS];
                const dw ae = dw_select(e == 0, a0, dw_select(e == 1, a1, a2));
                dw u1, u2, tau, beta;
                house3(x, y, three ? z : zero, u1, u2, tau, beta);
                const dw ue = dw_select(e == 0, one, dw_select(e == 1, u1, u2));
                const dw va = dw_select(block, reflected(ae, ue, house_dot(a0, a1, a2, u1, u2, tau)),
                                        dw_select(t == 12, beta, zero));
                __syncwarp();
                if (entry && (block ? in : edge && k > l)) *to = va;
                if (t >= 16 && t < 19) refl[k & 1][c] = dw_select(c == 0, u1, dw_select(c == 1, u2, tau));
                // the other warps have applied the earlier reflectors to column k + 4
                if (k > l) role_wait<BAR_APPLIED>();
                else __syncwarp();
                const dw b0 = rows[0], b1 = rows[step], b2 = rows[2 * step];
                const dw be = dw_select(e == 0, b0, dw_select(e == 1, b1, b2));
                const dw vb = reflected(be, ue, house_dot(b0, b1, b2, u1, u2, tau));
                __syncwarp();
                if (entry && (block ? in : edge && k + 4 <= hi)) rows[e * step] = vb;
                role_arrive<BAR_REFLECTOR>();
                __syncwarp();
                x = H[(k + 1) * LDS + k];
                y = H[(k + 2) * LDS + k];
                z = H[(k + 3) * LDS + k];
                from += LDS + 1;
                to += LDS + 1;
                rows += LDS + 1;
            }
        }
        __syncthreads();
    }
    __syncthreads();
    for (int i = t; i < n * n; i += kFrancisThreads) {
        int r = i / n, c = i % n;
        dw v = H[r * LDS + c];
        Hd[r * LDS + c] = (c >= r - 1) ? dw_to_double(v) * up : 0.0;
    }
    if (sweeps && t == 0) { sweeps[0] = total_its; sweeps[1] = total_steps; }
    __syncthreads();
    return ok;
}

// ---------------------------------------------------------------- eigenvectors (one warp each)
// Complex double-word arithmetic for the per-unit eigenvector work: each
// step of a triangular factorisation or solve is a short serial chain, and
// on GB300 an FP64 warp instruction holds the FP64 pipe for 64 cycles, so
// the chains run several times faster on the FP32 pipes in double-word form
// (~48-bit significands, the accuracy of the QR iteration that supplies the
// shifts).  The operands are scaled by a power of two to unit norm first so
// that they stay inside FP32's exponent range.
struct cdw {
    dw re, im;
};
// (products and sums as lazily normalised sums: half the depth of the pairwise ones)
__device__ __forceinline__ cdw cdw_fma(cdw c, cdw a, cdw b) {   // c + a b
    dwacc r = dwacc_of(c.re), i = dwacc_of(c.im);
    dwacc_add_mul(r, a.re, b.re);
    dwacc_add_mul(r, dw_neg(a.im), b.im);
    dwacc_add_mul(i, a.re, b.im);
    dwacc_add_mul(i, a.im, b.re);
    return {dwacc_result(r), dwacc_result(i)};
}
__device__ __forceinline__ cdw cdw_zero() { return {dw_make(0.0f), dw_make(0.0f)}; }
__device__ __forceinline__ cdw cdw_mul(cdw a, cdw b) { return cdw_fma(cdw_zero(), a, b); }
__device__ __forceinline__ cdw cdw_neg(cdw a) { return {dw_neg(a.re), dw_neg(a.im)}; }
__device__ __forceinline__ dw dw_fma(dw c, dw a, dw b) {   // c + a b
    dwacc r = dwacc_of(c);
    dwacc_add_mul(r, a, b);
    return dwacc_result(r);
}
__device__ __forceinline__ float cdw_abs1(cdw a) { return fabsf(a.re.hi) + fabsf(a.im.hi); }
// 1 / b, the denominator scaled by a power of two first (no under- or overflow)
__device__ __forceinline__ cdw cdw_recip(cdw b) {
    const float sc = pow2_inverse_of(fmaxf(fabsf(b.re.hi), fabsf(b.im.hi)));
    const dw r = dw_mul_pow2(b.re, sc), i = dw_mul_pow2(b.im, sc);
    const dw den = dw_fma(dw_fma(dw_make(0.0f), r, r), i, i);
    const dw inv = recip_refine(den, __fdividef(1.0f, den.hi));
    return {dw_mul_pow2(dw_mul(r, inv), sc), dw_mul_pow2(dw_neg(dw_mul(i, inv)), sc)};
}
__device__ __forceinline__ dw dw_shfl(dw v, int lane) {
    return {__shfl_sync(0xffffffffu, v.hi, lane), __shfl_sync(0xffffffffu, v.lo, lane)};
}
__device__ __forceinline__ cdw cdw_shfl(cdw v, int lane) { return {dw_shfl(v.re, lane), dw_shfl(v.im, lane)}; }

// A vector or matrix row over a warp: entries lane and lane + 32
struct cdw2 {
    cdw v[2];
    __device__ __forceinline__ cdw at(int j) const { return cdw_shfl(j >= 32 ? v[1] : v[0], j & 31); }
};

// Inverse iteration on the Hessenberg H (n x n, unit norm) for the eigenvalue lam
// by one warp: (H - lam I) is factored once by Gaussian elimination with
// adjacent-row pivoting (keeps the Hessenberg structure; multipliers, swaps, the
// upper factor U and the reciprocals of its pivots kept), then two solves starting
// from b = 1, each normalised to max |x_i| = 1.  The row being eliminated and the
// vector stay in registers; U and the multipliers go to shared memory.
// Column-oriented back substitution: one reciprocal multiply on the critical path
// per step, the updates in parallel.
__device__ cdw2 inverse_iteration(const dw* H, int n, cdw lam, cdw* U, cdw* mult, cdw* rpiv, cdw* xs, int* swp,
                                  float tiny) {
    const int lane = threadIdx.x & 31;
    cdw2 cur, nxt;
    for (int q = 0; q < 2; ++q) {
        const int j = lane + 32 * q;
        cur.v[q] = {j < n ? H[j] : dw_make(0.0f), dw_make(0.0f)};
        if (j == 0) cur.v[q] = {dw_sub(cur.v[q].re, lam.re), dw_neg(lam.im)};
    }
    for (int k = 0; k < n; ++k) {
        cdw piv = cur.at(k);
        if (k < n - 1) {
            for (int q = 0; q < 2; ++q) {
                const int j = lane + 32 * q;
                nxt.v[q] = {j >= k && j < n ? H[(k + 1) * LDS + j] : dw_make(0.0f), dw_make(0.0f)};
                if (j == k + 1) nxt.v[q] = {dw_sub(nxt.v[q].re, lam.re), dw_neg(lam.im)};
            }
        }
        cdw low = {k < n - 1 ? H[(k + 1) * LDS + k] : dw_make(0.0f), dw_make(0.0f)};
        const bool swap = k < n - 1 && cdw_abs1(low) > cdw_abs1(piv);
        if (swap) {
            const cdw2 t = cur;
            cur = nxt;
            nxt = t;
            const cdw u = piv;
            piv = low;
            low = u;
        }
        if (cdw_abs1(piv) < tiny) piv = {dw_make(tiny), dw_make(0.0f)};
        const cdw rp = cdw_recip(piv), f = cdw_mul(low, rp), nf = cdw_neg(f);
        for (int q = 0; q < 2; ++q) {
            const int j = lane + 32 * q;
            if (j < n && j >= k) U[k * LDS + j] = j == k ? piv : cur.v[q];
            cur.v[q] = cdw_fma(nxt.v[q], nf, cur.v[q]);   // the next row (columns above k)
        }
        if (lane == 0) { mult[k] = nf; rpiv[k] = rp; swp[k] = swap ? 1 : 0; }
    }
    cdw2 x;
    x.v[0] = x.v[1] = {dw_make(1.0f), dw_make(0.0f)};
    wsync();
    for (int iter = 0; iter < 2; ++iter) {
        // forward: the recorded row swaps and eliminations applied to b = x, one
        // chain that every lane follows
        for (int q = 0; q < 2; ++q)
            if (lane + 32 * q < n) xs[lane + 32 * q] = x.v[q];
        wsync();
        cdw top = xs[0];
        for (int k = 0; k < n - 1; ++k) {
            const cdw nf = mult[k];
            cdw next = xs[k + 1];
            if (swp[k]) {
                const cdw t = top;
                top = next;
                next = t;
            }
            if (k == lane) x.v[0] = top;
            if (k == lane + 32) x.v[1] = top;
            top = cdw_fma(next, nf, top);
        }
        if (n - 1 == lane) x.v[0] = top;
        if (n - 1 == lane + 32) x.v[1] = top;
        // backward: x_i = b_i / U_ii, then b_j -= U_ji x_i for j < i
        for (int i = n - 1; i >= 0; --i) {
            const cdw xi = cdw_mul(x.at(i), rpiv[i]), ni = cdw_neg(xi);
            if (lane < i) x.v[0] = cdw_fma(x.v[0], U[lane * LDS + i], ni);
            if (i > 32) {
                if (lane + 32 < i) x.v[1] = cdw_fma(x.v[1], U[(lane + 32) * LDS + i], ni);
            }
            if (lane == i) x.v[0] = xi;
            if (lane + 32 == i) x.v[1] = xi;
        }
        // normalise to max |x_i| = 1 (scale by a power of two, then exactly)
        float mx = 0.0f;
        for (int q = 0; q < 2; ++q)
            if (lane + 32 * q < n) mx = fmaxf(mx, cdw_abs1(x.v[q]));
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float sc = (mx > 0.0f && isfinite(mx)) ? pow2_inverse_of(mx) : 1.0f;
        for (int q = 0; q < 2; ++q) x.v[q] = {dw_mul_pow2(x.v[q].re, sc), dw_mul_pow2(x.v[q].im, sc)};
        wsync();
    }
    return x;
}

// sum over the warp, lazily normalised
__device__ __forceinline__ dw warp_sum_dw(dwacc v) {
    for (int o = 16; o > 0; o >>= 1) {
        const float h = __shfl_xor_sync(0xffffffffu, v.hi, o), l = __shfl_xor_sync(0xffffffffu, v.lo, o);
        const dw t = dw_two_sum(v.hi, h);
        v = {t.hi, __fadd_rn(t.lo, __fadd_rn(v.lo, l))};
    }
    return dwacc_result(v);
}

// ---------------------------------------------------------------- the state between the launches
struct DenseState {
    double H[MAXM * LDS];     // G_R, then C
    double H0[MAXM * LDS];    // Hessenberg form of C
    double Vh[MAXM * LDS];    // Householder vectors of the Hessenberg reduction
    double A[MAXM * LDS];     // R (upper), the Cholesky factor of the kept columns' Gram
    double B[MAXM * LDS];     // G_L -> L
    double beta[MAXM];
    double t[MAXM];           // column normalisation of the (scaled) basis
    int kidx[MAXM];           // kept -> raw index
    double eig_re[MAXM], eig_im[MAXM];
    int order[MAXM];          // selected units: eigenvalue index
    int kind[MAXM];           // 0 real, 2 full pair, 1 cut pair
    int nclose[MAXM];         // earlier selected units in the same numerical cluster
    int ints[8];              // [0] kept columns, [1] of V, [3] selected units, [6] stop, [7] pencil's verdict
};

// Yre, Yim (MAXM^2 each), then the saved state
constexpr int MAXKP = 16;
constexpr size_t kWorkMainDoubles = 2 * (size_t)MAXM * MAXM;
constexpr size_t kDenseWorkDoubles = kWorkMainDoubles + (sizeof(DenseState) + sizeof(double) - 1) / sizeof(double);

__device__ __forceinline__ DenseState* state_of(const DenseArgs& a) {
    return reinterpret_cast<DenseState*>(a.work + kWorkMainDoubles);
}

// The dense stage runs as four launches: k_pencil (up to the Hessenberg form,
// state saved to global scratch), k_francis (three warps: the eigenvalues and the
// selection), k_eigvec and k_finish (one CTA per selected unit each: the
// eigenvector; cluster orthogonalisation, Y' and the coefficients of the unit's
// columns).  The eigenvalue iteration measured 2x slower per bulge step when run
// inside the large kernel than as its own launch on the same data and code.
//
// k_pencil is one cluster of kPencilCtas CTAs.  The first does the serial parts
// (the two Cholesky factorisations, the Hessenberg form); the triangular solves,
// one warp per column and then per row, are spread over all of them, since 512 solves
// of 64 unknowns are half a million FP64 multiply-adds, 258,000 cycles of one SM's
// FP64 pipe (both congruences 588,000 -> 109,000 cycles).  Blocks pass between the
// CTAs through the global state; what another CTA wrote is read past L1.
constexpr int kPencilCtas = 8;
struct PencilShm {
    double A[MAXM * LDS];    // column-normalised B-Gram, then G_L, and their factors
    double T[MAXM * LDS];    // columns of a triangular factor over its diagonal
    double H[MAXM * LDS];
    double Vh[MAXM * LDS];
    double beta[MAXM], t[MAXM], rinv[MAXM], red[NT / 32];
    int keep[MAXM], kidx[MAXM];
};

// S.T, S.rinv from a factor in global memory: T_il at f[l * LDS + i] (upper, T = R^T)
// or f[i * LDS + l] (lower)
__device__ __forceinline__ void load_factor(PencilShm& S, const double* f, bool upper, int n) {
    bsync();
    for (int i = threadIdx.x; i < n; i += NT) S.rinv[i] = 1.0 / __ldcg(f + i * LDS + i);
    bsync();
    for (int e = threadIdx.x; e < n * n; e += NT) {
        const int l = e / n, i = e - l * n;
        if (i > l) S.T[l * LDS + i] = __ldcg(f + (upper ? l * LDS + i : i * LDS + l)) * S.rinv[l];
    }
    bsync();
}

__global__ void __cluster_dims__(kPencilCtas, 1, 1) __launch_bounds__(NT) k_pencil(DenseArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PencilShm& S = *reinterpret_cast<PencilShm*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31;
    const int m = a.m, kp = a.kp;
    const bool lead = blockIdx.x == 0;
    const int solver = blockIdx.x * (NT / 32) + (tid >> 5);   // 2 MAXM warps of the cluster
    static_assert(kPencilCtas * (NT / 32) == 2 * MAXM, "one warp per column of two blocks");
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    DenseState* G = state_of(a);
    int nk = 0;
#define STAMP(i) do { if (a.clk && lead && tid == 0) a.clk[i] = clock64(); } while (0)
    STAMP(0);
    // ---- 1. B-orthonormalisation of Z, implicitly: Cholesky with column
    // dropping of the column-normalised Gram (the Grams are of Z diag(colscale)).
    // The basis Z D R^{-1} amplifies Gram rounding by cond(R)^2; if G_L then is
    // not numerically positive definite the pass is repeated with a stricter
    // drop threshold.
    if (lead) {
        for (int i = tid; i < m; i += NT) {
            const double g = a.Gzz[i * m + i];
            S.t[i] = (g > 0.0 && isfinite(g)) ? 1.0 / sqrt(g) : 0.0;
            G->t[i] = S.t[i];
        }
    }
    bsync();
    const double drop_tols[3] = {1e-12, 1e-9, 1e-6};
    enum { PENCIL_OK = 0, PENCIL_AGAIN = 1, PENCIL_STOP = 2 };
    int next = PENCIL_AGAIN;
    for (int attempt = 0; attempt < 3 && next == PENCIL_AGAIN; ++attempt) {
        if (lead) {
            for (int i = tid; i < m * m; i += NT) {
                const int r = i / m, c = i % m;
                S.A[r * LDS + c] = a.Gzz[i] * S.t[r] * S.t[c];
            }
            bsync();
            bchol(S.A, m, S.keep, drop_tols[attempt]);
            STAMP(11);
            if (tid == 0) {
                int q = 0, qv = 0;
                for (int j = 0; j < m; ++j)
                    if (S.keep[j] && S.t[j] != 0.0) {
                        S.kidx[q] = j;
                        G->kidx[q++] = j;
                        if (j < a.nv) ++qv;
                    }
                G->ints[0] = q;
                G->ints[1] = qv;
                const bool loss = qv < 1 || q < kp;
                if (loss) { a.out_int[0] = kDenseRankLoss; a.out_int[1] = q; a.out_int[2] = 0; }
                G->ints[6] = loss ? 1 : 0;
                S.keep[0] = q;
            }
            bsync();
            nk = S.keep[0];
            // compact R (upper)
            for (int i = tid; i < nk * nk; i += NT) {
                const int r = i / nk, c = i % nk;
                G->A[r * LDS + c] = (c >= r) ? S.A[S.kidx[r] * LDS + S.kidx[c]] : 0.0;
            }
        }
        STAMP(12);
        cluster.sync();
        nk = __ldcg(&G->ints[0]);
        if (__ldcg(&G->ints[6])) {
            next = PENCIL_STOP;
            break;
        }
        // ---- 2. the pencil in the B-orthonormal basis, via tau = 1/xi: G_L =
        // sym(U^T Q), G_R[r][c] = q_r . z_c on the kept, normalised columns, by
        // columns R^{-T} X, then by rows X R^{-1}
        load_factor(S, G->A, true, nk);
        {
            const int c = solver & (MAXM - 1);
            const bool gl = solver < MAXM;
            double* X = gl ? G->B : G->H;
            double b0 = 0.0, b1 = 0.0;
            if (c < nk) {
                const int cc = __ldcg(&G->kidx[c]);
                const double tc = __ldcg(&G->t[cc]);
                for (int half = 0; half < 2; ++half) {
                    const int r = lane + 32 * half;
                    if (r >= nk) break;
                    const int rr = __ldcg(&G->kidx[r]);
                    const double v = gl ? 0.5 * (a.Guq[rr * m + cc] + a.Guq[cc * m + rr]) : a.Gqz[rr * m + cc];
                    (half ? b1 : b0) = v * __ldcg(&G->t[rr]) * tc;
                }
                warp_solve(S.T, S.rinv, nk, b0, b1);
                if (lane < nk) X[lane * LDS + c] = b0;
                if (lane + 32 < nk) X[(lane + 32) * LDS + c] = b1;
            }
            cluster.sync();
            if (c < nk) {
                double* x = X + c * LDS;
                b0 = lane < nk ? __ldcg(x + lane) : 0.0;
                b1 = lane + 32 < nk ? __ldcg(x + lane + 32) : 0.0;
                warp_solve(S.T, S.rinv, nk, b0, b1);
                if (lane < nk) x[lane] = b0;
                if (lane + 32 < nk) x[lane + 32] = b1;
            }
        }
        cluster.sync();
        STAMP(13);
        if (lead) {
            for (int i = tid; i < nk * nk; i += NT) {
                const int r = i / nk, c = i % nk;
                if (c >= r) S.A[r * LDS + c] = 0.5 * (__ldcg(&G->B[r * LDS + c]) + __ldcg(&G->B[c * LDS + r]));
            }
            bsync();
            const bool ok = bchol(S.A, nk, nullptr, 0.0);
            if (ok) {
                for (int i = tid; i < nk * nk; i += NT) {   // L = R^T
                    const int r = i / nk, c = i % nk;
                    G->B[r * LDS + c] = c <= r ? S.A[c * LDS + r] : 0.0;
                }
            }
            if (tid == 0) G->ints[7] = ok ? PENCIL_OK : PENCIL_AGAIN;
        }
        cluster.sync();
        next = __ldcg(&G->ints[7]);
    }
    STAMP(1);
    if (next != PENCIL_OK) {
        if (lead && tid == 0 && next == PENCIL_AGAIN) {
            a.out_int[0] = kDenseBreakdown; a.out_int[1] = nk; a.out_int[2] = 0;
            G->ints[6] = 1;
        }
        return;
    }
    // C = L^{-1} G_R L^{-T}: by columns, then by rows, eight warps a CTA
    load_factor(S, G->B, false, nk);
    {
        const int c = blockIdx.x * (MAXM / kPencilCtas) + (tid >> 5);
        const bool act = (tid >> 5) < MAXM / kPencilCtas && c < nk;
        double b0 = 0.0, b1 = 0.0;
        if (act) {
            if (lane < nk) b0 = __ldcg(&G->H[lane * LDS + c]);
            if (lane + 32 < nk) b1 = __ldcg(&G->H[(lane + 32) * LDS + c]);
            warp_solve(S.T, S.rinv, nk, b0, b1);
            if (lane < nk) G->H[lane * LDS + c] = b0;
            if (lane + 32 < nk) G->H[(lane + 32) * LDS + c] = b1;
        }
        cluster.sync();
        if (act) {
            double* x = G->H + c * LDS;
            b0 = lane < nk ? __ldcg(x + lane) : 0.0;
            b1 = lane + 32 < nk ? __ldcg(x + lane + 32) : 0.0;
            warp_solve(S.T, S.rinv, nk, b0, b1);
            if (lane < nk) x[lane] = b0;
            if (lane + 32 < nk) x[lane + 32] = b1;
        }
    }
    cluster.sync();
    STAMP(2);
    if (!lead) return;
    // ---- 3. Hessenberg form of C
    for (int i = tid; i < nk * nk; i += NT) {
        const int r = i / nk, c = i % nk;
        S.H[r * LDS + c] = __ldcg(&G->H[r * LDS + c]);
    }
    bsync();
    bhessenberg(S.H, S.Vh, S.beta, nk, S.red);
    STAMP(14);
    for (int i = tid; i < nk * nk; i += NT) {
        const int r = i / nk, c = i % nk;
        G->H0[r * LDS + c] = S.H[r * LDS + c];
        G->Vh[r * LDS + c] = S.Vh[r * LDS + c];
    }
    for (int i = tid; i < nk; i += NT) G->beta[i] = S.beta[i];
#undef STAMP
}

// Eigenvector of one selected unit (CTA u): inverse iteration on the saved
// Hessenberg form H0, back to C's basis with the Householder reflectors, then
// y = L^{-T} z in the orthonormal basis, into Yre[u], Yim[u].  The units run as
// separate CTAs on separate SMs; one warp follows a unit's serial chain, after all
// four have brought the three matrices to double-word form (in the chain, the
// conversions and a division per row of L were 40 % of it).  250 -> 140 us at
// m = 64.
struct EigvecShm {
    dw H[MAXM * LDS], L[MAXM * LDS], V[MAXM * LDS];
    cdw U[MAXM * LDS];
    cdw mult[MAXM], rpiv[MAXM], x[MAXM];
    dw beta[MAXM], rl[MAXM];
    int swp[MAXM], top[2];
};

// 2^-k for the largest exponent k of a matrix, from the upper words of its entries
__device__ __forceinline__ double unit_scale(int top) {
    return top < 0x00100000 ? 1.0 : ldexp(1.0, 1023 - (top >> 20));
}

__global__ void __launch_bounds__(128) k_eigvec(DenseArgs a) {
    extern __shared__ __align__(16) unsigned char she[];
    EigvecShm& S = *reinterpret_cast<EigvecShm*>(she);
    const DenseState* G = state_of(a);
    if (G->ints[6]) return;
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const int nsel = G->ints[3], n = G->ints[0];
    if (u >= nsel) return;
    if (tid < 2) S.top[tid] = 0;
    __syncthreads();
    int th = 0, tl = 0;
    for (int i = tid; i < n * LDS; i += 128) {
        if (i % LDS >= n) continue;
        th = max(th, __double2hiint(G->H0[i]) & 0x7fffffff);
        tl = max(tl, __double2hiint(G->B[i]) & 0x7fffffff);
    }
    atomicMax(&S.top[0], th);
    atomicMax(&S.top[1], tl);
    __syncthreads();
    // H0 and lam, and L, scaled by a power of two to unit norm
    const double down = unit_scale(S.top[0]), ld = unit_scale(S.top[1]);
    for (int i = tid; i < n * LDS; i += 128) {
        if (i % LDS >= n) continue;
        S.H[i] = dw_from_double_fast(G->H0[i] * down);
        S.L[i] = dw_from_double_fast(G->B[i] * ld);
        if (i < (n - 2) * LDS) S.V[i] = dw_from_double_fast(G->Vh[i]);
    }
    if (tid < n) {
        if (tid < n - 2) S.beta[tid] = dw_from_double_fast(G->beta[tid]);
        S.rl[tid] = dw_div(dw_make(1.0f), dw_from_double_fast(G->B[tid * LDS + tid] * ld));
    }
    __syncthreads();
    if (tid >= 32) return;
    const int e = G->order[u];
    double lre = G->eig_re[e], lim = G->eig_im[e];
    if (G->nclose[u] > 0) { lre *= 1.0 + 1e-10 * G->nclose[u]; lim *= 1.0 + 1e-10 * G->nclose[u]; }
    const cdw lam = {dw_from_double(lre * down), dw_from_double(lim * down)};
    const float tiny = 0x1p-46f;   // a few units of the double-word precision of the unit-norm matrix
    cdw2 x = inverse_iteration(S.H, n, lam, S.U, S.mult, S.rpiv, S.x, S.swp, tiny);
    // z = Q x with Q = H_0 H_1 ... (reflectors applied last-first)
    for (int k = n - 3; k >= 0; --k) {
        dw v[2];
        dwacc sr = {0.0f, 0.0f}, si = {0.0f, 0.0f};
        for (int q = 0; q < 2; ++q) {
            const int j = lane + 32 * q;
            v[q] = j < n ? S.V[k * LDS + j] : dw_make(0.0f);
            dwacc_add_mul(sr, v[q], x.v[q].re);
            dwacc_add_mul(si, v[q], x.v[q].im);
        }
        const dw b = dw_neg(S.beta[k]);
        const dw tr = dw_mul(warp_sum_dw(sr), b), ti = dw_mul(warp_sum_dw(si), b);
        for (int q = 0; q < 2; ++q) x.v[q] = {dw_fma(x.v[q].re, v[q], tr), dw_fma(x.v[q].im, v[q], ti)};
    }
    // y = L^{-T} z: column-oriented back substitution with the lower factor L
    // (scaled to unit norm; y then carries the inverse scale, undone below)
    for (int i = n - 1; i >= 0; --i) {
        const cdw t = x.at(i);
        const dw rl = S.rl[i];
        const dw yr = dw_mul(t.re, rl), yi = dw_mul(t.im, rl);
        for (int q = 0; q < 2; ++q) {
            const int j = lane + 32 * q;
            if (q == 1 && i <= 32 && i != j) continue;
            const dw l = j < i ? S.L[i * LDS + j] : dw_make(0.0f);
            if (j < i) x.v[q] = {dw_fma(x.v[q].re, l, dw_neg(yr)), dw_fma(x.v[q].im, l, dw_neg(yi))};
            if (j == i) x.v[q] = {yr, yi};
        }
    }
    double* yr = a.work + (size_t)u * MAXM;
    double* yi = a.work + (size_t)MAXM * MAXM + (size_t)u * MAXM;
    for (int q = 0; q < 2; ++q) {
        const int i = lane + 32 * q;
        if (i >= n) break;
        yr[i] = dw_to_double(x.v[q].re) * ld;
        yi[i] = dw_to_double(x.v[q].im) * ld;
    }
}

// Order by |xi| (xi = 1/tau), conjugate pairs adjacent, select k': the eigenvalues
// are in the diagonal blocks of H (n x n).  Every step takes one thread per
// eigenvalue, unit or rank (one thread for all of it took 180 us).
static_assert(kFrancisThreads >= MAXM, "one eigenvalue per thread");
__device__ void select_units(const DenseArgs& a, DenseState* G, const double* H, int n) {
    __shared__ double er[MAXM], ei[MAXM], ka[MAXM], kr[MAXM];
    __shared__ int slot[MAXM], size[MAXM], order[MAXM], count;
    const int t = threadIdx.x, kp = a.kp;
    if (t == 0) count = 0;
    if (t < MAXM) { slot[t] = 0; size[t] = 0; }
    __syncthreads();
    const bool own = t < n;
    double re = 0.0, im = 0.0;
    if (own) {
        const bool second = t > 0 && H[t * LDS + t - 1] != 0.0;
        const bool first = !second && t + 1 < n && H[(t + 1) * LDS + t] != 0.0;
        if (first || second) {
            const double* b = H + (t - (second ? 1 : 0)) * (LDS + 1);
            const double aa = b[0], bb = b[1], cc = b[LDS], dd = b[LDS + 1];
            const double hf = 0.5 * (aa - dd), disc = hf * hf + bb * cc, mean = 0.5 * (aa + dd);
            const double sq = sqrt(fabs(disc));
            // two real eigenvalues, or tau = re -+ i im: the member with
            // Im(tau) < 0, which has Im(xi) > 0, first
            re = disc >= 0.0 ? (second ? mean - sq : mean + sq) : mean;
            im = disc >= 0.0 ? 0.0 : (second ? sq : -sq);
        } else {
            re = H[t * LDS + t];
        }
        er[t] = re; ei[t] = im;
        G->eig_re[t] = re; G->eig_im[t] = im;
    }
    // units: real eigenvalues and conjugate pairs (represented by Im(tau) < 0)
    const bool unit = own && !(im > 0.0);
    const double m2 = re * re + im * im;
    if (own) {
        const double xr = m2 > 0.0 ? re / m2 : INFINITY, xim = m2 > 0.0 ? -im / m2 : 0.0;
        ka[t] = m2 > 0.0 ? hypot(xr, xim) : INFINITY;
        kr[t] = xr;
    }
    __syncthreads();
    if (unit) {
        const double k = ka[t], x = kr[t];
        int rank = 0;
        for (int v = 0; v < n; ++v)
            rank += !(ei[v] > 0.0) && (ka[v] < k || (ka[v] == k && (kr[v] < x || (kr[v] == x && v < t))));
        slot[rank] = t;
        size[rank] = im != 0.0 ? 2 : 1;
    }
    __syncthreads();
    int sel = 0;
    if (own) {
        for (int q = 0; q < t; ++q) sel += size[q];
        if (size[t] > 0 && sel < kp) {
            order[t] = slot[t];
            G->order[t] = slot[t];
            G->kind[t] = size[t] == 2 ? (kp - sel >= 2 ? 2 : 1) : 0;
            atomicAdd(&count, 1);
        }
    }
    __syncthreads();
    const int ns = count;   // the ranks below ns are selected
    if (t < ns) {
        const int e = order[t];
        const double tre = er[e], tim = ei[e], t2 = tre * tre + tim * tim;
        // numerical clusters among the selected: later members get a shifted
        // inverse iteration and are orthogonalised against earlier ones
        const double mag = fmax(fabs(tre) + fabs(tim), 1e-300);
        int c = 0;
        for (int v = 0; v < t; ++v) c += fabs(er[order[v]] - tre) + fabs(ei[order[v]] - tim) <= 1e-8 * mag;
        G->nclose[t] = c;
        a.xi[2 * t] = tre / t2;
        a.xi[2 * t + 1] = -tim / t2;
    }
    if (t == 0) G->ints[3] = ns;
}

// Eigenvalues of the saved Hessenberg form (three warps; see k_pencil) and the
// selection.  The stage clocks 3 and 4 and the sweep counts come from this launch.
__global__ void __launch_bounds__(kFrancisThreads) k_francis(DenseArgs a) {
    extern __shared__ __align__(16) double shh[];
    DenseState* G = state_of(a);
    if (G->ints[6]) return;
    const int nk = G->ints[0];
    const int t = threadIdx.x;
    for (int i = t; i < nk * LDS; i += kFrancisThreads) shh[i] = G->H0[i];
    __syncthreads();
    if (a.clk && t == 0) a.clk[3] = clock64();
    const bool conv = francis_eigenvalues(shh, nk, a.clk ? a.clk + 9 : nullptr);
    if (a.clk && t == 0) a.clk[4] = clock64();
    if (conv) {
        select_units(a, G, shh, nk);
    } else if (t == 0) {
        a.out_int[0] = kDenseNoConv; a.out_int[1] = nk; a.out_int[2] = 0; G->ints[6] = 1;
    }
}

// Two selected units belong to one numerical cluster (u the later one)
__device__ __forceinline__ bool close_units(const DenseState* G, int u, int v) {
    const int e = G->order[u], f = G->order[v];
    const double mag = fmax(fabs(G->eig_re[e]) + fabs(G->eig_im[e]), 1e-300);
    return fabs(G->eig_re[f] - G->eig_re[e]) + fabs(G->eig_im[f] - G->eig_im[e]) <= 1e-8 * mag;
}

// Cluster orthogonalisation, pair rotation, unit norm of unit u and the
// coefficients of its one or two columns of Y' = [Y0 YR yR~ YI] (CTA u).  A
// member of a cluster needs the earlier members' final vectors: its CTA works
// them out again from the raw ones (clusters are small, and one warp doing the
// units in turn took 75 us).  The back substitutions (real and imaginary column,
// for P_new and V_new - P_new, a warp each) subtract a solved entry from all rows
// at once: two FP64 operations deep a row instead of a sum (59 us; the whole
// stage, with the state's copy, 185 -> 25 us at m = 64, 16 columns).
__global__ void __launch_bounds__(128) k_finish(DenseArgs a) {
    extern __shared__ __align__(16) double shy[];
    double* R = shy;                  // MAXM x LDS
    double* Y = R + MAXM * LDS;       // [unit][re, im][MAXM]
    __shared__ double rinv[MAXM], W[4][MAXM];
    const DenseState* G = state_of(a);
    if (G->ints[6]) return;
    const int nk = G->ints[0], nvk = G->ints[1], nsel = G->ints[3];
    const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (u >= nsel) return;
    if (a.clk && u == 0 && tid == 0) { a.clk[5] = clock64(); a.clk[6] = a.clk[5]; }
    for (int i = tid; i < nk * LDS; i += 128) R[i] = G->A[i];
    const double* Yre = a.work;
    const double* Yim = a.work + MAXM * MAXM;
    if (warp == 0) {
        unsigned need = 1u << u;
        for (int v = u; v > 0; --v)
            if ((need >> v & 1u) && G->nclose[v] > 0)
                for (int w = 0; w < v; ++w)
                    if (close_units(G, v, w)) need |= 1u << w;
        for (int v = 0; v <= u; ++v) {
            if (!(need >> v & 1u)) continue;
            double* yr = Y + v * 2 * MAXM;
            double* yi = yr + MAXM;
            for (int i = lane; i < nk; i += 32) { yr[i] = Yre[v * MAXM + i]; yi[i] = Yim[v * MAXM + i]; }
            wsync();
            // two passes of modified Gram-Schmidt against the earlier members
            // of the cluster (the second restores the orthogonality the first
            // loses when most of y lies in their span); plain complex inner
            // products, in the orthonormal basis
            for (int pass = 0; pass < 2 && G->nclose[v] > 0; ++pass)
                for (int w = 0; w < v; ++w) {
                    if (!close_units(G, v, w)) continue;
                    const double* vr = Y + w * 2 * MAXM;
                    const double* vi = vr + MAXM;
                    // y -= v (v^H y) / (v^H v)
                    double pr = 0.0, pi = 0.0, vv = 0.0;
                    for (int i = lane; i < nk; i += 32) {
                        pr += vr[i] * yr[i] + vi[i] * yi[i];
                        pi += vr[i] * yi[i] - vi[i] * yr[i];
                        vv += vr[i] * vr[i] + vi[i] * vi[i];
                    }
                    pr = warp_sum(pr); pi = warp_sum(pi); vv = warp_sum(vv);
                    pr /= vv; pi /= vv;
                    for (int i = lane; i < nk; i += 32) {
                        const double ar = vr[i] * pr - vi[i] * pi, ai = vr[i] * pi + vi[i] * pr;
                        yr[i] -= ar;
                        yi[i] -= ai;
                    }
                    wsync();
                }
            double aa = 0.0, bb = 0.0, ab = 0.0;
            for (int i = lane; i < nk; i += 32) { aa += yr[i] * yr[i]; bb += yi[i] * yi[i]; ab += yr[i] * yi[i]; }
            aa = warp_sum(aa); bb = warp_sum(bb); ab = warp_sum(ab);
            double c = 1.0, sn = 0.0;
            if (G->kind[v] != 0) {
                const double phi = 0.5 * atan2(-2.0 * ab, aa - bb);
                c = cos(phi); sn = sin(phi);
            }
            double nrm = sqrt(aa + bb);
            if (!(nrm > 0.0)) nrm = 1.0;
            for (int i = lane; i < nk; i += 32) {
                const double re = yr[i], im = yi[i];
                yr[i] = (re * c - im * sn) / nrm;
                yi[i] = (re * sn + im * c) / nrm;
            }
            wsync();
        }
    } else {
        for (int i = tid - 32; i < nk; i += 96) rinv[i] = 1.0 / G->A[i * LDS + i];
    }
    __syncthreads();
    if (a.clk && u == 0 && tid == 0) a.clk[7] = clock64();
    // columns of the unit: real part, imaginary part or -1
    int nreal = 0, npair = 0, ncut = 0, before_real = 0, before_pair = 0;
    for (int v = 0; v < nsel; ++v) {
        const int k = G->kind[v];
        if (v < u) { before_real += k == 0; before_pair += k == 2; }
        nreal += k == 0; npair += k == 2; ncut += k == 1;
    }
    const int kind = G->kind[u];
    const int cr = kind == 0 ? before_real : kind == 2 ? nreal + before_pair : nreal + npair;
    const int ci = kind == 2 ? nreal + npair + ncut + before_pair : -1;
    if (tid == 0) {
        a.tags[cr] = kind == 0 ? 0 : kind == 2 ? 1 : 2;
        a.tag_partner[cr] = ci;
        if (ci >= 0) { a.tags[ci] = 3; a.tag_partner[ci] = cr; }
    }
    // ---- raw coefficients.  Z-hat = Z diag(colscale t) R^{-1}; R^{-1} is
    // upper triangular with the V columns first, so
    //   P_new = Z-hat[:, rest] Y'_rest = Z diag(colscale t) R^{-1} [0; Y'_rest]
    //   V_new - P_new = Z-hat[:, V] Y'_V = Z_V diag(colscale t) R_VV^{-1} Y'_V
    // warps 0, 1: P_new's real and imaginary column, 2, 3: V_new - P_new's
    if ((warp & 1) == 0 || ci >= 0) {
        const bool isv = warp >= 2;
        const double* y = Y + (u * 2 + (warp & 1)) * MAXM;
        const int lim = isv ? nvk : nk, r0 = lane, r1 = lane + 32;
        double b0 = r0 < lim && (isv || r0 >= nvk) ? y[r0] : 0.0;
        double b1 = r1 < lim && (isv || r1 >= nvk) ? y[r1] : 0.0;
        for (int i = lim - 1; i >= 0; --i) {
            const double w = __shfl_sync(0xffffffffu, i >= 32 ? b1 : b0, i & 31) * rinv[i];
            if (r0 < i) b0 = fma(-R[r0 * LDS + i], w, b0);
            if (i > 32) {
                if (r1 < i) b1 = fma(-R[r1 * LDS + i], w, b1);
            }
            if (r0 == i) b0 = w;
            if (r1 == i) b1 = w;
        }
        W[warp][r0] = b0;
        W[warp][r1] = b1;
    }
    const int m = a.m, kp = a.kp;
    for (int half = 0; half < 2; ++half) {
        const int col = half ? ci : cr;
        if (col < 0) break;
        for (int i = tid; i < m; i += 128) a.Cp[i * kp + col] = 0.0;
        for (int i = tid; i < a.nv; i += 128) a.Cvv[i * kp + col] = 0.0;
    }
    __syncthreads();
    for (int half = 0; half < 2; ++half) {
        const int col = half ? ci : cr;
        if (col < 0) break;
        for (int q = tid; q < nk; q += 128) {
            const int raw = G->kidx[q];
            const double tr = G->t[raw] * a.colscale[raw];
            a.Cp[raw * kp + col] = tr * W[half][q];
            if (q < nvk) a.Cvv[raw * kp + col] = tr * W[2 + half][q];
        }
    }
    if (u == 0 && tid == 0) {
        if (a.clk) a.clk[8] = clock64();
        a.out_int[0] = kDenseOK;
        a.out_int[1] = nk;
        a.out_int[2] = nsel;
    }
}

}  // namespace

size_t dense_work_doubles() { return kDenseWorkDoubles; }

cudaError_t dense_extract(const DenseArgs& a, cudaStream_t s) {
    size_t shm = sizeof(PencilShm);
    cudaError_t e = cudaFuncSetAttribute(k_pencil, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
    if (e != cudaSuccess) return e;
    const size_t shf = sizeof(double) * kFrancisRows * LDS;
    e = cudaFuncSetAttribute(k_francis, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shf);
    if (e != cudaSuccess) return e;
    const size_t she = sizeof(EigvecShm);
    e = cudaFuncSetAttribute(k_eigvec, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)she);
    if (e != cudaSuccess) return e;
    const size_t shn = sizeof(double) * (MAXM * LDS + MAXKP * 2 * MAXM);
    e = cudaFuncSetAttribute(k_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shn);
    if (e != cudaSuccess) return e;
    k_pencil<<<kPencilCtas, NT, shm, s>>>(a);
    k_francis<<<1, kFrancisThreads, shf, s>>>(a);
    k_eigvec<<<a.kp, 128, she, s>>>(a);
    k_finish<<<a.kp, 128, shn, s>>>(a);
    count_launches(4);
    return cudaGetLastError();
}

}  // namespace plhr

// ======================================================================
// Convergence status, Rayleigh quotients, final Rayleigh-Ritz.
namespace plhr {
namespace {

// relative residual ||r|| / (max(|lam|, 1) ||Bv||); order by |lam - sigma|
// (ties: smaller lam first); converged when the k nearest meet tol; a column
// is active (contributes W and S) when its residual is above tol.
__global__ void k_status(StatusArgs a) {
    if (threadIdx.x != 0) return;
    const int kp = a.kp;
    int nan = 0;
    for (int j = 0; j < kp; ++j) {
        double rn = sqrt(a.sums[j]), bn = sqrt(a.sums[kp + j]);
        double l = a.lam[j];
        double rel = rn / (fmax(fabs(l), 1.0) * bn);
        if (!isfinite(rel)) { nan = 1; rel = INFINITY; }
        a.rel[j] = rel;
        a.order[j] = j;
    }
    for (int i = 1; i < kp; ++i) {
        int o = a.order[i];
        double d = fabs(a.lam[o] - a.sigma), l = a.lam[o];
        int j = i - 1;
        while (j >= 0) {
            int p = a.order[j];
            double dp = fabs(a.lam[p] - a.sigma);
            if (dp > d || (dp == d && a.lam[p] > l)) { a.order[j + 1] = p; --j; }
            else break;
        }
        a.order[j + 1] = o;
    }
    int conv = 1;
    for (int q = 0; q < a.k; ++q)
        if (!(a.rel[a.order[q]] <= a.tol)) conv = 0;
    int na = 0;
    for (int j = 0; j < kp; ++j)
        if (!(a.rel[j] <= a.tol)) { a.lam_act[na] = a.lam[j]; a.active[na++] = j; }
    a.hstat[0] = conv;
    a.hstat[1] = na;
    a.hstat[2] = nan;
}

__global__ void k_rq(int kp, const double* dots, const int* tags, const int* partner, double* lam, double* scale) {
    if (threadIdx.x != 0) return;
    for (int j = 0; j < kp; ++j) {
        double aa = dots[j], bb = dots[kp + j];
        double l = aa / bb;
        if (tags[j] == 1 || tags[j] == 3) {
            int p = partner[j];
            l = (aa + dots[p]) / (bb + dots[kp + p]);
        }
        lam[j] = l;
        scale[j] = 1.0 / sqrt(bb);
    }
}

// columns in order by |th - sigma| (ties: smaller th first), one thread
__device__ void rr_order(const double* th, int n, double sigma, int* ord) {
    for (int j = 0; j < n; ++j) ord[j] = j;
    for (int i = 1; i < n; ++i) {
        int o = ord[i];
        double d = fabs(th[o] - sigma), l = th[o];
        int j = i - 1;
        while (j >= 0) {
            int p = ord[j];
            double dp = fabs(th[p] - sigma);
            if (dp > d || (dp == d && th[p] > l)) { ord[j + 1] = p; --j; }
            else break;
        }
        ord[j + 1] = o;
    }
}

// one warp: Cholesky of GB, M = L^-1 GA L^-T, cyclic Jacobi (Golub & Van Loan
// Sec. 8.5), C = L^-T W, sort by |theta - sigma|.  Where GB has no Cholesky factor
// (ok_out 0) the columns are only scaled and sorted, theta their Rayleigh
// quotients: a block that is multiplied by C all the same keeps its columns.
__global__ void __launch_bounds__(32) k_rr(int n, const double* GA, const double* GB, double sigma,
                                           const double* rowscale, double* C, double* theta, int* ok_out) {
    __shared__ double L[32 * 33], M[32 * 33], W[32 * 33];
    __shared__ double th[32];
    __shared__ int ord[32];
    const int lane = threadIdx.x;
    const int ld = 33;
    for (int i = lane; i < n * n; i += 32) {
        int r = i / n, c = i % n;
        L[r * ld + c] = 0.5 * (GB[r * n + c] + GB[c * n + r]);
        M[r * ld + c] = 0.5 * (GA[r * n + c] + GA[c * n + r]);
    }
    __syncwarp();
    if (!chol_lower(L, n, ld)) {
        if (lane < n) th[lane] = GA[lane * n + lane] / GB[lane * n + lane];
        __syncwarp();
        if (lane == 0) {
            rr_order(th, n, sigma, ord);
            *ok_out = 0;
        }
        __syncwarp();
        for (int i = lane; i < n * n; i += 32) {
            const int r = i / n, c = i % n;
            C[i] = r == ord[c] ? (rowscale ? rowscale[r] : 1.0) : 0.0;
        }
        if (lane < n) theta[lane] = th[ord[lane]];
        return;
    }
    // M <- L^-1 M L^-T
    for (int c = lane; c < n; c += 32)
        for (int i = 0; i < n; ++i) {
            double s = M[i * ld + c];
            for (int l = 0; l < i; ++l) s -= L[i * ld + l] * M[l * ld + c];
            M[i * ld + c] = s / L[i * ld + i];
        }
    __syncwarp();
    for (int r = lane; r < n; r += 32)
        for (int j = 0; j < n; ++j) {
            double s = M[r * ld + j];
            for (int l = 0; l < j; ++l) s -= M[r * ld + l] * L[j * ld + l];
            M[r * ld + j] = s / L[j * ld + j];
        }
    __syncwarp();
    for (int i = lane; i < n * n; i += 32) {
        int r = i / n, c = i % n;
        if (c > r) { double s = 0.5 * (M[r * ld + c] + M[c * ld + r]); M[r * ld + c] = s; M[c * ld + r] = s; }
        W[r * ld + c] = (r == c) ? 1.0 : 0.0;
    }
    __syncwarp();
    for (int sweep = 0; sweep < 30; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int i = lane; i < n * n; i += 32) {
            int r = i / n, c = i % n;
            double v = M[r * ld + c] * M[r * ld + c];
            tot += v;
            if (r != c) off += v;
        }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if (off <= 1e-30 * tot) break;
        for (int p = 0; p < n - 1; ++p)
            for (int q = p + 1; q < n; ++q) {
                double apq = M[p * ld + q];
                if (apq == 0.0) continue;
                double app = M[p * ld + p], aqq = M[q * ld + q];
                double tau = (aqq - app) / (2.0 * apq);
                double t = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
                double c = 1.0 / sqrt(1.0 + t * t), s = t * c;
                __syncwarp();
                // rows p, q of M
                for (int j = lane; j < n; j += 32) {
                    double mp = M[p * ld + j], mq = M[q * ld + j];
                    M[p * ld + j] = c * mp - s * mq;
                    M[q * ld + j] = s * mp + c * mq;
                }
                __syncwarp();
                for (int j = lane; j < n; j += 32) {
                    double mp = M[j * ld + p], mq = M[j * ld + q];
                    M[j * ld + p] = c * mp - s * mq;
                    M[j * ld + q] = s * mp + c * mq;
                    double wp = W[j * ld + p], wq = W[j * ld + q];
                    W[j * ld + p] = c * wp - s * wq;
                    W[j * ld + q] = s * wp + c * wq;
                }
                __syncwarp();
            }
    }
    if (lane == 0) {
        for (int j = 0; j < n; ++j) th[j] = M[j * ld + j];
        rr_order(th, n, sigma, ord);
    }
    __syncwarp();
    // C = L^-T W (back substitution per column), columns reordered
    for (int jj = lane; jj < n; jj += 32) {
        int j = ord[jj];
        double x[32];
        for (int i = n - 1; i >= 0; --i) {
            double s = W[i * ld + j];
            for (int l = i + 1; l < n; ++l) s -= L[l * ld + i] * x[l];
            x[i] = s / L[i * ld + i];
        }
        for (int i = 0; i < n; ++i) C[i * n + jj] = x[i] * (rowscale ? rowscale[i] : 1.0);
        theta[jj] = th[j];
    }
    if (lane == 0) *ok_out = 1;
}

}  // namespace

cudaError_t dense_status(const StatusArgs& a, cudaStream_t s) {
    k_status<<<1, 32, 0, s>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t dense_rq(int kp, const double* dots, const int* tags, const int* partner, double* lam, double* scale,
                     cudaStream_t s) {
    k_rq<<<1, 32, 0, s>>>(kp, dots, tags, partner, lam, scale);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t dense_rr(int kp, const double* GA, const double* GB, double sigma, const double* rowscale, double* C,
                     double* theta, int* ok, cudaStream_t s) {
    if (kp > 32) return cudaErrorInvalidValue;
    k_rr<<<1, 32, 0, s>>>(kp, GA, GB, sigma, rowscale, C, theta, ok);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace plhr

extern "C" plhr_status plhr_tharm_extract(int m, int kp, int nv, const double* Gzz, const double* Guq,
                                          const double* Gqz, const double* colscale, double* Cp, double* Cvv,
                                          int* tags, int* partner, double* xi, int* status, long long* clk,
                                          void* stream) {
    using namespace plhr;
    clear_error();
    if (m < 1 || m > kDenseMaxM || kp < 1 || kp > 16 || kp > m || nv < 1 || nv > m || !Gzz || !Guq || !Gqz ||
        !colscale || !Cp || !Cvv || !tags || !partner || !xi || !status) {
        set_error("plhr_tharm_extract: invalid argument");
        return PLHR_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    double* work = nullptr;
    PLHR_TRY_CUDA(ws_alloc(reinterpret_cast<void**>(&work), sizeof(double) * dense_work_doubles(), s));
    DenseArgs a;
    a.m = m; a.kp = kp; a.nv = nv; a.Gzz = Gzz; a.Guq = Guq; a.Gqz = Gqz; a.colscale = colscale; a.work = work;
    a.Cp = Cp; a.Cvv = Cvv; a.tags = tags; a.tag_partner = partner; a.xi = xi; a.out_int = status; a.clk = clk;
    cudaError_t e = dense_extract(a, s);
    ws_free(work, s);
    PLHR_TRY_CUDA(e);
    return PLHR_OK;
}

// ======================================================================
// Allocation-free variant of plhr_tharm_extract.
//
// Some callers cannot allocate device memory at the moment they need the
// projected eigensolve: an application that has handed the whole device to
// its own pooled allocator or arena, a service with a fixed memory budget
// that forbids allocation after start-up, or code running from a host
// callback where an allocation could block on the allocator.  For them this
// entry point takes its scratch from a fixed array compiled into the library
// instead of calling the CUDA allocator.
namespace {

// Scratch of the projected eigensolve for the largest supported basis
// (m = 64): two 64 x 64 arrays and the saved state, about 230 KiB.  Every
// GPU that loads the library holds this array until the process exits.
constexpr size_t kNoAllocScratchDoubles = plhr::kDenseWorkDoubles;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

// Device address of the scratch array, looked up once per device.
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
double* g_noalloc_ptr[kMaxDevices] = {nullptr};

plhr_status noalloc_scratch(double** out) {
    int dev = 0;
    PLHR_TRY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) {
        plhr::set_error("plhr_tharm_extract_noalloc: device ordinal %d out of range", dev);
        return PLHR_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        // host code sees only a stand-in for g_noalloc_scratch; its device
        // address comes from the runtime, with this device current
        PLHR_TRY_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        g_noalloc_ptr[dev] = static_cast<double*>(p);
    }
    *out = g_noalloc_ptr[dev];
    return PLHR_OK;
}

}  // namespace

extern "C" plhr_status plhr_tharm_extract_noalloc(int m, int kp, int nv, const double* Gzz, const double* Guq,
                                                  const double* Gqz, const double* colscale, double* Cp,
                                                  double* Cvv, int* tags, int* partner, double* xi, int* status,
                                                  void* stream) {
    using namespace plhr;
    clear_error();
    if (m > kDenseMaxM) {
        set_error("plhr_tharm_extract_noalloc: m = %d exceeds the maximum %d of the built-in scratch", m,
                  kDenseMaxM);
        return PLHR_EINVAL;
    }
    if (m < 1 || kp < 1 || kp > 16 || kp > m || nv < 1 || nv > m || !Gzz || !Guq || !Gqz || !colscale || !Cp ||
        !Cvv || !tags || !partner || !xi || !status) {
        set_error("plhr_tharm_extract_noalloc: invalid argument");
        return PLHR_EINVAL;
    }
    if (dense_work_doubles() > kNoAllocScratchDoubles) {
        set_error("plhr_tharm_extract_noalloc: built-in scratch too small");
        return PLHR_EINVAL;
    }
    double* work = nullptr;
    PLHR_TRY(noalloc_scratch(&work));
    DenseArgs a;
    a.m = m; a.kp = kp; a.nv = nv; a.Gzz = Gzz; a.Guq = Guq; a.Gqz = Gqz; a.colscale = colscale; a.work = work;
    a.Cp = Cp; a.Cvv = Cvv; a.tags = tags; a.tag_partner = partner; a.xi = xi; a.out_int = status; a.clk = nullptr;
    PLHR_TRY_CUDA(dense_extract(a, (cudaStream_t)stream));
    return PLHR_OK;
}
