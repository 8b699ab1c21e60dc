// The three projected Grams of FP64 blocks on the tensor cores (tcgen05), by
// fixed-point slices.
//
// With the trial basis Z (m <= 64 columns), its image A Z and the T-harmonic
// images Q, U = A Z - sigma Z and column scales D,
//     (Z D)^T (Z D),   (U D)^T (Q D),   (Q D)^T (Z D)       (Eq. THarm_evp)
// as FP64 m x m matrices.  GB300 issues FP64 at 1/64 of FP32 and a
// double-word multiply-add costs 13 FP32 instructions, so on the CUDA cores
// this pass is bound by arithmetic at 5-6 % of HBM; here it is a BF16 tensor
// contraction of integers.
//
// Slices (the splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59, 2012, in fixed point).  A column's
// entries are rounded to integers X of at most 53 bits below a power of two
// 2^E above the column's magnitude, and X is written in six balanced digits
// of base 2^9, d_k in [-256, 256], k = 0 the leading one.  Every such digit is
// a BF16 number (8 significant bits and a sign), also when it is stored as
// d_k 2^-9k.  The product of digits k and l of two values belongs to level
// k + l; levels 0 to 6 (26 products) are formed, of U^T Q level 7 too, which its
// MMAs of two levels bring with them.  The rest is below 2^-63 of 2^E 2^E' a row.
// Sums: over a period of 128 rows a level of L + 1 products is at most
// (L + 1) 128 2^16 (its two products with a leading digit, which is below 2^7, half
// of that), so levels 0 to 2, and level 3 except where all its products are near
// their largest, accumulate exactly in FP32 tensor memory.  Levels 4 to 6 share an
// accumulator, which drops what is below 2^-24 of its content with each MMA.  At the
// end of a period the accumulators are read back as integers into 64-bit sums
// in units of 2^-35 of the leading digit product (2^-53 of 2^E 2^E').
//
// Accuracy.  On columns whose entries are of one size, such as trial bases, an entry is
// correct to a few 2^-53 of the column norms: 2e-16 to 9e-16 of |x| |y| at 40,000 to
// 2,097,152 rows (FP64 multiply-adds 2e-16 to 1.3e-15, double-word ones 5e-15 to
// 2e-11).  A column with few large entries and a long tail of equal low digits loses
// up to 2^-40 of the product of the largest entries per 128 rows of an SM (128 MMAs
// at one unit of the shared accumulator); measured with one entry 1 and 10^-3, 10^-4 or
// 10^-6 elsewhere at 2,097,152 rows: 1e-13, 2.4e-12, 2e-13 where FP64 multiply-adds
// lose 1e-13, 6e-13, 6e-13 (without all of level 6, which has 2 d_1 d_5 and 2 d_2 d_4 of
// one sign there: 1.7e-12, 6.5e-12, 5e-13).
//
// Exponents.  E is kept per column and CTA: the largest exponent met so far
// plus two, in long runs from 32 rows spread over the CTA's share on.
// When a value exceeds it, the pending period is folded, the integers are
// shifted to the new exponents and the CTA goes on.  So the precision is relative to
// the columns' norms (what the Cholesky factorisation of a Gram matrix needs), not to
// each pair of entries.
// A column holding Inf or NaN or values outside the exponents' range (kExpFloor,
// kExpTop) and a wait that times out set the CTA's flag: the plain FP64 kernel, which
// is launched behind this one and returns at once otherwise, then redoes the Grams.
//
// Tiles (mp = m rounded up to 16).  A step of 32 rows is one K-major panel of
// operand rows per digit.  [Z_k; Q_k] with Z_l, 128 x mp x 16, gives Z^T Z and
// Q^T Z; five accumulators hold levels 0, 1, 2, 3 and the rest.  U^T Q fills the
// 128 lanes with two levels at once: [U_k-1; U_k] with Q_l adds to level
// k + l - 1 in the upper and k + l in the lower half, so three accumulators hold
// all eight levels and the eight fill the 512 columns of tensor memory at
// m = 64.  The 86 MMAs of a step take 4.2k cycles (49 each: operand reads from
// shared memory bind at N = 64).
//
// Roles.  Four warps issue the MMAs (issued by a converting warp, that warp
// stands still for the time they take); 16 warps convert, and read the
// accumulators back every 128 rows.  A converting warp takes 4 columns, all 32
// rows, so that it agrees on their exponents by shuffles; the next step's
// values are in flight in registers meanwhile.  A step takes about 12k cycles: the
// conversion, about 40 integer and FP32 instructions per value, 4.6k of them, the
// rest loads, the barrier and a period's share of the read-back.
//
// Measured on GB300 on trial bases of a Laplacian: m = 36, 262,144 rows 370 us a call
// (FP64 multiply-adds 2.64 ms, bound by the FP64 pipe); m = 64, 2,097,152 rows
// 2.61 ms a call, 2.53 of the kernel (double-word multiply-adds on the FP32 pipes 9.45 ms).
#include "blockops.h"
#include "tc.h"

namespace plhr {
namespace {

constexpr int kFxConv = 512;                   // threads that convert and read back
constexpr int kFxThreads = kFxConv + 128;      // and a warpgroup that issues the MMAs
constexpr int kFxK = 32;                       // rows per step
constexpr int kMaxPeriod = 4;                  // steps per period
constexpr int kDigits = 6;
// the 64-bit sums are in units of 2^-kUnit of the leading digit product: a period adds at
// most 2^58 of them, so a CTA writes its sums out where one may pass 2^62 (at 2^-36 the
// 128^3 trial basis does so: 2.68 ms against 2.65 at m = 64)
constexpr int kUnit = 35;
constexpr int kCore = 128;                     // core matrix: 8 rows x 16 bytes
// A step's panel: the U digits between two blocks of zeros (per core column of 8
// rows of the step: [0 | U0 | .. | U5 | 0], 8 mp operand rows), then per digit a
// slice [Z | Q] of 2 mp operand rows.  Core columns are 64 bytes further apart
// than their rows take, so that the stores of a warp (4 columns of all 4 core
// columns) use different banks.
__host__ __device__ constexpr int lbo_u_of(int mp) { return 8 * 16 * mp + 64; }
__host__ __device__ constexpr int lbo_z_of(int mp) { return 2 * 16 * mp + 64; }
__host__ __device__ constexpr int panel_of(int mp) { return 4 * (lbo_u_of(mp) + kDigits * lbo_z_of(mp)); }
constexpr int kFxOperand = 2 * panel_of(64) + 4096;  // A reads 128 rows: up to 2 KB past a narrow last slice
constexpr int kFxMeta = 10240;
constexpr int kLdD = 33;                       // staging of 32 columns of sums
constexpr int kFxSmem = kFxOperand + kFxMeta + 128 * kLdD * 8;
constexpr int kIssuers = 4;
// Exponents start at kExpFloor: a share of a column that has nothing from 2^-895 up, but
// not only zeros, is left to k_gram, and so are values from 2^1017 up, whose column
// factors could leave the range that their products with the column scales keep
constexpr int kExpFloor = 128;
constexpr int kExpTop = 0x7f8;
constexpr long long kFxWait = 4LL << 30;       // about 2 s

struct FxCols {
    const double* p[3][64];   // Z, AZ, Q
    int64_t ld[3][64];
};
struct FxMeta {
    uint64_t done[2];         // the MMAs that read this panel completed
    uint64_t full[2];         // this panel is converted
    uint32_t tmem;
    uint32_t carry[2];        // the step's MMAs add to the accumulators
    int stop;
    // of column j of Z, Q and U at j, mp + j and 2 mp + j: the exponent of the
    // sums, that of the panel being converted, the column scale times
    // 2^(exponent - 1022)
    int e[192];
    int en[192];
    int low[192];             // met a value other than zero while the exponent was the floor
    double fac[192];
    FxCols cols;
};
static_assert(sizeof(FxMeta) <= (size_t)kFxMeta, "meta area");

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// X = x 2^(1076 - e) rounded to an integer, |X| <= 2^53, for an exponent e >
// exp_field(x); returned as 2 (X + 2^17 (1 + 2^18 + 2^36)) + a fraction bit, so
// that the 18-bit fields from bit 1 on (the top one has 19) hold the digit
// pairs of X plus 2^17.  Zero and subnormal x, and Inf and NaN (flagged by the
// caller), shift out to 0.
__device__ __forceinline__ unsigned long long fields_of(double x, int e) {
    const unsigned hw = (unsigned)__double2hiint(x), lw = (unsigned)__double2loint(x);
    const unsigned sh = (unsigned)(e - (int)((hw >> 20) & 0x7ffu));
    const unsigned long long M = ((unsigned long long)((hw & 0xfffffu) | 0x100000u) << 32) | lw;
    unsigned long long X;
    asm("shr.u64 %0, %1, %2;" : "=l"(X) : "l"(M << 2), "r"(sh));   // a shift past 63 gives 0
    const unsigned long long sgn = (unsigned long long)((long long)(int)hw >> 63);
    constexpr unsigned long long B = 2 * ((1ull << 17) | (1ull << 35) | (1ull << 53)) + 1;
    return (X ^ sgn) + (B - sgn);
}

// digits 2 P and 2 P + 1 of a field word, times 2^-18P and 2^-18P-9, as FP32:
// the field in the mantissa of a power of two, less the power and the 2^17,
// is split at 2^9 by rounding (FMA-pipe instructions: the integer ones bind)
template <int P>
__device__ __forceinline__ void digit_pair(unsigned long long W, float& hi, float& lo) {
    const unsigned w0 = (unsigned)W, w1 = (unsigned)(W >> 32);
    const unsigned w = P == 2 ? w0 : P == 1 ? __funnelshift_r(w0, w1, 18) : w1 >> 4;
    constexpr unsigned mask = P == 0 ? 0xffffeu : 0x7fffeu;
    // low digit in units of 2^(9 - 18 (P + 1) + ...): bit 1 of the mantissa weighs 2^(-18 P - 9)
    constexpr unsigned big = (unsigned)(127 + 22 - 9 - 18 * P) << 23;
    constexpr unsigned half = (unsigned)(127 + 17 - 9 - 18 * P) << 23;
    const float f = __fsub_rn(__uint_as_float((w & mask) | big), __uint_as_float(big) + __uint_as_float(half));
    // 1.5 2^23 in units of the high digit
    constexpr unsigned grid = ((unsigned)(127 + 23 - 18 * P) << 23) | 0x400000u;
    hi = __fsub_rn(__fadd_rn(f, __uint_as_float(grid)), __uint_as_float(grid));
    lo = __fsub_rn(f, hi);
}

template <int P>
__device__ __forceinline__ void put_pair(unsigned char* dst, int slice, const unsigned long long* W) {
    float h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) digit_pair<P>(W[i], h[i], l[i]);
    auto pack = [](float x, float y) { return __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632); };
    *reinterpret_cast<uint2*>(dst + 2 * P * slice) = make_uint2(pack(h[0], h[1]), pack(h[2], h[3]));
    *reinterpret_cast<uint2*>(dst + (2 * P + 1) * slice) = make_uint2(pack(l[0], l[1]), pack(l[2], l[3]));
}

// the digits of four consecutive rows of one column: 8 bytes per digit, the
// digits slice bytes apart
__device__ __forceinline__ void put_digits(unsigned char* dst, int slice, const double* x, int e) {
    unsigned long long W[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) W[i] = fields_of(x[i], e);
    put_pair<0>(dst, slice, W);
    put_pair<1>(dst, slice, W);
    put_pair<2>(dst, slice, W);
}

// barrier of the converting threads: whether pred holds for any of them
__device__ __forceinline__ bool conv_any(bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "barrier.cta.red.or.pred p, 1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(r)
        : "r"((uint32_t)pred), "n"(kFxConv)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void conv_sync() { asm volatile("barrier.cta.sync 1, %0;\n" ::"n"(kFxConv) : "memory"); }

// Add 8 columns of the accumulator at TMEM column ta to acc: the values times
// mul (a power of two) are integers in units of 2^SHIFT of acc (rounded where
// they are not).  The integer is the mantissa of 1.5 2^23 + value (one FFMA;
// the conversion instruction runs at 1/8 of its rate), which holds below 2^22
// in magnitude; sums beyond that (columns of nearly constant magnitude) take
// the conversion.  kMagic 2^SHIFT too much is added per value: the caller
// takes all of them off at once.
constexpr unsigned kMagic = 0x4b400000u;       // 1.5 2^23
template <int SHIFT>
__device__ __forceinline__ void add8(unsigned long long* acc, const uint32_t* v, float mul) {
    unsigned chk = 0;
    uint32_t w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        w[i] = __float_as_uint(__fmaf_rn(__uint_as_float(v[i]), mul, __uint_as_float(kMagic)));
        chk |= w[i] ^ 0x4b000000u;
    }
    if (__any_sync(0xffffffffu, chk >= 0x00800000u)) {
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] = (uint32_t)__float2int_rn(__uint_as_float(v[i]) * mul) + kMagic;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        if (SHIFT >= 32) acc[i] += (unsigned long long)(w[i] << (SHIFT & 31)) << 32;
        else asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(acc[i]) : "r"(w[i]), "n"(1u << (SHIFT & 31)));
    }
}

__global__ void __launch_bounds__(kFxThreads, 1) k_gram_fx(int64_t n, int m, int mp, const __grid_constant__ FxCols C,
                                                           int has_q, double sigma, const double* __restrict__ csc,
                                                           double* __restrict__ partial, int* __restrict__ flags,
                                                           int period) {
    extern __shared__ __align__(1024) unsigned char smem[];
    FxMeta& S = *reinterpret_cast<FxMeta*>(smem + kFxOperand);
    double* D = reinterpret_cast<double*>(smem + kFxOperand + kFxMeta);   // [128][kLdD]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int lbo_u = lbo_u_of(mp), lbo_z = lbo_z_of(mp), slice = 4 * lbo_z, block = 16 * mp;   // block: mp rows

    for (int t = tid; t < 3 * 64; t += kFxThreads) {
        const int f = t >> 6, j = t & 63;
        S.cols.p[f][j] = C.p[f][j];
        S.cols.ld[f][j] = C.ld[f][j];
        S.e[t] = S.en[t] = kExpFloor;
        S.low[t] = 0;
    }
    // the zero block, padding columns and what A reads past a panel stay zero
    for (int t = tid; t < kFxOperand / 16; t += kFxThreads) reinterpret_cast<uint4*>(smem)[t] = make_uint4(0, 0, 0, 0);
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&S.done[i], kIssuers);
            tc::mbar_init(&S.full[i], 1);
        }
        S.stop = 0;
        tc::mbar_init_fence();
    }
    if (warp == 0) {
        tc::tmem_alloc(&S.tmem, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = S.tmem;

    // steps of this CTA: periods strided over the CTAs, from the middle one on
    const int64_t nblk = (n + period * kFxK - 1) / (period * kFxK);
    const int nloc = (int64_t)blockIdx.x < nblk ? (int)((nblk - 1 - blockIdx.x) / gridDim.x + 1) : 0;
    const int nst = period * nloc;
    bool ok = true, bad = false;
    int issued = 0;              // steps handed to the issuing warps

    if (warp >= kFxConv / 32) {
        // ------------------------------------------------------------ issue
        // 640 threads are launched with 96 registers: this warpgroup gives up 72 of
        // them, the other four take 16 more (128 x 24 + 512 x 112 <= 640 x 96)
        asm volatile("setmaxnreg.dec.sync.aligned.u32 24;\n");
        const int share = warp - kFxConv / 32;
        const uint32_t idesc = tc::idesc_bf16_f32(128, mp);
        const uint32_t ds = (uint32_t)slice >> 4, db = (uint32_t)block >> 4;
        const uint32_t kz = (uint32_t)lbo_z >> 3, ku = (uint32_t)lbo_u >> 3;   // two core columns
        for (int st = 0; st < nst; ++st) {
            const bool w = tc::mbar_wait(&S.full[st & 1], (uint32_t)((st >> 1) & 1), kFxWait);
            if (!w || *reinterpret_cast<volatile int*>(&S.stop)) break;
            if (lane == 0) {
                tc::fence_after_sync();
                const uint32_t pu = tc::smem_u32(smem) + (uint32_t)((st & 1) * panel_of(mp)), pz = pu + 4 * lbo_u;
                const uint32_t carry = S.carry[st & 1];
                // descriptors: addresses in units of 16 bytes in the low bits
                const uint64_t hz = tc::smem_desc(pz, lbo_z, kCore), hu = tc::smem_desc(pu, lbo_u, kCore);
                auto mma_z = [&](uint32_t d, int k, int l, uint32_t accum) {
                    // [Z_k; Q_k] (rows) with Z_l (columns)
                    const uint64_t ad = hz + k * ds, bd = hz + l * ds;
                    tc::mma_bf16(d, ad, bd, idesc, accum);
                    tc::mma_bf16(d, ad + kz, bd + kz, idesc, 1u);
                };
                auto mma_u = [&](uint32_t d, int b, int l, uint32_t accum) {
                    // [U_b-1; U_b] (U_-1 = U_6 = 0) with Q_l
                    const uint64_t ad = hu + b * db, bd = hz + l * ds + db;
                    tc::mma_bf16(d, ad, bd, idesc, accum);
                    tc::mma_bf16(d, ad + ku, bd + kz, idesc, 1u);
                };
                auto levels_z = [&](int first, int last, uint32_t start) {
                    for (int L = first; L >= last; --L)
                        for (int k = 0; k <= L; ++k)
                            mma_z(tmem + (uint32_t)((L < 4 ? L : 4) * mp), k, L - k, k ? 1u : start);
                };
                auto levels_u = [&](int p, uint32_t start) {
                    for (int l = 0; l <= 2 * p + 1; ++l)
                        mma_u(tmem + (uint32_t)((5 + p) * mp), 2 * p + 1 - l, l, l ? 1u : start);
                };
                // every accumulator has one issuer, so the order of its sums is fixed
                if (share == 0) {            // levels 6 to 4, the finest first
                    for (int k = 1; k <= 5; ++k) mma_z(tmem + 4 * mp, k, 6 - k, k == 1 ? carry : 1u);
                    levels_z(5, 4, 1u);
                } else if (share == 1) {
                    levels_z(3, 0, carry);
                } else if (share == 2) {     // levels 6 and 7 (U_6 = 0), then 4 and 5
                    for (int l = 5; l >= 1; --l) mma_u(tmem + 7 * mp, 7 - l, l, l == 5 ? carry : 1u);
                    levels_u(2, 1u);
                } else {
                    levels_u(1, carry);
                    levels_u(0, carry);
                }
                tc::mma_commit(&S.done[st & 1]);
            }
            __syncwarp();
        }
    } else {
        // ------------------------------------------------------------ conversion and read-back
        asm volatile("setmaxnreg.inc.sync.aligned.u32 112;\n");
        // A warp converts 4 columns: thread's column j, rows row .. row + 3 of the step;
        // all rows of a column are in one warp, which agrees on its exponents by shuffles
        const int j = 4 * warp + (lane >> 3), row = 4 * (lane & 7);
        const bool conv = j < m, convw = 4 * warp < m;
        const int at = (j >> 3) * kCore + (j & 7) * 16 + 8 * (lane & 1), ki = (lane & 7) >> 1;
        const int at_u = ki * lbo_u + block + at, at_z = 4 * lbo_u + ki * lbo_z + at;
        // read-back: TMEM lane r, columns cq ncol .. + ncol - 1 of every accumulator
        const int q = warp & 3, cq = warp >> 2;
        const int ncol = mp / 4;
        const int r = 32 * q + lane;
        const bool reads = 32 * q < 2 * mp;
        const float odd = r < mp ? 1.0f : 0x1p9f;          // rows mp.. of the U accumulators hold the odd levels
        constexpr float fine = (float)(1ull << kUnit);
        unsigned long long az[16], au[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) { az[c] = 0; au[c] = 0; }

        double z[4], a[4], qv[4];
        int64_t r0 = 0;        // the thread's first row of the step being loaded
        auto start_of = [&](int st) {
            int p = st / period + nloc / 2;
            if (p >= nloc) p -= nloc;
            r0 = ((int64_t)blockIdx.x + (int64_t)p * gridDim.x) * (period * kFxK) + (int64_t)(st % period) * kFxK + row;
        };
        auto load4 = [&](int f, double* v) {
            const int64_t ld = S.cols.ld[f][j];
            const double* p = S.cols.p[f][j] + r0 * ld;
            if (r0 + 3 < n) {
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = __ldg(p + i * ld);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = r0 + i < n ? __ldg(p + i * ld) : 0.0;
            }
        };
        // Add the accumulators of the MMAs issued so far (the last of them for step
        // st) to the integers; false when the wait timed out.  full: some integer is
        // from 2^62 up.
        bool full = false;
        auto drain = [&](int st) -> bool {
            if (!tc::mbar_wait(&S.done[st & 1], (uint32_t)((st >> 1) & 1), kFxWait)) return false;
            tc::fence_after_sync();
            unsigned top = 0;
            if (reads) {
                const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(cq * ncol);
                constexpr unsigned long long kB = kMagic;
#pragma unroll
                for (int c = 0; c < 16; c += 8) {
                    if (c < ncol) {
                        uint32_t v[8];
                        auto get = [&](int i) {
                            tc::tmem_ld8(ta + i * mp + c, v);
                            tc::tmem_ld_wait();
                        };
                        get(0);
                        add8<kUnit>(az + c, v, 1.0f);
                        get(1);
                        add8<kUnit - 9>(az + c, v, 0x1p9f);
                        get(2);
                        add8<kUnit - 18>(az + c, v, 0x1p18f);
                        get(3);
                        add8<kUnit - 27>(az + c, v, 0x1p27f);
                        get(4);
                        add8<0>(az + c, v, fine);
                        get(5);
                        add8<kUnit>(au + c, v, odd);
                        get(6);
                        add8<kUnit - 18>(au + c, v, odd * 0x1p18f);
                        get(7);
                        add8<0>(au + c, v, odd * fine);
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            az[c + i] -= (kB << kUnit) + (kB << (kUnit - 9)) + (kB << (kUnit - 18)) +
                                         (kB << (kUnit - 27)) + kB;
                            au[c + i] -= (kB << kUnit) + (kB << (kUnit - 18)) + kB;
                            const int hz = (int)(az[c + i] >> 32), hu = (int)(au[c + i] >> 32);
                            top |= (unsigned)(hz ^ (hz >> 31)) | (unsigned)(hu ^ (hu >> 31));
                        }
                    }
                }
            }
            full = top >= 1u << 30;
            tc::fence_before_sync();
            return true;
        };
        // Add the integers to the CTA's partial sums (first: write them) and clear
        // them, 8 columns of each quarter at a time through shared memory.
        double* out = partial + (int64_t)blockIdx.x * 3 * m * m;
        auto emit = [&](bool first) {
            if (tid < 3 * mp) {
                const int jj = tid % mp;
                S.fac[tid] = jj < m ? scalbn(csc[jj], S.e[tid] - 1022) : 0.0;
            }
            auto group = [&](unsigned long long* acc, int c, bool u) {
                conv_sync();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    D[r * kLdD + 8 * cq + i] = (double)(long long)acc[i];
                    acc[i] = 0;
                }
                conv_sync();
                for (int t = tid; t < 128 * 32; t += kFxConv) {
                    const int i = t >> 5, cc = t & 31;
                    const int y = (cc >> 3) * ncol + c + (cc & 7);
                    if (y >= m || c + (cc & 7) >= ncol) continue;
                    // units of 2^-kUnit of a leading digit product; a column's leading digit is
                    // in units of 2^-9 2^(exponent - 1022).  One factor after the other: the product
                    // of two factors can leave the range (large column scales) where the sum is 0.
                    constexpr double unit = 1.0 / (double)(1ull << (18 + kUnit));
                    if (u) {
                        // even levels in row i, odd ones in row mp + i; the upper triangle, mirrored
                        if (i >= m || i > y) continue;
                        const double v = (D[i * kLdD + cc] + D[(mp + i) * kLdD + cc] * 0x1p-9) * unit *
                                         S.fac[2 * mp + i] * S.fac[mp + y];
                        double* o = out + m * m;
                        const double s = first ? v : o[i * m + y] + v;
                        o[i * m + y] = s;
                        o[y * m + i] = s;
                    } else {
                        const int x = i < mp ? i : i - mp;
                        if (i >= 2 * mp || x >= m) continue;
                        // (x, y) and (y, x) of Z^T Z are rounded alike
                        const int a = i < mp ? min(x, y) : i, b = i < mp ? max(x, y) : y;
                        const double v = D[i * kLdD + cc] * unit * S.fac[a] * S.fac[b];
                        double* o = out + (i < mp ? 0 : 2 * m * m) + x * m + y;
                        *o = first ? v : *o + v;
                    }
                }
            };
#pragma unroll
            for (int c = 0; c < 16; c += 8) {
                if (c < ncol) {
                    group(az + c, c, false);
                    group(au + c, c, true);
                }
            }
        };

        // one binade of room: a column then settles after a few steps (32,768 rows, m = 36:
        // 183 -> 145 us a call), and the leading digit of one whose magnitude hardly changes
        // stays below 2^7, without which level 2 passes 2^24 and loses up to 1.4e-12 |x| |y|
        constexpr int room = 2;
        int ez = kExpFloor, eu = kExpFloor, eq = kExpFloor;   // exponents of the thread's column
        int mz = 0, mu = 0, mq = 0;                           // largest exponent fields of the loaded values
        // U = AZ - sigma Z and the exponents of the loaded step
        auto prepare = [&]() {
            mz = mu = mq = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a[i] = fma(-sigma, z[i], a[i]);
                if (!has_q) qv[i] = a[i];
                mz = max(mz, exp_field(z[i]));
                mu = max(mu, exp_field(a[i]));
                mq = max(mq, exp_field(qv[i]));
            }
        };
        // the thread's values of column at_col are not all zero
        auto note_low = [&](const double* v, int at_col) {
            bool any = false;
#pragma unroll
            for (int i = 0; i < 4; ++i) any |= (__double_as_longlong(v[i]) << 1) != 0;
            if (any) S.low[at_col] = 1;
        };
        // raise the exponents of the warp's columns to the loaded values (too large ones,
        // Inf and NaN set the flag, Inf and NaN leave them alone); whether this thread's had to
        auto raise = [&]() -> bool {
            const bool up = mz >= ez || mu >= eu || mq >= eq;
            if (!__any_sync(0xffffffffu, up)) return false;
            if (max(mz, max(mu, mq)) >= kExpTop) bad = true;
            auto one = [&](int& e, int mx, int at_col) {
                int x = mx >= e && mx != 0x7ff ? mx + room : e;
                for (int o = 4; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
                e = x;
                if ((lane & 7) == 0 && conv) S.en[at_col] = x;
            };
            one(ez, mz, j);
            one(eq, mq, mp + j);
            one(eu, mu, 2 * mp + j);
            return up;
        };
        bool pending = false, first = true;    // accumulators hold products not yet added / nothing written yet
        auto load = [&]() {
            if (conv) {
                load4(0, z);
                load4(1, a);
                if (has_q) load4(2, qv);
            }
        };
        if (nst > 16) {
            // 32 rows spread over the CTA's share set the first exponents: smooth columns
            // then hardly ever outgrow them (m = 36, 262,144 rows: 370 -> 302 us)
            start_of((int)((int64_t)(lane & 7) * nst / 8));
            load();
            if (conv) prepare();
            if (convw) raise();
            conv_sync();
            if (tid < 3 * mp) S.e[tid] = S.en[tid];
        }
        if (nst > 0) {
            start_of(0);
            load();
        }
        // one step more than there is: it drains the last period and writes the sums
        for (int st = 0; st <= nst; ++st) {
            const bool last = st == nst;
            bool grow = false, w = true;
            if (!last) {
                if (conv) prepare();
                if (convw) grow = raise();
                if (conv && min(ez, min(eu, eq)) == kExpFloor) {
                    if (ez == kExpFloor) note_low(z, j);
                    if (eq == kExpFloor) note_low(qv, mp + j);
                    if (eu == kExpFloor) note_low(a, 2 * mp + j);
                }
                // the MMAs of two steps ago have read this panel
                if (st >= 2) w = tc::mbar_wait(&S.done[st & 1], (uint32_t)(((st >> 1) - 1) & 1), kFxWait);
                unsigned char* pan = smem + (st & 1) * panel_of(mp);
                const bool more = st + 1 < nst;
                if (more) start_of(st + 1);
                if (conv) {
                    put_digits(pan + at_u, block, a, eu);
                    if (more) load4(1, a);
                    put_digits(pan + at_z, slice, z, ez);
                    if (more) load4(0, z);
                    put_digits(pan + at_z + block, slice, qv, eq);
                    if (more && has_q) load4(2, qv);
                }
                tc::fence_async_smem();

            }
            const bool any = conv_any(grow || !w);     // new exponents (or a wait that timed out)
            bool out_now = last;
            if (any && conv_any(!w)) { ok = false; break; }
            if (pending && (last || any || st % period == 0)) {
                w = drain(st - 1);
                pending = false;
                if (conv_any(!w || full)) {
                    if (conv_any(!w)) { ok = false; break; }
                    out_now = true;
                }
            }
            if (out_now) {
                emit(first);
                first = false;
                conv_sync();
                if (last) break;
            }
            if (any) {
                if (r < 2 * mp) {
                    // rows Z, Q against columns Z; rows U (twice) against columns Q
                    const int ru = 2 * mp + (r < mp ? r : r - mp);
                    const int dz = S.en[r] - S.e[r], du = S.en[ru] - S.e[ru];
                    auto down = [](unsigned long long x, int sh) -> unsigned long long {
                        return sh <= 0 ? x : sh > 62 ? 0 : (unsigned long long)(((long long)x + (1LL << (sh - 1))) >> sh);
                    };
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        if (c < ncol) {
                            const int pc = cq * ncol + c;
                            az[c] = down(az[c], dz + S.en[pc] - S.e[pc]);
                            au[c] = down(au[c], du + S.en[mp + pc] - S.e[mp + pc]);
                        }
                    }
                }
                conv_sync();
                if (tid < 3 * mp) S.e[tid] = S.en[tid];
                conv_sync();
            }
            if (tid == 0) {
                S.carry[st & 1] = pending ? 1u : 0u;
                tc::mbar_arrive(&S.full[st & 1]);
            }
            pending = true;
            ++issued;
        }
        if (tid < 3 * mp && S.low[tid] && S.e[tid] == kExpFloor) bad = true;
        if (!ok && tid == 0) {       // let the issuing warps go
            S.stop = 1;
            tc::mbar_arrive(&S.full[issued & 1]);
        }
    }
    bool redo = __syncthreads_or(!ok || bad);
    if (redo && issued > 0)   // bounded wait for the MMAs in flight before their memory is released
        tc::mbar_wait(&S.done[(issued - 1) & 1], (uint32_t)(((issued - 1) >> 1) & 1), kFxWait);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 512);
    }
    if (tid == 0) flags[blockIdx.x] = redo ? 1 : 0;
}

}  // namespace

// partial: grid * 3 m^2 doubles and grid ints behind them.  *grid_out CTAs
// wrote a partial sum and a flag each.
cudaError_t gram_fx_launch(int64_t n, int nb, const Blk<const double>* Z, const Blk<const double>* AZ,
                           const Blk<const double>* Q, double sigma, const double* colscale, double* partial,
                           int* grid_out, int** flags_out, cudaStream_t s) {
    FxCols C{};
    int m = 0;
    for (int b = 0; b < nb; ++b)
        for (int c = 0; c < Z[b].nc; ++c, ++m) {
            if (m >= 64) return cudaErrorInvalidValue;
            C.p[0][m] = Z[b].p + c;
            C.p[1][m] = AZ[b].p + c;
            C.p[2][m] = Q ? Q[b].p + c : nullptr;
            C.ld[0][m] = Z[b].ld;
            C.ld[1][m] = AZ[b].ld;
            C.ld[2][m] = Q ? Q[b].ld : 0;
        }
    const int mp = (m + 15) / 16 * 16;
    // steps per period: long ones read the accumulators back less often (about one
    // step's time), short ones spread few rows over more CTAs
    const int64_t steps = (n + kFxK - 1) / kFxK;
    int period = kMaxPeriod, grid = 1;
    int64_t best = -1;
    for (int p = kMaxPeriod; p >= 1; --p) {
        const int64_t blocks = (steps + p - 1) / p;
        const int64_t cost = (blocks + sm_count() - 1) / sm_count() * (p + 1);
        if (best < 0 || cost < best) {
            best = cost;
            period = p;
            grid = blocks < sm_count() ? (blocks > 0 ? (int)blocks : 1) : sm_count();
        }
    }
    int* flags = reinterpret_cast<int*>(partial + (int64_t)grid * 3 * m * m);
    // above the 48 KB default, on every device a process uses
    cudaError_t e = cudaFuncSetAttribute(k_gram_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, kFxSmem);
    if (e != cudaSuccess) return e;
    k_gram_fx<<<grid, kFxThreads, kFxSmem, s>>>(n, m, mp, C, Q ? 1 : 0, sigma, colscale, partial, flags,
                                                  period);
    count_launches(1);
    *grid_out = grid;
    *flags_out = flags;
    return cudaGetLastError();
}

}  // namespace plhr
