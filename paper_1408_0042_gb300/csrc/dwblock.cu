// Double-word form of the coefficient update on FP64 blocks, for the FP64
// phase of the mixed-precision solve.  The inputs are
// split once into double-word values (hi = the leading 24 bits, lo = the
// rest rounded to FP32: ~48-bit significands, dw_split_trunc); products are
// formed with the FMA exact product of the high
// parts plus the FP32 cross terms, and sums are accumulated with TwoSum on the
// high part, so every result carries ~2^-46 relative error of the sum of
// |terms| - FP64-class accuracy for the projected problem at a fraction of the
// FP64 pipe's cost on GB300.  Results are FP64.
#include "blockops.h"
#include "dword.h"

namespace plhr {
namespace {

struct FamD {
    const double* p[4];
    int64_t ld[4];
    int nc[4];
    int off[4];
};

FamD fam_d(const Blk<const double>* b, int nb) {
    FamD F{};
    int off = 0;
    for (int i = 0; i < 4; ++i) {
        if (i < nb) {
            F.p[i] = b[i].p; F.ld[i] = b[i].ld; F.nc[i] = b[i].nc; F.off[i] = off;
            off += b[i].nc;
        } else {
            F.p[i] = nullptr; F.ld[i] = 0; F.nc[i] = 0; F.off[i] = off;
        }
    }
    return F;
}


// Pout = F C_P, Vout = F_0 C_VV + F C_P in double-word arithmetic on FP64
// blocks (in place allowed: every output row depends only on the same input
// row and a chunk is staged before any of its rows is written)
// Thread t owns column j = t % kp of rows r = t / kp and r + `rows` of each chunk
// of 2 `rows` rows: the two rows share the coefficient loads and give each thread two
// independent sums.  Every output is summed over i in the same order as with one
// output per thread.  A chunk has as many rows as the threads allow, so that no warp
// idles where k' does not divide 256 (both families of an iteration at
// 112 x 96 x 80: 788 -> 692 us; fetching the next chunk into registers meanwhile
// was 4 % slower at 128^3, k' = 16).
__global__ void __launch_bounds__(256) k_update_dw(int64_t n, int m, int kp, int nb, int rows, FamD F,
                                                   const double* __restrict__ Cp, const double* __restrict__ Cvv,
                                                   double* __restrict__ Vout, int64_t ldvo, double* __restrict__ Pout,
                                                   int64_t ldpo) {
    extern __shared__ __align__(16) unsigned char raw[];
    dw* cp = reinterpret_cast<dw*>(raw);      // [m][kp]
    dw* cv = cp + m * kp;                     // [kp][kp]
    dw* zr = cv + kp * kp;                    // [2 rows][m]
    for (int t = threadIdx.x; t < m * kp; t += blockDim.x) cp[t] = dw_from_double(Cp[t]);
    for (int t = threadIdx.x; t < kp * kp; t += blockDim.x) cv[t] = dw_from_double(Cvv[t]);
    const int tid = threadIdx.x, chunk = 2 * rows, r0 = tid / kp, j = tid - r0 * kp;
    const int64_t nchunks = (n + chunk - 1) / chunk;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const int64_t row0 = ch * chunk;
        const int nrows = (int)((n - row0) < chunk ? (n - row0) : chunk);
        __syncthreads();
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (b >= nb) break;
            const int nc = F.nc[b];
            for (int t = tid; t < nrows * nc; t += 256) {
                const int r = t / nc, c = t - r * nc;
                zr[r * m + F.off[b] + c] = dw_split_trunc(F.p[b][(row0 + r) * F.ld[b] + c]);
            }
        }
        __syncthreads();
        if (r0 >= rows || r0 >= nrows) continue;
        const bool two = r0 + rows < nrows;
        const dw* z0 = zr + r0 * m;
        const dw* z1 = zr + (two ? r0 + rows : r0) * m;
        float ph0 = 0.0f, pl0 = 0.0f, ph1 = 0.0f, pl1 = 0.0f;
        for (int i = 0; i < m; ++i) {
            const dw c = cp[i * kp + j];
            dw_fma_acc(ph0, pl0, z0[i], c);
            dw_fma_acc(ph1, pl1, z1[i], c);
        }
        float vh0 = ph0, vl0 = pl0, vh1 = ph1, vl1 = pl1;
        for (int i = 0; i < kp; ++i) {
            const dw c = cv[i * kp + j];
            dw_fma_acc(vh0, vl0, z0[i], c);
            dw_fma_acc(vh1, vl1, z1[i], c);
        }
        const int64_t row = row0 + r0;
        Pout[row * ldpo + j] = dw_to_double_fast(dw{ph0, pl0});
        Vout[row * ldvo + j] = dw_to_double_fast(dw{vh0, vl0});
        if (two) {
            Pout[(row + rows) * ldpo + j] = dw_to_double_fast(dw{ph1, pl1});
            Vout[(row + rows) * ldvo + j] = dw_to_double_fast(dw{vh1, vl1});
        }
    }
}

}  // namespace

cudaError_t block_update_dw(int64_t n, int nb, const Blk<const double>* F, int kp, const double* Cp, const double* Cvv,
                            double* Vout, int64_t ldvo, double* Pout, int64_t ldpo, cudaStream_t s) {
    FamD FF = fam_d(F, nb);
    int m = 0, widest = kp;
    for (int i = 0; i < nb; ++i) {
        m += F[i].nc;
        widest = F[i].nc > widest ? F[i].nc : widest;
    }
    if (widest > 256) return cudaErrorInvalidValue;
    const int rows = 256 / widest;   // a family's values of a chunk: at most two per thread
    const size_t shm = sizeof(dw) * (m * kp + kp * kp + 2 * rows * m);
    k_update_dw<<<sm_count() * 4, 256, shm, s>>>(n, m, kp, nb, rows, FF, Cp, Cvv, Vout, ldvo, Pout, ldpo);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace plhr
