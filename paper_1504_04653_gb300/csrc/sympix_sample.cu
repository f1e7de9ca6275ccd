// Block sampling: M_qr = D^_qr + sum_p B^_pq N^-1_p B^_pr for q, r on the
// block's ring (Eq. Dhat, Eq. system-rewritten; Y2 = Y1).
//
// For a coupled neighbour ring rho with pair constants (P, Q, mmax) pixel q
// couples to the pixels p with |z| <= mmax, z = (2q+1)Q - (2p+1)P (a
// contiguous arc), and r = q - d couples to p iff |z - 2dQ| <= mmax.  The
// kernel value of (q, p) is table[(|z| - par) / 2].  One thread owns one
// column q of its block and accumulates the whole lower band row
// M[q][q-d], d = 0..w, in registers: per pixel p it forms w_p = B^_pq N^-1_p
// once and adds w_p B^_pr to every d whose arc holds p.
//
// Arithmetic (template PREC):
//   0  FP64 products and sums;
//   1  FP32 products and sums (kernel values and N^-1 rounded to FP32);
//   2  split FP32: every value is an unevaluated sum hi + lo of two floats,
//      products by the exact FMA-based two-product, sums by two-sum with
//      renormalisation, i.e. ~44-bit significands on the FP32 pipes.
#include "sympix_arith.cuh"
#include "sympix_internal.cuh"

namespace sympix {

template <int PREC, bool DENSE_OUT>
void launch_pband(sympix_plan_t pl, const double *ninv, double *blocks, cudaStream_t st);

// N^-1 split once per call into FP32 (hi, lo) planes, so the contraction
// never converts from FP64 in its inner loops.
__global__ void k_split_ninv(int64_t count, const double *__restrict__ ninv, float *__restrict__ n32,
                             float *__restrict__ nlo) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const F2 v = f2_from_bits(ninv[i]);
    n32[i] = v.hi;
    nlo[i] = v.lo;
}

// z reduced to (-half, half] (T2 = 2 half): the longitude separation index
// of a pixel pair on a pair of rings, as the kernel table is indexed.  Dense
// blocks have at most 8192 pixels and rings 30000, so that every index and
// T2 = 2 P n_rho fit 32 bits.
__device__ __forceinline__ int wrap_half(int z, int half, int T2) {
    z %= T2;
    if (z > half) z -= T2;
    if (z <= -half) z += T2;
    return z;
}

// Small or wrapping blocks (every pixel pair of the ring may couple), FP64.
// A CTA takes row q and up to 64 columns r <= q (M is symmetric: (r, q) is
// stored with (q, r)).  For eight neighbour rings at a time each of its eight
// warps forms one ring's weights b(q, p) N^-1_p over the pixels coupled to q
// (the arc |z_q| <= mmax, or the whole ring when the support covers it),
// kDensePix at a time; then warp k sums over them for the columns r = k, k + 8,
// ..., its lanes sharing the pixels, separation indices reduced to |dphi| <=
// pi and moved by a fixed step.  The partial sums meet in a fixed-order
// shuffle tree.  Bound by the FP64 pipe and the integer work per pixel: one
// multiply-add a pixel, half the pairs, against a product and a multiply-add
// for every (q, r) in 64-bit index arithmetic before (72 blocks of up to 128
// pixels at l_max 1000: 2.0 -> 0.35 ms).
constexpr int kDensePix = 256, kDenseWarps = 8, kDenseCols = 64;

__global__ void __launch_bounds__(32 * kDenseWarps) k_sample_dense(const SampleItem *__restrict__ items,
                                                                   const BlockDesc *__restrict__ blocks,
                                                                   const PairEntry *__restrict__ entries,
                                                                   int64_t nslots, int64_t npix,
                                                                   const double *__restrict__ tb,
                                                                   const double *__restrict__ td,
                                                                   const double *__restrict__ ninv,
                                                                   double *__restrict__ out, int dense_storage) {
    constexpr int NR = kDenseCols / kDenseWarps;
    __shared__ double wgt[kDenseWarps][kDensePix];
    __shared__ int s_len[kDenseWarps], s_pm[kDenseWarps];
    const SampleItem it = items[blockIdx.x];
    const BlockDesc bd = blocks[it.block];
    const int n = bd.n, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = it.q0 & 0xffff, r0 = (it.q0 >> 16) * kDenseCols + warp;
    const int64_t tbase = (int64_t)bd.op * nslots;
    const double *nv = ninv + (int64_t)bd.op * npix;
    double acc[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) acc[k] = 0.0;
    for (int e0 = 0; e0 < bd.npairs; e0 += kDenseWarps) {
        for (int c0 = 0;; c0 += kDensePix) {
            __syncthreads();  // the weights before are used
            int left = 0;     // pixels of this warp's ring from c0 on
            if (e0 + warp < bd.npairs) {
                const PairEntry pe = entries[bd.pair0 + e0 + warp];
                const int P = pe.P, m = pe.mmax, nr = pe.nrho, half = P * nr, T2 = 2 * half, d2 = 2 * P;
                const int Zq = (2 * q + 1) * pe.Q;
                int lo = 0, hi = nr - 1;
                if (m < half) {  // ceil((Z - m - P) / 2P) .. floor((Z + m - P) / 2P)
                    const int a = Zq - m - P, b = Zq + m - P;
                    lo = a >= 0 ? (a + d2 - 1) / d2 : -((-a) / d2);
                    hi = b >= 0 ? b / d2 : -((-b + d2 - 1) / d2);
                }
                const int len = hi - lo + 1;
                int pm0 = lo % nr;
                if (pm0 < 0) pm0 += nr;
                left = len - c0;
                if (lane == 0) {
                    s_len[warp] = left;
                    s_pm[warp] = pm0;
                }
                for (int i = lane; i < min(left, kDensePix); i += 32) {
                    const int pm = (pm0 + c0 + i) % nr;
                    const int z = wrap_half(Zq - (2 * pm + 1) * P, half, T2), az = z < 0 ? -z : z;
                    wgt[warp][i] = az <= m ? tb[tbase + pe.tab + ((az - pe.par) >> 1)] *
                                                 nv[pe.noff + (int64_t)pm * pe.nstride]
                                           : 0.0;
                }
            } else if (lane == 0) {
                s_len[warp] = 0;
            }
            const int more = __syncthreads_or(left > kDensePix);
            for (int k = 0; k < kDenseWarps; ++k) {
                const int len = min(s_len[k], kDensePix);
                if (len <= 0) continue;
                const PairEntry pe = entries[bd.pair0 + e0 + k];
                const int P = pe.P, m = pe.mmax, nr = pe.nrho, half = P * nr, T2 = 2 * half;
                const double *T = tb + tbase + pe.tab;
                // the lane's next pixel is 32 on (mod nr): z moves by a step reduced once
                const int dz = 2 * P * (32 % nr), pm = (s_pm[k] + c0 + lane) % nr;
#pragma unroll
                for (int u = 0; u < NR; ++u) {
                    const int r = r0 + kDenseWarps * u;
                    if (r > q) break;  // uniform in the warp
                    int z = wrap_half((2 * r + 1) * pe.Q - (2 * pm + 1) * P, half, T2);
                    double v = acc[u];
                    for (int i = lane; i < len; i += 32) {
                        const int az = z < 0 ? -z : z;
                        if (az <= m) v = fma(wgt[k][i], T[(az - pe.par) >> 1], v);
                        z -= dz;
                        if (z <= -half) z += T2;
                    }
                    acc[u] = v;
                }
            }
            if (!more) break;
        }
    }
    double *M = out + (dense_storage ? bd.off_dense : bd.off_pband);
#pragma unroll
    for (int u = 0; u < NR; ++u) {
        const int r = r0 + kDenseWarps * u;
        if (r > q) break;
        double v = acc[u];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0) {
            int k = q - r;
            if (n - k < k) k = n - k;
            if (k < bd.dK) v += td[tbase + bd.dtab + k];
            M[(int64_t)q * n + r] = v;
            M[(int64_t)r * n + q] = v;
        }
    }
}

}  // namespace sympix

using namespace sympix;

extern "C" int sympix_sample_blocks(sympix_plan_t pl, const double *ninv, int precision, int storage,
                                    double *blocks, void *stream) {
    if (!pl || !ninv || !blocks) return set_error(SYMPIX_EINVAL, "sympix_sample_blocks: NULL argument");
    if (precision < SYMPIX_PREC_FP64 || precision > SYMPIX_PREC_FP32X2)
        return set_error(SYMPIX_EINVAL, "sympix_sample_blocks: unknown precision %d", precision);
    if (storage != SYMPIX_STORE_PBAND && storage != SYMPIX_STORE_DENSE)
        return set_error(SYMPIX_EINVAL, "sympix_sample_blocks: unknown storage %d", storage);
    if (!pl->table_ready)
        return set_error(SYMPIX_EINVAL, "sympix_sample_blocks: sympix_kernel_table has not been called");
    cudaStream_t st = (cudaStream_t)stream;
    const bool dense = storage == SYMPIX_STORE_DENSE;
    trace_mark(pl, st, nullptr);
    if (dense) SPX_CUDA(cudaMemsetAsync(blocks, 0, (size_t)pl->size_dense * sizeof(double), st));
    if (precision != SYMPIX_PREC_FP64) {
        const int64_t cnt = (int64_t)pl->nops * pl->grid->npix;
        k_split_ninv<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, ninv, pl->d_ninv32.p, pl->d_ninvlo.p);
        trace_mark(pl, st, "k_split_ninv");
    }
    if (pl->tiles) {  // band blocks of a DP grid
        int rc = launch_tiles(pl, ninv, precision, blocks, st);
        if (rc) return rc;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_error(e, "sympix_sample_blocks: launch");
        return SYMPIX_OK;
    }
    if (precision == SYMPIX_PREC_FP64) {
        dense ? launch_pband<0, true>(pl, ninv, blocks, st) : launch_pband<0, false>(pl, ninv, blocks, st);
    } else if (precision == SYMPIX_PREC_FP32) {
        dense ? launch_pband<1, true>(pl, ninv, blocks, st) : launch_pband<1, false>(pl, ninv, blocks, st);
    } else {
        dense ? launch_pband<2, true>(pl, ninv, blocks, st) : launch_pband<2, false>(pl, ninv, blocks, st);
    }
    trace_mark(pl, st, "k_sample_pband");
    if (!pl->items_dense.empty())
        k_sample_dense<<<(unsigned)pl->items_dense.size(), 32 * kDenseWarps, 0, st>>>(
            pl->d_items_dense.p, pl->d_blocks.p, pl->d_entries.p, pl->nslots, pl->grid->npix, pl->d_tab_b.p,
            pl->d_tab_d.p, ninv, blocks, dense ? 1 : 0);
    trace_mark(pl, st, "k_sample_dense");
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "sympix_sample_blocks: launch");
    return SYMPIX_OK;
}
