// FP32 block sampling for bands wider than 16: a register-tiled correlation.
//
// On a neighbour ring of the same pixel count the kernel value of (q, p)
// depends on s = p - q alone, so the row sum is the correlation
//   M[q][q-d] += sum_s (T[|s|] N[q+s]) T[|s+d|],  |s|, |s+d| < K,
// and most of a band's terms are of this kind (92 % for beams of 10' to 60' at
// l_max 1000).  A thread takes 8 columns q and 4 offsets d: per s it forms the
// 8 weights and does 32 multiply-adds with three values in flight, the map's
// and the kernel's windows sliding through registers by one 16-byte shared
// load each per four s.  T is staged symmetric around s = 0 and with zeros
// past K - 1, the map as the tile's run of the ring, for eight rings between
// two barriers.  The last of the four offsets ends up to three terms early;
// those terms are products with a staged zero, which leave the sum as it is.
// A thread holds two groups of offsets, the g-th from the front and from the
// back, so that every thread has the same number of terms.  Each element is
// the same sum, in the same order and rounding, as in k_sample_pband, whose
// fully unrolled correlation of one column per thread covers K <= 17 and is
// held up by instruction fetches (tens of KB of code, each instruction used
// once per ring); the rest there takes about 15 instructions a term.  Four
// operators of 10' to 60' at l_max 1000 (2.8e10 terms, w up to 51): 10.4 ->
// 7.1 ms.  For 8 < w <= 16 the unrolled kernel stays: few terms per staged
// value (0.03 ms slower at l_max 3000 with 64 such blocks).  A product of
// staged weight and kernel tiles for every ring pair took 12.4 ms.
//
// Other ring pairs, and maps or tables with values of 1e19 and above, whose
// product might not be finite (0 x inf is not 0), take the direct walk: one element at a time, into shared memory, from where
// the threads add it to their sums.
#include <algorithm>

#include "sympix_sample_kernels.cuh"

namespace sympix {

constexpr int kWideCols = 128;   // columns of a CTA (the plan's sampling tile)
constexpr int kWalkCols = 64;    // columns walked directly at a time
constexpr int kWideRings = 8;    // rings staged between two barriers
constexpr int kWideKMax = 33;    // kernel values of a same-count ring: w <= 64
constexpr int kWideMap = kWideCols + 2 * kWideKMax + 14;   // staged map values per ring (a multiple of 4)
constexpr int kWideTab = (2 * kWideKMax - 1 + 7 + 3) / 4 * 4 + 4;  // staged kernel values per ring

// floor(a / d) for d > 0 and |a / d| < 2^20 (inv = 1 / d)
__device__ __forceinline__ int wide_floor(int a, int d, float inv) {
    int q = __float2int_rd((float)a * inv);
    const int r = a - q * d;
    q += r < 0 ? -1 : r >= d ? 1 : 0;
    return q;
}

// Arc length up to which the walk's weights are staged, for width w.
__host__ __device__ constexpr int wide_arc(int w) { return w + 16; }

// acc[a][b] += sum_s W_a(s) T[|s + d0 + b|] for columns a, offsets d0 + b;
// nm: the map at column a = 0, s = -(K-1); tab: T at s = -(K-1) (both 16-byte aligned).
__device__ __forceinline__ void wide_sweep(float (&acc)[8][4], int d0, int K, const float *nm, const float *tab) {
    const int len = 2 * K - 1 - d0;
    if (len <= 0) return;
    const float4 *n4 = reinterpret_cast<const float4 *>(nm), *t4 = reinterpret_cast<const float4 *>(tab);
    const float4 *u4 = reinterpret_cast<const float4 *>(tab + d0);
    float nw[12], tw[8];
    *reinterpret_cast<float4 *>(nw) = n4[0];
    *reinterpret_cast<float4 *>(nw + 4) = n4[1];
    *reinterpret_cast<float4 *>(tw) = u4[0];
    for (int i = 0; 4 * i < len; ++i) {
        *reinterpret_cast<float4 *>(nw + 8) = n4[i + 2];
        *reinterpret_cast<float4 *>(tw + 4) = u4[i + 1];
        const float4 t = t4[i];
        const float ts[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const float wv = ts[u] * nw[u + a];
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(wv, tw[u + b], acc[a][b]);
            }
        }
#pragma unroll
        for (int a = 0; a < 8; ++a) nw[a] = nw[a + 4];
#pragma unroll
        for (int b = 0; b < 4; ++b) tw[b] = tw[b + 4];
    }
}

template <int NT>
__global__ void __launch_bounds__(NT, 512 / NT) k_sample_wide32(
    const SampleItem *__restrict__ items, const BlockDesc *__restrict__ blocks, const PairEntry *__restrict__ entries,
    int64_t nslots, int64_t npix, const float *__restrict__ tb32, const float *__restrict__ td32,
    const float *__restrict__ ninv32, double *__restrict__ out) {
    constexpr int KTOP = 17;  // as in k_sample_pband
    // the staged rings, or one ring's directly walked sums [offset][column] and weights [pixel][column]
    extern __shared__ __align__(16) float wide_smem[];
    const SampleItem it = items[blockIdx.x];
    const BlockDesc bd = blocks[it.block];
    const int n = bd.n, w = bd.w, q0 = it.q0, nq = min(kWideCols, n - q0);
    const int nd = (w + 4) / 4, qt = threadIdx.x & 15, pr = threadIdx.x >> 4;
    const int qa = q0 + 8 * qt;
    // offset groups of this thread: d = 4 pr .. and 4 (nd - 1 - pr) ..
    const int da = 4 * pr, db = 4 * (nd - 1 - pr);
    const bool two = db > da, work = qa < n && db >= da;
    const float *tb = tb32 + (int64_t)bd.op * nslots, *nv = ninv32 + (int64_t)bd.op * npix;
    float acca[8][4], accb[8][4];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acca[a][b] = accb[a][b] = 0.0f;
    int e = 0;
    while (e < bd.npairs) {
        // a run of same-count rings, up to kWideRings
        int ne = 0;
        while (ne < kWideRings && e + ne < bd.npairs) {
            const PairEntry &pe = entries[bd.pair0 + e + ne];
            if (pe.P != 1 || pe.Q != 1) break;
            ++ne;
        }
        bool bad = false;
        __syncthreads();  // what was staged before is used
        for (int k = 0; k < ne; ++k) {
            const PairEntry pe = entries[bd.pair0 + e + k];
            const int K = pe.mmax / 2 + 1;
            float *nm = wide_smem + k * kWideMap, *tt = wide_smem + kWideRings * kWideMap + k * kWideTab;
            const float *N = nv + pe.noff, *T = tb + pe.tab;
            for (int i = threadIdx.x; i < kWideMap; i += NT) {  // columns q0 - (K-1) + i of the ring
                float v = 0.0f;
                if (i < nq + 2 * K - 2) {
                    int p = q0 - (K - 1) + i;
                    p += p < 0 ? n : 0;
                    p -= p >= n ? n : 0;
                    v = N[(int64_t)p * pe.nstride];
                }
                bad |= !(fabsf(v) < 1e19f);
                nm[i] = v;
            }
            for (int i = threadIdx.x; i < kWideTab; i += NT) {
                const int s = i - (K - 1), as = s < 0 ? -s : s;
                const float v = as < K ? T[as] : 0.0f;
                bad |= !(fabsf(v) < 1e19f);
                tt[i] = v;
            }
        }
        bad = __syncthreads_or(bad);
        if (ne > 0 && !bad) {
            if (work)
                for (int k = 0; k < ne; ++k) {
                    const int K = entries[bd.pair0 + e + k].mmax / 2 + 1;
                    const float *nm = wide_smem + k * kWideMap + 8 * qt, *tt = wide_smem + kWideRings * kWideMap + k * kWideTab;
                    if (K <= KTOP) {  // summed into the element itself
                        wide_sweep(acca, da, K, nm, tt);
                        if (two) wide_sweep(accb, db, K, nm, tt);
                    } else {
                        float s[8][4];
#pragma unroll 1
                        for (int g = 0; g < (two ? 2 : 1); ++g) {
#pragma unroll
                            for (int a = 0; a < 8; ++a)
#pragma unroll
                                for (int b = 0; b < 4; ++b) s[a][b] = 0.0f;
                            wide_sweep(s, g ? db : da, K, nm, tt);
#pragma unroll
                            for (int a = 0; a < 8; ++a)
#pragma unroll
                                for (int b = 0; b < 4; ++b) {
                                    if (g)
                                        accb[a][b] += s[a][b];
                                    else
                                        acca[a][b] += s[a][b];
                                }
                        }
                    }
                }
            e += ne;
            continue;
        }
        // one ring by the direct walk
        const PairEntry pe = entries[bd.pair0 + e];
        const int P = pe.P, Q = pe.Q, m = pe.mmax, par = pe.par, D2 = 2 * P;
        const float inv = 1.0f / (float)D2;
        const float *T = tb + pe.tab, *N = nv + pe.noff;
        const bool direct = P == 1 && Q == 1 && m / 2 + 1 <= KTOP;
        const int arc = m / P + 1;
        const bool staged = arc <= wide_arc(w);
        float *sums = wide_smem, *wt = wide_smem + (w + 1) * kWalkCols;
        for (int c0 = 0; c0 < nq; c0 += kWalkCols) {
            const bool mine = work && 8 * qt >= c0 && 8 * qt < c0 + kWalkCols;
            const int col = 8 * qt - c0, nc = min(kWalkCols, nq - c0);
            __syncthreads();  // the columns before are added
            if (direct && mine) {  // the walk goes on from the element
#pragma unroll
                for (int a = 0; a < 8; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        if (da + b <= w) sums[(da + b) * kWalkCols + col + a] = acca[a][b];
                        if (two && db + b <= w) sums[(db + b) * kWalkCols + col + a] = accb[a][b];
                    }
            }
            // the weights of every column's arc (while it fits), then the walk:
            // a weight and a kernel value a term
            if (staged)
                for (int i = threadIdx.x; i < arc * kWalkCols; i += NT) {
                    const int j = i / kWalkCols, c = i % kWalkCols, Zq = (2 * (q0 + c0 + c) + 1) * Q;
                    const int f = wide_floor(Zq - m - P + D2 - 1, D2, inv), z = Zq - (2 * (f + j) + 1) * P;
                    if (c >= nc || -z > m) continue;
                    int pm = (f + j) % pe.nrho;
                    if (pm < 0) pm += pe.nrho;
                    wt[i] = T[((z < 0 ? -z : z) - par) >> 1] * N[(int64_t)pm * pe.nstride];
                }
            __syncthreads();
            for (int i = threadIdx.x; i < (w + 1) * kWalkCols; i += NT) {
                const int d = i / kWalkCols, c = i % kWalkCols;
                if (c >= nc) continue;
                const int Zq = (2 * (q0 + c0 + c) + 1) * Q, f = wide_floor(Zq - m - P + D2 - 1, D2, inv);
                const int l = wide_floor(Zq - 2 * d * Q + m - P, D2, inv);
                float v = direct ? sums[i] : 0.0f;
                int z = Zq - (2 * f + 1) * P;
                if (staged) {
                    const float *x = wt + c;
                    z -= 2 * d * Q;
                    for (int p = f; p <= l; ++p) {
                        v = fmaf(*x, T[((z < 0 ? -z : z) - par) >> 1], v);
                        x += kWalkCols;
                        z -= D2;
                    }
                } else if (l >= f) {
                    int pm = f % pe.nrho;
                    if (pm < 0) pm += pe.nrho;
                    for (int p = f; p <= l; ++p) {
                        const int zr = z - 2 * d * Q;
                        const float x = T[((z < 0 ? -z : z) - par) >> 1] * N[(int64_t)pm * pe.nstride];
                        v = fmaf(x, T[((zr < 0 ? -zr : zr) - par) >> 1], v);
                        z -= D2;
                        if (++pm == pe.nrho) pm = 0;
                    }
                }
                sums[i] = v;
            }
            __syncthreads();
            if (mine) {
#pragma unroll
                for (int a = 0; a < 8; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        if (da + b <= w) {
                            const float v = sums[(da + b) * kWalkCols + col + a];
                            acca[a][b] = direct ? v : acca[a][b] + v;
                        }
                        if (two && db + b <= w) {
                            const float v = sums[(db + b) * kWalkCols + col + a];
                            accb[a][b] = direct ? v : accb[a][b] + v;
                        }
                    }
            }
        }
        ++e;
    }
    if (!work) return;
    const float *td = td32 + (int64_t)bd.op * nslots + bd.dtab;
    auto put = [&](const float (&acc)[8][4], int d0) {
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            const int q = qa + a;
            if (q >= n) continue;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int d = d0 + b;
                if (d <= w)
                    out[bd.off_pband + (int64_t)q * (w + 1) + d] = f32_to_f64_bits(d < bd.dK ? acc[a][b] + td[d] : acc[a][b]);
            }
        }
    };
    put(acca, da);
    if (two) put(accb, db);
}

template <int NT>
static void launch_wide32(sympix_plan_t pl, int list, double *blocks, cudaStream_t st) {
    if (pl->items_wide[list].empty()) return;
    const int w = pl->wide_list_w[list];
    const size_t staged = kWideRings * (size_t)(kWideMap + kWideTab), walked = (size_t)(w + 1 + wide_arc(w)) * kWalkCols;
    const size_t smem = std::max(staged, walked) * sizeof(float);  // at most 37 KB: no limit to raise
    k_sample_wide32<NT><<<(unsigned)pl->items_wide[list].size(), NT, smem, st>>>(
        pl->d_items_wide[list].p, pl->d_blocks.p, pl->d_entries.p, pl->nslots, pl->grid->npix, pl->d_tab_b32.p,
        pl->d_tab_d32.p, pl->d_ninv32.p, blocks);
}

// The plan's work lists (periodic bands of 17 .. 31, 32 .. 47 and 48 .. 64).
void launch_sample_wide32(sympix_plan_t pl, double *blocks, cudaStream_t st) {
    launch_wide32<64>(pl, 0, blocks, st);
    launch_wide32<96>(pl, 1, blocks, st);
    launch_wide32<160>(pl, 2, blocks, st);
}

}  // namespace sympix
