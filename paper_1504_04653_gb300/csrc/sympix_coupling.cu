// Blocks between rings.
//
// Off-diagonal blocks (Eq. system-rewritten, Eq. Dhat with rows on ring j
// and columns on ring k = j + delta):
//   M_qr = [gamma_qr <= r_s] d(x_qr) + sum_p B^_pq N^-1_p B^_pr,
// p over the pixels of every ring coupled to both.  Pixel q of ring j and
// pixel r of ring k are at separation index z = (2q+1) Q - (2r+1) P with
// P = n_j / g, Q = n_k / g, g = gcd(n_j, n_k).  M_qr vanishes unless
// gamma_qr <= 2 r_s (a pixel coupled to both is within r_s of each), so row
// q stores the columns with |z| <= zmax, zmax the largest separation index
// within 2 r_s: r = r0(q) + t (mod n_k), t = 0 .. K-1, with
//   r0(q) = ceil(((2q+1) Q - zmax - P) / (2P)),  K = floor(zmax / P) + 1,
// entries past the row's own count stored as zero; when K >= n_k the row
// holds every column (r0 = 0, K = n_k).  One thread per stored entry walks,
// for every ring rho coupled to both rings, the contiguous arc of pixels p
// coupled to q and adds b(q,p) N^-1_p b(r,p) where p also couples to r.
// Unwrapped pixel indices (longitudes continued past 2 pi) keep every
// separation index in one piece.
#include <cmath>

#include "sympix_internal.cuh"

namespace sympix {

__device__ __forceinline__ int fdiv(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }
__device__ __forceinline__ int cdiv(int a, int b) { return -fdiv(-a, b); }

// z reduced to its nearest image in (-half, half] (the separation of the
// nearest copies of the two pixels, |dphi| <= pi).
__device__ __forceinline__ int near_image(int z, int half) {
    z %= 2 * half;
    if (z < 0) z += 2 * half;
    return z > half ? z - 2 * half : z;
}

// Blocks whose arcs do not meet themselves around the ring (every ring but a
// few near the poles, unless the support is a good part of the sphere): no
// separation needs reducing, and the pixels coupled to both q and r are one
// run.  A CTA takes 32 rows q by up to 32 stored columns t; lane = row.  Per
// neighbour ring the four warps form the weights b(q, p) N^-1_p of the rows'
// arcs once, kCoupArc pixels at a time, in shared memory ([pixel][row]), then
// warp k walks the columns t = k, k + 4, ...: the lanes' rows meet column t in
// runs of nearly the same length, whose ends move by a fixed step from column
// to column.  One multiply-add, one shared load and one table load a pixel,
// against two FP64 operations, two table loads and six integer divisions in
// the kernel below; the same products in the same order.  l_max 1500, delta 1:
// 13.2 -> 4.66 ms; 1.5e9 multiply-adds take the FP64 pipe 2.6 ms.
constexpr int kCoupArc = 64;   // pixels of an arc staged at once
constexpr int kCoupCols = 32;  // columns per CTA

// floor(a / d) for d > 0, |a / d| < 2^20 (inv = 1 / d)
__device__ __forceinline__ int coup_floor(int a, int d, float inv) {
    int q = __float2int_rd((float)a * inv);
    const int r = a - q * d;
    q += r < 0 ? -1 : r >= d ? 1 : 0;
    return q;
}

__global__ void __launch_bounds__(128) k_sample_coupling_arcs(const CoupDesc *__restrict__ cds,
                                                              const int32_t *__restrict__ tile0, int ncd,
                                                              const BlockDesc *__restrict__ blocks,
                                                              const PairEntry *__restrict__ entries, int64_t nslots,
                                                              int64_t npix, const double *__restrict__ tb,
                                                              const double *__restrict__ td,
                                                              const double *__restrict__ ninv,
                                                              double *__restrict__ out) {
    constexpr int NU = kCoupCols / 4;
    __shared__ double wc[kCoupArc][32];
    int lo = 0, hi = ncd - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tile0[mid] <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const CoupDesc cd = cds[lo];
    const int tile = (int)blockIdx.x - tile0[lo], ntq = (cd.n + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = (tile % ntq) * 32 + lane, t0 = (tile / ntq) * kCoupCols + warp;
    const BlockDesc bj = blocks[cd.bj], bk = blocks[cd.bk];
    const double *tbo = tb + (int64_t)bj.op * nslots, *nv = ninv + (int64_t)bj.op * npix;
    const bool live = q < cd.n;
    const int Z = (2 * q + 1) * cd.Q;
    const int r0 = cd.dense ? 0 : cdiv(Z - cd.zmax - cd.P, 2 * cd.P);  // first column, unwrapped
    // which columns are stored entries, and D^ between the rings
    double acc[NU];
    unsigned on = 0;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
        const int t = t0 + 4 * u, z = Z - (2 * (r0 + t) + 1) * cd.P;
        acc[u] = 0.0;
        if (!live || t >= cd.K || z > cd.zmax || -z > cd.zmax) continue;
        on |= 1u << u;
        if (cd.dpair >= 0) {
            const PairEntry pd = entries[cd.dpair];
            const int zd = (2 * q + 1) * pd.Q - (2 * (r0 + t) + 1) * pd.P, az = zd < 0 ? -zd : zd;
            if (az <= pd.mmax) acc[u] = td[(int64_t)bj.op * nslots + pd.tab + ((az - pd.par) >> 1)];
        }
    }
    for (int a = 0; a < bj.npairs; ++a) {
        const PairEntry p1 = entries[bj.pair0 + a];
        int ib = bk.npairs > 0 ? p1.rho - entries[bk.pair0].rho : -1;  // coupled rings are consecutive
        if (ib < 0 || ib >= bk.npairs) continue;
        const PairEntry p2 = entries[bk.pair0 + ib];
        const int d1 = 2 * p1.P, d2 = 2 * p2.P;
        const float i1 = 1.0f / (float)d1, i2 = 1.0f / (float)d2;
        // the arc of q
        const int Z1 = (2 * q + 1) * p1.Q;
        const int plo = coup_floor(Z1 - p1.mmax - p1.P + d1 - 1, d1, i1);
        const int narc = live ? coup_floor(Z1 + p1.mmax - p1.P, d1, i1) - plo + 1 : 0;
        int pm0 = plo % p1.nrho;
        if (pm0 < 0) pm0 += p1.nrho;
        const int longest = p1.mmax / p1.P + 1;
        // the run of r = r0 + t0 within it (indices from plo), and its step per 4 columns
        const int Z2 = (2 * (r0 + t0) + 1) * p2.Q;
        const int e0 = Z2 - p2.mmax - p2.P + d2 - 1, e1 = Z2 + p2.mmax - p2.P;
        const int lo0 = coup_floor(e0, d2, i2), hi0 = coup_floor(e1, d2, i2);
        const int mlo0 = e0 - lo0 * d2, mhi0 = e1 - hi0 * d2;
        const int step = 8 * p2.Q, sq = step / d2, sr = step - sq * d2;
        const double *T1 = tbo + p1.tab, *T2 = tbo + p2.tab;
        double s[NU];
#pragma unroll
        for (int u = 0; u < NU; ++u) s[u] = 0.0;
        for (int c0 = 0; c0 < longest; c0 += kCoupArc) {
            const int c1 = min(longest, c0 + kCoupArc);
            __syncthreads();  // the weights of the chunk before are used
            for (int i = c0 + warp; i < c1; i += 4) {
                double w = 0.0;
                if (i < narc) {
                    const int z1 = Z1 - (2 * (plo + i) + 1) * p1.P;
                    int pm = pm0 + i;
                    if (pm >= p1.nrho) pm -= p1.nrho;
                    w = T1[((z1 < 0 ? -z1 : z1) - p1.par) >> 1] * nv[p1.noff + (int64_t)pm * p1.nstride];
                }
                wc[i - c0][lane] = w;
            }
            __syncthreads();
            int lo2 = lo0 - plo, hi2 = hi0 - plo, mlo = mlo0, mhi = mhi0;
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                if (t0 + 4 * u >= cd.K) break;  // uniform in the warp
                const int f = max(lo2, c0), l = on >> u & 1 ? min(min(hi2, narc - 1), c1 - 1) : -1;
                int z2 = Z2 + u * step - (2 * (plo + f) + 1) * p2.P;
                double v = s[u];
                for (int i = f; i <= l; ++i) {
                    v = fma(wc[i - c0][lane], T2[((z2 < 0 ? -z2 : z2) - p2.par) >> 1], v);
                    z2 -= d2;
                }
                s[u] = v;
                mlo += sr;
                lo2 += sq + (mlo >= d2 ? 1 : 0);
                mlo -= mlo >= d2 ? d2 : 0;
                mhi += sr;
                hi2 += sq + (mhi >= d2 ? 1 : 0);
                mhi -= mhi >= d2 ? d2 : 0;
            }
        }
#pragma unroll
        for (int u = 0; u < NU; ++u) acc[u] += s[u];
    }
#pragma unroll
    for (int u = 0; u < NU; ++u)
        if (live && t0 + 4 * u < cd.K) out[cd.off + (int64_t)q * cd.K + t0 + 4 * u] = acc[u];
}

// Every other block: one thread per entry, every separation reduced to its
// nearest image.
__global__ void __launch_bounds__(128) k_sample_coupling(int64_t total, const CoupDesc *__restrict__ cds,
                                                         const int64_t *__restrict__ first, int ncd,
                                                         const BlockDesc *__restrict__ blocks,
                                                         const PairEntry *__restrict__ entries, int64_t nslots,
                                                         int64_t npix, const double *__restrict__ tb,
                                                         const double *__restrict__ td,
                                                         const double *__restrict__ ninv, double *__restrict__ out) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= total) return;
    // the descriptor holding this entry
    int lo = 0, hi = ncd - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= gid) lo = mid;
        else hi = mid - 1;
    }
    const CoupDesc cd = cds[lo];
    const int64_t e = gid - first[lo];
    const int q = (int)(e / cd.K), t = (int)(e - (int64_t)q * cd.K);
    const int Z = (2 * q + 1) * cd.Q;
    const int ru = cd.dense ? t : cdiv(Z - cd.zmax - cd.P, 2 * cd.P) + t;  // column, unwrapped
    const int zqr = Z - (2 * ru + 1) * cd.P;
    double acc = 0.0;
    if (cd.dense || (zqr <= cd.zmax && zqr >= -cd.zmax)) {
        const BlockDesc bj = blocks[cd.bj], bk = blocks[cd.bk];
        const int64_t tbase = (int64_t)bj.op * nslots;
        const double *nv = ninv + (int64_t)bj.op * npix;
        // D^ between the two rings (the same support as B^)
        if (cd.dpair >= 0) {
            const PairEntry pd = entries[cd.dpair];
            // reduce the separation to the nearest image (|dphi| <= pi)
            const int64_t half = (int64_t)pd.P * pd.nrho;
            int64_t z = ((int64_t)(2 * q + 1) * pd.Q - (int64_t)(2 * ru + 1) * pd.P) % (2 * half);
            if (z < 0) z += 2 * half;
            if (z > half) z -= 2 * half;
            const int az = (int)(z < 0 ? -z : z);
            if (az <= pd.mmax) acc += td[tbase + pd.tab + ((az - pd.par) >> 1)];
        }
        for (int a = 0; a < bj.npairs; ++a) {
            const PairEntry p1 = entries[bj.pair0 + a];
            // the same neighbour ring in ring k's list
            int ib = -1;
            for (int b = 0; b < bk.npairs; ++b)
                if (entries[bk.pair0 + b].rho == p1.rho) {
                    ib = b;
                    break;
                }
            if (ib < 0) continue;
            const PairEntry p2 = entries[bk.pair0 + ib];
            // pixels p coupled to q: |Z1 - (2p+1) P1| <= m1, p unwrapped near q
            const int Z1 = (2 * q + 1) * p1.Q;
            const int plo = cdiv(Z1 - p1.mmax - p1.P, 2 * p1.P), phi = fdiv(Z1 + p1.mmax - p1.P, 2 * p1.P);
            // r's separation to p: z2 = (2 ru + 1) Q2 - (2 p + 1) P2 (the pair
            // constants of ring k with rho), the longitude difference of (r, p)
            // being pi z2 g2 / (n_k n_rho), taken at its nearest image
            const int Z2 = (2 * ru + 1) * p2.Q;
            int pm = plo % p1.nrho;
            if (pm < 0) pm += p1.nrho;
            // an arc as long as the ring (polar rings) holds every pixel once
            const int pend = min(phi, plo + p1.nrho - 1);
            double s = 0.0;
            for (int p = plo; p <= pend; ++p) {
                const int z1 = near_image(Z1 - (2 * p + 1) * p1.P, p1.P * p1.nrho);
                const int z2 = near_image(Z2 - (2 * p + 1) * p2.P, p2.P * p2.nrho);
                const int a1 = z1 < 0 ? -z1 : z1, a2 = z2 < 0 ? -z2 : z2;
                if (a1 <= p1.mmax && a2 <= p2.mmax) {
                    const double b1 = tb[tbase + p1.tab + ((a1 - p1.par) >> 1)];
                    const double b2 = tb[(int64_t)bk.op * nslots + p2.tab + ((a2 - p2.par) >> 1)];
                    s = fma(b1 * nv[p1.noff + (int64_t)pm * p1.nstride], b2, s);
                }
                if (++pm == p1.nrho) pm = 0;
            }
            acc += s;
        }
    }
    out[cd.off + e] = acc;
}

static long gcd_h(long a, long b) {
    while (b) {
        long t = a % b;
        a = b;
        b = t;
    }
    return a;
}

// Whether no separation of a block reaches around the ring: half a turn is
// separation index P Q g of a ring pair; a pixel p of q's arc, r within zmax of
// q and p's arc on ring k together stay within a full turn.  Also the coupled
// rings of both are consecutive, and every index times its step fits 2^20.
static bool coupling_plain(sympix_plan_t pl, const CoupDesc &cd) {
    const BlockDesc &bj = pl->blocks[cd.bj], &bk = pl->blocks[cd.bk];
    const double zt = (double)cd.zmax / ((double)cd.P * bk.n);  // turns, halved
    if (cd.dense || !(zt < 1.0)) return false;
    for (int i = 0; i < 2; ++i) {
        const BlockDesc &bd = i ? bk : bj;
        for (int e = 0; e < bd.npairs; ++e) {
            const PairEntry &pe = pl->entries[bd.pair0 + e];
            if (pe.rho != pl->entries[bd.pair0].rho + e || pe.nrho > (1 << 18)) return false;
        }
    }
    for (int e = 0; e < bj.npairs; ++e) {
        const PairEntry &p1 = pl->entries[bj.pair0 + e];
        for (int f = 0; f < bk.npairs; ++f) {
            const PairEntry &p2 = pl->entries[bk.pair0 + f];
            if (p1.rho != p2.rho) continue;
            const double t1 = (double)p1.mmax / ((double)p1.P * p1.nrho), t2 = (double)p2.mmax / ((double)p2.P * p2.nrho);
            if (!(t1 < 1.0) || !(t1 + zt + t2 < 1.99)) return false;
        }
    }
    return true;
}

}  // namespace sympix

using namespace sympix;

extern "C" int sympix_coupling_size(sympix_plan_t pl, int delta, size_t *bytes, int64_t *elements) {
    if (!pl) return set_error(SYMPIX_EINVAL, "sympix_coupling_size: NULL plan");
    if (pl->tiles) return set_error(SYMPIX_EUNSUPPORTED, "sympix_coupling_size: ring blocks only (k = 1)");
    if (delta < 1 || delta >= pl->grid->nrings)
        return set_error(SYMPIX_EINVAL, "sympix_coupling_size: ring offset %d out of [1, nrings)", delta);
    auto it = pl->coupling.find(delta);
    if (it == pl->coupling.end()) {
        it = pl->coupling.emplace(delta, CouplingPlan{}).first;  // built in place
        CouplingPlan &cp = it->second;
        const sympix_grid_s *g = pl->grid;
        const int nb = pl->ring1 - pl->ring0;
        int64_t off = 0;
        for (int o = 0; o < pl->nops; ++o) {
            const double r2 = std::min(2.0 * pl->r_s[o], kPi);
            const double h2 = std::sin(0.5 * r2), u2 = 2.0 * h2 * h2 * (1.0 + 1e-9);
            for (int j = pl->ring0; j + delta < pl->ring1; ++j) {
                const int k = j + delta;
                CoupDesc cd{};
                cd.bj = o * nb + (j - pl->ring0);
                cd.bk = o * nb + (k - pl->ring0);
                const long nj = g->nring[j], nk = g->nring[k], gg = gcd_h(nj, nk);
                cd.P = (int32_t)(nj / gg);
                cd.Q = (int32_t)(nk / gg);
                // largest separation index within 2 r_s (u grows with |z| up to |dphi| = pi)
                const double ta = g->theta[j], tb = g->theta[k];
                const double da = std::sin(0.5 * (ta - tb));
                const double base = 2.0 * da * da, st = 2.0 * std::sin(ta) * std::sin(tb);
                const long par = (cd.P + cd.Q) & 1, PQg = (long)cd.P * cd.Q * gg;
                const long mcap = PQg - ((PQg - par) & 1);
                long zmax = -1;
                for (long z = par; z <= mcap; z += 2) {
                    const double hh = std::sin(0.5 * kPi * (double)(z * gg) / ((double)nj * (double)nk));
                    if (r2 < kPi && base + st * hh * hh > u2) break;
                    zmax = z;
                }
                cd.zmax = (int32_t)std::max<long>(zmax, 0);
                const long K = zmax < 0 ? 1 : zmax / cd.P + 1;
                cd.dense = K >= nk ? 1 : 0;
                cd.K = (int32_t)(cd.dense ? nk : K);
                cd.n = (int32_t)nj;
                cd.off = off;
                cd.dpair = -1;
                const BlockDesc &bd = pl->blocks[cd.bj];
                for (int e = 0; e < bd.npairs; ++e)
                    if (pl->entries[bd.pair0 + e].rho == k) cd.dpair = (int32_t)(bd.pair0 + e);
                off += (int64_t)cd.n * cd.K;
                cp.desc.push_back(cd);
            }
        }
        cp.total = off;
        // the two kernels' blocks: no separation of the first list's reaches
        // around the ring
        std::vector<CoupDesc> arcs, rest;
        std::vector<int32_t> tile0;
        std::vector<int64_t> first;
        int64_t tiles = 0;
        for (const CoupDesc &cd : cp.desc) {
            if (coupling_plain(pl, cd)) {
                tile0.push_back((int32_t)tiles);
                tiles += (int64_t)((cd.n + 31) / 32) * ((cd.K + kCoupCols - 1) / kCoupCols);
                arcs.push_back(cd);
            } else {
                first.push_back(cp.total_rest);
                cp.total_rest += (int64_t)cd.n * cd.K;
                rest.push_back(cd);
            }
        }
        cp.tiles = tiles;
        int rc;
        if ((rc = tiles > INT32_MAX ? set_error(SYMPIX_EUNSUPPORTED, "sympix_coupling_size: too many blocks")
                                    : SYMPIX_OK) ||
            (rc = cp.d_arcs.upload(arcs)) || (rc = cp.d_tile0.upload(tile0)) || (rc = cp.d_rest.upload(rest)) ||
            (rc = cp.d_first.upload(first))) {
            pl->coupling.erase(it);
            return rc;
        }
        pl->all_d = true;  // D^ between rings needs d at every slot: the next table call evaluates it
    }
    if (bytes) *bytes = (size_t)it->second.total * sizeof(double);
    if (elements) *elements = it->second.total;
    return SYMPIX_OK;
}

extern "C" int sympix_coupling_layout(sympix_plan_t pl, int delta, int op, int ring, int64_t *offset, int32_t *geom) {
    if (!pl || !geom) return set_error(SYMPIX_EINVAL, "sympix_coupling_layout: NULL argument");
    if (pl->tiles) return set_error(SYMPIX_EUNSUPPORTED, "sympix_coupling_layout: ring blocks only (k = 1)");
    auto it = pl->coupling.find(delta);
    if (it == pl->coupling.end())
        return set_error(SYMPIX_EINVAL, "sympix_coupling_layout: call sympix_coupling_size(%d) first", delta);
    const int nb = pl->ring1 - pl->ring0;
    for (const CoupDesc &cd : it->second.desc) {
        const BlockDesc &bj = pl->blocks[cd.bj];
        if (bj.op != op || bj.ring != ring) continue;
        if (offset) *offset = cd.off;
        geom[0] = cd.n;
        geom[1] = pl->blocks[cd.bk].n;
        geom[2] = cd.K;
        geom[3] = cd.zmax;
        geom[4] = cd.P;
        geom[5] = cd.Q;
        geom[6] = cd.dense;
        return SYMPIX_OK;
    }
    (void)nb;
    return set_error(SYMPIX_EINVAL, "sympix_coupling_layout: no block (op %d, ring %d) for offset %d", op, ring, delta);
}

extern "C" int sympix_sample_coupling(sympix_plan_t pl, const double *ninv, int delta, double *out, void *stream) {
    if (!pl || !ninv || !out) return set_error(SYMPIX_EINVAL, "sympix_sample_coupling: NULL argument");
    if (pl->tiles) return set_error(SYMPIX_EUNSUPPORTED, "sympix_sample_coupling: ring blocks only (k = 1)");
    auto it = pl->coupling.find(delta);
    if (it == pl->coupling.end())
        return set_error(SYMPIX_EINVAL, "sympix_sample_coupling: call sympix_coupling_size(%d) first", delta);
    if (!pl->table_all_d)
        return set_error(SYMPIX_EINVAL,
                         "sympix_sample_coupling: call sympix_kernel_table after sympix_coupling_size "
                         "(the blocks between rings need d at every class)");
    cudaStream_t st = (cudaStream_t)stream;
    const CouplingPlan &cp = it->second;
    trace_mark(pl, st, nullptr);
    if (cp.total_rest > 0)
        k_sample_coupling<<<(unsigned)((cp.total_rest + 127) / 128), 128, 0, st>>>(
            cp.total_rest, cp.d_rest.p, cp.d_first.p, (int)cp.d_rest.n, pl->d_blocks.p, pl->d_entries.p, pl->nslots,
            pl->grid->npix, pl->d_tab_b.p, pl->d_tab_d.p, ninv, out);
    if (cp.tiles > 0)
        k_sample_coupling_arcs<<<(unsigned)cp.tiles, 128, 0, st>>>(cp.d_arcs.p, cp.d_tile0.p, (int)cp.d_arcs.n,
                                                                   pl->d_blocks.p, pl->d_entries.p, pl->nslots,
                                                                   pl->grid->npix, pl->d_tab_b.p, pl->d_tab_d.p, ninv,
                                                                   out);
    trace_mark(pl, st, "k_sample_coupling");
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "sympix_sample_coupling: launch");
    return SYMPIX_OK;
}
