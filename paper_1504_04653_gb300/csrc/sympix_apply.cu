// The preconditioner M^-1 x applied block by block (the diagonal ring blocks,
// block Jacobi): y = L^-T L^-1 x in FP64 with the factor of
// sympix_factor_blocks.
//
// Periodic bands up to w = 16 (k_apply_band).  RG = 8 or 16 lanes hold one
// open row of the substitution each: row k sits in slot k mod W, and when row
// i is solved, row i + W takes its slot.  A step scales row i by its
// reciprocal diagonal, hands z_i out by one shuffle and updates every lane's
// row with one multiply-add; a period is W steps.  In the gaps of a period's
// chain lane b adds the last period's z to border row b's dot product (the H =
// G / RG lane sets share the columns) and the next period's reciprocals are
// formed.  After the corner the back substitution runs the same way from the
// last row up (row i's entries are the coefficients), the border rows' part
// taken out of a period's values one period before they enter.  Band rows
// arrive by 16-byte asynchronous copies into a ring of four periods, border
// entries, x and z one or two periods ahead into registers.
//
// What bounds it: the chain.  An FP64 instruction takes its warp 64 cycles
// whatever the number of active lanes, and its result 19 more to a shuffle of
// about 30: 206 cycles a step in multiply, shuffle and multiply-add, 340 to
// 410 measured with everything else a step issues, for n steps each way.  One
// lane's recurrence per block (k_apply below, before: all widths) took about
// 2 W FP64 instructions a step.  l_max 500, two operators: 1.34 -> 0.40 ms;
// l_max 3000: 22.6 -> 2.9 ms (3.4 GB at l_max 3000, 0.5 ms).  Scaling the
// rows' coefficients by the reciprocals beforehand takes the multiplication
// out of the chain, but costs as many instructions: 3.03 ms at l_max 3000.
//
// Dense-format blocks up to 32 rows go to the same launch, a warp each with
// the matrix in shared memory and a row per lane; wider bands, larger dense
// blocks and dense storage to k_apply, one warp per block.
#include "sympix_window.cuh"

namespace sympix {

// 1/x: the FP32 estimate of the significand's reciprocal and the geometric
// series of the residual e = 1 - x y (|e| < 2^-21) to second order.
__device__ __forceinline__ double apply_recip_normal(double x) {
    const int ex = (__double2hiint(x) >> 20) & 0x7ff;
    const double y = window_widen(window_rcp32(window_narrow(x, 0)), ex - 1023);
    const double e = fma(-x, y, 1.0);
    return fma(fma(e, e, e), y, y);
}
__device__ __forceinline__ bool apply_normal(double x) { return window_normal(x) && __double2hiint(x) > 0; }
// x != 0 on the integer ALU
__device__ __forceinline__ bool apply_nonzero(double x) { return ((__double2hiint(x) << 1) | __double2loint(x)) != 0; }
__device__ __forceinline__ double apply_recip(double x) { return apply_normal(x) ? apply_recip_normal(x) : 1.0 / x; }

// 16 bytes at dst, the first `bytes` of them from src, the others zero
__device__ __forceinline__ void cp_async16_part(double *dst, const double *src, int bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ double apply_shfl(double x, int src, int width) {
    return __shfl_sync(0xffffffffu, x, src, width);
}

// One block's vector in global memory.
struct ApplyVec {
    const double *x;
    double *y;
    int64_t ps;
};

// n = 0: an idle group (`band` is then any 16-byte aligned address).
template <int W, int G>
__device__ __forceinline__ void apply_band(const double *__restrict__ band, int n, ApplyVec v, unsigned char *smem) {
    constexpr int RG = W <= 8 ? 8 : 16, H = G / RG, NB = (W + H - 1) / H;
    constexpr int RL = W + 1, PE = W * RL, NP = 4;
    const int lane = threadIdx.x & 31, gl = lane % G, r = gl % RG, h = gl / RG;
    const int rw = r < W ? r : 0;  // lanes past the band read row 0; their values reach no one
    double *ring = reinterpret_cast<double *>(smem) + (lane / G) * apply_elems(W);
    double *cs = ring + NP * PE;  // the corner, [row][column]
    const int m = n > 0 ? n - W : 0;
    const double *bord = band + (int64_t)n * RL;
    // Rows of period `per` into their place of the ring.  Rows past the m of
    // L11 are read, times zero, and L defines none of their entries: they are
    // staged as zeros.
    const int bend = m * RL;
    auto issue = [&](int per) {
        const double *src = band + per * PE + 2 * gl;
        double *dst = ring + (per % NP) * PE + 2 * gl;
        if (per >= 0 && (per + 1) * PE <= bend) {
#pragma unroll
            for (int i = 0; i < PE; i += 2 * G)
                if (i + 2 * G <= PE || i + 2 * gl < PE) cp_async16(dst + i, src + i);
        } else if (per >= 0) {
            for (int i = 0; i + 2 * gl < PE; i += 2 * G) {
                const int left = bend - (per * PE + i + 2 * gl);
                cp_async16_part(dst + i, left > 0 ? src + i : band, left < 0 ? 0 : left < 2 ? 8 * left : 16);
            }
        }
        cp_async_commit();
    };
    for (int i = gl; i < W * W; i += G) {
        const int b = i / W, c = i % W;
        cs[i] = m > 0 && c <= b ? __ldg(bord + (int64_t)b * n + m + c) : 1.0;
    }
    int mtop = m;
#pragma unroll
    for (int o = G; o < 32; o <<= 1) mtop = max(mtop, __shfl_xor_sync(0xffffffffu, mtop, o));
    const int np = (mtop + W - 1) / W;
    // 1 / L[k][k] of this lane's row of a staged period (0 past the band)
    auto diag = [&](const double *per, int k) { return r < W && k >= 0 && k < m ? per[rw * RL] : 0.0; };
    auto recip = [&](double d) { return apply_nonzero(d) ? apply_recip(d) : 0.0; };

    // -- forward: L11 z = x.  Lane b of each set also keeps border row b's dot
    // product, over the set's columns h NB .. of every period --------------------
    const double *xp = v.x + r * v.ps;
    auto load_x = [&](int k) { return r < W && k + r < m ? xp[k * v.ps] : 0.0; };
    const double *bp = bord + (int64_t)rw * n + h * NB;
    double bn[NB], dot = 0.0;
    auto border = [&](int k) {  // columns k + h NB .. of border row r
#pragma unroll
        for (int j = 0; j < NB; ++j) bn[j] = k < m && h * NB + j < W ? __ldg(bp + k + j) : 0.0;
        if (H == 1 && k + W > m) {  // a block's last period: see below
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (k + j >= m) bn[j] = 0.0;
        }
    };
    __syncwarp();
#pragma unroll
    for (int p = 0; p < NP; ++p) issue(p);
    border(0);
    double s = load_x(0), xn = load_x(W);  // right-hand sides: this period's rows and the next one's
    cp_async_wait<NP - 1>();
    __syncwarp();
    double rr = recip(diag(ring, r)), bc[NB], zl[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) bc[j] = zl[j] = 0.0;
    // a period's chain is W times shuffle and multiply-add; the next period's
    // reciprocals and the last one's products for the border fill its gaps
    for (int p = 0; p < np; ++p) {
        cp_async_wait<NP - 2>();  // period p + 1 has landed
        __syncwarp();
        const double *cur = ring + (p % NP) * PE, *nxt = ring + ((p + 1) % NP) * PE;
        const int k0 = p * W;
        const double xs = xn;
        xn = load_x(k0 + 2 * W);
        double bo[NB];
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            bo[j] = bc[j];
            bc[j] = bn[j];
        }
        border(k0 + W);
        const double dn = diag(nxt, k0 + W + r);
        double rn = apply_recip_normal(dn);
        double z = 0.0, zs[W];
#pragma unroll
        for (int q = 0; q < W; ++q) {
            // row of slot r: this period's while r > q, then the next one's
            const double c = rw > q ? cur[rw * RL + rw - q] : nxt[rw * RL + W - (q - rw)];
            const double t = s * rr;
            zs[q] = apply_shfl(t, q, G);
            if (r == q) {
                z = t;
                s = xs;
            }
            s = fma(-c, zs[q], s);
            if (q < NB) dot = fma(bo[q < NB ? q : 0], zl[q < NB ? q : 0], dot);
        }
        if (__any_sync(0xffffffffu, apply_nonzero(dn) && !apply_normal(dn))) rn = recip(dn);
        rr = apply_nonzero(dn) ? rn : 0.0;
#pragma unroll
        for (int j = 0; j < NB; ++j) zl[j] = H == 1 ? zs[j < W ? j : 0] : apply_shfl(z, h * NB + j, G);
        if (H == 1 && k0 + W > m) {
#pragma unroll
            for (int j = 0; j < NB; ++j)
                if (k0 + j >= m) zl[j] = 0.0;
        }
        if (h == 0 && r < W && k0 + r < m) v.y[(k0 + r) * v.ps] = z;
        __syncwarp();
        issue(p + NP);
    }
    cp_async_wait<0>();
    // A block's last period reaches past the m columns of L21: into the corner,
    // whose entries past the diagonal no one has written, and to rows whose z is
    // zero times what may be infinite.  Neither joins the dot product.  With one
    // block per warp that period is the last of the loop (the same test in the
    // loop: l_max 500 with two operators 0.403 ms against 0.397).
#pragma unroll
    for (int j = 0; j < NB; ++j)
        if ((np - 1) * W + h * NB + j < m) dot = fma(bc[j], zl[j], dot);
#pragma unroll
    for (int o = RG; o < G; o <<= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    // corner: lane b < W holds border row b
    double t = gl < W && m > 0 ? v.x[(m + gl) * v.ps] - dot : 0.0;
    const double rc = gl < W ? apply_recip(cs[gl * W + gl]) : 0.0;
    t *= rc;
#pragma unroll
    for (int c = 0; c < W; ++c) {
        const double zc = apply_shfl(t, c, G);
        if (gl > c && gl < W) t = fma(-cs[gl * W + c] * rc, zc, t);
    }
    t *= rc;
    double tail[NB];  // y of border rows b = h, h + H, ...
#pragma unroll
    for (int j = 0; j < NB; ++j) tail[j] = 0.0;
#pragma unroll
    for (int c = W - 1; c >= 0; --c) {
        const double yc = apply_shfl(t, c, G);
        if (c % H == h) tail[c / H] = yc;
        if (gl < c) t = fma(-cs[c * W + gl] * rc, yc, t);
    }
    if (gl < W && m > 0) v.y[(m + gl) * v.ps] = t;

    // -- back: L11^T y = z - L21^T y2, from the last row up ---------------------
    const int pt = (mtop - 1) / W;
    __syncwarp();
#pragma unroll
    for (int p = 0; p < NP; ++p) issue(pt - p);
    // z of column k + r less the border rows' part (each set takes rows h, h + H, ...)
    double zn;
    const double *bq = bord + (int64_t)h * n + r;
    auto load_z = [&](int k) {
        const bool on = r < W && k >= 0 && k + r < m;
        zn = on && h == 0 ? v.y[(k + r) * v.ps] : 0.0;
#pragma unroll
        for (int j = 0; j < NB; ++j) bn[j] = on && h + j * H < W ? __ldg(bq + k + j * H * n) : 0.0;
    };
    auto enter = [&]() {
#pragma unroll
        for (int j = 0; j < NB; ++j) zn = fma(-bn[j], tail[j], zn);
#pragma unroll
        for (int o = RG; o < G; o <<= 1) zn += __shfl_xor_sync(0xffffffffu, zn, o);
        return zn;
    };
    load_z(pt * W);
    s = enter();
    if (pt * W + r >= m) s = 0.0;
    load_z((pt - 1) * W);
    double xe = enter();  // entering values of the period before
    if ((pt - 1) * W + r >= m) xe = 0.0;
    load_z((pt - 2) * W);
    cp_async_wait<NP - 1>();
    __syncwarp();
    rr = recip(diag(ring + (pt >= 0 ? pt % NP : 0) * PE, pt * W + r));
    for (int p = pt; p >= 0; --p) {
        cp_async_wait<NP - 2>();  // period p - 1 has landed
        __syncwarp();
        const double *cur = ring + (p % NP) * PE, *prv = ring + ((p + NP - 1) % NP) * PE;
        const int k0 = p * W;
        const double xs = xe, dn = diag(prv, k0 - W + r);
        double rn = apply_recip_normal(dn);
        double yv = 0.0;
#pragma unroll
        for (int q = W - 1; q >= 0; --q) {
            // row q at column of slot r: this period's (r < q) or the one before
            const double c = cur[q * RL + (rw < q ? q - rw : W - (rw - q))];
            const double t1 = s * rr, yq = apply_shfl(t1, q, G);
            if (r == q) {
                yv = t1;
                s = xs;
            }
            s = fma(-c, yq, s);
            const int j = W - 1 - q;
            if (j < NB) zn = fma(-bn[j < NB ? j : 0], tail[j < NB ? j : 0], zn);
        }
        if (__any_sync(0xffffffffu, apply_nonzero(dn) && !apply_normal(dn))) rn = recip(dn);
        rr = apply_nonzero(dn) ? rn : 0.0;
        xe = zn;
#pragma unroll
        for (int o = RG; o < G; o <<= 1) xe += __shfl_xor_sync(0xffffffffu, xe, o);
        if (H == 1 && k0 - 2 * W + r >= m) xe = 0.0;
        load_z(k0 - 3 * W);
        if (h == 0 && r < W && k0 + r < m) v.y[(k0 + r) * v.ps] = yv;
        __syncwarp();
        issue(p - NP);
    }
    cp_async_wait<0>();
}

// A dense-format block of up to 32 rows: the matrix in shared memory (rows of
// 33), one row per lane.
__device__ __forceinline__ void apply_dense32(const double *__restrict__ A, int n, ApplyVec v, double *a) {
    const int lane = threadIdx.x & 31;
    for (int i = lane; i < n * n; i += 32) a[i / n * 33 + i % n] = __ldg(A + i);
    __syncwarp();
    const bool on = lane < n;
    const double rr = on ? apply_recip(a[lane * 33 + lane]) : 0.0;
    double s = on ? v.x[lane * v.ps] * rr : 0.0;
    for (int i = 0; i < n; ++i) {
        const double c = on && lane > i ? a[lane * 33 + i] * rr : 0.0;
        s = fma(-c, apply_shfl(s, i, 32), s);
    }
    s *= rr;
    for (int i = n - 1; i > 0; --i) {
        const double c = lane < i ? a[i * 33 + lane] * rr : 0.0;
        s = fma(-c, apply_shfl(s, i, 32), s);
    }
    if (on) v.y[lane * v.ps] = s;
}

constexpr int kApplyWarps = 4;  // independent warps per CTA, one per scheduler

// One warp per entry of `work`: blocks items[first .. first + count) of width
// w (w = -1: one dense-format block).  ONE: one block per warp.
template <bool ONE>
__global__ void __launch_bounds__(32 * kApplyWarps) k_apply_band(int count, int smem_warp, const int4 *__restrict__ work,
                                                                 const int32_t *__restrict__ items,
                                                                 const BlockDesc *__restrict__ blocks,
                                                                 const int32_t *__restrict__ info,
                                                                 const double *__restrict__ Lbuf,
                                                                 const int64_t *__restrict__ roff,
                                                                 const int32_t *__restrict__ rstr, int64_t npix,
                                                                 const double *__restrict__ x, double *y) {
    extern __shared__ __align__(16) unsigned char apply_all[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if ((int)blockIdx.x * kApplyWarps + warp >= count) return;
    unsigned char *smem = apply_all + warp * smem_warp;
    const int4 it = work[blockIdx.x * kApplyWarps + warp];  // first, count, w
    auto vec = [&](const BlockDesc &bd) {
        const int64_t px0 = (int64_t)bd.op * npix + roff[bd.ring];
        return ApplyVec{x + px0, y + px0, (int64_t)rstr[bd.ring]};
    };
    auto copy = [&](const ApplyVec &v, int n, int first, int step) {  // a failed block passes x through
        for (int c = first; c < n; c += step) v.y[c * v.ps] = v.x[c * v.ps];
    };
    StaticFor<1, kApplyWMax + 1>::run([&](auto Wc) {
        constexpr int W = decltype(Wc)::value, G = ONE ? 32 : apply_lanes(W);
        if (it.z != W) return;
        const int g = lane / G;
        const double *band = Lbuf;
        int n = 0;
        ApplyVec v{x, y, 1};
        if (g < it.y) {
            const int bi = items[it.x + g];
            const BlockDesc bd = blocks[bi];
            v = vec(bd);
            if (info[bi] == 0) {
                n = bd.n;
                band = Lbuf + bd.off_pband;
            } else {
                copy(v, bd.n, lane % G, G);
            }
        }
        __syncwarp();
        apply_band<W, G>(band, n, v, smem);
    });
    if (it.z > 0) return;
    for (int g = 0; g < it.y; ++g) {
        const int bi = items[it.x + g];
        const BlockDesc bd = blocks[bi];
        const ApplyVec v = vec(bd);
        const double *L = Lbuf + bd.off_pband;
        if (info[bi] != 0) {
            copy(v, bd.n, lane, 32);
        } else if (it.z == 0) {  // a diagonal block
            for (int c = lane; c < bd.n; c += 32) {
                const double rr = apply_recip(L[c]);
                v.y[c * v.ps] = v.x[c * v.ps] * rr * rr;
            }
        } else {
            apply_dense32(L, bd.n, v, reinterpret_cast<double *>(smem));
            __syncwarp();
        }
    }
}

// Every other block: one warp each.  Periodic band: the band rows by
// substitution along the band (one lane, from rows staged in shared memory
// with their reciprocal diagonals), the border rows as dense dot products by
// the whole warp; the back substitution first takes the border rows' entries
// out of every band row, in parallel.
constexpr int kApplyRows = 32;

__global__ void __launch_bounds__(32) k_apply(const int32_t *__restrict__ items, const BlockDesc *__restrict__ blocks,
                                              const int32_t *__restrict__ info, const double *__restrict__ Lbuf,
                                              int dense_storage, const int64_t *__restrict__ roff,
                                              const int32_t *__restrict__ rstr, int64_t npix, int max_ring,
                                              const double *__restrict__ x, double *__restrict__ y) {
    extern __shared__ double smem_apply[];
    double *v = smem_apply;           // the block's vector, n values
    double *stg = v + max_ring;       // staged band rows
    const int bi = items ? items[blockIdx.x] : blockIdx.x, lane = threadIdx.x;
    const BlockDesc bd = blocks[bi];
    const int n = bd.n;
    const int64_t px0 = (int64_t)bd.op * npix + roff[bd.ring];
    const int64_t ps = rstr[bd.ring];
    const double *xin = x + px0;
    double *yout = y + px0;
    if (info[bi] != 0) {
        for (int c = lane; c < n; c += 32) yout[c * ps] = xin[c * ps];
        return;
    }
    for (int c = lane; c < n; c += 32) v[c] = xin[c * ps];
    __syncwarp();
    auto wsum = [](double s) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        return s;
    };
    const bool pband = !dense_storage && bd.format == SYMPIX_BLOCK_PBAND;
    if (pband) {
        const int w = bd.w, RL = w + 1, m = n - w;
        const double *band = Lbuf + bd.off_pband;
        const double *bord = band + (int64_t)n * RL;
        double *rinv = stg + (kApplyRows + w) * RL;  // 1 / L[i][i] of the staged rows
        // stage band rows [r0, r1) and their reciprocal diagonals
        auto stage = [&](int r0, int r1) {
            const int cnt = (r1 - r0) * RL;
            for (int e = lane; e < cnt; e += 32) stg[e] = band[(int64_t)r0 * RL + e];
            for (int r = lane; r < r1 - r0; r += 32) rinv[r] = 1.0 / band[(int64_t)(r0 + r) * RL];
            __syncwarp();
        };
        // forward: band rows i < m
        for (int r0 = 0; r0 < m; r0 += kApplyRows) {
            const int r1 = min(m, r0 + kApplyRows);
            stage(r0, r1);
            if (lane == 0)
                for (int i = r0; i < r1; ++i) {
                    const double *row = stg + (i - r0) * RL;
                    double s = v[i];
                    for (int d = 1; d <= w && d <= i; ++d) s = fma(-row[d], v[i - d], s);
                    v[i] = s * rinv[i - r0];
                }
            __syncwarp();
        }
        // forward: the border rows (dense dot products)
        for (int b = 0; b < w; ++b) {
            const int i = m + b;
            double s = 0.0;
            for (int c = lane; c < i; c += 32) s = fma(bord[(int64_t)b * n + c], v[c], s);
            s = wsum(s);
            if (lane == 0) v[i] = (v[i] - s) / bord[(int64_t)b * n + i];
            __syncwarp();
        }
        // back: the border rows (columns i >= m of L^T)
        if (lane == 0)
            for (int i = n - 1; i >= m; --i) {
                double s = v[i];
                for (int c = i + 1; c < n; ++c) s = fma(-bord[(int64_t)(c - m) * n + i], v[c], s);
                v[i] = s / bord[(int64_t)(i - m) * n + i];
            }
        __syncwarp();
        // their contribution to every band row: v_i -= sum_b L21[b][i] v_{m+b}
        for (int i = lane; i < m; i += 32) {
            double s = v[i];
            for (int b = 0; b < w; ++b) s = fma(-bord[(int64_t)b * n + i], v[m + b], s);
            v[i] = s;
        }
        __syncwarp();
        // back: band rows, from the bottom; a chunk needs the w rows below it
        for (int r1 = m; r1 > 0; r1 -= kApplyRows) {
            const int r0 = max(0, r1 - kApplyRows);
            const int re = min(m, r1 + w);
            stage(r0, re);
            if (lane == 0)
                for (int i = r1 - 1; i >= r0; --i) {
                    double s = v[i];
                    for (int d = 1; d <= w && i + d < m; ++d) s = fma(-stg[(i + d - r0) * RL + d], v[i + d], s);
                    v[i] = s * rinv[i - r0];
                }
            __syncwarp();
        }
    } else {
        const double *A = Lbuf + (dense_storage ? bd.off_dense : bd.off_pband);
        for (int i = 0; i < n; ++i) {
            double s = 0.0;
            for (int c = lane; c < i; c += 32) s = fma(A[(int64_t)i * n + c], v[c], s);
            s = wsum(s);
            if (lane == 0) v[i] = (v[i] - s) / A[(int64_t)i * n + i];
            __syncwarp();
        }
        for (int i = n - 1; i >= 0; --i) {
            double s = 0.0;
            for (int c = i + 1 + lane; c < n; c += 32) s = fma(A[(int64_t)c * n + i], v[c], s);
            s = wsum(s);
            if (lane == 0) v[i] = (v[i] - s) / A[(int64_t)i * n + i];
            __syncwarp();
        }
    }
    for (int c = lane; c < n; c += 32) yout[c * ps] = v[c];
}

// Dynamic shared memory of one warp of k_apply_band on entries of width w, of
// the plan's widest entry, and of any.
static size_t apply_smem_width(int w, bool one) {
    const int g = one ? 32 : apply_lanes(w);
    const size_t e = w < 0 ? 32 * 33 : w == 0 ? 2 : (size_t)(32 / g) * apply_elems(w);
    return (e * sizeof(double) + 15) / 16 * 16;
}
static size_t apply_smem(sympix_plan_t pl, bool one) {
    size_t smem = 16;
    for (const int4 &it : pl->apply_work[one]) smem = std::max(smem, apply_smem_width(it.z, one));
    return smem;
}
static size_t apply_smem_max(bool one) {
    size_t smem = 16;
    for (int w = -1; w <= kApplyWMax; ++w) smem = std::max(smem, apply_smem_width(w, one));
    return smem;
}

template <bool ONE>
static void launch_apply_band(sympix_plan_t pl, const double *blocks, const int32_t *info, const double *x, double *y,
                              cudaStream_t st) {
    const int count = (int)pl->apply_work[ONE].size();
    if (!count) return;
    const size_t smem = apply_smem(pl, ONE);
    // the limit is the function's, not a launch's: the same for every plan,
    // whatever other threads and captured graphs launch
    cudaFuncSetAttribute(k_apply_band<ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(kApplyWarps * apply_smem_max(ONE)));
    k_apply_band<ONE><<<(unsigned)((count + kApplyWarps - 1) / kApplyWarps), 32 * kApplyWarps, kApplyWarps * smem, st>>>(
        count, (int)smem, pl->d_apply_work[ONE].p, pl->d_apply_items.p, pl->d_blocks.p, info, blocks, pl->d_ring_off.p,
        pl->d_ring_stride.p, pl->grid->npix, x, y);
}

// Work lists of sympix_apply on periodic-band storage: items by width (most
// expensive first), then the dense-format blocks of up to 32 rows, and the
// warps of both layouts, longest first.  One block per warp while that is at
// most two warps per scheduler (608 of them): a step then takes 340 cycles
// against 410 in a full warp, which serves 32 / G blocks.  Measured, one block
// per warp / full: l_max 500 0.344 / 0.433 ms, with two operators (1002
// blocks) 0.403 / 0.449 ms, l_max 1500 (1501 blocks) 1.54 / 1.42 ms, l_max 500
// with four operators 0.63 / 0.46 ms, l_max 3000 4.41 / 2.89 ms.
int plan_apply(sympix_plan_t pl, const std::vector<int32_t> &order) {
    std::vector<int32_t> items;
    std::vector<int32_t> rest;
    std::vector<int> width;
    for (int w = -1; w <= kApplyWMax; ++w)
        for (int b : order) {
            const BlockDesc &bd = pl->blocks[b];
            const bool band = bd.format == SYMPIX_BLOCK_PBAND;
            if (band ? bd.w != w : !(w == -1 && bd.n <= 32)) continue;
            items.push_back(b);
            width.push_back(w);
        }
    for (int b : order) {
        const BlockDesc &bd = pl->blocks[b];
        if (bd.format == SYMPIX_BLOCK_PBAND ? bd.w > kApplyWMax : bd.n > 32) rest.push_back(b);
    }
    for (int one = 0; one < 2; ++one) {
        std::vector<std::pair<double, int4>> work;
        for (size_t i = 0; i < items.size();) {
            const int w = width[i], g = one || w <= 0 ? 32 : apply_lanes(w);
            size_t e = i;
            while (e < items.size() && e < i + 32 / g && width[e] == w) ++e;
            // FP64 instructions of a step times steps
            const double step = w <= 0 ? 2.0 : 2.0 + (double)apply_lanes(w) / g + 3.0 / w;
            work.push_back({step * pl->blocks[items[i]].n, make_int4((int)i, (int)(e - i), w, 0)});
            i = e;
        }
        std::stable_sort(work.begin(), work.end(), [](const auto &a, const auto &b) { return a.first > b.first; });
        for (const auto &x : work) pl->apply_work[one].push_back(x.second);
        const int rc = pl->d_apply_work[one].upload(pl->apply_work[one]);
        if (rc) return rc;
    }
    pl->apply_one = pl->apply_work[1].size() <= 2 * 608;
    pl->apply_rest = (int)rest.size();
    const int rc = pl->d_apply_items.upload(items);
    return rc ? rc : pl->d_apply_rest.upload(rest);
}

}  // namespace sympix

using namespace sympix;

extern "C" int sympix_apply(sympix_plan_t pl, int storage, const double *blocks, const int32_t *info, const double *x,
                            double *y, void *stream) {
    if (!pl || !blocks || !info || !x || !y) return set_error(SYMPIX_EINVAL, "sympix_apply: NULL argument");
    if (pl->tiles) return set_error(SYMPIX_EUNSUPPORTED, "sympix_apply: ring blocks only (k = 1)");
    if (storage != SYMPIX_STORE_PBAND && storage != SYMPIX_STORE_DENSE)
        return set_error(SYMPIX_EINVAL, "sympix_apply: unknown storage %d", storage);
    if (x == y) return set_error(SYMPIX_EINVAL, "sympix_apply: x and y must not alias");
    cudaStream_t st = (cudaStream_t)stream;
    // the band rows are copied 16 bytes at a time: a buffer that is not
    // 16-byte aligned takes the other kernel
    const bool band = storage == SYMPIX_STORE_PBAND && (reinterpret_cast<uintptr_t>(blocks) & 15) == 0;
    trace_mark(pl, st, nullptr);
    const int nrest = band ? pl->apply_rest : (int)pl->blocks.size();
    if (nrest > 0) {
        // the vector, then kApplyRows + w staged rows of w + 1 values and their
        // reciprocal diagonals (the widest periodic band planned)
        const size_t W1 = (size_t)pl->max_w + 1;
        const size_t smem = ((size_t)pl->grid->max_ring + (kApplyRows + W1) * (W1 + 1)) * sizeof(double);
        cudaFuncSetAttribute(k_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);  // what a CTA may have
        k_apply<<<(unsigned)nrest, 32, smem, st>>>(band ? pl->d_apply_rest.p : nullptr, pl->d_blocks.p, info, blocks,
                                                   storage == SYMPIX_STORE_DENSE ? 1 : 0, pl->d_ring_off.p,
                                                   pl->d_ring_stride.p, pl->grid->npix, pl->grid->max_ring, x, y);
    }
    if (band) {
        if (pl->apply_one)
            launch_apply_band<true>(pl, blocks, info, x, y, st);
        else
            launch_apply_band<false>(pl, blocks, info, x, y, st);
    }
    trace_mark(pl, st, "k_apply");
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "sympix_apply: launch");
    return SYMPIX_OK;
}
