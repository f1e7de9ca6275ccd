// Sliding-window Cholesky of periodic-band blocks (w <= 12) in one pass, for
// the exact arithmetics: FP64 (V = double) and split FP32 (V = DF).
//
// The lower rows that column i updates are the W band rows i+1 .. i+W and the
// W border rows m .. n-1 (m = n - W), so the active part of the matrix is a
// symmetric window of 2W rows whose W columns are the band rows' indices.  RG
// = 8, 16 or 32 lanes hold one row each, every lane the row's entries at the
// W window columns (a band row the full symmetric row, so that every index
// below is static).  Band index k lives in slot k mod W: when column i has
// been eliminated, row i + W takes slot i mod W, and a loop body of W steps
// (one period) has every slot in a register of fixed name.  A step on column
// i with pivot d:
//   - every lane scales its entry of column i by f, formed in the step before
//     (the pivot's own lane takes the entering row's entry A[i+W][i], which
//     has had no update yet): t = entry x f;
//   - W shuffles of t and W multiply-adds update the lane's row, the entering
//     row's entries, read a step ahead, replacing the retired slot's; the
//     next column comes first, so that its pivot and f are formed among the
//     other updates.
// FP64 takes f = 1/sqrt(d), and t is L's entry.  Split FP32 takes f = 1/d (a
// shorter chain) and scales by 1/sqrt(d), one root per lane for a whole
// period, as the entries leave; in FP64 that form was slower (1570 against
// 1210 cycles a step at W = 8), each FP64 instruction holding its warp for
// 64 cycles.  Band rows arrive by 16-byte asynchronous copies into a ring of
// NP periods; the columns' entries take the place of the input rows in the
// ring (an entry is read before the same position is written) and leave a
// period at a time as contiguous 16-byte stores.  The border rows' entries
// go through a ring of 2G columns; every G columns they leave as contiguous
// rows and each lane adds one column's products to the W(W+1)/2 corner sums.
// At the end the sums meet in a halving exchange and the corner is eliminated
// by the same lanes.  Rows past m and steps past a block's end hold arbitrary
// values: they only ever reach each other.
//
// What bounds it: an FP64 instruction takes 64 cycles of its scheduler, and of
// its warp, whatever the number of active lanes (measured; 76 with the other
// three schedulers busy).  At W = 8 a step has 5 of them for the root, 1 for t,
// W (or W/2 with one block per warp) updates and W(W+1)/2G for the corner.
// One block per lane (the band pass of option 3) spends fewer instructions per
// block, but its step takes 1.8k cycles and the border needs a second pass of
// about the same length; here a block's n steps take 1210 cycles each in FP64
// and 780 in split FP32 for band and border together, and nothing is
// transposed.  Factor stage, before and now: l_max 64 FP64 0.47 -> 0.094 ms,
// l_max 500 3.3 -> 0.93 ms, l_max 1500 5.8 -> 3.0 ms, l_max 3000 12.9 -> 7.4 ms;
// split FP32 at l_max 750 with three operators 2.1 -> 1.4 ms, l_max 3000 6.0 ->
// 3.7 ms.
#pragma once

#include <algorithm>

#include "sympix_factor_kernels.cuh"

namespace sympix {

// The FP32 reciprocal estimate (relative error below 2^-22).
__device__ __forceinline__ float window_rcp32(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// A double from an FP32 value in (1/2, 1] times 2^-shift.
__device__ __forceinline__ double window_widen(float f, int shift) {
    const unsigned u = __float_as_uint(f);
    return __hiloint2double((int)((u >> 3) + (896u << 20)) - shift * (1 << 20), (int)(u << 29));
}
// x's significand as an FP32 value in [1, 2) (truncated), times 2 when `odd`.
__device__ __forceinline__ float window_narrow(double x, int odd) {
    const unsigned m = ((unsigned)(__double2hiint(x) & 0xfffff) << 3) | ((unsigned)__double2loint(x) >> 29);
    return __uint_as_float(((unsigned)(127 + odd) << 23) | m);
}
// Whether x is normal (with a normal reciprocal).
__device__ __forceinline__ bool window_normal(double x) {
    const unsigned ex = (unsigned)(__double2hiint(x) >> 20) & 0x7ffu;
    return ex - 1u < 2043u;
}
// 1/sqrt(x) for such x > 0: the FP32 estimate y from the significand (exponent
// made even) and the series of (1 - e)^(-1/2) to second order in the residual
// e = 1 - x y^2 (|e| < 2^-21, the next term is below 2^-63).
__device__ __forceinline__ double window_rsqrt_normal(double x) {
    const int ex = (__double2hiint(x) >> 20) & 0x7ff, odd = (ex + 1) & 1;
    const double y = window_widen(rsqrtf(window_narrow(x, odd)), (ex - 1023 - odd) / 2);
    const double e = fma(-x * y, y, 1.0);
    return fma(fma(e, 0.375, 0.5), y * e, y);
}
__device__ __forceinline__ double window_rsqrt(double x) { return window_normal(x) ? window_rsqrt_normal(x) : rsqrt(x); }
// 1/sqrt(x) in split FP32 the same way, e to second order (to first order, as
// in f2_rsqrt, 3 e^2 / 8 remains: |L L^T - M| / |M| 7.4e-15 against 4.5e-15 now,
// l_max 64 to 750).
__device__ __forceinline__ DF window_rsqrt(DF x) {
    const float y = rsqrtf(x.hi);
    const DF e = df_fma(-(x * DF(y)), DF(y), DF(1.0f));
    return to_df(f2_fast_two_sum(y, y * fmaf(0.5f, e.hi + e.lo, 0.375f * e.hi * e.hi)));
}
// What a column's entries are multiplied by: 1/sqrt(pivot) in FP64; 1/pivot in
// split FP32, by the series of the residual r = 1 - x y of the FP32 estimate.
__device__ __forceinline__ double window_factor_normal(double x) { return window_rsqrt_normal(x); }
__device__ __forceinline__ DF window_factor_normal(DF x) {
    const float y = window_rcp32(x.hi);
    const DF r = df_fma(DF(-y), x, DF(1.0f));
    return to_df(f2_fast_two_sum(y, y * (fmaf(r.hi, r.hi, r.hi) + r.lo)));
}
// Whether 2^-64 <= |x| < 2^64: 1/x then has both its words among FP32's normal
// numbers (alone it is flushed to zero for x > 2^126 and loses its low word
// from 2^104 on), and so have a column's entries times it.
__device__ __forceinline__ bool window_common(DF x) { return ((__float_as_uint(x.hi) >> 23) & 0xffu) - 63u < 128u; }
__device__ __forceinline__ DF window_scale(DF x, float g) { return DF(x.hi * g, x.lo * g); }
// For any x > 0: g, a power of two with x g^2 in [1, 4), and 1 / (x g^2).  The
// column's entries times g then stand for them in the step.
__device__ __forceinline__ DF window_factor_far(DF x, float &g) {
    const bool tiny = x.hi < 0x1p-100f;  // may be subnormal
    if (tiny) x = window_scale(x, 0x1p+100f);
    const int e = (int)((__float_as_uint(x.hi) >> 23) & 0xffu) - 127;
    g = __uint_as_float((unsigned)(127 - (e >> 1)) << 23);
    x = window_scale(window_scale(x, g), g);
    if (tiny) g *= 0x1p+50f;
    return window_factor_normal(x);
}
// (FP64's 1/sqrt needs neither)
__device__ __forceinline__ double window_scale(double x, float) { return x; }
__device__ __forceinline__ double window_factor_far(double x, float &) { return window_factor_normal(x); }

// x > 0 on the integer ALU (an FP64 compare costs as much as a multiply-add)
__device__ __forceinline__ bool window_positive(double x) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    return (hi > 0 || (hi == 0 && lo != 0u)) && (hi < 0x7ff00000 || (hi == 0x7ff00000 && lo == 0u));
}
__device__ __forceinline__ bool window_positive(DF x) { return x > DF(0.0f); }

__device__ __forceinline__ double window_shfl(double x, int src, int width) {
    return __shfl_sync(0xffffffffu, x, src, width);
}
__device__ __forceinline__ DF window_shfl(DF x, int src, int width) {
    return DF(__shfl_sync(0xffffffffu, x.hi, src, width), __shfl_sync(0xffffffffu, x.lo, src, width));
}
__device__ __forceinline__ double window_xor(double x, int o) { return __shfl_xor_sync(0xffffffffu, x, o); }
__device__ __forceinline__ DF window_xor(DF x, int o) {
    return DF(__shfl_xor_sync(0xffffffffu, x.hi, o), __shfl_xor_sync(0xffffffffu, x.lo, o));
}

// Lanes per block: `one` block per warp, or as many as the rows allow.
__host__ __device__ constexpr int window_rows(int W) { return W <= 4 ? 8 : W <= 8 ? 16 : 32; }

// FP64 instructions of one step with G lanes per block: the root, the scaled
// column, the row update, the corner products.  The plan compares the two
// layouts by it (plan: sympix_support).
inline double window_step_cost(int w, int G) {
    const int H = G / window_rows(w);
    return 6.0 + (w + H - 1) / H + 0.5 * w * (w + 1) / G;
}

// Shared memory of one block (elements of 8 bytes).
constexpr int kWindowPeriods = 4;  // staged periods of band rows
__host__ __device__ constexpr int window_elems(int W, int G) {
    return (kWindowPeriods * W * (W + 1) + W * (2 * G + 1) + W * W + 2 * G + 2 + 1) / 2 * 2;
}

// The block preconditioner on periodic bands (sympix_apply.cu): the widest
// band, lanes per block of a full warp, and one block's shared memory (doubles:
// four periods of band rows, the corner).
constexpr int kApplyWMax = 16;
__host__ __device__ constexpr int apply_lanes(int W) { return W <= 8 ? 8 : 16; }
__host__ __device__ constexpr int apply_elems(int W) { return (4 * W * (W + 1) + W * W + 1) / 2 * 2; }

// Sums of acc over the G lanes of a group: each exchange adds the halves of
// two lanes' arrays, so lane l ends with sums at, at + 1, ... of its own.
template <class V, int N, int O>
struct WindowReduce {
    __device__ __forceinline__ static void run(const V (&acc)[N], int lane, int at, int total, double *out) {
        constexpr int HALF = (N + 1) / 2;
        const bool up = (lane & O) != 0;
        V got[HALF];
#pragma unroll
        for (int i = 0; i < HALF; ++i) {
            const V hi = HALF + i < N ? acc[HALF + i < N ? HALF + i : 0] : V(0);
            got[i] = (up ? hi : acc[i]) + window_xor(up ? acc[i] : hi, O);
        }
        WindowReduce<V, HALF, O / 2>::run(got, lane, at + (up ? HALF : 0), up ? min(total, at + N) : min(total, at + HALF),
                                          out);
    }
};
template <class V, int N>
struct WindowReduce<V, N, 0> {
    __device__ __forceinline__ static void run(const V (&acc)[N], int, int at, int total, double *out) {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (at + i < total) out[at + i] = elem_to_f64(acc[i]);
    }
};

// W >= 1; G lanes per block (window_rows(W), or 32 for one block per warp).
// Every lane of the warp calls this; `bi` < 0: an idle group.
template <class V, int W, int G>
__device__ __forceinline__ void window_chol(const BlockDesc *__restrict__ blocks, int bi, double *__restrict__ out,
                                            int32_t *__restrict__ info, unsigned char *smem) {
    constexpr int RG = window_rows(W), H = G / RG, WC = (W + H - 1) / H;
    constexpr int RL = W + 1, PE = W * RL, NP = kWindowPeriods, HB = 2 * G, HS = HB + 1;
    constexpr int NPAIR = W * (W + 1) / 2;
    constexpr bool LDL = !std::is_same<V, double>::value;
    const int lane = threadIdx.x & 31, gl = lane % G, r = gl % RG, h = gl / RG;
    V *ring = reinterpret_cast<V *>(smem) + (lane / G) * window_elems(W, G);
    V *hist = ring + NP * PE;  // border values, [row][column mod HB]
    V *tail = hist + W * HS;   // A21 at the last W columns, [row][column]
    V *prs = tail + W * W;     // 1/sqrt(pivot), [column mod HB]
    V *spare = prs + HB;       // [0] zero, [1] takes what no one needs
    int n = 2 * W + 2;
    double *band = nullptr;
    if (bi >= 0) {
        const BlockDesc bd = blocks[bi];
        n = bd.n;
        band = out + bd.off_pband;
    }
    const int m = bi >= 0 ? n - W : 0;
    double *bord = band + (int64_t)n * RL;
    const PBandView view{band, bord, n, W, n - W};
    const int bend = bi >= 0 ? n * RL : 0;
    auto issue = [&](int per) {
        V *dst = ring + (per % NP) * PE;
        for (int i = 2 * gl; i < PE; i += 2 * G)
            if (per * PE + i < bend) cp_async16(dst + i, band + (int64_t)per * PE + i);
        cp_async_commit();
    };
    // a landed period in the kernel's arithmetic, in place
    auto convert = [&](int per) {
        if constexpr (!std::is_same<V, double>::value) {
            V *src = ring + (per % NP) * PE;
            for (int i = gl; i < PE; i += G) src[i] = elem_from_f64<V>(*reinterpret_cast<double *>(src + i));
        }
    };
#pragma unroll
    for (int p = 0; p < NP; ++p) issue(p);
    // the first window: rows 0 .. W-1 and the border rows at columns 0 .. W-1
    V x[WC];
#pragma unroll
    for (int j = 0; j < WC; ++j) {
        const int c = h * WC + j;
        x[j] = V(0);
        if (bi >= 0 && c < W && r < 2 * W)
            x[j] = elem_from_f64<V>(r < W ? band[max(r, c) * RL + abs(r - c)] : view.a(m + r - W, c));
    }
    for (int i = gl; i < W * W; i += G)
        tail[i] = bi >= 0 ? elem_from_f64<V>(view.a(m + i / W, m - W + i % W)) : V(0);
    // corner sums: all of them over this lane's columns, or for wide windows
    // (W > 8: too many registers) this lane's share of them over all columns
    constexpr bool SHARE = W > 8;
    constexpr int NACC = SHARE ? (NPAIR + G - 1) / G : NPAIR;
    V acc[NACC];
    int pb[NACC], pc[NACC];
#pragma unroll
    for (int i = 0; i < NACC; ++i) {
        acc[i] = V(0);
        if constexpr (SHARE) {
            int k = min(gl + i * G, NPAIR - 1), b = 0;
            while (k > b) k -= ++b;  // pair b (b + 1) / 2 + c
            pb[i] = b * HS;
            pc[i] = k * HS;
        }
    }
    int inf = 0, done = 0;
    // column 0's entry of this lane's row, the pivot and its reciprocal
    V a = x[0];
    if constexpr (H > 1) a = window_shfl(a, r, G);
    V d = window_shfl(x[0], 0, G);
    V f = window_factor_normal(d);
    if constexpr (!LDL)
        if (!window_normal(d)) f = rsqrt(d);
    if (gl == 0) spare[0] = V(0);
    cp_async_wait<NP - 1>();
    __syncwarp();
    convert(0);
    // Split FP32: a pivot is at most its row's diagonal entry, so the entries of
    // the rows that a period eliminates, looked at while it enters, say whether
    // one of its pivots can be too large (or the entry too small) for 1/pivot.
    // Such a period runs a copy of the steps with scaled columns.  A test per
    // pivot instead cost 12 to 27 % (l_max 750, three operators 1.81 ms; one a
    // period 1.44; none 1.42).
    bool far = false;
    if constexpr (LDL) {
        __syncwarp();
        far = __any_sync(0xffffffffu, gl < W && gl < m && !window_common(ring[(gl < W ? gl : 0) * RL]));
    }
    int mtop = m;
#pragma unroll
    for (int o = G; o < 32; o <<= 1) mtop = max(mtop, __shfl_xor_sync(0xffffffffu, mtop, o));

    // border columns done .. done + G - 1: out as rows, products into the corner sums
    auto flush_border = [&](bool ok) {
        const int k = done + gl;
        V xb[W];
#pragma unroll
        for (int b = 0; b < W; ++b) xb[b] = k < m ? (LDL ? hist[b * HS + k % HB] * prs[k % HB] : hist[b * HS + k % HB]) : V(0);
        if (ok && k < m) {
#pragma unroll
            for (int b = 0; b < W; ++b) bord[(int64_t)b * n + k] = elem_to_f64(xb[b]);
        }
        if constexpr (SHARE) {
#pragma unroll
            for (int b = 0; b < W; ++b) hist[b * HS + k % HB] = xb[b];
            __syncwarp();
            const V *x = hist + done % HB;  // G columns from done, a multiple of G
#pragma unroll 4
            for (int j = 0; j < G; ++j)
#pragma unroll
                for (int i = 0; i < NACC; ++i) acc[i] = band_fma(x[pb[i] + j], x[pc[i] + j], acc[i]);
        } else {
#pragma unroll
            for (int b = 0; b < W; ++b)
#pragma unroll
                for (int c = 0; c <= b; ++c) acc[b * (b + 1) / 2 + c] = band_fma(xb[b], xb[c], acc[b * (b + 1) / 2 + c]);
        }
        done += G;
    };

    const int np = (mtop + W - 1) / W;
    auto period = [&](int p, auto FARc) {
        constexpr bool FAR = decltype(FARc)::value;
        cp_async_wait<NP - 2>();  // period p + 1 has landed
        __syncwarp();
        convert(p + 1);
        __syncwarp();
        V *cur = ring + (p % NP) * PE, *nxt = ring + ((p + 1) % NP) * PE;
        // what step s takes from its entering row e = (p+1) W + s: the entry at
        // this lane's row (border rows: A21's last columns, else zero), the one
        // at column e - W, and the row itself for the lane that takes it over;
        // read a step ahead, before the step in between writes to the ring
        V nv, na, nrow[WC];
        auto enter = [&](auto Sc) {
            constexpr int s = decltype(Sc)::value;
            const int e = (p + 1) * W + s;
            const V *row = nxt + s * RL;
            const V *pn = row + (r > s ? W - (r - s) : s - r);
            if (r >= W) pn = (unsigned)(e - (m - W)) < (unsigned)W && r < 2 * W ? tail + (r - W) * W + e - (m - W) : spare;
            nv = *pn;
            na = row[W];
#pragma unroll
            for (int j = 0; j < WC; ++j) {
                const int c = h * WC + j;
                nrow[j] = row[c > s ? W - (c - s) : s - c];
            }
        };
        enter(std::integral_constant<int, 0>{});
        [[maybe_unused]] const V dn = nxt[(gl < W ? gl : 0) * RL];
        [[maybe_unused]] float g = 1.0f;
        if constexpr (FAR) f = window_factor_far(d, g);
        StaticFor<0, W>::run([&](auto Sc) {
            constexpr int s = decltype(Sc)::value, s1 = (s + 1) % W, js1 = s1 % WC;
            const int i = p * W + s;
            if (inf == 0 && i < m && !window_positive(d)) inf = i + 1;
            const V src = r == s ? na : a;
            V col = src;
            if constexpr (FAR) col = window_scale(src, g);
            const V t = col * f, left = LDL ? col : t;
            V base[WC];
#pragma unroll
            for (int j = 0; j < WC; ++j) {
                base[j] = r == s ? nrow[j] : x[j];
                if (h * WC + j == s) base[j] = nv;
            }
            if constexpr (s + 1 < W) enter(std::integral_constant<int, s + 1 < W ? s + 1 : 0>{});
            auto update = [&](int j) { x[j] = band_fma(-left, window_shfl(t, h * WC + j, G), base[j]); };
            const V a0 = a;
            [[maybe_unused]] const V f0 = f;
            update(js1);
            d = window_shfl(x[js1], s1 / WC * RG + s1, G);
            a = x[js1];
            if constexpr (H > 1) a = window_shfl(a, s1 / WC * RG + r, G);
            if constexpr (FAR)
                f = window_factor_far(d, g);
            else
                f = window_factor_normal(d);
#pragma unroll
            for (int j = 0; j < WC; ++j)
                if (j != js1) update(j);
            if constexpr (!LDL)
                if (__any_sync(0xffffffffu, !window_normal(d))) f = rsqrt(d);
            // column i's entries: rows of this period and the next, the border's
            // history; the pivot in its row's diagonal position
            V *pw = (r > s ? cur : nxt) + r * RL + (r > s ? r - s : W - (s - r));
            if (r >= W) pw = hist + (r - W) * HS + i % HB;
            if (h > 0 || r >= 2 * W) pw = spare + 1;
            *pw = LDL ? src : t;
            if (r == s && h == 0) {
                cur[s * RL] = a0;
                if constexpr (!LDL) prs[i % HB] = f0;
            }
            __syncwarp();
        });
        if constexpr (FAR) f = window_factor_normal(d);
        if constexpr (LDL) far = __any_sync(0xffffffffu, gl < W && (p + 1) * W + gl < m && !window_common(dn));
        // rows p W .. p W + W - 1 of L
        const int rows = min(W, m - p * W);
        const bool ok = inf == 0;
        if constexpr (LDL) {
            if (gl < W) prs[(p * W + gl) % HB] = window_rsqrt(cur[gl * RL]);
        } else {
            if (gl < W) cur[gl * RL] *= prs[(p * W + gl) % HB];
        }
        __syncwarp();
        if (ok) {
            double *dst = band + (int64_t)p * PE;
            auto l = [&](int i) {
                return elem_to_f64(LDL ? cur[i] * prs[(p * W + i / RL - i % RL) & (HB - 1)] : cur[i]);
            };
            if (p > 0) {
                for (int i = 2 * gl; i < rows * RL; i += 2 * G) {
                    const double y0 = l(i);
                    if (i + 1 < rows * RL)
                        *reinterpret_cast<double2 *>(dst + i) = make_double2(y0, l(i + 1));
                    else
                        dst[i] = y0;
                }
            } else {  // offsets past the first column keep the sampled values
                for (int i = gl; i < rows * RL; i += G)
                    if (i % RL <= i / RL) dst[i] = l(i);
            }
        }
        if ((p + 1) * W - done >= G) flush_border(ok);
        __syncwarp();
        issue(p + NP);
    };
    if constexpr (LDL) {
        for (int p = 0; p < np;) {
            for (; p < np && !far; ++p) period(p, std::false_type{});
            for (; p < np && far; ++p) period(p, std::true_type{});
        }
    } else {
        for (int p = 0; p < np; ++p) period(p, std::false_type{});
    }
    cp_async_wait<0>();
    while (done < np * W) flush_border(inf == 0);  // columns past m are zero
    __syncwarp();
    // the corner A22 - S, one row per lane, eliminated in FP64
    double *sums = reinterpret_cast<double *>(hist);
    if constexpr (SHARE) {
        double mine[NACC];
#pragma unroll
        for (int i = 0; i < NACC; ++i) mine[i] = elem_to_f64(acc[i]);
        __syncwarp();  // the history has been read
#pragma unroll
        for (int i = 0; i < NACC; ++i)
            if (gl + i * G < NPAIR) sums[gl + i * G] = mine[i];
    } else {
        WindowReduce<V, NPAIR, G / 2>::run(acc, gl, 0, NPAIR, sums);
    }
    __syncwarp();
    double cr[W];
#pragma unroll
    for (int c = 0; c < W; ++c)
        cr[c] = bi >= 0 && gl < W && c <= gl ? band[(int64_t)(m + gl) * RL + (gl - c)] - sums[gl * (gl + 1) / 2 + c] : 0.0;
#pragma unroll
    for (int s = 0; s < W; ++s) {
        const double d = window_shfl(cr[s], s, G);
        const bool go = inf == 0 && window_positive(d);
        if (inf == 0 && !go) inf = m + s + 1;
        const double v = cr[s] * window_rsqrt(go ? d : 1.0);
        if (bi >= 0 && go && gl < W && gl >= s) bord[(int64_t)gl * n + m + s] = v;
#pragma unroll
        for (int c = s + 1; c < W; ++c) cr[c] = fma(-v, window_shfl(v, c, G), cr[c]);
    }
    if (bi >= 0 && gl == 0) info[bi] = inf;
}

// W = 0: a diagonal block.
template <class V>
__device__ __forceinline__ void window_diag(const BlockDesc *__restrict__ blocks, int bi, double *__restrict__ out,
                                            int32_t *__restrict__ info) {
    const int lane = threadIdx.x & 31;
    if (bi < 0) return;
    const BlockDesc bd = blocks[bi];
    double *band = out + bd.off_pband;
    int first = bd.n;
    for (int i = lane; i < bd.n; i += 32)
        if (!window_positive(elem_from_f64<V>(band[i]))) {
            first = i;
            break;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) first = min(first, __shfl_xor_sync(0xffffffffu, first, o));
    for (int i = lane; i < first; i += 32) {
        const V d = elem_from_f64<V>(band[i]);
        band[i] = elem_to_f64(d * window_rsqrt(d));
    }
    if (lane == 0) info[bi] = first < bd.n ? first + 1 : 0;
}

// A dense-format block of up to 32 rows (polar rings), in FP64 whatever the
// arithmetic: the lower triangle in shared memory (rows of 33), one row per
// lane.  Beside the window's chains it costs nothing; as a launch of its own
// (k_factor_dense) it added 36 to 55 us to every factor.
__device__ __forceinline__ void window_dense(const BlockDesc *__restrict__ blocks, int bi, double *__restrict__ out,
                                             int32_t *__restrict__ info, double *a) {
    const int lane = threadIdx.x & 31;
    const BlockDesc bd = blocks[bi];
    const int n = bd.n;
    double *A = out + bd.off_pband;
    for (int i = lane; i < n * n; i += 32)
        if (i % n <= i / n) a[i / n * 33 + i % n] = A[i];
    __syncwarp();
    int inf = 0;
    for (int j = 0; j < n; ++j) {
        const double d = a[j * 33 + j];
        if (!window_positive(d)) {  // the same in every lane
            inf = j + 1;
            break;
        }
        double l = 0.0;
        if (lane >= j && lane < n) {
            l = a[lane * 33 + j] * window_rsqrt(d);
        }
        __syncwarp();  // the pivot has been read
        if (lane >= j && lane < n) a[lane * 33 + j] = l;
        for (int k = j + 1; k < n; ++k) {
            const double lk = window_shfl(l, k, 32);
            if (lane >= k && lane < n) a[lane * 33 + k] = fma(-l, lk, a[lane * 33 + k]);
        }
        __syncwarp();
    }
    if (inf == 0)
        for (int i = lane; i < n * n; i += 32)
            if (i % n <= i / n) A[i] = a[i / n * 33 + i % n];
    if (lane == 0) info[bi] = inf;
}

// One warp per item: blocks items[first .. first + count) of width w (-1: one
// small dense-format block).  ONE: one block per warp.  Four independent warps per CTA, one on each scheduler
// of its SM: CTAs of one warp were placed unevenly (up to three on one
// scheduler and none on another), which doubled the time.
constexpr int kWindowWarps = 4;
// (two CTAs per SM: the registers allow no more)
template <class V, bool ONE>
__global__ void __launch_bounds__(32 * kWindowWarps, 2) k_window_chol(int count, int smem_warp,
                                                                   const int4 *__restrict__ work,
                                                                   const int32_t *__restrict__ items,
                                                                   const BlockDesc *__restrict__ blocks,
                                                                   double *__restrict__ out,
                                                                   int32_t *__restrict__ info) {
    extern __shared__ __align__(16) unsigned char window_all[];
    const int warp = threadIdx.x >> 5;
    if ((int)blockIdx.x * kWindowWarps + warp >= count) return;
    unsigned char *window_smem = window_all + warp * smem_warp;
    const int4 it = work[blockIdx.x * kWindowWarps + warp];  // first, count, w
    StaticFor<1, kNarrowWMax + 1>::run([&](auto Wc) {
        constexpr int W = decltype(Wc)::value, G = ONE ? 32 : window_rows(W);
        if (it.z == W) {
            const int g = (threadIdx.x & 31) / G;
            window_chol<V, W, G>(blocks, g < it.y ? items[it.x + g] : -1, out, info, window_smem);
        }
    });
    if (it.z == 0)
        for (int g = 0; g < it.y; ++g) window_diag<V>(blocks, items[it.x + g], out, info);
    else if (it.z < 0)
        window_dense(blocks, items[it.x], out, info, reinterpret_cast<double *>(window_smem));
}

template <class V, bool ONE>
void launch_window_list(sympix_plan_t pl, double *blocks, int32_t *info, cudaStream_t st) {
    // one size for every plan: the limit is the function's, not a launch's
    size_t smem = 32 * 33 * sizeof(double);  // a small dense block
    for (int w = 1; w <= kNarrowWMax; ++w) {
        const int g = ONE ? 32 : window_rows(w);
        smem = std::max(smem, (size_t)(32 / g) * window_elems(w, g) * 8);
    }
    const int count = (int)pl->d_win[ONE].n;
    cudaFuncSetAttribute(k_window_chol<V, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(kWindowWarps * smem));
    k_window_chol<V, ONE><<<(unsigned)((count + kWindowWarps - 1) / kWindowWarps), 32 * kWindowWarps,
                            kWindowWarps * smem, st>>>(count, (int)smem, pl->d_win[ONE].p, pl->d_win_items.p,
                                                       pl->d_blocks.p, blocks, info);
}

template <class V>
void launch_window_lists(sympix_plan_t pl, int one, double *blocks, int32_t *info, cudaStream_t st) {
    one ? launch_window_list<V, true>(pl, blocks, info, st) : launch_window_list<V, false>(pl, blocks, info, st);
}

}  // namespace sympix
