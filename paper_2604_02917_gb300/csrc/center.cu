// mv_center_factor: mu = R 1/T, L = (R - mu 1^T)/sqrt(T-1), tr(Sigma) = ||L||_F^2 (Sec. 2.1).
//
// n x T output: one block per asset row sums the row and writes it centred;
// the second read of the row hits L2.  Transposed output: the same kernel
// leaves the means, then a tiled transpose reads R again along periods.
// Sums of squares go to one partial per block, added in a second,
// single-block kernel in fixed order, so tr(Sigma) is deterministic.
//
// Arithmetic.  The results are those of FP64 (mu, tr Sigma to FP64 rounding,
// every stored entry of L the rounding of the FP64 value), but GB300 retires
// about 2 FP64 operations per clock and SM, and one FP64 operation per entry
// of R already costs 0.45 ms at 5440 x 48374 (the copy rate would read R in
// 0.155 ms).  So an entry meets FP64 only when it has to:
//  * sum of a row: exact 64-bit integer sums of the entries' significands
//    (RowSum);
//  * centred entry: an FP32 pair with a proven error bound, FP64 when the
//    bound leaves the rounding open (centred());
//  * sum of squares: FP32 pairs, 16 entries at a time (SquareSum).
// With FP64 per entry 5440 x 48374 FP32 took 3.55 ms; so it takes 0.57 ms (0.74 ms
// transposed) at the same error of the trace: 0.9e-16 (root mean square over
// panels of 2000 x 20000) against 1.4e-16.
#include <stdio.h>
#include <string.h>

#include <algorithm>

#include "mv_internal.cuh"

namespace mv {

static thread_local char g_last_error[512] = "";

int record_cuda_error(cudaError_t e, const char *what, const char *file, int line) {
    const char *base = strrchr(file, '/');
    snprintf(g_last_error, sizeof(g_last_error), "%s (%s) at %s:%d: %s", cudaGetErrorName(e), cudaGetErrorString(e),
             base ? base + 1 : file, line, what);
    return MV_ERR_CUDA;
}

int record_message(int status, const char *msg) {
    snprintf(g_last_error, sizeof(g_last_error), "%s", msg);
    return status;
}

// Sum of FP32 values: exact within a flush, whose total (up to 256 values) is
// rounded to FP64 and added in FP64, as are the threads' sums.  A value is a
// 24-bit significand m (signed) times 2^(e - 150); m << (e - eb) is added to
// a 64-bit integer while e lies in [eb, eb + 30] (under 2^54 each, so 256 of
// them fit), eb being set so that the first value seen has 8 octaves of
// headroom (fewer above 2^119: the window ends below the field 255).
// Anything outside that window (a value 2^8 above or 2^-22 below the first,
// infinities, NaN) is added in FP64; a larger value also moves the window.  About 10 integer operations per value, against an FP64
// conversion and addition at 2 per clock and SM.
struct RowSum {
    long long acc = 0;
    double wide = 0.0;
    int eb = 1 << 20;              // no value seen yet: everything is out of the window

    __device__ __forceinline__ void flush() {
        if (acc != 0) wide += scalbn((double)acc, eb - 150);
        acc = 0;
    }
    __device__ __forceinline__ void add_wide(float x) {
        const unsigned b = __float_as_uint(x) & 0x7fffffffu;
        if (b == 0) return;
        const int e = (int)(b >> 23);
        if (e >= 1 && e < 255 && (eb == 1 << 20 || e > eb + 30)) {
            flush();
            // never 0: the significand of e = 0 has no implicit bit; at most 224: field 255 stays outside
            eb = e > 23 ? min(e - 22, 224) : 1;
            add_inside(x);
        } else {
            wide += (double)x;
        }
    }
    __device__ __forceinline__ bool inside(float x) const {
        return (unsigned)((int)((__float_as_uint(x) >> 23) & 0xff) - eb) <= 30u;
    }
    __device__ __forceinline__ void add_inside(float x) {
        const int b = __float_as_int(x);
        const int sh = ((b >> 23) & 0xff) - eb;
        const int m = (b & 0x7fffff) | 0x800000, sg = b >> 31;
        acc += (long long)((m ^ sg) - sg) * (long long)(1 << sh);
    }
    // K values; the window test is one branch for all of them.
    template <int K>
    __device__ __forceinline__ void add(const float (&x)[K]) {
        bool in = true;
#pragma unroll
        for (int k = 0; k < K; ++k) in = in && inside(x[k]);
        if (in) {
#pragma unroll
            for (int k = 0; k < K; ++k) add_inside(x[k]);
        } else {
#pragma unroll 1
            for (int k = 0; k < K; ++k) {
                float v = 0.f;
#pragma unroll
                for (int j = 0; j < K; ++j) v = j == k ? x[j] : v;
                if (inside(v)) add_inside(v); else add_wide(v);
            }
        }
    }
    __device__ __forceinline__ double total() {
        flush();
        return wide;
    }
};

// Constants of one row: mean and c = 1/sqrt(T-1) as FP32 pairs, and the
// absolute part of the error bound of centred().  `wide` is infinite where
// the FP32 range cannot be relied on (the row's largest |R| outside
// [2^-30, 2^50], infinities or NaN), and in small panels: every entry then
// takes the FP64 path.  A square of a pair is off by 2^-49 or so; over kPairMin
// of them that averages to FP64's own error, over fewer it would not.
constexpr int64_t kPairMin = 1 << 16;
struct RowConst {
    float mh, ml, ch, cl, wide;
};
__device__ __forceinline__ RowConst row_const(double mean, double c, float amax, bool small) {
    RowConst k;
    k.mh = (float)mean;
    k.ml = (float)(mean - (double)k.mh);
    k.ch = (float)c;
    k.cl = (float)(c - (double)k.ch);
    const bool ok = !small && amax >= 0x1p-30f && amax <= 0x1p50f && fabsf(k.mh) <= 0x1p50f;
    k.wide = ok ? fmaf(fabsf(k.mh) * k.ch, 0x1p-44f, 0x1p-120f) : INFINITY;
    return k;
}

// Two FP32 values per instruction (sm_100 and later): a centred entry is
// about 28 FP32 operations, and issue slots, not the pipe, bound the kernels.
__device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }

// Sum of squares of FP32 pairs (s, e), two at a time, without the factor c^2
// (which would bring in the error of c as a pair; the blocks divide by T - 1
// in FP64).  (s + e)^2 = s^2 + (2 s e + e^2), the first square as a product
// and its error, the second term rounded as one sum: every rounding is to
// nearest of a sum whose last bits vary, so none has a preferred sign (added
// after 2 s e, e^2 would be lost each time: 7e-16 of the sum).  The pair
// (h, l) that collects them (Knuth's error-free addition) goes to FP64 every
// kSquareFlush additions (4: 0.59 and 0.74 ms for 0.57 and 0.74, the same
// error).  Values centred in FP64 are added in FP64.
constexpr int kSquareFlush = 8;
struct SquareSum {
    float2 h = make_float2(0.f, 0.f), l = make_float2(0.f, 0.f);
    double wide = 0.0;
    __device__ __forceinline__ void add(float2 s, float2 e) {
        const float2 q = __fmul2_rn(s, s);
        const float2 m = __ffma2_rn(__fadd2_rn(s, s), e, __fmul2_rn(e, e));
        const float2 r = __fadd2_rn(__ffma2_rn(s, s, neg2(q)), m);
        const float2 t = __fadd2_rn(h, q), bb = sub2(t, h);         // h + q = t + (rounding error), exactly
        l = __fadd2_rn(l, __fadd2_rn(__fadd2_rn(sub2(h, sub2(t, bb)), sub2(q, bb)), r));
        h = t;
    }
    __device__ __forceinline__ void flush() {
        const float t = h.x + h.y, bb = t - h.x;                    // the two lanes' pairs as one
        const float r = ((h.x - (t - bb)) + (h.y - bb)) + (l.x + l.y);
        wide += (double)t + (double)r;
        h = l = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ double total() {
        flush();
        return wide;
    }
};

// FP32 roundings of d = (x - mean) c for two entries of a row.  x - mh is
// exact as the pair (s, e); the product with the pair (ch, cl) leaves d = p + r
// with an error below 7 x 2^-48 |p| + 3 x 2^-48 |mh| ch (unit roundoff 2^-24
// in each of the pair's low parts), and r +- tol adds 3 x 2^-48 |p| + 2^-48
// |mh| ch: inside tol = 2^-44 (|p| + |mh| ch) for rows inside row_const's
// limits.  Where p + r - tol and p + r + tol round to the same FP32 value that
// value is the rounding of the FP64 result too; elsewhere (about one entry in
// 2^18) d is formed in FP64.  BF16 adds one case: an FP32 value on a BF16 tie
// does not say which way the FP64 value rounds.  Returns the values to store
// (for BF16 already rounded to it on the FP64 path) and adds the squares of
// x - mean, to FP64 or as the pair (s, e), of the first `use` entries to q.
template <int DT>
__device__ __forceinline__ float2 centred(float2 x, const RowConst &k, double mean, double c, int use, SquareSum &q) {
    const float2 mh = splat(k.mh), ch = splat(k.ch);
    float2 s = sub2(x, mh);
    const float2 bb = sub2(s, x);
    float2 e = sub2(sub2(sub2(x, sub2(s, bb)), __fadd2_rn(mh, bb)), splat(k.ml));
    const float2 p = __fmul2_rn(s, ch);
    float2 r = __ffma2_rn(s, ch, neg2(p));
    r = __ffma2_rn(s, splat(k.cl), r);
    r = __ffma2_rn(e, ch, r);
    const float2 tol = __ffma2_rn(make_float2(fabsf(p.x), fabsf(p.y)), splat(0x1p-44f), splat(k.wide));
    float2 f = __fadd2_rn(p, sub2(r, tol));
    const float2 f1 = __fadd2_rn(p, __fadd2_rn(r, tol));
    bool wx = !(f.x == f1.x), wy = !(f.y == f1.y);
    if constexpr (DT == MV_BF16) {
        wx = wx || (__float_as_uint(f.x) & 0xffffu) == 0x8000u;
        wy = wy || (__float_as_uint(f.y) & 0xffffu) == 0x8000u;
    }
    if (wx || wy || use < 2) {
        auto in64 = [&](float v) {
            const double u = (double)v - mean, d = u * c;
            q.wide = fma(u, u, q.wide);
            return DT == MV_BF16 ? __bfloat162float(__double2bfloat16(d)) : (float)d;
        };
        if (wx || use < 1) {
            if (use >= 1) f.x = in64(x.x);
            s.x = e.x = 0.f;
        }
        if (wy || use < 2) {
            if (use >= 2) f.y = in64(x.y);
            s.y = e.y = 0.f;
        }
    }
    q.add(s, e);
    return f;
}

template <int DT>
__device__ __forceinline__ void store_elem(void *L, int64_t idx, float val, float inv_scale) {
    if constexpr (DT == MV_F32) {
        reinterpret_cast<float *>(L)[idx] = val;
    } else if constexpr (DT == MV_BF16) {
        reinterpret_cast<__nv_bfloat16 *>(L)[idx] = __float2bfloat16_rn(val);
    } else {
        reinterpret_cast<__nv_fp8_storage_t *>(L)[idx] = __nv_cvt_float_to_fp8(val * inv_scale, __NV_SATFINITE, __NV_E4M3);
    }
}

// One block of NT threads per asset row.  Pass 1: mu_i = sum_t R_it / T and
// the FP32 range of the row; the FP8 scale max_t |d_it| / 448 follows exactly
// from it, because d = ((double)x - mu) c is monotone in x.  Pass 2 (WRITE):
// the centred entries, stored in the storage type, and their squares for the
// trace; the re-read of the row mostly hits L2.  With WRITE = false
// (transposed layout) pass 2 is done by transpose_center_kernel, which finds
// the row's largest |R| in amax.  Entries are read one per lane (rows of a
// ragged panel share no 16-byte alignment), kCenterUnroll loads in flight.
// NT: FP64 runs once per thread and warp here (the thread totals and the
// shuffles over them), about 3000 cycles of the SM's FP64 pipe per block of
// 512, so long panels take 128 threads per row (more rows in flight instead);
// panels of fewer rows than that fills take 512.
constexpr int kCenterUnroll = 8;
constexpr int kRowThreads = 128, kRowThreadsFew = 512;
template <int DT, bool WRITE, int NT>
__global__ void __launch_bounds__(NT)
center_kernel(const float *__restrict__ R, int64_t ldR, unsigned T, void *__restrict__ L, int64_t ldL,
              float *__restrict__ row_scale, double *__restrict__ mu, double *__restrict__ rowsq,
              float *__restrict__ amax_out, int64_t i_base, bool small) {
    constexpr int U = kCenterUnroll;
    __shared__ double red[NT / kWarp + 1];
    __shared__ float s_lo[NT / kWarp], s_hi[NT / kWarp];
    const int64_t i = i_base + blockIdx.x;                 // asset; R holds rows i_base ..
    const float *r = R + (int64_t)blockIdx.x * ldR;
    RowSum sum;
    float xmin = INFINITY, xmax = -INFINITY;
    auto range = [&](float x) {
        if constexpr (DT == MV_FP8_E4M3) {
            xmin = fminf(xmin, x);
            xmax = fmaxf(xmax, x);
        } else {
            xmax = fmaxf(xmax, fabsf(x));                   // only the largest |x| is needed
        }
    };
    unsigned t = threadIdx.x;
    int since = 0;
    for (; t + (U - 1) * NT < T; t += U * NT) {
        float x[U];
#pragma unroll
        for (int k = 0; k < U; ++k) x[k] = r[t + k * NT];
        sum.add(x);
#pragma unroll
        for (int k = 0; k < U; ++k) range(x[k]);
        since += U;
        if (since >= 240) {                                 // at most 256 values in the integer
            sum.flush();
            since = 0;
        }
    }
    for (; t < T; t += NT) {                                // fewer than U values
        const float x[1] = {r[t]};
        sum.add(x);
        range(x[0]);
    }
    const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        xmin = fminf(xmin, __shfl_xor_sync(0xffffffffu, xmin, o));
        xmax = fmaxf(xmax, __shfl_xor_sync(0xffffffffu, xmax, o));
    }
    if (lane == 0) {
        s_lo[warp] = xmin;
        s_hi[warp] = xmax;
    }
    double s[1] = {sum.total()};
    block_sum<1, NT>(s, red);                               // its barriers publish s_lo and s_hi too
#pragma unroll
    for (int w = 0; w < NT / kWarp; ++w) {
        xmin = fminf(xmin, s_lo[w]);
        xmax = fmaxf(xmax, s_hi[w]);
    }
    const double mean = s[0] / (double)T;
    const double c = 1.0 / sqrt((double)(T - 1));
    float inv_scale = 1.f, ra = xmax;
    if constexpr (DT == MV_FP8_E4M3) {
        const double amax = fmax(((double)xmax - mean) * c, (mean - (double)xmin) * c);
        const float scale = amax > 0.0 ? (float)(amax / 448.0) : 1.f;
        inv_scale = 1.f / scale;
        if (threadIdx.x == 0) row_scale[i] = scale;
        ra = fmaxf(fabsf(xmin), fabsf(xmax));
    }
    if constexpr (WRITE) {
        const RowConst k = row_const(mean, c, ra, small);
        SquareSum q;
        const int64_t o = i * ldL;
        auto write2 = [&](float2 x, unsigned ta, unsigned tb, int use) {
            const float2 f = centred<DT>(x, k, mean, c, use, q);
            store_elem<DT>(L, o + ta, f.x, inv_scale);
            if (use > 1) store_elem<DT>(L, o + tb, f.y, inv_scale);
        };
        t = threadIdx.x;
        int adds = 0;
        for (; t + (U - 1) * NT < T; t += U * NT) {
            float x[U];
#pragma unroll
            for (int j = 0; j < U; ++j) x[j] = r[t + j * NT];
#pragma unroll
            for (int j = 0; j < U; j += 2) write2(make_float2(x[j], x[j + 1]), t + j * NT, t + (j + 1) * NT, 2);
            adds += U / 2;
            if (adds % kSquareFlush == 0) q.flush();
        }
        for (; t < T; t += 2 * NT) {
            const bool two = t + NT < T;
            write2(make_float2(r[t], two ? r[t + NT] : 0.f), t, t + NT, two ? 2 : 1);
        }
        for (int64_t z = (int64_t)T + threadIdx.x; z < ldL; z += NT) store_elem<DT>(L, o + z, 0.f, inv_scale);
        double v[1] = {q.total()};
        __syncthreads();
        block_sum<1, NT>(v, red);
        if (threadIdx.x == 0) rowsq[i] = v[0] / (double)(T - 1);
    } else if (threadIdx.x == 0) {
        amax_out[i] = ra;
    }
    if (threadIdx.x == 0) mu[i] = mean;
}

// L^T (T x ldM, row t = period t) from R (n x T).  A block owns kTile assets
// and one of `slices` period slices, walking it in kTile x kTileT tiles
// through shared memory: read along periods (one row per warp and
// instruction), written along assets; columns n..ldM-1 are written as zeros.
// Values as center_kernel's; each block leaves the sum of its squares in
// sqpart[asset tile x slices + slice] (added in fixed order by
// trace_kernel).  The slice count is chosen per call to fill the GPU.
constexpr int kTile = 32;
constexpr int kTileT = 64;                      // periods per tile
constexpr int kMaxSlices = 64;                  // period slices per asset tile (grid fill), at most
constexpr int kTransThreads = 128;             // 256: 724 against 707 us at 5440 x 48374 FP32, 179 against 162 at 3754 x 10162 FP8
template <int DT>
__global__ void __launch_bounds__(kTransThreads)
transpose_center_kernel(const float *__restrict__ R, int64_t ldR, int64_t n, int T, void *__restrict__ M, int64_t ldM,
                        const float *__restrict__ row_scale, const double *__restrict__ mu,
                        const float *__restrict__ amax, double *__restrict__ sqpart, int64_t i_base, int slices,
                        bool small) {
    constexpr int W = kTransThreads / kWarp, RPW = kTile / W;   // warps, asset rows per warp
    constexpr int H = kTileT / kWarp;                           // loads per row and tile
    __shared__ float tile[kTile][kTileT + 1];
    __shared__ double red[kTransThreads / kWarp + 1];
    __shared__ double s_mean[kTile];
    __shared__ RowConst s_k[kTile];
    const int64_t i0 = i_base + (int64_t)blockIdx.y * kTile;   // assets; R holds rows i_base ..
    const int slice = blockIdx.x;
    const int per = ((T + slices - 1) / slices + kTileT - 1) / kTileT * kTileT;
    const int tb = slice * per, te = min(T, tb + per);
    const double c = 1.0 / sqrt((double)(T - 1));
    const int lane = threadIdx.x % kWarp, warp = threadIdx.x / kWarp;
    if (threadIdx.x < kTile) {
        const int64_t i = i0 + threadIdx.x;
        s_mean[threadIdx.x] = i < n ? mu[i] : 0.0;
        s_k[threadIdx.x] = row_const(s_mean[threadIdx.x], c, i < n ? amax[i] : 1.f, small);
    }
    __syncthreads();
    const float inv = (DT == MV_FP8_E4M3 && i0 + lane < n) ? 1.f / row_scale[i0 + lane] : 1.f;
    SquareSum q;
    const bool inside = i0 + kTile <= n;               // every asset of the tile exists (and ldM >= n)
    const float *src = R + (i0 - i_base + warp) * ldR + lane;
    // the next tile's loads go out before this tile is centred
    float x[RPW][H], nx[RPW][H];
    auto fetch = [&](int t0, float (&v)[RPW][H]) {
        if (inside && te - t0 >= kTileT) {
#pragma unroll
            for (int j = 0; j < RPW; ++j)
#pragma unroll
                for (int h = 0; h < H; ++h) v[j][h] = src[(int64_t)(j * W) * ldR + t0 + h * kWarp];
        } else {
#pragma unroll
            for (int j = 0; j < RPW; ++j)
#pragma unroll
                for (int h = 0; h < H; ++h)
                    v[j][h] = i0 + warp + j * W < n && lane + h * kWarp < te - t0 ? src[(int64_t)(j * W) * ldR + t0 + h * kWarp]
                                                                                   : 0.f;
        }
    };
    fetch(tb, nx);
    for (int t0 = tb; t0 < te; t0 += kTileT) {
        const bool full = inside && te - t0 >= kTileT;
#pragma unroll
        for (int j = 0; j < RPW; ++j)
#pragma unroll
            for (int h = 0; h < H; ++h) x[j][h] = nx[j][h];
        if (t0 + kTileT < te) fetch(t0 + kTileT, nx);
#pragma unroll
        for (int j = 0; j < RPW; ++j) {
            const int a = warp + j * W;
            const RowConst k = s_k[a];
#pragma unroll
            for (int h = 0; h < H; h += 2) {
                // entries of the tile that exist: all, or those below te of an existing asset
                int use = 2;
                if (!full) use = i0 + a >= n ? 0 : min(2, max(0, (te - t0 - lane - h * kWarp + kWarp - 1) / kWarp));
                const float2 f = centred<DT>(make_float2(x[j][h], x[j][h + 1]), k, s_mean[a], c, use, q);
                tile[a][lane + h * kWarp] = use > 0 ? f.x : 0.f;
                tile[a][lane + (h + 1) * kWarp] = use > 1 ? f.y : 0.f;
            }
            if ((j + 1) * H % (2 * kSquareFlush) == 0) q.flush();
        }
        __syncthreads();
        if (i0 + lane < ldM) {
            const int64_t at = (int64_t)(t0 + warp) * ldM + i0 + lane;
#pragma unroll
            for (int j = 0; j < kTileT / W; ++j)
                if (full || j * W + warp < te - t0) store_elem<DT>(M, at + (int64_t)(j * W) * ldM, tile[lane][warp + j * W], inv);
        }
        __syncthreads();
    }
    double v[1] = {q.total()};
    block_sum<1, kTransThreads>(v, red);
    if (threadIdx.x == 0 && i0 < n) sqpart[(i0 / kTile) * slices + slice] = v[0] / (double)(T - 1);
}

// trace(Sigma): the sum of the blocks' partials, in a fixed order.
constexpr int kCenterThreads = 512;
__global__ void __launch_bounds__(kCenterThreads)
trace_kernel(const double *__restrict__ part, int64_t count, double *__restrict__ trace) {
    __shared__ double red[(kCenterThreads / kWarp + 1) * 1];
    double s[1] = {0.0};
    for (int64_t i = threadIdx.x; i < count; i += kCenterThreads) s[0] += part[i];
    block_sum<1, kCenterThreads>(s, red);
    if (threadIdx.x == 0) *trace = s[0];
}

// Centering of the asset rows [i0, i1) of R, whose row i0 is at R_rows.
// The last chunk of the transposed layout also zero-fills columns n..ldL-1.
// Period slices of the transposed write: about 32 blocks per SM over the
// asset tiles of a chunk of `rows` assets (several waves, so that the last
// one costs little).
static int center_slices(int64_t rows, int64_t T) {
    const int64_t tiles = (rows + kTile - 1) / kTile;
    int64_t sl = (32 * 152 + tiles - 1) / tiles;
    const int64_t max_by_T = (T + kTileT - 1) / kTileT;
    sl = sl < 1 ? 1 : (sl > kMaxSlices ? kMaxSlices : sl);
    return (int)(sl < max_by_T ? sl : max_by_T);
}

static void center_chunk(const float *R_rows, int64_t ldR, int64_t n, int64_t T, int out_dtype, bool tn, void *d_L,
                         int64_t ldL, float *d_row_scale, double *d_mu, double *rowsq, float *amax, int64_t i0,
                         int64_t i1, int slices, cudaStream_t s) {
    const unsigned rows = (unsigned)(i1 - i0);
    const bool small = n * T < kPairMin;
    const bool few = rows < 152 * 8;                           // one row per block: about 8 blocks of 128 per SM
    const int64_t wend = (tn && i1 == n) ? ldL : i1;          // transposed: columns written by this chunk
    const dim3 tgrid((unsigned)slices, (unsigned)((wend - i0 + kTile - 1) / kTile));
#define MV_CENTER_ROWS(DT, WRITE, NT, RS)                                                                        \
    center_kernel<DT, WRITE, NT><<<rows, NT, 0, s>>>(R_rows, ldR, (unsigned)T, WRITE ? d_L : nullptr, ldL, RS,   \
                                                     d_mu, rowsq, amax, i0, small)
#define MV_CENTER_CASE(DT, RS)                                                                                   \
    if (tn) {                                                                                                    \
        if (few) MV_CENTER_ROWS(DT, false, kRowThreadsFew, RS); else MV_CENTER_ROWS(DT, false, kRowThreads, RS); \
        transpose_center_kernel<DT><<<tgrid, kTransThreads, 0, s>>>(R_rows, ldR, n, (int)T, d_L, ldL, RS, d_mu,  \
                                                                    amax, rowsq, i0, slices, small);             \
    } else {                                                                                                     \
        if (few) MV_CENTER_ROWS(DT, true, kRowThreadsFew, RS); else MV_CENTER_ROWS(DT, true, kRowThreads, RS);   \
    }
    switch (out_dtype) {
        case MV_F32: MV_CENTER_CASE(MV_F32, nullptr) break;
        case MV_BF16: MV_CENTER_CASE(MV_BF16, nullptr) break;
        default: MV_CENTER_CASE(MV_FP8_E4M3, d_row_scale) break;
    }
#undef MV_CENTER_CASE
#undef MV_CENTER_ROWS
}

static int center_args(const void *R, int64_t n, int64_t T, int64_t ldR, int out_dtype, int layout, void *d_L,
                       int64_t ldL, float *d_row_scale, double *d_mu, double *d_trace) {
    if (R == nullptr || d_L == nullptr || d_mu == nullptr || d_trace == nullptr) return MV_ERR_INVALID_ARG;
    if (layout != MV_LAYOUT_NT && layout != MV_LAYOUT_TN) return MV_ERR_INVALID_ARG;
    const bool tn = layout == MV_LAYOUT_TN;
    if (n < 1 || T < 2 || ldR < T || ldL < (tn ? n : T) || n > (1LL << 31) - 1 || T > (1LL << 31) - 1)
        return MV_ERR_INVALID_ARG;
    if (dtype_size(out_dtype) == 0) return MV_ERR_INVALID_ARG;
    if (out_dtype == MV_FP8_E4M3 && d_row_scale == nullptr) return MV_ERR_INVALID_ARG;
    if (tn && (ldL + kTile - 1) / kTile > 65535)
        return record_message(MV_ERR_UNSUPPORTED, "mv_center_factor: the transposed output needs ldL <= 65535 * 32");
    return MV_OK;
}

// Workspace: the partial sums of squares (one per row, or per asset tile and
// slice), then the rows' largest |R| (transposed output).
static size_t center_amax_offset(int64_t n) { return align_up((size_t)((n + kTile - 1) / kTile) * kMaxSlices * 8, 256); }
static int64_t center_partials(int64_t n, bool tn, int slices) { return tn ? (n + kTile - 1) / kTile * slices : n; }

// Chunked host-to-device pipeline of mv_center_factor_host.
constexpr int64_t kHostChunkBytes = 64ll << 20;

static int64_t host_chunk_rows(int64_t n, int64_t T) {
    int64_t m = kHostChunkBytes / (T * 4);
    m = m / kTile * kTile;
    if (m < kTile) m = kTile;
    return m < n ? m : n;
}

}  // namespace mv

using namespace mv;

extern "C" {

size_t mv_center_workspace_size(int64_t n, int64_t T) {
    (void)T;
    return n > 0 ? std::max(align_up((size_t)n * 8 * kMaxSlices, 256), center_amax_offset(n) + align_up(4 * (size_t)n, 256)) : 0;
}

int mv_center_factor(const float *d_R, int64_t n, int64_t T, int64_t ldR, int out_dtype, int layout, void *d_L,
                     int64_t ldL, float *d_row_scale, double *d_mu, double *d_trace, void *d_ws, size_t ws_bytes,
                     mv_stream_t stream) {
    MV_TRY(center_args(d_R, n, T, ldR, out_dtype, layout, d_L, ldL, d_row_scale, d_mu, d_trace));
    const size_t need = mv_center_workspace_size(n, T);
    if (d_ws == nullptr || ws_bytes < need || ((uintptr_t)d_ws) % 256 != 0) return MV_ERR_WORKSPACE;
    (void)cudaGetLastError();
    cudaStream_t s = (cudaStream_t)stream;
    const bool tn = layout == MV_LAYOUT_TN;
    double *rowsq = reinterpret_cast<double *>(d_ws);
    float *amax = reinterpret_cast<float *>(reinterpret_cast<char *>(d_ws) + center_amax_offset(n));
    const int slices = center_slices(n, T);
    center_chunk(d_R, ldR, n, T, out_dtype, tn, d_L, ldL, d_row_scale, d_mu, rowsq, amax, 0, n, slices, s);
    trace_kernel<<<1, kCenterThreads, 0, s>>>(rowsq, center_partials(n, tn, slices), d_trace);
    MV_CUDA_TRY(cudaGetLastError());
    return MV_OK;
}

size_t mv_center_host_workspace_size(int64_t n, int64_t T) {
    if (n < 1 || T < 2) return 0;
    const int64_t m = host_chunk_rows(n, T);
    return mv_center_workspace_size(n, T) + 2 * align_up((size_t)m * (size_t)T * 4, 256);
}

int mv_center_factor_host(const float *h_R, int64_t n, int64_t T, int64_t ldR, int out_dtype, int layout, void *d_L,
                          int64_t ldL, float *d_row_scale, double *d_mu, double *d_trace, void *d_ws, size_t ws_bytes,
                          mv_stream_t stream) {
    MV_TRY(center_args(h_R, n, T, ldR, out_dtype, layout, d_L, ldL, d_row_scale, d_mu, d_trace));
    const size_t need = mv_center_host_workspace_size(n, T);
    if (d_ws == nullptr || ws_bytes < need || ((uintptr_t)d_ws) % 256 != 0) return MV_ERR_WORKSPACE;
    (void)cudaGetLastError();
    cudaStream_t s = (cudaStream_t)stream;
    const bool tn = layout == MV_LAYOUT_TN;
    const int64_t m = host_chunk_rows(n, T);
    const int slices = center_slices(m, T);
    char *ws = reinterpret_cast<char *>(d_ws);
    double *rowsq = reinterpret_cast<double *>(ws);
    float *amax = reinterpret_cast<float *>(ws + center_amax_offset(n));
    const size_t o_stage = mv_center_workspace_size(n, T), stage_bytes = align_up((size_t)m * (size_t)T * 4, 256);
    float *stage[2] = {reinterpret_cast<float *>(ws + o_stage), reinterpret_cast<float *>(ws + o_stage + stage_bytes)};
    // The copies run on a stream of their own, one chunk ahead of the kernels.
    cudaStream_t cs;
    MV_CUDA_TRY(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
    cudaEvent_t copied[2], used[2], start;
    for (int b = 0; b < 2; ++b) {
        MV_CUDA_TRY(cudaEventCreateWithFlags(&copied[b], cudaEventDisableTiming));
        MV_CUDA_TRY(cudaEventCreateWithFlags(&used[b], cudaEventDisableTiming));
    }
    MV_CUDA_TRY(cudaEventCreateWithFlags(&start, cudaEventDisableTiming));
    MV_CUDA_TRY(cudaEventRecord(start, s));
    MV_CUDA_TRY(cudaStreamWaitEvent(cs, start, 0));            // the copies follow earlier work on `stream`
    int st = MV_OK;
    int k = 0;
    for (int64_t i0 = 0; i0 < n && st == MV_OK; i0 += m, ++k) {
        const int64_t i1 = i0 + m < n ? i0 + m : n;
        const int b = k & 1;
        if (k >= 2 && cudaStreamWaitEvent(cs, used[b], 0) != cudaSuccess) st = MV_ERR_CUDA;
        if (st == MV_OK &&
            cudaMemcpy2DAsync(stage[b], (size_t)T * 4, h_R + i0 * ldR, (size_t)ldR * 4, (size_t)T * 4,
                              (size_t)(i1 - i0), cudaMemcpyHostToDevice, cs) != cudaSuccess)
            st = record_cuda_error(cudaGetLastError(), "cudaMemcpy2DAsync (host R chunk)", __FILE__, __LINE__);
        if (st == MV_OK && cudaEventRecord(copied[b], cs) != cudaSuccess) st = MV_ERR_CUDA;
        if (st == MV_OK && cudaStreamWaitEvent(s, copied[b], 0) != cudaSuccess) st = MV_ERR_CUDA;
        if (st == MV_OK) {
            center_chunk(stage[b], T, n, T, out_dtype, tn, d_L, ldL, d_row_scale, d_mu, rowsq, amax, i0, i1, slices, s);
            if (cudaEventRecord(used[b], s) != cudaSuccess) st = MV_ERR_CUDA;
        }
    }
    if (st == MV_OK) trace_kernel<<<1, kCenterThreads, 0, s>>>(rowsq, center_partials(n, tn, slices), d_trace);
    // `stream` waits for every copy before the events and the copy stream go away.
    cudaEvent_t fin;
    if (cudaEventCreateWithFlags(&fin, cudaEventDisableTiming) == cudaSuccess) {
        cudaEventRecord(fin, cs);
        cudaStreamWaitEvent(s, fin, 0);
        cudaEventDestroy(fin);
    }
    for (int b = 0; b < 2; ++b) {
        cudaEventDestroy(copied[b]);
        cudaEventDestroy(used[b]);
    }
    cudaEventDestroy(start);
    cudaStreamDestroy(cs);
    MV_TRY(st);
    MV_CUDA_TRY(cudaGetLastError());
    return MV_OK;
}

const char *mv_status_string(int status) {
    switch (status) {
        case MV_OK: return "MV_OK";
        case MV_ERR_INVALID_ARG: return "MV_ERR_INVALID_ARG: bad pointer, size, alignment or option";
        case MV_ERR_INFEASIBLE: return "MV_ERR_INFEASIBLE: the feasible set F is empty";
        case MV_ERR_NOT_CONVERGED: return "MV_ERR_NOT_CONVERGED: iteration budget reached";
        case MV_ERR_TIMEOUT: return "MV_ERR_TIMEOUT: a bounded device wait gave up";
        case MV_ERR_NUMERIC: return "MV_ERR_NUMERIC: NaN or Inf encountered";
        case MV_ERR_CUDA: return "MV_ERR_CUDA: a CUDA runtime call failed";
        case MV_ERR_UNSUPPORTED: return "MV_ERR_UNSUPPORTED: not implemented for these arguments";
        case MV_ERR_WORKSPACE: return "MV_ERR_WORKSPACE: workspace missing, too small or misaligned";
        default: return "unknown mv_status";
    }
}

const char *mv_version(void) { return "mv 0.1 sm_103a"; }

const char *mv_last_error(void) { return g_last_error; }

}  // extern "C"
