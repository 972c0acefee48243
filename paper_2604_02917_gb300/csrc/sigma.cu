// Explicit covariance Sigma = L L^T (the classical model of Sec. 3's remark:
// NPGA with grad f(x) = 2 Sigma x, O(n^2) per iteration) formed once on the
// tcgen05 tensor cores.
//
// Sigma is symmetric, so only the 256 x 256 tiles (I, J) with I <= J are
// multiplied, each by a pair of CTAs (cluster of 2, cta_group::2 MMAs); the
// epilogue writes each tile and its mirror, so the stored Sigma is exactly
// symmetric.  On a diagonal tile only the entries with col >= row are kept
// and mirrored.
//
// Operands are BF16, K-major (row t of L along T), FP32 accumulation:
//   MV_BF16  L itself, one K-segment;
//   MV_FP8   Q expanded exactly to BF16 (e4m3 values are BF16 values) in
//            the workspace, one segment; the epilogue multiplies by
//            s_i s_j, since Sigma = diag(s) Q Q^T diag(s);
//   MV_F32   L = H + D with H = bf16(L), D = bf16(L - H) in the workspace;
//            Sigma ~= H H^T + H D^T + D H^T: each k-step stages the four
//            boxes H_I, D_I, H_J, D_J once and issues the three products
//            into one accumulator (the dropped D D^T and the rounding of D
//            are below 2^-16 |L_i| |L_j| per product term).
//
// Bound: tensor.  A CTA of a pair loads its 128 rows of the I panel and its
// 128 of the J panel: 64 KB per k-step of 3 x 256 x 256 x 64 multiply-adds
// (FP32), half of what a CTA alone on a 128 x 128 tile needs per
// multiply-add, which had made the L2 the limit (1.16 PFLOP/s).
//
// Work split.  P pairs fit the chip (one per two SMs).  All tiles but the
// last N mod P run whole; those last r tiles would leave most of a wave
// idle, so each is cut into floor(P / r) K-ranges whose partial sums go to
// the workspace and are added in range order by a second kernel.  With few
// tiles (small n) all of them are cut, from two chunks on (kernels' time, cut
// against whole: 300 x 2000 BF16 13.1 / 19.2 us, 2000 x 1000 FP32 30.7 / 31.3,
// 1500 x 5000 FP32 55.8 / 89.5).
//
// Every store of the epilogue and of the joining kernel covers 128 bytes of a
// row.  With the accumulators' own layout, one row per lane, the epilogue alone
// held a small or short-T call up (300 x 700 BF16: 27.5 us of kernel, now 13.0;
// 4000 x 700 51 -> 29; 2500 x 3000 29).
//
// Pipeline per CTA as in gemm_chunk.cuh's pair kernel: warp 0 (one thread)
// TMA producer, warp 1 of rank 0 (one thread) MMA issuer, warps 2..9 the
// epilogue, which also carries the running sum in FP32 registers (see the
// accumulation note below).  Every wait is bounded in time; a timeout is
// recorded in the device error word and the call returns MV_ERR_TIMEOUT.
#include <cooperative_groups.h>

#include "gemm.cuh"

namespace mv {

int sm_count();          // solve.cu

constexpr int kSigTile = 256;                      // rows and columns of a pair's tile
constexpr int kSigHalf = kSigTile / 2;             // rows of each panel that one CTA loads
constexpr uint32_t kSigBox = kSigHalf * kBK * 2;   // one 128 x 64 BF16 operand box (16 KB)
constexpr int kSigEpiWarps = 8;                    // 128 rows x 2 column groups of 128
constexpr int kSigThreads = 64 + 32 * kSigEpiWarps;
// Stage geometry by number of products per k-step: one (BF16, FP8) = boxes
// A, B and 6 stages; three (FP32 split) = boxes H_I, D_I, H_J, D_J and 3 stages.
// A tensor-memory partial sums at most 64 MMAs (16 k-steps x 4, or 5 x 12).
template <int NSEG> struct SigGeo {
    static constexpr int BOXES = NSEG == 3 ? 4 : 2;
    static constexpr int S = NSEG == 3 ? 3 : 6;
    static constexpr uint32_t STAGE = BOXES * kSigBox;
    static constexpr int CHUNK = NSEG == 3 ? 5 : 16;
};
constexpr size_t kSigSmem = 1024 + 6 * (size_t)2 * kSigBox + (2 * 6 + 4) * 8 + 16;   // the larger of the two

// Tile order: the upper triangle is walked in super-blocks of kSigGroup x
// kSigGroup tiles (row-major inside each, super-blocks row-major over the
// upper triangle), so the pairs that run at the same time share about
// 2 kSigGroup operand panels and read them from L2 rather than HBM.
constexpr int kSigGroup = 6;

__host__ __device__ __forceinline__ void tile_of(int t, int nb, int &I, int &J) {
    const int nsb = (nb + kSigGroup - 1) / kSigGroup;
    for (int P = 0; P < nsb; ++P) {
        const int i0 = P * kSigGroup, ri = nb - i0 < kSigGroup ? nb - i0 : kSigGroup;
        for (int Q = P; Q < nsb; ++Q) {
            const int j0 = Q * kSigGroup, rj = nb - j0 < kSigGroup ? nb - j0 : kSigGroup;
            if (Q == P) {                             // triangle of ri (ri + 1) / 2 tiles
                const int cnt = ri * (ri + 1) / 2;
                if (t < cnt) {
                    int a = 0;
                    while (t >= ri - a) {
                        t -= ri - a;
                        ++a;
                    }
                    I = i0 + a;
                    J = i0 + a + t;
                    return;
                }
                t -= cnt;
            } else {                                  // rectangle of ri x rj tiles
                const int cnt = ri * rj;
                if (t < cnt) {
                    I = i0 + t / rj;
                    J = j0 + t % rj;
                    return;
                }
                t -= cnt;
            }
        }
    }
    I = J = 0;                                        // not reached: t < nb (nb + 1) / 2
}

// Whole tiles first, then `cut` tiles of `parts` K-ranges each.
struct SigSplit {
    int whole, cut, parts;
};
constexpr int kSigMaxParts = 64;
static SigSplit sigma_split(int64_t tiles, int pairs, int chunks) {
    SigSplit w;
    w.whole = (int)(tiles / pairs * pairs);
    w.cut = (int)(tiles - w.whole);
    w.parts = w.cut > 0 ? std::min(std::min(pairs / w.cut, chunks), kSigMaxParts) : 1;
    if (w.parts < 2) {
        w.whole = (int)tiles;
        w.cut = 0;
        w.parts = 1;
    }
    return w;
}

// Accumulation.  The tensor core adds each MMA's products into the FP32
// accumulator with a rounding that loses up to about an ulp of the running
// sum, with one sign when the terms have one sign (the diagonal of Sigma):
// over thousands of MMAs that is a bias of order 1e-4.  So a tile is
// accumulated in chunks of at most 64 MMAs (SigGeo::CHUNK k-steps), alternately
// into two 256-column tensor-memory buffers; the epilogue warps add every
// finished chunk into FP32 registers (round-to-nearest, fixed order) while
// the MMA warp fills the other buffer.
template <int NSEG>
__global__ void __launch_bounds__(kSigThreads, 1)
sigma_pair_kernel(const __grid_constant__ CUtensorMap tmH, const __grid_constant__ CUtensorMap tmD, int n, int K,
                  int nb, SigSplit w, const float *__restrict__ rs, float *__restrict__ Sig, int64_t ldS,
                  float *__restrict__ part) {
    using Geo = SigGeo<NSEG>;
    constexpr int S = Geo::S;
    constexpr uint32_t COLS = 2 * kSigTile;           // tensor-memory columns: all 512
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (uint32_t)(reinterpret_cast<uintptr_t>(smem_raw) & 1023u)) & 1023u);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + S * Geo::STAGE);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * S + 4);
    const uint32_t full0 = umma::smem_u32(bars), empty0 = umma::smem_u32(bars + S);
    const uint32_t tfull0 = umma::smem_u32(bars + 2 * S), tempty0 = umma::smem_u32(bars + 2 * S + 2);
    // box b of stage s
    auto box = [&](int st, int b) { return umma::smem_u32(smem + (size_t)st * Geo::STAGE + (size_t)b * kSigBox); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = umma::cluster_ctarank();    // 0: issues the MMAs
    const int unit = (int)blockIdx.x >> 1;
    int tile = unit, range = 0, slot = -1;            // slot: the partial's place, -1 for a whole tile
    if (unit >= w.whole) {
        slot = unit - w.whole;
        tile = w.whole + slot / w.parts;
        range = slot % w.parts;
    }
    int I, J;
    tile_of(tile, nb, I, J);
    const int m0 = I * kSigTile + (int)rank * kSigHalf;    // this CTA's rows of the tile and of panel I
    const int b0 = J * kSigTile + (int)rank * kSigHalf;    // its rows of panel J
    const int steps = (K + kBK - 1) / kBK;
    const int all = (steps + Geo::CHUNK - 1) / Geo::CHUNK;
    // chunks [c0, c1) of this unit
    const int c0 = slot < 0 ? 0 : (int)((int64_t)all * range / w.parts);
    const int c1 = slot < 0 ? all : (int)((int64_t)all * (range + 1) / w.parts);
    const int k0 = c0 * Geo::CHUNK, k1 = min(steps, c1 * Geo::CHUNK);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            umma::mbar_init(full0 + 8 * s, 1);
            umma::mbar_init(empty0 + 8 * s, 1);
        }
        for (int b = 0; b < 2; ++b) {
            umma::mbar_init(tfull0 + 8 * b, 1);                  // tcgen05.commit of a chunk
            umma::mbar_init(tempty0 + 8 * b, 2 * kSigEpiWarps);  // both CTAs' epilogue warps drained it
        }
        umma::mbar_fence_init();
    }
    if (warp == 1) {
        umma::tmem_alloc_pair(umma::smem_u32(tmem_slot), COLS);
        umma::tmem_relinquish_pair();
    }
    umma::fence_before_sync();
    cooperative_groups::this_cluster().sync();        // both CTAs' barriers exist
    umma::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    const uint32_t full_r0 = umma::mapa_rank(full0, 0);

    if (warp == 0) {
        if (lane == 0) {
            umma::prefetch_tensormap(&tmH);
            if (NSEG > 1) umma::prefetch_tensormap(&tmD);
            for (int g = k0; g < k1; ++g) {
                const int j = g - k0, s = j % S;
                if (!umma::mbar_wait(empty0 + 8 * s, ((uint32_t)(j / S) & 1u) ^ 1u, kWaitNs)) {
                    atomicExch(&g_gemm_err, 1);
                    break;
                }
                const uint32_t fb = full_r0 + 8u * (uint32_t)s;
                if (rank == 0) umma::mbar_arrive_expect_tx(full0 + 8 * s, 2 * Geo::STAGE);
                if (NSEG == 3) {                       // H_I, D_I, H_J, D_J
                    umma::tma_load_2d_pair(box(s, 0), &tmH, g * kBK, m0, fb);
                    umma::tma_load_2d_pair(box(s, 1), &tmD, g * kBK, m0, fb);
                    umma::tma_load_2d_pair(box(s, 2), &tmH, g * kBK, b0, fb);
                    umma::tma_load_2d_pair(box(s, 3), &tmD, g * kBK, b0, fb);
                } else {                               // A_I, A_J
                    umma::tma_load_2d_pair(box(s, 0), &tmH, g * kBK, m0, fb);
                    umma::tma_load_2d_pair(box(s, 1), &tmH, g * kBK, b0, fb);
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            constexpr uint32_t idesc = umma::idesc_bf16_f32(kSigTile, kSigTile);
            bool ok = true;
            for (int c = c0; c < c1 && ok; ++c) {
                const int i = c - c0, b = i & 1;
                if (i >= 2 && !umma::mbar_wait(tempty0 + 8 * b, (uint32_t)((i >> 1) - 1) & 1u, 2 * kWaitNs)) {
                    atomicExch(&g_gemm_err, 4);
                    break;
                }
                umma::fence_after_sync();
                const uint32_t acc = tmem + (uint32_t)(b * kSigTile);
                const int g0 = c * Geo::CHUNK, g1 = min(k1, g0 + Geo::CHUNK);
                for (int g = g0; g < g1; ++g) {
                    const int j = g - k0, s = j % S;
                    if (!umma::mbar_wait(full0 + 8 * s, (uint32_t)(j / S) & 1u, kWaitNs)) {
                        atomicExch(&g_gemm_err, 2);
                        ok = false;
                        break;
                    }
                    umma::fence_after_sync();
                    if (NSEG == 3) {
                        // H_I H_J^T + H_I D_J^T + D_I H_J^T from the one stage
                        const uint64_t hi = umma::desc_kmajor_sw128(box(s, 0)), di = umma::desc_kmajor_sw128(box(s, 1));
                        const uint64_t hj = umma::desc_kmajor_sw128(box(s, 2)), dj = umma::desc_kmajor_sw128(box(s, 3));
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k) {
                            umma::mma_bf16_pair(acc, hi + 2 * k, hj + 2 * k, idesc, (g != g0 || k != 0) ? 1u : 0u);
                            umma::mma_bf16_pair(acc, hi + 2 * k, dj + 2 * k, idesc, 1u);
                            umma::mma_bf16_pair(acc, di + 2 * k, hj + 2 * k, idesc, 1u);
                        }
                    } else {
                        const uint64_t da = umma::desc_kmajor_sw128(box(s, 0)), db = umma::desc_kmajor_sw128(box(s, 1));
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k)
                            umma::mma_bf16_pair(acc, da + 2 * k, db + 2 * k, idesc, (g != g0 || k != 0) ? 1u : 0u);
                    }
                    umma::mma_commit_pair(empty0 + 8 * s, (uint16_t)3);
                }
                if (ok) umma::mma_commit_pair(tfull0 + 8 * b, (uint16_t)3);
            }
        }
        __syncwarp();
    } else {
        const int q = warp & 3, grp = (warp - 2) >> 2;       // tile rows 32 q .., columns 128 grp ..
        const int row = m0 + 32 * q + lane, cb = J * kSigTile + grp * 128;
        const uint32_t tempty_r0 = umma::mapa_rank(tempty0, 0);
        float acc[128];
#pragma unroll
        for (int j = 0; j < 128; ++j) acc[j] = 0.f;
        bool ok = true;
        for (int c = c0; c < c1; ++c) {
            const int i = c - c0, b = i & 1;
            if (!umma::mbar_wait(tfull0 + 8 * b, (uint32_t)(i >> 1) & 1u, 4 * kWaitNs)) {
                ok = false;
                break;
            }
            umma::fence_after_sync();
            const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * kSigTile + grp * 128);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                uint32_t r[32];
                umma::tmem_ld_32x32b_x32(ta + (uint32_t)(p * 32), r);
                umma::tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[p * 32 + j] += __uint_as_float(r[j]);
            }
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma::mbar_arrive_cluster(tempty_r0 + 8u * (uint32_t)b);
        }
        if (!ok) {
            if (lane == 0) atomicExch(&g_gemm_err, 3);
        } else if (slot >= 0) {                              // a K-range's partial, added by sigma_join_kernel
            float *dst = part + (int64_t)slot * kSigTile * kSigTile + ((((int)rank * 4 + q) * 2 + grp) * 128) * 32 + lane;
#pragma unroll
            for (int j = 0; j < 128; ++j) dst[j * 32] = acc[j];
        } else {
            const bool diag = I == J;
            const float sr = (rs != nullptr && row < n) ? rs[row] : 1.f;
            if (rs != nullptr) {
#pragma unroll
                for (int j = 0; j < 128; ++j) acc[j] *= sr * (cb + j < n ? __ldg(rs + cb + j) : 0.f);
            }
            // Rows of the tile: the accumulators hold one row per lane, and a
            // store of 32 rows costs 32 memory sectors, so each 32 x 32 piece is
            // turned in shared memory (the stages are free: the last chunk's
            // MMAs have read them all) and written 128 bytes of a row at a time.
            const int r0 = m0 + 32 * q, rows = min(32, n - r0), cols = min(128, n - cb);
            float *turn = reinterpret_cast<float *>(smem) + (warp - 2) * (32 * 33);
            if (rows > 0 && cols > 0) {
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const int c = cb + p * 32, col = c + lane;
                    if (p * 32 >= cols || (diag && c + 31 < r0)) continue;      // nothing to store: the same in every lane
#pragma unroll
                    for (int j = 0; j < 32; ++j) turn[lane * 33 + j] = acc[p * 32 + j];
                    __syncwarp();
                    float *dst = Sig + (int64_t)r0 * ldS + col;
                    const int last = col >= n ? 0 : (diag ? min(rows, col - r0 + 1) : rows);   // rows of this column
#pragma unroll 8
                    for (int r = 0; r < rows; ++r, dst += ldS)
                        if (r < last) *dst = turn[r * 33 + lane];
                    __syncwarp();
                }
                // mirror: for fixed j the 32 lanes write 32 consecutive floats
                float *dst = Sig + (int64_t)cb * ldS + row;
                const int first = row >= n ? cols : (diag ? row - cb + 1 : 0);                   // columns above the diagonal
#pragma unroll
                for (int j = 0; j < 128; ++j, dst += ldS)
                    if (j >= first && j < cols) *dst = acc[j];
            }
        }
    }
    umma::fence_before_sync();
    cooperative_groups::this_cluster().sync();        // the peer no longer reads or signals this CTA
    umma::fence_after_sync();
    if (warp == 1) umma::tmem_dealloc_pair(tmem, COLS);
}

// The cut tiles: partials added in range order, scaled, written with their
// mirror.  One block of 32 x 8 threads per 32 x 32 piece of a tile.  A partial
// is stored as the epilogue's warps hold it, 32 rows by 128 columns each, the
// rows of a column side by side (both sides then move whole 128-byte lines).
__global__ void __launch_bounds__(256)
sigma_join_kernel(const float *__restrict__ part, SigSplit w, int nb, int n, const float *__restrict__ rs,
                  float *__restrict__ Sig, int64_t ldS) {
    __shared__ float t[32][33];
    int I, J;
    tile_of(w.whole + (int)blockIdx.y, nb, I, J);
    const int pr = (int)blockIdx.x / (kSigTile / 32) * 32, pc = (int)blockIdx.x % (kSigTile / 32) * 32;
    const int r0 = I * kSigTile + pr, c0 = J * kSigTile + pc;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    if (r0 >= n || c0 >= n || (I == J && pc < pr)) return;   // uniform: nothing on or above the diagonal here
    const float *src = part + (int64_t)blockIdx.y * w.parts * kSigTile * kSigTile +
                       (((pr / 32) * 2 + pc / 128) * 128 + pc % 128) * 32 + tx;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int p = 0; p < w.parts; ++p)
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] += __ldcg(src + (int64_t)p * kSigTile * kSigTile + (ty + 8 * k) * 32);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int c = ty + 8 * k, row = r0 + tx, col = c0 + c;
        if (rs != nullptr && row < n && col < n) s[k] *= rs[row] * rs[col];
        t[c][tx] = s[k];
        if (row < n && col < n && col >= row) Sig[(int64_t)col * ldS + row] = s[k];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = ty + 8 * k;
        const int row = r0 + r, col = c0 + tx;
        if (row < n && col < n && col > row) Sig[(int64_t)row * ldS + col] = t[tx][r];
    }
}

// H = bf16(L), D = bf16(L - H), row by row (4 columns per thread step).
__global__ void split_hi_lo_kernel(const float *__restrict__ L, int64_t ld, int n, int T, __nv_bfloat16 *__restrict__ H,
                                   __nv_bfloat16 *__restrict__ D, int64_t ldo) {
    const int64_t quads = (T + 3) / 4;
    for (int64_t r = blockIdx.y; r < n; r += gridDim.y) {
        const float *src = L + r * ld;
        for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < quads; q += (int64_t)gridDim.x * blockDim.x) {
            const int64_t c = 4 * q;
            const float4 x = *reinterpret_cast<const float4 *>(src + c);   // c + 3 < ld: ld is a multiple of 4
            const float xs[4] = {x.x, x.y, x.z, x.w};
            __nv_bfloat16 h[4], d[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float v = c + j < T ? xs[j] : 0.f;
                h[j] = __float2bfloat16_rn(v);
                d[j] = __float2bfloat16_rn(v - __bfloat162float(h[j]));
            }
            *reinterpret_cast<uint2 *>(H + r * ldo + c) = *reinterpret_cast<const uint2 *>(h);
            *reinterpret_cast<uint2 *>(D + r * ldo + c) = *reinterpret_cast<const uint2 *>(d);
        }
    }
}

// Q (e4m3) -> BF16, exact (every e4m3 value is a BF16 value).
__global__ void expand_fp8_kernel(const uint8_t *__restrict__ Q, int64_t ld, int n, int T, __nv_bfloat16 *__restrict__ B,
                                  int64_t ldo) {
    const int64_t quads = (T + 3) / 4;
    for (int64_t r = blockIdx.y; r < n; r += gridDim.y) {
        const uint8_t *src = Q + r * ld;
        for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < quads; q += (int64_t)gridDim.x * blockDim.x) {
            const int64_t c = 4 * q;
            const uint32_t w = *reinterpret_cast<const uint32_t *>(src + c);   // c + 3 < ld: ld is a multiple of 16
            float f[4];
            Store<MV_FP8_E4M3>::four(w, f);
            __nv_bfloat16 b[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = __float2bfloat16_rn(c + j < T ? f[j] : 0.f);
            *reinterpret_cast<uint2 *>(B + r * ldo + c) = *reinterpret_cast<const uint2 *>(b);
        }
    }
}

static int64_t sigma_ldo(int64_t T) { return (T + 7) / 8 * 8; }   // BF16 row pitch: 16-byte rows

static int sigma_check(const mv_problem *P) {
    if (P == nullptr || P->L == nullptr) return MV_ERR_INVALID_ARG;
    if (P->dtype != MV_F32 && P->dtype != MV_BF16 && P->dtype != MV_FP8_E4M3) return MV_ERR_INVALID_ARG;
    if (P->layout != MV_LAYOUT_NT) return MV_ERR_INVALID_ARG;
    if (P->n < 1 || P->T < 1 || P->ld < P->T) return MV_ERR_INVALID_ARG;
    if (P->n > 32768 || P->T >= (1LL << 31))
        return record_message(MV_ERR_UNSUPPORTED, "mv_sigma_form: n must be <= 32768 and T below 2^31");
    const int es = dtype_size(P->dtype);
    if (((uintptr_t)P->L) % 16 != 0 || (P->ld * es) % 16 != 0) return MV_ERR_INVALID_ARG;
    if (P->dtype == MV_FP8_E4M3 && P->row_scale == nullptr) return MV_ERR_INVALID_ARG;
    return MV_OK;
}

static size_t sigma_ws_bytes(const mv_problem *P) {
    const size_t plane = align_up((size_t)P->n * (size_t)sigma_ldo(P->T) * 2, 256);
    if (P->dtype == MV_F32) return 2 * plane;
    if (P->dtype == MV_FP8_E4M3) return plane;
    return 0;
}
// Partials of cut tiles: fewer than `pairs` units of one tile each.  Room for
// them is optional (without it no tile is cut); the SM count of the part,
// so that the size does not depend on the current device.
constexpr int kSigPairs = 152 / 2;
constexpr size_t kSigPartBytes = (size_t)kSigPairs * kSigTile * kSigTile * 4;

}  // namespace mv

using namespace mv;

extern "C" {

size_t mv_sigma_workspace_size(const mv_problem *P) {
    if (sigma_check(P) != MV_OK) return 0;
    return sigma_ws_bytes(P) + kSigPartBytes;
}

int mv_sigma_form(const mv_problem *P, float *d_Sigma, int64_t ldS, void *d_ws, size_t ws_bytes, mv_stream_t stream) {
    MV_TRY(sigma_check(P));
    if (d_Sigma == nullptr || ldS < P->n || (ldS & 3) != 0 || ((uintptr_t)d_Sigma) % 16 != 0) return MV_ERR_INVALID_ARG;
    const size_t need = sigma_ws_bytes(P);
    if (P->dtype != MV_BF16 && (d_ws == nullptr || ws_bytes < need || ((uintptr_t)d_ws) % 256 != 0))
        return MV_ERR_WORKSPACE;
    (void)cudaGetLastError();
    cudaStream_t s = (cudaStream_t)stream;
    const int n = (int)P->n, T = (int)P->T;
    const int nb = (n + kSigTile - 1) / kSigTile;
    const int64_t tiles = (int64_t)nb * (nb + 1) / 2;
    const int chunk = P->dtype == MV_F32 ? SigGeo<3>::CHUNK : SigGeo<1>::CHUNK;
    const int chunks = ((T + kBK - 1) / kBK + chunk - 1) / chunk;
    const bool room = d_ws != nullptr && ((uintptr_t)d_ws) % 256 == 0 && ws_bytes >= need + kSigPartBytes;
    const SigSplit w = sigma_split(tiles, room ? std::min(sm_count() / 2, kSigPairs) : 1, chunks);
    float *part = reinterpret_cast<float *>(reinterpret_cast<char *>(d_ws) + need);
    const int64_t ldo = sigma_ldo(T);
    const size_t plane = align_up((size_t)n * (size_t)ldo * 2, 256);
    CUtensorMap tmH, tmD;
    int nseg = 1;
    const float *rs = nullptr;
    dim3 cgrid((unsigned)std::min<int64_t>((T / 4 + 255) / 256 + 1, 8), (unsigned)std::min(n, 4096));
    if (P->dtype == MV_BF16) {
        MV_TRY(make_map_bf16(&tmH, P->L, n, T, P->ld, kSigHalf));
        tmD = tmH;
    } else if (P->dtype == MV_FP8_E4M3) {
        __nv_bfloat16 *B = reinterpret_cast<__nv_bfloat16 *>(d_ws);
        expand_fp8_kernel<<<cgrid, 256, 0, s>>>(reinterpret_cast<const uint8_t *>(P->L), P->ld, n, T, B, ldo);
        MV_TRY(make_map_bf16(&tmH, B, n, T, ldo, kSigHalf));
        tmD = tmH;
        rs = P->row_scale;
    } else {
        __nv_bfloat16 *H = reinterpret_cast<__nv_bfloat16 *>(d_ws);
        __nv_bfloat16 *D = reinterpret_cast<__nv_bfloat16 *>(reinterpret_cast<char *>(d_ws) + plane);
        split_hi_lo_kernel<<<cgrid, 256, 0, s>>>(reinterpret_cast<const float *>(P->L), P->ld, n, T, H, D, ldo);
        MV_TRY(make_map_bf16(&tmH, H, n, T, ldo, kSigHalf));
        MV_TRY(make_map_bf16(&tmD, D, n, T, ldo, kSigHalf));
        nseg = 3;
    }
    MV_CUDA_TRY(cudaGetLastError());
    static int attrs = -1;
    if (attrs < 0)
        attrs = (cudaFuncSetAttribute(sigma_pair_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kSigSmem) == cudaSuccess &&
                 cudaFuncSetAttribute(sigma_pair_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kSigSmem) == cudaSuccess)
                    ? MV_OK
                    : MV_ERR_CUDA;
    if (attrs != MV_OK) return record_message(MV_ERR_CUDA, "sigma GEMM: shared-memory attribute refused");
    int zero = 0;
    MV_CUDA_TRY(cudaMemcpyToSymbolAsync(g_gemm_err, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)(w.whole + w.cut * w.parts));
    cfg.blockDim = dim3(kSigThreads);
    cfg.dynamicSmemBytes = kSigSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (nseg == 3)
        MV_CUDA_TRY(cudaLaunchKernelEx(&cfg, sigma_pair_kernel<3>, tmH, tmD, n, T, nb, w, rs, d_Sigma, ldS, part));
    else
        MV_CUDA_TRY(cudaLaunchKernelEx(&cfg, sigma_pair_kernel<1>, tmH, tmD, n, T, nb, w, rs, d_Sigma, ldS, part));
    if (w.cut > 0)
        sigma_join_kernel<<<dim3((kSigTile / 32) * (kSigTile / 32), (unsigned)w.cut), 256, 0, s>>>(part, w, nb, n, rs, d_Sigma,
                                                                                                  ldS);
    MV_CUDA_TRY(cudaGetLastError());
    int err = 0;
    MV_CUDA_TRY(cudaMemcpyFromSymbolAsync(&err, g_gemm_err, sizeof(int), 0, cudaMemcpyDeviceToHost, s));
    MV_CUDA_TRY(cudaStreamSynchronize(s));
    if (err != 0) {
        char msg[96];
        snprintf(msg, sizeof(msg), "sigma GEMM pipeline wait timed out (stage code %d)", err);
        return record_message(MV_ERR_TIMEOUT, msg);
    }
    return MV_OK;
}

}  // extern "C"
