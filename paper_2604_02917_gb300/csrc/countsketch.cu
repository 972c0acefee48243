// CountSketch stage of STR (Sec. 2.3, construction (2)): tilde L = L Phi with
// Phi(t, h(t)) = s_t and every other entry 0, i.e. column j of tilde L is
// the signed sum of the columns t of L whose period hashes to bucket j.
//
// Deterministic by construction: the periods of each bucket are listed in
// ascending order (a histogram, a scan, an atomic fill and a per-bucket
// sort), and every output is summed over its list in that order.
//
//  * MV_LAYOUT_TN (L^T stored T x n): a CTA takes 8 buckets and a chunk of
//    256 x VEC assets.  The buckets' lists are one contiguous run, which the
//    CTA fetches first and each thread then walks from end to end, kCsLoads
//    signed 16-byte slices of rows of L^T in flight (a warp reads 512
//    contiguous bytes of a row) whatever the bucket boundaries; each finished
//    bucket parks its sum in shared memory, and the 8 results go out as 8
//    consecutive floats of tilde L's row (n x m, row-major).  Every row of L^T
//    is read once in total: HBM-bound.
//  * MV_LAYOUT_NT (L stored n x T): a CTA stages one asset row of L in
//    shared memory (T e bytes, at most 200 KB) and its threads gather the
//    buckets from it.
// FP8 rows are multiplied by their scale at the write.
#include <algorithm>

#include "mv_internal.cuh"
#include "umma.cuh"

namespace mv {

constexpr int kCsThreads = 256, kCsThreadsFew = 64;   // TN: per CTA, and where that leaves SMs idle
constexpr int kCsGroup = 8;                   // buckets per CTA (TN)
constexpr int kCsLoads = 8;                   // row slices in flight per thread (TN)
constexpr int kCsCacheMax = 2048;             // list entries a CTA keeps in shared memory, at most (TN)
constexpr int kCsNtThreads = 512;
constexpr size_t kCsNtMaxRow = 200 * 1024;    // staged row bytes (NT)
constexpr int kCsMaxBucket = 4096;            // periods per bucket the in-place sort accepts

struct CsWs {
    int *cnt, *off, *fill, *err;
    unsigned *list;                           // period | sign bit 31 (negative)
};

static size_t cs_ws_bytes(int64_t T, int64_t m) {
    return align_up(4 * (size_t)m, 256) * 2 + align_up(4 * ((size_t)m + 1), 256) + align_up(4 * (size_t)T, 256) + 256;
}

// Counters and the error word first: one memset clears them.
static size_t cs_zero_bytes(int64_t m) { return 2 * align_up(4 * (size_t)m, 256) + 256; }

static CsWs cs_carve(void *ws, int64_t T, int64_t m) {
    CsWs w;
    char *p = reinterpret_cast<char *>(ws);
    w.cnt = reinterpret_cast<int *>(p);
    p += align_up(4 * (size_t)m, 256);
    w.fill = reinterpret_cast<int *>(p);
    p += align_up(4 * (size_t)m, 256);
    w.err = reinterpret_cast<int *>(p);
    p += 256;
    w.off = reinterpret_cast<int *>(p);
    p += align_up(4 * ((size_t)m + 1), 256);
    w.list = reinterpret_cast<unsigned *>(p);
    return w;
}

// The kernels run as a chain of programmatic dependent launches: each starts
// while the one before drains, waits for it, then lets the next start.  What
// the ones before wrote (counts, offsets, list) is read by ordinary loads
// through plain pointers: the read-only path, which const __restrict__ and
// __ldg ask for, is for memory that nobody writes while the kernel lives, and
// this kernel may be alive before the writes.  The n x T gather is launched
// the ordinary way and keeps that path: every entry of the list is a load in
// every row of L (2000 x 40000 to 40000 columns FP32 799 us, in the chain with
// ordinary loads 877; 5440 x 12000 to 512 153 against 206).
__device__ __forceinline__ void cs_chain() {
    umma::grid_dependency_wait();
    umma::launch_dependents();
}
template <typename... Params, typename... Args>
static cudaError_t cs_start(void (*kern)(Params...), dim3 grid, int threads, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}

__global__ void cs_count_kernel(const int *__restrict__ h, int T, int m, int *__restrict__ cnt, int *__restrict__ err) {
    cs_chain();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
        const int b = h[t];
        if (b < 0 || b >= m) {
            atomicExch(err, 1);
            continue;
        }
        atomicAdd(&cnt[b], 1);
    }
}

// Exclusive scan of m counts by one block of 1024 threads (chunked).
__global__ void __launch_bounds__(1024) cs_scan_kernel(const int *cnt, int m, int *off) {
    __shared__ int part[1024];
    cs_chain();
    const int per = (m + 1023) / 1024;
    const int b0 = threadIdx.x * per, b1 = min(m, b0 + per);
    int s = 0;
    for (int b = b0; b < b1; ++b) s += cnt[b];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int d = 1; d < 1024; d <<= 1) {      // inclusive Hillis-Steele scan of the chunk sums
        const int v = threadIdx.x >= d ? part[threadIdx.x - d] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    int run = threadIdx.x == 0 ? 0 : part[threadIdx.x - 1];
    for (int b = b0; b < b1; ++b) {
        off[b] = run;
        run += cnt[b];
    }
    if (threadIdx.x == 1023) off[m] = part[1023];
}

__global__ void cs_fill_kernel(const int *__restrict__ h, const int8_t *__restrict__ sign, int T, int m,
                               const int *off, int *__restrict__ fill, unsigned *list) {
    cs_chain();
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < T; t += gridDim.x * blockDim.x) {
        const int b = h[t];
        if (b < 0 || b >= m) continue;
        const int pos = off[b] + atomicAdd(&fill[b], 1);
        list[pos] = (unsigned)t | (sign[t] < 0 ? 0x80000000u : 0u);
    }
}

constexpr int kCsShort = 16;                  // periods per bucket that one thread sorts

__device__ __forceinline__ unsigned cs_key(unsigned e) { return e & 0x7fffffffu; }

// Ascending periods within one bucket of nb <= kCsShort entries at
// list[p0..), in registers through a fixed odd-even transposition network (a
// uniform hash leaves a few periods per bucket).
__device__ __forceinline__ void cs_sort_bucket(unsigned *list, int p0, int nb) {
    unsigned v[kCsShort];
#pragma unroll
    for (int i = 0; i < kCsShort; ++i) v[i] = i < nb ? list[p0 + i] : 0xffffffffu;   // padding sorts last
#pragma unroll
    for (int r = 0; r < kCsShort; ++r) {
#pragma unroll
        for (int i = r & 1; i + 1 < kCsShort; i += 2) {
            const unsigned x = v[i], y = v[i + 1];
            const bool sw = cs_key(x) > cs_key(y);
            v[i] = sw ? y : x;
            v[i + 1] = sw ? x : y;
        }
    }
#pragma unroll
    for (int i = 0; i < kCsShort; ++i)
        if (i < nb) list[p0 + i] = v[i];
}

// Sort every bucket (a bucket above kCsMaxBucket periods is refused): short
// ones a thread each, longer ones by the whole warp, each lane placing its
// entries by counting the smaller keys (periods are distinct): nb^2 / 128
// reads of four keys from shared memory, a few ms at worst.  A warp takes
// `per` buckets, 32, or one where the average bucket is long.  (One thread
// inserting in global memory took most of the call where buckets are long:
// 100 x 30000 to 20 columns, 1500 periods each, 54 ms, and 234 ms in blocks of
// four warps; now 0.52 ms.)
__global__ void __launch_bounds__(kWarp)
cs_sort_kernel(const int *off, int m, int per, unsigned *list, int *__restrict__ err) {
    __shared__ __align__(16) unsigned buf[kCsMaxBucket];   // (period, sign) as 2 t + sign: the same order
    cs_chain();
    const int lane = threadIdx.x;
    for (int b0 = blockIdx.x * per; b0 < m; b0 += gridDim.x * per) {
        const int b = b0 + lane;
        const bool mine = lane < per && b < m;
        const int p0 = mine ? off[b] : 0, nb = mine ? off[b + 1] - p0 : 0;
        if (nb > kCsMaxBucket)
            atomicExch(err, 2);
        else if (nb <= kCsShort)
            cs_sort_bucket(list, p0, nb);
        for (unsigned todo = __ballot_sync(0xffffffffu, nb > kCsShort && nb <= kCsMaxBucket); todo != 0; todo &= todo - 1) {
            const int src = __ffs((int)todo) - 1;
            const int q0 = __shfl_sync(0xffffffffu, p0, src), nq = __shfl_sync(0xffffffffu, nb, src);
            for (int i = lane; i < nq + (-nq & 3); i += kWarp) {
                const unsigned e = i < nq ? list[q0 + i] : 0u;
                buf[i] = i < nq ? (e << 1) | (e >> 31) : 0xffffffffu;      // the padding counts nowhere
            }
            __syncwarp();
            for (int i = lane; i < nq; i += kWarp) {
                const unsigned x = buf[i];
                int rank = 0;
#pragma unroll 4
                for (int k = 0; k < nq; k += 4) {
                    const uint4 y = *reinterpret_cast<const uint4 *>(buf + k);
                    rank += (y.x < x ? 1 : 0) + (y.y < x ? 1 : 0) + (y.z < x ? 1 : 0) + (y.w < x ? 1 : 0);
                }
                list[q0 + rank] = (x >> 1) | (x << 31);
            }
            __syncwarp();
        }
    }
}

template <int DT, int NT>
__global__ void __launch_bounds__(NT)
cs_tn_kernel(const void *__restrict__ Lt, int64_t ld, int n, int m, const int *off,
             const unsigned *list, const float *__restrict__ rs, float *__restrict__ out, int64_t ldS,
             int ncache) {
    using St = Store<DT>;
    constexpr int VEC = St::VEC;
    constexpr int CHUNK = NT * VEC;
    extern __shared__ __align__(16) float tile[];                 // [kCsGroup][CHUNK]
    const int j0 = blockIdx.x * kCsGroup;
    const int a0 = blockIdx.y * CHUNK;
    const int my = a0 + threadIdx.x * VEC;
    const char *base = reinterpret_cast<const char *>(Lt);
    cs_chain();
    // the group's 9 bucket boundaries and its run of the list (what exceeds the cache is read as it comes)
    __shared__ int bnd[kCsGroup + 1];
    unsigned *cache = reinterpret_cast<unsigned *>(tile + kCsGroup * CHUNK);
    if (threadIdx.x <= kCsGroup) bnd[threadIdx.x] = off[min(j0 + (int)threadIdx.x, m)];
    __syncthreads();
    const int p0 = bnd[0], p1 = bnd[kCsGroup];
    for (int k = threadIdx.x; k < min(p1 - p0, ncache); k += NT) cache[k] = list[p0 + k];
    __syncthreads();
    float acc[VEC];
#pragma unroll
    for (int q = 0; q < VEC; ++q) acc[q] = 0.f;
    int g = 0;
    auto park = [&] {                              // bucket g is complete
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
            tile[g * CHUNK + threadIdx.x * VEC + q] = acc[q];
            acc[q] = 0.f;
        }
        ++g;
    };
    for (int p = p0; p < p1; p += kCsLoads) {
        unsigned e[kCsLoads];
        uint4 u[kCsLoads];
#pragma unroll
        for (int k = 0; k < kCsLoads; ++k) {
            const int at = p + k - p0;
            e[k] = p + k < p1 ? (at < ncache ? cache[at] : list[p + k]) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kCsLoads; ++k)
            u[k] = my < n && p + k < p1 ? ld_stream16(base + ((int64_t)(e[k] & 0x7fffffffu) * ld + my) *
                                                                 (int64_t)sizeof(typename St::elem))
                                        : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int k = 0; k < kCsLoads; ++k) {
            if (p + k >= p1) break;
            while (p + k >= bnd[g + 1]) park();     // the same in every thread
            float f[VEC];
            St::unpack(u[k], f);
            if (e[k] & 0x80000000u) {
#pragma unroll
                for (int q = 0; q < VEC; ++q) acc[q] -= f[q];
            } else {
#pragma unroll
                for (int q = 0; q < VEC; ++q) acc[q] += f[q];
            }
        }
    }
    while (g < kCsGroup) park();
    __syncthreads();
    // row a of tilde L gets the kCsGroup consecutive buckets j0 ..
    const bool full = j0 + kCsGroup <= m && (ldS & 3) == 0;
    for (int k = threadIdx.x; k < CHUNK; k += NT) {
        const int a = a0 + k;
        if (a >= n) break;
        const float s = rs ? rs[a] : 1.f;
        float v[kCsGroup];
#pragma unroll
        for (int g = 0; g < kCsGroup; ++g) v[g] = tile[g * CHUNK + k] * s;
        float *dst = out + (int64_t)a * ldS + j0;
        if (full) {
            *reinterpret_cast<float4 *>(dst) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4 *>(dst + 4) = make_float4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
            for (int g = 0; g < kCsGroup; ++g)
                if (j0 + g < m) dst[g] = v[g];
        }
    }
}

template <int DT>
__global__ void __launch_bounds__(kCsNtThreads)
cs_nt_kernel(const void *__restrict__ L, int64_t ld, int T, int m, const int *__restrict__ off,
             const unsigned *__restrict__ list, const float *__restrict__ rs, float *__restrict__ out, int64_t ldS) {
    using St = Store<DT>;
    using E = typename St::elem;
    extern __shared__ __align__(16) unsigned char row[];
    const int i = blockIdx.x;
    const int es = (int)sizeof(E);
    const int64_t bytes = ((int64_t)T * es + 15) / 16 * 16;       // within the row: ld e is a multiple of 16
    const char *src = reinterpret_cast<const char *>(L) + (int64_t)i * ld * es;
    for (int64_t o = (int64_t)threadIdx.x * 16; o < bytes; o += (int64_t)kCsNtThreads * 16)
        *reinterpret_cast<uint4 *>(row + o) = ld_stream16(src + o);
    __syncthreads();
    const E *r = reinterpret_cast<const E *>(row);
    const float s = rs ? rs[i] : 1.f;
    for (int j = threadIdx.x; j < m; j += kCsNtThreads) {
        float acc = 0.f;
        const int p1 = off[j + 1];
        for (int p = off[j]; p < p1; ++p) {
            const unsigned e = __ldg(list + p);
            const int t = (int)(e & 0x7fffffffu);
            float x;
            if constexpr (DT == MV_F32) {
                x = r[t];
            } else if constexpr (DT == MV_BF16) {
                x = __bfloat162float(r[t]);
            } else {
                __half_raw hh = __nv_cvt_fp8_to_halfraw(reinterpret_cast<const __nv_fp8_storage_t *>(r)[t], __NV_E4M3);
                x = __half2float(*reinterpret_cast<__half *>(&hh));
            }
            acc = (e & 0x80000000u) ? acc - x : acc + x;
        }
        out[(int64_t)i * ldS + j] = acc * s;
    }
}

template <typename K>
static int cs_smem_attr(K k, size_t bytes) {
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess
               ? MV_OK
               : record_message(MV_ERR_CUDA, "countsketch: shared-memory attribute refused");
}

template <int DT, int NT>
static int cs_launch_tn(const void *L, int64_t ld, int n, int T, int m, const CsWs &w, const float *rs, float *out, int64_t ldS,
                        cudaStream_t s) {
    constexpr int CHUNK = NT * Store<DT>::VEC;
    // room for twice the average run (it holds nearly every one of a uniform
    // hash); more would cost a resident CTA where the runs are short
    const int ncache = (int)std::min<int64_t>(kCsCacheMax, std::max<int64_t>(64, 2 * (int64_t)kCsGroup * T / m));
    const size_t smem = (size_t)kCsGroup * CHUNK * 4 + 4 * (size_t)ncache;
    MV_TRY(cs_smem_attr(cs_tn_kernel<DT, NT>, smem));
    dim3 grid((unsigned)((m + kCsGroup - 1) / kCsGroup), (unsigned)((n + CHUNK - 1) / CHUNK));
    MV_CUDA_TRY(cs_start(cs_tn_kernel<DT, NT>, grid, NT, smem, s, L, ld, n, m, w.off, w.list, rs, out, ldS,
                         ncache));
    return MV_OK;
}

template <int DT>
static int cs_launch(int layout, const void *L, int64_t ld, int n, int T, int m, const CsWs &w, const float *rs,
                     float *out, int64_t ldS, cudaStream_t s) {
    if (layout == MV_LAYOUT_TN) {
        // narrow CTAs where wide ones would not give every SM four
        constexpr int CHUNK = kCsThreads * Store<DT>::VEC;
        const int64_t wide = (int64_t)((m + kCsGroup - 1) / kCsGroup) * ((n + CHUNK - 1) / CHUNK);
        if (wide < 4 * 152) return cs_launch_tn<DT, kCsThreadsFew>(L, ld, n, T, m, w, rs, out, ldS, s);
        return cs_launch_tn<DT, kCsThreads>(L, ld, n, T, m, w, rs, out, ldS, s);
    } else {
        const size_t smem = ((size_t)T * dtype_size(DT) + 15) / 16 * 16;
        MV_TRY(cs_smem_attr(cs_nt_kernel<DT>, smem));
        cs_nt_kernel<DT><<<(unsigned)n, kCsNtThreads, smem, s>>>(L, ld, T, m, w.off, w.list, rs, out, ldS);
    }
    return MV_OK;
}

}  // namespace mv

using namespace mv;

extern "C" {

size_t mv_countsketch_workspace_size(int64_t T, int64_t m) {
    if (T < 1 || m < 1 || T >= (1LL << 31) || m >= (1LL << 30)) return 0;
    return cs_ws_bytes(T, m);
}

int mv_countsketch(const void *d_L, int32_t dtype, int32_t layout, const float *d_row_scale, int64_t n, int64_t T,
                   int64_t ldL, const int32_t *d_hash, const int8_t *d_sign, int64_t m, float *d_L_sketch,
                   int64_t ldS, void *d_ws, size_t ws_bytes, mv_stream_t stream) {
    if (d_L == nullptr || d_hash == nullptr || d_sign == nullptr || d_L_sketch == nullptr) return MV_ERR_INVALID_ARG;
    if (dtype != MV_F32 && dtype != MV_BF16 && dtype != MV_FP8_E4M3) return MV_ERR_INVALID_ARG;
    if (layout != MV_LAYOUT_NT && layout != MV_LAYOUT_TN) return MV_ERR_INVALID_ARG;
    if (n < 1 || T < 1 || m < 1 || ldS < m) return MV_ERR_INVALID_ARG;
    if (ldL < (layout == MV_LAYOUT_TN ? n : T)) return MV_ERR_INVALID_ARG;
    if (n >= (1LL << 31) || T >= (1LL << 31) || m >= (1LL << 30))
        return record_message(MV_ERR_UNSUPPORTED, "mv_countsketch: n and T must be below 2^31 and m below 2^30");
    const int es = dtype_size(dtype);
    if (((uintptr_t)d_L) % 16 != 0 || (ldL * es) % 16 != 0 || ((uintptr_t)d_L_sketch) % 16 != 0) return MV_ERR_INVALID_ARG;
    if (dtype == MV_FP8_E4M3 && d_row_scale == nullptr) return MV_ERR_INVALID_ARG;
    if (layout == MV_LAYOUT_NT && (size_t)T * es > kCsNtMaxRow)
        return record_message(MV_ERR_UNSUPPORTED, "countsketch: an n x T row above 200 KB does not fit shared memory; "
                                                  "store L transposed (MV_LAYOUT_TN)");
    const size_t need = cs_ws_bytes(T, m);
    if (d_ws == nullptr || ws_bytes < need || ((uintptr_t)d_ws) % 256 != 0) return MV_ERR_WORKSPACE;
    (void)cudaGetLastError();
    cudaStream_t s = (cudaStream_t)stream;
    CsWs w = cs_carve(d_ws, T, m);
    MV_CUDA_TRY(cudaMemsetAsync(w.cnt, 0, cs_zero_bytes(m), s));
    const int tb = (int)std::min<int64_t>((T + 255) / 256, 4096);
    const int per = T > (int64_t)kCsShort * m ? 1 : kWarp;       // buckets per warp of the sort
    const int sb = (int)std::min<int64_t>((m + per - 1) / per, 4096);
    MV_CUDA_TRY(cs_start(cs_count_kernel, dim3(tb), 256, 0, s, d_hash, (int)T, (int)m, w.cnt, w.err));
    MV_CUDA_TRY(cs_start(cs_scan_kernel, dim3(1), 1024, 0, s, w.cnt, (int)m, w.off));
    MV_CUDA_TRY(cs_start(cs_fill_kernel, dim3(tb), 256, 0, s, d_hash, d_sign, (int)T, (int)m, w.off, w.fill, w.list));
    MV_CUDA_TRY(cs_start(cs_sort_kernel, dim3(sb), kWarp, 0, s, w.off, (int)m, per, w.list, w.err));
    const float *rs = dtype == MV_FP8_E4M3 ? d_row_scale : nullptr;
    switch (dtype) {
        case MV_F32: MV_TRY(cs_launch<MV_F32>(layout, d_L, ldL, (int)n, (int)T, (int)m, w, rs, d_L_sketch, ldS, s)); break;
        case MV_BF16: MV_TRY(cs_launch<MV_BF16>(layout, d_L, ldL, (int)n, (int)T, (int)m, w, rs, d_L_sketch, ldS, s)); break;
        default: MV_TRY(cs_launch<MV_FP8_E4M3>(layout, d_L, ldL, (int)n, (int)T, (int)m, w, rs, d_L_sketch, ldS, s)); break;
    }
    MV_CUDA_TRY(cudaGetLastError());
    int err = 0;
    MV_CUDA_TRY(cudaMemcpyAsync(&err, w.err, sizeof(int), cudaMemcpyDeviceToHost, s));
    MV_CUDA_TRY(cudaStreamSynchronize(s));
    if (err == 1) return record_message(MV_ERR_INVALID_ARG, "countsketch: a bucket index lies outside [0, m)");
    if (err == 2) return record_message(MV_ERR_UNSUPPORTED, "countsketch: a bucket holds more than 4096 periods");
    return MV_OK;
}

}  // extern "C"
