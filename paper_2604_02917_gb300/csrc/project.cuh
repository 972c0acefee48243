// Cluster-cooperative exact projection onto F = {mu^T x >= R, 1^T x = 1, x >= 0}
// (Sec. 3.1, Eqs. simplex-tau, simplex-proj, projF-dualpath).
//
// Search (the same mathematics as the paper's scalar dual search):
//  * inner -- the simplex threshold at fixed nu: h(tau) = sum max(w - tau, 0) - 1
//    (w = v + nu mu) is convex, decreasing, piecewise linear.  A Newton step
//    from any tau lands at or left of the root, and from the left the
//    supports are nested, so the iteration ends exactly when |S| stops
//    changing: tau = (sum_S w - 1)/|S|.  It replaces the paper's sort.
//  * outer -- phi(nu) = mu^T x(nu) is continuous, nondecreasing, piecewise
//    linear.  On the support S at the current nu the budget and return rows
//        |S| tau - nu sum_S mu = sum_S v - 1
//        sum_S mu tau - nu sum_S mu^2 = sum_S mu v - R
//    give the exact (tau, nu) of that piece (a Newton step on phi).  A
//    bracket psi(lo) < 0 <= psi(hi), psi = phi - R, is kept; the paper's
//    geometric expansion nu = 1, 2, 4, ... and bisection take over when the
//    Newton point leaves it; the search stops when the support at nu
//    reproduces nu (exact finish).  psi(0) >= 0 means the return row is
//    inactive and the simplex projection is the answer.
//
// Arithmetic designed for GB300, whose FP64 rate is ~2 lane-ops/clk/SM:
//  * every step is one reduction of |S|, sum_S v, sum_S mu, sum_S mu v,
//    sum_S mu^2; the sums are EXACT integer additions of fixed-point images
//    of the FP64 values (62-bit magnitudes scaled by the largest element,
//    converted with integer bit operations, so each image carries the full
//    FP64 mantissa), so no FP64 add runs per element or in the reduction
//    tree and the sums are at least as accurate as FP64 ones.  An image is
//    three 21-bit limbs; a thread's and a warp's limb sums fit 32 bits (one
//    redux.sync each), a block's too, and only the cluster totals are
//    recombined;
//  * membership w_i > tau is decided in FP32 with a proven error margin;
//    only elements inside the margin repeat the test in FP64 (same result as
//    an FP64 evaluation of fma(nu, mu_i, v_i) > tau);
//  * the n elements are split over a cluster of CL thread blocks (one SM
//    each); block sums are exchanged through distributed shared memory and
//    added in rank order by every block, so all blocks hold bit-identical
//    sums and take identical decisions; the O(1) scalar FP64 logic runs on
//    one thread per block.
// The warm start (nu, tau of the previous call) only changes where the
// search begins, never the point it returns: the projection is unique.
// Warm-start shortcut: the support S0 at the hint gives, from the same
// reduction, the exact solution (nu*, tau*) of the budget and return rows on
// S0 (tau* alone at nu = 0 when the hint says the return row is inactive).
// A second, much lighter exchange only asks whether any element's membership
// at (nu*, tau*) differs from S0 (each thread kept its elements' bits); none
// means S0 is the support at (nu*, tau*), so (nu*, tau*) is exact and the
// search ends (the general search needs four reductions when the support
// does not move).  Otherwise the general search continues from (nu*, tau*).
// Scale hint: the fixed-point scales follow from the cluster maxima of four
// exponents, which would cost an exchange of their own before the first
// reduction.  A caller that projects similar points again and again (the
// solve loops) passes the exponents of its last projection: the images are
// made with those and the true maxima travel with the first reduction, which
// is repeated in the rare case that one of them moved.  The images, and so
// the results, are the same either way.
#pragma once

#include <cooperative_groups.h>

#include "mv_internal.cuh"

namespace mv {

namespace cg = cooperative_groups;

constexpr int kProjNT = 256;          // threads per block
constexpr int kProjMaxCL = 16;        // largest cluster
constexpr int kProjMaxLocal = 2048;   // elements per block (n <= 16 * 2048)
constexpr int kProjMaxN = kProjMaxCL * kProjMaxLocal;
constexpr int kFixBits = 62;          // fixed-point magnitude bound 2^62 (sums kept in 128 bits)

// round(d * 2^s) with integer operations only; |d| 2^s must stay below 2^62.
__device__ __forceinline__ long long to_fixed(double d, int s) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return 0;                                    // zero or subnormal
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = e - 1075 + s;
    long long r;
    if (sh >= 0) {
        r = (long long)(m << (sh > 9 ? 9 : sh));
    } else if (sh > -64) {
        r = (long long)((m + (1ull << (-sh - 1))) >> (-sh));
    } else {
        r = 0;
    }
    return (b >> 63) ? -r : r;
}

// Biased exponent field of |d| (0 for zero).
__device__ __forceinline__ int exp_field(double d) {
    return (int)(((unsigned long long)__double_as_longlong(d) >> 52) & 0x7ff);
}

// 2^-s as an exact double (0 below the normal range).
__device__ __forceinline__ double pow2_neg(int s) {
    const int e = 1023 - s;
    if (e <= 0) return 0.0;
    if (e >= 2047) return INFINITY;
    return __longlong_as_double((long long)e << 52);
}

// Scale s such that every |q| whose exponent field is <= e satisfies |q| 2^s < 2^kFixBits.
__host__ __device__ __forceinline__ int fixed_scale(int e) { return e == 0 ? 0 : kFixBits + 1022 - e; }

// Warp-wide sum and maximum of a 32-bit integer (one instruction).
__device__ __forceinline__ int redux_add(int v) { return __reduce_add_sync(0xffffffffu, v); }
__device__ __forceinline__ int redux_max(int v) { return __reduce_max_sync(0xffffffffu, v); }
// Adds the three 21-bit limbs of a fixed-point image (|x| < 2^62: the top
// limb, arithmetic, lies in [-2^20, 2^20)) to per-thread 32-bit sums.  Eight
// elements per thread (kProjMaxLocal) and 32 lanes stay below 2^29, a block
// of kProjMaxLocal below 2^32 (the top limb within int32).
__device__ __forceinline__ void add_limbs(int (&l)[3], long long x) {
    l[0] += (int)x & 0x1fffff;
    l[1] += (int)(x >> 21) & 0x1fffff;
    l[2] += (int)(x >> 42);
}
// The value of cluster-wide limb totals (l0, l1 < 2^36; |l2| < 2^35): the
// 128-bit sum as its high and low halves, each rounded to FP64.
__device__ __forceinline__ double from_limbs(long long l0, long long l1, long long l2) {
    const unsigned long long m = (unsigned long long)((l1 << 21) + l0);
    const unsigned long long lo = m + ((unsigned long long)l2 << 42);
    const long long hi = (l2 >> 22) + (lo < m ? 1 : 0);
    return (double)hi * 18446744073709551616.0 + (double)lo;
}

// Cluster totals of one support step, as thread 0 of every block holds them.
struct SupportSums {
    double cnt, sv, sm, smv, smm;
    int nan;
};

// Exponent fields of the last projection's scales (v, mu, mu v, mu^2); e[0] < 0: none.
struct ScaleHint {
    int e[4];
};

// Words a block contributes to a reduction: 0 |S|, 1 + 3q + l limb l of
// image q (v, mu, mu v, mu^2), 13 NaNs met, 14 and 15 the largest exponent
// fields of v and mu v (maxima, not sums).
constexpr int kProjWords = 16;
constexpr int kProjNW = kProjNT / kWarp;

struct ProjOut {
    double nu, tau;
    int status;
    int steps;
    int dykstra;      // 1 if the Dykstra safeguard ran
};

// Shared-memory workspace of one block of the projector.
struct ProjSmem {
    alignas(16) int part[2][kProjMaxCL][kProjWords];   // DSMEM slots: [parity][source rank][word]
    alignas(16) int wred[kProjNW][kProjWords];         // per-warp words
    alignas(16) int moved[kProjMaxCL];                 // verifying exchange: source rank's membership changes
    double dpart[2][kProjMaxCL];
    int emax[kProjMaxCL][4];
    double wredd[kProjNW], wredm[kProjNW];
    int wmax[kProjNW][4];
    // broadcast of the scalar state (written by warp 0)
    double nu, tau, dbcast, dmin, dmax;
    double mpart[2][kProjMaxCL][2];
    float nu32, tau32;
    int verify, redo;
    int done, status, steps;
    int e[4];                           // exponent fields the scales follow from
    double p_v, p_m, p_mv, p_mm;        // 2^-s of the four scales
    int parity;
};

// Must run once per block before the first reduction (all threads).
__device__ inline void proj_smem_init(ProjSmem *sh) {
    if (threadIdx.x == 0) {
        sh->parity = 0;
        sh->verify = 0;
        sh->redo = 0;
    }
    __syncthreads();
}

// Per-element arrays of the block's slice, in shared memory.
struct ProjElems {
    double *v, *mu;               // FP64 values
    float *v32, *mu32;            // FP32 images for screening
    long long *V, *M, *MV, *MM;   // fixed-point images
    int n;                        // elements in this block's slice
};

__host__ __device__ inline size_t proj_elem_bytes(int n_local) {
    return (size_t)n_local * (8 + 8 + 4 + 4 + 8 * 4) + 64;
}

__device__ inline ProjElems carve_elems(void *base, int n_local) {
    ProjElems e;
    char *p = reinterpret_cast<char *>(base);
    e.v = reinterpret_cast<double *>(p);
    p += 8 * (size_t)n_local;
    e.mu = reinterpret_cast<double *>(p);
    p += 8 * (size_t)n_local;
    e.V = reinterpret_cast<long long *>(p);
    p += 8 * (size_t)n_local;
    e.M = reinterpret_cast<long long *>(p);
    p += 8 * (size_t)n_local;
    e.MV = reinterpret_cast<long long *>(p);
    p += 8 * (size_t)n_local;
    e.MM = reinterpret_cast<long long *>(p);
    p += 8 * (size_t)n_local;
    e.v32 = reinterpret_cast<float *>(p);
    p += 4 * (size_t)n_local;
    e.mu32 = reinterpret_cast<float *>(p);
    e.n = n_local;
    return e;
}

__device__ __forceinline__ int warp_max_i(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

template <int CL>
__device__ __forceinline__ void cluster_barrier() {
    if constexpr (CL > 1) {
        cg::this_cluster().sync();
    } else {
        __syncthreads();
    }
}

// The same barrier in two halves, for work between them.  Every kernel that
// exchanges has one before its first exchange (arrive on entry, wait behind
// the loads): a peer's shared memory may only be written once the peer runs.
template <int CL>
__device__ __forceinline__ void cluster_arrive() {
    if constexpr (CL > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
template <int CL>
__device__ __forceinline__ void cluster_wait() {
    if constexpr (CL > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int CL>
__device__ __forceinline__ int cluster_rank() {
    if constexpr (CL > 1) {
        return (int)cg::this_cluster().block_rank();
    } else {
        return 0;
    }
}

template <int CL>
struct ClusterProj {
    ProjSmem *sh;
    ProjElems el;
    // Dykstra safeguard: 4 el.n doubles of global scratch for this block
    // (v, x, p, q) and the sweep budget; without scratch the safeguard is off.
    double *dyk = nullptr;
    int dyk_iters = 0;
    // Per thread: membership bits of its elements at the last reduction's
    // point, and, while the scales rest on a hint, its largest exponent
    // fields of v and mu v.
    unsigned in_bits = 0;
    int my_ev = 0, my_emv = 0;
    bool hinted = false;

    // Block-then-cluster total of the per-warp words in sh->wred (after a
    // __syncthreads): lane k of warp 0 of every block ends with the total of
    // word k mod 16 (integer sums and maxima: exact, so the order does not
    // matter).  Two lanes share a word, each taking half of the warps and
    // half of the ranks; the words go out as 16-byte pieces, two per lane.
    __device__ long long reduce_partials() {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int par = sh->parity;
        const int word = lane & (kProjWords - 1), half = lane / kProjWords;
        const bool is_max = word >= 14;
        auto join = [&](long long a, long long b) { return is_max ? (a > b ? a : b) : a + b; };
        long long t = 0;
        if (warp == 0) {
#pragma unroll
            for (int w = 0; w < kProjNW / 2; ++w) t = join(t, (long long)sh->wred[half * (kProjNW / 2) + w][word]);
            t = join(t, __shfl_xor_sync(0xffffffffu, t, kProjWords));
            if (lane == 0) sh->parity = par ^ 1;
        }
        // One block: no barrier here.  Warp 0's reads of wred come before the
        // block barrier that follows in every caller, and so before the next
        // reduction's writes.
        if constexpr (CL > 1) {
            if (warp == 0) {
                const int me = cluster_rank<CL>();
                if (lane < kProjWords) sh->part[par][me][word] = (int)(unsigned)t;   // limbs 0, 1 as unsigned
                __syncwarp();
                cg::cluster_group cl = cg::this_cluster();
                int4 *src = reinterpret_cast<int4 *>(&sh->part[par][me][0]);
                for (int p = lane; p < CL * (kProjWords / 4); p += kWarp) {
                    const int r = p / (kProjWords / 4), q = p % (kProjWords / 4);
                    if (r != me) *cl.map_shared_rank(src + q, r) = src[q];
                }
            }
            cluster_barrier<CL>();
            t = 0;
            if (warp == 0) {
                // limbs 0 and 1 of an image are unsigned block totals, every other word is signed
                const bool uns = word >= 1 && word <= 12 && (word - 1) % 3 != 2;
#pragma unroll
                for (int r = 0; r < CL / 2; ++r) {
                    const int x = sh->part[par][half * (CL / 2) + r][word];
                    t = join(t, uns ? (long long)(unsigned)x : (long long)x);
                }
                t = join(t, __shfl_xor_sync(0xffffffffu, t, kProjWords));
            }
            // The next exchange writes the other parity; the one after reuses this
            // one only after another cluster barrier, so no reader is overtaken.
        }
        return t;
    }

    // Whether any thread of the cluster passes a nonzero x; one barrier.
    // Its slots are rewritten only by the next call, with at least one full
    // reduction (a cluster barrier) between two calls.
    __device__ bool any_of(int x) {
        if constexpr (CL == 1) {
            return __syncthreads_or(x) != 0;
        } else {
            const int any = __syncthreads_or(x);
            if (threadIdx.x < CL)
                *cg::this_cluster().map_shared_rank(&sh->moved[cluster_rank<CL>()], (int)threadIdx.x) = any;
            cluster_barrier<CL>();
            int t = 0;
#pragma unroll
            for (int r = 0; r < CL; ++r) t |= sh->moved[r];
            return t != 0;
        }
    }

    // Cluster sum of one double per thread, added in a fixed order (every
    // block gets the same value); result returned to all threads.
    __device__ double reduce_double(double x) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        x = warp_sum(x);
        if (lane == 0) sh->wredd[warp] = x;
        __syncthreads();
        const int par = sh->parity;
        if (warp == 0) {
            double t = lane < kProjNW ? sh->wredd[lane] : 0.0;
#pragma unroll
            for (int o = kProjNW / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            t = __shfl_sync(0xffffffffu, t, 0);
            if (lane < CL) {
                double *dst = &sh->dpart[par][cluster_rank<CL>()];
                if constexpr (CL > 1) dst = cg::this_cluster().map_shared_rank(dst, lane);
                *dst = t;
            }
        }
        cluster_barrier<CL>();
        if (warp == 0) {
            double t = lane < CL ? sh->dpart[par][lane] : 0.0;
#pragma unroll
            for (int o = CL / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) {
                sh->dbcast = t;
                sh->parity = par ^ 1;
            }
        }
        __syncthreads();
        const double r = sh->dbcast;
        __syncthreads();
        return r;
    }

    // Cluster-wide min and max of one double per thread; result to all threads.
    __device__ void reduce_minmax(double &mn, double &mx) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        mn = warp_min(mn);
        mx = warp_max(mx);
        if (lane == 0) {
            sh->wredd[warp] = mn;
            sh->wredm[warp] = mx;
        }
        __syncthreads();
        const int par = sh->parity;
        if (threadIdx.x == 0) {
            double a = INFINITY, b = -INFINITY;
            for (int w = 0; w < kProjNW; ++w) {
                a = fmin(a, sh->wredd[w]);
                b = fmax(b, sh->wredm[w]);
            }
            const int me = cluster_rank<CL>();
            if constexpr (CL > 1) {
                cg::cluster_group cl = cg::this_cluster();
                for (int r = 0; r < CL; ++r) {
                    double *dst = cl.map_shared_rank(&sh->mpart[par][me][0], r);
                    dst[0] = a;
                    dst[1] = b;
                }
            } else {
                sh->mpart[par][0][0] = a;
                sh->mpart[par][0][1] = b;
            }
        }
        cluster_barrier<CL>();
        if (threadIdx.x == 0) {
            double a = INFINITY, b = -INFINITY;
            for (int r = 0; r < CL; ++r) {
                a = fmin(a, sh->mpart[par][r][0]);
                b = fmax(b, sh->mpart[par][r][1]);
            }
            sh->dmin = a;
            sh->dmax = b;
            sh->parity = par ^ 1;
        }
        __syncthreads();
        mn = sh->dmin;
        mx = sh->dmax;
        __syncthreads();
    }

    // The scales of the exponent fields sh->e (thread 0), for the conversions
    // of the totals.
    __device__ void set_scales() {
        sh->p_v = pow2_neg(fixed_scale(sh->e[0]));
        sh->p_m = pow2_neg(fixed_scale(sh->e[1]));
        sh->p_mv = pow2_neg(fixed_scale(sh->e[2]));
        sh->p_mm = pow2_neg(fixed_scale(sh->e[3]));
    }

    // prepare() on the scales of `hint` (none: the plain form).  The largest
    // exponent fields this thread meets go into the first reduction.
    __device__ void prepare(const ScaleHint &hint) {
        if (hint.e[0] < 0) {
            prepare();
            return;
        }
        const int s0 = fixed_scale(hint.e[0]), s1 = fixed_scale(hint.e[1]), s2 = fixed_scale(hint.e[2]),
                  s3 = fixed_scale(hint.e[3]);
        my_ev = my_emv = 0;
        for (int i = threadIdx.x; i < el.n; i += kProjNT) {
            const double v = el.v[i], m = el.mu[i];
            const double mv = m * v;
            my_ev = max(my_ev, exp_field(v));
            my_emv = max(my_emv, exp_field(mv));
            el.V[i] = to_fixed(v, s0);
            el.M[i] = to_fixed(m, s1);
            el.MV[i] = to_fixed(mv, s2);
            el.MM[i] = to_fixed(m * m, s3);
            el.v32[i] = (float)v;
            el.mu32[i] = (float)m;
        }
        hinted = true;
        if (threadIdx.x == 0) {
#pragma unroll
            for (int k = 0; k < 4; ++k) sh->e[k] = hint.e[k];
            set_scales();
        }
    }
    // Images of v and mu v again, on the scales of sh->e (a hint that did not hold).
    __device__ void rescale() {
        const int s0 = fixed_scale(sh->e[0]), s2 = fixed_scale(sh->e[2]);
        for (int i = threadIdx.x; i < el.n; i += kProjNT) {
            el.V[i] = to_fixed(el.v[i], s0);
            el.MV[i] = to_fixed(el.mu[i] * el.v[i], s2);
        }
    }
    // The exponent fields behind the present scales.
    __device__ ScaleHint scales() const {
        ScaleHint h;
#pragma unroll
        for (int k = 0; k < 4; ++k) h.e[k] = sh->e[k];
        return h;
    }

    // Cluster-wide maxima of the exponent fields of |v|, |mu|, |mu v|, mu^2,
    // then the fixed-point images of the slice.  Expects el.v and el.mu set.
    __device__ void prepare() {
        int e[4] = {0, 0, 0, 0};
        for (int i = threadIdx.x; i < el.n; i += kProjNT) {
            const double v = el.v[i], m = el.mu[i];
            const double mv = m * v, mm = m * m;
            e[0] = max(e[0], exp_field(v));
            e[1] = max(e[1], exp_field(m));
            e[2] = max(e[2], exp_field(mv));
            e[3] = max(e[3], exp_field(mm));
            el.MV[i] = __double_as_longlong(mv);   // converted in place below
            el.MM[i] = __double_as_longlong(mm);
            el.v32[i] = (float)v;
            el.mu32[i] = (float)m;
        }
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < 4; ++k) e[k] = warp_max_i(e[k]);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < 4; ++k) sh->wmax[warp][k] = e[k];
        __syncthreads();
        if (threadIdx.x == 0) {
            int t[4] = {0, 0, 0, 0};
            for (int w = 0; w < kProjNT / kWarp; ++w)
#pragma unroll
                for (int k = 0; k < 4; ++k) t[k] = max(t[k], sh->wmax[w][k]);
            const int me = cluster_rank<CL>();
            if constexpr (CL > 1) {
                cg::cluster_group cl = cg::this_cluster();
                for (int r = 0; r < CL; ++r) {
                    int *dst = cl.map_shared_rank(&sh->emax[me][0], r);
#pragma unroll
                    for (int k = 0; k < 4; ++k) dst[k] = t[k];
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) sh->emax[0][k] = t[k];
            }
        }
        cluster_barrier<CL>();
        if (threadIdx.x == 0) {
            int t[4] = {0, 0, 0, 0};
            for (int r = 0; r < CL; ++r)
#pragma unroll
                for (int k = 0; k < 4; ++k) t[k] = max(t[k], sh->emax[r][k]);
#pragma unroll
            for (int k = 0; k < 4; ++k) sh->e[k] = t[k];
            set_scales();
        }
        __syncthreads();
        hinted = false;
        const int sv = fixed_scale(sh->e[0]), sm = fixed_scale(sh->e[1]), smv = fixed_scale(sh->e[2]),
                  smm = fixed_scale(sh->e[3]);
        for (int i = threadIdx.x; i < el.n; i += kProjNT) {
            el.V[i] = to_fixed(el.v[i], sv);
            el.M[i] = to_fixed(el.mu[i], sm);
            el.MV[i] = to_fixed(__longlong_as_double(el.MV[i]), smv);
            el.MM[i] = to_fixed(__longlong_as_double(el.MM[i]), smm);
        }
        // emax slots are rewritten only by the next prepare(), after at least
        // one more cluster barrier.
        __syncthreads();
    }

    // i in S(nu, tau), i.e. fma(nu, mu_i, v_i) > tau in FP64, screened in FP32
    // with a proven margin (the FP64 test runs only inside it).
    __device__ __forceinline__ bool member(int i, double nu, double tau, float nu32, float tau32, float anu,
                                           float atau, bool &nan) const {
        const float c = 2.384185791015625e-07f;   // 2^-22
        const float v32 = el.v32[i], m32 = el.mu32[i];
        const float d = fmaf(nu32, m32, v32) - tau32;
        const float margin = c * (fmaf(anu, fabsf(m32), fabsf(v32)) + atau);
        if (d > margin) return true;
        if (d < -margin) return false;
        const double w = fma(nu, el.mu[i], el.v[i]);
        if (!(w == w)) nan = true;
        return w > tau;
    }

    // Sums over S = {i : fma(nu, mu_i, v_i) > tau}; totals valid in warp 0
    // (all lanes).  Leaves the thread's membership bits in in_bits.
    __device__ SupportSums support_sums(double nu, double tau, float nu32, float tau32) {
        while (true) {
            int lb[4][3];
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int q = 0; q < 3; ++q) lb[k][q] = 0;
            const float anu = fabsf(nu32), atau = isinf(tau32) ? 0.f : fabsf(tau32);
            bool nan = false;
            in_bits = 0;
            unsigned bit = 1;
            for (int i = threadIdx.x; i < el.n; i += kProjNT, bit <<= 1) {
                if (member(i, nu, tau, nu32, tau32, anu, atau, nan)) {
                    in_bits |= bit;
                    add_limbs(lb[0], el.V[i]);
                    add_limbs(lb[1], el.M[i]);
                    add_limbs(lb[2], el.MV[i]);
                    add_limbs(lb[3], el.MM[i]);
                }
            }
            const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
            __syncwarp();
            // |S| and the NaN count share a word: at most 256 of each per warp
            const int cn = redux_add(__popc(in_bits) + (nan ? 1 << 16 : 0));
            int mine = lane == 0 ? (cn & 0xffff) : (lane == 13 ? cn >> 16 : 0);
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    const int t = redux_add(lb[k][q]);
                    mine = lane == 1 + 3 * k + q ? t : mine;
                }
            if (hinted) {
                const int a = redux_max(my_ev), b = redux_max(my_emv);
                mine = lane == 14 ? a : (lane == 15 ? b : mine);
            }
            if (lane < kProjWords) sh->wred[warp][lane] = mine;
            __syncthreads();
            const long long t = reduce_partials();
            if (hinted) {
                hinted = false;
                if (warp == 0) {
                    const bool moved = (lane == 14 && t != sh->e[0]) || (lane == 15 && t != sh->e[2]);
                    const bool redo = __any_sync(0xffffffffu, moved);
                    const int ev = (int)__shfl_sync(0xffffffffu, t, 14), emv = (int)__shfl_sync(0xffffffffu, t, 15);
                    if (lane == 0) {
                        sh->redo = redo;
                        if (redo) {
                            sh->e[0] = ev;
                            sh->e[2] = emv;
                            set_scales();
                        }
                    }
                }
                __syncthreads();
                if (sh->redo) {
                    rescale();
                    continue;
                }
            }
            // lane k < 5 converts total k to FP64 (the four images with their scales)
            SupportSums out{};
            if (warp == 0) {
                const int base = lane >= 1 && lane < 5 ? 1 + 3 * (lane - 1) : 1;
                const long long l0 = __shfl_sync(0xffffffffu, t, base), l1 = __shfl_sync(0xffffffffu, t, base + 1),
                                l2 = __shfl_sync(0xffffffffu, t, base + 2);
                const double p = lane == 1 ? sh->p_v : (lane == 2 ? sh->p_m : (lane == 3 ? sh->p_mv : sh->p_mm));
                const double d = lane == 0 ? (double)t : from_limbs(l0, l1, l2) * p;
                out.cnt = __shfl_sync(0xffffffffu, d, 0);
                out.sv = __shfl_sync(0xffffffffu, d, 1);
                out.sm = __shfl_sync(0xffffffffu, d, 2);
                out.smv = __shfl_sync(0xffffffffu, d, 3);
                out.smm = __shfl_sync(0xffffffffu, d, 4);
                out.nan = (int)__shfl_sync(0xffffffffu, t, 13);
            }
            return out;
        }
    }

    // Whether the support at (nu, tau) is the one of the last reduction.
    __device__ bool same_support(double nu, double tau, float nu32, float tau32) {
        const float anu = fabsf(nu32), atau = isinf(tau32) ? 0.f : fabsf(tau32);
        bool nan = false;
        unsigned now = 0, bit = 1;
        for (int i = threadIdx.x; i < el.n; i += kProjNT, bit <<= 1)
            if (member(i, nu, tau, nu32, tau32, anu, atau, nan)) now |= bit;
        return !any_of(now != in_bits);
    }

    // Full search.  Returns (nu, tau, status) identically in all threads.
    // The scalar logic runs on warp 0 (every lane the same); `side` is run
    // meanwhile by the last warp, once.
    template <typename Side>
    __device__ ProjOut search(double R, int mode, double mu_min, double mu_max, double nu_hint, double tau_hint,
                             int budget, const Side &side) {
        // Search state of warp 0.
        double lo = -INFINITY, hi = INFINITY, nu = 0.0, tau = -INFINITY, prev_cnt = -1.0;
        bool have_lo = false, have_hi = false, zero_done = false, first = true;
        bool try_fast = true, refuted = false, side_done = false;
        int outer = 0, inner = 0, status = MV_OK;
        const bool ge = (mode == MV_RETURN_GE);
        if (threadIdx.x < kWarp) {
            const bool infeasible = !(R <= mu_max) || (!ge && !(R >= mu_min));
            if (!infeasible) {
                nu = (nu_hint == nu_hint) ? nu_hint : 0.0;
                if (ge && !(nu > 0.0)) nu = 0.0;
                tau = (tau_hint == tau_hint) ? tau_hint : -INFINITY;
            }
            if (threadIdx.x == 0) {
                sh->steps = 0;
                sh->verify = 0;
                sh->done = infeasible ? 1 : 0;
                sh->status = infeasible ? MV_ERR_INFEASIBLE : MV_OK;
                sh->nu = infeasible ? NAN : nu;
                sh->tau = infeasible ? NAN : tau;
                sh->nu32 = (float)nu;
                sh->tau32 = (float)tau;
            }
        }
        __syncthreads();
        double scaleR = 0.0;
        if (threadIdx.x < kWarp) scaleR = fmax(fabs(R), fmax(fabs(mu_max), fabs(mu_min)));
        while (true) {
            if (sh->done) break;                       // uniform: read after a barrier
            const double enu = sh->nu, etau = sh->tau;
            const float enu32 = sh->nu32, etau32 = sh->tau32;
            if (sh->verify) {
                // a candidate built on the support of the last reduction: exact iff the support is the same there
                const bool same = same_support(enu, etau, enu32, etau32);
                if (same) {
                    if (threadIdx.x == 0) sh->steps += 1;
                    break;                             // (nu, tau) and MV_OK stand in sh
                }
                refuted = true;
            }
            const SupportSums S = support_sums(enu, etau, enu32, etau32);
            if (!side_done && threadIdx.x >= kProjNT - kWarp) side();
            side_done = true;
            if (threadIdx.x < kWarp) {
                const double cnt = S.cnt, sv = S.sv, sm = S.sm, smv = S.smv, smm = S.smm;
                bool finish = false, handled = false, verify = false;
                double next_nu = enu, next_tau = etau;
                if (S.nan != 0) {
                    status = MV_ERR_NUMERIC;
                    finish = true;
                    handled = true;
                } else if (refuted) {
                    refuted = false;                   // the general search goes on from the candidate
                } else if (try_fast && cnt > 0.0) {
                    try_fast = false;
                    const double a = cnt, b = sm, c = smm;
                    double nc = NAN, tc = NAN;
                    bool ok = false;
                    if (ge && enu == 0.0) {            // hint: return row inactive; simplex threshold on S0
                        tc = (sv - 1.0) / a;
                        nc = 0.0;
                        ok = (smv - tc * b) - R >= 0.0;
                    } else {
                        const double det = a * c - b * b;
                        if (det > 1e-13 * a * c) {
                            // the two divisions as one: lane 0 the multiplier, the others 1/|S|, from which
                            // two corrections give the threshold's correctly rounded quotient (Markstein:
                            // with r = RN(1/a) and q within an ulp, q + (t - q a) r rounds to RN(t / a))
                            const double num = b * (sv - 1.0) - a * (smv - R);
                            const bool l0 = threadIdx.x == 0;
                            const double q = (l0 ? num : 1.0) / (l0 ? det : a);
                            nc = __shfl_sync(0xffffffffu, q, 0);
                            const double ra = __shfl_sync(0xffffffffu, q, 1);
                            const double t = fma(nc, b, sv) - 1.0, t0 = t * ra;
                            const double t1 = fma(fma(-t0, a, t), ra, t0);
                            tc = fma(fma(-t1, a, t), ra, t1);
                            ok = !ge || nc >= 0.0;
                        }
                    }
                    if (ok && nc == nc && tc == tc && isfinite(nc) && isfinite(tc)) {
                        verify = true;
                        next_nu = nc;
                        next_tau = tc;
                        handled = true;
                    }
                }
                if (handled) {
                    // decided above
                } else if (cnt == 0.0) {               // tau >= max w: restart from the left
                    next_tau = -INFINITY;
                    first = true;
                    if (++inner > 96) {
                        status = MV_ERR_NOT_CONVERGED;
                        finish = true;
                    }
                } else if (first || cnt != prev_cnt) {  // inner Newton step
                    first = false;
                    prev_cnt = cnt;
                    next_tau = (fma(enu, sm, sv) - 1.0) / cnt;
                    if (++inner > 96) {
                        status = MV_ERR_NOT_CONVERGED;
                        finish = true;
                    }
                } else {
                    // inner converged: etau is the threshold at enu, S its support
                    inner = 0;
                    nu = enu;
                    tau = etau;
                    if (nu == 0.0) zero_done = true;
                    const double a = cnt, b = sm, c = smm;
                    const double det = a * c - b * b;
                    const bool flat = !(det > 1e-13 * a * c);
                    const double psi = flat ? (b / a - R) : ((fma(nu, c, smv) - tau * b) - R);
                    double nu_c = NAN;
                    if (ge && nu == 0.0 && psi >= 0.0) {
                        finish = true;                 // return row inactive
                    } else if (psi == 0.0) {
                        finish = true;
                    } else if (flat && fabs(psi) <= 1e-12 * scaleR) {
                        finish = true;                 // target met on a flat piece
                    } else {
                        if (!flat) {
                            nu_c = (b * (sv - 1.0) - a * (smv - R)) / det;
                            if (fabs(nu_c - nu) <= 1e-13 * fmax(1.0, fabs(nu))) finish = true;   // exact finish
                        }
                        if (!finish) {
                            if (psi < 0.0) {
                                lo = nu;
                                have_lo = true;
                            } else {
                                hi = nu;
                                have_hi = true;
                            }
                            double nxt = nu_c;
                            if (ge && nxt == nxt && nxt <= 0.0 && !zero_done) nxt = 0.0;
                            const bool inside = (nxt == nxt) && (!have_lo || nxt > lo) && (!have_hi || nxt < hi) &&
                                                (!ge || nxt >= 0.0);
                            if (!inside) {
                                if (have_lo && have_hi) {
                                    nxt = 0.5 * (lo + hi);
                                } else if (have_lo) {          // expand right: 1, 2, 4, ...
                                    nxt = (lo < 0.0) ? 0.0 : (lo == 0.0 ? 1.0 : 2.0 * lo);
                                    if (nxt == 0.0 && zero_done) nxt = 1.0;
                                } else if (ge) {
                                    nxt = 0.0;
                                } else {                       // expand left (equality mode)
                                    nxt = (hi > 0.0) ? 0.0 : (hi == 0.0 ? -1.0 : 2.0 * hi);
                                    if (nxt == 0.0 && zero_done) nxt = -1.0;
                                }
                            }
                            if (nxt == nu || ++outer >= budget) {
                                status = MV_ERR_NOT_CONVERGED;
                                finish = true;
                            } else {
                                next_nu = nxt;
                                next_tau = (fma(nxt, b, sv) - 1.0) / a;   // threshold this support predicts
                                first = true;
                            }
                        }
                    }
                }
                if (threadIdx.x == 0) {
                    sh->steps += 1;
                    sh->verify = verify ? 1 : 0;
                    if (finish) {
                        sh->done = 1;
                        sh->status = status;
                        sh->nu = nu;
                        sh->tau = tau;
                        if (status == MV_ERR_NUMERIC || (status == MV_ERR_NOT_CONVERGED && !(tau == tau))) {
                            sh->nu = enu;
                            sh->tau = etau;
                        }
                    } else {
                        sh->nu = next_nu;
                        sh->tau = next_tau;
                        sh->nu32 = (float)next_nu;
                        sh->tau32 = (float)next_tau;
                    }
                }
            }
            __syncthreads();
        }
        if (!side_done && threadIdx.x >= kProjNT - kWarp) side();   // infeasible: no reduction ran
        __syncthreads();
        ProjOut o;
        o.nu = sh->nu;
        o.tau = sh->tau;
        o.status = sh->status;
        o.steps = sh->steps;
        o.dykstra = 0;
        __syncthreads();   // all threads read the result before the slots are reused
        return o;
    }

    __device__ ProjOut search(double R, int mode, double mu_min, double mu_max, double nu_hint, double tau_hint,
                             int budget) {
        return search(R, mode, mu_min, mu_max, nu_hint, tau_hint, budget, [] {});
    }

    // Dykstra's alternating projections between Delta and H (the safeguard
    // of Sec. 3.1), started at the v held in el.v: x = v, p = q = 0, then
    //   y = Pi_Delta(x + p), p <- x + p - y;  w = y + q,
    //   x = w + theta mu (theta = max(0, (R - mu^T w) / ||mu||^2), any sign
    //   in equality mode), q <- w - x = -theta mu,
    // until x and y agree and stop moving (1e-10 max(1, |v|_inf)) or the
    // sweep budget is spent.  Pi_Delta is the scalar search at nu = 0 with
    // the return row dropped (R = -inf).  Returns theta, the return-row
    // multiplier of the limit, and in tau_out the threshold it implies
    // (tau = v_i + theta mu_i - x_i on the support, averaged); el.v and its
    // fixed-point images are restored.
    __device__ double dykstra(double R, int mode, double mu_min, double mu_max, int budget, int &sweeps,
                              double &tau_out) {
        const int n = el.n;
        double *v0 = dyk, *x = dyk + n, *p = dyk + 2 * n, *q = dyk + 3 * n;
        double vmax = 0.0, mm = 0.0;
        for (int i = threadIdx.x; i < n; i += kProjNT) {
            const double v = el.v[i];
            v0[i] = v;
            x[i] = v;
            p[i] = 0.0;
            q[i] = 0.0;
            vmax = fmax(vmax, fabs(v));
            mm = fma(el.mu[i], el.mu[i], mm);
        }
        mm = reduce_double(mm);
        double lo = 0.0, hi = vmax;
        reduce_minmax(lo, hi);
        const double tol = 1e-10 * fmax(1.0, hi);
        double theta = 0.0;
        sweeps = 0;
        for (int it = 0; it < dyk_iters; ++it) {
            for (int i = threadIdx.x; i < n; i += kProjNT) el.v[i] = x[i] + p[i];
            __syncthreads();
            prepare();
            const ProjOut s = search(-INFINITY, MV_RETURN_GE, mu_min, mu_max, 0.0, -INFINITY, budget);
            // el.v holds x + p: y = Pi_Delta(x + p), p <- x + p - y, w = y + q (parked in q)
            double c = 0.0;
            for (int i = threadIdx.x; i < n; i += kProjNT) {
                const double y = fmax(el.v[i] - s.tau, 0.0);
                p[i] = el.v[i] - y;
                const double w = y + q[i];
                q[i] = w;
                c = fma(el.mu[i], w, c);
            }
            c = reduce_double(c);
            double th = mm > 0.0 ? (R - c) / mm : 0.0;
            if (mode == MV_RETURN_GE) th = fmax(th, 0.0);
            // x <- w + theta mu, q <- w - x; measure |x_new - x_old| and |x_new - y|
            double dev = 0.0;
            for (int i = threadIdx.x; i < n; i += kProjNT) {
                const double w = q[i];
                const double y = fmax(el.v[i] - s.tau, 0.0);
                const double xn = fma(th, el.mu[i], w);
                dev = fmax(dev, fmax(fabs(xn - x[i]), fabs(xn - y)));
                x[i] = xn;
                q[i] = w - xn;
            }
            double a = -dev, b = fabs(th - theta) * sqrt(mm);
            reduce_minmax(a, b);
            theta = th;
            sweeps = it + 1;
            if (s.status != MV_OK) break;
            if (-a <= tol && b <= tol) break;
        }
        double st = 0.0, sc = 0.0;
        for (int i = threadIdx.x; i < n; i += kProjNT) {
            el.v[i] = v0[i];
            if (x[i] > 0.0) {
                st += fma(theta, el.mu[i], v0[i]) - x[i];
                sc += 1.0;
            }
        }
        st = reduce_double(st);
        sc = reduce_double(sc);
        tau_out = sc > 0.0 ? st / sc : -INFINITY;
        prepare();
        return theta;
    }

    // The projection: the scalar search, and the Dykstra safeguard when the
    // search does not finish within its budget (scratch permitting), whose
    // (theta, tau) restarts the exact search, with at least 100 outer steps.
    // `side` runs on the last warp beside the first reduction's scalar logic;
    // what it leaves in shared memory is visible on return.
    template <typename Side>
    __device__ ProjOut solve(double R, int mode, double mu_min, double mu_max, double nu_hint, double tau_hint,
                             int budget, const Side &side) {
        ProjOut o = search(R, mode, mu_min, mu_max, nu_hint, tau_hint, budget, side);
        if (o.status != MV_ERR_NOT_CONVERGED || dyk == nullptr || dyk_iters <= 0) return o;
        ClusterProj safe = *this;              // a copy, so that this one stays in registers
        return safeguarded(safe, o.steps, R, mode, mu_min, mu_max, budget);
    }
    // The safeguard and the search restarted from it.  Out of line: it runs
    // almost never, and the instructions of a projection that does not need
    // it should lie together (a step executes them once per launch).
    __device__ __noinline__ static ProjOut safeguarded(ClusterProj &P, int steps, double R, int mode, double mu_min,
                                                       double mu_max, int budget) {
        int sweeps = 0;
        double tau_d = -INFINITY;
        const double theta = P.dykstra(R, mode, mu_min, mu_max, budget, sweeps, tau_d);
        ProjOut o = P.search(R, mode, mu_min, mu_max, theta, tau_d, budget > 100 ? budget : 100);
        o.steps += steps;
        o.dykstra = 1;
        return o;
    }
    __device__ ProjOut solve(double R, int mode, double mu_min, double mu_max, double nu_hint, double tau_hint,
                             int budget) {
        return solve(R, mode, mu_min, mu_max, nu_hint, tau_hint, budget, [] {});
    }
};

// Cluster size used for a problem of n assets: about 512 elements per block
// (two per thread), at most 16 blocks.
inline int proj_cluster_size(int64_t n) {
    if (n <= 512) return 1;
    if (n <= 1024) return 2;
    if (n <= 2048) return 4;
    if (n <= 4096) return 8;
    return 16;
}

}  // namespace mv
