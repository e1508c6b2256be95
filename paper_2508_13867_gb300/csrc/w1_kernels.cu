// 1-Wasserstein distance between the speed distributions of two ensembles of velocity fields
// (arXiv 2508.13867, Sec. 8.3: W1 of the numerical statistical solutions of |u|).
//
// For two empirical distributions on the real line, W1 is the integral of |F_a(x) - F_b(x)|.
// Both sets of speeds are counted into the same `bins` equal bins over [0, vmax]; the integral
// over the binned CDFs is exact for the binned values, which differ from the true ones by less
// than one bin width h, so |W1_binned - W1| < h.  Three kernels: the largest speed, the two
// histograms (global atomics; the counts do not depend on their order), and one cluster that scans the
// bins and sums |F_a - F_b| exactly.  Non-finite speeds (samples that became unstable) are left out of
// both distributions and counted.
//
// FP64 instructions issue at 1/75 of the FP32 rate on GB300, and these kernels have nothing else to wait
// for, so they use FP64 only where FP32 cannot decide:
//   largest speed: the squared speed in FP32 picks the candidates, FP64 decides between close ones;
//   bins: the speed as the sum of two FP32 numbers (error below 2^-42 of it) gives the bin unless the
//     speed lies close to an edge (2^-40 of the range and a little more); then the FP64 formula decides;
//   distance: sum |n_b C_a - n_a C_b| over the bins in integers (C: cumulative counts; 64-bit products,
//     128-bit sum), one division at the end.
// Measured on 128 x 127^2 and 256 x 255^2 FP32 speeds in 2^20 bins: 0.30 against 7.83 ms in all (two
// FP64 divisions per bin on one block took most of it).
#include <cmath>

#include <cooperative_groups.h>

#include "uqlb_internal.h"

namespace uqlb {

namespace {

constexpr int kBlocks = 1216, kThreads = 256;

// Squared speed and speed in FP64 (the reference of every decision).
__device__ __forceinline__ double speed_sq(double u, double v) { return u * u + v * v; }

// Calls f(u, v) for the speeds of this thread's share: the nodes of all samples in one sequence (S nodes is
// at most 4e9, so that 32-bit indices and divisions do), whatever the length of a row.  4 million speeds in
// rows of 16 / 225 / 5000 nodes, largest speed and histogram of 2^20 bins: FP32 49 / 50 / 49 us, FP64 177 /
// 177 / 177; chunks of one sample at a time, which leave threads idle on short rows, took 351 / 56 / 50 and 656
// / 196 / 201.
template <typename M, typename Fn>
__device__ __forceinline__ void for_each_velocity(const M* m, int64_t S, int64_t nodes, int64_t ld, Fn&& f) {
    const unsigned n = (unsigned)nodes, all = (unsigned)(S * nodes), step = gridDim.x * kThreads;
    for (unsigned i = blockIdx.x * kThreads + threadIdx.x; i < all; i += step) {
        const unsigned s = i / n;
        const M* at = m + (int64_t)s * ld + (i - s * n);
        f(at[0], at[n]);
    }
}

template <typename M>
__global__ void __launch_bounds__(kThreads) max_speed_kernel(const M* m, int64_t S, int64_t nodes, int64_t ld,
                                                             unsigned long long* vmax_bits) {
    double best = 0.0;            // largest squared speed decided in FP64
    M cu = M(0), cv = M(0);       // candidate: the largest by its FP32 square, cq
    float cq = 0.0f;
    auto decide = [&](M u, M v) {
        const double q = speed_sq((double)u, (double)v);
        if (isfinite(q)) best = fmax(best, q);
    };
    for_each_velocity(m, S, nodes, ld, [&](M u, M v) {
        const float fu = (float)u, fv = (float)v, q = fmaf(fu, fu, fv * fv);  // error below 2^-22 of it
        if (q <= cq * 0.999999f && q >= 1e-30f) return;
        if (q > cq * 1.000001f && q >= 1e-30f && q < 1e30f) {
            cq = q;
            cu = u;
            cv = v;
        } else if (q >= 1e-30f || fu != 0.0f || fv != 0.0f || sizeof(M) == 8) {
            decide(u, v);  // as large as the candidate, or outside FP32's range; NaN is no speed
        }
    });
    decide(cu, cv);
    best = sqrt(best);
    for (int o = 16; o > 0; o >>= 1) best = fmax(best, __shfl_xor_sync(0xffffffffu, best, o));
    // non-negative doubles order like their bit patterns
    if ((threadIdx.x & 31) == 0) atomicMax(vmax_bits, (unsigned long long)__double_as_longlong(best));
}

// Bin of the speed of (u, v) under scale = sh + sl bins per unit, as FP32 pairs: u^2 + v^2 with its
// rounding errors, the root by one Newton step on the approximate one, times the scale.  All errors
// together stay below 2^-42 of the result, which is at most `bins`; false where the result lies within delta =
// bins 2^-40 + 2^-30 of an edge (or outside FP32's range, or is not finite) and FP64 has to decide.
__device__ __forceinline__ bool bin_fp32(float u, float v, float sh, float sl, float delta, int& bin) {
    if (u == 0.0f && v == 0.0f) {
        bin = 0;
        return true;
    }
    const float p = __fmul_rn(u, u), pe = __fmaf_rn(u, u, -p), q = __fmul_rn(v, v), qe = __fmaf_rn(v, v, -q);
    const float s = __fadd_rn(p, q), bb = __fsub_rn(s, p);
    const float lo = __fadd_rn(__fadd_rn(__fsub_rn(p, __fsub_rn(s, bb)), __fsub_rn(q, bb)), __fadd_rn(pe, qe));
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(s));
    const float r = __fmul_rn(s, y);
    const float c = __fmul_rn(__fadd_rn(__fmaf_rn(-r, r, s), lo), __fmul_rn(0.5f, y));  // root = r + c
    const float xh = __fmul_rn(r, sh);
    const float xl = __fmaf_rn(c, sh, __fmaf_rn(r, sl, __fmaf_rn(r, sh, -xh)));
    float n = floorf(xh), frac = __fadd_rn(__fsub_rn(xh, n), xl);
    if (frac < 0.0f) {
        n -= 1.0f;
        frac += 1.0f;
    } else if (frac >= 1.0f) {
        n += 1.0f;
        frac -= 1.0f;
    }
    bin = (int)n;
    return s > 1e-30f && s < 1e30f && frac > delta && frac < 1.0f - delta;
}

// Histogram of the speeds.  Non-finite speeds (an unstable sample) are not binned; they are counted in
// *nonfinite.  LOCAL: few bins, counted in shared memory first (hot bins would serialise in L2).
constexpr int kLocalBins = 8192, kLocalBlocks = 4 * 152;
template <typename M, bool LOCAL>
__global__ void __launch_bounds__(kThreads) speed_hist_kernel(const M* m, int64_t S, int64_t nodes, int64_t ld,
                                                              const unsigned long long* vmax_bits, int bins,
                                                              unsigned int* counts, unsigned long long* nonfinite) {
    __shared__ unsigned int local[LOCAL ? kLocalBins : 1];
    if constexpr (LOCAL) {
        for (int b = threadIdx.x; b < bins; b += kThreads) local[b] = 0u;
        __syncthreads();
    }
    const double vmax = __longlong_as_double((long long)*vmax_bits);
    const double scale = vmax > 0.0 ? bins / vmax : 0.0;
    const bool in_range = scale > 1e-25 && scale < 1e25;
    const float sh = in_range ? (float)scale : 0.0f, sl = in_range ? (float)(scale - (double)sh) : 0.0f;
    const float delta = in_range ? (float)bins * 0x1p-40f + 0x1p-30f : 2.0f;  // 2: FP64 decides
    for_each_velocity(m, S, nodes, ld, [&](M u, M v) {
        int b = 0;
        bool decided = false;
        if (sizeof(M) == 4) decided = bin_fp32((float)u, (float)v, sh, sl, delta, b);
        if (!decided) {
            const double w = sqrt(speed_sq((double)u, (double)v));
            if (!isfinite(w)) {
                atomicAdd(nonfinite, 1ull);
                return;
            }
            b = (int)(w * scale);
            b = b < 0 ? 0 : (b >= bins ? bins - 1 : b);
        }
        if constexpr (LOCAL)
            atomicAdd(local + b, 1u);
        else
            atomicAdd(counts + b, 1u);
    });
    if constexpr (LOCAL) {
        __syncthreads();
        for (int b = threadIdx.x; b < bins; b += kThreads)
            if (local[b]) atomicAdd(counts + b, local[b]);
    }
}

// Distance from the two histograms: one cluster, each block a contiguous share of the bins.  The blocks
// exchange the totals of their shares, then walk them with running cumulative counts.  n_a and n_b are at
// most 4e9, so their products fit 64 bits and cumulative counts 32.
constexpr int kScanThreads = 1024, kScanBlocks = 8;
__device__ __forceinline__ unsigned __int128 shfl_xor_128(unsigned __int128 v, int o) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)v, o);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(v >> 64), o);
    return (unsigned __int128)hi << 64 | lo;
}
__global__ void __cluster_dims__(kScanBlocks, 1, 1) __launch_bounds__(kScanThreads)
    w1_scan_kernel(const unsigned int* ca, const unsigned int* cb, int bins, unsigned long long na_all,
                   unsigned long long nb_all, const unsigned long long* vmax_bits, const unsigned long long* nonfinite,
                   double* out) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    __shared__ unsigned int total[2];
    __shared__ unsigned int wsum[2][kScanThreads / 32];
    __shared__ unsigned long long part[2];
    __shared__ unsigned long long wpart[2][kScanThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = (int)cluster.block_rank();
    const unsigned long long na = na_all - nonfinite[0], nb = nb_all - nonfinite[1];
    const int per = (bins + kScanBlocks - 1) / kScanBlocks;
    const int lo = rank * per < bins ? rank * per : bins, hi = lo + per < bins ? lo + per : bins;
    unsigned int ta = 0, tb = 0;
    for (int b = lo + tid; b < hi; b += kScanThreads) {
        ta += ca[b];
        tb += cb[b];
    }
    ta = __reduce_add_sync(0xffffffffu, ta);
    tb = __reduce_add_sync(0xffffffffu, tb);
    if (lane == 0) {
        wsum[0][warp] = ta;
        wsum[1][warp] = tb;
    }
    __syncthreads();
    if (tid < 2) {
        unsigned int s = 0;
        for (int w = 0; w < kScanThreads / 32; ++w) s += wsum[tid][w];
        total[tid] = s;
    }
    cluster.sync();
    unsigned int ra = 0, rb = 0;  // counts before the current bins
    for (int q = 0; q < rank; ++q) {
        const unsigned int* t = cluster.map_shared_rank(total, q);
        ra += t[0];
        rb += t[1];
    }
    unsigned __int128 acc = 0;
    constexpr int kPer = 4;
    for (int b0 = lo; b0 < hi; b0 += kScanThreads * kPer) {
        unsigned int va[kPer], vb[kPer], sa = 0, sb = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int b = b0 + tid * kPer + k;
            va[k] = b < hi ? ca[b] : 0u;
            vb[k] = b < hi ? cb[b] : 0u;
            sa += va[k];
            sb += vb[k];
        }
        unsigned int ia = sa, ib = sb;  // inclusive sums over the warp, then over the block
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int x = __shfl_up_sync(0xffffffffu, ia, o), y = __shfl_up_sync(0xffffffffu, ib, o);
            if (lane >= o) {
                ia += x;
                ib += y;
            }
        }
        __syncthreads();
        if (lane == 31) {
            wsum[0][warp] = ia;
            wsum[1][warp] = ib;
        }
        __syncthreads();
        unsigned int pa = 0, pb = 0, all_a = 0, all_b = 0;
        {
            unsigned int xa = wsum[0][lane], xb = wsum[1][lane];
            all_a = __reduce_add_sync(0xffffffffu, xa);
            all_b = __reduce_add_sync(0xffffffffu, xb);
            pa = __reduce_add_sync(0xffffffffu, lane < warp ? xa : 0u);
            pb = __reduce_add_sync(0xffffffffu, lane < warp ? xb : 0u);
        }
        unsigned int qa = ra + pa + ia - sa, qb = rb + pb + ib - sb;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            qa += va[k];
            qb += vb[k];
            const unsigned long long x = (unsigned long long)qa * nb, y = (unsigned long long)qb * na;
            if (b0 + tid * kPer + k < hi) acc += x > y ? x - y : y - x;
        }
        ra += all_a;
        rb += all_b;
    }
    for (int o = 16; o > 0; o >>= 1) acc += shfl_xor_128(acc, o);
    if (lane == 0) {
        wpart[0][warp] = (unsigned long long)acc;
        wpart[1][warp] = (unsigned long long)(acc >> 64);
    }
    __syncthreads();
    if (tid == 0) {
        acc = 0;
        for (int w = 0; w < kScanThreads / 32; ++w) acc += (unsigned __int128)wpart[1][w] << 64 | wpart[0][w];
        part[0] = (unsigned long long)acc;
        part[1] = (unsigned long long)(acc >> 64);
    }
    cluster.sync();
    if (rank == 0 && tid == 0) {
        acc = 0;
        for (int q = 0; q < kScanBlocks; ++q) {
            const unsigned long long* t = cluster.map_shared_rank(part, q);
            acc += (unsigned __int128)t[1] << 64 | t[0];
        }
        const double h = __longlong_as_double((long long)*vmax_bits) / bins;
        const double sum = (double)(unsigned long long)(acc >> 64) * 0x1p64 + (double)(unsigned long long)acc;
        out[0] = (na > 0 && nb > 0) ? sum / ((double)na * (double)nb) * h : NAN;
        out[1] = h;
        out[2] = (double)nonfinite[0];
        out[3] = (double)nonfinite[1];
    }
    cluster.sync();  // the other blocks' shared memory stays until it has been read
}

template <typename M>
cudaError_t launch_max(const M* m, int64_t S, int64_t nodes, int64_t ld, unsigned long long* vmax, cudaStream_t s) {
    max_speed_kernel<M><<<kBlocks, kThreads, 0, s>>>(m, S, nodes, ld, vmax);
    return cudaGetLastError();
}

template <typename M>
cudaError_t launch_hist(const M* m, int64_t S, int64_t nodes, int64_t ld, const unsigned long long* vmax, int bins,
                        unsigned int* counts, unsigned long long* nonfinite, cudaStream_t s) {
    // Few bins: counted in shared memory, about eight speeds per thread, so that small sets spread over the
    // chip too, in at most four blocks per SM, which hold enough loads in flight (more only add counts to
    // flush).  Measured, blocks of eight speeds per thread / global atomics: 65536 speeds FP32 8 us / 13 us in
    // 8192 bins, 8 / 50 in one; 2 million 15..23 / 105..1414; FP64 13 / 17 and 58..66 / 109..1315 us.
    const int64_t blocks = (S * nodes + 8 * kThreads - 1) / (8 * kThreads);
    if (bins <= kLocalBins)
        speed_hist_kernel<M, true><<<(int)(blocks < kLocalBlocks ? blocks : kLocalBlocks), kThreads, 0, s>>>(
            m, S, nodes, ld, vmax, bins, counts, nonfinite);
    else
        speed_hist_kernel<M, false><<<kBlocks, kThreads, 0, s>>>(m, S, nodes, ld, vmax, bins, counts, nonfinite);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_w1_speed(const void* a, int dta, int64_t sa, int64_t na, int64_t lda, const void* b, int dtb,
                            int64_t sb, int64_t nb, int64_t ldb, int bins, void* ws, double* out_dev, cudaStream_t s) {
    auto* vmax = static_cast<unsigned long long*>(ws);
    auto* nonfinite = vmax + 1;  // two counters, one per set
    auto* ca = reinterpret_cast<unsigned int*>(static_cast<char*>(ws) + 256);
    unsigned int* cb = ca + bins;
    cudaError_t e;
    if ((e = cudaMemsetAsync(ws, 0, 256 + (size_t)2 * bins * sizeof(unsigned int), s))) return e;
    e = dta == UQLB_F64 ? launch_max(static_cast<const double*>(a), sa, na, lda, vmax, s)
                        : launch_max(static_cast<const float*>(a), sa, na, lda, vmax, s);
    if (e) return e;
    e = dtb == UQLB_F64 ? launch_max(static_cast<const double*>(b), sb, nb, ldb, vmax, s)
                        : launch_max(static_cast<const float*>(b), sb, nb, ldb, vmax, s);
    if (e) return e;
    e = dta == UQLB_F64 ? launch_hist(static_cast<const double*>(a), sa, na, lda, vmax, bins, ca, nonfinite, s)
                        : launch_hist(static_cast<const float*>(a), sa, na, lda, vmax, bins, ca, nonfinite, s);
    if (e) return e;
    e = dtb == UQLB_F64 ? launch_hist(static_cast<const double*>(b), sb, nb, ldb, vmax, bins, cb, nonfinite + 1, s)
                        : launch_hist(static_cast<const float*>(b), sb, nb, ldb, vmax, bins, cb, nonfinite + 1, s);
    if (e) return e;
    w1_scan_kernel<<<kScanBlocks, kScanThreads, 0, s>>>(ca, cb, bins, (unsigned long long)(sa * na),
                                                        (unsigned long long)(sb * nb), vmax, nonfinite, out_dev);
    return cudaGetLastError();
}

}  // namespace uqlb
