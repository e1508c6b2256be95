// gPC projection and ensemble statistics (arXiv 2508.13867, Sec. 4 and Algorithm 1).
//
//   coefficients (Eq. coef_discrete, gamma_k = 1):  C[k, f] = sum_s W[k, s] M[s, f],
//                                                     W[k, s] = a_s Phi_k(xi_s)
//   gPC mean / variance (Eq. gpc_mean, Eq. gpc_std):  mean = C[0, f], var = sum_{k>=1} C[k, f]^2
//   Monte Carlo (Eq. meanMCS, Eq. varMCS):           two passes over the samples in FP64, or (FP32 fields of
//     many samples) one pass with sums of three FP32 numbers
// All other accumulation is FP64; M may be FP32 (the ensemble's field output) or FP64.
// The contraction is [K x S] x [S x F] with K <= a few hundred and F up to ~10^6.  Three forms: one input at
// a time on tensor grids (sf_stage_kernel), over reflected samples on symmetric sample sets
// (reflect_kernel), dense (project_kernel).
#include <cmath>
#include <cstdio>
#include <mutex>
#include <type_traits>

#include "uqlb_internal.h"

namespace uqlb {

namespace {

constexpr int kProjThreads = 128;
constexpr int kSB = 128;  // samples per shared-memory stage

// Dense contraction, KB coefficients per block (blockIdx.y chunk) and FPT fields per thread.  FP64
// instructions bound it (one per warp in 19 cycles of an SM), so a term block that divides K badly costs
// in proportion: launch_dense_any() takes the KB with the least work for K (K = 35: 37 instructions
// per sample in one block of 36 against 51 in three of 16; the conversion of a value is shared by the
// block's terms), or the smallest blocks where few fields leave SMs idle.
template <typename M, int KB, int FPT>
__global__ void __launch_bounds__(kProjThreads) project_kernel(const double* __restrict__ W, int K, int S,
                                                               const M* __restrict__ m, int64_t F, int64_t ld,
                                                               double* __restrict__ C) {
    __shared__ double sw[KB][kSB];
    const int k0 = blockIdx.y * KB;
    const int64_t f0 = ((int64_t)blockIdx.x * kProjThreads) * FPT + threadIdx.x;
    double acc[FPT][KB];
#pragma unroll
    for (int a = 0; a < FPT; ++a)
#pragma unroll
        for (int k = 0; k < KB; ++k) acc[a][k] = 0.0;

    for (int s0 = 0; s0 < S; s0 += kSB) {
        const int sn = min(kSB, S - s0);
        for (int q = threadIdx.x; q < KB * kSB; q += kProjThreads) {
            const int kk = q / kSB, ss = q % kSB;
            sw[kk][ss] = (k0 + kk < K && ss < sn) ? W[(int64_t)(k0 + kk) * S + s0 + ss] : 0.0;
        }
        __syncthreads();
        for (int ss = 0; ss < sn; ++ss) {
            const M* row = m + (int64_t)(s0 + ss) * ld;
            double v[FPT];
#pragma unroll
            for (int a = 0; a < FPT; ++a) {
                const int64_t f = f0 + (int64_t)a * kProjThreads;
                v[a] = f < F ? (double)row[f] : 0.0;
            }
#pragma unroll
            for (int k = 0; k < KB; ++k) {
                const double w = sw[k][ss];
#pragma unroll
                for (int a = 0; a < FPT; ++a) acc[a][k] = fma(w, v[a], acc[a][k]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < FPT; ++a) {
        const int64_t f = f0 + (int64_t)a * kProjThreads;
        if (f >= F) continue;
#pragma unroll
        for (int k = 0; k < KB; ++k)
            if (k0 + k < K) C[(int64_t)(k0 + k) * F + f] = acc[a][k];
    }
}

// In integers: an FP64 comparison takes the units that bound these kernels.
__device__ __forceinline__ bool not_finite(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

// Contraction over reflected samples.  A sample set that is symmetric in every input (Clenshaw-Curtis
// Smolyak and Gauss-Legendre grids) falls into orbits of 2^m samples that differ in the signs of their m
// nonzero reference coordinates.  The weights of a term over an orbit are equal up to the sign that its
// odd degrees give, so with the signed sums h[p] = sum_b (-1)^(p.b) M[s_b] (m 2^m additions) an orbit adds
// w_k h[p_k] to term k, and nothing to terms of odd degree in a zero coordinate: 549 multiply-adds and 272
// additions per field where the dense contraction of 137 samples and 35 terms takes 4795.  Per-thread sums
// lie in shared memory (a term's index is data).  A field with a non-finite value, or whose signed sums
// leave the range of FP64, takes the products one by one, zero weights included, as the dense contraction
// does.  Measured, 137 samples x 35 terms x 130051 fields: 0.36 against 1.66 ms dense (with the statistics).
constexpr int kReflThreads = 128;
template <typename M>
__global__ void __launch_bounds__(kReflThreads) reflect_kernel(const ReflOrbit* __restrict__ orbits, int norbits,
                                                               const ReflTerm* __restrict__ terms,
                                                               const int* __restrict__ members, int K, int hrows,
                                                               const M* __restrict__ m, int64_t F, int64_t ld,
                                                               double* __restrict__ C) {
    extern __shared__ double s_refl[];
    double* const acc = s_refl + threadIdx.x;                       // [K][threads]
    double* const hs = s_refl + (int64_t)K * kReflThreads + threadIdx.x;  // [hrows][threads]
    const int64_t f = (int64_t)blockIdx.x * kReflThreads + threadIdx.x;
    if (f >= F) return;  // no barrier below
    for (int k = 0; k < K; ++k) acc[k * kReflThreads] = 0.0;
    auto at = [&](int s) { return (double)m[(int64_t)s * ld + f]; };
    bool finite = true;
    auto orbit = [&](auto m_c, const ReflOrbit& o) {
        constexpr int MM = decltype(m_c)::value, N = 1 << MM;
        double v[N];
#pragma unroll
        for (int b = 0; b < N; ++b) v[b] = at(__ldg(members + o.member + b));
#pragma unroll
        for (int d = 0; d < MM; ++d)
#pragma unroll
            for (int b = 0; b < N; ++b)
                if (!(b >> d & 1)) {
                    const double x = v[b], y = v[b | 1 << d];
                    v[b] = x + y;
                    v[b | 1 << d] = x - y;
                }
        finite = finite && !not_finite(v[0]);
#pragma unroll
        for (int b = 0; b < N; ++b) hs[b * kReflThreads] = v[b];
        for (int q = o.term; q < o.term + o.nterms; ++q) {
            const ReflTerm t = terms[q];
            acc[t.k * kReflThreads] = fma(t.w, hs[t.p * kReflThreads], acc[t.k * kReflThreads]);
        }
    };
    for (int i = 0; i < norbits; ++i) {
        const ReflOrbit o = orbits[i];
        switch (o.m) {
            case 0: orbit(std::integral_constant<int, 0>{}, o); break;
            case 1: orbit(std::integral_constant<int, 1>{}, o); break;
            case 2: orbit(std::integral_constant<int, 2>{}, o); break;
            case 3: orbit(std::integral_constant<int, 3>{}, o); break;
            default: orbit(std::integral_constant<int, 4>{}, o); break;
        }
    }
    for (int k = 0; k < K; ++k) {
        const double c = acc[k * kReflThreads];
        finite = finite && !not_finite(c);  // a difference can leave FP64's range where the sum v[0] does not
        C[(int64_t)k * F + f] = c;
    }
    if (!finite) {
        for (int k = 0; k < K; ++k) acc[k * kReflThreads] = 0.0;
        for (int i = 0; i < norbits; ++i) {
            const ReflOrbit o = orbits[i];
            for (int b = 0; b < 1 << o.m; ++b) {
                const double x = at(members[o.member + b]);
                int q = o.term;  // terms ascend in k
                for (int k = 0; k < K; ++k) {
                    double w = 0.0;
                    if (q < o.term + o.nterms && terms[q].k == k) {
                        w = (__popc(terms[q].p & b) & 1) ? -terms[q].w : terms[q].w;
                        ++q;
                    }
                    acc[k * kReflThreads] = fma(w, x, acc[k * kReflThreads]);
                }
            }
        }
        for (int k = 0; k < K; ++k) C[(int64_t)k * F + f] = acc[k * kReflThreads];
    }
}

__global__ void gpc_stats_kernel(const double* __restrict__ C, int K, int64_t F, double* mean, double* var) {
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < F; f += (int64_t)gridDim.x * blockDim.x) {
        double v = 0.0;
        for (int k = 1; k < K; ++k) {
            const double c = C[(int64_t)k * F + f];
            v = fma(c, c, v);
        }
        if (mean) mean[f] = C[f];
        if (var) var[f] = v;
    }
}

// ddof < 0: var receives the sum of squared deviations itself (M2 of a block, for merging blocks).
template <typename M>
__global__ void mc_stats_kernel(const M* __restrict__ m, int64_t S, int64_t F, int64_t ld, double* mean,
                                double* var, int ddof) {
    for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < F; f += (int64_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int64_t q = 0; q < S; ++q) s += (double)m[q * ld + f];
        const double mu = s / (double)S;
        double ss = 0.0;
        for (int64_t q = 0; q < S; ++q) {
            const double d = (double)m[q * ld + f] - mu;
            ss = fma(d, d, ss);
        }
        if (mean) mean[f] = mu;
        if (var) var[f] = ddof < 0 ? ss : ((S - ddof) > 0 ? ss / (double)(S - ddof) : NAN);
    }
}

// Monte Carlo statistics of FP32 fields in one pass and (almost) without FP64.  FP64 instructions issue at
// 1/75 of the FP32 rate on GB300, so the two-pass FP64 loop above is bound by its five of them per value.
// Here the deviations d = x - c from the field's first sample c are formed exactly (a sum of two FP32
// numbers), and sum d and sum d^2 are kept as sums of three FP32 numbers with exact rounding errors
// (Knuth's two-sum, products by FMA): about 70 bits, more than FP64 holds.  The rest,
// var = (sum d^2 - (sum d)^2 / S) / (S - ddof), takes pairs of FP64 numbers once per field, so that the
// cancellation of the shift costs nothing.  A field with a non-finite value, or a deviation outside
// [1e-15, 1e15] (whose square or its rounding error would leave FP32's range), is left to FP64.
// A block takes 32 fields, each of its eight warps every eighth sample.  Measured on 1024 samples of 2 x
// 512^2 + 1 fields: 0.92 against 5.09 ms (mc_one_pass() says for which sizes).
constexpr int kMcWarps = 8;
struct Sum3 {
    float a, b, c;
};
__device__ __forceinline__ float two_sum(float& s, float x) {  // s += x; returns the rounding error
    const float t = __fadd_rn(s, x), v = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, v)), __fsub_rn(x, v));
    s = t;
    return e;
}
__device__ __forceinline__ void add_low(Sum3& s, float x) { s.c = __fadd_rn(s.c, two_sum(s.b, x)); }
__device__ __forceinline__ void add(Sum3& s, float x) { add_low(s, two_sum(s.a, x)); }
__device__ __forceinline__ void add(Sum3& s, const Sum3& x) {
    add(s, x.a);
    add_low(s, x.b);
    s.c = __fadd_rn(s.c, x.c);
}
struct Pair64 {
    double h, l;
};
__device__ __forceinline__ Pair64 quick_sum(double a, double b) {  // Dekker's fast two-sum: |a| >= |b|, or a == 0
    const double h = a + b;
    return {h, b - (h - a)};
}
__device__ __forceinline__ Pair64 to_pair(const Sum3& s) {
    const Pair64 p = quick_sum((double)s.a, (double)s.b);
    return quick_sum(p.h, p.l + (double)s.c);
}

__global__ void __launch_bounds__(32 * kMcWarps) mc_stats_f32_kernel(const float* __restrict__ m, int64_t S, int64_t F,
                                                                     int64_t ld, double* mean, double* var, int ddof) {
    __shared__ Sum3 sd[kMcWarps][32], sq[kMcWarps][32];
    __shared__ double sx[kMcWarps][32];
    __shared__ int bad_warps[kMcWarps];
    const int lane = threadIdx.x, warp = threadIdx.y;
    const int64_t f = blockIdx.x * (int64_t)32 + lane;
    const float* col = m + (f < F ? f : F - 1);
    const float c = __ldg(col);
    Sum3 d{}, q{};
    bool bad = false;
    auto take = [&](float x) {
        float dh = x;
        const float dl = two_sum(dh, -c);
        const float t = fabsf(dh);
        bad = bad || !(t <= 1e15f) || (t < 1e-15f && t > 0.0f);
        const float p = __fmul_rn(dh, dh), e = __fmaf_rn(dh, dh, -p);
        add(d, dh);
        add(q, p);
        add_low(q, e);
        if (__any_sync(0xffffffffu, dl != 0.0f)) {  // values within a factor of two of c give none
            const float d2 = dh + dh, p2 = __fmul_rn(d2, dl), e2 = __fmaf_rn(d2, dl, -p2);
            add_low(d, dl);
            add_low(q, p2);
            q.c = __fadd_rn(q.c, __fmaf_rn(dl, dl, e2));
        }
    };
    constexpr int kAhead = 8;
    int64_t s = warp;
    for (; s + (kAhead - 1) * kMcWarps < S; s += kAhead * kMcWarps) {
        float x[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) x[k] = __ldg(col + (s + k * kMcWarps) * ld);
#pragma unroll
        for (int k = 0; k < kAhead; ++k) take(x[k]);
    }
    for (; s < S; s += kMcWarps) take(__ldg(col + s * ld));
    sd[warp][lane] = d;
    sq[warp][lane] = q;
    const unsigned bad_lanes = __ballot_sync(0xffffffffu, bad);
    if (lane == 0) bad_warps[warp] = (int)bad_lanes;
    __syncthreads();
    unsigned any_bad = 0;
#pragma unroll
    for (int w = 0; w < kMcWarps; ++w) any_bad |= (unsigned)bad_warps[w];
    if (warp == 0 && f < F && !((any_bad >> lane) & 1)) {
        for (int w = 1; w < kMcWarps; ++w) {
            add(d, sd[w][lane]);
            add(q, sq[w][lane]);
        }
        const double n = (double)S;
        const Pair64 D = to_pair(d), Q = to_pair(q);
        const double md = D.h / n, mr = (fma(-md, n, D.h) + D.l) / n;  // mean of d = md + mr
        if (mean) mean[f] = (double)c + (md + mr);
        if (var) {
            // T = D^2 / n = D md + D mr, as a pair; Q - T
            const double th = D.h * md, tl = fma(D.h, md, -th) + (D.l * md + D.h * mr);
            const double r = Q.h - th, v = r - Q.h, e = (Q.h - (r - v)) - (th + v);
            const double ss = fmax(r + (e + (Q.l - tl)), 0.0);
            var[f] = ddof < 0 ? ss : ((S - ddof) > 0 ? ss / (double)(S - ddof) : NAN);
        }
    }
    if (any_bad == 0) return;
    // FP64 in two passes for the fields left to it
    const bool mine = ((any_bad >> lane) & 1) && f < F;
    double acc = 0.0;
    if (mine)
        for (int64_t k = warp; k < S; k += kMcWarps) acc += (double)__ldg(col + k * ld);
    sx[warp][lane] = acc;
    __syncthreads();
    double mu = 0.0;
    for (int w = 0; w < kMcWarps; ++w) mu += sx[w][lane];
    mu /= (double)S;
    __syncthreads();
    acc = 0.0;
    if (mine)
        for (int64_t k = warp; k < S; k += kMcWarps) {
            const double x = (double)__ldg(col + k * ld) - mu;
            acc = fma(x, x, acc);
        }
    sx[warp][lane] = acc;
    __syncthreads();
    if (warp == 0 && mine) {
        double ss = 0.0;
        for (int w = 0; w < kMcWarps; ++w) ss += sx[w][lane];
        if (mean) mean[f] = mu;
        if (var) var[f] = ddof < 0 ? ss : ((S - ddof) > 0 ? ss / (double)(S - ddof) : NAN);
    }
}

// Sum factorization of the projection on a tensor Gauss-Legendre grid.  There W[k, s] is a product
// over the input dimensions, W[k, s] = prod_q G[alpha_kq][s_q] with G[a][s] = (w_s / 2) phi_a(x_s) (the
// 1-D probability weight times the orthonormal Legendre polynomial), so C = W M contracts one
// dimension at a time, the last (fastest) first.  One stage maps an input T[(r n + s) J' + j'][f] to
// T[r J + o(a, j')][f] = sum_{s < n} G[a][s] T[(r n + s) J' + j'][f] for every degree a that the
// multi-index set admits after the partial index j' (a prefix a = 0 .. c - 1 of the degrees; o(a, j') =
// -1 beyond it; at the last stage o is the coefficient's row k).  A thread owns one field and one
// group (r, j'): it loads the n inputs once and accumulates the c outputs as independent chains, so
// the FP64 pipe (a small fraction of the FP32 rate on GB300) always has several multiply-adds to
// issue.  FP64 throughout.
// The points of a Gauss-Legendre rule are symmetric, so G[a][n-1-q] = (-1)^a G[a][q] up to rounding: with the
// sums and differences of opposite inputs a degree takes half the multiply-adds (n = 5, five degrees: 4
// additions and 15 multiply-adds instead of 25; the middle input keeps its rounding-sized weight in the
// odd degrees, so that a non-finite value reaches every coefficient; a thread with a non-finite result takes
// the products one by one).  Points and degrees are compile-time (a runtime bound left the unrolled
// multiply-adds of 16 points and 9 degrees in the loop, predicated off).  Measured on 625 samples x 131073 fields, all four stages: 1.43 against 3.88 ms (with the statistics).
constexpr int kSfThreads = 256;

// One group of N points; true if its folded inputs left the range of FP64 (or were not finite).
template <int N, int CNT, typename TI>
__device__ __forceinline__ bool sf_group(const TI* src, int64_t step, const double (*G)[kSfMaxPoints], double* out,
                                         int64_t out_ld, const int* __restrict__ o) {
    constexpr int H = N / 2;
    double x[N], e[H > 0 ? H : 1], d[H > 0 ? H : 1];
#pragma unroll
    for (int q = 0; q < N; ++q) x[q] = (double)src[q * step];
#pragma unroll
    for (int q = 0; q < H; ++q) {
        e[q] = x[q] + x[N - 1 - q];
        d[q] = x[q] - x[N - 1 - q];
    }
    double y[CNT];
#pragma unroll
    for (int a = 0; a < CNT; ++a) {
        y[a] = N % 2 == 1 ? G[a][H] * x[H] : 0.0;
#pragma unroll
        for (int q = 0; q < H; ++q)
            y[a] = q == 0 && N % 2 == 0 ? G[a][q] * (a % 2 == 0 ? e[q] : d[q]) : fma(G[a][q], a % 2 == 0 ? e[q] : d[q], y[a]);
    }
#pragma unroll
    for (int a = 0; a < CNT; ++a) out[(int64_t)__ldg(o + a) * out_ld] = y[a];
    // a non-finite input, sum or difference of inputs reaches the first even or the first odd degree, whose
    // weights have no zeros; FP32 inputs have no sums beyond FP64's range
    return sizeof(TI) == 8 && N > 1 && (not_finite(y[0]) || (CNT > 1 && not_finite(y[CNT > 1 ? 1 : 0])));
}

// The same for n points that are not compiled in, without the fold: the inputs are loaded and converted once,
// and the degrees are CNT independent chains, with eight, four, two and one inputs in flight (n = 10 in fours
// with a remainder one by one: 12 % longer).  Measured with the statistics, FP32 / FP64 fields, 131073 fields:
// 16 x 16 points at degree 8 757 / 682 us, 10 x 10 at degree 4 195 / 167; one degree after the other, which
// reloads and converts the inputs for each, 1288 / 682 and 296 / 167; all nine degrees with predicates 887 / 813
// and 357 / 329.
template <int CNT, typename TI>
__device__ __forceinline__ void sf_group_any(const TI* src, int64_t step, int n, const double (*G)[kSfMaxPoints],
                                             double* out, int64_t out_ld, const int* __restrict__ o) {
    double y[CNT];
#pragma unroll
    for (int a = 0; a < CNT; ++a) y[a] = 0.0;
    int q = 0;
    auto take = [&](auto u_c) {
        constexpr int U = decltype(u_c)::value;
        TI v[U];
#pragma unroll
        for (int i = 0; i < U; ++i) v[i] = src[(q + i) * step];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const double x = (double)v[i];
#pragma unroll
            for (int a = 0; a < CNT; ++a) y[a] = fma(G[a][q + i], x, y[a]);
        }
        q += U;
    };
    while (n - q >= 8) take(std::integral_constant<int, 8>{});
    if (n - q >= 4) take(std::integral_constant<int, 4>{});
    if (n - q >= 2) take(std::integral_constant<int, 2>{});
    if (n - q >= 1) take(std::integral_constant<int, 1>{});
#pragma unroll
    for (int a = 0; a < CNT; ++a) out[(int64_t)__ldg(o + a) * out_ld] = y[a];
}

// Calls an expression with the compile-time count C of admitted degrees.
#define UQLB_SF_CASE(C_, CALL) \
    case C_: { \
        constexpr int C = C_; \
        CALL; \
        break; \
    }
#define UQLB_SF_SWITCH(...) \
    switch (cnt) { \
        UQLB_SF_CASE(1, (__VA_ARGS__)) \
        UQLB_SF_CASE(2, (__VA_ARGS__)) \
        UQLB_SF_CASE(3, (__VA_ARGS__)) \
        UQLB_SF_CASE(4, (__VA_ARGS__)) \
        UQLB_SF_CASE(5, (__VA_ARGS__)) \
        UQLB_SF_CASE(6, (__VA_ARGS__)) \
        UQLB_SF_CASE(7, (__VA_ARGS__)) \
        UQLB_SF_CASE(8, (__VA_ARGS__)) \
        UQLB_SF_CASE(9, (__VA_ARGS__)) \
    }

// N: points per input (0: runtime n).
template <typename TI, int N>
__global__ void __launch_bounds__(kSfThreads) sf_stage_kernel(const TI* __restrict__ in, int64_t in_ld,
                                                              double* __restrict__ out, int64_t out_ld,
                                                              int64_t groups, int jprev, int jout, int n, int p1,
                                                              const int* __restrict__ oidx,
                                                              const double* __restrict__ G, int64_t F) {
    __shared__ double sG[kSfMaxDegree + 1][kSfMaxPoints];
    for (int q = threadIdx.x; q < (kSfMaxDegree + 1) * kSfMaxPoints; q += kSfThreads) {
        const int a = q / kSfMaxPoints, c = q % kSfMaxPoints;
        double g = 0.0;
        if (a < p1 && c < n) {
            g = G[a * n + c];
            // both halves' weights, which differ by rounding only, as their mean
            if (N > 0 && 2 * c + 1 != n) g = 0.5 * (g + (a % 2 == 0 ? G[a * n + n - 1 - c] : -G[a * n + n - 1 - c]));
        }
        sG[a][c] = g;
    }
    __syncthreads();
    const int64_t f = (int64_t)blockIdx.x * kSfThreads + threadIdx.x;
    if (f >= F) return;  // no barrier below
    bool redo = false;
    for (int64_t g = blockIdx.y; g < groups; g += gridDim.y) {
        const int64_t r = g / jprev;
        const int jp = (int)(g - r * jprev);
        const int* o = oidx + jp * p1;
        int cnt = 0;  // admitted degrees: a prefix of 0 .. p1 - 1
        while (cnt < p1 && __ldg(o + cnt) >= 0) ++cnt;
        const TI* src = in + ((r * n) * jprev + jp) * in_ld + f;
        const int64_t step = (int64_t)jprev * in_ld;
        double* dst = out + (r * jout) * out_ld + f;
        if constexpr (N > 0) {
            UQLB_SF_SWITCH(redo |= sf_group<N, C>(src, step, sG, dst, out_ld, o))
        } else {
            UQLB_SF_SWITCH(sf_group_any<C>(src, step, n, sG, dst, out_ld, o))
        }
    }
    if (!redo) return;
    // this thread's groups once more, product by product (after the loop: tests and a second path within it
    // cost the 625 samples x 131073 fields 6 %)
    for (int64_t g = blockIdx.y; g < groups; g += gridDim.y) {
        const int64_t r = g / jprev;
        const int jp = (int)(g - r * jprev);
        for (int a = 0; a < p1; ++a) {
            const int to = __ldg(oidx + jp * p1 + a);
            if (to < 0) break;
            double y = 0.0;
            for (int q = 0; q < n; ++q) y = fma(sG[a][q], (double)in[((r * n + q) * jprev + jp) * in_ld + f], y);
            out[(r * jout + to) * out_ld + f] = y;
        }
    }
}
static_assert(kSfMaxDegree == 8, "sf_stage_kernel has a case for each count of degrees");

template <typename TI>
void launch_sf(dim3 grid, cudaStream_t s, const TI* in, int64_t in_ld, double* out, int64_t out_ld, int64_t groups,
               int jprev, int jout, int n, int p1, const int* oidx, const double* G, int64_t F) {
#define UQLB_SF_POINTS(N_) \
    case N_: \
        sf_stage_kernel<TI, N_><<<grid, kSfThreads, 0, s>>>(in, in_ld, out, out_ld, groups, jprev, jout, n, p1, oidx, G, F); \
        return;
    switch (n) {
        UQLB_SF_POINTS(2)
        UQLB_SF_POINTS(3)
        UQLB_SF_POINTS(4)
        UQLB_SF_POINTS(5)
        UQLB_SF_POINTS(6)
        UQLB_SF_POINTS(7)
        UQLB_SF_POINTS(8)
        UQLB_SF_POINTS(9)
    }
#undef UQLB_SF_POINTS
    sf_stage_kernel<TI, 0><<<grid, kSfThreads, 0, s>>>(in, in_ld, out, out_ld, groups, jprev, jout, n, p1, oidx, G, F);
}

template <typename M, int KB, int FPT>
void launch_dense(const double* W, int K, int S, const M* m, int64_t F, int64_t ld, double* C, cudaStream_t s) {
    const int64_t per_block = (int64_t)kProjThreads * FPT;
    const dim3 grid((unsigned)((F + per_block - 1) / per_block), (unsigned)((K + KB - 1) / KB));
    project_kernel<M, KB, FPT><<<grid, kProjThreads, 0, s>>>(W, K, S, m, F, ld, C);
}
template <typename M>
void launch_dense_any(const double* W, int K, int S, const M* m, int64_t F, int64_t ld, double* C, cudaStream_t s) {
    // FP64 instructions per sample of the busiest SM: a thread's terms and conversions times the blocks per SM.
    // One block saturates its SM's FP64 units, so many fields go by the total work alone, and few, which
    // leave SMs idle, take small blocks (137 samples, 70 terms, 2049 fields: 98 us, by total work 222; 41 samples,
    // 35 terms, 129 fields 39 / 79).
    struct Size {
        int kb, fpt;
    };
    constexpr Size kSizes[] = {{6, 2}, {12, 2}, {16, 2}, {24, 1}, {36, 1}};
    int best = 0;
    int64_t cost = 0;
    for (const Size& z : kSizes) {
        const int64_t blocks = (F + kProjThreads * z.fpt - 1) / (kProjThreads * z.fpt) * ((K + z.kb - 1) / z.kb);
        const int64_t c = (blocks + 151) / 152 * (z.fpt * (z.kb + 1));
        if (best == 0 || c < cost) {
            best = z.kb;
            cost = c;
        }
    }
    switch (best) {
        case 6: return launch_dense<M, 6, 2>(W, K, S, m, F, ld, C, s);
        case 12: return launch_dense<M, 12, 2>(W, K, S, m, F, ld, C, s);
        case 16: return launch_dense<M, 16, 2>(W, K, S, m, F, ld, C, s);
        case 24: return launch_dense<M, 24, 1>(W, K, S, m, F, ld, C, s);
        default: return launch_dense<M, 36, 1>(W, K, S, m, F, ld, C, s);
    }
}

template <typename M>
cudaError_t launch_refl(const ReflPlanView& p, int K, const M* m, int64_t F, int64_t ld, double* C, cudaStream_t s) {
    const int hrows = 1 << p.max_m;
    const size_t smem = (size_t)(K + hrows) * kReflThreads * sizeof(double);
    if (smem > 48 * 1024) {
        // the limit belongs to the current device, so it is set for each launch that needs it (1.5 us on the
        // host); always the same value, as threads of one process may launch at once
        const cudaError_t e = cudaFuncSetAttribute(reflect_kernel<M>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   kReflMaxRows * kReflThreads * (int)sizeof(double));
        if (e != cudaSuccess) return e;
    }
    reflect_kernel<M><<<(unsigned)((F + kReflThreads - 1) / kReflThreads), kReflThreads, smem, s>>>(
        p.orbits, p.norbits, p.terms, p.members, K, hrows, m, F, ld, C);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sf_stage(const void* in, int in_dtype, int64_t in_ld, double* out, int64_t out_ld, int64_t groups,
                            int jprev, int jout, int n, int p1, const int* oidx, const double* G, int64_t F,
                            cudaStream_t s) {
    if (F <= 0 || groups <= 0) return cudaSuccess;
    if (n < 1 || n > kSfMaxPoints || p1 < 1 || p1 > kSfMaxDegree + 1) return cudaErrorInvalidValue;
    // enough blocks to fill the chip several times; a block keeps its table for all its groups
    const int64_t gx = (F + kSfThreads - 1) / kSfThreads;
    int64_t gy = (16 * 152 + gx - 1) / gx;
    gy = gy < groups ? gy : groups;
    const dim3 grid((unsigned)gx, (unsigned)(gy < 65535 ? gy : 65535));
    if (in_dtype == UQLB_F64)
        launch_sf(grid, s, static_cast<const double*>(in), in_ld, out, out_ld, groups, jprev, jout, n, p1, oidx, G, F);
    else
        launch_sf(grid, s, static_cast<const float*>(in), in_ld, out, out_ld, groups, jprev, jout, n, p1, oidx, G, F);
    return cudaGetLastError();
}

cudaError_t launch_project(const double* W, int K, int S, const void* M, int dtype, int64_t F, int64_t ld,
                           double* C, cudaStream_t s) {
    if (F <= 0 || K <= 0) return cudaSuccess;
    if (dtype == UQLB_F64)
        launch_dense_any(W, K, S, static_cast<const double*>(M), F, ld, C, s);
    else
        launch_dense_any(W, K, S, static_cast<const float*>(M), F, ld, C, s);
    return cudaGetLastError();
}

// Over reflected samples or dense.  Few fields leave SMs idle under either, and a call is then a chain: 0.70 us
// per orbit and 0.086 per term (its sum lies in shared memory) against 0.56 per sample for blocks of six
// terms (fit of 14 sparse grids, one field, to 3 us).  On many terms per sample the dense chain is the shorter
// one: 69 samples x 84 terms, 129 fields 114 us over reflected samples, 56 dense; 177 x 35 156, 113.
bool reflect_pays(int K, int64_t S, int64_t F, int norbits, int nterms) {
    const int64_t blocks = (F + 2 * kProjThreads - 1) / (2 * kProjThreads) * ((K + 5) / 6);
    return blocks > 152 || 0.70 * norbits + 0.086 * nterms <= 0.56 * (double)S;
}

cudaError_t launch_reflect(const ReflPlanView& p, int K, const void* M, int dtype, int64_t F, int64_t ld, double* C,
                           cudaStream_t s) {
    if (F <= 0 || K <= 0) return cudaSuccess;
    return dtype == UQLB_F64 ? launch_refl(p, K, static_cast<const double*>(M), F, ld, C, s)
                             : launch_refl(p, K, static_cast<const float*>(M), F, ld, C, s);
}

cudaError_t launch_gpc_stats(const double* C, int K, int64_t F, double* mean, double* var, cudaStream_t s) {
    if (F <= 0) return cudaSuccess;
    const int64_t blocks = (F + 255) / 256;
    gpc_stats_kernel<<<(unsigned)(blocks < 65535 * 8 ? blocks : 65535 * 8), 256, 0, s>>>(C, K, F, mean, var);
    return cudaGetLastError();
}

// FP32 fields: one pass or two.  The merge of the warps' sums and the pairs of one pass cost some 60 FP64
// instructions per field whatever S is, the two passes five per value, so few samples of many fields take
// two; few fields do not fill the chip, and there the chains of the two passes are the longer ones.  One
// pass / two passes in us: 131073 fields 4 samples 45 / 28, 12 47 / 39, 16 48 / 46, 20 49 / 52; 524289 fields
// 4 123 / 55, 16 134 / 116, 20 141 / 136, 24 142 / 156; 2097153 fields 12 541 / 319, 24 600 / 548, 32 649 / 702;
// 32769 fields 4 27 / 24, 12 28 / 25, 20 28 / 28; 16385 fields 4 21 / 23, 16 22 / 25.
static bool mc_one_pass(int64_t S, int64_t F) {
    return F < (1 << 15) || S >= (F < (1 << 18) ? 16 : (F < (1 << 20) ? 20 : 28));
}

cudaError_t launch_mc_stats(const void* M, int dtype, int64_t S, int64_t F, int64_t ld, double* mean,
                            double* var, int ddof, cudaStream_t s) {
    if (F <= 0) return cudaSuccess;
    const int64_t blocks = (F + 255) / 256;
    const unsigned g = (unsigned)(blocks < 65535 * 8 ? blocks : 65535 * 8);
    if (dtype == UQLB_F64)
        mc_stats_kernel<double><<<g, 256, 0, s>>>(static_cast<const double*>(M), S, F, ld, mean, var, ddof);
    else if (!mc_one_pass(S, F))
        mc_stats_kernel<float><<<g, 256, 0, s>>>(static_cast<const float*>(M), S, F, ld, mean, var, ddof);
    else
        mc_stats_f32_kernel<<<(unsigned)((F + 31) / 32), dim3(32, kMcWarps), 0, s>>>(static_cast<const float*>(M), S, F, ld,
                                                                                     mean, var, ddof);
    return cudaGetLastError();
}

}  // namespace uqlb

// =========================================================================================
// Projection without allocation.
//
// Some callers cannot allocate device memory at the moment they need statistics: code running
// under a memory budget that forbids new allocations, host threads that must not take the
// allocator's locks, or embeddings that hand over only their own input and output buffers.
// uqlb_project needs a small device scratch for the weight matrix W, which it takes from a
// caller workspace.  This variant keeps W in a file-scope device array instead, so the caller
// passes nothing but the fields and the coefficient buffer and nothing is allocated.
// =========================================================================================

namespace {

// Capacity of the shared weight-matrix scratch: K x S <= 131072 doubles (1 MiB).  Every GPU
// that loads the library holds this array until the process exits.
constexpr int64_t kNoAllocWMax = 1 << 17;
static __device__ __align__(256) double g_noalloc_w[kNoAllocWMax];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double* g_noalloc_ptr[kMaxDevices] = {nullptr};

}  // namespace

extern "C" int uqlb_project_noalloc(uqlb_ctx* ctx, const void* m_dev, int dtype, int64_t n_fields, int64_t m_ld,
                                    double* coeffs_dev, void* stream) {
    using namespace uqlb;
    const double* W = nullptr;
    int K = 0, device = 0;
    int64_t S = 0;
    if (int rc = ctx_projection_view(ctx, &W, &K, &S, &device)) return rc;
    if (!m_dev || !coeffs_dev || n_fields < 0 || m_ld < n_fields)
        return ctx_fail(ctx, UQLB_ERR_ARG, "project_noalloc: bad arguments");
    if (dtype != UQLB_F64 && dtype != UQLB_F32)
        return ctx_fail(ctx, UQLB_ERR_ARG, "project_noalloc: dtype must be F64 or F32");
    if ((int64_t)K * S > kNoAllocWMax) {
        char buf[200];
        snprintf(buf, sizeof buf, "project_noalloc: K x S = %lld exceeds the fixed scratch of %lld weights; use uqlb_project",
                 (long long)K * S, (long long)kNoAllocWMax);
        return ctx_fail(ctx, UQLB_ERR_ARG, buf);
    }
    if (device < 0 || device >= kMaxDevices) return ctx_fail(ctx, UQLB_ERR_ARG, "project_noalloc: device index too large");
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return ctx_fail(ctx, UQLB_ERR_CUDA, cudaGetErrorString(e));
    double* w_dev = nullptr;
    {
        // First call on this device: resolve the device address of the array (host code cannot
        // use the symbol itself, which only stands in for it on the host).  The address is kept for
        // the life of the process; a device reset would invalidate it (documented in the header).
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (g_noalloc_ptr[device] == nullptr) {
            void* ptr = nullptr;
            e = cudaGetSymbolAddress(&ptr, g_noalloc_w);
            if (e != cudaSuccess) return ctx_fail(ctx, UQLB_ERR_CUDA, cudaGetErrorString(e));
            g_noalloc_ptr[device] = static_cast<double*>(ptr);
        }
        w_dev = g_noalloc_ptr[device];
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // W overwrites exactly the K x S entries the kernel reads, so nothing needs clearing.
    e = cudaMemcpyAsync(w_dev, W, (size_t)K * S * sizeof(double), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return ctx_fail(ctx, UQLB_ERR_CUDA, cudaGetErrorString(e));
    e = launch_project(w_dev, K, (int)S, m_dev, dtype, n_fields, m_ld, coeffs_dev, s);
    if (e != cudaSuccess) return ctx_fail(ctx, UQLB_ERR_CUDA, cudaGetErrorString(e));
    return 0;
}
