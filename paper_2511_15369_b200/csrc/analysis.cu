// Unified-Metric analysis of one layer (Sec. 3.5): every candidate function of the layer and the float layer in one pass
// over its calibration activations, reduced to (sum X^2, sum (X - Q)^2) per candidate.
//
// One launch per layer.  Launched as the candidates' own kernels followed by iptq_metric_*() -- four launches per
// candidate, the integer output written and read again, the float layer (fp64 exp or erf) evaluated once per
// candidate -- the 159 evaluations of a DeiT-Small encoder at batch 8 kept the device busy for 3.5 ms and the host for
// 9.7 ms.  Here the activations are read once, the float layer is evaluated once and the candidates run in registers on
// the device functions of the deployed kernels, so their integers are the same.
#include <climits>
#include <cmath>
#include <cstring>

#include "iptq_common.cuh"

namespace iptq {

constexpr unsigned kAllLanes = 0xffffffffu;
constexpr int kAnThreads = 256;
constexpr int kAnMaxCand = IPTQ_ANALYZE_MAX_CANDIDATES;
// scratch: the counter (256 bytes), the CTAs' pairs, the GELU terms.  The scratch is 16-byte aligned and a term is read with
// one 32-byte load, so the terms start at the 32-byte boundary at or below kAnPartialBytes; the pairs end 32 bytes ahead of it.
constexpr int kAnPartialBytes = 131072;
constexpr int kAnMaxBlocks = (kAnPartialBytes - 256 - 32) / (16 * kAnMaxCand);

__device__ __forceinline__ double an_warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kAllLanes, v, o);
    return v;
}

// An int32 as a double without the conversion unit: 2^52 + 2^31 + v in the bits, both offsets subtracted.
__device__ __forceinline__ double an_to_double(int v)
{
    return __hiloint2double(0x43300000, v ^ (int)0x80000000) - 4503601774854144.0;
}

// Adds the CTAs' pairs (x2[i], e2[i]), i < n, in an order that depends on the launch alone: lanes by butterfly, warps and
// CTAs in index order.  The CTA that finishes last does the final sum and leaves the counter at zero.
template <int THREADS = kAnThreads>
__device__ __forceinline__ void an_finish(const double (&x2)[kAnMaxCand], const double (&e2)[kAnMaxCand], int n, double* sums,
                                          unsigned* counter, double* partials)
{
    __shared__ double sh[2 * kAnMaxCand][THREADS / 32];
    __shared__ bool last;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < kAnMaxCand; ++i) {
        if (i < n) {
            const double a = an_warp_sum(x2[i]), b = an_warp_sum(e2[i]);
            if (lane == 0) { sh[2 * i][w] = a; sh[2 * i + 1][w] = b; }
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 * n) {
        double t = 0.0;
#pragma unroll
        for (int i = 0; i < THREADS / 32; ++i) t += sh[threadIdx.x][i];
        partials[(size_t)blockIdx.x * 2 * kAnMaxCand + threadIdx.x] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int i = w; i < 2 * n; i += THREADS / 32) {
        double t = 0.0;
        // eight reads in flight: one after the other they were the length of a small layer's whole row loop
        for (int b0 = lane; b0 < (int)gridDim.x; b0 += 256) {
            double q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                q[k] = b0 + 32 * k < (int)gridDim.x ? __ldcg(partials + (size_t)(b0 + 32 * k) * 2 * kAnMaxCand + i) : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k) t += q[k];
        }
        t = an_warp_sum(t);
        if (lane == 0) sums[i] = t;
    }
    if (threadIdx.x == 0) *counter = 0;
}

// ------------------------------------------------------------------------------------------------ Softmax
struct AnSoftmaxCand {
    ExpDev ex;
    int variant, M, f_shl, p_shr;
    double step;                       // value of one unit of the output byte (linear candidates)
};
struct AnSoftmax {
    AnSoftmaxCand c[kAnMaxCand];
};

template <int VARIANT, int NITER>
__device__ __forceinline__ double an_softmax_err(const AnSoftmaxCand& c, const int (&v)[NITER], const double (&X)[NITER], int mx)
{
    unsigned e[NITER];
    unsigned sum = 0;
#pragma unroll
    for (int k = 0; k < NITER; ++k) {
        e[k] = exp_core_nd<VARIANT>(exp_distance(mx, v[k]), c.ex);       // 0 for lanes past the row end
        sum += e[k];
    }
    sum = __reduce_add_sync(kAllLanes, sum);
    const unsigned f = VARIANT == IPTQ_SM_LOG2 ? 0u : intdiv_factor(sum, c.M) << c.f_shl;
    double err = 0.0;
#pragma unroll
    for (int k = 0; k < NITER; ++k) {
        double q;
        if (VARIANT == IPTQ_SM_LOG2) {
            const unsigned code = log2_code(sum, e[k]);
            q = code == IPTQ_LOG2_ZERO ? 0.0 : __hiloint2double((int)(1023u - code) << 20, 0);
        } else {
            q = an_to_double((int)(__umulhi(f, e[k]) >> c.p_shr)) * c.step;
        }
        const double d = X[k] - q;
        err = fma(d, d, err);
    }
    return err;
}

// exp(-d S) of an integer distance d >= 0 as the product of two tabulated exponentials, exp(-(d >> k) 2^k S) exp(-(d mod 2^k) S):
// two shared-memory reads and a multiply instead of some fifty fp64 instructions.  Each argument is rounded to 2^-53 of at most 70, each
// exp() is off by a unit in its last place and the product is rounded once more: below 2e-14 relative.  The tables cover d S < kAnExpRange, beyond which the exponential is below 1e-30 and counts as 0.
constexpr double kAnExpRange = 70.0;
constexpr int kAnExpMaxEntries = 4096;
struct AnExp {
    int shift, n_hi;                   // n_hi = 0: no tables (scales below about 1e-5), exp() per element
};
static AnExp an_exp(double in_scale)
{
    AnExp t{0, 0};
    const double n = kAnExpRange / in_scale + 1.0;
    while (t.shift < 30 && (double)(1 << t.shift) * (double)(1 << t.shift) < n) ++t.shift;
    const double hi = n / (double)(1 << t.shift) + 1.0;
    if (hi + (double)(1 << t.shift) <= (double)kAnExpMaxEntries) t.n_hi = (int)hi;
    return t;
}

// A warp per row, the row and its float Softmax in registers.  One CTA per SM, as many warps as the registers of NITER allow: the
// exponential tables (a thousand exp()) are built once per SM, and the launch is one wave (four CTAs of eight warps, of which
// three fitted an SM: 22.6 us per layer of 9456 x 197, 18.5 now).  Rows go round the CTAs first, so that few rows use all SMs.
template <int NITER>
constexpr int kAnSoftmaxThreads = NITER <= 7 ? 768 : NITER <= 16 ? 512 : 256;

template <int NITER>
__global__ void __launch_bounds__(kAnSoftmaxThreads<NITER>, 1)
analyze_softmax_kernel(const int32_t* __restrict__ scores, int64_t rows, int n, double in_scale, const __grid_constant__ AnSoftmax a,
                       int n_cand, const AnExp et, double* __restrict__ sums, unsigned* __restrict__ counter,
                       double* __restrict__ partials)
{
    extern __shared__ __align__(16) double exp_lo[];                     // 2^shift low entries, then n_hi high ones
    double* exp_hi = exp_lo + (1 << et.shift);
    grid_dep_launch();
    constexpr int T = kAnSoftmaxThreads<NITER>;
    if (et.n_hi) {
        for (int i = threadIdx.x; i < 1 << et.shift; i += T) exp_lo[i] = exp(-(double)i * in_scale);
        for (int i = threadIdx.x; i < et.n_hi; i += T) exp_hi[i] = exp(-((double)i * (double)(1 << et.shift)) * in_scale);
        __syncthreads();
    }
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    const int64_t nwarps = (int64_t)gridDim.x * (T >> 5);
    const int iters = (n + 31) >> 5;                                     // <= NITER
    double x2 = 0.0, e2[kAnMaxCand] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t row = warp; row < rows; row += nwarps) {
        const int32_t* sr = scores + row * n + lane;
        int v[NITER];
        int mx = INT_MIN;
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            v[k] = lane + 32 * k < n ? __ldg(sr + 32 * k) : kNoScore;
            mx = max(mx, v[k]);
        }
        mx = __reduce_max_sync(kAllLanes, mx);
        const double zmax = (double)mx * in_scale;
        double X[NITER];
        double den = 0.0;
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            X[k] = 0.0;
            if (k < iters) {                                             // uniform
                if (et.n_hi) {
                    // kNoScore is at a distance of 2^30 and more from every maximum: past the tables' range
                    const unsigned d = (unsigned)mx - (unsigned)v[k];
                    if ((d >> et.shift) < (unsigned)et.n_hi) X[k] = exp_hi[d >> et.shift] * exp_lo[d & ((1u << et.shift) - 1u)];
                } else if (lane + 32 * k < n) {
                    X[k] = exp(fma(an_to_double(v[k]), in_scale, -zmax));
                }
                den += X[k];
            }
        }
        const double inv = 1.0 / an_warp_sum(den);
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            X[k] *= inv;
            x2 = fma(X[k], X[k], x2);
        }
        // every element past the row end has X = 0 and an integer probability of 0, except a logarithm code of such a lane,
        // which is IPTQ_LOG2_ZERO = probability 0 as well
        for (int i = 0; i < n_cand; ++i) {
            const AnSoftmaxCand& c = a.c[i];
            double err;
            switch (c.variant) {
                case IPTQ_SM_BITEXP: err = an_softmax_err<IPTQ_SM_BITEXP, NITER>(c, v, X, mx); break;
                case IPTQ_SM_SHIFTMAX: err = an_softmax_err<IPTQ_SM_SHIFTMAX, NITER>(c, v, X, mx); break;
                case IPTQ_SM_POLY: err = an_softmax_err<IPTQ_SM_POLY, NITER>(c, v, X, mx); break;
                default: err = an_softmax_err<IPTQ_SM_LOG2, NITER>(c, v, X, mx); break;
            }
#pragma unroll
            for (int j = 0; j < kAnMaxCand; ++j) e2[j] += j == i ? err : 0.0;
        }
    }
    const double xs[kAnMaxCand] = {x2, x2, x2, x2};
    an_finish<T>(xs, e2, n_cand, sums, counter, partials);
}

// ------------------------------------------------------------------------------------------------ GELU
struct AnGelu {
    GeluDev c[kAnMaxCand];
};

__device__ __forceinline__ int an_gelu(int x, const GeluDev& c)
{
    switch (c.variant) {
        case IPTQ_GELU_POLY4: return requant_full(gelu_core<IPTQ_GELU_POLY4>(x, c), c.out);
        case IPTQ_GELU_POLY2: return requant_full(gelu_core<IPTQ_GELU_POLY2>(x, c), c.out);
        default: return requant_full(gelu_core<IPTQ_GELU_SHIFT>(x, c), c.out);
    }
}

// What an input code contributes to every sum: X^2 and (X - Q_i)^2.
struct AnGeluTerm {
    double x2, e2[3];
};
static_assert(sizeof(AnGeluTerm) == 32, "one 32-byte sector per code");

// A term of the table that the launch before has written: volatile and a memory operation to the compiler, so that it stays behind
// the dependency wait and behind the test for a table and the code's range.
__device__ __forceinline__ AnGeluTerm an_load_term(const AnGeluTerm* p)
{
    AnGeluTerm t;
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(t.x2), "=d"(t.e2[0]), "=d"(t.e2[1]), "=d"(t.e2[2]) : "l"(p) : "memory");
    return t;
}

__device__ __forceinline__ AnGeluTerm an_gelu_term(int x, double in_scale, double out_scale, int out_zp, const AnGelu& a, int n_cand)
{
    const double v = an_to_double(x) * in_scale;
    const double X = 0.5 * v * (1.0 + erf(v * 0.70710678118654752440));
    AnGeluTerm t;
    t.x2 = X * X;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        t.e2[i] = 0.0;
        if (i < n_cand) {
            const double d = X - an_to_double(an_gelu(x, a.c[i]) - out_zp) * out_scale;
            t.e2[i] = d * d;
        }
    }
    return t;
}

// Layers of kAnGeluTableMin elements and more: the terms of all 2^16 codes are tabulated first (2 MB, L2-resident) and an
// element then costs one 32-byte read and four additions instead of an fp64 erf and three integer functions
// (2.4 M elements: 54 us evaluated).  Below, the table would cost more than it saves.  The reads miss L1 line by line; from
// kAnGeluHistMin on a CTA counts its elements' codes in shared memory and then adds the terms of every code it has seen
// times its count, so the table is read once per CTA and not once per element.  Per layer, terms read / counted, codes spread
// over the whole range: 1 M elements 18.3 / 21.9 us, 2.4 M 24.9 / 23.0, 8.4 M 47.7 / 28.4, 33.6 M 143 / 87.
constexpr int64_t kAnGeluTableMin = 1 << 18, kAnGeluHistMin = 1 << 21;
constexpr int kAnHistThreads = 1024, kAnHistBytes = 2 * 65536;             // 16-bit counters: 128 KB, one CTA per SM
constexpr int kAnHistSteps = 15;                                         // 16-byte reads per thread between two emptyings:
static_assert(4 * kAnHistThreads * kAnHistSteps < 65536, "a counter holds what lies between two emptyings");

__global__ void __launch_bounds__(kAnThreads)
analyze_gelu_terms_kernel(AnGeluTerm* __restrict__ table, double in_scale, double out_scale, int out_zp,
                          const __grid_constant__ AnGelu a, int n_cand)
{
    grid_dep_launch();
    const int i = blockIdx.x * kAnThreads + threadIdx.x;
    const AnGeluTerm t = an_gelu_term(i - 32768, in_scale, out_scale, out_zp, a, n_cand);
    grid_dep_wait();                                                     // the previous layer may still be reading the table
    table[i] = t;
}

__global__ void __launch_bounds__(kAnThreads)
analyze_gelu_kernel(const int32_t* __restrict__ x, int64_t n, double in_scale, double out_scale, int out_zp,
                    const __grid_constant__ AnGelu a, int n_cand, const AnGeluTerm* table, double* __restrict__ sums,
                    unsigned* __restrict__ counter, double* __restrict__ partials)
{
    grid_dep_launch();
    grid_dep_wait();
    double x2 = 0.0, e2[kAnMaxCand] = {0.0, 0.0, 0.0, 0.0};
    auto element = [&](int xi) {
        // one 256-bit load per element, cached in L1: calibration activations fall on a few thousand codes
        const AnGeluTerm t = table && xi >= -32768 && xi < 32768 ? an_load_term(table + 32768 + xi)
                                                                : an_gelu_term(xi, in_scale, out_scale, out_zp, a, n_cand);
        x2 += t.x2; e2[0] += t.e2[0]; e2[1] += t.e2[1]; e2[2] += t.e2[2];
    };
    const int64_t nvec = n >> 2, stride = (int64_t)gridDim.x * kAnThreads, first = (int64_t)blockIdx.x * kAnThreads + threadIdx.x;
    const int4* xv = reinterpret_cast<const int4*>(x);
    for (int64_t i = first; i < nvec; i += stride) {
        const int4 q = __ldg(xv + i);
        element(q.x); element(q.y); element(q.z); element(q.w);
    }
    if ((nvec << 2) + first < n) element(__ldg(x + (nvec << 2) + first));
    const double xs[kAnMaxCand] = {x2, x2, x2, x2};
    an_finish(xs, e2, n_cand, sums, counter, partials);
}

__global__ void __launch_bounds__(kAnHistThreads, 1)
analyze_gelu_hist_kernel(const int32_t* __restrict__ x, int64_t n, double in_scale, double out_scale, int out_zp,
                         const __grid_constant__ AnGelu a, int n_cand, const AnGeluTerm* table, double* __restrict__ sums,
                         unsigned* __restrict__ counter, double* __restrict__ partials)
{
    extern __shared__ __align__(16) unsigned hist[];                     // word w: the counts of codes 2 w - 32768 and 2 w - 32767
    const int tid = threadIdx.x;
    grid_dep_launch();
    for (int i = tid; i < kAnHistBytes / 16; i += kAnHistThreads) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
    __syncthreads();
    grid_dep_wait();
    double x2 = 0.0, e2[kAnMaxCand] = {0.0, 0.0, 0.0, 0.0};
    auto evaluate = [&](int xi) {
        const AnGeluTerm t = an_gelu_term(xi, in_scale, out_scale, out_zp, a, n_cand);
        x2 += t.x2; e2[0] += t.e2[0]; e2[1] += t.e2[1]; e2[2] += t.e2[2];
    };
    auto element = [&](int xi) {
        const unsigned c = (unsigned)xi + 32768u;
        if (c < 65536u) atomicAdd(&hist[c >> 1], c & 1u ? 65536u : 1u);
        else evaluate(xi);
    };
    const int64_t nvec = n >> 2, stride = (int64_t)gridDim.x * kAnHistThreads;
    const int4* xv = reinterpret_cast<const int4*>(x);
    for (int64_t base = (int64_t)blockIdx.x * kAnHistThreads; base < nvec; base += kAnHistSteps * stride) {
        for (int k0 = 0; k0 < kAnHistSteps; k0 += 5) {
            int4 q[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const int64_t i = base + (k0 + k) * stride + tid;
                if (i < nvec) q[k] = __ldg(xv + i);
            }
#pragma unroll
            for (int k = 0; k < 5; ++k)
                if (base + (k0 + k) * stride + tid < nvec) { element(q[k].x); element(q[k].y); element(q[k].z); element(q[k].w); }
        }
        __syncthreads();
        const bool more = base + kAnHistSteps * stride < nvec;
#pragma unroll 4
        for (int w = tid; w < kAnHistBytes / 4; w += kAnHistThreads) {
            const unsigned c = hist[w];
            if (more) hist[w] = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const unsigned m = h ? c >> 16 : c & 0xffffu;
                if (m) {
                    const AnGeluTerm t = an_load_term(table + 2 * w + h);
                    const double f = an_to_double((int)m);
                    x2 = fma(f, t.x2, x2); e2[0] = fma(f, t.e2[0], e2[0]); e2[1] = fma(f, t.e2[1], e2[1]); e2[2] = fma(f, t.e2[2], e2[2]);
                }
            }
        }
        if (more) __syncthreads();
    }
    if (blockIdx.x == 0 && (nvec << 2) + tid < n) evaluate(__ldg(x + (nvec << 2) + tid));
    const double xs[kAnMaxCand] = {x2, x2, x2, x2};
    an_finish<kAnHistThreads>(xs, e2, n_cand, sums, counter, partials);
}

// ------------------------------------------------------------------------------------------------ LayerNorm
struct AnLayerNorm {
    int variant[kAnMaxCand];
    bool same_out[kAnMaxCand];         // reads its input and requantises as the candidate before it
    RequantDev out[kAnMaxCand];
};

// The layer's parameters: by value in the launch up to MAXD channels (a copy to the device in front of every launch would
// cost the stream more than a small layer's kernel); for wider layers in the scratch, where launches that hold them by
// value have put them (a copy from the caller's host memory would be recorded by a stream capture as a pointer to it).
template <int MAXD>
struct AnLnParams {
    float4 gamma[MAXD / 4], beta[MAXD / 4];
    int4 gamma_q[MAXD / 4], beta_q[MAXD / 4];
    __device__ __forceinline__ void get(int i, float4& g, float4& b, int4& gq, int4& bq) const
    {
        g = gamma[i]; b = beta[i]; gq = gamma_q[i]; bq = beta_q[i];
    }
};
template <>
struct AnLnParams<0> {
    const float4 *gamma, *beta;
    const int4 *gamma_q, *beta_q;
    __device__ __forceinline__ void get(int i, float4& g, float4& b, int4& gq, int4& bq) const
    {
        const int4 a = load_act(reinterpret_cast<const int4*>(gamma + i)), c = load_act(reinterpret_cast<const int4*>(beta + i));
        g = make_float4(__int_as_float(a.x), __int_as_float(a.y), __int_as_float(a.z), __int_as_float(a.w));
        b = make_float4(__int_as_float(c.x), __int_as_float(c.y), __int_as_float(c.z), __int_as_float(c.w));
        gq = load_act(gamma_q + i); bq = load_act(beta_q + i);
    }
};
constexpr int kAnLnMaxDim = 3072;
constexpr int kAnLnPart = 1536;                                          // channels per launch: 24 KB of parameters
__global__ void __launch_bounds__(kAnThreads)
analyze_layernorm_params_kernel(const __grid_constant__ AnLnParams<kAnLnPart> prm, int words, int first_word, int4* dst)
{
    grid_dep_launch();
    const AnLnParams<kAnLnPart>* pp = &prm;                              // as in the kernel below
    asm volatile("" : "+l"(pp));
    grid_dep_wait();                                                     // an earlier launch may still be using this part of the scratch
    const int i = blockIdx.x * kAnThreads + threadIdx.x;
    if (i >= words) return;
    float4 g, b;
    int4 gq, bq;
    pp->get(i, g, b, gq, bq);
    int4* d = dst + first_word + i;
    constexpr int W = kAnLnMaxDim / 4;
    d[0] = make_int4(__float_as_int(g.x), __float_as_int(g.y), __float_as_int(g.z), __float_as_int(g.w));
    d[W] = make_int4(__float_as_int(b.x), __float_as_int(b.y), __float_as_int(b.z), __float_as_int(b.w));
    d[2 * W] = gq;
    d[3 * W] = bq;
}
constexpr int kAnLnBytesPerChannel = 24;                                 // shared memory: two doubles, two ints

// A warp per row, under two readings of its input: index 0 plain, 1 with the power-of-two factors.  The row is read twice (the
// second time from L1); the parameters wait in shared memory.  Bound by latency at calibration sizes (a few rows per warp).
template <int MAXD>
__global__ void __launch_bounds__(kAnThreads)
analyze_layernorm_kernel(const int8_t* x, int64_t rows, int D, const __grid_constant__ AnLnParams<MAXD> prm,
                         const uint8_t* __restrict__ ptf, double out_scale, int out_zp, const __grid_constant__ AnLayerNorm a,
                         int n_cand, double* __restrict__ sums, unsigned* __restrict__ counter, double* __restrict__ partials)
{
    extern __shared__ __align__(16) double2 gb[];                        // (gamma, beta) [D], then (gamma_q, beta_q) [D]
    int2* gbq = reinterpret_cast<int2*>(gb + D);
    const int lane = threadIdx.x & 31, words = D >> 2;
    grid_dep_launch();
    if (MAXD == 0) grid_dep_wait();                                      // the launches before this one write the parameters
    // Read through a generic pointer the compiler cannot trace back: as constant-bank loads with an address per lane these
    // reads go one address after the other, each a miss (10 us for 384 channels).
    const AnLnParams<MAXD>* pp = &prm;
    asm volatile("" : "+l"(pp));
    for (int i = threadIdx.x; i < words; i += kAnThreads) {
        float4 g, b;
        int4 gq, bq;
        pp->get(i, g, b, gq, bq);
        gb[4 * i] = make_double2(g.x, b.x); gb[4 * i + 1] = make_double2(g.y, b.y);
        gb[4 * i + 2] = make_double2(g.z, b.z); gb[4 * i + 3] = make_double2(g.w, b.w);
        gbq[4 * i] = make_int2(gq.x, bq.x); gbq[4 * i + 1] = make_int2(gq.y, bq.y);
        gbq[4 * i + 2] = make_int2(gq.z, bq.z); gbq[4 * i + 3] = make_int2(gq.w, bq.w);
    }
    __syncthreads();
    if (MAXD != 0) grid_dep_wait();
    const int64_t warp = (int64_t)blockIdx.x * (kAnThreads >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (kAnThreads >> 5);
    bool any[2] = {false, false};
    for (int i = 0; i < n_cand; ++i) any[a.variant[i] == IPTQ_LN_PTF] = true;
    double x2[2] = {0.0, 0.0}, e2[kAnMaxCand] = {0.0, 0.0, 0.0, 0.0};
    for (int64_t row = warp; row < rows; row += nwarps) {
        const int* xr = reinterpret_cast<const int*>(x + row * D);
        int s1[2] = {0, 0};
        unsigned s2[2] = {0, 0};
        for (int wi = lane; wi < words; wi += 32) {
            const int w = load_act(xr + wi);
            if (any[0]) {
                s1[0] = __dp4a(w, 0x01010101, s1[0]);
                s2[0] = (unsigned)__dp4a(w, w, (int)s2[0]);
            }
            if (any[1]) {
                const unsigned sh = __ldg(reinterpret_cast<const unsigned*>(ptf) + wi);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int xv = ((int)(int8_t)(w >> (8 * t))) << ((sh >> (8 * t)) & 3);
                    s1[1] += xv;
                    s2[1] += (unsigned)(xv * xv);
                }
            }
        }
        double mu[2], inv_sd[2];
        int f4[kAnMaxCand];
        long long F[kAnMaxCand];
        bool same[kAnMaxCand];           // the candidate's integers in this row are those of the candidate before it
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            s1[p] = __reduce_add_sync(kAllLanes, s1[p]);
            s2[p] = __reduce_add_sync(kAllLanes, s2[p]);
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            if (!any[p]) continue;
            const long long V = (long long)D * (long long)s2[p] - (long long)s1[p] * (long long)s1[p];    // D^2 var
            mu[p] = (double)s1[p] / (double)D;
            inv_sd[p] = V > 0 ? (double)D * rsqrt((double)V) : 0.0;      // a constant row gives beta
            const double rt = ln_isqrt((double)V, IPTQ_LN_NEWTON);
            const long long Fn = (long long)ln_reciprocal(rt);
            // the fixed steps of LN_SHIFT can end elsewhere only where V + 1 is a perfect square
            const bool odd = rt > 0.0 && (rt + 1.0) * (rt + 1.0) == (double)V + 1.0;
#pragma unroll
            for (int i = 0; i < kAnMaxCand; ++i) {
                if (i < n_cand && (a.variant[i] == IPTQ_LN_PTF) == (p == 1)) {
                    F[i] = Fn;
                    if (a.variant[i] == IPTQ_LN_SHIFT && odd) {
                        F[i] = (long long)ln_reciprocal(ln_isqrt((double)V, IPTQ_LN_SHIFT));
                    }
                    f4[i] = F[i] < (1ll << 29) ? (int)(F[i] << 2) : 0;   // then (u F) >> 30 = hi32(u 4F)
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kAnMaxCand; ++i)
            same[i] = i > 0 && i < n_cand && a.same_out[i] && F[i] == F[i - 1];
        double er[kAnMaxCand] = {0.0, 0.0, 0.0, 0.0};
        for (int wi = lane; wi < words; wi += 32) {
            const unsigned w = (unsigned)load_act(xr + wi);
            const unsigned sh = any[1] ? __ldg(reinterpret_cast<const unsigned*>(ptf) + wi) : 0u;
            // the four channels side by side under each uniform test: a row is one chain of fp64 latencies otherwise
            int xv[2][4];
            double2 fp[4];
            int2 qp[4];
            double X[2][4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                xv[0][t] = (int)(int8_t)(w >> (8 * t));
                xv[1][t] = xv[0][t] << ((sh >> (8 * t)) & 3);
                fp[t] = gb[4 * wi + t];
                qp[t] = gbq[4 * wi + t];
            }
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (any[p]) {
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        X[p][t] = fma((an_to_double(xv[p][t]) - mu[p]) * inv_sd[p], fp[t].x, fp[t].y);
                        x2[p] = fma(X[p][t], X[p][t], x2[p]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < kAnMaxCand; ++i) {
                if (i < n_cand && !same[i]) {
                    const bool p = a.variant[i] == IPTQ_LN_PTF;
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int u = D * (p ? xv[1][t] : xv[0][t]) - (p ? s1[1] : s1[0]);
                        const int nq = f4[i] ? __mulhi(u, f4[i]) : (int)(((long long)u * F[i]) >> 30);
                        const int o = requant_full(nq * qp[t].x + qp[t].y, a.out[i]);
                        const double d = (p ? X[1][t] : X[0][t]) - an_to_double(o - out_zp) * out_scale;
                        er[i] = fma(d, d, er[i]);
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kAnMaxCand; ++i) {
            if (i > 0 && i < n_cand && same[i]) er[i] = er[i - 1];
            e2[i] += er[i];
        }
    }
    double xs[kAnMaxCand];
#pragma unroll
    for (int i = 0; i < kAnMaxCand; ++i) xs[i] = i < n_cand && a.variant[i] == IPTQ_LN_PTF ? x2[1] : x2[0];
    an_finish(xs, e2, n_cand, sums, counter, partials);
}

static int an_grid(int64_t blocks, int per_sm = 4)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>(blocks, std::min<int64_t>((int64_t)sm_count() * per_sm, kAnMaxBlocks)));
}

static int an_args_ok(const void* consts, int n_cand, const void* sums, const void* work)
{
    if (!consts || !sums || !work) return IPTQ_ERR_NULL;
    if (n_cand < 1 || n_cand > kAnMaxCand) return IPTQ_ERR_SHAPE;
    if (!aligned16(sums) || !aligned16(work)) return IPTQ_ERR_ALIGN;
    return IPTQ_OK;
}

}  // namespace iptq

using namespace iptq;

extern "C" {

int iptq_analyze_softmax(const int32_t* scores, int64_t rows, int row_len, double in_scale, const iptq_softmax_consts* consts,
                         int n_candidates, double* sums, void* work, iptq_stream_t stream)
{
    int rc = an_args_ok(consts, n_candidates, sums, work);
    if (rc != IPTQ_OK) return rc;
    if (rows < 0 || row_len < 1 || row_len > 1024) return IPTQ_ERR_SHAPE;
    if (!(in_scale > 0.0)) return IPTQ_ERR_SCALE_RANGE;
    if (rows > 0 && !scores) return IPTQ_ERR_NULL;
    if (!aligned16(scores)) return IPTQ_ERR_ALIGN;
    AnSoftmax a{};
    for (int i = 0; i < n_candidates; ++i) {
        const iptq_softmax_consts& c = consts[i];
        if (c.row_len != row_len) return IPTQ_ERR_SHAPE;
        if (c.out_bits < 4 || c.out_bits > 8) return IPTQ_ERR_BITS;
        if (c.x0 < 8 || c.M < 31 || c.M > 40) return IPTQ_ERR_SCALE_RANGE;
        if (c.variant < 0 || c.variant > 3) return IPTQ_ERR_VARIANT;
        a.c[i].ex = to_dev_exp(c);
        a.c[i].variant = c.variant; a.c[i].M = c.M; a.c[i].f_shl = c.f_shl; a.c[i].p_shr = c.p_shr;
        a.c[i].step = 1.0 / (double)(1 << (c.out_bits - 1));
    }
    unsigned* counter = static_cast<unsigned*>(work);
    double* partials = reinterpret_cast<double*>(static_cast<uint8_t*>(work) + 256);
    const AnExp et = an_exp(in_scale);
    const int grid = an_grid(rows, 1), it = (row_len + 31) / 32;
#define IPTQ_AN_SM(NI)                                                                                                    \
    launch_kernel(analyze_softmax_kernel<NI>, grid, kAnSoftmaxThreads<NI>, et.n_hi ? 8 * ((size_t)et.n_hi + (1u << et.shift)) : 0, stream, \
                  scores, rows, row_len, in_scale, a, n_candidates, et, sums, counter, partials)
    if (it <= 2) IPTQ_AN_SM(2);
    else if (it <= 4) IPTQ_AN_SM(4);
    else if (it <= 5) IPTQ_AN_SM(5);
    else if (it <= 7) IPTQ_AN_SM(7);
    else if (it <= 8) IPTQ_AN_SM(8);
    else if (it <= 16) IPTQ_AN_SM(16);
    else IPTQ_AN_SM(32);
#undef IPTQ_AN_SM
    note_launch();
    return last_launch_status();
}

int iptq_analyze_gelu(const int32_t* x, int64_t n, double in_scale, double out_scale, int out_zp,
                      const iptq_gelu_consts* consts, int n_candidates, double* sums, void* work, iptq_stream_t stream)
{
    int rc = an_args_ok(consts, n_candidates, sums, work);
    if (rc != IPTQ_OK) return rc;
    if (n < 0 || n_candidates > 3) return IPTQ_ERR_SHAPE;
    if (!(in_scale > 0.0) || !(out_scale > 0.0)) return IPTQ_ERR_SCALE_RANGE;
    if (n > 0 && !x) return IPTQ_ERR_NULL;
    if (!aligned16(x)) return IPTQ_ERR_ALIGN;
    AnGelu a{};
    for (int i = 0; i < n_candidates; ++i) {
        if (consts[i].in_bits < 8 || consts[i].in_bits > 16) return IPTQ_ERR_BITS;
        if (consts[i].variant < 0 || consts[i].variant > 2) return IPTQ_ERR_VARIANT;
        if ((rc = check_requant(&consts[i].out)) != IPTQ_OK) return rc;
        a.c[i] = to_dev(consts[i]);
    }
    unsigned* counter = static_cast<unsigned*>(work);
    double* partials = reinterpret_cast<double*>(static_cast<uint8_t*>(work) + 256);
    AnGeluTerm* table = nullptr;
    if (n >= kAnGeluTableMin) {
        table = reinterpret_cast<AnGeluTerm*>((reinterpret_cast<uintptr_t>(work) + kAnPartialBytes) & ~uintptr_t(31));
        launch_kernel(analyze_gelu_terms_kernel, 65536 / kAnThreads, kAnThreads, 0, stream, table, in_scale, out_scale, out_zp, a,
                      n_candidates);
        note_launch();
    }
    if (n >= kAnGeluHistMin) {
        static bool configured[64];
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return IPTQ_ERR_CUDA;
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(analyze_gelu_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAnHistBytes) != cudaSuccess)
                return IPTQ_ERR_CUDA;
            configured[dev] = true;
        }
        launch_kernel(analyze_gelu_hist_kernel, sm_count(), kAnHistThreads, kAnHistBytes, stream, x, n, in_scale, out_scale, out_zp, a,
                      n_candidates, table, sums, counter, partials);
    } else {
        launch_kernel(analyze_gelu_kernel, an_grid((n / 4 + kAnThreads - 1) / kAnThreads, table ? 6 : 4), kAnThreads, 0, stream, x, n,
                      in_scale, out_scale, out_zp, a, n_candidates, table, sums, counter, partials);
    }
    note_launch();
    return last_launch_status();
}

int iptq_analyze_layernorm(const int8_t* x, int64_t rows, int dim, const float* gamma, const float* beta,
                           const int32_t* gamma_q, const int32_t* beta_q, const uint8_t* ptf_shift, double out_scale,
                           int out_zp, const iptq_ln_consts* consts, int n_candidates, double* sums, void* work,
                           iptq_stream_t stream)
{
    int rc = an_args_ok(consts, n_candidates, sums, work);
    if (rc != IPTQ_OK) return rc;
    if (rows < 0 || dim < 4 || dim > kAnLnMaxDim || (dim & 3)) return IPTQ_ERR_SHAPE;
    if (!(out_scale > 0.0)) return IPTQ_ERR_SCALE_RANGE;
    if (!gamma || !beta || !gamma_q || !beta_q || (rows > 0 && !x)) return IPTQ_ERR_NULL;
    if (!aligned16(x) || (reinterpret_cast<uintptr_t>(ptf_shift) & 3u)) return IPTQ_ERR_ALIGN;
    AnLayerNorm a{};
    for (int i = 0; i < n_candidates; ++i) {
        if (consts[i].dim != dim) return IPTQ_ERR_SHAPE;
        if (consts[i].variant < 0 || consts[i].variant > 2) return IPTQ_ERR_VARIANT;
        if (consts[i].variant == IPTQ_LN_PTF && !ptf_shift) return IPTQ_ERR_NULL;
        if ((rc = check_requant(&consts[i].out)) != IPTQ_OK) return rc;
        a.variant[i] = consts[i].variant;
        a.out[i] = to_dev(consts[i].out);
        a.same_out[i] = i > 0 && (a.variant[i] == IPTQ_LN_PTF) == (a.variant[i - 1] == IPTQ_LN_PTF) &&
                        memcmp(&consts[i].out, &consts[i - 1].out, sizeof(iptq_requant)) == 0;
    }
    unsigned* counter = static_cast<unsigned*>(work);
    double* partials = reinterpret_cast<double*>(static_cast<uint8_t*>(work) + 256);
    const int grid = an_grid((rows + 7) / 8);
    const size_t smem = (size_t)kAnLnBytesPerChannel * dim, bytes = (size_t)dim * 4;
    auto by_value = [&](auto& prm, auto kern) {
        memcpy(prm.gamma, gamma, bytes); memcpy(prm.beta, beta, bytes);
        memcpy(prm.gamma_q, gamma_q, bytes); memcpy(prm.beta_q, beta_q, bytes);
        launch_kernel(kern, grid, kAnThreads, smem, stream, x, rows, dim, prm, ptf_shift, out_scale, out_zp, a, n_candidates, sums,
                      counter, partials);
    };
    if (dim <= 256) {
        AnLnParams<256> prm;
        by_value(prm, analyze_layernorm_kernel<256>);
    } else if (dim <= 512) {
        AnLnParams<512> prm;
        by_value(prm, analyze_layernorm_kernel<512>);
    } else if (dim <= 1024) {
        AnLnParams<1024> prm;
        by_value(prm, analyze_layernorm_kernel<1024>);
    } else {
        // where the GELU terms of another layer would be
        int4* dst = reinterpret_cast<int4*>(static_cast<uint8_t*>(work) + kAnPartialBytes);
        for (int first = 0; first < dim; first += kAnLnPart) {
            const int n = std::min(dim - first, kAnLnPart);
            AnLnParams<kAnLnPart> part;
            memcpy(part.gamma, gamma + first, (size_t)n * 4); memcpy(part.beta, beta + first, (size_t)n * 4);
            memcpy(part.gamma_q, gamma_q + first, (size_t)n * 4); memcpy(part.beta_q, beta_q + first, (size_t)n * 4);
            launch_kernel(analyze_layernorm_params_kernel, (n / 4 + kAnThreads - 1) / kAnThreads, kAnThreads, 0, stream, part, n / 4, first / 4, dst);
            note_launch();
        }
        constexpr int W = kAnLnMaxDim / 4;
        AnLnParams<0> prm{reinterpret_cast<const float4*>(dst), reinterpret_cast<const float4*>(dst + W), dst + 2 * W, dst + 3 * W};
        if (cudaFuncSetAttribute(analyze_layernorm_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAnLnBytesPerChannel * kAnLnMaxDim) != cudaSuccess)
            return IPTQ_ERR_CUDA;
        launch_kernel(analyze_layernorm_kernel<0>, grid, kAnThreads, smem, stream, x, rows, dim, prm, ptf_shift, out_scale, out_zp, a,
                      n_candidates, sums, counter, partials);
    }
    note_launch();
    return last_launch_status();
}

}  // extern "C"
