// Stand-alone integer Softmax / GELU kernels (row- and element-wise, HBM/ALU bound).
#include <climits>
#include <type_traits>

#include "iptq_common.cuh"

namespace iptq {

constexpr unsigned kFull = 0xffffffffu;

// ------------------------------------------------------------------------------------------------
// Softmax: one warp per row, the row lives in registers (NITER values per lane), row max / row sum
// by warp reduction, one fp64 division per row for floor(2^M / sum).
// ------------------------------------------------------------------------------------------------
struct SoftmaxDev {
    ExpDev ex;
    int M, f_shl, p_shr;
    int tab_n;                 // entries of the exponential table, 0: evaluate
    const uint16_t* tab_src;   // the table in device memory, or null: each CTA builds it
};

template <int VARIANT, int NITER, bool HAS_BIAS, bool PSHR>
__global__ void __launch_bounds__(256)
softmax_rows_kernel(const int32_t* __restrict__ scores, uint8_t* __restrict__ probs, int64_t rows, int n,
                    const int32_t* __restrict__ bias, int64_t bias_period, const SoftmaxDev c)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    grid_dep_launch();
    grid_dep_wait();
    for (int64_t row = warp; row < rows; row += nwarps) {
        const int32_t* sr = scores + row * n;
        const int32_t* br = HAS_BIAS ? bias + (row % bias_period) * n : nullptr;
        int v[NITER];
        int mx = INT_MIN;
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            const int j = lane + 32 * k;
            int s = kNoScore;                                  // lanes past the row end
            if (j < n) {
                s = __ldcs(sr + j);
                if (HAS_BIAS) s += __ldg(br + j);
            }
            v[k] = s;
            mx = max(mx, s);
        }
        mx = __reduce_max_sync(kFull, mx);                      // Eq. (6)
        unsigned sum = 0;
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            const unsigned e = exp_core_nd<VARIANT>(exp_distance(mx, v[k]), c.ex);
            v[k] = (int)e;
            sum += e;
        }
        sum = __reduce_add_sync(kFull, sum);
        uint8_t* pr = probs + row * n;
        if (VARIANT == IPTQ_SM_LOG2) {
#pragma unroll
            for (int k = 0; k < NITER; ++k) {
                const int j = lane + 32 * k;
                if (j < n) __stcs(pr + j, (uint8_t)log2_code(sum, (unsigned)v[k]));
            }
            continue;
        }
        const unsigned f = intdiv_factor(sum, c.M) << c.f_shl;  // Eq. (15)
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            const int j = lane + 32 * k;
            unsigned pv = __umulhi(f, (unsigned)v[k]);
            if (PSHR) pv >>= c.p_shr;
            if (j < n) __stcs(pr + j, (uint8_t)pv);
        }
    }
}

// Tabulated form: the integer exponential (Eq. (9), or the second-order polynomial of the other two candidates)
// depends on max - s alone, is 0 beyond a few multiples of x0 and below 2^16, so each CTA keeps it as a table in
// shared memory (copied from the one iptq_softmax_table() wrote, or
// built here with the same arithmetic) and a score costs one 16-bit shared-memory load instead of the evaluation.
// Two CTAs of 1024 threads per SM: 32 registers per thread, 64 warps to cover the load latency.
constexpr int kSmTabThreads = 1024;
constexpr int kSmTabMaxBytes = 2 * IPTQ_SOFTMAX_TABLE_MAX;
// Smallest inputs for which the table pays for its set-up (copied from device memory / built by every CTA).
constexpr int64_t kSmTabMinElemsCopy = 1 << 20, kSmTabMinElemsBuild = 16 << 20;

template <int VARIANT, int NITER, bool HAS_BIAS, bool PSHR>
__global__ void __launch_bounds__(kSmTabThreads, 2)
softmax_rows_tab_kernel(const int32_t* __restrict__ scores, uint8_t* __restrict__ probs, int64_t rows, int n,
                        const int32_t* __restrict__ bias, int64_t bias_period, const SoftmaxDev c, int tab_n,
                        const uint16_t* __restrict__ tab_src)
{
    constexpr int TPB = kSmTabThreads;
    extern __shared__ __align__(16) uint16_t exp_tab[];
    if (tab_src) {
        // Written by iptq_softmax_table() and fenced there, so it may be read ahead of the dependency wait.
        const int4* src = reinterpret_cast<const int4*>(tab_src);
        int4* dst = reinterpret_cast<int4*>(exp_tab);
        for (int i = threadIdx.x; i < (tab_n + 8) / 8; i += TPB) dst[i] = __ldg(src + i);
    } else {
        for (int d = threadIdx.x; d <= tab_n; d += TPB)
            exp_tab[d] = d < tab_n ? (uint16_t)exp_core_nd<VARIANT>(-d, c.ex) : (uint16_t)0;
    }
    __syncthreads();
    const uint32_t tab_addr = (uint32_t)__cvta_generic_to_shared(exp_tab);
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (TPB >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (TPB >> 5);
    grid_dep_launch();
    grid_dep_wait();
    // Only the last 32-column step of a row can pass the row end.
    const bool tail_ok = lane + 32 * (NITER - 1) < n;
    auto load_row = [&](int64_t row, int (&v)[NITER]) {
        const int32_t* sr = scores + row * n + lane;
        const int32_t* br = HAS_BIAS ? bias + (row % bias_period) * n + lane : nullptr;
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            int s = kNoScore;                                  // lanes past the row end
            if (k < NITER - 1 || tail_ok) {
                s = __ldcs(sr + 32 * k);
                if (HAS_BIAS) s += __ldg(br + 32 * k);
            }
            v[k] = s;
        }
    };
    auto finish_row = [&](int64_t row, int (&v)[NITER]) {
        int mx = INT_MIN;
#pragma unroll
        for (int k = 0; k < NITER; ++k) mx = max(mx, v[k]);
        mx = __reduce_max_sync(kFull, mx);                      // Eq. (6)
        unsigned sum = 0;
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            const unsigned d = min((unsigned)mx - (unsigned)v[k], (unsigned)tab_n);   // exact for any int32 pair
            unsigned e;
            asm volatile("ld.shared.u16 %0, [%1];" : "=r"(e) : "r"(tab_addr + 2u * d));
            v[k] = (int)e;
            sum += e;
        }
        sum = __reduce_add_sync(kFull, sum);
        uint8_t* pr = probs + row * n + lane;
        if constexpr (VARIANT == IPTQ_SM_LOG2) {
#pragma unroll
            for (int k = 0; k < NITER; ++k)
                if (k < NITER - 1 || tail_ok) __stcs(pr + 32 * k, (uint8_t)log2_code(sum, (unsigned)v[k]));
            return;
        }
        const unsigned f = intdiv_factor(sum, c.M) << c.f_shl;  // Eq. (15)
#pragma unroll
        for (int k = 0; k < NITER; ++k) {
            unsigned pv = __umulhi(f, (unsigned)v[k]);
            if (PSHR) pv >>= c.p_shr;
            if (k < NITER - 1 || tail_ok) __stcs(pr + 32 * k, (uint8_t)pv);
        }
    };
    int v[NITER];
    for (int64_t row = warp; row < rows; row += nwarps) {
        load_row(row, v);
        finish_row(row, v);
    }
}

template <int VARIANT, int NITER>
static int launch_softmax2(const int32_t* s, uint8_t* p, int64_t rows, int n, const int32_t* bias, int64_t period,
                           const SoftmaxDev& c, cudaStream_t st)
{
    if constexpr (NITER <= 8)
    if (c.tab_n > 0 && ((c.tab_n + 8) & ~7) <= IPTQ_SOFTMAX_TABLE_MAX &&
        rows * n >= (c.tab_src ? kSmTabMinElemsCopy : kSmTabMinElemsBuild)) {
        // Tabulated exponential: worth the per-CTA table set-up once every warp has several rows.
        const size_t smem = (2 * ((size_t)c.tab_n + 1) + 15) & ~(size_t)15;
        const int wpc = kSmTabThreads / 32;
        const int grid = (int)std::min<int64_t>((rows + wpc - 1) / wpc, (int64_t)sm_count() * 2);
#define IPTQ_SM_TAB(HB, PS)                                                                                         \
        do {                                                                                                        \
            auto kern = softmax_rows_tab_kernel<VARIANT, NITER, HB, PS>;                                            \
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmTabMaxBytes);              \
            launch_kernel(kern, grid, kSmTabThreads, smem, st, s, p, rows, n, bias, period, c, c.tab_n, c.tab_src); \
        } while (0)
        if (bias) { if (c.p_shr) IPTQ_SM_TAB(true, true); else IPTQ_SM_TAB(true, false); }
        else      { if (c.p_shr) IPTQ_SM_TAB(false, true); else IPTQ_SM_TAB(false, false); }
#undef IPTQ_SM_TAB
        note_launch();
        return last_launch_status();
    }
    const int threads = 256;
    const int64_t want = (rows + 7) / 8;
    const int grid = (int)std::min<int64_t>(want, (int64_t)sm_count() * 8);
    if (bias) {
        if (c.p_shr) launch_kernel(softmax_rows_kernel<VARIANT, NITER, true, true>, grid, threads, 0, st, s, p, rows, n, bias, period, c);
        else         launch_kernel(softmax_rows_kernel<VARIANT, NITER, true, false>, grid, threads, 0, st, s, p, rows, n, bias, period, c);
    } else {
        if (c.p_shr) launch_kernel(softmax_rows_kernel<VARIANT, NITER, false, true>, grid, threads, 0, st, s, p, rows, n, bias, period, c);
        else         launch_kernel(softmax_rows_kernel<VARIANT, NITER, false, false>, grid, threads, 0, st, s, p, rows, n, bias, period, c);
    }
    note_launch();
    return last_launch_status();
}

template <int VARIANT>
static int launch_softmax1(const int32_t* s, uint8_t* p, int64_t rows, int n, const int32_t* bias, int64_t period,
                           const SoftmaxDev& c, cudaStream_t st)
{
    const int it = (n + 31) / 32;
    switch (it) {
        case 1: return launch_softmax2<VARIANT, 1>(s, p, rows, n, bias, period, c, st);
        case 2: return launch_softmax2<VARIANT, 2>(s, p, rows, n, bias, period, c, st);
        case 3: return launch_softmax2<VARIANT, 3>(s, p, rows, n, bias, period, c, st);
        case 4: return launch_softmax2<VARIANT, 4>(s, p, rows, n, bias, period, c, st);
        case 5: return launch_softmax2<VARIANT, 5>(s, p, rows, n, bias, period, c, st);
        case 6: return launch_softmax2<VARIANT, 6>(s, p, rows, n, bias, period, c, st);
        case 7: return launch_softmax2<VARIANT, 7>(s, p, rows, n, bias, period, c, st);
        case 8: return launch_softmax2<VARIANT, 8>(s, p, rows, n, bias, period, c, st);
        default:
            if (it <= 16) return launch_softmax2<VARIANT, 16>(s, p, rows, n, bias, period, c, st);
            return launch_softmax2<VARIANT, 32>(s, p, rows, n, bias, period, c, st);
    }
}

// ------------------------------------------------------------------------------------------------
// GELU: element-wise; each warp iteration covers 512 elements with four coalesced 16-byte loads per
// lane and four coalesced 4-byte stores.
// ------------------------------------------------------------------------------------------------
template <int VARIANT, bool SAT8>
__device__ __forceinline__ unsigned gelu4(int4 a, const GeluDev& c)
{
    if (SAT8)
        return pack4_sat_s8(requant_nosat(gelu_core<VARIANT>(a.x, c), c.out), requant_nosat(gelu_core<VARIANT>(a.y, c), c.out),
                            requant_nosat(gelu_core<VARIANT>(a.z, c), c.out), requant_nosat(gelu_core<VARIANT>(a.w, c), c.out));
    return pack4_s8(requant_full(gelu_core<VARIANT>(a.x, c), c.out), requant_full(gelu_core<VARIANT>(a.y, c), c.out),
                    requant_full(gelu_core<VARIANT>(a.z, c), c.out), requant_full(gelu_core<VARIANT>(a.w, c), c.out));
}

template <int VARIANT, bool SAT8>
__global__ void __launch_bounds__(256)
gelu_kernel(const int32_t* __restrict__ x, int8_t* __restrict__ y, int64_t n, const GeluDev c)
{
    grid_dep_launch();
    grid_dep_wait();
    const int64_t nvec = n >> 2;                                 // int4 / 4-byte groups
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int4* xv = reinterpret_cast<const int4*>(x);
    unsigned* yv = reinterpret_cast<unsigned*>(y);
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // four independent groups per iteration for memory-level parallelism
    for (; i + 3 * stride < nvec; i += 4 * stride) {
        int4 a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = __ldcs(xv + i + u * stride);
#pragma unroll
        for (int u = 0; u < 4; ++u) __stcs(yv + i + u * stride, gelu4<VARIANT, SAT8>(a[u], c));
    }
    for (; i < nvec; i += stride) yv[i] = gelu4<VARIANT, SAT8>(__ldcs(xv + i), c);
    // ragged tail (n % 4 elements)
    const int64_t t = (nvec << 2) + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) y[t] = (int8_t)requant_full(gelu_core<VARIANT>(x[t], c), c.out);
}

// Tabulated form: with consts->table set (iptq_gelu_table) the whole function is a 64 KB table, copied once per CTA
// into shared memory; an element then costs a clamp to 16 bits and one byte load.  Two CTAs of 1024 threads per SM.
constexpr int kGeluTabThreads = 1024;

__global__ void __launch_bounds__(kGeluTabThreads, 2)
gelu_tab_kernel(const int32_t* __restrict__ x, int8_t* __restrict__ y, int64_t n, const int8_t* __restrict__ table)
{
    extern __shared__ __align__(16) int8_t gelu_tab[];
    {
        // written and fenced by iptq_gelu_table(): safe to read ahead of the dependency wait
        const int4* src = reinterpret_cast<const int4*>(table);
        int4* dst = reinterpret_cast<int4*>(gelu_tab);
        for (int i = threadIdx.x; i < IPTQ_GELU_TABLE_SIZE / 16; i += kGeluTabThreads) dst[i] = __ldg(src + i);
    }
    __syncthreads();
    const uint32_t mid = (uint32_t)__cvta_generic_to_shared(gelu_tab) + 32768u;      // address of table[0 + 32768]
    grid_dep_launch();
    grid_dep_wait();
    auto look = [&](int v) -> int {
        v = max(-32768, min(32767, v));
        int r;
        asm volatile("ld.shared.s8 %0, [%1];" : "=r"(r) : "r"(mid + (uint32_t)v));
        return r;
    };
    auto four = [&](int4 a) -> unsigned { return pack4_sat_s8(look(a.x), look(a.y), look(a.z), look(a.w)); };
    const int64_t nvec = n >> 2;
    const int64_t stride = (int64_t)gridDim.x * kGeluTabThreads;
    const int4* xv = reinterpret_cast<const int4*>(x);
    unsigned* yv = reinterpret_cast<unsigned*>(y);
    int64_t i = (int64_t)blockIdx.x * kGeluTabThreads + threadIdx.x;
    for (; i + 3 * stride < nvec; i += 4 * stride) {
        int4 a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = __ldcs(xv + i + u * stride);
#pragma unroll
        for (int u = 0; u < 4; ++u) __stcs(yv + i + u * stride, four(a[u]));
    }
    for (; i < nvec; i += stride) yv[i] = four(__ldcs(xv + i));
    const int64_t t = (nvec << 2) + (int64_t)blockIdx.x * kGeluTabThreads + threadIdx.x;
    if (t < n) y[t] = (int8_t)look(x[t]);
}

// table[x + 32768] = integer GELU of x for every 16-bit x (the input clamp to in_bits is part of gelu_core)
template <int VARIANT>
__global__ void __launch_bounds__(256)
gelu_table_kernel(int8_t* __restrict__ table, const GeluDev c)
{
    grid_dep_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    table[i] = (int8_t)requant_full(gelu_core<VARIANT>(i - 32768, c), c.out);
}

// table[d] = integer exponential of -d for d < n, 0 for n <= d < n_pad
template <int VARIANT>
__global__ void __launch_bounds__(256)
softmax_table_kernel(uint16_t* __restrict__ table, int n, int n_pad, const ExpDev ex)
{
    grid_dep_wait();
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d < n_pad) table[d] = d < n ? (uint16_t)exp_core_nd<VARIANT>(-d, ex) : (uint16_t)0;
}

// Launched without programmatic serialisation behind a table kernel: it starts only once the table is complete
// and visible, so a later kernel that reads the table ahead of its own dependency wait cannot overtake the writer.
__global__ void stream_fence_kernel() {}

}  // namespace iptq

using namespace iptq;

extern "C" {

int iptq_softmax(const int32_t* scores, uint8_t* probs, int64_t rows, int row_len, const int32_t* bias,
                 int64_t bias_period, const iptq_softmax_consts* consts, iptq_stream_t stream)
{
    if (!consts) return IPTQ_ERR_NULL;
    if (rows < 0 || row_len < 1 || row_len > 1024 || row_len != consts->row_len) return IPTQ_ERR_SHAPE;
    if (rows == 0) return IPTQ_OK;                      // empty input: nothing to read or write
    if (!scores || !probs) return IPTQ_ERR_NULL;
    if (bias && bias_period < 1) return IPTQ_ERR_SHAPE;
    if (!aligned16(scores) || !aligned16(probs) || (bias && !aligned16(bias))) return IPTQ_ERR_ALIGN;
    if (consts->out_bits < 4 || consts->out_bits > 8) return IPTQ_ERR_BITS;
    if (consts->x0 < 8 || consts->M < 31 || consts->M > 40) return IPTQ_ERR_SCALE_RANGE;
    if (rows == 0) return IPTQ_OK;
    SoftmaxDev c;
    c.ex = to_dev_exp(*consts);
    c.M = consts->M; c.f_shl = consts->f_shl; c.p_shr = consts->p_shr;
    c.tab_n = exp_table_entries(*consts);
    c.tab_src = (consts->table && consts->table_n == c.tab_n) ? consts->table : nullptr;
    switch (consts->variant) {
        case IPTQ_SM_BITEXP: return launch_softmax1<IPTQ_SM_BITEXP>(scores, probs, rows, row_len, bias, bias_period, c, stream);
        case IPTQ_SM_SHIFTMAX: return launch_softmax1<IPTQ_SM_SHIFTMAX>(scores, probs, rows, row_len, bias, bias_period, c, stream);
        case IPTQ_SM_POLY: return launch_softmax1<IPTQ_SM_POLY>(scores, probs, rows, row_len, bias, bias_period, c, stream);
        case IPTQ_SM_LOG2: return launch_softmax1<IPTQ_SM_LOG2>(scores, probs, rows, row_len, bias, bias_period, c, stream);
        default: return IPTQ_ERR_VARIANT;
    }
}

int iptq_gelu(const int32_t* x, int8_t* y, int64_t n, const iptq_gelu_consts* consts, iptq_stream_t stream)
{
    if (!consts) return IPTQ_ERR_NULL;
    if (n < 0) return IPTQ_ERR_SHAPE;
    if (n == 0) return IPTQ_OK;
    if (!x || !y) return IPTQ_ERR_NULL;
    if (!aligned16(x) || !aligned16(y)) return IPTQ_ERR_ALIGN;
    if (consts->in_bits < 8 || consts->in_bits > 16) return IPTQ_ERR_BITS;
    int rc = check_requant(&consts->out);
    if (rc != IPTQ_OK) return rc;
    if (n == 0) return IPTQ_OK;
    if (consts->table && n >= (1 << 20)) {
        // tabulated: worth the 64 KB copy per CTA once every thread has a few vectors
        if (!aligned16(consts->table)) return IPTQ_ERR_ALIGN;
        const int64_t vecs = (n + 3) / 4;
        const int grid = (int)std::min<int64_t>((vecs + kGeluTabThreads - 1) / kGeluTabThreads, (int64_t)sm_count() * 2);
        cudaFuncSetAttribute(gelu_tab_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, IPTQ_GELU_TABLE_SIZE);
        launch_kernel(gelu_tab_kernel, grid, kGeluTabThreads, IPTQ_GELU_TABLE_SIZE, stream, x, y, n, consts->table);
        note_launch();
        return last_launch_status();
    }
    const GeluDev c = to_dev(*consts);
    const int threads = 256;
    const int64_t groups = (n + 3) / 4;
    const int grid = (int)std::min<int64_t>((groups + threads - 1) / threads, (int64_t)sm_count() * 16);
    const bool sat8 = consts->out.qmin == -128 && consts->out.qmax == 127;
#define IPTQ_GELU_LAUNCH(V)                                                               \
    do {                                                                                  \
        if (sat8) launch_kernel(gelu_kernel<V, true>, grid, threads, 0, stream, x, y, n, c);         \
        else      launch_kernel(gelu_kernel<V, false>, grid, threads, 0, stream, x, y, n, c);        \
    } while (0)
    switch (consts->variant) {
        case IPTQ_GELU_POLY4: IPTQ_GELU_LAUNCH(IPTQ_GELU_POLY4); break;
        case IPTQ_GELU_POLY2: IPTQ_GELU_LAUNCH(IPTQ_GELU_POLY2); break;
        case IPTQ_GELU_SHIFT: IPTQ_GELU_LAUNCH(IPTQ_GELU_SHIFT); break;
        default: return IPTQ_ERR_VARIANT;
    }
#undef IPTQ_GELU_LAUNCH
    note_launch();
    return last_launch_status();
}

int iptq_gelu_table(const iptq_gelu_consts* consts, int8_t* table, iptq_stream_t stream)
{
    if (!consts || !table) return IPTQ_ERR_NULL;
    if (!aligned16(table)) return IPTQ_ERR_ALIGN;
    if (consts->in_bits < 8 || consts->in_bits > 16) return IPTQ_ERR_BITS;
    int rc = check_requant(&consts->out);
    if (rc != IPTQ_OK) return rc;
    const GeluDev c = to_dev(*consts);
    const int threads = 256, grid = IPTQ_GELU_TABLE_SIZE / threads;
    switch (consts->variant) {
        case IPTQ_GELU_POLY4: launch_kernel(gelu_table_kernel<IPTQ_GELU_POLY4>, grid, threads, 0, stream, table, c); break;
        case IPTQ_GELU_POLY2: launch_kernel(gelu_table_kernel<IPTQ_GELU_POLY2>, grid, threads, 0, stream, table, c); break;
        case IPTQ_GELU_SHIFT: launch_kernel(gelu_table_kernel<IPTQ_GELU_SHIFT>, grid, threads, 0, stream, table, c); break;
        default: return IPTQ_ERR_VARIANT;
    }
    stream_fence_kernel<<<1, 32, 0, stream>>>();
    note_launch();
    return last_launch_status();
}

int iptq_softmax_table(iptq_softmax_consts* consts, uint16_t* table, int32_t capacity, iptq_stream_t stream)
{
    if (!consts) return IPTQ_ERR_NULL;
    consts->table = nullptr;
    consts->table_n = 0;
    const int n = exp_table_entries(*consts);
    const int n_pad = (n + 8) & ~7;                     // at least one zero behind the last entry
    if (n == 0 || n_pad > IPTQ_SOFTMAX_TABLE_MAX) return IPTQ_OK;
    if (!table) return IPTQ_ERR_NULL;
    if (!aligned16(table)) return IPTQ_ERR_ALIGN;
    if (capacity < n_pad) return IPTQ_ERR_SHAPE;
    const ExpDev ex = to_dev_exp(*consts);
    const int threads = 256, grid = (n_pad + threads - 1) / threads;
    if (consts->variant == IPTQ_SM_BITEXP)        launch_kernel(softmax_table_kernel<IPTQ_SM_BITEXP>, grid, threads, 0, stream, table, n, n_pad, ex);
    else if (consts->variant == IPTQ_SM_SHIFTMAX) launch_kernel(softmax_table_kernel<IPTQ_SM_SHIFTMAX>, grid, threads, 0, stream, table, n, n_pad, ex);
    else                                          launch_kernel(softmax_table_kernel<IPTQ_SM_POLY>, grid, threads, 0, stream, table, n, n_pad, ex);   // also behind the logarithm candidate
    stream_fence_kernel<<<1, 32, 0, stream>>>();
    note_launch();
    const int rc = last_launch_status();
    if (rc == IPTQ_OK) { consts->table = table; consts->table_n = n; }
    return rc;
}

}  // extern "C"
