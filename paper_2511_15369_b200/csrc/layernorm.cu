// Integer LayerNorm (rows of int8 channels): statistics exact in 64 bits, square root and reciprocal as the variants define
// them, normalisation and requantisation in 32-bit fixed point.
#include <algorithm>
#include <type_traits>

#include "iptq_internal.cuh"

namespace iptq {

constexpr unsigned kFull = 0xffffffffu;

struct LnDev {
    int variant, dim;
    RequantDev out;
};

// The rows a LayerNorm reads: row i of x, or, with an index, the concatenation over p < parts of row index[i * parts + p] of a
// tensor whose rows are dim / parts channels (a negative entry: zeros).
struct LnSource {
    const int8_t* x;
    const int32_t* index;
    int parts, part_words;
};

__device__ __forceinline__ int ln_load_word(const LnSource& s, int64_t row, int wi)
{
    if (!s.index) return __ldcs(reinterpret_cast<const int*>(s.x) + row * s.part_words + wi);
    int part = 0;
#pragma unroll
    for (int p = 1; p < 4; ++p)
        if (wi >= s.part_words) { wi -= s.part_words; ++part; }
    const int r = __ldg(s.index + row * s.parts + part);
    return r < 0 ? 0 : load_act(reinterpret_cast<const int*>(s.x) + (int64_t)r * s.part_words + wi);
}

// ---- one row's constants.  n = ((D x - s1) F) >> 30 = hi32(v F) with v = 4 (D x - s1) and F up to 2^40: a high multiply by the
// low word of F with v times its high part as the addend.
struct LnRow {
    int s4, f_lo, f_hi;                // 4 s1; F = f_lo + 2^32 f_hi, f_lo signed
    __device__ __forceinline__ void set(int s1, double F)
    {
        const long long f = (long long)F;
        s4 = 4 * s1;
        f_lo = (int)f;
        f_hi = (int)((f - f_lo) >> 32);
    }
    // xm: input byte times 4 D (times the channel's power-of-two factor)
    template <bool WIDE>
    __device__ __forceinline__ int n(int xm) const
    {
        const int v = xm - s4;
        return WIDE ? mad_hi(v, f_lo, v * f_hi) : __mulhi(v, f_lo);      // not WIDE: F < 2^31, D std > 2^9
    }
};

// Power-of-two factors of a word of four channels: the bytes that have factor 2^j (m.x .. m.w for j = 0..3), the factors as bytes.
__device__ __forceinline__ int4 ln_ptf_masks(unsigned sh)
{
    const unsigned hi = ((sh >> 1) & 0x01010101u) * 255u, lo = (sh & 0x01010101u) * 255u;
    return make_int4((int)(~hi & ~lo), (int)(~hi & lo), (int)(hi & ~lo), (int)(hi & lo));
}
__device__ __forceinline__ int ln_ptf_factors(const int4& m)
{
    return (m.x & 0x01010101) | (m.y & 0x02020202) | (m.z & 0x04040404) | (m.w & 0x08080808);
}
// sum x 2^alpha: the factors as bytes; sum x^2 4^alpha: one sum per alpha over the bytes that have it
struct LnPtfSums {
    int s1 = 0, q0 = 0, q1 = 0, q2 = 0, q3 = 0;
    __device__ __forceinline__ void add(int w, const int4& m, int f)
    {
        s1 = __dp4a(w, f, s1);
        q0 = __dp4a(w & m.x, w, q0); q1 = __dp4a(w & m.y, w, q1);
        q2 = __dp4a(w & m.z, w, q2); q3 = __dp4a(w & m.w, w, q3);
    }
    __device__ __forceinline__ unsigned s2() const { return (unsigned)q0 + 4u * (unsigned)q1 + 16u * (unsigned)q2 + 64u * (unsigned)q3; }
};

// R with the zero point in the rounding constant; SAT8: the pack that follows saturates.
template <bool SAT8>
__device__ __forceinline__ int ln_requant(int y, const RequantDev& out)
{
    const int o = mad_hi(y, out.mult, out.rnd) >> out.shift;
    return SAT8 ? o : max(out.qmin, min(out.qmax, o));
}

// One packed word: normalise, n gamma + beta, R.  d4: 4 D per byte (times its power-of-two factor).
template <bool WIDE, bool SAT8>
__device__ __forceinline__ int ln_word(unsigned w, const int (&d4)[4], const LnRow& r, const int4& g, const int4& b, const RequantDev& out)
{
    return (int)pack4_sat_s8(ln_requant<SAT8>(r.n<WIDE>(sext_byte<0>(w) * d4[0]) * g.x + b.x, out),
                             ln_requant<SAT8>(r.n<WIDE>(sext_byte<1>(w) * d4[1]) * g.y + b.y, out),
                             ln_requant<SAT8>(r.n<WIDE>(sext_byte<2>(w) * d4[2]) * g.z + b.z, out),
                             ln_requant<SAT8>(r.n<WIDE>(sext_byte<3>(w) * d4[3]) * g.w + b.w, out));
}

// CTAs of 256 threads per SM that the compiler has to leave room for: with fewer registers per thread and more warps the kernel was
// faster up to here ([201728, 768]: 86.3 us with 24 warps per SM, 81.0 with 32; [60800, 384]: 18.3 with 32, 17.1 with 40).
constexpr int ln_ctas_per_sm(int words, int rows) { return words <= 2 ? 4 : words <= 4 ? 5 : words * rows <= 24 ? 4 : words * rows <= 32 ? 3 : 2; }

// A warp takes RW rows at a time; they live in registers as packed int8 words (NW per lane).  The per-row scalar work (variance,
// integer square root, reciprocal) is a long dependent chain; lane r of the warp runs it for row r, so its cost is shared by
// RW rows.  The channel parameters are in shared memory and are read once per word for all of them: in registers they
// halved the resident warps.  [201728, 768]: 95.8 -> 81.0 us (3.8 TB/s); [25216, 768] 14.8 -> 13.8; power-of-two factors 181 -> 112.
// Bound by the integer multiplier: two high multiplies and two multiply-adds per element are 12 of its clocks (the same
// launch without R takes 62 us, without any arithmetic 47 us).  Forms of the normalisation with fp64 or packed fp32 FMAs,
// exact as well, were not faster: they need operand pairs whose moves cost what the multiplier saves.
// EXACT: the row is exactly 32 * NW words, so no lane ever needs a bounds predicate.
template <int NW, int RW, bool PTF, bool EXACT, bool SAT8>
__global__ void __launch_bounds__(256, ln_ctas_per_sm(NW, RW))
layernorm_rows_kernel(const LnSource src, int8_t* __restrict__ y, int64_t rows, const int32_t* __restrict__ gamma_q,
                      const int32_t* __restrict__ beta_q, const uint8_t* __restrict__ ptf, const LnDev c)
{
    extern __shared__ __align__(16) int4 ln_prm[];            // gamma_q [words], beta_q [words]
    const int lane = threadIdx.x & 31;
    const int D = c.dim, words = EXACT ? 32 * NW : D >> 2;
    grid_dep_launch();
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t groups = (rows + RW - 1) / RW;
    for (int i = threadIdx.x; i < words; i += 256) {
        ln_prm[i] = __ldg(reinterpret_cast<const int4*>(gamma_q) + i);
        ln_prm[words + i] = __ldg(reinterpret_cast<const int4*>(beta_q) + i);
    }
    __syncthreads();
    const RequantDev out = c.out;
    grid_dep_wait();                                          // gamma / beta above are static; the rows come from the previous kernel
    for (int64_t grp = warp; grp < groups; grp += nwarps) {
        const int64_t row0 = grp * RW, left = rows - row0;
        int w[RW][NW];
        if (src.parts == 1) {
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                int64_t from = row0 + r;
                if (src.index) from = r < left ? __ldg(src.index + from) : -1;
                const bool read = r < left && from >= 0;
                const int* xr = reinterpret_cast<const int*>(src.x + (read ? from : 0) * D);
#pragma unroll
                for (int k = 0; k < NW; ++k) {
                    const int wi = lane + 32 * k;
                    w[r][k] = (read && (EXACT || wi < words)) ? __ldcs(xr + wi) : 0;
                }
            }
        } else {
#pragma unroll
            for (int r = 0; r < RW; ++r)
#pragma unroll
                for (int k = 0; k < NW; ++k) {
                    const int wi = lane + 32 * k;
                    w[r][k] = r < left && wi < words ? ln_load_word(src, row0 + r, wi) : 0;
                }
        }
        int s1[RW];
        unsigned s2[RW];
        if (!PTF) {
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                s1[r] = 0; s2[r] = 0;
#pragma unroll
                for (int k = 0; k < NW; ++k) {
                    s1[r] = __dp4a(w[r][k], 0x01010101, s1[r]);
                    s2[r] = (unsigned)__dp4a(w[r][k], w[r][k], (int)s2[r]);
                }
            }
        } else {
            LnPtfSums q[RW];
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                const int wi = lane + 32 * k;
                const int4 m = ln_ptf_masks(wi < words ? __ldg(reinterpret_cast<const unsigned*>(ptf) + wi) : 0u);
                const int f = ln_ptf_factors(m);
#pragma unroll
                for (int r = 0; r < RW; ++r) q[r].add(w[r][k], m, f);
            }
#pragma unroll
            for (int r = 0; r < RW; ++r) { s1[r] = q[r].s1; s2[r] = q[r].s2(); }
        }
        int my_s1 = 0;
        unsigned my_s2 = 0;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const int a1 = __reduce_add_sync(kFull, s1[r]);
            const unsigned a2 = __reduce_add_sync(kFull, s2[r]);
            if (lane == r) { my_s1 = a1; my_s2 = a2; }
        }
        // lane r: statistics of row r (the other lanes run the same instructions on zeros)
        const double s1d = (double)my_s1;
        const double F = ln_reciprocal(ln_isqrt(fma(-s1d, s1d, (double)D * (double)my_s2), c.variant));   // of D^2 var, exact
        int* yr = reinterpret_cast<int*>(y + row0 * D) + lane;
        LnRow mine;
        mine.set(my_s1, F);
        LnRow row[RW];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            row[r].s4 = __shfl_sync(kFull, mine.s4, r);
            row[r].f_lo = __shfl_sync(kFull, mine.f_lo, r);
            row[r].f_hi = __shfl_sync(kFull, mine.f_hi, r);
        }
        auto emit = [&](auto wide, auto full) {
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                const int wi = lane + 32 * k;
                if (EXACT || wi < words) {
                    const int4 g = ln_prm[wi], b = ln_prm[words + wi];
                    int d4[4] = {4 * D, 4 * D, 4 * D, 4 * D};
                    if (PTF) {
                        const unsigned sh = __ldg(reinterpret_cast<const unsigned*>(ptf) + wi);
#pragma unroll
                        for (int t = 0; t < 4; ++t) d4[t] <<= (sh >> (8 * t)) & 3u;
                    }
#pragma unroll
                    for (int r = 0; r < RW; ++r)
                        if (decltype(full)::value || r < left)
                            __stcs(yr + r * words + 32 * k, ln_word<decltype(wide)::value, SAT8>((unsigned)w[r][k], d4, row[r], g, b, out));
                }
            }
        };
        if (left < RW || __any_sync(kFull, mine.f_hi != 0)) emit(std::true_type{}, std::false_type{});
        else emit(std::false_type{}, std::true_type{});
    }
}

// Output constants whose zero point does not fit into the rounding constant: a warp per row, the row read twice.
template <bool PTF>
__global__ void __launch_bounds__(256)
layernorm_general_kernel(const LnSource src, int8_t* __restrict__ y, int64_t rows, const int32_t* __restrict__ gamma_q,
                         const int32_t* __restrict__ beta_q, const uint8_t* __restrict__ ptf, const LnDev c)
{
    const int lane = threadIdx.x & 31, words = c.dim >> 2;
    grid_dep_launch();
    grid_dep_wait();
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t row = warp; row < rows; row += nwarps) {
        int s1 = 0;
        unsigned s2 = 0;
        for (int wi = lane; wi < words; wi += 32) {
            const int w = ln_load_word(src, row, wi);
            const unsigned sh = PTF ? __ldg(reinterpret_cast<const unsigned*>(ptf) + wi) : 0u;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int xv = ((int)(int8_t)((unsigned)w >> (8 * t))) << ((sh >> (8 * t)) & 3);
                s1 += xv;
                s2 += (unsigned)(xv * xv);
            }
        }
        s1 = __reduce_add_sync(kFull, s1);
        s2 = __reduce_add_sync(kFull, s2);
        const double s1d = (double)s1;
        LnRow r;
        r.set(s1, ln_reciprocal(ln_isqrt(fma(-s1d, s1d, (double)c.dim * (double)s2), c.variant)));
        for (int wi = lane; wi < words; wi += 32) {
            const int w = ln_load_word(src, row, wi);
            const unsigned sh = PTF ? __ldg(reinterpret_cast<const unsigned*>(ptf) + wi) : 0u;
            const int4 g = __ldg(reinterpret_cast<const int4*>(gamma_q) + wi), b = __ldg(reinterpret_cast<const int4*>(beta_q) + wi);
            const int gg[4] = {g.x, g.y, g.z, g.w}, bb[4] = {b.x, b.y, b.z, b.w};
            int o[4];
#pragma unroll
            for (int t = 0; t < 4; ++t)
                o[t] = requant_full(r.n<true>(((int)(int8_t)((unsigned)w >> (8 * t))) * (4 * c.dim << ((sh >> (8 * t)) & 3))) * gg[t] + bb[t], c.out);
            reinterpret_cast<int*>(y + row * c.dim)[wi] = (int)pack4_s8(o[0], o[1], o[2], o[3]);
        }
    }
}

// Short rows (dim <= 128, dim % 16 == 0: the first Swin stage): LPR lanes share a row, so a warp step covers 32 / LPR
// rows.  Lane q of a row takes the VEC-word pieces q, q + LPR, ... of it (WPL words in all): with one word at a time every load
// touched a 32-byte sector per row for 8 bytes of it.  Row sums are xor-shuffles over the LPR lanes, and every lane then runs
// the scalar part (variance, square root, reciprocal) of its own row, so that part is shared by 32 / LPR rows
// without any broadcast.  [200704, 96]: 19.4 -> 15.6 us, with power-of-two factors 26.5 -> 15.9.  Two lanes per row up to 96 channels, four at 128, where twelve more words per lane would spill.
template <int LPR, int WPL, int VEC, bool PTF, bool SAT8>
__global__ void __launch_bounds__(256, PTF ? 3 : 4)
layernorm_short_rows_kernel(const LnSource src, int8_t* __restrict__ y, int64_t rows, const int32_t* __restrict__ gamma_q,
                            const int32_t* __restrict__ beta_q, const uint8_t* __restrict__ ptf, const LnDev c)
{
    const int lane = threadIdx.x & 31;
    constexpr int RPW = 32 / LPR, WORDS = LPR * WPL, D = 4 * WORDS;
    const int q = lane & (LPR - 1);                           // position inside the row's lanes
    grid_dep_launch();
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t steps = (rows + RPW - 1) / RPW;
    // The per-channel parameters live in shared memory (the lanes of a row read consecutive addresses, the rows of a
    // warp the same ones: no bank conflict): resident warps are what hides a row's chain of dependent steps.
    __shared__ int4 sg[WORDS], sb[WORDS], sd[PTF ? WORDS : 1], sm[PTF ? WORDS : 1];     // .., 4 D 2^alpha per channel, masks of the factors
    for (int i = threadIdx.x; i < WORDS; i += blockDim.x) {
        sg[i] = __ldg(reinterpret_cast<const int4*>(gamma_q) + i);
        sb[i] = __ldg(reinterpret_cast<const int4*>(beta_q) + i);
        if (PTF) {
            const unsigned sh = __ldg(reinterpret_cast<const unsigned*>(ptf) + i);
            sd[i] = make_int4(4 * D << (sh & 3u), 4 * D << ((sh >> 8) & 3u), 4 * D << ((sh >> 16) & 3u), 4 * D << ((sh >> 24) & 3u));
            sm[i] = ln_ptf_masks(sh);
        }
    }
    __syncthreads();
    const RequantDev out = c.out;
    grid_dep_wait();                                          // gamma / beta above are static; the rows come from the previous kernel
    using Vec = typename std::conditional<VEC == 4, int4, int2>::type;
    for (int64_t step = warp; step < steps; step += nwarps) {
        const int64_t row = step * RPW + lane / LPR;
        const bool live = row < rows;
        int64_t from = row;
        if (src.index) from = live ? __ldg(src.index + row) : -1;
        const bool read = live && from >= 0;
        const Vec* xr = reinterpret_cast<const Vec*>(src.x + (read ? from : 0) * D);
        int w[WPL];
#pragma unroll
        for (int k = 0; k < WPL / VEC; ++k) {
            Vec v{};
            if (read) v = __ldcs(xr + q + LPR * k);
            const int* p = reinterpret_cast<const int*>(&v);
#pragma unroll
            for (int i = 0; i < VEC; ++i) w[k * VEC + i] = p[i];
        }
        auto word_index = [&](int k) { return VEC * (q + LPR * (k / VEC)) + k % VEC; };
        int s1 = 0;
        unsigned s2 = 0;
        if (PTF) {
            LnPtfSums p;
#pragma unroll
            for (int k = 0; k < WPL; ++k) { const int4 m = sm[word_index(k)]; p.add(w[k], m, ln_ptf_factors(m)); }
            s1 = p.s1;
            s2 = p.s2();
        } else {
#pragma unroll
            for (int k = 0; k < WPL; ++k) {
                s1 = __dp4a(w[k], 0x01010101, s1);
                s2 = (unsigned)__dp4a(w[k], w[k], (int)s2);
            }
        }
        s1 += __shfl_xor_sync(kFull, s1, 1); s2 += __shfl_xor_sync(kFull, s2, 1);
        if (LPR == 4) { s1 += __shfl_xor_sync(kFull, s1, 2); s2 += __shfl_xor_sync(kFull, s2, 2); }
        const double s1d = (double)s1;
        const double F = ln_reciprocal(ln_isqrt(fma(-s1d, s1d, (double)D * (double)s2), c.variant));
        LnRow one;
        one.set(s1, F);
        auto emit = [&](auto wide) {
#pragma unroll
            for (int k = 0; k < WPL / VEC; ++k) {
                Vec v;
                int* p = reinterpret_cast<int*>(&v);
#pragma unroll
                for (int i = 0; i < VEC; ++i) {
                    const int wi = word_index(VEC * k + i);
                    const int4 d = PTF ? sd[wi] : make_int4(4 * D, 4 * D, 4 * D, 4 * D);
                    const int d4[4] = {d.x, d.y, d.z, d.w};
                    p[i] = ln_word<decltype(wide)::value, SAT8>((unsigned)w[k * VEC + i], d4, one, sg[wi], sb[wi], out);
                }
                if (live) __stcs(reinterpret_cast<Vec*>(y + row * D) + q + LPR * k, v);
            }
        };
        if (__any_sync(kFull, one.f_hi != 0)) emit(std::true_type{}); else emit(std::false_type{});
    }
}

// W16 = dim / 16
template <int W16>
static int launch_ln_short(const LnSource& src, int8_t* y, int64_t rows, const int32_t* gq, const int32_t* bq, const uint8_t* ptf,
                           const LnDev& c, cudaStream_t st)
{
    constexpr int LPR = W16 <= 6 ? 2 : 4, WPL = 4 * W16 / LPR, VEC = WPL % 4 == 0 ? 4 : 2;
    const int64_t want = ((rows + 32 / LPR - 1) / (32 / LPR) + 7) / 8;
    const int grid = (int)std::min<int64_t>(want, (int64_t)sm_count() * 8);
    const bool sat8 = c.out.qmin == -128 && c.out.qmax == 127;
#define IPTQ_LNS_GO(P, S8) launch_kernel(layernorm_short_rows_kernel<LPR, WPL, VEC, P, S8>, grid, 256, 0, st, src, y, rows, gq, bq, ptf, c)
    if (c.variant == IPTQ_LN_PTF) { if (sat8) IPTQ_LNS_GO(true, true); else IPTQ_LNS_GO(true, false); }
    else { if (sat8) IPTQ_LNS_GO(false, true); else IPTQ_LNS_GO(false, false); }
#undef IPTQ_LNS_GO
    note_launch();
    return last_launch_status();
}

template <int NW>
static int launch_ln(const LnSource& src, int8_t* y, int64_t rows, const int32_t* gq, const int32_t* bq, const uint8_t* ptf,
                     const LnDev& c, cudaStream_t st)
{
    // Up to 32 rows per SM a warp takes one row, so that the rows are spread over the chip ([1576, 384]: 3.8 -> 2.8 us), up to 128
    // rows two ([12608, 384]: 7.3 us with four, 6.3 with two), else four.
    constexpr int RW = NW <= 8 ? 4 : NW <= 16 ? 2 : 1, RM = RW < 2 ? 1 : 2;
    const int rw = rows <= (int64_t)sm_count() * 32 ? 1 : rows <= (int64_t)sm_count() * 128 ? RM : RW;
    const int64_t want = ((rows + rw - 1) / rw + 7) / 8;
    const int grid = (int)std::min<int64_t>(want, (int64_t)sm_count() * 32);
    const bool sat8 = c.out.qmin == -128 && c.out.qmax == 127;
    const bool exact = c.dim == 128 * NW;
    const size_t smem = 8 * (size_t)c.dim;
#define IPTQ_LN_GO(P, EX, S8)                                                                                                \
    do {                                                                                                                     \
        if (rw == 1) launch_kernel(layernorm_rows_kernel<NW, 1, P, EX, S8>, grid, 256, smem, st, src, y, rows, gq, bq, ptf, c); \
        else if (rw == RM) launch_kernel(layernorm_rows_kernel<NW, RM, P, EX, S8>, grid, 256, smem, st, src, y, rows, gq, bq, ptf, c); \
        else launch_kernel(layernorm_rows_kernel<NW, RW, P, EX, S8>, grid, 256, smem, st, src, y, rows, gq, bq, ptf, c);     \
    } while (0)
    if (c.variant == IPTQ_LN_PTF) { if (sat8) IPTQ_LN_GO(true, false, true); else IPTQ_LN_GO(true, false, false); }
    else if (!sat8) IPTQ_LN_GO(false, false, false);
    else if (exact) IPTQ_LN_GO(false, true, true);
    else IPTQ_LN_GO(false, false, true);
#undef IPTQ_LN_GO
    note_launch();
    return last_launch_status();
}

int layernorm_check(const LnArgs& a, const int8_t* y, int64_t rows, int dim)
{
    if (!a.consts) return IPTQ_ERR_NULL;
    if (rows < 0 || dim != a.consts->dim || dim < 2 || dim > 3072 || (dim & 3)) return IPTQ_ERR_SHAPE;
    if (a.parts < 1 || a.parts > 4 || dim % (4 * a.parts) || (a.parts > 1 && !a.index)) return IPTQ_ERR_SHAPE;
    if (rows == 0) return IPTQ_OK;
    if (!a.x || !y || !a.gamma || !a.beta) return IPTQ_ERR_NULL;
    if (a.consts->variant < 0 || a.consts->variant > 2) return IPTQ_ERR_VARIANT;
    if (a.consts->variant == IPTQ_LN_PTF && !a.ptf) return IPTQ_ERR_NULL;
    if (!aligned16(a.x) || !aligned16(y) || !aligned16(a.gamma) || !aligned16(a.beta) ||
        (a.ptf && (reinterpret_cast<uintptr_t>(a.ptf) & 3u)) || (reinterpret_cast<uintptr_t>(a.index) & 3u))
        return IPTQ_ERR_ALIGN;
    return check_requant(&a.consts->out);
}

// Used by the encoder block as well.
int layernorm_launch(const LnArgs& a, int8_t* y, int64_t rows, int dim, cudaStream_t st)
{
    const int rc = layernorm_check(a, y, rows, dim);
    if (rc != IPTQ_OK || rows == 0) return rc;
    LnDev c;
    c.variant = a.consts->variant; c.dim = dim; c.out = to_dev(a.consts->out);
    const LnSource src{a.x, a.index, a.parts, dim / 4 / a.parts};
    const bool is_ptf = c.variant == IPTQ_LN_PTF;
    // the other kernels have the zero point in the rounding constant, where the sum stays clear of 32-bit overflow (|hi32| < 2^30)
    const long long rz = (long long)c.out.rnd + ((long long)c.out.zp << c.out.shift);
    if (rz <= -(1ll << 30) || rz >= (1ll << 30)) {
        const int grid = (int)std::min<int64_t>((rows + 7) / 8, (int64_t)sm_count() * 8);
        if (is_ptf) launch_kernel(layernorm_general_kernel<true>, grid, 256, 0, st, src, y, rows, a.gamma, a.beta, a.ptf, c);
        else launch_kernel(layernorm_general_kernel<false>, grid, 256, 0, st, src, y, rows, a.gamma, a.beta, a.ptf, c);
        note_launch();
        return last_launch_status();
    }
    c.out.rnd = (int)rz; c.out.zp = 0;
    if ((dim & 15) == 0 && dim <= 128 && rows >= 64 && a.parts == 1) {
        switch (dim / 16) {
            case 1: return launch_ln_short<1>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            case 2: return launch_ln_short<2>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            case 3: return launch_ln_short<3>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            case 4: return launch_ln_short<4>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            case 6: return launch_ln_short<6>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            case 8: return launch_ln_short<8>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            default: break;                                   // other widths take the general kernel
        }
    }
    const int nw = (dim / 4 + 31) / 32;
    switch (nw) {
        case 1: return launch_ln<1>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
        case 2: return launch_ln<2>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
        case 3: return launch_ln<3>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
        case 4: return launch_ln<4>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
        case 5: case 6: return launch_ln<6>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
        case 7: case 8: return launch_ln<8>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
        default:
            if (nw <= 12) return launch_ln<12>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            if (nw <= 16) return launch_ln<16>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
            return launch_ln<24>(src, y, rows, a.gamma, a.beta, a.ptf, c, st);
    }
}

}  // namespace iptq

using namespace iptq;

extern "C" {

int iptq_layernorm(const int8_t* x, int8_t* y, int64_t rows, int dim, const int32_t* gamma_q,
                   const int32_t* beta_q, const uint8_t* ptf_shift, const iptq_ln_consts* consts,
                   iptq_stream_t stream)
{
    return layernorm_launch(LnArgs{x, gamma_q, beta_q, ptf_shift, consts}, y, rows, dim, stream);
}

int iptq_layernorm_gather(const int8_t* x, int8_t* y, int64_t rows, int dim, const int32_t* index, int parts,
                          const int32_t* gamma_q, const int32_t* beta_q, const uint8_t* ptf_shift,
                          const iptq_ln_consts* consts, iptq_stream_t stream)
{
    if (rows > 0 && !index) return IPTQ_ERR_NULL;
    return layernorm_launch(LnArgs{x, gamma_q, beta_q, ptf_shift, consts, index, parts}, y, rows, dim, stream);
}

}  // extern "C"
