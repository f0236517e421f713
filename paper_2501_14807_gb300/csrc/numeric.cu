// numeric.cu -- numeric layers (arXiv 2501.14807, Section 4.2): a data texture of 8/16/32-bit
// integers or 16/32-bit floats plus a mask texture (here one bit per texel).  Whole-layer
// operations, all HBM streams over the texture:
//   k_num_arith   arithmetic overlay a <op> b (or a <op> scalar): each lane takes a 16-byte chunk of
//                 data (warp-contiguous), the mask bits of its texels come from the word shared by
//                 the 2, 4 or 8 lanes of its group, and the group's output word is merged with
//                 shuffles and written by its first lane
//   k_num_select  selection by value into a label layer (the lane owns its texels' label bytes)
//   k_num_stats   zonal statistics: a warp walks down strips of 32 texels, four rows per step (a quad per
//                 lane); two runs of equal zone labels stay in registers, as integers, until the warp
//                 meets further zones, then are reduced across the warp, rounded to double and flushed
//                 into a shared-memory table (or the output, for many zones); min / max through
//                 order-preserving 64-bit keys
#include <algorithm>
#include <type_traits>

#include <cuda_fp16.h>

#include "lcl_impl.cuh"

namespace lcl {
namespace {

constexpr int kKindUnsigned = 1, kKindSigned = 2, kKindFloat = 3;
constexpr uint32_t kSmemZones = 1024;  // zone tables up to this size live in shared memory (48 KB)

template <int S>
__device__ __forceinline__ uint32_t width_mask() {
    return S == 4 ? 0xFFFFFFFFu : ((1u << (8 * S)) - 1u);
}

template <int S>
__device__ __forceinline__ int32_t sext(uint32_t v) {
    if (S == 1) return (int32_t)(int8_t)(uint8_t)v;
    if (S == 2) return (int32_t)(int16_t)(uint16_t)v;
    return (int32_t)v;
}

template <int S>
__device__ __forceinline__ float to_float(uint32_t v) {
    if (S == 2) return __half2float(__ushort_as_half((unsigned short)v));
    return __uint_as_float(v);
}

template <int S>
__device__ __forceinline__ uint32_t from_float(float f) {
    if (S == 2) return (uint32_t)__half_as_ushort(__float2half_rn(f));
    return __float_as_uint(f);
}

// One arithmetic operation on the bits of two values of the type (S bytes, KIND).
template <int S, int KIND>
__device__ __forceinline__ uint32_t arith(uint32_t a, uint32_t b, int op) {
    if (KIND == kKindFloat) {
        const float x = to_float<S>(a), y = to_float<S>(b);
        float r;
        switch (op) {
        case LCL_ADD: r = __fadd_rn(x, y); break;
        case LCL_SUB: r = __fsub_rn(x, y); break;
        case LCL_MUL: r = __fmul_rn(x, y); break;
        case LCL_DIV: r = __fdiv_rn(x, y); break;
        case LCL_MIN: r = x < y ? x : y; break;
        default: r = x > y ? x : y; break;
        }
        return from_float<S>(r);
    }
    uint32_t r;
    switch (op) {
    case LCL_ADD: r = a + b; break;
    case LCL_SUB: r = a - b; break;
    case LCL_MUL: r = a * b; break;
    case LCL_MIN: r = (KIND == kKindSigned ? sext<S>(a) < sext<S>(b) : a < b) ? a : b; break;
    default: r = (KIND == kKindSigned ? sext<S>(a) > sext<S>(b) : a > b) ? a : b; break;
    }
    return r & width_mask<S>();
}

// Element k of a 16-byte chunk of S-byte values.
template <int S>
__device__ __forceinline__ uint32_t elem(const uint32_t (&w)[4], int k) {
    if (S == 4) return w[k];
    if (S == 2) return (w[k >> 1] >> (16 * (k & 1))) & 0xFFFFu;
    return (w[k >> 2] >> (8 * (k & 3))) & 0xFFu;
}

template <int S>
__device__ __forceinline__ void set_elem(uint32_t (&w)[4], int k, uint32_t v) {
    if (S == 4) {
        w[k] = v;
    } else if (S == 2) {
        const int sh = 16 * (k & 1);
        w[k >> 1] = (w[k >> 1] & ~(0xFFFFu << sh)) | (v << sh);
    } else {
        const int sh = 8 * (k & 3);
        w[k >> 2] = (w[k >> 2] & ~(0xFFu << sh)) | (v << sh);
    }
}

struct ArithArgs {
    const uint4 *a, *b;
    uint4 *out;
    const uint32_t *ma, *mb, *cover;
    uint32_t *mout;
    uint32_t b_value;
    int op;
    int64_t n_chunks;  // 16-byte chunks over whole mask words: (n_texels / 32) * 32 texels
    int64_t n_texels;
};

// Texels of one lane's chunk: 16 / S, starting at texel c * (16 / S), inside mask word
// (c * (16 / S)) / 32 at bit (c * (16 / S)) % 32; 2S consecutive lanes share that word.  Float layers load
// the next chunk while they work on this one, which takes 48 registers and leaves room for five CTAs on an SM;
// the shorter work of integer layers is better hidden by eight.  16384^2, a + b: f32 560 us (650 with eight
// CTAs without the look-ahead), f16 350 (402), u32 513 without it (517 with), i16 285 (350), u8 235 (272).
// The grid is what fits: with eight CTAs per SM of which five fit, the last three ran alone.
template <int KIND>
struct ArithShape {
    static constexpr bool kAhead = KIND == kKindFloat;
    static constexpr int kCtas = kAhead ? 5 : 8;
};
template <int S, int KIND>
__global__ void __launch_bounds__(kThreads, ArithShape<KIND>::kCtas) k_num_arith(const __grid_constant__ ArithArgs p) {
    constexpr bool kAhead = ArithShape<KIND>::kAhead;
    constexpr int kPer = 16 / S;
    constexpr int kGroup = 32 / kPer;  // lanes per mask word
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // whole warps iterate together (the group merge uses shuffles over the full warp); out may be a or b: a
    // thread writes only chunks it has read
    const int64_t n_iter = (p.n_chunks + 31) & ~int64_t(31);
    uint4 A = make_uint4(0u, 0u, 0u, 0u), B = A;
    uint32_t ok = 0u;
    auto load = [&](int64_t c) {
        const int64_t t0 = c * kPer;
        if (c < p.n_chunks && LCL_IN(t0 + kPer - 1, p.n_texels)) {
            A = __ldcs(p.a + c);
            if (p.b) B = __ldcs(p.b + c);
            const uint32_t word = (uint32_t)(t0 >> 5);
            ok = __ldg(p.ma + word) & __ldg(p.cover + word);
            if (p.b) ok &= __ldg(p.mb + word);
        }
    };
    int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (kAhead) load(c);
    for (; c - (threadIdx.x & 31) < n_iter; c += stride) {
        if (!kAhead) load(c);
        const int64_t t0 = c * kPer;
        const bool live = c < p.n_chunks && LCL_IN(t0 + kPer - 1, p.n_texels);
        const uint32_t aw[4] = {A.x, A.y, A.z, A.w}, bw[4] = {B.x, B.y, B.z, B.w};
        const uint32_t now = ok;
        if (kAhead) load(c + stride);
        uint32_t bits = 0;
        if (live) {
            const int off = (int)(t0 & 31);
            const uint32_t valid = (now >> off) & (kPer == 32 ? 0xFFFFFFFFu : ((1u << kPer) - 1u));
            uint32_t rw[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int k = 0; k < kPer; ++k) {
                const uint32_t bv = p.b ? elem<S>(bw, k) : p.b_value;
                const uint32_t r = (valid >> k) & 1u ? arith<S, KIND>(elem<S>(aw, k), bv, p.op) : 0u;
                set_elem<S>(rw, k, r);
            }
            __stcs(p.out + c, make_uint4(rw[0], rw[1], rw[2], rw[3]));
            bits = valid << off;
        }
#pragma unroll
        for (int o = 1; o < kGroup; o <<= 1) bits |= __shfl_xor_sync(0xffffffffu, bits, o);
        if (live && (threadIdx.x & (kGroup - 1)) == 0) p.mout[t0 >> 5] = bits;
    }
    // the last n_texels % 32 texels (one partial mask word), by the grid's first thread
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t t_begin = (p.n_texels >> 5) << 5;
        if (t_begin < p.n_texels && LCL_IN(t_begin >> 5, (p.n_texels + 31) >> 5)) {
            const uint32_t word = (uint32_t)(t_begin >> 5);
            uint32_t valid = p.ma[word] & p.cover[word];
            if (p.b) valid &= p.mb[word];
            uint32_t bits = 0;
            for (int64_t t = t_begin; t < p.n_texels; ++t) {
                const int k = (int)(t - t_begin);
                uint32_t av, bv = p.b_value;
                if (S == 1) {
                    av = reinterpret_cast<const uint8_t *>(p.a)[t];
                    if (p.b) bv = reinterpret_cast<const uint8_t *>(p.b)[t];
                } else if (S == 2) {
                    av = reinterpret_cast<const uint16_t *>(p.a)[t];
                    if (p.b) bv = reinterpret_cast<const uint16_t *>(p.b)[t];
                } else {
                    av = reinterpret_cast<const uint32_t *>(p.a)[t];
                    if (p.b) bv = reinterpret_cast<const uint32_t *>(p.b)[t];
                }
                const bool v = (valid >> k) & 1u;
                const uint32_t r = v ? arith<S, KIND>(av, bv, p.op) : 0u;
                if (S == 1) reinterpret_cast<uint8_t *>(p.out)[t] = (uint8_t)r;
                else if (S == 2) reinterpret_cast<uint16_t *>(p.out)[t] = (uint16_t)r;
                else reinterpret_cast<uint32_t *>(p.out)[t] = r;
                bits |= (v ? 1u : 0u) << k;
            }
            p.mout[word] = bits;
        }
    }
}

// ---- selection by value ----------------------------------------------------------------------

template <int S, int KIND>
__device__ __forceinline__ bool compare(uint32_t v, uint32_t t, int cmp) {
    if (KIND == kKindFloat) {
        const float x = to_float<S>(v), y = to_float<S>(t);
        switch (cmp) {
        case LCL_LT: return x < y;
        case LCL_LE: return x <= y;
        case LCL_GT: return x > y;
        case LCL_GE: return x >= y;
        case LCL_EQ: return x == y;
        default: return x != y;
        }
    }
    if (KIND == kKindSigned) {
        const int32_t x = sext<S>(v), y = sext<S>(t);
        switch (cmp) {
        case LCL_LT: return x < y;
        case LCL_LE: return x <= y;
        case LCL_GT: return x > y;
        case LCL_GE: return x >= y;
        case LCL_EQ: return x == y;
        default: return x != y;
        }
    }
    switch (cmp) {
    case LCL_LT: return v < t;
    case LCL_LE: return v <= t;
    case LCL_GT: return v > t;
    case LCL_GE: return v >= t;
    case LCL_EQ: return v == t;
    default: return v != t;
    }
}

struct SelectArgs {
    const uint4 *data;
    const uint32_t *mask, *cover;
    void *layer;
    uint32_t threshold, label;
    int cmp;
    int64_t n_chunks;  // whole 16-byte chunks
    int64_t n_texels;
    unsigned long long *hits;
};

// Writes `label` (LB bytes) into the texels t0 .. t0 + n - 1 whose bit is set in `sel`.
template <int LB>
__device__ __forceinline__ void store_labels(void *layer, int64_t t0, int n, uint32_t sel, uint32_t label) {
    if (!sel) return;
    if (LB == 1) {
        uint8_t *l = static_cast<uint8_t *>(layer) + t0;
        for (int w = 0; w < n; w += 4) {  // t0 and n are multiples of 4
            const uint32_t m4 = (sel >> w) & 0xFu;
            if (!m4) continue;
            uint32_t *p = reinterpret_cast<uint32_t *>(l + w);
            uint32_t bm = ((m4 * 0x00204081u) & 0x01010101u) * 0xFFu;
            const uint32_t rep = label * 0x01010101u;
            *p = m4 == 0xFu ? rep : ((*p & ~bm) | (rep & bm));
        }
    } else {
        uint16_t *l = static_cast<uint16_t *>(layer) + t0;
        for (int w = 0; w < n; w += 2) {
            const uint32_t m2 = (sel >> w) & 0x3u;
            if (!m2) continue;
            uint32_t *p = reinterpret_cast<uint32_t *>(l + w);
            const uint32_t bm = ((m2 & 1u) ? 0x0000FFFFu : 0u) | ((m2 & 2u) ? 0xFFFF0000u : 0u);
            const uint32_t rep = label * 0x00010001u;
            *p = m2 == 0x3u ? rep : ((*p & ~bm) | (rep & bm));
        }
    }
}

template <int S, int KIND, int LB>
__global__ void __launch_bounds__(kThreads) k_num_select(SelectArgs p) {
    constexpr int kPer = 16 / S;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    uint32_t cnt = 0;
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < p.n_chunks; c += stride) {
        if (!LCL_IN(c * kPer + kPer - 1, p.n_texels)) continue;
        const uint4 D = __ldcs(p.data + c);
        const int64_t t0 = c * kPer;
        const uint32_t word = (uint32_t)(t0 >> 5);
        const uint32_t valid = ((__ldg(p.mask + word) & __ldg(p.cover + word)) >> (t0 & 31)) &
                               (kPer == 32 ? 0xFFFFFFFFu : ((1u << kPer) - 1u));
        if (!valid) continue;
        const uint32_t dw[4] = {D.x, D.y, D.z, D.w};
        uint32_t sel = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k)
            if ((valid >> k) & 1u) sel |= (compare<S, KIND>(elem<S>(dw, k), p.threshold, p.cmp) ? 1u : 0u) << k;
        store_labels<LB>(p.layer, t0, kPer, sel, p.label);
        cnt += __popc(sel);
    }
    // tail texels after the whole chunks (fewer than 16 / S), by the grid's first thread
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        for (int64_t t = p.n_chunks * kPer; t < p.n_texels; ++t) {
            if (!LCL_IN(t, p.n_texels)) break;
            const uint32_t word = (uint32_t)(t >> 5);
            if (!(((p.mask[word] & p.cover[word]) >> (t & 31)) & 1u)) continue;
            uint32_t v;
            if (S == 1) v = reinterpret_cast<const uint8_t *>(p.data)[t];
            else if (S == 2) v = reinterpret_cast<const uint16_t *>(p.data)[t];
            else v = reinterpret_cast<const uint32_t *>(p.data)[t];
            if (!compare<S, KIND>(v, p.threshold, p.cmp)) continue;
            if (LB == 1) static_cast<uint8_t *>(p.layer)[t] = (uint8_t)p.label;
            else static_cast<uint16_t *>(p.layer)[t] = (uint16_t)p.label;
            ++cnt;
        }
    }
    if (p.hits) {
        for (int o = 16; o; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(p.hits, (unsigned long long)cnt);
    }
}

// ---- zonal statistics ------------------------------------------------------------------------

// Order-preserving 64-bit key of a double (atomicMin / atomicMax on doubles).
__device__ __forceinline__ unsigned long long dkey(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double key_double(unsigned long long k) {
    return __longlong_as_double((long long)((k >> 63) ? (k & 0x7FFFFFFFFFFFFFFFull) : ~k));
}

// Accumulator layout of one zone while the kernel runs (same 48 bytes as lcl_zone_stats, with
// order-preserving keys in place of vmin / vmax).
struct ZoneAcc {
    unsigned long long count, area, kmin, kmax;
    double sum, wsum;
};
static_assert(sizeof(ZoneAcc) == sizeof(lcl_zone_stats), "zone accumulator must alias lcl_zone_stats");

__global__ void k_stats_init(ZoneAcc *z, uint32_t n) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        z[i].count = 0;
        z[i].area = 0;
        z[i].kmin = ~0ull;
        z[i].kmax = 0;
        z[i].sum = 0.0;
        z[i].wsum = 0.0;
    }
}

__global__ void k_stats_final(ZoneAcc *z, uint32_t n) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        lcl_zone_stats *o = reinterpret_cast<lcl_zone_stats *>(z + i);
        const unsigned long long kmin = z[i].kmin, kmax = z[i].kmax;
        const bool empty = z[i].count == 0;
        o->vmin = empty ? __longlong_as_double(0x7FF0000000000000ll) : key_double(kmin);
        o->vmax = empty ? __longlong_as_double((long long)0xFFF0000000000000ull) : key_double(kmax);
    }
}

// ---- per-texel value handling for the statistics ------------------------------------------
// Order-preserving 32-bit key of a value in its own type (integer min / max, no FP64):
// unsigned: the value; signed: value ^ 2^31 (of the sign-extended value); floats: the float32
// bits with the sign folded.  key_value turns a key back into the exact double.
template <int S, int KIND>
__device__ __forceinline__ uint32_t vkey(uint32_t f32_or_int_bits) {
    if (KIND == kKindFloat) {
        const uint32_t b = f32_or_int_bits;
        return (b >> 31) ? ~b : (b | 0x80000000u);
    }
    if (KIND == kKindSigned) return (uint32_t)sext<S>(f32_or_int_bits) ^ 0x80000000u;
    return f32_or_int_bits;
}

template <int S, int KIND>
__device__ __forceinline__ double key_value(uint32_t k) {
    if (KIND == kKindFloat) return (double)__uint_as_float((k >> 31) ? (k & 0x7FFFFFFFu) : ~k);
    if (KIND == kKindSigned) return (double)(int32_t)(k ^ 0x80000000u);
    return (double)k;
}

__device__ __forceinline__ void acc_add(ZoneAcc *z, unsigned long long cnt, unsigned long long area,
                                        unsigned long long kmin, unsigned long long kmax, double sum, double wsum) {
    atomicAdd(&z->count, cnt);
    atomicAdd(&z->area, area);
    atomicMin(&z->kmin, kmin);
    atomicMax(&z->kmax, kmax);
    atomicAdd(&z->sum, sum);
    atomicAdd(&z->wsum, wsum);
}

// x 2^k as a double (two roundings at most: the halves' sum; |k| <= 300).
__device__ __forceinline__ double i128_to_double(__int128 x, int k) {
    const bool neg = x < 0;
    const unsigned __int128 m = neg ? -(unsigned __int128)x : (unsigned __int128)x;
    const double v = __dadd_rn(__dmul_rn(__ull2double_rn((unsigned long long)(m >> 64)), 18446744073709551616.0),
                               __ull2double_rn((unsigned long long)m));
    const double r = __dmul_rn(v, __hiloint2double((1023 + k) << 20, 0));
    return neg ? -r : r;
}

// The sum of v over the warp's lanes, |v| < 2^63: 26-bit pieces whose sums stay below 2^31, the top one
// signed.
__device__ __forceinline__ __int128 warp_sum_i64(long long v) {
    const uint32_t a = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0x3FFFFFFu);
    const uint32_t b = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 26) & 0x3FFFFFFu);
    const int32_t c = __reduce_add_sync(0xffffffffu, (int32_t)(v >> 52));
    return (__int128)((long long)a + ((long long)b << 26)) + ((__int128)c << 52);
}
// A signed 96-bit integer, for the weighted sums.
struct Int96 {
    uint32_t w0, w1, w2;
};
__device__ __forceinline__ void add96(Int96 &a, uint32_t b0, uint32_t b1, uint32_t b2) {
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2)
        : "r"(b0), "r"(b1), "r"(b2));
}
// Its sum over the warp's lanes, in 26-bit pieces.
__device__ __forceinline__ __int128 warp_sum_i96(const Int96 &v) {
    const uint32_t a = __reduce_add_sync(0xffffffffu, v.w0 & 0x3FFFFFFu);
    const uint32_t b = __reduce_add_sync(0xffffffffu, __funnelshift_r(v.w0, v.w1, 26) & 0x3FFFFFFu);
    const uint32_t c = __reduce_add_sync(0xffffffffu, __funnelshift_r(v.w1, v.w2, 20) & 0x3FFFFFFu);
    const int32_t d = __reduce_add_sync(0xffffffffu, (int32_t)v.w2 >> 14);
    return (__int128)((long long)a + ((long long)b << 26)) + ((__int128)c << 52) + ((__int128)d << 78);
}

// The exact sums of a run of texels: integers in units of 2^(base - 150), the unit of a float32 whose
// biased exponent is `base`.  A float32 value (significand m of 24 bits, exponent e) adds m << (e - base)
// for exponents base .. base + kWindow; integer layers and float16 (multiples of 2^-24) have a fixed
// unit.  A lane takes at most kRunTexels texels before a flush, so |s| < 2^(24 + kWindow + 10) and the
// weighted sum (weights below 2^35) < 2^94.  Float32 values below the unit, subnormals and infinities are
// summed in binary64, per lane (OutSums).  The unit follows the values: it rises when a step holds a larger
// one than the window, and falls when a step's largest value has fallen kFallen below the one it was set
// for, kFallSteps steps at least after the last flush, so that it does not swing from step to step.
constexpr int kWindow = 25, kRunTexels = 1024;
constexpr int kHeadroom = 20, kFallen = 16, kFallSteps = 8;
// Steps of a warp at least: a warp's zones and a CTA's table are written out at the end of its work.
constexpr int kStatsSteps = 4;
// Times a step lets zones take over runs; a step of more than twice as many zones is noise, whose texels
// cost less one by one.
constexpr int kZoneRounds = 3;

struct StatsRun {
    uint32_t zone;
    uint32_t cnt, kmin, kmax;  // value keys (vkey) of the smallest and largest value
    unsigned long long area;
    long long s;
    Int96 w;
};

__device__ __forceinline__ void run_reset(StatsRun &r) {
    r.cnt = 0;
    r.area = 0;
    r.kmin = 0xFFFFFFFFu;
    r.kmax = 0u;
    r.s = 0;
    r.w.w0 = r.w.w1 = r.w.w2 = 0u;
}

struct StatsArgs {
    const void *data;
    const uint32_t *mask, *cover, *tri;
    const unsigned long long *area_w;
    const void *zones;  // NULL: one zone
    uint32_t n_labels;
    int64_t n_texels;
    int64_t n_tri;
    int32_t w4, h;      // quads per row, rows
    ZoneAcc *out;
};

// Four consecutive S-byte values of a quad.
template <int S>
struct Quad4 {
    uint32_t w[S];
    __device__ __forceinline__ void load(const void *data, int64_t q) {
        if constexpr (S == 1) {
            w[0] = __ldcs(static_cast<const uint32_t *>(data) + q);
        } else if constexpr (S == 2) {
            const uint2 v = __ldcs(static_cast<const uint2 *>(data) + q);
            w[0] = v.x;
            w[1] = v.y;
        } else {
            const uint4 v = __ldcs(static_cast<const uint4 *>(data) + q);
            w[0] = v.x;
            w[1] = v.y;
            w[2] = v.z;
            w[3] = v.w;
        }
    }
    __device__ __forceinline__ uint32_t get(int k) const {
        if (S == 4) return w[k];
        if (S == 2) return (w[k >> 1] >> (16 * (k & 1))) & 0xFFFFu;
        return (w[0] >> (8 * k)) & 0xFFu;
    }
};

// m 2^e as a double, rounded to nearest, by integer operations (0 < m < 2^64, the result a normal double; an
// FP64 operation costs a warp as much as 64 others on this part).
__device__ __forceinline__ double scaled_to_double(uint64_t m, int e, uint32_t sign) {
    const int lz = __clzll((long long)m);
    m <<= lz;
    const uint64_t q = (m >> 11) + ((m >> 10) & 1u);  // 53 bits, or 2^53, whose carry goes to the exponent
    return __longlong_as_double((long long)((((uint64_t)(e - lz + 63 + 1022) << 52) + q) | ((uint64_t)sign << 63)));
}

// The binary64 sums of a thread's texels that do not fit their run's unit: value and weight x value, by zone, until
// the end of a step in which a run changes its zone, or of the work: such a step holds texels of two zones and of
// the two before them (more go to the table one by one).  They lie in shared memory and are written to the table between steps, where registers are free: with a call in the
// middle of a step or in the flush of a run, a layer without such texels took 7 to 80% more time.  8192^2
// float32, one zone, of values near 1: 0.34 ms; with a value of 1e30 in each 4096 (256) texels 0.46 (0.61),
// where an atomic per texel, 32 lanes to one address, took 16 (26) and binary64 sums throughout 0.58; of
// values over 60 powers of two 0.64, and 17 with the atomics.
constexpr int kOutZones = 4;
struct OutSums {
    double s[kOutZones][kThreads], w[kOutZones][kThreads];
    uint32_t zone[kOutZones][kThreads];  // filled from the first place on; kNone: empty
};
// A texel of zone `zone`: float32 bits v (not 0), weight w.  v and the product go to binary64 by their bits: by
// conversions and products on the FP64 pipe layers of very wide range took 690 us for 8192^2, not 610.
__device__ __forceinline__ void outs_add(OutSums &o, uint32_t zone, uint32_t v, unsigned long long w, ZoneAcc *tab) {
    const uint32_t e = (v >> 23) & 0xFFu, f = v & 0x7FFFFFu;
    const double d = e - 1u < 254u ? __hiloint2double((int)((v & 0x80000000u) | ((e + 896u) << 20) | (f >> 3)), (int)(v << 29))
                                   : (double)__uint_as_float(v);
    const double wd = e < 255u && w ? scaled_to_double((uint64_t)(e ? f | 0x800000u : f) * w, (int)max(e, 1u) - 150, v >> 31)
                                    : __dmul_rn(__ull2double_rn(w), d);
    int i = 0;
    uint32_t held = o.zone[0][threadIdx.x];
#pragma unroll 1
    while (held != zone && held != kNone && ++i < kOutZones) held = o.zone[i][threadIdx.x];
    if (i == kOutZones) {
        atomicAdd(&tab[zone].sum, d);
        atomicAdd(&tab[zone].wsum, wd);
        return;
    }
    double &s = o.s[i][threadIdx.x], &t = o.w[i][threadIdx.x];
    if (held == zone) {
        s = __dadd_rn(s, d);
        t = __dadd_rn(t, wd);
    } else {
        o.zone[i][threadIdx.x] = zone;
        s = d;
        t = wd;
    }
}
// All of a warp's places into the table; every lane calls it.
__device__ __noinline__ void outs_end(OutSums &o, ZoneAcc *tab) {
#pragma unroll 1
    for (int i = 0; i < kOutZones; ++i) {
        uint32_t zone = o.zone[i][threadIdx.x];
        for (;;) {  // zone by zone
            const uint32_t bal = __ballot_sync(0xffffffffu, zone != kNone);
            if (!bal) break;
            const int leader = __ffs(bal) - 1;
            const uint32_t z = __shfl_sync(0xffffffffu, zone, leader);
            double s = zone == z ? o.s[i][threadIdx.x] : 0.0, t = zone == z ? o.w[i][threadIdx.x] : 0.0;
#pragma unroll 1
            for (int k = 16; k; k >>= 1) {
                s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, k));
                t = __dadd_rn(t, __shfl_xor_sync(0xffffffffu, t, k));
            }
            if ((threadIdx.x & 31) == 0) {
                atomicAdd(&tab[z].sum, s);
                atomicAdd(&tab[z].wsum, t);
            }
            if (zone == z) o.zone[i][threadIdx.x] = zone = kNone;
        }
    }
}

// One texel into the table.
template <int S, int KIND>
__device__ __noinline__ void stats_single(ZoneAcc *tab, uint32_t n_zones, uint32_t zone, uint32_t v,
                                          unsigned long long w) {
    if (!LCL_IN(zone, n_zones)) return;
    (void)n_zones;
    const double d = key_value<S, KIND>(vkey<S, KIND>(v));
    acc_add(tab + zone, 1ull, w, dkey(d), dkey(d), d, __dmul_rn(__ull2double_rn(w), d));
}

// Zonal statistics.  A warp walks down a strip of 32 texels, four rows per step, a quad of four texels
// per lane, the next step's loads issued ahead.  Two zones have a run each, per-lane sums in registers,
// all integers: count, area, min / max as keys of the value's own type, the values and weight x value.
// A strip meets few zones, and along a border the same two row after row.  When a step holds a third
// zone, a run (one that the step does not use, if there is one) is reduced into the table and taken over;
// what is left after three such rounds goes to the table texel by texel.
// The sums are rounded only when they go to the table.
// Bound by instructions.  Summing in binary64 per texel was held by the FP64 pipe (1/64 of the FP32 rate
// on this part).  8192^2 float32, 40 zones: 862 -> 390 us; strips of 64 or 128 texels, which meet more
// zones, 470 and 680.
template <int S, int KIND, int ZB, bool SMEM>
__global__ void __launch_bounds__(kThreads, 3) k_num_stats(StatsArgs p) {
    constexpr bool kF32 = KIND == kKindFloat && S == 4;
    constexpr bool kFloat = KIND == kKindFloat;
    extern __shared__ ZoneAcc sh_zone[];
    __shared__ OutSums outs;  // float layers only
    ZoneAcc *tab = SMEM ? sh_zone : p.out;
    if (kFloat)
        for (int i = 0; i < kOutZones; ++i) outs.zone[i][threadIdx.x] = kNone;
    if (SMEM) {
        for (uint32_t i = threadIdx.x; i < p.n_labels; i += blockDim.x) {
            sh_zone[i].count = 0;
            sh_zone[i].area = 0;
            sh_zone[i].kmin = ~0ull;
            sh_zone[i].kmax = 0;
            sh_zone[i].sum = 0.0;
            sh_zone[i].wsum = 0.0;
        }
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    // units of kStatsSteps to 32 steps: steps u / n_strips * per and on of strip u % n_strips, so that neighbouring
    // warps read neighbouring texels, and a warp's units lie apart (borders of zones cost more)
    constexpr int kCols = 8, kRows = 32 / kCols;  // lanes side by side, rows per step
    const int32_t n_strips = (p.w4 + kCols - 1) / kCols, n_groups = (p.h + kRows - 1) / kRows;
    const int32_t n_warps = (int32_t)((gridDim.x * blockDim.x) >> 5);
    const int32_t warp = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int32_t per = max(kStatsSteps, min(32, (int32_t)((int64_t)n_groups * n_strips / n_warps)));
    const int32_t n_units = n_strips * ((n_groups + per - 1) / per);
    const uint32_t ntri = p.n_tri < (int64_t)0xFFFFFFFFu ? (uint32_t)p.n_tri : 0xFFFFFFFFu;

    uint4 T = make_uint4(kNone, kNone, kNone, kNone);
    Quad4<S> V;
    Quad4<ZB> Z;
    uint32_t bits = 0u;
#pragma unroll
    for (int k = 0; k < S; ++k) V.w[k] = 0u;
#pragma unroll
    for (int k = 0; k < ZB; ++k) Z.w[k] = 0u;
    auto load = [&](int32_t strip, int32_t group) {
        const int32_t x = strip * kCols + (lane & (kCols - 1)), y = group * kRows + lane / kCols;
        const int32_t q = y * p.w4 + x;  // below 2^26
        bits = 0u;
        if (x < p.w4 && y < p.h && LCL_IN(4 * (int64_t)q + 3, p.n_texels)) {
            T = __ldcs(reinterpret_cast<const uint4 *>(p.tri) + q);
            V.load(p.data, q);
            if (p.zones) Z.load(p.zones, q);
            bits = (__ldg(p.mask + (q >> 3)) & __ldg(p.cover + (q >> 3))) >> ((q & 7) * 4);
        }
    };

    StatsRun run[2];
    run_reset(run[0]);
    run_reset(run[1]);
    run[0].zone = run[1].zone = kNone;
    int base = kF32 ? 1 : KIND == kKindFloat ? 126 : 150;  // float32: follows the values met; others: fixed
    int since = 0;                                          // steps since the runs were last empty
    // Run i's sums into the table; every lane of the warp calls it.
    auto flush = [&](int i) {
        StatsRun &r = run[i];
        const uint32_t cnt = __reduce_add_sync(0xffffffffu, r.cnt);
        if (cnt) {
            const __int128 area = warp_sum_i64((long long)r.area);
            const uint32_t kmin = __reduce_min_sync(0xffffffffu, r.kmin), kmax = __reduce_max_sync(0xffffffffu, r.kmax);
            const __int128 sum = warp_sum_i64(r.s), wsum = warp_sum_i96(r.w);
            if (lane == 0 && LCL_IN(r.zone, p.n_labels))
                acc_add(tab + r.zone, cnt, (unsigned long long)area, dkey(key_value<S, KIND>(kmin)),
                        dkey(key_value<S, KIND>(kmax)), i128_to_double(sum, base - 150), i128_to_double(wsum, base - 150));
        }
        run_reset(r);
    };
    for (int32_t u = warp; u < n_units; u += n_warps) {
    const int32_t strip = u % n_strips, g0 = u / n_strips * per, g1 = min(n_groups, g0 + per);
    if (g0 < g1) load(strip, g0);
    for (int32_t g = g0; g < g1; ++g) {
        const uint32_t ts[4] = {T.x, T.y, T.z, T.w};
        uint32_t v[4], z[4], ok = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = V.get(k);
            z[k] = p.zones ? Z.get(k) : 0u;
        }
        const uint32_t vb = bits;
        // weights (a texel whose triangle is its left neighbour's shares that one's)
        unsigned long long w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = ts[k] < ntri && (k == 0 || ts[k] != ts[k - 1]) ? __ldg(p.area_w + ts[k]) : 0ull;
        if (g + 1 < g1) load(strip, g + 1);
        uint32_t emax = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            bool good = ((vb >> k) & 1u) && ts[k] < ntri && z[k] < p.n_labels;
            if (KIND == kKindFloat) {
                if (S == 2) v[k] = __float_as_uint(__half2float(__ushort_as_half((unsigned short)v[k])));
                const uint32_t mag = v[k] & 0x7FFFFFFFu;
                good = good && mag <= 0x7F800000u;  // not NaN
                if (mag == 0u) v[k] = 0u;           // -0 counts as +0
                if (kF32 && good && mag < 0x7F800000u) emax = max(emax, mag >> 23);
            }
            ok |= (good ? 1u : 0u) << k;
        }
        const int top = kF32 ? (int)__reduce_max_sync(0xffffffffu, emax) : 0;  // 0: no normal value
        ++since;
        if (since > kRunTexels / 4 ||
            (kF32 && (top > base + kWindow ||
                      (top != 0 && base > 1 && top < base + kHeadroom - kFallen && since > kFallSteps)))) {  // uniform
            flush(0);
            flush(1);
            since = 1;
            if (kF32 && top != 0) base = max(top - kHeadroom, 1);
        }
#pragma unroll
        for (int k = 1; k < 4; ++k)
            if (ts[k] == ts[k - 1]) w[k] = w[k - 1];
        // adds the texels take0 and take1 to the lane's shares of the two runs (with1: some lane has a take1)
        auto add = [&](uint32_t take0, uint32_t take1, bool with1) {
            uint32_t miss = 0u;  // texels whose values do not fit the unit
            run[0].cnt += __popc(take0);
            run[1].cnt += __popc(take1);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool t0 = (take0 >> k) & 1u, t1 = (take1 >> k) & 1u;
                const uint32_t key = vkey<S, KIND>(v[k]);
                long long f;          // the value in units
                uint32_t b0, b1, b2;  // weight x value, 96 bits
                if (KIND == kKindFloat) {
                    // the value is m 2^sh units
                    const uint32_t e = (v[k] >> 23) & 0xFFu;
                    int32_t m = (int32_t)((v[k] & 0x7FFFFFu) | 0x800000u);
                    int sh = (int)e - base;
                    if (!kF32 && sh < 0) m >>= min(-sh, 31), sh = 0;  // float16: zeros are shifted out
                    const bool fits = (uint32_t)sh < 255u - (uint32_t)base;  // else below the window, zero, or infinite
                    m = (int32_t)v[k] < 0 ? -m : m;
                    m = fits && (kF32 || v[k] != 0u) ? m : 0;
                    sh = fits ? sh : 0;
                    f = (long long)m * (long long)(1 << sh);
                    // |m w| < 2^59: weight in parts of 30 and 5 bits, so that signed 32-bit products do
                    const long long pw = (long long)m * (int32_t)((uint32_t)w[k] & 0x3FFFFFFFu) +
                                         (long long)(m * (int32_t)(w[k] >> 30)) * (1 << 30);
                    const uint32_t lo = (uint32_t)pw, hi = (uint32_t)(pw >> 32);
                    b0 = lo << sh;
                    b1 = __funnelshift_l(lo, hi, sh);
                    b2 = __funnelshift_l(hi, (uint32_t)((int32_t)hi >> 31), sh);
                    if (!fits && v[k] != 0u) miss |= 1u << k;
                } else {
                    f = KIND == kKindSigned ? (long long)sext<S>(v[k]) : (long long)v[k];
                    if (S == 4) {
                        const __int128 fw = (__int128)f * (long long)w[k];
                        b0 = (uint32_t)fw;
                        b1 = (uint32_t)(fw >> 32);
                        b2 = (uint32_t)(fw >> 64);
                    } else {
                        const long long fw = f * (long long)w[k];
                        b0 = (uint32_t)fw;
                        b1 = (uint32_t)(fw >> 32);
                        b2 = (uint32_t)(fw >> 63);
                    }
                }
                auto acc = [&](StatsRun &r, bool t) {
                    if (!t) return;
                    r.kmin = min(r.kmin, key);
                    r.kmax = max(r.kmax, key);
                    r.area += w[k];
                    r.s += f;
                    add96(r.w, b0, b1, b2);
                };
                acc(run[0], t0);
                if (with1) acc(run[1], t1);
            }
            if (kFloat) {  // rare: a loop, so that its code stands once and takes few registers
#pragma unroll 1
                for (miss &= take0 | take1; miss; miss &= miss - 1u) {
                    const int k = __ffs(miss) - 1;
                    const bool b = (take0 >> k) & 1u;
                    outs_add(outs, b ? run[0].zone : run[1].zone, k & 2 ? (k & 1 ? v[3] : v[2]) : (k & 1 ? v[1] : v[0]),
                             k & 2 ? (k & 1 ? w[3] : w[2]) : (k & 1 ? w[1] : w[0]), tab);
                }
            }
        };
        uint32_t in0 = 0u, in1 = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t b = ok & (1u << k);
            if (z[k] == run[0].zone) in0 |= b;
            else if (z[k] == run[1].zone) in1 |= b;
        }
        uint32_t odd = ok & ~(in0 | in1);
        bool taken = false;  // a run has changed its zone
        // a zone not yet among the runs' takes over one that the step does not use (any more)
        auto take_over = [&](int i, uint32_t &in) {
            StatsRun &r = run[i];
            const uint32_t bal = __ballot_sync(0xffffffffu, odd != 0u);
            if (!bal || __any_sync(0xffffffffu, in != 0u)) return;  // uniform
            uint32_t last = kNone;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((odd >> k) & 1u) last = z[k];
            flush(i);
            taken = true;
            r.zone = __shfl_sync(0xffffffffu, last, 31 - __clz(bal));
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (((odd >> k) & 1u) && z[k] == r.zone) in |= 1u << k;
            odd &= ~in;
        };
        for (int round = 0; round < kZoneRounds; ++round) {
            take_over(0, in0);
            take_over(1, in1);
            if (__any_sync(0xffffffffu, (in0 | in1) != 0u)) add(in0, in1, __any_sync(0xffffffffu, in1 != 0u));
            in0 = in1 = 0u;
            if (!__any_sync(0xffffffffu, odd != 0u)) break;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)  // zones of a few texels: one by one, the lanes side by side
            if ((odd >> k) & 1u) stats_single<S, KIND>(tab, p.n_labels, z[k], v[k], w[k]);
        if (kFloat && taken) outs_end(outs, tab);  // uniform
    }
    }
    flush(0);
    flush(1);
    if (kFloat) outs_end(outs, tab);
    if (SMEM) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < p.n_labels; i += blockDim.x) {
            const ZoneAcc &a = sh_zone[i];
            if (a.count == 0) continue;
            acc_add(p.out + i, a.count, a.area, a.kmin, a.kmax, a.sum, a.wsum);
        }
    }
}

int stream_grid(int64_t work, int ctas_per_sm = 8) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sm_count() * ctas_per_sm, (work + kThreads - 1) / kThreads));
}

template <int S, int KIND>
void launch_arith(const ArithArgs &p, cudaStream_t st) {
    k_num_arith<S, KIND><<<stream_grid(p.n_chunks, ArithShape<KIND>::kCtas), kThreads, 0, st>>>(p);
}

template <int S, int KIND, int LB>
void launch_select(const SelectArgs &p, cudaStream_t st) {
    k_num_select<S, KIND, LB><<<stream_grid(p.n_chunks), kThreads, 0, st>>>(p);
}

template <int S, int KIND, int ZB, bool SMEM>
void launch_stats_smem(const StatsArgs &p, size_t shb, cudaStream_t st) {
    auto kernel = k_num_stats<S, KIND, ZB, SMEM>;
    constexpr size_t kOuts = KIND == kKindFloat ? sizeof(OutSums) : 0;
    if (SMEM && shb + kOuts > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shb);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, shb) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int64_t threads = (int64_t)((p.w4 + 7) / 8) * ((p.h + 3) / 4) / kStatsSteps * 32 + 32;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)sm_count() * per_sm,
                                                                 (threads + kThreads - 1) / kThreads));
    kernel<<<grid, kThreads, shb, st>>>(p);
}

template <int S, int KIND, int ZB>
void launch_stats(const StatsArgs &p, cudaStream_t st) {
    if (p.n_labels <= kSmemZones)
        launch_stats_smem<S, KIND, ZB, true>(p, (size_t)p.n_labels * sizeof(ZoneAcc), st);
    else
        launch_stats_smem<S, KIND, ZB, false>(p, 0, st);
}

template <int S, int KIND>
void launch_stats_z(const StatsArgs &p, int zb, cudaStream_t st) {
    if (zb == 2) launch_stats<S, KIND, 2>(p, st);
    else launch_stats<S, KIND, 1>(p, st);
}

}  // namespace

lcl_status numeric_arith_impl(const lcl_atlas *atlas, int type, const void *a, const uint32_t *ma, const void *b,
                              const uint32_t *mb, uint32_t b_value, void *out, uint32_t *mout, int op,
                              cudaStream_t st) {
    ArithArgs p;
    p.a = static_cast<const uint4 *>(a);
    p.b = static_cast<const uint4 *>(b);
    p.out = static_cast<uint4 *>(out);
    p.ma = ma;
    p.mb = mb;
    p.cover = atlas->cover;
    p.mout = mout;
    p.b_value = b_value;
    p.op = op;
    p.n_texels = (int64_t)atlas->width * atlas->height;
    const int bytes = type & 15;
    p.n_chunks = ((p.n_texels >> 5) << 5) * bytes / 16;
    switch (type) {
    case LCL_NUM_U8: launch_arith<1, kKindUnsigned>(p, st); break;
    case LCL_NUM_I8: launch_arith<1, kKindSigned>(p, st); break;
    case LCL_NUM_U16: launch_arith<2, kKindUnsigned>(p, st); break;
    case LCL_NUM_I16: launch_arith<2, kKindSigned>(p, st); break;
    case LCL_NUM_U32: launch_arith<4, kKindUnsigned>(p, st); break;
    case LCL_NUM_I32: launch_arith<4, kKindSigned>(p, st); break;
    case LCL_NUM_F16: launch_arith<2, kKindFloat>(p, st); break;
    default: launch_arith<4, kKindFloat>(p, st); break;
    }
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "lcl_numeric_arith launch");
    return LCL_OK;
}

lcl_status numeric_select_impl(const lcl_atlas *atlas, int type, const void *data, const uint32_t *mask, int cmp,
                               uint32_t threshold, void *layer, int label_bytes, uint32_t label, uint64_t *hits,
                               cudaStream_t st) {
    SelectArgs p;
    p.data = static_cast<const uint4 *>(data);
    p.mask = mask;
    p.cover = atlas->cover;
    p.layer = layer;
    p.threshold = threshold;
    p.label = label;
    p.cmp = cmp;
    p.n_texels = (int64_t)atlas->width * atlas->height;
    p.n_chunks = p.n_texels * (type & 15) / 16;
    p.hits = reinterpret_cast<unsigned long long *>(hits);
    if (hits) cudaMemsetAsync(hits, 0, sizeof(uint64_t), st);
#define LCL_SEL(S, K)                                                          \
    do {                                                                       \
        if (label_bytes == 1) launch_select<S, K, 1>(p, st);                   \
        else launch_select<S, K, 2>(p, st);                                    \
    } while (0)
    switch (type) {
    case LCL_NUM_U8: LCL_SEL(1, kKindUnsigned); break;
    case LCL_NUM_I8: LCL_SEL(1, kKindSigned); break;
    case LCL_NUM_U16: LCL_SEL(2, kKindUnsigned); break;
    case LCL_NUM_I16: LCL_SEL(2, kKindSigned); break;
    case LCL_NUM_U32: LCL_SEL(4, kKindUnsigned); break;
    case LCL_NUM_I32: LCL_SEL(4, kKindSigned); break;
    case LCL_NUM_F16: LCL_SEL(2, kKindFloat); break;
    default: LCL_SEL(4, kKindFloat); break;
    }
#undef LCL_SEL
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "lcl_numeric_select launch");
    return LCL_OK;
}

lcl_status numeric_stats_impl(const lcl_atlas *atlas, int type, const void *data, const uint32_t *mask,
                              const void *zones, int zone_bytes, uint32_t n_labels, lcl_zone_stats *out,
                              cudaStream_t st) {
    StatsArgs p;
    p.data = data;
    p.mask = mask;
    p.cover = atlas->cover;
    p.tri = atlas->tri;
    p.area_w = reinterpret_cast<const unsigned long long *>(atlas->area_w);
    p.zones = zones;
    p.n_labels = n_labels;
    p.n_texels = (int64_t)atlas->width * atlas->height;
    p.n_tri = atlas->n_tri;
    p.w4 = atlas->width / 4;
    p.h = atlas->height;
    p.out = reinterpret_cast<ZoneAcc *>(out);
    const unsigned zg = std::max(1u, std::min(1024u, (n_labels + kThreads - 1) / kThreads));
    k_stats_init<<<zg, kThreads, 0, st>>>(p.out, n_labels);
    switch (type) {
    case LCL_NUM_U8: launch_stats_z<1, kKindUnsigned>(p, zone_bytes, st); break;
    case LCL_NUM_I8: launch_stats_z<1, kKindSigned>(p, zone_bytes, st); break;
    case LCL_NUM_U16: launch_stats_z<2, kKindUnsigned>(p, zone_bytes, st); break;
    case LCL_NUM_I16: launch_stats_z<2, kKindSigned>(p, zone_bytes, st); break;
    case LCL_NUM_U32: launch_stats_z<4, kKindUnsigned>(p, zone_bytes, st); break;
    case LCL_NUM_I32: launch_stats_z<4, kKindSigned>(p, zone_bytes, st); break;
    case LCL_NUM_F16: launch_stats_z<2, kKindFloat>(p, zone_bytes, st); break;
    default: launch_stats_z<4, kKindFloat>(p, zone_bytes, st); break;
    }
    k_stats_final<<<zg, kThreads, 0, st>>>(p.out, n_labels);
    count_launches(3);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "lcl_numeric_stats launch");
    return LCL_OK;
}

}  // namespace lcl
