// spheres.cu -- sphere strokes without texture padding, on label and numeric layers
// (arXiv 2501.14807, Section 4.3.1: the selected value is stored in the texels that survive).
//
// Applying a call's strokes one by one leaves each texel with the value of the newest stroke that
// selects it, and a stroke's hit count does not depend on the others.  So one launch takes up to
// kManyStrokes strokes: it culls, tests and writes in one pass over the tiles, each texel is written
// at most once and a tile's positions are read once per launch however many strokes cross it.
//
// A CTA takes a block of up to 8 x 4 tiles (block_shape) in three steps, its warps in step:
//  1. the strokes are tested against the union of the tiles' boxes, a stroke per thread, and those
//     that can reach it are listed in shared memory, in order;
//  2. a warp per tile tests 32 listed strokes at a time against the tile's box: the ballots are the
//     masks of the strokes that reach the tile and of those that contain it;
//  3. tiles that no sphere's surface crosses are written from the coverage bits alone, with the value
//     of the newest stroke containing them (their hit counts come from the box's covered count); of
//     the others, a warp takes 32 quads at a time and tests the crossing strokes newest first; the
//     newest containing stroke gives the texels left open their value.
// No candidate lists pass through memory, and a call needs ceil(n / kManyStrokes) launches, where a
// cull and an apply launch per 32 strokes (label layers) or one launch per stroke (numeric layers,
// single strokes) ran before.  Those stay where they are the faster ones, for few strokes on large textures
// (by_lists in select.cu).
//
// What bounds it: latency of the crossing tiles' loads, then issue of their 64-bit distance tests
// (38% of issue slots, 21% of DRAM at 4096^2).  Measured on GB300, per call, before -> after: 250
// strokes of 1-30% of the diagonal on 16384^2 u8 1000 -> 350 us; 625 of 0.1-5% on a 4096^2 u16 chart
// atlas 225 -> 97 us; 40 value strokes on 5004 x 3310 i16 190 -> 39 us; one stroke on 1024^2 17 -> 15 us
// (two launches instead of three; two runs of one side differ by as much).  Tried and slower: a tile per warp from the culling on (the warps
// of a CTA drift apart and wait at its end: 121 us at 4096^2), the next 32 quads' positions held in
// registers (64 registers, four CTAs per SM: 105 us), CTAs of 128 threads (twice the staging: 106-113
// us and 490 us at 16384^2), six CTAs per SM (40 registers: spills).
#include <algorithm>

#include "select_common.cuh"

namespace lcl {
namespace {

constexpr int kFewStrokes = 32;    // strokes per launch of the small variant (1 KB of arguments)
constexpr int kManyStrokes = 512;  // strokes per launch (16 KB of arguments, 24 KB of shared memory)
constexpr int kCta = 256;          // threads per CTA
constexpr int kWarps = kCta / 32;
constexpr int kBlockTiles = 32;  // tiles of a block, at most

struct __align__(16) Stroke {
    int32_t cx, cy, cz;
    uint32_t value;
    int64_t r2;
    uint32_t erase;  // numeric layers: 1 clears the mask bit
    uint32_t pad;
};
static_assert(sizeof(Stroke) == 32, "Stroke must be 32 bytes");

// How a launch cuts the texture: blocks of (1 << ux) x (1 << uy) tiles, or of one of the 1 << parts
// bands of rows of a single tile.
struct BlockShape {
    int32_t ux, uy, parts;
    int32_t blocks_x;
    uint32_t n_blocks;
};

template <int CAP>
struct StrokesArg {
    BlockShape u;
    int32_t n;
    int32_t rows;  // 32-texel row segments are whole coverage words (tile side >= 32, width a multiple of 32)
    Stroke s[CAP];
};

// Squared distances from the stroke's centre to the box's nearest and farthest points.  Centres lie
// in [-2^22, 2^22 + 2^21] and boxes in [0, 2^21), so coordinate differences fit in 32 bits.
__device__ __forceinline__ int64_t near2(const int4 &lo, const int4 &hi, const Stroke &s) {
    const int32_t ex = max(max(lo.x - s.cx, s.cx - hi.x), 0), ey = max(max(lo.y - s.cy, s.cy - hi.y), 0),
                  ez = max(max(lo.z - s.cz, s.cz - hi.z), 0);
    return (int64_t)ex * ex + (int64_t)ey * ey + (int64_t)ez * ez;
}
__device__ __forceinline__ int64_t far2(const int4 &lo, const int4 &hi, const Stroke &s) {
    const int32_t fx = max(s.cx - lo.x, hi.x - s.cx), fy = max(s.cy - lo.y, hi.y - s.cy),
                  fz = max(s.cz - lo.z, hi.z - s.cz);
    return (int64_t)fx * fx + (int64_t)fy * fy + (int64_t)fz * fz;
}

// A quad's four texels selected by the stroke (bit k: texel k), among the covered ones `cov`.
// Uncovered texels (x = INT32_MIN) wrap around in the unsigned difference; `cov` drops them.
__device__ __forceinline__ uint32_t stroke_quad(const int4 &X, const int4 &Y, const int4 &Z, uint32_t cov, int32_t cx,
                                                int32_t cy, int32_t cz, int64_t r2) {
    const int32_t xs[4] = {X.x, X.y, X.z, X.w}, ys[4] = {Y.x, Y.y, Y.z, Y.w}, zs[4] = {Z.x, Z.y, Z.z, Z.w};
    uint32_t sel = 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int32_t dx = (int32_t)((uint32_t)xs[q] - (uint32_t)cx), dy = (int32_t)((uint32_t)ys[q] - (uint32_t)cy),
                      dz = (int32_t)((uint32_t)zs[q] - (uint32_t)cz);
        sel |= ((int64_t)dx * dx + (int64_t)dy * dy + (int64_t)dz * dz <= r2 ? 1u : 0u) << q;
    }
    return sel & cov;
}

// The values of a quad's texels, packed as they lie in the layer (sizeof(L) words).
template <typename L>
struct QuadValues {
    uint32_t w[sizeof(L)];
};

// Word j's lanes of the texels set in m (m a nibble, bit k: texel k), all ones.
template <typename L>
__device__ __forceinline__ uint32_t lanes_of(uint32_t m, int j) {
    if (sizeof(L) == 1) return ((m * 0x00204081u) & 0x01010101u) * 0xFFu;
    if (sizeof(L) == 2) return ((m >> (2 * j)) & 1u ? 0x0000FFFFu : 0u) | ((m >> (2 * j)) & 2u ? 0xFFFF0000u : 0u);
    return (m >> j) & 1u ? 0xFFFFFFFFu : 0u;
}

template <typename L>
__device__ __forceinline__ void put_value(QuadValues<L> &v, uint32_t m, uint32_t value) {
    const uint32_t rep = sizeof(L) == 1 ? value * 0x01010101u : sizeof(L) == 2 ? value * 0x00010001u : value;
#pragma unroll
    for (int j = 0; j < (int)sizeof(L); ++j) {
        const uint32_t b = lanes_of<L>(m, j);
        v.w[j] = (v.w[j] & ~b) | (rep & b);
    }
}

// What step 2 found out about a tile.
struct __align__(16) TileState {
    int32_t newest;  // list place of the newest stroke containing the tile, -1: none
    int32_t place;   // in the block
    int32_t tx, ty;
};

// A lane's quad: its positions and, for layers of one or two bytes, the values it holds, which a store
// of some of its texels puts back (loaded beside the positions, as waiting for them at the store costs
// a second trip to memory).
template <typename L>
struct Quad {
    int32_t l;  // first texel, -1: none
    int4 X, Y, Z;
    uint32_t old[sizeof(L) == 4 ? 1 : sizeof(L)];
};

template <typename L>
__device__ __forceinline__ void load_old(const L *layer, Quad<L> &v) {
    if constexpr (sizeof(L) == 1) {
        v.old[0] = *reinterpret_cast<const uint32_t *>(layer + v.l);
    } else if constexpr (sizeof(L) == 2) {
        const uint2 o = *reinterpret_cast<const uint2 *>(layer + v.l);
        v.old[0] = o.x;
        v.old[1] = o.y;
    }
}

// Writes the values of the quad's texels set in m (m != 0).
template <typename L>
__device__ __forceinline__ void store_quad(L *layer, const Quad<L> &v, uint32_t m, const QuadValues<L> &val) {
    if constexpr (sizeof(L) == 1) {
        const uint32_t b = lanes_of<L>(m, 0);
        *reinterpret_cast<uint32_t *>(layer + v.l) = (v.old[0] & ~b) | (val.w[0] & b);
    } else if constexpr (sizeof(L) == 2) {
        const uint32_t b0 = lanes_of<L>(m, 0), b1 = lanes_of<L>(m, 1);
        *reinterpret_cast<uint2 *>(layer + v.l) =
            make_uint2((v.old[0] & ~b0) | (val.w[0] & b0), (v.old[1] & ~b1) | (val.w[1] & b1));
    } else if (m == 0xFu) {
        *reinterpret_cast<uint4 *>(layer + v.l) = make_uint4(val.w[0], val.w[1], val.w[2], val.w[3]);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (m & (1u << k)) layer[v.l + k] = val.w[k];
    }
}

template <typename L, bool NUM, int CAP>
__global__ void __launch_bounds__(kCta, 5) k_spheres(AtlasDev a, L *__restrict__ layer,
                                                         uint32_t *__restrict__ mask,
                                                         const __grid_constant__ StrokesArg<CAP> g,
                                                         uint32_t *next_block, unsigned long long *hits) {
    constexpr int kWords = CAP / 32;
    __shared__ Stroke s_st[CAP];
    __shared__ uint32_t s_hits[CAP];              // below 2^28 texels per launch
    __shared__ uint32_t s_reach[kWords];          // strokes that reach the block, a bit each
    __shared__ uint16_t s_list[CAP];              // the same as a list, in order
    __shared__ uint2 s_mask[kBlockTiles][kWords]; // per tile and 32 listed strokes: cross the tile, contain it
    __shared__ TileState s_crossed[kBlockTiles], s_inside[kBlockTiles];  // tiles to test, tiles only contained
    __shared__ uint32_t s_n_crossed, s_n_inside, s_next;
    {
        // The strokes are read through their generic address: threads reading different places of
        // the constant bank are served one after another, generic loads are coalesced.
        const int4 *src = reinterpret_cast<const int4 *>(g.s);
        asm volatile("" : "+l"(src));
        for (int k = threadIdx.x; k < 2 * g.n; k += kCta) reinterpret_cast<int4 *>(s_st)[k] = src[k];
        for (int k = threadIdx.x; k < g.n; k += kCta) s_hits[k] = 0u;
    }
    __syncthreads();
    pdl_wait();
    pdl_allow_next();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n_tex = (int64_t)a.w * a.h, n_tiles = (int64_t)a.tiles_x * a.tiles_y;
    (void)n_tex;
    (void)n_tiles;
    const int tlog = __ffs(a.T) - 1, qlog = tlog - 2;             // texels, quads per tile row
    const int band_log = tlog - g.u.parts;                        // tile rows per band
    const int sub_log = max(band_log + qlog - 5, 0);              // 32-quad pieces per tile (band)
    const int32_t n_quads = 1 << (band_log + qlog);
    const int n_stroke_words = (g.n + 31) >> 5;
    // thread 0 fetches the number of the block after the next one, a block ahead of its use
    uint32_t fetched = blockIdx.x - gridDim.x;
    for (uint32_t u = blockIdx.x; u < g.u.n_blocks;) {  // uniform over the CTA
        if (threadIdx.x == 0) {
            s_next = fetched + 2 * gridDim.x;
            if (next_block) fetched = atomicAdd(next_block, 1u);
            else fetched += gridDim.x;
            s_n_crossed = s_n_inside = 0u;
        }
        const int32_t band = (int32_t)(u & ((1u << g.u.parts) - 1u)), blk = (int32_t)(u >> g.u.parts);
        const int32_t by = blk / g.u.blocks_x, bx = blk - by * g.u.blocks_x;
        const int32_t tx = (bx << g.u.ux) + (lane & ((1 << g.u.ux) - 1)), ty = (by << g.u.uy) + (lane >> g.u.ux);
        // the lane's tile of the block; an empty tile's box is the neutral element of the union
        int4 lo = make_int4(INT32_MAX, INT32_MAX, INT32_MAX, 0), hi = make_int4(INT32_MIN, INT32_MIN, INT32_MIN, 0);
        if (lane < (1 << (g.u.ux + g.u.uy)) && tx < a.tiles_x && ty < a.tiles_y &&
            LCL_IN((int64_t)ty * a.tiles_x + tx, n_tiles)) {
            const int4 *b = reinterpret_cast<const int4 *>(a.tile_box + 8 * ((int64_t)ty * a.tiles_x + tx));
            lo = __ldg(b);
            hi = __ldg(b + 1);
        }
        const uint32_t tiles = __ballot_sync(0xffffffffu, lo.w > 0);
        {
            int4 ulo, uhi;
            ulo.x = __reduce_min_sync(0xffffffffu, lo.x);
            ulo.y = __reduce_min_sync(0xffffffffu, lo.y);
            ulo.z = __reduce_min_sync(0xffffffffu, lo.z);
            uhi.x = __reduce_max_sync(0xffffffffu, hi.x);
            uhi.y = __reduce_max_sync(0xffffffffu, hi.y);
            uhi.z = __reduce_max_sync(0xffffffffu, hi.z);
            for (int i = warp; i < n_stroke_words; i += kWarps) {
                const int k = 32 * i + lane;
                bool reach = false;
                if (tiles && k < g.n) {
                    const Stroke s = s_st[k];
                    reach = near2(ulo, uhi, s) <= s.r2;
                }
                const uint32_t m = __ballot_sync(0xffffffffu, reach);
                if (lane == 0) s_reach[i] = m;
            }
        }
        __syncthreads();
        u = s_next;
        // lane i counts the strokes of word i and of the words before it
        const uint32_t word = lane < n_stroke_words ? s_reach[lane] : 0u;
        int before = __popc(word);
#pragma unroll
        for (int o = 1; o < kWords; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, before, o);
            if (lane >= o) before += t;
        }
        const int n_list = __shfl_sync(0xffffffffu, before, kWords - 1);
        before -= __popc(word);
        for (int i = warp; i < n_stroke_words; i += kWarps) {
            const uint32_t m = __shfl_sync(0xffffffffu, word, i);
            const int b = __shfl_sync(0xffffffffu, before, i);
            if ((m >> lane) & 1u) s_list[b + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(32 * i + lane);
        }
        __syncthreads();
        if (n_list == 0) continue;  // uniform over the CTA
        const int n_words = (n_list + 31) >> 5;
        // masks, a warp per tile
        for (int t = warp; t < kBlockTiles; t += kWarps) {
            if (!((tiles >> t) & 1u)) continue;  // uniform over the warp
            int4 tlo, thi;
            tlo.x = __shfl_sync(0xffffffffu, lo.x, t);
            tlo.y = __shfl_sync(0xffffffffu, lo.y, t);
            tlo.z = __shfl_sync(0xffffffffu, lo.z, t);
            tlo.w = __shfl_sync(0xffffffffu, lo.w, t);
            thi.x = __shfl_sync(0xffffffffu, hi.x, t);
            thi.y = __shfl_sync(0xffffffffu, hi.y, t);
            thi.z = __shfl_sync(0xffffffffu, hi.z, t);
            int newest = -1;
            bool crossed = false;
            for (int i = 0; i < n_words; ++i) {
                bool reach = false, inside = false;
                const int j = 32 * i + lane;
                if (j < n_list) {
                    const int k = s_list[j];
                    const Stroke s = s_st[k];
                    reach = near2(tlo, thi, s) <= s.r2;
                    inside = reach && far2(tlo, thi, s) <= s.r2;
                    // every covered texel of the tile counts for a stroke containing it
                    if (inside && hits && band == 0) atomicAdd(&s_hits[k], (uint32_t)tlo.w);
                }
                const uint32_t in = __ballot_sync(0xffffffffu, inside);
                const uint32_t c = __ballot_sync(0xffffffffu, reach) & ~in;
                if (lane == 0) s_mask[t][i] = make_uint2(c, in);
                if (in) newest = 32 * i + 31 - __clz(in);
                // without hit counts only crossing strokes newer than `newest` matter
                if (hits) crossed = crossed || c;
                else crossed = (in ? false : crossed) || (c && 32 * i + 31 - __clz(c) > newest);
            }
            if (lane == t) {  // the lane that holds this tile's place
                TileState st;
                st.newest = newest;
                st.place = t;
                st.tx = tx;
                st.ty = ty;
                if (crossed || (newest >= 0 && !g.rows)) s_crossed[atomicAdd(&s_n_crossed, 1u)] = st;
                else if (newest >= 0) s_inside[atomicAdd(&s_n_inside, 1u)] = st;
            }
        }
        __syncthreads();
        // 32-quad pieces of the tiles to test
        const int n_pieces = (int)s_n_crossed << sub_log;
        for (int piece = warp; piece < n_pieces; piece += kWarps) {  // uniform over the warp
            const TileState st = s_crossed[piece >> sub_log];
            const int32_t q = ((piece & ((1 << sub_log) - 1)) << 5) + lane;
            const int32_t x = (st.tx << tlog) + 4 * (q & ((1 << qlog) - 1));
            const int32_t y = (st.ty << tlog) + (band << band_log) + (q >> qlog);
            Quad<L> v;
            v.l = -1;
            v.X = v.Y = v.Z = make_int4(INT32_MIN, INT32_MIN, INT32_MIN, INT32_MIN);  // no texel covered
            if (q < n_quads && x < a.w && y < a.h && LCL_IN((int64_t)y * a.w + x + 3, n_tex)) {
                v.l = y * a.w + x;  // below 2^28
                v.X = __ldg(reinterpret_cast<const int4 *>(a.px + v.l));
                v.Y = __ldg(reinterpret_cast<const int4 *>(a.py + v.l));
                v.Z = __ldg(reinterpret_cast<const int4 *>(a.pz + v.l));
                load_old<L>(layer, v);
            }
            const int newest = st.newest, t = st.place;
            const uint32_t cov = (v.X.x != INT32_MIN ? 1u : 0u) | (v.X.y != INT32_MIN ? 2u : 0u) |
                                 (v.X.z != INT32_MIN ? 4u : 0u) | (v.X.w != INT32_MIN ? 8u : 0u);
            uint32_t open = cov, erased = 0u;
            QuadValues<L> val;
#pragma unroll
            for (int q = 0; q < (int)sizeof(L); ++q) val.w[q] = 0u;
            for (int i = n_words - 1; i >= 0; --i) {  // newest first (uniform)
                uint32_t m = s_mask[t][i].x;
                if (!hits && 32 * i + 31 <= newest) break;  // older strokes change nothing
                while (m) {
                    const int b = 31 - __clz(m);
                    m &= ~(1u << b);
                    const int place = 32 * i + b;
                    if (!hits && place < newest) break;
                    const int k = s_list[place];
                    const Stroke s = s_st[k];
                    const uint32_t sel = stroke_quad(v.X, v.Y, v.Z, cov, s.cx, s.cy, s.cz, s.r2);
                    if (hits) {
                        const uint32_t c = __reduce_add_sync(0xffffffffu, __popc(sel));
                        if (lane == 0 && c) atomicAdd(&s_hits[k], c);
                    }
                    if (place > newest) {
                        const uint32_t nw = sel & open;
                        put_value<L>(val, nw, s.value);
                        if (NUM && s.erase) erased |= nw;
                        open &= ~nw;
                    }
                }
            }
            if (newest >= 0) {
                const Stroke &s = s_st[s_list[newest]];
                put_value<L>(val, open, s.value);
                if (NUM && s.erase) erased |= open;
                open = 0u;
            }
            const uint32_t written = cov & ~open;
            if (written && LCL_IN(v.l + 3, n_tex)) store_quad<L>(layer, v, written, val);
            if (NUM) {
                if (g.rows) {  // the eight lanes of a mask word merge their bits
                    const int sh = (int)(v.l & 31);
                    uint32_t set = v.l >= 0 ? (written & ~erased) << sh : 0u;
                    uint32_t clr = v.l >= 0 ? (written & erased) << sh : 0u;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        set |= __shfl_xor_sync(0xffffffffu, set, o);
                        clr |= __shfl_xor_sync(0xffffffffu, clr, o);
                    }
                    if ((lane & 7) == 0 && (set | clr) && LCL_IN(v.l >> 5, (n_tex + 31) >> 5)) {
                        uint32_t *mp = mask + (v.l >> 5);
                        *mp = (*mp & ~clr) | set;
                    }
                } else if (written) {
                    ValMask vm;
                    vm.bits = mask;
                    vm.set = 1u;
                    if (written & ~erased) valid_update_atomic(vm, v.l, written & ~erased, n_tex);
                    vm.set = 0u;
                    if (written & erased) valid_update_atomic(vm, v.l, written & erased, n_tex);
                }
            }
        }
        // tiles only contained: a warp per tile, from the last warp down, a lane per 32-texel row segment
        for (int i = kWarps - 1 - warp; i < (int)s_n_inside; i += kWarps) {
            const TileState st = s_inside[i];
            const Stroke &s = s_st[s_list[st.newest]];
            const uint32_t value = s.value;
            const int wlog = tlog - 5;
            for (int32_t wi = lane; wi < (1 << (band_log + wlog)); wi += 32) {
                const int32_t x = (st.tx << tlog) + 32 * (wi & ((1 << wlog) - 1));
                const int32_t y = (st.ty << tlog) + (band << band_log) + (wi >> wlog);
                if (x >= a.w || y >= a.h) continue;  // x < w implies x + 31 < w
                const int64_t l = (int64_t)y * a.w + x;
                if (!LCL_IN(l + 31, n_tex)) continue;
                const uint32_t cov = __ldg(a.cover + (l >> 5));
                if (!cov) continue;
                store_word32<L>(layer, l, cov, value);
                if (NUM) {  // the segment's mask word belongs to this lane alone
                    uint32_t *mp = mask + (l >> 5);
                    *mp = s.erase ? (*mp & ~cov) : (*mp | cov);
                }
            }
        }
        __syncthreads();  // the block's lists and masks have been read
    }
    if (hits) {
        __syncthreads();
        for (int k = threadIdx.x; k < g.n; k += kCta)
            if (s_hits[k]) atomicAdd(hits + k, (unsigned long long)s_hits[k]);
    }
}

// Zeroes the block counters and the hit counts of a call.
__global__ void k_spheres_init(uint32_t *counters, int32_t n, unsigned long long *hits, int32_t n_hits) {
    pdl_wait();  // launched as a dependent: the previous grid no longer uses the counters
    pdl_allow_next();
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) counters[i] = 0u;
    if (hits && i < n_hits) hits[i] = 0ull;
}

// The blocks of a launch: several tiles, which share one list of strokes, as long as every CTA still
// gets four blocks; where there are fewer tiles than CTAs, bands of a tile's rows, of 32 quads (a
// quad per lane of a warp) at least.
BlockShape block_shape(const lcl_atlas *at, int64_t n_ctas) {
    BlockShape s;
    s.ux = s.uy = s.parts = 0;
    const int64_t tiles = (int64_t)at->tiles_x * at->tiles_y, quads = (int64_t)at->tile * at->tile / 4;
    while ((quads >> s.parts) > 32 && (tiles << (s.parts + 1)) <= n_ctas) ++s.parts;
    while (s.ux + s.uy < 5 && (tiles >> (s.ux + s.uy + 1)) >= 4 * n_ctas) {
        if (s.ux <= s.uy) ++s.ux;
        else ++s.uy;
    }
    s.blocks_x = (at->tiles_x + (1 << s.ux) - 1) >> s.ux;
    s.n_blocks = (uint32_t)(((int64_t)s.blocks_x * ((at->tiles_y + (1 << s.uy) - 1) >> s.uy)) << s.parts);
    return s;
}

template <typename L, bool NUM, int CAP>
cudaError_t launch_spheres(const lcl_atlas *atlas, const AtlasDev &a, L *layer, uint32_t *mask,
                           const lcl_sphere *strokes, int32_t n, unsigned long long *hits, uint32_t *counters,
                           cudaStream_t st) {
    const int grid_max = resident_per_sm(k_spheres<L, NUM, CAP>, kCta) * sm_count();
    static thread_local StrokesArg<CAP> g;  // kept off the stack
    g.u = block_shape(atlas, grid_max);
    g.rows = (a.T >= 32 && (a.w & 31) == 0) ? 1 : 0;
    const int grid = (int)std::min<int64_t>(grid_max, g.u.n_blocks);
    const int32_t n_launches = (n + CAP - 1) / CAP;
    // a block per CTA needs no counter; otherwise CTAs fetch blocks as they finish
    const bool fetch = g.u.n_blocks > (uint32_t)grid;
    cudaError_t e = cudaSuccess;
    if (fetch || hits) {
        const int32_t n_zero = std::max(fetch ? n_launches : 0, hits ? n : 0);
        e = launch_pdl(k_spheres_init, dim3((n_zero + kThreads - 1) / kThreads), st, counters, fetch ? n_launches : 0,
                       hits, n);
        count_launches(1);
    }
    for (int32_t i = 0; i < n_launches && e == cudaSuccess; ++i) {
        const int32_t k0 = i * CAP;
        g.n = std::min(CAP, n - k0);
        for (int32_t k = 0; k < g.n; ++k) {
            const lcl_sphere &in = strokes[k0 + k];
            Stroke &s = g.s[k];
            s.cx = in.cx;
            s.cy = in.cy;
            s.cz = in.cz;
            s.r2 = in.r2 > kR2Cap ? kR2Cap : in.r2;
            s.erase = NUM && (in.flags & LCL_ERASE) ? 1u : 0u;
            s.value = s.erase ? 0u : in.label;
            s.pad = 0u;
        }
        e = launch_pdl_shape(k_spheres<L, NUM, CAP>, dim3(grid), dim3(kCta), st, a, layer, mask, g,
                             fetch ? counters + i : nullptr, hits ? hits + k0 : nullptr);
        count_launches(1);
    }
    return e;
}

}  // namespace

template <typename L, bool NUM>
cudaError_t spheres_run(const lcl_atlas *atlas, L *layer, uint32_t *mask, const lcl_sphere *strokes, int32_t n,
                        unsigned long long *hits, uint32_t *counters, cudaStream_t st) {
    const AtlasDev a = dev_view(atlas);
    return n <= kFewStrokes ? launch_spheres<L, NUM, kFewStrokes>(atlas, a, layer, mask, strokes, n, hits, counters, st)
                            : launch_spheres<L, NUM, kManyStrokes>(atlas, a, layer, mask, strokes, n, hits, counters, st);
}

template cudaError_t spheres_run<uint8_t, false>(const lcl_atlas *, uint8_t *, uint32_t *, const lcl_sphere *, int32_t,
                                                 unsigned long long *, uint32_t *, cudaStream_t);
template cudaError_t spheres_run<uint16_t, false>(const lcl_atlas *, uint16_t *, uint32_t *, const lcl_sphere *,
                                                  int32_t, unsigned long long *, uint32_t *, cudaStream_t);
template cudaError_t spheres_run<uint8_t, true>(const lcl_atlas *, uint8_t *, uint32_t *, const lcl_sphere *, int32_t,
                                                unsigned long long *, uint32_t *, cudaStream_t);
template cudaError_t spheres_run<uint16_t, true>(const lcl_atlas *, uint16_t *, uint32_t *, const lcl_sphere *, int32_t,
                                                 unsigned long long *, uint32_t *, cudaStream_t);
template cudaError_t spheres_run<uint32_t, true>(const lcl_atlas *, uint32_t *, uint32_t *, const lcl_sphere *, int32_t,
                                                 unsigned long long *, uint32_t *, cudaStream_t);

}  // namespace lcl
