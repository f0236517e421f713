// batch.cu -- batched edits: many models, each with a queue of sphere and lasso strokes, edited
// by one cull launch and one persistent apply launch (capturable in a CUDA graph).
//
// The paper edits one layer of one model per operation (Section 4.3.1).  A server holding many
// models batches their queued strokes instead: the result must equal applying each model's
// strokes one by one, in queue order, so
//   k_batch_cull   gives every tile of every model a 64-bit mask of the model's queued strokes
//                  (queue order = bit order) whose conservative box test can reach the tile, and
//                  of those a `sure` mask (spheres containing the tile, lassos inside whose polygon
//                  it lies): a warp per four tiles of a row.  Tiles with a non-empty mask become
//                  work items (model, tile, masks);
//   k_batch_apply  takes units of one or more groups of 32 quads of an item from a work queue, a warp
//                  each.  A thread loads its four texels' positions once and evaluates the masked strokes
//                  from the newest down: the first stroke that selects a texel is the last one
//                  sequential application would have written there, so the texel is final and
//                  the thread stops once its four texels are final (or no stroke is left); each
//                  label word is written once.  Texture padding (Section 4.3.2) writes only
//                  uncovered texels, so for those the masked padded strokes are evaluated the
//                  same way (newest first, on the neighbours' positions), and a padded stroke's
//                  cull counts a tile whose 3 x 3 neighbourhood it may reach.
// Each texel belongs to one unit and one thread, so no two threads write a texel, and the label a
// texel receives is that of the newest stroke selecting it: the result is bit-identical to
// sequential single-stroke calls.
//
// The host uploads compact descriptors (models, strokes, each lasso's camera and polygon);
// k_batch_prep builds the lassos' culling boxes and y-band edge lists on the device, one warp per
// lasso.  Workspace layout and launch shape depend only on the limits (capacities) and the config,
// and the kernels read the batch's counts from the workspace header, so the launch is independent
// of the batch's contents: it can be captured once in a CUDA graph and replayed after each upload.
#include <cstring>

#include "select_common.cuh"

namespace lcl {
namespace {

struct BModel {
    AtlasDev a;
    void *layer;
    int32_t dtype_bytes;
    int32_t s0, ns;   // this model's strokes: [s0, s0 + ns) of the batch's stroke array, ns <= 64
    int32_t super0;   // first flattened super-tile of this model
};

struct BStroke {
    int32_t kind;     // LCL_STROKE_SPHERE or LCL_STROKE_LASSO
    int32_t lasso;    // index into the lasso array
    SphereArg sphere;
};

// Built on the device by k_batch_prep.  Every texel of a crossing tile goes through the edges of its y-band,
// so the edges have records (as in LassoShared) and the bands bit masks of them; with lists of bytes, and
// the records worked out from the vertices at each use, the batch at k_batch_apply took 859 us instead of 806.
struct BLasso : LassoHead {
    float4 rec[LCL_MAX_LASSO_VERTICES];  // {ay, by, lo, hi}
    uint2 band[kBands];                  // edges 0-31 and 32-63 of the band
    const float *depth;
    int32_t pad_r, pad_t;  // texture padding: kernel radius and outline thickness (0: none)
};
static_assert(sizeof(BLasso) % 16 == 0, "k_batch_prep copies it by 16-byte words");
constexpr size_t kBLassoRoom = 2792;  // bytes of the workspace per lasso, which programs may have stored
static_assert(sizeof(BLasso) <= kBLassoRoom, "lcl_batch_workspace_bytes");

// Kernels of batches whose limits hold no lassos leave out their code (LASSOS false).
template <typename F>
__device__ __forceinline__ void band_edges(const BLasso &L, int band, F f) {
    const uint2 b = L.band[band];
    for (uint32_t m = b.x; m; m &= m - 1) {
        const int e = __ffs(m) - 1;
        f(e, L.rec[e]);
    }
    for (uint32_t m = b.y; m; m &= m - 1) {
        const int e = 31 + __ffs(m);
        f(e, L.rec[e]);
    }
}

struct BLassoIn {  // what the host uploads per lasso
    float m[16];
    int32_t w_s, h_s;
    const float *depth;
    float poly[2 * LCL_MAX_LASSO_VERTICES];
    int32_t nv;
    uint32_t label;
    float bias;
    uint32_t flags;  // texture padding: radius = bits 0-3, thickness = bits 4-7
};

constexpr uint32_t kPadItem = 0x80000000u;  // bit of an item's tile: a stroke of its mask pads
struct BItem {
    uint32_t model, tile;
    unsigned long long mask;  // strokes that can write a texel of the tile
    unsigned long long sure;  // of those: spheres containing the tile's box (every covered texel
                              // selected) and unpadded lassos inside whose polygon the tile lies
};

// Capacities of a workspace's arrays (its limits), for the kernels' index checks.
struct BCaps {
    int32_t models, strokes, lassos, pad;
    int64_t supers, tiles;
};

// Can the stroke's descriptors be read: its index within the strokes and, for a lasso, the lasso's
// within the lassos (the debug build's checks; always true otherwise).
__device__ __forceinline__ bool stroke_in_bounds(const BStroke *strokes, int64_t si, const BCaps &caps) {
    if (!LCL_IN(si, caps.strokes)) return false;
    return strokes[si].kind == LCL_STROKE_SPHERE || LCL_IN(strokes[si].lasso, caps.lassos);
}

// Workspace header (first 256 bytes), uploaded with the descriptors; the counters are reset by
// k_batch_prep at every launch.
struct BHdr {
    int32_t n_models, n_strokes, n_lassos, n_supers;
    int32_t groups_log, tickets_log;  // of the largest tiles: groups of 32 quads, and tickets per item, powers of 2
    unsigned int n_items;          // written by k_batch_cull
    unsigned int next_cull;        // work queue of k_batch_cull
    unsigned long long next_unit;  // work queue of k_batch_apply
};

// Workspace: [hdr | models | strokes | lasso inputs | super-tile -> model] is uploaded (the
// staging holds its image); [lassos | items] is written by the kernels.  Another 16 bytes per tile are
// counted but not used, so that lcl_batch_workspace_bytes stays what programs may have stored.
struct BLayout {
    size_t hdr, models, strokes, lasso_in, super_model, upload, lassos, items, total;
};

BLayout b_layout(const lcl_batch_limits &lim) {
    BLayout L;
    L.hdr = 0;
    L.models = align256(sizeof(BHdr));
    L.strokes = L.models + align256((size_t)std::max(lim.models, 1) * sizeof(BModel));
    L.lasso_in = L.strokes + align256((size_t)std::max(lim.strokes, 1) * sizeof(BStroke));
    L.super_model = L.lasso_in + align256((size_t)std::max(lim.lassos, 1) * sizeof(BLassoIn));
    L.upload = L.super_model + align256((size_t)std::max<int64_t>(lim.supers, 1) * 4);
    L.lassos = L.upload;
    L.items = L.lassos + align256((size_t)std::max(lim.lassos, 1) * kBLassoRoom);
    L.total = L.items + align256((size_t)std::max<int64_t>(lim.tiles, 1) * sizeof(BItem)) +
              align256((size_t)std::max<int64_t>(lim.tiles, 1) * 16);
    return L;
}

__device__ __forceinline__ bool stroke_pads(const BStroke &st, const BLasso *lassos) {
    return st.kind == LCL_STROKE_SPHERE ? st.sphere.pad_r > 0 : lassos[st.lasso].pad_r > 0;
}

// Can lasso L select a texel of a box within r of box (bx, by) of a grid of nx x ny boxes (8 int32 each)?
// By an aligned group of 8 lanes.  With texture padding a texel may be written because a neighbour within
// 8 texels (at most one tile, and so one super-tile, away) is selected, so then r = 1.
__device__ __forceinline__ bool box_near(const BLasso &L, const int32_t *boxes, int32_t nx, int32_t ny, int32_t bx,
                                         int32_t by, int32_t r, const float *depth) {
    for (int32_t y = max(by - r, 0); y <= min(by + r, ny - 1); ++y)
        for (int32_t x = max(bx - r, 0); x <= min(bx + r, nx - 1); ++x) {
            if (!LCL_IN((int64_t)y * nx + x, (int64_t)nx * ny)) continue;
            const int4 *b = reinterpret_cast<const int4 *>(boxes + 8 * ((int64_t)y * nx + x));
            const int4 lo = b[0], hi = b[1];
            if (lo.w > 0 && box_may_touch_by<8>(L, lo, hi, depth)) return true;
        }
    return false;
}

constexpr int kPrepWarps = kThreads / 32;  // lassos per CTA of k_batch_prep
static_assert(kBands == 32, "k_batch_prep gives each y-band one lane");

// Resets the work counters and builds every lasso's argument, one warp per lasso:
// the lanes copy the vertices and reduce their bounding box, then lane b collects the edges of
// band b (the same predicate as the host builder).
__global__ void __launch_bounds__(kThreads) k_batch_prep(BHdr *hdr, const BLassoIn *__restrict__ in,
                                                         BLasso *__restrict__ out, BCaps caps) {
    pdl_allow_next();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        hdr->n_items = 0;
        hdr->next_cull = 0;
        hdr->next_unit = 0;
    }
    __shared__ BLasso s_arg[kPrepWarps];
    const int lane = threadIdx.x & 31;
    const int j = blockIdx.x * kPrepWarps + (int)(threadIdx.x / 32);
    if (j >= hdr->n_lassos) return;  // uniform over the warp
    if (!LCL_IN(j, caps.lassos)) return;
    (void)caps;
    const BLassoIn &L = in[j];
    BLasso &p = s_arg[threadIdx.x / 32];
    const int nv = L.nv;
    float x0 = INFINITY, x1 = -INFINITY, y0 = INFINITY, y1 = -INFINITY;
    for (int i = lane; i <= LCL_MAX_LASSO_VERTICES; i += 32) {  // vertices nv and on repeat vertex 0
        const float2 v = *reinterpret_cast<const float2 *>(L.poly + 2 * (i < nv ? i : 0));
        p.vx[i] = v.x;
        p.vy[i] = v.y;
        x0 = fminf(x0, v.x);
        x1 = fmaxf(x1, v.x);
        y0 = fminf(y0, v.y);
        y1 = fmaxf(y1, v.y);
    }
    for (int o = 16; o; o >>= 1) {
        x0 = fminf(x0, __shfl_xor_sync(0xffffffffu, x0, o));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, o));
        y0 = fminf(y0, __shfl_xor_sync(0xffffffffu, y0, o));
        y1 = fmaxf(y1, __shfl_xor_sync(0xffffffffu, y1, o));
    }
    if (lane < 16) p.m[lane] = L.m[lane];
    if (lane == 0) {
        lasso_arg_scalars(p, L.m, L.w_s, L.h_s, nv, L.label, L.bias);
        lasso_arg_box(p, x0, x1, y0, y1);
        p.depth = L.depth;
        p.pad_r = (int32_t)(L.flags & 15u);
        p.pad_t = (int32_t)((L.flags >> 4) & 15u);
    }
    __syncwarp();
    const float2 range = lasso_band_range(p, lane, lasso_band_height(p));
    unsigned long long has = 0ull;  // edges of band `lane`
    for (int e = 0; e < nv; ++e)
        if (lasso_band_has(p, range, e)) has |= 1ull << e;
    p.band[lane] = make_uint2((uint32_t)has, (uint32_t)(has >> 32));
    for (int e = lane; e < nv; e += 32) {
        const float2 r = edge_xrange(p.vx[e], p.vx[e + 1]);
        p.rec[e] = make_float4(p.vy[e], p.vy[e + 1], r.x, r.y);
    }
    __syncwarp();
    for (int i = lane; i < (int)(sizeof(BLasso) / 16); i += 32)
        reinterpret_cast<uint4 *>(&out[j])[i] = reinterpret_cast<const uint4 *>(&p)[i];
}

// Bit number n (from 0) of the set bits of m, which has more than n.
__device__ __forceinline__ int nth_bit(unsigned long long m, int n) {
    for (; n > 0; --n) m &= m - 1;
    return __ffsll((long long)m) - 1;
}

// OR of the lanes' values; every lane of the warp calls it.
__device__ __forceinline__ unsigned long long warp_or(unsigned long long v) {
    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)v), hi = __reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32));
    return (unsigned long long)hi << 32 | lo;
}

// The strokes that can write a texel of each tile.  A warp takes units of four tiles (neighbours in a row
// of a super-tile) from a work queue, 8 lanes per tile.  The warp first tests the model's lassos against
// the super-tile's box, four at a time; then each group of 8 lanes tests its tile: a lane per sphere, the
// whole group per lasso, so that the four groups go through the same lasso together.  A padded stroke
// counts a tile if it may reach any box of its 3 x 3 neighbourhood: a padded sphere tests the 18 boxes around a unit
// once each (with nine per tile a batch of 4 models of 2048^2 with tiles of 8 and 16 padded spheres took 489 us, of
// which the cull 257; now 262).  The queue evens out tiles under many
// large lassos; with a CTA per (super-tile, stroke) those ran on while the chip was idle (24 models of
// 512^2 to 2048^2, 48 spheres and 16 lassos each: 341 us with the compaction, now about 220; 3 models with
// 40 spheres each: 11.1 us and 8.5).  What is left is the latency of one warp's footprint scans.
constexpr int kCullTiles = 4;  // tiles of a unit
constexpr int kCullUnits = LCL_SUPER * LCL_SUPER / kCullTiles;
static_assert(LCL_SUPER % kCullTiles == 0 && kCullTiles == 4, "k_batch_cull: 8 lanes per tile");

__global__ void __launch_bounds__(kThreads, 4) k_batch_cull(BHdr *hdr, const BModel *__restrict__ models,
                                                            const BStroke *__restrict__ strokes,
                                                            const BLasso *__restrict__ lassos,
                                                            const uint32_t *__restrict__ super_model,
                                                            BItem *items, BCaps caps) {
    const int lane = threadIdx.x & 31, sub = lane & 7, group = lane / 8;
    pdl_wait();  // the counters are reset and the lassos built
    pdl_allow_next();
    const int64_t n_units = (int64_t)hdr->n_supers * kCullUnits;
    // a warp's first units are by its number, the others come from the queue, drawn one ahead
    const uint32_t n_warps = gridDim.x * (kThreads / 32);
    // Without lassos a unit is short, and a large model has more of them than the queue's one address serves
    // in time (4 spheres on 16384^2 with tiles of 8: 784 us with one unit per draw, now 630): several per draw then.
    const uint32_t chunk =
        hdr->n_lassos ? 1u : (uint32_t)max((int64_t)1, min((int64_t)16, n_units / (4 * (int64_t)n_warps)));
    uint32_t next = chunk * (blockIdx.x * (kThreads / 32) + threadIdx.x / 32);
    uint32_t u = 0u, end = 0u;
    for (;; ++u) {
        if (u == end) {
            u = __shfl_sync(0xffffffffu, next, 0);
            if (u >= n_units) break;  // uniform over the warp, as below
            end = min(u + chunk, (uint32_t)n_units);
            if (lane == 0) next = chunk * n_warps + atomicAdd(&hdr->next_cull, chunk);
        }
        const int32_t g = (int32_t)(u / kCullUnits), part = (int32_t)(u % kCullUnits);
        if (!LCL_IN(g, caps.supers)) break;
        const uint32_t mi = super_model[g];
        if (!LCL_IN(mi, caps.models)) continue;
        const BModel &M = models[mi];
        const AtlasDev &a = M.a;
        const int32_t sidx = g - M.super0;
        if (!LCL_IN(sidx, (int64_t)a.supers_x * a.supers_y)) continue;
        const int32_t sx = sidx % a.supers_x, sy = sidx / a.supers_x;
        const int32_t tx0 = sx * LCL_SUPER + part % (LCL_SUPER / kCullTiles) * kCullTiles, tx = tx0 + group;
        const int32_t ty = sy * LCL_SUPER + part / (LCL_SUPER / kCullTiles);
        if (tx0 >= a.tiles_x || ty >= a.tiles_y) continue;
        const int64_t n_tiles = (int64_t)a.tiles_x * a.tiles_y, tile = (int64_t)ty * a.tiles_x + tx;
        (void)n_tiles;
        const bool here = tx < a.tiles_x && LCL_IN(tile, n_tiles);  // uniform over the 8 lanes
        int4 lo = make_int4(0, 0, 0, 0), hi = lo;
        if (here) {
            const int4 *b = reinterpret_cast<const int4 *>(a.tile_box + 8 * tile);
            lo = b[0], hi = b[1];
        }
        // spheres: a lane tests strokes `lane` and `lane + 32` against the four tiles in turn
        unsigned long long mask = 0ull, sure = 0ull, pads = 0ull, las = 0ull;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (32 * h >= M.ns) break;  // uniform over the warp
            const int32_t k = 32 * h + lane;
            const bool mine = k < M.ns && stroke_in_bounds(strokes, (int64_t)M.s0 + k, caps);
            bool lasso = false, pad = false;
            SphereArg sp = {};
            if (mine) {
                const BStroke &st = strokes[M.s0 + k];
                lasso = st.kind != LCL_STROKE_SPHERE;
                sp = st.sphere;
                pad = stroke_pads(st, lassos);
            }
            const bool sphere = mine && !lasso;
            uint32_t near = 0u;  // padded spheres: bit c, some box of column tx0 - 1 + c of the three rows is in reach
            if (__any_sync(0xffffffffu, sphere && pad)) {
#pragma unroll 1
                for (int b = 0; b < 3 * (kCullTiles + 2); ++b) {  // uniform
                    const int c = b % (kCullTiles + 2);
                    const int32_t x = tx0 - 1 + c, y = ty - 1 + b / (kCullTiles + 2);
                    if (x < 0 || x >= a.tiles_x || y < 0 || y >= a.tiles_y || !LCL_IN((int64_t)y * a.tiles_x + x, n_tiles))
                        continue;
                    const int4 *bp = reinterpret_cast<const int4 *>(a.tile_box + 8 * ((int64_t)y * a.tiles_x + x));
                    const int4 blo = bp[0], bhi = bp[1];
                    if (blo.w > 0 && box_dist2(blo, bhi, sp) <= sp.r2) near |= 1u << c;
                }
            }
#pragma unroll
            for (int t = 0; t < kCullTiles; ++t) {
                int4 tlo, thi;
                tlo.x = __shfl_sync(0xffffffffu, lo.x, 8 * t), thi.x = __shfl_sync(0xffffffffu, hi.x, 8 * t);
                tlo.y = __shfl_sync(0xffffffffu, lo.y, 8 * t), thi.y = __shfl_sync(0xffffffffu, hi.y, 8 * t);
                tlo.z = __shfl_sync(0xffffffffu, lo.z, 8 * t), thi.z = __shfl_sync(0xffffffffu, hi.z, 8 * t);
                tlo.w = __shfl_sync(0xffffffffu, lo.w, 8 * t), thi.w = 0;
                bool can = false, in = false;
                if (sphere && pad) {
                    can = tx0 + t < a.tiles_x && ((near >> t) & 7u);
                } else if (sphere && tlo.w > 0) {
                    can = box_dist2(tlo, thi, sp) <= sp.r2;
                    in = can && box_far2(tlo, thi, sp) <= sp.r2;
                }
                const uint32_t bc = __ballot_sync(0xffffffffu, can), bi = __ballot_sync(0xffffffffu, in);
                if (group == t) {
                    mask |= (unsigned long long)bc << (32 * h);
                    sure |= (unsigned long long)bi << (32 * h);
                }
            }
            pads |= (unsigned long long)__ballot_sync(0xffffffffu, pad) << (32 * h);
            las |= (unsigned long long)__ballot_sync(0xffffffffu, lasso) << (32 * h);
        }
        if (las) {  // uniform over the warp
            unsigned long long reach = 0ull;
            const int n = __popcll(las);
            for (int i = group; i < n; i += 4) {  // uniform over the 8 lanes
                const int k = nth_bit(las, i);
                const BLasso &L = lassos[strokes[M.s0 + k].lasso];
                if (box_near(L, a.super_box, a.supers_x, a.supers_y, sx, sy, L.pad_r > 0 ? 1 : 0, nullptr))
                    reach |= 1ull << k;
            }
            __syncwarp();
            for (unsigned long long m = warp_or(reach); m; m &= m - 1) {  // uniform over the warp
                const int k = __ffsll((long long)m) - 1;
                const BLasso &L = lassos[strokes[M.s0 + k].lasso];
                int cls = kTileTest;
                bool can = false;
                if (pads >> k & 1ull)
                    can = here && box_near(L, a.tile_box, a.tiles_x, a.tiles_y, tx, ty, 1, L.depth);
                else if (lo.w > 0)
                    can = box_may_touch_by<8, true, 4>(L, lo, hi, L.depth, L.vx, L.vy, &cls);
                if (can) {
                    mask |= 1ull << k;
                    if (cls == kTileIn) sure |= 1ull << k;
                }
                __syncwarp();
            }
        }
        const bool item = mask != 0ull && sub == 0;
        const uint32_t bal = __ballot_sync(0xffffffffu, item);
        uint32_t base = 0;
        if (lane == 0 && bal) base = atomicAdd(&hdr->n_items, (unsigned)__popc(bal));
        const uint32_t slot = __shfl_sync(0xffffffffu, base, 0) + __popc(bal & ((1u << lane) - 1));
        if (item && LCL_IN(slot, caps.tiles)) {
            BItem it;
            it.model = mi;
            it.tile = (uint32_t)tile | (mask & pads ? kPadItem : 0u);
            it.mask = mask;
            it.sure = sure;
            items[slot] = it;
        }
    }
}

// Does stroke `st` select the covered texel n?
template <bool LASSOS>
__device__ __forceinline__ bool stroke_selects(const AtlasDev &a, const BStroke &st, const BLasso *__restrict__ lassos,
                                               int64_t n, int32_t qx) {
    if (!LASSOS || st.kind == LCL_STROKE_SPHERE) {
        const int64_t dx = (int64_t)qx - st.sphere.cx, dy = (int64_t)__ldg(a.py + n) - st.sphere.cy;
        const int64_t dz = (int64_t)__ldg(a.pz + n) - st.sphere.cz;
        return dx * dx + dy * dy + dz * dz <= st.sphere.r2;
    }
    const BLasso &ls = lassos[st.lasso];
    return lasso_hit(ls, ls, ls.depth, qx, __ldg(a.py + n), __ldg(a.pz + n));
}

// Texture padding of the uncovered texels `unc` of the quad at l: for each, the masked padded strokes
// from the newest down; the first whose outline (a covered texel within its thickness) and kernel
// (a texel it selects within its radius) both hold gives the label.  Returns the texels written.
template <bool LASSOS>
__device__ __noinline__ uint32_t pad_texels(const AtlasDev &a, int64_t l, uint32_t unc, unsigned long long mask, int32_t s0,
                               const BStroke *__restrict__ strokes, const BLasso *__restrict__ lassos,
                               uint32_t lab[4], const BCaps &caps) {
    const int32_t x0 = (int32_t)(l % a.w), y0 = (int32_t)(l / a.w);
    uint32_t written = 0u;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        if (!(unc & (1u << k))) continue;
        for (unsigned long long m = mask; m; ) {
            const int si = 63 - __clzll((long long)m);  // newest stroke left
            m &= ~(1ull << si);
            if (!stroke_in_bounds(strokes, (int64_t)s0 + si, caps)) continue;
            const BStroke &st = strokes[s0 + si];
            const int32_t pr = !LASSOS || st.kind == LCL_STROKE_SPHERE ? st.sphere.pad_r : lassos[st.lasso].pad_r;
            if (pr == 0) continue;
            const int32_t pt = !LASSOS || st.kind == LCL_STROKE_SPHERE ? st.sphere.pad_t : lassos[st.lasso].pad_t;
            const int32_t reach = max(pr, pt);
            bool outline = false, near = false;
            for (int32_t dy = -reach; dy <= reach && !(outline && near); ++dy) {
                const int32_t yy = y0 + dy;
                if (yy < 0 || yy >= a.h) continue;
                for (int32_t dx = -reach; dx <= reach; ++dx) {
                    const int32_t xx = x0 + k + dx;
                    if (xx < 0 || xx >= a.w) continue;
                    const int64_t n = (int64_t)yy * a.w + xx;
                    if (!LCL_IN(n, (int64_t)a.w * a.h)) continue;
                    const int32_t qx = __ldg(a.px + n);
                    if (qx == INT32_MIN) continue;
                    const int32_t ax = abs(dx), ay = abs(dy);
                    if (ax <= pt && ay <= pt) outline = true;
                    if (ax <= pr && ay <= pr && !near) near = stroke_selects<LASSOS>(a, st, lassos, n, qx);
                }
            }
            if (outline && near) {
                lab[k] = !LASSOS || st.kind == LCL_STROKE_SPHERE ? st.sphere.label : lassos[st.lasso].label;
                written |= 1u << k;
                break;
            }
        }
    }
    return written;
}

// The texels `open` of a quad that the lasso selects (sure: its tile lies inside the polygon).  Out of line
// it took 1001 us where the batch at k_batch_apply takes 887.
__device__ __forceinline__ uint32_t lasso_texels(const BLasso &ls, int4 X, int4 Y, int4 Z, uint32_t open, bool sure) {
    uint32_t sel = 0u;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {  // selects, not a runtime index into the arrays
        if (!(open & (1u << k))) continue;
        const int32_t qx = k == 0 ? X.x : k == 1 ? X.y : k == 2 ? X.z : X.w;
        const int32_t qy = k == 0 ? Y.x : k == 1 ? Y.y : k == 2 ? Y.z : Y.w;
        const int32_t qz = k == 0 ? Z.x : k == 1 ? Z.y : k == 2 ? Z.z : Z.w;
        if (sure ? lasso_hit<true>(ls, ls, ls.depth, qx, qy, qz)
                 : lasso_hit<false>(ls, ls, ls.depth, qx, qy, qz))
            sel |= 1u << k;
    }
    return sel;
}

// 32 quads from q0 of a work item's tile (quad = 4 consecutive texels of a tile row, row-major in
// the tile), one per lane.
template <bool LASSOS>
__device__ __forceinline__ void apply_quads(const BModel &M, const BItem &it, int32_t q0,
                                            const BStroke *__restrict__ strokes, const BLasso *__restrict__ lassos,
                                            const BCaps &caps) {
    const AtlasDev &a = M.a;
    const uint32_t tile = it.tile & ~kPadItem;
    if (!LCL_IN(tile, (int64_t)a.tiles_x * a.tiles_y)) return;
    int32_t tx, ty;
    tile_xy(a, tile, tx, ty);
    const int32_t qpr = a.T / 4, qd = q0 + (int32_t)(threadIdx.x & 31u);
    const int32_t x = tx * a.T + 4 * (qd & (qpr - 1)), y = ty * a.T + (qd >> (__ffs(qpr) - 1));
    if (qd >= a.T * qpr || x >= a.w || y >= a.h) return;
    const int64_t l = (int64_t)y * a.w + x;
    if (!LCL_IN(l + 3, (int64_t)a.w * a.h)) return;
    const int4 X = __ldg(reinterpret_cast<const int4 *>(a.px + l));
    const int4 Y = __ldg(reinterpret_cast<const int4 *>(a.py + l));
    const int4 Z = __ldg(reinterpret_cast<const int4 *>(a.pz + l));
    const int32_t xs[4] = {X.x, X.y, X.z, X.w}, ys[4] = {Y.x, Y.y, Y.z, Y.w}, zs[4] = {Z.x, Z.y, Z.z, Z.w};
    // uncovered texels (x = INT32_MIN) are never selected: they start final
    uint32_t open = 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) open |= (xs[k] != INT32_MIN ? 1u : 0u) << k;
    const uint32_t unc = ~open & 15u;
    uint32_t lab[4] = {0u, 0u, 0u, 0u}, hit = 0u;
    for (unsigned long long m = it.mask; m && open;) {
        const int si = 63 - __clzll((long long)m);  // newest stroke left
        m &= ~(1ull << si);
        if (!stroke_in_bounds(strokes, (int64_t)M.s0 + si, caps)) continue;
        const BStroke &st = strokes[M.s0 + si];
        uint32_t sel = 0u, label;
        const bool sure = (it.sure >> si) & 1ull;
        if (!LASSOS || st.kind == LCL_STROKE_SPHERE) {
            label = st.sphere.label;
            if (sure) {
                sel = open;  // the sphere contains the tile's box: every covered texel is selected
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int64_t dx = (int64_t)xs[k] - st.sphere.cx, dy = (int64_t)ys[k] - st.sphere.cy;
                    const int64_t dz = (int64_t)zs[k] - st.sphere.cz;
                    sel |= (dx * dx + dy * dy + dz * dz <= st.sphere.r2 ? 1u : 0u) << k;
                }
                sel &= open;
            }
        } else {
            const BLasso &ls = lassos[st.lasso];
            label = ls.label;
            sel = lasso_texels(ls, X, Y, Z, open, sure);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (sel & (1u << k)) lab[k] = label;
        hit |= sel;
        open &= ~sel;
    }
    // texture padding (Section 4.3.2) of the quad's uncovered texels: the newest padded stroke
    // that selects a texel within its kernel radius, with a covered texel within its outline
    // thickness, writes its label there
    if (unc && (it.tile & kPadItem)) {
        uint32_t plab[4];
        const uint32_t ph = pad_texels<LASSOS>(a, l, unc, it.mask, M.s0, strokes, lassos, plab, caps);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (ph & (1u << k)) lab[k] = plab[k];
        hit |= ph;
    }
    if (!hit) return;
    if (M.dtype_bytes == 1) store_labels<uint8_t>(static_cast<uint8_t *>(M.layer), l, hit, lab);
    else store_labels<uint16_t>(static_cast<uint16_t *>(M.layer), l, hit, lab);
}

// The work queue's tickets: an item has up to 16 * split, each an equal share of the tile's groups of 32 quads and a
// group at least (two where all strokes are spheres without padding, whose work is short), one warp per ticket.
// A warp draws its next ticket before it works on the current one, so the queue's latency is hidden; a ticket
// per CTA waited for the slowest of its warps.  24 models of 512^2 to 2048^2 with tiles of 32 (8 groups), 48 spheres
// and 16 lassos each: 8 tickets 959 us, 4 1024, 1 1498.  Tiles of 64 (32 groups), 4 models of 2048^2 with 16 padded
// spheres: 32 203, 16 264, 8 414; one of 16384^2 with 16 spheres and 4 lassos 934, 614, 614.  Tiles of 8 (one
// group) with seven empty tickets each: one of 4096^2 with 64 spheres 502, without them 163.  A group or two per
// ticket, 64 spheres on 4096^2 with tiles of 32: 72 and 61.
// The kernel waits for the lassos' arguments (cache hits) between dependent operations, so warps count for more
// than registers: with 3, 4, 5 and 6 CTAs per SM the batch of 24 took 1141, 1023, 1014 and 974 us.  Without
// lassos (LASSOS false) six, whose 40 registers spill, cost a tenth of five.  The four texels of a quad side by
// side, as in the single lasso's apply, need 80 registers and more code than the instruction cache holds: 1484
// us.  All of the batch: 1314 us before (a CTA per ticket, 3 per SM, padded strokes looked for at every
// uncovered texel), now 696.
constexpr int kItemTicketsLog = 4;

template <bool LASSOS>
__global__ void __launch_bounds__(256, LASSOS ? 6 : 5) k_batch_apply(const BHdr *__restrict__ hdr, const BModel *__restrict__ models,
                                                     const BStroke *__restrict__ strokes,
                                                     const BLasso *__restrict__ lassos,
                                                     const BItem *__restrict__ items, unsigned long long *next_unit,
                                                     int32_t split, BCaps caps) {
    pdl_wait();
    pdl_allow_next();
    const int lane = threadIdx.x & 31;
    const int plog = min(hdr->tickets_log + __ffs(split) - 1, hdr->groups_log);  // split is a power of 2
    const unsigned long long n_units = (unsigned long long)hdr->n_items << plog;
    const unsigned long long n_warps = (unsigned long long)gridDim.x * (blockDim.x / 32);
    unsigned long long next = (unsigned long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
    for (;;) {
        const unsigned long long u = __shfl_sync(0xffffffffu, next, 0);
        if (u >= n_units) break;  // uniform over the warp
        if (lane == 0) next = n_warps + atomicAdd(next_unit, 1ull);
        const unsigned long long i = u >> plog;
        if (!LCL_IN(i, caps.tiles)) continue;
        const BItem it = items[i];
        const int32_t part = (int32_t)(u & ((1u << plog) - 1u));
        if (!LCL_IN(it.model, caps.models)) continue;
        const BModel &M = models[it.model];
        const int32_t groups = max(M.a.T * (M.a.T / 4) / 32, 1);
        const int32_t g0 = groups * part >> plog, g1 = groups * (part + 1) >> plog;
        for (int32_t g = g0; g < g1; ++g) {
            apply_quads<LASSOS>(M, it, 32 * g, strokes, lassos, caps);
            __syncwarp();
        }
    }
}

}  // namespace

// ---- host side -------------------------------------------------------------------------

namespace {

lcl_status check_batch(const lcl_batch_model *models, int32_t n_models, const lcl_batch_stroke *strokes,
                       int32_t n_strokes, const lcl_batch_lasso *lassos, int32_t n_lassos, int64_t *n_supers,
                       int64_t *n_tiles) {
    if (n_models < 0 || n_strokes < 0 || n_lassos < 0) return fail(LCL_ERR_INVALID_ARG, "negative batch count");
    if ((n_models && !models) || (n_strokes && !strokes) || (n_lassos && !lassos))
        return fail(LCL_ERR_INVALID_ARG, "batch array is NULL");
    int64_t ns = 0, nt = 0;
    for (int32_t i = 0; i < n_models; ++i) {
        const lcl_batch_model &m = models[i];
        const lcl_atlas *a = m.atlas;
        if (!a || !a->pos_x || !a->tile_box || !a->super_box || a->tiles_x <= 0 || a->tiles_y <= 0)
            return fail(LCL_ERR_INVALID_ARG, "batch model needs a bound, whole atlas");
        if (m.dtype != LCL_U8 && m.dtype != LCL_U16) return fail(LCL_ERR_INVALID_ARG, "batch model dtype");
        if (!m.layer || (reinterpret_cast<uintptr_t>(m.layer) & 15))
            return fail(LCL_ERR_INVALID_ARG, "batch layers must be 16-byte aligned device pointers");
        if (m.n_strokes < 0 || m.n_strokes > LCL_BATCH_MAX_STROKES)
            return fail(LCL_ERR_UNSUPPORTED, "at most LCL_BATCH_MAX_STROKES (64) strokes per model per batch");
        if (m.first_stroke < 0 || (int64_t)m.first_stroke + m.n_strokes > n_strokes)
            return fail(LCL_ERR_INVALID_ARG, "batch model stroke range out of bounds");
        const uint32_t lab_max = m.dtype == LCL_U8 ? 0xFFu : 0xFFFFu;
        // a band of a texture's rows cannot pad (padding reads up to 8 rows beyond the band)
        const bool band = a->tex_height > 0 && a->height != a->tex_height;
        for (int32_t k = 0; k < m.n_strokes; ++k) {
            const lcl_batch_stroke &s = strokes[m.first_stroke + k];
            if (s.kind == LCL_STROKE_SPHERE) {
                const lcl_sphere &sp = s.sphere;
                const int32_t lo = -(1 << 22), hi = (1 << 22) + (1 << 21);
                if (sp.r2 < 0 || sp.label > lab_max || sp.cx < lo || sp.cx > hi || sp.cy < lo || sp.cy > hi ||
                    sp.cz < lo || sp.cz > hi || (sp.flags & ~0xFFu) || (sp.flags & 15u) > 8 ||
                    ((sp.flags >> 4) & 15u) > 8)
                    return fail(LCL_ERR_INVALID_ARG, "batch sphere stroke out of range");
                if (band && (sp.flags & 15u))
                    return fail(LCL_ERR_UNSUPPORTED, "texture padding needs the whole texture, not a band of its rows");
            } else if (s.kind == LCL_STROKE_LASSO) {
                if (s.lasso < 0 || s.lasso >= n_lassos) return fail(LCL_ERR_INVALID_ARG, "batch lasso index");
                if (lassos[s.lasso].label > lab_max) return fail(LCL_ERR_INVALID_ARG, "batch lasso label too wide");
                if (band && (lassos[s.lasso].flags & 15u))
                    return fail(LCL_ERR_UNSUPPORTED, "texture padding needs the whole texture, not a band of its rows");
            } else {
                return fail(LCL_ERR_INVALID_ARG, "unknown batch stroke kind");
            }
        }
        ns += (int64_t)a->supers_x * a->supers_y;
        nt += (int64_t)a->tiles_x * a->tiles_y;
    }
    for (int32_t j = 0; j < n_lassos; ++j) {
        const lcl_batch_lasso &L = lassos[j];
        const lcl_camera &c = L.camera;
        if (c.width < 1 || c.width > 16384 || c.height < 1 || c.height > 16384 || !L.depth || !L.poly_xy)
            return fail(LCL_ERR_INVALID_ARG, "batch lasso camera or buffers");
        for (int i = 0; i < 16; ++i)
            if (!std::isfinite(c.m[i])) return fail(LCL_ERR_INVALID_ARG, "batch lasso camera is not finite");
        if (L.n_vertices < 3 || L.n_vertices > LCL_MAX_LASSO_VERTICES)
            return fail(LCL_ERR_UNSUPPORTED, "lasso polygons need 3..64 vertices");
        for (int i = 0; i < 2 * L.n_vertices; ++i)
            if (!std::isfinite(L.poly_xy[i])) return fail(LCL_ERR_INVALID_ARG, "batch lasso vertex is not finite");
        if (!std::isfinite(L.bias)) return fail(LCL_ERR_INVALID_ARG, "batch lasso bias is not finite");
        if ((L.flags & ~0xFFu) || (L.flags & 15u) > 8 || ((L.flags >> 4) & 15u) > 8)
            return fail(LCL_ERR_INVALID_ARG, "batch lasso flags: padding radius and thickness at most 8");
    }
    if (ns > INT32_MAX || nt > UINT32_MAX) return fail(LCL_ERR_UNSUPPORTED, "batch too large");
    *n_supers = ns;
    *n_tiles = nt;
    return LCL_OK;
}

bool limits_ok(const lcl_batch_limits *lim) {
    return lim && lim->models >= 0 && lim->strokes >= 0 && lim->lassos >= 0 && lim->supers >= 0 &&
           lim->supers <= INT32_MAX && lim->tiles >= 0 && lim->tiles <= (int64_t)UINT32_MAX;
}

bool config_ok(const lcl_batch_config &c) {
    return (c.threads == 64 || c.threads == 128 || c.threads == 256) && c.ctas_per_sm >= 0 && c.ctas_per_sm <= 32 &&
           (c.split == 1 || c.split == 2 || c.split == 4 || c.split == 8);
}

lcl_batch_config default_config() {
    lcl_batch_config c;
    std::memset(&c, 0, sizeof(c));
    c.threads = 256;
    c.ctas_per_sm = 0;
    c.split = 1;
    return c;
}

struct BPtrs {
    BHdr *hdr;
    const BModel *models;
    const BStroke *strokes;
    const BLassoIn *lasso_in;
    BLasso *lassos;
    const uint32_t *super_model;
    BItem *items;
};

BPtrs b_ptrs(const BLayout &L, void *ws) {
    char *base = static_cast<char *>(ws);
    BPtrs p;
    p.hdr = reinterpret_cast<BHdr *>(base + L.hdr);
    p.models = reinterpret_cast<const BModel *>(base + L.models);
    p.strokes = reinterpret_cast<const BStroke *>(base + L.strokes);
    p.lasso_in = reinterpret_cast<const BLassoIn *>(base + L.lasso_in);
    p.lassos = reinterpret_cast<BLasso *>(base + L.lassos);
    p.super_model = reinterpret_cast<const uint32_t *>(base + L.super_model);
    p.items = reinterpret_cast<BItem *>(base + L.items);
    return p;
}

using ApplyKernel = void (*)(const BHdr *, const BModel *, const BStroke *, const BLasso *, const BItem *,
                             unsigned long long *, int32_t, BCaps);
ApplyKernel apply_kernel(const lcl_batch_limits &lim) { return lim.lassos > 0 ? k_batch_apply<true> : k_batch_apply<false>; }

cudaError_t launch_kernels(const BPtrs &p, const lcl_batch_limits &lim, const lcl_batch_config &c, cudaStream_t st) {
    BCaps caps;
    caps.models = lim.models;
    caps.strokes = lim.strokes;
    caps.lassos = lim.lassos;
    caps.pad = 0;
    caps.supers = lim.supers;
    caps.tiles = lim.tiles;
    const int pg = (std::max(lim.lassos, 1) + kPrepWarps - 1) / kPrepWarps;  // a warp per lasso
    k_batch_prep<<<pg, kThreads, 0, st>>>(p.hdr, p.lasso_in, p.lassos, caps);
    cudaError_t e = cudaSuccess;
    if (lim.supers > 0) {
        const int ug = (int)std::min<int64_t>(lim.supers * kCullUnits / (kThreads / 32), resident_grid(k_batch_cull));
        e = launch_pdl(k_batch_cull, dim3(ug), st, p.hdr, p.models, p.strokes, p.lassos, p.super_model, p.items, caps);
        if (e == cudaSuccess) {
            const auto apply = apply_kernel(lim);
            const int fit = resident_per_sm(apply, c.threads);
            const int per_sm = c.ctas_per_sm > 0 ? std::min(c.ctas_per_sm, fit) : fit;
            e = launch_pdl_shape(apply, dim3(per_sm * sm_count()), dim3(c.threads), st, (const BHdr *)p.hdr,
                                 p.models, p.strokes, p.lassos, (const BItem *)p.items, &p.hdr->next_unit,
                                 (int32_t)c.split, caps);
        }
    }
    count_launches(lim.supers > 0 ? 3 : 1);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e;
}

}  // namespace

lcl_status batch_limits_of(const lcl_batch_model *models, int32_t n_models, int32_t n_strokes, int32_t n_lassos,
                           lcl_batch_limits *out) {
    if (!out || n_models < 0 || n_strokes < 0 || n_lassos < 0 || (n_models && !models))
        return fail(LCL_ERR_INVALID_ARG, "batch limits: bad counts or NULL");
    int64_t ns = 0, nt = 0;
    for (int32_t i = 0; i < n_models; ++i) {
        const lcl_atlas *a = models[i].atlas;
        if (!a || a->tiles_x <= 0 || a->tiles_y <= 0) return fail(LCL_ERR_INVALID_ARG, "batch model without atlas");
        ns += (int64_t)a->supers_x * a->supers_y;
        nt += (int64_t)a->tiles_x * a->tiles_y;
    }
    std::memset(out, 0, sizeof(*out));
    out->models = n_models;
    out->strokes = n_strokes;
    out->lassos = n_lassos;
    out->supers = ns;
    out->tiles = nt;
    if (!limits_ok(out)) return fail(LCL_ERR_UNSUPPORTED, "batch too large");
    return LCL_OK;
}

size_t batch_ws_bytes(const lcl_batch_limits *lim) { return limits_ok(lim) ? b_layout(*lim).total : 0; }

size_t batch_host_bytes(const lcl_batch_limits *lim) { return limits_ok(lim) ? b_layout(*lim).upload : 0; }

namespace {
__global__ void k_copy16(uint4 *__restrict__ dst, const uint4 *__restrict__ src, int64_t n16) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n16; i += (int64_t)gridDim.x * blockDim.x)
        dst[i] = src[i];
}
}  // namespace

cudaError_t copy_by_kernel(void *dst, const void *src, size_t n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int64_t n16 = (int64_t)(n / 16);
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((n16 + kThreads - 1) / kThreads, 2 * sm_count()));
    k_copy16<<<grid, kThreads, 0, st>>>(static_cast<uint4 *>(dst), static_cast<const uint4 *>(src), n16);
    count_launches(1);
    return cudaGetLastError();
}

// staging_dev: the device address of host_staging (pinned, mapped) or NULL; with it the descriptors
// go to the workspace by a copy kernel instead of the copy engines.
lcl_status batch_upload_impl(const lcl_batch_limits *lim, const lcl_batch_model *models, int32_t n_models,
                             const lcl_batch_stroke *strokes, int32_t n_strokes, const lcl_batch_lasso *lassos,
                             int32_t n_lassos, void *ws, size_t ws_bytes, void *host_staging, size_t host_bytes,
                             cudaStream_t st, const void *staging_dev) {
    if (!limits_ok(lim)) return fail(LCL_ERR_INVALID_ARG, "batch limits out of range");
    if (!ws || !host_staging) return fail(LCL_ERR_INVALID_ARG, "batch workspace or staging is NULL");
    int64_t n_supers = 0, n_tiles = 0;
    lcl_status s = check_batch(models, n_models, strokes, n_strokes, lassos, n_lassos, &n_supers, &n_tiles);
    if (s != LCL_OK) return s;
    if (n_models > lim->models || n_strokes > lim->strokes || n_lassos > lim->lassos || n_supers > lim->supers ||
        n_tiles > lim->tiles)
        return fail(LCL_ERR_INVALID_ARG, "batch exceeds the workspace limits");
    const BLayout L = b_layout(*lim);
    if (ws_bytes < L.total) return fail(LCL_ERR_OUT_OF_MEMORY, "batch workspace smaller than lcl_batch_workspace_bytes");
    if (host_bytes < L.upload) return fail(LCL_ERR_OUT_OF_MEMORY, "batch staging smaller than lcl_batch_staging_bytes");
    char *img = static_cast<char *>(host_staging);  // image of the uploaded part of the workspace
    const size_t head = L.models + (size_t)n_models * sizeof(BModel);  // header + models
    std::memset(img, 0, head);
    BHdr hdr;
    std::memset(&hdr, 0, sizeof(hdr));
    hdr.n_models = n_models;
    hdr.n_strokes = n_strokes;
    hdr.n_lassos = n_lassos;
    hdr.n_supers = (int32_t)n_supers;
    for (int32_t i = 0; i < n_models; ++i)
        while ((32 << hdr.groups_log) < models[i].atlas->tile * models[i].atlas->tile / 4) ++hdr.groups_log;
    bool spheres = true;  // nothing but spheres without padding
    for (int32_t k = 0; k < n_strokes; ++k)
        spheres = spheres && strokes[k].kind == LCL_STROKE_SPHERE && !(strokes[k].sphere.flags & 15u);
    hdr.tickets_log = std::max(0, std::min(kItemTicketsLog, hdr.groups_log - (spheres ? 1 : 0)));
    std::memcpy(img + L.hdr, &hdr, sizeof(hdr));
    BModel *bm = reinterpret_cast<BModel *>(img + L.models);
    uint32_t *super_model = reinterpret_cast<uint32_t *>(img + L.super_model);
    int32_t super0 = 0;
    for (int32_t i = 0; i < n_models; ++i) {
        const lcl_batch_model &m = models[i];
        BModel d;
        std::memset(&d, 0, sizeof(d));
        d.a = dev_view(m.atlas);
        d.layer = m.layer;
        d.dtype_bytes = m.dtype == LCL_U8 ? 1 : 2;
        d.s0 = m.first_stroke;
        d.ns = m.n_strokes;
        d.super0 = super0;
        bm[i] = d;
        const int32_t nsup = m.atlas->supers_x * m.atlas->supers_y;
        for (int32_t k = 0; k < nsup; ++k) super_model[super0 + k] = (uint32_t)i;
        super0 += nsup;
    }
    BStroke *bs = reinterpret_cast<BStroke *>(img + L.strokes);
    for (int32_t k = 0; k < n_strokes; ++k) {
        BStroke d;
        std::memset(&d, 0, sizeof(d));
        d.kind = strokes[k].kind;
        d.lasso = strokes[k].lasso;
        d.sphere.cx = strokes[k].sphere.cx;
        d.sphere.cy = strokes[k].sphere.cy;
        d.sphere.cz = strokes[k].sphere.cz;
        d.sphere.r2 = strokes[k].sphere.r2 > kR2Cap ? kR2Cap : strokes[k].sphere.r2;
        d.sphere.label = strokes[k].sphere.label;
        d.sphere.pad_r = (int32_t)(strokes[k].sphere.flags & 15u);
        d.sphere.pad_t = (int32_t)((strokes[k].sphere.flags >> 4) & 15u);
        bs[k] = d;
    }
    BLassoIn *bl = reinterpret_cast<BLassoIn *>(img + L.lasso_in);
    for (int32_t j = 0; j < n_lassos; ++j) {
        BLassoIn &d = bl[j];
        std::memcpy(d.m, lassos[j].camera.m, sizeof(d.m));
        d.w_s = lassos[j].camera.width;
        d.h_s = lassos[j].camera.height;
        d.depth = lassos[j].depth;
        std::memcpy(d.poly, lassos[j].poly_xy, sizeof(float) * 2 * (size_t)lassos[j].n_vertices);
        d.nv = lassos[j].n_vertices;
        d.label = lassos[j].label;
        d.bias = lassos[j].bias;
        d.flags = lassos[j].flags;
    }
    // the used front of each region (the kernels read no further; the limits may be far larger)
    const size_t part[4][2] = {{0, head},
                               {L.strokes, (size_t)n_strokes * sizeof(BStroke)},
                               {L.lasso_in, (size_t)n_lassos * sizeof(BLassoIn)},
                               {L.super_model, (size_t)n_supers * 4}};
    char *dst = static_cast<char *>(ws);
    for (const auto &pc : part) {
        if (pc[1] == 0) continue;
        // by kernel: whole 16-byte words (regions are 256-byte aligned and sized, so rounding up stays
        // inside the region in both images)
        const cudaError_t e = staging_dev ? copy_by_kernel(dst + pc[0], static_cast<const char *>(staging_dev) + pc[0],
                                                           (pc[1] + 15) & ~size_t(15), st)
                                          : cudaMemcpyAsync(dst + pc[0], img + pc[0], pc[1], cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return cuda_fail(e, "batch descriptor upload");
    }
    return LCL_OK;
}

lcl_status batch_launch_impl(const lcl_batch_limits *lim, const lcl_batch_config *cfg, void *ws, size_t ws_bytes,
                             cudaStream_t st) {
    if (!limits_ok(lim)) return fail(LCL_ERR_INVALID_ARG, "batch limits out of range");
    const lcl_batch_config c = cfg ? *cfg : default_config();
    if (!config_ok(c)) return fail(LCL_ERR_INVALID_ARG, "batch config: threads 64/128/256, split 1/2/4/8, ctas_per_sm 0..32");
    const BLayout L = b_layout(*lim);
    if (!ws || ws_bytes < L.total) return fail(LCL_ERR_INVALID_ARG, "batch workspace NULL or smaller than the limits need");
    const cudaError_t e = launch_kernels(b_ptrs(L, ws), *lim, c, st);
    if (e != cudaSuccess) return cuda_fail(e, "batch launch");
    return LCL_OK;
}

lcl_status batch_tune_impl(const lcl_batch_limits *lim, void *ws, size_t ws_bytes, int32_t reps, cudaStream_t st,
                           lcl_batch_config *best, float *best_ms) {
    if (!best || reps < 1 || reps > 100) return fail(LCL_ERR_INVALID_ARG, "batch tune: best is NULL or reps not in 1..100");
    if (!limits_ok(lim)) return fail(LCL_ERR_INVALID_ARG, "batch limits out of range");
    const BLayout L = b_layout(*lim);
    if (!ws || ws_bytes < L.total) return fail(LCL_ERR_INVALID_ARG, "batch workspace NULL or smaller than the limits need");
    const BPtrs p = b_ptrs(L, ws);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    float t_best = INFINITY;
    lcl_batch_config c_best = default_config();
    const int threads[3] = {64, 128, 256}, splits[4] = {1, 2, 4, 8};
    for (int ti = 0; ti < 3 && e == cudaSuccess; ++ti)
        for (int si = 0; si < 4 && e == cudaSuccess; ++si)
            for (int half = 0; half < 2 && e == cudaSuccess; ++half) {
                lcl_batch_config c = default_config();
                c.threads = threads[ti];
                c.split = splits[si];
                const int fit = resident_per_sm(apply_kernel(*lim), c.threads);
                c.ctas_per_sm = half ? std::max(1, fit / 2) : 0;
                if (half && c.ctas_per_sm >= fit) continue;
                e = launch_kernels(p, *lim, c, st);  // warm-up
                if (e == cudaSuccess) e = cudaEventRecord(e0, st);
                for (int r = 0; r < reps && e == cudaSuccess; ++r) e = launch_kernels(p, *lim, c, st);
                if (e == cudaSuccess) e = cudaEventRecord(e1, st);
                if (e == cudaSuccess) e = cudaEventSynchronize(e1);
                float ms = 0.0f;
                if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
                if (e == cudaSuccess && ms / reps < t_best) {
                    t_best = ms / reps;
                    c_best = c;
                }
            }
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (e != cudaSuccess) return cuda_fail(e, "batch tune");
    *best = c_best;
    if (best_ms) *best_ms = t_best;
    return LCL_OK;
}

}  // namespace lcl
