// atlas.cu -- UV atlas build: the mesh rasterised in texture space once per model
// (arXiv 2501.14807, Section 4.3.1: the mesh is drawn with its texture coordinates as
// vertex positions, so each fragment is one texel of the layer).  The paper repeats that
// rasterisation on every edit; here it runs once and its result -- per texel the covering
// triangle and the 21-bit grid position of the surface point -- is kept in HBM so that
// every later edit is a streaming pass over the texels.
//
// Kernels, in launch order:
//   k_init        tri plane := none, coverage bits := 0, header reset
//   k_bbox        float bbox of all positions (order-preserving integer atomics)
//   k_scale       grid scale (2^21-1)/extent, one thread
//   k_quant       every vertex to the grid (as in binary64, rounded once per operation)
//   k_snap        every texture coordinate to 1/256 texel (round half to even)
//   k_raster      one thread per triangle: position planes, area weight, and the texels of
//                 small triangles; big triangles are split into 16x16-texel blocks appended to a
//                 work list
//   k_raster_big  one warp per (triangle, block) entry
//   k_resolve     one warp or CTA per tile, one texel per lane and step: position of every covered texel
//                 (from the triangle's planes where their rounding cannot matter, else exact
//                 barycentrics), coverage bits, tile box
//   k_super       one CTA per super-tile: union of its tile boxes
#include <algorithm>
#include <cstring>

#include "lcl_impl.cuh"

namespace lcl {
namespace {

__global__ void k_init(uint32_t *__restrict__ tri, int64_t n_texels, uint32_t *__restrict__ cover, int64_t n_words,
                       AtlasHdr *hdr) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int64_t stride = (int64_t)gridDim.x * blockDim.x;
    uint4 none = make_uint4(kNone, kNone, kNone, kNone);
    for (int64_t k = i; k < n_texels / 4; k += stride)
        if (LCL_IN(4 * k + 3, n_texels)) reinterpret_cast<uint4 *>(tri)[k] = none;
    for (int64_t k = i; k < n_words; k += stride)
        if (LCL_IN(k, n_words)) cover[k] = 0u;
    if (i == 0) {
        for (int a = 0; a < 3; ++a) {
            hdr->key_min[a] = 0x7FFFFFFF;
            hdr->key_max[a] = (int32_t)0x80000000;
        }
        hdr->flags = 0;
        hdr->n_big = 0;
    }
}

// Four vertices (three 16-byte loads) per thread and step; one set of atomics per CTA.
__global__ void __launch_bounds__(kThreads) k_bbox(const float *__restrict__ pos, int64_t n_pos, AtlasHdr *hdr) {
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY};
    bool bad = false;
    auto take = [&](int axis, float p) {
        bad |= !isfinite(p);
        mn[axis] = fminf(mn[axis], p);
        mx[axis] = fmaxf(mx[axis], p);
    };
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n_quads = (reinterpret_cast<uintptr_t>(pos) & 15) == 0 ? n_pos / 4 : 0;  // the array may start anywhere
    for (int64_t v = first; v < n_quads; v += stride) {
        if (!LCL_IN(12 * v + 11, 3 * n_pos)) continue;
        const float4 *p = reinterpret_cast<const float4 *>(pos) + 3 * v;
        const float4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
        take(0, a.x), take(1, a.y), take(2, a.z), take(0, a.w);
        take(1, b.x), take(2, b.y), take(0, b.z), take(1, b.w);
        take(2, c.x), take(0, c.y), take(1, c.z), take(2, c.w);
    }
    for (int64_t v = 4 * n_quads + first; v < n_pos; v += stride)
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (LCL_IN(3 * v + a, 3 * n_pos)) take(a, pos[3 * v + a]);
    __shared__ float red[6][kThreads / 32];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o; o >>= 1) {
            mn[a] = fminf(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], o));
            mx[a] = fmaxf(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], o));
        }
        if ((threadIdx.x & 31) == 0) {
            red[a][threadIdx.x >> 5] = mn[a];
            red[3 + a][threadIdx.x >> 5] = mx[a];
        }
    }
    bad = __syncthreads_or(bad);
    if (threadIdx.x < 3) {
        const int a = threadIdx.x;
        float lo = red[a][0], hi = red[3 + a][0];
        for (int w = 1; w < kThreads / 32; ++w) {
            lo = fminf(lo, red[a][w]);
            hi = fmaxf(hi, red[3 + a][w]);
        }
        if (lo <= hi) {
            atomicMin(&hdr->key_min[a], float_key(lo));
            atomicMax(&hdr->key_max[a], float_key(hi));
        }
        if (a == 0 && bad) atomicOr(&hdr->flags, kBadPos);
    }
}

__global__ void k_scale(AtlasHdr *hdr) {
    double ext = 0.0;
    for (int a = 0; a < 3; ++a) {
        float lo = key_float(hdr->key_min[a]), hi = key_float(hdr->key_max[a]);
        double e = __dsub_rn((double)hi, (double)lo);
        ext = e > ext ? e : ext;
        hdr->mn[a] = lo;
    }
    if (!(ext > 0.0)) {
        hdr->flags |= kFlatBBox;
        hdr->scale = 1.0;
    } else {
        hdr->scale = __ddiv_rn((double)kGridMax, ext);
    }
    hdr->pair = scale_pair(hdr->scale);
}

__global__ void k_quant(const float *__restrict__ pos, int64_t n_pos, const AtlasHdr *__restrict__ hdr,
                        int4 *__restrict__ q) {
    int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n_pos) return;
    const double S = hdr->scale;
    const ScalePair sp = hdr->pair;
    if (!LCL_IN(3 * v + 2, 3 * n_pos)) return;
    int4 r;
    r.x = quantize_coord(pos[3 * v + 0], hdr->mn[0], S, sp);
    r.y = quantize_coord(pos[3 * v + 1], hdr->mn[1], S, sp);
    r.z = quantize_coord(pos[3 * v + 2], hdr->mn[2], S, sp);
    r.w = 0;
    q[v] = r;
}

// rint(u * K), ties to even, for |u| <= 2 and an integer K <= 2^22 (exact in binary32): ph + pl is the
// product exactly (FMA), r = rint(ph) and d = ph - r are exact, and d is a multiple of ulp(ph) while
// |pl| is at most half of that, so pl changes the outcome only where d is a tie; a tie of ph that pl
// leaves alone goes to even as in rint.  (In binary64 the two products per vertex took 62 us for 4 M,
// FP64 being slow on this part.)
__device__ __forceinline__ int32_t snap_coord(float u, float K) {
    const float ph = __fmul_rn(u, K), pl = __fmaf_rn(u, K, -ph);
    const float r = rintf(ph), d = __fsub_rn(ph, r);
    return (int32_t)r + (d == 0.5f && pl > 0.0f ? 1 : 0) - (d == -0.5f && pl < 0.0f ? 1 : 0);
}

__global__ void k_snap(const float *__restrict__ uv, int64_t n_uv, int32_t w, int32_t h, AtlasHdr *hdr,
                       int2 *__restrict__ out) {
    int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n_uv) return;
    if (!LCL_IN(2 * v + 1, 2 * n_uv)) return;
    float u = uv[2 * v], t = uv[2 * v + 1];
    bool ok = isfinite(u) && isfinite(t) && u >= -1.0f && u <= 2.0f && t >= -1.0f && t <= 2.0f;
    if (!ok) {
        atomicOr(&hdr->flags, kBadUV);
        out[v] = make_int2(0, 0);
        return;
    }
    out[v] = make_int2(snap_coord(u, (float)(256 * w)), snap_coord(t, (float)(256 * h)));
}

// floor(sqrt(n)) for n < 2^88 (the squared length of a cross product of 21-bit differences,
// at most 3 * 2^86): a binary64 estimate, then exact integer corrections.  Converting n to binary64
// and the correctly rounded square root each err by at most half an ulp, so the estimate is within
// 2^-8 of sqrt(n) < 2^44, and its floor within one of the result.
__device__ __noinline__ uint64_t isqrt_u88(unsigned __int128 n) {
    const double d = (double)(uint64_t)(n >> 64) * 18446744073709551616.0 + (double)(uint64_t)n;
    uint64_t r = (uint64_t)__dsqrt_rn(d);
#pragma unroll 1
    for (int k = 0; k < 3 && (unsigned __int128)r * r > n; ++k) --r;
#pragma unroll 1
    for (int k = 0; k < 3 && (unsigned __int128)(r + 1) * (r + 1) <= n; ++k) ++r;
    return r;
}

// A 64-bit integer below 2^62 as a float to within 2^-22 of itself (a 64-bit conversion runs on the slow
// FP64 pipe).
__device__ __forceinline__ float to_float_fast(int64_t n) {
    return __fmaf_rn(__int2float_rn((int32_t)(n >> 31)), 2147483648.0f, __int2float_rn((int32_t)(n & 0x7FFFFFFF)));
}

// The same for n < 2^62 from binary32: the estimate is within 2^-21 sqrt(n) of sqrt(n) (2^10), and one
// Newton step with the exact remainder leaves an error below 2^20 / (2 sqrt(n)) of the squared term, 1/2
// of the rounding and 2^-20 of the step: two at most for n >= 2^38; smaller n have estimates within
// two to begin with.
__device__ __forceinline__ uint64_t isqrt_u62(uint64_t n) {
    const float f = __fsqrt_rn(to_float_fast((int64_t)n));
    int64_t r = (int64_t)(uint32_t)f;
    if (n >= (uint64_t(1) << 38)) r += __float2int_rn(__fdividef(__fmul_rn(0.5f, to_float_fast((int64_t)n - r * r)), f));
#pragma unroll 1
    for (int k = 0; k < 4 && (uint64_t)(r * r) > n; ++k) --r;
#pragma unroll 1
    for (int k = 0; k < 4 && (uint64_t)((r + 1) * (r + 1)) <= n; ++k) ++r;
    return (uint64_t)r;
}

// floor(r / A) for r < 2^39 given as r_float too, 0 < A < 2^31, inv = RN(1 / RN(A)), by a binary32 estimate and corrections
// (quotients up to 2^24 come out within 3 of it, those up to 2^8 within 1); r becomes the remainder.
__device__ __forceinline__ uint32_t div_step(uint64_t &r, uint32_t A, float r_float, float inv) {
    uint32_t q = (uint32_t)__fmul_rn(r_float, inv);
    int64_t rem = (int64_t)r - (int64_t)q * (int64_t)A;
#pragma unroll 1
    for (int k = 0; k < 4 && rem < 0; ++k) { --q; rem += A; }
#pragma unroll 1
    for (int k = 0; k < 4 && rem >= (int64_t)A; ++k) { ++q; rem -= A; }
    r = (uint64_t)rem;
    return q;
}

// floor(a 2^24 / A) for a < 2^24, 0 < A < 2^31: an integer quotient and three of eight bits each.
__device__ __forceinline__ uint64_t area_quotient(uint32_t a, uint32_t A, float inv) {
    uint64_t r = a;
    uint64_t q = div_step(r, A, __uint2float_rn(a), inv);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float f = __fmul_rn(__uint2float_rn((uint32_t)r), 256.0f);  // r < A < 2^31
        r <<= 8;
        q = (q << 8) + div_step(r, A, f, inv);
    }
    return q;
}

// The mesh as the kernels gather it: indices, grid positions and snapped texture coordinates.
struct MeshRefs {
    const uint32_t *tri_pos, *tri_uv;
    const int4 *q;
    const int2 *uvs;
    int64_t n_tri, n_pos, n_uv;
};

// Corners of a triangle, counter-clockwise in the texture: snapped texture coordinates, grid
// positions, and A, twice the texture area in sub-pixel units (0: it covers nothing).  Sub-pixel
// coordinates lie within [-2^22, 2^23] (sides <= 2^14, UVs in [-1, 2]): differences fit in 32 bits.
struct Corners {
    int32_t x[3], y[3], qx[3], qy[3], qz[3];
    int64_t A;
};

// False for an index out of range.
__device__ __forceinline__ bool load_corners(const MeshRefs &m, int64_t t, Corners &c) {
    uint32_t ip[3], iu[3];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ip[k] = m.tri_pos[3 * t + k];
        iu[k] = m.tri_uv[3 * t + k];
        ok &= ip[k] < (uint64_t)m.n_pos && iu[k] < (uint64_t)m.n_uv;
    }
    if (!ok) return false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int2 u = m.uvs[iu[k]];
        const int4 q = m.q[ip[k]];
        c.x[k] = u.x;
        c.y[k] = u.y;
        c.qx[k] = q.x;
        c.qy[k] = q.y;
        c.qz[k] = q.z;
    }
    c.A = edge_fn32(c.x[0], c.y[0], c.x[1], c.y[1], c.x[2], c.y[2]);
    if (c.A < 0) {  // swap corners 1 and 2
        int32_t tmp;
        tmp = c.x[1]; c.x[1] = c.x[2]; c.x[2] = tmp;
        tmp = c.y[1]; c.y[1] = c.y[2]; c.y[2] = tmp;
        tmp = c.qx[1]; c.qx[1] = c.qx[2]; c.qx[2] = tmp;
        tmp = c.qy[1]; c.qy[1] = c.qy[2]; c.qy[2] = tmp;
        tmp = c.qz[1]; c.qz[1] = c.qz[2]; c.qz[2] = tmp;
        c.A = -c.A;
    }
    return true;
}

struct RasterArgs {
    MeshRefs m;
    int32_t w;           // texture width
    int32_t row0, rows;  // the rows this atlas holds: [row0, row0 + rows)
    TriPlane *planes;
    uint64_t *area_w;
    uint32_t *tri_plane;
    AtlasHdr *hdr;
    uint2 *big;
    int64_t big_cap;
};

// Texel-centre range [i0, i1] of sub-pixel interval [lo, hi] clamped to [first, last].
__device__ __forceinline__ void texel_range(int32_t lo, int32_t hi, int32_t first, int32_t last, int32_t &i0,
                                            int32_t &i1) {
    i0 = max((lo + 127) >> 8, first);   // ceil((lo - 128) / 256)
    i1 = min((hi - 128) >> 8, last);    // floor((hi - 128) / 256)
}

// n as a sum of two floats, the second the first one's rounding error.
__device__ __forceinline__ void split_int(int64_t n, float &h, float &l) {
    if (n <= (1 << 30) && n >= -(1 << 30)) {
        const int32_t k = (int32_t)n;
        h = __int2float_rn(k);
        l = __int2float_rn(k - __float2int_rn(h));
    } else {
        h = __ll2float_rn(n);
        l = __ll2float_rn(n - __float2ll_rn(h));
    }
}

// The position planes of a triangle.  The slopes num / A (integers) are computed as float pairs, q plus
// the remainder's quotient, good to about 2^-44 of themselves, then rounded to 2^-s as integers below
// 2^30 in magnitude, so each errs by at most 1.01 * 2^-s (two roundings to an integer); over the
// triangle's extent (ex, ey) a position then errs by at most 1.01 (ex + ey) 2^-s, about 2^-18 for
// triangles of a few texels.  Triangles too steep for that (s < 8, or a margin of 1/2) get a margin
// that sends every texel to exact_position.
__device__ __forceinline__ TriPlane make_plane(const Corners &c, int32_t ex, int32_t ey) {
    TriPlane p;
    p.x0 = c.x[0];
    p.y0 = c.y[0];
    const int32_t ax = c.y[2] - c.y[0], ay = c.x[0] - c.x[2];  // d w1 / dx, d w1 / dy
    const int32_t bx = c.y[0] - c.y[1], by = c.x[1] - c.x[0];  // d w2 / dx, d w2 / dy
    float ah, al;
    split_int(c.A, ah, al);
    const float inv = __frcp_rn(ah);
    float g[6], gl[6], most = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int32_t *const q = k == 0 ? c.qx : k == 1 ? c.qy : c.qz;
        const int32_t d1 = q[1] - q[0], d2 = q[2] - q[0];
        p.q0[k] = q[0];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            float h, l;
            split_int(e ? (int64_t)ay * d1 + (int64_t)by * d2 : (int64_t)ax * d1 + (int64_t)bx * d2, h, l);
            const float v = __fmul_rn(h, inv);
            g[2 * k + e] = v;
            gl[2 * k + e] = __fmul_rn(__fadd_rn(__fmaf_rn(-v, ah, h), __fmaf_rn(-v, al, l)), inv);
            most = fmaxf(most, fabsf(v));
        }
    }
    const int32_t s = min(30, 29 - ((int32_t)(__float_as_uint(most) >> 23) - 127));  // most 2^s < 2^30
    const float scale = __uint_as_float((uint32_t)(127 + max(s, 0)) << 23);
    const float margin = __fmul_rn(1.02f * 4294967296.0f, __fdividef((float)(ex + ey), scale));
    const bool usable = s >= 8 && margin < 2147483000.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p.gx[k] = usable ? __float2int_rn(__fmul_rn(g[2 * k], scale)) + __float2int_rn(__fmul_rn(gl[2 * k], scale)) : 0;
        p.gy[k] = usable ? __float2int_rn(__fmul_rn(g[2 * k + 1], scale)) + __float2int_rn(__fmul_rn(gl[2 * k + 1], scale)) : 0;
    }
    p.fine = usable ? ((((uint32_t)margin + 64u) & ~31u) | (uint32_t)s) : (0x80000000u | 8u);
    return p;
}

// raster_rect for a triangle whose corners span at most 2^14 sub-pixels (64 texels) on each axis.
// The scanned texel centres lie within the corners' bounding box (the texel range is cut from it),
// and the values computed one texel past the last column or row within one texel of it, so with
// ex, ey <= 2^14 the extents: |edge value| <= ex (ey + 256) + ey (ex + 256) + 1 < 2^30, and the
// steps are at most 256 * 2^14.  The scan therefore runs in 32-bit integers after an exact start.
__device__ __forceinline__ void raster_rect_small(const Corners &s, uint32_t t, int32_t i0, int32_t i1, int32_t j0, int32_t j1,
                                  int32_t w, int32_t row0, int32_t rows, uint32_t *__restrict__ tri_plane) {
    const int32_t X0 = s.x[0], X1 = s.x[1], X2 = s.x[2], Y0 = s.y[0], Y1 = s.y[1], Y2 = s.y[2];
    const int32_t px = 256 * i0 + 128, py = 256 * j0 + 128;
    int32_t e0 = (int32_t)(edge_fn32(X1, Y1, X2, Y2, px, py) + edge_bias(X2 - X1, Y2 - Y1));
    int32_t e1 = (int32_t)(edge_fn32(X2, Y2, X0, Y0, px, py) + edge_bias(X0 - X2, Y0 - Y2));
    int32_t e2 = (int32_t)(edge_fn32(X0, Y0, X1, Y1, px, py) + edge_bias(X1 - X0, Y1 - Y0));
    const int32_t dx0 = -(Y2 - Y1) * 256, dy0 = (X2 - X1) * 256;
    const int32_t dx1 = -(Y0 - Y2) * 256, dy1 = (X0 - X2) * 256;
    const int32_t dx2 = -(Y1 - Y0) * 256, dy2 = (X1 - X0) * 256;
    const int32_t n_i = i1 - i0;
#pragma unroll 1
    for (int32_t j = j0; j <= j1; ++j) {
        int32_t r0 = e0, r1 = e1, r2 = e2;
        uint32_t *row = tri_plane + (j - row0) * (int64_t)w + i0;
#pragma unroll 1
        for (int32_t i = 0; i <= n_i; ++i) {
            if (min(r0, min(r1, r2)) > 0 && LCL_IN((j - row0) * (int64_t)w + i0 + i, (int64_t)w * rows))
                atomicMin(row + i, t);
            r0 += dx0;
            r1 += dx1;
            r2 += dx2;
        }
        e0 += dy0;
        e1 += dy1;
        e2 += dy2;
    }
}

// Rasterises texels [i0, i1] x [j0, j1] (texture rows j) of a set-up triangle into a plane that
// holds rows [row0, row0 + rows).
__device__ __noinline__ void raster_rect(const Corners &s, uint32_t t, int64_t i0, int64_t i1, int64_t j0, int64_t j1, int32_t w,
                            int32_t row0, int32_t rows, uint32_t *__restrict__ tri_plane) {
    int64_t X0 = s.x[0], X1 = s.x[1], X2 = s.x[2], Y0 = s.y[0], Y1 = s.y[1], Y2 = s.y[2];
    int64_t px = 256 * i0 + 128, py = 256 * j0 + 128;
    // w_k + bias_k > 0 <=> covered (integer edge values, owned edges get bias 1)
    int64_t e0 = edge_fn(X1, Y1, X2, Y2, px, py) + edge_bias(X2 - X1, Y2 - Y1);
    int64_t e1 = edge_fn(X2, Y2, X0, Y0, px, py) + edge_bias(X0 - X2, Y0 - Y2);
    int64_t e2 = edge_fn(X0, Y0, X1, Y1, px, py) + edge_bias(X1 - X0, Y1 - Y0);
    // steps per texel: dE/dx = -(by - ay) * 256, dE/dy = (bx - ax) * 256
    int64_t dx0 = -(Y2 - Y1) * 256, dy0 = (X2 - X1) * 256;
    int64_t dx1 = -(Y0 - Y2) * 256, dy1 = (X0 - X2) * 256;
    int64_t dx2 = -(Y1 - Y0) * 256, dy2 = (X1 - X0) * 256;
#pragma unroll 1
    for (int64_t j = j0; j <= j1; ++j) {
        int64_t r0 = e0, r1 = e1, r2 = e2;
        uint32_t *row = tri_plane + (j - row0) * (int64_t)w;
#pragma unroll 1
        for (int64_t i = i0; i <= i1; ++i) {
            if (r0 > 0 && r1 > 0 && r2 > 0 && LCL_IN((j - row0) * (int64_t)w + i, (int64_t)w * rows))
                atomicMin(row + i, t);
            r0 += dx0;
            r1 += dx1;
            r2 += dx2;
        }
        e0 += dy0;
        e1 += dy1;
        e2 += dy2;
    }
}

// Triangle t's planes and area weight, and its texels if it is a small triangle.
__device__ __forceinline__ void raster_triangle(const RasterArgs &a, int64_t t) {
    Corners c;
    if (!load_corners(a.m, t, c)) {
        atomicOr(&a.hdr->flags, kBadIndex);
        a.area_w[t] = 0;
        return;
    }
    // area weight: 3D area over UV area, floor(isqrt(|n|^2) * 2^(16+F) / A), capped
    {
        const int32_t d1x = c.qx[1] - c.qx[0], d1y = c.qy[1] - c.qy[0], d1z = c.qz[1] - c.qz[0];
        const int32_t d2x = c.qx[2] - c.qx[0], d2y = c.qy[2] - c.qy[0], d2z = c.qz[2] - c.qz[0];
        const int64_t nx = (int64_t)d1y * d2z - (int64_t)d1z * d2y, ny = (int64_t)d1z * d2x - (int64_t)d1x * d2z,
                      nz = (int64_t)d1x * d2y - (int64_t)d1y * d2x;
        uint64_t a3, wgt = 0;
        // components below 2^30: the sum of their squares is below 2^62
        const int64_t most = max(max(nx < 0 ? -nx : nx, ny < 0 ? -ny : ny), nz < 0 ? -nz : nz);
        if (most < (1 << 30)) {
            const int32_t sx = (int32_t)nx, sy = (int32_t)ny, sz = (int32_t)nz;
            a3 = isqrt_u62((uint64_t)((int64_t)sx * sx + (int64_t)sy * sy + (int64_t)sz * sz));
        } else {
            a3 = isqrt_u88((unsigned __int128)((__int128)nx * nx) + (unsigned __int128)((__int128)ny * ny) +
                           (unsigned __int128)((__int128)nz * nz));
        }
        if (c.A != 0) {
            if (a3 < (1u << 24) && c.A < (int64_t(1) << 31)) {
                wgt = area_quotient((uint32_t)a3, (uint32_t)c.A, __frcp_rn((float)(uint32_t)c.A));
            } else if (a3 < (uint64_t(1) << 40)) {
                wgt = (a3 << (16 + LCL_AREA_FRAC_BITS)) / (uint64_t)c.A;
            } else {
                const unsigned __int128 wq = ((unsigned __int128)a3 << (16 + LCL_AREA_FRAC_BITS)) / (uint64_t)c.A;
                wgt = wq > kWeightCap ? kWeightCap : (uint64_t)wq;
            }
            wgt = wgt > kWeightCap ? kWeightCap : wgt;
        }
        a.area_w[t] = wgt;
    }
    if (c.A == 0) return;
    const int32_t xmin = min(c.x[0], min(c.x[1], c.x[2])), xmax = max(c.x[0], max(c.x[1], c.x[2]));
    const int32_t ymin = min(c.y[0], min(c.y[1], c.y[2])), ymax = max(c.y[0], max(c.y[1], c.y[2]));
    int32_t i0, i1, j0, j1;
    texel_range(xmin, xmax, 0, a.w - 1, i0, i1);
    texel_range(ymin, ymax, a.row0, a.row0 + a.rows - 1, j0, j1);  // this atlas's rows only
    if (i0 > i1 || j0 > j1) return;
    a.planes[t] = make_plane(c, xmax - xmin, ymax - ymin);
    const int32_t nx = i1 - i0 + 1, ny = j1 - j0 + 1;  // up to 2^14 each
    if (nx * ny <= kSmallRaster) {
        if (xmax - xmin <= (1 << 14) && ymax - ymin <= (1 << 14))
            raster_rect_small(c, (uint32_t)t, i0, i1, j0, j1, a.w, a.row0, a.rows, a.tri_plane);
        else
            raster_rect(c, (uint32_t)t, i0, i1, j0, j1, a.w, a.row0, a.rows, a.tri_plane);
        return;
    }
    const int64_t nb = (int64_t)((nx + kBlockSide - 1) / kBlockSide) * ((ny + kBlockSide - 1) / kBlockSide);
    unsigned long long base = atomicAdd(&a.hdr->n_big, (unsigned long long)nb);
    if ((int64_t)base + nb <= a.big_cap) {
        for (int64_t b = 0; b < nb; ++b)
            if (LCL_IN((int64_t)base + b, a.big_cap)) a.big[base + b] = make_uint2((uint32_t)t, (uint32_t)b);
        return;
    }
    // list full: the reserved slots that lie below the capacity are read by k_raster_big, so they
    // get empty entries, and this thread rasterises the triangle itself
    for (int64_t b = 0; b < nb && (int64_t)base + b < a.big_cap; ++b)
        if (LCL_IN((int64_t)base + b, a.big_cap)) a.big[base + b] = make_uint2(kNone, 0u);
    raster_rect(c, (uint32_t)t, i0, i1, j0, j1, a.w, a.row0, a.rows, a.tri_plane);
}

// A thread per triangle.  Of the triangles that cover a texel the smallest id wins: atomicMin, whose rate of about
// one lane a cycle and SM bounds the kernel (16384^2, 8 M triangles: 1.05 ms).  Plain stores take 0.87, with a
// count of covered texels that shows whether two triangles share one, but then raster and resolve have to run
// again: the whole build took 2.51 ms, and 4.9 to 7.6 with a single shared texel or a mirrored unwrap, where
// it now takes 2.69, and 2.69 to 4.1; slivers that snapping folds over give nearly every unwrap such texels.
// Four triangles at a time by eight lanes each, so that a row is one request: 2.67, on charts 2.78 (2.59).
__global__ void __launch_bounds__(128) k_raster(const __grid_constant__ RasterArgs a) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < a.m.n_tri) raster_triangle(a, t);
}

// The blocks of big triangles, a warp each: a lane takes every second row of one of the block's 16 columns,
// its edge values stepping from row to row.  Bound by the latency of the chain entry -> indices -> corners,
// so a warp, not a CTA, waits on it: 400 000 triangles on 16384^2 (9 blocks each) took 6.06 ms with a CTA
// per entry and a texel per thread, now 1.43.
__global__ void __launch_bounds__(kThreads) k_raster_big(const uint2 *__restrict__ big, const AtlasHdr *hdr, int64_t cap,
                             const MeshRefs m, int32_t w, int32_t row0, int32_t rows,
                             uint32_t *__restrict__ tri_plane) {
    const int64_t n = min((int64_t)hdr->n_big, cap), n_warps = (int64_t)gridDim.x * (kThreads / 32);
    const int32_t lane = (int32_t)(threadIdx.x & 31u), col = lane % kBlockSide, row = lane / kBlockSide;
    constexpr int kStep = 32 / kBlockSide;  // rows of a warp's step
    int64_t e = (int64_t)blockIdx.x * (kThreads / 32) + threadIdx.x / 32;
    uint2 next = e < n && LCL_IN(e, cap) ? big[e] : make_uint2(kNone, 0u);
    for (; e < n; e += n_warps) {  // uniform over the warp
        const uint2 ent = next;
        next = e + n_warps < n && LCL_IN(e + n_warps, cap) ? big[e + n_warps] : make_uint2(kNone, 0u);
        if (ent.x == kNone) continue;  // a slot of a reservation that did not fit
        if (!LCL_IN(ent.x, m.n_tri)) continue;
        Corners s;
        if (!load_corners(m, ent.x, s)) continue;
        const int32_t xmin = min(s.x[0], min(s.x[1], s.x[2])), xmax = max(s.x[0], max(s.x[1], s.x[2]));
        const int32_t ymin = min(s.y[0], min(s.y[1], s.y[2])), ymax = max(s.y[0], max(s.y[1], s.y[2]));
        int32_t i0, i1, j0, j1;
        texel_range(xmin, xmax, 0, w - 1, i0, i1);
        texel_range(ymin, ymax, row0, row0 + rows - 1, j0, j1);  // as k_raster cut the blocks
        const uint32_t nbx = (uint32_t)(i1 - i0 + 1 + kBlockSide - 1) / kBlockSide;
        const int32_t i = i0 + (int32_t)(ent.y % nbx) * kBlockSide + col;
        int32_t j = j0 + (int32_t)(ent.y / nbx) * kBlockSide + row;
        if (i > i1) continue;
        const int32_t px = 256 * i + 128, py = 256 * j + 128;
        int64_t e0 = edge_fn32(s.x[1], s.y[1], s.x[2], s.y[2], px, py) + edge_bias(s.x[2] - s.x[1], s.y[2] - s.y[1]);
        int64_t e1 = edge_fn32(s.x[2], s.y[2], s.x[0], s.y[0], px, py) + edge_bias(s.x[0] - s.x[2], s.y[0] - s.y[2]);
        int64_t e2 = edge_fn32(s.x[0], s.y[0], s.x[1], s.y[1], px, py) + edge_bias(s.x[1] - s.x[0], s.y[1] - s.y[0]);
        const int64_t d0 = (int64_t)(s.x[2] - s.x[1]) * (256 * kStep), d1 = (int64_t)(s.x[0] - s.x[2]) * (256 * kStep);
        const int64_t d2 = (int64_t)(s.x[1] - s.x[0]) * (256 * kStep);
#pragma unroll
        for (int k = 0; k < kBlockSide / kStep; ++k) {
            if (j <= j1 && e0 > 0 && e1 > 0 && e2 > 0 && LCL_IN((j - row0) * (int64_t)w + i, (int64_t)w * rows))
                atomicMin(tri_plane + (j - row0) * (int64_t)w + i, ent.x);
            j += kStep;
            e0 += d0;
            e1 += d1;
            e2 += d2;
        }
    }
}

// Exact rounded barycentric interpolation of one axis, relative to corner 0:
// q = q0 + floor((2 (w1 (q1-q0) + w2 (q2-q0)) + A) / (2A)), which equals
// floor((2 sum_k w_k q_k + A) / (2A)) because q0 is an integer.  The quotient is estimated in
// FP32 with `rden` ~ 1/(2A) (error well under 2 units) and then made exact with integer
// remainder corrections.
__device__ __forceinline__ int32_t interp_axis(int64_t w1, int64_t w2, int64_t A, float rden, int32_t q0, int32_t q1,
                                               int32_t q2) {
    const int32_t d1 = q1 - q0, d2 = q2 - q0;  // |d| < 2^21
    if (A < (int64_t(1) << 40)) {
        const int64_t num = 2 * (w1 * d1 + w2 * d2) + A;  // |num| < 2^63 since w <= A < 2^40, |d| < 2^21
        const int64_t den = 2 * A;
        // the quotient lies within the corners' range (|num / den| <= 2^21 + 1): an int32 floor of the
        // estimate, which four roundings (num and 2A to FP32, the reciprocal, the product) leave within
        // 1/2 of num / den, so the corrections below take at most one step and usually none
        int32_t est = __float2int_rd(__fmul_rn((float)num, rden));
        int64_t r = num - (int64_t)est * den;
#pragma unroll 1
        for (int k = 0; k < 4 && r < 0; ++k) { est -= 1; r += den; }
#pragma unroll 1
        for (int k = 0; k < 4 && r >= den; ++k) { est += 1; r -= den; }
        return q0 + (int32_t)est;
    }
    __int128 num = 2 * ((__int128)w1 * d1 + (__int128)w2 * d2) + A, den = 2 * (__int128)A;
    double dn = (double)(int64_t)(num >> 64) * 18446744073709551616.0 + (double)(uint64_t)num;
    double dd = (double)(int64_t)(den >> 64) * 18446744073709551616.0 + (double)(uint64_t)den;
    int64_t est = (int64_t)floor(dn / dd);
    __int128 r = num - (__int128)est * den;
#pragma unroll 1
    for (int k = 0; k < 4 && r < 0; ++k) { est -= 1; r += den; }
#pragma unroll 1
    for (int k = 0; k < 4 && r >= den; ++k) { est += 1; r -= den; }
    return q0 + (int32_t)est;
}

// The position of triangle t's texel centre (cx, cy), exactly, from the mesh.
__device__ __noinline__ int3 exact_position(const MeshRefs &m, uint32_t t, int32_t cx, int32_t cy) {
    Corners c;
    if (!load_corners(m, t, c)) return make_int3(INT32_MIN, 0, 0);  // not a triangle that covers a texel
    const int64_t w1 = edge_fn32(c.x[2], c.y[2], c.x[0], c.y[0], cx, cy);
    const int64_t w2 = edge_fn32(c.x[0], c.y[0], c.x[1], c.y[1], cx, cy);
    const float rden = __frcp_rn((float)(2 * c.A));
    return make_int3(interp_axis(w1, w2, c.A, rden, c.qx[0], c.qx[1], c.qx[2]),
                     interp_axis(w1, w2, c.A, rden, c.qy[0], c.qy[1], c.qy[2]),
                     interp_axis(w1, w2, c.A, rden, c.qz[0], c.qz[1], c.qz[2]));
}

// The position of triangle t's texel (x, y): q0 + floor(v), v = (gx (cx - x0) + gy (cy - y0)) 2^-s + 1/2
// per axis as a 64-bit integer with s fraction bits; where the fraction is further than the planes'
// error from 0 and 1 the exact v has the same floor.
__device__ __forceinline__ int3 plane_position(const TriPlane *__restrict__ planes, const MeshRefs &mesh, uint32_t t,
                                               int32_t x, int32_t y) {
    const int4 *const r = reinterpret_cast<const int4 *>(planes + t);
    const int4 ra = __ldg(r), rb = __ldg(r + 1), rc = __ldg(r + 2);
    const int32_t cx = 256 * x + 128, cy = 256 * y + 128;
    const int32_t dx = cx - ra.x, dy = cy - ra.y;  // within +-2^24
    const uint32_t s = (uint32_t)rc.w & 31u, margin = (uint32_t)rc.w & ~31u;
    const int64_t half = (int64_t)(1u << (s - 1u));
    const int64_t vx = (int64_t)ra.z * dx + ((int64_t)rb.y * dy + half);
    const int64_t vy = (int64_t)ra.w * dx + ((int64_t)rb.z * dy + half);
    const int64_t vz = (int64_t)rb.x * dx + ((int64_t)rb.w * dy + half);
    const uint32_t lim = 0u - 2u * margin;  // settled: margin <= fraction < 2^32 - margin
    if (((uint32_t)vx << (32u - s)) - margin >= lim || ((uint32_t)vy << (32u - s)) - margin >= lim ||
        ((uint32_t)vz << (32u - s)) - margin >= lim)
        return exact_position(mesh, t, cx, cy);
    return make_int3(rc.x + (int32_t)__funnelshift_r((uint32_t)vx, (uint32_t)(vx >> 32), s),
                     rc.y + (int32_t)__funnelshift_r((uint32_t)vy, (uint32_t)(vy >> 32), s),
                     rc.z + (int32_t)__funnelshift_r((uint32_t)vz, (uint32_t)(vz >> 32), s));
}

// WORDS (tile side 32 or more, width a multiple of 32): a warp takes 32-texel row segments, each one
// aligned coverage word, a texel per lane; otherwise one texel per thread and step, a tile row after the
// other.  Either way warps read the triangle plane and write the position planes in long rows, and the
// texels of one triangle, which lie together, find its planes in L1.  WARP: a tile per warp, all its
// segments from top to bottom, else a tile per CTA.  Bound by the latency of the chain triangle id ->
// planes and by issue (140 instructions per segment, 55% of the cycles): with a CTA per tile of 32 a warp
// had four segments between the latency of its first ids and the reduction of the box.  16384^2, 8 M
// triangles: 1.83 ms by CTAs, 1.39 by warps; exact barycentrics for every texel (290 instructions) took
// 2.79.  Slower: planes in binary32 (their error sent a tenth of the warps to exact_position), four
// segments in flight per warp (spills), three or five CTAs per SM (1.69 and 1.61 ms), planes prefetched
// to L1 a segment ahead (no change by warps, 1.71 ms by CTAs).
// The rule: enough tiles that each of the chip's 4864 warps gets several, weighed by their rows.  With
// tiles of 32 the whole build takes 802 and 916 us (by warps, by CTAs) on 8192^2, 329 and 353 on 4096^2,
// 222 and 225 on 2048^2 (4096 tiles: below the line); of 64 on 16384^2 2610 and 2733, on 8192^2 (16384
// tiles: below the line) 838 and 832.
constexpr int32_t kWarpTiles = 16384;  // of 32 texels

template <bool WORDS, bool WARP>
__global__ void __launch_bounds__(kThreads, 4) k_resolve(const TriPlane *__restrict__ planes,
                                                      const __grid_constant__ MeshRefs mesh, int32_t w, int32_t h,
                                                      int32_t row0, int32_t T, int32_t tiles_x, int32_t n_tiles,
                                                      const uint32_t *__restrict__ tri_plane,
                                                      int32_t *__restrict__ px, int32_t *__restrict__ py,
                                                      int32_t *__restrict__ pz, uint32_t *__restrict__ cover,
                                                      int32_t *__restrict__ tile_box) {
    static_assert(WORDS || !WARP, "a warp per tile takes whole words");
    const int32_t tile = WARP ? (int32_t)(blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) : (int32_t)blockIdx.x;
    if (WARP && tile >= n_tiles) return;
    const int32_t ty = tile / tiles_x, tx = tile - ty * tiles_x;
    int32_t mn[3] = {INT32_MAX, INT32_MAX, INT32_MAX}, mx[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
    int32_t cnt = 0;
    const int tshift = __ffs(T) - 1;  // T is a power of two
    auto resolve = [&](uint32_t t, int32_t x, int32_t y, int32_t l) {  // writes the texel, returns whether it is covered
        int3 o = make_int3(INT32_MIN, 0, 0);
        const bool covered = t != kNone && LCL_IN(t, mesh.n_tri);
        if (covered) {
            o = plane_position(planes, mesh, t, x, y + row0);
            mn[0] = min(mn[0], o.x); mx[0] = max(mx[0], o.x);
            mn[1] = min(mn[1], o.y); mx[1] = max(mx[1], o.y);
            mn[2] = min(mn[2], o.z); mx[2] = max(mx[2], o.z);
        }
        __stcs(px + l, o.x);
        __stcs(py + l, o.y);
        __stcs(pz + l, o.z);
        return covered;
    };
    if (WORDS) {
        const int lane = threadIdx.x & 31, slog = tshift - 5;  // segments per row: 1 << slog
        const int n_words = 1 << (tshift + slog);
        // the triangle ids of the warp's next segment are loaded during this one
        auto place = [&](int i, int32_t &x, int32_t &y) {
            x = (tx << tshift) + ((i & ((1 << slog) - 1)) << 5);
            y = (ty << tshift) + (i >> slog);
            return i < n_words && x < w && y < h;  // x < w implies x + 31 < w
        };
        constexpr int kStep = WARP ? 1 : kThreads / 32;
        const int i0 = WARP ? 0 : (int)(threadIdx.x >> 5);
        int32_t nx, ny;
        bool nv = place(i0, nx, ny);
        uint32_t nt = nv ? __ldcs(tri_plane + (ny * w + nx + lane)) : kNone;
        for (int i = i0; i < n_words; i += kStep) {  // uniform over the warp
            const int32_t x = nx, y = ny;
            const bool v = nv;
            const uint32_t t = nt;
            nv = place(i + kStep, nx, ny);
            nt = nv ? __ldcs(tri_plane + (ny * w + nx + lane)) : kNone;
            if (!v) continue;
            const int32_t l = y * w + x + lane;  // below 2^28
            const bool covered = LCL_IN(l, (int64_t)w * h) && resolve(t, x + lane, y, l);
            const uint32_t bits = __ballot_sync(0xffffffffu, covered);
            cnt += __popc(bits);  // the warp's count, in every lane
            if (lane == 0) cover[l >> 5] = bits;  // the tile's CTA is the word's only writer
        }
        if (lane) cnt = 0;
    } else {
        for (int i = threadIdx.x; i - (int)(threadIdx.x & 31) < T * T; i += kThreads) {  // whole warps together
            const int32_t x = tx * T + (i & (T - 1)), y = ty * T + (i >> tshift);
            const bool valid = i < T * T && x < w && y < h && LCL_IN((int64_t)y * w + x, (int64_t)w * h);
            const int32_t l = valid ? y * w + x : 0;
            const bool covered = valid && resolve(__ldcs(tri_plane + l), x, y, l);
            cnt += covered;
            // lanes writing the same 32-bit word combine, one atomicOr per word
            const uint32_t word = (uint32_t)(l >> 5), val = covered ? 1u << (uint32_t)(l & 31) : 0u;
            const uint32_t peers = __match_any_sync(0xffffffffu, valid ? word : 0xFFFFFFFFu);
            const uint32_t orv = __reduce_or_sync(peers, val);
            if (valid && orv != 0 && (threadIdx.x & 31) == (__ffs(peers) - 1) &&
                LCL_IN(word, ((int64_t)w * h + 31) / 32))
                atomicOr(cover + word, orv);
        }
    }
    // tile box: block reduction
    __shared__ int32_t red[7][kThreads / 32];
    int32_t v[7];
    v[0] = __reduce_min_sync(0xffffffffu, mn[0]);
    v[1] = __reduce_min_sync(0xffffffffu, mn[1]);
    v[2] = __reduce_min_sync(0xffffffffu, mn[2]);
    v[3] = __reduce_add_sync(0xffffffffu, cnt);
    v[4] = __reduce_max_sync(0xffffffffu, mx[0]);
    v[5] = __reduce_max_sync(0xffffffffu, mx[1]);
    v[6] = __reduce_max_sync(0xffffffffu, mx[2]);
    if (!WARP) {
        const int wid = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0)
            for (int k = 0; k < 7; ++k) red[k][wid] = v[k];
        __syncthreads();
        if (threadIdx.x < 32) {  // lane j holds warp j's values
            const int j = threadIdx.x & (kThreads / 32 - 1);
            v[0] = __reduce_min_sync(0xffffffffu, red[0][j]);
            v[1] = __reduce_min_sync(0xffffffffu, red[1][j]);
            v[2] = __reduce_min_sync(0xffffffffu, red[2][j]);
            v[3] = __reduce_add_sync(0xffffffffu, threadIdx.x < kThreads / 32 ? red[3][j] : 0);
            v[4] = __reduce_max_sync(0xffffffffu, red[4][j]);
            v[5] = __reduce_max_sync(0xffffffffu, red[5][j]);
            v[6] = __reduce_max_sync(0xffffffffu, red[6][j]);
        }
    }
    if ((WARP ? threadIdx.x & 31u : threadIdx.x) == 0 && LCL_IN(tile, n_tiles)) {
        int32_t *b = tile_box + 8 * (int64_t)tile;
        reinterpret_cast<int4 *>(b)[0] = make_int4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<int4 *>(b)[1] = make_int4(v[4], v[5], v[6], 0);
    }
}

__global__ void __launch_bounds__(kThreads) k_super(const int32_t *__restrict__ tile_box, int32_t tiles_x,
                                                    int32_t tiles_y, int32_t *__restrict__ super_box) {
    const int32_t sx = blockIdx.x, sy = blockIdx.y;
    const int32_t tx = sx * LCL_SUPER + (threadIdx.x % LCL_SUPER), ty = sy * LCL_SUPER + (threadIdx.x / LCL_SUPER);
    int32_t v[7] = {INT32_MAX, INT32_MAX, INT32_MAX, 0, INT32_MIN, INT32_MIN, INT32_MIN};
    if (tx < tiles_x && ty < tiles_y && LCL_IN((int64_t)ty * tiles_x + tx, (int64_t)tiles_x * tiles_y)) {
        const int4 *b = reinterpret_cast<const int4 *>(tile_box + 8 * ((int64_t)ty * tiles_x + tx));
        int4 lo = b[0], hi = b[1];
        v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w; v[4] = hi.x; v[5] = hi.y; v[6] = hi.z;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        v[0] = min(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
        v[1] = min(v[1], __shfl_xor_sync(0xffffffffu, v[1], o));
        v[2] = min(v[2], __shfl_xor_sync(0xffffffffu, v[2], o));
        v[3] += __shfl_xor_sync(0xffffffffu, v[3], o);
        v[4] = max(v[4], __shfl_xor_sync(0xffffffffu, v[4], o));
        v[5] = max(v[5], __shfl_xor_sync(0xffffffffu, v[5], o));
        v[6] = max(v[6], __shfl_xor_sync(0xffffffffu, v[6], o));
    }
    __shared__ int32_t red[7][kThreads / 32];
    const int wid = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < 7; ++k) red[k][wid] = v[k];
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int j = 1; j < kThreads / 32; ++j) {
            v[0] = min(v[0], red[0][j]); v[1] = min(v[1], red[1][j]); v[2] = min(v[2], red[2][j]);
            v[3] += red[3][j];
            v[4] = max(v[4], red[4][j]); v[5] = max(v[5], red[5][j]); v[6] = max(v[6], red[6][j]);
        }
        const int64_t n_sup = (int64_t)((tiles_x + LCL_SUPER - 1) / LCL_SUPER) * ((tiles_y + LCL_SUPER - 1) / LCL_SUPER);
        if (LCL_IN((int64_t)sy * gridDim.x + sx, n_sup)) {
            int4 *b = reinterpret_cast<int4 *>(super_box + 8 * ((int64_t)sy * gridDim.x + sx));
            b[0] = make_int4(v[0], v[1], v[2], v[3]);
            b[1] = make_int4(v[4], v[5], v[6], 0);
        }
        (void)n_sup;
    }
}

struct WsLayout {
    size_t hdr, q, uvs, planes, big, total;
};

WsLayout ws_layout(int64_t n_pos, int64_t n_uv, int64_t n_tri, int32_t w, int32_t h) {
    WsLayout L;
    L.hdr = 0;
    L.q = align256(sizeof(AtlasHdr));
    L.uvs = L.q + align256((size_t)n_pos * sizeof(int4));
    L.planes = L.uvs + align256((size_t)n_uv * sizeof(int2));
    L.big = L.planes + align256((size_t)n_tri * 64);  // 64 bytes a triangle, of which its planes take 48
    L.total = L.big + align256((size_t)big_capacity(n_tri, w, h) * sizeof(uint2));
    return L;
}

}  // namespace

size_t big_capacity(int64_t n_tri, int32_t w, int32_t h) {
    int64_t blocks = ((int64_t)w / kBlockSide + 2) * ((int64_t)h / kBlockSide + 2);
    return (size_t)std::max<int64_t>(4096, n_tri / 8 + 4 * blocks);
}

size_t atlas_ws_bytes(int64_t n_pos, int64_t n_uv, int64_t n_tri, int32_t w, int32_t h) {
    return ws_layout(n_pos, n_uv, n_tri, w, h).total;
}

lcl_status atlas_build_impl(const lcl_mesh *mesh, lcl_atlas *at, void *ws, size_t ws_bytes, cudaStream_t st) {
    const WsLayout L = ws_layout(mesh->n_pos, mesh->n_uv, mesh->n_tri, at->width, at->height);
    if (ws_bytes < L.total) return fail(LCL_ERR_OUT_OF_MEMORY, "atlas workspace smaller than lcl_atlas_workspace_bytes");
    char *base = static_cast<char *>(ws);
    AtlasHdr *hdr = reinterpret_cast<AtlasHdr *>(base + L.hdr);
    int4 *q = reinterpret_cast<int4 *>(base + L.q);
    int2 *uvs = reinterpret_cast<int2 *>(base + L.uvs);
    TriPlane *planes = reinterpret_cast<TriPlane *>(base + L.planes);
    uint2 *big = reinterpret_cast<uint2 *>(base + L.big);
    const int64_t n_tex = (int64_t)at->width * at->height;
    const int64_t n_words = (n_tex + 31) / 32;
    const int sms = sm_count();

    k_init<<<sms * 8, kThreads, 0, st>>>(at->tri, n_tex, at->cover, n_words, hdr);
    k_bbox<<<std::max(1, std::min<int>(sms * 4, (int)((mesh->n_pos + kThreads - 1) / kThreads))), kThreads, 0, st>>>(
        mesh->pos, mesh->n_pos, hdr);
    k_scale<<<1, 1, 0, st>>>(hdr);
    k_quant<<<(unsigned)((mesh->n_pos + kThreads - 1) / kThreads), kThreads, 0, st>>>(mesh->pos, mesh->n_pos, hdr, q);
    const int32_t tex_h = at->tex_height > 0 ? at->tex_height : at->height;  // snapped against the whole texture
    k_snap<<<(unsigned)((mesh->n_uv + kThreads - 1) / kThreads), kThreads, 0, st>>>(mesh->uv, mesh->n_uv, at->width,
                                                                                   tex_h, hdr, uvs);
    count_launches(5);
    MeshRefs mr;
    mr.tri_pos = mesh->tri_pos;
    mr.tri_uv = mesh->tri_uv;
    mr.q = q;
    mr.uvs = uvs;
    mr.n_tri = mesh->n_tri;
    mr.n_pos = mesh->n_pos;
    mr.n_uv = mesh->n_uv;
    RasterArgs ra;
    ra.m = mr;
    ra.w = at->width;
    ra.row0 = at->row0;
    ra.rows = at->height;
    ra.planes = planes;
    ra.area_w = at->area_w;
    ra.tri_plane = at->tri;
    ra.hdr = hdr;
    ra.big = big;
    ra.big_cap = (int64_t)big_capacity(mesh->n_tri, at->width, at->height);  // blocks of this atlas's rows
    if (mesh->n_tri > 0) {
        k_raster<<<(unsigned)((mesh->n_tri + 127) / 128), 128, 0, st>>>(ra);
        k_raster_big<<<sms * 8, kThreads, 0, st>>>(big, hdr, ra.big_cap, mr, at->width, at->row0, at->height, at->tri);
        count_launches(2);
    }
    const int32_t n_tiles = at->tiles_x * at->tiles_y;
    const bool words = at->tile >= 32 && (at->width & 31) == 0;
    const bool by_warp = words && n_tiles >= kWarpTiles / 32 * at->tile;
    const auto resolve = by_warp ? k_resolve<true, true> : words ? k_resolve<true, false> : k_resolve<false, false>;
    const int per_cta = by_warp ? kThreads / 32 : 1;
    resolve<<<(n_tiles + per_cta - 1) / per_cta, kThreads, 0, st>>>(planes, mr, at->width, at->height, at->row0, at->tile,
                                                                    at->tiles_x, n_tiles, at->tri, at->pos_x, at->pos_y,
                                                                    at->pos_z, at->cover, at->tile_box);
    k_super<<<dim3(at->supers_x, at->supers_y), kThreads, 0, st>>>(at->tile_box, at->tiles_x, at->tiles_y, at->super_box);
    count_launches(2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "atlas build launch");
    AtlasHdr host;
    e = cudaMemcpyAsync(&host, hdr, sizeof(AtlasHdr), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "atlas build");
    if (host.flags & kBadPos) return fail(LCL_ERR_INVALID_ARG, "mesh positions contain a non-finite value");
    if (host.flags & kFlatBBox) return fail(LCL_ERR_INVALID_ARG, "mesh bounding box has zero extent");
    if (host.flags & kBadIndex) return fail(LCL_ERR_INVALID_ARG, "triangle index out of range");
    if (host.flags & kBadUV) return fail(LCL_ERR_INVALID_ARG, "texture coordinate outside [-1, 2] or non-finite");
    for (int a = 0; a < 3; ++a) at->bbox_min[a] = host.mn[a];
    at->scale = host.scale;
    return LCL_OK;
}

}  // namespace lcl
