// 2D Gaussian tile rasteriser for G-buffers (IRGS Sec. 3.3: the depth,
// normal, albedo and roughness maps of Eq. 9-10 come from 2DGS
// rasterisation; the shading then runs per pixel).
//
// Per pixel the surfels in front of the near plane are blended (Eq. 2) in
// ascending order of their centre's view depth (ties by user index), each
// with rho^2 = min(rho3^2, rho2^2): rho3 from the pixel ray's intersection
// with the surfel plane (Eq. 6-7; +inf when grazing or behind the camera),
// rho2 the distance of the pixel centre to the projected surfel centre over
// sigma = sqrt(1/2) pixel (the 2DGS screen-space low-pass filter). A surfel
// counts where rho^2 <= rho_c^2 and alpha = min(alpha_max, o exp(-rho^2/2))
// >= alpha_min; its depth is the intersection's tau when the ray term
// wins, else the centre's distance along the ray.
//
// Pipeline: per surfel a conservative pixel rectangle (the projected corners
// of its padded support box, united with the filter's disc around the
// projected centre), counted into the 16x16 tiles that it covers; one
// (depth, user index) key per covered tile, dropped into the tile's segment
// in any order; a block per 2,048 keys of a segment sorts them in shared
// memory, and longer segments are merged from such runs; then one block of
// 256 threads per tile walks its list in 256-surfel chunks staged in shared
// memory, each thread blending its pixel until T < T_min, the block stopping
// when every pixel is done. Segments of a few hundred keys sort in shared
// memory in a few microseconds, where radix sorting all (tile, depth) pairs
// takes six passes over memory with three launches each. 800 x 800 pixels,
// 300,000 surfels, 10 channels: 0.50 ms (1.49 with the radix sorts and every
// pixel of a tile tested against its whole list): preparation 22 us, segments
// 10, keys 26, sort 40, blending 330, the rest the host's wait for the count.
#include <cuda_runtime.h>

#include "camera.cuh"
#include "scene.h"
#include "trace.cuh"

namespace irgs {
namespace {

constexpr int kTileSide = 16;
constexpr int kTilePix = kTileSide * kTileSide;
constexpr int kPrepThreads = 256;
constexpr int kSortBlock = 256;
constexpr int kRun = 2048;             // keys sorted by a block
constexpr int kLengthBins = 128;       // a quarter of a power of two each
// Up to this many tiles start with the longest lists (a few waves of blocks,
// whose last one would otherwise wait for single long tiles: 542 us per image in
// order of place, 511 so, at 2,500 tiles); in larger images the end is short
// against the rest.
constexpr int64_t kOrderedTiles = 1 << 16;
constexpr int kRasterFB = 16;          // blended channels handled per pixel
constexpr float kFilterSigma2 = 0.5f;  // screen-space filter variance (pixels^2)

struct RasterCam {
    f3 o, fw, rt, up;
    float tan_half, aspect;
    int W, H, tiles_x, tiles_y;
};

__device__ __forceinline__ void project(const RasterCam& c, f3 p, float& z, float& px, float& py) {
    const f3 q = sub3(p, c.o);
    z = dot3(q, c.fw);
    const float xs = dot3(q, c.rt) / z, ys = dot3(q, c.up) / z;
    px = (xs / (c.tan_half * c.aspect) + 1.f) * 0.5f * (float)c.W - 0.5f;
    py = (1.f - ys / c.tan_half) * 0.5f * (float)c.H - 0.5f;
}

// fn(tile, source lane, first of the lanes that hold this tile with it, those
// lanes) for every tile of the warp's surfels, `area` of them in the rectangle
// t of this lane's (0: none). Called with all lanes of the warp; neighbouring
// surfels share tiles, which are handed out together.
constexpr int kOwnTiles = 32;   // larger rectangles are shared out among the lanes
template <class Fn>
__device__ __forceinline__ void each_tile(const RasterCam& c, int4 t, int area, Fn fn) {
    const int lane = threadIdx.x & 31;
    const int own = area <= kOwnTiles ? area : 0;
    int tx = t.x, ty = t.y;
    for (int k = 0; __any_sync(kFullWarp, k < own); ++k) {
        const bool on = k < own;
        const int tile = on ? ty * c.tiles_x + tx : -1 - lane;
        fn(tile, lane, __match_any_sync(kFullWarp, tile));
        if (++tx > t.z) {
            tx = t.x;
            ++ty;
        }
    }
    for (unsigned big = __ballot_sync(kFullWarp, area > kOwnTiles); big != 0u; big &= big - 1u) {
        const int src = __ffs(big) - 1;
        const int x0 = __shfl_sync(kFullWarp, t.x, src), y0 = __shfl_sync(kFullWarp, t.y, src);
        const int w = __shfl_sync(kFullWarp, t.z, src) - x0 + 1, all = __shfl_sync(kFullWarp, area, src);
        for (int k = lane; k - lane < all; k += 32)
            fn(k < all ? (y0 + k / w) * c.tiles_x + x0 + k % w : -1, src, 1u << lane);
    }
}

__device__ __forceinline__ int4 tile_rect(int4 r) {
    return make_int4(r.x / kTileSide, r.y / kTileSide, r.z / kTileSide, r.w / kTileSide);
}
__device__ __forceinline__ int tile_area(int4 r) {
    const int4 t = tile_rect(r);
    return r.z < r.x ? 0 : (t.z - t.x + 1) * (t.w - t.y + 1);
}

// Extent of a surfel's disc about its centre along one image axis, in units of
// the tangent: the disc's points are centre + cos A + sin B, and a line s of
// constant tangent touches it where (x_A - s z_A)^2 + (x_B - s z_B)^2 = (s z)^2,
// x seen from the centre's own tangent. Without bound where the disc comes near
// the camera plane (the roots keep 1e-5 of their size up to there, the axes are
// stretched by 1e-4).
__device__ __forceinline__ float2 outline(f3 along, const RasterCam& c, f3 mu, float z, float4 r1, float4 r2) {
    const float rc = 1.0001f * sqrtf(r1.w);
    const f3 u = mk3(r1.x, r1.y, r1.z), v = mk3(r2.x, r2.y, r2.z);   // axes over their squared lengths
    const float lu = rc / dot3(u, u), lv = rc / dot3(v, v);
    const float s0 = dot3(sub3(mu, c.o), along) / z;
    const float za = lu * dot3(u, c.fw), zb = lv * dot3(v, c.fw);
    const float xa = lu * dot3(u, along) - s0 * za, xb = lv * dot3(v, along) - s0 * zb;
    const float a = z * z - za * za - zb * zb, b = xa * za + xb * zb;
    if (!(a > 0.05f * z * z)) return make_float2(-INFINITY, INFINITY);
    const float h = sqrtf(b * b + a * (xa * xa + xb * xb));
    return make_float2((-b - h) / a, (h - b) / a);
}

// Covered pixels of a surfel (Morton slot m), r.z < r.x if none.
__device__ __forceinline__ int4 pixel_rect(const SceneView& S, const float* __restrict__ leaf_box, const RasterCam& c,
                                           float near, int64_t m, float& zc, float2& ctr) {
    const int4 none = make_int4(0, 0, -1, -1);
    const float4 r0 = __ldg(S.rec + m * kRecF4), r1 = __ldg(S.rec + m * kRecF4 + 1), r2 = __ldg(S.rec + m * kRecF4 + 2);
    const f3 mu = mk3(r0.x, r0.y, r0.z);
    project(c, mu, zc, ctr.x, ctr.y);
    if (!(zc > near) || r1.w < 0.f) return none;
    // the filter's support: rho2^2 <= rho_c^2 within rho_c sigma pixels of the centre
    const float rf = sqrtf(fmaxf(r1.w, 0.f) * kFilterSigma2);
    float x0 = ctr.x - rf, x1 = ctr.x + rf, y0 = ctr.y - rf, y1 = ctr.y + rf;
    // the ray term: the support disc lies in the padded leaf box; project its corners
    const float* b = leaf_box + m * 6;
    float zmin = zc, reach = fabsf(c.o.x) + fabsf(c.o.y) + fabsf(c.o.z);
#pragma unroll
    for (int k = 0; k < 3; ++k) reach += fmaxf(fabsf(b[k]), fabsf(b[3 + k]));
    for (int k = 0; k < 8; ++k) {
        const f3 p = mk3(b[(k & 1) ? 3 : 0], b[(k & 2) ? 4 : 1], b[(k & 4) ? 5 : 2]);
        float z, px, py;
        project(c, p, z, px, py);
        if (!(z > 1e-6f)) return make_int4(0, 0, c.W - 1, c.H - 1);   // the box reaches the camera plane: any pixel may see it
        zmin = fminf(zmin, z);
        x0 = fminf(x0, px); x1 = fmaxf(x1, px);
        y0 = fminf(y0, py); y1 = fmaxf(y1, py);
    }
    // The box's corners reach far beyond an oblique disc (139M pixels against
    // 53M for 300k surfels on 800 x 800), so that the disc's own outline bounds
    // it too where it stays clear of the camera plane.
    const float2 wx = outline(c.rt, c, mu, zc, r1, r2), wy = outline(c.up, c, mu, zc, r1, r2);
    const float kx = 0.5f * (float)c.W / (c.tan_half * c.aspect), ky = 0.5f * (float)c.H / c.tan_half;
    x0 = fmaxf(x0, fminf(ctr.x + kx * wx.x, ctr.x - rf));
    x1 = fminf(x1, fmaxf(ctr.x + kx * wx.y, ctr.x + rf));
    y0 = fmaxf(y0, fminf(ctr.y - ky * wy.y, ctr.y - rf));
    y1 = fminf(y1, fmaxf(ctr.y - ky * wy.x, ctr.y + rf));
    // A pixel of slack for the ray's own rounding, and the projection's: a
    // corner's view coordinates are off by less than 1e-6 of the lengths that
    // enter them, and as seen from the camera by that over the depth.
    const float e = 1e-6f * reach / zmin;
    const float sx = 1.f + 0.5f * (float)c.W * e * (1.f + 1.f / (c.tan_half * c.aspect));
    const float sy = 1.f + 0.5f * (float)c.H * e * (1.f + 1.f / c.tan_half);
    x0 = fmaxf(x0 - sx, -1.f); y0 = fmaxf(y0 - sy, -1.f);
    x1 = fminf(x1 + sx, (float)c.W); y1 = fminf(y1 + sy, (float)c.H);
    const int4 r = make_int4(max((int)ceilf(x0), 0), max((int)ceilf(y0), 0), min((int)floorf(x1), c.W - 1),
                             min((int)floorf(y1), c.H - 1));
    return r.z < r.x || r.w < r.y ? none : r;
}

// Per surfel (Morton slot): its key, covered pixels and projected centre, and
// its tiles' counts.
__global__ void __launch_bounds__(kPrepThreads) k_raster_prep(SceneView S, const float* __restrict__ leaf_box,
                                                              RasterCam c, float near, uint64_t* __restrict__ key,
                                                              int4* __restrict__ rect, float2* __restrict__ center,
                                                              uint32_t* __restrict__ count) {
    const int64_t m = blockIdx.x * (int64_t)kPrepThreads + threadIdx.x;
    int4 r = make_int4(0, 0, -1, -1);
    if (m < S.n) {
        float zc;
        float2 ctr;
        r = pixel_rect(S, leaf_box, c, near, m, zc, ctr);
        rect[m] = r;
        center[m] = ctr;
        // zc > 0 where counted: the float bits order like the values
        key[m] = (uint64_t)__float_as_uint(zc) << 32 | (uint32_t)uid_of(S.rec, (int32_t)m);
    }
    each_tile(c, tile_rect(r), tile_area(r), [&](int tile, int, unsigned peers) {
        if (tile >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(count + tile, (uint32_t)__popc(peers));
    });
}

// Segments of the tiles' keys, and the runs that the sort cuts them into.
struct RasterInfo {
    uint64_t pairs;
    uint32_t runs, longest;
};
// Longer lists have smaller numbers.
__device__ __forceinline__ int length_bin(uint32_t n) {
    return n == 0u ? kLengthBins - 1 : kLengthBins - 1 - (int)((__float_as_uint((float)n) >> 21) - (127u << 2));
}
__global__ void __launch_bounds__(1024) k_raster_tiles(uint32_t* __restrict__ count, int64_t n_tiles,
                                                       int2* __restrict__ range, uint32_t* __restrict__ first_run,
                                                       uint32_t* __restrict__ order, RasterInfo* __restrict__ info) {
    __shared__ uint32_t s_bin[kLengthBins];
    __shared__ uint64_t s_pairs[32];
    __shared__ uint32_t s_runs[32];
    __shared__ uint32_t s_max;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_max = 0u;
    if (threadIdx.x < kLengthBins) s_bin[threadIdx.x] = 0u;
    __syncthreads();
    uint64_t pairs = 0;
    uint32_t runs = 0, longest = 0;
    for (int64_t base = 0; base < n_tiles; base += 1024) {
        const int64_t t = base + threadIdx.x;
        const uint32_t n = t < n_tiles ? count[t] : 0u, nr = (n + kRun - 1u) / kRun;
        longest = max(longest, n);
        if (t < n_tiles) atomicAdd(s_bin + length_bin(n), 1u);
        uint64_t p = n;
        uint32_t r = nr;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t pp = __shfl_up_sync(kFullWarp, p, d);
            const uint32_t rr = __shfl_up_sync(kFullWarp, r, d);
            if (lane >= d) {
                p += pp;
                r += rr;
            }
        }
        if (lane == 31) {
            s_pairs[warp] = p;
            s_runs[warp] = r;
        }
        __syncthreads();
        uint64_t before = 0, all = 0;
        uint32_t runs_before = 0, runs_all = 0;
        for (int w = 0; w < 32; ++w) {
            if (w < warp) {
                before += s_pairs[w];
                runs_before += s_runs[w];
            }
            all += s_pairs[w];
            runs_all += s_runs[w];
        }
        if (t < n_tiles) {
            const uint64_t at = pairs + before + p - n;
            range[t] = make_int2((int)at, (int)(at + n));
            count[t] = (uint32_t)at;   // from here on the segment's next free place
            first_run[t] = runs + runs_before + r - nr;
        }
        pairs += all;
        runs += runs_all;
        __syncthreads();
    }
    atomicMax(&s_max, longest);
    __syncthreads();
    if (threadIdx.x == 0) {
        info->pairs = pairs;
        info->runs = runs;
        info->longest = s_max;
        uint32_t at = 0;
        for (int b = 0; b < kLengthBins; ++b) {
            const uint32_t n = s_bin[b];
            s_bin[b] = at;
            at += n;
        }
    }
    if (n_tiles > kOrderedTiles) return;
    __syncthreads();
    for (int64_t t = threadIdx.x; t < n_tiles; t += 1024) {
        const int2 r = range[t];
        order[atomicAdd(s_bin + length_bin((uint32_t)r.y - (uint32_t)r.x), 1u)] = (uint32_t)t;
    }
}

// The surfels' keys into the segments of their tiles.
__global__ void __launch_bounds__(kPrepThreads) k_raster_emit(int64_t n, RasterCam c, const uint64_t* __restrict__ key,
                                                              const int4* __restrict__ rect,
                                                              uint32_t* __restrict__ next,
                                                              uint64_t* __restrict__ keys) {
    const int64_t m = blockIdx.x * (int64_t)kPrepThreads + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const int4 r = m < n ? rect[m] : make_int4(0, 0, -1, -1);
    const uint64_t k = m < n ? key[m] : 0ull;
    each_tile(c, tile_rect(r), tile_area(r), [&](int tile, int src, unsigned peers) {
        const uint64_t ks = __shfl_sync(kFullWarp, k, src);
        const int first = __ffs(peers) - 1;
        uint32_t at = 0;
        if (tile >= 0 && lane == first) at = atomicAdd(next + tile, (uint32_t)__popc(peers));
        at = __shfl_sync(kFullWarp, at, first) + __popc(peers & ((1u << lane) - 1u));
        if (tile >= 0) keys[at] = ks;
    });
}

// Where key v at i of [0, len) goes when ascending runs of `width` (a power of
// two) are merged in pairs: behind the keys of the other run that are below it
// (the keys are distinct).
__device__ __forceinline__ uint32_t merged_place(const uint64_t* a, uint32_t i, uint32_t len, uint32_t width, uint64_t v) {
    const uint32_t pair = i & ~(2u * width - 1u);
    const uint32_t other = (i & width) != 0u ? pair : min(pair + width, len);
    uint32_t lo = other, n = min(other + width, len) - other;
    while (n > 0u) {
        const uint32_t half = n >> 1;
        if (a[lo + half] < v) {
            lo += half + 1u;
            n -= half + 1u;
        } else {
            n = half;
        }
    }
    return pair + (i & (width - 1u)) + (lo - other);
}

__device__ __forceinline__ uint64_t warp_sort(uint64_t v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            const uint64_t o = __shfl_xor_sync(kFullWarp, v, j);
            const bool low = ((lane & j) == 0) == ((lane & k) == 0);
            v = (o < v) == low ? o : v;
        }
    return v;
}

// The segment and run of sort block b: the last tile whose runs begin at or before it.
__device__ __forceinline__ int2 run_of(const uint32_t* __restrict__ first_run, int64_t n_tiles,
                                       const int2* __restrict__ range, int b, int2& seg) {
    int64_t lo = 0, n = n_tiles;
    while (n > 1) {
        const int64_t half = n >> 1;
        if (__ldg(first_run + lo + half) <= (uint32_t)b) {
            lo += half;
            n -= half;
        } else {
            n = half;
        }
    }
    seg = range[lo];
    const int begin = (b - (int)__ldg(first_run + lo)) * kRun;
    return make_int2(begin, min(begin + kRun, seg.y - seg.x));
}

// A run of a segment into ascending order: runs of 32 in registers, then
// merged in shared memory by each key's rank in the other run. To `slots` as
// Morton slots if no merges follow.
__global__ void __launch_bounds__(kSortBlock) k_raster_sort(const uint32_t* __restrict__ first_run, int64_t n_tiles,
                                                            const int2* __restrict__ range,
                                                            const uint64_t* __restrict__ keys,
                                                            const int32_t* __restrict__ inv_perm,
                                                            uint64_t* __restrict__ out, int32_t* __restrict__ slots) {
    __shared__ uint64_t buf[2][kRun];
    int2 seg;
    const int2 run = run_of(first_run, n_tiles, range, (int)blockIdx.x, seg);
    const int begin = seg.x + run.x, len = run.y - run.x;
    for (int i = threadIdx.x; i < ((len + 31) & ~31); i += kSortBlock)
        buf[0][i] = warp_sort(i < len ? keys[begin + i] : ~0ull);
    __syncthreads();
    int cur = 0;
    for (int width = 32; width < len; width *= 2) {
        for (int i = threadIdx.x; i < len; i += kSortBlock) {
            const uint64_t v = buf[cur][i];
            buf[cur ^ 1][merged_place(buf[cur], (uint32_t)i, (uint32_t)len, (uint32_t)width, v)] = v;
        }
        __syncthreads();
        cur ^= 1;
    }
    for (int i = threadIdx.x; i < len; i += kSortBlock) {
        const uint64_t v = buf[cur][i];
        if (slots != nullptr) slots[begin + i] = inv_perm[(uint32_t)v];
        else out[begin + i] = v;
    }
}

// One doubling of the runs of the segments that are longer than one.
__global__ void __launch_bounds__(kSortBlock) k_raster_merge(const uint32_t* __restrict__ first_run, int64_t n_tiles,
                                                             const int2* __restrict__ range,
                                                             const uint64_t* __restrict__ keys, int64_t width,
                                                             const int32_t* __restrict__ inv_perm,
                                                             uint64_t* __restrict__ out, int32_t* __restrict__ slots) {
    int2 seg;
    const int2 run = run_of(first_run, n_tiles, range, (int)blockIdx.x, seg);
    const int len = seg.y - seg.x;
    for (int i = run.x + (int)threadIdx.x; i < run.y; i += kSortBlock) {
        const uint64_t v = keys[seg.x + i];
        const int at = seg.x + (int)(width < len ? merged_place(keys + seg.x, (uint32_t)i, (uint32_t)len, (uint32_t)width, v) : (uint32_t)i);
        if (slots != nullptr) slots[at] = inv_perm[(uint32_t)v];
        else out[at] = v;
    }
}

// rho3^2 and tau of the pixel ray against one surfel (the ray origin is
// rebased to the closest approach to the centre, as in the tracer, so that
// u and v keep their digits for small surfels far from the camera). ah + al is
// the centre seen from the origin, the same for all pixels. Returns false when
// grazing or behind the camera.
__device__ __forceinline__ bool ray_term(const float4& ah, const float4& al, const float4& tu, const float4& tv,
                                         const float4& nn, f3 d, float& rho2, float& tau) {
    const float tr = __fmaf_rn(ah.x, d.x, __fmaf_rn(ah.y, d.y, __fmul_rn(ah.z, d.z)));   // |d| = 1
    const float dlx = __fadd_rn(__fmaf_rn(-tr, d.x, ah.x), al.x);
    const float dly = __fadd_rn(__fmaf_rn(-tr, d.y, ah.y), al.y);
    const float dlz = __fadd_rn(__fmaf_rn(-tr, d.z, ah.z), al.z);
    const float den = __fmaf_rn(nn.x, d.x, __fmaf_rn(nn.y, d.y, __fmul_rn(nn.z, d.z)));
    if (!(fabsf(den) >= 1e-8f)) return false;
    const float num = __fmaf_rn(nn.x, dlx, __fmaf_rn(nn.y, dly, __fmul_rn(nn.z, dlz)));
    const float tp = __fdiv_rn(num, den);
    tau = tr + tp;
    if (!(tau > 0.f)) return false;
    const float ex = __fmaf_rn(tp, d.x, -dlx), ey = __fmaf_rn(tp, d.y, -dly), ez = __fmaf_rn(tp, d.z, -dlz);
    const float u = __fmaf_rn(ex, tu.x, __fmaf_rn(ey, tu.y, __fmul_rn(ez, tu.z)));
    const float v = __fmaf_rn(ex, tv.x, __fmaf_rn(ey, tv.y, __fmul_rn(ez, tv.z)));
    rho2 = __fmaf_rn(u, u, __fmul_rn(v, v));
    return true;
}

// The warps of a tile (8 x 4 pixels each, two to a row) that a surfel's pixels reach.
__device__ __forceinline__ uint32_t covered_warps(int4 r, int x0, int y0) {
    const int ax = max(r.x - x0, 0), bx = min(r.z - x0, kTileSide - 1);
    const int ay = max(r.y - y0, 0), by = min(r.w - y0, kTileSide - 1);
    const uint32_t cols = (ax < 8 ? 1u : 0u) | (bx >= 8 ? 2u : 0u);
    uint32_t warps = 0;
    for (int row = ay >> 2; row <= by >> 2; ++row) warps |= cols << (2 * row);
    return warps;
}

// Bound by instruction issue (72% of the slots, 23 of 32 lanes on): some 80
// instructions per surfel and warp that it reaches. Each warp takes only the
// surfels whose pixel rectangle meets its own 8 x 4 pixels: 2.7M of 6.1M
// tests with the discs' outlines, 10.5M without rectangles (888 us).
template <int FB>
__global__ void __launch_bounds__(kTilePix) k_raster_render(SceneView S, RasterCam c, irgs_camera cam,
                                                            TraceParams P, const uint32_t* __restrict__ order,
                                                            const int2* __restrict__ range,
                                                            const int32_t* __restrict__ slots,
                                                            const int4* __restrict__ rect,
                                                            const float2* __restrict__ center,
                                                            float* __restrict__ feat, float* __restrict__ depth,
                                                            float* __restrict__ opac, int32_t* __restrict__ nhits) {
    __shared__ float4 s_rec[5][kTilePix];   // centre from the origin (high, low words), axes, normal, with o, rho_c^2, centre's pixel
    __shared__ float4 s_feat[(FB + 3) / 4][kTilePix];
    __shared__ uint8_t s_warps[kTilePix];
    const int tile = order != nullptr ? (int)order[blockIdx.x] : (int)blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x0 = tile % c.tiles_x * kTileSide, y0 = tile / c.tiles_x * kTileSide;
    const int px = x0 + (warp & 1) * 8 + (lane & 7), py = y0 + (warp >> 1) * 4 + (lane >> 3);
    const bool inside = px < c.W && py < c.H;
    const f3 d = camera_dir(cam, (float)px, (float)py);
    const float fpx = (float)px, fpy = (float)py;
    float C[FB];
#pragma unroll
    for (int k = 0; k < FB; ++k) C[k] = 0.f;
    float D = 0.f, T = 1.f;
    int nh = 0;
    bool done = !inside;
    const int2 rg = range[tile];
    for (int base = rg.x; base < rg.y; base += kTilePix) {
        if (__syncthreads_count(!done) == 0) break;
        const int j = base + (int)threadIdx.x;
        if (j < rg.y) {
            const int32_t m = slots[j];
            const float4* Rp = S.rec + (int64_t)m * kRecF4;
            const float4 r0 = __ldg(Rp), r1 = __ldg(Rp + 1), r2 = __ldg(Rp + 2), r3 = __ldg(Rp + 3);
            const float2 ctr = __ldg(center + m);
            float4 ah, al;
            two_sum(r0.x, -c.o.x, ah.x, al.x);
            two_sum(r0.y, -c.o.y, ah.y, al.y);
            two_sum(r0.z, -c.o.z, ah.z, al.z);
            ah.w = r0.w;
            al.w = r1.w;
            s_rec[0][threadIdx.x] = ah;
            s_rec[1][threadIdx.x] = al;
            s_rec[2][threadIdx.x] = make_float4(r1.x, r1.y, r1.z, ctr.x);
            s_rec[3][threadIdx.x] = make_float4(r2.x, r2.y, r2.z, ctr.y);
            s_rec[4][threadIdx.x] = r3;
            s_warps[threadIdx.x] = (uint8_t)covered_warps(__ldg(rect + m), x0, y0);
            const float* f = S.feat + (int64_t)m * S.F + P.off;
#pragma unroll
            for (int k = 0; k < FB; k += 4) {
                float4 v;
                v.x = k < P.fc ? __ldg(f + k) : 0.f;
                v.y = k + 1 < P.fc ? __ldg(f + k + 1) : 0.f;
                v.z = k + 2 < P.fc ? __ldg(f + k + 2) : 0.f;
                v.w = k + 3 < P.fc ? __ldg(f + k + 3) : 0.f;
                s_feat[k / 4][threadIdx.x] = v;
            }
        }
        __syncthreads();
        const int cnt = min(kTilePix, rg.y - base);
        for (int g = 0; g < cnt; g += 32) {
            if (__all_sync(kFullWarp, done)) break;
            unsigned some = __ballot_sync(kFullWarp, g + lane < cnt && (s_warps[g + lane] >> warp & 1u) != 0u);
            for (; some != 0u; some &= some - 1u) {
                const int i = g + __ffs(some) - 1;
                if (done) continue;
                const float4 ah = s_rec[0][i], al = s_rec[1][i], tu = s_rec[2][i], tv = s_rec[3][i];
                float rho3 = INFINITY, tau = 0.f;
                const bool hit3 = ray_term(ah, al, tu, tv, s_rec[4][i], d, rho3, tau);
                const float dx = fpx - tu.w, dy = fpy - tv.w;
                const float rho2d = (dx * dx + dy * dy) / kFilterSigma2;
                const float rho2 = hit3 ? fminf(rho3, rho2d) : rho2d;
                if (!(rho2 <= al.w)) continue;
                const float alpha = fminf(ah.w * __expf(-0.5f * rho2), P.alpha_max);
                if (!(alpha >= P.alpha_min)) continue;
                const float dep = (hit3 && rho3 <= rho2d) ? tau : dot3(mk3(ah.x, ah.y, ah.z), d);
                const float w = T * alpha;
#pragma unroll
                for (int k = 0; k < FB; k += 4) {
                    const float4 v = s_feat[k / 4][i];
                    const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int l = 0; l < 4 && k + l < FB; ++l) C[k + l] = fmaf(w, f[l], C[k + l]);
                }
                D = fmaf(w, dep, D);
                T *= 1.f - alpha;
                ++nh;
                if (T < P.T_min) done = true;
            }
        }
    }
    if (!inside) return;
    const int64_t p = (int64_t)py * c.W + px;
#pragma unroll
    for (int k = 0; k < FB; ++k)
        if (k < P.fc) feat[p * P.fc + k] = C[k];
    depth[p] = D;
    opac[p] = 1.f - T;
    if (nhits != nullptr) nhits[p] = nh;
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

}  // namespace

irgs_status launch_rasterize(const SceneView& S, const float* leaf_box, const irgs_camera& cam,
                             const irgs_trace_params& p, float* feat, float* depth, float* opac, int32_t* nhits,
                             cudaStream_t st) {
    const TraceParams P = to_params(p);
    RasterCam c;
    const auto v3 = [](const float* a) { f3 r; r.x = a[0]; r.y = a[1]; r.z = a[2]; return r; };
    c.o = v3(cam.origin);
    c.fw = v3(cam.forward);
    c.rt = v3(cam.right);
    c.up = v3(cam.up);
    c.tan_half = cam.tan_half_fov;
    c.aspect = (float)cam.width / (float)cam.height;
    c.W = cam.width;
    c.H = cam.height;
    c.tiles_x = (cam.width + kTileSide - 1) / kTileSide;
    c.tiles_y = (cam.height + kTileSide - 1) / kTileSide;
    const int64_t n_tiles = (int64_t)c.tiles_x * c.tiles_y;
    const int64_t n = S.n;
    // per-surfel scratch + per-tile segments
    const int64_t nn = n > 0 ? n : 1;
    unsigned char* base = nullptr;
    const size_t b_key = 8 * nn, b_rect = 16 * nn, b_ctr = 8 * nn, b_rng = 8 * n_tiles, b_cnt = 4 * n_tiles;
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t total_bytes = al(b_key) + al(b_rect) + al(b_ctr) + al(b_rng) + 3 * al(b_cnt) + al(sizeof(RasterInfo));
    cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&base), total_bytes, st);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? IRGS_ERR_OOM : IRGS_ERR_CUDA;
    size_t off = 0;
    auto take = [&](size_t b) { unsigned char* q = base + off; off += al(b); return q; };
    uint64_t* key = reinterpret_cast<uint64_t*>(take(b_key));
    int4* rect = reinterpret_cast<int4*>(take(b_rect));
    float2* center = reinterpret_cast<float2*>(take(b_ctr));
    int2* range = reinterpret_cast<int2*>(take(b_rng));
    uint32_t* count = reinterpret_cast<uint32_t*>(take(b_cnt));
    uint32_t* first_run = reinterpret_cast<uint32_t*>(take(b_cnt));
    uint32_t* tile_order = reinterpret_cast<uint32_t*>(take(b_cnt));
    RasterInfo* d_info = reinterpret_cast<RasterInfo*>(take(sizeof(RasterInfo)));
    unsigned char* pairs = nullptr;
    int32_t* slots = nullptr;
    RasterInfo info = {};
    if (n > 0) {
        e = cudaMemsetAsync(count, 0, b_cnt, st);
        k_raster_prep<<<grid_for(n, kPrepThreads), kPrepThreads, 0, st>>>(S, leaf_box, c, P.t_min, key, rect, center,
                                                                          count);
        k_raster_tiles<<<1, 1024, 0, st>>>(count, n_tiles, range, first_run, tile_order, d_info);
        count_launches(2);
        if (e == cudaSuccess) e = cudaMemcpyAsync(&info, d_info, sizeof(info), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    } else {
        e = cudaMemsetAsync(range, 0, b_rng, st);
    }
    if (e == cudaSuccess && info.pairs > (uint64_t)INT32_MAX) e = cudaErrorInvalidValue;
    if (e == cudaSuccess && info.pairs > 0) {
        const size_t b8 = al(8 * (size_t)info.pairs);
        e = scratch_alloc(reinterpret_cast<void**>(&pairs), (info.longest > kRun ? 2 : 1) * b8 + al(4 * (size_t)info.pairs),
                          st);
        if (e == cudaSuccess) {
            slots = reinterpret_cast<int32_t*>(pairs);
            uint64_t* from = reinterpret_cast<uint64_t*>(pairs + al(4 * (size_t)info.pairs));
            uint64_t* to = info.longest > kRun ? from + b8 / 8 : nullptr;
            k_raster_emit<<<grid_for(n, kPrepThreads), kPrepThreads, 0, st>>>(n, c, key, rect, count, from);
            k_raster_sort<<<info.runs, kSortBlock, 0, st>>>(first_run, n_tiles, range, from, S.inv_perm, to,
                                                            to != nullptr ? nullptr : slots);
            count_launches(2);
            for (int64_t width = kRun; width < (int64_t)info.longest; width *= 2) {
                uint64_t* sorted = to;
                to = from;
                from = sorted;
                k_raster_merge<<<info.runs, kSortBlock, 0, st>>>(first_run, n_tiles, range, from, width, S.inv_perm, to,
                                                                 2 * width < (int64_t)info.longest ? nullptr : slots);
                count_launches(1);
            }
        }
    }
    if (e == cudaSuccess) {
        const unsigned g = (unsigned)n_tiles;
        const uint32_t* order = n > 0 && n_tiles <= kOrderedTiles ? tile_order : nullptr;
        if (P.fc <= 3)
            k_raster_render<3><<<g, kTilePix, 0, st>>>(S, c, cam, P, order, range, slots, rect, center, feat, depth, opac, nhits);
        else if (P.fc <= 10)
            k_raster_render<10><<<g, kTilePix, 0, st>>>(S, c, cam, P, order, range, slots, rect, center, feat, depth, opac,
                                                        nhits);
        else
            k_raster_render<kRasterFB><<<g, kTilePix, 0, st>>>(S, c, cam, P, order, range, slots, rect, center, feat, depth,
                                                               opac, nhits);
        count_launches(1);
        e = cudaGetLastError();
    }
    const cudaError_t e1 = pairs ? cudaFreeAsync(pairs, st) : cudaSuccess;
    const cudaError_t e2 = cudaFreeAsync(base, st);
    if (e == cudaErrorMemoryAllocation) return IRGS_ERR_OOM;
    if (e == cudaErrorInvalidValue) return IRGS_ERR_UNSUPPORTED;
    return (e == cudaSuccess && e1 == cudaSuccess && e2 == cudaSuccess) ? IRGS_OK : IRGS_ERR_CUDA;
}

}  // namespace irgs
