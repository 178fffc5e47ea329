// Wavefront Monte Carlo shading (IRGS Eq. 13-15) and its gradient.
//
// The fused shading kernel traces the samples of one point from one warp:
// its 32 rays share an origin but spread over the hemisphere, so a warp
// walks 32 unrelated paths through the hierarchy. Here the secondary rays of
// a batch of points are made first (one thread per sample), regrouped by a
// 30-bit key -- a 6-bit octahedral bin of the direction above the 24-bit
// Morton code of the origin -- with a stable radix sort, and traced in that
// order, so the rays of a warp leave neighbouring points in similar
// directions and walk similar paths. These rays are still too spread for
// packets: each walks its own way, with a warp's 32 lanes working on it or,
// in the largest batches, a lane. The per-point estimate then reads the stored
// traces (L_ind, V) and applies the same per-sample arithmetic as the fused
// kernel (shade_point_warp), with the same fixed reduction order.
//
// The gradient reuses the regrouping: the forward pass of the backward also
// saves each ray's hit list; a per-point kernel turns the upstream gradient
// into albedo / roughness / environment gradients and into each ray's
// upstream (dL/dL_ind, dL/dO); the rays are then run backwards in sorted
// order from their hit lists (rays with longer lists replay the march).
//
// Rays are processed in chunks of whole points, at most kWaveChunkRays rays
// each, so the scratch (~330 bytes per ray with the gradient) stays bounded;
// a chunk is sorted as a whole, and the denser its points the more a warp's
// regrouped rays share their paths (one chunk of 41M rays traces 6-7%
// faster than three of at most 2^24).
#include <cuda_runtime.h>

#include "scene.h"
#include "shade.cuh"
#include "trace.cuh"
#include "trace_warp.cuh"
#include "trace_bwd.cuh"
#include "wave.cuh"

namespace irgs {
namespace {

constexpr int kWaveThreads = kTraceThreads;
constexpr int64_t kWaveChunkRays = int64_t(1) << 26;
constexpr int kWaveSavedHits = 64;   // 12% of secondary rays blend more than 32 hits, 0.02% more than 64
// Batches up to this size keep their order: at 61k rays the sort by origin and
// direction costs more than it gives (1.07 ms for a call without, 1.16 with),
// at 1M rays it pays (8.20 without, 7.94 with).
constexpr int64_t kWaveUnsortedMax = int64_t(1) << 19;
// Batches up to this size take a warp per ray, whose throughput does not depend
// on the size; a ray per lane catches up only where the pools are refilled many
// times. ms for scenes of 100k / 300k / 1M / 3M surfels, a warp per ray first:
//   0.26M rays   1.00 0.90 0.88 0.91    1.79 1.83 1.92 2.18
//   4.2M         14.6 13.2 12.1 12.2    13.0 12.4 12.3 13.8
//   8.4M         31.2 29.2 27.1 27.1    26.4 25.4 26.1 29.5
//   16.8M        57.2 54.6 52.1 51.6    48.4 46.6 48.2 53.7
//   41M          129.9 125.4 121.0 119.1    110.6 106.4 105.9 117.2
// Shading breaks even at about 2^22 rays, relighting, whose rays meet twice as
// many surfels, at 2^23 to 2^24 (relight.cu); the two share a line between.
constexpr int64_t kWaveWarpMax = int64_t(1) << 23;
constexpr int kWaveReplayBlocks = 152 * 4;   // blocks that share the few rays whose hit list did not fit

__device__ __forceinline__ f3 ld3w(const float* p, int64_t i) { return mk3(p[3 * i], p[3 * i + 1], p[3 * i + 2]); }

// One thread per sample of points [p0, p0 + rays / St): direction (w = 1 if
// the sample is valid, -1 if its ray is not finite and so meets nothing) and its
// regrouping key (invalid samples sort last).
// Point p draws the random numbers of point number key_base + p; a point
// whose `valid` entry (if given) is not above 0.5 traces nothing.
__global__ void k_wave_gen(const float* __restrict__ xg, const float* __restrict__ ng, const float* __restrict__ rg,
                           const float* __restrict__ wog, int64_t p0, int64_t rays, int St, int nd, int mode,
                           uint64_t seed, const uint32_t* __restrict__ bounds, float4* __restrict__ dir,
                           uint32_t* __restrict__ key, int32_t* __restrict__ val, uint64_t key_base,
                           const float* __restrict__ valid) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= rays) return;
    const int64_t p = p0 + i / St;
    const int s = (int)(i % St);
    if (valid != nullptr && !(valid[p] > 0.5f)) {
        dir[i] = make_float4(0.f, 0.f, 1.f, 0.f);
        key[i] = kInvalidWaveKey;
        val[i] = (int32_t)i;
        return;
    }
    const ShadeFrame F = shade_frame(ld3w(ng, p), ld3w(wog, p), rg[p]);
    const ShadeSample d = draw_sample(F, mode, key_base + (uint64_t)p, s, St, nd, seed);
    const f3 x = ld3w(xg, p);
    dir[i] = make_float4(d.wi.x, d.wi.y, d.wi.z, d.valid ? (can_hit(x, d.wi) ? 1.f : -1.f) : 0.f);
    key[i] = d.valid ? wave_key(x, d.wi, bounds) : kInvalidWaveKey;
    val[i] = (int32_t)i;
}

// Trace the rays in regrouped order; res[i] = (L_ind, V). With SAVE the blended
// hit ids (user order, -1 terminated) and the hit counts are kept for the
// backward.
template <bool SAVE>
struct WaveJob {
    const float* xg;
    int64_t p0;
    int St;
    const float4* dir;
    const int32_t* order;
    float4* res;
    int32_t* nh;
    int32_t* hit_ids;
    int max_ids;
    // FINITE: rays that are not finite are dealt with here, for the kernel that must
    // not walk them; asking costs the pools 0.4%.
    template <bool FINITE = false>
    __device__ __forceinline__ bool load(int j, f3& o, f3& d) const {
        const int64_t i = order[j];
        const float4 d4 = dir[i];
        if (FINITE ? !(d4.w > 0.f) : d4.w == 0.f) {   // every sample gets an entry, so no reader sees unwritten scratch
            res[i] = make_float4(0.f, 0.f, 0.f, FINITE && d4.w < 0.f ? 1.f : 0.f);
            if (SAVE) nh[i] = 0;
            return false;
        }
        o = ld3w(xg, p0 + i / St);
        d = mk3(d4.x, d4.y, d4.z);
        return true;
    }
    __device__ __forceinline__ int32_t* ids(int j) const {
        return SAVE ? hit_ids + order[j] * (int64_t)max_ids : nullptr;
    }
    __device__ __forceinline__ void finish(int j, const MarchState<3>& st) const {
        const int64_t i = order[j];
        res[i] = make_float4(st.C[0], st.C[1], st.C[2], st.T);
        if (SAVE) {
            nh[i] = st.nh;
            if (st.nh < max_ids) hit_ids[i * max_ids + st.nh] = -1;
        }
    }
};

template <bool SAVE>
__global__ void __launch_bounds__(kWaveThreads, kRayBlocks) k_wave_trace(SceneView S, TraceParams P, WaveJob<SAVE> job,
                                                                         int rays, uint32_t* next) {
    __shared__ SavedMarch<3> saved;
    walk_batch<3, kCap>(S, P, rays, next, job, saved);
}

// The same with a warp per ray, for batches that do not fill the chip with a
// ray per lane.
template <bool SAVE>
__global__ void __launch_bounds__(kWarpRayThreads, kWarpRayBlocks) k_wave_trace_ray(SceneView S, TraceParams P, WaveJob<SAVE> job,
                                                                                int rays) {
    const int j = blockIdx.x * kWarpRays + (threadIdx.x >> 5);
    f3 o, d;
    if (j >= rays || !job.template load<true>(j, o, d)) return;
    const Ray ray = make_ray(o, d);
    WarpMarch w;
    const bool ok = march_warp(S, ray, make_ray_box(ray), P, w, job.ids(j), job.max_ids, warp_ray_scratch());
    MarchState<3> st;
#pragma unroll
    for (int c = 0; c < 3; ++c) st.C[c] = __shfl_sync(kFullWarp, w.C, c);
    st.D = w.D;
    st.T = w.T;
    st.nh = w.nh;
    if ((threadIdx.x & 31) != 0) return;
    if (!ok) atomicOr(S.status, kErrStackOverflow);
    job.finish(j, st);
}

// Per-point estimate from the stored traces (warp per point).
__global__ void __launch_bounds__(kWaveThreads) k_wave_shade(SceneView S, const float* __restrict__ xg,
                                                             const float* __restrict__ ng,
                                                             const float* __restrict__ ag,
                                                             const float* __restrict__ rg,
                                                             const float* __restrict__ wog, int64_t p0, int64_t np,
                                                             const float* __restrict__ env, int H, int W, int nd,
                                                             int ns, int mode, uint64_t seed, TraceParams TP,
                                                             const float4* __restrict__ res, float* __restrict__ rgb,
                                                             float* __restrict__ vis, float* __restrict__ ind,
                                                             uint64_t key_base, const float* __restrict__ valid) {
    const int lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)(kWaveThreads / 32) + (threadIdx.x >> 5);
    if (k >= np) return;
    const int64_t p = p0 + k;
    const int St = nd + ns;
    ShadeSums o;
    if (valid != nullptr && !(valid[p] > 0.5f)) {   // background: no estimate (warp-uniform)
        o.rgb[0] = o.rgb[1] = o.rgb[2] = 0.f;
        o.ind[0] = o.ind[1] = o.ind[2] = 0.f;
        o.vis = 0.f;
    } else {
        shade_point_warp<false, true>(S, ld3w(xg, p), ld3w(ng, p), ld3w(wog, p), ld3w(ag, p), rg[p],
                                         key_base + (uint64_t)p, nd, ns, mode, seed, env, H, W, TP, o, res + k * St);
    }
    if (lane == 0) {
        for (int c = 0; c < 3; ++c) rgb[3 * p + c] = o.rgb[c];
        if (vis != nullptr) vis[p] = o.vis;
        if (ind != nullptr)
            for (int c = 0; c < 3; ++c) ind[3 * p + c] = o.ind[c];
    }
}

// Per-point gradient (warp per point): albedo, roughness and environment
// gradients, and up[i] = (dL/dL_ind, dL/dO) of each of its rays.
__global__ void __launch_bounds__(kWaveThreads) k_wave_grad_point(
    const float* __restrict__ ng, const float* __restrict__ ag, const float* __restrict__ rg,
    const float* __restrict__ wog, int64_t p0, int64_t np, const float* __restrict__ env, int H, int W, int nd,
    int ns, int mode, uint64_t seed, const float4* __restrict__ res, const float* __restrict__ g_rgb,
    float* __restrict__ g_albedo, float* __restrict__ g_rough, float* __restrict__ g_env, float4* __restrict__ up) {
    const int lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)(kWaveThreads / 32) + (threadIdx.x >> 5);
    if (k >= np) return;
    const int64_t p = p0 + k;
    const int St = nd + ns;
    const float g[3] = {g_rgb[3 * p], g_rgb[3 * p + 1], g_rgb[3 * p + 2]};
    const f3 a = ld3w(ag, p);
    const float av[3] = {a.x, a.y, a.z};
    const ShadeFrame F = shade_frame(ld3w(ng, p), ld3w(wog, p), rg[p]);
    float ga[3] = {0.f, 0.f, 0.f}, gr = 0.f;
    for (int s = lane; s < St; s += 32) {
        const ShadeSample d = draw_sample(F, mode, (uint64_t)p, s, St, nd, seed);
        float gL[3] = {0.f, 0.f, 0.f}, gO = 0.f;
        if (d.valid) {
            const float4 t = __ldg(res + k * St + s);
            const float C[3] = {t.x, t.y, t.z};
            sample_grad(F, d, mode, nd, ns, St, av, g, C, t.w, env, H, W, g_env, ga, gr, gL, gO);
        }
        up[k * St + s] = make_float4(gL[0], gL[1], gL[2], gO);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
        for (int off = 16; off > 0; off >>= 1) ga[c] += __shfl_xor_sync(0xffffffffu, ga[c], off);
    for (int off = 16; off > 0; off >>= 1) gr += __shfl_xor_sync(0xffffffffu, gr, off);
    if (lane == 0) {
        for (int c = 0; c < 3; ++c) g_albedo[3 * p + c] += ga[c];
        g_rough[p] += gr;
    }
}

// Backward from the saved hit lists, one thread per sorted ray; rays whose
// list did not fit (more than max_ids hits) are appended to replay_list for
// k_wave_replay.
__global__ void __launch_bounds__(kWaveThreads) k_wave_backward(SceneView S, TraceParams P,
                                                                const float* __restrict__ xg, int64_t p0, int St,
                                                                const float4* __restrict__ dir,
                                                                const int32_t* __restrict__ order, int64_t rays,
                                                                const float4* __restrict__ res,
                                                                const int32_t* __restrict__ nh,
                                                                const int32_t* __restrict__ ids, int max_ids,
                                                                const float4* __restrict__ up,
                                                                float* __restrict__ acc_rows,
                                                                int32_t* __restrict__ replay_list,
                                                                uint32_t* __restrict__ replay_count) {
    float4* scratch = warp_memory<32 * GradRow<3>::kStride / 4>();
    const int64_t j = blockIdx.x * (int64_t)kWaveThreads + threadIdx.x;
    if (j >= rays) return;
    const int64_t i = order[j];
    const int n_hits = nh[i];   // 0 for samples that drew no ray
    if (n_hits <= 0) return;
    const float4 u4 = up[i];
    if (u4.x == 0.f && u4.y == 0.f && u4.z == 0.f && u4.w == 0.f) return;
    if (n_hits > max_ids) {
        replay_list[atomicAdd(replay_count, 1u)] = (int32_t)j;
        return;
    }
    const float4 d4 = dir[i], t = res[i];
    const Ray ray = make_ray(ld3w(xg, p0 + i / St), mk3(d4.x, d4.y, d4.z));
    const float Cf[3] = {t.x, t.y, t.z}, gC[3] = {u4.x, u4.y, u4.z};
    listed_backward<3>(S, ray, P, ids + i * (int64_t)max_ids, n_hits, Cf, 0.f, t.w, gC, 0.f, u4.w, acc_rows,
                       reinterpret_cast<float*>(scratch));
}

// The rays of replay_list replay their march backwards, a warp per ray (the
// list's length is what the listing launch left in replay_count): as lanes of
// their own these few hundred longest rays took 0.9 of a gradient's 10.9 ms.
__global__ void __launch_bounds__(kWarpRayThreads) k_wave_replay(SceneView S, TraceParams P, const float* __restrict__ xg,
                                                                 int64_t p0, int St, const float4* __restrict__ dir,
                                                                 const int32_t* __restrict__ order,
                                                                 const float4* __restrict__ res,
                                                                 const int32_t* __restrict__ nh,
                                                                 const float4* __restrict__ up,
                                                                 float* __restrict__ acc_rows,
                                                                 const int32_t* __restrict__ replay_list,
                                                                 const uint32_t* __restrict__ replay_count) {
    const int64_t n = *replay_count;
    const int lane = threadIdx.x & 31;
    for (int64_t t = blockIdx.x * (int64_t)kWarpRays + (threadIdx.x >> 5); t < n; t += (int64_t)gridDim.x * kWarpRays) {
        const int64_t i = order[replay_list[t]];
        const float4 d4 = dir[i], c = res[i], u = up[i];
        const Ray ray = make_ray(ld3w(xg, p0 + i / St), mk3(d4.x, d4.y, d4.z));
        const float Cf = lane == 0 ? c.x : (lane == 1 ? c.y : c.z), gC = lane == 0 ? u.x : (lane == 1 ? u.y : u.z);
        const bool ok = backward_warp<3>(S, ray, P, nh[i], Cf, 0.f, c.w, gC, 0.f, u.w, acc_rows, warp_ray_scratch());
        if (!ok && lane == 0) atomicOr(S.status, kErrStackOverflow);
    }
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

// Scratch of one chunk (stream-ordered allocation).
struct WaveScratch {
    float4* dir = nullptr;
    uint32_t* key = nullptr;
    int32_t* val = nullptr;
    uint32_t* key_tmp = nullptr;
    int32_t* val_tmp = nullptr;
    uint32_t* hist = nullptr;
    float4* res = nullptr;
    int32_t* nh = nullptr;
    int32_t* ids = nullptr;
    float4* up = nullptr;
    int32_t* list = nullptr;     // [rays] rays to replay (sorted positions; gradient only)
    uint32_t* count = nullptr;   // [2] the batch's next pool; rays to replay
    unsigned char* base = nullptr;

    cudaError_t alloc(int64_t rays, bool backward, cudaStream_t st) {
        const int64_t hw = sort_hist_words(rays);
        size_t off = 0;
        auto take = [&](size_t bytes) {
            const size_t o = off;
            off += (bytes + 255) & ~size_t(255);
            return o;
        };
        const size_t o_dir = take(sizeof(float4) * rays), o_key = take(4 * rays), o_val = take(4 * rays);
        const size_t o_kt = take(4 * rays), o_vt = take(4 * rays), o_hist = take(4 * hw);
        const size_t o_res = take(sizeof(float4) * rays);
        const size_t o_count = take(8);
        size_t o_nh = 0, o_ids = 0, o_up = 0, o_list = 0;
        if (backward) {
            o_nh = take(4 * rays);
            o_ids = take(sizeof(int32_t) * kWaveSavedHits * rays);
            o_up = take(sizeof(float4) * rays);
            o_list = take(4 * rays);
        }
        cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&base), off, st);
        if (e != cudaSuccess) return e;
        dir = reinterpret_cast<float4*>(base + o_dir);
        key = reinterpret_cast<uint32_t*>(base + o_key);
        val = reinterpret_cast<int32_t*>(base + o_val);
        key_tmp = reinterpret_cast<uint32_t*>(base + o_kt);
        val_tmp = reinterpret_cast<int32_t*>(base + o_vt);
        hist = reinterpret_cast<uint32_t*>(base + o_hist);
        res = reinterpret_cast<float4*>(base + o_res);
        count = reinterpret_cast<uint32_t*>(base + o_count);
        if (backward) {
            nh = reinterpret_cast<int32_t*>(base + o_nh);
            ids = reinterpret_cast<int32_t*>(base + o_ids);
            up = reinterpret_cast<float4*>(base + o_up);
            list = reinterpret_cast<int32_t*>(base + o_list);
        }
        return cudaSuccess;
    }
    cudaError_t release(cudaStream_t st) { return base ? cudaFreeAsync(base, st) : cudaSuccess; }
};

int64_t chunk_points(int St) {
    const int64_t pc = kWaveChunkRays / St;
    return pc > 0 ? pc : 1;
}

// Trace the sorted rays of one chunk into w.res (and, with SAVE, the hit
// counts and lists).
template <bool SAVE>
cudaError_t wave_trace(const SceneView& S, const TraceParams& TP, const float* x, int64_t p0, int St, int64_t rays,
                       WaveScratch& w, cudaStream_t st) {
    const cudaError_t e = cudaMemsetAsync(w.count, 0, 2 * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    const WaveJob<SAVE> job{x, p0, St, w.dir, w.val, w.res, SAVE ? w.nh : nullptr, SAVE ? w.ids : nullptr,
                            SAVE ? kWaveSavedHits : 0};
    if (rays <= kWaveWarpMax) {
        k_wave_trace_ray<SAVE><<<warp_ray_grid(rays), kWarpRayThreads, 0, st>>>(S, TP, job, (int)rays);
        count_launches(1);
        return cudaGetLastError();
    }
    const unsigned blocks = batch_blocks(k_wave_trace<SAVE>, rays);
    if (blocks == 0u) return cudaGetLastError();
    k_wave_trace<SAVE><<<blocks, kWaveThreads, 0, st>>>(S, TP, job, (int)rays, w.count);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t wave_forward(const SceneView& S, const uint32_t* bounds, const float* x, const float* n, const float* a,
                         const float* r, const float* wo, int64_t P, const float* env, int H, int W, int nd, int ns,
                         int mode, uint64_t seed, const TraceParams& TP, float* rgb, float* vis, float* ind,
                         cudaStream_t st, uint64_t key_base, const float* valid) {
    const int St = nd + ns;
    const int64_t pc = chunk_points(St);
    WaveScratch w;
    cudaError_t e = w.alloc((P < pc ? P : pc) * St, false, st);
    if (e != cudaSuccess) return e;
    for (int64_t p0 = 0; p0 < P && e == cudaSuccess; p0 += pc) {
        const int64_t np = P - p0 < pc ? P - p0 : pc;
        const int64_t rays = np * St;
        k_wave_gen<<<grid_for(rays, 256), 256, 0, st>>>(x, n, r, wo, p0, rays, St, nd, mode, seed, bounds, w.dir,
                                                        w.key, w.val, key_base, valid);
        if (rays > kWaveUnsortedMax) e = sort_pairs(w.key, w.val, w.key_tmp, w.val_tmp, w.hist, rays, st);
        if (e != cudaSuccess) break;
        e = wave_trace<false>(S, TP, x, p0, St, rays, w, st);
        if (e != cudaSuccess) break;
        k_wave_shade<<<grid_for(np, kWaveThreads / 32), kWaveThreads, 0, st>>>(
            S, x, n, a, r, wo, p0, np, env, H, W, nd, ns, mode, seed, TP, w.res, rgb, vis, ind, key_base, valid);
        count_launches(2);
        e = cudaGetLastError();
    }
    const cudaError_t ef = w.release(st);
    return e != cudaSuccess ? e : ef;
}

cudaError_t wave_backward(const SceneView& S, const int32_t* perm, const uint32_t* bounds, const float* x,
                          const float* n, const float* a, const float* r, const float* wo, int64_t P,
                          const float* env, int H, int W, int nd, int ns, int mode, uint64_t seed,
                          const TraceParams& TP, const float* g_rgb, float* g_albedo, float* g_rough, float* g_env,
                          float* g_means, float* g_quats, float* g_scales, float* g_opacity, float* g_features,
                          cudaStream_t st) {
    constexpr int N = GradRow<3>::N;
    const int St = nd + ns;
    const int64_t pc = chunk_points(St);
    const size_t row_bytes = sizeof(float) * N * (size_t)(S.n > 0 ? S.n : 1);
    float* acc_rows = nullptr;
    cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&acc_rows), row_bytes, st);
    if (e != cudaSuccess) return e;
    WaveScratch w;
    e = cudaMemsetAsync(acc_rows, 0, row_bytes, st);
    if (e == cudaSuccess) e = w.alloc((P < pc ? P : pc) * St, true, st);
    for (int64_t p0 = 0; p0 < P && e == cudaSuccess; p0 += pc) {
        const int64_t np = P - p0 < pc ? P - p0 : pc;
        const int64_t rays = np * St;
        k_wave_gen<<<grid_for(rays, 256), 256, 0, st>>>(x, n, r, wo, p0, rays, St, nd, mode, seed, bounds, w.dir,
                                                        w.key, w.val, 0ull, nullptr);
        if (rays > kWaveUnsortedMax) e = sort_pairs(w.key, w.val, w.key_tmp, w.val_tmp, w.hist, rays, st);
        if (e != cudaSuccess) break;
        const unsigned g = grid_for(rays, kWaveThreads);
        e = wave_trace<true>(S, TP, x, p0, St, rays, w, st);
        if (e != cudaSuccess) break;
        k_wave_grad_point<<<grid_for(np, kWaveThreads / 32), kWaveThreads, 0, st>>>(
            n, a, r, wo, p0, np, env, H, W, nd, ns, mode, seed, w.res, g_rgb, g_albedo, g_rough, g_env, w.up);
        k_wave_backward<<<g, kWaveThreads, 0, st>>>(S, TP, x, p0, St, w.dir, w.val, rays, w.res, w.nh, w.ids,
                                                       kWaveSavedHits, w.up, acc_rows, w.list, w.count + 1);
        k_wave_replay<<<kWaveReplayBlocks, kWarpRayThreads, 0, st>>>(S, TP, x, p0, St, w.dir, w.val, w.res, w.nh,
                                                                     w.up, acc_rows, w.list, w.count + 1);
        count_launches(4);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && S.n > 0) {
        k_grad_scatter<3><<<grid_for(S.n, 256), 256, 0, st>>>(perm, S.n, acc_rows, TP.fc, S.F, TP.off, g_means,
                                                             g_quats, g_scales, g_opacity, g_features);
        count_launches(1);
        e = cudaGetLastError();
    }
    const cudaError_t ef = w.release(st);
    const cudaError_t ea = cudaFreeAsync(acc_rows, st);
    if (e != cudaSuccess) return e;
    return ef != cudaSuccess ? ef : ea;
}

irgs_status to_status(cudaError_t e) {
    if (e == cudaSuccess) return IRGS_OK;
    return e == cudaErrorMemoryAllocation ? IRGS_ERR_OOM : IRGS_ERR_CUDA;
}

}  // namespace

irgs_status launch_shade_wave(const SceneView& S, const uint32_t* bounds, const float* x, const float* n,
                              const float* albedo, const float* rough, const float* wo, int64_t P, const float* env,
                              int32_t H, int32_t W, int32_t n_diffuse, int32_t n_spec, uint64_t seed, int mode,
                              const irgs_trace_params& p, float* rgb, float* vis, float* ind, cudaStream_t st,
                              uint64_t key_base, const float* valid) {
    if (P == 0) return IRGS_OK;
    const TraceParams TP = to_params(p);
    if (p.k != 8 && p.k != 16) return IRGS_ERR_UNSUPPORTED;
    return to_status(wave_forward(S, bounds, x, n, albedo, rough, wo, P, env, H, W, n_diffuse, n_spec, mode, seed, TP,
                                  rgb, vis, ind, st, key_base, valid));
}

irgs_status launch_shade_wave_backward(const SceneView& S, const int32_t* perm, const uint32_t* bounds,
                                       const float* x, const float* n, const float* albedo, const float* rough,
                                       const float* wo, int64_t P, const float* env, int32_t H, int32_t W,
                                       int32_t n_diffuse, int32_t n_spec, uint64_t seed, int mode,
                                       const irgs_trace_params& p, const float* g_rgb, float* g_albedo,
                                       float* g_rough, float* g_env, float* g_means, float* g_quats, float* g_scales,
                                       float* g_opacity, float* g_features, cudaStream_t st) {
    if (P == 0) return IRGS_OK;
    const TraceParams TP = to_params(p);
    if (p.k != 8 && p.k != 16) return IRGS_ERR_UNSUPPORTED;
    return to_status(wave_backward(S, perm, bounds, x, n, albedo, rough, wo, P, env, H, W, n_diffuse, n_spec, mode,
                                   seed, TP, g_rgb, g_albedo, g_rough, g_env, g_means, g_quats, g_scales, g_opacity,
                                   g_features, st));
}

}  // namespace irgs
