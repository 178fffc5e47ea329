// Backward trace kernels: each ray's hits come from the forward's saved hit
// list or from a replay of its march (trace_bwd.cuh); the surfel gradients
// are accumulated in Morton order and then added into the caller's
// user-order arrays.
#include <cuda_runtime.h>

#include "scene.h"
#include "trace.cuh"
#include "trace_bwd.cuh"

namespace irgs {
namespace {

constexpr int kBwdThreads = kTraceThreads;

// Which rays a launch handles.
enum BwdMode {
    kReplayAll = 0,    // every ray replays the march (no hit lists)
    kListed = 1,       // rays whose whole hit list was saved; no traversal code
    kReplayLong = 2,   // rays whose hit list did not fit replay the march
};

// Rays whose hit list did not fit: the listing launch counts and lists them.
// Up to a sixteenth of the batch they take a warp each; beyond that the packets
// of kReplayLong replay them. Both launches follow, one of them finds nothing
// to do. The list has room for no more than that.
constexpr int kLongShare = 16;
__host__ __device__ __forceinline__ int64_t long_room(int64_t R) { return R < INT32_MAX ? R / kLongShare : 0; }
__device__ __forceinline__ bool few_long(uint32_t count, int64_t R) { return (int64_t)count <= long_room(R); }

// Per-ray inputs of the backward (forward outputs and upstream gradients).
template <int FB>
struct RayGrad {
    float gC[FB], Cf[FB];
    float gD, gO, Df, Tfin;
};

template <int FB>
__device__ __forceinline__ void load_ray_grad(RayGrad<FB>& g, int64_t q, const TraceParams& P,
                                              const float* __restrict__ out_feat, const float* __restrict__ out_depth,
                                              const float* __restrict__ out_opac, const float* __restrict__ g_featv,
                                              const float* __restrict__ g_depthv,
                                              const float* __restrict__ g_opacv) {
#pragma unroll
    for (int c = 0; c < FB; ++c) {
        g.gC[c] = c < P.fc ? g_featv[q * P.fc + c] : 0.f;
        g.Cf[c] = c < P.fc ? out_feat[q * P.fc + c] : 0.f;
    }
    g.gD = g_depthv != nullptr ? g_depthv[q] : 0.f;
    g.gO = g_opacv != nullptr ? g_opacv[q] : 0.f;
    g.Df = out_depth[q];
    g.Tfin = 1.0f - out_opac[q];
}

template <int FB, bool PACKET, int MODE>
__global__ void __launch_bounds__(kBwdThreads) k_trace_backward(
    SceneView S, const float* __restrict__ ro, const float* __restrict__ rd, int64_t R, TraceParams P,
    const float* __restrict__ out_feat, const float* __restrict__ out_depth, const float* __restrict__ out_opac,
    const int32_t* __restrict__ out_nhits, const int32_t* __restrict__ hit_ids, int max_ids,
    const float* __restrict__ g_featv, const float* __restrict__ g_depthv, const float* __restrict__ g_opacv,
    float* __restrict__ acc_rows, const int32_t* __restrict__ width, int32_t* __restrict__ long_list,
    uint32_t* __restrict__ long_count) {
    float4* scratch = warp_memory<MODE == kListed ? 32 * GradRow<FB>::kStride / 4 : replay_f4<FB, PACKET>()>();
    const int64_t t = blockIdx.x * (int64_t)kBwdThreads + threadIdx.x;
    if (S.n == 0) return;
    const int64_t r = t < R ? tiled_ray(t, R, width) : R;
    const int nh_total = r < R ? out_nhits[r] : 0;
    const bool mine = nh_total > 0 && (MODE == kReplayAll || (MODE == kListed) == (nh_total <= max_ids));
    if (MODE == kReplayLong && few_long(*long_count, R)) return;
    if (MODE == kListed) {
        const unsigned longer = __ballot_sync(kFullWarp, nh_total > max_ids);
        if (longer != 0u) {
            const int lane = threadIdx.x & 31, first = __ffs(longer) - 1;
            uint32_t base = 0u;
            if (lane == first) base = atomicAdd(long_count, (uint32_t)__popc(longer));
            base = __shfl_sync(kFullWarp, base, first);
            const int64_t at = (int64_t)base + __popc(longer & ((1u << lane) - 1u));
            if (nh_total > max_ids && at < long_room(R)) long_list[at] = (int32_t)r;
        }
        if (!mine) return;
    } else if (!__any_sync(kFullWarp, mine)) {
        return;   // the whole warp has nothing to replay
    }
    const int64_t q = mine ? r : 0;   // lanes without work follow the warp with a dummy ray
    const Ray ray = make_ray(mk3(ro[3 * q], ro[3 * q + 1], ro[3 * q + 2]),
                             mk3(rd[3 * q], rd[3 * q + 1], rd[3 * q + 2]));
    RayGrad<FB> g;
    load_ray_grad<FB>(g, q, P, out_feat, out_depth, out_opac, g_featv, g_depthv, g_opacv);
    if (MODE == kListed) {
        listed_backward<FB>(S, ray, P, hit_ids + q * (int64_t)max_ids, nh_total, g.Cf, g.Df, g.Tfin, g.gC, g.gD,
                            g.gO, acc_rows, reinterpret_cast<float*>(scratch));
    } else {
        const bool ok = march_backward<FB, PACKET>(S, ray, P, mine, nh_total, g.Cf, g.Df, g.Tfin, g.gC, g.gD, g.gO, acc_rows,
                                                   scratch);
        if (mine && !ok) atomicOr(S.status, kErrStackOverflow);
    }
}

// A warp per ray: all rays (list = nullptr), or those of the list while they
// are few, warps taking entries in turn.
template <int FB>
__global__ void __launch_bounds__(kWarpRayThreads) k_trace_backward_ray(
    SceneView S, const float* __restrict__ ro, const float* __restrict__ rd, int64_t R, TraceParams P,
    const float* __restrict__ out_feat, const float* __restrict__ out_depth, const float* __restrict__ out_opac,
    const int32_t* __restrict__ out_nhits, const float* __restrict__ g_featv, const float* __restrict__ g_depthv,
    const float* __restrict__ g_opacv, float* __restrict__ acc_rows, const int32_t* __restrict__ list,
    const uint32_t* __restrict__ count) {
    if (S.n == 0 || (list != nullptr && !few_long(*count, R))) return;
    const int64_t n = list != nullptr ? (int64_t)*count : R;
    const int lane = threadIdx.x & 31;
    for (int64_t t = blockIdx.x * (int64_t)kWarpRays + (threadIdx.x >> 5); t < n; t += (int64_t)gridDim.x * kWarpRays) {
        const int64_t r = list != nullptr ? (int64_t)list[t] : t;
        const int nh_total = out_nhits[r];
        if (nh_total <= 0) continue;
        const Ray ray = make_ray(mk3(ro[3 * r], ro[3 * r + 1], ro[3 * r + 2]),
                                 mk3(rd[3 * r], rd[3 * r + 1], rd[3 * r + 2]));
        const bool mine = lane < P.fc;
        const bool ok = backward_warp<FB>(S, ray, P, nh_total, mine ? out_feat[r * P.fc + lane] : 0.f, out_depth[r],
                                          1.0f - out_opac[r], mine ? g_featv[r * P.fc + lane] : 0.f,
                                          g_depthv != nullptr ? g_depthv[r] : 0.f,
                                          g_opacv != nullptr ? g_opacv[r] : 0.f, acc_rows, warp_ray_scratch());
        if (!ok && lane == 0) atomicOr(S.status, kErrStackOverflow);
    }
}

constexpr unsigned kLongBlocks = 152 * 4;   // blocks that share the listed rays

// Pointers of one backward call (see irgs_trace_backward).
struct BwdArgs {
    const int32_t* perm;
    const float *ro, *rd;
    int64_t R;
    const float *feat, *depth, *opac;
    const int32_t *nhits, *ids;
    int max_ids;
    const float *gf, *gd, *go;
    float *gm, *gq, *gs, *gop, *gfe;
};

template <int FB, bool PACKET>
cudaError_t launch(const SceneView& S, const TraceParams& P, const BwdArgs& a, bool warp_rays, cudaStream_t st) {
    constexpr int N = GradRow<FB>::N;
    const size_t row_bytes = sizeof(float) * N * (size_t)(S.n > 0 ? S.n : 1);
    // rows, then with hit lists the long rays' count and list
    const size_t list_at = (row_bytes + 255) / 256 * 256;
    const size_t bytes = a.ids != nullptr ? list_at + sizeof(uint32_t) * (size_t)(long_room(a.R) + 64) : row_bytes;
    unsigned char* base = nullptr;
    cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&base), bytes, st);
    if (e != cudaSuccess) return e;
    float* acc_rows = reinterpret_cast<float*>(base);
    uint32_t* long_count = a.ids != nullptr ? reinterpret_cast<uint32_t*>(base + list_at) : nullptr;
    int32_t* long_list = a.ids != nullptr ? reinterpret_cast<int32_t*>(long_count + 64) : nullptr;
    e = cudaMemsetAsync(base, 0, a.ids != nullptr ? list_at + 4 : row_bytes, st);
    if (e == cudaSuccess) {
        const int64_t blocks = (a.R + kBwdThreads - 1) / kBwdThreads;
        const unsigned grid = (unsigned)blocks;
        const RowWidth w(a.rd, a.R, PACKET && !(warp_rays && a.ids == nullptr), st);
#define IRGS_BWD(MODE)                                                                                  \
    k_trace_backward<FB, PACKET, MODE><<<grid, kBwdThreads, 0, st>>>(S, a.ro, a.rd, a.R, P, a.feat, a.depth, \
                                                                      a.opac, a.nhits, a.ids, a.max_ids, a.gf, \
                                                                      a.gd, a.go, acc_rows, w.get(), long_list, long_count)
        if (a.ids != nullptr) {
            IRGS_BWD(kListed);
            IRGS_BWD(kReplayLong);
            k_trace_backward_ray<FB><<<kLongBlocks, kWarpRayThreads, 0, st>>>(
                S, a.ro, a.rd, a.R, P, a.feat, a.depth, a.opac, a.nhits, a.gf, a.gd, a.go, acc_rows, long_list, long_count);
            count_launches(2);
        } else if (warp_rays) {
            k_trace_backward_ray<FB><<<warp_ray_grid(a.R), kWarpRayThreads, 0, st>>>(
                S, a.ro, a.rd, a.R, P, a.feat, a.depth, a.opac, a.nhits, a.gf, a.gd, a.go, acc_rows, nullptr, nullptr);
        } else {
            IRGS_BWD(kReplayAll);
        }
#undef IRGS_BWD
        if (S.n > 0)
            k_grad_scatter<FB><<<(unsigned)((S.n + 255) / 256), 256, 0, st>>>(a.perm, S.n, acc_rows, P.fc, S.F, P.off,
                                                                             a.gm, a.gq, a.gs, a.gop, a.gfe);
        count_launches(S.n > 0 ? 2 : 1);
        e = cudaGetLastError();
    }
    cudaError_t ef = cudaFreeAsync(base, st);
    return e != cudaSuccess ? e : ef;
}

template <bool PACKET>
cudaError_t launch_f(const SceneView& S, const TraceParams& P, const BwdArgs& a, bool warp_rays, cudaStream_t st) {
    if (P.fc <= 3) return launch<3, PACKET>(S, P, a, warp_rays, st);
    if (P.fc <= 10) return launch<10, PACKET>(S, P, a, warp_rays, st);
    return launch<16, PACKET>(S, P, a, warp_rays, st);
}

}  // namespace

irgs_status launch_trace_backward(const SceneView& S, const int32_t* perm, const float* ro, const float* rd, int64_t R,
                                  const irgs_trace_params& p, const float* feat, const float* depth,
                                  const float* opac, const int32_t* nhits, const int32_t* hit_ids,
                                  int32_t max_hit_ids, const float* g_feat, const float* g_depth, const float* g_opac,
                                  float* g_means, float* g_quats, float* g_scales, float* g_opacity,
                                  float* g_features, cudaStream_t st) {
    if (R == 0) return IRGS_OK;
    const TraceParams P = to_params(p);
    const BwdArgs a{perm,  ro,     rd,      R,       feat,     depth,     opac,      nhits,     hit_ids,
                    hit_ids != nullptr ? max_hit_ids : 0, g_feat, g_depth, g_opac, g_means, g_quats, g_scales,
                    g_opacity, g_features};
    const bool packet = (p.flags & IRGS_FLAG_PER_THREAD) == 0u;
    // without hit lists, batches that the forward gives a warp per ray are replayed so too
    const bool warp_rays = p.flags == 0u && R <= kWarpRayMax;
    const cudaError_t e = packet ? launch_f<true>(S, P, a, warp_rays, st) : launch_f<false>(S, P, a, false, st);
    if (e == cudaErrorMemoryAllocation) return IRGS_ERR_OOM;
    return e == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

}  // namespace irgs
