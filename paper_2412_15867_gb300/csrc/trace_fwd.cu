// Forward trace kernels, Trace(r_o, r_d) of IRGS Eq. 8: a warp per ray for small
// batches, else packets of 32 rays that walk together, or a lane per ray.
#include <cuda_runtime.h>

#include "scene.h"
#include "trace.cuh"
#include "trace_warp.cuh"

namespace irgs {
namespace {

// Rows at least this wide are regrouped (narrower ones are tiles already, or no rows at all).
constexpr int kMinRowWidth = 32;
constexpr int kMaxRowWidth = 1 << 13;

// Width of the image whose pixel rows the rays seem to be, else 0: the first
// neighbours whose directions differ by more than twice the first
// difference end a row, if the next row starts beside its start. A hint:
// it only decides which rays share a warp.
__global__ void __launch_bounds__(1024) k_row_width(const float* __restrict__ rd, int64_t R, int32_t* __restrict__ width) {
    __shared__ int s_first;
    if (threadIdx.x == 0) s_first = INT32_MAX;
    auto diff2 = [&](int64_t i, int64_t j) {
        const float x = rd[3 * i] - rd[3 * j], y = rd[3 * i + 1] - rd[3 * j + 1], z = rd[3 * i + 2] - rd[3 * j + 2];
        return x * x + y * y + z * z;
    };
    const float unit = diff2(0, 1);
    const int last = (int)(R - 1 < kMaxRowWidth ? R - 1 : kMaxRowWidth);
    __syncthreads();
    for (int i0 = 1; i0 < last; i0 += 1024) {
        const int i = i0 + threadIdx.x;
        if (i < last && diff2(i, i + 1) > 4.f * unit) atomicMin(&s_first, i);
        __syncthreads();
        if (s_first != INT32_MAX) break;   // the same for every thread: nothing writes it until the next pass
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const int64_t w = s_first == INT32_MAX ? 0 : (int64_t)s_first + 1;
        *width = w >= kMinRowWidth && w < R && diff2(0, w) < 9.f * unit ? (int32_t)w : 0;
    }
}


template <int FB, bool PACKET>
__global__ void __launch_bounds__(kTraceThreads, kPacketBlocks) k_trace_forward(SceneView S, const float* __restrict__ ro,
                                                                    const float* __restrict__ rd, int64_t R,
                                                                    TraceParams P, float* __restrict__ feat,
                                                                    float* __restrict__ depth,
                                                                    float* __restrict__ opac,
                                                                    int32_t* __restrict__ nhits,
                                                                    int32_t* __restrict__ ids, int max_ids,
                                                                    const int32_t* __restrict__ width) {
    const int64_t t = blockIdx.x * (int64_t)kTraceThreads + threadIdx.x;
    const bool live = t < R;
    const int64_t r = live ? tiled_ray(t, R, width) : 0, q = r;   // lanes without a ray follow the warp with a dummy ray
    const Ray ray = make_ray(mk3(ro[3 * q], ro[3 * q + 1], ro[3 * q + 2]),
                             mk3(rd[3 * q], rd[3 * q + 1], rd[3 * q + 2]));
    int32_t* my_ids = (ids != nullptr && live) ? ids + r * (int64_t)max_ids : nullptr;
    MarchState<FB> st;
    const bool ok = march_forward<FB, PACKET>(S, ray, P, st, my_ids, max_ids, live, warp_scratch<PACKET>());
    if (!live) return;
    if (my_ids != nullptr && st.nh < max_ids) my_ids[st.nh] = -1;   // terminator
    if (!ok) atomicOr(S.status, kErrStackOverflow);
#pragma unroll
    for (int c = 0; c < FB; ++c)
        if (c < P.fc) feat[r * P.fc + c] = st.C[c];
    depth[r] = st.D;
    opac[r] = 1.0f - st.T;
    if (nhits != nullptr) nhits[r] = st.nh;
}

// One warp per ray.
__global__ void __launch_bounds__(kWarpRayThreads, kWarpRayBlocks) k_trace_ray(SceneView S, const float* __restrict__ ro,
                                                                               const float* __restrict__ rd, int64_t R,
                                                                               TraceParams P, float* __restrict__ feat,
                                                                               float* __restrict__ depth,
                                                                               float* __restrict__ opac,
                                                                               int32_t* __restrict__ nhits,
                                                                               int32_t* __restrict__ ids, int max_ids) {
    const int64_t r = blockIdx.x * (int64_t)kWarpRays + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (r >= R) return;
    const Ray ray = make_ray(mk3(ro[3 * r], ro[3 * r + 1], ro[3 * r + 2]), mk3(rd[3 * r], rd[3 * r + 1], rd[3 * r + 2]));
    int32_t* my_ids = ids != nullptr ? ids + r * (int64_t)max_ids : nullptr;
    RayBox rb = make_ray_box(ray);
    if (!can_hit(ray)) {   // behind every box (a branch around the march cost 9%)
        rb.inv = mk3(0.f, 0.f, 0.f);
        rb.oinv = mk3(INFINITY, INFINITY, INFINITY);
    }
    WarpMarch st;
    const bool ok = march_warp(S, ray, rb, P, st, my_ids, max_ids, warp_ray_scratch());
    if (lane < P.fc) feat[r * P.fc + lane] = st.C;
    if (lane != 0) return;
    if (my_ids != nullptr && st.nh < max_ids) my_ids[st.nh] = -1;   // terminator
    if (!ok) atomicOr(S.status, kErrStackOverflow);
    depth[r] = st.D;
    opac[r] = 1.0f - st.T;
    if (nhits != nullptr) nhits[r] = st.nh;
}

// ---------------------------------------------------------------------------
// Compacted rounds (large packet batches). Most rays end in their first
// k-buffer round; a warp would walk as many rounds as its slowest ray with
// few lanes still active. Here round 1 runs on every ray; rays not done
// after it store their march state and are regrouped, in ray order, into
// full warps that run to completion. Per ray the rounds and their arithmetic
// are those of march_forward, so the results are bitwise the same; only
// which rays share a warp changes.
enum RoundMode { kRoundFirst = 0, kRoundLast = 1 };

// Between rounds: C[FB], D, T, hit count, next key (2 words), next user index.
template <int FB>
struct RoundState {
    static constexpr int kF4 = (FB + 6 + 3) / 4;
};

template <int FB, int MODE>
__global__ void __launch_bounds__(kTraceThreads, kPacketBlocks) k_trace_round(
    SceneView S, const float* __restrict__ ro, const float* __restrict__ rd, int64_t R, TraceParams P,
    float* __restrict__ feat, float* __restrict__ depth, float* __restrict__ opac, int32_t* __restrict__ nhits,
    int32_t* __restrict__ ids, int max_ids, const int32_t* __restrict__ list, const uint32_t* __restrict__ count,
    float4* __restrict__ state, uint32_t* __restrict__ flags, const int32_t* __restrict__ width) {
    constexpr int SW = RoundState<FB>::kF4;
    const int64_t t = blockIdx.x * (int64_t)kTraceThreads + threadIdx.x;
    const int64_t n = MODE == kRoundFirst ? R : (int64_t)*count;
    if (__all_sync(kFullWarp, t >= n)) return;   // nothing for this warp
    const bool live = t < n;
    // slot: the ray's place in the order the warps are made in
    const int64_t slot = live ? (MODE == kRoundFirst ? t : (int64_t)list[t]) : 0;
    const int64_t r = live ? tiled_ray(slot, R, width) : 0;
    const Ray ray = make_ray(mk3(ro[3 * r], ro[3 * r + 1], ro[3 * r + 2]),
                             mk3(rd[3 * r], rd[3 * r + 1], rd[3 * r + 2]));
    MarchState<FB> st;
    uint64_t last_key = depth_key(P.t_min, 0.f);
    int32_t last_u = INT32_MAX;
    if (MODE == kRoundFirst || !live) {
        st.init();
    } else {
        float w[4 * SW];
#pragma unroll
        for (int q = 0; q < SW; ++q) {
            const float4 v = state[slot * SW + q];
            w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
        }
#pragma unroll
        for (int c = 0; c < FB; ++c) st.C[c] = w[c];
        st.D = w[FB];
        st.T = w[FB + 1];
        st.nh = __float_as_int(w[FB + 2]);
        last_key = ((uint64_t)__float_as_uint(w[FB + 4]) << 32) | (uint64_t)__float_as_uint(w[FB + 3]);
        last_u = __float_as_int(w[FB + 5]);
    }
    int32_t* my_ids = (ids != nullptr && live) ? ids + r * (int64_t)max_ids : nullptr;
    KBuffer<kCap> kb;
    kb.bind();
    float4* scratch = warp_scratch<true>();
    bool ok = true, done = !live, packet = true;
    do {
        ok &= collect<true>(S, ray, P, last_key, last_u, st.T, kb, !done, packet, scratch);
        if (!done) done = blend_round<FB>(S, ray, P, kb, st, my_ids, max_ids, last_key, last_u);
    } while (MODE == kRoundLast && __any_sync(kFullWarp, !done));
    if (!live) return;
    if (!ok) atomicOr(S.status, kErrStackOverflow);
    if (done) {
        if (my_ids != nullptr && st.nh < max_ids) my_ids[st.nh] = -1;   // terminator
#pragma unroll
        for (int c = 0; c < FB; ++c)
            if (c < P.fc) feat[r * P.fc + c] = st.C[c];
        depth[r] = st.D;
        opac[r] = 1.0f - st.T;
        if (nhits != nullptr) nhits[r] = st.nh;
    } else {
        float w[4 * SW];
#pragma unroll
        for (int c = 0; c < FB; ++c) w[c] = st.C[c];
        w[FB] = st.D;
        w[FB + 1] = st.T;
        w[FB + 2] = __int_as_float(st.nh);
        w[FB + 3] = __uint_as_float((uint32_t)last_key);
        w[FB + 4] = __uint_as_float((uint32_t)(last_key >> 32));
        w[FB + 5] = __int_as_float(last_u);
#pragma unroll
        for (int c = FB + 6; c < 4 * SW; ++c) w[c] = 0.f;
#pragma unroll
        for (int q = 0; q < SW; ++q) state[slot * SW + q] = make_float4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
        flags[slot] = 1u;
    }
}

// Batches at least this large take the compacted rounds.
constexpr int64_t kRoundMinRays = int64_t(1) << 20;

template <int FB>
cudaError_t launch_rounds(const SceneView& S, const float* ro, const float* rd, int64_t R, const TraceParams& P,
                          float* feat, float* depth, float* opac, int32_t* nhits, int32_t* ids, int max_ids,
                          const int32_t* width, cudaStream_t st) {
    constexpr int threads = kTraceThreads;
    constexpr int SW = RoundState<FB>::kF4;
    const int64_t sums = scan_long_words(R + 1);
    // scratch: flags / positions [R + 1], list [R], count, scan sums, then the states (16-byte aligned)
    const int64_t words = (R + 1) + R + 1 + sums;
    const size_t state_off = (size_t)((words * 4 + 255) / 256 * 256);
    const size_t bytes = state_off + sizeof(float4) * SW * (size_t)R;
    unsigned char* base = nullptr;
    cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&base), bytes, st);
    if (e != cudaSuccess) return e;
    uint32_t* flags = reinterpret_cast<uint32_t*>(base);
    int32_t* list = reinterpret_cast<int32_t*>(flags + R + 1);
    uint32_t* count = reinterpret_cast<uint32_t*>(list + R);
    uint32_t* scan_sums = count + 1;
    float4* state = reinterpret_cast<float4*>(base + state_off);
    const unsigned grid = (unsigned)((R + threads - 1) / threads);
    e = cudaMemsetAsync(flags, 0, sizeof(uint32_t) * (R + 1), st);
    if (e == cudaSuccess) {
        k_trace_round<FB, kRoundFirst><<<grid, threads, 0, st>>>(S, ro, rd, R, P, feat, depth, opac, nhits, ids,
                                                                  max_ids, list, count, state, flags, width);
        e = flags_to_list(flags, R, scan_sums, list, count, st);
        if (e == cudaSuccess)
            k_trace_round<FB, kRoundLast><<<grid, threads, 0, st>>>(S, ro, rd, R, P, feat, depth, opac, nhits, ids,
                                                                    max_ids, list, count, state, flags, width);
        count_launches(2);
    }
    const cudaError_t ef = cudaFreeAsync(base, st);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e != cudaSuccess ? e : ef;
}

template <int FB, bool PACKET>
cudaError_t launch(const SceneView& S, const float* ro, const float* rd, int64_t R, const TraceParams& P,
                   float* feat, float* depth, float* opac, int32_t* nhits, int32_t* ids, int max_ids,
                   const int32_t* width, cudaStream_t st) {
    if constexpr (PACKET) {
        // the ray list holds int32 indices; without room for the scratch the
        // single-kernel march below does the same work
        if (R >= kRoundMinRays && R < INT32_MAX && S.n > 0) {
            const cudaError_t e = launch_rounds<FB>(S, ro, rd, R, P, feat, depth, opac, nhits, ids, max_ids, width, st);
            if (e != cudaErrorMemoryAllocation) return e;
            cudaGetLastError();   // clear the failed allocation
        }
    }
    const int64_t blocks = (R + kTraceThreads - 1) / kTraceThreads;
    k_trace_forward<FB, PACKET><<<(unsigned)blocks, kTraceThreads, 0, st>>>(S, ro, rd, R, P, feat, depth, opac,
                                                                           nhits, ids, max_ids, width);
    count_launches(1);
    return cudaGetLastError();
}

template <bool PACKET>
cudaError_t launch_f(const SceneView& S, const float* ro, const float* rd, int64_t R, const TraceParams& P,
                     float* feat, float* depth, float* opac, int32_t* nhits, int32_t* ids, int max_ids,
                     cudaStream_t st) {
    RowWidth w(rd, R, PACKET, st);
    const auto f = P.fc <= 3 ? launch<3, PACKET> : (P.fc <= 10 ? launch<10, PACKET> : launch<16, PACKET>);
    const cudaError_t e = f(S, ro, rd, R, P, feat, depth, opac, nhits, ids, max_ids, w.get(), st);
    return e;
}

// Diagnostic: the march with per-ray counters and a k-buffer of 16 entries (the
// other calls' has kCap, so they need fewer rounds and fewer walks), <= 10
// channels. A packet's node fetches count for each of its rays.
template <bool PACKET>
__global__ void __launch_bounds__(128) k_trace_stats(SceneView S, const float* __restrict__ ro,
                                                     const float* __restrict__ rd, int64_t R, TraceParams P,
                                                     int32_t* __restrict__ stats) {
    const int64_t r = blockIdx.x * (int64_t)128 + threadIdx.x;
    const bool live = r < R;
    const int64_t q = live ? r : 0;
    const Ray ray = make_ray(mk3(ro[3 * q], ro[3 * q + 1], ro[3 * q + 2]),
                             mk3(rd[3 * q], rd[3 * q + 1], rd[3 * q + 2]));
    MarchState<10> st;
    TraceStats ts = {0, 0, 0, 0};
    march_forward<10, PACKET, 16, true>(S, ray, P, st, nullptr, 0, live, warp_scratch<PACKET>(), &ts);
    if (!live) return;
    stats[4 * r] = ts.rounds;
    stats[4 * r + 1] = ts.nodes;
    stats[4 * r + 2] = ts.leaves;
    stats[4 * r + 3] = ts.inserts;
}

}  // namespace

RowWidth::RowWidth(const float* rd, int64_t R, bool wanted, cudaStream_t st) : st_(st) {
    if (!wanted || R < kRowMinRays || R >= INT32_MAX) return;
    if (scratch_alloc(reinterpret_cast<void**>(&width_), sizeof(int32_t), st) != cudaSuccess) {
        cudaGetLastError();   // no hint, then
        width_ = nullptr;
        return;
    }
    k_row_width<<<1, 1024, 0, st>>>(rd, R, width_);
    count_launches(1);
}

RowWidth::~RowWidth() {
    if (width_ != nullptr) cudaFreeAsync(width_, st_);
}

irgs_status launch_trace_stats(const SceneView& S, const float* ro, const float* rd, int64_t R,
                               const irgs_trace_params& p, int32_t* stats, cudaStream_t st) {
    if (R == 0) return IRGS_OK;
    const TraceParams P = to_params(p);
    const unsigned blocks = (unsigned)((R + 127) / 128);
    if ((p.flags & IRGS_FLAG_PER_THREAD) == 0u)
        k_trace_stats<true><<<blocks, 128, 0, st>>>(S, ro, rd, R, P, stats);
    else
        k_trace_stats<false><<<blocks, 128, 0, st>>>(S, ro, rd, R, P, stats);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

irgs_status launch_trace_forward(const SceneView& S, const float* ro, const float* rd, int64_t R,
                                 const irgs_trace_params& p, float* feat, float* depth, float* opac,
                                 int32_t* nhits, int32_t* ids, int32_t max_ids, cudaStream_t st) {
    if (R == 0) return IRGS_OK;
    const TraceParams P = to_params(p);
    if (p.flags == 0u && R <= kWarpRayMax) {
        k_trace_ray<<<warp_ray_grid(R), kWarpRayThreads, 0, st>>>(S, ro, rd, R, P, feat, depth, opac, nhits, ids, max_ids);
        count_launches(1);
        return cudaGetLastError() == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
    }
    const bool packet = (p.flags & IRGS_FLAG_PER_THREAD) == 0u;
    const cudaError_t e = packet ? launch_f<true>(S, ro, rd, R, P, feat, depth, opac, nhits, ids, max_ids, st)
                                 : launch_f<false>(S, ro, rd, R, P, feat, depth, opac, nhits, ids, max_ids, st);
    if (e == cudaErrorMemoryAllocation) return IRGS_ERR_OOM;
    return e == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

}  // namespace irgs
