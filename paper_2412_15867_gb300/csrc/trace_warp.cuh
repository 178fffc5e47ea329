// A warp per ray: the march of trace.cuh for rays that do not run together, in
// batches that do not fill the chip many times over with a ray per lane (a
// lane walks some 75 nodes and 65 surfels one after the other, a microsecond
// each, and the longest ray of a batch ten times that). The 32 lanes test 8
// nodes x 4 children, or 32 surfels, of the same ray at a time, and the
// round's nearest hits are kept in order in registers, the i-th in lane i.
// Bound by instruction issue (80% of the slots), so the rate hardly depends on
// the batch's size: 230 to 260 Mrays/s for camera rays, 260 for relighting's and 340
// for shading's samples, which meet fewer surfels. Half a warp per ray (two hits per lane) was 10% slower: its
// nodes and leaves come in smaller portions. Hits, order and blending
// arithmetic are those of march_forward, so the results are the same.
#pragma once

#include "trace.cuh"

namespace irgs {

struct WarpRayScratch {
    uint2 stack[kPacketStack];   // (wide node, entry depth bits)
    uint32_t leaf[64];
};

// The nearest hits of a round, in order: lane i holds the i-th of cnt.
struct WarpHits {
    uint32_t kh, kl;   // depth_key's words
    int32_t m;         // Morton slot
    float a;           // alpha
    int cnt;
    bool closed;       // bounded by its last entry: more hits may follow
    __device__ __forceinline__ void clear() {
        kh = kl = 0xffffffffu;
        m = 0;
        a = 0.f;
        cnt = 0;
    }
    __device__ __forceinline__ uint64_t key() const { return (uint64_t)kh << 32 | kl; }
    __device__ __forceinline__ uint64_t key_of(int i) const {
        return (uint64_t)__shfl_sync(kFullWarp, kh, i) << 32 | __shfl_sync(kFullWarp, kl, i);
    }
};

// A hit (the same for all lanes) into its place in the list; the 33rd falls off.
__device__ __forceinline__ void insert_hit(WarpHits& h, uint32_t nh, uint32_t nl, int32_t nm, float na,
                                           const float4* rec) {
    const int lane = threadIdx.x & 31;
    const uint64_t nk = (uint64_t)nh << 32 | nl;
    const bool there = lane < h.cnt;
    // the entries before it are a prefix of the lanes
    int pos = __popc(__ballot_sync(kFullWarp, there && h.key() < nk));
    const unsigned tie = __ballot_sync(kFullWarp, there && h.key() == nk);
    if (tie != 0u) {   // equal exact depths: by user index
        const int32_t nu = uid_of(rec, nm);
        pos += __popc(__ballot_sync(kFullWarp, ((tie >> lane) & 1u) && uid_of(rec, h.m) < nu));
    }
    if (pos < 32 && h.cnt < 32) ++h.cnt;
    const uint32_t ph = __shfl_up_sync(kFullWarp, h.kh, 1), pl = __shfl_up_sync(kFullWarp, h.kl, 1);
    const int32_t pm = __shfl_up_sync(kFullWarp, h.m, 1);
    const float pa = __shfl_up_sync(kFullWarp, h.a, 1);
    if (lane >= pos) {
        h.kh = lane > pos ? ph : nh;
        h.kl = lane > pos ? pl : nl;
        h.m = lane > pos ? pm : nm;
        h.a = lane > pos ? pa : na;
    }
}

// Gather the nearest hits of the warp's ray strictly after (last_key, last_u).
// Returns false if the stack overflowed.
__device__ __forceinline__ bool collect_warp(const SceneView& S, const Ray& ray, const RayBox& rb,
                                             const TraceParams& P, uint64_t last_key, int32_t last_u, float T,
                                             WarpRayScratch& ws, WarpHits& h) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const float t_lo = key_depth(last_key);
    const float lo_c = fmaxf(t_lo - tslack(t_lo), 0.f);
    const float bits = 16.f * __log2f(__fdividef(T, P.T_min)) + 2.f;
    const uint32_t need = P.T_min > 0.f && bits < 1e9f ? (uint32_t)fmaxf(bits, 1.f) : 0xffffffffu;
    h.clear();
    h.closed = false;
    uint64_t tail_key = ~0ull;
    float t_hi = P.t_max;
    int sp = 1, nleaf = 0;
    int visits = visit_cap(S);
    __syncwarp();   // the memory's last use is over
    if (lane == 0) ws.stack[0] = make_uint2(0u, 0u);
    __syncwarp();
    while (sp > 0 || nleaf > 0) {
        if (nleaf < 32 && sp > 0) {
            const float hi_c = t_hi + tslack(t_hi);
            // near the stack's end only its top is taken, as a plain depth-first walk would
            const int take = min(sp, sp <= kPacketStack - 96 ? 8 : 1);
            visits -= take;
            const int g = lane >> 2;
            bool in = g < take;
            uint32_t id = 0u;
            if (in) {
                const uint2 ent = ws.stack[sp - 1 - g];
                id = ent.x;
                in = __uint_as_float(ent.y) <= hi_c;
            }
            sp -= take;
            int child = kNoChild;
            float tn = 0.f;
            if (in) {
                const float4* w = S.child_box + (int64_t)id * 8 + (lane & 3) * 2;
                const float4 lo = ldg4(w), hi = ldg4(w + 1);
                child = __float_as_int(lo.w);
                const float x0 = fmaf(lo.x, rb.inv.x, -rb.oinv.x), x1 = fmaf(hi.x, rb.inv.x, -rb.oinv.x);
                const float y0 = fmaf(lo.y, rb.inv.y, -rb.oinv.y), y1 = fmaf(hi.y, rb.inv.y, -rb.oinv.y);
                const float z0 = fmaf(lo.z, rb.inv.z, -rb.oinv.z), z1 = fmaf(hi.z, rb.inv.z, -rb.oinv.z);
                tn = fmaxf(max3f(fminf(x0, x1), fminf(y0, y1), fminf(z0, z1)), lo_c);
                const float tf = fminf(min3f(fmaxf(x0, x1), fmaxf(y0, y1), fmaxf(z0, z1)), hi_c);
                in = tn <= tf && child != kNoChild;
            }
            const unsigned leaves = __ballot_sync(kFullWarp, in && child < 0);
            if (in && child < 0) ws.leaf[nleaf + __popc(leaves & lt)] = (uint32_t)~child;
            nleaf += __popc(leaves);
            const bool inner = in && child >= 0;
            const unsigned push = __ballot_sync(kFullWarp, inner);
            // farther siblings lie deeper, and so do the children of nodes farther down the stack; siblings'
            // depths are told apart but for their last two bits, then by their numbers
            const uint32_t td = inner ? (__float_as_uint(tn) & ~3u) | (uint32_t)(lane & 3) : 0u;
            int at = sp + __popc((push >> (4 * g)) >> 4);
#pragma unroll
            for (int x = 1; x < 4; ++x) at += __shfl_xor_sync(kFullWarp, td, x) > td ? 1 : 0;
            if (sp + __popc(push) > kPacketStack || visits < 0) return false;
            __syncwarp();   // the popped entries have been read
            if (inner) ws.stack[at] = make_uint2((uint32_t)child, __float_as_uint(tn));
            sp += __popc(push);
            __syncwarp();
            continue;
        }
        // up to 32 surfels, one per lane
        const int cnt = min(nleaf, 32);
        bool hit = false;
        uint64_t key = 0u;
        int32_t m = 0;
        float a = 0.f;
        if (lane < cnt) {
            m = (int32_t)ws.leaf[lane];
            const float4* R = S.rec + (int64_t)m * kRecF4;
            const float4 r0 = ldg4(R), r1 = ldg4(R + 1), r2 = ldg4(R + 2), r3 = ldg4(R + 3);
            float kh, kl;
            // the bounds are leaf_insert's
            if (surfel_hit<false>(r0, r1, r2, r3, ray, P.alpha_min, P.alpha_max, kh, kl, a, nullptr, t_lo, t_hi)) {
                key = depth_key(kh, kl);
                hit = (key > last_key || (key == last_key && __float_as_int(r2.w) > last_u)) &&
                      (kh < P.t_max || (kh == P.t_max && kl < 0.f)) && key <= tail_key;
            }
        }
        const uint32_t rest = 32 + lane < nleaf ? ws.leaf[32 + lane] : 0u;
        __syncwarp();
        if (32 + lane < nleaf) ws.leaf[lane] = rest;
        nleaf -= cnt;
        unsigned found = __ballot_sync(kFullWarp, hit);
        if (found == 0u) continue;
        while (found != 0u) {   // each into its place
            const int src = __ffs(found) - 1;
            found &= found - 1u;
            const uint32_t nh = __shfl_sync(kFullWarp, (uint32_t)(key >> 32), src);
            const uint32_t nl = __shfl_sync(kFullWarp, (uint32_t)key, src);
            const int32_t nm = __shfl_sync(kFullWarp, m, src);
            const float na = __shfl_sync(kFullWarp, a, src);
            insert_hit(h, nh, nl, nm, na, S.rec);
        }
        // the shortest prefix that is surely past T_min (the optical depths floor(-16 log2(1 - alpha)) add up to
        // `need`, as in KBuffer), else a full buffer, bounds the walk
        uint32_t sum = lane < h.cnt ? (uint32_t)fminf(fmaxf(-16.f * __log2f(1.f - h.a), 0.f), 255.f) : 0u;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(kFullWarp, sum, off);
            if (lane >= off) sum += y;
        }
        const unsigned past = __ballot_sync(kFullWarp, lane < h.cnt && sum >= need);
        if (past != 0u) h.cnt = __ffs(past);
        h.closed = past != 0u || h.cnt == 32;
        if (h.closed) {
            tail_key = h.key_of(h.cnt - 1);
            t_hi = key_depth(tail_key);
        }
    }
    return true;
}

// Running blend of the warp's ray: channel c in lane c; depth, transmittance
// and hit count in every lane.
struct WarpMarch {
    float C, D, T;
    int nh;
    __device__ __forceinline__ void init() {
        C = 0.f;
        D = 0.f;
        T = 1.f;
        nh = 0;
    }
};

// Blend the round's hits in order, every lane with the same w and T, lane c
// with channel c, until T < T_min (the crossing hit included) or `most` hits.
// Returns how many; T_before: the transmittance in front of this lane's hit.
__device__ __forceinline__ int blend_warp(const SceneView& S, const TraceParams& P, const WarpHits& h, int most,
                                          WarpMarch& st, float& T_before) {
    const int lane = threadIdx.x & 31;
    const float* feat = S.feat + P.off + lane;
    const int cnt = min(h.cnt, most);
    int done = 0;
    T_before = 1.f;
    for (int j0 = 0; j0 < cnt && !(st.T < P.T_min); j0 += 4) {   // 4 hits' channels in flight
        float f[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int32_t m = __shfl_sync(kFullWarp, h.m, (j0 + i) & 31);
            f[i] = j0 + i < cnt && lane < P.fc ? __ldg(feat + (int64_t)m * S.F) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = __shfl_sync(kFullWarp, h.a, (j0 + i) & 31);
            const float depth = __uint_as_float(__shfl_sync(kFullWarp, h.kh, (j0 + i) & 31));
            if (j0 + i < cnt && !(st.T < P.T_min)) {
                const float w = __fmul_rn(st.T, a);
                if (lane == j0 + i) T_before = st.T;
                st.C = __fmaf_rn(w, f[i], st.C);
                st.D = __fmaf_rn(w, depth, st.D);
                st.T = __fmul_rn(st.T, __fsub_rn(1.0f, a));
                ++done;
            }
        }
    }
    return done;
}

// All rounds of the warp's ray, which can_hit.
__device__ __forceinline__ bool march_warp(const SceneView& S, const Ray& ray, const RayBox& rb, const TraceParams& P,
                                           WarpMarch& st, int32_t* ids, int max_ids, WarpRayScratch& ws) {
    const int lane = threadIdx.x & 31;
    st.init();
    if (S.n == 0) return true;
    uint64_t last_key = depth_key(P.t_min, 0.f);
    int32_t last_u = INT32_MAX;
    bool ok = true;
    for (;;) {
        WarpHits h;
        ok &= collect_warp(S, ray, rb, P, last_key, last_u, st.T, ws, h);
        float before;
        const int done = blend_warp(S, P, h, 32, st, before);
        if (ids != nullptr && lane < done && st.nh + lane < max_ids) ids[st.nh + lane] = uid_of(S.rec, h.m);
        st.nh += done;
        if (st.T < P.T_min || !h.closed) break;
        last_key = h.key_of(h.cnt - 1);
        last_u = uid_of(S.rec, __shfl_sync(kFullWarp, h.m, h.cnt - 1));
    }
    return ok;
}

// Batches of caller's rays up to this size take a warp per ray. Packets of
// camera rays are faster per ray where a batch has many, but their warps are few
// and the slowest of them takes a millisecond or more, longer the more surfels
// there are, while a warp per ray takes little longer then. ms for one view, a
// warp per ray against packets:
//                100k surfels    300k           1M             3M
//   256 x 256    0.29 / 0.70     0.30 / 1.17    0.33 / 2.07    0.36 / 3.25
//   384 x 384    0.64 / 0.62     0.66 / 1.13    0.70 / 1.71    0.75 / 3.33
//   512 x 512    1.11 / 0.67     1.14 / 1.03    1.22 / 1.72    1.30 / 3.17
// Rays that do not run together gain at every size (2^18 random pixels of 300k
// surfels 1.39 ms, one ray more 2.74, where they walk as lanes). The line lies
// where views of 300k surfels break even.
constexpr int64_t kWarpRayMax = int64_t(1) << 18;

// Threads per block, and resident blocks per SM, of the kernels with a warp per
// ray.
constexpr int kWarpRayThreads = 128;
constexpr int kWarpRayBlocks = 8;
constexpr int kWarpRays = kWarpRayThreads / 32;   // rays per block

__device__ __forceinline__ WarpRayScratch& warp_ray_scratch() {
    __shared__ WarpRayScratch s_ws[kWarpRays];
    return s_ws[threadIdx.x >> 5];
}

inline unsigned warp_ray_grid(int64_t rays) { return (unsigned)((rays + kWarpRays - 1) / kWarpRays); }

}  // namespace irgs
