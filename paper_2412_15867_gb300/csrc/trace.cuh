// Traversal of the BVH with a shared-memory k-buffer and front-to-back
// compositing -- Trace(r_o, r_d) of IRGS Eq. 8 with the intersection of Eq. 6,
// the response of Eq. 7 and the blending of Eq. 2. Shared by the forward,
// backward and shading kernels, which must reproduce each other's hit order
// and arithmetic bit for bit; every operation whose rounding matters is
// therefore written with explicit round-to-nearest intrinsics.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace irgs {

struct TraceParams {
    float alpha_min, alpha_max, T_min, t_min, t_max;
    int32_t off, fc;
};

struct Ray {
    f3 o, d;           // origin and direction as given
    float inv_dd;      // 1 / |d|^2
    float graze;       // 1e-8 |d|
};

__device__ __forceinline__ Ray make_ray(f3 o, f3 d) {
    Ray r;
    r.o = o;
    r.d = d;
    float dd = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
    r.inv_dd = 1.0f / dd;
    r.graze = 1e-8f * sqrtf(dd);
    return r;
}

// Can the ray hit anything? With a component that is not finite every depth and
// response below is NaN, and every hit is refused. Such a ray must not keep its
// warp's others from walking together, nor walk itself: an axis that is NaN
// bounds nothing (30,000 such rays, a warp each, over 300,000 surfels: 134 ms).
__device__ __forceinline__ bool can_hit(f3 o, f3 d) {
    return fabsf(o.x) < INFINITY && fabsf(o.y) < INFINITY && fabsf(o.z) < INFINITY && fabsf(d.x) < INFINITY &&
           fabsf(d.y) < INFINITY && fabsf(d.z) < INFINITY;
}
__device__ __forceinline__ bool can_hit(const Ray& r) { return can_hit(r.o, r.d); }

// A ray's slab-test form.
struct RayBox {
    f3 inv;            // 1/d with zero components replaced
    f3 oinv;           // o * inv
    int nrx, nry, nrz; // row of a wide node holding each axis' entry plane (lo if inv >= 0, else hi)
};

__device__ __forceinline__ RayBox make_ray_box(const Ray& ray) {
    RayBox r;
    auto safe = [](float x) { return fabsf(x) < 1e-20f ? copysignf(1e-20f, x) : x; };
    r.inv = mk3(1.0f / safe(ray.d.x), 1.0f / safe(ray.d.y), 1.0f / safe(ray.d.z));
    r.oinv = mk3(ray.o.x * r.inv.x, ray.o.y * r.inv.y, ray.o.z * r.inv.z);
    r.nrx = r.inv.x >= 0.f ? 0 : 3;
    r.nry = r.inv.y >= 0.f ? 1 : 4;
    r.nrz = r.inv.z >= 0.f ? 2 : 5;
    return r;
}

// Geometry of an accepted hit that the backward pass needs.
struct HitGeom {
    f3 e;          // p - mu
    float u, v;    // Eq. 7 local coordinates
    float G;       // exp(-rho^2/2)
    float a_raw;   // o G before the clamp
    float den;     // n . d
};

// Ray/surfel test (Eq. 6-7) evaluated around a rebased origin
// o' = o + t_r d, t_r = (mu - o).d / |d|^2 (closest approach to mu), so the
// cancellation that plain FP32 suffers when |o - mu| >> scale disappears:
//   a   = mu - o exactly as a float pair (two_sum),
//   dl  = mu - o' = fma(-t_r, d, a_hi) + a_lo          (small, nearly exact)
//   tau = t_r + n.dl / n.d,  p - mu = (tau - t_r) d - dl.
// The depth is returned as the exact pair (kh, kl) = two_sum(t_r, tau - t_r).
// surfel_depth: that depth; false where the ray grazes the plane (|n.d| <
// 1e-8 |d|).
struct DepthParts {
    float dlx, dly, dlz, den, tp;
};
__device__ __forceinline__ bool surfel_depth(const float4& r0, const float4& r3, const Ray& ray, float& kh, float& kl,
                                             DepthParts* g = nullptr) {
    float ahx, alx, ahy, aly, ahz, alz;
    two_sum(r0.x, -ray.o.x, ahx, alx);
    two_sum(r0.y, -ray.o.y, ahy, aly);
    two_sum(r0.z, -ray.o.z, ahz, alz);
    const f3 d = ray.d;
    float tr = __fmul_rn(__fmaf_rn(ahx, d.x, __fmaf_rn(ahy, d.y, __fmul_rn(ahz, d.z))), ray.inv_dd);
    float dlx = __fadd_rn(__fmaf_rn(-tr, d.x, ahx), alx);
    float dly = __fadd_rn(__fmaf_rn(-tr, d.y, ahy), aly);
    float dlz = __fadd_rn(__fmaf_rn(-tr, d.z, ahz), alz);
    float den = __fmaf_rn(r3.x, d.x, __fmaf_rn(r3.y, d.y, __fmul_rn(r3.z, d.z)));
    if (!(fabsf(den) >= ray.graze)) return false;
    float num = __fmaf_rn(r3.x, dlx, __fmaf_rn(r3.y, dly, __fmul_rn(r3.z, dlz)));
    float tp = __fdiv_rn(num, den);
    two_sum(tr, tp, kh, kl);
    if (g != nullptr) *g = {dlx, dly, dlz, den, tp};
    return true;
}

// The whole test. A candidate whose rounded depth kh lies outside [kh_lo,
// kh_hi] is rejected before the support and opacity tests (callers pass
// bounds that only cut candidates their own key tests would reject).
template <bool GEOM>
__device__ __forceinline__ bool surfel_hit(const float4& r0, const float4& r1, const float4& r2, const float4& r3,
                                           const Ray& ray, float amin, float amax, float& kh, float& kl,
                                           float& alpha, HitGeom* g, float kh_lo = -INFINITY,
                                           float kh_hi = INFINITY) {
    DepthParts p;
    if (!surfel_depth(r0, r3, ray, kh, kl, &p)) return false;
    const f3 d = ray.d;
    if (kh < kh_lo || kh > kh_hi) return false;
    float ex = __fmaf_rn(p.tp, d.x, -p.dlx);
    float ey = __fmaf_rn(p.tp, d.y, -p.dly);
    float ez = __fmaf_rn(p.tp, d.z, -p.dlz);
    float u = __fmaf_rn(ex, r1.x, __fmaf_rn(ey, r1.y, __fmul_rn(ez, r1.z)));
    float v = __fmaf_rn(ex, r2.x, __fmaf_rn(ey, r2.y, __fmul_rn(ez, r2.z)));
    float rho2 = __fmaf_rn(u, u, __fmul_rn(v, v));
    if (!(rho2 <= r1.w)) return false;
    float G = __expf(__fmul_rn(-0.5f, rho2));
    float a_raw = __fmul_rn(r0.w, G);
    alpha = fminf(a_raw, amax);
    if (!(alpha >= amin)) return false;
    if (GEOM) {
        g->e = mk3(ex, ey, ez);
        g->u = u;
        g->v = v;
        g->G = G;
        g->a_raw = a_raw;
        g->den = p.den;
    }
    return true;
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// A wide node's child boxes as the ray meets them: for each axis the plane
// it enters through (lo where 1/d >= 0, else hi) and the one it leaves
// through, selected by which rows are loaded.
struct WideNodeRay {
    float4 nx, ny, nz, fx, fy, fz;
    int4 child;
};

__device__ __forceinline__ WideNodeRay load_wide_ray(const WideNode* w, int i, const RayBox& r) {
    const float4* p = reinterpret_cast<const float4*>(w + i);
    WideNodeRay n;
    n.nx = ldg4(p + r.nrx);
    n.ny = ldg4(p + r.nry);
    n.nz = ldg4(p + r.nrz);
    n.fx = ldg4(p + (r.nrx ^ 3));   // rows 0 <-> 3, 1 <-> 4, 2 <-> 5
    n.fy = ldg4(p + (r.nry ^ 5));
    n.fz = ldg4(p + (r.nrz ^ 7));
    n.child = ldg4i(reinterpret_cast<const int4*>(p + 6));
    return n;
}

// Slab intervals of the four children from the entry / exit planes
// (fma(v, inv, -oinv) is monotone in v for a fixed sign of inv, so the entry
// plane's distance is the smaller of the pair without a min/max).
__device__ __forceinline__ void slab4_ray(const WideNodeRay& w, const RayBox& r, float tn[4], float tf[4]) {
    const float nx[4] = {w.nx.x, w.nx.y, w.nx.z, w.nx.w}, fx[4] = {w.fx.x, w.fx.y, w.fx.z, w.fx.w};
    const float ny[4] = {w.ny.x, w.ny.y, w.ny.z, w.ny.w}, fy[4] = {w.fy.x, w.fy.y, w.fy.z, w.fy.w};
    const float nz[4] = {w.nz.x, w.nz.y, w.nz.z, w.nz.w}, fz[4] = {w.fz.x, w.fz.y, w.fz.z, w.fz.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        tn[k] = max3f(fmaf(nx[k], r.inv.x, -r.oinv.x), fmaf(ny[k], r.inv.y, -r.oinv.y),
                      fmaf(nz[k], r.inv.z, -r.oinv.z));
        tf[k] = min3f(fmaf(fx[k], r.inv.x, -r.oinv.x), fmaf(fy[k], r.inv.y, -r.oinv.y),
                      fmaf(fz[k], r.inv.z, -r.oinv.z));
    }
}

// Conservative slack on depths compared against box intervals.
__device__ __forceinline__ float tslack(float t) { return 1e-5f * (1.0f + fabsf(t)); }

__device__ __forceinline__ float key_depth(uint64_t k) { return __uint_as_float((uint32_t)(k >> 32)); }

// User index of the surfel in Morton slot m (carried in its record's r2.w).
__device__ __forceinline__ int32_t uid_of(const float4* rec, int32_t m) {
    return __float_as_int(__ldg(&rec[(int64_t)m * kRecF4 + 2].w));
}

// ---------------------------------------------------------------------------
// Threads per block of every tracing kernel (k-buffer slots and leaf queues
// are laid out per block thread).
constexpr int kTraceThreads = 128;

// Entries of the k-buffer. Results do not depend on it (the buffer holds the
// nearest hits after the last blended one, whatever its size), so the size a
// caller asks for selects no code. A ray that blends more walks once more:
// 640k points' shading takes 112.0 ms with 24 entries, 108.6 with 28, 105.8
// with 32, beyond which fewer blocks fit.
constexpr int kCap = 32;
constexpr int kPacketBlocks = 4;   // resident blocks per SM that the kernels are compiled for
constexpr int kRayBlocks = 5;

// Exact depth remainder kl and user index of surfel m, whose hit at the same
// rounded depth ties with another: out of line, since ties are rare.
static __device__ __noinline__ float2 tie_of(const float4* rec, int32_t m, f3 o, f3 d, float inv_dd) {
    Ray r;
    r.o = o;
    r.d = d;
    r.inv_dd = inv_dd;
    r.graze = 0.f;
    const float4* R = rec + (int64_t)m * kRecF4;
    const float4 r2 = ldg4(R + 2);
    float kh, kl;
    surfel_depth(ldg4(R), ldg4(R + 3), r, kh, kl);
    return make_float2(kl, r2.w);
}

// k-buffer of the nearest hits after the last blended one, ascending in
// (depth, user index), in shared memory as 8-byte entries: x the bits of the
// rounded depth kh, y the Morton index with the hit's optical depth in the
// top byte. Slot j of thread t lives at [j * kTraceThreads + t], so a warp
// touching one slot reads consecutive words. Two hits with the same rounded
// depth are ordered by the exact remainder and then the user index, both
// recomputed on that (rare) tie; alpha is recomputed when a hit is blended.
//
// The buffer is closed when it is full or when its hits alone bring the
// transmittance below T_min: the optical depths, floor(-16 log2(1 - alpha))
// each, add up to `need`, and entries behind the shortest such prefix are
// dropped. A closed buffer bounds the walk by its last depth. The sums round
// down, so a prefix is never cut short; if the blend does not end inside a
// closed buffer, another round continues behind its last entry.
template <int CAP>
struct KBuffer {
    uint2* e;
    int cnt;
    uint32_t sum, need, id_mask;
    uint32_t tail;   // depth bits of the last entry of a closed buffer

    // The kernel's one shared array of entries.
    __device__ __forceinline__ void bind() {
        __shared__ uint2 s_e[CAP * kTraceThreads];
        e = s_e + threadIdx.x;
        cnt = 0;
    }
    // An empty buffer for a ray of transmittance T (T >= T_min).
    __device__ __forceinline__ void open(int64_t n, float T, float T_min) {
        cnt = 0;
        sum = 0u;
        const bool packs = n <= (int64_t)1 << 24;   // 24-bit Morton indices leave a byte for the optical depth
        id_mask = packs ? 0xffffffu : 0xffffffffu;
        // optical depth that is surely past T_min; never reached when T_min = 0
        const float bits = 16.f * __log2f(__fdividef(T, T_min)) + 2.f;
        need = packs && T_min > 0.f && bits < 1e9f ? (uint32_t)fmaxf(bits, 1.f) : 0xffffffffu;
    }
    __device__ __forceinline__ bool closed() const { return cnt == CAP || sum >= need; }
    __device__ __forceinline__ int32_t m_at(int j) const { return (int32_t)(e[j * kTraceThreads].y & id_mask); }
    // does a hit at (kb = bits of kh, kl, user index u) come before entry v?
    __device__ __forceinline__ bool before(uint32_t kb, float kl, int32_t u, const uint2& v, const float4* rec,
                                           const Ray& ray) const {
        if (kb != v.x) return kb < v.x;
        const float2 t = tie_of(rec, (int32_t)(v.y & id_mask), ray.o, ray.d, ray.inv_dd);
        return kl < t.x || (kl == t.x && u < __float_as_int(t.y));
    }
    // Insert a hit unless the buffer is closed and it lies behind the last
    // entry. Returns whether it went in.
    __device__ __forceinline__ bool insert(float kh, float kl, int32_t m, int32_t u, float alpha, const float4* rec,
                                           const Ray& ray) {
        const uint32_t kb = __float_as_uint(kh + 0.0f);
        const bool was_closed = closed();
        if (was_closed &&
            !(kb < tail || (kb == tail && before(kb, kl, u, e[(cnt - 1) * kTraceThreads], rec, ray))))
            return false;
        int j = cnt - 1;
        if (cnt == CAP) {
            sum -= id_mask == 0xffffffu ? e[j * kTraceThreads].y >> 24 : 0u;
            --j;
        } else {
            ++cnt;
        }
        // entries behind the new one move up, eight at a time: their loads are in
        // flight together, and a warp waits out a shared-memory round trip per
        // step of its longest shift (7 entries on average). 800 x 800 view: 1.49 ms
        // by two, 1.36 by four, 1.33 by eight.
        bool found = false;
        while (!found && j >= 0) {
            uint2 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = j >= i ? e[(j - i) * kTraceThreads] : make_uint2(0u, 0u);
            int moved = 0;   // entries are in order: those behind the new one come first
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (j >= i && kb < v[i].x) {
                    e[(j - i + 1) * kTraceThreads] = v[i];
                    ++moved;
                }
            }
            j -= moved;
            if (moved == 8) continue;
            found = j < 0 || !before(kb, kl, u, e[j * kTraceThreads], rec, ray);
            if (!found) {   // a tie, and the entry comes after
                e[(j + 1) * kTraceThreads] = e[j * kTraceThreads];
                --j;
            }
        }
        uint32_t q = 0u;
        if (id_mask == 0xffffffu) q = (uint32_t)fminf(fmaxf(-16.f * __log2f(1.f - alpha), 0.f), 255.f);
        e[(j + 1) * kTraceThreads] = make_uint2(kb, (uint32_t)m | q << 24);
        sum += q;
        if (closed()) {
            uint2 t = e[(cnt - 1) * kTraceThreads];
            while (need != 0xffffffffu && cnt > 1 && sum - (t.y >> 24) >= need) {
                sum -= t.y >> 24;
                --cnt;
                t = e[(cnt - 1) * kTraceThreads];
            }
            tail = t.x;
        }
        return true;
    }
};

// Per-ray traversal counters of the diagnostic build (STATS = true).
struct TraceStats {
    int rounds, nodes, leaves, inserts;
};

// Shared working memory of one warp. The packet walk keeps its stack, its
// pending leaves and the records of a batch of 32 leaves; the per-ray walk
// its leaf queues (in the records' place).
constexpr int kPacketStack = 184;
constexpr int kLeafQueue = 12;   // pending leaves per ray
struct PacketScratch {
    float4 rec[32 * kRecF4];
    uint2 stack[kPacketStack];   // (wide node, entry depth bits)
    uint32_t leaf[64];
    float mid[8];                // origin and direction of the ray the leaves are ordered for
};
constexpr int kQueueF4 = kLeafQueue * 32 / 4;
static_assert(kQueueF4 <= 32 * kRecF4, "the leaf queues take the records' place");

static_assert(sizeof(PacketScratch) % sizeof(float4) == 0, "per-warp slots stay aligned");
// float4s of working memory that one warp's walk takes.
template <bool PACKET>
__host__ __device__ constexpr int scratch_f4() { return PACKET ? (int)(sizeof(PacketScratch) / sizeof(float4)) : kQueueF4; }

// Ray number of slot t when warps are made of 4 x 8 pixel tiles of an image
// of *width columns (rays row by row; nullptr or 0: the rays' own order). A
// packet of a tile meets a third of the leaves that one of a row strip
// does. A permutation of [0, R): the last rows that do not fill a band of
// eight keep their order.
__device__ __forceinline__ int64_t tiled_ray(int64_t t, int64_t R, const int32_t* __restrict__ width) {
    const uint32_t W = width != nullptr ? (uint32_t)__ldg(width) : 0u;
    if (W == 0u) return t;
    const int64_t band = t / (8 * (int64_t)W) * (8 * (int64_t)W);
    if (band + 8 * (int64_t)W > R) return t;
    const uint32_t u = (uint32_t)(t - band), full = W / 4 * 32, c = W % 4;   // whole tiles, then the columns left over
    const uint32_t v = u - full;
    const uint32_t col = u < full ? u / 32 * 4 + u % 4 : W / 4 * 4 + v % (c != 0u ? c : 1u);
    const uint32_t row = u < full ? u % 32 / 4 : v / (c != 0u ? c : 1u);
    return band + (int64_t)row * W + col;
}

// This warp's part of a block's working memory, F4 float4s per warp.
template <int F4>
__device__ __forceinline__ float4* warp_memory() {
    __shared__ float4 s_warp[kTraceThreads / 32 * F4];
    return s_warp + (threadIdx.x >> 5) * F4;
}
template <bool PACKET>
__device__ __forceinline__ float4* warp_scratch() { return warp_memory<scratch_f4<PACKET>()>(); }

// One ray against surfel records: into the buffer if its hit lies strictly
// after (last_key, last_u) and before t_max and the buffer's last entry.
template <class KB, bool STATS = false>
__device__ __forceinline__ bool leaf_insert(const SceneView& S, const Ray& ray, const TraceParams& P, int32_t m,
                                            const float4& r0, const float4& r1, const float4& r2, const float4& r3,
                                            uint64_t last_key, int32_t last_u, KB& kb, float& t_hi, TraceStats* ts) {
    if (STATS) ts->leaves++;
    float kh, kl, a;
    // a rounded depth below the last blended key's, or above the closed
    // buffer's last entry (t_hi, else t_max), cannot pass the key tests
    // below; kh >= key_depth(last_key) >= t_min >= 0 also makes the key
    // order that of the depths, and the first round's last_key = (t_min, 0)
    // with last_u = INT32_MAX admits exactly the depths beyond t_min
    if (!surfel_hit<false>(r0, r1, r2, r3, ray, P.alpha_min, P.alpha_max, kh, kl, a, nullptr, key_depth(last_key),
                           t_hi))
        return false;
    const uint64_t key = depth_key(kh, kl);
    const int32_t u = __float_as_int(r2.w);
    const bool after = key > last_key || (key == last_key && u > last_u);
    const bool inside = kh < P.t_max || (kh == P.t_max && kl < 0.f);
    if (!(after && inside && kb.insert(kh, kl, m, u, a, S.rec, ray))) return false;
    if (STATS) ts->inserts++;
    if (kb.closed()) t_hi = __uint_as_float(kb.tail);
    return true;
}

constexpr unsigned kFullWarp = 0xffffffffu;

// Upper bound on node fetches of one round in a valid tree.
__device__ __forceinline__ int visit_cap(const SceneView& S) {
    return S.n + 64 < (int64_t)INT32_MAX ? (int)(S.n + 64) : INT32_MAX;
}

// A ray's walk on its own: the node to visit next (-1: none), pending leaves in
// its queue, and a stack whose most recent entry is kept in a register. An
// entry is one word: the entry depth's leading bits (rounded down) above the
// node's number. The stacks live in local memory and share the L1 with nodes
// and records: at two words they took as much of it as those.
struct RayWalk {
    int ni, qn, sp, visits;
    uint32_t top;
    bool has_top, ok;
    float lo_c, t_hi;
    __device__ __forceinline__ void start(const SceneView& S, const TraceParams& P, uint64_t last_key) {
        ni = 0;
        qn = sp = 0;
        has_top = false;
        top = 0u;
        visits = visit_cap(S);
        const float t_lo = key_depth(last_key);
        lo_c = t_lo - tslack(t_lo);
        t_hi = P.t_max;
    }
    __device__ __forceinline__ bool can_walk() const { return ni >= 0 && qn <= kLeafQueue - 4; }
};

// One pending leaf of the ray.
template <class KB, bool STATS>
__device__ __forceinline__ void walk_leaf(const SceneView& S, const Ray& ray, const TraceParams& P, uint64_t last_key,
                                          int32_t last_u, KB& kb, RayWalk& w, const uint32_t* queue, TraceStats* ts) {
    --w.qn;
    const int32_t m = (int32_t)queue[32 * w.qn];
    const float4* R = S.rec + (int64_t)m * kRecF4;
    const float4 r0 = ldg4(R), r1 = ldg4(R + 1), r2 = ldg4(R + 2), r3 = ldg4(R + 3);
    leaf_insert<KB, STATS>(S, ray, P, m, r0, r1, r2, r3, last_key, last_u, kb, w.t_hi, ts);
}

// One node: its leaves that the ray's box test keeps go to the queue, the
// nearest inner one is next, the others go onto the stack, farthest first.
template <bool STATS>
__device__ __forceinline__ void walk_node(const SceneView& S, const RayBox& rb, RayWalk& w, uint32_t* stack,
                                          uint32_t* queue, TraceStats* ts) {
    const uint32_t id_mask = (1u << S.wide_bits) - 1u;
    auto entry_depth = [&](uint32_t e) { return __uint_as_float((e & ~id_mask) >> 1); };
    if (--w.visits < 0) {   // each wide node is fetched at most once per round in a valid tree
        w.ok = false;
        w.ni = -1;
        return;
    }
    const WideNodeRay nd = load_wide_ray(S.wide, w.ni, rb);
    if (STATS) ts->nodes++;
    float tn[4], tf[4];
    slab4_ray(nd, rb, tn, tf);
    const int c[4] = {nd.child.x, nd.child.y, nd.child.z, nd.child.w};
    const float hi_c = w.t_hi + tslack(w.t_hi);
    // children to enter, nearest first: entry depth (its last two bits
    // give way to the child's number, which only rounds it down)
    uint32_t key[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool h = tn[k] <= tf[k] && tf[k] >= w.lo_c && tn[k] <= hi_c;   // empty slots: empty box
        if (h && c[k] < 0) queue[32 * w.qn++] = (uint32_t)~c[k];
        key[k] = h && c[k] >= 0 ? (__float_as_uint(fmaxf(tn[k], 0.f)) & ~3u) | (uint32_t)k : 0xffffffffu;
    }
    auto order = [&](int a, int b) {
        const uint32_t lo = min(key[a], key[b]), hi = max(key[a], key[b]);
        key[a] = lo;
        key[b] = hi;
    };
    order(0, 1);
    order(2, 3);
    order(0, 2);
    order(1, 3);
    order(1, 2);
    auto child_of = [&](uint32_t k) {
        const uint32_t s = k & 3u;
        const int lo = (s & 1u) ? c[1] : c[0], hi = (s & 1u) ? c[3] : c[2];
        return (s & 2u) ? hi : lo;
    };
    auto entry = [&](uint32_t k) { return ((k << 1) & ~id_mask) | (uint32_t)child_of(k); };
    if (key[0] == 0xffffffffu) {
        w.ni = -1;
        if (w.has_top) {
            w.has_top = false;
            if (entry_depth(w.top) <= hi_c) w.ni = (int)(w.top & id_mask);
        }
        while (w.ni < 0 && w.sp > 0) {
            const uint32_t e = stack[--w.sp];
            if (entry_depth(e) <= hi_c) w.ni = (int)(e & id_mask);
        }
        return;
    }
    w.ni = child_of(key[0]);
    if (key[1] != 0xffffffffu) {
        if (w.sp + 3 > kStackSize) {
            w.ok = false;
        } else {
            if (w.has_top) stack[w.sp++] = w.top;
            if (key[3] != 0xffffffffu) stack[w.sp++] = entry(key[3]);
            if (key[2] != 0xffffffffu) stack[w.sp++] = entry(key[2]);
        }
        w.top = entry(key[1]);
        w.has_top = true;
    }
}

// One round, one traversal stack per ray: gather the nearest hits strictly
// after (last_key, last_u). All 32 lanes call this together (lanes without a
// ray pass active = false). The lanes of a warp walk different nodes, and on
// average less than one leaf child per node has to be tested, so testing
// each node's leaves on the spot leaves most lanes idle; here a lane queues
// its leaves and the warp takes the step, node visits or leaf tests, that
// more of its lanes are ready for. Returns false if a stack overflowed.
template <class KB, bool STATS = false>
__device__ __forceinline__ bool collect_round(const SceneView& S, const Ray& ray, const TraceParams& P,
                                              uint64_t last_key, int32_t last_u, KB& kb, bool active,
                                              float4* scratch, TraceStats* ts = nullptr) {
    uint32_t* queue = reinterpret_cast<uint32_t*>(scratch) + (threadIdx.x & 31);   // entry i at queue[32 i]
    const RayBox rb = make_ray_box(ray);
    uint32_t stack[kStackSize];
    RayWalk w;
    w.ok = true;
    w.start(S, P, last_key);
    if (!active || !can_hit(ray)) w.ni = -1;
    for (;;) {
        const unsigned walk = __ballot_sync(kFullWarp, w.can_walk());
        const unsigned have = __ballot_sync(kFullWarp, w.qn > 0);
        if ((walk | have) == 0u) break;
        if (__popc(walk) <= __popc(have)) {
            if (w.qn > 0) walk_leaf<KB, STATS>(S, ray, P, last_key, last_u, kb, w, queue, ts);
        } else {
            if (w.can_walk()) walk_node<STATS>(S, rb, w, stack, queue, ts);
        }
    }
    __syncwarp();   // the queues' memory may now take another use
    return w.ok;
}

// Bounds of a warp's rays for the packet walk. Axis k is the one the rays
// mostly run along; z = sign * (x_k - o_k) grows along every ray, and at z a
// ray is at o_a + s_a z, o_b + s_b z with slopes s = d / |d_k| of any sign.
struct Packet {
    int k, a, b;                        // axes
    float sign;
    float zo_min, zo_max;               // sign * o_k
    float oa_min, oa_max, ob_min, ob_max;
    float sa_min, sa_max, sb_min, sb_max;
    float dk_min, dk_max;               // |d_k|
    float o_abs;                        // largest |o| component, for the rounding margin
    float s_abs;
};

__device__ __forceinline__ float axis_of(f3 v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }

__device__ __forceinline__ float warp_min(float v, bool on) {
    const uint32_t u = on ? ordered_bits(v + 0.0f) : 0xffffffffu;
    const uint32_t m = __reduce_min_sync(kFullWarp, u);
    return __uint_as_float((m & 0x80000000u) ? (m & 0x7fffffffu) : ~m);
}
__device__ __forceinline__ float warp_max(float v, bool on) { return -warp_min(-v, on); }

// The packet of the active lanes' rays; false if they do not run together:
// a common dominant axis and direction along it, and slopes that spread by
// less than kPacketSpread (a strip of a coarse image; a strip is long and
// thin, so this alone says little, and collect_packet gives up on packets
// whose leaves miss most of their rays).
constexpr float kPacketSpread = 0.7f;
__device__ __forceinline__ bool make_packet(const Ray& ray, bool active, Packet& p) {
    const unsigned on = __ballot_sync(kFullWarp, active);
    if (on == 0u) return false;
    const int src = __ffs(on) - 1;
    const float ax = fabsf(__shfl_sync(kFullWarp, ray.d.x, src)), ay = fabsf(__shfl_sync(kFullWarp, ray.d.y, src)),
                az = fabsf(__shfl_sync(kFullWarp, ray.d.z, src));
    p.k = ax >= ay && ax >= az ? 0 : (ay >= az ? 1 : 2);
    p.a = p.k == 2 ? 0 : p.k + 1;
    p.b = p.a == 2 ? 0 : p.a + 1;
    p.sign = __shfl_sync(kFullWarp, axis_of(ray.d, p.k), src) >= 0.f ? 1.f : -1.f;
    const float dk = p.sign * axis_of(ray.d, p.k);
    const float inv = 1.0f / dk;
    const float sa = axis_of(ray.d, p.a) * inv, sb = axis_of(ray.d, p.b) * inv;
    const bool fits = dk > 1e-30f && dk < 1e30f && fabsf(sa) <= 2.5f && fabsf(sb) <= 2.5f &&
                      fabsf(ray.o.x) < 1e15f && fabsf(ray.o.y) < 1e15f && fabsf(ray.o.z) < 1e15f;
    if (!__all_sync(kFullWarp, fits || !active)) return false;
    p.sa_min = warp_min(sa, active);
    p.sa_max = warp_max(sa, active);
    p.sb_min = warp_min(sb, active);
    p.sb_max = warp_max(sb, active);
    if (!(p.sa_max - p.sa_min <= kPacketSpread && p.sb_max - p.sb_min <= kPacketSpread)) return false;
    const float zo = p.sign * axis_of(ray.o, p.k), oa = axis_of(ray.o, p.a), ob = axis_of(ray.o, p.b);
    p.zo_min = warp_min(zo, active);
    p.zo_max = warp_max(zo, active);
    p.oa_min = warp_min(oa, active);
    p.oa_max = warp_max(oa, active);
    p.ob_min = warp_min(ob, active);
    p.ob_max = warp_max(ob, active);
    p.dk_min = warp_min(dk, active);
    p.dk_max = warp_max(dk, active);
    p.o_abs = fmaxf(fmaxf(fmaxf(fabsf(p.zo_min), fabsf(p.zo_max)), fmaxf(fabsf(p.oa_min), fabsf(p.oa_max))),
                    fmaxf(fabsf(p.ob_min), fabsf(p.ob_max)));
    p.s_abs = 1.f + fmaxf(fmaxf(fabsf(p.sa_min), fabsf(p.sa_max)), fmaxf(fabsf(p.sb_min), fabsf(p.sb_max)));
    return true;
}

// Can a ray of the packet meet child `c` of wide node `id` between depths
// lo_t and hi_t? t_in: a lower bound on the depths inside the box. Margins of
// 2e-6 of the coordinates involved cover the rounding of every step, and
// comparisons with NaN keep the child.
__device__ __forceinline__ bool packet_child(const float4* boxes, int id, int c, const Packet& p, float lo_t,
                                             float hi_t, int& child, float& t_in) {
    const float4 lo = ldg4(boxes + (int64_t)id * 8 + 2 * c), hi = ldg4(boxes + (int64_t)id * 8 + 2 * c + 1);
    child = __float_as_int(lo.w);
    const f3 lo3 = mk3(lo.x, lo.y, lo.z), hi3 = mk3(hi.x, hi.y, hi.z);
    const float lok = axis_of(lo3, p.k), hik = axis_of(hi3, p.k);
    const float loa = axis_of(lo3, p.a), hia = axis_of(hi3, p.a);
    const float lob = axis_of(lo3, p.b), hib = axis_of(hi3, p.b);
    if (child == kNoChild) return false;
    const float ez = 2e-6f * (fmaxf(fabsf(lok), fabsf(hik)) + p.o_abs);
    const float zn = p.sign > 0.f ? lok : -hik, zf = p.sign > 0.f ? hik : -lok;
    const float z1 = fmaxf(fmaxf(zn - p.zo_max - ez, 0.f), lo_t * p.dk_min);
    const float z2 = fminf(zf - p.zo_min + ez, hi_t * p.dk_max);
    t_in = z1 / p.dk_max;
    if (z2 < z1) return false;
    const float e = 2e-6f * (p.o_abs + p.s_abs * z2);
    const float a_lo = p.oa_min + fminf(p.sa_min * z1, p.sa_min * z2), a_hi = p.oa_max + fmaxf(p.sa_max * z1, p.sa_max * z2);
    const float b_lo = p.ob_min + fminf(p.sb_min * z1, p.sb_min * z2), b_hi = p.ob_max + fmaxf(p.sb_max * z1, p.sb_max * z2);
    return !(a_hi + e < loa || a_lo - e > hia || b_hi + e < lob || b_lo - e > hib);
}

// Can a ray of the packet meet the support disk of a surfel? The disk against
// the packet's four side planes, x_j - s x_k sign >= c (or <= c): the largest
// value of such a form over the disk is its value at the centre plus
// rho_c |(U.N, V.N)| with U = s_u t_u, V = s_v t_v. The box of a tilted disk is
// much larger than the disk, so this drops half of the leaves whose boxes
// the packet meets; the margins are far above the rounding of the test.
__device__ __forceinline__ bool packet_disk(const Packet& p, const float4& r0, const float4& r1, const float4& r2) {
    if (!(r1.w >= 0.f)) return false;
    const f3 mu = mk3(r0.x, r0.y, r0.z), tu = mk3(r1.x, r1.y, r1.z), tv = mk3(r2.x, r2.y, r2.z);
    const float iu = __fdividef(1.f, dot3(tu, tu)), iv = __fdividef(1.f, dot3(tv, tv));   // s_u^2, s_v^2
    const float uk = p.sign * axis_of(tu, p.k) * iu, vk = p.sign * axis_of(tv, p.k) * iv;
    const float mk = p.sign * axis_of(mu, p.k);
    const float rc2 = r1.w * 1.001f;
    const float eps = 4e-6f * p.s_abs * (p.o_abs + fabsf(mu.x) + fabsf(mu.y) + fabsf(mu.z));
    // outside the plane with normal e_j - s e_k by more than the disk's extent
    auto beyond = [&](float gap, float uj, float vj, float s) {
        const float a = uj - s * uk, b = vj - s * vk;
        return gap > eps && (gap - eps) * (gap - eps) > rc2 * (a * a + b * b);
    };
    const float ma = axis_of(mu, p.a), ua = axis_of(tu, p.a) * iu, va = axis_of(tv, p.a) * iv;
    const float mb = axis_of(mu, p.b), ub = axis_of(tu, p.b) * iu, vb = axis_of(tv, p.b) * iv;
    const float a_lo = p.oa_min - fmaxf(p.sa_min * p.zo_min, p.sa_min * p.zo_max);
    const float a_hi = p.oa_max - fminf(p.sa_max * p.zo_min, p.sa_max * p.zo_max);
    const float b_lo = p.ob_min - fmaxf(p.sb_min * p.zo_min, p.sb_min * p.zo_max);
    const float b_hi = p.ob_max - fminf(p.sb_max * p.zo_min, p.sb_max * p.zo_max);
    return !(beyond(a_lo - (ma - p.sa_min * mk), ua, va, p.sa_min) || beyond((ma - p.sa_max * mk) - a_hi, ua, va, p.sa_max) ||
             beyond(b_lo - (mb - p.sb_min * mk), ub, vb, p.sb_min) || beyond((mb - p.sb_max * mk) - b_hi, ub, vb, p.sb_max));
}

// One step of a bitonic merge over the lanes, ascending.
__device__ __forceinline__ void bitonic_step(uint32_t& key, int32_t& m, int step) {
    const uint32_t ko = __shfl_xor_sync(kFullWarp, key, step);
    const int32_t mo = __shfl_xor_sync(kFullWarp, m, step);
    if ((threadIdx.x & step) == 0 ? ko < key : ko > key) {
        key = ko;
        m = mo;
    }
}

// One round for a packet of rays (32 lanes together): the hierarchy is walked
// once for the warp, 8 nodes a step with one child box per lane against the
// packet's bounds. Of the leaves that remain the records are fetched 32 at a
// time, one per lane (64 B each, in flight together); those whose disks miss
// the packet are dropped, the others put in the order in which the middle ray
// meets their planes. The nearer 32 of these and of those that waited are then
// staged in shared memory, where every ray tests every one; the rest waits for
// the next batch, so that hits come nearly in order (shifts in the k-buffer are
// most of the cost: 1.39 ms for an 800 x 800 view without the waiting ones,
// 1.37 with). Returns 0, or 1 if the hierarchy is broken, or 2 if
// the packet gave up (nothing is kept then; the caller walks per ray).
template <class KB, bool STATS = false>
__device__ __forceinline__ int collect_packet(const SceneView& S, const Ray& ray, const TraceParams& P,
                                              uint64_t last_key, int32_t last_u, KB& kb, bool active,
                                              PacketScratch& ws, TraceStats* ts = nullptr) {
    Packet pk;
    if (!make_packet(ray, active, pk)) return 2;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    {
        const unsigned on = __ballot_sync(kFullWarp, active);
        const int mid = (on >> 18) & 1u ? 18 : __ffs(on) - 1;   // lane 18: inside a 4 x 8 or 8 x 4 tile
        if (lane == mid) {
            ws.mid[0] = ray.o.x; ws.mid[1] = ray.o.y; ws.mid[2] = ray.o.z;
            ws.mid[3] = ray.d.x; ws.mid[4] = ray.d.y; ws.mid[5] = ray.d.z;
        }
        if (lane == 0) ws.stack[0] = make_uint2(0u, 0u);
    }
    __syncwarp();
    const float t_lo = key_depth(last_key);
    const float lo_t = fmaxf(warp_min(t_lo - tslack(t_lo), active), 0.f);
    float t_hi = P.t_max;
    float hi_t = P.t_max + tslack(P.t_max);
    int sp = 1, nleaf = 0, status = 0, batches = 0, hits = 0;
    int visits = visit_cap(S);
    uint32_t wait_key = 0xffffffffu;   // leaves that wait for nearer ones, in order, one per lane
    int32_t wait_m = 0;
    int waiting = 0;
    while (sp > 0 || nleaf > 0 || waiting > 0) {
        if (nleaf < 32 && sp > 0) {
            // near the stack's end only its top is taken, as a plain depth-first walk would
            const int take = min(sp, sp <= kPacketStack - 96 ? 8 : 1);
            visits -= take;
            const int g = lane >> 2;
            uint2 ent = make_uint2(0u, 0x7f800000u);
            bool in = g < take;
            if (in) ent = ws.stack[sp - 1 - g];
            in = in && __uint_as_float(ent.y) <= hi_t;
            sp -= take;
            int child = kNoChild;
            float t_in = 0.f;
            if (in) in = packet_child(S.child_box, (int)ent.x, lane & 3, pk, lo_t, hi_t, child, t_in);
            if (STATS && active) ts->nodes += take;
            const unsigned leaves = __ballot_sync(kFullWarp, in && child < 0);
            if (in && child < 0) ws.leaf[nleaf + __popc(leaves & lt)] = (uint32_t)~child;
            nleaf += __popc(leaves);
            const bool inner = in && child >= 0;
            const unsigned push = __ballot_sync(kFullWarp, inner);
            // farther siblings lie deeper, and so do the children of nodes farther down the stack
            const float td = inner ? t_in : -1.f;
            int deeper = __popc((push >> (4 * g)) >> 4);
#pragma unroll
            for (int x = 1; x < 4; ++x) {
                const float to = __shfl_xor_sync(kFullWarp, td, x);
                deeper += to > td || (to == td && (lane ^ x) > lane) ? 1 : 0;
            }
            if (sp + __popc(push) > kPacketStack || visits < 0) {
                status = visits < 0 ? 1 : 2;   // no room: the rays' own stacks hold less
                break;
            }
            __syncwarp();   // the popped entries have been read
            if (inner) ws.stack[sp + deeper] = make_uint2((uint32_t)child, __float_as_uint(t_in));
            sp += __popc(push);
            __syncwarp();
            continue;
        }
        const int cnt = min(nleaf, 32);
        uint32_t key = 0xffffffe0u | (uint32_t)lane;
        int32_t m = 0;
        bool keep = false;
        if (lane < cnt) {
            m = (int32_t)ws.leaf[lane];
            const float4* R = S.rec + (int64_t)m * kRecF4;
            const float4 r0 = ldg4(R), r1 = ldg4(R + 1), r2 = ldg4(R + 2), r3 = ldg4(R + 3);
            const f3 n3 = mk3(r3.x, r3.y, r3.z), w = mk3(r0.x - ws.mid[0], r0.y - ws.mid[1], r0.z - ws.mid[2]);
            const float tau = __fdividef(dot3(n3, w), dot3(n3, mk3(ws.mid[3], ws.mid[4], ws.mid[5])));
            keep = packet_disk(pk, r0, r1, r2);
            // order only: any value below the dropped lanes' will do
            if (keep) key = (tau > 0.f && tau < 1e30f ? __float_as_uint(tau) & ~31u : 0u) | (uint32_t)lane;
        }
        // the leaves behind the batch move to the front
        const uint32_t rest = 32 + lane < nleaf ? ws.leaf[32 + lane] : 0u;
        __syncwarp();
        if (32 + lane < nleaf) ws.leaf[lane] = rest;
        nleaf -= cnt;
        const int fresh = __popc(__ballot_sync(kFullWarp, keep));
        if (fresh > 0) {
            // bitonic sort of the lanes' keys
#pragma unroll
            for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
                for (int step = size >> 1; step > 0; step >>= 1) {
                    const uint32_t other = __shfl_xor_sync(kFullWarp, key, step);
                    const bool up = ((lane & size) == 0) == ((lane & step) == 0);
                    key = up ? min(key, other) : max(key, other);
                }
            m = __shfl_sync(kFullWarp, m, key & 31u);
            // the nearer half of these and the waiting ones, and the farther half, each in order
            const uint32_t ko = __shfl_sync(kFullWarp, key, 31 - lane);
            const int32_t mo = __shfl_sync(kFullWarp, m, 31 - lane);
            const bool swap = ko < wait_key;
            key = swap ? ko : wait_key;
            m = swap ? mo : wait_m;
            if (!swap) {
                wait_key = ko;
                wait_m = mo;
            }
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                bitonic_step(key, m, step);
                bitonic_step(wait_key, wait_m, step);
            }
        } else {
            key = wait_key;
            m = wait_m;
            wait_key = 0xffffffffu;
        }
        const int all = waiting + fresh, now = min(all, 32);
        if (all <= 32 && (sp > 0 || nleaf > 0)) {
            wait_key = key;
            wait_m = m;
            waiting = all;
            __syncwarp();
            continue;
        }
        waiting = all - now;
        if (lane < now) {
            const float4* R = S.rec + (int64_t)m * kRecF4;
            float4 r3 = ldg4(R + 3);
            r3.w = __int_as_float(m);
            ws.rec[lane * 4] = ldg4(R);
            ws.rec[lane * 4 + 1] = ldg4(R + 1);
            ws.rec[lane * 4 + 2] = ldg4(R + 2);
            ws.rec[lane * 4 + 3] = r3;
        }
        __syncwarp();
        for (int i = 0; i < now; ++i) {
            const float4* R = ws.rec + 4 * i;
            if (active) {
                const float4 r3 = R[3];
                hits += leaf_insert<KB, STATS>(S, ray, P, __float_as_int(r3.w), R[0], R[1], R[2], r3, last_key, last_u,
                                               kb, t_hi, ts);
            }
        }
        const float hi = __uint_as_float(__reduce_max_sync(kFullWarp, active ? __float_as_uint(t_hi) : 0u));
        hi_t = hi + tslack(hi);
        // a packet whose leaves miss nearly all of its rays is no packet
        if (++batches % 16 == 0 && __reduce_add_sync(kFullWarp, hits) < 10 * batches) {
            status = 2;
            break;
        }
        __syncwarp();
    }
    __syncwarp();
    return status;
}

// One round by the walk that suits the warp's rays: the packet walk where
// they run together (PACKET), else one stack per ray.
template <bool PACKET, class KB, bool STATS = false>
__device__ __forceinline__ bool collect(const SceneView& S, const Ray& ray, const TraceParams& P, uint64_t last_key,
                                        int32_t last_u, float T, KB& kb, bool active, bool& packet, float4* scratch,
                                        TraceStats* ts = nullptr) {
    kb.open(S.n, T, P.T_min);
    if (PACKET && packet) {
        const int status = collect_packet<KB, STATS>(S, ray, P, last_key, last_u, kb, active && can_hit(ray),
                                                     *reinterpret_cast<PacketScratch*>(scratch), ts);
        if (status != 2) return status == 0;
        packet = false;   // the later rounds of the same rays walk per ray at once
        kb.open(S.n, T, P.T_min);
    }
    return collect_round<KB, STATS>(S, ray, P, last_key, last_u, kb, active, scratch, ts);
}

// Full forward march of one ray: rounds of collect + blend until the
// transmittance drops below T_min or no further hit exists.
template <int FB>
struct MarchState {
    float C[FB];
    float D, T;
    int nh;
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int c = 0; c < FB; ++c) C[c] = 0.f;
        D = 0.f;
        T = 1.f;
        nh = 0;
    }
};

// The traced channels f[0..fc) of one surfel, zero beyond fc; as 8-byte
// pairs when f is 8-byte aligned for every surfel (even row length and
// offset).
template <int FB>
__device__ __forceinline__ void load_channels(const float* __restrict__ f, int fc, bool pairs, float (&fv)[FB]) {
    if (pairs) {
#pragma unroll
        for (int c = 0; c < FB; c += 2) {
            const float2 t = c + 1 < fc ? __ldg(reinterpret_cast<const float2*>(f + c))
                                        : make_float2(c < fc ? __ldg(f + c) : 0.f, 0.f);
            fv[c] = t.x;
            if (c + 1 < FB) fv[c + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int c = 0; c < FB; ++c) fv[c] = c < fc ? __ldg(f + c) : 0.f;
    }
}

// Blend the round's buffered hits in order (Eq. 2, Eq. 8) until the
// transmittance drops below T_min (the crossing hit included). Each hit is
// recomputed from its record, with the same arithmetic. Returns true when
// the ray is done: terminated, or no hit was left outside the buffer; else
// (last_key, last_u) move to the buffer's last entry for the next round.
template <int FB, class KB>
__device__ __forceinline__ bool blend_round(const SceneView& S, const Ray& ray, const TraceParams& P, const KB& kb,
                                            MarchState<FB>& st, int32_t* ids, int max_ids, uint64_t& last_key,
                                            int32_t& last_u) {
    bool done = false;
    float kh = 0.f, kl = 0.f;
    int32_t u = 0;
    for (int j = 0; j < kb.cnt && !done; ++j) {
        const int32_t m = kb.m_at(j);
        const float4* R = S.rec + (int64_t)m * kRecF4;
        const float4 r0 = ldg4(R), r1 = ldg4(R + 1), r2 = ldg4(R + 2), r3 = ldg4(R + 3);
        float fv[FB];
        load_channels<FB>(S.feat + (int64_t)m * S.F + P.off, P.fc, ((S.F | P.off) & 1) == 0, fv);
        float a;
        surfel_hit<false>(r0, r1, r2, r3, ray, P.alpha_min, P.alpha_max, kh, kl, a, nullptr);
        u = __float_as_int(r2.w);
        const float w = __fmul_rn(st.T, a);
#pragma unroll
        for (int c = 0; c < FB; ++c)
            if (c < P.fc) st.C[c] = __fmaf_rn(w, fv[c], st.C[c]);
        st.D = __fmaf_rn(w, kh + 0.0f, st.D);
        st.T = __fmul_rn(st.T, __fsub_rn(1.0f, a));
        if (ids != nullptr && st.nh < max_ids) ids[st.nh] = u;
        st.nh++;
        if (st.T < P.T_min) done = true;
    }
    if (!done) {
        if (!kb.closed()) {
            done = true;
        } else {
            last_key = depth_key(kh, kl);
            last_u = u;
        }
    }
    return done;
}

// The rounds of one ray until it is done. All 32 lanes of the warp call this
// together (lanes without a ray pass live = false).
template <int FB, bool PACKET, int CAP = kCap, bool STATS = false>
__device__ __forceinline__ bool march_forward(const SceneView& S, const Ray& ray, const TraceParams& P,
                                              MarchState<FB>& st, int32_t* ids, int max_ids, bool live,
                                              float4* scratch, TraceStats* ts = nullptr) {
    st.init();
    bool ok = true;
    if (S.n == 0) return ok;
    uint64_t last_key = depth_key(P.t_min, 0.f);
    int32_t last_u = INT32_MAX;
    KBuffer<CAP> kb;
    kb.bind();
    bool done = !live, packet = true;
    while (__any_sync(kFullWarp, !done)) {
        if (STATS && !done) ts->rounds++;
        ok &= collect<PACKET, KBuffer<CAP>, STATS>(S, ray, P, last_key, last_u, st.T, kb, !done, packet,
                                                         scratch, ts);
        if (done) continue;
        done = blend_round<FB>(S, ray, P, kb, st, ids, max_ids, last_key, last_u);
    }
    return ok;
}

// A long batch of rays that walk on their own, in the batch's order: each warp
// takes kPool of them at a time and keeps its lanes filled. A lane whose walk
// has ended waits until kFinishLanes lanes have (or nothing else is left to
// do); these blend together, and each then starts its ray's next round or
// takes the pool's next ray. (With one ray per lane a warp ran its longest
// ray's walk with few lanes left, and rays that needed more rounds did so in a
// launch of their own, mostly alone: 15 of 32 lanes per node step, and a third
// of the time for a sixth of the rays.) Per ray the rounds and their
// arithmetic are march_forward's, so the results are the same. The batch holds at most 2^31 - kPool rays.
//
// Job: bool load(j, o, d): ray j, or false if there is none to trace (the job
// has dealt with it); int32_t* ids(j), max_ids: where to save its hit ids;
// void finish(j, st): its blend. `next`: a zeroed counter of the batch.
constexpr int kPool = 64;
constexpr int kFinishLanes = 12;
template <int FB>
struct SavedMarch {
    float v[FB + 3][kTraceThreads];   // C, D, T, hits of each thread's ray between rounds
};
template <int FB, int CAP, class Job>
__device__ __forceinline__ void walk_batch(const SceneView& S, const TraceParams& P, int rays, uint32_t* next,
                                           const Job& job, SavedMarch<FB>& saved) {
    uint32_t* queue = reinterpret_cast<uint32_t*>(warp_scratch<false>()) + (threadIdx.x & 31);
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    uint32_t stack[kStackSize];
    KBuffer<CAP> kb;
    kb.bind();
    RayWalk w;
    w.ok = true;
    w.ni = -1;
    w.qn = 0;
    Ray ray = make_ray(mk3(0.f, 0.f, 0.f), mk3(0.f, 0.f, 1.f));
    RayBox rb = make_ray_box(ray);
    uint64_t last_key = 0u;
    int32_t last_u = 0;
    int j = -1;                      // this lane's ray
    bool fresh = false;              // in its first round
    int pool = 0, pool_end = 0;      // the warp's rays not yet taken
    bool dry = false;                // the batch has no more
    for (;;) {
        const unsigned walk = __ballot_sync(kFullWarp, w.can_walk());
        const unsigned have = __ballot_sync(kFullWarp, w.qn > 0);
        const unsigned wait = __ballot_sync(kFullWarp, w.ni < 0 && w.qn == 0 && (j >= 0 || !dry));
        if (__popc(wait) >= kFinishLanes || (walk | have) == 0u) {
            if (wait == 0u) break;
            bool want = false;
            if (w.ni < 0 && w.qn == 0) {
                want = true;
                if (j >= 0) {
                    MarchState<FB> st;
                    st.init();
                    if (!fresh) {
#pragma unroll
                        for (int c = 0; c < FB; ++c) st.C[c] = saved.v[c][threadIdx.x];
                        st.D = saved.v[FB][threadIdx.x];
                        st.T = saved.v[FB + 1][threadIdx.x];
                        st.nh = __float_as_int(saved.v[FB + 2][threadIdx.x]);
                    }
                    if (blend_round<FB>(S, ray, P, kb, st, job.ids(j), job.max_ids, last_key, last_u)) {
                        job.finish(j, st);
                        j = -1;
                    } else {
#pragma unroll
                        for (int c = 0; c < FB; ++c) saved.v[c][threadIdx.x] = st.C[c];
                        saved.v[FB][threadIdx.x] = st.D;
                        saved.v[FB + 1][threadIdx.x] = st.T;
                        saved.v[FB + 2][threadIdx.x] = __int_as_float(st.nh);
                        fresh = false;
                        want = false;
                        kb.open(S.n, st.T, P.T_min);
                        w.start(S, P, last_key);
                    }
                }
            }
            // new rays for the lanes that want one: the pool's, then one more pool's
            bool got = false;
            unsigned need = __ballot_sync(kFullWarp, want);
#pragma unroll
            for (int turn = 0; turn < 2; ++turn) {
                const int mine = pool + __popc(need & lt);
                if (want && mine < pool_end) {
                    j = mine;
                    want = false;
                    got = true;
                }
                pool = min(pool + __popc(need), pool_end);
                need = __ballot_sync(kFullWarp, want);
                if (turn == 0 && need != 0u && !dry) {
                    uint32_t first = 0u;
                    if (lane == 0) first = atomicAdd(next, 1u);
                    first = __shfl_sync(kFullWarp, first, 0);
                    dry = first >= (uint32_t)(rays + kPool - 1) / kPool;
                    pool = dry ? 0 : (int)first * kPool;
                    pool_end = dry ? 0 : min(pool + kPool, rays);
                }
            }
            if (got) {
                f3 o, d;
                if (job.load(j, o, d)) {
                    ray = make_ray(o, d);
                    rb = make_ray_box(ray);
                    last_key = depth_key(P.t_min, 0.f);
                    last_u = INT32_MAX;
                    fresh = true;
                    kb.open(S.n, 1.f, P.T_min);
                    w.start(S, P, last_key);
                } else {
                    j = -1;
                }
            }
            continue;
        }
        if (__popc(walk) <= __popc(have)) {
            if (w.qn > 0) walk_leaf<KBuffer<CAP>, false>(S, ray, P, last_key, last_u, kb, w, queue, nullptr);
        } else {
            if (w.can_walk()) walk_node<false>(S, rb, w, stack, queue, nullptr);
        }
    }
    if (!w.ok) atomicOr(S.status, kErrStackOverflow);
}

// Blocks of a walk_batch launch: what the device holds, or fewer for a batch
// that has not a pool for each of their warps. 0 on an error.
template <class Kernel>
inline unsigned batch_blocks(Kernel kernel, int64_t rays) {
    int device = 0, sms = 0, per_sm = 0;
    if (cudaGetDevice(&device) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kTraceThreads, 0) != cudaSuccess)
        return 0u;
    const int64_t need = (rays + kTraceThreads - 1) / kTraceThreads, hold = (int64_t)sms * per_sm;
    return (unsigned)(need < hold ? need : hold);
}

__host__ __device__ inline TraceParams to_params(const irgs_trace_params& p) {
    TraceParams t;
    t.alpha_min = p.alpha_min;
    t.alpha_max = p.alpha_max;
    t.T_min = p.T_min;
    t.t_min = p.t_min;
    t.t_max = p.t_max;
    t.off = p.feat_offset;
    t.fc = p.feat_count;
    return t;
}

}  // namespace irgs
