// Relighting query (IRGS supplementary "Relighting details", Eq. 18; Sec. 4,
// relighting paragraph).
//
// Under a new environment the surfels' optimised radiance no longer holds,
// so each incident ray instead blends the albedo, roughness and normal of
// the surfels it crosses (normalised blend weights) and that aggregate
// surface is shaded with pre-integrated maps of the environment:
//   L_ind = O (A_r Irr(N_r) + Pref(reflect(v, N_r), R_r) (F0 A + B)(N_r.v, R_r)),
// O = 1 - V the ray's opacity, v = -w_i, Irr the diffuse irradiance map,
// Pref the split-sum prefiltered radiance and (A, B) the split-sum BRDF
// table. Incident directions are drawn by importance sampling the
// environment's intensity. Pre-integration (once per environment):
//   irradiance  Irr(N) = 1/pi sum_t E_t max(0, w_t.N) dOmega_t      [32 x 64]
//   prefilter   Pref_l(R) = sum_t E_t D_l(R.h_t) (w_t.R)+ dOmega_t / sum_t D_l (w_t.R)+ dOmega_t,
//               roughness l/5, l = 1..5                               [64 x 128 each]
//   BRDF table  A, B over (n.v, roughness) cell centres, 1024 Hammersley
//               GGX half vectors per cell                             [32 x 32]
//   sampling    row and per-row column cdfs of lum(E) sin(theta_row), FP64
// over all environment texels t (centre direction w_t, exact band solid
// angle dOmega_t). The environment is cut into slices; a block sums one slice
// for a tile of output texels, and the slices are then added in order, so the
// maps are deterministic.
#include <cuda_runtime.h>

#include <new>

#include "scene.h"
#include "shade.cuh"
#include "trace.cuh"
#include "trace_warp.cuh"
#include "wave.cuh"

namespace irgs {
namespace {

constexpr int kIrrH = IRGS_RELIGHT_IRR_H, kIrrW = IRGS_RELIGHT_IRR_W;
constexpr int kLevels = IRGS_RELIGHT_LEVELS;
constexpr int kPrefH = IRGS_RELIGHT_PREF_H, kPrefW = IRGS_RELIGHT_PREF_W;
constexpr int kLutN = IRGS_RELIGHT_LUT_N;
constexpr int kLutSamples = 1024;
constexpr int kRelightThreads = kTraceThreads;

// Centre direction of texel (row, col) of an h x w equirect map. The azimuth over
// pi is one quotient of whole numbers in (-1, 1): the texel's weight at the peak
// of prefilter level 1 changes by 25 to 50 times the angle's error.
__device__ __forceinline__ f3 texel_dir(int h, int w, int row, int col) {
    float st, ct, sp, cp;
    sincospif(((float)row + 0.5f) / (float)h, &st, &ct);
    sincospif((float)(2 * col + 1 - w) / (float)w, &sp, &cp);
    return mk3(st * cp, st * sp, ct);
}

// Solid angle of a texel of `row`: (cos t0 - cos t1) 2 pi / W written as
// 2 sin((t0 + t1)/2) sin((t1 - t0)/2) 2 pi / W (no cancellation at the poles).
__device__ __forceinline__ float texel_solid_angle(int H, int W, int row) {
    const float m = sinpif(((float)row + 0.5f) / (float)H);
    const float h = sinpif(0.5f / (float)H);
    return 2.f * m * h * 2.f * kPi / (float)W;
}

// Sums over the environment for a tile of output texels. A sum over all
// texels costs a direction (two sincospi) and a weight per (output, texel)
// pair, 1.1e9 pairs for the prefilter of a 512 x 256 environment; computing
// both per pair took 25 ms (prefilter) and 1.2 ms (irradiance). Here a block
// makes the directions of 128 texels at a time once for its 128 x kMapTexels
// outputs, all prefilter levels share a pair's geometry, and a warp whose
// outputs (8 x 4 patches) all face away skips the weights.
//
// Bound by the FP32 pipe and the reciprocals' latency (issue active in 61% of
// the cycles): a thread's two outputs are one packed pair of
// FP32 lanes, which halves the arithmetic but for the reciprocals (one per output
// and level). A slice is every so-many-th chunk of 128 texels, so that each sees
// all of the sphere (contiguous ones face some tiles wholly and others not at
// all); an odd number of slices walks through the columns of maps of 2^k
// columns. An environment of 512 x 256 and the relighting of 4,096 points under
// it took 2.98 ms (3.50 without pairs; 27 prefilter slices, as many blocks as
// fit at once, 3.18; 127 slices 2.95, for twice the memory) before the groups below.
//
// Sums are made in three steps: kMapGroup texels in one accumulator, the groups
// of a slice in another, the slices with their rounding errors carried along.
// The errors of groups and of slices are independent, so what they leave of the
// total falls with the square root of their number: 4e-8 rms relative at
// 512 x 256 texels and 7e-8 at 2048 x 1024 (level 1: 7e-8 and 9e-8). A block-wide
// tree per output left 9e-8 and 2e-7 (1.4e-7 and 1.7e-6), one accumulator per
// slice 2e-7 and 1.2e-6 (3.5e-7 and 1e-5). With the tables' running sums the
// groups take 7% of an environment's time (512 x 256: 1.74 -> 1.86 ms; groups of
// 16 1.93, of 64 1.84, but 1.2e-7 at 32 x 16 texels, where the tree had 1e-7).
constexpr int kMapThreads = 128;
constexpr int kMapTexels = 2;      // output texels per thread
constexpr int kMapGroup = 32;      // environment texels per accumulator
constexpr int kMapSlice = 128;     // least environment texels per slice
constexpr int kPrefSlices = 63;    // x 32 tiles
constexpr int kIrrSlices = 217;    // x 8 tiles

// Output texel (row, col) of thread t of tile `tile`, its j-th: warps cover
// patches of 8 columns x 4 rows, the j-th patch 4 rows further down.
__device__ __forceinline__ void map_texel(int w, int tile, int j, int& row, int& col) {
    const int patch = tile * (kMapThreads / 32) + (threadIdx.x >> 5), across = w / 8;
    row = (patch / across * kMapTexels + j) * 4 + (threadIdx.x & 31) / 8;
    col = patch % across * 8 + (threadIdx.x & 7);
}

// A pair of FP32 lanes, each rounded as the scalar operation.
__device__ __forceinline__ uint64_t pack2(float2 a) { return (uint64_t)__float_as_uint(a.y) << 32 | __float_as_uint(a.x); }
__device__ __forceinline__ float2 unpack2(uint64_t a) {
    return make_float2(__uint_as_float((uint32_t)a), __uint_as_float((uint32_t)(a >> 32)));
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)), "l"(pack2(c)));
    return unpack2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a)), "l"(pack2(b)));
    return unpack2(r);
}
// Within 1 ulp for normal x (the division of __fdividef without its scaling of
// denormal divisors).
__device__ __forceinline__ float reciprocal(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

// A texel of the environment: direction, solid angle and radiance, each twice.
struct MapTexel {
    float2 dx, dy, dz, omega, ex, ey, ez, pad;
};

// The texels of slice blockIdx.y: fn(texel, whether the radiance of its chunk
// is finite) for each, group() after every kMapGroup of them. The second is a
// type: asked per texel and level it took a quarter of the kernel's time.
template <bool YES>
struct Finite {};
template <class Fn, class Group>
__device__ __forceinline__ void for_texels(const float* __restrict__ env, int H, int W, Fn fn, Group group) {
    __shared__ MapTexel s_tex[kMapThreads];
    const int64_t all = (int64_t)H * W;
    for (int64_t t0 = (int64_t)blockIdx.y * kMapThreads; t0 < all; t0 += (int64_t)gridDim.y * kMapThreads) {
        const int64_t t = t0 + threadIdx.x;
        bool finite = true;
        if (t < all) {
            const int r = (int)(t / W), c = (int)(t - (int64_t)r * W);
            const f3 d = texel_dir(H, W, r, c), e = mk3(env[3 * t], env[3 * t + 1], env[3 * t + 2]);
            MapTexel m;
            m.dx = both(d.x);
            m.dy = both(d.y);
            m.dz = both(d.z);
            m.omega = both(texel_solid_angle(H, W, r));
            m.ex = both(e.x);
            m.ey = both(e.y);
            m.ez = both(e.z);
            m.pad = both(0.f);
            s_tex[threadIdx.x] = m;
            finite = fabsf(e.x) < INFINITY && fabsf(e.y) < INFINITY && fabsf(e.z) < INFINITY;
        }
        finite = __syncthreads_and(finite);
        const int n = (int)(all - t0 < kMapThreads ? all - t0 : kMapThreads);
        for (int g = 0; g < n; g += kMapGroup) {
            const int e = min(g + kMapGroup, n);
            if (finite)
                for (int i = g; i < e; ++i) fn(s_tex[i], Finite<true>());
            else
                for (int i = g; i < e; ++i) fn(s_tex[i], Finite<false>());
            group();
        }
        __syncthreads();
    }
}

// Directions of a thread's two outputs, and their texels.
struct PairDir {
    float2 x, y, z;
};
__device__ __forceinline__ PairDir pair_dir(int h, int w, int (&id)[2]) {
    static_assert(kMapTexels == 2, "two outputs are a packed pair");
    f3 d[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        int row, col;
        map_texel(w, blockIdx.x, j, row, col);
        d[j] = texel_dir(h, w, row, col);
        id[j] = row * w + col;
    }
    return {make_float2(d[0].x, d[1].x), make_float2(d[0].y, d[1].y), make_float2(d[0].z, d[1].z)};
}

// Projected solid angle of a texel for a pair of outputs, zero for one that it
// does not face.
__device__ __forceinline__ float2 facing(float2 cs, const MapTexel& t) {
    return make_float2(cs.x > 0.f ? cs.x * t.omega.x : 0.f, cs.y > 0.f ? cs.y * t.omega.y : 0.f);
}

// acc += radiance x weight. Infinities and NaN must not meet the zero weight of
// the output that the texel does not face: chunks that hold any take the
// outputs one by one.
template <bool FINITE>
__device__ __forceinline__ void add_weighted(float2* acc, const MapTexel& t, float2 wgt, float2 cs, Finite<FINITE>) {
    const float2 e[3] = {t.ex, t.ey, t.ez};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (FINITE) {
            acc[c] = fma2(e[c], wgt, acc[c]);
        } else {
            if (cs.x > 0.f) acc[c].x = fmaf(e[c].x, wgt.x, acc[c].x);
            if (cs.y > 0.f) acc[c].y = fmaf(e[c].y, wgt.y, acc[c].y);
        }
    }
}

// Irradiance partial sums: part[slice][texel] = sum E max(0, w.N) dOmega.
__global__ void __launch_bounds__(kMapThreads) k_irradiance(const float* __restrict__ env, int H, int W,
                                                            float4* __restrict__ part) {
    int id[2];
    const PairDir N = pair_dir(kIrrH, kIrrW, id);
    float2 acc[3] = {both(0.f), both(0.f), both(0.f)}, group_acc[3] = {both(0.f), both(0.f), both(0.f)};
    bool some = false;   // has the group a texel that an output faces?
    for_texels(
        env, H, W,
        [&](const MapTexel& t, auto finite) {
            const float2 cs = fma2(t.dx, N.x, fma2(t.dy, N.y, mul2(t.dz, N.z)));
            if (!(cs.x > 0.f || cs.y > 0.f)) return;
            some = true;
            add_weighted(group_acc, t, facing(cs, t), cs, finite);
        },
        [&]() {
            if (!some) return;
            some = false;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                acc[c] = add2(acc[c], group_acc[c]);
                group_acc[c] = both(0.f);
            }
        });
    float4* out = part + (int64_t)blockIdx.y * (kIrrH * kIrrW);
    out[id[0]] = make_float4(acc[0].x, acc[1].x, acc[2].x, 0.f);
    out[id[1]] = make_float4(acc[0].y, acc[1].y, acc[2].y, 0.f);
}

// Prefilter partial sums of every level: part[slice][level - 1][texel] = sums
// of E wgt and wgt, wgt = (w.R)+ dOmega / q^2 (the constant a^2 / pi of D
// cancels in their ratio). With the half vector h of the unit vectors w and R,
// |R x h|^2 = |w - R|^2 / 4 and (R.h)^2 is one less that: no h is needed, and
// nothing cancels near the peak.
__global__ void __launch_bounds__(kMapThreads) k_prefilter(const float* __restrict__ env, int H, int W,
                                                           float4* __restrict__ part) {
    constexpr int kL = kLevels - 1;
    int id[2];
    const PairDir R = pair_dir(kPrefH, kPrefW, id);
    // the slice's sums lie in shared memory: in registers they would take half of the blocks
    __shared__ float2 s_acc[kL][4][kMapThreads];
    float2 group_acc[kL][4];
#pragma unroll
    for (int l = 0; l < kL; ++l)
#pragma unroll
        for (int c = 0; c < 4; ++c) s_acc[l][c][threadIdx.x] = group_acc[l][c] = both(0.f);
    bool some = false;
    for_texels(
        env, H, W,
        [&](const MapTexel& t, auto finite) {
            const float2 cs = fma2(t.dx, R.x, fma2(t.dy, R.y, mul2(t.dz, R.z)));
            if (!(cs.x > 0.f || cs.y > 0.f)) return;
            some = true;
            const float2 w = facing(cs, t);
            const float2 gx = fma2(R.x, both(-1.f), t.dx), gy = fma2(R.y, both(-1.f), t.dy), gz = fma2(R.z, both(-1.f), t.dz);
            const float2 x2 = mul2(both(0.25f), fma2(gx, gx, fma2(gy, gy, mul2(gz, gz))));
            const float2 nh2 = fma2(x2, both(-1.f), both(1.f));
#pragma unroll
            for (int l = 0; l < kL; ++l) {
                const float rho = (float)(l + 1) / (float)(kLevels - 1);
                const float2 q = fma2(nh2, both(rho * rho * rho * rho), x2);   // (n.h)^2 (a2 - 1) + 1
                const float2 qq = mul2(q, q);
                const float2 wgt = mul2(w, make_float2(reciprocal(qq.x), reciprocal(qq.y)));
                add_weighted(group_acc[l], t, wgt, cs, finite);
                group_acc[l][3] = add2(group_acc[l][3], wgt);
            }
        },
        [&]() {
            if (!some) return;
            some = false;
#pragma unroll
            for (int l = 0; l < kL; ++l)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    s_acc[l][c][threadIdx.x] = add2(s_acc[l][c][threadIdx.x], group_acc[l][c]);
                    group_acc[l][c] = both(0.f);
                }
        });
#pragma unroll
    for (int l = 0; l < kL; ++l) {
        float4* out = part + ((int64_t)blockIdx.y * kL + l) * (kPrefH * kPrefW);
        float2 acc[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] = s_acc[l][c][threadIdx.x];
        out[id[0]] = make_float4(acc[0].x, acc[1].x, acc[2].x, acc[3].x);
        out[id[1]] = make_float4(acc[0].y, acc[1].y, acc[2].y, acc[3].y);
    }
}

// s += v, its rounding error into e.
__device__ __forceinline__ void carry_sum(float& s, float& e, float v) {
    float t, d;
    two_sum(s, v, t, d);
    s = t;
    e += d;
}
// The sum with what it lost; as it is where it is not finite (the errors are NaN there).
__device__ __forceinline__ float carried(float s, float e) { return fabsf(e) < INFINITY ? s + e : s; }

// The slices' partial sums in order: irradiance texels, then prefilter texels
// of every level.
__global__ void k_map_sums(const float4* __restrict__ irr_part, const float4* __restrict__ pref_part, int irr_slices,
                           int pref_slices, float* __restrict__ irr, float* __restrict__ pref) {
    constexpr int kI = kIrrH * kIrrW, kP = (kLevels - 1) * kPrefH * kPrefW;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kI + kP) return;
    const bool is_irr = i < kI;
    const float4* p = is_irr ? irr_part + i : pref_part + (i - kI);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f), e = s;
#pragma unroll 8
    for (int k = 0; k < (is_irr ? irr_slices : pref_slices); ++k) {
        const float4 v = p[(int64_t)k * (is_irr ? kI : kP)];
        carry_sum(s.x, e.x, v.x);
        carry_sum(s.y, e.y, v.y);
        carry_sum(s.z, e.z, v.z);
        carry_sum(s.w, e.w, v.w);
    }
    s = make_float4(carried(s.x, e.x), carried(s.y, e.y), carried(s.z, e.z), carried(s.w, e.w));
    if (is_irr) {
        irr[3 * i] = s.x * (1.f / kPi);
        irr[3 * i + 1] = s.y * (1.f / kPi);
        irr[3 * i + 2] = s.z * (1.f / kPi);
    } else {
        float* o = pref + 3 * (int64_t)(i - kI);
        o[0] = s.w > 0.f ? s.x / s.w : 0.f;
        o[1] = s.w > 0.f ? s.y / s.w : 0.f;
        o[2] = s.w > 0.f ? s.z / s.w : 0.f;
    }
}

// One warp per table cell.
__global__ void k_brdf_table(float* __restrict__ lut) {
    const int cell = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x & 31;
    if (cell >= kLutN * kLutN) return;
    const int i = cell / kLutN, j = cell % kLutN;
    const float mu = ((float)i + 0.5f) / (float)kLutN, rho = ((float)j + 0.5f) / (float)kLutN;
    const float ag = rho * rho, a2 = ag * ag, kk = 0.5f * ag;
    const f3 v = mk3(sqrtf(1.f - mu * mu), 0.f, mu);
    float A = 0.f, B = 0.f;
    for (int s = lane; s < kLutSamples; s += 32) {
        const float u1 = ((float)s + 0.5f) / (float)kLutSamples;
        const float u2 = (float)__brev((unsigned)s) * 2.3283064365386963e-10f;   // radical inverse, base 2
        const float om = 1.f - u1;
        const float inv = 1.f / fmaf(a2, u1, om);
        const float ct = sqrtf(om * inv), st = sqrtf(a2 * u1 * inv);
        float sp, cp;
        sincospif(2.f * u2, &sp, &cp);
        const f3 h = mk3(st * cp, st * sp, ct);
        const float vh = dot3(v, h);
        const float lz = 2.f * vh * h.z - v.z;
        if (lz <= 0.f || vh <= 0.f) continue;
        const float G = (lz / (lz * (1.f - kk) + kk)) * (mu / (mu * (1.f - kk) + kk));
        const float gv = G * vh / (h.z * mu);
        const float om5 = 1.f - vh, om52 = om5 * om5;
        const float fc = om52 * om52 * om5;
        A += (1.f - fc) * gv;
        B += fc * gv;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        A += __shfl_xor_sync(0xffffffffu, A, off);
        B += __shfl_xor_sync(0xffffffffu, B, off);
    }
    if (lane == 0) {
        lut[cell * 2] = A / (float)kLutSamples;
        lut[cell * 2 + 1] = B / (float)kLutSamples;
    }
}

// Importance-sampling tables, FP64: one warp per row for the column cdfs,
// then one warp for the row cdf, as running sums in order: each entry is the
// one before it plus a term >= 0, rounded, so the tables never decrease and a
// black texel has no width at all (sums associated otherwise differ in the
// last bit there, and a sample that lands on such a bit of width has a pdf of
// 1e-16). The lanes make 32 terms at a time; all of them carry the sum.
// Bound by the chain of FP64 additions.
__device__ __forceinline__ double warp_running_sum(double v, double& run) {
    const int lane = threadIdx.x & 31;
    double mine = 0.0;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        run = __dadd_rn(run, __shfl_sync(0xffffffffu, v, i));
        if (lane == i) mine = run;
    }
    return mine;
}

__global__ void k_env_col_cdf(const float* __restrict__ env, int H, int W, double* __restrict__ col_cdf) {
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x & 31;
    if (r >= H) return;
    const double s = sin(((double)r + 0.5) * 3.14159265358979323846 / (double)H);
    double* cc = col_cdf + (int64_t)r * (W + 1);
    double run = 0.0;
    if (lane == 0) cc[0] = 0.0;
    for (int c0 = 0; c0 < W; c0 += 32) {
        const int c = c0 + lane;
        double v = 0.0;
        if (c < W) {
            const float* e = env + ((int64_t)r * W + c) * 3;
            const double lum = __dadd_rn(__dadd_rn(__dmul_rn(0.2126, (double)e[0]), __dmul_rn(0.7152, (double)e[1])),
                                         __dmul_rn(0.0722, (double)e[2]));
            v = __dmul_rn(lum, s);
        }
        v = warp_running_sum(v, run);
        if (c < W) cc[c + 1] = v;
    }
}

__global__ void k_env_row_cdf(const double* __restrict__ col_cdf, int H, int W, double* __restrict__ row_cdf) {
    double run = 0.0;
    if (threadIdx.x == 0) row_cdf[0] = 0.0;
    for (int r0 = 0; r0 < H; r0 += 32) {
        const int r = r0 + threadIdx.x;
        const double v = warp_running_sum(r < H ? col_cdf[(int64_t)r * (W + 1) + W] : 0.0, run);
        if (r < H) row_cdf[r + 1] = v;
    }
}

// Largest k in [0, n) with cdf[k] <= t (cdf[0] <= t < cdf[n]).
__device__ __forceinline__ int cdf_find(const double* __restrict__ cdf, int n, double t) {
    int lo = 0, hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (cdf[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

// Environment sample from (u1, u2) (row, then column within the row; the
// leftover fractions place the direction inside the texel). Returns false
// if the environment has no weight.
__device__ __forceinline__ bool env_sample(const double* __restrict__ row_cdf, const double* __restrict__ col_cdf,
                                           int H, int W, double u1, double u2, f3& w, float& pdf) {
    const double total = row_cdf[H];
    if (!(total > 0.0)) return false;
    const double t1 = u1 * total;
    const int r = cdf_find(row_cdf, H, t1);
    const double* cc = col_cdf + (int64_t)r * (W + 1);
    const double rw = cc[W];
    const double fv = (t1 - row_cdf[r]) / rw;
    const double t2 = u2 * rw;
    const int c = cdf_find(cc, W, t2);
    const double wt = cc[c + 1] - cc[c];
    const double fu = (t2 - cc[c]) / wt;
    double st, ct, sp, cp;
    sincospi(((double)r + fv) / (double)H, &st, &ct);
    sincospi(((double)c + fu) * 2.0 / (double)W - 1.0, &sp, &cp);
    w = mk3((float)(st * cp), (float)(st * sp), (float)ct);
    pdf = st > 0.0 ? (float)((wt / total) * (double)W * (double)H / (2.0 * 3.14159265358979323846 *
                                                                       3.14159265358979323846 * st))
                   : 0.f;
    return pdf > 0.f;
}

struct EnvMaps {
    const float *env, *irr, *pref, *lut;
    const double *row_cdf, *col_cdf;
    int H, W;
};

// Split-sum prefiltered radiance at roughness rho: linear between the two
// nearest levels (level 0 is the environment).
__device__ __forceinline__ f3 pref_lookup(const EnvMaps& M, f3 d, float rho) {
    rho = fminf(fmaxf(rho, 0.f), 1.f);
    const float t = rho * (float)(kLevels - 1);
    int l0 = (int)floorf(t);
    l0 = l0 > kLevels - 2 ? kLevels - 2 : l0;
    const float f = t - (float)l0;
    const f3 a = l0 == 0 ? env_lookup(M.env, M.H, M.W, d)
                         : env_lookup(M.pref + (int64_t)(l0 - 1) * kPrefH * kPrefW * 3, kPrefH, kPrefW, d);
    const f3 b = env_lookup(M.pref + (int64_t)l0 * kPrefH * kPrefW * 3, kPrefH, kPrefW, d);
    return add3(mul3(a, 1.f - f), mul3(b, f));
}

// Bilinear lookup of the BRDF table at (mu, rho), coordinates clamped to the
// cell centres.
__device__ __forceinline__ float2 lut_lookup(const float* __restrict__ lut, float mu, float rho) {
    const float x = fminf(fmaxf(mu * kLutN - 0.5f, 0.f), (float)(kLutN - 1));
    const float y = fminf(fmaxf(rho * kLutN - 0.5f, 0.f), (float)(kLutN - 1));
    int i0 = (int)floorf(x), j0 = (int)floorf(y);
    i0 = i0 > kLutN - 2 ? kLutN - 2 : i0;
    j0 = j0 > kLutN - 2 ? kLutN - 2 : j0;
    const float fx = x - (float)i0, fy = y - (float)j0;
    const float2* L = reinterpret_cast<const float2*>(lut);
    const float2 a = __ldg(L + i0 * kLutN + j0), b = __ldg(L + i0 * kLutN + j0 + 1);
    const float2 c = __ldg(L + (i0 + 1) * kLutN + j0), d = __ldg(L + (i0 + 1) * kLutN + j0 + 1);
    return make_float2((1.f - fx) * ((1.f - fy) * a.x + fy * b.x) + fx * ((1.f - fy) * c.x + fy * d.x),
                       (1.f - fx) * ((1.f - fy) * a.y + fy * b.y) + fx * ((1.f - fy) * c.y + fy * d.y));
}

__device__ __forceinline__ f3 ld3r(const float* p, int64_t i) { return mk3(p[3 * i], p[3 * i + 1], p[3 * i + 2]); }

// One environment sample w (density pdf) of a point, given its trace (the
// blended [albedo, roughness, normal] C and transmittance T): adds the
// estimate term f L_i (w.n) / pdf to acc[0..2], V to acc[3] and L_ind to
// acc[4..6].
__device__ __forceinline__ void relight_sample(const EnvMaps& M, const ShadeFrame& F, f3 a, f3 w, float pdf,
                                               const float (&C)[7], float T, float (&acc)[7]) {
    const float V = T, O = 1.f - T;
    f3 Lind = mk3(0.f, 0.f, 0.f);
    if (O > 0.f) {
        const f3 Ar = mul3(mk3(C[0], C[1], C[2]), 1.f / O);
        const float Rr = C[3] / O;
        const f3 v = mul3(w, -1.f);
        f3 Nr = mk3(C[4], C[5], C[6]);
        const float len2 = dot3(Nr, Nr);
        Nr = len2 > 1e-24f ? mul3(Nr, rsqrtf(len2)) : v;
        if (dot3(Nr, v) < 0.f) Nr = mul3(Nr, -1.f);
        const float mu = fminf(dot3(Nr, v), 1.f);
        const f3 refl = sub3(mul3(Nr, 2.f * mu), v);
        const f3 irr = env_lookup(M.irr, kIrrH, kIrrW, Nr);
        const f3 pf = pref_lookup(M, refl, Rr);
        const float2 AB = lut_lookup(M.lut, mu, Rr);
        const float spec = kF0 * AB.x + AB.y;
        Lind = mul3(add3(mk3(Ar.x * irr.x, Ar.y * irr.y, Ar.z * irr.z), mul3(pf, spec)), O);
    }
    acc[3] += V;
    acc[4] += Lind.x;
    acc[5] += Lind.y;
    acc[6] += Lind.z;
    const float ni = dot3(F.n, w);
    if (ni <= 0.f) return;
    const f3 h = normalize3(add3(w, F.wo));
    const float nh = dot3(F.n, h), oh = dot3(F.wo, h);
    const float q = ggx_q(F, h, nh);
    const float D = F.a2 / (kPi * q * q);
    const float G1i = ni / (ni * (1.f - F.kk) + F.kk);
    const float fs_cos = D * fresnel(oh) * G1i * F.G1o / (4.f * F.no);   // f_s (w.n)
    const f3 E = env_lookup(M.env, M.H, M.W, w);
    const float Li[3] = {V * E.x + Lind.x, V * E.y + Lind.y, V * E.z + Lind.z};
    const float av[3] = {a.x, a.y, a.z};
    const float inv_pdf = 1.f / pdf;
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c] += (av[c] * (1.f / kPi) * ni + fs_cos) * Li[c] * inv_pdf;
}

// Final per-point sums of a warp (fixed butterfly order).
__device__ __forceinline__ void relight_write(float (&acc)[7], int lane, int64_t p, int Sn, float* __restrict__ rgb,
                                              float* __restrict__ vis, float* __restrict__ ind) {
#pragma unroll
    for (int k = 0; k < 7; ++k)
        for (int off = 16; off > 0; off >>= 1) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], off);
    if (lane == 0) {
        const float inv = 1.f / (float)Sn;
        for (int c = 0; c < 3; ++c) rgb[3 * p + c] = acc[c] * inv;
        if (vis != nullptr) vis[p] = acc[3] * inv;
        if (ind != nullptr)
            for (int c = 0; c < 3; ++c) ind[3 * p + c] = acc[4 + c] * inv;
    }
}

// Environment sample s of point p (uniforms as in the shading estimate).
__device__ __forceinline__ bool relight_dir(const EnvMaps& M, int64_t p, int s, int Sn, uint64_t seed, f3& w,
                                            float& pdf) {
    const uint64_t i0 = ((uint64_t)p * (uint64_t)Sn + (uint64_t)s) * 2ull;
    const double u1 = (double)u01_from_bits(splitmix64_at(seed, i0));
    const double u2 = (double)u01_from_bits(splitmix64_at(seed, i0 + 1));
    return env_sample(M.row_cdf, M.col_cdf, M.H, M.W, u1, u2, w, pdf);
}

// One warp per point; lanes take samples s = lane, lane + 32, ...; the traced
// channels are [albedo (3), roughness, normal (3)].
__global__ void __launch_bounds__(kRelightThreads) k_relight(SceneView S, EnvMaps M, const float* __restrict__ xg,
                                                             const float* __restrict__ ng,
                                                             const float* __restrict__ ag,
                                                             const float* __restrict__ rg,
                                                             const float* __restrict__ wog, int64_t Pn, int Sn,
                                                             uint64_t seed, TraceParams TP, float* __restrict__ rgb,
                                                             float* __restrict__ vis, float* __restrict__ ind) {
    const int lane = threadIdx.x & 31;
    const int64_t p = blockIdx.x * (int64_t)(kRelightThreads / 32) + (threadIdx.x >> 5);
    if (p >= Pn) return;
    const f3 x = ld3r(xg, p), a = ld3r(ag, p);
    const ShadeFrame F = shade_frame(ld3r(ng, p), ld3r(wog, p), rg[p]);
    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};   // rgb, V, L_ind
    for (int s0 = 0; s0 < Sn; s0 += 32) {
        f3 w = mk3(0.f, 0.f, 1.f);
        float pdf = 0.f;
        const bool live = s0 + lane < Sn && relight_dir(M, p, s0 + lane, Sn, seed, w, pdf);
        MarchState<7> st;
        const bool ok = march_forward<7, false>(S, make_ray(x, w), TP, st, nullptr, 0, live, warp_scratch<false>());
        if (!live) continue;
        if (!ok) atomicOr(S.status, kErrStackOverflow);
        relight_sample(M, F, a, w, pdf, st.C, st.T, acc);
    }
    relight_write(acc, lane, p, Sn, rgb, vis, ind);
}

// Wavefront form: samples generated one thread each, regrouped by direction
// bin and origin, traced in that order (a warp per ray, in the largest batches
// a lane), then estimated per point from the stored traces with the same per-sample
// arithmetic and reduction order as k_relight.
__global__ void k_relight_gen(EnvMaps M, const float* __restrict__ xg, int64_t p0, int64_t rays, int Sn,
                              uint64_t seed, const uint32_t* __restrict__ bounds, float4* __restrict__ dir,
                              uint32_t* __restrict__ key, int32_t* __restrict__ val) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= rays) return;
    const int64_t p = p0 + i / Sn;
    f3 w = mk3(0.f, 0.f, 1.f);
    float pdf = 0.f;
    const bool ok = relight_dir(M, p, (int)(i % Sn), Sn, seed, w, pdf);
    const f3 x = ld3r(xg, p);
    dir[i] = make_float4(w.x, w.y, w.z, ok ? (can_hit(x, w) ? pdf : -pdf) : 0.f);   // < 0: a ray that meets nothing
    key[i] = ok ? wave_key(x, w, bounds) : kInvalidWaveKey;
    val[i] = (int32_t)i;
}

struct RelightJob {
    const float* xg;
    int64_t p0;
    int Sn;
    const float4* dir;
    const int32_t* order;
    float4* res;
    int max_ids;
    __device__ __forceinline__ bool load(int j, f3& o, f3& d) const {
        const int64_t i = order[j];
        const float4 d4 = dir[i];
        if (!(d4.w > 0.f)) {
            res[2 * i] = make_float4(0.f, 0.f, 0.f, 0.f);
            res[2 * i + 1] = make_float4(0.f, 0.f, 0.f, 1.f);
            return false;
        }
        o = ld3r(xg, p0 + i / Sn);
        d = mk3(d4.x, d4.y, d4.z);
        return true;
    }
    __device__ __forceinline__ int32_t* ids(int) const { return nullptr; }
    __device__ __forceinline__ void finish(int j, const MarchState<7>& st) const {
        const int64_t i = order[j];
        res[2 * i] = make_float4(st.C[0], st.C[1], st.C[2], st.C[3]);
        res[2 * i + 1] = make_float4(st.C[4], st.C[5], st.C[6], st.T);
    }
};

__global__ void __launch_bounds__(kRelightThreads, kRayBlocks) k_relight_trace(SceneView S, TraceParams P,
                                                                               RelightJob job, int rays,
                                                                               uint32_t* next) {
    __shared__ SavedMarch<7> saved;
    walk_batch<7, kCap>(S, P, rays, next, job, saved);
}

// The same with a warp per ray, for batches that do not fill the chip many
// times over with a ray per lane (the lines are shading's, shade_wave.cu). ms
// for scenes of 100k / 300k / 1M / 3M surfels, a warp per ray first:
//   0.26M rays   1.45 1.47 1.58 1.76    2.42 2.50 3.11 3.77
//   4.2M         21.4 21.7 22.4 24.1    22.7 24.1 27.4 33.7
//   8.4M         45.1 45.9 47.3 49.9    45.9 47.9 55.7 67.8
//   16.8M        73.5 73.8 74.6 76.8    70.9 72.1 81.3 93.9
constexpr int64_t kRelightUnsortedMax = int64_t(1) << 19;   // smaller batches gain less from the order than its sort costs
constexpr int64_t kRelightWarpMax = int64_t(1) << 23;
__global__ void __launch_bounds__(kWarpRayThreads, kWarpRayBlocks) k_relight_trace_ray(SceneView S, TraceParams P, RelightJob job,
                                                                                int rays) {
    const int j = blockIdx.x * kWarpRays + (threadIdx.x >> 5);
    f3 o, d;
    if (j >= rays || !job.load(j, o, d)) return;
    const Ray ray = make_ray(o, d);
    WarpMarch w;
    const bool ok = march_warp(S, ray, make_ray_box(ray), P, w, job.ids(j), job.max_ids, warp_ray_scratch());
    MarchState<7> st;
#pragma unroll
    for (int c = 0; c < 7; ++c) st.C[c] = __shfl_sync(kFullWarp, w.C, c);
    st.D = w.D;
    st.T = w.T;
    st.nh = w.nh;
    if ((threadIdx.x & 31) != 0) return;
    if (!ok) atomicOr(S.status, kErrStackOverflow);
    job.finish(j, st);
}

__global__ void __launch_bounds__(kRelightThreads) k_relight_shade(EnvMaps M, const float* __restrict__ ng,
                                                                   const float* __restrict__ ag,
                                                                   const float* __restrict__ rg,
                                                                   const float* __restrict__ wog, int64_t p0,
                                                                   int64_t np, int Sn, const float4* __restrict__ dir,
                                                                   const float4* __restrict__ res,
                                                                   float* __restrict__ rgb, float* __restrict__ vis,
                                                                   float* __restrict__ ind) {
    const int lane = threadIdx.x & 31;
    const int64_t k = blockIdx.x * (int64_t)(kRelightThreads / 32) + (threadIdx.x >> 5);
    if (k >= np) return;
    const int64_t p = p0 + k;
    const f3 a = ld3r(ag, p);
    const ShadeFrame F = shade_frame(ld3r(ng, p), ld3r(wog, p), rg[p]);
    float acc[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int s = lane; s < Sn; s += 32) {
        const int64_t i = k * Sn + s;
        const float4 d4 = __ldg(dir + i);
        if (d4.w == 0.f) continue;
        const float4 r0 = __ldg(res + 2 * i), r1 = __ldg(res + 2 * i + 1);
        const float C[7] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z};
        relight_sample(M, F, a, mk3(d4.x, d4.y, d4.z), fabsf(d4.w), C, r1.w, acc);
    }
    relight_write(acc, lane, p, Sn, rgb, vis, ind);
}

inline unsigned grid_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

constexpr int64_t kRelightChunkRays = int64_t(1) << 26;

cudaError_t relight_wave(const SceneView& S, const uint32_t* bounds, const EnvMaps& M, const float* x,
                         const float* n, const float* a, const float* r, const float* wo, int64_t P, int Sn,
                         uint64_t seed, const TraceParams& TP, float* rgb, float* vis, float* ind, cudaStream_t st) {
    const int64_t pc = kRelightChunkRays / Sn > 0 ? kRelightChunkRays / Sn : 1;
    const int64_t cap = (P < pc ? P : pc) * Sn;
    const int64_t hw = sort_hist_words(cap);
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t bytes = al(16 * cap) + 4 * al(4 * cap) + al(4 * hw) + al(32 * cap) + al(4);
    unsigned char* base = nullptr;
    cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&base), bytes, st);
    if (e != cudaSuccess) return e;
    size_t off = 0;
    auto take = [&](size_t b) { unsigned char* q = base + off; off += al(b); return q; };
    float4* dir = reinterpret_cast<float4*>(take(16 * cap));
    uint32_t* key = reinterpret_cast<uint32_t*>(take(4 * cap));
    int32_t* val = reinterpret_cast<int32_t*>(take(4 * cap));
    uint32_t* ktmp = reinterpret_cast<uint32_t*>(take(4 * cap));
    int32_t* vtmp = reinterpret_cast<int32_t*>(take(4 * cap));
    uint32_t* hist = reinterpret_cast<uint32_t*>(take(4 * hw));
    float4* res = reinterpret_cast<float4*>(take(32 * cap));
    uint32_t* next = reinterpret_cast<uint32_t*>(take(4));
    for (int64_t p0 = 0; p0 < P && e == cudaSuccess; p0 += pc) {
        const int64_t np = P - p0 < pc ? P - p0 : pc;
        const int64_t rays = np * Sn;
        k_relight_gen<<<grid_for(rays, 256), 256, 0, st>>>(M, x, p0, rays, Sn, seed, bounds, dir, key, val);
        if (rays > kRelightUnsortedMax) e = sort_pairs(key, val, ktmp, vtmp, hist, rays, st);
        if (e != cudaSuccess) break;
        const RelightJob job{x, p0, Sn, dir, val, res, 0};
        if (rays <= kRelightWarpMax) {
            k_relight_trace_ray<<<warp_ray_grid(rays), kWarpRayThreads, 0, st>>>(S, TP, job, (int)rays);
        } else {
            e = cudaMemsetAsync(next, 0, sizeof(uint32_t), st);
            const unsigned blocks = batch_blocks(k_relight_trace, rays);
            if (e == cudaSuccess && blocks == 0u) e = cudaGetLastError();
            if (e != cudaSuccess) break;
            k_relight_trace<<<blocks, kRelightThreads, 0, st>>>(S, TP, job, (int)rays, next);
        }
        count_launches(1);
        k_relight_shade<<<grid_for(np, kRelightThreads / 32), kRelightThreads, 0, st>>>(M, n, a, r, wo, p0, np, Sn,
                                                                                       dir, res, rgb, vis, ind);
        count_launches(2);
        e = cudaGetLastError();
    }
    const cudaError_t ef = cudaFreeAsync(base, st);
    return e != cudaSuccess ? e : ef;
}

}  // namespace

void free_envmap(irgs_envmap m) {
    if (m == nullptr) return;
    if (m->base) cudaFree(m->base);
    delete m;
}

irgs_status build_envmap_impl(const float* env, int32_t H, int32_t W, cudaStream_t st, irgs_envmap* out) {
    irgs_envmap m = new (std::nothrow) irgs_envmap_s();
    if (m == nullptr) return IRGS_ERR_OOM;
    cudaGetDevice(&m->device);
    m->H = H;
    m->W = W;
    // all maps in one allocation (each cudaMalloc and cudaFree costs as much as a small map)
    const size_t counts[6] = {sizeof(float) * (size_t)H * W * 3, sizeof(float) * kIrrH * kIrrW * 3,
                              sizeof(float) * (kLevels - 1) * kPrefH * kPrefW * 3, sizeof(float) * kLutN * kLutN * 2,
                              sizeof(double) * ((size_t)H + 1), sizeof(double) * (size_t)H * (W + 1)};
    size_t at[6], bytes = 0;
    for (int i = 0; i < 6; ++i) {
        at[i] = bytes;
        bytes += (counts[i] + 255) & ~size_t(255);
        m->bytes += (int64_t)counts[i];
    }
    cudaError_t e = cudaMalloc(&m->base, bytes);
    // the slices' partial sums
    const int64_t texels = (int64_t)H * W;
    const int64_t want = ((texels + kMapSlice - 1) / kMapSlice) | 1;
    const int irr_slices = (int)(want < kIrrSlices ? want : kIrrSlices);
    const int pref_slices = (int)(want < kPrefSlices ? want : kPrefSlices);
    constexpr int kIrr = kIrrH * kIrrW, kPref = kPrefH * kPrefW;
    float4* part = nullptr;
    if (e == cudaSuccess)
        e = scratch_alloc(reinterpret_cast<void**>(&part),
                          sizeof(float4) * ((size_t)irr_slices * kIrr + (size_t)pref_slices * (kLevels - 1) * kPref), st);
    if (e != cudaSuccess) {
        free_envmap(m);
        cudaGetLastError();
        return e == cudaErrorMemoryAllocation ? IRGS_ERR_OOM : IRGS_ERR_CUDA;
    }
    unsigned char* base = static_cast<unsigned char*>(m->base);
    m->env = reinterpret_cast<float*>(base + at[0]);
    m->irr = reinterpret_cast<float*>(base + at[1]);
    m->pref = reinterpret_cast<float*>(base + at[2]);
    m->lut = reinterpret_cast<float*>(base + at[3]);
    m->row_cdf = reinterpret_cast<double*>(base + at[4]);
    m->col_cdf = reinterpret_cast<double*>(base + at[5]);
    auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    A(cudaMemcpyAsync(m->env, env, sizeof(float) * (size_t)H * W * 3, cudaMemcpyDeviceToDevice, st));
    float4* pref_part = part + (size_t)irr_slices * kIrr;
    constexpr int kPer = kMapThreads * kMapTexels;
    static_assert(kIrr % kPer == 0 && kPref % kPer == 0 && kIrrW % 8 == 0 && kIrrH % (4 * kMapTexels) == 0 &&
                      kPrefH % (4 * kMapTexels) == 0, "whole tiles of patches");
    k_irradiance<<<dim3(kIrr / kPer, irr_slices), kMapThreads, 0, st>>>(m->env, H, W, part);
    k_prefilter<<<dim3(kPref / kPer, pref_slices), kMapThreads, 0, st>>>(m->env, H, W, pref_part);
    k_map_sums<<<(kIrr + (kLevels - 1) * kPref + 255) / 256, 256, 0, st>>>(part, pref_part, irr_slices, pref_slices, m->irr, m->pref);
    k_brdf_table<<<(kLutN * kLutN * 32 + 255) / 256, 256, 0, st>>>(m->lut);
    k_env_col_cdf<<<(unsigned)(((int64_t)H * 32 + 127) / 128), 128, 0, st>>>(m->env, H, W, m->col_cdf);
    k_env_row_cdf<<<1, 32, 0, st>>>(m->col_cdf, H, W, m->row_cdf);
    count_launches(6);
    A(cudaGetLastError());
    A(cudaFreeAsync(part, st));
    if (e != cudaSuccess) {
        cudaStreamSynchronize(st);
        free_envmap(m);
        return IRGS_ERR_CUDA;
    }
    *out = m;
    return IRGS_OK;
}

irgs_status export_envmap_impl(irgs_envmap m, float* irr, float* pref, float* lut, double* row_cdf,
                               double* col_cdf, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    const cudaMemcpyKind k = cudaMemcpyDefault;
    if (irr) A(cudaMemcpyAsync(irr, m->irr, sizeof(float) * kIrrH * kIrrW * 3, k, st));
    if (pref) A(cudaMemcpyAsync(pref, m->pref, sizeof(float) * (kLevels - 1) * kPrefH * kPrefW * 3, k, st));
    if (lut) A(cudaMemcpyAsync(lut, m->lut, sizeof(float) * kLutN * kLutN * 2, k, st));
    if (row_cdf) A(cudaMemcpyAsync(row_cdf, m->row_cdf, sizeof(double) * (m->H + 1), k, st));
    if (col_cdf) A(cudaMemcpyAsync(col_cdf, m->col_cdf, sizeof(double) * (size_t)m->H * (m->W + 1), k, st));
    return e == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

// Directions of the environment-importance samples the relighting traces:
// ray i = p * n_samples + s (they depend on the keys only, not on the point).
__global__ void k_relight_rays(EnvMaps M, int64_t rays, int Sn, uint64_t seed, float* __restrict__ dir,
                               float* __restrict__ pdf_out, int32_t* __restrict__ valid) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= rays) return;
    f3 w = mk3(0.f, 0.f, 1.f);
    float pdf = 0.f;
    const bool ok = relight_dir(M, i / Sn, (int)(i % Sn), Sn, seed, w, pdf);
    dir[3 * i] = w.x;
    dir[3 * i + 1] = w.y;
    dir[3 * i + 2] = w.z;
    if (pdf_out != nullptr) pdf_out[i] = ok ? pdf : 0.f;
    if (valid != nullptr) valid[i] = ok ? 1 : 0;
}

irgs_status launch_relight_rays(irgs_envmap m, int64_t P, int32_t n_samples, uint64_t seed, float* dir, float* pdf,
                                int32_t* valid, cudaStream_t st) {
    const int64_t rays = P * (int64_t)n_samples;
    if (rays == 0) return IRGS_OK;
    const EnvMaps M{m->env, m->irr, m->pref, m->lut, m->row_cdf, m->col_cdf, m->H, m->W};
    const int T = 256;
    k_relight_rays<<<(unsigned)((rays + T - 1) / T), T, 0, st>>>(M, rays, n_samples, seed, dir, pdf, valid);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

irgs_status launch_relight(const SceneView& S, const uint32_t* bounds, irgs_envmap m, const float* x,
                           const float* n, const float* albedo, const float* rough, const float* wo, int64_t P,
                           int32_t n_samples, uint64_t seed, const irgs_trace_params& p, float* rgb, float* vis,
                           float* ind, cudaStream_t st) {
    if (P == 0) return IRGS_OK;
    const TraceParams TP = to_params(p);
    const EnvMaps M{m->env, m->irr, m->pref, m->lut, m->row_cdf, m->col_cdf, m->H, m->W};
    if (p.k != 8 && p.k != 16) return IRGS_ERR_UNSUPPORTED;
    cudaError_t e = cudaSuccess;
    if ((p.flags & IRGS_FLAG_PER_THREAD) != 0u) {
        // fused: a warp per point tracing its own samples
        const int64_t blocks = (P + kRelightThreads / 32 - 1) / (kRelightThreads / 32);
        k_relight<<<(unsigned)blocks, kRelightThreads, 0, st>>>(S, M, x, n, albedo, rough, wo, P, n_samples, seed, TP,
                                                                rgb, vis, ind);
        count_launches(1);
        e = cudaGetLastError();
    } else {
        e = relight_wave(S, bounds, M, x, n, albedo, rough, wo, P, n_samples, seed, TP, rgb, vis, ind, st);
    }
    if (e == cudaErrorMemoryAllocation) return IRGS_ERR_OOM;
    return e == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

}  // namespace irgs
