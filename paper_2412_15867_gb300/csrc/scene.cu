// Scene construction: centre bounds, Morton codes and their stable radix sort
// (K1), surfel packing and support boxes in Morton order (K2), the binary
// hierarchy by locally-ordered clustering over the sorted leaves (K3; the
// Karras hierarchy as fallback), bottom-up box refit (K4) and the 4-wide
// collapse (K5). IRGS bounds each 2D Gaussian by a proxy enclosing the region
// where its response reaches alpha_min (Sec. 3.2, Eq. 5) and builds a BVH over
// the proxies; here the proxy is the axis-aligned box of the support disk and
// the BVH is a linear BVH built entirely on the device.
//
// K1, K3 and K5 are sequences of up to 100 short dependent steps. Each is one
// cooperative launch (one block of 1024 threads per SM) with a barrier over
// the grid between steps: as launches of their own the steps took 3 to 30 us
// each and 194 launches a build, most of them for levels and rounds that only
// some hierarchies have.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <mutex>
#include <new>

#include "common.cuh"
#include "scene.h"

namespace irgs {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortChunks = 16;                             // 32-key chunks per warp
constexpr int kTile = kSortThreads * kSortChunks;           // 4096 keys per tile

__device__ __forceinline__ uint32_t f2ord(float f) {
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}

// ---------------------------------------------------------------------------
// Cooperative kernels: at most kCoopBlocks blocks of kCoopThreads threads.
constexpr int kCoopThreads = 1024;
constexpr int kCoopBlocks = 160;

// Words of a scene's control array: the centre bounds, then per cooperative
// kernel an arrival count and a "gave up" flag, then the clustering build's
// fallback flag.
constexpr int kCtlOrder = 8, kCtlPloc = 10, kCtlWide = 12, kCtlFallback = 14;
constexpr int kCtlWords = 16;

// Barrier over the grid: every block of the (cooperative) launch calls it the
// same number of times. bar[0] counts arrivals, zero before the launch. A wait
// that runs out (it cannot, while the blocks are co-resident) sets bar[1],
// which ends every other wait, and false is returned to all threads.
__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t& target) {
    __shared__ int s_ok;
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        int ok = 0;
        for (int spin = 0; spin < (1 << 22); ++spin) {
            uint32_t v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int32_t)(v - target) >= 0) {
                ok = 1;
                break;
            }
            if ((spin & 255) == 255 && *(volatile uint32_t*)(bar + 1) != 0u) break;
        }
        if (!ok) atomicExch(bar + 1, 1u);
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Exclusive scan of one value per thread over the block (blockDim.x a
// multiple of 32); s_warp holds 33 words. Returns the prefix, *total the sum.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* s_warp, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < nw ? s_warp[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, off);
            if (lane >= off) wi += y;
        }
        if (lane < nw) s_warp[lane] = wi - w;
        if (lane == nw - 1) s_warp[32] = wi;
    }
    __syncthreads();
    const uint32_t r = s_warp[warp] + inc - v;
    *total = s_warp[32];
    __syncthreads();
    return r;
}

// ---------------------------------------------------------------------------
// K1: bounds of the centres, 30-bit Morton codes inside them, and their
// stable LSD radix sort, 8 bits per pass. A surfel whose values are not usable
// counts as centred at the origin in the bounds.
__device__ __forceinline__ uint32_t spread10(uint32_t v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

__device__ __forceinline__ bool usable(const float* q, float su, float sv, const float* mu, float o) {
    const bool q_ok = isfinite(q[0]) && isfinite(q[1]) && isfinite(q[2]) && isfinite(q[3]) &&
                      (q[0] != 0.f || q[1] != 0.f || q[2] != 0.f || q[3] != 0.f);
    return q_ok && su > 0.f && sv > 0.f && isfinite(su) && isfinite(sv) && isfinite(mu[0]) && isfinite(mu[1]) &&
           isfinite(mu[2]) && isfinite(o);
}

// Centre bounds over all threads of the grid into bounds (3 mins, 3 maxes).
__device__ __forceinline__ void centre_bounds(const float* __restrict__ means, const float* __restrict__ quats,
                                              const float* __restrict__ scales, const float* __restrict__ opac,
                                              int64_t n, uint32_t* bounds) {
    __shared__ uint32_t s_bounds[6];
    const int tid = threadIdx.x;
    float cmin[3] = {INFINITY, INFINITY, INFINITY}, cmax[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + tid; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float mu[3] = {means[3 * i], means[3 * i + 1], means[3 * i + 2]};
        const float q[4] = {quats[4 * i], quats[4 * i + 1], quats[4 * i + 2], quats[4 * i + 3]};
        const bool ok = usable(q, scales[2 * i], scales[2 * i + 1], mu, opac[i]);
        for (int k = 0; k < 3; ++k) {
            cmin[k] = fminf(cmin[k], ok ? mu[k] : 0.f);
            cmax[k] = fmaxf(cmax[k], ok ? mu[k] : 0.f);
        }
    }
    for (int k = 0; k < 3; ++k)
        for (int off = 16; off > 0; off >>= 1) {
            cmin[k] = fminf(cmin[k], __shfl_xor_sync(0xffffffffu, cmin[k], off));
            cmax[k] = fmaxf(cmax[k], __shfl_xor_sync(0xffffffffu, cmax[k], off));
        }
    if (tid < 6) s_bounds[tid] = tid < 3 ? 0xffffffffu : 0u;
    __syncthreads();
    if ((tid & 31) == 0 && cmin[0] <= cmax[0])
        for (int k = 0; k < 3; ++k) {
            atomicMin(&s_bounds[k], f2ord(cmin[k]));
            atomicMax(&s_bounds[3 + k], f2ord(cmax[k]));
        }
    __syncthreads();
    if (tid < 3) atomicMin(&bounds[tid], s_bounds[tid]);
    else if (tid < 6) atomicMax(&bounds[tid], s_bounds[tid]);
}

__global__ void __launch_bounds__(256) k_bounds(const float* __restrict__ means, const float* __restrict__ quats,
                                                const float* __restrict__ scales, const float* __restrict__ opac,
                                                int64_t n, uint32_t* __restrict__ bounds) {
    centre_bounds(means, quats, scales, opac, n, bounds);
}

// Sorts with passes > 0 (then even: the result ends in keys / vals); with
// passes = 0 only the codes are made. A block owns a contiguous piece of the
// keys; every block sums the digit counts of the pieces before its own. A
// barrier that gives up leaves an error bit and its flag, by which k_pack
// knows that the order is not there.
__global__ void __launch_bounds__(kCoopThreads, 1) k_order(
    const float* __restrict__ means, const float* __restrict__ quats, const float* __restrict__ scales,
    const float* __restrict__ opac, int64_t n, uint32_t* ctl, uint32_t* keys, int32_t* vals, uint32_t* keys_tmp,
    int32_t* vals_tmp, uint32_t* hist, int passes, uint32_t* status) {
    __shared__ uint32_t s_base[256], s_cnt[256];
    __shared__ uint32_t s_part[2][4][256];
    __shared__ uint16_t s_warp_cnt[kCoopThreads / 32][256];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t target = 0u;
    const uint32_t* bounds = ctl;
    auto meet = [&]() {
        const bool ok = grid_barrier(ctl + kCtlOrder, target);
        if (!ok && tid == 0) atomicOr(status, kErrBadTree);
        return ok;
    };
    centre_bounds(means, quats, scales, opac, n, ctl);
    if (!meet()) return;
    const int64_t piece = (n + gridDim.x - 1) / gridDim.x;
    const int64_t begin = blockIdx.x * piece, end = begin + piece < n ? begin + piece : n;
    {
        float lo[3], ext[3];
        for (int k = 0; k < 3; ++k) {
            lo[k] = ord2f(__ldcg(bounds + k));
            ext[k] = ord2f(__ldcg(bounds + 3 + k)) - lo[k];
        }
        for (int64_t i = begin + tid; i < end; i += kCoopThreads) {
            uint32_t q[3];
            for (int k = 0; k < 3; ++k) {
                const float t = ext[k] > 0.f ? (means[3 * i + k] - lo[k]) / ext[k] : 0.5f;
                int v = (int)(t * 1024.0f);
                v = v < 0 ? 0 : (v > 1023 ? 1023 : v);
                if (!(t == t)) v = 0;
                q[k] = (uint32_t)v;
            }
            keys[i] = (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
            vals[i] = (int32_t)i;
        }
    }
    const unsigned lt = (1u << lane) - 1u;
    for (int pass = 0; pass < passes; ++pass) {
        const uint32_t* kin = pass & 1 ? keys_tmp : keys;
        const int32_t* vin = pass & 1 ? vals_tmp : vals;
        uint32_t* kout = pass & 1 ? keys : keys_tmp;
        int32_t* vout = pass & 1 ? vals : vals_tmp;
        const int shift = 8 * pass;
        if (tid < 256) s_cnt[tid] = 0u;
        __syncthreads();
        for (int64_t i = begin + tid; i < end; i += kCoopThreads) atomicAdd(&s_cnt[(__ldcg(kin + i) >> shift) & 255u], 1u);
        __syncthreads();
        if (tid < 256) hist[blockIdx.x * 256 + tid] = s_cnt[tid];
        if (!meet()) return;
        // where this piece's keys of each digit go: all smaller digits, then the pieces before this one
        {
            const int d = tid & 255, quarter = tid >> 8;
            uint32_t before = 0u, all = 0u;
            for (int b = quarter; b < (int)gridDim.x; b += 4) {
                const uint32_t v = __ldcg(hist + b * 256 + d);
                all += v;
                before += b < (int)blockIdx.x ? v : 0u;
            }
            s_part[0][quarter][d] = before;
            s_part[1][quarter][d] = all;
        }
        __syncthreads();
        if (warp == 0) {   // exclusive scan of the 256 digit totals, 8 per lane
            uint32_t t[8], sum = 0u;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int d = lane * 8 + k;
                t[k] = s_part[1][0][d] + s_part[1][1][d] + s_part[1][2][d] + s_part[1][3][d];
                sum += t[k];
            }
            uint32_t inc = sum;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, off);
                if (lane >= off) inc += y;
            }
            uint32_t run = inc - sum;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int d = lane * 8 + k;
                s_base[d] = run + s_part[0][0][d] + s_part[0][1][d] + s_part[0][2][d] + s_part[0][3][d];
                run += t[k];
            }
        }
        for (int64_t i0 = begin; i0 < end; i0 += kCoopThreads) {
            const int64_t i = i0 + tid;
            for (int k = tid; k < kCoopThreads / 32 * 256 / 2; k += kCoopThreads)
                reinterpret_cast<uint32_t*>(&s_warp_cnt[0][0])[k] = 0u;
            __syncthreads();
            const uint32_t key = i < end ? __ldcg(kin + i) : 0u;
            const int32_t val = i < end ? __ldcg(vin + i) : 0;
            const uint32_t dg = i < end ? (key >> shift) & 255u : 256u;
            const unsigned peers = __match_any_sync(0xffffffffu, dg);
            if (dg < 256u && (peers & lt) == 0u) s_warp_cnt[warp][dg] = (uint16_t)__popc(peers);
            __syncthreads();
            uint32_t total = 0u;
            if (tid < 256) {
                uint32_t c[kCoopThreads / 32];
#pragma unroll
                for (int w = 0; w < kCoopThreads / 32; ++w) c[w] = s_warp_cnt[w][tid];
#pragma unroll
                for (int w = 0; w < kCoopThreads / 32; ++w) {
                    s_warp_cnt[w][tid] = (uint16_t)total;
                    total += c[w];
                }
            }
            __syncthreads();
            if (dg < 256u) {
                const uint32_t pos = s_base[dg] + s_warp_cnt[warp][dg] + __popc(peers & lt);
                kout[pos] = key;
                vout[pos] = val;
            }
            __syncthreads();
            if (tid < 256) s_base[tid] += total;
        }
        if (!meet()) return;
    }
}

// ---------------------------------------------------------------------------
// K2: per surfel, in Morton order: frame (FP64, then rounded once), support
// radius, packed record, padded support-disk box, raw quaternion and scales.
// Bound by the FP64 pipe, so its divisions and roots are few: 2 / |q|^2 and
// the two inverse scales (normalising q first took 12 divisions and 5 roots
// per surfel, 149 us for 300k surfels against 35), the logarithm of the support
// radius only where it is not capped, and the box extents' roots in FP32,
// whose error the boxes' padding of 1e-5 covers a hundred times.
// With `no_order` set and nonzero, perm and keys hold no order: the surfels
// then keep the user's, with equal keys, from which every later step builds a
// valid (if poor) hierarchy.
__global__ void __launch_bounds__(256) k_pack(int32_t* __restrict__ perm, uint32_t* __restrict__ keys,
                                              const uint32_t* __restrict__ no_order, const float* __restrict__ means,
                                              const float* __restrict__ quats, const float* __restrict__ scales,
                                              const float* __restrict__ opac, int64_t n, double alpha_min,
                                              float4* __restrict__ rec, float* __restrict__ leaf_box,
                                              float4* __restrict__ q_raw, float2* __restrict__ scale,
                                              int32_t* __restrict__ inv_perm) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= n) return;
    if (no_order != nullptr && *no_order != 0u) {
        perm[j] = (int32_t)j;
        keys[j] = 0u;
    }
    const int32_t i = perm[j];
    if (inv_perm != nullptr) inv_perm[i] = (int32_t)j;
    const float muf[3] = {means[3 * (int64_t)i], means[3 * (int64_t)i + 1], means[3 * (int64_t)i + 2]};
    const float qf[4] = {quats[4 * (int64_t)i], quats[4 * (int64_t)i + 1], quats[4 * (int64_t)i + 2],
                         quats[4 * (int64_t)i + 3]};
    const float suf = scales[2 * (int64_t)i], svf = scales[2 * (int64_t)i + 1], of = opac[i];
    q_raw[j] = make_float4(qf[0], qf[1], qf[2], qf[3]);
    scale[j] = make_float2(suf, svf);
    const bool ok = usable(qf, suf, svf, muf, of);
    double tu[3] = {1, 0, 0}, tv[3] = {0, 1, 0}, nn[3] = {0, 0, 1};
    double isu = 1.0, isv = 1.0;
    if (ok) {
        const double w = qf[0], x = qf[1], y = qf[2], z = qf[3];
        const double s = 2.0 / (w * w + x * x + y * y + z * z);
        // rotation columns of the unit quaternion (w,x,y,z) / |q|
        tu[0] = 1.0 - s * (y * y + z * z); tu[1] = s * (x * y + w * z); tu[2] = s * (x * z - w * y);
        tv[0] = s * (x * y - w * z); tv[1] = 1.0 - s * (x * x + z * z); tv[2] = s * (y * z + w * x);
        nn[0] = s * (x * z + w * y); nn[1] = s * (y * z - w * x); nn[2] = 1.0 - s * (x * x + y * y);
        isu = 1.0 / (double)suf;
        isv = 1.0 / (double)svf;
    }
    // support radius: alpha reaches alpha_min at rho^2 = 2 ln(o/alpha_min), capped at 3 sigma
    // (e^4.5 = 90.017131...: the cap is certain above 90.02 alpha_min)
    double rc2 = -1.0;
    if (ok && of > 0.f) {
        rc2 = 9.0;
        if ((double)of < 90.02 * alpha_min) {
            const double r2 = 2.0 * log((double)of / alpha_min);
            rc2 = r2 < 9.0 ? r2 : 9.0;
        }
    }
    if (!(rc2 >= 0.0)) rc2 = -1.0;
    float4* R = rec + 4 * j;
    R[0] = make_float4(muf[0], muf[1], muf[2], of);
    R[1] = make_float4((float)(tu[0] * isu), (float)(tu[1] * isu), (float)(tu[2] * isu), (float)rc2);
    R[2] = make_float4((float)(tv[0] * isv), (float)(tv[1] * isv), (float)(tv[2] * isv), __int_as_float(i));
    R[3] = make_float4((float)nn[0], (float)nn[1], (float)nn[2], 0.f);
    const float rc = rc2 >= 0.0 ? sqrtf((float)rc2) : 0.f;
    const float su = ok ? suf : 1.f, sv = ok ? svf : 1.f;
    float* B = leaf_box + 6 * j;
    for (int k = 0; k < 3; ++k) {
        const double m = ok ? (double)muf[k] : 0.0;
        const float a = su * (float)tu[k], b = sv * (float)tv[k], q = a * a + b * b;
        double e = rc * sqrtf(q);
        if (!(q < INFINITY)) {   // discs of 2^64 and more: the longer leg times a root of [1, 2]
            const float leg = fmaxf(fabsf(a), fabsf(b)), r = fminf(fabsf(a), fabsf(b)) / leg;
            e = (double)leg * (double)(rc * sqrtf(fmaf(r, r, 1.f)));
        }
        e = e * (1.0 + 1e-5) + 1e-6 * (1.0 + fabs(m));
        if (rc2 < 0.0) e = 0.0;   // never hit: a point box at the centre
        B[k] = __double2float_rd(m - e);
        B[3 + k] = __double2float_ru(m + e);
    }
}

// ---------------------------------------------------------------------------
// Radix sort of long key arrays (the wavefronts' rays; large scenes), a launch
// per step: stable LSD, 8 bits per pass. Per pass: tile histograms,
// one exclusive scan over (digit, tile), and a stable scatter that ranks keys
// inside a tile with warp match masks in (warp, chunk, lane) order.
__global__ void k_sort_hist(const uint32_t* __restrict__ keys, int64_t n, int shift, int tiles,
                            uint32_t* __restrict__ hist) {
    __shared__ uint32_t h[256];
    for (int d = threadIdx.x; d < 256; d += blockDim.x) h[d] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * kTile;
    for (int j = threadIdx.x; j < kTile; j += blockDim.x) {
        int64_t i = base + j;
        if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
    }
    __syncthreads();
    for (int d = threadIdx.x; d < 256; d += blockDim.x) hist[(int64_t)d * tiles + blockIdx.x] = h[d];
}

// Exclusive scan of `m` counters with one block of 1024 threads.
__global__ void k_scan_exclusive(uint32_t* __restrict__ a, int64_t m) {
    __shared__ uint32_t part[1024];
    int t = threadIdx.x;
    int64_t per = (m + 1023) / 1024;
    int64_t b = t * per, e = b + per < m ? b + per : m;
    uint32_t s = 0;
    for (int64_t i = b; i < e; ++i) s += a[i];
    part[t] = s;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        uint32_t v = t >= off ? part[t - off] : 0u;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    uint32_t run = part[t] - s;   // exclusive prefix of this thread's chunk
    for (int64_t i = b; i < e; ++i) {
        uint32_t v = a[i];
        a[i] = run;
        run += v;
    }
}

// Multi-block exclusive scan for long arrays: each block scans a tile of
// kScanTile words in place and records the tile total; the totals are scanned
// by k_scan_exclusive; a last pass adds each tile's offset.
constexpr int kScanThreads = 1024;
constexpr int kScanTile = 4 * kScanThreads;

__global__ void __launch_bounds__(kScanThreads) k_scan_tiles(uint32_t* __restrict__ a, int64_t m,
                                                              uint32_t* __restrict__ sums) {
    __shared__ uint32_t warp_tot[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + 4 * threadIdx.x;
    uint32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = base + k < m ? a[base + k] : 0u;
    const uint32_t t = v[0] + v[1] + v[2] + v[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = t;   // inclusive scan of the thread totals within the warp
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, off);
        if (lane >= off) inc += y;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < kScanThreads / 32 ? warp_tot[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, wi, off);
            if (lane >= off) wi += y;
        }
        if (lane < kScanThreads / 32) warp_tot[lane] = wi - w;   // exclusive warp offsets
        if (lane == kScanThreads / 32 - 1) sums[blockIdx.x] = wi;
    }
    __syncthreads();
    uint32_t run = warp_tot[warp] + inc - t;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (base + k < m) a[base + k] = run;
        run += v[k];
    }
}

__global__ void k_scan_add(uint32_t* __restrict__ a, int64_t m, const uint32_t* __restrict__ sums) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < m) a[i] += sums[i / kScanTile];
}

// Exclusive scan of m words using `sums` (ceil(m / kScanTile) words) as scratch.
void scan_long(uint32_t* a, int64_t m, uint32_t* sums, cudaStream_t st) {
    const int64_t tiles = (m + kScanTile - 1) / kScanTile;
    k_scan_tiles<<<(unsigned)tiles, kScanThreads, 0, st>>>(a, m, sums);
    k_scan_exclusive<<<1, 1024, 0, st>>>(sums, tiles);
    k_scan_add<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(a, m, sums);
}

__global__ void __launch_bounds__(kSortThreads) k_sort_scatter(
    const uint32_t* __restrict__ kin, const int32_t* __restrict__ vin, int64_t n, int shift, int tiles,
    const uint32_t* __restrict__ offs, uint32_t* __restrict__ kout, int32_t* __restrict__ vout) {
    __shared__ uint32_t wcnt[kSortWarps][256];
    __shared__ uint32_t gofs[256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < 256; d += blockDim.x) {
        gofs[d] = offs[(int64_t)d * tiles + blockIdx.x];
        for (int w = 0; w < kSortWarps; ++w) wcnt[w][d] = 0;
    }
    __syncthreads();
    const int64_t wbase = (int64_t)blockIdx.x * kTile + warp * (32 * kSortChunks);
    uint32_t key[kSortChunks];
    int32_t val[kSortChunks];
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int c = 0; c < kSortChunks; ++c) {
        int64_t i = wbase + c * 32 + lane;
        key[c] = i < n ? kin[i] : 0u;
        val[c] = i < n ? vin[i] : 0;
    }
    // phase 1: per-warp digit counts
#pragma unroll
    for (int c = 0; c < kSortChunks; ++c) {
        int64_t i = wbase + c * 32 + lane;
        uint32_t dg = i < n ? ((key[c] >> shift) & 255u) : 256u;
        unsigned peers = __match_any_sync(0xffffffffu, dg);
        if (dg < 256u && (peers & lt) == 0u) wcnt[warp][dg] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // phase 2: exclusive scan over warps per digit
    for (int d = threadIdx.x; d < 256; d += blockDim.x) {
        uint32_t run = 0;
        for (int w = 0; w < kSortWarps; ++w) {
            uint32_t v = wcnt[w][d];
            wcnt[w][d] = run;
            run += v;
        }
    }
    __syncthreads();
    // phase 3: stable scatter
#pragma unroll
    for (int c = 0; c < kSortChunks; ++c) {
        int64_t i = wbase + c * 32 + lane;
        uint32_t dg = i < n ? ((key[c] >> shift) & 255u) : 256u;
        unsigned peers = __match_any_sync(0xffffffffu, dg);
        if (dg < 256u) {
            uint32_t pos = gofs[dg] + wcnt[warp][dg] + __popc(peers & lt);
            kout[pos] = key[c];
            vout[pos] = val[c];
        }
        __syncwarp();
        if (dg < 256u && (peers & lt) == 0u) wcnt[warp][dg] += __popc(peers);
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// Features into Morton order.
__global__ void k_gather_feat(const int32_t* __restrict__ perm, int64_t n, int F, const float* __restrict__ fin,
                              float* __restrict__ fout) {
    int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= n * F) return;
    int64_t m = j / F, c = j - m * F;
    fout[j] = fin[(int64_t)perm[m] * F + c];
}

// ---------------------------------------------------------------------------
// K3 (fallback): Karras (2012) hierarchy. delta(i,j) is the common prefix length of the
// sorted keys, extended by the index bits when keys are equal.
__device__ __forceinline__ int kdelta(const uint32_t* __restrict__ k, int64_t n, int64_t i, int64_t j) {
    if (j < 0 || j >= n) return -1;
    uint32_t a = k[i], b = k[j];
    if (a == b) return 32 + __clz((uint32_t)i ^ (uint32_t)j);
    return __clz(a ^ b);
}

// With `gate` set it runs only if *gate != 0 (the clustering build's fallback).
__global__ void k_karras(const uint32_t* __restrict__ keys, int64_t n, Node* __restrict__ nodes,
                         int32_t* __restrict__ leaf_parent, int32_t* __restrict__ node_parent,
                         const uint32_t* __restrict__ gate) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n - 1 || (gate != nullptr && *gate == 0u)) return;
    int d = (kdelta(keys, n, i, i + 1) - kdelta(keys, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = kdelta(keys, n, i, i - d);
    int64_t lmax = 2;
    while (kdelta(keys, n, i, i + lmax * d) > dmin) lmax *= 2;
    int64_t l = 0;
    for (int64_t t = lmax / 2; t >= 1; t /= 2)
        if (kdelta(keys, n, i, i + (l + t) * d) > dmin) l += t;
    int64_t j = i + l * d;
    int dnode = kdelta(keys, n, i, j);
    int64_t s = 0, t = l;
    do {
        t = (t + 1) >> 1;
        if (kdelta(keys, n, i, i + (s + t) * d) > dnode) s += t;
    } while (t > 1);
    int64_t g = i + s * d + (d < 0 ? -1 : 0);
    int64_t lo = i < j ? i : j, hi = i < j ? j : i;
    int32_t left = (lo == g) ? ~(int32_t)g : (int32_t)g;
    int32_t right = (hi == g + 1) ? ~(int32_t)(g + 1) : (int32_t)(g + 1);
    nodes[i].d = make_int4(left, right, 0, 0);
    if (left < 0) leaf_parent[~left] = (int32_t)i; else node_parent[left] = (int32_t)i;
    if (right < 0) leaf_parent[~right] = (int32_t)i; else node_parent[right] = (int32_t)i;
    if (i == 0) node_parent[0] = -1;
}

// K4: bottom-up refit. The second thread to reach a node writes both child
// boxes into it and moves up; the first one stops.
__device__ __forceinline__ void child_box(const Node* nodes, const float* leaf_box, int32_t c, float b[6]) {
    if (c < 0) {
        const float* L = leaf_box + 6 * (int64_t)(~c);
        for (int k = 0; k < 6; ++k) b[k] = __ldcg(L + k);
    } else {
        const float4* p = reinterpret_cast<const float4*>(nodes + c);
        float4 a = __ldcg(p), bb = __ldcg(p + 1), cc = __ldcg(p + 2);
        b[0] = fminf(a.x, bb.z); b[1] = fminf(a.y, bb.w); b[2] = fminf(a.z, cc.x);
        b[3] = fmaxf(a.w, cc.y); b[4] = fmaxf(bb.x, cc.z); b[5] = fmaxf(bb.y, cc.w);
    }
}

__global__ void k_refit(int64_t n, const float* __restrict__ leaf_box, const int32_t* __restrict__ leaf_parent,
                        const int32_t* __restrict__ node_parent, Node* nodes, uint32_t* flags, uint32_t* status,
                        const uint32_t* __restrict__ gate) {
    int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (m >= n || (gate != nullptr && *gate == 0u)) return;
    int32_t p = leaf_parent[m];
    // a valid hierarchy is at most 62 levels deep (30 key bits + 32 index bits)
    for (int level = 0; p >= 0; ++level) {
        if (level > 128 || p >= n - 1) {
            atomicOr(status, kErrBadTree);
            return;
        }
        __threadfence();
        const uint32_t arrived = atomicAdd(&flags[p], 1u);
        if (arrived == 0u) return;
        if (arrived != 1u) {
            atomicOr(status, kErrBadTree);
            return;
        }
        int4 ch = __ldcg(&nodes[p].d);
        float b0[6], b1[6];
        child_box(nodes, leaf_box, ch.x, b0);
        child_box(nodes, leaf_box, ch.y, b1);
        nodes[p].a = make_float4(b0[0], b0[1], b0[2], b0[3]);
        nodes[p].b = make_float4(b0[4], b0[5], b1[0], b1[1]);
        nodes[p].c = make_float4(b1[2], b1[3], b1[4], b1[5]);
        p = node_parent[p];
    }
}

// Root of a one-surfel (or empty) scene: child 0 = leaf 0 (if any), child 1 absent.
__global__ void k_tiny_root(int64_t n, const float* __restrict__ leaf_box, Node* nodes) {
    float b[6] = {0, 0, 0, 0, 0, 0};
    if (n == 1)
        for (int k = 0; k < 6; ++k) b[k] = leaf_box[k];
    nodes[0].a = make_float4(b[0], b[1], b[2], b[3]);
    nodes[0].b = make_float4(b[4], b[5], 0.f, 0.f);
    nodes[0].c = make_float4(0.f, 0.f, 0.f, 0.f);
    nodes[0].d = make_int4(n == 1 ? ~0 : kNoChild, kNoChild, 0, 0);
}

// ---------------------------------------------------------------------------
// K3 (default): locally-ordered agglomerative clustering over the sorted
// leaves (PLOC, Meister and Bittner 2018). In each round every cluster looks
// at the kPlocRadius clusters on either side in Morton order and picks the
// one whose union box has the smallest surface area; mutually chosen pairs
// merge into a new internal node. Equal areas are ordered by (distance in
// the order, parity of the lower index, lower index): a strict order on
// pairs, so the best pair of a round is always mutual (every round merges)
// and runs of equal boxes pair up as (0,1), (2,3), ... Node ids follow
// (round, position), so the tree is the same on every run; the root is made
// last and gets id 0. A cluster is (id, lo, hi) with its subtree height in
// lo.w. The rounds run over the grid until at most kPlocFinishCap clusters are
// left; one block then merges the rest in shared memory. A tree higher than
// kPlocMaxHeight (possible only for contrived inputs) is replaced by the
// Karras hierarchy, whose depth the 4-wide collapse and the refit assume.
//
// Rounds shrink the clusters by a seventh, so most of the ~40 rounds of a
// large scene have fewer clusters than the chip has threads: a cluster's
// neighbours are then split over 2 to 16 threads, which shortens the round's
// chain instead of leaving SMs idle.
//
// Working memory: cluster boxes in rec_user (4 x n float4: lo and hi, two
// copies), cluster ids in keys_tmp / vals_tmp, per-tile kept lists in
// box_user (n int2), tile counts in hist.
constexpr int kPlocRadius = 16;
constexpr int kPlocFinishCap = kCoopThreads;
constexpr int kPlocMaxRounds = 64;
constexpr int kPlocMaxHeight = 60;

__device__ __forceinline__ float union_area(const float4& alo, const float4& ahi, const float4& blo,
                                            const float4& bhi) {
    const float dx = fmaxf(ahi.x, bhi.x) - fminf(alo.x, blo.x);
    const float dy = fmaxf(ahi.y, bhi.y) - fminf(alo.y, blo.y);
    const float dz = fmaxf(ahi.z, bhi.z) - fminf(alo.z, blo.z);
    const float a = dx * dy + dy * dz + dz * dx;
    return isnan(a) ? INFINITY : a;
}

// Nearest neighbour of cluster i among [i - R, i + R] of [0, count); boxes of
// cluster g at s_lo / s_hi[g - base]. 1 << lg adjacent lanes of a warp share
// the cluster and all return it (-1: none). The order of pairs as one integer:
// area (>= 0, so its bits order it), distance, then which of the two pairs at
// one distance has the even lower index, or the lower one.
__device__ __forceinline__ int64_t ploc_nearest(int64_t i, int64_t count, const float4* s_lo, const float4* s_hi,
                                                int64_t base, int lg) {
    uint64_t best = ~0ull;
    if (i >= 0 && i < count) {
        const float4 lo = s_lo[i - base], hi = s_hi[i - base];
        const int step = 1 << lg;
        for (int q = threadIdx.x & (step - 1); q < 2 * kPlocRadius; q += step) {
            const int o = q < kPlocRadius ? q - kPlocRadius : q - kPlocRadius + 1;
            const int64_t j = i + o;
            if (j < 0 || j >= count) continue;
            const uint32_t c = __float_as_uint(union_area(lo, hi, s_lo[j - base], s_hi[j - base]));
            const int d = o < 0 ? -o : o;
            // the pairs at distance d have the lower indices i - d and i
            const bool same = (d & 1) == 0;
            const bool worse = same ? o > 0 : (((o < 0 ? j : i) & 1) != 0);
            const uint64_t key = (uint64_t)c << 32 | (uint32_t)(d << 8 | (worse ? 128 : 0) | (o + kPlocRadius));
            best = key < best ? key : best;
        }
    }
    for (int x = 1; x < (1 << lg); x <<= 1) {
        const uint64_t other = __shfl_xor_sync(0xffffffffu, best, x);
        best = other < best ? other : best;
    }
    return best == ~0ull ? -1 : i + (int)(best & 127u) - kPlocRadius;
}

// Internal node k with children a, b (ids as in Node::d) and their boxes;
// returns the merged cluster's box (height in lo.w).
__device__ __forceinline__ void ploc_node(int32_t k, int32_t a, int32_t b, const float4& alo, const float4& ahi,
                                          const float4& blo, const float4& bhi, Node* nodes, int32_t* leaf_parent,
                                          int32_t* node_parent, float4& lo, float4& hi) {
    nodes[k].a = make_float4(alo.x, alo.y, alo.z, ahi.x);
    nodes[k].b = make_float4(ahi.y, ahi.z, blo.x, blo.y);
    nodes[k].c = make_float4(blo.z, bhi.x, bhi.y, bhi.z);
    nodes[k].d = make_int4(a, b, 0, 0);
    if (a < 0) leaf_parent[~a] = k; else node_parent[a] = k;
    if (b < 0) leaf_parent[~b] = k; else node_parent[b] = k;
    lo = make_float4(fminf(alo.x, blo.x), fminf(alo.y, blo.y), fminf(alo.z, blo.z), fmaxf(alo.w, blo.w) + 1.f);
    hi = make_float4(fmaxf(ahi.x, bhi.x), fmaxf(ahi.y, bhi.y), fmaxf(ahi.z, bhi.z), 0.f);
}

// Clusters per tile when 1 << lg threads share one: the tile's items are its
// clusters and kPlocRadius more on either side, whose choices decide
// mutuality; together they take the block's threads.
__device__ __forceinline__ int ploc_tile(int lg) { return (kCoopThreads >> lg) - 2 * kPlocRadius; }

struct PlocArgs {
    int64_t n;
    int rounds;
    const float* leaf_box;
    int32_t* cid[2];
    float4 *lo[2], *hi[2];
    int2* kept;
    uint32_t* tile_cnt;
    uint32_t* ctl;
    Node* nodes;
    int32_t *leaf_parent, *node_parent;
    uint32_t* status;
};

// Kept clusters and merges of tiles [0, upto) (the same for every thread).
__device__ __forceinline__ uint2 ploc_before(const uint32_t* tile_cnt, int64_t upto, uint32_t (*s_red)[32]) {
    uint32_t ko = 0u, mo = 0u;
    for (int64_t t = threadIdx.x; t < upto; t += kCoopThreads) {
        const uint2 v = __ldcg(reinterpret_cast<const uint2*>(tile_cnt) + t);
        ko += v.x;
        mo += v.y;
    }
    ko = __reduce_add_sync(0xffffffffu, ko);
    mo = __reduce_add_sync(0xffffffffu, mo);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();   // an earlier call's sums have been read
    if (lane == 0) {
        s_red[0][warp] = ko;
        s_red[1][warp] = mo;
    }
    __syncthreads();
    return make_uint2(__reduce_add_sync(0xffffffffu, s_red[0][lane]), __reduce_add_sync(0xffffffffu, s_red[1][lane]));
}

__global__ void __launch_bounds__(kCoopThreads, 1) k_ploc(PlocArgs A) {
    constexpr int H = 2 * kPlocRadius;
    constexpr int kItems = kCoopThreads + H;
    __shared__ float4 s_lo[kItems], s_hi[kItems];
    __shared__ int32_t s_nn[kCoopThreads], s_id[kCoopThreads];
    __shared__ uint32_t s_warp[33];
    __shared__ uint32_t s_red[2][32];
    const int tid = threadIdx.x;
    const int64_t n = A.n;
    uint32_t target = 0u;
    if (blockIdx.x == 0 && tid == 0) A.node_parent[0] = -1;
    for (int64_t i = blockIdx.x * (int64_t)kCoopThreads + tid; i < n; i += (int64_t)gridDim.x * kCoopThreads) {
        const float* b = A.leaf_box + 6 * i;
        A.cid[0][i] = ~(int32_t)i;
        A.lo[0][i] = make_float4(b[0], b[1], b[2], 0.f);
        A.hi[0][i] = make_float4(b[3], b[4], b[5], 0.f);
    }
    if (!grid_barrier(A.ctl + kCtlPloc, target)) {
        if (tid == 0) {
            atomicOr(A.status, kErrBadTree);
            A.ctl[kCtlFallback] = 1u;
        }
        return;
    }
    int64_t count = n, made = 0;
    int src = 0;
    for (int round = 0; round < A.rounds && count > kPlocFinishCap; ++round) {
        const int32_t* cid = A.cid[src];
        const float4 *clo = A.lo[src], *chi = A.hi[src];
        int32_t* cid2 = A.cid[src ^ 1];
        float4 *clo2 = A.lo[src ^ 1], *chi2 = A.hi[src ^ 1];
        // as many threads per cluster as still leave every tile a block of its own
        int lg = 4;
        while (lg > 0 && (int64_t)ploc_tile(lg) * gridDim.x < count) --lg;
        const int tile_size = ploc_tile(lg);
        const int64_t tiles = (count + tile_size - 1) / tile_size;
        // nearest neighbours, then each tile's kept clusters in order as
        // (source index, partner or -1) in kept[b0 ...], their number and the
        // number of merges in tile_cnt
        for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            const int64_t b0 = tile * tile_size, base = b0 - H;
            __syncthreads();
            for (int t = tid; t < tile_size + 2 * H; t += kCoopThreads) {
                const int64_t g = base + t;
                if (g >= 0 && g < count) {
                    s_lo[t] = __ldcg(clo + g);
                    s_hi[t] = __ldcg(chi + g);
                }
            }
            __syncthreads();
            const int item = tid >> lg;
            const int64_t nn = ploc_nearest(b0 - kPlocRadius + item, count, s_lo, s_hi, base, lg);
            if ((tid & ((1 << lg) - 1)) == 0) s_nn[item] = (int32_t)nn;
            __syncthreads();
            const int64_t i = b0 + tid;
            uint32_t keep = 0u, maker = 0u;
            int32_t j = -1;
            if (tid < tile_size && i < count) {
                const int32_t c = s_nn[tid + kPlocRadius];
                const bool mutual = c >= 0 && s_nn[c - (b0 - kPlocRadius)] == (int32_t)i;
                keep = (mutual && c < i) ? 0u : 1u;
                maker = (mutual && c > i) ? 1u : 0u;
                j = maker ? c : -1;
            }
            uint32_t tot;
            const uint32_t pre = block_scan(keep | (maker << 16), s_warp, &tot);
            if (keep) A.kept[b0 + (pre & 0xffffu)] = make_int2((int32_t)i, j);
            if (tid == 0) *reinterpret_cast<uint2*>(A.tile_cnt + 2 * tile) = make_uint2(tot & 0xffffu, tot >> 16);
        }
        if (!grid_barrier(A.ctl + kCtlPloc, target)) break;
        // compaction into the other buffers; merges become nodes numbered by
        // (nodes made before the round + merges before them)
        for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            const int64_t b0 = tile * tile_size;
            const uint2 before = ploc_before(A.tile_cnt, tile, s_red);
            const uint32_t nk = __ldcg(A.tile_cnt + 2 * tile);
            const int2 e = (uint32_t)tid < nk ? __ldcg(A.kept + b0 + tid) : make_int2(-1, -1);
            uint32_t tot;
            const uint32_t rank = block_scan((uint32_t)tid < nk && e.y >= 0 ? 1u : 0u, s_warp, &tot);
            if ((uint32_t)tid < nk) {
                const int64_t dst = (int64_t)before.x + tid;
                int32_t id = __ldcg(cid + e.x);
                float4 lo = __ldcg(clo + e.x), hi = __ldcg(chi + e.x);
                if (e.y >= 0) {
                    const int64_t idx = made + before.y + rank;
                    if (idx > n - 2) {
                        atomicOr(A.status, kErrBadTree);
                    } else {
                        const int32_t k = (int32_t)(n - 2 - idx);
                        float4 mlo, mhi;
                        ploc_node(k, id, __ldcg(cid + e.y), lo, hi, __ldcg(clo + e.y), __ldcg(chi + e.y), A.nodes,
                                  A.leaf_parent, A.node_parent, mlo, mhi);
                        id = k;
                        lo = mlo;
                        hi = mhi;
                    }
                }
                cid2[dst] = id;
                clo2[dst] = lo;
                chi2[dst] = hi;
            }
        }
        const uint2 all = ploc_before(A.tile_cnt, tiles, s_red);
        count = all.x;
        made += all.y;
        src ^= 1;
        if (!grid_barrier(A.ctl + kCtlPloc, target)) break;
    }
    if (blockIdx.x != 0) return;
    if (*(volatile uint32_t*)(A.ctl + kCtlPloc + 1) != 0u) {   // a barrier gave up
        if (tid == 0) {
            atomicOr(A.status, kErrBadTree);
            A.ctl[kCtlFallback] = 1u;
        }
        return;
    }
    // One block: the clusters left after the rounds (pairs of neighbours first
    // while more than kPlocFinishCap remain, which only contrived inputs
    // leave), then rounds in shared memory down to the root; a root higher
    // than kPlocMaxHeight raises the fallback flag.
    int64_t c = count;
    for (int level = 0; c > kPlocFinishCap && level < 64; ++level) {
        const int32_t* sid = A.cid[src];
        const float4 *slo = A.lo[src], *shi = A.hi[src];
        int32_t* did = A.cid[src ^ 1];
        float4 *dlo = A.lo[src ^ 1], *dhi = A.hi[src ^ 1];
        const int64_t half = c / 2;
        for (int64_t t = tid; t < (c + 1) / 2; t += kCoopThreads) {
            int32_t id = __ldcg(sid + 2 * t);
            float4 lo = __ldcg(slo + 2 * t), hi = __ldcg(shi + 2 * t);
            if (t < half) {
                const int64_t idx = made + t;
                if (idx > n - 2) {
                    atomicOr(A.status, kErrBadTree);
                    continue;
                }
                const int32_t k = (int32_t)(n - 2 - idx);
                float4 mlo, mhi;
                ploc_node(k, id, __ldcg(sid + 2 * t + 1), lo, hi, __ldcg(slo + 2 * t + 1), __ldcg(shi + 2 * t + 1),
                          A.nodes, A.leaf_parent, A.node_parent, mlo, mhi);
                id = k;
                lo = mlo;
                hi = mhi;
            }
            did[t] = id;
            dlo[t] = lo;
            dhi[t] = hi;
        }
        made += half;
        c = (c + 1) / 2;
        src ^= 1;
        __threadfence();
        __syncthreads();
    }
    if (c > kPlocFinishCap) {   // cannot happen: 64 halvings
        if (tid == 0) atomicOr(A.status, kErrBadTree);
        return;
    }
    __syncthreads();
    if (tid < c) {
        s_id[tid] = __ldcg(A.cid[src] + tid);
        s_lo[tid] = __ldcg(A.lo[src] + tid);
        s_hi[tid] = __ldcg(A.hi[src] + tid);
    }
    __syncthreads();
    for (int round = 0; c > 1 && round < kPlocFinishCap; ++round) {
        int lg = 4;
        while (lg > 0 && (kCoopThreads >> lg) < c) --lg;
        const int item = tid >> lg;
        const int64_t nn = ploc_nearest(item, c, s_lo, s_hi, 0, lg);
        if ((tid & ((1 << lg) - 1)) == 0) s_nn[item] = (int32_t)nn;
        __syncthreads();
        bool keep = false, maker = false;
        int32_t id = 0, pid = 0;
        float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo, plo = lo, phi = lo;
        if (tid < c) {
            const int32_t m = s_nn[tid];
            const bool mutual = m >= 0 && s_nn[m] == tid;
            keep = !(mutual && m < tid);
            maker = mutual && m > tid;
            id = s_id[tid];
            lo = s_lo[tid];
            hi = s_hi[tid];
            if (maker) {
                pid = s_id[m];
                plo = s_lo[m];
                phi = s_hi[m];
            }
        }
        uint32_t tot;
        const uint32_t pre = block_scan((keep ? 1u : 0u) | (maker ? 0x10000u : 0u), s_warp, &tot);
        if (maker) {
            const int64_t idx = made + (pre >> 16);
            if (idx > n - 2) {
                atomicOr(A.status, kErrBadTree);
            } else {
                const int32_t k = (int32_t)(n - 2 - idx);
                float4 mlo, mhi;
                ploc_node(k, id, pid, lo, hi, plo, phi, A.nodes, A.leaf_parent, A.node_parent, mlo, mhi);
                id = k;
                lo = mlo;
                hi = mhi;
            }
        }
        if (keep) {
            s_id[pre & 0xffffu] = id;
            s_lo[pre & 0xffffu] = lo;
            s_hi[pre & 0xffffu] = hi;
        }
        made += tot >> 16;
        c = tot & 0xffffu;
        __syncthreads();
    }
    if (tid == 0) {
        if (c != 1 || made != n - 1 || s_id[0] != 0) {
            atomicOr(A.status, kErrBadTree);
            A.ctl[kCtlFallback] = 1u;
        } else if (s_lo[0].w > (float)kPlocMaxHeight) {
            A.ctl[kCtlFallback] = 1u;
        }
    }
}

__device__ __forceinline__ void node_child(const Node& nd, int s, int32_t& c, float b[6]) {
    if (s == 0) {
        c = nd.d.x;
        b[0] = nd.a.x; b[1] = nd.a.y; b[2] = nd.a.z; b[3] = nd.a.w; b[4] = nd.b.x; b[5] = nd.b.y;
    } else {
        c = nd.d.y;
        b[0] = nd.b.z; b[1] = nd.b.w; b[2] = nd.c.x; b[3] = nd.c.y; b[4] = nd.c.z; b[5] = nd.c.w;
    }
}

// K5, greedy form: wide nodes are made top-down, level by level. A wide node
// starts from the two children of its binary node and repeatedly replaces the
// internal child of largest box surface area (one that is NaN counts as such) by
// that child's two children, until it has four (or only leaves). Its internal children get new wide
// indices, so a level's nodes are the range of indices the level before
// allocated; source[w] is the binary node behind wide node w. counters: the
// number of nodes each level allocates (zero before the launch).

__device__ __forceinline__ float box_area(const float b[6]) {
    const float dx = b[3] - b[0], dy = b[4] - b[1], dz = b[5] - b[2];
    return dx * dy + dy * dz + dz * dx;
}

// Wide root of a one-surfel (or empty) scene.
__device__ __forceinline__ void write_tiny_root(int64_t n, const float* __restrict__ leaf_box, WideNode* wide,
                                                float4* child_box) {
    WideNode o;
    const float e = INFINITY;   // empty slots: lo = +inf, hi = -inf
    float b[6] = {e, e, e, -e, -e, -e};
    if (n == 1)
        for (int k = 0; k < 6; ++k) b[k] = leaf_box[k];
    o.lox = make_float4(b[0], e, e, e);
    o.loy = make_float4(b[1], e, e, e);
    o.loz = make_float4(b[2], e, e, e);
    o.hix = make_float4(b[3], -e, -e, -e);
    o.hiy = make_float4(b[4], -e, -e, -e);
    o.hiz = make_float4(b[5], -e, -e, -e);
    o.child = make_int4(n == 1 ? ~0 : kNoChild, kNoChild, kNoChild, kNoChild);
    o.pad = make_int4(n == 1 ? 1 : 0, 0, 0, 0);
    wide[0] = o;
    child_box[0] = make_float4(b[0], b[1], b[2], __int_as_float(o.child.x));
    child_box[1] = make_float4(b[3], b[4], b[5], 0.f);
    for (int k = 1; k < 4; ++k) {
        child_box[2 * k] = make_float4(e, e, e, __int_as_float(kNoChild));
        child_box[2 * k + 1] = make_float4(-e, -e, -e, 0.f);
    }
}

__global__ void __launch_bounds__(kCoopThreads, 1) k_wide(const Node* __restrict__ nodes, int32_t* source,
                                                          uint32_t* counters, uint32_t* ctl, int64_t max_wide,
                                                          WideNode* __restrict__ wide,
                                                          float4* __restrict__ child_box, uint32_t* status) {
    uint32_t target = 0u;
    const int lane = threadIdx.x & 31;
    uint32_t begin = 0u, end = 1u;
    for (int level = 0; begin < end; ++level) {
        if (level >= kWideLevels) {
            if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, kErrBadTree);
            break;
        }
        const uint32_t stride = gridDim.x * kCoopThreads;
        // a warp's nodes lie next to each other; warps are dealt to the blocks in turn
        const uint32_t first = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32u;
        for (uint32_t i0 = begin + first; i0 < end; i0 += stride) {
            const uint32_t i = i0 + lane;
            const bool live = i < end;
            int32_t cid[4] = {kNoChild, kNoChild, kNoChild, kNoChild};
            float box[4][6] = {};
            int m = 0;
            if (live) {
                const Node nd = nodes[i == 0u ? 0 : __ldcg(source + i)];
                node_child(nd, 0, cid[0], box[0]);
                node_child(nd, 1, cid[1], box[1]);
                m = 2;
#pragma unroll
                for (int grown = 2; grown < 4; ++grown) {
                    int best = -1;
                    float ba = -1.f;
#pragma unroll
                    for (int k = 0; k < grown; ++k)
                        if (k < m && cid[k] >= 0) {
                            const float a = box_area(box[k]);
                            if (!(a <= ba)) {
                                ba = a;
                                best = k;
                            }
                        }
                    if (best < 0) break;
                    int32_t open = 0;
#pragma unroll
                    for (int k = 0; k < grown; ++k) open = k == best ? cid[k] : open;
                    const Node cn = nodes[open];
                    node_child(cn, 1, cid[grown], box[grown]);
#pragma unroll
                    for (int k = 0; k < grown; ++k)
                        if (k == best) node_child(cn, 0, cid[k], box[k]);
                    m = grown + 1;
                }
            }
            // indices of the warp's internal children: one atomic for all of them
            uint32_t inner = 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) inner += k < m && cid[k] >= 0 ? 1u : 0u;
            uint32_t inc = inner;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, inc, off);
                if (lane >= off) inc += y;
            }
            uint32_t w = 0u;
            if (lane == 31 && inc > 0u) w = atomicAdd(counters + level, inc);
            w = end + __shfl_sync(0xffffffffu, w, 31) + inc - inner;
            if (!live) continue;
            int32_t out[4] = {kNoChild, kNoChild, kNoChild, kNoChild};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (k >= m) {
                    // empty slots get an empty box (lo = +inf, hi = -inf): no ray's slab
                    // interval meets it, so the walks need no test of the child id
                    for (int j = 0; j < 3; ++j) {
                        box[k][j] = INFINITY;
                        box[k][3 + j] = -INFINITY;
                    }
                } else if (cid[k] < 0) {
                    out[k] = cid[k];
                } else if ((int64_t)w >= max_wide) {
                    atomicOr(status, kErrBadTree);
                } else {
                    source[w] = cid[k];
                    out[k] = (int32_t)w++;
                }
            }
            WideNode o;
            o.lox = make_float4(box[0][0], box[1][0], box[2][0], box[3][0]);
            o.loy = make_float4(box[0][1], box[1][1], box[2][1], box[3][1]);
            o.loz = make_float4(box[0][2], box[1][2], box[2][2], box[3][2]);
            o.hix = make_float4(box[0][3], box[1][3], box[2][3], box[3][3]);
            o.hiy = make_float4(box[0][4], box[1][4], box[2][4], box[3][4]);
            o.hiz = make_float4(box[0][5], box[1][5], box[2][5], box[3][5]);
            o.child = make_int4(out[0], out[1], out[2], out[3]);
            o.pad = make_int4(m, 0, 0, 0);
            wide[i] = o;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                child_box[8 * (int64_t)i + 2 * k] = make_float4(box[k][0], box[k][1], box[k][2], __int_as_float(out[k]));
                child_box[8 * (int64_t)i + 2 * k + 1] = make_float4(box[k][3], box[k][4], box[k][5], 0.f);
            }
        }
        if (!grid_barrier(ctl + kCtlWide, target)) {
            // the levels below were not made: nothing may be walked into (thread 0 of block 0 alone writes the root)
            if (threadIdx.x == 0) {
                atomicOr(status, kErrBadTree);
                if (blockIdx.x == 0) {
                    write_tiny_root(0, nullptr, wide, child_box);
                    counters[kWideLevels] = 1u;
                }
            }
            return;
        }
        begin = end;
        const int64_t now = (int64_t)end + __ldcg(counters + level);
        end = (uint32_t)(now < max_wide ? now : max_wide);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) counters[kWideLevels] = end;
}

__global__ void k_wide_tiny(int64_t n, const float* __restrict__ leaf_box, WideNode* wide, float4* child_box) {
    write_tiny_root(n, leaf_box, wide, child_box);
}

template <class T>
cudaError_t dalloc(T** p, size_t count, int64_t& bytes) {
    size_t b = sizeof(T) * (count > 0 ? count : 1);
    bytes += (int64_t)b;
    return cudaMalloc(reinterpret_cast<void**>(p), b);
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

// Keys that k_order sorts itself.
constexpr int64_t kOrderMaxKeys = int64_t(1) << 22;

// Words of a build's hist array: the sort's digit counts (a row per block of
// k_order, or sort_pairs' tiles), later the clustering's two counts per tile
// (its smallest tiles have ploc_tile(4) = 32 clusters, but only while every
// tile has a block; larger scenes have tiles of 992).
int64_t build_hist_words(int64_t n) {
    const int64_t order = 256 * kCoopBlocks, large = n > kOrderMaxKeys ? sort_hist_words(n) : 0;
    const int64_t tiles = 2 * (n / (kCoopThreads - 2 * kPlocRadius) + 1 + kCoopBlocks);
    return order > large ? (order > tiles ? order : tiles) : (large > tiles ? large : tiles);
}

}  // namespace

void free_scene(irgs_scene sc) {
    if (!sc) return;
    void* ptrs[] = {sc->nodes, sc->rec, sc->feat, sc->q_raw, sc->scale, sc->leaf_box, sc->keys,
                    sc->perm, sc->inv_perm, sc->status, sc->rec_user, sc->box_user, sc->keys_tmp, sc->vals_tmp,
                    sc->hist, sc->bounds, sc->leaf_parent, sc->node_parent, sc->refit_flag, sc->wide, sc->child_box,
                    sc->wide_source, sc->wide_counters};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    delete sc;
}

// Rounds of the clustering build for n leaves: about four per halving of the
// cluster count down to kPlocFinishCap, plus margin (rounds past that point
// return at once).
static int ploc_rounds(int64_t n) {
    int r = 8;
    for (int64_t c = n; c > kPlocFinishCap; c = (c + 1) / 2) r += 4;
    return r < kPlocMaxRounds ? r : kPlocMaxRounds;
}

// A cooperative launch of at most kCoopBlocks blocks, no more than are needed
// for `threads` threads' worth of work and than the device can hold at once.
template <class... Args>
static cudaError_t launch_coop(void (*kernel)(Args...), int device, int64_t threads, cudaStream_t st, Args... args) {
    int sms = 0, per_sm = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kCoopThreads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1 || sms < 1) return cudaErrorLaunchOutOfResources;
    int64_t blocks = (threads + kCoopThreads - 1) / kCoopThreads;
    if (blocks > sms) blocks = sms;
    if (blocks > kCoopBlocks) blocks = kCoopBlocks;
    if (blocks < 1) blocks = 1;
    void* argv[] = {&args...};
    e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kernel), dim3((unsigned)blocks), dim3(kCoopThreads),
                                    argv, 0, st);
    count_launches(1);
    return e;
}

// Enqueue the clustering build of the binary hierarchy (n > 1) over the
// sorted leaf boxes; ctl[kCtlFallback] is then nonzero when the Karras
// hierarchy has to replace it.
static cudaError_t enqueue_ploc(irgs_scene sc, cudaStream_t st) {
    const int64_t n = sc->n;
    PlocArgs A;
    A.n = n;
    A.rounds = ploc_rounds(n);
    A.leaf_box = sc->leaf_box;
    A.cid[0] = reinterpret_cast<int32_t*>(sc->keys_tmp);
    A.cid[1] = sc->vals_tmp;
    A.lo[0] = sc->rec_user;
    A.hi[0] = sc->rec_user + n;
    A.lo[1] = sc->rec_user + 2 * n;
    A.hi[1] = sc->rec_user + 3 * n;
    A.kept = reinterpret_cast<int2*>(sc->box_user);
    A.tile_cnt = sc->hist;
    A.ctl = sc->bounds;
    A.nodes = sc->nodes;
    A.leaf_parent = sc->leaf_parent;
    A.node_parent = sc->node_parent;
    A.status = sc->status;
    // a few threads per cluster still find work in the first round
    return launch_coop<PlocArgs>(k_ploc, sc->device, n > kPlocFinishCap ? 16 * n : 1, st, A);
}

// Enqueue the greedy 4-wide collapse of the scene's binary hierarchy (n > 1).
static cudaError_t enqueue_wide(irgs_scene sc, cudaStream_t st) {
    const cudaError_t e = cudaMemsetAsync(sc->wide_counters, 0, sizeof(uint32_t) * (kWideLevels + 1), st);
    if (e != cudaSuccess) return e;
    return launch_coop<const Node*, int32_t*, uint32_t*, uint32_t*, int64_t, WideNode*, float4*, uint32_t*>(
        k_wide, sc->device, sc->n, st, sc->nodes, sc->wide_source, sc->wide_counters, sc->bounds, sc->max_wide,
        sc->wide, sc->child_box, sc->status);
}

// Morton order of the surfels: keys and perm.
static cudaError_t enqueue_order(irgs_scene sc, const irgs_surfels* s, cudaStream_t st) {
    const int64_t n = sc->n;
    // beyond a few keys per thread the launches of sort_pairs cost less than a piece's serial steps
    const int passes = n <= kOrderMaxKeys ? 4 : 0;
    cudaError_t e = launch_coop<const float*, const float*, const float*, const float*, int64_t, uint32_t*, uint32_t*,
                                int32_t*, uint32_t*, int32_t*, uint32_t*, int, uint32_t*>(
        k_order, sc->device, n, st, s->means, s->quats, s->scales, s->opacity, n, sc->bounds, sc->keys, sc->perm,
        sc->keys_tmp, sc->vals_tmp, sc->hist, passes, sc->status);
    if (e == cudaSuccess && passes == 0)
        e = sort_pairs(sc->keys, sc->perm, sc->keys_tmp, sc->vals_tmp, sc->hist, n, st);
    return e;
}

// Records, boxes and features in the Morton order of sc->perm.
static cudaError_t enqueue_pack(irgs_scene sc, const irgs_surfels* s, cudaStream_t st) {
    const int64_t n = sc->n;
    const int32_t F = sc->F;
    const int T = 256;
    // (a refit keeps the last build's order and finds the flag zero)
    k_pack<<<blocks_for(n, T), T, 0, st>>>(sc->perm, sc->keys, sc->bounds + kCtlOrder + 1, s->means, s->quats, s->scales, s->opacity, n,
                                           (double)sc->alpha_min, sc->rec, sc->leaf_box, sc->q_raw, sc->scale,
                                           sc->inv_perm);
    if (F > 0) k_gather_feat<<<blocks_for(n * F, T), T, 0, st>>>(sc->perm, n, F, s->features, sc->feat);
    count_launches(1 + (F > 0));
    return cudaGetLastError();
}

// Centre bounds as no centre leaves them, barriers and flags zero.
static cudaError_t enqueue_control(irgs_scene sc, cudaStream_t st) {
    // mins start at the largest ordered value, maxes at the smallest
    cudaError_t e = cudaMemsetAsync(sc->bounds, 0xff, 3 * sizeof(uint32_t), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(sc->bounds + 3, 0x00, (kCtlWords - 3) * sizeof(uint32_t), st);
    return e;
}

// Enqueue the whole build (K1-K5) for surfels `s` into the scene's buffers.
static irgs_status enqueue_build(irgs_scene sc, const irgs_surfels* s, cudaStream_t st) {
    const int64_t n = sc->n;
    const int64_t nn = n > 1 ? n - 1 : 1;
    cudaError_t e = cudaSuccess;
    auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    A(cudaMemsetAsync(sc->nodes, 0, sizeof(Node) * nn, st));
    A(cudaMemsetAsync(sc->refit_flag, 0, sizeof(uint32_t) * nn, st));
    A(enqueue_control(sc, st));
    if (n > 0 && e == cudaSuccess) {
        const int T = 256;
        A(enqueue_order(sc, s, st));
        A(enqueue_pack(sc, s, st));
        if (n > 1) {
            // the radix tree runs when asked for, else only if the clustering raises its fallback flag
            const uint32_t* gate = nullptr;
            if (!(sc->build_flags & IRGS_BUILD_RADIX_TREE)) {
                A(enqueue_ploc(sc, st));
                gate = sc->bounds + kCtlFallback;
            }
            k_karras<<<blocks_for(n - 1, T), T, 0, st>>>(sc->keys, n, sc->nodes, sc->leaf_parent, sc->node_parent,
                                                         gate);
            k_refit<<<blocks_for(n, T), T, 0, st>>>(n, sc->leaf_box, sc->leaf_parent, sc->node_parent, sc->nodes,
                                                    sc->refit_flag, sc->status, gate);
            count_launches(2);
        }
    }
    if (n <= 1) {
        k_tiny_root<<<1, 1, 0, st>>>(n, sc->leaf_box, sc->nodes);
        count_launches(1);
    }
    if (sc->wide != nullptr) {
        if (n > 1) {
            A(enqueue_wide(sc, st));
        } else {
            k_wide_tiny<<<1, 1, 0, st>>>(n, sc->leaf_box, sc->wide, sc->child_box);
            count_launches(1);
        }
    }
    A(cudaGetLastError());
    return e == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

int64_t sort_hist_words(int64_t n) {
    const int64_t tiles = (n + kTile - 1) / kTile;
    const int64_t words = 256 * (tiles > 0 ? tiles : 1);
    return words + (words + kScanTile - 1) / kScanTile;   // digit counts, then the scan's tile sums
}

cudaError_t sort_pairs(uint32_t* keys, int32_t* vals, uint32_t* keys_tmp, int32_t* vals_tmp, uint32_t* hist,
                       int64_t n, cudaStream_t st, int key_bits) {
    if (n <= 0) return cudaSuccess;
    const int64_t tiles = (n + kTile - 1) / kTile;
    // an even number of 8-bit passes, so that the result ends in keys / vals
    const int passes = ((key_bits + 15) / 16) * 2;
    uint32_t* ka = keys; int32_t* va = vals;
    uint32_t* kb = keys_tmp; int32_t* vb = vals_tmp;
    for (int shift = 0; shift < 8 * passes; shift += 8) {
        k_sort_hist<<<(unsigned)tiles, 256, 0, st>>>(ka, n, shift, (int)tiles, hist);
        scan_long(hist, 256 * tiles, hist + 256 * tiles, st);
        k_sort_scatter<<<(unsigned)tiles, kSortThreads, 0, st>>>(ka, va, n, shift, (int)tiles, hist, kb, vb);
        uint32_t* tk = ka; ka = kb; kb = tk;
        int32_t* tv = va; va = vb; vb = tv;
    }
    count_launches(5 * passes);
    return cudaGetLastError();
}

int64_t scan_long_words(int64_t m) { return (m + kScanTile - 1) / kScanTile + 1; }

namespace {
// pos[0..m] = exclusive prefix of 0/1 flags: list[pos[j]] = j for every
// flagged j, *count = pos[m].
__global__ void k_flag_list(const uint32_t* __restrict__ pos, int64_t m, int32_t* __restrict__ list,
                            uint32_t* __restrict__ count) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j == 0) *count = pos[m];
    if (j < m && pos[j + 1] != pos[j]) list[pos[j]] = (int32_t)j;
}
}  // namespace

cudaError_t flags_to_list(uint32_t* flags, int64_t m, uint32_t* sums, int32_t* list, uint32_t* count,
                          cudaStream_t st) {
    cudaError_t e = scan_exclusive_long(flags, m + 1, sums, st);
    if (e != cudaSuccess) return e;
    k_flag_list<<<(unsigned)((m + 255) / 256 > 0 ? (m + 255) / 256 : 1), 256, 0, st>>>(flags, m, list, count);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t scan_exclusive_long(uint32_t* a, int64_t m, uint32_t* sums, cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    scan_long(a, m, sums, st);
    count_launches(3);
    return cudaGetLastError();
}

irgs_status build_scene_impl(const irgs_surfels* s, float alpha_min, uint32_t build_flags, cudaStream_t st,
                             irgs_scene* out) {
    const int64_t n = s->n;
    const int32_t F = s->num_features;
    irgs_scene sc = new (std::nothrow) irgs_scene_s();
    if (!sc) return IRGS_ERR_OOM;
    cudaGetDevice(&sc->device);
    sc->n = n;
    sc->F = F;
    sc->alpha_min = alpha_min;
    sc->build_flags = build_flags;
    const int64_t nn = n > 1 ? n - 1 : 1;
    int64_t& B = sc->bytes;
    cudaError_t e = cudaSuccess;
    auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    A(dalloc(&sc->nodes, nn, B));
    A(dalloc(&sc->rec, 4 * n, B));
    A(dalloc(&sc->feat, (size_t)n * F, B));
    A(dalloc(&sc->q_raw, n, B));
    A(dalloc(&sc->scale, n, B));
    A(dalloc(&sc->leaf_box, 6 * n, B));
    A(dalloc(&sc->keys, n, B));
    A(dalloc(&sc->perm, n, B));
    A(dalloc(&sc->inv_perm, n, B));
    A(dalloc(&sc->status, 1, B));
    A(dalloc(&sc->rec_user, 4 * n, B));
    A(dalloc(&sc->box_user, 6 * n, B));
    A(dalloc(&sc->keys_tmp, n, B));
    A(dalloc(&sc->vals_tmp, n, B));
    A(dalloc(&sc->hist, build_hist_words(n), B));
    A(dalloc(&sc->bounds, kCtlWords, B));
    A(dalloc(&sc->leaf_parent, n, B));
    A(dalloc(&sc->node_parent, nn, B));
    A(dalloc(&sc->refit_flag, nn, B));
    // Every wide node has four children, or two or three leaves: with p of the
    // latter among W, 4 (W - p) + 2 p <= W - 1 + n, and p <= n / 2.
    sc->max_wide = n > 1 ? (2 * n - 1) / 3 : 1;
    A(dalloc(&sc->wide, sc->max_wide, B));
    A(dalloc(&sc->child_box, 8 * sc->max_wide, B));
    A(dalloc(&sc->wide_source, sc->max_wide, B));
    A(dalloc(&sc->wide_counters, kWideLevels + 1, B));
    if (e != cudaSuccess) {
        cudaGetLastError();
        free_scene(sc);
        return e == cudaErrorMemoryAllocation ? IRGS_ERR_OOM : IRGS_ERR_CUDA;
    }
    if (cudaMemsetAsync(sc->status, 0, sizeof(uint32_t), st) != cudaSuccess) {
        free_scene(sc);
        return IRGS_ERR_CUDA;
    }
    irgs_status r = enqueue_build(sc, s, st);
    if (r != IRGS_OK) {
        cudaStreamSynchronize(st);
        free_scene(sc);
        return r;
    }
    *out = sc;
    return IRGS_OK;
}

irgs_status update_scene_impl(irgs_scene sc, const irgs_surfels* s, cudaStream_t st) {
    return enqueue_build(sc, s, st);
}

// Refit: new surfel values in the Morton order and hierarchy of the last
// build. Records, leaf boxes and features are recomputed and gathered with
// the kept permutation, the binary boxes are refitted bottom-up and the
// 4-wide nodes made from them again (the collapse opens children by box area,
// so their layout follows the new boxes). Every box still bounds its subtree, so traces stay exact; only
// the quality of the tree can degrade as surfels move.
irgs_status refit_scene_impl(irgs_scene sc, const irgs_surfels* s, cudaStream_t st) {
    const int64_t n = sc->n;
    const int64_t nn = n > 1 ? n - 1 : 1;
    cudaError_t e = cudaSuccess;
    auto A = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    A(cudaMemsetAsync(sc->refit_flag, 0, sizeof(uint32_t) * nn, st));
    A(enqueue_control(sc, st));
    const int T = 256;
    if (n > 0 && e == cudaSuccess) {
        // the centre bounds follow the new values, the order does not
        k_bounds<<<blocks_for(n, T), T, 0, st>>>(s->means, s->quats, s->scales, s->opacity, n, sc->bounds);
        A(enqueue_pack(sc, s, st));
        if (n > 1)
            k_refit<<<blocks_for(n, T), T, 0, st>>>(n, sc->leaf_box, sc->leaf_parent, sc->node_parent, sc->nodes,
                                                    sc->refit_flag, sc->status, nullptr);
        count_launches(n > 1 ? 2 : 1);
    }
    if (n > 1) {
        A(enqueue_wide(sc, st));
    } else {
        k_tiny_root<<<1, 1, 0, st>>>(n, sc->leaf_box, sc->nodes);
        k_wide_tiny<<<1, 1, 0, st>>>(n, sc->leaf_box, sc->wide, sc->child_box);
        count_launches(2);
    }
    A(cudaGetLastError());
    return e == cudaSuccess ? IRGS_OK : IRGS_ERR_CUDA;
}

// ---------------------------------------------------------------------------
// Allocation-free build: all working memory of the build comes from one
// file-scope device array; the caller provides the outputs.
namespace {

constexpr int64_t kNoallocMax = IRGS_NOALLOC_MAX_SURFELS;
constexpr size_t kAlign = 256;
constexpr size_t align_up(size_t b) { return (b + kAlign - 1) / kAlign * kAlign; }
constexpr size_t kNoallocBytes =
    align_up(sizeof(float4) * 4 * kNoallocMax) * 2 +      // records, the clusters' boxes
    align_up(sizeof(float) * 6 * kNoallocMax) +           // the clusters' kept lists
    align_up(sizeof(float4) * kNoallocMax) +              // raw quaternions
    align_up(sizeof(float2) * kNoallocMax) +              // scales
    align_up(sizeof(uint32_t) * kNoallocMax) * 2 +        // sort ping-pong keys / values
    align_up(sizeof(int32_t) * kNoallocMax) * 3 +         // leaf parents, node parents, refit flags
    align_up(sizeof(uint32_t) * 256 * kCoopBlocks) +      // digit counts
    align_up(sizeof(uint32_t) * kCtlWords) + align_up(sizeof(uint32_t));   // bounds and control words, status word

__device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

std::mutex g_noalloc_mutex;
void* g_noalloc_ptr[256] = {};

// Device address of the scratch array on the current device (looked up once
// per device). Returns nullptr if the lookup fails.
void* noalloc_scratch(int device) {
    if (device < 0 || device >= 256) return nullptr;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (g_noalloc_ptr[device] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        g_noalloc_ptr[device] = p;
    }
    return g_noalloc_ptr[device];
}

}  // namespace

// The scratch array's carve-out for one allocation-free build: the scene
// view's work buffers and its device status word. Returns the bytes used.
size_t noalloc_carve(unsigned char* base, irgs_scene_s& sc) {
    const int64_t M = kNoallocMax;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        unsigned char* p = base + off;
        off += align_up(bytes);
        return p;
    };
    sc.rec_user = reinterpret_cast<float4*>(take(sizeof(float4) * 4 * M));
    sc.rec = reinterpret_cast<float4*>(take(sizeof(float4) * 4 * M));
    sc.box_user = reinterpret_cast<float*>(take(sizeof(float) * 6 * M));
    sc.q_raw = reinterpret_cast<float4*>(take(sizeof(float4) * M));
    sc.scale = reinterpret_cast<float2*>(take(sizeof(float2) * M));
    sc.keys_tmp = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * M));
    sc.vals_tmp = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * M));
    sc.leaf_parent = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * M));
    sc.node_parent = reinterpret_cast<int32_t*>(take(sizeof(int32_t) * M));
    sc.refit_flag = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * M));
    sc.hist = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * 256 * kCoopBlocks));
    sc.bounds = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * kCtlWords));
    sc.status = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t)));
    return off;
}

irgs_status build_lbvh_noalloc_impl(const irgs_surfels* s, float alpha_min, int32_t* perm, uint32_t* keys,
                                    float* nodes, float* leaf_boxes, cudaStream_t st) {
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return IRGS_ERR_CUDA;
    unsigned char* base = static_cast<unsigned char*>(noalloc_scratch(device));
    if (base == nullptr) return IRGS_ERR_CUDA;
    irgs_scene_s sc;   // a view onto caller buffers and the scratch array
    sc.device = device;
    sc.n = s->n;
    sc.F = 0;
    sc.alpha_min = alpha_min;
    const size_t used = noalloc_carve(base, sc);
    sc.keys = keys;
    sc.perm = perm;
    sc.nodes = reinterpret_cast<Node*>(nodes);
    sc.leaf_box = leaf_boxes;
    if (used > kNoallocBytes) return IRGS_ERR_CUDA;   // carve-out mismatch (cannot happen)
    if (cudaMemsetAsync(sc.status, 0, sizeof(uint32_t), st) != cudaSuccess) return IRGS_ERR_CUDA;
    return enqueue_build(&sc, s, st);
}

irgs_status lbvh_noalloc_status_impl(cudaStream_t st, uint32_t* bits) {
    int device = 0;
    if (cudaGetDevice(&device) != cudaSuccess) return IRGS_ERR_CUDA;
    unsigned char* base = static_cast<unsigned char*>(noalloc_scratch(device));
    if (base == nullptr) return IRGS_ERR_CUDA;
    irgs_scene_s sc;
    noalloc_carve(base, sc);
    uint32_t h = 0;
    if (cudaStreamSynchronize(st) != cudaSuccess) return IRGS_ERR_CUDA;
    if (cudaMemcpy(&h, sc.status, sizeof(uint32_t), cudaMemcpyDeviceToHost) != cudaSuccess) return IRGS_ERR_CUDA;
    if (bits) *bits = h;
    return h == 0u ? IRGS_OK : IRGS_ERR_DEVICE;
}

}  // namespace irgs
