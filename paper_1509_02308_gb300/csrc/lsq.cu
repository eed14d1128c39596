// S7's judge: the exhaustive least-squares matcher.
//
// Per trace: keep the points at or below its 507th smallest value (drops the
// 5 largest of 512, the spike allowance); mask m_p.  For candidate g with
// miss rates r_gp the best affine fit y ~ alpha + beta r_g over kept points
// leaves residual Var_y - Cov^2 / Var_r (Var_y when Var_r is 0 or the slope is
// not positive).  The smallest residual wins; equal residuals go to the lower
// candidate index.
//
// Sums over 512 points for every trace x candidate pair are a contraction, but
// the answer is defined by FP32 sums in point order (dyr, dr, drr below), and
// two candidates' residuals may be closer than another order's rounding.  So
// the work is in two parts:
//   1. estimates of every pair's residual on the tcgen05 tensor cores, from
//      centred rows split into BF16 high and low parts (three products for the
//      covariance; the dropped points' share of the row's sum and square sum),
//      accurate to about 1e-5 of Var_y.  Each trace lists the candidates whose
//      estimate is within a margin of its best one: 1e-3 Var_y, far above both
//      the estimates' error and the FP32 sums', plus 2^-14 of the trace's
//      square sum, which takes over when Var_y is small against it (then FP32
//      sums cancel, the list overflows and every candidate is evaluated);
//   2. the listed candidates' residuals by the FP32 sums themselves, a lane
//      each, and the smallest of them.  Rows that are nearly constant (their
//      variance below 1/64 of their mean square), whose FP32 variance cancels,
//      are evaluated for every trace.
// Evaluating every pair on the CUDA cores (three FP32 accumulators, 64 x 64
// tiles) took 1388 us for 8192 traces x 1308 candidates, 80 % of it FP32 issue
// and shared-memory loads; the two parts take 233 us.  What bounds them:
// the operand tiles' L2 reads (0.9 MB per 128 x 128 tile).
#include <algorithm>

#include <cuda_bf16.h>

#include "pchase_internal.cuh"
#include "tc_common.cuh"
#include "tma_host.cuh"

namespace pchase {

namespace {

constexpr int kPoints = 512;
constexpr int kKeep = kPoints - 5;
constexpr uint32_t kLsqChunk = 2048;   // candidates converted at a time
constexpr uint32_t kLsqList = 32;      // listed candidates of a trace
constexpr uint32_t kLsqIll = 4096;     // nearly constant rows
constexpr int kYCols = 3 * kPoints;    // a trace's operand row: high, low, dropped mask
constexpr int kRCols = 4 * kPoints;    // a candidate's: high, low, square's high, low

struct RowStats {
    float thr, cnt, sy, syy;  // kept: v <= thr; their count, sum and square sum
    float mean, var;          // of the kept points, from centred sums
    float margin, pad;
};
struct Listed {
    float res;
    uint32_t g;
};
struct Flags {
    uint32_t all;    // 1: evaluate every candidate (a wait gave up, too many flat rows)
    uint32_t n_ill;  // nearly constant rows
};

// The workspace: per trace operands, statistics, best estimate, list; then a
// chunk of candidates.
struct LsqWork {
    __nv_bfloat16 *Y, *R;
    RowStats *stats;
    uint32_t *best, *count, *ill;
    Listed *list;
    float2 *cand;  // {sum, square sum} of the centred row
    Flags *flags;
    size_t bytes;
    LsqWork(void *base, size_t n) {
        uint8_t *p = static_cast<uint8_t *>(base);
        size_t o = 0;
        auto take = [&](size_t b) {
            uint8_t *q = p + o;
            o = (o + b + 255) & ~size_t(255);
            return q;
        };
        Y = reinterpret_cast<__nv_bfloat16 *>(take(n * kYCols * 2));
        stats = reinterpret_cast<RowStats *>(take(n * sizeof(RowStats)));
        best = reinterpret_cast<uint32_t *>(take(n * 4));
        count = reinterpret_cast<uint32_t *>(take(n * 4));
        list = reinterpret_cast<Listed *>(take(n * kLsqList * sizeof(Listed)));
        R = reinterpret_cast<__nv_bfloat16 *>(take((size_t)kLsqChunk * kRCols * 2));
        cand = reinterpret_cast<float2 *>(take((size_t)kLsqChunk * sizeof(float2)));
        ill = reinterpret_cast<uint32_t *>(take(kLsqIll * 4));
        flags = reinterpret_cast<Flags *>(take(sizeof(Flags)));
        bytes = o;
    }
};

__device__ __forceinline__ uint32_t order_key(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// One warp per trace: the 507th smallest value (the sixth largest: five times
// the largest of what is left is taken out), statistics, operand row.  Lane l
// holds points 4 l + 128 q .. + 3.
__global__ void __launch_bounds__(256) lsq_rows_kernel(const float *__restrict__ y, uint32_t n,
                                                       const uint32_t *n_dev, LsqWork w) {
    if (n_dev && *n_dev < n) n = *n_dev;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
        float v[16];
        const float *row = y + (size_t)i * kPoints;
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) v[4 * q + e] = row[4 * lane + 128 * q + e];
        uint32_t out = 0;  // values taken out
        uint32_t kth = 0;
        for (int round = 0; round < kPoints - kKeep + 1; ++round) {
            uint32_t top = 0, at = 0;
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const uint32_t k = order_key(v[e]);
                if (!((out >> e) & 1u) && k >= top) {
                    top = k;
                    at = (uint32_t)e;
                }
            }
            kth = __reduce_max_sync(kFull, top);
            const uint32_t who = __ballot_sync(kFull, top == kth);
            if (lane == (uint32_t)(__ffs(who) - 1)) out |= 1u << at;
        }
        const float thr = key_value(kth);
        float c = 0.0f, sy = 0.0f, syy = 0.0f;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const float m = v[e] <= thr ? 1.0f : 0.0f;
            c += m;
            sy += m * v[e];
            syy += m * v[e] * v[e];
        }
        c = warp_sum(c);
        sy = warp_sum(sy);
        syy = warp_sum(syy);
        const float mean = sy / c;
        float var = 0.0f;
        __nv_bfloat16 *o = w.Y + (size_t)i * kYCols;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            __nv_bfloat16 hi[4], lo[4], d[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool kept = v[4 * q + e] <= thr;
                const float z = kept ? v[4 * q + e] - mean : 0.0f;
                var += z * z;
                hi[e] = __float2bfloat16(z);
                lo[e] = __float2bfloat16(z - __bfloat162float(hi[e]));
                d[e] = __float2bfloat16(kept ? 0.0f : 1.0f);
            }
            const uint32_t p = 4 * lane + 128 * q;
            *reinterpret_cast<uint2 *>(o + p) = *reinterpret_cast<const uint2 *>(hi);
            *reinterpret_cast<uint2 *>(o + kPoints + p) = *reinterpret_cast<const uint2 *>(lo);
            *reinterpret_cast<uint2 *>(o + 2 * kPoints + p) = *reinterpret_cast<const uint2 *>(d);
        }
        var = warp_sum(var);
        if (lane == 0) {
            RowStats s;
            s.thr = thr;
            s.cnt = c;
            s.sy = sy;
            s.syy = syy;
            s.mean = mean;
            s.var = var;
            s.margin = 1e-3f * var + syy * (1.0f / 16384.0f);
            s.pad = 0.0f;
            w.stats[i] = s;
            w.best[i] = 0x7F800000u;
            w.count[i] = 0;
        }
    }
}

// One warp per candidate of the chunk: centred row, split, and its sums.
__global__ void __launch_bounds__(256) lsq_rates_kernel(const float *__restrict__ rates, uint32_t g0,
                                                        uint32_t ng, LsqWork w) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (k >= ng) return;
    const float *row = rates + (size_t)(g0 + k) * kPoints;
    float v[16], sum = 0.0f, raw = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float x = row[4 * lane + 128 * q + e];
            v[4 * q + e] = x;
            sum += x;
            raw += x * x;
        }
    const float mean = warp_sum(sum) * (1.0f / kPoints);
    raw = warp_sum(raw);
    float s1 = 0.0f, s2 = 0.0f;
    __nv_bfloat16 *o = w.R + (size_t)k * kRCols;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        __nv_bfloat16 t[4][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float z = v[4 * q + e] - mean, zz = z * z;
            s1 += z;
            s2 += zz;
            t[0][e] = __float2bfloat16(z);
            t[1][e] = __float2bfloat16(z - __bfloat162float(t[0][e]));
            t[2][e] = __float2bfloat16(zz);
            t[3][e] = __float2bfloat16(zz - __bfloat162float(t[2][e]));
        }
#pragma unroll
        for (int h = 0; h < 4; ++h)
            *reinterpret_cast<uint2 *>(o + h * kPoints + 4 * lane + 128 * q) =
                *reinterpret_cast<const uint2 *>(t[h]);
    }
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if (lane == 0) {
        w.cand[k] = make_float2(s1, s2);
        // (also rows whose sums are not finite)
        if (!(64.0f * s2 >= raw)) {
            const uint32_t at = atomicAdd(&w.flags->n_ill, 1u);
            if (at < kLsqIll) w.ill[at] = g0 + k;
            else w.flags->all = 1u;
        }
    }
}

// Estimates: persistent CTAs over 128 x 128 tiles (traces x candidates), the
// three sums side by side in TMEM (128 columns each).  A K block of 64 points
// is seven TMA tiles (112 KB) in one of two stages and 24 MMAs; one thread
// issues both.  Epilogue: a thread per trace and column half, first its best
// estimate, then the candidates to list.
constexpr uint32_t kTile = 128 * 128;  // bytes of a 128 x 64 BF16 tile
constexpr uint32_t kLsqStage = 7 * kTile;
constexpr uint32_t kLsqSmem = 1024 + 2 * kLsqStage + 128 * 8 + 64;
// M 128, N 128, BF16 operands, FP32 sums
constexpr uint32_t kIdescLsq = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

__global__ void __launch_bounds__(256)
    lsq_estimate_kernel(const __grid_constant__ CUtensorMap ymap, const __grid_constant__ CUtensorMap rmap,
                        uint32_t n, const uint32_t *n_dev, uint32_t g0, uint32_t ng, LsqWork w) {
    extern __shared__ uint8_t dsm[];
    const uint32_t raw = smem_u32(dsm);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *const gbase = dsm + (base - raw);
    float2 *const cand = reinterpret_cast<float2 *>(gbase + 2 * kLsqStage);
    // mbarriers: stage loaded [2], stage's MMAs done [2]
    const uint32_t full0 = base + 2 * kLsqStage + 128 * 8, done0 = full0 + 16u;
    uint32_t *const tslot = reinterpret_cast<uint32_t *>(gbase + 2 * kLsqStage + 128 * 8 + 32);
    volatile uint32_t *const abort_flag = tslot + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (n_dev && *n_dev < n) n = *n_dev;
    const uint32_t gt = (ng + 127u) / 128u, tiles = (n + 127u) / 128u * gt;
    constexpr int kBlocks = kPoints / 64;
    if (tid == 0) {
        for (int q = 0; q < 4; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8 * q) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *abort_flag = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tslot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    // K blocks are numbered through all of this CTA's tiles: block b uses stage
    // b mod 2, whose barriers it completes for the (b / 2)-th time
    auto load = [&](uint32_t tile, int kb, uint32_t b) {
        const uint32_t q = b & 1u, st = base + q * kLsqStage, bar = full0 + 8u * q;
        const int m0 = (int)(tile / gt) * 128, c0 = (int)(tile % gt) * 128, k0 = kb * 64;
        mbar_expect_tx(bar, kLsqStage);
#pragma unroll
        for (int h = 0; h < 3; ++h) tma_load_2d(st + h * kTile, &ymap, h * kPoints + k0, m0, bar);
#pragma unroll
        for (int h = 0; h < 4; ++h) tma_load_2d(st + (3 + h) * kTile, &rmap, h * kPoints + k0, c0, bar);
    };
    uint32_t b = 0;        // blocks consumed (thread 0)
    uint32_t loaded = 0;   // blocks requested (thread 0)
    auto load_next = [&]() {
        // block `loaded` of this CTA's sequence, if it has one
        const uint64_t tile = (uint64_t)blockIdx.x + (uint64_t)(loaded / kBlocks) * gridDim.x;
        if (tile < tiles) {
            load((uint32_t)tile, (int)(loaded % kBlocks), loaded);
            ++loaded;
        }
    };
    if (tid == 0) {
        load_next();
        load_next();
    }
    bool ok = true;
    uint32_t tno = 0;
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++tno) {
        if (tid < 128) {
            const uint32_t g = tile % gt * 128u + (uint32_t)tid;
            cand[tid] = g < ng ? w.cand[g] : make_float2(0.0f, 0.0f);
        }
        if (tid == 0) {
            for (int kb = 0; kb < kBlocks; ++kb, ++b) {
                const uint32_t q = b & 1u, par = (b >> 1) & 1u;
                if (!mbar_wait(full0 + 8u * q, par)) {
                    *abort_flag = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t st = base + q * kLsqStage;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const uint64_t yh = sw128_desc(st + 32u * s), yl = sw128_desc(st + kTile + 32u * s),
                                   dm = sw128_desc(st + 2 * kTile + 32u * s),
                                   rh = sw128_desc(st + 3 * kTile + 32u * s),
                                   rl = sw128_desc(st + 4 * kTile + 32u * s),
                                   qh = sw128_desc(st + 5 * kTile + 32u * s),
                                   ql = sw128_desc(st + 6 * kTile + 32u * s);
                    const uint32_t add = (kb | s) != 0 ? 1u : 0u;
                    mma_bf16_id(tmem, yh, rh, kIdescLsq, add);
                    mma_bf16_id(tmem, yh, rl, kIdescLsq, 1u);
                    mma_bf16_id(tmem, yl, rh, kIdescLsq, 1u);
                    mma_bf16_id(tmem + 128u, dm, rh, kIdescLsq, add);
                    mma_bf16_id(tmem + 256u, dm, qh, kIdescLsq, add);
                    mma_bf16_id(tmem + 256u, dm, ql, kIdescLsq, 1u);
                }
                asm volatile(
                    "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                        done0 + 8u * q)
                    : "memory");
                // the other stage's block (its MMAs went out a step ago) is
                // replaced once they are done
                if (b > 0) {
                    const uint32_t pb = b - 1u;
                    if (!mbar_wait(done0 + 8u * (pb & 1u), (pb >> 1) & 1u)) {
                        *abort_flag = 1;
                        break;
                    }
                    load_next();
                }
            }
        }
        __syncthreads();
        ok = *abort_flag == 0;
        if (!ok) break;
        const uint32_t lb = (tno + 1u) * kBlocks - 1u;  // the tile's last block
        const bool got = mbar_wait(done0 + 8u * (lb & 1u), (lb >> 1) & 1u);
        ok = __syncthreads_and(got);
        if (!ok) break;
        tc_fence_after();
        // epilogue: warps w and w + 4 share TMEM lanes 32 (w % 4) .., a column
        // half each
        const uint32_t half = (uint32_t)warp >> 2;
        const uint32_t i = tile / gt * 128u + 32u * ((uint32_t)warp & 3u) + (uint32_t)lane;
        const uint32_t taddr = tmem + ((32u * ((uint32_t)warp & 3u)) << 16) + 64u * half;
        const bool act = i < n;
        RowStats s{};
        if (act) s = w.stats[i];
        const float inv = act ? 1.0f / s.cnt : 0.0f;
        const uint32_t c0 = tile % gt * 128u + 64u * half;
        auto estimate = [&](float cov, float dr, float dq, float2 c) {
            const float d = c.x - dr, var = (c.y - dq) - d * d * inv;
            const float r = var > 1e-12f && cov > 0.0f ? s.var - cov * cov / var : s.var;
            return fmaxf(r, 0.0f);
        };
        float best = 3.0e38f;
        for (int pass = 0; pass < 2; ++pass) {
            float limit = 0.0f;
            if (pass == 1) {
                float all = best;
                if (act) {
                    const uint32_t old = atomicMin(w.best + i, __float_as_uint(best));
                    all = fminf(best, __uint_as_float(old));
                }
                limit = all + s.margin;
                if (!__any_sync(kFull, act && !(best > limit))) break;
            }
#pragma unroll 1
            for (uint32_t q = 0; q < 4; ++q) {
                uint32_t x[16], y[16], z[16];
                __syncwarp();
                tmem_ld16(taddr + 16u * q, x);
                tmem_ld16(taddr + 128u + 16u * q, y);
                tmem_ld16(taddr + 256u + 16u * q, z);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const uint32_t g = c0 + 16u * q + (uint32_t)e;
                    const float r = estimate(__uint_as_float(x[e]), __uint_as_float(y[e]),
                                             __uint_as_float(z[e]), cand[64u * half + 16u * q + e]);
                    if (g >= ng) continue;
                    if (pass == 0) {
                        best = fminf(best, r);
                    } else if (act && !(r > limit)) {
                        const uint32_t at = atomicAdd(w.count + i, 1u);
                        if (at < kLsqList) w.list[(size_t)i * kLsqList + at] = Listed{r, g0 + g};
                    }
                }
            }
        }
        // every thread is done with the sums before the next tile's MMAs
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }
    if (!ok && tid == 0) {
        w.flags->all = 1u;
        // loads and MMAs still in flight land before the CTA leaves
        for (uint32_t k = loaded > 2u ? loaded - 2u : 0u; k < loaded; ++k)
            mbar_wait(full0 + 8u * (k & 1u), (k >> 1) & 1u);
        if (b > 0) mbar_wait(done0 + 8u * ((b - 1u) & 1u), ((b - 1u) >> 1) & 1u);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                     : "memory");
}

// One warp per trace: the listed candidates' residuals by FP32 sums in point
// order, a candidate per lane; the smallest, then the lowest index.
constexpr int kExactWarps = 8;
__global__ void __launch_bounds__(kExactWarps * 32)
    lsq_exact_kernel(const float *__restrict__ y, uint32_t n, const uint32_t *n_dev,
                     const float *__restrict__ rates, uint32_t G, LsqWork w, uint32_t *idx_out,
                     float *res_out) {
    __shared__ float2 sh[kExactWarps][kPoints];  // {kept value, kept}
    if (n_dev && *n_dev < n) n = *n_dev;
    const uint32_t lane = threadIdx.x & 31u;
    float2 *const yv = sh[threadIdx.x >> 5];
    const uint32_t nw = gridDim.x * kExactWarps;
    const uint32_t n_ill = w.flags->n_ill;
    const bool vec = (reinterpret_cast<uintptr_t>(rates) & 15u) == 0;
    for (uint32_t i = blockIdx.x * kExactWarps + (threadIdx.x >> 5); i < n; i += nw) {
        const RowStats s = w.stats[i];
        for (uint32_t p = lane; p < kPoints; p += 32) {
            const float v = y[(size_t)i * kPoints + p], m = v <= s.thr ? 1.0f : 0.0f;
            yv[p] = make_float2(m * v, m);
        }
        const uint32_t listed = w.count[i];
        const bool every = w.flags->all || listed > kLsqList || listed == 0;
        const float limit = __uint_as_float(w.best[i]) + s.margin;
        const uint32_t total = every ? G : listed + n_ill;
        const float cnt = s.cnt, sy = s.sy, syy = s.syy;
        const float var_y = syy - sy * sy / cnt;
        __syncwarp();
        unsigned long long best = ~0ull;
        for (uint32_t c0 = 0; c0 < total; c0 += 32) {
            const uint32_t c = c0 + lane;
            uint32_t g = 0xFFFFFFFFu;
            if (c < total) {
                if (every) {
                    g = c;
                } else if (c < listed) {
                    const Listed l = w.list[(size_t)i * kLsqList + c];
                    if (!(l.res > limit)) g = l.g;
                } else {
                    g = w.ill[c - listed];
                }
            }
            if (g == 0xFFFFFFFFu) continue;
            const float *const r1 = rates + (size_t)g * kPoints;
            float dyr = 0.0f, dr = 0.0f, drr = 0.0f;
#pragma unroll 4
            for (int p = 0; p < kPoints / 4; ++p) {
                const float4 r = vec ? __ldg(reinterpret_cast<const float4 *>(r1) + p)
                                     : make_float4(__ldg(r1 + 4 * p), __ldg(r1 + 4 * p + 1),
                                                   __ldg(r1 + 4 * p + 2), __ldg(r1 + 4 * p + 3));
                const float rv[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 v = yv[4 * p + e];
                    dyr = fmaf(v.x, rv[e], dyr);
                    dr = fmaf(v.y, rv[e], dr);
                    drr = fmaf(v.y, rv[e] * rv[e], drr);
                }
            }
            const float cov = dyr - sy * dr / cnt;
            const float var_r = drr - dr * dr / cnt;
            float res = var_y;
            if (var_r > 1e-12f && cov > 0.0f) res = var_y - cov * cov / var_r;
            res = fmaxf(res, 0.0f);
            const unsigned long long key = ((unsigned long long)__float_as_uint(res) << 32) | g;
            best = key < best ? key : best;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(kFull, best, o);
            best = v < best ? v : best;
        }
        if (lane == 0) {
            idx_out[i] = (uint32_t)(best & 0xFFFFFFFFull);
            if (res_out) res_out[i] = __uint_as_float((uint32_t)(best >> 32));
        }
        __syncwarp();
    }
}

}  // namespace

size_t lsq_work_bytes(uint32_t n) { return LsqWork(nullptr, n).bytes; }

// The matcher over the first min(n, *n_dev) rows (n_dev NULL: all n).
cudaError_t lsq_run(const float *rates, uint32_t n_geoms, const float *y, uint32_t n,
                    const uint32_t *n_dev, uint32_t *best_out, float *resid_out, void *work, int sms,
                    cudaStream_t st) {
    const LsqWork w(work, n);
    const uint32_t full = (uint32_t)std::max(sms, 1);
    cudaError_t e = cudaMemsetAsync(w.flags, 0, sizeof(Flags), st);
    if (e != cudaSuccess) return e;
    const uint32_t row_blocks = (n + 7u) / 8u;
    lsq_rows_kernel<<<std::min(row_blocks, full * 8u), 256, 0, st>>>(y, n, n_dev, w);
    CUtensorMap ymap, rmap;
    if (!kmajor_map(w.Y, (int)n, kYCols, kYCols, 128, &ymap)) return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(lsq_estimate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kLsqSmem);
    if (e != cudaSuccess) return e;
    for (uint32_t g0 = 0; g0 < n_geoms; g0 += kLsqChunk) {
        const uint32_t ng = std::min(kLsqChunk, n_geoms - g0);
        lsq_rates_kernel<<<(ng + 7u) / 8u, 256, 0, st>>>(rates, g0, ng, w);
        if (!kmajor_map(w.R, (int)ng, kRCols, kRCols, 128, &rmap)) return cudaErrorInvalidValue;
        const uint64_t tiles = (uint64_t)((n + 127u) / 128u) * ((ng + 127u) / 128u);
        lsq_estimate_kernel<<<(unsigned)std::min<uint64_t>(tiles, full), 256, kLsqSmem, st>>>(
            ymap, rmap, n, n_dev, g0, ng, w);
    }
    lsq_exact_kernel<<<std::min((n + kExactWarps - 1u) / kExactWarps, full * 8u), kExactWarps * 32, 0, st>>>(
        y, n, n_dev, rates, n_geoms, w, best_out, resid_out);
    return cudaGetLastError();
}

}  // namespace pchase
