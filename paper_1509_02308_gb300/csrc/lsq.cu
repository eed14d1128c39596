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
// the work is in three parts:
//   1. every pair's covariance on the tcgen05 tensor cores, from centred rows
//      split into BF16 high and low parts (three products, accurate to about
//      1e-5 of Var_y).  Dropped points are zeros in the trace's row, so the
//      covariance needs no mask; Var_r does, but it lies between the row's
//      whole square sum and that less its five largest squares, which bounds
//      the residual from both sides without looking at the pair's points.  A
//      trace lists the candidates whose lower bound is within a margin of the
//      smallest upper bound seen;
//   2. the listed candidates' residuals from the covariance and the five
//      dropped points' rates.  The margin is 1e-3 Var_y, far above both these
//      estimates' error and the FP32 sums', plus 2^-14 of the trace's square
//      sum, which takes over when Var_y is small against it (then FP32 sums
//      cancel, the list overflows and every candidate is evaluated);
//   3. the residuals of the candidates within the margin of the best estimate
//      by the FP32 sums themselves, and the smallest of them.
// A row whose Var_r could lie below 1/64 of its square sum for some trace
// (nearly constant rows, and rows that five points can take nearly all of) has
// no estimate to rely on: differences cancel in it, and the FP32 sums may say
// anything.  Such a row sets no trace's bound and is evaluated for every trace.
// For the others the estimates stay within a fifth of half the margin of the
// FP32 sums' residuals (emulated, Var_r from 1/2 to 1/60 of the square sum).
// Evaluating every pair on the CUDA cores (three FP32 accumulators, 64 x 64
// tiles) took 1388 us for 8192 traces x 1308 candidates, 80 % of it FP32 issue
// and shared-memory loads; with the dropped points' sums as three more tensor
// products per pair, a 128 x 128 tile's load, MMA and epilogue one after the
// other and a trace to a warp in part 3, 232 us (150 the estimates, 66 part 3).
// Now 98 us: 37 the covariances (287 MB of operand tiles from L2 at 7.7 TB/s,
// tensor pipe 41 % active), 42 parts 2 and 3 (latency: 512 dependent adds a
// candidate, 19 % of issue slots used), 14 the traces' rows, 5 the candidates'.
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
constexpr uint32_t kLsqList = 128;     // listed candidates of a trace
constexpr uint32_t kLsqIll = 4096;     // rows without estimates
constexpr int kDrop = kPoints - kKeep; // points a trace drops, at most
constexpr int kCols = 2 * kPoints;     // an operand row: high parts, low parts

struct __align__(16) RowStats {
    float thr, cnt, sy, syy;  // kept: v <= thr; their count, sum and square sum
    float mean, var;          // of the kept points, from centred sums
    float margin;
    uint32_t n_drop;
    uint16_t drop[8];         // the dropped points
};
struct __align__(16) Listed {
    float cov;  // then the residual's estimate
    uint32_t g;
    float mean, s2;  // the candidate's mean and centred square sum
};
struct __align__(16) Cand {
    float inv_low, inv_s2;  // 1 / the least and the whole centred square sum
    float mean, s2;
};
struct Flags {
    uint32_t all;    // 1: evaluate every candidate (a wait gave up, too many rows without estimates)
    uint32_t n_ill;  // rows without estimates
    uint32_t n_every;  // traces that evaluate every candidate
};

// The workspace: per trace operands, statistics, best estimate, list; then a
// chunk of candidates.
struct LsqWork {
    __nv_bfloat16 *Y, *R;
    RowStats *stats;
    uint32_t *best, *count, *ill, *every;
    Listed *list;
    Cand *cand;
    Flags *flags;
    size_t bytes;
    // (the caller's buffer may start anywhere; the tensor maps' rows may not)
    LsqWork(void *base, size_t n) {
        uint8_t *const p = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(base) + 255) & ~uintptr_t(255));
        size_t o = 0;
        auto take = [&](size_t b) {
            uint8_t *q = p + o;
            o = (o + b + 255) & ~size_t(255);
            return q;
        };
        Y = reinterpret_cast<__nv_bfloat16 *>(take(n * kCols * 2));
        stats = reinterpret_cast<RowStats *>(take(n * sizeof(RowStats)));
        best = reinterpret_cast<uint32_t *>(take(n * 4));
        count = reinterpret_cast<uint32_t *>(take(n * 4));
        list = reinterpret_cast<Listed *>(take(n * kLsqList * sizeof(Listed)));
        R = reinterpret_cast<__nv_bfloat16 *>(take((size_t)kLsqChunk * kCols * 2));
        cand = reinterpret_cast<Cand *>(take((size_t)kLsqChunk * sizeof(Cand)));
        every = reinterpret_cast<uint32_t *>(take(n * 4));
        ill = reinterpret_cast<uint32_t *>(take(kLsqIll * 4));
        flags = reinterpret_cast<Flags *>(take(sizeof(Flags)));
        bytes = o + 255;
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
        uint32_t key[16], kth = 0;  // (a value taken out has key 0)
#pragma unroll
        for (int e = 0; e < 16; ++e) key[e] = order_key(v[e]);
        for (int round = 0; round < kDrop + 1; ++round) {
            uint32_t top = 0;
#pragma unroll
            for (int e = 0; e < 16; ++e) top = max(top, key[e]);
            kth = __reduce_max_sync(kFull, top);
            const uint32_t who = __ballot_sync(kFull, top == kth);
            bool mine = lane == (uint32_t)(__ffs(who) - 1);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const bool hit = mine && key[e] == kth;
                key[e] = hit ? 0u : key[e];
                mine = mine && !hit;
            }
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
        __nv_bfloat16 *o = w.Y + (size_t)i * kCols;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            __nv_bfloat16 hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool kept = v[4 * q + e] <= thr;
                const float z = kept ? v[4 * q + e] - mean : 0.0f;
                var += z * z;
                hi[e] = __float2bfloat16(z);
                lo[e] = __float2bfloat16(z - __bfloat162float(hi[e]));
            }
            const uint32_t p = 4 * lane + 128 * q;
            *reinterpret_cast<uint2 *>(o + p) = *reinterpret_cast<const uint2 *>(hi);
            *reinterpret_cast<uint2 *>(o + kPoints + p) = *reinterpret_cast<const uint2 *>(lo);
        }
        var = warp_sum(var);
        uint32_t nd = 0;  // dropped points (more than kDrop: values that compare with nothing)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            const bool gone = !(v[e] <= thr);
            const uint32_t who = __ballot_sync(kFull, gone);
            const uint32_t at = nd + (uint32_t)__popc(who & ((1u << lane) - 1u));
            if (gone && at < 8u) w.stats[i].drop[at] = (uint16_t)(4 * lane + 128 * (e >> 2) + (e & 3));
            nd += (uint32_t)__popc(who);
        }
        if (lane == 0) {
            RowStats &s = w.stats[i];
            s.thr = thr;
            s.cnt = c;
            s.sy = sy;
            s.syy = syy;
            s.mean = mean;
            s.var = var;
            s.margin = 1e-3f * var + syy * (1.0f / 16384.0f);
            s.n_drop = min(nd, (uint32_t)kDrop);
            w.best[i] = 0x7F800000u;
            w.count[i] = nd > (uint32_t)kDrop ? kLsqList + 1u : 0u;
        }
    }
}

// One warp per candidate of the chunk: centred row, split, its square sum and
// what is left of that without its five largest squares.
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
    float s2 = 0.0f, zz[16];
    __nv_bfloat16 *o = w.R + (size_t)k * kCols;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        __nv_bfloat16 hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float z = v[4 * q + e] - mean;
            zz[4 * q + e] = z * z;
            s2 += z * z;
            hi[e] = __float2bfloat16(z);
            lo[e] = __float2bfloat16(z - __bfloat162float(hi[e]));
        }
        const uint32_t p = 4 * lane + 128 * q;
        *reinterpret_cast<uint2 *>(o + p) = *reinterpret_cast<const uint2 *>(hi);
        *reinterpret_cast<uint2 *>(o + kPoints + p) = *reinterpret_cast<const uint2 *>(lo);
    }
    s2 = warp_sum(s2);
    float top = 0.0f;
    uint32_t out = 0;
    for (int round = 0; round < kDrop; ++round) {
        float mx = -1.0f;
        int at = 0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (!((out >> e) & 1u) && zz[e] > mx) {
                mx = zz[e];
                at = e;
            }
        }
        const uint32_t all = __reduce_max_sync(kFull, mx < 0.0f ? 0u : __float_as_uint(mx));
        const uint32_t who = __ballot_sync(kFull, mx >= 0.0f && __float_as_uint(mx) == all);
        if (lane == (uint32_t)(__ffs(who) - 1)) out |= 1u << at;
        top += __uint_as_float(all);
    }
    if (lane == 0) {
        // a trace's Var_r is s2 less its dropped points' squares and less
        // (their sum)^2 / 507, below a hundredth of their squares
        const float low = s2 * (1.0f - 1e-5f) - 1.02f * top;
        Cand c;
        // (also rows whose sums are not finite, and rows so small that Var_r
        // may be on either side of the 1e-12 that makes it 0; a row of zeros
        // has the trace's variance as its residual exactly)
        const bool ill = !(64.0f * low >= raw) || (raw > 0.0f && !(low > 1e-9f));
        c.inv_low = ill || raw == 0.0f ? 0.0f : 1.0f / low;
        c.inv_s2 = ill || raw == 0.0f ? 0.0f : 1.0f / s2;
        c.mean = mean;
        c.s2 = ill ? 0.0f : s2;  // (0: estimated at the trace's variance, above every residual)
        w.cand[k] = c;
        if (ill) {
            const uint32_t at = atomicAdd(&w.flags->n_ill, 1u);
            if (at < kLsqIll) w.ill[at] = g0 + k;
            else w.flags->all = 1u;
        }
    }
}

// A pair's residual from its covariance (a positive one's square), the
// candidate's mean and centred square sum, and its rates at the trace's
// dropped points.
__device__ __forceinline__ float estimate(float cov2, float mean, float s2, const float *__restrict__ row,
                                          const RowStats &s) {
    float dr = 0.0f, dq = 0.0f;
#pragma unroll
    for (uint32_t k = 0; k < (uint32_t)kDrop; ++k) {
        if (k < s.n_drop) {
            const float r = __ldg(row + s.drop[k]) - mean;
            dr += r;
            dq += r * r;
        }
    }
    const float var_r = (s2 - dq) - dr * dr / s.cnt;
    return var_r > 1e-12f ? fmaxf(s.var - cov2 / var_r, 0.0f) : s.var;
}

// Covariances and lists: persistent CTAs over tiles of 128 traces x N
// candidates, candidate-major, so that the first tiles leave most traces an
// upper bound for the others to list by.  A K block of 64 points is four TMA
// tiles (32 KB of traces, N / 4 KB of candidates) in a ring of stages and 12
// MMAs; the sums are double buffered in TMEM (columns 0 and 256), so the next
// tile's MMAs run under this one's epilogue.  Warps 0-7: epilogue, a thread per
// trace and column half; warp 8: loads; warp 9: MMAs (one thread each).
//
// N: bytes read per tile are 256 (N + 128) a K row, and a wave is a tile on
// every SM, so the N with the least waves (N + 128) (8192 x 1308: 192, three
// waves).
constexpr uint32_t kTile = 128 * 128;  // bytes of a 128 x 64 BF16 tile
constexpr uint32_t kLsqMaxN = 256, kLsqMaxStages = 5, kLsqRing = 200 * 1024;
constexpr uint32_t kLsqBars = 16;      // loaded, free [stages]; sums ready, read [2]
constexpr uint32_t kLsqSmem = 1024 + kLsqRing + kLsqMaxN * 16 + kLsqBars * 8 + 16;
constexpr uint32_t kLsqThreads = 320;
// M 128, BF16 operands, FP32 sums; N is added
constexpr uint32_t kIdescLsq = (1u << 4) | (1u << 7) | (1u << 10) | ((128u >> 4) << 24);

__host__ __device__ constexpr uint32_t lsq_stage_bytes(uint32_t N) { return 2 * kTile + 2 * N * 128; }

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

__global__ void __launch_bounds__(kLsqThreads, 1)
    lsq_estimate_kernel(const __grid_constant__ CUtensorMap ymap, const __grid_constant__ CUtensorMap rmap,
                        const float *__restrict__ rates, uint32_t n, const uint32_t *n_dev, uint32_t g0,
                        uint32_t ng, uint32_t N, LsqWork w) {
    extern __shared__ uint8_t dsm[];
    const uint32_t raw = smem_u32(dsm);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *const gbase = dsm + (base - raw);
    Cand *const cand = reinterpret_cast<Cand *>(gbase + kLsqRing);
    const uint32_t bars = base + kLsqRing + kLsqMaxN * 16;
    const uint32_t full0 = bars, free0 = bars + 8 * kLsqMaxStages, ready0 = free0 + 8 * kLsqMaxStages,
                   read0 = ready0 + 16;
    uint32_t *const tslot = reinterpret_cast<uint32_t *>(gbase + kLsqRing + kLsqMaxN * 16 + kLsqBars * 8);
    volatile uint32_t *const abort_flag = tslot + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (n_dev && *n_dev < n) n = *n_dev;
    const uint32_t stage = lsq_stage_bytes(N), S = min(kLsqMaxStages, kLsqRing / stage);
    const uint32_t mt = (n + 127u) / 128u, tiles = mt * ((ng + N - 1u) / N);
    constexpr int kBlocks = kPoints / 64;
    if (tid == 0) {
        for (uint32_t q = 0; q < 2 * kLsqMaxStages + 2; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bars + 8 * q) : "memory");
        for (uint32_t q = 0; q < 2; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(read0 + 8 * q) : "memory");
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
    // K blocks are numbered through all of this CTA's tiles: block b is in
    // stage b mod S, whose barriers it completes for the (b / S)-th time
    if (warp == 8) {
        if (lane == 0) {
            uint32_t b = 0, q = 0, par = 0;
            for (uint32_t tile = blockIdx.x; tile < tiles && !*abort_flag; tile += gridDim.x) {
                const int m0 = (int)(tile % mt) * 128, c0 = (int)(tile / mt * N);
                for (int kb = 0; kb < kBlocks; ++kb, ++b) {
                    if (!mbar_wait(free0 + 8u * q, par ^ 1u)) {
                        *abort_flag = 1;
                        break;
                    }
                    const uint32_t st = base + q * stage, bar = full0 + 8u * q;
                    mbar_expect_tx(bar, stage);
                    tma_load_2d(st, &ymap, kb * 64, m0, bar);
                    tma_load_2d(st + kTile, &ymap, kPoints + kb * 64, m0, bar);
                    tma_load_2d(st + 2 * kTile, &rmap, kb * 64, c0, bar);
                    tma_load_2d(st + 2 * kTile + N * 128, &rmap, kPoints + kb * 64, c0, bar);
                    if (++q == S) {
                        q = 0;
                        par ^= 1u;
                    }
                }
            }
            // loads in flight land before the CTA leaves
            for (uint32_t k = b > S ? b - S : 0u; k < b; ++k) mbar_wait(full0 + 8u * (k % S), (k / S) & 1u);
        }
    } else if (warp == 9) {
        if (lane == 0) {
            const uint32_t idesc = kIdescLsq | ((N >> 3) << 17);
            uint32_t b = 0, q = 0, par = 0, tno = 0;
            bool ok = true;
            for (uint32_t tile = blockIdx.x; ok && tile < tiles && !*abort_flag; tile += gridDim.x, ++tno) {
                const uint32_t buf = tno & 1u, d = tmem + 256u * buf;
                ok = mbar_wait(read0 + 8u * buf, ((tno >> 1) & 1u) ^ 1u);
                tc_fence_after();
                for (int kb = 0; ok && kb < kBlocks; ++kb) {
                    ok = mbar_wait(full0 + 8u * q, par);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t st = base + q * stage;
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        const uint64_t yh = sw128_desc(st + 32u * s), yl = sw128_desc(st + kTile + 32u * s),
                                       rh = sw128_desc(st + 2 * kTile + 32u * s),
                                       rl = sw128_desc(st + 2 * kTile + N * 128 + 32u * s);
                        mma_bf16_id(d, yh, rh, idesc, (kb | s) != 0 ? 1u : 0u);
                        mma_bf16_id(d, yh, rl, idesc, 1u);
                        mma_bf16_id(d, yl, rh, idesc, 1u);
                    }
                    mma_commit(free0 + 8u * q);
                    ++b;
                    if (++q == S) {
                        q = 0;
                        par ^= 1u;
                    }
                }
                if (ok) mma_commit(ready0 + 8u * buf);
            }
            if (!ok) *abort_flag = 1;
            // and so do the MMAs
            if (b) mbar_wait(free0 + 8u * ((b - 1u) % S), ((b - 1u) / S) & 1u);
        }
    } else {
        // warps w and w + 4 share TMEM lanes 32 (w % 4) .., a column half each
        const uint32_t quarter = (uint32_t)warp & 3u, half = (uint32_t)warp >> 2, cols = N / 2;
        uint32_t tno = 0;
        for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++tno) {
            const uint32_t buf = tno & 1u, c0 = tile / mt * N;
            // (every warp is done with the last tile's candidates)
            if (group_any(1, *abort_flag != 0)) break;
            for (uint32_t c = (uint32_t)tid; c < N; c += 256) {
                float4 f = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (c0 + c < ng) f = *reinterpret_cast<const float4 *>(w.cand + c0 + c);
                *reinterpret_cast<float4 *>(cand + c) = f;
            }
            const uint32_t i = tile % mt * 128u + 32u * quarter + (uint32_t)lane;
            const bool act = i < n;
            RowStats s{};
            if (act) s = w.stats[i];
            const bool got = mbar_wait(ready0 + 8u * buf, (tno >> 1) & 1u);
            if (group_any(1, !got)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t taddr = tmem + 256u * buf + ((32u * quarter) << 16) + half * cols;
            const Cand *const cd = cand + half * cols;
            // the residual is var - cov^2 / Var_r for a positive covariance
            float top = 0.0f;
            uint32_t arg = 0;
#pragma unroll 1
            for (uint32_t q = 0; q < cols; q += 16) {
                uint32_t x[16];
                __syncwarp();
                tmem_ld16(taddr + q, x);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float cov = fmaxf(__uint_as_float(x[e]), 0.0f), gain = cov * cov * cd[q + e].inv_s2;
                    if (gain > top) {
                        top = gain;
                        arg = q + (uint32_t)e;
                    }
                }
            }
            // the estimate of the one with the least upper bound: a third of
            // the listed candidates that the bound itself lets through
            float best = s.var;
            if (act && top > 0.0f) {
                const Cand f = cd[arg];
                best = estimate(top * f.s2, f.mean, f.s2, rates + (size_t)(g0 + c0 + half * cols + arg) * kPoints,
                                s);
            }
            if (act) best = fminf(best, __uint_as_float(atomicMin(w.best + i, __float_as_uint(best))));
            const float need = s.var - (best + s.margin);
            uint32_t take[kLsqMaxN / 64] = {}, found = 0;
#pragma unroll
            for (uint32_t h = 0; h < kLsqMaxN / 64; ++h) {
                if (32 * h >= cols) break;
#pragma unroll
                for (uint32_t q = 0; q < 32; q += 16) {
                    if (32 * h + q >= cols) break;
                    uint32_t x[16];
                    __syncwarp();
                    tmem_ld16(taddr + 32 * h + q, x);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float cov = __uint_as_float(x[e]);
                        const float gain = cov > 0.0f ? cov * cov * cd[32 * h + q + e].inv_low : 0.0f;
                        if (!(gain < need)) take[h] |= 1u << (q + (uint32_t)e);
                    }
                }
                // (columns past the last candidate)
                const uint32_t c = c0 + half * cols + 32 * h;
                if (!act || c >= ng) take[h] = 0;
                else if (ng - c < 32) take[h] &= (1u << (ng - c)) - 1u;
                found += (uint32_t)__popc(take[h]);
            }
            // one reservation a thread and tile: an atomic's round trip per
            // listed candidate cost more than the tile's MMAs
            uint32_t at = found ? atomicAdd(w.count + i, found) : 0u;
            Listed *const list = w.list + (size_t)i * kLsqList;
#pragma unroll
            for (uint32_t h = 0; h < kLsqMaxN / 64; ++h) {
                if (32 * h >= cols) break;
#pragma unroll
                for (uint32_t q = 0; q < 32; q += 16) {
                    if (32 * h + q >= cols) break;
                    if (!__any_sync(kFull, (take[h] >> q) & 0xFFFFu)) continue;
                    uint32_t x[16];
                    tmem_ld16(taddr + 32 * h + q, x);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if ((take[h] >> (q + (uint32_t)e)) & 1u) {
                            const uint32_t c = 32 * h + q + (uint32_t)e;
                            if (at < kLsqList)
                                list[at] = Listed{__uint_as_float(x[e]), g0 + c0 + half * cols + c, cd[c].mean,
                                                  cd[c].s2};
                            ++at;
                        }
                    }
                }
            }
            // the sums are read; their columns may take the tile after next
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(read0 + 8u * buf);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && *abort_flag) w.flags->all = 1u;
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u)
                     : "memory");
}

// A candidate's residual by FP32 sums in point order: v the kept values (0 at
// dropped points), kept a bit per point, both in shared memory.
struct Trace {
    float cnt, sy, var_y;
};
__device__ __forceinline__ float residual(const float *__restrict__ r1, bool vec, const float *v,
                                          const uint32_t *kept, const Trace &t) {
    float dyr = 0.0f, dr = 0.0f, drr = 0.0f;
    auto load = [&](int q, float4 (&r)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float *const p = r1 + 32 * q + 4 * k;
            r[k] = vec ? __ldg(reinterpret_cast<const float4 *>(p))
                       : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
        }
    };
    auto add = [&](int q, const float4 (&r)[8]) {
        const uint32_t bits = kept[q];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float4 y = *reinterpret_cast<const float4 *>(v + 32 * q + 4 * k);
            const float rv[4] = {r[k].x, r[k].y, r[k].z, r[k].w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float m = (bits >> (4 * k + e)) & 1u ? 1.0f : 0.0f;
                dyr = fmaf(yv[e], rv[e], dyr);
                dr = fmaf(m, rv[e], dr);
                drr = fmaf(m, rv[e] * rv[e], drr);
            }
        }
    };
    // 128 bytes of the row ahead of the adds
    float4 a[8], b[8];
    load(0, a);
#pragma unroll 1
    for (int q = 0; q < kPoints / 32; q += 2) {
        load(q + 1, b);
        add(q, a);
        if (q + 2 < kPoints / 32) load(q + 2, a);
        add(q + 1, b);
    }
    const float cov = dyr - t.sy * dr / t.cnt;
    const float var_r = drr - dr * dr / t.cnt;
    float res = t.var_y;
    if (var_r > 1e-12f && cov > 0.0f) res = t.var_y - cov * cov / var_r;
    return fmaxf(res, 0.0f);
}

// the kept values and bits of trace i, by a warp
__device__ __forceinline__ void load_trace(const float *__restrict__ y, uint32_t i, float thr, float *v,
                                           uint32_t *kept, uint32_t lane) {
#pragma unroll 4
    for (uint32_t q = 0; q < kPoints / 32; ++q) {
        const float x = y[(size_t)i * kPoints + 32 * q + lane], m = x <= thr ? 1.0f : 0.0f;
        v[32 * q + lane] = m * x;
        const uint32_t bits = __ballot_sync(kFull, x <= thr);
        if (lane == 0) kept[q] = bits;
    }
}

// What the warps of one left-over trace share, at the start of its list.
struct Shared {
    unsigned long long key;  // least residual, then candidate
    uint32_t done;           // parts evaluated
};

// Eight lanes to a trace: its listed candidates' estimates, then the residuals
// of those within the margin of the best (3 on average), a candidate per lane;
// the smallest, then the lowest index.  A residual is a chain of 512 dependent
// adds fed by 2 KB of its own row, so what counts is that every trace is in
// flight at once and a lane's loads go out 128 bytes at a time.
constexpr int kExactWarps = 4, kGroup = 8, kPerWarp = 32 / kGroup;
constexpr int kRowPad = kPoints + 4, kKeptPad = kPoints / 32 + 1;  // (the groups' banks differ)
__global__ void __launch_bounds__(kExactWarps * 32)
    lsq_exact_kernel(const float *__restrict__ y, uint32_t n, const uint32_t *n_dev,
                     const float *__restrict__ rates, LsqWork w, uint32_t *idx_out, float *res_out) {
    __shared__ __align__(16) float rows[kExactWarps][kPerWarp][kRowPad];
    __shared__ uint32_t keeps[kExactWarps][kPerWarp][kKeptPad];
    __shared__ uint32_t lists[kExactWarps][kPerWarp][kLsqList];
    if (n_dev && *n_dev < n) n = *n_dev;
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, grp = lane / kGroup, l = lane % kGroup;
    uint32_t *const near = lists[wid][grp];
    const uint32_t nw = gridDim.x * kExactWarps;
    const uint32_t n_ill = w.flags->n_ill;
    const bool all = w.flags->all != 0;
    const bool vec = (reinterpret_cast<uintptr_t>(rates) & 15u) == 0;
    for (uint32_t t0 = (blockIdx.x * kExactWarps + wid) * kPerWarp; t0 < n; t0 += nw * kPerWarp) {
        const uint32_t i = t0 + grp;
        const uint32_t listed = i < n ? w.count[i] : 0u;
        const bool every = all || listed > kLsqList || listed == 0;
        if (i < n && every && l == 0) {
            w.every[atomicAdd(&w.flags->n_every, 1u)] = i;
            *reinterpret_cast<Shared *>(w.list + (size_t)i * kLsqList) = Shared{~0ull, 0u};
        }
        const bool act = i < n && !every;
        if (!__any_sync(kFull, act)) continue;
        RowStats s{};
        if (act) s = w.stats[i];
        __syncwarp();  // (the last traces' rows are read)
#pragma unroll 1
        for (uint32_t q = 0; q < kPerWarp; ++q) {
            const float thr = __shfl_sync(kFull, s.thr, q * kGroup);
            if (__shfl_sync(kFull, act ? 1u : 0u, q * kGroup))
                load_trace(y, t0 + q, thr, rows[wid][q], keeps[wid][q], lane);
        }
        Listed *const list = w.list + (size_t)i * kLsqList;
        float best = 3.0e38f;
        if (act) {
            for (uint32_t c = l; c < listed; c += kGroup) {
                const Listed e = list[c];
                const float est =
                    e.cov > 0.0f ? estimate(e.cov * e.cov, e.mean, e.s2, rates + (size_t)e.g * kPoints, s) : s.var;
                list[c].cov = est;
                best = fminf(best, est);
            }
        }
#pragma unroll
        for (int o = kGroup / 2; o; o >>= 1) best = fminf(best, __shfl_xor_sync(kFull, best, o));
        const float limit = best + s.margin;
        uint32_t n_near = 0;
        const uint32_t trips = __reduce_max_sync(kFull, act ? listed : 0u);
        for (uint32_t c = l; c < trips + l; c += kGroup) {
            bool take = false;
            uint32_t g = 0;
            if (act && c < listed) {
                take = !(list[c].cov > limit);
                g = list[c].g;
            }
            const uint32_t who = (__ballot_sync(kFull, take) >> (grp * kGroup)) & ((1u << kGroup) - 1u);
            if (take) near[n_near + (uint32_t)__popc(who & ((1u << l) - 1u))] = g;
            n_near += (uint32_t)__popc(who);
        }
        __syncwarp();
        unsigned long long key = ~0ull;
        if (act) {
            const Trace t{s.cnt, s.sy, s.syy - s.sy * s.sy / s.cnt};
            for (uint32_t c = l; c < n_near + n_ill; c += kGroup) {
                const uint32_t g = c < n_near ? near[c] : w.ill[c - n_near];
                const float res = residual(rates + (size_t)g * kPoints, vec, rows[wid][grp], keeps[wid][grp], t);
                const unsigned long long k = ((unsigned long long)__float_as_uint(res) << 32) | g;
                key = k < key ? k : key;
            }
        }
#pragma unroll
        for (int o = kGroup / 2; o; o >>= 1) {
            const unsigned long long k = __shfl_xor_sync(kFull, key, o);
            key = k < key ? k : key;
        }
        if (act && l == 0) {
            idx_out[i] = (uint32_t)(key & 0xFFFFFFFFull);
            if (res_out) res_out[i] = __uint_as_float((uint32_t)(key >> 32));
        }
    }
}

// The traces left over: every candidate's residual, 32 candidates at a time.
// A trace's candidates are parted among the warps that there are for it (one
// trace of 1308 candidates by one warp: 0.4 ms).
constexpr int kEveryWarps = 8;
__global__ void __launch_bounds__(kEveryWarps * 32, 2)
    lsq_every_kernel(const float *__restrict__ y, const float *__restrict__ rates, uint32_t G, LsqWork w,
                     uint32_t *idx_out, float *res_out) {
    __shared__ __align__(16) float rows[kEveryWarps][kPoints];
    __shared__ uint32_t keeps[kEveryWarps][kPoints / 32];
    const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const uint32_t total = w.flags->n_every;
    if (!total) return;
    const uint32_t nw = gridDim.x * kEveryWarps, rounds = (G + 31u) / 32u;
    const uint32_t most = min(rounds, max(nw / total, 1u)), each = (rounds + most - 1u) / most,
                   parts = (rounds + each - 1u) / each;
    const bool vec = (reinterpret_cast<uintptr_t>(rates) & 15u) == 0;
    for (uint64_t k = blockIdx.x * kEveryWarps + wid; k < (uint64_t)total * parts; k += nw) {
        const uint32_t i = w.every[k / parts], part = (uint32_t)(k % parts);
        const RowStats s = w.stats[i];
        __syncwarp();
        load_trace(y, i, s.thr, rows[wid], keeps[wid], lane);
        __syncwarp();
        const Trace t{s.cnt, s.sy, s.syy - s.sy * s.sy / s.cnt};
        unsigned long long key = ~0ull;
        const uint32_t last = min(G, 32u * each * (part + 1u));
        for (uint32_t g = 32u * each * part + lane; g < last; g += 32) {
            const float res = residual(rates + (size_t)g * kPoints, vec, rows[wid], keeps[wid], t);
            const unsigned long long x = ((unsigned long long)__float_as_uint(res) << 32) | g;
            key = x < key ? x : key;
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            const unsigned long long x = __shfl_xor_sync(kFull, key, o);
            key = x < key ? x : key;
        }
        if (lane == 0) {
            Shared *const sh = reinterpret_cast<Shared *>(w.list + (size_t)i * kLsqList);
            if (parts > 1) {
                atomicMin(&sh->key, key);
                __threadfence();
                if (atomicAdd(&sh->done, 1u) + 1u < parts) continue;
                __threadfence();
                key = atomicMin(&sh->key, ~0ull);
            }
            idx_out[i] = (uint32_t)(key & 0xFFFFFFFFull);
            if (res_out) res_out[i] = __uint_as_float((uint32_t)(key >> 32));
        }
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
    if (!kmajor_map(w.Y, (int)n, kCols, kCols, 128, &ymap)) return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(lsq_estimate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kLsqSmem);
    if (e != cudaSuccess) return e;
    const uint32_t mt = (n + 127u) / 128u;
    for (uint32_t g0 = 0; g0 < n_geoms; g0 += kLsqChunk) {
        const uint32_t ng = std::min(kLsqChunk, n_geoms - g0);
        lsq_rates_kernel<<<(ng + 7u) / 8u, 256, 0, st>>>(rates, g0, ng, w);
        uint32_t N = 0;
        uint64_t least = ~0ull, tiles = 0;
        for (uint32_t c = 32; c <= kLsqMaxN; c += 32) {
            const uint64_t t = (uint64_t)mt * ((ng + c - 1u) / c), cost = (t + full - 1u) / full * (c + 128u);
            if (cost < least) {
                least = cost;
                N = c;
                tiles = t;
            }
        }
        if (!kmajor_map(w.R, (int)ng, kCols, kCols, (int)N, &rmap)) return cudaErrorInvalidValue;
        lsq_estimate_kernel<<<(unsigned)std::min<uint64_t>(tiles, full), kLsqThreads, kLsqSmem, st>>>(
            ymap, rmap, rates, n, n_dev, g0, ng, N, w);
    }
    constexpr uint32_t kPerBlock = kExactWarps * kPerWarp;
    lsq_exact_kernel<<<std::min((n + kPerBlock - 1u) / kPerBlock, full * 16u), kExactWarps * 32, 0, st>>>(
        y, n, n_dev, rates, w, best_out, resid_out);
    lsq_every_kernel<<<full * 2u, kEveryWarps * 32, 0, st>>>(
        y, rates, n_geoms, w, best_out, resid_out);
    return cudaGetLastError();
}

}  // namespace pchase
