// S4: latency -> hit/miss, and the matcher's canonical pick.
//
// Sec. 4.1 models a P-chase latency as t0 (hit) or t0 + t_m (miss); the paper
// states no cut rule.  The rule implemented (the same one the CPU oracle
// states): over one observation of n latencies, set aside the floor(n/200)
// largest, take the largest gap between consecutive distinct kept values (the
// lowest on ties) and cut at (lo + hi) * 0.5f.
//
// GPU form, without a sort.  Observations of up to 8 x 48K latencies take one
// launch (classify_cluster_kernel): a cluster of up to eight CTAs holds the
// observation in shared memory from end to end.  Longer ones take the same
// steps as launches over global memory:
//   1. radix select (four 8-bit digit passes over order-preserving keys) finds
//      the cut value v[keep-1] exactly, and the minimum;
//   2. maximum gap by pigeonhole (Gonzalez's linear-time maximum-gap method):
//      the kept values go into 2*keep equal-width buckets keeping each
//      bucket's min and max; a gap inside one bucket is at most half the
//      average gap, so the largest gap lies between consecutive non-empty
//      buckets, and is computed from the same two floats as a sort would give;
//   3. a block scans the buckets in order (first maximum wins) and a grid
//      writes the miss bits with __ballot_sync.
#include <mutex>

#include <algorithm>

#include <cooperative_groups.h>

#include "pchase_internal.cuh"

namespace pchase {

namespace {

__device__ __forceinline__ uint32_t fkey(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fval(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

struct ObsMeta {
    uint32_t cut_key;
    uint32_t min_key;
    uint32_t nb;   // buckets (0: no gap possible)
    float thr;
};

// ---- one launch per call: a cluster of CTAs per observation
// Each CTA keeps a slice of the observation's keys in shared memory.  The cut
// value is found by three histogram passes (11, 11 and 10 bits; a bin's count
// goes up by one per latency, which the hardware adds up within a warp), rank 0
// adding the CTAs' bins through distributed shared memory.  The maximum gap:
// kGapBuckets equal buckets first (min and max key of each); when the largest
// gap between neighbouring buckets is wider than a bucket no gap inside one
// can reach it, and it is the answer (two latency plateaus: always).  If not,
// or where the bucket arithmetic is not regular, the 2 * keep buckets of the
// pigeonhole method follow, kGapBuckets of them at a time.  Bound by the
// passes over shared memory and a dozen cluster barriers: 64 observations of
// 16K-64K latencies take 40 us against 288 us as four launches, one CTA per
// observation; one of 177K latencies, as the matcher pools, 39 against 458 us.
constexpr uint32_t kGapBuckets = 4096;
constexpr uint32_t kClusterThreads = 512;
constexpr uint32_t kClusterMaxKeys = 49152;  // of one CTA (192 KB, beside 33 KB of buckets)
constexpr uint32_t kClusterMax = 8;

struct ClusterShared {
    uint4 bucket4[kGapBuckets / 2];  // uint2 {min key, max key} per bucket; the histogram's bins before
    unsigned long long best;
    uint32_t warp_v[kClusterThreads / 32];
    uint32_t prefix, k, min_key, carry, found;
    float gap, lo, hi, thr;
};
constexpr size_t kClusterSmemBase = (sizeof(ClusterShared) + 15) & ~size_t(15);

// Exclusive prefix of v over the CTA's threads under op (identity id).
template <typename Op>
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t id, uint32_t *warp_v, Op op) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc = op(inc, x);
    }
    if (lane == 31) warp_v[w] = inc;
    __syncthreads();
    uint32_t before = id;
    for (int q = 0; q < w; ++q) before = op(before, warp_v[q]);
    const uint32_t up = __shfl_up_sync(kFull, inc, 1);
    __syncthreads();
    return lane ? op(before, up) : before;
}

__global__ void __launch_bounds__(kClusterThreads, 2)
    classify_cluster_kernel(const float *__restrict__ lat, const uint64_t *__restrict__ offsets,
                            uint64_t max_len, ObsMeta *meta, float *thresh_out, uint32_t *bits,
                            const uint64_t *__restrict__ word_offsets) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) uint8_t c_smem[];
    ClusterShared &S = *reinterpret_cast<ClusterShared *>(c_smem);
    uint32_t *const keys = reinterpret_cast<uint32_t *>(c_smem + kClusterSmemBase);
    uint32_t *const hist = reinterpret_cast<uint32_t *>(S.bucket4);
    uint2 *const bucket = reinterpret_cast<uint2 *>(S.bucket4);
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t C = cluster.num_blocks(), rank = cluster.block_rank();
    ClusterShared *const S0 = cluster.map_shared_rank(&S, 0);
    const uint32_t o = blockIdx.x / C, tid = threadIdx.x;
    const uint64_t b0 = offsets[o], n64 = offsets[o + 1] - b0;
    if (n64 == 0 || n64 > max_len) {
        // empty, or longer than the caller's max_len: refused (NaN cut, bits 0)
        const float thr = n64 ? __int_as_float(0x7FC00000) : 0.0f;
        if (rank == 0 && tid == 0) {
            meta[o] = ObsMeta{0, 0, 0, thr};
            if (thresh_out) thresh_out[o] = thr;
        }
        if (bits && n64) {
            const uint64_t words = (n64 + 31) / 32;
            for (uint64_t w = (uint64_t)rank * kClusterThreads + tid; w < words; w += (uint64_t)C * kClusterThreads)
                bits[word_offsets[o] + w] = 0;
        }
        return;
    }
    const uint32_t n = (uint32_t)n64, keep = n - n / 200;
    const uint32_t per = ((n + C - 1) / C + 31u) & ~31u;
    const uint32_t first = min(n, rank * per), cnt = min(n, first + per) - first;
    const float *const x = lat + b0 + first;
    if (tid == 0) {
        S.min_key = 0xFFFFFFFFu;
        S.prefix = 0;
        S.k = keep;
        S.carry = 0;
        S.gap = 0.0f;
        S.found = 0;
    }
    __syncthreads();
    uint32_t mn = 0xFFFFFFFFu;
    for (uint32_t i = tid; i < cnt; i += kClusterThreads) {
        const uint32_t k = fkey(x[i]);
        keys[i] = k;
        mn = min(mn, k);
    }
    mn = __reduce_min_sync(kFull, mn);
    if ((tid & 31) == 0) atomicMin(&S.min_key, mn);
    // ---- the cut value: keep-th smallest key
    uint32_t prefix = 0, mask = 0;
    for (int pass = 0; pass < 3; ++pass) {
        const uint32_t shift = pass == 0 ? 21u : pass == 1 ? 10u : 0u;
        const uint32_t bins = pass == 2 ? 1024u : 2048u;
        for (uint32_t i = tid; i < bins; i += kClusterThreads) hist[i] = 0;
        __syncthreads();
        for (uint32_t i = tid; i < cnt; i += kClusterThreads) {
            const uint32_t k = keys[i];
            if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & (bins - 1u)], 1u);
        }
        cluster.sync();
        if (rank == 0) {
            // four bins a thread, all CTAs' counts
            uint32_t m[4] = {0, 0, 0, 0};
            if (4 * tid < bins)
                for (uint32_t c = 0; c < C; ++c) {
                    const uint4 v = *reinterpret_cast<const uint4 *>(
                        cluster.map_shared_rank(hist, c) + 4 * tid);
                    m[0] += v.x;
                    m[1] += v.y;
                    m[2] += v.z;
                    m[3] += v.w;
                }
            uint32_t before = block_exclusive(m[0] + m[1] + m[2] + m[3], 0u, S.warp_v,
                                              [](uint32_t a, uint32_t b) { return a + b; });
            const uint32_t k = S.k;
            __syncthreads();
#pragma unroll
            for (uint32_t e = 0; e < 4; ++e) {
                if (before < k && k <= before + m[e]) {
                    S.prefix = prefix | ((4 * tid + e) << shift);
                    S.k = k - before;
                }
                before += m[e];
            }
            if (pass == 0 && tid < C) atomicMin(&S.min_key, cluster.map_shared_rank(&S, tid)->min_key);
        }
        cluster.sync();
        prefix = S0->prefix;
        mask |= (bins - 1u) << shift;
    }
    const uint32_t cut = prefix, mnk = S0->min_key;
    const float vlo = fval(mnk), vhi = fval(cut);
    float thr = vhi;  // no gap: every latency a hit
    if (cut != mnk) {
        // one round of buckets [w0, w0 + kGapBuckets) of `nb` over [vlo, vhi];
        // rank 0 adds the largest gap so far
        auto round = [&](uint32_t w0, uint32_t nb, float scale) {
            for (uint32_t i = tid; i < kGapBuckets; i += kClusterThreads) bucket[i] = make_uint2(0xFFFFFFFFu, 0u);
            __syncthreads();
            for (uint32_t i = tid; i < cnt; i += kClusterThreads) {
                const uint32_t k = keys[i];
                if (k > cut) continue;
                uint32_t bi = (uint32_t)((fval(k) - vlo) * scale);
                if (bi >= nb) bi = nb - 1;
                bi -= w0;
                if (bi >= kGapBuckets) continue;
                // (a look first: most latencies move neither end)
                if (k < bucket[bi].x) atomicMin(&bucket[bi].x, k);
                if (k > bucket[bi].y) atomicMax(&bucket[bi].y, k);
            }
            cluster.sync();
            if (rank == 0) {
                constexpr uint32_t B = kGapBuckets / kClusterThreads;  // buckets a thread
                uint2 m[B];
                uint32_t top = 0;
#pragma unroll
                for (uint32_t e = 0; e < B; ++e) m[e] = make_uint2(0xFFFFFFFFu, 0u);
                for (uint32_t c = 0; c < C; ++c) {
                    const uint4 *const r = cluster.map_shared_rank(S.bucket4, c) + B / 2 * tid;
#pragma unroll
                    for (uint32_t e = 0; e < B; e += 2) {
                        const uint4 a = r[e / 2];
                        m[e] = make_uint2(min(m[e].x, a.x), max(m[e].y, a.y));
                        m[e + 1] = make_uint2(min(m[e + 1].x, a.z), max(m[e + 1].y, a.w));
                        top = max(top, max(a.y, a.w));
                    }
                }
                const auto larger = [](uint32_t a, uint32_t b) { return max(a, b); };
                uint32_t prev = max(block_exclusive(top, 0u, S.warp_v, larger), S.carry);
                if (tid == 0) S.best = 0;
                const uint32_t last = max(prev, top);  // (the last thread's: the carry)
                float g = 0.0f, lo = 0.0f, hi = 0.0f;
                uint32_t at = 0;
#pragma unroll
                for (uint32_t e = 0; e < B; ++e) {
                    if (m[e].x == 0xFFFFFFFFu) continue;
                    if (prev) {
                        const float a = fval(prev), c = fval(m[e].x), d = c - a;
                        if (d > g) {
                            g = d;
                            lo = a;
                            hi = c;
                            at = B * tid + e;
                        }
                    }
                    prev = m[e].y;
                }
                __syncthreads();
                // the largest gap, the lowest one on ties
                const unsigned long long key =
                    g > 0.0f ? ((unsigned long long)__float_as_uint(g) << 32) | (0xFFFFFFFFu - at) : 0ull;
                if (key) atomicMax(&S.best, key);
                __syncthreads();
                if (key && key == S.best && g > S.gap) {
                    S.gap = g;
                    S.lo = lo;
                    S.hi = hi;
                    S.found = 1;
                }
                if (tid == kClusterThreads - 1) S.carry = last;
                __syncthreads();
            }
            cluster.sync();
        };
        const float range = vhi - vlo, width = range * (1.0f / kGapBuckets), coarse = (float)kGapBuckets / range;
        bool done = false;
        if (isfinite(range) && range > 1e-30f && isfinite(coarse)) {
            round(0, kGapBuckets, coarse);
            done = S0->gap > 1.01f * width;
            cluster.sync();
            if (!done && rank == 0 && tid == 0) {
                S.carry = 0;
                S.gap = 0.0f;
                S.found = 0;
            }
            cluster.sync();
        }
        if (!done) {
            const uint32_t nb = 2 * keep;
            const float scale = (float)nb / (vhi - vlo);
            for (uint32_t w0 = 0; w0 < nb; w0 += kGapBuckets) round(w0, nb, scale);
        }
        if (S0->found) thr = (S0->lo + S0->hi) * 0.5f;
    }
    if (rank == 0 && tid == 0) {
        meta[o] = ObsMeta{cut, mnk, cut == mnk ? 0u : 2u * keep, thr};
        if (thresh_out) thresh_out[o] = thr;
    }
    if (bits) {
        uint32_t *const out = bits + word_offsets[o] + (first >> 5);
        const uint32_t padded = (cnt + 31u) & ~31u;
        for (uint32_t i = tid; i < padded; i += kClusterThreads) {
            const uint32_t v = __ballot_sync(kFull, i < cnt && fval(keys[i]) > thr);
            if ((tid & 31) == 0) out[i >> 5] = v;
        }
    }
    cluster.sync();  // rank 0's shared memory outlives the others' reads
}

// CTAs of an observation's cluster (0: too long for one), and its launch: as
// few as hold it, more while its CTAs have above 8K latencies each and the
// call's CTAs still fit the GPU side by side, two to an SM (every CTA more
// shortens the passes and lengthens rank 0's sums: 64 observations of up to
// 64K latencies took 131 us with eight CTAs of 1024 threads each).
uint32_t cluster_ctas(uint64_t max_len, uint64_t n_obs, int sms) {
    uint32_t c = 1;
    while (c < kClusterMax && (max_len > (uint64_t)c * (kClusterMaxKeys - 32) ||
                               (max_len > 8192ull * c && n_obs * c <= (uint64_t)std::max(sms, 1))))
        c *= 2;
    return max_len <= (uint64_t)c * (kClusterMaxKeys - 32) ? c : 0;
}

cudaError_t launch_cluster(const float *lat, const uint64_t *offsets, uint32_t n_obs, uint64_t max_len,
                           ObsMeta *meta, float *thresh_out, uint32_t *bits,
                           const uint64_t *word_offsets, cudaStream_t st, uint32_t C) {
    const size_t per = ((max_len + C - 1) / C + 31) & ~size_t(31);
    const size_t smem = kClusterSmemBase + 4 * per;
    cudaError_t e = cudaFuncSetAttribute(classify_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(kClusterSmemBase + 4 * kClusterMaxKeys));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(n_obs * C);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, classify_cluster_kernel, lat, offsets, max_len, meta, thresh_out, bits,
                              word_offsets);
}

// One CTA per observation: cut value by radix select, minimum, bucket init.
__global__ void __launch_bounds__(1024) select_cut_kernel(const float *lat,
                                                          const uint64_t *offsets,
                                                          uint64_t max_len, ObsMeta *meta,
                                                          uint2 *buckets) {
    __shared__ uint32_t hist[256];
    __shared__ uint32_t s_prefix, s_mask, s_k, s_min;
    const uint32_t o = blockIdx.x;
    const uint64_t b0 = offsets[o], n = offsets[o + 1] - b0;
    const float *x = lat + b0;
    const uint64_t keep = n - n / 200;
    if (threadIdx.x == 0) {
        s_prefix = 0;
        s_mask = 0;
        s_k = (uint32_t)keep;
        s_min = 0xFFFFFFFFu;
    }
    __syncthreads();
    if (n == 0) {
        if (threadIdx.x == 0) meta[o] = ObsMeta{0, 0, 0, 0.0f};
        return;
    }
    if (n > max_len) {
        // the observation's bucket slice holds 2 * max_len buckets: an
        // observation longer than the caller's max_len is refused (NaN cut, so
        // no latency is above it and every bit stays 0) instead of writing
        // into the next observation's slice or past the scratch
        if (threadIdx.x == 0) meta[o] = ObsMeta{0, 0, 0, __int_as_float(0x7FC00000)};
        return;
    }
    for (int pass = 0; pass < 4; ++pass) {
        const int shift = 24 - 8 * pass;
        for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
        __syncthreads();
        const uint32_t prefix = s_prefix, mask = s_mask;
        uint32_t mn = 0xFFFFFFFFu;
        // (counts go up by one: lanes with the same digit are added up by the
        // shared-memory increment itself)
        for (uint64_t i = threadIdx.x; i < n; i += blockDim.x) {
            const uint32_t k = fkey(x[i]);
            if (pass == 0) mn = min(mn, k);
            if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], 1u);
        }
        if (pass == 0) {
            mn = __reduce_min_sync(kFull, mn);
            if ((threadIdx.x & 31) == 0) atomicMin(&s_min, mn);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t cum = 0, k = s_k;
            for (uint32_t d = 0; d < 256; ++d) {
                if (cum + hist[d] >= k) {
                    s_prefix = prefix | (d << shift);
                    s_mask = mask | (255u << shift);
                    s_k = k - cum;
                    break;
                }
                cum += hist[d];
            }
        }
        __syncthreads();
    }
    const uint32_t cut = s_prefix, mnk = s_min;
    const uint32_t nb = (cut == mnk) ? 0u : (uint32_t)(2 * keep);
    uint2 *bk = buckets + (uint64_t)o * 2 * max_len;
    for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x) bk[i] = make_uint2(0xFFFFFFFFu, 0u);
    if (threadIdx.x == 0) meta[o] = ObsMeta{cut, mnk, nb, fval(cut)};
}

// Kept values into buckets (min / max key per bucket).
__global__ void bucket_kernel(const float *lat, const uint64_t *offsets, uint64_t max_len,
                              const ObsMeta *meta, uint2 *buckets) {
    const uint32_t o = blockIdx.y;
    const ObsMeta m = meta[o];
    if (m.nb == 0) return;
    const uint64_t b0 = offsets[o], n = offsets[o + 1] - b0;
    const float lo = fval(m.min_key), hi = fval(m.cut_key);
    const float scale = (float)m.nb / (hi - lo);
    uint2 *bk = buckets + (uint64_t)o * 2 * max_len;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const float v = lat[b0 + i];
        const uint32_t k = fkey(v);
        if (k > m.cut_key) continue;
        uint32_t bi = (uint32_t)((v - lo) * scale);
        if (bi >= m.nb) bi = m.nb - 1;
        atomicMin(&bk[bi].x, k);
        atomicMax(&bk[bi].y, k);
    }
}

struct GapPart {
    uint32_t first_min, last_max;  // keys; first_min = 0xFFFFFFFF when empty
    float gap, lo, hi;
};

// One CTA per observation: the largest gap between consecutive non-empty
// buckets, first one on ties; each thread scans a contiguous range, then one
// warp-serial pass joins the ranges in order.
__global__ void __launch_bounds__(1024) gap_kernel(uint64_t max_len, ObsMeta *meta,
                                                   const uint2 *buckets, float *thresh_out) {
    __shared__ GapPart part[1024];
    const uint32_t o = blockIdx.x;
    ObsMeta m = meta[o];
    if (m.nb == 0) {
        if (threadIdx.x == 0 && thresh_out) thresh_out[o] = m.thr;
        return;
    }
    const uint2 *bk = buckets + (uint64_t)o * 2 * max_len;
    const uint32_t per = (m.nb + blockDim.x - 1) / blockDim.x;
    const uint32_t beg = threadIdx.x * per;
    const uint32_t end = min(m.nb, beg + per);
    GapPart p{0xFFFFFFFFu, 0u, -1.0f, 0.0f, 0.0f};
    for (uint32_t i = beg; i < end; ++i) {
        const uint2 b = bk[i];
        if (b.x == 0xFFFFFFFFu) continue;
        if (p.first_min == 0xFFFFFFFFu) {
            p.first_min = b.x;
        } else {
            const float a = fval(p.last_max), c = fval(b.x);
            const float g = c - a;
            if (g > p.gap) { p.gap = g; p.lo = a; p.hi = c; }
        }
        p.last_max = b.y;
    }
    part[threadIdx.x] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
        float best = 0.0f, lo = 0.0f, hi = 0.0f;
        bool found = false, have_prev = false;
        uint32_t prev_max = 0;
        for (uint32_t t = 0; t < blockDim.x; ++t) {
            const GapPart q = part[t];
            if (q.first_min == 0xFFFFFFFFu) continue;
            if (have_prev) {
                const float a = fval(prev_max), c = fval(q.first_min);
                const float g = c - a;
                if (g > best) { best = g; lo = a; hi = c; found = true; }
            }
            if (q.gap > best) { best = q.gap; lo = q.lo; hi = q.hi; found = true; }
            prev_max = q.last_max;
            have_prev = true;
        }
        m.thr = found ? (lo + hi) * 0.5f : fval(m.cut_key);
        meta[o].thr = m.thr;
        if (thresh_out) thresh_out[o] = m.thr;
    }
}

// Miss bits of segment s against the threshold of observation s / per_seg
// (per_seg segments per observation; 0: one pooled threshold)
// or of observation 0 (every segment pooled into one observation).
__global__ void bits_kernel(const float *lat, const uint64_t *seg_offsets, int per_seg,
                            uint32_t n_seg, const ObsMeta *meta, uint32_t *bits,
                            const uint64_t *word_offsets) {
    const uint32_t s = blockIdx.y;
    const float thr = meta[per_seg ? s / (uint32_t)per_seg : 0].thr;
    const uint64_t b0 = seg_offsets[s], n = seg_offsets[s + 1] - b0;
    const uint64_t words = (n + 31) / 32;
    const uint64_t wo = word_offsets[s];
    const int lane = threadIdx.x & 31;
    const uint64_t warp = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t w = 4 * warp; w < words; w += 4 * nwarps) {
        // four words' latencies in flight
        bool miss[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint64_t i = (w + q) * 32 + lane;
            miss[q] = i < n && lat[b0 + i] > thr;
        }
        uint32_t v = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t x = __ballot_sync(kFull, miss[q]);
            if (lane == q) v = x;
        }
        if (lane < 4 && w + lane < words) bits[wo + w + lane] = v;
    }
}

// Canonical pick: one block.
__device__ __forceinline__ bool better(const pchase_geom *g, const uint64_t *d, uint32_t x,
                                       uint32_t y) {
    if (d[x] != d[y]) return d[x] < d[y];
    const pchase_geom &a = g[x], &b = g[y];
    if (a.policy != b.policy) return a.policy < b.policy;
    if (a.line_bytes != b.line_bytes) return a.line_bytes > b.line_bytes;
    if (a.ways != b.ways) return a.ways < b.ways;
    if (a.C_bytes != b.C_bytes) return a.C_bytes < b.C_bytes;
    return x < y;
}

__global__ void __launch_bounds__(1024) pick_kernel(const pchase_geom *geoms, const uint64_t *dist,
                                                    uint32_t n, uint32_t *pick) {
    // block o picks for observation o: distances dist + o * n
    dist += (size_t)blockIdx.x * n;
    pick += 2ull * blockIdx.x;
    __shared__ uint32_t best[1024];
    __shared__ uint32_t count;
    uint32_t b = 0xFFFFFFFFu;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x)
        if (b == 0xFFFFFFFFu || better(geoms, dist, i, b)) b = i;
    best[threadIdx.x] = b;
    if (threadIdx.x == 0) count = 0;
    __syncthreads();
    for (uint32_t s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            const uint32_t x = best[threadIdx.x], y = best[threadIdx.x + s];
            if (y != 0xFFFFFFFFu && (x == 0xFFFFFFFFu || better(geoms, dist, y, x)))
                best[threadIdx.x] = y;
        }
        __syncthreads();
    }
    const uint32_t w = best[0];
    uint32_t c = 0;
    if (w != 0xFFFFFFFFu)
        for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) c += dist[i] == dist[w];
    atomicAdd(&count, c);
    __syncthreads();
    if (threadIdx.x == 0) {
        pick[0] = w == 0xFFFFFFFFu ? n : w;
        pick[1] = count;
    }
}

}  // namespace

size_t classify_meta_bytes(uint32_t n_obs) { return ((size_t)n_obs * sizeof(ObsMeta) + 255) & ~size_t(255); }

size_t classify_bucket_bytes(uint32_t n_obs, uint64_t max_len) {
    return (size_t)n_obs * 2 * (max_len ? max_len : 1) * sizeof(uint2);
}

// Thresholds for n_obs observations (lat + offsets), buckets in `work`.
cudaError_t classify_thresholds(const float *lat, const uint64_t *offsets, uint32_t n_obs,
                                uint64_t max_len, void *meta_mem, void *bucket_mem,
                                float *thresh_out, cudaStream_t st, int sms) {
    ObsMeta *meta = static_cast<ObsMeta *>(meta_mem);
    uint2 *bk = static_cast<uint2 *>(bucket_mem);
    if (const uint32_t C = cluster_ctas(max_len, n_obs, sms))
        return launch_cluster(lat, offsets, n_obs, max_len, meta, thresh_out, nullptr, nullptr, st, C);
    select_cut_kernel<<<n_obs, 1024, 0, st>>>(lat, offsets, max_len, meta, bk);
    uint32_t gx = (uint32_t)((max_len + 255) / 256);
    const uint32_t cap = (uint32_t)(sms > 0 ? sms : 1) * 8;
    if (gx > cap) gx = cap;
    if (gx < 1) gx = 1;
    bucket_kernel<<<dim3(gx, n_obs), 256, 0, st>>>(lat, offsets, max_len, meta, bk);
    gap_kernel<<<n_obs, 1024, 0, st>>>(max_len, meta, bk, thresh_out);
    return cudaGetLastError();
}

cudaError_t classify_bits(const float *lat, const uint64_t *seg_offsets, int per_seg,
                          uint32_t n_seg, uint64_t max_seg_len, const void *meta_mem,
                          uint32_t *bits, const uint64_t *word_offsets, cudaStream_t st,
                          int sms) {
    uint32_t gx = (uint32_t)((max_seg_len + 1023) / 1024);
    const uint32_t cap = (uint32_t)(sms > 0 ? sms : 1) * 8;
    if (gx > cap) gx = cap;
    if (gx < 1) gx = 1;
    bits_kernel<<<dim3(gx, n_seg), 256, 0, st>>>(lat, seg_offsets, per_seg, n_seg,
                                                  static_cast<const ObsMeta *>(meta_mem), bits,
                                                  word_offsets);
    return cudaGetLastError();
}

// Thresholds and each observation's own bits.
cudaError_t classify_all(const float *lat, const uint64_t *offsets, uint32_t n_obs, uint64_t max_len,
                         void *meta_mem, void *bucket_mem, float *thresh_out, uint32_t *bits,
                         const uint64_t *word_offsets, cudaStream_t st, int sms) {
    if (const uint32_t C = cluster_ctas(max_len, n_obs, sms))
        return launch_cluster(lat, offsets, n_obs, max_len, static_cast<ObsMeta *>(meta_mem), thresh_out, bits,
                              word_offsets, st, C);
    cudaError_t e = classify_thresholds(lat, offsets, n_obs, max_len, meta_mem, bucket_mem, thresh_out, st, sms);
    if (e == cudaSuccess)
        e = classify_bits(lat, offsets, 1, n_obs, max_len, meta_mem, bits, word_offsets, st, sms);
    return e;
}

cudaError_t canonical_pick(const pchase_geom *geoms, const uint64_t *dist, uint32_t n,
                           uint32_t *pick, cudaStream_t st, uint32_t n_obs) {
    pick_kernel<<<n_obs ? n_obs : 1, 1024, 0, st>>>(geoms, dist, n, pick);
    return cudaGetLastError();
}

// Segment and word offsets of n_obs observations laid out back to back, each
// L latencies in plan-trace order (T traces, seg[T + 1], owo[T]).
__global__ void batch_offsets_kernel(const uint64_t *seg, const uint64_t *owo, uint32_t T,
                                     uint32_t n_obs, uint64_t L, uint64_t obs_words,
                                     uint64_t *obs_off, uint64_t *seg_out, uint64_t *wo_out) {
    const uint64_t n = (uint64_t)n_obs * T;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t o = i / T, t = i % T;
        if (i == n) {
            seg_out[n] = n_obs * L;
        } else {
            seg_out[i] = o * L + seg[t];
            wo_out[i] = o * obs_words + owo[t];
        }
        if (i <= n_obs) obs_off[i] = i * L;
    }
}

cudaError_t batch_offsets(const uint64_t *seg, const uint64_t *owo, uint32_t T, uint32_t n_obs,
                          uint64_t L, uint64_t obs_words, uint64_t *obs_off, uint64_t *seg_out,
                          uint64_t *wo_out, cudaStream_t st) {
    const uint64_t n = (uint64_t)n_obs * T + 1;
    const unsigned blocks = (unsigned)std::min<uint64_t>((n + 255) / 256, 1024);
    batch_offsets_kernel<<<blocks, 256, 0, st>>>(seg, owo, T, n_obs, L, obs_words, obs_off,
                                                 seg_out, wo_out);
    return cudaGetLastError();
}

// ------------------------------------------------ classification without allocation
// Scratch of pchase_classify_noalloc: a fixed array in the library's own
// device memory, shared by every call on a device and kept until the process
// exits.  Host code cannot use the name g_noalloc_scratch as an address: it
// names a host-side stand-in, so the device address is looked up once per
// device with cudaGetSymbolAddress.
constexpr size_t kNoallocScratchBytes = 8u << 20;
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoallocScratchBytes];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[kMaxDevices];

// Device address of the scratch array for the current device (set up on the
// first call per device).
cudaError_t noalloc_scratch(void **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}
}  // namespace

}  // namespace pchase

extern "C" size_t pchase_classify_noalloc_limit_bytes(void) {
    return pchase::kNoallocScratchBytes;
}

extern "C" int pchase_classify_noalloc(const float *lat, const uint64_t *offsets, uint32_t n_obs,
                                       uint64_t max_len, uint32_t *bits_out,
                                       const uint64_t *bit_word_offsets, float *thresh_out,
                                       pchase_stream_t stream) {
    using namespace pchase;
    if (n_obs == 0) return PCHASE_OK;
    if (!lat || !offsets || !bits_out || !bit_word_offsets)
        return set_last_error(PCHASE_EINVAL, "pchase_classify_noalloc: NULL argument");
    const size_t meta = classify_meta_bytes(n_obs);
    const size_t bk = (classify_bucket_bytes(n_obs, max_len) + 255) & ~size_t(255);
    if (max_len > (kNoallocScratchBytes >> 4) || n_obs > (kNoallocScratchBytes >> 4) ||
        meta + bk > kNoallocScratchBytes)
        return set_last_error(PCHASE_ERANGE,
                              "pchase_classify_noalloc: n_obs * max_len too large for the "
                              "8 MiB static scratch (need 16 * n_obs * (max_len + 1) bytes, "
                              "rounded up); use pchase_classify with a workspace");
    void *scratch = nullptr;
    cudaError_t e = noalloc_scratch(&scratch);
    if (e != cudaSuccess)
        return set_last_error(PCHASE_ECUDA, "pchase_classify_noalloc: cudaGetSymbolAddress failed");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    uint8_t *w = static_cast<uint8_t *>(scratch);
    // the kernels write every metadata entry and initialise every bucket they
    // read, so nothing left by an earlier call is consumed
    e = classify_all(lat, offsets, n_obs, max_len, w, w + meta, thresh_out, bits_out, bit_word_offsets, st,
                     sms);
    if (e != cudaSuccess) return set_last_error(PCHASE_ECUDA, cudaGetErrorString(e));
    return PCHASE_OK;
}
