// Uniform chains: the items whose trace is Listing 1's chain with a stride that
// divides the array (every pass of the array visits the same lines in the same
// order), replayed without stepping a cache through their accesses.
//
// Over such a chain the accesses of one pass visit nl distinct lines in
// increasing order; number them kk = 0 .. nl - 1 (consecutive lines when the
// stride is at most a line, every st-th line when it is a multiple of one).
// Line kk falls in the set class kk mod T' (T' = T / gcd(st, T)), so each set
// is walked cyclically over the lines of its class, n of them:
//   - the first pass misses once per line (its first access, a run head);
//   - n <= a: the set holds all of them from then on, under every policy;
//   - n > a under LRU and FIFO (and one way under any policy): a line is
//     evicted by the n - 1 >= a other lines before it returns, so every run
//     head misses.  This is Eq. (2) of Sec. 4.1 made exact: class c overflows
//     when c < nl - a T';
//   - n > a under RANDOM and WEIGHTED: which lines a pass finds depends on the
//     victims, so these sets are played, each by itself, from their n lines and
//     the victim sequence (below).
// An analytic chain is uniform by definition.  An index array is compared
// with the chain its descriptor states, element by element, on every run; an
// item whose trace differs anywhere is left to the simulator's units, and the
// units of the items done here return at once.
//
// What bounds it: uniform_prep_kernel reads 4 B per access (HBM), the output
// kernel writes a bit per access; the played sets are chains of dependent
// events, so they are cut into one warp per set (or 32 small sets), long small
// sets into segments, and the costliest start first.  Against stepping the same
// items in the units, batches of 4096 items (0.63 G accesses, index arrays) went
// from 44 to 9-15 ms and the benchmark's from 21.8 to 4.4 (their longest played
// sets all but 1.1 ms of it), a 384-item batch of short traces from 519 to 155 us, matching 1308 candidates against 108 traces from 3.54 to
// 0.18 ms.
#include <algorithm>

#include "pchase_internal.cuh"

namespace pchase {

namespace {

extern __shared__ __align__(16) uint8_t u_smem[];

__device__ __forceinline__ uint32_t lt_mask() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// The chain of an eligible item, from any of its units.
struct Chain {
    uint32_t len, warmup;
    uint32_t per;    // accesses of one pass
    uint32_t s, lb;  // stride in elements, line shift (line = element >> lb)
    uint32_t nl;     // lines of one pass
    uint32_t st;     // line step (1: consecutive lines)
    bool strided;    // stride of a line or more: access k of a pass is line k
    uint32_t T, Tp;  // sets, classes
    uint32_t a, m;
    uint32_t thr;    // classes [0, thr) overflow (mapping 0)
    bool rnd;        // overflowing sets are played (RANDOM, WEIGHTED)
    uint32_t sm, ss1, ss2;  // division by the stride (DivMagic), below a line

    __device__ __forceinline__ explicit Chain(const SimItem &it) {
        len = it.len;
        warmup = it.warmup;
        s = it.stride;
        lb = it.lsh & 255u;
        per = s ? it.n_elems / s : 1u;
        strided = s > (1u << lb);
        nl = strided ? per : (((per - 1u) * s) >> lb) + 1u;
        st = strided ? s >> lb : 1u;
        T = it.kcnt > 1 ? it.gsets : it.sets;
        a = it.ways;
        m = (it.lsh >> 8) & 255u;
        // T / gcd(st, T); a line step is mostly a power of two
        if ((st & (st - 1u)) == 0u) {
            Tp = T >> min(__ffs(st) - 1, __ffs(T) - 1);
        } else {
            uint32_t x = st % T, y = T;
            while (x) {
                const uint32_t r = y % x;
                y = x;
                x = r;
            }
            Tp = T / y;
        }
        const uint64_t room = (uint64_t)a * Tp;
        thr = nl > room ? (uint32_t)min((uint64_t)Tp, nl - room) : 0u;
        rnd = it.policy >= PCHASE_RANDOM && a > 1;
        sm = ss1 = ss2 = 0;
    }
    // miss bits of accesses [t0, t0 + 32) (the played sets' only in the first
    // pass); held: no set misses after the first pass, all: every one does
    __device__ __forceinline__ uint32_t word(uint32_t t0, bool held, bool all) const {
        if (nl == 1u) return t0 == 0u ? 1u : 0u;
        uint32_t bits = 0, k = t0 % per;
        if (strided) {
            // every access is a head; x: its line's class
            uint32_t x = k % Tp;
            if (Tp >= 8u) {
                // runs of overflowing classes and of the others, a few a word
                for (uint32_t i = 0; i < 32u;) {
                    const bool cold = t0 + i < per, miss = cold || (!held && (all || x < thr));
                    uint32_t r = cold || all || held ? 32u : x < thr ? thr - x : Tp - x;
                    r = min(min(r, per - k), 32u - i);
                    bits |= (miss ? kFull >> (32u - r) : 0u) << i;
                    i += r;
                    k += r;
                    x += r;
                    if (k == per) k = x = 0;
                    if (x >= Tp) x = cold || all || held ? x % Tp : 0u;
                }
                return bits;
            }
#pragma unroll 8
            for (uint32_t i = 0; i < 32; ++i) {
                const bool miss = t0 + i < per || (!held && (all || x < thr));
                bits |= (miss ? 1u : 0u) << i;
                x = x + 1u == Tp ? 0u : x + 1u;
                if (++k == per) k = x = 0;
            }
            return bits;
        }
        // heads from the first one at or after t0
        uint32_t base = t0 - k, kk = k ? (((k - 1u) * s) >> lb) + 1u : 0u;
        if (kk == nl) {
            kk = 0;
            base += per;
        }
        uint32_t x = m || all || held ? 0u : kk % Tp;
        for (;;) {
            const uint32_t i = base + first(kk) - t0;
            if (i >= 32u) break;
            const bool miss = base == 0u || (!held && (all || (m ? over(kk) : x < thr)));
            bits |= (miss ? 1u : 0u) << i;
            x = x + 1u == Tp ? 0u : x + 1u;
            if (++kk == nl) {
                kk = x = 0;
                base += per;
            }
        }
        return bits;
    }
    // before first(): the stride's DivMagic (make_div_magic)
    __device__ __forceinline__ void prepare_first() {
        if (strided || s == 0) return;
        const uint32_t l = 32u - (uint32_t)__clz(s - 1u);  // ceil(log2 s), 0 for s = 1
        sm = (uint32_t)((((1ull << l) - s) << 32) / s + 1u);
        ss1 = min(l, 1u);
        ss2 = l > 1u ? l - 1u : 0u;
    }
    // lines of class c (mapping 0)
    __device__ __forceinline__ uint32_t lines_of(uint32_t c) const { return (nl - c - 1u) / Tp + 1u; }
    // whether the set of visited line kk overflows
    __device__ __forceinline__ bool over(uint32_t kk) const {
        if (m == 0) return kk % Tp < thr;
        // set = (line >> m) mod T, consecutive lines: whole blocks of 2^m
        // lines, and the part block at the end
        const uint32_t u = (kk >> m) % T, q = nl >> m;
        uint32_t n = (q > u ? (q - 1u - u) / T + 1u : 0u) << m;
        if (q % T == u) n += nl & ((1u << m) - 1u);
        return n > a;
    }
    // first access of line kk within a pass
    // (arrays of at most 2^31 elements: the sum does not wrap)
    __device__ __forceinline__ uint32_t first(uint32_t kk) const {
        return strided ? kk : div_q((kk << lb) + s - 1u, sm, ss1, ss2);
    }
};

__device__ __forceinline__ bool taken(const SimItem &it, const uint32_t *bad) {
    return ((it.lsh >> kUniformBit) & 1u) && bad[it.obs] == 0u;
}

// Clears the miss counts and compares the index arrays with their chains:
// 16-byte loads, four of a lane in flight, `parts` warps to a trace.  bad[t] is
// set where trace t differs.  HBM-bound on 4 B per access.
__global__ void __launch_bounds__(256) uniform_prep_kernel(const SimItem *__restrict__ items,
                                                           const uint32_t *__restrict__ trace_unit,
                                                           uint32_t n_trace, uint32_t parts,
                                                           uint64_t n_items, uint64_t *counts,
                                                           uint32_t *bad, uint32_t *head) {
    const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const uint64_t nthr = (uint64_t)gridDim.x * blockDim.x;
    if (head)  // the workspace's counters, unless a memset cleared them
        for (uint64_t i = tid; i < kQueueHeader / 4; i += nthr) head[i] = 0;
    if (counts)
        for (uint64_t i = tid; i < 2 * n_items; i += nthr) counts[i] = 0;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t tasks = (uint64_t)n_trace * parts;
    for (uint64_t task = tid >> 5; task < tasks; task += nthr >> 5) {
        const uint32_t tr = (uint32_t)(task / parts), part = (uint32_t)(task % parts);
        const uint32_t unit = trace_unit[tr];
        if (unit == 0xFFFFFFFFu) {
            if (parts == 1u && lane == 0) bad[tr] = 0;
            continue;
        }
        const SimItem &it = items[unit];
        const uint32_t *const p = it.idx;
        const uint32_t len = it.len, s = it.stride;
        const uint32_t per = s ? it.n_elems / s : 1u;
        // [0, e0) up to the first 16-byte boundary, quads from there, a tail
        const uint32_t e0 = min(len, (uint32_t)((0u - (uint32_t)(reinterpret_cast<uintptr_t>(p) >> 2)) & 3u));
        const uint32_t nq = (len - e0) >> 2, tail = e0 + 4u * nq;
        bool wrong = false;
        if (part == 0) {
            if (lane < e0) wrong = p[lane] != (lane % per) * s;
            if (tail + lane < len) wrong = wrong || p[tail + lane] != ((tail + lane) % per) * s;
        }
        const uint32_t chunk = (nq + parts - 1u) / parts;
        const uint32_t q0 = min(nq, part * chunk), q1 = min(nq, q0 + chunk);
        const uint4 *const v = reinterpret_cast<const uint4 *>(p + e0);
        auto differs = [&](uint4 x, uint32_t k) {
            bool w = x.x != k * s;
            k = k + 1u == per ? 0u : k + 1u;
            w = w || x.y != k * s;
            k = k + 1u == per ? 0u : k + 1u;
            w = w || x.z != k * s;
            k = k + 1u == per ? 0u : k + 1u;
            return w || x.w != k * s;
        };
        uint32_t k = (e0 + 4u * (q0 + lane)) % per;  // place of this lane's quad in its pass
        const uint32_t inc = 128u % per;             // a warp's quads hold 128 accesses
        uint32_t q = q0 + lane;
        for (; q + 96u < q1; q += 128u) {
            uint4 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = __ldcs(v + q + 32u * u);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                wrong = differs(x[u], k) || wrong;
                k += inc;
                k -= k >= per ? per : 0u;
            }
            if (wrong) break;
        }
        for (; !wrong && q < q1; q += 32u) {
            wrong = differs(__ldcs(v + q), k);
            k += inc;
            k -= k >= per ? per : 0u;
        }
        // (a warp that has the trace to itself says so either way)
        const bool any = __any_sync(kFull, wrong);
        if (lane == 0 && parts == 1u) bad[tr] = any ? 1u : 0u;
        else if (lane == 0 && any) atomicOr(bad + tr, 1u);
    }
}

// The words of every caller item: an item taken here gets its final words and
// counts (or its Hamming distance), the played sets' later misses apart; any
// other one is cleared for the simulator's units.  A warp takes 32 words at a
// time, one per lane.  A lane goes through its word's run heads (its accesses,
// where each is one): up to 32 short turns for 32 words, where a vote per word
// took 32 longer ones (a pass over the texture and Fermi sweeps of 9.6K items
// 284 -> 91 us; this kernel on the 4096-item batch 1519 -> 421 us).
__global__ void __launch_bounds__(256) uniform_out_kernel(const SimItem *__restrict__ items,
                                                          const uint32_t *__restrict__ units,
                                                          uint64_t n_units, uint32_t parts,
                                                          SimOut out, uint32_t *live) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    const bool ham = out.dist != nullptr;
    const uint32_t nrep = ham && out.n_rep ? out.n_rep : 1u;
    for (uint64_t task = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
         task < n_units * parts; task += nw) {
        const uint64_t ui = task / parts;
        const uint32_t part = (uint32_t)(task % parts);
        const SimItem it = items[units ? units[ui] : ui];
        if (!it.lead) continue;
        const bool mine = taken(it, out.uniform_bad) &&
                          (!ham || ((it.lsh >> kUniformMatchBit) & 1u));
        if (!mine && part == 0 && lane == 0) atomicOr(live, 1u);
        if (!mine && ham) continue;
        const uint32_t nwords = (it.len + 31u) >> 5;
        const uint32_t chunk = ((nwords + parts - 1u) / parts + 31u) & ~31u;
        const uint32_t w0 = min(nwords, part * chunk), w1 = min(nwords, w0 + chunk);
        uint32_t *const bm =
            out.bitmaps ? out.bitmaps + (out.word_offsets ? out.word_offsets[it.out_item] : it.word_off)
                        : nullptr;
        if (!mine) {
            if (bm)
                for (uint32_t w = w0 + lane; w < w1; w += 32) bm[w] = 0;
            continue;
        }
        Chain ch(it);
        ch.prepare_first();
        const bool held = ch.rnd || (ch.m == 0 && ch.thr == 0);  // later passes: nothing here
        const bool all = !ch.rnd && ch.m == 0 && ch.thr >= ch.Tp;
        const bool ones = all && ch.strided && ch.nl > 1;
        const uint64_t ob = ham ? out.obs_word_offsets[it.obs] : 0;
        uint32_t tot = 0, aft = 0;
        uint32_t dsum = 0;
        for (uint32_t wb = w0; wb < w1; wb += 32) {
            uint32_t word = 0;
            if (ones) {
                word = kFull;
            } else if (!(held && (wb << 5) >= ch.per)) {
                word = ch.word((wb + lane) << 5, held, all);
            }
            const uint32_t w = wb + lane, t = w << 5;
            if (w < w1) {
                const uint32_t valid = ch.len - t >= 32u ? kFull : (1u << (ch.len - t)) - 1u;
                word &= valid;
                if (bm) bm[w] = word;
                tot += (uint32_t)__popc(word);
                const uint32_t before = ch.warmup <= t ? 0u : ch.warmup - t;
                aft += before >= 32u ? 0u : (uint32_t)__popc(word >> before);
                if (ham && nrep == 1u) dsum += (uint32_t)__popc(word ^ (out.observed[ob + w] & valid));
            }
            if (nrep > 1u) {
                for (uint32_t r = 0; r < nrep; ++r) {
                    uint32_t d = 0;
                    if (w < w1) {
                        const uint32_t valid = ch.len - t >= 32u ? kFull : (1u << (ch.len - t)) - 1u;
                        d = (uint32_t)__popc(word ^ (out.observed[r * out.rep_obs_stride + ob + w] & valid));
                    }
                    d = __reduce_add_sync(kFull, d);
                    if (lane == 0 && d)
                        atomicAdd(reinterpret_cast<unsigned long long *>(
                                      out.dist + r * out.rep_dist_stride + it.cand),
                                  (unsigned long long)d);
                }
            }
        }
        if (ham) {
            if (nrep == 1u) {
                dsum = __reduce_add_sync(kFull, dsum);
                if (lane == 0 && dsum)
                    atomicAdd(reinterpret_cast<unsigned long long *>(out.dist + it.cand),
                              (unsigned long long)dsum);
            }
        } else if (out.miss_counts) {
            tot = __reduce_add_sync(kFull, tot);
            aft = __reduce_add_sync(kFull, aft);
            if (lane == 0) {
                unsigned long long *mc =
                    reinterpret_cast<unsigned long long *>(out.miss_counts + 2ull * it.out_item);
                if (tot) atomicAdd(mc, (unsigned long long)tot);
                if (aft) atomicAdd(mc + 1, (unsigned long long)aft);
            }
        }
    }
}

// The matcher's groups: a candidate's capacity decides only whether the run
// heads after the first pass all miss, all hit or are split by class, so most
// candidates of one line size predict the same words for a trace (1308
// candidates x 108 traces, 141K items: 864 groups).  A CTA works out a group's
// distance from one observation and adds it to its candidates' (161 us item by
// item; 8 us so, and 30 for the items that have a word of their own).
__global__ void __launch_bounds__(256) uniform_match_kernel(const SimItem *__restrict__ items,
                                                            const UniformGroup *__restrict__ groups,
                                                            uint32_t n_groups,
                                                            const uint32_t *__restrict__ cands,
                                                            SimOut out, uint32_t *live) {
    __shared__ uint32_t sums[8];
    const uint32_t tid = threadIdx.x, rep = blockIdx.y;
    const uint32_t *const observed = out.observed + rep * out.rep_obs_stride;
    unsigned long long *const dist =
        reinterpret_cast<unsigned long long *>(out.dist + rep * out.rep_dist_stride);
    for (uint32_t b = blockIdx.x; b < n_groups; b += gridDim.x) {
        const UniformGroup g = groups[b];
        const SimItem &it = items[g.unit];
        if (!taken(it, out.uniform_bad)) {
            if (tid == 0) atomicOr(live, 1u);
            continue;
        }
        Chain ch(it);
        ch.prepare_first();
        const bool held = ch.rnd || ch.thr == 0, all = !held;
        const bool ones = all && ch.strided && ch.nl > 1;
        const uint32_t *const obs = observed + out.obs_word_offsets[it.obs];
        const uint32_t nwords = (ch.len + 31u) >> 5;
        uint32_t d = 0;
        for (uint32_t w = tid; w < nwords; w += 256u) {
            const uint32_t t = w << 5;
            const uint32_t valid = ch.len - t >= 32u ? kFull : (1u << (ch.len - t)) - 1u;
            uint32_t word = 0;
            if (ones) word = kFull;
            else if (!held || t < ch.per) word = ch.word(t, held, all);
            d += (uint32_t)__popc((word ^ obs[w]) & valid);
        }
        d = __reduce_add_sync(kFull, d);
        if ((tid & 31u) == 0) sums[tid >> 5] = d;
        __syncthreads();
        uint32_t total = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) total += sums[q];
        if (total)
            for (uint32_t c = tid; c < g.count; c += 256u)
                atomicAdd(dist + cands[g.first + c], (unsigned long long)total);
        __syncthreads();
    }
}

// Sinks of one warp's misses in the played sets.
struct Sink {
    uint32_t *bm;
    const uint32_t *obs;  // observed words in shared memory (matcher)
    uint32_t warmup;
    uint32_t tot = 0, aft = 0;
    int32_t dsum = 0;

    __device__ __forceinline__ void finish(const SimItem &it, const SimOut &out, uint32_t rep,
                                           uint32_t lane) {
        if (out.dist) {
            // first-pass misses aside, the output kernel took every later
            // access of these sets for a hit
            const int32_t d = (int32_t)__reduce_add_sync(kFull, (uint32_t)dsum);
            if (lane == 0 && d)
                atomicAdd(reinterpret_cast<unsigned long long *>(out.dist + rep * out.rep_dist_stride +
                                                                 it.cand),
                          (unsigned long long)(long long)d);
        } else if (out.miss_counts) {
            const uint32_t x = __reduce_add_sync(kFull, tot), y = __reduce_add_sync(kFull, aft);
            if (lane == 0) {
                unsigned long long *mc =
                    reinterpret_cast<unsigned long long *>(out.miss_counts + 2ull * it.out_item);
                if (x) atomicAdd(mc, (unsigned long long)x);
                if (y) atomicAdd(mc + 1, (unsigned long long)y);
            }
        }
    }
};

// A warp's sink; the matcher's observed words take the arena's first part.
__device__ __forceinline__ uint8_t *open_sink(Sink &sink, const SimItem &it, const Chain &ch, const SimOut &out,
                                              uint32_t rep, uint8_t *arena, uint32_t lane) {
    sink.bm = nullptr;
    sink.obs = nullptr;
    sink.warmup = ch.warmup;
    if (out.dist) {
        uint32_t *const ob = reinterpret_cast<uint32_t *>(arena);
        const uint32_t nwords = (ch.len + 31u) >> 5;  // at most kUniformMatchLen / 32
        const uint32_t *const src = out.observed + rep * out.rep_obs_stride + out.obs_word_offsets[it.obs];
        for (uint32_t w = lane; w < nwords; w += 32) ob[w] = src[w];
        __syncwarp();
        sink.obs = ob;
        arena += kUniformMatchLen / 8;
    } else if (out.bitmaps) {
        sink.bm = out.bitmaps + (out.word_offsets ? out.word_offsets[it.out_item] : it.word_off);
    }
    return arena;
}

// Small sets (n <= 32 lines): one set per group of G lanes, miss by miss.
// The set's state is a mask of the lines not held, line j at bit 31 - j; all
// accesses up to the next line not held are hits, so the next miss is the
// mask's next set bit below the last one's, or its top bit in the next pass.
// It fills the way of the next eviction, and that way's line leaves.  The
// victims do not depend on the outcome: the lanes of a group hash G of them at
// a time, and the line a miss evicts is loaded before the miss ahead of it is
// known (which is that line when the two ways are one).  What is left is the
// chain that bounds it, one miss to the next: find-leading-one, shift, two
// logic operations and a select.  Lane q keeps the group's q-th miss, so the
// bits, counts and distances are worked out for G misses at once.
//
// arena: uint8 occ[32 ways][32 lanes], uint32 toff[32 lines][32 lanes]
// Where a small set is: lines not held (gone), those of them ahead in this pass
// (below), the last miss's line p and its pass's first access.
struct SmallSet {
    uint32_t gone, below, base, p;
};

// G misses in a row.  wv: 32 times the way of this lane's (miss r of the
// group's); mine_p, mine_base: that miss.
template <int G>
__device__ __forceinline__ void small_round(SmallSet &st, uint8_t *occ, uint32_t wv, uint32_t per,
                                            uint32_t glane, uint32_t r, uint32_t &mine_p,
                                            uint32_t &mine_base) {
    uint32_t p = 0;
    uint32_t w = G == 1 ? wv : __shfl_sync(kFull, wv, glane);
    uint32_t ld = occ[w];  // line of way w, but for the miss ahead
    bool again = false;    // the miss ahead took way w too
#pragma unroll
    for (int q = 0; q < G; ++q) {
        // (the miss ahead took the same way: it is the line that leaves)
        const uint32_t old = again ? p : ld;
        const bool wrap = st.below == 0;
        const uint32_t x = wrap ? st.gone : st.below;
        st.base += wrap ? per : 0u;
        p = 31u - (uint32_t)__clz(x);
        uint32_t wn = 0;
        if (q + 1 < G) {
            wn = __shfl_sync(kFull, wv, glane + q + 1);
            ld = occ[wn];
            again = wn == w;
        }
        occ[w] = (uint8_t)p;
        const uint32_t ob = 1u << old;
        st.below = (st.gone | ob) & ~(kFull << p);
        st.gone = (st.gone | ob) & ~(1u << p);
        mine_p = r == (uint32_t)q ? p : mine_p;
        mine_base = r == (uint32_t)q ? st.base : mine_base;
        w = wn;
    }
    st.p = p;
}

// A miss at access t of each lane where `count`, a group's in order.
template <int G>
__device__ __forceinline__ void small_sink(Sink &sink, bool count, uint32_t t, uint32_t r) {
    if (sink.obs) {
        if (count) sink.dsum += (sink.obs[t >> 5] >> (t & 31u)) & 1u ? -1 : 1;
        return;
    }
    sink.tot += count;
    sink.aft += count && t >= sink.warmup;
    if (sink.bm) {
        // a group's misses come in order: the first of each word
        // collects the others' bits
        const uint32_t wd = count ? t >> 5 : 0xFFFFFFFFu;
        uint32_t bits = 1u << (t & 31u);
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            const uint32_t vb = __shfl_down_sync(kFull, bits, o);
            const uint32_t vw = __shfl_down_sync(kFull, wd, o);
            if (r + o < (uint32_t)G && vw == wd) bits |= vb;
        }
        const uint32_t wp = __shfl_up_sync(kFull, wd, 1);
        if (count && (r == 0 || wp != wd)) atomicOr(sink.bm + wd, bits);
    }
}

// The set after its first pass: lines 0 .. a - 1 have filled the ways, the
// others have evicted n - a of them.
__device__ __forceinline__ SmallSet small_first_pass(uint8_t *occ, uint32_t n, uint32_t a, uint64_t seed,
                                                     uint32_t set, bool wtd) {
    uint32_t gone = 0;
    for (uint32_t w = 0; w < a; ++w) occ[32 * w] = (uint8_t)(31u - w);
    for (uint32_t j = a; j < n; ++j) {
        const uint32_t w = random_way(seed, set, j - a, a, wtd);
        gone |= 1u << occ[32 * w];
        occ[32 * w] = (uint8_t)(31u - j);
    }
    return SmallSet{gone, 0u, 0u, 31u - (n - 1u)};
}

template <int G>
__device__ __forceinline__ void play_small(const SimItem &it, const Chain &ch, uint32_t first,
                                           uint32_t nsets, uint8_t *arena, Sink &sink, uint32_t lane) {
    uint8_t *const occ = arena + lane;  // occ[32 w]: 31 - (line held by way w)
    uint32_t *const toff = reinterpret_cast<uint32_t *>(arena + 1024) + lane;
    const uint32_t slot = lane / G, r = lane % G;
    const bool on = slot < nsets;
    const uint32_t c = on ? first + slot : first;
    const uint32_t n = ch.lines_of(c), a = ch.a;
    const uint32_t set = (uint32_t)(((uint64_t)c * ch.st) % ch.T);
    const bool wtd = it.policy == PCHASE_WEIGHTED;
    const uint64_t seed = it.seed;
    for (uint32_t j = 0; j < n; ++j) toff[32 * (31u - j)] = ch.first(c + j * ch.Tp);
    SmallSet st = small_first_pass(occ, n, a, seed, set, wtd);
    uint32_t k = n - a;  // evictions
    const uint32_t glane = lane & ~(uint32_t)(G - 1);
    const uint32_t len = ch.len, per = ch.per;
    bool done = !on;
    while (!__all_sync(kFull, done)) {
        constexpr int kRounds = G >= 8 ? 1 : 8 / G;  // 8 misses at least to a vote
        for (int round = 0; round < kRounds; ++round) {
            const uint32_t wv = 32u * random_way(seed, set, k + r, a, wtd);
            k += G;
            uint32_t mine_p = 0, mine_base = 0;
            small_round<G>(st, occ, wv, per, glane, r, mine_p, mine_base);
            const uint32_t t = mine_base + toff[32 * mine_p];
            const bool count = !done && t < len;
            const uint32_t latest = __shfl_sync(kFull, t, glane + G - 1);
            done = done || latest >= len;
            small_sink<G>(sink, count, t, r);
        }
    }
    __syncwarp();
}

// ---- one long small set by many groups of lanes
// The chain of a set's misses is serial, and one of 300K misses (11.7 ms) set
// the time of a batch.  But what a miss depends on, the lines held counted from
// the last miss's line on, forgets where it came from: two plays of the same
// victims from different states become the same play, up to a rotation of the
// lines, within some tens to hundreds of misses where two lines or more are
// always out (4 ways, 6 lines: 34 on average, 250 at most of 300; 16 ways of 23
// lines: 374, 1837; 4 ways of 5 lines: never; 3 lines in 2 ways: at once).  So the evictions are cut into
// segments.  A survey plays each from a guess kUniformRun evictions long,
// after `warm` evictions to forget it, and notes the state at its start and
// end and the lines it went by.  Then every segment is played from the state
// noted at its start, rotated by the lines all segments before it went by: it
// is the true one if each of those ended in the state the next one's start
// noted.  Where one did not, the segment before plays on to the end alone.
// Segment i is evictions n - a + warm + i kUniformRun and on, the first one
// from n - a (the first pass's) on.
// (Not in the matcher: a set with enough misses for it is in an item of more
// than kUniformMatchLen accesses, which the matcher's runs leave to the units.)
constexpr int kSegG = 8;  // lanes of a segment: four segments a warp

__device__ __forceinline__ bool same_state(const uint8_t *x, const uint8_t *y) {
    const uint4 *const u = reinterpret_cast<const uint4 *>(x), *const v = reinterpret_cast<const uint4 *>(y);
    const uint4 a = u[0], b = v[0], c = u[1], d = v[1];
    return a.x == b.x && a.y == b.y && a.z == b.z && a.w == b.w && c.x == d.x && c.y == d.y && c.z == d.z &&
           c.w == d.w;
}

__global__ void __launch_bounds__(32) uniform_survey_kernel(const SimItem *__restrict__ items,
                                                            const UniformSeg *__restrict__ segs,
                                                            UniformSegState *__restrict__ states,
                                                            SimOut out) {
    __shared__ uint8_t arena[1024];
    const uint32_t lane = threadIdx.x, r = lane % kSegG, glane = lane & ~(uint32_t)(kSegG - 1);
    const UniformSeg sg = segs[blockIdx.x];
    const SimItem it = items[sg.unit];
    if (!taken(it, out.uniform_bad)) return;
    const Chain ch(it);
    const uint32_t i = sg.first + lane / kSegG;
    const uint32_t n = ch.lines_of(sg.cls), a = ch.a;
    const uint32_t set = (uint32_t)(((uint64_t)sg.cls * ch.st) % ch.T);
    const bool wtd = it.policy == PCHASE_WEIGHTED;
    uint8_t *const occ = arena + lane;
    SmallSet st;
    if (i == 0) {
        st = small_first_pass(occ, n, a, it.seed, set, wtd);
    } else {
        // (3 lines in 2 ways: every eviction swaps two of way 0's, way 1's and the
        // one out, so an odd number of them, 1 + i kUniformRun, leaves an odd
        // order; two plays of the same parity are one play but for a rotation)
        const uint32_t flip = n == 3u ? 1u : 0u;
        for (uint32_t w = 0; w < a; ++w) occ[32 * w] = (uint8_t)(31u - (w ^ flip));
        st = SmallSet{(kFull >> a) & ~(n < 32u ? kFull >> n : 0u), 0u, 0u, 31u - (a - 1u)};
        st.below = st.gone & ~(kFull << st.p);
    }
    __syncwarp();
    uint32_t k = n - a + i * kUniformRun;
    // (pass numbers times n: the lines gone by are base + 31 - p)
    uint32_t from = st.base + 31u - st.p;
    UniformSegState *const o = states + sg.state + i;
    auto note = [&](uint8_t *to) {
        if (i < sg.count)
            for (uint32_t w = r; w < 32u; w += kSegG) {
                // line of way w from the last miss's on
                const uint32_t d = w < a ? st.p + n - occ[32 * w] : 0u;
                to[w] = (uint8_t)(d >= n ? d - n : d);
            }
    };
    auto play = [&](uint32_t evictions) {
        for (uint32_t e = 0; e < evictions; e += kSegG) {
            const uint32_t wv = 32u * random_way(it.seed, set, k + r, a, wtd);
            k += kSegG;
            uint32_t mp = 0, mb = 0;
            small_round<kSegG>(st, occ, wv, n, glane, r, mp, mb);
        }
    };
    play(sg.warm);
    note(o->start);
    if (i) from = st.base + 31u - st.p;
    play(kUniformRun);
    note(o->end);
    if (i < sg.count && r == 0) o->lines = st.base + 31u - st.p - from;
}

__global__ void __launch_bounds__(32) uniform_segment_kernel(const SimItem *__restrict__ items,
                                                             const UniformSeg *__restrict__ segs,
                                                             const UniformSegState *__restrict__ states,
                                                             SimOut out) {
    uint8_t *const arena = u_smem;
    const uint32_t lane = threadIdx.x, r = lane % kSegG, glane = lane & ~(uint32_t)(kSegG - 1);
    const UniformSeg sg = segs[blockIdx.x];
    const SimItem it = items[sg.unit];
    if (!taken(it, out.uniform_bad)) return;
    Chain ch(it);
    ch.prepare_first();
    Sink sink;
    open_sink(sink, it, ch, out, 0, arena, lane);
    const uint32_t i = sg.first + lane / kSegG;
    const uint32_t n = ch.lines_of(sg.cls), a = ch.a;
    const uint32_t set = (uint32_t)(((uint64_t)sg.cls * ch.st) % ch.T);
    const bool wtd = it.policy == PCHASE_WEIGHTED;
    uint8_t *const occ = arena + lane;
    uint32_t *const toff = reinterpret_cast<uint32_t *>(arena + 1024) + lane;
    for (uint32_t j = 0; j < n; ++j) toff[32 * (31u - j)] = ch.first(sg.cls + j * ch.Tp);
    // the segments before this one: the lines they went by, and whether each
    // ended where the next one started
    const UniformSegState *const s0 = states + sg.state;
    uint32_t lines = 0;
    bool known = i < sg.count;
    for (uint32_t q = r; known && q < i; q += kSegG) {
        lines += s0[q].lines;
        known = same_state(s0[q].end, s0[q + 1].start);
    }
#pragma unroll
    for (int o = kSegG / 2; o; o >>= 1) {
        lines += __shfl_xor_sync(kFull, lines, o);
        known = __shfl_xor_sync(kFull, known ? 1 : 0, o) && known;
    }
    SmallSet st = small_first_pass(occ, n, a, it.seed, set, wtd);
    uint32_t k = n - a;
    if (i) {
        k += sg.warm + i * kUniformRun;
        lines += n - 1u;  // (the first pass)
        const uint32_t line = lines % n;
        st.base = lines / n * ch.per;
        st.p = 31u - line;
        st.gone = n < 32u ? ~(kFull >> n) : kFull;
        for (uint32_t w = 0; known && w < a; ++w) {
            uint32_t j = line + s0[i].start[w];
            j -= j >= n ? n : 0u;
            occ[32 * w] = (uint8_t)(31u - j);
            st.gone &= ~(0x80000000u >> j);
        }
        st.below = st.gone & ~(kFull << st.p);
    }
    const bool ends = known && i + 1u < sg.count && same_state(s0[i].end, s0[i + 1u].start);
    const uint32_t last = ends ? n - a + sg.warm + (i + 1u) * kUniformRun : 0xFFFFFFFFu;
    __syncwarp();
    const uint32_t len = ch.len, per = ch.per;
    bool done = !known || st.base >= len;
    while (!__all_sync(kFull, done)) {
        const uint32_t wv = 32u * random_way(it.seed, set, k + r, a, wtd);
        k += kSegG;
        uint32_t mine_p = 0, mine_base = 0;
        small_round<kSegG>(st, occ, wv, per, glane, r, mine_p, mine_base);
        const uint32_t t = mine_base + toff[32 * mine_p];
        const bool count = !done && t < len;
        const uint32_t latest = __shfl_sync(kFull, t, glane + kSegG - 1);
        done = done || latest >= len || k >= last;
        small_sink<kSegG>(sink, count, t, r);
    }
    sink.finish(it, out, 0, lane);
}

// Larger sets: one warp per set, a window of up to 32 H run heads at a time, H
// to a lane.  Number the set's evictions 0, 1, 2, ...  The way of each is known
// beforehand, so a line that came in with eviction k leaves with the next
// eviction of the same way: with leave[line] holding that number, a head misses
// exactly when leave[its line] is below the number of evictions before it.
// The lines of a window are distinct (n of them go by before one returns), so
// the heads need only the number at the window's start and how many heads
// before them in the window miss, a rule whose fixed point votes reach in a few
// rounds (a head that misses in one round misses in every later one).
//
// The ways are hashed 32 evictions at a time, 32 H ahead at least.  Of two
// evictions of one way in a row, the earlier one's line gets its number when
// the later one is hashed: through next[] (a ring) if the earlier one is still
// to come, else straight into leave[], by way of occ[], the line a way holds.
//
// A window costs two shared-memory round trips and three to five votes; its
// length, not its instructions, is what counts (one warp to a set), hence as
// many heads a lane as the set's lines allow.  (Tables of each eviction's next
// one of the same way, worked out in parallel beforehand, in place of the
// hashing: the batch 10.0 -> 10.9 ms, their loads being on the window's chain.)
//
// arena: int32 leave[n], uint32 last[a] (1 + the last hashed eviction of a
// way), int32 next[kAhead], uint16 occ[a], uint16 way[kAhead]
constexpr uint32_t kAhead = 256;  // ring of hashed evictions, above 32 (H + 1)
constexpr int32_t kNever = 0x7FFFFFFF;

template <int H>
__device__ __forceinline__ void play_window(const SimItem &it, const Chain &ch, uint32_t c,
                                            uint8_t *arena, Sink &sink, uint32_t lane) {
    const uint32_t n = ch.lines_of(c), a = ch.a;
    int32_t *const leave = reinterpret_cast<int32_t *>(arena);
    uint32_t *const last = reinterpret_cast<uint32_t *>(leave + n);
    int32_t *const next = reinterpret_cast<int32_t *>(last + a);
    uint16_t *const occ = reinterpret_cast<uint16_t *>(next + kAhead);
    uint16_t *const way = occ + a;
    const uint32_t set = (uint32_t)(((uint64_t)c * ch.st) % ch.T);
    const bool wtd = it.policy == PCHASE_WEIGHTED;
    const uint64_t seed = it.seed;
    const uint32_t lt = lt_mask();
    for (uint32_t w = lane; w < a; w += 32) {
        last[w] = 0;
        occ[w] = (uint16_t)w;
    }
    // the first pass has filled the ways with lines 0 .. a - 1
    for (uint32_t j = lane; j < n; j += 32) leave[j] = j < a ? kNever : -1;
    __syncwarp();
    const uint32_t W = H == 1 ? min(32u, n) : 32u * H;  // (H > 1: n >= 32 H)
    // one set walked line by line: consecutive heads are consecutive accesses
    const bool dense = ch.strided && ch.Tp == 1u;
    const uint32_t per = ch.per, len = ch.len;
    uint32_t k0 = 0, hashed = 0;  // evictions before the window; hashed so far
    uint32_t j[H], base[H], t[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        j[h] = a + 32u * h + lane;
        base[h] = 0;
        while (j[h] >= n) {
            j[h] -= n;
            base[h] += per;
        }
        t[h] = base[h] + ch.first(c + j[h] * ch.Tp);
    }
    const bool in = H > 1 || lane < W;
    for (;;) {
        while (hashed < k0 + 32u * H) {
            const uint32_t k = hashed + lane;
            const uint32_t w = random_way(seed, set, k, a, wtd);
            const uint32_t same = __match_any_sync(kFull, w);
            const uint32_t later = same & ~((2u << lane) - 1u);
            const bool head = (same & lt) == 0;
            const uint32_t before = head ? last[w] : 0u;
            way[k % kAhead] = (uint16_t)w;
            next[k % kAhead] = later ? (int32_t)(hashed + (uint32_t)__ffs(later) - 1u) : kNever;
            __syncwarp();
            if (later == 0) last[w] = k + 1u;
            if (head) {
                if (before > k0) next[(before - 1u) % kAhead] = (int32_t)k;
                else leave[occ[w]] = (int32_t)k;
            }
            __syncwarp();
            hashed += 32;
        }
        // heads in trace order: all of h = 0, then h = 1, ...
        int32_t e[H];
        bool valid[H];
        uint32_t bal[H];
#pragma unroll
        for (int h = 0; h < H; ++h) {
            valid[h] = in && t[h] < len;
            e[h] = valid[h] ? leave[j[h]] - (int32_t)k0 : kNever;
        }
#pragma unroll
        for (int h = 0; h < H; ++h) bal[h] = __ballot_sync(kFull, e[h] < 0);
        for (int round = 0; round < 32 * H + 2; ++round) {
            uint32_t change = 0, m = 0;
#pragma unroll
            for (int h = 0; h < H; ++h) {
                const uint32_t nb = __ballot_sync(kFull, e[h] < (int32_t)(m + __popc(bal[h] & lt)));
                change |= nb ^ bal[h];
                bal[h] = nb;
                m += (uint32_t)__popc(nb);
            }
            if (change == 0) break;
        }
        const bool more = __all_sync(kFull, valid[H - 1] || !in);  // the trace goes on
        uint32_t m = k0;
#pragma unroll
        for (int h = 0; h < H; ++h) {
            if ((bal[h] >> lane) & 1u) {
                const uint32_t k = (m + __popc(bal[h] & lt)) % kAhead;
                const int32_t nx = next[k];
                leave[j[h]] = nx;
                // the line its way holds, unless its leaving is known already
                if (nx == kNever) occ[way[k]] = (uint16_t)j[h];
                // (the first pass's misses are in the words already)
                if (t[h] >= per) {
                    if (sink.obs) {
                        sink.dsum += (sink.obs[t[h] >> 5] >> (t[h] & 31u)) & 1u ? -1 : 1;
                    } else {
                        sink.tot += 1;
                        sink.aft += t[h] >= sink.warmup;
                        if (sink.bm && !dense) atomicOr(sink.bm + (t[h] >> 5), 1u << (t[h] & 31u));
                    }
                }
            }
            if (dense && sink.bm && lane == 0 && bal[h]) {
                const uint32_t sh = t[h] & 31u;
                atomicOr(sink.bm + (t[h] >> 5), bal[h] << sh);
                if (sh && bal[h] >> (32u - sh))
                    atomicOr(sink.bm + (t[h] >> 5) + 1, bal[h] >> (32u - sh));
            }
            m += (uint32_t)__popc(bal[h]);
            j[h] += W;
            if (j[h] >= n) {
                j[h] -= n;
                base[h] += per;
            }
            t[h] = base[h] + ch.first(c + j[h] * ch.Tp);
        }
        if (!more) break;
        k0 = m;
        __syncwarp();
    }
    __syncwarp();
}

// One warp per task, costliest first; blockIdx.y: the observation (matcher).
__global__ void __launch_bounds__(32) uniform_play_kernel(const SimItem *__restrict__ items,
                                                          const UniformTask *__restrict__ tasks,
                                                          SimOut out) {
    const uint32_t lane = threadIdx.x;
    const UniformTask task = tasks[blockIdx.x];
    const SimItem it = items[task.unit];
    if (!taken(it, out.uniform_bad)) return;
    const bool ham = out.dist != nullptr;
    if (ham && !((it.lsh >> kUniformMatchBit) & 1u)) return;
    Chain ch(it);
    ch.prepare_first();
    Sink sink;
    uint8_t *const arena = open_sink(sink, it, ch, out, blockIdx.y, u_smem, lane);
    if (task.lanes) {
        const uint32_t per_warp = 32u / task.lanes;
        for (uint32_t c = 0; c < task.count; c += per_warp) {
            const uint32_t first = task.first + c, m = min(per_warp, task.count - c);
            switch (task.lanes) {
            case 1: play_small<1>(it, ch, first, m, arena, sink, lane); break;
            case 2: play_small<2>(it, ch, first, m, arena, sink, lane); break;
            case 4: play_small<4>(it, ch, first, m, arena, sink, lane); break;
            case 8: play_small<8>(it, ch, first, m, arena, sink, lane); break;
            case 16: play_small<16>(it, ch, first, m, arena, sink, lane); break;
            default: play_small<32>(it, ch, first, m, arena, sink, lane); break;
            }
        }
    } else {
        for (uint32_t c = task.first; c < task.first + task.count; ++c) {
            const uint32_t n = ch.lines_of(c);
            if (n >= 128) play_window<4>(it, ch, c, arena, sink, lane);
            else if (n >= 64) play_window<2>(it, ch, c, arena, sink, lane);
            else play_window<1>(it, ch, c, arena, sink, lane);
        }
    }
    sink.finish(it, out, blockIdx.y, lane);
}

}  // namespace

cudaError_t launch_uniform_prep(const SimItem *items, const uint32_t *trace_unit, uint32_t n_trace,
                                uint64_t n_explicit, uint64_t max_len, uint64_t n_items,
                                uint64_t *counts, uint32_t *head, uint32_t *bad, int sms,
                                cudaStream_t st) {
    // warps to a trace: enough of them to fill the GPU when traces are few, of
    // 2048 accesses at least; with one each, the launch needs nothing cleared
    // before it (97 traces of 432 accesses: 2 us of memset and 2 of idle CTAs)
    const uint64_t full = (uint64_t)std::max(sms, 1) * 64;
    uint32_t parts = 1;
    while (parts < 64 && n_explicit && n_explicit * parts < 4 * full && max_len > 2048ull * parts) parts *= 2;
    const bool alone = parts == 1 && n_explicit;
    if (!alone) {
        const cudaError_t e = cudaMemsetAsync(head, 0, kQueueHeader + 4ull * n_trace, st);
        if (e != cudaSuccess) return e;
    }
    const uint64_t warps = std::max<uint64_t>(n_explicit ? (uint64_t)n_trace * parts : 1,
                                              counts ? (2 * n_items + 31) / 32 : 1);
    const uint64_t blocks = std::min<uint64_t>((warps + 7) / 8, (uint64_t)std::max(sms, 1) * 8);
    uniform_prep_kernel<<<(unsigned)blocks, 256, 0, st>>>(items, trace_unit, n_explicit ? n_trace : 0u,
                                                          parts, n_items, counts, bad,
                                                          alone ? head : nullptr);
    return cudaGetLastError();
}

cudaError_t launch_uniform_match(const SimItem *items, const UniformGroup *groups, uint32_t n_groups,
                                 const uint32_t *cands, int sms, const SimOut &out, uint32_t *live,
                                 cudaStream_t st) {
    const uint32_t blocks = std::min(n_groups, (uint32_t)std::max(sms, 1) * 8u);
    uniform_match_kernel<<<dim3(blocks, out.n_rep ? out.n_rep : 1u), 256, 0, st>>>(
        items, groups, n_groups, cands, out, live);
    return cudaGetLastError();
}

cudaError_t launch_uniform_out(const SimItem *items, const uint32_t *units, uint64_t n_units,
                               uint64_t max_len, int sms, const SimOut &out, uint32_t *live,
                               cudaStream_t st) {
    if (!n_units) return cudaSuccess;
    // (a part is 32 words at least)
    const uint64_t full = (uint64_t)std::max(sms, 1) * 64;
    uint32_t parts = 1;
    while (parts < 32 && n_units * parts < 2 * full && max_len > 1024ull * parts) parts *= 2;
    const uint64_t warps = n_units * parts;
    const uint64_t blocks = std::min<uint64_t>((warps + 7) / 8, (uint64_t)std::max(sms, 1) * 8);
    uniform_out_kernel<<<(unsigned)blocks, 256, 0, st>>>(items, units, n_units, parts, out, live);
    return cudaGetLastError();
}

cudaError_t prepare_uniform(uint32_t smem_bytes) {
    return cudaFuncSetAttribute(uniform_play_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(smem_bytes + kUniformMatchLen / 8));
}

cudaError_t launch_uniform_play(const SimItem *items, const UniformTask *tasks, uint32_t n_tasks,
                                uint32_t smem_bytes, const SimOut &out, cudaStream_t st) {
    if (!n_tasks) return cudaSuccess;
    const bool ham = out.dist != nullptr;
    const uint32_t bytes = smem_bytes + (ham ? kUniformMatchLen / 8 : 0u);
    uniform_play_kernel<<<dim3(n_tasks, ham && out.n_rep ? out.n_rep : 1u), 32, bytes, st>>>(items, tasks,
                                                                                             out);
    return cudaGetLastError();
}

cudaError_t launch_uniform_segments(const SimItem *items, const UniformSeg *segs, uint32_t n_segs,
                                    UniformSegState *states, const SimOut &out, cudaStream_t st) {
    if (!n_segs) return cudaSuccess;
    uniform_survey_kernel<<<n_segs, 32, 0, st>>>(items, segs, states, out);
    uniform_segment_kernel<<<n_segs, 32, kUniformSmallBytes, st>>>(items, segs, states, out);
    return cudaGetLastError();
}

}  // namespace pchase
