// The learned inverse's network at inference (S7) on sm_103a's fifth-
// generation tensor cores: tcgen05.mma with both operands in shared memory
// and the FP32 accumulator in tensor memory (TMEM).  Three kernels: layers 1
// and 2 (conv12_tc_kernel), layers 3 and 4 (conv34_tc_kernel), FC + heads
// (fc_heads_tc_kernel).  The 64-channel layers (kernel 5, stride 2, zero
// padding 2) use an implicit im2col:
//
// out[b][p][co] = GELU(bias[co] + sum_k sum_ci W[co][k*64 + ci] * x[b][2p + k - 2][ci])
//
// One tile is 128 consecutive output rows (b, p) x 64 output channels, i.e.
// one M=128, N=64 accumulator, computed as 5 taps x 4 K-slices of 16 channels
// (20 MMAs, issued by one thread).  The A operand of tap k would be the input
// rows 2p + k - 2: rows two apart, which no shared-memory matrix descriptor
// can address.  So the tile's rows are taken in a transposed order, TMEM lane
// r = 8g + i holding output row o = 16i + g of the tile, and the input slab is
// staged as two planes (even and odd input offsets) whose row 8G + i holds
// input position 2*p(16i) + 2(G - 1) + plane.  Tap k then reads plane k % 2 from
// row group k / 2 on: 128 consecutive rows of 128 bytes (64 BF16 channels), a
// canonical K-major operand with the 128-byte swizzle, every tap starting on
// a 1024-byte swizzle-atom boundary.  The weights are five such N=64 x K=64
// tiles, loaded once per CTA.  An epilogue warp w reads TMEM lanes
// 32 (w % 4) .. +31 (the lanes its quarter of the CTA may access).
// Completion waits on an mbarrier give up after 2 s of %globaltimer: the
// kernel then ORs PCHASE_DEV_TIMEOUT into *status, stops, waits for its own
// copies and MMAs, frees its TMEM and returns.
#include <cuda_bf16.h>

#include <algorithm>

#include "conv_tc.cuh"
#include "tc_common.cuh"
#include "tma_host.cuh"

namespace pchase {
namespace {

constexpr int kCh = 64;
constexpr int kTaps = 5;
constexpr int kTileRows = 128;
constexpr int kGroups = 18;                           // 8-row groups per slab plane
constexpr uint32_t kPlaneBytes = kGroups * 8 * 128;   // 18 KB
constexpr uint32_t kSlabBytes = 2 * kPlaneBytes;      // 36 KB
constexpr uint32_t kWBytes = kTaps * kCh * 128;       // 40 KB
constexpr uint32_t kTmemCols = 128;                   // two 64-column accumulators

// Instruction descriptor of tcgen05.mma .kind::f16: FP32 accumulator (bits
// 4-5 = 1), BF16 A and B (bits 7-9, 10-12 = 1), both K-major (bits 15, 16 =
// 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(64 >> 3) << 17) |
                            ((uint32_t)(kTileRows >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t acc) {
    mma_bf16_id(d_tmem, a, b, kIdesc, acc);
}

// ------------------------------------------- first two layers, fused
// Inference of layers 1 and 2 without the first layer's activations ever
// leaving the SM.  One tile is one trace: layer 2's 128 output positions are
// exactly an M=128 accumulator.  Its input slab (the two planes of 18 x 8
// rows of layer-1 outputs described above, 36 KB) is computed by eight
// producer warps straight from the trace's 512 FP32 inputs (rounded to BF16
// as the unfused path rounds them): row 8G + i of plane pl holds layer-1
// position q = 32i + 2G - 2 + pl, channels in 16-byte chunks with the
// 128-byte swizzle, zeros outside 0 <= q < 256.  Eight more warps run the
// epilogue (bias, GELU, BF16 store) and one thread of the last warp issues the
// MMAs.  The roles meet on mbarriers: slab_full (the producers' 256 arrivals
// after a proxy fence), slab_empty (tcgen05.commit once the MMAs that read a
// slab are done; three slabs in flight), acc_full and acc_empty (two TMEM
// accumulators).
// The output tile goes through shared memory and leaves as one TMA store: a
// lane of the accumulator holds half a row, and 32 such rows stored from
// registers are 32 pieces of 16 bytes an instruction (65,536 traces 925 us with
// them, 793 us so).  What bounds it: no one pipe; FMA, tanh and shared-memory
// wavefronts each take 43-45 % of the cycles and issue 49 %, and a second group
// of producer warps adds nothing.
// Every wait gives up after 2 s: the CTA then ORs PCHASE_DEV_TIMEOUT into
// *status, each role leaves its loop at its next wait or group barrier, the
// MMAs already issued are waited for, and TMEM is freed.
constexpr uint32_t kOutTile = kTileRows * 128;  // a trace's 128 output positions, 16 KB
constexpr int kFusedThreads = 256 + 256 + 32;  // producers, epilogue, an MMA warp
constexpr int kFusedSlabs = 3;
constexpr uint32_t kFusedXs = 520;  // staged inputs: xs[q + 2] = x[q], zeros around
// two buffers of staged inputs, a trace's and the next one's
constexpr uint32_t kFusedSmem =
    1024 + kWBytes + kFusedSlabs * kSlabBytes + 2 * kOutTile + 2 * 4 * kFusedXs + 4 * kCh + 128;

__global__ void __launch_bounds__(kFusedThreads, 1)
    conv12_tc_kernel(const float *__restrict__ x, int nb, const __nv_bfloat16 *__restrict__ W1,
                     const float *__restrict__ bias1, const __nv_bfloat16 *__restrict__ W2,
                     const float *__restrict__ bias2, const __grid_constant__ CUtensorMap omap,
                     uint32_t *__restrict__ status) {
    constexpr int kLin = 512, kL1 = 256;
    extern __shared__ uint8_t dsm[];
    const uint32_t raw = smem_u32(dsm);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *const gbase = dsm + (base - raw);
    const uint32_t sW = base;
    const uint32_t sSlab = base + kWBytes;
    const uint32_t sOut = sSlab + kFusedSlabs * kSlabBytes;  // two output tiles
    float *const xs = reinterpret_cast<float *>(gbase + (sOut - base) + 2 * kOutTile);
    float *const sBias2 = xs + 2 * kFusedXs;
    const uint32_t sBar = sOut + 2 * kOutTile + 2 * 4 * kFusedXs + 4 * kCh;
    // barriers: slab_full[kFusedSlabs] at sBar + 8b, slab_empty[kFusedSlabs] at
    // sEmpty + 8b, acc_full[2] at sAcc + 8a, acc_empty[2] at sFree + 8a; then the TMEM
    // address and the abort flag
    const uint32_t sEmpty = sBar + 8u * kFusedSlabs, sAcc = sEmpty + 8u * kFusedSlabs, sFree = sAcc + 16u;
    uint32_t *const tslot = reinterpret_cast<uint32_t *>(gbase + (sFree - base) + 16);
    volatile uint32_t *const abort_flag = tslot + 1;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ntiles = nb;

    // layer 2's weights: tap k is W2[:, 64k .. 64k+63], 64 rows of 128 bytes, swizzled
    for (int e = tid; e < kTaps * kCh * 8; e += kFusedThreads) {
        const int k = e >> 9, co = (e >> 3) & 63, c = e & 7;
        cp_async16(sW + k * 8192 + co * 128 + ((c ^ (co & 7)) << 4),
                   W2 + (size_t)co * (kTaps * kCh) + k * kCh + c * 8, true);
    }
    cp_async_commit();
    if (tid == 0) {
        for (int q = 0; q < kFusedSlabs; ++q) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 256;" ::"r"(sBar + 8 * q) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sEmpty + 8 * q)
                         : "memory");
        }
        for (int a = 0; a < 2; ++a) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sAcc + 8 * a)
                         : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(sFree + 8 * a)
                         : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *abort_flag = 0;
    }
    if (tid < kCh) sBias2[tid] = bias2[tid];
    if (tid < 2 * (int)(kFusedXs - kLin)) {
        // the padding of each buffer: 2 words before the inputs, the rest after
        const int u = tid / (int)(kFusedXs - kLin), e = tid % (int)(kFusedXs - kLin);
        xs[u * (int)kFusedXs + (e < 2 ? e : kLin + e)] = 0.0f;
    }
    // slab rows of positions -2, -1 (row 0 of each plane) and 256, 257 (row
    // 8 * 17 + 7) are zero padding, written once: the producers never write them
    for (int e = tid; e < kFusedSlabs * 2 * 2 * 8; e += kFusedThreads) {
        const int sb = e / 32, pl = (e / 16) & 1, which = (e / 8) & 1, c = e & 7;
        const int row = which ? 8 * 17 + 7 : 0;
        uint4 *d = reinterpret_cast<uint4 *>(gbase + kWBytes + (size_t)sb * kSlabBytes +
                                             (size_t)pl * kPlaneBytes + (size_t)row * 128 + c * 16);
        *d = make_uint4(0u, 0u, 0u, 0u);
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tslot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    cp_async_wait_all();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    if (warp < 8) {
        // ---------------- producers: layer 1 into the slabs (barrier id 2)
        const int p = tid;             // 0..255
        const int c = p & 7;           // the 8 channels this thread computes
        const int r0 = p >> 3;         // rows r0, r0 + 32, ... of the 288 slab rows
        // the weights and biases of channels (2jj, 2jj + 1) of this thread's
        // 8, halved (exactly), so that the sums come out halved for gelu2h_bf16
        uint64_t w2[4][kTaps], b2[4];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const int c0 = c * 8 + 2 * jj;
            b2[jj] = f2(0.5f * bias1[c0], 0.5f * bias1[c0 + 1]);
#pragma unroll
            for (int k = 0; k < kTaps; ++k)
                w2[jj][k] = f2(0.5f * __bfloat162float(W1[c0 * kTaps + k]),
                               0.5f * __bfloat162float(W1[(c0 + 1) * kTaps + k]));
        }
        // the next trace's inputs are loaded while this one's slab is computed
        float xa = 0.0f, xb = 0.0f;
        if ((int)blockIdx.x < ntiles) {
            xa = x[(size_t)blockIdx.x * kLin + p];
            xb = x[(size_t)blockIdx.x * kLin + 256 + p];
        }
        for (int j = 0;; ++j) {
            const int t = blockIdx.x + j * (int)gridDim.x;
            if (t >= ntiles) break;
            const int b = j % kFusedSlabs;
            bool ok = true;
            if (j >= kFusedSlabs) ok = mbar_wait(sEmpty + 8 * b, (uint32_t)(j / kFusedSlabs - 1) & 1u);
            // this trace's inputs into buffer j mod 2 (every producer finished
            // trace j - 2, the last user of that buffer, before the barrier of
            // trace j - 1), then one barrier: the inputs are in, and no wait
            // gave up
            float *const xb_ = xs + (j & 1) * kFusedXs;
            xb_[p + 2] = __bfloat162float(__float2bfloat16(xa));
            xb_[p + 258] = __bfloat162float(__float2bfloat16(xb));
            if (group_any(2, !ok || *abort_flag != 0)) {
                if (p == 0) *abort_flag = 1;
                break;
            }
            const int tn = t + (int)gridDim.x;
            if (tn < ntiles) {
                xa = x[(size_t)tn * kLin + p];
                xb = x[(size_t)tn * kLin + 256 + p];
            }
            const uint32_t slab = sSlab + (uint32_t)b * kSlabBytes;
            // each layer-1 position once (a warp takes 4 consecutive ones, so
            // its input reads fall in different banks), stored to the slab row
            // that holds it and, for the positions two row groups repeat, to
            // the second one too; the rows outside 0..255 stay zero
#pragma unroll 2
            for (int q = r0; q < kL1; q += 32) {
                uint64_t xin[kTaps];
#pragma unroll
                for (int k = 0; k < kTaps; ++k) {
                    const float xv = xb_[2 * q + k];  // x[2q + k - 2]
                    xin[k] = f2(xv, xv);
                }
                uint32_t pk[4];
#pragma unroll
                for (int jj = 0; jj < 4; ++jj) {
                    // channels 2jj and 2jj + 1 side by side: the bias, then the
                    // taps in order from 0, as one FMA chain (all halved)
                    uint64_t acc = fma2(w2[jj][0], xin[0], b2[jj]);
#pragma unroll
                    for (int k = 1; k < kTaps; ++k) acc = fma2(w2[jj][k], xin[k], acc);
                    pk[jj] = gelu2h_bf16(acc);
                }
                // q = 32i + 2G - 2 + pl: row 8G + i of plane pl (i < 8), and
                // row 8(G + 16) + (i - 1) when G < 2 and i > 0
                const int pl = q & 1, u = (q + 2 - pl) >> 1;
                const int i = u >> 4, G = u & 15;
                const uint32_t pbase = slab + (uint32_t)pl * kPlaneBytes;
                uint32_t dst;
                if (i < 8) {
                    dst = pbase + (uint32_t)(8 * G + i) * 128u + ((uint32_t)(c ^ i) << 4);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst),
                                 "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3])
                                 : "memory");
                }
                if (G < 2 && i > 0) {
                    dst = pbase + (uint32_t)(8 * (G + 16) + i - 1) * 128u +
                          ((uint32_t)(c ^ (i - 1)) << 4);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst),
                                 "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3])
                                 : "memory");
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(sBar + 8 * b)
                         : "memory");
        }
    } else if (warp < 16) {
        // ---------------- epilogue: tile j from accumulator j mod 2, handed
        // back as soon as its values are in registers.  Warp w reads TMEM lane
        // quarter w mod 4 (its hardware quarter), column half w / 4
        const int gw = warp - 8, quarter = gw & 3, half = gw >> 2;
        const int r = quarter * 32 + lane;  // TMEM lane r: output position 16 (r & 7) + (r >> 3)
        const ulonglong2 *const b2 = reinterpret_cast<const ulonglong2 *>(sBias2 + half * 32);
        for (int j = 0;; ++j) {
            const int t = blockIdx.x + j * (int)gridDim.x;
            if (t >= ntiles) break;
            // (a wait that gives up is told to the others at the tile's barrier)
            const bool bad = !mbar_wait(sAcc + 8 * (j & 1), (uint32_t)(j >> 1) & 1u);
            __syncwarp();
            tc_fence_after();
            const uint32_t taddr = tmem + (uint32_t)(j & 1) * 64u + (uint32_t)half * 32u +
                                   ((uint32_t)(quarter * 32) << 16);
            uint32_t v[2][16];
#pragma unroll
            for (int qq = 0; qq < 2; ++qq) tmem_ld16(taddr + qq * 16, v[qq]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            tc_fence_before();
            if (lane == 0)
                asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(sFree + 8 * (j & 1))
                             : "memory");
            // the tile in shared memory, row r as it comes (the store's tensor map
            // puts it at its position), 128-byte swizzle: 8 lanes write 8 chunks
            const uint32_t row = sOut + (uint32_t)(j & 1) * kOutTile + (uint32_t)r * 128u;
            auto put = [&](int c, const uint32_t *q) {
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                                 row + (uint32_t)(((half * 4 + c) ^ (r & 7)) << 4)),
                             "r"(q[0]), "r"(q[1]), "r"(q[2]), "r"(q[3])
                             : "memory");
            };
#pragma unroll
            for (int qq = 0; qq < 2; ++qq) {
                uint32_t pk[8];
#pragma unroll
                for (int e = 0; e < 16; e += 4) {
                    const ulonglong2 bb = b2[qq * 4 + (e >> 2)];
                    pk[e >> 1] = gelu2_bf16(add2(f2(__uint_as_float(v[qq][e]), __uint_as_float(v[qq][e + 1])), bb.x));
                    pk[(e >> 1) + 1] =
                        gelu2_bf16(add2(f2(__uint_as_float(v[qq][e + 2]), __uint_as_float(v[qq][e + 3])), bb.y));
                }
                put(2 * qq, pk);
                put(2 * qq + 1, pk + 4);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            // the tile before this one has left its buffer (issued a tile ago),
            // which the warps fill after this barrier
            if (gw == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            if (group_any(1, bad || *abort_flag != 0)) {
                if (lane == 0) *abort_flag = 1;
                break;
            }
            if (gw == 0 && lane == 0) {
                asm volatile(
                    "cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::
                        "l"(reinterpret_cast<uint64_t>(&omap)), "r"(0), "r"(0), "r"(0), "r"(t),
                    "r"(sOut + (uint32_t)(j & 1) * kOutTile)
                    : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
        }
        if (gw == 0 && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    } else if (lane == 0) {
        // ---------------- MMA issue: one thread, ahead of the epilogue by one
        // tile (two accumulators)
        uint64_t da[kTaps], db[kTaps];  // tap k in slab 0, and its weights
#pragma unroll
        for (int q = 0; q < kTaps; ++q) {
            da[q] = sw128_desc(sSlab + (uint32_t)(q & 1) * kPlaneBytes + (uint32_t)(q >> 1) * 1024u);
            db[q] = sw128_desc(sW + (uint32_t)q * 8192u);
        }
        int issued = 0;
        for (int j = 0;; ++j) {
            const int t = blockIdx.x + j * (int)gridDim.x;
            if (t >= ntiles || *abort_flag) break;
            const int b = j % kFusedSlabs;
            // the epilogue has tile j - 2's values, and slab j is written
            if ((j >= 2 && !mbar_wait(sFree + 8 * (j & 1), (uint32_t)((j >> 1) - 1) & 1u)) ||
                !mbar_wait(sBar + 8 * b, (uint32_t)(j / kFusedSlabs) & 1u)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(j & 1) * 64u;
            const uint64_t off = (uint64_t)((uint32_t)b * kSlabBytes >> 4);  // slab b's, in 16 bytes
#pragma unroll
            for (int q = 0; q < kTaps; ++q)
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    mma_bf16(d, da[q] + off + 2u * s, db[q] + 2u * s, (q | s) != 0 ? 1u : 0u);
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    sAcc + 8u * (uint32_t)(j & 1))
                : "memory");
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    sEmpty + 8u * (uint32_t)b)
                : "memory");
            issued = j + 1;
        }
        // every commit's arrival lands, and every MMA issued finishes, before
        // TMEM is freed and the CTA leaves
        for (int jj = issued > kFusedSlabs ? issued - kFusedSlabs : 0; jj < issued; ++jj)
            mbar_wait(sEmpty + 8 * (jj % kFusedSlabs), (uint32_t)(jj / kFusedSlabs) & 1u);
        for (int jj = issued > 2 ? issued - 2 : 0; jj < issued; ++jj)
            mbar_wait(sAcc + 8 * (jj & 1), (uint32_t)(jj >> 1) & 1u);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && *abort_flag) atomicOr(status, PCHASE_DEV_TIMEOUT);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kTmemCols)
                     : "memory");
}

// ------------------------------------------------------------ FC + heads
// logits[m][h] = bias5[h] + sum_n bf16(GELU(bias4[n] + sum_k act[m][k] W4[n][k])) W5[h][n]
// act [B][2048] BF16, W4 [256][2048] BF16, W5 [31][256] BF16.  CTA t takes
// rows 128t .. 128t+127 and all 256 hidden units, so each activation row is
// read once:
//   * FC on the tensor cores: M128 N256, K = 2048 in 32 blocks of 64; a block
//     is two TMA tile loads (the activation tile and W4's, 2-D tensor maps with
//     the 128-byte swizzle; rows past the batch read as zeros) into a 4-stage
//     ring three blocks ahead, one thread issuing loads and MMAs; a stage's
//     mbarrier counts its bytes in, a second one frees it once its MMAs are done;
//   * epilogue: bias, GELU, BF16 rounding of the 128 x 256 hidden tile into
//     four swizzled 64-column K blocks in shared memory (the ring's space),
//     then the heads as a second MMA (M128 N32 K256, W5 padded to 32 rows)
//     into 32 more TMEM columns, read back and stored with bias5 (no atomics:
//     each CTA owns its rows).
constexpr int kFcK = 2048, kFcN = 256, kHeads = 31, kHeadsPad = 32;
constexpr int kFcStages = 4;   // ring stages, loaded kFcStages - 1 blocks ahead
constexpr uint32_t kFcABytes = kTileRows * 128, kFcBBytes = kFcN * 128;
constexpr uint32_t kFcStageBytes = kFcABytes + kFcBBytes;  // 48 KB
constexpr uint32_t kW5Bytes = 4 * kHeadsPad * 128;         // 4 K blocks of 32 rows x 64 BF16
constexpr uint32_t kFcSmemBytes =
    1024 + kFcStages * kFcStageBytes + kW5Bytes + 8 * (2 * kFcStages + 1) + 16;
constexpr uint32_t kFcTmemCols = 512;  // 256 FC + 32 heads, rounded to a power of two
constexpr uint32_t kIdescFc = (1u << 4) | (1u << 7) | (1u << 10) |
                              ((uint32_t)(kFcN >> 3) << 17) | ((uint32_t)(kTileRows >> 4) << 24);
constexpr uint32_t kIdescHeads = (1u << 4) | (1u << 7) | (1u << 10) |
                                 ((uint32_t)(kHeadsPad >> 3) << 17) |
                                 ((uint32_t)(kTileRows >> 4) << 24);

__global__ void __launch_bounds__(128, 1)
    fc_heads_tc_kernel(const __grid_constant__ CUtensorMap amap,
                       const __grid_constant__ CUtensorMap wmap, int nb, const float *__restrict__ bias4,
                       const __nv_bfloat16 *__restrict__ W5, const float *__restrict__ bias5,
                       float *__restrict__ logits, uint32_t *__restrict__ status) {
    extern __shared__ uint8_t dsm[];
    const uint32_t raw = smem_u32(dsm);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *const gbase = dsm + (base - raw);
    const uint32_t sStage = base;
    const uint32_t sW5 = base + kFcStages * kFcStageBytes;  // 1024-aligned
    // mbarriers: stage loaded [S] at sBar + 8s, stage's MMAs done [S] at
    // sBar + 8 (S + s), the heads MMAs at sBar + 16 S
    const uint32_t sBar = sW5 + kW5Bytes;
    const uint32_t full0 = sBar, done0 = sBar + 8u * kFcStages, hbar = sBar + 16u * kFcStages;
    uint32_t *const tslot = reinterpret_cast<uint32_t *>(
        gbase + kFcStages * kFcStageBytes + kW5Bytes + 8 * (2 * kFcStages + 1));
    volatile uint32_t *const abort_flag = tslot + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * kTileRows;
    constexpr int kBlocks = kFcK / 64;

    // W5 as the heads' B operand: K block kb holds hidden units 64kb .. +63 of
    // its 32 rows (row 31 zero), 128-byte swizzle
    for (int e = tid; e < 4 * kHeadsPad * 8; e += 128) {
        const int kb = e >> 8, h = (e >> 3) & 31, c = e & 7;
        const bool ok = h < kHeads;
        cp_async16(sW5 + kb * (kHeadsPad * 128) + h * 128 + ((c ^ (h & 7)) << 4),
                   ok ? W5 + (size_t)h * kFcN + kb * 64 + c * 8 : W5, ok);
    }
    // block kb's activation and W4 tiles into stage kb mod S (one thread)
    auto load = [&](int kb) {
        const uint32_t q = (uint32_t)(kb % kFcStages);
        const uint32_t st = sStage + q * kFcStageBytes;
        mbar_expect_tx(full0 + 8u * q, kFcStageBytes);
        tma_load_2d(st, &amap, kb * 64, m0, full0 + 8u * q);
        tma_load_2d(st + kFcABytes, &wmap, kb * 64, 0, full0 + 8u * q);
    };
    cp_async_commit();
    if (tid == 0) {
        for (int q = 0; q <= 2 * kFcStages; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(sBar + 8 * q) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *abort_flag = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tslot)),
                     "r"(kFcTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;  // columns 0..255: FC; 256..287: heads

    int loaded = 0;  // blocks whose loads went out (thread 0)
    if (tid == 0) {
        for (; loaded < kFcStages - 1; ++loaded) load(loaded);
        for (int kb = 0; kb < kBlocks; ++kb) {
            const uint32_t q = (uint32_t)(kb % kFcStages);
            if (!mbar_wait(full0 + 8u * q, (uint32_t)(kb / kFcStages) & 1u)) {
                *abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t st = sStage + q * kFcStageBytes;
#pragma unroll
            for (int s = 0; s < 4; ++s)
                mma_bf16_id(tmem, sw128_desc(st + 32u * s), sw128_desc(st + kFcABytes + 32u * s),
                            kIdescFc, (kb | s) != 0 ? 1u : 0u);
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    done0 + 8u * q)
                : "memory");
            // the stage of block kb - 1 (its MMAs went out a step ago) takes block kb + S - 1
            if (loaded < kBlocks) {
                const int pj = loaded - kFcStages;
                if (pj >= 0 && !mbar_wait(done0 + 8u * (uint32_t)(pj % kFcStages),
                                          (uint32_t)(pj / kFcStages) & 1u)) {
                    *abort_flag = 1;
                    break;
                }
                load(loaded++);
            }
        }
    }
    cp_async_wait_all();  // W5
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    bool ok = *abort_flag == 0;
    if (ok) {
        const int lb = kBlocks - 1;  // the last commit covers every earlier MMA
        const bool got = mbar_wait(done0 + 8u * (uint32_t)(lb % kFcStages), (uint32_t)(lb / kFcStages) & 1u);
        ok = __syncthreads_and(got);
    }
    const int r = warp * 32 + lane;  // TMEM lane = tile row
    if (ok) {
        // hidden tile -> BF16 A operand of the heads MMA: K block kb (hidden
        // units 64kb .. +63) at sStage + kb * 16 KB, rows of 128 bytes swizzled
        tc_fence_after();
        const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int q = 0; q < 16; ++q) {
            uint32_t v[16];
            tmem_ld16(taddr + q * 16, v);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            uint32_t pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
                const int n = q * 16 + e;
                pk[e >> 1] = gelu2_bf16(add2(f2(__uint_as_float(v[e]), __uint_as_float(v[e + 1])),
                                             f2(__ldg(bias4 + n), __ldg(bias4 + n + 1))));
            }
            // 16 columns = chunks 2(q % 4), +1 of row r in K block q / 4
            uint4 *row = reinterpret_cast<uint4 *>(gbase + (q >> 2) * kFcABytes + r * 128);
            const int c0 = 2 * (q & 3);
            row[c0 ^ (r & 7)] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            row[(c0 + 1) ^ (r & 7)] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (tid == 0) {
#pragma unroll
            for (int kb = 0; kb < 4; ++kb)
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    mma_bf16_id(tmem + 256u, sw128_desc(sStage + kb * kFcABytes + 32u * s),
                                sw128_desc(sW5 + kb * (kHeadsPad * 128) + 32u * s), kIdescHeads,
                                (kb | s) != 0 ? 1u : 0u);
            asm volatile(
                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    hbar)
                : "memory");
        }
        const bool got = mbar_wait(hbar, 0u);
        ok = __syncthreads_and(got);
        if (ok) {
            tc_fence_after();
            uint32_t v[2][16];
            tmem_ld16(taddr + 256, v[0]);
            tmem_ld16(taddr + 272, v[1]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            const int m = m0 + r;
            if (m < nb) {
#pragma unroll
                for (int h = 0; h < kHeads; ++h)
                    logits[(size_t)m * kHeads + h] = __uint_as_float(v[h >> 4][h & 15]) + __ldg(bias5 + h);
            }
        }
    }
    if (!ok && tid == 0) {
        atomicOr(status, PCHASE_DEV_TIMEOUT);
        // the loads and MMAs issued land before TMEM is freed and the CTA leaves
        for (int j = loaded > kFcStages ? loaded - kFcStages : 0; j < loaded; ++j)
            mbar_wait(full0 + 8u * (uint32_t)(j % kFcStages), (uint32_t)(j / kFcStages) & 1u);
        if (loaded > 0)
            mbar_wait(done0 + 8u * (uint32_t)((loaded - 1) % kFcStages),
                      (uint32_t)((loaded - 1) / kFcStages) & 1u);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kFcTmemCols)
                     : "memory");
}

// ------------------------------------------------------------ layers 3 + 4
// Inference of layers 3 and 4 in one kernel.  An iteration takes 4 traces
// (one 128-row tile of layer 4): the layer-3 outputs of its two 128-row tiles
// (2 traces each) go from TMEM through bias and GELU straight into layer 4's
// input slab in shared memory, laid out as the implicit im2col above wants
// (row 8g + i of plane pl holds position 32 (i & 1) + 2 (g - 1) + pl of the
// tile's trace i / 2), and layer 4's MMAs run from there; only layer 4's
// outputs go to global memory.  A layer-3 position q of trace b lands in row
// 8 ((q >> 1) + 1) + 2b when q <= 33 and in row 8 ((q >> 1) - 15) + 2b + 1
// when q >= 30 (plane q & 1); rows 2b of group 0 and 2b + 1 of group 17 are
// the zero padding, written once.
//
// Roles: sixteen epilogue warps, one thread that loads, one that issues the
// MMAs.  A layer-3 slab is two planes, each a stage of its own in a ring of
// five (three TMA loads: groups 1-16, and the first and last group, whose rows
// are the neighbouring blocks of 32 positions', zeros where the trace ends).
// Layer 3's accumulators are double-buffered and its MMAs run up to two
// iterations ahead of the epilogue, so a stage is free again as soon as its
// tile's MMAs are done; layer 4's are double-buffered too, and its epilogue
// runs under the next iteration's layer-4 MMAs.  The outputs go through shared
// memory and leave as TMA stores, one per lane quarter (4 warps, 32 rows).
// With cp.async loads by eight of the warps, one accumulator a tile, block
// barriers between the phases and rows stored from registers the network took
// 1325 us for 65,536 traces, 1210 us so.  An iteration moves 80 KB through
// HBM and some 500 KB through an SM's shared memory (MMA operands 360 KB,
// loads, slab and output writes and reads): those two bound it about equally.
constexpr int kL34Epi = 16;                        // epilogue warps
constexpr int kL34Threads = 32 * (kL34Epi + 2);
constexpr int kL34Planes = 5;                      // ring stages
constexpr uint32_t kL34TmemCols = 512;  // layer 3: 128 p + 64 X; layer 4: 256 + 64 p
constexpr uint32_t kL34Bars = 2 * kL34Planes + 4 + 2 + 1;
constexpr uint32_t kL34Smem =
    1024 + 2 * kWBytes + kL34Planes * kPlaneBytes + kSlabBytes + kOutTile + 8 * kL34Bars + 16;
static_assert(kL34Smem <= 232448, "shared memory");

__device__ __forceinline__ void mma_commit_to(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

__global__ void __launch_bounds__(kL34Threads, 1)
    conv34_tc_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap emap,
                     int nb, const __nv_bfloat16 *__restrict__ W3, const float *__restrict__ bias3,
                     const __nv_bfloat16 *__restrict__ W4, const float *__restrict__ bias4,
                     const __grid_constant__ CUtensorMap omap, uint32_t *__restrict__ status) {
    extern __shared__ uint8_t dsm[];
    const uint32_t raw = smem_u32(dsm);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *const gbase = dsm + (base - raw);
    const uint32_t sW3 = base, sW4 = base + kWBytes;
    const uint32_t sRing = base + 2 * kWBytes;                // planes of layer-3 input slabs
    const uint32_t sL4 = sRing + kL34Planes * kPlaneBytes;    // layer-4 input slab
    const uint32_t sOut = sL4 + kSlabBytes;                   // output tile
    // barriers: plane loaded [5], plane free [5], layer-3 tile done [2 p + X],
    // layer-4 tile done [p], layer-4 slab written
    const uint32_t full0 = sOut + kOutTile, free0 = full0 + 8u * kL34Planes,
                   done3 = free0 + 8u * kL34Planes, done4 = done3 + 32u, ready4 = done4 + 16u;
    uint32_t *const tslot = reinterpret_cast<uint32_t *>(gbase + (ready4 + 8u - base));
    volatile uint32_t *const abort_flag = tslot + 1;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int iters = (nb - 1) / 4 + 1;  // of 4 traces

    for (int e = tid; e < kTaps * kCh * 8; e += kL34Threads) {
        const int k = e >> 9, co = (e >> 3) & 63, c = e & 7;
        const uint32_t off = k * 8192 + co * 128 + ((c ^ (co & 7)) << 4);
        const size_t src = (size_t)co * (kTaps * kCh) + k * kCh + c * 8;
        cp_async16(sW3 + off, W3 + src, true);
        cp_async16(sW4 + off, W4 + src, true);
    }
    cp_async_commit();
    // the layer-4 slab's padding rows (never written again)
    if (tid < 2 * 4 * 2 * 8) {
        const int pl = tid >> 6, b = (tid >> 4) & 3, which = (tid >> 3) & 1, c = tid & 7;
        const int row = which ? 8 * 17 + 2 * b + 1 : 2 * b;
        *reinterpret_cast<uint4 *>(gbase + (sL4 - base) + pl * kPlaneBytes + row * 128 +
                                   ((c ^ (row & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
    }
    if (tid == 0) {
        for (uint32_t q = 0; q + 1 < kL34Bars; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8 * q) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(ready4), "r"(kL34Epi) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *abort_flag = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tslot)),
                     "r"(kL34TmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    cp_async_wait_all();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;

    if (warp == kL34Epi) {
        // ---------------- loads: planes are numbered through all of this CTA's
        // tiles; plane b is in stage b mod 5
        if (lane == 0) {
            uint32_t b = 0, q = 0, par = 1;
            for (int it = blockIdx.x; it < iters && !*abort_flag; it += (int)gridDim.x) {
                for (int k = 0; k < 4; ++k, ++b) {
                    if (!mbar_wait(free0 + 8u * q, par)) {
                        *abort_flag = 1;
                        break;
                    }
                    const int trace = 4 * it + 2 * (k >> 1), pl = k & 1;
                    const uint32_t st = sRing + q * kPlaneBytes, bar = full0 + 8u * q;
                    mbar_expect_tx(bar, kPlaneBytes);
                    tma_load_5d(st + 1024u, &xmap, 0, 0, trace, 0, pl, bar);
                    tma_load_5d(st, &emap, 0, -1, trace, 15, pl, bar);
                    tma_load_5d(st + 17u * 1024u, &emap, 0, 1, trace, 0, pl, bar);
                    if (++q == kL34Planes) {
                        q = 0;
                        par ^= 1u;
                    }
                }
            }
            // loads in flight land before the CTA leaves
            for (uint32_t k = b > kL34Planes ? b - kL34Planes : 0u; k < b; ++k)
                mbar_wait(full0 + 8u * (k % kL34Planes), (k / kL34Planes) & 1u);
        }
    } else if (warp == kL34Epi + 1) {
        // ---------------- MMAs
        if (lane == 0) {
            uint32_t b = 0;
            bool ok = true;
            auto tap = [&](uint32_t d, int k, uint32_t plane, uint32_t sw) {
                const uint32_t a0 = plane + (uint32_t)(k >> 1) * 1024u, b0 = sw + (uint32_t)k * 8192u;
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    mma_bf16(d, sw128_desc(a0 + 32u * s), sw128_desc(b0 + 32u * s), (k | s) != 0 ? 1u : 0u);
            };
            // both layer-3 tiles of this CTA's iteration j
            auto layer3 = [&](int j) {
                for (uint32_t X = 0; ok && X < 2; ++X) {
                    const uint32_t q0 = b % kL34Planes, q1 = (b + 1u) % kL34Planes;
                    ok = mbar_wait(full0 + 8u * q0, (b / kL34Planes) & 1u) &&
                         mbar_wait(full0 + 8u * q1, ((b + 1u) / kL34Planes) & 1u);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t p0 = sRing + q0 * kPlaneBytes, p1 = sRing + q1 * kPlaneBytes;
                    const uint32_t buf = 2u * ((uint32_t)j & 1u) + X;
#pragma unroll
                    for (int k = 0; k < kTaps; ++k) tap(tmem + 64u * buf, k, (k & 1) ? p1 : p0, sW3);
                    mma_commit_to(free0 + 8u * q0);
                    mma_commit_to(free0 + 8u * q1);
                    mma_commit_to(done3 + 8u * buf);
                    b += 2;
                }
            };
            const int mine = ((int)blockIdx.x < iters)
                                 ? (iters - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
            for (int j = 0; j < 2 && j < mine; ++j) layer3(j);
            int sent = 0;
            for (int j = 0; ok && j < mine && !*abort_flag; ++j) {
                // the slab of iteration j is written, and every epilogue warp has
                // read iteration j's layer-3 sums and iteration j - 2's layer-4 sums
                ok = mbar_wait(ready4, (uint32_t)j & 1u);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int k = 0; k < kTaps; ++k)
                    tap(tmem + 256u + 64u * ((uint32_t)j & 1u), k, sL4 + (uint32_t)(k & 1) * kPlaneBytes, sW4);
                mma_commit_to(done4 + 8u * ((uint32_t)j & 1u));
                sent = j + 1;
                if (j + 2 < mine) layer3(j + 2);
            }
            if (!ok) *abort_flag = 1;
            // the MMAs issued finish before TMEM is freed
            if (b) mbar_wait(free0 + 8u * ((b - 1u) % kL34Planes), ((b - 1u) / kL34Planes) & 1u);
            if (sent) mbar_wait(done4 + 8u * ((uint32_t)(sent - 1) & 1u), (uint32_t)((sent - 1) >> 1) & 1u);
        }
    } else {
        // ---------------- epilogues: warp w reads TMEM lane quarter w mod 4 (its
        // hardware quarter) and columns 16 (w / 4) .. + 15: a thread holds 16
        // values of one tile row
        const int quarter = warp & 3, colq = warp >> 2;
        const int r = quarter * 32 + lane;       // this thread's TMEM lane
        const int mt = 16 * (r & 7) + (r >> 3);  // ... and the tile row it holds
        const uint32_t tlane = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)colq * 16u;
        const bool storer = colq == 0 && lane == 0;
        // 16 columns of accumulator acc, bias, GELU, as BF16 pairs
        auto finish = [&](uint32_t acc, const float *bias, uint32_t (&pk)[8]) {
            uint32_t v[16];
            tmem_ld16(tlane + acc, v);
            float4 f[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                f[e] = __ldg(reinterpret_cast<const float4 *>(bias + colq * 16) + e);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                pk[2 * e] = gelu2_bf16(add2(f2(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1])),
                                            f2(f[e].x, f[e].y)));
                pk[2 * e + 1] = gelu2_bf16(
                    add2(f2(__uint_as_float(v[4 * e + 2]), __uint_as_float(v[4 * e + 3])), f2(f[e].z, f[e].w)));
            }
        };
        // the two 16-byte chunks of a row written in an order that alternates
        // with the lane, so that a store instruction's lanes spread over more banks
        auto put_row = [&](uint32_t pbase, uint32_t row, const uint32_t (&pk)[8]) {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int cc = k ^ (lane & 1);
                const uint32_t dst =
                    pbase + row * 128u + ((uint32_t)((colq * 2 + cc) ^ (int)(row & 7)) << 4);
                const uint32_t w0 = cc ? pk[4] : pk[0], w1 = cc ? pk[5] : pk[1];
                const uint32_t w2 = cc ? pk[6] : pk[2], w3 = cc ? pk[7] : pk[3];
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w0), "r"(w1),
                             "r"(w2), "r"(w3)
                             : "memory");
            }
        };
        bool bad = false;  // a wait gave up (the quarter learns of it at its next barrier)
        // layer 4's outputs of this CTA's iteration j, traces 4 it ..; false: leave
        auto outputs = [&](int j, int it) {
            tc_fence_after();
            uint32_t pk[8];
            finish(256u + 64u * ((uint32_t)j & 1u), bias4, pk);
            // the quarter's rows of the last tile have left
            if (storer) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            if (quarter_any(1 + quarter, bad || *abort_flag != 0)) return false;
            // a quarter's row is its lane: the store's box has position / 16
            // before position mod 16, as the accumulator's lanes do
            put_row(sOut + (uint32_t)quarter * 4096u, (uint32_t)lane, pk);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("bar.sync %0, 128;" ::"r"(1 + quarter) : "memory");
            if (storer) {
                // (traces past the batch are out of the tensor)
                asm volatile(
                    "cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                        reinterpret_cast<uint64_t>(&omap)),
                    "r"(0), "r"(8 * it), "r"(4 * quarter), "r"(sOut + (uint32_t)quarter * 4096u)
                    : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            }
            return true;
        };
        int j = 0;
        bool go = true;
        for (int it = blockIdx.x; it < iters; it += (int)gridDim.x, ++j) {
            // layer 3's outputs, worked out before the slab is free
            uint32_t pk[2][8];
#pragma unroll
            for (uint32_t X = 0; X < 2; ++X) {
                const uint32_t buf = 2u * ((uint32_t)j & 1u) + X;
                if (!mbar_wait(done3 + 8u * buf, (uint32_t)(j >> 1) & 1u)) bad = true;
                __syncwarp();
                tc_fence_after();
                finish(64u * buf, bias3, pk[X]);
            }
            // the slab's last MMAs are done
            if (j > 0 && !mbar_wait(done4 + 8u * ((uint32_t)(j - 1) & 1u), (uint32_t)((j - 1) >> 1) & 1u))
                bad = true;
#pragma unroll
            for (int X = 0; X < 2; ++X) {
                const int b = 2 * X + (mt >> 6), q = mt & 63;
                const uint32_t pbase = sL4 + (uint32_t)(q & 1) * kPlaneBytes;
                if (q <= 33) put_row(pbase, 8u * (uint32_t)((q >> 1) + 1) + 2u * (uint32_t)b, pk[X]);
                if (q >= 30) put_row(pbase, 8u * (uint32_t)((q >> 1) - 15) + 2u * (uint32_t)b + 1u, pk[X]);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(ready4) : "memory");
            if (j > 0 && !outputs(j - 1, it - (int)gridDim.x)) {
                go = false;
                break;
            }
        }
        if (go && j > 0) {
            if (!mbar_wait(done4 + 8u * ((uint32_t)(j - 1) & 1u), (uint32_t)((j - 1) >> 1) & 1u)) bad = true;
            __syncwarp();
            go = outputs(j - 1, (int)blockIdx.x + (j - 1) * (int)gridDim.x);
        }
        if (!go) *abort_flag = 1;
        if (storer) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        tc_fence_before();
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 0 && *abort_flag) atomicOr(status, PCHASE_DEV_TIMEOUT);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(kL34TmemCols)
                     : "memory");
}

// Layer 3's inputs [nb][128][64] BF16 as a 5-D tensor (channel, block of 32
// positions, trace, pair in the block, parity).  A plane's groups 1-16 are a
// box of 4 blocks x 2 traces x 16 pairs; its groups 0 and 17 are the last
// (first) pair of the blocks before (after), a box of one pair that starts one
// block early (late): zeros where that leaves the trace.
static bool conv3_in_map(const __nv_bfloat16 *x, int nb, uint32_t pairs, CUtensorMap *map) {
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[5] = {64, 4, (cuuint64_t)nb, 16, 2};
    const cuuint64_t strides[4] = {32 * 128, 128 * 128, 2 * 128, 128};
    const cuuint32_t box[5] = {64, 4, 2, pairs, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<__nv_bfloat16 *>(x), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Layer 4's outputs [nb][32][64] BF16 as (channel, row / 16, row mod 16) of
// the nb 32 rows: a lane quarter's rows are a box of 8 x 4
static bool conv4_out_map(__nv_bfloat16 *out, int nb, CUtensorMap *map) {
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[3] = {64, (cuuint64_t)nb * 2, 16};
    const cuuint64_t strides[2] = {16 * 128, 128};
    const cuuint32_t box[3] = {64, 8, 4};
    const cuuint32_t estr[3] = {1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, out, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

cudaError_t conv34_tc(const __nv_bfloat16 *x, int nb, const __nv_bfloat16 *W3, const float *bias3,
                      const __nv_bfloat16 *W4, const float *bias4, __nv_bfloat16 *out,
                      uint32_t *status, int sms, cudaStream_t st) {
    if (nb <= 0) return cudaSuccess;
    if (!status) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(conv34_tc_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kL34Smem);
    if (e != cudaSuccess) return e;
    const int grid = std::min((nb - 1) / 4 + 1, std::max(1, sms));
    CUtensorMap xmap, emap, omap;
    if (!conv3_in_map(x, nb, 16, &xmap) || !conv3_in_map(x, nb, 1, &emap) || !conv4_out_map(out, nb, &omap))
        return cudaErrorInvalidValue;
    conv34_tc_kernel<<<grid, kL34Threads, kL34Smem, st>>>(xmap, emap, nb, W3, bias3, W4, bias4, omap, status);
    return cudaGetLastError();
}

// Layer 2's outputs [nb][128][64] BF16 as a 4-D tensor (channel, position / 16,
// position mod 16, trace): a box is a trace's tile with its rows in the order
// of the accumulator's lanes, lane 8g + i holding position 16i + g
static bool conv12_out_map(__nv_bfloat16 *out, int nb, CUtensorMap *map) {
    const PFN_cuTensorMapEncodeTiled_v12000 encode = tensor_map_encoder();
    if (!encode) return false;
    const cuuint64_t dims[4] = {64, 8, 16, (cuuint64_t)nb};
    const cuuint64_t strides[3] = {16 * 128, 128, 128 * 128};
    const cuuint32_t box[4] = {64, 8, 16, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, out, dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

cudaError_t conv12_tc(const float *x, int nb, const __nv_bfloat16 *W1, const float *bias1,
                      const __nv_bfloat16 *W2, const float *bias2, __nv_bfloat16 *out,
                      uint32_t *status, int sms, cudaStream_t st) {
    if (nb <= 0) return cudaSuccess;
    if (!status) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(conv12_tc_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kFusedSmem);
    if (e != cudaSuccess) return e;
    const int grid = std::min(nb, std::max(1, sms));
    CUtensorMap omap;
    if (!conv12_out_map(out, nb, &omap)) return cudaErrorInvalidValue;
    conv12_tc_kernel<<<grid, kFusedThreads, kFusedSmem, st>>>(x, nb, W1, bias1, W2, bias2, omap,
                                                               status);
    return cudaGetLastError();
}

cudaError_t fc_heads_tc(const __nv_bfloat16 *act, int nb, const __nv_bfloat16 *W4,
                        const float *bias4, const __nv_bfloat16 *W5, const float *bias5,
                        float *logits, uint32_t *status, cudaStream_t st) {
    if (nb <= 0) return cudaSuccess;
    if (!status) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(fc_heads_tc_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kFcSmemBytes);
    if (e != cudaSuccess) return e;
    if ((reinterpret_cast<uintptr_t>(act) & 15) || (reinterpret_cast<uintptr_t>(W4) & 15))
        return cudaErrorInvalidValue;
    alignas(64) CUtensorMap amap, wmap;
    if (!kmajor_map(act, nb, kFcK, kFcK, kTileRows, &amap) ||
        !kmajor_map(W4, kFcN, kFcK, kFcK, kFcN, &wmap))
        return cudaErrorInvalidValue;
    const int grid = (nb + kTileRows - 1) / kTileRows;
    fc_heads_tc_kernel<<<grid, 128, kFcSmemBytes, st>>>(amap, wmap, nb, bias4, W5, bias5, logits,
                                                        status);
    return cudaGetLastError();
}

}  // namespace pchase
