// Hidden 64 -> 64 layers of the learned denoiser on the 5th-generation
// tensor cores (tcgen05, sm_103a): an implicit GEMM whose output strips are
// 128 pixels of one image row,
//   D[m][co] = sum_{tap, ci} A_tap[m][ci] W[co][tap*64 + ci],
// M = 128 pixels, 64 output channels per strip, K = 9 x 64.
//
// Operands are K-major with the 128-byte swizzle: a pixel's 64 channels are
// one 128-byte row, exactly as the activations lie in global memory
// ([B][H][W][64] BF16), so one TMA copy (box 64 channels x 130 pixels, zero
// fill outside the image = the convolution's zero padding) brings a whole
// halo row, and tap column dx of it starts dx rows later.
//
// An input row is multiplied once, for all the output rows it touches: image
// row i gives output row i - 1 its dy = 2 taps, row i its dy = 1 taps and row
// i + 1 its dy = 0 taps, so with the weights of one dx stacked [dy = 0; 1; 2]
// one MMA of N = 192 adds into three neighbouring 64-column accumulators.  An
// MMA of N = 64 is bound by its operand reads (54.6 cycles measured per
// 128 x 64 x 16, where the arithmetic is 32); N = 192 takes 96.2, which is the
// arithmetic alone, and reads the pixels once instead of three times.  Every
// output row still sums its taps in the order dy, dx, ci, as a per-row kernel
// would, so the results do not depend on the split.
//
// A CTA takes a contiguous range of strips, consecutive rows of one
// 128-column band, and the accumulators of its output rows pass through
// tensor memory as a ring of eight.  The epilogue (tcgen05.ld, bias + ReLU or
// the mask, BF16) leaves a strip in shared memory, and one TMA copy stores it.
//
// One 512 x 512 layer: 28.3 us with an N = 64 MMA per tap, 19.1 us in this
// form (ncu; the 17 layers of dgamp_ct_cnn_denoise 512 -> 332 us).  The MMAs
// used to wait for their issue (see mma_bf16); now a row takes about 1450
// cycles, of which its 12 MMAs' arithmetic is 1152: the operands (10 KB per
// MMA), the incoming row and the outgoing strip (twice) share the 128 bytes
// per cycle of shared memory.
//
// Every wait is bounded and reports a timeout through *err instead of hanging.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "internal.cuh"

namespace dgct {
namespace tc {

constexpr int CH = 64;
constexpr int M = 128;                    // pixels per strip (MMA M)
constexpr int HWL = M + 2;                // halo pixels loaded per row
constexpr int HWP = 136;                  // row slot: 136 pixels x 128 B = 17 x 1024 B
constexpr int A_ROW = HWP * 128;          // bytes of one row slot (pixel-major, 128-byte swizzle)
constexpr int RING = 6;                   // row slots: one being multiplied, the others landing
constexpr int FOLD_RING = 2;              // FOLD: slots of three shifted rows (the loads of one overlap the MMAs of the other)
constexpr int A_BYTES = RING * A_ROW;     // the ring
constexpr int ROW_BYTES = HWL * 128;      // bytes one row load delivers (130 pixels x 64 channels)
constexpr int B_TAP = 64 * 128;           // one tap of the weights: 64 co x 64 ci, 128-byte swizzle
constexpr int B_BYTES = 9 * B_TAP;        // [dx][dy][co][ci]
constexpr int O_BYTES = M * 128;          // one strip on its way out (and its mask on the way in)
static_assert(FOLD_RING * 3 * O_BYTES <= A_BYTES, "the shifted rows use the ring's memory");
constexpr int EPI_GROUPS = 2;             // epilogue groups of four warps: group g drains strips k % 2 == g
constexpr int SMEM = 1024 + B_BYTES + A_BYTES + EPI_GROUPS * O_BYTES;   // + alignment slack
constexpr int EPI_WARP0 = 4;              // warps 4..11: epilogue; warp 0: TMA; warp 1: MMA
                                          // (the epilogue warps start at a multiple of 4: warp % 4 is
                                          // the TMEM lane quarter a warp may read)
constexpr int THREADS = 32 * (EPI_WARP0 + 4 * EPI_GROUPS);
constexpr int ACCS = 8;                   // ring of 64-column FP32 accumulators
constexpr unsigned TMEM_COLS = 64 * ACCS;
constexpr unsigned long long WAIT_NS = 2000000000ull;   // bound of every mbarrier wait (2 s)

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// K-major operand with 128-byte swizzle (rows of 64 BF16 = 128 B, 8-row groups
// 1024 B apart): start address and SBO = 1024.  The swizzle follows the
// absolute shared-memory address (the TMA wrote with the same rule), so a
// start moved by whole 128-byte rows or by 32 bytes within a row needs no
// base offset.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1u << 16) | ((uint64_t)(1024u >> 4) << 32) |
           (1ull << 46) | (2ull << 61);
}

// kind::f16 instruction descriptor: D FP32, A and B BF16, both K-major, N = 64 count, M = 128
constexpr uint32_t IDESC0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(M >> 4) << 24);
__device__ __forceinline__ uint32_t idesc_n(int count) { return IDESC0 | ((uint32_t)(count * (64 >> 3)) << 17); }

// Called by a whole converged warp; elect.sync picks the one lane that issues
// (always the same one, so its commits cover its MMAs).  Issued from a branch
// that only lane 0 takes, an MMA took 146 cycles to issue, more than it takes to
// execute; from the converged warp they issue at the rate they execute.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        :
        : "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(mbar)
        : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t mbar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `parity` of the mbarrier; false once about `bound_ns`
// has passed, counted in SM clocks (at most 2.07 per ns; a slower clock only
// lengthens the bound).  The SM's own counter, because a read of the global
// timer takes about as long as a strip's arithmetic and every wait of the
// pipeline that is not satisfied at once would pay for one.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity,
                                          unsigned long long bound_ns = WAIT_NS) {
    if (mbar_try(mbar, parity)) return true;
    const long long t0 = clock64(), bound = 2 * (long long)bound_ns;
    for (;;) {
        if (mbar_try(mbar, parity)) return true;
        if (clock64() - t0 > bound) return false;
    }
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes) : "memory");
}

// TMA tiled loads (zero fill outside the tensor), completion counted on mbar
__device__ __forceinline__ void tma_4d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                       uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(mbar)
        : "memory");
}
__device__ __forceinline__ void tma_5d(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                       uint32_t mbar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5, %6}], [%7];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(mbar)
        : "memory");
}

// TMA tiled store (pixels outside the tensor are dropped), and its group
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* map, uint32_t src, int c0, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];\n" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void tma_store_read_wait() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void tma_store_wait() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// barrier of `threads` threads (whole warps) of the block
__device__ __forceinline__ void named_bar(int id, int threads) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

// 32 consecutive FP32 accumulator columns of this warp's 32 TMEM lanes (no wait)
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

typedef __nv_bfloat16 bf16;

// Strip s of the batch (row fastest): band = s / H is a 128-column band of
// image b = band / nx at x0 = (band % nx) * 128, row y = s % H.  A CTA takes a
// contiguous range of strips, so its consecutive strips are consecutive rows
// of one band and share two of their three input rows.
struct Strip {
    int b, y, x0;
};
__device__ __forceinline__ Strip strip_of(int s, int H, int nx) {
    const int band = s / H;
    Strip t;
    t.b = band / nx;
    t.y = s - band * H;
    t.x0 = (band - t.b * nx) * M;
    return t;
}

// Strips come in runs: the strips [s_a, s_e] of a CTA that lie in one band.  A
// run needs input rows y(s_a) - 1 .. y(s_e) + 1 (rows -1 and H load as zeros).
__device__ __forceinline__ int run_end(int s_a, int s1, int H) {
    const int e = (s_a / H + 1) * H;
    return (e < s1 ? e : s1) - 1;
}

// accumulator of a CTA's output row k: descending, so that the rows one input
// row adds to (newest first) take ascending columns and weight blocks
__device__ __forceinline__ int acc_of(int k) { return ACCS - 1 - k % ACCS; }

// Two channels (2j, 2j + 1) of the accumulator columns r: bias + ReLU
// (MODE 0) or zero where the mask is not positive (MODE 1), rounded to BF16
template <int MODE>
__device__ __forceinline__ uint32_t finish2(uint32_t r0, uint32_t r1, float2 b, uint32_t mask2) {
    float v0 = __uint_as_float(r0), v1 = __uint_as_float(r1);
    if (MODE == 0) {
        v0 = fmaxf(v0 + b.x, 0.f);
        v1 = fmaxf(v1 + b.y, 0.f);
    }
    __nv_bfloat162 p = __floats2bfloat162_rn(v0, v1);
    uint32_t o = *reinterpret_cast<uint32_t*>(&p);
    if (MODE == 1) {
        const __nv_bfloat162 m = *reinterpret_cast<__nv_bfloat162*>(&mask2);
        o &= __hgt2_mask(m, __floats2bfloat162_rn(0.f, 0.f));
    }
    return o;
}

// MODE 0: out = relu(bias + conv(in, Wk)); MODE 1: out = conv(in, Wk) * (mask > 0).
// stall_ns > 0 is the timeout test: before any copy or MMA is issued, thread 0
// waits at most stall_ns on an mbarrier that nothing arrives at, records the
// timeout in *err and the CTA returns without computing (after freeing its
// tensor memory), exactly as a wait that ran out in the loop reports it.
// Wk = layer `layer` of a [layers][co][tap*64 + ci] BF16 array (map_w); input,
// mask and output are [B][H][W][64] BF16.  CTA k takes strips [k per, (k+1) per).
// Warp-specialised, with no block barrier inside the loop:
//   warp 0 (one lane): TMA producer -- weights, then input rows into the ring,
//     a slot refilled once the MMAs of its previous row are done;
//   warp 1 (one lane): MMA issuer -- per input row 12 MMAs (3 dx x 4 channel
//     steps) over the up to three output rows it touches, then releases the
//     row's slot and hands over the output row it completes.  The first MMA of
//     an output row overwrites its accumulator, so it is issued apart;
//   warps 4..11: epilogue, two groups of four warps on alternate strips --
//     wait acc_full, read TMEM, free the accumulator (acc_empty), then bias +
//     ReLU or mask, a lane's pixel as one 128-byte row of the group's buffer
//     (swizzled, so the eight lanes of a store phase hit distinct banks), and
//     one TMA store.  The mask of the group's next strip is loaded into the
//     same buffer once the store has read it: each lane overwrites just the
//     mask chunk it has read.
//
// FOLD (images at most 64 pixels wide, the training patches): a strip is the
// same row of two images, 2 x 64 pixels, where a strip of one row would
// multiply 64 pixels of padding.  The halo columns of the two rows cannot share
// one buffer, so each row is loaded once per dx, already shifted; a slot holds
// the three copies.
template <int MODE, bool FOLD>
__global__ void __launch_bounds__(THREADS, 1)
k_conv64_tc(const __grid_constant__ CUtensorMap map_in, const __grid_constant__ CUtensorMap map_w,
            const __grid_constant__ CUtensorMap map_out, const __grid_constant__ CUtensorMap map_mask, int layer,
            const float* __restrict__ bias, int B, int H, int W, int per, unsigned* err,
            unsigned long long stall_ns) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(16) float s_bias[CH];
    __shared__ __align__(8) uint64_t row_full[RING];
    __shared__ __align__(8) uint64_t row_empty[RING];
    __shared__ __align__(8) uint64_t acc_full[ACCS];
    __shared__ __align__(8) uint64_t acc_empty[ACCS];
    __shared__ __align__(8) uint64_t mask_full[EPI_GROUPS];
    __shared__ __align__(8) uint64_t w_bar;
    __shared__ __align__(8) uint64_t never_bar;   // the timeout test's barrier: nothing arrives
    __shared__ uint32_t tmem_slot;
    __shared__ int stalled;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sB = (raw + 1023u) & ~1023u, sA = sB + B_BYTES, sO = sA + A_BYTES;
    constexpr int ring = FOLD ? FOLD_RING : RING;
    constexpr uint32_t slot_bytes = FOLD ? 3 * O_BYTES : A_ROW, dx_bytes = FOLD ? O_BYTES : 128;
    constexpr int ib = FOLD ? 2 : 1;      // images per strip
    const int nx = (W + M - 1) / M;
    const int nstrips = (B + ib - 1) / ib * H * nx;
    const int s0 = (int)blockIdx.x * per;
    const int s1 = s0 + per < nstrips ? s0 + per : nstrips;
    if (s0 >= s1) return;
    pdl_launch();   // the next layer's CTAs set up as soon as this one's shared memory is free
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int r = 0; r < RING; ++r) {
            mbar_init(smem_u32(&row_full[r]), 1);
            mbar_init(smem_u32(&row_empty[r]), 1);
        }
        for (int b = 0; b < ACCS; ++b) {
            mbar_init(smem_u32(&acc_full[b]), 1);
            mbar_init(smem_u32(&acc_empty[b]), 4);   // one arrival per warp of the group
        }
        for (int g = 0; g < EPI_GROUPS; ++g) mbar_init(smem_u32(&mask_full[g]), 1);
        mbar_init(smem_u32(&w_bar), 1);
        mbar_init(smem_u32(&never_bar), 1);
        stalled = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (MODE == 0 && tid < CH) s_bias[tid] = bias[tid];
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    bool ok = true;
    if (stall_ns) {
        if (tid == 0 && !mbar_wait(smem_u32(&never_bar), 0u, stall_ns)) stalled = 1;
        __syncthreads();
        ok = stalled == 0;
    }
    if (!ok) {
        // timeout test: nothing was issued, so nothing is in flight
    } else if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer ----
            mbar_expect_tx(smem_u32(&w_bar), B_BYTES);
            tma_5d(sB, &map_w, 0, 0, 0, 0, layer, smem_u32(&w_bar));   // weights: no kernel before this one writes them
            pdl_wait();   // the input rows are the previous layer's output
            int q = 0;
            for (int s_a = s0; s_a < s1;) {
                const int s_e = run_end(s_a, s1, H);
                const Strip t = strip_of(s_a, H, nx);
                for (int i = 0; i < s_e - s_a + 3; ++i, ++q) {
                    const int slot = q % ring;
                    if (q >= ring && !mbar_wait(smem_u32(&row_empty[slot]), (uint32_t)((q / ring - 1) & 1))) ok = false;
                    const uint32_t bar = smem_u32(&row_full[slot]);
                    const uint32_t dst = sA + (uint32_t)slot * slot_bytes;
                    mbar_expect_tx(bar, FOLD ? 3 * O_BYTES : ROW_BYTES);
                    if (FOLD) {
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx)
                            tma_4d(dst + dx * dx_bytes, &map_in, 0, dx - 1, t.y - 1 + i, ib * t.b, bar);
                    } else {
                        tma_4d(dst, &map_in, 0, t.x0 - 1, t.y - 1 + i, t.b, bar);
                    }
                }
                s_a = s_e + 1;
            }
        }
    } else if (warp == 1) {
        {
            // ---- MMA issuer (the whole warp, one elected lane issues) ----
            if (!mbar_wait(smem_u32(&w_bar), 0u)) ok = false;
            const uint64_t bdesc0 = sdesc_sw128(sB);
            // waits of input row q (ring slot, phase) and, where an output row starts with it, of
            // that row's accumulator; they run in the middle of the row before, so that the tensor
            // core still has MMAs queued
            auto ready = [&](int q, int k, bool fresh) {
                bool got = true;
                if (fresh && k >= ACCS) got = mbar_wait(smem_u32(&acc_empty[acc_of(k)]), (uint32_t)((k / ACCS - 1) & 1));
                got = mbar_wait(smem_u32(&row_full[q % ring]), (uint32_t)((q / ring) & 1)) && got;
                __syncwarp();
                fence_after();
                if (!got) ok = false;
            };
            ready(0, 0, true);
            int q = 0, k0 = 0;   // input row, and the first output row of the run, in the CTA's sequence
            for (int s_a = s0; s_a < s1;) {
                const int s_e = run_end(s_a, s1, H), R = s_e - s_a + 1;
                for (int i = 0; i < R + 2; ++i, ++q) {
                    const int slot = q % ring;
                    const int lo = i > 2 ? i - 2 : 0, hi = i < R ? i : R - 1;   // output rows this row adds to
                    const bool fresh = i < R;                                     // row i starts here (dy = 0)
                    const uint64_t a0 = sdesc_sw128(sA + (uint32_t)slot * slot_bytes);
                    // output rows hi, hi - 1, .. lo (accumulators ascending, dy = i - hi ascending) as
                    // one or, where the accumulator ring wraps, two MMAs
                    const int first = acc_of(k0 + hi), cnt = hi - lo + 1;
                    const int n1 = first + cnt > ACCS ? ACCS - first : cnt, n2 = cnt - n1;
                    const uint32_t d1 = tmem + (uint32_t)(first * 64);
                    const uint64_t w1 = bdesc0 + (uint64_t)(((i - hi) * B_TAP) >> 4);
                    const uint64_t w2 = w1 + (uint64_t)((n1 * B_TAP) >> 4);
                    const uint32_t i1 = idesc_n(n1), i2 = idesc_n(n2);
                    // first tap (dx = 0, channels 0..15): a fresh row overwrites, the older rows accumulate
                    mma_bf16(d1, a0, w1, fresh ? idesc_n(1) : i1, fresh ? 0u : 1u);
                    if (fresh && n1 > 1) mma_bf16(d1 + 64, a0, w1 + (uint64_t)(B_TAP >> 4), idesc_n(n1 - 1), 1u);
                    if (n2) mma_bf16(tmem, a0, w2, i2, 1u);
                    // pixel m of the strip reads halo pixel m + dx (dx = t / 4 rows later; FOLD: its copy);
                    // 16 channels (32 bytes of each row) per MMA
                    auto taps = [&](int t0, int t1) {
                        if (n2 == 0) {
#pragma unroll
                            for (int t = t0; t < t1; ++t)
                                mma_bf16(d1, a0 + (uint64_t)(((t / 4) * dx_bytes + (t % 4) * 32) >> 4),
                                         w1 + (uint64_t)(((t / 4) * 3 * B_TAP + (t % 4) * 32) >> 4), i1, 1u);
                        } else {
#pragma unroll
                            for (int t = t0; t < t1; ++t) {
                                const uint64_t ad = a0 + (uint64_t)(((t / 4) * dx_bytes + (t % 4) * 32) >> 4);
                                const uint64_t wo = (uint64_t)(((t / 4) * 3 * B_TAP + (t % 4) * 32) >> 4);
                                mma_bf16(d1, ad, w1 + wo, i1, 1u);
                                mma_bf16(tmem, ad, w2 + wo, i2, 1u);
                            }
                        }
                    };
                    taps(1, 6);
                    if (i < R + 1)
                        ready(q + 1, k0 + i + 1, i + 1 < R);
                    else if (s_e + 1 < s1)
                        ready(q + 1, k0 + R, true);
                    taps(6, 12);
                    mma_commit(smem_u32(&row_empty[slot]));
                    if (i >= 2) mma_commit(smem_u32(&acc_full[acc_of(k0 + i - 2)]));
                }
                k0 += R;
                s_a = s_e + 1;
            }
        }
    } else if (warp >= EPI_WARP0) {
        // ---- epilogue ----
        const int g = (warp - EPI_WARP0) >> 2, quad = warp & 3;
        const bool leader = quad == 0 && lane == 0;
        const uint32_t buf = sO + (uint32_t)(g * O_BYTES);
        const int pix = quad * 32 + lane;
        const uint32_t row = buf + (uint32_t)(pix * 128);
        auto load_mask = [&](int s) {
            const Strip t = strip_of(s, H, nx);
            mbar_expect_tx(smem_u32(&mask_full[g]), O_BYTES);
            tma_4d(buf, &map_mask, 0, t.x0, t.y, ib * t.b, smem_u32(&mask_full[g]));
        };
        if (leader) pdl_wait();   // the mask, and the buffer the output replaces, belong to earlier kernels
        if (MODE == 1 && leader && s0 + g < s1) load_mask(s0 + g);
        for (int k = g; s0 + k < s1; k += EPI_GROUPS) {
            const int a = acc_of(k);
            if (!mbar_wait(smem_u32(&acc_full[a]), (uint32_t)((k / ACCS) & 1))) ok = false;
            __syncwarp();
            fence_after();
            uint32_t v[64];
            const uint32_t taddr = tmem + (uint32_t)(a * 64) + ((uint32_t)(quad * 32) << 16);
            tmem_ld32(taddr, v);
            tmem_ld32(taddr + 32, v + 32);
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            fence_before();               // the reads are complete: the accumulator may be reused
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acc_empty[a])) : "memory");
            if (MODE == 1) {
                if (!mbar_wait(smem_u32(&mask_full[g]), (uint32_t)((k / EPI_GROUPS) & 1))) ok = false;
            } else {
                if (leader) tma_store_read_wait();      // the buffer's previous strip has been read
                named_bar(1 + g, 128);
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) {   // 16 bytes = 8 channels, at its swizzled place in the pixel's row
                const uint32_t at = row + (uint32_t)((c ^ (pix & 7)) * 16);
                uint32_t m[4] = {0u, 0u, 0u, 0u}, o[4];
                if (MODE == 1)
                    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                                 : "=r"(m[0]), "=r"(m[1]), "=r"(m[2]), "=r"(m[3])
                                 : "r"(at));
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float2 b = make_float2(0.f, 0.f);
                    if (MODE == 0) b = *reinterpret_cast<const float2*>(&s_bias[8 * c + 2 * j]);
                    o[j] = finish2<MODE>(v[8 * c + 2 * j], v[8 * c + 2 * j + 1], b, m[j]);
                }
                asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};\n" ::"r"(at), "r"(o[0]), "r"(o[1]), "r"(o[2]),
                             "r"(o[3])
                             : "memory");
            }
            fence_async_smem();
            named_bar(1 + g, 128);
            if (leader) {
                const Strip t = strip_of(s0 + k, H, nx);
                tma_store_4d(&map_out, buf, 0, t.x0, t.y, ib * t.b);
                if (MODE == 1 && s0 + k + EPI_GROUPS < s1) {
                    tma_store_read_wait();
                    load_mask(s0 + k + EPI_GROUPS);
                }
            }
        }
        if (leader) tma_store_wait();
    }
    if (!ok && (!stall_ns || tid == 0)) atomicOr(err, 1u);
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// ---------------------------------------------------- weight gradient ----
// For a layer with input activations a and output gradient g,
//   partial[tap][ci][co] = sum over pixels p of a[p + (dy - 1, dx - 1)][ci] g[p][co],  tap = 3 dy + dx,
// and the bias gradient sum_p g[p][co]: GEMMs with the pixels as K.  Both
// operands lie pixel-major in global memory (one pixel's 64 channels = one
// 128-byte row), which read with pixels as K is the MN-major operand layout
// with the 128-byte swizzle, so the convolution's TMA copies (a halo row of
// 130 activation pixels, a strip of 128 gradient pixels) feed the MMAs as they
// land.
//
// All nine taps of an activation row take two MMAs per 16 pixels, both M = 128,
// N = 192:
//   B = the gradient rows above, at and below the activation row (N = 3 x 64,
//       one row slot apart; they are its dy = 2, 1 and 0 taps);
//   A = the activation row twice, the second copy starting one pixel later
//       (M = 2 x 64, the leading-dimension offset is one 128-byte row): dx = 0
//       and 1; then from pixel 2 (and 3, which nothing reads): dx = 2.
// M = 64 halves fill half of the tensor core, and separate CTAs per dy read
// both operands three times: that form took 25.5 us per layer on 32 patches of
// 64 x 64 and two more kernels for the bias; this one takes
// 12 us per layer (ncu; the whole training pass 1296 -> 891 us).
//
// One launch covers several layers (blockIdx.y): each CTA sums its layer over a
// contiguous range of strips.  The tensor core truncates as it accumulates, an
// error that grows with the number of additions, so after a fiftieth of a layer's
// steps of 16 pixels (WG_SHARES: as many chains as a launch of one layer had CTAs
// per tap row), and WG_CHAIN at most, the sums move from tensor memory to the CTA's partial,
// where one thread per element adds them up in FP32 (1e-5 relative without, at
// 816 steps).  Sums of one sign on 32 patches of 64 x 64 are then 3.5e-7 off, with
// WG_CHAIN alone 9.0e-7, for 1% of the pass (833 against 826 us; 3% on 8 patches).
// The bias sums, terms of one sign more often than the others', are
// added in FP32 by two warps of their own from the gradient rows in shared memory:
// rows of ones beside the third tap gave them for nothing, but cut off as above
// they were up to 1.1e-6 of sum |g| away (16 images of 256 x 256, mean 1).  Warp 0
// (one lane) loads rows, warp 1 issues the MMAs, warps 2 and 3 sum the bias, warps
// 4..7 move the sums; gradient rows pass through a ring, and where three of them
// wrap around its end the MMA is split in two.
constexpr int WG_G_SLOT = M * 128;                     // 128 gradient pixels
constexpr int WG_NA = 4, WG_NG = 6;                    // row slots of the two rings
constexpr int WG_SMEM = 1024 + WG_NA * A_ROW + WG_NG * WG_G_SLOT;
constexpr int WG_THREADS = 256;
constexpr int WG_CHAIN = 320;                          // most accumulation steps (a row may start below, and end past it)
constexpr int WG_SHARES = 50;                          // chains a layer's pixels are cut into at least
constexpr unsigned WG_TMEM_COLS = 512;                 // two 192-column accumulators (a power of two)
// One partial as it lies in tensor memory, [column][lane], so that a warp's lanes write whole lines.  Column
// 64 r + co of the first accumulator: tap dy = 2 - r, dx = lane / 64, ci = lane % 64; of the second: lanes below 64
// dx = 2.  Lane 64 of the second's columns 64 + co holds the bias; its other lanes from 64 on are not written.
constexpr int WG_OUT = 2 * 192 * 128;
// kind::f16 instruction descriptor: D FP32, A and B BF16, both MN-major, M = 128, N = 64 count
__device__ __forceinline__ uint32_t idesc_wg(int count) { return idesc_n(count) | (1u << 15) | (1u << 16); }

// accumulation steps of strip s (past the image the gradient is 0)
__device__ __forceinline__ int wg_steps(int s, int H, int W, int nx) {
    const int wide = W - strip_of(s, H, nx).x0;
    return ((wide < M ? wide : M) + 15) / 16;
}

// MN-major operand, 128-byte swizzle: 64 elements along M or N per 128-byte
// row, rows are successive K (pixels), 8-row groups 1024 bytes apart, the next
// 64 elements along M or N `lbo` bytes on.  The swizzle follows the absolute
// shared-memory address, as the TMA wrote it, so a start may move by whole rows.
__device__ __forceinline__ uint64_t sdesc_sw128_mn(uint32_t saddr, uint32_t lbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)(1024u >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

__global__ void __launch_bounds__(WG_THREADS, 1)
k_wgrad64_tc(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_g, int a_first,
             int g_first, int g_step, int B, int H, int W, int per, int chain_max, float* __restrict__ partial, unsigned* err,
             unsigned long long stall_ns) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t a_full[WG_NA], a_empty[WG_NA], g_full[WG_NG], g_empty[WG_NG];
    __shared__ __align__(8) uint64_t acc_full, acc_empty;
    __shared__ __align__(8) uint64_t never_bar;
    __shared__ float bias_sum[2][CH];
    __shared__ uint32_t tmem_slot;
    __shared__ int stalled;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform
    const int group = blockIdx.x, z = blockIdx.y;
    const int la = a_first - z, lg = g_first + g_step * z;    // layer slots of the two tensors
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sA = (raw + 1023u) & ~1023u, sG = sA + WG_NA * A_ROW;
    const int nx = (W + M - 1) / M;
    const int nstrips = B * H * nx;
    const int s0 = group * per;
    const int s1 = s0 + per < nstrips ? s0 + per : nstrips;
    float* out = partial + ((size_t)z * gridDim.x + group) * WG_OUT;
    if (s0 >= s1) {   // no strips: zero partials
        for (int i = tid; i < WG_OUT; i += WG_THREADS) out[i] = 0.f;
        return;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_slot)),
                     "r"(WG_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int s = 0; s < WG_NA; ++s) {
            mbar_init(smem_u32(&a_full[s]), 1);
            mbar_init(smem_u32(&a_empty[s]), 1);
        }
        for (int s = 0; s < WG_NG; ++s) {
            mbar_init(smem_u32(&g_full[s]), 1);
            mbar_init(smem_u32(&g_empty[s]), 3);     // the MMAs and the two bias warps
        }
        mbar_init(smem_u32(&acc_full), 1);
        mbar_init(smem_u32(&acc_empty), 4);
        mbar_init(smem_u32(&never_bar), 1);
        stalled = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
    bool run = true;   // false only in the timeout test: nothing is issued
    if (stall_ns) {
        if (tid == 0 && !mbar_wait(smem_u32(&never_bar), 0u, stall_ns)) stalled = 1;
        __syncthreads();
        run = stalled == 0;
    }
    bool ok = run;
    if (run && warp == 0 && lane == 0) {
        // ---- TMA producer: per run of activation rows y .. y + R - 1 of a band, gradient rows y - 1 .. y + R ----
        int qa = 0, qg = 0;
        auto put = [&](bool act, const Strip& t, int y) {
            int& q = act ? qa : qg;
            const int n = act ? WG_NA : WG_NG, slot = q % n;
            uint64_t* full = act ? a_full : g_full;
            uint64_t* empty = act ? a_empty : g_empty;
            if (q >= n && !mbar_wait(smem_u32(&empty[slot]), (uint32_t)((q / n - 1) & 1))) return false;
            const uint32_t bar = smem_u32(&full[slot]);
            mbar_expect_tx(bar, act ? ROW_BYTES : WG_G_SLOT);
            if (act)
                tma_5d(sA + (uint32_t)(slot * A_ROW), &map_a, 0, t.x0 - 1, y, t.b, la, bar);
            else
                tma_5d(sG + (uint32_t)(slot * WG_G_SLOT), &map_g, 0, t.x0, y, t.b, lg, bar);
            ++q;
            return true;
        };
        for (int s_a = s0; ok && s_a < s1;) {
            const int s_e = run_end(s_a, s1, H);
            const Strip t = strip_of(s_a, H, nx);
            ok = put(false, t, t.y - 1) && put(false, t, t.y);
            for (int i = 0; ok && i <= s_e - s_a; ++i) ok = put(false, t, t.y + i + 1) && put(true, t, t.y + i);
            s_a = s_e + 1;
        }
        // every copy issued has landed before the CTA may exit (bounded)
        for (int j = qa > WG_NA ? qa - WG_NA : 0; j < qa; ++j)
            if (!mbar_wait(smem_u32(&a_full[j % WG_NA]), (uint32_t)((j / WG_NA) & 1))) ok = false;
        for (int j = qg > WG_NG ? qg - WG_NG : 0; j < qg; ++j)
            if (!mbar_wait(smem_u32(&g_full[j % WG_NG]), (uint32_t)((j / WG_NG) & 1))) ok = false;
    } else if (run && warp == 1) {
        // ---- MMA issuer (the whole warp, one elected lane issues) ----
        int qa = 0, qg = 0, seen = 0;   // activation row, first of its gradient rows, gradient rows waited for
        int chain = 0, flushes = 0;     // steps since the accumulators were emptied, and how often they were
        for (int s_a = s0; ok && s_a < s1;) {
            const int s_e = run_end(s_a, s1, H);
            const int nks = wg_steps(s_a, H, W, nx);
            for (int i = 0; i <= s_e - s_a; ++i, ++qa, ++qg) {
                bool got = true;
                if (chain >= chain_max) {
                    mma_commit(smem_u32(&acc_full));
                    got = mbar_wait(smem_u32(&acc_empty), (uint32_t)(flushes & 1));
                    ++flushes;
                    chain = 0;
                }
                got = mbar_wait(smem_u32(&a_full[qa % WG_NA]), (uint32_t)((qa / WG_NA) & 1)) && got;
                for (; seen < qg + 3; ++seen)
                    got = mbar_wait(smem_u32(&g_full[seen % WG_NG]), (uint32_t)((seen / WG_NG) & 1)) && got;
                if (!__all_sync(0xffffffffu, got)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t a0 = sA + (uint32_t)((qa % WG_NA) * A_ROW);
                const int gs = qg % WG_NG, n1 = gs + 3 > WG_NG ? WG_NG - gs : 3, n2 = 3 - n1;
                const uint64_t g1 = sdesc_sw128_mn(sG + (uint32_t)(gs * WG_G_SLOT), WG_G_SLOT);
                const uint64_t g2 = sdesc_sw128_mn(sG, WG_G_SLOT);
                const uint32_t d2 = tmem + (uint32_t)(n1 * 64), i1 = idesc_wg(n1), i2 = idesc_wg(n2);
#pragma unroll 1
                for (int ks = 0; ks < nks; ++ks) {
                    const uint32_t acc = (chain | ks) != 0 ? 1u : 0u;
                    const uint64_t go = (uint64_t)((ks * 16 * 128) >> 4);
                    const uint32_t at = a0 + (uint32_t)(ks * 16 * 128);
                    const uint64_t a01 = sdesc_sw128_mn(at, 128u), a2 = sdesc_sw128_mn(at + 256u, 128u);
                    mma_bf16(tmem, a01, g1 + go, i1, acc);
                    if (n2) mma_bf16(d2, a01, g2 + go, i2, acc);
                    mma_bf16(tmem + 192u, a2, g1 + go, i1, acc);
                    if (n2) mma_bf16(d2 + 192u, a2, g2 + go, i2, acc);
                }
                chain += nks;
                mma_commit(smem_u32(&a_empty[qa % WG_NA]));
                mma_commit(smem_u32(&g_empty[qg % WG_NG]));
            }
            if (ok)   // the run's last two gradient rows
                for (int k = 0; k < 2; ++k, ++qg) mma_commit(smem_u32(&g_empty[qg % WG_NG]));
            s_a = s_e + 1;
        }
        // arrives once every MMA issued above has completed
        mma_commit(smem_u32(&acc_full));
    } else if (run && warp < 4 && warp >= 2) {
        // ---- bias: each gradient row of the strips once; a thread takes 8 channels of every eighth pixel, adds a
        // row's pixels apart and joins them to its total with Kahan's correction ----
        const int t = tid - 64, chunk = t & 7, p0 = t >> 3;
        const uint32_t at = sG + (uint32_t)(p0 * 128 + ((chunk ^ p0) * 16));      // swizzled as the TMA wrote it
        float tot[8] = {}, corr[8] = {};
        int qg = 0;
        for (int s_a = s0; ok && s_a < s1;) {
            const int R = run_end(s_a, s1, H) - s_a + 1, eights = 2 * wg_steps(s_a, H, W, nx);
            for (int i = 0; i < R + 2; ++i, ++qg) {      // rows 0 and R + 1 lie outside the run
                const int slot = qg % WG_NG;
                if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&g_full[slot]), (uint32_t)((qg / WG_NG) & 1)))) {
                    ok = false;
                    break;
                }
                if (i >= 1 && i <= R) {
                    float row[8] = {};
                    for (int j = 0; j < eights; ++j) {
                        uint32_t v[4];
                        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                                     : "r"(at + (uint32_t)(slot * WG_G_SLOT + j * 1024)));
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            row[2 * k] += __uint_as_float(v[k] << 16);
                            row[2 * k + 1] += __uint_as_float(v[k] & 0xFFFF0000u);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float y = row[k] - corr[k], n = tot[k] + y;
                        corr[k] = (n - tot[k]) - y;
                        tot[k] = n;
                    }
                }
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&g_empty[slot])) : "memory");
            }
            s_a += R;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], 8);
            tot[k] += __shfl_xor_sync(0xffffffffu, tot[k], 16);
            if (lane < 8) bias_sum[warp - 2][chunk * 8 + k] = tot[k];
        }
        named_bar(1, 64);
        out[(256 + t) * 128 + 64] = bias_sum[0][t] + bias_sum[1][t];
    } else if (run && warp >= 4) {
        // ---- sums from tensor memory to the partial: stored the first time, then added (each element by
        // one thread, so in a fixed order) ----
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const int m = (warp & 3) * 32 + lane;
        int chain = 0, flushes = 0;
        for (int s = s0; s < s1; ++s) {
            chain += wg_steps(s, H, W, nx);
            if (chain < chain_max && s + 1 < s1) continue;
            if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&acc_full), (uint32_t)(flushes & 1)))) {
                ok = false;
                break;
            }
            fence_after();
#pragma unroll 1
            for (int c = 0; c < 12; ++c) {   // 32 columns: accumulator c / 6, gradient row c / 2 % 3, half of co
                uint32_t v[32];
                __syncwarp();
                tmem_ld32(tmem + lane_base + (uint32_t)(c * 32), v);   // warp-collective
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                if (c >= 6 && m >= 64) continue;
                float* dst = out + c * 32 * 128 + m;
                if (flushes == 0) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) dst[j * 128] = __uint_as_float(v[j]);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        asm volatile("red.global.add.f32 [%0], %1;\n" ::"l"(dst + j * 128), "f"(__uint_as_float(v[j]))
                                     : "memory");
                }
            }
            fence_before();               // the reads are complete: the accumulators may be overwritten
            __syncwarp();
            if (lane == 0)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acc_empty)) : "memory");
            ++flushes;
            chain = 0;
        }
    }
    __syncwarp();
    if (!ok && (run || tid == 0)) atomicOr(err, 1u);
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(WG_TMEM_COLS)
                     : "memory");
    }
}

}  // namespace tc
}  // namespace dgct

namespace dgct {

int conv64_tc_init() {
    const void* convs[] = {(const void*)tc::k_conv64_tc<0, false>, (const void*)tc::k_conv64_tc<1, false>,
                           (const void*)tc::k_conv64_tc<0, true>, (const void*)tc::k_conv64_tc<1, true>};
    for (const void* k : convs)
        DGCT_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::SMEM));
    DGCT_CUDA(cudaFuncSetAttribute(tc::k_wgrad64_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, tc::WG_SMEM));
    return DGAMP_CT_OK;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn tensor_map_encoder() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

static int encode(CUtensorMap* map, cuuint32_t rank, const void* base, const cuuint64_t* dims,
                  const cuuint64_t* strides, const cuuint32_t* box) {
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn) return cuda_fail(cudaErrorNotSupported);
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), dims, strides, box,
                          es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? DGAMP_CT_OK : cuda_fail(cudaErrorInvalidValue);
}

// in: [B][H][W][64] BF16; wk_all: [layers][64][576] BF16 (layer `layer` used);
// out (mode 0: bias + ReLU, mode 1: times mask > 0) like in.
int launch_conv64_tc(int mode, const void* in, const void* wk_all, int layers, int layer, const float* bias,
                     const void* mask, void* out, int B, int H, int W, int grid_cap, unsigned* err, cudaStream_t st,
                     unsigned long long stall_ns) {
    // rows of at most half a strip are taken two images at a time: 64-pixel rows as they are cost a whole
    // strip each (32 patches of 64 x 64, the training pass 891 -> 847 us; bound by the L2 reads
    // of the three copies)
    const bool fold = W <= tc::M / 2 && B > 1;
    const long long nstrips = (long long)(fold ? (B + 1) / 2 : B) * H * ((W + tc::M - 1) / tc::M);
    if (nstrips <= 0) return DGAMP_CT_OK;
    if (layer < 0 || layer >= layers) return DGAMP_CT_ERR_INVALID_ARG;
    CUtensorMap map_in, map_w, map_out, map_mask;
    {
        const cuuint64_t dims[4] = {64, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
        const cuuint64_t strides[3] = {128, (cuuint64_t)W * 128, (cuuint64_t)H * W * 128};
        const cuuint32_t box[4] = {64, (cuuint32_t)tc::HWL, 1, 1};
        const cuuint32_t whole[4] = {64, (cuuint32_t)tc::M, 1, 1}, pair[4] = {64, (cuuint32_t)tc::M / 2, 1, 2};
        const cuuint32_t* strip = fold ? pair : whole;
        DGCT_TRY(encode(&map_in, 4, in, dims, strides, fold ? pair : box));
        DGCT_TRY(encode(&map_out, 4, out, dims, strides, strip));
        DGCT_TRY(encode(&map_mask, 4, mode == 1 ? mask : in, dims, strides, strip));
    }
    {
        // [layers][co][dy][dx][ci], fetched as [dx][dy][co][ci]
        const cuuint64_t dims[5] = {64, 64, 3, 3, (cuuint64_t)layers};
        const cuuint64_t strides[4] = {1152, 384, 128, 1152 * 64};
        const cuuint32_t box[5] = {64, 64, 3, 3, 1};
        DGCT_TRY(encode(&map_w, 5, wk_all, dims, strides, box));
    }
    // contiguous ranges of strips, one per CTA, at most grid_cap CTAs
    const int cap = grid_cap > 0 ? grid_cap : 1;
    const int per = (int)((nstrips + cap - 1) / cap);
    const int grid = (int)((nstrips + per - 1) / per);
    const auto kernel = fold ? (mode == 0 ? tc::k_conv64_tc<0, true> : tc::k_conv64_tc<1, true>)
                             : (mode == 0 ? tc::k_conv64_tc<0, false> : tc::k_conv64_tc<1, false>);
    DGCT_CUDA(launch_pdl(kernel, dim3(grid), dim3(tc::THREADS), tc::SMEM, st,
                         map_in, map_w, map_out, map_mask, layer, bias, B, H, W, per, err, stall_ns));
    return DGAMP_CT_OK;
}

// Layers z = 0 .. nl - 1: input activations in slot a_first - z of `acts`,
// output gradients in slot g_first + g_step z of `grads`, both
// [slots][slot][64] BF16 with slot = slot_pix pixels of which the first B H W
// are used; partial: [nl][groups][wgrad64_partial_floats()] FP32 in the kernel's
// [column][lane] layout, whose entries without a meaning are left unwritten
// (a group without strips is all zeros).
int wgrad64_partial_floats() { return tc::WG_OUT; }
int launch_wgrad64_tc(const void* acts, int act_slots, int a_first, const void* grads, int grad_slots, int g_first,
                      int g_step, long long slot_pix, int nl, int B, int H, int W, int groups, float* partial,
                      unsigned* err, cudaStream_t st, unsigned long long stall_ns) {
    if (groups < 1 || nl < 1) return DGAMP_CT_ERR_INVALID_ARG;
    const long long nstrips = (long long)B * H * ((W + tc::M - 1) / tc::M);
    if (nstrips <= 0) {
        DGCT_CUDA(cudaMemsetAsync(partial, 0, (size_t)nl * groups * tc::WG_OUT * sizeof(float), st));
        return DGAMP_CT_OK;
    }
    CUtensorMap map_a, map_g;
    const cuuint64_t strides[4] = {128, (cuuint64_t)W * 128, (cuuint64_t)H * W * 128, (cuuint64_t)slot_pix * 128};
    {
        const cuuint64_t dims[5] = {64, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B, (cuuint64_t)act_slots};
        const cuuint32_t box[5] = {64, (cuuint32_t)tc::HWL, 1, 1, 1};
        DGCT_TRY(encode(&map_a, 5, acts, dims, strides, box));
    }
    {
        const cuuint64_t dims[5] = {64, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B, (cuuint64_t)grad_slots};
        const cuuint32_t box[5] = {64, (cuuint32_t)tc::M, 1, 1, 1};
        DGCT_TRY(encode(&map_g, 5, grads, dims, strides, box));
    }
    const int per = (int)((nstrips + groups - 1) / groups);
    long long steps = 0;      // of a layer: 16 pixels each
    for (int x = 0; x < W; x += tc::M) steps += (std::min(W - x, tc::M) + 15) / 16;
    steps *= (long long)B * H;
    const int chain_max = (int)std::min<long long>(tc::WG_CHAIN, (steps + tc::WG_SHARES - 1) / tc::WG_SHARES);
    tc::k_wgrad64_tc<<<dim3(groups, nl), tc::WG_THREADS, tc::WG_SMEM, st>>>(map_a, map_g, a_first, g_first, g_step, B, H,
                                                                           W, per, chain_max, partial, err, stall_ns);
    DGCT_LAUNCH_CHECK();
    return DGAMP_CT_OK;
}

}  // namespace dgct
