// 3x3 circular convolution of the surrogate as an implicit GEMM on the fifth-
// generation tensor cores: tcgen05.mma (kind::f16, BF16 operands from shared
// memory, FP32 accumulator in tensor memory), issued by one elected lane of a warp.
//
// Tiling.  A CTA computes MT tiles of 128 output pixels (each 16 rows x 8 columns;
// the MT tiles side by side) for BN output channels: the accumulator
// D[pixel][co] of tile j sits in tensor-memory lanes 0..127 (lane = pixel) and
// columns j BN .. j BN + BN - 1 (two such accumulators, alternating between output
// blocks).  The input block with its one-pixel halo ((16 + 2) x (8 MT + 2) pixels)
// is staged per 16-channel chunk as two planes of 8 channels, one 16-byte row per
// pixel: the K-major operand layout without swizzle, whose 8-row core matrices are
// then 8 consecutive pixels of one image row.  A stencil tap (dy, dx) is a
// descriptor into that same block, started dy halo rows and dx pixels further on,
// with the stride between 8-row groups (SBO) = one halo row and between the two K
// halves (LBO) = one plane; no im2col copy is made.  The weights of a chunk's nine
// taps arrive by one tensor copy as rows of 32 bytes (an output channel's 16 input
// channels) in the 32-byte swizzled layout; they stay resident for the whole kernel
// when all chunks fit in shared memory.
//
// Precision is that of the mma.sync kernels: activations split into BF16 hi + lo
// (two MMAs per tap; one with act_bf16), BF16 weights, FP32 accumulation.
//
// Pipeline (conv3_tc_kernel below): persistent CTAs, one per SM, with warp roles.
// Producer warps load the FP32 chunks a few steps ahead into registers and convert
// them into the BF16 operand buffers; one warp issues the MMAs; four warps read the
// accumulators (tcgen05.ld), add the bias, apply ReLU and store FP32 (or add into
// the destination); one warp streams the weights when they are not resident.  The
// roles hand buffers and accumulators to each other through mbarriers.
//
// Every wait is bounded (about two seconds of SM clock).  A wait that runs out
// sets a device flag (read by conv3_tc_take_timeout) and makes every role leave its
// loop; the MMA warp waits (bounded) for the MMAs it has in flight, and the CTA
// frees its tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "lbm_tma.cuh"
#include "nn_conv_tc.h"

#ifndef LBM_CONV_TC_STAGES
#define LBM_CONV_TC_STAGES 0    // BF16 operand buffers; 0 = three
#endif
#ifndef LBM_CONV_TC_DEPTH
#define LBM_CONV_TC_DEPTH 3     // FP32 chunks in flight per producer thread (registers)
#endif

namespace {

__device__ int g_tc_timeout;

constexpr int kMaxStages = 4;
constexpr long long kWaitCycles = 4000000000LL;
constexpr int kSmemLimit = 227 * 1024 - 1024;   // dynamic shared memory per CTA (static part kept below 1 KB)
constexpr int kTmemColumns = 512;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor in two words.  Low: start address and leading-dimension (K) byte
// offset, each >> 4 in 14 bits; high: stride-dimension (M / N) byte offset >> 4 in 14 bits, descriptor
// version 1 at bits 46-47, swizzle mode at bits 61-63.  Addresses stay below 2^14 * 16 bytes, so a
// descriptor further on is the low word plus the distance >> 4.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return (addr >> 4) | ((lbo >> 4) << 16); }
constexpr uint32_t kNoSwizzle = 0u, kSwizzle32 = 6u;
constexpr uint32_t desc_hi(uint32_t sbo, uint32_t swizzle) { return (sbo >> 4) | (1u << 14) | (swizzle << 29); }

// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A and B BF16
// (bits 7-9 = 1, 10-12 = 1), no negation, both K-major (bits 15, 16 = 0), dense,
// N >> 3 at bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t idesc_bf16_f32(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// D (+)= A B^T with A, B in shared memory (descriptors) and D in tensor memory.  Executed by a
// whole converged warp: one lane (elect.sync) issues the instruction, so that the operands can
// stay in warp-uniform registers.
template <uint32_t A_HI, uint32_t B_HI, uint32_t IDESC>
__device__ __forceinline__ void mma_bf16_ss_elect(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t.reg .b64 da, db;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %3, 0;\n\t"
        "mov.b64 da, {%1, %4};\n\t"
        "mov.b64 db, {%2, %5};\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %6, p;\n\t"
        "}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(b_lo), "r"(accumulate), "n"(A_HI), "n"(B_HI), "r"(IDESC)
        : "memory");
}

// arrive on the mbarrier once every tcgen05 operation issued so far by the elected lane has completed
__device__ __forceinline__ void mma_commit_elect(uint32_t bar)
{
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t"
        "}\n" ::"r"(bar)
        : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t"
        "}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// wait for the completion of the barrier's phase with this parity; false after ~2 s
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try(bar, parity))
        if (clock64() - t0 > kWaitCycles) return false;
    return true;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld_16x32_issue(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
// keeps the uses of loaded registers behind the wait
__device__ __forceinline__ void behind_the_wait(uint32_t (&r)[16])
{
    asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                      "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                      "+r"(r[15]));
}

// 16 lanes x 32 columns of an accumulator as matrix fragments: v[4 j + 2 h + e] is lane lane/4 + 8 h,
// column 8 j + 2 (lane % 4) + e.  Two of them per wait.
__device__ __forceinline__ void tmem_ld_16x32_pair(uint32_t taddr0, uint32_t taddr1, uint32_t (&r)[2][16])
{
    tmem_ld_16x32_issue(taddr0, r[0]);
    tmem_ld_16x32_issue(taddr1, r[1]);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    behind_the_wait(r[0]);
    behind_the_wait(r[1]);
}

__device__ __forceinline__ void tmem_ld_16x32(uint32_t taddr, uint32_t (&r)[16])
{
    tmem_ld_16x32_issue(taddr, r);
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    behind_the_wait(r);
}

__device__ __forceinline__ uint32_t bf16x2_bits(__nv_bfloat162 v) { return *reinterpret_cast<const uint32_t*>(&v); }

// warp roles
constexpr int kProducerWarps = 12;      // warps 0-11: activations (FP32 -> BF16 hi / lo)
constexpr int kEpilogueWarp0 = 12;      // warps 12-15: accumulator -> global (TMEM lanes 32 (w % 4) ..)
constexpr int kMmaWarp = 16;            // warp 16: tensor-memory allocation; the MMA loop (elected lane issues)
constexpr int kWeightWarp = 17;         // warp 17: tensor copies of the weights
constexpr int kThreads = 18 * 32;
constexpr int kProducers = kProducerWarps * 32;
static_assert(kEpilogueWarp0 % 4 == 0 && kEpilogueWarp0 == kProducerWarps && kEpilogueWarp0 + 4 == kMmaWarp, "warp roles");

template <int BN, int MT, bool LO>
struct TcShape {
    static constexpr int TH = 16, TW = 8 * MT;               // output block (MT tiles of 16 x 8)
    static constexpr int HWD = TW + 2, HP = (TH + 2) * HWD;  // halo block width, pixels
    static constexpr int NQ = (HP * 2 + kProducers - 1) / kProducers;   // 8-channel items per producer thread per chunk
    static constexpr int PLANE = HP * 16;                    // 8 channels of every halo pixel (BF16)
    static constexpr int A_HALF = 2 * PLANE;                 // one BF16 half of a 16-channel chunk
    static constexpr int A_BYTES = (LO ? 2 : 1) * A_HALF;
    static constexpr int B_TAP = BN * 32;                    // BN weight rows of 16 input channels, 32-byte swizzle
    static constexpr int B_BYTES = 9 * B_TAP;                // weights of one 16-channel chunk
    static constexpr int ACC = MT * BN;                      // accumulator columns of one block
    static constexpr int COLS = 2 * ACC <= 32 ? 32 : 2 * ACC <= 64 ? 64 : 2 * ACC <= 128 ? 128
                                : 2 * ACC <= 256 ? 256 : 512;   // two accumulators
    static constexpr uint32_t IDESC = idesc_bf16_f32(128, BN);
    static constexpr uint32_t A_HI = desc_hi(HWD * 16, kNoSwizzle), B_HI = desc_hi(256, kSwizzle32);
    // operand buffers rounded up so that the weights start on a 256-byte boundary (the swizzle's period)
    static constexpr int ring_bytes(int stages) { return (stages * A_BYTES + 255) / 256 * 256; }
    static_assert(BN % 16 == 0 && BN >= 32 && BN <= 128 && MT >= 1 && MT <= 2, "tile");
};

template <int I> struct Const { static constexpr int value = I; };

struct TcConf {
    int stages;     // BF16 operand buffers (and weight buffers when not resident)
    int resident;   // the weights of all chunks stay in shared memory
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// bounded wait that also gives up once another role has given up (`abort_flag`)
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort_flag = 1;
            return false;
        }
    }
}

// Persistent, warp-specialised.  CTA b takes the output blocks b, b + gridDim.x, ...
// (output channels of blockIdx.y) and walks their 16-channel chunks as one sequence
// g = 0 .. G-1.  Barriers: full[s] (activations of the chunk in buffer s staged: one
// arrival per producer warp), wfull[s] (weights of the chunk in buffer s landed; resident weights:
// wfull[0], all of them), empty[s] (the MMAs that read buffer s completed: tcgen05.commit),
// acc_full[b] (the MMAs of the block in accumulator b completed), acc_empty[b] (the epilogue warps
// have read accumulator b: one arrival per warp).
// Shared memory: [BF16 operand buffers][weights].
//
// What bounds it: an MMA takes max(32 + BN / 4, BN / 2) clocks (128 rows of A and BN of B read from
// shared memory at 128 bytes per clock, or the arithmetic), measured alike for every operand layout and
// alignment: 1450 clocks per chunk at BN = 32, 2300 at 128.  At BN = 128 the MMAs take three quarters
// of the time (the rest: the first chunk's way in and the last block's way out, one or two blocks per
// CTA); at BN = 32 shared memory is shared with the conversion and the stores (about 2000 clocks per
// chunk).  Before, the weights came by one warp's 16-byte copies (2.4 us per chunk at BN = 128; now one
// tensor copy, box 16 channels x BN x 9 taps), and eight warps converted 4-channel items (1.5 us per
// chunk).  16 samples: 32 -> 32 channels at 256^2 100 -> 76 us, 64 + 32 -> 32 229 -> 170, 128 + 64 -> 64
// at 128^2 146 -> 100, 256 + 128 -> 128 at 64^2 117 -> 78, 256 -> 256 at 32^2 47 -> 35.
template <int BN, int MT, bool LO>
__global__ void __launch_bounds__(kThreads, 1)
    conv3_tc_kernel(const __grid_constant__ CUtensorMap wmap, ConvTcArgs a, TcConf cf)
{
    using S = TcShape<BN, MT, LO>;
    extern __shared__ __align__(128) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], wfull[kMaxStages], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    volatile int* abort_v = &abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tiles_x = a.W / S::TW, tiles_y = a.H / S::TH;      // powers of two
    const int ltx = 31 - __clz(tiles_x), lty = 31 - __clz(tiles_y);
    const int ntiles = a.B * tiles_x * tiles_y;
    const int co0 = blockIdx.y * BN;
    const int Cin = a.C1 + a.C2;
    const int nchunk = Cin / 16;
    const int my_tiles = (int)blockIdx.x < ntiles ? (ntiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int G = my_tiles * nchunk;
    const int stages = cf.stages;
    uint8_t* const ring = smem_raw + (0u - smem_addr(smem_raw) & 255u);
    const uint32_t wts = smem_addr(ring) + S::ring_bytes(stages);

    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(&tmem_slot)),
                     "r"((uint32_t)S::COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < stages; ++i) {
            mbar_init(smem_addr(&full[i]), kProducerWarps);   // one arrival per warp
            mbar_init(smem_addr(&empty[i]), 1);
            mbar_init(smem_addr(&wfull[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_addr(&acc_full[i]), 1);
            mbar_init(smem_addr(&acc_empty[i]), 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    auto tile_of = [&](int t, int& n, int& ty0, int& tx0) {
        const int tile = (int)blockIdx.x + t * (int)gridDim.x;
        n = tile >> (ltx + lty);
        ty0 = ((tile >> ltx) & (tiles_y - 1)) * S::TH;
        tx0 = (tile & (tiles_x - 1)) * S::TW;
    };

    if (warp < kProducerWarps) {
        // ---- activations: the FP32 loads of chunk g + DEPTH are issued once chunk g is converted.
        // An item is one pixel's 8 channels of a plane: 32 bytes read, 16 bytes of hi and of lo written
        // (the two planes lie 64 bytes apart modulo 128, so eight lanes' stores share no bank).  This
        // loop paced the kernel with 4-channel items on eight warps and divisions per chunk: 1.5 us per
        // chunk, with one MMA per tap as with two. ----
        constexpr int DEPTH = LBM_CONV_TC_DEPTH;
        static_assert(S::PLANE % 128 == 64, "planes half a line apart");
        // element offsets of this thread's halo pixels in the block being loaded: full resolution, and
        // halved for an x1 stored at half size
        uint32_t pix_full[S::NQ], pix_half[S::NQ];
        float4 v[DEPTH][S::NQ][2];
        int lt = 0, lc = 0;                                // block and chunk of the next load
        auto load = [&](float4 (&u)[S::NQ][2]) {
            if (lt == my_tiles) return;
            if (lc == 0) {
                int n, ty0, tx0;
                tile_of(lt, n, ty0, tx0);
#pragma unroll
                for (int i = 0; i < S::NQ; ++i) {
                    const int hp = (tid + kProducers * i) >> 1;
                    const int hy = hp / S::HWD, hx = hp - hy * S::HWD;
                    const int sy = (ty0 + hy - 1) & (a.H - 1), sx = (tx0 + hx - 1) & (a.W - 1);
                    pix_full[i] = ((uint32_t)n * (uint32_t)a.H + (uint32_t)sy) * (uint32_t)a.W + (uint32_t)sx;
                    pix_half[i] = ((uint32_t)n * (uint32_t)(a.H >> 1) + (uint32_t)(sy >> 1)) * (uint32_t)(a.W >> 1) +
                                  (uint32_t)(sx >> 1);
                }
            }
            const int ci0 = lc * 16;
            const bool from1 = ci0 < a.C1;
            const float* base = (from1 ? a.x1 + ci0 : a.x2 + (ci0 - a.C1)) + (tid & 1) * 8;
            const uint32_t cstride = (uint32_t)(from1 ? a.C1 : a.C2);
            const bool half = from1 && a.x1_half;          // nearest upsampling of a half-size x1
#pragma unroll
            for (int i = 0; i < S::NQ; ++i)
                if (tid + kProducers * i < S::HP * 2) {
                    const float4* p = reinterpret_cast<const float4*>(
                        base + (unsigned long long)(half ? pix_half[i] : pix_full[i]) * cstride);
                    u[i][0] = __ldg(p);
                    u[i][1] = __ldg(p + 1);
                }
            if (++lc == nchunk) {
                lc = 0;
                ++lt;
            }
        };
#pragma unroll
        for (int d = 0; d < DEPTH; ++d) load(v[d]);
        bool ok = true;
        int s = 0;
        uint32_t ph = 1;                                   // the first round of buffers is free
        for (int g0 = 0; g0 < G && ok; g0 += DEPTH) {
#pragma unroll
            for (int d = 0; d < DEPTH; ++d) {
                const int g = g0 + d;
                if (g >= G) break;
                // (warp-uniform, so that the whole warp leaves together after an abort)
                if (g >= stages) ok = __all_sync(0xffffffffu, wait_or_abort(smem_addr(&empty[s]), ph, abort_v));
                if (!ok) break;
                uint8_t* st = ring + s * S::A_BYTES + (tid & 1) * S::PLANE;
#pragma unroll
                for (int i = 0; i < S::NQ; ++i) {
                    const int q = tid + kProducers * i;
                    if (q < S::HP * 2) {
                        uint32_t hi[4], lo[4];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float4 u = v[d][i][e];
                            const __nv_bfloat162 h01 = __floats2bfloat162_rn(u.x, u.y), h23 = __floats2bfloat162_rn(u.z, u.w);
                            hi[2 * e] = bf16x2_bits(h01);
                            hi[2 * e + 1] = bf16x2_bits(h23);
                            if constexpr (LO) {
                                const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
                                lo[2 * e] = bf16x2_bits(__floats2bfloat162_rn(u.x - f01.x, u.y - f01.y));
                                lo[2 * e + 1] = bf16x2_bits(__floats2bfloat162_rn(u.z - f23.x, u.w - f23.y));
                            }
                        }
                        const int off = (q >> 1) * 16;
                        *reinterpret_cast<uint4*>(st + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                        if constexpr (LO)
                            *reinterpret_cast<uint4*>(st + S::A_HALF + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> tensor core
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&full[s]));              // for the whole warp
                load(v[d]);
                if (++s == stages) {
                    s = 0;
                    ph ^= 1u;
                }
            }
        }
    } else if (warp < kEpilogueWarp0 + 4) {
        // ---- epilogue: accumulator of block t -> bias, ReLU, FP32 stores ----
        // Read as matrix fragments (16 pixels x 32 channels per load): four lanes then hold 8 adjacent
        // channels of a pixel and a store covers whole 32-byte sectors.  One pixel per lane stored
        // 16-byte pieces of 32 different lines at a time, every sector twice.
        // With one warp per scheduler the loop is bound by its own instructions' latency, so addresses
        // are one base per block plus 32-bit offsets and the bias stays in registers.
        const int q = warp & 3, gr = lane >> 2, t4 = lane & 3;
        constexpr int NC = BN / 32;                          // 32-column pieces of a tile's accumulator
        const int Co2 = a.Cout - a.Co1;
        float2 bias[BN / 8];
#pragma unroll
        for (int j = 0; j < BN / 8; ++j)
            bias[j] = a.bias ? __ldg(reinterpret_cast<const float2*>(a.bias + co0 + 8 * j + 2 * t4)) : make_float2(0.f, 0.f);
        for (int t = 0; t < my_tiles; ++t) {
            const bool ok = wait_or_abort(smem_addr(&acc_full[t & 1]), (uint32_t)((t >> 1) & 1), abort_v);
            if (!__all_sync(0xffffffffu, ok)) break;
            tc_fence_after();
            int n, ty0, tx0;
            tile_of(t, n, ty0, tx0);
            // TMEM lane m = pixel (m >> 3, m & 7) of a tile; this lane's first pixel
            const long long p0 = ((long long)n * a.H + ty0 + q * 4) * a.W + tx0 + gr;
            float* const y1 = a.y1 + p0 * a.Co1 + 2 * t4;
            float* const y2 = a.y2 + p0 * Co2 + 2 * t4 - a.Co1;
            const uint32_t acc = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)((t & 1) * S::ACC);
            // 16 lanes (half hh) x 32 columns (piece c) of tile j
            auto put = [&](const uint32_t (&v)[16], int j, int hh, auto piece) {
                constexpr int c = decltype(piece)::value;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int dp = (2 * hh + h) * a.W + 8 * j;
                    float* const r1 = y1 + dp * a.Co1;
                    float* const r2 = y2 + dp * Co2;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int co = co0 + 32 * c + 8 * k;            // 8 channels, all in y1 or all in y2
                        float* const dst = (co < a.Co1 ? r1 : r2) + co;
                        float2 r = make_float2(__uint_as_float(v[4 * k + 2 * h]), __uint_as_float(v[4 * k + 2 * h + 1]));
                        if (a.bias) {
                            r.x += bias[4 * c + k].x;
                            r.y += bias[4 * c + k].y;
                        }
                        if (a.relu) {
                            r.x = fmaxf(r.x, 0.f);
                            r.y = fmaxf(r.y, 0.f);
                        }
                        if (a.beta) {
                            const float2 o = *reinterpret_cast<const float2*>(dst);
                            r.x += o.x;
                            r.y += o.y;
                        }
                        *reinterpret_cast<float2*>(dst) = r;
                    }
                }
            };
            uint32_t v[2][16];
            if constexpr (NC == 1) {
#pragma unroll 1
                for (int j = 0; j < MT; ++j) {
                    tmem_ld_16x32_pair(acc + j * BN, acc + (16u << 16) + j * BN, v);
                    put(v[0], j, 0, Const<0>());
                    put(v[1], j, 1, Const<0>());
                }
            } else {
#pragma unroll 1
                for (int jh = 0; jh < 2 * MT; ++jh) {
                    const int j = jh >> 1, hh = jh & 1;
                    const uint32_t at = acc + ((uint32_t)(16 * hh) << 16) + j * BN;
                    tmem_ld_16x32_pair(at, at + 32, v);
                    put(v[0], j, hh, Const<0>());
                    put(v[1], j, hh, Const<1>());
                    if constexpr (NC == 4) {
                        tmem_ld_16x32_pair(at + 64, at + 96, v);
                        put(v[0], j, hh, Const<2>());
                        put(v[1], j, hh, Const<3>());
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&acc_empty[t & 1]));
        }
    } else if (warp == kMmaWarp) {
        // ---- MMAs: the whole warp runs the loop (warp-uniform control flow and operands),
        //      one elected lane issues each instruction ----
        int last = -1, t = 0, c = 0, s = 0;
        uint32_t ph = 0;
        // Operands of chunk g (buffer s, phase ph) staged, and the accumulator of a new block read by the
        // epilogue of the block two before.  A look at a barrier takes some 200 clocks while the MMAs
        // read shared memory, which idled the tensor core between chunks: the first look at the next
        // chunk's barriers comes before the last taps of this one, and only a failed one waits.
        auto ready = [&](int g, int t, int c, int s, uint32_t ph, auto wait) {
            return !(c == 0 && t >= 2 && !wait(smem_addr(&acc_empty[t & 1]), (uint32_t)(((t >> 1) - 1) & 1))) &&
                   ((cf.resident && g > 0) || wait(smem_addr(&wfull[s]), ph)) && wait(smem_addr(&full[s]), ph);
        };
        auto look = [](uint32_t bar, uint32_t parity) { return mbar_try(bar, parity); };
        auto block = [&](uint32_t bar, uint32_t parity) { return wait_or_abort(bar, parity, abort_v); };
        bool ok = G == 0 || __all_sync(0xffffffffu, ready(0, 0, 0, 0, 0, block));
        for (int g = 0; g < G && ok; ++g) {
            tc_fence_after();
            const uint32_t ad = desc_lo(smem_addr(ring) + s * S::A_BYTES, S::PLANE);
            const uint32_t bd = desc_lo(wts + (cf.resident ? c : s) * S::B_BYTES, 0);
            const uint32_t acc = tmem + (uint32_t)((t & 1) * S::ACC);
            const uint32_t empty_bar = smem_addr(&empty[s]), acc_bar = smem_addr(&acc_full[t & 1]);
            const uint32_t first = (uint32_t)c;
            if (++s == stages) {
                s = 0;
                ph ^= 1u;
            }
            const bool block_done = ++c == nchunk;
            if (block_done) {
                c = 0;
                ++t;
            }
            bool next = false;
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int dy = tap / 3, dx = tap - dy * 3;
                if (tap == 6 && g + 1 < G) next = __all_sync(0xffffffffu, ready(g + 1, t, c, s, ph, look));
#pragma unroll
                for (int j = 0; j < MT; ++j) {
                    const uint32_t aoff = (uint32_t)(dy * S::HWD + 8 * j + dx);     // 16-byte pixels
                    const uint32_t d = acc + (uint32_t)(j * BN);
                    mma_bf16_ss_elect<S::A_HI, S::B_HI, S::IDESC>(d, ad + aoff, bd + tap * (S::B_TAP / 16),
                                                                  tap != 0 ? 1u : first);
                    if constexpr (LO)
                        mma_bf16_ss_elect<S::A_HI, S::B_HI, S::IDESC>(d, ad + S::A_HALF / 16 + aoff,
                                                                      bd + tap * (S::B_TAP / 16), 1u);
                }
            }
            mma_commit_elect(empty_bar);
            if (block_done) mma_commit_elect(acc_bar);
            last = g;
            if (!next && g + 1 < G) ok = __all_sync(0xffffffffu, ready(g + 1, t, c, s, ph, block));
        }
        // after an abort: wait (bounded) for the MMAs in flight before the memory is freed
        if (*abort_v && last >= 0) mbar_wait(smem_addr(&empty[last % stages]), (uint32_t)((last / stages) & 1));
        __syncwarp();
    } else if (warp == kWeightWarp && lane == 0 && G > 0) {
        // ---- weights: all chunks once, or chunk g as soon as buffer g % stages is free ----
        lbmt::prefetch_map(&wmap);
        if (cf.resident) {
            lbmt::mbar_arrive_expect_tx(smem_addr(&wfull[0]), (uint32_t)(nchunk * S::B_BYTES));
            for (int c = 0; c < nchunk; ++c)
                lbmt::tma_load_3d(wts + c * S::B_BYTES, &wmap, 16 * c, co0, 0, smem_addr(&wfull[0]));
            lbmt::mbar_drain(smem_addr(&wfull[0]), 0);
        } else {
            int g = 0;
            for (; g < G; ++g) {
                const int s = g % stages;
                if (g >= stages && !wait_or_abort(smem_addr(&empty[s]), (uint32_t)((g / stages - 1) & 1), abort_v)) break;
                lbmt::mbar_arrive_expect_tx(smem_addr(&wfull[s]), (uint32_t)S::B_BYTES);
                lbmt::tma_load_3d(wts + s * S::B_BYTES, &wmap, 16 * (g % nchunk), co0, 0, smem_addr(&wfull[s]));
            }
            // every copy issued has landed before the block leaves
            for (int q = g > stages ? g - stages : 0; q < g; ++q)
                lbmt::mbar_drain(smem_addr(&wfull[q % stages]), (uint32_t)((q / stages) & 1));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && *abort_v) atomicExch(&g_tc_timeout, 1);
    if (warp == kMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)S::COLS)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// 3x3 weight gradient, dW[co][dy][dx][ci] = sum over pixels of dY[p][co] X[p + (dy, dx) - 1][ci], on
// 16 x 16 pixel blocks.  A CTA takes CB output x 32 input channels, all nine taps and a range of blocks
// (gridDim.z ranges; partials summed in fixed order by the caller).
//
// Both operands have their channels contiguous and the pixels as the K index: the M / N-major layout
// without swizzle, 16-byte rows of 8 channels, 16 pixels of an image row per MMA.  A block's dY lies in
// shared memory as [row][8-channel plane][16 pixels], X with its halo as [row][plane][18 pixels], both
// with 288 bytes per plane, so that the planes of consecutive rows follow each other at one stride and
//   A = dY of 2 rows x CB channels (M = 2 CB),  B = X of the 4 halo rows around them x 32 channels (N = 128):
// block (i, j) of the product, dY row i against X row j, is the tap dy = j - i: six of the eight blocks
// are taps.  The tap dx is B started dx pixels further on, each with its own accumulator D_dx (128
// columns).  Per row pair and dx three MMAs: dY_hi X_hi + dY_hi X_lo + dY_lo X_hi.
//
// What bounds it: 72 MMAs of 64 clocks per block (M = 64 takes as long as 128): 33 us of the 50 us that
// 32 x 32 channels take at 8 x 256 x 256 (20 us of memory traffic; 43 us with one part per range).  The mma.sync kernel before, one warp
// per tap reading its fragments with ldmatrix, took 104 us there at half of mma.sync's rate (47 us);
// 384 -> 128 channels at 16 x 64 x 64, whole layer: 855 -> 377 us.
// Sixteen warps load, split into BF16 halves and stage a block while the MMAs of the one before run.
// ---------------------------------------------------------------------------
constexpr int kWgProducerWarps = 16;
constexpr int kWgEpilogueWarp0 = 16;     // four warps: accumulators -> partials
constexpr int kWgMmaWarp = 20;
constexpr int kWgThreads = 21 * 32;
constexpr int kWgProducers = kWgProducerWarps * 32;

template <int CB>
struct WgShape {
    static constexpr int PLANE = 288;                                   // bytes of 8 channels of a row
    static constexpr int Y_BYTES = 16 * (CB / 8) * PLANE;               // one BF16 half of dY
    static constexpr int X_BYTES = 18 * 4 * PLANE;                      // one BF16 half of X
    static constexpr int STAGE = 2 * (Y_BYTES + X_BYTES);
    static constexpr int SMEM = 2 * STAGE + 128;
    static constexpr int YQ = 256 * (CB / 8) / kWgProducers;            // 8-channel items per thread: dY
    static constexpr int XQ = (18 * 18 * 4 + kWgProducers - 1) / kWgProducers;   // and X
    static constexpr int M = 2 * CB;
    // both operands M / N-major (bits 15, 16)
    static constexpr uint32_t IDESC = idesc_bf16_f32(M, 128) | (1u << 15) | (1u << 16);
    static constexpr uint32_t HI = desc_hi(PLANE, kNoSwizzle);          // 8 channels further: one plane
    static_assert(256 * (CB / 8) % kWgProducers == 0, "dY items per thread");
};

template <int CB>
__global__ void __launch_bounds__(kWgThreads, 1) conv3_wgrad_tc_kernel(ConvTcWgradArgs a)
{
    using S = WgShape<CB>;
    extern __shared__ __align__(128) uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full[2], empty[2], acc_full, acc_empty;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    volatile int* abort_v = &abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Cin = a.C1 + a.C2;
    const int co0 = blockIdx.x * CB, ci0 = blockIdx.y * 32;
    const int lbx = 31 - __clz(a.W / 16), lby = 31 - __clz(a.H / 16);   // powers of two
    const int nblocks = a.B << (lbx + lby);
    // range z of gridDim.z, in a.subs parts of at least one block each: part u ends before block end(u)
    const int b0 = (int)((long long)nblocks * blockIdx.z / gridDim.z);
    const int G = (int)((long long)nblocks * (blockIdx.z + 1) / gridDim.z) - b0;
    auto end = [&](int u) { return (int)((long long)G * (u + 1) / a.subs); };
    uint8_t* const ring = smem_raw + ((0u - smem_addr(smem_raw)) & 127u);

    if (warp == kWgMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(&tmem_slot))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_addr(&full[i]), kWgProducerWarps);
            mbar_init(smem_addr(&empty[i]), 1);
        }
        mbar_init(smem_addr(&acc_full), 1);
        mbar_init(smem_addr(&acc_empty), 4);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp < kWgProducerWarps) {
        // input channels ci0 .. ci0 + 31 lie in x1 or in x2 (C1 is a multiple of 32)
        const bool from1 = ci0 < a.C1;
        const int half = (from1 && a.x1_half) ? 1 : 0;                  // nearest upsampling of a half-size x1
        const int xc = from1 ? a.C1 : a.C2;
        const float* const xs = (from1 ? a.x1 + ci0 : a.x2 + (ci0 - a.C1)) + (tid & 3) * 8;
        const float* const ys = a.dy + co0 + (tid & (CB / 8 - 1)) * 8;
        float4 vy[S::YQ][2], vx[S::XQ][2];
        auto load = [&](int b) {
            const int n = b >> (lbx + lby), ty0 = ((b >> lbx) & ((1 << lby) - 1)) * 16, tx0 = (b & ((1 << lbx) - 1)) * 16;
#pragma unroll
            for (int i = 0; i < S::YQ; ++i) {
                const int p = (tid + kWgProducers * i) / (CB / 8);
                const long long q = ((long long)n * a.H + ty0 + (p >> 4)) * a.W + tx0 + (p & 15);
                const float4* src = reinterpret_cast<const float4*>(ys + q * a.Cout);
                vy[i][0] = __ldg(src);
                vy[i][1] = __ldg(src + 1);
            }
#pragma unroll
            for (int i = 0; i < S::XQ; ++i) {
                const int hp = (tid + kWgProducers * i) >> 2;
                if (hp < 18 * 18) {
                    const int hy = hp / 18, hx = hp - hy * 18;
                    const int sy = (ty0 + hy - 1) & (a.H - 1), sx = (tx0 + hx - 1) & (a.W - 1);
                    const long long q = ((long long)n * (a.H >> half) + (sy >> half)) * (a.W >> half) + (sx >> half);
                    const float4* src = reinterpret_cast<const float4*>(xs + q * xc);
                    vx[i][0] = __ldg(src);
                    vx[i][1] = __ldg(src + 1);
                }
            }
        };
        auto put = [&](uint8_t* dst, int lo_off, const float4 (&u)[2]) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const __nv_bfloat162 h01 = __floats2bfloat162_rn(u[e].x, u[e].y), h23 = __floats2bfloat162_rn(u[e].z, u[e].w);
                const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
                hi[2 * e] = bf16x2_bits(h01);
                hi[2 * e + 1] = bf16x2_bits(h23);
                lo[2 * e] = bf16x2_bits(__floats2bfloat162_rn(u[e].x - f01.x, u[e].y - f01.y));
                lo[2 * e + 1] = bf16x2_bits(__floats2bfloat162_rn(u[e].z - f23.x, u[e].w - f23.y));
            }
            *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(dst + lo_off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        };
        load(b0);
        for (int g = 0; g < G; ++g) {
            const int s = g & 1;
            if (g >= 2 &&
                !__all_sync(0xffffffffu, wait_or_abort(smem_addr(&empty[s]), (uint32_t)(((g >> 1) - 1) & 1), abort_v)))
                break;
            uint8_t* const y = ring + s * S::STAGE;
            uint8_t* const x = y + 2 * S::Y_BYTES;
#pragma unroll
            for (int i = 0; i < S::YQ; ++i) {
                const int q = tid + kWgProducers * i, p = q / (CB / 8), c = q & (CB / 8 - 1);
                put(y + ((p >> 4) * (CB / 8) + c) * S::PLANE + (p & 15) * 16, S::Y_BYTES, vy[i]);
            }
#pragma unroll
            for (int i = 0; i < S::XQ; ++i) {
                const int q = tid + kWgProducers * i, hp = q >> 2;
                if (hp < 18 * 18) {
                    const int hy = hp / 18, hx = hp - hy * 18;
                    put(x + (hy * 4 + (q & 3)) * S::PLANE + hx * 16, S::X_BYTES, vx[i]);
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> tensor core
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&full[s]));
            if (g + 1 < G) load(b0 + g + 1);
        }
    } else if (warp < kWgMmaWarp) {
        // ---- accumulators -> partials: dY row i of the pairs is a partial of its own ----
        // M rows 32 w .. 32 w + 31 in this warp's 32 lanes (M = 128), or 16 w .. in its first 16
        constexpr int HALVES = CB / 32;
        const int w = warp - kWgEpilogueWarp0, gr = lane >> 2, t4 = lane & 3;
        for (int u = 0; u < a.subs; ++u) {
            if (!__all_sync(0xffffffffu, wait_or_abort(smem_addr(&acc_full), (uint32_t)(u & 1), abort_v))) break;
            tc_fence_after();
#pragma unroll 1
            for (int hh = 0; hh < HALVES; ++hh) {
                const int m = w * 16 * HALVES + 16 * hh, i = m / CB, co = co0 + m % CB;
                float* const out = a.partial + (2LL * (blockIdx.z * a.subs + u) + i) * a.Cout * 9 * Cin + ci0 + 2 * t4;
#pragma unroll 1
                for (int tap = 0; tap < 9; ++tap) {
                    const int dy = tap / 3, dx = tap - 3 * dy;
                    uint32_t v[16];
                    tmem_ld_16x32(tmem + ((uint32_t)(32 * w + 16 * hh) << 16) + 128 * dx + 32 * (i + dy), v);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            *reinterpret_cast<float2*>(out + ((long long)(co + gr + 8 * h) * 9 + tap) * Cin + 8 * k) =
                                make_float2(__uint_as_float(v[4 * k + 2 * h]), __uint_as_float(v[4 * k + 2 * h + 1]));
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&acc_empty));
        }
    } else {
        // ---- MMAs ----
        bool ok = true;
        int last = -1, u = 0, g0 = 0;                       // part and its first block
        for (int g = 0; g < G; ++g) {
            const int s = g & 1;
            ok = __all_sync(0xffffffffu, wait_or_abort(smem_addr(&full[s]), (uint32_t)((g >> 1) & 1), abort_v));
            if (ok && g == g0 && u > 0)                     // the epilogue has read the part before
                ok = __all_sync(0xffffffffu, wait_or_abort(smem_addr(&acc_empty), (uint32_t)((u - 1) & 1), abort_v));
            if (!ok) break;
            tc_fence_after();
            const uint32_t y = desc_lo(smem_addr(ring) + s * S::STAGE, 128);   // 8 pixels further: 128 bytes
            const uint32_t x = y + 2 * S::Y_BYTES / 16;
#pragma unroll
            for (int r = 0; r < 16; r += 2)
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    const uint32_t yr = y + r * (CB / 8) * (S::PLANE / 16), xr = x + r * 4 * (S::PLANE / 16) + dx;
                    const uint32_t d = tmem + 128 * dx;
                    mma_bf16_ss_elect<S::HI, S::HI, S::IDESC>(d, yr, xr, r > 0 ? 1u : (uint32_t)(g - g0));
                    mma_bf16_ss_elect<S::HI, S::HI, S::IDESC>(d, yr, xr + S::X_BYTES / 16, 1u);
                    mma_bf16_ss_elect<S::HI, S::HI, S::IDESC>(d, yr + S::Y_BYTES / 16, xr, 1u);
                }
            mma_commit_elect(smem_addr(&empty[s]));
            if (g + 1 == end(u)) {
                mma_commit_elect(smem_addr(&acc_full));
                ++u;
                g0 = g + 1;
            }
            last = g;
        }
        // after an abort: wait (bounded) for the MMAs in flight before the memory is freed
        if (!ok && last >= 0) mbar_wait(smem_addr(&empty[last & 1]), (uint32_t)((last >> 1) & 1));
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && *abort_v) atomicExch(&g_tc_timeout, 1);
    if (warp == kWgMmaWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

constexpr int kMaxDevices = 64;

struct VariantInfo {
    int ready;          // attributes set and read
    int regs_per_cta;   // registers allocated to one CTA (per-warp granularity of 256)
    int static_smem;
};
// filled on the first launch of a variant on a device; first launches racing from several host
// threads write the same values
VariantInfo g_var[kMaxDevices][12];
int g_sms[kMaxDevices], g_smem_sm[kMaxDevices], g_smem_reserved[kMaxDevices];

// CTAs that fit on one SM with `smem` bytes of dynamic shared memory: the limits of
// threads, registers and shared memory (carveout at its maximum, which the variant requests)
int ctas_per_sm(const VariantInfo& v, int dev, long long smem)
{
    int k = 2048 / kThreads;
    const int by_regs = 65536 / v.regs_per_cta;
    if (by_regs < k) k = by_regs;
    const long long by_smem = g_smem_sm[dev] / (smem + v.static_smem + g_smem_reserved[dev]);
    if (by_smem < k) k = (int)by_smem;
    return k;
}

template <int BN, int MT, bool LO>
bool launch_variant(const ConvTcArgs& a, cudaStream_t s, int stages, int slot)
{
    using S = TcShape<BN, MT, LO>;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    VariantInfo& v = g_var[dev][slot];
    if (!v.ready) {
        cudaFuncAttributes fa;
        if (cudaFuncSetAttribute(conv3_tc_kernel<BN, MT, LO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSmemLimit) != cudaSuccess ||
            cudaFuncSetAttribute(conv3_tc_kernel<BN, MT, LO>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, conv3_tc_kernel<BN, MT, LO>) != cudaSuccess ||
            cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&g_smem_sm[dev], cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
                cudaSuccess ||
            cudaDeviceGetAttribute(&g_smem_reserved[dev], cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
                cudaSuccess)
            return false;
        v.regs_per_cta = (kThreads / 32) * ((fa.numRegs * 32 + 255) / 256 * 256);
        v.static_smem = (int)fa.sharedSizeBytes;
        v.ready = 1;
    }
    const int nchunk = (a.C1 + a.C2) / 16;
    CUtensorMap wmap;
    if (!lbmh::encode_conv3_weights_map(&wmap, a.w, a.C1 + a.C2, a.Cout, BN)) return false;
    TcConf cf{stages > 0 ? stages : 3, 1};
    if (cf.stages < 2 || cf.stages > kMaxStages) return false;
    // largest configuration that fits: resident weights first, then fewer operand buffers
    long long smem = 0;
    for (;;) {
        const long long base = 256 + S::ring_bytes(cf.stages);       // 256: alignment
        const long long res = base + (long long)nchunk * S::B_BYTES;
        const long long str = base + (long long)cf.stages * S::B_BYTES;
        if (res <= kSmemLimit) { cf.resident = 1; smem = res; break; }
        if (str <= kSmemLimit) { cf.resident = 0; smem = str; break; }
        if (cf.stages > 2) --cf.stages;
        else return false;
    }
    const int per_sm = ctas_per_sm(v, dev, smem);
    // the CTAs resident on one SM must fit in its tensor memory together, so that no
    // allocation ever waits for another CTA
    if (per_sm < 1 || per_sm * S::COLS > kTmemColumns) return false;
    const long long ntiles = (long long)a.B * (a.H / S::TH) * (a.W / S::TW);
    const int cob = a.Cout / BN;
    long long gx = ((long long)per_sm * g_sms[dev] + cob - 1) / cob;
    if (gx > ntiles) gx = ntiles;
    if (gx < 1) gx = 1;
    conv3_tc_kernel<BN, MT, LO><<<dim3((unsigned)gx, (unsigned)cob), kThreads, (size_t)smem, s>>>(wmap, a, cf);
    return true;
}

template <int BN>
bool launch_bn(const ConvTcArgs& a, cudaStream_t s, int stages, int mt)
{
    const int base = (BN == 128 ? 8 : BN == 64 ? 4 : 0);
    if (mt == 2) return a.act_bf16 ? launch_variant<BN, 2, false>(a, s, stages, base + 0)
                                   : launch_variant<BN, 2, true>(a, s, stages, base + 1);
    return a.act_bf16 ? launch_variant<BN, 1, false>(a, s, stages, base + 2)
                      : launch_variant<BN, 1, true>(a, s, stages, base + 3);
}

template <int CB>
bool launch_wgrad(const ConvTcWgradArgs& a, int ranges, cudaStream_t s)
{
    static bool ready[kMaxDevices] = {};    // racing first launches set the same attribute
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
    if (!ready[dev]) {
        if (cudaFuncSetAttribute(conv3_wgrad_tc_kernel<CB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 WgShape<CB>::SMEM) != cudaSuccess)
            return false;
        ready[dev] = true;
    }
    const dim3 grid((unsigned)(a.Cout / CB), (unsigned)((a.C1 + a.C2) / 32), (unsigned)ranges);
    conv3_wgrad_tc_kernel<CB><<<grid, kWgThreads, WgShape<CB>::SMEM, s>>>(a);
    return true;
}

}  // namespace

bool conv3_tc_launch(const ConvTcArgs& a, cudaStream_t s, int stages)
{
    const auto aligned = [](const void* p) { return ((uintptr_t)p & 15) == 0; };
    if (a.H < 16 || a.W < 8 || a.C1 % 32 || a.C2 % 32 || a.Co1 % 16 || a.Cout % 32 || a.Co1 > a.Cout ||
        a.B <= 0 || (long long)a.B * a.H * a.W > (1LL << 31) - 1 || !aligned(a.x1) || !aligned(a.x2) ||
        !aligned(a.w) || !aligned(a.bias) || !aligned(a.y1) || !aligned(a.y2))
        return false;
    if (stages <= 0) stages = LBM_CONV_TC_STAGES;
    const int bn = a.Cout % 128 == 0 ? 128 : a.Cout % 64 == 0 ? 64 : 32;
#ifdef LBM_CONV_TC_MT
    const int mt = (LBM_CONV_TC_MT == 2 && a.W >= 16) ? 2 : 1;
#else
    // two 128-pixel tiles per CTA (one B operand for both) wherever the width allows
    const int mt = a.W >= 16 ? 2 : 1;
#endif
    if (bn == 128) return launch_bn<128>(a, s, stages, mt);
    if (bn == 64) return launch_bn<64>(a, s, stages, mt);
    return launch_bn<32>(a, s, stages, mt);
}

// One CTA per SM: ranges of blocks for 152 of them.  The tensor core's FP32 sums round towards zero, so
// their error grows with the number of MMAs in a row; a part of a range is at most twice the blocks that
// fill 4 x 152 CTAs of 32 x 32 channels (each of a pair's two rows has its own sums, 24 MMAs per block),
// the length that the kernel before had (relative error of a 32-channel layer's gradients at 8 x 256 x
// 256: 5.1e-6 then, 6.5e-6 with one part per range, 4.9e-6 so).
ConvTcWgradSplit conv3_wgrad_tc_split(int Cin, int Cout, int B, int H, int W)
{
    const long long nblocks = (long long)B * (H / 16) * (W / 16);
    const long long tiles32 = (long long)(Cout / 32) * (Cin / 32), tiles = Cout % 64 == 0 ? tiles32 / 2 : tiles32;
    const long long ranges = std::max(1LL, std::min(152 / tiles, nblocks));
    const long long splits = std::min((4 * 152 + tiles32 - 1) / tiles32, nblocks);
    const long long part = 2 * ((nblocks + splits - 1) / splits), per = (nblocks + ranges - 1) / ranges;
    return {(int)ranges, (int)((per + part - 1) / part)};
}

bool conv3_wgrad_tc_launch(ConvTcWgradArgs a, cudaStream_t s)
{
    const ConvTcWgradSplit sp = conv3_wgrad_tc_split(a.C1 + a.C2, a.Cout, a.B, a.H, a.W);
    a.subs = sp.parts;
    return a.Cout % 64 == 0 ? launch_wgrad<64>(a, sp.ranges, s) : launch_wgrad<32>(a, sp.ranges, s);
}

bool conv3_tc_take_timeout(cudaStream_t s)
{
    int v = 0, zero = 0;
    if (cudaMemcpyFromSymbolAsync(&v, g_tc_timeout, sizeof(int), 0, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return false;
    if (cudaStreamSynchronize(s) != cudaSuccess) return false;
    if (v) {
        cudaMemcpyToSymbolAsync(g_tc_timeout, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s);
        cudaStreamSynchronize(s);
    }
    return v != 0;
}
