// Several time steps per pass for the population formats stored in FP32 / BF16 / FP16 (FP32
// arithmetic), periodic or homogeneous-Dirichlet lattices without body load, omega = 2: two
// adjacent columns per thread in packed FP32 arithmetic (fma.rn.f32x2 / add.rn.f32x2).  Every
// packed operation rounds each half as the scalar one does and the operations are those of
// collide() (lbm_kernels.cuh) up to exact sign changes, so FP32 results equal single steps.
// (Packed products that are added are merged into one packed multiply-add; the update has none.)
//
// Block = NW compute warps + 1 producer warp over a tile of OUT = NW OUTW output columns and `rows`
// output rows (TbpGeom: a warp's 64 columns are OUTW = 64 - 2 LEAD stored ones and LEAD on each side
// that feed them; 56 and 4 in FP32, 60 and 2 in the 16-bit formats' single lattices).  The producer's
// elected lane streams the input rows y0 - NL .. y1 + NL - 1 of
// all 20 planes, columns [X0 - HL, X0 + OUT + HL), into a ring of shared-memory stages, one
// tensor copy per row (lbm_tma.cuh).  A lane of warp w owns the columns X0 - LEAD + OUTW w + 2 lane
// and the next one.  Level 1, S1 = f*(t+dt) of row r, is pulled from the staged rows r-1, r,
// r+1; level l + 1 of row r - l is pulled from level l's rows r-l-1 .. r-l+1, which stay in
// registers (x-neighbours: one shuffle per component and direction for both columns); level NL
// of row r - NL + 1 is stored by lanes LEAD / 2 .. 31 - LEAD / 2.  Per level and node only what later rows still
// read is kept: the shifted (1,0) and (-1,0) populations of the last row and the (0,1)
// populations of the last two.
//
// What bounds it: instruction issue before, memory and latency now (FP32: DRAM 74 % busy, 40 % of the
// issue slots, two warps per scheduler; BF16: 61 %, 56 %).  One column per thread took 164 thread
// instructions per node and step in the three-step kernel it replaces (scalar arithmetic, a shuffle
// per component and column, register copies of the kept rows); here it is 97 in FP32 and 106 in BF16,
// the columns and rows around a tile included.
// Measured at 8192^2 periodic: FP32 110k -> 154k MLUPS at four steps per pass (three: 117k, bound by
// HBM at 53 B per node and step; five spill), 0.91 of the copy bandwidth at 40 B; BF16 158k -> 215k at
// three, 0.85 of it at 26.7 B.  FP32: 3 compute warps, 2 blocks per SM, 232 registers (168 spill: 17k);
// 16-bit: 4 warps, 2 blocks, 168 registers, ring of 5 (8 stages: 157k -> 150k at 2048^2).
//
// Signs: with f given, o = U/2 + (Phi - f) needs -f as an addend, which packed operations have
// no modifier for.  Odd levels therefore compute n = -o for the directions (1,0) and (0,1) (all
// their constants negated: the exact negative of every intermediate), and even levels, reading
// n, compute o again; stores after an odd number of levels negate back.
//
// Edges: the blocks that touch x = 0 or x = nx - 1 (on a Dirichlet lattice also those that touch
// row 0 or ny - 1) run the EDGE instantiation of the body; the others hold no edge code.
// Periodic lattices wider than a tile stage the wrapped columns too (two more tensor copies per
// row, 32 bytes of columns each, from the other end of the row), narrower ones hold every
// column in the tile; each lane then reads each of its columns through its own address and
// plane stride.  Dirichlet lattices overwrite the missing links.  Rows
// outside a Dirichlet lattice are not loaded: what level l computes for them is replaced by the
// wall reflection before a row of the lattice reads it.
#pragma once

#include "lbm_kernels.cuh"
#include "lbm_tma.cuh"

namespace lbmk {

// r modulo ny in [0, ny) for r within four rows of the lattice (the rows staged for up to four
// steps): one wrap suffices unless ny is 2 or 3, where the remainder is taken
__device__ __forceinline__ int wrap_row(int r, int ny)
{
    if (r < 0) r += ny;
    else if (r >= ny) r -= ny;
    if ((unsigned)r >= (unsigned)ny) {
        const int q = r % ny;
        r = q < 0 ? q + ny : q;
    }
    return r;
}

typedef unsigned long long f32x2;       // two FP32 values, the lower column in the low half

__device__ __forceinline__ f32x2 pk(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk(f32x2 v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ float lo_of(f32x2 v)
{
    float a, b;
    upk(v, a, b);
    return a;
}
__device__ __forceinline__ float hi_of(f32x2 v)
{
    float a, b;
    upk(v, a, b);
    return b;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// both halves' signs (exact)
__device__ __forceinline__ f32x2 neg2(f32x2 v) { return v ^ 0x8000000080000000ull; }

// two adjacent stored elements <-> a pair
template <int K> struct Pair;
template <> struct Pair<K_F32> {
    static __device__ __forceinline__ f32x2 lds(uint32_t a)
    {
        f32x2 v;
        asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
        return v;
    }
    template <bool NEG> static __device__ __forceinline__ void st(float* p, f32x2 v)
    {
        *reinterpret_cast<f32x2*>(p) = NEG ? neg2(v) : v;
    }
};
template <int K> struct Pair16 {
    static __device__ __forceinline__ f32x2 lds(uint32_t a)
    {
        uint32_t w;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w) : "r"(a) : "memory");
        return pk(Fmt<K>::ld((unsigned short)(w & 0xFFFFu)), Fmt<K>::ld((unsigned short)(w >> 16)));
    }
    template <bool NEG> static __device__ __forceinline__ void st(unsigned short* p, f32x2 v)
    {
        float a, b;
        upk(v, a, b);
        if (NEG) {
            a = -a;
            b = -b;
        }
        *reinterpret_cast<uint32_t*>(p) = (uint32_t)Fmt<K>::st(a) | ((uint32_t)Fmt<K>::st(b) << 16);
    }
};
template <> struct Pair<K_BF16> : Pair16<K_BF16> {
    template <bool NEG> static __device__ __forceinline__ void st(unsigned short* p, f32x2 v)
    {
        float a, b;
        upk(v, a, b);
        const __nv_bfloat162 h = NEG ? __floats2bfloat162_rn(-a, -b) : __floats2bfloat162_rn(a, b);
        *reinterpret_cast<__nv_bfloat162*>(p) = h;
    }
};
template <> struct Pair<K_F16> : Pair16<K_F16> {
    template <bool NEG> static __device__ __forceinline__ void st(unsigned short* p, f32x2 v)
    {
        float a, b;
        upk(v, a, b);
        const __half2 h = NEG ? __floats2half2_rn(-a, -b) : __floats2half2_rn(a, b);
        *reinterpret_cast<__half2*>(p) = h;
    }
};

// constants of the update, duplicated in both halves
struct TbpConst {
    f32x2 a, na, b, nb, h, nh, m1;      // a = cK/c, b = cmu/c, 1/2, -1
    __device__ __forceinline__ TbpConst(float fa, float fb)
        : a(pk(fa, fa)), na(pk(-fa, -fa)), b(pk(fb, fb)), nb(pk(-fb, -fb)), h(pk(.5f, .5f)), nh(pk(-.5f, -.5f)),
          m1(pk(-1.f, -1.f))
    {
    }
};

// node update of two columns.  NEG = false: x0 .. x3 are the pulled populations of (1,0), (0,1),
// (-1,0), (0,-1); o[0], o[1] are returned negated.  NEG = true: x0, x1 come negated; o[0], o[1]
// are returned as they are.  Operation for operation collide() of lbm_kernels.cuh.
template <bool NEG>
__device__ __forceinline__ void tbp_update(const TbpConst& C, const f32x2 (&x0)[5], const f32x2 (&x1)[5],
                                           const f32x2 (&x2)[5], const f32x2 (&x3)[5], f32x2 (&o)[4][5])
{
    f32x2 rx[5], ry[5], U[5], t0[5], t1[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        rx[k] = NEG ? fma2(C.m1, x1[k], x3[k]) : add2(x1[k], x3[k]);
        ry[k] = NEG ? fma2(C.m1, x0[k], x2[k]) : add2(x0[k], x2[k]);
        U[k] = add2(rx[k], ry[k]);
    }
    const f32x2 a = NEG ? C.a : C.na, b = NEG ? C.b : C.nb, mb = NEG ? C.nb : C.b, h = NEG ? C.h : C.nh;
    t0[0] = fma2(a, U[2], fma2(b, U[3], x0[0]));
    t0[1] = fma2(b, U[4], x0[1]);
    t0[2] = fma2(a, U[0], x0[2]);
    t0[3] = fma2(b, U[0], x0[3]);
    t0[4] = fma2(b, U[1], x0[4]);
    t1[0] = fma2(b, U[4], x1[0]);
    t1[1] = fma2(a, U[2], fma2(mb, U[3], x1[1]));
    t1[2] = fma2(a, U[1], x1[2]);
    t1[3] = fma2(mb, U[1], x1[3]);
    t1[4] = fma2(b, U[0], x1[4]);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        o[0][k] = fma2(h, U[k], t0[k]);
        o[1][k] = fma2(h, U[k], t1[k]);
        o[2][k] = NEG ? fma2(C.m1, o[0][k], rx[k]) : add2(rx[k], o[0][k]);
        o[3][k] = NEG ? fma2(C.m1, o[1][k], ry[k]) : add2(ry[k], o[1][k]);
    }
}

struct TbpArgs {
    void* dst;             // f*(t + NL dt) planes; f*(t) is read through the row maps
    int nx, ny, pitch;
    long long plane;
    float af, bf;          // cK/c, cmu/c in FP32
    int rows;              // output rows per block
    int* timeout;          // device flag: set when a bounded wait ran out
    int withhold;          // test hook: staged input row the producer never copies (-1: none)
};

#ifndef LBM_TBP_NL4
#define LBM_TBP_NL4 4                   // steps per pass of the FP32 format
#endif
// compute warps per block, stages of the row ring, resident blocks per SM (registers: 65536 /
// (threads x blocks))
#ifndef LBM_TBP_NW4
#define LBM_TBP_NW4 3
#endif
#ifndef LBM_TBP_NW2
#define LBM_TBP_NW2 4
#endif
#ifndef LBM_TBP_LEAD4
#define LBM_TBP_LEAD4 4
#endif
#ifndef LBM_TBP_LEAD2
#define LBM_TBP_LEAD2 2
#endif
#ifndef LBM_TBP_NST4
#define LBM_TBP_NST4 7
#endif
#ifndef LBM_TBP_NST2
#define LBM_TBP_NST2 5
#endif
#ifndef LBM_TBP_MIN4
#define LBM_TBP_MIN4 2
#endif
#ifndef LBM_TBP_MIN2
#define LBM_TBP_MIN2 2
#endif

// BATCH: the 16-bit formats take FP32's tile there.  Most tiles of a batch of small lattices touch an
// edge, and the Dirichlet edge code spills 180 bytes at the 168 registers of five warps (two blocks put
// three warps on a scheduler); at four warps it has 203 and none.  48 steps, before this tile
// and with it: 64 Dirichlet lattices of 256 x 512 in BF16 5069 -> 3639 us, periodic ones 3791 -> 3032.
// Single lattices keep the wider tile: 8192^2 periodic 312 us a step against 371.
template <int ES, bool BATCH = false>
struct TbpGeom {
    static constexpr bool TALL = ES == 4 || BATCH;
    static constexpr int NLMAX = (ES == 4) ? LBM_TBP_NL4 : 3;          // steps per pass at most
    static constexpr int NW = TALL ? LBM_TBP_NW4 : LBM_TBP_NW2;
    static constexpr int MIN_BLOCKS = TALL ? LBM_TBP_MIN4 : LBM_TBP_MIN2;
    static constexpr int LEAD = TALL ? LBM_TBP_LEAD4 : LBM_TBP_LEAD2;        // columns a warp computes left and right of
                                                                       // its output (even, at least NLMAX - 1)
    static constexpr int OUTW = 64 - 2 * LEAD;                         // output columns per warp
    static constexpr int OUT = NW * OUTW;
    static constexpr int THREADS = 32 * (NW + 1);
    static constexpr int HL = (LEAD + 1) * ES > 16 ? 32 / ES : 16 / ES;   // staged columns left and right of the tile
    static constexpr int WIN = HL + OUT + HL;
    static constexpr int WRAP = 32 / ES;                               // columns of a wrap copy
    static constexpr int ROW_BYTES = 20 * WIN * ES;
    static constexpr int WRAP_BYTES = 20 * WRAP * ES;                  // 640
    static constexpr int LOFF = (ROW_BYTES + 127) / 128 * 128;         // columns wrapped below x = 0
    static constexpr int ROFF = LOFF + WRAP_BYTES;                     // columns wrapped beyond x = nx - 1
    static constexpr int STAGE_BYTES = ROFF + WRAP_BYTES;
    static constexpr int NST = TALL ? LBM_TBP_NST4 : LBM_TBP_NST2;
    static constexpr int SMEM = NST * STAGE_BYTES + 128;
    static_assert(LEAD % 2 == 0 && LEAD >= NLMAX - 1, "columns lost per level");
    static_assert((WIN * ES) % 16 == 0 && WIN <= 256, "staged row geometry");
    static_assert((OUT * ES) % 16 == 0, "a tensor copy starts on a 16-byte boundary");
    static_assert(WRAP_BYTES % 128 == 0 && STAGE_BYTES % 128 == 0, "copies land on 128-byte boundaries");
};

// Rows per block.  A block of r rows computes r + 2 (NL - 1) rows of level 1 and stages r + 2 NL,
// and the last wave of blocks leaves part of the chip idle.  Measured over rows 2..64 on lattices
// from 256^2 to 4096^2 (FP32, four steps per pass; also the 16-bit formats), the time of a pass
// follows (W + 0.6 (ceil W - W)) (r + 4.4), W the waves of resident blocks, within a tenth; the
// rule takes the r up to 96 that makes it smallest.  With the fixed 12 (FP32) and 64 (16-bit) rows
// before, a BF16 lattice of 256^2 ran in 8 blocks.  `blocks(r)`: blocks of a pass at r rows.
template <typename Blocks>
inline int tbp_rows(long long resident, int ny, Blocks blocks)
{
    int best = 1;
    double cost = 1e300;
    for (int r = 2; r <= 96; ++r) {
        const double w = (double)blocks(r) / (double)resident, up = (double)(long long)(w + 0.999999);
        const double c = (w + 0.6 * ((up > w ? up : w) - w)) * (r + 4.4);
        if (c < cost) {
            cost = c;
            best = r;
        }
        if (r >= ny) break;
    }
    return best;
}

// Sizes of `count` passes that make n steps, as equal as they can be: pass i of plan(n, count)
inline int tbp_pass(long long n, long long count, long long i)
{
    const long long q = n / count;
    return (int)(q + (i < n - q * count ? 1 : 0));
}

// first column of the copy that holds the columns nx - LEAD - 1 .. nx - 1
template <typename G>
__device__ __forceinline__ int tbp_wrap_x(int nx) { return (nx - G::LEAD - 1) & ~(G::WRAP / 2 - 1); }

// the compute warps' part of a block.  EDGE: the tile touches x = 0 or x = nx - 1.
template <typename G, int K, int NL, bool DIRICHLET, bool EDGE>
__device__ __forceinline__ void tbp_compute(const TbpArgs& A, int X0, int y0, int y1, uint32_t sbase,
                                            unsigned long long* full_bar, unsigned long long* empty_bar,
                                            volatile int* abort_flag)
{
    using E = typename Fmt<K>::E;
    constexpr int NST = G::NST, WIN = G::WIN, HL = G::HL;
    constexpr uint32_t ES = sizeof(E), PL = WIN * sizeof(E);
    constexpr bool NEGOUT = (NL & 1) != 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nx = A.nx, ny = A.ny;
    const int nin = (y1 - y0) + 2 * NL;
    const int xs = X0 - G::LEAD + G::OUTW * warp + 2 * lane;   // this lane's lower column (even)
    const bool out_lane = lane >= G::LEAD / 2 && lane < 32 - G::LEAD / 2 && xs < nx;
    const bool both = xs + 1 < nx;
    const uint32_t own = (uint32_t)(xs - X0 + HL) * ES;
    const TbpConst C(A.af, A.bf);

    // EDGE, periodic: where the columns xs - 1 .. xs + 2 sit in a stage, and their plane strides
    uint32_t eo[4], es[4];
    if (EDGE && !DIRICHLET) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int c = (xs - 1 + q) % nx;
            c = c < 0 ? c + nx : c;
            const int m = c - X0 + HL, xl = tbp_wrap_x<G>(nx);
            if (m >= 0 && m < WIN) {
                eo[q] = m * ES;
                es[q] = PL;
            } else if (c >= xl && c < xl + G::WRAP) {
                eo[q] = G::LOFF + (c - xl) * ES;
                es[q] = G::WRAP * ES;
            } else {
                eo[q] = G::ROFF + (c < G::WRAP ? c : 0) * ES;     // others feed no stored column
                es[q] = G::WRAP * ES;
            }
        }
    }
    const bool wl = EDGE && DIRICHLET && xs == 0;                        // lower column on the left wall
    const bool wr0 = EDGE && DIRICHLET && xs == nx - 1, wr1 = EDGE && DIRICHLET && xs + 1 == nx - 1;

    // where this lane's pulled (1,0) population of the lower column and its two (-1,0) ones sit in the
    // staged row, from its own column on; on a Dirichlet wall, with BYADDR, the node's own opposite
    // populations (a missing link is D f* of the opposite direction, D = (-1, -1, 1, 1, 1)).  In the
    // 16-bit formats that saves the second loads (BF16 Dirichlet, us a step: 2048^2 33.4 -> 31.1, 2500 x
    // 5000 93 -> 80, 8192^2 334 -> 316); in FP32 the offsets spill at four steps (4095 x 4001: 114 -> 120).
    constexpr bool BYADDR = EDGE && DIRICHLET && ES == 2;
    const uint32_t wo0 = BYADDR && wl ? 10 * PL : 0u - ES, wo2 = BYADDR && wr0 ? 0u : 10 * PL + ES;
    const uint32_t wo3 = BYADDR && wr1 ? ES : 10 * PL + 2 * ES;

    // level l + 1 reads: s0 / s2 the pulled (1,0) / (-1,0) populations of its row, k1 the (0,1)
    // populations of the row below, c1 those of its own row (the next row's k1)
    f32x2 s0[NL - 1][5], s2[NL - 1][5], k1[NL - 1][5], c1[NL - 1][5];
#pragma unroll
    for (int l = 0; l < NL - 1; ++l)
#pragma unroll
        for (int k = 0; k < 5; ++k) s0[l][k] = s2[l][k] = k1[l][k] = c1[l][k] = 0ull;

    auto wait = [&](int j) {
        return lbmt::mbar_wait(lbmt::smem_u32(&full_bar[j % NST]), (j / NST) & 1, abort_flag);
    };
    bool ok = wait(0) && wait(1);
    uint32_t st_m = sbase, st_c = sbase + (1 % NST) * G::STAGE_BYTES;
    int sp = 2 % NST, ph = (2 / NST) & 1, se = 0;          // stage and phase of row i + 2, stage of row i
    E* __restrict__ dst = static_cast<E*>(A.dst);
    for (int i = 0; i + 2 < nin; ++i) {
        const int r = y0 - (NL - 1) + i;                   // level 1's row, from staged rows i, i+1, i+2
        ok = ok && lbmt::mbar_wait(lbmt::smem_u32(&full_bar[sp]), ph, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) break;
        const uint32_t st_p = sbase + sp * G::STAGE_BYTES;
        f32x2 cur[4][5];
        {
            f32x2 x0[5], x1[5], x2[5], x3[5];
            if (EDGE && !DIRICHLET) {
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    x0[k] = pk(Fmt<K>::ld(lbmt::lds<E>(st_c + eo[0] + k * es[0])),
                               Fmt<K>::ld(lbmt::lds<E>(st_c + eo[1] + k * es[1])));
                    x2[k] = pk(Fmt<K>::ld(lbmt::lds<E>(st_c + eo[2] + (10 + k) * es[2])),
                               Fmt<K>::ld(lbmt::lds<E>(st_c + eo[3] + (10 + k) * es[3])));
                    x1[k] = pk(Fmt<K>::ld(lbmt::lds<E>(st_m + eo[1] + (5 + k) * es[1])),
                               Fmt<K>::ld(lbmt::lds<E>(st_m + eo[2] + (5 + k) * es[2])));
                    x3[k] = pk(Fmt<K>::ld(lbmt::lds<E>(st_p + eo[1] + (15 + k) * es[1])),
                               Fmt<K>::ld(lbmt::lds<E>(st_p + eo[2] + (15 + k) * es[2])));
                }
            } else {
                const uint32_t c = st_c + own;
                uint32_t a1 = st_m + own + 5 * PL, a3 = st_p + own + 15 * PL;
                if (BYADDR && r == 0) a1 = c + 15 * PL;
                if (BYADDR && r == ny - 1) a3 = c + 5 * PL;
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    float l0 = Fmt<K>::ld(lbmt::lds<E>(c + wo0 + k * PL)), l2 = Fmt<K>::ld(lbmt::lds<E>(c + wo2 + k * PL));
                    float h2 = Fmt<K>::ld(lbmt::lds<E>(c + wo3 + k * PL));
                    x1[k] = Pair<K>::lds(a1 + k * PL);
                    x3[k] = Pair<K>::lds(a3 + k * PL);
                    if (BYADDR && k < 2) {
                        if (wl) l0 = -l0;
                        if (wr0) l2 = -l2;
                        if (wr1) h2 = -h2;
                        if (r == 0) x1[k] = neg2(x1[k]);
                        if (r == ny - 1) x3[k] = neg2(x3[k]);
                    }
                    x0[k] = pk(l0, Fmt<K>::ld(lbmt::lds<E>(c + k * PL)));
                    x2[k] = pk(l2, h2);
                }
                if (EDGE && DIRICHLET && !BYADDR) {
                    // missing links: D f* of the opposite direction at the node, D = (-1, -1, 1, 1, 1)
#pragma unroll
                    for (int k = 0; k < 5; ++k) {
                        const float Dk = k < 2 ? -1.f : 1.f;
                        if (wl) x0[k] = pk(Dk * Fmt<K>::ld(lbmt::lds<E>(c + (10 + k) * PL)), hi_of(x0[k]));
                        if (wr0) x2[k] = pk(Dk * Fmt<K>::ld(lbmt::lds<E>(c + k * PL)), hi_of(x2[k]));
                        if (wr1) x2[k] = pk(lo_of(x2[k]), Dk * Fmt<K>::ld(lbmt::lds<E>(c + k * PL + ES)));
                    }
                    if (r == 0) {
#pragma unroll
                        for (int k = 0; k < 5; ++k) {
                            const f32x2 v = Pair<K>::lds(c + (15 + k) * PL);
                            x1[k] = k < 2 ? neg2(v) : v;
                        }
                    }
                    if (r == ny - 1) {
#pragma unroll
                        for (int k = 0; k < 5; ++k) {
                            const f32x2 v = Pair<K>::lds(c + (5 + k) * PL);
                            x3[k] = k < 2 ? neg2(v) : v;
                        }
                    }
                }
            }
            tbp_update<false>(C, x0, x1, x2, x3, cur);
        }
        // staged row i (row r - 1) is not read again
        __syncwarp();
        if (lane == 0) lbmt::mbar_arrive(lbmt::smem_u32(&empty_bar[se]));
        st_m = st_c;
        st_c = st_p;
        se = se + 1 == NST ? 0 : se + 1;
        if (++sp == NST) {
            sp = 0;
            ph ^= 1;
        }
        // level l + 1 of row r - l from level l; cur holds level l's row r - l + 1
#pragma unroll
        for (int l = 1; l < NL; ++l) {
            const int q = r - l;
            const int s = l - 1;
            const bool neg = (l & 1) != 0;                 // cur[0], cur[1], s0, k1, c1 hold -f
            f32x2 out[4][5];
            {
                f32x2 x3[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) x3[k] = cur[3][k];
                if (EDGE && DIRICHLET && q == ny - 1)
#pragma unroll
                    for (int k = 0; k < 5; ++k) x3[k] = ((k < 2) != neg) ? neg2(c1[s][k]) : c1[s][k];
                if (neg) tbp_update<true>(C, s0[s], k1[s], s2[s], x3, out);
                else tbp_update<false>(C, s0[s], k1[s], s2[s], x3, out);
            }
            // level l's row r - l + 1 becomes the last one
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const float up = __shfl_up_sync(0xffffffffu, hi_of(cur[0][k]), 1);
                const float dn = __shfl_down_sync(0xffffffffu, lo_of(cur[2][k]), 1);
                s0[s][k] = pk(up, lo_of(cur[0][k]));
                s2[s][k] = pk(hi_of(cur[2][k]), dn);
                if (EDGE && DIRICHLET) {
                    const float Dk = ((k < 2) != neg) ? -1.f : 1.f;
                    if (wl) s0[s][k] = pk(Dk * lo_of(cur[2][k]), lo_of(cur[0][k]));
                    if (wr0) s2[s][k] = pk(Dk * lo_of(cur[0][k]), dn);
                    if (wr1) s2[s][k] = pk(hi_of(cur[2][k]), Dk * hi_of(cur[0][k]));
                }
                k1[s][k] = c1[s][k];
                c1[s][k] = cur[1][k];
            }
            if (EDGE && DIRICHLET && q + 1 == 0)             // the wall below row 0
#pragma unroll
                for (int k = 0; k < 5; ++k) k1[s][k] = ((k < 2) != neg) ? neg2(cur[3][k]) : cur[3][k];
#pragma unroll
            for (int d = 0; d < 4; ++d)
#pragma unroll
                for (int k = 0; k < 5; ++k) cur[d][k] = out[d][k];
        }
        const int q = r - (NL - 1);
        if (q >= y0 && out_lane) {
            E* p = dst + (long long)q * A.pitch + xs;
            if (both) {
#pragma unroll
                for (int d = 0; d < 4; ++d)
#pragma unroll
                    for (int k = 0; k < 5; ++k) {
                        if (NEGOUT && d < 2) Pair<K>::template st<true>(p + (d * 5 + k) * A.plane, cur[d][k]);
                        else Pair<K>::template st<false>(p + (d * 5 + k) * A.plane, cur[d][k]);
                    }
            } else {                                       // odd nx: the last column alone
#pragma unroll
                for (int d = 0; d < 4; ++d)
#pragma unroll
                    for (int k = 0; k < 5; ++k)
                        p[(d * 5 + k) * A.plane] =
                            Fmt<K>::st(NEGOUT && d < 2 ? -lo_of(cur[d][k]) : lo_of(cur[d][k]));
            }
        }
    }
    if (lane == 0 && *abort_flag) atomicExch(A.timeout, 1);
}

// One block's work: output columns X0 .. and rows y0 .. of the lattice A describes; maps[0]: its
// row map (box WIN), maps[1]: the wrap map (box WRAP), as kernel parameters or in global memory.
template <typename G, int K, int NL, bool DIRICHLET>
__device__ __forceinline__ void tbp_body(const CUtensorMap* map, const CUtensorMap* wmap, const TbpArgs& A, int X0,
                                         int y0)
{
    constexpr int NST = G::NST;
    extern __shared__ __align__(128) unsigned char tbp_smem_raw[];
    __shared__ __align__(8) unsigned long long full_bar[NST], empty_bar[NST];
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nx = A.nx, ny = A.ny;
    const int y1 = min(ny, y0 + A.rows);
    const int nin = (y1 - y0) + 2 * NL;              // staged input rows y0 - NL .. y1 + NL - 1
    const int nact = min(G::NW, (nx - X0 + G::OUTW - 1) / G::OUTW);   // warps with output columns
    const bool edge = X0 == 0 || X0 + G::OUT + G::LEAD + 1 >= nx ||
                      (DIRICHLET && (y0 < NL || y1 + NL - 1 >= ny));
    const uint32_t sbase = (lbmt::smem_u32(tbp_smem_raw) + 127u) & ~127u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            lbmt::mbar_init(lbmt::smem_u32(&full_bar[s]), 1);
            lbmt::mbar_init(lbmt::smem_u32(&empty_bar[s]), nact);
        }
        abort_flag = 0;
        lbmt::fence_mbar_init();
    }
    __syncthreads();

    if (warp == G::NW) {
        if (lane == 0) {
            lbmt::prefetch_map(map);
            const bool wrap = !DIRICHLET && edge && nx > G::OUT;   // columns beyond the row's ends, copied apart
            const uint32_t bytes = G::ROW_BYTES + (wrap ? 2 * G::WRAP_BYTES : 0);
            const int xl = tbp_wrap_x<G>(nx);
            lbmt::grid_dependency_wait();
            int j = 0, s = 0, ph = 1;
            for (; j < nin; ++j) {
                const uint32_t fb = lbmt::smem_u32(&full_bar[s]);
                bool go = j != A.withhold;                         // test hook: this row never arrives
                if (go && j >= NST) go = lbmt::mbar_wait(lbmt::smem_u32(&empty_bar[s]), ph, &abort_flag);
                if (!go && j != A.withhold) break;
                if (go) {
                    int y = y0 - NL + j;
                    if (DIRICHLET && (y < 0 || y >= ny)) {
                        lbmt::mbar_arrive(fb);                     // row outside the lattice
                    } else {
                        if (!DIRICHLET) y = wrap_row(y, ny);
                        const uint32_t st = sbase + s * G::STAGE_BYTES;
                        lbmt::mbar_arrive_expect_tx(fb, bytes);
                        lbmt::tma_load_3d(st, map, X0 - G::HL, y, 0, fb);
                        if (wrap) {
                            lbmt::tma_load_3d(st + G::LOFF, wmap, xl, y, 0, fb);
                            lbmt::tma_load_3d(st + G::ROFF, wmap, 0, y, 0, fb);
                        }
                    }
                }
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
            // every copy issued has landed before the block leaves
            for (int q = (j > NST ? j - NST : 0); q < j; ++q)
                if (q != A.withhold) lbmt::mbar_drain(lbmt::smem_u32(&full_bar[q % NST]), (q / NST) & 1);
            if (abort_flag) atomicExch(A.timeout, 1);
        }
        return;
    }
    if (warp >= nact) return;
    // the previous launch's last blocks may still read what this one overwrites
    lbmt::grid_dependency_wait();
    if (edge) tbp_compute<G, K, NL, DIRICHLET, true>(A, X0, y0, y1, sbase, full_bar, empty_bar, &abort_flag);
    else tbp_compute<G, K, NL, DIRICHLET, false>(A, X0, y0, y1, sbase, full_bar, empty_bar, &abort_flag);
}

template <int K, int NL, bool DIRICHLET>
__global__ void __launch_bounds__(TbpGeom<(int)sizeof(typename Fmt<K>::E)>::THREADS,
                                  TbpGeom<(int)sizeof(typename Fmt<K>::E)>::MIN_BLOCKS)
    tbp_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap wmap, TbpArgs A)
{
    using G = TbpGeom<(int)sizeof(typename Fmt<K>::E)>;
    tbp_body<G, K, NL, DIRICHLET>(&map, &wmap, A, blockIdx.x * G::OUT, blockIdx.y * A.rows);
}

// ---------------------------------------------------------------------------
// Batches of lattices, several steps per pass (lbm_batch.cu, mode 2): one block per tile
// {lattice, X0, y0, Dirichlet} of a flat list, each running tbp_body on its lattice with that
// lattice's row and wrap maps of the source arena.  Periodic and Dirichlet tiles share the launch: a
// launch for each, one behind the other, left half the chip idle where either kind fills it less than
// once (128 lattices of 64^2 in FP32, 48 steps: 941 us, 556 so).  The maps live in global memory, written by the host before
// the launch; a lattice's planes sit at its element offset in each arena.
// ---------------------------------------------------------------------------
struct BatchLatT3 {
    long long off;         // element offset of plane 0 in each arena
    long long plane;       // elements per plane = ny * pitch
    int nx, ny, pitch;
    float af, bf;          // cK / c, cmu / c in FP32
};

struct BatchTbpArgs {
    const int4* tiles;          // {lattice, X0, y0, 1 if Dirichlet} per block
    const BatchLatT3* lat;
    const CUtensorMap* maps;    // [lattice][arena][2]: row map, wrap map
    void* arenaA;
    void* arenaB;
    int parity;                 // 0: read arena A, write arena B
    int rows;                   // output rows per tile
    int* timeout;               // set when a bounded wait ran out
};

template <int K, int NL>
__global__ void __launch_bounds__(TbpGeom<(int)sizeof(typename Fmt<K>::E), true>::THREADS,
                                  TbpGeom<(int)sizeof(typename Fmt<K>::E), true>::MIN_BLOCKS)
    batch_tbp_kernel(BatchTbpArgs B)
{
    using E = typename Fmt<K>::E;
    const int4 t = B.tiles[blockIdx.x];
    const BatchLatT3 L = B.lat[t.x];
    E* a = static_cast<E*>(B.arenaA) + L.off;
    E* b = static_cast<E*>(B.arenaB) + L.off;
    TbpArgs A;
    A.dst = B.parity ? a : b;
    A.nx = L.nx;
    A.ny = L.ny;
    A.pitch = L.pitch;
    A.plane = L.plane;
    A.af = L.af;
    A.bf = L.bf;
    A.rows = B.rows;
    A.timeout = B.timeout;
    A.withhold = -1;
    const CUtensorMap* m = B.maps + 2 * (2 * t.x + B.parity);
    using G = TbpGeom<(int)sizeof(E), true>;
    if (t.w) tbp_body<G, K, NL, true>(m, m + 1, A, t.y, t.z);
    else tbp_body<G, K, NL, false>(m, m + 1, A, t.y, t.z);
}

}  // namespace lbmk
