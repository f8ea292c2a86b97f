// Two or three time steps per pass of the moment-space formats (lbm_ms.cuh), two adjacent columns
// per thread in packed FP32 arithmetic: the scheme of lbm_tbp.cuh with one level more in registers.
// The staged rows hold the moments (5 FP32 planes, 15 16-bit planes of scaled deviations); level 0
// is the rebuilding of a row's populations, done once per node, and level l + 1 is pulled from
// level l's last three rows exactly as there (shuffles for the x-neighbours at every level, so a
// warp loses one column per level and side: 56 of its 64 columns are stored).  The last level is
// stored as moments; nothing in between is rounded to 16 bits.
//
// Words.  The words a pass stores are those of the scalar kernel that came before this one, whose
// roundings the compiler chose: every sum with one product fused, but (all formats except periodic
// block floating point) Phi_x[4] = b m0[1] and Phi_y[3] = -b m0[1], one product used twice, rounded
// before the deviation was added.  Its warps each took 28 columns (30 in the two-step kernel) and
// rebuilt f_x of the columns just outside their halo alone, with that sum fused: so at each seam
// (a column c that is a multiple of 28, of 30 in two steps) the value pulled into c from the left and
// into c - 1 from the right starts from a fused Phi_x[4] + dx[4] three (two) columns away.  Only
// components 1 and 4 of those two chains differ (tbpms_seam_update); the last level takes them at the
// seams.  Without them the 16-bit roundings part from there on within a few hundred steps: the fields
// of a run differ by as much as the format's own error (1e-5).  About a tenth more instructions.
//
// What bounds it: latency, with at most two compute warps per scheduler (236 to 255 registers): 47 % of
// the issue slots and 32 % of DRAM in block floating point.  One column per thread took about 470 thread
// instructions per node and step there at 3 blocks per SM, two columns take 217.  Measured, block
// floating point, 300 steps on 4095 x 4001 from the initial fields to the moments: 104.7 ms before
// (three steps per pass, one column per thread), 67.5 ms now; the floor at 33.3 bytes per node and step
// is 24 ms.  30 steps of 4095 x 4001, one column per thread / now: BF16 and FP16 deviations 6.47 / 4.97 ms,
// Dirichlet 6.97 / 5.53, Dirichlet block floating point 9.57 / 7.17.
#pragma once

#include "lbm_ms.cuh"
#include "lbm_tbp.cuh"

namespace lbmk {

__device__ __forceinline__ f32x2 dup2(float v) { return pk(v, v); }

// the three words of one component of two columns (low half: the lower column) <-> their scaled
// deviations; decode returns them unscaled (inv = 1/scale)
template <typename Codec> struct PairCodec;

template <int H> struct PairCodec<MsFloatCodec<H>> {
    static __device__ __forceinline__ f32x2 one(uint32_t w, float inv)
    {
        return mul2(pk(Fmt<H>::ld((unsigned short)(w & 0xFFFFu)), Fmt<H>::ld((unsigned short)(w >> 16))), dup2(inv));
    }
    static __device__ __forceinline__ void decode(uint32_t wx, uint32_t wy, uint32_t wz, float inv, f32x2& x, f32x2& y,
                                                  f32x2& z)
    {
        x = one(wx, inv);
        y = one(wy, inv);
        z = one(wz, inv);
    }
    static __device__ __forceinline__ uint32_t word(f32x2 v)
    {
        float a, b;
        upk(v, a, b);
        return (uint32_t)Fmt<H>::st(a) | ((uint32_t)Fmt<H>::st(b) << 16);
    }
    static __device__ __forceinline__ void encode(f32x2 x, f32x2 y, f32x2 z, uint32_t& wx, uint32_t& wy, uint32_t& wz,
                                                  bool&, bool&)
    {
        wx = word(x);
        wy = word(y);
        wz = word(z);
    }
};

template <> struct PairCodec<MsBfpCodec> {
    // 2 m of a word's mantissa m as FP32, both columns: the word without its exponent bit, sign
    // bit turned, placed under the exponent of 2^23 is 2^23 + 2^15 + 2 m
    static __device__ __forceinline__ f32x2 mant2(uint32_t w)
    {
        const float lo = __uint_as_float((w & 0xFFFEu) ^ 0x4B008000u);
        const float hi = __uint_as_float(((w >> 16) & 0xFFFEu) ^ 0x4B008000u);
        return add2(pk(lo, hi), dup2(-8421376.f));
    }
    static __device__ __forceinline__ void decode(uint32_t wx, uint32_t wy, uint32_t wz, float inv, f32x2& x, f32x2& y,
                                                  f32x2& z)
    {
        const uint32_t t = (wx & 0x00010001u) | ((wy & 0x00010001u) << 1) | ((wz & 0x00010001u) << 2);
        // 2^(e-7) inv / 2: inv is a power of two in the normal range
        const uint32_t base = __float_as_uint(inv) - (8u << 23);
        const f32x2 f = pk(__uint_as_float((t << 23) + base), __uint_as_float(((t << 7) & 0x03800000u) + base));
        x = mul2(mant2(wx), f);
        y = mul2(mant2(wy), f);
        z = mul2(mant2(wz), f);
    }
    // exponent field of the block, clamped to the format's range, its scale factor 2^(7-e)
    static __device__ __forceinline__ uint32_t block(float X, float Y, float Z, float& f, bool& sat)
    {
        float m;
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(fabsf(X)), "f"(fabsf(Y)));
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(m), "f"(fabsf(Z)));
        uint32_t E = __float_as_uint(m) & 0x7F800000u;                 // (127 + q) << 23; NaN: the largest
        sat |= E > (140u << 23);
        E = min(max(E, 133u << 23), 140u << 23);                       // e = q - 6 in 0 .. 7
        f = __uint_as_float((267u << 23) - E);
        return E - (133u << 23);
    }
    // rounded mantissas of both columns, each within +-16383, in 16-bit halves
    static __device__ __forceinline__ uint32_t mants(f32x2 v, f32x2 f)
    {
        float a, b;
        upk(mul2(v, f), a, b);
        short i, j;
        asm("cvt.rni.s16.f32 %0, %1;" : "=h"(i) : "f"(a));             // saturates; NaN gives 0
        asm("cvt.rni.s16.f32 %0, %1;" : "=h"(j) : "f"(b));
        const uint32_t p = (uint32_t)(unsigned short)i | ((uint32_t)(unsigned short)j << 16);
        return __vmaxs2(__vmins2(p, 0x3FFF3FFFu), 0xC001C001u);
    }
    // satl, sath: set when the lower / upper column's block saturated
    static __device__ __forceinline__ void encode(f32x2 x, f32x2 y, f32x2 z, uint32_t& wx, uint32_t& wy, uint32_t& wz,
                                                  bool& satl, bool& sath)
    {
        float fl, fh;
        const uint32_t el = block(lo_of(x), lo_of(y), lo_of(z), fl, satl);
        const uint32_t eh = block(hi_of(x), hi_of(y), hi_of(z), fh, sath);
        const uint32_t t = (el >> 23) | (eh >> 7);                     // e of both columns in bits 0.., 16..
        const f32x2 f = pk(fl, fh);
        wx = ((mants(x, f) << 1) & 0xFFFEFFFEu) | (t & 0x00010001u);
        wy = ((mants(y, f) << 1) & 0xFFFEFFFEu) | ((t >> 1) & 0x00010001u);
        wz = ((mants(z, f) << 1) & 0xFFFEFFFEu) | ((t >> 2) & 0x00010001u);
    }
};

// populations of two columns from their moments (ms_dir).  SPLIT (see tbpms_compute): Phi_x[4] =
// b m0[1] and Phi_y[3] = -b m0[1] are rounded before the deviation is added, and f0h, f2h return
// f[0][4], f[2][4] with the fused sum instead; else every sum with one product is fused.  The
// separate roundings are scalar: a packed product and a packed sum are merged into one packed
// multiply-add whatever their rounding modifiers (seen in the results).
template <bool SPLIT>
__device__ __forceinline__ void tbpms_rebuild(const f32x2 (&m0)[5], const f32x2 (&dx)[5], const f32x2 (&dy)[5],
                                              const f32x2 (&dd)[5], const TbpConst& C, f32x2 (&f)[4][5], f32x2& f0h,
                                              f32x2& f2h)
{
    const f32x2 two = dup2(2.f), mtwo = dup2(-2.f), quarter = dup2(.25f);
    // T = Phi/c + deviation, per axis
    f32x2 tx[5], ty[5];
    tx[0] = add2(fma2(C.a, m0[2], mul2(C.b, m0[3])), dx[0]);
    tx[1] = fma2(C.b, m0[4], dx[1]);
    tx[2] = fma2(C.a, m0[0], dx[2]);
    tx[3] = fma2(C.b, m0[0], dx[3]);
    tx[4] = fma2(C.b, m0[1], dx[4]);
    ty[0] = fma2(C.b, m0[4], dy[0]);
    ty[1] = add2(fma2(C.a, m0[2], mul2(C.nb, m0[3])), dy[1]);
    ty[2] = fma2(C.a, m0[1], dy[2]);
    ty[3] = fma2(C.nb, m0[1], dy[3]);
    ty[4] = fma2(C.b, m0[0], dy[4]);
    if (SPLIT) {
        f0h = mul2(quarter, add2(fma2(two, tx[4], m0[4]), dd[4]));
        f2h = mul2(quarter, add2(fma2(mtwo, tx[4], m0[4]), dd[4]));
        const float pl = __fmul_rn(lo_of(C.b), lo_of(m0[1])), ph = __fmul_rn(lo_of(C.b), hi_of(m0[1]));
        tx[4] = pk(__fadd_rn(pl, lo_of(dx[4])), __fadd_rn(ph, hi_of(dx[4])));
        ty[3] = pk(__fsub_rn(lo_of(dy[3]), pl), __fsub_rn(hi_of(dy[3]), ph));
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        f[0][k] = mul2(quarter, add2(fma2(two, tx[k], m0[k]), dd[k]));
        f[2][k] = mul2(quarter, add2(fma2(mtwo, tx[k], m0[k]), dd[k]));
        f[1][k] = mul2(quarter, fma2(C.m1, dd[k], fma2(two, ty[k], m0[k])));
        f[3][k] = mul2(quarter, fma2(C.m1, dd[k], fma2(mtwo, ty[k], m0[k])));
    }
}

// Components 1 and 4 of the directions (1,0) and (-1,0) of tbp_update with X0, X2 in the place of
// x0, x2 in those components ([0]: component 1, [1]: component 4; the others do not enter)
template <bool NEG>
__device__ __forceinline__ void tbpms_seam_update(const TbpConst& C, const f32x2 (&X0)[2], const f32x2 (&x1)[5],
                                                  const f32x2 (&X2)[2], const f32x2 (&x3)[5], f32x2 (&o0)[2],
                                                  f32x2 (&o2)[2])
{
    f32x2 rx[2], U[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int k = j ? 4 : 1;
        rx[j] = NEG ? fma2(C.m1, x1[k], x3[k]) : add2(x1[k], x3[k]);
        U[j] = add2(rx[j], NEG ? fma2(C.m1, X0[j], X2[j]) : add2(X0[j], X2[j]));
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        o0[j] = fma2(NEG ? C.h : C.nh, U[j], fma2(NEG ? C.b : C.nb, U[1 - j], X0[j]));
        o2[j] = NEG ? fma2(C.m1, o0[j], rx[j]) : add2(rx[j], o0[j]);
    }
}

// moments of two columns' populations (ms_moments)
__device__ __forceinline__ void tbpms_moments(const f32x2 (&o)[4][5], const TbpConst& C, f32x2 (&m0)[5], f32x2 (&dx)[5],
                                              f32x2 (&dy)[5], f32x2 (&dd)[5])
{
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const f32x2 sx = add2(o[0][k], o[2][k]), sy = add2(o[1][k], o[3][k]);
        m0[k] = add2(sx, sy);
        dx[k] = fma2(C.m1, o[2][k], o[0][k]);
        dy[k] = fma2(C.m1, o[3][k], o[1][k]);
        dd[k] = fma2(C.m1, sy, sx);
    }
    dx[0] = fma2(C.m1, fma2(C.a, m0[2], mul2(C.b, m0[3])), dx[0]);
    dx[1] = fma2(C.nb, m0[4], dx[1]);
    dx[2] = fma2(C.na, m0[0], dx[2]);
    dx[3] = fma2(C.nb, m0[0], dx[3]);
    dx[4] = fma2(C.nb, m0[1], dx[4]);
    dy[0] = fma2(C.nb, m0[4], dy[0]);
    dy[1] = fma2(C.m1, fma2(C.a, m0[2], mul2(C.nb, m0[3])), dy[1]);
    dy[2] = fma2(C.na, m0[1], dy[2]);
    dy[3] = fma2(C.b, m0[1], dy[3]);
    dy[4] = fma2(C.nb, m0[0], dy[4]);
}

#ifndef LBM_TBPMS_NST
#define LBM_TBPMS_NST 7
#endif

constexpr int up128(int b) { return (b + 127) / 128 * 128; }   // copies land on 128-byte boundaries

struct TbpMsGeom {
    static constexpr int NLMAX = 3;
    static constexpr int NW = 3;                                       // compute warps
    static constexpr int MIN_BLOCKS = 2;
    static constexpr int LEAD = 4;                                     // NLMAX columns lost per side, made even
    static constexpr int OUTW = 64 - 2 * LEAD;
    static constexpr int OUT = NW * OUTW;                              // 168
    static constexpr int THREADS = 32 * (NW + 1);
    static constexpr int HL = 8;                                       // 16 bytes of 16-bit words
    static constexpr int WIN = HL + OUT + HL;
    static constexpr int WRAP = 16;                                    // columns of a wrap copy
    static constexpr int M0_BYTES = 5 * WIN * 4, DEV_BYTES = 15 * WIN * 2;
    static constexpr int WM0_BYTES = 5 * WRAP * 4, WDEV_BYTES = 15 * WRAP * 2;
    static constexpr int DEV = up128(M0_BYTES);                        // offsets in a stage
    static constexpr int WL0 = DEV + up128(DEV_BYTES), WLD = WL0 + up128(WM0_BYTES);
    static constexpr int WR0 = WLD + up128(WDEV_BYTES), WRD = WR0 + up128(WM0_BYTES);
    static constexpr int STAGE_BYTES = WRD + up128(WDEV_BYTES);
    static constexpr int NST = LBM_TBPMS_NST;
    static constexpr int SMEM = NST * STAGE_BYTES + 128;
    static_assert(LEAD % 2 == 0 && LEAD >= NLMAX && HL >= LEAD, "columns lost per level");
    static_assert((WIN * 2) % 16 == 0 && (OUT * 2) % 16 == 0 && WIN <= 256, "staged row geometry");
};

__device__ __forceinline__ int tbpms_wrap_x(int nx) { return (nx - TbpMsGeom::LEAD) & ~7; }

struct TbpMsArgs {
    void* dst;             // state at t + NL dt
    int nx, ny, pitch;
    long long plane;
    float af, bf;          // cK/c, cmu/c in FP32
    float scale, inv_s;    // scale of the stored deviations and its reciprocal (powers of two)
    int rows;              // output rows per block
    int* timeout;          // device flag: set when a bounded wait ran out
    int* sat;              // block floating point: set when a stored block saturated
    int withhold;          // test hook: staged input row the producer never copies (-1: none)
};

template <int K, int NL, bool DIRICHLET, bool EDGE>
__device__ __forceinline__ void tbpms_compute(const TbpMsArgs& A, int X0, int y0, int y1, uint32_t sbase,
                                              unsigned long long* full_bar, unsigned long long* empty_bar,
                                              volatile int* abort_flag)
{
    using G = TbpMsGeom;
    using Codec = PairCodec<typename Ms<K>::C>;
    constexpr int NST = G::NST, WIN = G::WIN;
    constexpr bool SPLIT = !(K == K_MSBFP && !DIRICHLET);
    constexpr int SEAM = NL == 3 ? 28 : 30;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nx = A.nx, ny = A.ny;
    const int nin = (y1 - y0) + 2 * NL;
    const int xs = X0 - G::LEAD + G::OUTW * warp + 2 * lane;   // this lane's lower column (even)
    const bool out_lane = lane >= G::LEAD / 2 && lane < 32 - G::LEAD / 2 && xs < nx;
    const bool both = xs + 1 < nx;
    const int own = xs - X0 + G::HL;
    const TbpConst C(A.af, A.bf);

    // EDGE, periodic: where the columns xs, xs + 1 sit in a stage, and their plane strides
    uint32_t e0[2], ed[2], s0e[2], sde[2];
    if (EDGE && !DIRICHLET) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            int c = (xs + q) % nx;
            c = c < 0 ? c + nx : c;
            const int m = c - X0 + G::HL, xl = tbpms_wrap_x(nx);
            if (m >= 0 && m < WIN) {
                e0[q] = 4u * m;
                ed[q] = G::DEV + 2u * m;
                s0e[q] = WIN * 4;
                sde[q] = WIN * 2;
            } else {
                const bool left = c >= xl && c < xl + G::WRAP;
                const int w = left ? c - xl : (c < G::WRAP ? c : 0);     // others feed no stored column
                e0[q] = (left ? G::WL0 : G::WR0) + 4u * w;
                ed[q] = (left ? G::WLD : G::WRD) + 2u * w;
                s0e[q] = G::WRAP * 4;
                sde[q] = G::WRAP * 2;
            }
        }
    }
    const bool wl = EDGE && DIRICHLET && xs == 0;
    const bool wr0 = EDGE && DIRICHLET && xs == nx - 1, wr1 = EDGE && DIRICHLET && xs + 1 == nx - 1;

    // The columns of a seam (header) this lane holds: c - 1 in its upper half, c in its lower half
    const bool seam_r = SPLIT && (xs + 2) % SEAM == 0, seam_l = SPLIT && xs % SEAM == 0;
    // [level][0, 1]: components 1, 4 that the level's seam update reads (level 0: component 4 only)
    f32x2 seam[NL - 1][2];
#pragma unroll
    for (int l = 0; l < NL - 1; ++l) seam[l][0] = seam[l][1] = 0ull;

    // per level as in tbp_compute; level 0 is the rebuilt state itself
    f32x2 s0[NL][5], s2[NL][5], k1[NL][5], c1[NL][5];
#pragma unroll
    for (int l = 0; l < NL; ++l)
#pragma unroll
        for (int k = 0; k < 5; ++k) s0[l][k] = s2[l][k] = k1[l][k] = c1[l][k] = 0ull;

    float* __restrict__ m0p = static_cast<float*>(A.dst);
    unsigned short* __restrict__ dvp = reinterpret_cast<unsigned short*>(m0p + 5 * A.plane);
    bool sat = false;
    int st = 0, ph = 0;
    for (int i = 0; i < nin; ++i) {
        const int R = y0 - NL + i;                         // the row rebuilt now
        const bool ok = lbmt::mbar_wait(lbmt::smem_u32(&full_bar[st]), ph, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) break;
        const uint32_t sb = sbase + st * G::STAGE_BYTES;
        f32x2 cur[4][5], sr[2], sl[2];                     // sr, sl: the seam values of cur (directions 0, 2)
        {
            f32x2 m0[5], dx[5], dy[5], dd[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                uint32_t w[3];
                if (EDGE && !DIRICHLET) {
                    m0[k] = pk(lbmt::lds_f32(sb + e0[0] + k * s0e[0]), lbmt::lds_f32(sb + e0[1] + k * s0e[1]));
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        w[j] = (uint32_t)lbmt::lds_u16(sb + ed[0] + (5 * j + k) * sde[0]) |
                               ((uint32_t)lbmt::lds_u16(sb + ed[1] + (5 * j + k) * sde[1]) << 16);
                } else {
                    m0[k] = Pair<K_F32>::lds(sb + 4 * own + k * (WIN * 4));
#pragma unroll
                    for (int j = 0; j < 3; ++j)
                        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w[j]) : "r"(sb + G::DEV + 2 * own + (5 * j + k) * (WIN * 2)) : "memory");
                }
                Codec::decode(w[0], w[1], w[2], A.inv_s, dx[k], dy[k], dd[k]);
            }
            tbpms_rebuild<SPLIT>(m0, dx, dy, dd, C, cur, sr[1], sl[1]);
        }
        __syncwarp();
        if (lane == 0) lbmt::mbar_arrive(lbmt::smem_u32(&empty_bar[st]));
        if (++st == NST) {
            st = 0;
            ph ^= 1;
        }
        // level l + 1 of row R - 1 - l from level l; cur holds level l's row R - l
#pragma unroll
        for (int l = 0; l < NL; ++l) {
            const int q = R - 1 - l;
            const bool neg = (l & 1) != 0;                 // cur[0], cur[1], s0, k1, c1 hold -f
            f32x2 out[4][5], nr[2], nl[2];
            {
                f32x2 x3[5];
#pragma unroll
                for (int k = 0; k < 5; ++k) x3[k] = cur[3][k];
                if (EDGE && DIRICHLET && q == ny - 1)
#pragma unroll
                    for (int k = 0; k < 5; ++k) x3[k] = ((k < 2) != neg) ? neg2(c1[l][k]) : c1[l][k];
                if (neg) tbp_update<true>(C, s0[l], k1[l], s2[l], x3, out);
                else tbp_update<false>(C, s0[l], k1[l], s2[l], x3, out);
                if (SPLIT && l < NL - 1) {
                    // level 1 of three: column c - 2 (lower half) pulls the seam value rightwards, c + 1
                    // (upper) leftwards; the level before the last: c - 1 (upper), c (lower)
                    const bool outer = NL == 3 && l == 0;
                    f32x2 p0[2], p2[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int k = j ? 4 : 1;
                        const f32x2 v = seam[l][j];
                        p0[j] = s0[l][k];
                        p2[j] = s2[l][k];
                        if (l == 0 && j == 0) continue;
                        if (outer) {
                            p0[j] = pk(lo_of(v), hi_of(p0[j]));
                            if (!wr1) p2[j] = pk(lo_of(p2[j]), hi_of(v));
                        } else {
                            p0[j] = pk(lo_of(p0[j]), hi_of(v));
                            if (!wr0) p2[j] = pk(lo_of(v), hi_of(p2[j]));
                        }
                    }
                    if (neg) tbpms_seam_update<true>(C, p0, k1[l], p2, x3, nr, nl);
                    else tbpms_seam_update<false>(C, p0, k1[l], p2, x3, nr, nl);
                }
            }
            if (SPLIT && l == 0 && NL == 3)
                seam[0][1] = pk(__shfl_up_sync(0xffffffffu, hi_of(sr[1]), 1), __shfl_down_sync(0xffffffffu, lo_of(sl[1]), 1));
            else if (SPLIT && l < NL - 1)
#pragma unroll
                for (int j = l == 0 ? 1 : 0; j < 2; ++j) seam[l][j] = pk(hi_of(sl[j]), lo_of(sr[j]));
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                float r0 = hi_of(cur[0][k]), l2 = lo_of(cur[2][k]);
                if (SPLIT && l == NL - 1 && (k == 1 || k == 4)) {
                    if (seam_r) r0 = hi_of(sr[k / 4]);
                    if (seam_l) l2 = lo_of(sl[k / 4]);
                }
                const float up = __shfl_up_sync(0xffffffffu, r0, 1);
                const float dn = __shfl_down_sync(0xffffffffu, l2, 1);
                s0[l][k] = pk(up, lo_of(cur[0][k]));
                s2[l][k] = pk(hi_of(cur[2][k]), dn);
                if (EDGE && DIRICHLET) {
                    const float Dk = ((k < 2) != neg) ? -1.f : 1.f;
                    if (wl) s0[l][k] = pk(Dk * lo_of(cur[2][k]), lo_of(cur[0][k]));
                    if (wr0) s2[l][k] = pk(Dk * lo_of(cur[0][k]), dn);
                    if (wr1) s2[l][k] = pk(hi_of(cur[2][k]), Dk * hi_of(cur[0][k]));
                }
                k1[l][k] = c1[l][k];
                c1[l][k] = cur[1][k];
            }
            if (EDGE && DIRICHLET && q + 1 == 0)           // the wall below row 0
#pragma unroll
                for (int k = 0; k < 5; ++k) k1[l][k] = ((k < 2) != neg) ? neg2(cur[3][k]) : cur[3][k];
#pragma unroll
            for (int d = 0; d < 4; ++d)
#pragma unroll
                for (int k = 0; k < 5; ++k) cur[d][k] = out[d][k];
            if (SPLIT && l < NL - 1)
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    sr[j] = nr[j];
                    sl[j] = nl[j];
                }
        }
        const int q = R - NL;
        if (q >= y0) {
            if (NL & 1)
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    cur[0][k] = neg2(cur[0][k]);
                    cur[1][k] = neg2(cur[1][k]);
                }
            f32x2 m0[5], dx[5], dy[5], dd[5];
            tbpms_moments(cur, C, m0, dx, dy, dd);
            if (out_lane) {
                const f32x2 sc = dup2(A.scale);
                const long long off = (long long)q * A.pitch + xs;
                bool clipl = false, cliph = false;
#pragma unroll
                for (int k = 0; k < 5; ++k) {
                    uint32_t w[3];
                    Codec::encode(mul2(dx[k], sc), mul2(dy[k], sc), mul2(dd[k], sc), w[0], w[1], w[2], clipl, cliph);
                    if (both) {
                        *reinterpret_cast<f32x2*>(m0p + k * A.plane + off) = m0[k];
#pragma unroll
                        for (int j = 0; j < 3; ++j)
                            *reinterpret_cast<uint32_t*>(dvp + (5 * j + k) * A.plane + off) = w[j];
                    } else {                               // odd nx: the last column alone
                        m0p[k * A.plane + off] = lo_of(m0[k]);
#pragma unroll
                        for (int j = 0; j < 3; ++j) dvp[(5 * j + k) * A.plane + off] = (unsigned short)(w[j] & 0xFFFFu);
                    }
                }
                sat |= clipl || (both && cliph);           // column nx of an odd width is not stored
            }
        }
    }
    if (sat && A.sat) atomicOr(A.sat, 1);
    if (lane == 0 && *abort_flag) atomicExch(A.timeout, 1);
}

// maps: row maps of the FP32 and the 16-bit part (box WIN), wrap maps of both (box WRAP)
template <int K, int NL, bool DIRICHLET>
__global__ void __launch_bounds__(TbpMsGeom::THREADS, TbpMsGeom::MIN_BLOCKS)
    tbpms_kernel(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap mapd,
                 const __grid_constant__ CUtensorMap wmap0, const __grid_constant__ CUtensorMap wmapd, TbpMsArgs A)
{
    using G = TbpMsGeom;
    constexpr int NST = G::NST;
    extern __shared__ __align__(128) unsigned char tbp_smem_raw[];
    __shared__ __align__(8) unsigned long long full_bar[NST], empty_bar[NST];
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nx = A.nx, ny = A.ny;
    const int X0 = blockIdx.x * G::OUT, y0 = blockIdx.y * A.rows;
    const int y1 = min(ny, y0 + A.rows);
    const int nin = (y1 - y0) + 2 * NL;              // staged input rows y0 - NL .. y1 + NL - 1
    const int nact = min(G::NW, (nx - X0 + G::OUTW - 1) / G::OUTW);
    const bool edge = X0 == 0 || X0 + G::OUT + G::LEAD >= nx ||
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
            lbmt::prefetch_map(&map0);
            lbmt::prefetch_map(&mapd);
            const bool wrap = !DIRICHLET && edge && nx > G::OUT;
            const uint32_t bytes = G::M0_BYTES + G::DEV_BYTES + (wrap ? 2 * (G::WM0_BYTES + G::WDEV_BYTES) : 0);
            const int xl = tbpms_wrap_x(nx);
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
                        lbmt::tma_load_3d(st, &map0, X0 - G::HL, y, 0, fb);
                        lbmt::tma_load_3d(st + G::DEV, &mapd, X0 - G::HL, y, 0, fb);
                        if (wrap) {
                            lbmt::tma_load_3d(st + G::WL0, &wmap0, xl, y, 0, fb);
                            lbmt::tma_load_3d(st + G::WLD, &wmapd, xl, y, 0, fb);
                            lbmt::tma_load_3d(st + G::WR0, &wmap0, 0, y, 0, fb);
                            lbmt::tma_load_3d(st + G::WRD, &wmapd, 0, y, 0, fb);
                        }
                    }
                }
                if (++s == NST) {
                    s = 0;
                    ph ^= 1;
                }
            }
            for (int q = (j > NST ? j - NST : 0); q < j; ++q)      // every copy issued has landed
                if (q != A.withhold) lbmt::mbar_drain(lbmt::smem_u32(&full_bar[q % NST]), (q / NST) & 1);
            if (abort_flag) atomicExch(A.timeout, 1);
        }
        return;
    }
    if (warp >= nact) return;
    lbmt::grid_dependency_wait();
    if (edge) tbpms_compute<K, NL, DIRICHLET, true>(A, X0, y0, y1, sbase, full_bar, empty_bar, &abort_flag);
    else tbpms_compute<K, NL, DIRICHLET, false>(A, X0, y0, y1, sbase, full_bar, empty_bar, &abort_flag);
}

}  // namespace lbmk
