// Instantiates every kernel for one storage format; compiled once per format
// with -DLBM_KIND=<0..6> (FP64, FP32, BF16, FP16, and moment space with BF16, FP16
// or block-floating-point deviations).
#include "lbm_dispatch.h"

#include <algorithm>

#ifndef LBM_KIND
#error "LBM_KIND must be defined"
#endif

namespace {

#ifndef LBM_VEC_F64
#define LBM_VEC_F64 2
#endif
#ifndef LBM_VEC_F32
#define LBM_VEC_F32 4
#endif
#ifndef LBM_VEC_F16
#define LBM_VEC_F16 4
#endif
#ifndef LBM_VEC_SPLIT
#define LBM_VEC_SPLIT 1
#endif

constexpr int K = LBM_KIND;
constexpr bool MS = (K >= lbmk::K_MSBF16);
// nodes per thread in the step kernel (one vector access per plane and thread)
constexpr int V = (K == lbmk::K_F64) ? LBM_VEC_F64 : (K == lbmk::K_F32) ? LBM_VEC_F32 : MS ? 4 : LBM_VEC_F16;
#ifndef LBM_VEC_STEP
#define LBM_VEC_STEP 2
#endif
// nodes per thread of the single step (measured beside step_kernel)
constexpr int VS = (K == lbmk::K_F64 || MS) ? V : LBM_VEC_STEP;
constexpr int ELEM = (K == lbmk::K_F64) ? 8 : (K == lbmk::K_F32) ? 4 : 2;
// nodes per thread in the batch kernel (FP64 runs the split collision, at its width)
constexpr int VB = (K == lbmk::K_F64) ? LBM_VEC_SPLIT : V;
constexpr int NODE_BYTES = MS ? 5 * 4 + 15 * 2 : 20 * ELEM;

template <bool D, bool F, bool T, bool O, unsigned long long SPLIT = 0>
cudaError_t step_v(const lbmk::StepArgs& a, dim3 g, dim3 b, cudaStream_t s)
{
    if constexpr (MS) lbmk::ms_step_kernel<K, V, D, F, T, O><<<g, b, 0, s>>>(a);
    else if constexpr (SPLIT > 0) lbmk::step_kernel<K, LBM_VEC_SPLIT, D, F, T, O, SPLIT><<<g, b, 0, s>>>(a);
    else if constexpr (K == lbmk::K_F64) lbmk::step_kernel<K, V, D, F, T, O><<<g, b, 0, s>>>(a);
    else {
        // 16-bit populations without load, tracking or omega: four nodes per thread (8-byte accesses) from
        // 2^19 nodes on (us per step of four / two nodes, periodic: 5000 x 6000 345 / 389, 1024^2 8.9 / 10.7,
        // Dirichlet: 349 / 398, 1024^2 12.5 / 13.4, but 512^2 6.5 / 5.7, 256^2 6.5 / 5.1)
        if constexpr (ELEM == 2 && !F && !T && !O)
            if ((long long)a.nx * a.ny >= 1 << 19) {
                const int nchunk = (a.nx + 3) / 4, bx = std::min(64, (nchunk + 31) / 32 * 32);
                return lbmh::launch_dependent(lbmk::step_kernel<K, 4, D, F, T, O>, dim3((nchunk + bx - 1) / bx, a.ny),
                                              dim3(bx), 0, s, a);
            }
        return lbmh::launch_dependent(lbmk::step_kernel<K, VS, D, F, T, O>, g, b, 0, s, a);
    }
    return cudaGetLastError();
}

// FP64 without body load and with omega = 2: the number of the node's 35
// additions computed on the integer pipes (lbmh::split_adds of the level)
template <bool D, bool T>
cudaError_t step_split(const lbmk::StepArgs& a, int level, dim3 g, dim3 b, cudaStream_t s)
{
    if constexpr (K != lbmk::K_F64) {
        return cudaErrorNotSupported;
    } else {
        switch (level) {
        case 1: return step_v<D, false, T, false, lbmh::split_mask(1)>(a, g, b, s);
        case 2: return step_v<D, false, T, false, lbmh::split_mask(2)>(a, g, b, s);
        case 3: return step_v<D, false, T, false, lbmh::split_mask(3)>(a, g, b, s);
        case 4: return step_v<D, false, T, false, lbmh::split_mask(4)>(a, g, b, s);
        case 5: return step_v<D, false, T, false, lbmh::split_mask(5)>(a, g, b, s);
        case 6: return step_v<D, false, T, false, lbmh::split_mask(6)>(a, g, b, s);
        case 7: return step_v<D, false, T, false, lbmh::split_mask(7)>(a, g, b, s);
        case 8: return step_v<D, false, T, false, lbmh::split_mask(8)>(a, g, b, s);
        case 9: return step_v<D, false, T, false, lbmh::split_mask(9)>(a, g, b, s);
        case 10: return step_v<D, false, T, false, lbmh::split_mask(10)>(a, g, b, s);
        case 11: return step_v<D, false, T, false, lbmh::split_mask(11)>(a, g, b, s);
        case 12: return step_v<D, false, T, false, lbmh::split_mask(12)>(a, g, b, s);
        default: return cudaErrorInvalidValue;
        }
    }
}

#ifndef LBM_SA_MASK
#define LBM_SA_MASK lbmh::split_mask(1)   // the additions of split level 1 on the integer pipes
#endif

// FP64 at split level 1 or 12 with the rows staged by asynchronous copies (lbm_f64stage.cuh),
// a body load at level 12 only; other formats, levels and variants return cudaErrorNotSupported
template <bool D, bool T, bool F, unsigned long long M>
cudaError_t step_staged_dt(const lbmk::StepArgs& a, int rows, cudaStream_t s)
{
    if constexpr (K != lbmk::K_F64) {
        return cudaErrorNotSupported;
    } else {
        const dim3 g((a.nx + lbmk::SA_THREADS - 1) / lbmk::SA_THREADS, (a.ny + rows - 1) / rows);
        return lbmh::launch_dependent(lbmk::step_f64_staged_kernel<D, T, F, M>, g, dim3(lbmk::SA_THREADS), 0, s, a, rows);
    }
}

template <bool F, unsigned long long M>
cudaError_t step_staged_m(const lbmk::StepArgs& a, bool d, bool t, int rows, cudaStream_t s)
{
    return d ? (t ? step_staged_dt<true, true, F, M>(a, rows, s) : step_staged_dt<true, false, F, M>(a, rows, s))
             : (t ? step_staged_dt<false, true, F, M>(a, rows, s) : step_staged_dt<false, false, F, M>(a, rows, s));
}

// split levels 1 (LBM_SA_MASK) and 12 (fixed point)
cudaError_t step_staged(const lbmk::StepArgs& a, int variant, int rows, cudaStream_t s)
{
    constexpr unsigned long long FX = lbmh::split_mask(lbmh::STEP_SPLIT_FIXED);
    const int level = (variant >> lbmh::STEP_SPLIT_SHIFT) & 15;
    const bool force = variant & lbmh::STEP_FORCING;
    if ((level != 1 && level != lbmh::STEP_SPLIT_FIXED) || (variant & lbmh::STEP_OMEGA) ||
        (force && level != lbmh::STEP_SPLIT_FIXED) || rows < 1)
        return cudaErrorNotSupported;
    const bool d = variant & lbmh::STEP_DIRICHLET, t = variant & lbmh::STEP_TRACK;
    if (level == 1) return step_staged_m<false, LBM_SA_MASK>(a, d, t, rows, s);
    return force ? step_staged_m<true, FX>(a, d, t, rows, s) : step_staged_m<false, FX>(a, d, t, rows, s);
}

// `steps` FP64 steps of a small lattice at split level 12 in one cooperative launch
// (multi_f64_kernel); cudaErrorNotSupported where one launch per step is the better form
template <bool D, bool T, bool F>
cudaError_t step_multi_dtf(const lbmk::StepArgs& a, int steps, unsigned int* flags, int max_flags, int* timeout,
                           int withhold, cudaStream_t s)
{
    if constexpr (K != lbmk::K_F64) {
        return cudaErrorNotSupported;
    } else {
        constexpr int W = lbmk::MULTI_WARPS;
        lbmk::MultiArgs q;
        q.A = a;
        q.steps = steps;
        q.nseg = (a.nx + 31) / 32;
        const long long ntask = (long long)q.nseg * a.ny;
        int dev = 0, sms = 0, occ = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, lbmk::multi_f64_kernel<D, T, F>, 32 * W, 0);
        if (e != cudaSuccess) return e;
        // up to half of the blocks that fit on the chip (two per SM), so that two such lattices on streams
        // of their own run side by side: one that takes more makes the others wait for its whole call (200
        // steps, us, this kernel / a launch per step before: two of 208^2 2057 / 2645, but four 4112 / 3418,
        // sixteen 16829 / 8671).  Alone, beyond three blocks per SM a launch per step is as fast (us per step,
        // this kernel / launches: 64^2 3.3 / 5.0, 128^2 3.4 / 5.2, 256^2 5.9 / 5.6; with body load and
        // tracking 4.1 / 5.1, 4.3 / 6.3, 6.6 / 6.6)
        const long long cap = std::min((long long)std::min(occ, 4) * sms / 2, (long long)max_flags / lbmk::MULTI_FLAG) * W;
        if (cap < W || ntask > cap) return cudaErrorNotSupported;
        q.ntask = (int)ntask;
        q.nblk = (q.ntask + W - 1) / W;
        // a node's sources lie within nseg segments of its own, cyclically; one block more for the
        // shorter last block, one for the rounding
        q.reach = std::min((q.nseg + W - 1) / W + 2, q.nblk - 1);
        q.flags = flags;
        q.timeout = timeout;
        q.withhold = withhold;
        e = cudaMemsetAsync(flags, 0, (size_t)q.nblk * lbmk::MULTI_FLAG * sizeof(unsigned int), s);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(q.nblk);
        cfg.blockDim = dim3(32 * W);
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, lbmk::multi_f64_kernel<D, T, F>, q);
        if (e == cudaErrorCooperativeLaunchTooLarge) {       // part of the chip reserved for others
            cudaGetLastError();
            return cudaErrorNotSupported;
        }
        return e;
    }
}

cudaError_t step_multi(const lbmk::StepArgs& a, int variant, int steps, unsigned int* flags, int max_flags,
                       int* timeout, int withhold, cudaStream_t s)
{
    switch (variant & 7) {
    case 0: return step_multi_dtf<false, false, false>(a, steps, flags, max_flags, timeout, withhold, s);
    case 1: return step_multi_dtf<true, false, false>(a, steps, flags, max_flags, timeout, withhold, s);
    case 2: return step_multi_dtf<false, false, true>(a, steps, flags, max_flags, timeout, withhold, s);
    case 3: return step_multi_dtf<true, false, true>(a, steps, flags, max_flags, timeout, withhold, s);
    case 4: return step_multi_dtf<false, true, false>(a, steps, flags, max_flags, timeout, withhold, s);
    case 5: return step_multi_dtf<true, true, false>(a, steps, flags, max_flags, timeout, withhold, s);
    case 6: return step_multi_dtf<false, true, true>(a, steps, flags, max_flags, timeout, withhold, s);
    default: return step_multi_dtf<true, true, true>(a, steps, flags, max_flags, timeout, withhold, s);
    }
}

template <bool O>
cudaError_t step_o(const lbmk::StepArgs& a, int variant, dim3 g, dim3 b, cudaStream_t s)
{
    switch (variant & 7) {
    case 0: return step_v<false, false, false, O>(a, g, b, s);
    case 1: return step_v<true, false, false, O>(a, g, b, s);
    case 2: return step_v<false, true, false, O>(a, g, b, s);
    case 3: return step_v<true, true, false, O>(a, g, b, s);
    case 4: return step_v<false, false, true, O>(a, g, b, s);
    case 5: return step_v<true, false, true, O>(a, g, b, s);
    case 6: return step_v<false, true, true, O>(a, g, b, s);
    default: return step_v<true, true, true, O>(a, g, b, s);
    }
}

// FP64 with a body load at split level 12 (omega = 2): the fixed-point node update with it
template <bool D, bool T>
cudaError_t step_fixed_forced(const lbmk::StepArgs& a, dim3 g, dim3 b, cudaStream_t s)
{
    if constexpr (K != lbmk::K_F64) {
        return cudaErrorNotSupported;
    } else {
        return step_v<D, true, T, false, lbmh::split_mask(lbmh::STEP_SPLIT_FIXED)>(a, g, b, s);
    }
}

cudaError_t step(const lbmk::StepArgs& a, int variant, dim3 g, dim3 b, cudaStream_t s)
{
    const int level = (variant >> lbmh::STEP_SPLIT_SHIFT) & 15;
    if (level == lbmh::STEP_SPLIT_FIXED && (variant & lbmh::STEP_FORCING) && !(variant & lbmh::STEP_OMEGA)) {
        const bool d = variant & lbmh::STEP_DIRICHLET, t = variant & lbmh::STEP_TRACK;
        return d ? (t ? step_fixed_forced<true, true>(a, g, b, s) : step_fixed_forced<true, false>(a, g, b, s))
                 : (t ? step_fixed_forced<false, true>(a, g, b, s) : step_fixed_forced<false, false>(a, g, b, s));
    }
    if (level && !(variant & (lbmh::STEP_FORCING | lbmh::STEP_OMEGA))) {
        const bool d = variant & lbmh::STEP_DIRICHLET, t = variant & lbmh::STEP_TRACK;
        return d ? (t ? step_split<true, true>(a, level, g, b, s) : step_split<true, false>(a, level, g, b, s))
                 : (t ? step_split<false, true>(a, level, g, b, s) : step_split<false, false>(a, level, g, b, s));
    }
    return (variant & lbmh::STEP_OMEGA) ? step_o<true>(a, variant, g, b, s) : step_o<false>(a, variant, g, b, s);
}

cudaError_t init(const lbmk::NodeArgs& a, const double* U0, const double* Ux, const double* Uy,
                 const double* B0, const double* u0, cudaStream_t s)
{
    // enough blocks for several per SM, then more rows per block: a thread's constants cost
    // about as many FP64 operations as a tenth of a node
    const int nbx = (a.nx + 127) / 128;
    const dim3 b(128), g(nbx, std::min(a.ny, std::max(1, 152 * 48 / nbx)));
    if (B0) lbmk::init_kernel<K, true><<<g, b, 0, s>>>(a, U0, Ux, Uy, B0, u0);
    else lbmk::init_kernel<K, false><<<g, b, 0, s>>>(a, U0, Ux, Uy, B0, u0);
    return cudaGetLastError();
}

cudaError_t moments(const lbmk::NodeArgs& a, double* out, dim3 g, dim3 b, cudaStream_t s)
{
    lbmk::moments_kernel<K><<<g, b, 0, s>>>(a, out);
    return cudaGetLastError();
}

cudaError_t get_pop(const lbmk::NodeArgs& a, double* f, double* ustar, dim3 g, dim3 b, cudaStream_t s)
{
    lbmk::get_populations_kernel<K><<<g, b, 0, s>>>(a, f, ustar);
    return cudaGetLastError();
}

cudaError_t set_pop(const lbmk::NodeArgs& a, const double* f, const double* ustar, dim3 g, dim3 b,
                    cudaStream_t s)
{
    lbmk::set_populations_kernel<K><<<g, b, 0, s>>>(a, f, ustar);
    return cudaGetLastError();
}

cudaError_t energy(const lbmk::NodeArgs& a, double* partial, dim3 g, dim3 b, cudaStream_t s)
{
    lbmk::energy_kernel<K><<<g, b, 0, s>>>(a, partial);
    return cudaGetLastError();
}

cudaError_t error(const lbmk::NodeArgs& a, const double* exact, double* partial, dim3 g, dim3 b,
                  cudaStream_t s)
{
    lbmk::error_kernel<K><<<g, b, 0, s>>>(a, exact, partial);
    return cudaGetLastError();
}

cudaError_t finite(const lbmk::NodeArgs& a, int* flag, dim3 g, dim3 b, cudaStream_t s)
{
    lbmk::finite_kernel<K><<<g, b, 0, s>>>(a, flag);
    return cudaGetLastError();
}

template <int KK>
cudaError_t batch_step_t(const lbmk::BatchArgs& a, bool persistent, int grid, cudaStream_t s)
{
    if constexpr (KK >= lbmk::K_MSBF16) {
        return cudaErrorNotSupported;        // batches use the population formats only
    } else {
        if (!persistent) {
            lbmk::batch_step_kernel<KK, VB, false><<<grid, 256, 0, s>>>(a);
            return cudaGetLastError();
        }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = 0;
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, lbmk::batch_step_kernel<KK, VB, true>, a);
    }
}

template <int KK>
cudaError_t batch_occupancy_t(int* n)
{
    if constexpr (KK >= lbmk::K_MSBF16) {
        *n = 1;
        return cudaSuccess;
    } else {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, lbmk::batch_step_kernel<KK, VB, true>, 256, 0);
    }
}

cudaError_t batch_step(const lbmk::BatchArgs& a, bool persistent, int grid, cudaStream_t s)
{
    return batch_step_t<K>(a, persistent, grid, s);
}

template <int KK>
cudaError_t tb2_t(const lbmk::TbArgs& a, bool dirichlet, dim3 g, dim3 b, cudaStream_t s)
{
    if constexpr (KK == lbmk::K_F32 || KK == lbmk::K_BF16 || KK == lbmk::K_F16) {
        if (dirichlet) lbmk::tb2_kernel<KK, true><<<g, b, 0, s>>>(a);
        else lbmk::tb2_kernel<KK, false><<<g, b, 0, s>>>(a);
        return cudaGetLastError();
    } else {
        return cudaErrorNotSupported;
    }
}

cudaError_t tb2_step(const lbmk::TbArgs& a, bool dirichlet, dim3 g, dim3 b, cudaStream_t s)
{
    return tb2_t<K>(a, dirichlet, g, b, s);
}

// 2 .. TbpGeom::NLMAX fused steps of the population formats (lbm_tbp.cuh)
template <int KK, int NL>
cudaError_t tbp_nl(const CUtensorMap* maps, const lbmk::TbpArgs& a, bool dirichlet, cudaStream_t s)
{
    using G = lbmk::TbpGeom<(int)sizeof(typename lbmk::Fmt<KK>::E)>;
    void (*kern)(CUtensorMap, CUtensorMap, lbmk::TbpArgs) =
        dirichlet ? lbmk::tbp_kernel<KK, NL, true> : lbmk::tbp_kernel<KK, NL, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
    if (e != cudaSuccess) return e;
    const dim3 g((a.nx + G::OUT - 1) / G::OUT, (a.ny + a.rows - 1) / a.rows);
    return lbmh::launch_dependent(kern, g, dim3(G::THREADS), G::SMEM, s, maps[0], maps[1], a);
}

template <int KK>
cudaError_t tbp_t(const CUtensorMap* maps, const lbmk::TbpArgs& a, int steps, bool dirichlet, cudaStream_t s)
{
    if constexpr (KK == lbmk::K_F32 || KK == lbmk::K_BF16 || KK == lbmk::K_F16) {
        constexpr int MX = lbmk::TbpGeom<(int)sizeof(typename lbmk::Fmt<KK>::E)>::NLMAX;
        switch (steps) {
        case 2: return tbp_nl<KK, 2>(maps, a, dirichlet, s);
        case 3: return tbp_nl<KK, 3>(maps, a, dirichlet, s);
        case 4: if constexpr (MX >= 4) return tbp_nl<KK, 4>(maps, a, dirichlet, s); break;
        }
    }
    return cudaErrorNotSupported;
}

cudaError_t tbp_step(const CUtensorMap* maps, const lbmk::TbpArgs& a, int steps, bool dirichlet, cudaStream_t s)
{
    return tbp_t<K>(maps, a, steps, dirichlet, s);
}

// two or three fused steps of the moment-space formats (lbm_tbpms.cuh)
template <int KK, int NL>
cudaError_t tbpms_nl(const CUtensorMap* maps, const lbmk::TbpMsArgs& a, bool dirichlet, cudaStream_t s)
{
    using G = lbmk::TbpMsGeom;
    void (*kern)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, lbmk::TbpMsArgs) =
        dirichlet ? lbmk::tbpms_kernel<KK, NL, true> : lbmk::tbpms_kernel<KK, NL, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
    if (e != cudaSuccess) return e;
    const dim3 g((a.nx + G::OUT - 1) / G::OUT, (a.ny + a.rows - 1) / a.rows);
    return lbmh::launch_dependent(kern, g, dim3(G::THREADS), G::SMEM, s, maps[0], maps[1], maps[2], maps[3], a);
}

template <int KK>
cudaError_t tbpms_t(const CUtensorMap* maps, const lbmk::TbpMsArgs& a, int steps, bool dirichlet, cudaStream_t s)
{
    if constexpr (KK == lbmk::K_MSBF16 || KK == lbmk::K_MSF16 || KK == lbmk::K_MSBFP) {
        if (steps == 3) return tbpms_nl<KK, 3>(maps, a, dirichlet, s);
        if (steps == 2) return tbpms_nl<KK, 2>(maps, a, dirichlet, s);
    }
    return cudaErrorNotSupported;
}

cudaError_t tbpms_step(const CUtensorMap* maps, const lbmk::TbpMsArgs& a, int steps, bool dirichlet, cudaStream_t s)
{
    return tbpms_t<K>(maps, a, steps, dirichlet, s);
}

template <int KK, int NL>
cudaError_t batch_tbp_nl(const lbmk::BatchTbpArgs& a, int ntiles, cudaStream_t s)
{
    using G = lbmk::TbpGeom<(int)sizeof(typename lbmk::Fmt<KK>::E), true>;
    void (*kern)(lbmk::BatchTbpArgs) = lbmk::batch_tbp_kernel<KK, NL>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM);
    if (e != cudaSuccess) return e;
    return lbmh::launch_dependent(kern, dim3(ntiles), dim3(G::THREADS), G::SMEM, s, a);
}

template <int KK>
cudaError_t batch_tbp_t(const lbmk::BatchTbpArgs& a, int steps, int ntiles, cudaStream_t s)
{
    if (ntiles <= 0) return cudaSuccess;
    if constexpr (KK == lbmk::K_F32 || KK == lbmk::K_BF16 || KK == lbmk::K_F16) {
        constexpr int MX = lbmk::TbpGeom<(int)sizeof(typename lbmk::Fmt<KK>::E)>::NLMAX;
        switch (steps) {
        case 2: if constexpr (MX >= 4) return batch_tbp_nl<KK, 2>(a, ntiles, s); break;
        case 3: return batch_tbp_nl<KK, 3>(a, ntiles, s);
        case 4: if constexpr (MX >= 4) return batch_tbp_nl<KK, 4>(a, ntiles, s); break;
        }
    }
    return cudaErrorNotSupported;
}

cudaError_t batch_tbp_step(const lbmk::BatchTbpArgs& a, int steps, int ntiles, cudaStream_t s)
{
    return batch_tbp_t<K>(a, steps, ntiles, s);
}

cudaError_t batch_occupancy(int* n)
{
    return batch_occupancy_t<K>(n);
}

}  // namespace

namespace lbmh {

#define LBM_OPS_NAME2(k) kind_ops_##k
#define LBM_OPS_NAME(k) LBM_OPS_NAME2(k)

const KindOps LBM_OPS_NAME(LBM_KIND) = {
    K, VS, ELEM, NODE_BYTES,
    step, init, moments, get_pop, set_pop, energy, error, finite, batch_step, batch_occupancy, tb2_step, tbp_step,
    tbpms_step, step_staged, step_multi, batch_tbp_step,
    LBM_VEC_SPLIT, VB,
};

}  // namespace lbmh
