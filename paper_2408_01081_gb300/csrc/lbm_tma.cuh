// Tensor-memory-access (TMA) row staging for the lattice kernels: mbarrier and
// cp.async.bulk.tensor helpers in inline PTX (sm_103a).
//
// A lattice buffer of P planes [P][ny][pitch] is described by a 3D tensor map
// (x = column, extent nx; y = row, extent ny; z = plane, extent P) whose box is
// {W, 1, P}: one copy brings W consecutive columns of one row of every plane into
// shared memory as [P][W] (x fastest).  Columns outside [0, nx) and rows outside
// [0, ny) arrive as zeros.  The x coordinate of every copy is a multiple of
// 16 bytes / element size, as the tensor copy requires.
//
// Every wait is bounded (about two seconds of SM clock); a wait that runs out
// returns false, and the kernels then record a timeout in a device flag and leave.
#pragma once

#include <cuda.h>
#include <stdint.h>

namespace lbmt {

constexpr long long kWaitCycles = 4000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// For kernels launched by lbmh::launch_dependent: let the next kernel's blocks become resident
// as soon as every block of this one has started, and wait for the previous kernel's completion
// (before the first access to anything an earlier kernel of the stream reads or writes).
__device__ __forceinline__ void grid_dependency_wait()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// make the initialised barriers visible to the tensor-copy unit
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
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

// wait until the phase with this parity has completed; false once the limit runs out
// or another role of the block has given up (*abort set)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort) return false;
        if (clock64() - t0 > kWaitCycles) {
            *abort = 1;
            return false;
        }
    }
}

// bounded wait that ignores the abort flag (draining copies in flight before the block exits)
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity)
{
    const long long t0 = clock64();
    while (!mbar_try(bar, parity))
        if (clock64() - t0 > kWaitCycles) return false;
    return true;
}

// shared-memory loads by 32-bit shared address (explicitly in the shared state space)
__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ unsigned short lds_u16(uint32_t addr)
{
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}

template <typename E> __device__ __forceinline__ E lds(uint32_t addr);
template <> __device__ __forceinline__ float lds<float>(uint32_t addr) { return lds_f32(addr); }
template <> __device__ __forceinline__ unsigned short lds<unsigned short>(uint32_t addr) { return lds_u16(addr); }

// one 3D tensor copy global -> shared, completion counted in bytes on `bar`
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

}  // namespace lbmt
