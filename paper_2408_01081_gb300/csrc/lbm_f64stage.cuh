// FP64 step (omega = 2; the node update of split level 1, the IEEE operation sequence, without
// body load, or 12, the fixed-point update, with or without one) with each node's inputs staged in shared memory
// by per-thread asynchronous copies (cp.async), one row ahead.
//
// The register step kernel loads the 20 inputs of a node and then waits for them:
// with 80 registers and three 256-thread blocks per SM, about a sixth of its warp
// cycles go to that wait (long scoreboard) while the integer pipe, which shares the
// bound of the split collision with the FP64 pipe, idles.  Here a block of 128 threads
// owns 128 consecutive columns and walks down `rows` rows (the library passes up to 2 at level 1
// and up to 4 at level 12, fewer on small lattices), thread t computing column t of each row.  The copies of the next row are issued as soon as
// the current row has been read out of shared memory, so they are in flight during its
// whole collision and occupy no registers.  Each thread copies exactly the 20 values its
// own node pulls (f*_(1,0) from x - 1, f*_(-1,0) from x + 1, f*_(0,1) from y - 1,
// f*_(0,-1) from y + 1, with the periodic wrap or the Dirichlet edge reflection in the
// source address), so no value crosses threads and no barrier or wait loop is needed: a
// thread's copies of a row complete by cp.async.wait_group.  The node arithmetic is
// collide_split of the same level (collide_fixed_forced with a body load) as in step_kernel (lbm_kernels.cuh) on the same inputs,
// so results are bit-identical to it.
#pragma once

#include "lbm_kernels.cuh"
#include "lbm_tma.cuh"

namespace lbmk {

#ifndef LBM_SA_THREADS
#define LBM_SA_THREADS 128
#endif
constexpr int SA_THREADS = LBM_SA_THREADS;            // columns per block, one per thread
constexpr int SA_SLOTS = 20;                          // inputs per node
#ifndef LBM_SA_MIN_BLOCKS
#define LBM_SA_MIN_BLOCKS 6                           // 6 x 128 threads at <= 85 registers
#endif
#ifndef LBM_SA_FX_MIN_BLOCKS
#define LBM_SA_FX_MIN_BLOCKS 4                        // fixed-point node update: <= 128 registers
#endif

__device__ __forceinline__ void cp_async8(uint32_t dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ double lds_f64(uint32_t a)
{
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// The missing incoming links of a node on a Dirichlet edge: f_ij = D f*_{-i,-j}(x) + S_ij(x_b,
// t + dt/2), as in step_kernel; f holds the node's own opposite populations there.  g: the step's
// wall data or nullptr.
__device__ __forceinline__ void wall_links(const StepArgs& A, const double* g, int x, int y, bool le, bool ri, bool bot,
                                           bool top, double (&f)[4][5])
{
    if (!(le || ri || bot || top)) return;
    const int nx = A.nx, ny = A.ny;
    const double Dk[5] = {-1.0, -1.0, 1.0, 1.0, 1.0};
    double S[5];
    if (le) {
        double gx = 0.0, gy = 0.0;
        if (g) { gx = g[y]; gy = g[A.nwall + y]; }
        wall_source(1, 0, gx, gy, A.a, A.b, S);
#pragma unroll
        for (int k = 0; k < 5; ++k) f[0][k] = Dk[k] * f[0][k] + S[k];
    }
    if (ri) {
        double gx = 0.0, gy = 0.0;
        if (g) { gx = g[ny + y]; gy = g[A.nwall + ny + y]; }
        wall_source(-1, 0, gx, gy, A.a, A.b, S);
#pragma unroll
        for (int k = 0; k < 5; ++k) f[2][k] = Dk[k] * f[2][k] + S[k];
    }
    if (bot) {
        double gx = 0.0, gy = 0.0;
        if (g) { gx = g[2 * ny + x]; gy = g[A.nwall + 2 * ny + x]; }
        wall_source(0, 1, gx, gy, A.a, A.b, S);
#pragma unroll
        for (int k = 0; k < 5; ++k) f[1][k] = Dk[k] * f[1][k] + S[k];
    }
    if (top) {
        double gx = 0.0, gy = 0.0;
        if (g) { gx = g[2 * ny + nx + x]; gy = g[A.nwall + 2 * ny + nx + x]; }
        wall_source(0, -1, gx, gy, A.a, A.b, S);
#pragma unroll
        for (int k = 0; k < 5; ++k) f[3][k] = Dk[k] * f[3][k] + S[k];
    }
}

// grid: (ceil(nx / SA_THREADS), ceil(ny / rows)), block SA_THREADS; block (cb, r) computes
// the rows r * rows ... of column block cb, one after the other
template <bool DIRICHLET, bool TRACK, bool FORCE, unsigned long long SPLIT>
__global__ void __launch_bounds__(SA_THREADS, (SPLIT & kSplitFixed) ? LBM_SA_FX_MIN_BLOCKS : LBM_SA_MIN_BLOCKS)
    step_f64_staged_kernel(StepArgs A, int rows)
{
    __shared__ __align__(16) double slot[SA_SLOTS][SA_THREADS];
    __shared__ double coef[FORCE ? SA_THREADS / 32 : 1][32];   // per warp: body_coef of the row, [r][c]
    const int t = threadIdx.x;
    const int nx = A.nx, ny = A.ny;
    const int xg = blockIdx.x * SA_THREADS + t;
    const bool active = xg < nx;
    const int x = active ? xg : nx - 1;                // lanes past nx mirror column nx - 1
    const int y0 = blockIdx.y * rows;
    const int y1 = min(ny, y0 + rows);
    const long long plane = A.plane, pitch = A.pitch;
    const double* __restrict__ src = static_cast<const double*>(A.src);
    double* __restrict__ dst = static_cast<double*>(A.dst);
    const int xl = (x == 0) ? nx - 1 : x - 1, xr = (x == nx - 1) ? 0 : x + 1;
    const bool le = DIRICHLET && x == 0, ri = DIRICHLET && x == nx - 1;
    const uint32_t s0 = lbmt::smem_u32(&slot[0][t]);
    constexpr uint32_t SL = SA_THREADS * 8;            // bytes from one slot to the next

    // source of slot d * 5 + k: the population of direction d, component k that node (x, y)
    // pulls; on a Dirichlet edge the missing link's slot gets the node's own opposite population
    auto sources = [&](int y, const double* (&p)[4]) {
        const int ym = (y == 0) ? ny - 1 : y - 1, yp = (y == ny - 1) ? 0 : y + 1;
        const bool bot = DIRICHLET && y == 0, top = DIRICHLET && y == ny - 1;
        const long long r = (long long)y * pitch;
        p[0] = src + (le ? 10 * plane + r + x : r + xl);
        p[1] = src + (bot ? 15 * plane + r + x : 5 * plane + (long long)ym * pitch + x);
        p[2] = src + (ri ? r + x : 10 * plane + r + xr);
        p[3] = src + (top ? 5 * plane + r + x : 15 * plane + (long long)yp * pitch + x);
    };
    auto issue = [&](int y, uint32_t sb) {
        const double* p[4];
        sources(y, p);
#pragma unroll
        for (int k = 0; k < 5; ++k)
#pragma unroll
            for (int d = 0; d < 4; ++d) cp_async8(sb + (d * 5 + k) * SL, p[d] + k * plane);
    };

    const double hdt = 0.5 * A.dt;
    lbmt::grid_dependency_wait();
    // one commit group per row
    if (y0 < y1) issue(y0, s0);
    cp_async_commit();
    for (int y = y0; y < y1; ++y) {
        double hx = 0.0, hy = 0.0;
        if (FORCE) warp_body_load(A, A.T, hdt, coef[t >> 5], x, y, hx, hy);   // the row's copies are in flight
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        double f[4][5];
#pragma unroll
        for (int d = 0; d < 4; ++d)
#pragma unroll
            for (int k = 0; k < 5; ++k) f[d][k] = lds_f64(s0 + (d * 5 + k) * SL);
        // the slots have been read: the copies of row y + 1 may overwrite them
        __syncwarp();
        if (y + 1 < y1) issue(y + 1, s0);
        cp_async_commit();
        const long long off = (long long)y * pitch + x;
        double w0 = 0.0, w1 = 0.0;                     // loaded before the collision, not after it
        if (TRACK) {
            w0 = A.w[off];
            w1 = A.w[plane + off];
        }
        if (DIRICHLET) wall_links(A, A.g, x, y, le, ri, y == 0, y == ny - 1, f);
        double U[5], o[4][5];
        if constexpr (FORCE) collide_fixed_forced(f, hx, hy, A.a, A.b, U, o);
        else collide_split<SPLIT>(f, A.a, A.b, U, o);
        if (active) {
#pragma unroll
            for (int d = 0; d < 4; ++d)
#pragma unroll
                for (int k = 0; k < 5; ++k) dst[(d * 5 + k) * plane + off] = o[d][k];
            if (TRACK) {
                // u*(t+2dt) = u*(t+dt) + dt v(t+dt)  (steps 1(b) and 2(c) of the summary, Sec. 3.6)
                A.w[off] = fma(A.dt, U[0], w0);
                A.w[plane + off] = fma(A.dt, U[1], w1);
            }
        }
    }
    // no copy is left in flight: the group committed after the last row is empty
}

// ---------------------------------------------------------------------------
// Many steps of a small lattice in one cooperative launch (split level 12).
//
// A step of a lattice that fills the chip at most a few times over is bound by latency, not by
// bytes or pipes: launch and drain, the loads, one node's chain of about a thousand instructions,
// the stores.  Here every warp keeps one segment of 32 columns of a row (segments in row-major
// order) for all steps, and a step of a block waits only for the
// blocks within `reach` of it to have finished the step before: each block counts its finished
// steps in a flag of its own (release after the block's barrier) and warp 0 polls its neighbours'
// flags (acquire).  Having seen them also means that the neighbours no longer read what the block
// is about to overwrite (two buffers).  The body load is computed before the wait.  Loads bypass
// L1, which another SM's stores do not reach.  Same node arithmetic on the same inputs as the
// staged kernel, hence the same bits.
// Measured (us per step, one launch per step without programmatic launch before): 64^2 with body
// load and displacement tracking 6.2 -> 4.1, without 6.2 -> 3.3, 128^2 6.2 -> 3.4.
// Waits are bounded (two seconds of SM clock); one that runs out sets `timeout` and ends the block.
// ---------------------------------------------------------------------------
struct MultiArgs {
    StepArgs A;            // src: the state at entry, dst: the other buffer, T and g: the first step's rows
    int steps;
    int ntask, nseg;       // segments in all and per row
    int nblk, reach;       // blocks; neighbours on each side whose flags a step waits for
    unsigned int* flags;   // [nblk * MULTI_FLAG], zero at launch
    int* timeout;
    int withhold;          // test hook: the block whose flag never rises (-1: none)
};
constexpr int MULTI_WARPS = 4;
constexpr int MULTI_FLAG = 8;        // 32 bytes apart

__device__ __forceinline__ bool multi_wait(const unsigned int* flag, unsigned int want)
{
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v >= want) return true;
    const long long t0 = clock64();
    do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v >= want) return true;
    } while (clock64() - t0 < lbmt::kWaitCycles);
    return false;
}

template <bool DIRICHLET, bool TRACK, bool FORCE>
__global__ void __launch_bounds__(32 * MULTI_WARPS, LBM_SA_FX_MIN_BLOCKS) multi_f64_kernel(const MultiArgs Q)
{
    __shared__ double coef[MULTI_WARPS][32];
    __shared__ int quit;
    const StepArgs& A = Q.A;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nx = A.nx, ny = A.ny;
    const long long plane = A.plane, pitch = A.pitch;
    const int t = blockIdx.x * MULTI_WARPS + warp;
    const bool live = t < Q.ntask;                     // a warp without a segment only takes part in the barriers
    const int y = live ? t / Q.nseg : 0, xg = live ? (t - y * Q.nseg) * 32 + lane : 0;
    const int x = xg < nx ? xg : nx - 1;               // lanes past nx mirror column nx - 1
    const bool le = DIRICHLET && x == 0, ri = DIRICHLET && x == nx - 1;
    const bool bot = DIRICHLET && y == 0, top = DIRICHLET && y == ny - 1;
    const int xl = (x == 0) ? nx - 1 : x - 1, xr = (x == nx - 1) ? 0 : x + 1;
    const int ym = (y == 0) ? ny - 1 : y - 1, yp = (y == ny - 1) ? 0 : y + 1;
    const long long off = (long long)y * pitch + x;
    // the sources; on a Dirichlet edge the missing link gets the node's own opposite population
    const long long o0 = le ? 10 * plane + off : (long long)y * pitch + xl;
    const long long o1 = bot ? 15 * plane + off : 5 * plane + (long long)ym * pitch + x;
    const long long o2 = ri ? off : 10 * plane + (long long)y * pitch + xr;
    const long long o3 = top ? 5 * plane + off : 15 * plane + (long long)yp * pitch + x;
    const double hdt = 0.5 * A.dt;
    const double* src = static_cast<const double*>(A.src);
    double* dst = static_cast<double*>(A.dst);
    const double* T = A.T;
    const double* g = A.g;
    if (threadIdx.x == 0) quit = 0;
    for (int s = 0; s < Q.steps; ++s) {
        double hx = 0.0, hy = 0.0;
        if (FORCE && live) warp_body_load(A, T, hdt, coef[warp], x, y, hx, hy);
        if (s > 0 && warp == 0)
            for (int j = lane - Q.reach; j <= Q.reach; j += 32) {
                int b = (int)blockIdx.x + j;
                b = b < 0 ? b + Q.nblk : (b >= Q.nblk ? b - Q.nblk : b);
                if (!multi_wait(Q.flags + b * MULTI_FLAG, (unsigned)s)) quit = 1;
            }
        __syncthreads();
        if (quit) {
            if (threadIdx.x == 0) atomicExch(Q.timeout, 1);
            return;
        }
        if (live) {
            double f[4][5], w0 = 0.0, w1 = 0.0;
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                f[0][k] = __ldcg(src + o0 + k * plane);
                f[1][k] = __ldcg(src + o1 + k * plane);
                f[2][k] = __ldcg(src + o2 + k * plane);
                f[3][k] = __ldcg(src + o3 + k * plane);
            }
            if (TRACK) {
                w0 = A.w[off];
                w1 = A.w[plane + off];
            }
            if (DIRICHLET) wall_links(A, g, x, y, le, ri, bot, top, f);
            double U[5], o[4][5];
            if constexpr (FORCE) collide_fixed_forced(f, hx, hy, A.a, A.b, U, o);
            else collide_fixed(f, A.a, A.b, U, o);
            if (xg < nx) {
#pragma unroll
                for (int d = 0; d < 4; ++d)
#pragma unroll
                    for (int k = 0; k < 5; ++k) dst[(d * 5 + k) * plane + off] = o[d][k];
                if (TRACK) {
                    A.w[off] = fma(A.dt, U[0], w0);
                    A.w[plane + off] = fma(A.dt, U[1], w1);
                }
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && (int)blockIdx.x != Q.withhold) {
            __threadfence();
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(Q.flags + blockIdx.x * MULTI_FLAG),
                         "r"((unsigned)(s + 1))
                         : "memory");
        }
        double* n = const_cast<double*>(src);
        src = dst;
        dst = n;
        if (FORCE) T += 2 * A.R;
        if (g) g += 2 * A.nwall;
    }
}

}  // namespace lbmk
