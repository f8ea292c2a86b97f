// Internal interface of the tcgen05 3x3 convolution (nn_conv_tc.cu), called by
// the convolution entry point of nn_kernels.cu.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

struct ConvTcArgs {
    const float* x1;            // first input, C1 channels, [B][H][W][C1] (or [B][H/2][W/2][C1] with x1_half)
    const float* x2;            // second input (channels after x1), C2 channels, or null
    int C1, C2;                 // multiples of 32
    const uint16_t* w;          // BF16 weights [Cout][3][3][C1 + C2]
    const float* bias;          // [Cout] or null
    float* y1;                  // output channels [0, Co1)
    float* y2;                  // output channels [Co1, Cout), or null
    int Co1, Cout;              // Co1 a multiple of 16
    int B, H, W;                // powers of two
    int relu, beta, x1_half, act_bf16;
};

// Launches the tensor-core convolution when its tiling applies to these sizes and
// returns true; returns false (nothing launched) otherwise, and the caller uses
// another kernel.  `stages` = 0 picks the pipeline depth.
bool conv3_tc_launch(const ConvTcArgs& a, cudaStream_t s, int stages);

struct ConvTcWgradArgs {
    const float* dy;            // [B][H][W][Cout]
    const float* x1;            // as in ConvTcArgs
    const float* x2;
    int C1, C2, Cout;           // multiples of 32
    int B, H, W;                // H, W powers of two, at least 16
    int x1_half;
    float* partial;             // [ranges][parts][2][Cout][3][3][C1 + C2]
    int subs;                   // parts per range, set by the launch
};

// 3x3 weight gradient: ranges of 16 x 16 pixel blocks the work is split into and parts per range (two
// partial sums each), and the launch (false: the device refused the kernel's attributes)
struct ConvTcWgradSplit {
    int ranges, parts;
    int partials() const { return 2 * ranges * parts; }
};
ConvTcWgradSplit conv3_wgrad_tc_split(int Cin, int Cout, int B, int H, int W);
bool conv3_wgrad_tc_launch(ConvTcWgradArgs a, cudaStream_t s);

// Reads and clears the flag that a bounded wait inside the kernel ran out
// (the output of that launch is invalid); synchronises `s`.
bool conv3_tc_take_timeout(cudaStream_t s);

namespace lbmh {
// tensor map of BF16 weights [cout][3][3][cin]: box {16 input channels, box_co, 9 taps} with the
// 32-byte swizzle, defined in lbm_capi.cu
bool encode_conv3_weights_map(CUtensorMap* m, const void* w, int cin, int cout, int box_co);
}  // namespace lbmh
