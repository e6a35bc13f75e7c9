// Learned warm-start network: shared declarations of the tensor-core
// convolution and the element-wise kernels (unet.cu) used by the network
// driver (unet_net.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace purify {

using bf16 = __nv_bfloat16;

struct ConvArgs {
    const bf16* in;          // NHWC, channel stride in_cs, first channel in_co
    int B, H, W, Cin, in_cs, in_co;
    const bf16* w;           // [k][k][Cinp / 8][Npad][8], zero padded
    int k, Cinp, Npad;
    const float* bias;       // [Cout] or null
    int Cout, relu;
    bf16* out;               // NHWC BF16 (channel stride out_cs, offset out_co) or null: output channels
    int out_cs, out_co;      // from bf_from on
    float* out_f32;          // NHWC FP32 [pixels][f32_ch] of the first f32_ch channels, or null
    const float* residual;   // added to out_f32 when not null ([pixels][f32_ch])
    int* err;                // set to 1 when a bounded wait gives up
    const bf16* mask;        // not null: `out` is zero where this activation (same pixels; channel
    int mask_cs, mask_co;    // stride, first channel) is not positive
    int f32_ch, bf_from;     // f32_ch 0: all channels
    int vec_out, vec_f32;    // set by the launch: `out` (and the mask), `out_f32` take 16-byte accesses
    int up;                  // 1: the input is the (H/2, W/2) image read through a x2 nearest upsampling
};

void conv_tc_launch(const ConvArgs& a, cudaStream_t st);
// weight gradient of a k x k convolution added to dW (channels in multiples of 8)
bool dw_tc_ok(int Cout, int Cin, int xcs, int xco);
void dw_tc_launch(const bf16* gz, int Cout, const bf16* x, int xcs, int xco, int Cin, int B, int H, int W, int up, int k,
                  float* dW, int* err, cudaStream_t st);
int round16(int v);
__global__ void k_f32_to_bf16(const float* __restrict__ x, bf16* __restrict__ y, int64_t n);
__global__ void k_pack_weights(const float* __restrict__ w, bf16* __restrict__ wp, int Cout, int k, int Cin, int Npad,
                               int Cinp);

}  // namespace purify
