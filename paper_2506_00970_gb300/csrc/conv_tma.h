// Forward convolutions of the proposal network's layers 2-6 and the data
// gradients of its layers 3-6 on tcgen05 with TMA-fed operands (conv_tma.cu).  Internal to the library.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace gs2d {
namespace net {

// out = bfloat16(ReLU(conv3x3_stride2_pad1(x, w) + bias)) for conv layer
// `layer` (0-based: 1 .. 5 = the network's layers 2-6): x NHWC [B][H][W][C_in] bfloat16, w [C_out][9 C_in] bfloat16
// (k = (ky * 3 + kx) C_in + c), bias [C_out] FP32, out NHWC [B][Ho][Wo][C_out];
// device pointers, 16-byte aligned.  A wait that runs out sets *err to 1.
// GS2D_ERR_CUDA if the tensor maps cannot be made (nothing is launched).
int conv_tma_forward(int layer, const __nv_bfloat16* x, int B, const __nv_bfloat16* w,
                     const float* bias, __nv_bfloat16* out, int* err, cudaStream_t st);

// out = bfloat16(the gradient of conv layer `layer` (2 .. 5) with respect to
// its input, zero where act <= 0): dz NHWC [B][Ho][Wo][C_out] bfloat16, w as
// above, act and out NHWC [B][H][W][C_in] bfloat16; pointers and errors as
// above.  Each parity class 2 py + px of the input pixels sums its products
// (over taps, then output channels) in pieces of steps[class] blocks of 64
// output channels, and the pieces in order.
struct DgradSplits {
  int steps[4];
};
int dgrad_tma(int layer, const __nv_bfloat16* dz, int B, const __nv_bfloat16* w,
              const __nv_bfloat16* act, __nv_bfloat16* out, const DgradSplits& splits, int* err,
              cudaStream_t st);

}  // namespace net
}  // namespace gs2d
