// lf_sur_conv.cuh -- the surrogate's tensor-core convolution (lf_sur_conv.cu) as
// the network calls it (lf_sur.cu); lf_sur_conv3x3 of lf_sur.h is one plain call.
#pragma once

#include <cuda_bf16.h>

#include "lf_internal.cuh"

namespace lf {
namespace sur {

struct ConvArgs {
    const __nv_bfloat16* in;     // padded NHWC, CIN channels
    const __nv_bfloat16* w;      // [9][COUT][CIN], tap t = 3 (dy + 1) + (dx + 1)
    const float* bias;           // [COUT] or null
    const __nv_bfloat16* resid;  // padded NHWC COUT, added after the activation, or null
    const __nv_bfloat16* mask;   // padded NHWC COUT: out2 = out * (mask > 0), or null
    __nv_bfloat16* out;          // padded NHWC COUT, or null
    __nv_bfloat16* out2;         // padded NHWC COUT (masked copy of out), or null
    __nv_bfloat16* zout;         // padded NHWC COUT: pre-activation value, or null
    const float* x4;             // [B][NY][NX][4]: y4 = x4 + (acc + bias)[0..3], or null
    float* y4;
    float* raw;                  // [B][4][NY][NX]: y4 scale + offset in place of y4, or null
    float scale[4], offset[4];
    // training: one bit per pre-activation value, (value > 0), [B NY][4][NX]
    // 16-channel words of COUT = 64: written by the forward pass in place of
    // zout, read by the backward pass in place of mask
    uint16_t* zbits;
    const uint16_t* mbits;
    float* bsum;                 // [COUT] += sums over pixels of out2 (the next bias gradient), or null
    int relu;
    int B, NY, NX;
    int* err;
    // the weights are older than the kernel before this one on the stream (which
    // was itself started after they were written), so they may be read before
    // that kernel has finished
    int old_weights;
    int sectors;                 // set by conv3x3: out, out2, zout and resid are 32-byte aligned
};

// `mbits` selects the backward form: acc (+ resid) -> out (may be null) and out2 = out where the bit is set.
cudaError_t conv3x3(int cin, int cout, const ConvArgs& a, cudaStream_t s);

}  // namespace sur
}  // namespace lf
