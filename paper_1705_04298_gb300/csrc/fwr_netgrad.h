// Backward pass of the warm-start network (fwr_net.cu): kernels and launchers
// in fwr_netgrad.cu. Not installed.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>

namespace fwr {
namespace net {

typedef __nv_bfloat16 bf16;

// One 3 x 3 layer's backward: the channel concatenation of A (ca channels; at
// half resolution when upA) and B (cb, may be null) went in at H x H.
struct ConvBwd {
    int ca, cb, cout, H;
    bool upA;
    const bf16 *A, *B;
    bool simt;  // FP32 pipe only
};

// dW, db of a 3 x 3 layer into g (flat: W[cout][3][3][cin], then the biases),
// from dZ [Bn][H][H][cout]; ws: wgrad_ws_floats() of workspace.
cudaError_t conv_wgrad(const ConvBwd& L, const float* dZ, int Bn, float* ws, float* g, int sms, cudaStream_t s);
size_t wgrad_ws_floats(int cin, int cout, int H, int sms);

// Input gradient of a 3 x 3 layer with weights Wt. Without concatenation
// (lo = nullptr): dIn [Bn][H][H][ca], zeroed where act (the layer's input,
// null: no mask) is not positive. With it: the A part is summed over the 2 x 2
// pixels that read each half-resolution one into lo [Bn][H/2][H/2][ca] (zeroed
// where lo_act is not positive), the B part goes to dIn [Bn][H][H][cb].
cudaError_t conv_dgrad(const ConvBwd& L, const float* dZ, const bf16* Wt, int Bn, const bf16* act, float* dIn,
                       float* lo, const bf16* lo_act, int sms, cudaStream_t s);

// Tensor-core forms of the two (fwr_netgradtc.cu), which conv_wgrad and
// conv_dgrad take for layers whose channel counts are multiples of 16 (weight
// gradients also for fewer than 16 input channels); wgrad_tc leaves the sums of *chunks parts in ws.
bool wgrad_tc_shape(int ca, int cb, int cout);
bool dgrad_tc_shape(int ca, int cb, int cout);
bool grad_tc_fits(int cin, int cout, int H);
size_t wgrad_tc_ws_floats(int cin, int cout, int H, int sms);
bool wgrad_tc_fits(const ConvBwd& L, const float* dZ);
cudaError_t wgrad_tc(const ConvBwd& L, const float* dZ, int Bn, float* ws, int* chunks, int sms, cudaStream_t s);
bool dgrad_tc_fits(const ConvBwd& L, const float* dZ, const bf16* Wt);
cudaError_t dgrad_tc(const ConvBwd& L, const float* dZ, const bf16* Wt, int Bn, const bf16* act, float* dIn,
                     float* lo, const bf16* lo_act, int sms, cudaStream_t s);

// Masked mean squared error of pred against T and the backward of the 1 x 1
// output layer (C input channels a, two outputs): dIn [npix][C] (zeroed where
// a is not positive), g = W[2][C], b[2] gradients, *loss.
cudaError_t out_backward(const float* pred, const float* T, const float* LM, const unsigned* cnt, int npix, int C,
                         const bf16* a, const bf16* Wt, float* dIn, float* ws, float* g, float* loss, int sms,
                         cudaStream_t s);
size_t out_ws_floats(int C, int sms);

// whether the kernels above can run a layer (shared memory)
bool netgrad_fits(int ca, int cb, int cout, int H);

}  // namespace net
}  // namespace fwr
