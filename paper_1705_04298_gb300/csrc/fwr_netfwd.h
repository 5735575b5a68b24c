// Forward pass of the width-16 warm-start network in one kernel (fwr_netfwd.cu).
// Not installed.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace fwr {
namespace net {

typedef __nv_bfloat16 bf16;

constexpr float IN_SCALE = 0.5f;
constexpr int GRID = 128, LOW = 32, POOL = 4;

struct FwdArgs {
    const float* slopes;      // [F][2][n][n]
    const uint8_t* mask;      // [n][n]
    int n, off, F;
    const bf16* w_first;      // W[16][3][3][3]
    const bf16* w_out;        // W[2][16]
    const uint2* wp[14];      // packed weights of layers 1 .. 13 (k_pack_tc's order); [0] unused
    const float* bias[15];
    // outputs: any may be null
    float* ext;               // warm start [F][2][128][128]
    float* pred;              // [F][32][32][2]
    bf16* X;                  // network input [F][32][32][3]
    bf16* act[14];            // layer outputs (NHWC); all or none
    bf16* pool[3];            // pooled outputs of layers 1, 3, 5
};

constexpr int FUSED_WIDTH = 16;
cudaError_t unet_forward_prepare();
cudaError_t unet_forward(const FwdArgs& a, int sms, cudaStream_t s);

}  // namespace net
}  // namespace fwr
