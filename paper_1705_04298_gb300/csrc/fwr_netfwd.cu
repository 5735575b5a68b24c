// Forward pass of the width-16 warm-start network (definition: fwr_net.cu) in
// one kernel (sm_103a): a CTA takes an image through all 15 layers with every
// activation in shared memory.
//
// The layered path reads and writes each activation through L2 (0.9 MB per
// image with halos, for 38 M multiply-adds) and pays 21 launches; here HBM sees
// the slopes and the prediction (or the warm start), and L2 the packed weights
// (0.6 MB per image). What bounds it is the mma.sync rate and its operand
// loads. Every output is the same bits as the layered path's: each sum runs
// over the same operands in the same order (taps, then channels in chunks of
// 16; first and last layer in FP32 FMA chains).
//
// Layout: activations are [pixel][channel] BF16, the 16-byte chunks of a pixel
// permuted by its index so that ldmatrix (8 pixels x one chunk) and the
// epilogue's stores hit all banks; taps outside the image read a zero chunk.
// 256 threads; the lifetimes are packed into 106 KB, so two CTAs share an SM
// and one's barriers and epilogues overlap the other's products.
// Measured, 1000 images and the warm start written: 1040 us layer by layer, 320 us.

#include "fwr_netfwd.h"

#include <algorithm>

namespace fwr {
namespace net {

namespace {

constexpr int NT = 256;
constexpr int KB = 1024;
// byte offsets of the activations (see the order of the layers in the kernel)
constexpr int R0 = 0, R1 = 32 * KB, S2 = 64 * KB, S3 = 80 * KB, A11 = 88 * KB, ZERO = 104 * KB, WF = ZERO + 128,
              WO = WF + 27 * 16 * 4, BF = WO + 32 * 4, SMEM = BF + 32 * 4;
constexpr int P1 = R0, A2 = R0 + 8 * KB, P2 = R0, A4 = R0 + 4 * KB, P3 = R0 + 24 * KB, A6 = R0 + 26 * KB,
              A7 = R0 + 28 * KB, A8 = R0, A9 = R0 + 8 * KB, A10 = R0 + 16 * KB, A12 = R0, A13 = R1;
static_assert(34 * 34 * 3 * 4 <= 16 * KB, "the input plane fits the space of layer 11's output");

// permutation of a pixel's 16-byte chunks (2, 4 or 8 of them: C channels)
template <int C> __device__ __forceinline__ int perm(int p) {
    constexpr int n = C / 8;
    return n == 2 ? (p >> 2) & 1 : n == 4 ? (p >> 1) & 3 : p & 7;
}
// byte offset of chunk c of pixel p
template <int C> __device__ __forceinline__ uint32_t chunk_at(int p, int c) {
    return uint32_t(p * C * 2 + ((c ^ perm<C>(p)) << 4));
}

__device__ __forceinline__ void ldsm_x4(uint32_t (&a)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(addr));
}
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// One 3 x 3 layer at H x H: input channels [A (CA, at half resolution when UP) |
// B (CB)], COUT outputs, ReLU. WN warps across the output channels, 8 / WN across
// the pixels. src*, dst: byte offsets of the activations in shared memory. Starts
// with the barrier that completes its input.
template <int H, int CA, bool UP, int CB, int COUT, int WN>
__device__ __forceinline__ void conv(unsigned char* sm, int srcA, int srcB, int dst, const uint2* __restrict__ wp,
                                     const float* __restrict__ bias, bf16* __restrict__ save) {
    constexpr int WM = 8 / WN, MTT = H * H / 16, NTT = COUT / 8, CH = (CA + CB) / 16;
    constexpr int MT = MTT / WM, NTW = NTT / WN;
    static_assert(MT * WM == MTT && NTW * WN == NTT, "warps cover the layer");
    // taps whose weights are loaded together, where the registers allow it (they
    // come from L2: 1000 images 370 us a tap at a time, 320 with this and without
    // a second warp on the same pixels at 16 x 16)
    constexpr int TG = 3 * CH * NTW * 2 + MT * NTW * 4 <= 100 ? 3 : 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = warp / WN, wn = warp % WN;
    const uint2* w = wp + (wn * NTW) * 32 + lane;
    __syncthreads();
    {
        const uint32_t base = uint32_t(__cvta_generic_to_shared(sm));
        const int kh = lane >> 4;  // which 16-byte half of a 16-channel chunk
        const int p0 = wm * MT * 16 + (lane & 15);
        float acc[MT][NTW][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int t = 0; t < NTW; ++t) acc[m][t][0] = acc[m][t][1] = acc[m][t][2] = acc[m][t][3] = 0.f;
#pragma unroll 1
        for (int t0 = 0; t0 < 9; t0 += TG) {
            uint2 b[TG][CH][NTW];
#pragma unroll
            for (int i = 0; i < TG * CH; ++i)
#pragma unroll
                for (int t = 0; t < NTW; ++t) b[i / CH][i % CH][t] = __ldg(w + (i * NTT + t) * 32);
            w += TG * CH * NTT * 32;
#pragma unroll
            for (int g = 0; g < TG; ++g) {
                const int dy = t0 / 3 - 1, dx = TG == 3 ? g - 1 : t0 - (t0 / 3) * 3 - 1;
                // this lane's pixel of tile m is p0 + 16 m; a tap's chunk permutation
                // is the same for all tiles where the rows hold whole tiles' low bits
                const int x0 = p0 % H + dx, y0 = p0 / H + dy;
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    const int x = x0 + (16 * m) % H, y = y0 + (16 * m) / H;
                    const bool in = y >= 0 && y < H && x >= 0 && x < H;
                    const int pa = UP ? (y >> 1) * (H / 2) + (x >> 1) : y * H + x, pb = y * H + x;
                    const uint32_t am = base + (in ? uint32_t(srcA + pa * CA * 2) : uint32_t(ZERO));
                    const uint32_t bm = base + (in ? uint32_t(srcB + pb * CB * 2) : uint32_t(ZERO));
                    const int sa = perm<CA>(pa), sb = perm<CB ? CB : 16>(pb);
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        uint32_t a[4];
                        if (16 * c < CA) ldsm_x4(a, am + (((2 * c + kh) ^ sa) << 4));
                        else ldsm_x4(a, bm + (((2 * c - CA / 8 + kh) ^ sb) << 4));
#pragma unroll
                        for (int t = 0; t < NTW; ++t) mma_16816(acc[m][t], a, b[g][c][t]);
                    }
                }
            }
        }
        const int g = lane >> 2, q = lane & 3;
#pragma unroll
        for (int t = 0; t < NTW; ++t) {
            const int nt = wn * NTW + t, co = nt * 8 + 2 * q;
            const float b0 = bias[co], b1 = bias[co + 1];
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int p = (wm * MT + m) * 16 + g + 8 * h;
                    const __nv_bfloat162 v = __floats2bfloat162_rn(fmaxf(acc[m][t][2 * h] + b0, 0.f),
                                                                   fmaxf(acc[m][t][2 * h + 1] + b1, 0.f));
                    *reinterpret_cast<__nv_bfloat162*>(sm + dst + chunk_at<COUT>(p, nt) + 4 * q) = v;
                    if (save) *reinterpret_cast<__nv_bfloat162*>(save + size_t(p) * COUT + co) = v;
                }
        }
    }
}

// 2 x 2 average pooling of an H x H x C activation; starts with a barrier
template <int H, int C>
__device__ __forceinline__ void pool(unsigned char* sm, int src, int dst, bf16* __restrict__ save) {
    constexpr int Ho = H / 2;
    __syncthreads();
    for (int i = threadIdx.x; i < Ho * Ho * (C / 8); i += NT) {
        const int c = i % (C / 8), p = i / (C / 8), y = p / Ho, x = p % Ho;
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int ps = (2 * y + (a >> 1)) * H + 2 * x + (a & 1);
            const uint4 v = *reinterpret_cast<const uint4*>(sm + src + chunk_at<C>(ps, c));
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                s[2 * k] += __uint_as_float(u[k] << 16);
                s[2 * k + 1] += __uint_as_float(u[k] & 0xFFFF0000u);
            }
        }
        __nv_bfloat162 o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = __floats2bfloat162_rn(0.25f * s[2 * k], 0.25f * s[2 * k + 1]);
        const uint4 v = *reinterpret_cast<uint4*>(o);
        *reinterpret_cast<uint4*>(sm + dst + chunk_at<C>(p, c)) = v;
        if (save) *reinterpret_cast<uint4*>(save + size_t(p) * C + 8 * c) = v;
    }
}

__global__ void __launch_bounds__(NT, 2) k_unet_forward(const __grid_constant__ FwdArgs a) {
    extern __shared__ __align__(128) unsigned char sm[];
    const int tid = threadIdx.x;
    float* const wf = reinterpret_cast<float*>(sm + WF);  // first layer: [tap][cin][cout]
    float* const wo = reinterpret_cast<float*>(sm + WO);  // output layer: [cout][cin]
    float* const bf = reinterpret_cast<float*>(sm + BF);  // their biases: 16, 2
    float* const xp = reinterpret_cast<float*>(sm + A11); // input [3][34][34], zero border
    for (int i = tid; i < 27 * 16; i += NT) wf[i] = __bfloat162float(a.w_first[(i % 16) * 27 + i / 16]);
    if (tid < 32) wo[tid] = __bfloat162float(a.w_out[tid]);
    if (tid < 16) bf[tid] = a.bias[0][tid];
    if (tid < 2) bf[16 + tid] = a.bias[14][tid];
    if (tid < 32) reinterpret_cast<uint32_t*>(sm + ZERO)[tid] = 0u;
    const int n = a.n, nn = n * n;
    for (int f = blockIdx.x; f < a.F; f += gridDim.x) {
        auto at = [&](bf16* p, int per) { return p ? p + size_t(f) * per : nullptr; };
        __syncthreads();
        // input: 4 x 4 block means of the measured slopes and the pupil
        for (int i = tid; i < 3 * 34 * 34; i += NT) {
            const int x = i % 34, y = (i / 34) % 34;
            if (x == 0 || x == 33 || y == 0 || y == 33) xp[i] = 0.f;
        }
        const float* s = a.slopes + size_t(f) * 2 * nn;
        for (int p = tid; p < LOW * LOW; p += NT) {
            const int Y = p / LOW, X = p % LOW;
            float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
            for (int i = 0; i < POOL; ++i)
#pragma unroll
                for (int j = 0; j < POOL; ++j) {
                    const int bi = POOL * Y + i - a.off, bj = POOL * X + j - a.off;
                    if (bi >= 0 && bi < n && bj >= 0 && bj < n && a.mask[bi * n + bj]) {
                        a0 += s[bi * n + bj];
                        a1 += s[nn + bi * n + bj];
                        a2 += 1.f;
                    }
                }
            const float k = 1.f / (POOL * POOL);
            const bf16 v0 = __float2bfloat16(a0 * IN_SCALE * k), v1 = __float2bfloat16(a1 * IN_SCALE * k),
                       v2 = __float2bfloat16(a2 * k);
            float* const o = xp + (Y + 1) * 34 + X + 1;
            o[0] = __bfloat162float(v0);
            o[34 * 34] = __bfloat162float(v1);
            o[2 * 34 * 34] = __bfloat162float(v2);
            if (a.X) {
                bf16* const g = a.X + (size_t(f) * LOW * LOW + p) * 3;
                g[0] = v0;
                g[1] = v1;
                g[2] = v2;
            }
        }
        __syncthreads();
        // layer 0: a thread takes 4 adjacent pixels of a row, all 16 channels
        {
            const int y = tid / 8, x0 = (tid % 8) * 4;
            float acc[4][16];
#pragma unroll
            for (int g = 0; g < 4; ++g)
#pragma unroll
                for (int c = 0; c < 16; ++c) acc[g][c] = bf[c];
#pragma unroll 1
            for (int dy = 0; dy < 3; ++dy) {
                float v[3][6];
#pragma unroll
                for (int c = 0; c < 3; ++c)
#pragma unroll
                    for (int i = 0; i < 6; ++i) v[c][i] = xp[c * 34 * 34 + (y + dy) * 34 + x0 + i];
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                    for (int c = 0; c < 3; ++c)
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const float4 w = *reinterpret_cast<const float4*>(wf + ((dy * 3 + dx) * 3 + c) * 16 + 4 * q);
#pragma unroll
                            for (int g = 0; g < 4; ++g) {
                                acc[g][4 * q] = fmaf(w.x, v[c][g + dx], acc[g][4 * q]);
                                acc[g][4 * q + 1] = fmaf(w.y, v[c][g + dx], acc[g][4 * q + 1]);
                                acc[g][4 * q + 2] = fmaf(w.z, v[c][g + dx], acc[g][4 * q + 2]);
                                acc[g][4 * q + 3] = fmaf(w.w, v[c][g + dx], acc[g][4 * q + 3]);
                            }
                        }
            }
            bf16* const save = at(a.act[0], LOW * LOW * 16);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const int p = y * LOW + x0 + g;
                __nv_bfloat162 o[8];
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    o[c] = __floats2bfloat162_rn(fmaxf(acc[g][2 * c], 0.f), fmaxf(acc[g][2 * c + 1], 0.f));
                const uint4 lo = reinterpret_cast<uint4*>(o)[0], hi = reinterpret_cast<uint4*>(o)[1];
                *reinterpret_cast<uint4*>(sm + R0 + chunk_at<16>(p, 0)) = lo;
                *reinterpret_cast<uint4*>(sm + R0 + chunk_at<16>(p, 1)) = hi;
                if (save) {
                    reinterpret_cast<uint4*>(save + size_t(p) * 16)[0] = lo;
                    reinterpret_cast<uint4*>(save + size_t(p) * 16)[1] = hi;
                }
            }
        }
        conv<32, 16, false, 0, 16, 1>(sm, R0, 0, R1, a.wp[1], a.bias[1], at(a.act[1], 1024 * 16));
        pool<32, 16>(sm, R1, P1, at(a.pool[0], 256 * 16));
        conv<16, 16, false, 0, 32, 1>(sm, P1, 0, A2, a.wp[2], a.bias[2], at(a.act[2], 256 * 32));
        conv<16, 32, false, 0, 32, 1>(sm, A2, 0, S2, a.wp[3], a.bias[3], at(a.act[3], 256 * 32));
        pool<16, 32>(sm, S2, P2, at(a.pool[1], 64 * 32));
        conv<8, 32, false, 0, 64, 4>(sm, P2, 0, A4, a.wp[4], a.bias[4], at(a.act[4], 64 * 64));
        conv<8, 64, false, 0, 64, 4>(sm, A4, 0, S3, a.wp[5], a.bias[5], at(a.act[5], 64 * 64));
        pool<8, 64>(sm, S3, P3, at(a.pool[2], 16 * 64));
        conv<4, 64, false, 0, 64, 8>(sm, P3, 0, A6, a.wp[6], a.bias[6], at(a.act[6], 16 * 64));
        conv<4, 64, false, 0, 64, 8>(sm, A6, 0, A7, a.wp[7], a.bias[7], at(a.act[7], 16 * 64));
        conv<8, 64, true, 64, 64, 4>(sm, A7, S3, A8, a.wp[8], a.bias[8], at(a.act[8], 64 * 64));
        conv<8, 64, false, 0, 64, 4>(sm, A8, 0, A9, a.wp[9], a.bias[9], at(a.act[9], 64 * 64));
        conv<16, 64, true, 32, 32, 1>(sm, A9, S2, A10, a.wp[10], a.bias[10], at(a.act[10], 256 * 32));
        conv<16, 32, false, 0, 32, 1>(sm, A10, 0, A11, a.wp[11], a.bias[11], at(a.act[11], 256 * 32));
        conv<32, 32, true, 16, 16, 1>(sm, A11, R1, A12, a.wp[12], a.bias[12], at(a.act[12], 1024 * 16));
        conv<32, 16, false, 0, 16, 1>(sm, A12, 0, A13, a.wp[13], a.bias[13], at(a.act[13], 1024 * 16));
        // output layer; the warm start repeats it over 4 x 4 blocks
        __syncthreads();
        for (int p = tid; p < LOW * LOW; p += NT) {
            const uint4 c0 = *reinterpret_cast<const uint4*>(sm + A13 + chunk_at<16>(p, 0));
            const uint4 c1 = *reinterpret_cast<const uint4*>(sm + A13 + chunk_at<16>(p, 1));
            const uint32_t u[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
            float o0 = bf[16], o1 = bf[17];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const float lo = __uint_as_float(u[k] << 16), hi = __uint_as_float(u[k] & 0xFFFF0000u);
                o0 = fmaf(wo[2 * k], lo, o0);
                o1 = fmaf(wo[16 + 2 * k], lo, o1);
                o0 = fmaf(wo[2 * k + 1], hi, o0);
                o1 = fmaf(wo[16 + 2 * k + 1], hi, o1);
            }
            if (a.pred) reinterpret_cast<float2*>(a.pred)[size_t(f) * LOW * LOW + p] = make_float2(o0, o1);
            if (a.ext) {
                const float e0 = o0 * (1.f / IN_SCALE), e1 = o1 * (1.f / IN_SCALE);
                const int Y = p / LOW, X = p % LOW;
                float* const e = a.ext + size_t(f) * 2 * GRID * GRID + size_t(POOL * Y) * GRID + POOL * X;
#pragma unroll
                for (int i = 0; i < POOL; ++i) {
                    *reinterpret_cast<float4*>(e + i * GRID) = make_float4(e0, e0, e0, e0);
                    *reinterpret_cast<float4*>(e + GRID * GRID + i * GRID) = make_float4(e1, e1, e1, e1);
                }
            }
        }
    }
}

}  // namespace

cudaError_t unet_forward_prepare() {
    return cudaFuncSetAttribute(k_unet_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
}

cudaError_t unet_forward(const FwdArgs& a, int sms, cudaStream_t s) {
    k_unet_forward<<<std::min(a.F, 2 * sms), NT, SMEM, s>>>(a);
    return cudaGetLastError();
}

}  // namespace net
}  // namespace fwr
