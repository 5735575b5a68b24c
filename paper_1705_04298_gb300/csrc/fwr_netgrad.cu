// Backward pass of the warm-start network's convolutions (sm_103a).
//
// Weight gradients and input gradients are contractions with one FP32 operand
// (the activations' gradients stay FP32; weights and activations are BF16).
// Layers whose channel counts are multiples of 16 (and the first layer, three
// input channels) take the tensor-core kernels of fwr_netgradtc.cu; those of
// other widths run here on the FP32 pipe, with the packed two-lane FMA
// (fma.rn.f32x2, half the issue slots of scalar FMA at the same lane rate),
// which bounds them. Each thread keeps a register tile whose
// operands come from shared memory in 16-byte loads, few loads per FMA.
// Measured on 256 images at width 16, the whole gradient call: 90.6 ms with
// scalar kernels (one block per output channel and tap, operands from global
// memory), 2.5 ms with these, 0.96 ms with the tensor cores'.

#include <stdint.h>

#include <algorithm>

#include "fwr_internal.h"
#include "fwr_netgrad.h"

namespace fwr {
namespace net {

namespace {

typedef unsigned long long u64;

__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 dup2(float a) {
    u64 d;
    asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(a));
    return d;
}
__device__ __forceinline__ float2 un2(u64 a) {
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(a));
    return v;
}
__device__ __forceinline__ bool positive(bf16 a) { return __bfloat162float(a) > 0.f; }

constexpr int THREADS = 256;
// shared memory of a weight-gradient CTA: two fit an SM
constexpr size_t WGRAD_SMEM = 108 * 1024;

// ------------------------------------------------------------ weight gradient
//
// dW[co][dy][dx][ci] = sum over pixels dZ[p][co] in[p + (dy - 1, dx - 1)][ci].
// A thread owns 8 output channels x 4 input channels x the 3 taps of one
// kernel row: 96 sums, fed per pixel by two 16-byte loads of dZ and one of the
// input (the three columns of the window slide along the row in registers). The
// CTA's thread tiles cover one range of outputs (blockIdx.y) S times over, the
// S copies on different image rows; it stages RS rows of dZ and of the input
// (with halo, widened to FP32) at a time. The copies are summed through shared
// memory and every CTA (a chunk of rows) writes its sums to ws; k_reduce adds
// the chunks in order, so the result does not depend on timing.

// i / d for 0 <= i < 2^16 and 1 <= d < 2^16 as one multiply
struct FastDiv {
    unsigned d, m;
};
FastDiv fast_div(int d) { return FastDiv{unsigned(d), unsigned(((1ull << 32) + d - 1) / d)}; }
__device__ __forceinline__ int div_by(int i, FastDiv f) { return f.d == 1u ? i : int(__umulhi(unsigned(i), f.m)); }

struct WgradShape {
    FastDiv by_ncib, by_q;
    int cin4, cout8, ncib, ncob, T, ny, TG, S, threads, RS, zrow, irow;
    size_t smem;
};

WgradShape wgrad_shape(int cin, int cout, int H) {
    WgradShape w;
    w.cin4 = (cin + 3) / 4 * 4;
    w.cout8 = (cout + 7) / 8 * 8;
    w.ncib = w.cin4 / 4;
    w.ncob = w.cout8 / 8;
    w.by_ncib = fast_div(w.ncib);
    w.by_q = fast_div(std::max(1, H * cout / 4));
    w.T = w.ncib * w.ncob * 3;
    w.ny = (w.T + THREADS - 1) / THREADS;
    w.TG = (w.T + w.ny - 1) / w.ny;
    w.S = THREADS / w.TG;
    w.threads = (w.TG * w.S + 31) / 32 * 32;
    // rows 8 floats apart beyond their data: the S copies read different banks
    w.zrow = H * w.cout8 + 8;
    w.irow = (H + 2) * w.cin4 + 8;
    auto bytes = [&](int rs) { return (size_t(rs) * w.zrow + size_t(rs + 2) * w.irow) * sizeof(float); };
    int rs = w.S;
    while (rs > 1 && bytes(rs) > WGRAD_SMEM) --rs;
    while (rs % w.S == 0 && bytes(rs + w.S) <= WGRAD_SMEM) rs += w.S;
    w.RS = rs;
    const size_t red = size_t(w.S / 2) * w.TG * 97 * sizeof(float);
    w.smem = std::max(bytes(rs), red);
    return w;
}

// chunks of image rows (one CTA each): two CTAs per SM, whole turns of the
// copies where there is more than one. (A few images do not fill the copies of
// one CTA; they are spread all the same: one image of width 3, 12 x 32 x 32, 29
// us in one CTA, 7 in 32.)
int wgrad_rows(const WgradShape& w, long long rows, int sms) {
    const long long want = std::max(1, 2 * sms / w.ny);
    long long r = (rows + want - 1) / want;
    const int unit = w.S < w.RS ? w.S : w.RS;
    if (r > unit) r = (r + unit - 1) / unit * unit;
    return int(r);
}

template <int H>
__global__ void __launch_bounds__(THREADS)
k_wgrad3(const float* __restrict__ dZ, int cout, const bf16* __restrict__ A, int ca, int upA,
         const bf16* __restrict__ Bt, int cb, int rows, int rows_cta, WgradShape w, float* __restrict__ ws) {
    extern __shared__ __align__(16) float sm[];
    float* const zs = sm;                      // [RS][H][cout8]
    float* const is = sm + size_t(w.RS) * w.zrow;  // [RS + 2][H + 2][cin4]
    constexpr int W = H;
    const int cin = ca + cb;
    const int tid = threadIdx.x;
    const int s = tid / w.TG, t = blockIdx.y * w.TG + tid % w.TG;
    const bool active = s < w.S && t < w.T;
    const int cib = t % w.ncib, cob = (t / w.ncib) % w.ncob, dy = t / (w.ncib * w.ncob);
    const bool biased = active && cib == 0 && dy == 1;
    u64 acc[3][4][4];  // [dx][pair of output channels][input channel]
    u64 bacc[4];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[d][a][b] = 0ull;
#pragma unroll
    for (int a = 0; a < 4; ++a) bacc[a] = 0ull;

    const int r_begin = blockIdx.x * rows_cta, r_end = min(rows, r_begin + rows_cta);
    for (int r0 = r_begin; r0 < r_end; r0 += w.RS) {
        const int nr = min(w.RS, r_end - r0);
        __syncthreads();
        // dZ rows (contiguous in memory)
        if ((cout & 7) == 0) {
            const int q = W * cout / 4;
#pragma unroll 4
            for (int i = tid; i < nr * q; i += blockDim.x) {
                const int r = div_by(i, w.by_q), c = i - r * q;
                reinterpret_cast<float4*>(zs + r * w.zrow)[c] =
                    __ldg(reinterpret_cast<const float4*>(dZ + size_t(r0 + r) * W * cout) + c);
            }
        } else {
            for (int i = tid; i < nr * W * w.cout8; i += blockDim.x) {
                const int c = i % w.cout8, x = (i / w.cout8) % W, r = i / (w.cout8 * W);
                zs[r * w.zrow + x * w.cout8 + c] = c < cout ? dZ[(size_t(r0 + r) * W + x) * cout + c] : 0.f;
            }
        }
        // input rows r0 - 1 .. r0 + nr, one zero column on each side
        const bool vec = (ca & 3) == 0 && (cb & 3) == 0;
#pragma unroll 4
        for (int i = tid; i < (nr + 2) * (W + 2) * w.ncib; i += blockDim.x) {
            const int q = div_by(i, w.by_ncib), c = (i - q * w.ncib) * 4, xx = q % (W + 2), r = q / (W + 2);
            const int gr = r0 - 1 + r, x = xx - 1;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gr >= 0 && gr < rows && x >= 0 && x < W) {
                size_t pa = size_t(gr) * W + x;
                if (upA) {
                    const int b = gr / H, y = gr - b * H;
                    pa = (size_t(b) * (H / 2) + y / 2) * (W / 2) + x / 2;
                }
                const size_t pb = size_t(gr) * W + x;
                if (vec) {
                    const bf16* src = c < ca ? A + pa * ca + c : Bt + pb * cb + (c - ca);
                    const uint2 u = __ldg(reinterpret_cast<const uint2*>(src));
                    v = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u),
                                    __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
                } else {
                    float e[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int cc = c + k;
                        e[k] = cc >= cin ? 0.f
                               : cc < ca ? __bfloat162float(A[pa * ca + cc])
                                         : __bfloat162float(Bt[pb * cb + (cc - ca)]);
                    }
                    v = make_float4(e[0], e[1], e[2], e[3]);
                }
            }
            *reinterpret_cast<float4*>(is + r * w.irow + xx * w.cin4 + c) = v;
        }
        __syncthreads();
        if (!active) continue;
        for (int row = s; row < nr; row += w.S) {
            const int y = (r0 + row) % H, yy = y + dy - 1;
            if (yy < 0 || yy >= H) continue;
            const float* zp = zs + row * w.zrow + 4 * cob;
            const float* ip = is + (row + dy) * w.irow + 4 * cib;
            u64 w0[4], w1[4];
            {
                const float4 a = *reinterpret_cast<const float4*>(ip);
                const float4 b = *reinterpret_cast<const float4*>(ip + w.cin4);
                w0[0] = dup2(a.x), w0[1] = dup2(a.y), w0[2] = dup2(a.z), w0[3] = dup2(a.w);
                w1[0] = dup2(b.x), w1[1] = dup2(b.y), w1[2] = dup2(b.z), w1[3] = dup2(b.w);
            }
            ip += 2 * w.cin4;
#pragma unroll 4
            for (int x = 0; x < W; ++x) {
                const float4 c = *reinterpret_cast<const float4*>(ip);
                const ulonglong2 z0 = *reinterpret_cast<const ulonglong2*>(zp);
                const ulonglong2 z1 = *reinterpret_cast<const ulonglong2*>(zp + 4 * w.ncob);
                ip += w.cin4;
                zp += w.cout8;
                const u64 z[4] = {z0.x, z0.y, z1.x, z1.y};
                const u64 w2[4] = {dup2(c.x), dup2(c.y), dup2(c.z), dup2(c.w)};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        acc[0][a][b] = fma2(z[a], w0[b], acc[0][a][b]);
                        acc[1][a][b] = fma2(z[a], w1[b], acc[1][a][b]);
                        acc[2][a][b] = fma2(z[a], w2[b], acc[2][a][b]);
                    }
                if (biased) {
#pragma unroll
                    for (int a = 0; a < 4; ++a) bacc[a] = add2(bacc[a], z[a]);
                }
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    w0[b] = w1[b];
                    w1[b] = w2[b];
                }
            }
        }
    }
    // sum the copies (those that had a row), pairwise halves, one kernel column at a time
    const int tl = tid % w.TG, copies = min(w.S, rows_cta);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        for (int n = copies; n > 1; n = (n + 1) / 2) {
            const int half = (n + 1) / 2;
            u64* const red = reinterpret_cast<u64*>(sm);  // [copy][tile][21]
            __syncthreads();
            if (active && s >= half && s < n) {
                u64* o = red + (size_t(s - half) * w.TG + tl) * 21;
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) o[4 * a + b] = acc[d][a][b];
                if (d == 0) {
#pragma unroll
                    for (int a = 0; a < 4; ++a) o[16 + a] = bacc[a];
                }
            }
            __syncthreads();
            if (active && s + half < n) {
                const u64* o = red + (size_t(s) * w.TG + tl) * 21;
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) acc[d][a][b] = add2(acc[d][a][b], o[4 * a + b]);
                if (d == 0) {
#pragma unroll
                    for (int a = 0; a < 4; ++a) bacc[a] = add2(bacc[a], o[16 + a]);
                }
            }
        }
    }
    if (!active || s != 0) return;
    const int nw = cout * 9 * cin;
    float* const o = ws + size_t(blockIdx.x) * (nw + cout);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int co = 4 * cob + (a < 2 ? 0 : 4 * w.ncob) + 2 * (a & 1);
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float2 v = un2(acc[d][a][b]);
                const int ci = 4 * cib + b;
                if (ci < cin) {
                    if (co < cout) o[(co * 9 + dy * 3 + d) * cin + ci] = v.x;
                    if (co + 1 < cout) o[((co + 1) * 9 + dy * 3 + d) * cin + ci] = v.y;
                }
            }
        if (biased) {
            const float2 v = un2(bacc[a]);
            if (co < cout) o[nw + co] = v.x;
            if (co + 1 < cout) o[nw + co + 1] = v.y;
        }
    }
}

// g[i] = sum over chunks of ws[chunk][i]; the last of `n` sums goes to *last
// when given. 32 sums x LANES chunk lanes per block, four of a lane's loads in
// flight together: 32 lanes where there are few sums (2320 sums of 304 chunks:
// 5 us, 8 with 8 lanes), 8 where the blocks fill the chip (36928 sums of 147:
// 7.5 us, 12 with 32).
template <int LANES>
__global__ void __launch_bounds__(32 * LANES)
k_reduce(const float* __restrict__ ws, int chunks, int n, float* g, float* last) {
    __shared__ float part[LANES][33];
    const int c = threadIdx.x & 31, q = threadIdx.x >> 5, i = blockIdx.x * 32 + c;
    float u[4] = {0.f, 0.f, 0.f, 0.f};
    if (i < n) {
        for (int k = q; k < chunks; k += 4 * LANES)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (k + LANES * j < chunks) u[j] += ws[size_t(k + LANES * j) * n + i];
    }
    part[q][c] = (u[0] + u[1]) + (u[2] + u[3]);
    __syncthreads();
#pragma unroll
    for (int h = LANES / 2; h > 0; h /= 2) {
        if (q < h) part[q][c] += part[q + h][c];
        __syncthreads();
    }
    if (q == 0 && i < n) {
        if (last && i == n - 1) *last = part[0][c];
        else g[i] = part[0][c];
    }
}
cudaError_t reduce_chunks(const float* ws, int chunks, int n, float* g, float* last, int sms, cudaStream_t s) {
    const int blocks = (n + 31) / 32;
    if (blocks < 2 * sms) k_reduce<32><<<blocks, 1024, 0, s>>>(ws, chunks, n, g, last);
    else k_reduce<8><<<blocks, 256, 0, s>>>(ws, chunks, n, g, last);
    return cudaGetLastError();
}

// ------------------------------------------------------------- input gradient
//
// dIn[y][x][ci] = sum over (co, dy, dx) dZ[y - dy + 1][x - dx + 1][co] W[co][dy][dx][ci].
// A thread owns 2 x 4 pixels x 8 input channels (64 sums); per output channel
// it reads the 4 x 6 window of dZ and the 9 x 8 weights: 30 shared-memory loads
// for 288 packed FMAs. The 2 x 4 tile holds whole 2 x 2 blocks, so the
// upsampled half of a concatenated input is summed to half resolution in
// registers. A CTA covers `tiles` of them (whole row pairs) x 8 cb input
// channels and stages 16 output channels of dZ (channel-major rows with zero
// halo) and of the weights (widened to FP32) at a time.

constexpr int DG_CO = 16;
constexpr size_t DGRAD_SMEM = 100 * 1024;

struct DgradShape {
    int cb, ny, pairs, S, threads, slots, portion;  // portion: row pairs per image part
    int block;  // threads of the launch: those beyond `threads` stage only
    size_t smem;
};

DgradShape dgrad_shape(int cin, int H, long long total_pairs, int sms) {
    DgradShape d;
    const int blk = (cin + 7) / 8;
    d.ny = (blk + 7) / 8;
    d.cb = (blk + d.ny - 1) / d.ny;
    const int per_pair = H / 4;  // tiles of a row pair
    const int img = H / 2;
    auto slots = [&](int pairs) {
        const int portion = pairs < img ? pairs : img;
        return pairs / portion * (2 * portion + 2);
    };
    auto bytes = [&](int pairs) {
        return (size_t(slots(pairs)) * DG_CO * (H + 8) + size_t(DG_CO) * 9 * 8 * d.cb) * sizeof(float);
    };
    // 128 to 254 threads (several CTAs fit an SM's registers) unless dZ's rows
    // would leave room for one CTA only (few channels on the smallest images)
    d.pairs = 1;
    while (d.cb * per_pair * d.pairs < 128 && bytes(2 * d.pairs) <= DGRAD_SMEM) d.pairs *= 2;
    // the small images' layers have few tiles: fewer per CTA, each shared by S
    // threads over the output channels, until there are two CTAs per SM (256
    // images of 8 x 8 and 64 channels: 161 us with S = 1, 64 with 4)
    d.S = 1;
    while (d.S < 8 && (total_pairs + d.pairs - 1) / d.pairs * d.ny < 2 * sms) {
        if (d.pairs > 1) d.pairs /= 2;
        else if (2 * d.S * d.cb * per_pair > THREADS) break;
        d.S *= 2;
    }
    d.portion = d.pairs < img ? d.pairs : img;
    d.slots = slots(d.pairs);
    d.threads = d.cb * per_pair * d.pairs * d.S;
    // CTAs that have an SM each get a few more warps for the staging
    d.block = (total_pairs + d.pairs - 1) / d.pairs * d.ny <= sms ? std::max(d.threads, 128) : d.threads;
    d.smem = std::max(bytes(d.pairs), size_t(d.threads / 2) * 33 * sizeof(u64));
    return d;
}

template <int H>
__global__ void __launch_bounds__(THREADS)
k_dgrad3(const float* __restrict__ dZ, int cout, const bf16* __restrict__ Wt, int ca, int cb2, int total_pairs,
         DgradShape d, const bf16* __restrict__ act, float* __restrict__ dIn, float* __restrict__ lo,
         const bf16* __restrict__ lo_act) {
    extern __shared__ __align__(16) float sm[];
    constexpr int W = H, ZS = W + 8;
    const int cin = ca + cb2, n8 = 8 * d.cb;
    float* const zs = sm;                                     // [slots][DG_CO][ZS], column x at 4 + x
    float* const wsm = sm + size_t(d.slots) * DG_CO * ZS;     // [DG_CO][9][n8]
    constexpr int img = H / 2;
    const int tid = threadIdx.x, tt = d.threads / d.S, sp = tid / tt, tl = tid - sp * tt;
    const int cib = tl % d.cb, tile = tl / d.cb;
    const int xt = tile % (W / 4), pr = tile / (W / 4);       // tile column, row pair in the CTA
    const int pair0 = blockIdx.x * d.pairs, ci0 = blockIdx.y * n8;
    const int part = pr / d.portion, slot0 = part * (2 * d.portion + 2) + 2 * (pr - part * d.portion);
    u64 acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;

    // the zero columns of every staged row
    for (int i = tid; i < d.slots * DG_CO * 2; i += blockDim.x) zs[(i >> 1) * ZS + ((i & 1) ? W + 4 : 3)] = 0.f;
    for (int c0 = 0; c0 < cout; c0 += DG_CO) {
        const int nc = min(DG_CO, cout - c0);
        __syncthreads();
#pragma unroll 4
        for (int i = tid; i < d.slots * (DG_CO / 4) * W; i += blockDim.x) {
            const int x = i % W, c4 = (i / W) % (DG_CO / 4), slot = i / (W * (DG_CO / 4));
            const int p = slot / (2 * d.portion + 2), j = slot - p * (2 * d.portion + 2);
            const int gp = pair0 + p * d.portion;             // first row pair of this part
            const int b = gp / img, y = 2 * (gp - b * img) - 1 + j;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gp < total_pairs && y >= 0 && y < H) {
                const float* src = dZ + ((size_t(b) * H + y) * W + x) * cout + c0 + 4 * c4;
                if ((cout & 3) == 0) {
                    if (4 * c4 < nc) v = __ldg(reinterpret_cast<const float4*>(src));
                } else {
                    if (4 * c4 < nc) v.x = src[0];
                    if (4 * c4 + 1 < nc) v.y = src[1];
                    if (4 * c4 + 2 < nc) v.z = src[2];
                    if (4 * c4 + 3 < nc) v.w = src[3];
                }
            }
            float* o = zs + (slot * DG_CO + 4 * c4) * ZS + 4 + x;
            o[0] = v.x;
            o[ZS] = v.y;
            o[2 * ZS] = v.z;
            o[3 * ZS] = v.w;
        }
        // weight rows (output channel, tap): two rows per warp at a time, 16 lanes
        // each; several loads in flight, along the row where it is long, over the
        // rows where it is short
        const bf16* const wsrc = Wt + size_t(c0) * 9 * cin + ci0;
        if (n8 > 32) {
            for (int ct = tid >> 4; ct < nc * 9; ct += blockDim.x >> 4)
#pragma unroll 4
                for (int c = tid & 15; c < n8; c += 16)
                    wsm[ct * n8 + c] = ci0 + c < cin ? __bfloat162float(wsrc[size_t(ct) * cin + c]) : 0.f;
        } else {
            for (int c = tid & 15; c < n8; c += 16)
#pragma unroll 8
                for (int ct = tid >> 4; ct < nc * 9; ct += blockDim.x >> 4)
                    wsm[ct * n8 + c] = ci0 + c < cin ? __bfloat162float(wsrc[size_t(ct) * cin + c]) : 0.f;
        }
        __syncthreads();
        const float* zp = zs + (slot0 * DG_CO + sp) * ZS + 4 + 4 * xt;
        const float* wp = wsm + sp * 9 * n8 + 4 * cib;
#pragma unroll 1
        for (int co = sp < d.S ? sp : nc; co < nc; co += d.S, zp += d.S * ZS, wp += d.S * 9 * n8) {
            u64 z[4][6];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float* q = zp + r * DG_CO * ZS;
                const float4 m = *reinterpret_cast<const float4*>(q);
                z[r][0] = dup2(q[-1]);
                z[r][1] = dup2(m.x);
                z[r][2] = dup2(m.y);
                z[r][3] = dup2(m.z);
                z[r][4] = dup2(m.w);
                z[r][5] = dup2(q[4]);
            }
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int dy = tap / 3, dx = tap % 3;
                const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(wp + tap * n8);
                const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(wp + tap * n8 + 4 * d.cb);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const u64 zz = z[(i >> 2) - dy + 2][(i & 3) - dx + 2];
                    acc[i][0] = fma2(zz, a.x, acc[i][0]);
                    acc[i][1] = fma2(zz, a.y, acc[i][1]);
                    acc[i][2] = fma2(zz, b.x, acc[i][2]);
                    acc[i][3] = fma2(zz, b.y, acc[i][3]);
                }
            }
        }
    }
    // sum the S copies, pairwise halves
    for (int n = d.S; n > 1; n /= 2) {
        u64* const red = reinterpret_cast<u64*>(sm);  // [copy][tile][33]
        __syncthreads();
        if (sp >= n / 2 && sp < n) {
            u64* o = red + size_t((sp - n / 2) * tt + tl) * 33;
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) o[4 * i + j] = acc[i][j];
        }
        __syncthreads();
        if (sp < n / 2) {
            const u64* o = red + size_t(sp * tt + tl) * 33;
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = add2(acc[i][j], o[4 * i + j]);
        }
    }
    const int gp = pair0 + pr;
    if (sp != 0 || gp >= total_pairs) return;
    const int b = gp / img, y0 = 2 * (gp - b * img), x0 = 4 * xt;
    const bool vec = (cin & 3) == 0 && (ca & 3) == 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int ci = ci0 + 4 * cib + 4 * d.cb * h;  // four adjacent input channels
        if (ci >= cin) continue;
        float v[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 p = un2(acc[i][2 * h]), q = un2(acc[i][2 * h + 1]);
            v[i][0] = p.x;
            v[i][1] = p.y;
            v[i][2] = q.x;
            v[i][3] = q.y;
        }
        const int nch = lo ? cb2 : cin;  // channels of dIn
        if (vec) {
            if (lo && ci < ca) {
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const size_t o = ((size_t(b) * (H / 2) + y0 / 2) * (W / 2) + x0 / 2 + k) * ca + ci;
                    const uint2 m = __ldg(reinterpret_cast<const uint2*>(lo_act + o));
                    const bf16* mb = reinterpret_cast<const bf16*>(&m);
                    float s[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        s[e] = positive(mb[e]) ? ((v[2 * k][e] + v[2 * k + 1][e]) + v[4 + 2 * k][e]) + v[5 + 2 * k][e]
                                               : 0.f;
                    *reinterpret_cast<float4*>(lo + o) = make_float4(s[0], s[1], s[2], s[3]);
                }
            } else {
                const int c = lo ? ci - ca : ci;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const size_t o = ((size_t(b) * H + y0 + (i >> 2)) * W + x0 + (i & 3)) * nch + c;
                    if (act) {
                        const uint2 m = __ldg(reinterpret_cast<const uint2*>(act + o));
                        const bf16* mb = reinterpret_cast<const bf16*>(&m);
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (!positive(mb[e])) v[i][e] = 0.f;
                    }
                    *reinterpret_cast<float4*>(dIn + o) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
                }
            }
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int cc = ci + e;
                if (cc >= cin) break;
                if (lo && cc < ca) {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const size_t o = ((size_t(b) * (H / 2) + y0 / 2) * (W / 2) + x0 / 2 + k) * ca + cc;
                        lo[o] = positive(lo_act[o])
                                    ? ((v[2 * k][e] + v[2 * k + 1][e]) + v[4 + 2 * k][e]) + v[5 + 2 * k][e]
                                    : 0.f;
                    }
                } else {
                    const int c = lo ? cc - ca : cc;
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const size_t o = ((size_t(b) * H + y0 + (i >> 2)) * W + x0 + (i & 3)) * nch + c;
                        dIn[o] = act && !positive(act[o]) ? 0.f : v[i][e];
                    }
                }
            }
        }
    }
}

// ------------------------------------------------------------ loss, 1 x 1 layer
//
// One pass over the pixels: the masked error, its gradient, the output layer's
// input gradient (written) and weight gradient (summed per thread over a
// channel, then over the CTA). Sums per CTA go to ws[cta] = W[2][C], b[2], loss.
__global__ void __launch_bounds__(256)
k_out_bwd(const float2* __restrict__ pred, const float2* __restrict__ T, const float* __restrict__ LM,
          const unsigned* __restrict__ cnt, int npix, int pix_cta, int C, const bf16* __restrict__ a,
          const bf16* __restrict__ Wt, float* __restrict__ dIn, float* __restrict__ ws) {
    __shared__ float red[5][256];
    const int parts = 256 / C, c = threadIdx.x % C, part = threadIdx.x / C;
    // the reciprocal of the count with what its rounding leaves out: alone it is
    // one relative error of every gradient, and adds to the tensor cores'
    // truncation where their signs agree (3 and 6 images: 9.1e-8 and 8.9e-8 of a
    // layer's gradient, 6.9e-8 and 6.6e-8 so; scalar FP32 sums 8.2e-8 and 9.3e-8).
    // (A division per gradient: 256 images 964 -> 972 us.)
    const float norm = fmaxf(1.f, 2.f * float(*cnt)), inv = 1.f / norm, rest = fmaf(-inv, norm, 1.f) / norm;
    auto over_norm = [&](float e) {  // (an infinite error stays one)
        return fmaf(e, inv, fminf(fmaxf(e, -3e38f), 3e38f) * rest);
    };
    const float w0 = __bfloat162float(Wt[c]), w1 = __bfloat162float(Wt[C + c]);
    float s0 = 0.f, s1 = 0.f, b0 = 0.f, b1 = 0.f, l = 0.f;
    const int p_end = min(npix, int(blockIdx.x + 1) * pix_cta);
    if (part < parts) {
#pragma unroll 4
        for (int p = blockIdx.x * pix_cta + part; p < p_end; p += parts) {
            const float m = LM[p];
            const float2 q = pred[p], t = T[p];
            const float d0 = (q.x - t.x) * m, d1 = (q.y - t.y) * m;
            const float g0 = over_norm(2.f * d0), g1 = over_norm(2.f * d1);
            const bf16 av = a[size_t(p) * C + c];
            const float v = __bfloat162float(av);
            s0 += g0 * v;
            s1 += g1 * v;
            b0 += g0;
            b1 += g1;
            l += (d0 * d0 + d1 * d1) * inv;
            dIn[size_t(p) * C + c] = v > 0.f ? fmaf(w1, g1, w0 * g0) : 0.f;
        }
    }
    red[0][threadIdx.x] = s0;
    red[1][threadIdx.x] = s1;
    red[2][threadIdx.x] = b0;
    red[3][threadIdx.x] = b1;
    red[4][threadIdx.x] = l;
    __syncthreads();
    // thread i < 2 C + 3: one of the CTA's sums
    const int i = threadIdx.x;
    if (i < 2 * C + 3) {
        const int row = i < 2 * C ? i / C : i - 2 * C + 2, col = i < 2 * C ? i % C : 0;
        float v = 0.f;
        for (int q = 0; q < parts; ++q) v += red[row][q * C + col];
        ws[size_t(blockIdx.x) * (2 * C + 3) + i] = v;
    }
}

int out_ctas(int sms) { return 4 * sms; }

}  // namespace

size_t wgrad_ws_floats(int cin, int cout, int H, int sms) {
    const WgradShape w = wgrad_shape(cin, cout, H);
    const size_t n = size_t(std::max(1, 2 * sms / w.ny)) * (size_t(cout) * 9 * cin + cout);
    return (cin % 16 == 0 || cin < 16) && cout % 16 == 0 ? std::max(n, wgrad_tc_ws_floats(cin, cout, H, sms)) : n;
}

cudaError_t conv_wgrad(const ConvBwd& L, const float* dZ, int Bn, float* ws, float* g, int sms, cudaStream_t s) {
    const int cin = L.ca + L.cb, rows = Bn * L.H, n = L.cout * 9 * cin + L.cout;
    if (wgrad_tc_fits(L, dZ)) {
        int chunks = 0;
        const cudaError_t e = wgrad_tc(L, dZ, Bn, ws, &chunks, sms, s);
        return e == cudaSuccess ? reduce_chunks(ws, chunks, n, g, nullptr, sms, s) : e;
    }
    const WgradShape w = wgrad_shape(cin, L.cout, L.H);
    const int rc = wgrad_rows(w, rows, sms), chunks = (rows + rc - 1) / rc;
    auto kern = L.H == 32 ? k_wgrad3<32> : L.H == 16 ? k_wgrad3<16> : L.H == 8 ? k_wgrad3<8> : k_wgrad3<4>;
    // limits are raised at the launches: a network that is never trained loads
    // no kernel of the backward pass
    const cudaError_t e = raise_smem_limit(kern, w.smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(chunks, w.ny), w.threads, w.smem, s>>>(dZ, L.cout, L.A, L.ca, L.upA ? 1 : 0, L.B, L.cb, rows, rc, w,
                                                       ws);
    return reduce_chunks(ws, chunks, n, g, nullptr, sms, s);
}

cudaError_t conv_dgrad(const ConvBwd& L, const float* dZ, const bf16* Wt, int Bn, const bf16* act, float* dIn,
                       float* lo, const bf16* lo_act, int sms, cudaStream_t s) {
    if (dgrad_tc_fits(L, dZ, Wt)) return dgrad_tc(L, dZ, Wt, Bn, act, dIn, lo, lo_act, sms, s);
    const int pairs = Bn * (L.H / 2);
    const DgradShape d = dgrad_shape(L.ca + L.cb, L.H, pairs, sms);
    auto kern = L.H == 32 ? k_dgrad3<32> : L.H == 16 ? k_dgrad3<16> : L.H == 8 ? k_dgrad3<8> : k_dgrad3<4>;
    const cudaError_t e = raise_smem_limit(kern, d.smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3((pairs + d.pairs - 1) / d.pairs, d.ny), d.block, d.smem, s>>>(dZ, L.cout, Wt, L.ca, L.cb, pairs, d,
                                                                               act, dIn, lo, lo_act);
    return cudaGetLastError();
}

size_t out_ws_floats(int C, int sms) { return size_t(out_ctas(sms)) * (2 * C + 3); }

cudaError_t out_backward(const float* pred, const float* T, const float* LM, const unsigned* cnt, int npix, int C,
                         const bf16* a, const bf16* Wt, float* dIn, float* ws, float* g, float* loss, int sms,
                         cudaStream_t s) {
    const int ctas = out_ctas(sms), per = (npix + ctas - 1) / ctas, used = (npix + per - 1) / per;
    k_out_bwd<<<used, 256, 0, s>>>(reinterpret_cast<const float2*>(pred), reinterpret_cast<const float2*>(T), LM, cnt,
                                   npix, per, C, a, Wt, dIn, ws);
    const int n = 2 * C + 3;
    return reduce_chunks(ws, used, n, g, loss, sms, s);
}

bool netgrad_fits(int ca, int cb, int cout, int H) {
    const int cin = ca + cb;
    if (H != 32 && H != 16 && H != 8 && H != 4) return false;
    if ((wgrad_tc_shape(ca, cb, cout) || dgrad_tc_shape(ca, cb, cout)) && !grad_tc_fits(cin, cout, H)) return false;
    return std::max(wgrad_shape(cin, cout, H).smem, dgrad_shape(cin, H, 1ll << 40, 1).smem) <= size_t(227) * 1024;
}

}  // namespace net
}  // namespace fwr
