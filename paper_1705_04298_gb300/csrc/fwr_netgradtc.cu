// Tensor-core weight and input gradients of the warm-start network's 3 x 3
// layers whose channel counts are multiples of 16 (sm_103a); the first layer's
// three input channels are padded.
//
// One operand of each contraction is FP32 (the activations' gradient dZ), the
// other BF16 (activations or weights). dZ is split exactly into three BF16
// values (its 24 significand bits, eight each, by truncation), so the products
// of mma.sync are exact; a 16-deep sum of all three splits is formed from zero
// on the tensor cores and added to the FP32 sums kept in registers, so no long
// sum is accumulated with the tensor cores' rounding. The FP32-FMA kernels
// (fwr_netgrad.cu) serve all other channel counts.
//
// Why: a layer's gradients are 2 to 7 GFLOP for 256 images, three times that
// in split products, which the tensor pipe (about 590 TFLOP/s for mma.sync)
// does in 10 to 36 us and the FP32 pipe (78 TFLOP/s) in 30 to 90. Measured
// against the FP32-FMA kernels, 256 images at width 16 (us, weight / input
// gradient): 48 -> 16 channels at 32 x 32: 51 / 45 against 153 / 113; 96 -> 32
// at 16 x 16: 47 / 44 against 210 / 120; 64 -> 64 at 8 x 8: 27 / 25 against
// 62 / 57; 128 -> 128 at 4 x 4: 27 / 33 against 66 / 85; the whole gradient
// call 2234 -> 1057 us (1004 with the first layer padded, chunk sums and pool
// gradients by wider kernels; 961 with the weight gradient's input rows copied
// asynchronously). Error against 64-bit sums: input gradient 0.75 to 1.0
// of the FP32-FMA kernel's, weight gradient 0.7 to 1.0 of it (and 1.0 to 1.2
// for a few images, where both are below 1e-7).

#include <stdint.h>

#include <algorithm>

#include "fwr_internal.h"
#include "fwr_netgrad.h"

namespace fwr {
namespace net {

namespace {

constexpr size_t TC_SMEM = 108 * 1024;  // two CTAs per SM

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// acc += A B over 16 of the contraction, A = a[0] + a[1] + a[2], largest
// first: the parts are summed from zero, the smallest first
__device__ __forceinline__ void mma3(float (&acc)[4], const uint32_t (&a)[3][4], uint32_t b0, uint32_t b1) {
    float t[4] = {0.f, 0.f, 0.f, 0.f};
    mma(t, a[2], b0, b1);
    mma(t, a[1], b0, b1);
    mma(t, a[0], b0, b1);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] += t[i];
}

// asynchronous 16-byte copy global -> shared; zeros when !ok (src is not read)
__device__ __forceinline__ void cp16(void* dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// the three BF16 parts of x and y, packed (x in the lower half); an infinity
// stays in the first part
__device__ __forceinline__ void split2(float x, float y, uint32_t (&p)[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint32_t ux = __float_as_uint(x), uy = __float_as_uint(y);
        p[k] = __byte_perm(ux, uy, 0x7632);
        if (k < 2) {
            x = (ux & 0x7FFFFFFFu) == 0x7F800000u ? 0.f : x - __uint_as_float(ux & 0xFFFF0000u);
            y = (uy & 0x7FFFFFFFu) == 0x7F800000u ? 0.f : y - __uint_as_float(uy & 0xFFFF0000u);
        }
    }
}
// four values at `dst` of each plane
__device__ __forceinline__ void store_split(unsigned char* dst, size_t plane, float4 v) {
    uint32_t a[3], b[3];
    split2(v.x, v.y, a);
    split2(v.z, v.w, b);
#pragma unroll
    for (int k = 0; k < 3; ++k) *reinterpret_cast<uint2*>(dst + k * plane) = make_uint2(a[k], b[k]);
}

__device__ __forceinline__ bool pos_lo(uint32_t v) { return __uint_as_float(v << 16) > 0.f; }
__device__ __forceinline__ bool pos_hi(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u) > 0.f; }

// i / d for 0 <= i < 2^16 and 1 <= d < 2^16 as one multiply
struct FastDiv {
    unsigned d, m;
};
FastDiv fast_div(int d) { return FastDiv{unsigned(d), unsigned(((1ull << 32) + d - 1) / d)}; }
__device__ __forceinline__ int div_by(int i, FastDiv f) { return f.d == 1u ? i : int(__umulhi(unsigned(i), f.m)); }

// ------------------------------------------------------------ weight gradient
//
// dW[co][tap][ci] = sum over pixels: A = dZ^T (16 output channels x 16 pixels),
// B = the input at the shifted pixels (16 pixels x 16 input channels), both
// transposed out of pixel-major shared memory by ldmatrix. A warp owns 16
// output x 16 input channels x 9 taps (72 sums a thread): per 16 pixels three
// loads of dZ and nine of the input for 54 MMAs. A CTA's mt x nt warp tiles
// cover one block of outputs (blockIdx.y) S times over, the S copies on
// different pixels; each CTA of blockIdx.x takes a range of image rows, RS at
// a time. Pixels outside the image are read from zeros. What bounds it: the
// tensor pipe and staging (dZ is split in the CTA).
struct WgTc {
    int ncin, nt, mt, S, ny, threads, pin, pz, RS, unit;  // pin, pz: bytes of a pixel
    FastDiv by_in, by_z;
    size_t smem, zoff;
};

WgTc wg_tc(int cin, int cout, int H) {
    WgTc w;
    w.ncin = (cin + 15) / 16;
    const int ncout = cout / 16;
    w.nt = 1;
    for (int d = 2; d <= 8; ++d)
        if (w.ncin % d == 0) w.nt = d;
    w.mt = 1;
    for (int d = 2; d <= 8 / w.nt; ++d)
        if (ncout % d == 0) w.mt = d;
    w.S = 8 / (w.nt * w.mt);
    w.ny = (w.ncin / w.nt) * (ncout / w.mt);
    w.threads = 32 * w.nt * w.mt * w.S;
    // pixels an odd number of 16 bytes apart: eight of them are conflict free
    w.pin = 32 * w.nt + 16;
    w.pz = 32 * w.mt + 16;
    w.by_in = fast_div(2 * w.nt);
    w.by_z = fast_div(4 * w.mt);
    w.unit = H < 16 ? 16 / H : 1;
    const int step = std::max(w.unit, w.S * 16 / H);  // every copy has pixels
    auto bytes = [&](int rs) {
        return size_t(3 * w.pin) + size_t(rs + 2) * (H + 2) * w.pin + size_t(3) * rs * H * w.pz;
    };
    w.RS = step;
    while (bytes(w.RS + step) <= TC_SMEM) w.RS += step;
    w.zoff = size_t(3 * w.pin) + size_t(w.RS + 2) * (H + 2) * w.pin;
    w.smem = std::max(bytes(w.RS), size_t((w.S + 1) / 2) * w.nt * w.mt * 76 * 32 * sizeof(float));
    return w;
}

int wg_tc_rows(const WgTc& w, long long rows, int sms) {
    const long long want = std::max(1, 2 * sms / w.ny);
    long long r = (rows + want - 1) / want;
    return int((r + w.unit - 1) / w.unit * w.unit);
}

template <int H>
__global__ void __launch_bounds__(256, 2)
k_wgrad_tc(const float* __restrict__ dZ, int cout, const bf16* __restrict__ A, int ca, int upA,
           const bf16* __restrict__ Bt, int cb, int rows, int rows_cta, WgTc w, float* __restrict__ ws) {
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int W = H;
    const int cin = ca + cb, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tiles = w.nt * w.mt, s = warp / tiles, tile = warp - s * tiles, tm = tile / w.nt, ti = tile - tm * w.nt;
    const int cgs = w.ncin / w.nt, cg = blockIdx.y % cgs, mg = blockIdx.y / cgs;
    const int c0 = cg * w.nt * 16, m0 = mg * w.mt * 16;
    unsigned char* const in = sm + 3 * w.pin;
    unsigned char* const zp = sm + w.zoff;
    const int plane = w.RS * W * w.pz, rpitch = (W + 2) * w.pin;
    const bool biased = cg == 0 && ti == 0;
    float acc[9][2][4], bias[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[t][b][k] = 0.f;
    for (int i = tid; i < 3 * w.pin / 16; i += blockDim.x) reinterpret_cast<uint4*>(sm)[i] = make_uint4(0, 0, 0, 0);
    // ldmatrix roles: pixel of the 16 and byte offset of the 8 channels
    const int pb = ((lane >> 3) & 1) * 8 + (lane & 7), ob = (ti * 16 + (lane >> 4) * 8) * 2;
    const int pa = (lane >> 4) * 8 + (lane & 7), oa = (tm * 16 + ((lane >> 3) & 1) * 8) * 2;
    const uint32_t zero_a = smem_u32(sm) + ob, in_a = smem_u32(in) + ob, z_a = smem_u32(zp) + oa;

    const int r_begin = blockIdx.x * rows_cta, r_end = min(rows, r_begin + rows_cta);
    for (int r0 = r_begin; r0 < r_end; r0 += w.RS) {
        const int nr = min(w.RS, r_end - r0);
        __syncthreads();
        // input rows r0 - 1 .. r0 + nr, one zero column on each side
#pragma unroll 4
        for (int i = tid; i < (nr + 2) * (W + 2) * 2 * w.nt; i += blockDim.x) {
            const int q = div_by(i, w.by_in), v = i - q * 2 * w.nt, xx = q % (W + 2), r = q / (W + 2);
            const int gr = r0 - 1 + r, x = xx - 1, c = c0 + 8 * v;
            const bool ok = gr >= 0 && gr < rows && x >= 0 && x < W;
            unsigned char* const dst = in + q * w.pin + 16 * v;
            size_t p = ok ? size_t(gr) * W + x : 0;
            if (cin < 16) {  // the rest of the 16 channels is zero
                const uint16_t* a = reinterpret_cast<const uint16_t*>(A) + p * cin;
                uint16_t e[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) e[k] = ok && c + k < cin ? __ldg(a + c + k) : uint16_t(0);
                *reinterpret_cast<uint4*>(dst) = make_uint4(e[0] | uint32_t(e[1]) << 16, e[2] | uint32_t(e[3]) << 16,
                                                            e[4] | uint32_t(e[5]) << 16, e[6] | uint32_t(e[7]) << 16);
            } else if (c < ca) {
                if (upA) {
                    const int b = gr / H, y = gr - b * H;
                    p = ok ? (size_t(b) * (H / 2) + y / 2) * (W / 2) + x / 2 : 0;
                }
                cp16(dst, A + p * ca + c, ok);
            } else {
                cp16(dst, Bt + p * cb + (c - ca), ok);
            }
        }
#pragma unroll 4
        for (int i = tid; i < nr * W * 4 * w.mt; i += blockDim.x) {
            const int q = div_by(i, w.by_z), c = i - q * 4 * w.mt;
            const float4 v = __ldg(reinterpret_cast<const float4*>(dZ + (size_t(r0) * W + q) * cout + m0) + c);
            store_split(zp + q * w.pz + 8 * c, plane, v);
        }
        cp_wait();
        __syncthreads();
        for (int ch = s; ch < nr * W / 16; ch += w.S) {
            uint32_t a[3][4];
#pragma unroll
            for (int k = 0; k < 3; ++k) ldsm4t(a[k], z_a + k * plane + (ch * 16 + pa) * w.pz);
            const int px = ch * 16 + pb, row = px / W, x = px % W, y = (r0 + row) % H;
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const bool ok = y + dy >= 1 && y + dy <= H;
                const uint32_t ad = ok ? in_a + (row + dy) * rpitch + x * w.pin : zero_a;
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    uint32_t b[4];
                    ldsm4t(b, ad + dx * w.pin);
                    mma3(acc[3 * dy + dx][0], a, b[0], b[1]);
                    mma3(acc[3 * dy + dx][1], a, b[2], b[3]);
                }
            }
            if (biased) mma3(bias, a, 0x3F803F80u, 0x3F803F80u);  // times one
        }
    }
    // sum the S copies, pairwise halves
    float* const red = reinterpret_cast<float*>(sm);  // [copy][tile][76][32]
    for (int n = w.S; n > 1; n = (n + 1) / 2) {
        const int half = (n + 1) / 2;
        __syncthreads();
        if (s >= half && s < n) {
            float* o = red + size_t((s - half) * tiles + tile) * 76 * 32 + lane;
#pragma unroll
            for (int i = 0; i < 72; ++i) o[32 * i] = acc[i / 8][(i / 4) & 1][i & 3];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[32 * (72 + k)] = bias[k];
        }
        __syncthreads();
        if (s + half < n) {
            const float* o = red + size_t(s * tiles + tile) * 76 * 32 + lane;
#pragma unroll
            for (int i = 0; i < 72; ++i) acc[i / 8][(i / 4) & 1][i & 3] += o[32 * i];
#pragma unroll
            for (int k = 0; k < 4; ++k) bias[k] += o[32 * (72 + k)];
        }
    }
    if (s != 0) return;
    const int nw = cout * 9 * cin, g = lane >> 2, t2 = 2 * (lane & 3);
    float* const o = ws + size_t(blockIdx.x) * (nw + cout);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int co = m0 + tm * 16 + g + 8 * h;
#pragma unroll
        for (int t = 0; t < 9; ++t)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int ci = c0 + ti * 16 + 8 * b + t2;
                float* q = o + (co * 9 + t) * cin + ci;
                if (cin >= 16) {
                    *reinterpret_cast<float2*>(q) = make_float2(acc[t][b][2 * h], acc[t][b][2 * h + 1]);
                } else {
                    if (ci < cin) q[0] = acc[t][b][2 * h];
                    if (ci + 1 < cin) q[1] = acc[t][b][2 * h + 1];
                }
            }
        if (biased && t2 == 0) o[nw + co] = bias[2 * h];
    }
}

// ------------------------------------------------------------- input gradient
//
// dIn[p][ci] = sum over (tap, co) dZ[p - tap][co] W[co][tap][ci]: A = dZ (16
// pixels x 16 output channels, the three parts), B = W (16 output x 8 input
// channels). A warp owns 32 pixels x 16 NW input channels; its 16-pixel tiles
// are 2 x 8 pixels (4 x 4 at H = 4), pixel g + 8 below pixel g, so 2 x 2
// blocks are summed in a thread and one shuffle. A CTA (one block of 16 NW
// input channels, blockIdx.y) takes `warps` such pairs of tiles, each with one warp or
// (S = 3) a warp per kernel row, and stages 16 output channels of dZ (with zero
// halo) and of the weights at a time.
struct DgTc {
    int warps, S, pairs, portion, slots, nw, logw;  // row pairs: per CTA, per image part
    size_t smem, woff;
};
constexpr int DG_PX = 48;  // bytes of a staged pixel: 16 channels and 16 bytes (conflict-free ldmatrix)

DgTc dg_tc(int cin, int H, long long total_pairs, int sms) {
    DgTc d;
    const int m = cin / 16;
    d.nw = m % 4 == 0 ? 4 : m % 3 == 0 ? 3 : m % 2 == 0 ? 2 : 1;
    d.logw = H == 32 ? 5 : H == 16 ? 4 : H == 8 ? 3 : 2;
    d.warps = 8;
    // smaller CTAs until there are two per SM
    while (d.warps > (H == 32 ? 2 : 1) &&
           (total_pairs + 16 * d.warps / H - 1) / (16 * d.warps / H) * (m / d.nw) < 2 * sms)
        d.warps /= 2;
    // few warps: three per pair of tiles, a kernel row each
    d.S = d.warps <= 2 ? 3 : 1;
    d.pairs = 16 * d.warps / H;
    d.portion = std::min(d.pairs, H / 2);
    d.slots = d.pairs / d.portion * (2 * d.portion + 2);
    d.woff = size_t(3) * d.slots * (H + 2) * DG_PX;
    d.smem = std::max(d.woff + size_t(9 * 16) * (32 * d.nw + 16),
                      size_t(d.S - 1) * d.warps * 16 * d.nw * 32 * sizeof(float));
    return d;
}

template <int NW>
__global__ void __launch_bounds__(256, 2)
k_dgrad_tc(const float* __restrict__ dZ, int cout, const bf16* __restrict__ Wt, int ca, int cb, int H,
           int total_pairs, DgTc d, const bf16* __restrict__ act, float* __restrict__ dIn, float* __restrict__ lo,
           const bf16* __restrict__ lo_act) {
    extern __shared__ __align__(16) unsigned char sm[];
    constexpr int PW = 32 * NW + 16;
    const int W = H, img = H / 2, cin = ca + cb, tid = threadIdx.x, lane = tid & 31;
    const int sp = (tid >> 5) / d.warps, warp = (tid >> 5) - sp * d.warps;
    const int dy0 = d.S == 3 ? sp : 0, dy1 = d.S == 3 ? sp + 1 : 3;
    const int pair0 = blockIdx.x * d.pairs, ci0 = blockIdx.y * 16 * NW, per = 2 * d.portion + 2;
    const int plane = d.slots * (W + 2) * DG_PX;
    unsigned char* const wsm = sm + d.woff;
    // row pair (in the CTA) and column of pixel g (0..7; g + 8 is below) of tile T
    auto pair_of = [&](int T, int g) { return H == 4 ? 2 * T + (g >> 2) : T >> (d.logw - 3); };
    auto col_of = [&](int T, int g) { return H == 4 ? (g & 3) : ((T & (W / 8 - 1)) << 3) + g; };
    uint32_t az[2];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        const int T = 2 * warp + mt, g = lane & 7, pr = pair_of(T, g), part = pr / d.portion;
        const int slot = part * per + 1 + 2 * (pr - part * d.portion) + ((lane >> 3) & 1);
        az[mt] = smem_u32(sm) + (slot * (W + 2) + col_of(T, g) + 1) * DG_PX + (lane >> 4) * 16;
    }
    const uint32_t bw = smem_u32(wsm) + (((lane >> 3) & 1) * 8 + (lane & 7)) * PW + (lane >> 4) * 16;
    float acc[2][2 * NW][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int b = 0; b < 2 * NW; ++b)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[mt][b][k] = 0.f;
    // the zero columns of every staged row
    for (int i = tid; i < 3 * d.slots * 2 * (DG_PX / 16); i += blockDim.x) {
        const int q = i / (DG_PX / 16), row = q >> 1, x = (q & 1) ? W + 1 : 0;
        *reinterpret_cast<uint4*>(sm + (row * (W + 2) + x) * DG_PX + 16 * (i % (DG_PX / 16))) = make_uint4(0, 0, 0, 0);
    }
    for (int k0 = 0; k0 < cout; k0 += 16) {
        __syncthreads();
#pragma unroll 4
        for (int i = tid; i < d.slots * W * 4; i += blockDim.x) {
            const int c4 = i & 3, x = (i >> 2) & (W - 1), slot = i >> (2 + d.logw);
            const int part = slot / per, j = slot - part * per, gp = pair0 + part * d.portion;
            const int b = gp / img, y = 2 * (gp - b * img) - 1 + j;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (gp < total_pairs && y >= 0 && y < H)
                v = __ldg(reinterpret_cast<const float4*>(dZ + ((size_t(b) * H + y) * W + x) * cout + k0) + c4);
            store_split(sm + (slot * (W + 2) + x + 1) * DG_PX + 8 * c4, plane, v);
        }
        for (int i = tid; i < 9 * 16 * 2 * NW; i += blockDim.x) {
            const int q = i / (2 * NW), v = i - q * 2 * NW, co = q / 9, tap = q - 9 * co;
            *reinterpret_cast<uint4*>(wsm + (tap * 16 + co) * PW + 16 * v) =
                __ldg(reinterpret_cast<const uint4*>(Wt + (size_t(k0 + co) * 9 + tap) * cin + ci0 + 8 * v));
        }
        __syncthreads();
#pragma unroll 1
        for (int dy = dy0; dy < dy1; ++dy) {
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                const int off = ((1 - dy) * (W + 2) + 1 - dx) * DG_PX;
                uint32_t b[NW][4];
#pragma unroll
                for (int j = 0; j < NW; ++j) ldsm4t(b[j], bw + (3 * dy + dx) * 16 * PW + 32 * j);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    uint32_t a[3][4];
#pragma unroll
                    for (int k = 0; k < 3; ++k) ldsm4(a[k], az[mt] + k * plane + off);
#pragma unroll
                    for (int j = 0; j < NW; ++j) {
                        mma3(acc[mt][2 * j], a, b[j][0], b[j][1]);
                        mma3(acc[mt][2 * j + 1], a, b[j][2], b[j][3]);
                    }
                }
            }
        }
    }
    if (d.S == 3) {
        float* const red = reinterpret_cast<float*>(sm);  // [kernel row 1, 2][warp][16 NW][32]
        __syncthreads();
        if (sp > 0) {
            float* o = red + size_t((sp - 1) * d.warps + warp) * 16 * NW * 32 + lane;
#pragma unroll
            for (int i = 0; i < 16 * NW; ++i) o[32 * i] = acc[i / (8 * NW)][(i / 4) % (2 * NW)][i & 3];
        }
        __syncthreads();
        if (sp > 0) return;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float* o = red + size_t(k * d.warps + warp) * 16 * NW * 32 + lane;
#pragma unroll
            for (int i = 0; i < 16 * NW; ++i) acc[i / (8 * NW)][(i / 4) % (2 * NW)][i & 3] += o[32 * i];
        }
    }
    const int g = lane >> 2, t2 = 2 * (lane & 3), nch = lo ? cb : cin;
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
        const int T = 2 * warp + mt, gp = pair0 + pair_of(T, g), x = col_of(T, g);
        const bool live = gp < total_pairs;
        const int b = gp / img, y = 2 * (gp - b * img);
#pragma unroll
        for (int j = 0; j < 2 * NW; ++j) {
            const float(&v)[4] = acc[mt][j];
            const int ci = ci0 + 8 * j + t2;
            if (lo && ci < ca) {
                // 2 x 2 sum: rows in the thread, columns g and g ^ 1
                float s0 = v[0] + v[2], s1 = v[1] + v[3];
                s0 += __shfl_xor_sync(0xffffffffu, s0, 4);
                s1 += __shfl_xor_sync(0xffffffffu, s1, 4);
                if (live && (g & 1) == 0) {
                    const size_t o = ((size_t(b) * (H / 2) + y / 2) * (W / 2) + x / 2) * ca + ci;
                    const uint32_t m = __ldg(reinterpret_cast<const uint32_t*>(lo_act + o));
                    *reinterpret_cast<float2*>(lo + o) = make_float2(pos_lo(m) ? s0 : 0.f, pos_hi(m) ? s1 : 0.f);
                }
            } else if (live) {
                const int c = lo ? ci - ca : ci;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const size_t o = ((size_t(b) * H + y + h) * W + x) * nch + c;
                    float2 q = make_float2(v[2 * h], v[2 * h + 1]);
                    if (act) {
                        const uint32_t m = __ldg(reinterpret_cast<const uint32_t*>(act + o));
                        q = make_float2(pos_lo(m) ? q.x : 0.f, pos_hi(m) ? q.y : 0.f);
                    }
                    *reinterpret_cast<float2*>(dIn + o) = q;
                }
            }
        }
    }
}

typedef void (*DgKernel)(const float*, int, const bf16*, int, int, int, int, DgTc, const bf16*, float*, float*,
                         const bf16*);
DgKernel dg_kernel(int nw) {
    return nw == 4 ? k_dgrad_tc<4> : nw == 3 ? k_dgrad_tc<3> : nw == 2 ? k_dgrad_tc<2> : k_dgrad_tc<1>;
}
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

bool dgrad_tc_shape(int ca, int cb, int cout) {
    return (ca + cb) % 16 == 0 && ca % 8 == 0 && cb % 8 == 0 && cout % 16 == 0;
}
// fewer than 16 input channels are padded with zeros (3 -> 16 channels at 32 x
// 32, 256 images: 50 us by the FP32-FMA kernel, 27 so)
bool wgrad_tc_shape(int ca, int cb, int cout) {
    return dgrad_tc_shape(ca, cb, cout) || (ca < 16 && cb == 0 && cout % 16 == 0);
}

size_t wgrad_tc_ws_floats(int cin, int cout, int H, int sms) {
    return size_t(std::max(1, 2 * sms / wg_tc(cin, cout, H).ny)) * (size_t(cout) * 9 * cin + cout);
}

bool wgrad_tc_fits(const ConvBwd& L, const float* dZ) {
    if (L.simt || !wgrad_tc_shape(L.ca, L.cb, L.cout) || !aligned16(dZ)) return false;
    return L.ca + L.cb < 16 ? !L.upA : aligned16(L.A) && aligned16(L.B);
}

cudaError_t wgrad_tc(const ConvBwd& L, const float* dZ, int Bn, float* ws, int* chunks, int sms, cudaStream_t s) {
    const int rows = Bn * L.H;
    const WgTc w = wg_tc(L.ca + L.cb, L.cout, L.H);
    const int rc = wg_tc_rows(w, rows, sms);
    *chunks = (rows + rc - 1) / rc;
    auto kern = L.H == 32 ? k_wgrad_tc<32> : L.H == 16 ? k_wgrad_tc<16> : L.H == 8 ? k_wgrad_tc<8> : k_wgrad_tc<4>;
    const cudaError_t e = raise_smem_limit(kern, w.smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(*chunks, w.ny), w.threads, w.smem, s>>>(dZ, L.cout, L.A, L.ca, L.upA ? 1 : 0, L.B, L.cb, rows, rc, w,
                                                        ws);
    return cudaGetLastError();
}

bool dgrad_tc_fits(const ConvBwd& L, const float* dZ, const bf16* Wt) {
    return !L.simt && dgrad_tc_shape(L.ca, L.cb, L.cout) && aligned16(dZ) && aligned16(Wt);
}

cudaError_t dgrad_tc(const ConvBwd& L, const float* dZ, const bf16* Wt, int Bn, const bf16* act, float* dIn,
                     float* lo, const bf16* lo_act, int sms, cudaStream_t s) {
    const int pairs = Bn * (L.H / 2);
    const DgTc d = dg_tc(L.ca + L.cb, L.H, pairs, sms);
    const cudaError_t e = raise_smem_limit(dg_kernel(d.nw), d.smem);
    if (e != cudaSuccess) return e;
    dg_kernel(d.nw)<<<dim3((pairs + d.pairs - 1) / d.pairs, (L.ca + L.cb) / (16 * d.nw)), 32 * d.warps * d.S, d.smem, s>>>(
        dZ, L.cout, Wt, L.ca, L.cb, L.H, pairs, d, act, dIn, lo, lo_act);
    return cudaGetLastError();
}

bool grad_tc_fits(int cin, int cout, int H) {
    return std::max(wg_tc(cin, cout, H).smem, dg_tc(cin, H, 1ll << 40, 1).smem) <= size_t(227) * 1024;
}

}  // namespace net
}  // namespace fwr
