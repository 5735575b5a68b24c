// FP32 Gerchberg kernel of one frame per thread-block cluster, grid 128^2
// (sm_103a): the path of few frames.
//
// One CTA per frame (fwr_fused.cuh) spends 9 us per iteration and 20 us before
// and after, on one SM: half of it waiting for instructions, since a few warps
// run 58 KB of straight-line code per iteration. Here 8 or 16 CTAs share a frame
// and the line transforms are cut finer (128 = 4 x 8 x 4 with 8 cells per lane),
// so each SM's share is an eighth or less and the code a third. A warp keeps two
// lines: rows 2w, 2w + 1 of its CTA in the row phases (inverse transform,
// reinsertion (Algorithm 1 step 4), x part of Eq. PC, forward transform) and a
// pair of columns kx, -kx in the column phases (forward transform with the y
// part of Eq. PC, the projection or final filter on the pair's bins, inverse
// transform). So nothing inside a phase crosses a warp; between phases every
// lane stores its results straight into the shared memory of the CTA that owns
// the line, and a cluster barrier follows.
//
// The arithmetic is the fused kernel's, operation by operation: its 32-point
// networks cut after three stages (the last two with the lane's own factors),
// its twiddles, sums, fills and spectral steps. The phase is the same bits.
//
// Shared memory: cell (p, line) of a phase at 18 p + p / 8 + p / 32 + line:
// neighbouring lines adjacent (the remote stores of a warp are runs of them),
// reads along p and of the last two stages free of bank conflicts, the 8-point
// passes two-way. What bounds it is latency: shared-memory passes, two cluster
// barriers per iteration that wait for the remote stores (14 bytes per clock and
// SM), few warps. Measured, 40 x 40 lenslets, one frame (us, before / now): k = 0
// 23 / 10.5, k = 2 41 / 17, k = 10 113 / 45.

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <utility>
#include <vector>

#include "fwr_internal.h"

namespace fwr {

#include "fwr_fft.cuh"
#include "fwr_fused.cuh"
#include "fwr_cluster.cuh"

namespace {

constexpr int N = 128;
constexpr int CELLS = 18 * N + N / 8 + N / 32;
template <int CL> constexpr size_t smem_bytes() {
    return 2 * size_t(CELLS) * sizeof(float2) + 2 * size_t(N) * sizeof(float2) + 8 * size_t(16 * N / CL) * sizeof(float);
}

__device__ __forceinline__ int cell(int p, int line) { return 18 * p + (p >> 3) + (p >> 5) + line; }

// The last two stages of a 32-point network for the pairs at J, J + 8, J + 16,
// J + 24: factors w_32^(2 J), w_32^J and w_32^(J + 8) in the tangent form of
// bfly (fwr_fft.cuh), w = s (1 + i r) or s (r + i), chosen per lane.
struct Tail {
    float s[3], r[3];
    bool c[3];  // the first form
};
__device__ __forceinline__ Tail make_tail(int J) {
    Tail t;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int i = k == 0 ? 2 * J : k == 1 ? J : J + 8;
        const float2 f = c_t32f[i];
        t.s[k] = f.x;
        t.r[k] = i == 8 ? 0.f : f.y;  // w = -i
        t.c[k] = i <= 4 || i >= 12;
    }
    return t;
}
// bfly with the factor k of t
template <bool INV> __device__ __forceinline__ void bfly_rt(float2& a, float2& b, const Tail& t, int k) {
    const bool c = t.c[k];
    const float r = INV ? -t.r[k] : t.r[k], s = INV && !c ? -t.s[k] : t.s[k];
    const float P = c ? b.y : b.x, Q = c ? b.x : b.y;
    const float2 u = make_float2(fmaf(c ? -r : r, P, c ? Q : -Q), fmaf(r, Q, P));
    const float2 a0 = a;
    a = make_float2(fmaf(s, u.x, a0.x), fmaf(s, u.y, a0.y));
    b = make_float2(fmaf(-s, u.x, a0.x), fmaf(-s, u.y, a0.y));
}

// Two lines (l0, l1) of buf through the 32-point DFTs over s for each of the
// four q: in natural order at (p = 32 q + s), out in registers, y[line][i] = s =
// J + 8 i of lane J + 8 q.
template <bool INV>
__device__ __forceinline__ void dft32(float2* buf, int l0, int l1, const Tail& t, int lane, float2 (&y)[2][4]) {
    {
        const int c = lane & 3, q = (lane >> 2) & 3, l = lane >> 4 ? l1 : l0;
        float2 x[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) x[m] = buf[cell(32 * q + 4 * m + c, l)];
        dft_reg<8, INV>(x);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j) buf[cell(32 * q + 8 * c + j, l)] = x[j];
    }
    __syncwarp();
    const int J = lane & 7, q = lane >> 3;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int l = h ? l1 : l0;
        // blocks in the network's (bit-reversed) order
        float2 v0 = buf[cell(32 * q + J, l)], v1 = buf[cell(32 * q + 16 + J, l)];
        float2 v2 = buf[cell(32 * q + 8 + J, l)], v3 = buf[cell(32 * q + 24 + J, l)];
        bfly_rt<INV>(v0, v1, t, 0);
        bfly_rt<INV>(v2, v3, t, 0);
        bfly_rt<INV>(v0, v2, t, 1);
        bfly_rt<INV>(v1, v3, t, 2);
        y[h][0] = v0;
        y[h][1] = v1;
        y[h][2] = v2;
        y[h][3] = v3;
    }
}

__device__ __forceinline__ void put(float2* buf, int l0, int l1, int lane, const float2 (&y)[2][4]) {
    const int J = lane & 7, q = lane >> 3;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 4; ++i) buf[cell(32 * q + J + 8 * i, h ? l1 : l0)] = y[h][i];
}

template <int CL>
__global__ void __launch_bounds__(16 * N / CL, 2) cluster128_kernel(Params<float> p, int clusters) {
    constexpr int SL = N / CL, SC = SL / 2, NT = 32 * SC;
    extern __shared__ __align__(16) unsigned char smem[];
    float2* const R = reinterpret_cast<float2*>(smem);       // row phase: (kx, row)
    float2* const C = R + CELLS;                             // column phase: (row, line)
    float2* const At = C + CELLS;                            // a(u), T(u)
    float2* const Tt = At + N;
    float* const wf = reinterpret_cast<float*>(Tt + N);      // final weights of each thread's bins
    const uint32_t rbase = uint32_t(__cvta_generic_to_shared(R)), cbase = uint32_t(__cvta_generic_to_shared(C));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, rank = cluster_rank();
    const int n = p.n, off = p.off, nn = n * n, mode = p.periodic;
    cluster_arrive();  // matched before the first remote store: every CTA runs

    const int J = lane & 7, q = lane >> 3;
    const Tail tail = make_tail(J);
    if (tid < N) {
        At[tid] = p.tab.A[tid];
        Tt[tid] = p.tab.Tt[tid];
    }
    // twiddles w^(lane k) between the 4- and 32-point parts, and w^q
    float2 tw[3];
#pragma unroll
    for (int k = 1; k < 4; ++k) tw[k - 1] = p.tab.tw[lane * k];
    const float2 tq[4] = {p.tab.tw[0], p.tab.tw[1], p.tab.tw[2], p.tab.tw[3]};
    // column phase: lines warp and warp + SC; bins ky = q + 4 (J + 8 i)
    const int l0 = warp, l1 = warp + SC;
    const bool self = rank == 0 && warp == 0;  // columns 0 and N/2 are their own partners
    int kx[2];
    float al[2][4], be[2][4], ga[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        kx[h] = owned_column<N, SC>(rank, h ? l1 : l0);
        const float4 u = __ldg(reinterpret_cast<const float4*>(p.tab.pt) + kx[h]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int ky = q + 4 * (J + 8 * i), wi = ky <= N / 2 ? ky * N + kx[h] : (N - ky) * N + ((N - kx[h]) & (N - 1));
            const float4 v = __ldg(reinterpret_cast<const float4*>(p.tab.pt) + ky);
            lsq_coefs(__ldg(p.tab.iota + wi), u.x, u.y, 0.5f * u.z, 0.5f * u.w, quad<float>{v.x, v.y, v.z, v.w},
                      al[h][i], be[h][i], ga[h][i]);
            wf[(4 * h + i) * NT + tid] = __ldg(p.tab.wfin + wi);
        }
    }
    // row phase: rows 2 warp, 2 warp + 1 of the CTA, cells q + 4 (J + 8 i)
    const int r0 = SL * rank + 2 * warp;
    unsigned valid = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int ii = r0 + h - off, j = q + 4 * (J + 8 * i) - off;
            if (ii >= 0 && ii < n && j >= 0 && j < n && p.mask[ii * n + j]) valid |= 1u << (4 * h + i);
        }
    __syncthreads();
    cluster_wait();

    bool finite = true;
    const bool fill_first = fills_first(mode, p.iters);
    for (int f = int(blockIdx.x) / CL; f < p.F; f += clusters) {
        const float* const sl = p.slopes + size_t(f) * 2 * nn;
        const float* const ext = p.ext_init ? p.ext_init + size_t(f) * 2 * N * N : nullptr;
        const uint16_t* const exth = p.ext_init_h ? p.ext_init_h + size_t(f) * 2 * N * N : nullptr;
        float2 y[2][4], meas[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int row = r0 + h, c = q + 4 * (J + 8 * i), ii = row - off, j = c - off, gi = row * N + c;
                float2 v = make_float2(0.f, 0.f);
                if (ext) {
                    v = make_float2(ext[gi], ext[N * N + gi]);
                } else if (exth) {
                    v = make_float2(__uint_as_float(uint32_t(exth[gi]) << 16),
                                    __uint_as_float(uint32_t(exth[N * N + gi]) << 16));
                } else if (p.hud) {
                    // Hudgin extension from the pupil's edge slopes
                    if (j >= 0 && j < n) {
                        const int e0 = p.hud[j], e1 = p.hud[n + j];
                        if (e0 >= 0 && (ii < e0 || ii > e1)) v.x = sl[(ii < e0 ? e0 : e1) * n + j];
                    }
                    if (ii >= 0 && ii < n) {
                        const int e0 = p.hud[2 * n + ii], e1 = p.hud[3 * n + ii];
                        if (e0 >= 0 && (j < e0 || j > e1)) v.y = sl[nn + ii * n + (j < e0 ? e0 : e1)];
                    }
                }
                // replaced by Eq. PC, as in the fused kernel
                if (fill_first && row == N - 1) v.y = 0.f;
                if (valid & (1u << (4 * h + i))) {
                    v = make_float2(sl[ii * n + j], sl[nn + ii * n + j]);
                    finite &= isfinite(v.x) && isfinite(v.y);
                }
                y[h][i] = meas[h][i] = v;
            }
        for (int it = 0; it <= p.iters; ++it) {
            const bool final = it == p.iters;
            const bool fill = mode == PERIODIC_BEFORE_EACH_FFT || (mode == PERIODIC_FINAL_ONLY && final);
            if (fill) {
                // x part of Eq. PC, the fused kernel's tree: over J + 8 i of each
                // quarter, then the quarters
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float t3 = y[h][3].x;
                    if (lane == 31) t3 = 0.f;
                    float s = (y[h][0].x + y[h][2].x) + (y[h][1].x + t3);
#pragma unroll
                    for (int o = 4; o >= 1; o /= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
                    const float s0 = __shfl_sync(0xffffffffu, s, 0), s1 = __shfl_sync(0xffffffffu, s, 8);
                    const float s2 = __shfl_sync(0xffffffffu, s, 16), s3 = __shfl_sync(0xffffffffu, s, 24);
                    if (lane == 31) y[h][3].x = -(((s0 + s1) + s2) + s3);
                }
            }
            // ---- forward rows: 32-point over the cells of each quarter, twiddles,
            // 4-point over the quarters; bins lane + 32 a to the columns' owners
            {
                const int a0 = 2 * warp, a1 = a0 + 1;
                __syncwarp();
                put(R, a0, a1, lane, y);
                __syncwarp();
                dft32<false>(R, a0, a1, tail, lane, y);
                put(R, a0, a1, lane, y);
                __syncwarp();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 z[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) z[a] = R[cell(32 * a + lane, a0 + h)];
#pragma unroll
                    for (int a = 1; a < 4; ++a) z[a] = twiddle<false>(z[a], tw[a - 1]);
                    dft_reg<4, false>(z);
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        int owner, line;
                        column_owner<N, SC>(lane + 32 * a, owner, line);
                        st_rank(cbase + uint32_t(cell(r0 + h, line) * sizeof(float2)), owner, z[a]);
                    }
                }
            }
            cluster_arrive();
            cluster_wait();
            // ---- forward columns: 4-point over rows 32 apart, twiddles, 32-point
            {
                float2 z[2][4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int a = 0; a < 4; ++a) z[h][a] = C[cell(lane + 32 * a, h ? l1 : l0)];
                    dft_reg<4, false>(z[h]);
#pragma unroll
                    for (int a = 1; a < 4; ++a) z[h][a] = twiddle<false>(z[h][a], tw[a - 1]);
                }
                if (fill) {
                    // the columns' ky = 0 bins; lane 31 holds the last inputs
                    float2 d0 = z[0][0], d1 = z[1][0];
#pragma unroll
                    for (int o = 16; o >= 1; o /= 2) {
                        d0 = cadd(d0, make_float2(__shfl_xor_sync(0xffffffffu, d0.x, o), __shfl_xor_sync(0xffffffffu, d0.y, o)));
                        d1 = cadd(d1, make_float2(__shfl_xor_sync(0xffffffffu, d1.x, o), __shfl_xor_sync(0xffffffffu, d1.y, o)));
                    }
                    const float2 p0 = self ? d0 : d1, p1 = self ? d1 : d0;
                    if (lane == 31) {
#pragma unroll
                        for (int a = 0; a < 4; ++a) {
                            z[0][a] = fill_input(z[0][a], d0, p0, tq[a]);
                            z[1][a] = fill_input(z[1][a], d1, p1, tq[a]);
                        }
                    }
                }
                __syncwarp();
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int a = 0; a < 4; ++a) C[cell(32 * a + lane, h ? l1 : l0)] = z[h][a];
            }
            __syncwarp();
            dft32<false>(C, l0, l1, tail, lane, y);
            put(C, l0, l1, lane, y);
            __syncwarp();
            // ---- spectral step: partner (-ky, -kx) at quarter qn, place 31 - s (or 32 - s)
            {
                const int qn = (4 - q) & 3;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int pl = (h != 0) == self ? l1 : l0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int s = J + 8 * i, sn = q ? 31 - s : (32 - s) & 31;
                        const float2 z2 = C[cell(32 * qn + sn, pl)];
                        if (!final)
                            y[h][i] = lsq_apply(al[h][i], be[h][i], ga[h][i], y[h][i], z2);
                        else
                            y[h][i] = final_bin(y[h][i], z2, At[kx[h]], Tt[kx[h]], At[q + 4 * s], Tt[q + 4 * s],
                                                0.5f * wf[(4 * h + i) * NT + tid]);
                    }
                }
            }
            __syncwarp();
            // ---- inverse columns: 32-point, twiddles, 4-point; rows lane + 32 a to their owners
            put(C, l0, l1, lane, y);
            __syncwarp();
            dft32<true>(C, l0, l1, tail, lane, y);
            put(C, l0, l1, lane, y);
            __syncwarp();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 z[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) z[a] = C[cell(32 * a + lane, h ? l1 : l0)];
#pragma unroll
                for (int a = 1; a < 4; ++a) z[a] = twiddle<true>(z[a], tw[a - 1]);
                dft_reg<4, true>(z);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    const int row = lane + 32 * a;
                    st_rank(rbase + uint32_t(cell(kx[h], row % SL) * sizeof(float2)), row / SL, z[a]);
                }
            }
            cluster_arrive();
            cluster_wait();
            // ---- inverse rows: 4-point over bins 32 apart, twiddles, 32-point
            {
                const int a0 = 2 * warp, a1 = a0 + 1;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 z[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) z[a] = R[cell(lane + 32 * a, a0 + h)];
                    dft_reg<4, true>(z);
#pragma unroll
                    for (int a = 1; a < 4; ++a) z[a] = twiddle<true>(z[a], tw[a - 1]);
#pragma unroll
                    for (int a = 0; a < 4; ++a) R[cell(32 * a + lane, a0 + h)] = z[a];
                }
                __syncwarp();
                dft32<true>(R, a0, a1, tail, lane, y);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (final)
                        p.phase[(size_t(f) * N + r0 + h) * N + q + 4 * (J + 8 * i)] = y[h][i].x;
                    else if (valid & (1u << (4 * h + i)))
                        y[h][i] = meas[h][i];
                }
        }
    }
    if (!finite) atomicOr(p.status, STATUS_NONFINITE);
}

}  // namespace

// Frames that run at once: 7 with clusters of 16 CTAs, 30 with 8 (two CTAs per
// SM); the fused kernel takes a frame per SM in the time of one. Measured, k = 5
// (us, clusters of 16 / of 8 / fused kernel): 1 to 7 frames 28 / 37 / 68, 15: 62 /
// 39 / 68, 30: 94 / 57 / 68, 40: - / 89 / 68. A call cannot know what other
// streams run, and a cluster takes more SM time per frame (2.6 to 4 us of the
// chip against 0.5): several calls at once, in sum (us, this / fused kernel; a
// graph with parallel branches): 10 x 1 frames 48 / 82, 64 x 1 217 / 225, 5 x 4
// 65 / 74, 10 x 4 111 / 83, 2 x 15 56 / 70, 5 x 15 142 / 74, 2 x 30 111 / 70, 5 x
// 30 257 / 74. So the line lies at 15 frames, where a lone call gains 1.7 times.
bool cluster128_wanted(int F, int sms) { return F <= sms / 10; }

template <int CL> static cudaError_t launch_cl(const Params<float>& p, cudaStream_t s) {
    static std::mutex mu;
    static std::vector<std::pair<int, int>> cache;
    return launch_clusters(cluster128_kernel<CL>, p, CL, 16 * N / CL, smem_bytes<CL>(), mu, cache, s);
}

cudaError_t launch_cluster_f32(const Params<float>& p, int sms, cudaStream_t s) {
    if (16 * p.F <= 3 * sms / 4) {
        const cudaError_t e = launch_cl<16>(p, s);
        if (e == cudaSuccess) return e;
        cudaGetLastError();  // no cluster of 16 to be had (not a portable size)
    }
    return launch_cl<8>(p, s);
}

}  // namespace fwr
