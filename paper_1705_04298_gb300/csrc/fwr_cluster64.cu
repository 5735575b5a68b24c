// FP64 Gerchberg kernel of one frame per thread-block cluster, grids 32^2 and
// 64^2 (sm_103a).
//
// What bounds the FP64 path is the FP64 unit: it takes 64 cycles per warp
// instruction and SM quarter, whatever the number of active lanes (measured:
// 2 to 32 lanes alike, 76 cycles with all four quarters busy), so one CTA per
// frame took 29 us per iteration at 32^2 with most of the chip idle. Here a
// cluster of 8 CTAs shares a frame, a warp takes a line and a lane N / 32 of its
// elements: full warps, one line per SM quarter at 32^2 (two at 64^2), and four
// FP64 instructions per butterfly stage and lane: out = A + W B with W = +-w^J of
// the lane, both halves of a pair doing their own output.
//
// Line transforms are N/4-point DFTs over elements 4 apart, twiddles and
// 4-point DFTs (the factors of fwr_fused.cuh, with as few rounded products), each
// a decimation-in-time network over lanes (shuffles; the last stage of 64 points
// inside the lane) from bit-reversed to natural order; the bit reversal is taken
// where the data pass through shared memory
// anyway. CTA r works rows SL r .. SL r + SL - 1 in the row phases (inverse
// transform, reinsertion (Algorithm 1 step 4), x part of Eq. PC, forward
// transform) and SL columns in pairs kx, -kx in the column phases (forward
// transform, the LSQ projection of Sec. 3.3 or the final filter of Eqs. 2-3
// with the y part of Eq. PC, inverse transform); results are stored straight
// into the shared memory of the CTA that needs them, and a cluster barrier ends
// each phase. The y part of Eq. PC is added to the last row's input of each
// column transform, from the column sums of kx and -kx (taking it out of the
// finished spectrum is shorter by ten FP64 instructions, but its cancellation
// doubles the rounding error after ten iterations).
// Measured, k = 10, one frame: 16 x 16 lenslets on 32^2 322 -> 71 us, 31 x 31 on
// 64^2 1093 -> 185 us.

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

constexpr int CL = 8;  // CTAs per frame

__device__ __forceinline__ double2 shfl_xor2(double2 v, int h) {
    return make_double2(__shfl_xor_sync(0xffffffffu, v.x, h), __shfl_xor_sync(0xffffffffu, v.y, h));
}

template <int N> struct C64 {
    static constexpr int E = N / 32, SL = N / CL, SC = SL / 2, H = N / 2, NT = 32 * SL, LOG = N == 64 ? 6 : 5;
    static constexpr int LS = N + 1;  // line stride (cells)
    static constexpr size_t rbuf = 0, cbuf = rbuf + size_t(SL) * LS * 16, sbuf = cbuf + size_t(SL) * LS * 16,
                            dc = sbuf + size_t(SL) * LS * 16, bytes = dc + size_t(SL) * 16;
};

// this lane's constants: signs of the trivial stages, +-w_8^J and +-w_16^J of
// the others (J: the pair's place in its block), the twiddles w_N^(n2 k1) of its
// elements, and whether a stage turns the pair's second element by -i
template <int N> struct Tw64 {
    double2 w8, w16, t[N / 32];
    double sg1, sg2, sg8, sg16;  // lane bits 0, 1, 3, 4: -1 where set
    bool rot2, rot16;
};

// one output of a pair (lanes l and l ^ h): a + W b, the lane's own W
__device__ __forceinline__ void pair_of(double2 v, int h, int lane, double2& a, double2& b) {
    const double2 o = shfl_xor2(v, h);
    const bool up = lane & h;
    a = up ? o : v;
    b = up ? v : o;
}
template <bool INV> __device__ __forceinline__ double2 turned(double2 b, bool on) {
    return !on ? b : INV ? make_double2(-b.y, b.x) : make_double2(b.y, -b.x);
}
__device__ __forceinline__ double2 add_s(double2 a, double sg, double2 b) {
    return make_double2(fma(sg, b.x, a.x), fma(sg, b.y, a.y));
}
template <bool INV> __device__ __forceinline__ double2 add_w(double2 a, double2 w, double2 b) {
    const double wy = INV ? -w.y : w.y;
    return make_double2(fma(w.x, b.x, fma(-wy, b.y, a.x)), fma(w.x, b.y, fma(wy, b.x, a.y)));
}

// In: slot j = lane + 32 e holds element bitrev(j); out: element j.
template <bool INV, int N>
__device__ __forceinline__ void line_dft(double2 (&x)[N / 32], const Tw64<N>& t, int lane) {
    constexpr int E = N / 32;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        double2 v = x[e], a, b;
        // N/4-point DFT
        pair_of(v, 1, lane, a, b);
        v = add_s(a, t.sg1, b);
        pair_of(v, 2, lane, a, b);
        v = add_s(a, t.sg2, turned<INV>(b, t.rot2));
        pair_of(v, 4, lane, a, b);
        v = add_w<INV>(a, t.w8, b);
        if (N == 64) {
            pair_of(v, 8, lane, a, b);
            v = add_w<INV>(a, t.w16, b);
        }
        // twiddle; 4-point DFT over the N/4-lane groups
        v = INV ? cmulc(t.t[e], v) : cmul(v, t.t[e]);
        if (N == 32) {
            pair_of(v, 8, lane, a, b);
            v = add_s(a, t.sg8, b);
            pair_of(v, 16, lane, a, b);
            v = add_s(a, t.sg16, turned<INV>(b, t.rot16));
        } else {
            pair_of(v, 16, lane, a, b);
            v = add_s(a, t.sg16, b);
        }
        x[e] = v;
    }
    if (E == 2) {
        const double2 a = x[0], b = turned<INV>(x[E - 1], t.rot16);
        x[0] = cadd(a, b);
        x[E - 1] = csub(a, b);
    }
}

template <int N>
__global__ void __launch_bounds__(C64<N>::NT) cluster64_kernel(Params<double> p, int clusters) {
    typedef C64<N> G;
    constexpr int E = G::E, SL = G::SL, SC = G::SC, H = G::H, LS = G::LS;
    extern __shared__ __align__(16) unsigned char smem[];
    double2* const R = reinterpret_cast<double2*>(smem + G::rbuf);  // [row][kx]
    double2* const C = reinterpret_cast<double2*>(smem + G::cbuf);  // [line][row]
    double2* const S = reinterpret_cast<double2*>(smem + G::sbuf);  // [line][ky]
    double2* const dc = reinterpret_cast<double2*>(smem + G::dc);   // [line] column sums
    const uint32_t rbase = uint32_t(__cvta_generic_to_shared(R)), cbase = uint32_t(__cvta_generic_to_shared(C));
    const int lane = threadIdx.x & 31, line = threadIdx.x >> 5;
    const int rank = cluster_rank(), n = p.n, off = p.off, nn = n * n, mode = p.periodic;
    cluster_arrive();  // matched before the first remote store: every CTA runs

    Tw64<N> tw;
    {
        auto sign = [&](int bit) { return lane & bit ? -1.0 : 1.0; };
        auto stage = [&](int h) {  // +-w_{2h}^J
            const double2 w = p.tab.tw[(lane & (h - 1)) * (N / (2 * h))];
            return lane & h ? make_double2(-w.x, -w.y) : w;
        };
        tw.sg1 = sign(1);
        tw.sg2 = sign(2);
        tw.sg8 = sign(8);
        tw.sg16 = sign(16);
        tw.rot2 = lane & 1;
        tw.rot16 = N == 32 ? lane & 8 : lane & 16;
        tw.w8 = stage(4);
        tw.w16 = stage(8);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int j = lane + 32 * e, g = j / (N / 4), n2 = 2 * (g & 1) + (g >> 1);
            tw.t[e] = p.tab.tw[n2 * (j % (N / 4))];
        }
    }
    // column of this warp's line, the line of its partner -kx
    const int kx = owned_column<N, SC>(rank, line);
    const int kxn = (N - kx) & (N - 1);
    const int pl = (rank == 0 && (line & (SC - 1)) == 0) ? line : (line ^ SC);
    // this lane's elements j = lane + 32 e: bin (j, kx), row j of a column,
    // column j of row SL rank + line
    double al[E], be[E], ga[E], wfin[E];
    int rev[E];
    const double2 Akx = p.tab.A[kx], Tkx = p.tab.Tt[kx];
    {
        const double *u = p.tab.pt + 4 * kx;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int j = lane + 32 * e;
            rev[e] = __brev(unsigned(j)) >> (32 - G::LOG);
            const int wi = j <= H ? j * N + kx : (N - j) * N + kxn;
            const double* v = p.tab.pt + 4 * j;
            lsq_coefs(p.tab.iota[wi], u[0], u[1], 0.5 * u[2], 0.5 * u[3], quad<double>{v[0], v[1], v[2], v[3]}, al[e],
                      be[e], ga[e]);
            wfin[e] = p.tab.wfin[wi];
        }
    }
    const int row = SL * rank + line, i0 = row - off;
    bool valid[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int j = lane + 32 * e - off;
        valid[e] = i0 >= 0 && i0 < n && j >= 0 && j < n && p.mask[i0 * n + j];
    }
    cluster_wait();

    bool finite = true;
    const bool fill_first = fills_first(mode, p.iters);
    for (int f = int(blockIdx.x) / CL; f < p.F; f += clusters) {
        const double* const sl = p.slopes + size_t(f) * 2 * nn;
        const double* const ext = p.ext_init ? p.ext_init + size_t(f) * 2 * N * N : nullptr;
        // this lane's measured slopes, and the embedding
        double2 meas[E], x[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int c = lane + 32 * e, j = c - off, gi = row * N + c;
            x[e] = make_double2(0.0, 0.0);
            if (ext) {
                x[e] = make_double2(ext[gi], ext[N * N + gi]);
            } else if (p.hud) {
                // Hudgin extension from the pupil's edge slopes
                if (j >= 0 && j < n) {
                    const int t = p.hud[j], b = p.hud[n + j];
                    if (t >= 0 && (i0 < t || i0 > b)) x[e].x = sl[(i0 < t ? t : b) * n + j];
                }
                if (i0 >= 0 && i0 < n) {
                    const int l = p.hud[2 * n + i0], r = p.hud[3 * n + i0];
                    if (l >= 0 && (j < l || j > r)) x[e].y = sl[nn + i0 * n + (j < l ? l : r)];
                }
            }
            // replaced by Eq. PC, as in the fused kernel
            if (fill_first && row == N - 1) x[e].y = 0.0;
            if (valid[e]) {
                meas[e] = make_double2(sl[i0 * n + j], sl[nn + i0 * n + j]);
                finite &= isfinite(meas[e].x) && isfinite(meas[e].y);
                x[e] = meas[e];
            }
        }
        for (int it = 0; it <= p.iters; ++it) {
            const bool final = it == p.iters;
            const bool fill = mode == PERIODIC_BEFORE_EACH_FFT || (mode == PERIODIC_FINAL_ONLY && final);
            if (fill) {
                double s = x[0].x;
                if (E == 1 && lane == 31) s = 0.0;
                if (E == 2 && lane != 31) s += x[E - 1].x;
#pragma unroll
                for (int o = 1; o < 32; o *= 2) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 31) x[E - 1].x = -s;
            }
            // ---- forward rows
            double2* const scr = R + line * LS;  // this warp's: the permutation's
            __syncwarp();
#pragma unroll
            for (int e = 0; e < E; ++e) scr[lane + 32 * e] = x[e];
            __syncwarp();
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = scr[rev[e]];
            line_dft<false, N>(x, tw, lane);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                int owner, l;
                column_owner<N, SC>(lane + 32 * e, owner, l);
                st_rank(cbase + uint32_t((l * LS + row) * 16), owner, x[e]);
            }
            cluster_arrive();
            cluster_wait();
            // ---- forward columns
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = C[line * LS + rev[e]];
            if (fill) {
                // -i Sy(0, kx) onto row N - 1, Sy(0, kx) = (Z(0, kx) - conj Z(0, -kx)) / (2i)
                double2 z0 = E == 2 ? cadd(x[0], x[E - 1]) : x[0];
#pragma unroll
                for (int o = 16; o >= 1; o /= 2) z0 = cadd(z0, shfl_xor2(z0, o));
                if (lane == 0) dc[line] = z0;
                __syncthreads();
                const double2 z0p = dc[pl];
                // slot N - 1 holds row N - 1
                if (lane == 31) {
                    x[E - 1].x += 0.5 * (z0p.x - z0.x);
                    x[E - 1].y -= 0.5 * (z0.y + z0p.y);
                }
            }
            line_dft<false, N>(x, tw, lane);
#pragma unroll
            for (int e = 0; e < E; ++e) S[line * LS + lane + 32 * e] = x[e];
            __syncthreads();
            // ---- spectral step
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int ky = lane + 32 * e;
                const double2 z1 = x[e], z2 = S[pl * LS + ((N - ky) & (N - 1))];
                if (!final) x[e] = lsq_apply(al[e], be[e], ga[e], z1, z2);
                else x[e] = final_bin(z1, z2, Akx, Tkx, p.tab.A[ky], p.tab.Tt[ky], 0.5 * wfin[e]);
            }
            // ---- inverse columns (C's line is this warp's until the next row phase)
            __syncwarp();
#pragma unroll
            for (int e = 0; e < E; ++e) C[line * LS + lane + 32 * e] = x[e];
            __syncwarp();
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = C[line * LS + rev[e]];
            line_dft<true, N>(x, tw, lane);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int r = lane + 32 * e;
                st_rank(rbase + uint32_t(((r % SL) * LS + kx) * 16), r / SL, x[e]);
            }
            cluster_arrive();
            cluster_wait();
            // ---- inverse rows
#pragma unroll
            for (int e = 0; e < E; ++e) x[e] = R[line * LS + rev[e]];
            line_dft<true, N>(x, tw, lane);
            if (!final) {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (valid[e]) x[e] = meas[e];
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) p.phase[(size_t(f) * N + row) * N + lane + 32 * e] = x[e].x;
            }
        }
    }
    if (!finite) atomicOr(p.status, STATUS_NONFINITE);
}

template <int N> cudaError_t launch_n(const Params<double>& p, cudaStream_t s) {
    static std::mutex mu;
    static std::vector<std::pair<int, int>> cache;
    return launch_clusters(cluster64_kernel<N>, p, CL, C64<N>::NT, C64<N>::bytes, mu, cache, s);
}

}  // namespace

// Up to 15 frames run at once, more take turns, while the fused kernel takes a
// frame per SM in the time of one. Measured at k = 10 (us, this / fused): 32^2,
// 76 frames: 204 / 326, 100: 261 / 326, 152: 360 / 327; 64^2, 76 frames: 835 / 1098,
// 100: 1019 / 1097. Several such calls at once cost more SM time than one CTA per
// frame: 38 frames on 32^2 alone 131 / 324, two at once 202 / 325, four 383 / 326,
// eight 716 / 498; single frames gain on any number of streams (64: 272 / 987).
bool cluster64_wanted(int N, int F, int sms) {
    return N == 32 ? F <= 3 * sms / 4 : N == 64 ? F <= 2 * sms / 3 : false;
}

cudaError_t launch_cluster_f64(int N, const Params<double>& p, cudaStream_t s) {
    return N == 32 ? launch_n<32>(p, s) : N == 64 ? launch_n<64>(p, s) : cudaErrorInvalidValue;
}

}  // namespace fwr
