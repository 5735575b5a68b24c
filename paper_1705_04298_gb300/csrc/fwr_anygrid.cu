// Gerchberg kernel for grids of any even size 18 <= N <= 62 that is no power
// of two (sm_103a): the paper's small windows, where the pupil of n lenslets is
// padded by w cells on each side (N = n + 2w, e.g. 46 and 52 for 40 lenslets
// with w = 3 and 6, Sec. 4.1).
//
// One CTA owns one frame at a time; its whole N x N packed grid Z = sx + i sy
// stays in shared memory for every iteration of Algorithm 1 (Sec. 3.3) and the
// final reconstruction (Eqs. 2-3), as in the power-of-two kernels; several CTAs
// share an SM.
//
// 1-D transforms, N = 2 M: the M-point DFTs E and O of the even and the odd
// elements as direct sums, folded about their middle: with a_j = v[j] + v[M-j]
// and b_j = v[j] - v[M-j],
//   E[k], E[M-k] = sum_j a_j cos(2 pi j k / M) -+ i sum_j b_j sin(2 pi j k / M),
// then X[k], X[k+M] = E[k] +- w_N^k O[k]. That is a quarter of the direct
// sum's multiplications, for every M (23 is prime, so there is no FFT to be had
// at N = 46), and it has the shape of a small matrix product: a thread takes
// one line and K of the k = 0 .. M/2, 8 K real sums whose inputs are two
// 16-byte loads per j (four 8-byte ones down a column) and whose coefficients,
// the same for the whole warp, K 8-byte ones: 8 K FMAs per 2 + K / 2 shared
// loads. What bounds it is the FP32 pipe and, for few frames, latency.
// Measured: 1000 frames of 40 x 40 lenslets on 46^2, 10 iterations: 3335 us
// with one output per lane and a twiddle look-up per product, 290 us now; one
// frame 68 us.
//
// Fusions: the x part of Eq. PC is a rank-1 correction of each row's spectrum
// (the row's sum comes out of the same loop), the y part one of each column's
// (from the column sums of kx and -kx, published through shared memory), and
// the reinsertion of the measured slopes is done where the inverse row
// transform stores its outputs. The spectral step works on (k, -k) pairs with
// coefficients computed once per launch.

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <vector>

#include "fwr_internal.h"

namespace fwr {

#include "fwr_fft.cuh"
#include "fwr_fused.cuh"

namespace {

constexpr int AG_NT = 256;  // most threads per CTA

// Sizes and shared-memory layout of a launch.
struct AgShape {
    int N, S, M, J, Kc, kt, tpf, NP, KP;
    size_t z, s0, cf, pa, ct, tw, dc, bytes;
};

template <typename T> struct alignas(4 * sizeof(T)) Quad { T x, y, z, w; };

template <typename T>
AgShape ag_shape(int N, int n, int K) {
    typedef typename cvec<T>::type V;
    AgShape a;
    a.N = N;
    a.S = (N / 2) % 2 ? N : N + 2;  // rows an odd number of 16-byte units apart
    a.M = N / 2;
    a.J = (a.M - 1) / 2;
    a.Kc = a.M / 2 + 1;             // k = 0 .. M/2
    a.kt = (a.Kc + K - 1) / K;
    a.KP = a.kt * K;
    a.tpf = N * a.kt;               // threads at work
    a.NP = (N / 2 - 1) * N + 2 * (N / 2 + 1);
    auto up = [](size_t b) { return (b + 31) & ~size_t(31); };
    a.z = 0;
    a.s0 = up(a.z + size_t(N) * a.S * sizeof(V));
    a.cf = up(a.s0 + size_t(n) * n * sizeof(V));
    a.pa = up(a.cf + size_t(a.NP) * 4 * sizeof(T));
    a.ct = up(a.pa + size_t(a.NP) * sizeof(uint32_t));
    a.tw = up(a.ct + size_t(a.J + 1) * a.KP * sizeof(V));
    a.dc = up(a.tw + size_t(N) * sizeof(V));
    a.bytes = a.dc + size_t(N) * sizeof(V);
    return a;
}

// two adjacent cells (16-byte aligned pair)
__device__ __forceinline__ void load2(const float2* p, float2& a, float2& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void load2(const double2* p, double2& a, double2& b) {
    a = p[0];
    b = p[1];
}

// The sums of one line for k = k0 .. k0 + K - 1: P = sum a_j cos, Q = sum b_j
// sin of the even (e) and odd (o) elements.
template <typename V, int K> struct AgSums {
    V pe[K], qe[K], po[K], qo[K];
};

// x: the line's first cell; elements 1 (ROWS) or S cells apart. sum: the sum of
// all elements (FILL; ROWS: without the real part of the last one, which is
// also left out of the transform).
template <bool ROWS, bool FILL, typename V, int K>
__device__ __forceinline__ void ag_accumulate(const V* x, const AgShape& a, const V* ct, int k0, AgSums<V, K>& s, V& sum) {
    typedef decltype(V().x) T;
    const int st = ROWS ? 1 : a.S;
    V e, o;
    if (ROWS) load2(x, e, o);
    else e = x[0], o = x[st];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        s.pe[k] = e;
        s.po[k] = o;
        s.qe[k] = s.qo[k] = mk(T(0), T(0));
    }
    if (FILL) sum = cadd(e, o);
    const V* lo = x + 2 * st;
    const V* hi = x + 2 * (a.M - 1) * st;
    const V* c = ct + a.KP + k0;
#pragma unroll 1
    for (int j = 1; j <= a.J; ++j, lo += 2 * st, hi -= 2 * st, c += a.KP) {
        V ej, oj, em, om;
        if (ROWS) {
            load2(lo, ej, oj);
            load2(hi, em, om);
            if (FILL && j == 1) om.x = T(0);
        } else {
            ej = lo[0], oj = lo[st], em = hi[0], om = hi[st];
        }
        const V ae = cadd(ej, em), be = csub(ej, em), ao = cadd(oj, om), bo = csub(oj, om);
        if (FILL) sum = cadd(sum, cadd(ae, ao));
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const V w = c[k];
            s.pe[k] = mk(fmadd(ae.x, w.x, s.pe[k].x), fmadd(ae.y, w.x, s.pe[k].y));
            s.po[k] = mk(fmadd(ao.x, w.x, s.po[k].x), fmadd(ao.y, w.x, s.po[k].y));
            s.qe[k] = mk(fmadd(be.x, w.y, s.qe[k].x), fmadd(be.y, w.y, s.qe[k].y));
            s.qo[k] = mk(fmadd(bo.x, w.y, s.qo[k].x), fmadd(bo.y, w.y, s.qo[k].y));
        }
    }
    if ((a.M & 1) == 0) {  // the middle element of an even M: cos(pi k)
        if (ROWS) load2(x + a.M, e, o);
        else e = x[a.M * st], o = x[(a.M + 1) * st];
        if (FILL) sum = cadd(sum, cadd(e, o));
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool odd = (k0 + k) & 1;
            s.pe[k] = odd ? csub(s.pe[k], e) : cadd(s.pe[k], e);
            s.po[k] = odd ? csub(s.po[k], o) : cadd(s.po[k], o);
        }
    }
}

// Outputs of the line: f(position, value, slot), slot = 4 i + {0: k, 1: k + M,
// 2: M - k, 3: N - k}. FILL: plus d conj(w^k), the transform of a value d added
// to the last element.
template <bool INV, bool FILL, typename V, int K, typename Fn>
__device__ __forceinline__ void ag_outputs(const AgSums<V, K>& s, const AgShape& a, const V* tw, int k0, V d, Fn f) {
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const int k = k0 + i;
        if (k >= a.Kc) break;
        const V pe = s.pe[i], qe = s.qe[i], po = s.po[i], qo = s.qo[i];
        // p - i q and p + i q (exchanged for the inverse)
        const V em = mk(pe.x + qe.y, pe.y - qe.x), ep = mk(pe.x - qe.y, pe.y + qe.x);
        const V om = mk(po.x + qo.y, po.y - qo.x), op = mk(po.x - qo.y, po.y + qo.x);
        const V e1 = INV ? ep : em, e2 = INV ? em : ep, o1 = INV ? op : om, o2 = INV ? om : op;
        const V w1 = tw[k];
        V t = INV ? cmulc_rn(w1, o1) : cmul_rn(o1, w1);
        if (FILL) t = cadd(t, cmulc_rn(w1, d));
        f(k, cadd(e1, t), 4 * i);
        f(k + a.M, csub(e1, t), 4 * i + 1);
        if (k != 0 && 2 * k != a.M) {
            const V w2 = tw[a.M - k];
            t = INV ? cmulc_rn(w2, o2) : cmul_rn(o2, w2);
            if (FILL) t = cadd(t, cmulc_rn(w2, d));
            f(a.M - k, cadd(e2, t), 4 * i + 2);
            f(a.N - k, csub(e2, t), 4 * i + 3);
        }
    }
}

// Final filter (Eq. 2) over the (k, -k) pairs, one frame's threads.
template <typename T, typename V>
__device__ __forceinline__ void ag_final(V* Z, const Tables<T>& tab, const uint32_t* pa, const AgShape& a, int t) {
    const T half = T(0.5);
    for (int p = t; p < a.NP; p += a.tpf) {
        const int a1 = pa[p] & 0xFFFF, a2 = pa[p] >> 16, ky = a1 / a.S, kx = a1 - ky * a.S;
        const V z1 = Z[a1], z2 = Z[a2];
        const V ph = final_bin(z1, z2, tab.A[kx], tab.Tt[kx], tab.A[ky], tab.Tt[ky], half * tab.wfin[ky * a.N + kx]);
        Z[a2] = mk(ph.x, -ph.y);
        Z[a1] = ph;
    }
}

// Eq. PC in direct space, for the extended-slope output (one frame's threads):
// out[l] = (last x slope of row l, last y slope of column l). The grid is left
// as it is: the transforms apply the fill themselves.
template <typename T, typename V>
__device__ __forceinline__ void ag_fill_values(const V* Z, V* out, const AgShape& a, int t) {
    for (int l = t; l < a.N; l += a.tpf) {
        T sx = T(0), sy = T(0);
        for (int i = 0; i < a.N - 1; ++i) {
            sx += Z[l * a.S + i].x;
            sy += Z[i * a.S + l].y;
        }
        out[l] = mk(-sx, -sy);
    }
}

template <typename T, int K>
__global__ void __launch_bounds__(AG_NT, 2) anygrid_kernel(Params<T> p, AgShape a) {
    typedef typename cvec<T>::type V;
    extern __shared__ __align__(32) unsigned char smem_raw[];
    Quad<T>* const cf = reinterpret_cast<Quad<T>*>(smem_raw + a.cf);  // al, be, ga of a pair's first bin, al of its second
    uint32_t* const pa = reinterpret_cast<uint32_t*>(smem_raw + a.pa);  // its two cells
    V* const ct = reinterpret_cast<V*>(smem_raw + a.ct);  // [j][k]: cos, sin of 2 pi j k / M
    V* const tw = reinterpret_cast<V*>(smem_raw + a.tw);
    const int N = a.N, S = a.S, M = a.M, H = N / 2, n = p.n, off = p.off, nn = n * n;

    for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = p.tab.tw[i];
    for (int i = threadIdx.x; i < (a.J + 1) * a.KP; i += blockDim.x) {
        const int j = i / a.KP, k = i - j * a.KP;
        const V w = p.tab.tw[(2 * j * k) % N];
        ct[i] = mk(w.x, -w.y);
    }
    // pairs: rows ky = 1 .. N/2 - 1 with every kx, rows 0 and N/2 with kx = 0 ..
    // N/2 (their partners lie in the same row)
    for (int q = threadIdx.x; q < a.NP; q += blockDim.x) {
        int ky, kx;
        if (q < (H - 1) * N) {
            ky = 1 + q / N;
            kx = q % N;
        } else {
            const int r = q - (H - 1) * N;
            ky = r <= H ? 0 : H;
            kx = r <= H ? r : r - (H + 1);
        }
        const int my = ky == 0 ? 0 : N - ky, mx = kx == 0 ? 0 : N - kx;
        pa[q] = uint32_t(ky * S + kx) | uint32_t(my * S + mx) << 16;
        const T w = p.tab.iota[ky * N + kx];
        const T *u = p.tab.pt + 4 * kx, *v = p.tab.pt + 4 * ky, *un = p.tab.pt + 4 * mx, *vn = p.tab.pt + 4 * my;
        T al, be, ga, al2, none;
        lsq_coefs(w, u[0], u[1], T(0.5) * u[2], T(0.5) * u[3], quad<T>{v[0], v[1], v[2], v[3]}, al, be, ga);
        lsq_coefs(w, un[0], un[1], T(0.5) * un[2], T(0.5) * un[3], quad<T>{vn[0], vn[1], vn[2], vn[3]}, al2, none,
                  none);
        cf[q] = Quad<T>{al, be, ga, al2};
    }
    // roles: line, first k
    const int t = threadIdx.x;
    const bool act = t < a.tpf;
    const int line = t % N, k0 = (t / N) * K;
    V* const Z = reinterpret_cast<V*>(smem_raw + a.z);
    V* const s0 = reinterpret_cast<V*>(smem_raw + a.s0);
    V* const dc = reinterpret_cast<V*>(smem_raw + a.dc);
    // which of this thread's row outputs (ag_outputs' slots) are pupil cells
    uint32_t vbits = 0;
    const int li = line - off;
    if (li >= 0 && li < n) {
#pragma unroll
        for (int s = 0; s < 4 * K; ++s) {
            const int k = k0 + s / 4, q = s & 3;
            const int col = q == 0 ? k : q == 1 ? k + M : q == 2 ? M - k : N - k, j = col - off;
            if (k < a.Kc && j >= 0 && j < n && p.mask[li * n + j]) vbits |= 1u << s;
        }
    }
    V* const row = Z + line * S;
    V* const col = Z + line;
    const V* const s0r = s0 + li * n - off;  // dereferenced only under vbits
    const V zero = mk(T(0), T(0));
    const bool fill_first = fills_first(p.periodic, p.iters);
    __syncthreads();

    bool finite = true;
    for (int f = blockIdx.x; f < p.F; f += gridDim.x) {
        if (act) {
            const T* sl = p.slopes + size_t(f) * 2 * nn;
            const T* ext = p.ext_init ? p.ext_init + size_t(f) * 2 * N * N : nullptr;
            for (int c = t; c < nn; c += a.tpf) s0[c] = mk(sl[c], sl[nn + c]);
            for (int r = t / N; r < N; r += a.kt) {
                const int c = line, i = r - off, j = c - off;
                V v = ext ? mk(ext[r * N + c], ext[N * N + r * N + c]) : zero;
                // Eq. PC replaces the last row's y slopes (and the last column's x
                // slopes, which the row transforms leave out): what a warm start
                // holds there must not reach the column sums
                if (fill_first && r == N - 1) v.y = T(0);
                if (i >= 0 && i < n && j >= 0 && j < n && p.mask[i * n + j]) {
                    v = mk(sl[i * n + j], sl[nn + i * n + j]);
                    finite &= isfinite(v.x) && isfinite(v.y);
                }
                Z[r * S + c] = v;
            }
        }
        __syncthreads();
        for (int it = 0; it <= p.iters; ++it) {
            const bool final = it == p.iters;
            const bool fill = p.periodic == PERIODIC_BEFORE_EACH_FFT || (p.periodic == PERIODIC_FINAL_ONLY && final);
            if (final && p.ext_out) {
                if (act && fill) ag_fill_values<T>(Z, dc, a, t);
                __syncthreads();
                if (act) {
                    T* eo = p.ext_out + size_t(f) * 2 * N * N;
                    for (int r = t / N; r < N; r += a.kt) {
                        V z = Z[r * S + line];
                        if (fill && line == N - 1) z.x = dc[r].x;
                        if (fill && r == N - 1) z.y = dc[line].y;
                        eo[r * N + line] = z.x;
                        eo[N * N + r * N + line] = z.y;
                    }
                }
                if (!p.phase) break;
            }
            AgSums<V, K> s;
            V sum = zero;
            // ---- forward rows, x part of Eq. PC
            if (act) {
                if (fill) ag_accumulate<true, true>(row, a, ct, k0, s, sum);
                else ag_accumulate<true, false>(row, a, ct, k0, s, sum);
            }
            __syncthreads();
            if (act) {
                auto put = [&](int q, V v, int) { row[q] = v; };
                if (fill) ag_outputs<false, true>(s, a, tw, k0, mk(-sum.x, T(0)), put);
                else ag_outputs<false, false>(s, a, tw, k0, zero, put);
            }
            __syncthreads();
            // ---- forward columns, y part of Eq. PC
            if (act) {
                if (fill) {
                    ag_accumulate<false, true>(col, a, ct, k0, s, sum);
                    if (k0 == 0) dc[line] = sum;
                } else {
                    ag_accumulate<false, false>(col, a, ct, k0, s, sum);
                }
            }
            __syncthreads();
            if (act) {
                auto put = [&](int q, V v, int) { col[q * S] = v; };
                if (fill) {
                    // -i Sy(0, kx), Sy(0, kx) = (Z(0, kx) - conj Z(0, -kx)) / (2i)
                    const V z0 = dc[line], z0p = dc[line == 0 ? 0 : N - line];
                    ag_outputs<false, true>(s, a, tw, k0,
                                            mk(T(0.5) * (z0p.x - z0.x), T(-0.5) * (z0.y + z0p.y)), put);
                } else {
                    ag_outputs<false, false>(s, a, tw, k0, zero, put);
                }
            }
            __syncthreads();
            // ---- Algorithm 1 step 2, or the final filter
            if (act) {
                if (!final) {
#pragma unroll 4
                    for (int q = t; q < a.NP; q += a.tpf) {
                        const uint32_t ad = pa[q];
                        const Quad<T> c = cf[q];
                        const V z1 = Z[ad & 0xFFFF], z2 = Z[ad >> 16];
                        Z[ad >> 16] = lsq_apply(c.w, c.y, c.z, z2, z1);
                        Z[ad & 0xFFFF] = lsq_apply(c.x, c.y, c.z, z1, z2);
                    }
                } else {
                    ag_final(Z, p.tab, pa, a, t);
                }
            }
            __syncthreads();
            // ---- inverse columns
            if (act) ag_accumulate<false, false>(col, a, ct, k0, s, sum);
            __syncthreads();
            if (act) ag_outputs<true, false>(s, a, tw, k0, zero, [&](int q, V v, int) { col[q * S] = v; });
            __syncthreads();
            // ---- inverse rows; Algorithm 1 step 4: measured slopes back in the pupil
            if (act) ag_accumulate<true, false>(row, a, ct, k0, s, sum);
            __syncthreads();
            if (act) {
                if (!final)
                    ag_outputs<true, false>(s, a, tw, k0, zero, [&](int q, V v, int sl) {
                        if (vbits & (1u << sl)) v = s0r[q];
                        row[q] = v;
                    });
                else
                    ag_outputs<true, false>(s, a, tw, k0, zero, [&](int q, V v, int) { row[q] = v; });
            }
            __syncthreads();
        }
        if (act && p.phase) {
            T* ph = p.phase + size_t(f) * N * N;
            for (int r = t / N; r < N; r += a.kt) ph[r * N + line] = Z[r * S + line].x;
        }
        __syncthreads();
    }
    if (!finite) atomicOr(p.status, STATUS_NONFINITE);
}

// resident CTAs per SM and SM count, per (device, kernel, threads, shared memory)
struct AgLaunch {
    int dev, threads, sms, per_sm;
    const void* kern;
    size_t smem;
};

template <typename T> using AgKernel = void (*)(Params<T>, AgShape);

AgKernel<float> ag_kernel(float, int K) {
    switch (K) {
        case 3: return anygrid_kernel<float, 3>;
        case 4: return anygrid_kernel<float, 4>;
        case 5: return anygrid_kernel<float, 5>;
        case 6: return anygrid_kernel<float, 6>;
        default: return anygrid_kernel<float, 7>;
    }
}
AgKernel<double> ag_kernel(double, int K) { return K <= 3 ? anygrid_kernel<double, 3> : anygrid_kernel<double, 4>; }

// K: four threads per line, the shortest time for few frames (46^2, 10
// iterations, one frame: 68 us, 87 with two threads); many frames of the
// smaller grids take two (K up to 6: 1000 frames 290 us against 307; 26^2: 89
// against 106), the larger ones not (62^2: 617 against 539). FP64 keeps four
// (its sums take twice the registers). The phase of a frame is the same bits
// whichever is taken.
template <typename T> AgShape ag_choose(int N, int n, int F, int sms, int* K) {
    const int Kc = N / 4 + 1;
    const bool two = sizeof(T) == 4 && N <= 48 && F > 5 * sms / 2;
    *K = two ? (Kc + 1) / 2 : (Kc + 3) / 4;
    if (*K < 3) *K = 3;
    return ag_shape<T>(N, n, *K);
}

template <typename T>
cudaError_t launch_any(int N, const Params<T>& p, cudaStream_t s) {
    static std::mutex mu;
    static std::vector<AgLaunch> cache;
    if (N < 18 || N > 62 || (N & 1)) return cudaErrorInvalidValue;
    int dev = 0, sms = 0, per_sm = 0, K = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::unique_lock<std::mutex> lock(mu);
    for (const AgLaunch& c : cache)
        if (c.dev == dev) sms = c.sms;
    if (sms == 0 && (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const AgShape a = ag_choose<T>(N, p.n, p.F, sms, &K);
    const AgKernel<T> kern = ag_kernel(T(0), K);
    const void* k = reinterpret_cast<const void*>(kern);
    const int threads = (a.tpf + 31) / 32 * 32;
    for (const AgLaunch& c : cache)
        if (c.dev == dev && c.kern == k && c.threads == threads && c.smem == a.bytes) per_sm = c.per_sm;
    if (per_sm == 0) {
        // the limit is a property of the function: the most any launch needs
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, a.bytes)) != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        cache.push_back(AgLaunch{dev, threads, sms, per_sm, k, a.bytes});
    }
    lock.unlock();
    int grid = sms * per_sm;
    if (p.ctas > 0 && p.ctas < grid) grid = p.ctas;
    if (grid > p.F) grid = p.F;
    kern<<<grid, threads, a.bytes, s>>>(p, a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_anygrid_f32(int N, const Params<float>& p, cudaStream_t s) { return launch_any<float>(N, p, s); }
cudaError_t launch_anygrid_f64(int N, const Params<double>& p, cudaStream_t s) { return launch_any<double>(N, p, s); }

}  // namespace fwr
