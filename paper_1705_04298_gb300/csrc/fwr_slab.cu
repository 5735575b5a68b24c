// Gerchberg kernel for 256^2 and 512^2 grids (sm_103a): kernels and launchers. The
// slab-streamed device code is in fwr_slab.cuh.

#include <cuda_runtime.h>
#include <stdint.h>

#include "fwr_internal.h"

namespace fwr {

#include "fwr_fft.cuh"
#include "fwr_slab.cuh"

template <int N, int GROUPS>
__global__ void __launch_bounds__(SNT, 1)
slab_kernel(Params<float> p, float2* scratch) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_bad;
    if (threadIdx.x == 0) s_bad = 0;
    SlabCtx c;
    slab_setup<N>(c, smem, p.tab, p.mask, p.n, p.off, p.periodic);
    float2* G = scratch + size_t(blockIdx.x) * N * N;
    const int nn = p.n * p.n;
    bool finite = true;
    for (int f = blockIdx.x; f < p.F; f += gridDim.x) {
        finite &= slab_frame<N, GROUPS>(c, p.tab, p.slopes + size_t(f) * 2 * nn,
                                        p.ext_init ? p.ext_init + size_t(f) * 2 * N * N : nullptr,
                                        p.phase + size_t(f) * N * N, p.iters, G, p.hud);
        __syncthreads();
    }
    if (!finite) atomicOr(&s_bad, 1);
    __syncthreads();
    if (threadIdx.x == 0 && s_bad) atomicOr(p.status, STATUS_NONFINITE);
}

// Few frames: a team of CTAs per frame. One frame's phases have too little
// arithmetic and too few bytes in flight for more than one SM's share, and the
// other SMs idle; the exchange through L2 is the same whoever does the slabs.
// The grid is whole teams, all resident (a cooperative launch); bitwise the
// results of slab_kernel (each line's and each bin's arithmetic is the same).
// After a barrier's wait ran out (STATUS_TIMEOUT) the plan's team launches do
// nothing until the status has been read, which also resets the counters.
template <int N>
__global__ void __launch_bounds__(SNT, 1)
slab_team_kernel(Params<float> p, float2* scratch, unsigned* counters, int team) {
    extern __shared__ __align__(16) unsigned char smem[];
    if (*reinterpret_cast<volatile unsigned*>(p.status) & STATUS_TIMEOUT) return;
    SlabCtx c;
    slab_setup<N>(c, smem, p.tab, p.mask, p.n, p.off, p.periodic);
    const int teams = int(gridDim.x) / team, id = int(blockIdx.x) % teams, rank = int(blockIdx.x) / teams;
    float2* G = scratch + size_t(id) * N * N;
    TeamBar bar{counters + id * TEAM_COUNTER_STRIDE, 0u, team, p.team_wait, false};
    const int nn = p.n * p.n;
    bool finite = true;
    for (int f = id; f < p.F && !bar.dead; f += teams)
        finite &= slab_frame<N, 2, true>(c, p.tab, p.slopes + size_t(f) * 2 * nn,
                                         p.ext_init ? p.ext_init + size_t(f) * 2 * N * N : nullptr,
                                         p.phase + size_t(f) * N * N, p.iters, G, p.hud, rank, &bar);
    if (!bar.dead) team_leave(bar);
    if (!finite) atomicOr(p.status, STATUS_NONFINITE);
    if (bar.dead && threadIdx.x == 0) atomicOr(p.status, STATUS_TIMEOUT);
}

namespace {

typedef void (*SlabKernel)(Params<float>, float2*);
typedef void (*SlabTeamKernel)(Params<float>, float2*, unsigned*, int);

// the kernel of grid N and a shape (1 or 2 warp groups; 0 is 2) with its
// shared-memory limit raised for n lenslets
cudaError_t slab_kernel_for(int N, int shape, int n, SlabKernel* k) {
    if (N == 512) *k = shape == 1 ? slab_kernel<512, 1> : slab_kernel<512, 2>;
    else *k = shape == 1 ? slab_kernel<256, 1> : slab_kernel<256, 2>;
    return raise_smem_limit(*k, slab_layout_bytes_n(N, n));
}

}  // namespace

size_t slab_smem_bytes(int N, int n) { return slab_layout_bytes_n(N, n); }

size_t slab_scratch_elems_per_cta(int N) { return size_t(N) * N; }

size_t slab_counter_bytes(int max_ctas) { return size_t(max_ctas) * TEAM_COUNTER_STRIDE * sizeof(unsigned); }

int slab_max_ctas() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    return sms;
}

namespace {

// CTAs per frame. Cost of one wave of teams that fills the SMs (us, 128 x 128
// on 256^2 and 200 x 200 on 512^2 lenslets, five iterations, 152 SMs; 1 is
// slab_kernel; 8 and 32 slabs, two per CTA and step): a wave takes the same
// time with fewer frames, so the least number of waves times their cost wins.
// At 512^2 teams of 8 also win for many frames: 19 grids of 2 MB in flight stay
// in L2, 152 do not. Measured with / without teams: 256^2, F = 1: 142 / 398,
// F = 38: 157 / 398, F = 200: 753 / 855; 512^2, F = 1: 181 / 2043, F = 16: 312 /
// 2047, F = 76: 1238 / 2470, F = 152: 2475 / 2741. Several calls at once: 256^2,
// 8 of F = 1: 157 / 406, 2 of F = 38: 314 / 402, 4 of F = 38: 631 / 461; 512^2, 8 of
// F = 16: 2559 / 2647.
int team_size(int N, int F, int ctas) {
    struct Cost {
        int team, us;
    };
    static const Cost c256[] = {{1, 460}, {2, 259}, {4, 160}};
    static const Cost c512[] = {{1, 2749}, {2, 1370}, {3, 937}, {4, 638}, {6, 443}, {8, 316}, {16, 186}};
    const Cost* c = N == 512 ? c512 : c256;
    const int nc = N == 512 ? 7 : 3;
    int best = 1;
    long long least = 0;
    for (int i = 0; i < nc; ++i) {
        const int teams = ctas / c[i].team;
        if (teams < 1) continue;
        const long long us = (long long)((F + teams - 1) / teams) * c[i].us;
        if (i == 0 || us < least) {
            least = us;
            best = c[i].team;
        }
    }
    return best;
}

cudaError_t launch_team(int N, int team, const Params<float>& p, float2* scratch, unsigned* counters, int max_ctas,
                        cudaStream_t s) {
    const SlabTeamKernel kern = N == 512 ? slab_team_kernel<512> : slab_team_kernel<256>;
    const size_t smem = slab_smem_bytes(N, p.n);
    cudaError_t e = raise_smem_limit(kern, smem);
    if (e != cudaSuccess) return e;
    int teams = max_ctas / team;
    if (p.F < teams) teams = p.F;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(teams * team));
    cfg.blockDim = dim3(SNT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p, scratch, counters, team);
}

}  // namespace

cudaError_t launch_slab(int N, const Params<float>& p, float2* scratch, unsigned* counters, int max_ctas,
                        cudaStream_t s) {
    if (N != 256 && N != 512) return cudaErrorInvalidValue;
    if (!p.one_cta && p.l2_bytes == 0) {
        const int team = team_size(N, p.F, max_ctas);
        if (team > 1) {
            cudaError_t e = launch_team(N, team, p, scratch, counters, max_ctas, s);
            // fewer SMs to this context than the device has: one CTA per frame
            if (e != cudaErrorCooperativeLaunchTooLarge) return e;
            cudaGetLastError();
        }
    }
    SlabKernel kern = nullptr;
    cudaError_t e = slab_kernel_for(N, p.shape, p.n, &kern);
    if (e != cudaSuccess) return e;
    int grid = max_ctas;
    if (p.ctas > 0 && p.ctas < grid) grid = p.ctas;
    if (grid > p.F) grid = p.F;
    if (grid < 1) return cudaErrorInvalidConfiguration;
    if (p.l2_bytes == 0) {
        kern<<<grid, SNT, slab_smem_bytes(N, p.n), s>>>(p, scratch);
        return cudaGetLastError();
    }
    // the scratch's lines persist in L2 (the context's set-aside holds them)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(SNT);
    cfg.dynamicSmemBytes = slab_smem_bytes(N, p.n);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
    attr[0].val.accessPolicyWindow.base_ptr = scratch;
    attr[0].val.accessPolicyWindow.num_bytes = p.l2_bytes;
    attr[0].val.accessPolicyWindow.hitRatio = p.l2_hit;
    attr[0].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
    attr[0].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p, scratch);
}

// ---------------------------------------------------------------------------
// Variant without any allocation: the scratch is this file-scope array, sized
// for STATIC_SLAB_GRIDS concurrent frames (8 MB). It exists on every GPU that
// loads the library, for the life of the process.
// ---------------------------------------------------------------------------
static __device__ __align__(256) float2 g_static_slab_scratch[STATIC_SLAB_GRIDS * 256 * 256];

// Host code cannot use the array's name as a device address: look the address
// up with the device current (this also loads the module on that device, so a
// later call does no loading) and raise the kernel's shared-memory limit.
cudaError_t static_slab_prepare(int n, float2** addr) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_slab_scratch);
    if (e != cudaSuccess) return e;
    SlabKernel kern = nullptr;
    if ((e = slab_kernel_for(256, 1, n, &kern)) != cudaSuccess || (e = slab_kernel_for(256, 2, n, &kern)) != cudaSuccess)
        return e;
    *addr = static_cast<float2*>(ptr);
    return cudaSuccess;
}

cudaError_t launch_slab_static(const Params<float>& p, float2* scratch, int ctas, cudaStream_t s) {
    if (ctas < 1 || ctas > STATIC_SLAB_GRIDS || !scratch) return cudaErrorInvalidValue;
    const int grid = ctas < p.F ? ctas : p.F;
    auto kern = p.shape == 1 ? slab_kernel<256, 1> : slab_kernel<256, 2>;
    kern<<<grid, SNT, slab_smem_bytes(256, p.n), s>>>(p, scratch);
    return cudaGetLastError();
}

}  // namespace fwr
