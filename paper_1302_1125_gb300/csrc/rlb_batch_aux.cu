// Batched tubes: initialisation, macroscopic output and per-tube totals over
// the tube storage (packed fields in, packed fields out), and the dispatch of
// the persistent step kernel.
#include "rlb_cellops_f32.cuh"
#include "rlb_kernels.cuh"
#include "rlb_internal.h"

namespace rlb {
namespace batch {

cudaError_t launch_tubes(const Args &a, int threads, int bound, int cluster, cudaStream_t s,
                         int *nclusters_out)
{
    if (cluster < 1 || cluster > 8) return cudaErrorInvalidValue;
    return a.np == 7 ? launch_tubes_7(a, threads, bound, cluster, s, nclusters_out)
                     : launch_tubes_19(a, threads, bound, cluster, s, nclusters_out);
}

// tubes are stored in blocks of 32 cells, 38 populations each (f, then h)
constexpr long long kStep = f32::kBlk;            // floats between populations
constexpr int kH = 19 * f32::kBlk;                // from f to h

// grid (ceil(max_nx / 256), B): cells x0 = 2 t and x0 + 1 of tube blockIdx.y
__global__ void tubes_init_kernel(const Tube *__restrict__ tubes, const long long *__restrict__ pack,
                                  const double *__restrict__ n, const double *__restrict__ T,
                                  const double *__restrict__ ux, float *__restrict__ f,
                                  float *__restrict__ prev, unsigned *status)
{
    const int b = blockIdx.y;
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const Tube t = tubes[b];
    if (x0 >= t.nx) return;
    const bool has1 = x0 + 1 < t.nx;
    const long long s0 = pack[b] + x0, d0 = (long long)f32::blk_at(t.off + x0), p0 = (long long)f32::blk_prev_at(t.off + x0);
    const f32::CellPair c{s0, has1 ? s0 + 1 : s0, d0, d0 + 1, has1, p0, p0 + 1};
    f32::init_pair<0, true>(c, kStep, n, T, ux, nullptr, nullptr, f, f + kH, prev, status);
}

__global__ void tubes_macro_kernel(const Tube *__restrict__ tubes, const long long *__restrict__ pack,
                                   const int *__restrict__ par, long long total,
                                   const float *__restrict__ f0, const float *__restrict__ f1,
                                   double *__restrict__ out, unsigned *status)
{
    const int b = blockIdx.y;
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const Tube t = tubes[b];
    if (x0 >= t.nx) return;
    const bool has1 = x0 + 1 < t.nx;
    const bool one = par[b] != 0;
    const long long s0 = (long long)f32::blk_at(t.off + x0), d0 = pack[b] + x0;
    const float *f = one ? f1 : f0;
    const f32::CellPair c{s0, has1 ? s0 + 1 : s0, d0, d0 + 1, has1, 0, 0};
    f32::macro_pair<0, true>(c, kStep, f, f + kH, out, total, status);
}

// class of population i under the 1-D symmetry reduction, as the plane of
// its representative: rest, +x, -x, y/z axis, x+ diagonals, x- diagonals,
// y-z diagonals
__device__ __forceinline__ int class_plane(int i)
{
    if (i < 3) return i;
    if (i < 7) return 3;
    if (i >= 15) return 15;
    const int j = (i - 7) & 3;   // 7..10 and 11..14: signs (+,+) (+,-) (-,+) (-,-)
    return j < 2 ? 7 : 9;
}

__global__ void tubes_expand_kernel(const Tube *__restrict__ tubes, const int *__restrict__ par,
                                    float *__restrict__ f0, float *__restrict__ f1)
{
    const int b = blockIdx.y;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const Tube t = tubes[b];
    if (x >= t.nx) return;
    const bool one = par[b] != 0;
    float *f = one ? f1 : f0, *h = f + kH;
    const long long idx = (long long)f32::blk_at(t.off + x), ps = kStep;
    for (int i = 3; i < 19; ++i) {
        const int r = class_plane(i);
        if (r == i) continue;
        f[i * ps + idx] = f[r * ps + idx];
        h[i * ps + idx] = h[r * ps + idx];
    }
}

// one block per tube, fixed reduction order (deterministic)
constexpr int kTubeTotBlock = 256;
__global__ void __launch_bounds__(kTubeTotBlock) tubes_totals_kernel(const Tube *__restrict__ tubes,
                                                                     const int *__restrict__ par,
                                                                     const float *__restrict__ f0,
                                                                     const float *__restrict__ f1,
                                                                     double *__restrict__ out)
{
    const int b = blockIdx.x;
    const Tube t = tubes[b];
    const bool one = par[b] != 0;
    const float *f = one ? f1 : f0, *h = f + kH;
    constexpr long long ps = kStep;
    double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    for (int x = threadIdx.x; x < t.nx; x += blockDim.x) {
        const long long idx = (long long)f32::blk_at(t.off + x);
        for_pops(RLB_POPS, [&](auto ic) {
            constexpr int I = decltype(ic)::value;
            const double fv = double(f[I * ps + idx]);
            acc[0] += kXi0Sq * fv;
            if constexpr (cdir<I, 0>() != 0) acc[1] += kXi0 * double(cdir<I, 0>()) * fv;
            if constexpr (cdir<I, 1>() != 0) acc[2] += kXi0 * double(cdir<I, 1>()) * fv;
            if constexpr (cdir<I, 2>() != 0) acc[3] += kXi0 * double(cdir<I, 2>()) * fv;
            acc[4] += kXi0 * double(h[I * ps + idx]);
        });
    }
    __shared__ double sm[5][kTubeTotBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        double v = acc[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) sm[k][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        double v = 0.0;
        for (int w = 0; w < kTubeTotBlock / 32; ++w) v += sm[threadIdx.x][w];
        out[5 * (long long)b + threadIdx.x] = v;
    }
}

cudaError_t launch_tubes_init(int B, int max_nx, const Tube *tubes, const long long *pack, const double *n,
                              const double *T, const double *ux, float *f, float *prev, unsigned *status, cudaStream_t s)
{
    const dim3 grid((max_nx + 255) / 256, B, 1);
    tubes_init_kernel<<<grid, 128, 0, s>>>(tubes, pack, n, T, ux, f, prev, status);
    return cudaGetLastError();
}

cudaError_t launch_tubes_macro(int B, int max_nx, const Tube *tubes, const long long *pack, const int *par,
                               long long total, const float *f0, const float *f1, double *out, unsigned *status,
                               cudaStream_t s)
{
    const dim3 grid((max_nx + 255) / 256, B, 1);
    tubes_macro_kernel<<<grid, 128, 0, s>>>(tubes, pack, par, total, f0, f1, out, status);
    return cudaGetLastError();
}

cudaError_t launch_tubes_expand(int B, int max_nx, const Tube *tubes, const int *par, float *f0, float *f1,
                                cudaStream_t s)
{
    const dim3 grid((max_nx + 127) / 128, B, 1);
    tubes_expand_kernel<<<grid, 128, 0, s>>>(tubes, par, f0, f1);
    return cudaGetLastError();
}

cudaError_t launch_tubes_totals(int B, const Tube *tubes, const int *par, const float *f0,
                                const float *f1, double *out,
                                cudaStream_t s)
{
    tubes_totals_kernel<<<B, kTubeTotBlock, 0, s>>>(tubes, par, f0, f1, out);
    return cudaGetLastError();
}

}  // namespace batch
}  // namespace rlb
