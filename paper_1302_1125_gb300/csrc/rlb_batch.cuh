// rlb_batch.cuh -- the batched form of the FP32-storage step: B independent
// 1-D tubes (zero-gradient ends, Sec. III), each with its own length, eta/s
// and bulk coefficient, advanced by one persistent launch.
//
// Work division.  A cluster of C blocks (C = 1: one block) takes a job, one
// tube or a few consecutive tubes of similar length, and runs all of the
// job's steps; its C x blockDim threads split the job's cell pairs and meet
// at a barrier after each step (the block barrier for C = 1, the hardware
// cluster barrier otherwise).  No block ever waits on a block outside its
// own cluster, so there is no grid-wide barrier and no software spin.  Jobs
// are assigned to clusters on the host, longest first, each to the least
// loaded cluster; the grid holds exactly as many clusters as fit on the GPU
// at once.
#pragma once

#include "rlb_step_f32.cuh"

namespace rlb {
namespace batch {

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ unsigned cluster_index()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}

// hardware barrier over every thread of the cluster; release/acquire order
// each thread's earlier global stores before the other blocks' later loads
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// the x stencil of the pair (x0, x0 + 1) of a tube of nx cells stored at `off`
// (zero-gradient at both ends; an odd tube's last pair holds one pad cell):
// distances of the pairs it takes for x0-2 and x0+2, and the fix-ups
__device__ __forceinline__ void tube_ends(int nx, int x0, int &ol, int &orr, unsigned &xfix)
{
    ol = -2;
    orr = 2;
    xfix = 0u;
    if (x0 == 0) {
        ol = 0;
        xfix |= f32::XF_LO_CLAMP;
    }
    if (x0 + 2 >= nx) {
        orr = 0;
        xfix |= x0 + 1 < nx ? f32::XF_HI_CLAMP : f32::XF_HI_ODD1;
    } else if (x0 + 3 == nx) {
        xfix |= f32::XF_HI_ODD3;
    }
}

// Populations in blocks of 32 cells and stencils straight into registers, as
// on grids (f32::BlockIO); plain loads, which after the block or cluster
// barrier see what the other threads of the cluster wrote in the step before.
// MAXT = launch bound: 512 caps the kernel at 128 registers, 384 at 168, 256
// leaves it unconstrained (147; none spills); the autotuner picks.
template <int MAXT, int NP>
__global__ void __launch_bounds__(MAXT, 1) tubes_kernel(const Args a)
{
    __shared__ int s_off[kMaxJobTubes], s_nx[kMaxJobTubes], s_steps[kMaxJobTubes], s_par[kMaxJobTubes];
    __shared__ int s_tube[kMaxJobTubes], s_p0[kMaxJobTubes + 1];
    __shared__ float s_eos[kMaxJobTubes], s_kb[kMaxJobTubes];
    extern __shared__ f2 s_dyn[];   // parked coefficients (see update_pair)

    const int C = a.cluster;
    const unsigned rank = C > 1 ? cluster_rank() : 0u;
    const int cid = C > 1 ? int(cluster_index()) : int(blockIdx.x);
    if (cid >= a.nclusters) return;   // uniform over the cluster
    const int stride = C * int(blockDim.x);
    const int base = int(rank) * int(blockDim.x) + int(threadIdx.x);

    for (int j = a.cl_start[cid]; j < a.cl_start[cid + 1]; ++j) {
        const Job J = a.jobs[j];
        __syncthreads();   // the previous job's readers of the tables are done
        if (int(threadIdx.x) < J.count) {
            const int t = a.order[J.first + threadIdx.x];
            const Tube T = a.tubes[t];
            s_tube[threadIdx.x] = t;
            s_off[threadIdx.x] = T.off;
            s_nx[threadIdx.x] = T.nx;
            s_eos[threadIdx.x] = T.eos;
            s_kb[threadIdx.x] = T.kb;
            s_steps[threadIdx.x] = a.steps[t];
            s_par[threadIdx.x] = a.par[t];
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int acc = 0;
            for (int i = 0; i < J.count; ++i) {
                s_p0[i] = acc;
                acc += (s_nx[i] + 1) >> 1;
            }
            s_p0[J.count] = acc;
        }
        __syncthreads();

        for (int s = 0; s < J.steps; ++s) {
            for (int q = base; q < J.pairs; q += stride) {
                int i = 0;
                while (i + 1 < J.count && q >= s_p0[i + 1]) ++i;
                if (s < s_steps[i]) {
                    const int x0 = 2 * (q - s_p0[i]), i0 = s_off[i] + x0, nx = s_nx[i];
                    const bool odd = ((s_par[i] + s) & 1) != 0;
                    const char *src = reinterpret_cast<const char *>(odd ? a.f1 : a.f0);
                    char *dst = reinterpret_cast<char *>(odd ? a.f0 : a.f1);
                    auto at = [](int k) { return sizeof(float) * f32::blk_at(k); };
                    f32::BlockIO<1, false, NP, 0, false> io{a.p};
                    int ol, orr;
                    tube_ends(nx, x0, ol, orr, io.xfix);
                    io.c = src + at(i0);
                    io.l = src + at(i0 + ol);
                    io.r = src + at(i0 + orr);
                    io.o = dst + at(i0);
                    io.pv = a.prev + f32::blk_prev_at(i0);
                    io.kb = s_kb[i];
                    // the slots of the shared-memory array are MAXT apart (the
                    // launch bound, a compile-time constant: fixed offsets
                    // from one base address), whatever blockDim.x <= MAXT is
                    f32::update_pair<false, f32::EQ_FOLD, NP, 0, false>(a.p, io, x0 + 1 < nx, s_eos[i], s_dyn + threadIdx.x, MAXT);
                }
            }
            if (C > 1) cluster_barrier();
            else __syncthreads();
        }
        if (rank == 0 && int(threadIdx.x) < J.count)
            a.par[s_tube[threadIdx.x]] = (s_par[threadIdx.x] + s_steps[threadIdx.x]) & 1;
    }
}

template <int MAXT, int NP>
cudaError_t launch_variant(const Args &a, int threads, int cluster, cudaStream_t s, int *nclusters_out)
{
    auto kern = tubes_kernel<MAXT, NP>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nclusters_out ? unsigned(cluster) : unsigned(a.nclusters * cluster), 1, 1);
    cfg.blockDim = dim3(unsigned(threads), 1, 1);
    const size_t smem = f32::park_bytes(MAXT, 1);   // slots MAXT apart
    cfg.dynamicSmemBytes = smem;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
    }
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    if (cluster > 1) {
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = unsigned(cluster);
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
    if (nclusters_out) {
        if (cluster > 1) return cudaOccupancyMaxActiveClusters(nclusters_out, kern, &cfg);
        int per_sm = 0, dev = 0, sms = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (e == cudaSuccess) e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        *nclusters_out = per_sm * sms;
        return e;
    }
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int NP>
cudaError_t launch_np(const Args &a, int threads, int bound, int cluster, cudaStream_t s, int *nclusters_out)
{
    if (threads < 32 || threads > bound || threads % 32 != 0) return cudaErrorInvalidValue;
    if (bound == 256) return launch_variant<256, NP>(a, threads, cluster, s, nclusters_out);
    if (bound == 384) return launch_variant<384, NP>(a, threads, cluster, s, nclusters_out);
    if (bound == 512) return launch_variant<512, NP>(a, threads, cluster, s, nclusters_out);
    return cudaErrorInvalidValue;
}

}  // namespace batch
}  // namespace rlb
