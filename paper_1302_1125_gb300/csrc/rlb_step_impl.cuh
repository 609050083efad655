// rlb_step_impl.cuh -- launch configuration of the fused step kernel, shared
// by the FP64 and FP32-storage translation units.
#pragma once

#include "rlb_kernels.cuh"

namespace rlb {

// SMs of the current device (looked up once per device)
inline int sm_count()
{
    constexpr int kMaxDevices = 64;
    static int cache[kMaxDevices] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (dev < kMaxDevices && cache[dev] > 0) return cache[dev];
    int n = 1;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
    if (dev < kMaxDevices) cache[dev] = n;
    return n;
}

// Grids that the small-grid kernels take, unless the mapping asks for tiles (1;
// 3: FP32 tiles): fewer than 128 cells per SM, four blocks of 32 cells.  us a
// step on 152 SMs: 1-D 16.3 at 64 cells an SM, 25.8 at 96, 26.0 at 128 (tiles of
// 128 cells 33), 2-D 20.6, 30.2, 30.0 (45.6), 3-D 32.2 at 42, 33.8 at 96, 34.0 at
// 121 (56).  Under the 1-D reduction 80 cells per SM: five of its blocks fit on
// an SM, and up to two and a half to an SM those of the next step (which start
// while a step runs) all find room.  Beyond, the SMs that finish first take the
// rest, up to five to an SM: 15.0 at 79 cells per SM, 22.5 from 86 on (tiles 18.0).
inline bool f64_below(const StepParams &p, int cells_per_sm)
{
    return (long long)p.nx * p.ny * p.nz < (long long)cells_per_sm * sm_count();
}
inline bool f64_small(const StepParams &p) { return f64_below(p, p.sym == 1 ? 80 : 128) && p.mapping != 1 && p.mapping != 3; }

template <typename T, int DIM, bool EULER, int LAT, int NP>
cudaError_t launch_step_np(const StepParams &p, const T *f, const T *h, T *fo, T *ho, T *prev,
                          cudaStream_t s)
{
    const long long cells = (long long)p.nx * p.ny * p.nz;
    // Small grids: four warps to 32 cells (step_split_kernel); in Euler mode
    // blocks of one to four warps of consecutive cells (x-fastest order) spread
    // the cells over more SMs.
    int bs = 128;
    const bool small = f64_small(p);
    if constexpr (!EULER) {
        if (small)
            return launch_overlapped(step_split_kernel<DIM, LAT, NP>, unsigned((cells + 31) / 32), dim3(32, 4, 1), 0, s, p,
                                     f, h, fo, ho, prev);
    } else if (small) {
        const int nsm = sm_count();
        bs = int(((cells + nsm - 1) / nsm + 31) / 32 * 32);
        bs = bs < 32 ? 32 : (bs > 128 ? 128 : bs);
    }
    const unsigned nb = unsigned((cells + bs - 1) / bs);
    if constexpr (DIM == 1) {
        if constexpr (EULER) {
            // (whatever the mapping, so that its kernels agree bit for bit)
            if (f64_below(p, 128))
                return launch_overlapped(step_kernel<T, 1, true, LAT, false, NP, FX_NONE>, nb, bs, 0, s, p, f, h, fo, ho,
                                         prev);
        }
        return launch_overlapped(step_kernel<T, DIM, EULER, LAT, false, NP>, nb, bs, 0, s, p, f, h, fo, ho, prev);
    } else {
        // tiles of 32 x 4 cells when nx and ny fill them, else 128 consecutive
        // cells of the x-fastest order per block
        const long long tiles_x = (p.nx + 31) / 32, tiles_y = (p.ny + 3) / 4;
        const double fill = double(p.nx) * p.ny / double(tiles_x * 32 * tiles_y * 4);
        if (small || p.mapping == 2 || (p.mapping == 0 && fill < 0.97)) {
            return launch_overlapped(step_kernel<T, DIM, EULER, LAT, true, NP>, nb, bs, 0, s, p, f, h, fo, ho, prev);
        } else {
            const dim3 grid(unsigned(tiles_x), unsigned(tiles_y), p.nz);
            // (a block or less an SM: see FX_CALL)
            if constexpr (!EULER) {
                if (f64_below(p, 128))
                    return launch_overlapped(step_kernel<T, DIM, EULER, LAT, false, NP, FX_CALL>, grid, dim3(32, 4, 1), 0, s,
                                             p, f, h, fo, ho, prev);
            }
            return launch_overlapped(step_kernel<T, DIM, EULER, LAT, false, NP>, grid, dim3(32, 4, 1), 0, s, p, f, h, fo,
                                     ho, prev);
        }
    }
}

// the symmetry reductions (p.sym: 1 on 1-D grids, 2 on 2-D grids; viscous)
template <typename T, int DIM, bool EULER, int LAT>
cudaError_t launch_step_t(const StepParams &p, const T *f, const T *h, T *fo, T *ho, T *prev,
                          cudaStream_t s)
{
    if constexpr (DIM == 1 && !EULER) {
        if (p.sym == 1) return launch_step_np<T, 1, false, LAT, 7>(p, f, h, fo, ho, prev, s);
    }
    if constexpr (DIM == 2 && !EULER) {
        if (p.sym == 2) return launch_step_np<T, 2, false, LAT, 14>(p, f, h, fo, ho, prev, s);
    }
    return launch_step_np<T, DIM, EULER, LAT, 19>(p, f, h, fo, ho, prev, s);
}

template <typename T, int LAT>
cudaError_t launch_step_lat(const StepParams &p, int dim, int euler, const T *f, const T *h, T *fo, T *ho,
                            T *prev, cudaStream_t s)
{
    if (euler) {
        if (dim == 1) return launch_step_t<T, 1, true, LAT>(p, f, h, fo, ho, prev, s);
        if (dim == 2) return launch_step_t<T, 2, true, LAT>(p, f, h, fo, ho, prev, s);
        return launch_step_t<T, 3, true, LAT>(p, f, h, fo, ho, prev, s);
    }
    if (dim == 1) return launch_step_t<T, 1, false, LAT>(p, f, h, fo, ho, prev, s);
    if (dim == 2) return launch_step_t<T, 2, false, LAT>(p, f, h, fo, ho, prev, s);
    return launch_step_t<T, 3, false, LAT>(p, f, h, fo, ho, prev, s);
}

template <typename T>
cudaError_t launch_step_any(const StepParams &p, int dim, int euler, const T *f, const T *h, T *fo,
                            T *ho, T *prev, cudaStream_t s)
{
    if (p.lat == 1) return launch_step_lat<T, 1>(p, dim, euler, f, h, fo, ho, prev, s);
    return launch_step_lat<T, 0>(p, dim, euler, f, h, fo, ho, prev, s);
}

}  // namespace rlb
