// The persistent tube kernel with the 7 classes of the 1-D symmetry reduction, in a
// unit of its own so that the two compile in parallel.
#include "rlb_batch.cuh"

namespace rlb {
namespace batch {

cudaError_t launch_tubes_7(const Args &a, int threads, int bound, int cluster, cudaStream_t s, int *nclusters_out)
{
    return launch_np<7>(a, threads, bound, cluster, s, nclusters_out);
}

}  // namespace batch
}  // namespace rlb
