// Instantiations of the face-flux kernels for the 10-point TENO-AA scheme.
#include "teno_face.cuh"

namespace teno {

cudaError_t launch_chunk10(int nd, const SweepArgs &a, cudaStream_t s)
{
    if (nd == 1) return launch_chunk<1, 5>(a, s);
    if (nd == 2) return launch_chunk<2, 5>(a, s);
    return launch_chunk<3, 5>(a, s);
}

}  // namespace teno
