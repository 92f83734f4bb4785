// Instantiations of the face-flux kernels for the 12-point TENO-AA scheme.
#include "teno_face.cuh"

namespace teno {

cudaError_t launch_chunk12(int nd, const SweepArgs &a, cudaStream_t s)
{
    if (nd == 1) return launch_chunk<1, 6>(a, s);
    if (nd == 2) return launch_chunk<2, 6>(a, s);
    return launch_chunk<3, 6>(a, s);
}

}  // namespace teno
