// Instantiations of the face-flux kernels for the 8-point TENO-AA scheme.
#include "teno_face.cuh"

namespace teno {

cudaError_t launch_chunk8(int nd, const SweepArgs &a, cudaStream_t s)
{
    if (nd == 1) return launch_chunk<1, 4>(a, s);
    if (nd == 2) return launch_chunk<2, 4>(a, s);
    return launch_chunk<3, 4>(a, s);
}

}  // namespace teno
