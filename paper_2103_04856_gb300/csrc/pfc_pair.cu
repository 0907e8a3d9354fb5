// pfc_pair.cu -- the packed FP32 sweep for general polynomials.
#include "pfc_pair_kernel.cuh"

namespace pfc {

template <int MAXI>
cudaError_t launch_pair(Launch<float, MAXI>& L, int mode, int tile_y, int max_run, cudaStream_t s)
{
    return launch_pair_mode<MAXI, false, false>(L, mode, tile_y, max_run, s);
}
template cudaError_t launch_pair<1>(Launch<float, 1>&, int, int, int, cudaStream_t);
template cudaError_t launch_pair<BATCH_MAX>(Launch<float, BATCH_MAX>&, int, int, int, cudaStream_t);

}  // namespace pfc
