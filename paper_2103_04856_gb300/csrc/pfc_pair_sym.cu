// pfc_pair_sym.cu -- the packed FP32 sweep for launches whose problems all
// have c3 = c5 = 0 (polynomials symmetric in kappa1, kappa2): the sqrt(D+)
// terms of eq. Feps have weight c3 T + c5 q = 0 there and are not compiled in.
// Its own translation unit, so that the instantiations build in parallel.
#include "pfc_pair_kernel.cuh"

namespace pfc {

template <int MAXI>
cudaError_t launch_pair_sym(Launch<float, MAXI>& L, int mode, int tile_y, int max_run, cudaStream_t s)
{
    return launch_pair_mode<MAXI, true, false>(L, mode, tile_y, max_run, s);
}
template cudaError_t launch_pair_sym<1>(Launch<float, 1>&, int, int, int, cudaStream_t);
template cudaError_t launch_pair_sym<BATCH_MAX>(Launch<float, BATCH_MAX>&, int, int, int, cudaStream_t);

}  // namespace pfc
