// pfc_pair_slab.cu -- the packed FP32 sweep of a z-slab: the planes beyond the
// slab's ends come from its halo buffer instead of the periodic wrap.
#include "pfc_pair_kernel.cuh"

namespace pfc {

cudaError_t launch_pair_halo(Launch<float, 1>& L, int mode, int tile_y, int max_run, cudaStream_t s)
{
    return L.inst[0].C.nform ? launch_pair_mode<1, true, true>(L, mode, tile_y, max_run, s)
                           : launch_pair_mode<1, false, true>(L, mode, tile_y, max_run, s);
}

}  // namespace pfc
