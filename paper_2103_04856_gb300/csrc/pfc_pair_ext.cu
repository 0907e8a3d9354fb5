// pfc_pair_ext.cu -- the packed FP32 sweep with the Sec. 5.2 extensions: the
// orientation term, and coefficients from a field c(x).
#include "pfc_pair_kernel.cuh"

namespace pfc {

cudaError_t launch_pair_ext(Launch<float, 1>& L, int mode, int max_run, cudaStream_t s)
{
    const Inst<float>& in = L.inst[0];
    if (in.halo) return in.cf ? cudaErrorInvalidValue : launch_pair_ext_mode<true, 1>(L, mode, max_run, s);
    return in.cf ? launch_pair_ext_mode<false, 2>(L, mode, max_run, s) : launch_pair_ext_mode<false, 1>(L, mode, max_run, s);
}

}  // namespace pfc
