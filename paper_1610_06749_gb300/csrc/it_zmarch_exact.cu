// it_zmarch_exact.cu -- the staged march's instances with compensated sums.
#include "it_zmarch.cuh"

namespace itk {

template cudaError_t zm_prepare_shape<true>(bool, int, int, bool, bool, size_t, int *);
template void zm_launch_shape<true>(bool, int, int, bool, bool, int, const ZmMaps &, const float *, const float *,
                                    float *, float *, int, int, int,
                                    const ZmConf &, const Coef<float> &, double *, int *, cudaStream_t);

}  // namespace itk
