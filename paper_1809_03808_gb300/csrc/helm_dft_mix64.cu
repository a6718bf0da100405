// The mixed-radix transforms in complex128.
#include "helm_dft_mix.cuh"

namespace helm {

template cudaError_t run_mix<double, false, false>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);
template cudaError_t run_mix<double, false, true>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);
template cudaError_t run_mix<double, true, false>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);
template cudaError_t run_mix<double, true, true>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);

}  // namespace helm
