// The mixed-radix transforms in complex64.
#include "helm_dft_mix.cuh"

namespace helm {

template cudaError_t run_mix<float, false, false>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);
template cudaError_t run_mix<float, false, true>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);
template cudaError_t run_mix<float, true, false>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);
template cudaError_t run_mix<float, true, true>(const MixArgs&, int, const void*, int, void*, int, int64_t, int64_t,
                                          int64_t, int, double, double, const void*, const void*, const int*,
                                          cudaStream_t);

}  // namespace helm
