// Launch arguments of the mixed-radix transforms, shared by their planner
// (helm_dft_mix.cu) and the kernels of each precision.
#pragma once

#include "helm_dft.h"
#include "helm_kernels.cuh"

namespace helm {

constexpr int kMixThreads = 256;  // largest CTA

struct MixArgs {
  MixPlan m;
  const void* tw;  // complex64: mix_tables of m; complex128: e^{-2 pi i k / m.n}
  const void* bw;  // chirp (Bluestein)
  const void* bf;  // its spectrum
};

// Shared memory a CTA can have; dft_supported accepts lengths of which it holds
// two bare lines.
constexpr size_t kMixSmem = 227 * 1024;
constexpr int kMixRoots = 64;  // a prime pass's roots beside the lines

// Lines per CTA, column slots, threads and exchange buffers of one launch.
struct MixShape {
  int L, lt, threads, nbuf;
};
MixShape mix_shape(const MixPlan& m, bool cols, size_t es, int64_t nlines, int64_t outer, int64_t inner);

// One launch (see helm_dft_mix.cuh), instantiated per precision T for rows
// and columns, with and without Bluestein.
template <typename T, bool COLS, bool BS>
cudaError_t run_mix(const MixArgs& a, int len, const void* in, int kind, void* out, int out_mode, int64_t nlines,
                    int64_t outer, int64_t inner, int sign, double scale, double accum_scale, const void* sc_in,
                    const void* sc_out, const int* skip, cudaStream_t st);

}  // namespace helm
