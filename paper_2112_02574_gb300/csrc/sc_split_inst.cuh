// Instantiation helper of the two-pass step: included by one translation unit per storage type.
#pragma once

#include "sc_dispatch.h"
#include "sc_step_split.cuh"

namespace scgb {

// A launch that may start while the launch before it in the stream drains (see pass_begin).
template <class... P, class... A>
cudaError_t launch_pass(void (*kernel)(P...), unsigned blocks, cudaStream_t stream, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(blocks);
  c.blockDim = dim3(kSplitThreads);
  c.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

template <class ST, class CT>
cudaError_t launch_split(int sten, const SplitArgs<CT> &m, cudaStream_t st) {
  const unsigned blocks = (unsigned)((m.a.N + kSplitThreads - 1) / kSplitThreads);
  cudaError_t e = launch_pass(sc_split_moments<ST, CT>, blocks, st, m);
  if (e != cudaSuccess) return e;
  return launch_pass(sten == kE6 ? sc_split_collide<kE6, ST, CT> : sc_split_collide<kE4, ST, CT>, blocks, st, m);
}

template <class ST, class CT>
cudaError_t launch_split_batch(int sten, const SplitArgs<CT> *args, const int2 *items, int nitems, int swap,
                               cudaStream_t st) {
  cudaError_t e = launch_pass(sc_split_moments_batched<ST, CT>, (unsigned)nitems, st, args, items, swap);
  if (e != cudaSuccess) return e;
  return launch_pass(sten == kE6 ? sc_split_collide_batched<kE6, ST, CT> : sc_split_collide_batched<kE4, ST, CT>,
                     (unsigned)nitems, st, args, items, swap);
}

}  // namespace scgb
