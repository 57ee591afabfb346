// Instantiation helper of the two-pass step: included by one translation unit per storage type.
#pragma once

#include "sc_step_inst.cuh"
#include "sc_step_split.cuh"

namespace scgb {

template <class ST, class CT>
cudaError_t launch_split(int sten, const SplitArgs<CT> &m, cudaStream_t st) {
  const unsigned blocks = (unsigned)((m.a.N + kSplitThreads - 1) / kSplitThreads);
  cudaError_t e = launch_pass(sc_split_moments<ST, CT>, blocks, kSplitThreads, 0, st, m);
  if (e != cudaSuccess) return e;
  auto *collide = sten == kE6 ? sc_split_collide<kE6, ST, CT, false> : sc_split_collide<kE4, ST, CT, false>;
  if constexpr (sizeof(CT) == 4)  // FP64 has one register budget
    if (m.a.self_on && m.a.N <= kSmallCollide)
      collide = sten == kE6 ? sc_split_collide<kE6, ST, CT, true> : sc_split_collide<kE4, ST, CT, true>;
  return launch_pass(collide, blocks, kSplitThreads, 0, st, m);
}

template <class ST, class CT>
cudaError_t launch_split_batch(int sten, const SplitArgs<CT> *args, const int2 *items, int nitems, int swap,
                               cudaStream_t st) {
  cudaError_t e = launch_pass(sc_split_moments_batched<ST, CT>, nitems, kSplitThreads, 0, st, args, items, swap);
  if (e != cudaSuccess) return e;
  return launch_pass(sten == kE6 ? sc_split_collide_batched<kE6, ST, CT> : sc_split_collide_batched<kE4, ST, CT>,
                     nitems, kSplitThreads, 0, st, args, items, swap);
}

}  // namespace scgb
