// Two-pass step instantiations: FP16 storage.
#include "sc_split_inst.cuh"
cudaError_t scgb::launch_split_f16(int stencil, const SplitArgs<float> &m, cudaStream_t st) {
  return launch_split<__half, float>(stencil, m, st);
}
cudaError_t scgb::launch_split_batch_f16(int stencil, const SplitArgs<float> *args, const int2 *items, int nitems,
                                         int swap, cudaStream_t st) {
  return launch_split_batch<__half, float>(stencil, args, items, nitems, swap, st);
}
