// Two-pass step instantiations: FP32 storage.
#include "sc_split_inst.cuh"
cudaError_t scgb::launch_split_f32(int stencil, const SplitArgs<float> &m, cudaStream_t st) {
  return launch_split<float, float>(stencil, m, st);
}
cudaError_t scgb::launch_split_batch_f32(int stencil, const SplitArgs<float> *args, const int2 *items, int nitems,
                                         int swap, cudaStream_t st) {
  return launch_split_batch<float, float>(stencil, args, items, nitems, swap, st);
}
