// Two-pass step instantiations: BF16 storage.
#include "sc_split_inst.cuh"
cudaError_t scgb::launch_split_bf16(int stencil, const SplitArgs<float> &m, cudaStream_t st) {
  return launch_split<__nv_bfloat16, float>(stencil, m, st);
}
cudaError_t scgb::launch_split_batch_bf16(int stencil, const SplitArgs<float> *args, const int2 *items, int nitems,
                                         int swap, cudaStream_t st) {
  return launch_split_batch<__nv_bfloat16, float>(stencil, args, items, nitems, swap, st);
}
