// Two-pass step instantiations: FP64 storage.
#include "sc_split_inst.cuh"
cudaError_t scgb::launch_split_f64(int stencil, const SplitArgs<double> &m, cudaStream_t st) {
  return launch_split<double, double>(stencil, m, st);
}
cudaError_t scgb::launch_split_batch_f64(int stencil, const SplitArgs<double> *args, const int2 *items, int nitems,
                                         int swap, cudaStream_t st) {
  return launch_split_batch<double, double>(stencil, args, items, nitems, swap, st);
}
