// Instantiation of the fine-operator hop passes for f64 storage.
#include "dwf_kernels.cuh"

namespace hdcg {
void launch_hop_f64(int v, int pass, bool mob, const HopArgs& a, dim3 grid, int threads, cudaStream_t st) {
  launch_hop_variant<f64_t>(v, pass, mob, a, grid, threads, st);
}
}  // namespace hdcg
