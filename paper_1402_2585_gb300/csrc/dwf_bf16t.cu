// Instantiation of the fine-operator hop passes for bf16t storage.
#include "dwf_kernels.cuh"

namespace hdcg {
void launch_hop_bf16t(int v, int pass, bool mob, const HopArgs& a, dim3 grid, int threads, cudaStream_t st) {
  launch_hop_variant<bf16t_t>(v, pass, mob, a, grid, threads, st);
}
}  // namespace hdcg
