// hybrid_attn_fma128.cu -- the CUDA-core step for head_dim 128 (attn_fma.cuh).
#include "attn_fma.cuh"

namespace hyb {
namespace fma {
cudaError_t launch_attn_d128(const AttnArgs &a, int n_req, int rt, cudaStream_t st) { return launch_attn_d<128>(a, n_req, rt, st); }
}  // namespace fma
}  // namespace hyb
