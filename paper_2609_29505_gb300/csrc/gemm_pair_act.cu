// Instantiations of the CTA-pair GEMM (gemm_pair_kernel.cuh) with gated and RoPE epilogues.
#include "gemm_pair_kernel.cuh"

namespace sgd {
namespace gk {

template cudaError_t launch_pair<256, kEpGated>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<224, kEpGated>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<256, kEpRope>(const GemmPlan&, const TcArgs&, cudaStream_t);

}  // namespace gk
}  // namespace sgd
