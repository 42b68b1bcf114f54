// Instantiations of the CTA-pair GEMM (gemm_pair_kernel.cuh) with the residual epilogue.
#include "gemm_pair_kernel.cuh"

namespace sgd {
namespace gk {

template cudaError_t launch_pair<256, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<224, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<192, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<160, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<128, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);

}  // namespace gk
}  // namespace sgd
