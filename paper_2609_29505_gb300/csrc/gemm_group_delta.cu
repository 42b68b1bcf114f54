// Instantiations of gemm_group_kernel.cuh with the residual epilogue.
#include "gemm_group_kernel.cuh"

namespace sgd {
namespace gk {

template cudaError_t launch_group<2, 256, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 224, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 192, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 160, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 128, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 256, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 128, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 64, kEpDelta>(const GemmPlan&, const TcArgs&, cudaStream_t);

}  // namespace gk
}  // namespace sgd
