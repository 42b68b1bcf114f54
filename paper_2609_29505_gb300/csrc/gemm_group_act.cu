// Instantiations of gemm_group_kernel.cuh with gated and RoPE epilogues.
#include "gemm_group_kernel.cuh"

namespace sgd {
namespace gk {

template cudaError_t launch_group<2, 256, kEpGated>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 224, kEpGated>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 256, kEpGated>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 128, kEpGated>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 256, kEpRope>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 256, kEpRope>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 128, kEpRope>(const GemmPlan&, const TcArgs&, cudaStream_t);

}  // namespace gk
}  // namespace sgd
