// Instantiations of gemm_group_kernel.cuh with plain, GELU and fp32 epilogues.
#include "gemm_group_kernel.cuh"

namespace sgd {
namespace gk {

template cudaError_t launch_group<2, 256, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 224, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 192, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 160, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<2, 128, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 256, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 128, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_group<1, 64, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);

}  // namespace gk
}  // namespace sgd
