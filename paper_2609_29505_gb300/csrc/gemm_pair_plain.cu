// Instantiations of the CTA-pair GEMM (gemm_pair_kernel.cuh) with plain, GELU and fp32 epilogues.
#include "gemm_pair_kernel.cuh"

namespace sgd {
namespace gk {

template cudaError_t launch_pair<256, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<224, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<192, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<160, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);
template cudaError_t launch_pair<128, kEpPlain>(const GemmPlan&, const TcArgs&, cudaStream_t);

}  // namespace gk
}  // namespace sgd
