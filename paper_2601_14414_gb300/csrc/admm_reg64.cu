// admm_reg64.cu -- the FP64 kernels of the register-resident schedule (admm_reg.cuh).
#include "admm_reg.cuh"

namespace pimpc {

cudaError_t launch_reg64(const AdmmLaunch &s, const RegLaunch &rl, cudaStream_t stream) {
  return reg_launch_t<double>(s, rl, stream);
}

}  // namespace pimpc
