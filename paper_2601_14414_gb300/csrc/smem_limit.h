// smem_limit.h -- the dynamic shared-memory limit of a kernel, raised and never lowered (internal,
// host code: it compiles without the CUDA compiler, the runtime calls come in as Rt).
#pragma once
#include <cstddef>
#include <mutex>

namespace pimpc {

// The limit belongs to the kernel on a device, not to a launch: a thread that set it to what its own
// launch needs could lower it between another thread's setting and launch, which is then refused.
// Rt: get(bytes *) reads the limit, set(bytes) writes it; each returns 0 or an error. One mutex for
// all kernels and threads, so that no limit changes between the two.
template <typename Rt>
int raise_smem_limit(Rt rt, std::mutex &mu, std::size_t bytes) {
  std::lock_guard<std::mutex> lock(mu);
  std::size_t now = 0;
  const int rc = rt.get(&now);
  if (rc != 0 || now >= bytes) return rc;
  return rt.set(bytes);
}

}  // namespace pimpc
