// static_arrays.h -- the device arrays of the no-allocation entry point and when they may be used
// (internal, host code: it compiles without the CUDA compiler, the runtime calls come in as Rt).
#pragma once
#include <cmath>
#include <vector>

namespace pimpc {

// Momentum factors (alpha_m - 1) / alpha_{m+1} of Algorithm 1 step 6 after m consecutive momentum
// steps, alpha_0 = 1, alpha_{m+1} = (1 + sqrt(1 + 4 alpha_m^2)) / 2, rounded as the device rounds
// them (multiply-adds fused).
inline std::vector<double> momentum_factors(int len) {
  std::vector<double> tab(len);
  double al = 1.0;
  for (int m = 0; m < len; ++m) {
    const double an = std::fma(0.5, std::sqrt(std::fma(4.0 * al, al, 1.0)), 0.5);
    tab[m] = (al - 1.0) / an;
    al = an;
  }
  return tab;
}

// Addresses on one device; scratch is null until both arrays may be used.
struct StaticArrays {
  void *scratch = nullptr;
  double *coefs = nullptr;
};

// The first call on a device: looks up both arrays and fills the table. A copy from pageable memory
// may return once the data are staged, and the stream that the caller solves on need not be ordered
// after the copy's, so the copy is waited for before the addresses can be seen by anyone.
// Rt: scratch(void **), table(double **), copy(double *device, const double *host, int count), wait()
// for that copy; each returns 0 or an error, which leaves `a` unset.
template <typename Rt>
int ensure_static_arrays(Rt &rt, StaticArrays &a, int table_len) {
  if (a.scratch) return 0;
  StaticArrays t;
  int rc = rt.scratch(&t.scratch);
  if (rc == 0) rc = rt.table(&t.coefs);
  if (rc != 0) return rc;
  const std::vector<double> tab = momentum_factors(table_len);
  rc = rt.copy(t.coefs, tab.data(), table_len);
  const int waited = rt.wait();  // also after an error: the host buffer goes away
  if (rc == 0) rc = waited;
  if (rc == 0) a = t;
  return rc;
}

}  // namespace pimpc
