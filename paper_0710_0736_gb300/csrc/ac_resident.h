// ac_resident.h -- a value queried once per kernel (plain C++).
#pragma once

namespace ac {

// q(K, THREADS) of the first call for this kernel and block size.  The kernel
// is a template argument and not a parameter: kernels of one pointer type
// (k_smooth_settled with and without MASK, k_coarse_pair for every N and
// smoother) would share one static, and the first of them used in the process
// would set the others' grids.
template <auto K, int THREADS, class Query>
int once_per_kernel(Query q) {
  static const int value = q(K, THREADS);
  return value;
}

}  // namespace ac
