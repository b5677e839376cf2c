// ns_k2_f64e.cu -- size-specialised kernels (double, N in {32, 48, 64}).
// One translation unit per group of sizes so the build compiles them in parallel.
#include "ns_kernels2.cuh"

namespace ns {

bool k2_lookup_f64e(int N, K2Entry<double>* e) {
  switch (N) {
    case 32:
      *e = make_k2_entry<double, 32>();
      return true;
    case 48:
      *e = make_k2_entry<double, 48>();
      return true;
    case 64:
      *e = make_k2_entry<double, 64>();
      return true;
    default:
      return false;
  }
}

}  // namespace ns
