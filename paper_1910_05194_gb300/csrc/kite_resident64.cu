// kite_resident64.cu -- the FP64 kernels of the on-chip sweep of mid-size lattices
// (kite_resident.cuh).
#include "kite_resident.cuh"

namespace kite {

const void* resident_kernel64(int lattice, int dbl, int var, int sites) {
  return res_kernel<double, 16>(lattice, dbl, var, sites);
}

}  // namespace kite
