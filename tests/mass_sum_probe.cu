// Runs the library's mass sum on a workspace of the caller's: n masses at
// `mass` (device), every word of the plan's scratch inside `scratch` (device, at
// least 4096 bytes, whatever it holds).  Leaves the sum at scratch[0] and the ray
// pass's work counter at scratch[1] (8 bytes each).
#include <string.h>

#include "irs_common.cuh"

extern "C" int probe_mass_sum(const double* mass, int64_t n, unsigned char* scratch, int32_t* cells, int64_t ncells,
                              void* stream) {
  irs_plan_t P;
  memset(&P, 0, sizeof P);
  P.g.a1 = P.g.b1 = -1.0;
  P.g.a2 = P.g.b2 = 1.0;
  P.d_msum = reinterpret_cast<double*>(scratch);
  P.d_queue = reinterpret_cast<unsigned long long*>(scratch + 8);
  P.d_status = reinterpret_cast<int*>(scratch + 16);
#ifdef HAVE_MDONE
  P.d_mdone = reinterpret_cast<unsigned int*>(scratch + 64);
#endif
  P.d_mpart = reinterpret_cast<double*>(scratch + 256);
  P.d_zero = cells;
  P.n_zero = ncells;
  return (int)irs::launch_mass_sum(&P, mass, n, static_cast<cudaStream_t>(stream));
}
