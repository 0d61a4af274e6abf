// Subdomain ILU(0) factorisation in FP64, boxes in narrow groups (ras.cuh).  A unit
// of its own: the generated elimination code takes half a minute to compile.
#include <algorithm>

#include "factor.cuh"

kkt_status ras_factor_launch64_narrow(ras_precond* m, cudaStream_t s) {
  return factor_launch<double, narrow_group(64)>(m, (double*)m->F, s);
}
