// The resident PCG (pm_resident.cuh) of FP64 systems.
#include "pm_resident.cuh"

namespace pm {
namespace resident {

int launch_fp64(Args& a, int prec, bool cluster, int num_sms, cudaStream_t s) {
  return launch<double, double>(a, prec, cluster, num_sms, s);
}

}  // namespace resident
}  // namespace pm
