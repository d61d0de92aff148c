// The resident PCG (pm_resident.cuh) of FP32 operator values.
#include "pm_resident.cuh"

namespace pm {
namespace resident {

int launch_fp32(Args& a, int prec, int num_sms, cudaStream_t s) {
  return launch<float, float>(a, prec, num_sms, s);
}

}  // namespace resident
}  // namespace pm
