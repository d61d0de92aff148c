// The resident PCG (pm_resident.cuh) of BF16 operator values.
#include "pm_resident.cuh"

namespace pm {
namespace resident {

int launch_bf16(Args& a, int prec, int num_sms, cudaStream_t s) {
  return launch<float, __nv_bfloat16>(a, prec, num_sms, s);
}

}  // namespace resident
}  // namespace pm
