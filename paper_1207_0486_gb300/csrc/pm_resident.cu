// The resident PCG (pm_resident.cuh) of FP64 systems.
#include "pm_resident.cuh"

namespace pm {
namespace resident {

int launch_fp64(Args& a, int prec, int num_sms, cudaStream_t s) {
  return launch<double, double>(a, prec, num_sms, s);
}

// One block takes the parts of both: as rank 1 of two it waits for an arrival that never comes, then it
// reports a result as rank 0.
__global__ void __launch_bounds__(NT, 1) k_timeout_probe(Args a) {
  __shared__ Scratch scratch;
  Team<false> team(a, &scratch);
  team.G = 2;
  Result o = {};
  report(a.out, 1, team.barrier(), o);
  report(a.out, 0, true, o);
}

int debug_timeout(cudaStream_t s) {
  char* d = nullptr;
  int st = cuda_check(cudaMalloc((void**)&d, sizeof(Ctl) + sizeof(Out)), "probe memory");
  if (st) return st;
  Args a = {};
  a.out = reinterpret_cast<Out*>(d);
  a.ctl = reinterpret_cast<Ctl*>(d + sizeof(Out));
  Out h = {};
  st = cuda_check(cudaMemsetAsync(d, 0, sizeof(Ctl) + sizeof(Out), s), "probe memory");
  if (!st) {
    k_timeout_probe<<<1, NT, 0, s>>>(a);
    count_launch();
    st = cuda_check(cudaGetLastError(), "k_timeout_probe");
  }
  if (!st) st = cuda_check(cudaMemcpyAsync(&h, d, sizeof(Out), cudaMemcpyDeviceToHost, s), "probe results");
  if (!st) st = cuda_check(cudaStreamSynchronize(s), "probe");
  cudaFree(d);
  return st ? st : outcome(h);
}

}  // namespace resident
}  // namespace pm
