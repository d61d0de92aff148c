// pm_pcg_solve_noalloc: the Jacobi / plain PCG solve with every scratch buffer taken from one
// file-scope device array instead of allocated memory.
//
// Some callers cannot allocate device memory while they solve: hosts whose device memory is
// owned by a custom pool or a framework allocator (a cudaMalloc behind its back would escape its
// accounting or fail against its reservation), and embedded callers that must not grow the
// device footprint after start-up. This entry point serves them. It calls no cudaMalloc,
// cudaFree, cudaMallocHost or any other allocating routine (torch's included): the Krylov
// vectors r, p, w, the projected right-hand side, the Jacobi inverse diagonal, the block sums, the
// barrier and the results all live in g_pm_noalloc_scratch below, which every GPU that
// loads the library holds until the process exits (about 21 MB). The results are read into stack
// memory.
//
// The solve is one resident launch (pm_resident.cuh). As three kernels per iteration, with slots tested
// one by one in the SpMV, 0.51M rows took 78 us per iteration; resident 39.
//
// Limits and sharing rules:
//   - n (rows) <= PM_NOALLOC_MAX_ROWS; larger systems are rejected with PM_EINVAL.
//   - Jacobi or no preconditioner, FP64 (the IC0 and line factors would need storage).
//   - The operator's device must be the current device (PM_EINVAL otherwise).
//   - The call reads its results back to the host and synchronises the stream, so it is rejected
//     with PM_EINVAL when the stream is being captured.
//   - All calls on a device share the one array, which keeps the last call's contents; every
//     call re-initialises what must start at zero (the barrier). Calls that
//     overlap on the GPU (different streams, or different host threads) race on the array.
//   - The first call on a device (with that device current) looks the array's device address up
//     with cudaGetSymbolAddress.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <mutex>

#include "pm_internal.cuh"
#include "pm_resident.cuh"

namespace pm {
namespace na {

constexpr int64_t MAXR = PM_NOALLOC_MAX_ROWS;
constexpr int TPB = 256;
constexpr int64_t OFF_R = 0;
constexpr int64_t OFF_P = 1 * MAXR;
constexpr int64_t OFF_W = 2 * MAXR;
constexpr int64_t OFF_BW = 3 * MAXR;
constexpr int64_t OFF_DINV = 4 * MAXR;
constexpr int64_t OFF_PART = 5 * MAXR;
constexpr int64_t OFF_CTL = OFF_PART + ((int64_t)NPART * MAX_GRID + 31) / 32 * 32;
constexpr int64_t OFF_OUT = OFF_CTL + 32;
constexpr int64_t TOTAL = OFF_OUT + 32;
static_assert(sizeof(resident::Ctl) <= 256 && sizeof(resident::Out) <= 256, "scratch layout");

}  // namespace na
}  // namespace pm

// The scratch array. In host code its name is only a stand-in: the device address comes from
// cudaGetSymbolAddress (see scratch_for_current_device).
static __device__ __align__(256) double g_pm_noalloc_scratch[pm::na::TOTAL];

namespace pm {
namespace na {
namespace {

// Jacobi inverse diagonal (1 on Dirichlet rows).
__global__ void k_dinv(Geom g, const double* __restrict__ val, int maskc, double* __restrict__ dinv) {
  for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < g.n; row += (int64_t)gridDim.x * blockDim.x) {
    const int col = fdiv(g.nzd, (int)row), k = (int)row - col * g.nz;
    double d = 1.0;
    if (maskc < 0 || !is_dirichlet(g.colflag[col], k, g.nz, maskc)) d = 1.0 / val[DIAG_SLOT * g.npad + row];
    dinv[row] = d;
  }
}

int grid_of(int64_t n, int sms) {
  int64_t g = (n + TPB - 1) / TPB;
  int64_t cap = std::min<int64_t>((int64_t)sms * 8, MAX_GRID);
  return (int)std::max<int64_t>(1, std::min(g, cap));
}

// Device address of the scratch array for the current device, looked up once per device.
double* scratch_for_current_device() {
  static std::mutex mu;
  static double* addr[256] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return nullptr;
  std::lock_guard<std::mutex> lk(mu);
  if (!addr[dev]) {
    double* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress((void**)&p, g_pm_noalloc_scratch);
    if (e != cudaSuccess) {
      cuda_check(e, "cudaGetSymbolAddress(g_pm_noalloc_scratch)");
      return nullptr;
    }
    addr[dev] = p;
  }
  return addr[dev];
}

int run(pm_operator* op, int which, const double* b, double* x, const pm_solve_opts* o, pm_solve_stats* stats,
        cudaStream_t s, double* base) {
  auto t0 = std::chrono::steady_clock::now();
  const int64_t n = op->n;
  const int mc = which_mask(which);
  resident::Args a;
  std::memset(&a, 0, sizeof(a));
  a.g = geom_of(op);
  a.val64 = op->d_val[which_valset(which)];
  a.val = a.val64;
  a.mask = mc >= 0 ? op->d_keep[mc] : op->d_struct;
  a.b = b;
  a.x = x;
  a.r = base + OFF_R;
  a.p = base + OFF_P;
  a.w = base + OFF_W;
  a.bw = base + OFF_BW;
  a.m = op->d_m;
  a.rtol = o->rtol;
  a.one_m = op->one_m;
  a.max_iter = o->max_iter;
  a.max_restarts = o->max_restarts;
  a.x0_is_guess = o->x0_is_guess ? 1 : 0;
  a.proj = which == PM_OP_PRESSURE ? 1 : 0;
  a.ctl = reinterpret_cast<resident::Ctl*>(base + OFF_CTL);
  a.part = base + OFF_PART;
  a.out = reinterpret_cast<resident::Out*>(base + OFF_OUT);
  if (o->prec == PM_PREC_JACOBI) {
    k_dinv<<<grid_of(n, op->num_sms), TPB, 0, s>>>(a.g, a.val64, mc, base + OFF_DINV);
    count_launch();
    a.dinv = base + OFF_DINV;
  }
  int st = cuda_check(cudaMemsetAsync(a.out, 0xff, sizeof(resident::Out), s), "noalloc results");
  if (st) return st;
  if ((st = resident::launch_fp64(a, PM_PREC_JACOBI, op->num_sms, s))) return st;
  resident::Out got;
  if ((st = cuda_check(cudaMemcpyAsync(&got, a.out, sizeof(got), cudaMemcpyDeviceToHost, s), "noalloc results"))) return st;
  if ((st = cuda_check(cudaStreamSynchronize(s), "noalloc pcg"))) return st;
  if ((st = resident::outcome(got))) return st;
  const resident::Result& h = got.res;
  stats->iters = h.iters;
  stats->outer_iters = h.restarts;
  stats->first_pass_iters = h.first_pass;
  stats->status = h.status;
  stats->rel_residual_true = h.rel_true;
  stats->rel_residual_rec = h.rel_rec;
  stats->rel_residual_floor = h.floor;
  stats->bytes_moved = (double)h.iters * (double)n * (15 * 8 + 8 + 8 + 5 * 8 + 2 * 8 + 3 * 8 + 8);
  stats->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  if (h.status != PM_OK)
    return set_error(h.status, h.status == PM_NOT_CONVERGED ? "PCG did not reach rtol within max_iter"
                                                            : "PCG breakdown: (p, Ap) <= 0 or non-finite");
  return PM_OK;
}

}  // namespace
}  // namespace na
}  // namespace pm

extern "C" int pm_pcg_solve_noalloc(pm_operator* op, pm_which which, const double* b, double* x,
                                    const pm_solve_opts* opts, pm_solve_stats* stats, pm_stream stream) {
  using namespace pm;
  if (!op || !b || !x || !opts) return set_error(PM_EINVAL, "null argument");
  if (!which_symmetric((int)which)) return set_error(PM_EINVAL, "pcg needs a symmetric operator");
  if (opts->prec != PM_PREC_JACOBI && opts->prec != PM_PREC_NONE)
    return set_error(PM_EINVAL, "pm_pcg_solve_noalloc supports PM_PREC_JACOBI and PM_PREC_NONE only");
  if (opts->precision != PM_FP64) return set_error(PM_EINVAL, "pm_pcg_solve_noalloc solves in FP64 only");
  if (!(opts->rtol > 0.0) || opts->max_iter < 0) return set_error(PM_EINVAL, "rtol must be > 0, max_iter >= 0");
  if (op->n > na::MAXR)
    return set_error(PM_EINVAL, "pm_pcg_solve_noalloc: the system has " + std::to_string(op->n) +
                                    " rows, more than PM_NOALLOC_MAX_ROWS = " + std::to_string(na::MAXR));
  cudaStream_t s = (cudaStream_t)stream;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  int st = cuda_check(cudaStreamIsCapturing(s, &cap), "cudaStreamIsCapturing");
  if (st) return st;
  if (cap != cudaStreamCaptureStatusNone)
    return set_error(PM_EINVAL, "pm_pcg_solve_noalloc synchronises its stream; it cannot be called on a stream "
                                "that is being captured");
  int dev = -1;
  if ((st = cuda_check(cudaGetDevice(&dev), "cudaGetDevice"))) return st;
  if (dev != op->device)
    return set_error(PM_EINVAL, "pm_pcg_solve_noalloc: the operator lives on device " + std::to_string(op->device) +
                                    ", the current device is " + std::to_string(dev));
  double* base = na::scratch_for_current_device();
  if (!base) return PM_ECUDA;
  NvtxRange range(std::string("pcg_noalloc ") + which_name((int)which) + " " + prec_name(opts->prec));
  pm_solve_stats local = {};
  st = na::run(op, (int)which, b, x, opts, &local, s, base);
  const int bs = bounds_status("pm_pcg_solve_noalloc");
  if (bs) st = bs;
  if (stats) *stats = local;
  if (log_enabled()) log_solve("pcg_solve_noalloc", op, (int)which, opts->prec, PM_FP64, local);
  return st;
}
