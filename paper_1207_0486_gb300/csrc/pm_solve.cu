// SpMV, preconditioner apply and preconditioned conjugate gradient on the column-sliced ELL
// layout (Section 5 remark: the linear systems are solved by PCG; IC0 for the velocity and mass
// systems, DIAG (Jacobi) for the pressure system with a zero-mean Lagrange multiplier).
//
// PCG follows Saad's preconditioned CG step for step (same order of updates, same stopping test
// ||r|| <= rtol ||b|| on the recursive residual, then a true-residual check with restarts):
//   K1 k_cg_spmv   : w = A p and the grid reduction (p, w); the last block forms alpha
//   K2 k_cg_update : x += alpha p, r -= alpha w, z = D^{-1} r (Jacobi, never stored), the grid
//                    reductions (r, r), (r, z) [and m'z, 1'r for the pressure]; the last block
//                    tests convergence and forms beta
//   K3 k_cg_pupd   : p = z + beta p
// This file's kernels run one phase each over the whole GPU (PM_KERNEL_STREAM, and large systems);
// below resident_auto's lines one launch runs the whole solve (pm_resident.cuh).
// IC0 replaces the inline z by 8 forward and 7 backward colour sweeps, with (r, z) = (y, y) between them.
// Grid reductions are deterministic: each block reduces its rows in a fixed tree, writes one
// partial, and the last block to arrive (atomic ticket) sums the partials in block order.
// All scalars (alpha, beta, rho, status) stay on the device; the host reads one small struct
// every few dozen iterations to see whether the solve has finished. Kernels of iterations
// issued after convergence return at once (the device "done" flag), so the result is the same
// as testing after every iteration.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <chrono>
#include <type_traits>

#include "pm_internal.cuh"
#include "pm_resident.cuh"

namespace pm {

struct SolveCtx {
  int64_t n = 0;
  // Resident blocks of the fused line kernels on the operator's device (0: not looked up yet): any nz; 32 levels with
  // tasks of 16 and of 32 columns; FP32 without and with the projection.
  int line_slots = 0, line_w_slots[2] = {0, 0}, line32_slots[2] = {0, 0};
  double *r = nullptr, *p = nullptr, *w = nullptr, *z = nullptr, *bw = nullptr;
  double* partials = nullptr;
  PcgScalars* sc = nullptr;
  PcgScalars* sc_host = nullptr;
  // mixed precision (allocated on first use)
  float *r32 = nullptr, *p32 = nullptr, *w32 = nullptr, *z32 = nullptr, *d32 = nullptr;
  PcgScalars* sc_in = nullptr;
  PcgScalars* sc_in_host = nullptr;
  void* res_ctl = nullptr;        // barrier of the resident solve (device)
  void* res_out = nullptr;   // its results (pinned; the kernel writes them there)
};

struct ColourMap;  // pm_assemble.cu
}  // namespace pm

namespace pm {

// ---- live kernel timing (CUDA events on the launching stream) ------------------------------------
// When enabled, the host PCG loop brackets each launch of the timed kernel classes with a pair of
// events on the solve's stream; elapsed times are collected where that loop synchronises anyway.
// Process-global, not thread-safe: enable it from one host thread only.
struct KernelTimer {
  bool on = false;
  std::vector<cudaEvent_t> pool;
  struct Pending { cudaEvent_t a, b; int kind; int launches; };
  std::vector<Pending> pending;
  double total_ms[PM_KT_COUNT] = {};
  int64_t launches[PM_KT_COUNT] = {};
};
static KernelTimer g_kt;

static cudaEvent_t kt_event() {
  if (!g_kt.pool.empty()) {
    cudaEvent_t e = g_kt.pool.back();
    g_kt.pool.pop_back();
    return e;
  }
  cudaEvent_t e;
  cudaEventCreate(&e);
  return e;
}

struct KtScope {
  cudaEvent_t a = nullptr;
  cudaStream_t s;
  int kind, launches;
  KtScope(int kind_, int launches_, cudaStream_t s_) : s(s_), kind(kind_), launches(launches_) {
    if (g_kt.on) {
      a = kt_event();
      cudaEventRecord(a, s);
    }
  }
  ~KtScope() {
    if (a) {
      cudaEvent_t b = kt_event();
      cudaEventRecord(b, s);
      g_kt.pending.push_back({a, b, kind, launches});
    }
  }
};

static void kt_collect() {
  for (auto& p : g_kt.pending) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, p.a, p.b) == cudaSuccess) {
      g_kt.total_ms[p.kind] += ms;
      g_kt.launches[p.kind] += p.launches;
    }
    g_kt.pool.push_back(p.a);
    g_kt.pool.push_back(p.b);
  }
  g_kt.pending.clear();
}

namespace {

constexpr int TPB = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Reduce NV per-thread values over the block; thread 0 receives the sums. sm: NV * 32 doubles.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* sm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    v[i] = warp_sum(v[i]);
    if (lane == 0) sm[i * 32 + wid] = v[i];
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      double t = lane < nw ? sm[i * 32 + lane] : 0.0;
      v[i] = warp_sum(t);
    }
  }
  __syncthreads();
}

// Grid reduction with a last-block finish. Returns true in the last block; there, thread 0 holds
// the grid totals in v. partials: NV * gridDim.x doubles; ticket: a zero-initialised counter
// that the last block resets.
template <int NV>
__device__ __forceinline__ bool grid_sum(double (&v)[NV], double* partials, uint32_t* ticket) {
  __shared__ double sm[NV * 32];
  __shared__ bool last;
  block_sum<NV>(v, sm);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) partials[i * gridDim.x + blockIdx.x] = v[i];
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double acc[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) {
    double a = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) a += __ldcg(partials + i * gridDim.x + b);
    acc[i] = a;
  }
  block_sum<NV>(acc, sm);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = acc[i];
    *ticket = 0;
  }
  return true;
}

__device__ __forceinline__ bool sc_done(const PcgScalars* sc) {
  return *((volatile const int32_t*)&sc->done) != 0;
}

// Row r of the (optionally masked) operator times x. MASKC >= 0: symmetric elimination of
// component MASKC's Dirichlet set (identity row, zero column).
// Branch-free: all 15 value loads are unconditional (absent slots hold 0), an absent or
// eliminated neighbour reads x[row] and multiplies a selected 0, so every load of a row can be
// in flight at once. 32-bit indices: the library caps n so that 15 * n_pad < 2^31.
template <int MASKC, typename TV, typename TX>
__device__ __forceinline__ double row_dot(const Geom& g, const TV* __restrict__ val, const TX* __restrict__ x,
                                          int row, int col, int k, bool& is_dir) {
  const int nz = g.nz;
  const int npad = (int)g.npad;
  int nb[NNBR];
  uint8_t fl[NNBR];
  nb[0] = col;
#pragma unroll
  for (int q = 1; q < NNBR; ++q) nb[q] = nbr_of(g, col, q);
  if (MASKC >= 0) {
#pragma unroll
    for (int q = 0; q < NNBR; ++q) fl[q] = __ldg(g.colflag + (nb[q] >= 0 ? nb[q] : col));
  }
  TV a[NSLOT];
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) a[s] = __ldg(val + s * npad + row);
  double sum = 0.0;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const int q = slot_q(s);
    const int kk = k + slot_dk(s);
    bool ok = nb[q] >= 0;
    if (slot_dk(s) < 0) ok = ok && kk >= 0;
    if (slot_dk(s) > 0) ok = ok && kk < nz;
    if (MASKC >= 0) ok = ok && !is_dirichlet(fl[q], kk, nz, MASKC);
    const double xv = (double)x[ok ? nb[q] * nz + kk : row];
    const double av = ok ? (double)a[s] : 0.0;
    sum = fma(av, xv, sum);
  }
  if (MASKC >= 0) {
    is_dir = is_dirichlet(fl[0], k, nz, MASKC);
    if (is_dir) sum = (double)x[row];
  }
  return sum;
}

// Row r of component c's eliminated velocity operator times x, with the kept slots of the row
// read from its precomputed mask (bit s: slot s's neighbour present and not Dirichlet; bit 15:
// identity row). Same result as row_dot<c>, without the dependent column-flag loads.
template <typename TV, typename TX>
__device__ __forceinline__ double row_dot_keep(const Geom& g, const TV* __restrict__ val, const TX* __restrict__ x,
                                               const uint16_t* __restrict__ keep, int row, int col, int k) {
  const int nz = g.nz;
  const int npad = (int)g.npad;
  const uint32_t km = __ldg(keep + row);
  if (km & 0x8000u) return (double)x[row];
  int nb[NNBR];
  nb[0] = col;
#pragma unroll
  for (int q = 1; q < NNBR; ++q) nb[q] = nbr_of(g, col, q);
  TV a[NSLOT];
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) a[s] = __ldg(val + s * npad + row);
  double sum = 0.0;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const bool ok = (km >> s) & 1u;
    const double xv = (double)x[ok ? nb[slot_q(s)] * nz + k + slot_dk(s) : row];
    sum = fma(ok ? (double)a[s] : 0.0, xv, sum);
  }
  return sum;
}

template <int MASKC>
__global__ void __launch_bounds__(TPB) k_spmv(Geom g, const double* __restrict__ val,
                                              const double* __restrict__ x, double* __restrict__ y) {
  const int n = (int)g.n;
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < n; row += gridDim.x * blockDim.x) {
    const int col = row / g.nz;
    const int k = row - col * g.nz;
    bool d = false;
    y[row] = row_dot<MASKC>(g, val, x, row, col, k, d);
  }
}

// ---- PCG setup ---------------------------------------------------------------------------------

// Pressure only: lam = 1'b / 1'm, xshift = m'x / 1'm.
__global__ void __launch_bounds__(TPB) k_cg_press_sums(int64_t n, const double* __restrict__ b,
                                                       const double* __restrict__ x, const double* __restrict__ m,
                                                       int use_x, double* partials, PcgScalars* sc) {
  double v[2] = {0.0, 0.0};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    v[0] += b[i];
    if (use_x) v[1] = fma(m[i], x[i], v[1]);
  }
  if (grid_sum<2>(v, partials, &sc->count[0]) && threadIdx.x == 0) {
    sc->lam = v[0] / sc->one_m;
    sc->xshift = use_x ? v[1] / sc->one_m : 0.0;
  }
}

// Pressure with a guess: bw = b - lam m and x = x - xshift.
__global__ void k_cg_prepare(int64_t n, const double* __restrict__ b, const double* __restrict__ m,
                             double* __restrict__ bw, double* __restrict__ x, const PcgScalars* sc) {
  const double lam = sc->lam, xs = sc->xshift;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    bw[i] = b[i] - lam * m[i];
    x[i] = x[i] - xs;
  }
}

// Scalars of a solve from ||b||^2 and the first ||r||^2: target, zero right-hand side, first convergence test.
__device__ __forceinline__ void start_scalars(PcgScalars* sc, double rtol, double bb, double rr) {
  sc->bb = bb;
  sc->rr = rr;
  sc->tol2 = rtol * rtol * bb;
  sc->zero_rhs = bb == 0.0;
  sc->iter = 0;
  sc->status = PM_OK;
  sc->done = (bb == 0.0 || rr <= sc->tol2) ? 1 : 0;
  if (!sc->done && sc->max_iter == 0) {  // no iteration allowed: report the initial residual
    sc->status = PM_NOT_CONVERGED;
    sc->done = 1;
  }
}

// A solve from x = 0: bw = b - lam m (pressure), r = bw itself, (bw, bw). The residual kernel would spend 1.5 ms at
// 5M rows on forming b - A 0.
__global__ void __launch_bounds__(TPB) k_cg_start_zero(int64_t n, const double* __restrict__ b, const double* __restrict__ m,
                                                       double* __restrict__ bw, double* __restrict__ x,
                                                       double* __restrict__ r, int press, double rtol, double* partials,
                                                       PcgScalars* sc) {
  const double lam = press ? sc->lam : 0.0;
  double v[1] = {0.0};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double bi = b[i];
    if (press) {
      bi = bi - lam * m[i];
      bw[i] = bi;
    }
    x[i] = 0.0;
    r[i] = bi;
    v[0] = fma(bi, bi, v[0]);
  }
  if (grid_sum<1>(v, partials, &sc->count[1]) && threadIdx.x == 0) start_scalars(sc, rtol, v[0], v[0]);
}

// r = bw - A x, row by row in compensated arithmetic (row_residual_dot2); grid sums (bw, bw),
// (r, r) and the floor's (|A||x| + |bw|)^2. MODE 0: first setup (also sets tol2, zero_rhs and
// the initial convergence test); MODE 1: true residual at exit (stores (r, r) in aux[0]).
template <int MASKC, int MODE>
__global__ void __launch_bounds__(TPB) k_cg_residual(Geom g, const double* __restrict__ val,
                                                     const double* __restrict__ bw, const double* __restrict__ x,
                                                     double* __restrict__ r, double rtol, double* partials,
                                                     PcgScalars* sc) {
  double v[3] = {0.0, 0.0, 0.0};
  const int n = (int)g.n;
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < n; row += gridDim.x * blockDim.x) {
    const int col = row / g.nz;
    const int k = row - col * g.nz;
    double asum = 0.0;
    const double bi = bw[row];
    const double ri = row_residual_dot2<MASKC, MODE == 1>(g, val, x, bi, row, col, k, asum);
    r[row] = ri;
    v[0] = fma(bi, bi, v[0]);
    v[1] = fma(ri, ri, v[1]);
    if (MODE == 1) {
      const double f = asum + fabs(bi);
      v[2] = fma(f, f, v[2]);
    }
  }
  if (grid_sum<3>(v, partials, &sc->count[1]) && threadIdx.x == 0) {
    if (MODE == 0) {
      start_scalars(sc, rtol, v[0], v[1]);
    } else {
      sc->aux[0] = v[1];
      sc->aux[1] = v[2];
    }
  }
}

// First preconditioned residual (Jacobi): rho = (r, z') with z' = z - c 1,
// c = m'z / 1'm for the pressure (PROJ), p = z'; beta = 0.
template <int PROJ>
__global__ void __launch_bounds__(TPB) k_cg_rho(int64_t n, const double* __restrict__ r, const double* __restrict__ dinv,
                                                const double* __restrict__ m, double* partials, PcgScalars* sc) {
  double v[3] = {0.0, 0.0, 0.0};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double ri = r[i];
    const double zi = dinv[i] * ri;
    v[0] = fma(ri, zi, v[0]);
    if (PROJ) {
      v[1] = fma(m[i], zi, v[1]);
      v[2] += ri;
    }
  }
  if (grid_sum<3>(v, partials, &sc->count[2]) && threadIdx.x == 0) {
    const double c = PROJ ? v[1] / sc->one_m : 0.0;
    const double rho_new = v[0] - c * v[2];
    sc->proj_c = c;
    sc->rho = rho_new;
    sc->beta = 0.0;
    if ((!(rho_new > 0.0) || !isfinite(rho_new)) && !sc->done) {
      sc->status = PM_BREAKDOWN;
      sc->done = 1;
    }
  }
}

// p = (z - c) + beta p; beta = 0 on the first step. STORED: z from zbuf, else dinv r.
template <int STORED>
__global__ void __launch_bounds__(TPB) k_cg_pupd(int64_t n, const double* __restrict__ r, const double* __restrict__ dinv,
                                                 const double* __restrict__ zbuf, double* __restrict__ p,
                                                 const PcgScalars* sc, int is_first) {
  if (!is_first && sc_done(sc)) return;
  const double beta = sc->beta, c = sc->proj_c;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double zi = (STORED ? zbuf[i] : dinv[i] * r[i]) - c;
    p[i] = is_first ? zi : fma(beta, p[i], zi);
  }
}

// ---- PCG iteration -----------------------------------------------------------------------------

// 256 threads, at most 64 registers: 4 blocks (32 warps) per SM to hide the gather latency.
template <int MASKC>
__global__ void __launch_bounds__(TPB, 4) k_cg_spmv(Geom g, const double* __restrict__ val, const double* __restrict__ p,
                                                    double* __restrict__ w, const uint16_t* __restrict__ keep,
                                                    double* partials, PcgScalars* sc) {
  if (sc_done(sc)) return;
  double v[1] = {0.0};
  const int n = (int)g.n;
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < n; row += gridDim.x * blockDim.x) {
    const int col = row / g.nz;
    const int k = row - col * g.nz;
    bool d = false;
    const double wi = MASKC >= 0 ? row_dot_keep(g, val, p, keep, row, col, k) : row_dot<MASKC>(g, val, p, row, col, k, d);
    w[row] = wi;
    v[0] = fma(p[row], wi, v[0]);
  }
  if (grid_sum<1>(v, partials, &sc->count[3]) && threadIdx.x == 0) {
    const double pap = v[0];
    sc->pAp = pap;
    if (!(pap > 0.0) || !isfinite(pap)) {
      sc->status = PM_BREAKDOWN;
      sc->done = 1;
    } else {
      sc->alpha = sc->rho / pap;
    }
  }
}

// x += alpha p; r -= alpha w; (Jacobi, INLINE_Z) z = dinv r and its dots, else only (r, r).
template <int PROJ, int INLINE_Z>
__global__ void __launch_bounds__(TPB) k_cg_update(int64_t n, double* __restrict__ x, double* __restrict__ r,
                                                   const double* __restrict__ p, const double* __restrict__ w,
                                                   const double* __restrict__ dinv, const double* __restrict__ m,
                                                   double* partials, PcgScalars* sc) {
  if (sc_done(sc)) return;
  const double alpha = sc->alpha;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] = fma(alpha, p[i], x[i]);
    const double ri = fma(-alpha, w[i], r[i]);
    r[i] = ri;
    v[0] = fma(ri, ri, v[0]);
    if (INLINE_Z) {
      const double zi = dinv[i] * ri;
      v[1] = fma(ri, zi, v[1]);
      if (PROJ) {
        v[2] = fma(m[i], zi, v[2]);
        v[3] += ri;
      }
    }
  }
  if (grid_sum<4>(v, partials, &sc->count[4]) && threadIdx.x == 0) {
    sc->iter += 1;
    sc->rr = v[0];
    if (v[0] <= sc->tol2) {
      sc->done = 1;
    } else if (sc->iter >= sc->max_iter) {
      sc->status = PM_NOT_CONVERGED;
      sc->done = 1;
    } else if (v[0] <= sc->aux[2]) {
      sc->done = 2;  // residual replacement requested (mixed precision): the host finishes the step
    } else if (INLINE_Z) {
      const double c = PROJ ? v[2] / sc->one_m : 0.0;
      const double rho_new = v[1] - c * v[3];
      sc->proj_c = c;
      sc->beta = rho_new / sc->rho;
      sc->rho = rho_new;
      if (!(rho_new > 0.0) || !isfinite(rho_new)) {
        sc->status = PM_BREAKDOWN;
        sc->done = 1;
      }
    }
  }
}

// ---- IC0 colour sweeps -------------------------------------------------------------------------
// The sweeps' work vector y (then z) is kept in colour order, the order of the factor's rows: position
// cbase[colour] + (index of the column in its parity class) * levels + level / 2. A colour's rows are every
// other level of their columns, so in the natural order each gathered or stored sector would be half
// used; in colour order a warp's accesses to every neighbour are runs. The neighbours' class indices
// come from a table in class order (d_ccls), one load each. Before (natural order, 64-bit index
// divisions, two dependent index loads per neighbour): 23.8 us per colour phase at 4.9M rows; 18.9 with this
// layout, 16.1 launched ahead (below).
struct SweepGeo {
  int32_t n, nz, ncols;
  const int32_t* cnbr;
  const int32_t* ccls;
  const int32_t* colpos;
  int32_t cbase[8], cls_off[4], cls_cnt[4];
  FastDiv nlev[2], nzd;
};

__device__ __forceinline__ int ccls_of(const SweepGeo& g, int i, int q) {
  const int nb = __ldg(g.ccls + q * g.ncols + i);
#ifdef PM_CHECKED
  if (nb < -1 || nb >= g.ncols) {
    record_bad_index(SITE_NBR, nb, g.ncols);
    return -1;
  }
#endif
  return nb;
}

// Colour-ordered position of a row in natural order.
__device__ __forceinline__ int colour_pos(const SweepGeo& g, int row) {
  const int col = fdiv(g.nzd, row), k = row - col * g.nz;
  return __ldg(g.colpos + (k & 1) * g.ncols + col) + (k >> 1);
}

// Forward (FWD = 1): y_i = (r_i - sum_{colour(j) < C} L_ij y_j) / L_ii over rows of colour C.
// Backward (FWD = 0): z_i = (y_i - sum_{colour(j) > C} L_ji z_j) / L_ii, in place on y.
// The factor's diagonal slot holds 1 / L_ii (a multiply instead of an FP64 division).
// Position t of colour C: column t / nlev of its class, level 2 (t % nlev) + parity. All of a row's
// loads but the neighbours' values are independent of one another.
//
// Launched ahead of the previous kernel's end (programmatic dependent launch): a block that finds room
// while that kernel's last blocks run fetches its factor row and neighbour indices, which no kernel of a solve
// writes, and waits for the previous kernel only then. r and y are not __restrict__: earlier kernels write them
// while this one is already resident, so neither may be read as constant for the kernel's life (ld.global.nc,
// or a load moved above the wait).
template <int C, int FWD, typename T>
__global__ void __launch_bounds__(TPB, 4) k_ic0_sweep(SweepGeo g, const T* __restrict__ F, const T* r, T* y,
                                                      const PcgScalars* sc, int check_done) {
  asm volatile("griddepcontrol.launch_dependents;");
  constexpr int kpar = C >> 2, cls = C & 3;
  const int total = g.cls_cnt[cls] * g.nlev[kpar].d;
  const int n = g.n;
  const int t = blockIdx.x * blockDim.x + threadIdx.x, tc = min(t, total - 1);   // the grid covers the rows
  const int i = fdiv(g.nlev[kpar], tc), kk = tc - i * g.nlev[kpar].d, at = g.cls_off[cls] + i, pos = g.cbase[C] + tc;
  T f[NSLOT], v[NSLOT];
  int nb[NNBR];
  nb[0] = i;
#pragma unroll
  for (int q = 1; q < NNBR; ++q) nb[q] = ccls_of(g, at, q);
  const int own = FWD ? __ldg(g.cnbr + at) * g.nz + 2 * kk + kpar : pos;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const int cj = C ^ slot_flip(s);
    if (s == DIAG_SLOT || (FWD ? cj < C : cj > C)) f[s] = __ldg(F + s * n + pos);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (check_done && sc_done(sc)) return;
  T acc = FWD ? r[own] : y[own];
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const int cj = C ^ slot_flip(s);
    if (s == DIAG_SLOT || !(FWD ? cj < C : cj > C)) continue;
    const int dk = slot_dk(s);
    const int lv = kk + (dk == 0 ? 0 : dk > 0 ? kpar : kpar - 1);   // the neighbour's level / 2
    const int nl = g.nlev[cj >> 2].d;
    const bool ok = nb[slot_q(s)] >= 0 && lv >= 0 && lv < nl;
    v[s] = ok ? y[g.cbase[cj] + nb[slot_q(s)] * nl + lv] : (T)0;
  }
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    const int cj = C ^ slot_flip(s);
    if (s == DIAG_SLOT || !(FWD ? cj < C : cj > C)) continue;
    acc = fma(-f[s], v[s], acc);
  }
  if (t < total) y[pos] = acc * f[DIAG_SLOT];
}

// Between the sweeps: (y, y), which is (r, z) since y = L^-1 r and z = L^-T y, and colour 7's backward rows
// z = y / L_ii (no higher colour). FINISH: rho, beta, breakdown test, as k_cg_rho.
template <typename T, int FINISH>
__global__ void __launch_bounds__(TPB) k_ic0_mid(SweepGeo g, const T* __restrict__ F, T* __restrict__ y, double* partials,
                                                 PcgScalars* sc, int is_first) {
  if (!is_first && sc_done(sc)) return;
  AccFor<T> a;
  const int n = g.n, last = g.cbase[7];
  for (int i = (FINISH ? 0 : last) + blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const T yi = y[i];
    if (FINISH) a.add_prod(yi, yi);
    if (i >= last) y[i] = yi * __ldg(F + DIAG_SLOT * n + i);
  }
  if (!FINISH) return;
  double v[1] = {a.value()};
  if (grid_sum<1>(v, partials, &sc->count[2]) && threadIdx.x == 0) {
    sc->proj_c = 0.0;
    sc->beta = is_first ? 0.0 : v[0] / sc->rho;
    sc->rho = v[0];
    if ((!(v[0] > 0.0) || !isfinite(v[0])) && !sc->done) {
      sc->status = PM_BREAKDOWN;
      sc->done = 1;
    }
  }
}

__device__ __forceinline__ void ic0_add_m(Acc64& acc, const double* m, int i, double z) { acc.add_prod(m[i], z); }
__device__ __forceinline__ void ic0_add_m(DF& acc, const float2* m, int i, float z) {
  acc.add_prod(m[i].x, z);
  acc.add_prod(m[i].y, z);
}

// Pressure: rho = (r, z'), z' = z - c, c = m'z / 1'm, with z in colour order (k_cg_rho otherwise).
template <typename T, typename TM>
__global__ void __launch_bounds__(TPB) k_ic0_rho_proj(SweepGeo g, const T* __restrict__ r, const T* __restrict__ z,
                                                      const TM* __restrict__ m, double* partials, PcgScalars* sc,
                                                      int is_first) {
  if (!is_first && sc_done(sc)) return;
  AccFor<T> a0, a1, a2;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += gridDim.x * blockDim.x) {
    const T ri = r[i], zi = z[colour_pos(g, i)];
    a0.add_prod(ri, zi);
    ic0_add_m(a1, m, i, zi);
    a2.add(ri);
  }
  double v[3] = {a0.value(), a1.value(), a2.value()};
  if (grid_sum<3>(v, partials, &sc->count[2]) && threadIdx.x == 0) {
    const double c = v[1] / sc->one_m, rho = v[0] - c * v[2];
    sc->proj_c = c;
    sc->beta = is_first ? 0.0 : rho / sc->rho;
    sc->rho = rho;
    if ((!(rho > 0.0) || !isfinite(rho)) && !sc->done) {
      sc->status = PM_BREAKDOWN;
      sc->done = 1;
    }
  }
}

// p = (z - c) + beta p with z in colour order; FIRST step: p = z - c.
template <typename T>
__global__ void __launch_bounds__(TPB) k_ic0_pupd(SweepGeo g, const T* __restrict__ z, T* __restrict__ p,
                                                  const PcgScalars* sc, int is_first) {
  if (!is_first && sc_done(sc)) return;
  const T beta = (T)sc->beta, c = (T)sc->proj_c;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.n; i += gridDim.x * blockDim.x) {
    const T zi = z[colour_pos(g, i)] - c;
    p[i] = is_first ? zi : fma(beta, p[i], zi);
  }
}

// Grid of the reduction kernels: at most MAX_GRID blocks (the size of the partials buffer).
// ---- vertical-line block Jacobi ----------------------------------------------------------------
// P = block diagonal of A made of each column's tridiagonal block (rows k, couplings k-1 / k+1
// inside the column, the same Dirichlet elimination as A). Thomas factors per row, stored
// level-major (index k * ncols + column) so that one thread per column reads them coalesced:
//   lo_k = A[k, k-1],  w_k = 1 / (A[k, k] - lo_k cp_{k-1}),  cp_k = A[k, k+1] w_k.
__global__ void k_line_factor(Geom g, const double* __restrict__ val, int maskc, double* __restrict__ F,
                              int* __restrict__ breakdown) {
  const int nz = g.nz;
  const int64_t n = g.n;
  for (int64_t col = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; col < g.ncols;
       col += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t fl = g.colflag[col];
    double cprev = 0.0;
    for (int k = 0; k < nz; ++k) {
      const int64_t row = col * nz + k;
      const bool di = maskc >= 0 && is_dirichlet(fl, k, nz, maskc);
      const double d = di ? 1.0 : val[(int64_t)DIAG_SLOT * g.npad + row];
      double lo = 0.0, up = 0.0;
      if (k > 0 && !di && !(maskc >= 0 && is_dirichlet(fl, k - 1, nz, maskc))) lo = val[row];
      if (k < nz - 1 && !di && !(maskc >= 0 && is_dirichlet(fl, k + 1, nz, maskc)))
        up = val[2 * g.npad + row];
      double piv = d - lo * cprev;
      if (!(piv > 0.0)) {
        atomicExch(breakdown, 1);
        piv = 1.0;
      }
      const double w = 1.0 / piv;
      const double cp = up * w;
      const int64_t li = (int64_t)k * g.ncols + col;
      F[li] = lo;
      F[n + li] = w;
      F[2 * n + li] = cp;
      cprev = cp;
    }
  }
}

constexpr int LINE_COLS = 64;
constexpr int LINE_TPB = 128;

// z = P^{-1} r for whole columns staged in shared memory, fused with the (r, z) [m'z, 1'r]
// reductions and the beta update (as k_cg_rho).
template <int PROJ>
__global__ void __launch_bounds__(LINE_TPB) k_line_rho(Geom g, const double* __restrict__ F,
                                                       const double* __restrict__ r, double* __restrict__ z,
                                                       const double* __restrict__ m, double* partials,
                                                       PcgScalars* sc, int is_first) {
  extern __shared__ double smem[];
  if (!is_first && sc_done(sc)) return;
  const int nz = g.nz, ld = nz + 1;
  double* sr = smem;
  double* sz = smem + LINE_COLS * ld;
  const int64_t n = g.n;
  const int64_t ntiles = (g.ncols + LINE_COLS - 1) / LINE_COLS;
  double v[3] = {0.0, 0.0, 0.0};
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t c0 = tile * LINE_COLS;
    const int cc = (int)min((int64_t)LINE_COLS, (int64_t)g.ncols - c0);
    const int64_t row0 = c0 * nz;
    const int rows = cc * nz;
    for (int i = threadIdx.x; i < rows; i += blockDim.x) sr[(i / nz) * ld + i % nz] = r[row0 + i];
    __syncthreads();
    if ((int)threadIdx.x < cc) {
      const int64_t col = c0 + threadIdx.x;
      const int base = threadIdx.x * ld;
      double y = 0.0;
      for (int k = 0; k < nz; ++k) {
        const int64_t li = (int64_t)k * g.ncols + col;
        y = (sr[base + k] - F[li] * y) * F[n + li];
        sz[base + k] = y;
      }
      double zn = sz[base + nz - 1];
      for (int k = nz - 2; k >= 0; --k) {
        const int64_t li = (int64_t)k * g.ncols + col;
        zn = fma(-F[2 * n + li], zn, sz[base + k]);
        sz[base + k] = zn;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
      const int si = (i / nz) * ld + i % nz;
      const double zi = sz[si], ri = sr[si];
      z[row0 + i] = zi;
      v[0] = fma(ri, zi, v[0]);
      if (PROJ) {
        v[1] = fma(m[row0 + i], zi, v[1]);
        v[2] += ri;
      }
    }
    __syncthreads();
  }
  if (grid_sum<3>(v, partials, &sc->count[2]) && threadIdx.x == 0) {
    const double c = PROJ ? v[1] / sc->one_m : 0.0;
    const double rho_new = v[0] - c * v[2];
    sc->proj_c = c;
    if (is_first) {
      sc->rho = rho_new;
      sc->beta = 0.0;
    } else {
      sc->beta = rho_new / sc->rho;
      sc->rho = rho_new;
    }
    if (!(rho_new > 0.0) || !isfinite(rho_new)) {
      if (!sc->done) {
        sc->status = PM_BREAKDOWN;
        sc->done = 1;
      }
    }
  }
}

// One PCG iteration's update with the vertical-line preconditioner fused in:
//   x += alpha p, r -= alpha w (rows of LINE_FCOLS whole columns, staged in shared memory),
//   z = P^{-1} r column by column (one thread per column, in place), then the reductions
//   (r, r), (r, z) [m'z, 1'r]. The last block tests convergence on (r, r) and forms beta, as
//   k_cg_update + k_line_rho would; the z of the converged iteration is simply not used.
#ifndef PM_LINE_FCOLS
#define PM_LINE_FCOLS 64
#endif
#ifndef PM_LINE_UNROLL
#define PM_LINE_UNROLL 8
#endif
constexpr int LINE_FCOLS = PM_LINE_FCOLS;  // FP64 fused kernel: columns per block (128 threads stage them)
constexpr int LINE_FTPB = 128;
constexpr int LINE_UNROLL = PM_LINE_UNROLL;  // levels of Thomas factors in flight per sweep thread

// NZ > 0: compile-time column height (shifts instead of divisions); NZ == 0: g.nz at run time.
template <int PROJ, int NZ>
__global__ void __launch_bounds__(LINE_FTPB) k_update_line(Geom g, const double* __restrict__ F,
                                                         double* __restrict__ x, double* __restrict__ r,
                                                         const double* __restrict__ p, const double* __restrict__ w,
                                                         double* __restrict__ z, const double* __restrict__ m,
                                                         double* partials, PcgScalars* sc, int nfull_max) {
  extern __shared__ double smem[];
  if (sc_done(sc)) return;
  const double alpha = sc->alpha;
  const int nz = NZ > 0 ? NZ : g.nz, ld = nz + 1;
  const int ncols = g.ncols;
  const int n = (int)g.n;
  const int ntiles = (ncols + LINE_FCOLS - 1) / LINE_FCOLS;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  // Tiles 0 .. nfull-1 are LINE_FCOLS columns wide (one per resident block: the first wave); the
  // columns left after them go in half-width tiles, so the second wave is short.
  const int nfull = min(ntiles, nfull_max);
  const int rest0 = nfull * LINE_FCOLS;
  const int nhalf = rest0 < ncols ? (ncols - rest0 + LINE_FCOLS / 2 - 1) / (LINE_FCOLS / 2) : 0;
  for (int tile = blockIdx.x; tile < nfull + nhalf; tile += gridDim.x) {
    const int c0 = tile < nfull ? tile * LINE_FCOLS : rest0 + (tile - nfull) * (LINE_FCOLS / 2);
    const int cc = min(tile < nfull ? LINE_FCOLS : LINE_FCOLS / 2, ncols - c0);
    const int row0 = c0 * nz;
    const int rows = cc * nz;
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
      const int row = row0 + i;
      x[row] = fma(alpha, p[row], x[row]);
      const double ri = fma(-alpha, w[row], r[row]);
      r[row] = ri;
      smem[(i / nz) * ld + i % nz] = ri;
      v[0] = fma(ri, ri, v[0]);
    }
    __syncthreads();
    if ((int)threadIdx.x < cc) {
      const int col = c0 + threadIdx.x;
      double* col_s = smem + threadIdx.x * ld;
      double y = 0.0;
#pragma unroll (LINE_UNROLL)
      for (int k = 0; k < nz; ++k) {
        const int li = k * ncols + col;
        y = (col_s[k] - F[li] * y) * F[n + li];
        col_s[k] = y;
      }
      double zn = y;
#pragma unroll (LINE_UNROLL)
      for (int k = nz - 2; k >= 0; --k) {
        const int li = k * ncols + col;
        zn = fma(-F[2 * n + li], zn, col_s[k]);
        col_s[k] = zn;
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
      const int row = row0 + i;
      const double zi = smem[(i / nz) * ld + i % nz];
      const double ri = r[row];
      z[row] = zi;
      v[1] = fma(ri, zi, v[1]);
      if (PROJ) {
        v[2] = fma(m[row], zi, v[2]);
        v[3] += ri;
      }
    }
    __syncthreads();
  }
  if (grid_sum<4>(v, partials, &sc->count[4]) && threadIdx.x == 0) {
    sc->iter += 1;
    sc->rr = v[0];
    if (v[0] <= sc->tol2) {
      sc->done = 1;
    } else if (sc->iter >= sc->max_iter) {
      sc->status = PM_NOT_CONVERGED;
      sc->done = 1;
    } else {
      const double c = PROJ ? v[2] / sc->one_m : 0.0;
      const double rho_new = v[1] - c * v[3];
      sc->proj_c = c;
      sc->beta = rho_new / sc->rho;
      sc->rho = rho_new;
      if (!(rho_new > 0.0) || !isfinite(rho_new)) {
        sc->status = PM_BREAKDOWN;
        sc->done = 1;
      }
    }
  }
}

// The same fused iteration for 32-level columns, organised by warp instead of by block. A task is
// TCOLS = 32 whole columns (TCOLS * 32 consecutive rows, since node id = column * 32 + k); every
// warp owns an even, contiguous share of the tasks and the grid is exactly the resident blocks,
// so each SM gets the same work. Per task:
//   A (all lanes, coalesced): x += alpha p, r -= alpha w for level k = lane of each column, r
//     staged into the warp's own shared-memory tile [column][level];
//   B (lane = column): the Thomas sweep down and up the column in that tile;
//   C (all lanes, coalesced): z written, m'z.
// Warps never wait for one another (only __syncwarp), so one warp's sequential sweep overlaps
// other warps' streaming. (r, z) comes out of the sweep without reading r again: with the factors
// T = L U of the column block (L lower bidiagonal, diagonal 1/w_k, sub-diagonal lo_k; U unit
// upper bidiagonal, cp_k), a symmetric T has U = diag(w) L^T, so with t_k = r_k - lo_k y_{k-1},
// y_k = t_k w_k and z = U^{-1} y,  (r, z) = y' diag(1/w) y = sum_k t_k y_k.
constexpr int LINE_WNZ = 32;
constexpr int LINE_WTPB = 256;   // 8 warps per block
template <int PROJ, int TCOLS>
__global__ void __launch_bounds__(LINE_WTPB, TCOLS == 32 ? 3 : 4) k_update_line_w(
    Geom g, const double* __restrict__ F, double* __restrict__ x, double* __restrict__ r,
    const double* __restrict__ p, const double* __restrict__ w, double* __restrict__ z,
    const double* __restrict__ m, double* partials, PcgScalars* sc) {
  constexpr int NZ = LINE_WNZ, LD = NZ + 1;
  extern __shared__ double smem[];
  if (sc_done(sc)) return;
  const double alpha = sc->alpha;
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  double* ws = smem + wib * (TCOLS * LD);
  const int ncols = g.ncols;
  const int n = (int)g.n;
  const int nwarps = gridDim.x * (LINE_WTPB / 32);
  const int wg = blockIdx.x * (LINE_WTPB / 32) + wib;
  // this warp's tasks (TCOLS columns each, the last one ragged): an even split of all tasks over
  // all warps, so every block, hence every SM, gets the same work and every lane sweeps a column
  const int ntask = (ncols + TCOLS - 1) / TCOLS;
  const int tbeg = (int)((int64_t)ntask * wg / nwarps);
  const int tend = (int)((int64_t)ntask * (wg + 1) / nwarps);
  double v[4] = {0.0, 0.0, 0.0, 0.0};   // (r, r), (r, z), m'z, 1'r
  for (int t = tbeg; t < tend; ++t) {
    const int c0 = t * TCOLS;
    const int cc = min(TCOLS, ncols - c0);
    const int row0 = c0 * NZ + lane;
#pragma unroll 8
    for (int j = 0; j < cc; ++j) {
      const int row = row0 + j * NZ;
      x[row] = fma(alpha, p[row], x[row]);
      const double ri = fma(-alpha, w[row], r[row]);
      r[row] = ri;
      ws[j * LD + lane] = ri;
      v[0] = fma(ri, ri, v[0]);
      if (PROJ) v[3] += ri;
    }
    __syncwarp();
    if (lane < cc) {
      const int col = c0 + lane;
      double* cs = ws + lane * LD;
      double y = 0.0, rz = 0.0;
#pragma unroll 8
      for (int k = 0; k < NZ; ++k) {
        const int li = k * ncols + col;
        const double tk = fma(-F[li], y, cs[k]);
        y = tk * F[n + li];
        rz = fma(tk, y, rz);
        cs[k] = y;
      }
      double zn = y;
#pragma unroll 8
      for (int k = NZ - 2; k >= 0; --k) {
        const int li = k * ncols + col;
        zn = fma(-F[2 * n + li], zn, cs[k]);
        cs[k] = zn;
      }
      v[1] += rz;
    }
    __syncwarp();
#pragma unroll 8
    for (int j = 0; j < cc; ++j) {
      const int row = row0 + j * NZ;
      const double zi = ws[j * LD + lane];
      z[row] = zi;
      if (PROJ) v[2] = fma(m[row], zi, v[2]);
    }
    __syncwarp();
  }
  if (grid_sum<4>(v, partials, &sc->count[4]) && threadIdx.x == 0) {
    sc->iter += 1;
    sc->rr = v[0];
    if (v[0] <= sc->tol2) {
      sc->done = 1;
    } else if (sc->iter >= sc->max_iter) {
      sc->status = PM_NOT_CONVERGED;
      sc->done = 1;
    } else {
      const double c = PROJ ? v[2] / sc->one_m : 0.0;
      const double rho_new = v[1] - c * v[3];
      sc->proj_c = c;
      sc->beta = rho_new / sc->rho;
      sc->rho = rho_new;
      if (!(rho_new > 0.0) || !isfinite(rho_new)) {
        sc->status = PM_BREAKDOWN;
        sc->done = 1;
      }
    }
  }
}

// Columns per task: 32, so that every lane of a warp sweeps a column (an FP64 instruction costs the
// FP64 pipe the same with idle lanes, and the sweep is a third of the kernel's FP64 work), unless
// that leaves fewer tasks than resident warps (basins under about 600 x 600 columns of 32 levels):
// then 16, twice the warps and half the lanes sweeping. line_w_setup gives the resident blocks of
// one choice.
//
// Function attributes are per device, so they are set for every operator, not once in the process.
constexpr int LINE_SMEM = 200 * 1024;
int smem_limit(const void* kernel, size_t bytes) {
  return cuda_check(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes), "line shared memory");
}

template <int TC>
int line_w_setup(pm_operator* op, int* slots) {
  const size_t smem = (size_t)(LINE_WTPB / 32) * TC * (LINE_WNZ + 1) * sizeof(double);
  int st, per_sm = 0;
  if ((st = smem_limit((const void*)k_update_line_w<0, TC>, smem))) return st;
  if ((st = smem_limit((const void*)k_update_line_w<1, TC>, smem))) return st;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_update_line_w<1, TC>, LINE_WTPB, smem);
  *slots = std::max(1, per_sm) * op->num_sms;
  return PM_OK;
}

// What the FP64 line kernels need before their first launch for this operator.
int line_setup(pm_operator* op) {
  SolveCtx* c = op->ctx;
  if (c->line_slots) return PM_OK;
  int st, per_sm = 0;
  if ((st = smem_limit((const void*)k_line_rho<0>, LINE_SMEM))) return st;
  if ((st = smem_limit((const void*)k_line_rho<1>, LINE_SMEM))) return st;
  if ((st = smem_limit((const void*)k_update_line<0, 0>, LINE_SMEM))) return st;
  if ((st = smem_limit((const void*)k_update_line<1, 0>, LINE_SMEM))) return st;
  if ((st = line_w_setup<16>(op, &c->line_w_slots[0]))) return st;
  if ((st = line_w_setup<32>(op, &c->line_w_slots[1]))) return st;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_update_line<1, 0>, LINE_FTPB,
                                                (size_t)LINE_FCOLS * (op->nz + 1) * sizeof(double));
  c->line_slots = std::max(1, per_sm) * op->num_sms;
  return PM_OK;
}

template <int TC>
void launch_line_w(pm_operator* op, int which, bool proj, double* x, int slots, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  Geom g = geom_of(op);
  const size_t smem = (size_t)(LINE_WTPB / 32) * TC * (LINE_WNZ + 1) * sizeof(double);
  int64_t blocks = std::min<int64_t>(slots, (int64_t)NPART * MAX_GRID / 4);
  const int64_t ntask = (op->ncols + TC - 1) / TC;
  blocks = std::min<int64_t>(blocks, (ntask + LINE_WTPB / 32 - 1) / (LINE_WTPB / 32));
  const int grid = (int)std::max<int64_t>(1, blocks);
  const double* F = op->d_line[which];
  if (proj)
    k_update_line_w<1, TC><<<grid, LINE_WTPB, smem, s>>>(g, F, x, c->r, c->p, c->w, c->z, op->d_m, c->partials, c->sc);
  else
    k_update_line_w<0, TC><<<grid, LINE_WTPB, smem, s>>>(g, F, x, c->r, c->p, c->w, c->z, op->d_m, c->partials, c->sc);
}

// Launch of k_update_line_w: exactly the resident blocks (capped by the partials buffer, 4 lanes
// per block, and by one task per warp).
void update_line_w(pm_operator* op, int which, bool proj, double* x, cudaStream_t s) {
  const int slots16 = op->ctx->line_w_slots[0], slots32 = op->ctx->line_w_slots[1];
  const int64_t tasks32 = (op->ncols + 31) / 32;
  if (tasks32 >= (int64_t)slots32 * (LINE_WTPB / 32)) launch_line_w<32>(op, which, proj, x, slots32, s);
  else launch_line_w<16>(op, which, proj, x, slots16, s);
  count_launch();
}

void update_line(pm_operator* op, int which, bool proj, double* x, cudaStream_t s) {
  if (op->nz == LINE_WNZ) {
    update_line_w(op, which, proj, x, s);
    return;
  }
  SolveCtx* c = op->ctx;
  Geom g = geom_of(op);
  const size_t smem = (size_t)LINE_FCOLS * (op->nz + 1) * sizeof(double);
  // The full-width tiles fill exactly one wave of the resident blocks;
  // four partial lanes per block must fit the partials buffer (NPART x MAX_GRID doubles)
  const int nfull_max = (int)std::min<int64_t>(c->line_slots, (int64_t)NPART * MAX_GRID / 4);
  const int64_t nt_full = (op->ncols + LINE_FCOLS - 1) / LINE_FCOLS;
  const int64_t nfull = std::min<int64_t>(nt_full, nfull_max);
  const int64_t rest = std::max<int64_t>(0, op->ncols - nfull * LINE_FCOLS);
  const int64_t ntiles = nfull + (rest + LINE_FCOLS / 2 - 1) / (LINE_FCOLS / 2);
  int grid = (int)std::min<int64_t>(ntiles, nfull_max);
  if (grid < 1) grid = 1;
  const double* F = op->d_line[which];
#define PM_UL(P, NZ)                                                                                     \
  k_update_line<P, NZ><<<grid, LINE_FTPB, smem, s>>>(g, F, x, c->r, c->p, c->w, c->z, op->d_m, c->partials, c->sc, \
                                                     nfull_max)
  if (op->nz == 32) {
    if (proj) PM_UL(1, 32);
    else PM_UL(0, 32);
  } else {
    if (proj) PM_UL(1, 0);
    else PM_UL(0, 0);
  }
#undef PM_UL
  count_launch();
}

void line_apply_rho(pm_operator* op, int which, bool proj, int is_first, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  Geom g = geom_of(op);
  const int64_t ntiles = (op->ncols + LINE_COLS - 1) / LINE_COLS;
  int grid = (int)std::min<int64_t>(ntiles, std::min<int64_t>((int64_t)op->num_sms * 8, MAX_GRID));
  if (grid < 1) grid = 1;
  const size_t smem = 2 * (size_t)LINE_COLS * (op->nz + 1) * sizeof(double);
  if (proj)
    k_line_rho<1><<<grid, LINE_TPB, smem, s>>>(g, op->d_line[which], c->r, c->z, op->d_m, c->partials, c->sc, is_first);
  else
    k_line_rho<0><<<grid, LINE_TPB, smem, s>>>(g, op->d_line[which], c->r, c->z, op->d_m, c->partials, c->sc, is_first);
  count_launch();
}

int line_factor(pm_operator* op, int which, cudaStream_t s) {
  if (op->line_ok[which]) return PM_OK;
  int st;
  if (!op->d_line[which]) {
    if ((st = cuda_check(cudaMalloc((void**)&op->d_line[which], 3 * (size_t)op->n * sizeof(double)), "cudaMalloc line")))
      return st;
    op->device_bytes += 3 * op->n * 8;
  }
  int* d_bd = nullptr;
  if ((st = cuda_check(cudaMallocAsync((void**)&d_bd, sizeof(int), s), "cudaMallocAsync"))) return st;
  cudaMemsetAsync(d_bd, 0, sizeof(int), s);
  Geom g = geom_of(op);
  int grid = (int)std::min<int64_t>((op->ncols + 127) / 128, (int64_t)op->num_sms * 16);
  if (grid < 1) grid = 1;
  k_line_factor<<<grid, 128, 0, s>>>(g, op->d_val[which_valset(which)], which_mask(which), op->d_line[which], d_bd);
  count_launch();
  int h = 0;
  st = cuda_check(cudaMemcpyAsync(&h, d_bd, sizeof(int), cudaMemcpyDeviceToHost, s), "memcpy");
  if (!st) st = cuda_check(cudaStreamSynchronize(s), "line factor");
  cudaFreeAsync(d_bd, s);
  if (st) return st;
  if (h) return set_error(PM_BREAKDOWN, "vertical-line preconditioner: non-positive pivot");
  op->line_ok[which] = true;
  return cuda_check(cudaGetLastError(), "k_line_factor");
}

int grid_for(int64_t n, int threads, int sms) {
  int64_t gsz = (n + threads - 1) / threads;
  int64_t cap = (int64_t)sms * 8;
  if (cap > MAX_GRID) cap = MAX_GRID;
  if (gsz > cap) gsz = cap;
  if (gsz < 1) gsz = 1;
  return (int)gsz;
}

struct CMap {
  int64_t cbase[8];
  int32_t nlev[2];
};
CMap cmap_of(const pm_operator* op) {
  CMap cm;
  cm.nlev[0] = (op->nz + 1) / 2;
  cm.nlev[1] = op->nz / 2;
  int64_t acc = 0;
  for (int c = 0; c < 8; ++c) {
    cm.cbase[c] = acc;
    acc += (int64_t)op->cls_count[c & 3] * cm.nlev[c >> 2];
  }
  return cm;
}

SweepGeo sweep_geo(const pm_operator* op) {
  SweepGeo g;
  const CMap cm = cmap_of(op);
  g.n = (int32_t)op->n;
  g.nz = op->nz;
  g.ncols = op->ncols;
  g.cnbr = op->d_cnbr;
  g.ccls = op->d_ccls;
  g.colpos = op->d_colpos;
  for (int c = 0; c < 8; ++c) g.cbase[c] = (int32_t)cm.cbase[c];
  for (int q = 0, off = 0; q < 4; ++q) {
    g.cls_off[q] = off;
    g.cls_cnt[q] = op->cls_count[q];
    off += op->cls_count[q];
  }
  g.nlev[0] = fast_div(cm.nlev[0]);
  g.nlev[1] = fast_div(cm.nlev[1]);
  g.nzd = fast_div(op->nz);
  return g;
}

// z = (L L^T)^{-1} r into z (colour order), and rho, beta (m: the projection's mass vector, null: none).
// is_first: the step that starts a recurrence; its kernels run whatever the done flag says.
template <typename T, typename TM>
void ic0_apply(pm_operator* op, const T* F, const T* r, T* z, const TM* m, double* partials, PcgScalars* sc, int is_first,
               cudaStream_t s) {
  const SweepGeo g = sweep_geo(op);
  const int G = grid_for(op->n, TPB, op->num_sms), check = is_first ? 0 : 1;
  cudaLaunchAttribute ahead;
  ahead.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  ahead.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(TPB);
  cfg.stream = s;
  cfg.attrs = &ahead;
  cfg.numAttrs = 1;
#define PM_SWEEP(C, FW)                                                                                         \
  {                                                                                                             \
    const int64_t tot = (int64_t)g.cls_cnt[(C) & 3] * g.nlev[(C) >> 2].d;                                       \
    if (tot > 0) {                                                                                              \
      cfg.gridDim = dim3((unsigned)((tot + TPB - 1) / TPB));                                                    \
      cudaLaunchKernelEx(&cfg, k_ic0_sweep<C, FW, T>, g, F, r, z, (const PcgScalars*)sc, check);                \
      count_launch();                                                                                           \
    }                                                                                                           \
  }
  {
    KtScope t(PM_KT_IC0, 16, s);
    PM_SWEEP(0, 1) PM_SWEEP(1, 1) PM_SWEEP(2, 1) PM_SWEEP(3, 1)
    PM_SWEEP(4, 1) PM_SWEEP(5, 1) PM_SWEEP(6, 1) PM_SWEEP(7, 1)
    if (m) k_ic0_mid<T, 0><<<G, TPB, 0, s>>>(g, F, z, partials, sc, is_first);
    else k_ic0_mid<T, 1><<<G, TPB, 0, s>>>(g, F, z, partials, sc, is_first);
    PM_SWEEP(6, 0) PM_SWEEP(5, 0) PM_SWEEP(4, 0)
    PM_SWEEP(3, 0) PM_SWEEP(2, 0) PM_SWEEP(1, 0) PM_SWEEP(0, 0)
  }
#undef PM_SWEEP
  if (m) k_ic0_rho_proj<T, TM><<<G, TPB, 0, s>>>(g, r, z, m, partials, sc, is_first);
  count_launch(m ? 2 : 1);
}

int ensure_ctx(pm_operator* op) {
  if (op->ctx) return PM_OK;
  SolveCtx* c = new SolveCtx();
  c->n = op->n;
  const size_t vb = (size_t)op->n * sizeof(double);
  cudaError_t e = cudaSuccess;
  e = e ? e : cudaMalloc((void**)&c->r, vb);
  e = e ? e : cudaMalloc((void**)&c->p, vb);
  e = e ? e : cudaMalloc((void**)&c->w, vb);
  e = e ? e : cudaMalloc((void**)&c->z, vb);
  e = e ? e : cudaMalloc((void**)&c->bw, vb);
  e = e ? e : cudaMalloc((void**)&c->partials, (size_t)NPART * MAX_GRID * sizeof(double));
  e = e ? e : cudaMalloc((void**)&c->sc, sizeof(PcgScalars));
  e = e ? e : cudaMallocHost((void**)&c->sc_host, sizeof(PcgScalars));
  e = e ? e : cudaMalloc(&c->res_ctl, 64);
  e = e ? e : cudaMallocHost(&c->res_out, 64);
  if (e == cudaSuccess) e = cudaMemset(c->sc, 0, sizeof(PcgScalars));
  op->ctx = c;
  if (e != cudaSuccess) return cuda_check(e, "solve workspace");
  op->device_bytes += 5 * (int64_t)vb + (int64_t)NPART * MAX_GRID * 8 + (int64_t)sizeof(PcgScalars);
  return PM_OK;
}

template <int MASKC>
void launch_iter(pm_operator* op, int which, const double* val, double* x, bool proj, int prec,
                 const double* dinv, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  Geom g = geom_of(op);
  const int G = grid_for(op->n, TPB, op->num_sms);
  const bool ic0 = prec == PM_PREC_IC0;
  {
    KtScope t(PM_KT_SPMV, 1, s);
    k_cg_spmv<MASKC><<<G, TPB, 0, s>>>(g, val, c->p, c->w, MASKC >= 0 ? op->d_keep[MASKC < 0 ? 0 : MASKC] : nullptr,
                                       c->partials, c->sc);
  }
  if (prec == PM_PREC_LINE) {
    {
      KtScope t(PM_KT_LINE, 1, s);
      update_line(op, which, proj, x, s);
    }
    {
      KtScope t(PM_KT_PUPDATE, 1, s);
      k_cg_pupd<1><<<G, TPB, 0, s>>>(op->n, c->r, dinv, c->z, c->p, c->sc, 0);
    }
    count_launch(1);
  } else if (!ic0) {
    {
      KtScope t(PM_KT_UPDATE, 1, s);
      if (proj) {
        k_cg_update<1, 1><<<G, TPB, 0, s>>>(op->n, x, c->r, c->p, c->w, dinv, op->d_m, c->partials, c->sc);
      } else {
        k_cg_update<0, 1><<<G, TPB, 0, s>>>(op->n, x, c->r, c->p, c->w, dinv, op->d_m, c->partials, c->sc);
      }
    }
    {
      KtScope t(PM_KT_PUPDATE, 1, s);
      k_cg_pupd<0><<<G, TPB, 0, s>>>(op->n, c->r, dinv, nullptr, c->p, c->sc, 0);
    }
    count_launch(3);
  } else {
    {
      KtScope t(PM_KT_UPDATE, 1, s);
      k_cg_update<0, 0><<<G, TPB, 0, s>>>(op->n, x, c->r, c->p, c->w, dinv, op->d_m, c->partials, c->sc);
    }
    count_launch(1);
    ic0_apply(op, op->ic0[which].F, c->r, c->z, proj ? op->d_m : nullptr, c->partials, c->sc, 0, s);
    {
      KtScope t(PM_KT_PUPDATE, 1, s);
      k_ic0_pupd<<<G, TPB, 0, s>>>(sweep_geo(op), c->z, c->p, c->sc, 0);
    }
    count_launch(2);
  }
}

template <int MASKC>
void launch_residual(pm_operator* op, const double* val, const double* bw, const double* x, double rtol,
                     int mode, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  Geom g = geom_of(op);
  const int G = grid_for(op->n, TPB, op->num_sms);
  if (mode == 0)
    k_cg_residual<MASKC, 0><<<G, TPB, 0, s>>>(g, val, bw, x, c->r, rtol, c->partials, c->sc);
  else
    k_cg_residual<MASKC, 1><<<G, TPB, 0, s>>>(g, val, bw, x, c->r, rtol, c->partials, c->sc);
  count_launch();
}

// Projected right-hand side (pressure: returned in the workspace), initial guess, first residual in c->r and the
// scalars that start a solve.
template <int MASKC>
const double* launch_start(pm_operator* op, const double* val, const double* b, double* x, bool proj, const pm_solve_opts* o,
                           cudaStream_t s) {
  SolveCtx* c = op->ctx;
  const int G = grid_for(op->n, TPB, op->num_sms), guess = o->x0_is_guess ? 1 : 0;
  if (proj) {
    k_cg_press_sums<<<G, TPB, 0, s>>>(op->n, b, x, op->d_m, guess, c->partials, c->sc);
    count_launch();
  }
  const double* bw = proj ? c->bw : b;
  if (!guess) {
    k_cg_start_zero<<<G, TPB, 0, s>>>(op->n, b, op->d_m, c->bw, x, c->r, proj ? 1 : 0, o->rtol, c->partials, c->sc);
    count_launch();
    return bw;
  }
  if (proj) {
    k_cg_prepare<<<G, TPB, 0, s>>>(op->n, b, op->d_m, c->bw, x, c->sc);
    count_launch();
  }
  launch_residual<MASKC>(op, val, bw, x, o->rtol, 0, s);
  return bw;
}

// z, p, rho from the current r (first step or restart). The kernels run even when "done" is
// set by the setup so that a zero initial residual still leaves consistent scalars.
void launch_first(pm_operator* op, int which, bool proj, int prec, const double* dinv, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  const int G = grid_for(op->n, TPB, op->num_sms);
  if (prec == PM_PREC_LINE) {
    line_apply_rho(op, which, proj, 1, s);
    k_cg_pupd<1><<<G, TPB, 0, s>>>(op->n, c->r, dinv, c->z, c->p, c->sc, 1);
    count_launch(1);
    return;
  }
  if (prec == PM_PREC_IC0) {
    ic0_apply(op, op->ic0[which].F, c->r, c->z, proj ? op->d_m : nullptr, c->partials, c->sc, 1, s);
    k_ic0_pupd<<<G, TPB, 0, s>>>(sweep_geo(op), c->z, c->p, c->sc, 1);
  } else {
    if (proj) k_cg_rho<1><<<G, TPB, 0, s>>>(op->n, c->r, dinv, op->d_m, c->partials, c->sc);
    else k_cg_rho<0><<<G, TPB, 0, s>>>(op->n, c->r, dinv, op->d_m, c->partials, c->sc);
    k_cg_pupd<0><<<G, TPB, 0, s>>>(op->n, c->r, dinv, nullptr, c->p, c->sc, 1);
  }
  count_launch(2);
}

__global__ void k_fill(double* x, int64_t n, double v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) x[i] = v;
}
__global__ void k_shift_by(double* x, int64_t n, const PcgScalars* sc) {
  const double v = sc->xshift;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) x[i] -= v;
}

int read_scalars(SolveCtx* c, cudaStream_t s) {
  int st = cuda_check(cudaMemcpyAsync(c->sc_host, c->sc, sizeof(PcgScalars), cudaMemcpyDeviceToHost, s), "scalars");
  if (st) return st;
  st = cuda_check(cudaStreamSynchronize(s), "pcg sync");
  if (!st && !g_kt.pending.empty()) kt_collect();
  return st;
}

// Algorithmic bytes of one PCG iteration per row (FP64), each array once per pass:
//   SpMV: 15 values + p read + w write = 136;
//   Jacobi: update x, r read/write + p, w, dinv read (z = dinv r inline) = 56, p-update r, dinv,
//           p read + p write = 32;
//   IC0: update x, r read/write + p, w read = 48, the factor (8 of its 15 slots per row in each
//        sweep direction) 128 and r, y, z traffic 32, the (r, z) pass 16, p-update z, p, p = 24;
//   LINE: update 48, the three line factors and the z write 32 (fused with the update), p-update 24.
// The pressure adds m (8) where m'z is taken.
double bytes_per_iter(const pm_operator* op, int prec, bool proj) {
  const double n = (double)op->n;
  double b = n * (15 * 8 + 8 + 8);
  if (prec == PM_PREC_IC0) b += n * (48 + 2 * 8 * 8 + 4 * 8 + 16 + 24);
  else if (prec == PM_PREC_LINE) b += n * (48 + 3 * 8 + 8 + 24);
  else b += n * (56 + 32);
  if (proj) b += n * 8;
  return b;
}

template <int MASKC>
int pcg_run(pm_operator* op, int which, const double* b, double* x, const pm_solve_opts* o,
            pm_solve_stats* stats, cudaStream_t s) {
  auto t0 = std::chrono::steady_clock::now();
  SolveCtx* c = op->ctx;
  const bool proj = which == PM_OP_PRESSURE;
  const bool ic0 = o->prec == PM_PREC_IC0;
  const int prec = o->prec;
  const double* val = op->d_val[which_valset(which)];
  int st;
  // Preconditioner set-up.
  const double* dinv = nullptr;
  if ((st = launch_dinv(op, which, s))) return st;
  dinv = op->d_dinv[which];
  double* ones_buf = nullptr;
  if (o->prec == PM_PREC_NONE) {
    ones_buf = c->z;  // plain CG: z = r, held as dinv = 1 in a scratch vector
    k_fill<<<grid_for(op->n, TPB, op->num_sms), TPB, 0, s>>>(ones_buf, op->n, 1.0);
    count_launch();
    dinv = ones_buf;
  }
  if (ic0) {
    Ic0Factor& f = op->ic0[which];
    if (!f.ok) {
      int bd = 0;
      double shift = 0.0;
      for (int m = -1; m <= 10; ++m) {
        shift = m < 0 ? 0.0 : 1e-3 * std::pow(2.0, m);
        if ((st = launch_ic0_factor(op, which, shift, &bd, s))) return st;
        if (!bd) break;
      }
      if (bd) return set_error(PM_BREAKDOWN, "IC0 pivot failure after the shift limit");
    }
  }
  if (prec == PM_PREC_LINE && ((st = line_setup(op)) || (st = line_factor(op, which, s)))) return st;
  // Right-hand side and initial guess.
  const int G = grid_for(op->n, TPB, op->num_sms);
  PcgScalars init;
  std::memset(&init, 0, sizeof(init));
  init.one_m = op->one_m;
  init.max_iter = o->max_iter;
  if ((st = cuda_check(cudaMemcpyAsync(c->sc, &init, sizeof(init), cudaMemcpyHostToDevice, s), "scalars init"))) return st;
  const double* bw = launch_start<MASKC>(op, val, b, x, proj, o, s);
  launch_first(op, which, proj, prec, dinv, s);
  if ((st = read_scalars(c, s))) return st;
  int restarts = 0;
  int first_pass = 0;
  int status = PM_OK;
  double rel_true = 0.0, rel_floor = 0.0, prev_true = -1.0;
  bool accepted = false;
  if (c->sc_host->zero_rhs) {
    k_fill<<<G, TPB, 0, s>>>(x, op->n, 0.0);
    count_launch();
    if ((st = read_scalars(c, s))) return st;
  } else {
    int64_t issued = 0;
    for (;;) {
      int chunk = 4;
      while (!c->sc_host->done) {
        // the device stops itself at max_iter; this bound only guards the host loop
        if (issued > (int64_t)o->max_iter + 4096)
          return set_error(PM_ECUDA, "PCG driver: device never reported completion");
        for (int it = 0; it < chunk; ++it) launch_iter<MASKC>(op, which, val, x, proj, prec, dinv, s);
        issued += chunk;
        if ((st = read_scalars(c, s))) return st;
        if (chunk < 64) chunk *= 2;
      }
      status = c->sc_host->status;
      if (restarts == 0) first_pass = c->sc_host->iter;
      // true residual
      launch_residual<MASKC>(op, val, bw, x, o->rtol, 1, s);
      if ((st = read_scalars(c, s))) return st;
      rel_true = std::sqrt(c->sc_host->aux[0] / c->sc_host->bb);
      rel_floor = std::ldexp(1.0, -53) * std::sqrt(c->sc_host->aux[1] / c->sc_host->bb);
      // Accepted when the (compensated, hence exact to one rounding) true residual meets rtol,
      // or when it lies below the floor that rounding x to FP64 alone can cause (backward error
      // at the unit roundoff) and restarts no longer lower it: the last restart did not halve
      // it, or no restart is left.
      const bool stalled = prev_true >= 0.0 && rel_true > 0.5 * prev_true;
      const bool last = restarts >= o->max_restarts || c->sc_host->iter >= o->max_iter;
      accepted = rel_true <= o->rtol || (rel_true <= rel_floor && (stalled || last));
      if (status != PM_OK || accepted || last) break;
      prev_true = rel_true;
      ++restarts;
      // restart from the true residual held in r
      PcgScalars* hs = c->sc_host;
      hs->done = 0;
      hs->rr = hs->aux[0];
      if ((st = cuda_check(cudaMemcpyAsync(c->sc, hs, sizeof(PcgScalars), cudaMemcpyHostToDevice, s), "scalars"))) return st;
      launch_first(op, which, proj, prec, dinv, s);
      if ((st = read_scalars(c, s))) return st;
    }
    if (status == PM_OK && !accepted) status = PM_NOT_CONVERGED;
  }
  if (proj) {
    // keep m'x = 0 exactly as returned result
    k_cg_press_sums<<<G, TPB, 0, s>>>(op->n, b, x, op->d_m, 1, c->partials, c->sc);
    k_shift_by<<<G, TPB, 0, s>>>(x, op->n, c->sc);
    count_launch(2);
    if ((st = read_scalars(c, s))) return st;
  }
  const PcgScalars* h = c->sc_host;
  if (stats) {
    stats->iters = h->iter;
    stats->outer_iters = restarts;
    stats->first_pass_iters = first_pass;
    stats->rel_residual_floor = rel_floor;
    stats->status = status;
    stats->rel_residual_true = h->zero_rhs ? 0.0 : rel_true;
    stats->rel_residual_rec = h->zero_rhs ? 0.0 : std::sqrt(h->rr / h->bb);
    stats->bytes_moved = h->iter * bytes_per_iter(op, prec, proj);
    stats->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  }
  if ((st = cuda_check(cudaGetLastError(), "pcg kernels"))) return st;
  if (status != PM_OK) {
    return set_error(status, status == PM_NOT_CONVERGED ? "PCG did not reach rtol within max_iter"
                                                        : "PCG breakdown: (p, Ap) <= 0 or non-finite");
  }
  return PM_OK;
}

// ---- resident solve: one launch runs the whole PCG (pm_resident.cuh) ---------------------------
constexpr int64_t RESIDENT_MAX_ROWS = 1 << 20;    // accepted when requested explicitly
// Automatic choice of the resident solve (measured lines: resident_auto).
constexpr int64_t RESIDENT_AUTO_ROWS = 3 << 20, RESIDENT_AUTO_IC0 = 2 << 20, RESIDENT_AUTO_MIXED_LINE = 5 << 18;

static_assert(sizeof(resident::Out) <= 64 && sizeof(resident::Ctl) <= 64, "resident buffers");

// Preconditioner data a solve reads: Jacobi diagonal, line or IC0 factor.
int ensure_prec(pm_operator* op, int which, int prec, cudaStream_t s) {
  int st;
  if ((st = launch_dinv(op, which, s))) return st;
  if (prec == PM_PREC_IC0 && !op->ic0[which].ok) {
    int bd = 0;
    for (int m = -1; m <= 10; ++m) {
      if ((st = launch_ic0_factor(op, which, m < 0 ? 0.0 : 1e-3 * std::pow(2.0, m), &bd, s))) return st;
      if (!bd) break;
    }
    if (bd) return set_error(PM_BREAKDOWN, "IC0 pivot failure after the shift limit");
  }
  return prec == PM_PREC_LINE ? line_factor(op, which, s) : PM_OK;
}

// The operands of a resident solve that do not depend on its precision.
resident::Args resident_args(pm_operator* op, int which, const double* b, double* x, const pm_solve_opts* o) {
  SolveCtx* c = op->ctx;
  resident::Args a;
  std::memset(&a, 0, sizeof(a));
  const int mc = which_mask(which);
  a.g = geom_of(op);
  a.val64 = op->d_val[which_valset(which)];
  a.mask = mc >= 0 ? op->d_keep[mc] : op->d_struct;
  a.b = b;
  a.x = x;
  a.bw = c->bw;
  a.m = op->d_m;
  a.cnbr = op->d_cnbr;
  a.ccls = op->d_ccls;
  a.colpos = op->d_colpos;
  const CMap cm = cmap_of(op);
  for (int q = 0, off = 0; q < 4; ++q) {
    a.cls_off[q] = off;
    a.cls_cnt[q] = op->cls_count[q];
    off += op->cls_count[q];
  }
  for (int q = 0; q < 8; ++q) a.cbase[q] = (int32_t)cm.cbase[q];
  a.nlev[0] = fast_div(cm.nlev[0]);
  a.nlev[1] = fast_div(cm.nlev[1]);
  a.rtol = o->rtol;
  a.inner_rtol = o->inner_rtol > 0.0 ? o->inner_rtol : 1e-2;
  a.one_m = op->one_m;
  a.max_iter = o->max_iter;
  a.max_restarts = o->max_restarts;
  a.x0_is_guess = o->x0_is_guess ? 1 : 0;
  a.proj = which == PM_OP_PRESSURE ? 1 : 0;
  a.ctl = static_cast<resident::Ctl*>(c->res_ctl);
  a.part = c->partials;
  a.out = static_cast<resident::Out*>(c->res_out);
  return a;
}

// ---- mixed precision: FP32 / BF16 operator values, FP32 inner PCG, FP64 outer refinement -------
// Outer (FP64): r = b - A x with the FP64 operator; stop when ||r|| <= rtol ||b|| or below the
// FP64 floor. Inner: PCG on A d = r with the operator values in FP32 (or BF16), FP32 vectors and
// FP32 SpMV / preconditioner arithmetic, FP64 dot products and alpha / beta, to a relative
// reduction inner_rtol; then x += d in FP64.

// m'z with m held exactly as two floats (hi + lo = m in FP64 to 48 bits) for the FP32 kernels.
__device__ __forceinline__ void add_mz(DF& acc, float2 m2, float z) {
  acc.add_prod(m2.x, z);
  acc.add_prod(m2.y, z);
}

__device__ __forceinline__ float ldv(const float* p, int i) { return __ldg(p + i); }
__device__ __forceinline__ float ldv(const __nv_bfloat16* p, int i) { return __bfloat162float(p[i]); }

// Low-precision operator in difference form. The low-precision copy keeps the 14 off-diagonal
// values and stores, in the diagonal slot, the FP64 row sum rs_i = sum_j a_ij (0 for the pure-
// Neumann pressure operator). Then
//   (A x)_i = (rs_i - sum_{j eliminated} a_ij) x_i + sum_{j kept, j != i} a_ij (x_j - x_i),
// which is A x exactly, but rounds each a_ij (x_j - x_i) instead of cancelling large a_ij x_j
// terms: for vectors that are smooth along the strong (vertical) couplings this keeps the
// relative accuracy that FP32 / BF16 would otherwise lose on the thin-domain operators, and the
// constant null space of the pressure operator is exact in any precision.
template <int MASKC, typename TV>
__device__ __forceinline__ float row_dot32(const Geom& g, const TV* __restrict__ val, const float* __restrict__ x,
                                           int row, int col, int k) {
  const int nz = g.nz;
  const int npad = (int)g.npad;
  int nb[NNBR];
  uint8_t fl[NNBR];
  nb[0] = col;
#pragma unroll
  for (int q = 1; q < NNBR; ++q) nb[q] = nbr_of(g, col, q);
  if (MASKC >= 0) {
#pragma unroll
    for (int q = 0; q < NNBR; ++q) fl[q] = __ldg(g.colflag + (nb[q] >= 0 ? nb[q] : col));
    if (is_dirichlet(fl[0], k, nz, MASKC)) return x[row];
  }
  float a[NSLOT];
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) a[s] = ldv(val, s * npad + row);
  const float xi = x[row];
  float sum = 0.f, drop = 0.f;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    if (s == DIAG_SLOT) continue;
    const int q = slot_q(s);
    const int kk = k + slot_dk(s);
    bool ok = nb[q] >= 0;
    if (slot_dk(s) < 0) ok = ok && kk >= 0;
    if (slot_dk(s) > 0) ok = ok && kk < nz;
    bool keep = ok;
    if (MASKC >= 0) {
      const bool dj = ok && is_dirichlet(fl[q], kk, nz, MASKC);
      keep = ok && !dj;
      drop += dj ? a[s] : 0.f;
    }
    const float xv = x[keep ? nb[q] * nz + kk : row];
    sum = fmaf(keep ? a[s] : 0.f, xv - xi, sum);
  }
  return fmaf(a[DIAG_SLOT] - drop, xi, sum);
}

// row_dot32 for a velocity component through its keep mask (see row_dot_keep): a slot whose
// neighbour is present but eliminated adds its value to the drop term.
template <typename TV>
__device__ __forceinline__ float row_dot32_keep(const Geom& g, const TV* __restrict__ val, const float* __restrict__ x,
                                                const uint16_t* __restrict__ keep, int row, int col, int k) {
  const int nz = g.nz;
  const int npad = (int)g.npad;
  const uint32_t km = __ldg(keep + row);
  if (km & 0x8000u) return x[row];
  int nb[NNBR];
  nb[0] = col;
#pragma unroll
  for (int q = 1; q < NNBR; ++q) nb[q] = nbr_of(g, col, q);
  float a[NSLOT];
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) a[s] = ldv(val, s * npad + row);
  const float xi = x[row];
  float sum = 0.f, drop = 0.f;
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) {
    if (s == DIAG_SLOT) continue;
    const int q = slot_q(s);
    const int kk = k + slot_dk(s);
    bool exists = nb[q] >= 0;
    if (slot_dk(s) < 0) exists = exists && kk >= 0;
    if (slot_dk(s) > 0) exists = exists && kk < nz;
    const bool keep_s = (km >> s) & 1u;
    drop += (exists && !keep_s) ? a[s] : 0.f;
    const float xv = x[keep_s ? nb[q] * nz + kk : row];
    sum = fmaf(keep_s ? a[s] : 0.f, xv - xi, sum);
  }
  return fmaf(a[DIAG_SLOT] - drop, xi, sum);
}

// Low-precision copy in difference form: off-diagonals rounded, diagonal slot = FP64 row sum
// (zero_rowsum: exactly 0, the pure-Neumann operator).
template <typename T>
__global__ void k_cvt_diff(int64_t n, int64_t npad, const double* __restrict__ val, T* __restrict__ out,
                           int zero_rowsum) {
  for (int64_t row = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; row < npad; row += (int64_t)gridDim.x * blockDim.x) {
    double rs = 0.0;
#pragma unroll
    for (int s = 0; s < NSLOT; ++s) {
      const double v = val[s * npad + row];
      rs += v;
      if (s != DIAG_SLOT) {
        if constexpr (std::is_same<T, float>::value) out[s * npad + row] = (float)v;
        else out[s * npad + row] = __double2bfloat16(v);
      }
    }
    if (zero_rowsum || row >= n) rs = 0.0;
    if constexpr (std::is_same<T, float>::value) out[DIAG_SLOT * npad + row] = (float)rs;
    else out[DIAG_SLOT * npad + row] = __double2bfloat16(rs);
  }
}

// Four consecutive rows of one slot's values.
__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(p));
  v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
}
__device__ __forceinline__ void ld4(const __nv_bfloat16* p, float (&v)[4]) {
  const uint2 t = __ldg(reinterpret_cast<const uint2*>(p));   // bf16 is the upper half of an FP32 number
  v[0] = __uint_as_float(t.x << 16), v[1] = __uint_as_float(t.x & 0xffff0000u);
  v[2] = __uint_as_float(t.y << 16), v[3] = __uint_as_float(t.y & 0xffff0000u);
}

// k32_spmv for level counts that are multiples of 4: four consecutive rows of a column per thread, so that a
// slot's values and a neighbour column's entries are one 16-byte load each (the entry above or below the four is a
// load of its own): 37 loads for four rows instead of 148. The FP32 SpMV is bound by load instructions,
// not by its 68 bytes a row. Slots by the mask (structural slots, or a component's kept ones): a clear
// bit's value is 0 or, eliminated, goes to the drop term.
template <typename TV>
__global__ void __launch_bounds__(TPB, 2) k32_spmv4(Geom g, const TV* __restrict__ val, const float* __restrict__ p,
                                                    float* __restrict__ w, const uint16_t* __restrict__ mask,
                                                    double* partials, PcgScalars* sc) {
  if (sc_done(sc)) return;
  DF dot;
  const int n4 = (int)(g.n >> 2), nz = g.nz, npad = (int)g.npad;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n4; j += gridDim.x * blockDim.x) {
    const int row = 4 * j, col = fdiv(g.nzd, row), k = row - col * nz;
    const uint2 mk = __ldg(reinterpret_cast<const uint2*>(mask + row));
    const uint32_t km[4] = {mk.x & 0xffffu, mk.x >> 16, mk.y & 0xffffu, mk.y >> 16};
    float x[NNBR][6];   // entries k - 1 .. k + 4 of each neighbour column (unused ones never loaded)
#pragma unroll
    for (int q = 0; q < NNBR; ++q) {
      const int nb = q == 0 ? col : nbr_of(g, col, q);
      const bool up = q == 0 || (q & 1), down = q == 0 || !(q & 1);   // slots with dk = +1, dk = -1
      const float* c = p + (nb >= 0 ? nb * nz + k : row);
      float t[4];
      ld4(c, t);
#pragma unroll
      for (int u = 0; u < 4; ++u) x[q][u + 1] = t[u];
      x[q][0] = down && k > 0 ? (nb >= 0 ? c[-1] : 0.f) : 0.f;
      x[q][5] = up && k + 4 < nz ? (nb >= 0 ? c[4] : 0.f) : 0.f;
    }
    float sum[4] = {0.f, 0.f, 0.f, 0.f}, drop[4] = {0.f, 0.f, 0.f, 0.f}, diag[4];
#pragma unroll
    for (int s = 0; s < NSLOT; ++s) {
      float a[4];
      ld4(val + s * npad + row, a);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (s == DIAG_SLOT) {
          diag[u] = a[u];
          continue;
        }
        const bool keep = (km[u] >> s) & 1u;
        drop[u] += keep ? 0.f : a[u];
        sum[u] = fmaf(keep ? a[u] : 0.f, x[slot_q(s)][u + 1 + slot_dk(s)] - x[0][u + 1], sum[u]);
      }
    }
    float4 out;
    float* o = &out.x;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float xi = x[0][u + 1];
      o[u] = (km[u] & 0x8000u) ? xi : fmaf(diag[u] - drop[u], xi, sum[u]);
      dot.add_prod(xi, o[u]);
    }
    *reinterpret_cast<float4*>(w + row) = out;
  }
  double v[1] = {dot.value()};
  if (grid_sum<1>(v, partials, &sc->count[3]) && threadIdx.x == 0) {
    const double pap = v[0];
    sc->pAp = pap;
    if (!(pap > 0.0) || !isfinite(pap)) {
      sc->status = PM_BREAKDOWN;
      sc->done = 1;
    } else {
      sc->alpha = sc->rho / pap;
    }
  }
}

template <int MASKC, typename TV>
__global__ void __launch_bounds__(TPB, 4) k32_spmv(Geom g, const TV* __restrict__ val, const float* __restrict__ p,
                                                   float* __restrict__ w, const uint16_t* __restrict__ keep,
                                                   double* partials, PcgScalars* sc) {
  if (sc_done(sc)) return;
  double v[1] = {0.0};
  DF a0;
  const int n = (int)g.n;
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < n; row += gridDim.x * blockDim.x) {
    const int col = row / g.nz;
    const int k = row - col * g.nz;
    const float wi = MASKC >= 0 ? row_dot32_keep<TV>(g, val, p, keep, row, col, k) : row_dot32<MASKC, TV>(g, val, p, row, col, k);
    w[row] = wi;
    a0.add_prod(p[row], wi);
  }
  v[0] = a0.value();
  if (grid_sum<1>(v, partials, &sc->count[3]) && threadIdx.x == 0) {
    const double pap = v[0];
    sc->pAp = pap;
    if (!(pap > 0.0) || !isfinite(pap)) {
      sc->status = PM_BREAKDOWN;
      sc->done = 1;
    } else {
      sc->alpha = sc->rho / pap;
    }
  }
}

// d += alpha p, r -= alpha w (FP32; d is the correction since the last residual replacement,
// folded into the FP64 x there); INLINE_Z: z = dinv r (Jacobi) and its reductions.
template <int PROJ, int INLINE_Z>
__global__ void __launch_bounds__(TPB) k32_update(int64_t n, float* __restrict__ d, float* __restrict__ r,
                                                  const float* __restrict__ p, const float* __restrict__ w,
                                                  const float* __restrict__ dinv, const float2* __restrict__ m2,
                                                  double* partials, PcgScalars* sc) {
  if (sc_done(sc)) return;
  const double alpha_d = sc->alpha;
  const float alpha = (float)alpha_d;
  DF a[4];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    d[i] = fmaf(alpha, p[i], d[i]);
    const float ri = fmaf(-alpha, w[i], r[i]);
    r[i] = ri;
    a[0].add_prod(ri, ri);
    if (INLINE_Z) {
      const float zi = dinv[i] * ri;
      a[1].add_prod(ri, zi);
      if (PROJ) {
        add_mz(a[2], m2[i], zi);
        a[3].add(ri);
      }
    }
  }
  double v[4] = {a[0].value(), a[1].value(), a[2].value(), a[3].value()};
  if (grid_sum<4>(v, partials, &sc->count[4]) && threadIdx.x == 0) {
    sc->iter += 1;
    sc->rr = v[0];
    if (v[0] <= sc->tol2) {
      sc->done = 1;
    } else if (sc->iter >= sc->max_iter) {
      sc->status = PM_NOT_CONVERGED;
      sc->done = 1;
    } else if (v[0] <= sc->aux[2]) {
      sc->done = 2;  // residual replacement requested (mixed precision): the host finishes the step
    } else if (INLINE_Z) {
      const double c = PROJ ? v[2] / sc->one_m : 0.0;
      const double rho_new = v[1] - c * v[3];
      sc->proj_c = c;
      sc->beta = rho_new / sc->rho;
      sc->rho = rho_new;
      if (!(rho_new > 0.0) || !isfinite(rho_new)) {
        sc->status = PM_BREAKDOWN;
        sc->done = 1;
      }
    }
  }
}

// First preconditioned residual: rho = (r, z') with z' = z - c (pressure), z = dinv r; beta = 0.
template <int PROJ>
__global__ void __launch_bounds__(TPB) k32_rho(int64_t n, const float* __restrict__ r, const float* __restrict__ dinv,
                                               const float2* __restrict__ m2, double* partials, PcgScalars* sc) {
  DF a[3];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float ri = r[i];
    const float zi = dinv[i] * ri;
    a[0].add_prod(ri, zi);
    if (PROJ) {
      add_mz(a[1], m2[i], zi);
      a[2].add(ri);
    }
  }
  double v[3] = {a[0].value(), a[1].value(), a[2].value()};
  if (grid_sum<3>(v, partials, &sc->count[2]) && threadIdx.x == 0) {
    const double c = PROJ ? v[1] / sc->one_m : 0.0;
    const double rho_new = v[0] - c * v[2];
    sc->proj_c = c;
    sc->rho = rho_new;
    sc->beta = 0.0;
    if ((!(rho_new > 0.0) || !isfinite(rho_new)) && !sc->done) {
      sc->status = PM_BREAKDOWN;
      sc->done = 1;
    }
  }
}

template <int STORED>
__global__ void __launch_bounds__(TPB) k32_pupd(int64_t n, const float* __restrict__ r, const float* __restrict__ dinv,
                                                const float* __restrict__ zbuf, float* __restrict__ p,
                                                const PcgScalars* sc, int is_first) {
  if (!is_first && sc_done(sc)) return;
  const float beta = (float)sc->beta, c = (float)sc->proj_c;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float zi = (STORED ? zbuf[i] : dinv[i] * r[i]) - c;
    p[i] = is_first ? zi : fmaf(beta, p[i], zi);
  }
}

// k32_pupd<1> after the first step, four entries per thread (16-byte loads: 4.7M rows 18.5 -> 13.8 us).
__global__ void __launch_bounds__(TPB) k32_pupd4(int n, const float* __restrict__ z, float* __restrict__ p,
                                                 const PcgScalars* sc) {
  if (sc_done(sc)) return;
  const float beta = (float)sc->beta, c = (float)sc->proj_c;
  const int n4 = n >> 2, stride = gridDim.x * blockDim.x, t = blockIdx.x * blockDim.x + threadIdx.x;
  const float4* z4 = reinterpret_cast<const float4*>(z);
  float4* p4 = reinterpret_cast<float4*>(p);
  for (int i = t; i < n4; i += stride) {
    const float4 zi = z4[i], pi = p4[i];
    p4[i] = make_float4(fmaf(beta, pi.x, zi.x - c), fmaf(beta, pi.y, zi.y - c), fmaf(beta, pi.z, zi.z - c),
                        fmaf(beta, pi.w, zi.w - c));
  }
  for (int i = 4 * n4 + t; i < n; i += stride) p[i] = fmaf(beta, p[i], z[i] - c);
}

// m = hi + lo as two floats (hi = fl32(m), lo = fl32(m - hi)) for the FP32 kernels' m'z.
__global__ void k_split_m(int64_t n, const double* __restrict__ m, float2* __restrict__ m2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float hi = (float)m[i];
    m2[i] = make_float2(hi, (float)(m[i] - (double)hi));
  }
}

// x += d (FP64), d = 0: the inner solve's FP32 correction folded into the FP64 iterate.
__global__ void k32_fold(int64_t n, double* __restrict__ x, float* __restrict__ d) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    x[i] += (double)d[i];
    d[i] = 0.f;
  }
}

__global__ void k32_from64(int64_t n, const double* __restrict__ r64, float* __restrict__ r32) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    r32[i] = (float)r64[i];
}

__global__ void k_fill32(float* x, int64_t n, float v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) x[i] = v;
}

template <typename T>
__global__ void k_cvt(int64_t n, const double* __restrict__ in, T* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if constexpr (std::is_same<T, float>::value) out[i] = (float)in[i];
    else out[i] = __double2bfloat16(in[i]);
  }
}

// FP32 version of k_update_line_w (warp tasks of TC columns, no block barriers), for any number of
// levels that fits (NZ = 0: g.nz, rows of a task taken flat); the FP32 correction d takes alpha p (folded into
// the FP64 x at each refinement) and the dots are accumulated in compensated FP32. mode 0: first step (z,
// rho, beta = 0); 1: a full iteration (d, r update, z, rho, beta). (r, z) = sum_k t_k y_k from the sweep (symmetric column blocks, see
// k_update_line_w). Half-wide tasks (TC = 16): the FP32 pipe has room for idle lanes, and more tasks per warp keep
// some warps streaming while others sweep.
template <int PROJ, int TC, int NZ>
__global__ void __launch_bounds__(LINE_WTPB, 4) k32_update_line_w(Geom g, const float* __restrict__ F,
                                                              float* __restrict__ d, float* __restrict__ r,
                                                              const float* __restrict__ p, const float* __restrict__ w,
                                                              float* __restrict__ z, const float2* __restrict__ m2,
                                                              double* partials, PcgScalars* sc, int mode) {
  extern __shared__ float smf[];
  const int update = mode == 1;
  if (mode != 0 && sc_done(sc)) return;
  const double alpha_d = update ? sc->alpha : 0.0;
  const float alpha = (float)alpha_d;
  const int nz = NZ > 0 ? NZ : g.nz, ld = nz | 1;
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  float* ws = smf + wib * (TC * ld);
  const int ncols = g.ncols;
  const int n = (int)g.n;
  const int nwarps = gridDim.x * (LINE_WTPB / 32);
  const int wg = blockIdx.x * (LINE_WTPB / 32) + wib;
  const int ntask = (ncols + TC - 1) / TC;
  const int tbeg = (int)((int64_t)ntask * wg / nwarps);
  const int tend = (int)((int64_t)ntask * (wg + 1) / nwarps);
  // place of the task's i-th row in the tile of columns
  const auto at = [&](int i) {
    if (NZ > 0) return (i / (NZ > 0 ? NZ : 1)) * ld + i % (NZ > 0 ? NZ : 1);
    const int c = fdiv(g.nzd, i);
    return c * ld + i - c * nz;
  };
  DF a[4];   // (r, r), (r, z), m'z, 1'r
  for (int t = tbeg; t < tend; ++t) {
    const int c0 = t * TC;
    const int cc = min(TC, ncols - c0);
    const int row0 = c0 * nz, rows = cc * nz;
#pragma unroll 8
    for (int i = lane; i < rows; i += 32) {
      const int row = row0 + i;
      float ri = r[row];
      if (update) {
        d[row] = fmaf(alpha, p[row], d[row]);
        ri = fmaf(-alpha, w[row], ri);
        r[row] = ri;
      }
      ws[at(i)] = ri;
      a[0].add_prod(ri, ri);
      if (PROJ) a[3].add(ri);
    }
    __syncwarp();
    if (lane < cc) {
      const int col = c0 + lane;
      float* cs = ws + lane * ld;
      float y = 0.f;
#pragma unroll 8
      for (int k = 0; k < nz; ++k) {
        const int li = k * ncols + col;
        const float tk = fmaf(-F[li], y, cs[k]);
        y = tk * F[n + li];
        a[1].add_prod(tk, y);
        cs[k] = y;
      }
      float zn = y;
#pragma unroll 8
      for (int k = nz - 2; k >= 0; --k) {
        const int li = k * ncols + col;
        zn = fmaf(-F[2 * n + li], zn, cs[k]);
        cs[k] = zn;
      }
    }
    __syncwarp();
#pragma unroll 8
    for (int i = lane; i < rows; i += 32) {
      const int row = row0 + i;
      const float zi = ws[at(i)];
      z[row] = zi;
      if (PROJ) add_mz(a[2], m2[row], zi);
    }
    __syncwarp();
  }
  double v[4] = {a[0].value(), a[1].value(), a[2].value(), a[3].value()};
  if (grid_sum<4>(v, partials, &sc->count[4]) && threadIdx.x == 0) {
    const double c = PROJ ? v[2] / sc->one_m : 0.0;
    const double rho_new = v[1] - c * v[3];
    if (mode == 0) {
      sc->proj_c = c;
      sc->rho = rho_new;
      sc->beta = 0.0;
      if ((!(rho_new > 0.0) || !isfinite(rho_new)) && !sc->done) {
        sc->status = PM_BREAKDOWN;
        sc->done = 1;
      }
    } else {
      sc->iter += 1;
      sc->rr = v[0];
      if (v[0] <= sc->tol2) {
        sc->done = 1;
      } else if (sc->iter >= sc->max_iter) {
        sc->status = PM_NOT_CONVERGED;
        sc->done = 1;
      } else if (v[0] <= sc->aux[2]) {
        sc->done = 2;
      } else {
        sc->proj_c = c;
        sc->beta = rho_new / sc->rho;
        sc->rho = rho_new;
        if (!(rho_new > 0.0) || !isfinite(rho_new)) {
          sc->status = PM_BREAKDOWN;
          sc->done = 1;
        }
      }
    }
  }
}

// The FP32 fused update + line solve (mode as k32_update_line_w). One launch; the caller counts it.
constexpr int LINE32_TC = 16;
constexpr size_t LINE32_TILE = 200 * 1024;   // shared memory of a block's warp tiles: up to 399 levels
size_t line32_tile(int nz) { return (size_t)(LINE_WTPB / 32) * LINE32_TC * (nz | 1) * sizeof(float); }

template <int PROJ, int NZ>
int line32_setup(pm_operator* op) {
  int& slots = op->ctx->line32_slots[PROJ];
  if (slots) return PM_OK;
  const void* kern = (const void*)k32_update_line_w<PROJ, LINE32_TC, NZ>;
  int st, per_sm = 0;
  if ((st = smem_limit(kern, LINE32_TILE))) return st;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, LINE_WTPB, line32_tile(op->nz));
  slots = std::max(1, per_sm) * op->num_sms;
  return PM_OK;
}
// What the FP32 line kernel needs before its first launch for this operator.
int line32_setup(pm_operator* op, bool proj) {
  if (op->nz == LINE_WNZ) return proj ? line32_setup<1, LINE_WNZ>(op) : line32_setup<0, LINE_WNZ>(op);
  return proj ? line32_setup<1, 0>(op) : line32_setup<0, 0>(op);
}

template <int PROJ, int NZ>
void launch_line32_w(pm_operator* op, int which, int mode, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  // the resident blocks, capped by the partials buffer (4 lanes per block) and by one task per warp
  const int64_t ntask = (op->ncols + LINE32_TC - 1) / LINE32_TC;
  int64_t blocks = std::min<int64_t>(c->line32_slots[PROJ], (int64_t)NPART * MAX_GRID / 4);
  blocks = std::min<int64_t>(blocks, (ntask + LINE_WTPB / 32 - 1) / (LINE_WTPB / 32));
  k32_update_line_w<PROJ, LINE32_TC, NZ><<<(int)std::max<int64_t>(1, blocks), LINE_WTPB, line32_tile(op->nz), s>>>(
      geom_of(op), op->d_line32[which], c->d32, c->r32, c->p32, c->w32, c->z32, op->d_m2f, c->partials, c->sc_in, mode);
}

void update_line32(pm_operator* op, int which, bool proj, int mode, cudaStream_t s) {
  if (op->nz == LINE_WNZ) proj ? launch_line32_w<1, LINE_WNZ>(op, which, mode, s) : launch_line32_w<0, LINE_WNZ>(op, which, mode, s);
  else proj ? launch_line32_w<1, 0>(op, which, mode, s) : launch_line32_w<0, 0>(op, which, mode, s);
}

int ensure_mixed(pm_operator* op, int which, int precision, int prec, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  const size_t fb = (size_t)op->n * sizeof(float);
  if (!c->r32) {
    cudaError_t e = cudaSuccess;
    e = e ? e : cudaMalloc((void**)&c->r32, fb);
    e = e ? e : cudaMalloc((void**)&c->p32, fb);
    e = e ? e : cudaMalloc((void**)&c->w32, fb);
    e = e ? e : cudaMalloc((void**)&c->z32, fb);
    e = e ? e : cudaMalloc((void**)&c->d32, fb);
    e = e ? e : cudaMalloc((void**)&c->sc_in, sizeof(PcgScalars));
    e = e ? e : cudaMallocHost((void**)&c->sc_in_host, sizeof(PcgScalars));
    if (e != cudaSuccess) return cuda_check(e, "mixed-precision workspace");
    op->device_bytes += 5 * (int64_t)fb;
  }
  if (!op->d_m2f) {
    int st = cuda_check(cudaMalloc((void**)&op->d_m2f, (size_t)op->n * sizeof(float2)), "cudaMalloc m split");
    if (st) return st;
    op->device_bytes += op->n * 8;
    k_split_m<<<grid_for(op->n, TPB, op->num_sms), TPB, 0, s>>>(op->n, op->d_m, op->d_m2f);
    count_launch();
  }
  const int vs = which_valset(which);
  const int64_t nv = (int64_t)NSLOT * op->npad;
  const int G = grid_for(nv, TPB, op->num_sms);
  const int zero_rs = vs == VS_KI ? 1 : 0;
  const int Gr = grid_for(op->npad, TPB, op->num_sms);
  (void)G;
  if (precision == PM_FP32_REFINE && !op->d_val32[vs]) {
    int st = cuda_check(cudaMalloc((void**)&op->d_val32[vs], nv * sizeof(float)), "cudaMalloc fp32 values");
    if (st) return st;
    op->device_bytes += nv * 4;
    k_cvt_diff<float><<<Gr, TPB, 0, s>>>(op->n, op->npad, op->d_val[vs], op->d_val32[vs], zero_rs);
    count_launch();
  }
  if (precision == PM_BF16_REFINE && !op->d_val16[vs]) {
    int st = cuda_check(cudaMalloc((void**)&op->d_val16[vs], nv * sizeof(uint16_t)), "cudaMalloc bf16 values");
    if (st) return st;
    op->device_bytes += nv * 2;
    k_cvt_diff<__nv_bfloat16><<<Gr, TPB, 0, s>>>(op->n, op->npad, op->d_val[vs],
                                                reinterpret_cast<__nv_bfloat16*>(op->d_val16[vs]), zero_rs);
    count_launch();
  }
  if (prec == PM_PREC_LINE && !op->d_line32[which]) {
    int st = cuda_check(cudaMalloc((void**)&op->d_line32[which], 3 * fb), "cudaMalloc fp32 line");
    if (st) return st;
    op->device_bytes += 3 * (int64_t)fb;
    k_cvt<float><<<grid_for(3 * op->n, TPB, op->num_sms), TPB, 0, s>>>(3 * op->n, op->d_line[which], op->d_line32[which]);
    count_launch();
  }
  if (prec == PM_PREC_IC0 && !op->d_ic0_32[which]) {
    int st = cuda_check(cudaMalloc((void**)&op->d_ic0_32[which], (size_t)NSLOT * fb), "cudaMalloc fp32 ic0");
    if (st) return st;
    op->device_bytes += (int64_t)NSLOT * fb;
    k_cvt<float><<<grid_for(NSLOT * op->n, TPB, op->num_sms), TPB, 0, s>>>(NSLOT * op->n, op->ic0[which].F,
                                                                          op->d_ic0_32[which]);
    count_launch();
  }
  return cuda_check(cudaGetLastError(), "mixed set-up");
}

int read_inner(SolveCtx* c, cudaStream_t s) {
  int st = cuda_check(cudaMemcpyAsync(c->sc_in_host, c->sc_in, sizeof(PcgScalars), cudaMemcpyDeviceToHost, s), "scalars");
  if (st) return st;
  st = cuda_check(cudaStreamSynchronize(s), "mixed pcg sync");
  if (!st && !g_kt.pending.empty()) kt_collect();
  return st;
}

// Algorithmic bytes per inner iteration per row (values at vbytes each; vectors FP32, the
// correction d read and written in FP32).
double bytes_per_inner(const pm_operator* op, int prec, int vbytes, bool proj) {
  const double n = (double)op->n;
  double b = n * (15 * vbytes + 4 + 4);                       // SpMV: values, p, w
  if (prec == PM_PREC_LINE) b += n * (8 + 8 + 4 + 4 + 12 + 4 + 12);  // d, r r/w; p, w; factors; z; p-update
  else if (prec == PM_PREC_IC0) b += n * (8 + 8 + 4 + 4 + 2 * 8 * 4 + 4 * 4 + 8 + 12);
  else b += n * (8 + 8 + 4 + 4 + 4 + 4 * 4);                   // Jacobi update (z inline), p-update
  if (proj) b += n * 8;                                         // m'z
  return b;
}

// FP64 residual, and the fold of the correction into x, of one refinement step.
double bytes_per_refine(const pm_operator* op) { return (double)op->n * (15 * 8 + 3 * 8 + 16 + 8); }

// Whether the automatic choice runs a solve resident. Measured against the stream of kernels, us per
// iteration, stream / resident:
//   FP64  IC0 n = 0.12M 132 / 51, 0.29M 170 / 63, 0.99M 231 / 150, 2.0M 266 / 269, 3.0M 336 / 362;
//         line 0.31M 64 / 35, 1.0M 110 / 88, 1.8M 152 / 130, 4.7M 316 / 327;
//         Jacobi 2.0M 140 / 126, 5.1M 275 / 296
//   FP32  IC0 0.12M 226 / 46, 2.0M 198 / 190, 3.0M 231 / 258; line 0.31M 40 / 25, 0.63M 48 / 32, 1.0M 67 / 62,
//         4.7M 150 / 218; Jacobi 1.0M 77 / 41, 2.25M 112 / 98, 5.1M 196 / 201.
bool resident_auto(const pm_operator* op, int prec, bool mixed) {
  return op->n <= (prec == PM_PREC_IC0             ? RESIDENT_AUTO_IC0
                   : mixed && prec == PM_PREC_LINE ? RESIDENT_AUTO_MIXED_LINE
                                                   : RESIDENT_AUTO_ROWS);
}

int resident_run(pm_operator* op, int which, const double* b, double* x, const pm_solve_opts* o,
                 pm_solve_stats* stats, cudaStream_t s) {
  auto t0 = std::chrono::steady_clock::now();
  SolveCtx* c = op->ctx;
  const int prec = o->prec;
  const bool mixed = o->precision != PM_FP64;
  int st;
  if ((st = ensure_prec(op, which, prec, s))) return st;
  if (mixed && (st = ensure_mixed(op, which, o->precision, prec, s))) return st;
  resident::Args a = resident_args(op, which, b, x, o);
  const int vs = which_valset(which);
  a.out->res.status = -1;
  a.out->timeout = 0;
  if (mixed) {
    a.val = o->precision == PM_FP32_REFINE ? (const void*)op->d_val32[vs] : (const void*)op->d_val16[vs];
    a.r = c->r32;
    a.p = c->p32;
    a.w = c->w32;
    a.z = c->z32;
    a.d = c->d32;
    a.m2 = op->d_m2f;
    a.dinv = prec == PM_PREC_NONE ? nullptr : op->d_dinv32[which];
    a.ic0 = op->d_ic0_32[which];
    a.line = op->d_line32[which];
    KtScope t(PM_KT_RESIDENT, 1, s);
    st = o->precision == PM_FP32_REFINE ? resident::launch_fp32(a, prec, op->num_sms, s)
                                        : resident::launch_bf16(a, prec, op->num_sms, s);
  } else {
    a.val = a.val64;
    a.r = c->r;
    a.p = c->p;
    a.w = c->w;
    a.z = c->z;
    a.dinv = prec == PM_PREC_NONE ? nullptr : op->d_dinv[which];
    a.ic0 = op->ic0[which].F;
    a.line = op->d_line[which];
    KtScope t(PM_KT_RESIDENT, 1, s);
    st = resident::launch_fp64(a, prec, op->num_sms, s);
  }
  if (st) return st;
  if ((st = cuda_check(cudaStreamSynchronize(s), "resident pcg"))) return st;
  if (!g_kt.pending.empty()) kt_collect();
  if ((st = resident::outcome(*a.out))) return st;
  const resident::Result h = a.out->res;
  if (stats) {
    stats->iters = h.iters;
    stats->outer_iters = h.restarts;
    stats->first_pass_iters = h.first_pass;
    stats->status = h.status;
    stats->rel_residual_true = h.rel_true;
    stats->rel_residual_rec = h.rel_rec;
    stats->rel_residual_floor = h.floor;
    stats->bytes_moved = mixed ? h.iters * bytes_per_inner(op, prec, o->precision == PM_FP32_REFINE ? 4 : 2, a.proj) +
                                     h.restarts * bytes_per_refine(op)
                               : h.iters * bytes_per_iter(op, prec, a.proj);
    stats->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  }
  if (h.status != PM_OK)
    return set_error(h.status, h.status == PM_NOT_CONVERGED
                                   ? mixed ? "mixed-precision PCG did not reach rtol" : "PCG did not reach rtol within max_iter"
                               : mixed ? "mixed-precision PCG breakdown"
                                       : "PCG breakdown: (p, Ap) <= 0 or non-finite");
  return PM_OK;
}

template <int MASKC, typename TV>
void inner_iter(pm_operator* op, int which, const TV* val32, bool proj, int prec, const float* dinv32,
                cudaStream_t s) {
  SolveCtx* c = op->ctx;
  Geom g = geom_of(op);
  const int G = grid_for(op->n, TPB, op->num_sms);
  {
    KtScope t(PM_KT_SPMV, 1, s);
    if (op->nz % 4 == 0)
      k32_spmv4<TV><<<grid_for(op->n / 4, TPB, op->num_sms), TPB, 0, s>>>(
          g, val32, c->p32, c->w32, MASKC >= 0 ? op->d_keep[MASKC < 0 ? 0 : MASKC] : op->d_struct, c->partials, c->sc_in);
    else
      k32_spmv<MASKC, TV><<<G, TPB, 0, s>>>(g, val32, c->p32, c->w32, MASKC >= 0 ? op->d_keep[MASKC < 0 ? 0 : MASKC] : nullptr,
                                            c->partials, c->sc_in);
  }
  if (prec == PM_PREC_LINE) {
    {
      KtScope t(PM_KT_LINE, 1, s);
      update_line32(op, which, proj, 1, s);
    }
    {
      KtScope t(PM_KT_PUPDATE, 1, s);
      k32_pupd4<<<grid_for(op->n / 4 + 1, TPB, op->num_sms), TPB, 0, s>>>((int)op->n, c->z32, c->p32, c->sc_in);
    }
    count_launch(3);
  } else if (prec == PM_PREC_IC0) {
    {
      KtScope t(PM_KT_UPDATE, 1, s);
      k32_update<0, 0><<<G, TPB, 0, s>>>(op->n, c->d32, c->r32, c->p32, c->w32, dinv32, op->d_m2f, c->partials, c->sc_in);
    }
    ic0_apply(op, op->d_ic0_32[which], c->r32, c->z32, proj ? op->d_m2f : nullptr, c->partials, c->sc_in, 0, s);
    {
      KtScope t(PM_KT_PUPDATE, 1, s);
      k_ic0_pupd<<<G, TPB, 0, s>>>(sweep_geo(op), c->z32, c->p32, c->sc_in, 0);
    }
    count_launch(3);
  } else {
    {
      KtScope t(PM_KT_UPDATE, 1, s);
      if (proj) k32_update<1, 1><<<G, TPB, 0, s>>>(op->n, c->d32, c->r32, c->p32, c->w32, dinv32, op->d_m2f, c->partials, c->sc_in);
      else k32_update<0, 1><<<G, TPB, 0, s>>>(op->n, c->d32, c->r32, c->p32, c->w32, dinv32, op->d_m2f, c->partials, c->sc_in);
    }
    {
      KtScope t(PM_KT_PUPDATE, 1, s);
      k32_pupd<0><<<G, TPB, 0, s>>>(op->n, c->r32, dinv32, nullptr, c->p32, c->sc_in, 0);
    }
    count_launch(3);
  }
}

// z = P^{-1} r32, rho = (r, z'), beta = 0, p = z': the first step of an inner solve.
void inner_first(pm_operator* op, int which, bool proj, int prec, const float* dinv32, cudaStream_t s) {
  SolveCtx* c = op->ctx;
  const int G = grid_for(op->n, TPB, op->num_sms);
  if (prec == PM_PREC_LINE) {
    update_line32(op, which, proj, 0, s);
    k32_pupd<1><<<G, TPB, 0, s>>>(op->n, c->r32, dinv32, c->z32, c->p32, c->sc_in, 1);
  } else if (prec == PM_PREC_IC0) {
    ic0_apply(op, op->d_ic0_32[which], c->r32, c->z32, proj ? op->d_m2f : nullptr, c->partials, c->sc_in, 1, s);
    k_ic0_pupd<<<G, TPB, 0, s>>>(sweep_geo(op), c->z32, c->p32, c->sc_in, 1);
  } else {
    if (proj) k32_rho<1><<<G, TPB, 0, s>>>(op->n, c->r32, dinv32, op->d_m2f, c->partials, c->sc_in);
    else k32_rho<0><<<G, TPB, 0, s>>>(op->n, c->r32, dinv32, op->d_m2f, c->partials, c->sc_in);
    k32_pupd<0><<<G, TPB, 0, s>>>(op->n, c->r32, dinv32, nullptr, c->p32, c->sc_in, 1);
  }
  count_launch(2);
}

template <int MASKC, typename TV>
int mixed_run(pm_operator* op, int which, const double* b, double* x, const pm_solve_opts* o, pm_solve_stats* stats,
              cudaStream_t s) {
  auto t0 = std::chrono::steady_clock::now();
  SolveCtx* c = op->ctx;
  const bool proj = which == PM_OP_PRESSURE;
  const int prec = o->prec;
  const double* val64 = op->d_val[which_valset(which)];
  int st;
  if (prec == PM_PREC_LINE && line32_tile(op->nz) > LINE32_TILE)
    return set_error(PM_ECUDA, "line preconditioner: columns too tall for shared memory");
  if (prec == PM_PREC_LINE && (st = line32_setup(op, proj))) return st;
  if ((st = ensure_prec(op, which, prec, s))) return st;
  if ((st = ensure_mixed(op, which, o->precision, prec, s))) return st;
  const int vs = which_valset(which);
  const TV* val32 = std::is_same<TV, float>::value ? reinterpret_cast<const TV*>(op->d_val32[vs])
                                                   : reinterpret_cast<const TV*>(op->d_val16[vs]);
  const float* dinv32 = op->d_dinv32[which];
  if (prec == PM_PREC_NONE) {  // plain CG: z = r, held as an all-ones diagonal in z32
    k_fill32<<<grid_for(op->n, TPB, op->num_sms), TPB, 0, s>>>(c->z32, op->n, 1.f);
    count_launch();
    dinv32 = c->z32;
  }
  // residual replacement each time the recursive residual has dropped by this factor
  const double inner_rtol = o->inner_rtol > 0.0 ? o->inner_rtol : 1e-2;
  const int G = grid_for(op->n, TPB, op->num_sms);
  PcgScalars init;
  std::memset(&init, 0, sizeof(init));
  init.one_m = op->one_m;
  init.max_iter = o->max_iter;
  if ((st = cuda_check(cudaMemcpyAsync(c->sc, &init, sizeof(init), cudaMemcpyHostToDevice, s), "scalars init"))) return st;
  const double* bw = launch_start<MASKC>(op, val64, b, x, proj, o, s);
  if ((st = read_scalars(c, s))) return st;
  const double bb = c->sc_host->bb;
  int outer = 0, inner_total = 0, status = PM_OK;
  double rel_true = 0.0, rel_floor = 0.0, bytes = 0.0;
  const int vbytes = std::is_same<TV, float>::value ? 4 : 2;
  if (c->sc_host->zero_rhs) {
    k_fill<<<G, TPB, 0, s>>>(x, op->n, 0.0);
    count_launch();
  } else if (c->sc_host->done) {
    // x0 already meets rtol (PM_OK), or max_iter = 0 (PM_NOT_CONVERGED): no inner solve runs
    status = c->sc_host->status;
    rel_true = std::sqrt(c->sc_host->rr / bb);
  } else {
    // Restarted refinement: inner PCG solves with r, p, w, z and the correction d in FP32 (dots
    // in compensated FP32 reduced in FP64, alpha and beta in FP64). Each time the recursive
    // residual has dropped by inner_rtol, or claims convergence, d is folded into the FP64 x, the
    // FP64 true residual b - A x (compensated) is formed, and a new inner solve starts from it.
    const double rr_drop = inner_rtol * inner_rtol;
    PcgScalars in;
    std::memset(&in, 0, sizeof(in));
    in.one_m = op->one_m;
    in.max_iter = o->max_iter;
    in.tol2 = c->sc_host->tol2;
    in.bb = bb;
    in.aux[2] = rr_drop * c->sc_host->rr;   // replacement threshold on the recursive (r, r)
    if ((st = cuda_check(cudaMemcpyAsync(c->sc_in, &in, sizeof(in), cudaMemcpyHostToDevice, s), "scalars"))) return st;
    k32_from64<<<G, TPB, 0, s>>>(op->n, c->r, c->r32);
    count_launch();
    if ((st = cuda_check(cudaMemsetAsync(c->d32, 0, (size_t)op->n * sizeof(float), s), "d32"))) return st;
    inner_first(op, which, proj, prec, dinv32, s);
    if ((st = read_inner(c, s))) return st;
    int64_t issued = 0;
    const int32_t zero = 0;
    int stalled = 0;
    double prev_true = 1e300;
    for (;;) {
      int chunk = 4;
      while (!c->sc_in_host->done) {
        if (issued > (int64_t)o->max_iter + 4096) return set_error(PM_ECUDA, "mixed PCG: device never reported completion");
        for (int it = 0; it < chunk; ++it) inner_iter<MASKC, TV>(op, which, val32, proj, prec, dinv32, s);
        issued += chunk;
        if ((st = read_inner(c, s))) return st;
        if (chunk < 64) chunk *= 2;
      }
      // fold the FP32 correction into x, then the FP64 true residual into c->r
      k32_fold<<<G, TPB, 0, s>>>(op->n, x, c->d32);
      count_launch();
      launch_residual<MASKC>(op, val64, bw, x, o->rtol, 1, s);
      if ((st = read_scalars(c, s))) return st;
      ++outer;
      bytes += bytes_per_refine(op);
      rel_true = std::sqrt(c->sc_host->aux[0] / bb);
      rel_floor = std::ldexp(1.0, -53) * std::sqrt(c->sc_host->aux[1] / bb);
      // the refinement step did not halve the (compensated) true residual
      const bool stalled_now = rel_true > 0.5 * prev_true;
      if (rel_true <= o->rtol || (rel_true <= rel_floor && stalled_now)) break;
      // stagnation above the floor: three replacements in a row that did not halve it
      stalled = stalled_now ? stalled + 1 : 0;
      prev_true = rel_true;
      if (stalled >= 3) {
        status = PM_NOT_CONVERGED;
        break;
      }
      if (c->sc_in_host->status == PM_BREAKDOWN) {
        status = PM_BREAKDOWN;
        break;
      }
      if (c->sc_in_host->iter >= o->max_iter) {  // no iteration left: accepted only below the floor
        status = rel_true <= rel_floor ? PM_OK : PM_NOT_CONVERGED;
        break;
      }
      // the next inner solve starts from r32 = (float)(b - A x)
      const double thr = rr_drop * c->sc_host->aux[0];
      if ((st = cuda_check(cudaMemcpyAsync(&c->sc_in->done, &zero, sizeof(zero), cudaMemcpyHostToDevice, s), "scalars")))
        return st;
      if ((st = cuda_check(cudaMemcpyAsync(&c->sc_in->aux[2], &thr, sizeof(thr), cudaMemcpyHostToDevice, s), "scalars")))
        return st;
      k32_from64<<<G, TPB, 0, s>>>(op->n, c->r, c->r32);
      count_launch();
      inner_first(op, which, proj, prec, dinv32, s);
      if ((st = read_inner(c, s))) return st;
    }
    inner_total = c->sc_in_host->iter;
    bytes += inner_total * bytes_per_inner(op, prec, vbytes, proj);
  }
  if (proj) {
    k_cg_press_sums<<<G, TPB, 0, s>>>(op->n, b, x, op->d_m, 1, c->partials, c->sc);
    k_shift_by<<<G, TPB, 0, s>>>(x, op->n, c->sc);
    count_launch(2);
    if ((st = read_scalars(c, s))) return st;
  }
  if (stats) {
    stats->iters = inner_total;
    stats->outer_iters = outer;
    stats->first_pass_iters = inner_total;
    stats->status = status;
    stats->rel_residual_true = c->sc_host->zero_rhs ? 0.0 : rel_true;
    stats->rel_residual_rec = stats->rel_residual_true;
    stats->rel_residual_floor = rel_floor;
    stats->bytes_moved = bytes;
    stats->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  }
  if ((st = cuda_check(cudaGetLastError(), "mixed pcg kernels"))) return st;
  if (status != PM_OK)
    return set_error(status, status == PM_NOT_CONVERGED ? "mixed-precision PCG did not reach rtol"
                                                        : "mixed-precision PCG breakdown");
  return PM_OK;
}

}  // namespace

int spmv(pm_operator* op, int which, const double* x, double* y, cudaStream_t s) {
  const int vs = which_valset(which);
  if (vs < 0) return set_error(PM_EINVAL, "unknown operator");
  Geom g = geom_of(op);
  const int G = grid_for(op->n, TPB, op->num_sms);
  switch (which_mask(which)) {
    case 0: k_spmv<0><<<G, TPB, 0, s>>>(g, op->d_val[vs], x, y); break;
    case 1: k_spmv<1><<<G, TPB, 0, s>>>(g, op->d_val[vs], x, y); break;
    case 2: k_spmv<2><<<G, TPB, 0, s>>>(g, op->d_val[vs], x, y); break;
    default: k_spmv<-1><<<G, TPB, 0, s>>>(g, op->d_val[vs], x, y); break;
  }
  count_launch();
  return cuda_check(cudaGetLastError(), "k_spmv");
}

namespace {
// r = b - A x by row_residual_dot2, with the grid sums (r, r), (|A||x| + |b|)^2 and (b, b) left
// in aux[2..4] of the operator's scalar block (ticket 5).
template <int MASKC>
__global__ void __launch_bounds__(TPB) k_residual_any(Geom g, const double* __restrict__ val,
                                                      const double* __restrict__ b, const double* __restrict__ x,
                                                      double* __restrict__ r, double* partials, PcgScalars* sc) {
  double v[3] = {0.0, 0.0, 0.0};
  const int n = (int)g.n;
  for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < n; row += gridDim.x * blockDim.x) {
    const int col = row / g.nz;
    const int k = row - col * g.nz;
    double asum = 0.0;
    const double bi = b[row];
    const double ri = row_residual_dot2<MASKC>(g, val, x, bi, row, col, k, asum);
    r[row] = ri;
    v[0] = fma(ri, ri, v[0]);
    const double f = asum + fabs(bi);
    v[1] = fma(f, f, v[1]);
    v[2] = fma(bi, bi, v[2]);
  }
  if (grid_sum<3>(v, partials, &sc->count[5]) && threadIdx.x == 0) {
    sc->aux[2] = v[0];
    sc->aux[3] = v[1];
    sc->aux[4] = v[2];
  }
}
}  // namespace

int residual(pm_operator* op, int which, const double* b, const double* x, double* r, double* norms,
             cudaStream_t s) {
  const int vs = which_valset(which);
  if (vs < 0) return set_error(PM_EINVAL, "unknown operator");
  int st = ensure_ctx(op);
  if (st) return st;
  SolveCtx* c = op->ctx;
  Geom g = geom_of(op);
  const int G = grid_for(op->n, TPB, op->num_sms);
  switch (which_mask(which)) {
    case 0: k_residual_any<0><<<G, TPB, 0, s>>>(g, op->d_val[vs], b, x, r, c->partials, c->sc); break;
    case 1: k_residual_any<1><<<G, TPB, 0, s>>>(g, op->d_val[vs], b, x, r, c->partials, c->sc); break;
    case 2: k_residual_any<2><<<G, TPB, 0, s>>>(g, op->d_val[vs], b, x, r, c->partials, c->sc); break;
    default: k_residual_any<-1><<<G, TPB, 0, s>>>(g, op->d_val[vs], b, x, r, c->partials, c->sc); break;
  }
  count_launch();
  if ((st = cuda_check(cudaGetLastError(), "k_residual_any"))) return st;
  if (!norms) return PM_OK;
  if ((st = read_scalars(c, s))) return st;
  norms[0] = c->sc_host->aux[2];
  norms[1] = c->sc_host->aux[3];
  norms[2] = c->sc_host->aux[4];
  return PM_OK;
}

int pcg_solve(pm_operator* op, int which, const double* b, double* x, const pm_solve_opts* o,
              pm_solve_stats* st, cudaStream_t s) {
  if (!which_symmetric(which)) return set_error(PM_EINVAL, "pcg needs a symmetric operator");
  if (o->prec < 0 || o->prec > PM_PREC_LINE) return set_error(PM_EINVAL, "unknown preconditioner");
  if (!(o->rtol > 0.0) || o->max_iter < 0) return set_error(PM_EINVAL, "rtol must be > 0, max_iter >= 0");
  if (o->precision < PM_FP64 || o->precision > PM_BF16_REFINE) return set_error(PM_EINVAL, "unknown precision");
  if (o->kernel < PM_KERNEL_AUTO || o->kernel > PM_KERNEL_RESIDENT) return set_error(PM_EINVAL, "unknown kernel choice");
  NvtxRange range(std::string("pcg ") + which_name(which) + " " + prec_name(o->prec) + " " + precision_name(o->precision));
  int r = ensure_ctx(op);
  if (r) return r;
  // PM_KERNEL_RESIDENT (and its limit) is of FP64 solves; a mixed-precision one runs as AUTO then
  const bool mixed = o->precision != PM_FP64, asked = !mixed && o->kernel == PM_KERNEL_RESIDENT;
  if (asked && op->n > RESIDENT_MAX_ROWS)
    return set_error(PM_EINVAL, "PM_KERNEL_RESIDENT: at most " + std::to_string(RESIDENT_MAX_ROWS) + " rows");
  if (asked || (o->kernel != PM_KERNEL_STREAM && resident_auto(op, o->prec, mixed)))
    return resident_run(op, which, b, x, o, st, s);
  if (o->precision == PM_FP32_REFINE) {
    switch (which_mask(which)) {
      case 0: return mixed_run<0, float>(op, which, b, x, o, st, s);
      case 1: return mixed_run<1, float>(op, which, b, x, o, st, s);
      case 2: return mixed_run<2, float>(op, which, b, x, o, st, s);
      default: return mixed_run<-1, float>(op, which, b, x, o, st, s);
    }
  }
  if (o->precision == PM_BF16_REFINE) {
    switch (which_mask(which)) {
      case 0: return mixed_run<0, __nv_bfloat16>(op, which, b, x, o, st, s);
      case 1: return mixed_run<1, __nv_bfloat16>(op, which, b, x, o, st, s);
      case 2: return mixed_run<2, __nv_bfloat16>(op, which, b, x, o, st, s);
      default: return mixed_run<-1, __nv_bfloat16>(op, which, b, x, o, st, s);
    }
  }
  switch (which_mask(which)) {
    case 0: return pcg_run<0>(op, which, b, x, o, st, s);
    case 1: return pcg_run<1>(op, which, b, x, o, st, s);
    case 2: return pcg_run<2>(op, which, b, x, o, st, s);
    default: return pcg_run<-1>(op, which, b, x, o, st, s);
  }
}

// Everything a batched solve reads from one operator: Jacobi diagonals, line or IC0 factors, and
// for FP32 the difference-form values and FP32 factors.
int prepare_for_batch(pm_operator* op, int which, int prec, int precision, cudaStream_t s) {
  int st = ensure_ctx(op);
  if (st) return st;
  if ((st = ensure_prec(op, which, prec, s))) return st;
  if (precision != PM_FP64 && (st = ensure_mixed(op, which, precision, prec, s))) return st;
  return PM_OK;
}

}  // namespace pm

extern "C" int pm_kernel_timing(int32_t enable) {
  using namespace pm;
  if (!g_kt.pending.empty()) {
    cudaDeviceSynchronize();
    kt_collect();
  }
  g_kt.on = enable != 0;
  for (int k = 0; k < PM_KT_COUNT; ++k) {
    g_kt.total_ms[k] = 0.0;
    g_kt.launches[k] = 0;
  }
  return PM_OK;
}

extern "C" int pm_kernel_timing_get(int32_t kind, double* total_ms, int64_t* launches) {
  using namespace pm;
  if (kind < 0 || kind >= PM_KT_COUNT) return set_error(PM_EINVAL, "unknown kernel class");
  if (!g_kt.pending.empty()) {
    cudaDeviceSynchronize();
    kt_collect();
  }
  if (total_ms) *total_ms = g_kt.total_ms[kind];
  if (launches) *launches = g_kt.launches[kind];
  return PM_OK;
}

namespace pm {

void destroy_ctx(pm_operator* op) {
  SolveCtx* c = op->ctx;
  if (!c) return;
  cudaFree(c->r);
  cudaFree(c->p);
  cudaFree(c->w);
  cudaFree(c->z);
  cudaFree(c->bw);
  cudaFree(c->partials);
  cudaFree(c->sc);
  cudaFreeHost(c->sc_host);
  cudaFree(c->r32);
  cudaFree(c->p32);
  cudaFree(c->w32);
  cudaFree(c->z32);
  cudaFree(c->d32);
  cudaFree(c->sc_in);
  if (c->sc_in_host) cudaFreeHost(c->sc_in_host);
  cudaFree(c->res_ctl);
  if (c->res_out) cudaFreeHost(c->res_out);
  delete c;
  op->ctx = nullptr;
}

}  // namespace pm
