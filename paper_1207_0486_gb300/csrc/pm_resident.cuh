// Resident PCG: one launch runs a whole solve (Section 5 remark), its blocks in step.
//
// A PCG iteration is a chain of short dependent phases: with IC0, 18 of them. As separate kernels
// each costs a launch on the host and a drain and ramp on the GPU, 8 to 12 us measured per phase
// whatever its size, far more than the work of a phase below a few hundred thousand rows. Here a
// team of blocks keeps the GPU (one block per SM) from the first residual to the last and separates
// the phases by its own barrier; convergence is tested by every block from the same sums, so no
// iteration is issued in vain and the host waits once.
//
// Two teams run the same code:
//   - grid: one block per SM (cooperative launch), a counter in L2 as the barrier (bounded wait): 2400
//     cycles, 3000 with stores to publish;
//   - cluster: 16 blocks of one thread-block cluster, the hardware cluster barrier (550 to 980 cycles, 2000
//     with global stores to publish), block sums exchanged through distributed shared memory: for systems so
//     small that the grid barrier would cost more than the work the other SMs take over. The smallest have a
//     team of one block, whose barrier is the block's own: no fence, and L1 keeps what it holds between phases.
//
// Rows: the line preconditioner works on whole columns, dealt evenly and contiguously to the blocks; without it
// a block takes an even share of the rows, however few columns they make up (16 columns of 20,000 levels, Jacobi:
// 32 us per iteration, 172 by whole columns, 71 as a stream); an IC0 colour phase deals the colour's rows (in class order, as the
// factor is stored) evenly to the blocks. Vectors that other blocks read (p, x, the IC0 work vector)
// go through L2: a barrier's release / acquire pair orders them, and the acquire drops stale L1 lines,
// so plain loads may use L1 within a phase.
//
// One iteration, phases | team barriers:
//   w = A p, (p, w)                                                              | sum
//   r -= alpha w, (r, r); Jacobi / line: z and its dots; IC0: y of colour 0        | sum
//   IC0: y of colours 1..7 (forward), z of colour 7 with its y, (y, y) = (r, z)        | 6, then sum
//   x += alpha p, p = z - c + beta p; IC0: with z of colours 6..0 (backward)            | 1 (IC0: 7)
// (r, z) = (y, y) because z = L^-T y and y = L^-1 r; it is known before the backward sweep, so that
// sweep can form p at once. The pressure's projection needs m'z first: its IC0 sums and p follow the
// sweeps as passes of their own.
//
// What bounds it: barriers and load latency below about 0.3M rows (IC0 49 us per iteration at 0.12M rows; the stream of
// kernels takes 132 now, and took 218 before its sweeps were in colour order), the FP64 pipe (64 cycles per warp
// instruction and sub-core) above.
//
// A grid team holds every SM to the end of its solve (512 threads of 128 registers fill the register file): solves on
// other streams queue behind it, where the stream's kernels interleave. Several solves at once, one operator
// and host thread each, us per system and iteration, 1 / 2 / 4 / 8 threads: FP64 line, 0.12M rows, resident 24 whatever
// the number, stream 53 / 30 / 19 / 13; FP32 line 19 and 37 / 19 / 11 / 7; FP64 IC0 40 and 76 / 43 / 29 / 21, 2.0M rows 272 and
// 284 / 212 / 188 / 194. Solves by one cluster or one block run side by side (2,048 rows, IC0: 7.0 / 3.6 / 1.8 / 1.2).
#pragma once

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "pm_internal.cuh"

namespace pm {
namespace resident {

// Threads per block, one block per SM: 128 registers a thread hold the 15 values and 15 gathered
// entries of a row, or the factor row fetched ahead of a barrier, without spills.
constexpr int NT = 512;
constexpr int CLUSTER = 16;

struct Ctl {
  uint32_t arrive;   // barrier arrivals of this launch (zeroed before it)
  int32_t err;       // set by a wait that ran out
};

struct Result {
  int32_t iters, restarts, first_pass, status, zero_rhs, pad;
  double rel_true, rel_rec, floor;
};
// Rank 0 writes the result. A block whose wait ran out writes the other field: rank 0 may have passed the last
// barrier all the same and report its result after that, but the block that left did not do its rows.
struct Out {
  Result res;
  int32_t timeout, pad;
};

struct Args {
  Geom g;
  const void* val;        // operator values: FP64, or the FP32 / BF16 difference form
  const double* val64;
  const uint16_t* mask;   // bit s: slot s counts; bit 15: identity row
  const double* b;
  double* x;
  double* bw;             // projected right-hand side (pressure)
  void *r, *p, *w, *z;    // Krylov vectors (T)
  float* d;               // FP32 correction since the last residual (mixed precision)
  const void* dinv;       // T inverse diagonal; null: plain CG
  const double* m;        // M 1
  const float2* m2;       // M 1 as two floats (mixed precision)
  const void* ic0;        // IC0 factor, colour-ordered rows, 1 / L_ii in the diagonal slot
  const void* line;       // line factors, level-major
  const int32_t* cnbr;    // columns in class order
  const int32_t* ccls;    // [7][ncols]: their neighbours' indices within their classes
  const int32_t* colpos;  // [2][ncols]: first colour-ordered position of a column's even / odd levels
  int32_t cls_off[4], cls_cnt[4];
  int32_t cbase[8];
  FastDiv nlev[2];        // levels of even / odd parity
  double rtol, inner_rtol, one_m;
  int32_t max_iter, max_restarts, x0_is_guess, proj, z_in_smem;
  Ctl* ctl;
  double* part;           // 2 x 4 x blocks block sums (grid team)
  Out* out;               // pinned host memory
};

__device__ __forceinline__ void red_release(uint32_t* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Polls of a grid barrier before it gives up: each takes about a microsecond.
constexpr uint32_t WAIT_LIMIT = 1u << 22;

// Block-level part of a team sum: FP64 adds run at 1/64 of the FP32 rate on this GPU, so the values
// go through shared memory and full warps add them (NT / 32 + 12 warp-wide adds per value), where
// shuffles in every warp would take 5 NT / 32.
struct Scratch {
  double v[4][NT];
  double q[4][128];
  double res[4];
  double sc[3];                // block_scalars
  double xch[2][4][CLUSTER];   // cluster team: the blocks' sums
  int ok;
  int first[8], past[8];       // this block's share of each colour's rows
};

template <bool CL>
struct Team {
  Ctl* ctl;
  double* part;
  Scratch* s;
  int G, rank;
  uint32_t target;
  int buf;

  __device__ Team(const Args& a, Scratch* s_)
      : ctl(a.ctl), part(a.part), s(s_), G(gridDim.x), rank(blockIdx.x), target(0), buf(0) {}

  // This block's stores so far are published; wait() returns when every block has arrived.
  __device__ __forceinline__ void arrive() {
    if (CL) {
      if (G > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    } else {
      __syncthreads();
      if (threadIdx.x == 0) red_release(&ctl->arrive);
      target += (uint32_t)G;
    }
  }
  __device__ __forceinline__ bool wait() {
    if (CL) {
      if (G > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      else __syncthreads();
      return true;
    }
    if (threadIdx.x == 0) {
      int ok = 1;
      uint32_t polls = 0;
      while ((int32_t)(ld_acquire(&ctl->arrive) - target) < 0) {
        ++polls;
        if (polls > WAIT_LIMIT || ((polls & 1023u) == 0 && *(volatile int32_t*)&ctl->err)) {
          atomicExch(&ctl->err, 1);
          ok = 0;
          break;
        }
      }
      s->ok = ok;
    }
    __syncthreads();
    return s->ok != 0;
  }
  __device__ __forceinline__ bool barrier() {
    arrive();
    return wait();
  }

  // Team totals of NV values in every thread, added in a fixed order. A barrier as well.
  template <int NV>
  __device__ __forceinline__ bool sum(double (&v)[NV]) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const bool alone = CL && G == 1;
    static_assert(NT == 512 && NV <= 4, "four warps per value");
#pragma unroll
    for (int i = 0; i < NV; ++i) s->v[i][tid] = v[i];
    __syncthreads();
    if (wid < 4 * NV) {
      const double* c = s->v[wid >> 2] + (wid & 3) * 128 + lane;
      s->q[wid >> 2][(wid & 3) * 32 + lane] = (c[0] + c[32]) + (c[64] + c[96]);
    }
    __syncthreads();
    if (wid < NV) {
      const double* c = s->q[wid] + lane;
      double t = warp_sum((c[0] + c[32]) + (c[64] + c[96]));
      if (alone) {
        if (lane == 0) s->res[wid] = t;
      } else if (CL) {
        t = __shfl_sync(0xffffffffu, t, 0);
        if (lane < G) {
          const uint32_t local = (uint32_t)__cvta_generic_to_shared(&s->xch[buf][wid][rank]);
          uint32_t remote;
          asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(lane));
          asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(t) : "memory");
        }
        __syncwarp();
      } else if (lane == 0) {
        part[(buf * 4 + wid) * G + rank] = t;
      }
    }
    arrive();
    if (!wait()) return false;
    if (wid < NV && !alone) {
      double t = 0.0;
      if (CL) {
        t = lane < G ? s->xch[buf][wid][lane] : 0.0;
      } else {
        for (int j = lane; j < G; j += 32) t += __ldcg(part + (buf * 4 + wid) * G + j);
      }
      t = warp_sum(t);
      if (lane == 0) s->res[wid] = t;
    }
    if (!alone) __syncthreads();
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = s->res[i];
    buf ^= 1;
    return true;
  }
};

// Scalars formed from a sum, by one thread for its block. A division takes some ten instructions of the FP64 pipe, 64
// cycles each per warp and sub-core: repeated by 16 warps, the three of an iteration held the pipe for about 7,500
// cycles. By one thread: 512 rows, Jacobi pressure, 3.06 -> 2.38 ms (one block of 8 warps had taken 2.82); 0.06M 9 to 14 %
// less by the diagonal, 6 to 10 % by columns, 4 % IC0; nothing from 2M rows on.
template <int NV, typename F>
__device__ __forceinline__ void block_scalars(Scratch* s, double (&out)[NV], F f) {
  static_assert(NV <= 3, "Scratch::sc");
  if (threadIdx.x == 0) f(s->sc);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < NV; ++i) out[i] = s->sc[i];
}

// A block's share: whole columns [c0, c1) with the line preconditioner, else rows. Only one of the pairs is kept
// in registers (with both, line solves of 1M to 3M rows were 3 to 7 % slower).
template <int PREC>
struct Share {
  int first, past;
  __device__ __forceinline__ Share(const Geom& g, int rank, int G) {
    if (PREC == PM_PREC_LINE) {
      first = (int)((int64_t)g.ncols * rank / G);
      past = (int)((int64_t)g.ncols * (rank + 1) / G);
    } else {   // in runs of 32 rows, so that a warp's accesses are aligned
      const int64_t runs = (g.n + 31) / 32;
      first = (int)min(g.n, 32 * (runs * rank / G));
      past = (int)min(g.n, 32 * (runs * (rank + 1) / G));
    }
  }
  __device__ __forceinline__ int row0(const Geom& g) const { return PREC == PM_PREC_LINE ? first * g.nz : first; }
  __device__ __forceinline__ int row1(const Geom& g) const { return PREC == PM_PREC_LINE ? past * g.nz : past; }
  __device__ __forceinline__ int col0() const { return first; }   // line preconditioner
  __device__ __forceinline__ int col1() const { return past; }
};

// Neighbour q, by its index within its class, of the column at place i in class order (-1: none).
__device__ __forceinline__ int ccls_of(const Args& a, int i, int q) {
  const int nb = __ldg(a.ccls + q * a.g.ncols + i);
#ifdef PM_CHECKED
  if (nb < -1 || nb >= a.g.ncols) {
    record_bad_index(SITE_NBR, nb, a.g.ncols);
    return -1;
  }
#endif
  return nb;
}

__device__ __forceinline__ double ldval(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldval(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ldval(const __nv_bfloat16* p) {
  return __bfloat162float(__ushort_as_bfloat16(__ldg(reinterpret_cast<const unsigned short*>(p))));
}

// Row of A times x. The mask's clear bits are slots that do not count: absent neighbours (their
// values are 0) and, for a velocity, Dirichlet ones. FP32: the difference form (row sum in the
// diagonal slot, eliminated slots' values taken off it).
template <typename T, typename TV>
__device__ __forceinline__ T row_apply(const Geom& g, const TV* __restrict__ val, const T* x,
                                       const uint16_t* __restrict__ mask, int row, int col, int k) {
  const int nz = g.nz, npad = (int)g.npad;
  const uint32_t km = __ldg(mask + row);
  if (km & 0x8000u) return x[row];
  int nb[NNBR];
  nb[0] = col;
#pragma unroll
  for (int q = 1; q < NNBR; ++q) nb[q] = nbr_of(g, col, q);
  T a[NSLOT], xv[NSLOT];
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) a[s] = ldval(val + s * npad + row);
#pragma unroll
  for (int s = 0; s < NSLOT; ++s) xv[s] = x[((km >> s) & 1u) ? nb[slot_q(s)] * nz + k + slot_dk(s) : row];
  T sum = 0;
  if constexpr (std::is_same<T, double>::value) {
#pragma unroll
    for (int s = 0; s < NSLOT; ++s) sum = fma(((km >> s) & 1u) ? a[s] : 0.0, xv[s], sum);
    return sum;
  } else {
    const float xi = xv[DIAG_SLOT];
    float drop = 0.f;
#pragma unroll
    for (int s = 0; s < NSLOT; ++s) {
      if (s == DIAG_SLOT) continue;
      const bool keep = (km >> s) & 1u;
      drop += keep ? 0.f : a[s];
      sum = fmaf(keep ? a[s] : 0.f, xv[s] - xi, sum);
    }
    return fmaf(a[DIAG_SLOT] - drop, xi, sum);
  }
}

// b_i - (A x)_i by Dot2 (row_residual_dot2), slots by the mask.
__device__ __forceinline__ double row_residual(const Geom& g, const double* __restrict__ val, const double* x,
                                               const uint16_t* __restrict__ mask, double bi, int row, int col, int k,
                                               double& abs_sum) {
  const int nz = g.nz, npad = (int)g.npad;
  const uint32_t km = __ldg(mask + row);
  if (km & 0x8000u) {
    const double xi = x[row];
    abs_sum = fabs(xi);
    return __dsub_rn(bi, xi);
  }
  int nb[NNBR];
  nb[0] = col;
#pragma unroll
  for (int q = 1; q < NNBR; ++q) nb[q] = nbr_of(g, col, q);
  double s = bi, c = 0.0, asum = 0.0;
#pragma unroll
  for (int sl = 0; sl < NSLOT; ++sl) {
    const bool ok = (km >> sl) & 1u;
    const double av = ok ? __ldg(val + sl * npad + row) : 0.0;
    const double xv = x[ok ? nb[slot_q(sl)] * nz + k + slot_dk(sl) : row];
    double pe, se;
    const double pr = two_product(av, xv, pe);
    s = two_sum(s, -pr, se);
    c = __dadd_rn(c, __dsub_rn(se, pe));
    asum += fabs(pr);
  }
  abs_sum = asum;
  return __dadd_rn(s, c);
}

// ---- IC0 ---------------------------------------------------------------------------------------

// Sums of one sweep pass: (r, r), (y, y) = (r, z), m'z, 1'r.
template <typename T>
struct Dots {
  AccFor<T> rr, rz, mz, sr;
};

__device__ __forceinline__ void add_m(Acc64& acc, const Args& a, int row, double z) { acc.add_prod(__ldg(a.m + row), z); }
__device__ __forceinline__ void add_m(DF& acc, const Args& a, int row, float z) {
  const float2 m = __ldg(a.m2 + row);
  acc.add_prod(m.x, z);
  acc.add_prod(m.y, z);
}

// The vector that alpha p is added to: the FP64 iterate, or the FP32 correction of a mixed-precision solve.
template <typename T>
__device__ __forceinline__ T* iterate(const Args& a) {
  if constexpr (std::is_same<T, double>::value) return a.x;
  else return a.d;
}
// x += alpha p, p = z + beta p on one row.
template <typename T>
__device__ __forceinline__ void move_row(const Args& a, int row, T alpha, T beta, T z) {
  T* p = static_cast<T*>(a.p);
  T* x = iterate<T>(a);
  const T pv = p[row];
  x[row] = fma(alpha, pv, x[row]);
  p[row] = fma(beta, pv, z);
}

// The sweeps' work vector (y, then z) is in colour order, as the factor's rows are: position cbase[colour] +
// (index of the column in its parity class) * levels + level / 2. A colour's rows are every other level of
// their columns; in colour order a warp's reads of each neighbour are runs, in the natural order every other
// entry of each sector.
__device__ __forceinline__ int colour_pos(const Args& a, int col, int k) {
  return __ldg(a.colpos + (k & 1) * a.g.ncols + col) + (k >> 1);
}

// Constant operands of one row of a colour phase: its places, neighbours and factor row.
template <typename T, int C, bool FWD>
struct ColourRow {
  static constexpr int kpar = C >> 2, cls = C & 3;
  int row, pos, kk;   // in natural order, in colour order; level / 2
  int nb[NNBR];
  T f[NSLOT];
  // The slots read: lower colours forward, higher ones backward.
  static __host__ __device__ constexpr bool uses(int s) {
    return s != DIAG_SLOT && (FWD ? (C ^ slot_flip(s)) < C : (C ^ slot_flip(s)) > C);
  }
  // t: place within the colour. Reads stay inside the arrays for t = 0 of an empty colour.
  __device__ __forceinline__ void load(const Args& a, int t) {
    const T* __restrict__ F = static_cast<const T*>(a.ic0);
    const int i = fdiv(a.nlev[kpar], t), n = (int)a.g.n;
    const int at = min(a.cls_off[cls] + i, a.g.ncols - 1);
    pos = min(a.cbase[C] + t, n - 1);
    kk = t - i * a.nlev[kpar].d;
    nb[0] = i;
#pragma unroll
    for (int q = 1; q < NNBR; ++q) nb[q] = ccls_of(a, at, q);
#pragma unroll
    for (int s = 0; s < NSLOT; ++s)
      if (uses(s) || s == DIAG_SLOT) f[s] = __ldg(F + (s * n + pos));
    row = __ldg(a.cnbr + at) * a.g.nz + 2 * kk + kpar;
  }
  // (v - sum f_s y_s) / L_ii
  __device__ __forceinline__ T value(const Args& a, T v, const T* y) const {
    T yv[NSLOT];
#pragma unroll
    for (int s = 0; s < NSLOT; ++s) {
      if (!uses(s)) continue;
      const int cj = C ^ slot_flip(s), dk = slot_dk(s), nl = a.nlev[cj >> 2].d;
      const int lv = kk + (dk == 0 ? 0 : dk > 0 ? kpar : kpar - 1);   // the neighbour's level / 2
      const bool ok = nb[slot_q(s)] >= 0 && lv >= 0 && lv < nl;
      yv[s] = ok ? y[a.cbase[cj] + nb[slot_q(s)] * nl + lv] : (T)0;
    }
#pragma unroll
    for (int s = 0; s < NSLOT; ++s)
      if (uses(s)) v = fma(-f[s], yv[s], v);
    return v * f[DIAG_SLOT];
  }
};

// One colour phase over this block's share of the colour's rows. Forward (FWD): y_i = (r_i - sum L_ij y_j) / L_ii
// over lower colours; colour 7 goes straight on to its backward value z_i = y_i / L_ii (no higher
// colour exists). Backward: z_i = (y_i - sum L_ji z_j) / L_ii over higher colours, in place, and
// (FUSEP) x_i += alpha p_i, p_i = z_i + beta p_i. The constant operands of a thread's first row are fetched before
// the barrier that its neighbours' values wait for (SYNC). acc takes (y, y) on forward phases.
template <typename T, int C, bool FWD, bool FUSEP, bool SYNC, bool CL, typename Acc>
__device__ __forceinline__ bool colour_phase(const Args& a, Team<CL>& team, T alpha, T beta, Acc& acc) {
  using Row = ColourRow<T, C, FWD>;
  const T* r = static_cast<const T*>(a.r);
  T* y = static_cast<T*>(a.z);
  const int t1 = team.s->past[C];
  int t = team.s->first[C] + (int)threadIdx.x;
  Row w;
  if (SYNC) {
    // without a condition (a clamped place instead): loaded under one, the row went to local memory
    w.load(a, max(0, min(t, t1 - 1)));
    if (!team.wait()) return false;
  }
#pragma unroll 1
  for (bool first = SYNC; t < t1; t += NT, first = false) {
    if (!first) w.load(a, t);
    T v = w.value(a, FWD ? r[w.row] : y[w.pos], y);
    if (FWD) {
      acc.add_prod(v, v);
      if (C == 7) v *= w.f[DIAG_SLOT];
    }
    y[w.pos] = v;
    if (FUSEP) move_row(a, w.row, alpha, beta, v);
  }
  return true;
}

// y of colour 0 for one row in natural order: r / L_ii (no lower colour). Other rows: nothing.
template <typename T, typename Acc>
__device__ __forceinline__ void colour0_y(const Args& a, int col, int k, T ri, Acc& acc) {
  if (k & 1) return;
  const int pos = colour_pos(a, col, k);
  if (pos >= a.cbase[1]) return;
  const T v = ri * __ldg(static_cast<const T*>(a.ic0) + DIAG_SLOT * (int)a.g.n + pos);
  static_cast<T*>(a.z)[pos] = v;
  acc.add_prod(v, v);
}

// Forward sweep after colour 0; (y, y) = (r, z) is summed over the team (a barrier).
template <typename T, bool CL, typename Acc>
__device__ __forceinline__ bool ic0_forward(const Args& a, Team<CL>& team, Acc& acc, double& yy) {
  if (!colour_phase<T, 1, true, false, false>(a, team, (T)0, (T)0, acc)) return false;
#define PM_FWD(C)                                                                          \
  team.arrive();                                                                           \
  if (!colour_phase<T, C, true, false, true>(a, team, (T)0, (T)0, acc)) return false;
  PM_FWD(2) PM_FWD(3) PM_FWD(4) PM_FWD(5) PM_FWD(6) PM_FWD(7)
#undef PM_FWD
  double v[1] = {acc.value()};
  if (!team.template sum<1>(v)) return false;
  yy = v[0];
  return true;
}

// Backward sweep from colour 6 on, with x and p when FUSEP, and the barrier after it.
template <typename T, bool FUSEP, bool CL>
__device__ __forceinline__ bool ic0_backward(const Args& a, Team<CL>& team, T alpha, T beta) {
  Acc64 unused;
  if (FUSEP) {   // rows of colour 7 have their z already: x and p where this block formed it
    for (int t = team.s->first[7] + (int)threadIdx.x; t < team.s->past[7]; t += NT) {
      const int i = fdiv(a.nlev[1], t);
      const int row = __ldg(a.cnbr + a.cls_off[3] + i) * a.g.nz + 2 * (t - i * a.nlev[1].d) + 1;
      move_row(a, row, alpha, beta, static_cast<const T*>(a.z)[a.cbase[7] + t]);
    }
  }
  if (!colour_phase<T, 6, false, FUSEP, false>(a, team, alpha, beta, unused)) return false;
#define PM_BWD(C)                                                                          \
  team.arrive();                                                                           \
  if (!colour_phase<T, C, false, FUSEP, true>(a, team, alpha, beta, unused)) return false;
  PM_BWD(5) PM_BWD(4) PM_BWD(3) PM_BWD(2) PM_BWD(1) PM_BWD(0)
#undef PM_BWD
  return team.barrier();
}

// ---- the update and the column-local preconditioners ------------------------------------------

// r -= alpha w (UPDATE), then z by the preconditioner, on this block's rows. LINE: zt is the
// block's tile of columns, ld apart (shared memory, or its part of the z vector).
template <typename T, int PREC, bool UPDATE>
__device__ __forceinline__ void update_rows(const Args& a, const Share<PREC>& sh, T alpha, T* zt, int ld, Dots<T>& dots) {
  const Geom& g = a.g;
  const int nz = g.nz, row1 = sh.row1(a.g);
  T* r = static_cast<T*>(a.r);
  const T* w = static_cast<const T*>(a.w);
  const T* dinv = static_cast<const T*>(a.dinv);
  constexpr int U = 4;   // rows whose loads are in flight together
  for (int i0 = sh.row0(a.g) + (int)threadIdx.x; i0 < row1; i0 += U * NT) {
    T rv[U], wv[U], dv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = min(i0 + u * NT, row1 - 1);
      rv[u] = r[row];
      if (UPDATE) wv[u] = w[row];
      if (PREC == PM_PREC_JACOBI) dv[u] = dinv ? __ldg(dinv + row) : (T)1;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = i0 + u * NT;
      if (row >= row1) break;
      T ri = rv[u];
      if (UPDATE) {
        ri = fma(-alpha, wv[u], ri);
        r[row] = ri;
      }
      dots.rr.add_prod(ri, ri);
      if (a.proj) dots.sr.add(ri);
      if (PREC == PM_PREC_JACOBI) {
        const T zi = dv[u] * ri;
        dots.rz.add_prod(ri, zi);
        if (a.proj) add_m(dots.mz, a, row, zi);
      } else {
        const int col = fdiv(g.nzd, row), k = row - col * nz;
        if (PREC == PM_PREC_LINE) zt[(col - sh.col0()) * ld + k] = ri;
        else colour0_y(a, col, k, ri, dots.rz);
      }
    }
  }
  if (PREC != PM_PREC_LINE) return;
  __syncthreads();
  // Thomas solve of each column, one thread per column; (r, z) = sum_k t_k y_k (symmetric blocks)
  const T* F = static_cast<const T*>(a.line);
  const int nc = g.ncols, n = (int)g.n;
  for (int col = sh.col0() + (int)threadIdx.x; col < sh.col1(); col += NT) {
    T* cs = zt + (col - sh.col0()) * ld;
    T y = 0;
#pragma unroll 8
    for (int k = 0; k < nz; ++k) {
      const int li = k * nc + col;
      const T tk = fma(-__ldg(F + li), y, cs[k]);
      y = tk * __ldg(F + n + li);
      dots.rz.add_prod(tk, y);
      cs[k] = y;
    }
    T zn = y;
#pragma unroll 8
    for (int k = nz - 2; k >= 0; --k) {
      zn = fma(-__ldg(F + 2 * n + k * nc + col), zn, cs[k]);
      cs[k] = zn;
    }
  }
  __syncthreads();
  if (!a.proj) return;
  for (int row = sh.row0(a.g) + (int)threadIdx.x; row < row1; row += NT) {
    const int col = fdiv(g.nzd, row);
    add_m(dots.mz, a, row, zt[(col - sh.col0()) * ld + row - col * nz]);
  }
}

// x += alpha p and p = (z - c) + beta p on the block's rows. x moves here, a pass after r, because p is read
// here anyway. FIRST: p = z - c.
// LAST: x alone, when no further direction is needed.
template <typename T, int PREC, bool FIRST, bool LAST>
__device__ __forceinline__ void direction(const Args& a, const Share<PREC>& sh, T alpha, T beta, T c, const T* zt, int ld) {
  const Geom& g = a.g;
  const int nz = g.nz, row1 = sh.row1(a.g);
  T* p = static_cast<T*>(a.p);
  T* x = iterate<T>(a);
  const T* r = static_cast<const T*>(a.r);
  const T* zv = static_cast<const T*>(a.z);
  const T* dinv = static_cast<const T*>(a.dinv);
  constexpr int U = 4;
  for (int i0 = sh.row0(a.g) + (int)threadIdx.x; i0 < row1; i0 += U * NT) {
    T z[U], pv[U], xv[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = min(i0 + u * NT, row1 - 1);
      if (!LAST) {
        if (PREC == PM_PREC_JACOBI) {
          z[u] = (dinv ? __ldg(dinv + row) : (T)1) * r[row];
        } else if (PREC == PM_PREC_LINE) {
          const int col = fdiv(g.nzd, row);
          z[u] = zt[(col - sh.col0()) * ld + row - col * nz];
        } else {
          const int col = fdiv(g.nzd, row);
          z[u] = zv[colour_pos(a, col, row - col * nz)];
        }
      }
      if (!FIRST) {
        pv[u] = p[row];
        xv[u] = x[row];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = i0 + u * NT;
      if (row >= row1) break;
      if (!FIRST) x[row] = fma(alpha, pv[u], xv[u]);
      if (!LAST) p[row] = FIRST ? z[u] - c : fma(beta, pv[u], z[u] - c);
    }
  }
}

// State of the PCG recurrence, the same in every thread of the team.
struct Cg {
  double rho = 0.0, rr = 0.0;
  int iter = 0, status = PM_OK;
};

// r -= alpha w (not FIRST), z = P^{-1} r, (r, r), then x += alpha p, rho, beta and p, and the barrier
// after which every block may read p. FIRST: from r alone, beta = 0. STOP is asked once cg.rr = (r, r) is
// known: true ends the step with x moved (the recursion has met its target). cg.status is PM_BREAKDOWN
// when rho is not positive. Returns false when a wait ran out.
template <typename T, int PREC, bool FIRST, bool CL, typename Stop>
__device__ __forceinline__ bool advance(const Args& a, Team<CL>& team, const Share<PREC>& sh, T* zt, int ld,
                                        double alpha, Cg& cg, bool& stopped, Stop stop) {
  Dots<T> dots;
  update_rows<T, PREC, !FIRST>(a, sh, (T)alpha, zt, ld, dots);
  double c = 0.0, rho = 0.0, beta64 = 0.0;
  const auto scalars = [&](double rz, double mz, double sr) {
    double u[3];
    block_scalars(team.s, u, [&](double* o) {
      o[0] = a.proj ? mz / a.one_m : 0.0;
      o[1] = a.proj ? rz - o[0] * sr : rz;
      o[2] = FIRST ? 0.0 : o[1] / cg.rho;
    });
    c = u[0];
    rho = u[1];
    beta64 = u[2];
  };
  if (PREC == PM_PREC_IC0) {
    double v[1] = {dots.rr.value()};
    if (!team.template sum<1>(v)) return false;
    cg.rr = v[0];
    stopped = stop();
    if (!stopped && !ic0_forward<T>(a, team, dots.rz, rho)) return false;
    if (!stopped && !a.proj) scalars(rho, 0.0, 0.0);
    if (!stopped && a.proj) {   // the projection needs the whole z before p
      if (!ic0_backward<T, false>(a, team, (T)0, (T)0)) return false;
      const T* r = static_cast<const T*>(a.r);
      const T* z = static_cast<const T*>(a.z);
      AccFor<T> rz;
      for (int row = sh.row0(a.g) + (int)threadIdx.x; row < sh.row1(a.g); row += NT) {
        const int col = fdiv(a.g.nzd, row);
        const T zi = z[colour_pos(a, col, row - col * a.g.nz)];
        rz.add_prod(r[row], zi);
        add_m(dots.mz, a, row, zi);
      }
      double u[3] = {rz.value(), dots.mz.value(), dots.sr.value()};
      if (!team.template sum<3>(u)) return false;
      scalars(u[0], u[1], u[2]);
    }
  } else if (a.proj) {
    double v[4] = {dots.rr.value(), dots.rz.value(), dots.mz.value(), dots.sr.value()};
    if (!team.template sum<4>(v)) return false;
    cg.rr = v[0];
    scalars(v[1], v[2], v[3]);
    stopped = stop();
  } else {
    double v[2] = {dots.rr.value(), dots.rz.value()};
    if (!team.template sum<2>(v)) return false;
    cg.rr = v[0];
    scalars(v[1], 0.0, 0.0);
    stopped = stop();
  }
  const bool broken = !stopped && (!(rho > 0.0) || !isfinite(rho));
  if (broken) cg.status = PM_BREAKDOWN;
  if (stopped || broken) {
    direction<T, PREC, FIRST, true>(a, sh, (T)alpha, (T)0, (T)0, zt, ld);
    return team.barrier();
  }
  const T beta = (T)beta64;
  cg.rho = rho;
  if (PREC == PM_PREC_IC0 && !a.proj) {
    if (!FIRST) return ic0_backward<T, true>(a, team, (T)alpha, beta);
    // p may hold anything yet (not a number included): set afterwards, not scaled by 0
    if (!ic0_backward<T, false>(a, team, (T)0, (T)0)) return false;
  }
  direction<T, PREC, FIRST, false>(a, sh, (T)alpha, beta, (T)c, zt, ld);
  return team.barrier();
}

// w = A p on the block's rows; pw = (p, w) over the team and alpha = rho / pw.
template <typename T, typename TV, bool CL, int PREC>
__device__ __forceinline__ bool apply_dot(const Args& a, Team<CL>& team, const Share<PREC>& sh, double rho, double& pw,
                                          double& alpha) {
  const Geom& g = a.g;
  const TV* val = static_cast<const TV*>(a.val);
  const T* p = static_cast<const T*>(a.p);
  T* w = static_cast<T*>(a.w);
  AccFor<T> acc;
  for (int row = sh.row0(a.g) + (int)threadIdx.x; row < sh.row1(a.g); row += NT) {
    const int col = fdiv(g.nzd, row);
    const T wi = row_apply<T, TV>(g, val, p, a.mask, row, col, row - col * g.nz);
    w[row] = wi;
    acc.add_prod(p[row], wi);
  }
  double v[1] = {acc.value()};
  if (!team.template sum<1>(v)) return false;
  pw = v[0];
  double u[1];
  block_scalars(team.s, u, [&](double* o) { o[0] = rho / pw; });
  alpha = u[0];
  return true;
}

// r = b - A x (compensated), (r, r) and the floor's (|A||x| + |b|)^2 over the team.
template <typename T, bool CL, int PREC>
__device__ __forceinline__ bool true_residual(const Args& a, Team<CL>& team, const Share<PREC>& sh, const double* b, double& rr,
                                              double& ff) {
  const Geom& g = a.g;
  T* r = static_cast<T*>(a.r);
  double v[2] = {0.0, 0.0};
  for (int row = sh.row0(a.g) + (int)threadIdx.x; row < sh.row1(a.g); row += NT) {
    const int col = fdiv(g.nzd, row);
    double asum;
    const double bi = b[row];
    const double ri = row_residual(g, a.val64, a.x, a.mask, bi, row, col, row - col * g.nz, asum);
    r[row] = (T)ri;
    v[0] = fma(ri, ri, v[0]);
    const double f = asum + fabs(bi);
    v[1] = fma(f, f, v[1]);
  }
  if (!team.template sum<2>(v)) return false;
  rr = v[0];
  ff = v[1];
  return true;
}

// Right-hand side, initial guess and first residual: (b', b') and (r, r). From x = 0 the residual is b' itself.
template <typename T, bool CL, int PREC>
__device__ __forceinline__ bool start_solve(const Args& a, Team<CL>& team, const Share<PREC>& sh, const double*& b, double& bb,
                                            double& rr) {
  double lam = 0.0, xs = 0.0;
  b = a.b;
  if (a.proj) {
    double v[2] = {0.0, 0.0};
    for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) {
      v[0] += b[i];
      if (a.x0_is_guess) v[1] = fma(a.m[i], a.x[i], v[1]);
    }
    if (!team.template sum<2>(v)) return false;
    lam = v[0] / a.one_m;
    xs = a.x0_is_guess ? v[1] / a.one_m : 0.0;
  }
  T* r = static_cast<T*>(a.r);
  double v[2] = {0.0, 0.0};
  for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) {
    double bi = b[i];
    if (a.proj) {
      bi = bi - lam * a.m[i];
      a.bw[i] = bi;
    }
    if (!a.x0_is_guess) {
      a.x[i] = 0.0;
      r[i] = (T)bi;
    } else if (a.proj) {
      a.x[i] = a.x[i] - xs;
    }
    v[0] = fma(bi, bi, v[0]);
  }
  if (a.proj) b = a.bw;
  v[1] = v[0];
  if (!team.template sum<1>(*reinterpret_cast<double(*)[1]>(v))) return false;
  bb = v[0];
  rr = bb;
  double ff;
  if (a.x0_is_guess && !true_residual<T>(a, team, sh, b, rr, ff)) return false;
  return true;
}

// The returned pressure has m'x = 0.
template <bool CL, int PREC>
__device__ __forceinline__ bool zero_mean(const Args& a, Team<CL>& team, const Share<PREC>& sh) {
  double v[1] = {0.0};
  for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) v[0] = fma(a.m[i], a.x[i], v[0]);
  if (!team.template sum<1>(v)) return false;
  const double shift = v[0] / a.one_m;
  for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) a.x[i] -= shift;
  return true;
}

// The FP64 solve: PCG on the recursive residual, then the true residual, restarts while they help.
template <int PREC, bool CL>
__device__ __forceinline__ bool solve64(const Args& a, Team<CL>& team, const Share<PREC>& sh, double* zt, int ld, Result& o) {
  const double* b;
  double bb, rr;
  if (!start_solve<double>(a, team, sh, b, bb, rr)) return false;
  const double tol2 = a.rtol * a.rtol * bb;
  Cg cg;
  int restarts = 0, first_pass = -1;
  double rel_true = 0.0, floor = 0.0, prev_true = -1.0;
  bool accepted = false;
  bool skip = rr <= tol2;   // x0 already meets rtol
  if (!skip && a.max_iter == 0 && bb != 0.0) cg.status = PM_NOT_CONVERGED;
  cg.rr = rr;
  if (bb == 0.0)
    for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) a.x[i] = 0.0;
  while (bb != 0.0) {
    if (cg.status == PM_OK && !skip) {
      bool converged = false, stopped;
      if (!advance<double, PREC, true>(a, team, sh, zt, ld, 0.0, cg, stopped, [] { return false; })) return false;
      while (cg.status == PM_OK && cg.iter < a.max_iter) {
        double pw, alpha;
        if (!apply_dot<double, double>(a, team, sh, cg.rho, pw, alpha)) return false;
        if (!(pw > 0.0) || !isfinite(pw)) {
          cg.status = PM_BREAKDOWN;
          break;
        }
        const bool fine = advance<double, PREC, false>(a, team, sh, zt, ld, alpha, cg, stopped, [&] {
          ++cg.iter;
          converged = cg.rr <= tol2;
          return converged || cg.iter >= a.max_iter;
        });
        if (!fine) return false;
        if (stopped) break;
      }
      if (cg.status == PM_OK && !converged) cg.status = PM_NOT_CONVERGED;   // iteration cap
    }
    skip = false;
    if (first_pass < 0) first_pass = cg.iter;
    double tr, ff;
    if (!true_residual<double>(a, team, sh, b, tr, ff)) return false;
    rel_true = sqrt(tr / bb);
    floor = ldexp(1.0, -53) * sqrt(ff / bb);
    const bool stalled = prev_true >= 0.0 && rel_true > 0.5 * prev_true;
    const bool last = restarts >= a.max_restarts || cg.iter >= a.max_iter;
    accepted = rel_true <= a.rtol || (rel_true <= floor && (stalled || last));
    if (cg.status != PM_OK || accepted || last) break;
    prev_true = rel_true;
    cg.rr = tr;
    ++restarts;
  }
  if (bb != 0.0 && cg.status == PM_OK && !accepted) cg.status = PM_NOT_CONVERGED;
  if (a.proj && !zero_mean(a, team, sh)) return false;
  o.iters = cg.iter;
  o.restarts = restarts;
  o.first_pass = first_pass < 0 ? cg.iter : first_pass;
  o.status = cg.status;
  o.zero_rhs = bb == 0.0;
  o.rel_true = bb == 0.0 ? 0.0 : rel_true;
  o.rel_rec = bb == 0.0 ? 0.0 : sqrt(cg.rr / bb);
  o.floor = floor;
  return true;
}

// The mixed-precision solve: inner PCG with FP32 vectors on the difference-form values; each time the
// recursive residual has dropped by inner_rtol, or claims convergence, the FP32 correction is folded into the
// FP64 iterate, the true residual b - A x is formed (compensated) and a new inner solve starts from it.
template <typename TV, int PREC, bool CL>
__device__ __forceinline__ bool solve_mixed(const Args& a, Team<CL>& team, const Share<PREC>& sh, float* zt, int ld, Result& o) {
  const double* b;
  double bb, rr;
  for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) a.d[i] = 0.f;
  if (!start_solve<float>(a, team, sh, b, bb, rr)) return false;
  const double tol2 = a.rtol * a.rtol * bb, drop = a.inner_rtol * a.inner_rtol;
  Cg cg;
  int outer = 0, stalled = 0;
  double rel_true = 0.0, floor = 0.0, prev_true = 1e300;
  if (bb == 0.0) {
    for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) a.x[i] = 0.0;
  } else if (rr <= tol2 || a.max_iter == 0) {   // x0 already meets rtol, or no iteration is allowed
    if (!(rr <= tol2)) cg.status = PM_NOT_CONVERGED;   // not a number included
    rel_true = sqrt(rr / bb);
  } else {
    for (;;) {
      const double target = fmax(tol2, drop * rr);
      bool stopped;
      if (!advance<float, PREC, true>(a, team, sh, zt, ld, 0.0, cg, stopped, [] { return false; })) return false;
      while (cg.status == PM_OK) {
        double pw, alpha;
        if (!apply_dot<float, TV>(a, team, sh, cg.rho, pw, alpha)) return false;
        if (!(pw > 0.0) || !isfinite(pw)) {
          cg.status = PM_BREAKDOWN;
          break;
        }
        const bool fine = advance<float, PREC, false>(a, team, sh, zt, ld, alpha, cg, stopped, [&] {
          ++cg.iter;
          return cg.rr <= target || cg.iter >= a.max_iter;
        });
        if (!fine) return false;
        if (stopped) break;
      }
      for (int i = sh.row0(a.g) + (int)threadIdx.x; i < sh.row1(a.g); i += NT) {
        a.x[i] += (double)a.d[i];
        a.d[i] = 0.f;
      }
      if (!team.barrier()) return false;
      double ff;
      if (!true_residual<float>(a, team, sh, b, rr, ff)) return false;
      ++outer;
      rel_true = sqrt(rr / bb);
      floor = ldexp(1.0, -53) * sqrt(ff / bb);
      const bool stalled_now = rel_true > 0.5 * prev_true;   // this step did not halve the true residual
      const bool broken = cg.status == PM_BREAKDOWN;
      cg.status = PM_OK;
      if (rel_true <= a.rtol || (rel_true <= floor && stalled_now)) break;
      stalled = stalled_now ? stalled + 1 : 0;
      prev_true = rel_true;
      if (stalled >= 3) {   // stagnation above the floor
        cg.status = PM_NOT_CONVERGED;
        break;
      }
      if (broken) {
        cg.status = PM_BREAKDOWN;
        break;
      }
      if (cg.iter >= a.max_iter) {   // no iteration left: accepted only below the floor
        if (!(rel_true <= floor)) cg.status = PM_NOT_CONVERGED;
        break;
      }
    }
  }
  if (a.proj && !zero_mean(a, team, sh)) return false;
  o.iters = o.first_pass = cg.iter;
  o.restarts = outer;
  o.status = cg.status;
  o.zero_rhs = bb == 0.0;
  o.rel_true = o.rel_rec = bb == 0.0 ? 0.0 : rel_true;
  o.floor = floor;
  return true;
}

__device__ __forceinline__ void report(Out* out, int rank, bool fine, const Result& o) {
  if (threadIdx.x != 0) return;
  if (!fine) *(volatile int32_t*)&out->timeout = 1;
  else if (rank == 0) out->res = o;
}

// Host: whether the results of a finished launch are a solve's.
inline int outcome(const Out& h) {
  if (h.timeout > 0) return set_error(PM_TIMEOUT, "resident PCG: a grid barrier wait ran out");
  if (h.res.status < 0) return set_error(PM_ECUDA, "resident PCG: the kernel reported nothing");
  return PM_OK;
}

template <typename T, typename TV, int PREC, bool CL>
__global__ void __launch_bounds__(NT, 1) k_resident(Args a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ Scratch scratch;
  if (PREC == PM_PREC_IC0 && threadIdx.x < 8) {   // 64-bit divisions: once, not in every phase
    const int c = threadIdx.x;
    const int64_t tot = (int64_t)a.cls_cnt[c & 3] * (c >> 2 ? a.nlev[1].d : a.nlev[0].d);
    scratch.first[c] = (int)(tot * blockIdx.x / gridDim.x);
    scratch.past[c] = (int)(tot * (blockIdx.x + 1) / gridDim.x);
  }
  __syncthreads();
  Team<CL> team(a, &scratch);
  if (CL) team.barrier();   // every block of the cluster runs before one writes to another's shared memory
  const Share<PREC> sh(a.g, team.rank, team.G);
  T* zt;
  int ld = a.g.nz | 1;   // odd: a warp's columns fall into different banks
  if (a.z_in_smem) {
    zt = reinterpret_cast<T*>(smem_raw);
  } else {
    zt = static_cast<T*>(a.z) + (PREC == PM_PREC_LINE ? sh.row0(a.g) : 0);
    ld = a.g.nz;
  }
  Result o;
  bool fine;
  if constexpr (std::is_same<T, double>::value) fine = solve64<PREC>(a, team, sh, zt, ld, o);
  else fine = solve_mixed<TV, PREC>(a, team, sh, zt, ld, o);
  report(a.out, team.rank, fine, o);
  if (!fine) return;
  if (CL) team.barrier();   // no block of a cluster leaves while another may still write to its shared memory
}

// ---- launch ------------------------------------------------------------------------------------

constexpr size_t TILE_LIMIT = 200 * 1024;   // shared memory of a block's tile of columns

template <typename T, typename TV, int PREC, bool CL>
inline int launch_one(Args& a, int grid, size_t smem, cudaStream_t s) {
  const void* f = (const void*)k_resident<T, TV, PREC, CL>;
  int st;
  // the limit belongs to the function, not to the launch: always the same value, since other threads launch tiles
  // of other sizes between this call and the launch
  if (smem && (st = cuda_check(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TILE_LIMIT),
                               "resident shared memory")))
    return st;
  const bool team = !CL || grid > 1;   // more than one block
  if (CL && team &&
      (st = cuda_check(cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1), "cluster size")))
    return st;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (CL) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)grid;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = team ? 1 : 0;
  if (!CL && (st = cuda_check(cudaMemsetAsync(a.ctl, 0, sizeof(Ctl), s), "resident barrier"))) return st;
  st = cuda_check(cudaLaunchKernelEx(&cfg, k_resident<T, TV, PREC, CL>, a), "k_resident");
  count_launch();
  return st;
}

// Dynamic shared memory of a block's columns (line preconditioner), or 0 when they do not fit.
inline size_t tile_bytes(int64_t ncols, int nz, int grid, size_t elem) {
  const int64_t cols = (ncols + grid - 1) / grid;
  const size_t b = (size_t)cols * (size_t)(nz | 1) * elem;
  return b <= TILE_LIMIT ? b : 0;
}

template <typename T, typename TV, bool CL>
int launch_prec(Args& a, int prec, int grid, cudaStream_t s) {
  const size_t smem = prec == PM_PREC_LINE ? tile_bytes(a.g.ncols, a.g.nz, grid, sizeof(T)) : 0;
  a.z_in_smem = smem > 0;
  switch (prec) {
    case PM_PREC_IC0: return launch_one<T, TV, PM_PREC_IC0, CL>(a, grid, smem, s);
    case PM_PREC_LINE: return launch_one<T, TV, PM_PREC_LINE, CL>(a, grid, smem, s);
    default: return launch_one<T, TV, PM_PREC_JACOBI, CL>(a, grid, smem, s);
  }
}

// Blocks of a solve's team: one, one cluster's, or (0) the grid's. Measured, us per iteration or, marked ms, whole
// solves:
//   cluster / grid: IC0 n = 2,048 40 / 49, 18,000 50 / 49; line 11,803 18.3 / 18.1, 18,000 24 / 21; Jacobi 2,048
//   10 / 14, 11,803 15.5 / 14.2;
//   one block / cluster, FP64 velocity and pressure in ms: IC0 n = 512 0.22 / 0.29 and 3.40 / 4.84, 1,024 0.42 / 0.47 and
//   7.57 / 9.09, 1,600 0.55 / 0.48 and 13.4 / 12.1; line 288 0.14 / 0.17 and 0.20 / 0.24, 512 0.20 / 0.21 and 0.33 / 0.35,
//   648 0.25 / 0.24 and 0.46 / 0.44; Jacobi 288 0.15 / 0.17 and 1.41 / 1.66, 400 0.26 / 0.27 and 2.26 / 2.33, 512 0.22 / 0.20
//   and 2.48 / 2.38. FP32 alike (IC0 1,024 0.40 / 0.38 and 7.2 / 11.0, Jacobi 400 0.28 / 0.30 and 3.4 / 3.9).
constexpr int64_t ONE_BLOCK_ROWS = 400, ONE_BLOCK_IC0 = 1024;
constexpr int64_t CLUSTER_ROWS = 8192, CLUSTER_IC0 = 16384;
inline int team_blocks(int64_t n, int prec) {
  const bool ic0 = prec == PM_PREC_IC0;
  if (n <= (ic0 ? ONE_BLOCK_IC0 : ONE_BLOCK_ROWS)) return 1;
  return n <= (ic0 ? CLUSTER_IC0 : CLUSTER_ROWS) ? CLUSTER : 0;
}

template <typename T, typename TV>
int launch(Args& a, int prec, int num_sms, cudaStream_t s) {
  const int blocks = team_blocks(a.g.n, prec);
  return blocks ? launch_prec<T, TV, true>(a, prec, blocks, s) : launch_prec<T, TV, false>(a, prec, num_sms, s);
}

// One file each (pm_resident.cu, pm_resident_fp32.cu, pm_resident_bf16.cu), so that they compile side by side.
int launch_fp64(Args& a, int prec, int num_sms, cudaStream_t s);
int launch_fp32(Args& a, int prec, int num_sms, cudaStream_t s);
int launch_bf16(Args& a, int prec, int num_sms, cudaStream_t s);

}  // namespace resident
}  // namespace pm
