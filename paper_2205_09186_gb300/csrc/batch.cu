// Batched D2Q9 droplets of uneven sizes and parameters in one persistent
// launch.  Cases of FP32-deviation batches at tau = 1 advance on their moments, an
// even number of steps per call (k_batch_mom, a launch of its own); an odd step and
// the other cases run on the populations.  There (k_batch_split) the CTAs (collision
// items) and warps (mu units) claim the work of each phase from an atomic
// counter in guided runs; other precisions (k_batch_persistent) fetch their
// (case, tile) items one at a time from an atomic counter per phase.
// Compact-scheme cases (Eq. 21-24, OCFDS4 of Sec. 3.1) add phases to every
// step: their chemical-potential field (k_batch_persistent; the mu phase of
// k_batch_split already has one), then the periodic tridiagonal line solves
// for grad mu and grad rho along x and y (groups of lines as work items), each
// behind the same bounded barrier, before the collision reads the derivative
// fields.
// Steps and phases are separated by a device-wide barrier whose waits are
// bounded (about one second), after which the kernel records LBM_ETIMEOUT and
// returns.  lbm_batch_step captures the launches (plus the counter resets) in a
// CUDA graph and replays it; lbm_batch_autotune picks the tile shape.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/lbm.h"
#include "compact_dev.cuh"
#include "iir.cuh"
#include "launch.cuh"
#include "mom2d.cuh"
#include "step2d.cuh"
#include "step2d_split.cuh"

using namespace lbmd;

namespace {

constexpr int TXB = 32, TYB = 8;
constexpr unsigned long long BARRIER_NS = 1000000000ull;  // longest wait at a barrier

struct CaseDev {
  KParams kp;
  void* f[2];
  void* rho[2];  // density field: double (FP64) or float rho - rho_ref (FP32DEV)
  void* snap;
  float* mu;     // mu field (split FP32DEV path)
  unsigned long long* bad;
  int scheme;
  int tiles_x, tiles_y;
  int item_begin, item_end;      // observation / single-phase items
  int mtiles_x, ctiles_x;        // split path: mu tiles (32 wide) and collision tiles (30 wide) per row
  Mrt mrt;                       // collision operator of the case
  // compact schemes: order of the explicit Laplacian (4, 6, 8; 0 = not
  // compact), line coefficients (row of c_lines), mu field (type P::Tm; the
  // split path's mu), grad mu (P::Tm) and grad rho (P::Tc), 2 N each
  int lap, lci;
  void* cmu;
  void* gmu;
  void* grho;
  // steps on the moments (k_batch_mom); mom = 0: on the populations
  int mom;
  Mom2Geo mg;
};

// line coefficients of CFDS4, CFDS6, CFDS8, OCFDS4: [0] all PCR levels (FP64
// lines), [1] the levels that move a float (FP32 lines)
__constant__ LineCoef c_lines[2][4];

__host__ __device__ __forceinline__ bool is_compact(int scheme) { return scheme >= S_CFDS4 && scheme <= S_OCFDS4; }

struct Item {
  int c, tile;
};

struct BatchCtl {
  unsigned int count;
  unsigned int gen;
  unsigned int work[4];  // k_batch_split: [(2 step + phase) % 4]; k_batch_persistent: [step parity]
  int status;
  int skip_block;  // fault injection for tests: this CTA never arrives (-1: none)
  long long t;     // step counter of the batch
};

__device__ __forceinline__ unsigned long long gtime() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Device-wide barrier with a bounded wait.  Returns false (for every thread of
// the CTA) when the wait timed out or another CTA already reported an error.
__device__ bool grid_barrier(BatchCtl* ctl, unsigned long long timeout_ns) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    if (int(blockIdx.x) == ctl->skip_block) {
      ok = 0;  // injected non-arrival: leave without arriving
    } else {
      __threadfence();
      const unsigned gen = ld_acquire(&ctl->gen);
      __threadfence();
      const unsigned arrived = atomicAdd(&ctl->count, 1u);
      if (arrived == gridDim.x - 1) {
        atomicExch(&ctl->count, 0u);
        __threadfence();
        atomicAdd(&ctl->gen, 1u);
      } else {
        const unsigned long long t0 = gtime();
        while (ld_acquire(&ctl->gen) == gen) {
          if (gtime() - t0 > timeout_ns) {
            atomicExch(&ctl->status, LBM_ETIMEOUT);
            ok = 0;
            break;
          }
          __nanosleep(256);
        }
      }
      __threadfence();
      if (atomicAdd(&ctl->status, 0) != 0) ok = 0;
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <class P>
__device__ void run_item(const CaseDev& cd, int tile, long long t, unsigned char* smem, int mode, double* partial) {
  using Tf = typename P::Tf;
  using Tr = typename P::Tr;
  const int par = int(t & 1);
  const int x0 = (tile % cd.tiles_x) * TXB, y0 = (tile / cd.tiles_x) * TYB;
  StepAux aux;
  aux.t = t;
  aux.bad_step = cd.bad;
  aux.partials = nullptr;
  aux.rho_snap = cd.snap;
  FieldOut fo{nullptr, nullptr};
  GradIn gi{cd.gmu, cd.grho, cd.cmu};
  const Tf* fin = static_cast<const Tf*>(cd.f[par]);
  Tf* fout = static_cast<Tf*>(cd.f[par ^ 1]);
  const Tr* rin = static_cast<const Tr*>(cd.rho[par]);
  Tr* rout = static_cast<Tr*>(cd.rho[par ^ 1]);
#define LBM_ITEM_CASE(S)                                                                                   \
  case S:                                                                                                  \
    if (mode == MODE_STEP)                                                                                 \
      step2d_tile<S, P, TXB, TYB, MODE_STEP>(cd.kp, fin, fout, rin, rout, aux, fo, gi, cd.mrt, x0, y0, smem, partial); \
    else                                                                                                   \
      step2d_tile<S, P, TXB, TYB, MODE_OBS>(cd.kp, fin, fout, rin, rout, aux, fo, gi, cd.mrt, x0, y0, smem, partial); \
    break;
  switch (cd.scheme) {
    LBM_ITEM_CASE(S_EFDS2)
    LBM_ITEM_CASE(S_EFDS4)
    LBM_ITEM_CASE(S_EFDS6)
    LBM_ITEM_CASE(S_E4)
    LBM_ITEM_CASE(S_E8)
    default:
      if (is_compact(cd.scheme)) {  // derivatives from the line solves of this step
        if (mode == MODE_STEP)
          step2d_tile<S_CFDS4, P, TXB, TYB, MODE_STEP>(cd.kp, fin, fout, rin, rout, aux, fo, gi, cd.mrt, x0, y0, smem,
                                                        partial);
        else
          step2d_tile<S_CFDS4, P, TXB, TYB, MODE_OBS>(cd.kp, fin, fout, rin, rout, aux, fo, gi, cd.mrt, x0, y0, smem,
                                                       partial);
      }
      break;
  }
#undef LBM_ITEM_CASE
}

// compact case: mu of one 32 x 8 tile (one node per thread of NT2)
template <class P>
__device__ void cmu_tile(const CaseDev& cd, int tile, long long t) {
  using Tm = typename P::Tm;
  using Tr = typename P::Tr;
  const Tr* rin = static_cast<const Tr*>(cd.rho[int(t & 1)]);
  const int x = (tile % cd.tiles_x) * TXB + int(threadIdx.x) % TXB;
  const int y = (tile / cd.tiles_x) * TYB + int(threadIdx.x) / TXB;
  if (x < cd.kp.nx && y < cd.kp.ny) {
    const long long n = (long long)y * cd.kp.nx + x;
    static_cast<Tm*>(cd.cmu)[n] = mu_field_node_order<Tm, Tr>(cd.lap, cd.kp, 2, P::DEV, rin, n);
  }
}

// compact case: one group of lines (code = group * 4 + set; set = 2 axis +
// field, field 0 mu -> grad mu, 1 rho -> grad rho) by a CTA of NTH threads
template <int NTH, class P>
__device__ void line_item(const CaseDev& cd, int code, long long t, int lpb, int lpb_shift, unsigned char* smem) {
  using Tm = typename P::Tm;
  using Tr = typename P::Tr;
  using Tc = typename P::Tc;
  const int set = code & 3, grp = code >> 2, axis = set >> 1;
  const long long N = cd.kp.n;
  const int nx = cd.kp.nx, ny = cd.kp.ny;
  if ((set & 1) == 0) {
    lines_block<NTH, Tm, Tm>(axis, nx, ny, 1, static_cast<const Tm*>(cd.cmu), static_cast<Tm*>(cd.gmu) + axis * N,
                             c_lines[sizeof(Tm) == 4][cd.lci], lpb, lpb_shift, grp, smem);
  } else {
    lines_block<NTH, Tr, Tc>(axis, nx, ny, 1, static_cast<const Tr*>(cd.rho[int(t & 1)]),
                             static_cast<Tc*>(cd.grho) + axis * N, c_lines[sizeof(Tc) == 4][cd.lci], lpb, lpb_shift,
                             grp, smem);
  }
}

// Every step: [mu tiles of the compact cases] -> [their line groups] -> the
// step items of all cases, each phase followed by the bounded barrier.  Phase
// k of a launch counts on work[k % 4]; block 0 zeroes work[(k + 2) % 4], last
// used two phases back, before it arrives at the phase's barrier (the launch
// starts from zeroed counters).
template <class P>
__global__ void __launch_bounds__(NT2) k_batch_persistent(const CaseDev* __restrict__ cases,
                                                          const Item* __restrict__ items, int nitems, int nsteps,
                                                          BatchCtl* ctl, unsigned long long timeout_ns,
                                                          const Item* __restrict__ cmu_items, int ncmu,
                                                          const Item* __restrict__ line_items, int nline, int lpb,
                                                          int lpb_shift) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  const long long t0 = *((volatile long long*)&ctl->t);
  int k = 0;  // phase of the launch
  // items of one phase, fetched one at a time by the CTAs; false if the
  // barrier after it failed
  auto phase = [&](const Item* its, int n, auto&& fn) {
    unsigned* ctr = &ctl->work[k & 3];
    for (;;) {
      if (threadIdx.x == 0) s_item = int(atomicAdd(ctr, 1u));
      __syncthreads();
      const int it = s_item;
      __syncthreads();
      if (it >= n) break;
      fn(its[it]);
      __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->work[(k + 2) & 3] = 0u;
    ++k;
    return grid_barrier(ctl, timeout_ns);
  };
  for (int s = 0; s < nsteps; ++s) {
    const long long t = t0 + s;
    if (ncmu > 0 && !phase(cmu_items, ncmu, [&](const Item& itm) { cmu_tile<P>(cases[itm.c], itm.tile, t); })) return;
    if (nline > 0 && !phase(line_items, nline, [&](const Item& itm) {
          line_item<NT2, P>(cases[itm.c], itm.tile, t, lpb, lpb_shift, smem);
        }))
      return;
    if (!phase(items, nitems, [&](const Item& itm) { run_item<P>(cases[itm.c], itm.tile, t, smem, MODE_STEP, nullptr); }))
      return;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->t = t0 + nsteps;
}

// FP32DEV: per step a mu phase over all cases' mu tiles (warp units of eight
// rows, read straight from global memory) and a collision phase over their
// collision tiles, each followed by the bounded device barrier.  A collision
// item is staged in shared memory: the copies of the next item are in flight
// while the current one is computed from the other buffer.
template <int RPT>
__device__ void coll_load(const CaseDev& cd, int tile, long long t, unsigned char* buf) {
  constexpr int T2Y = Tile2<RPT>::T2Y;
  const int par = int(t & 1);
  const float* rin = static_cast<const float*>(cd.rho[par]);
  const int x0 = (tile % cd.ctiles_x) * T2X, y0 = (tile / cd.ctiles_x) * T2Y;
  const float* fin = static_cast<const float*>(cd.f[par]);
  switch (cd.scheme) {
    case S_EFDS2: coll2d_load<S_EFDS2, RPT>(cd.kp, fin, rin, cd.mu, x0, y0, buf); break;
    case S_EFDS4: coll2d_load<S_EFDS4, RPT>(cd.kp, fin, rin, cd.mu, x0, y0, buf); break;
    case S_EFDS6: coll2d_load<S_EFDS6, RPT>(cd.kp, fin, rin, cd.mu, x0, y0, buf); break;
    case S_E4: coll2d_load<S_E4, RPT>(cd.kp, fin, rin, cd.mu, x0, y0, buf); break;
    case S_E8: coll2d_load<S_E8, RPT>(cd.kp, fin, rin, cd.mu, x0, y0, buf); break;
    default:
      if (is_compact(cd.scheme))
        coll2d_load<S_CFDS4, RPT>(cd.kp, fin, rin, cd.mu, x0, y0, buf, static_cast<const float*>(cd.gmu),
                                  static_cast<const float*>(cd.grho));
      break;
  }
}

// one warp's mu unit: rows part * MU_UNIT_ROWS .. + MU_UNIT_ROWS - 1 of a mu tile
template <int RPT>
__device__ void mu_unit(const CaseDev& cd, int tile, int part, long long t, int lane) {
  constexpr int M2Y = Tile2<RPT>::M2Y;
  const int par = int(t & 1);
  const float* rin = static_cast<const float*>(cd.rho[par]);
  const int x0 = (tile % cd.mtiles_x) * M2X, y0 = (tile / cd.mtiles_x) * M2Y + part * MU_UNIT_ROWS;
  if (y0 >= cd.kp.ny) return;
  switch (cd.scheme) {
    case S_EFDS2: mu2d_rows<S_EFDS2>(cd.kp, rin, cd.mu, x0, y0, lane); break;
    case S_EFDS4: mu2d_rows<S_EFDS4>(cd.kp, rin, cd.mu, x0, y0, lane); break;
    case S_EFDS6: mu2d_rows<S_EFDS6>(cd.kp, rin, cd.mu, x0, y0, lane); break;
    case S_E4: mu2d_rows<S_E4>(cd.kp, rin, cd.mu, x0, y0, lane); break;
    case S_E8: mu2d_rows<S_E8>(cd.kp, rin, cd.mu, x0, y0, lane); break;
    default:
      if (is_compact(cd.scheme)) {
        // the compact scheme's chemical potential, node by node as in the
        // single-case path (explicit Laplacian of the scheme's order)
        const int gx = x0 + lane;
        if (gx >= cd.kp.nx) break;
        for (int r = 0; r < MU_UNIT_ROWS && y0 + r < cd.kp.ny; ++r) {
          const long long n = (long long)(y0 + r) * cd.kp.nx + gx;
          cd.mu[n] = mu_field_node_order<float, float>(cd.lap, cd.kp, 2, true, rin, n);
        }
      }
      break;
  }
}

template <int RPT>
__device__ void coll_compute(const CaseDev& cd, int tile, long long t, unsigned char* buf) {
  constexpr int T2Y = Tile2<RPT>::T2Y;
  const int par = int(t & 1);
  const int x0 = (tile % cd.ctiles_x) * T2X, y0 = (tile / cd.ctiles_x) * T2Y;
  float* fout = static_cast<float*>(cd.f[par ^ 1]);
  float* rout = static_cast<float*>(cd.rho[par ^ 1]);
  const bool tau1 = cd.kp.omega == 1.0;
#define LBM_SPLIT_CASE(SS)                                                              \
  case SS:                                                                              \
    if (tau1) coll2d_compute<SS, true, RPT>(cd.kp, fout, rout, cd.bad, t, x0, y0, buf, cd.mrt); \
    else coll2d_compute<SS, false, RPT>(cd.kp, fout, rout, cd.bad, t, x0, y0, buf, cd.mrt);     \
    break;
  switch (cd.scheme) {
    LBM_SPLIT_CASE(S_EFDS2)
    LBM_SPLIT_CASE(S_EFDS4)
    LBM_SPLIT_CASE(S_EFDS6)
    LBM_SPLIT_CASE(S_E4)
    LBM_SPLIT_CASE(S_E8)
    default:
      if (is_compact(cd.scheme)) {
        if (tau1) coll2d_compute<S_CFDS4, true, RPT>(cd.kp, fout, rout, cd.bad, t, x0, y0, buf, cd.mrt);
        else coll2d_compute<S_CFDS4, false, RPT>(cd.kp, fout, rout, cd.bad, t, x0, y0, buf, cd.mrt);
      }
      break;
  }
#undef LBM_SPLIT_CASE
}

// Items of a phase are dealt dynamically in guided runs: a CTA claims a run of
// consecutive items from the phase's counter, up to 16 while much work is
// left and shrinking to single items at the end.  Item costs differ by scheme
// (E8's 5 x 5 stencils against EFDS2's 3-point lines) and by how much of a
// ragged tile lies on the lattice, so equal static shares left the average CTA
// waiting 29% of the step at the grid barriers; runs keep neighbouring tiles of
// one case on one CTA (halo lines reused from L1).  In the collision phase
// the claimant is the CTA: thread 0 claims its next run when it starts the
// current one, so the atomic's round trip is hidden, and each item's index
// reaches the other threads through a two-slot shared queue at the barrier
// every item already has.  The mu phase needs no CTA barrier: each warp claims
// units of eight tile rows itself (lane 0, broadcast by a shuffle), which
// also balances the warps of a CTA.  Phase k of a launch (k = 2 step +
// phase) counts on work[k % 4]; block 0 zeroes work[(k + 2) % 4], last used
// two phases back, before it arrives at the phase's barrier, and the launch
// starts from zeroed counters.
// Dynamic shared memory: NBUF buffers of buf_bytes (a multiple of 16); two
// 30 x 30 tiles' buffers (~48 KB each) keep two CTAs resident per SM.
constexpr int NBUF = 2;

// one claimant's claims in a phase of n units: the run [lo, hi) being worked
// through and the run of nc units from nlo claimed after it
constexpr int RUN_MU = 16, RUN_COLL = 16, RUN_DIV = 4;
struct Claims {
  int lo, hi, nlo, nc, cap, g;
  // a run: 1/RUN_DIV of an equal share (over g claimants) of what is left, 1..cap units
  __device__ int size(int n, int v) const {
    const int share = (n - v) / (RUN_DIV * g);
    return share < 1 ? 1 : (share > cap ? cap : share);
  }
  __device__ void start(unsigned* ctr, int n, int run_cap, int claimants) {
    cap = run_cap;
    g = claimants;
    const int c = size(n, 0);
    lo = int(atomicAdd(ctr, unsigned(c)));
    hi = lo + c;
    nc = size(n, lo);
    nlo = int(atomicAdd(ctr, unsigned(nc)));
  }
  // the next unit index (>= n: the phase has no more work for this claimant)
  __device__ int next(unsigned* ctr, int n) {
    if (lo >= hi) {
      lo = nlo;
      hi = nlo + nc;
      nc = size(n, lo);
      nlo = int(atomicAdd(ctr, unsigned(nc)));
    }
    return lo++;
  }
};

template <int RPT>  // rows per thread of the tiles (1, 2, 4)
__global__ void __launch_bounds__(NT2S, RPT >= 4 ? 1 : 2) k_batch_split(const CaseDev* __restrict__ cases,
                                                      const Item* __restrict__ mitems, int nmu,
                                                      const Item* __restrict__ citems, int ncoll, int nsteps,
                                                      BatchCtl* ctl, unsigned long long timeout_ns, int buf_bytes,
                                                      const Item* __restrict__ litems, int nline, int lpb,
                                                      int lpb_shift) {
  static_assert(NBUF == 2, "one item in flight: the claim queue has two slots");
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_q[2];
  __shared__ Claims s_cl[NT2S / 32];  // in shared memory: registers are at the cap
  const long long t0 = *((volatile long long*)&ctl->t);
  int k = 0;  // phase of the launch: mu, [lines,] collision per step
  for (int s = 0; s < nsteps; ++s) {
    const long long t = t0 + s;
    for (int phase = 0; phase < 3; ++phase) {
      if (phase == 1 && nline == 0) continue;
      const Item* items = phase == 0 ? mitems : (phase == 1 ? litems : citems);
      const int nitems = phase == 0 ? nmu : (phase == 1 ? nline : ncoll);
      unsigned* ctr = &ctl->work[k & 3];
      if (phase == 1) {
        // line groups of the compact cases, one at a time per CTA
        for (;;) {
          if (threadIdx.x == 0) s_q[0] = int(atomicAdd(ctr, 1u));
          __syncthreads();
          const int it = s_q[0];
          __syncthreads();
          if (it >= nitems) break;
          const Item itm = items[it];
          line_item<NT2S, PrecF32>(cases[itm.c], itm.tile, t, lpb, lpb_shift, smem);
          __syncthreads();
        }
      } else if (phase == 0) {
        // mu: each warp claims units of MU_UNIT_ROWS rows of a mu tile and
        // reads their stencils with cached global loads; no staging, no CTA barrier
        constexpr int UPI = Tile2<RPT>::M2Y / MU_UNIT_ROWS;
        const int n = nitems * UPI, lane = int(threadIdx.x) & 31;
        Claims& cl = s_cl[threadIdx.x / 32];  // lane 0's
        if (lane == 0) cl.start(ctr, n, RUN_MU, int(gridDim.x) * (NT2S / 32));
        for (;;) {
          int u = 0;
          if (lane == 0) u = cl.next(ctr, n);
          u = __shfl_sync(0xffffffffu, u, 0);
          if (u >= n) break;
          const Item itm = items[u / UPI];
          mu_unit<RPT>(cases[itm.c], itm.tile, u % UPI, t, lane);
        }
      } else {
        Claims& cl = s_cl[0];  // thread 0's
        if (threadIdx.x == 0) {
          cl.start(ctr, nitems, RUN_COLL, int(gridDim.x));
          s_q[0] = cl.next(ctr, nitems);
        }
        __syncthreads();
        int cur = s_q[0], q = 1;
        // a slot is rewritten two items after it was read, by thread 0 past
        // the barrier that every reader reached after reading it
        int b = 0;
        if (cur < nitems) {
          const Item itm = items[cur];
          coll_load<RPT>(cases[itm.c], itm.tile, t, smem);
        }
        cpa_commit();
        while (cur < nitems) {
          if (threadIdx.x == 0) s_q[q] = cl.next(ctr, nitems);
          // this item's copies have landed, every thread is past the
          // computation of the item before, and the next index is published:
          // one barrier covers the data, the reuse of the other buffer and the claim
          cpa_wait_all();
          __syncthreads();
          const int nxt = s_q[q];
          q ^= 1;
          if (nxt < nitems) {
            const Item itm = items[nxt];
            coll_load<RPT>(cases[itm.c], itm.tile, t, smem + (b ^ 1) * buf_bytes);
          }
          cpa_commit();
          const Item itm = items[cur];
          coll_compute<RPT>(cases[itm.c], itm.tile, t, smem + b * buf_bytes);
          cur = nxt;
          b ^= 1;
        }
        cpa_wait_all();
      }
      if (blockIdx.x == 0 && threadIdx.x == 0) ctl->work[(k + 2) & 3] = 0u;
      ++k;
      if (!grid_barrier(ctl, timeout_ns)) return;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->t = t0 + nsteps;
}

// An even number of steps of the cases that advance on their moments (mom2d.cuh):
// gather, then nsteps times every tile, the last time forming the populations,
// each phase followed by the bounded barrier.  Compact cases make a step three
// phases: their mu, F / rho along their lines (iir.cuh) with the other cases'
// tiles behind them, their tiles. (48 cases, 8 of them compact: 79 us a step so; 85
// with the other cases' tiles beside the mu or the compact tiles, 86 with a third
// in each phase, whose ends then all wait for part-filled waves. On the populations
// the batch took 231; its 40 explicit cases alone 125 and now 44.)
// Item b of a phase goes to CTA b, further ones are
// claimed from the phase's counter while the one before is being computed.  The
// moments live in the buffers the populations are not in; after an even number of
// steps the populations belong in the buffers they started in.  set_t: this
// launch ends the batch's step.
struct IirAll {
  IirK<float> k[4];  // CFDS4, CFDS6, CFDS8, OCFDS4
};

template <bool FINAL>
__device__ __forceinline__ void mom_tile(const CaseDev& cd, int par, int s, long long t, int tile, float* smem) {
  const int row = tile / cd.mg.nt, x0 = (tile - row * cd.mg.nt) * cd.mg.TW, y0 = row * cd.mg.TH;
  const int vw = min(cd.mg.TW, cd.kp.nx - x0), vh = min(cd.mg.TH, cd.kp.ny - y0);
  float* m = static_cast<float*>(cd.f[par ^ 1]);
  float* f = static_cast<float*>(cd.f[par]);
  float* rho = static_cast<float*>(cd.rho[par]);
  const int a = s & 1, P = cd.mg.P;
  const float *r = m + a * P, *j = m + (2 + 2 * a) * P;
  float *ro = FINAL ? rho : m + (a ^ 1) * P, *jo = m + (2 + 2 * (a ^ 1)) * P;
#define LBM_MOM_CASE(SS) \
  case SS: mom2_tile<SS, FINAL>(cd.kp, cd.mg.LX, P, r, j, ro, jo, f, cd.bad, t, x0, y0, vw, vh, smem); break;
  switch (cd.scheme) {
    LBM_MOM_CASE(S_EFDS2)
    LBM_MOM_CASE(S_EFDS4)
    LBM_MOM_CASE(S_EFDS6)
    LBM_MOM_CASE(S_E4)
    LBM_MOM_CASE(S_E8)
    default:
      mom2_tile<S_CFDS4, FINAL>(cd.kp, cd.mg.LX, P, r, j, ro, jo, f, cd.bad, t, x0, y0, vw, vh, smem,
                                static_cast<const float*>(cd.gmu));
      break;
  }
#undef LBM_MOM_CASE
}

// mu of a compact case: 64 columns x 32 rows per CTA (tiles across: ceil(nx / 64))
__device__ __forceinline__ void mom_cmu(const CaseDev& cd, int par, int s, int tile) {
  const int nt = (cd.kp.nx + 63) / 64, row = tile / nt, w = int(threadIdx.x >> 5);
  const int x0 = (tile - row * nt) * 64 + 32 * (w & 1), y0 = row * 32 + 8 * (w >> 1);
  const float* r = static_cast<const float*>(cd.f[par ^ 1]) + (s & 1) * cd.mg.P;
  if (cd.lap == 4) mom2_mu_rows<4>(cd.kp, cd.mg.LX, r, cd.mu, x0, y0);
  else if (cd.lap == 6) mom2_mu_rows<6>(cd.kp, cd.mg.LX, r, cd.mu, x0, y0);
  else mom2_mu_rows<8>(cd.kp, cd.mg.LX, r, cd.mu, x0, y0);
}

// F / rho of a compact case: groups of lines along x, then of columns
__device__ __noinline__ void mom_acc(const CaseDev& cd, const IirAll& ia, int par, int s, int g, float* smem) {
  const int nx = cd.kp.nx, ny = cd.kp.ny, rows = (ny + IIR_CTA_ROWS - 1) / IIR_CTA_ROWS, LX = cd.mg.LX;
  const float* r = static_cast<const float*>(cd.f[par ^ 1]) + (s & 1) * cd.mg.P;
  const float rref = float(cd.kp.rho_ref);
  float* acc = static_cast<float*>(cd.gmu);
  float* kf = smem + IIR_CTA_FLOATS;
  const IirK<float>& c = *reinterpret_cast<const IirK<float>*>(kf);
  if (threadIdx.x < sizeof(IirK<float>) / 4) kf[threadIdx.x] = reinterpret_cast<const float*>(&ia.k[cd.lci])[threadIdx.x];
  __syncthreads();
  if (g < rows) {
    iir_cta_rows(c, nx, ny, LX, 8, r, cd.mu, acc, rref, g * IIR_CTA_ROWS, smem);
  } else {
    const int x0 = (g - rows) * iir_cta_cols_n(ny);
    acc += cd.kp.n;
    if (ny <= 256) iir_cta_cols<16>(c, nx, ny, LX, 8, r, cd.mu, acc, rref, x0, smem);
    else iir_cta_cols<8>(c, nx, ny, LX, 8, r, cd.mu, acc, rref, x0, smem);
  }
}

static_assert(sizeof(float) * IIR_CTA_FLOATS + sizeof(IirK<float>) <= T2_SMEM, "line groups of a batch");

// work lists of k_batch_mom: tiles of the explicit cases; the compact cases' mu
// tiles, line groups and tiles
struct MomWork {
  const Item *tiles, *cmp[3];
  int ntiles, ncmp[3];
};

__global__ void __launch_bounds__(T2NT, T2_CTAS) k_batch_mom(const CaseDev* __restrict__ cases, const MomWork work,
                                                             int nsteps, BatchCtl* ctl, unsigned long long timeout_ns,
                                                             int set_t, const __grid_constant__ IirAll ia) {
  extern __shared__ __align__(16) unsigned char smem_[];
  float* smem = reinterpret_cast<float*>(smem_);
  __shared__ int s_q[2];
  const long long t0 = *((volatile long long*)&ctl->t);
  const int par = int(t0 & 1), w = int(threadIdx.x >> 5);
  const int ph = work.ncmp[2] > 0 ? 3 : 1;  // phases of a step
  int q = 0, s = 0, f = 2;                  // step and its phase
  unsigned k = 0;                           // phase of the launch, modulo 2^32 (three times INT_MAX steps exceed an int)
  for (bool gather = true;; gather = false, ++k) {
    const bool last = s == nsteps - 1;
    const Item* cmp = work.cmp[f];
    const int nc = work.ncmp[f], n = nc + (gather || ph == 1 || f == 1 ? work.ntiles : 0);
    unsigned* ctr = &ctl->work[k & 3];
    for (int u = int(blockIdx.x); u < n;) {
      // (a slot is rewritten two items after it was read, past the barrier below)
      if (threadIdx.x == 0) s_q[q] = int(gridDim.x) + int(atomicAdd(ctr, 1u));
      const Item itm = u < nc ? cmp[u] : work.tiles[u - nc];
      const CaseDev& cd = cases[itm.c];
      if (gather) {
        const int row = itm.tile / cd.mg.nt, x0 = (itm.tile - row * cd.mg.nt) * cd.mg.TW, y0 = row * cd.mg.TH;
        const int vw = min(cd.mg.TW, cd.kp.nx - x0), vh = min(cd.mg.TH, cd.kp.ny - y0);
        for (int y = y0 + w; y < y0 + vh; y += T2NT / 32)
          mom2_gather(cd.kp, cd.mg.LX, cd.mg.P, static_cast<const float*>(cd.f[par]),
                      static_cast<const float*>(cd.rho[par]), static_cast<float*>(cd.f[par ^ 1]),
                      static_cast<float*>(cd.f[par ^ 1]) + 2 * cd.mg.P, cd.bad, t0, x0, vw, y, y + 1);
      } else if (u < nc && f < 2) {
        if (f == 0) mom_cmu(cd, par, s, itm.tile);
        else mom_acc(cd, ia, par, s, itm.tile, smem);
      } else {
        if (last) mom_tile<true>(cd, par, s, t0 + s, itm.tile, smem);
        else mom_tile<false>(cd, par, s, t0 + s, itm.tile, smem);
      }
      __syncthreads();
      u = s_q[q];
      q ^= 1;
    }
    if (!gather && last && f == ph - 1) break;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->work[(k + 2) & 3] = 0u;
    if (!grid_barrier(ctl, timeout_ns)) return;
    if (gather) {
      f = 0;
    } else if (++f == ph) {
      f = 0;
      ++s;
    }
  }
  if (set_t && blockIdx.x == 0 && threadIdx.x == 0) ctl->t = t0 + nsteps;
}

// derivative fields of the compact cases for the current state (before an
// observation pass): mu tiles, then line groups, one CTA per item
template <class P>
__global__ void __launch_bounds__(NT2) k_batch_cmu(const CaseDev* __restrict__ cases, const Item* __restrict__ items,
                                                   const BatchCtl* ctl) {
  const Item itm = items[blockIdx.x];
  cmu_tile<P>(cases[itm.c], itm.tile, ctl->t);
}
template <class P>
__global__ void __launch_bounds__(NT2) k_batch_clines(const CaseDev* __restrict__ cases, const Item* __restrict__ items,
                                                      const BatchCtl* ctl, int lpb, int lpb_shift) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Item itm = items[blockIdx.x];
  line_item<NT2, P>(cases[itm.c], itm.tile, ctl->t, lpb, lpb_shift, smem);
}

// observation pass: one CTA per work item (not persistent)
template <class P>
__global__ void __launch_bounds__(NT2) k_batch_obs(const CaseDev* __restrict__ cases, const Item* __restrict__ items,
                                                   const BatchCtl* ctl, double* partials) {
  extern __shared__ __align__(16) unsigned char smem[];
  const Item itm = items[blockIdx.x];
  run_item<P>(cases[itm.c], itm.tile, ctl->t, smem, MODE_OBS, partials + 4 * blockIdx.x);
}

// per case: reduce its items' partials; out[c*8 + ...]
__global__ void k_batch_obs_final(const CaseDev* __restrict__ cases, const BatchCtl* ctl, const double* partials,
                                  double* out, int dev) {
  __shared__ double red[4][256];
  const CaseDev& cd = cases[blockIdx.x];
  double a = 0, b = 0, c = 0, d = 0;
  for (int i = cd.item_begin + threadIdx.x; i < cd.item_end; i += blockDim.x) {
    a = fmax(a, partials[4 * i]);
    b = fmax(b, partials[4 * i + 1]);
    c += partials[4 * i + 2];
    d = fmax(d, partials[4 * i + 3]);
  }
  red[0][threadIdx.x] = a; red[1][threadIdx.x] = b; red[2][threadIdx.x] = c; red[3][threadIdx.x] = d;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      red[0][threadIdx.x] = fmax(red[0][threadIdx.x], red[0][threadIdx.x + s]);
      red[1][threadIdx.x] = fmax(red[1][threadIdx.x], red[1][threadIdx.x + s]);
      red[2][threadIdx.x] += red[2][threadIdx.x + s];
      red[3][threadIdx.x] = fmax(red[3][threadIdx.x], red[3][threadIdx.x + s]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int par = int(ctl->t & 1);
    const long long center = (long long)(cd.kp.ny / 2) * cd.kp.nx + cd.kp.nx / 2;
    double* o = out + 8 * blockIdx.x;
    o[0] = red[0][0]; o[1] = red[1][0]; o[2] = red[2][0]; o[3] = red[3][0];
    if (dev) {
      const float* r = static_cast<const float*>(cd.rho[par]);
      o[4] = cd.kp.rho_ref + double(r[center]);
      o[5] = cd.kp.rho_ref + double(r[0]);
    } else {
      const double* r = static_cast<const double*>(cd.rho[par]);
      o[4] = r[center];
      o[5] = r[0];
    }
    reinterpret_cast<unsigned long long*>(o)[6] = *cd.bad;
  }
}

// rho snapshot of every case (for the max |d rho / dt| observable)
template <typename Tr>
__global__ void k_batch_snap(const CaseDev* __restrict__ cases, const BatchCtl* ctl) {
  const CaseDev& cd = cases[blockIdx.y];
  const int par = int(ctl->t & 1);
  const Tr* r = static_cast<const Tr*>(cd.rho[par]);
  Tr* s = static_cast<Tr*>(cd.snap);
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < cd.kp.n; n += (long long)gridDim.x * blockDim.x)
    s[n] = r[n];
}

template <class P>
size_t batch_smem() {
  size_t m = Step2DShape<S_CFDS4, P, TXB, TYB>::bytes;
  m = std::max(m, Step2DShape<S_EFDS2, P, TXB, TYB>::bytes);
  m = std::max(m, Step2DShape<S_EFDS4, P, TXB, TYB>::bytes);
  m = std::max(m, Step2DShape<S_EFDS6, P, TXB, TYB>::bytes);
  m = std::max(m, Step2DShape<S_E4, P, TXB, TYB>::bytes);
  m = std::max(m, Step2DShape<S_E8, P, TXB, TYB>::bytes);
  return m;
}

}  // namespace

struct lbm_batch {
  int n = 0, prec = 0;
  cudaStream_t stream = nullptr;
  lbm_allocator alloc{};
  std::vector<lbm_params> p;
  std::vector<CaseDev> host_cases;
  std::vector<int> order;  // case c is host index order[k]... (identity: cases keep input order)
  CaseDev* d_cases = nullptr;
  Item* d_items = nullptr;
  int nitems = 0;
  BatchCtl* ctl = nullptr;
  double* d_partials = nullptr;
  double* d_out = nullptr;
  long long t = 0, t_snap = 0;
  int grid = 0;
  size_t smem = 0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  long long graph_steps = -1;
  bool split = false;
  Item* d_mitems = nullptr;
  Item* d_citems = nullptr;
  int nmu = 0, ncoll = 0, grid_split = 0;
  size_t smem_split = 0;
  int buf_split = 0;  // bytes of one item buffer of the split kernel
  int rpt = 0;        // split kernel: tile rows per thread (1, 2, 4)
  int item_cap = 0;   // capacity of d_mitems and of d_citems
  // cases on the moments: their tiles; they come first in the work lists above,
  // nmu_mom and ncoll_mom items of them
  Item* d_tiles = nullptr;
  MomWork work{};
  int grid_mom = 0, nmu_mom = 0, ncoll_mom = 0, nline_mom = 0;
  bool populations = false;  // lbm_batch_autotune: every case on the populations
  std::vector<int> case_order;  // split path: cases in work-list order
  // compact-scheme cases: their mu tiles (TXB x TYB), their line groups
  // (rebuilt with the group size lpb of the tile shape), longest line
  bool compact = false;
  Item* d_cmu = nullptr;
  int ncmu = 0;
  Item* d_litems = nullptr;
  int nline = 0, line_cap = 0, lpb = 8, lpb_shift = 3, lmax = 0;
  std::vector<std::pair<void*, size_t>> blocks;
};

// line groups of the compact cases for groups of lpb lines: code = group * 4
// + 2 axis + field (field 0: mu, 1: rho)
static int build_line_items(lbm_batch* b, int lpb) {
  int sh = 0;
  while ((1 << sh) < lpb) ++sh;
  std::vector<Item> li;
  for (const int c : b->case_order) {
    const CaseDev& cd = b->host_cases[c];
    if (!cd.lap) continue;
    for (int axis = 0; axis < 2; ++axis) {
      const int lines = axis == 0 ? b->p[c].ny : b->p[c].nx;
      const int groups = (lines + lpb - 1) / lpb;
      for (int g = 0; g < groups; ++g)
        for (int field = 0; field < 2; ++field) li.push_back({c, g * 4 + 2 * axis + field});
    }
    if (cd.mom) b->nline_mom = int(li.size());
  }
  if (int(li.size()) > b->line_cap) return LBM_ECUDA;
  if (!li.empty() && cudaMemcpyAsync(b->d_litems, li.data(), sizeof(Item) * li.size(), cudaMemcpyHostToDevice,
                                     b->stream) != cudaSuccess)
    return LBM_ECUDA;
  if (cudaStreamSynchronize(b->stream) != cudaSuccess) return LBM_ECUDA;
  b->nline = int(li.size());
  b->lpb = lpb;
  b->lpb_shift = sh;
  return LBM_OK;
}

static void* balloc(lbm_batch* b, size_t bytes) {
  void* p = b->alloc.alloc(bytes ? bytes : 256, b->alloc.ctx);
  if (p) b->blocks.push_back({p, bytes ? bytes : 256});
  return p;
}
static void cuda_free_b(void* p, size_t, void*) { cudaFree(p); }

extern "C" void lbm_batch_destroy(lbm_batch* b) {
  if (!b) return;
  cudaStreamSynchronize(b->stream);
  if (b->gexec) cudaGraphExecDestroy(b->gexec);
  if (b->graph) cudaGraphDestroy(b->graph);
  for (auto& blk : b->blocks) b->alloc.free(blk.first, blk.second, b->alloc.ctx);
  delete b;
}

template <int RPT>
static int setup_split_t(lbm_batch* b) {
  constexpr int M2Y = Tile2<RPT>::M2Y, T2Y = Tile2<RPT>::T2Y;
  std::vector<Item> mitems, citems;
  for (const int c : b->case_order) {
    const CaseDev& cd = b->host_cases[c];
    const int ny = b->p[c].ny;
    const int mt = cd.mtiles_x * ((ny + M2Y - 1) / M2Y);
    const int ct = cd.ctiles_x * ((ny + T2Y - 1) / T2Y);
    for (int tl = 0; tl < mt; ++tl) mitems.push_back({c, tl});
    for (int tl = 0; tl < ct; ++tl) citems.push_back({c, tl});
    if (cd.mom) {
      b->nmu_mom = int(mitems.size());
      b->ncoll_mom = int(citems.size());
    }
  }
  if (int(mitems.size()) > b->item_cap || int(citems.size()) > b->item_cap) return LBM_ECUDA;
  cudaError_t e = cudaMemcpyAsync(b->d_mitems, mitems.data(), sizeof(Item) * mitems.size(), cudaMemcpyHostToDevice,
                                  b->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->d_citems, citems.data(), sizeof(Item) * citems.size(), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return LBM_ECUDA;
  size_t m = Split2DShape<S_EFDS2, RPT>::bytes;
  m = std::max(m, Split2DShape<S_EFDS4, RPT>::bytes);
  m = std::max(m, Split2DShape<S_EFDS6, RPT>::bytes);
  m = std::max(m, Split2DShape<S_E4, RPT>::bytes);
  m = std::max(m, Split2DShape<S_E8, RPT>::bytes);
  if (b->compact) m = std::max(m, Split2DShape<S_CFDS4, RPT>::bytes);
  // compact cases: groups of up to 16 lines (one per warp) whose two float
  // line buffers fit the items' shared memory
  int lpb = 16;
  if (b->compact) {
    while (lpb > 1 && size_t(2) * lpb * (b->lmax + 1) * 4 > NBUF * m) lpb /= 2;
    m = std::max(m, (size_t(2) * lpb * (b->lmax + 1) * 4 + NBUF - 1) / NBUF);
  }
  const int buf = int((m + 15) / 16 * 16);
  const size_t smem = NBUF * size_t(buf);  // items in flight
  int dev = 0, sms = 0, ps = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaFuncSetAttribute(k_batch_split<RPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, k_batch_split<RPT>, NT2S, smem) != cudaSuccess || ps < 1)
    return LBM_ENOTSUP;
  if (b->compact && build_line_items(b, lpb) != LBM_OK) return LBM_ECUDA;
  b->nmu = int(mitems.size());
  b->ncoll = int(citems.size());
  b->buf_split = buf;
  b->smem_split = smem;
  b->grid_split = std::max(1, std::min(ps * sms, std::max(b->nmu, b->ncoll)));
  b->rpt = RPT;
  // the captured launch depends on the shape: capture again at the next step
  if (b->gexec) { cudaGraphExecDestroy(b->gexec); b->gexec = nullptr; }
  if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
  b->graph_steps = -1;
  return LBM_OK;
}

// work lists of the cases on the moments, the dearest schemes' tiles first
static int setup_moments(lbm_batch* b) {
  int dev = 0, sms = 0, ps = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  std::vector<Item> list, cmp[3];
  MomWork& wk = b->work;
  wk = MomWork{};
  for (const int s : {S_E8, S_EFDS6, S_E4, S_EFDS4, S_EFDS2, S_CFDS4})
    for (const int c : b->case_order) {
      const CaseDev& cd = b->host_cases[c];
      if (!cd.mom || (is_compact(cd.scheme) ? int(S_CFDS4) : cd.scheme) != s) continue;
      for (int u = 0; u < cd.mg.nt * cd.mg.nr; ++u) (s == S_CFDS4 ? cmp[2] : list).push_back({c, u});
      if (s != S_CFDS4) continue;
      const int nx = cd.kp.nx, ny = cd.kp.ny;
      for (int u = 0; u < (nx + 63) / 64 * ((ny + 31) / 32); ++u) cmp[0].push_back({c, u});
      const int groups = (ny + IIR_CTA_ROWS - 1) / IIR_CTA_ROWS + (nx + iir_cta_cols_n(ny) - 1) / iir_cta_cols_n(ny);
      for (int g = groups - 1; g >= 0; --g) cmp[1].push_back({c, g});
    }
  if (list.empty() && cmp[2].empty()) return LBM_OK;
  if (cudaFuncSetAttribute(k_batch_mom, cudaFuncAttributeMaxDynamicSharedMemorySize, T2_SMEM) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ps, k_batch_mom, T2NT, T2_SMEM) != cudaSuccess || ps < 1)
    return LBM_ECUDA;
  wk.ntiles = int(list.size());
  const int most = int(list.size() + std::max(cmp[1].size(), cmp[2].size()));
  for (int f = 0; f < 3; ++f) {
    wk.ncmp[f] = int(cmp[f].size());
    list.insert(list.end(), cmp[f].begin(), cmp[f].end());
  }
  b->grid_mom = std::max(1, std::min(ps * sms, most));
  b->d_tiles = static_cast<Item*>(balloc(b, sizeof(Item) * list.size()));
  if (!b->d_tiles) return LBM_ENOMEM;
  wk.tiles = b->d_tiles;
  for (int f = 0, at = wk.ntiles; f < 3; at += wk.ncmp[f++]) wk.cmp[f] = wk.tiles + at;
  if (cudaMemcpyAsync(b->d_tiles, list.data(), sizeof(Item) * list.size(), cudaMemcpyHostToDevice, b->stream) != cudaSuccess ||
      cudaStreamSynchronize(b->stream) != cudaSuccess)
    return LBM_ECUDA;
  return LBM_OK;
}

static int setup_split(lbm_batch* b, int rpt) {
  if (rpt == 1) return setup_split_t<1>(b);
  if (rpt == 2) return setup_split_t<2>(b);
  if (rpt == 4) return setup_split_t<4>(b);
  return LBM_EINVAL;
}

extern "C" int lbm_batch_create(const lbm_params* cases, int n, void* stream, const lbm_allocator* alloc,
                                lbm_batch** out) {
  if (!out || !cases || n < 1) return LBM_EINVAL;
  *out = nullptr;
  const int prec0 = cases[0].precision;
  const int mu0 = cases[0].mu_fp64;
  for (int c = 0; c < n; ++c) {
    const lbm_params& q = cases[c];
    if (q.lattice != LBM_D2Q9 || q.nz != 1 || q.nx < 8 || q.ny < 8) return LBM_EINVAL;
    if (!(q.a > 0 && q.b > 0 && q.R > 0 && q.Tr > 0 && q.k > 0 && q.kappa >= 0 && q.tau > 0.5)) return LBM_EINVAL;
    if (q.precision != prec0 || q.mu_fp64 != mu0 || (q.precision != LBM_FP64 && q.precision != LBM_FP32DEV))
      return LBM_EINVAL;
    if (q.scheme < LBM_EFDS2 || q.scheme > LBM_E8) return LBM_EINVAL;
    if (q.collision != LBM_BGK && q.collision != LBM_MRT) return LBM_EINVAL;
    if (q.eos < LBM_EOS_CS || q.eos > LBM_EOS_RKS) return LBM_EINVAL;
  }
  lbm_batch* b = new (std::nothrow) lbm_batch();
  if (!b) return LBM_ENOMEM;
  b->n = n;
  b->stream = static_cast<cudaStream_t>(stream);
  if (alloc && alloc->alloc && alloc->free) b->alloc = *alloc;
  else { b->alloc.alloc = device_malloc; b->alloc.free = cuda_free_b; b->alloc.ctx = nullptr; }
  b->prec = prec0 == LBM_FP64 ? 0 : (mu0 ? 2 : 1);
  b->p.assign(cases, cases + n);
  b->host_cases.resize(n);
  // work items: cases grouped by scheme, larger cases first (dynamic fetch
  // then ends with small items, which balances the step)
  std::vector<int> idx(n);
  for (int c = 0; c < n; ++c) idx[c] = c;
  std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) {
    if (cases[x].scheme != cases[y].scheme) return cases[x].scheme < cases[y].scheme;
    return (long long)cases[x].nx * cases[x].ny > (long long)cases[y].nx * cases[y].ny;
  });
  std::vector<Item> items, cmu_items;
  const size_t fs = prec0 == LBM_FP64 ? 8 : 4;
  // compact cases: mu type (float only in FP32DEV with FP32 mu), gradient types
  const size_t tm = (prec0 == LBM_FP32DEV && !mu0) ? 4 : 8, tc = prec0 == LBM_FP64 ? 8 : 4;
  long long line_cap = 0;
  bool ok = true;
  for (int k = 0; k < n && ok; ++k) {
    const int c = idx[k];
    const lbm_params& q = cases[c];
    CaseDev& cd = b->host_cases[c];
    if (params_to_kp(&q, &cd.kp) != LBM_OK) { ok = false; break; }
    const long long N = cd.kp.n;
    b->p[c].rho_ref = cd.kp.rho_ref;
    cd.scheme = q.scheme;
    cd.mrt = make_mrt(q.collision == LBM_MRT, q.mrt_s, q.tau);
    cd.tiles_x = (q.nx + TXB - 1) / TXB;
    cd.tiles_y = (q.ny + TYB - 1) / TYB;
    cd.item_begin = int(items.size());
    for (int tl = 0; tl < cd.tiles_x * cd.tiles_y; ++tl) items.push_back({c, tl});
    cd.item_end = int(items.size());
    cd.f[0] = balloc(b, size_t(9) * N * fs);
    cd.f[1] = balloc(b, size_t(9) * N * fs);
    cd.rho[0] = balloc(b, size_t(N) * fs);
    cd.rho[1] = balloc(b, size_t(N) * fs);
    cd.snap = balloc(b, size_t(N) * fs);
    cd.bad = static_cast<unsigned long long*>(balloc(b, 8));
    cd.mu = nullptr;
    cd.mtiles_x = (q.nx + M2X - 1) / M2X;
    cd.ctiles_x = (q.nx + T2X - 1) / T2X;
    if (prec0 == LBM_FP32DEV && !mu0) cd.mu = static_cast<float*>(balloc(b, size_t(N) * 4));
    ok = cd.f[0] && cd.f[1] && cd.rho[0] && cd.rho[1] && cd.snap && cd.bad && (cd.mu || prec0 != LBM_FP32DEV || mu0);
    cd.lap = cd.lci = 0;
    cd.cmu = cd.gmu = cd.grho = nullptr;
    // (compact cases: the fit and tau as for an explicit scheme, lines of at most 512)
    const bool comp = is_compact(q.scheme);
    cd.mom = prec0 == LBM_FP32DEV && !mu0 && (!comp || iir_ok(cd.kp)) &&
             mom2d_ok(cd.kp, comp ? S_EFDS4 : q.scheme, 1, cd.mrt.on != 0);
    cd.mg = Mom2Geo{};
    if (cd.mom) cd.mg = mom2_geo(cd.kp, 1);
    if (ok && q.scheme >= LBM_CFDS4 && q.scheme <= LBM_OCFDS4) {
      b->compact = true;
      cd.lap = q.scheme == LBM_CFDS6 ? 6 : (q.scheme == LBM_CFDS8 ? 8 : 4);
      cd.lci = q.scheme - LBM_CFDS4;
      cd.cmu = cd.mu ? static_cast<void*>(cd.mu) : balloc(b, size_t(N) * tm);
      cd.gmu = balloc(b, size_t(2) * N * tm);
      cd.grho = balloc(b, size_t(2) * N * tc);
      ok = cd.cmu && cd.gmu && cd.grho;
      for (int tl = cd.item_begin; tl < cd.item_end; ++tl) cmu_items.push_back(items[tl]);
      line_cap += 2LL * (q.nx + q.ny);
      b->lmax = std::max(b->lmax, std::max(q.nx, q.ny));
    }
  }
  if (!ok) { lbm_batch_destroy(b); return LBM_ENOMEM; }
  b->nitems = int(items.size());
  b->split = prec0 == LBM_FP32DEV && !mu0;
  std::stable_partition(idx.begin(), idx.end(), [&](int c) { return b->host_cases[c].mom != 0; });
  b->case_order.assign(idx.begin(), idx.end());
  if (const int rm = setup_moments(b); rm != LBM_OK) { lbm_batch_destroy(b); return rm; }
  if (b->compact) {
    // the line coefficients of the four compact schemes (the same for every batch)
    LineCoef lc[2][4];
    for (int j = 0; j < 4; ++j) {
      const LineCoef full = make_line_coef(S_CFDS4 + j);
      lc[0][j] = line_coef_for(full, false);
      lc[1][j] = line_coef_for(full, true);
    }
    b->ncmu = int(cmu_items.size());
    b->line_cap = int(line_cap);
    b->d_cmu = static_cast<Item*>(balloc(b, sizeof(Item) * cmu_items.size()));
    b->d_litems = static_cast<Item*>(balloc(b, sizeof(Item) * line_cap));
    if (!b->d_cmu || !b->d_litems ||
        cudaMemcpyToSymbolAsync(c_lines, lc, sizeof(lc), 0, cudaMemcpyHostToDevice, b->stream) != cudaSuccess ||
        cudaMemcpyAsync(b->d_cmu, cmu_items.data(), sizeof(Item) * cmu_items.size(), cudaMemcpyHostToDevice,
                        b->stream) != cudaSuccess) {
      lbm_batch_destroy(b);
      return LBM_ECUDA;
    }
    // the persistent kernel of FP64 (and FP64-mu) batches: groups of 8 lines
    if (!b->split && build_line_items(b, 8) != LBM_OK) { lbm_batch_destroy(b); return LBM_ECUDA; }
  }
  if (b->split) {
    // work lists are rebuilt per tile shape; the shortest tiles (one row per
    // thread) give the longest lists
    long long cap = 0;
    for (int k = 0; k < n; ++k) {
      const int c = idx[k];
      const CaseDev& cd = b->host_cases[c];
      cap += (long long)std::max(cd.mtiles_x * ((cases[c].ny + Tile2<1>::M2Y - 1) / Tile2<1>::M2Y),
                                 cd.ctiles_x * ((cases[c].ny + Tile2<1>::T2Y - 1) / Tile2<1>::T2Y));
    }
    b->item_cap = int(cap);
    b->d_mitems = static_cast<Item*>(balloc(b, sizeof(Item) * cap));
    b->d_citems = static_cast<Item*>(balloc(b, sizeof(Item) * cap));
    if (!b->d_mitems || !b->d_citems) { lbm_batch_destroy(b); return LBM_ENOMEM; }
  }
  b->d_cases = static_cast<CaseDev*>(balloc(b, sizeof(CaseDev) * n));
  b->d_items = static_cast<Item*>(balloc(b, sizeof(Item) * items.size()));
  b->ctl = static_cast<BatchCtl*>(balloc(b, sizeof(BatchCtl)));
  b->d_partials = static_cast<double*>(balloc(b, size_t(4) * 8 * items.size()));
  b->d_out = static_cast<double*>(balloc(b, size_t(8) * 8 * n));
  if (!b->d_cases || !b->d_items || !b->ctl || !b->d_partials || !b->d_out) { lbm_batch_destroy(b); return LBM_ENOMEM; }
  BatchCtl c0{};
  c0.skip_block = -1;
  cudaError_t e = cudaMemcpyAsync(b->d_cases, b->host_cases.data(), sizeof(CaseDev) * n, cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->d_items, items.data(), sizeof(Item) * items.size(), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->ctl, &c0, sizeof(c0), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  // residency: CTAs per SM x SMs, all resident at once
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  auto setup = [&](auto kern, size_t smem) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT2, smem);
  };
  // line groups of 8 lines of 8-byte values beside the step tiles (compact cases)
  const size_t line_bytes = b->compact ? size_t(2) * 8 * (b->lmax + 1) * 8 : 0;
  if (b->prec == 0) { b->smem = std::max(batch_smem<PrecF64>(), line_bytes); setup(k_batch_persistent<PrecF64>, b->smem);
                      cudaFuncSetAttribute(k_batch_obs<PrecF64>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(b->smem)); }
  else if (b->prec == 1) { b->smem = std::max(batch_smem<PrecF32>(), line_bytes); setup(k_batch_persistent<PrecF32>, b->smem);
                           cudaFuncSetAttribute(k_batch_obs<PrecF32>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(b->smem)); }
  else { b->smem = std::max(batch_smem<PrecF32M64>(), line_bytes); setup(k_batch_persistent<PrecF32M64>, b->smem);
         cudaFuncSetAttribute(k_batch_obs<PrecF32M64>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(b->smem)); }
  b->grid = std::max(1, std::min(per_sm * sms, b->nitems));
  if (b->split && e == cudaSuccess && setup_split(b, RPT_DEFAULT) != LBM_OK) {
    lbm_batch_destroy(b);
    return LBM_ECUDA;
  }
  if (e != cudaSuccess || per_sm < 1 || cudaGetLastError() != cudaSuccess) { lbm_batch_destroy(b); return LBM_ECUDA; }
  *out = b;
  return LBM_OK;
}

namespace {
__constant__ double cb_w9[9] = {4.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 9, 1.0 / 36, 1.0 / 36, 1.0 / 36, 1.0 / 36};

// Eq. 26 droplet centred at node (nx/2, ny/2) for every case; f_i = w_i rho
template <typename Tf>
__global__ void k_batch_init(const CaseDev* __restrict__ cases, const double* radius, const double* rl,
                             const double* rg, double width) {
  const int c = blockIdx.y;
  const CaseDev& cd = cases[c];
  for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < cd.kp.n; n += (long long)gridDim.x * blockDim.x) {
    const int x = int(n % cd.kp.nx), y = int(n / cd.kp.nx);
    const double dx = x - double(cd.kp.nx / 2), dy = y - double(cd.kp.ny / 2);
    const double r = sqrt(dx * dx + dy * dy);
    const double r0 = 0.5 * (rl[c] + rg[c]) - 0.5 * (rl[c] - rg[c]) * tanh(2.0 * (r - radius[c]) / width);
    Tf* f = static_cast<Tf*>(cd.f[0]);
    Tf* rho = static_cast<Tf*>(cd.rho[0]);
    Tf* snap = static_cast<Tf*>(cd.snap);
    if constexpr (sizeof(Tf) == 8) {
      double acc = 0;
      for (int i = 0; i < 9; ++i) { const double fi = cb_w9[i] * r0; f[i * cd.kp.n + n] = fi; acc += fi; }
      rho[n] = acc;
    } else {
      FSum acc;
      for (int i = 0; i < 9; ++i) { const float d = float(cb_w9[i] * (r0 - cd.kp.rho_ref)); f[i * cd.kp.n + n] = d; acc.add(d); }
      rho[n] = acc.fvalue();
    }
    snap[n] = rho[n];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *cd.bad = ULLONG_MAX;
}
}  // namespace

extern "C" int lbm_batch_init_droplets(lbm_batch* b, const double* radius, double width) {
  if (!b || !radius || !(width > 0)) return LBM_EINVAL;
  std::vector<double> host(3 * size_t(b->n));
  long long maxn = 0;
  for (int c = 0; c < b->n; ++c) {
    double g, l;
    if (!(radius[c] >= 0) || lbm_maxwell(&b->p[c], &g, &l) != LBM_OK) return LBM_EINVAL;
    host[c] = radius[c];
    host[b->n + c] = l;
    host[2 * b->n + c] = g;
    maxn = std::max(maxn, (long long)b->p[c].nx * b->p[c].ny);
  }
  double* d = static_cast<double*>(b->alloc.alloc(host.size() * 8, b->alloc.ctx));
  if (!d) return LBM_ENOMEM;
  cudaError_t e = cudaMemcpyAsync(d, host.data(), host.size() * 8, cudaMemcpyHostToDevice, b->stream);
  dim3 grid(unsigned(std::min<long long>((maxn + 255) / 256, 1024)), unsigned(b->n));
  if (e == cudaSuccess) {
    if (b->prec == 0) k_batch_init<double><<<grid, 256, 0, b->stream>>>(b->d_cases, d, d + b->n, d + 2 * b->n, width);
    else k_batch_init<float><<<grid, 256, 0, b->stream>>>(b->d_cases, d, d + b->n, d + 2 * b->n, width);
    e = cudaGetLastError();
  }
  BatchCtl c0{};
  c0.skip_block = -1;
  if (e == cudaSuccess) e = cudaMemcpyAsync(b->ctl, &c0, sizeof(c0), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  b->alloc.free(d, host.size() * 8, b->alloc.ctx);
  b->t = 0;
  b->t_snap = 0;
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

// the split kernel over all cases, or over those not on the moments
static cudaError_t launch_split(lbm_batch* b, int nsteps, bool all) {
  cudaLaunchConfig_t cs{};
  cs.gridDim = dim3(unsigned(b->grid_split));
  cs.blockDim = dim3(NT2S);
  cs.dynamicSmemBytes = b->smem_split;
  cs.stream = b->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cs.attrs = at;
  cs.numAttrs = 1;
  auto kern = b->rpt == 1 ? k_batch_split<1> : (b->rpt == 4 ? k_batch_split<4> : k_batch_split<2>);
  const int m0 = all ? 0 : b->nmu_mom, c0 = all ? 0 : b->ncoll_mom, l0 = all ? 0 : b->nline_mom;
  return cudaLaunchKernelEx(&cs, kern, (const CaseDev*)b->d_cases, (const Item*)b->d_mitems + m0, b->nmu - m0,
                            (const Item*)b->d_citems + c0, b->ncoll - c0, nsteps, b->ctl, BARRIER_NS, b->buf_split,
                            (const Item*)b->d_litems + l0, b->nline - l0, b->lpb, b->lpb_shift);
}

// nsteps steps of every case: on the populations in one persistent launch, or,
// with cases that advance on their moments, an odd step on the populations, then
// the moments' launch and the remaining cases'
static cudaError_t launch_persistent(lbm_batch* b, int nsteps) {
  const unsigned long long timeout_ns = BARRIER_NS;
  // counters and barrier state (status and skip_block are left as they are)
  auto reset = [&] { return cudaMemsetAsync(b->ctl, 0, offsetof(BatchCtl, status), b->stream); };
  cudaError_t e = reset();
  if (e != cudaSuccess) return e;
  if (b->split) {
    const int even = b->work.tiles && !b->populations ? nsteps / 2 * 2 : 0;
    if (nsteps - even > 0 && (e = launch_split(b, nsteps - even, true)) != cudaSuccess) return e;
    if (even == 0) return e;
    const bool rest = b->nmu > b->nmu_mom;
    cudaLaunchConfig_t cs{};
    cs.gridDim = dim3(unsigned(b->grid_mom));
    cs.blockDim = dim3(T2NT);
    cs.dynamicSmemBytes = T2_SMEM;
    cs.stream = b->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cs.attrs = at;
    cs.numAttrs = 1;
    if ((e = reset()) != cudaSuccess) return e;
    IirAll ia;
    for (int k = 0; k < 4; ++k) ia.k[k] = iir_coef(S_CFDS4 + k);
    e = cudaLaunchKernelEx(&cs, k_batch_mom, (const CaseDev*)b->d_cases, b->work, even, b->ctl, timeout_ns, rest ? 0 : 1, ia);
    if (e != cudaSuccess || !rest) return e;
    if ((e = reset()) != cudaSuccess) return e;
    return launch_split(b, even, false);
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(b->grid));
  cfg.blockDim = dim3(NT2);
  cfg.dynamicSmemBytes = b->smem;
  cfg.stream = b->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const Item* cmu = b->d_cmu;
  const Item* li = b->d_litems;
  if (b->prec == 0)
    return cudaLaunchKernelEx(&cfg, k_batch_persistent<PrecF64>, (const CaseDev*)b->d_cases, (const Item*)b->d_items,
                              b->nitems, nsteps, b->ctl, timeout_ns, cmu, b->ncmu, li, b->nline, b->lpb, b->lpb_shift);
  if (b->prec == 1)
    return cudaLaunchKernelEx(&cfg, k_batch_persistent<PrecF32>, (const CaseDev*)b->d_cases, (const Item*)b->d_items,
                              b->nitems, nsteps, b->ctl, timeout_ns, cmu, b->ncmu, li, b->nline, b->lpb, b->lpb_shift);
  return cudaLaunchKernelEx(&cfg, k_batch_persistent<PrecF32M64>, (const CaseDev*)b->d_cases, (const Item*)b->d_items,
                            b->nitems, nsteps, b->ctl, timeout_ns, cmu, b->ncmu, li, b->nline, b->lpb, b->lpb_shift);
}

// n steps = one persistent launch, two or three with cases on their moments
// (each preceded by the reset of the barrier and work counters), captured once in a CUDA graph per distinct n and replayed
extern "C" int lbm_batch_step(lbm_batch* b, long long n) {
  if (!b || n < 0 || n > INT_MAX) return LBM_EINVAL;
  if (n == 0) return LBM_OK;
  if (b->graph_steps != n) {
    if (b->gexec) { cudaGraphExecDestroy(b->gexec); b->gexec = nullptr; }
    if (b->graph) { cudaGraphDestroy(b->graph); b->graph = nullptr; }
    cudaStream_t cap;
    if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) return LBM_ECUDA;
    cudaStream_t saved = b->stream;
    b->stream = cap;
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
      const cudaError_t el = launch_persistent(b, int(n));
      e = cudaStreamEndCapture(cap, &b->graph);
      if (e == cudaSuccess) e = el;
    }
    b->stream = saved;
    cudaStreamDestroy(cap);
    if (e != cudaSuccess) return LBM_ECUDA;
    if (cudaGraphInstantiate(&b->gexec, b->graph, 0) != cudaSuccess) return LBM_ECUDA;
    b->graph_steps = n;
  }
  if (cudaGraphLaunch(b->gexec, b->stream) != cudaSuccess) return LBM_ECUDA;
  b->t += n;
  return LBM_OK;
}

extern "C" int lbm_batch_set_tiles(lbm_batch* b, int rows) {
  if (!b || (rows != 1 && rows != 2 && rows != 4)) return LBM_EINVAL;
  if (!b->split) return LBM_ENOTSUP;
  return setup_split(b, rows);
}

extern "C" int lbm_batch_autotune(lbm_batch* b, int steps, int* rows_out) {
  if (!b || steps < 1 || steps > 100000) return LBM_EINVAL;
  if (rows_out) *rows_out = b->rpt;
  if (!b->split) return LBM_OK;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return LBM_ECUDA;
  if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return LBM_ECUDA; }
  // three interleaved rounds, each shape's fastest launch counting: shapes
  // a few percent apart are otherwise ordered by noise and by the state each
  // launch happens to step through
  const int shapes[3] = {1, 2, 4};
  float shape_ms[3] = {1e30f, 1e30f, 1e30f};
  int rc = LBM_OK;
  // where every case advances on its moments, only odd steps run on the tiles that
  // are tuned: all of the timed ones do
  b->populations = b->nmu == b->nmu_mom;
  for (int round = 0; round < 3 && rc == LBM_OK; ++round) {
    for (int j = 0; j < 3; ++j) {
      if (setup_split(b, shapes[j]) != LBM_OK) continue;  // shape without a resident configuration
      if ((rc = lbm_batch_step(b, steps)) != LBM_OK) break;  // capture and warm up
      cudaEventRecord(e0, b->stream);
      if ((rc = lbm_batch_step(b, steps)) != LBM_OK) break;
      cudaEventRecord(e1, b->stream);
      if (cudaEventSynchronize(e1) != cudaSuccess) { rc = LBM_ECUDA; break; }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      shape_ms[j] = std::min(shape_ms[j], ms);
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  b->populations = false;
  b->graph_steps = -1;
  if (rc != LBM_OK) return rc;
  int best = 0;
  float best_ms = 1e30f;
  for (int j = 0; j < 3; ++j)
    if (shape_ms[j] < best_ms) { best_ms = shape_ms[j]; best = shapes[j]; }
  if (best == 0) return LBM_ECUDA;
  if ((rc = setup_split(b, best)) != LBM_OK) return rc;
  if (rows_out) *rows_out = best;
  return LBM_OK;
}

// compact cases: mu and derivative fields of the current state
template <class P>
static cudaError_t compact_fields(lbm_batch* b) {
  if (!b->compact) return cudaSuccess;
  const size_t lb = size_t(2) * b->lpb * (b->lmax + 1) * 8;
  if (cudaError_t e = ensure_smem(k_batch_clines<P>, lb); e != cudaSuccess) return e;
  if (b->ncmu > 0) k_batch_cmu<P><<<b->ncmu, NT2, 0, b->stream>>>(b->d_cases, b->d_cmu, b->ctl);
  if (b->nline > 0)
    k_batch_clines<P><<<b->nline, NT2, lb, b->stream>>>(b->d_cases, b->d_litems, b->ctl, b->lpb, b->lpb_shift);
  return cudaGetLastError();
}

extern "C" int lbm_batch_observables(lbm_batch* b, lbm_obs* out) {
  if (!b || !out) return LBM_EINVAL;
  cudaError_t e = b->prec == 0 ? compact_fields<PrecF64>(b)
                               : (b->prec == 1 ? compact_fields<PrecF32>(b) : compact_fields<PrecF32M64>(b));
  if (e != cudaSuccess) return LBM_ECUDA;
  if (b->prec == 0) k_batch_obs<PrecF64><<<b->nitems, NT2, b->smem, b->stream>>>(b->d_cases, b->d_items, b->ctl, b->d_partials);
  else if (b->prec == 1) k_batch_obs<PrecF32><<<b->nitems, NT2, b->smem, b->stream>>>(b->d_cases, b->d_items, b->ctl, b->d_partials);
  else k_batch_obs<PrecF32M64><<<b->nitems, NT2, b->smem, b->stream>>>(b->d_cases, b->d_items, b->ctl, b->d_partials);
  k_batch_obs_final<<<b->n, 256, 0, b->stream>>>(b->d_cases, b->ctl, b->d_partials, b->d_out, b->prec != 0);
  if (b->prec == 0) k_batch_snap<double><<<dim3(64, unsigned(b->n)), 256, 0, b->stream>>>(b->d_cases, b->ctl);
  else k_batch_snap<float><<<dim3(64, unsigned(b->n)), 256, 0, b->stream>>>(b->d_cases, b->ctl);
  e = cudaGetLastError();
  std::vector<double> host(size_t(8) * b->n);
  BatchCtl hc{};
  if (e == cudaSuccess) e = cudaMemcpyAsync(host.data(), b->d_out, host.size() * 8, cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, b->ctl, sizeof(hc), cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return LBM_ECUDA;
  int rc = LBM_OK;
  for (int c = 0; c < b->n; ++c) {
    const double* o = host.data() + 8 * c;
    lbm_obs& r = out[c];
    r.max_v = o[0]; r.max_u = o[1]; r.mass = o[2];
    r.max_drho = b->t > b->t_snap ? o[3] / double(b->t - b->t_snap) : 0.0;
    r.rho_center = o[4]; r.rho_corner = o[5];
    unsigned long long bad;
    std::memcpy(&bad, &o[6], 8);
    r.step = b->t;
    r.status = LBM_OK;
    if (bad != ULLONG_MAX) { r.status = LBM_EUNSTABLE; r.step = (long long)bad; }
    if (hc.status != 0) r.status = hc.status;
  }
  b->t_snap = b->t;
  if (hc.status != 0) rc = hc.status;
  return rc;
}

extern "C" int lbm_batch_get_density(lbm_batch* b, int c, double* host) {
  if (!b || !host || c < 0 || c >= b->n) return LBM_EINVAL;
  const CaseDev& cd = b->host_cases[c];
  const size_t n = size_t(cd.kp.n);
  cudaError_t e;
  if (b->prec == 0) {
    e = cudaMemcpyAsync(host, cd.rho[b->t & 1], n * 8, cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
  }
  std::vector<float> tmp(n);
  e = cudaMemcpyAsync(tmp.data(), cd.rho[b->t & 1], n * 4, cudaMemcpyDeviceToHost, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  for (size_t i = 0; i < n; ++i) host[i] = cd.kp.rho_ref + double(tmp[i]);
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

extern "C" long long lbm_batch_get_step(const lbm_batch* b) { return b ? b->t : -1; }

// CTAs of the batch's launches (the smallest, where there are two kinds)
static int resident(const lbm_batch* b) {
  const int g = b->split ? b->grid_split : b->grid;
  return b->work.tiles ? std::min(g, b->grid_mom) : g;
}

extern "C" int lbm_batch_inject_stall(lbm_batch* b, int cta) {
  if (!b || cta < -1 || cta >= resident(b)) return LBM_EINVAL;
  cudaError_t e = cudaMemcpyAsync(&b->ctl->skip_block, &cta, sizeof(int), cudaMemcpyHostToDevice, b->stream);
  int zero = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&b->ctl->status, &zero, sizeof(int), cudaMemcpyHostToDevice, b->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
  return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}

extern "C" int lbm_batch_size(const lbm_batch* b, int* ncases, int* nitems, int* grid) {
  if (!b) return LBM_EINVAL;
  if (ncases) *ncases = b->n;
  if (nitems) *nitems = (b->split ? b->nmu + b->ncoll : b->nitems + b->ncmu) + b->nline;
  if (grid) *grid = resident(b);
  return LBM_OK;
}
