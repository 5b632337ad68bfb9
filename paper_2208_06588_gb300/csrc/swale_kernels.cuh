// Device side of the GB300 (sm_103a) FP64 solver for the well-balanced ALE-WENO hybrid scheme
// (Zhang, Xia & Xu, arXiv 2208.06588): data layout and the stage kernels.
//
// One SSP-RK3 step (Eq. RK32D) is a fixed sequence of launches on one stream:
//   k_prologue                 per-instance scalar resets
//   [k_mesh_gauss]             fluid-driven node velocities
//   k_recon<1>, k_update<1>    stage 1 on the mesh at t_n
//   k_recon<2>, k_update<2>    stage 2 on the mesh at t_{n+1}
//   k_recon<3>, k_update<3>    stage 3 on the mesh at t_{n+1/2}
//   k_commit                   the step's time and step count, or its roll-back after an error
// (A mesh of few blocks runs whole steps in one launch instead: k_steps in swale_steps.cuh. Between steps of one
// sequence k_commit does the next step's prologue as well.)
// Every launch serves all instances of a batch: blocks walk a work list of (instance, tile)
// entries in grid-stride order (one pass when the grid has one block per tile, a persistent
// loop when it is smaller). A single instance uses the implicit list t -> (0, t * T + first).
// The reconstruction also reduces the per-instance global wave speed of Eq. alpha2D (warp
// shuffle, shared memory, one atomicMax per tile on the order-preserving bit pattern of a
// non-negative double); in stage 1 the last tile of each instance computes that instance's
// dt, so dt, alpha and t never visit the host and steps replay as CUDA graphs.
//
// Error contract: an error bit (kErrBits) raised in a step stops the instance. Kernels skip an
// instance whose status holds one; the stage-3 update writes q^{n+1}, J^{n+1} and the nodes only
// if no error was raised before it (keeping q^n, J^n and x^n in backup arrays), and k_commit
// restores them if the stage-3 update itself raised one. The state is then that of the last
// good step; later steps (also inside a captured graph) are no-ops for the instance.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/swale.h"
#include "swale_cell.cuh"

namespace swale_dev {

using swale::EdgeState;
using swale::SchemeConst;

constexpr int kMaxGaussHalf = 64;
// Resident threads per SM that the launch bounds of the stage kernels ask for (72 registers a thread; 640 to
// 1024 threads are within 1 %).
constexpr int kReconThreads = 896, kUpdateThreads = 896;
constexpr int kMeshThreads = 256;
constexpr int kMeshNodes = kMeshThreads - 1;  // nodes a mesh-velocity tile advances by
constexpr double kTwoPi = 6.283185307179586476925286766559;  // (the host's bound on the node speeds)

// Per-instance device scalars. Maxima of non-negative doubles are kept as their bit patterns
// (unsigned order equals numeric order for non-negative IEEE doubles).
struct DevScalars {
  double t, dt, sdiff, Wbar, alpha1;
  unsigned int st3;                  // status bits raised by the stage-3 update (folded by k_commit)
  unsigned int pad_;
  unsigned long long A[3];           // max edge wave speed per stage
  unsigned long long Jmax[3];        // max width of the stage meshes J^n, J^(1), J^(2)
  unsigned long long Jmin0;          // min J^n
  unsigned long long JmaxN, JminN;   // of J^{n+1} (the minimum accumulated by stage 1)
  unsigned long long Wabs, dWabs;    // fluid-driven motion: max |w|, max |w_{j+1} - w_j|
  long long steps;
  long long step_idx;                // index of the step in progress (set by the prologue)
  unsigned int status;
  unsigned int counter;              // reconstruction tiles finished in stage 1
  int done;
  int clipped;
  // Mesh cache: stage 2 stores the mesh-only values (GEO_*) of the t_{n+1} mesh, which the next
  // step's stage 1 reuses when the tag (context epoch, step index) matches.
  unsigned long long geo_tag;
};

// Per-instance constants.
struct InstConst {
  int64_t N;           // cells
  int64_t coff;        // first cell in the concatenated cell arrays (nodes: coff + i,
                       // edge arrays: coff + 2 i)
  double cfl;
  double Wbar_profile; // (2 pi / T) max |P| of the prescribed motion
  int32_t ntiles_r;    // forward reconstruction tiles of the instance
  int32_t pad_;
};

struct Tile {
  int32_t inst, c0;  // instance and first cell (reconstruction tiles start at cell -1)
};

// Constants of the whole launch.
struct StepConst {
  SchemeConst sc;
  double t_end, dt_fixed, mesh_T, inv_T;
  double gauss_iwsum;  // reciprocal of the full Gaussian window's sum (from -H to H)
  int32_t bc, mesh, gauss_half, B;
  // Stage viscosities: log of 3 values per step and instance (index (step * B + i) * 3 + s - 1);
  // alpha_mode 1 records the computed values, 2 replays the logged ones (the adjoint's and the
  // finite-difference checks' convention: alpha held fixed).
  double* alpha_log;
  int64_t alpha_cap;   // steps the log holds
  int64_t alpha_base;  // step counter value of log row 0
  int32_t alpha_mode;
  int32_t scheme;  // SWALE_SCHEME_*
  uint32_t geo_epoch;  // bumped by the host whenever the state is set or restored
  // Wave speeds of alpha (Eq. alpha2D): 1 = relative to the node velocity, |u - w| + sqrt(g h)
  // (w known when the stage runs), 0 = |u| + sqrt(g h), with the step bound Wbar of |w| added to
  // the maximum (stage 1 of the secant motion, whose w depends on dt; or on request).
  int32_t wave_rel;
  // L2-projection bottom (Eq. baverage); bot_pieces == 0: b evolves by Eq. bottomrk.
  int32_t bot_pieces, bot_deg;
  const double* bot_breaks;  // bot_pieces + 1 breakpoints
  const double* bot_coef;    // piece p: sum_k bot_coef[p (bot_deg + 1) + k] (x - break_p)^k
  // Bounded waits for bulk copies: polls before a wait gives up, and bytes expected beyond the
  // copies (0; swale_set_wait_test raises it so that the waits run out, to test that path).
  int32_t wait_tries;
  uint32_t tx_pad;
  int32_t barrier_tries;  // polls of a grid-wide wait of k_steps
};

// Stage viscosity of instance i in stage s of step `step` (DevScalars::step_idx): the computed
// value, or the logged one in replay mode; recorded in record mode.
__device__ __forceinline__ double stage_alpha(const StepConst& K, int i, int s, double computed, long long step) {
  step -= K.alpha_base;
  if (K.alpha_mode == 0 || K.alpha_log == nullptr || step < 0 || step >= K.alpha_cap) return computed;
  double* slot = K.alpha_log + ((int64_t)step * K.B + i) * 3 + (s - 1);
  if (K.alpha_mode == 2) return *slot;
  *slot = computed;
  return computed;
}

// Mesh-only values that stage 2 keeps for the next step's stage 1, which runs on the same mesh: the
// reciprocal sums of the widths (see k_recon) and the source term's ratios (per interface, at the
// edge index of its left cell, and per cell).
enum { GEO_IP, GEO_IT, GEO_IQ, GEO_IV, GEO_RHO, GEO_SIG, GEO_RHO2, GEO_SIG2, GEO_GX, GEO_GY, GEO_K3, GEO_ARRAYS };

// Weights exp(-m^2 / 2 sigma^2), m = -H..H, of a configuration's filter, and the same times 2^56.
struct GaussTable {
  double w[2 * kMaxGaussHalf + 1];
  swale::Limbs q[2 * kMaxGaussHalf + 1];
  long long need;  // filter_need of q
};

// Device arrays of a batch (concatenated over instances).
struct DevState {
  double *E0, *M0, *B0;        // q^n (updated in place by stage 3)
  double *Ea, *Ma, *Ba;        // q^(1)
  double *Eb, *Mb, *Bb;        // q^(2)
  double *YE, *YM, *YB;        // running RK combination J q
  double *J0, *J1, *J2;        // J^n, J^(1), J^(2)
  double *x, *w, *P;           // nodes, node velocities, motion profile (N_i + 1 per instance)
  // Edge arrays hold cells -1..N_i of each instance (N_i + 2 per instance).
  double *eEL, *eER, *eBL, *eBR, *ehL, *ehR, *euL, *euR;
  double *ipair, *itri;        // 1/(J_c + J_{c+1}) and 1/(J_{c-1} + J_c + J_{c+1}) of the stage mesh
  double* xn;                  // nodes at t_{n+1}, written by stage 2 (L2-projection bottom only)
  // Backups of q^n, J^n (cells) and x^n (nodes) written by the stage-3 update before it commits
  // the step, restored by k_commit if that update raised an error (null: no roll-back).
  double *bE, *bM, *bB, *bJ, *bx;
  double *eG1, *eG2;           // interior Gauss-Lobatto points of eta, as smooth_points has them (special source scheme only)
  // Mesh cache: GEO_ARRAYS arrays in the edge layout, geo[k * geo_stride + idx] (null: every stage forms
  // these values, bit for bit the same).
  double* geo;
  int64_t geo_stride;
  // Per cell of the stage input in the edge layout, written by the reconstruction for the update of
  // the same stage: differences of eta and h to the next cell, and the depth.
  double *dE, *dH, *H;
  double *iJ1, *iJ2;           // 1 / J^(1), 1 / J^(2) (cells)
  // What the reverse of a stage reads besides the edge states, arrays in the edge layout
  // (gK[k * geo_stride + idx], ADJ_*); set only for the adjoint's recomputes, which store them.
  double* gK;
  uint8_t* flags;              // stage-1 classes, edge layout
  GaussTable* gauss;           // fluid-driven motion
  InstConst* IC;
  DevScalars* S;
  const Tile* mtiles;  // work lists (null: one instance, implicit tiles)
  int32_t nm;          // tiles in each list
  // The forward update's tiles: T - 1 cells for a block of T threads, so that its T interfaces
  // take one pass.
  const Tile* ftiles;
  int32_t nf;
  // The forward reconstruction's tiles: T - 4 cells for a block of T threads.
  const Tile* rftiles;
  int32_t nrf;
  InstConst ic1;  // the constants of a single instance (the stage kernels need no load for them)
};

// Status bits that stop an instance (SWALE_BIT_NEGDEPTH is a warning).
constexpr unsigned int kErrBits =
    swale::ST_EWEIGHT | swale::ST_NONFINITE | swale::ST_EMESH | swale::ST_NODT | swale::ST_TIMEOUT;

// Whether the mesh cache holds the values of stage STAGE's mesh: that of the step before's stage 2 is the
// mesh of this step's stage 1; a static mesh has one for all stages of all later steps.
template <int STAGE>
__device__ __forceinline__ bool cached_mesh(const StepConst& K, const DevState& D, const DevScalars* S) {
  if (!D.geo || (STAGE != 1 && K.mesh != SWALE_MESH_STATIC)) return false;
  const unsigned long long tag = S->geo_tag;
  if ((unsigned)(tag >> 32) != K.geo_epoch) return false;
  const int ahead = (int)((unsigned)S->step_idx - (unsigned)tag);
  return K.mesh == SWALE_MESH_STATIC ? ahead >= 0 : ahead == 0;
}

// An instance takes no further part in the step: finished (t_end), or an error was raised.
__device__ __forceinline__ bool inst_idle(const DevScalars* S) {
  return S->done || (*(volatile const unsigned int*)&S->status & kErrBits);
}

// Node velocity array of a batch: the motion profile itself for the linear motion (constant
// node velocities), else the node-velocity array (zero for a static mesh).
__device__ __forceinline__ const double* node_velocities(const StepConst& K, const DevState& D) {
  return K.mesh == SWALE_MESH_LINEAR ? D.P : D.w;
}

__device__ __forceinline__ int32_t ghost(int32_t i, int32_t N, int bc) {
  if (i >= 0 && i < N) return i;
  if (bc == SWALE_BC_PERIODIC) {
    i %= N;
    return i < 0 ? i + N : i;
  }
  return i < 0 ? -1 - i : N - 1 - (i - N);
}

// L2 projection of the bottom onto one cell [a, c] (Eq. baverage): on each piece the cell
// overlaps (the first found by bisection of the breakpoints), the mean of the polynomial by the
// 5-point Gauss-Legendre rule, exact for degree <= 8, taken about the middle value so that constants
// come out exact; the cell average weights these means by the overlap lengths.
// (Differences of antiderivatives would cancel on short cells far from the breakpoint.)
// A cell within one piece (nearly all of them) takes the mean as the middle value plus the weighted
// differences from it, with no division, and a constant piece its value. (With a division per
// piece and cell and the constants copied to the stack, the projected bottom cost the dam break over the bump 27 %.)
__device__ __noinline__ double bottom_average(const double* br, const double* coef, int pieces, int deg, double a, double c) {
  int lo = 0, hi = pieces;  // the piece p with br[p] <= a < br[p + 1] (clamped)
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (!swale::dlt(a, br[mid])) lo = mid;
    else hi = mid;
  }
  const double x1 = 0.9061798459386639928, x2 = 0.5384693101056830910;
  const double w1 = 0.5 * 0.2369268850561890875, w2 = 0.5 * 0.4786286704993664680;
  auto mean = [&](int p, double l, double h) {
    const double* ck = coef + p * (deg + 1);
    if (deg == 0) return ck[0];
    const double t = 0.5 * (l + h) - br[p], hw = 0.5 * (h - l);
    auto v = [&](double y) {
      double r = ck[deg];
      for (int k = deg - 1; k >= 0; --k) r = fma(r, y, ck[k]);
      return r;
    };
    const double v0 = v(t);
    const double a1 = fma(-2.0, v0, v(fma(hw, x1, t)) + v(fma(-hw, x1, t)));
    const double a2 = fma(-2.0, v0, v(fma(hw, x2, t)) + v(fma(-hw, x2, t)));
    return fma(w1, a1, fma(w2, a2, v0));
  };
  if (!swale::dlt(a, br[lo]) && !swale::dlt(br[lo + 1], c)) return mean(lo, a, c);
  double s = 0.0;
  for (int p = lo; p < pieces && br[p] < c; ++p) {
    const double l = fmax(a, br[p]), h = fmin(c, br[p + 1]);
    if (h > l) s += (h - l) * mean(p, l, h);
  }
  return s / (c - a);
}
__device__ __forceinline__ double bottom_average(const StepConst& K, double a, double c) {
  return bottom_average(K.bot_breaks, K.bot_coef, K.bot_pieces, K.bot_deg, a, c);
}

__device__ __forceinline__ unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }

__device__ __forceinline__ double bitsd(unsigned long long b) { return __longlong_as_double((long long)b); }

// Block-wide max of non-negative doubles, one atomicMax per block. The bit
// patterns of doubles >= +0 order like unsigned integers, so the reductions run on the integer
// pipe (the FP64 pipe is the bottleneck of the stage kernels). A NaN wins the max.
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) { return a > b ? a : b; }

__device__ __forceinline__ void block_max_to(unsigned long long* dst, double v) {
  __shared__ unsigned long long red[32];
  unsigned long long b = dbits(v);
  for (int o = 16; o > 0; o >>= 1) b = umax64(b, __shfl_xor_sync(0xffffffffu, b, o));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = b;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    b = lane < nw ? red[lane] : 0ull;
    for (int o = 16; o > 0; o >>= 1) b = umax64(b, __shfl_xor_sync(0xffffffffu, b, o));
    if (lane == 0) atomicMax(dst, b);
  }
  __syncthreads();
}

// Maximum over a warp of non-negative doubles as bit patterns, by the 32-bit reduction unit: the
// high words, then the low words of those that hold the largest.
__device__ __forceinline__ unsigned long long warp_umax64(unsigned long long v) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(v >> 32) == hi ? (unsigned)v : 0u);
  return ((unsigned long long)hi << 32) | lo;
}

// Raises *dst to v unless it is there already (most callers find that it is).
__device__ __forceinline__ void raise_to(unsigned long long* dst, unsigned long long v) {
  if (v > *(volatile const unsigned long long*)dst) atomicMax(dst, v);
}

// One edge state of the wave speed: depth, velocity and node velocity.
struct WaveEdge {
  double h, u, w;
  __device__ bool same(const WaveEdge& o) const {
    return dbits(h) == dbits(o.h) && dbits(u) == dbits(o.u) && dbits(w) == dbits(o.w);
  }
  __device__ double speed(double g) const { return swale::wave_speed(g, h, swale::sub_(u, w)); }
};

// Exact maximum of the edge wave speeds |u - w| + sqrt(g h) (Eq. alpha2D) of a block's cells, raised
// into *A, with few FP64 operations. FP32 bounds lo <= speed <= hi of every edge (relative error
// below 2^-20 of each term, 1e-15 for inputs below the FP32 range) rule out every edge whose hi is
// below the largest lo of the block or below `seen`, a value *A has held; the edges left are
// evaluated in FP64, once for a warp, or for several, whose edges left are all the same (flat water).
// On the 2^20-cell dam break, mostly still water, the evaluations cost about 20 of the
// reconstruction's 105 FP64 instructions per cell when every warp made its own; now about 2.
template <int T>
__device__ __forceinline__ void block_wave(unsigned long long* A, double seen, double g, bool useL, bool useR,
                                           const WaveEdge& L, const WaveEdge& R) {
  __shared__ unsigned s_lo[T / 32];
  __shared__ WaveEdge s_edge[T / 32];
  __shared__ int s_kind[T / 32];  // 0: no edge left, 1: all left are s_edge, 2: several
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const float gf = swale::f32_trunc(g);
  auto bounds = [&](bool use, const WaveEdge& e, float& lo, float& hi) {
    const float uf = swale::f32_trunc(e.u), wf = swale::f32_trunc(e.w), q = gf * fmaxf(swale::f32_trunc(e.h), 0.0f);
    float sq;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(sq) : "f"(q));
    const float v = fabsf(uf - wf) + sq, m = (fabsf(uf) + fabsf(wf)) * 4.8e-7f + 1e-15f;
    lo = use ? fmaxf(fmaf(v, 1.0f - 4e-6f, -m), 0.0f) : 0.0f;
    hi = use ? fmaf(v, 1.0f + 4e-6f, m) : -1.0f;
  };
  float lol, hil, lor, hir;
  bounds(useL, L, lol, hil);
  bounds(useR, R, lor, hir);
  const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(lol, lor)));
  if (lane == 0) s_lo[wid] = m;
  __syncthreads();
  unsigned bm = __float_as_uint(swale::f32_trunc(seen));
#pragma unroll
  for (int w = 0; w < T / 32; ++w) bm = bm > s_lo[w] ? bm : s_lo[w];
  const float thr = __uint_as_float(bm);
  const bool cl = !(hil < thr), cr = !(hir < thr);  // (a NaN stays)
  const bool kl = useL && cl, kr = useR && cr;
  const unsigned cand = __ballot_sync(0xffffffffu, kl || kr);
  int kind = 0;
  WaveEdge first{0.0, 0.0, 0.0};
  if (cand) {
    const int src = __ffs(cand) - 1;
    const bool r0 = !kl;  // the first left edge of this lane is its right one
    first.h = __shfl_sync(0xffffffffu, r0 ? R.h : L.h, src);
    first.u = __shfl_sync(0xffffffffu, r0 ? R.u : L.u, src);
    first.w = __shfl_sync(0xffffffffu, r0 ? R.w : L.w, src);
    kind = __all_sync(0xffffffffu, (!kl || L.same(first)) && (!kr || R.same(first))) ? 1 : 2;
    if (lane == 0) s_edge[wid] = first;
  }
  if (lane == 0) s_kind[wid] = kind;
  __syncthreads();
  if (kind == 1)
    for (int w = 0; w < wid; ++w)
      if (s_kind[w] == 1 && first.same(s_edge[w])) kind = 0;  // another warp evaluates it
  if (kind == 0) return;
  unsigned long long v;
  if (kind == 1) {
    v = dbits(first.speed(g));
  } else {
    v = 0ull;
    if (kl || kr) v = dbits((kl ? L : R).speed(g));
    if (kl && kr) v = umax64(v, dbits(R.speed(g)));
    v = warp_umax64(v);
  }
  if (lane == 0) raise_to(A, v);
}

__device__ __forceinline__ void block_or_status(unsigned int* dst, uint32_t st) {
  st = __reduce_or_sync(0xffffffffu, st);
  if ((threadIdx.x & 31) == 0 && st) atomicOr(dst, st);
}

// Programmatic dependent launch: a kernel lets the next one of its stream be scheduled when all its
// blocks have got to their last statements, and waits here for the one before it (complete, its
// writes visible) before it touches what that wrote. Every kernel launched with the attribute waits, so the
// chain orders a step's kernels as plain launches do; the launch latency overlaps the tail of the
// kernel before. (Triggered at the kernels' start instead, the next one's blocks filled the multiprocessors
// that came free first: 7 on some and 3 on others where 5 each would do, 12 % slower on 100003 cells.)
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------------------------
// Bulk (TMA) copies global -> shared, completed on an mbarrier. A copy needs 16-byte aligned
// source and destination and a size that is a multiple of 16 bytes (callers check all three).
// ------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
}
// Orders this thread's generic-proxy shared-memory accesses before later async-proxy ones.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for the phase `parity` of bar to complete, at most `tries` polls (each poll itself
// blocks for a short hardware-defined time). Returns false if it gave up. kWaitTries bounds the
// wait for a tile's copies; when it runs out, the block waits kDrainTries more polls for those
// copies before it leaves (a block must not exit while its copies can still write its shared
// memory, which the SM hands to the next block).
constexpr int kWaitTries = 1 << 20;
constexpr int kDrainTries = 1 << 24;
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, int tries) {
  for (int i = 0; i < tries; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// ------------------------------------------------------------------------------------
// Per-step prologue, one thread per instance: stage maxima reset, J^{n+1} statistics become
// those of J^n; an instance whose time reached t_end (t_end > 0) is marked done.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void prologue(const StepConst& K, const DevState& D, int i) {
  DevScalars* S = D.S + i;
  // An error in an earlier step, or the end time reached: the instance is done.
  if ((S->status & kErrBits) || (K.t_end > 0.0 && S->t >= K.t_end)) {
    S->done = 1;
    return;
  }
  S->done = 0;
  S->clipped = 0;
  S->step_idx = S->steps;
  S->Jmax[0] = S->JmaxN;
  S->Jmin0 = S->JminN;
  S->JmaxN = 0ull;
  S->JminN = 0x7ff0000000000000ull;  // +inf
  S->A[0] = S->A[1] = S->A[2] = 0ull;
  S->Jmax[1] = S->Jmax[2] = 0ull;
  S->Wabs = S->dWabs = 0ull;
  S->counter = 0u;
  S->st3 = 0u;
  if (K.mesh != SWALE_MESH_FLUID_GAUSS) S->Wbar = D.IC[i].Wbar_profile;
}
__global__ void k_prologue(StepConst K, DevState D) {
  pdl_wait();
  pdl_trigger();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < K.B) prologue(K, D, i);
}

// ------------------------------------------------------------------------------------
// Fluid-driven node velocity: raw_k = (u_{k-1} + u_k)/2 for k = 1..N-1 (u = hu/h, dry -> 0),
// truncated renormalised Gaussian filter, w_0 = w_N = 0. A block filters kMeshThreads nodes in
// one pass, one per thread, and tiles advance by kMeshNodes = kMeshThreads - 1 nodes: the last
// node of a tile is the next tile's first, filtered by both (the same to rounding: a tile scales by its own largest velocity),
// which gives the tile the right neighbour of its last node for max |w_{k+1} - w_k| without a
// second pass for one node.
//
// The filter's 2 H + 1 products run on the integer multiplier in fixed point: an FP64 FMA holds the sub-partition
// for 64 cycles, four 32-bit multiply-adds with 64-bit sums about ten. The raw velocities of the
// tile's window are scaled by a power of two to integers of b = 55 to 58 bits (filter_bits), the largest of them to the
// full length, the weights exp(-m^2 / 2 sigma^2) are 57-bit ones, both in limbs of 28 bits, and the sums
// are exact for every window that a configuration may ask for (filter_sum). With |v| the largest raw velocity and W the
// sum of the weights, rounding the velocities, the weights and the sum leaves at most ((W + 1) 2^(-b - 1) + (2 H + 1) 2^-57) |v|
// before the division by W: no more than an FP64 sum leaves where the window's velocities have 53 bits or more in that scale,
// in the mean (filter_fits). The other nodes, those of quiet water beside fast, take the FP64 sum, and so do nodes whose
// window is cut off by an end, and tiles whose largest velocity is beyond 2^900, below 2^-902 or a NaN.
// The kernel issues 14 FP64 instructions per node (61 with the FP64 sum alone) and takes 40 us at 2^20 cells (118), 15 at 131071,
// where the tiles at the fronts are the longest.
// The block stages the cell velocities and the raw node velocities in shared memory (dynamic, and
// the limbs in place of the former), and the weights in both forms: 3 T + 8 H + 5 doubles.
// ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(kMeshThreads) k_mesh_gauss(StepConst K, DevState D) {
  extern __shared__ double sh[];
  __shared__ unsigned wmax[kMeshThreads / 32];
  const int H = K.gauss_half, T = kMeshThreads, tid = threadIdx.x, bits = swale::filter_bits(2 * H + 1);
  const int nu = T + 2 * H + 2, nr = T + 2 * H + 1;
  double* su = sh;         // cell velocities, cells [k0 - H - 1, k0 + T + H]; then the limbs of sraw
  double* sraw = sh + nu;  // raw node velocities, nodes [k0 - H, k0 + T + H]
  double* sw = sraw + nr;  // filtered velocities, nodes [k0, k0 + T)
  double* gw = sw + T;     // the weights
  swale::Limbs* gq = reinterpret_cast<swale::Limbs*>(gw + 2 * H + 1);
  swale::Limbs* sx = reinterpret_cast<swale::Limbs*>(su);
  if (tid <= 2 * H) {  // (written before the first step)
    gw[tid] = D.gauss->w[tid];
    gq[tid] = D.gauss->q[tid];
  }
  const long long need = D.gauss->need;
  pdl_wait();
  for (int t = blockIdx.x; t < D.nm; t += gridDim.x) {
    const Tile tl = D.mtiles ? D.mtiles[t] : Tile{0, t * kMeshNodes};
    DevScalars* S = D.S + tl.inst;
    if (S->done) continue;
    const InstConst ic = D.IC[tl.inst];
    const int64_t N = ic.N, k0 = tl.c0;
    const double* E0 = D.E0 + ic.coff;
    const double* M0 = D.M0 + ic.coff;
    const double* B0 = D.B0 + ic.coff;
    double* w = D.w + ic.coff + tl.inst;
    __syncthreads();
    for (int i = tid; i < nu; i += T) {
      const int64_t c = k0 - H - 1 + i;
      double u = 0.0;
      if (c >= 0 && c < N) {
        const double h = E0[c] - B0[c];
        u = swale::dlt(K.sc.h_dry, h) ? M0[c] * swale::recip(h) : 0.0;
      }
      su[i] = u;
    }
    __syncthreads();
    unsigned top = 0u;  // high word of the largest magnitude
    for (int i = tid; i < nr; i += T) {
      const int64_t k = k0 - H + i;
      const double v = (k >= 1 && k <= N - 1) ? 0.5 * (su[i] + su[i + 1]) : 0.0;
      sraw[i] = v;
      const unsigned hi = (unsigned)__double2hiint(v) & 0x7fffffffu;
      top = top > hi ? top : hi;
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if ((tid & 31) == 0) wmax[tid >> 5] = top;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kMeshThreads / 32; ++q) top = top > wmax[q] ? top : wmax[q];
    // |v| < 2^(ex - 1022) for every raw velocity.
    const int ex = (int)(top >> 20);
    const bool fixed = ex > 120 && ex < 1923;  // (2^-902 to 2^900, and no NaN or infinity)
    if (fixed)
      for (int i = tid; i < nr; i += T) sx[i] = swale::fixed_point(sraw[i], ex, bits);
    __syncthreads();
    {
      const int i = tid;
      const int64_t k = k0 + i;
      const bool whole = k - H >= 1 && k + H <= N - 1;  // the window
      // (A warp takes one of the sums: an FP64 instruction costs the same for one lane as for 32.)
      const bool fits = fixed && __all_sync(0xffffffffu, !whole || swale::filter_fits(sx + i, gq, H, need));
      double v = 0.0;
      if (top == 0u) {
        v = 0.0;  // still water
      } else if (whole && fits) {
        // (2^(1022 - ex + bits) times the filtered value)
        v = (double)swale::filter_sum(sx + i, gq, 2 * H + 1) * (K.gauss_iwsum * bitsd((unsigned long long)(ex + 1 - bits) << 52));
      } else if (whole) {
        double acc = 0.0;
        for (int m = 0; m <= 2 * H; ++m) acc += gw[m] * sraw[i + m];
        v = acc * K.gauss_iwsum;
      } else if (k >= 1 && k <= N - 1) {
        double acc = 0.0, wsum = 0.0;
        for (int m = -H; m <= H; ++m) {
          const int64_t q = k + m;
          if (q < 1 || q > N - 1) continue;
          acc += gw[m + H] * sraw[i + m + H];
          wsum += gw[m + H];
        }
        v = acc / wsum;
      }
      sw[i] = v;
    }
    __syncthreads();
    const int64_t k = k0 + tid;
    double wa = 0.0, dwa = 0.0;
    if (tid < kMeshNodes && k <= N) {
      w[k] = sw[tid];
      wa = fabs(sw[tid]);
      if (k < N) dwa = fabs(sw[tid + 1] - sw[tid]);
    }
    if (t + gridDim.x >= D.nm) pdl_trigger();
    block_max_to(&S->Wabs, wa);
    block_max_to(&S->dWabs, dwa);
  }
}

// ------------------------------------------------------------------------------------
// Reconstruction + limiter of cells -1..N_i (rows a2-a7) for stage STAGE. A block of T threads
// holds T consecutive cells, one per thread, and reconstructs the T - 4 inner ones: the
// differences of order two to five that the stencils share (pairs, triples, quadruples,
// quintuples of cells) are formed once each, one per thread and order, through shared memory, so
// that every phase is a single pass of the block (a tile of T cells with a halo would leave four
// entries of each phase to a second pass of one warp). It stores the edge states, the pair / triple reciprocals and
// pair differences that the update kernel of the same stage reads, reduces the wave speed, and in
// stage 1 the instance's last tile computes its dt (and the secant factor of the prescribed motion).
// What bounds it: FP64 instructions, each of which holds its SM sub-partition for 64 cycles, and beside them
// about 1000 others at 0.5-1 cycle. Per cell it issues 81 / 85 / 85 of them in stages 1 / 2 / 3 (83 / 151 / 149 when the
// mesh geometry was formed per cell and cached in 28 arrays); at 2^20 cells a launch takes 170 / 172 / 170 us
// (182 / 301 / 293) with the FP64 pipe 83-86 % busy and DRAM at 9-13 %, at 131071 cells 35 us at 65-71 %, where the
// loads and the drain of the one wave of blocks are a seventh of the time. The cells come by bulk copies: plain loads
// make a step of 2^20 cells 1.3 % slower.
// ------------------------------------------------------------------------------------
// Shared-memory rows of a tile that the out-of-line path of an open cell reads (row i: cell, pair,
// triple starting at cell c0 - 2 + i).
struct TileRows {
  const double *J, *E, *M, *H, *D2, *D3;
  int ld;  // distance between the rows of the three variables in D2, D3
};
struct OpenOut {
  EdgeState o;
  double etaG[2];
  uint32_t st;
  uint8_t flag;
};
// A cell of the non-well-balanced or special scheme whose smooth class the FP32 test leaves open (or
// whose widths are not moderate), out of line: the mesh geometry with its checks, the FP64 detector and
// the edge values of its class. A call, not inlined, so that this rare path's registers do not weigh
// on the smooth cells' code.
template <int SCHEME>
__device__ __noinline__ OpenOut recon_open_cell(const SchemeConst P, const TileRows R, int i, double dxe) {
  swale::CellGeom G;
  swale::StencilDD DD;
  double h[5], v0[3][3];
  const double* V[3] = {R.E, R.M, R.H};
#pragma unroll
  for (int k = 0; k < 5; ++k) h[k] = R.J[i - 2 + k];
#pragma unroll
  for (int v = 0; v < 3; ++v) {
#pragma unroll
    for (int a = 0; a < 3; ++a) v0[v][a] = V[v][i - 2 + a];
#pragma unroll
    for (int a = 0; a < 4; ++a) DD.D2[v][a] = R.D2[v * R.ld + i - 2 + a];
#pragma unroll
    for (int a = 0; a < 3; ++a) DD.D3[v][a] = R.D3[v * R.ld + i - 2 + a];
  }
  OpenOut r;
  r.st = 0;
  r.etaG[0] = r.etaG[1] = 0.0;
  swale::cell_geom(h, dxe, G, r.st);
  if (SCHEME == 1) {
    swale::recon_cell_nonwb_g(P, G, v0, DD, r.o, r.flag, r.st, swale::nonwb_proj(P, v0), nullptr, true);
  } else {
    swale::recon_cell_special_g(P, G, h, v0, DD, r.o, r.flag, r.st, r.etaG);
  }
  return r;
}

// a / b rounded once: the product with the reciprocal, corrected by its remainder (Markstein 1990), two operations where
// the division is a chain of a dozen (an accuracy run at N = 50 takes 5 % longer with divisions). Operands and
// quotients near the ends of the range take the division.
__device__ __forceinline__ double quotient(double a, double b) {
  const double y = swale::recip(b), q = a * y;
  const auto mid = [](double v) { return swale::gt_pos(v, 1e-250) && swale::lt_pos(v, 1e250); };
  if (!mid(a) || !mid(b) || !mid(q)) return a / b;
  return fma(fma(-b, q, a), y, q);
}

// A step's dt and the secant factor of the prescribed motion from alpha_1, by whole warps (every
// lane computes dt: an FP64 instruction costs the same for one lane as for 32). The secant factor
// (sin(2 pi (t + dt) / T) - sin(2 pi t / T)) / dt is formed as
// 2 cos(pi (2 t + dt) / T) sin(pi dt / T) / dt, which does not cancel, with the cosine and the sine in two lanes
// of the same instructions. inv_T: 1 / T of the profile motion, 0 for the others.
struct StepDt {
  double dt, alpha1, sdiff;
  int clipped, nodt;
};
__device__ __noinline__ StepDt step_dt(double cfl, double alpha1, double dwmax, double jmin, double tn, double dt_fixed,
                                       double t_end, double inv_T) {
  StepDt r{dt_fixed, alpha1, 0.0, 0, 0};
  if (!(dt_fixed > 0.0)) {
    r.dt = quotient(cfl * jmin, alpha1);
    if (dwmax > 0.0) r.dt = fmin(r.dt, quotient(0.5 * jmin, dwmax));
  }
  if (t_end > 0.0 && t_end - tn <= r.dt) {
    r.dt = t_end - tn;
    r.clipped = 1;
  }
  // alpha = 0 (a dry state at rest on a mesh that does not move) leaves the CFL condition
  // with no bound; without an end time there is no step to take: dt = 0, flagged.
  if (!(r.dt < INFINITY)) {
    r.dt = 0.0;
    r.nodt = 1;
  }
  if (inv_T > 0.0 && r.dt > 0.0) {
    const bool first = (threadIdx.x & 31) == 0;
    const double x = (first ? 2.0 * tn + r.dt : r.dt) * inv_T;
    double v;
    if (x < 1e12) v = swale::trig_pi(x, !first);
    else v = first ? cospi(x) : sinpi(x);
    const double cs0 = __shfl_sync(0xffffffffu, v, 0), sn1 = __shfl_sync(0xffffffffu, v, 1);
    r.sdiff = r.dt > 1e-290 ? 2.0 * cs0 * sn1 * swale::recip(r.dt) : 2.0 * cs0 * sn1 / r.dt;
  }
  return r;
}

// The same for the stage kernels, by one warp of the instance's last stage-1 tile.
__device__ __forceinline__ void stage1_dt(const StepConst& K, DevScalars* S, const InstConst& ic, int inst) {
  __threadfence();
  const int lane = threadIdx.x & 31;
  const bool fluid = K.mesh == SWALE_MESH_FLUID_GAUSS;
  const double A1 = bitsd(*(volatile const unsigned long long*)&S->A[0]);
  const double Wbar = fluid ? bitsd(*(volatile const unsigned long long*)&S->Wabs) : S->Wbar;
  const double dwmax = fluid ? bitsd(*(volatile const unsigned long long*)&S->dWabs) : 0.0;
  double alpha1 = K.wave_rel ? A1 : A1 + Wbar;
  if (K.alpha_mode != 0) {
    if (lane == 0) alpha1 = stage_alpha(K, inst, 1, alpha1, S->step_idx);
    alpha1 = __shfl_sync(0xffffffffu, alpha1, 0);
  }
  const StepDt r = step_dt(ic.cfl, alpha1, dwmax, bitsd(S->Jmin0), S->t, K.dt_fixed, K.t_end,
                           K.mesh == SWALE_MESH_PROFILE ? K.inv_T : 0.0);
  if (lane == 0) {
    if (r.nodt) atomicOr(&S->status, (unsigned int)swale::ST_NODT);
    S->Wbar = Wbar;
    S->dt = r.dt;
    S->alpha1 = r.alpha1;
    S->clipped = r.clipped;
    S->sdiff = r.sdiff;
    S->counter = 0u;
  }
}

// Shared rows of the phases. Every phase runs on all threads: the last rows hold nothing that a
// reconstructed cell reads (they are padded for the reads past the block).
template <int T, int SCHEME>
struct ReconRows {
  static constexpr int NV32 = SCHEME == 1 ? 3 : 2;
  double H[T + 2], P[T + 2], Q[T];            // depths; pair and quadruple sums of widths
  double D2[3][T + 2], D3[3][T + 2], D4[3][T];  // divided differences of eta, hu, h (non-well-balanced scheme: of the bottom)
  // FP32 copies for the smooth-class test: widths, triple reciprocals, pair differences (hu, h, and
  // for the non-well-balanced scheme eta)
  float Jf[T], ITf[T], D2f[NV32][T];
  // Hydrostatic scheme: the cells that the test leaves open, and their edge values [edge][variable][cell],
  // classes and status bits.
  static constexpr int TX = SCHEME == 0 ? T : 1;
  double X[2][3][TX];
  uint16_t open[TX];
  uint8_t cls[TX], xst[TX];
  int nopen;
};
// Reciprocal sums of the widths a thread takes from the mesh cache (see k_recon): `pair`, `next` say
// which it has, `all_pair`, `all_next` whether its whole warp has them (no reciprocal is formed then).
struct MeshRecips {
  double ip, it, iq, iv;
  bool pair, next, all_pair, all_next;
};

// The mesh checks of a cell whose widths are not moderate (see moderate_widths), as cell_geom makes them.
__device__ __noinline__ uint32_t width_status(const double* J) {
  double h[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) h[k] = J[k];
  swale::CellGeom G;
  uint32_t st = 0;
  swale::cell_geom(h, h[2], G, st, false);
  return st;
}

// Edge `right` of the open cell i of a block (hydrostatic scheme): its values into R.X, and (by the left
// edge's thread) its class and status.
// (A call: its registers do not weigh on the smooth cells' code.)
template <int T, int SCHEME>
__device__ __noinline__ void open_edge(const SchemeConst P, ReconRows<T, SCHEME>& R, const double* sE, const double* sM,
                                          const double* sJ, int i, bool right, double dxmax) {
  double h[5], p[4], v[3], d2[3][4], d3[3][3], d4[3][2], out[3];
#pragma unroll
  for (int k = 0; k < 5; ++k) h[k] = sJ[i - 2 + k];
#pragma unroll
  for (int k = 0; k < 4; ++k) p[k] = R.P[i - 2 + k];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    v[q] = (q == 0 ? sE : q == 1 ? sM : R.H)[i];
#pragma unroll
    for (int a = 0; a < 4; ++a) d2[q][a] = R.D2[q][i - 2 + a];
#pragma unroll
    for (int a = 0; a < 3; ++a) d3[q][a] = R.D3[q][i - 2 + a];
#pragma unroll
    for (int a = 0; a < 2; ++a) d4[q][a] = R.D4[q][i - 2 + a];
  }
  // (the same sum as the quintuple's: the quadruple that starts at i - 2, and the last width)
  const double iv = swale::recip(swale::add_(swale::add_(p[0], p[2]), h[4]));
  const uint8_t flag = swale::open_edge_values(P, h, p, P.beta_dx_global ? dxmax : h[2], iv, v, d2, d3, d4, right, out);
#pragma unroll
  for (int q = 0; q < 3; ++q) R.X[right ? 1 : 0][q][i] = out[q];
  if (!right) {
    R.cls[i] = flag;
    R.xst[i] = (uint8_t)(swale::moderate_widths(R.Jf[i - 2], R.Jf[i - 1], R.Jf[i], R.Jf[i + 1], R.Jf[i + 2])
                             ? 0u
                             : width_status(sJ + i - 2));
  }
}

// The same by eight lanes a cell (four for each edge), a chain of about 67 operations instead of 118: lane r
// of an edge forms the indicator, the linear weight and the nonlinear weight of sub-stencil r, then the edge value
// of variable r, every number by the same operations as open_edge_values, bit for bit. Called by whole
// warps; n cells, four to a warp and pass. It costs more lanes than it saves operations, so it serves blocks
// that have their SM to themselves, where the chain is what is waited for: an accuracy run to t = 0.1 at N = 50,
// most of whose cells are open, takes 35.1 ms instead of 39.0 (4 to 16 open cells in its one block).
template <int T, int SCHEME>
__device__ __noinline__ void open_cells_split(const SchemeConst P, ReconRows<T, SCHEME>& R, const double* sE, const double* sM,
                                              const double* sJ, int n, double dxmax) {
  using swale::add_;
  using swale::fma_;
  using swale::mul_;
  using swale::sub_;
  const int lane = threadIdx.x & 31, r = min(lane & 3, 2);
  const bool right = (lane & 4) != 0;
  for (int c0 = (threadIdx.x >> 5) * 4; c0 < n; c0 += T / 8) {
    const int k = c0 + (lane >> 3);
    const int i = R.open[min(k, n - 1)];
    auto from = [&](double v, int q) { return __shfl_sync(0xffffffffu, v, (lane & ~3) + q); };
    double h[5], p[4];
#pragma unroll
    for (int q = 0; q < 5; ++q) h[q] = sJ[i - 2 + q];
#pragma unroll
    for (int q = 0; q < 4; ++q) p[q] = R.P[i - 2 + q];
    const double dx = P.beta_dx_global ? dxmax : h[2];
    const int a = 2 - r;  // the sub-stencil's first cell
    const double hh = mul_(0.5, h[2]);
    double F = fma_(3.0, hh, p[0]);
    F = add_(a == 0 ? F : hh, a == 2 ? h[3] : h[1]);
    if (a == 2) F = -F;
    const double c4 = mul_(mul_(4.0, dx), h[2]), kap = fma_(mul_(9.0, dx), dx, mul_(mul_(3.0, hh), hh));
    const double d3h = R.D3[2][i - 2 + a], d3m = R.D3[1][i - 2 + a];
    const double qh = fma_(d3h, F, R.D2[2][i - 2 + a]), qm = fma_(d3m, F, R.D2[1][i - 2 + a]);
    const double beta = mul_(c4, fma_(kap, fma_(d3m, d3m, mul_(d3h, d3h)), fma_(qm, qm, mul_(qh, qh))));
    const double b0 = from(beta, 0), b1 = from(beta, 1), b2 = from(beta, 2);
    const double tau = swale::dabs(sub_(b0, b2));
    const double den = fma_(add_(add_(b0, b1), b2), 1.0 / 3.0, P.eps_weno);
    const uint8_t flag = swale::le_nn(tau, mul_(0.5, den)) ? 0 : (swale::le_nn(den, tau) ? 2 : 1);
    // Linear weights.
    const double Sa = add_(p[0], p[2]), Sb = add_(Sa, h[4]), Sc = add_(p[1], p[3]);
    const double inv = swale::recip(mul_(mul_(Sa, Sb), Sc));
    const double sum = r == 2 ? add_(p[2], h[4]) : add_(p[0], h[2]);
    const double fa = r == 2 ? (right ? h[3] : p[2]) : (right ? p[1] : h[1]);
    const double fb = r == 2 ? (right ? p[3] : sum) : (right ? sum : p[0]);
    double d = mul_(mul_(fa, fb), mul_(r == 2 ? Sc : Sa, inv));
    const double dm = sub_(sub_(1.0, from(d, 0)), from(d, 2));
    if (r == 1) d = dm;
    // WENO-Z weights and the blend.
    const double e = add_(beta, P.eps_weno);
    const double e0 = from(e, 0), e1 = from(e, 1), e2 = from(e, 2);
    const double ie = mul_(tau, swale::recip(mul_(mul_(e0, e1), e2)));
    const double q = mul_(mul_(r == 0 ? e1 : e0, r == 2 ? e1 : e2), ie);
    const double al = mul_(d, fma_(q, q, 1.0));
    const double is = swale::recip(add_(add_(from(al, 0), from(al, 1)), from(al, 2)));
    double phi = mul_(al, is);
    const double mg = fma_(2.0, mul_(tau, swale::recip(den)), -1.0);
    const double bl = fma_(mg, sub_(phi, d), d);
    if (flag == 1) phi = bl;
    const double f0 = from(phi, 0), f1 = from(phi, 1), f2 = from(phi, 2);
    // Variable r.
    const double v = (r == 0 ? sE : r == 1 ? sM : R.H)[i];
    const double d2l = R.D2[r][i - 1], d2r = R.D2[r][i], d3l = R.D3[r][i - 2], d3c = R.D3[r][i - 1], d3r = R.D3[r][i];
    double out;
    if (flag == 0) {
      const double iv = swale::recip(add_(Sa, h[4]));
      const swale::SmoothWidths w = {h[1], h[2], h[3], p[0], p[1], p[2], p[3]};
      const double d4l = R.D4[r][i - 2], d4r = R.D4[r][i - 1], d5 = mul_(sub_(d4r, d4l), iv);
      out = right ? swale::smooth_right(w, v, d2r, d3c, d4r, d5) : swale::smooth_left(w, v, d2l, d3c, d4l, d5);
    } else {
      const double dn = right ? d2r : d2l, df = right ? d2l : d2r;
      const double g = right ? -h[3] : h[1], gf = right ? p[1] : -p[2];
      const double s1 = fma_(g, d3c, dn);
      const double sa = fma_(g, right ? d3r : d3l, dn);
      const double sb = fma_(gf, right ? d3l : d3r, df);
      const double s = fma_(right ? f2 : f0, sb, fma_(right ? f0 : f2, sa, mul_(f1, s1)));
      out = fma_(right ? h[2] : -h[2], s, v);
    }
    if (k < n && (lane & 3) < 3) {
      R.X[right ? 1 : 0][r][i] = out;
      if ((lane & 7) == 0) {
        R.cls[i] = flag;
        R.xst[i] = (uint8_t)(swale::moderate_widths(R.Jf[i - 2], R.Jf[i - 1], R.Jf[i], R.Jf[i + 1], R.Jf[i + 2])
                                 ? 0u
                                 : width_status(sJ + i - 2));
      }
    }
  }
}

// The reconstruction of a block's T cells, thread i holding cell i: width jv, averages ev, mv of eta
// and hu, depth hv, also in the shared rows sE, sM, sJ (a barrier lies behind their stores). Threads
// with mine set (2 <= i <= T - 3) get the limited edge state o, the class and, for the special scheme,
// the interior points of eta. The sink is handed each thread's pair differences and reciprocals as
// they are formed: pair(ip, de, dh), triple(it), quad(iq), quint(iv). SPLIT: up to how many open cells
// open_cells_split takes them (dxmax, the stage's largest width, is read behind the first barrier): 16 (one warp per sub-partition) where the block is alone on its SM; none where
// other blocks fill it (up to 4 cells, one warp: 8580 us instead of 8556 for 8 steps of 10^6 cells).
template <int T, int SCHEME, int SPLIT, class Sink>
__device__ __forceinline__ void recon_phases(const SchemeConst& P, ReconRows<T, SCHEME>& R, const double* sE, const double* sM,
                                             const double* sJ, double jv, double ev, double mv, double hv, const double& dxmax,
                                             const MeshRecips& g, bool mine, Sink& sink, EdgeState& o, uint8_t& flag,
                                             swale::PointPair& pts, uint32_t& st, bool* limited = nullptr) {
  const int tid = threadIdx.x;
  R.H[tid] = hv;  // the depth is reconstructed in place of the bottom
  R.Jf[tid] = swale::f32_trunc(jv);
  if (SCHEME == 0 && tid == 0) R.nopen = 0;
  __syncthreads();
  // Order 2: the pair (i, i+1).
  double d2[3], d3[3];
  const double p = swale::add_(jv, sJ[tid + 1]);
  {
    const double de = swale::sub_(sE[tid + 1], ev), dm = swale::sub_(sM[tid + 1], mv), dh = swale::sub_(R.H[tid + 1], hv);
    double ip = g.ip;
    if (!g.all_pair) ip = g.pair ? g.ip : swale::recip(p);
    d2[0] = swale::mul_(de, ip);
    d2[1] = swale::mul_(dm, ip);
    // (the non-well-balanced scheme reconstructs the bottom, and its edge depths are eta's less the bottom's: the other
    // way round the rounding of eta's and h's edge values stays in the bottom's, and doubles the error of its right-hand side)
    d2[2] = swale::mul_(SCHEME == 1 ? swale::sub_(de, dh) : dh, ip);
    R.P[tid] = p;
#pragma unroll
    for (int v = 0; v < 3; ++v) R.D2[v][tid] = d2[v];
    R.D2f[0][tid] = swale::f32_trunc(d2[1]);
    R.D2f[1][tid] = swale::f32_trunc(d2[2]);
    if (SCHEME == 1) R.D2f[R.NV32 - 1][tid] = swale::f32_trunc(d2[0]);
    sink.pair(ip, de, dh);
  }
  __syncthreads();
  // Order 3: the triple (i, i+1, i+2).
  {
    double it = g.it;
    if (!g.all_next) it = g.next ? g.it : swale::recip(swale::add_(p, sJ[tid + 2]));
#pragma unroll
    for (int v = 0; v < 3; ++v) R.D3[v][tid] = d3[v] = swale::mul_(swale::sub_(R.D2[v][tid + 1], d2[v]), it);
    R.ITf[tid] = swale::f32_trunc(it);
    sink.triple(it);
  }
  __syncthreads();
  // Order 4: the quadruple (i .. i+3).
  {
    double iq = g.iq;
    if (!g.all_pair || !g.all_next) {  // (the quintuple's sum needs it where that is not cached)
      const double q = swale::add_(p, R.P[tid + 2]);
      R.Q[tid] = q;
      iq = g.next ? g.iq : swale::recip(q);
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) R.D4[v][tid] = swale::mul_(swale::sub_(R.D3[v][tid + 1], d3[v]), iq);
    sink.quad(iq);
  }
  const double dxe = P.beta_dx_global ? dxmax : jv;
  flag = 0;
  // The smooth class, when FP32 can tell it for sure; else the FP64 detector decides.
  bool smooth = false;
  if (mine) {
    if (!swale::gt0(jv)) st |= swale::ST_EMESH;
    const float hf[5] = {R.Jf[tid - 2], R.Jf[tid - 1], R.Jf[tid], R.Jf[tid + 1], R.Jf[tid + 2]};
    float F32[3], itf[3], c4f, c3f, d2h[4], d2m[4];
    swale::indicator_factors_f32(hf, swale::f32_trunc(dxe), F32, c4f, c3f);
#pragma unroll
    for (int a = 0; a < 3; ++a) itf[a] = R.ITf[tid - 2 + a];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      d2h[a] = R.D2f[1][tid - 2 + a];
      d2m[a] = R.D2f[0][tid - 2 + a];
    }
    const float epsf = swale::f32_trunc(P.eps_weno);
    if (SCHEME == 1) {
      float d2e[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) d2e[a] = R.D2f[R.NV32 - 1][tid - 2 + a];
      smooth = swale::sure_smooth_nonwb_f32(P.g, P.h_dry, hv, mv, F32, c4f, c3f, d2e, d2m, d2h, itf, epsf, true);
    } else {
      smooth = swale::sure_smooth_f32(F32, c4f, c3f, d2h, d2m, itf, epsf);
    }
    smooth = smooth && swale::moderate_widths(hf[0], hf[1], hf[2], hf[3], hf[4]);
  }
  // The open cells of the hydrostatic scheme: an FP64 instruction costs a warp the same for one lane
  // as for 32, so they are gathered and spread over the block's threads, two to a cell (one per edge),
  // instead of taking their own warps one by one through about twice the work. (The barrier is the
  // one that the differences of order 4 need anyway.)
  if constexpr (SCHEME == 0) {
    const bool open = mine && !smooth;
    if (open) R.open[atomicAdd(&R.nopen, 1)] = (uint16_t)tid;
    if (__syncthreads_or(open)) {
      const int n = R.nopen;
      if (SPLIT > 0 && n <= SPLIT) {
        open_cells_split<T, SCHEME>(P, R, sE, sM, sJ, n, dxmax);
      } else {
        for (int e = tid; e < 2 * n; e += T) open_edge<T, SCHEME>(P, R, sE, sM, sJ, R.open[e >> 1], e & 1, dxmax);
      }
      __syncthreads();
    }
  } else {
    __syncthreads();
  }
  if (!mine) return;
  // Order 5, the quintuple centred at i.
  double iv = g.iv;
  if (!g.all_pair) iv = g.pair ? g.iv : swale::recip(swale::add_(R.Q[tid - 2], sJ[tid + 2]));
  sink.quint(iv);
  if (SCHEME != 0 && !smooth) {
    const TileRows rows = {sJ, sE, sM, R.H, &R.D2[0][0], &R.D3[0][0], T + 2};
    const OpenOut r = recon_open_cell<SCHEME>(P, rows, tid, dxe);
    o = r.o;
    flag = r.flag;
    pts = swale::point_pair(ev, r.etaG[0], r.etaG[1]);
    st |= r.st;
    return;
  }
  double evl[3][2];
  if (smooth) {
    const swale::SmoothWidths w = {sJ[tid - 1], jv, sJ[tid + 1], R.P[tid - 2], R.P[tid - 1], p, R.P[tid + 1]};
    const double vj[3] = {ev, mv, SCHEME == 1 ? swale::sub_(ev, hv) : hv};
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      const double d4l = R.D4[v][tid - 2], d4r = R.D4[v][tid - 1], d3c = R.D3[v][tid - 1];
      const double d5 = swale::mul_(swale::sub_(d4r, d4l), iv);
      evl[v][0] = swale::smooth_left(w, vj[v], R.D2[v][tid - 1], d3c, d4l, d5);
      evl[v][1] = swale::smooth_right(w, vj[v], d2[v], d3c, d4r, d5);
      if (SCHEME == 2 && v == 0) pts = swale::smooth_points(w, ev, evl[0][0], evl[0][1], d4r, d5);
    }
    if (SCHEME == 1)
#pragma unroll
      for (int e = 0; e < 2; ++e) evl[2][e] = swale::sub_(evl[0][e], evl[2][e]);
  } else {
#pragma unroll
    for (int v = 0; v < 3; ++v) {
      evl[v][0] = R.X[0][v][tid];
      evl[v][1] = R.X[1][v][tid];
    }
    flag = R.cls[tid];
    st |= R.xst[tid];
  }
  swale::limit_cell(P, evl, hv, mv, o, st);
  if (limited) *limited = dbits(o.hL) != dbits(evl[2][0]) || dbits(o.hR) != dbits(evl[2][1]);
}

// Arrays of DevState::gK (see swale_adjoint_kernels.cuh).
enum { ADJ_IQ, ADJ_IV, ADJ_RHO, ADJ_SIG, ADJ_GX, ADJ_GY, ADJ_K3, ADJ_CLS, ADJ_DE, ADJ_DH, ADJ_H, ADJ_ARRAYS };

// Where k_recon's differences and reciprocals go: the arrays that the update of the stage reads, in
// stage 2 the mesh cache, and (STOREK) the arrays of the adjoint.
template <int STAGE, int SCHEME, bool STOREK>
struct ReconSink {
  const DevState& D;
  int32_t idx;      // edge-array index of the thread's cell
  bool mine, next_mine, use_geo, put_geo;
  double hv;
  __device__ __forceinline__ void pair(double ip, double de, double dh) const {
    if (!mine) return;
    if (SCHEME == 2 || STOREK || !use_geo) D.ipair[idx] = ip;  // (on the cache the update needs neither)
    D.dE[idx] = de;
    D.dH[idx] = dh;
    D.H[idx] = hv;
    if (STAGE == 2 && put_geo) D.geo[GEO_IP * D.geo_stride + idx] = ip;
  }
  __device__ __forceinline__ void triple(double it) const {
    if (!next_mine) return;
    if (SCHEME == 2 || STOREK || !use_geo) D.itri[idx + 1] = it;
    if (STAGE == 2 && put_geo) D.geo[GEO_IT * D.geo_stride + idx + 1] = it;
  }
  __device__ __forceinline__ void quad(double iq) const {
    if (STAGE == 2 && put_geo && next_mine) D.geo[GEO_IQ * D.geo_stride + idx + 1] = iq;
    if (STOREK && next_mine) D.gK[ADJ_IQ * D.geo_stride + idx + 1] = iq;
  }
  __device__ __forceinline__ void quint(double iv) const {
    if (STAGE == 2 && put_geo) D.geo[GEO_IV * D.geo_stride + idx] = iv;
    if (STOREK) D.gK[ADJ_IV * D.geo_stride + idx] = iv;
  }
};

// STOREK: an instantiation of the hydrostatic scheme that also stores what the reverse reads (the
// adjoint's recomputes). CACHE: one that may take the reciprocals from the mesh cache (stage 1, and every
// stage of a static mesh; in the others the values to be taken would only cost registers).
template <int STAGE, int T, int SCHEME = 0, bool STOREK = false, bool CACHE = STAGE == 1>
__global__ void __launch_bounds__(T, kReconThreads / T) k_recon(StepConst K, DevState D, const double* __restrict__ Eg,
                                             const double* __restrict__ Mg, const double* __restrict__ Bg,
                                             const double* __restrict__ Jg) {
  constexpr int TO = T - 4;                        // cells reconstructed
  __shared__ __align__(16) double sRaw[4][T + 8];  // E, M, B, J of cells c0-2 .. c0+T-3 as bulk-copied
  __shared__ ReconRows<T, SCHEME> rows;
  __shared__ bool sIdle;
  __shared__ __align__(8) uint64_t sBar;           // completion of the tile's bulk copies
  __shared__ __align__(8) uint64_t sPad;           // test hook: a barrier no copy completes
  __shared__ bool last;
  const int tid = threadIdx.x;
  const bool refl = (K.bc == SWALE_BC_REFLECTIVE);
  if (tid == 0) {
    mbar_init(&sBar);
    mbar_init(&sPad);
    fence_proxy_async();  // the initialised barriers, visible to the copy engine
  }
  __syncthreads();
  uint32_t phase = 0;
  pdl_wait();
  for (int t = blockIdx.x; t < D.nrf; t += gridDim.x) {
    const Tile tl = D.rftiles ? D.rftiles[t] : Tile{0, t * TO - 1};
    DevScalars* S = D.S + tl.inst;
    const InstConst ic = D.rftiles ? D.IC[tl.inst] : D.ic1;
    const int32_t N = (int32_t)ic.N, c0 = tl.c0;
    const double* E = Eg + ic.coff;
    const double* M = Mg + ic.coff;
    const double* B = Bg + ic.coff;
    const double* J = Jg + ic.coff;
    const int64_t eb = ic.coff + 2 * (int64_t)tl.inst;  // edge-array base of the instance
    // One thread reads the flags, for the whole block (the status may change meanwhile); the
    // copies start before they are known.
    if (tid == 0) sIdle = inst_idle(S);
    // The cells of the tile that lie in the instance, [cs, ce], arrive by four bulk copies (E, M,
    // B, J). The copied span [ga, ge] (global element indices) is widened to 16-byte boundaries:
    // one element before cs where needed (it exists: ga >= 1), one after ce when that element is
    // in the arrays (the instance is not the last one, or ce < N - 1), else one fewer (that cell
    // is loaded directly). Shared rows are shifted by `off` so that the first copied element
    // lands on a 16-byte boundary as well. Ghost cells and anything not copied take the direct
    // loads below.
    const int32_t cs = c0 - 2 < 0 ? 0 : c0 - 2, ce = c0 + T - 3 < N - 1 ? c0 + T - 3 : N - 1;
    int64_t ga = (ic.coff + cs) & ~(int64_t)1, ge = ic.coff + ce;
    if (!(ge & 1)) ge += (ce + 1 < N || tl.inst + 1 < K.B) ? 1 : -1;
    const int rel = (int)(ga - ic.coff - (c0 - 2));  // shared index of ga before the shift
    const int off = 2 - (rel & 1);
    const uint32_t bytes = ge >= ga ? (uint32_t)((ge - ga + 1) * 8) : 0u;
    const bool bulk = bytes >= 16 && ((((uintptr_t)(Eg + ga)) | ((uintptr_t)(Mg + ga)) | ((uintptr_t)(Bg + ga)) |
                                       ((uintptr_t)(Jg + ga))) & 15) == 0;
    const int32_t c = c0 - 2 + tid;                   // this thread's cell
    const int32_t idx = (int32_t)(eb + c + 1);        // its edge-array index
    const int32_t ca = (int32_t)(ga - ic.coff), cz = (int32_t)(ge - ic.coff);  // the cells copied
    // Reciprocal sums of the widths: as an earlier stage 2 stored them (the same mesh), or
    // formed below. Those that lie at cells -1..N are in the cache: the pair starting at c, the triple
    // and quadruple whose second cell is c + 1, the quintuple centred at c.
    const bool use_geo = CACHE && cached_mesh<STAGE>(K, D, S), put_geo = STAGE == 2 && D.geo && !use_geo;
    MeshRecips mr{0.0, 0.0, 0.0, 0.0, use_geo && c >= -1 && c <= N, use_geo && c >= -2 && c + 1 <= N, false, false};
    if (CACHE && use_geo) {
      mr.all_pair = __all_sync(0xffffffffu, mr.pair);
      mr.all_next = __all_sync(0xffffffffu, mr.next);
      if (mr.pair) {
        mr.ip = D.geo[GEO_IP * D.geo_stride + idx];
        mr.iv = D.geo[GEO_IV * D.geo_stride + idx];
      }
      if (mr.next) {
        mr.it = D.geo[GEO_IT * D.geo_stride + idx + 1];
        mr.iq = D.geo[GEO_IQ * D.geo_stride + idx + 1];
      }
    }
    const double seen = bitsd(*(volatile const unsigned long long*)&S->A[STAGE - 1]);
    const double dxmax = bitsd(S->Jmax[STAGE - 1]);
    // Node velocities of the cell's two edges (Eq. alpha2D: speeds relative to the node).
    double wl = 0.0, wr = 0.0;
    if (K.wave_rel && c >= -1 && c <= N) {
      const double* wv = node_velocities(K, D) + ic.coff + tl.inst;
      if (c >= 0) wl = wv[c];
      if (c < N) wr = wv[c + 1];
    }
    if (bulk) {
      if (tid == 0) {
        fence_proxy_async();  // the previous tile's reads of sRaw come before these writes
        mbar_arrive_expect_tx(&sBar, 4 * bytes);
        bulk_copy_g2s(&sRaw[0][rel + off], Eg + ga, bytes, &sBar);
        bulk_copy_g2s(&sRaw[1][rel + off], Mg + ga, bytes, &sBar);
        bulk_copy_g2s(&sRaw[2][rel + off], Bg + ga, bytes, &sBar);
        bulk_copy_g2s(&sRaw[3][rel + off], Jg + ga, bytes, &sBar);
        // Test hook: a second barrier expects bytes that no copy delivers.
        if (K.tx_pad) mbar_arrive_expect_tx(&sPad, K.tx_pad);
      }
      bool landed = mbar_wait_bounded(&sBar, phase, kWaitTries);
      bool ok = landed;
      if (!landed) landed = mbar_wait_bounded(&sBar, phase, kDrainTries);  // drain before leaving
      if (K.tx_pad && landed) ok = mbar_wait_bounded(&sPad, 0u, K.wait_tries > 0 ? K.wait_tries : kWaitTries);
      phase ^= 1u;
      // The copies did not complete in time (or the test barrier ran out): give the stage up.
      // Every copy of this block has landed here unless the drain wait ran out as well.
      if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicOr(&S->status, (unsigned int)swale::ST_TIMEOUT);
        return;
      }
    } else {
      __syncthreads();
    }
    if (sIdle) {
      __syncthreads();  // every thread has read the flag before the next tile's is written
      continue;
    }
    double* const sE = &sRaw[0][off];
    double* const sM = &sRaw[1][off];
    double* const sJ = &sRaw[3][off];
    double jv = 1.0, ev = 0.0, mv = 0.0, hv = 0.0;  // filler beyond the last ghost cell
    if (bulk && c >= 0 && c < N && c >= ca && c <= cz) {
      ev = sE[tid];
      mv = sM[tid];
      jv = sJ[tid];
      hv = swale::sub_(ev, sRaw[2][off + tid]);
    } else {
      if (c >= -3 && c <= N + 2) {
        const int32_t s = ghost(c, N, K.bc);
        jv = J[s];
        ev = E[s];
        mv = M[s];
        if (refl && (c < 0 || c >= N)) mv = -mv;
        hv = swale::sub_(ev, B[s]);
      }
      sE[tid] = ev;
      sM[tid] = mv;
      sJ[tid] = jv;
    }
    // Cells of the tile that are reconstructed and stored.
    const bool mine = tid >= 2 && tid < 2 + TO && c <= N;
    const bool next_mine = tid >= 1 && tid < 1 + TO && c + 1 <= N;  // cell c + 1 is
    ReconSink<STAGE, SCHEME, STOREK> sink{D, idx, mine, next_mine, use_geo, put_geo, hv};
    bool limited = false;
    EdgeState o;
    uint8_t flag = 0;
    swale::PointPair pts{0.0, 0.0};
    uint32_t st = 0;
    recon_phases<T, SCHEME, 0>(K.sc, rows, sE, sM, sJ, jv, ev, mv, hv, dxmax, mr, mine, sink, o, flag, pts, st, &limited);
    if (STAGE == 2 && put_geo && c0 == -1 && tid == 0)
      S->geo_tag = ((unsigned long long)K.geo_epoch << 32) | (unsigned long long)((S->step_idx + 1) & 0xffffffffLL);
    WaveEdge eL{0.0, 0.0, 0.0}, eR{0.0, 0.0, 0.0};
    bool useL = false, useR = false;
    if (mine) {
      // (with the limiter's mark, for the reverse)
      if (STOREK) D.gK[ADJ_CLS * D.geo_stride + idx] = (double)(flag + (limited ? 4 : 0));
      D.eEL[idx] = o.EL;
      D.eER[idx] = o.ER;
      D.eBL[idx] = o.BL;
      D.eBR[idx] = o.BR;
      D.ehL[idx] = o.hL;
      D.ehR[idx] = o.hR;
      D.euL[idx] = o.uL;
      D.euR[idx] = o.uR;
      if (SCHEME == 2) {
        D.eG1[idx] = pts.sum;
        D.eG2[idx] = pts.diff;
      }
      if (STAGE == 1) D.flags[idx] = flag;
      // Edges that touch interfaces 0..N only.
      useL = (c != -1);
      useR = (c != N);
      eL = {o.hL, o.uL, wl};
      eR = {o.hR, o.uR, wr};
    }
    if (t + gridDim.x >= D.nrf) pdl_trigger();
    block_wave<T>(&S->A[STAGE - 1], seen, K.sc.g, useL, useR, eL, eR);
    block_or_status(&S->status, st);
    if (STAGE == 1) {
      __syncthreads();  // the block's atomics come before its ticket
      if (tid == 0) {
        __threadfence();
        const unsigned int ticket = atomicAdd(&S->counter, 1u);
        last = (ticket == (unsigned)ic.ntiles_r - 1u);
      }
      __syncthreads();
      if (last && tid < 32) stage1_dt(K, S, ic, tl.inst);
    } else {
      __syncthreads();  // block_wave's shared rows are read before the next tile's are written
    }
  }
}

// ------------------------------------------------------------------------------------
// Fluxes, source and the RK combination of stage STAGE for cells 0..N_i-1 (rows a1, a8, a9;
// MODE 0), or the bare right-hand side of one instance (MODE 1, used by swale_rhs). A tile is
// T - 1 consecutive cells for a block of T threads: thread i forms the fluxes of interface
// j0 + i, once, and passes them to the cell on its left through shared memory (a tile of T cells
// would leave its last interface to a second pass of a single thread). Bound by FP64
// instructions like the reconstruction, so everything is at twice its value (the halves of the
// Lax-Friedrichs flux are then free) and the pressure terms are combined with the source in the
// cell (source_pressure_form in swale_cell.cuh).
//
// The three stages advance increments instead of the products J q: with the width recursion of
// Eq. Jacobi2D in closed form, J^(1) = J^{n+1} = J + dt dw and J^(2) = J + dt dw / 2, the
// combination of Eq. RK32D reads J^(s) q^(s) = J q + dt (b_s . R), so
//   q^(s) = q + (dt (b_s . R) - q (J^(s) - J)) / J^(s),  b = (1), (1/4, 1/4), (1/6, 1/6, 2/3):
// fewer operations, and the rounding of the products J q stays out of the state.
// ------------------------------------------------------------------------------------
struct RhsOut {
  double *RE, *RM, *RB;
  double alpha;
};

// Largest a and b over the block (non-negative doubles), raised into mx[0], mx[1], and the smallest c,
// lowered into *mn (or, with COMPL, its complement raised there), by three lanes after one barrier.
template <int T, bool COMPL>
__device__ __forceinline__ void block_widths(unsigned long long* mx, unsigned long long* mn, double a, double b, double c) {
  __shared__ unsigned long long red[3][T / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const unsigned long long ma = warp_umax64(dbits(a)), mb = warp_umax64(dbits(b)), mc = warp_umax64(~dbits(c));
  if (lane < 3) red[lane][wid] = lane == 0 ? ma : lane == 1 ? mb : mc;
  __syncthreads();
  if (threadIdx.x < 3) {
    unsigned long long m = 0ull;
#pragma unroll
    for (int w = 0; w < T / 32; ++w) m = umax64(m, red[threadIdx.x][w]);
    if (threadIdx.x < 2) raise_to(mx + threadIdx.x, m);
    else if (COMPL) raise_to(mn, m);
    else if (~m < *(volatile const unsigned long long*)mn) atomicMin(mn, ~m);
  }
}

// Update of stage STAGE (MODE 0) or the right-hand side for a given viscosity (MODE 1): blocks of T threads take
// T - 1 cells, so that their T interfaces are one pass, one flux each, shared with the right neighbour through
// shared memory; then the source joined with the edge pressures, and the RK combination as an increment of q^n.
// Bound by FP64 instructions: 73 / 91 / 92 a cell in stages 1 / 2 / 3 (95 / 132 / 142 with the source as a bilinear
// form with six mesh-only entries and J q combined), 148 / 186 / 189 us at 2^20 cells (190 / 263 / 285), the FP64
// pipe 87 % busy, DRAM at 20 %. Launch bound as the reconstruction's.
// SCHEME: 0 hydrostatic, 1 non-well-balanced, 2 special source. BOT: an instantiation with the
// L2-projection bottom. STOREK: one that also stores the source's ratios in D.gK (the adjoint's
// recomputes).
template <int STAGE, int MODE, int T, int SCHEME = 0, bool BOT = false, bool STOREK = false>
__global__ void __launch_bounds__(T, kUpdateThreads / T) k_update(StepConst K, DevState D, const double* __restrict__ Eg,
                                              const double* __restrict__ Mg, const double* __restrict__ Bg,
                                              const double* __restrict__ Jsg, RhsOut ro) {
  __shared__ double sF[3][T], sW[T];      // interfaces / nodes j0 .. j0+T-1: fluxes FE, FMl, FB
  __shared__ double sG[2][T], sDe[2][T];  // their sig and rho^2 (PairRatio); differences of eta and h
  __shared__ bool sIdle;
  const int tid = threadIdx.x;
  (void)Mg;
  constexpr int TC = T - 1;  // cells of a tile; its T interfaces j0 .. j0 + TC, one per thread
  pdl_wait();
  for (int t = blockIdx.x; t < D.nf; t += gridDim.x) {
    const Tile tl = D.ftiles ? D.ftiles[t] : Tile{0, t * TC};
    const int inst = tl.inst;
    DevScalars* S = D.S + inst;
    // Skip a finished instance and one whose step has failed (below, when the loads are under way).
    // In stage 3 the status does not change during the launch (this kernel raises its bits in
    // st3), so every tile of an instance decides alike: all commit the step or none does.
    if (MODE == 0 && tid == 0) sIdle = inst_idle(S);
    const InstConst ic = D.ftiles ? D.IC[inst] : D.ic1;
    const int32_t N = (int32_t)ic.N, j0 = tl.c0;
    const int64_t cb = ic.coff, nb = ic.coff + inst, eb = ic.coff + 2 * (int64_t)inst;
    const double* E = Eg + cb;
    const double* B = Bg + cb;
    const double* Js = Jsg + cb;
    double alpha, dt = 0.0;
    if (MODE == 1) {
      alpha = ro.alpha;
    } else {
      alpha = (STAGE == 1) ? S->alpha1 : bitsd(S->A[STAGE - 1]);
      if (STAGE > 1 && !K.wave_rel) alpha = swale::add_(alpha, S->Wbar);
      if (STAGE > 1) {
        // Replay of stages 2 and 3 (recorded below; stage 1 is handled where alpha1 is formed).
        if (K.alpha_mode == 2) alpha = stage_alpha(K, inst, STAGE, alpha, S->step_idx);
      }
      dt = S->dt;
    }
    const bool fresh_w = (MODE == 0 && STAGE == 1 && K.mesh == SWALE_MESH_PROFILE);
    // The source's mesh-only values are cached beside the reconstruction's reciprocals: stage 2
    // stores them and the next step's stage 1, on the same mesh, reads them under the same tag.
    const bool use_sgeo = MODE == 0 && cached_mesh<STAGE>(K, D, S), put_sgeo = STAGE == 2 && MODE == 0 && D.geo && !use_sgeo;
    const bool still = use_sgeo && K.mesh == SWALE_MESH_STATIC;  // 1 / J^(1), 1 / J^(2) are there too
    const double sdiff = fresh_w ? S->sdiff : 0.0;
    const int32_t k = j0 + tid;  // this thread's node / interface and cell
    const int32_t el = (int32_t)(eb + k), er = el + 1;
    swale::Flux2 F{0.0, 0.0, 0.0, 0.0};
    swale::PairRatio pr{0.0, 0.0, 0.0, 0.0};
    double wk = 0.0, ELj = 0.0, BLj = 0.0, hLj = 0.0, dE = 0.0, dH = 0.0;
    if (k <= N) {
      if (fresh_w) {
        wk = swale::mul_(D.P[nb + k], sdiff);
      } else if (MODE == 0 && K.mesh == SWALE_MESH_STATIC) {
        wk = 0.0;
      } else if (MODE == 0 && K.mesh == SWALE_MESH_LINEAR) {
        wk = D.P[nb + k];  // constant node velocity (Eq. velocity)
      } else {
        wk = D.w[nb + k];
      }
      // Interface k: left state = right edge of cell k-1 (edge index k), right state = left
      // edge of cell k (edge index k+1).
      ELj = D.eEL[er];
      BLj = D.eBL[er];
      hLj = D.ehL[er];
      dE = D.dE[el];  // eta_k - eta_{k-1}
      dH = D.dH[el];
      if (use_sgeo) {
        pr.rho = D.geo[GEO_RHO * D.geo_stride + el];
        pr.sig = D.geo[GEO_SIG * D.geo_stride + el];
        pr.rho2 = D.geo[GEO_RHO2 * D.geo_stride + el];
        pr.sig2 = D.geo[GEO_SIG2 * D.geo_stride + el];
      } else {
        const double Jl = Js[ghost(k - 1, N, K.bc)], Jr = Js[ghost(k, N, K.bc)];
        pr = swale::pair_ratio(Jl, Jr, D.ipair[el]);
      }
      F = swale::interface_flux2<SCHEME>(K.sc.g, alpha, wk, D.eER[el], ELj, D.eBR[el], BLj, D.ehR[el], hLj, D.euR[el],
                                         D.euL[er]);
      sF[0][tid] = F.FE;
      sF[1][tid] = F.FMl;
      sF[2][tid] = F.FB;
      sW[tid] = wk;
      sG[0][tid] = pr.sig;
      sG[1][tid] = pr.rho2;
      sDe[0][tid] = dE;
      sDe[1][tid] = dH;
    }
    __syncthreads();
    if (MODE == 0 && sIdle) {
      __syncthreads();  // every thread has read the flag before the next tile's is written
      continue;
    }
    if (MODE == 0 && k <= N) {
      // The node velocities of the step, where this stage makes them (a tile's last node is the
      // next tile's first).
      if (STAGE == 1 && (fresh_w || K.mesh == SWALE_MESH_LINEAR) && (tid < TC || k == N)) D.w[nb + k] = wk;
      if (put_sgeo) {
        D.geo[GEO_RHO * D.geo_stride + el] = pr.rho;
        D.geo[GEO_SIG * D.geo_stride + el] = pr.sig;
        D.geo[GEO_RHO2 * D.geo_stride + el] = pr.rho2;
        D.geo[GEO_SIG2 * D.geo_stride + el] = pr.sig2;
      }
      if (STOREK) {
        D.gK[ADJ_RHO * D.geo_stride + el] = pr.rho;
        D.gK[ADJ_SIG * D.geo_stride + el] = pr.sig;
      }
      // Every tile has the same viscosity; the first one of the instance records it.
      if (STAGE > 1 && K.alpha_mode == 1 && k == 0) stage_alpha(K, inst, STAGE, alpha, S->step_idx);
    }
    const int32_t j = k;
    double jmaxa = 0.0, jmaxb = 0.0, jminb = INFINITY;
    uint32_t st = 0;
    if (tid < TC && j < N) {
      const double ERj = D.eER[er], BRj = D.eBR[er], hRj = D.ehR[er];
      const double hj = D.H[er], Ej = E[j];
      // Twice the momentum's right-hand side: the fluxes, then the pressure and source terms.
      double Rm = swale::sub_(F.FMr, sF[1][tid + 1]);
      const double Jm = use_sgeo && SCHEME != 2 ? 0.0 : Js[ghost(j - 1, N, K.bc)];
      const double Jc = use_sgeo && SCHEME != 2 ? 0.0 : Js[j];
      const double Jp = use_sgeo && SCHEME != 2 ? 0.0 : Js[ghost(j + 1, N, K.bc)];
      if (SCHEME == 2) {
        const double bd[5] = {B[ghost(j - 1, N, K.bc)], B[j], B[ghost(j + 1, N, K.bc)], BLj, BRj};
        double iJm, iJc, iJp;
        // 1 / J of the neighbours: stored by the previous stage's update, or formed here. On a moving mesh stage 1 forms
        // it although the last step left it in iJ1 (the same value): this launch's other threads write 1 / J^(1)
        // there. A static mesh's iJ1 is not written again.
        if (MODE == 0 && (STAGE > 1 || still)) {
          const double* iJ = (STAGE == 3 ? D.iJ2 : D.iJ1) + cb;
          iJm = iJ[ghost(j - 1, N, K.bc)];
          iJc = iJ[j];
          iJp = iJ[ghost(j + 1, N, K.bc)];
        } else {
          iJm = swale::recip(Jm);
          iJc = swale::recip(Jc);
          iJp = swale::recip(Jp);
        }
        const swale::SourceGeom sg = swale::source_geom(Jm, Jc, iJm, iJc, iJp, D.ipair[el], D.ipair[er], D.itri[er]);
        const swale::PointPair pts = {D.eG1[er], D.eG2[er]};
        Rm = swale::add_(Rm, swale::source_special2(K.sc.g, Ej, ELj, ERj, pts, bd, sg, D.eBR[er - 1], D.eBL[er + 1]));
      } else {
        swale::SourceRatio sr;
        if (use_sgeo) {
          sr.GX = D.geo[GEO_GX * D.geo_stride + er];
          sr.GY = D.geo[GEO_GY * D.geo_stride + er];
          sr.K3 = D.geo[GEO_K3 * D.geo_stride + er];
        } else {
          // 1 / J of the stage mesh: stored by the previous stage's update, or formed here
          double iJm, iJp;
          if (MODE == 0 && STAGE > 1) {
            const double* iJ = (STAGE == 2 ? D.iJ1 : D.iJ2) + cb;
            iJm = iJ[ghost(j - 1, N, K.bc)];
            iJp = iJ[ghost(j + 1, N, K.bc)];
          } else {
            iJm = swale::recip(Jm);
            iJp = swale::recip(Jp);
          }
          sr = swale::source_ratio(Jm, Jc, Jp, iJm, iJp, D.itri[er]);
        }
        if (put_sgeo) {
          D.geo[GEO_GX * D.geo_stride + er] = sr.GX;
          D.geo[GEO_GY * D.geo_stride + er] = sr.GY;
          D.geo[GEO_K3 * D.geo_stride + er] = sr.K3;
        }
        if (STOREK) {
          D.gK[ADJ_GX * D.geo_stride + er] = sr.GX;
          D.gK[ADJ_GY * D.geo_stride + er] = sr.GY;
          D.gK[ADJ_K3 * D.geo_stride + er] = sr.K3;
        }
        const double acc = swale::source_pressure_form(hj, hLj, hRj, swale::sub_(ELj, Ej), swale::sub_(ERj, Ej), dE, dH, sDe[0][tid + 1],
                                                       sDe[1][tid + 1], pr.rho, pr.sig2, sG[0][tid + 1],
                                                       sG[1][tid + 1], sr);
        Rm = swale::fma_(-K.sc.g, acc, Rm);
      }
      // Twice the right-hand sides.
      const double R2[3] = {swale::sub_(F.FE, sF[0][tid + 1]), Rm, swale::sub_(sF[2][tid + 1], F.FB)};
      if (MODE == 1) {
        ro.RE[j] = 0.5 * R2[0];
        ro.RM[j] = 0.5 * R2[1];
        ro.RB[j] = 0.5 * R2[2];
      } else {
        const int32_t g = (int32_t)cb + j;  // global cell index
        const double wl = wk, wr = sW[tid + 1];
        const double J0 = D.J0[g];
        // The width's increment over the step (stage 2: half of it).
        const double dJ = swale::mul_(STAGE == 2 ? swale::down_<1>(dt) : dt, swale::sub_(wr, wl));
        const double q0[3] = {D.E0[g], D.M0[g], D.B0[g]};
        if (STAGE == 1) {
          const double J1 = swale::add_(J0, dJ), J2 = swale::fma_(0.5, dJ, J0);
          D.J1[g] = J1;
          D.J2[g] = J2;
          jmaxa = J1;
          jmaxb = J2;
          jminb = J1;
          if (!swale::gt0(J1) || !swale::gt0(J2)) st |= swale::ST_EMESH;
          double inv;
          if (still) inv = D.iJ1[g];
          else D.iJ1[g] = inv = swale::recip(J1);
          D.YE[g] = R2[0];
          D.YM[g] = R2[1];
          D.YB[g] = R2[2];
          const double hdt = swale::down_<1>(dt);
          D.Ea[g] = swale::rk_advance(q0[0], hdt, R2[0], dJ, inv);
          D.Ma[g] = swale::rk_advance(q0[1], hdt, R2[1], dJ, inv);
          if (!BOT) D.Ba[g] = swale::rk_advance(q0[2], hdt, R2[2], dJ, inv);
          else  // bottom of stage 2: projection onto the mesh at t_{n+1}
            D.Ba[g] = bottom_average(K, D.x[nb + j] + dt * wl, D.x[nb + j + 1] + dt * wr);
        } else if (STAGE == 2) {
          const double Y[3] = {swale::add_(D.YE[g], R2[0]), swale::add_(D.YM[g], R2[1]), swale::add_(D.YB[g], R2[2])};
          D.YE[g] = Y[0];
          D.YM[g] = Y[1];
          D.YB[g] = Y[2];
          double inv;
          if (still) inv = D.iJ2[g];
          else D.iJ2[g] = inv = swale::recip(D.J2[g]);
          const double edt = swale::down_<3>(dt);
          D.Eb[g] = swale::rk_advance(q0[0], edt, Y[0], dJ, inv);
          D.Mb[g] = swale::rk_advance(q0[1], edt, Y[1], dJ, inv);
          if (!BOT) {
            D.Bb[g] = swale::rk_advance(q0[2], edt, Y[2], dJ, inv);
          } else {  // bottom of stage 3: projection onto the mesh at t_{n+1/2}
            const double xl = D.x[nb + j], xr = D.x[nb + j + 1];
            D.Bb[g] = bottom_average(K, xl + 0.5 * dt * wl, xr + 0.5 * dt * wr);
            D.xn[nb + j] = xl + dt * wl;  // nodes at t_{n+1} for the projection after the step
            if (j == N - 1) D.xn[nb + N] = xr + dt * wr;
          }
        } else {
          const double J3 = D.J1[g], inv = D.iJ1[g];  // J^{n+1} = J^(1)
          if (D.bE) {  // q^n, J^n, x^n kept for a roll-back by k_commit
            D.bE[g] = q0[0];
            D.bM[g] = q0[1];
            D.bB[g] = q0[2];
            D.bJ[g] = J0;
            D.bx[nb + j] = D.x[nb + j];
            if (j == N - 1) D.bx[nb + N] = D.x[nb + N];
          }
          const double tdt = dt * (1.0 / 12.0);
          const double En = swale::rk_advance(q0[0], tdt, swale::fma_(4.0, R2[0], D.YE[g]), dJ, inv);
          const double Mn = swale::rk_advance(q0[1], tdt, swale::fma_(4.0, R2[1], D.YM[g]), dJ, inv);
          double Bn = swale::rk_advance(q0[2], tdt, swale::fma_(4.0, R2[2], D.YB[g]), dJ, inv);
          if (BOT) {  // bottom after the step: projection onto the mesh at t_{n+1}
            const double xl = D.xn[nb + j], xr = D.xn[nb + j + 1];
            if (swale::bad(Bn)) st |= swale::ST_NONFINITE;
            Bn = bottom_average(K, xl, xr);
            D.x[nb + j] = xl;
            if (j == N - 1) D.x[nb + N] = xr;
          } else {
            D.x[nb + j] = swale::fma_(dt, wl, D.x[nb + j]);
            if (j == N - 1) D.x[nb + N] = swale::fma_(dt, wr, D.x[nb + N]);
          }
          D.E0[g] = En;
          D.M0[g] = Mn;
          D.B0[g] = Bn;
          D.J0[g] = J3;
          if (swale::bad(En) || swale::bad(Mn) || (!BOT && swale::bad(Bn))) st |= swale::ST_NONFINITE;
        }
      }
    }
    if (t + gridDim.x >= D.nf) pdl_trigger();
    if (MODE == 0) {
      block_or_status(STAGE == 3 ? &S->st3 : &S->status, st);
      if (STAGE == 1) block_widths<T, false>(&S->Jmax[1], &S->JminN, jmaxa, jmaxb, jminb);
    }
    __syncthreads();  // this tile's reads of the shared rows come before the next tile's writes
  }
}

// ------------------------------------------------------------------------------------
// End of a step, one block per instance (grid-stride): a clean step advances the instance's time
// and step count; a step whose stage-3 update raised an error (after committing its cells) is
// rolled back from the backups, and one that failed earlier wrote nothing. The stage-3 bits
// join the status word here. next: another step follows in the same sequence of launches, whose
// prologue is done here too.
// ------------------------------------------------------------------------------------
__global__ void k_commit(StepConst K, DevState D, int next) {
  pdl_wait();
  pdl_trigger();
  for (int i = blockIdx.x; i < K.B; i += gridDim.x) {
    DevScalars* S = D.S + i;
    const bool skip = S->done;
    const unsigned int before = S->status & kErrBits, bad3 = S->st3 & kErrBits;
    __syncthreads();  // every thread has read the words before thread 0 changes them
    if (skip) continue;
    if (!before && bad3 && D.bE) {
      const InstConst ic = D.IC[i];
      const int64_t cb = ic.coff, nb = ic.coff + i;
      for (int64_t j = threadIdx.x; j < ic.N; j += blockDim.x) {
        D.E0[cb + j] = D.bE[cb + j];
        D.M0[cb + j] = D.bM[cb + j];
        D.B0[cb + j] = D.bB[cb + j];
        D.J0[cb + j] = D.bJ[cb + j];
      }
      for (int64_t k = threadIdx.x; k <= ic.N; k += blockDim.x) D.x[nb + k] = D.bx[nb + k];
    }
    if (threadIdx.x == 0) {
      S->status |= S->st3;
      if (!before && !bad3) {
        S->t = S->clipped ? K.t_end : S->t + S->dt;
        S->steps += 1;
        S->JmaxN = S->Jmax[1];  // J^{n+1} = J^(1)
      } else {  // the widths stay those of J^n
        S->JmaxN = S->Jmax[0];
        S->JminN = S->Jmin0;
      }
      if (next) prologue(K, D, i);
    }
  }
}

// Detector classes of every instance into a dense array (N_i bytes per instance, in order).
__global__ void k_gather_flags(DevState D, int32_t B, uint8_t* out) {
  for (int i = blockIdx.x; i < B; i += gridDim.x) {
    const InstConst ic = D.IC[i];
    const int64_t eb = ic.coff + 2 * (int64_t)i;
    for (int64_t c = threadIdx.x; c < ic.N; c += blockDim.x) out[ic.coff + c] = D.flags[eb + c + 1];
  }
}

// Max of the widths of one instance into S->Jmax[0] and S->Jmax[1] (used by swale_rhs and
// swale_rhs_noalloc, which evaluate a stage outside a step).
__global__ void k_widths_max(const double* __restrict__ J, int64_t N, DevScalars* S) {
  double m = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x)
    m = fmax(m, J[i]);
  block_max_to(&S->Jmax[0], m);
}

}  // namespace swale_dev
