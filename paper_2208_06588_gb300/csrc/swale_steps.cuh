// Whole SSP-RK3 steps in one launch, for meshes of up to five blocks an SM (93 thousand cells): there a step
// of the stage kernels is eight dependent launches of ten to twenty microseconds each, much of it launch, load
// and drain latency. Here the cells stay in registers across stages and steps.
#pragma once

#include "swale_kernels.cuh"

namespace swale_dev {

constexpr int kStepThreads = 128;
constexpr int kStepCells = kStepThreads - 6;  // cells a block owns: three on each side are its neighbours'

// Per-instance scratch of k_steps, zero at its launch. The maxima and status words of a step live in
// set (step mod 3); the next but one is cleared while a step runs.
struct StepScratch {
  unsigned int arrived;  // barrier arrivals since the launch, and kGaveUp
  unsigned int pad_;
  unsigned long long mx[3][6];  // A of the three stages, max J^(1), max J^(2), complement of min J^(1)
  unsigned int st[3][6];        // status bits raised before each of the step's barriers
};

// Barrier of the nb blocks of an instance: arrivals are counted in global memory and every block
// waits until all have come. All blocks are resident (a cooperative launch), so the wait ends; it is
// bounded all the same (`tries` polls). A block that runs out of them marks the counter, unless the last arrival has
// come meanwhile (one compare-and-swap decides), and no block passes this barrier then: all of an instance's
// blocks give up at the same one, so that they leave the state of the same step. (A mark set at the next barrier
// follows an arrival there, a count above this barrier's.)
constexpr int kBarrierTries = 1 << 22;  // (seconds)
constexpr unsigned int kGaveUp = 0x80000000u;
__device__ __forceinline__ bool meet(unsigned int* arrived, unsigned int target, int tries) {
  // (the release and the acquire order the whole block's accesses through the two block barriers)
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(arrived) : "memory");
  unsigned int v = 0;
  for (int i = 0; i < tries && v < target; ++i)  // (ends on a mark too)
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
  while (v < target) {  // (repeated once for every arrival at most: ends)
    const unsigned int old = atomicCAS(arrived, v, v | kGaveUp);
    v = old == v ? v | kGaveUp : old;
    __threadfence();
  }
  return v < kGaveUp || (v & ~kGaveUp) > target;
}
__device__ __forceinline__ bool inst_barrier(unsigned int* arrived, unsigned int nb, unsigned int& target, int tries) {
  target += nb;  // (at most 6 arrivals a step and block: far below kGaveUp)
  if (nb == 1) {
    __syncthreads();
    return true;
  }
  __shared__ bool ok;
  __syncthreads();
  if (threadIdx.x == 0) ok = meet(arrived, target, tries);
  __syncthreads();
  return ok;
}

// Pair differences and reciprocals kept in the thread's registers.
struct StepSink {
  double ip, it, iq, iv, de, dh;
  __device__ __forceinline__ void pair(double a, double b, double c) {
    ip = a;
    de = b;
    dh = c;
  }
  __device__ __forceinline__ void triple(double a) { it = a; }
  __device__ __forceinline__ void quad(double a) { iq = a; }
  __device__ __forceinline__ void quint(double a) { iv = a; }
};

// nsteps steps of every instance (fewer where it reaches t_end or stops on an error), the same
// arithmetic as the stage kernels, bit for bit. Block (instance, b) owns the cells b * 122 .. and keeps
// their state in registers, one cell per thread; per stage it reads three cells on either side
// from its neighbours (through L2), reconstructs one of them, so that the fluxes need no exchange,
// and meets the other blocks of the instance twice: after the wave speeds (alpha), and after the new
// stage values. Bound by the chain of a warp's FP64 instructions (64 cycles each, whatever the
// number of warps or lanes: about 170 a stage, 67 more where cells are open) and by
// the six barriers (one to two microseconds each with several blocks). 16 steps at N = 200 take 830 us (1599 by
// the stage kernels at first, 1077 by today's), at 16300 cells 862 (1554, 993); an accuracy run of N = 50 to
// t = 0.1 35 ms (79). One block per SM runs a warp on each
// sub-partition; hydrostatic and non-well-balanced schemes, static, profile and linear motion. PER_SM:
// blocks that an SM holds (2: 255 registers; 4: 128, 5: 96, the rest spilled).
template <int SCHEME, int PER_SM>
__global__ void __launch_bounds__(kStepThreads, PER_SM) k_steps(StepConst K, DevState D, StepScratch* scratch, const Tile* blocks,
                                                           int wave_rel1, long long nsteps) {
  constexpr int T = kStepThreads;
  __shared__ double rE[T + 8], rM[T + 8], rJ[T + 8];
  __shared__ ReconRows<T, SCHEME> rows;
  __shared__ double sR[4][T], sPair[4][T];  // right edges (eta, b, h, u); ip, it, de, dh of the pair that starts there
  __shared__ double sF[3][T], sG[2][T], sW[T + 1], sI[T];
  const int tid = threadIdx.x;
  const Tile tl = blocks ? blocks[blockIdx.x] : Tile{0, (int32_t)blockIdx.x};
  const InstConst ic = blocks ? D.IC[tl.inst] : D.ic1;
  DevScalars* S = D.S + tl.inst;
  StepScratch* X = scratch + tl.inst;
  const int32_t N = (int32_t)ic.N;
  const unsigned int nb = (unsigned)((N + kStepCells - 1) / kStepCells);
  unsigned int target = 0;
  const int32_t c = tl.c0 * kStepCells - 3 + tid;  // this thread's cell, and its left node
  const int64_t cb = ic.coff, nbase = ic.coff + tl.inst;
  const int32_t idx = (int32_t)(ic.coff + 2 * (int64_t)tl.inst) + c + 1;
  const bool in_own = tid >= 3 && tid < T - 3;
  const bool own = in_own && c < N;
  const bool has_node = c >= 0 && c <= N;
  const bool own_node = own || (c == N && tid >= 4 && tid <= T - 3);
  const bool mine = tid >= 2 && tid < T - 2 && c <= N;  // reconstructed
  const bool face = tid >= 3 && tid < T - 2 && c <= N;  // left interface of an owned cell, or the last one
  const bool real_cell = c >= -3 && c <= N + 2;
  const int32_t g = (int32_t)cb + (real_cell ? ghost(c, N, K.bc) : 0);  // where the cell's values come from
  const bool flip = K.bc == SWALE_BC_REFLECTIVE && (c < 0 || c >= N);
  const bool moving = K.mesh != SWALE_MESH_STATIC;

  // State at t_n.
  double q0[3] = {0.0, 0.0, 0.0}, J0 = 1.0, w = 0.0;
  if (own) {
    q0[0] = D.E0[g];
    q0[1] = D.M0[g];
    q0[2] = D.B0[g];
    J0 = D.J0[g];
  }
  double tn = S->t;
  const double Wbar = S->Wbar;
  long long taken = 0;
  unsigned int bits = 0;
  bool timeout = false, written = false;
  int done = 0;
  StepDt sd{S->dt, S->alpha1, S->sdiff, 0, 0};
  // Kept in shared memory, for want of registers (in registers an accuracy run at N = 50 takes 2.3 % longer, 16 steps at N = 200 and
  // 16300 2 %): max J^n, J^(1), J^(2), min J^n (written by the first thread behind a barrier of the
  // instance, read behind the next barrier of the block), and what the instance's first thread reports of the last step, A of the
  // stages, alpha_1 and the secant factor. Per thread its node and the node's profile.
  __shared__ double sJm[4], sEnd[5], sX[2][T];
  sX[0][tid] = has_node ? D.x[nbase + c] : 0.0;
  sX[1][tid] = has_node ? D.P[nbase + c] : 0.0;
  if (K.mesh == SWALE_MESH_LINEAR) w = sX[1][tid];
  if (tid == 0) {
    sJm[0] = sJm[1] = sJm[2] = bitsd(S->JmaxN);
    sJm[3] = bitsd(S->JminN);
    sEnd[0] = sEnd[1] = sEnd[2] = 0.0;
    sEnd[3] = S->alpha1;
    sEnd[4] = S->sdiff;
  }
  if (S->status & kErrBits) done = 1;
  // Mesh-only values, kept from stage 2 for the next step's stage 1 (the same mesh; every stage of a
  // static one).
  MeshRecips mr{0.0, 0.0, 0.0, 0.0, false, false, false, false};
  swale::PairRatio kept_pr{0.0, 0.0, 0.0, 0.0};
  swale::SourceRatio kept_sr{0.0, 0.0, 0.0};
  double iJ0 = 1.0;  // 1 / J^n of the thread's cell
  bool have_mesh = false;

  // The values of the cells that other threads own, for the next stage: read as soon as the barrier has
  // passed, beside the status and the maxima.
  double pe = 0.0, pm = 0.0, pb = 0.0, pj = 1.0, pi = 1.0;
  const bool foreign = !own && real_cell;
  auto fetch = [&](const double* gE, const double* gM, const double* gB, const double* gJ, const double* gi) {
    if (!foreign) return;
    pe = __ldcg(gE + g);
    pm = __ldcg(gM + g);
    pb = __ldcg(gB + g);
    pj = __ldcg(gJ + g);
    if (gi) pi = __ldcg(gi + g);
    if (flip) pm = -pm;
  };
  fetch(D.E0, D.M0, D.B0, D.J0, nullptr);

  while (taken < nsteps && !done) {
    if (K.t_end > 0.0 && tn >= K.t_end) {
      done = 1;
      break;
    }
    const int set = (int)(taken % 3);
    double qs[3] = {q0[0], q0[1], q0[2]}, Js = J0, iJs = iJ0, J1 = J0, iJ1 = iJ0, dJ = 0.0, Y[3] = {0.0, 0.0, 0.0};
    unsigned int err = 0;
#pragma unroll 1
    for (int stage = 1; stage <= 3; ++stage) {
      // The stage's cells: owned ones from registers, the others as their owners (or images) have them
      // (filler beyond the last ghost cell).
      const double ev = own ? qs[0] : pe, mv = own ? qs[1] : pm, bv = own ? qs[2] : pb, jv = own ? Js : pj;
      double iv = own ? iJs : pi;
      if (stage == 1 && taken == 0) {
        iv = swale::recip(jv);
        if (own) iJ0 = iv;
      }
      rE[tid] = ev;
      rM[tid] = mv;
      rJ[tid] = jv;
      sI[tid] = iv;
      sW[tid] = w;
      const double hv = swale::sub_(ev, bv);
      const bool keep = have_mesh && (stage == 1 || !moving);
      mr.pair = mr.next = mr.all_pair = mr.all_next = keep;
      StepSink sink{mr.ip, mr.it, mr.iq, mr.iv, 0.0, 0.0};
      EdgeState o{0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
      uint8_t flag = 0;
      swale::PointPair pts{0.0, 0.0};
      uint32_t st = 0;
      recon_phases<T, SCHEME, 16>(K.sc, rows, rE, rM, rJ, jv, ev, mv, hv, sJm[stage - 1], mr, mine, sink,
                              o, flag, pts, st);
      if (stage == 2 || !moving) {
        mr.ip = sink.ip;
        mr.it = sink.it;
        mr.iq = sink.iq;
        mr.iv = sink.iv;
      }
      if (stage == 1 && own) D.flags[idx] = flag;
      sR[0][tid] = o.ER;
      sR[1][tid] = o.BR;
      sR[2][tid] = o.hR;
      sR[3][tid] = o.uR;
      sPair[0][tid] = sink.ip;
      sPair[1][tid] = sink.it;
      sPair[2][tid] = sink.de;
      sPair[3][tid] = sink.dh;
      const bool rel = stage == 1 ? wave_rel1 : K.wave_rel;
      block_wave<T>(&X->mx[set][stage - 1], 0.0, K.sc.g, mine && c != -1, mine && c != N,
                    WaveEdge{o.hL, o.uL, rel ? w : 0.0}, WaveEdge{o.hR, o.uR, rel && tid < T - 1 ? sW[tid + 1] : 0.0});
      block_or_status(&X->st[set][2 * stage - 2], st);
      if (!inst_barrier(&X->arrived, nb, target, K.barrier_tries)) {
        timeout = true;
        break;
      }
      const double A = bitsd(__ldcg(&X->mx[set][stage - 1]));
      const unsigned int raised = __ldcg(&X->st[set][2 * stage - 2]);
      if (tid == 0) sEnd[stage - 1] = A;
      bits |= raised;
      err = raised & kErrBits;
      if (err) break;
      double alpha;
      if (stage == 1) {
        // Everybody has left the last step's set: it is cleared for the step after the next one.
        if (tl.c0 == 0 && tid < 12) {
          const int z = (int)((taken + 2) % 3);
          if (tid < 6) X->mx[z][tid] = 0ull;
          else X->st[z][tid - 6] = 0u;
        }
        sd = step_dt(ic.cfl, wave_rel1 ? A : A + Wbar, 0.0, sJm[3], tn, K.dt_fixed, K.t_end,
                     K.mesh == SWALE_MESH_PROFILE ? K.inv_T : 0.0);
        if (sd.nodt) {
          err = swale::ST_NODT;
          bits |= err;
          break;
        }
        if (tid == 0) {
          sEnd[3] = sd.alpha1;
          sEnd[4] = sd.sdiff;
        }
        if (K.mesh == SWALE_MESH_PROFILE) w = swale::mul_(sX[1][tid], sd.sdiff);
        sW[tid] = w;
        alpha = sd.alpha1;
      } else {
        alpha = A;
        if (!K.wave_rel) alpha = swale::add_(A, Wbar);
      }
      const double dt = sd.dt;
      // Left interface of the cell: its left state is the right edge of cell c - 1.
      swale::Flux2 F{0.0, 0.0, 0.0, 0.0};
      swale::PairRatio pr = kept_pr;
      swale::SourceRatio sr = kept_sr;
      double dE = 0.0, dH = 0.0;
      if (face) {
        dE = sPair[2][tid - 1];
        dH = sPair[3][tid - 1];
        if (!keep) pr = swale::pair_ratio(rJ[tid - 1], jv, sPair[0][tid - 1]);
        F = swale::interface_flux2<SCHEME>(K.sc.g, alpha, w, sR[0][tid - 1], o.EL, sR[1][tid - 1], o.BL, sR[2][tid - 1],
                                           o.hL, sR[3][tid - 1], o.uL);
        sF[0][tid] = F.FE;
        sF[1][tid] = F.FMl;
        sF[2][tid] = F.FB;
        sG[0][tid] = pr.sig;
        sG[1][tid] = pr.rho2;
      }
      __syncthreads();
      double jmaxa = 0.0, jmaxb = 0.0, jminb = INFINITY;
      st = 0;
      if (own) {
        if (!keep) sr = swale::source_ratio(rJ[tid - 1], jv, rJ[tid + 1], sI[tid - 1], sI[tid + 1], sPair[1][tid - 1]);
        double Rm = swale::sub_(F.FMr, sF[1][tid + 1]);
        const double acc = swale::source_pressure_form(hv, o.hL, o.hR, swale::sub_(o.EL, ev), swale::sub_(o.ER, ev), dE, dH,
                                                       sink.de, sink.dh, pr.rho, pr.sig2, sG[0][tid + 1], sG[1][tid + 1], sr);
        Rm = swale::fma_(-K.sc.g, acc, Rm);
        const double R2[3] = {swale::sub_(F.FE, sF[0][tid + 1]), Rm, swale::sub_(sF[2][tid + 1], F.FB)};
        if (stage == 1) {
          dJ = swale::mul_(dt, swale::sub_(sW[tid + 1], w));
          J1 = swale::add_(J0, dJ);
          Js = J1;
          const double J2 = swale::fma_(0.5, dJ, J0);
          jmaxa = J1;
          jmaxb = J2;
          jminb = J1;
          if (!swale::gt0(J1) || !swale::gt0(J2)) st |= swale::ST_EMESH;
          iJ1 = moving ? swale::recip(J1) : iv;
          iJs = iJ1;
          const double hdt = swale::down_<1>(dt);
#pragma unroll
          for (int v = 0; v < 3; ++v) {
            Y[v] = R2[v];
            qs[v] = swale::rk_advance(q0[v], hdt, R2[v], dJ, iJ1);
          }
          D.J1[g] = J1;
          D.iJ1[g] = iJ1;
          D.Ea[g] = qs[0];
          D.Ma[g] = qs[1];
          D.Ba[g] = qs[2];
        } else if (stage == 2) {
          Js = swale::fma_(0.5, dJ, J0);
          iJs = moving ? swale::recip(Js) : iv;
          const double edt = swale::down_<3>(dt), hdJ = 0.5 * dJ;
#pragma unroll
          for (int v = 0; v < 3; ++v) {
            Y[v] = swale::add_(Y[v], R2[v]);
            qs[v] = swale::rk_advance(q0[v], edt, Y[v], hdJ, iJs);
          }
          D.J2[g] = Js;
          D.iJ2[g] = iJs;
          D.Eb[g] = qs[0];
          D.Mb[g] = qs[1];
          D.Bb[g] = qs[2];
        } else {
          const double tdt = dt * (1.0 / 12.0);
#pragma unroll
          for (int v = 0; v < 3; ++v) qs[v] = swale::rk_advance(q0[v], tdt, swale::fma_(4.0, R2[v], Y[v]), dJ, iJ1);
          if (swale::bad(qs[0]) || swale::bad(qs[1]) || swale::bad(qs[2])) st |= swale::ST_NONFINITE;
          D.E0[g] = qs[0];
          D.M0[g] = qs[1];
          D.B0[g] = qs[2];
          D.J0[g] = J1;
        }
      }
      if (stage == 1 && moving) block_widths<T, true>(&X->mx[set][3], &X->mx[set][5], jmaxa, jmaxb, jminb);
      block_or_status(&X->st[set][2 * stage - 1], st);
      if (stage == 2 || !moving) {
        kept_pr = pr;
        kept_sr = sr;
        have_mesh = true;
      }
      if (!inst_barrier(&X->arrived, nb, target, K.barrier_tries)) {
        timeout = true;
        written = stage == 3;
        break;
      }
      if (stage == 1) fetch(D.Ea, D.Ma, D.Ba, D.J1, D.iJ1);
      else if (stage == 2) fetch(D.Eb, D.Mb, D.Bb, D.J2, D.iJ2);
      else fetch(D.E0, D.M0, D.B0, D.J0, D.iJ1);
      const unsigned int raised2 = __ldcg(&X->st[set][2 * stage - 1]);
      if (stage == 1 && moving && tid == 0) {
        sJm[1] = bitsd(__ldcg(&X->mx[set][3]));
        sJm[2] = bitsd(__ldcg(&X->mx[set][4]));
      }
      bits |= raised2;
      err = raised2 & kErrBits;
      if (err) {
        if (stage == 3 && own) {  // the step failed after its cells were written: q^n, J^n back
          D.E0[g] = q0[0];
          D.M0[g] = q0[1];
          D.B0[g] = q0[2];
          D.J0[g] = J0;
        }
        break;
      }
    }
    if (timeout) break;
    if (err) {
      done = 1;
      break;
    }
    // The step is good.
#pragma unroll
    for (int v = 0; v < 3; ++v) q0[v] = qs[v];
    J0 = J1;
    iJ0 = iJ1;
    sX[0][tid] = swale::fma_(sd.dt, w, sX[0][tid]);
    if (moving && tid == 0) {
      sJm[0] = sJm[1];
      sJm[3] = bitsd(~__ldcg(&X->mx[set][5]));
    }
    tn = sd.clipped ? K.t_end : tn + sd.dt;
    ++taken;
  }
  if (timeout) {  // (not folded into the steps' error path: that costs 100 bytes of spills a thread, 2 to 5 % of the time)
    if (written && own) {  // the step's cells are written: q^n, J^n back
      D.E0[g] = q0[0];
      D.M0[g] = q0[1];
      D.B0[g] = q0[2];
      D.J0[g] = J0;
    }
    bits |= swale::ST_TIMEOUT;
    done = 1;
  }
  if (own_node && taken > 0) D.x[nbase + c] = sX[0][tid];
  if (tl.c0 == 0 && tid == 0) {
    S->status |= bits;
    S->done = done;
    S->t = tn;
    S->steps += taken;
    S->step_idx = S->steps;
    S->dt = sd.dt;
    S->alpha1 = sEnd[3];
    S->sdiff = sEnd[4];
    S->clipped = sd.clipped;
    for (int s = 0; s < 3; ++s) S->A[s] = dbits(sEnd[s]);
    S->Jmax[0] = S->JmaxN = dbits(sJm[0]);
    S->Jmin0 = S->JminN = dbits(sJm[3]);
    S->Jmax[1] = dbits(sJm[1]);
    S->Jmax[2] = dbits(sJm[2]);
    S->geo_tag = 0ull;
  }
}

// A width as a candidate for the largest: its bit pattern, zero for a negative one or a NaN (whose patterns lie above
// infinity's), so that a bad cell spoils its neighbours only.
__device__ __forceinline__ unsigned long long width_bits(double J) {
  const unsigned long long b = dbits(J);
  return b <= 0x7ff0000000000000ull ? b : 0ull;
}

// Largest of n widths, by one block, into *out; *wave (if given) is cleared.
__global__ void __launch_bounds__(1024) k_rhs_widths(const double* __restrict__ J, int32_t n, unsigned long long* out,
                                                     unsigned long long* wave) {
  __shared__ unsigned long long red[32];
  unsigned long long m = 0ull;
  pdl_wait();
  pdl_trigger();
#pragma unroll 8
  for (int32_t i = threadIdx.x; i < n; i += 1024) m = umax64(m, width_bits(J[i]));
  m = warp_umax64(m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = warp_umax64(red[threadIdx.x]);
    if (threadIdx.x == 0) {
      *out = m;
      if (wave) *wave = 0ull;
    }
  }
}

// One right-hand side for a given viscosity in one launch: alpha is known, so the fluxes need no grid-wide
// maximum between them and the reconstruction, and the edge values stay on the chip (a block owns 122
// cells and reconstructs one more on each side, as in k_steps). dxmax: the largest width, or null: every block
// scans the N widths (cheaper than a launch of its own up to 8192 cells). Bound by the chain of a warp's 139 FP64
// instructions (64 cycles each, 4.3 us) and the loads before it: 11.6 us a call at N = 200 (30.7 as stage kernels with
// their launches), 27 at 65536 (59), where FP64 throughput is the bound. wave: where the largest
// edge speed goes (null: not wanted), relative to w if wave_rel.
template <int SCHEME>
__global__ void __launch_bounds__(kStepThreads, 4) k_rhs(SchemeConst P, int bc, int wave_rel, int32_t N, double alpha,
                                                         const double* __restrict__ E, const double* __restrict__ M,
                                                         const double* __restrict__ B, const double* __restrict__ J,
                                                         const double* __restrict__ w, const unsigned long long* dxmax,
                                                         unsigned long long* wave, double* __restrict__ RE,
                                                         double* __restrict__ RM, double* __restrict__ RB,
                                                         uint8_t* __restrict__ flags) {
  constexpr int T = kStepThreads;
  __shared__ double rE[T + 8], rM[T + 8], rJ[T + 8];
  __shared__ ReconRows<T, SCHEME> rows;
  __shared__ double sR[4][T], sBL[T], sPair[4][T];  // right edges, left bottoms; ip, it, de, dh of the pair that starts there
  __shared__ double sF[3][T], sG[2][T], sB[T], sI[T];
  __shared__ unsigned long long red[T / 32];
  const int tid = threadIdx.x;
  const int32_t c = (int32_t)blockIdx.x * kStepCells - 3 + tid;  // this thread's cell, and its left node
  const bool own = tid >= 3 && tid < T - 3 && c < N;
  const bool mine = tid >= 2 && tid < T - 2 && c <= N;  // reconstructed
  const bool face = tid >= 3 && tid < T - 2 && c <= N;  // left interface of an owned cell, or the last one
  pdl_wait();
  double ev = 0.0, mv = 0.0, bv = 0.0, jv = 1.0, wl = 0.0, wr = 0.0;
  if (c >= -3 && c <= N + 2) {
    const int32_t g = ghost(c, N, bc);
    ev = E[g];
    mv = M[g];
    bv = B[g];
    jv = J[g];
    if (bc == SWALE_BC_REFLECTIVE && (c < 0 || c >= N)) mv = -mv;
    if (c >= 0 && c <= N) wl = w[c];
    if (c >= -1 && c < N) wr = w[c + 1];
  }
  double dx;
  if (dxmax || !P.beta_dx_global) {
    dx = dxmax ? bitsd(*dxmax) : 0.0;
  } else {
    unsigned long long m = 0ull;
#pragma unroll 4
    for (int32_t i = tid; i < N; i += T) m = umax64(m, width_bits(J[i]));
    m = warp_umax64(m);
    if ((tid & 31) == 0) red[tid >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < T / 32; ++k) m = umax64(m, red[k]);
    dx = bitsd(m);
  }
  rE[tid] = ev;
  rM[tid] = mv;
  rJ[tid] = jv;
  sB[tid] = bv;
  const double hv = swale::sub_(ev, bv), iv = swale::recip(jv);
  sI[tid] = iv;
  const MeshRecips none{0.0, 0.0, 0.0, 0.0, false, false, false, false};
  StepSink sink{0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  EdgeState o{0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  uint8_t flag = 0;
  swale::PointPair pts{0.0, 0.0};
  uint32_t st = 0;
  recon_phases<T, SCHEME, 16>(P, rows, rE, rM, rJ, jv, ev, mv, hv, dx, none, mine, sink, o, flag, pts, st);
  if (own && flags) flags[c] = flag;
  sR[0][tid] = o.ER;
  sR[1][tid] = o.BR;
  sR[2][tid] = o.hR;
  sR[3][tid] = o.uR;
  sBL[tid] = o.BL;
  sPair[0][tid] = sink.ip;
  sPair[1][tid] = sink.it;
  sPair[2][tid] = sink.de;
  sPair[3][tid] = sink.dh;
  if (wave)
    block_wave<T>(wave, 0.0, P.g, mine && c != -1, mine && c != N, WaveEdge{o.hL, o.uL, wave_rel ? wl : 0.0},
                  WaveEdge{o.hR, o.uR, wave_rel ? wr : 0.0});
  __syncthreads();
  swale::Flux2 F{0.0, 0.0, 0.0, 0.0};
  swale::PairRatio pr{0.0, 0.0, 0.0, 0.0};
  if (face) {
    pr = swale::pair_ratio(rJ[tid - 1], jv, sPair[0][tid - 1]);
    F = swale::interface_flux2<SCHEME>(P.g, alpha, wl, sR[0][tid - 1], o.EL, sR[1][tid - 1], o.BL, sR[2][tid - 1], o.hL,
                                       sR[3][tid - 1], o.uL);
    sF[0][tid] = F.FE;
    sF[1][tid] = F.FMl;
    sF[2][tid] = F.FB;
    sG[0][tid] = pr.sig;
    sG[1][tid] = pr.rho2;
  }
  __syncthreads();
  pdl_trigger();
  if (!own) return;
  double Rm = swale::sub_(F.FMr, sF[1][tid + 1]);
  if (SCHEME == 2) {
    const double bd[5] = {sB[tid - 1], bv, sB[tid + 1], o.BL, o.BR};
    const swale::SourceGeom sg = swale::source_geom(rJ[tid - 1], jv, sI[tid - 1], iv, sI[tid + 1], sPair[0][tid - 1],
                                                    sink.ip, sPair[1][tid - 1]);
    Rm = swale::add_(Rm, swale::source_special2(P.g, ev, o.EL, o.ER, pts, bd, sg, sR[1][tid - 1], sBL[tid + 1]));
  } else {
    const swale::SourceRatio sr =
        swale::source_ratio(rJ[tid - 1], jv, rJ[tid + 1], sI[tid - 1], sI[tid + 1], sPair[1][tid - 1]);
    const double acc = swale::source_pressure_form(hv, o.hL, o.hR, swale::sub_(o.EL, ev), swale::sub_(o.ER, ev),
                                                   sPair[2][tid - 1], sPair[3][tid - 1], sink.de, sink.dh, pr.rho, pr.sig2,
                                                   sG[0][tid + 1], sG[1][tid + 1], sr);
    Rm = swale::fma_(-P.g, acc, Rm);
  }
  RE[c] = 0.5 * swale::sub_(F.FE, sF[0][tid + 1]);
  RM[c] = 0.5 * Rm;
  RB[c] = 0.5 * swale::sub_(sF[2][tid + 1], F.FB);
}

}  // namespace swale_dev
