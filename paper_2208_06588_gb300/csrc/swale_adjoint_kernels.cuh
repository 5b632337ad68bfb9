// Device kernels of the discrete adjoint of one SSP-RK3 step (Eq. RK32D) of the well-balanced
// ALE-WENO hybrid scheme: one kernel per stage reverses its RK combination, fluxes, source,
// limiter and reconstruction, and the gauge misfit seeds the adjoint of the state.
#pragma once

#include "swale_adjoint.cuh"
#include "swale_kernels.cuh"

namespace swale_dev {

// What the reverse of a stage reads per cell besides its edge states, kept by the recompute's kernels
// in DevState::gK (ADJ_*): reciprocal sums of four and five widths, the interfaces' width ratios and the
// source's, the class (0, 1, 2, plus 4 where the limiter acted), and the differences and depths of the
// stage (DevState::dE, dH, H point there).
static_assert(ADJ_ARRAYS <= 14, "swale_adjoint_bytes counts 14 arrays per stage");

// Adjoint work arrays (concatenated like the state).
struct AdjState {
  const double *lE, *lM, *lB;  // lambda: adjoint of q^{n+1}
  double *oE, *oM, *oB;        // adjoint of q^n (another buffer: neighbours still read lambda)
  double *a3[3], *a2[3];       // adjoints of the inputs of stages 3 and 2
  const double *sJ;            // J^n of the step being reversed
  const Tile* tiles;           // blocks (instance, index), null: one instance
};

constexpr int kAdjThreads = 128;
constexpr int kAdjCells = kAdjThreads - 8;  // cells a block owns at most: four on each side are its neighbours'

// Cells of block b of an instance of N cells: the blocks are balanced, so that the last three cells of
// an instance, whose ghost images the block folds back itself, are in one block.
__device__ __host__ __forceinline__ int32_t adj_blocks(int64_t N) { return (int32_t)((N + kAdjCells - 1) / kAdjCells); }
__device__ __forceinline__ int32_t adj_first(int32_t b, int32_t nb, int32_t N) { return (int32_t)((int64_t)b * N / nb); }

// The reverse of a cell that is not smooth or whose limiter acted, out of line.
struct AdjCellIn {
  double J[5], E[5], M[5], H[5];
  swale::EdgeAdj ob;
};
struct AdjCellOut {
  swale::SmoothAdj s[3];
};
__device__ __noinline__ AdjCellOut adj_general_cell(const SchemeConst P, const AdjCellIn c, double dxmax) {
  AdjCellOut r;
  swale::cell_rev_general(P, c.J, c.E, c.M, c.H, dxmax, c.ob, r.s);
  return r;
}

// Reverse of stage STAGE. With Y3 = lambda / J^{n+1}, y2 = (2/3) Y3 + a3 / J^(2), y1 = y2 / 4 + a2 / J^(1) (a_s the adjoint of
// stage s's input), twice the stages' right-hand sides have the adjoints dt Y3 / 3, dt y2 / 8, dt y1 / 2, and the
// adjoint of q^n is J^n (Y3 / 3 + 3 y2 / 4 + y1) + a1: every block forms these for its cells and their
// neighbours from lambda, a3 and a2, which nobody writes meanwhile, so no kernel of its own
// combines them. A block owns up to 120 cells, one per thread, and takes four more on each side: it
// gathers what falls on its cells from the cells and interfaces around them (the transpose of the
// differences runs through shared memory, order by order, as the forward builds them), instead of
// scattering 15 atomic additions per cell; ghost cells' shares are folded back to their images.
// Per cell 224 to 249 FP64 instructions, which bound it: 38-41 us a stage at 65536 cells, the FP64 pipe 77 % busy,
// against 61 us of the four kernels that scattered (3, 4, 5 and 6 blocks on an SM are within 1 %); in a smooth cell whose limiter did not act
// nothing of the forward is formed again but the source's functionals.
// E, M, B, J: the stage's input and widths. Runs are bitwise reproducible up to the misfit's seeds.
template <int STAGE>
__global__ void __launch_bounds__(kAdjThreads, 4) k_adj_stage(StepConst K, DevState D, AdjState A, const double* __restrict__ Eg,
                                                              const double* __restrict__ Mg, const double* __restrict__ Bg,
                                                              const double* __restrict__ Jg) {
  constexpr int T = kAdjThreads;
  __shared__ double rE[T], rM[T], rH[T], rJ[T + 4];
  __shared__ double sRho[3][T], sR[4][T], sX[3][T], sDl[2][T];
  __shared__ double sD2l[3][T], sD3[3][T], sD4l[3][T], sD4r[3][T], sT[3][T];
  const int tid = threadIdx.x;
  pdl_wait();
  const Tile tl = A.tiles ? A.tiles[blockIdx.x] : Tile{0, (int32_t)blockIdx.x};
  const InstConst ic = A.tiles ? D.IC[tl.inst] : D.ic1;
  const DevScalars* S = D.S + tl.inst;
  const int32_t N = (int32_t)ic.N, nb = adj_blocks(N);
  const int32_t first = adj_first(tl.c0, nb, N), last = adj_first(tl.c0 + 1, nb, N);  // owned cells [first, last)
  const int32_t c = first - 4 + tid;
  const bool own = tid >= 4 && c < last;
  const bool near = c <= last + 3;  // within the cells that contribute
  const bool per = K.bc == SWALE_BC_PERIODIC;
  // A cell of the domain (periodic: of its continuation), one whose edges were reconstructed, an interface.
  const bool real = near && (per || (c >= 0 && c < N));
  const bool recon = near && (per || (c >= -1 && c <= N));
  const bool face = near && tid >= 1 && (per || (c >= 0 && c <= N));
  const int32_t gl = near ? ghost(c, N, K.bc) : 0;          // where its averages lie
  const int32_t g = (int32_t)ic.coff + gl;
  const int32_t eb = (int32_t)(ic.coff + 2 * (int64_t)tl.inst);
  const int32_t e = eb + (recon ? (per ? gl : c) + 1 : 1);  // its edge-array index
  const bool flip = K.bc == SWALE_BC_REFLECTIVE && (c < 0 || c >= N);
  const double dt = S->dt, dxmax = bitsd(S->Jmax[STAGE - 1]);
  double alpha = (STAGE == 1) ? S->alpha1 : bitsd(S->A[STAGE - 1]) + S->Wbar;
  if (STAGE > 1 && K.alpha_mode == 2) alpha = stage_alpha(K, tl.inst, STAGE, alpha, S->step_idx);

  const double ev = Eg[g], jv = near ? Jg[g] : 1.0;
  const double hv = swale::sub_(ev, Bg[g]);
  rE[tid] = ev;
  rM[tid] = flip ? -Mg[g] : Mg[g];
  rH[tid] = hv;
  rJ[tid] = jv;
  double q[3] = {0.0, 0.0, 0.0};  // Y3 / 3 + 3 y2 / 4 + y1 (stage 1)
  {
    double rho[3] = {0.0, 0.0, 0.0};
    if (real) {
      const double i1 = swale::recip(D.J1[g]);  // J^{n+1} = J^(1)
      const double i2 = STAGE < 3 ? swale::recip(D.J2[g]) : 0.0;
      const double l[3] = {A.lE[g], A.lM[g], A.lB[g]};
#pragma unroll
      for (int v = 0; v < 3; ++v) {
        const double Y3 = l[v] * i1;
        if (STAGE == 3) {
          rho[v] = (1.0 / 3.0) * dt * Y3;
        } else {
          const double y2 = (2.0 / 3.0) * Y3 + A.a3[v][g] * i2;
          if (STAGE == 2) {
            rho[v] = 0.125 * dt * y2;
          } else {
            const double y1 = 0.25 * y2 + A.a2[v][g] * i1;
            rho[v] = 0.5 * dt * y1;
            q[v] = (1.0 / 3.0) * Y3 + (0.75 * y2 + y1);
          }
        }
      }
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) sRho[v][tid] = rho[v];
  }
  // Edge state of the cell; its right edge for the interface on its right.
  swale::EdgeState o{0.0, 0.0, 0.0, 0.0, 1.0, 1.0, 0.0, 0.0};
  if (recon) o = {D.eEL[e], D.eER[e], D.eBL[e], D.eBR[e], D.ehL[e], D.ehR[e], D.euL[e], D.euR[e]};
  sR[0][tid] = o.ER;
  sR[1][tid] = o.BR;
  sR[3][tid] = o.uR;
  __syncthreads();
  // Fluxes: interface c, between cells c - 1 and c. The right edge of cell c - 1 gets its share through sX.
  swale::FaceAdj f{0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (face) {
    // (A periodic domain whose end nodes move apart: each cell has its own end's velocity.)
    const double* wv = D.w + ic.coff + tl.inst;
    const bool moving = K.mesh != SWALE_MESH_STATIC;
    const double wr = moving ? wv[per ? gl : c] : 0.0, wl = moving && per && gl == 0 ? wv[N] : wr;
    const double* l = &sRho[0][tid - 1];
    const double* r = &sRho[0][tid];
    const bool both = wl == wr;
    for (int p = both ? 1 : 0; p < 2; ++p) {  // p = 1: the right cell's share (or both), 0: the left one's
      const double zl = p && !both ? 0.0 : 1.0, zr = p ? 1.0 : 0.0;
      const swale::FaceAdj h = swale::interface_flux2_rev(K.sc.g, alpha, p ? wr : wl, sR[0][tid - 1], o.EL, sR[1][tid - 1],
                                                          o.BL, sR[3][tid - 1], o.uL, zr * r[0] - zl * l[0], -(zl * l[T]),
                                                          zr * r[T], zl * l[2 * T] - zr * r[2 * T]);
      f.EL += h.EL;
      f.BL += h.BL;
      f.uL += h.uL;
      f.ER += h.ER;
      f.BR += h.BR;
      f.uR += h.uR;
    }
  }
  sX[0][tid] = f.EL;
  sX[1][tid] = f.BL;
  sX[2][tid] = f.uL;
  __syncthreads();
  const bool inner = recon && tid < T - 1;
  swale::EdgeAdj ob{f.ER, 0.0, f.BR, 0.0, 0.0, 0.0, f.uR, 0.0};
  if (inner) {
    ob.ER = sX[0][tid + 1];
    ob.BR = sX[1][tid + 1];
    ob.uR = sX[2][tid + 1];
  }
  // Pressure and source.
  double Eb = 0.0, Hb = 0.0, dEr = 0.0, dHr = 0.0, dEl = 0.0, dHl = 0.0;
  if (real && tid >= 1 && tid < T - 1) {
    const int64_t gs = D.geo_stride;
    const double* G = D.gK;
    // the interfaces' ratios are stored at the edge index of their left cell, the differences too
    const int32_t el = per ? eb + ghost(c - 1, N, K.bc) + 1 : e - 1;
    const double rho_l = G[ADJ_RHO * gs + el], sig_l = G[ADJ_SIG * gs + el], rho_r = G[ADJ_RHO * gs + e],
                 sig_r = G[ADJ_SIG * gs + e];
    const swale::SourceRatio sr = {G[ADJ_GX * gs + e], G[ADJ_GY * gs + e], G[ADJ_K3 * gs + e]};
    const swale::SourceAdj a = swale::source_pressure_rev(
        hv, o.hL, o.hR, o.EL - ev, o.ER - ev, D.dE[el], D.dH[el], D.dE[e], D.dH[e], rho_l, sig_l * sig_l, sig_r,
        rho_r * rho_r, sr, -(K.sc.g * sRho[1][tid]));
    ob.hL = a.hL;
    ob.hR = a.hR;
    ob.EL += a.deL;
    ob.ER += a.deR;
    Eb = -(a.deL + a.deR);
    Hb = a.hc;
    dEl = a.dEl;
    dHl = a.dHl;
    dEr = a.dEr;
    dHr = a.dHr;
  }
  sDl[0][tid] = dEl;
  sDl[1][tid] = dHl;
  // Limiter and reconstruction.
  swale::SmoothAdj r[3] = {};
  if (recon && tid >= 2 && tid < T - 2) {
    const int cls = (int)D.gK[ADJ_CLS * D.geo_stride + e];
    if (cls == 0) {  // smooth, limiter not active
      const swale::SmoothWidths w = {rJ[tid - 1], jv, rJ[tid + 1], rJ[tid - 2] + rJ[tid - 1], rJ[tid - 1] + jv,
                                     jv + rJ[tid + 1], rJ[tid + 1] + rJ[tid + 2]};
      const double iv = D.gK[ADJ_IV * D.geo_stride + e];
      // B = E - h and u = m / h on wet edges
      const bool wetL = swale::gt_pos(o.hL, K.sc.h_dry), wetR = swale::gt_pos(o.hR, K.sc.h_dry);
      const double hLs = wetL ? o.hL : 1.0, hRs = wetR ? o.hR : 1.0, ihh = swale::recip(hLs * hRs);
      const double mL = wetL ? ob.uL * (hRs * ihh) : 0.0, mR = wetR ? ob.uR * (hLs * ihh) : 0.0;
      r[0] = swale::smooth_rev(w, iv, ob.EL + ob.BL, ob.ER + ob.BR);
      r[1] = swale::smooth_rev(w, iv, mL, mR);
      r[2] = swale::smooth_rev(w, iv, (ob.hL - ob.BL) - mL * o.uL, (ob.hR - ob.BR) - mR * o.uR);
    } else {
      AdjCellIn in;
      in.ob = ob;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        in.J[k] = rJ[tid - 2 + k];
        in.E[k] = rE[tid - 2 + k];
        in.M[k] = rM[tid - 2 + k];
        in.H[k] = rH[tid - 2 + k];
      }
      const AdjCellOut ro = adj_general_cell(K.sc, in, dxmax);
#pragma unroll
      for (int v = 0; v < 3; ++v) r[v] = ro.s[v];
    }
  }
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    sD2l[v][tid] = r[v].d2l;
    sD3[v][tid] = r[v].d3;
    sD4l[v][tid] = r[v].d4l;
    sD4r[v][tid] = r[v].d4r;
  }
  // Reciprocal sums of the pair, triple and quadruple that start at this cell: as stored for cells
  // -1..N (the triple and quadruple by their second cell), formed for the outer ghost cells.
  double ip = 0.0, it = 0.0, iq = 0.0;
  if (near) {
    const int32_t cp = per ? gl : c, cn = per ? ghost(c + 1, N, K.bc) : c + 1;
    if (cp >= -1 && cp <= N) ip = D.ipair[eb + cp + 1];
    else if (tid < T - 1) ip = swale::recip(jv + rJ[tid + 1]);
    if (cn >= -1 && cn <= N) {
      it = D.itri[eb + cn + 1];
      iq = D.gK[ADJ_IQ * D.geo_stride + eb + cn + 1];
    } else if (tid < T - 3) {
      const double p = jv + rJ[tid + 1];
      it = swale::recip(p + rJ[tid + 2]);
      iq = swale::recip(p + (rJ[tid + 2] + rJ[tid + 3]));
    }
  }
  __syncthreads();
  // Transpose of the differences: quadruples, triples, pairs, cells (rows past the block count as zero).
#pragma unroll
  for (int v = 0; v < 3; ++v) sT[v][tid] = tid < T - 2 ? (sD4l[v][tid + 2] + sD4r[v][tid + 1]) * iq : 0.0;
  __syncthreads();
  double t3[3];
#pragma unroll
  for (int v = 0; v < 3; ++v)
    t3[v] = tid < T - 1 ? (sD3[v][tid + 1] + ((tid > 0 ? sT[v][tid - 1] : 0.0) - sT[v][tid])) * it : 0.0;
#pragma unroll
  for (int v = 0; v < 3; ++v) sD4l[v][tid] = t3[v];  // (read above as D4 shares, before the barrier)
  __syncthreads();
  const double src[3] = {dEr + (tid < T - 1 ? sDl[0][tid + 1] : 0.0), 0.0, dHr + (tid < T - 1 ? sDl[1][tid + 1] : 0.0)};
  double t2[3];
#pragma unroll
  for (int v = 0; v < 3; ++v) {
    const double s2 = (r[v].d2r + (tid < T - 1 ? sD2l[v][tid + 1] : 0.0)) + ((tid > 0 ? sD4l[v][tid - 1] : 0.0) - t3[v]);
    t2[v] = s2 * ip + src[v];
    sD4r[v][tid] = t2[v];
  }
  __syncthreads();
  double a[3];
#pragma unroll
  for (int v = 0; v < 3; ++v) a[v] = r[v].v + ((tid > 0 ? sD4r[v][tid - 1] : 0.0) - t2[v]);
  a[0] += Eb;
  a[2] += Hb;
  // (eta, hu, h) to (eta, hu, b): h = eta - b.
  a[0] += a[2];
  a[2] = -a[2];
  if (!per && (first < 3 || last > N - 3)) {  // ghost cells' shares go to their images
#pragma unroll
    for (int v = 0; v < 3; ++v) sD3[v][tid] = (flip && v == 1) ? -a[v] : a[v];
    __syncthreads();
    if (own) {
      if (c < 3) {  // image of cell -1 - c
#pragma unroll
        for (int v = 0; v < 3; ++v) a[v] += sD3[v][tid - (2 * c + 1)];
      }
      if (c >= N - 3) {  // image of cell 2 N - 1 - c
#pragma unroll
        for (int v = 0; v < 3; ++v) a[v] += sD3[v][tid + 2 * (N - 1 - c) + 1];
      }
    }
  }
  pdl_trigger();
  if (!own) return;
  if (STAGE == 1) {
    const double J0 = A.sJ[g];
    A.oE[g] = J0 * q[0] + a[0];
    A.oM[g] = J0 * q[1] + a[1];
    A.oB[g] = J0 * q[2] + a[2];
  } else {
#pragma unroll
    for (int v = 0; v < 3; ++v) (STAGE == 3 ? A.a3 : A.a2)[v][g] = a[v];
  }
}

// The evolving state of one context or state set (q^n, J^n, nodes, scalars) copied to another, in
// one launch: cells, nodes and 8-byte words of the scalars.
struct StateArrays {
  double *E, *M, *B, *J, *x;
  DevScalars* S;
};
__global__ void __launch_bounds__(256) k_copy_state(StateArrays to, StateArrays from, int64_t cells, int64_t nodes,
                                                    int64_t words) {
  static_assert(sizeof(DevScalars) % 8 == 0, "the scalars are copied in 8-byte words");
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  pdl_wait();
  pdl_trigger();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nodes || i < words; i += step) {
    if (i < cells) {
      to.E[i] = from.E[i];
      to.M[i] = from.M[i];
      to.B[i] = from.B[i];
      to.J[i] = from.J[i];
    }
    if (i < nodes) to.x[i] = from.x[i];
    if (i < words) ((long long*)to.S)[i] = ((const long long*)from.S)[i];
  }
}

// Gauge misfit of the state after a step: gauge g of instance i sits at x = gx[i * G + g]; its
// depth is the average of the cell that contains x on the current mesh. MODE 0 adds
// dt (h - obs)^2 to Jout[i]; MODE 1 adds its gradient 2 dt (h - obs) to lambda (eta: +, b: -).
// obs points at the row of the observed depths for this step (B x G values).
// gcell[id] caches the gauge's cell between calls (-1: not located yet): from there a short walk
// finds the cell on the new mesh (a node moves by less than a cell per step); the first call
// bisects. Either way the cell is c with x[c] <= xg < x[c+1] (clamped to 0..N-1).
template <int MODE>
__global__ void k_misfit(DevState D, double* lE, double* lB, int32_t B, int32_t G, const double* __restrict__ gx,
                         const double* __restrict__ obs, double* Jout, int64_t* gcell) {
  pdl_wait();
  pdl_trigger();
  const int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= (int64_t)B * G) return;
  const int i = (int)(id / G);
  const InstConst ic = D.IC[i];
  const double* x = D.x + ic.coff + i;
  const double xg = gx[id];
  int64_t lo = gcell[id];
  if (lo < 0 || lo >= ic.N) {
    lo = 0;
    int64_t hi = ic.N;
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (x[mid] <= xg) lo = mid;
      else hi = mid;
    }
  } else {
    while (lo + 1 < ic.N && x[lo + 1] <= xg) ++lo;
    while (lo > 0 && x[lo] > xg) --lo;
  }
  gcell[id] = lo;
  const int64_t g = ic.coff + lo;
  const double r = (D.E0[g] - D.B0[g]) - obs[id];
  const double dt = D.S[i].dt;
  if (MODE == 0) {
    atomicAdd(&Jout[i], dt * r * r);
  } else {
    atomicAdd(&lE[g], 2.0 * dt * r);
    atomicAdd(&lB[g], -2.0 * dt * r);
  }
}

}  // namespace swale_dev
