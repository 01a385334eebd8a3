// stepper.cuh -- the cluster time stepper: every backward-Euler solve of the pass.
//
// One thread-block cluster owns one independent time-stepping system (one Parareal slice,
// one coarse step, or the sequential correction sweep).  Its CTAs split the node rows into
// slabs held on chip (ptg_device.cuh); each thread owns NG aligned groups of 4 consecutive
// nodes of a row.  Each solve of (C/dt + K) x = b (Eq. 2.7 / 4.4) is a Jacobi-preconditioned
// CG in precision Real inside an FP64 residual loop:
//     r = b - A x            (FP64, per-node FP64 weights: 9 FMAs per node)
//     while ||r|| > rtol ||b||:   CG on A d = r / 2^k,  x += 2^k d,  r = b - A x
// With Real = double the CG works in pairs of floats (ff.cuh) on the same per-node weights and the
// first CG already meets the tolerance; with Real = float the CG uses FP32 element weights held in shared memory
// and this is iterative refinement with FP64 residuals.  CG carries q = A p by the recurrence
// q_{k+1} = A z_{k+1} + beta q_k, so z is the only stencil operand and an iteration has one
// exchange of its halo rows and one reduction.
//
// Task kinds (StepParams::kind), one task per cluster:
//   FINE_PRI    Alg. 1 repeated M times from u_s (or chained over slices), history written.
//   COARSE_PRI  Alg. 1 with dt -> dtau, Nt -> Ntau, one step ending at t_{M(s+1)}.
//   CORRECT_PRI Eq. 4.9 forward sweep: u_{s+1} = G(u_s) + F[s] - G_old[s].
//   FINE_ADJ    Alg. 2 repeated M times from v_{s+1} (or chained), g accumulated.
//   COARSE_ADJ  Alg. 2 with dt -> dtau, Nt -> Ntau, n+1 -> n+M, n-1 -> n-M.
//   CORRECT_ADJ Eq. 4.14 reverse sweep: v_s = G(v_{s+1}) + F[s] - G_old[s], v_Ntau = 0.
#pragma once
#include <type_traits>
#include "comm.cuh"
#include "ptg_device.cuh"
#include "ptg_internal.h"

namespace ptg {

// COARSE: the kinds that solve with C/dtau + K, which alone have the two-level preconditioners.
template <class Real, int NG, class Comm, bool COARSE>
struct Stepper {
  static constexpr bool kMixed = std::is_same<Real, float>::value;
  // the CG's vectors and scalars: floats, or float pairs for the FP64 kinds (ff.cuh)
  using V = typename std::conditional<kMixed, float, ff>::type;

  const StepParams& P;
  Comm& comm;
  Slab sb;
  // shared memory (each pointer at the first non-slack entry)
  double* x64;      // FP64 state, rows -1..R
  double* b64;      // FP64 right-hand side, rows 0..R-1
  float* zbuf;      // CG stencil operand, rows -1..R
  float* dinv;      // Jacobi inverse diagonal, rows 0..R-1 (0 on Dirichlet and pad nodes)
  float* wk = nullptr;  // FP32 element weights, element rows r0-1..r0+R-1 (FP32 CG, V-cycle): the conductivity
  float* wm = nullptr;  // and the capacity part, k_e / 6 and c_e h^2 / (36 step) (stencil_km32)
  // per-thread groups: loc0[k] = offset of the group's first node in the halo buffers, -1 if none
  int loc0[NG];
  unsigned fmask = 0;   // bit 4k+j: node j of group k is an unknown (free, not a pad)
  NodeWeights A;    // per-node FP64 weights of the current operator
  FFWeights ffw;    // the same as float pairs (FP64 kinds)
  double step_dt = 0.0;
  double inv_dt = 0.0;
  int gshift = 0;   // offset from a halo-buffer node to the same node of the global padded arrays
  double* ax64;     // A x64 from the last residual evaluation, rows 0..R-1 (reused by the next step;
                    // null when the plan leaves it out, P.keep_ax == 0)
  bool ax_valid = false;
  // two-level preconditioner of the coarse-step solves: see coarse_restrict_push
  bool tl = false;
  bool tl_loaded = false;
  int aj0 = 0, naj = 0;      // this CTA's aggregate rows [aj0, aj0 + naj)
  float* tl_ainv = nullptr;  // rows of Ainv for the CTA's aggregates, [naj * naxp][ncp]
  float* tl_slot = nullptr;  // restricted partials of every rank, [cs][ncp]
  float* tl_qc = nullptr;    // restricted vector summed over the covering ranks, [ncp]
  float* tl_ec = nullptr;    // coarse correction Ac^-1 P^T r on the CTA's aggregates, [naj * naxp]
  float* tl_gs = nullptr;    // group sums of the vector being restricted, [R * G]
  int* tl_gagg = nullptr;    // local aggregate (row-major in [naj][nax]) of every group, [R * G]
  int* tl_cov = nullptr;     // first / last rank covering each aggregate row, [nay][2]
  unsigned tl_bytes = 0;     // restricted partials that every rank receives from all ranks together
  // V(1,1) two-grid cycle (P.tl_vc), see vcycle; aj0 / naj then cover the halo rows too
  bool vc = false;
  int ajo0 = 0, najo = 0;    // aggregate rows of the owned rows (the restriction's partials)
  V* vrh = nullptr;       // r on the halo rows -1 and R, [2][W]
  float* vy = nullptr;       // y = S r, then u = y + P ec, rows -1..R
  float* vsd = nullptr;      // S = omega D^-1, rows -1..R (0 off the unknowns)
  float* ve0 = nullptr;      // slab-local smoothing (P.tl_nu >= 2): ping-pong iterates, rows -1..R,
  float* ve1 = nullptr;      // halo rows kept at zero
  // three-level cycle (P.tl_l3, see vcycle3): the 2h rows [J0, J0 + R1) of this CTA (R1b: those
  // of the CTA below), padded 2h row width W1, stride own1s of the owned-row 2h arrays
  bool l3 = false;
  int J0 = 0, R1 = 0, R1b = 0, W1 = 0, own1s = 0;
  // this thread's owned 2h nodes: offset in the halo buffers (-1 if none) and local aggregate
  static constexpr int K1 = NG + 1;
  int n1o[K1], n1a[K1];
  float* vw = nullptr;       // fine residual w0 = r - A e0, rows -1..R
  float* b1x = nullptr;      // 2h rows -1..R1: e1 = S1 r1 (halo rows from the neighbours)
  float* b1u = nullptr;      //                 u1 = e1 + P2 ec (owned and halo rows, computed here)
  float* b1z = nullptr;      //                 z1 = u1 + S1 (r1 - A1 u1) (halo rows from the neighbours)
  float* s1a = nullptr;      //                 slab-local smoothing iterates (halo rows kept at zero)
  float* s1b = nullptr;
  float* a1w = nullptr;      // [9][own1s] A1 weights of the owned 2h nodes, k = (dJ + 1) * 3 + (dI + 1)
  float* s1d = nullptr;      // omega / diag(A1) of the owned 2h nodes

  __device__ Stepper(const StepParams& P_, Comm& comm_, unsigned char* dyn) : P(P_), comm(comm_) {
    sb.nx = P.nx;
    sb.ny = P.ny;
    sb.cs = P.cs;
    sb.rank = comm.rank();
    slab_rows(P.ny + 1, P.cs, sb.rank, sb.r0, sb.R);
    sb.W = P.W;
    sb.G = P.W / kGroup;
    sb.ngroups = sb.R * sb.G;
    const int W = sb.W;
    const int halo = (P.rmax + 2) * W + 2 * kSlack;
    const int own = P.rmax * W + 2 * kSlack;
    const int elems = (P.rmax + 1) * W + 2 * kSlack;
    unsigned char* p = dyn;
    double* x64b = reinterpret_cast<double*>(p);  p += sizeof(double) * halo;
    double* b64b = reinterpret_cast<double*>(p);  p += sizeof(double) * own;
    double* axb = reinterpret_cast<double*>(p);   p += P.keep_ax ? sizeof(double) * own : 0;
    float* zb = reinterpret_cast<float*>(p);      p += sizeof(float) * halo;
    float* db = reinterpret_cast<float*>(p);      p += sizeof(float) * own;
    float* eb = reinterpret_cast<float*>(p);
    for (int i = threadIdx.x; i < halo; i += blockDim.x) {
      x64b[i] = 0.0;
      zb[i] = 0.f;
    }
    for (int i = threadIdx.x; i < own; i += blockDim.x) {
      b64b[i] = 0.0;
      if (P.keep_ax) axb[i] = 0.0;
      db[i] = 0.f;
    }
    if constexpr (kMixed) {
      for (int i = threadIdx.x; i < 2 * elems; i += blockDim.x) eb[i] = 0.f;
    }
    {
      if (P.tl_naj > 0) {
        const int naxp = coarse_row_stride(P.nax), ncp = naxp * P.nay;
        const int groups = P.rmax * (W / kGroup);
        // after the element weights (FP32 CG only); 16-byte aligned: every earlier array is a
        // multiple of 4 words
        float* t = eb + (kMixed ? 2 * elems : 0);
        tl_ainv = t;  t += P.tl_naj * naxp * ncp;
        tl_slot = t;  t += P.wide ? 0 : P.cs * ncp;   // grid-wide: the partials are in global memory
        tl_qc = t;    t += ncp;
        tl_ec = t;    t += P.tl_naj * naxp;
        if (P.tl_vc) {
          // every array a multiple of 4 words, so each starts 16-byte aligned
          constexpr int rw = (int)(sizeof(V) / 4);
          float* v0 = t;
          vrh = reinterpret_cast<V*>(t);  t += 2 * W * rw;
          vy = t + kSlack;   t += halo;
          vsd = t + kSlack;  t += halo;
          if (P.tl_nu >= 2) {
            ve0 = t + kSlack;  t += halo;
            ve1 = t + kSlack;  t += halo;
          }
          if constexpr (!kMixed) {
            wk = t + kSlack;
            wm = t + elems + kSlack;
            t += 2 * elems;
          }
          for (float* z = v0 + threadIdx.x; z < t; z += blockDim.x) *z = 0.f;
        }
        if (P.tl_l3) {
          float* l0 = t;
          vw = t + kSlack;  t += halo;
          W1 = P.l3_W1;
          const int halo1 = (P.l3_r1max + 2) * W1 + 2 * kSlack;
          own1s = P.l3_r1max * W1 + 2 * kSlack;
          b1x = t + kSlack;  t += halo1;
          b1u = t + kSlack;  t += halo1;
          b1z = t + kSlack;  t += halo1;
          s1a = t + kSlack;  t += halo1;
          s1b = t + kSlack;  t += halo1;
          a1w = t + kSlack - W1; t += 9 * own1s;     // indexed like the halo buffers from lr1 = 0
          s1d = t + kSlack - W1; t += own1s;
          for (float* z = l0 + threadIdx.x; z < t; z += blockDim.x) *z = 0.f;
          tl_cov = reinterpret_cast<int*>(t);
          l1_rows_of_slab(sb.r0, sb.R, J0, R1);
          if (sb.rank > 0) {
            int r0b, Rb, J0b;
            slab_rows(P.ny + 1, P.cs, sb.rank - 1, r0b, Rb);
            l1_rows_of_slab(r0b, Rb, J0b, R1b);
          }
          const int ny1 = P.l3_ny1;
          aj0 = l3_agg(J0 > 0 ? J0 - 1 : 0, P.cm, P.nay);
          naj = l3_agg(J0 + R1 <= ny1 ? J0 + R1 : ny1, P.cm, P.nay) - aj0 + 1;
          ajo0 = l3_agg(J0, P.cm, P.nay);
          najo = l3_agg(J0 + R1 - 1, P.cm, P.nay) - ajo0 + 1;
#pragma unroll
          for (int u = 0; u < K1; ++u) {
            const int n1 = P.l3_nx1 + 1, i = threadIdx.x + u * blockDim.x;
            n1o[u] = -1;
            n1a[u] = 0;
            if (i < R1 * n1) {
              const int lr1 = i / n1, I = i - lr1 * n1;
              n1o[u] = (lr1 + 1) * W1 + I + 1;
              n1a[u] = (l3_agg(J0 + lr1, P.cm, P.nay) - aj0) * naxp + l3_agg(I, P.cm, P.nax);
            }
          }
          for (int J = threadIdx.x; J < P.nay; J += blockDim.x) {
            int lo = -1, hi = -1;
            for (int q = 0; q < P.cs; ++q) {
              int r0q, Rq, J0q, R1q;
              slab_rows(P.ny + 1, P.cs, q, r0q, Rq);
              l1_rows_of_slab(r0q, Rq, J0q, R1q);
              if (R1q > 0 && J >= l3_agg(J0q, P.cm, P.nay) && J <= l3_agg(J0q + R1q - 1, P.cm, P.nay)) {
                if (lo < 0) lo = q;
                hi = q;
              }
            }
            tl_cov[2 * J] = lo;
            tl_cov[2 * J + 1] = hi;
          }
          for (int q = 0; q < P.cs; ++q) {
            int r0q, Rq, J0q, R1q;
            slab_rows(P.ny + 1, P.cs, q, r0q, Rq);
            l1_rows_of_slab(r0q, Rq, J0q, R1q);
            tl_bytes += 4u * naxp * (l3_agg(J0q + R1q - 1, P.cm, P.nay) - l3_agg(J0q, P.cm, P.nay) + 1);
          }
        } else {
        tl_gs = t;    t += groups;
        tl_gagg = reinterpret_cast<int*>(t);  t += P.tl_vc ? groups + 2 * (W / kGroup) : groups;
        tl_cov = reinterpret_cast<int*>(t);
        int ajhi, ajo1;
        coarse_rows_of_slab(sb.r0, sb.R, P.cm, P.nay, ajo0, ajo1);
        najo = ajo1 - ajo0 + 1;
        if (P.tl_vc) {
          coarse_rows_of_halo_slab(sb.r0, sb.R, P.ny, P.cm, P.nay, aj0, ajhi);
          // rows -1..R: group gi of row gi / G - 1 (no aggregate outside the grid)
          for (int gi = threadIdx.x; gi < (sb.R + 2) * sb.G; gi += blockDim.x) {
            const int lr = gi / sb.G - 1, g = gi - (lr + 1) * sb.G, row = sb.r0 + lr;
            tl_gagg[gi] = (row < 0 || row > P.ny)
                              ? -1
                              : (coarse_agg_y(row, P.cm, P.nay) - aj0) * naxp + coarse_agg_x(g, P.cm, P.nax);
          }
        } else {
          aj0 = ajo0;
          ajhi = ajo1;
          for (int gi = threadIdx.x; gi < sb.ngroups; gi += blockDim.x) {
            const int lr = gi / sb.G, g = gi - lr * sb.G;
            tl_gagg[gi] = (coarse_agg_y(sb.r0 + lr, P.cm, P.nay) - aj0) * naxp + coarse_agg_x(g, P.cm, P.nax);
          }
        }
        naj = ajhi - aj0 + 1;
        for (int q = 0; q < P.cs; ++q) {
          int r0q, Rq, a, bq;
          slab_rows(P.ny + 1, P.cs, q, r0q, Rq);
          coarse_rows_of_slab(r0q, Rq, P.cm, P.nay, a, bq);
          tl_bytes += 4u * naxp * (bq - a + 1);
        }
        for (int J = threadIdx.x; J < P.nay; J += blockDim.x) {
          int lo = -1, hi = -1;
          for (int q = 0; q < P.cs; ++q) {
            int r0q, Rq, a, bq;
            slab_rows(P.ny + 1, P.cs, q, r0q, Rq);
            coarse_rows_of_slab(r0q, Rq, P.cm, P.nay, a, bq);
            if (J >= a && J <= bq) {
              if (lo < 0) lo = q;
              hi = q;
            }
          }
          tl_cov[2 * J] = lo;
          tl_cov[2 * J + 1] = hi;
        }
        }
      }
    }
    x64 = x64b + kSlack;
    b64 = b64b + kSlack - W;   // b64[loc] for loc in own rows (loc >= W)
    ax64 = P.keep_ax ? axb + kSlack - W : nullptr;
    zbuf = zb + kSlack;
    dinv = db + kSlack - W;    // dinv[loc] likewise
    if constexpr (kMixed) {
      wk = eb + kSlack;
      wm = eb + elems + kSlack;
    }
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int gi = threadIdx.x + k * blockDim.x;
      loc0[k] = -1;
      if (gi < sb.ngroups) {
        const int lr = gi / sb.G, g = gi - lr * sb.G;
        loc0[k] = (lr + 1) * W + kGroup * g;
      }
    }
    gshift = sb.r0 * W;
  }

  // global node index of node j of a group, or -1 for a pad node
  __device__ __forceinline__ int gnode(int l0, int j) const {
    const int lr = l0 / sb.W - 1;
    const int ix = (l0 - (lr + 1) * sb.W) + j - 1;
    return (ix >= 0 && ix <= P.nx) ? (sb.r0 + lr) * (P.nx + 1) + ix : -1;
  }

  template <class T, int NV, int NX = 0, class Post = NoPost>
  __device__ __forceinline__ void allreduce(T (&v)[NV + NX], Post post = Post()) {
    comm.template allreduce<T, NV, NX, Post>(v, sb.cs, post);
  }

  // Select the operator C/dt + K (fine) or C/dtau + K (coarse): per-node FP64 weights for the
  // residual, and, of the operator times ffw.scale, float pairs (FP64 kinds' CG), FP32 element weights
  // in shared memory (FP32 CG, V-cycle) and the Jacobi inverse diagonal (zero on Dirichlet and pad
  // nodes).  The 2h level and the aggregates' inverse are built from the operator times scale too.
  __device__ void set_operator() {
    constexpr bool coarse = COARSE;
    A = coarse ? P.A_coarse : P.A_fine;
    ffw = coarse ? P.ff_coarse : P.ff_fine;
    step_dt = coarse ? P.dtau : P.dt;
    inv_dt = 1.0 / step_dt;
    ax_valid = false;
    tl = coarse && P.tl_naj > 0 && P.Ainv != nullptr;
    vc = tl && P.tl_vc;
    l3 = vc && P.tl_l3;
    if (tl && !tl_loaded) {        // rows of the aggregate rows aj0 .. aj0+naj-1 of Ainv, 16-byte copies
      const int naxp = coarse_row_stride(P.nax), ncp = naxp * P.nay;
      const int n4 = naj * naxp * ncp / 4;
      const float4* src = reinterpret_cast<const float4*>(P.Ainv + (size_t)aj0 * naxp * ncp);
      float4* dst = reinterpret_cast<float4*>(tl_ainv);
      for (int i = threadIdx.x; i < n4; i += blockDim.x) dst[i] = src[i];
      tl_loaded = true;
    }
    const int W = sb.W;
    __syncthreads();
    if (kMixed || vc) {
      const double* wE = coarse ? P.wE_coarse : P.wE_fine;
      const int PE = (P.ny + 2) * W + 2 * kSlack;      // one element array incl. slack
      const int n = (sb.R + 1) * W;
      const double* src = wE + sb.r0 * W;               // padded element row r0 = element row r0 - 1
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double Dw = src[i], Sw = src[PE + i];   // 4 (k + m) and 2 m - k
        wk[i] = (float)(ffw.scale * (fma(-2.0, Sw, Dw) * (1.0 / 6.0)));
        wm[i] = (float)(ffw.scale * (fma(4.0, Sw, Dw) * (1.0 / 12.0)));
      }
    }
    fmask = 0;
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const int g = gnode(l0, j);
        float v = 0.f;
        if (g >= 0 && P.dirichlet[g] == 0) {
          v = 1.f / (float)(ffw.scale * A.C[l0 + gshift + j]);
          fmask |= 1u << (kGroup * k + j);
        }
        dinv[l0 + j] = v;
      }
    }
    if (l3) {
      // the 2h stencil and omega / diag of the owned 2h nodes (FP32)
      const int n1 = P.l3_nx1 + 1, nn1 = n1 * (P.l3_ny1 + 1);
      for (int t = threadIdx.x; t < R1 * n1; t += blockDim.x) {
        const int lr1 = t / n1, I = t - lr1 * n1, o = (lr1 + 1) * W1 + I + 1;
        const int g = (J0 + lr1) * n1 + I;
#pragma unroll
        for (int k = 0; k < 9; ++k) a1w[k * own1s + o] = (float)P.A1[(size_t)k * nn1 + g];
        s1d[o] = (float)((double)P.tl_omega / P.A1[(size_t)4 * nn1 + g]);
      }
    }
    if (vc) {
      // S = omega / diag on rows -1..R; 0 on Dirichlet, pad and out-of-grid nodes
      for (int i = threadIdx.x; i < (sb.R + 2) * W; i += blockDim.x) {
        const int lr = i / W - 1, ix = i - (lr + 1) * W - 1, row = sb.r0 + lr;
        float v = 0.f;
        if (row >= 0 && row <= P.ny && ix >= 0 && ix <= P.nx && P.dirichlet[row * (P.nx + 1) + ix] == 0)
          v = (float)((double)P.tl_omega / (ffw.scale * A.C[i + gshift]));
        vsd[i] = v;
      }
    }
    __syncthreads();
  }

  __device__ __forceinline__ bool unknown(int k, int j) const { return (fmask >> (kGroup * k + j)) & 1u; }

  // Load a node vector from global memory into x64: owned rows and both halo rows
  // (Dirichlet nodes forced to zero).  Ends with __syncthreads.
  __device__ void load_x64(const double* __restrict__ src) {
    ax_valid = false;
    __syncthreads();
    const int nn = P.nx + 1;
    const int rows = sb.R + 2;
    for (int t = threadIdx.x; t < rows * nn; t += blockDim.x) {
      const int row = t / nn, ix = t - row * nn;
      const int g = sb.r0 - 1 + row;
      if (g >= 0 && g <= P.ny) {
        const int gi = g * nn + ix;
        x64[row * sb.W + ix + 1] = P.dirichlet[gi] ? 0.0 : src[gi];
      }
    }
    __syncthreads();
  }

  __device__ void zero_x64() {
    ax_valid = false;
    __syncthreads();
    for (int i = threadIdx.x; i < (P.rmax + 2) * sb.W; i += blockDim.x) x64[i] = 0.0;
    __syncthreads();
  }

  // Correction sweeps: the start of a step is G_old plus the polynomial extrapolation of the
  // sweep's increments G(x^new) - G(x^old) through the last m of them (1 <= m <= 3):
  //   x64 = G + inc,  inc = d0 (m = 1), 2 d0 - d1 (m = 2), 3 (d0 - d1) + d2 (m = 3),
  // with d_i = X_i - Fm[i] the increment of the i-th step before, which by the correction itself
  // is the corrected state X_i that step produced minus the fine result Fm[i] of its slice; X_0
  // is x64 (the state the step propagates), X_1, X_2 node vectors of earlier corrected states.
  // On the owned and both halo rows: every CTA evaluates the same expression on the same
  // operands (x64's halos are exact), so the halos stay exact.  Ends with __syncthreads.
  __device__ void load_x64_increment(const double* __restrict__ G, int m, const double* const* Fm,
                                     const double* const* X) {
    ax_valid = false;
    __syncthreads();
    const int nn = P.nx + 1;
    const int rows = sb.R + 2;
    for (int t = threadIdx.x; t < rows * nn; t += blockDim.x) {
      const int row = t / nn, ix = t - row * nn;
      const int g = sb.r0 - 1 + row;
      if (g >= 0 && g <= P.ny) {
        const int gi = g * nn + ix;
        double& x = x64[row * sb.W + ix + 1];
        const double d0 = x - Fm[0][gi];
        double inc = d0;
        if (m == 2) inc = fma(2.0, d0, -(X[1][gi] - Fm[1][gi]));
        if (m == 3) inc = fma(3.0, d0 - (X[1][gi] - Fm[1][gi]), X[2][gi] - Fm[2][gi]);
        x = P.dirichlet[gi] ? 0.0 : G[gi] + inc;
      }
    }
    __syncthreads();
  }

  // Polynomial extrapolation in time of the initial guess: with x64 = x_1 (the last state) and
  // X[i-2] = x_i, i = 2..n, the states of the n previous equidistant steps (global node vectors),
  // x64 becomes the value at the next step of the polynomial of degree n-1 through them,
  //   n = 2: 2 x_1 - x_2;  n = 3: 3 x_1 - 3 x_2 + x_3;  n = 4: 4 x_1 - 6 x_2 + 4 x_3 - x_4,
  // on the owned rows and both halo rows.  x64's halo rows hold the neighbours' x_1, so every
  // CTA evaluates the same expression on the same operands and the halos stay exact: no
  // exchange is needed.  If wr is given, x_1 is first saved there on the owned rows (the
  // slice's ring of states; wr is none of the X).  Ends with __syncthreads.
  // The ring's rows are padded node rows (P.W entries a row, rows 0 .. ny), so a thread moves groups
  // of 4 with 16-byte loads; pads and Dirichlet nodes are zero in every state.
  __device__ void extrapolate_x64(int n, const double* const* X, double* __restrict__ wr) {
    ax_valid = false;
    __syncthreads();
    const int G = sb.G, total = (sb.R + 2) * G;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      const int row = t / G, y = sb.r0 - 1 + row;
      if (y < 0 || y > P.ny) continue;
      double* x = x64 + kGroup * t;
      const size_t o = (size_t)(sb.r0 - 1) * P.W + kGroup * t;
      double x1[4], v[4], a[4], b[4], c[4];
      load4(x, x1);
      if (n >= 2) load4(X[0] + o, a);
      if (n >= 3) load4(X[1] + o, b);
      if (n >= 4) load4(X[2] + o, c);
      if (wr && row >= 1 && row <= sb.R) {
        *reinterpret_cast<double2*>(wr + o) = make_double2(x1[0], x1[1]);
        *reinterpret_cast<double2*>(wr + o + 2) = make_double2(x1[2], x1[3]);
      }
      if (n < 2) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        if (n == 2)
          v[j] = fma(2.0, x1[j], -a[j]);
        else if (n == 3)
          v[j] = fma(3.0, x1[j] - a[j], b[j]);
        else
          v[j] = fma(4.0, x1[j] + b[j], -fma(6.0, a[j], c[j]));
      }
      *reinterpret_cast<double2*>(x) = make_double2(v[0], v[1]);
      *reinterpret_cast<double2*>(x + 2) = make_double2(v[2], v[3]);
    }
    __syncthreads();
  }

  // Store the owned nodes of x64 to a global node vector.
  __device__ void store_x64(double* __restrict__ dst) const {
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const int g = gnode(l0, j);
        if (g >= 0) dst[g] = x64[l0 + j];
      }
    }
  }

  // Refresh every CTA's halo rows of a buffer from the neighbours' owned rows.
  template <class T>
  __device__ void exchange(T* buf) {
    __syncthreads();
    comm.exchange(buf, sb);
  }
  __device__ void exchange_x64() { exchange(x64); }

  // (C/dt) x64 on a group.  With a uniform capacity the mass stencil is (c h^2/36) (1 4 1) x (1 4 1)
  // (2 instead of 4 on the boundary): 4 FP64 instructions per node and no weights, instead of 9.
  __device__ __forceinline__ void mass_dt(int l0, double (&y)[4]) const {
    if (P.has_dc) {
      stencil_node64<double>(x64, l0, P.mass, l0 + gshift, sb.W, y);
#pragma unroll
      for (int j = 0; j < kGroup; ++j) y[j] *= inv_dt;
      return;
    }
    const int lr = l0 / sb.W - 1, iy = sb.r0 + lr, ix0 = l0 - (lr + 1) * sb.W - 1;
    const double dy = iy == 0 || iy == P.ny ? 2.0 : 4.0, s = P.mass_uniform * inv_dt;
    double xl[6], xm[6], xh[6];
    load_window(x64, l0 - sb.W, xl);
    load_window(x64, l0, xm);
    load_window(x64, l0 + sb.W, xh);
#pragma unroll
    for (int i = 0; i < 6; ++i) xm[i] = fma(dy, xm[i], xl[i] + xh[i]);
#pragma unroll
    for (int j = 0; j < kGroup; ++j) {
      const double dx = ix0 + j == 0 || ix0 + j == P.nx ? 2.0 : 4.0;
      y[j] = s * fma(dx, xm[j + 1], xm[j] + xm[j + 2]);
    }
  }

  // b64 = (C/dt) x64 + src, with src(global node) supplied per owned free node.
  template <class Src>
  __device__ void build_rhs(Src src) {
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
      double y[4];
      mass_dt(l0, y);
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const bool free_node = dinv[l0 + j] != 0.f;
        b64[l0 + j] = free_node ? y[j] + src(gnode(l0, j)) : 0.0;
      }
    }
  }

  // r64 = b - A x64 on the owned groups (0 off the unknowns); returns the local sum of r^2.
  __device__ __forceinline__ double residual(double (&r64)[NG][4]) const {
    double rr = 0.0;
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) r64[k][j] = 0.0;
      if (l0 < 0) continue;
      double y[4];
      stencil_node64<double>(x64, l0, A, l0 + gshift, sb.W, y);
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        if (ax64) ax64[l0 + j] = y[j];
        if (unknown(k, j)) {
          r64[k][j] = b64[l0 + j] - y[j];
          rr = fma(r64[k][j], r64[k][j], rr);
        }
      }
    }
    return rr;
  }

  // r64 = b - (A x64 saved by the last residual evaluation); valid while x64 is unchanged.
  __device__ __forceinline__ double residual_saved(double (&r64)[NG][4]) const {
    double rr = 0.0;
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) r64[k][j] = 0.0;
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        if (unknown(k, j)) {
          r64[k][j] = b64[l0 + j] - ax64[l0 + j];
          rr = fma(r64[k][j], r64[k][j], rr);
        }
      }
    }
    return rr;
  }

  // A z on group k with the FP32 element weights; every lane calls it (a lane without the group
  // computes on the first one)
  __device__ __forceinline__ void apply32(const float* z, int k, float (&y)[4], bool no_lo = false,
                                          bool no_hi = false) const {
    stencil_km32(z, wk, wm, loc0[k] < 0 ? sb.W : loc0[k], sb.W, threadIdx.x & 31, y, no_lo, no_hi);
  }

  // Two-level preconditioner M^-1 = D^-1 + P Ac^-1 P^T of the coarse-step solves (CG in either
  // precision; the coarse part is applied in FP32, the FP64 residual loop around the CG fixes
  // the accuracy); P is piecewise constant on aggregates of m x m nodes aligned to the 4-node groups, so the
  // restriction P^T v is a sum of group sums and the prolongation adds one value per group.
  // Every CTA sends its partial sums for the aggregates its slab touches to every CTA of the
  // cluster (16-byte stores of 4 aggregates); comm.finish_tl() waits for all of them.
  // coarse_gather then adds, chunk by chunk, the partials of the covering ranks in rank order
  // and multiplies by the CTA's rows of Ac^-1.
  template <class T>
  __device__ void coarse_restrict_push(const T (&v)[NG][4]) {
    const int G = sb.G, m4 = P.cm / 4, nax = P.nax, naxp = coarse_row_stride(nax), ncp = naxp * P.nay;
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      if (loc0[k] < 0) continue;
      tl_gs[threadIdx.x + k * blockDim.x] = (f32(v[k][0]) + f32(v[k][1])) + (f32(v[k][2]) + f32(v[k][3]));
    }
    __syncthreads();
    // 4 lanes per local aggregate (16 lanes per chunk of 4 aggregates), each summing every
    // 4th node row; padding aggregates (ax >= nax) sum to 0
    const int items = najo * naxp, padded = ((4 * items + 31) / 32) * 32;
    const int rlast = sb.r0 + sb.R - 1;
    const int lane = threadIdx.x & 31;
    for (int t = threadIdx.x; t < padded; t += blockDim.x) {
      const int item = t >> 2, part = t & 3;
      const int ajl = item / naxp, ax = item - ajl * naxp;
      const int ay = ajo0 + ajl;
      float acc = 0.f;
      if (item < items && ax < nax) {
        const int y0 = max(ay * P.cm, sb.r0), y1 = min(ay == P.nay - 1 ? P.ny : ay * P.cm + P.cm - 1, rlast);
        const int g0 = ax * m4, g1 = ax == nax - 1 ? G - 1 : g0 + m4 - 1;
        for (int iy = y0 + part; iy <= y1; iy += 4) {
          const float* row = tl_gs + (iy - sb.r0) * G;
          for (int g = g0; g <= g1; ++g) acc += row[g];
        }
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      // the 16 lanes of a chunk: lane (c, p) holds aggregate c's sum; collect all four
      const int base = lane & 16;
      float4 chunk;
      chunk.x = __shfl_sync(0xffffffffu, acc, base + 0);
      chunk.y = __shfl_sync(0xffffffffu, acc, base + 4);
      chunk.z = __shfl_sync(0xffffffffu, acc, base + 8);
      chunk.w = __shfl_sync(0xffffffffu, acc, base + 12);
      const int item0 = (t & ~15) >> 2;              // first aggregate of the chunk
      if (item0 < items) {
        const int ajl0 = item0 / naxp, ax0 = item0 - ajl0 * naxp;
        const int dst = sb.rank * ncp + (ajo0 + ajl0) * naxp + ax0;
        comm.publish_tl(tl_slot, dst, chunk, lane & 15, sb.cs);
      }
    }
    comm.expect_tl(tl_bytes);
  }

  // After the phase that follows coarse_restrict_push: qc = sum over the covering ranks of the
  // partials (in rank order), then ec = Ac^-1 qc on the CTA's aggregate rows (8 lanes per row of
  // Ac^-1, 16-byte loads).
  __device__ void coarse_gather() {
    const int naxp = coarse_row_stride(P.nax), ncp = naxp * P.nay;
    const float* slots = comm.tl_slots(tl_slot);
    for (int L4 = threadIdx.x; L4 < ncp / 4; L4 += blockDim.x) {
      const int J = (4 * L4) / naxp;            // a 16-byte chunk lies in one aggregate row
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int q = tl_cov[2 * J]; q <= tl_cov[2 * J + 1]; ++q) {
        const float4 u = comm.tl_load4(slots, q * ncp + 4 * L4);
        acc.x += u.x; acc.y += u.y; acc.z += u.z; acc.w += u.w;
      }
      reinterpret_cast<float4*>(tl_qc)[L4] = acc;
    }
    __syncthreads();
    const int nrows = naj * naxp, n4 = ncp / 4;
    const int padded = ((8 * nrows + 31) / 32) * 32;
    const float4* q4 = reinterpret_cast<const float4*>(tl_qc);
    for (int t = threadIdx.x; t < padded; t += blockDim.x) {
      const int row = t >> 3, part = t & 7;
      float acc = 0.f;
      if (row < nrows) {
        const float4* a4 = reinterpret_cast<const float4*>(tl_ainv + (size_t)row * ncp);
        float ax = 0.f, ay = 0.f, az = 0.f, aw = 0.f;
#pragma unroll 4
        for (int L = part; L < n4; L += 8) {
          const float4 a = a4[L], r = q4[L];
          ax = fmaf(a.x, r.x, ax);
          ay = fmaf(a.y, r.y, ay);
          az = fmaf(a.z, r.z, az);
          aw = fmaf(a.w, r.w, aw);
        }
        acc = (ax + ay) + (az + aw);
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      acc += __shfl_xor_sync(0xffffffffu, acc, 4);
      if (part == 0 && row < nrows) tl_ec[row] = acc;
    }
    __syncthreads();
  }

  // z = D^-1 r + P ec on the owned nodes (0 off the unknowns), written to zbuf; returns the
  // local part of (r, z).
  __device__ V prolong_precondition(const V (&r)[NG][4]) {
    V rz = V{};
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
      const float e = tl_ec[tl_gagg[threadIdx.x + k * blockDim.x]];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const float z = unknown(k, j) ? fmaf(dinv[l0 + j], f32(r[k][j]), e) : 0.f;
        zbuf[l0 + j] = z;
        rz = vdot(rz, r[k][j], z);
      }
    }
    return rz;
  }

  // The owned edge rows (0 and R-1) of a per-thread vector into the neighbours' two-row buffer
  // `edge` ([0]: the row below the slab, [1]: the row above), straight from registers; visible
  // after comm.finish_edges().
  __device__ void put_edges(V* edge, const V (&v)[NG][4]) {
    comm.begin_edges();
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
      const int lr = l0 / sb.W - 1;
      if (lr == 0 || lr == sb.R - 1) comm.put_edge(edge, lr, l0 - (lr + 1) * sb.W, v[k], sb);
    }
    comm.end_edges(edge, sb);
  }

  // offset in a rows -1..R buffer of entry i of the two halo rows ([0, W): row -1, [W, 2W): row R)
  __device__ __forceinline__ int halo_offset(int i) const { return i < sb.W ? i : (sb.R + 1) * sb.W + (i - sb.W); }

  // V(1,1) two-grid cycle z = M^-1 r in FP32 over the owned rows and the two halo rows:
  //   y = S r,  ec = Ac^-1 P^T (r - A y),  u = y + P ec (in place of y),  z = u + S (r - A u),
  // with the damped-Jacobi smoother S = omega D^-1 and A applied with the FP32 element weights,
  // so that I - M^-1 A = (I - S A)(I - P Ac^-1 P^T A)(I - S A) (symmetric).  The halo rows of r
  // (vrh) are the owners' rows, and every CTA computes ec for the
  // aggregate rows its halo rows touch from the same restricted vector, so y and u on a halo
  // row equal the owner's values: M^-1 is one operator across the CTAs.  One all-to-all
  // phase (the restricted partials).  z goes to zbuf on the owned rows; returns the local (r, z).
  __device__ V vcycle(const V (&r)[NG][4]) {
    const int W = sb.W, G = sb.G;
    float rf[NG][4];   // r in FP32, converted once (FP64 conversions run on the FP64 pipe)
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) rf[k][j] = f32(r[k][j]);
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) vy[l0 + j] = vsd[l0 + j] * rf[k][j];
    }
    for (int i = threadIdx.x; i < 2 * W; i += blockDim.x) {
      const int l = halo_offset(i);
      vy[l] = vsd[l] * f32(vrh[i]);
    }
    __syncthreads();
    float w[NG][4];
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = 0.f;
      float t[4];
      apply32(vy, k, t);
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = unknown(k, j) ? rf[k][j] - t[j] : 0.f;
    }
    coarse_restrict_push(w);
    comm.finish_tl();
    coarse_gather();
    for (int gi = threadIdx.x; gi < (sb.R + 2) * G; gi += blockDim.x) {
      const int a = tl_gagg[gi];
      const float e = a >= 0 ? tl_ec[a] : 0.f;
      const int l = (gi / G) * W + kGroup * (gi % G);   // row gi / G - 1, group gi % G
#pragma unroll
      for (int j = 0; j < kGroup; ++j) vy[l + j] = vsd[l + j] != 0.f ? vy[l + j] + e : 0.f;
    }
    __syncthreads();
    V rz = V{};
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      float t[4];
      apply32(vy, k, t);
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const float z = unknown(k, j) ? fmaf(vsd[l0 + j], rf[k][j] - t[j], vy[l0 + j]) : 0.f;
        zbuf[l0 + j] = z;
        rz = vdot(rz, r[k][j], z);
      }
    }
    return rz;
  }

  // Slab-local damped-Jacobi smoothing of A e = s: P.tl_nu steps from e = 0 over the owned rows
  // with the halo rows held at zero (the slab's diagonal block A_s of A), in FP32, the iterate
  // ping-ponging between two buffers; e returned in registers.  The result is a fixed polynomial
  // in D^-1 A_s times D^-1, a symmetric operator, so the cycle that uses it stays symmetric; it
  // needs no communication.
  __device__ void smooth_local(const float (&s)[NG][4], float (&e)[NG][4]) {
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) e[k][j] = l0 >= 0 ? vsd[l0 + j] * s[k][j] : 0.f;
    }
    for (int it = 1; it < P.tl_nu; ++it) {
      float* buf = (it & 1) ? ve0 : ve1;
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int l0 = loc0[k];
        if (l0 < 0) continue;
#pragma unroll
        for (int j = 0; j < kGroup; ++j) buf[l0 + j] = e[k][j];
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int l0 = loc0[k];
        float t[4];
        apply32(buf, k, t);
        if (l0 < 0) continue;
#pragma unroll
        for (int j = 0; j < kGroup; ++j) e[k][j] = fmaf(vsd[l0 + j], s[k][j] - t[j], e[k][j]);
      }
    }
  }

  // Two-grid cycle with the slab-local smoother S_s of smooth_local before and after the coarse
  // correction: e1 = S_s r;  ec = Ac^-1 P^T (r - A e1);  u = e1 + P ec;  z = u + S_s (r - A u),
  // so that I - M^-1 A = (I - S_s A)(I - P Ac^-1 P^T A)(I - S_s A).  e1's edge rows are
  // exchanged before the residual; u on the halo rows is then the owner's value (e1 from the
  // owner, ec computed from the same restricted vector).  One neighbour exchange and one
  // all-to-all phase.  z goes to zbuf on the owned rows; returns the local (r, z).
  __device__ V vcycle_local(const V (&r)[NG][4]) {
    const int W = sb.W, G = sb.G;
    float rf[NG][4], e[NG][4], w[NG][4];
#pragma unroll
    for (int k = 0; k < NG; ++k)
#pragma unroll
      for (int j = 0; j < kGroup; ++j) rf[k][j] = f32(r[k][j]);
    smooth_local(rf, e);
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) vy[l0 + j] = e[k][j];
    }
    exchange(vy);
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = 0.f;
      float t[4];
      apply32(vy, k, t);
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = unknown(k, j) ? rf[k][j] - t[j] : 0.f;
    }
    coarse_restrict_push(w);
    comm.finish_tl();
    coarse_gather();
    for (int gi = threadIdx.x; gi < (sb.R + 2) * G; gi += blockDim.x) {
      const int a = tl_gagg[gi];
      const float ea = a >= 0 ? tl_ec[a] : 0.f;
      const int l = (gi / G) * W + kGroup * (gi % G);   // row gi / G - 1, group gi % G
#pragma unroll
      for (int j = 0; j < kGroup; ++j) vy[l + j] = vsd[l + j] != 0.f ? vy[l + j] + ea : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      float t[4];
      apply32(vy, k, t);
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = unknown(k, j) ? f32(r[k][j]) - t[j] : 0.f;
    }
    smooth_local(w, e);
    V rz = V{};
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const float z = vy[l0 + j] + e[k][j];
        zbuf[l0 + j] = z;
        rz = vdot(rz, r[k][j], z);
      }
    }
    return rz;
  }

  // ---------------------------------------------------------------- three-level cycle
  // 2h buffers: halo buffers (rows -1..R1) at (lr1 + 1) W1 + I + 1; the owned-row arrays a1w and s1d
  // are addressed by the same offset

  // (A1 x) at the owned 2h node with offset c from a halo buffer x (zero outside the 2h grid)
  __device__ __forceinline__ float a1_apply(const float* __restrict__ x, int c) const {
    const float* w = a1w + c;
    float lo = 0.f, mid = 0.f, hi = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo = fmaf(w[k * own1s], x[c - W1 + k - 1], lo);
      mid = fmaf(w[(3 + k) * own1s], x[c + k - 1], mid);
      hi = fmaf(w[(6 + k) * own1s], x[c + W1 + k - 1], hi);
    }
    return (lo + hi) + mid;
  }

  // refresh the 2h halo rows of every CTA from the neighbours' owned rows
  __device__ void exchange_l1(float* buf) {
    __syncthreads();
    comm.exchange_rows(buf, W1, R1, R1b, sb.rank, sb.cs);
  }

  // P.tl_nu damped-Jacobi steps of A1_s e = s from e = 0 on the owned 2h rows, with the 2h halo
  // rows held at zero (the diagonal block of A1 of this CTA's rows: a fixed polynomial in
  // S1 A1_s times S1, symmetric, no communication).  Every thread keeps its nodes in registers; the
  // iterates ping-pong through s1a and s1b.
  __device__ __forceinline__ void smooth_l1(const float (&sv)[K1], float (&e)[K1]) {
#pragma unroll
    for (int u = 0; u < K1; ++u) e[u] = n1o[u] >= 0 ? s1d[n1o[u]] * sv[u] : 0.f;
    float* cur = s1a;
    for (int it = 1; it < P.tl_nu; ++it) {
#pragma unroll
      for (int u = 0; u < K1; ++u)
        if (n1o[u] >= 0) cur[n1o[u]] = e[u];
      __syncthreads();
#pragma unroll
      for (int u = 0; u < K1; ++u)
        if (n1o[u] >= 0) e[u] = fmaf(s1d[n1o[u]], sv[u] - a1_apply(cur, n1o[u]), e[u]);
      cur = cur == s1a ? s1b : s1a;
    }
  }

  // The 2h part of the three-level cycle, from the fine residual w0 in vw (halo rows exchanged):
  //   r1 = P1^T w0;  e1 = S1 r1;  ec = A2^-1 P2^T (r1 - A1 e1);  u1 = e1 + P2 ec;
  //   z1 = u1 + S1 (r1 - A1 u1) into b1z with its halo rows exchanged.
  // The plan gives the block a thread per owned 2h node, so a pass over them is one trip with
  // precomputed offsets: the passes are bound by latency (barriers, shared-memory round trips).
  __device__ __forceinline__ void l1_correct() {
    const int W = sb.W, n1 = P.l3_nx1 + 1, ny1 = P.l3_ny1;
    const int naxp = coarse_row_stride(P.nax), ncp = naxp * P.nay;
    // r1 = P1^T w0 on the owned 2h rows: fine rows 2J-1 .. 2J+1 lie in -1 .. R.  The 2h node at
    // offset o = (lr1 + 1) W1 + I + 1 sits on the fine offset of row 2 (J0 + lr1) - r0, column 2I.
    float r1[K1], e1[K1];
    const int fshift = (2 * J0 - sb.r0 + 1) * W - 1;
#pragma unroll
    for (int u = 0; u < K1; ++u) {
      r1[u] = 0.f;
      if (n1o[u] < 0) continue;
      const int lr1 = n1o[u] / W1 - 1, I1 = n1o[u] - (lr1 + 1) * W1;   // I1 = I + 1
      const float* c = vw + fshift + 2 * (lr1 * W + I1);
      const float mid = fmaf(0.5f, c[-1] + c[1], c[0]);
      const float lo = fmaf(0.5f, c[-W - 1] + c[-W + 1], c[-W]);
      const float hi = fmaf(0.5f, c[W - 1] + c[W + 1], c[W]);
      r1[u] = fmaf(0.5f, lo + hi, mid);
    }
    // 2h pre-smoothing e1 = S1 r1, exchanged
    smooth_l1(r1, e1);
#pragma unroll
    for (int u = 0; u < K1; ++u)
      if (n1o[u] >= 0) b1x[n1o[u]] = e1[u];
    exchange_l1(b1x);
    // 2h residual r1 - A1 e1 (in b1u's owned rows), summed per aggregate of the owned rows by 4
    // lanes each and published to every CTA (16 lanes per 16-byte chunk of 4 aggregates)
#pragma unroll
    for (int u = 0; u < K1; ++u)
      if (n1o[u] >= 0) b1u[n1o[u]] = r1[u] - a1_apply(b1x, n1o[u]);
    __syncthreads();
    const int items = najo * naxp, padded = ((4 * items + 31) / 32) * 32, lane = threadIdx.x & 31;
    for (int t = threadIdx.x; t < padded; t += blockDim.x) {
      const int item = t >> 2, ajl = item / naxp, ax = item - ajl * naxp, ay = ajo0 + ajl;
      float acc = 0.f;
      if (item < items && ax < P.nax) {
        const int ya = max(ay * P.cm, J0), yb = min(ay == P.nay - 1 ? ny1 : ay * P.cm + P.cm - 1, J0 + R1 - 1);
        const int xa = ax * P.cm, xb = ax == P.nax - 1 ? n1 - 1 : ax * P.cm + P.cm - 1;
        for (int J = ya + (t & 3); J <= yb; J += 4) {
          const float* row = b1u + (J - J0 + 1) * W1 + 1;
          for (int I = xa; I <= xb; ++I) acc += row[I];
        }
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      const int base = lane & 16;
      float4 chunk;
      chunk.x = __shfl_sync(0xffffffffu, acc, base + 0);
      chunk.y = __shfl_sync(0xffffffffu, acc, base + 4);
      chunk.z = __shfl_sync(0xffffffffu, acc, base + 8);
      chunk.w = __shfl_sync(0xffffffffu, acc, base + 12);
      const int item0 = (t & ~15) >> 2;                // first aggregate of the chunk
      if (item0 < items) {
        const int ajl0 = item0 / naxp, ax0 = item0 - ajl0 * naxp;
        comm.publish_tl(tl_slot, sb.rank * ncp + (ajo0 + ajl0) * naxp + ax0, chunk, lane & 15, sb.cs);
      }
    }
    comm.expect_tl(tl_bytes);
    comm.finish_tl();
    coarse_gather();
    // u1 = e1 + P2 ec on the owned and halo 2h rows (b1u's owned rows have been read: coarse_gather
    // ends with a block barrier)
#pragma unroll
    for (int u = 0; u < K1; ++u) {
      if (n1o[u] < 0) continue;
      e1[u] += tl_ec[n1a[u]];
      b1u[n1o[u]] = e1[u];
    }
    for (int t = threadIdx.x; t < 2 * n1; t += blockDim.x) {
      const int lr1 = t < n1 ? -1 : R1, I = t < n1 ? t : t - n1, J = J0 + lr1;
      if (J < 0 || J > ny1) continue;
      const int o = (lr1 + 1) * W1 + I + 1;
      b1u[o] = b1x[o] + tl_ec[(l3_agg(J, P.cm, P.nay) - aj0) * naxp + l3_agg(I, P.cm, P.nax)];
    }
    __syncthreads();
    // 2h post-smoothing z1 = u1 + S1 (r1 - A1 u1), exchanged
    float z1[K1];
#pragma unroll
    for (int u = 0; u < K1; ++u)
      if (n1o[u] >= 0) r1[u] -= a1_apply(b1u, n1o[u]);
    smooth_l1(r1, z1);
#pragma unroll
    for (int u = 0; u < K1; ++u)
      if (n1o[u] >= 0) b1z[n1o[u]] = e1[u] + z1[u];
    exchange_l1(b1z);
  }

  // P1 z1 on the fine group g of local row lr: columns 4g-1 .. 4g+2 take the 2h columns 2g-1, 2g and
  // 2g+1, an odd row the mean of the 2h rows below and above
  __device__ __forceinline__ void prolong_l1(int lr, int g, float (&v)[4]) const {
    const int y = sb.r0 + lr;
    const float* ra = b1z + ((y >> 1) - J0 + 1) * W1 + 2 * g;
    const float* rb = b1z + (((y + 1) >> 1) - J0 + 1) * W1 + 2 * g;
    const float z0 = 0.5f * (ra[0] + rb[0]), z1 = 0.5f * (ra[1] + rb[1]), z2 = 0.5f * (ra[2] + rb[2]);
    v[0] = 0.5f * (z0 + z1);
    v[1] = z1;
    v[2] = 0.5f * (z1 + z2);
    v[3] = z2;
  }

  // Three-level cycle z = M^-1 r in FP32 over the fine, 2h and aggregate levels:
  //   e0 = S0 r;  w0 = r - A e0;  r1 = P1^T w0;
  //   e1 = S1 r1;  ec = A2^-1 P2^T (r1 - A1 e1);  u1 = e1 + P2 ec;  z1 = u1 + S1 (r1 - A1 u1);
  //   u0 = e0 + P1 z1;  z = u0 + S0 (r - A u0),
  // S0, S1 the slab-local damped-Jacobi smoothers of smooth_local / smooth_l1, P1 bilinear from
  // the 2h nodes (2I, 2J), P2 piecewise constant on the aggregates, A1 = P1^T A P1,
  // A2 = P2^T A1 P2.  Each level's correction is the exact adjoint of its restriction and every
  // smoother is symmetric, so M^-1 is symmetric.  Values on halo rows equal the owners' (e0 and
  // e1 exchanged, ec from the same restricted vector in every CTA, z1 exchanged), so M^-1 is one
  // operator across the CTAs.  Four neighbour exchanges and one all-to-all
  // phase.  z goes to zbuf; returns the local (r, z).
  __device__ V vcycle3(const V (&r)[NG][4]) {
    const int W = sb.W;
    float e[NG][4], w[NG][4];
    // fine pre-smoothing e0 = S0 r, exchanged (r in FP32 in w)
#pragma unroll
    for (int k = 0; k < NG; ++k)
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = f32(r[k][j]);
    smooth_local(w, e);
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) vy[l0 + j] = e[k][j];
    }
    exchange(vy);
    // fine residual w0 = r - A e0 on the owned rows, exchanged
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      float t[4];
      apply32(vy, k, t);
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) vw[l0 + j] = unknown(k, j) ? w[k][j] - t[j] : 0.f;
    }
    exchange(vw);
    l1_correct();
    // u0 = e0 + P1 z1 on the owned and halo fine rows (in vy); 0 off the unknowns
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
      const int lr = l0 / W - 1;
      float v[4];
      prolong_l1(lr, (l0 - (lr + 1) * W) / kGroup, v);
#pragma unroll
      for (int j = 0; j < kGroup; ++j)
        if (unknown(k, j)) vy[l0 + j] += v[j];
    }
    for (int t = threadIdx.x; t < 2 * sb.G; t += blockDim.x) {
      const int lr = t < sb.G ? -1 : sb.R, g = t < sb.G ? t : t - sb.G, y = sb.r0 + lr;
      if (y < 0 || y > P.ny) continue;
      const int l0 = (lr + 1) * W + kGroup * g;
      float v[4];
      prolong_l1(lr, g, v);
#pragma unroll
      for (int j = 0; j < kGroup; ++j)
        if (vsd[l0 + j] != 0.f) vy[l0 + j] += v[j];
    }
    __syncthreads();
    // fine post-smoothing z = u0 + S0 (r - A u0)
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = 0.f;
      float t[4];
      apply32(vy, k, t);
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) w[k][j] = unknown(k, j) ? f32(r[k][j]) - t[j] : 0.f;
    }
    smooth_local(w, e);
    V rz = V{};
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const float z = vy[l0 + j] + e[k][j];
        zbuf[l0 + j] = z;
        rz = vdot(rz, r[k][j], z);
      }
    }
    return rz;
  }

  // Two damped-Jacobi steps on the slab's diagonal block A_s (the rows of the other slabs left
  // out): z = S r + S (r - A_s S r) = (2S - S A_s S) r, S = omega D^-1, a symmetric operator,
  // positive definite while omega lambda_max(D^-1 A_s) < 2 (at most 0.8 * 2.25).  FP32 CG only
  // (the FP32 element weights); the first step's iterate goes through zbuf, whose halo rows are
  // not read, so the neighbours may already be writing their new edge rows into them.  No
  // communication; two block barriers.  z goes to zbuf; returns the local (r, z).
  __device__ V precond_local2(const V (&r)[NG][4]) {
    const float om = P.tl_omega;
    float e[NG][4];
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) e[k][j] = 0.f;
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        e[k][j] = om * dinv[l0 + j] * f32(r[k][j]);
        zbuf[l0 + j] = e[k][j];
      }
    }
    __syncthreads();
    float z[NG][4];
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
#pragma unroll
      for (int j = 0; j < kGroup; ++j) z[k][j] = 0.f;
      const int lr = l0 / sb.W - 1;
      float t[4];
      apply32(zbuf, k, t, lr <= 0, lr < 0 || lr == sb.R - 1);   // (lr = -1: no group, computes on the first row)
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) z[k][j] = fmaf(om * dinv[l0 + j], f32(r[k][j]) - t[j], e[k][j]);
    }
    __syncthreads();
    V rz = V{};
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        zbuf[l0 + j] = z[k][j];
        rz = vdot(rz, r[k][j], z[k][j]);
      }
    }
    return rz;
  }

  // z = M^-1 r to zbuf (owned rows); returns the local (r, z)
  __device__ V precondition(const V (&r)[NG][4]) {
    if constexpr (COARSE) {
      if (l3) return vcycle3(r);
      if (vc && P.tl_nu >= 2) return vcycle_local(r);
      if (vc) return vcycle(r);
      if (tl) return prolong_precondition(r);
    }
    if constexpr (kMixed) {
      if (P.local_steps >= 2) return precond_local2(r);
    }
    V rz = V{};
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const float z = dinv[l0 + j] * f32(r[k][j]);
        zbuf[l0 + j] = z;
        rz = vdot(rz, r[k][j], z);
      }
    }
    return rz;
  }

  // Preconditioned CG on A d = r, where r (given per node) is the FP64 residual scaled by a power
  // of two to a squared 2-norm rr0 in [1, 4); on return x64 += unscale * d.  Stops when
  // ||r||^2 <= target2 (scaled units) or at the iteration limit; returns the iteration count.
  // Vectors, scalars and dot products are V; z is float.
  // One reduction per iteration (after Chronopoulos and Gear): A z instead of A p, with q = A p by
  // recurrence, so the iteration waits for the neighbours' rows of z and for one all-reduce instead of
  // two.  (p, q) of the new direction p = z + beta p_old comes from that reduction as well,
  //   (p, q) = (z, w) + beta (2 (z, q_old) + beta (p, q)_old),
  // or, where K does not outweigh C/dt by much (P.cg_dots == 0), as (z, w) - beta^2 (p, q)_old.  That takes z
  // for conjugate to p_old, which it is to 2^-24 only, being the FP32 result of a preconditioner, and where
  // (p, q) is far below (z, w) the error decides: with K over C/dt of 1e5 and more it took 1.2 to 4 times
  // the iterations of a CG with a dot product of its own for (p, q) (16 x 16 nodes, FP64 kinds), or
  // 16 000 instead of 400 without an end (FP32 kinds).  With (z, q_old) it takes as many.  In FP32
  // (p, q)_old carried from iteration to iteration loses its own bits there too, so it is a dot product
  // of the same reduction.  One more dot product costs 3 to 4% of a pass (128 x 128 FP64 43.0 -> 44.4 ms,
  // 96 x 96 gradient 99.9 -> 104.8), the two of FP32 5% (100 x 100 28.0 -> 29.6): hence the rule.
  // The float pairs of the FP64 kinds: on a slab of 9 x 132 nodes (128 x 128 over 16 CTAs) an
  // iteration's stencil, updates and dot products took 10 100 cycles on the FP64 pipe (17 FP64
  // instructions per node) and take about 180 FP32 instructions per node in pairs.
  __device__ int cg_correct(V (&r)[NG][4], float rr0, float target2, double unscale) {
    V d[NG][4], p[NG][4], q[NG][4];
#pragma unroll
    for (int k = 0; k < NG; ++k) {
#pragma unroll
      for (int j = 0; j < kGroup; ++j) d[k][j] = p[k][j] = q[k][j] = V{};
    }
    const bool additive = COARSE && tl && !vc;                   // needs r restricted
    const bool global1 = COARSE && vc && !l3 && P.tl_nu < 2;     // needs r on the halo rows
    V rz_old = V{}, pq_old = V{};
    int it = 0;
    for (;;) {
      if (additive) {
        coarse_restrict_push(r);
        comm.finish_tl();
        coarse_gather();
      } else if (global1) {
        put_edges(vrh, r);
        comm.finish_edges();
      }
      // z = M^-1 r and w = A z; (r, z), (z, w), (r, r) and what (p, q) needs in one reduction; then beta,
      // (p, q) and alpha = (r, z) / (p, q).  (r, r), for the stop alone, needs no more than a float.
      const V rz_part = precondition(r);
      exchange(zbuf);
      V w[NG][4], zw = V{}, zq = V{}, pq = V{};
      float rr = 0.f;
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int l0 = loc0[k];
        if constexpr (kMixed) apply32(zbuf, k, w[k]);
        if (l0 < 0) continue;
        if constexpr (!kMixed) stencil_ff(zbuf, l0, ffw, l0 + gshift, sb.W, w[k]);
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
          if (!unknown(k, j)) w[k][j] = V{};
          zw = vdot(zw, w[k][j], zbuf[l0 + j]);
          rr = fmaf(f32(r[k][j]), f32(r[k][j]), rr);
        }
      }
      if (P.cg_dots) {
#pragma unroll
        for (int k = 0; k < NG; ++k) {
          const int l0 = loc0[k];
          if (l0 < 0) continue;
#pragma unroll
          for (int j = 0; j < kGroup; ++j) {
            zq = vdot(zq, q[k][j], zbuf[l0 + j]);
            if constexpr (kMixed) pq = vdot(pq, p[k][j], q[k][j]);
          }
        }
      }
      const bool start = it == 0;
      // alpha, beta and (p, q) into o, from (r, z), (z, w) and what (p, q) has beside (z, w)
      auto lengths = [start](const V& rz_, const V& zw_, const V& b, const V& more, V* o) {
        o[1] = start ? V{} : b;
        o[2] = zw_;
        if (!start) o[2] = vfma(b, more, zw_);
        if (!(f32(o[2]) > 0.f)) {        // nothing left of (p, q) but rounding: start again from z
          o[1] = V{};
          o[2] = zw_;
        }
        o[0] = vdiv(rz_, o[2]);
      };
      V o[3];
      if (P.cg_dots) {
        constexpr int NV = kMixed ? 5 : 4;
        V v[NV + 3] = {rz_part, zw, vfloat<V>(rr), zq};
        if constexpr (kMixed) v[4] = pq;
        allreduce<V, NV, 3>(v, [&lengths, rz_old, pq_old](V* t) {
          const V b = vdiv(t[0], rz_old), pq_ = kMixed ? t[NV - 1] : pq_old;
          lengths(t[0], t[1], b, vfma(b, pq_, t[3] + t[3]), t + NV);
        });
        rr = f32(v[2]);
        rz_old = v[0];
        for (int i = 0; i < 3; ++i) o[i] = v[NV + i];
      } else {
        V v[6] = {rz_part, zw, vfloat<V>(rr)};
        allreduce<V, 3, 3>(v, [&lengths, rz_old, pq_old](V* t) {
          const V b = vdiv(t[0], rz_old);
          lengths(t[0], t[1], b, vneg(vmul(b, pq_old)), t + 3);
        });
        rr = f32(v[2]);
        rz_old = v[0];
        for (int i = 0; i < 3; ++i) o[i] = v[3 + i];
      }
      const V alpha = o[0], beta = o[1];
      pq_old = o[2];
      if (!((start ? rr0 : rr) > target2)) break;
      const V nalpha = vneg(alpha);
      // p = z + beta p, q = w + beta q, d += alpha p, r -= alpha q
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int l0 = loc0[k];
        if (l0 < 0) continue;
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
          p[k][j] = vfma(beta, p[k][j], zbuf[l0 + j]);
          q[k][j] = vfma(beta, q[k][j], w[k][j]);
          d[k][j] = vfma(alpha, p[k][j], d[k][j]);
          r[k][j] = vfma(nalpha, q[k][j], r[k][j]);
        }
      }
      if (++it >= P.itmax) break;
    }
    if constexpr (kMixed) {
      // d with its halo rows in zbuf
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int l0 = loc0[k];
        if (l0 < 0) continue;
#pragma unroll
        for (int j = 0; j < kGroup; ++j) zbuf[l0 + j] = d[k][j];
      }
      exchange(zbuf);
    }
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        double x = x64[l0 + j];
        if constexpr (!kMixed) x = fma(widen(d[k][j].l), unscale, x);
        x64[l0 + j] = fma(widen(f32(d[k][j])), unscale, x);
      }
    }
    return it;
  }

  // After an FP32 CG (d with its halo rows in zbuf): x64's halo rows follow their owners' update bit
  // for bit, without an exchange.
  __device__ void update_halos(double unscale) {
    for (int i = threadIdx.x; i < 2 * sb.W; i += blockDim.x) {
      const int l = halo_offset(i);
      x64[l] = fma(widen(zbuf[l]), unscale, x64[l]);
    }
    __syncthreads();
  }

  // Solve (C/dt + K) x = b64 with x64 (owned + halos) as initial guess; on return x64 holds
  // the solution with valid halos in every CTA.  `step` is the fine index for error reports.
  // What decides is b - A x in FP64, evaluated after every CG: a residual that follows x by
  // recurrence misses the rounding of x and that of A d, and would accept solves that do not meet rtol.
  // An FP32 kind ends a solve that rounding keeps above rtol too (kRounding2); an FP64 kind reports it.
  // `reuse_ax`: x64 is the previous solution of the same operator, so the A x64 saved by that
  // solve's final residual check gives the first residual without another stencil.
  __device__ void solve(int step, bool reuse_ax = false) {
    double r64[NG][4];
    double bb_rr[2] = {0.0, 0.0};
    bb_rr[1] = (reuse_ax && ax_valid && ax64) ? residual_saved(r64) : residual(r64);
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) bb_rr[0] = fma(b64[l0 + j], b64[l0 + j], bb_rr[0]);
    }
    allreduce<double, 2>(bb_rr);
    const double bb = bb_rr[0];
    double rr = bb_rr[1];
    const double tol2 = P.rtol * P.rtol * bb;
    int sweeps = 0, its = 0;
    bool rounded = false;
    while (rr > tol2 && !rounded && sweeps < P.refmax) {
      // scale the residual by 2^-k to a squared norm in [1, 4), so that the CG works on O(1) values
      const int k2 = (((__double2hiint(rr) >> 20) & 0x7ff) - 1023) >> 1;
      const double rr0 = rr * exp2_int(-k2) * exp2_int(-k2);
      V r[NG][4];
#pragma unroll
      for (int k = 0; k < NG; ++k) {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) {
          const ff s = split_scaled(r64[k][j], -k2);
          if constexpr (kMixed)
            r[k][j] = s.h + s.l;
          else
            r[k][j] = s;
        }
      }
      // (the pairs carry a residual to about 1e-15 of its start)
      const double inner2 = P.inner_rtol * P.inner_rtol, final2 = 0.25 * tol2 / rr;
      const float target2 = fmaxf((float)(fmax(inner2, final2) * rr0), 1e-30f);
      // (scale A) d = r gives d / scale
      const double unscale = exp2_int(k2) * ffw.scale;
      its += cg_correct(r, (float)rr0, target2, unscale);
      ++sweeps;
      if constexpr (kMixed)
        update_halos(unscale);
      else
        exchange_x64();
      double v[1] = {residual(r64)};
      allreduce<double, 1>(v);
      if constexpr (kMixed) {
        // a CG that aimed at the tolerance, or gained little: whether rounding is what is left
        if (v[0] > tol2 && (inner2 <= final2 || v[0] > 0.01 * rr)) {
          double u[1] = {diag_x2()};
          allreduce<double, 1>(u);
          rounded = v[0] <= kRounding2 * u[0];
        }
      }
      rr = v[0];
    }
    ax_valid = true;
    if (threadIdx.x == 0 && sb.rank == 0) {
      atomicAdd(&P.stats->solves, 1ull);
      atomicAdd(&P.stats->cg_iters, (unsigned long long)its);
      atomicAdd(&P.stats->refinements, (unsigned long long)sweeps);
      atomicMax(&P.stats->max_cg_iters, (unsigned long long)its);
      atomicAdd(&P.stats->kind_solves[P.stats_kind], 1ull);
      atomicAdd(&P.stats->kind_cg_iters[P.stats_kind], (unsigned long long)its);
      atomicAdd(&P.stats->kind_refinements[P.stats_kind], (unsigned long long)sweeps);
      if (!(rr == rr) || !(bb == bb) || isinf(rr)) {
        record_error(P.stats, PTG_ENONFINITE, P.stats_kind, step);
      } else if (rr > tol2 && !rounded) {
        record_error(P.stats, PTG_ENOCONV, P.stats_kind, step);
      }
    }
  }

  // the local sum of (diag(A) x)^2 (kRounding2)
  __device__ double diag_x2() const {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const double t = unknown(k, j) ? A.C[l0 + gshift + j] * x64[l0 + j] : 0.0;
        s = fma(t, t, s);
      }
    }
    return s;
  }

  // sum over owned free nodes of x64^p, reduced over the cluster (FP64)
  __device__ double pnorm_p() {
    double v[1] = {0.0};
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j)
        if (dinv[l0 + j] != 0.f) v[0] += ipow(x64[l0 + j], P.p_int);
    }
    allreduce<double, 1>(v);
    return v[0];
  }

  // Element term of Eq. 4.7 for the owned elements:
  //   g[e] = gsrc[e] - (1/nnorm) * ( dk_e lambda_e^T Ke T_j,e + dc_e/dt lambda_e^T Me (T_j - T_jm)_e )
  //          (+ addF[e] - subG[e] when given)
  // lambda is x64 (valid halos), T_j / T_jm are full global node vectors.
  __device__ void accumulate_g(const double* __restrict__ Tj, const double* __restrict__ Tjm, double dt_step,
                               double nnorm, const double* __restrict__ gsrc, double* __restrict__ gdst,
                               const double* __restrict__ addF, const double* __restrict__ subG) const {
    const int nx = P.nx, nn = P.nx + 1;
    const int er = min(sb.R, P.ny - sb.r0);  // owned element rows ey in [r0, r0+er)
    const int nel = er > 0 ? er * nx : 0;
    const double mass_scale = P.h * P.h / dt_step, inv_norm = 1.0 / nnorm;
    for (int t = threadIdx.x; t < nel; t += blockDim.x) {
      const int ler = t / nx, ex = t - ler * nx;
      const int ey = sb.r0 + ler;
      const int e = ey * nx + ex;
      const int l0 = (ler + 1) * sb.W + ex + 1;   // SW node in x64
      const Modes l = elem_modes(x64[l0], x64[l0 + 1], x64[l0 + sb.W + 1], x64[l0 + sb.W]);
      const int g0 = ey * nn + ex;
      const double tsw = Tj[g0], tse = Tj[g0 + 1], tne = Tj[g0 + nn + 1], tnw = Tj[g0 + nn];
      double term = P.dk[e] * elem_stiffness(l, elem_modes(tsw, tse, tne, tnw));
      if (P.has_dc)
        term = fma(P.dc[e] * mass_scale,
                   elem_mass(l, elem_modes(tsw - Tjm[g0], tse - Tjm[g0 + 1], tne - Tjm[g0 + nn + 1], tnw - Tjm[g0 + nn])),
                   term);
      double g = fma(-inv_norm, term, gsrc ? gsrc[e] : 0.0);
      if (addF) g += addF[e] - subG[e];
      gdst[e] = g;
    }
  }

  __device__ __forceinline__ double* hist_row(int j) const {
    const int r = j - P.hist_j0;
    if (P.hist == nullptr || r < 0 || r >= P.hist_rows) return nullptr;
    return P.hist + (size_t)r * P.Nn;
  }

  // correction x64 = x64 + F - G on the owned nodes, written to X (and Y if given)
  __device__ void apply_correction(const double* __restrict__ Fs, const double* __restrict__ Gs, double* __restrict__ X,
                                   double* __restrict__ Y) {
    ax_valid = false;
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
#pragma unroll
      for (int j = 0; j < kGroup; ++j) {
        const int g = gnode(l0, j);
        if (g < 0) continue;
        const double t = dinv[l0 + j] != 0.f ? (x64[l0 + j] + Fs[g]) - Gs[g] : 0.0;
        x64[l0 + j] = t;
        X[g] = t;
        if (Y) Y[g] = t;
      }
    }
  }

  // Cumulative objective update with increment sp / N (N Ne the divisor, sp = ||T||_p^p / Ne
  // folded by the caller): the power mean of Sec. 4.4, or the plain sum of the modified
  // objective Theta~ = Theta^p (Sec. 7.1).
  __device__ __forceinline__ double accumulate_theta(double theta, double inc) const {
    return P.objective == PTG_OBJ_MODIFIED ? theta + inc : pow(ipow(theta, P.p_int) + inc, 1.0 / P.p);
  }
  // Factor of T^(p-1) in the adjoint source: Theta^(1-p)/Ne (Eq. 4.6) or p/Ne (Sec. 7.1).
  __device__ __forceinline__ double adjoint_scale(double Theta) const {
    return (P.objective == PTG_OBJ_MODIFIED ? P.p : pow(Theta, 1.0 - P.p)) / (double)P.Ne;
  }

  // Copy the own rows of a node field (stride Nn) from src to dst (and to hist if given).
  __device__ void copy_field(const double* src, double* dst, double* hist) {
#pragma unroll
    for (int k = 0; k < NG; ++k) {
      const int l0 = loc0[k];
      if (l0 < 0) continue;
      for (int j = 0; j < kGroup; ++j) {
        const int g = gnode(l0, j);
        if (g < 0) continue;
        const double v = src[g];
        dst[g] = v;
        if (hist) hist[g] = v;
      }
    }
  }

  // ------------------------------------------------------------------ task bodies
  __device__ void fine_primal(int task) {
    const int sa = P.chained ? P.s0 : P.s0 + task;
    const int sb_end = P.chained ? P.s0 + P.ns : sa + 1;
    const int M = P.M;
    const double inv_norm = 1.0 / ((double)P.Nt * (double)P.Ne);
    set_operator();
    load_x64(P.in_field + (size_t)sa * P.Nn);
    // theta^p (or theta of the modified objective), a plain sum over the steps: the root is taken at
    // the end of a slice only (an FP64 pow takes 6 000 cycles of the one thread that needs it)
    const bool power = P.objective != PTG_OBJ_MODIFIED;
    double theta = power ? ipow(P.in_aux[sa], P.p_int) : P.in_aux[sa];
    if (P.chained) {                              // a sequential run also records its start
      if (double* row = hist_row(M * sa)) store_x64(row);
    }
    const int nring = P.extrap;
    double* ring = nring > 1 && P.prev_field ? P.prev_field + (size_t)task * nring * P.ring_stride : nullptr;
    int saved = 0;                                // states of this slice in the ring
    for (int s = sa; s < sb_end; ++s) {
      for (int j = M * s + 1; j <= M * (s + 1); ++j) {
        const double qj = P.q_time[j];
        build_rhs([&](int g) { return qj * P.fload[g]; });
        // initial guess: the polynomial extrapolation through T_{j-1} (in x64) .. T_{j-n}, kept in
        // a ring of P.extrap rows per task (T_k in row k mod P.extrap; step j writes row
        // (j-1) mod P.extrap and reads the others).  Each slice starts afresh, in a chained run
        // too, so that a slice recomputed alone from its start state (checkpointed
        // differentiation) repeats every solve bit for bit.
        if (ring) {
          if (j == M * s + 1) saved = 0;
          const int n = min(saved + 1, nring);
          const double* X[kMaxExtrap - 1];
          for (int i = 2; i <= n; ++i) X[i - 2] = ring + (size_t)((j - i) % nring) * P.ring_stride;
          if (n >= 2) comm.order_global();   // the neighbours' ring rows
          extrapolate_x64(n, X, ring + (size_t)((j - 1) % nring) * P.ring_stride);
          ++saved;
        }
        solve(j, ring == nullptr);
        const double sp = pnorm_p();
        theta = fma(sp, inv_norm, theta);
        if (double* row = hist_row(j)) store_x64(row);
      }
      store_x64(P.out_field + (size_t)s * P.Nn);
      if (threadIdx.x == 0 && sb.rank == 0) P.out_aux[s] = power ? pow(theta, 1.0 / P.p) : theta;
    }
  }

  __device__ void coarse_primal(int task) {
    const int s = P.s0 + task;
    set_operator();
    load_x64(P.in_field + (size_t)s * P.Nn);
    const double theta0 = P.in_aux[s];
    const int j = P.M * (s + 1);
    if (P.src_field) {                          // a given source per slice (coarse-mesh G)
      const double* src = P.src_field + (size_t)s * P.Nn;
      build_rhs([&](int g) { return src[g]; });
    } else {
      const double qj = P.q_time[j];
      build_rhs([&](int g) { return qj * P.fload[g]; });
    }
    if (P.guess_next) load_x64(P.in_field + (size_t)(s + 1) * P.Nn);   // start from the guess u_{s+1}
    solve(j);
    const double sp = pnorm_p();
    store_x64(P.out_field + (size_t)s * P.Nn);
    if (threadIdx.x == 0 && sb.rank == 0) P.out_aux[s] = accumulate_theta(theta0, sp / ((double)P.Ntau * (double)P.Ne));
  }

  __device__ void correct_primal() {
    if (!P.plt) set_operator();
    double theta;
    if (P.in_field) {                           // u_0 taken from the guess states, copied to X[0]
      load_x64(P.in_field);
      store_x64(P.out_field);
      theta = P.in_aux[0];
      if (threadIdx.x == 0 && sb.rank == 0) P.out_aux[0] = theta;
    } else {                                    // u_0 given in X[0]
      load_x64(P.out_field);
      theta = P.out_aux[0];
    }
    if (double* row = hist_row(0)) store_x64(row);
    if (P.plt) {                                // G = 0 (Sec. 7, Eq. 7.2): u_{s+1} = F(u_s^old)
      for (int s = 0; s < P.Ntau; ++s) {
        copy_field(P.F_field + (size_t)s * P.Nn, P.out_field + (size_t)(s + 1) * P.Nn, hist_row(P.M * (s + 1)));
        if (threadIdx.x == 0 && sb.rank == 0) P.out_aux[s + 1] = P.F_aux[s];
      }
      return;
    }
    for (int s = 0; s < P.Ntau; ++s) {
      const int j = P.M * (s + 1);
      if (P.src_field) {                        // a given source per slice (coarse-mesh G)
        const double* src = P.src_field + (size_t)s * P.Nn;
        build_rhs([&](int g) { return src[g]; });
      } else {
        const double qj = P.q_time[j];
        build_rhs([&](int g) { return qj * P.fload[g]; });
      }
      // initial guess G(u_s^old) plus the extrapolation of the increments G(u^new) - G(u^old) of
      // the last min(extrap - 1, s) steps, the increment of step s-1-i being u_{s-i}^new - F[s-1-i]
      // by the correction itself (plain: G(u_s^old))
      const int m = min(P.extrap - 1, min(s, 3));
      if (m >= 1) {
        const double* Fm[3];
        const double* X[3] = {nullptr, nullptr, nullptr};
        for (int i = 0; i < m; ++i) Fm[i] = P.F_field + (size_t)(s - 1 - i) * P.Nn;
        for (int i = 1; i < m; ++i) X[i] = P.out_field + (size_t)(s - i) * P.Nn;
        if (m >= 2) comm.order_global();      // the neighbours' rows of the corrected states
        load_x64_increment(P.G_field + (size_t)s * P.Nn, m, Fm, X);
      } else {
        load_x64(P.G_field + (size_t)s * P.Nn);
      }
      solve(j);
      const double sp = pnorm_p();
      apply_correction(P.F_field + (size_t)s * P.Nn, P.G_field + (size_t)s * P.Nn,
                       P.out_field + (size_t)(s + 1) * P.Nn, hist_row(j));
      if (threadIdx.x == 0) {                    // theta is needed by thread 0 only
        const double theta_g = accumulate_theta(theta, sp / ((double)P.Ntau * (double)P.Ne));
        theta = (theta_g + P.F_aux[s]) - P.G_aux[s];
        if (sb.rank == 0) P.out_aux[s + 1] = theta;
      }
      exchange_x64();
    }
  }

  __device__ void fine_adjoint(int task) {
    const int s_lo = P.chained ? P.s0 : P.s0 + task;
    const int s_hi = P.chained ? P.s0 + P.ns - 1 : s_lo;
    const int M = P.M;
    const double Theta = *P.Theta;
    const double scale = adjoint_scale(Theta);
    set_operator();
    load_x64(P.in_field + (size_t)(s_hi + 1) * P.Nn);
    const double* gsrc = P.in_aux + (size_t)(s_hi + 1) * P.Ne;
    // initial guess: the extrapolation through lambda_{j+1} (in x64) .. lambda_{j+n}, kept in a
    // ring of P.extrap rows per task, lambda_k in row k mod P.extrap; step j writes row
    // (j+1) mod P.extrap and reads the n-1 <= P.extrap-1 others, so no CTA writes a row that a
    // neighbour reads in the same step
    const int nring = P.extrap;
    double* ring = nring > 1 && P.prev_field ? P.prev_field + (size_t)task * nring * P.ring_stride : nullptr;
    int saved = 0;   // states of this slice in the ring
    for (int s = s_hi; s >= s_lo; --s) {
      double* gdst = P.out_aux + (size_t)s * P.Ne;
      saved = 0;     // each slice starts afresh, as in the primal
      for (int j = M * (s + 1); j >= M * s + 1; --j) {
        const double* Tj = hist_row(j);
        const double* Tjm = hist_row(j - 1);
        if (Tj == nullptr || Tjm == nullptr) {   // host validation makes this unreachable
          if (threadIdx.x == 0 && sb.rank == 0) record_error(P.stats, PTG_EINVAL, P.stats_kind, j);
          return;
        }
        build_rhs([&](int g) { return scale * ipow(Tj[g], P.p_int - 1); });
        if (ring) {
          const int n = min(saved + 1, nring);
          const double* X[kMaxExtrap - 1];
          for (int i = 2; i <= n; ++i) X[i - 2] = ring + (size_t)((j + i) % nring) * P.ring_stride;
          if (n >= 2) comm.order_global();   // the neighbours' ring rows
          extrapolate_x64(n, X, ring + (size_t)((j + 1) % nring) * P.ring_stride);
          ++saved;
        }
        solve(j, ring == nullptr);
        accumulate_g(Tj, Tjm, P.dt, (double)P.Nt, gsrc, gdst, nullptr, nullptr);
        gsrc = gdst;
        __syncthreads();
      }
      store_x64(P.out_field + (size_t)s * P.Nn);
    }
  }

  // G_adj of slice s; with P.src_mode 1 or 2 one of its two parts (G_adj is affine in the source
  // scale c of Eq. 4.6): 1 the solve and g update driven by v_{s+1} with c = 0, 2 those of the
  // unit source (c = 1) from lambda = 0 and g = 0.  The parts start from the state they
  // propagate (zero for part 2).
  __device__ void coarse_adjoint(int task) {
    const int s = P.s0 + task;
    const int kidx = P.M * s + 1;
    const int kprev = max(kidx - P.M, 0);
    const double scale = P.src_mode == 0 ? adjoint_scale(*P.Theta) : (P.src_mode == 1 ? 0.0 : 1.0);
    const double* Tk = P.hist + (size_t)kidx * P.Nn;
    const double* Tkm = P.hist + (size_t)kprev * P.Nn;
    set_operator();
    if (P.src_mode == 2)
      zero_x64();
    else
      load_x64(P.in_field + (size_t)(s + 1) * P.Nn);
    build_rhs([&](int g) { return scale * ipow(Tk[g], P.p_int - 1); });
    if (P.guess_next && P.src_mode == 0) load_x64(P.in_field + (size_t)s * P.Nn);   // start from the guess lambda_s
    solve(kidx);
    accumulate_g(Tk, Tkm, P.dtau, (double)P.Ntau, P.src_mode == 2 ? nullptr : P.in_aux + (size_t)(s + 1) * P.Ne,
                 P.out_aux + (size_t)s * P.Ne, nullptr, nullptr);
    store_x64(P.out_field + (size_t)s * P.Nn);
  }

  __device__ void correct_adjoint() {
    const double Theta = *P.Theta;
    const double scale = adjoint_scale(Theta);
    if (!P.plt) set_operator();
    // v_Ntau = 0
    {
      double* Xl = P.out_field + (size_t)P.Ntau * P.Nn;
#pragma unroll
      for (int k = 0; k < NG; ++k) {
        const int l0 = loc0[k];
        if (l0 < 0) continue;
        for (int j = 0; j < kGroup; ++j) {
          const int g = gnode(l0, j);
          if (g >= 0) Xl[g] = 0.0;
        }
      }
      const int er = min(sb.R, P.ny - sb.r0);
      double* Xg = P.out_aux + (size_t)P.Ntau * P.Ne;
      for (int t = threadIdx.x; t < (er > 0 ? er * P.nx : 0); t += blockDim.x) Xg[sb.r0 * P.nx + t] = 0.0;
    }
    if (P.plt) {                                // G = 0 (Sec. 7, Eq. 7.2): v_s = F(v_{s+1}^old)
      const int er = min(sb.R, P.ny - sb.r0);
      for (int s = P.Ntau - 1; s >= 0; --s) {
        copy_field(P.F_field + (size_t)s * P.Nn, P.out_field + (size_t)s * P.Nn, nullptr);
        const double* Fg = P.F_aux + (size_t)s * P.Ne + sb.r0 * P.nx;
        double* Xg = P.out_aux + (size_t)s * P.Ne + sb.r0 * P.nx;
        for (int t = threadIdx.x; t < (er > 0 ? er * P.nx : 0); t += blockDim.x) Xg[t] = Fg[t];
      }
      return;
    }
    zero_x64();
    for (int s = P.Ntau - 1; s >= 0; --s) {
      const int kidx = P.M * s + 1;
      const int kprev = max(kidx - P.M, 0);
      const double* Tk = P.hist + (size_t)kidx * P.Nn;
      const double* Tkm = P.hist + (size_t)kprev * P.Nn;
      build_rhs([&](int g) { return scale * ipow(Tk[g], P.p_int - 1); });
      // initial guess G(v_{s+1}^old) plus the extrapolation of the increments of the last
      // min(extrap - 1, Ntau - 1 - s) steps, the increment of step s+1+i being
      // v_{s+1+i}^new - F[s+1+i] (plain: G(v_{s+1}^old))
      const int m = min(P.extrap - 1, min(P.Ntau - 1 - s, 3));
      if (m >= 1) {
        const double* Fm[3];
        const double* X[3] = {nullptr, nullptr, nullptr};
        for (int i = 0; i < m; ++i) Fm[i] = P.F_field + (size_t)(s + 1 + i) * P.Nn;
        for (int i = 1; i < m; ++i) X[i] = P.out_field + (size_t)(s + 1 + i) * P.Nn;
        load_x64_increment(P.G_field + (size_t)s * P.Nn, m, Fm, X);
      } else {
        load_x64(P.G_field + (size_t)s * P.Nn);
      }
      solve(kidx);
      // g_s = g_{s+1} - (1/Ntau) term(lambda_G) + F_g[s] - G_g[s]
      accumulate_g(Tk, Tkm, P.dtau, (double)P.Ntau, P.out_aux + (size_t)(s + 1) * P.Ne, P.out_aux + (size_t)s * P.Ne,
                   P.F_aux + (size_t)s * P.Ne, P.G_aux + (size_t)s * P.Ne);
      comm.sync();                              // every CTA is done reading lambda_G halos; also orders the
                                                // corrected states of the steps before for the next start
      apply_correction(P.F_field + (size_t)s * P.Nn, P.G_field + (size_t)s * P.Nn, P.out_field + (size_t)s * P.Nn,
                       nullptr);
      exchange_x64();
    }
  }
};

// One kernel per (precision, groups per thread, task kind); each kernel inlines a single task
// body, which keeps register pressure and compile time down.  Up to 512 threads per CTA (the
// plan picks the block size), at most 128 registers per thread.
constexpr int kStepMaxThreads = 512;
// Blocks of at most kStepNarrowThreads threads run a second instantiation of the same kernel that
// may use 168 registers: at 128 the CG of the FP32 kinds with two or three groups per thread and the
// three-level cycle spill (up to 750 bytes a thread).

template <int KIND>
constexpr bool kCoarseStep = KIND != KIND_FINE_PRI && KIND != KIND_FINE_ADJ;

template <class Real, int NG, int KIND, class Comm>
__device__ __forceinline__ void run_task(Stepper<Real, NG, Comm, kCoarseStep<KIND>>& st, int task) {
  if constexpr (KIND == KIND_FINE_PRI) st.fine_primal(task);
  if constexpr (KIND == KIND_COARSE_PRI) st.coarse_primal(task);
  if constexpr (KIND == KIND_CORRECT_PRI) st.correct_primal();
  if constexpr (KIND == KIND_FINE_ADJ) st.fine_adjoint(task);
  if constexpr (KIND == KIND_COARSE_ADJ) st.coarse_adjoint(task);
  if constexpr (KIND == KIND_CORRECT_ADJ) st.correct_adjoint();
}

template <class Real, int NG, int KIND, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) stepper_kernel(const __grid_constant__ StepParams P) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  __shared__ RedSmem rs;
  ClusterComm comm(rs);
  comm.bind(P);
  Stepper<Real, NG, ClusterComm, kCoarseStep<KIND>> st(P, comm, dyn_smem);
  // every CTA of the cluster has initialised its shared memory before any DSMEM traffic
  cluster_sync_all();
  run_task<Real, NG, KIND>(st, (int)(blockIdx.x / (unsigned)P.cs));
  // no CTA leaves while another may still read or write its shared memory
  cluster_sync_all();
  comm.drain();
}

// Systems spread over groups of CTAs of a cooperative launch: the grid holds gridDim.x / P.cs
// groups of P.cs CTAs (one slab each); group g runs tasks g, g + groups, ... < P.wide_tasks one
// after the other.  Halo rows, reduction partials and the two-level partials go through global
// memory (GridComm).  Used for one FP64 system over every SM, and for grids whose slabs do not
// fit the 16 CTAs of a cluster.
template <class Real, int NG, int KIND>
__global__ void __launch_bounds__(kStepMaxThreads, 1) stepper_wide_kernel(const __grid_constant__ StepParams P) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  __shared__ RedSmem rs;
  GridComm comm(P, rs);
  const int ngroups = (int)gridDim.x / P.cs;
  for (int task = comm.gid; task < P.wide_tasks; task += ngroups) {
    Stepper<Real, NG, GridComm, kCoarseStep<KIND>> st(P, comm, dyn_smem);
    run_task<Real, NG, KIND>(st, task);
    comm.sync();                               // the group's halo slots are free again
  }
}

// Persistent multi-design variant: `tasks` lists (design, task) pairs, largest designs first;
// every cluster claims the next pair from the work queue until the list is exhausted, and
// runs it with that design's parameters (table[design]).  All designs share the precision,
// the cluster size, the block size and NG; shared memory is carved per task for the design's
// geometry from the largest footprint that the launch reserves.
template <class Real, int NG, int KIND>
__global__ void __launch_bounds__(kStepMaxThreads, 1) stepper_batch_kernel(const StepParams* __restrict__ table,
                                                                       const int2* __restrict__ tasks, int ntasks,
                                                                       int* __restrict__ queue) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  __shared__ RedSmem rs;
  __shared__ int s_task, s_dead;               // s_dead (of rank 0): a CTA of the cluster gave up
  ClusterComm comm(rs);
  const unsigned rank = comm.cl.block_rank();
  if (threadIdx.x == 0) s_dead = 0;
  cluster_sync_all();                          // all CTAs running before any DSMEM store
  for (;;) {
    // rank 0 claims the next task and writes it into every CTA of the cluster; the barrier
    // publishes it (and orders it after the previous task's last shared-memory access).  Once a wait has
    // run out the cluster's exchanges are of no use any more: it claims on (~t), so that the designs
    // whose tasks it takes learn of it, and runs none of them.
    if (rank == 0 && threadIdx.x == 0) {
      const int t = atomicAdd(queue, 1), claim = s_dead ? ~t : t;
      for (unsigned r = 0; r < comm.cl.num_blocks(); ++r) *comm.cl.map_shared_rank(&s_task, r) = claim;
    }
    cluster_sync_all();
    const int claim = s_task, t = claim < 0 ? ~claim : claim;   // identical in every CTA: the loop is uniform
    if (t >= ntasks) break;
    const int2 tk = tasks[t];
    if (claim < 0) {
      if (rank == 0 && threadIdx.x == 0) record_error(table[tk.x].stats, PTG_ETIMEOUT, table[tk.x].stats_kind, -1);
    } else {
      comm.bind(table[tk.x]);
      Stepper<Real, NG, ClusterComm, kCoarseStep<KIND>> st(table[tk.x], comm, dyn_smem);
      cluster_sync_all();
      run_task<Real, NG, KIND>(st, tk.y);
      __syncthreads();
      if (threadIdx.x == 0 && comm.dead()) *comm.cl.map_shared_rank(&s_dead, 0u) = 1;
    }
    cluster_sync_all();
  }
  comm.drain();
}

}  // namespace ptg
