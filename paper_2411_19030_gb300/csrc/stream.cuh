// stream.cuh -- propagators of large grids with the Krylov vectors in global memory: the fine
// propagators (a2, a5), and the coarse propagators (a3) and correction sweeps (a4) with FP64 CG;
// each CG preconditioned by Jacobi or by a geometric multigrid V-cycle in FP32 of its step's
// operator (see "multigrid" below).
//
// The cluster stepper keeps a system's CG vectors on chip, so at 512 x 512 a slice needs the
// shared memory and registers of about 50 SMs and only 3 of 128 slices run at once.  Here every
// slice is a group of G CTAs of one launch (G = 1 or 2 at 512 x 512, one or two per SM), and
// its vectors stream from HBM: x (FP64, two buffers: the state a step starts from and the one
// it solves for), the right-hand side b and the residual (FP64), and the CG vectors r, p, q, d.
// All Ntau slices then advance together and the solves are bound by HBM bandwidth.
//
// Each step is the same as the stepper's (stepper.cuh): b = (C/dt) x_{j-1} + source, the start
// extrapolated through the slice's last states (the same ring of states per task), the FP64
// residual loop around a preconditioned CG on A d = r / 2^k, then theta (primal) or the Eq. 4.7
// element sums (adjoint).  The CG's vectors are floats, or float pairs (ff.cuh) in the FP64 kinds,
// its preconditioned vector z a float.  Per CG iteration the group sums two sets of dot products
// (fixed order, identical in every CTA of the group: GridComm) and each CTA streams its rows.
//
// What bounds the passes: at one CTA of 512 threads per SM a pass that loads its stencil operands
// straight from global memory waits for them (256 x 256 and 512 x 512: 5 100 cycles per 512 groups
// of 4 nodes, 12% of the HBM bandwidth).  The passes of the multigrid cycle's large levels and the
// FP32 CG's operator therefore march down the rows through a ring in shared memory that bulk copies
// (cp.async.bulk) fill several rows ahead (march below).
#pragma once
#include "comm.cuh"

namespace ptg {

constexpr int kStreamThreads = 512;   // one CTA per SM, 128 registers per thread
constexpr int kPipeRows = 32;         // most rows of a ring (one mbarrier each)

// Weights of a ring row per node: level 0 has the element form (omega/diag, k, m: stencil_km32's k_e/6
// and c_e h^2/(36 step)), which halves the bytes of a pass (the passes of 128 slices were bound by
// the weights' way from L2: 12 bytes per cycle and SM); a Galerkin level its six node weights.
constexpr int kElemWeights = 3, kNodeWeights = 6;
constexpr int kPipeBytes = 200 * 1024;
// rows of the ring that holds a level's residual until it is restricted (G4 groups per row): those
// of two trips of 512 groups and the ones that wait for their last row
inline __host__ __device__ int res_rows(int G4) { return 2 * ((kStreamThreads - 1) / G4 + 2) + 4; }
// rows that 512 consecutive groups touch, with a row on each side
inline __host__ __device__ int trip_rows(int G4) { return (kStreamThreads - 1) / G4 + 4; }
// Rows of a level's ring: a trip's rows and up to 16 ahead if the shared memory allows; 0 where
// fewer than 2 ahead remain (short rows, whose 512 groups span too many of them, and rows of more
// than 3 KB): such levels load straight from global memory.
inline __host__ __device__ int pipe_rows(int G4, int weights) {
  const int need = trip_rows(G4);
  const int cap = (kPipeBytes / (16 * G4) - res_rows(G4)) / (1 + weights);
  const int rows = cap < need + 16 ? cap : need + 16;
  return need <= 32 && rows >= need + 2 ? rows : 0;
}
// Rows of a bulk copy: the largest chunk of which the ring holds a trip's rows, wherever they
// start, and one more chunk.  A bulk copy costs about 175 cycles of the copy engine whatever its
// size (1 KB and 2 KB rows alike), so the weights of a level are interleaved row by row and a
// chunk is two copies.
inline __host__ __device__ int chunk_rows(int S, int need) {
  int c = (S - need + 1) / 2;
  while (c > 1 && (S / c) * c < need + 2 * c - 1) --c;
  return c < 1 ? 1 : c;
}
// shared memory of a level's rings
inline size_t pipe_bytes(int G4, int weights) {
  return 16 * (size_t)G4 * (size_t)((1 + weights) * pipe_rows(G4, weights) + res_rows(G4));
}

template <class Real, int KIND>
struct Streamer {
  static constexpr bool kMixed = std::is_same<Real, float>::value;
  using V = typename std::conditional<kMixed, float, ff>::type;
  const StepParams& P;
  GridComm& comm;
  int rank = 0, r0 = 0, R = 0;   // this CTA's node rows [r0, r0 + R) of the group's system
  int nn = 0;                    // nodes per row (nx + 1)
  int G4 = 0;                    // groups of 4 nodes per padded row (W / 4)
  // group workspace, padded node layout (node (iy, ix) at (iy + 1) W + ix + 1, the layout of the
  // per-node weights), zero off the unknowns
  double *xa = nullptr, *xb = nullptr, *b = nullptr, *res = nullptr;
  float *r = nullptr, *z = nullptr, *p = nullptr, *q = nullptr, *d = nullptr;   // high parts; low parts
  size_t lo = 0;                                                                // `lo` floats after (FP64 kinds)
  double step_dt = 0.0, inv_dt = 0.0;
  static constexpr bool kCoarse = KIND == KIND_COARSE_PRI || KIND == KIND_COARSE_ADJ || KIND == KIND_CORRECT_PRI ||
                                  KIND == KIND_CORRECT_ADJ;
  NodeWeights A64;               // the operator of the kind's step: C/dt + K or C/dtau + K
  FFWeights ffw;                 // the same as float pairs
  float* mgws = nullptr;         // the group's multigrid workspace
  // the row ring: shared memory, one mbarrier per row slot and the parity each waits for next
  float* ring_sm;
  unsigned long long* ring_bar;
  unsigned& ring_phase;
  bool& ring_dead;               // a wait for rows ran out (the same in every thread)

  __device__ Streamer(const StepParams& P_, GridComm& comm_, float* sm, unsigned long long* bar, unsigned& phase, bool& dead)
      : P(P_), comm(comm_), ring_sm(sm), ring_bar(bar), ring_phase(phase), ring_dead(dead) {
    rank = comm.rank();
    slab_rows(P.ny + 1, P.cs, rank, r0, R);
    nn = P.nx + 1;
    G4 = P.W / kGroup;
    const int grp = (int)blockIdx.x / P.cs;
    const size_t pv = (size_t)P.st_pv;                 // entries of one padded vector incl. slack
    double* w64 = P.st_w64 + (size_t)grp * 4 * pv + kSlack;
    xa = w64;
    xb = w64 + pv;
    b = w64 + 2 * pv;
    res = w64 + 3 * pv;
    constexpr int kParts = kMixed ? 1 : 2;
    float* wr = reinterpret_cast<float*>(P.st_wr) + (size_t)grp * 5 * kParts * pv + kSlack;
    lo = pv;
    r = wr;
    z = wr + kParts * pv;
    p = wr + 2 * kParts * pv;
    q = wr + 3 * kParts * pv;
    d = wr + 4 * kParts * pv;
    step_dt = kCoarse ? P.dtau : P.dt;
    inv_dt = 1.0 / step_dt;
    A64 = kCoarse ? P.A_coarse : P.A_fine;
    ffw = kCoarse ? P.ff_coarse : P.ff_fine;
    if (P.mg_levels > 0) mgws = P.mg_ws + (size_t)grp * P.mg_ws_stride;
  }

  // Visit this CTA's groups of 4 nodes (columns 4g-1 .. 4g+2 of an owned row): f(loc, iy, g) with
  // loc the padded index of the group's first node (16-byte aligned).
  template <class F>
  __device__ __forceinline__ void for_groups(F f) const {
    for (int t = threadIdx.x; t < R * G4; t += blockDim.x) {
      const int lr = t / G4, g = t - lr * G4, iy = r0 + lr;
      f((iy + 1) * P.W + kGroup * g, iy, g);
    }
  }

  // Two groups per loop trip (t and t + blockDim.x): f(loc[2], ok[2]) loads both groups' operands
  // before it computes, so each thread keeps twice the memory requests in flight.
  template <class F>
  __device__ __forceinline__ void for_group_pairs(F f) const {
    const int n = R * G4;
    for (int t0 = threadIdx.x; t0 < n; t0 += 2 * blockDim.x) {
      int loc[2];
      bool ok[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int t = t0 + u * (int)blockDim.x;
        ok[u] = t < n;
        const int lr = ok[u] ? t / G4 : 0, g = ok[u] ? t - lr * G4 : 0;
        loc[u] = (r0 + lr + 1) * P.W + kGroup * g;
      }
      f(loc, ok);
    }
  }

  // node index of column 4g-1+j of row iy, or -1 for a pad column
  __device__ __forceinline__ int gnode(int iy, int g, int j) const {
    const int ix = kGroup * g - 1 + j;
    return (ix >= 0 && ix <= P.nx) ? iy * nn + ix : -1;
  }

  // 1/C of the 4 nodes (0 off the unknowns)
  __device__ __forceinline__ void dinv4(int loc, float (&v)[4]) const { ld4f(P.w32_inv, loc, v); }
  __device__ __forceinline__ void ld4f(const float* __restrict__ a, int loc, float (&v)[4]) const {
    const float4 c = *reinterpret_cast<const float4*>(a + loc);
    v[0] = c.x; v[1] = c.y; v[2] = c.z; v[3] = c.w;
  }
  __device__ __forceinline__ void st4f(float* __restrict__ a, int loc, const float (&v)[4]) const {
    *reinterpret_cast<float4*>(a + loc) = make_float4(v[0], v[1], v[2], v[3]);
  }
  // a CG vector's entries on a group
  __device__ __forceinline__ void ldv(const float* __restrict__ a, int loc, V (&v)[4]) const {
    if constexpr (kMixed) {
      ld4f(a, loc, v);
    } else {
      float h[4], l[4];
      ld4f(a, loc, h);
      ld4f(a + lo, loc, l);
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = make_ff(h[j], l[j]);
    }
  }
  __device__ __forceinline__ void stv(float* __restrict__ a, int loc, const V (&v)[4]) const {
    if constexpr (kMixed) {
      st4f(a, loc, v);
    } else {
      float h[4], l[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h[j] = v[j].h;
        l[j] = v[j].l;
      }
      st4f(a, loc, h);
      st4f(a + lo, loc, l);
    }
  }
  __device__ __forceinline__ void st4d(double* __restrict__ a, int loc, const double (&v)[4]) const {
    *reinterpret_cast<double2*>(a + loc) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(a + loc + 2) = make_double2(v[2], v[3]);
  }

  // Group barriers after a pass whose stores bulk copies of the next may read (r, z, the right-hand
  // side of a large level): every thread orders its stores before the barrier for the async proxy.
  __device__ __forceinline__ void sync() {
    asm volatile("fence.proxy.async.global;" ::: "memory");
    comm.sync();
  }
  template <class T, int NV, int NX = 0, class Post = NoPost>
  __device__ __forceinline__ void allreduce(T (&v)[NV + NX], Post post = Post()) {
    asm volatile("fence.proxy.async.global;" ::: "memory");
    comm.template allreduce<T, NV, NX, Post>(v, P.cs, post);
  }

  // ------------------------------------------------------------------ row rings
  static __device__ __forceinline__ void bulk_load(unsigned dst, const float* src, unsigned bytes, unsigned bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
  }
  // Waits for a chunk; false where the wait ran out (P.wait_limit).
  __device__ __forceinline__ bool ring_wait(int slot) {
    unsigned long long* bar = ring_bar + slot;
    const unsigned parity = (ring_phase >> slot) & 1u;
    if (!mbar_test(bar, parity) && !mbar_wait(bar, parity, P.wait_limit)) return false;
    ring_phase ^= 1u << slot;
    return true;
  }
  // The rows below, at and above a group's row in the ring: the vector (v) and the weights (w, array
  // a of C, E, N, NE, NW, omega/diag, or of omega/diag, k, m)
  template <int NW>
  struct RowRef {
    const float *vec, *wts;   // the ring's vector rows and weight rows
    int W, so, sm, su;        // row indexes in the ring
    __device__ __forceinline__ const float* v(int s) const { return vec + s * W; }
    __device__ __forceinline__ const float* w(int s, int a) const { return wts + (NW * s + a) * W; }
    __device__ __forceinline__ const float* wd(int s) const { return w(s, NW == kNodeWeights ? 5 : 0); }
  };
  // Visit the groups of rows ya .. yb of level l, 512 consecutive groups at a time: body(rows, y, g,
  // ok) finds the rows y-1, y, y+1 of the vector `vec` (padded layout of the level) and of the
  // level's weights in shared memory (every lane calls it; one without a group has ok = false and
  // the last group's operands), then after(y_done) runs behind a block barrier, rows below y_done
  // visited.  The rows ya-1 .. yb+1 (all inside the padded layout) come in chunks of CR rows, one
  // mbarrier and two bulk copies each; a chunk's slot is filled again once its rows are done.  Where a
  // wait of any thread runs out, the CTA learns of it at the trip's block barrier: thread 0 waits for the
  // copies in flight, the group gives up (its reductions return NaN, which ends the solve), and this CTA
  // starts no march any more.
  template <int NW, class Body, class After>
  __device__ __forceinline__ void march(int l, const float* vec, int ya, int yb, Body body, After after) {
    if (ring_dead) return;
    const int Wl = P.mg[l].W, G4l = Wl / kGroup, first = ya - 1, nr = yb - ya + 3, n = (yb - ya + 1) * G4l;
    const int Smax = pipe_rows(G4l, NW), CR = nr <= Smax ? nr : chunk_rows(Smax, trip_rows(G4l));
    const int NS = Smax / CR, S = NS * CR, nchunks = (nr + CR - 1) / CR;
    float* svec = ring_sm;
    float* swts = ring_sm + Smax * Wl;
    const float* gvec = vec + (size_t)(first + 1) * Wl;
    const float* gwts = (NW == kNodeWeights ? lwb(l) : P.mg_elem + kSlack) + (size_t)(first + 1) * NW * Wl;
    int issued = 0, ready = 0;
    auto issue = [&](int upto) {           // chunks
      if (threadIdx.x != 0) return;
      for (; issued < upto; ++issued) {
        const int slot = issued % NS, row = issued * CR, rows = min(CR, nr - row);
        const unsigned bytes = 4u * (unsigned)(rows * Wl), bar = smem_u32(ring_bar + slot);
        mbar_expect(ring_bar + slot, (1u + NW) * bytes);
        bulk_load(smem_u32(svec + slot * CR * Wl), gvec + (size_t)row * Wl, bytes, bar);
        bulk_load(smem_u32(swts + slot * CR * NW * Wl), gwts + (size_t)row * NW * Wl, NW * bytes, bar);
      }
    };
    if (threadIdx.x == 0) asm volatile("fence.proxy.async;" ::: "memory");
    issue(min(NS, nchunks));
    for (int t0 = 0; t0 < n; t0 += kStreamThreads) {
      const int t = t0 + (int)threadIdx.x, tc = min(t, n - 1);
      const int need = ((min(n, t0 + kStreamThreads) - 1) / G4l + 2) / CR;   // last chunk of the trip
      bool out = false;
      for (; ready <= need; ++ready) {
        out = !ring_wait(ready % NS);
        if (out) break;
      }
      const int ry = tc / G4l, g = tc - ry * G4l;
      RowRef<NW> rr;
      rr.vec = svec;
      rr.wts = swts;
      rr.W = Wl;
      rr.so = ry % S;
      rr.sm = rr.so + 1 == S ? 0 : rr.so + 1;
      rr.su = rr.sm + 1 == S ? 0 : rr.sm + 1;
      body(rr, ya + ry, g, t < n);
      if (__syncthreads_or(out)) {
        ring_dead = true;
        if (threadIdx.x == 0) {
          for (; ready < issued; ++ready) mbar_wait(ring_bar + ready % NS, (ring_phase >> (ready % NS)) & 1u, 0);
          comm.give_up();
        }
        break;
      }
      const int done = min(n, t0 + kStreamThreads) / G4l;   // whole rows visited: chunks below are free
      issue(min(nchunks, done / CR + NS));
      after(ya + done);
    }
    // the ring is free for the next pass, whose copies may overwrite what `after` left in it
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
  }
  // 6-entry window of a group in a ring row; entries beyond the lane's own 16 bytes come from the
  // neighbouring lanes (their groups follow one another, a row's last entry is a zero pad)
  __device__ __forceinline__ void rwin(const float* row, int g, int G4l, float (&w)[6]) const {
    const int lane = threadIdx.x & 31;
    const float* x = row + kGroup * g;
    const float4 c = *reinterpret_cast<const float4*>(x);
    float e = 0.f;
    if (lane == 0 && g > 0) e = x[-1];
    if (lane == 31 && g < G4l - 1) e = x[4];
    const float l = __shfl_up_sync(0xffffffffu, c.w, 1), u = __shfl_down_sync(0xffffffffu, c.x, 1);
    w[0] = lane == 0 ? e : l;
    w[1] = c.x; w[2] = c.y; w[3] = c.z; w[4] = c.w;
    w[5] = lane == 31 ? e : u;
  }
  // A v on a group from v's windows and the weights' rows in the ring
  __device__ __forceinline__ void rstencil(const RowRef<kElemWeights>& rr, int g, int G4l, const float (&vl)[6],
                                           const float (&vm)[6], const float (&vh)[6], float (&y)[4]) const {
    float kl[6], ml[6], ku[6], mu[6];
    rwin(rr.w(rr.so, 1), g, G4l, kl);
    rwin(rr.w(rr.so, 2), g, G4l, ml);
    rwin(rr.w(rr.sm, 1), g, G4l, ku);
    rwin(rr.w(rr.sm, 2), g, G4l, mu);
    km_combine(vl, vm, vh, kl, ml, ku, mu, y);
  }
  __device__ __forceinline__ void rstencil(const RowRef<kNodeWeights>& rr, int g, int G4l, const float (&vl)[6],
                                           const float (&vm)[6], const float (&vh)[6], float (&y)[4]) const {
    float c4[4], n4[4], ne4[4], nw4[4], nb[4], e6[6], s6[6], t6[6];
    ld4f(rr.w(rr.sm, 0), kGroup * g, c4);
    rwin(rr.w(rr.sm, 1), g, G4l, e6);
    ld4f(rr.w(rr.sm, 2), kGroup * g, n4);
    ld4f(rr.w(rr.sm, 3), kGroup * g, ne4);
    ld4f(rr.w(rr.sm, 4), kGroup * g, nw4);
    ld4f(rr.w(rr.so, 2), kGroup * g, nb);
    rwin(rr.w(rr.so, 3), g, G4l, s6);     // NE of the row below: the south-west neighbours' weights
    rwin(rr.w(rr.so, 4), g, G4l, t6);     // NW of the row below: the south-east neighbours' weights
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float a = c4[j] * vm[j + 1];
      a = fmaf(e6[j + 1], vm[j + 2], a);
      a = fmaf(e6[j], vm[j], a);
      a = fmaf(n4[j], vh[j + 1], a);
      a = fmaf(nb[j], vl[j + 1], a);
      a = fmaf(ne4[j], vh[j + 2], a);
      a = fmaf(s6[j], vl[j], a);
      a = fmaf(nw4[j], vh[j], a);
      a = fmaf(t6[j + 2], vl[j + 2], a);
      y[j] = a;
    }
  }

  // ------------------------------------------------------------------ multigrid
  // z = M^-1 r by one V(1, 1)-cycle over the levels of mg.cu, all in FP32:
  //   level l < L-1: u = S f (one damped-Jacobi step from zero), f_{l+1} = P^T (f - A u),
  //                  e_{l+1} from the level below, u' = u + P e_{l+1}, e = u' + S (f - A u');
  //   level L-1:     e = mg_coarse_steps damped-Jacobi steps from zero,
  // with f = r (its high parts) on level 0 and e = z there.  Pre- and post-smoothing are the same
  // symmetric step and restriction is the transpose of prolongation, so M^-1 is symmetric (and
  // positive definite: omega lambda_max(D^-1 A) < 2), as CG needs.  Levels with few rows run on the
  // group's first CTA alone with block barriers; a barrier between passes on two such levels is
  // a block barrier, every other one the group's barrier.  A large level is one march down (the
  // residual is restricted from shared memory) and one up (u is formed again from f).
  // level l's weights: six arrays (C, E, N, NE, NW, omega/diag) interleaved row by row, so array a of
  // node (iy, ix) is at (6 (iy + 1) + a) W + ix + 1
  __device__ __forceinline__ const float* lwb(int l) const { return P.mg_w + P.mg[l].woff + kSlack; }
  __device__ __forceinline__ const float* lw(int l, int a) const { return lwb(l) + a * P.mg[l].W; }
  __device__ __forceinline__ float* lv(int l, int a) const {
    return mgws + P.mg[l].voff + (size_t)a * P.mg[l].plen + kSlack;
  }
  __device__ __forceinline__ bool solo(int l) const { return P.cs == 1 || P.mg[l].ny + 1 <= P.mg_solo_rows; }
  __device__ __forceinline__ bool piped(int l) const { return pipe_rows(P.mg[l].W / kGroup, l == 0 ? kElemWeights : kNodeWeights) > 0; }
  // Barrier between passes on levels a and b.  `bulk`: the pass before it wrote a vector that bulk
  // copies read (the fence costs 400 cycles of 512 threads, as much as a pass of a small level).
  __device__ __forceinline__ void xsync(int a, int b, bool bulk = false) {
    if (bulk) asm volatile("fence.proxy.async.global;" ::: "memory");
    if (solo(a) && solo(b))
      __syncthreads();
    else
      comm.sync();
  }
  // this CTA's node rows [y0, y0 + n) of level l
  __device__ __forceinline__ void lrows(int l, int& y0, int& n) const {
    y0 = 0;
    n = 0;
    if (solo(l))
      n = rank == 0 ? P.mg[l].ny + 1 : 0;
    else
      slab_rows(P.mg[l].ny + 1, P.cs, rank, y0, n);
  }
  // f(loc, wloc) for this CTA's groups of 4 nodes of level l: their padded index, and the index of
  // their weights
  template <class F>
  __device__ __forceinline__ void for_lgroups(int l, F f) const {
    int r0l, Rl;
    lrows(l, r0l, Rl);
    const int Wl = P.mg[l].W, G4l = Wl / kGroup;
    for (int t = threadIdx.x; t < Rl * G4l; t += blockDim.x) {
      const int lr = t / G4l, g = t - lr * G4l;
      const int row = r0l + lr + 1;
      f(row * Wl + kGroup * g, 6 * row * Wl + kGroup * g);
    }
  }
  // The node weights of a group's stencil on level l: its own and those of the row below and to the left
  struct GroupWeights {
    float c[4], e[5], n[4], nb[4], ne[4], neb[4], nw[4], nwb[4];
  };
  __device__ __forceinline__ void lweights(int l, int wloc, GroupWeights& w) const {
    const int Wl = P.mg[l].W, wb = wloc - 6 * Wl;       // the row below
    const float *C = lw(l, 0), *E = lw(l, 1), *N = lw(l, 2), *NE = lw(l, 3), *NW = lw(l, 4);
    ld4f(C, wloc, w.c);
    ld4f(N, wloc, w.n);
    ld4f(N, wb, w.nb);
    ld4f(NE, wloc, w.ne);
    ld4f(NW, wloc, w.nw);
    load_ewindow(E, wloc, w.e);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      w.neb[j] = NE[wb - 1 + j];            // NE weights of the row below, shifted left
      w.nwb[j] = NW[wb + 1 + j];            // NW weights of the row below, shifted right
    }
  }
  // y = A_l v on a group from v's windows on the rows below, at and above it (FP32 node weights)
  static __device__ __forceinline__ void lapply(const GroupWeights& w, const float (&vl)[6], const float (&vm)[6],
                                                const float (&vh)[6], float (&y)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float a = w.c[j] * vm[j + 1];
      a = fmaf(w.e[j + 1], vm[j + 2], a);
      a = fmaf(w.e[j], vm[j], a);
      a = fmaf(w.n[j], vh[j + 1], a);
      a = fmaf(w.nb[j], vl[j + 1], a);
      a = fmaf(w.ne[j], vh[j + 2], a);
      a = fmaf(w.neb[j], vl[j], a);
      a = fmaf(w.nw[j], vh[j], a);
      a = fmaf(w.nwb[j], vl[j + 2], a);
      y[j] = a;
    }
  }
  __device__ __forceinline__ void lstencil(int l, int wloc, const float (&vl)[6], const float (&vm)[6],
                                           const float (&vh)[6], float (&y)[4]) const {
    GroupWeights w;
    lweights(l, wloc, w);
    lapply(w, vl, vm, vh, y);
  }
  // windows on the rows below, at and above (rows `stride` floats apart)
  __device__ __forceinline__ void lwindows(const float* __restrict__ v, int loc, int stride, float (&a)[6],
                                           float (&b)[6], float (&c)[6]) const {
    load_window(v, loc - stride, a);
    load_window(v, loc, b);
    load_window(v, loc + stride, c);
  }
  // a large level on the way down: u = S f and res = f - A u row by row, f_{l+1} = P^T res.  The CTA
  // writes the coarse rows J with 2J among its rows, for which it also forms the residual on the
  // row on each side of them; the residual waits in a ring of its own behind the arrays'.
  template <int NW>
  __device__ __forceinline__ void mg_down_march(int l, const float* __restrict__ f) {
    int y0, n;
    lrows(l, y0, n);
    const int ny = P.mg[l].ny, Wl = P.mg[l].W, G4l = Wl / kGroup, Wc = P.mg[l + 1].W, G4c = Wc / kGroup;
    const int nxc = P.mg[l + 1].nx;
    if (n > 0) {
      const int ya = max(y0 - 1, 0), yb = min(y0 + n, ny), SR = res_rows(G4l);
      float* res = ring_sm + (1 + NW) * pipe_rows(G4l, NW) * Wl;
      const float* wdc = lw(l + 1, 5);
      float* fc = lv(l + 1, 0);
      int J = (y0 + 1) / 2;
      const int Jend = (y0 + n + 1) / 2;           // coarse rows J .. Jend - 1
      march<NW>(l, f, ya, yb,
               [&](const RowRef<NW>& rr, int y, int g, bool ok) {
                 float vl[6], vm[6], vh[6], dw[6], t[4], fc4[4], o[4];
                 rwin(rr.v(rr.so), g, G4l, vl);
                 rwin(rr.wd(rr.so), g, G4l, dw);
#pragma unroll
                 for (int i = 0; i < 6; ++i) vl[i] *= dw[i];
                 rwin(rr.v(rr.su), g, G4l, vh);
                 rwin(rr.wd(rr.su), g, G4l, dw);
#pragma unroll
                 for (int i = 0; i < 6; ++i) vh[i] *= dw[i];
                 rwin(rr.v(rr.sm), g, G4l, vm);
                 rwin(rr.wd(rr.sm), g, G4l, dw);
#pragma unroll
                 for (int j = 0; j < 4; ++j) fc4[j] = vm[j + 1];
#pragma unroll
                 for (int i = 0; i < 6; ++i) vm[i] *= dw[i];
                 rstencil(rr, g, G4l, vl, vm, vh, t);
#pragma unroll
                 for (int j = 0; j < 4; ++j) o[j] = dw[j + 1] != 0.f ? fc4[j] - t[j] : 0.f;
                 if (ok) st4f(res, ((y - ya) % SR) * Wl + kGroup * g, o);
               },
               [&](int ydone) {
                 // coarse rows whose fine rows 2J-1 .. 2J+1 are all there
                 const int Jn = ydone > yb ? Jend : max(J, min(Jend, ydone / 2));
                 for (int t = threadIdx.x; t < (Jn - J) * G4c; t += kStreamThreads) {
                   const int jr = t / G4c, gc = t - jr * G4c, Jc = J + jr, I0 = kGroup * gc - 1;
                   float dv[4], o[4] = {0.f, 0.f, 0.f, 0.f};
                   const int loc = (Jc + 1) * Wc + kGroup * gc;
                   ld4f(wdc, 6 * (Jc + 1) * Wc + kGroup * gc, dv);
#pragma unroll
                   for (int b = -1; b <= 1; ++b) {
                     const int y = 2 * Jc + b;
                     if (y < 0 || y > ny) continue;
                     // entries 8 gc - 4 .. 8 gc + 7 of the row: column 2 I of node j is entry 3 + 2 j
                     const float* row = res + ((y - ya) % SR) * Wl + 2 * kGroup * gc - 4;
                     // (those outside the row belong to pads of the coarse row)
                     const int at = 2 * kGroup * gc;
                     float4 ca = make_float4(0.f, 0.f, 0.f, 0.f), cb = ca, cc = ca;
                     if (gc > 0) ca = *reinterpret_cast<const float4*>(row);
                     if (at < Wl) cb = *reinterpret_cast<const float4*>(row + 4);
                     if (at + 4 < Wl) cc = *reinterpret_cast<const float4*>(row + 8);
                     const float hb = b == 0 ? 1.f : 0.5f;
                     o[0] = fmaf(hb, fmaf(0.5f, ca.z + cb.x, ca.w), o[0]);
                     o[1] = fmaf(hb, fmaf(0.5f, cb.x + cb.z, cb.y), o[1]);
                     o[2] = fmaf(hb, fmaf(0.5f, cb.z + cc.x, cb.w), o[2]);
                     o[3] = fmaf(hb, fmaf(0.5f, cc.x + cc.z, cc.y), o[3]);
                   }
#pragma unroll
                   for (int j = 0; j < 4; ++j)
                     if (dv[j] == 0.f || I0 + j < 0 || I0 + j > nxc) o[j] = 0.f;
                   st4f(fc, loc, o);
                 }
                 J = Jn;
               });
    }
  }
  // a large level on the way up: u' = S f + P e_{l+1}, out = u' + S (f - A u'); level 0 writes z and
  // returns the local (r, z)
  template <int NW>
  __device__ __forceinline__ V mg_up_march(int l, const float* __restrict__ f) {
    int y0, n;
    lrows(l, y0, n);
    V rz = V{};
    if (n == 0) return rz;
    const int Wl = P.mg[l].W, G4l = Wl / kGroup, Wc = P.mg[l + 1].W;
    const float* ec = lv(l + 1, 3);
    float* out = l == 0 ? z : lv(l, 3);
    march<NW>(l, f, y0, y0 + n - 1,
             [&](const RowRef<NW>& rr, int y, int g, bool ok) {
               // coarse rows A, B, C: row y-1 takes A and B (y even) or A, row y B or A and B, row
               // y+1 B and C or B; columns 2g-1 .. 2g+2
               const bool even = (y & 1) == 0;
               const int c0 = 2 * g;
               const float* eA = ec + (((y - 1) >> 1) + 1) * Wc + c0;
               const float* eB = ec + (((y + 1) >> 1) + 1) * Wc + c0;
               const float* eC = ec + (((y + 2) >> 1) + 1) * Wc + c0;
               float pa[4], pb[4], pc[4];
               auto ld = [](const float* q_, float (&v)[4]) {
                 const float2 a = *reinterpret_cast<const float2*>(q_), b = *reinterpret_cast<const float2*>(q_ + 2);
                 v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
               };
               ld(eA, pa);
               ld(eB, pb);
               ld(eC, pc);
               const int loc = (y + 1) * Wl + kGroup * g;
               V rv[4];
               if (l == 0) ldv(r, loc, rv);
               float vl[6], vm[6], vh[6], dw[6], t[4], fc4[4], o[4];
               // the row's window of P e: even window columns on coarse columns, odd ones between
               auto add = [&](float (&v)[6], const float (&c)[4]) {
#pragma unroll
                 for (int i = 0; i < 6; ++i) {
                   const float pe = i & 1 ? 0.5f * (c[i >> 1] + c[(i >> 1) + 1]) : c[i >> 1];
                   v[i] = dw[i] != 0.f ? fmaf(v[i], dw[i], pe) : 0.f;
                 }
               };
               float m[4];
#pragma unroll
               for (int i = 0; i < 4; ++i) m[i] = 0.5f * (pa[i] + pb[i]);
               rwin(rr.v(rr.so), g, G4l, vl);
               rwin(rr.wd(rr.so), g, G4l, dw);
               float c_[4];
#pragma unroll
               for (int i = 0; i < 4; ++i) c_[i] = even ? m[i] : pa[i];
               add(vl, c_);
               rwin(rr.v(rr.su), g, G4l, vh);
               rwin(rr.wd(rr.su), g, G4l, dw);
#pragma unroll
               for (int i = 0; i < 4; ++i) c_[i] = even ? 0.5f * (pb[i] + pc[i]) : pb[i];
               add(vh, c_);
               rwin(rr.v(rr.sm), g, G4l, vm);
               rwin(rr.wd(rr.sm), g, G4l, dw);
#pragma unroll
               for (int j = 0; j < 4; ++j) fc4[j] = vm[j + 1];
#pragma unroll
               for (int i = 0; i < 4; ++i) c_[i] = even ? pb[i] : m[i];
               add(vm, c_);
               rstencil(rr, g, G4l, vl, vm, vh, t);
#pragma unroll
               for (int j = 0; j < 4; ++j) o[j] = fmaf(dw[j + 1], fc4[j] - t[j], vm[j + 1]);
               if (!ok) return;
               if (l == 0) {
#pragma unroll
                 for (int j = 0; j < 4; ++j) rz = vdot(rz, rv[j], o[j]);
               }
               st4f(out, loc, o);
             },
             [](int) {});
    return rz;
  }
  // a small level on the way down: u = S f and res = f - A u (u of the neighbours from their f)
  __device__ __forceinline__ void mg_pre(int l, const float* __restrict__ f) {
    const int Wl = P.mg[l].W;
    const float* wd = lw(l, 5);
    float* u = lv(l, l == 0 ? 0 : 1);
    float* res = lv(l, l == 0 ? 1 : 2);
    for_lgroups(l, [&](int loc, int wloc) {
      float fl[6], fm[6], fh[6], dl[6], dm[6], dh[6], y[4], uo[4], ro[4], fc[4];
      lwindows(f, loc, Wl, fl, fm, fh);
      lwindows(wd, wloc, 6 * Wl, dl, dm, dh);
#pragma unroll
      for (int j = 0; j < 4; ++j) fc[j] = fm[j + 1];
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        fl[i] *= dl[i];
        fm[i] *= dm[i];
        fh[i] *= dh[i];
      }
      lstencil(l, wloc, fl, fm, fh, y);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        ro[j] = dm[j + 1] != 0.f ? fc[j] - y[j] : 0.f;
        uo[j] = fm[j + 1];
      }
      st4f(u, loc, uo);
      st4f(res, loc, ro);
    });
  }
  // f_{l+1} = P^T res_l on the nodes of level l+1 (0 off its unknowns)
  __device__ __forceinline__ void mg_restrict(int l) {
    const int c = l + 1, Wf = P.mg[l].W, nxc = P.mg[c].nx;
    const float* res = lv(l, l == 0 ? 1 : 2);
    const float* wdc = lw(c, 5);
    float* fc = lv(c, 0);
    const int Wc = P.mg[c].W;
    for_lgroups(c, [&](int loc, int wloc) {
      const int J = loc / Wc - 1, I0 = loc - (J + 1) * Wc - 1;
      float dv[4], o[4];
      ld4f(wdc, wloc, dv);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int I = I0 + j;
        float acc = 0.f;
        if (dv[j] != 0.f && I >= 0 && I <= nxc) {
          const float* r0 = res + (2 * J + 1) * Wf + 2 * I + 1;   // fine node (2I, 2J)
#pragma unroll
          for (int b = -1; b <= 1; ++b) {
            const float* rr = r0 + b * Wf;
            const float row = fmaf(0.5f, rr[-1] + rr[1], rr[0]);
            acc = fmaf(b == 0 ? 1.f : 0.5f, row, acc);
          }
        }
        o[j] = acc;
      }
      st4f(fc, loc, o);
    });
  }
  // coarsest level: e = mg_coarse_steps damped-Jacobi steps from zero, the last into e.  A level of at
  // most 32 groups on one CTA (9 x 9 nodes: 27) is one warp's: the iterate and the weights stay in
  // registers, the neighbours' values come by shuffles, and a step has no barrier.
  __device__ __forceinline__ void mg_coarsest(int l) {
    const int Wl = P.mg[l].W, n = P.mg_coarse_steps;
    const float* f = lv(l, 0);
    const float* wd = lw(l, 5);
    const int G4l = Wl / kGroup, cnt = (P.mg[l].ny + 1) * G4l;
    if (solo(l) && cnt <= 32) {
      if (rank == 0 && threadIdx.x < 32) {
        const int lane = threadIdx.x, t = min(lane, cnt - 1), lr = t / G4l, g = t - lr * G4l;
        const int loc = (lr + 1) * Wl + kGroup * g, wloc = 6 * (lr + 1) * Wl + kGroup * g;
        GroupWeights w;
        lweights(l, wloc, w);
        float fv[4], dv[4], v[4];
        ld4f(f, loc, fv);
        ld4f(wd, wloc, dv);
        // lanes beyond the level and rows beyond it hold 0; a row's first and last entries are zero
        // pads, so the window's ends may come from the lane of another row
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (lane >= cnt) dv[j] = fv[j] = 0.f;
          v[j] = dv[j] * fv[j];
        }
        const bool below = lane >= G4l, above = lane + G4l < cnt;
        auto from = [&](float x, int src) { return __shfl_sync(0xffffffffu, x, src & 31); };
        for (int k = 2; k <= n; ++k) {
          float vl[6], vm[6], vh[6], y[4];
          vm[0] = from(v[3], lane - 1);
          vm[5] = from(v[0], lane + 1);
          vl[0] = from(v[3], lane - G4l - 1);
          vl[5] = from(v[0], lane - G4l + 1);
          vh[0] = from(v[3], lane + G4l - 1);
          vh[5] = from(v[0], lane + G4l + 1);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            vm[j + 1] = v[j];
            vl[j + 1] = from(v[j], lane - G4l);
            vh[j + 1] = from(v[j], lane + G4l);
          }
#pragma unroll
          for (int i = 0; i < 6; ++i) {
            vl[i] = below ? vl[i] : 0.f;
            vh[i] = above ? vh[i] : 0.f;
          }
          lapply(w, vl, vm, vh, y);
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = fmaf(dv[j], fv[j] - y[j], v[j]);
        }
        if (lane < cnt) st4f(lv(l, 3), loc, v);
      }
      xsync(l, l);
      return;
    }
    float* bufs[2] = {lv(l, 3), lv(l, 1)};   // step k writes bufs[(n - k) % 2]: the last lands in e
    for (int k = 1; k <= n; ++k) {
      float* dst = bufs[(n - k) & 1];
      const float* src = bufs[(n - k + 1) & 1];
      for_lgroups(l, [&](int loc, int wloc) {
        float fv[4], dv[4], o[4];
        ld4f(f, loc, fv);
        ld4f(wd, wloc, dv);
        if (k == 1) {
#pragma unroll
          for (int j = 0; j < 4; ++j) o[j] = dv[j] * fv[j];
        } else {
          float vl[6], vm[6], vh[6], y[4];
          lwindows(src, loc, Wl, vl, vm, vh);
          lstencil(l, wloc, vl, vm, vh, y);
#pragma unroll
          for (int j = 0; j < 4; ++j) o[j] = fmaf(dv[j], fv[j] - y[j], vm[j + 1]);
        }
        st4f(dst, loc, o);
      });
      xsync(l, l);
    }
  }
  // a small level on the way up: the prolongation and the post-smoothing step in one pass, with
  // u' = u + P e_{l+1} formed on the window from u and the coarse e
  __device__ __forceinline__ V mg_up(int l, const float* __restrict__ f) {
    const int c = l + 1, Wl = P.mg[l].W, Wc = P.mg[c].W;
    const float* ec = lv(c, 3);
    const float* wd = lw(l, 5);
    const float* u = lv(l, l == 0 ? 0 : 1);
    V rz = V{};
    for_lgroups(l, [&](int loc, int wloc) {
      const int y = loc / Wl - 1, x0 = loc - (y + 1) * Wl - 1;   // first node of the group
      // x0 = 4g - 1 is odd, so window column i (node x0 - 1 + i) lies between coarse columns
      // cx0 + i/2 and cx0 + (i+1)/2 (equal for even i)
      const int cx0 = (x0 - 1) >> 1;
      float win[3][6];
#pragma unroll
      for (int r_ = 0; r_ < 3; ++r_) {
        const int row = loc + (r_ - 1) * Wl;
        float v[6], d_[6];
        load_window(u, row, v);
        load_window(wd, wloc + (r_ - 1) * 6 * Wl, d_);
        const int yy = y - 1 + r_, Ja = yy >> 1, Jb = (yy + 1) >> 1;
        const float* ra = ec + (Ja + 1) * Wc + 1 + cx0;
        const float* rb = ec + (Jb + 1) * Wc + 1 + cx0;
        float cc[4];
#pragma unroll
        for (int q_ = 0; q_ < 4; ++q_) cc[q_] = 0.5f * (ra[q_] + rb[q_]);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          const float pv = i & 1 ? 0.5f * (cc[i >> 1] + cc[(i >> 1) + 1]) : cc[i >> 1];
          win[r_][i] = d_[i] != 0.f ? v[i] + pv : v[i];
        }
      }
      float t[4], dv[4], fv[4], o[4];
      lstencil(l, wloc, win[0], win[1], win[2], t);
      ld4f(wd, wloc, dv);
      ld4f(f, loc, fv);
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = fmaf(dv[j], fv[j] - t[j], win[1][j + 1]);
      if (l == 0) {
        V rv[4];
        ldv(r, loc, rv);
#pragma unroll
        for (int j = 0; j < 4; ++j) rz = vdot(rz, rv[j], o[j]);
        st4f(z, loc, o);
      } else {
        st4f(lv(l, 3), loc, o);
      }
    });
    return rz;
  }

  // z = M^-1 r from r (every row of r visible); returns the local (r, z).  z is visible to the
  // group after the next group barrier.
  __device__ __forceinline__ V vcycle() {
    const int L = P.mg_levels;
    for (int l = 0; l < L - 1; ++l) {
      const float* f = l == 0 ? r : lv(l, 0);
      if (piped(l)) {
        if (l == 0)
          mg_down_march<kElemWeights>(0, f);
        else
          mg_down_march<kNodeWeights>(l, f);
        xsync(l, l + 1, piped(l + 1));
      } else {
        mg_pre(l, f);
        xsync(l, l + 1);
        mg_restrict(l);
        xsync(l + 1, l + 1, piped(l + 1));
      }
    }
    mg_coarsest(L - 1);                 // ends with a barrier
    V rz = V{};
    for (int l = L - 2; l >= 0; --l) {
      if (l < L - 2) xsync(l + 1, l);   // e_{l+1} of the level above is visible
      else if (!(solo(l + 1) && solo(l))) comm.sync();
      const float* f = l == 0 ? r : lv(l, 0);
      if (l == 0)
        rz = piped(0) ? mg_up_march<kElemWeights>(0, f) : mg_up(0, f);
      else if (piped(l))
        mg_up_march<kNodeWeights>(l, f);
      else
        mg_up(l, f);
    }
    return rz;
  }

  // res = b - A x (FP64, 0 off the unknowns); the local (b, b) and (r, r)
  __device__ __forceinline__ void residual(const double* __restrict__ x, double& bb, double& rr) const {
    bb = 0.0;
    rr = 0.0;
    for_groups([&](int loc, int, int) {
      double y[4], bv[4];
      float di[4];
      stencil_node64<double>(x, loc, A64, loc, P.W, y);
      load4(b + loc, bv);
      dinv4(loc, di);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        bb = fma(bv[j], bv[j], bb);
        bv[j] = di[j] != 0.f ? bv[j] - y[j] : 0.0;
        rr = fma(bv[j], bv[j], rr);
      }
      st4d(res, loc, bv);
    });
  }
  // the local sum of (diag(A) x)^2 (kRounding2); x is 0 off the unknowns
  __device__ __forceinline__ double diag_x2(const double* __restrict__ x) const {
    double s = 0.0;
    for_groups([&](int loc, int, int) {
      double xv[4], cv[4];
      load4(x + loc, xv);
      load4(A64.C + loc, cv);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const double t = cv[j] * xv[j];
        s = fma(t, t, s);
      }
    });
    return s;
  }
  // After a CG: x += unscale d
  __device__ __forceinline__ void update(double* __restrict__ x, double unscale) const {
    for_groups([&](int loc, int, int) {
      V dv[4];
      double xv[4];
      ldv(d, loc, dv);
      load4(x + loc, xv);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if constexpr (!kMixed) xv[j] = fma(widen(dv[j].l), unscale, xv[j]);
        xv[j] = fma(widen(f32(dv[j])), unscale, xv[j]);
      }
      st4d(x, loc, xv);
    });
  }
  // The same in an FP32 kind, with the residual following: res <- res - unscale A d, A d summed in
  // float pairs.  Cheaper than a new residual (3 FP64 instructions per node instead of 11), but
  // without the rounding of x and with the pairs' 48 bits: good enough for the next CG to work on, never to
  // end a solve.  Returns the local (r, r).
  __device__ __forceinline__ double update_residual(double* __restrict__ x, double unscale) const {
    const double us = -unscale / ffw.scale;
    double rr = 0.0;
    for_groups([&](int loc, int, int) {
      ff y[4];
      stencil_ff(d, loc, ffw, loc, P.W, y);
      float dv[4], di[4];
      double xv[4], rv[4];
      ld4f(d, loc, dv);
      load4(x + loc, xv);
      load4(res + loc, rv);
      dinv4(loc, di);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        xv[j] = fma(widen(dv[j]), unscale, xv[j]);
        rv[j] = di[j] != 0.f ? fma(widen(y[j].l), us, fma(widen(y[j].h), us, rv[j])) : 0.0;
        rr = fma(rv[j], rv[j], rr);
      }
      st4d(x, loc, xv);
      st4d(res, loc, rv);
    });
    return rr;
  }

  // q = A z + beta q, p = z + beta p on the own rows (q = A z, p = z at the start); the local (p, q)
  __device__ __forceinline__ V direction(bool start, const V& beta) {
    V pq = V{};
    auto update = [&](int loc, const V (&w)[4], const float (&zv)[4], const float (&di)[4]) {
      V qv[4] = {V{}, V{}, V{}, V{}}, pv[4] = {V{}, V{}, V{}, V{}};
      if (!start) {
        ldv(q, loc, qv);
        ldv(p, loc, pv);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        qv[j] = di[j] != 0.f ? vfma(beta, qv[j], w[j]) : V{};
        pv[j] = vfma(beta, pv[j], zv[j]);
        pq = vdot(pq, pv[j], qv[j]);
      }
      stv(q, loc, qv);
      stv(p, loc, pv);
    };
    if constexpr (kMixed) {
      if (P.mg_levels > 0 && piped(0)) {
        const int W = P.W;
        constexpr int NW = kElemWeights;
        march<NW>(0, z, r0, r0 + R - 1,
                 [&](const RowRef<NW>& rr, int y, int g, bool ok) {
                   float vl[6], vm[6], vh[6], w[4], zv[4], di[4];
                   rwin(rr.v(rr.so), g, G4, vl);
                   rwin(rr.v(rr.sm), g, G4, vm);
                   rwin(rr.v(rr.su), g, G4, vh);
                   rstencil(rr, g, G4, vl, vm, vh, w);
                   ld4f(rr.wd(rr.sm), kGroup * g, di);
#pragma unroll
                   for (int j = 0; j < 4; ++j) zv[j] = vm[j + 1];
                   if (ok) update((y + 1) * W + kGroup * g, w, zv, di);
                 },
                 [](int) {});
        return pq;
      }
    }
    for_groups([&](int loc, int iy, int g) {
      V w[4];
      float zv[4], di[4];
      if constexpr (!kMixed) {
        stencil_ff(z, loc, ffw, loc, P.W, w);
      } else if (P.mg_levels > 0) {
        float zl[6], zm[6], zh[6];
        lwindows(z, loc, P.W, zl, zm, zh);
        lstencil(0, 6 * (iy + 1) * P.W + kGroup * g, zl, zm, zh, w);
      } else {
        stencil_elem32(z, P.w32, P.w32 + P.w32_stride, P.w32 + 2 * P.w32_stride, loc, P.W, w);
      }
      ld4f(z, loc, zv);
      dinv4(loc, di);
      update(loc, w, zv, di);
    });
    return pq;
  }

  // z = D^-1 r on a group; acc + (r, z)
  __device__ __forceinline__ V jacobi(int loc, const V (&rv)[4], V acc) const {
    float di[4], zv[4];
    dinv4(loc, di);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      zv[j] = di[j] * f32(rv[j]);
      acc = vdot(acc, rv[j], zv[j]);
    }
    st4f(z, loc, zv);
    return acc;
  }

  // Solve (C/dt + K) x = b from the start in x (every row of x readable).  What decides is b - A x in FP64.
  // After a CG that was to reach the tolerance it is evaluated; after one that was to reach inner_rtol
  // alone the residual may follow x (update_residual), and it is evaluated before it ends the solve.  A
  // solve that rounding keeps above rtol ends too (kRounding2).
  __device__ __forceinline__ void solve(double* __restrict__ x, int step) {
    double v2[2];
    residual(x, v2[0], v2[1]);
    allreduce<double, 2>(v2);
    const double bb = v2[0];
    double rr = v2[1];
    const double tol2 = P.rtol * P.rtol * bb;
    const bool mg = P.mg_levels > 0;
    int sweeps = 0, its = 0;
    bool rounded = false;
    while (rr > tol2 && !rounded && sweeps < P.refmax) {
      // r / 2^k of squared norm in [1, 4)
      const int k2 = (((__double2hiint(rr) >> 20) & 0x7ff) - 1023) >> 1;
      const double rr0 = rr * exp2_int(-k2) * exp2_int(-k2);
      const double inner2 = P.inner_rtol * P.inner_rtol, final2 = 0.25 * tol2 / rr;
      const float target2 = fmaxf((float)(fmax(inner2, final2) * rr0), 1e-30f);
      V rz = V{}, beta = V{};
      int it = -1;                     // -1: the start, whose z and (r, z) open the iteration
      bool done = !((float)rr0 > target2);
      const bool none = done;
      for (;;) {
        V v[3] = {V{}, V{}, V{}};
        const bool start = it < 0;
        if (start) {
          for_groups([&](int loc, int, int) {
            double bv[4];
            V rv[4];
            load4(res + loc, bv);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const ff s = split_scaled(bv[j], -k2);
              if constexpr (kMixed)
                rv[j] = s.h + s.l;
              else
                rv[j] = s;
            }
            stv(r, loc, rv);
            if (!mg) v[0] = jacobi(loc, rv, v[0]);
          });
        } else {
          // alpha = rz / (p, q)
          V pq[1] = {direction(it == 0, beta)};
          const V rz_c = rz;
          comm.template allreduce<V, 1, 0>(pq, P.cs, [rz_c](V* t) { t[0] = vdiv(rz_c, t[0]); });   // p, q: no bulk copies
          const V alpha = pq[0], nalpha = vneg(alpha);
          // d += alpha p (d = alpha p at first), r -= alpha q; (r, r)
          const bool first = it == 0;
          for_group_pairs([&](const int (&loc)[2], const bool (&ok)[2]) {
            V dv[2][4], pv[2][4], rv[2][4], qv[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              if (!ok[u]) continue;
#pragma unroll
              for (int j = 0; j < 4; ++j) dv[u][j] = V{};
              if (!first) ldv(d, loc[u], dv[u]);
              ldv(p, loc[u], pv[u]);
              ldv(r, loc[u], rv[u]);
              ldv(q, loc[u], qv[u]);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              if (!ok[u]) continue;
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                dv[u][j] = vfma(alpha, pv[u][j], dv[u][j]);
                rv[u][j] = vfma(nalpha, qv[u][j], rv[u][j]);
                v[1] = vdot(v[1], rv[u][j], rv[u][j]);
              }
              stv(d, loc[u], dv[u]);
              stv(r, loc[u], rv[u]);
              if (!mg) v[0] = jacobi(loc[u], rv[u], v[0]);
            }
          });
        }
        // z = M^-1 r; (r, z), (r, r), beta = (r, z)_new / (r, z)
        if (mg) {
          sync();
          v[0] = vcycle();
        }
        const V rz_c = rz;
        allreduce<V, 2, 1>(v, [rz_c, start](V* t) { if (!start) t[2] = vdiv(t[0], rz_c); });
        ++it;
        if (!start && !(f32(v[1]) > target2)) done = true;   // a NaN ends it too
        beta = v[2];
        rz = v[0];
        if (done || it >= P.itmax) break;
      }
      its += it;
      ++sweeps;
      if (none) break;                             // no iteration: there is no d
      const double unscale = exp2_int(k2) * ffw.scale;
      bool follow = kMixed && inner2 > final2;
      double w1[1];
      if constexpr (kMixed) {
        if (follow) {
          w1[0] = update_residual(x, unscale);
          allreduce<double, 1>(w1);
          rr = w1[0];
          follow = rr > tol2;
        } else {
          update(x, unscale);
          comm.sync();
        }
      } else {
        update(x, unscale);
        comm.sync();
      }
      if (!follow) {
        const double before = rr;
        residual(x, v2[0], w1[0]);
        allreduce<double, 1>(w1);
        rr = w1[0];
        // a CG that aimed at the tolerance, or gained little: whether rounding is what is left
        if (rr > tol2 && (inner2 <= final2 || rr > 0.01 * before)) {
          double u[1] = {diag_x2(x)};
          allreduce<double, 1>(u);
          rounded = rr <= kRounding2 * u[0];
        }
      }
    }
    if (threadIdx.x == 0 && rank == 0) {
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

  __device__ __forceinline__ double* hist_row(int j) const {
    const int rr = j - P.hist_j0;
    if (P.hist == nullptr || rr < 0 || rr >= P.hist_rows) return nullptr;
    return P.hist + (size_t)rr * P.Nn;
  }

  __device__ __forceinline__ double accumulate_theta(double theta, double inc) const {
    return P.objective == PTG_OBJ_MODIFIED ? theta + inc : pow(ipow(theta, P.p_int) + inc, 1.0 / P.p);
  }
  __device__ __forceinline__ double adjoint_scale(double Theta) const {
    return (P.objective == PTG_OBJ_MODIFIED ? P.p : pow(Theta, 1.0 - P.p)) / (double)P.Ne;
  }

  // (C/dt) x on a group: without weights where the capacity is uniform (see Stepper::mass_dt)
  __device__ __forceinline__ void mass_dt(const double* __restrict__ x, int loc, int iy, int g, double (&y)[4]) const {
    if (P.has_dc) {
      stencil_node64<double>(x, loc, P.mass, loc, P.W, y);
#pragma unroll
      for (int j = 0; j < 4; ++j) y[j] *= inv_dt;
      return;
    }
    const double dy = iy == 0 || iy == P.ny ? 2.0 : 4.0, s = P.mass_uniform * inv_dt;
    double xl[6], xm[6], xh[6];
    load_window(x, loc - P.W, xl);
    load_window(x, loc, xm);
    load_window(x, loc + P.W, xh);
#pragma unroll
    for (int i = 0; i < 6; ++i) xm[i] = fma(dy, xm[i], xl[i] + xh[i]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int ix = kGroup * g - 1 + j;
      const double dx = ix == 0 || ix == P.nx ? 2.0 : 4.0;
      y[j] = s * fma(dx, xm[j + 1], xm[j] + xm[j + 2]);
    }
  }

  // b = (C/dt) xp + src(node) on the own rows; xn = the start of the step: the extrapolation
  // through xp and the ring rows X[0..n-2] (n = 1: xp itself); the ring row wr receives xp.
  // The ring rows are padded node rows 0 .. ny; pads and Dirichlet nodes are zero in every state.
  template <class Src>
  __device__ __forceinline__ void begin_step(const double* __restrict__ xp, double* __restrict__ xn, int n, const double* const* X,
                             double* __restrict__ wr, Src src) {
    for_groups([&](int loc, int iy, int g) {
      double y[4], x1[4], bv[4], xv[4], a[4], b_[4], c[4];
      const int o = loc - P.W;
      load4(xp + loc, x1);
      if (n >= 2) load4(X[0] + o, a);
      if (n >= 3) load4(X[1] + o, b_);
      if (n >= 4) load4(X[2] + o, c);
      mass_dt(xp, loc, iy, g, y);
      if (wr) st4d(wr, o, x1);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        bv[j] = gi < 0 || P.dirichlet[gi] ? 0.0 : y[j] + src(gi);
        if (n <= 1)
          xv[j] = x1[j];
        else if (n == 2)
          xv[j] = fma(2.0, x1[j], -a[j]);
        else if (n == 3)
          xv[j] = fma(3.0, x1[j] - a[j], b_[j]);
        else
          xv[j] = fma(4.0, x1[j] + b_[j], -fma(6.0, a[j], c[j]));
      }
      st4d(b, loc, bv);
      st4d(xn, loc, xv);
    });
    comm.sync();
  }

  // a node vector ([Nn]) into the own rows of a padded vector (0 off the unknowns), and back
  __device__ void load(const double* __restrict__ src, double* __restrict__ dst) const {
    for_groups([&](int loc, int iy, int g) {
      double v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        v[j] = (gi >= 0 && !P.dirichlet[gi]) ? src[gi] : 0.0;
      }
      st4d(dst, loc, v);
    });
  }
  __device__ void store(const double* __restrict__ src, double* __restrict__ dst) const {
    if (!dst) return;
    for_groups([&](int loc, int iy, int g) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        if (gi >= 0) dst[gi] = src[loc + j];
      }
    });
  }

  // sum of x^p over the nodes; x is stored to the node vector dst (if given) in the same pass
  __device__ __forceinline__ double pnorm_store(const double* __restrict__ x, double* __restrict__ dst) {
    double v[1] = {0.0};
    for_groups([&](int loc, int iy, int g) {
      double xv[4];
      load4(x + loc, xv);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        if (gi < 0) continue;
        v[0] += ipow(xv[j], P.p_int);   // 0 on Dirichlet nodes
        if (dst) dst[gi] = xv[j];
      }
    });
    allreduce<double, 1>(v);
    return v[0];
  }

  // Eq. 4.7 element sums of the own element rows (rows r0 .. r0 + R - 1 below ny); lam padded,
  // Tj and Tjm node vectors
  // (the gsrc row is 0 if null; addF - subG is added if given)
  __device__ __forceinline__ void accumulate_g(const double* __restrict__ lam, const double* __restrict__ Tj,
                               const double* __restrict__ Tjm, const double* __restrict__ gsrc,
                               double* __restrict__ gdst, double nnorm, const double* __restrict__ addF = nullptr,
                               const double* __restrict__ subG = nullptr) const {
    const int nx = P.nx, Wp = P.W;
    const int er = min(R, P.ny - r0);
    const int nel = er > 0 ? er * nx : 0;
    const double mass_scale = P.h * P.h / step_dt, inv_norm = 1.0 / nnorm;
    for (int t = threadIdx.x; t < nel; t += blockDim.x) {
      const int ler = t / nx, ex = t - ler * nx;
      const int ey = r0 + ler;
      const int e = ey * nx + ex;
      const int g0 = ey * nn + ex;
      const int l0 = (ey + 1) * Wp + ex + 1;
      const Modes l = elem_modes(lam[l0], lam[l0 + 1], lam[l0 + Wp + 1], lam[l0 + Wp]);
      const double tsw = Tj[g0], tse = Tj[g0 + 1], tne = Tj[g0 + nn + 1], tnw = Tj[g0 + nn];
      double term = P.dk[e] * elem_stiffness(l, elem_modes(tsw, tse, tne, tnw));
      if (P.has_dc)
        term = fma(P.dc[e] * mass_scale,
                   elem_mass(l, elem_modes(tsw - Tjm[g0], tse - Tjm[g0 + 1], tne - Tjm[g0 + nn + 1], tnw - Tjm[g0 + nn])),
                   term);
      double gv = fma(-inv_norm, term, gsrc ? gsrc[e] : 0.0);
      if (addF) gv += addF[e] - subG[e];
      gdst[e] = gv;
    }
  }

  // b = (C/dt) xp + src(node) on the own rows (xp padded, every row visible), 0 off the unknowns
  template <class Src>
  __device__ __forceinline__ void build_rhs(const double* __restrict__ xp, Src src) {
    for_groups([&](int loc, int iy, int g) {
      double y[4], bv[4];
      mass_dt(xp, loc, iy, g, y);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        bv[j] = (gi < 0 || P.dirichlet[gi]) ? 0.0 : y[j] + src(gi);
      }
      st4d(b, loc, bv);
    });
  }
  // x = Gs + inc on the own rows, 0 off the unknowns: the start G(u^old) plus the polynomial
  // extrapolation of the last m (1..3) increments of the correction sweep (as the stepper's
  // load_x64_increment): d_i = X_i - Fm[i], X_0 = xc (padded, the state the step propagates),
  // X_1, X_2 node vectors of earlier corrected states; inc = d0, 2 d0 - d1 or 3 (d0 - d1) + d2
  __device__ __forceinline__ void load_increment(const double* __restrict__ Gs, int m, const double* const* Fm,
                                 const double* const* X, const double* __restrict__ xc,
                                 double* __restrict__ x) const {
    for_groups([&](int loc, int iy, int g) {
      double v[4], c[4];
      load4(xc + loc, c);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        if (gi < 0 || P.dirichlet[gi]) {
          v[j] = 0.0;
          continue;
        }
        const double d0 = c[j] - Fm[0][gi];
        double inc = d0;
        if (m == 2) inc = fma(2.0, d0, -(X[1][gi] - Fm[1][gi]));
        if (m == 3) inc = fma(3.0, d0 - (X[1][gi] - Fm[1][gi]), X[2][gi] - Fm[2][gi]);
        v[j] = Gs[gi] + inc;
      }
      st4d(x, loc, v);
    });
  }
  // Parareal correction (Eq. 4.9 / 4.14): x = xs + Fs - Gs on the own rows into the padded x and
  // the node vectors X (and Y if given); 0 off the unknowns
  __device__ __forceinline__ void correction(const double* __restrict__ xs, const double* __restrict__ Fs,
                             const double* __restrict__ Gs, double* __restrict__ x, double* __restrict__ X,
                             double* __restrict__ Y) const {
    for_groups([&](int loc, int iy, int g) {
      double v[4], c[4];
      load4(xs + loc, c);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        v[j] = (gi >= 0 && !P.dirichlet[gi]) ? (c[j] + Fs[gi]) - Gs[gi] : 0.0;
        if (gi >= 0) {
          X[gi] = v[j];
          if (Y) Y[gi] = v[j];
        }
      }
      st4d(x, loc, v);
    });
  }
  __device__ void zero_padded(double* __restrict__ x) const {
    for_groups([&](int loc, int, int) {
      const double zero[4] = {0.0, 0.0, 0.0, 0.0};
      st4d(x, loc, zero);
    });
  }

  // ------------------------------------------------------------------ task bodies
  __device__ __forceinline__ void fine_primal(int task) {
    const int s = P.s0 + task;
    const int M = P.M;
    const double inv_norm = 1.0 / ((double)P.Nt * (double)P.Ne);
    double* x_prev = xa;
    double* x_cur = xb;
    load(P.in_field + (size_t)s * P.Nn, x_prev);
    comm.sync();
    const bool power = P.objective != PTG_OBJ_MODIFIED;   // (see the stepper: one root per slice)
    double theta = power ? ipow(P.in_aux[s], P.p_int) : P.in_aux[s];
    const int nring = P.extrap;
    double* ring = nring > 1 && P.prev_field ? P.prev_field + (size_t)task * nring * P.ring_stride : nullptr;
    int saved = 0;
    for (int j = M * s + 1; j <= M * (s + 1); ++j) {
      const double qj = P.q_time[j];
      const double* X[kMaxExtrap - 1];
      int n = 1;
      double* wr = nullptr;
      if (ring) {
        n = min(saved + 1, nring);
        for (int i = 2; i <= n; ++i) X[i - 2] = ring + (size_t)((j - i) % nring) * P.ring_stride;
        wr = ring + (size_t)((j - 1) % nring) * P.ring_stride;
        ++saved;
      }
      begin_step(x_prev, x_cur, n, X, wr, [&](int g) { return qj * P.fload[g]; });
      solve(x_cur, j);
      theta = fma(pnorm_store(x_cur, hist_row(j)), inv_norm, theta);
      double* t = x_prev;
      x_prev = x_cur;
      x_cur = t;
    }
    store(x_prev, P.out_field + (size_t)s * P.Nn);
    if (threadIdx.x == 0 && rank == 0) P.out_aux[s] = power ? pow(theta, 1.0 / P.p) : theta;
  }

  __device__ __forceinline__ void fine_adjoint(int task) {
    const int s = P.s0 + task;
    const int M = P.M;
    const double scale = adjoint_scale(*P.Theta);
    double* x_prev = xa;
    double* x_cur = xb;
    load(P.in_field + (size_t)(s + 1) * P.Nn, x_prev);
    comm.sync();
    const double* gsrc = P.in_aux + (size_t)(s + 1) * P.Ne;
    double* gdst = P.out_aux + (size_t)s * P.Ne;
    const int nring = P.extrap;
    double* ring = nring > 1 && P.prev_field ? P.prev_field + (size_t)task * nring * P.ring_stride : nullptr;
    int saved = 0;
    for (int j = M * (s + 1); j >= M * s + 1; --j) {
      const double* Tj = hist_row(j);
      const double* Tjm = hist_row(j - 1);
      if (Tj == nullptr || Tjm == nullptr) {   // host validation makes this unreachable
        if (threadIdx.x == 0 && rank == 0) record_error(P.stats, PTG_EINVAL, P.stats_kind, j);
        return;
      }
      const double* X[kMaxExtrap - 1];
      int n = 1;
      double* wr = nullptr;
      if (ring) {
        n = min(saved + 1, nring);
        for (int i = 2; i <= n; ++i) X[i - 2] = ring + (size_t)((j + i) % nring) * P.ring_stride;
        wr = ring + (size_t)((j + 1) % nring) * P.ring_stride;
        ++saved;
      }
      begin_step(x_prev, x_cur, n, X, wr, [&](int g) { return scale * ipow(Tj[g], P.p_int - 1); });
      solve(x_cur, j);
      accumulate_g(x_cur, Tj, Tjm, gsrc, gdst, (double)P.Nt);
      gsrc = gdst;
      double* t = x_prev;
      x_prev = x_cur;
      x_cur = t;
      __syncthreads();
    }
    store(x_prev, P.out_field + (size_t)s * P.Nn);
  }

  // G_pri of slice s (one step of size dtau from u_s, started from the guess u_{s+1})
  __device__ __forceinline__ void coarse_primal(int task) {
    const int s = P.s0 + task;
    const int j = P.M * (s + 1);
    load(P.in_field + (size_t)s * P.Nn, xa);
    comm.sync();
    if (P.src_field) {
      const double* src = P.src_field + (size_t)s * P.Nn;
      build_rhs(xa, [&](int g) { return src[g]; });
    } else {
      const double qj = P.q_time[j];
      build_rhs(xa, [&](int g) { return qj * P.fload[g]; });
    }
    load(P.in_field + (size_t)(P.guess_next ? s + 1 : s) * P.Nn, xb);
    comm.sync();
    solve(xb, j);
    const double sp = pnorm_store(xb, P.out_field + (size_t)s * P.Nn);
    if (threadIdx.x == 0 && rank == 0)
      P.out_aux[s] = accumulate_theta(P.in_aux[s], sp / ((double)P.Ntau * (double)P.Ne));
  }

  // G_adj of slice s; src_mode 1 / 2 one of its two Theta-free parts (as the stepper)
  __device__ __forceinline__ void coarse_adjoint(int task) {
    const int s = P.s0 + task;
    const int kidx = P.M * s + 1;
    const int kprev = max(kidx - P.M, 0);
    const double scale = P.src_mode == 0 ? adjoint_scale(*P.Theta) : (P.src_mode == 1 ? 0.0 : 1.0);
    const double* Tk = P.hist + (size_t)kidx * P.Nn;
    const double* Tkm = P.hist + (size_t)kprev * P.Nn;
    if (P.src_mode == 2)
      zero_padded(xa);
    else
      load(P.in_field + (size_t)(s + 1) * P.Nn, xa);
    comm.sync();
    build_rhs(xa, [&](int g) { return scale * ipow(Tk[g], P.p_int - 1); });
    if (P.guess_next && P.src_mode == 0)
      load(P.in_field + (size_t)s * P.Nn, xb);
    else if (P.src_mode == 2)
      zero_padded(xb);
    else
      load(P.in_field + (size_t)(s + 1) * P.Nn, xb);
    comm.sync();
    solve(xb, kidx);
    accumulate_g(xb, Tk, Tkm, P.src_mode == 2 ? nullptr : P.in_aux + (size_t)(s + 1) * P.Ne,
                 P.out_aux + (size_t)s * P.Ne, (double)P.Ntau);
    store(xb, P.out_field + (size_t)s * P.Nn);
  }

  // Eq. 4.9 forward correction sweep (one task): u_{s+1} = G(u_s) + F[s] - G_old[s]
  __device__ __forceinline__ void correct_primal() {
    double theta;
    if (P.in_field) {                           // u_0 taken from the guess states, copied to X[0]
      load(P.in_field, xa);
      theta = P.in_aux[0];
      comm.sync();
      store(xa, P.out_field);
      if (threadIdx.x == 0 && rank == 0) P.out_aux[0] = theta;
    } else {
      load(P.out_field, xa);
      theta = P.out_aux[0];
    }
    store(xa, hist_row(0));
    if (P.plt) {                                // G = 0 (Sec. 7, Eq. 7.2): u_{s+1} = F(u_s^old)
      for (int s = 0; s < P.Ntau; ++s) {
        load(P.F_field + (size_t)s * P.Nn, xb);
        store(xb, P.out_field + (size_t)(s + 1) * P.Nn);
        store(xb, hist_row(P.M * (s + 1)));
        if (threadIdx.x == 0 && rank == 0) P.out_aux[s + 1] = P.F_aux[s];
      }
      return;
    }
    comm.sync();
    for (int s = 0; s < P.Ntau; ++s) {
      const int j = P.M * (s + 1);
      if (P.src_field) {
        const double* src = P.src_field + (size_t)s * P.Nn;
        build_rhs(xa, [&](int g) { return src[g]; });
      } else {
        const double qj = P.q_time[j];
        build_rhs(xa, [&](int g) { return qj * P.fload[g]; });
      }
      // start G(u_s^old) plus the extrapolated increments of the last min(extrap - 1, s) steps
      const int m = min(P.extrap - 1, min(s, 3));
      if (m >= 1) {
        const double* Fm[3];
        const double* X[3] = {nullptr, nullptr, nullptr};
        for (int i = 0; i < m; ++i) Fm[i] = P.F_field + (size_t)(s - 1 - i) * P.Nn;
        for (int i = 1; i < m; ++i) X[i] = P.out_field + (size_t)(s - i) * P.Nn;
        load_increment(P.G_field + (size_t)s * P.Nn, m, Fm, X, xa, xb);
      } else {
        load(P.G_field + (size_t)s * P.Nn, xb);
      }
      comm.sync();
      solve(xb, j);
      const double sp = pnorm_store(xb, nullptr);
      correction(xb, P.F_field + (size_t)s * P.Nn, P.G_field + (size_t)s * P.Nn, xa,
                 P.out_field + (size_t)(s + 1) * P.Nn, hist_row(j));
      if (threadIdx.x == 0) {
        const double theta_g = accumulate_theta(theta, sp / ((double)P.Ntau * (double)P.Ne));
        theta = (theta_g + P.F_aux[s]) - P.G_aux[s];
        if (rank == 0) P.out_aux[s + 1] = theta;
      }
      comm.sync();
    }
  }

  // Eq. 4.14 reverse correction sweep (one task): v_s = G(v_{s+1}) + F[s] - G_old[s], v_Ntau = 0
  __device__ __forceinline__ void correct_adjoint() {
    const double scale = adjoint_scale(*P.Theta);
    const int er = min(R, P.ny - r0);
    const int ne_own = er > 0 ? er * P.nx : 0;
    double* Xl = P.out_field + (size_t)P.Ntau * P.Nn;
    for_groups([&](int loc, int iy, int g) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int gi = gnode(iy, g, j);
        if (gi >= 0) Xl[gi] = 0.0;
      }
    });
    double* Xg = P.out_aux + (size_t)P.Ntau * P.Ne + (size_t)r0 * P.nx;
    for (int t = threadIdx.x; t < ne_own; t += blockDim.x) Xg[t] = 0.0;
    if (P.plt) {                                // G = 0: v_s = F(v_{s+1}^old)
      for (int s = P.Ntau - 1; s >= 0; --s) {
        load(P.F_field + (size_t)s * P.Nn, xb);
        store(xb, P.out_field + (size_t)s * P.Nn);
        const double* Fg = P.F_aux + (size_t)s * P.Ne + (size_t)r0 * P.nx;
        double* Og = P.out_aux + (size_t)s * P.Ne + (size_t)r0 * P.nx;
        for (int t = threadIdx.x; t < ne_own; t += blockDim.x) Og[t] = Fg[t];
      }
      return;
    }
    zero_padded(xa);
    comm.sync();
    for (int s = P.Ntau - 1; s >= 0; --s) {
      const int kidx = P.M * s + 1;
      const int kprev = max(kidx - P.M, 0);
      const double* Tk = P.hist + (size_t)kidx * P.Nn;
      const double* Tkm = P.hist + (size_t)kprev * P.Nn;
      build_rhs(xa, [&](int g) { return scale * ipow(Tk[g], P.p_int - 1); });
      // start G(v_{s+1}^old) plus the extrapolated increments of the last min(extrap - 1,
      // Ntau - 1 - s) steps
      const int m = min(P.extrap - 1, min(P.Ntau - 1 - s, 3));
      if (m >= 1) {
        const double* Fm[3];
        const double* X[3] = {nullptr, nullptr, nullptr};
        for (int i = 0; i < m; ++i) Fm[i] = P.F_field + (size_t)(s + 1 + i) * P.Nn;
        for (int i = 1; i < m; ++i) X[i] = P.out_field + (size_t)(s + 1 + i) * P.Nn;
        load_increment(P.G_field + (size_t)s * P.Nn, m, Fm, X, xa, xb);
      } else {
        load(P.G_field + (size_t)s * P.Nn, xb);
      }
      comm.sync();
      solve(xb, kidx);
      // g_s = g_{s+1} - (1/Ntau) term(lambda_G) + F_g[s] - G_g[s]
      accumulate_g(xb, Tk, Tkm, P.out_aux + (size_t)(s + 1) * P.Ne, P.out_aux + (size_t)s * P.Ne,
                   (double)P.Ntau, P.F_aux + (size_t)s * P.Ne, P.G_aux + (size_t)s * P.Ne);
      correction(xb, P.F_field + (size_t)s * P.Nn, P.G_field + (size_t)s * P.Nn, xa,
                 P.out_field + (size_t)s * P.Nn, nullptr);
      comm.sync();
    }
  }
};

// ngroups groups of P.cs CTAs; group g runs tasks g, g + ngroups, ... < P.wide_tasks (the
// correction sweeps are one task).
template <class Real, int KIND>
__global__ void __launch_bounds__(kStreamThreads, 1) stream_kernel(const __grid_constant__ StepParams P) {
  extern __shared__ __align__(128) float stream_smem[];
  __shared__ RedSmem rs;
  __shared__ unsigned long long ring_bar[kPipeRows];
  if (threadIdx.x == 0) {
    for (int i = 0; i < kPipeRows; ++i) mbar_init(&ring_bar[i]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  unsigned ring_phase = 0;
  bool ring_dead = false;
  GridComm comm(P, rs);
  Streamer<Real, KIND> st(P, comm, stream_smem, ring_bar, ring_phase, ring_dead);
  const int ngroups = (int)gridDim.x / P.cs;
  for (int task = comm.gid; task < P.wide_tasks; task += ngroups) {
    if constexpr (KIND == KIND_FINE_PRI) st.fine_primal(task);
    if constexpr (KIND == KIND_FINE_ADJ) st.fine_adjoint(task);
    if constexpr (KIND == KIND_COARSE_PRI) st.coarse_primal(task);
    if constexpr (KIND == KIND_COARSE_ADJ) st.coarse_adjoint(task);
    if constexpr (KIND == KIND_CORRECT_PRI) st.correct_primal();
    if constexpr (KIND == KIND_CORRECT_ADJ) st.correct_adjoint();
    comm.sync();                           // the group's workspace is free for its next task
  }
}

// The kernels of one task kind (FP32 and FP64 CG), instantiated in stream_inst.cu.
using StreamKernel = void (*)(const StepParams);
struct StreamKernels {
  StreamKernel f32, f64;
};
StreamKernels stream_select_0();
StreamKernels stream_select_1();
StreamKernels stream_select_2();
StreamKernels stream_select_3();
StreamKernels stream_select_4();
StreamKernels stream_select_5();

}  // namespace ptg
