// ptg_device.cuh -- device-side building blocks of the cluster time stepper.
//
// Layout (one thread-block cluster per independent time-stepping system):
//   * The (ny+1) node rows of the grid are split into CS horizontal slabs, one per CTA of
//     the cluster.  CTA `rank` owns node rows [r0, r0+R).
//   * Every grid-shaped buffer uses the padded row layout of ptg_internal.h: columns
//     ix = -1 .. W-2 at offsets ix+1 with W = roundup(nx+3, 4), zeros outside the domain,
//     kSlack entries of zero slack before and after.  Node buffers that a stencil reads hold
//     local rows lr = -1..R (one halo row on each side, filled by the neighbouring CTAs
//     through distributed shared memory stores); element buffers hold element rows r0-1 ..
//     r0+R-1.  Each thread works on aligned groups of 4 consecutive nodes of a row, so a
//     9-point stencil is a handful of 16-byte loads and needs no boundary branches.
//
// Operator (Sec. 2.2): for the bilinear square element with local node order SW, SE, NE,
// NW the matrix a*Ke + b*Me has only three distinct entries: a diagonal D, an edge-neighbour
// S and an opposite-corner T.  For C/dt + K with conductivity k_e and capacity c_e:
//   D = 4k/6 + 4m,  S = -k/6 + 2m,  T = -2k/6 + m,  m = c_e h^2 / (36 dt).
// Summing the four elements around a node gives the 9-point stencil used below.
#pragma once
#include <cooperative_groups.h>
#include <cstdint>
#include "ff.cuh"
#include "ptg_internal.h"

namespace ptg {
namespace cg = cooperative_groups;

constexpr int kMaxCluster = 16;
constexpr int kMaxWarps = 32;

// First device-side error wins: status code, the task kind and the time index.
__device__ __forceinline__ void record_error(DevStats* st, int code, int kind, int step) {
  if (atomicCAS(&st->status, 0, code) == 0) {
    st->fail_kind = 10 + kind;
    st->fail_step = step;
  }
}

// ---------------------------------------------------------------------------- cluster sync
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// the shared::cluster address of the same variable in CTA `rank` of the cluster
__device__ __forceinline__ unsigned mapa_u32(unsigned addr, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// 16 bytes into another CTA's shared memory; on arrival they count on that CTA's mbarrier
__device__ __forceinline__ void st_async16(unsigned addr, const uint4& v, unsigned bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
               "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
// this CTA's arrival, with the bytes that the phase waits for
__device__ __forceinline__ void mbar_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// whether the phase is complete, without waiting; mbar_try may wait a little
__device__ __forceinline__ bool mbar_test(unsigned long long* bar, unsigned parity) {
  unsigned done;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(done)
               : "r"(smem_u32(bar)), "r"(parity)
               : "memory");
  return done != 0;
}
__device__ __forceinline__ bool mbar_try(unsigned long long* bar, unsigned parity) {
  unsigned done;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(done)
               : "r"(smem_u32(bar)), "r"(parity)
               : "memory");
  return done != 0;
}

// A bounded wait: false where it ran out, after kMbarPolls polls (of 7 800 cycles when nothing arrives: four
// seconds) or after `limit` of them if positive
// (then without the waiting form of the poll, so that a limit of one poll runs out at once).
constexpr int kMbarPolls = 1 << 20;
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity, long long limit) {
  if (limit > 0) {
    for (long long i = 1; i < limit; ++i)
      if (mbar_test(bar, parity)) return true;
    return false;
  }
  for (int i = 0; i < kMbarPolls; ++i)
    if (mbar_try(bar, parity)) return true;
  return false;
}

// A not-a-number: what the reductions of a launch return once a wait of theirs has run out
template <class T> __device__ __forceinline__ T not_a_number();
template <> __device__ __forceinline__ float not_a_number<float>() { return __int_as_float(0x7fffffff); }
template <> __device__ __forceinline__ double not_a_number<double>() { return __hiloint2double(0x7fffffff, -1); }
template <> __device__ __forceinline__ ff not_a_number<ff>() { return make_ff(__int_as_float(0x7fffffff)); }

// Shared scratch for reductions (static shared memory of the stepper kernel).
constexpr int kMaxReduce = 5;      // values of one all-reduce (of floats; 4 of the 8-byte types)
struct RedSmem {
  // per-warp partials of this CTA and finalised values, of whatever type is being reduced: partials are
  // read between the two block barriers of a reduction and written outside them, final values the other way
  // round, so reductions of different types share the memory
  double warp[kMaxWarps * kMaxReduce];
  double bcast[8];
  uint4 slot[2][kRedWords][kMaxCluster]; // [phase][16-byte word][source rank]: that rank's partials
  unsigned long long bar[4];     // the cluster's mbarriers (comm.cuh): two for all-to-all, two for neighbour phases
  volatile int dead;             // a wait of this CTA ran out (ClusterComm)
};
template <class T>
struct RedBank {
  T (*warp)[kMaxReduce];
  T* bcast;
  __device__ __forceinline__ explicit RedBank(RedSmem& rs)
      : warp(reinterpret_cast<T (*)[kMaxReduce]>(rs.warp)), bcast(reinterpret_cast<T*>(rs.bcast)) {}
};

struct NoPost {
  template <class T>
  __device__ __forceinline__ void operator()(T*) const {}
};

// Sum over the warp, the same bits in every lane; half_warp_sum: over lanes 0..15, in lane 0 .. 15
// (the others' values are not used there).
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ ff warp_sum(ff v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = v + make_ff(__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o));
  return v;
}
__device__ __forceinline__ float half_warp_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ ff half_warp_sum(ff v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
    v = v + make_ff(__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o));
  return v;
}
// In double: an FP64 instruction of a warp holds its FP64 pipe for 64 cycles on this chip
// (measured, whatever the number of active lanes), so a butterfly costs 320 cycles per warp and
// value.  Instead the lanes' mantissas are aligned to the largest exponent as 57-bit integers (4
// guard bits below the 53 of a double, 5 bits of headroom for 32 terms) and summed by three
// integer reductions; one conversion brings the sum back.  The truncation is at most 32 x 2^-56 of
// the largest term.  Non-finite, huge and tiny operands take the butterfly.
__device__ __forceinline__ double warp_sum(double v) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  const int emax = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  if (emax < 128 || emax > 0x7f0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
  // lanes far below the largest term (denormals among them) shift out to zero
  const int sh = emax - e;
  unsigned long long m =
      (((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(v)) << 4;
  m = sh < 58 ? m >> sh : 0ull;
  const long long s = hi < 0 ? -(long long)m : (long long)m;
  const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)s & 0x3fffffu);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(s >> 22) & 0x3fffffu);
  const int l2 = __reduce_add_sync(0xffffffffu, (int)(s >> 44));
  const long long t = (long long)l0 + ((long long)l1 << 22) + ((long long)l2 << 44);
  if (t == 0) return 0.0;
  const double d = __ll2double_rn(t);
  return __hiloint2double(__double2hiint(d) + ((emax - (1023 + 56)) << 20), __double2loint(d));
}

// (the lanes from 16 on hold zeros where this is called)
__device__ __forceinline__ double half_warp_sum(double v) { return warp_sum(v); }

// ---------------------------------------------------------------------------- slab geometry
struct Slab {
  int nx, ny;      // elements per side
  int cs, rank;    // cluster size, this CTA's rank
  int r0, R;       // first owned node row, owned rows
  int W, G;        // padded row width and groups of 4 nodes per row
  int ngroups;     // owned groups R*G
};

__device__ __forceinline__ void slab_rows(int rows_total, int cs, int rank, int& r0, int& R) {
  const int base = rows_total / cs, rem = rows_total % cs;
  r0 = rank * base + (rank < rem ? rank : rem);
  R = base + (rank < rem ? 1 : 0);
}

// The residual that rounding leaves: x rounded to FP64 and A x evaluated in FP64 each contribute up to
// 2^-53 || |A| |x| ||, and |A| |x| is about 2 diag(A) |x| (the couplings of a Q1 element's node add up to about
// its diagonal), so || b - A x ||^2 of about 2^-102 sum (diag(A) x)^2 cannot be lowered.
constexpr double kRounding2 = 0x1p-102;

// x^e for an integer exponent e >= 1 by squaring, without the multiplications by one (exact
// operation order is fixed so every CTA and every run computes the same value).
__device__ __forceinline__ double ipow(double x, int e) {
  while (!(e & 1)) {
    x *= x;
    e >>= 1;
  }
  double r = x;
  while ((e >>= 1) > 0) {
    x *= x;
    if (e & 1) r *= x;
  }
  return r;
}

// ---------------------------------------------------------------------------- stencils
// 6-entry window of a row around a group: w[0] = offset b-1, w[1..4] = b..b+3, w[5] = b+4
// (b a multiple of 4).  One 16-byte load for the centre in float, two in double.
template <class T>
__device__ __forceinline__ void load_window(const T* __restrict__ x, int b, T (&w)[6]) {
  w[0] = x[b - 1];
  if constexpr (sizeof(T) == 4) {
    const float4 c = *reinterpret_cast<const float4*>(x + b);
    w[1] = c.x; w[2] = c.y; w[3] = c.z; w[4] = c.w;
  } else {
    const double2 c0 = *reinterpret_cast<const double2*>(x + b);
    const double2 c1 = *reinterpret_cast<const double2*>(x + b + 2);
    w[1] = c0.x; w[2] = c0.y; w[3] = c1.x; w[4] = c1.y;
  }
  w[5] = x[b + 4];
}

// 5-entry window of an element row: e[0] = offset b-1, e[1..4] = b..b+3 (b a multiple of 4).
__device__ __forceinline__ void load_ewindow(const float* __restrict__ w, int b, float (&e)[5]) {
  e[0] = w[b - 1];
  const float4 c = *reinterpret_cast<const float4*>(w + b);
  e[1] = c.x; e[2] = c.y; e[3] = c.z; e[4] = c.w;
}

__device__ __forceinline__ void load4(const double* __restrict__ p, double (&v)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  const double2 b = *reinterpret_cast<const double2*>(p + 2);
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// y = A x for the 4 nodes of a group, FP64 per-node weights (global memory).
// x: node buffer (rows -1..R); loc0: offset of the group's first node in x;
// go: offset of the same node in the padded global node arrays; W: row width.
template <class T>
__device__ __forceinline__ void stencil_node64(const T* __restrict__ x, int loc0, const NodeWeights& nw, int go, int W,
                                               double (&y)[4]) {
  T xl[6], xm[6], xh[6];
  load_window(x, loc0 - W, xl);
  load_window(x, loc0, xm);
  load_window(x, loc0 + W, xh);
  double C[4], No[4], Nb[4], NEo[4], NWo[4];
  load4(nw.C + go, C);
  load4(nw.N + go, No);
  load4(nw.N + go - W, Nb);
  load4(nw.NE + go, NEo);
  load4(nw.NW + go, NWo);
  double E[5];
  E[0] = nw.E[go - 1];
  {
    double e4[4];
    load4(nw.E + go, e4);
    E[1] = e4[0]; E[2] = e4[1]; E[3] = e4[2]; E[4] = e4[3];
  }
  const double* neb = nw.NE + go - W - 1;      // NE weights of the row below, shifted left
  const double* nwb = nw.NW + go - W + 1;      // NW weights of the row below, shifted right
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    double a = C[j] * (double)xm[j + 1];
    a = fma(E[j + 1], (double)xm[j + 2], a);   // east
    a = fma(E[j], (double)xm[j], a);           // west  = east weight of the west neighbour
    a = fma(No[j], (double)xh[j + 1], a);      // north
    a = fma(Nb[j], (double)xl[j + 1], a);      // south = north weight of the south neighbour
    a = fma(NEo[j], (double)xh[j + 2], a);     // north-east
    a = fma(neb[j], (double)xl[j], a);         // south-west = NE weight of the SW neighbour
    a = fma(NWo[j], (double)xh[j], a);         // north-west
    a = fma(nwb[j], (double)xl[j + 2], a);     // south-east = NW weight of the SE neighbour
    y[j] = a;
  }
}

// y = A z for the 4 nodes of a group: z in float, the per-node weights as float pairs (FFWeights,
// global memory), summed in pairs.  Row by row, which keeps few weights live.
__device__ __forceinline__ void stencil_ff(const float* __restrict__ z, int loc0, const FFWeights& nw, int go, int W,
                                           ff (&y)[4]) {
  const float *hi = nw.w + go, *lo = hi + 5 * (size_t)nw.stride;
  const size_t st = (size_t)nw.stride;
  auto ld = [](const float* p, float (&v)[4]) {
    const float4 c = *reinterpret_cast<const float4*>(p);
    v[0] = c.x; v[1] = c.y; v[2] = c.z; v[3] = c.w;
  };
  float v[6], ah[4], al[4], bh[4], bl[4], ch[4], cl[4];
  // the node's row: C, E of the node, E of the west neighbour
  load_window(z, loc0, v);
  ld(hi, ah);
  ld(lo, al);
  ld(hi + st, bh);
  ld(lo + st, bl);
  ch[0] = hi[st - 1];
  cl[0] = lo[st - 1];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float p, e;
    ff_prod(make_ff(ah[j], al[j]), v[j + 1], p, e);
    ff a = make_ff(p, e);
    a = ff_acc(a, make_ff(bh[j], bl[j]), v[j + 2]);
    y[j] = ff_acc(a, j == 0 ? make_ff(ch[0], cl[0]) : make_ff(bh[j - 1], bl[j - 1]), v[j]);
  }
  // the row above: N, NE, NW of the node
  load_window(z, loc0 + W, v);
  ld(hi + 2 * st, ah);
  ld(lo + 2 * st, al);
  ld(hi + 3 * st, bh);
  ld(lo + 3 * st, bl);
  ld(hi + 4 * st, ch);
  ld(lo + 4 * st, cl);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    y[j] = ff_acc(y[j], make_ff(ah[j], al[j]), v[j + 1]);
    y[j] = ff_acc(y[j], make_ff(bh[j], bl[j]), v[j + 2]);
    y[j] = ff_acc(y[j], make_ff(ch[j], cl[j]), v[j]);
  }
  // the row below: N of the south, NE of the south-west, NW of the south-east neighbour
  load_window(z, loc0 - W, v);
  ld(hi + 2 * st - W, ah);
  ld(lo + 2 * st - W, al);
  ld(hi + 3 * st - W, bh);
  ld(lo + 3 * st - W, bl);
  ld(hi + 4 * st - W, ch);
  ld(lo + 4 * st - W, cl);
  const ff ne = make_ff(hi[3 * st - W - 1], lo[3 * st - W - 1]), nw4 = make_ff(hi[4 * st - W + 4], lo[4 * st - W + 4]);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    y[j] = ff_acc(y[j], make_ff(ah[j], al[j]), v[j + 1]);
    y[j] = ff_acc(y[j], j == 0 ? ne : make_ff(bh[j - 1], bl[j - 1]), v[j]);
    y[j] = ff_acc(y[j], j == 3 ? nw4 : make_ff(ch[j + 1], cl[j + 1]), v[j + 2]);
  }
}

// y = A z for the 4 nodes of a group, FP32 element weights (D, S, T).
// For the node at window position c = j+1: elements a, b below-left / below-right and c, d
// above-left / above-right, i.e. element windows lower[j], lower[j+1], upper[j], upper[j+1].
__device__ __forceinline__ void stencil_elem32(const float* __restrict__ z, const float* __restrict__ wd,
                                               const float* __restrict__ ws, const float* __restrict__ wt, int loc0,
                                               int W, float (&y)[4]) {
  float zl[6], zm[6], zh[6];
  load_window(z, loc0 - W, zl);
  load_window(z, loc0, zm);
  load_window(z, loc0 + W, zh);
  float dl[5], sl[5], tl[5], du[5], su[5], tu[5];
  const int el = loc0 - W, eu = loc0;   // element windows share the node buffers' row offsets
  load_ewindow(wd, el, dl);
  load_ewindow(ws, el, sl);
  load_ewindow(wt, el, tl);
  load_ewindow(wd, eu, du);
  load_ewindow(ws, eu, su);
  load_ewindow(wt, eu, tu);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float Da = dl[j], Db = dl[j + 1], Dc = du[j], Dd = du[j + 1];
    const float Sa = sl[j], Sb = sl[j + 1], Sc = su[j], Sd = su[j + 1];
    float a = ((Da + Db) + (Dc + Dd)) * zm[j + 1];
    a = fmaf(Sa + Sc, zm[j], a);           // west:  shared by a, c
    a = fmaf(Sb + Sd, zm[j + 2], a);       // east:  shared by b, d
    a = fmaf(Sa + Sb, zl[j + 1], a);       // south: shared by a, b
    a = fmaf(Sc + Sd, zh[j + 1], a);       // north: shared by c, d
    a = fmaf(tl[j], zl[j], a);             // south-west corner of a
    a = fmaf(tl[j + 1], zl[j + 2], a);     // south-east corner of b
    a = fmaf(tu[j], zh[j], a);             // north-west corner of c
    a = fmaf(tu[j + 1], zh[j + 2], a);     // north-east corner of d
    y[j] = a;
  }
}

// The same from the elements' conductivity and capacity parts k = k_e/6 and m = c_e h^2/(36 step),
// D = 4 (k + m), S = 2 m - k, T = m - 2 k, and with the window entries beyond a lane's own 16 bytes
// taken from the neighbouring lanes: the groups of a warp are consecutive in the row-padded
// buffers (from one row's last group to the next row's first, whose pads are zero), so only the
// warp's first and last lane load them.  A 4-byte load at a 16-byte stride takes 4 shared-memory
// wavefronts, like the 16-byte load beside it; this form takes about 45 wavefronts per warp where
// stencil_elem32 takes 84, and the smoothers and the FP32 CG are bound by them (17 x 132 nodes in
// two CTAs: 2 860 cycles per application).  Every lane of the warp calls it.
__device__ __forceinline__ void warp_window(const float* __restrict__ x, int b, int lane, float (&w)[6]) {
  const float4 c = *reinterpret_cast<const float4*>(x + b);
  float e = 0.f;
  if (lane == 0 || lane == 31) e = x[lane == 0 ? b - 1 : b + 4];
  const float l = __shfl_up_sync(0xffffffffu, c.w, 1), r = __shfl_down_sync(0xffffffffu, c.x, 1);
  w[0] = lane == 0 ? e : l;
  w[1] = c.x; w[2] = c.y; w[3] = c.z; w[4] = c.w;
  w[5] = lane == 31 ? e : r;
}
__device__ __forceinline__ void warp_ewindow(const float* __restrict__ x, int b, int lane, float (&w)[5]) {
  const float4 c = *reinterpret_cast<const float4*>(x + b);
  float e = 0.f;
  if (lane == 0) e = x[b - 1];
  const float l = __shfl_up_sync(0xffffffffu, c.w, 1);
  w[0] = lane == 0 ? e : l;
  w[1] = c.x; w[2] = c.y; w[3] = c.z; w[4] = c.w;
}
// A z on a group from z's windows and the element windows (columns b-1 .. b+3) below and above
template <int N>
__device__ __forceinline__ void km_combine(const float (&zl)[6], const float (&zm)[6], const float (&zh)[6],
                                           const float (&kl)[N], const float (&ml)[N], const float (&ku)[N],
                                           const float (&mu)[N], float (&y)[4]) {
  float d[5], sl[5], su[5], tl[5], tu[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    d[i] = (kl[i] + ml[i]) + (ku[i] + mu[i]);
    sl[i] = fmaf(2.f, ml[i], -kl[i]);
    su[i] = fmaf(2.f, mu[i], -ku[i]);
    tl[i] = fmaf(-2.f, kl[i], ml[i]);
    tu[i] = fmaf(-2.f, ku[i], mu[i]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float a = 4.f * (d[j] + d[j + 1]) * zm[j + 1];
    a = fmaf(sl[j] + su[j], zm[j], a);             // west
    a = fmaf(sl[j + 1] + su[j + 1], zm[j + 2], a); // east
    a = fmaf(sl[j] + sl[j + 1], zl[j + 1], a);     // south
    a = fmaf(su[j] + su[j + 1], zh[j + 1], a);     // north
    a = fmaf(tl[j], zl[j], a);
    a = fmaf(tl[j + 1], zl[j + 2], a);
    a = fmaf(tu[j], zh[j], a);
    a = fmaf(tu[j + 1], zh[j + 2], a);
    y[j] = a;
  }
}
__device__ __forceinline__ void stencil_km32(const float* __restrict__ z, const float* __restrict__ wk,
                                             const float* __restrict__ wm, int loc0, int W, int lane, float (&y)[4],
                                             bool no_lo = false, bool no_hi = false) {
  float zl[6], zm[6], zh[6], kl[5], ml[5], ku[5], mu[5];
  // (a row that is left out is not read either: a neighbour may be writing it)
  warp_window(z, no_lo ? loc0 : loc0 - W, lane, zl);
  warp_window(z, loc0, lane, zm);
  warp_window(z, no_hi ? loc0 : loc0 + W, lane, zh);
  warp_ewindow(wk, loc0 - W, lane, kl);
  warp_ewindow(wm, loc0 - W, lane, ml);
  warp_ewindow(wk, loc0, lane, ku);
  warp_ewindow(wm, loc0, lane, mu);
  if (no_lo) {
#pragma unroll
    for (int i = 0; i < 6; ++i) zl[i] = 0.f;
  }
  if (no_hi) {
#pragma unroll
    for (int i = 0; i < 6; ++i) zh[i] = 0.f;
  }
  km_combine(zl, zm, zh, kl, ml, ku, mu, y);
}

// Element bilinear forms of Eq. 4.7 in the modes that Ke and Me share as eigenvectors: with the
// corner values in the order SW, SE, NE, NW the sums a = (1, 1, 1, 1), b = (-1, 1, 1, -1),
// c = (-1, -1, 1, 1) and d = (1, -1, 1, -1) have the eigenvalues 0, 1, 1, 2/3 of Ke and
// (h^2/36) (9, 3, 3, 1) of Me, so
//   lambda^T Ke T = (b b' + c c' + (2/3) d d') / 4,
//   lambda^T Me T = (h^2/36) (9 a a' + 3 (b b' + c c') + d d') / 4.
// The sums are bound by the FP64 pipe (an FP64 instruction of a warp takes 64 cycles on this
// chip): 8 additions per field and 3 or 4 products replace the 20 multiply-adds of each 4 x 4 form.
struct Modes {
  double a, b, c, d;
};
__device__ __forceinline__ Modes elem_modes(double sw, double se, double ne, double nw) {
  const double p = se - sw, q = ne - nw, bot = sw + se, top = nw + ne;
  return Modes{top + bot, p + q, top - bot, q - p};
}
__device__ __forceinline__ double elem_stiffness(const Modes& l, const Modes& t) {
  return fma(l.d * t.d, 1.0 / 6.0, 0.25 * fma(l.b, t.b, l.c * t.c));
}
// (times h^2)
__device__ __forceinline__ double elem_mass(const Modes& l, const Modes& t) {
  return fma(l.a * t.a, 1.0 / 16.0, fma(l.d * t.d, 1.0 / 144.0, fma(l.b, t.b, l.c * t.c) * (1.0 / 48.0)));
}

// Eq. 4.7 for H elements above one another over the contiguous steps ja..jb (ja <= jb): the sums
// over j of lambda_j,e^T ( dke Ke T_j,e + dce Me (T_j - T_{j-1})_e ), dce already divided by the
// step size.  g0 is the lowest element's SW node, nn = nx + 1, Nn the node count; lambda_j is row
// j - j0 of lam and T_j row j - hist_j0 of T; rows from `rows` on (1 <= rows <= H) are left out.
// The row differences and sums of two neighbouring elements are shared, and each step's modes of
// T serve the next one as T_{j-1}, so a step costs 13 FP64 instructions per element, 23 with the
// capacity term (has_dc).
template <int H>
__device__ __forceinline__ void sens_strip_sum(int g0, int nn, int Nn, double h2, const double (&dke)[H],
                                               const double (&dce)[H], bool has_dc, int rows,
                                               const double* __restrict__ lam, int j0, const double* __restrict__ T,
                                               int hist_j0, int ja, int jb, double (&out)[H]) {
  double k1[H], k2[H], m9[H], m3[H], m1[H];
  Modes prev[H];
#pragma unroll
  for (int i = 0; i < H; ++i) k1[i] = k2[i] = m9[i] = m3[i] = m1[i] = 0.0;
  const double* Tp = T + (size_t)(ja - 1 - hist_j0) * Nn + g0;
  const double* Lj = lam + (size_t)(ja - j0) * Nn + g0;
  if (has_dc) {
#pragma unroll
    for (int i = 0; i < H; ++i)
      if (i < rows) prev[i] = elem_modes(Tp[i * nn], Tp[i * nn + 1], Tp[(i + 1) * nn + 1], Tp[(i + 1) * nn]);
  }
  for (int j = ja; j <= jb; ++j) {
    Tp += Nn;                                  // T_j
    double tp, ts, lp, ls;                     // difference and sum along the row below
    {
      const double t0 = Tp[0], t1 = Tp[1], l0 = Lj[0], l1 = Lj[1];
      tp = t1 - t0;
      ts = t0 + t1;
      lp = l1 - l0;
      ls = l0 + l1;
    }
#pragma unroll
    for (int i = 0; i < H; ++i) {
      if (i >= rows) break;
      const double t0 = Tp[(i + 1) * nn], t1 = Tp[(i + 1) * nn + 1], l0 = Lj[(i + 1) * nn], l1 = Lj[(i + 1) * nn + 1];
      const double tq = t1 - t0, tt = t0 + t1, lq = l1 - l0, lt = l0 + l1;
      const Modes t{has_dc ? tt + ts : 0.0, tp + tq, tt - ts, tq - tp};
      const Modes l{has_dc ? lt + ls : 0.0, lp + lq, lt - ls, lq - lp};
      k1[i] = fma(l.b, t.b, fma(l.c, t.c, k1[i]));
      k2[i] = fma(l.d, t.d, k2[i]);
      if (has_dc) {
        m9[i] = fma(l.a, t.a - prev[i].a, m9[i]);
        m3[i] = fma(l.b, t.b - prev[i].b, fma(l.c, t.c - prev[i].c, m3[i]));
        m1[i] = fma(l.d, t.d - prev[i].d, m1[i]);
        prev[i] = t;
      }
      tp = tq;
      ts = tt;
      lp = lq;
      ls = lt;
    }
    Lj += Nn;
  }
#pragma unroll
  for (int i = 0; i < H; ++i) {
    out[i] = dke[i] * 0.25 * fma(2.0 / 3.0, k2[i], k1[i]);
    if (has_dc) out[i] += dce[i] * h2 * (1.0 / 144.0) * fma(9.0, m9[i], fma(3.0, m3[i], m1[i]));
  }
}

}  // namespace ptg
