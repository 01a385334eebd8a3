// comm.cuh -- how the CTAs that share one linear system talk to each other.
//
// The stepper (stepper.cuh) needs four collective operations: an all-reduce of a few
// scalars, the exchange of the first and last owned node rows with the neighbouring slabs
// (halo rows), a barrier, and the broadcast of the two-level preconditioner's restricted
// partials.  Two implementations:
//
//   ClusterComm  one thread-block cluster (up to 16 CTAs): asynchronous stores to distributed
//                shared memory that count on the receiver's mbarriers.  Used wherever several independent
//                systems run side by side (one cluster each).
//   GridComm     groups of G CTAs of one cooperative launch (up to kMaxGrid CTAs in all, one
//                per SM), each group running one system at a time: global memory and a
//                counting barrier per group.  Used for a single large FP64 system, spread over
//                every SM instead of one cluster (kWideMinNodes in api.cu has the times), and for
//                grids whose slabs do not fit 16 CTAs.
//
// Both produce bitwise identical reductions in every CTA (fixed summation orders).
#pragma once
#include "ptg_device.cuh"

namespace ptg {

constexpr long kGridSpinLimit = 1L << 20; // polls of a grid barrier before it reports PTG_ETIMEOUT

// ---------------------------------------------------------------------------- cluster
// Everything a CTA sends goes out as 16-byte st.async stores that count their bytes on an mbarrier
// of the receiving CTA, which waits for the bytes it expects: one one-way trip instead of remote
// stores followed by the hardware cluster barrier (16 CTAs, measured: 430 against 1100 cycles at
// 320 threads; an all-reduce inside a CG iteration is mostly this latency).
//
// Phases.  An all-to-all phase (all-reduce, restricted partials) receives bytes from every CTA, a
// neighbour phase (halo rows) from the slabs above and below.  Each of the two uses its own pair
// of mbarriers in turn.  A pair is enough: a CTA sends in phase n + 2 only after it has completed
// phase n + 1, for which it needed the receiver's bytes, which the receiver sent after it had
// completed phase n (in a neighbour phase senders and receivers are mutual).  Buffers written
// remotely are safe by the same argument wherever an all-to-all phase lies between the last read
// of a buffer and the next send into it; the stepper has one between any two sends into the same
// buffer.
//
// Every wait is bounded (P.wait_limit polls, kMbarPolls if not positive).  A thread whose wait runs out
// records PTG_ETIMEOUT, and its CTA gives up: from the next reduction on no thread of it sends, expects
// bytes or waits, and every reduction returns NaN, which ends each CG and each residual loop at once.
// The other CTAs, whose waits for it run out in turn, follow.  So
//   - an mbarrier is never armed for a phase while its phase before is open (only thread 0 arms them, and
//     only after its own wait for the phase before);
//   - loop decisions come from values that warp 0 publishes to the whole CTA, and the hardware barriers
//     (sync, order_global) stand outside those loops: every CTA passes the same number of them;
//   - a CTA that has given up may still be sent the bytes of a phase or two (a few KB, within an
//     mbarrier's range).  drain() keeps it until they have landed.

struct ClusterComm {
  cg::cluster_group cl;
  RedSmem& rs;
  const StepParams* P = nullptr;   // for error reports
  unsigned na = 0, nn = 0;         // all-to-all and neighbour phases completed
  unsigned pend_a = 0, pend_n = 0; // bytes this CTA expects in the next phase of each kind
  bool broken = false;             // a wait of this thread ran out, or it has seen that the CTA gave up

  // Before the first use: the CTA's mbarriers; the caller follows with cluster_sync_all().
  __device__ ClusterComm(RedSmem& rs_) : cl(cg::this_cluster()), rs(rs_) {
    if (threadIdx.x == 0) {
      rs.dead = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) mbar_init(&rs.bar[i]);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  __device__ void bind(const StepParams& P_) { P = &P_; }
  __device__ int rank() const { return (int)cl.block_rank(); }
  __device__ void sync() { cluster_sync_all(); }
  // Orders the cluster's global stores before its global loads: between a CTA's stores to a global row
  // and a neighbour's loads of it.  The phases above order shared memory alone: the completion of
  // an st.async releases that store, not the earlier global stores of the CTA's other threads, and
  // a row that is written again may still sit in the reader's L1.  The hardware barrier's release and
  // acquire cover both (16 CTAs: 430 cycles, once per time step).
  __device__ void order_global() { cluster_sync_all(); }

  __device__ __forceinline__ unsigned long long* bar_a() { return &rs.bar[na & 1]; }
  __device__ __forceinline__ unsigned long long* bar_n() { return &rs.bar[2 + (nn & 1)]; }
  __device__ __forceinline__ void wait(unsigned long long* bar, unsigned parity) {
    if (broken || mbar_test(bar, parity)) return;
    if (mbar_wait(bar, parity, P->wait_limit)) return;
    broken = true;
    rs.dead = 1;
    record_error(P->stats, PTG_ETIMEOUT, P->stats_kind, -1);
  }
  // After a block barrier behind the last wait: whether this CTA gave up.
  __device__ bool dead() const { return rs.dead != 0; }
  // The end of a launch, after the cluster barrier behind which no CTA sends: where this CTA gave up,
  // nobody has counted the bytes that are still on their way to its shared memory (they take about a
  // microsecond); it stays for 200 000 cycles.
  __device__ void drain() const {
    if (threadIdx.x != 0 || !dead()) return;
    const long long t0 = clock64();
    for (int i = 0; i < (1 << 16) && clock64() - t0 < 200000; ++i) __nanosleep(100);
  }
  __device__ __forceinline__ void done_a() {
    ++na;
    pend_a = 0;
  }
  // The end of a phase whose sends are on their way: every thread waits for the expected bytes.
  __device__ void finish_a() {
    if (threadIdx.x == 0 && !broken) mbar_expect(bar_a(), pend_a);
    wait(bar_a(), (na >> 1) & 1);
    done_a();
  }
  __device__ void finish_n() {
    if (threadIdx.x == 0 && !broken) mbar_expect(bar_n(), pend_n);
    wait(bar_n(), (nn >> 1) & 1);
    ++nn;
    pend_n = 0;
  }

  // All-reduce of the first NV entries of v, then `post` as in GridComm.  Warp sums, then warp 0
  // adds the warps' partials and sends the CTA's sums to every rank; warp 0 waits, adds the ranks'
  // sums, applies `post` and hands the result to the CTA.  Every rank adds the same values in the
  // same order: the same bits everywhere.
  template <class T, int NV, int NX, class Post>
  __device__ void allreduce(T (&v)[NV + NX], int cs, Post post) {
    constexpr int kWords = (NV * (int)sizeof(T) + 15) / 16;
    static_assert(NV <= kMaxReduce && NV + NX <= 8 && kWords <= kRedWords, "16-byte words per rank");
    const RedBank<T> rb(rs);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i) rb.warp[warp][i] = v[i];
    }
    __syncthreads();
    if (warp == 0) {
      // the same in the whole warp: every earlier wait of the CTA lies before the block barrier
      broken = dead();
      union { uint4 u[kWords]; T t[16 * kWords / sizeof(T)]; } pk;
#pragma unroll
      for (int w = 0; w < kWords; ++w) pk.u[w] = make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int i = 0; i < NV; ++i) pk.t[i] = half_warp_sum(lane < nwarps ? rb.warp[lane][i] : T{});
      if (lane < cs && !broken) {
        const unsigned b = mapa_u32(smem_u32(bar_a()), (unsigned)lane);
#pragma unroll
        for (int w = 0; w < kWords; ++w)
          st_async16(mapa_u32(smem_u32(&rs.slot[na & 1][w][rank()]), (unsigned)lane), pk.u[w], b);
      }
      if (lane == 0 && !broken) mbar_expect(bar_a(), pend_a + 16u * kWords * (unsigned)cs);
      wait(bar_a(), (na >> 1) & 1);
#pragma unroll
      for (int w = 0; w < kWords; ++w) pk.u[w] = rs.slot[na & 1][w][lane < cs ? lane : 0];
      T t[NV + NX];
#pragma unroll
      for (int i = 0; i < NV; ++i) t[i] = half_warp_sum(broken ? not_a_number<T>() : lane < cs ? pk.t[i] : T{});
#pragma unroll
      for (int i = NV; i < NV + NX; ++i) t[i] = T{};
      post(t);
      if (lane == 0) {
#pragma unroll
        for (int i = 0; i < NV + NX; ++i) rb.bcast[i] = t[i];
      }
    }
    done_a();
    __syncthreads();
    broken = dead();
#pragma unroll
    for (int i = 0; i < NV + NX; ++i) v[i] = rb.bcast[i];
  }

  // Rows of `words16` 16-byte words: the own first / last row into the halo rows of the CTAs below
  // and above (their rows dst_lo / dst_hi), counting on `bar` there.
  __device__ __forceinline__ void send_rows(const void* first, const void* last, const void* dst_lo, const void* dst_hi,
                                            int words16, int rank_, int cs, unsigned long long* bar) {
    if (broken) return;
    if (rank_ > 0) {
      const unsigned d = mapa_u32(smem_u32(dst_lo), (unsigned)(rank_ - 1)), b = mapa_u32(smem_u32(bar), (unsigned)(rank_ - 1));
      const uint4* s = reinterpret_cast<const uint4*>(first);
      for (int i = threadIdx.x; i < words16; i += blockDim.x) st_async16(d + 16 * i, s[i], b);
    }
    if (rank_ < cs - 1) {
      const unsigned d = mapa_u32(smem_u32(dst_hi), (unsigned)(rank_ + 1)), b = mapa_u32(smem_u32(bar), (unsigned)(rank_ + 1));
      const uint4* s = reinterpret_cast<const uint4*>(last);
      // from the block's other end, so that different threads carry the two rows
      for (int i = (int)blockDim.x - 1 - (int)threadIdx.x; i < words16; i += blockDim.x) st_async16(d + 16 * i, s[i], b);
    }
  }
  __device__ __forceinline__ unsigned row_bytes(int words16, int rank_, int cs) const {
    return 16u * (unsigned)words16 * ((rank_ > 0 ? 1u : 0u) + (rank_ < cs - 1 ? 1u : 0u));
  }
  // Own first / last rows of a halo buffer (`buf` at row -1, row lr at buf + (lr+1) W) into the
  // neighbours' halo rows; on return the own halo rows are the neighbours' rows.  The caller's
  // block barrier has made this CTA's rows visible.
  template <class T>
  __device__ void exchange(T* buf, const Slab& sb) {
    const int n16 = sb.W * (int)sizeof(T) / 16;
    int r0n = 0, Rn = 0;
    if (sb.rank > 0) slab_rows(sb.ny + 1, sb.cs, sb.rank - 1, r0n, Rn);
    send_rows(buf + sb.W, buf + sb.R * sb.W, buf + (Rn + 1) * sb.W, buf, n16, sb.rank, sb.cs, bar_n());
    pend_n += row_bytes(n16, sb.rank, sb.cs);
    finish_n();
  }
  // The same for a buffer on the 2h level of the three-level cycle: rows of W1 floats, R1 owned
  // rows here, R1b owned rows in the CTA below (whose halo row lr = R1b receives row 0).
  __device__ void exchange_rows(float* buf, int W1, int R1, int R1b, int rank_, int cs) {
    const int n16 = W1 / 4;
    send_rows(buf + W1, buf + R1 * W1, buf + (R1b + 1) * W1, buf, n16, rank_, cs, bar_n());
    pend_n += row_bytes(n16, rank_, cs);
    finish_n();
  }
  // Edge rows sent straight from registers: the thread holding columns [col, col+4) of the
  // owned row lr (0 or R-1) stores them into the neighbour's two-row buffer `edge` ([0]: the
  // row below that CTA's slab, [1]: the row above); a neighbour phase that finish_edges ends.
  __device__ void begin_edges() {}
  template <class T>
  __device__ void put_edge(T* edge, int lr, int col, const T (&v)[4], const Slab& sb) {
    if (broken) return;
    unsigned long long* bar = bar_n();
    union { uint4 u[sizeof(T) / 4]; T t[4]; } pk;
#pragma unroll
    for (int j = 0; j < 4; ++j) pk.t[j] = v[j];
    if (lr == 0 && sb.rank > 0) {
      const unsigned r = (unsigned)(sb.rank - 1);
      const unsigned d = mapa_u32(smem_u32(edge + sb.W + col), r), b = mapa_u32(smem_u32(bar), r);
#pragma unroll
      for (int w = 0; w < (int)sizeof(T) / 4; ++w) st_async16(d + 16 * w, pk.u[w], b);
    }
    if (lr == sb.R - 1 && sb.rank < sb.cs - 1) {
      const unsigned r = (unsigned)(sb.rank + 1);
      const unsigned d = mapa_u32(smem_u32(edge + col), r), b = mapa_u32(smem_u32(bar), r);
#pragma unroll
      for (int w = 0; w < (int)sizeof(T) / 4; ++w) st_async16(d + 16 * w, pk.u[w], b);
    }
  }
  template <class T>
  __device__ void end_edges(T*, const Slab& sb) {
    pend_n += row_bytes(sb.W * (int)sizeof(T) / 16, sb.rank, sb.cs);
  }
  __device__ void finish_edges() { finish_n(); }
  // a 16-byte chunk of restricted partials, written at offset dst of every rank's slot array;
  // the 16 lanes `sub` = 0..15 of a half-warp share the destinations.  Part of the next all-to-all
  // phase; expect_tl adds the bytes that all ranks together send to each.
  __device__ void publish_tl(float* slot, int dst, const float4& chunk, int sub, int cs) {
    if (broken) return;
    const uint4 u = make_uint4(__float_as_uint(chunk.x), __float_as_uint(chunk.y), __float_as_uint(chunk.z),
                               __float_as_uint(chunk.w));
    for (int q = sub; q < cs; q += 16)
      st_async16(mapa_u32(smem_u32(slot + dst), (unsigned)q), u, mapa_u32(smem_u32(bar_a()), (unsigned)q));
  }
  __device__ void expect_tl(unsigned bytes) { pend_a += bytes; }
  __device__ void finish_tl() { finish_a(); }
  __device__ const float* tl_slots(const float* local) const { return local; }
  __device__ float4 tl_load4(const float* slots, int idx) const {
    return *reinterpret_cast<const float4*>(slots + idx);
  }
};

// ---------------------------------------------------------------------------- grid
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
template <class T>
__device__ __forceinline__ T ldcg(const T* p) { return __ldcg(p); }
__device__ __forceinline__ ff ldcg(const ff* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return make_ff(v.x, v.y);
}
__device__ __forceinline__ void st_release_gpu(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void red_release_add_gpu(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// The CTAs of a cooperative launch form groups of G = P.cs consecutive CTAs; each group runs
// one system at a time.  Reduction partials, halo rows and two-level partials are indexed by
// the global block index (every group owns its range); the barrier has one set of counters per
// group.
struct GridComm {
  const StepParams& P;
  RedSmem& rs;
  int phase = 0;
  const int G;                   // CTAs of the group
  const int gid;                 // group index
  const int base;                // first block of the group
  // halo rows published by push_halos and pulled in after the next barrier; pushes alternate
  // between two slot sets, so a CTA that has passed a barrier never overwrites slots that a
  // slower CTA of the group may still be pulling from the push before it
  unsigned char* pending_lo = nullptr;   // where the row below the slab goes (null: nothing pending)
  unsigned char* pending_hi = nullptr;   // where the row above goes
  int pending_bytes = 0;         // bytes of one row
  int hset = 0;                  // slot set of the latest push
  unsigned epoch = 0;            // barriers this CTA has passed in the launch
  bool broken = false;           // thread 0: a wait of the group ran out; its reductions return NaN

  __device__ GridComm(const StepParams& P_, RedSmem& rs_)
      : P(P_), rs(rs_), G(P_.cs), gid((int)blockIdx.x / P_.cs), base(((int)blockIdx.x / P_.cs) * P_.cs) {}
  __device__ int rank() const { return (int)blockIdx.x - base; }

  // Counting barrier over the CTAs of the group (co-resident: cooperative launch).  The group's
  // arrival count (zeroed before the launch) only grows: thread 0 of each CTA adds 1 with release
  // semantics, which publishes the CTA's global writes ordered before it by the block barrier, and
  // polls with acquire loads until the count reaches G times the barriers passed, which makes
  // every other CTA's writes before its arrival visible.  One global round trip after the last
  // arrival; no reset.  A wait that reaches P.wait_limit polls (kGridSpinLimit if not positive)
  // records PTG_ETIMEOUT and returns; once any CTA has recorded it (the group's broken flag,
  // P.g_bar[4 gid + 2]), every later wait returns at once, so a broken launch ends quickly with
  // the error instead of waiting out every barrier.
  __device__ __forceinline__ void barrier() {
    __syncthreads();
    if (G == 1) {                // a group of one CTA: the block barrier orders its global accesses
      pull_halos();
      return;
    }
    if (threadIdx.x == 0) arrive_and_wait();
    __syncthreads();
    pull_halos();
  }
  // One thread's part, after a block barrier (or its own stores).  The release of the arrival and
  // the acquire of the poll order every store of the CTA that the block barrier put before it, and
  // every load after the next block barrier; a fence on top of each would cost a round trip.
  __device__ __forceinline__ void arrive_and_wait() {
    unsigned* count = P.g_bar + 4 * gid;
    unsigned* flag = count + 2;
    ++epoch;
    const unsigned target = epoch * (unsigned)G;
    red_release_add_gpu(count, 1u);
    if (broken) return;
    const long long limit = P.wait_limit > 0 ? P.wait_limit : (long long)kGridSpinLimit;
    long long spins = 0;
    while ((int)(ld_acquire_gpu(count) - target) < 0) {
      if ((++spins & 255) == 0 && ld_acquire_gpu(flag) != 0u) {
        broken = true;
        break;
      }
      if (spins >= limit) {
        give_up();
        break;
      }
    }
  }
  // One thread: a wait ran out.  Every later wait of the group returns at once.
  __device__ void give_up() {
    record_error(P.stats, PTG_ETIMEOUT, P.stats_kind, -1);
    atomicExch(P.g_bar + 4 * gid + 2, 1u);
    broken = true;
  }
  __device__ void sync() { barrier(); }
  // every phase of a group is its barrier, a release and an acquire at gpu scope: nothing left to order
  __device__ void order_global() {}

  template <class T, int NV, int NX, class Post>
  __device__ __forceinline__ void allreduce(T (&v)[NV + NX], int /*cs*/, Post post) {
    const RedBank<T> rb(rs);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i) rb.warp[warp][i] = v[i];
    }
    __syncthreads();
    // the same bytes per block whatever T: the groups of a launch are not in step, and one may reduce floats
    // while another reduces doubles
    constexpr int kPer = 16 * kRedWords / (int)sizeof(T);
    static_assert(NV <= kPer && NV <= kMaxReduce && NV + NX <= 8, "a block's part of g_red");
    T* slots = reinterpret_cast<T*>(P.g_red + (size_t)phase * kMaxGrid * 2 * kRedWords);
    // warp 0 alone: the CTA's sums into its slots, the barrier, lane-strided sums over the ranks and
    // the warp's sum, then `post`; broadcast
    if (warp == 0) {
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        const T s = half_warp_sum(lane < nwarps ? rb.warp[lane][i] : T{});
        if (lane == 0) slots[(int)blockIdx.x * kPer + i] = s;
      }
      if (lane == 0 && G > 1) arrive_and_wait();
      __syncwarp();
      T t[NV + NX];
#pragma unroll
      for (int i = 0; i < NV; ++i) {
        T a = broken ? not_a_number<T>() : T{};
        for (int r = lane; r < G; r += 32) a = a + ldcg(slots + (base + r) * kPer + i);
        t[i] = warp_sum(a);
      }
#pragma unroll
      for (int i = NV; i < NV + NX; ++i) t[i] = T{};
      post(t);
      if (lane == 0) {
#pragma unroll
        for (int i = 0; i < NV + NX; ++i) rb.bcast[i] = t[i];
      }
    }
    __syncthreads();
    pull_halos();
#pragma unroll
    for (int i = 0; i < NV + NX; ++i) v[i] = rb.bcast[i];
    phase ^= 1;
  }

  __device__ size_t halo_slot(int set, int block) const {
    return ((size_t)set * kMaxGrid + (size_t)block) * 2 * (size_t)P.g_halo_row_bytes;
  }
  // Publish the own first and last rows (local rows 0 and R-1 of buf, which points at row -1)
  // to this CTA's two global halo slots of the next set; the neighbours pull them after the
  // next barrier.
  template <class T>
  __device__ void push_halos(T* buf, const Slab& sb) {
    const int nb = sb.W * (int)sizeof(T);           // bytes per row, a multiple of 16
    hset ^= 1;
    unsigned char* out = reinterpret_cast<unsigned char*>(P.g_halo) + halo_slot(hset, (int)blockIdx.x);
    const uint4* s0 = reinterpret_cast<const uint4*>(buf + 1 * sb.W);
    const uint4* s1 = reinterpret_cast<const uint4*>(buf + sb.R * sb.W);
    uint4* d0 = reinterpret_cast<uint4*>(out);
    uint4* d1 = reinterpret_cast<uint4*>(out + P.g_halo_row_bytes);
    for (int i = threadIdx.x; i < nb / 16; i += blockDim.x) {
      d0[i] = s0[i];
      d1[i] = s1[i];
    }
    __threadfence();                                // each writer orders its own stores
    pending_lo = reinterpret_cast<unsigned char*>(buf);
    pending_hi = reinterpret_cast<unsigned char*>(buf + (sb.R + 1) * sb.W);
    pending_bytes = nb;
  }
  // 2h-level rows (see ClusterComm::push_halos_rows) through the global halo slots.
  __device__ void push_halos_rows(float* buf, int W1, int R1, int /*R1b*/, int /*rank*/, int /*cs*/) {
    const int nb = W1 * (int)sizeof(float);
    hset ^= 1;
    unsigned char* out = reinterpret_cast<unsigned char*>(P.g_halo) + halo_slot(hset, (int)blockIdx.x);
    const uint4* s0 = reinterpret_cast<const uint4*>(buf + 1 * W1);
    const uint4* s1 = reinterpret_cast<const uint4*>(buf + R1 * W1);
    uint4* d0 = reinterpret_cast<uint4*>(out);
    uint4* d1 = reinterpret_cast<uint4*>(out + P.g_halo_row_bytes);
    for (int i = threadIdx.x; i < nb / 16; i += blockDim.x) {
      d0[i] = s0[i];
      d1[i] = s1[i];
    }
    __threadfence();
    pending_lo = reinterpret_cast<unsigned char*>(buf);
    pending_hi = reinterpret_cast<unsigned char*>(buf + (R1 + 1) * W1);
    pending_bytes = nb;
  }
  template <class T>
  __device__ void exchange(T* buf, const Slab& sb) {
    push_halos(buf, sb);
    sync();
  }
  __device__ void exchange_rows(float* buf, int W1, int R1, int R1b, int rank_, int cs) {
    push_halos_rows(buf, W1, R1, R1b, rank_, cs);
    sync();
  }
  // Edge rows from registers (see ClusterComm::put_edge): into this CTA's slots of the next set.
  __device__ void begin_edges() { hset ^= 1; }
  template <class T>
  __device__ void put_edge(T*, int lr, int col, const T (&v)[4], const Slab& sb) {
    unsigned char* out = reinterpret_cast<unsigned char*>(P.g_halo) + halo_slot(hset, (int)blockIdx.x);
    if (lr == 0) {
      T* d = reinterpret_cast<T*>(out) + col;
#pragma unroll
      for (int j = 0; j < 4; ++j) d[j] = v[j];
    }
    if (lr == sb.R - 1) {
      T* d = reinterpret_cast<T*>(out + P.g_halo_row_bytes) + col;
#pragma unroll
      for (int j = 0; j < 4; ++j) d[j] = v[j];
    }
    __threadfence();                                // each writer orders its own stores
  }
  template <class T>
  __device__ void end_edges(T* edge, const Slab& sb) {
    pending_lo = reinterpret_cast<unsigned char*>(edge);
    pending_hi = reinterpret_cast<unsigned char*>(edge + sb.W);
    pending_bytes = sb.W * (int)sizeof(T);
  }
  // After a barrier: the neighbours' last / first rows into the local halo rows -1 and R.
  __device__ void pull_halos() {
    if (!pending_lo) return;
    const unsigned char* hb = reinterpret_cast<const unsigned char*>(P.g_halo);
    const size_t rb = P.g_halo_row_bytes;
    const int n16 = pending_bytes / 16;
    uint4* lo = reinterpret_cast<uint4*>(pending_lo);   // row -1
    uint4* hi = reinterpret_cast<uint4*>(pending_hi);   // row R
    const int r = rank(), b = (int)blockIdx.x;
    if (r > 0) {
      const uint4* src = reinterpret_cast<const uint4*>(hb + halo_slot(hset, b - 1) + rb);
      for (int i = threadIdx.x; i < n16; i += blockDim.x) lo[i] = __ldcg(src + i);
    }
    if (r < G - 1) {
      const uint4* src = reinterpret_cast<const uint4*>(hb + halo_slot(hset, b + 1));
      for (int i = threadIdx.x; i < n16; i += blockDim.x) hi[i] = __ldcg(src + i);
    }
    pending_lo = pending_hi = nullptr;
    __syncthreads();
  }

  // the partials live in one global array read by every CTA of the group after the barrier
  // (dst is rank-relative; the group's range starts at its first block)
  __device__ void publish_tl(float* /*slot*/, int dst, const float4& chunk, int sub, int /*cs*/) {
    if (sub == 0) {
      *reinterpret_cast<float4*>(P.g_tl + (size_t)base * tl_ncp() + dst) = chunk;
      __threadfence();
    }
  }
  __device__ void finish_edges() { sync(); }
  __device__ void expect_tl(unsigned) {}
  __device__ void finish_tl() { sync(); }
  __device__ void bind(const StepParams&) {}
  __device__ int tl_ncp() const { return coarse_row_stride(P.nax) * P.nay; }
  __device__ const float* tl_slots(const float* /*local*/) const { return P.g_tl + (size_t)base * tl_ncp(); }
  __device__ float4 tl_load4(const float* slots, int idx) const {
    return __ldcg(reinterpret_cast<const float4*>(slots + idx));
  }
};

}  // namespace ptg
