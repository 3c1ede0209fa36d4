// Chunk gradients (Sec. I): g_{D_i} = sum_{rows r of chunk i} grad l(x_r, y_r, w)
//                                    = X_i^T (f(X_i w) - y01_i),
// f = identity (least squares) or the logistic sigmoid, un-normalised as in
// Sec. I; the loss L = (1/N~) sum_r l(x_r, y_r, w) is fused in.
//
// GB300 design: the path is HBM bound (2 flops per element read), so X is read
// exactly once.  A cluster of CL CTAs owns a contiguous range of rows (a flat
// partition of all batches, so every SM gets the same amount of X); CTA rank q
// of the cluster owns the column slice [q*Wc, (q+1)*Wc).  Rows arrive through
// a ring of S shared-memory stages filled by TMA bulk copies
// (cp.async.bulk, one per row slice, completion on an mbarrier).  For each
// batch of RB rows:
//   pass 1: every thread forms partial dot products of its columns with w and
//           leaves x in tensor memory; its warp's sums go to the reducer warp;
//   the reducer warp adds the warps' sums, exchanges them across the cluster
//           when CL > 1 (st.async into distributed shared memory), and
//           publishes the residuals r = f(z) - y01 (and adds the loss terms);
//   pass 2: acc[col] += r * x[row, col], x from tensor memory, two batches
//           behind pass 1.
// What the two separate: a stage is free as soon as its dot products are formed,
// so nearly the whole ring is in flight (tensor memory holds the three batches
// between the passes, 256 KB an SM that the kernel has no other use for), and
// no warp waits at a block barrier or for the exchange.  bf16 d = 65536, 8.6 GB:
// 1.74 ms (73% of the copy rate) with both passes from the stage, a named
// barrier per batch and the exchange by the consumers; 1.74 with x in tensor
// memory alone; 1.29 with the reducer warp, which then spent its time in the
// release fence of the remote arrive; 1.22 with st.async (104%).  fp32 d =
// 16384 .. 65536, 2 GB: 61-77% before, 86-98% now.
// acc lives in registers; when the row range crosses into a new chunk the
// cluster writes its partial chunk gradient to a scratch slot, and a small
// second kernel adds the (at most a few) partials of every chunk in a fixed
// order, so results are deterministic.
//
// Rows whose slices do not all start on a 16-byte boundary (a row length that
// is no multiple of 16 bytes, an unaligned X) take the same kernel with
// ALIGNED = false: a row is copied from the boundary below its start, so it
// lands in its stage row displaced by (start mod 16 bytes), and the threads
// take columns tid, tid + NT, ... one element a load -- consecutive lanes read
// consecutive elements whatever the displacement, so a warp's load is one
// wavefront, as many bytes a wavefront as the 16-byte loads of aligned rows.
//
// A batch is RB = RBM rows of one chunk; the last batch of a chunk has fewer
// when RB does not divide n_c.
#pragma once

#include <type_traits>

#include "gc_internal.cuh"
#include "tc_ptx.cuh"

namespace gc {
namespace cg {

// the CTA-local mbarrier wrappers are the shared ones (tc_ptx.cuh); the
// cluster-scope ones below are this kernel's own
using tcw::mbar_expect_tx;
using tcw::mbar_init;
using tcw::mbar_try_wait;
using tcw::smem_u32;

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(addr), "r"(rank));
  return out;
}
// R floats into a peer's shared memory, counted as 4 R bytes on the peer's
// mbarrier: no fence between the data and the signal (an arrive.release.cluster
// after plain remote stores held the sending warp for over a microsecond).
template <int R>
__device__ __forceinline__ void st_async(uint32_t addr, const float (&z)[R], uint32_t bar) {
  static_assert(R == 1 || R == 2 || R == 4, "rows per batch must be 1, 2 or 4");
  if constexpr (R == 1)
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                     addr),
                 "r"(__float_as_uint(z[0])), "r"(bar)
                 : "memory");
  else if constexpr (R == 2)
    asm volatile(
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(
            addr),
        "r"(__float_as_uint(z[0])), "r"(__float_as_uint(z[1])), "r"(bar)
        : "memory");
  else
    asm volatile(
        "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, "
        "[%5];" ::"r"(addr),
        "r"(__float_as_uint(z[0])), "r"(__float_as_uint(z[1])), "r"(__float_as_uint(z[2])),
        "r"(__float_as_uint(z[R - 1])), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// V elements (16 bytes) of a row slice, as they lie and as floats.
template <typename T>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int V = 4;
  __device__ static __forceinline__ uint4 load_raw(const float* p) {
    return *reinterpret_cast<const uint4*>(p);
  }
  __device__ static __forceinline__ void unpack(const uint4& u, float (&o)[4]) {
    o[0] = __uint_as_float(u.x); o[1] = __uint_as_float(u.y);
    o[2] = __uint_as_float(u.z); o[3] = __uint_as_float(u.w);
  }
};
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int V = 8;
  __device__ static __forceinline__ uint4 load_raw(const __nv_bfloat16* p) {
    return *reinterpret_cast<const uint4*>(p);
  }
  __device__ static __forceinline__ void unpack(const uint4& u, float (&o)[8]) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      o[2 * k] = __uint_as_float(w[k] << 16);
      o[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
  }
};

// V elements of a stage row: one 16-byte vector (aligned rows), or V single
// elements NT apart.
template <typename T, bool ALIGNED, int NT>
struct Elems {
  static constexpr int V = Vec<T>::V;
  using Raw = uint4;
  __device__ static __forceinline__ Raw load(const T* p) { return Vec<T>::load_raw(p); }
  __device__ static __forceinline__ void unpack(const Raw& r, float (&o)[V]) {
    Vec<T>::unpack(r, o);
  }
  __device__ static __forceinline__ uint4 words(const Raw& r) { return r; }
};
template <typename T, int NT>
struct Elems<T, false, NT> {
  static constexpr int V = Vec<T>::V;
  struct Raw {
    float f[V];
  };
  __device__ static __forceinline__ Raw load(const T* p) {
    Raw r;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      if constexpr (sizeof(T) == 4)
        r.f[e] = p[e * NT];
      else
        r.f[e] = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(p)[e * NT] << 16);
    }
    return r;
  }
  __device__ static __forceinline__ void unpack(const Raw& r, float (&o)[V]) {
#pragma unroll
    for (int e = 0; e < V; ++e) o[e] = r.f[e];
  }
  // the 16 bytes they came from
  __device__ static __forceinline__ uint4 words(const Raw& r) {
    auto bits = [&](int e) { return __float_as_uint(r.f[e]); };
    if constexpr (sizeof(T) == 4) {
      return make_uint4(bits(0), bits(1), bits(2), bits(3));
    } else {
      auto two = [&](int e) { return (bits(e) >> 16) | bits(e + 1); };
      return make_uint4(two(0), two(2), two(4), two(6));
    }
  }
};

constexpr int kMaxStages = 4;
// Pass 1 of batch n + kAhead runs before pass 2 of batch n, which leaves the
// reducer (and a cluster's exchange) two batches' time.
constexpr int kAhead = 2;
// Slots of the warps' partial dots and of the residuals, by batch.  A consumer
// warp that writes its partials of batch m has taken the residuals of batch
// m - kAhead - 1, so the reducer has read the partials up to m - kAhead; the
// reducer publishes the residuals of batch n after every warp's partials of
// batch n or later, which follow pass 2 of batch n - kAhead - 1.
constexpr int kSlots = kAhead + 2;
// DSMEM exchange slots.  A peer's reducer sends batch n after it has all sums of
// batch n - 2, so this CTA has sent n - 2, having read the sums up to n - 4.
constexpr int kZSlots = 8;
// Tensor memory as the place of x between the two passes: a batch is at most 32
// words a thread, one word a lane in 32 columns of its warp's lane quarter;
// batches n .. n + kAhead are held.
constexpr int kParkBatches = 4;
constexpr int kParkCols = 32 * kParkBatches;  // columns a warp
static_assert(kParkBatches > kAhead && kSlots > kAhead + 1, "slots");

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint4& v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(v.x),
               "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint4 tmem_ld4(uint32_t taddr) {
  uint4 v;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(taddr)
               : "memory");
  return v;
}
// The values of loads issued before this are complete after it.
template <int N>
__device__ __forceinline__ void tmem_wait_ld(uint4 (&v)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < N; ++k)  // no use of the values moves above the wait
    asm volatile("" : "+r"(v[k].x), "+r"(v[k].y), "+r"(v[k].z), "+r"(v[k].w)::"memory");
}
constexpr long long kSpinLimit = 1LL << 31;  // clock cycles (~1 s) per wait
constexpr long long kLandCycles = 1LL << 17;  // ~70 us, far above a remote store's latency

struct CGArgs {
  const void* X;
  const float* y;
  const float* w;
  int d;          // row length (elements)
  int Wc;         // columns per CTA slice (multiple of V)
  int ld_s;       // shared-memory row stride of a stage (elements, multiple of V)
  int n_c;        // rows per chunk
  long long Ntil; // rows
  int nbc;        // batches per chunk: ceil(n_c / RBM)
  long long nbatch;  // batches in all: chunks * nbc
  long long bpc;  // batches per cluster
  int S;          // stages
  int maxt;       // chunk slots per cluster in `parts`
  int by_warp;    // short rows: a range of batches is a warp's, not a block's
  int loss;
  int want_loss;
  long long spin_limit;  // clock cycles a wait may take before the kernel gives up
  int stall;             // failure-path test: the loader issues nothing
  float* parts;        // [clusters][maxt][d]
  double* loss_parts;  // [clusters]
  uint32_t* status;
};

__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; `cl` selects cluster-scope acquire (remote arrivals).
__device__ __forceinline__ bool bounded_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                             uint32_t* status, long long limit, bool cl = false) {
  auto tw = [&]() { return cl ? mbar_try_wait_cluster(bar, parity) : mbar_try_wait(bar, parity); };
  if (tw()) return true;
  const long long t0 = clock64();
  while (!tw()) {
    if (*abort_flag) return false;
    if (clock64() - t0 > limit) {
      atomicOr(status, ST_TIMEOUT);
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}
// A warp's bounded wait: every lane waits, then the warp goes on together.
__device__ __forceinline__ void warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          uint32_t* status, long long limit, bool cl = false) {
  bounded_wait(bar, parity, abort_flag, status, limit, cl);
  __syncwarp();
}

// Warp sums of R row partials with a halving butterfly: log2(R) exchange
// levels that each halve the vector, then plain xor levels -- 5 + R - 1
// shuffles instead of 5 R.  Lane l ends with the warp sum of row l >> (5 - log2 R).
template <int R>
__device__ __forceinline__ float warp_sum_rows(const float (&p)[R], int lane) {
  constexpr int LR = R >= 16 ? 4 : R >= 8 ? 3 : (R >= 4 ? 2 : (R >= 2 ? 1 : 0));
  static_assert((1 << LR) == R, "rows per batch must be a power of two up to 16");
  float v[R];
#pragma unroll
  for (int j = 0; j < R; ++j) v[j] = p[j];
#pragma unroll
  for (int lvl = 0; lvl < LR; ++lvl) {
    const int off = 16 >> lvl;
    const int half = R >> (lvl + 1);
    const bool hi = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < half; ++j) {
      const float keep = hi ? v[half + j] : v[j];
      const float send = hi ? v[j] : v[half + j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (int lvl = LR; lvl < 5; ++lvl) v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16 >> lvl);
  return v[0];
}

// Position in the sequence of batches: the ring stage and the parity of its
// phase, the batch's index within its chunk and the low bits of its first
// row's element index (only its remainder mod V is used).
struct Ring {
  int s;
  uint32_t ph;
  int bi;
  uint32_t e0;
  template <bool ALIGNED>
  __device__ __forceinline__ void next(const CGArgs& a, int RB) {
    if (++s == a.S) {
      s = 0;
      ph ^= 1u;
    }
    const bool wrap = ++bi == a.nbc;
    if (!ALIGNED) e0 += (uint32_t)(wrap ? a.n_c - (a.nbc - 1) * RB : RB) * (uint32_t)a.d;
    if (wrap) bi = 0;
  }
};

// NT consumer threads (warps 0 .. NW-1), a producer warp (warp NW) and a reducer
// warp (warp NW + 1).
template <typename T, bool ALIGNED, int CL, int NT, int NVT, int RBM>
__device__ __forceinline__ void chunkgrad_body(const CGArgs& a) {
  constexpr int V = Vec<T>::V;
  using EL = Elems<T, ALIGNED, NT>;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(128) unsigned char smem[];
  T* stages = reinterpret_cast<T*>(smem);
  const size_t stage_elems = (size_t)RBM * a.ld_s;
  float* red = reinterpret_cast<float*>(smem + a.S * stage_elems * sizeof(T));  // [kSlots][NW][RBM]
  float* zcl = red + kSlots * NW * RBM;                                         // [kZSlots][CL][RBM]
  float* resid = zcl + kZSlots * CL * RBM;                                      // [kSlots][RBM]
  uint64_t* bars = reinterpret_cast<uint64_t*>(resid + kSlots * RBM);           // 16-byte aligned
  uint64_t* full = bars;                    // [kMaxStages] data landed
  uint64_t* empty = full + kMaxStages;      // [kMaxStages] consumers done with the stage
  uint64_t* part = empty + kMaxStages;      // [kSlots] every warp's partial dots written
  uint64_t* ready = part + kSlots;          // [kSlots] residuals written
  uint64_t* zfull = ready + kSlots;         // [kZSlots] every peer's partial dots arrived
  volatile int* abort_flag = reinterpret_cast<volatile int*>(zfull + kZSlots);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(zfull + kZSlots) + 1;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = CL > 1 ? (int)cluster_rank() : 0;
  const long long q = blockIdx.x / CL;
  const long long g0 = q * a.bpc;  // first batch
  const int nb = (int)max(0LL, min(a.bpc, a.nbatch - g0));
  const long long first_chunk = g0 / a.nbc;
  const int bi0 = (int)(g0 - first_chunk * a.nbc);
  const long long r0 = first_chunk * a.n_c + (long long)bi0 * RBM;  // first row
  const int last_rows = a.n_c - (a.nbc - 1) * RBM;  // rows of a chunk's last batch
  const int c0 = rank * a.Wc;
  const int width = min(a.Wc, a.d - c0);  // columns of this CTA's slice
  const T* X = static_cast<const T*>(a.X);
  // column of element e of vector u of this thread, within the slice
  auto col_of = [&](int u, int e) {
    return ALIGNED ? (tid + u * NT) * V + e : (u * V + e) * NT + tid;
  };
  // elements between the 16-byte boundary below X and X
  const uint32_t xo = ALIGNED ? 0u : (uint32_t)((reinterpret_cast<uintptr_t>(X) & 15) / sizeof(T));

  if (tid == 0) {
    *abort_flag = 0;
    for (int s = 0; s < a.S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], NW);
    }
    for (int z = 0; z < kSlots; ++z) {
      mbar_init(&part[z], NW);
      mbar_init(&ready[z], 1);
    }
    for (int z = 0; z < kZSlots; ++z) mbar_init(&zfull[z], 1);
    fence_mbar_init();
  }
  {
    // Stage bytes the producer never writes are zeroed once, so that the
    // consumers read whole stage rows without masks (zeros add nothing to
    // either pass): with aligned rows the vectors past the slice; otherwise
    // everything, and the producer rewrites the ragged end of every row.
    const int vpr = a.ld_s / V;  // 16-byte vectors per stage row
    const int vfrom = ALIGNED ? width / V : 0;
    for (int s = 0; s < a.S; ++s) {
      uint4* st = reinterpret_cast<uint4*>(stages + (size_t)s * stage_elems);
      for (int r = 0; r < RBM; ++r)
        for (int v = vfrom + tid; v < vpr; v += blockDim.x)
          st[(size_t)r * vpr + v] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (!ALIGNED) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  constexpr uint32_t kTmemCols = NW / 4 * kParkCols;  // 1, 2 or 4 warps a lane quarter: 128, 256, 512
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_holder)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcw::fence_before();
  __syncthreads();
  tcw::fence_after();
  const uint32_t tmem_base = *tmem_holder;
  if (CL > 1) cluster_sync_all();  // every peer has started and initialised its barriers

  if (warp == NW) {
    // ------------------------------------------------------------ producer warp
    // A batch is issued only while no wait has failed: then every earlier
    // batch of the stage has landed (its consumers' waits succeeded), so each
    // stage holds at most one copy in flight and the phases stay in order.
    // The decision is warp-uniform.
    int issued = 0;
    long long row = r0;
    int bi = bi0;
    const int nbs = a.stall ? 0 : nb;
    auto rows_at = [&](int k) { return k == a.nbc - 1 ? last_rows : RBM; };  // rows of batch k of a chunk
    // the stage of batch n is free
    auto stage_free = [&](int n) {
      const bool ok = bounded_wait(&empty[n % a.S], (uint32_t)((n / a.S) & 1) ^ 1, abort_flag, a.status,
                                   a.spin_limit);
      return (bool)__all_sync(0xffffffffu, ok && !*abort_flag);
    };
    if constexpr (ALIGNED) {
      for (int n = 0; n < nbs; ++n) {
        const int s = n % a.S, nr = rows_at(bi);
        if (!stage_free(n)) break;
        if (lane == 0) {
          T* st = stages + s * stage_elems;
          const uint32_t row_bytes = (uint32_t)(width * sizeof(T));
          mbar_expect_tx(&full[s], row_bytes * nr);
          for (int r = 0; r < nr; ++r)
            bulk_g2s(st + (size_t)r * a.ld_s, X + (row + r) * a.d + c0, row_bytes, &full[s]);
        }
        issued = n + 1;
        row += nr;
        if (++bi == a.nbc) bi = 0;
      }
    } else {
      // Row r's slice starts o elements past a 16-byte boundary.  Its whole
      // 16-byte pieces up to element pt of the stage row arrive by one bulk copy;
      // the 2 V elements from pt on -- the last columns, then zeros over what an
      // earlier row with a larger o may have left there -- are stored by the
      // lanes, read from X one batch ahead.
      constexpr int NTL = (RBM * 2 * V + 31) / 32;
      struct Tail {
        T v[NTL];
        int pos[NTL];  // in the stage, -1: none
      };
      const uint32_t dv = (uint32_t)a.d;
      auto load_tail = [&](long long row, int nr, Tail& t) {
        const uint32_t e0 = (uint32_t)row * dv + (uint32_t)c0 + xo;
#pragma unroll
        for (int k = 0; k < NTL; ++k) {
          const int i = k * 32 + lane, r = i / (2 * V);
          const uint32_t o = (e0 + (uint32_t)r * dv) & (V - 1);
          const int pos = (int)((o + (uint32_t)width) & ~(uint32_t)(V - 1)) + i % (2 * V);
          const int c = pos - (int)o;
          t.pos[k] = r < nr ? r * a.ld_s + pos : -1;
          t.v[k] = T(0.f);
          if (r < nr && c >= 0 && c < width) t.v[k] = X[(row + r) * a.d + c0 + c];
        }
      };
      // issue batch n, whose tail is `cur`; load the next one's
      auto issue = [&](int n, const Tail& cur, Tail& next) {
        const int s = n % a.S, nr = rows_at(bi);
        const int nbi = bi + 1 == a.nbc ? 0 : bi + 1;
        if (n + 1 < nbs) load_tail(row + nr, rows_at(nbi), next);
        if (!stage_free(n)) return false;
        T* st = stages + s * stage_elems;
#pragma unroll
        for (int k = 0; k < NTL; ++k)
          if (cur.pos[k] >= 0) st[cur.pos[k]] = cur.v[k];
        const uint32_t o =
            ((uint32_t)row * dv + (uint32_t)c0 + xo + (uint32_t)lane * dv) & (V - 1);
        const T* src = X + (row + lane) * a.d + c0 - o;  // 16-byte aligned
        T* dst = st + (size_t)lane * a.ld_s;
        uint32_t pt = lane < nr ? (o + (uint32_t)width) & ~(uint32_t)(V - 1) : 0u;
        if (lane < nr && pt > 0 && src < X) {
          // rows in the first 16 bytes of an unaligned X: the piece that begins
          // before X is read element by element
          for (int c = 0; c < (int)(V - o) && c < width; ++c) dst[o + c] = src[o + c];
          src += V;
          dst += V;
          pt -= V;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        const uint32_t bytes = pt * (uint32_t)sizeof(T);
        const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);  // orders the stores, too
        __syncwarp();
        if (lane == 0) mbar_expect_tx(&full[s], total);
        __syncwarp();
        if (bytes > 0) bulk_g2s(dst, src, bytes, &full[s]);
        issued = n + 1;
        row += nr;
        bi = nbi;
        return true;
      };
      Tail t0, t1;
      if (nbs > 0) load_tail(row, rows_at(bi), t0);
      for (int n = 0; n < nbs; n += 2) {
        if (!issue(n, t0, t1)) break;
        if (n + 1 < nbs && !issue(n + 1, t1, t0)) break;
      }
    }
    // drain: the CTA must not exit with copies in flight
    if (lane == 0) {
      volatile int no_abort = 0;
      for (int n = max(0, issued - a.S); n < issued; ++n)
        bounded_wait(&full[n % a.S], (uint32_t)((n / a.S) & 1), &no_abort, a.status, kSpinLimit);
    }
  } else if (warp == NW + 1) {
    // ------------------------------------------------------------ reducer warp
    // Per batch: the CTA's sums of the warps' partial dots, with clusters their
    // exchange, the residuals and the loss; none of it in the consumers' way.
    double loss_acc = 0.0;
    // y of the next batches for lane r < their rows
    const float* yp = a.y + r0 + lane;
    int ybi = bi0, yleft = nb;
    auto load_y = [&]() {
      const int nr = ybi == a.nbc - 1 ? last_rows : RBM;
      const float v = (lane < nr && yleft > 0) ? __ldg(yp) : 0.f;
      yp += nr;
      --yleft;
      if (++ybi == a.nbc) ybi = 0;
      return v;
    };
    float y0 = load_y(), y1 = load_y();
    int bi = bi0;
    // CTA sums of batch n, in every lane: the NW x RBM partials are spread over
    // the lanes (entry j*32 + lane is warp idx % NW of row idx / NW), summed over
    // aligned groups of NW lanes, then row r is read from the first of its group.
    auto cta_sums = [&](int n, float (&z)[RBM]) {
      warp_wait(&part[n % kSlots], (uint32_t)((n / kSlots) & 1), abort_flag, a.status, a.spin_limit);
      const float* redn = red + (n % kSlots) * NW * RBM;
      constexpr int E = NW * RBM, NCH = (E + 31) / 32;
      float cs[NCH];
#pragma unroll
      for (int j = 0; j < NCH; ++j) {
        const int idx = j * 32 + lane;
        float t = idx < E ? redn[(idx % NW) * RBM + idx / NW] : 0.f;
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        cs[j] = t;
      }
#pragma unroll
      for (int r = 0; r < RBM; ++r) z[r] = __shfl_sync(0xffffffffu, cs[(r * NW) / 32], (r * NW) % 32);
    };
    // Lane p writes the CTA's sums into peer p's slot; the slot's barrier waits for
    // all peers' bytes.  After a failed wait the CTA sends no more: a peer then
    // never receives more bytes in one phase than it expects.
    auto send = [&](int n, const float (&z)[RBM]) {
      uint64_t* bar = &zfull[n % kZSlots];
      float* mine = zcl + (n % kZSlots) * CL * RBM + rank * RBM;
      if (lane == 0) mbar_expect_tx(bar, CL * RBM * (uint32_t)sizeof(float));
      if constexpr (CL > 1)
        if (lane < CL && !*abort_flag)
          st_async<RBM>(mapa(smem_u32(mine), (uint32_t)lane), z, mapa(smem_u32(bar), (uint32_t)lane));
    };
    // Cluster sums of batch n once every peer's have arrived: lane p * RBM + r
    // reads peer p's sum of row r, a xor tree adds the peers.
    auto cluster_sums = [&](int n, float (&z)[RBM]) {
      warp_wait(&zfull[n % kZSlots], (uint32_t)((n / kZSlots) & 1), abort_flag, a.status,
                a.spin_limit, true);
      const float* zc = zcl + (n % kZSlots) * CL * RBM;
      float t = lane < CL * RBM ? zc[lane] : 0.f;
#pragma unroll
      for (int o = RBM; o < CL * RBM; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
#pragma unroll
      for (int r = 0; r < RBM; ++r) z[r] = __shfl_sync(0xffffffffu, t, r);
    };
    // Residuals of batch n from its row sums (lane r takes row r), and the loss.
    auto publish = [&](int n, const float (&z)[RBM]) {
      const int nr = bi == a.nbc - 1 ? last_rows : RBM;
      if (++bi == a.nbc) bi = 0;
      const float yv = y0;
      y0 = y1;
      y1 = load_y();
      float zr = z[0];
#pragma unroll
      for (int r = 1; r < RBM; ++r) zr = lane == r ? z[r] : zr;
      const float mine =
          a.loss == GC_LSQ ? zr - yv : 1.f / (1.f + __expf(-zr)) - 0.5f * (yv + 1.f);
      if (lane < RBM) resid[(n % kSlots) * RBM + lane] = mine;
      __syncwarp();
      if (lane == 0) tcw::mbar_arrive(&ready[n % kSlots]);
      // ---- the loss: lane r adds its rows in fp64
      if (a.want_loss && rank == 0) {
        float lr = 0.f;
        if (lane < nr) {
          if (a.loss == GC_LSQ) {
            const float e = zr - yv;
            lr = 0.5f * e * e;
          } else {
            // log(1 + e^t) = max(t, 0) + log(1 + e^-|t|); the fast intrinsics
            // are accurate to ~1e-6 absolute per row here (1 + e^-|t| lies in
            // [1, 2]), far below the loss's 1e-5 relative tolerance
            const float t = -yv * zr;
            lr = fmaxf(t, 0.f) + __logf(1.f + __expf(-fabsf(t)));
          }
        }
        loss_acc += (double)lr;
      }
    };
    for (int n = 0; n < nb; ++n) {
      float z[RBM];
      cta_sums(n, z);
      if constexpr (CL == 1) {
        publish(n, z);
      } else {
        send(n, z);
        // the sums of the batch before have had this one's time to arrive
        if (n > 0) {
          cluster_sums(n - 1, z);
          publish(n - 1, z);
        }
      }
    }
    if (CL > 1 && nb > 0) {
      float z[RBM];
      cluster_sums(nb - 1, z);
      publish(nb - 1, z);
    }
    if (a.want_loss && rank == 0) {
#pragma unroll
      for (int o = RBM / 2; o > 0; o >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
      if (lane == 0) a.loss_parts[q] = loss_acc;
    }
  } else {
    // ------------------------------------------------------------ consumer warps
    // w and the gradient accumulators as column pairs: the passes use packed
    // two-wide FMAs (__ffma2_rn, the rounding of two fmaf)
    constexpr int V2 = V / 2;
    float2 wv[NVT][V2];
#pragma unroll
    for (int u = 0; u < NVT; ++u) {
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const int c = col_of(u, e);
        const float wc = c < width ? a.w[c0 + c] : 0.f;
        if (e & 1)
          wv[u][e >> 1].y = wc;
        else
          wv[u][e >> 1].x = wc;
      }
    }
    float2 acc[NVT][V2];
#pragma unroll
    for (int u = 0; u < NVT; ++u)
#pragma unroll
      for (int e = 0; e < V2; ++e) acc[u][e] = make_float2(0.f, 0.f);
    long long cur = -1;     // chunk whose gradient acc holds
    auto flush = [&](long long chunk) {
      float* dst = a.parts + ((size_t)q * a.maxt + (size_t)(chunk - first_chunk)) * a.d;
#pragma unroll
      for (int u = 0; u < NVT; ++u) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const int c = col_of(u, e);
          if (c < width) dst[c0 + c] = (e & 1) ? acc[u][e >> 1].y : acc[u][e >> 1].x;
        }
      }
    };

    // Stage access.  Every stage row is NVT * NT vectors long and the parts
    // the producer never writes are zero, so the reads need no masks.
    auto wait_stage = [&](const Ring& g) {
      warp_wait(&full[g.s], g.ph, abort_flag, a.status, a.spin_limit);
    };
    auto from_stage = [&](const Ring& g) {
      const T* st = stages + (size_t)g.s * stage_elems + (ALIGNED ? tid * V : tid);
      const int ld = a.ld_s;
      if constexpr (ALIGNED) {
        return [=](int r, int u) { return EL::load(st + r * ld + u * NT * V); };
      } else {
        const uint32_t o0 = g.e0, dv = (uint32_t)a.d;
        return [=](int r, int u) {
          return EL::load(st + r * ld + ((o0 + (uint32_t)r * dv) & (V - 1)) + u * NT * V);
        };
      }
    };
    // hand a stage back to the producer (every lane of the warp is done reading it)
    auto release = [&](const Ring& g) {
      __syncwarp();
      if (lane == 0) tcw::mbar_arrive(&empty[g.s]);
    };
    const uint32_t park0 =
        tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * kParkCols);
    auto park_slot = [&](int n) { return park0 + (uint32_t)(n % kParkBatches) * 32u; };
    // Pass 1 of the batch at g: its dot products, reduced over the warp and left
    // for the reducer.  x waits for pass 2 in tensor memory, so that the stage
    // goes back to the producer at once (held until pass 2, one of a cluster's
    // three stages was left to be in flight).
    auto pass1 = [&](int n, const Ring& g) {
      const uint32_t at = park_slot(n);
      wait_stage(g);  // ends converged, as the warp-collective tensor-memory instructions need
      auto xget = from_stage(g);
      // two packed partial sums a row (vectors u even / odd), so that the
      // FMA chain of a row is a quarter as long
      float pd[RBM];
#pragma unroll
      for (int r = 0; r < RBM; ++r) {
        float2 p2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int u = 0; u < NVT; ++u) {
          float x[V];
          const typename EL::Raw raw = xget(r, u);
          tmem_st4(at + (uint32_t)((r * NVT + u) * 4), EL::words(raw));
          EL::unpack(raw, x);
#pragma unroll
          for (int e = 0; e < V2; ++e)
            p2[u & 1] = __ffma2_rn(make_float2(x[2 * e], x[2 * e + 1]), wv[u][e], p2[u & 1]);
        }
        pd[r] = (p2[0].x + p2[0].y) + (p2[1].x + p2[1].y);
      }
      release(g);
      __syncwarp();
      tmem_wait_st();
      constexpr int kRowShift = 5 - (RBM >= 8 ? 3 : (RBM >= 4 ? 2 : (RBM >= 2 ? 1 : 0)));
      const float ws_ = warp_sum_rows<RBM>(pd, lane);
      if ((lane & ((1 << kRowShift) - 1)) == 0)
        red[((n % kSlots) * NW + warp) * RBM + (lane >> kRowShift)] = ws_;
      __syncwarp();
      if (lane == 0) tcw::mbar_arrive(&part[n % kSlots]);
    };
    // Pass 2 (acc += r * x) of the batch at g.
    auto pass2 = [&](int n, const Ring& g) {
      if (cur < 0 || g.bi == 0) {  // a new chunk (a batch never straddles chunks)
        if (cur >= 0) flush(cur);
#pragma unroll
        for (int u = 0; u < NVT; ++u)
#pragma unroll
          for (int e = 0; e < V2; ++e) acc[u][e] = make_float2(0.f, 0.f);
        cur = cur < 0 ? first_chunk : cur + 1;
      }
      const int nr = g.bi == a.nbc - 1 ? last_rows : RBM;
      const uint32_t at = park_slot(n);
      warp_wait(&ready[n % kSlots], (uint32_t)((n / kSlots) & 1), abort_flag, a.status, a.spin_limit);
      float res[RBM];
#pragma unroll
      for (int r = 0; r < RBM; ++r) res[r] = resid[(n % kSlots) * RBM + r];
      // rows past nr hold an earlier batch's values: skipped
      auto add_row = [&](int r) {
        uint4 xr[NVT];
#pragma unroll
        for (int u = 0; u < NVT; ++u) xr[u] = tmem_ld4(at + (uint32_t)((r * NVT + u) * 4));
        tmem_wait_ld(xr);
        const float2 rr = make_float2(res[r], res[r]);
#pragma unroll
        for (int u = 0; u < NVT; ++u) {
          float x[V];
          Vec<T>::unpack(xr[u], x);
#pragma unroll
          for (int e = 0; e < V2; ++e)
            acc[u][e] = __ffma2_rn(rr, make_float2(x[2 * e], x[2 * e + 1]), acc[u][e]);
        }
      };
      if (nr == RBM) {
#pragma unroll
        for (int r = 0; r < RBM; ++r) add_row(r);
      } else {
#pragma unroll
        for (int r = 0; r < RBM - 1; ++r)
          if (r < nr) add_row(r);
      }
    };

    Ring g{0, 0u, bi0, (uint32_t)r0 * (uint32_t)a.d + (uint32_t)c0 + xo};
    Ring g1 = g;
    for (int n = 0; n < min(kAhead, nb); ++n, g1.next<ALIGNED>(a, RBM)) pass1(n, g1);
    for (int n = 0; n < nb; ++n, g.next<ALIGNED>(a, RBM)) {
      if (n + kAhead < nb) {
        pass1(n + kAhead, g1);
        g1.next<ALIGNED>(a, RBM);
      }
      pass2(n, g);
    }
    // the reduction kernel may be scheduled now (it waits for this grid to
    // finish); not earlier, so that work on other streams keeps the SMs' room
    if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (cur >= 0) flush(cur);
  }
  tcw::fence_before();
  if (CL > 1)
    cluster_sync_all();  // no CTA leaves while a peer may still address it
  else
    __syncthreads();
  tcw::fence_after();
  if (CL > 1 && *abort_flag) {
    // after a failed wait sums that peers sent before the barrier may still be
    // on their way into this CTA's shared memory: let them land
    for (const long long t0 = clock64(); clock64() - t0 < kLandCycles;) {
    }
  }
  __syncwarp();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(kTmemCols)
                 : "memory");
}

template <typename T, bool ALIGNED, int CL, int NT, int NVT, int RBM>
__global__ void __launch_bounds__(NT + 64, 1) k_chunkgrad(CGArgs a) {
  chunkgrad_body<T, ALIGNED, CL, NT, NVT, RBM>(a);
}

using Kernel = void (*)(CGArgs);

// The instance for a shape, null when it is not built: the shapes that the
// host's choice of slices (make_plan) leads to.
template <typename T, bool ALIGNED, int CL>
Kernel pick_shape(int NT, int NVT) {
  constexpr bool kF32 = std::is_same<T, float>::value;
  if constexpr (CL == 1) {
    if (NT == 512 && NVT == 2) return k_chunkgrad<T, ALIGNED, 1, 512, 2, 4>;
    if (NT == 256 && NVT == 4) return k_chunkgrad<T, ALIGNED, 1, 256, 4, 2>;
    if (NT == 256 && NVT == 2) return k_chunkgrad<T, ALIGNED, 1, 256, 2, 4>;
    if (NT == 256 && NVT == 1) return k_chunkgrad<T, ALIGNED, 1, 256, 1, 8>;
    if (NT == 128 && NVT == 2) return k_chunkgrad<T, ALIGNED, 1, 128, 2, 4>;
    if constexpr (!kF32)
      if (NT == 128 && NVT == 1) return k_chunkgrad<T, ALIGNED, 1, 128, 1, 8>;
  }
  if constexpr (kF32 ? CL <= 4 : CL != 2)
    if (NT == 512 && NVT == 4) return k_chunkgrad<T, ALIGNED, CL, 512, 4, 2>;
  if constexpr (kF32) {
    if (NT == 512 && NVT == 5) return k_chunkgrad<T, ALIGNED, CL, 512, 5, 1>;
    if (NT == 512 && NVT == 6) return k_chunkgrad<T, ALIGNED, CL, 512, 6, 1>;
    if constexpr (CL >= 4)
      if (NT == 512 && NVT == 8) return k_chunkgrad<T, ALIGNED, CL, 512, 8, 1>;
  } else {
    if (NT == 512 && NVT == 3) return k_chunkgrad<T, ALIGNED, CL, 512, 3, 2>;
    if constexpr (CL == 2 || CL == 4) {
      if (NT == 512 && NVT == 2) return k_chunkgrad<T, ALIGNED, CL, 512, 2, 4>;
      if (NT == 256 && NVT == 4) return k_chunkgrad<T, ALIGNED, CL, 256, 4, 2>;
    }
  }
  return nullptr;
}
template <typename T, bool ALIGNED>
Kernel pick_cl(int CL, int NT, int NVT) {
  switch (CL) {
    case 1: return pick_shape<T, ALIGNED, 1>(NT, NVT);
    case 2: return pick_shape<T, ALIGNED, 2>(NT, NVT);
    case 4: return pick_shape<T, ALIGNED, 4>(NT, NVT);
    case 8: return pick_shape<T, ALIGNED, 8>(NT, NVT);
    default: return nullptr;
  }
}
// one translation unit each (they compile side by side)
Kernel pick_f32(int CL, int NT, int NVT);
Kernel pick_f32_ragged(int CL, int NT, int NVT);
Kernel pick_bf16(int CL, int NT, int NVT);
Kernel pick_bf16_ragged(int CL, int NT, int NVT);
// rows of at most 32 K vectors, a warp a row (k_chunkgrad_short.cu); four vectors of
// bf16 a lane do not fit the registers (d = 1000: 81% of the copy rate against the
// ring kernel's 75% at 2 GB, but 256 chunks of 16 rows 15 us against 9)
constexpr int short_vecs(bool bf16) { return bf16 ? 96 : 128; }
constexpr int kShortThreads = 256;
// rows a batch: 16 vectors a lane (half of that for bf16, whose unpacked values
// would not fit the registers)
constexpr int short_rows(int K, bool bf16) { return (K == 1 ? 16 : (K == 2 ? 8 : 4)) >> (bf16 ? 1 : 0); }
Kernel pick_short(bool bf16, bool aligned, int K);

}  // namespace cg
}  // namespace gc
