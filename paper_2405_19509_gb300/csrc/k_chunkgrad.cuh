// Chunk gradients (Sec. I): g_{D_i} = sum_{rows r of chunk i} grad l(x_r, y_r, w)
//                                    = X_i^T (f(X_i w) - y01_i),
// f = identity (least squares) or the logistic sigmoid, un-normalised as in
// Sec. I; the loss L = (1/N~) sum_r l(x_r, y_r, w) is fused in.
//
// GB300 design: the path is HBM bound (2 flops per element read), so X is read
// exactly once.  A cluster of CL CTAs owns a contiguous range of rows (a flat
// partition of all N~ rows, so every SM gets the same amount of X); CTA rank q
// of the cluster owns the column slice [q*Wc, (q+1)*Wc).  Rows arrive through
// a ring of S shared-memory stages filled by TMA bulk copies
// (cp.async.bulk, one per row slice, completion on an mbarrier).  For each
// stage of RB rows:
//   pass 1: every thread forms partial dot products of its columns with w;
//           they are reduced across the CTA (warp shuffles + shared memory)
//           and, when CL > 1, across the cluster through distributed shared
//           memory (st.shared::cluster + barrier.cluster);
//   then:   residual r = f(z) - y01 per row (and the loss term);
//   pass 2: acc[col] += r * x[row, col] from the same shared-memory stage.
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
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// Load V elements (16 bytes) of a row slice from shared memory as floats.
template <typename T>
struct Vec;
template <>
struct Vec<float> {
  static constexpr int V = 4;
  __device__ static __forceinline__ void load(const float* p, float (&o)[4]) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  }
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
  __device__ static __forceinline__ void load(const __nv_bfloat16* p, float (&o)[8]) {
    unpack(load_raw(p), o);
  }
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
};

constexpr int kMaxStages = 4;
// DSMEM exchange slots: a peer can run at most ~1.5 batches ahead of this CTA
// (it needs this CTA's sums of batch n + 1 before writing batch n + 4), so
// four slots keep a slot from being rewritten before it is read.
constexpr int kZSlots = 4;
constexpr long long kSpinLimit = 1LL << 31;  // clock cycles (~1 s) per wait

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
  int loss;
  int want_loss;
  long long spin_limit;  // clock cycles a wait may take before the kernel gives up
  int stall;             // failure-path test: the loader issues nothing
  float* parts;        // [clusters][maxt][d]
  double* loss_parts;  // [clusters]
  uint32_t* status;
};

// Arrive on the mbarrier at the same offset in cluster peer `rank`, releasing
// this thread's prior shared::cluster stores to it.
__device__ __forceinline__ void mbar_arrive_remote(uint64_t* bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                   mapa(smem_u32(bar), rank))
               : "memory");
}
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
__device__ __forceinline__ void consumer_sync(int nthreads) {
  asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// Warp sums of R row partials with a halving butterfly: log2(R) exchange
// levels that each halve the vector, then plain xor levels -- 5 + R - 1
// shuffles instead of 5 R.  Lane l ends with the warp sum of row l >> (5 - log2 R).
template <int R>
__device__ __forceinline__ float warp_sum_rows(const float (&p)[R], int lane) {
  constexpr int LR = R >= 4 ? 2 : (R >= 2 ? 1 : 0);
  static_assert((1 << LR) == R, "rows per batch must be 1, 2 or 4");
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

// NT consumer threads (warps 0 .. NW-1) plus one producer warp (warp NW).
template <typename T, bool ALIGNED, int CL, int NT, int NVT, int RBM>
__device__ __forceinline__ void chunkgrad_body(const CGArgs& a) {
  constexpr int V = Vec<T>::V;
  using EL = Elems<T, ALIGNED, NT>;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(128) unsigned char smem[];
  T* stages = reinterpret_cast<T*>(smem);
  const size_t stage_elems = (size_t)RBM * a.ld_s;
  float* red = reinterpret_cast<float*>(smem + a.S * stage_elems * sizeof(T));  // [2][NW][RBM]
  float* zcl = red + 2 * NW * RBM;                                               // [kZSlots][CL][RBM]
  uint64_t* bars = reinterpret_cast<uint64_t*>(zcl + kZSlots * CL * RBM + 2);    // 8-byte aligned
  uint64_t* full = bars;                    // [kMaxStages] data landed
  uint64_t* empty = bars + kMaxStages;      // [kMaxStages] consumers done with the stage
  uint64_t* zfull = bars + 2 * kMaxStages;  // [kZSlots] every peer's partial dots arrived
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 2 * kMaxStages + kZSlots);

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
    for (int z = 0; z < kZSlots; ++z) mbar_init(&zfull[z], CL);
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
  __syncthreads();
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
    for (int n = 0; n < (a.stall ? 0 : nb); ++n) {
      const int s = n % a.S;
      const uint32_t ph = (uint32_t)((n / a.S) & 1);
      const int nr = bi == a.nbc - 1 ? last_rows : RBM;  // rows of this batch
      T* st = stages + s * stage_elems;
      if constexpr (ALIGNED) {
        const bool ok = bounded_wait(&empty[s], ph ^ 1, abort_flag, a.status, a.spin_limit);
        if (!__all_sync(0xffffffffu, ok && !*abort_flag)) break;
        if (lane == 0) {
          const uint32_t row_bytes = (uint32_t)(width * sizeof(T));
          mbar_expect_tx(&full[s], row_bytes * nr);
          for (int r = 0; r < nr; ++r)
            bulk_g2s(st + (size_t)r * a.ld_s, X + (row + r) * a.d + c0, row_bytes, &full[s]);
        }
      } else {
        // Row r's slice starts o elements past a 16-byte boundary.  Its whole
        // 16-byte pieces up to element pt of the stage row arrive by one bulk
        // copy; the 2 V elements from pt on -- the last columns, then zeros
        // over what an earlier row with a larger o may have left there -- are
        // stored by the lanes (read from X before the wait, which hides them).
        const uint32_t e0 = (uint32_t)row * (uint32_t)a.d + (uint32_t)c0 + xo;
        const uint32_t dv = (uint32_t)a.d;
        constexpr int NTL = (RBM * 2 * V + 31) / 32;
        T tv[NTL];
        T* tp[NTL];
#pragma unroll
        for (int k = 0; k < NTL; ++k) {
          const int t = k * 32 + lane, r = t / (2 * V);
          const uint32_t o = (e0 + (uint32_t)r * dv) & (V - 1);
          const int pos = (int)((o + (uint32_t)width) & ~(uint32_t)(V - 1)) + t % (2 * V);
          const int c = pos - (int)o;
          tp[k] = r < nr ? st + (size_t)r * a.ld_s + pos : nullptr;
          tv[k] = T(0.f);
          if (r < nr && c >= 0 && c < width) tv[k] = X[(row + r) * a.d + c0 + c];
        }
        const bool ok = bounded_wait(&empty[s], ph ^ 1, abort_flag, a.status, a.spin_limit);
        if (!__all_sync(0xffffffffu, ok && !*abort_flag)) break;
#pragma unroll
        for (int k = 0; k < NTL; ++k)
          if (tp[k]) *tp[k] = tv[k];
        const uint32_t o = (e0 + (uint32_t)lane * dv) & (V - 1);
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
      }
      issued = n + 1;
      row += nr;
      if (++bi == a.nbc) bi = 0;
    }
    // drain: the CTA must not exit with copies in flight
    if (lane == 0) {
      volatile int no_abort = 0;
      for (int n = max(0, issued - a.S); n < issued; ++n)
        bounded_wait(&full[n % a.S], (uint32_t)((n / a.S) & 1), &no_abort, a.status, kSpinLimit);
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
    double loss_acc = 0.0;
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
      bounded_wait(&full[g.s], g.ph, abort_flag, a.status, a.spin_limit);
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
    // x of a batch copied to registers once (kept from the dot products to pass 2)
    auto load_x = [&](const Ring& g, typename EL::Raw (&xr)[RBM][NVT]) {
      auto src = from_stage(g);
#pragma unroll
      for (int r = 0; r < RBM; ++r)
#pragma unroll
        for (int u = 0; u < NVT; ++u) xr[r][u] = src(r, u);
    };
    // hand a stage back to the producer (every lane of the warp is done reading it)
    auto release = [&](const Ring& g) {
      __syncwarp();
      if (lane == 0) tcw::mbar_arrive(&empty[g.s]);
    };
    // Dot products of batch n, reduced over the CTA (warp butterfly, then
    // lane-parallel over (warp, row) pairs) and, with clusters, sent to every
    // peer.  Returns the CTA sums in every lane.
    auto dots = [&](int n, auto&& xget, float (&z)[RBM]) {
      // two packed partial sums a row (vectors u even / odd), so that the
      // FMA chain of a row is a quarter as long
      float pd[RBM];
#pragma unroll
      for (int r = 0; r < RBM; ++r) {
        float2 p2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int u = 0; u < NVT; ++u) {
          float x[V];
          EL::unpack(xget(r, u), x);
#pragma unroll
          for (int e = 0; e < V2; ++e)
            p2[u & 1] = __ffma2_rn(make_float2(x[2 * e], x[2 * e + 1]), wv[u][e], p2[u & 1]);
        }
        pd[r] = (p2[0].x + p2[0].y) + (p2[1].x + p2[1].y);
      }
      constexpr int kRowShift = 5 - (RBM >= 4 ? 2 : (RBM >= 2 ? 1 : 0));
      const float ws_ = warp_sum_rows<RBM>(pd, lane);
      float* redn = red + (n & 1) * NW * RBM;
      if ((lane & ((1 << kRowShift) - 1)) == 0) redn[warp * RBM + (lane >> kRowShift)] = ws_;
      consumer_sync(NT);
      // CTA sums: the NW x RBM partials are spread over the lanes (entry
      // j*32 + lane is warp (idx % NW) of row idx / NW), summed over aligned
      // groups of NW lanes, then row r is read from the first lane of its group.
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
      if (CL > 1 && tid < CL && !*abort_flag) {
        // thread p writes the CTA sums into peer p's slot and arrives there
        // (release).  After a failed wait the CTA sends no more: a peer then
        // never receives more arrivals in one phase than it expects.
        float* zc = zcl + (n % kZSlots) * CL * RBM;
        const uint32_t peer = (uint32_t)tid;
#pragma unroll
        for (int r = 0; r < RBM; ++r)
          st_cluster_f32(mapa(smem_u32(zc + rank * RBM + r), peer), z[r]);
        mbar_arrive_remote(&zfull[n % kZSlots], peer);
      }
    };
    // Cluster sums of batch n once every peer's CTA sums have arrived: lane
    // p * RBM + r reads peer p's sum of row r, a xor tree adds the peers.
    auto cluster_sums = [&](int n, float (&z)[RBM]) {
      bounded_wait(&zfull[n % kZSlots], (uint32_t)((n / kZSlots) & 1), abort_flag, a.status,
                   a.spin_limit, true);
      const float* zc = zcl + (n % kZSlots) * CL * RBM;
      float t = lane < CL * RBM ? zc[lane] : 0.f;
#pragma unroll
      for (int o = RBM; o < CL * RBM; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
#pragma unroll
      for (int r = 0; r < RBM; ++r) z[r] = __shfl_sync(0xffffffffu, t, r);
    };

    // y of a batch for lane r < its rows, loaded two batches ahead (off the
    // critical path between the dot products and the residuals)
    const float* yp = a.y + r0 + lane;  // row of the batch y is loaded for next
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
    // Residuals, loss and pass 2 (acc += r * x) of the batch at g from its row sums z.
    auto finish = [&](const Ring& g, const float (&z)[RBM], auto&& xget) {
      if (cur < 0 || g.bi == 0) {  // a new chunk (a batch never straddles chunks)
        if (cur >= 0) flush(cur);
#pragma unroll
        for (int u = 0; u < NVT; ++u)
#pragma unroll
          for (int e = 0; e < V2; ++e) acc[u][e] = make_float2(0.f, 0.f);
        cur = cur < 0 ? first_chunk : cur + 1;
      }
      const int nr = g.bi == a.nbc - 1 ? last_rows : RBM;
      const float yv = y0;
      y0 = y1;
      y1 = load_y();
      // ---- residuals: lane r < RBM takes row r, then a broadcast
      float zr = z[0];
#pragma unroll
      for (int r = 1; r < RBM; ++r) zr = lane == r ? z[r] : zr;
      const float mine =
          a.loss == GC_LSQ ? zr - yv : 1.f / (1.f + __expf(-zr)) - 0.5f * (yv + 1.f);
      float res[RBM];
#pragma unroll
      for (int r = 0; r < RBM; ++r) res[r] = __shfl_sync(0xffffffffu, mine, r);
      // ---- the loss: lane r < RB of warp 0 takes row r (fp32), one fp64 add per batch
      if (a.want_loss && rank == 0 && warp == 0) {
        float lr = 0.f;
        if (lane < nr) {
          if (a.loss == GC_LSQ) {
            const float e = zr - yv;
            lr = 0.5f * e * e;
          } else {
            // log(1 + e^t) = max(t, 0) + log(1 + e^-|t|); the fast intrinsics
            // are accurate to ~1e-6 absolute per row here (1 + e^-|t| lies in
            // [1, 2]), far below the loss's 1e-5 relative tolerance, and keep
            // warp 0 from lagging behind the others at every batch
            const float t = -yv * zr;
            lr = fmaxf(t, 0.f) + __logf(1.f + __expf(-fabsf(t)));
          }
        }
#pragma unroll
        for (int o = 2; o > 0; o >>= 1) lr += __shfl_xor_sync(0xffffffffu, lr, o);
        if (lane == 0) loss_acc += (double)lr;
      }
      // ---- pass 2 (rows past nr hold an earlier batch's values: skipped)
      auto add_row = [&](int r) {
        const float2 rr = make_float2(res[r], res[r]);
#pragma unroll
        for (int u = 0; u < NVT; ++u) {
          float x[V];
          EL::unpack(xget(r, u), x);
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

    // x in registers when they fit beside acc and w (fp32 rows; not bf16,
    // whose unpacked vectors would spill)
    constexpr bool kXRegs = NVT * RBM * V <= 32;
    Ring g{0, 0u, bi0, (uint32_t)r0 * (uint32_t)a.d + (uint32_t)c0 + xo};
    if (CL == 1 && kXRegs) {
      // One pass over the stage: x stays in registers from the dot products to
      // pass 2, so the stage goes back to the producer as soon as it is read.
      for (int n = 0; n < nb; ++n, g.next<ALIGNED>(a, RBM)) {
        typename EL::Raw xr[RBM][NVT];
        float z[RBM];
        wait_stage(g);
        load_x(g, xr);
        release(g);
        auto xget = [&](int r, int u) { return xr[r][u]; };
        dots(n, xget, z);
        finish(g, z, xget);
      }
    } else if (CL == 1) {
      for (int n = 0; n < nb; ++n, g.next<ALIGNED>(a, RBM)) {
        float z[RBM];
        wait_stage(g);
        dots(n, from_stage(g), z);
        finish(g, z, from_stage(g));
        release(g);
      }
    } else {
      // Clusters: batch n + 1's dot products and send run before the wait for
      // batch n's cluster sums (software pipelining); pass 2 re-reads the
      // stage, which is handed back afterwards.
      float znext[RBM];
      Ring g1 = g;
      if (nb > 0) {
        wait_stage(g1);
        dots(0, from_stage(g1), znext);
        g1.next<ALIGNED>(a, RBM);
      }
      for (int n = 0; n < nb; ++n, g.next<ALIGNED>(a, RBM), g1.next<ALIGNED>(a, RBM)) {
        if (n + 1 < nb) {
          wait_stage(g1);
          dots(n + 1, from_stage(g1), znext);
        }
        float z[RBM];
        cluster_sums(n, z);
        finish(g, z, from_stage(g));
        release(g);
      }
    }
    // the reduction kernel may be scheduled now (it waits for this grid to
    // finish); not earlier, so that work on other streams keeps the SMs' room
    if (tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (cur >= 0) flush(cur);
    if (tid == 0 && rank == 0) a.loss_parts[q] = loss_acc;
  }
  if (CL > 1) cluster_sync_all();  // no CTA leaves while a peer may still address it
}

template <typename T, bool ALIGNED, int CL, int NT, int NVT, int RBM>
__global__ void __launch_bounds__(NT + 32, 1) k_chunkgrad(CGArgs a) {
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
    if (NT == 256 && NVT == 1) return k_chunkgrad<T, ALIGNED, 1, 256, 1, 4>;
    if (NT == 128 && NVT == 2) return k_chunkgrad<T, ALIGNED, 1, 128, 2, 4>;
    if (NT == 128 && NVT == 1) return k_chunkgrad<T, ALIGNED, 1, 128, 1, 4>;
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
    if constexpr (CL == 4) {
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

}  // namespace cg
}  // namespace gc
