// Chunk gradients of short rows (at most 512 fp32 or 768 bf16 columns).
//
// In the ring kernel a batch of such rows is a few KB, and its chain -- copy,
// partial dots of every warp, reducer, residuals -- outlasts the copy by far.
// Here a warp takes whole rows: a lane holds K vectors of w, of the accumulators
// and of RB rows of x, loaded straight from global memory; the dots of the RB rows
// are summed by one halving butterfly, a row's residual is formed by its lanes and
// broadcast, and x is still in registers for the second pass.  No shared memory,
// barrier or other warp is in a row's way; 16 warps an SM with RB rows each keep
// the loads in flight.  The warps of a block take the batches of its range in turn
// and meet once per chunk to add their partial gradients (in warp order) for the
// reduction that follows, which is the ring kernel's; with few batches a chunk each
// warp has a range and a partial gradient of its own.
//
// Bound by HBM from about 100 fp32 columns on, below that by the bytes that RB rows
// a warp have in flight, ragged bf16 by its instructions.  Share of the copy rate at
// 2 GB, ring kernel -> here: fp32 d = 64 14% -> 74%, 301 46 -> 95, 512 82 -> 104;
// bf16 d = 64 5% -> 27%, 501 28 -> 54, 504 39 -> 94.  256 chunks of 4 rows 7.3 ->
// 5.3 us, of 70 rows (fp32 d = 512) 12.6 -> 9.7; 20000 chunks of one row 85 -> 56.
#include "k_chunkgrad.cuh"

namespace gc {
namespace cg {

constexpr int kShortWarps = kShortThreads / 32;

// Column of element e of a lane's vector u: V together when the row is aligned, else
// as 4-byte words 32 lanes apart.
template <typename T, bool ALIGNED>
__device__ __forceinline__ int short_col(int u, int e, int lane) {
  constexpr int V = Vec<T>::V, E = sizeof(T) == 4 ? 1 : 2;  // elements a word
  return ALIGNED ? (lane + 32 * u) * V + e : ((u * 4 + e / E) * 32 + lane) * E + e % E;
}

// One 16-byte piece of a row, zero past d.  Ragged bf16 one element at a time: the
// first and the last rows of X alone take this form.
template <typename T, bool ALIGNED>
__device__ __forceinline__ uint4 short_load(const T* __restrict__ row, int u, int lane, int d) {
  if constexpr (ALIGNED) {
    const int c = short_col<T, true>(u, 0, lane);
    return c < d ? __ldcs(reinterpret_cast<const uint4*>(row + c)) : make_uint4(0u, 0u, 0u, 0u);
  } else {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if constexpr (sizeof(T) == 4) {
        const int c = short_col<T, false>(u, k, lane);
        w[k] = c < d ? __ldg(reinterpret_cast<const uint32_t*>(row) + c) : 0u;
      } else {
        const int c = short_col<T, false>(u, 2 * k, lane);
        const uint16_t* p = reinterpret_cast<const uint16_t*>(row);
        const uint32_t lo = c < d ? __ldg(p + c) : 0u, hi = c + 1 < d ? __ldg(p + c + 1) : 0u;
        w[k] = lo | (hi << 16);
      }
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Ragged bf16 rows inside X: the aligned 4-byte words that hold the row (its first
// element may be the upper half of one) ...
template <int K>
__device__ __forceinline__ void words_load(const __nv_bfloat16* row, int lane, int d,
                                           uint4 (&x)[K]) {
  const int o = (int)(reinterpret_cast<uintptr_t>(row) >> 1) & 1;
  const uint32_t* p = reinterpret_cast<const uint32_t*>(row - o);
  const int nw = (d + o + 1) >> 1;  // at most 128 K words: d < 256 K
  auto word = [&](int i) { return i * 32 + lane < nw ? __ldg(p + i * 32 + lane) : 0u; };
#pragma unroll
  for (int u = 0; u < K; ++u)
    x[u] = make_uint4(word(4 * u), word(4 * u + 1), word(4 * u + 2), word(4 * u + 3));
}
// ... and, for such a row, the upper half with the next word's lower one; nothing of
// the next row is left.
template <int K>
__device__ __forceinline__ void words_shift(const __nv_bfloat16* row, int lane, int d,
                                            uint4 (&x)[K]) {
  const int o = (int)(reinterpret_cast<uintptr_t>(row) >> 1) & 1;
  uint32_t w[4 * K + 1];
#pragma unroll
  for (int u = 0; u < K; ++u) {
    w[4 * u] = x[u].x, w[4 * u + 1] = x[u].y, w[4 * u + 2] = x[u].z, w[4 * u + 3] = x[u].w;
  }
  w[4 * K] = 0u;
  if (o) {
#pragma unroll
    for (int i = 0; i < 4 * K; ++i) {
      // lane 31's next word is lane 0's of the block that follows
      const uint32_t next = __shfl_sync(0xffffffffu, lane == 0 ? w[i + 1] : w[i], (lane + 1) & 31);
      w[i] = __funnelshift_r(w[i], next, 16);
    }
  }
#pragma unroll
  for (int i = 0; i < 4 * K; ++i) {
    const int c = (i * 32 + lane) * 2;
    w[i] = c + 1 < d ? w[i] : (c < d ? w[i] & 0xffffu : 0u);
  }
#pragma unroll
  for (int u = 0; u < K; ++u)
    x[u] = make_uint4(w[4 * u], w[4 * u + 1], w[4 * u + 2], w[4 * u + 3]);
}

template <typename T, bool ALIGNED, int K, int RB>
__global__ void __launch_bounds__(32 * kShortWarps, 2) k_chunkgrad_short(CGArgs a) {
  constexpr int V = Vec<T>::V, V2 = V / 2;
  constexpr int LR = RB >= 16 ? 4 : (RB >= 8 ? 3 : (RB >= 4 ? 2 : 1)), kShift = 5 - LR;  // lanes of a row: 1 << kShift
  __shared__ float s_acc[kShortWarps][K * 32 * V];
  __shared__ double s_loss[kShortWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T* X = static_cast<const T*>(a.X);
  const long long rows = a.nbatch / a.nbc * a.n_c;
  auto col_of = [&](int u, int e) {
    return short_col<T, ALIGNED>(u, e, lane);
  };
  float2 wv[K][V2];
#pragma unroll
  for (int u = 0; u < K; ++u)
#pragma unroll
    for (int e = 0; e < V2; ++e) {
      const int c0 = col_of(u, 2 * e), c1 = col_of(u, 2 * e + 1);
      wv[u][e] = make_float2(c0 < a.d ? __ldg(a.w + c0) : 0.f, c1 < a.d ? __ldg(a.w + c1) : 0.f);
    }
  // whose range: the block's, or (few batches a chunk) this warp's own
  const int stride = a.by_warp ? 1 : kShortWarps;
  const long long q = a.by_warp ? (long long)blockIdx.x * kShortWarps + warp : (long long)blockIdx.x;
  const long long g0 = q * a.bpc, g1 = min(g0 + a.bpc, a.nbatch);
  const long long first_chunk = g0 / a.nbc;
  double loss_acc = 0.0;
  for (long long g = g0; g < g1;) {
    const long long chunk = g / a.nbc;
    const int b0 = (int)(g - chunk * a.nbc), b1 = (int)min((long long)a.nbc, b0 + (g1 - g));
    float2 acc[K][V2];
#pragma unroll
    for (int u = 0; u < K; ++u)
#pragma unroll
      for (int e = 0; e < V2; ++e) acc[u][e] = make_float2(0.f, 0.f);
    for (int b = b0 + (a.by_warp ? 0 : warp); b < b1; b += stride) {
      const int nr = min(RB, a.n_c - b * RB);
      const long long row0 = chunk * a.n_c + (long long)b * RB;
      uint4 x[RB][K];
      // Ragged bf16: by words 501 columns run at 54% of the copy rate, by elements 27%.
      // Rows whose words lie inside X (a first or last word may reach beyond its row)
      // and fit a lane's 4 K (256 K columns from an odd element on would need one more)
      const bool inside = sizeof(T) == 2 && !ALIGNED && row0 > 0 && row0 + nr < rows && a.d % 256;
      if (inside) {
        if constexpr (sizeof(T) == 2) {
#pragma unroll
          for (int r = 0; r < RB; ++r) words_load<K>(X + (row0 + min(r, nr - 1)) * a.d, lane, a.d, x[r]);
#pragma unroll
          for (int r = 0; r < RB; ++r) {
            words_shift<K>(X + (row0 + min(r, nr - 1)) * a.d, lane, a.d, x[r]);
            if (r >= nr)
#pragma unroll
              for (int u = 0; u < K; ++u) x[r][u] = make_uint4(0u, 0u, 0u, 0u);
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
          for (int u = 0; u < K; ++u)
            x[r][u] = r < nr ? short_load<T, ALIGNED>(X + (row0 + r) * a.d, u, lane, a.d)
                             : make_uint4(0u, 0u, 0u, 0u);
      }
      const int my = lane >> kShift;  // this lane's row
      const float yv = my < nr ? __ldg(a.y + row0 + my) : 0.f;
      float pd[RB];
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        float2 p2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < K; ++u) {
          float xv[V];
          Vec<T>::unpack(x[r][u], xv);
#pragma unroll
          for (int e = 0; e < V2; ++e)
            p2 = __ffma2_rn(make_float2(xv[2 * e], xv[2 * e + 1]), wv[u][e], p2);
        }
        pd[r] = p2.x + p2.y;
      }
      const float z = warp_sum_rows<RB>(pd, lane);
      // a row past the chunk's end is zeros, whose dot with an infinite w is NaN: its
      // residual is zero whatever the dot
      const float mine = my >= nr ? 0.f
                         : a.loss == GC_LSQ ? z - yv : 1.f / (1.f + __expf(-z)) - 0.5f * (yv + 1.f);
      if (a.want_loss && my < nr && (lane & ((1 << kShift) - 1)) == 0) {
        if (a.loss == GC_LSQ) {
          const float e = z - yv;
          loss_acc += (double)(0.5f * e * e);
        } else {
          // as in the ring kernel: log(1 + e^t), about 1e-6 absolute per row
          const float t = -yv * z;
          loss_acc += (double)(fmaxf(t, 0.f) + __logf(1.f + __expf(-fabsf(t))));
        }
      }
      __syncwarp();
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const float res = __shfl_sync(0xffffffffu, mine, r << kShift);
        const float2 rr = make_float2(res, res);
#pragma unroll
        for (int u = 0; u < K; ++u) {
          float xv[V];
          Vec<T>::unpack(x[r][u], xv);
#pragma unroll
          for (int e = 0; e < V2; ++e)
            acc[u][e] = __ffma2_rn(rr, make_float2(xv[2 * e], xv[2 * e + 1]), acc[u][e]);
        }
      }
    }
    g += b1 - b0;
    float* dst = a.parts + ((size_t)q * a.maxt + (size_t)(chunk - first_chunk)) * a.d;
    if (a.by_warp) {
#pragma unroll
      for (int u = 0; u < K; ++u)
#pragma unroll
        for (int e = 0; e < V2; ++e) {
          const int c0 = col_of(u, 2 * e), c1 = col_of(u, 2 * e + 1);
          if constexpr (ALIGNED) {  // d is a multiple of V
            if (e % 2 == 0 && c0 < a.d)
              *reinterpret_cast<float4*>(dst + c0) =
                  make_float4(acc[u][e].x, acc[u][e].y, acc[u][e + 1].x, acc[u][e + 1].y);
          } else {
            if (c0 < a.d) dst[c0] = acc[u][e].x;
            if (c1 < a.d) dst[c1] = acc[u][e].y;
          }
        }
      continue;
    }
    // the warps' partial gradients of this chunk, added in warp order
#pragma unroll
    for (int u = 0; u < K; ++u)
#pragma unroll
      for (int e = 0; e < V2; ++e) {
        if (ALIGNED || sizeof(T) == 2) {
          *reinterpret_cast<float2*>(&s_acc[warp][col_of(u, 2 * e)]) = acc[u][e];
        } else {
          s_acc[warp][col_of(u, 2 * e)] = acc[u][e].x;
          s_acc[warp][col_of(u, 2 * e + 1)] = acc[u][e].y;
        }
      }
    __syncthreads();
    for (int c = threadIdx.x; c < a.d; c += 32 * kShortWarps) {
      float t = 0.f;
#pragma unroll
      for (int k = 0; k < kShortWarps; ++k) t += s_acc[k][c];
      dst[c] = t;
    }
    __syncthreads();
  }
  // the reduction kernel may be scheduled now (it waits for this grid to finish)
  if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (a.want_loss) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
    if (lane == 0) s_loss[warp] = loss_acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int k = 0; k < kShortWarps; ++k) t += s_loss[k];
      a.loss_parts[blockIdx.x] = t;
    }
  }
}

template <typename T, bool ALIGNED>
static Kernel pick_short_t(int K) {
  constexpr bool kBf16 = sizeof(T) == 2;
  switch (K) {
    case 1: return k_chunkgrad_short<T, ALIGNED, 1, short_rows(1, kBf16)>;
    case 2: return k_chunkgrad_short<T, ALIGNED, 2, short_rows(2, kBf16)>;
    case 3: return k_chunkgrad_short<T, ALIGNED, 3, short_rows(3, kBf16)>;
    case 4:
      if constexpr (!kBf16) return k_chunkgrad_short<T, ALIGNED, 4, short_rows(4, false)>;
      return nullptr;
    default: return nullptr;
  }
}
Kernel pick_short(bool bf16, bool aligned, int K) {
  if (bf16) return aligned ? pick_short_t<__nv_bfloat16, true>(K) : pick_short_t<__nv_bfloat16, false>(K);
  return aligned ? pick_short_t<float, true>(K) : pick_short_t<float, false>(K);
}

}  // namespace cg
}  // namespace gc
