// Completion times and the encode-and-transmit trigger (Sec. II-A and
// Sec. IV), batched over simulated realizations of the cluster.
//
// Realization r gives every worker a time per chunk tau[r][j] (+inf for a
// failed worker).  W_j finishes the chunk in its slot p (1-based) at p *
// tau_j, so chunk D_i has been processed n_i(T) = #{holders j : O_ij tau_j
// <= T} times by time T, and the PS's error estimate (eq. (7) and the
// sentence after it) is est(T) = sum_i max(0, ell - n_i(T)).  With t_i^(k)
// the k-th smallest completion time of D_i, est(T) = #{(i, k <= ell) :
// t_i^(k) > T}; the first time the estimate reaches theta or less is
// therefore the (N ell - theta)-th smallest of the N ell values t_i^(k).
// theta = 0 gives the time at which every chunk has been processed ell
// times, i.e. exact recovery becomes possible.  The same time counting a
// copy only when its worker has finished all of its chunks (at delta_j
// tau_j) is the completion time of the original protocol (Sec. IV).
//
// GB300 design: one warp per realization.  theta = 0 asks for the largest of
// the chunks' ell-th completion times, and almost all of that can be decided in
// fp32: the times tau are truncated to fp32 (exact to 2^-23, products to 2^-22),
// lanes take chunks and keep the ell smallest of their holders' fp32 times, and
// only the chunks whose value comes within 2^-20 of the warp's largest are
// formed again with the defining double products, by the whole warp; when more
// than a few do (workers of one speed), the products themselves are compared.
// The fp64 pipe (2 operations a clock per SM) and the 64-bit comparisons are what
// bounded the kernel that did it all in double (N = m = 200, delta = 8, ell = 2,
// 10^5 realizations: 0.92 ms; 0.34 this way, 0.42 with all chunks tied).  A
// realization with a time outside [2^-100, 2^100] takes the double form below.
// In the double form, and for theta > 0, lanes gather their holders'
// completion times as 64-bit keys (the bit patterns of non-negative doubles
// order like the values) and keep the ell smallest in registers; for theta > 0
// the N ell values go to shared memory and a most-significant-digit radix
// select (4-bit digits, per-lane packed counters summed with warp reductions)
// finds the order statistic without sorting.
// Every time that leaves the kernel is the double multiply of the definition,
// so times and psi are bit-exact.
#include <math.h>

#include <algorithm>

#include "gc_internal.cuh"

namespace gc {
namespace {

constexpr int kWarpsPerBlock = 4;
// Resident blocks per SM the kernel is compiled for and the grid is sized
// to: 12 (at most 40 registers a thread) while the 2 x ELL running minima
// fit, else 8 (64 registers).  Many warps per SM keep the fp64 products and
// the tau loads of many realizations in flight.
constexpr int blocks_per_sm(int ell) { return ell <= 3 ? 12 : 8; }

// k-th smallest (1-based, 1 <= k <= n) of n keys in shared memory, by warp: a radix
// select over the 4-bit digits in which the keys that are left differ, until they are all
// the same (N = m = 200, delta = 8, ell = 2, theta = 10, 10^5 realizations: 1.31 ms; 1.92 with
// all sixteen digits).
__device__ unsigned long long warp_select(const unsigned long long* keys, int n, int k, int lane) {
  unsigned long long prefix = 0, mask = 0;
  for (;;) {
    unsigned long long all = ~0ull, any = 0;
    for (int t = lane; t < n; t += 32) {
      const unsigned long long key = keys[t];
      if ((key & mask) == prefix) {
        all &= key;
        any |= key;
      }
    }
    all = ((unsigned long long)__reduce_and_sync(0xffffffffu, (unsigned)(all >> 32)) << 32) |
          __reduce_and_sync(0xffffffffu, (unsigned)all);
    any = ((unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)(any >> 32)) << 32) |
          __reduce_or_sync(0xffffffffu, (unsigned)any);
    if (all == any) return all;
    const int shift = (63 - __clzll((long long)(all ^ any))) & ~3;  // the digits above are common
    unsigned long long lo = 0, hi = 0;  // 8-bit counters for digits 0..7 and 8..15
    for (int t = lane; t < n; t += 32) {
      const unsigned long long key = keys[t];
      if ((key & mask) == prefix) {
        const int dg = (int)((key >> shift) & 15u);
        if (dg < 8) lo += 1ull << (8 * dg);
        else hi += 1ull << (8 * (dg - 8));
      }
    }
    int cum = 0, digit = 15;
    for (int dg = 0; dg < 16; ++dg) {
      const unsigned c = (unsigned)(((dg < 8 ? lo : hi) >> (8 * (dg & 7))) & 255u);
      const int tot = (int)__reduce_add_sync(0xffffffffu, c);
      if (cum + tot >= k) {
        digit = dg;
        break;
      }
      cum += tot;
    }
    k -= cum;
    mask = ~0ull << shift;
    prefix = (all & (mask << 4)) | ((unsigned long long)digit << shift);
  }
}

// Keep the ELL smallest keys seen so far (ascending).  Keys are the bit
// patterns of non-negative doubles, which order like the values, so the
// comparisons are integer ones (GB300's fp64 pipe is 1/64 of fp32; only the
// multiplies that define the times stay in fp64).  Branch-free with static
// indices, so the array stays in registers: position k of the result is
// b[k-1] when v goes before it, else min(v, b[k]).
template <int ELL>
__device__ __forceinline__ void insert_smallest(unsigned long long (&b)[ELL], unsigned long long v) {
#pragma unroll
  for (int k = ELL - 1; k > 0; --k) b[k] = v < b[k - 1] ? b[k - 1] : (v < b[k] ? v : b[k]);
  b[0] = v < b[0] ? v : b[0];
}
__device__ __forceinline__ unsigned long long dbits(double x) {
  return (unsigned long long)__double_as_longlong(x);
}
// isfinite on the bit pattern (integer ops; a double compare would use the fp64 pipe)
__device__ __forceinline__ bool finite_bits(double x) {
  return (dbits(x) & 0x7ff0000000000000ull) != 0x7ff0000000000000ull;
}
// A float near a finite non-negative double, from its bits (integer ops; the
// mantissa is truncated, magnitudes outside the float range are clamped).
// Only a starting point for an exact search, so its accuracy is not critical.
__device__ __forceinline__ float approx_float(double x) {
  const unsigned long long b = dbits(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023 + 127;
  if (e <= 0) return 0.f;
  if (e >= 255) return 3.0e38f;
  return __uint_as_float(((unsigned)e << 23) | (unsigned)((b >> 29) & 0x7fffffu));
}

// outside [2^-100, 2^100], or negative (from the sign and the exponent)
__device__ __forceinline__ bool far_out(double x) {
  const unsigned e = (unsigned)(dbits(x) >> 52);
  return e < 1023u - 100u || e > 1023u + 100u;
}

// The ELL smallest of the values seen (ascending), fp32.
template <int ELL>
__device__ __forceinline__ void insert_smallest_f(float (&b)[ELL], float v) {
#pragma unroll
  for (int k = 0; k < ELL; ++k) {
    const float lo = fminf(b[k], v);
    v = fmaxf(b[k], v);
    b[k] = lo;
  }
}
__device__ __forceinline__ unsigned long long warp_min(unsigned long long x) {
  const unsigned hi = (unsigned)(x >> 32);
  const unsigned mh = __reduce_min_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_min_sync(0xffffffffu, hi == mh ? (unsigned)x : 0xffffffffu);
  return ((unsigned long long)mh << 32) | ml;
}
// ell-th smallest of the 32 lanes' keys
__device__ __forceinline__ unsigned long long warp_ell_th(unsigned long long key, int ell, int lane) {
  unsigned long long mn = 0;
  for (int k = 0; k < ell; ++k) {
    mn = warp_min(key);
    const unsigned who = __ballot_sync(0xffffffffu, key == mn);
    if (lane == __ffs(who) - 1) key = ~0ull;
  }
  return mn;
}

constexpr float kBelow = 1.f - 0x1p-20f, kAbove = 1.f + 0x1p-20f;
// Chunks about the largest time that a warp forms one by one; more of them are ties.
constexpr int kTrigExact = 2;
constexpr int kTrigHolders = 8192;  // holder words staged in shared memory (32 KB)

// ZERO: theta = 0 (two kernels, each with the registers it needs).
template <int ELL, bool ZERO>
__global__ void __launch_bounds__(32 * kWarpsPerBlock, blocks_per_sm(ELL))
    k_trigger(const int32_t* __restrict__ order, Holders h, int N, int m, int delta, int hs,
              const double* __restrict__ tau, long long nsim, int theta, double* __restrict__ T_out,
              int32_t* __restrict__ psi_out, double* __restrict__ Tfull_out) {
  extern __shared__ unsigned long long s_dyn[];
  // the integers 0..GC_MAX_REPL as doubles: the slot factors (p + 1) of the
  // completion times are read here rather than converted per product (an
  // int -> double conversion runs on the fp64 pipe, 1/64 of fp32 on GB300)
  __shared__ double s_kd[GC_MAX_REPL + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // per warp: every worker's fp32 time and fp32 finishing time, or in the
  // double form its finishing time (m words), and for theta > 0 2 N ELL
  // completion keys; per block: delta_j of every worker and the first hs
  // holders of every chunk, [holder][chunk], worker in the low half of a word
  // and the slot factor p + 1 as the upper half of its fp32 pattern (exact)
  unsigned long long* fin = s_dyn + (size_t)warp * m;
  float2* tf = reinterpret_cast<float2*>(fin);
  unsigned long long* keys = s_dyn + (size_t)kWarpsPerBlock * m + (size_t)warp * 2 * N * ELL;
  unsigned long long* keysF = keys + (size_t)N * ELL;
  uint32_t* s_h = reinterpret_cast<uint32_t*>(
      s_dyn + (size_t)kWarpsPerBlock * (m + (ZERO ? 0 : 2 * N * ELL)));
  int8_t* s_dj = reinterpret_cast<int8_t*>(s_h + (size_t)hs * N);
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    int c = 0;
    for (int p = 0; p < delta; ++p) c += order[(size_t)j * delta + p] >= 0;
    s_dj[j] = (int8_t)c;
  }
  auto holder = [&](int i, int q) {
    const int w = h.w[(size_t)i * GC_MAX_REPL + q], p = h.p[(size_t)i * GC_MAX_REPL + q];
    return (uint32_t)w | (__float_as_uint((float)(p + 1)) & 0xffff0000u);
  };
  for (int t = threadIdx.x; t < hs * N; t += blockDim.x) {
    const int q = t / N, i = t - q * N;
    s_h[t] = q < h.cnt[i] ? holder(i, q) : 0u;
  }
  for (int c = threadIdx.x; c <= GC_MAX_REPL; c += blockDim.x) s_kd[c] = (double)c;
  __syncthreads();
  const unsigned long long kInf = dbits(INFINITY);
  const int n = N * ELL;
  const int kth = n - theta;
  for (long long r = (long long)blockIdx.x * kWarpsPerBlock + warp; r < nsim;
       r += (long long)gridDim.x * kWarpsPerBlock) {
    const double* tr = tau + r * m;
    unsigned long long Tb = 0, TFb = 0;
    bool wild = false;  // a time outside the range in which fp32 decides
    unsigned tied = 0;  // 1: T, 2: T_full: more chunks about the largest time than are formed one by one
    float topT = 0.f, topF = 0.f;
    if (ZERO) {
      // fp32 times (truncated); +inf for a failed worker
      for (int j = lane; j < m; j += 32) {
        const double tj = tr[j];
        const bool fb = finite_bits(tj);
        wild |= fb && far_out(tj);
        const float f = fb ? approx_float(tj) : INFINITY;
        tf[j] = make_float2(f, f * (float)s_dj[j]);
      }
      wild = __any_sync(0xffffffffu, wild);
      __syncwarp();
    }
    if (ZERO && !wild) {
      // every lane's largest ell-th value, its chunk, and its second largest
      float best = -1.f, second = -1.f, bestF = -1.f, secondF = -1.f;
      int bi = 0, biF = 0;
      for (int i = lane; i < N; i += 32) {
        float b[ELL], bf[ELL];
#pragma unroll
        for (int k = 0; k < ELL; ++k) b[k] = bf[k] = INFINITY;
        const int cnt = h.cnt[i];
        for (int q = 0; q < cnt; ++q) {
          const uint32_t w = q < hs ? s_h[q * N + i] : holder(i, q);
          const float2 v = tf[w & 0xffffu];
          insert_smallest_f<ELL>(b, __uint_as_float(w & 0xffff0000u) * v.x);
          insert_smallest_f<ELL>(bf, v.y);
        }
        const float t = b[ELL - 1], u = bf[ELL - 1];
        second = fmaxf(second, fminf(best, t));
        if (t > best) {
          best = t;
          bi = i;
        }
        secondF = fmaxf(secondF, fminf(bestF, u));
        if (u > bestF) {
          bestF = u;
          biF = i;
        }
      }
      // non-negative floats order like their bits; lanes without a chunk hold -1
      const float A = __uint_as_float(__reduce_max_sync(0xffffffffu, best < 0.f ? 0u : __float_as_uint(best)));
      const float AF = __uint_as_float(__reduce_max_sync(0xffffffffu, bestF < 0.f ? 0u : __float_as_uint(bestF)));
      // exact ell-th time of chunk i: lane q takes its q-th holder (<= 32)
      auto exact = [&](int i, bool full) {
        unsigned long long key = kInf;
        if (lane < h.cnt[i]) {
          const int w = h.w[(size_t)i * GC_MAX_REPL + lane];
          const double tj = tr[w];
          const int c = full ? (int)s_dj[w] : h.p[(size_t)i * GC_MAX_REPL + lane] + 1;
          if (finite_bits(tj)) key = dbits(s_kd[c] * tj);
        }
        return min(warp_ell_th(key, ELL, lane), kInf);
      };
      // the largest time: of the few chunks about top (one as a rule); else a tie
      auto largest = [&](float top, float bst, float scd, int chunk, bool full) {
        const float lim = top * kBelow;
        unsigned lanes = __ballot_sync(0xffffffffu, bst >= lim);
        unsigned long long mx = 0;
        for (int left = kTrigExact; lanes; lanes &= lanes - 1) {
          const int src = __ffs(lanes) - 1;
          if (left-- == 0 || __shfl_sync(0xffffffffu, scd, src) >= lim) {
            tied |= full ? 2u : 1u;
            break;
          }
          mx = max(mx, exact(__shfl_sync(0xffffffffu, chunk, src), full));
        }
        return mx;
      };
      Tb = largest(A, best, second, bi, false);
      if (Tfull_out) {
        // a finishing time is one worker's, so when a single worker's fp32 time
        // lies about AF it is the answer; else the chunks about AF
        int js = -1, count = 0;
        for (int j = lane; j < m; j += 32) {
          const float u = tf[j].y;
          if (u >= AF * kBelow && u <= AF * kAbove) {
            js = j;
            ++count;
          }
        }
        const unsigned has = __ballot_sync(0xffffffffu, count > 0);
        if (AF < INFINITY && __popc(has) == 1 && !__any_sync(0xffffffffu, count > 1)) {
          js = __shfl_sync(0xffffffffu, js, __ffs(has) - 1);
          TFb = dbits(s_kd[s_dj[js]] * tr[js]);
        } else {
          TFb = largest(AF, bestF, secondF, biF, true);
        }
      }
      topT = A;
      topF = AF;
    }
    if (tied) {
      // The answer is one of the double products whose fp32 value lies about topT, and a
      // worker has at most one of them (two slots are 3% apart): when they are all the same
      // number, however many workers and chunks are tied, that is it.  So for T_full.
      // Otherwise the double form decides.  (Chunk by chunk, 10^5 realizations of 200
      // workers at equal speeds took 5.3 ms; 0.42 so, 0.93 all in double.)
      unsigned left = 0;
#pragma unroll 1
      for (; tied; tied &= tied - 1) {
        const bool full = !(tied & 1u);
        const float top = full ? topF : topT;
        unsigned long long mn = ~0ull, mx = 0;
        for (int j = lane; j < m; j += 32) {
          const float f = tf[j].x, dj = (float)s_dj[j];
          const float c = full ? dj : rintf(__fdividef(top, f)), u = c * f;
          if (u >= top * kBelow && u <= top * kAbove && c >= 1.f && c <= dj) {
            const unsigned long long key = dbits(s_kd[(int)c] * tr[j]);
            mn = min(mn, key);
            mx = max(mx, key);
          }
        }
        mn = warp_min(mn);
        const bool inf = !(top < INFINITY);  // a chunk without ell finite copies
        if (!inf && mn != ~warp_min(~mx)) left = 1;
        if (inf) mn = kInf;
        if (full) TFb = mn;
        else Tb = mn;
      }
      tied = left;
    }
    if (!ZERO || wild || tied) {
      // the double form; each worker's finishing time delta_j tau_j (+inf for a
      // failed worker)
      __syncwarp();
      for (int j = lane; j < m; j += 32) {
        const double tj = tr[j];
        const bool fb = finite_bits(tj);
        wild |= fb && far_out(tj);
        fin[j] = fb ? dbits(s_kd[s_dj[j]] * tj) : kInf;
      }
      wild = __any_sync(0xffffffffu, wild);  // for psi below
      __syncwarp();
      // theta = 0: the order statistic is the largest of the N ell values, i.e.
      // the largest ell-th completion time -- a max, no selection needed
      unsigned long long lmax = 0, lmaxF = 0;
      for (int i = lane; i < N; i += 32) {
        unsigned long long b[ELL], bf[ELL];
#pragma unroll
        for (int k = 0; k < ELL; ++k) b[k] = bf[k] = kInf;
        const int cnt = h.cnt[i];
        for (int q = 0; q < cnt; ++q) {
          const int j = h.w[(size_t)i * GC_MAX_REPL + q];
          const int p = h.p[(size_t)i * GC_MAX_REPL + q];
          const double tj = tr[j];
          if (finite_bits(tj)) {
            insert_smallest<ELL>(b, dbits(s_kd[p + 1] * tj));
            insert_smallest<ELL>(bf, fin[j]);
          }
        }
        if (ZERO) {
          lmax = max(lmax, b[ELL - 1]);
          lmaxF = max(lmaxF, bf[ELL - 1]);
        } else {
#pragma unroll
          for (int k = 0; k < ELL; ++k) {
            keys[(size_t)i * ELL + k] = b[k];
            keysF[(size_t)i * ELL + k] = bf[k];
          }
        }
      }
      __syncwarp();
      if (ZERO) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          lmax = max(lmax, (unsigned long long)__shfl_xor_sync(0xffffffffu, lmax, o));
          lmaxF = max(lmaxF, (unsigned long long)__shfl_xor_sync(0xffffffffu, lmaxF, o));
        }
        Tb = lmax;
        TFb = lmaxF;
      } else if (kth >= 1) {
        Tb = warp_select(keys, n, kth, lane);
        TFb = warp_select(keysF, n, kth, lane);
      }
    }
    const double T = __longlong_as_double((long long)Tb);
    const double TF = __longlong_as_double((long long)TFb);
    if (lane == 0) {
      if (T_out) T_out[r] = T;
      if (Tfull_out) Tfull_out[r] = TF;
    }
    if (psi_out) {
      const float Tf = approx_float(T);
      for (int j = lane; j < m; j += 32) {
        // slots finish in order: psi_j is the largest c <= delta_j with
        // c tau_j <= T (the products are monotone in c).  An fp32 estimate of
        // T / tau_j (exact to 2^-20 when no time is wild) decides it unless it
        // lies next to a whole number or a time is wild: then it is corrected
        // with the exact double products.
        const double tj = tr[j];
        const int dj = s_dj[j];
        int c = 0;
        if (finite_bits(tj) && dj > 0) {
          const float q = __fdividef(Tf, approx_float(tj));
          c = q >= (float)dj ? dj : (q > 0.f ? (int)q : 0);
          const float near = rintf(q);
          if (wild || (fabsf(q - near) <= near * 0x1p-18f && near <= (float)dj)) {
            while (c > 0 && dbits(s_kd[c] * tj) > Tb) --c;
            while (c < dj && dbits(s_kd[c + 1] * tj) <= Tb) ++c;
          }
        }
        psi_out[r * m + j] = c;
      }
    }
    __syncwarp();
  }
}

template <int ELL>
int launch_one(const int32_t* order, Holders h, int N, int m, int delta, const double* tau,
               long long nsim, int theta, double* T, int32_t* psi, double* TF, cudaStream_t s) {
  const size_t keys = theta == 0 ? 0 : (size_t)kWarpsPerBlock * 2 * N * ELL;
  // holders of a chunk staged: delta of them (all, when every chunk has at most
  // delta copies); none in the double form, which does not read them, nor where
  // the workers' times alone fill a good part of the shared memory
  const int hs = theta == 0 && m <= 2048 ? std::min(delta, kTrigHolders / N) : 0;
  const size_t smem = ((size_t)kWarpsPerBlock * m + keys) * 8 + (size_t)hs * N * 4 + (size_t)m;
  auto kern = theta == 0 ? k_trigger<ELL, true> : k_trigger<ELL, false>;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(e, "cudaFuncSetAttribute(k_trigger)");
  }
  const long long blocks_needed = (nsim + kWarpsPerBlock - 1) / kWarpsPerBlock;
  const int blocks =
      (int)std::min<long long>(blocks_needed, (long long)device_sm_count() * blocks_per_sm(ELL));
  kern<<<blocks, 32 * kWarpsPerBlock, smem, s>>>(order, h, N, m, delta, hs, tau, nsim, theta,
                                                           T, psi, TF);
  count_launches(1);
  return cuda_check(cudaGetLastError(), "k_trigger");
}

}  // namespace

int launch_trigger(const int32_t* order, Holders h, int N, int m, int delta, const double* tau,
                   long long nsim, int ell, int theta, double* T, int32_t* psi, double* TF,
                   cudaStream_t s) {
  switch (ell) {
    case 1: return launch_one<1>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    case 2: return launch_one<2>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    case 3: return launch_one<3>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    case 4: return launch_one<4>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    case 5: return launch_one<5>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    case 6: return launch_one<6>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    case 7: return launch_one<7>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    case 8: return launch_one<8>(order, h, N, m, delta, tau, nsim, theta, T, psi, TF, s);
    default: return fail(GC_ERR_UNSUPPORTED, "ell=%d exceeds GC_MAX_ELL", ell);
  }
}

}  // namespace gc
