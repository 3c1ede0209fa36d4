// The errors of a batch of patterns straight from their counts psi (the sweep
// over completion rates): coefficient error, estimate and gradient MSE, without
// the decode matrix in between.
//
// As in k_mse_gram.cu the MSE is a quadratic form in the Gram matrix H of the
// chunk blocks, ||ghat_b - s||^2 = sum_k v_k H v_k^T, where row k of the decode
// matrix minus the identity, v_k, is non-zero only in the blocks of the chunks
// with fewer than ell copies: v_k[i*ell + k'] = (Pi_i - I)[k][k'].  One warp
// takes a pattern: it forms its chunks' completion masks, takes the blocks of
// those chunks from Algorithm 1's memo table into a list in shared memory --
// all ell rows have the same support, so an entry holds its ell values -- and
// then lane e' sums u_k[e'] = sum_e v_k[e] H[a_e][a_e'], one read of H for ell
// multiply-adds.  (Through the plan: 102 MB of bf16 planes written and read for
// 10^5 patterns of N = 64, ell = 2, 75 + 99 us; here 85 us.)  The blocks
// enter in fp32 (the plan holds them as bf16 hi + lo).
//
// GB300 retires two fp64 operations a clock per SM, 16 clocks a warp
// instruction whatever its active lanes, so the fp64 parts are batched: the
// lanes' coefficient errors of four patterns are summed by one halving tree
// (the same pairs added as by a tree each: 6 additions instead of 20), and the
// rows' sums of 32 patterns wait in one lane each for the final additions.
#include <algorithm>
#include <type_traits>

#include "k_solve.cuh"

namespace gc {
namespace {

// words of a list entry: ell values, then the row offset a*K in H (low half)
// and a (high half); 8- or 16-byte pieces
constexpr int entry_words(int ell) { return ell == 1 ? 2 : (ell <= 3 ? 4 : 8); }

// Lanes without bit `off` go on with a, the others with b: sums over the pairs
// of lanes that differ in it.
__device__ __forceinline__ double halve(double a, double b, int off, int lane) {
  const bool hi = (lane & off) != 0;
  return (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, off);
}

template <int ELL, int CPL, bool HS, bool PAD>
__global__ void __launch_bounds__(1024, 1) k_mse_patterns(
    const double* __restrict__ R, const int32_t* __restrict__ psi, Holders hd, int N, int m,
    int delta, int npat, Table tb, const float* __restrict__ H, const float* __restrict__ H_last,
    double inv_d, double* __restrict__ coef_err, double* __restrict__ est,
    double* __restrict__ grad_mse, uint32_t* status) {
  extern __shared__ __align__(16) float s_dyn[];
  constexpr int EW = entry_words(ELL);
  const int K = N * ELL;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  uint32_t* list = reinterpret_cast<uint32_t*>(s_dyn) + (size_t)warp * K * EW;  // [K][EW]
  float* s_h = s_dyn + (size_t)warps * K * EW;                                   // [K][K] when HS
  if (HS) {
#pragma unroll 4
    for (int t = threadIdx.x; t < K * K; t += blockDim.x) s_h[t] = __ldg(H + t);
    __syncthreads();
  }
  LaneHolders<CPL> lh;
  lh.load(hd, N, lane);
  const long long b0 = (long long)blockIdx.x * warps + warp, stride = (long long)gridDim.x * warps;
  // sums waiting for the fp64 additions: row sums of pattern (it & ~31) + lane
  // of the warp, its estimate, and the lanes' errors of up to three patterns
  float wait_q[ELL];
  int wait_def = 0;
#pragma unroll
  for (int k = 0; k < ELL; ++k) wait_q[k] = 0.f;
  double err_a = 0.0, err_ab = 0.0;
  auto flush_rows = [&](int it) {  // patterns (it & ~31) .. it of the warp
    const long long b = b0 + ((it & ~31) + lane) * stride;
    if (lane <= (it & 31)) {
      double tot = 0.0;
#pragma unroll
      for (int k = 0; k < ELL; ++k) tot += (double)wait_q[k];
      grad_mse[b] = tot * inv_d;
      if (est) est[b] = (double)wait_def;
    }
  };
  auto add_err = [&](int it, double err) {
    if ((it & 1) == 0) {
      err_a = err;
    } else if ((it & 2) == 0) {
      err_ab = halve(err_a, err, 16, lane);
    } else {
      double t = halve(err_ab, halve(err_a, err, 16, lane), 8, lane);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      // lanes 0, 16, 8, 24 hold the four patterns in turn
      const int u = ((lane >> 4) & 1) + 2 * ((lane >> 3) & 1);
      const long long b = b0 + ((it & ~3) + u) * stride;
      if ((lane & 7) == 0 && b < npat) coef_err[b] = t;
    }
  };
  // a chunk with more holders than the table has bits (explicit orders) is
  // solved per pattern; a warp without such chunks runs a loop without the solve
  auto run = [&](auto big) {
  constexpr bool BIG = decltype(big)::value;
  int it = 0;
  for (long long b = b0; b < npat; b += stride, ++it) {
    uint32_t mask[CPL];
    const bool bad = lh.masks(hd, psi + (size_t)b * m, (uint32_t)delta, lane, mask);
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, ST_BAD_PSI);
    // blocks below full rank: their errors and the list (entry pos*ELL + k'
    // is column i*ELL + k'), chunks in ascending order
    double err = 0.0;
    int def = 0, n = 0;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int i = lane + 32 * c;
      const int D = __popc(mask[c]);
      const bool low = i < N && D < ELL;
      const unsigned bal = __ballot_sync(0xffffffffu, low);
      if (low) {
        float pi[ELL * ELL];
        double e_i;
        if (!BIG || lh.cnt[c] <= tb.bits) {
          const size_t e = ((size_t)i << tb.bits) | mask[c];
          const float* src = tb.pi + e * ELL * ELL;
          if constexpr (ELL == 2) {
            const float4 q = __ldg(reinterpret_cast<const float4*>(src));
            pi[0] = q.x; pi[1] = q.y; pi[ELL] = q.z; pi[ELL + 1] = q.w;
          } else {
#pragma unroll
            for (int q = 0; q < ELL * ELL; ++q) pi[q] = __ldg(src + q);
          }
          e_i = __ldg(tb.err + e);
        } else {
          double Pi[ELL][ELL];
          solve_block<ELL>(R, m, lh.cnt[c], hd.w + (size_t)i * GC_MAX_REPL, mask[c], Pi, e_i, status,
                           [](int, int, double) {});
#pragma unroll
          for (int q = 0; q < ELL * ELL; ++q) pi[q] = (float)Pi[q / ELL][q % ELL];
        }
        err = c == 0 ? e_i : err + e_i;
        def += ELL - D;
        const int pos = n + __popc(bal & ((1u << lane) - 1u));
#pragma unroll
        for (int kp = 0; kp < ELL; ++kp) {
          uint32_t* ent = list + (size_t)(pos * ELL + kp) * EW;
          const int a = i * ELL + kp;
          uint32_t w[EW];
#pragma unroll
          for (int k = 0; k < EW; ++k)
            w[k] = k < ELL ? __float_as_uint(pi[(k < ELL ? k : 0) * ELL + kp] - (k == kp ? 1.f : 0.f))
                           : (k == ELL ? (uint32_t)(a * K) | ((uint32_t)a << 16) : 0u);
          if constexpr (EW == 2) {
            *reinterpret_cast<uint2*>(ent) = make_uint2(w[0], w[1]);
          } else {
#pragma unroll
            for (int k = 0; k < EW; k += 4)
              *reinterpret_cast<uint4*>(ent + k) = make_uint4(w[k], w[k + 1], w[k + 2], w[k + 3]);
          }
        }
      }
      n += __popc(bal);
    }
    float q[ELL];
#pragma unroll
    for (int k = 0; k < ELL; ++k) q[k] = 0.f;
    if (n > 0) {
      __syncwarp();
      const int nz = n * ELL;
      // the rows' forms, over the lanes; SKIP leaves the entries that are zero in a row out of it
      auto forms = [&](auto skip) {
        constexpr bool SKIP = decltype(skip)::value;
#pragma unroll
        for (int k = 0; k < ELL; ++k) q[k] = 0.f;
        for (int t0 = 0; t0 < nz; t0 += 32) {
          // lane's own entry e' = t0 + lane (past the end: zero values)
          const bool in = t0 + lane < nz;
          const uint32_t* own = list + (size_t)(in ? t0 + lane : 0) * EW;
          const uint32_t a2 = own[ELL] >> 16;
          float u[ELL];
#pragma unroll
          for (int k = 0; k < ELL; ++k) u[k] = 0.f;
#pragma unroll (SKIP ? 1 : 4)
          for (int e = 0; e < nz; ++e) {
            uint32_t w[EW];
            if constexpr (EW == 2) {
              const uint2 x = *reinterpret_cast<const uint2*>(list + (size_t)e * EW);
              w[0] = x.x;
              w[1] = x.y;
            } else {
#pragma unroll
              for (int k = 0; k < EW; k += 4) {
                if (k <= ELL) {
                  const uint4 x = *reinterpret_cast<const uint4*>(list + (size_t)e * EW + k);
                  w[k] = x.x;
                  w[k + 1] = x.y;
                  w[k + 2] = x.z;
                  w[k + 3] = x.w;
                }
              }
            }
            const uint32_t at = (w[ELL] & 0xffffu) + a2;
            const float hv = HS ? s_h[at] : __ldg(H + at);
#pragma unroll
            for (int k = 0; k < ELL; ++k) {
              const float v = __uint_as_float(w[k]);
              const float f = fmaf(v, PAD && k == ELL - 1 ? __ldg(H_last + at) : hv, u[k]);
              u[k] = SKIP && v == 0.f ? u[k] : f;
            }
          }
          if (in) {
#pragma unroll
            for (int k = 0; k < ELL; ++k) {
              const float v = __uint_as_float(own[k]);
              q[k] = SKIP && v == 0.f ? q[k] : fmaf(v, u[k], q[k]);
            }
          }
        }
        // each row over the lanes
#pragma unroll
        for (int k = 0; k < ELL; ++k) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) q[k] += __shfl_xor_sync(0xffffffffu, q[k], o);
        }
      };
      forms(std::false_type{});
      // the list is that of all rows; an entry that is zero in one of them must not
      // meet an infinite value of H there
      bool finite = true;
#pragma unroll
      for (int k = 0; k < ELL; ++k) finite &= fabsf(q[k]) <= 3.4028235e38f;
      if (ELL > 1 && !finite) forms(std::true_type{});  // warp-uniform
      def = (int)__reduce_add_sync(0xffffffffu, (unsigned)def);
      __syncwarp();  // the list is rewritten by the next pattern
    }
    if (lane == (it & 31)) {
#pragma unroll
      for (int k = 0; k < ELL; ++k) wait_q[k] = q[k];
      wait_def = def;
    }
    if ((it & 31) == 31) flush_rows(it);
    if (coef_err) add_err(it, err);
  }
  if (it & 31) flush_rows(it - 1);
  if (coef_err)
    for (; it & 3; ++it) add_err(it, 0.0);  // the last four with zeros
  };
  bool over = false;
#pragma unroll
  for (int c = 0; c < CPL; ++c) over |= lh.cnt[c] > tb.bits;
  if (__any_sync(0xffffffffu, over))
    run(std::true_type{});
  else
    run(std::false_type{});
}

struct Shape {
  bool hs;
  int warps;
  size_t smem;
};
// H in shared memory when it fits beside the lists of at least 16 warps; with ell = 3
// past 128 rows the warps are worth more (N = 64, delta = 5, 20,000 patterns: 0.90 ms, 0.61
// through the cache; ell = 2, N = 100 0.35 and 0.48, ell = 4, N = 40 0.35 and 0.60)
Shape shape_of(int N, int ell) {
  const size_t K = (size_t)N * ell, list = K * entry_words(ell) * 4, limit = 220 * 1024;
  for (int w : {32, 24, 16})
    if ((ell != 3 || K <= 128) && K * K * 4 + w * list <= limit) return {true, w, K * K * 4 + w * list};
  for (int w : {32, 24, 16})
    if (w * list <= limit) return {false, w, w * list};
  return {false, 0, 0};
}

template <int ELL, int CPL, bool HS, bool PAD>
cudaError_t launch_t(const Shape& sh, int blocks, const double* R, const int32_t* psi, Holders h,
                     int N, int m, int delta, int npat, const Table& tb, const float* H,
                     const float* H_last, double inv_d, double* coef_err, double* est,
                     double* grad_mse, uint32_t* status, cudaStream_t s) {
  auto kern = k_mse_patterns<ELL, CPL, HS, PAD>;
  static SmemOptIn allow;
  const cudaError_t e = allow(kern, 220 * 1024);
  if (e != cudaSuccess) return e;
  kern<<<blocks, sh.warps * 32, sh.smem, s>>>(R, psi, h, N, m, delta, npat, tb, H, H_last, inv_d,
                                              coef_err, est, grad_mse, status);
  return cudaSuccess;
}

}  // namespace

// Taken when the memo table is (its blocks are gathered), for the sizes the
// register-resident holders cover.  Past N*ell = 160 a warp's pattern costs more here
// than in k_mse_gram, whose warps hold a row's entries in registers, until there are
// several for each warp: N = 100, delta = 6, ell = 2, p = 0.5 2,000 patterns 40 us from the plan and
// 74 here, 20,000 102 and 105; N = 64, ell = 4 2,000 206 and 306, 20,000 1517 and 1677; but
// N = 128, ell = 2, 10^5 patterns 513 and 260.
bool mse_patterns_applies(int N, int ell, int bits, int npat) {
  const int K = N * ell;
  return bits >= 0 && ell <= 4 && N <= 128 && shape_of(N, ell).warps > 0 &&
         (K <= 160 || (npat >= 16384 && (ell < 4 || K < 256)));
}

int launch_mse_patterns(const double* R, int ell, const int32_t* psi, Holders h, int N, int m,
                        int delta, int npat, void* table_mem, int bits, const float* H,
                        const float* H_last, int d, double* coef_err, double* est,
                        double* grad_mse, uint32_t* status, cudaStream_t s) {
  const Shape sh = shape_of(N, ell);
  const Table tb = table_at(table_mem, N, ell, bits);
  const int blocks = (int)std::min<long long>(((long long)npat + sh.warps - 1) / sh.warps, device_sm_count());
  const double inv_d = 1.0 / (double)d;
  cudaError_t e = cudaSuccess;
#define GC_MP2(E_, C_, H_, P_)                                                                  \
  e = launch_t<E_, C_, H_, P_>(sh, blocks, R, psi, h, N, m, delta, npat, tb, H, H_last, inv_d,  \
                               coef_err, est, grad_mse, status, s)
#define GC_MP1(E_, C_)                                                        \
  if (sh.hs) {                                                                \
    if (H_last) GC_MP2(E_, C_, true, true); else GC_MP2(E_, C_, true, false);   \
  } else {                                                                    \
    if (H_last) GC_MP2(E_, C_, false, true); else GC_MP2(E_, C_, false, false); \
  }
#define GC_MP(E_)                          \
  case E_:                                 \
    if (N <= 32) { GC_MP1(E_, 1) }         \
    else if (N <= 64) { GC_MP1(E_, 2) }    \
    else { GC_MP1(E_, 4) }                 \
    break;
  switch (ell) {
    GC_MP(1)
    GC_MP(2)
    GC_MP(3)
    GC_MP(4)
    default: return fail(GC_ERR_UNSUPPORTED, "ell=%d", ell);
  }
#undef GC_MP
#undef GC_MP1
#undef GC_MP2
  if (e != cudaSuccess) return cuda_check(e, "cudaFuncSetAttribute(k_mse_patterns)");
  count_launches(1);
  return cuda_check(cudaGetLastError(), "k_mse_patterns");
}

}  // namespace gc
