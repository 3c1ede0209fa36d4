// Batched decode in residual form.
//
// The decode block of chunk i in pattern b is Pi_{b,i} = R_{S_i} X^+, which is
// exactly I_ell whenever Delta_i >= ell (Sec. II-A: X = R[:, S_i] then has full
// row rank).  Writing D_{b,i} = Pi_{b,i} - I_ell, the decoded gradient is
//
//   ghat_b[k*L + c] = s[k*L + c] + sum_{i : D_{b,i} != 0} sum_k' D_{b,i}[k][k'] g_{D_i}[k'*L + c],
//   s = sum_i g_{D_i}  (the full gradient; Sec. I),
//
// the same linear map as the combine GEMM (Ghat = C . G, C = [Pi_{b,1} ... Pi_{b,N}]),
// evaluated with the identity blocks summed once per batch.  A pattern with few
// non-identity blocks is the write of ghat_b plus one read of g_{D_i} per such
// block; a pattern with many is cheaper on the tensor-core GEMM
// (k_combine_tc.cu).  The choice is made per pattern on the device, from the
// decode plan itself:
//
//   k_plan_scan     one warp per pattern: the ordered list of its non-identity
//                   blocks (chunk, D) and its length; the batch's totals that
//                   decide whether the GEMM runs at all.
//   k_gsum          s = sum_i g_{D_i} over all of d (one pass over G).
//   k_decode_resid  one CTA per (tile of patterns, 1024-column range of each
//                   block): every pattern below the threshold gets s, or s plus
//                   its corrections (all ell output blocks at once, so that
//                   each g_{D_i} is read once); the tiles of one column range
//                   run side by side, so each range of g_{D_i} is read from
//                   HBM about once.  ||ghat_b - s||^2 = ||corrections||^2 is
//                   left as one partial per (pattern, range).
// The patterns above the threshold are gathered by the GEMM's operand split.
// (A path per 128-row tile of the plan -- the GEMM for every tile with one
// heavy pattern -- took 4.56 ms for N = m = 256, delta = 16, ell = 4, d = 2^20,
// 1,024 patterns, of which one in eight is heavy but every 32 in a row hold
// one; the path per pattern takes 2.19 ms.)
#include <algorithm>

#include "gc_internal.cuh"

namespace gc {

int resid_ksp(int ell) { return ell <= 2 ? 32 : (ell <= 4 ? 16 : 8); }

static int resid_parts(int L) { return (L + kResidW - 1) / kResidW; }

size_t resid_ws_bytes(int N, int ell, int npat, int d) {
  Carve c(nullptr);
  carve_resid(c, N, ell, npat, d, true);
  return c.bytes() - kHeaderBytes;
}

ResidLists carve_resid(Carve& c, int N, int ell, int npat, int d, bool want_mse) {
  const int L = (d + ell - 1) / ell;
  ResidLists r{};
  r.ksp = std::min(resid_ksp(ell), N);
  r.parts = resid_parts(L);
  r.nnz = c.take<int32_t>(npat);
  r.idx = c.take<int32_t>((size_t)npat * r.ksp);
  r.D = c.take<float>((size_t)npat * r.ksp * ell * ell);
  r.stat = c.take<int32_t>(4);
  r.dpat = c.take<int32_t>(npat);
  r.dtile = c.take<int32_t>(npat / (128 / ell) + 1);
  float* msp = c.take<float>((size_t)npat * r.parts);
  r.msp = want_mse ? msp : nullptr;
  return r;
}

// ---------------------------------------------------------------------------
// Plan scan: non-identity blocks per pattern, totals of the batch.
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;  // one warp per pattern
constexpr int kScanWarps = kScanThreads / 32;

// ELL consecutive plan entries from p (p is 2 ELL-byte aligned for ELL = 2, 4)
template <int ELL>
__device__ __forceinline__ void plan_load(const __nv_bfloat16* p, float (&v)[ELL]) {
  if constexpr (ELL == 4) {
    const uint2 q = __ldg(reinterpret_cast<const uint2*>(p));
    v[0] = __uint_as_float(q.x << 16);
    v[1] = __uint_as_float(q.x & 0xffff0000u);
    v[2] = __uint_as_float(q.y << 16);
    v[3] = __uint_as_float(q.y & 0xffff0000u);
  } else if constexpr (ELL == 2) {
    const uint32_t q = __ldg(reinterpret_cast<const uint32_t*>(p));
    v[0] = __uint_as_float(q << 16);
    v[1] = __uint_as_float(q & 0xffff0000u);
  } else {
#pragma unroll
    for (int k = 0; k < ELL; ++k) v[k] = __bfloat162float(p[k]);
  }
}

template <int ELL>
__global__ void __launch_bounds__(kScanThreads) k_plan_scan(const __nv_bfloat16* __restrict__ Cs, int Kp,
                                                   int N, int npat, int budget, ResidLists rl,
                                                   unsigned int* counters) {
  // the sum of the chunk gradients (next in the stream) does not read the
  // lists: let it start now
  if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const size_t plane = (size_t)npat * ELL * Kp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ int s_over, s_extra;
  if (threadIdx.x == 0) s_over = s_extra = 0;
  __syncthreads();
  const long long b = (long long)blockIdx.x * kScanWarps + warp;
  if (b < npat) {
    int count = 0;
    for (int i0 = 0; i0 < N; i0 += 32) {
      const int i = i0 + lane;
      float Dv[ELL][ELL];
      bool nz = false;
#pragma unroll
      for (int a = 0; a < ELL; ++a) {
        float h[ELL], l[ELL];
#pragma unroll
        for (int k = 0; k < ELL; ++k) h[k] = l[k] = a == k ? 0.5f : 0.f;
        if (i < N) {
          const size_t e = ((size_t)b * ELL + a) * Kp + (size_t)i * ELL;
          plan_load<ELL>(Cs + e, h);
          plan_load<ELL>(Cs + plane + e, l);
        }
#pragma unroll
        for (int k = 0; k < ELL; ++k) {
          Dv[a][k] = h[k] + l[k] - (a == k ? 1.f : 0.f);
          nz |= Dv[a][k] != 0.f;
        }
      }
      const unsigned bal = __ballot_sync(0xffffffffu, nz);
      const int pos = count + __popc(bal & ((1u << lane) - 1u));
      if (nz && pos < rl.ksp) {
        rl.idx[(size_t)b * rl.ksp + pos] = i;
        float* dst = rl.D + ((size_t)b * rl.ksp + pos) * ELL * ELL;
#pragma unroll
        for (int a = 0; a < ELL; ++a)
#pragma unroll
          for (int k = 0; k < ELL; ++k) dst[a * ELL + k] = Dv[a][k];
      }
      count += __popc(bal);
    }
    if (lane == 0) {
      rl.nnz[b] = count;
      if (count > rl.ksp) atomicAdd(&s_over, 1);
      else if (count > budget) atomicAdd(&s_extra, count - budget);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_over) atomicAdd(counters + 1, (unsigned)s_over);
    if (s_extra) atomicAdd(counters + 2, (unsigned)s_extra);
    __threadfence();
    // the last CTA hands the totals over and leaves the counters at zero, as
    // the next launch expects them (the first wraps by itself)
    if (atomicInc(counters, gridDim.x - 1) == gridDim.x - 1) {
      __threadfence();
      rl.stat[0] = (int)atomicExch(counters + 1, 0u);
      rl.stat[1] = (int)atomicExch(counters + 2, 0u);
      rl.stat[2] = rl.stat[3] = 0;  // counted by the operand split
    }
  }
}

// ---------------------------------------------------------------------------
// s = sum_i g_{D_i} (chunks added in order 0..N-1).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void gsum_cols(const float* __restrict__ G, int N, int d, int vec,
                                          float* __restrict__ gsum) {
  const long long c0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (c0 >= d) return;
  if (vec) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* p = G + c0;
    int i = 0;
    for (; i + 8 <= N; i += 8) {
      float4 q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = __ldg(reinterpret_cast<const float4*>(p + (size_t)(i + u) * d));
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        acc.x += q[u].x;
        acc.y += q[u].y;
        acc.z += q[u].z;
        acc.w += q[u].w;
      }
    }
    for (; i < N; ++i) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(p + (size_t)i * d));
      acc.x += q.x;
      acc.y += q.y;
      acc.z += q.z;
      acc.w += q.w;
    }
    *reinterpret_cast<float4*>(gsum + c0) = acc;
  } else {
    for (int v = 0; v < 4; ++v) {
      const long long c = c0 + v;
      if (c >= d) break;
      float acc = 0.f;
      for (int i = 0; i < N; ++i) acc += __ldg(G + (size_t)i * d + c);
      gsum[c] = acc;
    }
  }
}

// Launched as a programmatic dependent of the plan scan, which it does not
// read: the two run side by side.  It waits for the scan before it exits, so
// that work ordered after it (the residual decode, which reads both) finds
// the scan complete.
__global__ void __launch_bounds__(128) k_gsum(const float* __restrict__ G, int N, int d, int vec,
                                              float* __restrict__ gsum) {
  gsum_cols(G, N, d, vec, gsum);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Residual decode.  Block (pattern tile, range r, slice z): columns
// [r*W, r*W + W) of every block k (the same offsets in all ell blocks, so one
// load of g_{D_i}[k'] serves every output block).  A thread takes four columns:
// 4 t .. 4 t + 3 when rows are 16-byte pieces (VEC), else t, t + 256, ...
// ---------------------------------------------------------------------------
template <bool VEC>
__device__ __forceinline__ int resid_col(int v) {
  return VEC ? 4 * (int)threadIdx.x + v : (int)threadIdx.x + kResidThreads * v;
}
// the thread's four columns of a row; ok: bit v = column v exists (VEC: all or none)
template <bool VEC>
__device__ __forceinline__ float4 ld4(const float* __restrict__ row, uint32_t ok) {
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
  if constexpr (VEC) {
    if (ok) x = __ldg(reinterpret_cast<const float4*>(row + resid_col<true>(0)));
  } else {
    if (ok & 1u) x.x = __ldg(row + resid_col<false>(0));
    if (ok & 2u) x.y = __ldg(row + resid_col<false>(1));
    if (ok & 4u) x.z = __ldg(row + resid_col<false>(2));
    if (ok & 8u) x.w = __ldg(row + resid_col<false>(3));
  }
  return x;
}
// written once, never re-read here
template <bool VEC>
__device__ __forceinline__ void st4(float* __restrict__ row, uint32_t ok, float4 x) {
  if constexpr (VEC) {
    if (ok) __stcs(reinterpret_cast<float4*>(row + resid_col<true>(0)), x);
  } else {
    if (ok & 1u) __stcs(row + resid_col<false>(0), x.x);
    if (ok & 2u) __stcs(row + resid_col<false>(1), x.y);
    if (ok & 4u) __stcs(row + resid_col<false>(2), x.z);
    if (ok & 8u) __stcs(row + resid_col<false>(3), x.w);
  }
}

template <int ELL, bool VEC>
__global__ void __launch_bounds__(kResidThreads, ELL <= 2 ? 4 : (ELL <= 4 ? 3 : 2))
    k_decode_resid(const float* __restrict__ G, const float* __restrict__ gsum, ResidLists rl,
                   GemmChoice gemm, int npat, int d, int L, int ppt, float* __restrict__ Ghat) {
  __shared__ int s_nnz[128];
  __shared__ float s_sq[128][kResidThreads / 32];
  // a programmatic dependent of the sum of the chunk gradients: s and the
  // scan's lists are complete once this wait returns
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // the operand split may start beside this grid's last blocks
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int thr = gemm.threshold(rl);
  const int pps = (ppt + gridDim.z - 1) / gridDim.z;  // patterns per slice of a tile (<= 128)
  const int b_lo = blockIdx.x * ppt + blockIdx.z * pps;
  const int b_hi = min(min(b_lo + pps, (int)(blockIdx.x + 1) * ppt), npat);
  const int nb = b_hi - b_lo;
  if (nb <= 0) return;
  const int r = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int)threadIdx.x < nb) s_nnz[threadIdx.x] = __ldg(rl.nnz + b_lo + threadIdx.x);
  // columns that exist in block k (padding past L and past d excluded), and s there
  uint32_t ok[ELL];
  float4 sv[ELL];
#pragma unroll
  for (int k = 0; k < ELL; ++k) {
    ok[k] = 0;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int c = r * kResidW + resid_col<VEC>(v);
      if (c < L && (long long)k * L + c < d) ok[k] |= 1u << v;
    }
    sv[k] = Ghat ? ld4<VEC>(gsum + (size_t)k * L + r * kResidW, ok[k]) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();
  for (int q = 0; q < nb; ++q) {
    const int nz = s_nnz[q];
    if (nz > thr) continue;  // the GEMM's pattern
    const int b = b_lo + q;
    float* out = Ghat ? Ghat + (size_t)b * d + r * kResidW : nullptr;
    if (nz == 0) {  // exact pattern: ghat_b = s, zero error
      if (out) {
#pragma unroll
        for (int k = 0; k < ELL; ++k) st4<VEC>(out + (size_t)k * L, ok[k], sv[k]);
      }
      continue;
    }
    float4 cr[ELL];
#pragma unroll
    for (int k = 0; k < ELL; ++k) cr[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int* idx = rl.idx + (size_t)b * rl.ksp;
    const float* Db = rl.D + (size_t)b * rl.ksp * ELL * ELL;
#pragma unroll (ELL <= 2 ? 4 : 1)
    for (int e = 0; e < nz; ++e) {
      const float* gi = G + (size_t)__ldg(idx + e) * d + r * kResidW;
      float4 g[ELL];
#pragma unroll
      for (int kp = 0; kp < ELL; ++kp) g[kp] = ld4<VEC>(gi + (size_t)kp * L, ok[kp]);
#pragma unroll
      for (int kp = 0; kp < ELL; ++kp)
#pragma unroll
        for (int k = 0; k < ELL; ++k) {
          const float w = __ldg(Db + (e * ELL + k) * ELL + kp);
          if (w == 0.f) continue;
          cr[k].x = fmaf(w, g[kp].x, cr[k].x);
          cr[k].y = fmaf(w, g[kp].y, cr[k].y);
          cr[k].z = fmaf(w, g[kp].z, cr[k].z);
          cr[k].w = fmaf(w, g[kp].w, cr[k].w);
        }
    }
    float sq = 0.f;
#pragma unroll
    for (int k = 0; k < ELL; ++k) {
      // corrections only on the output columns that exist
      if (ok[k] & 1u) sq = fmaf(cr[k].x, cr[k].x, sq);
      if (ok[k] & 2u) sq = fmaf(cr[k].y, cr[k].y, sq);
      if (ok[k] & 4u) sq = fmaf(cr[k].z, cr[k].z, sq);
      if (ok[k] & 8u) sq = fmaf(cr[k].w, cr[k].w, sq);
      if (out)
        st4<VEC>(out + (size_t)k * L, ok[k],
                 make_float4(sv[k].x + cr[k].x, sv[k].y + cr[k].y, sv[k].z + cr[k].z, sv[k].w + cr[k].w));
    }
    if (rl.msp) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (lane == 0) s_sq[q][warp] = sq;
    }
  }
  if (!rl.msp) return;
  __syncthreads();
  const int q = threadIdx.x;
  if (q < nb && s_nnz[q] > 0 && s_nnz[q] <= thr) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < kResidThreads / 32; ++w) t += s_sq[q][w];
    rl.msp[(size_t)(b_lo + q) * rl.parts + r] = t;
  }
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
int launch_plan_scan(const __nv_bfloat16* Cs, int Kp, int N, int ell, int npat, int budget,
                     const ResidLists& rl, unsigned int* counters, cudaStream_t s) {
  if (npat == 0) return GC_OK;
  const unsigned blocks = (unsigned)(((long long)npat + kScanWarps - 1) / kScanWarps);
#define GC_SCAN(E) \
  case E: k_plan_scan<E><<<blocks, kScanThreads, 0, s>>>(Cs, Kp, N, npat, budget, rl, counters); break;
  switch (ell) {
    GC_SCAN(1)
    GC_SCAN(2)
    GC_SCAN(3)
    GC_SCAN(4)
    GC_SCAN(5)
    GC_SCAN(6)
    GC_SCAN(7)
    GC_SCAN(8)
    default: return fail(GC_ERR_UNSUPPORTED, "ell=%d exceeds GC_MAX_ELL", ell);
  }
#undef GC_SCAN
  count_launches(1);
  return cuda_check(cudaGetLastError(), "k_plan_scan");
}

int launch_gsum(const float* G, int N, int d, float* gsum, cudaStream_t s) {
  const bool vec = d % 4 == 0 && reinterpret_cast<uintptr_t>(G) % 16 == 0 &&
                   reinterpret_cast<uintptr_t>(gsum) % 16 == 0;
  const long long quads = ((long long)d + 3) / 4;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)((quads + 127) / 128));
  cfg.blockDim = dim3(128);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, k_gsum, G, N, d, vec ? 1 : 0, gsum);
  if (e != cudaSuccess) return cuda_check(e, "cudaLaunchKernelEx(k_gsum)");
  count_launches(1);
  return GC_OK;
}

template <int ELL>
static cudaError_t launch_resid_t(const cudaLaunchConfig_t& cfg, bool vec, const float* G,
                                  const float* gsum, const ResidLists& rl, const GemmChoice& gemm,
                                  int npat, int d, int L, int ppt, float* Ghat) {
  return vec ? cudaLaunchKernelEx(&cfg, k_decode_resid<ELL, true>, G, gsum, rl, gemm, npat, d, L, ppt, Ghat)
             : cudaLaunchKernelEx(&cfg, k_decode_resid<ELL, false>, G, gsum, rl, gemm, npat, d, L, ppt, Ghat);
}

int launch_decode_resid(const float* G, const float* gsum, const ResidLists& rl,
                        const GemmChoice& gemm, int ell, int npat, int d, float* Ghat,
                        cudaStream_t s) {
  if (npat == 0) return GC_OK;
  const int L = (d + ell - 1) / ell;
  const bool vec = d % 4 == 0 && L % 4 == 0 && reinterpret_cast<uintptr_t>(G) % 16 == 0 &&
                   reinterpret_cast<uintptr_t>(gsum) % 16 == 0 &&
                   (!Ghat || reinterpret_cast<uintptr_t>(Ghat) % 16 == 0);
  const int ppt = 128 / ell;  // patterns per tile
  const long long ntile = ((long long)npat + ppt - 1) / ppt;
  const long long nranges = resid_parts(L);
  if (ntile > (1LL << 31) - 1 || nranges > 65535) return fail(GC_ERR_UNSUPPORTED, "residual decode grid too large");
  // tiles fastest: the CTAs of one column range run side by side and share
  // its chunk-gradient lines in L2; small batches split each tile's patterns
  // over up to 8 blocks so that every SM has a few
  int slices = 1;
  while (slices < 8 && ntile * nranges * slices < 16LL * device_sm_count()) slices *= 2;
  // a programmatic dependent of k_gsum (the launch overlaps its tail)
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)ntile, (unsigned)nranges, (unsigned)slices);
  cfg.blockDim = dim3(kResidThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaSuccess;
#define GC_RESID(E) \
  case E: e = launch_resid_t<E>(cfg, vec, G, gsum, rl, gemm, npat, d, L, ppt, Ghat); break;
  switch (ell) {
    GC_RESID(1)
    GC_RESID(2)
    GC_RESID(3)
    GC_RESID(4)
    GC_RESID(5)
    GC_RESID(6)
    GC_RESID(7)
    GC_RESID(8)
    default: return fail(GC_ERR_UNSUPPORTED, "ell=%d exceeds GC_MAX_ELL", ell);
  }
#undef GC_RESID
  if (e != cudaSuccess) return cuda_check(e, "cudaLaunchKernelEx(k_decode_resid)");
  count_launches(1);
  return GC_OK;
}

}  // namespace gc
