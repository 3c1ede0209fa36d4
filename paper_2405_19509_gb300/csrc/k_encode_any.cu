// Worker encoding (eq. 2) for orders that are not cyclic (Algorithm 2's
// orders of a regular assignment, explicit orders):
//   T[b][j][c] = sum_{p < psi[b][j]} sum_k E[b][j][p][k] * g_{order[j][p]}[k*L + c].
//
// Such workers share no window of chunks, so each of the delta*ell terms of an
// output is a read of its chunk's block.  From the cache those reads bound the
// kernel (N = m = 200, delta = 8, ell = 3, d = 262147, 4 patterns: 1.48 ms,
// one row and one pattern at a time).  Here one block an SM keeps the
// coefficients of PB patterns in shared memory (converted to fp32 once) and
// walks over tiles of 32 columns: it stages the tile of every chunk block --
// the next tile's values wait in registers -- and its warps take four workers
// at a time, eight lanes of four columns a worker, so that a term of four
// workers is one 16-byte read of g and one of the PB coefficients a lane (the
// eight lanes of a worker read the same) and 4 PB multiply-adds.  Bound by the
// instruction rate of those (0.22 ms; 63% of the issue slots); G and T cross HBM
// once per PB patterns, 0.49 GB or 73 us.  (A column a lane, one worker a warp, coefficients converted per tile: 413 us at
// the sizes above; four workers a warp, still converted per tile: 425 us.)
//
// The sums run over slots p ascending, blocks k ascending within a slot.  The
// other forms skip the slots past psi; here their coefficients are zero, which
// adds nothing unless a staged value is infinite or NaN: a tile that holds one
// takes the loop that skips.
#include <algorithm>

#include "gc_internal.cuh"

namespace gc {
namespace {

constexpr int kAnyThreads = 1024;
constexpr int kAnyWarps = kAnyThreads / 32;
constexpr int kAnyCols = 32;
constexpr int kAnyPre = 20;  // values of the next tile a thread holds (N*ell <= 640)

// Words of one worker's coefficients in shared memory: the four workers of a
// warp read the same entry at once, from banks PB words apart.
__host__ __device__ inline int any_estride(int ne, int PB) {
  return ne + ((PB - ne) % 32 + 32) % 32;
}

// ... and of all workers' (a whole number of 16-byte pieces).
__host__ __device__ inline size_t any_ewords(int m, int es) {
  return ((size_t)m * es + 3) / 4 * 4;
}

// (float)x, round to nearest even.  GB300 converts fp64 at 2 values a clock per
// SM; normal results take integer operations instead.
__device__ __forceinline__ float to_float(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned hi = (unsigned)(u >> 32), lo = (unsigned)u;
  if ((u << 1) == 0) return __uint_as_float(hi);  // +-0
  const int e = (int)((hi >> 20) & 0x7ffu) - 896;  // biased fp32 exponent
  if (e < 1 || e > 254) return (float)x;
  // the 52-bit fraction's top 23 bits, and the 29 below them
  unsigned f = ((unsigned)e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  const unsigned rest = lo & 0x1fffffffu;
  f += rest > 0x10000000u || (rest == 0x10000000u && (f & 1u));  // may carry into the exponent
  return __uint_as_float((hi & 0x80000000u) | f);
}

// PB patterns at a time; VEC: rows of G and T are 16-byte pieces.  J: workers
// per group of the cyclic kernel, which has written the groups whose orders
// are all cyclic.
template <int PB, int ELL, bool VEC>
__global__ void __launch_bounds__(kAnyThreads, 1)
    k_encode_any(const double* __restrict__ E, const int32_t* __restrict__ order,
                 const int32_t* __restrict__ psi, int N, int m, int delta, int npat,
                 const float* __restrict__ G, int d, int L, int J, float* __restrict__ T) {
  extern __shared__ __align__(16) float s_any[];
  const int de = delta * ELL, es = any_estride(de * PB, PB);
  const int rows = N * ELL, nquad = (m + 3) / 4;
  float* s_g = s_any;                                  // [rows][kAnyCols]
  float* s_e = s_g + (size_t)rows * kAnyCols;          // [m][es]: entry (p*ELL + k)*PB + q
  float* s_t = s_e + any_ewords(m, es);                // [warps][4][kAnyCols] when !VEC
  int16_t* s_o = reinterpret_cast<int16_t*>(s_t + (VEC ? 0 : kAnyWarps * 4 * kAnyCols));  // [m][delta]
  int8_t* s_np = reinterpret_cast<int8_t*>(s_o + (size_t)m * delta);  // [m][PB], -1: not written
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int l8 = lane & 7, w4 = lane >> 3;  // columns 4 l8 .. + 3 of worker w4 of the warp's four
  // groups whose orders are not cyclic: marked in s_np before it is filled
  const int ngroups = (m + J - 1) / J;
  for (int t = threadIdx.x; t < ngroups; t += kAnyThreads) s_np[t] = 0;
  __syncthreads();
  int mine = 0;
  for (int t = threadIdx.x; t < m * delta; t += kAnyThreads) {
    const int j = t / delta, p = t - j * delta, i = order[t];
    s_o[t] = (int16_t)(i < 0 || i >= N ? -1 : i);
    if (i != (j + p) % N) {
      s_np[j / J] = 1;
      mine = 1;
    }
  }
  if (__syncthreads_or(mine)) {
    // worker j < 32 * kAnyThreads is thread j % kAnyThreads's bit j / kAnyThreads
    uint32_t act = 0;
    for (int u = 0, j = threadIdx.x; j < m; ++u, j += kAnyThreads)
      if (s_np[j / J]) act |= 1u << u;
    __syncthreads();
    const int ntile = (L + kAnyCols - 1) / kAnyCols;
    const long long nitem = (long long)ntile * ((npat + PB - 1) / PB);
    const long long lo = nitem * blockIdx.x / gridDim.x, hi = nitem * (blockIdx.x + 1) / gridDim.x;
    const bool ahead = rows * kAnyCols <= kAnyPre * kAnyThreads;
    // value u of the tile at column c0 for this thread (VEC four columns): row
    // r0 + u * rstep, column cl of the tile.  Block k ends at L or where the row does,
    // which for d < (ELL - 1) L is before the last block (d = 5, ELL = 4: L = 2, blocks
    // of 2, 2, 1 and no columns).
    const int r0 = threadIdx.x / (VEC ? kAnyCols / 4 : kAnyCols);
    constexpr int kRstep = kAnyThreads / (VEC ? kAnyCols / 4 : kAnyCols);
    const int cl = VEC ? 4 * (threadIdx.x % (kAnyCols / 4)) : lane;
    auto fetch = [&](int c0, int u, float (&v)[VEC ? 4 : 1]) {
      const int r = r0 + u * kRstep, i = r / ELL, k = r - i * ELL;
      const int col = k * L + c0 + cl;
      const bool in = r < rows && c0 + cl < L && col < d;
      const float* src = G + (size_t)i * d + col;
      if constexpr (VEC) {
        const float4 q = in ? __ldg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
      } else {
        v[0] = in ? __ldg(src) : 0.f;
      }
    };
    constexpr int kW = VEC ? 4 : 1, kU = kAnyPre / kW;
    float pre[kU][kW];
    if (ahead && lo < hi) {
#pragma unroll
      for (int u = 0; u < kU; ++u) fetch((int)(lo % ntile) * kAnyCols, u, pre[u]);
    }
    int b0 = -1, tile = (int)(lo % ntile), bnext = (int)(lo / ntile) * PB;
    for (long long item = lo; item < hi; ++item) {
      const int c0 = tile * kAnyCols;
      __syncthreads();  // the previous tile has been read
      int odd = 0;      // an infinite or NaN value in the tile
      auto stage = [&](int u, const float (&v)[kW]) {
        const int t = threadIdx.x + u * kAnyThreads;
        if (t * kW < rows * kAnyCols) {
          if constexpr (VEC)
            *reinterpret_cast<float4*>(s_g + (size_t)t * 4) = make_float4(v[0], v[1], v[2], v[3]);
          else
            s_g[t] = v[0];
#pragma unroll
          for (int w = 0; w < kW; ++w)
            odd |= (__float_as_uint(v[w]) & 0x7f800000u) == 0x7f800000u;
        }
      };
      if (ahead) {
#pragma unroll
        for (int u = 0; u < kU; ++u) stage(u, pre[u]);
      } else {
        for (int u = 0; u * kAnyThreads * kW < rows * kAnyCols; ++u) {
          float v[kW];
          fetch(c0, u, v);
          stage(u, v);
        }
      }
      if (bnext != b0) {  // the next patterns' counts and coefficients
        b0 = bnext;
        for (int u = 0, j = threadIdx.x; j < m; ++u, j += kAnyThreads)
#pragma unroll
          for (int q = 0; q < PB; ++q) {
            int v = -1;
            if (((act >> u) & 1u) && b0 + q < npat) {
              v = __ldg(psi + (size_t)(b0 + q) * m + j);
              v = v < 0 ? 0 : (v > delta ? delta : v);  // bad values are flagged by the solve
            }
            s_np[j * PB + q] = (int8_t)v;
          }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < PB; ++q)
          for (int t = threadIdx.x; t < m * de; t += kAnyThreads) {
            const int j = t / de, x = t - j * de, p = x / ELL;
            float e = 0.f;
            if (p < s_np[j * PB + q] && s_o[j * delta + p] >= 0)
              e = to_float(__ldg(E + (size_t)(b0 + q) * m * de + t));
            s_e[(size_t)j * es + x * PB + q] = e;
          }
      }
      odd = __syncthreads_or(odd);
      if (++tile == ntile) {
        tile = 0;
        bnext += PB;
      }
      if (ahead && item + 1 < hi) {
#pragma unroll
        for (int u = 0; u < kU; ++u) fetch(tile * kAnyCols, u, pre[u]);
      }
      for (int quad = warp; quad < nquad; quad += kAnyWarps) {
        const int j = 4 * quad + w4, jc = j < m ? j : m - 1;
        int top = -1;
        uint32_t on = 0;  // bit q: pattern b0 + q of this worker is written here
        if (j < m) {
#pragma unroll
          for (int q = 0; q < PB; ++q) {
            const int v = s_np[j * PB + q];
            top = max(top, v);
            on |= v >= 0 ? 1u << q : 0u;
          }
        }
        top = __reduce_max_sync(0xffffffffu, top);
        if (top < 0) continue;
        float acc[PB][4];
#pragma unroll
        for (int q = 0; q < PB; ++q)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[q][v] = 0.f;
        const float* e = s_e + (size_t)jc * es;
        const int16_t* o = s_o + jc * delta;
        if (!odd) {
          for (int p = 0; p < top; ++p) {
            const float* g = s_g + max((int)o[p], 0) * (ELL * kAnyCols) + 4 * l8;
#pragma unroll
            for (int k = 0; k < ELL; ++k, e += PB) {
              const float4 x = *reinterpret_cast<const float4*>(g + k * kAnyCols);
              float ev[PB];
              if constexpr (PB == 4) {
                const float4 w = *reinterpret_cast<const float4*>(e);
                ev[0] = w.x; ev[1] = w.y; ev[2] = w.z; ev[3] = w.w;
              } else if constexpr (PB == 2) {
                const float2 w = *reinterpret_cast<const float2*>(e);
                ev[0] = w.x; ev[1] = w.y;
              } else {
                ev[0] = *e;
              }
#pragma unroll
              for (int q = 0; q < PB; ++q) {
                acc[q][0] = fmaf(ev[q], x.x, acc[q][0]);
                acc[q][1] = fmaf(ev[q], x.y, acc[q][1]);
                acc[q][2] = fmaf(ev[q], x.z, acc[q][2]);
                acc[q][3] = fmaf(ev[q], x.w, acc[q][3]);
              }
            }
          }
        } else if (j < m) {
          for (int p = 0; p < top; ++p) {
            if (o[p] < 0) continue;
            const float* g = s_g + o[p] * (ELL * kAnyCols) + 4 * l8;
#pragma unroll 1
            for (int k = 0; k < ELL; ++k)
#pragma unroll
              for (int q = 0; q < PB; ++q)
                if (p < s_np[j * PB + q])
#pragma unroll
                  for (int v = 0; v < 4; ++v)
                    acc[q][v] = fmaf(e[(p * ELL + k) * PB + q], g[k * kAnyCols + v], acc[q][v]);
          }
        }
        float* out = T + ((size_t)b0 * m + (VEC ? j : 4 * quad)) * L + c0 + (VEC ? 4 * l8 : lane);
        const size_t pstep = (size_t)m * L;  // next pattern
        if constexpr (VEC) {
          if (c0 + 4 * l8 < L) {
#pragma unroll
            for (int q = 0; q < PB; ++q, out += pstep)
              if ((on >> q) & 1u)
                __stcs(reinterpret_cast<float4*>(out),
                       make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]));
          }
        } else {
          // through shared memory, so that a store covers consecutive columns
          float* st = s_t + warp * 4 * kAnyCols;
          uint32_t won[4];
#pragma unroll
          for (int w = 0; w < 4; ++w)
            won[w] = __shfl_sync(0xffffffffu, on, 8 * w) & (c0 + lane < L ? ~0u : 0u);
#pragma unroll
          for (int q = 0; q < PB; ++q, out += pstep) {
            __syncwarp();
            *reinterpret_cast<float4*>(st + w4 * kAnyCols + 4 * l8) =
                make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
            __syncwarp();
#pragma unroll
            for (int w = 0; w < 4; ++w)
              if ((won[w] >> q) & 1u) __stcs(out + (size_t)w * L, st[w * kAnyCols + lane]);
          }
        }
      }
    }
  }
  // runs beside the cyclic kernel's tail (a programmatic dependent); work
  // ordered after this kernel must find that one complete, too
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

size_t any_smem(int N, int m, int delta, int ell, int PB) {
  return ((size_t)N * ell * kAnyCols + any_ewords(m, any_estride(delta * ell * PB, PB)) +
          (size_t)kAnyWarps * 4 * kAnyCols) * sizeof(float) +
         (size_t)m * delta * sizeof(int16_t) + (size_t)m * PB;
}

// Patterns at a time: as many as fit beside the tile, no more than there are (0: none fits).
int any_patterns(int N, int m, int delta, int ell, int npat) {
  for (int PB = npat >= 3 ? 4 : (npat == 2 ? 2 : 1); PB >= 1; PB /= 2)
    if (any_smem(N, m, delta, ell, PB) <= kEncodeAnySmem) return PB;
  return 0;
}

// rows of G and T are 16-byte pieces
bool any_vec(int L, int d, const float* G, const float* T) {
  return L % 4 == 0 && d % 4 == 0 &&
         (reinterpret_cast<uintptr_t>(G) | reinterpret_cast<uintptr_t>(T)) % 16 == 0;
}

template <int PB, int ELL, bool VEC>
int launch_any_t(size_t smem, const double* E, const int32_t* order, const int32_t* psi, int N,
                 int m, int delta, int npat, const float* G, int d, int L, int J, float* T,
                 cudaStream_t s) {
  auto kern = k_encode_any<PB, ELL, VEC>;
  static SmemOptIn allow;
  cudaError_t e = allow(kern, kEncodeAnySmem);
  if (e != cudaSuccess) return cuda_check(e, "cudaFuncSetAttribute(k_encode_any)");
  const long long items = (long long)((L + kAnyCols - 1) / kAnyCols) * ((npat + PB - 1) / PB);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)std::min<long long>(items, device_sm_count()));
  cfg.blockDim = dim3(kAnyThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, E, order, psi, N, m, delta, npat, G, d, L, J, T);
  if (e != cudaSuccess) return cuda_check(e, "cudaLaunchKernelEx(k_encode_any)");
  count_launches(1);
  return GC_OK;
}

}  // namespace

// Whether k_encode_any takes the groups that are not cyclic.  The order lies on
// the device, so the launch is paid for cyclic orders as well (about 2 us with
// its scan of the order): only from 2^26 multiply-adds on, where the form that
// reads the cache takes 35-55 us.  That form takes 0.5-1 us per 2^20 multiply-adds, of
// whole blocks of 512 columns, by the sizes and by how many slots are finished; a tile here
// 1.2 us (rows that are no 16-byte pieces 0.9 us more a pattern) and its multiply-adds at 43
// a nanosecond.  So few workers or few blocks on long rows stay there: ell = 1, delta = 4,
// L = 2^20, m = 16 53 us against 256 here, m = 50 182 and 287; ell = 2, L = 2^19, m = 50 147 and 163,
// m = 64 199 and 172; ell = 4, delta = 8, L = 2^18, m = 20 126 and 91.
bool encode_any_applies(int N, int m, int delta, int ell, int npat, int d, const float* G,
                        const float* T) {
  const int L = (d + ell - 1) / ell;
  const double fmas = (double)npat * m * L * delta * ell;
  if (ell > 4 || N >= 32768 || m > 4096 || fmas < (double)(1 << 26)) return false;
  const int PB = any_patterns(N, m, delta, ell, npat);
  if (PB == 0) return false;
  const long long items = (long long)((L + kAnyCols - 1) / kAnyCols) * ((npat + PB - 1) / PB);
  const long long rounds = (items + device_sm_count() - 1) / device_sm_count();
  const double item_us = 1.25 + (any_vec(L, d, G, T) ? 0.0 : 0.9 * PB) +
                         (double)m * delta * ell * kAnyCols * PB / 43e3;
  const double whole = (double)((L + 511) / 512 * 512) / L;
  return (double)rounds * item_us < fmas * whole / (1 << 20) * 0.7;
}

int launch_encode_any(const double* E, const int32_t* order, const int32_t* psi, int N, int m,
                      int delta, int ell, int npat, const float* G, int d, int J, float* T,
                      cudaStream_t s) {
  const int L = (d + ell - 1) / ell;
  const int PB = any_patterns(N, m, delta, ell, npat);
  const size_t smem = any_smem(N, m, delta, ell, PB);
  const bool vec = any_vec(L, d, G, T);
  auto go = [&](auto launch) {
    return launch(smem, E, order, psi, N, m, delta, npat, G, d, L, J, T, s);
  };
#define GC_ANY(E_)                                                                          \
  case E_:                                                                                  \
    if (PB == 4) return vec ? go(launch_any_t<4, E_, true>) : go(launch_any_t<4, E_, false>); \
    if (PB == 2) return vec ? go(launch_any_t<2, E_, true>) : go(launch_any_t<2, E_, false>); \
    return vec ? go(launch_any_t<1, E_, true>) : go(launch_any_t<1, E_, false>);
  switch (ell) {
    GC_ANY(1)
    GC_ANY(2)
    GC_ANY(3)
    GC_ANY(4)
    default: return fail(GC_ERR_UNSUPPORTED, "ell=%d", ell);
  }
#undef GC_ANY
}

}  // namespace gc
