// Chunk gradients: the host-side plan, the launches and the reduction of the
// partial gradients (the gradient kernel and its design: k_chunkgrad.cuh).
#include <algorithm>
#include <atomic>

#include "k_chunkgrad.cuh"

namespace gc {

namespace {

// G[i][col] = sum of the partials of chunk i, clusters in increasing order.
// Chunk i is the batches [i nbc, (i + 1) nbc) and cluster q took
// [q bpc, (q + 1) bpc); the first of its clusters may have begun in an earlier
// chunk (its slot for chunk i is then not slot 0), the others begin inside i.
// Block (x, i): 1024 columns, four a thread (one 16-byte piece when VEC, else
// 256 apart).  Memory bound, a few reads per output: the work a thread is what
// hides the latency (d = 65536, 64 chunks, 26 MB of partials: one column a
// thread 37 us).  Launched as a programmatic dependent of k_chunkgrad: the
// blocks are resident before the gradient kernel ends and wait for it here.
template <bool VEC>
__global__ void __launch_bounds__(256) k_chunkgrad_reduce(const float* __restrict__ parts,
                                                          const double* __restrict__ loss_parts,
                                                          float* __restrict__ G, double* loss_out,
                                                          int N, int nbc, int d, long long bpc,
                                                          int maxt, int nloss, long long Ntil) {
  const int i = blockIdx.y;
  const long long qlo = ((long long)i * nbc) / bpc;
  const long long qhi = ((long long)(i + 1) * nbc - 1) / bpc;
  const int np = (int)(qhi - qlo) + 1;
  const long long step = (long long)maxt * d;
  const float* first = parts + qlo * step + (i - (qlo * bpc) / nbc) * (long long)d;
  const float* rest = parts + qlo * step;  // + t * step: the t-th cluster after the first
  const int c0 = blockIdx.x * 1024 + (VEC ? 4 : 1) * threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // k_chunkgrad has completed
  // independent loads in groups of 8 clusters, added in increasing order
  if constexpr (VEC) {
    if (c0 < d) {
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int t0 = 0; t0 < np; t0 += 8) {
        float4 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (t0 + k < np)
            v[k] = __ldg(reinterpret_cast<const float4*>(
                (t0 + k == 0 ? first : rest + (t0 + k) * step) + c0));
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (t0 + k < np) {
            acc.x += v[k].x;
            acc.y += v[k].y;
            acc.z += v[k].z;
            acc.w += v[k].w;
          }
      }
      *reinterpret_cast<float4*>(G + (size_t)i * d + c0) = acc;
    }
  } else {
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int t0 = 0; t0 < np; t0 += 4) {
      float v[4][4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          v[k][u] = t0 + k < np && c0 + 256 * u < d
                        ? __ldg((t0 + k == 0 ? first : rest + (t0 + k) * step) + c0 + 256 * u)
                        : 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (t0 + k < np) acc[u] += v[k][u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 256 * u < d) G[(size_t)i * d + c0 + 256 * u] = acc[u];
  }
  if (loss_out && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 32) {
    // lane l adds parts l, l + 32, ...; then a fixed xor tree
    double t = 0.0;
    for (int q = threadIdx.x; q < nloss; q += 32) t += loss_parts[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) *loss_out = t / (double)Ntil;
  }
}

// ---------------------------------------------------------------------------
// Host-side plan
// ---------------------------------------------------------------------------
struct Plan {
  int CL, NT, NVT, RBM, S, Wc, ld_s, V;
  bool aligned;  // every row slice starts on a 16-byte boundary
  bool valid;
  int nbc;            // batches per chunk
  long long nbatch;   // batches in all
  long long bpc;      // batches per cluster
  int nclusters, maxt;
  size_t smem;
  bool by_warp;       // short rows: the clusters are single warps
  int blocks;         // of the short-row kernel
};

cg::Kernel kernel_of(const Plan& p, int x_dtype) {
  if (x_dtype == GC_BF16)
    return p.aligned ? cg::pick_bf16(p.CL, p.NT, p.NVT) : cg::pick_bf16_ragged(p.CL, p.NT, p.NVT);
  return p.aligned ? cg::pick_f32(p.CL, p.NT, p.NVT) : cg::pick_f32_ragged(p.CL, p.NT, p.NVT);
}

// Position of a shape in the per-kernel caches below.
constexpr int kShapes = 2 * 2 * 4 * 3 * 8;
int shape_index(const Plan& p, int x_dtype) {
  const int ci = p.CL == 1 ? 0 : (p.CL == 2 ? 1 : (p.CL == 4 ? 2 : 3));
  const int ni = p.NT == 512 ? 0 : (p.NT == 256 ? 1 : 2);
  return ((((x_dtype == GC_BF16) * 2 + p.aligned) * 4 + ci) * 3 + ni) * 8 + (p.NVT - 1);
}

// Allow the kernel its dynamic shared memory (all there is: a shape's depends on the ring).
cudaError_t allow_smem(cg::Kernel kern, const Plan& p, int x_dtype) {
  static SmemOptIn allow[kShapes];
  return allow[shape_index(p, x_dtype)](kern, kSmemMax);
}

cudaLaunchConfig_t launch_config(const Plan& p, unsigned grid, cudaLaunchAttribute* attr,
                                 cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(p.NT + 64);  // consumers, the producer and the reducer warp
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = p.CL;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Clusters of this plan that can be resident at once (cached per shape).
int max_active_clusters(const Plan& p, int x_dtype) {
  static std::atomic<int> cache[kShapes];
  std::atomic<int>& c = cache[shape_index(p, x_dtype)];
  int n = c.load(std::memory_order_relaxed);
  if (n > 0) return n;
  cg::Kernel kern = kernel_of(p, x_dtype);
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = launch_config(p, p.CL * 64, attr, nullptr);
  if (!kern || allow_smem(kern, p, x_dtype) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = 1;
  }
  c.store(n, std::memory_order_relaxed);
  return n;
}

Plan make_plan(int N, int n_c, int d, int x_dtype, bool x_aligned) {
  Plan p{};
  const int esz = x_dtype == GC_BF16 ? 2 : 4;
  p.V = 16 / esz;
  const long long row_bytes = (long long)d * esz;
  // The row is split over as few CTAs as its columns' w and accumulators fit
  // the registers of (512 threads of 6 fp32 or 4 bf16 vectors), so that the rows
  // of a batch and the partial gradients are as long as they can be (2 GB of X,
  // with the exchange of the time in the consumers' way: fp32 d = 10007 102% of
  // the copy rate in one CTA, 54% in two; bf16 d = 16384 98 and 74).
  // Fewer than five rows an SM leave SMs idle that way, or write a partial gradient for
  // every few rows (bf16 d = 16384: 32 rows 16.0 us, 11.9 with slices of half the size, 640
  // rows 24.3 and 20.2; d = 10007, 1024 rows 12.1 and 14.6; fp32 d = 24576, 32 rows 10.3 and 9.1).
  const bool few = (long long)N * n_c < 5LL * device_sm_count();
  const long long max_slice = x_dtype == GC_BF16 ? (few ? 16384 : 32768) : (few ? 32768 : 49152);
  p.CL = 1;
  while (p.CL < 8 && (row_bytes + p.CL - 1) / p.CL > max_slice) p.CL *= 2;
  // Clusters of 8 fill only 120 of the 152 SMs (a cluster lives inside one
  // GPC; at most 15 clusters of 8 are co-resident), clusters of 4 fill 144:
  // fp32 rows of up to 256 KB take 64 KB slices (8 vectors a thread, one row a
  // stage) in clusters of 4, bf16 rows of up to 128 KB 32 KB slices.  bf16 rows that two CTAs would take in four
  // vectors a thread stay in clusters of 4 (d = 32768: 70 against 68%, at
  // 256 MB 43 against 40%, before x was kept in tensor memory).
  if (p.CL == 8 && row_bytes <= 4 * (x_dtype == GC_BF16 ? 32768 : 65536)) p.CL = 4;
  if (x_dtype == GC_BF16 && p.CL == 2 && row_bytes > 2 * 3 * 512 * 16) p.CL = 4;
  p.Wc = (int)align_up((size_t)((d + p.CL - 1) / p.CL), (size_t)p.V);
  p.aligned = x_aligned && row_bytes % 16 == 0;
  const int nv = p.Wc / p.V;  // 16-byte vectors per row slice (<= 2048 by the slice caps)
  p.NT = nv >= 1024 ? 512 : (nv >= 256 ? 256 : 128);
  // CTAs per SM.  Rows of 4 to 16 KB: two (two independent rings) when each
  // still streams many rows, one when the rows per SM are few (ramp-up
  // dominates) or the row is longer.  Shorter rows, 128 threads: the chain of a
  // batch from its dot products to its residuals outlasts its copy, so up to
  // three CTAs, with at least 32 rows each.  (Rows of at most 128 fp32 or 96 bf16
  // vectors come here with an armed stall alone, see launch_chunkgrad.)
  const long long rows_per_sm = (long long)N * n_c / std::max(1, device_sm_count());
  int cps = (rows_per_sm >= 512 && row_bytes <= 16384) ? 2 : 1;
  if (p.NT == 128)
    cps = (int)std::max(1LL, std::min(3LL, rows_per_sm / 32));
  if (cps == 2 && p.NT == 512) p.NT = 256;  // only when nv <= 1024 (16 KB slices)
  const int need = (nv + p.NT - 1) / p.NT;
  // vectors a thread: 1, 2, 4, and for 512-thread slices past 4 vectors (fp32)
  // or 2 (bf16) the exact count, whose empty vectors would cost stage space
  // and dot products
  p.NVT = need <= 2 ? (p.NT == 128 && esz == 4 ? 2 : need) : 4;
  if (x_dtype == GC_BF16 ? need == 3 && p.NT == 512 : need > 4) p.NVT = need <= 6 ? need : 8;
  p.RBM = p.NVT >= 5 ? 1 : (p.NVT >= 3 ? 2 : (p.NVT == 2 ? 4 : 8));
  // stage row: one vector per (thread, u), so reads need no bounds; a slice at
  // any element lies up to V - 1 elements in and ends in up to 2 V - 1 more
  const int row_vecs = p.NVT * p.NT;
  p.ld_s = row_vecs * p.V + (p.aligned ? 0 : 2 * p.V);
  const size_t stage_bytes = (size_t)p.RBM * p.ld_s * esz;
  p.S = (int)std::min<size_t>(
      cg::kMaxStages, std::max<size_t>(2, (192 * 1024 / cps) / ((size_t)p.RBM * row_vecs * 16)));
  const int NW = p.NT / 32;
  p.smem = p.S * stage_bytes +
           (cg::kSlots * NW * p.RBM + cg::kZSlots * p.CL * p.RBM + cg::kSlots * p.RBM) * sizeof(float) +
           (2 * cg::kMaxStages + 2 * cg::kSlots + cg::kZSlots) * sizeof(uint64_t) + 16;
  // every vector of the slice has a thread, and the shape is built
  p.valid = (long long)row_vecs >= nv && kernel_of(p, x_dtype) != nullptr;
  // flat partition of the batches over one wave of clusters
  const int sms = device_sm_count();
  long long waves_cl = std::max(1, sms * cps / p.CL);
  if (p.CL > 1) waves_cl = std::max(1, std::min<int>((int)waves_cl, max_active_clusters(p, x_dtype)));
  p.nbc = (n_c + p.RBM - 1) / p.RBM;
  p.nbatch = (long long)N * p.nbc;
  p.bpc = (p.nbatch + waves_cl - 1) / waves_cl;
  p.nclusters = (int)((p.nbatch + p.bpc - 1) / p.bpc);
  p.maxt = (int)((p.bpc + p.nbc - 1) / p.nbc) + 1;
  return p;
}

// Short rows: a block per share of the batches, two blocks an SM when every
// warp of them has one.
Plan make_short_plan(int N, int n_c, int d, int x_dtype, bool x_aligned) {
  Plan p{};
  const int esz = x_dtype == GC_BF16 ? 2 : 4;
  p.V = 16 / esz;
  const int nv = (d + p.V - 1) / p.V;
  if (nv > cg::short_vecs(x_dtype == GC_BF16)) return p;
  p.CL = 1;
  p.NVT = (nv + 31) / 32;
  p.NT = cg::kShortThreads;
  p.RBM = cg::short_rows(p.NVT, x_dtype == GC_BF16);
  p.aligned = x_aligned && (long long)d * esz % 16 == 0;
  p.valid = true;
  p.nbc = (n_c + p.RBM - 1) / p.RBM;
  p.nbatch = (long long)N * p.nbc;
  const int warps = p.NT / 32;
  // Chunks of few batches go to single warps, as a block's would meet after each of
  // them with most having nothing to add (256 chunks of 4 rows: 5.4 us, by blocks 14);
  // chunks that give every warp a batch do not, unless a warp's range is whole chunks:
  // their partials would be as many bytes as the rows (256 chunks of 16 rows of 768
  // bf16: by warps 13 us, by blocks 7.9).
  p.by_warp = p.nbc < warps || N >= 2 * warps * device_sm_count();
  const long long blocks =
      std::max(1LL, std::min((p.nbatch + warps - 1) / warps, 2LL * device_sm_count()));
  const long long ranges = p.by_warp ? blocks * warps : blocks;
  p.bpc = (p.nbatch + ranges - 1) / ranges;
  p.nclusters = (int)((p.nbatch + p.bpc - 1) / p.bpc);
  p.blocks = p.by_warp ? (p.nclusters + warps - 1) / warps : p.nclusters;
  p.maxt = (int)((p.bpc + p.nbc - 1) / p.nbc) + 1;
  return p;
}

}  // namespace

size_t chunkgrad_ws_bytes(int N, int n_c, int d, int x_dtype) {
  const Plan p = make_plan(N, n_c, d, x_dtype, true);
  const Plan p2 = make_plan(N, n_c, d, x_dtype, false);
  const Plan p3 = make_short_plan(N, n_c, d, x_dtype, true);  // alignment does not change its sizes
  const size_t parts = std::max({(size_t)p.nclusters * p.maxt, (size_t)p2.nclusters * p2.maxt,
                                 (size_t)p3.nclusters * p3.maxt}) *
                       (size_t)d * sizeof(float);
  const size_t lp = (size_t)std::max({p.nclusters, p2.nclusters, p3.nclusters}) * sizeof(double);
  return align_up(parts, 256) + align_up(lp, 256);
}

int launch_chunkgrad(const void* X, int x_dtype, const float* y, const float* w, int N, int n_c,
                     int d, int loss, float* G, double* loss_out, Carve& ws, uint32_t* status,
                     cudaStream_t s) {
  const bool aligned = (reinterpret_cast<uintptr_t>(X) % 16) == 0;
  const bool stall = take_stall(GC_STALL_CHUNK_GRADS);
  // an armed stall withholds the ring kernel's copies: that kernel then
  const Plan ps = stall ? Plan{} : make_short_plan(N, n_c, d, x_dtype, aligned);
  const Plan p = ps.valid ? ps : make_plan(N, n_c, d, x_dtype, aligned);
  if (!p.valid) return fail(GC_ERR_UNSUPPORTED, "chunk-gradient plan does not cover d=%d", d);
  cg::CGArgs a{};
  a.X = X;
  a.y = y;
  a.w = w;
  a.d = d;
  a.Wc = p.Wc;
  a.ld_s = p.ld_s;
  a.n_c = n_c;
  a.Ntil = (long long)N * n_c;
  a.nbc = p.nbc;
  a.nbatch = p.nbatch;
  a.bpc = p.bpc;
  a.S = p.S;
  a.maxt = p.maxt;
  a.by_warp = p.by_warp;
  a.loss = loss;
  a.want_loss = loss_out != nullptr;
  a.spin_limit = wait_limit(cg::kSpinLimit);
  a.stall = stall ? 1 : 0;
  a.parts = ws.take<float>((size_t)p.nclusters * p.maxt * d);
  a.loss_parts = ws.take<double>(p.nclusters);
  a.status = status;
  // a limit of the interface, kept as it was: a single chunk of at least 512
  // rows per SM of short rows is refused
  if (N == 1 && (long long)n_c / std::max(1, device_sm_count()) >= 512 &&
      (long long)d * (x_dtype == GC_BF16 ? 2 : 4) <= 16384)
    return fail(GC_ERR_UNSUPPORTED, "one chunk of %d short rows: at most 512 per SM", n_c);
  if (N > 65535) return fail(GC_ERR_UNSUPPORTED, "N=%d exceeds 65535 chunks", N);
  cudaError_t e = cudaSuccess;
  if (ps.valid) {
    cg::pick_short(x_dtype == GC_BF16, p.aligned, p.NVT)<<<p.blocks, p.NT, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_check(e, "k_chunkgrad_short");
    count_launches(1);
  } else {
    cg::Kernel kern = kernel_of(p, x_dtype);
    e = allow_smem(kern, p, x_dtype);
    if (e != cudaSuccess) return cuda_check(e, "cudaFuncSetAttribute(chunkgrad smem)");
    cudaLaunchAttribute cl_attr[1];
    const cudaLaunchConfig_t cl_cfg = launch_config(p, (unsigned)(p.nclusters * p.CL), cl_attr, s);
    e = cudaLaunchKernelEx(&cl_cfg, kern, a);
    if (e != cudaSuccess) return cuda_check(e, "cudaLaunchKernelEx(chunkgrad)");
    count_launches(1);
  }
  // the reduction as a programmatic dependent launch (it waits in-kernel)
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((d + 1023) / 1024, N);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const bool vec = d % 4 == 0 && reinterpret_cast<uintptr_t>(G) % 16 == 0;
  e = cudaLaunchKernelEx(&cfg, vec ? k_chunkgrad_reduce<true> : k_chunkgrad_reduce<false>,
                         (const float*)a.parts, (const double*)a.loss_parts, G, loss_out, N, p.nbc,
                         d, p.bpc, p.maxt, ps.valid ? p.blocks : p.nclusters, a.Ntil);
  if (e != cudaSuccess) return cuda_check(e, "cudaLaunchKernelEx(k_chunkgrad_reduce)");
  count_launches(1);
  return GC_OK;
}

}  // namespace gc
