// Device code shared by the kernels that solve Algorithm 1's blocks
// (k_solve.cu, k_mse_patterns.cu): one block, the memo table, completion masks.
#pragma once

#include "gc_internal.cuh"

namespace gc {

// ---------------------------------------------------------------------------
// One least-squares block: chunk i, completion mask over its holders.
// emit(h, k, v) receives X^+ row of holder h (0 for holders not in S_i).
// Returns Delta; Pi (ell x ell) and err = ||I - Pi||_F^2 by reference.
// ---------------------------------------------------------------------------
template <bool SHARED>
__device__ __forceinline__ double r_load(const double* p) {
  if constexpr (SHARED) return *p;
  return __ldg(p);
}
// SHARED: R lies in shared memory.
template <int ELL, bool SHARED = false, typename Emit>
__device__ __forceinline__ int solve_block(const double* __restrict__ R, int m, int cnt,
                                           const int16_t* __restrict__ hw, uint32_t mask,
                                           double (&Pi)[ELL][ELL], double& err, uint32_t* status,
                                           Emit emit) {
  const int D = __popc(mask);
#pragma unroll
  for (int a = 0; a < ELL; ++a)
#pragma unroll
    for (int k = 0; k < ELL; ++k) Pi[a][k] = 0.0;

  if (D >= ELL) {
    // Gram matrix M = X X^T (lower triangle) and its Cholesky factor.
    double Lc[ELL][ELL];
#pragma unroll
    for (int a = 0; a < ELL; ++a)
#pragma unroll
      for (int c = 0; c < ELL; ++c) Lc[a][c] = 0.0;
    for (int h = 0; h < cnt; ++h) {
      if (!((mask >> h) & 1u)) continue;
      const int j = hw[h];
      double x[ELL];
#pragma unroll
      for (int a = 0; a < ELL; ++a) x[a] = r_load<SHARED>(R + (size_t)a * m + j);
#pragma unroll
      for (int a = 0; a < ELL; ++a)
#pragma unroll
        for (int c = 0; c <= a; ++c) Lc[a][c] = fma(x[a], x[c], Lc[a][c]);
    }
    // The diagonal is kept as reciprocals (one rsqrt per pivot): GB300's
    // fp64 divisions and square roots are long instruction sequences.
    bool bad = false;
    double rdiag[ELL];
#pragma unroll
    for (int a = 0; a < ELL; ++a) {
      double s = Lc[a][a];
#pragma unroll
      for (int c = 0; c < a; ++c) s -= Lc[a][c] * Lc[a][c];
      const double ref = Lc[a][a];
      // pivot^2 / M_aa below 1e-14 (kappa(X) of order 1e7 or more): numerically
      // rank deficient in fp64; flagged, and clamped so the result stays finite
      if (!(s > 1e-14 * ref) || !isfinite(s)) {
        bad = true;
        s = ref > 0.0 ? 1e-14 * ref : 1e-300;
      }
      const double rp = rsqrt(s);
      rdiag[a] = rp;
#pragma unroll
      for (int r = a + 1; r < ELL; ++r) {
        double t = Lc[r][a];
#pragma unroll
        for (int c = 0; c < a; ++c) t -= Lc[r][c] * Lc[a][c];
        Lc[r][a] = t * rp;
      }
    }
    if (bad) atomicOr(status, ST_SINGULAR);
    // Cholesky solve of M Y = Bm in place (column by column).
    auto chol_solve = [&](double (&Bm)[ELL][ELL]) {
#pragma unroll
      for (int k = 0; k < ELL; ++k) {
        double yv[ELL];
#pragma unroll
        for (int a = 0; a < ELL; ++a) {
          double t = Bm[a][k];
#pragma unroll
          for (int c = 0; c < a; ++c) t -= Lc[a][c] * yv[c];
          yv[a] = t * rdiag[a];
        }
#pragma unroll
        for (int a = ELL - 1; a >= 0; --a) {
          double t = yv[a];
#pragma unroll
          for (int c = a + 1; c < ELL; ++c) t -= Lc[c][a] * Bm[c][k];
          Bm[a][k] = t * rdiag[a];
        }
      }
    };
    double Lam[ELL][ELL];
#pragma unroll
    for (int a = 0; a < ELL; ++a)
#pragma unroll
      for (int k = 0; k < ELL; ++k) Lam[a][k] = (a == k) ? 1.0 : 0.0;
    chol_solve(Lam);
    // One refinement step on the residual of X b_k = e_k, b_k = X^T Lambda e_k.
    double Res[ELL][ELL];
#pragma unroll
    for (int a = 0; a < ELL; ++a)
#pragma unroll
      for (int k = 0; k < ELL; ++k) Res[a][k] = (a == k) ? 1.0 : 0.0;
    for (int h = 0; h < cnt; ++h) {
      if (!((mask >> h) & 1u)) continue;
      const int j = hw[h];
      double x[ELL];
#pragma unroll
      for (int a = 0; a < ELL; ++a) x[a] = r_load<SHARED>(R + (size_t)a * m + j);
#pragma unroll
      for (int k = 0; k < ELL; ++k) {
        double bk = 0.0;
#pragma unroll
        for (int c = 0; c < ELL; ++c) bk = fma(x[c], Lam[c][k], bk);
#pragma unroll
        for (int a = 0; a < ELL; ++a) Res[a][k] = fma(-x[a], bk, Res[a][k]);
      }
    }
    chol_solve(Res);
#pragma unroll
    for (int a = 0; a < ELL; ++a)
#pragma unroll
      for (int k = 0; k < ELL; ++k) Lam[a][k] += Res[a][k];
    // Coefficients and the projector Pi = X X^+.
    for (int h = 0; h < cnt; ++h) {
      if (!((mask >> h) & 1u)) {
#pragma unroll
        for (int k = 0; k < ELL; ++k) emit(h, k, 0.0);
        continue;
      }
      const int j = hw[h];
      double x[ELL];
#pragma unroll
      for (int a = 0; a < ELL; ++a) x[a] = r_load<SHARED>(R + (size_t)a * m + j);
#pragma unroll
      for (int k = 0; k < ELL; ++k) {
        double bk = 0.0;
#pragma unroll
        for (int c = 0; c < ELL; ++c) bk = fma(x[c], Lam[c][k], bk);
        emit(h, k, bk);
#pragma unroll
        for (int a = 0; a < ELL; ++a) Pi[a][k] = fma(x[a], bk, Pi[a][k]);
      }
    }
  } else if (D > 0) {
    constexpr int MQ = ELL > 1 ? ELL - 1 : 1;
    int jq[MQ];
    {
      int q = 0;
      for (int h = 0; h < cnt; ++h) {
        if (!((mask >> h) & 1u)) continue;
#pragma unroll
        for (int qq = 0; qq < MQ; ++qq)
          if (qq == q) jq[qq] = hw[h];
        ++q;
      }
    }
    double Xc[MQ][ELL], Q[MQ][ELL], Rr[MQ][MQ], Xp[MQ][ELL], rr[MQ];
#pragma unroll
    for (int qq = 0; qq < MQ; ++qq) {
#pragma unroll
      for (int r = 0; r < MQ; ++r) Rr[r][qq] = 0.0;
#pragma unroll
      for (int a = 0; a < ELL; ++a) {
        Xc[qq][a] = (qq < D) ? r_load<SHARED>(R + (size_t)a * m + jq[qq]) : 0.0;
        Q[qq][a] = 0.0;
        Xp[qq][a] = 0.0;
      }
    }
    bool bad = false;
#pragma unroll
    for (int qq = 0; qq < MQ; ++qq) {
      if (qq < D) {
        double v[ELL];
        double n0 = 0.0;
#pragma unroll
        for (int a = 0; a < ELL; ++a) {
          v[a] = Xc[qq][a];
          n0 = fma(v[a], v[a], n0);
        }
#pragma unroll
        for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
          for (int r = 0; r < MQ; ++r) {
            if (r < qq) {
              double dot = 0.0;
#pragma unroll
              for (int a = 0; a < ELL; ++a) dot = fma(Q[r][a], v[a], dot);
#pragma unroll
              for (int a = 0; a < ELL; ++a) v[a] = fma(-dot, Q[r][a], v[a]);
              Rr[r][qq] += dot;
            }
          }
        }
        double nn = 0.0;
#pragma unroll
        for (int a = 0; a < ELL; ++a) nn = fma(v[a], v[a], nn);
        if (!(nn > 1e-14 * n0) || !isfinite(nn)) {  // same criterion as the Cholesky pivot
          bad = true;
          nn = n0 > 0.0 ? 1e-14 * n0 : 1e-300;
        }
        const double rn = rsqrt(nn);
        Rr[qq][qq] = nn * rn;
        rr[qq] = rn;
#pragma unroll
        for (int a = 0; a < ELL; ++a) Q[qq][a] = v[a] * rn;
      }
    }
    if (bad) atomicOr(status, ST_SINGULAR);
    // X^+ = Rr^{-1} Q^T by back substitution.
#pragma unroll
    for (int qq = MQ - 1; qq >= 0; --qq) {
      if (qq < D) {
#pragma unroll
        for (int k = 0; k < ELL; ++k) {
          double t = Q[qq][k];
#pragma unroll
          for (int r = qq + 1; r < MQ; ++r)
            if (r < D) t -= Rr[qq][r] * Xp[r][k];
          Xp[qq][k] = t * rr[qq];
        }
      }
    }
    // Pi = X X^+
#pragma unroll
    for (int qq = 0; qq < MQ; ++qq)
      if (qq < D) {
#pragma unroll
        for (int a = 0; a < ELL; ++a)
#pragma unroll
          for (int k = 0; k < ELL; ++k) Pi[a][k] = fma(Xc[qq][a], Xp[qq][k], Pi[a][k]);
      }
    int q = 0;
    for (int h = 0; h < cnt; ++h) {
      const bool in = (mask >> h) & 1u;
#pragma unroll
      for (int k = 0; k < ELL; ++k) {
        double v = 0.0;
        if (in) {
#pragma unroll
          for (int qq = 0; qq < MQ; ++qq)
            if (qq == q) v = Xp[qq][k];
        }
        emit(h, k, v);
      }
      if (in) ++q;
    }
  } else {
    for (int h = 0; h < cnt; ++h)
#pragma unroll
      for (int k = 0; k < ELL; ++k) emit(h, k, 0.0);
  }
  double e = 0.0;
#pragma unroll
  for (int a = 0; a < ELL; ++a)
#pragma unroll
    for (int k = 0; k < ELL; ++k) {
      const double t = ((a == k) ? 1.0 : 0.0) - Pi[a][k];
      e = fma(t, t, e);
    }
  err = e;
  return D;
}

// Table of every holder subset: entry (i, mask) holds X^+ (cnt x ell), Pi and err.
struct Table {
  int bits;     // masks per chunk = 1 << bits
  double* xp;   // [N][1<<bits][bits][ell]
  float* pi;    // [N][1<<bits][ell][ell] (fp32: the decode matrix is emitted in fp32)
  double* err;  // [N][1<<bits]
};

// The layout of a table of `bits` masks per chunk (log2) in caller memory.
inline Table table_at(void* mem, int N, int ell, int bits) {
  Table tb{bits < 0 ? 0 : bits, nullptr, nullptr, nullptr};
  if (bits < 0 || !mem) return tb;
  const size_t ent = (size_t)N << bits;
  char* p = static_cast<char*>(mem);
  tb.xp = reinterpret_cast<double*>(p);
  p += align_up(ent * bits * ell * sizeof(double), 256);
  tb.pi = reinterpret_cast<float*>(p);
  p += align_up(ent * ell * ell * sizeof(float), 256);
  tb.err = reinterpret_cast<double*>(p);
  return tb;
}

// Chunks lane, lane + 32, ... (CPL of them) of a warp that takes whole
// patterns: their first eight holders (worker and slot) stay in registers.
template <int CPL>
struct LaneHolders {
  int cnt[CPL];
  uint4 hw8[CPL];
  uint2 hp8[CPL];
  __device__ __forceinline__ void load(const Holders& hd, int N, int lane) {
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      const int i = lane + 32 * c;
      cnt[c] = 0;
      hw8[c] = make_uint4(0u, 0u, 0u, 0u);
      hp8[c] = make_uint2(0u, 0u);
      if (i < N) {
        cnt[c] = hd.cnt[i];
        hw8[c] = *reinterpret_cast<const uint4*>(hd.w + (size_t)i * GC_MAX_REPL);
        hp8[c] = *reinterpret_cast<const uint2*>(hd.p + (size_t)i * GC_MAX_REPL);
      }
    }
  }
  // completion masks of the lane's chunks under the counts ps; a count outside
  // [0, delta] is taken as 0 and reported
  __device__ __forceinline__ bool masks(const Holders& hd, const int32_t* __restrict__ ps,
                                        uint32_t udelta, int lane, uint32_t (&mask)[CPL]) const {
    bool bad = false;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      uint32_t mk = 0;
      const uint32_t ww[4] = {hw8[c].x, hw8[c].y, hw8[c].z, hw8[c].w};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q < cnt[c]) {
          const int wq = (int)(int16_t)(ww[q >> 1] >> (16 * (q & 1)));
          const int pq = (int)(int8_t)(((q < 4 ? hp8[c].x : hp8[c].y) >> (8 * (q & 3))) & 0xffu);
          uint32_t v = (uint32_t)__ldg(ps + wq);
          if (v > udelta) {
            bad = true;
            v = 0;
          }
          if (pq < (int)v) mk |= 1u << q;
        }
      }
      // holders past the eighth (chunks with more than eight copies), eight a load
      for (int h0 = 8; h0 < cnt[c]; h0 += 8) {
        const size_t row = (size_t)(lane + 32 * c) * GC_MAX_REPL + h0;
        const uint4 w8 = *reinterpret_cast<const uint4*>(hd.w + row);
        const uint2 p8 = *reinterpret_cast<const uint2*>(hd.p + row);
        const uint32_t wx[4] = {w8.x, w8.y, w8.z, w8.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (h0 + q < cnt[c]) {
            const int wq = (int)(int16_t)(wx[q >> 1] >> (16 * (q & 1)));
            const int pq = (int)(int8_t)(((q < 4 ? p8.x : p8.y) >> (8 * (q & 3))) & 0xffu);
            uint32_t v = (uint32_t)__ldg(ps + wq);
            if (v > udelta) {
              bad = true;
              v = 0;
            }
            if (pq < (int)v) mk |= 1u << (h0 + q);
          }
        }
      }
      mask[c] = mk;
    }
    return bad;
  }
};

}  // namespace gc
