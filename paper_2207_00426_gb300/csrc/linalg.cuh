// Small dense linear algebra held in registers (one thread per matrix).
//
// Matrices are row-major arrays with compile-time shapes; every loop is fully
// unrolled so that the arrays stay in registers.  Tria (Sec. 2.2) is an LQ
// factorisation by Householder reflections applied from the right.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#define SQSM_DEV __device__ __forceinline__

namespace sqsm {

template <typename T> struct Tiny;
template <> struct Tiny<float> { static constexpr float value = 1e-30f; };
template <> struct Tiny<double> { static constexpr double value = 1e-280; };

SQSM_DEV float sq_sqrt(float x) { return sqrtf(x); }
SQSM_DEV double sq_sqrt(double x) { return sqrt(x); }
SQSM_DEV float sq_log(float x) { return logf(x); }
SQSM_DEV double sq_log(double x) { return log(x); }

// Square root and reciprocal for the reflector of one Householder step and
// the diagonal of triangular solves (normal x > 0).  FP32 starts from the hardware reciprocal square root and
// reciprocal estimates and takes one Newton step each (on y^2 = x from
// y = x rsqrt(x), and on 1/x, as in Markstein's refinements), which keeps
// them within about an ulp without the slow-path branch of the IEEE
// operations, so that a whole Tria is one branch-free block the compiler can
// schedule across reflections.  FP64 keeps the correctly rounded operations.
SQSM_DEV float hh_sqrt(float x) {
  const float r = rsqrtf(x);
  const float y = x * r;
  return fmaf(fmaf(-y, y, x), 0.5f * r, y);
}
SQSM_DEV double hh_sqrt(double x) { return sqrt(x); }
SQSM_DEV float hh_rcp(float x) {
  const float r = __fdividef(1.0f, x);
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}
SQSM_DEV double hh_rcp(double x) { return 1.0 / x; }

// Products and fused multiply-adds the compiler may not regroup.
SQSM_DEV float mul_rn(float a, float b) { return __fmul_rn(a, b); }
SQSM_DEV double mul_rn(double a, double b) { return __dmul_rn(a, b); }
SQSM_DEV float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
SQSM_DEV double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// x / c for a constant c > 1: the product with the rounded reciprocal,
// corrected by the remainder (a division by a divisor known in advance;
// Brisebarre, Muller and Raina, IEEE Trans. Computers 2004).  Equal to the
// rounded quotient, for the divisors the sigma-point rules use (10, 12 and
// once and twice sqrt(5), sqrt(6)) and away from underflow: in FP32 checked
// over every significand, in FP64 over every one whose quotient is near enough
// to a rounding boundary for the correction's error to matter.  An infinite x
// has no remainder and gives the product.
template <typename T> struct ConstDivisor {
  T c, rc;
  __host__ __device__ constexpr explicit ConstDivisor(T c_) : c(c_), rc(T(1) / c_) {}
};
// (in FP64 by the exponent's bits: a comparison would hold the FP64 unit)
SQSM_DEV bool finite_bits(float x) { return isfinite(x); }
SQSM_DEV bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
template <typename T>
SQSM_DEV T div_const(T x, const ConstDivisor<T>& d) {
  const T q = mul_rn(x, d.rc);
  const T r = fma_rn(fma_rn(-q, d.c, x), d.rc, q);
  return finite_bits(q) ? r : q;
}

// Which entries of a matrix handed to Tria can be nonzero: row(i) is the bit
// mask of the columns of row i that may be (bit j: column j).  Nearly every
// matrix the method triangularises is a block matrix with triangular, empty
// or identity blocks, and a reflection only ever spreads a row's columns onto
// the rows below it, so the columns each step has to touch are known at
// compile time: 6 of 10, 9, 8, ... in every n_x x 2 n_x Tria at n_x = 5.  The
// terms left out are products with an exact zero, so the factor is the full
// loops' (in FP32 bit for bit, the order of the remaining operations being
// kept).  The kernels are bound by instruction issue and fetch: 4096 sequences
// (1.04e7 steps, two FP32 iterations) 19.3 -> 16.8 ms, n = 1e5 linear smoother
// 258 -> 243 us, n = 4000 FP64 track 21.5 -> 18.7 ms per ten iterations.
template <int C> struct DenseRows {
  __host__ __device__ static constexpr uint32_t row(int) { return (1u << C) - 1; }
};
// [X | L]: X with D columns, L lower triangular.
template <int D> struct DenseThenLower {
  __host__ __device__ static constexpr uint32_t row(int i) { return ((1u << D) - 1) | (((2u << i) - 1) << D); }
};
// [X | Y] where only the first K of X's D columns are nonzero and Y has its
// first K2 columns full beside a lower triangle.
template <int K, int D, int K2> struct FewThenFewLower {
  __host__ __device__ static constexpr uint32_t row(int i) {
    return ((1u << K) - 1) | ((((2u << i) - 1) | ((1u << K2) - 1)) << D);
  }
};
// The first K columns only.
template <int K> struct FewColumns {
  __host__ __device__ static constexpr uint32_t row(int) { return (1u << K) - 1; }
};
// [X | I].
template <int K, int D> struct FewThenIdentity {
  __host__ __device__ static constexpr uint32_t row(int i) { return ((1u << K) - 1) | (1u << (D + i)); }
};
// [X^T | I] where only the first K of X's D columns (the first K rows of X^T)
// are nonzero.
template <int K, int D> struct FewRowsThenIdentity {
  __host__ __device__ static constexpr uint32_t row(int i) {
    return (i < K ? (1u << D) - 1 : 0u) | (1u << (D + i));
  }
};
// [[X, S], [N, 0]]: K rows of a dense D-column X beside a lower S, above a
// lower N.
template <int K, int D> struct DenseLowerOverLower {
  __host__ __device__ static constexpr uint32_t row(int i) {
    return i < K ? DenseThenLower<D>::row(i) : (2u << (i - K)) - 1;
  }
};

// The rows' masks at each step of Tria: at[i][r] before step i, v[i] the
// columns of step i's reflection (pivot column i included).
template <int R, int C, int NREF, typename PAT> struct TriaFill {
  uint32_t at[NREF + 1][R] = {}, v[NREF] = {};
  __host__ __device__ constexpr TriaFill() {
    for (int r = 0; r < R; ++r) at[0][r] = PAT::row(r) & (C < 32 ? (1u << C) - 1 : ~0u);
    for (int i = 0; i < NREF; ++i) {
      v[i] = ((at[i][i] >> i) << i) | (1u << i);
      for (int r = 0; r < R; ++r) {
        const bool hit = r > i && (at[i][r] & v[i]) != 0;
        at[i + 1][r] = at[i][r] | (hit ? v[i] : 0u);
      }
    }
  }
};

template <int R, int C, int NREF, typename PAT> struct TriaFillOf {
  static constexpr TriaFill<R, C, NREF, PAT> fill{};
};

// f(I), ..., f(N - 1) with the index as a compile-time constant (the masks
// above decide which statements exist; a loop the compiler only half unrolls
// would put the matrix in local memory).
template <int I, int N, typename F>
SQSM_DEV void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// Tria(A) for an R x C matrix `a` (Sec. 2.2): on return columns 0..R-1 of
// `a` hold the lower-triangular L with L L^T = A A^T and diag(L) >= 0 (the
// strictly upper part of those columns and columns R..C-1 are left as
// scratch).  Step i reflects row i onto its pivot: v = x + sign(x0)|x| e_0,
// applied to rows i+1.., after which column i of L is final; its sign is
// flipped so that L_ii = |x|.  A row whose remaining part is zero (rank
// deficiency) takes the identity reflector.  With NREF < R only the first
// NREF reflections are applied: rows 0..NREF-1 of L and columns 0..NREF-1 of
// the remaining rows are then final (used where only the leading block
// columns of the factor are needed).  PAT: the entries that can be nonzero;
// the others are not read.
template <typename T, int R, int C, typename PAT = DenseRows<C>, int NREF = R>
SQSM_DEV void tria(T* a) {
  static_assert(R <= C && C <= 32, "tria is only used on R x C blocks with R <= C <= 32");
  static_assert(NREF <= R, "at most R reflections");
  using F = TriaFillOf<R, C, NREF, PAT>;
  // Branch-free: a zero row selects the identity reflector (tau = 0, column
  // left as is).  Dot products use two partial sums to halve their chains.
  static_for<0, NREF>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr uint32_t pivot = F::fill.at[i][i], v = F::fill.v[i];
    T s2a = T(0), s2b = T(0);
    static_for<i, C>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      if constexpr (pivot >> j & 1) {
        if constexpr ((j - i) % 2 == 0) s2a += a[i * C + j] * a[i * C + j];
        else s2b += a[i * C + j] * a[i * C + j];
      }
    });
    const T s2 = s2a + s2b;
    T x0 = T(0);
    if constexpr (pivot >> i & 1) x0 = a[i * C + i];
    // (a NaN is no zero row: L_ii carries it on, also where no other entry of
    // the factor would read that column)
    const bool nz = !(s2 <= Tiny<T>::value);
    const T alpha = hh_sqrt(nz ? s2 : T(1));
    const T sgn = x0 >= T(0) ? T(1) : T(-1);
    const T v0 = x0 + sgn * alpha;
    const T tau = nz ? hh_rcp(alpha * (alpha + (x0 >= T(0) ? x0 : -x0))) : T(0);
    static_for<i + 1, R>([&](auto rc) {
      constexpr int r = decltype(rc)::value;
      constexpr uint32_t row = F::fill.at[i][r], both = row & v;
      if constexpr (both == 0) {
        a[r * C + i] = T(0);
      } else {
        // the order of the multiply-adds is written out: left to the
        // compiler, which of two products is fused depends on the code around
        T wa = T(0), wb = T(0), a0 = T(0);
        constexpr bool has0 = row >> i & 1, has1 = i + 1 < C && (both >> (i + 1) & 1);
        if constexpr (has0) a0 = a[r * C + i];
        if constexpr (has1) wa = mul_rn(a[r * C + i + 1], a[i * C + i + 1]);
        if constexpr (has0) wa = fma_rn(a0, v0, wa);
        static_for<i + 2, C>([&](auto jc) {
          constexpr int j = decltype(jc)::value;
          if constexpr (both >> j & 1) {
            if constexpr ((j - i) % 2) wa = fma_rn(a[r * C + j], a[i * C + j], wa);
            else wb = fma_rn(a[r * C + j], a[i * C + j], wb);
          }
        });
        const T w = (wa + wb) * tau;
        // column i of L, with the sign flip that makes L_ii = alpha > 0
        const T ci = -sgn * (a0 - w * v0);
        a[r * C + i] = nz ? ci : a0;
        static_for<i + 1, C>([&](auto jc) {
          constexpr int j = decltype(jc)::value;
          if constexpr (v >> j & 1) {
            if constexpr (row >> j & 1) a[r * C + j] = a[r * C + j] - w * a[i * C + j];
            else a[r * C + j] = T(0) - w * a[i * C + j];
          }
        });
      }
    });
    a[i * C + i] = nz ? alpha : T(0);
  });
}

// The same with every loop run in full and the order of the multiply-adds left
// to the compiler (see its uses).
template <typename T, int R, int C>
SQSM_DEV void tria_full(T* a) {
  static_assert(R <= C, "tria is only used on R x C blocks with R <= C");
  // Branch-free: a zero row selects the identity reflector (tau = 0, column
  // left as is).  Dot products use two partial sums to halve their chains.
#pragma unroll
  for (int i = 0; i < R; ++i) {
    T s2a = T(0), s2b = T(0);
#pragma unroll
    for (int j = i; j < C; j += 2) {
      s2a += a[i * C + j] * a[i * C + j];
      if (j + 1 < C) s2b += a[i * C + j + 1] * a[i * C + j + 1];
    }
    const T s2 = s2a + s2b;
    const T x0 = a[i * C + i];
    const bool nz = s2 > Tiny<T>::value;
    const T alpha = hh_sqrt(nz ? s2 : T(1));
    const T sgn = x0 >= T(0) ? T(1) : T(-1);
    const T v0 = x0 + sgn * alpha;
    const T tau = nz ? hh_rcp(alpha * (alpha + (x0 >= T(0) ? x0 : -x0))) : T(0);
#pragma unroll
    for (int r = i + 1; r < R; ++r) {
      T wa = a[r * C + i] * v0, wb = T(0);
#pragma unroll
      for (int j = i + 1; j < C; j += 2) {
        wa += a[r * C + j] * a[i * C + j];
        if (j + 1 < C) wb += a[r * C + j + 1] * a[i * C + j + 1];
      }
      const T w = (wa + wb) * tau;
      // column i of L, with the sign flip that makes L_ii = alpha > 0
      const T ci = -sgn * (a[r * C + i] - w * v0);
      a[r * C + i] = nz ? ci : a[r * C + i];
#pragma unroll
      for (int j = i + 1; j < C; ++j) a[r * C + j] -= w * a[i * C + j];
    }
    a[i * C + i] = nz ? alpha : T(0);
  }
}

// Copy the R x R lower factor out of the first R columns of an R x C array.
template <typename T, int R, int C>
SQSM_DEV void take_lower(const T* a, T* L) {
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int j = 0; j < R; ++j) L[r * R + j] = (j <= r && j < C) ? a[r * C + j] : T(0);
}

// C[M][N] = A[M][K] B[K][N]
template <typename T, int M, int K, int N>
SQSM_DEV void mm(const T* A, const T* B, T* Cm) {
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) {
      T s = T(0);
#pragma unroll
      for (int k = 0; k < K; ++k) s += A[i * K + k] * B[k * N + j];
      Cm[i * N + j] = s;
    }
}

// C[M][N] = A[K][M]^T B[K][N]
template <typename T, int M, int K, int N>
SQSM_DEV void mtm(const T* A, const T* B, T* Cm) {
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) {
      T s = T(0);
#pragma unroll
      for (int k = 0; k < K; ++k) s += A[k * M + i] * B[k * N + j];
      Cm[i * N + j] = s;
    }
}

// C[M][N] = A[M][K] B[N][K]^T
template <typename T, int M, int K, int N>
SQSM_DEV void mmt(const T* A, const T* B, T* Cm) {
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) {
      T s = T(0);
#pragma unroll
      for (int k = 0; k < K; ++k) s += A[i * K + k] * B[j * K + k];
      Cm[i * N + j] = s;
    }
}

// y[M] = A[M][N] x[N]
template <typename T, int M, int N>
SQSM_DEV void mv(const T* A, const T* x, T* y) {
#pragma unroll
  for (int i = 0; i < M; ++i) {
    T s = T(0);
#pragma unroll
    for (int k = 0; k < N; ++k) s += A[i * N + k] * x[k];
    y[i] = s;
  }
}

// y[N] = A[M][N]^T x[M]
template <typename T, int M, int N>
SQSM_DEV void mtv(const T* A, const T* x, T* y) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    T s = T(0);
#pragma unroll
    for (int k = 0; k < M; ++k) s += A[k * N + i] * x[k];
    y[i] = s;
  }
}

// Lower Cholesky factor in place (upper part cleared).  A non-positive pivot
// gives NaN, as the standard form does when a covariance loses definiteness.
template <typename T, int N>
SQSM_DEV void chol_inplace(T* A) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    T s = A[j * N + j];
#pragma unroll
    for (int k = 0; k < j; ++k) s -= A[j * N + k] * A[j * N + k];
    const T d = sq_sqrt(s);
    const T inv = T(1) / d;
    A[j * N + j] = d;
#pragma unroll
    for (int i = j + 1; i < N; ++i) {
      T t = A[i * N + j];
#pragma unroll
      for (int k = 0; k < j; ++k) t -= A[i * N + k] * A[j * N + k];
      A[i * N + j] = t * inv;
    }
#pragma unroll
    for (int i = 0; i < j; ++i) A[i * N + j] = T(0);
  }
}

// Triangular solves divide once per diagonal entry and multiply by the
// reciprocal elsewhere.

// x = L^{-1} b for lower L (N x N); in place on b.
template <typename T, int N>
SQSM_DEV void lsolve(const T* L, T* b) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    T s = b[i];
#pragma unroll
    for (int k = 0; k < i; ++k) s -= L[i * N + k] * b[k];
    b[i] = s / L[i * N + i];
  }
}

// x = L^{-T} b for lower L (N x N); in place on b.
template <typename T, int N>
SQSM_DEV void ltsolve(const T* L, T* b) {
#pragma unroll
  for (int i = N - 1; i >= 0; --i) {
    T s = b[i];
#pragma unroll
    for (int k = i + 1; k < N; ++k) s -= L[k * N + i] * b[k];
    b[i] = s / L[i * N + i];
  }
}

// X <- X L^{-1} for X (M x N), lower L (N x N): each row x solves z L = x.
template <typename T, int M, int N>
SQSM_DEV void rsolve(T* X, const T* L) {
  T inv[N];
#pragma unroll
  for (int i = 0; i < N; ++i) inv[i] = hh_rcp(L[i * N + i]);
#pragma unroll
  for (int r = 0; r < M; ++r) {
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      T s = X[r * N + i];
#pragma unroll
      for (int k = i + 1; k < N; ++k) s -= X[r * N + k] * L[k * N + i];
      X[r * N + i] = s * inv[i];
    }
  }
}

// X <- X L^{-T} for X (M x N), lower L (N x N): each row x solves z L^T = x.
template <typename T, int M, int N>
SQSM_DEV void rsolve_t(T* X, const T* L) {
  T inv[N];
#pragma unroll
  for (int i = 0; i < N; ++i) inv[i] = hh_rcp(L[i * N + i]);
#pragma unroll
  for (int r = 0; r < M; ++r) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      T s = X[r * N + i];
#pragma unroll
      for (int k = 0; k < i; ++k) s -= X[r * N + k] * L[i * N + k];
      X[r * N + i] = s * inv[i];
    }
  }
}

template <typename T, int N>
SQSM_DEV void load(const T* __restrict__ g, T* r) {
#pragma unroll
  for (int i = 0; i < N; ++i) r[i] = g[i];
}

template <typename T, int N>
SQSM_DEV void store(T* __restrict__ g, const T* r) {
#pragma unroll
  for (int i = 0; i < N; ++i) g[i] = r[i];
}

// Load an N x N lower factor, zeroing the strictly upper part.
template <typename T, int N>
SQSM_DEV void load_lower(const T* __restrict__ g, T* r) {
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) r[i * N + j] = j <= i ? g[i * N + j] : T(0);
}

// N consecutive elements through 16-byte vector accesses (g 16-byte aligned,
// N * sizeof(T) a multiple of 16).
template <typename T, int N>
SQSM_DEV void vload(const T* __restrict__ g, T* r) {
  static_assert((N * sizeof(T)) % 16 == 0, "vector access of whole 16-byte words");
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
      const float4 v = reinterpret_cast<const float4*>(g)[i];
      r[4 * i] = v.x; r[4 * i + 1] = v.y; r[4 * i + 2] = v.z; r[4 * i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const double2 v = reinterpret_cast<const double2*>(g)[i];
      r[2 * i] = v.x; r[2 * i + 1] = v.y;
    }
  }
}

template <typename T, int N>
SQSM_DEV void vstore(T* __restrict__ g, const T* r) {
  static_assert((N * sizeof(T)) % 16 == 0, "vector access of whole 16-byte words");
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i)
      reinterpret_cast<float4*>(g)[i] = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
  } else {
#pragma unroll
    for (int i = 0; i < N / 2; ++i)
      reinterpret_cast<double2*>(g)[i] = make_double2(r[2 * i], r[2 * i + 1]);
  }
}

// Store an N x N lower factor with explicit zeros above the diagonal.
template <typename T, int N>
SQSM_DEV void store_lower(T* __restrict__ g, const T* r) {
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) g[i * N + j] = j <= i ? r[i * N + j] : T(0);
}

template <typename T> SQSM_DEV bool finite(T x) { return isfinite(x); }

}  // namespace sqsm
