// Upper scan levels in FP64 with each combine spread over lanes.
//
// This GPU has few FP64 units: a warp's FP64 multiply-add holds its
// scheduler's unit for 64 cycles however many lanes take part and whatever
// its neighbours depend on (measured; four warps on an SM share it at 19
// cycles each).  With one thread per combine (some 2200 FP64 instructions
// at n_x = 5) a Kogge-Stone round therefore takes about 100 us however few
// combines it has, and a level of a thousand items keeps 32 of the GPU's 608
// schedulers busy.  Here a matrix has one row per lane (8 lanes, n_x of them
// used), so a combine issues about 430 FP64 instructions per warp:
//   filter combine    two rows-of-lanes halves (16 lanes) side by side; the
//                     two factors of Table 3 are the same computation on
//                     exchanged operands,
//                       U_ij = Tria([A_j   U_i Tria([M,   I])^{-T}, U_j]),
//                       Z_ij = Tria([A_i^T Z_j Tria([M^T, I])^{-T}, Z_i]),
//                     M = U_i^T Z_j, so one half computes U_ij and the other
//                     Z_ij in the same instructions;
//   filter apply, smoother combine and apply   one half (8 lanes) each.
// Tria is modified Gram-Schmidt on the rows (the same L as Householder's and
// as backward stable: Bjorck, Linear Algebra Appl. 1994): per row one inner
// product, one reciprocal square root and one update, where a reflection
// also needs a quotient; the rows' inner products with the pivot row are the
// lanes' own.  With one step per leaf (default_shape) the FP64 track of
// n = 4000 went from 18.7 to 6.6 ms per ten iterations (filter upper levels
// 1000 -> 220 us per iteration, smoother's 228 -> 112), the n_x = 6 linear
// smoother of n = 20011 from 3.45 to 1.60 ms.
#pragma once

#include "wscan.cuh"

namespace sqsm {

constexpr int kLaneRows = 8;        // lanes of a half: one matrix row each
// Items of a Kogge-Stone chunk: four warps, one per scheduler of an SM.
constexpr int kLaneFilterChunk = 8;
constexpr int kLaneSmootherChunk = 16;
constexpr int kLaneFold = 4;        // items folded by one group at larger levels

// Tria([X | Q]) with row r in lane r of each half: x[NX] dense, q[c] the
// lower Q (c <= r).  l[c] = L[r][c] (0 above the diagonal), rinv[c] =
// 1 / L[c][c] (0 for a zero row) in every lane; x and q are consumed.
template <typename T, int NX>
SQSM_DEV void lane_tria(T* x, T* q, T* l, T* rinv, int r) {
  constexpr unsigned kAll = 0xffffffffu;
#pragma unroll
  for (int i = 0; i < NX; ++i) {
    T xi[NX], qi[NX];
#pragma unroll
    for (int c = 0; c < NX; ++c) xi[c] = __shfl_sync(kAll, x[c], i, kLaneRows);
#pragma unroll
    for (int c = 0; c <= i; ++c) qi[c] = __shfl_sync(kAll, q[c], i, kLaneRows);
    T dot = T(0);
#pragma unroll
    for (int c = 0; c < NX; ++c) dot += x[c] * xi[c];
#pragma unroll
    for (int c = 0; c <= i; ++c) dot += q[c] * qi[c];
    const T s2 = __shfl_sync(kAll, dot, i, kLaneRows);
    const bool nz = s2 > Tiny<T>::value;
    const T ri = nz ? rsqrt(nz ? s2 : T(1)) : T(0);
    const T li = dot * ri;
    l[i] = r >= i ? li : T(0);
    rinv[i] = ri;
    const T w = r > i ? li * ri : T(0);
    if (i + 1 < NX) {
#pragma unroll
      for (int c = 0; c < NX; ++c) x[c] -= w * xi[c];
#pragma unroll
      for (int c = 0; c <= i; ++c) q[c] -= w * qi[c];
    }
  }
}

// A 16-lane group's scratch in shared memory, and what it holds of a
// combine's result: lane (h, r) row r of U_ij (h = 0) or Z_ij (h = 1), its
// half's columns of row r of A_ij, and b_ij or eta_ij [r].
template <typename T, int NX> struct LaneWs {
  T mt[NX * NX], x11[NX * NX], rx[NX], k[NX * NX];
};
template <typename T, int NX> struct LaneFilterOut {
  static constexpr int CA = (NX + 1) / 2;   // columns of A_ij in half 0
  T a[CA], v, l[NX];
  SQSM_DEV void store(T* o, int h, int r) const {
    using R = FRec<NX>;
    if (r >= NX) return;
#pragma unroll
    for (int c = 0; c < CA; ++c)
      if (h * CA + c < NX) o[R::A + r * NX + h * CA + c] = a[c];
    o[(h ? R::eta : R::b) + r] = v;
#pragma unroll
    for (int c = 0; c < NX; ++c) o[(h ? R::Z : R::U) + r * NX + c] = l[c];
  }
};

// Table 3 on records in shared memory (see filter_combine for the formulas;
// here A_ij = A_j A_i - V K^T with V = A_j U_i Xi_11^{-T} and
// K = A_i^T Z_j M^T Xi_11^{-T}, and b_ij, eta_ij from the same factors).
// Every lane of the warp takes part.
template <typename T, int NX>
SQSM_DEV void lane_filter_combine(const T* ei, const T* ej, LaneWs<T, NX>& ws,
                                  LaneFilterOut<T, NX>& out) {
  using R = FRec<NX>;
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int CA = LaneFilterOut<T, NX>::CA;
  const int lane = threadIdx.x % kWarp, r = lane % kLaneRows, h = lane / kLaneRows % 2;
  const int rr = r < NX ? r : NX - 1;
  const T* X = h ? ej + R::Z : ei + R::U;
  const T* Y = h ? ei + R::U : ej + R::Z;
  T P[NX], xc[NX], yc[NX];   // row rr of A_j or A_i^T, columns rr of X and Y
#pragma unroll
  for (int k = 0; k < NX; ++k) {
    P[k] = h ? ei[R::A + k * NX + rr] : ej[R::A + rr * NX + k];
    xc[k] = X[k * NX + rr];
    yc[k] = Y[k * NX + rr];
  }
  // row rr of M (M^T), and of A_j U_i (A_i^T Z_j)
  T m[NX], mc[NX], q[NX], V[NX];
#pragma unroll
  for (int c = 0; c < NX; ++c) {
    T s = T(0), v = T(0);
#pragma unroll
    for (int k = c; k < NX; ++k) {
      s += xc[k] * Y[k * NX + c];
      v += P[k] * X[k * NX + c];
    }
    m[c] = mc[c] = s;
    V[c] = v;
    q[c] = c == rr ? T(1) : T(0);
    if (h && r < NX) ws.mt[r * NX + c] = s;
  }
  T l[NX], rinv[NX];
  lane_tria<T, NX>(m, q, l, rinv, r);
  if (!h && r < NX) {
#pragma unroll
    for (int c = 0; c < NX; ++c) ws.x11[r * NX + c] = l[c];
    if (r == 0) {
#pragma unroll
      for (int c = 0; c < NX; ++c) ws.rx[c] = rinv[c];
    }
  }
  __syncwarp();
  // row rr of A_j A_i (half 0), of A_i^T Z_j M^T Xi_11^{-T} = K (half 1)
  T w[NX], kk[NX];
  const T* W = h ? ws.mt : ei + R::A;
#pragma unroll
  for (int c = 0; c < NX; ++c) {
    T s = T(0);
#pragma unroll
    for (int k = 0; k < NX; ++k) s += (h ? V[k] : P[k]) * W[k * NX + c];
    w[c] = s;
  }
#pragma unroll
  for (int c = 0; c < NX; ++c) {
    T s = w[c], v = V[c];
#pragma unroll
    for (int k = 0; k < c; ++k) {
      s -= kk[k] * ws.x11[c * NX + k];
      v -= V[k] * __shfl_sync(kAll, l[k], c, kLaneRows);
    }
    kk[c] = s * ws.rx[c];
    V[c] = v * rinv[c];       // row rr of A_j U_i Xi_11^{-T} (A_i^T W)
    if (h && r < NX) ws.k[r * NX + c] = kk[c];
  }
  // x = b_i + U_i U_i^T eta_j (half 0), z = eta_j - Z_j Z_j^T b_i (half 1)
  T t = T(0), sv = T(0);
#pragma unroll
  for (int k = 0; k < NX; ++k) t += xc[k] * (h ? ei[R::b + k] : ej[R::eta + k]);
#pragma unroll
  for (int k = 0; k < NX; ++k) sv += X[rr * NX + k] * __shfl_sync(kAll, t, k, kLaneRows);
  const T x = h ? ej[R::eta + rr] - sv : ei[R::b + rr] + sv;
  T xv[NX], u = T(0), u2 = T(0);
#pragma unroll
  for (int k = 0; k < NX; ++k) {
    xv[k] = __shfl_sync(kAll, x, k, kLaneRows);
    u += yc[k] * xv[k];       // Z_j^T x, U_i^T z
  }
#pragma unroll
  for (int k = 0; k < NX; ++k) u2 += mc[k] * __shfl_sync(kAll, u, k, kLaneRows);
  T y = h ? u : u2;           // then y <- Xi_11^{-1} (M Z_j^T x, U_i^T z)
  T v = h ? ei[R::eta + rr] : ej[R::b + rr];
#pragma unroll
  for (int k = 0; k < NX; ++k) {
    const T yk = __shfl_sync(kAll, y, k, kLaneRows) * ws.rx[k];
    y -= ws.x11[rr * NX + k] * yk;
    v += P[k] * xv[k];
    v -= (h ? kk[k] : V[k]) * yk;
  }
  out.v = v;
  __syncwarp();
  // this half's columns of row rr of A_ij
  T v0[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) {
    const T o = __shfl_xor_sync(kAll, V[k], kLaneRows);
    v0[k] = h ? o : V[k];
  }
#pragma unroll
  for (int c = 0; c < CA; ++c) {
    const T o = c + CA < NX ? __shfl_xor_sync(kAll, w[c + CA < NX ? c + CA : 0], kLaneRows) : T(0);
    const int col = h && c + CA < NX ? c + CA : c;
    T s = h ? o : w[c];
#pragma unroll
    for (int k = 0; k < NX; ++k) s -= v0[k] * ws.k[col * NX + k];
    out.a[c] = s;
  }
  const T* Bk = h ? ei + R::Z : ej + R::U;
#pragma unroll
  for (int c = 0; c < NX; ++c) q[c] = Bk[rr * NX + c];
  lane_tria<T, NX>(V, q, out.l, rinv, r);
  __syncwarp();
}

// Carry of one half in shared memory: vector and lower factor (full square,
// zeros above the diagonal).
template <typename T, int NX> struct LaneCarry {
  T v[NX], L[NX * NX];
};

// Table 3 with A_i = 0 (filter_apply): lane r returns row r of U_ij and
// b_ij[r] for the carry (b_i, U_i) and the record ej.
template <typename T, int NX>
SQSM_DEV void lane_filter_apply(const LaneCarry<T, NX>& ci, const T* ej, T& bo, T* l) {
  using R = FRec<NX>;
  constexpr unsigned kAll = 0xffffffffu;
  const int r = threadIdx.x % kLaneRows, rr = r < NX ? r : NX - 1;
  T P[NX], xc[NX], yc[NX], m[NX], mc[NX], q[NX], V[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) {
    P[k] = ej[R::A + rr * NX + k];
    xc[k] = ci.L[k * NX + rr];
    yc[k] = ej[R::Z + k * NX + rr];
  }
#pragma unroll
  for (int c = 0; c < NX; ++c) {
    T s = T(0), v = T(0);
#pragma unroll
    for (int k = c; k < NX; ++k) {
      s += xc[k] * ej[R::Z + k * NX + c];
      v += P[k] * ci.L[k * NX + c];
    }
    m[c] = mc[c] = s;
    V[c] = v;
    q[c] = c == rr ? T(1) : T(0);
  }
  T x11[NX], rinv[NX];
  lane_tria<T, NX>(m, q, x11, rinv, r);
#pragma unroll
  for (int c = 0; c < NX; ++c) {
    T v = V[c];
#pragma unroll
    for (int k = 0; k < c; ++k) v -= V[k] * __shfl_sync(kAll, x11[k], c, kLaneRows);
    V[c] = v * rinv[c];
  }
  T t = T(0), sv = T(0), u = T(0), y = T(0);
#pragma unroll
  for (int k = 0; k < NX; ++k) t += xc[k] * ej[R::eta + k];
#pragma unroll
  for (int k = 0; k < NX; ++k) sv += ci.L[rr * NX + k] * __shfl_sync(kAll, t, k, kLaneRows);
  const T x = ci.v[rr] + sv;
  T xv[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) {
    xv[k] = __shfl_sync(kAll, x, k, kLaneRows);
    u += yc[k] * xv[k];
  }
#pragma unroll
  for (int k = 0; k < NX; ++k) y += mc[k] * __shfl_sync(kAll, u, k, kLaneRows);
  bo = ej[R::b + rr];
#pragma unroll
  for (int k = 0; k < NX; ++k) {
    const T yk = __shfl_sync(kAll, y, k, kLaneRows) * rinv[k];
    y -= x11[k] * yk;
    bo += P[k] * xv[k];
    bo -= V[k] * yk;
  }
#pragma unroll
  for (int c = 0; c < NX; ++c) q[c] = ej[R::U + rr * NX + c];
  lane_tria<T, NX>(V, q, l, rinv, r);
}

// Table 5 (smoother_combine; E_ij left out with APPLY, the right operand
// then a carry): lane r returns row r of E_ij and D_ij and g_ij[r].
template <typename T, int NX, bool APPLY>
SQSM_DEV void lane_smoother_combine(const T* ei, const T* Ej, const T* gj, const T* Dj, T* eo,
                                    T& go, T* l) {
  using R = SRec<NX>;
  const int r = threadIdx.x % kLaneRows, rr = r < NX ? r : NX - 1;
  T e[NX], x[NX], q[NX], rinv[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) e[k] = ei[R::E + rr * NX + k];
  T g = T(0);
#pragma unroll
  for (int k = 0; k < NX; ++k) g += e[k] * gj[k];
  go = g + ei[R::g + rr];
#pragma unroll
  for (int c = 0; c < NX; ++c) {
    T s = T(0), d = T(0);
#pragma unroll
    for (int k = 0; k < NX; ++k) {
      if (!APPLY) s += e[k] * Ej[k * NX + c];
      if (k >= c) d += e[k] * Dj[k * NX + c];
    }
    if (!APPLY) eo[c] = s;
    x[c] = d;
    q[c] = ei[R::D + rr * NX + c];
  }
  lane_tria<T, NX>(x, q, l, rinv, r);
}

// n values from global memory into shared memory by `lanes` lanes.
template <typename T>
SQSM_DEV void lane_copy(T* dst, const T* __restrict__ src, int n, int lane, int lanes) {
  for (int i = lane; i < n; i += lanes) dst[i] = src[i];
}

// A packed carry record (RowsPacked) to and from a LaneCarry.
template <typename T, int NX>
SQSM_DEV void lane_load_carry(LaneCarry<T, NX>& c, const T* __restrict__ g, int r) {
  if (r < NX) {
    c.v[r] = g[r];
#pragma unroll
    for (int k = 0; k < NX; ++k) c.L[r * NX + k] = k <= r ? g[NX + r * (r + 1) / 2 + k] : T(0);
  }
}
template <typename T, int NX>
SQSM_DEV void lane_store_carry(T* __restrict__ g, T v, const T* l, int r) {
  if (r < NX) {
    g[r] = v;
#pragma unroll
    for (int k = 0; k < NX; ++k)
      if (k <= r) g[NX + r * (r + 1) / 2 + k] = l[k];
  }
}

// ---------------------------------------------------------------------------
// Filter
// ---------------------------------------------------------------------------

// Kogge-Stone rounds over the c <= kLaneFilterChunk records of S, one 16-lane
// group per item (blockDim 16 kLaneFilterChunk).
template <typename T, int NX>
SQSM_DEV void lane_filter_ks(T* S, LaneWs<T, NX>* ws, int c) {
  constexpr int REC = FRec<NX>::size;
  const int t = threadIdx.x / (2 * kLaneRows);
  const int h = threadIdx.x / kLaneRows % 2, r = threadIdx.x % kLaneRows;
  for (int d = 1; d < c; d <<= 1) {
    // a warp holds items t and t + 1 (t even): it idles when neither combines
    const int t1 = t | 1;
    const bool warp_on = t1 >= d && (t & ~1) < c;
    const bool act = t < c && t >= d;
    LaneFilterOut<T, NX> o;
    if (warp_on)
      lane_filter_combine<T, NX>(S + (act ? t - d : 0) * REC, S + (act ? t : 0) * REC, ws[t], o);
    __syncthreads();
    if (act) o.store(S + t * REC, h, r);
    __syncthreads();
  }
}

// Chunk-scan up level (see filter_up_cs): one block per chunk.
template <typename T, int NX>
__global__ void __launch_bounds__(2 * kLaneRows * kLaneFilterChunk)
filter_up_lane_ks(DevLevel lv, T* __restrict__ items, T* __restrict__ out) {
  constexpr int REC = FRec<NX>::size;
  __shared__ T S[kLaneFilterChunk * REC];
  __shared__ LaneWs<T, NX> ws[kLaneFilterChunk];
  const int64_t c = blockIdx.x;
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  lane_copy(S, items + i0 * REC, cnt * REC, threadIdx.x, blockDim.x);
  __syncthreads();
  lane_filter_ks<T, NX>(S, ws, cnt);
  lane_copy(items + i0 * REC, S, cnt * REC, threadIdx.x, blockDim.x);
  lane_copy(out + c * REC, S + (cnt - 1) * REC, REC, threadIdx.x, blockDim.x);
}

// Top of the tree (see filter_top_ks): one block per sequence.
template <typename T, int NX>
__global__ void __launch_bounds__(2 * kLaneRows * kLaneFilterChunk)
filter_top_lane_ks(const int64_t* __restrict__ seq_item_off, const T* __restrict__ items,
                   T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int REC = FRec<NX>::size;
  __shared__ T S[kLaneFilterChunk * REC];
  __shared__ LaneWs<T, NX> ws[kLaneFilterChunk];
  const int b = blockIdx.x;
  const int64_t i0 = seq_item_off[b];
  const int c = (int)(seq_item_off[b + 1] - i0);
  lane_copy(S, items + i0 * REC, c * REC, threadIdx.x, blockDim.x);
  __syncthreads();
  lane_filter_ks<T, NX>(S, ws, c);
  const int t = threadIdx.x;
  if (t < c) {
    if (t > 0) {
      const T* p = S + (t - 1) * REC;
      RowsPacked<T, NX>{carry_out}.store(i0 + t, p + FRec<NX>::b, p + FRec<NX>::U);
    }
    flag_out[i0 + t] = t > 0 ? 1 : 0;
  }
}

// Fold of a level's chunks (see filter_up), one 16-lane group per chunk, one
// warp (two chunks) per block.
template <typename T, int NX>
__global__ void __launch_bounds__(kWarp)
filter_up_lane(DevLevel lv, const T* __restrict__ items, T* __restrict__ out) {
  constexpr int REC = FRec<NX>::size, G = 2 * kLaneRows;
  __shared__ T S[2][2 * REC];
  __shared__ LaneWs<T, NX> ws[2];
  const int g = threadIdx.x / G, gl = threadIdx.x % G, h = gl / kLaneRows, r = gl % kLaneRows;
  const int64_t c = blockIdx.x * (int64_t)2 + g;
  const bool in = c < lv.n_chunks;
  const int64_t i0 = in ? lv.first[c] : 0;
  const int cnt = in ? lv.count[c] : 0;
  const int most = max(cnt, __shfl_xor_sync(0xffffffffu, cnt, G));
  T *agg = S[g], *el = S[g] + REC;
  lane_copy(agg, items + i0 * REC, cnt > 0 ? REC : 0, gl, G);
  for (int j = 1; j < most; ++j) {
    lane_copy(el, items + (i0 + j) * REC, j < cnt ? REC : 0, gl, G);
    __syncwarp();
    LaneFilterOut<T, NX> o;
    lane_filter_combine<T, NX>(agg, el, ws[g], o);
    if (j < cnt) o.store(agg, h, r);
    __syncwarp();
  }
  __syncwarp();
  lane_copy(out + c * REC, agg, in ? REC : 0, gl, G);
}

// Down-sweep of a chunk-scan level (see filter_down_cs): 8 lanes per item,
// one block per chunk.
template <typename T, int NX>
__global__ void __launch_bounds__(kLaneRows * kLaneFilterChunk)
filter_down_lane_ks(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                    const int* __restrict__ flag_in, T* __restrict__ carry_out,
                    int* __restrict__ flag_out) {
  constexpr int REC = FRec<NX>::size, XS = XRow<NX>::size;
  using R = FRec<NX>;
  __shared__ T S[kLaneFilterChunk * REC];
  __shared__ LaneCarry<T, NX> ci;
  const int64_t c = blockIdx.x;
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  const int flag = flag_in[c];
  const int j = threadIdx.x / kLaneRows, r = threadIdx.x % kLaneRows;
  lane_copy(S, items + i0 * REC, (cnt - 1) * REC, threadIdx.x, blockDim.x);
  if (j == 0) lane_load_carry<T, NX>(ci, carry_in + c * XS, r);
  __syncthreads();
  const int rr = r < NX ? r : NX - 1;
  T v = ci.v[rr], l[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) l[k] = ci.L[rr * NX + k];
  // a warp holds four items: it skips the apply when none of them has one
  const bool warp_on = flag && (j & ~3) < cnt && cnt > 1;
  if (warp_on) {
    const int p = j > 0 && j < cnt ? j - 1 : 0;
    T nv, nl[NX];
    lane_filter_apply<T, NX>(ci, S + p * REC, nv, nl);
    if (j > 0) {
      v = nv;
#pragma unroll
      for (int k = 0; k < NX; ++k) l[k] = nl[k];
    }
  } else if (!flag && j > 0 && j < cnt) {
    v = S[(j - 1) * REC + R::b + rr];
#pragma unroll
    for (int k = 0; k < NX; ++k) l[k] = S[(j - 1) * REC + R::U + rr * NX + k];
  }
  if (j < cnt) {
    lane_store_carry<T, NX>(carry_out + (i0 + j) * XS, v, l, r);
    if (r == 0) flag_out[i0 + j] = j == 0 ? flag : 1;
  }
}

// Down-sweep of a folded level (see filter_down): 8 lanes per chunk, one warp
// (four chunks) per block.
template <typename T, int NX>
__global__ void __launch_bounds__(kWarp)
filter_down_lane(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                 const int* __restrict__ flag_in, T* __restrict__ carry_out,
                 int* __restrict__ flag_out) {
  constexpr int REC = FRec<NX>::size, XS = XRow<NX>::size, NG = kWarp / kLaneRows;
  using R = FRec<NX>;
  __shared__ T S[NG][REC];
  __shared__ LaneCarry<T, NX> cs[NG];
  const int g = threadIdx.x / kLaneRows, r = threadIdx.x % kLaneRows, rr = r < NX ? r : NX - 1;
  const int64_t c = blockIdx.x * (int64_t)NG + g;
  const bool in = c < lv.n_chunks;
  const int64_t i0 = in ? lv.first[c] : 0;
  const int cnt = in ? lv.count[c] : 0;
  int flag = in ? flag_in[c] : 0;
  const int most = __reduce_max_sync(0xffffffffu, cnt);
  LaneCarry<T, NX>& ci = cs[g];
  if (in) lane_load_carry<T, NX>(ci, carry_in + c * XS, r);
  __syncwarp();
  T v = in ? ci.v[rr] : T(0), l[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) l[k] = in ? ci.L[rr * NX + k] : T(0);
  for (int j = 0; j < most; ++j) {
    if (j < cnt) {
      lane_store_carry<T, NX>(carry_out + (i0 + j) * XS, v, l, r);
      if (r == 0) flag_out[i0 + j] = flag;
    }
    if (j + 1 >= most) break;
    const bool more = j + 1 < cnt;
    lane_copy(S[g], items + (i0 + j) * REC, more ? REC : 0, r, kLaneRows);
    __syncwarp();
    T nv, nl[NX];
    lane_filter_apply<T, NX>(ci, S[g], nv, nl);
    __syncwarp();
    if (more) {
      if (!flag) {
        nv = S[g][R::b + rr];
#pragma unroll
        for (int k = 0; k < NX; ++k) nl[k] = S[g][R::U + rr * NX + k];
        flag = 1;
      }
      v = nv;
#pragma unroll
      for (int k = 0; k < NX; ++k) l[k] = nl[k];
      if (r < NX) {
        ci.v[r] = v;
#pragma unroll
        for (int k = 0; k < NX; ++k) ci.L[r * NX + k] = l[k];
      }
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Smoother (reverse scan), 8 lanes per combine
// ---------------------------------------------------------------------------

template <typename T, int NX>
SQSM_DEV void lane_smoother_store(T* o, const T* e, T g, const T* l, int r) {
  using R = SRec<NX>;
  if (r >= NX) return;
#pragma unroll
  for (int c = 0; c < NX; ++c) {
    o[R::E + r * NX + c] = e[c];
    o[R::D + r * NX + c] = l[c];
  }
  o[R::g + r] = g;
}

// Kogge-Stone rounds over the c <= kLaneSmootherChunk records of S (inclusive
// suffixes), 8 lanes per item.
template <typename T, int NX>
SQSM_DEV void lane_smoother_ks(T* S, int c) {
  constexpr int REC = SRec<NX>::size;
  using R = SRec<NX>;
  const int t = threadIdx.x / kLaneRows, r = threadIdx.x % kLaneRows;
  for (int d = 1; d < c; d <<= 1) {
    const bool act = t + d < c;
    const bool warp_on = (t & ~3) + d < c;
    T e[NX], g, l[NX];
    if (warp_on) {
      const T* ej = S + (act ? t + d : 0) * REC;
      lane_smoother_combine<T, NX, false>(S + (act ? t : 0) * REC, ej + R::E, ej + R::g, ej + R::D,
                                          e, g, l);
    }
    __syncthreads();
    if (act) lane_smoother_store<T, NX>(S + t * REC, e, g, l, r);
    __syncthreads();
  }
}

template <typename T, int NX>
__global__ void __launch_bounds__(kLaneRows * kLaneSmootherChunk)
smoother_up_lane_ks(DevLevel lv, T* __restrict__ items, T* __restrict__ out) {
  constexpr int REC = SRec<NX>::size;
  __shared__ T S[kLaneSmootherChunk * REC];
  const int64_t c = blockIdx.x;
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  lane_copy(S, items + i0 * REC, cnt * REC, threadIdx.x, blockDim.x);
  __syncthreads();
  lane_smoother_ks<T, NX>(S, cnt);
  lane_copy(items + i0 * REC, S, cnt * REC, threadIdx.x, blockDim.x);
  lane_copy(out + c * REC, S, REC, threadIdx.x, blockDim.x);
}

template <typename T, int NX>
__global__ void __launch_bounds__(kLaneRows * kLaneSmootherChunk)
smoother_top_lane_ks(const int64_t* __restrict__ seq_item_off, const T* __restrict__ items,
                     T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int REC = SRec<NX>::size;
  __shared__ T S[kLaneSmootherChunk * REC];
  const int b = blockIdx.x;
  const int64_t i0 = seq_item_off[b];
  const int c = (int)(seq_item_off[b + 1] - i0);
  lane_copy(S, items + i0 * REC, c * REC, threadIdx.x, blockDim.x);
  __syncthreads();
  lane_smoother_ks<T, NX>(S, c);
  const int t = threadIdx.x;
  if (t < c) {
    if (t + 1 < c) {
      const T* p = S + (t + 1) * REC;
      RowsPacked<T, NX>{carry_out}.store(i0 + t, p + SRec<NX>::g, p + SRec<NX>::D);
    }
    flag_out[i0 + t] = t + 1 < c ? 1 : 0;
  }
}

// Fold of a level's chunks right to left (see smoother_up), 8 lanes per chunk,
// one warp (four chunks) per block.
template <typename T, int NX>
__global__ void __launch_bounds__(kWarp)
smoother_up_lane(DevLevel lv, const T* __restrict__ items, T* __restrict__ out) {
  constexpr int REC = SRec<NX>::size, NG = kWarp / kLaneRows;
  using R = SRec<NX>;
  __shared__ T S[NG][2 * REC];
  const int g = threadIdx.x / kLaneRows, r = threadIdx.x % kLaneRows;
  const int64_t c = blockIdx.x * (int64_t)NG + g;
  const bool in = c < lv.n_chunks;
  const int64_t i0 = in ? lv.first[c] : 0;
  const int cnt = in ? lv.count[c] : 0;
  const int most = __reduce_max_sync(0xffffffffu, cnt);
  T *agg = S[g], *el = S[g] + REC;
  lane_copy(agg, items + (i0 + cnt - 1) * REC, cnt > 0 ? REC : 0, r, kLaneRows);
  for (int j = 1; j < most; ++j) {
    lane_copy(el, items + (i0 + cnt - 1 - j) * REC, j < cnt ? REC : 0, r, kLaneRows);
    __syncwarp();
    T e[NX], gg, l[NX];
    lane_smoother_combine<T, NX, false>(el, agg + R::E, agg + R::g, agg + R::D, e, gg, l);
    __syncwarp();
    if (j < cnt) lane_smoother_store<T, NX>(agg, e, gg, l, r);
    __syncwarp();
  }
  __syncwarp();
  lane_copy(out + c * REC, agg, in ? REC : 0, r, kLaneRows);
}

// Down-sweep of a chunk-scan level (see smoother_down_cs): 8 lanes per item,
// one block per chunk.
template <typename T, int NX>
__global__ void __launch_bounds__(kLaneRows * kLaneSmootherChunk)
smoother_down_lane_ks(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                      const int* __restrict__ flag_in, T* __restrict__ carry_out,
                      int* __restrict__ flag_out) {
  constexpr int REC = SRec<NX>::size, XS = XRow<NX>::size;
  using R = SRec<NX>;
  __shared__ T S[kLaneSmootherChunk * REC];
  __shared__ LaneCarry<T, NX> ci;
  const int64_t c = blockIdx.x;
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  const int flag = flag_in[c];
  const int j = threadIdx.x / kLaneRows, r = threadIdx.x % kLaneRows, rr = r < NX ? r : NX - 1;
  lane_copy(S, items + i0 * REC, cnt * REC, threadIdx.x, blockDim.x);
  if (j == 0) lane_load_carry<T, NX>(ci, carry_in + c * XS, r);
  __syncthreads();
  T v = ci.v[rr], l[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) l[k] = ci.L[rr * NX + k];
  const bool warp_on = flag && (j & ~3) + 1 < cnt;
  const bool mid = j + 1 < cnt;
  if (warp_on) {
    T e[1], nv, nl[NX];
    lane_smoother_combine<T, NX, true>(S + (mid ? j + 1 : 0) * REC, nullptr, ci.v, ci.L, e, nv, nl);
    if (mid) {
      v = nv;
#pragma unroll
      for (int k = 0; k < NX; ++k) l[k] = nl[k];
    }
  } else if (!flag && mid) {
    v = S[(j + 1) * REC + R::g + rr];
#pragma unroll
    for (int k = 0; k < NX; ++k) l[k] = S[(j + 1) * REC + R::D + rr * NX + k];
  }
  if (j < cnt) {
    lane_store_carry<T, NX>(carry_out + (i0 + j) * XS, v, l, r);
    if (r == 0) flag_out[i0 + j] = j == cnt - 1 ? flag : 1;
  }
}

// Down-sweep of a folded level (see smoother_down): 8 lanes per chunk, one
// warp (four chunks) per block.
template <typename T, int NX>
__global__ void __launch_bounds__(kWarp)
smoother_down_lane(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                   const int* __restrict__ flag_in, T* __restrict__ carry_out,
                   int* __restrict__ flag_out) {
  constexpr int REC = SRec<NX>::size, XS = XRow<NX>::size, NG = kWarp / kLaneRows;
  using R = SRec<NX>;
  __shared__ T S[NG][REC];
  __shared__ LaneCarry<T, NX> cs[NG];
  const int g = threadIdx.x / kLaneRows, r = threadIdx.x % kLaneRows, rr = r < NX ? r : NX - 1;
  const int64_t c = blockIdx.x * (int64_t)NG + g;
  const bool in = c < lv.n_chunks;
  const int64_t i0 = in ? lv.first[c] : 0;
  const int cnt = in ? lv.count[c] : 0;
  int flag = in ? flag_in[c] : 0;
  const int most = __reduce_max_sync(0xffffffffu, cnt);
  LaneCarry<T, NX>& ci = cs[g];
  if (in) lane_load_carry<T, NX>(ci, carry_in + c * XS, r);
  __syncwarp();
  T v = in ? ci.v[rr] : T(0), l[NX];
#pragma unroll
  for (int k = 0; k < NX; ++k) l[k] = in ? ci.L[rr * NX + k] : T(0);
  for (int j = 0; j < most; ++j) {   // item cnt - 1 - j
    const int64_t i = i0 + cnt - 1 - j;
    if (j < cnt) {
      lane_store_carry<T, NX>(carry_out + i * XS, v, l, r);
      if (r == 0) flag_out[i] = flag;
    }
    if (j + 1 >= most) break;
    const bool more = j + 1 < cnt;
    lane_copy(S[g], items + i * REC, more ? REC : 0, r, kLaneRows);
    __syncwarp();
    T e[1], nv, nl[NX];
    lane_smoother_combine<T, NX, true>(S[g], nullptr, ci.v, ci.L, e, nv, nl);
    __syncwarp();
    if (more) {
      if (!flag) {
        nv = S[g][R::g + rr];
#pragma unroll
        for (int k = 0; k < NX; ++k) nl[k] = S[g][R::D + rr * NX + k];
        flag = 1;
      }
      v = nv;
#pragma unroll
      for (int k = 0; k < NX; ++k) l[k] = nl[k];
      if (r < NX) {
        ci.v[r] = v;
#pragma unroll
        for (int k = 0; k < NX; ++k) ci.L[r * NX + k] = l[k];
      }
    }
    __syncwarp();
  }
}

}  // namespace sqsm
