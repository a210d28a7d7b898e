// Upper scan levels with one warp per chunk (see warp_ops.cuh); used for the
// levels that hold few chunks, where one thread per chunk leaves most of the
// GPU idle and each combine's latency sets the time.
#pragma once

#include "scan.cuh"
#include "warp_ops.cuh"

namespace sqsm {

constexpr int kWarpsPerBlock = 4;
constexpr int64_t kWarpLevelMaxChunks = 2048;

template <typename T, int NX> struct WFilterBuf {
  T a[FRec<NX>::size], b[FRec<NX>::size], c[FRec<NX>::size];
  T cb[NX], cU[NX * NX], nb[NX], nU[NX * NX];
  WFilterWs<T, NX> ws;
};

// Lane-parallel forms of RowsPacked::load / store for the warp kernels: a
// scan carry (vector v, lower factor L) in the XRow layout at g.
template <typename T, int NX>
SQSM_DEV void wload_carry(const T* __restrict__ g, T* v, T* L, int lane) {
  for (int i = lane; i < NX * NX; i += kWarp) {
    const int r = i / NX, q = i % NX;
    L[i] = q <= r ? g[NX + r * (r + 1) / 2 + q] : T(0);
  }
  for (int i = lane; i < NX; i += kWarp) v[i] = g[i];
}

template <typename T, int NX>
SQSM_DEV void wstore_carry(T* __restrict__ g, const T* v, const T* L, int lane) {
  for (int i = lane; i < NX * NX; i += kWarp) {
    const int r = i / NX, q = i % NX;
    if (q <= r) g[NX + r * (r + 1) / 2 + q] = L[i];
  }
  for (int i = lane; i < NX; i += kWarp) g[i] = v[i];
}

template <typename T, int NX>
__global__ void __launch_bounds__(kWarp * kWarpsPerBlock)
filter_up_w(DevLevel lv, const T* __restrict__ in, T* __restrict__ out) {
  constexpr int REC = FRec<NX>::size;
  __shared__ WFilterBuf<T, NX> sh[kWarpsPerBlock];
  const int wid = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
  const int64_t c = blockIdx.x * (int64_t)kWarpsPerBlock + wid;
  if (c >= lv.n_chunks) return;   // uniform per warp
  WFilterBuf<T, NX>& B = sh[wid];
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  T* agg = B.a;
  T* el = B.b;
  T* tmp = B.c;
  for (int i = lane; i < REC; i += kWarp) agg[i] = in[i0 * REC + i];
  __syncwarp();
  for (int j = 1; j < cnt; ++j) {
    for (int i = lane; i < REC; i += kWarp) el[i] = in[(i0 + j) * REC + i];
    __syncwarp();
    wfilter_combine<T, NX>(agg, el, tmp, B.ws, lane);
    T* t = agg;
    agg = tmp;
    tmp = t;
  }
  for (int i = lane; i < REC; i += kWarp) out[c * REC + i] = agg[i];
}

template <typename T, int NX>
__global__ void __launch_bounds__(kWarp * kWarpsPerBlock)
filter_down_w(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
              const int* __restrict__ flag_in, T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int REC = FRec<NX>::size, XS = XRow<NX>::size;
  __shared__ WFilterBuf<T, NX> sh[kWarpsPerBlock];
  const int wid = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
  const int64_t c = blockIdx.x * (int64_t)kWarpsPerBlock + wid;
  if (c >= lv.n_chunks) return;
  WFilterBuf<T, NX>& B = sh[wid];
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  int flag = flag_in[c];
  wload_carry<T, NX>(carry_in + c * XS, B.cb, B.cU, lane);
  __syncwarp();
  for (int j = 0; j < cnt; ++j) {
    const int64_t it = i0 + j;
    wstore_carry<T, NX>(carry_out + it * XS, B.cb, B.cU, lane);
    if (lane == 0) flag_out[it] = flag;
    __syncwarp();
    if (j + 1 < cnt) {
      if (flag) {
        for (int i = lane; i < REC; i += kWarp) B.a[i] = items[it * REC + i];
        __syncwarp();
        wfilter_apply<T, NX>(B.cb, B.cU, B.a, B.nb, B.nU, B.ws, lane);
        for (int i = lane; i < NX * NX; i += kWarp) B.cU[i] = B.nU[i];
        if (lane < NX) B.cb[lane] = B.nb[lane];
      } else {
        for (int i = lane; i < NX; i += kWarp) B.cb[i] = items[it * REC + FRec<NX>::b + i];
        for (int i = lane; i < NX * NX; i += kWarp) B.cU[i] = items[it * REC + FRec<NX>::U + i];
        flag = 1;
      }
      __syncwarp();
    }
  }
}

template <typename T, int NX> struct WSmootherBuf {
  T a[SRec<NX>::size], b[SRec<NX>::size], c[SRec<NX>::size];
  T cg[NX], cD[NX * NX];
  WSmootherWs<T, NX> ws;
};

template <typename T, int NX>
__global__ void __launch_bounds__(kWarp * kWarpsPerBlock)
smoother_up_w(DevLevel lv, const T* __restrict__ in, T* __restrict__ out) {
  constexpr int REC = SRec<NX>::size;
  __shared__ WSmootherBuf<T, NX> sh[kWarpsPerBlock];
  const int wid = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
  const int64_t c = blockIdx.x * (int64_t)kWarpsPerBlock + wid;
  if (c >= lv.n_chunks) return;
  WSmootherBuf<T, NX>& B = sh[wid];
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  T* agg = B.a;
  T* el = B.b;
  T* tmp = B.c;
  for (int i = lane; i < REC; i += kWarp) agg[i] = in[(i0 + cnt - 1) * REC + i];
  __syncwarp();
  for (int j = cnt - 2; j >= 0; --j) {
    for (int i = lane; i < REC; i += kWarp) el[i] = in[(i0 + j) * REC + i];
    __syncwarp();
    wsmoother_combine<T, NX>(el, agg, tmp, B.ws, lane);
    T* t = agg;
    agg = tmp;
    tmp = t;
  }
  for (int i = lane; i < REC; i += kWarp) out[c * REC + i] = agg[i];
}

template <typename T, int NX>
__global__ void __launch_bounds__(kWarp * kWarpsPerBlock)
smoother_down_w(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                const int* __restrict__ flag_in, T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int REC = SRec<NX>::size, XS = XRow<NX>::size;
  __shared__ WSmootherBuf<T, NX> sh[kWarpsPerBlock];
  const int wid = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
  const int64_t c = blockIdx.x * (int64_t)kWarpsPerBlock + wid;
  if (c >= lv.n_chunks) return;
  WSmootherBuf<T, NX>& B = sh[wid];
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  int flag = flag_in[c];
  wload_carry<T, NX>(carry_in + c * XS, B.cg, B.cD, lane);
  __syncwarp();
  for (int j = cnt - 1; j >= 0; --j) {
    const int64_t it = i0 + j;
    wstore_carry<T, NX>(carry_out + it * XS, B.cg, B.cD, lane);
    if (lane == 0) flag_out[it] = flag;
    __syncwarp();
    if (j > 0) {
      if (flag) {
        for (int i = lane; i < REC; i += kWarp) B.a[i] = items[it * REC + i];
        __syncwarp();
        wsmoother_apply<T, NX>(B.a, B.cg, B.cD, B.ws, lane);
      } else {
        for (int i = lane; i < NX; i += kWarp) B.cg[i] = items[it * REC + SRec<NX>::g + i];
        for (int i = lane; i < NX * NX; i += kWarp) B.cD[i] = items[it * REC + SRec<NX>::D + i];
        flag = 1;
      }
      __syncwarp();
    }
  }
}

inline unsigned wgrid_for(int64_t chunks) {
  return (unsigned)((chunks + kWarpsPerBlock - 1) / kWarpsPerBlock);
}

}  // namespace sqsm

namespace sqsm {

// Top of the tree in one launch: when every sequence has at most KS items at
// a level, one block per sequence runs a Kogge-Stone inclusive scan of them in
// shared memory (ceil(log2 KS) dependent combines) and writes each item's
// exclusive prefix (filter) / suffix (smoother) as its carry, replacing all
// higher up- and down-levels.
// Block width: 128 (FP32) / 64 (FP64) items, fewer if the records would not
// fit in 48 KB of static shared memory.
template <typename T, int REC> struct KsMax {
  static constexpr int cap = sizeof(T) == 4 ? 128 : 64;
  static constexpr int fit = (int)((48 * 1024) / (REC * sizeof(T)) / 32 * 32);
  static constexpr int value = cap < fit ? cap : fit;
};

template <typename T, int NX>
__global__ void __launch_bounds__((KsMax<T, FRec<NX>::size>::value))
filter_top_ks(const int64_t* __restrict__ seq_item_off, const T* __restrict__ items,
              T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int REC = FRec<NX>::size, KS = KsMax<T, REC>::value;
  __shared__ __align__(16) T S[KS * REC];
  const int b = blockIdx.x, t = threadIdx.x;
  const int64_t i0 = seq_item_off[b];
  const int c = (int)(seq_item_off[b + 1] - i0);
  T mine[REC], tmp[REC];
  if (t < c) vload<T, REC>(items + (i0 + t) * REC, mine);
  for (int d = 1; d < c; d <<= 1) {
    if (t < c) vstore<T, REC>(S + t * REC, mine);
    __syncthreads();
    if (t < c && t >= d) {
      filter_combine<T, NX>(S + (t - d) * REC, mine, tmp);
      copy<T, REC>(tmp, mine);
    }
    __syncthreads();
  }
  if (t < c) vstore<T, REC>(S + t * REC, mine);
  __syncthreads();
  if (t < c) {
    if (t > 0) {
      const T* p = S + (t - 1) * REC;
      RowsPacked<T, NX>{carry_out}.store(i0 + t, p + FRec<NX>::b, p + FRec<NX>::U);
    }
    flag_out[i0 + t] = t > 0 ? 1 : 0;
  }
}

template <typename T, int NX>
__global__ void __launch_bounds__((KsMax<T, SRec<NX>::size>::value))
smoother_top_ks(const int64_t* __restrict__ seq_item_off, const T* __restrict__ items,
                T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int REC = SRec<NX>::size, KS = KsMax<T, REC>::value;
  __shared__ __align__(16) T S[KS * REC];
  const int b = blockIdx.x, t = threadIdx.x;
  const int64_t i0 = seq_item_off[b];
  const int c = (int)(seq_item_off[b + 1] - i0);
  T mine[REC], tmp[REC];
  if (t < c) vload<T, REC>(items + (i0 + t) * REC, mine);
  for (int d = 1; d < c; d <<= 1) {
    if (t < c) vstore<T, REC>(S + t * REC, mine);
    __syncthreads();
    if (t + d < c) {
      smoother_combine<T, NX>(mine, S + (t + d) * REC, tmp);
      copy<T, REC>(tmp, mine);
    }
    __syncthreads();
  }
  if (t < c) vstore<T, REC>(S + t * REC, mine);
  __syncthreads();
  if (t < c) {
    if (t + 1 < c) {
      const T* p = S + (t + 1) * REC;
      RowsPacked<T, NX>{carry_out}.store(i0 + t, p + SRec<NX>::g, p + SRec<NX>::D);
    }
    flag_out[i0 + t] = t + 1 < c ? 1 : 0;
  }
}

}  // namespace sqsm

namespace sqsm {

// Upper levels in "chunk scan" form (radix kChunkScan = one warp): the up
// kernel scans each chunk with Kogge-Stone inside one warp, overwriting the
// items with their in-chunk inclusive prefixes (filter) / suffixes (smoother)
// and writing the chunk total; the down kernel gives every item its carry in
// one step, the chunk's carry applied to the neighbour's in-chunk prefix.
constexpr int kChunkScan = 32;

template <typename T, int NX>
__global__ void __launch_bounds__(kChunkScan)
filter_up_cs(DevLevel lv, T* __restrict__ items, T* __restrict__ out) {
  constexpr int REC = FRec<NX>::size;
  __shared__ __align__(16) T S[kChunkScan * REC];
  const int64_t c = blockIdx.x;
  const int t = threadIdx.x;
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  T mine[REC], tmp[REC];
  if (t < cnt) vload<T, REC>(items + (i0 + t) * REC, mine);
  for (int d = 1; d < cnt; d <<= 1) {
    if (t < cnt) vstore<T, REC>(S + t * REC, mine);
    __syncwarp();
    if (t < cnt && t >= d) {
      filter_combine<T, NX>(S + (t - d) * REC, mine, tmp);
      copy<T, REC>(tmp, mine);
    }
    __syncwarp();
  }
  if (t < cnt) vstore<T, REC>(items + (i0 + t) * REC, mine);
  if (t == cnt - 1) vstore<T, REC>(out + c * REC, mine);
}

// The carries of one chunk (cnt consecutive items, lane j holding item j's
// vector b[NX] and lower factor U[NX*NX]) written to their contiguous block
// of XRow records at g: packed into the warp's shared rows, then copied in
// 16-byte words, lane-strided, so that every store instruction covers
// consecutive words.
template <typename T, int NX>
SQSM_DEV void warp_store_carries(T* __restrict__ g, T* sh, const T* b, const T* U, int j, int cnt,
                                 bool active) {
  constexpr int XS = XRow<NX>::size, WPR = XS * (int)sizeof(T) / 16;
  static_assert(XS * sizeof(T) % 16 == 0, "whole 16-byte words per record");
  const int lane = threadIdx.x % kWarp;
  if (active) {
    T* o = sh + j * XS;
#pragma unroll
    for (int k = 0; k < NX; ++k) o[k] = b[k];
#pragma unroll
    for (int r = 0; r < NX; ++r)
#pragma unroll
      for (int q = 0; q <= r; ++q) o[NX + r * (r + 1) / 2 + q] = U[r * NX + q];
#pragma unroll
    for (int k = NX + NX * (NX + 1) / 2; k < XS; ++k) o[k] = T(0);
  }
  __syncwarp();
  if constexpr (sizeof(T) == 4) {
    const float4* s4 = reinterpret_cast<const float4*>(sh);
    float4* g4 = reinterpret_cast<float4*>(g);
    for (int k = lane; k < cnt * WPR; k += kWarp) g4[k] = s4[k];
  } else {
    const double2* s4 = reinterpret_cast<const double2*>(sh);
    double2* g4 = reinterpret_cast<double2*>(g);
    for (int k = lane; k < cnt * WPR; k += kWarp) g4[k] = s4[k];
  }
}

// The W-value rows of one chunk's cnt consecutive items (lane j holding item
// j's row v) written to their contiguous block g: staged in the warp's
// shared rows sh, then stored lane-strided, each store instruction covering
// consecutive words.
template <typename T, int W>
SQSM_DEV void warp_store_rows(T* __restrict__ g, T* sh, const T* v, int j, int cnt, bool active) {
  const int lane = threadIdx.x % kWarp;
  if (active) {
#pragma unroll
    for (int k = 0; k < W; ++k) sh[j * W + k] = v[k];
  }
  __syncwarp();
  for (int k = lane; k < cnt * W; k += kWarp) g[k] = sh[k];
}

// The carry of item j of chunk c of a chunk-scanned level (one warp per
// chunk, lane j): the chunk's carry applied to the in-chunk prefix before the
// item, that prefix itself where the chunk starts its sequence (flag 0).
// Returns whether the item has a carry.
template <typename T, int NX>
SQSM_DEV bool filter_item_carry(const T* __restrict__ items, const T* __restrict__ carry_in,
                                int flag, int64_t c, int64_t i, int j, bool active, T* cb, T* cU) {
  constexpr int REC = FRec<NX>::size;
  const RowsPacked<T, NX> cin{(T*)carry_in};
  if (!active) {
  } else if (j == 0) {
    cin.load(c, cb, cU);
  } else if (flag) {
    T pb[NX], pU[NX * NX], el[REC];
    cin.load(c, pb, pU);
    vload<T, REC>(items + (i - 1) * REC, el);
    filter_apply<T, NX>(pb, pU, el, cb, cU);
  } else {
    load<T, NX>(items + (i - 1) * REC + FRec<NX>::b, cb);
    load<T, NX * NX>(items + (i - 1) * REC + FRec<NX>::U, cU);
  }
  return j == 0 ? flag != 0 : true;
}

// One thread per item of the level; each warp is one chunk.
template <typename T, int NX>
__global__ void __launch_bounds__(kBlock)
filter_down_cs(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
               const int* __restrict__ flag_in, T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int XS = XRow<NX>::size;
  static_assert(kChunkScan == kWarp && kBlock % kWarp == 0, "one chunk per warp");
  __shared__ __align__(16) T SO[kBlock / kWarp][kWarp * XS];
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t c = tid / kChunkScan;
  if (c >= lv.n_chunks) return;   // uniform per warp
  const int j = (int)(tid - c * kChunkScan);
  const int cnt = lv.count[c];
  const bool active = j < cnt;
  const int64_t i0 = lv.first[c];
  const int64_t i = i0 + j;
  T cb[NX], cU[NX * NX];
  const bool have = filter_item_carry<T, NX>(items, carry_in, flag_in[c], c, i, j, active, cb, cU);
  warp_store_carries<T, NX>(carry_out + i0 * XS, SO[threadIdx.x / kWarp], cb, cU, j, cnt,
                            active);
  if (active) flag_out[i] = have;
}

// filter_down_cs of level 1 and filter_leaf_down in one launch: item i of the
// level is leaf chunk i, so its thread goes on with the chunk's steps and the
// carries stay in registers.  For scans of at most 65536 leaf chunks, where
// the two launches and the carries' way through memory cost more than the
// lower occupancy: with the smoother's pair a track of n = 1000 takes 98 ->
// 90 us an iteration, of 1e5 (two passes) 336 -> 323, the population model at
// n = 10000 27 -> 23.  A batch whose chunks leave lanes idle would spread its
// leaf steps over more warps and keeps the two.
template <typename T, int NX, int NY, typename GV, typename FO>
__global__ void __launch_bounds__(kBlock)
filter_down_leaf(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                 const int* __restrict__ flag_in, DevLevel leaf, DevSeqs sq, GV gv,
                 const T* __restrict__ y, const T* __restrict__ m0, const T* __restrict__ N0,
                 FO fo, double* __restrict__ partial, int* status) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t c = tid / kChunkScan;
  if (c >= lv.n_chunks) return;
  const int j = (int)(tid - c * kChunkScan);
  if (j >= lv.count[c]) return;
  const int64_t i = lv.first[c] + j;
  T m[NX], N[NX * NX];
  const bool have = filter_item_carry<T, NX>(items, carry_in, flag_in[c], c, i, j, true, m, N);
  filter_leaf_steps<T, NX, NY, GV, FO>(leaf, sq, gv, y, m0, N0, fo, partial, status, i, have, m,
                                       N);
}

template <typename T, int NX>
__global__ void __launch_bounds__(kChunkScan)
smoother_up_cs(DevLevel lv, T* __restrict__ items, T* __restrict__ out) {
  constexpr int REC = SRec<NX>::size;
  __shared__ __align__(16) T S[kChunkScan * REC];
  const int64_t c = blockIdx.x;
  const int t = threadIdx.x;
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  T mine[REC], tmp[REC];
  if (t < cnt) vload<T, REC>(items + (i0 + t) * REC, mine);
  for (int d = 1; d < cnt; d <<= 1) {
    if (t < cnt) vstore<T, REC>(S + t * REC, mine);
    __syncwarp();
    if (t + d < cnt) {
      smoother_combine<T, NX>(mine, S + (t + d) * REC, tmp);
      copy<T, REC>(tmp, mine);
    }
    __syncwarp();
  }
  if (t < cnt) vstore<T, REC>(items + (i0 + t) * REC, mine);
  if (t == 0 && cnt > 0) vstore<T, REC>(out + c * REC, mine);
}

// As filter_item_carry, for the smoother's suffixes.
template <typename T, int NX>
SQSM_DEV bool smoother_item_carry(const T* __restrict__ items, const T* __restrict__ carry_in,
                                  int flag, int64_t c, int64_t i, int j, int cnt, bool active,
                                  T* cg, T* cD) {
  constexpr int REC = SRec<NX>::size;
  const RowsPacked<T, NX> cin{(T*)carry_in};
  if (!active) {
  } else if (j == cnt - 1) {
    cin.load(c, cg, cD);
  } else if (flag) {
    T el[REC];
    cin.load(c, cg, cD);
    vload<T, REC>(items + (i + 1) * REC, el);
    smoother_apply<T, NX>(el, cg, cD);
  } else {
    load<T, NX>(items + (i + 1) * REC + SRec<NX>::g, cg);
    load<T, NX * NX>(items + (i + 1) * REC + SRec<NX>::D, cD);
  }
  return j == cnt - 1 ? flag != 0 : true;
}

template <typename T, int NX>
__global__ void __launch_bounds__(kBlock)
smoother_down_cs(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                 const int* __restrict__ flag_in, T* __restrict__ carry_out, int* __restrict__ flag_out) {
  constexpr int XS = XRow<NX>::size;
  static_assert(kChunkScan == kWarp && kBlock % kWarp == 0, "one chunk per warp");
  __shared__ __align__(16) T SO[kBlock / kWarp][kWarp * XS];
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t c = tid / kChunkScan;
  if (c >= lv.n_chunks) return;   // uniform per warp
  const int j = (int)(tid - c * kChunkScan);
  const int cnt = lv.count[c];
  const bool active = j < cnt;
  const int64_t i0 = lv.first[c];
  const int64_t i = i0 + j;
  T cg[NX], cD[NX * NX];
  const bool have =
      smoother_item_carry<T, NX>(items, carry_in, flag_in[c], c, i, j, cnt, active, cg, cD);
  warp_store_carries<T, NX>(carry_out + i0 * XS, SO[threadIdx.x / kWarp], cg, cD, j, cnt,
                            active);
  if (active) flag_out[i] = have;
}

// smoother_down_cs of level 1 and smoother_leaf_down in one launch (see
// filter_down_leaf).
template <typename T, int NX, int NY, typename GV, typename FO, typename SO>
__global__ void __launch_bounds__(kBlock)
smoother_down_leaf(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry_in,
                   const int* __restrict__ flag_in, DevLevel leaf, DevSeqs sq, GV gv, FO fo,
                   SO out_rows, int* status, bool add_nominal, unsigned* dmax, PriorMean<T> pm) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t c = tid / kChunkScan;
  if (c >= lv.n_chunks) return;
  const int j = (int)(tid - c * kChunkScan);
  const int cnt = lv.count[c];
  if (j >= cnt) return;
  const int64_t i = lv.first[c] + j;
  T gm[NX], Dm[NX * NX];
  smoother_item_carry<T, NX>(items, carry_in, flag_in[c], c, i, j, cnt, true, gm, Dm);
  smoother_leaf_steps<T, NX, NY, GV, FO, SO>(leaf, sq, gv, fo, out_rows, status, add_nominal, dmax,
                                             pm, i, gm, Dm);
}

// Leaf kernels of short FP32 scans with the steps of a leaf chunk side by
// side: the elements of a chunk's kLeafPar rows do not depend on one another,
// so each is built by a thread of its own warp (lane: chunk) and only the
// combines, or the RTS steps, are one after another.  A call of a few thousand
// steps has fewer warps than schedulers either way, and its leaf kernels take
// one element's chain instead of three.  Same operations on the same values
// as the one-thread kernels.  Four iterations over one track (us, one thread
// against side by side): n = 300 344 -> 276, 3000 407 -> 329, 12000 490 -> 422,
// 49000 574 -> 544; smoother of a linear model, n = 3000, 99 -> 79.
constexpr int kLeafPar = 3;

template <typename T, int NX, int NY, typename GV, typename FO>
SQSM_DEV void smoother_row_element(const DevSeqs& sq, const GV& gv, const FO& fo, int b, int64_t e,
                                   T* el) {
  T m[NX], N[NX * NX];
  const int64_t k = e - (sq.offsets[b] + b);
  const int64_t nb = sq.offsets[b + 1] - sq.offsets[b];
  fo.load(e, m, N);
  if (k == nb) {
    smoother_element_last<T, NX>(m, N, el);
  } else {
    Gamma<T, NX, NY> g;
    g.load_transition(gv, sq.offsets[b] + k);
    smoother_element<T, NX, NY>(g, m, N, el);
  }
}

// See smoother_leaf_up.
template <typename T, int NX, int NY, typename GV, typename FO>
__global__ void __launch_bounds__(kWarp * kLeafPar)
smoother_leaf_up_par(DevLevel lv, DevSeqs sq, GV gv, FO fo, T* __restrict__ items,
                     T* __restrict__ etab) {
  constexpr int REC = SRec<NX>::size;
  __shared__ __align__(16) T S[kLeafPar][kWarp * REC];
  const int lane = threadIdx.x % kWarp, j = threadIdx.x / kWarp;
  const int64_t c = blockIdx.x * (int64_t)kWarp + lane;
  const bool in = c < lv.n_chunks;
  const int cnt = in ? lv.count[c] : 0;
  if (j < cnt) {
    const int b = lv.seq[c];
    const int64_t e = lv.first[c] + j;
    T el[REC];
    smoother_row_element<T, NX, NY, GV, FO>(sq, gv, fo, b, e, el);
    if (etab && e != sq.offsets[b + 1] + b)
      vstore<T, ETab<NX>::size>(etab + e * ETab<NX>::size, el + SRec<NX>::E);
    vstore<T, REC>(S[j] + lane * REC, el);
  }
  __syncthreads();
  if (j == 0 && in) {
    T agg[REC], el[REC], tmp[REC];
    vload<T, REC>(S[cnt - 1] + lane * REC, agg);
    for (int i = cnt - 2; i >= 0; --i) {
      vload<T, REC>(S[i] + lane * REC, el);
      smoother_combine<T, NX>(el, agg, tmp);
      copy<T, REC>(tmp, agg);
    }
    vstore<T, REC>(items + c * REC, agg);
  }
}

// See smoother_leaf_down and smoother_down_leaf (FUSED: lv is level 1 and a
// block one of its chunks; otherwise carry / flag are the leaf chunks').  The
// last warp takes the carry while the others build the elements.
template <typename T, int NX, int NY, bool FUSED, typename GV, typename FO, typename SO>
__global__ void __launch_bounds__(kWarp * (kLeafPar + 1))
smoother_leaf_down_par(DevLevel lv, const T* __restrict__ items, const T* __restrict__ carry,
                       const int* __restrict__ flag, DevLevel leaf, DevSeqs sq, GV gv, FO fo,
                       SO out_rows, int* status, bool add_nominal, unsigned* dmax,
                       PriorMean<T> prior) {
  static_assert(kChunkScan == kWarp, "one chunk per block");
  constexpr int REC = SRec<NX>::size;
  __shared__ __align__(16) T S[kLeafPar][kWarp * REC];
  const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
  int64_t c;
  bool in;
  if constexpr (FUSED) {
    in = lane < lv.count[blockIdx.x];
    c = lv.first[blockIdx.x] + lane;
  } else {
    c = blockIdx.x * (int64_t)kWarp + lane;
    in = c < leaf.n_chunks;
  }
  const int cnt = in ? leaf.count[c] : 0;
  const int b = in ? leaf.seq[c] : 0;
  const int64_t e0 = in ? leaf.first[c] : 0;
  const int64_t r0 = sq.offsets[b] + b, nb = sq.offsets[b + 1] - sq.offsets[b];
  T gm[NX], Dm[NX * NX];
  if (w < kLeafPar) {
    if (w < cnt) {
      T el[REC];
      smoother_row_element<T, NX, NY, GV, FO>(sq, gv, fo, b, e0 + w, el);
      vstore<T, REC>(S[w] + lane * REC, el);
    }
  } else if (in) {
    if constexpr (FUSED)
      smoother_item_carry<T, NX>(items, carry, flag[blockIdx.x], blockIdx.x, c, lane,
                                 lv.count[blockIdx.x], true, gm, Dm);
    else if (flag[c]) RowsPacked<T, NX>{(T*)carry}.load(c, gm, Dm);
  }
  __syncthreads();
  if (w < kLeafPar || !in) return;
  float change = 0.f;
  bool ok = true;
  const bool need_old = add_nominal || dmax != nullptr;
  for (int j = cnt - 1; j >= 0; --j) {
    const int64_t e = e0 + j;
    T el[REC], old[NX], out[NX];
    vload<T, REC>(S[j] + lane * REC, el);
    if (need_old) out_rows.load_mean(e, old);
    if (e - r0 == nb) {
#pragma unroll
      for (int i = 0; i < NX; ++i) gm[i] = el[SRec<NX>::g + i];
#pragma unroll
      for (int i = 0; i < NX * NX; ++i) Dm[i] = el[SRec<NX>::D + i];
    } else {
      smoother_apply<T, NX>(el, gm, Dm);
    }
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      out[i] = add_nominal ? old[i] + gm[i] : gm[i];
      if (dmax) change = fmaxf(change, fabsf((float)(add_nominal ? gm[i] : gm[i] - old[i])));
      ok = ok && finite(gm[i]);
    }
    out_rows.store(e, out, Dm);
    if (e == r0 && prior.dm0) {
#pragma unroll
      for (int i = 0; i < NX; ++i)
        prior.dm0[(int64_t)b * NX + i] = prior.m0[(int64_t)b * NX + i] - out[i];
    }
  }
  if (!ok) flag_status(status, 8);
  if (dmax) {   // see smoother_leaf_steps
    unsigned bits = __float_as_uint(ok ? change : INFINITY);
    const unsigned mask = __activemask();
    bits = __reduce_max_sync(mask, bits);
    if (lane == __ffs(mask) - 1) atomicMax(dmax, bits);
  }
}

// See filter_leaf_up: the elements side by side, then each combine by three
// threads, one per part (see filter_ks3).
template <typename T, int NX, int NY, typename GV>
__global__ void __launch_bounds__(kWarp * kLeafPar)
filter_leaf_up_par(DevLevel lv, DevSeqs sq, GV gv, const T* __restrict__ y,
                   const T* __restrict__ m0, const T* __restrict__ N0, T* __restrict__ items) {
  using R = FRec<NX>;
  constexpr int REC = R::size, NZ = NX < NY ? NX : NY;
  __shared__ __align__(16) T S[kLeafPar][kWarp * REC];
  const int lane = threadIdx.x % kWarp, w = threadIdx.x / kWarp;
  const int64_t c = blockIdx.x * (int64_t)kWarp + lane;
  const bool in = c < lv.n_chunks;
  const int cnt = in ? lv.count[c] : 0;
  if (w < cnt) {
    const int b = lv.seq[c];
    const int64_t s = lv.first[c] + w;
    T el[REC], ys[NY], m0b[NX], N0b[NX * NX];
    load<T, NX>(m0 + (int64_t)b * NX, m0b);
    load_lower<T, NX>(N0 + (int64_t)b * NX * NX, N0b);
    Gamma<T, NX, NY> g;
    g.load_all(gv, s);
    load<T, NY>(y + s * NY, ys);
    filter_element<T, NX, NY>(g, ys, s == sq.offsets[b], m0b, N0b, el);
    if (cnt == 1) lower_Z<T, NX, NY>(el + R::Z);
    vstore<T, REC>(S[w] + lane * REC, el);
  }
  __syncthreads();
  T* agg = S[0] + lane * REC;
  if constexpr (NX < 5) {
    // (at n_x = 4 the parts' separate code would fuse other products than the
    // whole combine's, and round differently)
    if (w == 0 && cnt > 1) {
      T acc[REC], el[REC], tmp[REC];
      vload<T, REC>(agg, acc);
      for (int i = 1; i < cnt; ++i) {
        vload<T, REC>(S[i] + lane * REC, el);
        filter_combine<T, NX, 7, true, NZ>(acc, el, tmp);
        copy<T, REC>(tmp, acc);
      }
      vstore<T, REC>(agg, acc);
    }
    __syncthreads();
  } else {
    for (int i = 1; i < kLeafPar; ++i) {
      T part[REC];
      const T* ej = S[i] + lane * REC;
      if (i < cnt) {
        if (w == 0) filter_combine<T, NX, 1, true, NZ>(agg, ej, part);
        else if (w == 1) filter_combine<T, NX, 2, true, NZ>(agg, ej, part);
        else filter_combine<T, NX, 4, true, NZ>(agg, ej, part);
      }
      __syncthreads();
      if (i < cnt) {
        if (w == 0) {
#pragma unroll
          for (int k = R::A; k < R::U; ++k) agg[k] = part[k];
#pragma unroll
          for (int k = R::eta; k < R::Z; ++k) agg[k] = part[k];
        } else if (w == 1) {
#pragma unroll
          for (int k = R::U; k < R::eta; ++k) agg[k] = part[k];
        } else {
#pragma unroll
          for (int k = R::Z; k < R::Z + NX * NX; ++k) agg[k] = part[k];
        }
      }
      __syncthreads();
    }
  }
  // the block's chunks are consecutive: their records go out as one block
  const int64_t c0 = blockIdx.x * (int64_t)kWarp;
  const int n = lv.n_chunks - c0 < kWarp ? (int)(lv.n_chunks - c0) : kWarp;
  const float4* S4 = reinterpret_cast<const float4*>(S[0]);
  float4* I4 = reinterpret_cast<float4*>(items + c0 * REC);
  for (int k = threadIdx.x; k < n * REC * (int)sizeof(T) / 16; k += blockDim.x) I4[k] = S4[k];
}

inline unsigned cs_down_grid(int64_t chunks) {
  return (unsigned)((chunks * kChunkScan + kBlock - 1) / kBlock);
}

// Where a full filter pass stores, for one level, what the mean-only
// refinement passes replay (refine_scan.cuh); rec null: nothing is stored.
// For Kogge-Stone round r and item i of the level (n items): the record at
// the round's start at rec[(r * n + i) * FRec] and the combine's G and
// A_j (I - U_i G^T) at gm[(r * n + i) * FGm]; for chunk levels also the
// records the scan leaves at fin[i * FRec] (fin null at the top).
template <typename T> struct FMeansTab {
  T* rec;
  T* gm;
  T* fin;
  int64_t n;
};

// Filter scans with three threads per combine.  In the latency-bound top
// levels (few chunks, one warp per SM or less) a combine's chain of dependent
// instructions sets the time per Kogge-Stone round.  Thread (role r, item t)
// computes only part r of S[t - d] (x) S[t] (r = 0: A, b, eta; 1: U; 2: Z;
// each forms the factors it needs itself), which shortens that chain; role
// r runs in warps of its own, so no warp diverges.
//
// With STORE, the rounds also store what the mean-only refinement passes
// replay (FMeansTab, here offset to the first item): the records at the
// start of round r at trec[(r * n + t) * REC] and each combine's G and
// A_j (I - U_i G^T) at tgm[(r * n + t) * FGm].
template <typename T, int NX, int CAP, bool STORE = false>
SQSM_DEV void filter_ks3(T* S, int c, T* trec = nullptr, T* tgm = nullptr, int64_t n = 0) {
  using R = FRec<NX>;
  constexpr int REC = R::size, W = REC * sizeof(T) / 16, GMS = FGm<NX>::size;
  static_assert(CAP % 32 == 0, "roles in whole warps");
  const int role = threadIdx.x / CAP, t = threadIdx.x - role * CAP;
  int r = 0;
  for (int d = 1; d < c; d <<= 1, ++r) {
    if constexpr (STORE) {   // S is read-only until the barrier below
      const float4* S4 = reinterpret_cast<const float4*>(S);
      float4* D4 = reinterpret_cast<float4*>(trec + r * n * REC);
      for (int w = threadIdx.x; w < c * W; w += blockDim.x) D4[w] = S4[w];
    }
    T part[REC];
    const bool act = t < c && t >= d;
    if (act) {
      const T* ei = S + (t - d) * REC;
      const T* ej = S + t * REC;
      if (role == 0) {
        if constexpr (STORE) filter_combine<T, NX, 1>(ei, ej, part, tgm + (r * n + t) * GMS);
        else filter_combine<T, NX, 1>(ei, ej, part);
      } else if (role == 1) filter_combine<T, NX, 2>(ei, ej, part);
      else filter_combine<T, NX, 4>(ei, ej, part);
    }
    __syncthreads();
    if (act) {
      T* o = S + t * REC;
      if (role == 0) {
#pragma unroll
        for (int i = R::A; i < R::U; ++i) o[i] = part[i];      // A, b
#pragma unroll
        for (int i = R::eta; i < R::Z; ++i) o[i] = part[i];    // eta
      } else if (role == 1) {
#pragma unroll
        for (int i = R::U; i < R::eta; ++i) o[i] = part[i];
      } else {
#pragma unroll
        for (int i = R::Z; i < R::Z + NX * NX; ++i) o[i] = part[i];
      }
    }
    __syncthreads();
  }
}

// Chunk-scan up level (see filter_up_cs) with three threads per combine: one
// block of 3 x 32 threads per chunk.  STORE: also fill tb (a full pass
// followed by mean-only ones).
template <typename T, int NX, bool STORE>
__global__ void __launch_bounds__(3 * kChunkScan)
filter_up_cs3(DevLevel lv, T* __restrict__ items, T* __restrict__ out, FMeansTab<T> tb) {
  constexpr int REC = FRec<NX>::size, W = REC * sizeof(T) / 16;   // 16-byte words
  __shared__ __align__(16) T S[kChunkScan * REC];
  const int64_t c = blockIdx.x;
  const int64_t i0 = lv.first[c];
  const int cnt = lv.count[c];
  float4* S4 = reinterpret_cast<float4*>(S);
  float4* I4 = reinterpret_cast<float4*>(items + i0 * REC);
  for (int w = threadIdx.x; w < cnt * W; w += blockDim.x) S4[w] = I4[w];
  __syncthreads();
  if constexpr (STORE)
    filter_ks3<T, NX, kChunkScan, true>(S, cnt, tb.rec + i0 * REC, tb.gm + i0 * FGm<NX>::size,
                                        tb.n);
  else
    filter_ks3<T, NX, kChunkScan>(S, cnt);
  for (int w = threadIdx.x; w < cnt * W; w += blockDim.x) I4[w] = S4[w];
  if constexpr (STORE) {
    float4* F4 = reinterpret_cast<float4*>(tb.fin + i0 * REC);
    for (int w = threadIdx.x; w < cnt * W; w += blockDim.x) F4[w] = S4[w];
  }
  float4* O4 = reinterpret_cast<float4*>(out + c * REC);
  for (int w = threadIdx.x; w < W; w += blockDim.x) O4[w] = S4[(cnt - 1) * W + w];
}

// Top of the tree (see filter_top_ks) with three threads per combine, for
// sequences of at most Ks3Max items at that level (64, fewer where the
// records would not fit 48 KB of static shared memory).
constexpr int ks3_max_items(int rec_bytes) {
  return (48 * 1024) / rec_bytes / 32 * 32 < 64 ? (48 * 1024) / rec_bytes / 32 * 32 : 64;
}
template <typename T, int REC> struct Ks3Max {
  static constexpr int value = ks3_max_items(REC * (int)sizeof(T));
};

template <typename T, int NX, bool STORE>
__global__ void __launch_bounds__(3 * Ks3Max<T, FRec<NX>::size>::value)
filter_top_ks3(const int64_t* __restrict__ seq_item_off, const T* __restrict__ items,
               T* __restrict__ carry_out, int* __restrict__ flag_out, FMeansTab<T> tb) {
  constexpr int REC = FRec<NX>::size, W = REC * sizeof(T) / 16;
  constexpr int KS = Ks3Max<T, REC>::value;
  __shared__ __align__(16) T S[KS * REC];
  const int b = blockIdx.x;
  const int64_t i0 = seq_item_off[b];
  const int c = (int)(seq_item_off[b + 1] - i0);
  float4* S4 = reinterpret_cast<float4*>(S);
  const float4* I4 = reinterpret_cast<const float4*>(items + i0 * REC);
  for (int w = threadIdx.x; w < c * W; w += blockDim.x) S4[w] = I4[w];
  __syncthreads();
  if constexpr (STORE)
    filter_ks3<T, NX, KS, true>(S, c, tb.rec + i0 * REC, tb.gm + i0 * FGm<NX>::size, tb.n);
  else
    filter_ks3<T, NX, KS>(S, c);
  const int t = threadIdx.x;
  if (t < c) {
    if (t > 0) {
      const T* p = S + (t - 1) * REC;
      RowsPacked<T, NX>{carry_out}.store(i0 + t, p + FRec<NX>::b, p + FRec<NX>::U);
    }
    flag_out[i0 + t] = t > 0 ? 1 : 0;
  }
}

}  // namespace sqsm
