// Kernels shared by all paths.
#include <algorithm>

#include "dispatch.h"

namespace sqsm {

// Sum of part[lo], part[lo + stride], ... below hi by a block of 256 threads,
// in a fixed order (strided partial sums, then a tree), so that the result does
// not depend on scheduling (valid in thread 0).
__device__ double block_sum(const double* part, int64_t lo, int64_t hi, int64_t stride) {
  __shared__ double buf[256];
  double acc = 0.0;
  for (int64_t i = lo + threadIdx.x * stride; i < hi; i += blockDim.x * stride) acc += part[i];
  buf[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) buf[threadIdx.x] += buf[threadIdx.x + w];
    __syncthreads();
  }
  return buf[0];
}

// One block per sequence.
__global__ void loglik_reduce(DevSeqs sq, const double* __restrict__ partial, int64_t stride,
                              double* __restrict__ loglik, int* status) {
  const int b = blockIdx.x;
  const double v = block_sum(partial, sq.leaf_chunk_off[b], sq.leaf_chunk_off[b + 1], stride);
  if (threadIdx.x == 0) {
    loglik[b] = v;
    if (!isfinite(v) && status) atomicOr(status, 8);
  }
}

// First stage for long sequences: block (slice, sequence) puts the sum of its
// slice in the slice's first entry.
__global__ void loglik_slices(DevSeqs sq, double* partial, int64_t slice) {
  const int b = blockIdx.y;
  const int64_t hi = sq.leaf_chunk_off[b + 1], lo = sq.leaf_chunk_off[b] + blockIdx.x * slice;
  if (lo >= hi) return;
  const double v = block_sum(partial, lo, lo + slice < hi ? lo + slice : hi, 1);
  if (threadIdx.x == 0) partial[lo] = v;
}

// One SM adds a warp of doubles in 19 cycles, so a block per sequence takes
// 0.7 us a slice (13 us for the 33334 chunks of n = 1e5), and sequences of
// more than a slice are summed in slices by many blocks first (7 us, both
// launches).  The grid has the longest sequence's slices for every sequence
// (0.6 ns a block, empty or not), and many sequences fill the GPU with a block
// each: for one sequence of 123 slices among B short ones the sum takes 130 us
// in one launch at any B up to 3000, and sliced 16 at B = 100, 76 at 1000, 210
// at 3000, 3998 at 60000 (in one launch 269); for 300 sequences of 4 slices
// 13 us in one launch, 18 sliced.
constexpr int64_t kLoglikSlice = 2048;

void enqueue_loglik_reduce(DevSeqs sq, double* partial, int64_t max_chunks, double* loglik,
                           int* status, cudaStream_t s, Prof* P) {
  const int64_t slices = (max_chunks + kLoglikSlice - 1) / kLoglikSlice;
  const bool sliced = slices > 1 && sq.B <= std::min<int64_t>(32 * slices, 1000);
  if (sliced) {
    ProfScope ps(P, K_LOGLIK, s);
    loglik_slices<<<dim3((unsigned)slices, (unsigned)sq.B), 256, 0, s>>>(sq, partial,
                                                                          kLoglikSlice);
  }
  ProfScope ps(P, K_LOGLIK, s);
  loglik_reduce<<<sq.B, 256, 0, s>>>(sq, partial, sliced ? kLoglikSlice : 1, loglik, status);
}

namespace {

// N0 = chol(P0) per sequence in FP64 (one thread per sequence; the lower
// triangle of P0 is read, the factor is written with zeros above the
// diagonal).  A pivot that is not positive (P0 not positive definite) or not
// finite makes the whole factor NaN and sets SQSM_ERR_NOT_PD (4).
template <typename T>
__global__ void prior_cholesky(int64_t batch, int nx, const T* __restrict__ P0,
                               T* __restrict__ N0, int* status) {
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b >= batch) return;
  const T* P = P0 + b * nx * nx;
  T* N = N0 + b * nx * nx;
  double L[kMaxPriorNx * kMaxPriorNx];
  bool pd = true;
  for (int j = 0; j < nx; ++j) {
    double d = (double)P[j * nx + j];
    for (int k = 0; k < j; ++k) d -= L[j * kMaxPriorNx + k] * L[j * kMaxPriorNx + k];
    if (!(d > 0.0) || !isfinite(d)) pd = false;
    const double ljj = sqrt(d > 0.0 ? d : 1.0);
    L[j * kMaxPriorNx + j] = ljj;
    for (int i = j + 1; i < nx; ++i) {
      double v = (double)P[i * nx + j];
      for (int k = 0; k < j; ++k) v -= L[i * kMaxPriorNx + k] * L[j * kMaxPriorNx + k];
      L[i * kMaxPriorNx + j] = v / ljj;
    }
  }
  for (int i = 0; i < nx; ++i)
    for (int j = 0; j < nx; ++j)
      N[i * nx + j] = !pd ? T(NAN) : j <= i ? (T)L[i * kMaxPriorNx + j] : T(0);
  if (!pd && status) atomicOr(status, 4);
}

__global__ void ipls_tol_check(unsigned* dmax, int* iters, int max_iters, float tol,
                               cudaGraphConditionalHandle handle, int use_handle, int* go) {
  const float d = __uint_as_float(*dmax);
  const int it = *iters + 1;
  *iters = it;
  *dmax = 0u;
  const unsigned more = (!(d < tol) && it < max_iters) ? 1u : 0u;
  if (use_handle) cudaGraphSetConditional(handle, more);
  if (go) *go = (int)more;
}

// One group of a grouped NLL + gradient evaluation: g = {nll, grad[n_theta],
// adj_change, ipls_change} of the group; the first group is copied, later
// ones are added (nll, grad) or maxed (changes; NaN, an unsettled change,
// stays NaN).
__global__ void nll_grad_group_add(int first, int n_theta, const double* __restrict__ g,
                                   double* nll, double* grad, double* adj_change,
                                   double* ipls_change) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  auto mx = [](double a, double b) { return (a != a || b != b) ? NAN : (a > b ? a : b); };
  if (first) {
    nll[0] = g[0];
    for (int i = 0; i < n_theta; ++i) grad[i] = g[1 + i];
    if (adj_change) adj_change[0] = g[5];
    if (ipls_change) ipls_change[0] = g[6];
  } else {
    nll[0] += g[0];
    for (int i = 0; i < n_theta; ++i) grad[i] += g[1 + i];
    if (adj_change) adj_change[0] = mx(adj_change[0], g[5]);
    if (ipls_change) ipls_change[0] = mx(ipls_change[0], g[6]);
  }
}

}  // namespace

void enqueue_nll_grad_group_add(int first, int n_theta, const double* g, double* nll, double* grad,
                                double* adj_change, double* ipls_change, cudaStream_t s) {
  nll_grad_group_add<<<1, 1, 0, s>>>(first, n_theta, g, nll, grad, adj_change, ipls_change);
}

void enqueue_prior_cholesky(int dtype_f64, int64_t batch, int nx, const void* P0, void* N0,
                            int* status, cudaStream_t s) {
  const unsigned blocks = (unsigned)((batch + 127) / 128);
  if (dtype_f64)
    prior_cholesky<double><<<blocks, 128, 0, s>>>(batch, nx, (const double*)P0, (double*)N0,
                                                  status);
  else
    prior_cholesky<float><<<blocks, 128, 0, s>>>(batch, nx, (const float*)P0, (float*)N0, status);
}

void enqueue_tol_check(unsigned* dmax, int* iters, int max_iters, float tol,
                       cudaGraphConditionalHandle handle, int use_handle, int* go, cudaStream_t s) {
  ipls_tol_check<<<1, 1, 0, s>>>(dmax, iters, max_iters, tol, handle, use_handle, go);
}

}  // namespace sqsm
