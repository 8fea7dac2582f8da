// Pre-selection kernels' host side and the finish kernels; the tensor-core
// kernel is in kernel_presel.cuh, instantiated here for the shared time-grid
// operand (VAR 0) and in kernel_presel_permode.cu / kernel_presel_polres.cu for the
// per-mode (relative binning) and polarisation-resolved operands, so that the
// three instantiation sets compile in parallel.
#include "kernel_presel.cuh"

namespace dotpe {

template <int VAR>
cudaError_t launch_presel_var(const CUtensorMap &mapG, const CUtensorMap &mapBank, const PreselParams &p, bool bf16,
                              bool split, int grid, cudaStream_t st);
template <>
cudaError_t launch_presel_var<0>(const CUtensorMap &mapG, const CUtensorMap &mapBank, const PreselParams &p,
                                 bool bf16, bool split, int grid, cudaStream_t st) {
  return launch_presel_pm<0>(mapG, mapBank, p, bf16, split, grid, st);
}

// Per row: ln L^ML_{ik} and (o, t) from the packed maxima, ln L^inco.ML_i =
// sum_k (FP64), and the running maximum of ln L^inco.ML (order-preserving
// bits of a non-negative double).
__global__ void presel_rows_kernel(int64_t n, int D, int n_phi, const unsigned long long *__restrict__ keys,
                                   float *__restrict__ ml, int *__restrict__ arg_ot, double *__restrict__ inco,
                                   unsigned long long *max_bits) {
  __shared__ unsigned long long smax[8];
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  unsigned long long mb = 0;
  if (i < n) {
    double s = 0.0;
    for (int k = 0; k < D; ++k) {
      const unsigned long long key = keys[i * D + k];
      const float v = __uint_as_float((uint32_t)(key >> 32));
      const uint32_t idx = 0xffffffffu - (uint32_t)(key & 0xffffffffu);
      ml[i * D + k] = v;
      arg_ot[(i * D + k) * 2] = (int)(idx % (uint32_t)n_phi);
      arg_ot[(i * D + k) * 2 + 1] = (int)(idx / (uint32_t)n_phi);
      s += (double)v;
    }
    inco[i] = s;
    mb = (unsigned long long)__double_as_longlong(s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mb, o);
    mb = v > mb ? v : mb;
  }
  if ((threadIdx.x & 31) == 0) smax[threadIdx.x >> 5] = mb;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long m = 0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) m = smax[q] > m ? smax[q] : m;
    atomicMax(max_bits, m);
  }
}

// Sec. IV.D selection: rows with ln L^inco.ML >= max - delta, in increasing
// order, and the lowest row that attains the maximum.  A block of PS_NT threads takes
// PS_ROWS rows (8 consecutive ones per thread); the first kernel leaves each block's
// count and its first row at the maximum, the second writes the rows at the prefix of
// the earlier blocks' counts.  One block walking the rows was a chain of scans on one
// SM: 67 us for 65,536 rows; the two kernels take 4.4 and 4.6 us.
namespace {
constexpr int PS_NT = 256, PS_ROWS = PS_NT * 8;
}

__device__ __forceinline__ uint32_t presel_keep(int64_t n, int64_t r0, const double *__restrict__ inco, double thr) {
  uint32_t keep = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q)
    if (r0 + q < n && inco[r0 + q] >= thr) keep |= 1u << q;
  return keep;
}

// blk[block] = count << 32 | first row at the maximum within the block (PS_ROWS: none)
__global__ void __launch_bounds__(PS_NT)
presel_count_kernel(int64_t n, double delta, const double *__restrict__ inco, const unsigned long long *max_bits,
                    unsigned long long *__restrict__ blk) {
  __shared__ unsigned cnt, first;
  if (threadIdx.x == 0) { cnt = 0; first = PS_ROWS; }
  __syncthreads();
  const double mx = __longlong_as_double((long long)*max_bits);
  const int64_t r0 = (int64_t)blockIdx.x * PS_ROWS + threadIdx.x * 8;
  const uint32_t keep = presel_keep(n, r0, inco, mx - delta);
  unsigned at = PS_ROWS;
#pragma unroll
  for (int q = 7; q >= 0; --q)
    if (r0 + q < n && inco[r0 + q] == mx) at = threadIdx.x * 8 + q;
  const unsigned c = __reduce_add_sync(0xffffffffu, __popc(keep));
  at = __reduce_min_sync(0xffffffffu, at);
  if ((threadIdx.x & 31) == 0) {
    if (c) atomicAdd(&cnt, c);
    if (at < PS_ROWS) atomicMin(&first, at);
  }
  __syncthreads();
  if (threadIdx.x == 0) blk[blockIdx.x] = (unsigned long long)cnt << 32 | first;
}

__global__ void __launch_bounds__(PS_NT)
presel_select_kernel(int64_t n, double delta, const double *__restrict__ inco, const unsigned long long *max_bits,
                     const unsigned long long *__restrict__ blk, int64_t *__restrict__ sel, PreselOut *out) {
  __shared__ long long wsum[PS_NT / 32], wbase[PS_NT / 32];
  __shared__ int s_arg_blk;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const double mx = __longlong_as_double((long long)*max_bits);
  const double thr = mx - delta;
  const bool last = blockIdx.x == gridDim.x - 1;
  if (threadIdx.x == 0) s_arg_blk = (int)gridDim.x;
  __syncthreads();
  long long base = 0;  // rows kept by the earlier blocks
  for (int j = threadIdx.x; j < (int)blockIdx.x; j += PS_NT) base += (long long)(blk[j] >> 32);
  if (last)
    for (int j = threadIdx.x; j < (int)gridDim.x; j += PS_NT)
      if ((uint32_t)blk[j] < PS_ROWS) { atomicMin(&s_arg_blk, j); break; }
  const int64_t r0 = (int64_t)blockIdx.x * PS_ROWS + threadIdx.x * 8;
  const uint32_t keep = presel_keep(n, r0, inco, thr);
  const int cnt = __popc(keep);
  long long x = cnt;  // inclusive over the lanes
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) base += __shfl_xor_sync(0xffffffffu, base, o);
  if (lane == 31) { wsum[wid] = x; wbase[wid] = base; }
  __syncthreads();
  long long at = x - cnt, total = 0;
#pragma unroll
  for (int j = 0; j < PS_NT / 32; ++j) {
    at += wbase[j] + (j < wid ? wsum[j] : 0);
    total += wbase[j] + wsum[j];
  }
#pragma unroll
  for (int q = 0; q < 8; ++q)
    if (keep >> q & 1u) sel[at++] = r0 + q;
  if (last && threadIdx.x == 0) {
    const int j = s_arg_blk;
    out->max_inco = mx;
    out->threshold = thr;
    out->arg_i = j < (int)gridDim.x ? (int64_t)j * PS_ROWS + (uint32_t)blk[j] : 0;
    out->n_selected = total;
  }
}

int launch_presel(const CUtensorMap &mapG, const CUtensorMap &mapBank, const PreselParams &p, bool bf16, bool split,
                  bool per_mode, bool pol, int n_sms, cudaStream_t st) {
  const int total = p.n_itile * p.n_ctile;
  const int grid = total < n_sms ? (total > 0 ? total : 1) : n_sms;
  const cudaError_t e = pol ? launch_presel_var<2>(mapG, mapBank, p, bf16, split, grid, st)
                            : per_mode ? launch_presel_var<1>(mapG, mapBank, p, bf16, split, grid, st)
                                       : launch_presel_var<0>(mapG, mapBank, p, bf16, split, grid, st);
  return (int)e;
}

void launch_presel_finish(int64_t n, int D, int n_phi, double delta, unsigned long long *keys, float *ml,
                          int *arg_ot, double *inco, unsigned long long *max_bits, int64_t *sel, PreselOut *out,
                          cudaStream_t st) {
  const int64_t blocks = (n + 255) / 256;
  presel_rows_kernel<<<(unsigned)(blocks > 0 ? blocks : 1), 256, 0, st>>>(n, D, n_phi, keys, ml, arg_ot, inco,
                                                                          max_bits);
  // the rows' packed maxima are read: their first words hold the blocks' counts
  const unsigned nb = (unsigned)(n > 0 ? (n + PS_ROWS - 1) / PS_ROWS : 1);
  presel_count_kernel<<<nb, PS_NT, 0, st>>>(n, delta, inco, max_bits, keys);
  presel_select_kernel<<<nb, PS_NT, 0, st>>>(n, delta, inco, max_bits, keys, sel, out);
}

}  // namespace dotpe
