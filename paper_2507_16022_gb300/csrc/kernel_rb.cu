// Relative-binning weights (App. A, Eqs. dh_weights, hh_weights).
//
// The components m are the bank's modes, or its (mode, polarisation) pairs
// m = 2 m_az + p for a polarisation-resolved bank (W_{kmpb}, W_{kmm'pp'b}); up to
// 2 MAXM of them.  For detector d, component m (and m') and coarse node b:
//   W^{<d|h>}_{d m b}    = sum_n 4 dff_n d_d(f_n) h0_dm^*(f_n) s_b(f_n) / S_d(f_n)  /  h0_dm^*(f_b)
//   W^{<h|h>}_{d m m' b} = sum_n 4 dff_n h0_dm(f_n) h0_dm'^*(f_n) s_b(f_n) / S_d(f_n) / (h0_dm(f_b) h0_dm'^*(f_b))
// with h0_dm(f) = h0_m(f) e^{-2 pi i f t0_d} (the reference arriving at the
// detector at t0_d) and s_b the piecewise-linear hat function of node b on the
// fine grid (1 at f_b, 0 at the neighbouring nodes), so the sums run over the
// fine points between nodes b-1 and b+1, in FP64 (the weights are made once per
// event) and in a fixed order.  W^{<h|h>} is Hermitian in (m, m'): the upper triangle
// is summed and mirrored; the arrival phase drops out of it.
//
// FP64 runs at 2 operations per clock and SM, and all of this is FP64: the kernel is
// bound by its instruction count, not by the 20 MB or so that it reads.  A block takes up
// to RB_PART points of one interval between nodes (intervals differ 50-fold in length, so
// a block per node leaves the chip waiting for the longest); a point's phase, weight and
// products are formed once and added to both neighbouring nodes; |h_m|^2 has no imaginary
// part to sum.  The threads' sums are added column by column from shared memory (an FP64
// shuffle reduction costs each warp 10 instructions per sum).  A second kernel adds a
// node's parts and divides by h0(f_b), a lane per weight.
// 131,072 points, 378 nodes, 3 detectors, 4 modes: 188 us and 12 us for the second kernel
// (531 us with a block per node).
#include "common.cuh"
#include "kernels.h"

namespace dotpe {

namespace {
constexpr int RB_THREADS = 128, RB_FIN_THREADS = 64;
constexpr int RB_PART = 512;  // points per block
// NC: components per weight set, MAXM modes or 2 MAXM (mode, polarisation) pairs.
// Sums of a node: NC complex <d|h>, NC real |h_m|^2, then the complex pairs m < m'.
// With MAXM components a thread keeps the sums for both nodes of its interval (48
// doubles); with 2 MAXM (80 doubles a node) a block sums for one of the nodes.
template <int NC> struct RbAcc {
  static constexpr int NPAIR = NC * (NC - 1) / 2;
  static constexpr int NACC = 3 * NC + 2 * NPAIR;
  static constexpr bool BOTH = NC <= MAXM;
};

// e^{-2 pi i f t} in FP64 (the phase reduced with sincospi of the product f t)
__device__ __forceinline__ double2 shift64(double f, double t) {
  double s, c;
  sincospi(2.0 * f * t, &s, &c);
  return make_double2(c, -s);
}
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {  // a b^*
  return make_double2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
__device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
  const double den = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / den, (a.y * b.x - a.x * b.y) / den);
}
}  // namespace

// hat function of node b (frequencies of its neighbours and its own) at f
__device__ __forceinline__ double rb_hat(double f, double fbm, double fb, double fbp, bool first, bool last) {
  if (!first && f >= fbm && f <= fb) return (f - fbm) / (fb - fbm);
  if (!last && f >= fb && f <= fbp) return (fbp - f) / (fbp - fb);
  return f == fb ? 1.0 : 0.0;
}

// grid (parts, D, BOTH ? 1 : 2 sides).  Part p of the intervals' list lies in the interval
// j with first[j] <= p < first[j + 1]; interval j runs from node j up to node j + 1
// (exclusive; the last: node B - 1 alone).  part [D][parts][2][NACC]: the sums for node j
// (0) and node j + 1 (1).
template <int NC>
__global__ void __launch_bounds__(RB_THREADS)
    rb_parts_kernel(int M, int64_t N, const double *__restrict__ ff, const double *__restrict__ dff,
                    const double *__restrict__ psd, const double2 *__restrict__ data, const double2 *__restrict__ h0,
                    const double *__restrict__ t0, int B, const int64_t *__restrict__ node,
                    const int64_t *__restrict__ first, double *__restrict__ part, int *status) {
  using A = RbAcc<NC>;
  constexpr int NACC = A::NACC, NT = RB_THREADS, LD = NT + 1;
  constexpr int SETS = A::BOTH ? 2 : 1, CHUNK = 16;  // columns added per round of the reduction
  __shared__ double col[CHUNK * LD];
  const int d = blockIdx.y, tid = threadIdx.x;
  const bool right = !A::BOTH && blockIdx.z == 1;  // one set: which node of the interval
  int lo = 0, hi = B - 1;                          // largest j with first[j] <= part
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first[mid] <= (int64_t)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const int j = lo;
  auto fnode = [&](int b) { return b >= 0 && b < B ? ff[node[b]] : 0.0; };
  const double fm = fnode(j - 1), f0 = fnode(j), f1 = fnode(j + 1), f2 = fnode(j + 2);
  const double td = t0 ? t0[d] : 0.0;
  const int64_t end = j + 1 < B ? node[j + 1] : node[j] + 1;
  const int64_t n0 = node[j] + ((int64_t)blockIdx.x - first[j]) * RB_PART;
  const int64_t n1 = n0 + RB_PART < end ? n0 + RB_PART : end;
  double cur[NACC], nxt[A::BOTH ? NACC : 1];
#pragma unroll
  for (int q = 0; q < NACC; ++q) cur[q] = 0.0;
  if constexpr (A::BOTH) {
#pragma unroll
    for (int q = 0; q < NACC; ++q) nxt[q] = 0.0;
  }
  for (int64_t n = n0 + tid; n < n1; n += NT) {
    const double f = ff[n];
    // the weight for node j (wl) and for node j + 1 (wr); with one set, for the block's node
    double wl = 0.0, wr = 0.0;
    if (A::BOTH || !right) wl = rb_hat(f, fm, f0, f1, j == 0, j == B - 1);
    if ((A::BOTH || right) && j + 1 < B) wr = rb_hat(f, f0, f1, f2, false, j + 1 == B - 1);
    if constexpr (!A::BOTH) wl = right ? wr : wl;
    if (wl == 0.0 && (!A::BOTH || wr == 0.0)) continue;
    const double S = psd[(int64_t)d * N + n];
    const double base = 4.0 * dff[n] / S;
    wl *= base;
    wr *= base;
    if (!(S > 0.0) || !isfinite(wl) || !isfinite(wr)) {
      atomicCAS(status, 0, DEV_E_NONFINITE);
      continue;
    }
    const double2 dt = cmulc(data[(int64_t)d * N + n], shift64(f, td));
    double2 hv[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) hv[m] = (m < M) ? h0[(int64_t)m * N + n] : make_double2(0.0, 0.0);
    auto add = [&](int q, double v) {
      cur[q] += wl * v;
      if constexpr (A::BOTH) nxt[q] += wr * v;
    };
#pragma unroll
    for (int m = 0; m < NC; ++m) {
      const double2 v = cmulc(dt, hv[m]);  // d (h0 e^{-2 pi i f t})^*
      add(2 * m, v.x);
      add(2 * m + 1, v.y);
      add(2 * NC + m, hv[m].x * hv[m].x + hv[m].y * hv[m].y);
    }
    int p = 3 * NC;
#pragma unroll
    for (int m = 0; m < NC; ++m)
#pragma unroll
      for (int mp = m + 1; mp < NC; ++mp, p += 2) {
        const double2 v = cmulc(hv[m], hv[mp]);  // h0_m h0_m'^*
        add(p, v.x);
        add(p + 1, v.y);
      }
  }
  double *out = part + ((int64_t)d * gridDim.x + blockIdx.x) * 2 * NACC + (right ? NACC : 0);
#pragma unroll
  for (int c0 = 0; c0 < SETS * NACC; c0 += CHUNK) {
    if (c0 > 0) __syncthreads();
#pragma unroll
    for (int c = 0; c < CHUNK; ++c) {
      const int q = c0 + c;
      if (q < NACC) col[c * LD + tid] = cur[q < NACC ? q : 0];
      else if constexpr (A::BOTH) {
        if (q < 2 * NACC) col[c * LD + tid] = nxt[q < 2 * NACC ? q - NACC : 0];
      }
    }
    __syncthreads();
    // NT / CHUNK neighbouring lanes per column, each a run of CHUNK threads
    constexpr int LPC = NT / CHUNK;
    const int c = tid / LPC, r = tid % LPC;
    double v0 = 0.0, v1 = 0.0;
    for (int k = r; k < NT; k += 2 * LPC) {
      v0 += col[c * LD + k];
      v1 += col[c * LD + k + LPC];
    }
    double v = v0 + v1;
#pragma unroll
    for (int o = LPC / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (r == 0 && c0 + c < SETS * NACC) out[c0 + c] = v;
  }
}

// grid (B, D): node j's sums are the left sets of interval j's parts and the right sets of
// interval j - 1's, in order.
template <int NC>
__global__ void __launch_bounds__(RB_FIN_THREADS)
    rb_finish_kernel(int M, int64_t N, const double *__restrict__ ff, const double2 *__restrict__ h0,
                     const double *__restrict__ t0, int B, int64_t n_parts, const int64_t *__restrict__ node,
                     const int64_t *__restrict__ first, const double *__restrict__ part, double2 *__restrict__ w_dh,
                     double2 *__restrict__ w_hh, int *status) {
  constexpr int NACC = RbAcc<NC>::NACC, NT = RB_FIN_THREADS;
  __shared__ double tot[NACC];
  const int j = blockIdx.x, d = blockIdx.y, tid = threadIdx.x;
  const double *pd = part + (int64_t)d * n_parts * 2 * NACC;
  for (int q = tid; q < NACC; q += NT) {
    double v = 0.0;
    if (j > 0)
      for (int64_t p = first[j - 1]; p < first[j]; ++p) v += pd[(2 * p + 1) * NACC + q];
    for (int64_t p = first[j]; p < first[j + 1]; ++p) v += pd[2 * p * NACC + q];
    tot[q] = v;
  }
  __syncthreads();
  const int64_t nb = node[j];
  if (tid < M) {  // W^{<d|h>}: over the conjugate of h0(f_b) e^{-2 pi i f_b t}
    const double2 h = cmul(h0[(int64_t)tid * N + nb], shift64(ff[nb], t0 ? t0[d] : 0.0));
    if (h.x == 0.0 && h.y == 0.0) atomicCAS(status, 0, DEV_E_SHAPE);
    w_dh[((int64_t)d * M + tid) * B + j] = cdiv(make_double2(tot[2 * tid], tot[2 * tid + 1]), make_double2(h.x, -h.y));
  }
  for (int q = tid; q < NC * NC; q += NT) {  // W^{<h|h>} of m <= m' and its mirror
    const int m = q / NC, mp = q % NC;
    if (mp < m || mp >= M) continue;
    const int p = 3 * NC + 2 * (m * (2 * NC - m - 1) / 2 + mp - m - 1);
    const double2 num = mp == m ? make_double2(tot[2 * NC + m], 0.0) : make_double2(tot[p], tot[p + 1]);
    const double2 w = cdiv(num, cmulc(h0[(int64_t)m * N + nb], h0[(int64_t)mp * N + nb]));
    w_hh[(((int64_t)d * M + m) * M + mp) * B + j] = w;
    if (mp != m) w_hh[(((int64_t)d * M + mp) * M + m) * B + j] = make_double2(w.x, -w.y);
  }
}

std::vector<int64_t> rb_parts(int B, const int64_t *node) {
  std::vector<int64_t> first(B + 1, 0);
  for (int j = 0; j < B; ++j)
    first[j + 1] = first[j] + (j + 1 < B ? (node[j + 1] - node[j] + RB_PART - 1) / RB_PART : 1);
  return first;
}
size_t rb_part_doubles(int M) { return 2 * (M <= MAXM ? RbAcc<MAXM>::NACC : RbAcc<2 * MAXM>::NACC); }

template <int NC>
static void launch_rb(int D, int M, int64_t N, const double *ff, const double *dff, const double *psd,
                      const double2 *data, const double2 *h0, const double *t0, int B, int64_t n_parts,
                      const int64_t *node, const int64_t *first, double *part, double2 *w_dh, double2 *w_hh,
                      int *status, cudaStream_t st) {
  rb_parts_kernel<NC><<<dim3((unsigned)n_parts, D, RbAcc<NC>::BOTH ? 1 : 2), RB_THREADS, 0, st>>>(
      M, N, ff, dff, psd, data, h0, t0, B, node, first, part, status);
  rb_finish_kernel<NC><<<dim3(B, D), RB_FIN_THREADS, 0, st>>>(M, N, ff, h0, t0, B, n_parts, node, first, part, w_dh,
                                                             w_hh, status);
}

void launch_rb_weights(int D, int M, int64_t N, const double *ff, const double *dff, const double *psd,
                       const double2 *data, const double2 *h0, const double *t0, int B, int64_t n_parts,
                       const int64_t *node, const int64_t *first, double *part, double2 *w_dh, double2 *w_hh,
                       int *status, cudaStream_t st) {
  if (M <= MAXM)
    launch_rb<MAXM>(D, M, N, ff, dff, psd, data, h0, t0, B, n_parts, node, first, part, w_dh, w_hh, status, st);
  else
    launch_rb<2 * MAXM>(D, M, N, ff, dff, psd, data, h0, t0, B, n_parts, node, first, part, w_dh, w_hh, status, st);
}

}  // namespace dotpe
