// K6: cross-tile reduction (Eq. Z_sum with w_o = 1; Eqs. posterior_element,
// int_ess, ext_ess).  Each fused-kernel tile left log-sum-exp partials (max, sum)
// in FP32; they are combined with FP64 accumulation:
//   ln S1 = ln sum_ieo p_ieo,  ln S2 = ln sum_ieo p_ieo^2,  p_ieo = w_i w_e Lbar_ieo
//   ln Z  = ln S1 - ln(N_i N_e N_phi)
//   N_eff = S1^2 / S2, N_eff,int = S1^2 / sum_i P_i^2, N_eff,ext = S1^2 / sum_e P_e^2
// Tiles' totals and merges: two passes per log-sum-exp, the maximum (FP32, exact), then the sum
// of s * exp(m - max) with the exponential and the accumulation in FP64, which adds only FP64
// rounding to the FP32 partials.  Row and column marginals: FP32 exponentials (about 2^-22
// relative), FP64 products and sums.
// A slice processed as several bank blocks merges each block's (max, sum) pairs,
// its column marginals and its best ln L^ML into FP64 accumulators in block
// order; the final kernel turns them into the evidence.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace dotpe {

namespace {
constexpr int RB = 256;  // threads per block
constexpr int NB = 128;  // blocks of the parallel passes
constexpr int NQ = 3;    // log-sum-exp inputs of a bank block: tile m1, tile m2, 2 ln P_i
}

// ln P over partials [nparts][n] (row or column marginal).  A block takes 32
// consecutive entries (coalesced) and splits the parts over its 8 thread rows;
// each thread keeps an online (max, FP64 sum) and the rows merge in shared memory.  With
// acc != nullptr the value is merged into the FP64 accumulator acc[k] = (m, s) (s = 0: empty) instead of written to out.
constexpr int LX = 32, LY = 8;

__device__ __forceinline__ void lse_add(double &m, double &s, double x, double w) {
  if (!(w > 0.0)) return;
  if (!(s > 0.0)) { m = x; s = w; return; }
  if (x > m) { s = s * exp(m - x) + w; m = x; }
  else s += w * exp(x - m);
}
// A thread takes LG parts at a time: all LG loads are in flight together and the group has one
// maximum, so that the sum is scaled at most once per group.  The exponentials are FP32 (the
// partials carry FP32 precision), the products and their sum FP64: two conversions and a fused
// multiply-add per part (figures at launch_reduce_block).
constexpr int LG = 8;

__global__ void __launch_bounds__(LX * LY) reduce_lines_kernel(int64_t n, int nparts, const float2 *__restrict__ part,
                                                               double *__restrict__ out, double2 *__restrict__ acc,
                                                               int first) {
  __shared__ double sm[LY][LX], ss[LY][LX];
  const int64_t k = blockIdx.x * (int64_t)LX + threadIdx.x;
  float mf = 0.f;
  double s = 0.0;
  if (k < n)
    for (int p = threadIdx.y * LG; p < nparts; p += LY * LG) {
      const float2 *src = part + (int64_t)p * n + k;
      float2 v[LG];
      float gm = -INFINITY;
#pragma unroll
      for (int j = 0; j < LG; ++j) v[j] = (p + j < nparts) ? src[j * n] : make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 0; j < LG; ++j) {
        if (!(v[j].y > 0.f)) v[j] = make_float2(-INFINITY, 0.f);  // empty
        gm = fmaxf(gm, v[j].x);
      }
      if (gm == -INFINITY) continue;
      if (!(s > 0.0)) mf = gm;
      else if (gm > mf) { s *= (double)__expf(mf - gm); mf = gm; }
      // (finite, so that a value that overflowed leaves +inf)
      const float c = fminf(mf, 3.402823466e38f);
#pragma unroll
      for (int j = 0; j < LG; ++j) s = fma((double)v[j].y, (double)__expf(v[j].x - c), s);
    }
  double m = mf;
  sm[threadIdx.y][threadIdx.x] = m;
  ss[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y != 0 || k >= n) return;
  for (int y = 1; y < LY; ++y) lse_add(m, s, sm[y][threadIdx.x], ss[y][threadIdx.x]);
  if (!acc) {
    out[k] = (s > 0.0) ? m + log(s) : -INFINITY;
    return;
  }
  double2 a = first ? make_double2(0.0, 0.0) : acc[k];
  lse_add(a.x, a.y, m, s);
  acc[k] = a;
}

__device__ __forceinline__ float block_max(float v, float *sh) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = (threadIdx.x < blockDim.x / 32) ? sh[threadIdx.x] : -INFINITY;
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (threadIdx.x == 0) sh[0] = v;
  }
  __syncthreads();
  v = sh[0];
  __syncthreads();
  return v;
}

__device__ __forceinline__ double block_sum(double v, double *sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = (threadIdx.x < blockDim.x / 32) ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) sh[0] = v;
  }
  __syncthreads();
  v = sh[0];
  __syncthreads();
  return v;
}

// Pass 1 over one bank block: per-block maxima of the log-sum-exp inputs, the
// argmax and the marginalised count.
__global__ void __launch_bounds__(RB) reduce_pass1_kernel(ReduceArgs a, float *__restrict__ bmax,
                                                           float *__restrict__ bml, long long *__restrict__ barg,
                                                           long long *__restrict__ bnp) {
  __shared__ float shf[32];
  __shared__ double shd[32];
  __shared__ float sv[RB];
  __shared__ long long sa[RB];
  const int64_t n_tiles = (int64_t)a.n_itile * a.n_etile;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t k0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  float m1 = -INFINITY, m2 = -INFINITY, mr = -INFINITY, best = -1.f;
  long long arg = 0x7fffffffffffffffLL, np = 0;
  for (int64_t k = k0; k < n_tiles; k += stride) {
    float4 v = a.tile_part[k];
    if (v.y > 0.f) m1 = fmaxf(m1, v.x);
    if (v.w > 0.f) m2 = fmaxf(m2, v.z);
    float ml = a.tile_ml[k];
    long long g = a.tile_arg[k];
    if (ml > best || (ml == best && g < arg)) { best = ml; arg = g; }
    np += a.tile_npass[k];
  }
  const double *lpi = a.ln_p_int + a.row_offset;
  for (int64_t k = k0; k < a.n_int; k += stride) mr = fmaxf(mr, (float)(2.0 * lpi[k]));
  float r[NQ] = {m1, m2, mr};
  for (int q = 0; q < NQ; ++q) {
    float v = block_max(r[q], shf);
    if (threadIdx.x == 0) bmax[q * gridDim.x + blockIdx.x] = v;
  }
  sv[threadIdx.x] = best;
  sa[threadIdx.x] = arg;
  __syncthreads();
  for (int w = RB / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      if (sv[threadIdx.x + w] > sv[threadIdx.x] ||
          (sv[threadIdx.x + w] == sv[threadIdx.x] && sa[threadIdx.x + w] < sa[threadIdx.x])) {
        sv[threadIdx.x] = sv[threadIdx.x + w];
        sa[threadIdx.x] = sa[threadIdx.x + w];
      }
    }
    __syncthreads();
  }
  double npd = block_sum((double)np, shd);  // counts < 2^53
  if (threadIdx.x == 0) {
    bml[blockIdx.x] = sv[0];
    barg[blockIdx.x] = sa[0];
    bnp[blockIdx.x] = (long long)npd;
  }
}

// Pass 2: per-block FP64 sums of s * exp(m - M) against the bank block's maxima.
__global__ void __launch_bounds__(RB) reduce_pass2_kernel(ReduceArgs a, const float *__restrict__ bmax,
                                                           double *__restrict__ bsum) {
  __shared__ double shd[32];
  __shared__ float M[NQ];
  if (threadIdx.x < NQ) {
    float m = -INFINITY;
    for (int b = 0; b < (int)gridDim.x; ++b) m = fmaxf(m, bmax[threadIdx.x * gridDim.x + b]);
    M[threadIdx.x] = m;
  }
  __syncthreads();
  const int64_t n_tiles = (int64_t)a.n_itile * a.n_etile;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t k0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double s[NQ] = {0.0, 0.0, 0.0};
  for (int64_t k = k0; k < n_tiles; k += stride) {
    float4 v = a.tile_part[k];
    if (v.y > 0.f) s[0] += (double)v.y * exp((double)v.x - (double)M[0]);
    if (v.w > 0.f) s[1] += (double)v.w * exp((double)v.z - (double)M[1]);
  }
  const double *lpi = a.ln_p_int + a.row_offset;
  for (int64_t k = k0; k < a.n_int; k += stride) {
    double v = lpi[k];
    if (v != -INFINITY) s[2] += exp(2.0 * v - (double)M[2]);
  }
  for (int q = 0; q < NQ; ++q) {
    double v = block_sum(s[q], shd);
    if (threadIdx.x == 0) bsum[q * gridDim.x + blockIdx.x] = v;
  }
}

__device__ __forceinline__ void acc_merge(double &am, double &as, double bm, double bs) {
  if (!(bs > 0.0)) return;
  if (!(as > 0.0)) { am = bm; as = bs; return; }
  if (bm > am) { as = as * exp(am - bm) + bs; am = bm; }
  else as += bs * exp(bm - am);
}

// Merges one bank block into the event's FP64 accumulators (fixed order: deterministic).
__global__ void reduce_block_merge_kernel(ReduceArgs a, int nb, const float *__restrict__ bmax,
                                          const double *__restrict__ bsum, const float *__restrict__ bml,
                                          const long long *__restrict__ barg, const long long *__restrict__ bnp) {
  // one warp; lane l takes the per-block entries l, l + 32, ...; fixed shuffle order
  const int lane = threadIdx.x;
  double m[NQ], sm[NQ];
  for (int q = 0; q < NQ; ++q) {
    float mq = -INFINITY;
    double sq = 0.0;
    for (int b = lane; b < nb; b += 32) {
      mq = fmaxf(mq, bmax[q * nb + b]);
      sq += bsum[q * nb + b];
    }
    for (int o = 16; o > 0; o >>= 1) {
      mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o));
      sq += __shfl_xor_sync(0xffffffffu, sq, o);
    }
    m[q] = mq;
    sm[q] = sq;
  }
  // arguments are packed ((i * n_ext + e) * n_phi + o) with i relative to the block
  const long long shift = (long long)a.row_offset * a.n_ext * a.n_phi;
  float best = -1.f;
  long long arg = 0x7fffffffffffffffLL, np = 0;
  for (int b = lane; b < nb; b += 32) {
    const long long g = barg[b] + shift;
    if (bml[b] > best || (bml[b] == best && g < arg)) { best = bml[b]; arg = g; }
    np += bnp[b];
  }
  for (int o = 16; o > 0; o >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
    const long long oa = __shfl_xor_sync(0xffffffffu, arg, o);
    if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; }
    np += __shfl_xor_sync(0xffffffffu, np, o);
  }
  // The sums are the same in every lane: lane q < NQ merges pair q, lane NQ the maximum and the count
  double *dst = &a.acc->s1_m;  // the (max, sum) pairs lie one after the other
#pragma unroll
  for (int q = 1; q < NQ; ++q)
    if (lane == q) { m[0] = m[q]; sm[0] = sm[q]; dst += 2 * q; }
  if (lane < NQ) {
    double am = 0.0, as = 0.0;
    if (!a.first) { am = dst[0]; as = dst[1]; }
    if (m[0] != -INFINITY) acc_merge(am, as, m[0], sm[0]);
    dst[0] = am;
    dst[1] = as;
  } else if (lane == NQ) {
    float cb = a.first ? -1.f : a.acc->best;
    long long ca = a.first ? 0x7fffffffffffffffLL : a.acc->arg;
    if (best > cb || (best == cb && arg < ca)) { cb = best; ca = arg; }
    a.acc->best = cb;
    a.acc->arg = ca;
    a.acc->n_marg = (a.first ? 0 : a.acc->n_marg) + np;
  }
}

// After the last block: column marginals, Sum_e P_e^2 (two passes) and the evidence.
// The marginals' FP64 logarithms and exponentials are bound by the FP64 pipe, so
// they are spread over up to NB blocks, each leaving the maximum of its 2 ln P_e and
// the sum against it; the last kernel merges those in a fixed order (figures at
// launch_reduce_final).
__global__ void __launch_bounds__(RB) reduce_ext_kernel(ReduceArgs a, float *__restrict__ bmax,
                                                        double *__restrict__ bsum) {
  __shared__ float shf[32];
  __shared__ double shd[32];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t k0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  float mc = -INFINITY;
  for (int64_t k = k0; k < a.n_ext; k += stride) {
    const double2 v = a.acc_col[k];
    const double l = (v.y > 0.0) ? v.x + log(v.y) : -INFINITY;
    a.ln_p_ext[k] = l;
    mc = fmaxf(mc, (float)(2.0 * l));
  }
  mc = block_max(mc, shf);
  double sc = 0.0;
  if (mc != -INFINITY)
    for (int64_t k = k0; k < a.n_ext; k += stride) {
      const double l = a.ln_p_ext[k];
      if (l != -INFINITY) sc += exp(2.0 * l - (double)mc);
    }
  sc = block_sum(sc, shd);
  if (threadIdx.x == 0) { bmax[blockIdx.x] = mc; bsum[blockIdx.x] = sc; }
}

__global__ void reduce_final_kernel(ReduceArgs a, int nb, const float *__restrict__ bmax,
                                    const double *__restrict__ bsum) {
  // One warp.  FP64 logarithms and exponentials are chains of ~40 dependent operations:
  // those of a step run in one lane each, side by side.
  const EvAcc c = *a.acc;
  const int lane = threadIdx.x;
  float mc = -INFINITY;
  for (int b = lane; b < nb; b += 32) mc = fmaxf(mc, bmax[b]);
  for (int o = 16; o > 0; o >>= 1) mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, o));
  double sc = 0.0;
  for (int b = lane; b < nb; b += 32)
    if (bsum[b] > 0.0) sc += bsum[b] * exp((double)bmax[b] - (double)mc);
  for (int o = 16; o > 0; o >>= 1) sc += __shfl_xor_sync(0xffffffffu, sc, o);
  double x = 1.0;  // the argument of lane's logarithm
  if (lane == 0) x = c.s1_s;
  if (lane == 1) x = c.s2_s;
  if (lane == 2) x = c.pi_s;
  if (lane == 3) x = sc;
  if (lane == 4) x = (double)a.n_int_total;
  if (lane == 5) x = (double)a.n_ext;
  if (lane == 6) x = (double)a.n_phi;
  const double lx = log(x);
  auto lnv = [&](int l, double m, double s) {
    const double v = __shfl_sync(0xffffffffu, lx, l);
    return (s > 0.0) ? m + v : -INFINITY;
  };
  const double l1 = lnv(0, c.s1_m, c.s1_s), l2 = lnv(1, c.s2_m, c.s2_s), lpi = lnv(2, c.pi_m, c.pi_s);
  const double lpe = lnv(3, mc, sc);
  const double ln_i = lnv(4, 0.0, 1.0), ln_e = lnv(5, 0.0, 1.0), ln_o = lnv(6, 0.0, 1.0);
  const double ex = exp(2.0 * l1 - (lane == 0 ? l2 : lane == 1 ? lpi : lpe));
  const double n_eff_int = __shfl_sync(0xffffffffu, ex, 1), n_eff_ext = __shfl_sync(0xffffffffu, ex, 2);
  if (lane != 0) return;
  ReduceOut o;
  o.ln_s1 = l1;
  o.ln_s2 = l2;
  o.ln_z = l1 - ln_i - ln_e - ln_o;
  o.n_eff = (l1 == -INFINITY) ? 0.0 : ex;
  o.n_eff_int = (l1 == -INFINITY) ? 0.0 : n_eff_int;
  o.n_eff_ext = (l1 == -INFINITY) ? 0.0 : n_eff_ext;
  o.max_ml = c.best;
  o.arg = c.arg;
  o.n_marg = c.n_marg;
  o.threshold = (a.cut_delta > 0.f) ? (double)(*a.ml_running) - (double)a.cut_delta : -INFINITY;
  o.status = *a.status;
  o.n_refined = a.n_refined ? *a.n_refined : -1;
  o.n_cand = a.n_cand ? (long long)a.n_cand[0] : -1;
  o.n_eval = a.n_cand ? (long long)a.n_cand[1] : -1;
  *a.out = o;
}

size_t reduce_scratch_bytes() {
  return (size_t)NB * (NQ * sizeof(float) + NQ * sizeof(double) + sizeof(float) + 2 * sizeof(long long)) + 256;
}

namespace {
struct BlockScratch {  // per-block results of the parallel passes, in ReduceArgs::scratch
  float *bmax;
  double *bsum;
  float *bml;
  long long *barg, *bnp;
  explicit BlockScratch(void *scratch) {
    uint8_t *w = (uint8_t *)scratch;
    bmax = (float *)w;
    bsum = (double *)(w + NB * NQ * sizeof(float));
    bml = (float *)(bsum + NB * NQ);
    barg = (long long *)(((uintptr_t)(bml + NB) + 7) & ~(uintptr_t)7);
    bnp = barg + NB;
  }
};
}  // namespace

// The two line reductions stream 84 MB of partials for 65,536 rows x 4,096 samples: 44 us
// (67 us a part at a time); 148 us (238 us) over four blocks of 65,536 rows x 2,048 samples.
// Summing a group in two floats instead takes 34 and 106 us, with 46 bits of the sum where
// FP64 has 53.
void launch_reduce_block(const ReduceArgs &a, cudaStream_t st) {
  const dim3 lb(LX, LY);
  reduce_lines_kernel<<<(unsigned)((a.n_int + LX - 1) / LX), lb, 0, st>>>(a.n_int, a.n_etile, a.row_part,
                                                                         a.ln_p_int + a.row_offset, nullptr, 0);
  reduce_lines_kernel<<<(unsigned)((a.n_ext + LX - 1) / LX), lb, 0, st>>>(a.n_ext, a.n_itile, a.col_part, nullptr,
                                                                         a.acc_col, a.first);
  const BlockScratch s(a.scratch);
  reduce_pass1_kernel<<<NB, RB, 0, st>>>(a, s.bmax, s.bml, s.barg, s.bnp);
  reduce_pass2_kernel<<<NB, RB, 0, st>>>(a, s.bmax, s.bsum);
  reduce_block_merge_kernel<<<1, 32, 0, st>>>(a, NB, s.bmax, s.bsum, s.bml, s.barg, s.bnp);
}

// 4,096 samples: 5.8 us for the marginals and 6.9 us for the record (24.8 us in one block).
void launch_reduce_final(const ReduceArgs &a, cudaStream_t st) {
  const int nb = (int)std::min<int64_t>(NB, (a.n_ext + RB - 1) / RB);
  const BlockScratch s(a.scratch);
  reduce_ext_kernel<<<nb, RB, 0, st>>>(a, s.bmax, s.bsum);
  reduce_final_kernel<<<1, 32, 0, st>>>(a, nb, s.bmax, s.bsum);
}

// ---------------------------------------------------------------------------
// Refinement selection (after a screening pass).  Tile t of event k is refined
// when its screened best ln L^ML reaches max_k - window - 2 margin(max_k): the
// exact value of any pair differs from its screened one by at most one margin,
// and so does the exact maximum.  Two kernels keep the list in event order and
// banded tile order within an event: per-block counts, then each block writes
// its items at the prefix of the earlier counts.
// ---------------------------------------------------------------------------
namespace {
constexpr int SB = 1024;  // tiles per selection block
}

__device__ __forceinline__ bool select_tile(const SelectBatch &a, int w, int &k, int &t) {
  if (w >= a.begin[a.n]) return false;
  int lo = 0, hi = a.n - 1;  // largest k with begin[k] <= w
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (a.begin[mid] <= w) lo = mid;
    else hi = mid - 1;
  }
  k = lo;
  const SelectEvent &v = a.ev[k];
  int it, et;
  super_tile(w - a.begin[k], v.n_itile, v.n_etile, v.band, it, et);
  t = it * v.n_etile + et;
  const float mx = *v.ml_screen;
  const float thr = mx - v.window - 2.f * screen_margin(mx, v.margin_k, *v.sqrt_dd);
  return v.tile_ml[t] >= thr;
}

__global__ void __launch_bounds__(SB) select_count_kernel(SelectBatch a) {
  int k = -1, t;
  const bool f = select_tile(a, blockIdx.x * SB + threadIdx.x, k, t);
  const int c = __syncthreads_count(f);
  if (threadIdx.x == 0) a.counts[blockIdx.x] = c;
  // per-event counts: one atomic per (warp, event)
  const unsigned grp = __match_any_sync(0xffffffffu, f ? k : -1);
  const int lane = threadIdx.x & 31;
  if (f && lane == __ffs(grp) - 1) atomicAdd(a.ev[k].n_refined, __popc(grp));
}

__global__ void __launch_bounds__(SB) select_write_kernel(SelectBatch a) {
  __shared__ int wsum[SB / 32];
  __shared__ int base_s;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // prefix of the earlier blocks' counts (and, in block 0, the total)
  {
    const int upto = (blockIdx.x == 0) ? (int)gridDim.x : (int)blockIdx.x;
    int v = 0;
    for (int q = tid; q < upto; q += SB) v += a.counts[q];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) wsum[wid] = v;
    __syncthreads();
    if (tid == 0) {
      int s = 0;
      for (int q = 0; q < SB / 32; ++q) s += wsum[q];
      base_s = (blockIdx.x == 0) ? 0 : s;
      if (blockIdx.x == 0) *a.n_list = s;
    }
    __syncthreads();
  }
  int k = 0, t = 0;
  const bool f = select_tile(a, blockIdx.x * SB + tid, k, t);
  const unsigned bal = __ballot_sync(0xffffffffu, f);
  if (lane == 0) wsum[wid] = __popc(bal);
  __syncthreads();
  if (tid == 0) {
    int s = 0;
    for (int q = 0; q < SB / 32; ++q) {
      const int c = wsum[q];
      wsum[q] = s;
      s += c;
    }
  }
  __syncthreads();
  if (f) a.list[base_s + wsum[wid] + __popc(bal & ((1u << lane) - 1u))] = make_int2(k, t);
}

// Per event: the frozen refinement maximum; the refined-tile count starts at 0.
__global__ void select_events_kernel(SelectBatch a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.n) return;
  const SelectEvent &v = a.ev[k];
  const float mx = *v.ml_screen;
  *v.ml_refine = fmaxf(mx - screen_margin(mx, v.margin_k, *v.sqrt_dd), 0.f);
  *v.n_refined = 0;
  if (a.sep) a.sep[k] = (mx > v.sep_ml) ? 1 : 0;
}

int select_count_blocks(int n_tiles) { return (n_tiles + SB - 1) / SB; }

void launch_select(const SelectBatch &a, cudaStream_t st) {
  const int nb = select_count_blocks(a.begin[a.n]);
  if (nb < 1) return;
  select_events_kernel<<<(a.n + 63) / 64, 64, 0, st>>>(a);
  select_count_kernel<<<nb, SB, 0, st>>>(a);
  select_write_kernel<<<nb, SB, 0, st>>>(a);
}

}  // namespace dotpe
