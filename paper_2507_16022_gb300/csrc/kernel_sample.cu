// Posterior samples of a finished event: resampling with the weights
// p_ieo = w_i w_e w_o Lbar_ieo (Eq. posterior_element; Sec. III resampling;
// w_o = 1) and a distance per sample drawn from the summand of the distance
// marginal (App. C: phase and distance drawn per (intrinsic, extrinsic) pair).
//
// Per sample, four uniforms in [0, 1):
//   u1 -> i  from the row marginals ln sum_{e,o} p_ieo (the event's FP64 row weights),
//   u2 -> e  from row i of the stored ln Lbar_ie plus ln w_e,
//   u3 -> o  from the pair's phases that pass the event's ML cut, weights Lbar_ieo
//            (the pair recomputed in FP64 from the event's inputs: per-mode
//            components and mode overlaps, Eqs. dh_ieo, hh_ieo, per (mode,
//            polarisation) component with real antenna patterns F_edp for a
//            polarisation-resolved bank; Lbar from the same device distance
//            marginal as the fused kernels),
//   u4 -> d_L / d_L^0 = 1/u from the density of u on [u_min, inf),
//            proportional to u^-4 exp(dh u - hh u^2 / 2) (pi(d_L) ~ d_L^2).
// Each draw takes the smallest index whose cumulative weight exceeds u times
// the total.  The distance is inverted on a 1,024-node grid of v = sqrt(hh) u
// over [s, max(s, x, v*) + 12] (x = dh/sqrt(hh), s = sqrt(hh) u_min), the
// log-density linear within each interval (integrated and inverted in closed
// form).
//
// All of it is FP64, and an SM has two FP64 lanes per cycle: the draws are bound
// by the number of FP64 operations on the busiest SM.  So one block of two warps per
// sample (512 draws fill every SM; eight samples per block left half of the SMs
// without one), the quadrature weights formed once per call, each row overlap of the
// Hermitian matrix once, e^{ikphi} from one sincospi per phase, one logarithm and
// one exponential per distance node, and no exponentials for pairs below the cut.
// 512 draws of a 16,384 x 2,048 event: 0.37 ms for the kernel and the row weights (1.94 +
// 0.20 ms with one warp per sample and the row weights from a single block).
#include "common.cuh"
#include "dist_marg.cuh"
#include "kernels.h"

namespace dotpe {

namespace {
constexpr int ST = 64;        // threads per sample
constexpr int SNODE = 1024;   // distance grid nodes
constexpr int SPT = SNODE / ST;
constexpr int RBLK = 256;     // rows per block of the row weights

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double wmax(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// inclusive prefix sum over the warp's lanes
__device__ __forceinline__ double wscan(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}
// doubles as integers of the same order (for atomicMax), and back
__device__ __forceinline__ unsigned long long ord64(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double unord64(unsigned long long u) {
  return __longlong_as_double((long long)((u >> 63) ? (u & 0x7fffffffffffffffull) : ~u));
}

// The smallest k in [0, n) with f(k) > target for a non-decreasing f, by a whole
// warp (32 probes per step); n - 1 if there is none.
template <typename F>
__device__ __forceinline__ int64_t warp_search(int64_t n, double target, int lane, F f) {
  int64_t lo = 0, len = n;
  while (true) {
    const int64_t k = lo + ((lane + 1) * len + 31) / 32 - 1;
    const unsigned b = __ballot_sync(0xffffffffu, f(k) > target);
    if (!b) return n - 1;
    const int first = __ffs(b) - 1;
    const int64_t hi = __shfl_sync(0xffffffffu, k, first);
    const int64_t below = __shfl_sync(0xffffffffu, k, first > 0 ? first - 1 : 0);
    if (first > 0) lo = below + 1;
    len = hi - lo + 1;
    if (len <= 1) return hi;
  }
}

// The block draws an index from weights exp(x_k - mx), k in [0, n) (get(k) gives x_k,
// -inf for a weight of zero; mx their maximum, finite): the smallest k whose cumulative
// weight exceeds u * total.  Each warp sums half of the range, the half that holds the
// target is halved again, down to 32 entries.
template <typename Get>
__device__ int block_pick(int n, double u, double mx, double *sh, Get get) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int a = 0, b = n;
  double target = -1.0;
  while (b - a > 32 || target < 0.0) {
    const int mid = a + ((b - a + 1) / 2 + 31) / 32 * 32 < b ? a + ((b - a + 1) / 2 + 31) / 32 * 32 : b;
    const int k0 = w == 0 ? a : mid, k1 = w == 0 ? mid : b;
    double loc = 0.0;
    for (int k = k0 + lane; k < k1; k += 32) {
      const double x = get(k);
      if (x > -INFINITY) loc += exp(x - mx);
    }
    loc = wsum(loc);
    __syncthreads();
    if (lane == 0) sh[w] = loc;
    __syncthreads();
    const double t0 = sh[0], t1 = sh[1];
    if (target < 0.0) target = u * (t0 + t1);
    // (rounding may leave the target at the very top: the last half of positive weight)
    if (target < t0 || !(t1 > 0.0)) {
      b = mid;
    } else {
      target -= t0;
      a = mid;
    }
  }
  // 32 entries, in every warp alike
  const int k = a + lane;
  const double x = k < b ? get(k) : -INFINITY;
  const double wt = x > -INFINITY ? exp(x - mx) : 0.0;
  const double incl = wscan(wt, lane);
  // (a lane of zero weight can differ from its neighbour in the scan's last bit: never taken)
  const unsigned hit = __ballot_sync(0xffffffffu, wt > 0.0 && incl > target);
  const unsigned pos = __ballot_sync(0xffffffffu, wt > 0.0);
  __syncthreads();
  if (hit) return a + __ffs(hit) - 1;
  return pos ? a + 31 - __clz(pos) : -1;
}
}  // namespace

// ---- row weights: cumulative sums of exp(ln_p - max), a block of RBLK rows each ----
__global__ void sample_row_max_kernel(int64_t n, const double *__restrict__ ln_p,
                                      unsigned long long *__restrict__ mx) {
  double m = -INFINITY;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    m = fmax(m, ln_p[k]);
  m = wmax(m);
  if ((threadIdx.x & 31) == 0 && m > -INFINITY) atomicMax(mx, ord64(m));
}

// cdf[k]: sum within the block of rows of k; tot[block]: its total
__global__ void __launch_bounds__(RBLK) sample_row_cdf_kernel(int64_t n, const double *__restrict__ ln_p,
                                                              const unsigned long long *__restrict__ mx,
                                                              double *__restrict__ cdf, double *__restrict__ tot) {
  __shared__ double red[RBLK / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t k = blockIdx.x * (int64_t)RBLK + threadIdx.x;
  const double lp = k < n ? ln_p[k] : -INFINITY;
  const double v = lp > -INFINITY ? exp(lp - unord64(*mx)) : 0.0;
  double incl = wscan(v, lane);
  if (lane == 31) red[w] = incl;
  __syncthreads();
  for (int q = 0; q < w; ++q) incl += red[q];
  if (k < n) cdf[k] = incl;
  if (threadIdx.x == RBLK - 1) tot[blockIdx.x] = incl;
}

// pre[b] = sum of the totals before block b, pre[nb] = the total; one block
__global__ void __launch_bounds__(256) sample_row_prefix_kernel(int nb, const double *__restrict__ tot,
                                                                double *__restrict__ pre) {
  __shared__ double red[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double base = 0.0;
  for (int b0 = 0; b0 < nb; b0 += 256) {
    const int b = b0 + threadIdx.x;
    const double v = b < nb ? tot[b] : 0.0;
    double incl = wscan(v, lane);
    if (lane == 31) red[w] = incl;
    __syncthreads();
    double all = 0.0;
    for (int q = 0; q < 8; ++q) {
      if (q < w) incl += red[q];
      all += red[q];
    }
    if (b < nb) pre[b + 1] = base + incl;
    base += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) pre[0] = 0.0;
}

// Quadrature and data weights in FP64: om = 4 w / S, c = om conj(d) (Eq. inner_product).
__global__ void sample_weights_kernel(int D, int B, const double *__restrict__ w, const double *__restrict__ psd,
                                      const double2 *__restrict__ data, double *__restrict__ om,
                                      double2 *__restrict__ c) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= D * B) return;
  const double o = 4.0 * w[k % B] / psd[k];
  const double2 d = data[k];
  om[k] = o;
  c[k] = make_double2(o * d.x, -o * d.y);
}

// NP = 2: polarisation-resolved bank, components j = (m, p) with master row
// [Re h_m+ | Im h_m+ | Re h_mx | Im h_mx] and response F_edp (real).
template <int NP>
__global__ void __launch_bounds__(ST)
    sample_kernel(const SampleArgs a, int64_t n, const double *__restrict__ uni, const double *__restrict__ cdf,
                  const double *__restrict__ pre, int64_t *__restrict__ i_out, int64_t *__restrict__ e_out,
                  int32_t *__restrict__ o_out, double *__restrict__ d_out) {
  constexpr int MJ = MAXM * NP;
  constexpr int NQ = MJ * (MJ - 1) / 2;        // pairs j > jp
  constexpr int NV = 2 * MAXM + 7;             // Z_k by azimuthal number, C_0, C_1..C_3
  __shared__ double sh[ST / 32];
  __shared__ double red[ST / 32][NV];
  __shared__ double cz[NV];
  __shared__ double sl[MAXPHI];                // ln Lbar per phase, -inf below the cut
  __shared__ double pn[SNODE + SNODE / SPT], en[SNODE + SNODE / SPT];  // log-density and density per node (padded)
  __shared__ long long s_i;
  __shared__ float smx[ST / 32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t s = blockIdx.x;
  const double u1 = uni[4 * s], u2 = uni[4 * s + 1], u3 = uni[4 * s + 2], u4 = uni[4 * s + 3];
  const int M = a.n_modes, D = a.n_det, B = a.n_bins;
  // ---- i: the smallest row whose cumulative weight exceeds u1 * total
  // (the block of rows, then the row; at each level the target is kept below the last
  // entry, so that rounding cannot lead past the last row of positive weight)
  if (w == 0) {
    const int64_t nb = (a.n_int + RBLK - 1) / RBLK;
    const double tot = pre[nb];
    int64_t r = a.n_int - 1;
    if (tot > 0.0) {
      auto below = [](double v) { return __longlong_as_double(__double_as_longlong(v) - 1); };
      const double target = fmin(u1 * tot, below(tot));
      const int64_t bl = warp_search(nb, target, lane, [&](int64_t k) { return pre[k + 1]; });
      const int64_t r0 = bl * RBLK, nr = min((int64_t)RBLK, a.n_int - r0);
      const double p0 = pre[bl], last = p0 + cdf[r0 + nr - 1];
      r = r0 + warp_search(nr, fmin(target, below(last)), lane, [&](int64_t k) { return p0 + cdf[r0 + k]; });
    }
    if (lane == 0) {
      // (the scan's last bit again: not a row of zero weight while there is another)
      int64_t q = r;
      while (q > 0 && a.ln_p_int[q] == -INFINITY) --q;
      if (a.ln_p_int[q] == -INFINITY)
        for (q = r; q + 1 < a.n_int && a.ln_p_int[q] == -INFINITY;) ++q;
      s_i = q;
    }
  }
  __syncthreads();
  const int64_t i = s_i;
  // ---- e: row i of the stored ln Lbar_ie plus ln w_e
  const float *lrow = a.lnl + i * a.n_ext;
  auto lnw = [&](int k) -> double {
    const float v = lrow[k];
    return (v == -INFINITY) ? -INFINITY : (double)v + (a.lw_ext ? a.lw_ext[k] : 0.0);
  };
  double mx = -INFINITY;
  if (!a.lw_ext) {
    float m = -INFINITY;
    for (int k = tid; k < a.n_ext; k += ST) m = fmaxf(m, lrow[k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) smx[w] = m;
    __syncthreads();
    mx = (double)fmaxf(smx[0], smx[1]);
  } else {
    for (int k = tid; k < a.n_ext; k += ST) mx = fmax(mx, lnw(k));
    mx = wmax(mx);
    if (lane == 0) sh[w] = mx;
    __syncthreads();
    mx = fmax(sh[0], sh[1]);
  }
  const int e = (mx > -INFINITY) ? block_pick((int)a.n_ext, u2, mx, sh, lnw) : -1;
  // ---- the pair in FP64, per component j = (m, p): z_j = sum_d R_edj sum_b c_djb T_db h_j(b) and,
  // for j >= jp, H_jjp = sum_d R_edj R*_edjp sum_b W_djjpb h_j h*_jp (R_edj = R_edm, or F_edp).
  // The <h|h> of both orders of a pair is one term of weight (W_jjp + W*_jpj) / 2 (omega for
  // the plain quadrature), so that Re<h|h>(phi) = sum_j H_jj + 2 Re sum_{j > jp} H_jjp e^{i(m_j - m_jp) phi}.
  const int J = M * NP;
  double acc[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = 0.0;
  const int64_t ib = a.i_base + i;
  if (e >= 0)
    for (int d = 0; d < D; ++d) {
      double sr[MJ] = {}, si[MJ] = {}, qd[MJ] = {}, qr[NQ] = {}, qi[NQ] = {};
      const double td = a.t[(int64_t)e * D + d];
      for (int b = tid; b < B; b += ST) {
        double sn, cs;
        sincospi(2.0 * a.f[b] * td, &sn, &cs);
        double hr[MJ], hi[MJ];
#pragma unroll
        for (int j = 0; j < MJ; ++j) {
          const int m = j / NP, p = j % NP;
          const float *row = a.master + ((int64_t)m * a.bank_rows + ib) * a.kpad + 2 * p * B;
          hr[j] = (j < J) ? (double)row[b] : 0.0;
          hi[j] = (j < J) ? (double)row[B + b] : 0.0;
        }
        const int64_t db = (int64_t)d * B + b;
        if (!a.rb_dh) {
          const double om = a.om[db];
          const double2 c = a.cw[db];
          const double ctr = c.x * cs + c.y * sn, cti = c.y * cs - c.x * sn;  // c e^{-2 pi i f t}
          int p = 0;
#pragma unroll
          for (int j = 0; j < MJ; ++j) {
            if (j >= J) break;
            sr[j] += ctr * hr[j] - cti * hi[j];
            si[j] += ctr * hi[j] + cti * hr[j];
            const double wr = om * hr[j], wi = om * hi[j];
            qd[j] += wr * hr[j] + wi * hi[j];
#pragma unroll
            for (int jp = 0; jp < j; ++jp, ++p) {
              qr[p] += wr * hr[jp] + wi * hi[jp];
              qi[p] += wi * hr[jp] - wr * hi[jp];
            }
          }
        } else {
          int p = 0;
#pragma unroll
          for (int j = 0; j < MJ; ++j) {
            if (j >= J) break;
            const double2 wd = a.rb_dh[((int64_t)d * J + j) * B + b];
            const double ctr = wd.x * cs - wd.y * sn, cti = -wd.y * cs - wd.x * sn;  // conj(W) e^{-2 pi i f t}
            sr[j] += ctr * hr[j] - cti * hi[j];
            si[j] += ctr * hi[j] + cti * hr[j];
            const double wjj = a.rb_hh[(((int64_t)d * J + j) * J + j) * B + b].x;
            qd[j] += wjj * (hr[j] * hr[j] + hi[j] * hi[j]);
#pragma unroll
            for (int jp = 0; jp < j; ++jp, ++p) {
              const double2 w1 = a.rb_hh[(((int64_t)d * J + j) * J + jp) * B + b];
              const double2 w2 = a.rb_hh[(((int64_t)d * J + jp) * J + j) * B + b];
              const double wr = 0.5 * (w1.x + w2.x), wi = 0.5 * (w1.y - w2.y);
              const double pr = hr[j] * hr[jp] + hi[j] * hi[jp], pi = hi[j] * hr[jp] - hr[j] * hi[jp];
              qr[p] += wr * pr - wi * pi;
              qi[p] += wr * pi + wi * pr;
            }
          }
        }
      }
      // the detector's share of Z_k and C_delta (both orders of a pair: twice its real part)
      auto resp = [&](int j) -> double2 {
        if (NP == 2) return make_double2(a.F[((int64_t)e * D + d) * 2 + (j % 2)], 0.0);
        return a.R[((int64_t)e * D + d) * M + j];
      };
      int p = 0;
#pragma unroll
      for (int j = 0; j < MJ; ++j) {
        if (j >= J) break;
        const double2 R = resp(j);
#pragma unroll
        for (int k = 0; k < MAXM; ++k)
          if (a.mode_m[j / NP] == k + 1) {
            acc[2 * k] += R.x * sr[j] - R.y * si[j];
            acc[2 * k + 1] += R.x * si[j] + R.y * sr[j];
          }
        acc[2 * MAXM] += (R.x * R.x + R.y * R.y) * qd[j];
#pragma unroll
        for (int jp = 0; jp < j; ++jp, ++p) {
          const double2 Rp = resp(jp);
          const double rr = R.x * Rp.x + R.y * Rp.y, ri = R.y * Rp.x - R.x * Rp.y;  // R R'^*
          const double hre = 2.0 * (rr * qr[p] - ri * qi[p]), him = 2.0 * (rr * qi[p] + ri * qr[p]);
          const int dl = a.mode_m[j / NP] - a.mode_m[jp / NP];
          if (dl == 0) acc[2 * MAXM] += hre;
#pragma unroll
          for (int k = 1; k <= 3; ++k)
            if (dl == k) {
              acc[2 * MAXM + 2 * k - 1] += hre;
              acc[2 * MAXM + 2 * k] += him;
            }
        }
      }
    }
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const double v = wsum(acc[q]);
    if (lane == 0) red[w][q] = v;
  }
  __syncthreads();
  if (tid < NV) cz[tid] = red[0][tid] + red[1][tid];
  __syncthreads();
  // ---- o: phases that pass the cut, weights Lbar_ieo
  const int np = a.n_phi;
  auto dhh = [&](int o, double &dh, double &hh) {
    double s1, c1;
    sincospi(2.0 * (double)o / (double)np, &s1, &c1);
    const double c2 = c1 * c1 - s1 * s1, s2 = 2.0 * c1 * s1;
    const double c3 = c2 * c1 - s2 * s1, s3 = s2 * c1 + c2 * s1;
    const double c4 = c2 * c2 - s2 * s2, s4 = 2.0 * c2 * s2;
    dh = cz[0] * c1 - cz[1] * s1 + cz[2] * c2 - cz[3] * s2 + cz[4] * c3 - cz[5] * s3 + cz[6] * c4 - cz[7] * s4;
    hh = cz[8] + (cz[9] * c1 - cz[10] * s1) + (cz[11] * c2 - cz[12] * s2) + (cz[13] * c3 - cz[14] * s3);
  };
  double lmx = -INFINITY;
  if (e >= 0)
    for (int k = tid; k < np; k += ST) {
      double dh, hh;
      dhh(k, dh, hh);
      const double ml = (dh > 0.0 && hh > 0.0) ? dh * dh / (2.0 * hh) : 0.0;
      double l = -INFINITY;
      if (ml >= a.threshold) {
        const float d1[1] = {(float)dh}, h1[1] = {(float)hh};
        float l1[1];
        dm_lnlbar_n<1>(d1, h1, a.u_min, a.dm_table, l1);
        l = (double)l1[0];
      }
      sl[k] = l;
      lmx = fmax(lmx, l);
    }
  lmx = wmax(lmx);
  __syncthreads();
  if (lane == 0) sh[w] = lmx;
  __syncthreads();
  lmx = fmax(sh[0], sh[1]);
  const int o = (e >= 0 && lmx > -INFINITY) ? block_pick(np, u3, lmx, sh, [&](int k) { return sl[k]; }) : -1;
  // ---- distance
  double dist = 0.0;
  if (o >= 0) {
    double dh, hh;
    dhh(o, dh, hh);
    if (!(hh > 0.0)) {
      dist = cbrt(1.0 - u4) / (double)a.u_min;
    } else {
      const double r = sqrt(hh), x = dh / r, sv = r * (double)a.u_min;
      double vmax = sv;
      if (x > 4.0) vmax = fmax(vmax, 0.5 * (x + sqrt(x * x - 16.0)));
      const double vhi = fmax(fmax(sv, x), vmax) + 12.0;
      const double h = (vhi - sv) / (SNODE - 1);
      auto at = [](int k) { return k + k / SPT; };  // padded: a thread's run of nodes in other banks than its neighbour's
      double pm = -INFINITY;
      for (int k = tid; k < SNODE; k += ST) {
        const double v = sv + k * h;
        const double p = -4.0 * log(v) - 0.5 * (v - x) * (v - x);
        pn[at(k)] = p;
        pm = fmax(pm, p);
      }
      pm = wmax(pm);
      __syncthreads();
      if (lane == 0) sh[w] = pm;
      __syncthreads();
      pm = fmax(sh[0], sh[1]);
      // (beyond the peak a density below e^-90 of it changes no bit of the sums; before it
      // even the smallest one is the first interval of the smallest uniforms)
      for (int k = tid; k < SNODE; k += ST) {
        const double p = pn[at(k)] - pm;
        pn[at(k)] = p;
        en[at(k)] = (p > -90.0 || sv + k * h < x) ? exp(p) : 0.0;
      }
      __syncthreads();
      // interval k = [v_k, v_{k+1}], k < SNODE - 1; each thread takes SPT in a row
      auto area = [&](int k) {
        if (k >= SNODE - 1) return 0.0;
        const double dp = pn[at(k + 1)] - pn[at(k)], e0 = en[at(k)], e1 = en[at(k + 1)];
        if (!(e0 > 0.0) && !(e1 > 0.0)) return 0.0;
        return (fabs(dp) < 1e-12) ? h * e0 : h * (e1 - e0) / dp;
      };
      double ak[SPT], loc = 0.0;
#pragma unroll
      for (int q = 0; q < SPT; ++q) {
        ak[q] = area(tid * SPT + q);
        loc += ak[q];
      }
      double incl = wscan(loc, lane);
      if (lane == 31) sh[w] = incl;
      __syncthreads();
      const double total = sh[0] + sh[1];
      if (w == 1) incl += sh[0];
      const double target = u4 * total;
      double vres = -1.0;
      if (incl - loc <= target && target < incl) {
        double c = incl - loc;
#pragma unroll
        for (int q = 0; q < SPT; ++q) {
          const int k = tid * SPT + q;
          if (vres < 0.0 && c + ak[q] > target && k < SNODE - 1) {
            const double e0 = en[at(k)];
            const double slope = (pn[at(k + 1)] - pn[at(k)]) / h, rem = target - c;
            const double v0 = sv + k * h;
            vres = (fabs(slope) < 1e-12) ? v0 + rem / e0 : v0 + log1p(slope * rem / e0) / slope;
          }
          c += ak[q];
        }
      }
      vres = wmax(vres);
      __syncthreads();
      if (lane == 0) sh[w] = vres;
      __syncthreads();
      vres = fmax(sh[0], sh[1]);
      if (!(vres >= 0.0)) vres = vhi;
      dist = r / vres;
    }
  }
  if (tid == 0) {
    if (i_out) i_out[s] = i;
    if (e_out) e_out[s] = e;
    if (o_out) o_out[s] = o;
    if (d_out) d_out[s] = dist;
    if (e < 0 || o < 0) atomicCAS(a.status, 0, DEV_E_SHAPE);
  }
}

// scratch of the row weights, after the cdf: block totals and their prefix, the maximum
size_t sample_scratch_doubles(int64_t n_int) { return (size_t)(n_int + 2 * ((n_int + RBLK - 1) / RBLK) + 2); }

void launch_sample(const SampleArgs &a, int64_t n, const double *uni, double *scr, int64_t *i_out, int64_t *e_out,
                   int32_t *o_out, double *d_out, cudaStream_t st) {
  const int nb = (int)((a.n_int + RBLK - 1) / RBLK);
  double *cdf = scr, *tot = cdf + a.n_int, *pre = tot + nb;
  unsigned long long *mx = (unsigned long long *)(pre + nb + 1);
  cudaMemsetAsync(mx, 0, 8, st);  // below every ordered value
  sample_row_max_kernel<<<nb < 256 ? nb : 256, 256, 0, st>>>(a.n_int, a.ln_p_int, mx);
  sample_row_cdf_kernel<<<nb, RBLK, 0, st>>>(a.n_int, a.ln_p_int, mx, cdf, tot);
  sample_row_prefix_kernel<<<1, 256, 0, st>>>(nb, tot, pre);
  if (!a.rb_dh)
    sample_weights_kernel<<<(unsigned)((a.n_det * a.n_bins + 127) / 128), 128, 0, st>>>(a.n_det, a.n_bins, a.w, a.psd,
                                                                                       a.data, a.om, a.cw);
  if (a.n_pol == 2)
    sample_kernel<2><<<(unsigned)n, ST, 0, st>>>(a, n, uni, cdf, pre, i_out, e_out, o_out, d_out);
  else
    sample_kernel<1><<<(unsigned)n, ST, 0, st>>>(a, n, uni, cdf, pre, i_out, e_out, o_out, d_out);
}

}  // namespace dotpe
