// Fused per-pair epilogue shared by the FP32 SIMT and tcgen05 kernels.
//
// Given the per-mode components Z_m = sum_b h_{im}(b) G_m[b,e] of one (i,e)
// pair (Eq. dh_ieo: Re<d|h>(phi) = Re sum_m Z_m e^{i m phi}) and the <h|h>
// coefficients C_0, C_delta (Eq. hh_ieo: <h|h>(phi) = C_0 + 2 Re sum_delta
// C_delta e^{i delta phi}), evaluate on the regular phase grid phi_o:
//   ln L^ML_o   (Eq. bestfit_lnl),
//   the coherent-ML selection (Eq. coherent_ML_selection) against `thr`,
//   ln Lbar_o   (Eq. lnl_dist_marginalized, device table),
//   and the phase sums ln sum_o Lbar_o, ln sum_o Lbar_o^2 (w_o = 1).
#pragma once
#include "common.cuh"
#include "dist_marg.cuh"

namespace dotpe {

struct PairRes {
  float lsum;   // ln sum_o Lbar_o (-inf if no phase marginalised)
  float lsum2;  // ln sum_o Lbar_o^2
  float ml;     // max_o ln L^ML_o
  int argo;     // its phase index (lowest on ties)
  int npass;    // phases marginalised
};

// Phase table in shared memory: e^{i k phi_o}, k = 1..4, as ph[2 o] = (c1, s1, c2, s2),
// ph[2 o + 1] = (c3, s3, c4, s4).  The azimuthal numbers of a bank's modes are in 1..4
// and the delta of <h|h> in 1..3, so one row of 32 bytes per phase serves both; Z is
// held by azimuthal number (zero where the bank has no such mode).
__device__ __forceinline__ void fill_phase_tables(float4 *ph, const EpiParams &P, int tid, int nthreads) {
  float2 *t = reinterpret_cast<float2 *>(ph);
  for (int q = tid; q < 4 * MAXPHI; q += nthreads) {
    const int o = q / 4, k = q % 4 + 1;
    float s, c;
    // angle = k * 2 pi o / n_phi, reduced exactly in integers first
    const int num = (k * o) % (P.n_phi > 0 ? P.n_phi : 1);
    sincospif(2.0f * (float)num / (float)P.n_phi, &s, &c);
    t[q] = make_float2(c, s);
  }
}

// <h|h> coefficients for a polarisation-resolved bank (Eqs. hh_ieo with the
// polarisation index): H_{mm'} = sum_d sum_{pp'} F_p F_p' <h_{mp}|h_{m'p'}>_d.
// The row record of detector d (mrow + d REC_P, read through the cache) holds
// the overlaps grouped by delta = m - m': [X0, Y0, W0] for delta = 0 (real), then
// for delta = 1..3 (X, Y, W) complex, with X = sum <h_a+|h_c+>, Y = sum (<h_a+|h_cx>
// + <h_ax|h_c+>), W = sum <h_ax|h_cx>; the column record holds (F+^2, F+ Fx, Fx^2).
__device__ __forceinline__ void hh_coeffs_pol(const float *__restrict__ mrow, const float *__restrict__ qrec,
                                              const EpiParams &P, float &C0, float Cr[3], float Ci[3]) {
  C0 = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) { Cr[k] = 0.f; Ci[k] = 0.f; }
  for (int d = 0; d < P.n_det; ++d) {
    const float *r = mrow + d * REC_P;
    const float *q = qrec + d * REC;
    const float q0 = q[0], q1 = q[1], q2 = q[2];
    C0 += q0 * __ldg(r) + q1 * __ldg(r + 1) + q2 * __ldg(r + 2);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float *g = r + 3 + 6 * k;
      Cr[k] += q0 * __ldg(g) + q1 * __ldg(g + 2) + q2 * __ldg(g + 4);
      Ci[k] += q0 * __ldg(g + 1) + q1 * __ldg(g + 3) + q2 * __ldg(g + 5);
    }
  }
}

// One detector's share of the <h|h> coefficients, added to c0, cr, ci (see hh_coeffs_by).
template <bool CONSEC, class Row>
__device__ __forceinline__ void hh_det(Row mr, const float *__restrict__ q, const EpiParams &P, float &c0,
                                       float (&cr)[3], float (&ci)[3]) {
  const float4 *q4 = reinterpret_cast<const float4 *>(q);
  float qr[REC];
#pragma unroll
  for (int v = 0; v < REC / 4; ++v) {
    const float4 x = q4[v];
    qr[4 * v] = x.x; qr[4 * v + 1] = x.y; qr[4 * v + 2] = x.z; qr[4 * v + 3] = x.w;
  }
#pragma unroll
  for (int m = 0; m < MAXM; ++m) c0 = fmaf(mr(m), qr[m], c0);
  int p = 0;
#pragma unroll
  for (int a = 1; a < MAXM; ++a)
#pragma unroll
    for (int b = 0; b < a; ++b, ++p) {
      const float ar = mr(4 + 2 * p), ai = mr(5 + 2 * p);
      const float br = qr[4 + 2 * p], bi = qr[5 + 2 * p];
      if (CONSEC) {
        const int k = a - b - 1;
        cr[k] = fmaf(ar, br, fmaf(-ai, bi, cr[k]));
        ci[k] = fmaf(ar, bi, fmaf(ai, br, ci[k]));
      } else {
        const float hr = ar * br - ai * bi, hi = ar * bi + ai * br;
        const int dl = P.pdelta[p];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const bool sel = (dl == k + 1);
          cr[k] += sel ? hr : 0.f;
          ci[k] += sel ? hi : 0.f;
        }
      }
    }
}

// <h|h> coefficients for one pair from the row record (mrec) and column record (qrec):
// C_0 = sum_d sum_m M_d[m,m] Q_d[m,m];  C_delta = sum_d sum_{a>b, m_a-m_b=delta} M_d[a,b] Q_d[a,b].
// CONSEC: the modes' azimuthal numbers are consecutive, so pair (a, b) has delta = a - b.
// Each detector accumulates into its own partial sums (independent FMA chains),
// added at the end; records of detectors d >= n_det are zero.
// The row record's entry k of detector d is mr_at(d REC + k) (registers or memory).
template <bool CONSEC, class Row>
__device__ __forceinline__ void hh_coeffs_by(Row mr_at, const float *__restrict__ qrec, const EpiParams &P,
                                             float &C0, float Cr[3], float Ci[3]) {
  float c0[MAXD], cr[MAXD][3], ci[MAXD][3];
#pragma unroll
  for (int d = 0; d < MAXD; ++d) {
    c0[d] = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) { cr[d][k] = 0.f; ci[d][k] = 0.f; }
  }
  const int nd = P.n_det;
#pragma unroll
  for (int d = 0; d < MAXD; ++d) {
    if (d >= nd) break;
    hh_det<CONSEC>([&](int k) { return mr_at(d * REC + k); }, qrec + d * REC, P, c0[d], cr[d], ci[d]);
  }
  C0 = (c0[0] + c0[1]) + c0[2];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    Cr[k] = (cr[0][k] + cr[1][k]) + cr[2][k];
    Ci[k] = (ci[0][k] + ci[1][k]) + ci[2][k];
  }
}

template <bool CONSEC>
__device__ __forceinline__ void hh_coeffs(const float *__restrict__ mrec, const float *__restrict__ qrec,
                                          const EpiParams &P, float &C0, float Cr[3], float Ci[3]) {
  hh_coeffs_by<CONSEC>([&](int k) { return mrec[k]; }, qrec, P, C0, Cr, Ci);
}

// Polarisation-resolved bank, row records held in registers (tensor-core
// epilogue): mrec [POL_TC_MAXD][REC_POL] as hh_coeffs_pol reads them from
// memory, the column record's (F+^2, F+ Fx, Fx^2) as one float4 per detector.
__device__ __forceinline__ void hh_coeffs_pol_reg(const float *mrec, const float *__restrict__ qrec,
                                                  const EpiParams &P, float &C0, float Cr[3], float Ci[3]) {
  C0 = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) { Cr[k] = 0.f; Ci[k] = 0.f; }
#pragma unroll
  for (int d = 0; d < POL_TC_MAXD; ++d) {
    if (d >= P.n_det) break;
    const float4 q = *reinterpret_cast<const float4 *>(qrec + d * REC);
    const float *r = mrec + d * REC_POL;
    C0 += q.x * r[0] + q.y * r[1] + q.z * r[2];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      Cr[k] += q.x * r[3 + 6 * k] + q.y * r[5 + 6 * k] + q.z * r[7 + 6 * k];
      Ci[k] += q.x * r[4 + 6 * k] + q.y * r[6 + 6 * k] + q.z * r[8 + 6 * k];
    }
  }
}

// <h|h> coefficients of the tensor-core epilogue: HH = 0 general modes, 1
// consecutive modes, 2 polarisation-resolved bank (registers as above).
template <int HH>
__device__ __forceinline__ void hh_tile(const float *mrec, const float *__restrict__ qrec, const EpiParams &P,
                                        float &C0, float Cr[3], float Ci[3]) {
  if constexpr (HH == 2) hh_coeffs_pol_reg(mrec, qrec, P, C0, Cr, Ci);
  else hh_coeffs<HH == 1>(mrec, qrec, P, C0, Cr, Ci);
}

// <h|h> coefficients from bank row i's record in memory (mx, n_det records per row), over
// detectors d0 <= d < d1: a partial sum per detector, added in detector order.
template <int HH>
__device__ __forceinline__ void hh_row(const float *__restrict__ mx, int64_t i, const float *__restrict__ qrec,
                                       const EpiParams &P, int d0, int d1, float &C0, float (&Cr)[3],
                                       float (&Ci)[3]) {
  C0 = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) { Cr[k] = 0.f; Ci[k] = 0.f; }
  constexpr int RL = HH == 2 ? REC_P : REC;
#pragma unroll 1
  for (int d = d0; d < d1; ++d) {
    const float4 *src = reinterpret_cast<const float4 *>(mx + (i * P.n_det + d) * RL);
    float m[RL];
#pragma unroll
    for (int v = 0; v < RL / 4; ++v) {
      const float4 x = __ldg(src + v);
      m[4 * v] = x.x; m[4 * v + 1] = x.y; m[4 * v + 2] = x.z; m[4 * v + 3] = x.w;
    }
    float c0 = 0.f, cr[3] = {0.f, 0.f, 0.f}, ci[3] = {0.f, 0.f, 0.f};
    if constexpr (HH == 2) {
      const float4 q = *reinterpret_cast<const float4 *>(qrec + d * REC);
      c0 = q.x * m[0] + q.y * m[1] + q.z * m[2];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        cr[k] = q.x * m[3 + 6 * k] + q.y * m[5 + 6 * k] + q.z * m[7 + 6 * k];
        ci[k] = q.x * m[4 + 6 * k] + q.y * m[6 + 6 * k] + q.z * m[8 + 6 * k];
      }
    } else {
      hh_det<HH == 1>([&](int k) { return m[k]; }, qrec + d * REC, P, c0, cr, ci);
    }
    C0 += c0;
#pragma unroll
    for (int k = 0; k < 3; ++k) { Cr[k] += cr[k]; Ci[k] += ci[k]; }
  }
}

// Upper bound of max_o ln L^ML_o of a pair: |dh| <= sum_m |Z_m| and
// hh >= C_0 - 2 sum |C_delta| at every phase; +inf when that lower bound is not positive.
__device__ __forceinline__ float pair_bound(const float Zr[MAXM], const float Zi[MAXM], float C0, const float Cr[3],
                                            const float Ci[3]) {
  float a = 0.f, hmin = C0;
#pragma unroll
  for (int m = 0; m < MAXM; ++m) a += sqrtf(Zr[m] * Zr[m] + Zi[m] * Zi[m]);
#pragma unroll
  for (int k = 0; k < 3; ++k) hmin -= 2.f * sqrtf(Cr[k] * Cr[k] + Ci[k] * Ci[k]);
  return hmin > 0.f ? __fdividef(0.5f * a * a, hmin) * 1.000001f : INFINITY;
}

// dh and hh of phase o: the rows' rotations, summed in the order of the azimuthal numbers.
__device__ __forceinline__ void phase_at(const float (&Zr)[4], const float (&Zi)[4], float C0, const float (&Cr)[3],
                                         const float (&Ci)[3], const float4 *__restrict__ ph, int o, float &dh,
                                         float &hh) {
  const float4 e = ph[2 * o], f = ph[2 * o + 1];
  const float c[4] = {e.x, e.z, f.x, f.z}, s[4] = {e.y, e.w, f.y, f.w};
  dh = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) dh = fmaf(Zr[k], c[k], fmaf(-Zi[k], s[k], dh));
  float hs = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) hs = fmaf(Cr[k], c[k], fmaf(-Ci[k], s[k], hs));
  hh = fmaf(2.f, hs, C0);
}

// dh and hh of the four phases o + j n_phi / 4, j = 0..3, from one rotation of each Z_k
// and C_delta: e^{i k (phi + j pi / 2)} = i^{jk} e^{i k phi} (about 9 operations and half
// a shared load per phase instead of 14 and 7).
__device__ __forceinline__ void phase_quad(const float (&Zr)[4], const float (&Zi)[4], float C0, const float (&Cr)[3],
                                           const float (&Ci)[3], const float4 *__restrict__ ph, int o, float (&dh)[4],
                                           float (&hh)[4]) {
  const float4 e = ph[2 * o], f = ph[2 * o + 1];
  const float z2 = fmaf(Zr[1], e.z, -Zi[1] * e.w), z4 = fmaf(Zr[3], f.z, -Zi[3] * f.w);
  const float zr = fmaf(Zr[0], e.x, fmaf(-Zi[0], e.y, fmaf(Zr[2], f.x, -Zi[2] * f.y)));   // Re (Z_1 + Z_3)
  const float zi = fmaf(Zr[2], f.y, fmaf(Zi[2], f.x, -fmaf(Zr[0], e.y, Zi[0] * e.x)));    // Im (Z_3 - Z_1)
  const float zp = z4 + z2, zm = z4 - z2;
  dh[0] = zp + zr;
  dh[1] = zm + zi;
  dh[2] = zp - zr;
  dh[3] = zm - zi;
  const float h2 = fmaf(Cr[1], e.z, -Ci[1] * e.w);
  const float hr = fmaf(Cr[0], e.x, fmaf(-Ci[0], e.y, fmaf(Cr[2], f.x, -Ci[2] * f.y)));
  const float hi = fmaf(Cr[2], f.y, fmaf(Ci[2], f.x, -fmaf(Cr[0], e.y, Ci[0] * e.x)));
  // (one rounding at the size of C_0, as in phase_at: the sums of the other terms are smaller)
  hh[0] = fmaf(2.f, h2 + hr, C0);
  hh[1] = fmaf(2.f, hi - h2, C0);
  hh[2] = fmaf(2.f, h2 - hr, C0);
  hh[3] = fmaf(-2.f, h2 + hi, C0);
}

__device__ __forceinline__ float lnl_ml_of(float dh, float hh) {
  return (dh > 0.f && hh > 0.f) ? __fdividef(0.5f * dh * dh, hh) : 0.f;
}

// The maximum as the sums' reference: finite also where nothing has been added yet (-inf,
// whose terms are then zero) and where a value has overflowed (its sum stays +inf).
__device__ __forceinline__ float lse_ref(float m) { return fminf(fmaxf(m, -3.402823466e38f), 3.402823466e38f); }

// Online sums of exp(l) and exp(2 l) over N more values (-inf: none).
template <int N>
__device__ __forceinline__ void lse2_add(float &mx, float &s1, float &s2, const float (&l)[N]) {
  float m = mx;
#pragma unroll
  for (int k = 0; k < N; ++k) m = fmaxf(m, l[k]);
  const float c = lse_ref(m);
  const float r = __expf(mx - c);
  s1 *= r;
  s2 *= r * r;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const float q = __expf(l[k] - c);
    s1 += q;
    s2 = fmaf(q, q, s2);
  }
  mx = m;
}

// What the phases of one pair leave: online sums of Lbar and Lbar^2, the best ln L^ML.
struct PhaseSums {
  float mx, s1, s2, best;
  int argo, npass;
  __device__ __forceinline__ void init() {
    mx = -INFINITY; s1 = 0.f; s2 = 0.f; best = -1.f; argo = 0; npass = 0;
  }
  // with the sums of the lane o away (every lane of the warp calls it)
  __device__ __forceinline__ void merge_xor(int o) {
    const float om = __shfl_xor_sync(0xffffffffu, mx, o), o1 = __shfl_xor_sync(0xffffffffu, s1, o),
                o2 = __shfl_xor_sync(0xffffffffu, s2, o), ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oa = __shfl_xor_sync(0xffffffffu, argo, o);
    npass += __shfl_xor_sync(0xffffffffu, npass, o);
    const float m = fmaxf(mx, om), c = lse_ref(m);
    const float r = __expf(mx - c), q = __expf(om - c);
    s1 = fmaf(s1, r, o1 * q);
    s2 = fmaf(s2, r * r, o2 * q * q);
    mx = m;
    if (ob > best || (ob == best && oa < argo)) { best = ob; argo = oa; }
  }
  __device__ __forceinline__ PairRes result() const {
    PairRes R;
    R.ml = best;
    R.argo = argo;
    R.npass = npass;
    R.lsum = npass > 0 ? mx + __logf(s1) : -INFINITY;
    R.lsum2 = npass > 0 ? 2.f * mx + __logf(s2) : -INFINITY;
    return R;
  }
};

// phase_quad's sums differ from phase_at's by the order of their additions and the entries
// of the phase table that they start from: by less than 2^-18 of sum |Z| and of
// C_0 + 2 sum |C_delta| (the entries agree to 5e-7, each sum rounds at most 8 times).
constexpr float PHASE_SLACK = 3.8146973e-6f;

// One pair over the phase grid, or the part of it with base phases b0, b0 + step, ...
// Without a cut (thr <= 0: every phase has ln L^ML >= 0) phases go four at a time (a
// quarter turn apart when n_phi is a multiple of 4, else phase by phase) and all are
// marginalised as they come, two gathers of the distance table in flight.
// With a cut a phase is kept where its ln L^ML, from phase_at, reaches thr: one decision
// for every kernel, grid and option, so that an event keeps the same phases whichever way
// its pairs are evaluated.  The phases that may pass are marked first, four at a time, by
// dh > 0 and dh^2 >= 2 thr hh with the slack of the quick sums, and then evaluated two at a
// time, each thread taking its own next ones: a warp takes as many steps as its busiest
// lane has marked phases, not one for every phase that any of its lanes passes.  ln L^ML
// itself is needed for those only (the maximum is among them), or with want_best (stored
// values) for all phases, which then go through phase_at one by one.
__device__ __forceinline__ void pair_phases(const float (&Zr)[4], const float (&Zi)[4], float C0,
                                            const float (&Cr)[3], const float (&Ci)[3], float thr, bool want_best,
                                            const EpiParams &P, const float4 *__restrict__ ph, int b0, int step,
                                            PhaseSums &S) {
  const int n = P.n_phi, nb = (n + 3) >> 2;
  const bool quad = (n & 3) == 0, all = !(thr > 0.f), exact = !quad || (want_best && !all);
  const float thr2 = 2.f * thr;
  float dh_slack = 0.f, hh_slack = 0.f;
  if (!exact) {
    float a = 0.f, h = fabsf(C0);
#pragma unroll
    for (int k = 0; k < 4; ++k) a += fabsf(Zr[k]) + fabsf(Zi[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) h += 2.f * (fabsf(Cr[k]) + fabsf(Ci[k]));
    dh_slack = PHASE_SLACK * a;
    hh_slack = PHASE_SLACK * h * thr2;
  }
  uint32_t mk[4] = {0u, 0u, 0u, 0u};  // bit b of mk[j]: phase b + j nb may pass (nb <= 32)
#pragma unroll 1
  for (int b = b0; b < nb; b += step) {
    float dh[4], hh[4];
    if (!exact) {
      phase_quad(Zr, Zi, C0, Cr, Ci, ph, b, dh, hh);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        phase_at(Zr, Zi, C0, Cr, Ci, ph, min(b + j * nb, n - 1), dh[j], hh[j]);
        if (b + j * nb >= n) { dh[j] = -1.f; hh[j] = -1.f; }
      }
    }
    if (all || want_best) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int o = b + j * nb;
        const bool on = quad || o < n;
        const float ml = lnl_ml_of(dh[j], hh[j]);
        if (on && (ml > S.best || (ml == S.best && o < S.argo))) { S.best = ml; S.argo = o; }
        mk[j] |= (on && ml >= thr) ? 1u << b : 0u;
      }
    } else if (exact) {
#pragma unroll
      for (int j = 0; j < 4; ++j) mk[j] |= lnl_ml_of(dh[j], hh[j]) >= thr ? 1u << b : 0u;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float d = fmaxf(dh[j] + dh_slack, 0.f);
        mk[j] |= d * d >= fmaf(thr2, hh[j], -hh_slack) ? 1u << b : 0u;
      }
    }
    if (all) {
      float l[4];
#pragma unroll
      for (int q = 0; q < 4; q += 2) {
        const float d2[2] = {dh[q], dh[q + 1]}, h2[2] = {hh[q], hh[q + 1]};
        float l2[2];
        dm_lnlbar_n<2>(d2, h2, P.u_min, P.dm_table, l2);
        l[q] = l2[0];
        l[q + 1] = l2[1];
      }
      if (!quad) {
#pragma unroll
        for (int j = 1; j < 4; ++j) l[j] = (b + j * nb < n) ? l[j] : -INFINITY;
      }
      lse2_add<4>(S.mx, S.s1, S.s2, l);
    }
  }
  if (all) {
    S.npass = __popc(mk[0]) + __popc(mk[1]) + __popc(mk[2]) + __popc(mk[3]);
    return;
  }
  // up to 32 phases in one word, else a word per quarter of the grid
  const bool one = nb <= 8;
  if (one) mk[0] |= (mk[1] << 8) | (mk[2] << 16) | (mk[3] << 24);
#pragma unroll 1
  for (int w = 0; w < (one ? 1 : 4); ++w) {
    uint32_t m = mk[0];
#pragma unroll
    for (int q = 1; q < 4; ++q)
      if (w == q) m = mk[q];
    auto phase_of = [&](int bit) { return one ? (bit & 7) + (bit >> 3) * nb : bit + w * nb; };
    while (m) {
      const int o0 = phase_of(__ffs(m) - 1);
      m &= m - 1;
      const bool two = m != 0;
      const int o1 = two ? phase_of(__ffs(m) - 1) : o0;
      m &= m - 1;
      float dh[2], hh[2], l[2];
      phase_at(Zr, Zi, C0, Cr, Ci, ph, o0, dh[0], hh[0]);
      phase_at(Zr, Zi, C0, Cr, Ci, ph, o1, dh[1], hh[1]);
      const float m0 = lnl_ml_of(dh[0], hh[0]), m1 = lnl_ml_of(dh[1], hh[1]);
      // (in increasing o: the lowest keeps a tie)
      if (m0 > S.best) { S.best = m0; S.argo = o0; }
      if (m1 > S.best) { S.best = m1; S.argo = o1; }
      const bool k0 = m0 >= thr, k1 = two && m1 >= thr;
      S.npass += (int)k0 + (int)k1;
      dm_lnlbar_n<2>(dh, hh, P.u_min, P.dm_table, l);
      if (!k0) l[0] = -INFINITY;
      if (!k1) l[1] = -INFINITY;
      lse2_add<2>(S.mx, S.s1, S.s2, l);
    }
  }
}

__device__ __forceinline__ PairRes pair_eval(const float (&Zr)[4], const float (&Zi)[4], float C0,
                                             const float (&Cr)[3], const float (&Ci)[3], float thr,
                                             bool allow_skip, const EpiParams &P, const float4 *__restrict__ ph) {
  PhaseSums S;
  S.init();
  if (allow_skip && thr > 0.f) {
    // upper bound of max_o ln L^ML: |dh| <= sum |Z_m|, hh >= C_0 - 2 sum |C_delta|
    float a = 0.f, hmin = C0;
#pragma unroll
    for (int m = 0; m < MAXM; ++m) a += sqrtf(Zr[m] * Zr[m] + Zi[m] * Zi[m]);
#pragma unroll
    for (int k = 0; k < 3; ++k) hmin -= 2.f * sqrtf(Cr[k] * Cr[k] + Ci[k] * Ci[k]);
    if (hmin > 0.f && a * a < 2.f * hmin * thr) {
      S.best = 0.f;
      return S.result();
    }
  }
  pair_phases(Zr, Zi, C0, Cr, Ci, thr, !allow_skip, P, ph, 0, 1, S);
  return S.result();
}

// Screening evaluation (no distance marginal): max_o ln L^ML_o and its phase.
// A pair whose upper bound (as in pair_eval) is below thr returns ml = -1: it
// cannot reach the cut.
__device__ __forceinline__ float pair_ml(const float (&Zr)[4], const float (&Zi)[4], float C0, const float (&Cr)[3],
                                         const float (&Ci)[3], float thr, bool allow_skip, const EpiParams &P,
                                         const float4 *__restrict__ ph, int &argo) {
  argo = 0;
  if (allow_skip && thr > 0.f) {
    float a = 0.f, hmin = C0;
#pragma unroll
    for (int m = 0; m < MAXM; ++m) a += sqrtf(Zr[m] * Zr[m] + Zi[m] * Zi[m]);
#pragma unroll
    for (int k = 0; k < 3; ++k) hmin -= 2.f * sqrtf(Cr[k] * Cr[k] + Ci[k] * Ci[k]);
    if (hmin > 0.f && a * a < 2.f * hmin * thr) return -1.f;
  }
  float best = -1.f;
#pragma unroll 4
  for (int o = 0; o < P.n_phi; ++o) {
    float dh, hh;
    phase_at(Zr, Zi, C0, Cr, Ci, ph, o, dh, hh);
    const float ml = lnl_ml_of(dh, hh);
    if (ml > best) { best = ml; argo = o; }
  }
  return best;
}

// Cut threshold of a tile (Eq. coherent_ML_selection): running maximum - cut_delta,
// lowered by twice the screening margin in a screening pass (so that no pair the
// exact product would keep is skipped); -inf when the cut is off.
__device__ __forceinline__ float tile_threshold(const EpiParams &P) {
  if (!(P.cut_delta > 0.f)) return -INFINITY;
  const float run = *(volatile float *)P.ml_running;
  float thr = run - P.cut_delta;
  if (P.margin_k > 0.f) thr -= 2.f * screen_margin(run, P.margin_k, *P.sqrt_dd);
  return thr;
}

// Online log-sum-exp accumulator.
struct Lse {
  float m, s;
  __device__ __forceinline__ void init() { m = -INFINITY; s = 0.f; }
  __device__ __forceinline__ void add(float x) {
    if (x == -INFINITY) return;
    if (x > m) { s = fmaf(s, __expf(m - x), 1.f); m = x; }
    else s += __expf(x - m);
  }
  __device__ __forceinline__ void merge(float om, float os) {
    if (om == -INFINITY) return;
    if (m == -INFINITY) { m = om; s = os; return; }
    if (om > m) { s = fmaf(s, __expf(m - om), os); m = om; }
    else s = fmaf(os, __expf(om - m), s);
  }
};

__device__ __forceinline__ void warp_merge_lse(Lse &a) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float om = __shfl_xor_sync(0xffffffffu, a.m, o);
    float os = __shfl_xor_sync(0xffffffffu, a.s, o);
    a.merge(om, os);
  }
}

// (value, packed index) max with lowest index on ties
__device__ __forceinline__ void warp_argmax(float &v, long long &idx) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    float ov = __shfl_xor_sync(0xffffffffu, v, o);
    long long oi = __shfl_xor_sync(0xffffffffu, idx, o);
    if (ov > v || (ov == v && oi < idx)) { v = ov; idx = oi; }
  }
}

}  // namespace dotpe
