// Incoherent single-detector pre-selection (Sec. IV.D, App. B) of a
// polarisation-resolved bank, in FP32 on the CUDA cores.
//
// For bank row i, detector k, arrival time t_{kt} and phase phi_o:
//   Z_{ikmpt}     = sum_b h_{imp}(f_b) c_{kb} e^{-2 pi i f_b t_{kt}}       (Eq. dh_itop, per component)
//   <d|h>_{iktop} = Re sum_m e^{i m phi_o} Z_{ikmpt}
//   <h|h>_{ikopp'}: from the row's records of the bank's own overlaps grouped by
//                   delta = m - m' (cross_terms_pol_kernel): hh_{++} = X0 + 2 Re sum X_d e^{i d phi},
//                   hh_{xx} = W0 + 2 Re sum W_d e^{i d phi}, hh_{+x} = Y0 / 2 + Re sum Y_d e^{i d phi}
//   ln L^ML_{ikot} = dh^T [hh]^+ dh / 2                                   (Eqs. x_ML, single_det_ML)
// and, per (i, k), the maximum over (o, t) as the 64-bit key the tensor-core
// pre-selection writes (lowest t, then lowest o, on ties), so the same finish
// kernels form the per-row sums and the selection.
//
// One block per (4 rows, detector).  A thread holds the complex Z of 2 rows x M x 2
// components at 2 times, (re, im) packed: one fma.rn.f32x2 with (g.x, g.x) and (h.x, h.y),
// one with (g.y, g.y) and (-h.y, h.x); the rows' components lie in shared memory in
// both forms, 16 bytes per bin, and a warp's 16 lanes x 2 row pairs read two addresses in
// one wavefront.  The time-grid operand [D][B][n_tpad] (times innermost) is two 8-byte
// loads per bin and thread, held four bins ahead.  Per bin that is 64 packed FMAs to 16 shared and 2 global loads.
// With relative binning (App. A) the data weights differ per (mode, polarisation)
// component j = 2m + p, the time shifts do not: sum_b h_ij(b) W*_kjb e^{-2 pi i f_b t} takes
// the weighted row h_ij W*_kj, formed once per chunk for all times, against one operand
// e^{-2 pi i f_b t} for every component.  Each chunk of bins is summed on its own and added to
// the total kept in shared memory, so the sums' rounding grows with the bins of a chunk.
// What bounds it is the FMA pipe (57% busy) with the issue slots (57%) close behind: 16,384
// rows x 3 detectors x 128 times, 378 nodes, relative binning: 3.9 ms (2.1 ms at the pipe's
// rate); 5.25 ms with a lane per time, 4 rows and an operand per component (load unit 100%,
// FMA pipe 42%).  Measured on the way: an operand per component with this lane layout 4.8 ms,
// one operand and scalar FMAs 4.2 ms, this without the operand held four bins ahead 4.6 ms.
#include "common.cuh"
#include "kernels.h"

namespace dotpe {

namespace {
constexpr int PP_NT = 128;   // threads
constexpr int PP_TT = 128;   // time slots per pass: 32 per warp
constexpr int PP_RPB = 4;    // bank rows per block
constexpr int PP_RPT = 2;    // of them per thread
constexpr int PP_TPT = 2;    // times per thread, 16 apart
constexpr int PP_BCH = 32;   // bins per shared-memory chunk
constexpr int PP_GB = 4;     // bins of the operand held ahead
constexpr int PP_HROW = MAXM * 2 * PP_BCH;         // float4 of one row's chunk
constexpr int PP_HPAIR = PP_RPT * PP_HROW + 1;     // of a thread's rows (the next pair's 16 bytes on in the banks)
constexpr int PP_NACC = PP_RPT * MAXM * 2 * PP_TPT;  // complex sums per thread

struct PpSmem {
  float4 hs[PP_RPB / PP_RPT * PP_HPAIR];  // (h.x, h.y, -h.y, h.x)
  float2 tot[PP_NACC][PP_NT];             // each thread's sums of the earlier chunks
  float4 tab[PP_RPB][PS_MAXPHI];          // (a, 2b, c): ln L^ML = a dp^2 + 2b dp dx + c dx^2
  float2 ph[PS_MAXPHI][MAXM];             // e^{i m phi_o}
};

__device__ __forceinline__ uint64_t pp_dup(float x) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ uint64_t pp_fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
}  // namespace

template <bool RB>
__global__ void __launch_bounds__(PP_NT, 4) presel_pol_kernel(const PreselPolArgs a) {
  extern __shared__ __align__(16) uint8_t pp_smem[];
  PpSmem &S = *reinterpret_cast<PpSmem *>(pp_smem);
  auto &hs = S.hs;
  auto &tab = S.tab;
  auto &ph = S.ph;
  const int tid = threadIdx.x;
  // the detector is the fastest block index: the D blocks of one row group run
  // together and share the rows' FP32 components in L2
  const int k = (int)(blockIdx.x % (unsigned)a.n_det);
  const int64_t r0 = (int64_t)(blockIdx.x / (unsigned)a.n_det) * PP_RPB;
  const int M = a.n_modes, B = a.n_bins, D = a.n_det, np = a.n_phi;
  // phase factors (angles reduced in integers first)
  for (int q = tid; q < PS_MAXPHI * MAXM; q += PP_NT) {
    const int o = q / MAXM, m = q % MAXM;
    float s = 0.f, c = 1.f;
    if (o < np && m < M) sincospif(2.0f * (float)((a.mode_m[m] * o) % np) / (float)np, &s, &c);
    ph[o][m] = make_float2(c, s);
  }
  // [hh]^+ / 2 of the block's rows on every phase, from the rows' records
  for (int q = tid; q < PP_RPB * PS_MAXPHI; q += PP_NT) {
    const int r = q / PS_MAXPHI, o = q % PS_MAXPHI;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r0 + r < a.n_rows && o < np) {
      const float *rec = a.mx + ((r0 + r) * D + k) * REC_P;
      float A = __ldg(rec), Bx = 0.5f * __ldg(rec + 1), C = __ldg(rec + 2);
#pragma unroll
      for (int dl = 0; dl < 3; ++dl) {
        float s, c;
        sincospif(2.0f * (float)(((dl + 1) * o) % np) / (float)np, &s, &c);
        const float *g = rec + 3 + 6 * dl;
        A += 2.f * (__ldg(g) * c - __ldg(g + 1) * s);
        Bx += __ldg(g + 2) * c - __ldg(g + 3) * s;
        C += 2.f * (__ldg(g + 4) * c - __ldg(g + 5) * s);
      }
      const float det = A * C - Bx * Bx;
      if (det > a.rank_tol * A * C) {
        const float inv = 0.5f / det;
        v = make_float4(C * inv, -2.f * Bx * inv, A * inv, 0.f);
      } else if (A > 0.f || C > 0.f) {
        const float sm = A + C;
        const float inv = 0.5f / (sm * sm);
        v = make_float4(A * inv, 2.f * Bx * inv, C * inv, 0.f);
      }
    }
    tab[r][o] = v;
  }
  const int lane = tid & 31, w = tid >> 5;
  const int pair = lane >> 4;  // this thread's rows: 2 pair, 2 pair + 1
  const int64_t TP = a.n_tpad;
  for (int t0 = 0; t0 < a.n_t; t0 += PP_TT) {
    const int t = t0 + w * 32 + (lane & 15);  // and t + 16
    const bool any = t0 + w * 32 < a.n_t;     // (warp-uniform)
    // this thread's columns of the operand, bins TP apart (a time past the grid reads the
    // last one), four bins ahead of their use; a bin past the end is the last one again
    // (the rows' components are zero there)
    const float2 *ga = a.G + (int64_t)k * B * TP + min(t, a.n_t - 1);
    const float2 *gb = a.G + (int64_t)k * B * TP + min(t + 16, a.n_t - 1);
    float2 gn[PP_GB][PP_TPT];
    auto fetch = [&](int b) {
#pragma unroll
      for (int q = 0; q < PP_GB; ++q) {
        const int64_t off = (int64_t)min(b + q, B - 1) * TP;
        gn[q][0] = __ldg(ga + off);
        gn[q][1] = __ldg(gb + off);
      }
    };
    fetch(0);
    for (int b0 = 0; b0 < B; b0 += PP_BCH) {
      __syncthreads();  // the previous chunk is consumed (and, first time, the tables are written)
      for (int q = tid; q < PP_RPB * MAXM * 2 * PP_BCH; q += PP_NT) {
        const int bb = q % PP_BCH, rest = q / PP_BCH;
        const int p = rest % 2, m = (rest / 2) % MAXM, r = rest / (2 * MAXM);
        float2 v = make_float2(0.f, 0.f);
        if (r0 + r < a.n_rows && m < M && b0 + bb < B) {
          const float *row = a.master + ((int64_t)m * a.bank_rows + a.row0 + r0 + r) * a.kpad + 2 * p * B;
          v = make_float2(__ldg(row + b0 + bb), __ldg(row + B + b0 + bb));
          if constexpr (RB) {
            const float2 c = __ldg(a.c + ((int64_t)k * 2 * M + 2 * m + p) * B + b0 + bb);
            v = make_float2(v.x * c.x - v.y * c.y, v.x * c.y + v.y * c.x);
          }
        }
        hs[(r / PP_RPT) * PP_HPAIR + (r % PP_RPT) * PP_HROW + (2 * m + p) * PP_BCH + bb] =
            make_float4(v.x, v.y, -v.y, v.x);
      }
      __syncthreads();
      if (any) {
        uint64_t acc[PP_RPT][MAXM][2][PP_TPT];
#pragma unroll
        for (int r = 0; r < PP_RPT; ++r)
#pragma unroll
          for (int m = 0; m < MAXM; ++m)
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
              for (int u = 0; u < PP_TPT; ++u) acc[r][m][p][u] = 0ull;
        const int nb = min(PP_BCH, B - b0);
        const ulonglong2 *hb = reinterpret_cast<const ulonglong2 *>(hs + pair * PP_HPAIR);
#pragma unroll 1
        for (int bb = 0; bb < nb; bb += PP_GB, hb += PP_GB) {
          float2 gc[PP_GB][PP_TPT];
#pragma unroll
          for (int q = 0; q < PP_GB; ++q) {
            gc[q][0] = gn[q][0];
            gc[q][1] = gn[q][1];
          }
          fetch(b0 + bb + PP_GB);
#pragma unroll
          for (int q = 0; q < PP_GB; ++q) {
            const uint64_t x0 = pp_dup(gc[q][0].x), y0 = pp_dup(gc[q][0].y);
            const uint64_t x1 = pp_dup(gc[q][1].x), y1 = pp_dup(gc[q][1].y);
#pragma unroll
            for (int m = 0; m < MAXM; ++m) {
              if (m >= M) break;
#pragma unroll
              for (int p = 0; p < 2; ++p)
#pragma unroll
                for (int r = 0; r < PP_RPT; ++r) {
                  const ulonglong2 h = hb[r * PP_HROW + (2 * m + p) * PP_BCH + q];
                  acc[r][m][p][0] = pp_fma2(x0, h.x, pp_fma2(y0, h.y, acc[r][m][p][0]));
                  acc[r][m][p][1] = pp_fma2(x1, h.x, pp_fma2(y1, h.y, acc[r][m][p][1]));
                }
            }
          }
        }
#pragma unroll
        for (int r = 0; r < PP_RPT; ++r)
#pragma unroll
          for (int m = 0; m < MAXM; ++m)
#pragma unroll
            for (int p = 0; p < 2; ++p)
#pragma unroll
              for (int u = 0; u < PP_TPT; ++u) {
                float2 &s = S.tot[((r * MAXM + m) * 2 + p) * PP_TPT + u][tid];
                const uint64_t v = acc[r][m][p][u];
                const float2 z = make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
                s = b0 == 0 ? z : make_float2(s.x + z.x, s.y + z.y);
              }
      }
    }
    // per row: best (ln L^ML, o) over the phases of each time, the best over the warp's 32
    // times, one atomic per warp and row
#pragma unroll 1
    for (int r = 0; r < PP_RPT; ++r) {
      unsigned long long key = 0ull;
      const int rl = pair * PP_RPT + r;
#pragma unroll 1
      for (int u = 0; u < PP_TPT; ++u) {
        const int tu = t + 16 * u;
        if (tu >= a.n_t || r0 + rl >= a.n_rows) continue;
        float2 z[MAXM][2];
#pragma unroll
        for (int m = 0; m < MAXM; ++m)
#pragma unroll
          for (int p = 0; p < 2; ++p) z[m][p] = S.tot[((r * MAXM + m) * 2 + p) * PP_TPT + u][tid];
        float best = -1.f;
        int bo = 0;
        for (int o = 0; o < np; ++o) {
          float dp = 0.f, dx = 0.f;
#pragma unroll
          for (int m = 0; m < MAXM; ++m) {
            const float2 e = ph[o][m];
            dp += z[m][0].x * e.x - z[m][0].y * e.y;
            dx += z[m][1].x * e.x - z[m][1].y * e.y;
          }
          const float4 T = tab[rl][o];
          const float qv = fmaf(dp, fmaf(T.y, dx, T.x * dp), T.z * dx * dx);
          if (qv > best) { best = qv; bo = o; }
        }
        const unsigned long long ku = ((unsigned long long)__float_as_uint(fmaxf(best, 0.f)) << 32) |
                                      (unsigned long long)(0xffffffffu - (uint32_t)(tu * np + bo));
        key = ku > key ? ku : key;
      }
#pragma unroll
      for (int sh = 8; sh > 0; sh >>= 1) {
        const unsigned long long o2 = __shfl_xor_sync(0xffffffffu, key, sh);
        key = o2 > key ? o2 : key;
      }
      if ((lane & 15) == 0 && key != 0ull) atomicMax(a.keys + (r0 + rl) * D + k, key);
    }
  }
}

void launch_presel_pol(const PreselPolArgs &a, cudaStream_t st) {
  const dim3 grid((unsigned)(((a.n_rows + PP_RPB - 1) / PP_RPB) * a.n_det));
  auto go = [&](auto kern) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PpSmem));
    kern<<<grid, PP_NT, sizeof(PpSmem), st>>>(a);
  };
  if (a.c) go(presel_pol_kernel<true>);
  else go(presel_pol_kernel<false>);
}

}  // namespace dotpe
