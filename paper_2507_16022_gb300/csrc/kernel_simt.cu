// K7: plain FP32 path.  Fused <d|h> GEMM (FFMA on the CUDA cores) and the
// marginalisation epilogue, one 64 x 32 (i, e) tile per block.
//
// Per mode m the GEMM is the real-ified complex product of Eq. dh_ieo:
//   [h_r | h_i] (K = 2B) x [(e,re): (G_r | -G_i), (e,im): (G_i | G_r)]
// so each extrinsic sample e has two output columns, Re Z_m and Im Z_m.  The
// FP32 extrinsic operand interleaves them along K, [m][e][Kpad][2].
//
// Mainloop: 64 threads per mode (a block has 64 n_modes), each with 8 rows x 4
// samples of its mode in registers, (re, im) packed so that one instruction
// (fma.rn.f32x2: both halves round as fmaf does) advances both.  K in chunks of 16 through two
// cp.async stages that a mode's threads fill and order by a barrier of their own.  Per k-quad
// a thread reads 8 + 8 times 16 bytes for 128 packed FMAs, every read one wavefront (rows 20
// and samples 36 words apart), so shared memory is half busy and the FMA pipe is what is
// left: 8,192 x 1,024, B 512, M 4 takes 2.6 ms without the epilogue (1.85 ms at the pipe's
// rate), 2.8 ms with it and 3.3 ms with every pair stored under a cut.  It was 4.5 ms with every mode in each
// thread (4 rows x 2 samples, shared memory 78% busy).  Measured and not kept: scalar FMAs
// (3.7 ms), 4 rows x 8 samples (3.3 ms), sums split into even and odd k so that the
// operands need no copy of the row's value into both halves (4 x 4 per thread, 3.7 ms).
// The products of a pair are summed in k order.
//
// Epilogue: Z through shared memory (free after the mainloop), then a warp per row and a
// lane per sample: the row's record is a broadcast, stored values are written in whole lines.
#include <algorithm>

#include "common.cuh"
#include "epilogue.cuh"
#include "kernels.h"

namespace dotpe {

namespace {
constexpr int TI = SIMT_TI, TE = SIMT_TE, KC = 16;
constexpr int GT = 64;             // threads per mode
constexpr int AS_LD = KC + 4;      // words per bank row of a stage
constexpr int BS_LD = 2 * KC + 4;  // words per extrinsic sample of a stage ((re, im) per k)
constexpr int A_W = TI * AS_LD, B_W = TE * BS_LD;  // words of one mode's chunk
constexpr int Z_W = TI * TE;                       // words of one component of Z
constexpr int QS_LD = MAXD * REC + 4;  // words per column record: 16-byte reads of 8 lanes in 8 bank groups
constexpr int MAXW = 2 * MAXM;         // warps of a block
static_assert(2 * (A_W + B_W) >= 2 * Z_W, "Z fits in the stages");

struct SimtSmem {
  alignas(16) float qs[TE * QS_LD];
  double lwe[TE];
  float4 ph[2 * MAXPHI];
  float2 col[MAXW][TE];                     // column partials of each warp's rows
  float w_m1[MAXW], w_s1[MAXW], w_m2[MAXW], w_s2[MAXW], w_ml[MAXW];
  long long w_arg[MAXW];
  int w_np[MAXW];
};

// the stages (or Z) of n_modes modes, then SimtSmem
__host__ __device__ constexpr size_t stage_bytes(int n_modes) { return (size_t)n_modes * 2 * (A_W + B_W) * 4; }

__device__ __forceinline__ void cp_async16(uint32_t smem, const void *gmem, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem), "l"(gmem),
               "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// c + a b for both halves of b and c
__device__ __forceinline__ uint64_t fma2(float a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("{\n\t.reg .b64 t;\n\tmov.b64 t, {%1, %1};\n\tfma.rn.f32x2 %0, t, %2, %3;\n\t}"
      : "=l"(d)
      : "f"(a), "l"(b), "l"(c));
  return d;
}
// Z of (component c, row, sample): eight samples of four consecutive rows in other banks
__device__ __forceinline__ int z_at(int c, int row, int el) { return c * Z_W + row * TE + (el ^ ((row & 3) << 3)); }
}  // namespace

__global__ void __launch_bounds__(GT * MAXM, 2) simt_fused_kernel(SimtArgs g, EpiParams P, int tile0, int n_etile) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int M = P.n_modes;
  float *stage = reinterpret_cast<float *>(smem_raw);
  SimtSmem &S = *reinterpret_cast<SimtSmem *>(smem_raw + stage_bytes(M));
  const int tid = threadIdx.x, nt = blockDim.x;
  const int tile = tile0 + (int)blockIdx.x, it = tile / n_etile, et = tile % n_etile;
  const int64_t i0 = (int64_t)it * TI, e0 = (int64_t)et * TE;
  const int m = tid / GT, t = tid % GT;  // this thread's mode
  const int ty = t / 8, tx = t % 8;      // rows ty + 8 r, samples tx + 8 j

  fill_phase_tables(S.ph, P, tid, nt);
  for (int k = tid; k < TE * P.n_det * REC; k += nt) {
    const int e = k / (P.n_det * REC), q = k % (P.n_det * REC);
    S.qs[e * QS_LD + q] = (e0 + e < P.n_ext) ? P.qx[(e0 + e) * P.n_det * REC + q] : 0.f;
  }
  for (int k = tid; k < TE; k += nt) S.lwe[k] = (P.lw_ext && e0 + k < P.n_ext) ? P.lw_ext[e0 + k] : 0.0;

  // (re, im) packed: one instruction adds both (each half rounds as fmaf does)
  uint64_t acc[8][4];
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[r][j] = 0ull;

  // one chunk of this mode's operands into stage s (zero-filled outside the
  // slice and the extrinsic samples)
  const int nch = (g.K + KC - 1) / KC;
  // (a thread's copies: 16 bytes of rows t / 4 + 16 p and of samples t / 8 + 8 p, p = 0..3;
  // pointers, strides and the in-range bits are set up once)
  const float *ap = g.A + ((int64_t)m * g.I_bank + P.i_base + i0 + t / 4) * g.Kpad + 4 * (t % 4);
  const float *bp = g.Bm + (((int64_t)m * P.n_ext + e0 + t / 8) * g.Kpad) * 2 + 4 * (t % 8);
  uint32_t inb = 0;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    inb |= (i0 + t / 4 + 16 * p < P.n_int) ? 1u << p : 0u;
    inb |= (e0 + t / 8 + 8 * p < P.n_ext) ? 16u << p : 0u;
  }
  const uint32_t sdst = smem_u32(stage + m * 2 * (A_W + B_W)) + 4 * (t / 4 * AS_LD + 4 * (t % 4));
  const uint32_t tdst = smem_u32(stage + m * 2 * (A_W + B_W) + A_W) + 4 * (t / 8 * BS_LD + 4 * (t % 8));
  const int astep = 16 * g.Kpad, bstep = 16 * g.Kpad;
  auto load_chunk = [&](int s) {
    const uint32_t so = s * (A_W + B_W) * 4;
#pragma unroll
    for (int p = 0; p < 4; ++p)
      cp_async16(sdst + so + p * 16 * AS_LD * 4, (inb >> p) & 1 ? ap + p * astep : g.A, (inb >> p) & 1);
#pragma unroll
    for (int p = 0; p < 4; ++p)
      cp_async16(tdst + so + p * 8 * BS_LD * 4, (inb >> (4 + p)) & 1 ? bp + p * bstep : g.Bm, (inb >> (4 + p)) & 1);
    cp_async_commit();
    ap += KC;
    bp += 2 * KC;
  };

  load_chunk(0);
#pragma unroll 1
  for (int c = 0; c < nch; ++c) {
    if (c + 1 < nch) {
      load_chunk((c + 1) & 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    named_bar_sync(1 + m, GT);
    const float *A = stage + (m * 2 + (c & 1)) * (A_W + B_W), *B = A + A_W;
#pragma unroll
    for (int kq = 0; kq < KC / 4; ++kq) {
      float4 a[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) a[r] = *reinterpret_cast<const float4 *>(A + (ty + 8 * r) * AS_LD + 4 * kq);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // (re, im) of k, k+1 and of k+2, k+3
        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(B + (tx + 8 * j) * BS_LD + 8 * kq);
        const ulonglong2 b1 = *reinterpret_cast<const ulonglong2 *>(B + (tx + 8 * j) * BS_LD + 8 * kq + 4);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          acc[r][j] = fma2(a[r].x, b0.x, acc[r][j]);
          acc[r][j] = fma2(a[r].y, b0.y, acc[r][j]);
          acc[r][j] = fma2(a[r].z, b1.x, acc[r][j]);
          acc[r][j] = fma2(a[r].w, b1.y, acc[r][j]);
        }
      }
    }
    named_bar_sync(1 + m, GT);
  }

  const float thr = tile_threshold(P);
  const bool store = (P.lnl_tile != nullptr);
  const float zs = P.z_scale / (P.g_scale ? *P.g_scale : 1.f);
  __syncthreads();  // every mode's operands consumed: the stages become Z
#pragma unroll
  for (int r = 0; r < 8; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      stage[z_at(2 * m, ty + 8 * r, tx + 8 * j)] = __uint_as_float((uint32_t)acc[r][j]) * zs;
      stage[z_at(2 * m + 1, ty + 8 * r, tx + 8 * j)] = __uint_as_float((uint32_t)(acc[r][j] >> 32)) * zs;
    }
  __syncthreads();

  // a warp per row, a lane per sample
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const bool pol = (P.n_pol == 2), ve = e0 + lane < P.n_ext;
  const double lwe = S.lwe[lane];
  Lse col, t1, t2;
  col.init();
  t1.init();
  t2.init();
  float best = -1.f;
  long long barg = 0x7fffffffffffffffLL;
  int np = 0;
#pragma unroll 1
  for (int rl = warp; rl < TI; rl += nw) {
    const int64_t i = i0 + rl, e = e0 + lane;
    if (i >= P.n_int) break;
    float x = -INFINITY;
    if (ve) {
      float Zr[MAXM], Zi[MAXM];
#pragma unroll
      for (int k = 0; k < MAXM; ++k) {
        const int mk = P.kmode[k];  // (zero where the bank has no such mode)
        Zr[k] = mk >= 0 ? stage[z_at(2 * mk, rl, lane)] : 0.f;
        Zi[k] = mk >= 0 ? stage[z_at(2 * mk + 1, rl, lane)] : 0.f;
      }
      if (P.gemm_only) {
        x = 0.f;
#pragma unroll
        for (int k = 0; k < MAXM; ++k) x += Zr[k] + Zi[k];
        t2.add(x);
        best = fmaxf(best, 0.f);
      } else {
        const float *mrow = P.mx + i * P.n_det * (pol ? REC_P : REC);
        float C0, Cr[3], Ci[3];
        if (pol) hh_coeffs_pol(mrow, &S.qs[lane * QS_LD], P, C0, Cr, Ci);
        else if (P.consec) hh_coeffs_by<true>([&](int k) { return __ldg(mrow + k); }, &S.qs[lane * QS_LD], P, C0, Cr, Ci);
        else hh_coeffs_by<false>([&](int k) { return __ldg(mrow + k); }, &S.qs[lane * QS_LD], P, C0, Cr, Ci);
        const PairRes pr = pair_eval(Zr, Zi, C0, Cr, Ci, thr, !store, P, S.ph);
        const float lw = (float)((P.lw_int ? P.lw_int[i] : 0.0) + lwe);
        x = pr.lsum + lw;
        t2.add(pr.lsum2 + 2.f * lw);
        np += pr.npass;
        const long long gi = (i * P.n_ext + e) * (long long)P.n_phi + pr.argo;
        if (pr.ml > best || (pr.ml == best && gi < barg)) { best = pr.ml; barg = gi; }
        if (store) {
          P.lnl_tile[i * P.n_ext + e] = pr.lsum - P.ln_nphi;
          P.ml_tile[i * P.n_ext + e] = pr.ml;
        }
      }
    }
    col.add(x);
    Lse row;
    row.init();
    row.add(x);
    warp_merge_lse(row);
    t1.merge(row.m, row.s);
    if (lane == 0) P.row_part[(int64_t)et * P.n_int + i] = make_float2(row.m, row.s);
  }
  S.col[warp][lane] = make_float2(col.m, col.s);
  warp_merge_lse(t2);
  warp_argmax(best, barg);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) np += __shfl_xor_sync(0xffffffffu, np, o);
  if (lane == 0) {
    S.w_m1[warp] = t1.m; S.w_s1[warp] = t1.s; S.w_m2[warp] = t2.m; S.w_s2[warp] = t2.s;
    S.w_ml[warp] = best; S.w_arg[warp] = barg; S.w_np[warp] = np;
  }
  __syncthreads();
  if (tid < TE) {
    Lse a;
    a.init();
    for (int q = 0; q < nw; ++q) a.merge(S.col[q][tid].x, S.col[q][tid].y);
    if (e0 + tid < P.n_ext) P.col_part[(int64_t)it * P.n_ext + e0 + tid] = make_float2(a.m, a.s);
  }
  if (tid == 32) {
    Lse a, b;
    a.init();
    b.init();
    float bv = -1.f;
    long long bi = 0x7fffffffffffffffLL;
    int n = 0;
    for (int q = 0; q < nw; ++q) {
      a.merge(S.w_m1[q], S.w_s1[q]);
      b.merge(S.w_m2[q], S.w_s2[q]);
      n += S.w_np[q];
      if (S.w_ml[q] > bv || (S.w_ml[q] == bv && S.w_arg[q] < bi)) { bv = S.w_ml[q]; bi = S.w_arg[q]; }
    }
    P.tile_part[tile] = make_float4(a.m, a.s, b.m, b.s);
    P.tile_ml[tile] = bv;
    P.tile_arg[tile] = bi;
    P.tile_npass[tile] = n;
    if (bv > 0.f && P.track_max) atomic_max_nonneg(P.ml_running, bv);
  }
}

// A block's cut is the maximum that it finds when its products are done, so what is in flight
// at first is marginalised whole: two blocks per SM with three or four modes, whose registers
// fill it.  Of one or two modes more blocks fit, up to all of a small event's (6,456 x 207, two
// modes, best ln L 36: every phase kept and ln Z 5e-4 higher).  Under a running cut the first two
// blocks per SM are then a launch of their own, and the others find its maximum; 8,192 x 1,024,
// B 512, two modes 2.20 ms (2.27 ms in one launch with twice the phases kept).
constexpr int PILOT_PER_SM = 2;

void launch_simt(const SimtArgs &g, const EpiParams &P, int n_sms, cudaStream_t st) {
  const int n_etile = (int)((P.n_ext + TE - 1) / TE);
  const int n = n_etile * (int)((P.n_int + TI - 1) / TI);
  const size_t smem = stage_bytes(P.n_modes) + sizeof(SimtSmem);
  cudaFuncSetAttribute(simt_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)(stage_bytes(MAXM) + sizeof(SimtSmem)));
  const int pilot = (P.track_max && P.n_modes <= 2) ? std::min(n, PILOT_PER_SM * n_sms) : 0;
  if (pilot > 0) simt_fused_kernel<<<pilot, GT * P.n_modes, smem, st>>>(g, P, 0, n_etile);
  if (n > pilot) simt_fused_kernel<<<n - pilot, GT * P.n_modes, smem, st>>>(g, P, pilot, n_etile);
}

}  // namespace dotpe
