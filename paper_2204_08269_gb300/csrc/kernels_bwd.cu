// Backward JTFS kernels (Sec. 5: reverse-ordered adjoints of the forward operators), FP32
// on CUDA cores.  Only the first-order scalogram U1 is checkpointed by the forward; the
// backward recomputes x-hat, U1-hat, Y_alpha and Z, and the first-order coefficients z.
//
//   k_uh_from_u1       : U1-hat = FFT of every checkpointed U1 row
//   k_joint_bwd_simt   : per (alpha, 32- or 16-column chunk, signal): for every spin pair, then
//                        phi_F: Z = W_c Y of both spins, g|Z| = adjoint of phi_T x phi_F pooling
//                        applied to g_S2, gZ = g|Z| Z / |Z| (0 at Z = 0), gY += W_c^H gZ
//   k_gy_spectra       : DFT of every gY row, in place (G rows of one rate per CTA)
//   k_second_order_bwd : per (lambda', signal): sum over alpha of the adjoint of the
//                        fold / psi_alpha product on those spectra, real part of the inverse
//                        of the row FFT, plus the adjoint of S1's pooling -> g_U1 row
//   k_stage1_bwd       : per (lambda, signal): recompute z, gz = g_U1 z / |z|, FFT -> gF
//   k_gxh              : g_x-hat[k] = sum_lambda psi_lambda[k] gF_lambda[k mod L_lambda], plus
//                        the spectrum of S0's adjoint
//   k_gx               : g_x = Re(inverse DFT of g_x-hat)
#include <mutex>

#include "stages.cuh"

namespace jtfs {
namespace {

__global__ void __launch_bounds__(kFftThreads)
k_uh_from_u1(DevPlan P, const float* __restrict__ u1, float2* __restrict__ uh) {
  pdl_enter();
  extern __shared__ float2 sm[];
  const int lam = blockIdx.x, b = blockIdx.y;
  const Row1 R = P.rows1[lam];
  const float* ub = u1 + (size_t)b * P.u1_len + R.off_u;
  for (int m = threadIdx.x; m < R.L; m += blockDim.x)
    sm[fft_pos(bitrev(m, R.logL), R.logL)] = make_float2(ub[m], 0.f);
  __syncthreads();
  fft_dit_rows_r16<-1>(sm, R.logL, 1, twl_for(P, R.logL));
  float2* hb = uh + (size_t)b * P.uh_len + R.off_uh;
  for (int k = threadIdx.x; k < (R.L >> 1); k += blockDim.x) hb[k] = sm[fft_pos(k, R.logL)];
}

// ---------------------------------------------------------------------------------------
// Joint backward on CUDA cores (plain FP32 plans, and the rates past the tensor-core form's
// lambda' range).  One CTA per (alpha, NC-column chunk, signal); it walks the spin pairs and then
// the phi_F channel, whose filters W = Wr + i Wi serve both spins (the spin-down filter is the
// conjugate of the spin-up one): Z_up = W Y and Z_down = conj(W) Y from one h per (row, lambda').
// Each is summed product by product.  As P1 -/+ P2 of the real products Wr Y and Wi Y they take
// half the FMAs, but a weak spin is then a difference of two sums of the strong one's size, and
// gZ = g Z / |Z| weighs its cells like all others (a spin 54 times weaker, 151 rows: gradient
// error 8.3e-7 so, 3.4e-6 as the difference).
// With S = gZ_up + gZ_down, T = (Im gZ_up - Im gZ_down) + i (Re gZ_down - Re gZ_up) the adjoint
// is gY += Wr^T S + Wi^T T (phi_F: Wi = 0, T unused).  Both products are bound by their FMAs: a
// thread owns 4 consecutive rows x 4 columns, W is Toeplitz, so consecutive k shift a 4-entry
// window of h by one and a step loads one h and four columns for 64 packed FMAs (32 in the
// adjoint).  The gY accumulators rest in shared memory while the Z product holds the registers.
// Eight rows to a thread need fewer loads a product, but twice the registers and half the
// threads, which short banks and many frames miss in the pooling adjoint.  Contraction backward in
// plain FP32, 8 -> 4 rows (8 rows with Z as a difference in brackets): N = 2^12, n1 = 34, B = 1,
// 64 frames 620 -> 265 us (572); N = 2^16, n1 = 151, B = 8 36.0 -> 22.8 ms (28.3).  With the five
// lowest rates alone here (B = 16, N = 2^17, n1 = 167) 5.84 -> 5.25 ms (5.11).
constexpr int kJR = 4;        // rows (or lambda') of a thread
constexpr int kJC = 4;        // columns of a thread
constexpr int kJT = 512;      // most threads (32 columns fit the shared memory up to 220 rows, 448)

struct JointBwdLayout {       // float offsets in shared memory
  int rows, threads, y, st, gacc, h, g1, wt, total;
};

__host__ __device__ inline JointBwdLayout joint_bwd_layout(int n1, int nt, int nc) {
  JointBwdLayout s;
  s.rows = (n1 + kJR - 1) / kJR * kJR;
  s.threads = (s.rows / kJR * (nc / kJC) + 31) / 32 * 32;
  s.st = 0;                                   // [rows][nc] (S, T)
  s.y = s.st + s.rows * nc * 4;               // [rows][nc] Y
  s.gacc = s.y + s.rows * nc * 2;             // [2 kJR kJC][threads]
  s.wt = s.gacc + 2 * kJR * kJC * s.threads;  // [nt][nc]
  s.h = s.wt + nt * nc;                       // h[d], -rows <= d < rows
  s.g1 = s.h + 4 * s.rows;                    // [2 spins][n1][nt]
  s.total = s.g1 + 2 * n1 * nt;
  return s;
}

template <int NC>
__global__ void __launch_bounds__(kJT)
k_joint_bwd_simt(DevPlan P, const int2* __restrict__ items, const float2* __restrict__ y,
                 const float* __restrict__ gs2, float2* __restrict__ gy) {
  pdl_enter();
  extern __shared__ float4 smraw[];
  float* smf = reinterpret_cast<float*>(smraw);
  const int2 it = items[blockIdx.x];
  const int a = it.x, n0 = it.y + (int)blockIdx.z * NC, b = blockIdx.y;
  const Rate2 A = P.rates2[a];
  if (n0 >= A.L) return;
  const int n1 = P.n1, nt = P.n_t, K = A.K, l0 = A.lam_min, nfm = P.N_fr - 1;
  const JointBwdLayout lay = joint_bwd_layout(n1, nt, NC);
  const int Kp = (K + kJR - 1) / kJR * kJR, Rp = lay.rows;
  float4* st = reinterpret_cast<float4*>(smf + lay.st);
  float2* yt = reinterpret_cast<float2*>(smf + lay.y);
  float* gacc = smf + lay.gacc;
  float* wt = smf + lay.wt;
  float2* sh = reinterpret_cast<float2*>(smf + lay.h) + Rp;   // sh[d], -Rp <= d < Rp
  float* g1 = smf + lay.g1;
  const int tid = threadIdx.x, nthr = blockDim.x;
  const float2* ya = y + (size_t)b * P.y_len + A.off_y;
  for (int i = tid; i < Kp * NC; i += nthr) {
    const int k = i / NC, col = i % NC;
    yt[i] = (k < K && n0 + col < A.L) ? ya[(size_t)k * A.L + n0 + col] : make_float2(0.f, 0.f);
  }
  for (int i = tid; i < nt * NC; i += nthr) {
    const int t = i / NC, n = n0 + i % NC;
    wt[i] = (n < A.L) ? __ldg(&P.phiT[(t * P.T - n * A.s) & (P.N - 1)]) * (float)A.s : 0.f;
  }
  // the products' threads; the others only stage
  const int na = lay.threads;
  if (tid < na)
    for (int i = 0; i < 2 * kJR * kJC; ++i) gacc[i * na + tid] = 0.f;
  // columns col0 + CS j: neighbouring lanes read neighbouring columns
  constexpr int CS = NC / kJC;
  const int col0 = tid % CS, r0 = tid / CS * kJR;
  const bool has_rows = r0 < Rp, has_k = r0 < Kp;

  for (int p = 0; p <= P.n_fr; ++p) {
    const bool pair = p < P.n_fr;               // a spin pair, or the phi_F channel
    const int c = pair ? p : 2 * P.n_fr;
    __syncthreads();
    for (int i = tid; i < 2 * Rp; i += nthr)
      sh[i - Rp] = P.h[(size_t)c * P.N_fr + ((i - Rp) & nfm)];
    for (int i = tid; i < (pair ? 2 : 1) * n1 * nt; i += nthr) {
      const int d = i >= n1 * nt ? 1 : 0, j = i - d * n1 * nt;
      const float* g = gs2 + (size_t)b * P.s2_stride +
                       ((size_t)a * P.C + c + d * P.n_fr) * P.n_lo * nt;
      float v;
      if (P.average_fr) {
        const int r = j / nt, t = j - r * nt;
        v = 0.f;
        for (int lo = 0; lo < P.n_lo; ++lo)
          v += __ldg(&P.phiF[(lo * P.s_F - r) & nfm]) * __ldg(&g[lo * nt + t]);
      } else {
        v = g[j];
      }
      g1[i] = v;
    }
    __syncthreads();
    // Z of both spins, rows r0 + i, columns col0 + CS j
    float2 zu[kJR][kJC], zd[kJR][kJC];
#pragma unroll
    for (int i = 0; i < kJR; ++i)
#pragma unroll
      for (int j = 0; j < kJC; ++j) zu[i][j] = zd[i][j] = make_float2(0.f, 0.f);
    if (has_rows) {
      // row i's filter entry at step k is h[r0 + i - k - l0], in slot (i - k) mod kJR
      float2 win[kJR];
#pragma unroll
      for (int i = 1; i < kJR; ++i) win[i] = sh[r0 + i - l0];
      for (int k0 = 0; k0 < Kp; k0 += kJR) {
#pragma unroll
        for (int e = 0; e < kJR; ++e) {
          const int k = k0 + e;
          win[(kJR - e) & (kJR - 1)] = sh[max(r0 - k - l0, -Rp)];
          float2 yv[kJC], yi[kJC], yc[kJC];   // y, i y, -i y
#pragma unroll
          for (int j = 0; j < kJC; ++j) {
            yv[j] = yt[k * NC + col0 + CS * j];
            yi[j] = make_float2(-yv[j].y, yv[j].x);
            yc[j] = make_float2(yv[j].y, -yv[j].x);
          }
#pragma unroll
          for (int i = 0; i < kJR; ++i) {
            const float2 w = win[(i - e + kJR) & (kJR - 1)];
#pragma unroll
            for (int j = 0; j < kJC; ++j) {
              zu[i][j] = __ffma2_rn(make_float2(w.x, w.x), yv[j], zu[i][j]);
              zu[i][j] = __ffma2_rn(make_float2(w.y, w.y), yi[j], zu[i][j]);
              zd[i][j] = __ffma2_rn(make_float2(w.x, w.x), yv[j], zd[i][j]);
              zd[i][j] = __ffma2_rn(make_float2(w.y, w.y), yc[j], zd[i][j]);
            }
          }
        }
      }
      // g|Z| of both spins from the pooling adjoint, gZ = g|Z| Z / |Z|, then S and T
#pragma unroll
      for (int i = 0; i < kJR; ++i) {
        const int r = r0 + i;
        float gu[kJC] = {0.f, 0.f, 0.f, 0.f}, gd[kJC] = {0.f, 0.f, 0.f, 0.f};
        if (r < n1) {
          const float *gur = g1 + r * nt, *gdr = gur + n1 * nt;
          for (int t = 0; t < nt; ++t) {
            const float u = gur[t], d = pair ? gdr[t] : 0.f;
#pragma unroll
            for (int j = 0; j < kJC; ++j) {
              const float wv = wt[t * NC + col0 + CS * j];
              gu[j] = fmaf(u, wv, gu[j]);
              gd[j] = fmaf(d, wv, gd[j]);
            }
          }
        }
#pragma unroll
        for (int j = 0; j < kJC; ++j) {
          const float2 u = zu[i][j], d = zd[i][j];
          const float mu = sqrtf(u.x * u.x + u.y * u.y), md = sqrtf(d.x * d.x + d.y * d.y);
          const float fu = mu > 0.f ? gu[j] / mu : 0.f, fd = md > 0.f ? gd[j] / md : 0.f;
          const float2 zgu = make_float2(u.x * fu, u.y * fu), zgd = make_float2(d.x * fd, d.y * fd);
          st[r * NC + col0 + CS * j] =
              pair ? make_float4(zgu.x + zgd.x, zgu.y + zgd.y, zgu.y - zgd.y, zgd.x - zgu.x)
                   : make_float4(zgu.x, zgu.y, 0.f, 0.f);
        }
      }
    }
    __syncthreads();
    if (has_k) {
      // gY[k][col] += sum_r Wr[r][k] S[r][col] + Wi[r][k] T[r][col], k = r0 + i: the filter entry
      // h[r - k - l0] is in slot (r - i) mod kJR
      float2 acc[kJR][kJC];
#pragma unroll
      for (int i = 0; i < kJR; ++i)
#pragma unroll
        for (int j = 0; j < kJC; ++j)
          acc[i][j] = make_float2(gacc[2 * (i * kJC + j) * na + tid],
                                  gacc[(2 * (i * kJC + j) + 1) * na + tid]);
      float2 win[kJR];
#pragma unroll
      for (int i = 1; i < kJR; ++i) win[kJR - i] = sh[max(-(r0 + i) - l0, -Rp)];
      for (int rr = 0; rr < Rp; rr += kJR) {
#pragma unroll
        for (int e = 0; e < kJR; ++e) {
          const int r = rr + e;
          win[e] = sh[max(r - r0 - l0, -Rp)];
#pragma unroll
          for (int j = 0; j < kJC; ++j) {
            const float4 v = st[r * NC + col0 + CS * j];
#pragma unroll
            for (int i = 0; i < kJR; ++i) {
              const float2 w = win[(e - i + kJR) & (kJR - 1)];
              acc[i][j] = __ffma2_rn(make_float2(w.x, w.x), make_float2(v.x, v.y), acc[i][j]);
              acc[i][j] = __ffma2_rn(make_float2(w.y, w.y), make_float2(v.z, v.w), acc[i][j]);
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kJR; ++i)
#pragma unroll
        for (int j = 0; j < kJC; ++j) {
          gacc[2 * (i * kJC + j) * na + tid] = acc[i][j].x;
          gacc[(2 * (i * kJC + j) + 1) * na + tid] = acc[i][j].y;
        }
    }
  }
  float2* go = gy + (size_t)b * P.y_len + A.off_y;
  if (has_k) {
#pragma unroll
    for (int i = 0; i < kJR; ++i)
#pragma unroll
      for (int j = 0; j < kJC; ++j) {
        const int k = r0 + i, n = n0 + col0 + CS * j;
        if (k < K && n < A.L)
          go[(size_t)k * A.L + n] = make_float2(gacc[2 * (i * kJC + j) * na + tid],
                                                gacc[(2 * (i * kJC + j) + 1) * na + tid]);
      }
  }
}

// Parts 1, 2, ... of the gY rows of the rates [a0, a1) (the tensor-core backward of small batches).
struct GyParts {
  const float2* gy2;
  long long sub_off, sub_len;
  int a0, a1, parts;
};

// Spectra of the gY rows, in place: G rows of one rate per CTA (the Y producer's row items),
// batched forward FFT (padded radix-16 passes, bit-reversed loads), written back in natural
// order.
__global__ void __launch_bounds__(kRowBound)
k_gy_spectra(DevPlan P, const int4* __restrict__ items, float2* __restrict__ gy, GyParts gp) {
  pdl_enter();
  extern __shared__ float2 sm[];
  const int4 it = items[blockIdx.x];
  const int a = it.x, lam0 = it.y, G = it.z, b = blockIdx.y;
  const Rate2 A = P.rates2[a];
  const int L = A.L, logL = A.logL;
  float2* g = gy + (size_t)b * P.y_len + A.off_y + (size_t)(lam0 - A.lam_min) * L;
  const int total = G * L, step = blockDim.x;
  // two samples per 16-byte access where the block's rows start 16-byte aligned (rows hold an
  // even number of samples), else one
  const bool pair = L >= 2 && ((uintptr_t)g & 15) == 0;
  if (gp.parts > 1 && a >= gp.a0 && a < gp.a1) {
    // rows whose gY was summed in parts
    const float2* g2 = gp.gy2 + (size_t)b * P.y_len + (A.off_y - gp.sub_off) + (size_t)(lam0 - A.lam_min) * L;
    for (int idx = threadIdx.x; idx < total; idx += step) {
      float2 v = g[idx];
      for (int q = 1; q < gp.parts; ++q) v = cadd(v, g2[(q - 1) * gp.sub_len + idx]);
      sm[fft_pos(((idx >> logL) << logL) + bitrev(idx & (L - 1), logL), logL)] = v;
    }
  } else if (pair) {
    // four 16-byte loads in flight per thread before their shared-memory stores
    const float4* g4 = reinterpret_cast<const float4*>(g);
    const int total2 = total >> 1;
    for (int base = threadIdx.x; base < total2; base += 4 * step) {
      float4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i2 = base + q * step;
        v[q] = i2 < total2 ? g4[i2] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int idx = 2 * (base + q * step);
        if (idx < total) {
          const int r0 = (idx >> logL) << logL, k = idx & (L - 1);
          sm[fft_pos(r0 + bitrev(k, logL), logL)] = make_float2(v[q].x, v[q].y);
          sm[fft_pos(r0 + bitrev(k + 1, logL), logL)] = make_float2(v[q].z, v[q].w);
        }
      }
    }
  } else {
    // eight loads in flight per thread before their shared-memory stores
    for (int base = threadIdx.x; base < total; base += 8 * step) {
      float2 v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int idx = base + q * step;
        v[q] = idx < total ? g[idx] : make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int idx = base + q * step;
        if (idx < total) sm[fft_pos(((idx >> logL) << logL) + bitrev(idx & (L - 1), logL), logL)] = v[q];
      }
    }
  }
  __syncthreads();
  fft_dit_rows_r16<-1>(sm, logL, G, twl_for(P, logL));
  if (pair) {
    float4* g4 = reinterpret_cast<float4*>(g);
    for (int i2 = threadIdx.x; i2 < total >> 1; i2 += blockDim.x) {
      const float2 a = sm[fft_pos(2 * i2, logL)], c = sm[fft_pos(2 * i2 + 1, logL)];
      g4[i2] = make_float4(a.x, a.y, c.x, c.y);
    }
  } else {
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) g[idx] = sm[fft_pos(idx, logL)];
  }
}

// shared memory of k_second_order_bwd: the padded row, then its rate table
static size_t sob_table(const jtfs_plan* p) { return ((size_t)p->L1max * 17 / 2 + 15) & ~(size_t)15; }
static size_t sob_smem(const jtfs_plan* p) {
  return sob_table(p) + (size_t)(p->n2 + 3) * 16 + (size_t)(p->n2 / 4 + 2) * 4;
}

// g_U1 row lambda': sum over rates alpha of the adjoint of psi2 (the gY row's spectrum / Lr
// times psi-hat_alpha on the row's positive bins), then Re of the inverse row DFT, plus S1's
// adjoint.
template <int TH>   // threads: three 256-thread blocks per SM, or one of 512
__global__ void __launch_bounds__(TH, TH == kRowLaunch ? 3 : 1)
k_second_order_bwd(DevPlan P, int table, const float2* __restrict__ gys,
                   const float* __restrict__ gs1, float* __restrict__ gu1) {
  pdl_enter();
  extern __shared__ float2 sm[];
  const int lam = blockIdx.x, b = blockIdx.y;
  const Row1 R = P.rows1[lam];
  const int half = R.L >> 1;
  float2* tmp = sm;                // [L] padded
  const float invLr = 1.f / (float)R.L;
  const float* g1 = gs1 ? gs1 + ((size_t)b * P.n1 + lam) * P.n_t : nullptr;
  const float2* gyb = gys + (size_t)b * P.y_len;
  // the row's rates in increasing alpha: offset of its gY spectrum, L_alpha - 1, support end and
  // offset in psi2, then three empty entries; s_end: past it no rate from this group of four on
  // has support.  Supports shrink with alpha, so most bins stop after the first group.  Rate
  // records read per bin and all rates visited took the kernel and the gY spectra before it 1.05 ms,
  // this 0.93 ms (B = 64, N = 2^16).
  int4* s_rate = reinterpret_cast<int4*>(reinterpret_cast<char*>(sm) + table);
  int* s_end = reinterpret_cast<int*>(s_rate + P.n2 + 3);
  if (threadIdx.x == 0) {
    int n = 0;
    for (int a = 0; a < P.n2; ++a) {
      const Rate2 A = P.rates2[a];
      if (A.s != 0 && lam >= A.lam_min)
        s_rate[n++] = make_int4((int)(A.off_y + (long long)(lam - A.lam_min) * A.L), A.L - 1, A.k2e, a * P.K2max);
    }
    for (int i = n; i < n + 3; ++i) s_rate[i] = make_int4(0, 0, 0, 0);
    int end = 0;
    s_end[(n + 3) >> 2] = 0;
    for (int g = ((n + 3) >> 2) - 1; g >= 0; --g) {
      for (int i = 4 * g; i < min(4 * g + 4, n); ++i) end = max(end, s_rate[i].z);
      s_end[g] = end;
    }
  }
  __syncthreads();
  // guh[k] for k <= half, built in registers per bin and stored bit-reversed; g_U1 is the real
  // part of its inverse DFT.  Two terms:
  //  - the rates' adjoint: the gY row spectra / Lr times psi-hat_alpha on bins 0 < k < half;
  //  - S1's adjoint g[m] = s sum_t phi_T[t T - m s] g_S1[t], whose length-L DFT is
  //    G[k mod n_t] sum_r phi-hat[k + r L] (the spikes of g_S1 sit tau = T / s apart and
  //    phi_T at stride s aliases phi-hat): nonzero only where phi-hat is, taken one-sided
  //    (bins 0 and L / 2 once, the others twice), with phi-hat on the bins phi_T is built from.
  for (int k = threadIdx.x; k < R.L; k += blockDim.x) {
    float2 acc = make_float2(0.f, 0.f);
    if (k >= 1 && k < half) {
      // the rates in groups of four whose loads are in flight together, summed in increasing alpha
      // (a rate outside its support adds 0 * 0)
      for (int i0 = 0; k < s_end[i0 >> 2]; i0 += 4) {
        float2 v[4];
        float f[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int4 r = s_rate[i0 + q];
          v[q] = make_float2(0.f, 0.f);
          f[q] = 0.f;
          if (k < r.z) {
            v[q] = gyb[r.x + (k & r.y)];
            f[q] = __ldg(&P.psi2[r.w + k]) * invLr;
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          acc.x += v[q].x * f[q];
          acc.y += v[q].y * f[q];
        }
      }
    }
    if (g1 && k <= half) {
      // signed representatives k + r L of the N-grid bins: r >= 0, then r < 0
      // (|k + r L| = |r| L - k, below the Nyquist bin, which the first loop holds)
      float ph = 0.f;
      const int qneg = min(P.phiT_kmax, (P.N >> 1) - 1);
      for (int q = k; q <= P.phiT_kmax; q += R.L) ph += __ldg(&P.phiThat[q]);
      for (int q = R.L - k; q <= qneg; q += R.L) ph += __ldg(&P.phiThat[q]);
      if (ph != 0.f) {
        const int f = k & (P.n_t - 1);
        float2 G = make_float2(0.f, 0.f);
        for (int t = 0; t < P.n_t; ++t) {   // G[f] = sum_t g_S1[t] exp(-2 pi i f t / n_t)
          float sn, cs;
          sincospif(2.f * (float)((f * t) & (P.n_t - 1)) / (float)P.n_t, &sn, &cs);
          G.x += g1[t] * cs;
          G.y -= g1[t] * sn;
        }
        const float c = ((k == 0 || k == half) ? 1.f : 2.f) * invLr * ph;
        acc.x += c * G.x;
        acc.y += c * G.y;
      }
    }
    tmp[fft_pos(bitrev(k, R.logL), R.logL)] = acc;
  }
  __syncthreads();
  fft_dit_rows_r16<+1>(tmp, R.logL, 1, twl_for(P, R.logL));
  float* out = gu1 + (size_t)b * P.u1_len + R.off_u;
  for (int m = threadIdx.x; m < R.L; m += blockDim.x) out[m] = tmp[fft_pos(m, R.logL)].x;
}

template <int TH>   // threads: three 256-thread blocks per SM, or one of 512
__global__ void __launch_bounds__(TH, TH == kRowLaunch ? 3 : 1)
k_stage1_bwd(DevPlan P, const float2* __restrict__ xh, const float* __restrict__ gu1,
             float2* __restrict__ gf) {
  pdl_enter();
  extern __shared__ float2 sm[];
  const int lam = blockIdx.x, b = blockIdx.y;
  const Row1 R = P.rows1[lam];
  fold_first_order(P, R, xh + (size_t)b * (P.N >> 1), sm);
  __syncthreads();
  fft_dit_rows_r16<+1>(sm, R.logL, 1, twl_for(P, R.logL));
  // gz = g_U1 z / |z| (0 at z = 0), stored bit-reversed for the forward FFT: every thread
  // handles the pairs (m, bitrev(m)) with m <= bitrev(m), so the permutation is in place
  const float* g = gu1 + (size_t)b * P.u1_len + R.off_u;
  for (int m = threadIdx.x; m < R.L; m += blockDim.x) {
    const int r = bitrev(m, R.logL);
    if (m > r) continue;
    const float2 zm = sm[fft_pos(m, R.logL)], zr = sm[fft_pos(r, R.logL)];   // N * z
    const float am = hypotf(zm.x, zm.y), ar = hypotf(zr.x, zr.y);
    const float fm = (am > 0.f) ? g[m] / am : 0.f, fr = (ar > 0.f) ? g[r] / ar : 0.f;
    sm[fft_pos(r, R.logL)] = make_float2(zm.x * fm, zm.y * fm);
    sm[fft_pos(m, R.logL)] = make_float2(zr.x * fr, zr.y * fr);
  }
  __syncthreads();
  fft_dit_rows_r16<-1>(sm, R.logL, 1, twl_for(P, R.logL));
  const float invN = 1.f / (float)P.N;
  float2* out = gf + (size_t)b * P.u1_len + R.off_u;
  for (int k = threadIdx.x; k < R.L; k += blockDim.x) {
    const float2 v = sm[fft_pos(k, R.logL)];
    out[k] = make_float2(v.x * invN, v.y * invN);
  }
}

// S0's adjoint sum_t phi_T[(tT - n) mod N] g_S0[t] has the length-N DFT
// DFT(g_S0)[k mod n_t] phi-hat[k] (spikes T apart), nonzero for k <= phiT_kmax: it is added
// to those bins of the one-sided g_x spectrum (bin 0 once, the others twice, / N).  When
// phi-hat reaches the Nyquist bin (T <= 2), k_gx adds it in the time domain instead.
__global__ void k_gxh(DevPlan P, const float2* __restrict__ gf, const float* __restrict__ gs0,
                      float2* __restrict__ gxh) {
  pdl_enter();
  const int b = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int half = P.N >> 1;
  const int2 rng = P.gx_lam[blockIdx.x];
  float2 acc = make_float2(0.f, 0.f);
  if (k < half) {
    const float2* gb = gf + (size_t)b * P.u1_len;
    for (int lam = rng.x; lam < rng.y; ++lam) {
      const Row1 R = P.rows1[lam];
      const int i = k - R.ks;
      if (i >= 0 && i < R.kl) {
        const float f = __ldg(&P.psi1[R.off_v + i]);
        const float2 v = gb[R.off_u + (k & (R.L - 1))];
        acc.x += f * v.x;
        acc.y += f * v.y;
      }
    }
    if (gs0 && k <= P.phiT_kmax && P.phiT_kmax < half) {
      const float* g0 = gs0 + (size_t)b * P.n_t;
      const int f = k & (P.n_t - 1);
      float2 G = make_float2(0.f, 0.f);
      for (int t = 0; t < P.n_t; ++t) {
        float sn, cs;
        sincospif(2.f * (float)((f * t) & (P.n_t - 1)) / (float)P.n_t, &sn, &cs);
        G.x += g0[t] * cs;
        G.y -= g0[t] * sn;
      }
      const float c = (k == 0 ? 1.f : 2.f) * __ldg(&P.phiThat[k]) / (float)P.N;
      acc.x += c * G.x;
      acc.y += c * G.y;
    }
    gxh[(size_t)b * half + k] = acc;
  }
}

// g_x[r + D m] = Re(sum_k' e^{2 pi i k' m / M} sum_q H[k' + q M] e^{2 pi i (k' + q M) r / N})
// (S0's adjoint is already in H unless phi-hat reaches the Nyquist bin)
template <int TH>   // threads: two 512-thread blocks per SM, or one of 1024
__global__ void __launch_bounds__(TH, TH == kFftThreads ? 2 : 1)
k_gx(DevPlan P, const float2* __restrict__ gxh, const float* __restrict__ gs0, float* __restrict__ gx) {
  pdl_enter();
  extern __shared__ float2 sm[];
  const int r = blockIdx.x, b = blockIdx.y;
  const int half = P.N >> 1;
  const int step = P.TW / P.N;
  const float2* H = gxh + (size_t)b * half;
  for (int kp = threadIdx.x; kp < P.M; kp += blockDim.x) {
    float2 acc = make_float2(0.f, 0.f);
    for (int k = kp; k < half; k += P.M) {
      const float2 v = H[k];
      const int idx = (int)(((long long)k * r) & (P.N - 1)) * step;
      float2 w = __ldg(&P.tw[idx]);
      w.y = -w.y;
      acc.x += v.x * w.x - v.y * w.y;
      acc.y += v.x * w.y + v.y * w.x;
    }
    sm[fft_pos(bitrev(kp, P.logM), P.logM)] = acc;
  }
  __syncthreads();
  fft_dit_rows_r16<+1>(sm, P.logM, 1, twl_for(P, P.logM));
  const float* g0 = (gs0 && P.phiT_kmax >= half) ? gs0 + (size_t)b * P.n_t : nullptr;
  float* out = gx + (size_t)b * P.N;
  for (int m = threadIdx.x; m < P.M; m += blockDim.x) {
    const int n = r + P.D * m;
    float v = sm[fft_pos(m, P.logM)].x;
    if (g0)
      for (int t = 0; t < P.n_t; ++t) v += __ldg(&P.phiT[(t * P.T - n) & (P.N - 1)]) * g0[t];
    out[n] = v;
  }
}

// Time scattering (Scattering1D) backward of the second order: Y_alpha rows recomputed in
// shared memory as in the forward, then gY = g_|Y| Y / |Y| (0 where Y = 0) with
// g_|Y|[m] = sum_t s_alpha phi_T[(t T - m s_alpha) mod N] g_S2t[t], written in the layout of the
// transform's gY so that the second-order adjoint that follows is shared.  A thread takes the FB
// samples m = (q0 + j) tau + rho, j < FB, of one row (tau = T / s_alpha): their weights for
// consecutive frames are a sliding window over the rate's weights (DevPlan.poolw), so a frame
// costs one weight and one cotangent for FB products.  B = 32, N = 2^16, 167 rows, 32 frames:
// 5.48 -> 0.55 ms (every product gathered its own weight from phi_T at the rate's stride before).
template <int FB>
__global__ void __launch_bounds__(kRowBound)
k_scat1d_bwd_rows(DevPlan P, const int4* __restrict__ items, const float2* __restrict__ uh,
                  const float* __restrict__ gs2t, float2* __restrict__ gy) {
  pdl_enter();
  extern __shared__ float2 sm[];
  __shared__ int s_off[kMaxRowsPerItem], s_kend[kMaxRowsPerItem];
  __shared__ float s_inv[kMaxRowsPerItem];
  const int4 it = items[blockIdx.x];
  const int a = it.x, lam0 = it.y, G = it.z, b = blockIdx.y;
  const Rate2 A = P.rates2[a];
  const int L = A.L, logL = A.logL, nt = P.n_t, tau = P.T / A.s, logtau = 31 - __clz(tau);
  second_order_rows_ifft(P, A, a, lam0, G, uh + (size_t)b * P.uh_len, sm, s_off, s_kend, s_inv);
  __syncthreads();
  const float* g = gs2t + (((size_t)b * P.n2 + a) * P.n1 + lam0) * nt;
  const float* w = P.poolw + A.off_pw;
  float2* out = gy + (size_t)b * P.y_len + A.off_y + (size_t)(lam0 - A.lam_min) * L;
  constexpr int kLogFB = FB == 8 ? 3 : (FB == 4 ? 2 : FB - 1);
  const int logpr = logL - kLogFB, per_row = 1 << logpr;
  for (int i = threadIdx.x; i < G * per_row; i += blockDim.x) {
    const int r = i >> logpr, rest = i & (per_row - 1);
    const int rho = rest & (tau - 1), q0 = (rest >> logtau) * FB;
    const float* gr = g + r * nt;
    // slot (j - t) mod FB holds the weight of sample j in frame t
    float win[FB], ga[FB];
#pragma unroll
    for (int j = 0; j < FB; ++j) {
      ga[j] = 0.f;
      win[j] = j ? __ldg(&w[(q0 + j) * tau + rho]) : 0.f;
    }
    for (int t0 = 0; t0 < nt; t0 += FB) {
#pragma unroll
      for (int e = 0; e < FB; ++e) {
        const int t = t0 + e;
        win[(FB - e) & (FB - 1)] = __ldg(&w[((q0 - t) & (nt - 1)) * tau + rho]);
        const float gt = __ldg(&gr[t]);
#pragma unroll
        for (int j = 0; j < FB; ++j) ga[j] = fmaf(win[(j - e + FB) & (FB - 1)], gt, ga[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < FB; ++j) {
      const int idx = (r << logL) + (q0 + j) * tau + rho;
      const float2 v = sm[fft_pos(idx, logL)];
      const float mag = sqrtf(v.x * v.x + v.y * v.y);
      const float sc = mag > 0.f ? ga[j] / mag : 0.f;
      out[idx] = make_float2(v.x * sc, v.y * sc);
    }
  }
}

// cudaFuncSetAttribute acts on the current device only, so the raised shared-memory limits
// are recorded per device (the plan's device is current in every call that launches).
std::mutex g_attrs_mu;
bool g_attrs_set[256] = {};

jtfs_status set_attrs(const jtfs_plan* p) {
  if (p->device < 0 || p->device >= 256) {
    set_error("device ordinal out of range");
    return JTFS_ERR_INVALID_ARG;
  }
  std::lock_guard<std::mutex> lk(g_attrs_mu);
  if (g_attrs_set[p->device]) return JTFS_OK;
  const int big = 227 * 1024;
  const void* fns[] = {(const void*)k_uh_from_u1, (const void*)k_joint_bwd_simt<32>,
                       (const void*)k_joint_bwd_simt<16>,
                       (const void*)k_second_order_bwd<kRowLaunch>,
                       (const void*)k_second_order_bwd<2 * kRowLaunch>,
                       (const void*)k_stage1_bwd<kRowLaunch>, (const void*)k_stage1_bwd<2 * kRowLaunch>,
                       (const void*)k_gx<kFftThreads>, (const void*)k_gx<2 * kFftThreads>,
                       (const void*)k_xfft_sub<kFftThreads>, (const void*)k_xfft_sub<2 * kFftThreads>};
  for (const void* f : fns) {
    jtfs_status st = cuda_check(
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, big), "attr");
    if (st != JTFS_OK) return st;
  }
  // the row producer holds at most 2^14 complex samples (padded one per 16) next to its
  // static row tables
  for (const void* f : {(const void*)k_second_order_rows<0>, (const void*)k_second_order_rows<1>,
                        (const void*)k_gy_spectra, (const void*)k_scat1d_bwd_rows<1>,
                        (const void*)k_scat1d_bwd_rows<2>, (const void*)k_scat1d_bwd_rows<4>,
                        (const void*)k_scat1d_bwd_rows<8>}) {
    jtfs_status st = cuda_check(
        cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 140 * 1024), "attr");
    if (st != JTFS_OK) return st;
  }
  g_attrs_set[p->device] = true;
  return JTFS_OK;
}

}  // namespace

// The CUDA-core joint backward over 32-column items: 32 columns at a time where the shared memory
// holds them (every configuration but those with many rows and frames), else 16.  Where the blocks
// do not fill the SMs once they take at least 256 threads, whose surplus only stages: N = 512,
// n1 = 9, 32 frames, B = 1 137 -> 107 us.
static void launch_joint_bwd_simt(const jtfs_plan* p, int n_items, const int* items, int B,
                                  const float2* y, const float* gs2, float2* gy, cudaStream_t st) {
  const JointBwdLayout w = joint_bwd_layout(p->n1, p->n_t, 32);
  const bool wide = (size_t)w.total * 4 <= 227 * 1024;
  const JointBwdLayout l = wide ? w : joint_bwd_layout(p->n1, p->n_t, 16);
  auto* kernel = wide ? k_joint_bwd_simt<32> : k_joint_bwd_simt<16>;
  const int threads = few_blocks(p, (long long)n_items * B) ? std::max(l.threads, 256) : l.threads;
  launch_spread(kernel, dim3((unsigned)n_items, B, wide ? 1 : 2), threads, (size_t)l.total * 4, st,
                p->dp, reinterpret_cast<const int2*>(items), y, gs2, gy);
}

static void launch_second_order_bwd(const jtfs_plan* p, int B, const float2* gys, const float* gs1,
                                    float* gu1, cudaStream_t st) {
  const bool few = few_blocks(p, (long long)p->n1 * B);
  launch_pdl(few ? k_second_order_bwd<2 * kRowLaunch> : k_second_order_bwd<kRowLaunch>, dim3(p->n1, B),
             few ? 2 * kRowLaunch : kRowLaunch, sob_smem(p), st, p->dp, (int)sob_table(p), gys, gs1, gu1);
}

static void launch_stage1_bwd(const jtfs_plan* p, int B, const float2* xh, const float* gu1, float2* gf,
                              cudaStream_t st) {
  const bool few = few_blocks(p, (long long)p->n1 * B);
  launch_pdl(few ? k_stage1_bwd<2 * kRowLaunch> : k_stage1_bwd<kRowLaunch>, dim3(p->n1, B),
             few ? 2 * kRowLaunch : kRowLaunch, (size_t)p->L1max * 17 / 2, st, p->dp, xh, gu1, gf);
}

static void launch_gx(const jtfs_plan* p, int B, const float2* gxh, const float* gs0, float* gx,
                      cudaStream_t st) {
  const bool few = few_blocks(p, (long long)p->dp.D * B);
  launch_pdl(few ? k_gx<2 * kFftThreads> : k_gx<kFftThreads>, dim3(p->dp.D, B),
             few ? 2 * kFftThreads : kFftThreads, (size_t)p->dp.M * 17 / 2, st, p->dp, gxh, gs0, gx);
}

bool backward_reuses_forward(const jtfs_plan* p) {
  // the forward's BF16 Y planes are the backward's operands (not for TF32, whose forward
  // writes FP32 planes)
  return p->use_tc && p->use_tcb && p->cfg.precision != JTFS_PREC_TF32;
}

jtfs_status launch_backward(const jtfs_plan* p, const float* x, const float* u1, int B,
                            const float* gs0, const float* gs1, const float* gs2, float* gx,
                            const Workspace& w, cudaStream_t st, bool fused) {
  jtfs_status rc = set_attrs(p);
  if (rc != JTFS_OK) return rc;
  const DevPlan& d = p->dp;
  // fused: x-hat, U1-hat (and the BF16 Y planes) are still in the workspace from the forward
  // of the same call; otherwise recompute them from x and the checkpoint
  const bool reuse_y = fused && backward_reuses_forward(p);
  if (!fused) {
    {
      StageScope sc(p, kStXfft, st, 2);
      launch_xfft_sub(p, B, x, w.xsub, st);
      launch_pdl(k_xfft_combine, dim3((p->N / 2 + 255) / 256, B), 256, 0, st, d, w.xsub, w.xh);
    }
    {
      StageScope sc(p, kStUhFromU1, st, 1);
      launch_pdl(k_uh_from_u1, dim3(p->n1, B), kFftThreads, (size_t)p->L1max * 17 / 2, st, d, u1,
                 w.uh);
    }
  }
  const size_t n_items = p->items.size() / 2;
  if (gs2 && n_items > 0 && p->use_tcb) {
    if (!reuse_y) {
      StageScope sc(p, kStSecondOrder, st, 1);
      launch_pdl(k_second_order_rows<1>, dim3((unsigned)(p->rowitems.size() / 4), B),
                 p->row_threads, (size_t)p->rows_cap * 17 / 2, st, d,
                 reinterpret_cast<const int4*>(p->d_rowitems), w.uh, nullptr, (__nv_bfloat16*)w.ybh,
                 (__nv_bfloat16*)w.ybl, B);
    }
    StageScope sc(p, kStJointBwd, st, 0);   // the launcher counts its kernels
    jtfs_status r2 = launch_joint_bwd_tc(p, B, w.ybh, w.ybl, gs2, w.g1, w.gy, w.y, st);
    if (r2 != JTFS_OK) return r2;
    if (!p->tcb_fb_items.empty()) {
      // rates beyond the tensor-core backward's lambda' capacity: FP32 Y rows of those rates
      // only, then the CUDA-core backward on them
      launch_pdl(k_second_order_rows<0>, dim3((unsigned)(p->tcb_fb_rowitems.size() / 4), B),
                 p->row_threads, (size_t)p->tcb_fb_cap * 17 / 2, st, d,
                 reinterpret_cast<const int4*>(p->d_tcb_fb_rowitems), w.uh, w.y, nullptr, nullptr,
                 B);
      launch_joint_bwd_simt(p, (int)(p->tcb_fb_items.size() / 2), p->d_tcb_fb_items, B, w.y, gs2,
                            w.gy, st);
      p->prof.launches += 2;
    }
  } else if (gs2 && n_items > 0) {
    {
      StageScope sc(p, kStSecondOrder, st, 1);
      launch_pdl(k_second_order_rows<0>, dim3((unsigned)(p->rowitems.size() / 4), B),
                 p->row_threads, (size_t)p->rows_cap * 17 / 2, st, d,
                 reinterpret_cast<const int4*>(p->d_rowitems), w.uh, w.y, nullptr, nullptr, B);
    }
    StageScope sc(p, kStJointBwd, st, 1);
    launch_joint_bwd_simt(p, (int)n_items, p->d_items, B, w.y, gs2, w.gy, st);
  } else if (p->y_len > 0) {
    cudaMemsetAsync(w.gy, 0, (size_t)B * p->y_len * sizeof(float2), st);
  }
  const GyParts gp = {w.y, p->tcbf_sub_off, p->tcbf_sub_len, p->tcbf_sub_a0, p->tcbf_sub_a1,
                      gs2 && n_items > 0 && p->use_tcb ? tcb_parts(p, B) : 1};
  {
    StageScope sc(p, kStSecondOrderBwd, st, 2);
    if (!p->rowitems.empty())
      launch_pdl(k_gy_spectra, dim3((unsigned)(p->rowitems.size() / 4), B), p->row_threads,
                 (size_t)p->rows_cap * 17 / 2, st, d, reinterpret_cast<const int4*>(p->d_rowitems),
                 w.gy, gp);
    launch_second_order_bwd(p, B, w.gy, gs1, w.gu1, st);
  }
  {
    StageScope sc(p, kStStage1Bwd, st, 1);
    launch_stage1_bwd(p, B, w.xh, w.gu1, w.gf, st);
  }
  {
    StageScope sc(p, kStGx, st, 2);
    launch_pdl(k_gxh, dim3((p->N / 2 + 255) / 256, B), 256, 0, st, d, w.gf, gs0, w.gxh);
    launch_gx(p, B, w.gxh, gs0, gx, st);
  }
  return cuda_check(cudaGetLastError(), "backward launch");
}

// Time scattering backward: x-hat and U1-hat rebuilt from x and the checkpoint, the second
// order's gY from g_S2t, then the transform's own adjoint chain from gY down to g_x.
jtfs_status launch_scat1d_backward(const jtfs_plan* p, const float* x, const float* u1, int B,
                                   const float* gs0, const float* gs1, const float* gs2t,
                                   float* gx, const Workspace& w, cudaStream_t st) {
  jtfs_status rc = set_attrs(p);
  if (rc != JTFS_OK) return rc;
  const DevPlan& d = p->dp;
  {
    StageScope sc(p, kStXfft, st, 2);
    launch_xfft_sub(p, B, x, w.xsub, st);
    launch_pdl(k_xfft_combine, dim3((p->N / 2 + 255) / 256, B), 256, 0, st, d, w.xsub, w.xh);
  }
  {
    StageScope sc(p, kStUhFromU1, st, 1);
    launch_pdl(k_uh_from_u1, dim3(p->n1, B), kFftThreads, (size_t)p->L1max * 17 / 2, st, d, u1,
               w.uh);
  }
  if (gs2t && !p->rowitems.empty()) {
    StageScope sc(p, kStJointBwd, st, 1);
    auto* kernel = p->n_t >= 8 ? k_scat1d_bwd_rows<8>
                   : p->n_t == 4 ? k_scat1d_bwd_rows<4>
                   : p->n_t == 2 ? k_scat1d_bwd_rows<2> : k_scat1d_bwd_rows<1>;
    launch_pdl(kernel, dim3((unsigned)(p->rowitems.size() / 4), B), p->row_threads,
               (size_t)p->rows_cap * 17 / 2, st, d, reinterpret_cast<const int4*>(p->d_rowitems),
               w.uh, gs2t, w.gy);
  } else if (p->y_len > 0) {
    cudaMemsetAsync(w.gy, 0, (size_t)B * p->y_len * sizeof(float2), st);
  }
  {
    StageScope sc(p, kStSecondOrderBwd, st, 2);
    if (!p->rowitems.empty())
      launch_pdl(k_gy_spectra, dim3((unsigned)(p->rowitems.size() / 4), B), p->row_threads,
                 (size_t)p->rows_cap * 17 / 2, st, d, reinterpret_cast<const int4*>(p->d_rowitems),
                 w.gy, GyParts{nullptr, 0, 0, 0, 0, 1});
    launch_second_order_bwd(p, B, w.gy, gs1, w.gu1, st);
  }
  {
    StageScope sc(p, kStStage1Bwd, st, 1);
    launch_stage1_bwd(p, B, w.xh, w.gu1, w.gf, st);
  }
  {
    StageScope sc(p, kStGx, st, 2);
    launch_pdl(k_gxh, dim3((p->N / 2 + 255) / 256, B), 256, 0, st, d, w.gf, gs0, w.gxh);
    launch_gx(p, B, w.gxh, gs0, gx, st);
  }
  return cuda_check(cudaGetLastError(), "time scattering backward");
}

}  // namespace jtfs
