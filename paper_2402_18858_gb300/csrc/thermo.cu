// Mixture thermo and transport properties per cell (the paper's Sec. 2.1 property update:
// Newton's method for T from h, and temperature polynomials for the species properties).
//
// The species-major SoA layout makes every Y[k][*] load coalesced over cells.  c_p, h and the
// Newton solve are FP64.  The Wilke viscosity and the conductivity combining rule cost O(K^2) per
// cell; on GB300 FP64 issue (one warp instruction per 64 cycles in each SM sub-partition) would
// make them compute-bound far above the HBM time.  The mixed-precision mode therefore evaluates
// those sums in FP32 (the fits themselves are accurate to percent level), and the FP64 mode
// evaluates Wilke's in 55-bit fixed point on the integer pipe (thermo64_kernel).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "internal.h"

namespace chem {

// Shared-memory copy of the tables one block of the mixed mode needs: NASA-7 coefficients divided by
// the molar mass and transposed to [range][coefficient][species] (cp/R: a1..a5, h/RT: a6 is the
// only extra term), the FP32 transport fits and the three Wilke coefficients of the expanded form.
struct ThermoSmem {
  double* c;     // [2][6][K]  a_qk / W_k
  float* tr;     // [8][K]     ln mu (4), ln lambda (4)
  float4* w3;    // [K][K] (A, A B, A B^2, 0)
  float* invW;   // [K]
};

__host__ __device__ inline size_t thermo_smem_bytes(int K, bool transport) {
  if (!transport) return (size_t)12 * K * sizeof(double);
  return (size_t)12 * K * sizeof(double) + (size_t)8 * K * sizeof(float) + (size_t)K * K * sizeof(float4) +
         (size_t)K * sizeof(float) + 16;
}

// mixture polynomial coefficients A_i = sum_k Y_k (a_ik / W_k) (one FMA per coefficient and
// species), then c_p = R sum_i A_i T^i and h = R T (sum_i A_i T^i / (i+1) + A_5 / T)
template <int KC>
__device__ __forceinline__ void mix_coeffs(const double* __restrict__ cr, int K, const double* yv, double (&A)[6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i) A[i] = 0.0;
#pragma unroll
  for (int k = 0; k < (KC ? KC : K); ++k) {
    const double y = yv[k];
#pragma unroll
    for (int i = 0; i < 6; ++i) A[i] = fma(y, cr[i * K + k], A[i]);
  }
}
__device__ __forceinline__ void cp_h_of(const double (&A)[6], double T, double& cp, double& h) {
  // T A4, common to both, is rounded by itself, so that c_p has the same bits whether or not h is wanted
  const double t4 = __dmul_rn(T, A[4]);
  cp = kR * (A[0] + T * (A[1] + T * (A[2] + T * __dadd_rn(A[3], t4))));
  h = kR * (T * (A[0] + T * (A[1] * 0.5 + T * (A[2] * (1.0 / 3.0) + T * fma(A[3], 0.25, __dmul_rn(t4, 0.2))))) + A[5]);
}

// T from h(T) = ht by Newton's method.  The mixture coefficients belong to a temperature range, not
// to an iterate: they are formed once (coeffs(range, A)) and again only when the iterate crosses
// T_mid, so an iteration costs 11 multiply-adds instead of 6 per species (53 species, T from h in
// mixed precision: 583 -> 330 us at 120,007 cells).  On return A, cp and h belong to Tc.
// WARP: every lane of the warp calls it together and coeffs exchanges between lanes, so that the
// iterations run until all lanes are done and the coefficients are formed by all lanes again when
// any lane crosses (lanes that stay get the same values).
template <bool WARP, typename Coeffs>
__device__ __forceinline__ void solve_T(double& Tc, bool newton, double ht, double Tmid, Coeffs coeffs, double (&A)[6],
                                        double& cp, double& h) {
  bool hi = Tc >= Tmid;
  coeffs(hi, A);
  cp_h_of(A, Tc, cp, h);
  if (!newton) return;
  bool done = false;
  for (int it = 0; it < 50; ++it) {
    if (!done) {
      double Tn = Tc - (h - ht) / cp;
      Tn = fmin(fmax(Tn, 200.0), 6000.0);
      done = fabs(Tn - Tc) < 1e-9;
      Tc = Tn;
    }
    const bool cross = (Tc >= Tmid) != hi;
    if (WARP ? __any_sync(0xffffffffu, cross) : cross) {
      hi = Tc >= Tmid;
      coeffs(hi, A);
    }
    cp_h_of(A, Tc, cp, h);
    if (WARP ? __all_sync(0xffffffffu, done) : done) break;
  }
}

// One thread per cell: the mixed mode, and either mode without transport outputs (TR = false), where c_p and
// h are the same FP64 sums in both and the kernel holds only them: bound by its loads, where
// thermo64_kernel's registers and shared memory leave few warps to hide them (FP64 mode, 200,000 cells,
// thermo64_kernel -> this one: c_p of 12 species 74 -> 44 us, 30 species 117 -> 64, 53 species 220 -> 111; T from
// h of 30 species 249 -> 171).
// FROM_H: T from h first (decided at run time without an unrolled species loop, where the split lost 17 %);
// unrolled, the solve in the same kernel cost calls without it 3 % (53 species, all outputs of 200,000 cells 375
// -> 361 us).
template <int KC, bool TR, bool FROM_H>
__global__ void __launch_bounds__(128) thermo_kernel(DevMech m, int64_t n, int64_t ld, const double* T,
                                                     const double* Y, double* cp_out, double* h_out,
                                                     double* mu_out, double* kappa_out, const double* h_in,
                                                     double* T_out) {
  extern __shared__ double tsm[];
  const int K = KC ? KC : m.K;
  ThermoSmem S;
  S.c = tsm;
  if constexpr (TR) {
    S.tr = (float*)(tsm + 12 * K);
    // float4 table 16-byte aligned after the FP32 fits
    S.w3 = (float4*)(((uintptr_t)(S.tr + 8 * K) + 15) & ~(uintptr_t)15);
    S.invW = (float*)(S.w3 + K * K);
  }
  for (int i = threadIdx.x; i < 12 * K; i += blockDim.x) {
    const int rg = i / (6 * K), q = (i / K) % 6, k = i % K;
    const double* a = m.th + ((size_t)k * 2 + rg) * kThermoStride;
    S.c[i] = __ldg(a + (q < 5 ? q : 10)) * __ldg(m.invW + k);   // cp/R coefficients a1..a5, then a6
  }
  if constexpr (TR) {
    for (int i = threadIdx.x; i < 8 * K; i += blockDim.x) S.tr[i] = (float)__ldg(m.tr + (size_t)(i % K) * 8 + i / K);
    for (int i = threadIdx.x; i < K * K; i += blockDim.x) {
      const double A = __ldg(m.wA + i), B = __ldg(m.wB + i);
      S.w3[i] = make_float4((float)A, (float)(A * B), (float)(A * B * B), 0.0f);
    }
    for (int i = threadIdx.x; i < K; i += blockDim.x) S.invW[i] = (float)__ldg(m.invW + i);
  }
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    double yv[KC ? KC : CHEM_MAX_SPECIES];
    double sYW = 0.0;
#pragma unroll
    for (int k = 0; k < (KC ? KC : K); ++k) {
      yv[k] = Y[(size_t)k * ld + i];
      if (TR) sYW = fma(yv[k], __ldg(m.invW + k), sYW);
    }
    double Tc = T[i], cp, h, A[6];
    const bool newton = KC ? FROM_H : h_in != nullptr;
    solve_T<false>(Tc, newton, newton ? h_in[i] : 0.0, m.Tmid,
                   [&](bool hi, double (&a)[6]) { mix_coeffs<KC>(S.c + (hi ? 6 * K : 0), K, yv, a); }, A, cp, h);
    if (newton) T_out[i] = Tc;
    if (cp_out) cp_out[i] = cp;
    if (h_out) h_out[i] = h;
    if constexpr (!TR) continue;
    // FP32 transport.  Wilke's denominator D_k = sum_j X_j A_kj (1 + s_k B_kj / s_j)^2 with
    // s = sqrt(mu) expands into three sums over j with per-cell vectors X_j, X_j / s_j and
    // X_j / s_j^2: D_k = sum A X + 2 s_k sum (A B) (X / s) + s_k^2 sum (A B^2)(X / s^2),
    // all terms positive (no cancellation), 3 FMAs per species pair.
    float X[KC ? KC : CHEM_MAX_SPECIES], sm[KC ? KC : CHEM_MAX_SPECIES];
    float vx[KC ? KC : CHEM_MAX_SPECIES], wx[KC ? KC : CHEM_MAX_SPECIES];
    const float isYW = __frcp_rn(narrow_f32(sYW));
    const float L = logf(narrow_f32(Tc));
    float l1 = 0.0f, l2 = 0.0f;
#pragma unroll
    for (int k = 0; k < (KC ? KC : K); ++k) {
      X[k] = narrow_f32(yv[k]) * S.invW[k] * isYW;
      const float lnmu = S.tr[k] + L * (S.tr[K + k] + L * (S.tr[2 * K + k] + L * S.tr[3 * K + k]));
      const float lnlam = S.tr[4 * K + k] + L * (S.tr[5 * K + k] + L * (S.tr[6 * K + k] + L * S.tr[7 * K + k]));
      sm[k] = expf(0.5f * lnmu);
      const float ism = expf(-0.5f * lnmu);
      l1 = fmaf(X[k], expf(lnlam), l1);
      l2 = fmaf(X[k], expf(-lnlam), l2);
      vx[k] = X[k] * ism;
      wx[k] = vx[k] * ism;
    }
    if (kappa_out) kappa_out[i] = 0.5 * ((double)l1 + (double)__frcp_rn(l2));
    if (mu_out) {
      float mu = 0.0f;
#pragma unroll 2
      for (int k = 0; k < (KC ? KC : K); ++k) {
        const float4* W3 = S.w3 + k * K;
        float d0 = 0.0f, d1 = 0.0f, d2 = 0.0f;
#pragma unroll
        for (int j = 0; j < (KC ? KC : K); ++j) {
          const float4 c = W3[j];
          d0 = fmaf(c.x, X[j], d0);
          d1 = fmaf(c.y, vx[j], d1);
          d2 = fmaf(c.z, wx[j], d2);
        }
        const float sk = sm[k];
        const float den = fmaf(sk, fmaf(sk, d2, 2.0f * d1), d0);
        mu = fmaf(X[k] * sk * sk, __frcp_rn(den), mu);
      }
      mu_out[i] = (double)mu;
    }
  }
}

// ------------------------------------------------------------------------------------------
// FP64 mode.  With C_kj = (W_j + W_k)^(-1/2), u_k = W_k^(1/4) mu_k^(-1/2) and p_k = Y_k W_k^(-1/2)
// (proportional to X_k W_k^(1/2)), Wilke's rule (Phi_kj = (1 + sqrt(mu_k/mu_j) (W_j/W_k)^(1/4))^2 /
// sqrt(8 (1 + W_k/W_j))) is
//   mu = sqrt(8) sum_k p_k / S_k,   S_k = sum_j p_j C_kj (u_k + u_j)^2 = u_k^2 P_k + 2 u_k Q_k + R_k,
//   P = C p, Q = C (p u), R = C (p u^2):
// three products of one constant symmetric matrix with per-cell vectors of positive terms (no
// cancellation), and one exponential per species for the viscosity instead of two.
//
// The FP64 pipe (64 cycles per warp instruction) bounds any FP64 form: 3 K^2 = 2,700 FMAs at 30
// species took 57 % of the kernel's time.  So these products run in fixed point on the integer pipe:
// entries as two limbs (55 bits relative to the largest of the vector), three 32 x 32 + 64-bit
// multiply-adds (4 cycles each) per term, exact 64-bit sums, rounded once when they return to FP64.
// About 25 FP64 operations per species are left (c_p and h sums, transport fits, products,
// reciprocals).  1 M cells, 30 species: 6.49 -> 2.27 ms (8.96 -> 2.75 ms with T from h); 400,000 cells,
// 53 species: 8.23 -> 2.76 ms.  Errors against 64 bits no larger than the FP64 form's: viscosity
// 7.3e-16 (7.7e-16), c_p 1.4e-16 (1.5e-16), conductivity 3.2e-16 (4.8e-16).
//
// Layout: SPLIT threads per cell (1 for K <= 9, 2 above: two threads with 15 species each need 128
// registers, 128 bytes of them spilled, and hide more latency than one with 30 at 255: 2.48 -> 2.09 ms before the
// limbs were rounded instead of cut), thread h of a cell keeping
// the limbs of species h JC .. h JC + JC - 1 in registers (JC compile-time: every index is static);
// rows of C are read as broadcasts from shared memory.  With two threads the halves' sums of a row are
// exchanged and each finishes every other row.  The exponentials stay in a rolled loop: unrolled over
// the species they overran the instruction cache (7.8 ms).  Cells with non-finite or extreme inputs take the plain FP64
// form (thermo_cell_plain).
// ------------------------------------------------------------------------------------------
constexpr int kFxExpLo = 1023 - 400, kFxExpHi = 1023 + 400;   // exponents the fixed-point form takes

// one cell in plain FP64 (any input: NaN and infinities propagate)
__device__ __noinline__ void thermo_cell_plain(const DevMech& m, int64_t i, int64_t ld, double Tc, const double* Y,
                                               const double* h_in, double* T_out, double* cp_out, double* h_out,
                                               double* mu_out, double* kappa_out) {
  const int K = m.K;
  double A[6], cp, h, sYW = 0.0;
  for (int k = 0; k < K; ++k) sYW = fma(Y[(size_t)k * ld + i], __ldg(m.invW + k), sYW);
  auto coeffs = [&](bool hi, double (&a)[6]) {
    for (int q = 0; q < 6; ++q) a[q] = 0.0;
    for (int k = 0; k < K; ++k) {
      const double* c = m.th + ((size_t)k * 2 + (hi ? 1 : 0)) * kThermoStride;
      const double yw = Y[(size_t)k * ld + i] * __ldg(m.invW + k);
      for (int q = 0; q < 6; ++q) a[q] = fma(yw, __ldg(c + (q < 5 ? q : 10)), a[q]);
    }
  };
  solve_T<false>(Tc, h_in != nullptr, h_in ? h_in[i] : 0.0, m.Tmid, coeffs, A, cp, h);
  if (h_in) T_out[i] = Tc;
  if (cp_out) cp_out[i] = cp;
  if (h_out) h_out[i] = h;
  if (!mu_out && !kappa_out) return;
  const double isYW = 1.0 / sYW, L = log(Tc);
  double s[CHEM_MAX_SPECIES], l1 = 0.0, l2 = 0.0, mu = 0.0;
  for (int k = 0; k < K; ++k) {
    const double* b = m.tr + (size_t)k * 8;
    const double X = Y[(size_t)k * ld + i] * __ldg(m.invW + k) * isYW;
    const double lam = exp(b[4] + L * (b[5] + L * (b[6] + L * b[7])));
    s[k] = exp(0.5 * (b[0] + L * (b[1] + L * (b[2] + L * b[3]))));
    l1 = fma(X, lam, l1);
    l2 += X / lam;
  }
  if (kappa_out) kappa_out[i] = 0.5 * (l1 + 1.0 / l2);
  if (!mu_out) return;
  for (int k = 0; k < K; ++k) {
    double D = 0.0;
    for (int j = 0; j < K; ++j) {
      const double f = 1.0 + s[k] * __ldg(m.wB + (size_t)k * K + j) / s[j];
      D += Y[(size_t)j * ld + i] * __ldg(m.invW + j) * isYW * __ldg(m.wA + (size_t)k * K + j) * f * f;
    }
    mu += Y[(size_t)k * ld + i] * __ldg(m.invW + k) * isYW * s[k] * s[k] / D;
  }
  mu_out[i] = mu;
}

template <int JC, int SPLIT>
struct Thermo64Cfg {
  static constexpr int JE = (JC + 1) & ~1;     // row length of one half of C (16-byte loads)
  static constexpr int KP = JC * SPLIT;
  static constexpr size_t FX = (size_t)2 * KP * 6 * sizeof(double);
  static constexpr size_t CT = (size_t)KP * SPLIT * JE * sizeof(int2);
  static constexpr size_t TAB = FX + CT + (size_t)KP * 11 * sizeof(double);
  static size_t smem(int threads) { return TAB + (size_t)2 * JC * threads * sizeof(double); }
};

template <int JC, int SPLIT>
__global__ void __launch_bounds__(128, JC <= 16 ? 4 : 2) thermo64_kernel(DevMech m, int64_t n, int64_t ld, const double* T, const double* Y,
                                                       double* cp_out, double* h_out, double* mu_out,
                                                       double* kappa_out, const double* h_in, double* T_out) {
  using Cf = Thermo64Cfg<JC, SPLIT>;
  extern __shared__ __align__(16) uint8_t tsm8[];
  const int K = m.K, nt = blockDim.x, tid = threadIdx.x;
  double* fx = (double*)tsm8;                       // [2][KP][6] NASA-7 a1..a5, a6
  int2* ct = (int2*)(tsm8 + Cf::FX);                // [KP][SPLIT][JE]
  double* trs = (double*)(tsm8 + Cf::FX + Cf::CT);  // [KP][11]
  double* us = trs + 11 * Cf::KP;                   // [JC][threads] u
  double* ps = us + (size_t)JC * nt;                // [JC][threads] p
  const int2 z2 = make_int2(0, 0);
  for (int e = tid; e < 2 * Cf::KP * 6; e += nt) {
    const int q = e % 6, k = (e / 6) % Cf::KP, rg = e / (6 * Cf::KP);
    fx[e] = k < K ? __ldg(m.th + ((size_t)k * 2 + rg) * kThermoStride + (q < 5 ? q : 10)) : 0.0;
  }
  for (int e = tid; e < Cf::KP * 11; e += nt) trs[e] = e < K * 11 ? __ldg(m.fx_tr + e) : 0.0;
  if (mu_out)
    for (int e = tid; e < Cf::KP * SPLIT * Cf::JE; e += nt) {
      const int jj = e % Cf::JE, hf = (e / Cf::JE) % SPLIT, k = e / (Cf::JE * SPLIT), j = hf * JC + jj;
      ct[e] = (k < K && j < K && jj < JC) ? __ldg(m.fxC + (size_t)k * K + j) : z2;
    }
  __syncthreads();
  // thread -> (cell, half): with two threads per cell, lanes 0-15 hold the first halves
  const int half = SPLIT == 1 ? 0 : (tid >> 4) & 1;
  const int cell = SPLIT == 1 ? tid : (tid >> 5) * 16 + (tid & 15);
  const int64_t per = nt / SPLIT, stride = (int64_t)gridDim.x * per;
  // every thread of a warp runs the same rounds (the halves exchange by shuffles)
  for (int64_t base = (int64_t)blockIdx.x * per; base < n; base += stride) {
    const bool have = base + cell < n;
    const int64_t i = have ? base + cell : n - 1;
    double v[JC];
    double sYW = 0.0;
    int E = 0;
#pragma unroll
    for (int j = 0; j < JC; ++j) {
      const int k = half * JC + j;
      v[j] = k < K ? Y[(size_t)k * ld + i] * trs[11 * k + 8] : 0.0;   // Y/W
      sYW += v[j];
      E = max(E, fix_exp(v[j]));
    }
    if (SPLIT == 2) {
      E = max(E, __shfl_xor_sync(0xffffffffu, E, 16));
      sYW += __shfl_xor_sync(0xffffffffu, sYW, 16);
    }
    double Tc = have ? T[i] : 300.0, A[6], cp, h;
    bool plain = E < kFxExpLo || E > kFxExpHi;
    // mixture coefficients A_q = sum_k (Y_k/W_k) a_qk of a temperature range (the lanes of a warp may
    // be in different ranges), in FP64: the coefficients of one polynomial term differ between species
    // by more than the fixed-point form's spare bits, and the FP64 pipe has the time
    auto coeffs = [&](bool hi, double (&a)[6]) {
      const double2* c2 = (const double2*)(fx + ((hi ? Cf::KP : 0) + half * JC) * 6);
#pragma unroll
      for (int q = 0; q < 6; ++q) a[q] = 0.0;
#pragma unroll
      for (int j = 0; j < JC; ++j) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const double2 c = c2[3 * j + q];
          a[2 * q] = fma(v[j], c.x, a[2 * q]);
          a[2 * q + 1] = fma(v[j], c.y, a[2 * q + 1]);
        }
      }
      if (SPLIT == 2)
#pragma unroll
        for (int q = 0; q < 6; ++q) a[q] += __shfl_xor_sync(0xffffffffu, a[q], 16);
    };
    solve_T<SPLIT == 2>(Tc, h_in != nullptr, h_in ? h_in[i] : 0.0, m.Tmid, coeffs, A, cp, h);
    double l1 = 0.0, l2 = 0.0, mu = 0.0;
    const double L = log_t_fix(Tc, m.flogtab);
#pragma unroll
    for (int j = 0; j < JC; ++j) ps[j * nt + tid] = v[j];
    int Ep = 0, Eq = 0, Er = 0, ex = 0;
    // not unrolled: the three exponentials per species would not fit the instruction cache
#pragma unroll 1
    for (int j = 0; j < JC; ++j) {
      const int k = half * JC + j;
      const double* b = trs + 11 * k;
      const double yw = ps[j * nt + tid];
      const double xu = b[0] + L * (b[1] + L * (b[2] + L * b[3]));
      const double xl = b[4] + L * (b[5] + L * (b[6] + L * b[7]));
      const double u = b[10] * exp2_fix(fix_exp_arg(xu), m.fexptab);
      const long long fl = fix_exp_arg(xl);
      l1 = fma(yw, exp2_fix(fl, m.fexptab), l1);
      l2 = fma(yw, exp2_fix(-fl, m.fexptab), l2);
      const double p = yw * b[9], q = p * u;
      us[j * nt + tid] = u;
      ps[j * nt + tid] = p;
      Ep = max(Ep, fix_exp(p));
      Eq = max(Eq, fix_exp(q));
      Er = max(Er, fix_exp(q * u));
      ex = max(ex, max(fix_exp(xu), fix_exp(xl)));
    }
    plain = plain || ex > 1023 + 8;   // an exponential's argument beyond 512, or not finite
    if (SPLIT == 2) {
      Ep = max(Ep, __shfl_xor_sync(0xffffffffu, Ep, 16));
      Eq = max(Eq, __shfl_xor_sync(0xffffffffu, Eq, 16));
      Er = max(Er, __shfl_xor_sync(0xffffffffu, Er, 16));
      l1 += __shfl_xor_sync(0xffffffffu, l1, 16);
      l2 += __shfl_xor_sync(0xffffffffu, l2, 16);
      plain = __shfl_xor_sync(0xffffffffu, (int)plain, 16) || plain;
    }
    plain = plain || min(Ep, min(Eq, Er)) < kFxExpLo || max(Ep, max(Eq, Er)) > kFxExpHi;
    if (mu_out) {
      if (SPLIT == 2) __syncwarp();
      int2 p2[JC], q2[JC], r2[JC];
#pragma unroll
      for (int j = 0; j < JC; ++j) {
        const double p = ps[j * nt + tid], u = us[j * nt + tid], q = p * u;
        p2[j] = fix_vec(p, Ep);
        q2[j] = fix_vec(q, Eq);
        r2[j] = fix_vec(q * u, Er);
      }
      const int x0 = -1024 - m.fxC_e;
#pragma unroll 1
      for (int k0 = 0; k0 < K; k0 += SPLIT) {
        long long P[SPLIT], Q[SPLIT], R[SPLIT];
#pragma unroll
        for (int s = 0; s < SPLIT; ++s) {
          // (SPLIT = 2, odd K: the second row may be the zero row K < KP)
          const int4* c4 = (const int4*)(ct + ((size_t)(k0 + s) * SPLIT + half) * Cf::JE);
          long long ph = 0, pl = 0, qh = 0, ql = 0, rh = 0, rl = 0;
#pragma unroll
          for (int j = 0; j < JC; j += 2) {
            const int4 c = c4[j / 2];
            mad_wide(ph, c.x, p2[j].x);
            mad_wide(pl, c.x, p2[j].y);
            mad_wide(pl, c.y, p2[j].x);
            mad_wide(qh, c.x, q2[j].x);
            mad_wide(ql, c.x, q2[j].y);
            mad_wide(ql, c.y, q2[j].x);
            mad_wide(rh, c.x, r2[j].x);
            mad_wide(rl, c.x, r2[j].y);
            mad_wide(rl, c.y, r2[j].x);
            if (j + 1 < JC) {
              mad_wide(ph, c.z, p2[j + 1].x);
              mad_wide(pl, c.z, p2[j + 1].y);
              mad_wide(pl, c.w, p2[j + 1].x);
              mad_wide(qh, c.z, q2[j + 1].x);
              mad_wide(ql, c.z, q2[j + 1].y);
              mad_wide(ql, c.w, q2[j + 1].x);
              mad_wide(rh, c.z, r2[j + 1].x);
              mad_wide(rl, c.z, r2[j + 1].y);
              mad_wide(rl, c.w, r2[j + 1].x);
            }
          }
          P[s] = fix_fold(ph, pl);
          Q[s] = fix_fold(qh, ql);
          R[s] = fix_fold(rh, rl);
        }
        long long Pk = P[0], Qk = Q[0], Rk = R[0];
        int k = k0;
        if (SPLIT == 2) {
          // the first half's thread finishes row k0, the second's row k0 + 1
          const int o = half;
          Pk = P[o ? SPLIT - 1 : 0] + __shfl_xor_sync(0xffffffffu, P[o ? 0 : SPLIT - 1], 16);
          Qk = Q[o ? SPLIT - 1 : 0] + __shfl_xor_sync(0xffffffffu, Q[o ? 0 : SPLIT - 1], 16);
          Rk = R[o ? SPLIT - 1 : 0] + __shfl_xor_sync(0xffffffffu, R[o ? 0 : SPLIT - 1], 16);
          k = k0 + half;
        }
        if (k < K) {
          // u_k and p_k from the thread that owns species k
          const int own = SPLIT == 1 ? tid : (tid & ~16) | (k >= JC ? 16 : 0);
          const int at = (SPLIT == 1 ? k : (k >= JC ? k - JC : k)) * nt + own;
          const double u = us[at];
          const double S = fma(u, fma(u, fix_to_double(Pk, x0 + Ep), fix_to_double(Qk, x0 + Eq + 1)),
                               fix_to_double(Rk, x0 + Er));
          mu = fma(ps[at], rcp_nr(S), mu);
        }
      }
      if (SPLIT == 2) {
        mu += __shfl_xor_sync(0xffffffffu, mu, 16);
        __syncwarp();   // the next round overwrites us and ps
      }
      mu *= 2.8284271247461903;   // sqrt(8)
    }
    if (!have || half != 0) continue;
    if (plain) {
      thermo_cell_plain(m, i, ld, T[i], Y, h_in, T_out, cp_out, h_out, mu_out, kappa_out);
      continue;
    }
    if (h_in) T_out[i] = Tc;
    if (cp_out) cp_out[i] = cp;
    if (h_out) h_out[i] = h;
    if (mu_out) mu_out[i] = mu;
    if (kappa_out) kappa_out[i] = 0.5 * (l1 * rcp_nr(sYW) + sYW * rcp_nr(l2));
  }
}

static int thermo_sms() {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <int KC, bool TR, bool FROM_H>
static int launch_thermo_cell(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* Y, double* cp,
                              double* h, double* mu, double* kappa, const double* h_in, double* T_out, cudaStream_t s) {
  const size_t smem = thermo_smem_bytes(m.K, TR);
  int rc = cuda_check(cudaFuncSetAttribute(thermo_kernel<KC, TR, FROM_H>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                      "thermo smem attribute");
  if (rc) return rc;
  const int64_t blocks = std::min<int64_t>((n + 127) / 128, (int64_t)thermo_sms() * 8);
  thermo_kernel<KC, TR, FROM_H><<<(int)blocks, 128, smem, s>>>(m, n, ld, T, Y, cp, h, mu, kappa, h_in, T_out);
  return cuda_check(cudaGetLastError(), "thermo_kernel launch");
}

template <int JC, int SPLIT>
static int launch_thermo64(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* Y, double* cp,
                           double* h, double* mu, double* kappa, const double* h_in, double* T_out, cudaStream_t s) {
  using Cf = Thermo64Cfg<JC, SPLIT>;
  const int sms = thermo_sms();
  // blocks small enough that every SM has one
  int threads = 128;
  while (threads > 32 && n * SPLIT < (int64_t)sms * threads) threads /= 2;
  int rc = cuda_check(cudaFuncSetAttribute(thermo64_kernel<JC, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)Cf::smem(128)), "thermo64 smem attribute");
  if (rc) return rc;
  const int64_t blocks = std::min<int64_t>((n * SPLIT + threads - 1) / threads, (int64_t)sms * 8);
  thermo64_kernel<JC, SPLIT><<<(int)blocks, threads, Cf::smem(threads), s>>>(m, n, ld, T, Y, cp, h, mu, kappa, h_in, T_out);
  return cuda_check(cudaGetLastError(), "thermo64_kernel launch");
}

int launch_thermo(const DevMech& m, int64_t n, int64_t ld, const double* T, const double* Y,
                  double* cp, double* h, double* mu, double* kappa, const double* h_in,
                  double* T_out, int mixed, cudaStream_t s) {
  // Without transport outputs both modes are the same FP64 sums, by a thread per cell.  Species counts
  // of the shipped workloads get fully unrolled kernels; others run the generic loop
  const bool transport = mu || kappa;
#define CHEM_THERMO_CELL(KC)                                                                                        \
  return (transport ? h_in && KC ? launch_thermo_cell<KC, true, KC != 0> : launch_thermo_cell<KC, true, false>         \
                    : h_in && KC ? launch_thermo_cell<KC, false, KC != 0> : launch_thermo_cell<KC, false, false>)(     \
      m, n, ld, T, Y, cp, h, mu, kappa, h_in, T_out, s)
  if (mixed || !transport) {
    if (m.K == 9) CHEM_THERMO_CELL(9);
    if (m.K == 30) CHEM_THERMO_CELL(30);
    if (m.K == 53) CHEM_THERMO_CELL(53);
    CHEM_THERMO_CELL(0);
  }
#undef CHEM_THERMO_CELL
  // the narrowest instantiation that holds the species (the rest of its slots are zeros)
#define CHEM_THERMO64(JC, SPLIT) \
  if (m.K <= JC * SPLIT) return launch_thermo64<JC, SPLIT>(m, n, ld, T, Y, cp, h, mu, kappa, h_in, T_out, s);
  CHEM_THERMO64(9, 1)
  CHEM_THERMO64(8, 2)
  CHEM_THERMO64(12, 2)
  CHEM_THERMO64(15, 2)
  CHEM_THERMO64(20, 2)
  CHEM_THERMO64(27, 2)
  CHEM_THERMO64(32, 2)
#undef CHEM_THERMO64
  return set_error(CHEM_E_UNSUPPORTED, "thermo_props: too many species");
}

// ------------------------------------------------------------------------------------------
// FP64 FMA throughput probe (the DI roofline denominator): 8 independent FMA chains per
// thread, 4 blocks of 256 threads per SM.
// ------------------------------------------------------------------------------------------
__global__ void dfma_probe_kernel(double* sink, int iters, double a, double b) {
  double x0 = threadIdx.x, x1 = x0 + 1, x2 = x0 + 2, x3 = x0 + 3, x4 = x0 + 4, x5 = x0 + 5, x6 = x0 + 6, x7 = x0 + 7;
  for (int i = 0; i < iters; ++i) {
    x0 = fma(x0, a, b); x1 = fma(x1, a, b); x2 = fma(x2, a, b); x3 = fma(x3, a, b);
    x4 = fma(x4, a, b); x5 = fma(x5, a, b); x6 = fma(x6, a, b); x7 = fma(x7, a, b);
  }
  const double s = x0 + x1 + x2 + x3 + x4 + x5 + x6 + x7;
  if (s == 1.2345678) sink[threadIdx.x] = s;   // never true; keeps the chains alive
}

int launch_fp64_probe(double* gflops, cudaStream_t s) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  double* sink = nullptr;
  int rc = cuda_check(cudaMallocAsync((void**)&sink, 256 * sizeof(double), s), "probe alloc");
  if (rc) return rc;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  const int iters = 4096, blocks = sms * 4, threads = 256, reps = 3;
  dfma_probe_kernel<<<blocks, threads, 0, s>>>(sink, iters, 0.999, 1e-3);
  cudaEventRecord(e0, s);
  for (int r = 0; r < reps; ++r) dfma_probe_kernel<<<blocks, threads, 0, s>>>(sink, iters, 0.999, 1e-3);
  cudaEventRecord(e1, s);
  rc = cuda_check(cudaEventSynchronize(e1), "probe sync");
  float ms = 0;
  if (!rc) {
    cudaEventElapsedTime(&ms, e0, e1);
    const double flops = 2.0 * 8.0 * iters * (double)blocks * threads * reps;
    *gflops = flops / (ms * 1e-3) / 1e9;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFreeAsync(sink, s);
  return rc;
}

}  // namespace chem
