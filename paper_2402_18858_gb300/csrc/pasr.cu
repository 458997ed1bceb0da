// PaSR filtered reaction source from one chemistry step (the paper couples the learned step
// or DI to turbulence through the partially stirred reactor model, Sec. 3): per cell
//   kappa   = tau_c / (tau_c + tau_mix),
//   tau_mix = sqrt(sqrt(nu / eps) * k / eps)      (Kolmogorov time x sub-grid time k / eps),
//   tau_c   = max over species formed during the step (Y(t+dt) >= y_min and a gain
//             Y(t+dt) - Y(t) > r_min Y(t+dt)) of Y(t+dt) / ((Y(t+dt) - Y(t)) / dt)
//             (the slowest formation; r_min keeps rounding-level changes out),
//   omega_k = kappa rho (Y_k(t+dt) - Y_k(t)) / dt.
//
// One thread per cell over the species-major SoA state (coalesced loads and stores).  The kernel
// moves (3K + 5) doubles per cell, so it should be HBM-bound; on GB300 the K FP64 differences and
// K products already cost about as much FP64 issue (64 cycles per warp instruction) as the bytes
// cost HBM time, so everything else stays off the FP64 pipe: presence compares bit patterns, the
// formed decision (one IEEE product r_min Y(t+dt) per species before) is taken in FP32 wherever
// that settles it, the search for the slowest formation compares cross products in FP32 (only the
// winner's time is formed, in FP64), and the mixing time is FP32 from correctly rounded inputs
// (relative error below 1e-6).  1 M cells, 30 species: 223 -> 160 us (4.75 TB/s), same bits.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "internal.h"

namespace chem {

// Y1 and Y0 arrive by asynchronous copies into a ring of kRing chunks of kChunk species per thread:
// with plain loads the compiler placed each load before its use, one latency after the other (25 to
// 39 thousand cycles per cell of a warp, 2.7 to 3.4 TB/s).  A thread copies and reads only its own
// cells' slots, so no barrier is involved and any alignment of the rows (8 bytes) will do.  The species'
// differences stay in registers, so there is a kernel for each number of chunks (NB), and one more for a
// last chunk that is whole (WHOLE: no guards; 30 species, 900,000 cells 164 -> 160 us).  900,000 cells,
// thread-local arrays and plain loads -> ring: 12 species 109 -> 93 us, 20 species 154 -> 124, 36 species 244 ->
// 185, 44 species 287 -> 226, 62 species 392 -> 362.
constexpr int kChunk = 10, kRing = 2, kThreads = 128;
constexpr int kSlots = 2 * kChunk + 4;   // the cell's rho, k, eps and nu come with its last chunk
// blocks per SM by chunks, as the registers for the differences allow (six chunks: two blocks 305 us, three
// 264 us at 900,000 cells of 53 species; four chunks: three blocks 185 us, four 189 us at 36 species)
constexpr int kBlocks[8] = {0, 4, 4, 4, 3, 3, 3, 2};

__device__ __forceinline__ void copy_async8(double* smem_dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned int)__cvta_generic_to_shared(smem_dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// slowest formation: the largest y1 / d over formed, present species (Y1 >= y_min, d > r_min Y1),
// compared by FP32 cross products (all candidates have d > 0); y = 0: none.
struct Slowest {
  float y, d;
  double y1, dk;
};

// with the comparison itself, one IEEE product per species
__device__ __noinline__ Slowest slowest_exact(int K, int64_t i, int64_t ld, const double* Y0, const double* Y1,
                                              long long ymin_bits, double r_min) {
  Slowest b{0.0f, 1.0f, 0.0, 1.0};
  bool any = false;
  for (int k = 0; k < K; ++k) {
    const double y1 = Y1[(size_t)k * ld + i], dk = y1 - Y0[(size_t)k * ld + i];
    // y1 >= y_min >= 0 makes r_min y1 >= 0, so dk > r_min y1 orders like the bit patterns
    if (__double_as_longlong(y1) >= ymin_bits &&
        __double_as_longlong(dk) > __double_as_longlong(__dmul_rn(r_min, y1))) {
      const float yf = narrow_f32(y1), df = narrow_f32(dk);
      if (!any || yf * b.d > b.y * df) b = Slowest{yf, df, y1, dk};
      any = true;
    }
  }
  if (!any) b.dk = 0.0;
  return b;
}

// one species, without branches (the lanes differ in every decision) and without an FP64 product:
// d against r_min y1 in FP32, which settles all but gains within 2^-20 of the threshold and values
// outside FP32's normal range; those set `unsure`
__device__ __forceinline__ void slowest_step(double y1, double dk, long long ymin_bits, float r_hi, float r_lo,
                                             Slowest& b, bool& unsure) {
  const unsigned int yh = (unsigned int)__double2hiint(y1), dh = (unsigned int)__double2hiint(dk);
  // FP32 (truncated) of positive doubles with exponents in FP32's normal range: exponent rebias
  const float yf = __uint_as_float(__funnelshift_l((unsigned int)__double2loint(y1), yh, 3) - (384u << 23));
  const float df = __uint_as_float(__funnelshift_l((unsigned int)__double2loint(dk), dh, 3) - (384u << 23));
  const bool in_range = (yh - 0x38100000u < 0x0fe00000u) & (dh - 0x38100000u < 0x0fe00000u);
  const float th = r_hi * yf, tl = r_lo * yf;
  const bool present = __double_as_longlong(y1) >= ymin_bits;
  const bool above = df > th, settled = in_range & (tl > 1e-36f) & (above | (df < tl));
  unsure |= present & (__double_as_longlong(dk) > 0) & !settled;
  const bool take = present & settled & above & (yf * b.d > b.y * df);
  b.y = take ? yf : b.y;
  b.d = take ? df : b.d;
  b.y1 = take ? y1 : b.y1;
  b.dk = take ? dk : b.dk;
}

template <int NB, bool WHOLE>
__global__ void __launch_bounds__(kThreads, kBlocks[NB]) pasr_kernel(int Kr, int64_t n, int64_t ld, double dt, double inv_dt,
                                                   const double* __restrict__ rho, const double* __restrict__ Y0,
                                                   const double* __restrict__ Y1, const double* __restrict__ ksgs,
                                                   const double* __restrict__ eps, const double* __restrict__ nu,
                                                   long long ymin_bits, double r_min, double* __restrict__ omega,
                                                   double* __restrict__ kappa) {
  const int K = WHOLE ? NB * kChunk : Kr;
  const float r_minf = __double2float_rn(r_min);
  // With r_min = 0 every gain is above the threshold, r_hi y1 = 0, and any r_lo > 0 lets that settle it
  // (0 did not: every cell went through slowest_exact, 30 species, 900,000 cells 328 us).
  const float r_hi = r_minf * (1.0f + 0x1p-20f), r_lo = r_min == 0.0 ? 1.0f : r_minf * (1.0f - 0x1p-20f);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  extern __shared__ double ring[];                          // [kRing][kSlots][kThreads]
  double* mine = ring + threadIdx.x;
  int64_t fi = first;    // the cell and chunk fetched next
  int fc = 0, fslot = 0, slot = 0;
  auto fetch = [&]() {
    if (fi < n) {
      double* dst = mine + (size_t)fslot * kSlots * kThreads;
#pragma unroll
      for (int u = 0; u < kChunk; ++u) {
        const int k = fc * kChunk + u;
        if (k < K) {
          copy_async8(dst + 2 * u * kThreads, Y1 + (size_t)k * ld + fi);
          copy_async8(dst + (2 * u + 1) * kThreads, Y0 + (size_t)k * ld + fi);
        }
      }
      if (fc == NB - 1) {
        dst += 2 * kChunk * kThreads;
        copy_async8(dst, rho + fi);
        copy_async8(dst + kThreads, ksgs + fi);
        copy_async8(dst + 2 * kThreads, eps + fi);
        copy_async8(dst + 3 * kThreads, nu + fi);
      }
    }
    copy_commit();       // also an empty group: the waits below count groups
    fslot = fslot + 1 == kRing ? 0 : fslot + 1;
    if (++fc == NB) {
      fc = 0;
      fi += stride;
    }
  };
#pragma unroll
  for (int q = 0; q < kRing - 1; ++q) fetch();
  for (int64_t i = first; i < n; i += stride) {
    double d[NB * kChunk];
    Slowest b{0.0f, 1.0f, 0.0, 0.0};
    bool unsure = false;
    const double* last = nullptr;   // rho, k, eps, nu of the cell
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      fetch();
      copy_wait<kRing - 1>();   // all but the kRing - 1 newest groups: this chunk is here
      const double* src = mine + (size_t)slot * kSlots * kThreads;
      slot = slot + 1 == kRing ? 0 : slot + 1;
#pragma unroll
      for (int u = 0; u < kChunk; ++u)
        if (c < NB - 1 || c * kChunk + u < K) {
          const double y1 = src[2 * u * kThreads], dk = y1 - src[(2 * u + 1) * kThreads];
          d[c * kChunk + u] = dk;
          slowest_step(y1, dk, ymin_bits, r_hi, r_lo, b, unsure);
        }
      last = src + 2 * kChunk * kThreads;
    }
    if (unsure) b = slowest_exact(K, i, ld, Y0, Y1, ymin_bits, r_min);
    // dk > 0 for every candidate, 0 when there is none
    const double tau_c = __double_as_longlong(b.dk) > 0 ? dt * b.y1 * rcp_nr(b.dk) : 0.0;
    float tau_mix = 0.0f;
    const double rr = last[0], kk = last[kThreads], ee = last[2 * kThreads], nn = last[3 * kThreads];
    if (__double_as_longlong(kk) > 0 && __double_as_longlong(ee) > 0) {
      const float ie = __frcp_rn(__double2float_rn(ee));
      tau_mix = sqrtf(sqrtf(__double2float_rn(nn) * ie) * (__double2float_rn(kk) * ie));
    }
    const double tot = tau_c + (double)tau_mix;
    const double kap = tot > 0.0 ? tau_c * rcp_nr(tot) : 1.0;
    if (kappa) kappa[i] = kap;
    const double s = kap * rr * inv_dt;
#pragma unroll
    for (int k = 0; k < NB * kChunk; ++k)
      if (k < (NB - 1) * kChunk || k < K) omega[(size_t)k * ld + i] = s * d[k];
  }
}

int launch_pasr(const DevMech& m, int64_t n, int64_t ld, double dt, const double* rho, const double* Y0,
                const double* Y1, const double* ksgs, const double* eps, const double* nu, double y_min,
                double r_min, double* omega, double* kappa, cudaStream_t s) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t smem = (size_t)kRing * kSlots * kThreads * sizeof(double);   // 48 KB
  long long yb = 0;
  std::memcpy(&yb, &y_min, sizeof yb);
  const double inv_dt = 1.0 / dt;
  const int chunks = (m.K + kChunk - 1) / kChunk;
#define CHEM_PASR_CHUNKS(NB)                                                                                 \
  if (chunks == NB) {                                                                                        \
    auto kern = m.K % kChunk ? pasr_kernel<NB, false> : pasr_kernel<NB, true>;                               \
    int rc = cuda_check(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),  \
                        "pasr smem attribute");                                                              \
    if (rc) return rc;                                                                                       \
    const int blocks = (int)std::min<int64_t>((n + kThreads - 1) / kThreads, (int64_t)sms * kBlocks[NB]);    \
    kern<<<blocks, kThreads, smem, s>>>(m.K, n, ld, dt, inv_dt, rho, Y0, Y1, ksgs, eps, nu, yb, r_min, omega, kappa); \
    return cuda_check(cudaGetLastError(), "pasr_kernel launch");                                             \
  }
  CHEM_PASR_CHUNKS(1)
  CHEM_PASR_CHUNKS(2)
  CHEM_PASR_CHUNKS(3)
  CHEM_PASR_CHUNKS(4)
  CHEM_PASR_CHUNKS(5)
  CHEM_PASR_CHUNKS(6)
  CHEM_PASR_CHUNKS(7)
#undef CHEM_PASR_CHUNKS
  return set_error(CHEM_E_UNSUPPORTED, "chem_pasr_source: too many species");
}

}  // namespace chem
