// Binned power spectrum (Sec. 3.1 of arXiv 2502.02294; cross spectrum for r_c, Sec. 3.2).
// Bins of width k_f = 2 pi / L, index round(|k| / k_f); the half spectrum counts twice for
// 0 < k_x < n/2. Each CTA histograms its modes in shared memory (FP64) and adds its bins
// to the global sums once.
#include <algorithm>

#include "pm.cuh"

namespace dh {

// Bin round(|k|) of a mode with k2 = |k|^2 in units of k_f, in integers: the float square
// root is within one of it, and |k| lies in (b - 1/2, b + 1/2) exactly when
// b^2 - b < k2 <= b^2 + b (k2 is an integer, so |k| is never a half).
__device__ __forceinline__ int mode_bin(int k2, float& root) {
  root = __fsqrt_rn((float)k2);
  int b = __float2int_rn(root);
  if (k2 > b * b + b) ++b;
  if (k2 <= b * b - b) --b;
  return b;
}

// (hi, lo) += (v, vlo): float pairs, the sum hi + v by Knuth's two-sum (error-free while nothing
// overflows; neither operand needs to be the larger)
__device__ __forceinline__ void pair_add(float v, float vlo, float& hi, float& lo) {
  const float s = __fadd_rn(hi, v), t = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(vlo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(v, t))));
  hi = s;
}

// Sum of the float pair over the lanes lane .. last (inclusive) of a contiguous run of lanes,
// right for the first lane of each run (all lanes of the warp call it).
__device__ __forceinline__ void run_sum(int lane, int last, float& hi, float& lo) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const float h = __shfl_down_sync(0xffffffffu, hi, d), l = __shfl_down_sync(0xffffffffu, lo, d);
    if (lane + d <= last) pair_add(h, l, hi, lo);
  }
}

__device__ __forceinline__ void run_sum(int lane, int last, double& v) {
#pragma unroll 1
  for (int d = 1; d < 32; d <<= 1) {
    const double o = __shfl_down_sync(0xffffffffu, v, d);
    if (lane + d <= last) v += o;
  }
}

// hi + lo += x y as a float pair, the product exact while its low word stays representable
// (kPairMin); m: the largest |product| so far
__device__ __forceinline__ void dot2(float x, float y, float& hi, float& lo, float& m) {
  const float p = __fmul_rn(x, y);
  pair_add(p, __fmaf_rn(x, y, -p), hi, lo);
  m = fmaxf(m, fabsf(p));
}

// Products for which float pairs are as good as doubles: a low word is a multiple of 2^-149,
// 2^-59 of kPairMin, and the at most 512 products of a run stay below 2^110.
constexpr float kPairMin = 0x1p-90f, kPairMax = 0x1p100f;

// The powers of a warp's modes in FP64 (see spectrum_bin_kernel), added to the histogram once per
// run of lanes; out of line, so that it costs the common path no registers.
template <int NP>
__device__ __noinline__ void spectrum_wide_run(const cufftComplex* a, const cufftComplex* b, int n,
                                               int nbins, int kx, int ky, int kz, int bin,
                                               bool two_y, bool two_z, int wx, int lane, int last,
                                               bool head, double* hist) {
  const unsigned nh = n / 2 + 1;
#pragma unroll 1
  for (int q = 0; q < NP; ++q) {  // |a|^2, |b|^2, Re(a conj b); NP = 1: the last alone
    const cufftComplex* p = NP == 3 && q == 1 ? b : a;
    const cufftComplex* r = NP == 3 && q == 0 ? a : b;
    double v = 0.0;
    if (bin >= 0)
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        if (((c & 1) && !two_y) || ((c & 2) && !two_z)) continue;
        const long long o =
            ((long long)((c & 2) ? n - kz : kz) * n + ((c & 1) ? n - ky : ky)) * nh + kx;
        const cufftComplex x = p[o], y = r[o];
        v += (double)x.x * y.x + (double)x.y * y.y;
      }
    v *= (double)wx;
    run_sum(lane, last, v);
    if (head && bin >= 0) atomicAdd(hist + (size_t)(1 + q) * nbins + bin, v);
  }
}

// Sums per bin 1 .. nbins: mode weight, weight |k|, and NP weighted powers (NP = 0: the weight
// alone; 1: Re(a conj b); 3: |a|^2, |b|^2, Re(a conj b)), [2 + NP][nbins] doubles ([nbins] for
// NP = 0), accumulated. A thread takes the modes (k_x, +-k_y, +-k_z) of one |k| together (up
// to four, of 8-byte loads coalesced along k_x), so the bin, |k| and the histogram updates are
// paid once for all four. FP64 runs at 1/64 of the FP32 rate here, so the work per mode is in
// float: the bin in integers, |k| as a float root plus its residual, the products exact in
// float pairs; only the histograms are double, updated once per run of lanes of one bin (|k|
// grows along a row; a shared-memory double atomic is a compare-and-swap loop). At 128^3, 64
// bins, this took 80 us (108 us for NP = 3) with one FP64 update of every sum per mode, 21 us
// (32 us) with one per thread; now 10 us (16 us).
// A float pair has float's exponent range, the modes of a field in any units do not keep to it:
// a warp with a product outside [kPairMin, kPairMax] (infinities among them) forms its powers
// in FP64. For the cross product of NP = 3 the two auto products decide: its error counts
// against the root of theirs.
template <int NP>
__global__ void __launch_bounds__(512) spectrum_bin_kernel(const cufftComplex* __restrict__ a,
                                                           const cufftComplex* __restrict__ b, int n,
                                                           int nbins, double* __restrict__ sums) {
  pdl_enter();
  extern __shared__ double hist[];  // [1 + NP][nbins] (weight |k|, powers; none for NP = 0), counts
  constexpr int ND = NP ? 1 + NP : 0;
  unsigned* cnt = reinterpret_cast<unsigned*>(hist + (size_t)ND * nbins);
  for (int j = threadIdx.x; j < ND * nbins; j += blockDim.x) hist[j] = 0.0;
  for (int j = threadIdx.x; j < nbins; j += blockDim.x) cnt[j] = 0u;
  __syncthreads();
  const unsigned nh = n / 2 + 1;  // 0 <= |k| <= n / 2 along every axis
  const unsigned total = nh * nh * nh;
  const int lane = threadIdx.x & 31;
  // whole warps stay in the loop for the warp-wide sums
  for (unsigned i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < total;
       i0 += gridDim.x * blockDim.x) {
    const unsigned i = i0 + lane;
    const int kx = i % nh;
    const unsigned r = i / nh;
    const int ky = r % nh, kz = r / nh;
    float root;
    const int k2 = kx * kx + ky * ky + kz * kz;
    int bin = i < total ? mode_bin(k2, root) - 1 : -1;
    if (bin >= nbins) bin = -1;
    // k and -k are distinct modes except at 0 and, for even n, at the Nyquist index
    const bool two_y = ky != 0 && 2 * ky != n, two_z = kz != 0 && 2 * kz != n;
    const int wx = (kx == 0 || 2 * kx == n) ? 1 : 2;
    const int mult = wx << ((int)two_y + (int)two_z);
    if (bin >= 0) atomicAdd(cnt + bin, (unsigned)mult);
    if (NP) {
      // |k| = root + (k2 - root^2) / (2 root) to 1e-14; mult is a power of two
      float khi = 0.0f, klo = 0.0f;
      float hi[NP ? NP : 1], lo[NP ? NP : 1], m[NP ? NP : 1];
#pragma unroll
      for (int q = 0; q < NP; ++q) hi[q] = lo[q] = m[q] = 0.0f;
      unsigned nzx = 0u, nzy = 0u;  // bits of the components: zero modes are exact
      if (bin >= 0) {
        const float fm = (float)mult;
        khi = fm * root;
        klo = fm * __fdividef(__fmaf_rn(-root, root, (float)k2), 2.0f * root);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (((c & 1) && !two_y) || ((c & 2) && !two_z)) continue;
          const long long o =
              ((long long)((c & 2) ? n - kz : kz) * n + ((c & 1) ? n - ky : ky)) * nh + kx;
          const cufftComplex x = a[o], y = b[o];
          if (NP == 3) {
            dot2(x.x, x.x, hi[0], lo[0], m[0]);
            dot2(x.y, x.y, hi[0], lo[0], m[0]);
            dot2(y.x, y.x, hi[1], lo[1], m[1]);
            dot2(y.y, y.y, hi[1], lo[1], m[1]);
          }
          dot2(x.x, y.x, hi[NP - 1], lo[NP - 1], m[NP - 1]);
          dot2(x.y, y.y, hi[NP - 1], lo[NP - 1], m[NP - 1]);
          nzx |= __float_as_uint(x.x) | __float_as_uint(x.y);
          nzy |= __float_as_uint(y.x) | __float_as_uint(y.y);
        }
        const float fw = (float)wx;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          hi[q] *= fw;
          lo[q] *= fw;
        }
      }
      // |k| grows along a row, so lanes of one bin are neighbours: one update per run of them
      const int left = __shfl_up_sync(0xffffffffu, bin, 1);
      const bool head = lane == 0 || left != bin;
      const unsigned heads = __ballot_sync(0xffffffffu, head);
      const unsigned after = lane == 31 ? 0u : heads >> (lane + 1);
      const int last = after ? lane + __ffs(after) - 1 : 31;
      run_sum(lane, last, khi, klo);
      if (head && bin >= 0) atomicAdd(hist + bin, (double)khi + (double)klo);
      const bool zx = (nzx << 1) == 0u, zy = (nzy << 1) == 0u;
      bool wide;
      if (NP == 3)
        wide = !(zx || (m[0] >= kPairMin && m[0] <= kPairMax)) ||
               !(zy || (m[1] >= kPairMin && m[1] <= kPairMax));
      else
        wide = !(zx || zy || (m[0] >= kPairMin && m[0] <= kPairMax));
      if (__any_sync(0xffffffffu, wide)) {
        spectrum_wide_run<NP>(a, b, n, nbins, kx, ky, kz, bin, two_y, two_z, wx, lane, last, head, hist);
      } else {
#pragma unroll
        for (int q = 0; q < NP; ++q) run_sum(lane, last, hi[q], lo[q]);
        if (head && bin >= 0)
#pragma unroll
          for (int q = 0; q < NP; ++q)
            atomicAdd(hist + (size_t)(1 + q) * nbins + bin, (double)hi[q] + (double)lo[q]);
      }
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < nbins; j += blockDim.x)
    if (cnt[j]) atomicAdd(&sums[j], (double)cnt[j]);
  for (int j = threadIdx.x; j < ND * nbins; j += blockDim.x)
    if (hist[j] != 0.0) atomicAdd(&sums[nbins + j], hist[j]);
}

sim_status launch_spectrum_bins(const cufftComplex* a, const cufftComplex* b, int n, int nbins,
                                int powers, double* sums, cudaStream_t st) {
  const long long nh = n / 2 + 1;
  const int blocks = std::min(cdiv(nh * nh * nh, 512), 152 * 2);
  const size_t smem = (size_t)nbins * ((powers ? 1 + powers : 0) * sizeof(double) + sizeof(unsigned));
  switch (powers) {
    case 0: DH_CUDA_TRY((launch_pdl(spectrum_bin_kernel<0>, blocks, 512, smem, st, a, b, n, nbins, sums))); break;
    case 1: DH_CUDA_TRY((launch_pdl(spectrum_bin_kernel<1>, blocks, 512, smem, st, a, b, n, nbins, sums))); break;
    default: DH_CUDA_TRY((launch_pdl(spectrum_bin_kernel<3>, blocks, 512, smem, st, a, b, n, nbins, sums))); break;
  }
  DH_LAUNCH_CHECK();
  return SIM_OK;
}

__global__ void pk_finish_kernel(const double* __restrict__ sums, int nbins, double kf,
                                 double norm, double* __restrict__ k, double* __restrict__ pk,
                                 double* __restrict__ nm) {
  pdl_enter();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= nbins) return;
  const double w = sums[j];
  nm[j] = w;
  k[j] = w > 0 ? kf * sums[nbins + j] / w : 0.0;
  pk[j] = w > 0 ? norm * sums[2 * nbins + j] / w : 0.0;
}

// Adjoint of the binned spectrum: for the half-complex mode k of bin b,
//   ak <- ak * 2 norm dL/dP_b / W_b   (W_b the bin's mode weight, from weights[0..nbins)),
// modes outside bins 1..nbins <- 0. The unnormalised c2r of the result is dL/da: each P_b is
// norm / W_b sum_half w |a_k|^2, and the half-complex weights w make sum_half w Re(conj(a_k)
// e^{-ikx}) the full-grid sum that c2r evaluates. The factors of the bins are formed once per
// block (an FP64 division per bin instead of one per mode: 56 us at 128^3, now 9 us).
__global__ void __launch_bounds__(256) pk_adj_scale_kernel(cufftComplex* __restrict__ ak, int n,
                                                           int nbins,
                                                           const double* __restrict__ dL_dpk,
                                                           const double* __restrict__ weights,
                                                           double norm) {
  pdl_enter();
  extern __shared__ float coef[];  // [nbins]
  for (int j = threadIdx.x; j < nbins; j += blockDim.x)
    coef[j] = weights[j] > 0 ? (float)(2.0 * norm * dL_dpk[j] / weights[j]) : 0.0f;
  __syncthreads();
  const unsigned nh = n / 2 + 1;
  const unsigned NC = (unsigned)n * n * nh;
  for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < NC; i += gridDim.x * blockDim.x) {
    const int kx = i % nh;
    const unsigned r = i / nh;
    int ky = r % (unsigned)n, kz = r / (unsigned)n;
    if (ky > n / 2) ky -= n;
    if (kz > n / 2) kz -= n;
    float root;
    const int bin = mode_bin(kx * kx + ky * ky + kz * kz, root);
    const float c = bin >= 1 && bin <= nbins ? coef[bin - 1] : 0.0f;
    cufftComplex v = ak[i];
    v.x *= c;
    v.y *= c;
    ak[i] = v;
  }
}

}  // namespace dh

using namespace dh;

extern "C" sim_status sim_power_spectrum_adjoint(const float* a, int32_t n, double box,
                                                 int32_t nbins, const double* dL_dpk,
                                                 float* dL_da, void* stream) {
  if (!a || !dL_dpk || !dL_da || n < 2 || !(box > 0) || nbins < 1 || nbins > 2048) {
    set_error("sim_power_spectrum_adjoint: invalid arguments (1 <= nbins <= 2048)");
    return SIM_EINVAL;
  }
  FFTPlans* plans = shared_plans(n);
  if (!plans) return SIM_ECUDA;
  cudaStream_t st = (cudaStream_t)stream;
  const long long NC = (long long)n * n * (n / 2 + 1);
  cufftComplex* ak = nullptr;
  double* sums = nullptr;
  DH_CUDA_TRY(scratch_alloc((void**)&ak, NC * sizeof(cufftComplex) + nbins * sizeof(double), st));
  sums = reinterpret_cast<double*>(ak + NC);
  sim_status r = plans->set_stream(st);
  if (r == SIM_OK && cudaMemsetAsync(sums, 0, nbins * sizeof(double), st) != cudaSuccess) {
    set_error("cudaMemsetAsync failed");
    r = SIM_ECUDA;
  }
  if (r == SIM_OK && cufftExecR2C(plans->r2c1, const_cast<float*>(a), ak) != CUFFT_SUCCESS) {
    set_error("cufftExecR2C failed");
    r = SIM_ECUDA;
  }
  // mode weights per bin (the power sums are not needed)
  if (r == SIM_OK) r = launch_spectrum_bins(ak, ak, n, nbins, 0, sums, st);
  if (r == SIM_OK) {
    const double norm = box * box * box / ((double)n * n * n * (double)n * n * n);
    const int blocks = std::min(cdiv(NC, 256), 152 * 8);
    cudaError_t e = launch_pdl(pk_adj_scale_kernel, blocks, 256, nbins * sizeof(float), st, ak, n, nbins,
                               dL_dpk, sums, norm);
    count_launch();
    if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) {
      set_error("pk_adj_scale_kernel launch failed");
      r = SIM_ECUDA;
    }
  }
  if (r == SIM_OK && cufftExecC2R(plans->c2r1, ak, dL_da) != CUFFT_SUCCESS) {
    set_error("cufftExecC2R failed");
    r = SIM_ECUDA;
  }
  cudaFreeAsync(ak, st);
  return r;
}

extern "C" sim_status sim_power_spectrum(const float* a, const float* b, int32_t n, double box,
                                         int32_t nbins, double* k, double* pk, double* nmodes,
                                         void* stream) {
  if (!a || !k || !pk || !nmodes || n < 2 || !(box > 0) || nbins < 1 || nbins > 2048) {
    set_error("sim_power_spectrum: invalid arguments (1 <= nbins <= 2048)");
    return SIM_EINVAL;
  }
  FFTPlans* plans = shared_plans(n);
  if (!plans) return SIM_ECUDA;
  cudaStream_t st = (cudaStream_t)stream;
  const long long NC = (long long)n * n * (n / 2 + 1);
  cufftComplex* buf = nullptr;
  double* sums = nullptr;
  DH_CUDA_TRY(scratch_alloc((void**)&buf, 2 * NC * sizeof(cufftComplex) + 3 * nbins * sizeof(double), st));
  sums = reinterpret_cast<double*>(buf + 2 * NC);
  sim_status r = SIM_OK;
  cufftComplex* ak = buf;
  cufftComplex* bk = b ? buf + NC : buf;
  if (plans->set_stream(st) != SIM_OK) r = SIM_ECUDA;
  if (r == SIM_OK && cudaMemsetAsync(sums, 0, 3 * nbins * sizeof(double), st) != cudaSuccess) {
    set_error("cudaMemsetAsync failed");
    r = SIM_ECUDA;
  }
  if (r == SIM_OK && cufftExecR2C(plans->r2c1, const_cast<float*>(a), ak) != CUFFT_SUCCESS) {
    set_error("cufftExecR2C failed");
    r = SIM_ECUDA;
  }
  if (r == SIM_OK && b && cufftExecR2C(plans->r2c1, const_cast<float*>(b), bk) != CUFFT_SUCCESS) {
    set_error("cufftExecR2C failed");
    r = SIM_ECUDA;
  }
  if (r == SIM_OK) r = launch_spectrum_bins(ak, bk, n, nbins, 1, sums, st);
  if (r == SIM_OK) {
    const double norm = box * box * box / ((double)n * n * n * (double)n * n * n);
    DH_CUDA_TRY((launch_pdl(pk_finish_kernel, cdiv(nbins, 128), 128, 0, st, sums, nbins, 2.0 * M_PI / box, norm, k,
                                                        pk, nmodes)));
    count_launch();
    if (cudaGetLastError() != cudaSuccess) {
      set_error("pk_finish_kernel launch failed");
      r = SIM_ECUDA;
    }
  }
  cudaFreeAsync(buf, st);
  return r;
}
