// Range-Doppler imaging with range-cell migration correction and a
// range-dependent azimuth filter (Section VI's RCMC stage of the range-Doppler
// chain, on the paper's FP16 block-floating-point transforms).
//
// For a target at slant range R seen with the hyperbolic range history
// sqrt(R^2 + v^2 t^2), at Doppler frequency f it sits dR(f) = R (1/D(f) - 1)
// further out, D(f) = sqrt(1 - (lambda f / (2 v))^2), and its azimuth chirp
// has the FM rate k_a(R) = 2 v^2 / (lambda R PRF^2) cycles per pulse^2.  The
// line kernels here are the two steps the migration-free chain lacks:
//
//   rcmc_rows       one line per Doppler bin f, along range: the band-limited
//                   shift of the line by s = dR(f, R0) / range_cell cells back
//                   towards near range, as DFT, a linear phase
//                   exp(+2 pi i q s / N) on the signed frequency q (the Nyquist
//                   bin takes cos(pi s)), 1/N shift and inverse (Eq. 1's
//                   schedule);
//   azimuth_rows    one line per range bin r, along Doppler: the bin's own
//                   matched filter H_r = conj(DFT(ref_r)) (optionally divided by
//                   max |DFT(ref_r)|), ref_r the chirp exp(-i pi k_a(R_r) n^2),
//                   n in [-L/2, L/2), circularly centred at index 0, generated
//                   and transformed in registers, then H_r times the line, the
//                   1/N shift and the inverse.  No table of n_rg filters is read
//                   from HBM.
//
// Both run the radix-16 Stockham line transform of fft_rows.cuh in FP32
// registers; storage is FP16 (half2) or FP32 (float2).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "fft_rows.cuh"
#include "rda.h"

namespace bfp {

namespace {

// Phases.  Every phase of a line is an integer multiple of one number of turns
// that the line fixes: q s / N for the shift, k_a n^2 / 2 for the chirp.  That
// number's fractional part is kept as a 64-bit binary fraction, so a multiple
// is one integer product whose overflow drops whole turns exactly; its top 32
// bits give the phase to FP32 accuracy.  The line numbers themselves are
// computed in FP64 once per line by rda_lines_kernel: evaluated by every
// thread, with the reductions modulo 2 pi, they kept the FP64 pipe (two
// operations a cycle per SM) 60 % busy and took half of both kernels' time
// (4096 x 4096, FP16: RCMC rows 128 -> 68 us, azimuth rows 137 -> 73 us).
__device__ __forceinline__ unsigned long long turns_to_fixed(double turns) {
  const double f = turns - floor(turns);                       // in [0, 1)
  return static_cast<unsigned long long>(f * 18446744073709551616.0);
}
// exp(2 pi i phase / 2^64)
__device__ __forceinline__ float2 unit_of(unsigned long long phase) {
  float s, c;
  sincospif(float(int(phase >> 32)) * 4.656612873077393e-10f, &s, &c);   // half turns in [-1, 1): 2^-31 each
  return make_float2(c, s);
}

// shift[k] for the n_az Doppler bins: s / n_rg turns, s = dR(f, R0) / range_cell
// cells; rate[r] for the n_rg range bins: k_a(R_r) / 2 turns.
__global__ void rda_lines_kernel(RdaGeometry geo, int range_dependent, int n_az, int n_rg,
                                 unsigned long long* __restrict__ shift, unsigned long long* __restrict__ rate) {
  chain_begin();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_az) {
    const int k = i < n_az / 2 ? i : i - n_az;
    const double f = double(k) * geo.prf_hz / double(n_az);
    const double u = geo.wavelength_m * f / (2.0 * geo.speed_mps);
    const double s = geo.centre_range_m * (1.0 / sqrt(1.0 - u * u) - 1.0) / geo.range_cell_m;
    shift[i] = turns_to_fixed(s / double(n_rg));
  } else if (i < n_az + n_rg) {
    const int r = i - n_az;
    const double r_m = range_dependent ? geo.centre_range_m + (double(r) - 0.5 * double(n_rg)) * geo.range_cell_m
                                       : geo.centre_range_m;
    const double ka = 2.0 * geo.speed_mps * geo.speed_mps / (geo.wavelength_m * r_m * geo.prf_hz * geo.prf_hz);
    rate[r] = turns_to_fixed(0.5 * ka);
  }
}

template <int N, class TIn, class TOut, bool AZIMUTH>
__global__ void __launch_bounds__(RowShape<N>::kThreads, RowShape<N>::kMinBlocksDense)
rda_rows_kernel(const RdaArgs a) {
  using S = RowShape<N>;
  constexpr int P = S::P, T = S::T, G = S::G;
  extern __shared__ float2 smem_rda[];
  __shared__ float warp_max[32];
  __shared__ float2 ramp[AZIMUTH ? 1 : G][P];
  chain_begin();
  const int g = threadIdx.x / T;
  const int t = threadIdx.x - g * T;
  const long long line = (long long)blockIdx.x * G + g;
  const bool active = line < a.lines;
  float2* sm = smem_rda + g * S::kSmemPerLine;
  const float inv_n = 1.0f / float(N);
  const TIn* in = static_cast<const TIn*>(a.in) + line * (long long)N + t;
  const unsigned long long turns = active ? a.line_turns[line] : 0ull;
  float2 v[P];
  if constexpr (AZIMUTH) {
    // The line is wanted after its filter's transform only: into L2 meanwhile.
    if (t == 0 && active) prefetch_l2_bulk(in, uint32_t(N * sizeof(TIn)));
    // The line's reference chirp, exp(-i pi k_a n^2) at n in [-L/2, L/2).
    const int half = a.aperture / 2;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const int i = t + T * m;
      const int n = i < N / 2 ? i : i - N;
      v[m] = make_float2(0.f, 0.f);
      if (n >= -half && n < a.aperture - half) v[m] = cconj(unit_of(turns * (unsigned long long)(n * n)));
    }
    line_dft<N>(v, a.tw, sm, t);
    __syncthreads();   // the exchange buffer is reused by the data transform
    float scale = 1.0f;
    if (a.peak_normalise) {
      float mx = 0.f;
#pragma unroll
      for (int m = 0; m < P; ++m) mx = fmaxf(mx, v[m].x * v[m].x + v[m].y * v[m].y);
      if constexpr (T < 32) {
#pragma unroll
        for (int o = T / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      } else {
        constexpr int W = T / 32;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = mx;
        __syncthreads();
        mx = 0.f;
#pragma unroll
        for (int w = 0; w < W; ++w) mx = fmaxf(mx, warp_max[g * W + w]);
      }
      scale = mx > 0.f ? rsqrtf(mx) : 1.0f;
    }
    // The azimuth lines arrive as spectra: times the filter conj(DFT) scale,
    // four at a time to bound live registers.
#pragma unroll
    for (int m0 = 0; m0 < P; m0 += 4) {
      float2 x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = active ? Storage<TIn>::load(in + T * (m0 + i)) : make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        v[m0 + i] = cscale(cconj(cmul(x[i], make_float2(v[m0 + i].x * scale, -v[m0 + i].y * scale))), inv_n);
      asm volatile("" ::: "memory");
    }
  } else {
    // Bulk RCMC of this Doppler bin: y(r) = x(r + s) as exp(+2 pi i q s / N) on
    // the signed frequency q of bin t + T m: the phase of t times that of T m
    // (minus N from the Nyquist bin on), the second shared by the line.
    if (t < P) ramp[g][t] = unit_of(turns * (unsigned long long)(T * t - (t < P / 2 ? 0 : N)));
    if (active) {
#pragma unroll
      for (int m = 0; m < P; ++m) v[m] = Storage<TIn>::load(in + T * m);
    } else {
#pragma unroll
      for (int m = 0; m < P; ++m) v[m] = make_float2(0.f, 0.f);
    }
    line_dft<N>(v, a.tw, sm, t);
    const float2 first = unit_of(turns * (unsigned long long)t);
#pragma unroll
    for (int m = 0; m < P; ++m) {
      float2 h = cmul(first, ramp[g][m]);
      if (m == P / 2 && t == 0) h.y = 0.f;                     // the Nyquist bin: cos(pi s)
      v[m] = cscale(cconj(cmul(v[m], h)), inv_n);
    }
  }
  // the inverse as conj(DFT(conj(.) / N)) (Eq. 1)
  int t2;
  asm volatile("mov.b32 %0, %1;" : "=r"(t2) : "r"(t));
  line_dft<N>(v, a.tw, sm, t2);
  if (active) {
    TOut* out = static_cast<TOut*>(a.out) + line * (long long)N + t;
#pragma unroll
    for (int m = 0; m < P; ++m) Storage<TOut>::store(out + T * m, cconj(v[m]));
  }
}

template <int N, class TS, bool AZIMUTH>
cudaError_t launch_rda_n(const RdaArgs& a, cudaStream_t s) {
  using S = RowShape<N>;
  auto kern = rda_rows_kernel<N, TS, TS, AZIMUTH>;
  static const LaunchSetup setup = setup_kernel(kern, S::kThreads, S::kSmemBytes);
  if (setup.err != cudaSuccess) return setup.err;
  if (a.lines <= 0) return cudaSuccess;
  const long long grid = (a.lines + S::G - 1) / S::G;
  return launch_chained(kern, grid, S::kThreads, S::kSmemBytes, 1, true, s, a);
}

template <class TS, bool AZIMUTH>
cudaError_t launch_rda_typed(int log2n, const RdaArgs& a, cudaStream_t s) {
  switch (log2n) {
    case 8: return launch_rda_n<256, TS, AZIMUTH>(a, s);
    case 9: return launch_rda_n<512, TS, AZIMUTH>(a, s);
    case 10: return launch_rda_n<1024, TS, AZIMUTH>(a, s);
    case 11: return launch_rda_n<2048, TS, AZIMUTH>(a, s);
    case 12: return launch_rda_n<4096, TS, AZIMUTH>(a, s);
    case 13: return launch_rda_n<8192, TS, AZIMUTH>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_rda_lines(const RdaGeometry& geo, bool range_dependent, int n_az, int n_rg,
                             unsigned long long* shift, unsigned long long* rate, cudaStream_t s) {
  const long long grid = (n_az + n_rg + 127) / 128;
  return launch_chained(rda_lines_kernel, grid, 128, 0, 1, true, s, geo, int(range_dependent), n_az, n_rg, shift, rate);
}

cudaError_t launch_rcmc_rows(int log2n, bool f16, const RdaArgs& a, cudaStream_t s) {
  return f16 ? launch_rda_typed<__half2, false>(log2n, a, s) : launch_rda_typed<float2, false>(log2n, a, s);
}

cudaError_t launch_azimuth_rows(int log2n, bool f16, const RdaArgs& a, cudaStream_t s) {
  return f16 ? launch_rda_typed<__half2, true>(log2n, a, s) : launch_rda_typed<float2, true>(log2n, a, s);
}

}  // namespace bfp
