// Entropy phase autofocus: the image entropy of the azimuth-compressed image
// under a per-pulse phase correction, and its gradient by a hand-written
// adjoint that recomputes the forward transforms instead of storing them.
//
// Model (the paper has no autofocus section; this is standard SAR entropy
// autofocus on top of its azimuth compression, Fig. 1):
//   v[r][n] = rc[r][n] exp(-j phi[n])          rc rows: range bin r, pulse n
//   I[r]    = A v[r],  A = IDFT(DFT(.) . Ha)   azimuth compression of one range bin
//   q = |I|^2,  S = sum q,  p = q / S,  E = -sum p ln p = ln S - (1/S) sum q ln q
// Adjoint:
//   G = dE/dI* = -(ln p + E) / S * I           (0 where q = 0)
//   A^H = IDFT(DFT(.) . conj(Ha))              the same chain with the conjugate filter
//   dE/dphi[n] = 2 sum_r Im( conj((A^H G)[r][n]) * v[r][n] )
//
// Kernels (persistent, one group of N/16 threads per range bin, lines held on
// chip exactly as in fft_rows.cuh):
//   af_phase_kernel         e^{-j phi[n]} table
//   af_kernel<kAfEntropy>   per-CTA FP64 partials of S and sum q ln q; for a gradient
//                           it also keeps I[r] (FP32) in scratch, where there is room
//   af_stats_kernel         S, Q, E, ln S (one block, FP64 tree over the partials)
//   af_kernel<kAfAdjoint>   per-CTA partial gradients from the kept I
//   af_kernel<kAfRecompute> the same without scratch: I[r] is computed again
//   af_grad_kernel          sum of the partial gradients in FP64 (32 slices per 32 pulses)
//
// A gradient step costs its transforms: four with I kept, six when it is computed
// again.  Neither pass fills a pipe (entropy and adjoint: issue slots 52 and 53 %
// busy, FMA 44 %, L1 52 and 46 %, at two CTAs of 256 threads per SM).  Keeping I
// costs the entropy pass 11 us of stores and saves the adjoint 77 us (104 instead
// of 181; 4096 x 4096, FP16 rc, GB300).  The whole step: see kAfKeepBytes.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "autofocus.h"
#include "fft_rows.cuh"

namespace bfp {

namespace {

struct AfArgs {
  const void* rc;
  float2* img;           // I [n_rg][n_az]: written by the entropy pass when not null, read by kAfAdjoint
  const float2* ph;      // e^{-j phi[n]}
  const float2* ha;
  const float2* tw;
  long long rows;        // n_rg
  double* stats;         // S, Q, E, ln S
  double* sq_part;       // [grid][2]
  float* g_part;         // [grid][n_az]
  bool prefetch;         // rc in device memory: prefetch each CTA's next rows into L2
};

__global__ void af_phase_kernel(const float* __restrict__ phi, float2* __restrict__ ph, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    float s, c;
    sincosf(phi[i], &s, &c);
    ph[i] = make_float2(c, -s);
  }
}

// One compression of the line held in v with filter h (conjugated if CONJ_H):
// v <- conj(DFT(conj(DFT(v) . h) / N)).
template <int N, bool CONJ_H, bool OPAQUE = false>
__device__ __forceinline__ void af_compress(float2 (&v)[kPointsPerThread], const float2* __restrict__ h,
                                            const float2* __restrict__ tw, float2* sm, int t) {
  constexpr int P = kPointsPerThread, T = N / P;
  const float inv_n = 1.0f / float(N);
  // The second transform runs on an opaque copy of t: the compiler must not
  // keep the first one's shared-memory and twiddle addresses live for it.  With
  // OPAQUE (four transforms in one kernel) so does the first.
  int t1 = t;
  if (OPAQUE) asm volatile("mov.b32 %0, %1;" : "=r"(t1) : "r"(t));
  line_dft<N>(v, tw, sm, t1);
  // Filter loads in groups of four, so the compiler does not hoist all
  // sixteen next to the line (register pressure at 3 CTAs / SM).
#pragma unroll
  for (int m0 = 0; m0 < P; m0 += 4) {
    float2 hv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) hv[i] = __ldg(h + t + T * (m0 + i));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = CONJ_H ? cconj(hv[i]) : hv[i];
      v[m0 + i] = cscale(cconj(cmul(v[m0 + i], f)), inv_n);
    }
    asm volatile("" ::: "memory");
  }
  int t2;
  asm volatile("mov.b32 %0, %1;" : "=r"(t2) : "r"(t));
  line_dft<N>(v, tw, sm, t2);
#pragma unroll
  for (int m = 0; m < P; ++m) v[m] = cconj(v[m]);
}

// Cached loads (not streaming): the backward kernel reads each row twice and
// the second read should come from L2.
__device__ __forceinline__ float2 load_cached(const float2* p) { return __ldg(p); }
__device__ __forceinline__ float2 load_cached(const __half2* p) {
  const unsigned int u = __ldg(reinterpret_cast<const unsigned int*>(p));
  return __half22float2(*reinterpret_cast<const __half2*>(&u));
}

template <int N, class TIn>
__device__ __forceinline__ void af_load(float2 (&v)[kPointsPerThread], const AfArgs& a, long long row, int t,
                                        bool active) {
  constexpr int P = kPointsPerThread, T = N / P;
  const TIn* in = static_cast<const TIn*>(a.rc) + row * N + t;
  // The line first, then its phases four at a time.
#pragma unroll
  for (int m = 0; m < P; ++m) v[m] = active ? load_cached(in + T * m) : make_float2(0.f, 0.f);
#pragma unroll
  for (int m0 = 0; m0 < P; m0 += 4) {
    float2 p[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) p[i] = __ldg(a.ph + t + T * (m0 + i));
#pragma unroll
    for (int i = 0; i < 4; ++i) v[m0 + i] = cmul(v[m0 + i], p[i]);
    asm volatile("" ::: "memory");
  }
}

enum AfPass : int { kAfEntropy = 0, kAfAdjoint = 1, kAfRecompute = 2 };

// Resident CTAs per SM: two of 256 threads at 128 registers, one of 512.  More
// do not help: the entropy pass takes 98 to 102 us a call at two, three or four
// (issue slots 52 % busy at two), the adjoint pass is slower at four (a step
// takes 249 us against 224) and leaves more partial gradients to sum.  The
// number also fixes which rows a CTA's FP32 partial of the entropy adds up.
template <int N, int PASS>
constexpr int af_min_blocks() {
  return RowShape<N>::kThreads >= 512 ? 1 : 2;
}

template <int N, class TIn, int PASS>
__global__ void __launch_bounds__(RowShape<N>::kThreads, af_min_blocks<N, PASS>())
af_kernel(const AfArgs a) {
  using S = RowShape<N>;
  constexpr int P = S::P, T = S::T, G = S::G;
  constexpr bool BACKWARD = PASS != kAfEntropy;
  extern __shared__ float2 smem_af[];
  const int g = threadIdx.x / T;
  const int t = threadIdx.x - g * T;
  float2* sm = smem_af + g * S::kSmemPerLine;
  const long long groups = (a.rows + G - 1) / G;

  float s_acc = 0.f, q_acc = 0.f;
  // Gradient passes: the sums of this thread's pulses t + T m over the group's
  // rows, in registers; kAfRecompute, short of those, keeps them in shared memory.
  constexpr bool kShared = PASS == kAfRecompute;
  float* gsm = reinterpret_cast<float*>(smem_af + (kShared ? G * S::kSmemPerLine : 0)) + g * N;
  float grad[P];
#pragma unroll
  for (int m = 0; m < P; ++m) {
    grad[m] = 0.f;
    if (kShared) gsm[t + T * m] = 0.f;
  }
  float ln_s_minus_e = 0.f, inv_s = 0.f;
  if (BACKWARD) {
    ln_s_minus_e = float(a.stats[3] - a.stats[2]);   // ln S - E
    inv_s = float(1.0 / a.stats[0]);
  }

  for (long long i = blockIdx.x; i < groups; i += gridDim.x) {
    // The adjoint pass takes the rows last written first: those are in L2.
    const long long grp = PASS == kAfAdjoint ? groups - 1 - i : i;
    if (i + gridDim.x < groups && threadIdx.x == 0) {
      // The rows of this CTA's next group, into L2.
      const long long r0 = (PASS == kAfAdjoint ? grp - gridDim.x : grp + gridDim.x) * G;
      const long long cnt = a.rows - r0 < G ? a.rows - r0 : G;
      if (a.prefetch)
        prefetch_l2_bulk(static_cast<const TIn*>(a.rc) + r0 * N, uint32_t(cnt * N * sizeof(TIn)));
      if (PASS == kAfAdjoint) prefetch_l2_bulk(a.img + r0 * N, uint32_t(cnt * N * sizeof(float2)));
    }
    const long long row = grp * G + g;
    const bool active = row < a.rows;
    int ti = t;
    if (PASS == kAfRecompute) asm volatile("mov.b32 %0, %1;" : "=r"(ti) : "r"(t));
    float2 v[P];
    if constexpr (PASS == kAfAdjoint) {
      const float2* img = a.img + row * N + ti;
#pragma unroll
      for (int m = 0; m < P; ++m) v[m] = active ? Storage<float2>::load(img + T * m) : make_float2(0.f, 0.f);
    } else {
      af_load<N, TIn>(v, a, row, ti, active);
      af_compress<N, false, PASS == kAfRecompute>(v, a.ha, a.tw, sm, ti);          // v = I[row]
    }
    if (!BACKWARD) {
      if (active) {
#pragma unroll
        for (int m = 0; m < P; ++m) {
          const float q = v[m].x * v[m].x + v[m].y * v[m].y;
          s_acc += q;
          if (q > 0.f) q_acc += q * logf(q);
        }
        if (a.img != nullptr) {
          float2* img = a.img + row * N + ti;
#pragma unroll
          for (int m = 0; m < P; ++m) img[T * m] = v[m];
        }
      }
    } else {
      // G = -(ln p + E) / S * I, with ln p = ln q - ln S.
#pragma unroll
      for (int m = 0; m < P; ++m) {
        const float q = v[m].x * v[m].x + v[m].y * v[m].y;
        const float w = q > 0.f ? (ln_s_minus_e - logf(q)) * inv_s : 0.f;
        v[m] = cscale(v[m], w);
      }
      af_compress<N, true, PASS == kAfRecompute>(v, a.ha, a.tw, sm, ti);         // v = (A^H G)[row]
      if (active) {
        // v[row] again (from L2), four points at a time to bound live registers.
        const TIn* in = static_cast<const TIn*>(a.rc) + row * N + ti;
#pragma unroll
        for (int m0 = 0; m0 < P; m0 += 4) {
          float2 x[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = cmul(load_cached(in + T * (m0 + j)), __ldg(a.ph + ti + T * (m0 + j)));
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 b = v[m0 + j];
            const float d = 2.f * (b.x * x[j].y - b.y * x[j].x);      // 2 Im(conj(b) x)
            if (kShared) gsm[ti + T * (m0 + j)] += d;
            else grad[m0 + j] += d;
          }
          asm volatile("" ::: "memory");
        }
      }
    }
  }

  if (!BACKWARD) {
    __shared__ double red[2][32];
    double s = s_acc, q = q_acc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s += __shfl_down_sync(0xffffffffu, s, o);
      q += __shfl_down_sync(0xffffffffu, q, o);
    }
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = s;
      red[1][threadIdx.x >> 5] = q;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double ss = 0.0, qq = 0.0;
      for (int w = 0; w < S::kThreads / 32; ++w) {
        ss += red[0][w];
        qq += red[1][w];
      }
      a.sq_part[2 * blockIdx.x] = ss;
      a.sq_part[2 * blockIdx.x + 1] = qq;
    }
  } else {
    // Groups of one CTA cover the same pulses: add their sums, by way of the
    // row buffers (free once every group is past its last exchange).
    float* dst = a.g_part + (long long)blockIdx.x * N;
    if constexpr (G == 1 && !kShared) {
#pragma unroll
      for (int m = 0; m < P; ++m) dst[t + T * m] = grad[m];
    } else {
      __syncthreads();
      if (!kShared) {
#pragma unroll
        for (int m = 0; m < P; ++m) gsm[t + T * m] = grad[m];
        __syncthreads();
      }
      const float* g0 = gsm - g * N;
      for (int i = threadIdx.x; i < N; i += S::kThreads) {
        float acc = 0.f;
#pragma unroll
        for (int gg = 0; gg < G; ++gg) acc += g0[gg * N + i];
        dst[i] = acc;
      }
    }
  }
}

// S and sum q ln q from the per-CTA partials: one block of kAfRedThreads, each
// thread summing a strided share in FP64, then a shuffle and shared-memory
// reduction.
constexpr int kAfRedThreads = 256;

__global__ void __launch_bounds__(kAfRedThreads) af_stats_kernel(const double* __restrict__ sq_part, int grid,
                                                                 double* __restrict__ stats,
                                                                 double* __restrict__ kept,
                                                                 double* __restrict__ entropy) {
  __shared__ double red[2][kAfRedThreads / 32];
  double s = 0.0, q = 0.0;
  for (int b = threadIdx.x; b < grid; b += kAfRedThreads) {
    s += sq_part[2 * b];
    q += sq_part[2 * b + 1];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, o);
    q += __shfl_down_sync(0xffffffffu, q, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s;
    red[1][threadIdx.x >> 5] = q;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    s = 0.0;
    q = 0.0;
    for (int w = 0; w < kAfRedThreads / 32; ++w) {
      s += red[0][w];
      q += red[1][w];
    }
    const double ln_s = s > 0.0 ? log(s) : 0.0;
    const double e = s > 0.0 ? ln_s - q / s : 0.0;
    const double out[4] = {s, q, e, ln_s};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      stats[i] = out[i];
      if (kept != nullptr) kept[i] = out[i];
    }
    if (entropy != nullptr) *entropy = e;
  }
}

// grad[i] = sum over CTAs b of g_part[b][i], in FP64: a block covers 32
// consecutive pulses (one per lane: coalesced rows) with 32 warps splitting
// the CTAs between them, then adds the 32 partial sums.
constexpr int kAfGradSlices = 32;

// scale (may be null) multiplies the result, as FP32; `kept` statistics go to
// stats_out as well.
__global__ void __launch_bounds__(32 * kAfGradSlices) af_grad_kernel(const float* __restrict__ g_part, int grid,
                                                                    int n, float* __restrict__ grad,
                                                                    const double* __restrict__ scale,
                                                                    const double* __restrict__ kept,
                                                                    double* __restrict__ stats_out) {
  if (stats_out != nullptr && blockIdx.x == 0 && threadIdx.x < 4) stats_out[threadIdx.x] = kept[threadIdx.x];
  __shared__ double red[kAfGradSlices][32];
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  double acc = 0.0;
  if (i < n)
    for (int b = slice; b < grid; b += kAfGradSlices) acc += g_part[(long long)b * n + i];
  red[slice][lane] = acc;
  __syncthreads();
  if (slice == 0 && i < n) {
    double t = 0.0;
#pragma unroll
    for (int k = 0; k < kAfGradSlices; ++k) t += red[k][lane];
    grad[i] = scale != nullptr ? float(*scale) * float(t) : float(t);
  }
}

template <int N, class TIn, int PASS>
cudaError_t launch_af_n(const AfArgs& a, int* grid_out, cudaStream_t s) {
  using S = RowShape<N>;
  auto kern = af_kernel<N, TIn, PASS>;
  constexpr size_t kBytes = S::kSmemBytes + (PASS == kAfRecompute ? size_t(S::G) * N * sizeof(float) : 0);
  // One-time, thread-safe set-up (function-local static): resident CTAs,
  // capped by the workspace's partial-gradient slots.
  static const LaunchSetup setup = setup_kernel(kern, S::kThreads, kBytes);
  if (setup.err != cudaSuccess) return setup.err;
  const int cap = setup.resident < kAfMaxCtas ? setup.resident : kAfMaxCtas;
  const long long groups = (a.rows + S::G - 1) / S::G;
  const int grid = int(groups < cap ? groups : cap);
  *grid_out = grid;
  kern<<<grid, S::kThreads, kBytes, s>>>(a);
  return cudaGetLastError();
}

template <class TIn, int PASS>
cudaError_t launch_af_typed(int log2n, const AfArgs& a, int* grid, cudaStream_t s) {
  switch (log2n) {
    case 8: return launch_af_n<256, TIn, PASS>(a, grid, s);
    case 9: return launch_af_n<512, TIn, PASS>(a, grid, s);
    case 10: return launch_af_n<1024, TIn, PASS>(a, grid, s);
    case 11: return launch_af_n<2048, TIn, PASS>(a, grid, s);
    case 12: return launch_af_n<4096, TIn, PASS>(a, grid, s);
    case 13: return launch_af_n<8192, TIn, PASS>(a, grid, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int PASS>
cudaError_t launch_af(int log2n, bool rc16, const AfArgs& a, int* grid, cudaStream_t s) {
  return rc16 ? launch_af_typed<__half2, PASS>(log2n, a, grid, s) : launch_af_typed<float2, PASS>(log2n, a, grid, s);
}

}  // namespace

size_t af_workspace_bytes(long long n_az) {
  return size_t(kAfMaxCtas) * 2 * sizeof(double) + size_t(kAfMaxCtas) * size_t(n_az) * sizeof(float) +
         size_t(n_az) * sizeof(float2) + size_t(kAfMaxCtas) * sizeof(float) + 256;
}

AfWorkspaceLayout af_workspace_layout(void* workspace, long long n_az) {
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  AfWorkspaceLayout l;
  l.sq_part = reinterpret_cast<double*>(ws);
  ws += size_t(kAfMaxCtas) * 2 * sizeof(double);
  l.g_part = reinterpret_cast<float*>(ws);
  ws += size_t(kAfMaxCtas) * size_t(n_az) * sizeof(float);
  l.ph = reinterpret_cast<float2*>(ws);
  ws += size_t(n_az) * sizeof(float2);
  l.q_part = reinterpret_cast<float*>(ws);
  ws += size_t(kAfMaxCtas) * sizeof(float);
  l.qmax = reinterpret_cast<float*>(ws);
  return l;
}

cudaError_t af_phase_table(const float* phi, float2* ph, long long n_az, cudaStream_t s) {
  af_phase_kernel<<<int((n_az + 255) / 256), 256, 0, s>>>(phi, ph, int(n_az));
  return cudaGetLastError();
}

cudaError_t af_entropy_stats(const double* sq_part, int grid, double* stats, cudaStream_t s, double* kept,
                             double* entropy) {
  af_stats_kernel<<<1, kAfRedThreads, 0, s>>>(sq_part, grid, stats, kept, entropy);
  return cudaGetLastError();
}

cudaError_t af_gradient_sum(const float* g_part, int grid, int n_az, float* grad, cudaStream_t s,
                            const double* scale, const double* kept, double* stats_out) {
  af_grad_kernel<<<(n_az + 31) / 32, 32 * kAfGradSlices, 0, s>>>(g_part, grid, n_az, grad, scale, kept, stats_out);
  return cudaGetLastError();
}

namespace {

// The kept state: the four statistics, then the image.
struct AfState {
  double* stats;
  float2* image;
};
AfState af_state(void* state) {
  if (state == nullptr) return {nullptr, nullptr};
  unsigned char* p = static_cast<unsigned char*>(state);
  return {reinterpret_cast<double*>(p), reinterpret_cast<float2*>(p + kAfStateHead)};
}

AfArgs af_args(int log2n, const void* rc, const float2* ha, const float2* tw, long long n_rg, double* stats,
               void* workspace, float2* image, bool prefetch) {
  const AfWorkspaceLayout l = af_workspace_layout(workspace, 1LL << log2n);
  AfArgs a;
  a.rc = rc;
  a.img = image;
  a.ph = l.ph;
  a.ha = ha;
  a.tw = tw;
  a.rows = n_rg;
  a.stats = stats;
  a.sq_part = l.sq_part;
  a.g_part = l.g_part;
  a.prefetch = prefetch;
  return a;
}

}  // namespace

cudaError_t launch_autofocus_entropy(int log2n, bool rc16, const void* rc, const float* phi, const float2* ha,
                                     const float2* tw, long long n_rg, double* stats, void* workspace,
                                     void* state, double* entropy, bool prefetch, cudaStream_t s) {
  const AfState keep = af_state(state);
  const AfArgs a = af_args(log2n, rc, ha, tw, n_rg, stats, workspace, keep.image, prefetch);
  cudaError_t e = af_phase_table(phi, af_workspace_layout(workspace, 1LL << log2n).ph, 1LL << log2n, s);
  if (e != cudaSuccess) return e;
  int grid = 0;
  if ((e = launch_af<kAfEntropy>(log2n, rc16, a, &grid, s)) != cudaSuccess) return e;
  return af_entropy_stats(a.sq_part, grid, stats, s, keep.stats, entropy);
}

cudaError_t launch_autofocus_gradient(int log2n, bool rc16, const void* rc, const float* phi, const float2* ha,
                                      const float2* tw, long long n_rg, double* stats, float* grad, void* workspace,
                                      void* state, const double* scale, bool prefetch, cudaStream_t s) {
  const AfState kept = af_state(state);
  const AfArgs a = af_args(log2n, rc, ha, tw, n_rg, state != nullptr ? kept.stats : stats, workspace, kept.image,
                           prefetch);
  cudaError_t e = cudaSuccess;
  if (phi != nullptr)
    e = af_phase_table(phi, af_workspace_layout(workspace, 1LL << log2n).ph, 1LL << log2n, s);
  if (e != cudaSuccess) return e;
  int grid = 0;
  e = state != nullptr ? launch_af<kAfAdjoint>(log2n, rc16, a, &grid, s)
                       : launch_af<kAfRecompute>(log2n, rc16, a, &grid, s);
  if (e != cudaSuccess) return e;
  return af_gradient_sum(a.g_part, grid, 1 << log2n, grad, s, scale, kept.stats, state != nullptr ? stats : nullptr);
}

}  // namespace bfp
