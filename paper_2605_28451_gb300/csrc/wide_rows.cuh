// Dense row transforms with 32 or 64 points per thread: lines of 512 ... 16384
// points in two or three passes of radix 16, 32 or 64.
//
// The 16-point-per-thread kernel of fft_rows.cuh takes a 4096-point line
// through three radix-16 passes: two exchanges through shared memory and two
// sets of twiddle loads, 13.75 L1 / shared-memory wavefronts and 48
// instructions per thread for every point a thread moves through them; it is
// bound by those two pipes (78 % and 61 % busy) at 63 % of the HBM copy rate.
// With 64 points per thread the line is 64 x 64: one exchange, one set of
// twiddles, 8 wavefronts and 39 instructions a point.  Passes (N = P * ...):
//   512 = 32 x 16, 1024 = 32 x 32 (32 points per thread; a line is a half or a
//   whole warp, so the exchange needs no CTA barrier), 2048 = 64 x 32 (one
//   warp), 4096 = 64 x 64 (two warps), 8192 = 32 x 16 x 16 and 16384 =
//   32 x 32 x 16 (one CTA of 256 or 512 threads).
// Measured on GB300, FP16 storage, 2^27 points, forward, against the
// 16-point kernel (algorithmic GB/s; the copy rate is 6790): 512: 4720 ->
// 6390, 1024: 4440 -> 6650, 2048: 4360 -> 5560, 4096: 4130 -> 5030, 8192:
// 2880 -> 3640, 16384: 2300 -> 2870.  Lines up to 1024 points then run at the
// copy rate; 2048 and 4096 are left with 12 warps per SM (the registers of 64
// points a thread), too few to cover the exchange and twiddle latencies.
//
// Exchange.  The first pass writes its R = P outputs of butterfly t to points
// t P + r with 16-byte stores, two slots of padding every P points (so eight
// lanes hit 32 banks); later passes write and read consecutive points across
// a warp.  kSplit sends the real and then the imaginary parts through half the
// shared memory: for those shapes the larger L1 that this leaves (the 32 KB
// twiddle table stays in it) is worth two more barriers.
//
// Twiddles.  Table per length, FP64 sincospi rounded once, pass-major: for the
// pass with sub-length Ns and radix R, W_{Ns R}^{k r} sits at entry
// off + 2 ((r / 2) Ns + k) + (r & 1), off = 0 for the second pass and Ns for the
// third, so one 16-byte load fetches the twiddles of points r and r + 1.
//
// Included by fft_rows.cuh, whose RowArgs and launch helpers it uses.
#pragma once

namespace bfp {

constexpr int kWideMinLog2 = 9, kWideMaxLog2 = 14;

template <int N>
struct WideShape {
  static constexpr int P = (N == 2048 || N == 4096) ? 64 : 32;   // points per thread
  static constexpr int T = N / P;                                // threads per line
  static constexpr int kThreads = T < 64 ? 64 : T;               // threads per CTA
  static constexpr int G = kThreads / T;                         // lines per CTA
  // Resident CTAs asked of the register allocator: 168 registers for 64
  // points a thread, 96 (T <= 32) or 128 for 32 points; no spills in the
  // plain transforms.
  static constexpr int kMinBlocks = P == 64 ? 6 : T <= 32 ? 10 : T == 256 ? 2 : 1;
};

// Radix of the pass with sub-length Ns.
template <int N>
__host__ __device__ constexpr int wide_radix(int ns) {
  const int p = WideShape<N>::P, left = N / ns;
  return left <= p ? left : left >= 16 * p || left == p * p ? p : 16;
}

template <int N, bool SPLIT>
__host__ __device__ constexpr int wide_line_floats() {
  return SPLIT ? N + 4 * (N / WideShape<N>::P) : 2 * N + 4 * (N / WideShape<N>::P);
}
template <int N>
__host__ __device__ constexpr int wide_pad(int i) { return i + 2 * (i / WideShape<N>::P); }

// Barrier of the threads that share a line.
template <int N>
__device__ __forceinline__ void wide_sync() {
  if constexpr (WideShape<N>::T <= 32) __syncwarp();
  else __syncthreads();
}

struct WideNoHook {
  __device__ __forceinline__ void operator()() const {}
};

template <int N, int Ns, bool SPLIT, bool FINE>
struct WidePass {
  static constexpr int P = WideShape<N>::P, T = WideShape<N>::T;
  static constexpr int R = wide_radix<N>(Ns);
  static constexpr int B = P / R;
  static constexpr bool kLast = Ns * R == N;

  // v[m] = point t + T m of this pass, as read from the exchange, times its
  // twiddle: butterfly b takes points m = b + B r.
  __device__ __forceinline__ static void twiddle(float2 (&v)[P], const float4* __restrict__ tw, int t) {
    constexpr int kOff = Ns == P ? 0 : Ns;
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const float4* row = tw + kOff / 2 + ((t + T * b) & (Ns - 1));
#pragma unroll
      for (int h = 0; h < R / 2; ++h) {
        const float4 w = __ldg(row + h * Ns);
        if (h > 0) v[b + B * 2 * h] = cmul(v[b + B * 2 * h], make_float2(w.x, w.y));
        v[b + B * (2 * h + 1)] = cmul(v[b + B * (2 * h + 1)], make_float2(w.z, w.w));
      }
    }
  }

  // The line from this pass on: v[m] = twiddled point t + T m -> X[t + T m].
  // war: the exchange buffer may still be being read.  after_last_read runs
  // once the thread has read the last exchange back.
  template <class H>
  __device__ __forceinline__ static void run(float2 (&v)[P], const float4* __restrict__ tw, float* __restrict__ sm,
                                             int t, bool war, const H& after_last_read) {
    if constexpr (SPLIT && !kLast) {
      static_assert(Ns == 1 && R == P && P % 4 == 0 && WidePass<N, R, SPLIT, FINE>::kLast, "split exchange: two passes");
      Dft<R, FINE>::run(v);
      if (war) wide_sync<N>();
      constexpr int kPitch = P + 4;
      float4* dst = reinterpret_cast<float4*>(sm + t * kPitch);
#pragma unroll
      for (int r = 0; r < P; r += 4) dst[r / 4] = make_float4(v[r].x, v[r + 1].x, v[r + 2].x, v[r + 3].x);
      wide_sync<N>();
      float re[P];
#pragma unroll
      for (int m = 0; m < P; ++m) re[m] = sm[t + (T * m / P) * kPitch + T * m % P];
      wide_sync<N>();
#pragma unroll
      for (int r = 0; r < P; r += 4) dst[r / 4] = make_float4(v[r].y, v[r + 1].y, v[r + 2].y, v[r + 3].y);
      wide_sync<N>();
#pragma unroll
      for (int m = 0; m < P; ++m) v[m] = make_float2(re[m], sm[t + (T * m / P) * kPitch + T * m % P]);
      WidePass<N, R, SPLIT, FINE>::twiddle(v, tw, t);
      after_last_read();
      WidePass<N, R, SPLIT, FINE>::run(v, tw, sm, t, true, after_last_read);
    } else {
      if constexpr (!kLast) {
        if (war) wide_sync<N>();
      }
      float2* sm2 = reinterpret_cast<float2*>(sm);
      float2 o[P];
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int j = t + T * b;
        float2 u[R];
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = v[b + B * r];
        Dft<R, FINE>::run(u);
        if constexpr (kLast) {
#pragma unroll
          for (int r = 0; r < R; ++r) o[b + B * r] = u[r];
        } else if constexpr (Ns == 1) {
          float4* dst = reinterpret_cast<float4*>(sm2 + wide_pad<N>(j * R));
#pragma unroll
          for (int r = 0; r < R; r += 2) dst[r / 2] = make_float4(u[r].x, u[r].y, u[r + 1].x, u[r + 1].y);
        } else {
          const int base = (j / Ns) * Ns * R + (j & (Ns - 1));
#pragma unroll
          for (int r = 0; r < R; ++r) sm2[wide_pad<N>(base + r * Ns)] = u[r];
        }
      }
      if constexpr (kLast) {
#pragma unroll
        for (int m = 0; m < P; ++m) v[m] = o[m];
      } else {
        using Next = WidePass<N, Ns * R, SPLIT, FINE>;
        wide_sync<N>();
#pragma unroll
        for (int m = 0; m < P; ++m) v[m] = sm2[wide_pad<N>(t + T * m)];
        Next::twiddle(v, tw, t);
        if constexpr (Next::kLast) after_last_read();
        Next::run(v, tw, sm, t, true, after_last_read);
      }
    }
  }
};

// Forward DFT of the line held in v (v[m] = x[t + T m] -> X[t + T m]); FINE: see
// mul_root.
template <int N, bool SPLIT, bool FINE, class H = WideNoHook>
__device__ __forceinline__ void wide_dft(float2 (&v)[WideShape<N>::P], const float4* __restrict__ tw,
                                         float* __restrict__ sm, int t, bool war, const H& after_last_read = H()) {
  WidePass<N, 1, SPLIT, FINE>::run(v, tw, sm, t, war, after_last_read);
}

// v <- conj(v h) / N (Eq. 1's shift and conjugation behind the filter), h the
// thread's first filter point.  Loads go in groups of eight, for the short
// lines one group ahead of the products; more in flight do not fit beside the
// line's registers (nor does the second group at 8192 points and more, 3 %
// slower with it).  No __restrict__: an earlier kernel may have written h (see
// chain_begin).
template <int N>
__device__ __forceinline__ void wide_filter(float2 (&v)[WideShape<N>::P], const float2* h) {
  constexpr int P = WideShape<N>::P, T = WideShape<N>::T;
  constexpr float kInvN = 1.0f / float(N);
  constexpr int kAhead = N <= 4096 ? 8 : 0;
  float2 w[2][8];
#pragma unroll
  for (int i = 0; i < kAhead; ++i) w[0][i] = h[T * i];
#pragma unroll
  for (int m0 = 0; m0 < P; m0 += 8) {
    const int load = m0 + kAhead;
    if (load < P) {
#pragma unroll
      for (int i = 0; i < 8; ++i) w[(load / 8) & 1][i] = h[T * (load + i)];
    }
    if (kAhead > 0) asm volatile("" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i)
      v[m0 + i] = cmul_parts(cmul(v[m0 + i], w[(m0 / 8) & 1][i]), make_float2(kInvN, -kInvN));
    if (kAhead == 0) asm volatile("" ::: "memory");
  }
}

// What precedes and follows the transform(s): block exponents, Eq. 1's
// conjugate and 1/N, the output conjugate.
template <int N, int MODE, bool SCALED>
__device__ __forceinline__ void wide_head(float2 (&v)[WideShape<N>::P], const RowArgs& a) {
  constexpr int P = WideShape<N>::P;
  constexpr float kInvN = 1.0f / float(N);
  if constexpr (SCALED || MODE == kInverse) {
    const float s = (SCALED ? a.in_scale : 1.0f) * (MODE == kInverse ? kInvN : 1.0f);   // powers of two: exact
    const float2 f = make_float2(s, MODE == kInverse ? -s : s);
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = cmul_parts(v[m], f);
  }
}
template <int N, int MODE, bool SCALED>
__device__ __forceinline__ void wide_tail(float2 (&v)[WideShape<N>::P], const RowArgs& a) {
  constexpr int P = WideShape<N>::P;
  if constexpr (SCALED) {
    const float2 f = make_float2(a.out_scale, MODE == kForward ? a.out_scale : -a.out_scale);
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = cmul_parts(v[m], f);
  } else if constexpr (MODE != kForward) {
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = cconj(v[m]);
  }
}

// Shapes whose exchange is split (see the top): 4096 points forward 4810 ->
// 5030 GB/s; 4096 points inverse and 2048 points measured 1 to 4 % slower
// with it.
template <int N, int MODE>
constexpr bool kWideSplit = N == 4096 && MODE == kForward;

// Which lines this kernel takes, FP16 storage unless said (16-point kernel's
// time over this one's, GB300):
//   512, 1024, 8192, 16384 points: all (batches of 2^18 ... 2^26 points: 1.07
//     to 1.50, FP32 storage of 512 and 1024 points 0.99 to 1.31).
//   2048 and 4096 points: 64 points a thread make one line slow (4.4 against
//     3.6 us for 128 lines of 2048), so only batches that fill the GPU with
//     lines: 2048 points 0.90 at 512 lines, 1.07 at 1280, 1.17 at 32769; 4096
//     points 0.76 at 256, 1.00 at 1024, 1.10 at 4097, 1.18 at 16385.  Not with
//     FP32 storage (0.85 to 1.0: HBM-bound in both) and not for
//     forward-filter-inverse lines (0.95 at 1024, 1.07 at 16385 lines; 0.92 to
//     1.00 with a filter per line).
template <int N, class TIn, int MODE>
constexpr bool kWideOffered = WideShape<N>::P == 32 || (MODE != kCompress && !std::is_same<TIn, float2>::value);
template <int N>
constexpr int kWideLinesPerSm = N == 2048 ? 8 : N == 4096 ? 12 : 0;   // at least: 1216 and 1824 lines on 152 SMs

template <int N, class TIn, class TOut, int MODE, bool SCALED>
__global__ void __launch_bounds__(WideShape<N>::kThreads, WideShape<N>::kMinBlocks)
fft_wide_kernel(const RowArgs a) {
  using S = WideShape<N>;
  constexpr int P = S::P, T = S::T, G = S::G;
  constexpr bool kSplit = kWideSplit<N, MODE>;
  constexpr bool kFine = std::is_same<TOut, float2>::value;
  static_assert(kWideOffered<N, TIn, MODE>, "see kWideOffered");
  extern __shared__ float4 smem_wide[];
  chain_begin();
  const int g = threadIdx.x / T;
  const int t = threadIdx.x - g * T;
  const long long line = (long long)blockIdx.x * G + g;
  const bool active = line < a.lines;
  float* sm = reinterpret_cast<float*>(smem_wide) + g * wide_line_floats<N, kSplit>();
  float2 v[P];
  if (active) {
    if (a.pf_ahead > 0) {   // the lines of the CTA one resident wave later, into L2 (as fft_rows_kernel)
      const long long l0 = ((long long)blockIdx.x + a.pf_ahead) * G;
      if (a.line_off == nullptr) {
        const long long cnt = a.lines - l0 < G ? a.lines - l0 : G;
        if (threadIdx.x == 0 && cnt > 0)
          prefetch_l2_bulk(static_cast<const TIn*>(a.in) + l0 * N, uint32_t(cnt * N * sizeof(TIn)));
      } else if (t == 0 && l0 + g < a.lines) {
        prefetch_l2_bulk(static_cast<const TIn*>(a.in) + a.line_off[l0 + g], uint32_t(N * sizeof(TIn)));
      }
    }
    // This line's own filter is read once, from HBM, after the first transform.
    if (MODE == kCompress && a.h_prefetch && t == 0)
      prefetch_l2_bulk(a.h + line * a.h_stride, uint32_t(N * sizeof(float2)));
    const TIn* in = static_cast<const TIn*>(a.in) + line_start(a, line, a.in_stride) + t;
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = Storage<TIn>::load(in + T * m);
  } else {
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = make_float2(0.f, 0.f);
  }
  wide_head<N, MODE, SCALED>(v, a);
  if constexpr (MODE == kCompress) {
    const float2* h = a.h + (active ? line : 0) * a.h_stride + t;
    if constexpr (N <= 4096) {
      // One copy of the transform's code, run twice: two copies miss the
      // instruction cache (1024 points: 0.338 -> 0.321 ms per 2^27 points; the
      // longer lines' CTAs of 256 and 512 threads keep together and do not).
#pragma unroll 1
      for (int it = 0; it < 2; ++it) {
        wide_dft<N, false, kFine>(v, a.tw_wide, sm, t, it > 0);
        if (it == 0) wide_filter<N>(v, h);
      }
    } else {
      wide_dft<N, false, kFine>(v, a.tw_wide, sm, t, false);
      wide_filter<N>(v, h);
      int t2;   // opaque copy: the first transform's addresses are not kept live for the second
      asm volatile("mov.b32 %0, %1;" : "=r"(t2) : "r"(t));
      wide_dft<N, false, kFine>(v, a.tw_wide, sm, t2, true);
    }
  } else {
    wide_dft<N, kSplit, kFine>(v, a.tw_wide, sm, t, false);
  }
  wide_tail<N, MODE, SCALED>(v, a);
  if (active) {
    TOut* out = static_cast<TOut*>(a.out) + line_start(a, line, a.out_stride) + t;
#pragma unroll
    for (int m = 0; m < P; ++m) Storage<TOut>::store(out + T * m, v[m]);
    check_finite<Storage<TOut>, P>(a.finite_flag, [&](int m) { return v[m]; });
  }
}

// Lines of 16384 points, one CTA per SM: nothing else on the SM covers the
// line's load, so the CTAs are persistent and the next line arrives by bulk
// copy in the exchange buffer itself, which is free from the last exchange's
// reads on (FP16: 2600 -> 2880 GB/s, FP32: 4410 -> 5060 over 2^27 points).
// Smaller lines have other CTAs on the SM and measured slower this way.
// Waits are bounded: on expiry the CTA records a timeout, waits once more
// (bounded) for the copy it still has in flight and returns.
template <int N, class TIn, class TOut, int MODE, bool SCALED>
__global__ void __launch_bounds__(WideShape<N>::kThreads, WideShape<N>::kMinBlocks)
fft_wide_stream_kernel(const RowArgs a) {
  using S = WideShape<N>;
  constexpr int P = S::P, T = S::T;
  constexpr bool kFine = std::is_same<TOut, float2>::value;
  static_assert(S::G == 1 && T > 32 && MODE != kCompress, "one line per CTA");
  static_assert(N * sizeof(TIn) <= wide_line_floats<N, false>() * sizeof(float), "the line fits the exchange buffer");
  extern __shared__ float4 smem_wide[];
  __shared__ __align__(8) uint64_t bar;
  chain_begin();
  float* sm = reinterpret_cast<float*>(smem_wide);
  auto issue = [&](long long l) {
    mbar_arrive_expect_tx(&bar, uint32_t(N * sizeof(TIn)));
    bulk_load(sm, static_cast<const TIn*>(a.in) + line_start(a, l, a.in_stride), uint32_t(N * sizeof(TIn)), &bar);
  };
  long long line = blockIdx.x;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_proxy_async_shared();
    if (line < a.lines) issue(line);
  }
  __syncthreads();
  uint32_t phase = 0;
#pragma unroll 1
  for (; line < a.lines; line += gridDim.x) {
    const bool arrived = mbar_wait_bounded(&bar, phase, a.status);
    int t;   // opaque per iteration: no address arithmetic carried across the loop
    asm volatile("mov.b32 %0, %1;" : "=r"(t) : "r"(int(threadIdx.x)));
    float2 v[P];
    const TIn* staged = reinterpret_cast<const TIn*>(sm) + t;
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = Storage<TIn>::load_smem(staged + T * m);
    // All threads agree on a timeout, and have read the staged line.
    if (__syncthreads_or(!arrived)) {
      if (threadIdx.x == 0) mbar_wait_bounded(&bar, phase, nullptr);
      __syncthreads();
      return;
    }
    phase ^= 1;
    wide_head<N, MODE, SCALED>(v, a);
    wide_dft<N, false, kFine>(v, a.tw_wide, sm, t, false, [&]() {
      __syncthreads();
      if (threadIdx.x == 0 && line + gridDim.x < a.lines) {
        fence_proxy_async_shared();
        issue(line + gridDim.x);
      }
    });
    wide_tail<N, MODE, SCALED>(v, a);
    TOut* out = static_cast<TOut*>(a.out) + line_start(a, line, a.out_stride) + t;
#pragma unroll
    for (int m = 0; m < P; ++m) Storage<TOut>::store(out + T * m, v[m]);
    check_finite<Storage<TOut>, P>(a.finite_flag, [&](int m) { return v[m]; });
  }
}

template <int N, class TIn, class TOut, int MODE, bool SCALED>
cudaError_t launch_wide_n(const RowArgs& a, cudaStream_t stream, bool l2_prefetch) {
  using S = WideShape<N>;
  if constexpr (N == 16384 && MODE != kCompress) {
    // Bulk copies need device memory and 16-byte aligned lines (a stride of N).
    if (l2_prefetch && a.in_stride == N) {
      constexpr size_t kBytes = wide_line_floats<N, false>() * sizeof(float);
      auto kern = fft_wide_stream_kernel<N, TIn, TOut, MODE, SCALED>;
      static const LaunchSetup setup = setup_kernel(kern, S::kThreads, kBytes);
      if (setup.err != cudaSuccess) return setup.err;
      if (a.lines <= 0) return cudaSuccess;
      const int grid = int(a.lines < setup.resident ? a.lines : setup.resident);
      return launch_chained(kern, grid, S::kThreads, kBytes, 1, true, stream, a);
    }
  }
  constexpr size_t kBytes = size_t(S::G) * wide_line_floats<N, kWideSplit<N, MODE>>() * sizeof(float);
  auto kern = fft_wide_kernel<N, TIn, TOut, MODE, SCALED>;
  static const LaunchSetup setup = setup_kernel(kern, S::kThreads, kBytes);
  if (setup.err != cudaSuccess) return setup.err;
  if (a.lines <= 0) return cudaSuccess;
  const long long grid = (a.lines + S::G - 1) / S::G;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  RowArgs b = a;
  b.pf_ahead = l2_prefetch && a.in_stride == N ? setup.resident : 0;
  return launch_chained(kern, grid, S::kThreads, kBytes, 1, true, stream, b);
}

}  // namespace bfp
