// Lines of 32768 and 65536 points, N = A * 1024 (A = 32, 64), over a
// thread-block cluster of A / 8 CTAs of 128 threads, 64 points per thread.
//
// With n = n2 + 1024 n1 and k = k1 + A k2:
//   X[k1 + A k2] = sum_n2 W_1024^{n2 k2} W_N^{n2 k1} sum_n1 x[n2 + 1024 n1] W_A^{n1 k1}.
// Columns: CTA c loads the columns n2 in [c W, (c + 1) W), W = 1024 / (A / 8),
//   runs their A-point DFTs in registers (one column of 64 or two of 32 a
//   thread), multiplies by W_N^{n2 k1} and sends row k1 to CTA k1 / 8 with
//   asynchronous remote stores counted on that CTA's mbarrier.
// Rows: every CTA holds eight consecutive rows k1 = 8 c ... 8 c + 7 and
//   transforms them as 1024 = 64 x 16: sixteen threads a row for the radix-64
//   pass, then, through shared memory, eight rows across eight lanes for the
//   radix-16 pass, so that the results X[8 c ... 8 c + 7 + A k2] leave as full
//   32-byte sectors (FP16) in natural order with no second exchange.
// The only exchange between CTAs is the row hand-over; it waits on data, not on
// a cluster barrier.
//
// The four-step kernel of fft_rows.cuh (16 CTAs of 4096 points, 16 points a
// thread, N1 x 4096) needs a second exchange of the whole line between CTAs to
// store in natural order, and three shared-memory passes where this one has
// two.  Measured on GB300 (ms, four-step -> this kernel; 2^27 points, FP32
// 2^26): 65536 points FP16 0.689 -> 0.447, FP32 0.528 -> 0.264, E4M3 0.658 ->
// 0.475, FP16 with the row exchange in FP16 words 0.614 -> 0.401; 32768 points
// FP16 0.628 -> 0.416, FP32 0.451 -> 0.244.  Its stalls are the loads of the
// line and of the factors (three CTAs per SM, 168 registers a thread, are too
// few to cover them) and the hand-over itself: without any arithmetic the same
// data movement takes 0.39 ms.
#pragma once

namespace bfp {

template <int N>
struct LongShape {
  static constexpr int A = N / 1024;           // column length, rows
  static constexpr int C = A / 8;              // CTAs per line (cluster size)
  static constexpr int W = 1024 / C;           // columns per CTA
  static constexpr int kThreads = 128, P = 64;
  static constexpr int kCols = P / A;          // columns per thread
  static constexpr int kRowPitch = 1024 + 2 * 16 + 2;   // padded row of the radix-16 pass (banks: 2 per row)
  static constexpr size_t kSmemBytes = size_t(8) * kRowPitch * sizeof(float2);
  static_assert(W == kThreads * kCols, "one thread per kCols columns");
};

// A line is read once: no L1 allocation, which leaves L1 to the tables (the
// three CTAs leave it about 28 KB; 5 % faster so).
template <class T>
__device__ __forceinline__ float2 load_once(const T* p) {
  if constexpr (sizeof(T) == 8) {
    float2 r;
    asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
  } else if constexpr (sizeof(T) == 4) {
    uint32_t r;
    asm volatile("ld.global.L1::no_allocate.b32 %0, [%1];" : "=r"(r) : "l"(p));
    return bits_half2(r);
  } else {
    T r;
    asm volatile("ld.global.L1::no_allocate.b16 %0, [%1];" : "=h"(r.bits) : "l"(p));
    return Storage<T>::load_smem(&r);
  }
}

// The A-point DFT of z over n1 with output k1 times w^{k1}, w = W_N^{n2}: the
// DFT ends with radix-R2 butterflies over r1 at fixed k2 (k1 = k2 + 8 q), so
// w^{k2} goes onto a butterfly's inputs and w^{8 q} onto its outputs.  That
// takes 7 + A / 8 - 1 factors per column from the table instead of A - 1: the
// full table is twice the line's bytes through L2, and the kernel waits for
// those loads long before it runs out of FMA slots (FP16, 65536 points, 2048
// lines: 0.492 ms with it).
//   f[0 .. 7): w^1 ... w^7;  f[7 .. 7 + A / 8 - 1): w^8, w^16, ...
template <int A, bool FINE, class F>
__device__ __forceinline__ void twiddled_column_dft(float2 (&z)[A], const float2 (&f)[6 + A / 8], const F& emit) {
  constexpr int R2 = A / 8;                      // radix of the last butterflies: 8 or 4
  dft8_column<0, R2, FINE>(z);
  dft8_column<1, R2, FINE>(z);
  dft8_column<2, R2, FINE>(z);
  dft8_column<3, R2, FINE>(z);
  if constexpr (R2 == 8) {
    dft8_column<4, R2, FINE>(z);
    dft8_column<5, R2, FINE>(z);
    dft8_column<6, R2, FINE>(z);
    dft8_column<7, R2, FINE>(z);
  }
#pragma unroll
  for (int k2 = 0; k2 < 8; ++k2) {
    float2 x[R2];
#pragma unroll
    for (int i = 0; i < R2; ++i) x[i] = k2 == 0 ? z[i] : cmul(z[R2 * k2 + i], f[k2 - 1]);
    Dft<R2>::run(x);
#pragma unroll
    for (int q = 0; q < R2; ++q) emit(k2 + 8 * q, q == 0 ? x[0] : cmul(x[q], f[6 + q]));
  }
}

template <int N, class TS, int MODE, bool SCALED, bool H16ROW>
__global__ void __launch_bounds__(128, 3) fft_long_kernel(const RowArgs a) {
  using S = LongShape<N>;
  constexpr int A = S::A, C = S::C, P = S::P;
  constexpr float kInvN = 1.0f / float(N);
  constexpr bool kFine = std::is_same<TS, float2>::value;   // see mul_root
  extern __shared__ float4 smem_long[];
  __shared__ __align__(8) uint64_t bar;
  chain_begin();
  float2* sm = reinterpret_cast<float2*>(smem_long);
  const int u = threadIdx.x;
  const int c = int(cooperative_groups::this_cluster().block_rank());
  const long long line = blockIdx.x / C;
  const TS* in = static_cast<const TS*>(a.in) + line_start(a, line, a.in_stride);
  TS* out = static_cast<TS*>(a.out) + line_start(a, line, a.out_stride);
  constexpr uint32_t kWord = H16ROW ? 4 : 8;   // bytes of a point in the row hand-over
  if (u == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_arrive_expect_tx(&bar, 8192 * kWord);
    if (a.pf_ahead > 0 && line + a.pf_ahead < a.lines)
      prefetch_l2_bulk(static_cast<const TS*>(a.in) + line_start(a, line + a.pf_ahead, N) + c * 8192,
                       uint32_t(8192 * sizeof(TS)));
  }
  // Every CTA running and every mbarrier initialised before the first send
  // (the initialisation has its own release fence); the loads are issued in
  // between.
  cluster_arrive_relaxed();
  float2 v[P];
#pragma unroll
  for (int b = 0; b < S::kCols; ++b)
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) v[b * A + n1] = load_once(in + c * S::W + u + 128 * b + 1024 * n1);
  if constexpr (SCALED || MODE == kInverse) {
    const float s = (SCALED ? a.in_scale : 1.0f) * (MODE == kInverse ? kInvN : 1.0f);   // powers of two: exact
    const float2 f = make_float2(s, MODE == kInverse ? -s : s);
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = cmul_parts(v[m], f);
  }
  cluster_wait_acquire();
  const uint32_t base = smem_addr(sm), bar_local = smem_addr(&bar);
#pragma unroll
  for (int b = 0; b < S::kCols; ++b) {
    const int n2 = c * S::W + u + 128 * b;
    float2 z[A];
#pragma unroll
    for (int i = 0; i < A; ++i) z[i] = v[b * A + i];
    constexpr int kF = 6 + A / 8;                // factors per column, in [f / 2][n2] pairs
    float2 f[kF];
#pragma unroll
    for (int i = 0; i < kF; i += 2) {
      const float4 w = __ldg(a.tw_long + (i / 2) * 1024 + n2);
      f[i] = make_float2(w.x, w.y);
      if (i + 1 < kF) f[i + 1] = make_float2(w.z, w.w);
    }
    uint32_t slot[C], rbar[C];                   // this column in row 0 of every CTA, and its mbarrier
#pragma unroll
    for (int d = 0; d < C; ++d) {
      slot[d] = mapa(base + uint32_t(n2) * kWord, d);
      rbar[d] = mapa(bar_local, d);
    }
    twiddled_column_dft<A, kFine>(z, f, [&](int k1, float2 x) {
      if constexpr (H16ROW) {
        st_async_b32(slot[k1 / 8] + uint32_t((k1 % 8) * 1024) * kWord, half2_bits(x), rbar[k1 / 8]);
      } else {
        st_async_f2(slot[k1 / 8] + uint32_t((k1 % 8) * 1024) * kWord, x, rbar[k1 / 8]);
      }
    });
  }
  // All eight rows have landed (bounded wait).
  const bool arrived = mbar_wait_bounded(&bar, 0, a.status);
  {
    const int row = u >> 4, t = u & 15;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const int i = row * 1024 + t + 16 * m;
      v[m] = H16ROW ? bits_half2(reinterpret_cast<const uint32_t*>(sm)[i]) : sm[i];
    }
    if (__syncthreads_or(!arrived)) {
      // Nothing is stored; what peers may still be sending here lands (or its
      // wait expires once more) before the CTA's shared memory goes away.
      if (u == 0) mbar_wait_bounded(&bar, 0, nullptr);
      cluster_barrier_relaxed();
      return;
    }
    Dft<64, kFine>::run(v);
    float4* dst = reinterpret_cast<float4*>(sm + row * S::kRowPitch + t * 66);
#pragma unroll
    for (int r = 0; r < P; r += 2) dst[r / 2] = make_float4(v[r].x, v[r].y, v[r + 1].x, v[r + 1].y);
  }
  __syncthreads();
  const int row = u & 7, j0 = u >> 3;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int j = j0 + 16 * b;
    float2 z[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) z[r] = sm[row * S::kRowPitch + j + 66 * r];
#pragma unroll
    for (int r = 0; r < 16; r += 2) {
      const float4 w = __ldg(a.tw_row1024 + (r / 2) * 64 + j);
      if (r > 0) z[r] = cmul(z[r], make_float2(w.x, w.y));
      z[r + 1] = cmul(z[r + 1], make_float2(w.z, w.w));
    }
    Dft<16>::run(z);
    if constexpr (SCALED) {
      const float2 f = make_float2(a.out_scale, MODE == kForward ? a.out_scale : -a.out_scale);
#pragma unroll
      for (int r = 0; r < 16; ++r) z[r] = cmul_parts(z[r], f);
    } else if constexpr (MODE != kForward) {
#pragma unroll
      for (int r = 0; r < 16; ++r) z[r] = cconj(z[r]);
    }
    TS* o = out + 8 * c + row + A * j;
#pragma unroll
    for (int r = 0; r < 16; ++r) Storage<TS>::store(o + A * 64 * r, z[r]);
    check_finite<Storage<TS>, 16>(a.finite_flag, [&](int m) { return z[m]; });
  }
}

// Batches below this many points (ten lines of 65536) keep the four-step
// kernel, whose 16 CTAs of 256 threads finish a single line sooner (65536
// points, 5 lines: 10.2 against 12.6 us; 10 lines: 12.6 against 12.3; 38
// lines: 22.8 against 17.0; 32768 points: even at 20 to 40 lines).
constexpr long long kLongMinPoints = 10 * 65536;

template <int N, class TS, int MODE, bool SCALED, bool H16ROW = false>
cudaError_t launch_long_n(const RowArgs& a, cudaStream_t stream) {
  using S = LongShape<N>;
  auto kern = fft_long_kernel<N, TS, MODE, SCALED, H16ROW>;
  static const LaunchSetup setup = setup_cluster_kernel(kern, S::C, S::kThreads, S::kSmemBytes);
  if (setup.err != cudaSuccess) return setup.err;
  if (a.lines <= 0) return cudaSuccess;
  const long long grid = a.lines * S::C;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  RowArgs b = a;
  b.pf_ahead = (a.variant == kRowsPlainL2 || a.variant == kRowsPlain4L2 || a.variant == kRowsPlainHL2 ||
                a.variant == kRowsPlainH4L2 || a.variant == kRowsPlainHS4L2)
                   ? setup.resident
                   : 0;
  return launch_chained(kern, grid, S::kThreads, S::kSmemBytes, S::C, true, stream, b);
}

}  // namespace bfp
