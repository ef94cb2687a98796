// Range-Doppler imaging with RCMC and range-dependent azimuth filters (rda.cu).
#pragma once

#include <cuda_runtime.h>

namespace bfp {

struct RdaGeometry {
  double range_cell_m;     // slant-range sample spacing
  double prf_hz;           // pulse repetition frequency
  double wavelength_m;
  double speed_mps;        // platform speed
  double centre_range_m;   // slant range of range cell n_rg / 2
};

struct RdaArgs {
  const void* in;          // [lines][N] in the storage type
  void* out;               // [lines][N]; may equal in
  const float2* tw;        // pass-major FP32 twiddles of length N
  long long lines;
  const unsigned long long* line_turns;   // per line: its phase unit as a binary fraction of a turn (launch_rda_lines)
  int aperture;            // azimuth chirp length L (pulses)
  int peak_normalise;      // azimuth lines: H_r / max |H_r|
};

constexpr int kRdaMinLog2 = 8;
constexpr int kRdaMaxLog2 = 13;

// The phase units of the lines: shift[n_az] for RCMC lines, rate[n_rg] for
// azimuth lines (range_dependent: k_a of each bin's own range, else of the
// centre range).
cudaError_t launch_rda_lines(const RdaGeometry& geo, bool range_dependent, int n_az, int n_rg,
                             unsigned long long* shift, unsigned long long* rate, cudaStream_t s);

// RCMC lines (along range, one per Doppler bin) and azimuth lines (along
// Doppler, one per range bin); f16 selects half2 storage, else float2.
cudaError_t launch_rcmc_rows(int log2n, bool f16, const RdaArgs& a, cudaStream_t s);
cudaError_t launch_azimuth_rows(int log2n, bool f16, const RdaArgs& a, cudaStream_t s);

}  // namespace bfp
