// Out-of-place transpose of a row-major [rows][cols] array of complex values
// (4-byte half2 or 8-byte float2): out[c][r] = in[r][c].
//
// The SAR pipeline (Fig. 1) compresses range lines (rows of the raw data) and
// azimuth lines (columns); between the two the data is turned.  One CTA moves
// a tile through shared memory; the reads (tile rows), the writes (rows of the
// turned tile) and the shared accesses between them are 16-byte vectors.
#include <cuda_runtime.h>

#include <cstdint>

#include "launch.h"

namespace bfp {

namespace {

// One 16-byte vector of elements, read and written whole.
template <class T>
struct alignas(16) TileVec {
  T v[16 / sizeof(T)];
};

// Tiles of TILE x TILE elements, TILE * sizeof(T) = 256 bytes: 64 x 64 half2
// or 32 x 32 float2.  256 threads, 16 x 16: each takes a block of VEC x VEC
// elements, VEC rows of one 16-byte vector, turns it by the naming of its
// registers alone and hands over VEC vectors of VEC rows each.  Vector accesses
// need the row pitch to be a multiple of 16 bytes; ragged edge tiles and other
// pitches use element accesses.
//
// The vectors of a turned column lie XORed with the column block's number: the
// eight lanes of a quarter-warp, eight column blocks on the way in and eight
// row blocks on the way out, meet all 32 banks.  Element by element the same
// exchange kept the L1 pipe 60 % busy with two-way conflicts, with the shared
// memory queue as the top stall; now HBM and L2 bound it.  From buffer to buffer
// to buffer: 4096 x 4096 half2 22.2 -> 20.8 us (6.45 TB/s), 16384 x 4096 92.5 ->
// 87.0, the latter in float2 178.8 -> 161.8.  Five CTAs per SM, 45 registers:
// eight (32 registers, spills) take 22.3 us, six 20.7 but 6.3 for 1024 x 4096,
// which five turn in 5.3.
//
// Each CTA takes tiles b, b + gridDim.x, ... and loads its next tile into
// registers before it writes the current one out, so the loads of one tile
// overlap the shared-memory reads and global stores of the one before.
template <class T>
struct TileIo {
  static constexpr int VEC = 16 / sizeof(T);
  static constexpr int TILE = 16 * VEC;
  long long rows, cols;
  unsigned col_tiles;

  __device__ void origin(unsigned b, long long& r0, long long& c0) const {
    r0 = (long long)(b / col_tiles) * TILE;
    c0 = (long long)(b % col_tiles) * TILE;
  }
  // This thread's block of tile b: rows VEC rb ... of columns VEC cb ....
  __device__ void load(const T* in, unsigned b, int cb, int rb, TileVec<T> (&e)[VEC]) const {
    long long r0, c0;
    origin(b, r0, c0);
    const bool vec = r0 + TILE <= rows && c0 + TILE <= cols && cols % VEC == 0;
    const long long r = r0 + rb * VEC, c = c0 + cb * VEC;
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
      if (vec) {
        *reinterpret_cast<uint4*>(&e[k]) = __ldcs(reinterpret_cast<const uint4*>(in + (r + k) * cols + c));
      } else {
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
          if (r + k < rows && c + i < cols) e[k].v[i] = in[(r + k) * cols + c + i];
        }
      }
    }
  }
};

template <class T>
__global__ void __launch_bounds__(256, 5) transpose_kernel(const T* in, T* out, long long rows, long long cols,
                                                        unsigned col_tiles, unsigned tiles) {
  using Io = TileIo<T>;
  constexpr int VEC = Io::VEC, TILE = Io::TILE;
  __shared__ uint4 tile[TILE * 16];   // column c, row block q: tile[16 c + (q ^ (c / VEC % 8))]
  chain_begin();
  const Io io{rows, cols, col_tiles};
  const int lane16 = threadIdx.x % 16, row16 = threadIdx.x / 16;
  unsigned b = blockIdx.x;
  if (b >= tiles) return;
  TileVec<T> e[VEC];
  io.load(in, b, lane16, row16, e);
  for (; b < tiles; b += gridDim.x) {
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
      TileVec<T> w;
#pragma unroll
      for (int k = 0; k < VEC; ++k) w.v[k] = e[k].v[i];
      tile[16 * (lane16 * VEC + i) + (row16 ^ (lane16 & 7))] = *reinterpret_cast<const uint4*>(&w);
    }
    __syncthreads();
    if (b + gridDim.x < tiles) io.load(in, b + gridDim.x, lane16, row16, e);   // in flight while this tile is written
    long long r0, c0;
    io.origin(b, r0, c0);
    const bool vec_out = r0 + TILE <= rows && c0 + TILE <= cols && rows % VEC == 0;
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
      const int tc = row16 + 16 * k;                   // column of the tile = row of the output
      const long long oc = c0 + tc, orow = r0 + lane16 * VEC;
      const uint4 v = tile[16 * tc + (lane16 ^ (tc / VEC & 7))];
      if (vec_out) {
        __stcs(reinterpret_cast<uint4*>(out + oc * rows + orow), v);
      } else {
        const T* w = reinterpret_cast<const T*>(&v);
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
          if (oc < cols && orow + i < rows) out[oc * rows + orow + i] = w[i];
        }
      }
    }
    __syncthreads();                                   // the tile buffer is free for the next tile
  }
}

}  // namespace

cudaError_t launch_transpose(const void* in, void* out, long long rows, long long cols, int elem_bytes,
                             cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return cudaSuccess;
  if (elem_bytes != 4 && elem_bytes != 8) return cudaErrorInvalidValue;
  const int tile = elem_bytes == 4 ? 64 : 32;
  const long long gx = (cols + tile - 1) / tile, gy = (rows + tile - 1) / tile;
  const long long tiles = gx * gy;
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;   // 2^31 tiles: at least 512 GB of data
  // Resident CTAs of the kernel on this device, once per element size.
  static int resident[2] = {0, 0};
  int& res = resident[elem_bytes == 4 ? 0 : 1];
  if (res == 0) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = elem_bytes == 4
              ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, transpose_kernel<unsigned int>, 256, 0)
              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, transpose_kernel<float2>, 256, 0);
    if (e != cudaSuccess) return e;
    res = sms * per_sm > 0 ? sms * per_sm : 1;
  }
  // Every CTA takes the same number of tiles (the last ones one fewer at most);
  // below two each they are taken singly, half the CTAs with two would leave the
  // others' places idle.
  const long long per_cta = tiles < 2LL * res ? 1 : (tiles + res - 1) / res;
  const long long grid = (tiles + per_cta - 1) / per_cta;
  if (elem_bytes == 4)
    return launch_chained(transpose_kernel<unsigned int>, grid, 256, 0, 1, true, s,
                          static_cast<const unsigned int*>(in), static_cast<unsigned int*>(out), rows, cols, unsigned(gx),
                          unsigned(tiles));
  return launch_chained(transpose_kernel<float2>, grid, 256, 0, 1, true, s, static_cast<const float2*>(in),
                        static_cast<float2*>(out), rows, cols, unsigned(gx), unsigned(tiles));
}

}  // namespace bfp
