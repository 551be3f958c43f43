// transpose.cu -- front end: time-major filterbank samples (the order a
// receiver or a SIGPROC file delivers, X_tm[t][c]) to the channel-major rows
// the dedispersion kernels read (X[c][t]).
//
// HBM-bound: reads and writes every sample once.  131072 x 4096 bytes in
// 164 us = 6.5 TB/s (the earlier 4-byte loads and stores of 32-word tiles, and a
// zero fill of the output, took 475 us).  A CTA moves a tile of 128
// bytes of channels x 256 / E times (E bytes a
// sample): every thread issues all its 16-byte loads first (8 of them for
// bytes), the tile waits in shared memory, and each thread then takes 16 / E
// times x 4 / E channels (one word column), transposes them in registers and
// writes 16 bytes along time per channel: 256 contiguous bytes per channel
// row.  Only samples with t in [t_begin, t_end) and c < n_chan are written;
// pieces off the 16-byte grid are written word by word, a piece that straddles
// t_end sample by sample.
#include <cuda_runtime.h>

#include <cstdint>

#include "dd_internal.h"

namespace dd {

namespace {

constexpr int kRowWords = 32;   // words of a tile row: 128 bytes of channels
constexpr int kThreads = 256;

// Transpose of an R x R block held as R words (word r = time r, samples =
// channels): out[j] = channel j, samples = times.
template <int R>
__device__ __forceinline__ void block_transpose(const uint32_t (&in)[R], uint32_t (&out)[R]) {
  if constexpr (R == 4) {
    // Bytes: in[r] = (c0 c1 c2 c3) at time r.
    const uint32_t a = __byte_perm(in[0], in[1], 0x5140);  // t0c0 t1c0 t0c1 t1c1
    const uint32_t b = __byte_perm(in[2], in[3], 0x5140);  // t2c0 t3c0 t2c1 t3c1
    const uint32_t c = __byte_perm(in[0], in[1], 0x7362);  // t0c2 t1c2 t0c3 t1c3
    const uint32_t d = __byte_perm(in[2], in[3], 0x7362);  // t2c2 t3c2 t2c3 t3c3
    out[0] = __byte_perm(a, b, 0x5410);
    out[1] = __byte_perm(a, b, 0x7632);
    out[2] = __byte_perm(c, d, 0x5410);
    out[3] = __byte_perm(c, d, 0x7632);
  } else if constexpr (R == 2) {
    out[0] = __byte_perm(in[0], in[1], 0x5410);
    out[1] = __byte_perm(in[0], in[1], 0x7632);
  } else {
    out[0] = in[0];
  }
}

// Tile row i keeps its words in pairs at word ^ 2 (i / (16 / E)): the 16
// threads that read one word column at 16 / E rows' distance, and the two
// columns of a warp, fall on 32 different banks.
template <int E>
__global__ void __launch_bounds__(kThreads) transpose_kernel(
    const uint8_t* __restrict__ in, int64_t in_stride_bytes, int32_t n_chan,
    uint8_t* __restrict__ out, int64_t out_stride_bytes, int64_t t_begin, int64_t t_end,
    int32_t chan_tiles) {
  constexpr int R = 4 / E;               // samples per word
  constexpr int kTimes = 16 / E;         // times per 16 output bytes
  constexpr int kRows = 16 * kTimes;     // times per tile
  constexpr int kLoads = kRows * 8 / kThreads;
  static_assert(kRows * 8 % kThreads == 0, "whole loads per thread");
  __shared__ __align__(16) uint32_t tile[kRows][kRowWords];
  const int tid = threadIdx.x;
  const int64_t t0 = t_begin + static_cast<int64_t>(blockIdx.x / chan_tiles) * kRows;
  const int32_t c0 = (blockIdx.x % chan_tiles) * (kRowWords * R);
  const int64_t b0 = static_cast<int64_t>(c0) * E;

  // 8 lanes per 128-byte row (rows and strides are 16-byte aligned).  Only
  // pieces with channels below n_chan: the rows may be columns of wider ones,
  // and the last of them ends with its memory.
  uint4 v[kLoads];
#pragma unroll
  for (int k = 0; k < kLoads; ++k) {
    const int i = (tid + k * kThreads) / 8, g = tid % 8;
    v[k] = make_uint4(0u, 0u, 0u, 0u);
    if (t0 + i < t_end && b0 + 16 * g < static_cast<int64_t>(n_chan) * E)
      v[k] = __ldcs(reinterpret_cast<const uint4*>(in + (t0 + i) * in_stride_bytes + b0) + g);
  }
#pragma unroll
  for (int k = 0; k < kLoads; ++k) {
    const int i = (tid + k * kThreads) / 8, g = tid % 8, sw = 2 * (i / kTimes);
    *reinterpret_cast<uint2*>(&tile[i][(4 * g) ^ sw]) = make_uint2(v[k].x, v[k].y);
    *reinterpret_cast<uint2*>(&tile[i][(4 * g + 2) ^ sw]) = make_uint2(v[k].z, v[k].w);
  }
  __syncthreads();

  // Lane: times t0 + kTimes bt .., word columns 2 q + (lane / 16).
  const int lane = tid & 31, bt = lane & 15;
  const int64_t t = t0 + static_cast<int64_t>(kTimes) * bt;
  if (t >= t_end) return;
  const bool whole = t + kTimes <= t_end && (t * E) % 16 == 0;
  for (int q = tid >> 5; q < kRowWords / 2; q += kThreads / 32) {
    const int col = 2 * q + (lane >> 4);
    uint32_t w[kTimes], o[R][4];
#pragma unroll
    for (int r = 0; r < kTimes; ++r) w[r] = tile[kTimes * bt + r][col ^ (2 * bt)];
#pragma unroll
    for (int m = 0; m < 4; ++m) {  // R times each
      uint32_t x[R], y[R];
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = w[R * m + r];
      block_transpose<R>(x, y);
#pragma unroll
      for (int j = 0; j < R; ++j) o[j][m] = y[j];
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int32_t c = c0 + R * col + j;
      if (c >= n_chan) continue;
      uint8_t* dst = out + static_cast<int64_t>(c) * out_stride_bytes + t * E;
      if (whole) {
        __stcs(reinterpret_cast<uint4*>(dst), make_uint4(o[j][0], o[j][1], o[j][2], o[j][3]));
      } else if (t + kTimes <= t_end) {  // t_begin is a multiple of a word's samples
#pragma unroll
        for (int m = 0; m < 4; ++m) reinterpret_cast<uint32_t*>(dst)[m] = o[j][m];
      } else {
#pragma unroll
        for (int k = 0; k < kTimes; ++k) {
          if (t + k >= t_end) break;
          const uint32_t s = o[j][k / R] >> (8 * E * (k % R));
          if constexpr (E == 1) dst[k] = static_cast<uint8_t>(s);
          else if constexpr (E == 2) reinterpret_cast<uint16_t*>(dst)[k] = static_cast<uint16_t>(s);
          else reinterpret_cast<uint32_t*>(dst)[k] = s;
        }
      }
    }
  }
}

}  // namespace

int launch_transpose(int elem_bytes, const void* d_in, int64_t in_row_stride, int32_t n_chan,
                     void* d_out, int64_t out_row_stride, int64_t t_begin, int64_t t_end,
                     void* stream) {
  if (t_end <= t_begin) return 0;
  const int chans = kRowWords * 4 / elem_bytes, rows = 256 / elem_bytes;
  const int32_t chan_tiles = (n_chan + chans - 1) / chans;
  const int64_t time_tiles = (t_end - t_begin + rows - 1) / rows;
  const int64_t grid = time_tiles * chan_tiles;
  if (grid <= 0 || grid > 0x7fffffffLL) return static_cast<int>(cudaErrorInvalidConfiguration);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const auto* in = static_cast<const uint8_t*>(d_in);
  auto* out = static_cast<uint8_t*>(d_out);
  const int64_t isb = in_row_stride * elem_bytes, osb = out_row_stride * elem_bytes;
  const unsigned g = static_cast<unsigned>(grid);
  switch (elem_bytes) {
    case 1: transpose_kernel<1><<<g, kThreads, 0, st>>>(in, isb, n_chan, out, osb, t_begin, t_end, chan_tiles); break;
    case 2: transpose_kernel<2><<<g, kThreads, 0, st>>>(in, isb, n_chan, out, osb, t_begin, t_end, chan_tiles); break;
    case 4: transpose_kernel<4><<<g, kThreads, 0, st>>>(in, isb, n_chan, out, osb, t_begin, t_end, chan_tiles); break;
    default: return static_cast<int>(cudaErrorInvalidValue);
  }
  return static_cast<int>(cudaGetLastError());
}

}  // namespace dd
