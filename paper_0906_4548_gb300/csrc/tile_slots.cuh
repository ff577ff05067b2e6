// Four-step transforms inside a 128-byte swizzled shared-memory tile.
//
// A tile of 16 pencils has one 128-byte line per sample, pencil r's complex value in the line's
// 8-byte slot r, with the TMA 128-byte swizzle (16-byte chunk index XOR line mod 8).  A pencil of
// N = N1 N2 values belongs to N2 lanes of one warp, a warp to 32 / N2 pencils (lane bit 0 is the
// pencil's parity, so the 16 lanes of a shared-memory phase hold 8 lanes of an even and an odd
// pencil).  Lane c does the N1-point transforms of column c and the N2-point transforms of rows
// k1 = c, c + N2, ...; in between, value (k1, c) sits in line k1 N2 + (c ^ (k1 & 7)) of its own
// pencil.  Both directions are free of bank conflicts for N2 >= 8, and no other warp touches the
// pencil's slots, so a transform needs __syncwarp only.  Lines from N / 2 on lie `FOLD` bytes further
// (in a second tile).  When N1 is a multiple of N2, the values of lane c after the second
// stage, k1 + N1 k2 with k1 = c mod N2, are again samples of its column.
#pragma once

#include "fft_core.cuh"

namespace dgp {

template <int N1, int N2, int FOLD> struct TileSlots {
  static constexpr int M = N2 < 8 ? N2 - 1 : 7;
  static_assert(N2 == 4 || N2 == 8 || N2 == 16, "the lanes of a pencil divide a warp");
  static_assert((N1 * N2) % 16 == 0 && N1 % 2 == 0, "whole swizzle periods in both halves");
  static __host__ __device__ constexpr int col(int k1) { return k1 * N2 * 128 + (k1 >= N1 / 2 ? FOLD : 0); }
  static __host__ __device__ constexpr int odd4(int k1) { return N2 == 4 ? (k1 & 1) << 6 : 0; }
  // byte offset of line l, pencil r (first tile)
  static __device__ __forceinline__ int line(int l, int r) { return l * 128 + ((r * 8) ^ ((l & 7) << 4)); }
  // line l of the N lines across both tiles, pencil r
  static __device__ __forceinline__ int folded(int l, int r) { return line(l, r) + (l >= N1 * N2 / 2 ? FOLD : 0); }
  // sample N2 j1 + c, given line(c, r)
  static __device__ __forceinline__ int sample(int base, int j1) {
    return (base + j1 * N2 * 128) ^ (N2 == 4 ? (j1 & 1) << 6 : 0);
  }
  // value (k1, c) for a compile-time k1, given line(c, r)
  static __device__ __forceinline__ int by_col(int base, int k1) {
    return col(k1) + (base ^ ((k1 & M) * 144) ^ odd4(k1));
  }
  // value (k1, j2) for a compile-time j2: base = by_row_base(k1, r)
  static __device__ __forceinline__ int by_row_base(int k1, int r) {
    return col(k1) + (((k1 & M) * 144) ^ (r * 8) ^ odd4(k1));
  }
  static __device__ __forceinline__ int by_row(int base, int j2) { return (base ^ ((j2 & 7) * 144)) + (j2 >> 3) * 1024; }
};

__device__ __forceinline__ float2& tile_at(unsigned char* buf, int off) {
  return *reinterpret_cast<float2*>(buf + off);
}
__device__ __forceinline__ float2 tile_at(const unsigned char* buf, int off) {
  return *reinterpret_cast<const float2*>(buf + off);
}

}  // namespace dgp
