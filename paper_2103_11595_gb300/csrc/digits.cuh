// Fixed-point digit form of FP64 / FP32 GEMM operands (host and device arithmetic; the kernels are
// in dg_gemm.cu). The FP64 CUDA-core rate of GB300 (1.25 TFLOP/s) is 1/1500 of its fp16
// tensor-core rate, so a product of FP64 matrices is cheaper as a sum of exact fp16 products of
// their digits (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59,
// 2012, with a row-wise quantum).
//
// Digits. For an operand row with largest magnitude m let E = floor(log2 m) and q = 2^(E - 7), so
// that |x / q| < 2^8 for every x of the row. X = x / (q 2^-54) is rounded to an integer
// (|X| <= 2^62; exact for entries within 2^-9 of m) and written in balanced base 512:
//   X = sum_{t < T} d_t 2^(54 - 9 t) + rest,   d_0 in [-256, 256], d_t in [-256, 255] (t >= 1).
// Every digit is an integer that fp16 holds exactly. The last digit also takes the rest, rounded
// to fp16's 11 significant bits. T = 6 keeps x to 2^-56 m (FP64 operands), T = 4 to 2^-38 m
// (operands of the FP32 mode): normwise per row, an entry below m in the fewer bits the smaller it is. On
// rows graded over 10^6 the error over sum |a||b| is 1.6e-14 (FP64 sums: 4e-16), and 4.4e-12 where the two
// operands are graded oppositely along the sum (tests/test_gpu_dg_gemm.py). The networks contracted here
// do not show it: n = 8 .. 16 circuits with noises of 1e-2 down to 1e-12 (692 GEMMs) gave the same largest
// |dF| as FP64 sums, 4.2e-15, and every one of 4096 traces to 3.2e-15 of its own Kraus weight, since an
// open Kraus index is a row index; FP32: 5.7e-9 against 2.1e-8 on CUDA cores.
//
// Layout of a digit operand of R rows (a power of two >= 16) and Kr = 2K real columns (a power of
// two >= 16): [row block of RB = min(R, 128)][chunk of 64 columns][slot][RB rows x 128 bytes], each
// RB x 128-byte tile in the 128-byte swizzle that the MMA reads, so a tile is one contiguous bulk
// copy. With Kr >= 64 slot t holds digit t. A narrower operand packs 2 (Kr = 32) or 4 (Kr = 16)
// digits side by side in one 128-byte row, so that no bytes are spent on padding columns (with six digits
// and four to a row, two of the eight places stay unused).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "device.h"

namespace ajf {
namespace dg {

constexpr int kTileRows = 128;  // rows of an operand row block

__host__ __device__ constexpr int digit_terms(int mode) { return mode == OPM_DIG6 ? 6 : 4; }
// log2 of the digits that share a 128-byte row; kcols = real columns (2K)
__host__ __device__ constexpr int pack_bits(int64_t kcols) { return kcols >= 64 ? 0 : (kcols >= 32 ? 1 : 2); }
__host__ __device__ constexpr int slots_of(int terms, int pack) { return (terms + (1 << pack) - 1) >> pack; }
__host__ __device__ constexpr int64_t chunks_of(int64_t kcols) { return kcols >= 64 ? kcols >> 6 : 1; }
__host__ __device__ constexpr int64_t block_rows(int64_t rows) { return rows < kTileRows ? rows : kTileRows; }
// bytes of a digit operand
__host__ __device__ constexpr int64_t operand_bytes(int64_t rows, int64_t kcols, int terms) {
  return rows * chunks_of(kcols) * slots_of(terms, pack_bits(kcols)) * 128;
}
// Place of the 16-byte piece that holds columns kr .. kr + 7 (kr a multiple of 8) of row r of an
// operand of 2^row_bits rows and 2^col_bits real columns: at(t) is its byte for digit t.
struct Piece {
  int64_t base;      // the chunk's first tile, plus the row
  int64_t tile;      // bytes of a tile
  int pack, piece, x;
  __host__ __device__ Piece(int row_bits, int col_bits, int terms, int64_t r, int64_t kr) {
    const int rb = row_bits < 7 ? row_bits : 7;
    pack = col_bits >= 6 ? 0 : 6 - col_bits;
    tile = int64_t(128) << rb;
    const int64_t chunk = ((r >> rb) << (col_bits >= 6 ? col_bits - 6 : 0)) + (kr >> 6);
    const int row = static_cast<int>(r) & ((1 << rb) - 1);
    base = chunk * slots_of(terms, pack) * tile + row * 128;
    piece = static_cast<int>(kr & 63) >> 3;
    x = row & 7;
  }
  __host__ __device__ int64_t at(int t) const {
    const int sub = (t & ((1 << pack) - 1)) << (3 - pack);
    return base + (t >> pack) * tile + (((piece + sub) ^ x) << 4);
  }
};

// X + bias for an FP64 value given by its bits and its row's largest exponent field E (>= its own):
// digit t >= 1 is then ((Y >> (54 - 9 t)) & 511) - 256 and d_0 = Y >> 54. A zero exponent field (zero
// and subnormal values, below 2^-1022) counts as zero. terms = 6 (the bias of the digits 1..5). An
// infinity or a NaN gives digits without a meaning: its row's exponent says so, and the product's epilogue
// writes NaN for the row.
__host__ __device__ inline int64_t biased_fixed(uint64_t bits, int row_field, int terms) {
  const int f = static_cast<int>((bits >> 52) & 0x7FF);
  int64_t x = 0;
  if (f != 0) {
    const int64_t m = static_cast<int64_t>((bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);
    const int d = row_field - f;  // >= 0
    if (d <= 9) {
      x = m << (9 - d);
    } else if (d <= 63) {
      x = (m + (int64_t(1) << (d - 10))) >> (d - 9);  // round to nearest, ties up
    }
    if (bits >> 63) x = -x;
  }
  int64_t bias = 0;
  for (int t = 1; t < terms; ++t) bias += int64_t(256) << (54 - 9 * t);
  return x + bias;
}

}  // namespace dg
}  // namespace ajf
