// Output tiles of the FP64 integer-slice contraction (tc_oz.cuh) and the layout of its operands.
#pragma once
#include <stddef.h>

namespace osv {
namespace oz {

constexpr int BM = 128;       // tile rows = TMEM lanes = MMA M
constexpr int BN = 64;        // most columns of a tile with eight or five slices (level accumulators: 512 columns)
constexpr int BN4 = 128;      // and with four
constexpr __host__ __device__ int tile_cols(int ns) { return ns == 4 ? BN4 : BN; }
constexpr int BK = 32;        // k per stage (one 64-byte swizzle row of BF16)
constexpr int NSL = 8;        // slices per operand
constexpr int MXSL = 5;       // in the mixed form's pair build
constexpr int MXSOLVE = 4;    // and in its amplitude iterations
constexpr int CHUNK = 256;    // k-extent that shares one power-of-two scale per row
constexpr int EX_ZERO = -(1 << 20);   // chunk exponent of an all-zero chunk
constexpr int EX_NAN = 1 << 20;       // and of one that holds a NaN or an Inf

// An operand matrix: rows with K innermost, BF16 digits of slice s, row r at store row s * (rows of the store) + row + r
// (in units of the store's row stride), exponent of chunk c of row r at ex[eb + r * es + c] (es = 0: one
// exponent for all rows).
struct Mat {
  int row, eb, es;
};
// out += coef * A B^T over K
struct Seg {
  Mat a, b;
  int K;
  int pad;
  double coef;
};
struct Job {
  int seg0, nseg;          // the tile sums segments [seg0, seg0 + nseg)
  int m0, n0;              // first row / column of the tile in the output
  int m_valid, n_valid;    // rows (<= 128) and columns (<= tile_cols) to store
  int ld_out;
  int skip;                // index of a flag that makes the kernel leave the tile out, or -1
  int o_row, o_e;          // digit-writing epilogue: output matrix in its store, index of its exponent
  double s;                // epilogue scalar
  void* out;               // the output's first element (not the tile's)
};

inline int n_chunks(int K) { return (K + CHUNK - 1) / CHUNK; }
inline int ld_of(int K) { return (K + 7) & ~7; }   // row stride: 16-byte TMA rows

}  // namespace oz
}  // namespace osv
