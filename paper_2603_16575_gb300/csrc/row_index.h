// Row of an element of a row-major matrix by a multiplication (a division takes about twenty instructions).
#pragma once

#ifdef __CUDACC__
#define OSV_HD __host__ __device__ __forceinline__
#else
#define OSV_HD inline
#endif

namespace osv {

// ceil(2^32 / r), modulo 2^32 (r = 1: 0, and every row is 0).
OSV_HD unsigned row_magic(unsigned r) { return 0xffffffffu / r + 1; }

// idx / r for idx < r^2, r < 2^16.  The upper half of idx * magic is idx / r while idx r < 2^32 and at most one more
// beyond (from r = 1649 on for some idx), which the comparison takes back.
OSV_HD unsigned row_of(unsigned idx, unsigned r, unsigned magic) {
  const unsigned a = (unsigned)(((unsigned long long)idx * magic) >> 32);
  return a * r > idx ? a - 1 : a;
}

}  // namespace osv
