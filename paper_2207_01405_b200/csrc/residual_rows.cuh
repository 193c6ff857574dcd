// Which rows of a repeating residual a Dense epilogue fetches (plain C++, so that it can be run on the host too).
#pragma once

#ifdef __CUDACC__
#define IVIT_ROWS_FN __host__ __device__ __forceinline__
#else
#define IVIT_ROWS_FN inline
#endif

namespace ivit {

// Row of the residual that belongs to output row `row0 + off` of M, off < 32, where first = row0 % res_rows and res_rows >=
// 32; -1: there is no such output row, and the residual need not have one for it either (res_rows may be any number from M
// on when nothing repeats).
IVIT_ROWS_FN int residual_row(int row0, int first, int off, int M, int res_rows) {
  if (off >= M - row0) return -1;
  const int r = first + off;
  return r >= res_rows ? r - res_rows : r;
}

}  // namespace ivit
