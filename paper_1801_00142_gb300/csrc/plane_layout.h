// Layout of a batch of row-major matrices held as BF16 split planes,
// [plane][batch][row][ld] (host code, no CUDA header needed).
#pragma once

// Row stride of an operand buffer with k columns: whole 16-byte units.
static inline long long tc_ld(long long k) { return (k + 7) / 8 * 8; }

// Strides in elements.  The one place that forms them: the conversion that
// writes the planes, the GEMM that reads them and the size of the scratch that
// holds them all take them from here.  64 bits throughout: batch * rows alone
// passes 2^31 within a card's memory (65535 matrices of 32769 rows and one
// column fill 69 GB as two planes).
struct PlaneLayout {
  long long ld, batch_stride, plane_stride;
};
static inline PlaneLayout plane_layout(int rows, int cols, int batch) {
  PlaneLayout p;
  p.ld = tc_ld(cols);
  p.batch_stride = (long long)rows * p.ld;
  p.plane_stride = (long long)batch * p.batch_stride;
  return p;
}
