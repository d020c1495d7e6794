// cell_index.h — columns of tiles, whose halos reach beyond the mesh, in 32-bit arithmetic that does not overflow
// up to the largest mesh.
#pragma once

#ifdef __CUDACC__
#define DG_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define DG_HOST_DEVICE inline
#endif

namespace dgk {

// The cell of column x of a periodic row of n cells. (The remainder keeps the sign of a column below 0; adding n
// before a second remainder overflows from n = 2^30 on.)
DG_HOST_DEVICE int wrap_column(int x, int n) {
  const int r = x % n;
  return r < 0 ? r + n : r;
}

// 1D rows hold up to 2^31 - 1 cells, so a column past their end is no int: an unsigned number counted from COLUMN0
// columns before the mesh (at least the widest halo).
constexpr unsigned COLUMN0 = 8;
DG_HOST_DEVICE unsigned column_of(long long x) { return (unsigned)(x + COLUMN0); }
DG_HOST_DEVICE bool column_inside(unsigned c, int n) { return c >= COLUMN0 && c < COLUMN0 + (unsigned)n; }
// The cell that a column less than 2^30 past the end stands for: across a periodic boundary, else the nearest.
DG_HOST_DEVICE int cell_column(unsigned c, int n, bool periodic) {
  const bool past = c >= COLUMN0 + (unsigned)n;
  if (!periodic) return c < COLUMN0 ? 0 : (past ? n - 1 : (int)(c - COLUMN0));
  return wrap_column((int)(c - COLUMN0 - (past ? (unsigned)n : 0u)), n);
}

// Tiles of `out` cells in n.
DG_HOST_DEVICE long long tiles_of(long long n, long long out) { return (n + out - 1) / out; }

}  // namespace dgk
