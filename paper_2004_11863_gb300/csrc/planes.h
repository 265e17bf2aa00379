// Rows and elements of a level's z-planes: the storage pitch, and the walk of
// the 3D updates along a plane's elements.  Plain C++, for the layout, the
// launches and the kernels alike.
#pragma once

#ifdef __CUDACC__
#define MLBM_BOTH __host__ __device__ __forceinline__
#else
#define MLBM_BOTH inline
#endif

namespace mlbm {

#ifndef MLBM_ROW_ALIGN
#define MLBM_ROW_ALIGN 32
#endif
#ifndef MLBM_ROW_ALIGN_3D
#define MLBM_ROW_ALIGN_3D 8
#endif

inline int round_up(int x, int m) { return (x + m - 1) / m * m; }

// Row pitch SX and rows SY of a plane of n0 x n1 nodes with g0 and g1 ghost
// nodes at either end of an axis.  Rows are padded to MLBM_ROW_ALIGN elements
// in 2D; in 3D, whose updates walk the elements of a plane, to eight elements (a
// 32-byte sector in binary32), with rows added until a plane is whole
// 32-element lines -- unless that takes more memory than padded rows.
inline void plane_pitch(int D, int n0, int n1, int g0, int g1, int& SX, int& SY) {
  SX = round_up(n0 + 2 * g0, MLBM_ROW_ALIGN);
  SY = n1 + 2 * g1;
  if (D == 3) {
    const int sx = round_up(n0 + 2 * g0, MLBM_ROW_ALIGN_3D);
    const int lines = sx % 32 == 0 ? 1 : sx % 16 == 0 ? 2 : sx % 8 == 0 ? 4 : 8;
    const int sy = round_up(SY, lines);
    if ((long long)sx * sy <= (long long)SX * SY) {
      SX = sx;
      SY = sy;
    }
  }
}

// Elements from the first node to the last one of `rows` rows of `width`
// elements each, `pitch` apart.  A thread may stand for two of a row (pitch and
// width in pairs) or of two rows (rows in pairs).
inline long long plane_elements(int pitch, int width, int rows) {
  return (long long)(rows - 1) * pitch + width;
}

// Column and row of element e; a column of `width` or more lies between rows.
MLBM_BOTH void plane_node(unsigned pitch, unsigned e, int& x, int& y) {
  const unsigned r = e / pitch;
  y = (int)r;
  x = (int)(e - r * pitch);
}

}  // namespace mlbm
