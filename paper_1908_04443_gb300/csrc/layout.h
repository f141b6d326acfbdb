// Layout of the distribution buffers f[a][z][y][x] (host rules; no device code).
#pragma once

namespace lbmwet {

// Grids that the TMA-staged z-march takes: the window of a box (36 columns and 14 rows with the rows beyond
// it) leaves the grid on one side at most, also where the last column is moved inside.
inline bool ztma_marches(int nx, int ny, int nz) { return nx >= 40 && ny >= 16 && nz >= 4; }

// Nodes per stored row.  2D: a multiple of 32 (128-byte rows in FP32: TMA needs 16-byte row strides, and a row
// that starts a cache line keeps a warp's 32 consecutive nodes in one line).  3D: a multiple of 4 where the
// z-march runs (`zmarch`), so that every width has tensor maps; its direction offsets are 64-bit.  The other
// kernels form a * stride + node in 32 bits, which the limit on the nodes (2^31 / 19) covers only as long as the
// rows are not padded: 3D rows are not, nor are those of 2D grids so narrow and tall (15 columns or fewer, 7.4
// million rows or more) that the padding would pass it.
inline int row_pitch(int dim, bool zmarch, int nx, int ny) {
    const int pad = dim == 2 ? 32 : (zmarch ? 4 : 1), fp = (nx + pad - 1) / pad * pad;
    return dim == 2 && 9LL * fp * ny > 0x7fffffff ? nx : fp;
}

}  // namespace lbmwet
