// dg_brick.cuh -- the cells that a block of the face kernels takes: a brick of
// 4 x 4 x 2 cells, rows r = 0..31 with x fastest.  Index arithmetic alone, for
// device and host.
#pragma once

#ifdef __CUDACC__
#define DG_BRICK_FN __host__ __device__ __forceinline__
#else
#define DG_BRICK_FN inline
#endif

namespace dg {
namespace sf {

struct Brick {
    int N, x0, y0, z0;
    DG_BRICK_FN Brick(unsigned block, int n) : N(n)
    {
        const unsigned nbx = (unsigned)(n + 3) >> 2, q = block / nbx;
        x0 = 4 * (int)(block - q * nbx);
        y0 = 4 * (int)(q % nbx);
        z0 = 2 * (int)(q / nbx);
    }
    static DG_BRICK_FN int count(int n) { return ((n + 3) / 4) * ((n + 3) / 4) * ((n + 1) / 2); }
    // cell of brick coordinates (-1..4, -1..4, -1..2), periodic: past the end of the
    // mesh the images of its cells, the neighbours that the last cells need
    DG_BRICK_FN long cell(int i, int j, int k) const
    {
        int x = x0 + i, y = y0 + j, z = z0 + k;
        x = x < 0 ? N - 1 : (x < N ? x : x % N);
        y = y < 0 ? N - 1 : (y < N ? y : y % N);
        z = z < 0 ? N - 1 : (z < N ? z : z % N);
        return ((long)z * N + y) * N + x;
    }
    DG_BRICK_FN bool inside(int i, int j, int k) const { return x0 + i < N && y0 + j < N && z0 + k < N; }
    // cell of row r that this brick updates, -1 where the row lies past the end of the
    // mesh: its image belongs to another brick, whose block writes it in the same launch
    DG_BRICK_FN long own(int r) const
    {
        const int i = r & 3, j = (r >> 2) & 3, k = r >> 4;
        return inside(i, j, k) ? cell(i, j, k) : -1;
    }
};

}  // namespace sf
}  // namespace dg
