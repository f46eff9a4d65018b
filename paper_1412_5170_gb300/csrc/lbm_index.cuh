// lbm_index.cuh -- index walks of the kernels, safe for every lattice that
// lbm_create accepts (up to 2^31 - 1 nodes in any shape).  Compiled by the
// host too (tests), so no CUDA built-ins here.
#pragma once

namespace lbm {

// Walks a thread over the nodes of an nx-wide lattice in steps of the grid's
// threads, keeping (x, y) without a division per node.  Unsigned throughout:
// id and x run past 2^31 before the walk ends on the largest lattices.
struct NodeWalk {
    unsigned id, step, x, y, nx, sx, sy;
    __host__ __device__ __forceinline__ NodeWalk(unsigned first, unsigned step_, int nx_)
        : id(first), step(step_), nx(unsigned(nx_))
    {
        y = id / nx;
        x = id - y * nx;
        sy = step / nx;
        sx = step - sy * nx;
    }
    __host__ __device__ __forceinline__ void next()
    {
        id += step;
        x += sx;
        y += sy;
        if (x >= nx) { x -= nx; ++y; }
    }
};

// Rows [y0, y1) of chunk b of `rows` rows (the last one shorter), b rows < ny.
struct RowChunk { int y0, y1; };
__host__ __device__ __forceinline__ RowChunk row_chunk(unsigned b, int rows, int ny)
{
    const unsigned y0 = b * unsigned(rows), end = y0 + unsigned(rows);
    return RowChunk{int(y0), int(end < unsigned(ny) ? end : unsigned(ny))};
}

// Tiles of H rows down rows [y0, y1): even(y) and odd(y) in turn.  (The
// counter is unsigned: it runs past y1, which may be 2^31 - 1.)
template <int H, class Even, class Odd>
__host__ __device__ __forceinline__ void walk_tiles(int y0, int y1, Even even, Odd odd)
{
    for (unsigned y = y0; y < unsigned(y1); y += 2 * H) {
        even(int(y));
        if (y + H < unsigned(y1)) odd(int(y + H));
    }
}

}  // namespace lbm
