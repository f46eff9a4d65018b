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

}  // namespace lbm
