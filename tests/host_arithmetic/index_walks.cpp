// The kernels' index walks (lbm_index.cuh) compiled by a host compiler, so
// that CPU tests can run them on the largest shapes a lattice may have.
#define __device__
#define __host__
#define __forceinline__ inline
#include "lbm_index.cuh"

// Walks the thread that starts at node `first`, in steps of `step`, over an
// nx x ny lattice; returns the nodes visited, or -1 if one came out wrong.
extern "C" long long walk_nodes(int nx, int ny, unsigned step, unsigned first)
{
    const unsigned n = unsigned(nx) * unsigned(ny);
    long long seen = 0;
    for (lbm::NodeWalk w(first, step, nx); w.id < n; w.next()) {
        const unsigned long long want = first + (unsigned long long)step * (unsigned long long)seen;
        if (w.id != want || w.x != want % (unsigned)nx || w.y != want / (unsigned)nx) return -1;
        ++seen;
    }
    return seen;
}
