// The kernels' index walks (lbm_index.cuh) and the cuts of the walks of tiles
// (lbm_host.cpp), compiled by a host compiler, so that CPU tests can run them
// on the largest shapes a lattice may have.
#include "lbm_host.h"
#include "lbm_index.cuh"

using namespace lbm;

extern "C" {

// Walks the thread that starts at node `first`, in steps of `step`, over an
// nx x ny lattice; returns the nodes visited, or -1 if one came out wrong.
long long walk_nodes(int nx, int ny, unsigned step, unsigned first)
{
    const unsigned n = unsigned(nx) * unsigned(ny);
    long long seen = 0;
    for (NodeWalk w(first, step, nx); w.id < n; w.next()) {
        const unsigned long long want = first + (unsigned long long)step * (unsigned long long)seen;
        if (w.id != want || w.x != want % (unsigned)nx || w.y != want / (unsigned)nx) return -1;
        ++seen;
    }
    return seen;
}

// Rows that chunk b of `rows` rows walks in tiles of eight; -1 if a tile
// starts outside the chunk or out of order.
long long walk_chunk(int ny, int rows, unsigned b)
{
    const RowChunk c = row_chunk(b, rows, ny);
    if (c.y0 < 0 || c.y1 <= c.y0 || c.y1 > ny) return -1;
    long long seen = 0;
    bool ok = true;
    int want = c.y0, turn = 0;
    auto tile = [&](int y, int parity) {
        ok = ok && y == want && turn == parity && y < c.y1;
        const int h = c.y1 - y < 8 ? c.y1 - y : 8;
        seen += h;
        want = c.y1 - y > 8 ? y + 8 : c.y1;
        turn ^= 1;
    };
    walk_tiles<8>(c.y0, c.y1, [&](int y) { tile(y, 0); }, [&](int y) { tile(y, 1); });
    return ok && want == c.y1 ? seen : -1;
}

void walk_plan(int nx, int ny, int nsm, int ctas, int out[3])
{
    const WalkPlan w = plan_walk(nx, ny, nsm, ctas);
    out[0] = w.sx;
    out[1] = w.sy;
    out[2] = w.rows;
}

}  // extern "C"
