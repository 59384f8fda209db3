// Index of a neighbour in a row off the y and z faces of the box.
//
// One subtraction gives the neighbour n - e in the interior of such a row
// (0 < y < ny - 1, 0 < z < nz - 1), a shift by nx the wrapped one of a lane on a
// periodic x face.  Beyond a wall there is no neighbour, and the subtraction
// leaves the row and, with D3Q15's (1,1,1) at (0,1,1), the array: the lane reads
// its own node there and drops what it read.  So every load is inside the
// lattice and none waits for a branch.  Standard C++, also compiled for the
// host.
#pragma once

#ifdef __CUDACC__
#define ROW_FN __host__ __device__ __forceinline__
#else
#define ROW_FN inline
#endif

namespace lbmmb {

// Where row lane x stands: what the subtraction is off by for e_x = +1 and -1,
// and whether those neighbours lie beyond a wall.
struct RowLane {
    int cm, cp;
    bool wm, wp;
};
ROW_FN RowLane row_lane(int x, int nx, bool periodic) {
    RowLane r = {0, 0, false, false};
    if (x == 0) {
        if (periodic) r.cm = nx;
        else r.wm = true;
    }
    if (x == nx - 1) {
        if (periodic) r.cp = -nx;
        else r.wp = true;
    }
    return r;
}
ROW_FN bool row_wall(const RowLane &r, int ex) { return (ex > 0 && r.wm) || (ex < 0 && r.wp); }
// the index of node n's neighbour n - e, or n itself beyond a wall
ROW_FN int row_neighbour(int n, int nx, int nxy, const RowLane &r, int ex, int ey, int ez) {
    return row_wall(r, ex) ? n : n - (ex + nx * ey + nxy * ez) + (ex > 0 ? r.cm : (ex < 0 ? r.cp : 0));
}

}  // namespace lbmmb
