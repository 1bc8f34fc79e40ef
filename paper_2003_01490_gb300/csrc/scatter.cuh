// scatter.cuh -- registration of particles in the candidate lists of the
// mapping tiles their influence spheres touch (map.cu reads the lists).
#pragma once

#include "common.cuh"
#include "launch.h"

namespace lbmdem {

__device__ __forceinline__ int axis_pieces(double xc, double r, int n, int per, int (&a)[2], int (&b)[2]) {
    // cells whose centre (i + 1/2) lies in [xc - r, xc + r]
    long long lo = (long long)ceil(xc - r - 0.5);
    long long hi = (long long)floor(xc + r - 0.5);
    if (hi < lo) return 0;
    if (!per) {
        if (lo < 0) lo = 0;
        if (hi > n - 1) hi = n - 1;
        if (hi < lo) return 0;
        a[0] = (int)lo; b[0] = (int)hi;
        return 1;
    }
    if (hi - lo + 1 >= n) { a[0] = 0; b[0] = n - 1; return 1; }
    long long lw, hw;
    if (lo >= -n && hi < 2LL * n) {   // a centre in the box: no 64-bit remainders
        lw = lo < 0 ? lo + n : (lo >= n ? lo - n : lo);
        hw = hi < 0 ? hi + n : (hi >= n ? hi - n : hi);
    } else {
        lw = ((lo % n) + n) % n;
        hw = ((hi % n) + n) % n;
    }
    if (lw <= hw) { a[0] = (int)lw; b[0] = (int)hw; return 1; }
    a[0] = (int)lw; b[0] = n - 1; a[1] = 0; b[1] = (int)hw;
    return 2;
}

// distinct tile indices covering the cell pieces of one axis
__device__ __forceinline__ int axis_tiles(int np, const int (&a)[2], const int (&b)[2], int tsize, int (&t0)[2],
                          int (&t1)[2]) {
    if (np == 0) return 0;
    t0[0] = a[0] / tsize; t1[0] = b[0] / tsize;
    if (np == 1) return 1;
    int s = a[1] / tsize, e = b[1] / tsize;
    // trim the part of the second range already covered by the first
    if (e >= t0[0]) e = t0[0] - 1;
    if (s > e) return 1;
    t0[1] = s; t1[1] = e;
    return 2;
}

// particle i at xc; lane of lanes share out the tiles of its box
__device__ __forceinline__ void tile_scatter_particle(const MapParams& p, int i, const double (&xc)[3], int lane,
                                                      int lanes) {
    const double r = p.P.R[i] + fmax(p.shell_width, 1.4142135623730951) + 0.02;
    const int ts[3] = {TILE_X, TILE_Y, TILE_Z};
    int na[3], t0[3][2], t1[3][2], cnt[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int a[2], b[2];
        int np = axis_pieces(xc[d], r, p.g.n[d], p.g.per[d], a, b);
        na[d] = axis_tiles(np, a, b, ts[d], t0[d], t1[d]);
        if (na[d] == 0) return;
        cnt[d] = 0;
        for (int k = 0; k < na[d]; ++k) cnt[d] += t1[d][k] - t0[d][k] + 1;
    }
    const int total = cnt[0] * cnt[1] * cnt[2];
    for (int k = lane; k < total; k += lanes) {
        int rest = k;
        int tt[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            int m = rest % cnt[d];
            rest /= cnt[d];
            // the m-th tile of the axis' pieces
            const int len0 = t1[d][0] - t0[d][0] + 1;
            tt[d] = m < len0 ? t0[d][0] + m : t0[d][1] + (m - len0);
        }
        const long long t = ((long long)tt[2] * p.ntile[1] + tt[1]) * p.ntile[0] + tt[0];
        const int slot = atomicAdd(p.tile_count + t, 1);
        if (slot < TILE_CAP) p.tile_list[t * TILE_CAP + slot] = i;
        else atomicOr(p.status, ST_TILE_OVERFLOW);
    }
}

}  // namespace lbmdem
