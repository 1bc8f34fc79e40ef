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

// Particle i (on: it exists) at x, coordinate d in lane d of its LANES lanes:
// lanes 0-2 find the tiles of one axis each (with all three axes in every lane the
// 27 float64 instructions of 64 cycles took most of the scatter: 10,000 particles
// mapped without history 144 us per call, this way 131), then all lanes share out
// the tiles of the box. All lanes of the warp take part.
template <int LANES>
__device__ __forceinline__ void tile_scatter_particle(const MapParams& p, int i, bool on, double x, int lane) {
    const unsigned FULL = 0xffffffffu;
    const int d = lane < 2 ? lane : 2;
    int first = 0, len = 0, second = 0, cnt = 0;
    if (on && lane < 3) {
        const double r = p.P.R[i] + fmax(p.shell_width, 1.4142135623730951) + 0.02;
        int a[2], b[2], t0[2], t1[2];
        const int np = axis_pieces(x, r, p.g.n[d], p.g.per[d], a, b);
        const int na = axis_tiles(np, a, b, d == 0 ? TILE_X : (d == 1 ? TILE_Y : TILE_Z), t0, t1);
        if (na > 0) {
            first = t0[0];
            len = t1[0] - t0[0] + 1;
            second = na > 1 ? t0[1] : 0;
            cnt = len + (na > 1 ? t1[1] - t0[1] + 1 : 0);
        }
    }
    int f3[3], l3[3], s3[3], c3[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        f3[e] = __shfl_sync(FULL, first, e, LANES);
        l3[e] = __shfl_sync(FULL, len, e, LANES);
        s3[e] = __shfl_sync(FULL, second, e, LANES);
        c3[e] = __shfl_sync(FULL, cnt, e, LANES);
    }
    const int total = c3[0] * c3[1] * c3[2];
    for (int k = lane; k < total; k += LANES) {
        int rest = k;
        int tt[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const int m = rest % c3[e];
            rest /= c3[e];
            // the m-th tile of the axis' pieces
            tt[e] = m < l3[e] ? f3[e] + m : s3[e] + (m - l3[e]);
        }
        const long long t = ((long long)tt[2] * p.ntile[1] + tt[1]) * p.ntile[0] + tt[0];
        const int slot = atomicAdd(p.tile_count + t, 1);
        if (slot < TILE_CAP) p.tile_list[t * TILE_CAP + slot] = i;
        else atomicOr(p.status, ST_TILE_OVERFLOW);
    }
}

}  // namespace lbmdem
