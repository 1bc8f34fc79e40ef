// map.cu -- explicit particle mapping (Sec. 2.2), TRT+aB shell (Sec. 2.3.2),
// refill of uncovered cells (Eq. (18)) and the field read-out.
//
// Mapping: every particle registers itself in the candidate list of each
// 32x4x4 tile that its influence sphere (R + max(delta_aB, sqrt 2)) touches;
// then the tile's cells are tested against its candidates, eight cells a
// thread. The solid test |x_c - x_p|^2 <= R^2 and the shell
// test R^2 < |x_c - x_p|^2 <= (R + delta_aB)^2 are decided in float32 when the
// margin is clear and re-evaluated in float64 with round-to-nearest and no
// contraction, ((dx dx + dy dy) + dz dz), when a value lies within 1e-5
// (relative) of a threshold, so the flags are exactly those of a plain float64
// evaluation. The lowest particle index owns a cell inside several spheres;
// fluid cells have owner -1. Cells that were solid and are now fluid go to the
// refill list with their former particle. Fluid cells within R + sqrt(2) of a
// particle get the NEAR flag; solid cells next to another body (candidates for
// missing links) go to the missing-link list that the boundary kernel of the
// next step reads. The solid and shell cells are also written as one bit per
// cell (a tile row of 32 cells is one word), from which the dense kernel finds
// the particle links.
#include <cstddef>

#include "common.cuh"
#include "gang.cuh"
#include "launch.h"
#include "sc_common.cuh"
#include "scatter.cuh"

// minimum resident mapping blocks per SM (a register cap)
#ifndef LBM_MAP_MIN_BLOCKS
#define LBM_MAP_MIN_BLOCKS 16
#endif
#ifndef LBM_MAP_DEPTH_MAX
#define LBM_MAP_DEPTH_MAX 4
#endif

namespace lbmdem {

constexpr int MAP_BLOCKS_WANTED = 152 * LBM_MAP_MIN_BLOCKS, MAP_DEPTH_MAX = LBM_MAP_DEPTH_MAX;

__device__ __forceinline__ double min_image_dd(double d, int n, int per) {
    if (per) {
        double half = 0.5 * (double)n;
        if (d > half) d -= (double)n;
        if (d < -half) d += (double)n;
    }
    return d;
}
// ------------------------------------------------------------ tile scatter

// one warp per particle
__device__ __forceinline__ void tile_scatter_body(const MapParams& p, int bx) {
    const int i = (bx * blockDim.x + threadIdx.x) >> 5;
    if (i >= p.P.n) return;   // warp-uniform
    const int lane = threadIdx.x & 31;
    tile_scatter_particle<32>(p, i, true, lane < 3 ? p.P.x[3 * i + lane] : 0.0, lane);
}

__global__ void tile_scatter_kernel(const MapParams p) { tile_scatter_body(p, (int)blockIdx.x); }

__global__ void tile_scatter_gang_kernel(const MapParams* __restrict__ table, const int* __restrict__ off, int n) {
    __shared__ __align__(16) MapParams sp;
    const int i = gang_instance(off, n, (int)blockIdx.x);
    gang_load(table, i, sp);
    tile_scatter_body(sp, (int)blockIdx.x - off[i]);
}

void launch_tile_scatter(const MapParams& p, cudaStream_t st) {
    if (p.P.n == 0) return;
    const long long threads = 32LL * p.P.n;
    tile_scatter_kernel<<<(int)((threads + 127) / 128), 128, 0, st>>>(p);
}

// ------------------------------------------------------------ mapping

// Exact float64 decision of the solid and shell tests for a cell centre whose
// float32 distance lies within the tolerance of a threshold (kept out of line:
// it runs for a tiny fraction of the tests). Returns bit 0 inside, bit 1 shell.
__device__ __noinline__ int exact_tests(const MapParams& p, int id, int x, int y, int z) {
    const int cpos[3] = {x, y, z};
    const double R = p.P.R[id];
    double dd[3];
#pragma unroll
    for (int d = 0; d < 3; ++d)
        dd[d] = min_image_dd(((double)cpos[d] + 0.5) - p.P.x[3 * id + d], p.g.n[d], p.g.per[d]);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dd[0], dd[0]), __dmul_rn(dd[1], dd[1])), __dmul_rn(dd[2], dd[2]));
    const double rs = __dadd_rn(R, p.shell_width);
    const bool inside = d2 <= __dmul_rn(R, R);
    const bool in_shell = !inside && d2 <= __dmul_rn(rs, rs);
    return (inside ? 1 : 0) | (in_shell ? 2 : 0);
}

// minimum image on a short periodic axis, decided on 2 (n + g) against L
__device__ __forceinline__ float short_axis_image(float n, float g, int L) {
    const float tw = 2.0f * n + 2.0f * g;
    const float fl = (float)L;
    return tw > fl ? n - fl : (tw < -fl ? n + fl : n);
}

constexpr int MAP_THREADS = 64;
constexpr int MISS_HELD = 256;     // missing-link cells a block holds back before it appends them
static_assert(TILE_X == 32 && TILE_Y == 4 && TILE_Z == 4 && MAP_THREADS * 8 == TILE_X * TILE_Y * TILE_Z,
              "a thread takes four cells of a tile row in two planes");
static_assert(MAP_THREADS >= TILE_CAP, "one thread stages one candidate");

// candidate k of a tile: the integer offset n of the tile's first cell from the
// particle's base cell (an exact float; on long periodic axes already moved to
// the image nearest to the tile), the common fractional offset g = 1/2 - frac,
// R^2, (R + shell)^2, the near threshold and the tolerance of the float32 tests
struct MapShared {
    float4 cn[2][TILE_CAP];   // n, particle
    float4 ca[2][TILE_CAP];   // g, R^2
    float4 cb[2][TILE_CAP];   // (R + shell)^2, near, tolerance, axes (bits) without one image per tile
    unsigned miss[MISS_HELD + TILE_X * TILE_Y * TILE_Z];
    unsigned n_miss, base, n_solid[MAP_THREADS / 32];
};

// the first 36 bytes of a view: base, frac, R (as two 16-byte words and one of 4)
struct MapView {
    int4 a;
    float4 b;
};
__device__ __forceinline__ MapView load_map_view(const PartView* v) {
    static_assert(offsetof(PartView, frac) == 12 && offsetof(PartView, R) == 24, "two words hold base, frac and R");
    const int4* q = reinterpret_cast<const int4*>(v);
    MapView m;
    m.a = q[0];
    m.b = reinterpret_cast<const float4*>(q)[1];
    return m;
}

__device__ __forceinline__ void stage_candidate(const MapParams& p, MapShared& sh, int buf, int k, int i,
                                                const MapView& v, int ox, int oy, int oz) {
    const int org[3] = {ox, oy, oz}, base[3] = {v.a.x, v.a.y, v.a.z};
    const float frac[3] = {__int_as_float(v.a.w), v.b.x, v.b.y};
    const int ts[3] = {TILE_X, TILE_Y, TILE_Z};
    const float R = v.b.z;
    const float sw = (float)p.shell_width;
    const float reach = R + fmaxf(sw, 1.4142136f) + 0.02f;
    float n0[3], g[3];
    unsigned small = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int n = org[d] - base[d];
        g[d] = 0.5f - frac[d];
        if (p.g.per[d]) {
            const int L = p.g.n[d];
            if ((float)L <= 2.0f * reach + (float)(ts[d] + 2)) {
                small |= 1u << d;   // some cells of the tile may be nearer to another image
            } else {
                // image nearest to the tile centre
                const float cc = (float)(2 * n + ts[d] - 1) + 2.0f * g[d];   // twice the centre offset
                if (cc > (float)L) n -= L;
                else if (cc < -(float)L) n += L;
            }
        }
        n0[d] = (float)n;
    }
    const float Rs = R + sw;
    const float Rn = R + 1.4142135f + 0.02f;
    const float R2 = R * R, Rs2 = Rs * Rs;
    // d2 <= Rn^2 as d2 < the next float
    const float near = __int_as_float(__float_as_int(Rn * Rn) + 1);
    sh.cn[buf][k] = make_float4(n0[0], n0[1], n0[2], __int_as_float(i));
    sh.ca[buf][k] = make_float4(g[0], g[1], g[2], R2);
    sh.cb[buf][k] = make_float4(Rs2, near, 1e-5f * (Rs2 + 1.0f), __uint_as_float(small));
}

__device__ __forceinline__ float lo_of(F2 a) {
    float lo, hi;
    split(a, lo, hi);
    return lo;
}
__device__ __forceinline__ float hi_of(F2 a) {
    float lo, hi;
    split(a, lo, hi);
    return hi;
}
// bit j of the result: the sign of t[j]
__device__ __forceinline__ unsigned signs(const F2 (&t)[4]) {
    unsigned m = __float_as_uint(hi_of(t[3])) >> 31;
    m = __funnelshift_l(__float_as_uint(lo_of(t[3])), m, 1);
#pragma unroll
    for (int k = 2; k >= 0; --k) {
        m = __funnelshift_l(__float_as_uint(hi_of(t[k])), m, 1);
        m = __funnelshift_l(__float_as_uint(lo_of(t[k])), m, 1);
    }
    return m;
}
// bit j of m to bit 0 of byte j
__device__ __forceinline__ unsigned bytes_of(unsigned m) { return (m * 0x00204081u) & 0x01010101u; }

// Mapping of the tiles (bx, by, z0) .. (bx, by, z1 - 1) by one block. A warp takes
// half a tile, the 16x4x4 brick at x in 16 warp .. (a compact brick meets fewer
// spheres than rows of 32 cells), lane l eight cells: x from 4 (l & 3), y = (l >> 2)
// & 3, z = 2 (l >> 4) and the next; bit 4 h + j of its masks is cell x + j of plane
// z + h. Offsets are (n + l) + g with the integer part formed first, so no float32
// intermediate is larger than the offset itself. Each warp first drops the
// candidates that cannot reach its brick. While a tile is tested the candidates of
// the next one are on their way.
//
// Bound by instruction issue and, in small boxes, by the chain from the tile's
// count to its list, the views and the tests. A thread per (x, y) column with a
// test per cell and byte-wide flags issued 787 warp instructions per 128 cells
// at 76 % of the slots: 204 us for 256x256x512 cells and 10,000 spheres, 35 us for
// 128x128x256 and 1,250, and without history 312 us plus 50 us for clearing the
// outputs. Here the distances of eight cells are packed float32 arithmetic, every
// decision is a mask of eight bits from the signs of the differences, flags are
// written as words and owners as vectors (bytes and single words where a side is
// no multiple of four), and a block appends to the shared counters once: 725
// instructions per 256 cells at 59 %, 113 us, 25 us and 87 us without clearing.
// (Four cells a thread: 137 us. 12 resident blocks 119 us, 20 136 us; walks of 8
// tiles 115 us, 16 123 us.)
//
// FRESH: the outputs of a box without history (flags and owner only: the owner
// of every cell is written, nothing is read, no list is kept).
template <bool FRESH>
__device__ __forceinline__ void map_body(const MapParams& p, int bx, int by, int z0, int z1) {
    __shared__ MapShared sh;
    const unsigned FULL = 0xffffffffu;
    int tid;   // opaque, or the compiler reads the special register again and again
    asm volatile("mov.u32 %0, %%tid.x;" : "=r"(tid));
    const int warp = tid >> 5, lane = tid & 31;
    const int lx = 16 * warp + 4 * (lane & 3), ly = (lane >> 2) & 3, lz = 2 * (lane >> 4);
    const int nx = p.g.n[0], ny = p.g.n[1], nz = p.g.n[2];
    const int ox = bx * TILE_X, oy = by * TILE_Y;
    const int x = ox + lx, y = oy + ly;
    const int plane = nx * ny;   // cells and words of a box are counted in 31 bits
    const int nt = p.ntile[0] * p.ntile[1], words = p.ntile[0] * ny;
    const bool vec = ((nx & 3) | ((unsigned)(uintptr_t)p.flags & 3) | ((unsigned)(uintptr_t)p.owner & 15)) == 0;
    const unsigned valid_xy = y < ny ? (x + 4 <= nx ? 15u : (x < nx ? (1u << (nx - x)) - 1u : 0u)) : 0u;
    // cells of the quad next to a wall in x or y
    unsigned wall_xy = 0;
    if (!p.g.per[0]) {
        if (x == 0) wall_xy |= 1u;
        if (nx - 1 >= x && nx - 1 < x + 4) wall_xy |= 1u << (nx - 1 - x);
    }
    if (!p.g.per[1] && (y == 0 || y == ny - 1)) wall_xy = 15u;
    wall_xy *= 0x11u;
    const float flx = (float)lx, fly = (float)ly, flz = (float)lz;

    int t = (z0 * p.ntile[1] + by) * p.ntile[0] + bx;
    int c_cur = min(p.tile_count[t], TILE_CAP);
    int c_nxt = z0 + 1 < z1 ? min(p.tile_count[t + nt], TILE_CAP) : 0;
    if (tid == 0) sh.n_miss = 0;
    if (tid < c_cur) {
        const int i = p.tile_list[(long long)t * TILE_CAP + tid];
        stage_candidate(p, sh, 0, tid, i, load_map_view(p.P.view + i), ox, oy, z0 * TILE_Z);
    }
    __syncthreads();

    unsigned solid_count = 0;
    int z = z0 * TILE_Z + lz;
    int idx = z * plane + y * nx + x;
    int half = 2 * (z * words + y * p.ntile[0] + bx) + warp;   // the row's 16 cells in the bits
    for (int bz = z0; bz < z1; ++bz, t += nt, z += TILE_Z, idx += TILE_Z * plane, half += 2 * TILE_Z * words) {
        const int buf = (bz - z0) & 1;
        const unsigned valid = (z < nz ? valid_xy : 0u) | (z + 1 < nz ? valid_xy << 4 : 0u);
        // the next tile's list entry, the count after it, the cells solid before
        int next_i = 0;
        const bool stage = tid < c_nxt;
        if (stage) next_i = p.tile_list[(long long)(t + nt) * TILE_CAP + tid];
        const int c_after = bz + 2 < z1 ? min(p.tile_count[t + 2 * nt], TILE_CAP) : 0;
        unsigned old0 = 0, old1 = 0;
        if (!FRESH && (valid & 15u)) old0 = reinterpret_cast<const unsigned short*>(p.solid)[half];
        if (!FRESH && (valid >> 4)) old1 = reinterpret_cast<const unsigned short*>(p.solid)[half + 2 * words];

        int own[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) own[j] = 0x7fffffff;
        unsigned near1 = 0, near2 = 0;     // cells near one / two particles
        unsigned solid = 0, multi = 0, shell = 0;
        for (int k0 = 0; k0 < c_cur; k0 += 32) {
            // candidates that may reach this warp's brick (conservative float bound)
            bool rel = false;
            if (k0 + lane < c_cur) {
                const float4 N = sh.cn[buf][k0 + lane], A = sh.ca[buf][k0 + lane], B = sh.cb[buf][k0 + lane];
                const float xlo = (N.x + (float)(16 * warp)) + A.x, xhi = xlo + 15.0f;
                const float ylo = N.y + A.y, yhi = ylo + 3.0f;
                const float zlo = N.z + A.z, zhi = zlo + 3.0f;
                const float dx = fmaxf(fmaxf(xlo, -xhi), 0.f), dy = fmaxf(fmaxf(ylo, -yhi), 0.f),
                            dz = fmaxf(fmaxf(zlo, -zhi), 0.f);
                const float far = fmaxf(B.y, B.x + B.z) * 1.0001f + 0.01f;
                rel = dx * dx + dy * dy + dz * dz <= far || __float_as_uint(B.w) != 0u;
            }
            unsigned mm = __ballot_sync(FULL, rel);
            while (mm) {
                const int k = __ffs(mm) - 1 + k0;
                mm &= mm - 1;
                const float4 N = sh.cn[buf][k], A = sh.ca[buf][k], B = sh.cb[buf][k];
                const int id = __float_as_int(N.w);
                const float fx = N.x + flx;
                float fy = N.y + fly, fz0 = N.z + flz, fz1 = fz0 + 1.0f;
                F2 x01 = f2(fx, fx + 1.0f), x23 = f2(fx + 2.0f, fx + 3.0f);
                const unsigned small = __float_as_uint(B.w);
                if (small) {
                    if (small & 1u) {
                        x01 = f2(short_axis_image(fx, A.x, nx), short_axis_image(fx + 1.0f, A.x, nx));
                        x23 = f2(short_axis_image(fx + 2.0f, A.x, nx), short_axis_image(fx + 3.0f, A.x, nx));
                    }
                    if (small & 2u) fy = short_axis_image(fy, A.y, ny);
                    if (small & 4u) {
                        fz0 = short_axis_image(fz0, A.z, nz);
                        fz1 = short_axis_image(fz1, A.z, nz);
                    }
                }
                const float dy = fy + A.y, dz0 = fz0 + A.z, dz1 = fz1 + A.z;
                const float dy2 = __fmul_rn(dy, dy);
                const F2 gx = f2(A.x, A.x), vy = f2(dy2, dy2), va = f2(dz0, dz0), vb = f2(dz1, dz1);
                const F2 dx01 = x01 + gx, dx23 = x23 + gx;
                const F2 p01 = mad(dx01, dx01, vy), p23 = mad(dx23, dx23, vy);
                const F2 d[4] = {mad(va, va, p01), mad(va, va, p23), mad(vb, vb, p01), mad(vb, vb, p23)};
                const F2 r2 = f2(A.w, A.w), s2 = f2(B.x, B.x), n2 = f2(B.y, B.y);
                const F2 di[4] = {d[0] - r2, d[1] - r2, d[2] - r2, d[3] - r2};
                const F2 dh[4] = {d[0] - s2, d[1] - s2, d[2] - s2, d[3] - s2};
                const F2 dn[4] = {d[0] - n2, d[1] - n2, d[2] - n2, d[3] - n2};
                const unsigned near = signs(dn);
                unsigned in = signs(di), within = signs(dh);
                float least = fabsf(lo_of(di[0]));
#pragma unroll
                for (int k2 = 0; k2 < 4; ++k2) {
                    least = fminf(fminf(least, fabsf(lo_of(di[k2]))), fabsf(hi_of(di[k2])));
                    least = fminf(fminf(least, fabsf(lo_of(dh[k2]))), fabsf(hi_of(dh[k2])));
                }
                if (least <= B.z) {
                    // within the tolerance of a threshold: the float64 decision
                    unsigned close = 0;
#pragma unroll
                    for (int k2 = 0; k2 < 4; ++k2) {
                        if (fabsf(lo_of(di[k2])) <= B.z || fabsf(lo_of(dh[k2])) <= B.z) close |= 1u << (2 * k2);
                        if (fabsf(hi_of(di[k2])) <= B.z || fabsf(hi_of(dh[k2])) <= B.z) close |= 2u << (2 * k2);
                    }
                    close &= valid;
                    while (close) {
                        const int j = __ffs(close) - 1;
                        close &= close - 1;
                        const int r = exact_tests(p, id, x + (j & 3), y, z + (j >> 2));
                        in = (in & ~(1u << j)) | (unsigned)(r & 1) << j;
                        within = (within & ~(1u << j)) | (unsigned)(r != 0) << j;
                    }
                }
                near2 |= near1 & near;
                near1 |= near;
                shell |= within & ~in;
                if (in) {
                    multi |= solid & in;
                    solid |= in;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (in & (1u << j)) own[j] = min(own[j], id);
                }
            }
        }

        // the next tile's views
        MapView nv{};
        if (stage) nv = load_map_view(p.P.view + next_i);

        solid &= valid;
        const unsigned fluid = valid & ~solid;
        shell &= fluid;
        unsigned wall = wall_xy;
        if (!p.g.per[2]) {
            if (z == 0 || z == nz - 1) wall |= 0x0fu;
            if (z + 1 == nz - 1) wall |= 0xf0u;
        }
        const unsigned miss = solid & (near2 | wall);
        unsigned fresh = 0;   // uncovered now
        if (!FRESH) fresh = (((old0 >> (4 * (lane & 3))) & 15u) | ((old1 >> (4 * (lane & 3))) & 15u) << 4) & fluid;
        near1 &= fluid;
        multi &= solid;
        // refill with the former particle's velocity
        for (unsigned m = fresh; m; m &= m - 1) {
            const int j = __ffs(m) - 1, c = idx + (j & 3) + (j >> 2) * plane;
            const int prev = p.owner[c];
            p.owner[c] = -1;
            const int slot = atomicAdd(p.refill_count, 1);
            if (slot < p.refill_cap) {
                p.refill_list[slot] = (unsigned int)c;
                p.refill_owner[slot] = prev;
            } else {
                atomicOr(p.status, ST_REFILL_OVERFLOW);
            }
        }
        const unsigned write_own = FRESH ? valid : solid;
        if (FRESH) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (own[j] == 0x7fffffff) own[j] = -1;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            auto quad = [&](unsigned m) { return bytes_of((m >> (4 * h)) & 15u); };
            unsigned word = quad(solid) * FL_SOLID + quad(shell) * FL_SHELL + quad(near1) * FL_NEAR;
            if (miss | multi | fresh) word += quad(miss) * FL_MISS + quad(multi) * FL_MULTI + quad(fresh) * FL_NEWFLUID;
            const unsigned v = (valid >> (4 * h)) & 15u, wo = (write_own >> (4 * h)) & 15u;
            uint8_t* const fl = p.flags + (idx + h * plane);
            int* const ow = p.owner + (idx + h * plane);
            if (vec) {
                if (v) *reinterpret_cast<unsigned*>(fl) = word;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (v & (1u << j)) fl[j] = (uint8_t)(word >> (8 * j));
            }
            if (vec && wo == 15u) {
                *reinterpret_cast<int4*>(ow) = make_int4(own[4 * h], own[4 * h + 1], own[4 * h + 2], own[4 * h + 3]);
            } else if (wo) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (wo & (1u << j)) ow[j] = own[4 * h + j];
            }
        }
        bool flush_it = false;
        if (!FRESH) {
            // solid and shell bits of the rows' 16 cells, from their four lanes
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                unsigned bits = (((solid >> (4 * h)) & 15u) | ((shell >> (4 * h)) & 15u) << 16) << (4 * (lane & 3));
                bits |= __shfl_xor_sync(FULL, bits, 1);
                bits |= __shfl_xor_sync(FULL, bits, 2);
                if ((lane & 3) == 0 && y < ny && z + h < nz) {
                    reinterpret_cast<unsigned short*>(p.solid)[half + 2 * h * words] = (unsigned short)bits;
                    reinterpret_cast<unsigned short*>(p.shell)[half + 2 * h * words] = (unsigned short)(bits >> 16);
                }
            }
            solid_count += __popc(solid);
            if (__any_sync(FULL, miss != 0u)) {
                const int n = __popc(miss);
                int at = n;   // inclusive sum over the lanes
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int v = __shfl_up_sync(FULL, at, o);
                    if (lane >= o) at += v;
                }
                unsigned base = 0;
                if (lane == 31) base = atomicAdd(&sh.n_miss, (unsigned)at);
                base = __shfl_sync(FULL, base, 31);
                const unsigned end = base + (unsigned)__shfl_sync(FULL, at, 31);
                flush_it = end > (unsigned)MISS_HELD;
                unsigned slot = base + (unsigned)(at - n);
                for (unsigned m = miss; m; m &= m - 1) {
                    const int j = __ffs(m) - 1;
                    sh.miss[slot++] = (unsigned)(idx + (j & 3) + (j >> 2) * plane);
                }
            }
        }
        if (stage) stage_candidate(p, sh, buf ^ 1, tid, next_i, nv, ox, oy, (bz + 1) * TILE_Z);
        if (tid == 0) p.tile_count[t] = 0;   // consumed: zero for the next scatter
        c_cur = c_nxt;
        c_nxt = c_after;
        if (FRESH) {
            __syncthreads();
        } else if (__syncthreads_or(flush_it || bz + 1 == z1)) {
            // append the cells held back to the list
            const unsigned n = sh.n_miss;
            if (tid == 0 && n) sh.base = (unsigned)atomicAdd(p.miss_count, (int)n);
            __syncthreads();
            for (unsigned k = tid; k < n; k += MAP_THREADS) {
                const unsigned slot = sh.base + k;
                if (slot < (unsigned)p.miss_cap) p.miss_list[slot] = sh.miss[k];
                else atomicOr(p.status, ST_REFILL_OVERFLOW);
            }
            if (tid == 0) sh.n_miss = 0;
            __syncthreads();
        }
    }
    if (!FRESH) {
        const unsigned ws = __reduce_add_sync(FULL, solid_count);
        if (lane == 0) sh.n_solid[warp] = ws;
        __syncthreads();
        if (tid == 0) {
            unsigned n = 0;
#pragma unroll
            for (int w = 0; w < MAP_THREADS / 32; ++w) n += sh.n_solid[w];
            if (n) atomicAdd(p.n_solid, (unsigned long long)n);
        }
    }
}

template <bool FRESH>
__global__ void __launch_bounds__(MAP_THREADS, LBM_MAP_MIN_BLOCKS)
    map_kernel(const __grid_constant__ MapParams p, int depth) {
    const int z0 = (int)blockIdx.z * depth;
    map_body<FRESH>(p, (int)blockIdx.x, (int)blockIdx.y, z0, min(z0 + depth, p.ntile[2]));
}

// Tiles in z that a block walks: as many as keep the blocks resident at once,
// at most four (a longer walk hides more of the loads but leaves an emptier end)
int map_depth(const int* ntile) {
    const long long columns = (long long)ntile[0] * ntile[1];
    const long long d = (columns * ntile[2] + MAP_BLOCKS_WANTED - 1) / MAP_BLOCKS_WANTED;
    return (int)(d < 1 ? 1 : (d > MAP_DEPTH_MAX ? MAP_DEPTH_MAX : d));
}

int map_blocks(const int* ntile) {
    const int d = map_depth(ntile);
    return ntile[0] * ntile[1] * ((ntile[2] + d - 1) / d);
}

// instance i's tiles are walked by its blocks off[i] .. off[i + 1] - 1, x fastest
__global__ void __launch_bounds__(MAP_THREADS, LBM_MAP_MIN_BLOCKS)
    map_gang_kernel(const MapParams* __restrict__ table, const int* __restrict__ off, int n) {
    __shared__ __align__(16) MapParams sp;
    const int i = gang_instance(off, n, (int)blockIdx.x);
    gang_load(table, i, sp);
    const int b = (int)blockIdx.x - off[i];
    const int t0 = sp.ntile[0], t1 = sp.ntile[1], layers = (off[i + 1] - off[i]) / (t0 * t1);
    const int depth = (sp.ntile[2] + layers - 1) / layers;
    const int z0 = b / (t0 * t1) * depth;
    map_body<false>(sp, b % t0, (b / t0) % t1, z0, min(z0 + depth, sp.ntile[2]));
}

void launch_map(const MapParams& p, cudaStream_t st) {
    const int d = map_depth(p.ntile);
    const dim3 grid(p.ntile[0], p.ntile[1], (p.ntile[2] + d - 1) / d);
    if (p.solid) map_kernel<false><<<grid, MAP_THREADS, 0, st>>>(p, d);
    else map_kernel<true><<<grid, MAP_THREADS, 0, st>>>(p, d);
}

// one thread per word of 32 cells
__global__ void cell_bits_kernel(const __grid_constant__ MapParams p) {
    const int nx = p.g.n[0], W = p.ntile[0];
    const long long words = (long long)W * p.g.n[1] * p.g.n[2];
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < words; k += stride) {
        const long long row = k / W;
        const int x0 = (int)(k % W) * 32;
        uint32_t so = 0, sh = 0;
        for (int b = 0; b < 32 && x0 + b < nx; ++b) {
            const uint8_t f = p.flags[row * nx + x0 + b];
            so |= (uint32_t)((f & FL_SOLID) != 0) << b;
            sh |= (uint32_t)((f & FL_SHELL) != 0) << b;
        }
        p.solid[k] = so;
        p.shell[k] = sh;
    }
}

void launch_cell_bits(const MapParams& p, cudaStream_t st) {
    static_assert(TILE_X == 32, "a tile row is one word");
    cell_bits_kernel<<<152 * 8, 128, 0, st>>>(p);
}

// ------------------------------------------------------------ refill

// One warp per uncovered cell: lane q (1..18) reads the neighbour x + c_q
// (its 19 PDFs, when it was fluid before and after the update), the warp sums
// densities and shares the axis neighbours' velocities, and lane q (0..18)
// writes f_q of Eq. (18).
template <typename S>
__device__ __forceinline__ void refill_body(const RefillParams& p, int bx, int gx) {
    using T = typename Store<S>::T;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int count = min(*p.count, p.cap);
    const S* f = static_cast<const S*>(p.f);
    S* fw = static_cast<S*>(p.f);
    const long long N = p.g.ncells;
    const int nx = p.g.n[0], ny = p.g.n[1];
    const T ax = (T)p.accel[0], ay = (T)p.accel[1], az = (T)p.accel[2];
    constexpr unsigned long long PX = pack_dirs(0), PY = pack_dirs(1), PZ = pack_dirs(2);
    const int warps = gx * (blockDim.x >> 5);
    for (int k = bx * (blockDim.x >> 5) + (threadIdx.x >> 5); k < count; k += warps) {   // warp-uniform
        const unsigned cell = p.list[k];
        const long long idx = cell;
        const unsigned yz = cell / (unsigned)nx;
        const int x = (int)(cell % (unsigned)nx);
        const int y = (int)(yz % (unsigned)ny);
        const int z = (int)(yz / (unsigned)ny);
        const int cpos[3] = {x, y, z};
        const int i = p.list_owner[k];
        const int q = lane < Q ? lane : 0;
        const int c[3] = {dir_c(PX, q), dir_c(PY, q), dir_c(PZ, q)};
        // lane q: neighbour x + c_q, fluid before and after the update
        bool ok = false;
        T dr = T(0), jx = T(0), jy = T(0), jz = T(0);
        if (q >= 1) {
            int nb[3] = {x + c[0], y + c[1], z + c[2]};
            bool out = false;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                if (p.g.per[d]) nb[d] = wrap_idx(nb[d], p.g.n[d]);
                else if (nb[d] < 0 || nb[d] >= p.g.n[d]) out = true;
            }
            if (!out) {
                const long long j = ((long long)nb[2] * ny + nb[1]) * nx + nb[0];
                if (!(p.flags[j] & (FL_SOLID | FL_NEWFLUID))) {
                    ok = true;
#pragma unroll
                    for (int r = 0; r < Q; ++r) {
                        const T v = Store<S>::load(f + (long long)r * N + j);
                        dr += v;
                        if (cx(r)) jx += cx(r) > 0 ? v : -v;
                        if (cy(r)) jy += cy(r) > 0 ? v : -v;
                        if (cz(r)) jz += cz(r) > 0 ? v : -v;
                    }
                }
            }
        }
        T drho_sum = dr;   // neighbour densities minus rho0 (shifted, no cancellation)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) drho_sum += __shfl_xor_sync(FULL, drho_sum, o);
        const unsigned okm = __ballot_sync(FULL, ok);
        const int nnb = __popc(okm);
        // velocities of the axis neighbours +x -x +y -y +z -z (lanes 4, 3, 1, 2, 5, 6)
        const T vx = jx - T(0.5) * ax, vy = jy - T(0.5) * ay, vz = jz - T(0.5) * az;
        constexpr int SLOT_Q[6] = {4, 3, 1, 2, 5, 6};
        T uax[6][3];
        bool okax[6];
#pragma unroll
        for (int sl = 0; sl < 6; ++sl) {
            uax[sl][0] = __shfl_sync(FULL, vx, SLOT_Q[sl]);
            uax[sl][1] = __shfl_sync(FULL, vy, SLOT_Q[sl]);
            uax[sl][2] = __shfl_sync(FULL, vz, SLOT_Q[sl]);
            okax[sl] = (okm >> SLOT_Q[sl]) & 1u;
        }
        const T drb = nnb ? drho_sum / (T)nnb : T(0);
        const T rb = T(1) + drb;
        // velocity of the former particle at the cell centre (rigid body)
        T ut[3], rr[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double dd = ((double)cpos[d] + 0.5) - p.P.x[3 * i + d];
            if (p.g.per[d]) {
                double half = 0.5 * p.g.n[d];
                if (dd > half) dd -= p.g.n[d];
                if (dd < -half) dd += p.g.n[d];
            }
            rr[d] = (T)dd;
        }
        const T om0 = (T)p.P.om[3 * i], om1 = (T)p.P.om[3 * i + 1], om2 = (T)p.P.om[3 * i + 2];
        ut[0] = (T)p.P.u[3 * i] + (om1 * rr[2] - om2 * rr[1]);
        ut[1] = (T)p.P.u[3 * i + 1] + (om2 * rr[0] - om0 * rr[2]);
        ut[2] = (T)p.P.u[3 * i + 2] + (om0 * rr[1] - om1 * rr[0]);
        T g[3][3];   // g[a][b] = d u_a / d x_b
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int sp = 2 * b, sm = 2 * b + 1;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (okax[sp] && okax[sm]) g[a][b] = T(0.5) * (uax[sp][a] - uax[sm][a]);
                else if (okax[sp]) g[a][b] = uax[sp][a] - ut[a];
                else if (okax[sm]) g[a][b] = ut[a] - uax[sm][a];
                else g[a][b] = T(0);
            }
        }
        if (lane < Q) {
            const T coef = (T)p.cs2_over_s_nu;
            const T cf[3] = {(T)c[0], (T)c[1], (T)c[2]};
            T second = T(0);
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const T pab = rb * ut[a] * ut[b] - rb * coef * (g[a][b] + g[b][a]);
                    second += pab * (cf[a] * cf[b] - (a == b ? T(1) / T(3) : T(0)));
                }
            const T cu = cf[0] * ut[0] + cf[1] * ut[1] + cf[2] * ut[2];
            const int cc = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
            const T w = cc == 0 ? T(1) / T(3) : (cc == 1 ? T(1) / T(18) : T(1) / T(36));
            // f_q - w_q written without forming f_q: w_q (rho_bar - 1) + ...
            const T dfq = w * (drb + T(3) * rb * cu + T(4.5) * second);
            Store<S>::store(fw + (long long)q * N + idx, dfq);
        }
    }
}

template <typename S>
__global__ void __launch_bounds__(128) refill_kernel(const RefillParams p) {
    refill_body<S>(p, (int)blockIdx.x, (int)gridDim.x);
}

template <typename S>
__global__ void __launch_bounds__(128) refill_gang_kernel(const RefillParams* __restrict__ table,
                                                          const int* __restrict__ off, int n) {
    __shared__ __align__(16) RefillParams sp;
    const int i = gang_instance(off, n, (int)blockIdx.x);
    gang_load(table, i, sp);
    refill_body<S>(sp, (int)blockIdx.x - off[i], off[i + 1] - off[i]);
}

void launch_map_gang(int kind, int storage, const void* table, const int* off, int n, int blocks, cudaStream_t st) {
    if (n <= 0 || blocks <= 0) return;
    if (kind == GANG_SCATTER) {
        tile_scatter_gang_kernel<<<blocks, 128, 0, st>>>(static_cast<const MapParams*>(table), off, n);
    } else if (kind == GANG_MAP) {
        map_gang_kernel<<<blocks, MAP_THREADS, 0, st>>>(static_cast<const MapParams*>(table), off, n);
    } else {
        const RefillParams* t = static_cast<const RefillParams*>(table);
        switch (storage) {
            case 0: refill_gang_kernel<double><<<blocks, 128, 0, st>>>(t, off, n); break;
            case 1: refill_gang_kernel<float><<<blocks, 128, 0, st>>>(t, off, n); break;
            case 2: refill_gang_kernel<__half><<<blocks, 128, 0, st>>>(t, off, n); break;
            default: refill_gang_kernel<__nv_bfloat16><<<blocks, 128, 0, st>>>(t, off, n); break;
        }
    }
}

void launch_refill(const RefillParams& p, cudaStream_t st) {
    // 4 warps (cells) per block; some 32 cells a particle at once, more take turns
    const int blocks = p.P.n < 152 ? 8 * p.P.n : 152 * 8, threads = 128;
    switch (p.storage) {
        case 0: refill_kernel<double><<<blocks, threads, 0, st>>>(p); break;
        case 1: refill_kernel<float><<<blocks, threads, 0, st>>>(p); break;
        case 2: refill_kernel<__half><<<blocks, threads, 0, st>>>(p); break;
        default: refill_kernel<__nv_bfloat16><<<blocks, threads, 0, st>>>(p); break;
    }
}

// ------------------------------------------------------------ fields

template <typename S>
__global__ void fields_kernel(const FieldsParams p) {
    using T = typename Store<S>::T;
    const S* f = static_cast<const S*>(p.f);
    const long long N = p.g.ncells;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < p.count;
         k += (long long)gridDim.x * blockDim.x) {
        const long long idx = p.first_cell + k;
        double rho = 0, u[3] = {0, 0, 0};
        if (!(p.flags[idx] & FL_SOLID)) {
            // moments in the compute precision (float64 sums cost ten times
            // the read-out on GB300 and change u by less than 1e-8 relative)
            T dr = T(0), jx = T(0), jy = T(0), jz = T(0);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const T v = Store<S>::load(f + (long long)q * N + idx);
                dr += v;
                jx += (T)cx(q) * v;
                jy += (T)cy(q) * v;
                jz += (T)cz(q) * v;
            }
            rho = 1.0 + (double)dr;
            u[0] = (double)jx - 0.5 * p.accel[0];
            u[1] = (double)jy - 0.5 * p.accel[1];
            u[2] = (double)jz - 0.5 * p.accel[2];
        }
        p.out[k] = rho;
        p.out[p.count + k] = u[0];
        p.out[2 * p.count + k] = u[1];
        p.out[3 * p.count + k] = u[2];
    }
}

void launch_fields(const FieldsParams& p, cudaStream_t st) {
    const int blocks = 152 * 8, threads = 256;
    switch (p.storage) {
        case 0: fields_kernel<double><<<blocks, threads, 0, st>>>(p); break;
        case 1: fields_kernel<float><<<blocks, threads, 0, st>>>(p); break;
        case 2: fields_kernel<__half><<<blocks, threads, 0, st>>>(p); break;
        default: fields_kernel<__nv_bfloat16><<<blocks, threads, 0, st>>>(p); break;
    }
}

// density at sample points: trilinear interpolation of the cell-centred
// density (cell i has its centre at i + 1/2); periodic axes wrap, wall axes
// clamp to the first and last cell; solid cells count with the reference
// density 1. Eight lanes per point, one per corner cell: a thread per point read
// the corners one after the other, eight times the latency of the PDFs.
template <typename S>
__global__ void sample_density_kernel(const SampleParams p) {
    using T = typename Store<S>::T;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = t >> 3, c = t & 7;
    if (t == 0 && p.status_out) *p.status_out = *p.status;
    const bool on = k < p.n;
    const S* f = static_cast<const S*>(p.f);
    const long long N = p.g.ncells;
    double wgt = 1.0, rho = 1.0;
    if (on) {
        int idx3[3];
        for (int d = 0; d < 3; ++d) {
            const double g = p.pos[3 * k + d] - 0.5;
            const double b = floor(g);
            const double w = g - b;
            const int o = (c >> d) & 1;
            int i = (int)b + o;
            const int n = p.g.n[d];
            if (p.g.per[d]) i = ((i % n) + n) % n;
            else i = i < 0 ? 0 : (i >= n ? n - 1 : i);
            idx3[d] = i;
            wgt *= o ? w : 1.0 - w;
        }
        const long long idx = ((long long)idx3[2] * p.g.n[1] + idx3[1]) * p.g.n[0] + idx3[0];
        if (!(p.flags[idx] & FL_SOLID)) {
            T dr = T(0);
#pragma unroll
            for (int q = 0; q < Q; ++q) dr += Store<S>::load(f + (long long)q * N + idx);
            rho = 1.0 + (double)dr;
        }
    }
    double v = 0.0;   // the corners in order
    for (int o = 0; o < 8; ++o) {
        const double w = __shfl_sync(0xffffffffu, wgt, o, 8), r = __shfl_sync(0xffffffffu, rho, o, 8);
        v += w * r;
    }
    if (on && c == 0) p.out[k] = v;
}

void launch_sample_density(const SampleParams& p, cudaStream_t st) {
    if (p.n <= 0) return;
    const int blocks = (8 * p.n + 127) / 128;
    switch (p.storage) {
        case 0: sample_density_kernel<double><<<blocks, 128, 0, st>>>(p); break;
        case 1: sample_density_kernel<float><<<blocks, 128, 0, st>>>(p); break;
        case 2: sample_density_kernel<__half><<<blocks, 128, 0, st>>>(p); break;
        default: sample_density_kernel<__nv_bfloat16><<<blocks, 128, 0, st>>>(p); break;
    }
}

}  // namespace lbmdem
