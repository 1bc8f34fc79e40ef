// stream_collide.cu -- the dense kernel of one lattice Boltzmann step with
// moving particles (Algorithm 1, lines 1-3): pull streaming (Eq. (2)), the
// particle links (CLI moving no-slip condition, Eq. (14), and momentum
// exchange, Eqs. (15)-(17)), halfway bounce-back on the walls of the box
// (Eq. (14), delta = 1/2, wall velocity), then the two-relaxation-time
// collision (Eq. (10), magic parameter Eq. (11)) with Guo forcing; in TRT+aB
// shell cells (Sec. 2.3.2) and for Lambda_b,bulk != 1 the two bulk moments m4,
// m5 relax with s_b (Eq. (12)) through a rank-2 correction in moment space.
//
// PDFs are stored shifted (f_q - w_q) in SoA layout f[q][z][y][x], read from
// one buffer and written to the other. What a solid cell's slots hold is
// never used: which pulls are particle links is read from the mapping's bit
// per cell (solid), so a warp finds the links of a row of 32 cells with a few
// word operations per direction instead of testing 18 pulled values per cell.
//
// A warp works alone (no block barriers) on 32 x 2 cells (32 x 1 in float64) of
// one z plane after the other. For each plane it
//   1. forms the link words of its cells, lane q for direction q: fluid(x) &
//      solid(x - c_q), starts its pulls, and queues the links in shared memory,
//      the left half of the cells first (links of one sphere then mostly share
//      a chunk);
//   2. takes the queue 32 links at a time, one per lane: CLI value into the
//      cell's slot in shared memory, force and torque into the lane's open sums
//      of the particle, kept in shared memory over the planes for the last few
//      particles (added to a particle when its slot is needed and at the end);
//   3. patches the linked values in, collides and stores. Float32 collides the
//      two rows in packed arithmetic.
// Sectors of 32 bytes with a fluid cell are written whole (solid cells get
// whatever the arithmetic gives), so DRAM never has to merge part of one.
//
// What bounds it (256 x 256 x 512 cells, 10,000 spheres, 27 % solids, float32):
// instruction issue and latency together, 900 warp instructions per row of 32
// cells (1,310 with a test of every pulled value for a marker, one row per warp
// and force sums flushed when a lane's particle changed) at 51 % issue; 1.38 ms
// against 1.58 ms that way, 128 x 128 x 256 cells 216 us against 284 us, float16
// 192^3 with 2,000 spheres 334 us against 466 us. Streaming alone takes the
// memory's time (95 us of the 128 x 128 x 256 case at 6.7 TB/s).
//
// Per-particle sums. Float64 storage: float64 sums per lane and warp, float64
// atomics. Float32 compute: the link force splits into the constant part
// 2 w_p c_p and the small remainder c_p (f~_p + f_q) - u_b (f~_p - f_q). The
// constant parts and their torques over a particle's fluid links are minus
// those over its other links (the links of a set of cells to its outside
// cancel), so boundary.cu adds them from the few cells that have others; the
// remainder is summed per lane and warp in float32 and per particle in 64-bit
// fixed point (scale 2^32) through integer atomics. The sums depend on the
// chunk of planes a warp marches, not on the tile width.
//
// A box with one particle, float32 compute, has a form of its own. The force and
// torque on a sphere of an array are a small rest of their links' parts (a torque
// of 1e-5 to 1e-3 where the parts add up to 10), so the order in which float32
// adds them shows in the fifth digit. This form adds them per row, in the order of
// the row's cells and directions, cut into runs of equal length of which column c
// of the row's sums takes the c-th: each torque of an array is then the one that a
// warp per row has, bit for bit. It costs nothing: with one particle there is no
// owner to look up, no slot to find, and the words of the row's directions, once
// turned into the lane's own directions, serve to patch the values in too (a pass
// of the 80x80x160 box 2.63 ms against 2.62 with the sums by slot, 16 boxes of a
// batch 8.55 against 8.52, 480x160x80 cells 9.36 and 9.37).
#include <cstring>

#include "sc_common.cuh"

// resident blocks of 128 threads per SM (a register cap); tuned on GB300
#ifndef LBM_SC_MIN_BLOCKS
#define LBM_SC_MIN_BLOCKS 4
#endif
// the same for float64 storage
#ifndef LBM_SC_MIN_BLOCKS_F64
#define LBM_SC_MIN_BLOCKS_F64 4
#endif
// longest chunk of consecutive z planes marched by one block (shorter when
// the box is too small to give every SM several blocks); tuned on GB300
#ifndef LBM_SC_ZCHUNK
#define LBM_SC_ZCHUNK 16
#endif

namespace lbmdem {

constexpr int SC_WARPS = 4;       // warps per block
constexpr int QUEUE_CAP = 256;    // links queued at a time

// Shared memory of one warp. A cell is numbered half (x < 16 or not) << 5 |
// row << 4 | x & 15; a queue entry is q << 11 | p << 6 | cell, p opposite to q (p
// is put in when it is read in the form for one particle).
template <typename T>
struct SCWarp {
    static constexpr int ROWS = Pack<T>::ROWS;
    T v[Q - 1][32 * ROWS];                   // CLI values
    OpenParts<T> open;
    alignas(8) uint32_t w[Q + 2][ROWS];      // link words of directions 1 .. 18, fluid, shell
    unsigned short queue[QUEUE_CAP];
};
// cell number of x = lane, row 0 (row 1: + 16)
template <typename T>
__device__ __forceinline__ int cell_of(int lane) {
    return Pack<T>::ROWS == 1 ? lane : ((lane & 16) << 1) | (lane & 15);
}

// what one link reads: queue entry (bit 16: CLI), particle, PDFs
template <typename T>
struct LinkIn {
    int e, key;
    T fout, fin, fdown;
};

// a lane's words of one plane (see sc_warp)
struct PlaneWords {
    uint32_t at[2], side[2];
};

// g = *v where bit is set: a predicated load. The statement says that it reads
// memory, which costs nothing (256 x 256 x 512 cells 16.42 ms a pass with and 16.41
// without); `if (bit) g = *v` takes 16.54 and a load with a select 16.75.
__device__ __forceinline__ void patch_link(float& g, uint32_t bit, const float* v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p ld.shared.f32 %0, [%2];\n\t}"
                 : "+f"(g) : "r"(bit), "r"((uint32_t)__cvta_generic_to_shared(v)) : "memory");
}
__device__ __forceinline__ void patch_link(double& g, uint32_t bit, const double* v) {
    if (bit) g = *v;
}

// what a kernel is compiled for: boxes with one particle (see the header), other
// boxes, both
enum Boxes { BOXES_MORE, BOXES_ONE, BOXES_BOTH };

// One warp's cells: x = 32 wx + lane, rows y0 .. y0 + ROWS - 1, planes
// z_begin .. z_end - 1 marched in order.
template <typename S, typename T, Boxes KIND>
__device__ __forceinline__ void sc_warp(const SCArgs<S, T>& a, int wx, int y0, int z_begin, int z_end, SCWarp<T>& sm,
                                        const DirTable<S>& dt) {
    using P = Pack<T>;
    constexpr int ROWS = P::ROWS;
    const int nx = a.g.n[0], ny = a.g.n[1], nz = a.g.n[2];
    const unsigned FULL = 0xffffffffu;
    int lane;   // opaque, or the compiler reads the special register again and again
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    const int plane = nx * ny;
    const int W = a.words;
    const int x = 32 * wx + lane;
    const int xl = x < nx ? x : nx - 1;          // lanes past the row load its last cell
    const bool last_word = wx == W - 1;
    const uint32_t valid = last_word && (nx & 31) ? (1u << (nx & 31)) - 1u : FULL;
    const bool rowB = ROWS > 1 && y0 + 1 < ny;   // the second row exists
    // pull offsets in the plane: rows y0 - 1 .. y0 + ROWS, columns x - 1 .. x + 1
    const int xo[3] = {xl == 0 ? nx - 1 : xl - 1, xl, xl == nx - 1 ? 0 : xl + 1};
    int yo[ROWS + 2];
#pragma unroll
    for (int r = 0; r < ROWS + 2; ++r) {
        int yy = y0 - 1 + r;
        yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
        yo[r] = yy * nx;
    }
    const T ax = a.accel[0], ay = a.accel[1], az = a.accel[2];
    const Sinks sk{a.acc_d, a.acc_i, nullptr, a.status};

    SlotKeys<T> keys;
#pragma unroll
    for (int j = 0; j < OpenParts<T>::SLOTS; ++j) keys.k[j] = -1;
    keys.next = 0;

    // Words of a plane: lane q - 1 holds direction q's upstream words and the
    // neighbouring ones whose bit shifts in (behind a wall there are no links),
    // lane 18 the solid, lane 19 the shell words of the warp's own rows; loaded
    // a plane ahead.
    const int ql = lane < Q - 1 ? lane + 1 : 0;
    int wz = 0;               // the words' plane: z - wz
    int woff[ROWS], wside;    // word of each row, of the neighbouring word relative to it
    uint32_t wcfg;            // rows on in bits 0-1, shift left / right 2-3, carry on 4, side bit 8-12, carry bit 16-20
    {
        const int qi = dt.qi[ql];
        const int c0 = (qi & 3) - 1, c1 = ((qi >> 2) & 3) - 1;
        wz = ((qi >> 4) & 3) - 1;
        const bool carry = c0 != 0 && (a.g.per[0] || !((c0 > 0 && wx == 0) || (c0 < 0 && last_word)));
        wcfg = (c0 > 0 ? 4u : 0u) | (c0 < 0 ? 8u : 0u) | (carry ? 16u : 0u) |
               (c0 > 0 ? (uint32_t)(wx > 0 ? 31 : (nx - 1) & 31) << 8 : (uint32_t)(last_word ? (nx - 1) & 31 : 31) << 16);
        wside = c0 > 0 ? (wx > 0 ? -1 : W - 1) : (c0 < 0 ? (last_word ? 1 - W : 1) : 0);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            int yu = y0 + r - c1;
            if (ql ? a.g.per[1] || (yu >= 0 && yu < ny) : true) wcfg |= 1u << r;
            yu = yu < 0 ? yu + ny : (yu >= ny ? yu - ny : yu);
            woff[r] = yu * W + wx;
        }
    }
    const uint32_t* const wbase = lane == Q ? a.shell : a.solid;
    auto load_words = [&](int z) {
        PlaneWords s;
        int zu = z - wz;
        const bool in = a.g.per[2] || (unsigned)zu < (unsigned)nz;
        zu = zu < 0 ? zu + nz : (zu >= nz ? zu - nz : zu);
        const uint32_t* p = wbase + zu * (ny * W);
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            s.at[r] = p[woff[r]];
            s.side[r] = p[woff[r] + wside];
            if (!in) s.at[r] = s.side[r] = 0u;
        }
        return s;
    };
    PlaneWords pw = load_words(z_begin);

    const bool one = KIND == BOXES_ONE || (KIND == BOXES_BOTH && a.np == 1);
    int lanes[2] = {0, 0};   // one: lanes with a sum, per row

    // the gathers of queue entry e of a plane; edges: bit d, the warp's cells
    // reach the box's faces on axis d
    auto fetch = [&](int e, int z, int edges) {
        LinkIn<T> l;
        const int q = e >> 11, p = (e >> 6) & 31, row = (e >> 4) & (ROWS - 1);
        const int xb = ROWS == 1 ? e & 31 : (e & 15) | ((e >> 1) & 16);
        const int idx = z * plane + y0 * nx + 32 * wx + (row ? nx : 0) + xb, dq = dt.dq[q];
        // x + c_q must be fluid and inside the box for CLI; its post-collision
        // f_p is the cell's own pull in direction p
        bool cli = !((sm.w[p][row] >> xb) & 1u);
        int is = idx - dq, id = idx + dq;
        if (edges) {
            const int qi = dt.qi[q];
            const int pos[3] = {32 * wx + xb, y0 + row, z};
            const int step[3] = {nx, plane, (int)a.g.ncells};
#pragma unroll
            for (int d = 0; d < 3; ++d)
                if ((edges >> d) & 1) {
                    const int n_d = a.g.n[d], c = ((qi >> (2 * d)) & 3) - 1, us = pos[d] - c, ds = pos[d] + c;
                    if (!a.g.per[d] && (unsigned)ds >= (unsigned)n_d) cli = false;
                    is += us < 0 ? step[d] : (us >= n_d ? -step[d] : 0);
                    id += ds < 0 ? step[d] : (ds >= n_d ? -step[d] : 0);
                }
        }
        const S* const sp = dt.src[p];
        l.key = one ? 0 : a.owner[is];
        l.fout = Store<S>::load(sp + idx);
        l.fin = Store<S>::load(dt.src[q] + idx);
        const T fd = Store<S>::load(sp + id);
        l.fdown = cli ? fd : T(0);
        l.e = e | (cli ? 0x10000 : 0);
        return l;
    };

    // link l of particle key: its value into the cell's slot, its force and torque
    // into the sums of slot, column col (float64: to the particle at once without a
    // slot)
    auto add_link = [&](const LinkIn<T>& l, int key, int slot, int col, int z, bool wrap) {
        const int q = (l.e >> 11) & 31, row = (l.e >> 4) & (ROWS - 1);
        const int xb = ROWS == 1 ? l.e & 31 : (l.e & 15) | ((l.e >> 1) & 16);
        T F[6];
        sm.v[q - 1][l.e & (32 * ROWS - 1)] =
            link_value<S>(a, key, sm.open.view[sizeof(T) == 4 && !one ? slot : 0], 32 * wx + xb, y0 + row, z, dt.qi[q],
                          dt.cf[q], (l.e & 0x10000) != 0, wrap, l.fout, l.fin, l.fdown, F);
        if (sizeof(T) == 4 || slot >= 0) {
            T* p = &sm.open.f[slot][0][col];
#pragma unroll
            for (int d = 0; d < 6; ++d) p[32 * d] += F[d];
        } else {
#pragma unroll
            for (int d = 0; d < 6; ++d) add_float(sk, key, d, F[d]);
        }
    };

    // axes on which the warp's cells lie next to the box's faces, and z planes
    // in which no image of a particle near the tile's links matters
    const int wall_axes = (a.g.per[0] ? 0 : 1) | (a.g.per[1] ? 0 : 2) | (a.g.per[2] ? 0 : 4);
    const int edges_xy = (wx == 0 || last_word ? 1 : 0) | (y0 == 0 || y0 + ROWS >= ny ? 2 : 0);
    const int mx = a.g.per[0] ? a.margin : 1, my = a.g.per[1] ? a.margin : 1, mz = a.g.per[2] ? a.margin : 1;
    const bool deep_xy = 32 * wx >= mx && 32 * wx + 31 < nx - mx && y0 >= my && y0 + ROWS <= ny - my;

    for (int z = z_begin; z < z_end; ++z) {
        // 1. link words and queue
        __syncwarp();   // the last plane's words and values are read
        uint32_t link[2] = {0u, 0u};
        {
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                const uint32_t u = pw.at[r];
                const uint32_t carry = wcfg & 16u ? ((pw.side[r] >> ((wcfg >> 8) & 31)) & 1u) << ((wcfg >> 16) & 31) : 0u;
                const uint32_t v = ((u << ((wcfg >> 2) & 1)) >> ((wcfg >> 3) & 1)) | carry;
                link[r] = (wcfg >> r) & 1u ? v : 0u;
                // the second row of the last pair may not exist
                if (lane == Q - 1) link[r] = r == 0 || rowB ? ~v & valid : 0u;
                if (lane < Q + 1) sm.w[lane + 1][r] = link[r];
            }
        }
        if (z + 1 < z_end) pw = load_words(z + 1);
        __syncwarp();
        uint32_t fluid[2] = {sm.w[Q][0], ROWS > 1 ? sm.w[Q][ROWS - 1] : 0u};
        if ((fluid[0] | fluid[1]) == 0u) continue;   // warp-uniform
        link[0] = ql ? link[0] & fluid[0] : 0u;
        link[1] = ql ? link[1] & fluid[1] : 0u;
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
            if (ql) sm.w[ql][r] = link[r];
        // the pulls are under way while the links are worked on; lanes of a
        // sector without fluid idle
        constexpr int SECT = 32 / (int)sizeof(S) < 32 ? 32 / (int)sizeof(S) : 32;
        const uint32_t sect = (uint32_t)((1ull << SECT) - 1ull) << (lane & ~(SECT - 1));
        const bool actA = (fluid[0] & sect) != 0u, actB = ROWS > 1 && (fluid[1] & sect) != 0u;
        const int zoff[3] = {(z == 0 ? nz - 1 : z - 1) * plane, z * plane, (z == nz - 1 ? 0 : z + 1) * plane};
        typename P::V f[Q];
        if (actA || actB) {
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                T g[ROWS];
#pragma unroll
                for (int r = 0; r < ROWS; ++r)
                    g[r] = Store<S>::load(a.src[q] + (zoff[1 - cz(q)] + yo[1 + r - cy(q)] + xo[1 - cx(q)]));
                f[q] = P::make(g);
            }
        }
        const int edges = edges_xy | (z == 0 || z == nz - 1 ? 4 : 0);
        bool links;   // warp-uniform
        int cl = 0, cr = 0, incl = 0, left = 0, total = 0;
        if (one) {
            links = __any_sync(FULL, (link[0] | link[1]) != 0u);
        } else {
            // links of the left half (low 16 bits) and of the right half (high); with
            // one row all count as left, the order in which they are queued below
            cl = ROWS == 1 ? __popc(link[0]) : __popc(link[0] & 0xffffu) + __popc(link[1] & 0xffffu);
            cr = ROWS == 1 ? 0 : __popc(link[0] >> 16) + __popc(link[1] >> 16);
            incl = warp_incl_scan(cl | (cr << 16), lane);
            const int all = __shfl_sync(FULL, incl, 31);
            left = all & 0xffff;
            total = left + (all >> 16);
            links = total > 0;
        }
        uint32_t of_cell[2] = {0u, 0u};   // one: bit q - 1, the lane's cell has a link in direction q
        if (one && links) {
            // 2. the links of each row in the order of its cells, cut into runs of equal
            // length, one per lane
            const bool wrap = !(deep_xy && z >= mz && z < nz - mz);
            if ((lanes[0] | lanes[1]) == 0) open_single<T>(sm.open, a.view, lane);
            __syncwarp();   // the words of all directions
#pragma unroll
            for (int q = Q - 1; q >= 1; --q)
#pragma unroll
                for (int r = 0; r < ROWS; ++r)
                    of_cell[r] = __funnelshift_l(sm.w[q][r] << (31 - lane), of_cell[r], 1);
            const int count = __popc(of_cell[0]) | __popc(of_cell[1]) << 16;
            const int end = warp_incl_scan(count, lane), all = __shfl_sync(FULL, end, 31);
            const int first[2] = {((end - count) & 0xffff), (end - count) >> 16}, n[2] = {all & 0xffff, all >> 16};
            int run[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                run[r] = (n[r] + 31) >> 5;
                lanes[r] = max(lanes[r], run[r] > 1 ? (n[r] + run[r] - 1) / run[r] : n[r]);
            }
            constexpr int CAP = QUEUE_CAP / 2;   // of a row's links queued at a time
            for (int base = 0; base < max(n[0], n[1]); base += CAP) {
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    int pos = first[r] - base;
                    for (uint32_t m = of_cell[r]; m; m &= m - 1, ++pos)
                        if ((unsigned)pos < (unsigned)CAP)
                            sm.queue[CAP * r + pos] = (unsigned short)(__ffs((int)m) << 11 | (cell_of<T>(lane) + 16 * r));
                }
                __syncwarp();
                // 32 links at a time, the j-th of each run of the first row and then of
                // the second
                for (int j = 0; j < max(run[0], run[1]); ++j) {
                    int runs[2];   // with a j-th link
#pragma unroll
                    for (int r = 0; r < 2; ++r)
                        runs[r] = j >= run[r] ? 0 : (run[r] > 1 ? (n[r] - j + run[r] - 1) / run[r] : n[r]);
                    for (int u0 = 0; u0 < runs[0] + runs[1]; u0 += 32) {
                        const int u = u0 + lane, r = u < runs[0] ? 0 : 1;
                        const int col = r ? u - runs[0] : u;
                        const int k = col * (r ? run[1] : run[0]) + j - base;
                        if (u < runs[0] + runs[1] && (unsigned)k < (unsigned)CAP) {
                            const int e = sm.queue[CAP * r + k];
                            add_link(fetch(e | ((dt.qi[e >> 11] >> 6) & 31) << 6, z, edges), 0, r, col, z, wrap);
                        }
                        __syncwarp();   // queue read, values and sums written
                    }
                }
            }
        } else if (links) {
            const bool wrap = !(deep_xy && z >= mz && z < nz - mz);
            const int pl = (incl & 0xffff) - cl, pr = left + (incl >> 16) - cr;
            for (int base = 0; base < total; base += QUEUE_CAP) {
                // this lane's links of direction ql with places in [base, base + QUEUE_CAP)
                const bool all_fit = total <= QUEUE_CAP;
#pragma unroll
                for (int h = 0; h < (ROWS == 1 ? 1 : 2); ++h) {
                    int pos = (h == 0 ? pl : pr) - base;
                    const int e0 = (ql << 11) | (((dt.qi[ql] >> 6) & 31) << 6) | (h << 5);
                    uint32_t m = ROWS == 1 ? link[0]
                                           : (h == 0 ? __byte_perm(link[0], link[1], 0x5410)
                                                     : __byte_perm(link[0], link[1], 0x7632));
                    while (m) {
                        const int b = 31 - __clz((int)m);
                        m ^= 1u << b;
                        if (all_fit || (unsigned)pos < (unsigned)QUEUE_CAP) sm.queue[pos] = (unsigned short)(e0 + b);
                        ++pos;
                    }
                }
                __syncwarp();
                // 2. one link per lane (the last one for lanes past the end); the
                // gathers of the next 32 are under way while these are worked on
                const int n = min(total - base, QUEUE_CAP);
                LinkIn<T> l = fetch(sm.queue[min(lane, n - 1)], z, edges);
                for (int k0 = 0; k0 < n; k0 += 32) {
                    const LinkIn<T> cur = l;
                    if (k0 + 32 < n) l = fetch(sm.queue[min(k0 + 32 + lane, n - 1)], z, edges);
                    // solid cells have an owner below np
                    int key = k0 + lane < n && (unsigned)cur.key < (unsigned)a.np ? cur.key : -1;
                    // once, but where more particles meet than there are slots. A float64 link
                    // is 150 instructions of 64 cycles and is worked on once all the same
                    // (6,000 spheres of diameter 5 in 96x96x128 cells 3.26 ms with a turn per
                    // group of slots, 1.63 this way)
                    do {
                        const int slot = find_slot<T>(sm.open, keys, key, a.view, sk, lane);
                        if (slot >= 0 || (sizeof(T) == 8 && key >= 0)) {
                            add_link(cur, key, slot, lane, z, wrap);
                            key = -1;
                        }
                    } while (__any_sync(FULL, key >= 0));
                }
                __syncwarp();   // queue read, values written
            }
        }
        // 3. patch, collide, store
        if (actA || actB) {
            const uint32_t me = 1u << lane;
            const bool edge = (edges & wall_axes) != 0;
            if (edge) {
                // halfway bounce-back on the box walls (Eq. (14) with delta = 1/2)
#pragma unroll
                for (int q = 1; q < Q; ++q) {
                    const int p = opp(q);
                    T g[ROWS];
                    P::get(f[q], g);
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        // upstream outside: direction +1 from the low face, -1 from the high one
                        const bool oz = cz(q) && !a.g.per[2] && z == (cz(q) > 0 ? 0 : nz - 1);
                        const bool oy = cy(q) && !a.g.per[1] && y0 + r == (cy(q) > 0 ? 0 : ny - 1);
                        const bool ox = cx(q) && !a.g.per[0] && xl == (cx(q) > 0 ? 0 : nx - 1);
                        if (!(oz || oy || ox)) continue;
                        T ucp = T(0);   // c_p . u_wall, the z face before the y face before the x face
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const int cd = d == 0 ? cx(q) : (d == 1 ? cy(q) : cz(q));
                            const T uz = a.uw[cz(q) > 0 ? 0 : 1][2][d], uy = a.uw[cy(q) > 0 ? 0 : 1][1][d],
                                    ux = a.uw[cx(q) > 0 ? 0 : 1][0][d];
                            ucp += (oz ? uz : (oy ? uy : ux)) * (T)(-cd);
                        }
                        g[r] = Store<S>::load(a.src[p] + (zoff[1] + yo[1 + r] + xl)) - T(6) * wq<T>(p) * ucp;
                    }
                    f[q] = P::make(g);
                }
            }
            if (links) {
#pragma unroll
                for (int q = 1; q < Q; ++q) {
                    T g[ROWS];
                    P::get(f[q], g);
#pragma unroll
                    for (int r = 0; r < ROWS; ++r)
                        patch_link(g[r], one ? of_cell[r] & (1u << (q - 1)) : sm.w[q][r] & me,
                                   &sm.v[q - 1][cell_of<T>(lane) + 16 * r]);
                    f[q] = P::make(g);
                }
            }
            bool sh[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) sh[r] = (sm.w[Q + 1][r] & me) != 0u;
            T dr[ROWS];
            // without a body force its sums are left out: float64, each instruction 64
            // cycles of the unit, 32x32x64 cells 43.0 -> 39.4 us; boxes with one particle
            // in float32, a pass of the 80x80x160 box 2.67 -> 2.63 ms. With many
            // particles the second copy of the collision costs more than it gives
            // (256 x 256 x 512 cells 1380 us without, 1411 with it).
            if ((sizeof(T) == 8 || KIND == BOXES_ONE) && ax == T(0) && ay == T(0) && az == T(0))
                P::get(collide_core<T, false>(f, sh, ax, ay, az, dt.force, a.s_plus, a.s_minus, a.gp, a.s_b_shell,
                                             a.s_b_bulk, a.bulk_corr),
                       dr);
            else
                P::get(collide_core<T, true>(f, sh, ax, ay, az, dt.force, a.s_plus, a.s_minus, a.gp, a.s_b_shell,
                                            a.s_b_bulk, a.bulk_corr),
                       dr);
            bool stable = true;
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
                if ((fluid[r] & me) && !(dr[r] < T(0.5) && dr[r] > T(-0.5))) stable = false;
            if (!stable) atomicOr(a.status, ST_UNSTABLE);
            const int iA = zoff[1] + yo[1] + xl, iB = zoff[1] + yo[ROWS] + xl;
            const bool stA = actA && x < nx, stB = actB && x < nx;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                T g[ROWS];
                P::get(f[q], g);
                if (stA) Store<S>::store(a.dst[q] + iA, g[0]);
                if (ROWS > 1 && stB) Store<S>::store(a.dst[q] + iB, g[ROWS - 1]);
            }
        }
    }
    if (one) {
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
            if (lanes[r] > 0) commit_lanes<T>(sm.open, r, lanes[r], sk, lane);
    } else {
        commit_open<T>(sm.open, keys, sk, lane);
    }
}

__constant__ int k_qinfo[Q] = {qinfo(0), qinfo(1), qinfo(2), qinfo(3), qinfo(4), qinfo(5), qinfo(6),
                               qinfo(7), qinfo(8), qinfo(9), qinfo(10), qinfo(11), qinfo(12), qinfo(13),
                               qinfo(14), qinfo(15), qinfo(16), qinfo(17), qinfo(18)};

// the direction table into shared memory (before the first tile)
template <typename S, typename T>
__device__ __forceinline__ void load_dirs(DirTable<S>& dt, const SCArgs<S, T>& a) {
    const int t = threadIdx.x;
    if (t < Q) {
        const int qi = k_qinfo[t];
        const float c0 = (float)((qi & 3) - 1), c1 = (float)(((qi >> 2) & 3) - 1), c2_ = (float)(((qi >> 4) & 3) - 1);
        dt.qi[t] = qi;
        dt.dq[t] = (qi & 3) - 1 + (((qi >> 2) & 3) - 1) * a.g.n[0] + (((qi >> 4) & 3) - 1) * a.g.n[0] * a.g.n[1];
        dt.src[t] = a.src[t];
        dt.cf[t] = make_float4(-c0, -c1, -c2_, c0 * c0 + c1 * c1 + c2_ * c2_);
        dt.force[t] = force_terms<T>(qi, a.accel[0], a.accel[1], a.accel[2], a.gp, a.gm);
    }
}

// the warp of a tile of bx x (SC_WARPS ROWS 32 / bx) cells at (x0, y0)
template <typename S, typename T, Boxes KIND>
__device__ __forceinline__ void sc_tile(const SCArgs<S, T>& a, int x0, int y0, int z_begin, SCWarp<T>* sm,
                                        const DirTable<S>& dt) {
    // opaque, or the compiler derives them from special registers again and again
    int warp, wx, y;
    asm volatile("mov.u32 %0, %1;" : "=r"(warp) : "r"((int)threadIdx.x >> 5));
    const int across = a.bx >> 5;                       // 1, 2 or 4 warps along x
    asm volatile("mov.u32 %0, %1;" : "=r"(wx) : "r"((x0 >> 5) + (warp & (across - 1))));
    asm volatile("mov.u32 %0, %1;"
                 : "=r"(y)
                 : "r"(y0 + Pack<T>::ROWS * (across == 1 ? warp : (across == 2 ? warp >> 1 : 0))));
    if (wx < a.words && y < a.g.n[1])
        sc_warp<S, T, KIND>(a, wx, y, z_begin, min(a.g.n[2], z_begin + a.zchunk), sm[warp], dt);
}

// One box: block (x, y) tiles, a chunk of a.zchunk planes from blockIdx.z.
template <typename S, typename T, Boxes KIND>
__global__ void __launch_bounds__(32 * SC_WARPS, sizeof(S) == 8 ? LBM_SC_MIN_BLOCKS_F64 : LBM_SC_MIN_BLOCKS)
    stream_collide_kernel(const __grid_constant__ SCArgs<S, T> a) {
    __shared__ SCWarp<T> sm[SC_WARPS];
    __shared__ DirTable<S> dt;
    load_dirs<S, T>(dt, a);
    __syncthreads();
    sc_tile<S, T, KIND>(a, blockIdx.x * a.bx, blockIdx.y * sc_tile_rows(sizeof(S), a.bx), blockIdx.z * a.zchunk, sm, dt);
}

// Many boxes in one persistent launch: block b takes the work items b,
// b + gridDim.x, ... of the table (instance, x0, y0, z0), copies the
// arguments of the item's instance into shared memory and runs its tile
// (a.zchunk planes from z0). A batch of boxes of one kind has a kernel without
// the other kind's code and its registers.
template <typename S, typename T, Boxes KIND>
__global__ void __launch_bounds__(32 * SC_WARPS, sizeof(S) == 8 ? LBM_SC_MIN_BLOCKS_F64 : LBM_SC_MIN_BLOCKS)
    stream_collide_batch_kernel(const SCArgs<S, T>* __restrict__ args, const int4* __restrict__ items, int n_items) {
    __shared__ SCWarp<T> sm[SC_WARPS];
    __shared__ DirTable<S> dt;
    __shared__ __align__(16) SCArgs<S, T> s_a;
    constexpr int WORDS = (int)(sizeof(SCArgs<S, T>) / 4);
    static_assert(sizeof(SCArgs<S, T>) % 4 == 0, "argument block copied in words");
    for (int it = blockIdx.x; it < n_items; it += gridDim.x) {
        const int4 item = items[it];
        __syncthreads();                 // the previous tile is done with s_a
        const int* src = reinterpret_cast<const int*>(args + item.x);
        int* dst = reinterpret_cast<int*>(&s_a);
        for (int w = threadIdx.x; w < WORDS; w += blockDim.x) dst[w] = src[w];
        __syncthreads();
        load_dirs<S, T>(dt, s_a);
        __syncthreads();
        sc_tile<S, T, KIND>(s_a, item.y, item.z, item.w, sm, dt);
    }
}

// Tile width of a box nx cells wide: 4, 2 or 1 words of 32 cells, the widest
// that leaves at most an eighth of the warps idle at the end of a row
// (neighbouring warps of a block share the sectors their shifted pulls overlap in).
int default_tile_bx(int nx) {
    const int W = (nx + 31) / 32;
    int best = 1;
    for (int b : {2, 4})
        if (8 * ((W + b - 1) / b * b) <= 9 * W) best = b;
    return 32 * best;
}

// Planes a warp marches: as many as leave about 4 blocks of 256 cells per SM,
// beyond 8 only while 8 times as many blocks are left (longer marches commit
// fewer force sums: 256 x 256 x 512 cells 1400 us with 8 planes, 1366 us with
// 16; but 128 x 128 x 256 cells 216 and 226 us, the last wave being emptier).
static int default_zchunk(int nx, int ny, int nz, int sms) {
    const int bx = nx >= 128 ? 128 : (nx + 31) / 32 * 32, by = 256 / bx;
    const long long bxy = (long long)((nx + bx - 1) / bx) * ((ny + by - 1) / by);
    const long long zc = bxy * nz / (4LL * sms);
    if (zc <= 8) return zc < 1 ? 1 : (int)zc;
    return zc / 8 < 8 ? 8 : (zc / 8 > LBM_SC_ZCHUNK ? LBM_SC_ZCHUNK : (int)(zc / 8));
}

template <typename S>
void launch_stream_collide_t(const LbmStepParams& p, cudaStream_t st) {
    using T = typename Store<S>::T;
    SCArgs<S, T> a;
    fill_sc_args<S, T>(p, a);
    const int nx = p.g.n[0];
    a.bx = default_tile_bx(nx);
    while (p.g.n[1] > 65535 * sc_tile_rows(sizeof(S), a.bx)) a.bx /= 2;   // grid limit in y
    const int by = sc_tile_rows(sizeof(S), a.bx);
    a.zchunk = default_zchunk(nx, p.g.n[1], p.g.n[2], p.num_sms > 0 ? p.num_sms : 152);
    dim3 grid((nx + a.bx - 1) / a.bx, (p.g.n[1] + by - 1) / by, (p.g.n[2] + a.zchunk - 1) / a.zchunk);
    if (sc_one(p.storage, p.P.n))
        stream_collide_kernel<S, T, sizeof(T) == 4 ? BOXES_ONE : BOXES_MORE><<<grid, 32 * SC_WARPS, 0, st>>>(a);
    else
        stream_collide_kernel<S, T, BOXES_MORE><<<grid, 32 * SC_WARPS, 0, st>>>(a);
}

// ------------------------------------------------------------ batched launch

template <typename S>
static void fill_batch_args_t(const LbmStepParams& p, int tile_bx, int zchunk, void* out) {
    using T = typename Store<S>::T;
    SCArgs<S, T> a;
    std::memset(&a, 0, sizeof(a));
    fill_sc_args<S, T>(p, a);
    a.bx = tile_bx;
    a.zchunk = zchunk;
    std::memcpy(out, &a, sizeof(a));
}

size_t batch_args_bytes(int storage) {
    switch (storage) {
        case 0: return sizeof(SCArgs<double, double>);
        case 1: return sizeof(SCArgs<float, float>);
        case 2: return sizeof(SCArgs<__half, float>);
        default: return sizeof(SCArgs<__nv_bfloat16, float>);
    }
}

void fill_batch_args(const LbmStepParams& p, int tile_bx, int zchunk, void* out) {
    switch (p.storage) {
        case 0: fill_batch_args_t<double>(p, tile_bx, zchunk, out); break;
        case 1: fill_batch_args_t<float>(p, tile_bx, zchunk, out); break;
        case 2: fill_batch_args_t<__half>(p, tile_bx, zchunk, out); break;
        default: fill_batch_args_t<__nv_bfloat16>(p, tile_bx, zchunk, out); break;
    }
}

template <typename S>
static void launch_batch_t(const void* d_args, const int4* d_items, int n_items, bool one, bool more, int grid,
                           cudaStream_t st) {
    using T = typename Store<S>::T;
    const SCArgs<S, T>* args = static_cast<const SCArgs<S, T>*>(d_args);
    if constexpr (sizeof(T) == 4) {
        if (one) {
            if (more)
                stream_collide_batch_kernel<S, T, BOXES_BOTH><<<grid, 32 * SC_WARPS, 0, st>>>(args, d_items, n_items);
            else
                stream_collide_batch_kernel<S, T, BOXES_ONE><<<grid, 32 * SC_WARPS, 0, st>>>(args, d_items, n_items);
            return;
        }
    }
    stream_collide_batch_kernel<S, T, BOXES_MORE><<<grid, 32 * SC_WARPS, 0, st>>>(args, d_items, n_items);
}

void launch_stream_collide_batch(int storage, const void* d_args, const int4* d_items, int n_items, bool one, bool more,
                                 int grid, cudaStream_t st) {
    switch (storage) {
        case 0: launch_batch_t<double>(d_args, d_items, n_items, one, more, grid, st); break;
        case 1: launch_batch_t<float>(d_args, d_items, n_items, one, more, grid, st); break;
        case 2: launch_batch_t<__half>(d_args, d_items, n_items, one, more, grid, st); break;
        default: launch_batch_t<__nv_bfloat16>(d_args, d_items, n_items, one, more, grid, st); break;
    }
}

void launch_stream_collide(const LbmStepParams& p, cudaStream_t st) {
    switch (p.storage) {
        case 0: launch_stream_collide_t<double>(p, st); break;
        case 1: launch_stream_collide_t<float>(p, st); break;
        case 2: launch_stream_collide_t<__half>(p, st); break;
        default: launch_stream_collide_t<__nv_bfloat16>(p, st); break;
    }
}

}  // namespace lbmdem
