// sc_common.cuh -- arithmetic of the dense stream/collide kernel: the CLI
// moving no-slip value of one particle link with its momentum-exchange force
// and torque (Eqs. (14)-(17)), and the TRT(+aB) collision with Guo forcing
// (Eqs. (5), (10)-(12), Sec. 2.3.2). See stream_collide.cu for the data layout.
#pragma once

#include "common.cuh"
#include "launch.h"
#include "links.cuh"

namespace lbmdem {

// Two float32 values in one 64-bit register pair: one packed instruction
// (add, sub, mul, fma .f32x2, each rounded like its scalar form) works on
// both, which halves the instructions of the collision.
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 f2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void split(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.v));
}
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 mad(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

// the cells a thread collides together: V holds ROWS values of type T
template <typename T> struct Pack;
template <> struct Pack<float> {
    using V = F2;
    static constexpr int ROWS = 2;
    __device__ static V all(float a) { return f2(a, a); }
    __device__ static V make(const float (&a)[2]) { return f2(a[0], a[1]); }
    __device__ static void get(V v, float (&a)[2]) { split(v, a[0], a[1]); }
};
template <> struct Pack<double> {
    using V = double;
    static constexpr int ROWS = 1;
    __device__ static V all(double a) { return a; }
    __device__ static V make(const double (&a)[1]) { return a[0]; }
    __device__ static void get(V v, double (&a)[1]) { a[0] = v; }
};

// sign of the first non-zero component of c_q
__host__ __device__ constexpr int lead(int q) { return cx(q) ? cx(q) : (cy(q) ? cy(q) : cz(q)); }

// Weights w2 = 2 w (even parts), w6 = 6 w (odd parts) per class (axis,
// diagonal) and w0. In float32 they are chosen within 1.2e-7 of the exact
// fractions such that w0 + 3 w2_axis + 6 w2_diag = 1 and w6_axis + 4 w6_diag = 1
// hold exactly: the relaxation towards the equilibrium then keeps the mass and
// momentum of every cell, where the plain roundings of 1/18, 1/36 and 1/3 would
// leave a steady source of relative size 3e-8 per step that builds up over a
// long run.
template <typename T>
struct Weights {
    const T w2d = sizeof(T) == 4 ? T(0.0555555522441864) : T(1) / T(18);
    const T w2a = T(2) * w2d;
    const T w0 = T(1) - T(12) * w2d;
    const T w6d = T(1) / T(6);
    const T w6a = T(1) - T(4) * w6d;
};

// What the collision reads of the body force a per pair of directions (q, qbar),
// the same for every cell, once per packed cell: even = 2 lead(q) c_q.a, in
// float64 times (1 - s_plus / 2) w_q already (a multiply-add less per pair), and
// odd = (1 - s_minus / 2) (6 w_q / 2) lead(q) c_q.a.
template <typename T>
struct __align__(16) ForceTerms {
    T even[Pack<T>::ROWS], odd[Pack<T>::ROWS];
};
template <typename T>
__device__ __forceinline__ ForceTerms<T> force_terms(int qi, T ax, T ay, T az, T gp, T gm) {
    const int c0 = (qi & 3) - 1, c1 = ((qi >> 2) & 3) - 1, c2_ = ((qi >> 4) & 3) - 1;
    const int sg = c0 ? c0 : (c1 ? c1 : c2_);
    T ca = T(0);
    if (c0) ca += c0 * sg > 0 ? ax : -ax;
    if (c1) ca += c1 * sg > 0 ? ay : -ay;
    if (c2_) ca += c2_ * sg > 0 ? az : -az;
    const Weights<T> w{};
    const bool axis = c0 * c0 + c1 * c1 + c2_ * c2_ == 1;
    const T g = T(0.5) * gm * (axis ? w.w6a : w.w6d);
    const T e = sizeof(T) == 8 ? T(0.5) * gp * (axis ? w.w2a : w.w2d) : T(1);
    ForceTerms<T> t;
#pragma unroll
    for (int r = 0; r < Pack<T>::ROWS; ++r) {
        t.even[r] = e * (ca + ca);
        t.odd[r] = g * ca;
    }
    return t;
}

template <typename S, typename T>
struct SCArgs {
    // the arrays of each direction: their addresses come from the argument
    // block, so a load costs one 32-bit index and one multiply-add
    const S* src[Q];
    S* dst[Q];
    Geom g;
    // one bit per cell, x in the bits of a row's words (bits past nx are 0)
    const uint32_t* __restrict__ solid;
    const uint32_t* __restrict__ shell;
    int words;                       // 32-bit words per row
    T s_plus, s_minus, s_b_shell, s_b_bulk;
    T gp, gm;                        // weights of the body force, 1 - s_plus / 2 and 1 - s_minus / 2
    T uw[2][3][3];                   // wall velocities [side][axis][component]
    int bulk_corr;
    const T* __restrict__ accel;     // [3]
    int* status;
    int zchunk;                      // z planes per block
    int bx;                          // x extent of a block's tile (32, 64 or 128)
    // particles (for the links)
    int np;
    int margin;                      // cells from a periodic face within which images matter
    const int* __restrict__ owner;   // particle of a solid cell, -1 for fluid
    const double* __restrict__ px;
    const double* __restrict__ pu;
    const double* __restrict__ pom;
    const double* __restrict__ pR;
    const PartView* __restrict__ view;
    double* acc_d;
    long long* acc_i;
};

// kernel arguments from the step parameters
template <typename S, typename T>
void fill_sc_args(const LbmStepParams& p, SCArgs<S, T>& a) {
    for (int q = 0; q < Q; ++q) {
        a.src[q] = static_cast<const S*>(p.src) + q * p.g.ncells;
        a.dst[q] = static_cast<S*>(p.dst) + q * p.g.ncells;
    }
    a.g = p.g;
    a.solid = p.solid;
    a.shell = p.shell;
    a.words = (p.g.n[0] + 31) / 32;
    a.s_plus = (T)p.s_plus;
    a.s_minus = (T)p.s_minus;
    a.s_b_shell = (T)p.s_b_shell;
    a.s_b_bulk = (T)p.s_b_bulk;
    a.gp = T(1) - T(0.5) * a.s_plus;
    a.gm = T(1) - T(0.5) * a.s_minus;
    for (int s = 0; s < 2; ++s)
        for (int ax = 0; ax < 3; ++ax)
            for (int c = 0; c < 3; ++c) a.uw[s][ax][c] = (T)p.g.wall_vel[s][ax][c];
    a.bulk_corr = p.bulk_corr;
    a.accel = reinterpret_cast<const T*>(sizeof(T) == 8 ? (const void*)p.accel_d : (const void*)p.accel_f);
    a.status = p.status;
    a.zchunk = 0;
    a.bx = 128;
    a.np = p.P.n;
    a.margin = p.margin;
    a.owner = p.owner;
    a.px = p.P.x;
    a.pu = p.P.u;
    a.pom = p.P.om;
    a.pR = p.P.R;
    a.view = p.P.view;
    a.acc_d = p.P.acc_d;
    a.acc_i = p.P.acc_i;
}

// per-direction word of the link code: c_q + 1 in bits 0-1, 2-3, 4-5, the
// opposite direction in bits 6-10 (read from shared memory: a warp's lanes
// hold different directions)
__host__ __device__ constexpr int qinfo(int q) { return (cx(q) + 1) | ((cy(q) + 1) << 2) | ((cz(q) + 1) << 4) | (opp(q) << 6); }

// link codes and (-c_q, |c_q|^2) of the directions, in shared memory
template <typename S>
struct DirTable {
    float4 cf[Q];
    const S* src[Q];
    int qi[Q];
    int dq[Q];   // cell index offset of c_q
    ForceTerms<typename Store<S>::T> force[Q];   // of the body force, for the first of each pair of directions
};

// One particle link: cell (x, y, z) pulls direction q (velocity c) from a solid
// cell of particle i. fout = f~_p(x), fin = f~_q(x), fdown = f~_p(x + c_q) (p
// the opposite direction; cli: that cell is fluid and inside the box, else
// bounce-back coefficients). Returns f_q(x, t+1) of Eq. (14) and the link's
// force and torque (Eqs. (15)-(17)).
template <typename S>
__device__ __forceinline__ double link_value(const SCArgs<S, double>& a, int i, const PartView&, int x, int y, int z, int qi, float4,
                                             bool cli, bool, double fout, double fin, double fdown, double (&F)[6]) {
    double r[3], R, u[3], om[3];
    int n[3];
    const int c[3] = {(qi & 3) - 1, ((qi >> 2) & 3) - 1, ((qi >> 4) & 3) - 1};
    PartOps<double>::load(a, i, x, y, z, r, n, R, u, om);
    const double cp0 = -c[0], cp1 = -c[1], cp2 = -c[2];
    const int cc2 = c[0] * c[0] + c[1] * c[1] + c[2] * c[2];
    const double w = cc2 == 1 ? 1.0 / 18.0 : 1.0 / 36.0;
    const double delta = link_root<double>(r, surface_cc<double>(r, R), cp0, cp1, cp2, (double)cc2);
    const double dbc = cli ? delta : 0.5;
    const double inv = 1.0 / (1.0 + 2.0 * dbc);
    const double kappa = (1.0 - 2.0 * dbc) * inv;
    const double rb[3] = {r[0] + delta * cp0, r[1] + delta * cp1, r[2] + delta * cp2};
    const double ub[3] = {u[0] + (om[1] * rb[2] - om[2] * rb[1]), u[1] + (om[2] * rb[0] - om[0] * rb[2]),
                          u[2] + (om[0] * rb[1] - om[1] * rb[0])};
    const double ubc = ub[0] * cp0 + ub[1] * cp1 + ub[2] * cp2;
    const double v = fout + kappa * (fdown - fin) - (12.0 * w * inv) * ubc;
    // Eq. (15) on shifted PDFs: F = c_p (2 w + f~_p + f_q) - u_b (f~_p - f_q)
    const double dif = fout - v, sum = 2.0 * w + fout + v;
    F[0] = cp0 * sum - ub[0] * dif;
    F[1] = cp1 * sum - ub[1] * dif;
    F[2] = cp2 * sum - ub[2] * dif;
    F[3] = rb[1] * F[2] - rb[2] * F[1];
    F[4] = rb[2] * F[0] - rb[0] * F[2];
    F[5] = rb[0] * F[1] - rb[1] * F[0];
    return v;
}

// The same in float32, without the constant part 2 w_p c_p of the force and
// its torque (boundary.cu adds their sum over the particle). wrap: the tile is
// near a periodic face, where the particle's nearest image has to be chosen;
// a link cell lies within R + 2 cells of the centre on every axis and a
// periodic side is longer than 2 R + 4, so exactly one image has
// |n_d| <= floor(n / 2). |n|^2 is a whole number below 2^24, exact in float32.
// The link enters the sphere between t = 0 and 1, so |r + t c|^2 falls from
// above R^2 to at most R^2: r.c < -|c|^2 / 2 and the smaller root is
// cc / (sqrt(disc) - r.c) without cancellation.
template <typename S>
__device__ __forceinline__ float link_value(const SCArgs<S, float>& a, int, const PartView& v, int x, int y, int z, int, float4 cf,
                                            bool cli, bool wrap, float fout, float fin, float fdown, float (&F)[6]) {
    int nd[3] = {x - v.base[0], y - v.base[1], z - v.base[2]};
    if (wrap) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int L = a.g.per[d] ? a.g.n[d] : 0x7fffffff, half = L >> 1;
            if (nd[d] > half) nd[d] -= L;
            if (nd[d] < -half) nd[d] += L;
        }
    }
    const float n0 = (float)nd[0], n1 = (float)nd[1], n2 = (float)nd[2];
    const float g0 = 0.5f - v.frac[0], g1 = 0.5f - v.frac[1], g2 = 0.5f - v.frac[2];
    const float cp0 = cf.x, cp1 = cf.y, cp2 = cf.z;   // c_p
    // |r|^2 - R^2 = (|n|^2 + C) + (2 n.g + C_lo): only the small terms round
    const float nn = fmaf(n2, n2, fmaf(n1, n1, n0 * n0));
    const float ng = fmaf(n2, g2, fmaf(n1, g1, n0 * g0));
    const float cc = (nn + v.C) + fmaf(2.0f, ng, v.C_lo);
    const float r0 = n0 + g0, r1 = n1 + g1, r2 = n2 + g2;
    const float rc = fmaf(r2, cp2, fmaf(r1, cp1, r0 * cp0));
    const float disc = fmaxf(fmaf(rc, rc, -cf.w * cc), 0.0f);
    const float delta = __saturatef(fast_div(cc, fast_sqrt(disc) - rc));
    const float dbc = cli ? delta : 0.5f;
    const float inv = fast_div(1.0f, fmaf(2.0f, dbc, 1.0f));
    const float kappa = fmaf(-2.0f, dbc, 1.0f) * inv;
    const float b0 = fmaf(delta, cp0, r0), b1 = fmaf(delta, cp1, r1), b2 = fmaf(delta, cp2, r2);
    const float u0 = v.u[0] + (v.om[1] * b2 - v.om[2] * b1), u1 = v.u[1] + (v.om[2] * b0 - v.om[0] * b2),
                u2 = v.u[2] + (v.om[0] * b1 - v.om[1] * b0);
    const float ubc = fmaf(u2, cp2, fmaf(u1, cp1, u0 * cp0));
    const float w12 = cf.w == 1.0f ? 12.0f / 18.0f : 12.0f / 36.0f;
    const float val = fmaf(kappa, fdown - fin, fout) - (w12 * inv) * ubc;
    const float dif = fout - val, sum = fout + val;
    F[0] = cp0 * sum - u0 * dif;
    F[1] = cp1 * sum - u1 * dif;
    F[2] = cp2 * sum - u2 * dif;
    F[3] = b1 * F[2] - b2 * F[1];
    F[4] = b2 * F[0] - b0 * F[2];
    F[5] = b0 * F[1] - b1 * F[0];
    return val;
}

// TRT+aB collision of the cells packed in f, in place, with the body force
// a = (ax, ay, az); shell[r]: cell r lies in the shell. Returns the density
// deviations. The arithmetic is that of the moment-space update with S of
// Eq. (12) written per pair of opposite directions (q, qbar): with
// s = f_q + f_qbar and d = f_q - f_qbar the even part relaxes with s_nu and
// the odd part with s_nu^- (Eq. (10)),
//   dp = -s_nu (s/2 - w X) + (1 - s_nu/2) w Y + corr,   X = drho - 3/2 u^2 + 9/2 (c.u)^2
//   dm = -s_nu^- (d/2 - 3 w c.u) + (1 - s_nu^-/2) 3 w c.a, Y = -3 u.a + 9 (c.u)(c.a)
//   f_q += dp + dm,  f_qbar += dp - dm,
// the Guo source in Y and 3 w c.a; corr is the rank-2 bulk correction of the
// shell cells. Each pair costs one chain of fused multiply-adds. The source
// is added at the size of the pair's correction: taken into the equilibrium's
// velocities (u + k a in place of u) a body force some hundred times smaller
// than u is rounded to the last bit of u in every step, which made the float32
// velocities 1.3 to 1.9 times less exact over 50 steps. FORCE = false is the
// form for a = 0 (the same values), which leaves out the sums with a; force: the
// parts of the source that are the same for every cell (force_terms).
template <typename T, bool FORCE>
__device__ __forceinline__ typename Pack<T>::V collide_core(typename Pack<T>::V (&f)[Q],
                                                            const bool (&shell)[Pack<T>::ROWS], T ax, T ay, T az,
                                                            const ForceTerms<T>* force, T sp, T sm, T gp, T s_b_shell,
                                                            T s_b_bulk, int bulk_corr) {
    using P = Pack<T>;
    using V = typename P::V;
    const Weights<T> k_w{};
    // pair sums and differences are formed twice (here and in the update):
    // keeping them takes 36 registers more than the cell's PDFs
    V drho = f[0], jx = P::all(T(0)), jy = jx, jz = jx;
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const int qb = opp(q);
        if (qb < q) continue;
        const int sg = lead(q);
        const V d = sg > 0 ? f[q] - f[qb] : f[qb] - f[q];
        drho = drho + (f[q] + f[qb]);
        if (cx(q)) jx = cx(q) * sg > 0 ? jx + d : jx - d;
        if (cy(q)) jy = cy(q) * sg > 0 ? jy + d : jy - d;
        if (cz(q)) jz = cz(q) * sg > 0 ? jz + d : jz - d;
    }
    const V ux = FORCE ? jx + P::all(T(0.5) * ax) : jx, uy = FORCE ? jy + P::all(T(0.5) * ay) : jy,
            uz = FORCE ? jz + P::all(T(0.5) * az) : jz;
    const V usq = mad(uz, uz, mad(ux, ux, uy * uy));
    V ua = P::all(T(0)), m3ua = ua;
    if constexpr (FORCE) {
        ua = mad(uz, P::all(az), mad(ux, P::all(ax), uy * P::all(ay)));
        m3ua = P::all(T(-3)) * ua;
    }
    // bulk moments m4 = sum (c^2 - 1) f and m5 (row 6 of M) of the streamed
    // PDFs relax with s_b in shell cells (and everywhere when Lambda_b,bulk != 1)
    bool bulk = bulk_corr != 0;
#pragma unroll
    for (int r = 0; r < P::ROWS; ++r) bulk |= shell[r];
    V k4 = P::all(T(0)), k5 = k4;
    if (bulk) {
        T dsr[P::ROWS];
#pragma unroll
        for (int r = 0; r < P::ROWS; ++r) dsr[r] = shell[r] ? s_b_shell - sp : (bulk_corr ? s_b_bulk - sp : T(0));
        const V ds = P::make(dsr);
        V saxis = P::all(T(0)), sdiag = saxis;
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            if (opp(q) < q) continue;
            if (c2(q) == 1) saxis = saxis + (f[q] + f[opp(q)]); else sdiag = sdiag + (f[q] + f[opp(q)]);
        }
        const V m4 = sdiag - f[0];
        const V m5 = mad(P::all(T(-2)), saxis, f[0]) + sdiag;
        // M^-1 e_k = w_q M_kq / (sum_q w_q M_kq^2): norms 2/3 (row 4) and 2 (row 5)
        k4 = P::all(T(1.5)) * (ds * (FORCE ? (usq - m4) - ua : usq - m4));
        k5 = P::all(T(-0.5)) * (ds * m5);
    }
    // equilibrium part common to all directions
    const V drp = mad(P::all(T(-1.5)), usq, drho);
    const V mw2[2] = {P::all(-k_w.w2a), P::all(-k_w.w2d)}, mw6[2] = {P::all(-k_w.w6a), P::all(-k_w.w6d)};
    const V gpw[2] = {P::all(T(0.5) * gp * k_w.w2a), P::all(T(0.5) * gp * k_w.w2d)};
    V corr[2] = {mw2[0] * k5, P::all(T(0.5) * k_w.w2d) * (k4 + k5)};
    if constexpr (FORCE && sizeof(T) == 8) {
        corr[0] = mad(gpw[0], m3ua, corr[0]);
        corr[1] = mad(gpw[1], m3ua, corr[1]);
    }
    V f0 = mad(P::all(sp), mad(P::all(k_w.w0), drp, P::all(T(0)) - f[0]), f[0]);
    if constexpr (FORCE) f0 = mad(P::all(gp), P::all(k_w.w0) * m3ua, f0);
    f[0] = mad(P::all(k_w.w0), k5 - k4, f0);
    const V hsp = P::all(T(-0.5) * sp), hsm = P::all(T(-0.5) * sm), c45 = P::all(T(4.5));
    // each part relaxes as rate x (value - its equilibrium). The pair sums and
    // differences as (exact) multiply-adds, which the compiler does not merge
    // with the first ones
    const V one = P::all(T(1)), mone = P::all(T(-1));
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const int qb = opp(q);
        if (qb < q) continue;
        const int k = c2(q) == 1 ? 0 : 1;
        const int sg = lead(q);
        // c.u times lead(q), which its products with itself, c.a and the odd part share
        V cu = cx(q) ? ux : (cy(q) ? uy : uz);
        if (cx(q) && cy(q)) cu = cy(q) * sg > 0 ? cu + uy : cu - uy;
        if ((cx(q) || cy(q)) && cz(q)) cu = cz(q) * sg > 0 ? cu + uz : cu - uz;
        const V cu45 = c45 * cu;
        const V X = mad(cu45, cu, drp);
        // In float32 the zero is read from memory: the compiler merges a product with the
        // sums that follow (rounded once less than with a body force). Float64 gains
        // the nine instructions (32x32x64 cells 41.5 -> 39.8 us).
        V src = corr[k], odd = P::all(sizeof(T) == 4 ? ax : T(-0.0));
        if constexpr (FORCE) {
            const V even = P::make(force[q].even);
            src = sizeof(T) == 8 ? mad(cu45, even, corr[k]) : mad(gpw[k], mad(cu45, even, m3ua), corr[k]);
            odd = P::make(force[q].odd);
        }
        const V dp = mad(hsp, mad(mw2[k], X, mad(one, f[q], f[qb])), src);
        // lead(q) dm
        const V dm = mad(hsm, mad(mw6[k], cu, sg > 0 ? mad(mone, f[qb], f[q]) : mad(mone, f[q], f[qb])), odd);
        f[q] = f[q] + (sg > 0 ? dp + dm : dp - dm);
        f[qb] = f[qb] + (sg > 0 ? dp - dm : dp + dm);
    }
    return drho;
}

}  // namespace lbmdem
