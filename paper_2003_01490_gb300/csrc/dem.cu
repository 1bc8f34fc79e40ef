// dem.cu -- particle side of Algorithm 1: force finalisation and two-step
// averaging of the momentum-exchange force (Sec. 4.2), neighbour search,
// lubrication correction (Eqs. (25)-(33)), linear spring-dashpot contact with
// Coulomb-limited tangential spring (Eqs. (39)-(52)) and the Velocity-Verlet
// subcycles (Eqs. (37)-(38)); the prescribed-motion update. Particle state
// and integration are float64; the pair and wall laws run in float64 for
// float64 PDF storage and in float32 (gaps of pairs from positions held as sums
// of two floats, of walls from float64 positions) for the other formats.
//
// Each particle gathers every interaction of its own with eight lanes, so no
// force atomics are needed; a pair is evaluated by both partners with mirrored
// operands (n_ji = -n_ij, u_ji = -u_ij, ...). Each particle keeps its own copy of
// the tangential spring of every active contact (double buffered per
// subcycle). All subcycles of a step run in one launch: one block for up to 32
// particles, one cluster for up to 512 with float32 laws, a cooperative launch as
// long as its blocks fit the GPU at once.
#include <cstring>

#include "common.cuh"
#include "gang.cuh"
#include "launch.h"
#include "scatter.cuh"

namespace lbmdem {

template <typename T>
struct Vec3 {
    T x, y, z;
};
using V3 = Vec3<double>;
__device__ __forceinline__ V3 mk(double x, double y, double z) { return {x, y, z}; }
template <typename T>
__device__ __forceinline__ Vec3<T> zero3() { return {T(0), T(0), T(0)}; }
template <typename T>
__device__ __forceinline__ Vec3<T> operator+(Vec3<T> a, Vec3<T> b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
template <typename T>
__device__ __forceinline__ Vec3<T> operator-(Vec3<T> a, Vec3<T> b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
template <typename T>
__device__ __forceinline__ Vec3<T> operator-(Vec3<T> a) { return {-a.x, -a.y, -a.z}; }
// Products and multiply-adds of the interaction laws are written out, so that
// every kernel they are compiled into rounds them alike (a batch then ends where
// its instances end alone).
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
template <typename T>
__device__ __forceinline__ Vec3<T> operator*(T s, Vec3<T> a) { return {mul_rn(s, a.x), mul_rn(s, a.y), mul_rn(s, a.z)}; }
template <typename T>
__device__ __forceinline__ T dot(Vec3<T> a, Vec3<T> b) { return mad(a.z, b.z, mad(a.x, b.x, mul_rn(a.y, b.y))); }
template <typename T>
__device__ __forceinline__ Vec3<T> cross(Vec3<T> a, Vec3<T> b) {
    return {mad(a.y, b.z, -mul_rn(a.z, b.y)), mad(a.z, b.x, -mul_rn(a.x, b.z)), mad(a.x, b.y, -mul_rn(a.y, b.x))};
}
__device__ __forceinline__ V3 ld3(const double* p, int i) { return {p[3 * i], p[3 * i + 1], p[3 * i + 2]}; }
__device__ __forceinline__ Vec3<float> ld3(const float* p, int i) { return {p[3 * i], p[3 * i + 1], p[3 * i + 2]}; }
__device__ __forceinline__ void st3(double* p, int i, V3 v) {
    p[3 * i] = v.x;
    p[3 * i + 1] = v.y;
    p[3 * i + 2] = v.z;
}
template <typename T, typename U>
__device__ __forceinline__ Vec3<T> cvt3(Vec3<U> v) { return {(T)v.x, (T)v.y, (T)v.z}; }
__device__ __forceinline__ float tlog(float x) { return logf(x); }
__device__ __forceinline__ double tlog(double x) { return log(x); }
__device__ __forceinline__ float tsqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double tsqrt(double x) { return sqrt(x); }
// the interaction constants in the pair arithmetic's precision
template <typename T>
__device__ __forceinline__ const DemConsts<T>& consts(const DemParams& p);
template <> __device__ __forceinline__ const DemConsts<double>& consts<double>(const DemParams& p) { return p.kd; }
template <> __device__ __forceinline__ const DemConsts<float>& consts<float>(const DemParams& p) { return p.kf; }
__device__ __forceinline__ float mimgf(float d, int n, int per) {
    if (per) {
        const float half = 0.5f * (float)n;
        if (d > half) d -= (float)n;
        if (d < -half) d += (float)n;
    }
    return d;
}
__device__ __forceinline__ double mimg(double d, int n, int per) {
    if (per) {
        double half = 0.5 * (double)n;
        if (d > half) d -= (double)n;
        if (d < -half) d += (double)n;
    }
    return d;
}

// ------------------------------------------------------------ particle view

__device__ __forceinline__ void write_view(const Particles& P, int i) {
    PartView v;
    for (int d = 0; d < 3; ++d) {
        const double x = P.x[3 * i + d];
        const double b = floor(x);
        v.base[d] = (int)b;
        v.frac[d] = (float)(x - b);
        v.u[d] = (float)P.u[3 * i + d];
        v.om[d] = (float)P.om[3 * i + d];
        P.xf[3 * i + d] = (float)x;
    }
    v.R = (float)P.R[i];
    set_view_c(v, P.R[i]);
    P.view[i] = v;
}

// x as a sum of two floats
__device__ __forceinline__ float trailing(double x) { return (float)(x - (double)(float)x); }

// the record of particle i in buffer 0, for the float32 laws
__device__ __forceinline__ void write_record(const Particles& P, int i) {
    DemRec r;
    float* w = reinterpret_cast<float*>(&r);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        w[d] = (float)P.x[3 * i + d];
        w[4 + d] = trailing(P.x[3 * i + d]);
        w[8 + d] = (float)P.u[3 * i + d];
        w[12 + d] = (float)P.om[3 * i + d];
    }
    r.a.w = (float)P.R[i];
    r.b.w = trailing(P.R[i]);
    r.c.w = (float)P.m[i];
    r.d.w = 0.f;
    P.rec[0][i] = r;
}

// rebuild the float view of every particle (after insertion or a velocity
// change): the link arithmetic of Eqs. (14)-(17) reads it
__global__ void view_kernel(const Particles P) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    write_view(P, i);
}

__global__ void read_state_kernel(const Particles P, double* __restrict__ out, const int* __restrict__ status,
                                  int* __restrict__ status_out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x, n3 = 3 * P.n;
    if (k == 0) *status_out = *status;
    if (k >= n3) return;
    out[k] = P.x[k];
    out[n3 + k] = P.u[k];
    out[2 * n3 + k] = P.om[k];
    const int i = k / 3, d = k % 3;
    out[3 * n3 + k] = P.fp[6 * i + d];
    out[4 * n3 + k] = P.fp[6 * i + 3 + d];
}

void launch_read_state(const Particles& P, double* out, const int* status, int* status_out, cudaStream_t st) {
    read_state_kernel<<<(3 * P.n + 127) / 128, 128, 0, st>>>(P, out, status, status_out);
}

__global__ void set_velocity_kernel(const Particles P, int n, const double* __restrict__ vel,
                                    const double* __restrict__ omega, const int* __restrict__ status,
                                    int* __restrict__ status_out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *status_out = *status;
    if (i >= P.n) return;
    for (int d = 0; d < 3 && i < n; ++d) {
        if (vel) P.u[3 * i + d] = vel[3 * i + d];
        if (omega) P.om[3 * i + d] = omega[3 * i + d];
    }
    write_view(P, i);
}

void launch_set_velocity(const Particles& P, int n, const double* vel, const double* omega, const int* status,
                         int* status_out, cudaStream_t st) {
    set_velocity_kernel<<<(P.n + 127) / 128, 128, 0, st>>>(P, n, vel, omega, status, status_out);
}

void launch_view_update(const Particles& P, cudaStream_t st) {
    if (P.n == 0) return;
    view_kernel<<<(P.n + 127) / 128, 128, 0, st>>>(P);
}

// ------------------------------------------------------------ finalisation

// per particle: the step's hydrodynamic force and torque (Eqs. (16)-(17)) from
// the float64 or fixed-point link sums and the exact integer missing-link
// sums, their two-step average (Sec. 4.2), and the accumulators cleared
// (component c of particle i)
__device__ __forceinline__ void finalize_component(const FinalizeParams& p, int i, int c) {
    double v;
    if (p.use_fixed) {
        // constant link parts, exact integers (see boundary.cu):
        // K = 36 sum 2 w c and 36 sum 2 w (n x c); torque adds g x (K / 36)
        // with g = 1/2 - (x - floor(x)) the common fractional cell offset
        // (two components per word: lo + hi 2^32)
        const unsigned long long w = (unsigned long long)p.P.acc_k[3 * i + (c >> 1)];
        const long long lo = (long long)(int)(unsigned)(w & 0xffffffffull);
        const long long k = c & 1 ? (long long)(w - (unsigned long long)lo) >> 32 : lo;
        double exact = __dmul_rn((double)k, 1.0 / 36.0);
        if (c >= 3) {
            const int a = (c - 2) % 3, b = (c - 1) % 3;   // cross product axes
            double kf[2], g[2];
            for (int e = 0; e < 2; ++e) {
                const int d = e == 0 ? a : b;
                const unsigned long long wd = (unsigned long long)p.P.acc_k[3 * i + (d >> 1)];
                const long long lod = (long long)(int)(unsigned)(wd & 0xffffffffull);
                kf[e] = (double)(d & 1 ? (long long)(wd - (unsigned long long)lod) >> 32 : lod) * (1.0 / 36.0);
                const double x = p.P.x[3 * i + d];
                g[e] = 0.5 - (x - floor(x));
            }
            exact += fma(g[0], kf[1], -__dmul_rn(g[1], kf[0]));
        }
        v = fma((double)p.P.acc_i[6 * i + c], 1.0 / FIX_SCALE, exact);
    } else {
        v = p.P.acc_d[6 * i + c];
    }
    const double old = p.first_step ? v : p.P.fp_old[6 * i + c];
    p.P.fp[6 * i + c] = v;
    p.P.fbar[6 * i + c] = p.averaging ? 0.5 * (v + old) : v;
    p.P.fp_old[6 * i + c] = v;
}

// the accumulators cleared (after every component has been read)
__device__ __forceinline__ void finalize_clear(const FinalizeParams& p, int i, int c) {
    if (p.use_fixed) {
        p.P.acc_i[6 * i + c] = 0;
        if (c < 3) p.P.acc_k[3 * i + c] = 0;
    } else {
        p.P.acc_d[6 * i + c] = 0.0;
    }
}

// lane s (0-5) of the particle's eight takes component s
__device__ __forceinline__ void finalize_lane(const FinalizeParams& p, int i, int s) {
    const bool on = i < p.P.n && s < 6;
    if (on) finalize_component(p, i, s);
    __syncwarp();
    if (on) finalize_clear(p, i, s);
}

// eight lanes per particle (a thread per particle issued its six components' float64
// instructions one after the other: with float32 sums 9.3 us, this way 7.4)
__device__ __forceinline__ void finalize_body(const FinalizeParams& p, int bx) {
    const int t = bx * blockDim.x + threadIdx.x;
    finalize_lane(p, t >> 3, t & 7);
}

__global__ void finalize_kernel(const FinalizeParams p) { finalize_body(p, (int)blockIdx.x); }

__global__ void finalize_gang_kernel(const FinalizeParams* __restrict__ table, const int* __restrict__ off, int n) {
    __shared__ __align__(16) FinalizeParams sp;
    const int i = gang_instance(off, n, (int)blockIdx.x);
    gang_load(table, i, sp);
    finalize_body(sp, (int)blockIdx.x - off[i]);
}

void launch_finalize(const FinalizeParams& p, cudaStream_t st) {
    if (p.P.n == 0) return;
    finalize_kernel<<<(8 * p.P.n + 127) / 128, 128, 0, st>>>(p);
}

// ------------------------------------------------------------ neighbour bins

__device__ __forceinline__ int bin_coord(float x, float bs, int nb) {
    int b = (int)(x / bs);
    return b < 0 ? 0 : (b >= nb ? nb - 1 : b);
}

// particles into uniform bins no smaller than the largest interaction reach,
// for the neighbour search of the lubrication and contact pairs (Secs. 3.1, 4.1)
__device__ __forceinline__ void bin_fill_body(const DemParams& p, int bx) {
    const int i = bx * blockDim.x + threadIdx.x;
    if (i >= p.P.n) return;
    int b[3];
    for (int d = 0; d < 3; ++d) b[d] = bin_coord(p.P.xf[3 * i + d], (float)p.binsize[d], p.nbins[d]);
    const long long bi = ((long long)b[2] * p.nbins[1] + b[1]) * p.nbins[0] + b[0];
    if (p.pair_f32) write_record(p.P, i);
    const int slot = atomicAdd(p.P.bin_count + bi, 1);
    if (slot < BIN_CAP) p.P.bin_list[bi * BIN_CAP + slot] = i;
    else atomicOr(p.status, ST_BIN_OVERFLOW);
}

__global__ void bin_fill_kernel(const DemParams p) { bin_fill_body(p, (int)blockIdx.x); }

__global__ void bin_fill_gang_kernel(const DemParams* __restrict__ table, const int* __restrict__ off, int n) {
    __shared__ __align__(16) DemParams sp;
    const int i = gang_instance(off, n, (int)blockIdx.x);
    gang_load(table, i, sp);
    bin_fill_body(sp, (int)blockIdx.x - off[i]);
}

void launch_bins(const DemParams& p, cudaStream_t st) {
    if (p.P.n == 0) return;
    bin_fill_kernel<<<(p.P.n + 127) / 128, 128, 0, st>>>(p);
}

// one warp per particle: lane k tests entry k of each of the 27 bins around it
// (a bin holds at most BIN_CAP = 32 particles); hits are appended in bin order
__device__ __forceinline__ void neighbour_body(const DemParams& p, int bx) {
    static_assert(BIN_CAP == 32, "one lane per bin entry");
    const int i = (bx * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (bx == 0 && threadIdx.x == 0) *p.barrier = 0u;   // for the step's DEM launch
    if (i >= p.P.n) return;   // warp-uniform
    const unsigned FULL = 0xffffffffu;
    const float xi[3] = {p.P.xf[3 * i], p.P.xf[3 * i + 1], p.P.xf[3 * i + 2]};
    const float Ri = (float)p.P.R[i];
    const float extra = (float)(p.cut_max + NBR_SKIN) + 0.01f;
    int b[3], lo[3], hi[3];
    for (int d = 0; d < 3; ++d) {
        b[d] = bin_coord(xi[d], (float)p.binsize[d], p.nbins[d]);
        if (p.nbins[d] < 3) { lo[d] = 0; hi[d] = p.nbins[d] - 1; }
        else if (p.g.per[d]) { lo[d] = b[d] - 1; hi[d] = b[d] + 1; }
        else { lo[d] = b[d] > 0 ? b[d] - 1 : 0; hi[d] = b[d] < p.nbins[d] - 1 ? b[d] + 1 : b[d]; }
    }
    int cnt = 0;
    for (int bz = lo[2]; bz <= hi[2]; ++bz)
        for (int by = lo[1]; by <= hi[1]; ++by)
            for (int bx = lo[0]; bx <= hi[0]; ++bx) {
                const int wx = (p.nbins[0] >= 3) ? wrap_idx(bx, p.nbins[0]) : bx;
                const int wy = (p.nbins[1] >= 3) ? wrap_idx(by, p.nbins[1]) : by;
                const int wz = (p.nbins[2] >= 3) ? wrap_idx(bz, p.nbins[2]) : bz;
                const long long bi = ((long long)wz * p.nbins[1] + wy) * p.nbins[0] + wx;
                const int nb = min(p.P.bin_count[bi], BIN_CAP);
                bool hit = false;
                int j = -1;
                if (lane < nb) {
                    j = p.P.bin_list[bi * BIN_CAP + lane];
                    if (j != i) {
                        float d2 = 0.f;
                        for (int d = 0; d < 3; ++d) {
                            const float dd = mimgf(xi[d] - p.P.xf[3 * j + d], p.g.n[d], p.g.per[d]);
                            d2 += dd * dd;
                        }
                        const float reach = Ri + (float)p.P.R[j] + extra;
                        hit = d2 < reach * reach;
                    }
                }
                const unsigned m = __ballot_sync(FULL, hit);
                if (hit) {
                    const int slot = cnt + __popc(m & ((1u << lane) - 1u));
                    if (slot < NBR_CAP) p.P.nbr[i * NBR_CAP + slot] = j;
                }
                cnt += __popc(m);
            }
    // ascending partner order (a bitonic sort over the warp), so that the
    // subcycles' pair sums (each lane its slots in order, then the lanes in a
    // fixed order) do not depend on the order in which atomics filled the bins
    const int m = cnt < NBR_CAP ? cnt : NBR_CAP;
    __syncwarp();
    int v = lane < m ? p.P.nbr[i * NBR_CAP + lane] : 0x7fffffff;
    for (int k = 2; k <= 32; k <<= 1)
        for (int j2 = k >> 1; j2 > 0; j2 >>= 1) {
            const int o = __shfl_xor_sync(FULL, v, j2);
            v = (((lane & j2) == 0) == ((lane & k) == 0)) ? min(v, o) : max(v, o);
        }
    if (lane < m) p.P.nbr[i * NBR_CAP + lane] = v;
    if (lane == 0) {
        if (cnt > NBR_CAP) {
            atomicOr(p.status, ST_NBR_OVERFLOW);
            cnt = NBR_CAP;
        }
        p.P.nbr_count[i] = cnt;
    }
}

__global__ void neighbour_kernel(const DemParams p) { neighbour_body(p, (int)blockIdx.x); }

__global__ void neighbour_gang_kernel(const DemParams* __restrict__ table, const int* __restrict__ off, int n) {
    __shared__ __align__(16) DemParams sp;
    const int i = gang_instance(off, n, (int)blockIdx.x);
    gang_load(table, i, sp);
    neighbour_body(sp, (int)blockIdx.x - off[i]);
}

void launch_neighbours(const DemParams& p, cudaStream_t st) {
    if (p.P.n == 0) return;
    const long long threads = 32LL * p.P.n;
    neighbour_kernel<<<(int)((threads + 127) / 128), 128, 0, st>>>(p);
}

// ------------------------------------------------------------ Velocity Verlet

__device__ __forceinline__ double wrap_pos(double x, int n, int per) {
    if (per) {
        const double L = (double)n;
        if (x >= L) x -= L;
        if (x < 0.0) x += L;
    }
    return x;
}

__device__ __forceinline__ void position_update(const DemParams& p, int i) {
    // Eq. (37): x += dt u + dt^2 / (2 m) F, every operation rounded as in oct_move
    const double c = __dmul_rn(p.dt, __dmul_rn(p.dt, p.P.hm[i]));
    for (int d = 0; d < 3; ++d) {
        const double x = wrap_pos(fma(c, p.P.F_prev[3 * i + d], fma(p.dt, p.P.u[3 * i + d], p.P.x[3 * i + d])), p.g.n[d],
                                  p.g.per[d]);
        p.P.x[3 * i + d] = x;
        p.P.xf[3 * i + d] = (float)x;
    }
    if (p.pair_f32) write_record(p.P, i);
}

// the first Velocity-Verlet position update of a step (Eq. (37)); later
// subcycles update positions inside the subcycle kernel
__global__ void position_kernel(const DemParams p) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.P.n) return;
    position_update(p, i);
}

void launch_dem_position(const DemParams& p, cudaStream_t st) {
    if (p.P.n == 0) return;
    position_kernel<<<(p.P.n + 127) / 128, 128, 0, st>>>(p);
}

// prescribed motion: every particle moves by its velocity over one time step
// (Eq. (37) with no force and dt = 1), then its view is rebuilt
__global__ void prescribed_move_kernel(const Particles P, const Geom g) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    for (int d = 0; d < 3; ++d) P.x[3 * i + d] = wrap_pos(P.x[3 * i + d] + P.u[3 * i + d], g.n[d], g.per[d]);
    write_view(P, i);
}

void launch_prescribed_move(const Particles& P, const Geom& g, cudaStream_t st) {
    if (P.n == 0) return;
    prescribed_move_kernel<<<(P.n + 127) / 128, 128, 0, st>>>(P, g);
}


// ------------------------------------------------------------ interaction laws

// lubrication force and torque on i due to j, Eqs. (27)-(33)
template <typename T>
__device__ void lubrication_on_i(const DemConsts<T>& k, int tangential, T Ri, T Rj, T delta, Vec3<T> n,
                                 Vec3<T> uij, Vec3<T> omi, Vec3<T> omj, T dmin, Vec3<T>& F, Vec3<T>& Tq) {
    // no term acts outside (0, largest cut-off): a far wall or partner costs nothing
    if (!(delta > T(0) && delta < k.cut_max)) return;
    const T pi = T(3.14159265358979323846);
    const T mu = k.mu_f;
    const T dl = delta > dmin ? delta : dmin;
    const Vec3<T> un = dot(uij, n) * n;
    const Vec3<T> ut = uij - un;
    T c_n, c_ftt, c_ttt, c_ftr, c_ttr;
    Vec3<T> om_ftr, om_ttr;
    if (Rj == Ri) {
        // k = 1: the coefficients below are exact binary fractions or the
        // correctly rounded quotients the general formulas give
        c_n = T(0.25); c_ftt = T(1.0 / 6.0); c_ttt = T(0.125); c_ftr = T(1.0 / 30.0); c_ttr = T(0.2);
        const Vec3<T> oms = omi + omj;
        om_ftr = oms + T(4) * omi + T(4) * omj;
        om_ttr = omi + T(0.25) * omj;
    } else {
        const T kr = Rj / Ri;
        const T k1 = T(1) + kr;
        const T i1 = T(1) / k1;
        const T i2 = i1 * i1;
        c_n = kr * kr * i2;
        c_ftt = T(4) * kr * mad(T(2) * kr, kr, T(2) + kr) * (i2 * i1) * T(1.0 / 15.0);
        c_ttt = kr * (T(4) + kr) * i2 * T(0.1);
        c_ftr = T(2) * kr * kr * i2 * T(1.0 / 15.0);
        c_ttr = T(2) * kr * i1 * T(0.2);
        const Vec3<T> oms = omi + omj;
        om_ftr = oms + (T(4) * Ri / Rj) * omi + (T(4) * kr) * omj;
        om_ttr = omi + (kr * T(0.25)) * omj;
    }
    if (delta > T(0) && delta < k.cut_n)
        F = F + (T(-6) * pi * mu * Ri * Ri * c_n * (T(1) / dl - k.inv_cut_n)) * un;
    const bool tt = tangential && delta > T(0) && delta < k.cut_tt;
    const bool tr = tangential && delta > T(0) && delta < k.cut_tr;
    if (tt || tr) {
        const T lg_tt = tlog(dl * k.inv_cut_tt);
        const T lg_tr = k.cut_tr == k.cut_tt ? lg_tt : tlog(dl * k.inv_cut_tr);
        if (tt) {
            F = F + (T(6) * pi * mu * Ri * c_ftt * lg_tt) * ut;
            Tq = Tq + (T(8) * pi * mu * Ri * Ri * c_ttt * lg_tt) * cross(uij, n);
        }
        if (tr) {
            F = F + (T(-6) * pi * mu * Ri * Ri * c_ftr * lg_tr) * cross(om_ftr, n);
            Tq = Tq + (T(8) * pi * mu * Ri * Ri * Ri * c_ttr * lg_tr) * (om_ttr - dot(om_ttr, n) * n);
        }
    }
}

// normal + Coulomb-limited tangential contact force on i, Eqs. (41)-(50)
template <typename T>
__device__ void contact_force(const DemConsts<T>& k, Vec3<T> n, T delta, Vec3<T> ucp, Vec3<T> uij, T m_eff,
                              T Tc, Vec3<T> dt_old, Vec3<T>& Fn, Vec3<T>& Ft, Vec3<T>& dt_new) {
    const T iT = T(1) / Tc;
    const T kn = m_eff * k.pi2_log_e2 * (iT * iT);
    const T dn = T(-2) * m_eff * k.log_e * iT;
    const T kt = k.kappa * kn, dtg = k.sqrt_kappa * dn;
    const Vec3<T> un = dot(uij, n) * n;
    const Vec3<T> ut = ucp - un;
    Fn = (-kn * delta) * n - dn * un;
    const Vec3<T> proj = dt_old - dot(dt_old, n) * n;
    const T lp = tsqrt(dot(proj, proj));
    const Vec3<T> rot = lp > T(0) ? (tsqrt(dot(dt_old, dt_old)) / lp) * proj : zero3<T>();
    const Vec3<T> Fsd = (-kt) * rot - dtg * ut;
    const T fc = k.mu_p * tsqrt(dot(Fn, Fn));
    const T lsd = tsqrt(dot(Fsd, Fsd));
    if (lsd < fc) {
        Ft = Fsd;
        dt_new = rot + k.dt * ut;
    } else {
        const Vec3<T> t = lsd > T(0) ? (T(1) / lsd) * Fsd : zero3<T>();
        Ft = fc * t;
        dt_new = (T(-1) / kt) * (fc * t + dtg * ut);
    }
}

template <typename T>
__device__ __forceinline__ T collision_time(T diameter, T Tc) {
    return Tc > T(0) ? Tc : T(2.31) * diameter * T(1.7320508075688772);
}

// periodic shift (0 or -+n) that takes the separation of a close pair to its
// minimum image, decided on the float32 copy of the separation
__device__ __forceinline__ int image_shift(float d, int n, int per) {
    if (per) {
        const float half = 0.5f * (float)n;
        if (d > half) return -n;
        if (d < -half) return n;
    }
    return 0;
}

// Loads of particle state that other threads of the launch write between the
// subcycles: CG from L2 (other multiprocessors' writes never reach this one's
// L1), else plain.
template <bool CG, typename U>
__device__ __forceinline__ U ld_state(const U* p) {
    if constexpr (CG) return __ldcg(p);
    else return *p;
}
template <bool CG, typename U>
__device__ __forceinline__ Vec3<U> ld3s(const U* p, int i) {
    return {ld_state<CG>(p + 3 * i), ld_state<CG>(p + 3 * i + 1), ld_state<CG>(p + 3 * i + 2)};
}

// a float64 pair's state
struct PairState {
    V3 xi, xj, ui, uj, omi, omj;
};

template <bool CG>
__device__ __forceinline__ PairState load_pair(const Particles& P, int cur, int i, int j) {
    PairState s;
    s.xi = ld3s<CG>(P.xs[cur], i);
    s.xj = ld3s<CG>(P.xs[cur], j);
    s.ui = ld3s<CG>(P.us[cur], i); s.omi = ld3s<CG>(P.oms[cur], i);
    s.uj = ld3s<CG>(P.us[cur], j); s.omj = ld3s<CG>(P.oms[cur], j);
    return s;
}

template <bool CG>
__device__ __forceinline__ DemRec load_record(const DemRec* r) {
    DemRec v;
    const float4* q = reinterpret_cast<const float4*>(r);
    v.a = ld_state<CG>(q);
    v.b = ld_state<CG>(q + 1);
    v.c = ld_state<CG>(q + 2);
    v.d = ld_state<CG>(q + 3);
    return v;
}

// Force and torque on particle i from its neighbour j (lubrication,
// Eqs. (25)-(33), and contact, Eqs. (39)-(50)) at separation d = x_i - x_j
// (nearest image) of length dist and gap delta; contact = the spring of the
// pair continues, dnew its new value.
template <typename T>
__device__ __forceinline__ void pair_law(const DemParams& p, Vec3<T> d, T dist, T delta, T Ri, T Rj, T mi, T mj,
                                         Vec3<T> ui, Vec3<T> uj, Vec3<T> omi, Vec3<T> omj, int hin, int i, int j,
                                         Vec3<T>& F, Vec3<T>& Tq, bool& contact, Vec3<T>& dnew) {
    const Particles& P = p.P;
    const DemConsts<T>& k = consts<T>(p);
    F = zero3<T>();
    Tq = zero3<T>();
    contact = false;
    dnew = zero3<T>();
    if (delta >= k.cut_max && delta >= T(0)) return;
    const Vec3<T> n = (T(1) / dist) * d;
    const Vec3<T> uij = ui - uj;
    if (p.lubrication) {
        const T Rm = T(0.5) * (Ri + Rj);
        const T dmin = mad(k.min_b, Rm, k.min_a) * Rm;
        lubrication_on_i<T>(k, p.tangential, Ri, Rj, delta, n, uij, omi, omj, dmin, F, Tq);
    }
    if (delta < T(0)) {
        const Vec3<T> ri = T(-0.5) * d, rj = T(0.5) * d;
        const Vec3<T> ucp = (ui + cross(omi, ri)) - (uj + cross(omj, rj));
        const T m_eff = mi * mj / (mi + mj);
        const T Tc = collision_time<T>(Ri + Rj, k.Tc);
        Vec3<T> old = zero3<T>();
        const int nin = P.hist_n[hin][i];
        for (int h = 0; h < nin; ++h)
            if (P.hist_id[hin][i * NBR_CAP + h] == j) {
                const double* sp = P.hist_d[hin] + 3 * (i * NBR_CAP + h);
                old = Vec3<T>{(T)sp[0], (T)sp[1], (T)sp[2]};
                break;
            }
        Vec3<T> Fn, Ft;
        contact_force<T>(k, n, delta, ucp, uij, m_eff, Tc, old, Fn, Ft, dnew);
        F = F + (Fn + Ft);
        Tq = Tq + cross(ri, Ft);
        contact = true;
    }
}

// all in float64
__device__ __forceinline__ void pair_force(const DemParams& p, const PairState& s, int hin, int i, int j, V3& F, V3& Tq,
                                           bool& contact, V3& dnew) {
    const Particles& P = p.P;
    const V3 d = mk(mimg(s.xi.x - s.xj.x, p.g.n[0], p.g.per[0]), mimg(s.xi.y - s.xj.y, p.g.n[1], p.g.per[1]),
                    mimg(s.xi.z - s.xj.z, p.g.n[2], p.g.per[2]));
    const double dist = sqrt(dot(d, d)), Ri = P.R[i], Rj = P.R[j];
    pair_law<double>(p, d, dist, dist - (Ri + Rj), Ri, Rj, P.m[i], P.m[j], s.ui, s.uj, s.omi, s.omj, hin, i, j, F, Tq,
                     contact, dnew);
}

// Sums of two floats: h the leading part, l what it leaves. Every operation is
// rounded on its own, so that h + l is exact where the formulas say so (Knuth's
// two-sum, Dekker's products by a fused multiply-add).
struct Two {
    float h, l;
};
__device__ __forceinline__ Two two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Two two_square(float a) {
    const float p = __fmul_rn(a, a);
    return {p, fmaf(a, a, -p)};
}
// (ah + al) - (bh + bl) + shift
__device__ __forceinline__ Two two_diff(float ah, float al, float bh, float bl, int shift) {
    Two s = two_sum(ah, -bh);
    if (shift) {
        const Two t = two_sum(s.h, (float)shift);
        s.h = t.h;
        s.l = __fadd_rn(s.l, t.l);
    }
    const float l = __fadd_rn(s.l, __fsub_rn(al, bl));
    const float h = __fadd_rn(s.h, l);
    return {h, __fsub_rn(l, __fsub_rn(h, s.h))};
}

// In float32: the separation and e = |d|^2 - (Ri + Rj)^2 as sums of two floats
// (the gap delta = e / (|d| + Ri + Rj) keeps float32 relative accuracy: e is
// known to 2e-11 in boxes of 512 cells, a thousandth of its float32 spacing at
// the smallest gap the lubrication resolves, and to 3e-9 in boxes of 65,535), the
// laws in float32. In float64
// the separation issued 17 instructions of 64 cycles per pair and warp, and the
// partner's state was 18 loads: the DEM of a step took 115 us with 10,000
// particles, 66 us with 1,250 and 61 us with 150, this way 91, 59 and 54 us.
__device__ __forceinline__ void pair_force(const DemParams& p, const DemRec& ri, const DemRec& rj, int hin, int i, int j,
                                           Vec3<float>& F, Vec3<float>& Tq, bool& contact, Vec3<float>& dnew) {
    const Two x = two_diff(ri.a.x, ri.b.x, rj.a.x, rj.b.x, image_shift(ri.a.x - rj.a.x, p.g.n[0], p.g.per[0])),
              y = two_diff(ri.a.y, ri.b.y, rj.a.y, rj.b.y, image_shift(ri.a.y - rj.a.y, p.g.n[1], p.g.per[1])),
              z = two_diff(ri.a.z, ri.b.z, rj.a.z, rj.b.z, image_shift(ri.a.z - rj.a.z, p.g.n[2], p.g.per[2]));
    Two S = two_sum(ri.a.w, rj.a.w);
    S.l = __fadd_rn(S.l, __fadd_rn(ri.b.w, rj.b.w));
    // |d|^2 - S^2: the leading squares exactly, then everything small
    const Two xx = two_square(x.h), yy = two_square(y.h), zz = two_square(z.h), SS = two_square(S.h);
    const Two t1 = two_sum(xx.h, yy.h), t2 = two_sum(t1.h, zz.h), t3 = two_sum(t2.h, -SS.h);
    float low = mad(x.h, x.l, mad(y.h, y.l, mad(z.h, z.l, -mul_rn(S.h, S.l))));
    low = __fadd_rn(__fadd_rn(low, low), __fadd_rn(__fadd_rn(xx.l, yy.l), __fsub_rn(zz.l, SS.l)));
    low = __fadd_rn(low, __fadd_rn(__fadd_rn(t1.l, t2.l), t3.l));
    const float e = __fadd_rn(t3.h, low);
    const Vec3<float> d = {x.h, y.h, z.h};
    const float dist = sqrtf(dot(d, d));
    pair_law<float>(p, d, dist, e / __fadd_rn(dist, S.h), ri.a.w, rj.a.w, ri.c.w, rj.c.w, {ri.c.x, ri.c.y, ri.c.z},
                    {rj.c.x, rj.c.y, rj.c.z}, {ri.d.x, ri.d.y, ri.d.z}, {rj.d.x, rj.d.y, rj.d.z}, hin, i, j, F, Tq,
                    contact, dnew);
}

// ------------------------------------------------------------ subcycles
//
// Eight lanes per particle. Lane s holds neighbour slots s, s + 8, ... and, on
// walled axes, face s (axis s / 2, side s % 2): it evaluates their pair and wall
// laws; the sums of the eight lanes are formed by a butterfly that leaves
// component s of (F, T) in lane s. Lanes 0-2 integrate the translation (Eqs.
// (37)-(38)), lanes 3-5 the rotation, one component each, with the state in
// registers: a float64 instruction occupies a scheduler's float64 unit for 64
// cycles whatever its lanes do, and one lane per particle issued about a hundred
// of them per subcycle where this takes about fifteen.
//
// Float64 pair laws cost some 250 float64 instructions, so there the pairs of
// the block that pass the float32 prefilter are queued and evaluated by full
// warps; float32 ones are evaluated where they are found.
constexpr int DEM_LANES = 8;
constexpr int DEM_THREADS = 128;                     // of a multi-block launch
constexpr int DEM_PPB = DEM_THREADS / DEM_LANES;     // its particles per block
constexpr int ONE_BLOCK_THREADS = DEM_ONE_BLOCK_MAX * DEM_LANES;

template <int PPB>
struct PairQueue {
    int count[(DEM_LANES * PPB + 31) / 32];   // pairs of each warp
    unsigned short entry[PPB * NBR_CAP];   // particle of the block << 5 | slot
    double res[DEM_LANES * PPB][6];
};

// one lane's registers over the subcycles of a step
struct OctLane {
    int i, s;            // particle, lane of its eight
    bool on;             // the particle exists
    int nn;              // its neighbour slots
    int j[NBR_CAP / DEM_LANES];
    float reach2[NBR_CAP / DEM_LANES];
    double x, v, f_prev, f_const;   // position (lanes 0-2), velocity component, force of the last subcycle,
                                    // averaged fluid force + external force
    double coef, dcoef;             // dt / (2 m) or dt / (2 I), dt times it
    float xf, vf, R;                // float32 copies for the tests that decide most cases
    float xl, Rl, m;                // trailing parts of position and radius, the mass, for the float32 laws
    float side;                     // of the box on the lane's axis (lanes 0-2)
    float face;                     // face o.s is in reach where the position (negated for the upper face) is at most
                                    // this, minus infinity without a wall
};

// lane s's share of the particle's record
__device__ __forceinline__ void oct_publish(const DemParams& p, const OctLane& o, int buf) {
    float* r = reinterpret_cast<float*>(p.P.rec[buf] + o.i);
    if (o.s < 3) {
        r[o.s] = o.xf;
        r[4 + o.s] = o.xl;
        r[8 + o.s] = o.vf;
    } else if (o.s < 6) {
        r[9 + o.s] = o.vf;
    } else if (o.s == 6) {
        r[3] = o.R;
        r[7] = o.Rl;
    } else {
        r[11] = o.m;
    }
}

template <bool CG>
__device__ __forceinline__ void oct_load(const DemParams& p, OctLane& o, int i, int s, int cur) {
    const Particles& P = p.P;
    o.i = i;
    o.s = s;
    o.on = i < P.n;
    o.nn = 0;
    o.x = o.v = o.f_prev = o.f_const = o.coef = o.dcoef = 0.0;
    o.xf = o.vf = o.R = o.xl = o.Rl = o.m = o.side = 0.f;
    o.face = -INFINITY;
    if (!o.on) return;
    o.nn = P.nbr_count[i];
    o.R = (float)P.R[i];
    o.Rl = trailing(P.R[i]);
    o.m = (float)P.m[i];
    const float reach = o.R + ((float)p.cut_max + 1e-3f);
    if (s < 3) o.side = (float)p.g.n[s];
    if (s < 6 && !p.g.per[s >> 1]) {
        // the float32 position is within 1e-4 of the float64 one for boxes of up to
        // 2^11 cells; the exact gap decides where the face is in reach
        const float n = (float)p.g.n[s >> 1];
        o.face = reach + 1e-6f * n - (s & 1 ? n : 0.f);
    }
#pragma unroll
    for (int k = 0; k < NBR_CAP / DEM_LANES; ++k) {
        const int slot = s + DEM_LANES * k;
        if (slot < o.nn) {
            o.j[k] = P.nbr[i * NBR_CAP + slot];
            const float r = reach + (float)P.R[o.j[k]];
            o.reach2[k] = r * r;
        }
    }
    if (s < 3) {
        o.x = P.xs[cur][3 * i + s];
        o.v = P.us[cur][3 * i + s];
        o.f_prev = P.F_prev[3 * i + s];
        o.f_const = P.fbar[6 * i + s] + P.ext[3 * i + s];
        o.coef = __dmul_rn(p.dt, P.hm[i]);
    } else if (s < 6) {
        o.v = P.oms[cur][3 * i + s - 3];
        o.f_prev = P.T_prev[3 * i + s - 3];
        o.f_const = P.fbar[6 * i + s];
        o.coef = __dmul_rn(p.dt, P.hI[i]);
    }
    o.dcoef = __dmul_rn(p.dt, o.coef);
    o.xf = (float)o.x;
    o.xl = trailing(o.x);
    o.vf = (float)o.v;
}

// whether the warp (float32 laws) or the block has a neighbour slot
template <typename T>
__device__ __forceinline__ bool oct_pairs(const OctLane& o) {
    if constexpr (sizeof(T) == 4) return __any_sync(0xffffffffu, o.nn > 0);
    else return __syncthreads_or(o.nn > 0);
}

// Eq. (37) for lanes 0-2; the periodic wrap is decided in float64 only for
// positions within half a cell of a face
__device__ __forceinline__ void oct_move(const DemParams& p, OctLane& o) {
    o.x = fma(o.dcoef, o.f_prev, fma(p.dt, o.v, o.x));
    o.xf = (float)o.x;
    if (!(o.xf > 0.5f && o.xf < o.side - 0.5f)) {
        o.x = wrap_pos(o.x, p.g.n[o.s], p.g.per[o.s]);
        o.xf = (float)o.x;
    }
    o.xl = trailing(o.x);
}

// float positions are within 1e-4 of the float64 ones, so a gap above cut_max +
// 1e-3 there is above cut_max exactly
__device__ __forceinline__ bool may_touch(const DemParams& p, Vec3<float> a, Vec3<float> b, float reach2) {
    const float dx = mimgf(a.x - b.x, p.g.n[0], p.g.per[0]), dy = mimgf(a.y - b.y, p.g.n[1], p.g.per[1]),
                dz = mimgf(a.z - b.z, p.g.n[2], p.g.per[2]);
    return dx * dx + dy * dy + dz * dz < reach2;
}

// The tangential spring of the wall contact of face s, in lane s, over the
// subcycles of a launch: components along the two axes that follow the face's
// (the one along the normal is zero), and for float64 the contact's constants
// from the first subcycle that needs them.
template <typename T>
struct WallSpring {
    bool on = false, have = false;
    T b = T(0), c = T(0);
    T kn, dn, kt, dtg, ikt;
};

// whether the particle touches the face: a contact that ends takes its spring with it
template <typename T>
__device__ __forceinline__ void wall_touch(WallSpring<T>& w, bool touch) {
    w.on = touch;
    if (!touch) w.b = w.c = T(0);
}

template <typename T>
__device__ __forceinline__ void wall_load(const DemParams& p, const OctLane& o, WallSpring<T>& w, int hin) {
    const int a = o.s >> 1;
    if (!o.on || o.s >= 6 || p.g.per[a]) return;
    w.on = p.P.wact[hin][6 * o.i + o.s];
    if (w.on) {
        const double* sd = p.P.whist[hin] + 3 * (6 * o.i + o.s);
        w.b = (T)sd[a == 2 ? 0 : a + 1];
        w.c = (T)sd[a == 0 ? 2 : a - 1];
    }
}

template <typename T>
__device__ __forceinline__ void wall_store(const DemParams& p, const OctLane& o, const WallSpring<T>& w, int hout) {
    const int a = o.s >> 1;
    if (!o.on || o.s >= 6 || p.g.per[a]) return;
    p.P.wact[hout][6 * o.i + o.s] = w.on;
    if (w.on) {
        double* sd = p.P.whist[hout] + 3 * (6 * o.i + o.s);
        sd[a] = 0.0;
        sd[a == 2 ? 0 : a + 1] = (double)w.b;
        sd[a == 0 ? 2 : a - 1] = (double)w.c;
    }
}

// a < b of non-negative numbers; float64 ones by their bits, off the float64 unit
__device__ __forceinline__ bool less_pos(float a, float b) { return a < b; }
__device__ __forceinline__ bool less_pos(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b);
}
__device__ __forceinline__ bool negative(float a) { return a < 0.f; }
__device__ __forceinline__ bool negative(double a) { return __double2hiint(a) < 0; }

// Wall law of face s (axis a = s / 2, inward normal n = sg e_a) on the particle:
// lubrication (Eqs. (27)-(33) for a plane) or contact (Eqs. (41)-(50)) with
// everything resolved along a and the two axes b, c that follow it cyclically:
// n x and n . pick components, the spring has none along a and keeps its length
// when turned into the plane, and |Fn| is its one component. A float64
// instruction occupies the unit for 64 cycles; the laws on three-vectors, with
// four square roots and three divisions and the spring in memory between the
// subcycles, took a sphere resting on a wall from 2.0 us per subcycle to 8.9 in
// float64 and 3.9 in float32, this form takes 4.4 and 3.4 (a step of ten
// subcycles in a box of 32x32x64: 138 -> 93 us; float32, 40x40x80: 73 -> 68).
// F, Tq are the components along (a, b, c); returns whether the law acts.
template <typename T>
__device__ bool wall_force(const DemParams& p, const OctLane& o, WallSpring<T>& w, double xa, T ua, T ub, T uc, T omb,
                           T omc, int init, T (&F)[3], T (&Tq)[3]) {
    const Particles& P = p.P;
    const DemConsts<T>& k = consts<T>(p);
    const int a = o.s >> 1, side = o.s & 1;
    const double Rid = P.R[o.i];
    const T delta = (T)(side == 0 ? xa - Rid : ((double)p.g.n[a] - xa) - Rid);
    const bool touch = negative(delta);
    if (!init) wall_touch(w, touch);
    if (!touch && !less_pos(delta, k.cut_max)) return false;
    const T Ri = (T)Rid;
    const T sg = side == 0 ? T(1) : T(-1);
    const double* uw = p.g.wall_vel[side][a];
    ua -= (T)uw[a];
    ub -= (T)uw[a == 2 ? 0 : a + 1];
    uc -= (T)uw[a == 0 ? 2 : a - 1];
    F[0] = F[1] = F[2] = Tq[0] = Tq[1] = Tq[2] = T(0);
    if (!touch) {
        if (!p.lubrication || !(delta > T(0))) return true;
        const T pm = T(3.14159265358979323846) * k.mu_f;
        const T dmin = mad(k.min_b, Ri, k.min_a) * Ri;
        const T dl = less_pos(dmin, delta) ? delta : dmin;
        if (less_pos(delta, k.cut_n)) F[0] = mul_rn(T(-6) * pm * Ri * Ri * (T(1) / dl - k.inv_cut_n), ua);
        const bool tt = p.tangential && less_pos(delta, k.cut_tt);
        const bool tr = p.tangential && less_pos(delta, k.cut_tr);
        if (tt || tr) {
            const T lg_tt = tlog(dl * k.inv_cut_tt);
            const T lg_tr = k.cut_tr == k.cut_tt ? lg_tt : tlog(dl * k.inv_cut_tr);
            const T vb = sg * uc, vc = -sg * ub;      // u x n
            const T ob = sg * omc, oc = -sg * omb;    // omega x n
            if (tt) {
                const T cf = T(6.0 * 8.0 / 15.0) * pm * Ri * lg_tt, ct = T(0.8) * pm * Ri * Ri * lg_tt;
                F[1] = mul_rn(cf, ub); F[2] = mul_rn(cf, uc);
                Tq[1] = mul_rn(ct, vb); Tq[2] = mul_rn(ct, vc);
            }
            if (tr) {
                const T cf = T(-0.8) * pm * Ri * Ri * lg_tr, ct = T(3.2) * pm * Ri * Ri * Ri * lg_tr;
                F[1] = mad(cf, ob, F[1]); F[2] = mad(cf, oc, F[2]);
                Tq[1] = mad(ct, omb, Tq[1]); Tq[2] = mad(ct, omc, Tq[2]);
            }
        }
        return true;
    }
    if (sizeof(T) == 4 || !w.have) {
        const T iT = T(1) / collision_time<T>(T(2) * Ri, k.Tc), mi = (T)P.m[o.i];
        w.kn = mi * k.pi2_log_e2 * (iT * iT);
        w.dn = T(-2) * mi * k.log_e * iT;
        w.kt = k.kappa * w.kn;
        w.dtg = k.sqrt_kappa * w.dn;
        if (sizeof(T) == 8) w.ikt = T(1) / w.kt;
        w.have = true;
    }
    const T r = sg * -mad(T(0.5), delta, Ri);   // contact point on axis a
    const T utb = mad(r, omc, ub), utc = mad(-r, omb, uc);
    F[0] = mad(-w.kn * delta, sg, -mul_rn(w.dn, ua));
    const T sb = mad(-w.kt, w.b, -mul_rn(w.dtg, utb)), sc = mad(-w.kt, w.c, -mul_rn(w.dtg, utc));
    const T fc = k.mu_p * fabs(F[0]);
    const T l2 = mad(sb, sb, mul_rn(sc, sc));
    T nb, nc;
    if (sizeof(T) == 8 ? l2 < fc * fc : tsqrt(l2) < fc) {
        F[1] = sb;
        F[2] = sc;
        nb = mad(k.dt, utb, w.b);
        nc = mad(k.dt, utc, w.c);
    } else {
        const T m = l2 > T(0) ? fc / tsqrt(l2) : T(0);
        F[1] = mul_rn(m, sb);
        F[2] = mul_rn(m, sc);
        const T ik = sizeof(T) == 8 ? w.ikt : T(1) / w.kt;
        nb = -ik * mad(w.dtg, utb, F[1]);
        nc = -ik * mad(w.dtg, utc, F[2]);
    }
    Tq[1] = -mul_rn(r, F[2]);
    Tq[2] = mul_rn(r, F[1]);
    if (!init) {
        w.b = nb;
        w.c = nc;
    }
    return true;
}

// One subcycle of the particle of o (Algorithm 1, inner loop): pair and wall
// laws at the state in buffer cur, the velocities (Eq. (38)) and, unless it is
// the last subcycle, the positions of the next one (Eq. (37)), published in
// buffer 1 - cur, where the particle has neighbours (which then have it as
// theirs). init = 1 evaluates the initial force F(t = 0) only (no state or history
// update). All threads of the block take part; pairs: the block (float32: the
// warp) has a neighbour slot; put_n: hist_n is to be written.
template <typename T, bool CG, int PPB>
__device__ __forceinline__ void oct_subcycle(const DemParams& p, OctLane& o, WallSpring<T>& w, PairQueue<PPB>* queue,
                                             bool pairs, int cur, int hin, int hout, bool put_n, int init, int last) {
    const Particles& P = p.P;
    const unsigned FULL = 0xffffffffu;
    T f[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
    bool acts = false;
    if constexpr (sizeof(T) == 4) {
        if (pairs) {
            // the own record from the particle's lanes
            const int base = (threadIdx.x & 31) & ~(DEM_LANES - 1);
            DemRec me;
            me.a = make_float4(__shfl_sync(FULL, o.xf, base), __shfl_sync(FULL, o.xf, base + 1),
                               __shfl_sync(FULL, o.xf, base + 2), o.R);
            me.b = make_float4(__shfl_sync(FULL, o.xl, base), __shfl_sync(FULL, o.xl, base + 1),
                               __shfl_sync(FULL, o.xl, base + 2), o.Rl);
            me.c = make_float4(__shfl_sync(FULL, o.vf, base), __shfl_sync(FULL, o.vf, base + 1),
                               __shfl_sync(FULL, o.vf, base + 2), o.m);
            me.d = make_float4(__shfl_sync(FULL, o.vf, base + 3), __shfl_sync(FULL, o.vf, base + 4),
                               __shfl_sync(FULL, o.vf, base + 5), 0.f);
#pragma unroll
            for (int k = 0; k < NBR_CAP / DEM_LANES; ++k) {
                const int slot = o.s + DEM_LANES * k;
                if (slot >= o.nn) continue;
                const DemRec you = load_record<CG>(P.rec[cur] + o.j[k]);
                bool contact = false;
                if (may_touch(p, {me.a.x, me.a.y, me.a.z}, {you.a.x, you.a.y, you.a.z}, o.reach2[k])) {
                    Vec3<T> F, Tq, dnew;
                    pair_force(p, me, you, hin, o.i, o.j[k], F, Tq, contact, dnew);
                    f[0] += F.x; f[1] += F.y; f[2] += F.z;
                    f[3] += Tq.x; f[4] += Tq.y; f[5] += Tq.z;
                    acts = true;
                    if (contact && !init) {
                        double* sd = P.hist_d[hout] + 3 * (o.i * NBR_CAP + slot);
                        sd[0] = (double)dnew.x; sd[1] = (double)dnew.y; sd[2] = (double)dnew.z;
                    }
                }
                if (!init) P.hist_id[hout][o.i * NBR_CAP + slot] = contact ? o.j[k] : -1;
            }
        }
    } else if (pairs) {
        // pairs that pass the prefilter into the block's queue, in the order of the
        // threads and their slots, evaluated by full warps; each lane then collects its
        // slots'. The places, and with them the order of every sum, are the same in
        // every run (taken by an atomic counter 1 % faster: 150 particles 132.7 us a
        // step, this way 134.3).
        const int pl = threadIdx.x / DEM_LANES, lane = (int)threadIdx.x & 31, warp = (int)threadIdx.x >> 5;
        const int threads = (int)blockDim.x;
        bool near[NBR_CAP / DEM_LANES];
        int mine = 0;
#pragma unroll
        for (int k = 0; k < NBR_CAP / DEM_LANES; ++k) {
            const int slot = o.s + DEM_LANES * k;
            near[k] = slot < o.nn && may_touch(p, ld3s<CG>(P.xfs[cur], o.i), ld3s<CG>(P.xfs[cur], o.j[k]), o.reach2[k]);
            mine += near[k];
            if (slot < o.nn && !near[k] && !init) P.hist_id[hout][o.i * NBR_CAP + slot] = -1;
        }
        int at = mine;   // inclusive sum over the lanes
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(FULL, at, d);
            if (lane >= d) at += v;
        }
        if (lane == 31) queue->count[warp] = at;
        __syncthreads();
        at -= mine;
        int total = 0;
        for (int w = 0; w < threads / 32; ++w) {
            const int n = queue->count[w];
            at += w < warp ? n : 0;
            total += n;
        }
        int place[NBR_CAP / DEM_LANES];
#pragma unroll
        for (int k = 0; k < NBR_CAP / DEM_LANES; ++k) {
            place[k] = near[k] ? at++ : -1;
            if (near[k]) queue->entry[place[k]] = (unsigned short)((pl << 5) | (o.s + DEM_LANES * k));
        }
        __syncthreads();
        for (int c0 = 0; c0 < total; c0 += threads) {
            const int e = c0 + (int)threadIdx.x;
            if (e < total) {
                const int q = queue->entry[e], slot = q & 31;
                const int i = o.i - pl + (q >> 5), j = P.nbr[i * NBR_CAP + slot];
                Vec3<T> F, Tq, dnew;
                bool contact;
                pair_force(p, load_pair<CG>(P, cur, i, j), hin, i, j, F, Tq, contact, dnew);
                double* r = queue->res[threadIdx.x];
                r[0] = F.x; r[1] = F.y; r[2] = F.z; r[3] = Tq.x; r[4] = Tq.y; r[5] = Tq.z;
                if (!init) {
                    P.hist_id[hout][i * NBR_CAP + slot] = contact ? j : -1;
                    if (contact) {
                        double* sd = P.hist_d[hout] + 3 * (i * NBR_CAP + slot);
                        sd[0] = dnew.x; sd[1] = dnew.y; sd[2] = dnew.z;
                    }
                }
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < NBR_CAP / DEM_LANES; ++k)
                if (place[k] >= c0 && place[k] < c0 + threads) {
                    const double* r = queue->res[place[k] - c0];
#pragma unroll
                    for (int c = 0; c < 6; ++c) f[c] += (T)r[c];
                    acts = true;
                }
            __syncthreads();
        }
    }
    bool face = false;
    if (!(p.g.per[0] && p.g.per[1] && p.g.per[2])) {
        const float xa = __shfl_sync(FULL, o.xf, o.s >> 1, DEM_LANES);
        face = (o.s & 1 ? -xa : xa) <= o.face;
        if (!face && !init) wall_touch(w, false);
    }
    if (__any_sync(FULL, face)) {
        // what face s needs of the particle's position and velocities, from its lanes
        const int base = (threadIdx.x & 31) & ~(DEM_LANES - 1);
        const int a = o.s < 6 ? o.s >> 1 : 0, b = a == 2 ? 0 : a + 1, c = a == 0 ? 2 : a - 1;
        const T v = (T)o.v;
        const double xa = __shfl_sync(FULL, o.x, base + a);
        const T ua = __shfl_sync(FULL, v, base + a), ub = __shfl_sync(FULL, v, base + b),
                uc = __shfl_sync(FULL, v, base + c);
        const T omb = __shfl_sync(FULL, v, base + 3 + b), omc = __shfl_sync(FULL, v, base + 3 + c);
        T F[3], Tq[3];
        if (face && wall_force<T>(p, o, w, xa, ua, ub, uc, omb, omc, init, F, Tq)) {
            f[0] += a == 0 ? F[0] : (a == 1 ? F[2] : F[1]);
            f[1] += a == 0 ? F[1] : (a == 1 ? F[0] : F[2]);
            f[2] += a == 0 ? F[2] : (a == 1 ? F[1] : F[0]);
            f[3] += a == 0 ? Tq[0] : (a == 1 ? Tq[2] : Tq[1]);
            f[4] += a == 0 ? Tq[1] : (a == 1 ? Tq[0] : Tq[2]);
            f[5] += a == 0 ? Tq[2] : (a == 1 ? Tq[1] : Tq[0]);
            acts = true;
        }
    }
    double fs = o.f_const;
    if (__any_sync(FULL, acts)) {
        // component s of the particle's pair and wall sums
        const bool b4 = o.s & 4, b2 = o.s & 2, b1 = o.s & 1;
        T g[4], h[2];
        g[0] = (b4 ? f[4] : f[0]) + __shfl_xor_sync(FULL, b4 ? f[0] : f[4], 4);
        g[1] = (b4 ? f[5] : f[1]) + __shfl_xor_sync(FULL, b4 ? f[1] : f[5], 4);
        g[2] = (b4 ? T(0) : f[2]) + __shfl_xor_sync(FULL, b4 ? f[2] : T(0), 4);
        g[3] = (b4 ? T(0) : f[3]) + __shfl_xor_sync(FULL, b4 ? f[3] : T(0), 4);
        h[0] = (b2 ? g[2] : g[0]) + __shfl_xor_sync(FULL, b2 ? g[0] : g[2], 2);
        h[1] = (b2 ? g[3] : g[1]) + __shfl_xor_sync(FULL, b2 ? g[1] : g[3], 2);
        fs += (double)((b1 ? h[1] : h[0]) + __shfl_xor_sync(FULL, b1 ? h[0] : h[1], 1));
    }
    if (!o.on) return;
    if (init) {
        if (o.s < 3) P.F_prev[3 * o.i + o.s] = fs;
        else if (o.s < 6) P.T_prev[3 * o.i + o.s - 3] = fs;
        return;
    }
    if (put_n && o.s == 6) P.hist_n[hout][o.i] = o.nn;
    // Eq. (38) for u and its rotational analogue for omega
    o.v = fma(o.coef, o.f_prev + fs, o.v);
    o.f_prev = fs;
    o.vf = (float)o.v;
    const int nxt = 1 - cur;
    // the next subcycle's positions; the last subcycle keeps its own
    if (o.s < 3 && !last) oct_move(p, o);
    if constexpr (sizeof(T) == 4) {
        if (!last && o.nn > 0) oct_publish(p, o, nxt);
    } else if (o.nn > 0 && o.s < 3) {
        if (!last) {
            P.xs[nxt][3 * o.i + o.s] = o.x;
            P.xfs[nxt][3 * o.i + o.s] = o.xf;
        }
        P.us[nxt][3 * o.i + o.s] = o.v;
    } else if (o.nn > 0 && o.s < 6) {
        P.oms[nxt][3 * o.i + o.s - 3] = o.v;
    }
}

// The particle's speed stays below 0.5 cells per step (checked per subcycle on
// the squared components of lanes 0-2).
__device__ __forceinline__ void oct_check_speed(const DemParams& p, const OctLane& o) {
    const unsigned FULL = 0xffffffffu;
    // three components below 0.288 are below the limit together
    if (!__any_sync(FULL, o.on && o.s < 3 && !(fabsf(o.vf) < 0.288f))) return;
    const double sq = o.v * o.v;
    const double q1 = __shfl_down_sync(FULL, sq, 1, DEM_LANES), q2 = __shfl_down_sync(FULL, sq, 2, DEM_LANES);
    if (o.on && o.s == 0 && !((sq + q1) + q2 < 0.25)) atomicOr(p.status, ST_FAST_PARTICLE);
}

// the state after the last subcycle into buffer 0 of the particle arrays and
// the float32 view
template <typename T>
__device__ __forceinline__ void oct_store(const DemParams& p, const OctLane& o) {
    const Particles& P = p.P;
    if (!o.on || o.s >= 6) return;
    if (o.s < 3) {
        P.x[3 * o.i + o.s] = o.x;
        P.xf[3 * o.i + o.s] = o.xf;
        P.u[3 * o.i + o.s] = o.v;
        P.F_prev[3 * o.i + o.s] = o.f_prev;
    } else {
        P.om[3 * o.i + o.s - 3] = o.v;
        P.T_prev[3 * o.i + o.s - 3] = o.f_prev;
    }
}
// the view of the particle by its first lane, from the stored state's registers
__device__ __forceinline__ void oct_store_view(const DemParams& p, const OctLane& o) {
    const unsigned FULL = 0xffffffffu;
    const int base = (threadIdx.x & 31) & ~(DEM_LANES - 1);
    const double fl = floor(o.x);
    const int b = (int)fl;
    const float fr = (float)(o.x - fl), v = o.vf;
    PartView w;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        w.base[d] = __shfl_sync(FULL, b, base + d);
        w.frac[d] = __shfl_sync(FULL, fr, base + d);
        w.u[d] = __shfl_sync(FULL, v, base + d);
        w.om[d] = __shfl_sync(FULL, v, base + 3 + d);
    }
    if (o.on && o.s == 0) {
        w.R = (float)p.P.R[o.i];
        set_view_c(w, p.P.R[o.i]);
        p.P.view[o.i] = w;
    }
}

// the first Velocity-Verlet position update of a step (Eq. (37))
template <typename T>
__device__ __forceinline__ void oct_first_position(const DemParams& p, OctLane& o) {
    const Particles& P = p.P;
    if (!o.on) return;
    if (o.s < 3) oct_move(p, o);
    if constexpr (sizeof(T) == 4) {
        oct_publish(p, o, 0);
    } else if (o.s < 3) {
        P.xs[0][3 * o.i + o.s] = o.x;
        P.xfs[0][3 * o.i + o.s] = o.xf;
    }
}

// one DEM subcycle of Algorithm 1 as a launch of its own (the initial force,
// and more particles than fit one cooperative launch)
template <typename T>
__device__ __forceinline__ void subcycle_body(const DemParams& p, int cur, int hin, int hout, int init, int last,
                                              int pblock) {
    __shared__ PairQueue<sizeof(T) == 8 ? DEM_PPB : 1> queue;
    OctLane o;
    oct_load<false>(p, o, pblock * DEM_PPB + (int)threadIdx.x / DEM_LANES, threadIdx.x % DEM_LANES, cur);
    WallSpring<T> w;
    wall_load<T>(p, o, w, hin);
    oct_subcycle<T, false, sizeof(T) == 8 ? DEM_PPB : 1>(p, o, w, &queue, oct_pairs<T>(o), cur, hin, hout, true, init,
                                                        last);
    if (init) return;
    wall_store<T>(p, o, w, hout);
    oct_check_speed(p, o);
    const Particles& P = p.P;
    const int nxt = 1 - cur;
    if (o.on && o.s < 3) {
        P.xs[nxt][3 * o.i + o.s] = o.x;
        P.xfs[nxt][3 * o.i + o.s] = o.xf;
        P.us[nxt][3 * o.i + o.s] = o.v;
        P.F_prev[3 * o.i + o.s] = o.f_prev;
    } else if (o.on && o.s < 6) {
        P.oms[nxt][3 * o.i + o.s - 3] = o.v;
        P.T_prev[3 * o.i + o.s - 3] = o.f_prev;
    }
    if (last) oct_store_view(p, o);
}

template <typename T>
__global__ void __launch_bounds__(DEM_THREADS) subcycle_kernel(const __grid_constant__ DemParams p, int cur, int init,
                                                               int last) {
    subcycle_body<T>(p, cur, p.hin, p.hout, init, last, blockIdx.x);
}

// A barrier of all blocks of a cooperative launch: *count rises by one per block
// and barrier (0 at the launch). Gives up after a second with ST_TIMEOUT.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target, int* status) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(count, 1u);
        unsigned long long t0, t1;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
        unsigned now;
        ok = 1;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(now) : "l"(count) : "memory");
            if (now >= target) break;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
            if (t1 - t0 > 1000000000ull) {
                atomicOr(status, ST_TIMEOUT);
                ok = 0;
                break;
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// A barrier of all threads of a cluster, with the memory order of a release and
// an acquire at cluster scope.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

enum DemSpan { SPAN_BLOCK, SPAN_CLUSTER, SPAN_GRID };

// All subcycles of a step in one launch: the particles' state stays in
// registers, buffers 0 and 1 only carry what partners read. One block, one
// cluster or a cooperative launch, with the barrier of each. With fin, the force
// finalisation of the step comes first, with sc the counters' reset and the
// tile scatter of the mapping last: a step of Algorithm 1 between the dense
// kernel and the mapping is this one launch.
template <typename T, DemSpan SPAN, int PPB>
__device__ __forceinline__ void dem_step_body(const DemParams& p, const FinalizeParams* fin, const MapParams* sc,
                                              PairQueue<PPB>* queue, int hcur, int n_sub, int first_particle) {
    const int s = threadIdx.x % DEM_LANES, i = first_particle + (int)threadIdx.x / DEM_LANES;
    if (fin) {
        finalize_lane(*fin, i, s);
        __syncwarp();
    }
    OctLane o;
    constexpr bool CG = SPAN != SPAN_BLOCK;   // partners' state is written by other multiprocessors
    oct_load<CG>(p, o, i, s, 0);
    WallSpring<T> w;
    wall_load<T>(p, o, w, hcur);
    oct_first_position<T>(p, o);
    const bool pairs = oct_pairs<T>(o);
    unsigned target = 0;
    bool ok = true;
    auto barrier = [&]() {
        if constexpr (SPAN == SPAN_CLUSTER) {
            cluster_barrier();
        } else if constexpr (SPAN == SPAN_GRID) {
            target += gridDim.x;
            ok = grid_barrier(p.barrier, target, p.status);
        } else {
            __syncthreads();
        }
    };
    for (int k = 0; k < n_sub && ok; ++k) {
        barrier();
        if (!ok) break;
        oct_subcycle<T, CG, PPB>(p, o, w, queue, pairs, k & 1, hcur, 1 - hcur, k < 2, 0, k == n_sub - 1);
        oct_check_speed(p, o);
        hcur = 1 - hcur;
    }
    // float64 laws read u, omega of buffer 0 in the last of an odd number of subcycles
    if (sizeof(T) == 8 && (n_sub & 1)) barrier();
    oct_store<T>(p, o);
    wall_store<T>(p, o, w, hcur);
    oct_store_view(p, o);
    if (sc) {
        if (first_particle == 0 && threadIdx.x < 4) reinterpret_cast<int*>(sc->n_solid)[threadIdx.x] = 0;
        tile_scatter_particle<DEM_LANES>(*sc, o.i, o.on, o.x, s);
    }
}

template <typename T>
__global__ void __launch_bounds__(ONE_BLOCK_THREADS)
    dem_step_one_block_kernel(const __grid_constant__ DemParams p, const __grid_constant__ FinalizeParams fin,
                              const __grid_constant__ MapParams sc, int hcur, int n_sub) {
    __shared__ PairQueue<sizeof(T) == 8 ? DEM_ONE_BLOCK_MAX : 1> queue;
    dem_step_body<T, SPAN_BLOCK, sizeof(T) == 8 ? DEM_ONE_BLOCK_MAX : 1>(p, &fin, &sc, &queue, hcur, n_sub, 0);
}

template <typename T>
__global__ void __launch_bounds__(DEM_THREADS, 5)
    dem_step_grid_kernel(const __grid_constant__ DemParams p, const __grid_constant__ FinalizeParams fin,
                         const __grid_constant__ MapParams sc, int hcur, int n_sub) {
    __shared__ PairQueue<sizeof(T) == 8 ? DEM_PPB : 1> queue;
    dem_step_body<T, SPAN_GRID, sizeof(T) == 8 ? DEM_PPB : 1>(p, &fin, &sc, &queue, hcur, n_sub,
                                                            (int)blockIdx.x * DEM_PPB);
}

// Float32 laws, one cluster of CLUSTER_BLOCKS blocks: the cluster's hardware
// barrier takes the place of the counter in memory, which costs a subcycle of few
// particles a fifth of its time. 150 particles 54 -> 45 us per step of ten
// subcycles, 500 particles 65 -> 61 us; with 1,250 the particles crowd 16
// multiprocessors (20 warps each on their float64 units): 59 -> 77 us, so the
// cluster ends at two warps per scheduler.
constexpr int CLUSTER_BLOCKS = 16, CLUSTER_THREADS = 256;   // at most, in steps of a warp
static_assert(DEM_CLUSTER_MAX == CLUSTER_BLOCKS * CLUSTER_THREADS / DEM_LANES, "particles of a cluster");

__global__ void __launch_bounds__(CLUSTER_THREADS)
    dem_step_cluster_kernel(const __grid_constant__ DemParams p, const __grid_constant__ FinalizeParams fin,
                            const __grid_constant__ MapParams sc, int hcur, int n_sub) {
    dem_step_body<float, SPAN_CLUSTER, 1>(p, &fin, &sc, nullptr, hcur, n_sub,
                                          (int)(blockIdx.x * blockDim.x) / DEM_LANES);
}

// The one-block DEM steps of many instances in one launch: block b runs the
// step of entry b of the table (its parameters, history parity and subcycle
// count), exactly as dem_step_one_block_kernel does for one instance.
struct DemBatchEntry {
    DemParams p;
    int hcur, n_sub;
};

template <typename T>
__global__ void __launch_bounds__(ONE_BLOCK_THREADS) dem_step_batch_kernel(const DemBatchEntry* __restrict__ table) {
    __shared__ __align__(16) DemBatchEntry e;
    __shared__ PairQueue<sizeof(T) == 8 ? DEM_ONE_BLOCK_MAX : 1> queue;
    constexpr int WORDS = (int)(sizeof(DemBatchEntry) / 4);
    static_assert(sizeof(DemBatchEntry) % 4 == 0, "entry copied in words");
    const int* src = reinterpret_cast<const int*>(table + blockIdx.x);
    int* dst = reinterpret_cast<int*>(&e);
    for (int w = threadIdx.x; w < WORDS; w += blockDim.x) dst[w] = src[w];
    __syncthreads();
    dem_step_body<T, SPAN_BLOCK, sizeof(T) == 8 ? DEM_ONE_BLOCK_MAX : 1>(e.p, nullptr, nullptr, &queue, e.hcur, e.n_sub,
                                                                       0);
}

size_t dem_batch_entry_bytes() { return sizeof(DemBatchEntry); }

void fill_dem_batch_entry(const DemParams& p, int hcur, int n_sub, void* out) {
    DemBatchEntry e;
    std::memset(&e, 0, sizeof(e));
    e.p = p;
    e.hcur = hcur;
    e.n_sub = n_sub;
    std::memcpy(out, &e, sizeof(e));
}

void launch_dem_step_batch(const void* d_table, int count, int pair_f32, cudaStream_t st) {
    if (count <= 0) return;
    const DemBatchEntry* t = static_cast<const DemBatchEntry*>(d_table);
    if (pair_f32) dem_step_batch_kernel<float><<<count, ONE_BLOCK_THREADS, 0, st>>>(t);
    else dem_step_batch_kernel<double><<<count, ONE_BLOCK_THREADS, 0, st>>>(t);
}

cudaError_t dem_grid_capacity(int storage_f64, int num_sms, int* particles) {
    int blocks = 0;
    const cudaError_t e = storage_f64
        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, dem_step_grid_kernel<double>, DEM_THREADS, 0)
        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, dem_step_grid_kernel<float>, DEM_THREADS, 0);
    *particles = e == cudaSuccess ? blocks * num_sms * DEM_PPB : 0;
    return e;
}

static cudaLaunchConfig_t cluster_config(int threads, cudaLaunchAttribute* attr, cudaStream_t st) {
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = CLUSTER_BLOCKS;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(CLUSTER_BLOCKS);
    c.blockDim = dim3(threads);
    c.stream = st;
    c.attrs = attr;
    c.numAttrs = 1;
    return c;
}

int dem_cluster_capacity() {
    int clusters = 0;
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t c = cluster_config(CLUSTER_THREADS, &attr, nullptr);
    if (cudaFuncSetAttribute(dem_step_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, dem_step_cluster_kernel, &c) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return clusters > 0 ? DEM_CLUSTER_MAX : 0;
}

cudaError_t launch_dem_step(const DemParams& p, const FinalizeParams& fin, const MapParams& sc, int hcur, int n_sub,
                            int cluster_particles, cudaStream_t st) {
    if (p.P.n <= DEM_ONE_BLOCK_MAX) {
        // no idle warps: a block of as many as the particles need
        const int threads = (p.P.n * DEM_LANES + 31) / 32 * 32;
        if (p.pair_f32) dem_step_one_block_kernel<float><<<1, threads, 0, st>>>(p, fin, sc, hcur, n_sub);
        else dem_step_one_block_kernel<double><<<1, threads, 0, st>>>(p, fin, sc, hcur, n_sub);
        return cudaGetLastError();
    }
    if (p.pair_f32 && p.P.n <= cluster_particles) {
        const int warps = (p.P.n * DEM_LANES + 32 * CLUSTER_BLOCKS - 1) / (32 * CLUSTER_BLOCKS);   // per block
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t c = cluster_config(32 * warps, &attr, st);
        return cudaLaunchKernelEx(&c, dem_step_cluster_kernel, p, fin, sc, hcur, n_sub);
    }
    void* args[] = {const_cast<DemParams*>(&p), const_cast<FinalizeParams*>(&fin), const_cast<MapParams*>(&sc), &hcur,
                    &n_sub};
    const void* k = p.pair_f32 ? (const void*)dem_step_grid_kernel<float> : (const void*)dem_step_grid_kernel<double>;
    return cudaLaunchCooperativeKernel(k, dim3((p.P.n + DEM_PPB - 1) / DEM_PPB), dim3(DEM_THREADS), args, 0, st);
}

void launch_dem_subcycle(const DemParams& p, int cur, int init, int last, cudaStream_t st) {
    if (p.P.n == 0) return;
    const int blocks = (p.P.n + DEM_PPB - 1) / DEM_PPB;
    if (p.pair_f32) subcycle_kernel<float><<<blocks, DEM_THREADS, 0, st>>>(p, cur, init, last);
    else subcycle_kernel<double><<<blocks, DEM_THREADS, 0, st>>>(p, cur, init, last);
}

// copy state buffer 1 into buffer 0 (after an odd number of subcycles)
__global__ void state_copy_kernel(const Particles P) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 3 * P.n) return;
    P.xs[0][k] = P.xs[1][k];
    P.us[0][k] = P.us[1][k];
    P.oms[0][k] = P.oms[1][k];
    P.xfs[0][k] = P.xfs[1][k];
}

void launch_state_copy(const Particles& P, cudaStream_t st) {
    if (P.n == 0) return;
    state_copy_kernel<<<(3 * P.n + 255) / 256, 256, 0, st>>>(P);
}

// F^fp and T^fp of each particle ([n][6]) into two blocks [n][3] | [n][3],
// the layout of the host read-out
__global__ void fp_split_kernel(const double* __restrict__ fp, double* __restrict__ out, int n) {
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= 6LL * n) return;
    const long long i = k / 6;
    const int c = (int)(k - 6 * i);
    out[(c < 3 ? 0 : 3LL * n) + 3 * i + (c < 3 ? c : c - 3)] = fp[k];
}

// The multi-block DEM step and prescribed motion of many instances: one
// launch per phase (first position update, each subcycle, the copy back after
// an odd count, the prescribed move), each block running its block of one
// instance's grid with that instance's entry.
template <typename T>
__global__ void __launch_bounds__(128) dem_gang_kernel(const DemGangEntry* __restrict__ table,
                                                       const int* __restrict__ off, int n, int kind) {
    __shared__ __align__(16) DemGangEntry e;
    const int i = gang_instance(off, n, (int)blockIdx.x);
    gang_load(table, i, e);
    const int bx = (int)blockIdx.x - off[i];
    const Particles& P = e.p.P;
    if (kind == DEM_GANG_SUBCYCLE) {
        subcycle_body<T>(e.p, e.cur, e.p.hin, e.p.hout, 0, e.last, bx);
        return;
    }
    const int k = bx * blockDim.x + threadIdx.x;
    if (kind == DEM_GANG_POSITION) {
        if (k < P.n) position_update(e.p, k);
    } else if (kind == DEM_GANG_COPY) {
        if (k < 3 * P.n) {
            P.xs[0][k] = P.xs[1][k];
            P.us[0][k] = P.us[1][k];
            P.oms[0][k] = P.oms[1][k];
            P.xfs[0][k] = P.xfs[1][k];
        }
    } else if (k < P.n) {   // prescribed motion
        for (int d = 0; d < 3; ++d)
            P.x[3 * k + d] = wrap_pos(P.x[3 * k + d] + P.u[3 * k + d], e.p.g.n[d], e.p.g.per[d]);
        write_view(P, k);
    }
}

void launch_dem_gang(int kind, int pair_f32, const void* table, const int* off, int n, int blocks, cudaStream_t st) {
    if (n <= 0 || blocks <= 0) return;
    const DemGangEntry* t = static_cast<const DemGangEntry*>(table);
    if (pair_f32) dem_gang_kernel<float><<<blocks, 128, 0, st>>>(t, off, n, kind);
    else dem_gang_kernel<double><<<blocks, 128, 0, st>>>(t, off, n, kind);
}

// words set to zero, per instance a span (the counters a step starts from)
__global__ void zero_gang_kernel(const ZeroSpan* __restrict__ table, const int* __restrict__ off, int n) {
    const int i = gang_instance(off, n, (int)blockIdx.x);
    const ZeroSpan z = table[i];
    const int bx = (int)blockIdx.x - off[i], gx = off[i + 1] - off[i];
    for (int k = bx * blockDim.x + threadIdx.x; k < z.words; k += gx * blockDim.x) z.p[k] = 0;
}

void launch_gang(int kind, const void* table, const int* off, int n, int blocks, cudaStream_t st) {
    if (n <= 0 || blocks <= 0) return;
    switch (kind) {
        case GANG_FINALIZE:
            finalize_gang_kernel<<<blocks, 128, 0, st>>>(static_cast<const FinalizeParams*>(table), off, n);
            break;
        case GANG_BINS:
            bin_fill_gang_kernel<<<blocks, 128, 0, st>>>(static_cast<const DemParams*>(table), off, n);
            break;
        case GANG_NEIGHBOURS:
            neighbour_gang_kernel<<<blocks, 128, 0, st>>>(static_cast<const DemParams*>(table), off, n);
            break;
        default:
            zero_gang_kernel<<<blocks, 128, 0, st>>>(static_cast<const ZeroSpan*>(table), off, n);
            break;
    }
}

void launch_fp_split(const double* fp, double* out, int n, cudaStream_t st) {
    if (n <= 0) return;
    fp_split_kernel<<<(int)((6LL * n + 255) / 256), 256, 0, st>>>(fp, out, n);
}

}  // namespace lbmdem
