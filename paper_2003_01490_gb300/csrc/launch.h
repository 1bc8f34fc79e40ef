// launch.h -- host-side launchers of the device kernels (internal to the library).
#pragma once

#include <string>

#include "common.cuh"

namespace lbmdem {

struct LbmStepParams {
    int storage;                 // 0 f64, 1 f32, 2 f16, 3 bf16
    const void* src;
    void* dst;
    const uint8_t* flags;
    const uint32_t* solid;           // one bit per cell (x in the bits of a row's words): solid,
    const uint32_t* shell;           // in the TRT+aB shell
    const int* owner;                // particle of a solid cell, -1 for fluid
    Geom g;
    double s_plus, s_minus, s_b_shell, s_b_bulk;
    int bulk_corr;
    double a_user[3];
    double ext_total[3];
    const unsigned long long* n_solid;
    int counterforce;
    Particles P;
    int missing_links;               // the missing-link correction is on
    int other_links;                 // the missing-link list is walked
    int* status;
    const unsigned int* miss_list;   // solid cells with possible missing links
    const int* miss_count;
    int miss_cap;
    int margin;                      // cells from a periodic face within which particle images matter
    int num_sms;                     // multiprocessors of the device (grid sizing)
    double* accel_d;                 // out: fluid body force of the step [3]
    float* accel_f;
};
// BC_ACCEL: the fluid body force of the step; BC_LINKS: the missing links
constexpr int BC_ACCEL = 1, BC_LINKS = 2;
void launch_boundary(const LbmStepParams& p, cudaStream_t st, int mode);
void launch_stream_collide(const LbmStepParams& p, cudaStream_t st);
// rows in y of the dense kernel's tile bx (32, 64 or 128) cells wide: 4 warps
// of 32 x 2 cells (elem: bytes of a stored PDF), 32 x 1 for float64
__host__ __device__ constexpr int sc_tile_rows(int elem, int bx) { return (elem == 8 ? 1 : 2) * 128 / bx; }
// the dense kernel has a form for boxes with one particle (not in float64)
constexpr bool sc_one(int storage, int particles) { return storage != 0 && particles == 1; }
// the dense kernels of many boxes in one persistent launch: per instance one
// argument block (batch_args_bytes(storage) bytes, filled by fill_batch_args)
// in device memory, and a table of work items (instance, x0, y0, z0); one, more:
// there are boxes that sc_one takes, that it does not
size_t batch_args_bytes(int storage);
void fill_batch_args(const LbmStepParams& p, int tile_bx, int zchunk, void* out);
int default_tile_bx(int nx);
void launch_stream_collide_batch(int storage, const void* d_args, const int4* d_items, int n_items, bool one, bool more,
                                 int grid, cudaStream_t st);

struct MapParams {
    Geom g;
    Particles P;
    uint8_t* flags;
    int* owner;
    uint32_t* solid;        // one bit per cell: solid, in the shell (both NULL: a mapping without history)
    uint32_t* shell;
    int ntile[3];
    int* tile_count;
    int* tile_list;
    double shell_width;
    unsigned int* refill_list;
    int* refill_owner;      // former particle of each refill-list cell
    int* refill_count;
    int refill_cap;
    unsigned long long* n_solid;
    unsigned int* miss_list;
    int* miss_count;
    int miss_cap;
    int* status;
};
void launch_tile_scatter(const MapParams& p, cudaStream_t st);
void launch_map(const MapParams& p, cudaStream_t st);
int map_blocks(const int* ntile);   // blocks of a box in a gang launch of the mapping
// the bits per cell from the flags (after a restore)
void launch_cell_bits(const MapParams& p, cudaStream_t st);

struct RefillParams {
    int storage;
    void* f;
    const uint8_t* flags;
    const int* list_owner;  // former particle of each list cell
    Geom g;
    Particles P;
    const unsigned int* list;
    const int* count;
    int cap;
    double cs2_over_s_nu;  // 1 / (3 s_nu)
    const double* accel;   // fluid body force of the step [3]
};
void launch_refill(const RefillParams& p, cudaStream_t st);

struct FieldsParams {
    int storage;
    const void* f;
    const uint8_t* flags;
    Geom g;
    long long first_cell;   // slab of cells [first_cell, first_cell + count)
    long long count;
    const double* accel;
    double* out;            // [4 * count]: rho, ux, uy, uz blocks
};
void launch_fields(const FieldsParams& p, cudaStream_t st);

struct SampleParams {
    int storage;
    const void* f;
    const uint8_t* flags;
    Geom g;
    int n;
    const double* pos;      // [3n] sample points
    double* out;            // [n] density at each point
    const int* status;      // copied to status_out (or status_out NULL)
    int* status_out;
};
void launch_sample_density(const SampleParams& p, cudaStream_t st);

struct FinalizeParams {
    Particles P;
    int use_fixed;          // accumulators in fixed point (float32 path)
    int first_step;
    int averaging;
};
void launch_finalize(const FinalizeParams& p, cudaStream_t st);

// interaction constants of the DEM in the precision of its pair arithmetic
template <typename T>
struct DemConsts {
    T mu_f, cut_n, cut_tt, cut_tr, cut_max, inv_cut_n, inv_cut_tt, inv_cut_tr, min_a, min_b;
    T log_e, pi2_log_e2, kappa, sqrt_kappa, mu_p, Tc, dt;
};

struct DemParams {
    Geom g;
    Particles P;
    int nbins[3];
    double binsize[3];
    double cut_max;         // largest lubrication cut-off
    double e_dry, Tc, nu_p, mu_p;
    double cut_n, cut_tt, cut_tr, min_a, min_b;
    // derived on the host: 1 / cut-offs, log e_dry, pi^2 + (log e_dry)^2,
    // kappa = 2 (1 - nu) / (2 - nu) and its square root
    double inv_cut_n, inv_cut_tt, inv_cut_tr, log_e, pi2_log_e2, kappa, sqrt_kappa;
    double gravity[3];
    double mu_f;            // dynamic fluid viscosity rho0 nu
    int lubrication, tangential;
    double dt;              // subcycle time step 1/n_sub
    int hin, hout;          // history buffers to read and write
    // 1: pair and wall laws in float32 (separations and overlaps from the
    // float64 positions), 0: all in float64
    int pair_f32;
    DemConsts<double> kd;
    DemConsts<float> kf;
    int* status;
    unsigned* barrier;      // arrivals at the barriers of the step's cooperative launch
};
// the one-block DEM steps of many instances in one launch (batches)
size_t dem_batch_entry_bytes();
void fill_dem_batch_entry(const DemParams& p, int hcur, int n_sub, void* out);
void launch_dem_step_batch(const void* d_table, int count, int pair_f32, cudaStream_t st);
void launch_bins(const DemParams& p, cudaStream_t st);
void launch_neighbours(const DemParams& p, cudaStream_t st);
void launch_dem_position(const DemParams& p, cudaStream_t st);
void launch_dem_subcycle(const DemParams& p, int cur, int init, int last, cudaStream_t st);
// The force finalisation, the position update, all subcycles, the counters'
// reset and the tile scatter of a step in one launch: one block for at most
// DEM_ONE_BLOCK_MAX particles, one cluster for at most cluster_particles with
// float32 laws, else a cooperative launch, for at most the particles of
// dem_grid_capacity().
constexpr int DEM_ONE_BLOCK_MAX = 32, DEM_CLUSTER_MAX = 512;
constexpr int DEM_BLOCK_PARTICLES = 16;   // particles per block of a multi-block launch
cudaError_t dem_grid_capacity(int storage_f64, int num_sms, int* particles);
int dem_cluster_capacity();               // DEM_CLUSTER_MAX, or 0 where no such cluster fits the device
cudaError_t launch_dem_step(const DemParams& p, const FinalizeParams& fin, const MapParams& sc, int hcur, int n_sub,
                            int cluster_particles, cudaStream_t st);
void launch_state_copy(const Particles& P, cudaStream_t st);
// state of n particles (positions, velocities, angular velocities, F^fp, T^fp,
// 3n values each) to out and the status to status_out, in page-locked host memory
void launch_read_state(const Particles& P, double* out, const int* status, int* status_out, cudaStream_t st);
// velocities of particles 0 .. n - 1 from page-locked host memory (either NULL:
// kept), the views of all particles, the status to status_out
void launch_set_velocity(const Particles& P, int n, const double* vel, const double* omega, const int* status,
                         int* status_out, cudaStream_t st);
void launch_fp_split(const double* fp, double* out, int n, cudaStream_t st);

// Gang launches (gang.cuh): one launch of a per-step kernel for many
// instances; table holds n parameter blocks in device memory, off the n + 1
// prefix sums of their block counts (blocks = off[n]).
enum { GANG_FINALIZE = 1, GANG_BINS, GANG_NEIGHBOURS, GANG_ZERO, GANG_SCATTER, GANG_MAP, GANG_REFILL };
struct ZeroSpan {
    int* p;        // words set to zero
    int words;
    int pad;
};
void launch_gang(int kind, const void* table, const int* off, int n, int blocks, cudaStream_t st);
void launch_map_gang(int kind, int storage, const void* table, const int* off, int n, int blocks, cudaStream_t st);
// an instance's entry of a DEM gang launch: its parameters (hin, hout for a
// subcycle), the subcycle's state buffer and whether it is the last one
enum { DEM_GANG_POSITION = 1, DEM_GANG_SUBCYCLE, DEM_GANG_COPY, DEM_GANG_PRESCRIBED };
struct DemGangEntry {
    DemParams p;
    int cur, last, pad0, pad1;
};
void launch_dem_gang(int kind, int pair_f32, const void* table, const int* off, int n, int blocks, cudaStream_t st);
size_t bc_args_bytes();
void fill_bc_args(const LbmStepParams& p, void* out);
void launch_boundary_gang(int storage, const void* table, const int* off, int n, int blocks, int mode,
                          cudaStream_t st);
void launch_view_update(const Particles& P, cudaStream_t st);
void launch_prescribed_move(const Particles& P, const Geom& g, cudaStream_t st);

// message returned by lbm_last_error(NULL)
void set_global_error(const std::string& msg);

}  // namespace lbmdem
