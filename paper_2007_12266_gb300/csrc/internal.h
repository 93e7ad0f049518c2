// Host-side context and the device view shared by the CUDA translation units.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include <cstdint>
#include <string>
#include <vector>

#include "../../include/lbpm.h"
#include "lattice.cuh"

namespace lbm {

// Where a site's neighbours are. Sites are numbered in x-fastest order, so in
// the x-row through x + (0, dy, dz) the site at the row's middle voxel has the
// rank r of that voxel (the number of pore voxels before it, defined at solids
// too), the one at dx = +1 has r + 1 (r if the middle voxel is solid) and the
// one at dx = -1 has r - 1: eight ranks and one bit per direction give all 18
// neighbour ids. The ranks of the rows next to a known one are stored as 16-bit
// differences, so a site's record is 24 bytes, read with two coalesced vector
// loads.
struct SiteLinks {
    int4 a;             // x: ranks of rows (+y, -y) minus the site's own id (low, high 16 bits);
                        // y, z: ranks of rows +z, -z; w: bit q - 1 set when x + xi_q is a pore
                        // site (q = 1..18), kIrregular when the record does not hold for the site
    int2 b;             // ranks of rows (+z +y, +z -y) minus that of +z; (-z +y, -z -y) minus that of -z
};
// Sites next to a periodic x face (where the next voxel of the row is at its
// other end), and those whose differences exceed 16 bits: their neighbours are
// looked up in the dense grid of site ids.
constexpr int kIrregular = static_cast<int>(0x80000000u);

// Everything a step kernel needs, passed by value as a kernel parameter.
// Grids are "padded": (nx+2)(ny+2)(nz+2) voxels, one halo layer per face, so
// neighbour voxel = v + off[q] never leaves the allocation. The halo of a
// periodic axis mirrors the opposite face; on a non-periodic axis it is wall.
struct DomainView {
    int n_sites;        // N: pore sites
    int pitch;          // P: row length of the per-site arrays, N rounded up (see kPitch)
    int px, pxpy;       // padded-grid strides in y and z: xi_q is at offset cx + cy px + cz pxpy
    const int* site_vox;   // [N] padded voxel of each site
    const int* vsite;      // [Vp] site id; negative for solid (the complement of its rank) and wall (-1)
    const int4* link_a;    // [N] SiteLinks::a
    const int2* link_b;    // [N] SiteLinks::b
    float* phi[2];         // [N] phase of each site by step parity: the phase pass of a step of parity P
                           //     writes phi[P] and the collision reads it; with fp16 storage the
                           //     previous step's phi[P ^ 1] is the reference of the stored
                           //     components (with fp32 storage both point to one array)
    unsigned phis_at[2];   // where the grid of phi_s (phi_s of solid voxels, 0 at pores and walls) lies
                           //     relative to phi[P], in entries modulo 2^32: behind phi[1] with fp16
                           //     storage, otherwise before
    float* nsum;           // [N] Na + Nb of the current step (phase pass -> collision)
    float* rsum;           // [N] fp16 store: sum_q w_q phi_w(q) of the component references that the
                           //     next phase pass reads (collision -> phase pass, see StoreF16)
    float* drho;           // [N] rho - 1 of each site at the last even step, fp16 store: the
                           //     reference of the stored momentum deviations
    void* f;               // [19][P] momentum distributions (AA in place)
    void* a;               // [7][P]  component A
    void* b;               // [7][P]  component B
    unsigned long long* acc;     // [N] sum form: packed fixed-point (Na, Nb) of each site (see pack_sums)
    float tau_a, tau_b, alpha, beta;
    float fx, fy, fz;
    float fterm[9];        // 3 t_q xi_q . F of the odd directions q = 2k + 1 (forcing term per pair), in
                           // the collision's working units (times 2^14 with fp16 storage)
    float s_nu, s_m;       // rates when tau_a == tau_b
    int uniform_tau;
};

// offset of x + xi_q from x in the view's padded grids
__host__ __device__ __forceinline__ int stencil_off(const DomainView& d, int q) {
    return stencil_offset(q, d.px, d.pxpy);
}

// Per-site arrays are allocated for N rounded up to a multiple of kPitch
// entries, which is also the distance between the rows of f, a and b: every row
// then starts on a 128-byte (fp32; 64-byte, fp16) boundary, so that a warp's
// accesses to a row at an even step touch no extra sector, and two neighbouring
// sites can be accessed at once.
constexpr long long kPitch = 32;
inline long long pitch_of(long long n) { return (n + kPitch - 1) / kPitch * kPitch; }

struct Allocation {
    void* ptr;
    size_t bytes;
};

}  // namespace lbm

struct lbpm_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    std::string err;
    // allocator
    lbpm_alloc_fn alloc = nullptr;
    lbpm_free_fn free_fn = nullptr;
    void* alloc_user = nullptr;
    std::vector<lbm::Allocation> allocs;
    // image
    int nx = 0, ny = 0, nz = 0;
    int px = 0, py = 0, pz = 0;
    long long V = 0, Vp = 0;
    long long N = 0;
    bool have_image = false, have_fluids = false, unstable = false;
    uint16_t* d_labels = nullptr;   // [V]
    int* d_site_vox = nullptr;      // [N]
    int* d_vsite = nullptr;         // [Vp]
    float* d_phases = nullptr;      // one block: d_phi_alt (fp16 storage), d_phis, d_phi
    float* d_phis = nullptr;        // [Vp] phi_s of solid voxels, 0 at pores and walls
    int4* d_link_a = nullptr;       // [N] SiteLinks
    int2* d_link_b = nullptr;       // [N]
    float* d_phi = nullptr;         // [N] phase of each site
    float* d_phi_alt = nullptr;     // [N] fp16 storage: the phase at odd steps
    float* d_nsum = nullptr;        // [N]
    float* d_rsum = nullptr;        // [N] fp16 storage
    double* d_face_part = nullptr;          // flux inlet: per-block sums (2 * kFaceBlocks)
    float* d_face_rho = nullptr;            // flux inlet: (rho, rho - 1) of the inlet face, block counter (kFaceWords)
    float* d_drho = nullptr;                // [N] fp16 store
    void* d_f = nullptr;
    void* d_a = nullptr;
    void* d_b = nullptr;
    unsigned long long* d_acc = nullptr;   // [N] sum form: packed component sums
    int step_form = LBPM_STEP_AUTO;        // lbpm_set_step_form
    int* d_slab_site = nullptr;     // reservoir sites
    signed char* d_slab_side = nullptr;
    long long n_slab = 0;
    double* d_partials = nullptr;   // measure partial sums
    long long n_partials = 0;
    // parameters and state
    lbpm_params params{};
    long long step = 0;
    long long launches = 0;
    int block = 256;
    // captured step bundles: graphs[0] = 2 timesteps, graphs[1] = 16 timesteps (population form);
    // sum_graphs[0] / [1]: 2 / 16 middle timesteps of the sum form
    cudaStream_t cap_stream = nullptr;
    cudaGraphExec_t graphs[2] = {nullptr, nullptr};
    cudaGraphExec_t sum_graphs[2] = {nullptr, nullptr};
    bool use_graphs = true;
    // kernel timing
    bool timing = false;
    std::vector<cudaEvent_t> ev_pool;
    std::vector<std::pair<int, int>> ev_collide, ev_phase;  // (start, end) indices
    size_t ev_next = 0;
};

namespace lbm {

// device memory through the ctx's allocator
void* dalloc(lbpm_ctx* c, size_t bytes);
void dfree(lbpm_ctx* c, void* p);

// Enqueue the copy of `bytes` device bytes to the caller's host buffer on `s`
// (host_copy.cu; the caller synchronizes the stream).
cudaError_t copy_to_host(void* dst, const void* src, size_t bytes, cudaStream_t s);

// launchers (return cudaError_t of the launch)
cudaError_t launch_flag_pore(const uint16_t* labels, long long V, int* flags, cudaStream_t s);
cudaError_t exclusive_scan(lbpm_ctx* c, const int* in, int* out, long long n);
cudaError_t launch_scatter_sites(const lbpm_ctx* c, const int* scan, cudaStream_t s);
cudaError_t launch_fill_halo(const lbpm_ctx* c, cudaStream_t s);
cudaError_t launch_affinity_table(const lbpm_ctx* c, const float* table, int n_labels, cudaStream_t s);
cudaError_t launch_affinity_map(const lbpm_ctx* c, const float* map, cudaStream_t s);
cudaError_t launch_slab_flags(const lbpm_ctx* c, int* flags, cudaStream_t s);
cudaError_t launch_slab_scatter(const lbpm_ctx* c, const int* flags, const int* scan, cudaStream_t s);
cudaError_t launch_export_index(const lbpm_ctx* c, long long* site2vox, int* nbr, cudaStream_t s);
cudaError_t launch_links(const lbpm_ctx* c, cudaStream_t s);

// Look up (once per device, with that device current) the device address of
// the static staging array of lbpm_read_field_noalloc; called by lbpm_create.
cudaError_t noalloc_setup(int device);

DomainView make_view(const lbpm_ctx* c);
cudaError_t launch_init_fluids(const lbpm_ctx* c, const float* phi0, cudaStream_t s);
cudaError_t launch_ref_sum(const lbpm_ctx* c, int parity, cudaStream_t s);
// Phase pass from the populations (sums: also set the component sums, for a
// collision of the sum form next) and the collision storing populations.
cudaError_t launch_phase(const lbpm_ctx* c, int parity, bool sums, cudaStream_t s);
cudaError_t launch_collide(const lbpm_ctx* c, int parity, cudaStream_t s);
// Sum form of a timestep (components carried as per-site sums, see pack_sums):
// phase pass from the sums, and the collision moving its recolored values
// between the sums.
cudaError_t launch_phase_sum(const lbpm_ctx* c, int parity, cudaStream_t s);
cudaError_t launch_collide_sum(const lbpm_ctx* c, int parity, cudaStream_t s);
// Whether a context can run the sum form (no pressure or flux faces, the
// population form not forced).
bool sum_form_capable(const lbpm_ctx* c);
// Reservoir slabs or faces after a collision, for the next step (parity `parity`):
// the reset state (slabs; sums: the components' into the sums) or what enters
// (faces, population form only).
cudaError_t launch_reservoir(const lbpm_ctx* c, int parity, bool sums, cudaStream_t s);
// flux inlet: blocks of the fixed-order face reduction
constexpr int kFaceBlocks = 64;
constexpr int kFaceWords = 4;   // (rho, rho - 1) of the inlet and the counter of finished blocks
cudaError_t launch_morph(const lbpm_ctx* c, int parity, float delta, int R, int apply, float* phi_grid,
                         float* dist_grid, float* ntot, int3* off, long long* off_lin, float* off_len, int n_off,
                         unsigned long long* counts, cudaStream_t s);

constexpr int NSUM = 27;  // per-site sums reduced by the measure kernel
void fill_measures(const lbpm_ctx* c, const double* S, lbpm_measures* out);

// One tile of a batched launch: `first` is the first site of job `job` that the
// block handles.
struct BatchTile {
    int job;
    int first;
};
// Job table of one batched step launch, passed by value in the kernel's
// parameter space (at most kBatchLaunchJobs jobs per launch; larger batches
// take several launches per kernel). Tiles of bt threads are numbered job by
// job: job j owns tiles [tile_begin[j], tile_begin[j + 1]). Every thread of a
// block finds its job from blockIdx alone, so the job index and the view's
// fields are warp-uniform values read from the constant bank.
constexpr int kBatchLaunchJobs = 128;
struct BatchLaunch {
    int n_jobs;
    int tile_begin[kBatchLaunchJobs + 1];
    DomainView v[kBatchLaunchJobs];
};
// form: phase pass 0 = populations, 1 = sums, 2 = populations setting the sums;
// collision 0 = populations, 1 = sums.
cudaError_t launch_batch(int kernel, int form, int par, bool fp16, int bt, unsigned grid, cudaStream_t s,
                         const BatchLaunch& p);
cudaError_t launch_batch_measure(bool fp16, unsigned grid, cudaStream_t s, const DomainView* v, const int* parity,
                                 const BatchTile* t, int nt, double* partials, const int* tile_begin, int n_jobs,
                                 double* out);
int batch_max_blocks(int kernel, bool fp16, int bt);
// nsteps (>= 2) timesteps of one job of a batch in the sum form, enqueued on s
// instead of the context's own stream; adds the kernels launched to *launches.
lbpm_status advance_job(lbpm_ctx* c, long long nsteps, cudaStream_t s, long long* launches);
// Capture the graphs that such a run uses, without advancing the job.
lbpm_status capture_job(lbpm_ctx* c, long long nsteps);
cudaError_t launch_measure(lbpm_ctx* c, int parity, const double** out, cudaStream_t s);
cudaError_t launch_field(const lbpm_ctx* c, int parity, int which, float* dense, cudaStream_t s);
cudaError_t launch_export_dist(const lbpm_ctx* c, int parity, int which, float* out, cudaStream_t s);
cudaError_t launch_read_box(const lbpm_ctx* c, int parity, int which, const int* lo, const int* hi, float* out,
                            cudaStream_t s);
cudaError_t launch_import_dist(const lbpm_ctx* c, int parity, int which, const float* in, cudaStream_t s);

}  // namespace lbm
