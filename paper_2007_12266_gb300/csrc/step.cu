// Single-domain launchers of the timestep kernels (Sec. 3.1) and fluid
// initialisation.
#include "step_kernels.cuh"

namespace lbm {

namespace {

constexpr int kBlock = 256;

// Launch with programmatic stream serialization (see wait_prior_grid()).
template <class... KArgs, class... Args>
cudaError_t launch_pdl_bt(void (*kernel)(KArgs...), unsigned grid, unsigned block, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), unsigned grid, cudaStream_t s, Args... args) {
    return launch_pdl_bt(kernel, grid, kBlock, s, args...);
}

template <int PAR, class S, bool SUMS>
__global__ void __launch_bounds__(kBlock) k_phase(DomainView d) {
    const int t = blockIdx.x * kBlock + threadIdx.x;
    phase_thread<PAR, S, SUMS>(d, t);
}

constexpr int kPhaseSumPer = 2;   // sites per thread of the sum-form phase pass (1, 2, 4, 8 measured; 2 fastest)

template <int PAR>
__global__ void __launch_bounds__(kBlock) k_phase_sum(DomainView d) {
    phase_sum_thread<PAR, kPhaseSumPer>(d, blockIdx.x * kBlock * kPhaseSumPer + threadIdx.x, kBlock);
}

// Launch shape of the collision: 64 registers and 32 resident warps per SM; 56
// registers and 36 warps spill at odd steps, and gain nothing at even ones, where they
// do not. Blocks of 128 threads in FP16, and in FP32 below kSmallSites: there a launch
// is a few waves out of L2, which smaller blocks end more evenly (256 / 128 threads, us
// per step: 3.78 / 3.36 at 7 k sites, 10.8 / 10.3 at 247 k, 24.7 / 24.5 at 657 k, 38.7 /
// 38.9 at 901 k). Above it the step runs from DRAM and 256 threads are as fast or
// faster (53.1 / 53.3 at 1.2 M, 66.8 / 67.8 at 1.6 M, 102 / 104 at 2.5 M).
constexpr long long kSmallSites = 1LL << 20;

// CF: component form of the collision (see collide_site)
template <int PAR, class S, int CF, int BT>
__global__ void __launch_bounds__(BT, 1024 / BT) k_collide(DomainView d) {
    // odd steps: slot (and fp16 reference) cache, see SlotCache; even steps of
    // the sum form: the six face neighbours
    constexpr int kSlots = PAR == 1 ? (Q19 - 1) * BT : (CF != 0 ? (Q7 - 1) * BT : 1);
    constexpr int kRefs = PAR == 1 && S::kRef ? (Q19 - 1) * BT : 1;
    __shared__ int slot[kSlots];
    __shared__ float ref[kRefs];
    const int n = blockIdx.x * BT + threadIdx.x;
    if (n < d.n_sites) collide_thread<PAR, S, CF>(d, n, SlotCache{slot + threadIdx.x, ref + threadIdx.x, BT});
}

// The boundary kernels run after the collision with programmatic launch: the
// next phase pass, which waits for them, must not start before the collision has
// completed, so every thread waits first.
template <int PAR, class S>
__global__ void __launch_bounds__(kBlock) k_pressure_faces(DomainView d, const int* sites,
                                                           const signed char* side, int n_face,
                                                           float rho_in, float rho_out, float drho_in,
                                                           float drho_out, const float* face) {
    wait_prior_grid();
    allow_next_grid();
    const int i = blockIdx.x * kBlock + threadIdx.x;
    if (i < n_face) pressure_face_thread<PAR, S>(d, sites[i], side[i], rho_in, rho_out, drho_in, drho_out, face);
}

__device__ __forceinline__ double warp_total(double v) {
    #pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Flux inlet: per-block sums (fixed grid, fixed order: the result does not
// depend on scheduling) of D_s over the inlet sites and their count; the block
// that finishes last adds them up, again in a fixed order, and sets the inlet's
// density,
//   rho_in - 1 = (sum D + Q) / (n_in - Q), from sum_s (1 + D_s) / (n_in - Q).
// A few thousand sites: latency is all of it, so the sums are warp trees (one
// thread's 64 dependent fp64 additions took longer than the rest).
template <int PAR, class S>
__global__ void __launch_bounds__(kBlock) k_face_rho(DomainView d, const int* sites, const signed char* side,
                                                     int n_face, double* part, double flux, float* face) {
    constexpr int kWarps = kBlock / 32;
    __shared__ double sd[kWarps];
    __shared__ int sc[kWarps];
    __shared__ bool last;
    static_assert(kFaceBlocks == 64 && kWarps >= 1, "the last block's first warp adds two partial sums per lane");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    wait_prior_grid();
    allow_next_grid();
    double acc = 0.0;
    int cnt = 0;
    for (int i = blockIdx.x * kBlock + threadIdx.x; i < n_face; i += kFaceBlocks * kBlock) {
        if (side[i] != 1) continue;
        int nb[Q19];
        float dv[Q19], nx, ny;
        acc += face_deviations<PAR, S>(d, sites[i], 1.0f, nb, dv, nx, ny);
        ++cnt;
    }
    acc = warp_total(acc);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) {
        sd[warp] = acc;
        sc[warp] = cnt;
    }
    __syncthreads();
    unsigned* const finished = reinterpret_cast<unsigned*>(face + 2);
    if (threadIdx.x == 0) {
        double D = 0.0;
        int n = 0;
        for (int w = 0; w < kWarps; ++w) {
            D += sd[w];
            n += sc[w];
        }
        part[2 * blockIdx.x] = D;
        part[2 * blockIdx.x + 1] = static_cast<double>(n);
        __threadfence();
        last = atomicAdd(finished, 1u) + 1u == kFaceBlocks;
    }
    __syncthreads();
    if (!last || warp != 0) return;
    __threadfence();
    const volatile double* const p = part;
    const double D = warp_total(p[2 * lane] + p[2 * (lane + 32)]);
    const double n = warp_total(p[2 * lane + 1] + p[2 * (lane + 32) + 1]);
    if (lane != 0) return;
    const double drho = n > flux ? (D + flux) / (n - flux) : 0.0;
    face[0] = static_cast<float>(1.0 + drho);
    face[1] = static_cast<float>(drho);
    *finished = 0u;                        // for the next launch
}

template <int PAR, class S, bool SUMS>
__global__ void __launch_bounds__(kBlock) k_reservoir(DomainView d, const int* sites,
                                                      const signed char* side, int n_slab,
                                                      float rho_in, float rho_out) {
    wait_prior_grid();
    allow_next_grid();
    const int i = blockIdx.x * kBlock + threadIdx.x;
    if (i < n_slab) reservoir_thread<PAR, S, SUMS>(d, sites[i], side[i], rho_in, rho_out);
}

__device__ __forceinline__ float phi0_of_site(const DomainView& d, int n, const float* phi0, int nx, int ny,
                                              int px, int pxpy) {
    const int v = d.site_vox[n];
    const int z = v / pxpy - 1;
    const int r = v - (z + 1) * pxpy;
    const int y = r / px - 1;
    const int x = r - (y + 1) * px - 1;
    const float p = phi0[static_cast<size_t>(x) + static_cast<size_t>(nx) * (y + static_cast<size_t>(ny) * z)];
    return fminf(1.0f, fmaxf(-1.0f, p));
}

// The phases that step 0 reads as the previous step's: phi0 (fp16
// storage: the references of the initial component values).
__global__ void __launch_bounds__(kBlock) k_init_phase(DomainView d, const float* phi0, int nx, int ny, int px,
                                                       int pxpy) {
    const int n = blockIdx.x * kBlock + threadIdx.x;
    if (n >= d.n_sites) return;
    d.phi[1][n] = phi0_of_site(d, n, phi0, nx, ny, px, pxpy);
}

// fp16 storage: the references' phase sum of every site for a step of parity
// PAR (what the collision stores in rsum), after an initialisation or an import.
template <int PAR>
__global__ void __launch_bounds__(kBlock) k_ref_sum(DomainView d) {
    const int n = blockIdx.x * kBlock + threadIdx.x;
    if (n >= d.n_sites) return;
    d.rsum[n] = reference_phase_sum<PAR>(d, n);
}

// Initial state consistent with phi0 (rho = 1, u = 0), written in the even
// (natural) layout: Na = (1 + phi0)/2, Nb = (1 - phi0)/2. With fp16 storage the
// density reference is rho = 1 and the component references come from the
// phases that k_init_phase wrote.
template <class S>
__global__ void __launch_bounds__(kBlock) k_init(DomainView d, const float* phi0, int nx, int ny,
                                                 int px, int pxpy) {
    const int n = blockIdx.x * kBlock + threadIdx.x;
    if (n >= d.n_sites) return;
    const float p = phi0_of_site(d, n, phi0, nx, ny, px, pxpy);
    const float na = 0.5f * (1.0f + p), nb = 0.5f * (1.0f - p);
    int face[Q7];
    if constexpr (S::kRef) {
        d.drho[n] = 0.0f;
        face_neighbours(d, n, face);
    }
    const size_t P = d.pitch;
    static_for<0, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        S::template st_f<q>(d.f, q * P + n, t19(q));
        if constexpr (q < Q7) {
            float av = w7(q) * na, bv = w7(q) * nb;
            if constexpr (S::kRef) {
                const float pw = writer_phase<0, q>(d, n, face);
                av -= w7(q) * 0.5f * (1.0f + pw);
                bv -= w7(q) * 0.5f * (1.0f - pw);
            }
            S::template st_c<q>(d.a, q * P + n, av);
            S::template st_c<q>(d.b, q * P + n, bv);
        }
    });
}

inline unsigned blocks_for(long long n) { return static_cast<unsigned>((n + kBlock - 1) / kBlock); }

}  // namespace

DomainView make_view(const lbpm_ctx* c) {
    DomainView d{};
    d.n_sites = static_cast<int>(c->N);
    d.pitch = static_cast<int>(pitch_of(c->N));
    d.px = static_cast<int>(c->px);
    d.pxpy = static_cast<int>(c->px * c->py);
    d.site_vox = c->d_site_vox;
    d.vsite = c->d_vsite;
    d.phi[0] = c->d_phi;
    d.phi[1] = c->d_phi_alt ? c->d_phi_alt : c->d_phi;
    d.link_a = c->d_link_a;
    d.link_b = c->d_link_b;
    for (int k = 0; k < 2; ++k) d.phis_at[k] = static_cast<unsigned>(c->d_phis - d.phi[k]);
    d.nsum = c->d_nsum;
    d.drho = c->d_drho;
    d.rsum = c->d_rsum;
    d.f = c->d_f;
    d.a = c->d_a;
    d.b = c->d_b;
    d.acc = c->d_acc;
    const lbpm_params& p = c->params;
    d.tau_a = static_cast<float>(p.tau_a);
    d.tau_b = static_cast<float>(p.tau_b);
    d.alpha = static_cast<float>(p.alpha);
    d.beta = static_cast<float>(p.beta);
    d.fx = static_cast<float>(p.force[0]);
    d.fy = static_cast<float>(p.force[1]);
    d.fz = static_cast<float>(p.force[2]);
    const float K = p.precision == LBPM_FP16 ? StoreF16::kK : StoreF32::kK;
    for (int k = 0; k < 9; ++k) {
        const int q = 2 * k + 1;
        d.fterm[k] = K * (3.0f * t19(q) * (cx(q) * d.fx + cy(q) * d.fy + cz(q) * d.fz));
    }
    d.uniform_tau = p.tau_a == p.tau_b;
    const float s_nu = 1.0f / static_cast<float>(p.tau_a);
    d.s_nu = s_nu;
    d.s_m = 8.0f * (2.0f - s_nu) / (8.0f - s_nu);
    return d;
}

cudaError_t launch_init_fluids(const lbpm_ctx* c, const float* phi0, cudaStream_t s) {
    DomainView d = make_view(c);
    if (c->N == 0) return cudaSuccess;
    const bool h = c->params.precision == LBPM_FP16;
    if (h) {
        k_init_phase<<<blocks_for(c->N), kBlock, 0, s>>>(d, phi0, c->nx, c->ny, c->px, c->px * c->py);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        k_init<StoreF16><<<blocks_for(c->N), kBlock, 0, s>>>(d, phi0, c->nx, c->ny, c->px, c->px * c->py);
        k_ref_sum<0><<<blocks_for(c->N), kBlock, 0, s>>>(d);
    } else {
        k_init<StoreF32><<<blocks_for(c->N), kBlock, 0, s>>>(d, phi0, c->nx, c->ny, c->px, c->px * c->py);
    }
    return cudaGetLastError();
}

cudaError_t launch_ref_sum(const lbpm_ctx* c, int parity, cudaStream_t s) {
    if (c->params.precision != LBPM_FP16 || c->N == 0) return cudaSuccess;
    if (parity == 0) k_ref_sum<0><<<blocks_for(c->N), kBlock, 0, s>>>(make_view(c));
    else k_ref_sum<1><<<blocks_for(c->N), kBlock, 0, s>>>(make_view(c));
    return cudaGetLastError();
}

template <class S, bool SUMS>
cudaError_t launch_phase_form(const lbpm_ctx* c, int parity, cudaStream_t s) {
    const unsigned g = blocks_for(c->N);
    if (g == 0) return cudaSuccess;
    DomainView d = make_view(c);
    return parity == 0 ? launch_pdl(k_phase<0, S, SUMS>, g, s, d) : launch_pdl(k_phase<1, S, SUMS>, g, s, d);
}

cudaError_t launch_phase(const lbpm_ctx* c, int parity, bool sums, cudaStream_t s) {
    if (c->params.precision == LBPM_FP16)
        return sums ? launch_phase_form<StoreF16, true>(c, parity, s) : launch_phase_form<StoreF16, false>(c, parity, s);
    return sums ? launch_phase_form<StoreF32, true>(c, parity, s) : launch_phase_form<StoreF32, false>(c, parity, s);
}

// one collision launch of the given parity, storage, component form and block size
template <int PAR, class S, int CF, int BT>
cudaError_t launch_collide_shape(const lbpm_ctx* c, cudaStream_t s) {
    return launch_pdl_bt(k_collide<PAR, S, CF, BT>, static_cast<unsigned>((c->N + BT - 1) / BT), BT, s, make_view(c));
}
template <int PAR, int CF>
cudaError_t launch_collide_form(const lbpm_ctx* c, cudaStream_t s) {
    if (c->N == 0) return cudaSuccess;
    if (c->params.precision == LBPM_FP16) return launch_collide_shape<PAR, StoreF16, CF, 128>(c, s);
    return c->N < kSmallSites ? launch_collide_shape<PAR, StoreF32, CF, 128>(c, s)
                              : launch_collide_shape<PAR, StoreF32, CF, 256>(c, s);
}

cudaError_t launch_collide(const lbpm_ctx* c, int parity, cudaStream_t s) {
    return parity == 0 ? launch_collide_form<0, 0>(c, s) : launch_collide_form<1, 0>(c, s);
}

cudaError_t launch_phase_sum(const lbpm_ctx* c, int parity, cudaStream_t s) {
    const unsigned g = blocks_for((c->N + kPhaseSumPer - 1) / kPhaseSumPer);
    if (g == 0) return cudaSuccess;
    DomainView d = make_view(c);
    return parity == 0 ? launch_pdl(k_phase_sum<0>, g, s, d) : launch_pdl(k_phase_sum<1>, g, s, d);
}

cudaError_t launch_collide_sum(const lbpm_ctx* c, int parity, cudaStream_t s) {
    return parity == 0 ? launch_collide_form<0, 1>(c, s) : launch_collide_form<1, 1>(c, s);
}

// parity = parity of the step that will READ the reset values; reservoir slabs
// (reservoir_z = 1) or the boundary at the z faces (2: pressure, 3: flux inlet)
template <int PAR, class S, bool SUMS>
cudaError_t launch_reservoir_form(const lbpm_ctx* c, cudaStream_t s) {
    const DomainView d = make_view(c);
    const unsigned g = blocks_for(c->n_slab);
    const int ns = static_cast<int>(c->n_slab);
    const lbpm_params& p = c->params;
    const float ri = static_cast<float>(p.rho_in), ro = static_cast<float>(p.rho_out);
    const int* const st = c->d_slab_site;
    const signed char* const sd = c->d_slab_side;
    if (p.reservoir_z == 1) return launch_pdl(k_reservoir<PAR, S, SUMS>, g, s, d, st, sd, ns, ri, ro);
    // rho - 1 formed in double, so the small difference keeps full fp32 precision
    const float di = static_cast<float>(p.rho_in - 1.0), dout = static_cast<float>(p.rho_out - 1.0);
    const float* face = nullptr;
    if (p.reservoir_z == 3) {
        const cudaError_t e = launch_pdl(k_face_rho<PAR, S>, kFaceBlocks, s, d, st, sd, ns, c->d_face_part, p.flux_in,
                                         c->d_face_rho);
        if (e != cudaSuccess) return e;
        face = c->d_face_rho;
    }
    return launch_pdl(k_pressure_faces<PAR, S>, g, s, d, st, sd, ns, ri, ro, di, dout, face);
}
template <int PAR>
cudaError_t launch_reservoir_par(const lbpm_ctx* c, bool sums, cudaStream_t s) {
    if (c->params.precision == LBPM_FP16)
        return sums ? launch_reservoir_form<PAR, StoreF16, true>(c, s) : launch_reservoir_form<PAR, StoreF16, false>(c, s);
    return sums ? launch_reservoir_form<PAR, StoreF32, true>(c, s) : launch_reservoir_form<PAR, StoreF32, false>(c, s);
}

cudaError_t launch_reservoir(const lbpm_ctx* c, int parity, bool sums, cudaStream_t s) {
    if (c->n_slab == 0) return cudaSuccess;
    return parity == 0 ? launch_reservoir_par<0>(c, sums, s) : launch_reservoir_par<1>(c, sums, s);
}

}  // namespace lbm
