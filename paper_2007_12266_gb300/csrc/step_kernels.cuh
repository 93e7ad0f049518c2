// Device code of one color-gradient LBM timestep (Sec. 3.1), shared by the
// single-domain launchers and the batched launcher.
//
// State layout (structure of arrays, population-major, in place):
//   F[q*P + n], A[q*P + n], B[q*P + n]      (P: N rounded up, DomainView::pitch)
// AA streaming: at an even step site n reads its own slots F[q][n] and writes
// the post-collision value of direction q to F[opp(q)][n]. At an odd step it
// reads direction q from F[opp(q)][m] where m is the upstream neighbour
// (x - xi_q) or, if that voxel is solid, from F[q][n] (bounce-back), and it
// writes direction q to F[q][m'] with m' = x + xi_q, or to F[opp(q)][n] when
// x + xi_q is solid (halfway bounce-back). Each site reads and writes the same
// slots within a step, so one array suffices and no two sites collide.
#pragma once

#include "internal.h"
#include "lattice.cuh"
#include "links.cuh"

namespace lbm {

// explicitly rounded fp32 operations (never contracted)
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// ---------------------------------------------------------------------------
// storage of the distributions
// ---------------------------------------------------------------------------

// Plain fp32 storage. ld_fdev / st_fdev exchange deviations f_q - t_q from
// the rest state, which the collision works with.
struct StoreF32 {
    using T = float;
    static constexpr bool kRef = false;   // component values stored as they are
    // Hot-path forms: p points at the slot itself; the stored number as it
    // is (see collide_thread).
    static constexpr float kK = 1.0f;
    static __device__ __forceinline__ float ld_s(const T* p) { return *p; }
    static __device__ __forceinline__ void st_s(T* p, float v) { *p = v; }
    // a stored momentum population as a deviation from rest, and back
    template <int Q>
    static __device__ __forceinline__ float deviation(float x, float) { return sub(x, t19(Q)); }
    template <int Q>
    static __device__ __forceinline__ float stored(float dev) { return add(t19(Q), dev); }
    template <int Q>
    static __device__ __forceinline__ float ld_fdev(const void* p, size_t i) {
        return static_cast<const float*>(p)[i] - t19(Q);
    }
    template <int Q>
    static __device__ __forceinline__ void st_fdev(void* p, size_t i, float dev) {
        static_cast<float*>(p)[i] = t19(Q) + dev;
    }
    template <int Q>
    static __device__ __forceinline__ float ld_f(const void* p, size_t i) {
        return static_cast<const float*>(p)[i];
    }
    template <int Q>
    static __device__ __forceinline__ void st_f(void* p, size_t i, float v) {
        static_cast<float*>(p)[i] = v;
    }
    template <int Q>
    static __device__ __forceinline__ float ld_c(const void* p, size_t i) {
        return static_cast<const float*>(p)[i];
    }
    template <int Q>
    static __device__ __forceinline__ void st_c(void* p, size_t i, float v) {
        static_cast<float*>(p)[i] = v;
    }
};

// fp16 storage of deviations from a local rest-state equilibrium, arithmetic
// in fp32. Momentum: f_q - t_q rho(s), with rho of a reference site s kept in
// fp32 per site (DomainView::drho): the writing site for values written at an
// even step (read at the next odd step through the neighbour table) and the
// destination site, with its density of the last even step, for values
// written at an odd step (read at the next even step by that destination with
// one coalesced load); drho is written only at even steps.
// Components: A_q - w_q (1 + phi_w)/2 and B_q - w_q (1 - phi_w)/2, with phi_w
// the phase of the site w that wrote the value, at that step. The writer uses
// its own phase; the reader finds phi_w in the previous step's phases
// (DomainView::phi is double-buffered by step parity) at the upstream site
// x - xi_q, or at its own when that link bounced back. The phase pass needs only the sum
// of the references over the seven directions, Na = sum_q s_q + (1 + S)/2
// with S = sum_q w_q phi_w(q) (likewise Nb with -S; the writers' rest values
// absorb the fp32 weights' excess over 1); the collision, which holds those
// phases for its colour gradient, stores S per site (DomainView::rsum), so the
// phase pass reads one coalesced number instead of six phases. Against the
// writer's own (Na, Nb) the stored number gains w_q (N - 1)(1 +- phi_w)/2;
// N = Na + Nb follows the density, within a few 1e-2 of 1.
// Storing A, B themselves let every site of a pure phase round the same value
// the same way on the fp16 grid, a biased error that leaked 3e-3 of the
// component mass per 1,000 steps; storing f - t_q left the local density
// excursion (up to a few 1e-2 under a body force and capillary pressure) in
// the stored number and cost the velocity its precision. Referencing the
// components to the phase of the reading site instead (known to the reader
// without any lookup) left (phi_w - phi_r)/2, up to w_q at a sharp interface,
// in the stored numbers and raised the flux error against the oracle tenfold.
// ld_fdev / st_fdev below exchange the stored number; the kernels add the
// reference.
// Values are scaled by 2^14 (an exact power of two) to keep small deviations
// out of fp16's subnormal range; |deviation| up to 4 stays representable.
struct StoreF16 {
    using T = __half;
    static constexpr bool kRef = true;
    static constexpr float kScale = 16384.0f;
    static constexpr float kInv = 1.0f / 16384.0f;
    // Hot-path forms: the collision works in units of 2^-14 (kK = 2^14 times
    // the deviations), so the stored number is used as it is and the scale
    // costs no multiplication per value.
    static constexpr float kK = kScale;
    static __device__ __forceinline__ float ld_s(const T* p) { return __half2float(*p); }
    static __device__ __forceinline__ void st_s(T* p, float v) { *p = __float2half_rn(v); }
    // a stored momentum population, relative to the reference density deviation
    // `ref`, as a deviation from rest in working units
    template <int Q>
    static __device__ __forceinline__ float deviation(float x, float ref) { return fma(t19(Q) * kK, ref, x); }
    template <int Q>
    static __device__ __forceinline__ float stored(float dev) { return dev; }
    template <int Q>
    static __device__ __forceinline__ float ld_fdev(const void* p, size_t i) {
        return __half2float(static_cast<const __half*>(p)[i]) * kInv;
    }
    template <int Q>
    static __device__ __forceinline__ void st_fdev(void* p, size_t i, float dev) {
        static_cast<__half*>(p)[i] = __float2half_rn(dev * kScale);
    }
    template <int Q>
    static __device__ __forceinline__ float ld_f(const void* p, size_t i) {
        return t19(Q) + ld_fdev<Q>(p, i);
    }
    template <int Q>
    static __device__ __forceinline__ void st_f(void* p, size_t i, float v) {
        st_fdev<Q>(p, i, v - t19(Q));
    }
    template <int Q>
    static __device__ __forceinline__ float ld_c(const void* p, size_t i) {
        return __half2float(static_cast<const __half*>(p)[i]) * kInv;
    }
    template <int Q>
    static __device__ __forceinline__ void st_c(void* p, size_t i, float v) {
        static_cast<__half*>(p)[i] = __float2half_rn(v * kScale);
    }
};

// Programmatic dependent launch (sm_90+): a kernel launched with programmatic
// stream serialization may start while the previous kernel in the stream is
// still running. wait_prior_grid() blocks until that kernel has completed and
// its writes are visible; allow_next_grid() lets the next kernel start its
// blocks. Without the launch attribute both are no-ops.
// Data written by an earlier kernel of the step chain (phi, nsum, the
// fp16 reference densities, the populations) is read with plain coherent
// loads only: a read-only (__ldg / .nc) load may legally be hoisted by the
// compiler above wait_prior_grid(), which would read the previous step's
// values. __ldg is kept for the static index arrays.
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next_grid() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------
// sum form: component densities carried as per-site fixed-point sums
// ---------------------------------------------------------------------------
// The recolored populations of Eqs. LBE-mass-a/b are a function of the
// writing site's Na, Nb, velocity and colour normal, and the next step uses
// the populations a site receives only through their sums Na, Nb. In the sum
// form the collision moves each recolored value A*_q, B*_q from the sums of its
// site to the sums of the site that receives it, x + xi_q (on a bounce-back link
// it stays). The sums are updated in place: the collision itself reads N and phi,
// which the phase pass formed from them, and only adds to them. A site's (Na, Nb)
// is one 64-bit word: Na in the high and Nb in the
// low 32 bits, each in units of 2^-28 (|N| < 8). Adding packed words adds both
// halves exactly as long as the low sum stays within 32 bits, and integer sums
// do not depend on the order of the additions, so the result is deterministic
// and each component's mass is conserved exactly.
constexpr float kSumOne = 268435456.0f;          // 2^28
constexpr float kSumInv = 1.0f / 268435456.0f;

__device__ __forceinline__ unsigned long long pack_sums(int a, int b) {
    return (static_cast<unsigned long long>(static_cast<unsigned>(a)) << 32) +
           static_cast<unsigned long long>(static_cast<long long>(b));
}
__device__ __forceinline__ void unpack_sums(unsigned long long s, int& a, int& b) {
    b = static_cast<int>(static_cast<unsigned>(s));
    a = static_cast<int>((static_cast<long long>(s) - static_cast<long long>(b)) >> 32);
}
// N = Na + Nb and phi = (Na - Nb)/(Na + Nb) of a site from its sums, in fp32
// (32-bit integer to float conversions: a 64-bit conversion runs on the fp64
// pipe, which is slow on this GPU).
__device__ __forceinline__ void sums_phase(int a, int b, float& Nt, float& phi) {
    const float fa = static_cast<float>(a), fb = static_cast<float>(b);
    const float nt = fa + fb;
    Nt = nt * kSumInv;
    phi = nt > 0.0f ? (fa - fb) / nt : 0.0f;
}
// The sums (8 bytes per site, touched by both kernels of every step) are accessed
// with an L2 evict-last policy, so that they stay in L2 while the populations
// stream through it.
__device__ __forceinline__ unsigned long long l2_keep() {
    unsigned long long pol;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void red_add(unsigned long long* p, unsigned long long v, unsigned long long pol) {
    asm volatile("red.relaxed.gpu.global.add.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(p), "l"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ unsigned long long ld_keep(const unsigned long long* p, unsigned long long pol) {
    unsigned long long v;
    asm volatile("ld.global.L2::cache_hint.u64 %0, [%1], %2;" : "=l"(v) : "l"(p), "l"(pol) : "memory");
    return v;
}
__device__ __forceinline__ void st_keep(unsigned long long* p, unsigned long long v, unsigned long long pol) {
    asm volatile("st.global.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(p), "l"(v), "l"(pol) : "memory");
}

// ---------------------------------------------------------------------------
// AA read map: where the value of direction Q of site n lives at a step of
// parity PAR (the same slot the step writes direction opp(Q) to).
// ---------------------------------------------------------------------------
template <int PAR, int Q>
__device__ __forceinline__ size_t read_slot(const DomainView& d, int n, const int* nb) {
    const size_t P = static_cast<size_t>(d.pitch);
    if constexpr (Q == 0 || PAR == 0) {
        return static_cast<size_t>(Q) * P + n;
    } else {
        // upstream site x - xi_Q = x + xi_opp(Q), or -1 (bounce-back)
        const int up = nb[opp(Q)];
        return up >= 0 ? static_cast<size_t>(opp(Q)) * P + up : static_cast<size_t>(Q) * P + n;
    }
}

// ---------------------------------------------------------------------------
// component populations (D3Q7, Eqs. LBE-mass-a/b)
// ---------------------------------------------------------------------------
// The site that wrote slot read_slot<PAR, Q>(n) during the previous step: the
// upstream neighbour x - xi_Q if it is a pore, else n itself (bounce-back).
template <int Q>
__device__ __forceinline__ int writer_of(int n, const int* nb) {
    if constexpr (Q == 0) {
        return n;
    } else {
        const int up = nb[opp(Q)];
        return up >= 0 ? up : n;
    }
}

// Site whose density is the reference of the momentum population read as
// direction Q by site n at a step of parity PAR (see StoreF16).
template <int PAR, int Q>
__device__ __forceinline__ int f_ref_read(int n, const int* nb) {
    if constexpr (PAR == 0) return n;
    else return writer_of<Q>(n, nb);
}

// Phase of the site that wrote the component value read as direction Q by site
// n at a step of parity PAR (fp16 storage, see StoreF16): from the previous
// step's phases, at the upstream site x - xi_Q, or at n when x - xi_Q is solid
// (nb: the face neighbours' ids, negative where there is none).
template <int PAR, int Q>
__device__ __forceinline__ float writer_phase(const DomainView& d, int n, const int* nb) {
    return d.phi[PAR ^ 1][writer_of<Q>(n, nb)];
}

// A_q, B_q of site n at a step of parity PAR (nb[1..6]: face neighbours, needed
// where need_face_nb() says so).
template <int PAR, class S>
__device__ __forceinline__ void load_components(const DomainView& d, int n, const int* nb, float (&a)[Q7],
                                                float (&b)[Q7]) {
    static_for<0, Q7>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const size_t i = read_slot<PAR, q>(d, n, nb);
        a[q] = S::template ld_c<q>(d.a, i);
        b[q] = S::template ld_c<q>(d.b, i);
        if constexpr (S::kRef) {
            const float pw = writer_phase<PAR, q>(d, n, nb);
            a[q] = fmaf(w7(q) * 0.5f, 1.0f + pw, a[q]);
            b[q] = fmaf(w7(q) * 0.5f, 1.0f - pw, b[q]);
        }
    });
}

// fp16 storage: S = sum_q w_q phi_w(q) over the seven component values that
// site n reads at a step of parity PAR (see writer_phase).
template <int PAR>
__device__ __forceinline__ float reference_phase_sum(const DomainView& d, int n) {
    int nb[Q7];
    face_neighbours(d, n, nb);
    float S = 0.0f;
    static_for<0, Q7>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        S = fmaf(w7(q), writer_phase<PAR, q>(d, n, nb), S);
    });
    return S;
}

// Whether the face-neighbour ids are needed to read or write the components:
// for their slots at odd steps, for their references with fp16 storage.
template <int PAR, class S>
constexpr bool need_face_nb() { return PAR == 1 || S::kRef; }

// ---------------------------------------------------------------------------
// phase pass: Na, Nb -> phi and N of each site                      Sec. 3.1
// ---------------------------------------------------------------------------
// Phase pass of one site. Ordering with the neighbouring kernels under
// programmatic launch: only the static index is read before wait_prior_grid();
// A and B (written by the previous collision) are read, and phi / nsum (read by
// the previous collision) are written, only after it. Dependents are released
// after the wait, so the next collision never starts before the previous
// one has completed.
// SUMS: the first step of a run of the sum form, whose collision finds the
// site's sums set to its Na, Nb.
template <int PAR, class S, bool SUMS = false>
__device__ __forceinline__ void phase_thread(const DomainView& d, int n) {
    const bool ok = n < d.n_sites;
    int nb[Q7];
    if constexpr (PAR == 1) {
        if (ok) face_neighbours(d, n, nb);
    }
    wait_prior_grid();
    allow_next_grid();
    if (!ok) return;
    float Na = 0.0f, Nb = 0.0f;
    if constexpr (S::kRef) {
        // stored deviations plus the references' sum, (1 +- rsum)/2 (the
        // writers' rest values absorb the fp32 weights' excess over 1)
        static_for<0, Q7>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            const size_t i = read_slot<PAR, q>(d, n, nb);
            Na += S::template ld_c<q>(d.a, i);
            Nb += S::template ld_c<q>(d.b, i);
        });
        const float Sr = d.rsum[n];
        Na = fmaf(0.5f, 1.0f + Sr, Na);
        Nb = fmaf(0.5f, 1.0f - Sr, Nb);
    } else {
        float a[Q7], b[Q7];
        load_components<PAR, S>(d, n, nb, a, b);
        static_for<0, Q7>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            Na += a[q];
            Nb += b[q];
        });
    }
    const float Nt = Na + Nb;
    const float phi = Nt > 0.0f ? (Na - Nb) / Nt : 0.0f;
    d.phi[PAR][n] = phi;
    d.nsum[n] = Nt;
    if constexpr (SUMS) {
        const float half = mul(0.5f * kSumOne, Nt);
        st_keep(d.acc + n,
                pack_sums(__float2int_rn(mul(half, add(1.0f, phi))), __float2int_rn(mul(half, sub(1.0f, phi)))),
                l2_keep());
    }
}

// Phase pass of the sum form: phi and N from the site's component sums, for
// PER sites per thread (t0 + k * stride). Ordering as in phase_thread: the sums
// were completed by the collision before.
template <int PAR, int PER>
__device__ __forceinline__ void phase_sum_thread(const DomainView& d, int t0, int stride) {
    const unsigned long long pol = l2_keep();
    wait_prior_grid();
    allow_next_grid();
    unsigned long long s[PER];
    #pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int n = t0 + k * stride;
        s[k] = n < d.n_sites ? ld_keep(d.acc + n, pol) : 0ull;
    }
    #pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int n = t0 + k * stride;
        if (n >= d.n_sites) continue;
        int a, b;
        unpack_sums(s[k], a, b);
        float Nt, phi;
        sums_phase(a, b, Nt, phi);
        d.phi[PAR][n] = phi;
        d.nsum[n] = Nt;
    }
}

// ---------------------------------------------------------------------------
// fused collide + stream                                            Sec. 3.1
// ---------------------------------------------------------------------------
// Component forms of the collision (CF): 0 stores the recolored populations
// (AA slots); 1 moves them between the sites' sums (sum form). Both take Na, Nb
// from the phase pass, as N and phi.
// At an odd step site n reads direction opp(q) from, and writes direction q
// to, the same slot: row q at the downstream neighbour x + xi_q, or row
// opp(q) at n itself when that voxel is solid. With fp16 storage both also
// use the same density reference (that neighbour's density of the last even
// step, which odd steps do not change); SlotCache keeps it between the gather
// and the scatter, in shared memory laid out [row][thread] so that a warp's
// accesses fall in distinct banks.
// The neighbours' ids come from the site's record (DENSE = false: every lane's
// record is regular), formed again from its eight ranks wherever one is used,
// or from the dense grid of ids (DENSE = true), each looked up once and kept in
// the slot cache.
struct SlotCache {
    int* slot;      // DENSE: entry of direction 1 of this thread, direction q at slot[(q - 1) * stride]:
                    // slot_word of q (odd steps), the face neighbour's site id (even steps
                    // of the sum form)
    float* ref;     // the density reference of direction q's slot at ref[(q - 1) * stride] (fp16, odd steps)
    int stride;     // threads per block
};

// What a site reads before anything is known about its neighbours.
template <class S>
struct SiteState {
    SiteLinks l;
    float f[Q19];                   // even steps: the populations in the own slots (stored numbers); odd: f[0]
    float ref = 0.0f;               // fp16: the own slots' reference density (deviation)
    int v;                          // the site's voxel
};

// Collision, recoloring and streaming of site n. The arithmetic is written in
// explicitly rounded operations (no contraction is left to the compiler), so a
// site's result is the same bit for bit in every kernel this is compiled into.
// Which operations they are, and in which order, is part of the result: where the
// colour gradient nearly cancels, in pockets of a few voxels, the normal hangs on
// the last bits, and any other rounding moves single sites by a thousandth and more
// within a few hundred steps, in both storages. (A form over pairs of opposite
// directions with the solids' part of the gradient summed beforehand took a hundred
// instructions fewer per site and 137 / 130 us per step (fp32 / fp16) instead of 151 /
// 136, and was nearer to 64 bits in norm, but single sites of a 256^3 pack, and of
// batches, came out up to 4e-3 of the largest value away.)
//
// What bounds it: DRAM with fp32 storage, with fp16 the latency of the loads, with 32
// warps per SM resident, and the instructions (689 and 870 per site at even and odd
// steps in fp32, 738 and 1043 in fp16). So neighbours come from a 24-byte
// record per site and the phase is kept per site: against gathering 18 phases and 18
// (odd) or 6 site ids from dense voxel grids, where the 32 sites of a warp span about
// 150 voxels, the phase pass needs no site -> voxel map and no scattered stores, and
// only the solid neighbours (2 of 18 on average in a sphere pack of porosity 0.22) are
// read by voxel. And the component sums are updated in place, in one array that stays
// in L2 instead of two of which the collision reads one and clears it. Together, us per
// step before and now: 167 and 151 in fp32 and 157 and 136 in fp16 on 3.69 M sites of
// a 256^3 pack, 8.1 and 6.3 in fp32 on 79 k sites. Not everywhere a gain in fp32: on
// 734 k sites with a periodic x axis 29.2 and 30.8, on 1.02 M 44.7 and 46.3, where the
// step runs out of L2 and 36 instead of 32 warps cover its latency better.
template <int PAR, class S, int CF, bool DENSE>
__device__ __forceinline__ void collide_site(const DomainView& d, int n, const SiteState<S>& in, SlotCache sc) {
    SiteLinks l = in.l;
    using T = typename S::T;
    constexpr float K = S::kK;                      // working units: deviations times K
    constexpr float iK = 1.0f / K;
    int pitch = d.pitch;
    T* const F = static_cast<T*>(d.f);
    const unsigned long long pol = l2_keep();
    const int v = in.v;
    // id of x + xi_q where has(q)
    auto has = [&](auto qc) { return link_has<decltype(qc)::value>(l); };
    auto id = [&](auto qc) {
        constexpr int q = decltype(qc)::value;
        if constexpr (!DENSE) return link_id<q>(n, l);
        else if constexpr (PAR == 1 || (CF != 0 && q < Q7)) return sc.slot[(q - 1) * sc.stride];
        else return __ldg(d.vsite + v + stencil_off(d, q));
    };
    // slot that direction q is written to (and opp(q) read from) at odd steps
    auto slot = [&](auto qc, T* base) {
        constexpr int q = decltype(qc)::value;
        T* const row = base + q * static_cast<size_t>(pitch);
        if constexpr (DENSE) return slot_at<q>(row, static_cast<unsigned>(sc.slot[(q - 1) * sc.stride]));
        else return slot_at<q>(row, slot_word<q>(has(qc), id(qc), n, pitch));
    };
    // the record and the pitch from here on are values the compiler knows nothing
    // about: ids, slots and row addresses formed before are formed again instead
    // of being kept in registers (in the batched kernels, whose views are not
    // compile-time uniform, keeping them spilled 140-290 bytes per thread and took
    // 270 / 284 us per step of a 12-job set in fp32 / fp16 against 246 / 229)
    auto forget_ids = [&] {
        if constexpr (!DENSE) asm volatile("" : "+r"(l.a.x), "+r"(l.a.y), "+r"(l.a.z), "+r"(l.b.x), "+r"(l.b.y));
        asm volatile("" : "+r"(l.a.w), "+r"(n), "+r"(pitch));
    };

    // incoming distributions as deviations d_q = f_q - t_q from the rest state
    // (exact in fp32 near rest), so that density and momentum are sums of small
    // numbers and the relaxation acts on small quantities; in working units
    float f[Q19];
    const float ref_own = in.ref;
    static_for<0, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        if constexpr (PAR == 0 || q == 0) f[q] = S::template deviation<q>(in.f[q], ref_own);
    });
    if constexpr (PAR == 1) {
        static_for<1, Q19>([&](auto qc) {
            constexpr int q = decltype(qc)::value;   // direction of the downstream slot
            constexpr int o = opp(q);                // direction read from it
            if constexpr (DENSE) {
                const int m = __ldg(d.vsite + v + stencil_off(d, q));
                sc.slot[(q - 1) * sc.stride] = static_cast<int>(slot_word<q>(m >= 0, m, n, pitch));
            }
            const float x = S::ld_s(slot(qc, F));
            float r = 0.0f;
            if constexpr (S::kRef) {
                r = d.drho[has(qc) ? id(qc) : n];
                sc.ref[(q - 1) * sc.stride] = r;
            }
            f[o] = S::template deviation<o>(x, r);
        });
    }
    if constexpr (DENSE && CF != 0 && PAR == 0) {
        // sum form, even step: the face neighbours that receive the component values
        static_for<1, Q7>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            sc.slot[(q - 1) * sc.stride] = __ldg(d.vsite + v + stencil_off(d, q));
        });
    }
    forget_ids();

    // Everything above (neighbour ids and f from the previous collision) is safe to
    // read before the phase pass of this step completes; phi and nsum are its outputs,
    // and the A/B slots written below are its inputs.
    allow_next_grid();
    wait_prior_grid();

    // colour gradient C = sum_q g_q xi_q phi(x + xi_q), summed in the order of the
    // directions: pores' phases per site, solids' phi_s from the voxel grid, which lies
    // within 32-bit reach of the phases so that one load takes either, at a selected
    // index. On 256^3 in fp32 / fp16: 151 / 136 us per step; loads under opposite
    // predicates took 162 / 145, one through a selected pointer 151 / 141, the solids'
    // values packed site after site (8 B per site more) 147 / 139.
    const float* const phi = d.phi[PAR];
    const unsigned vs = static_cast<unsigned>(v) + d.phis_at[PAR];
    float Cx = 0.0f, Cy = 0.0f, Cz = 0.0f;
    static_for<1, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        constexpr float g = grad_w(q);
        const unsigned i = has(qc) ? static_cast<unsigned>(id(qc)) : vs + static_cast<unsigned>(stencil_off(d, q));
        const float p = S::kRef && PAR == 1 ? phi[i] : phi[static_cast<int>(i)];
        if constexpr (cx(q) != 0) Cx = fma(g * cx(q), p, Cx);
        if constexpr (cy(q) != 0) Cy = fma(g * cy(q), p, Cy);
        if constexpr (cz(q) != 0) Cz = fma(g * cz(q), p, Cz);
    });
    const float phi_c = phi[n];
    const float Nt = d.nsum[n];
    if constexpr (S::kRef && CF == 0) {
        // references of the values the next phase pass reads at this site: the
        // phase of x - xi_q, which this step writes, or this site's own on a
        // bounce-back link; every face direction has the same weight
        float Sf = 0.0f;
        static_for<1, Q7>([&](auto qc) { Sf += has(qc) ? phi[id(qc)] : phi_c; });
        d.rsum[n] = fmaf(w7(1), Sf, w7(0) * phi_c);
    }
    forget_ids();

    // macroscopic moments: drho = rho - 1 and j from the deviations
    float drho = f[0], jx = 0.0f, jy = 0.0f, jz = 0.0f;
    static_for<1, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        drho = add(drho, f[q]);
        if constexpr (cx(q) > 0) jx = add(jx, f[q]);
        if constexpr (cx(q) < 0) jx = sub(jx, f[q]);
        if constexpr (cy(q) > 0) jy = add(jy, f[q]);
        if constexpr (cy(q) < 0) jy = sub(jy, f[q]);
        if constexpr (cz(q) > 0) jz = add(jz, f[q]);
        if constexpr (cz(q) < 0) jz = sub(jz, f[q]);
    });

    const float C2 = fma(Cz, Cz, fma(Cx, Cx, mul(Cy, Cy)));
    float nx = 0.0f, ny = 0.0f, nz = 0.0f, Cmag = 0.0f;
    if (C2 > 0.0f) {
        const float inv = rsqrtf(C2);
        Cmag = mul(C2, inv);
        nx = mul(Cx, inv);
        ny = mul(Cy, inv);
        nz = mul(Cz, inv);
    }

    // relaxation rates from the viscosity (tau mixed linearly in phi)
    float s_nu = d.s_nu, s_m = d.s_m;
    if (!d.uniform_tau) {
        const float half = mul(d.tau_a - d.tau_b, 0.5f), pa = add(1.0f, phi_c);
        const float tau = fma(half, pa, d.tau_b);
        s_nu = __fdiv_rn(1.0f, tau);
        s_m = __fdiv_rn(mul(8.0f, sub(2.0f, s_nu)), sub(8.0f, s_nu));
    }

    // MRT collision, evaluated in its equivalent two-relaxation-time form.
    // With S from the viscosity, every non-conserved even moment (m1, m2,
    // m9..m15) relaxes with s_nu and every non-conserved odd moment (m4, m6,
    // m8, m16..m18) with s_m; the conserved ones equal their equilibria. So
    //   f* = f - s_nu (f+ - feq+) - s_m (f- - feq-) + 3 t_q xi_q . F
    // with f+- the even/odd parts over opposite pairs and feq the velocity-
    // space equilibrium whose moments are m^eq:
    //   feq+ = t_q (rho + 4.5 (xi.j)^2 - 1.5 j.j) + M^-1 dm_alpha
    //   feq- = 3 t_q xi.j
    // where dm_alpha holds the interfacial-tension terms of m1, m9, m11,
    // m13, m14, m15 (rho0 = 1). Everything below is relative to the rest
    // state t_q (rho = 1), i.e. in deviations, and in working units: the
    // equilibrium's quadratic terms take one factor 1/K, the interfacial terms
    // and the forcing (d.fterm is stored in working units) one factor K.
    const float jj = fma(jz, jz, fma(jx, jx, mul(jy, jy)));
    const float ac = mul(mul(d.alpha, K), Cmag);
    const float hac = mul(0.5f, ac);
    float dma[Q19];
    dma[1] = -ac;
    {
        const float i9 = fma(mul(2.0f, nx), nx, -mul(ny, ny));
        dma[9] = mul(hac, fma(-nz, nz, i9));
        dma[11] = mul(hac, fma(-nz, nz, mul(ny, ny)));
    }
    dma[13] = mul(mul(hac, nx), ny);
    dma[14] = mul(mul(hac, ny), nz);
    dma[15] = mul(mul(hac, nx), nz);
    const float drho_iso = fma(-1.5f * iK, jj, drho);

    // recoloring weights Nb/N and Na/N are (1 - phi)/2 and (1 + phi)/2
    const float bxa = mul(mul(d.beta, 0.5f), sub(1.0f, phi_c));
    const float bxb = mul(mul(d.beta, 0.5f), add(1.0f, phi_c));

    // destination of direction q (q >= 1): row opp(q) at n (even step) or the
    // slot of row q it was read from (odd step)
    auto store = [&](auto qc, T* base, float x) {
        constexpr int q = decltype(qc)::value;
        if constexpr (PAR == 0) S::st_s(base + opp(q) * static_cast<size_t>(pitch) + n, x);
        else S::st_s(slot(qc, base), x);
    };

    // The increments of the moving populations sum to minus the rest
    // increment in exact arithmetic; taking the rest increment as that sum
    // keeps fp32 mass exact up to unbiased rounding.
    float dsum = 0.0f;
    static_for<0, 9>([&](auto pc) {
        constexpr int q = 2 * decltype(pc)::value + 1;   // q odd, opp(q) = q + 1
        constexpr int o = q + 1;
        constexpr float t = t19(q), t3 = 3.0f * t;
        float cu;
        if constexpr (q == 1) cu = jx;
        if constexpr (q == 3) cu = jy;
        if constexpr (q == 5) cu = jz;
        if constexpr (q == 7) cu = add(jx, jy);
        if constexpr (q == 9) cu = sub(jx, jy);
        if constexpr (q == 11) cu = add(jx, jz);
        if constexpr (q == 13) cu = sub(jx, jz);
        if constexpr (q == 15) cu = add(jy, jz);
        if constexpr (q == 17) cu = sub(jy, jz);
        float eqp = mul(t, fma(mul(4.5f * iK, cu), cu, drho_iso));
        static_for<1, 16>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            if constexpr (k == 1 || k == 9 || k == 11 || k == 13 || k == 14 || k == 15) {
                if constexpr (mrow(k, q) != 0) eqp = fma(minv(q, k), dma[k], eqp);
            }
        });
        const float ev = fma(0.5f, add(f[q], f[o]), -eqp);          // f+ - feq+
        const float D = sub(f[q], f[o]);
        const float od = fma(0.5f, D, -mul(t3, cu));   // f- - feq-
        const float dmi = fma(-s_m, od, d.fterm[q >> 1]);
        const float inc_q = fma(-s_nu, ev, dmi);
        const float inc_o = fma(-s_nu, ev, -dmi);
        if constexpr (q == 1) dsum = add(inc_q, inc_o);
        else dsum = add(dsum, add(inc_q, inc_o));
        float vq = add(f[q], inc_q), vo = add(f[o], inc_o);
        if constexpr (S::kRef) {
            // even step: relative to this site's rest state t_q rho; odd step:
            // relative to the destination's density of the last even step
            if constexpr (PAR == 0) {
                vq = fma(-t, drho, vq);
                vo = fma(-t, drho, vo);
            } else {
                vq = fma(-t * K, sc.ref[(q - 1) * sc.stride], vq);
                vo = fma(-t * K, sc.ref[(o - 1) * sc.stride], vo);
            }
        }
        store(std::integral_constant<int, q>{}, F, S::template stored<q>(vq));
        store(std::integral_constant<int, o>{}, F, S::template stored<o>(vo));
    });
    {
        float r0 = sub(f[0], dsum);
        if constexpr (S::kRef && PAR == 0) {
            r0 = fma(-t19(0), drho, r0);
            d.drho[n] = mul(iK, drho);
        }
        if constexpr (S::kRef && PAR == 1) r0 = fma(-t19(0) * K, ref_own, r0);
        S::st_s(F + n, S::template stored<0>(r0));
    }

    // recolored component distributions (Eqs. LBE-mass-a/b), streamed on the
    // fly; the rest populations take the remainder of Na and Nb so that the
    // fp32 weights (whose sum is not exactly 1) create no mass. With fp16
    // storage the stored quantity is the deviation from w_q (1 +- phi_c)/2: the
    // deviation from w_q Na (w_q Nb), which the formula gives directly as
    // w_q Na (4.5 u.xi + beta Nb/N n.xi), plus w_q times
    //   Na - (1 + phi_c)/2 = (N - 1)(1 + phi_c)/2   (likewise for Nb).
    // (working units: Na, Nb times K, j divided by K back to u)
    const float pa1 = add(1.0f, phi_c), pb1 = sub(1.0f, phi_c);   // 1 + phi, 1 - phi
    const float j3[3] = {jx, jy, jz}, n3[3] = {nx, ny, nz};
    if constexpr (CF != 0) {
        // Sum form: A*_q = w_q Na [1 + 4.5 u.xi_q + beta (Nb/N) n.xi_q] (likewise B*_q)
        // in fixed point, moved from the site's sums to those of the site that
        // receives it; the rest value, and the values of bounce-back links, stay.
        unsigned long long out = 0;
        unsigned long long* const acc = d.acc;
        const float NS = mul(0.5f * kSumOne, Nt);
        const float PA = mul(w7(1), mul(NS, pa1)), PB = mul(w7(1), mul(NS, pb1));
        static_for<1, Q7>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            constexpr int i = (q - 1) >> 1;
            const float base = fma(q & 1 ? 4.5f * iK : -4.5f * iK, j3[i], 1.0f);
            const float ma = mul(bxa, n3[i]), mb = mul(bxb, n3[i]);
            const float ya = q & 1 ? add(base, ma) : sub(base, ma);
            const float yb = q & 1 ? sub(base, mb) : add(base, mb);
            if (has(qc)) {
                const unsigned long long x = pack_sums(__float2int_rn(mul(PA, ya)), __float2int_rn(mul(PB, yb)));
                out -= x;
                red_add(acc + id(qc), x, pol);
            }
        });
        red_add(acc + n, out, pol);
    } else {
        T* const A = static_cast<T*>(d.a);
        T* const B = static_cast<T*>(d.b);
        const float NK = mul(0.5f * K, Nt);
        const float Na = mul(NK, pa1), Nb = mul(NK, pb1);
        const float PA = mul(w7(1), Na), PB = mul(w7(1), Nb);
        if constexpr (S::kRef) {
            // K (N - 1)(1 +- phi_c)/2, the offsets of the references; the values
            // of opposite directions cancel in the sum of the six
            const float hN = mul(0.5f * K, add(Nt, -1.0f));
            const float eA = mul(hN, pa1), eB = mul(hN, pb1);
            static_for<0, 3>([&](auto ic) {
                constexpr int i = decltype(ic)::value;
                const std::integral_constant<int, 2 * i + 1> q;
                const std::integral_constant<int, 2 * i + 2> o;
                const float av = mul(PA, fma(4.5f * iK, j3[i], mul(bxa, n3[i])));
                const float bv = mul(PB, fma(4.5f * iK, j3[i], -mul(bxb, n3[i])));
                store(q, A, fma(w7(1), eA, av));
                store(q, B, fma(w7(1), eB, bv));
                store(o, A, fma(w7(1), eA, -av));
                store(o, B, fma(w7(1), eB, -bv));
            });
            // The phase pass adds (1 + S)/2 to the seven values a site reads, S
            // holding w_q phi_c for this site's value of direction q; the seven
            // stored values above sum to Wsum (Na - (1 + phi_c)/2) with Wsum the
            // fp32 weights' sum 1 + 2^-26. The rest value takes the difference,
            // K (1 - Wsum)(Na - 1/2), so that its readers rebuild exactly Na (and
            // Nb) and the fp32 weights create no mass.
            constexpr double kWsum = static_cast<double>(w7(0)) + 6.0 * static_cast<double>(w7(1));
            constexpr float kWerr = static_cast<float>(1.0 - kWsum);
            S::st_s(A + n, fma(kWerr, add(-0.5f * K, Na), mul(w7(0), eA)));
            S::st_s(B + n, fma(kWerr, add(-0.5f * K, Nb), mul(w7(0), eB)));
        } else {
            float asum = 0.0f, bsum = 0.0f;
            static_for<1, Q7>([&](auto qc) {
                constexpr int q = decltype(qc)::value;
                constexpr int i = (q - 1) >> 1;
                constexpr float sgn = q & 1 ? 1.0f : -1.0f;
                const float base = fma(sgn * 4.5f * iK, j3[i], 1.0f);
                const float av = mul(PA, fma(bxa, sgn * n3[i], base)), bv = mul(PB, fma(-bxb, sgn * n3[i], base));
                asum = q == 1 ? av : add(asum, av);
                bsum = q == 1 ? bv : add(bsum, bv);
                store(qc, A, av);
                store(qc, B, bv);
            });
            S::st_s(A + n, sub(Na, asum));
            S::st_s(B + n, sub(Nb, bsum));
        }
    }
}

// The loads that need no neighbour come first, then one path per warp: through
// the records if all of them are regular, else through the dense grid of ids.
template <int PAR, class S, int CF>
__device__ __forceinline__ void collide_thread(const DomainView& d, int n, SlotCache sc) {
    using T = typename S::T;
    const size_t P = static_cast<size_t>(d.pitch);
    const T* const F = static_cast<const T*>(d.f);
    SiteState<S> in;
    in.l = SiteLinks{__ldg(d.link_a + n), __ldg(d.link_b + n)};
    static_for<0, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        if constexpr (PAR == 0 || q == 0) in.f[q] = S::ld_s(F + q * P + n);
    });
    if constexpr (S::kRef) in.ref = d.drho[n];
    in.v = __ldg(d.site_vox + n);
    if (__any_sync(__activemask(), in.l.a.w & kIrregular)) collide_site<PAR, S, CF, true>(d, n, in, sc);
    else collide_site<PAR, S, CF, false>(d, n, in, sc);
}

// ---------------------------------------------------------------------------
// reservoir reset (unsteady protocol, Sec. 4.1): write the rest state into
// the slots the NEXT step (parity PAR) reads.
// ---------------------------------------------------------------------------
// SUMS: the sum form, where the next step reads the component sums (set to
// the reset state Na = 1, Nb = 0 at the inlet, 0 and 1 at the outlet) instead
// of the D3Q7 populations.
template <int PAR, class S, bool SUMS = false>
__device__ __forceinline__ void reservoir_thread(const DomainView& d, int n, int side, float rho_in,
                                                 float rho_out) {
    const int v = d.site_vox[n];
    int nb[Q19];
    if constexpr (PAR == 1) {
        static_for<1, Q19>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            nb[q] = __ldg(d.vsite + v + stencil_off(d, q));
        });
    }
    // fp16: the component references of the next step's reads (see StoreF16)
    if constexpr (S::kRef && PAR == 0) face_neighbours(d, n, nb);
    const float rho = side == 1 ? rho_in : rho_out;
    const float na = side == 1 ? 1.0f : 0.0f;
    static_for<0, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        const size_t i = read_slot<PAR, q>(d, n, nb);
        if constexpr (S::kRef) {
            const float dw = d.drho[f_ref_read<PAR, q>(n, nb)];
            S::template st_fdev<q>(d.f, i, t19(q) * (rho - 1.0f - dw));
        } else {
            S::template st_f<q>(d.f, i, t19(q) * rho);
        }
        if constexpr (q < Q7 && !SUMS) {
            float av = w7(q) * na, bv = w7(q) * (1.0f - na);
            if constexpr (S::kRef) {
                const float pw = writer_phase<PAR, q>(d, n, nb);
                av -= w7(q) * 0.5f * (1.0f + pw);
                bv -= w7(q) * 0.5f * (1.0f - pw);
            }
            S::template st_c<q>(d.a, i, av);
            S::template st_c<q>(d.b, i, bv);
        }
    });
    if constexpr (SUMS) {
        constexpr int one = 1 << 28;   // kSumOne
        d.acc[n] = side == 1 ? pack_sums(one, 0) : pack_sums(0, one);
    }
}

// ---------------------------------------------------------------------------
// pressure boundary at the z faces (Sec. 4.1: constant inlet and outlet
// pressures; Zou and He's non-equilibrium bounce-back): after streaming, the
// five populations that enter a face site from outside the domain (c_z = +1
// at the inlet z = 0, c_z = -1 at the outlet z = nz - 1) are set so that the
// site's density is the face density and its tangential velocity is zero:
//   u_z = +-(1 - (S_0 + 2 S_out) / rho)      S_0: c_z = 0, S_out: leaving
//   f_in(normal) = f_out(normal) +- rho u_z / 3
//   f_in(edge)   = f_out(opposite edge) +- rho u_z / 6 -+ N_t,
//   N_t = (1/2) sum_{c_z = 0} c_t f   (t = x, y, the tangential momentum)
// The one entering D3Q7 population of each component is the reservoir
// fluid's equilibrium at the face velocity: inlet A = w rho_in (1 + 4.5 u_z),
// B = 0; outlet B = w rho_out (1 - 4.5 u_z), A = 0. The values go into the
// slots the NEXT step (parity PAR) reads.
// ---------------------------------------------------------------------------
// Incoming populations of the next step at face site n as deviations
// d_q = f_q - t_q, and D = S_0 + 2 S_out - 1 in deviations (the weights of
// S_0 + 2 S_out add up to one): u_n is then formed from small numbers and
// rho - 1 instead of cancelling O(1) sums. nb: neighbour ids (filled here).
template <int PAR, class S>
__device__ __forceinline__ float face_deviations(const DomainView& d, int n, float sgn, int (&nb)[Q19],
                                                 float (&dv)[Q19], float& nx, float& ny) {
    const int v = d.site_vox[n];
    if constexpr (PAR == 1) {
        static_for<1, Q19>([&](auto qc) {
            constexpr int q = decltype(qc)::value;
            nb[q] = __ldg(d.vsite + v + stencil_off(d, q));
        });
    }
    static_for<0, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        dv[q] = S::template ld_fdev<q>(d.f, read_slot<PAR, q>(d, n, nb));
        if constexpr (S::kRef) dv[q] = fmaf(t19(q), d.drho[f_ref_read<PAR, q>(n, nb)], dv[q]);
    });
    float D = 0.0f;
    nx = 0.0f;
    ny = 0.0f;
    static_for<0, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        if constexpr (cz(q) == 0) {
            D += dv[q];
            if constexpr (cx(q) != 0) nx += cx(q) * dv[q];
            if constexpr (cy(q) != 0) ny += cy(q) * dv[q];
        } else {
            if (cz(q) * sgn < 0.0f) D += 2.0f * dv[q];   // leaving the domain through this face
        }
    });
    return D;
}

// face: (rho, rho - 1) of the inlet computed on the device (flux inlet), or
// nullptr to take rho_in, drho_in
template <int PAR, class S>
__device__ __forceinline__ void pressure_face_thread(const DomainView& d, int n, int side, float rho_in,
                                                     float rho_out, float drho_in, float drho_out,
                                                     const float* face) {
    if (face && side == 1) {
        rho_in = face[0];
        drho_in = face[1];
    }
    int nb[Q19];
    float dv[Q19];
    const float sgn = side == 1 ? 1.0f : -1.0f;       // face normal into the domain
    const float rho = side == 1 ? rho_in : rho_out;
    const float drho = side == 1 ? drho_in : drho_out;
    float nx, ny;
    const float D = face_deviations<PAR, S>(d, n, sgn, nb, dv, nx, ny);
    nx *= 0.5f;
    ny *= 0.5f;
    const float un = (drho - D) / rho;                // velocity along the inward normal
    const float j3 = rho * un * (1.0f / 3.0f), j6 = rho * un * (1.0f / 6.0f);
    static_for<1, Q19>([&](auto qc) {
        constexpr int q = decltype(qc)::value;
        if constexpr (cz(q) != 0) {
            if (cz(q) * sgn > 0.0f) {
                float dev = dv[opp(q)] + (cx(q) == 0 && cy(q) == 0 ? j3 : j6);
                if constexpr (cx(q) != 0) dev -= cx(q) * nx;
                if constexpr (cy(q) != 0) dev -= cy(q) * ny;
                const size_t i = read_slot<PAR, q>(d, n, nb);
                if constexpr (S::kRef) dev = fmaf(-t19(q), d.drho[f_ref_read<PAR, q>(n, nb)], dev);
                S::template st_fdev<q>(d.f, i, dev);
            }
        }
    });
    // the entering component population
    const float uz = sgn * un;
    static_for<5, 7>([&](auto qc) {
        constexpr int q = decltype(qc)::value;   // 5: +z, 6: -z
        if (cz(q) * sgn > 0.0f) {
            const float y = fma(4.5f * cz(q), uz, 1.0f);
            const float eq = mul(mul(w7(q), rho), y);
            float av = side == 1 ? eq : 0.0f, bv = side == 1 ? 0.0f : eq;
            if constexpr (S::kRef) {
                // the reference the next step reads it with (see StoreF16)
                if constexpr (PAR == 0) face_neighbours(d, n, nb);
                const float pw = writer_phase<PAR, q>(d, n, nb);
                // av - h (1 + pw), bv - h (1 - pw); the operations are part of the result,
                // as in collide_site
                constexpr float h = 0.5f * w7(q);
                const float ra = mul(h, add(1.0f, pw)), rb = sub(1.0f, pw);
                av = side == 1 ? fma(mul(w7(q), rho), y, -ra) : -ra;
                if constexpr (PAR == 0) bv = side == 1 ? -mul(h, rb) : fma(mul(w7(q), rho), y, -mul(h, rb));
                else bv = side == 1 ? -mul(h, rb) : fma(-h, rb, eq);
            }
            const size_t i = read_slot<PAR, q>(d, n, nb);
            S::template st_c<q>(d.a, i, av);
            S::template st_c<q>(d.b, i, bv);
        }
    });
}

}  // namespace lbm
