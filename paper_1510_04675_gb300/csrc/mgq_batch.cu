// libmgq batched driver: many independent lattices of (possibly) different
// extents, couplings and RNG streams advanced together -- the parallel
// rethermalisation of N_s prolongated configurations (Sec. II: "embarrassingly
// parallel").  Each sub-sweep is ONE launch over all lattices: the grid is a
// flattened list of 128-site blocks, block b belongs to the lattice l with
// prefix[l] <= b < prefix[l+1].  The lattice descriptors travel as kernel
// parameters (no device-side table), so a whole call can be captured into a
// CUDA graph as is.
#include <cstring>

#include "mgq_internal.h"
#include "mgq_columns.cuh"
#include "mgq_stencil.cuh"
#include "mgq_terms.cuh"

namespace mgq {

constexpr int BATCH_CHUNK = 128;  // lattices per launch (kernel-parameter table)
constexpr int BATCH_THREADS = 128;     // the kernels' maximal block size
constexpr int BATCH_MIN_THREADS = 32;  // the smallest tunable block size (sizes the partial sums)

template <class T>
struct LatDesc {
    Cx<T>* links;
    Geom g;
    T beta;
    uint2 key;
};

template <class T>
struct Batch {
    int n;
    int prefix[BATCH_CHUNK + 1];  // block offsets
    LatDesc<T> d[BATCH_CHUNK];
};

template <class T>
__device__ __forceinline__ int find_lattice(const Batch<T>& B, int b) {
    int lo = 0, hi = B.n;  // prefix[lo] <= b < prefix[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (B.prefix[mid] <= b) lo = mid; else hi = mid;
    }
    return lo;
}

template <class T>
__device__ __forceinline__ const Geom& geom_of(const LatDesc<T>& d) {
    return d.g;
}

// The staple of U_MU(x) and the link itself: staged through shared memory for
// FP32 12-real links (staple_staged; the launch gives STAGED_THREADS threads and
// STAGED_SMEM bytes), as in the single-lattice kernels, so that batched and
// single-lattice updates agree bit for bit; plain loads otherwise.
// early(), PACKED and FMA as in staple_staged (48 uneven lattices, one compound sweep: 3.05 ->
// 2.99 ms with the draws early and single-FMA rotations).
template <class T, int NP, int MU, bool PACKED = false, bool FMA = true, class Work = NoWork>
__device__ __forceinline__ void staple_and_link(const Links<T, NP>& U, const Geom& g, const int x[4], int h, int par,
                                                M3<T>& A, M3<T>& u, Work early = Work()) {
    if constexpr (sizeof(T) == 4 && NP == 6) {
        extern __shared__ float4 staged_sm[];
        A = staple_staged<PACKED, FMA>(U, g, x, h, MU, par, staged_sm, u, early);
    } else {
        A = staple(U, g, x, h, MU, par);
        u = U.load(MU, par, h);
    }
}

// blocks per SM the kernels are compiled for: the staged ones fill shared memory with five
template <class T, int NP> constexpr int batch_blocks() { return sizeof(T) == 8 ? 2 : (NP == 6 ? 5 : 4); }

// NHB1: single-attempt instance (the attempt loop is removed at compile time; staged
// links: the draws are taken while the first loads are in flight)
template <class T, int NP, int MU, bool NHB1>
__global__ void __launch_bounds__(BATCH_THREADS, NHB1 ? batch_blocks<T, NP>() : 4 - 2 * (sizeof(T) == 8))
    k_heatbath_batched(const __grid_constant__ Batch<T> B, int par, uint32_t idx_lo, uint32_t idx_hi, int n_hb) {
    if constexpr (NHB1) n_hb = 1;
    pdl_launch_dependents();
    const int l = find_lattice(B, blockIdx.x);
    const LatDesc<T>& d = B.d[l];
    const int h = (blockIdx.x - B.prefix[l]) * (int)blockDim.x + threadIdx.x;
    pdl_wait();
    if (h >= d.g.Vh) return;
    const Geom g = geom_of(d);
    Links<T, NP> U;
    U.p = d.links;
    U.S = d.g.S;
    RngKey rk;
    rk.key = d.key;
    rk.idx_lo = idx_lo;
    rk.idx_hi = idx_hi;
    int x[4];
    cb_coords(g, par, h, x);
    M3<T> A, u;
    const uint32_t lex = (uint32_t)lex_of(g, x);
    if constexpr (NHB1 && sizeof(T) == 4 && NP == 6) {
        uint4 r[3];
        staple_and_link<T, NP, MU, true>(U, g, x, h, par, A, u, [&]() {
#pragma unroll
            for (int s = 0; s < 3; s++) r[s] = draw(rk, lex, (uint32_t)MU, (uint32_t)s, 0u, KIND_HB);
        });
        hb_link_drawn(u, A, d.beta, r);
    } else {
        // packed throughout: beside the attempt loop single FMAs cost more (24 lattices of
        // 8^3x16 to 16^4, three attempts: 456 us a sweep against 430)
        staple_and_link<T, NP, MU, true, false>(U, g, x, h, par, A, u);
        hb_link<true>(u, A, d.beta, n_hb, rk, lex, (uint32_t)MU, (uint8_t*)nullptr);
    }
    U.store(MU, par, h, u);
}

template <class T, int NP, int MU>
__global__ void __launch_bounds__(BATCH_THREADS, batch_blocks<T, NP>()) k_overrelax_batched(const __grid_constant__ Batch<T> B, int par) {
    pdl_launch_dependents();
    const int l = find_lattice(B, blockIdx.x);
    const LatDesc<T>& d = B.d[l];
    const int h = (blockIdx.x - B.prefix[l]) * (int)blockDim.x + threadIdx.x;
    pdl_wait();
    if (h >= d.g.Vh) return;
    const Geom g = geom_of(d);
    Links<T, NP> U;
    U.p = d.links;
    U.S = d.g.S;
    int x[4];
    cb_coords(g, par, h, x);
    M3<T> A, u;
    staple_and_link<T, NP, MU>(U, g, x, h, par, A, u);
    or_link<(NP == 9)>(u, A);
    U.store(MU, par, h, u);
}

// Launches over few links in all, as for single lattices: FP32 with a staple term per
// warp (blocks of TERMS_LINKS links), FP64 with a column per lane (12 lattices of 6^4,
// 8^4 and 4^3x8, one compound sweep with plaquettes: 12-real 273 -> 170 us, FP64 6.9 -> 2.1
// ms).
template <int NP, int KIND, int WARPS, bool FMA>
__global__ void __launch_bounds__(WARPS * TERMS_LINKS, 24 / WARPS)
    k_update_terms_batched(const __grid_constant__ Batch<float> B, int mu, int par, uint32_t idx_lo, uint32_t idx_hi,
                           double* __restrict__ partials) {
    const int l = find_lattice(B, blockIdx.x);
    const LatDesc<float>& d = B.d[l];
    Links<float, NP> U;
    U.p = d.links;
    U.S = d.g.S;
    RngKey rk;
    rk.key = d.key;
    rk.idx_lo = idx_lo;
    rk.idx_hi = idx_hi;
    update_terms<NP, KIND, WARPS, FMA>(U, geom_of(d), blockIdx.x - B.prefix[l], mu, par, d.beta, rk,
                                  KIND == TERMS_OVERRELAX_LAST ? partials + par * B.prefix[B.n] + blockIdx.x : nullptr);
}

template <bool HB, int LPL>
__global__ void __launch_bounds__(COL_THREADS)
    k_update_columns_batched(const __grid_constant__ Batch<double> B, int mu, int par, uint32_t idx_lo, uint32_t idx_hi, int n_hb) {
    const int l = find_lattice(B, blockIdx.x);
    const LatDesc<double>& d = B.d[l];
    Links<double, 9> U;
    U.p = d.links;
    U.S = d.g.S;
    RngKey rk;
    rk.key = d.key;
    rk.idx_lo = idx_lo;
    rk.idx_hi = idx_hi;
    update_columns<HB, LPL>(U, geom_of(d), blockIdx.x - B.prefix[l], mu, par, d.beta, rk, n_hb, nullptr, nullptr);
}

// The last overrelaxation sweep's direction-3 sub-sweeps with the plaquette
// folded in, as in the single-lattice driver: partial sums per block at
// partials[par * nblocks + blockIdx.x].
template <class T, int NP>
__global__ void __launch_bounds__(BATCH_THREADS, sizeof(T) == 8 ? 2 : 4)
    k_overrelax_batched_last(const __grid_constant__ Batch<T> B, int par, double* __restrict__ partials) {
    pdl_launch_dependents();
    const int l = find_lattice(B, blockIdx.x);
    const LatDesc<T>& d = B.d[l];
    const int h = (blockIdx.x - B.prefix[l]) * (int)blockDim.x + threadIdx.x;
    pdl_wait();
    double acc = 0.0;
    if (h < d.g.Vh) {
        const Geom g = geom_of(d);
        Links<T, NP> U;
        U.p = d.links;
        U.S = d.g.S;
        int x[4];
        cb_coords(g, par, h, x);
        M3<T> A, u;
        staple_and_link<T, NP, 3>(U, g, x, h, par, A, u);
        if (par == 1) acc = (double)retr_nn(u, A);
        or_link<(NP == 9)>(u, A);
        U.store(3, par, h, u);
        acc += site_plaquettes<T, NP, 3>(U, g, par, h);
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) partials[par * B.prefix[B.n] + blockIdx.x] = acc;
}

// one block per lattice: both parities' partials of its blocks, times 1/(18 V)
template <class T>
__global__ void k_overrelax_batched_last_final(const __grid_constant__ Batch<T> B, const double* __restrict__ partials,
                                               double* __restrict__ out) {
    const int l = blockIdx.x, nb = B.prefix[B.n];
    double v = 0.0;
    for (int i = B.prefix[l] + threadIdx.x; i < B.prefix[l + 1]; i += blockDim.x) v += partials[i] + partials[nb + i];
    v = block_sum(v);
    if (threadIdx.x == 0) out[l] = v / (18.0 * (double)B.d[l].g.V);
}

// per-lattice plaquette: blocks of 256 sites, partial sums at the global block index
template <class T, int NP>
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 1 : 2) k_plaquette_batched(const __grid_constant__ Batch<T> B, double* __restrict__ partials) {
    const int l = find_lattice(B, blockIdx.x);
    const LatDesc<T>& d = B.d[l];
    const int idx = (blockIdx.x - B.prefix[l]) * 256 + threadIdx.x;
    double acc = 0.0;
    if (idx < d.g.V) {
        Links<T, NP> U;
        U.p = d.links;
        U.S = d.g.S;
        const int par = idx >= d.g.Vh, h = idx - par * d.g.Vh;
        acc = site_plaquettes(U, geom_of(d), par, h);
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// one block per lattice: fixed-order sum of its partials, times 1/(18 V)
template <class T>
__global__ void k_plaquette_batched_final(const __grid_constant__ Batch<T> B, const double* __restrict__ partials,
                                          double* __restrict__ out) {
    const int l = blockIdx.x;
    double v = 0.0;
    for (int i = B.prefix[l] + threadIdx.x; i < B.prefix[l + 1]; i += blockDim.x) v += partials[i];
    v = block_sum(v);
    if (threadIdx.x == 0) out[l] = v / (18.0 * (double)B.d[l].g.V);
}

// one FP32 sub-sweep of the launch over `links` links with `warps` warps per 32 links
template <int NP, int KIND>
static void launch_terms_batched(int warps, long links, const Batch<float>& B, int mu, int par, uint64_t sweep, double* partials, cudaStream_t st) {
    launch_pdl(warps == 6                 ? k_update_terms_batched<NP, KIND, 6, true>
               : term_single_fma(links) ? k_update_terms_batched<NP, KIND, 3, true>
                                        : k_update_terms_batched<NP, KIND, 3, NP == 9>,  // 18-real launches stay below
               B.prefix[B.n], warps * TERMS_LINKS, st, B, mu, par, (uint32_t)(sweep & 0xffffffffu), (uint32_t)(sweep >> 32), partials);
}
// one FP64 sub-sweep with `lanes` lanes per link
template <bool HB>
static void launch_columns_batched(int lanes, const Batch<double>& B, int mu, int par, uint64_t sweep, int n_hb, cudaStream_t st) {
    launch_pdl(lanes == 3 ? k_update_columns_batched<HB, 3> : k_update_columns_batched<HB, 6>, B.prefix[B.n], COL_THREADS, st, B, mu,
               par, (uint32_t)(sweep & 0xffffffffu), (uint32_t)(sweep >> 32), n_hb);
}

template <class T>
static void fill_batch(Batch<T>& B, const mgq_lattice* lats, const double* betas, int first, int n, int sites_per_block,
                       bool half) {
    B.n = n;
    B.prefix[0] = 0;
    for (int i = 0; i < n; i++) {
        const mgq_lattice& L = lats[first + i];
        const Geom g = make_geom(L.dims);
        LatDesc<T>& d = B.d[i];
        d.links = reinterpret_cast<Cx<T>*>(L.links);
        d.g = g;
        d.beta = betas ? (T)betas[first + i] : T(1);
        const RngKey rk = make_rng(L.seed, L.lattice_id, 0);
        d.key = rk.key;
        const int units = half ? g.Vh : g.V;
        B.prefix[i + 1] = B.prefix[i] + (units + sites_per_block - 1) / sites_per_block;
    }
}

// partial-sum slots: two per 128-site half-lattice block (the plaquette-
// measuring overrelaxation sub-sweeps), which also covers one per 256-site
// block (the plaquette kernel)
uint64_t batch_partials(const mgq_lattice* lats, int n) {
    uint64_t nb = 0;
    for (int i = 0; i < n; i++) {
        const Geom g = make_geom(lats[i].dims);
        nb += 2 * (uint64_t)((g.Vh + BATCH_MIN_THREADS - 1) / BATCH_MIN_THREADS);
    }
    return nb;
}

}  // namespace mgq

using namespace mgq;

extern "C" {

int mgq_launch_threads(int kernel, const mgq_lattice* lats, int n_lat, int* tunable) {
    if (tunable) *tunable = 0;
    if (kernel < 0 || kernel >= MGQ_NKERNELS || !lats || n_lat < 1) return 0;
    const bool batched = kernel == MGQ_KERNEL_HEATBATH_BATCHED || kernel == MGQ_KERNEL_OVERRELAX_BATCHED;
    if (!batched && kernel != MGQ_KERNEL_APE && n_lat != 1) return 0;
    const int prec = lats[0].prec;
    if (prec < MGQ_F64 || prec > MGQ_F32_C12) return 0;
    for (int i = 0; i < n_lat; i++)
        if (!valid_dims(lats[i].dims) || lats[i].prec != prec) return 0;
    const int set = block_size(kernel, prec);
    int first_threads = 0;
    for (int first = 0; first < n_lat; first += BATCH_CHUNK) {
        long links = 0;
        for (int i = first; i < n_lat && i < first + BATCH_CHUNK; i++) links += make_geom(lats[i].dims).Vh;
        const int warps = term_warps(prec, links);
        const bool columns = prec == MGQ_F64 && update_lanes(links) > 1;
        const int fixed = kernel == MGQ_KERNEL_APE ? 0 : columns ? COL_THREADS : warps ? warps * TERMS_LINKS : prec == MGQ_F32_C12 ? STAGED_THREADS : 0;
        if (!fixed) {
            if (tunable) *tunable = 1;
            return set;
        }
        if (!first) first_threads = fixed;
    }
    return first_threads;
}

uint64_t mgq_batch_workspace_bytes(const mgq_lattice* lats, int n_lat, int n_sweeps) {
    if (!lats || n_lat < 1 || n_sweeps < 0) return 0;
    for (int i = 0; i < n_lat; i++)
        if (!valid_dims(lats[i].dims)) return 0;
    return round256(batch_partials(lats, n_lat) * sizeof(double)) + round256((uint64_t)n_sweeps * n_lat * sizeof(double));
}

mgq_status mgq_update_sweeps_batched(mgq_lattice* lats, int n_lat, const double* betas, uint64_t sweep0, int n_sweeps,
                                     int n_hb, int n_or, double* plaq_out, void* batch_work, uint64_t batch_work_bytes,
                                     void* stream) {
    Trace trace("mgq_update_sweeps_batched");
    if (!lats || n_lat < 1) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: need at least one lattice");
    if (!betas) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: betas is NULL");
    mgq_status s;
    for (int i = 0; i < n_lat; i++) {
        if ((s = check_lattice(&lats[i], false, "mgq_update_sweeps_batched"))) return s;
        if (lats[i].prec != lats[0].prec) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: all lattices need one precision");
        if (!(betas[i] > 0.0) || betas[i] > 1e6) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: beta[%d] invalid", i);
    }
    if (n_hb < 1 || n_hb > 256) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: n_hb must be in [1, 256]");
    if (n_sweeps < 0 || n_or < 0) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: negative counts");
    const uint64_t need = mgq_batch_workspace_bytes(lats, n_lat, n_sweeps);
    if (plaq_out) {
        if (!batch_work) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: plaquettes need batch_work");
        if (((uintptr_t)batch_work & 255) != 0) return fail(MGQ_EINVAL, "mgq_update_sweeps_batched: batch_work not 256-byte aligned");
        if (batch_work_bytes < need)
            return fail(MGQ_ENOMEM, "mgq_update_sweeps_batched: batch_work has %llu bytes, needs %llu",
                        (unsigned long long)batch_work_bytes, (unsigned long long)need);
    }
    cudaStream_t st = as_stream(stream);
    double* partials = reinterpret_cast<double*>(batch_work);
    double* results =
        plaq_out ? reinterpret_cast<double*>((char*)batch_work + round256(batch_partials(lats, n_lat) * sizeof(double)))
                 : nullptr;
    for (int i = 0; i < n_sweeps; i++) {
        const uint64_t sweep = sweep0 + (uint64_t)i;
        for (int first = 0; first < n_lat; first += BATCH_CHUNK) {
            const int n = (n_lat - first < BATCH_CHUNK) ? n_lat - first : BATCH_CHUNK;
            dispatch_prec(lats[0].prec, [&]<class T, int NP>() {
                const bool staged = sizeof(T) == 4 && NP == 6;
                const int bh = staged ? STAGED_THREADS : block_size(MGQ_KERNEL_HEATBATH_BATCHED, lats[0].prec);
                const int bo = staged ? STAGED_THREADS : block_size(MGQ_KERNEL_OVERRELAX_BATCHED, lats[0].prec);
                const size_t smem = staged ? (size_t)STAGED_SMEM : 0;
                Batch<T> Bl, Bo;
                fill_batch(Bl, lats, betas, first, n, bh, true);
                fill_batch(Bo, lats, betas, first, n, bo, true);
                const int nblocks = Bl.prefix[n], oblocks = Bo.prefix[n];
                // with a plaquette record, the last overrelaxation sweep's
                // direction-3 sub-sweeps measure it (per-chunk partials)
                const bool fold = plaq_out && n_or > 0;
                long links = 0;
                for (int l = 0; l < n; l++) links += Bl.d[l].g.Vh;
                auto heatbath = [&](int mu, int par) {
                    dispatch_mu(mu, [&]<int MU>() {
                        if (n_hb == 1)
                            launch_pdl_smem(k_heatbath_batched<T, NP, MU, true>, nblocks, bh, smem, st, Bl, par,
                                       (uint32_t)(sweep & 0xffffffffu), (uint32_t)(sweep >> 32), n_hb);
                        else
                            launch_pdl_smem(k_heatbath_batched<T, NP, MU, false>, nblocks, bh, smem, st, Bl, par,
                                       (uint32_t)(sweep & 0xffffffffu), (uint32_t)(sweep >> 32), n_hb);
                    });
                };
                auto overrelax = [&](int mu, int par) {
                    dispatch_mu(mu, [&]<int MU>() {
                        launch_pdl_smem(k_overrelax_batched<T, NP, MU>, oblocks, bo, smem, st, Bo, par);
                    });
                };
                auto overrelax_last = [&](int par) {
                    launch_pdl_smem(k_overrelax_batched_last<T, NP>, oblocks, bo, smem, st, Bo, par, partials);
                };
                auto sweeps = [&](auto&& hb, auto&& orx, auto&& last) {
                    for (int mu = 0; mu < 4; mu++)
                        for (int par = 0; par < 2; par++) hb(mu, par);
                    for (int k = 0; k < n_or; k++)
                        for (int mu = 0; mu < 4; mu++)
                            for (int par = 0; par < 2; par++)
                                if (fold && k == n_or - 1 && mu == 3) last(par);
                                else orx(mu, par);
                };
                if constexpr (sizeof(T) == 4) {
                    if (const int warps = term_warps(lats[0].prec, links)) {
                        Batch<T> Bt;
                        fill_batch(Bt, lats, betas, first, n, TERMS_LINKS, true);
                        sweeps([&](int mu, int par) {
                            if (n_hb == 1) launch_terms_batched<NP, TERMS_HEATBATH>(warps, links, Bt, mu, par, sweep, nullptr, st);
                            else heatbath(mu, par);
                        }, [&](int mu, int par) {
                            launch_terms_batched<NP, TERMS_OVERRELAX>(warps, links, Bt, mu, par, sweep, nullptr, st);
                        }, [&](int par) {
                            launch_terms_batched<NP, TERMS_OVERRELAX_LAST>(warps, links, Bt, 3, par, sweep, partials, st);
                        });
                        if (fold)
                            k_overrelax_batched_last_final<T><<<n, 256, 0, st>>>(Bt, partials, results + (size_t)i * n_lat + first);
                        return;
                    }
                } else if (const int lanes = update_lanes(links); lanes > 1) {
                    Batch<T> Bc;
                    fill_batch(Bc, lats, betas, first, n, lanes == 3 ? ColumnLane<3>::kPerBlock : ColumnLane<6>::kPerBlock, true);
                    sweeps([&](int mu, int par) { launch_columns_batched<true>(lanes, Bc, mu, par, sweep, n_hb, st); },
                           [&](int mu, int par) { launch_columns_batched<false>(lanes, Bc, mu, par, 0, 0, st); }, overrelax_last);
                    if (fold)
                        k_overrelax_batched_last_final<T><<<n, 256, 0, st>>>(Bo, partials, results + (size_t)i * n_lat + first);
                    return;
                }
                sweeps(heatbath, overrelax, overrelax_last);
                if (fold)
                    k_overrelax_batched_last_final<T><<<n, 256, 0, st>>>(Bo, partials, results + (size_t)i * n_lat + first);
            });
            if ((s = cuda_check("mgq_update_sweeps_batched"))) return s;
        }
        if (plaq_out && n_or == 0) {
            uint64_t poff = 0;
            for (int first = 0; first < n_lat; first += BATCH_CHUNK) {
                const int n = (n_lat - first < BATCH_CHUNK) ? n_lat - first : BATCH_CHUNK;
                dispatch_prec(lats[0].prec, [&]<class T, int NP>() {
                    Batch<T> Bl;
                    fill_batch(Bl, lats, betas, first, n, 256, false);
                    k_plaquette_batched<T, NP><<<Bl.prefix[n], 256, 0, st>>>(Bl, partials + poff);
                    k_plaquette_batched_final<T><<<n, 256, 0, st>>>(Bl, partials + poff, results + (size_t)i * n_lat + first);
                    poff += (uint64_t)Bl.prefix[n];
                });
            }
            if ((s = cuda_check("mgq_update_sweeps_batched: plaquette"))) return s;
        }
    }
    if (plaq_out) return deliver(results, plaq_out, (size_t)n_sweeps * n_lat, st, "mgq_update_sweeps_batched");
    return MGQ_OK;
}

}  // extern "C"
