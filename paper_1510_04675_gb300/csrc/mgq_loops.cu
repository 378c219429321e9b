// libmgq Wilson loops and rethermalisation diagnostics (Sec. III: Wilson
// lines and m x n loops, partial plaquettes W^{1x1}_d, displaced loops
// W^{2x2}_d; Sec. IV.C: smoothness s_p = N_c [1 - W^{1x1}_p] and
// h = max_p s_p).  Measurement kernels: one thread per site, FP64 sums.
#include "mgq_internal.h"
#include "mgq_stencil.cuh"

namespace mgq {

// P <- P times the `len` links in direction mu from the site (lexicographic index
// lex, coordinate c along mu, parity par) on, which move along.
template <class T, int NP>
__device__ __forceinline__ void extend_line(M3<T>& P, const Links<T, NP>& U, int mu, int len, int L, int stride, int& lex,
                                            int& c, int& par) {
    for (int k = 0; k < len; k++) {
        P = mul_nn(P, U.load(mu, par, lex >> 1));
        const bool last = ++c == L;
        lex += last ? stride * (1 - L) : stride;
        if (last) c = 0;
        par ^= 1;
    }
}

// L^m_mu(x) L^n_nu(x + m mu): the path along mu, then nu
template <class T, int NP>
__device__ __forceinline__ M3<T> corner_path(const Links<T, NP>& U, const Geom& g, const int x[4], int par, int mu, int m, int nu,
                                             int n) {
    const int st[4] = {1, g.L[0], g.L[0] * g.L[1], g.L[0] * g.L[1] * g.L[2]};
    const int smu = pick(st, mu), Lmu = pick(g.L, mu);
    int lex = lex_of(g, x), c = pick(x, mu);
    M3<T> P = U.load(mu, par, lex >> 1);
    const bool last = ++c == Lmu;
    lex += last ? smu * (1 - Lmu) : smu;
    if (last) c = 0;
    par ^= 1;
    extend_line(P, U, mu, m - 1, Lmu, smu, lex, c, par);
    c = pick(x, nu);
    extend_line(P, U, nu, n, pick(g.L, nu), pick(st, nu), lex, c, par);
    return P;
}

__device__ __forceinline__ int plane_mu(int p) { return p < 3 ? 0 : (p < 5 ? 1 : 2); }
__device__ __forceinline__ int plane_nu(int p) { return p < 3 ? p + 1 : (p < 5 ? p - 1 : 3); }

// Re Tr L^m_mu(x) L^n_nu(x+m mu) [L^n_nu(x) L^m_mu(x+n nu)]^+, one thread per site
// and plane (block row y): two paths of m + n links, all rows multiplied out (2x3 loops
// of 24^3x48, FP32 12-real, a call: 383 us with a thread for a site's six planes, 296
// us so; 209 us with rows 0, 1 of the paths only, which added 10 to 30 % to the rounding
// error of the loops)
template <class T, int NP>
__global__ void __launch_bounds__(128) k_wilson_loop(Links<T, NP> U, Geom g, int m, int n, double* __restrict__ partials) {
    const int mu = plane_mu(blockIdx.y), nu = plane_nu(blockIdx.y);
    double acc = 0.0;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.V; idx += gridDim.x * blockDim.x) {
        const int par = idx >= g.Vh, h = idx - par * g.Vh;
        int x[4];
        cb_coords(g, par, h, x);
        const M3<T> a = corner_path(U, g, x, par, mu, m, nu, n), b = corner_path(U, g, x, par, nu, n, mu, m);
        acc += (double)retr_nd(a, b);
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.y * gridDim.x + blockIdx.x] = acc;
}

// 8 class sums of Re Tr (1x1 loops by chi_munu = 0..2, 2x2 loops by chi = 0..4) and
// the least Re Tr of the 1x1 loops: partials[q * nb + block] for q = 0..7, minima in
// partials[8 * nb + block], nb = gridDim.x * 6.  One thread per site and plane
// (block row y); U2 holds the lines of two links.  24^3x48, a call: FP32 12-real 634 us
// with the 2x2 loops multiplied out link by link and thirds taken in FP64 per loop, now
// 299 us, of which 40 us for the lines; 18-real 647 -> 326 us (538 us where the compiler
// is left to choose 96 registers).
template <class T, int NP>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 1 : 4) k_partial_loops(Links<T, NP> U, Links<T, 9> U2, Geom g, double* __restrict__ partials) {
    const int mu = plane_mu(blockIdx.y), nu = plane_nu(blockIdx.y);
    double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    T least = T(3);
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.V; idx += gridDim.x * blockDim.x) {
        const int par = idx >= g.Vh, h = idx - par * g.Vh;
        int x[4];
        cb_coords(g, par, h, x);
        const int chi = (x[0] & 1) + (x[1] & 1) + (x[2] & 1) + (x[3] & 1);
        const int cmn = chi - (pick(x, mu) & 1) - (pick(x, nu) & 1);
        const T w1 = loop_retr(U, make_hops(g, x), par, par ^ 1, mu, nu);
        const T w2 = loop_retr(U2, make_hops(g, x, 2), par, par, mu, nu);
        least = w1 < least ? w1 : least;
        // the sites of a warp mostly share their classes: one branch taken
#pragma unroll
        for (int d = 0; d < 3; d++)
            if (d == cmn) a[d] += (double)w1;
#pragma unroll
        for (int d = 0; d < 5; d++)
            if (d == chi) a[3 + d] += (double)w2;
    }
    const int nb = gridDim.x * gridDim.y, b = blockIdx.y * gridDim.x + blockIdx.x;
#pragma unroll
    for (int q = 0; q < 8; q++) {
        const double s = block_sum(a[q]);
        if (threadIdx.x == 0) partials[q * nb + b] = s;
    }
    // h's part 3 (1 - W) of a loop, W = Re Tr / 3, is largest where Re Tr is least
    __shared__ double smax[128];
    smax[threadIdx.x] = 3.0 * (1.0 - (double)least / 3.0);
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) partials[8 * nb + b] = smax[0];
}

struct LoopScales {
    double s[8];
};

// block q < 8: the q-th class sum times its scale; block 8: the maximum of the last set
__global__ void k_partial_final(const double* __restrict__ partials, int n, LoopScales sc, double* out) {
    const int q = blockIdx.x;
    partials += (size_t)q * n;
    if (q < 8) {
        double v = 0.0;
        for (int i = threadIdx.x; i < n; i += blockDim.x) v += partials[i];
        v = block_sum(v);
        if (threadIdx.x == 0) out[q] = v * sc.s[q];
        return;
    }
    __shared__ double sm[512];
    double m = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, partials[i]);
    sm[threadIdx.x] = m;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sm[threadIdx.x] = fmax(sm[threadIdx.x], sm[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) out[8] = sm[0];
}

static double binom(int n, int k) {
    double r = 1;
    for (int i = 1; i <= k; i++) r = r * (n - k + i) / i;
    return r;
}

}  // namespace mgq

using namespace mgq;

extern "C" {

mgq_status mgq_wilson_loop(const mgq_lattice* lat, int m, int n, double* out, void* stream) {
    Trace trace("mgq_wilson_loop");
    mgq_status s = check_lattice(lat, true, "mgq_wilson_loop");
    if (s) return s;
    if (m < 1 || n < 1 || m > 64 || n > 64) return fail(MGQ_EINVAL, "mgq_wilson_loop: need 1 <= m, n <= 64");
    if (!out) return fail(MGQ_EINVAL, "mgq_wilson_loop: out is NULL");
    const Geom g = make_geom(lat->dims);
    cudaStream_t st = as_stream(stream);
    const int nb = reduction_blocks(g.V, 128);  // at most 1184: 6 x 1184 partial sums
    dispatch_prec(lat->prec, [&]<class T, int NP>() {
        k_wilson_loop<T, NP><<<dim3(nb, 6), 128, 0, st>>>(links_of<T, NP>(lat), g, m, n, ws_partials(lat));
    });
    double* sc = ws_scalars(lat);
    launch_final_sum(ws_partials(lat), 6 * nb, 1.0 / (18.0 * (double)g.V), sc + 24, st);
    if ((s = cuda_check("mgq_wilson_loop"))) return s;
    return deliver(sc + 24, out, 1, st, "mgq_wilson_loop");
}

mgq_status mgq_partial_loops(const mgq_lattice* lat, double* out, void* stream) {
    Trace trace("mgq_partial_loops");
    mgq_status s = check_lattice(lat, true, "mgq_partial_loops");
    if (s) return s;
    if (!out) return fail(MGQ_EINVAL, "mgq_partial_loops: out is NULL");
    const Geom g = make_geom(lat->dims);
    cudaStream_t st = as_stream(stream);
    int nbx = reduction_blocks(g.V, 128);
    if (nbx > (int)(WS_NPARTIALS / 54)) nbx = (int)(WS_NPARTIALS / 54);
    const int nb = 6 * nbx;
    line_field(lat, 2, st);
    dispatch_prec(lat->prec, [&]<class T, int NP>() {
        k_partial_loops<T, NP><<<dim3(nbx, 6), 128, 0, st>>>(links_of<T, NP>(lat), links_at<T, 9>(ws_lines(lat), lat->dims), g,
                                                             ws_partials(lat));
    });
    double* sc = ws_scalars(lat);
    const double V = (double)g.V;
    LoopScales sc9;
    for (int d = 0; d < 3; d++) sc9.s[d] = 1.0 / (6.0 * (4 - d) * (3 - d) * binom(4, d) * V / 16.0);
    for (int d = 0; d < 5; d++) sc9.s[3 + d] = 1.0 / (18.0 * binom(4, d) * V / 16.0);
    k_partial_final<<<9, 512, 0, st>>>(ws_partials(lat), nb, sc9, sc + 24);
    if ((s = cuda_check("mgq_partial_loops"))) return s;
    return deliver(sc + 24, out, 9, st, "mgq_partial_loops");
}

}  // extern "C"
