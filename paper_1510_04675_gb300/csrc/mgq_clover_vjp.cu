// libmgq: gradients of the clover energy density E and charge Q (Sec. IV.B-C)
// with respect to the links, for the backward pass of flowed clover
// observables (the cotangent that the adjoint flow then pulls back).
//
// With g_p(x) = t(TA(Q_p(x)))/4 the algebra coefficients of the clover field
// strength of plane p at x (Q_p the four leaves), an observable O(g) has
// dO = sum_{x,p} c_p(x) . dg_p(x), c = dO/dg:
//   E = (1/V) sum_x 1/2 sum_p |g_p|^2           -> c_p = g_p / V
//   Q = 1/(8 pi^2) sum_x (g01.g23 - g02.g13 + g03.g12) -> c01 = g23/(8 pi^2), ...
// and dg = t(TA(dQ))/4, c . t(TA(N)) = -2 Re Tr(C N) (C = sum c_a X_a), so
// dO = -1/2 sum Re Tr(C_p(x) dQ_p(x)).  Each plaquette is a leaf of the clovers at
// its four corners, so it carries the four C of its corners, each inserted once.
// For a link m = U_rho(y) of it, traced from m as m X1 X2 X3 past the corners
// y, y1, y2, y3, the link's cotangent gets (variation U_m -> exp(e) U_m)
//   s/4 TA(m R),  R = C(y1) X1 X2 X3 + X1 C(y2) X2 X3 + X1 X2 C(y3) X3 + X1 X2 X3 C(y),
// s = +1 when that is the leaf's sense (a then b for plane a < b), -1 when it is
// the reverse, as C^+ = -C and TA(M^+) = -TA(M).
#include "mgq_internal.h"
#include "mgq_stencil.cuh"

namespace mgq {

// plane index of (a, b), a < b: 01 02 03 12 13 23
__host__ __device__ constexpr int plane_of(int a, int b) { return a == 0 ? b - 1 : (a == 1 ? b + 1 : 5); }

template <class T>
struct Planes6 {  // c_p(x): [p][parity][a][h] (scratch of this file only)
    T* p;
    int S;
    __device__ __forceinline__ T* at(int pl, int par, int h) const { return p + (size_t)(pl * 2 + par) * 8 * S + h; }
};

// Pass 1: c_p(x) for every site and plane, one thread per site and dual pair of
// planes (block row y).
template <class T, int NP>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 1 : 4) k_clover_cotangent(Links<T, NP> U, Geom g, int obs, Planes6<T> C) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x, p = blockIdx.y;
    if (idx >= g.V) return;
    const int par = idx >= g.Vh, h = idx - par * g.Vh;
    int x[4];
    cb_coords(g, par, h, x);
    const Hops H = make_hops(g, x);
    T Ga[8], Gb[8];
    clover_coeffs(U, H, par, par ^ 1, 0, p + 1, Ga);
    clover_coeffs(U, H, par, par ^ 1, dual_mu(p), dual_nu(p), Gb);
    // E: c = g / V; Q: c of a plane is +- g of its dual plane / (8 pi^2): 01<->23 (+), 02<->13 (-), 03<->12 (+)
    const T f = obs == 0 ? T(1) / (T)g.V : (p == 1 ? T(-1.0 / (8.0 * 9.869604401089358)) : T(1.0 / (8.0 * 9.869604401089358)));
    T* oa = C.at(p, par, h);
    T* ob = C.at(5 - p, par, h);
#pragma unroll
    for (int a = 0; a < 8; a++) {
        oa[(size_t)a * C.S] = f * (obs == 0 ? Ga[a] : Gb[a]);
        ob[(size_t)a * C.S] = f * (obs == 0 ? Gb[a] : Ga[a]);
    }
}

// the antihermitian C of plane pl at site (par, h)
template <class T> __device__ __forceinline__ M3<T> corner(const Planes6<T>& C, int pl, int par, int h) {
    T c[8];
    const T* p = C.at(pl, par, h);
#pragma unroll
    for (int q = 0; q < 8; q++) c[q] = p[(size_t)q * C.S];
    return alg_matrix(c);
}

// Pass 2: lam_m += scale * dO/de_m for every link m = U_rho(y): two plaquettes in each
// of three planes.  The product rule runs along the loop: with P = X1 X2 and
// S = P X3, R = C(y1) S + (X1 C(y2) X2 + P C(y3)) X3 + S C(y), and since every
// plaquette of a plane has the same C(y), the sum of s S takes it once per plane:
// 15 products a plane, where a gather over the 8 leaves of a plane that hold the
// link, each multiplied out on its own, took about 44 and as many link loads.  A
// plane's two sides run one after the other and the planes in a rolled loop, which
// keeps the live matrices in registers (16^4, FP32 12-real: 296 -> 70 us).
template <class T, int NP>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 1 : 3) k_clover_vjp(Links<T, NP> U, Geom g, Planes6<T> C, T scl, Alg<T> Lam) {
    const int rho = blockIdx.y >> 1, par = blockIdx.y & 1, op = par ^ 1, h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= g.Vh) return;
    int y[4];
    cb_coords(g, par, h, y);
    const Hops H = make_hops(g, y);
    const int frho = pick(H.fwd, rho), h1 = (H.lex + frho) >> 1;  // y + rho (op)
    M3<T> R;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) R.e[i][j] = mk(T(0), T(0));
#pragma unroll 1
    for (int K = 0; K < 3; K++) {
        const int nu = K < rho ? K : K + 1;
        const int pl = rho < nu ? plane_of(rho, nu) : plane_of(nu, rho);
        M3<T> Sd;  // s (S_up - S_dn) summed over the sides, and R's part of the plane
        M3<T> Rp;
        {
            const int h3 = (H.lex + pick(H.fwd, nu)) >> 1, h2 = (H.lex + frho + pick(H.fwd, nu)) >> 1;  // y + nu (op), y + rho + nu (par)
            const M3<T> X1 = U.load(nu, op, h1), X2d = U.load(rho, op, h3);
            const M3<T> P = mul_nd(X1, X2d);
            M3<T> Q = mul_nd(mul_nn(X1, corner(C, pl, par, h2)), X2d);
            acc_add(Q, mul_nn(P, corner(C, pl, op, h3)));
            const M3<T> X3d = U.load(nu, par, h);
            Rp = mul_nd(Q, X3d);
            Sd = mul_nd(P, X3d);
        }
        {
            const int bnu = pick(H.bwd, nu), h3 = (H.lex + bnu) >> 1, h2 = (H.lex + frho + bnu) >> 1;  // y - nu (op), y + rho - nu (par)
            const M3<T> Y1d = U.load(nu, par, h2), Y2d = U.load(rho, op, h3);
            const M3<T> P = mul_dd(Y1d, Y2d);
            M3<T> Q = mul_nd(mul_dn(Y1d, corner(C, pl, par, h2)), Y2d);
            acc_add(Q, mul_nn(P, corner(C, pl, op, h3)));
            const M3<T> Y3 = U.load(nu, op, h3);
            acc_sub(Rp, mul_nn(Q, Y3));
            acc_sub(Sd, mul_nn(P, Y3));
        }
        acc_add(Rp, mul_nn(corner(C, pl, op, h1), Sd));
        acc_add(Rp, mul_nn(Sd, corner(C, pl, par, h)));
        if (rho < nu) acc_add(R, Rp);
        else acc_sub(R, Rp);
    }
    T t[8];
    ta_coeffs(mul_nn(U.load(rho, par, h), R), t);
    T* out = Lam.at(rho, par, h);
    const T f = T(0.25) * scl;
#pragma unroll
    for (int q = 0; q < 8; q++) out[q * Alg<T>::kStep] += f * t[q];
}

static inline int nblk(long n, int t) { return (int)((n + t - 1) / t); }

uint64_t clover_vjp_scratch(const mgq_lattice* lat) {
    return round256(6ull * 2ull * 8ull * site_stride(lat->dims) * (lat->prec == MGQ_F64 ? 8 : 4));
}

}  // namespace mgq

using namespace mgq;

extern "C" {

uint64_t mgq_clover_vjp_scratch_bytes(const mgq_lattice* lat) {
    if (!lat || !links_bytes(lat)) return 0;
    return clover_vjp_scratch(lat);
}

mgq_status mgq_clover_vjp(const mgq_lattice* lat, int observable, double scale, void* lambda, void* scratch,
                          uint64_t scratch_bytes, void* stream) {
    Trace trace("mgq_clover_vjp");
    mgq_status s = check_lattice(lat, false, "mgq_clover_vjp");
    if (s) return s;
    if (observable != 0 && observable != 1) return fail(MGQ_EINVAL, "mgq_clover_vjp: observable must be 0 (E) or 1 (Q)");
    if (!lambda || ((uintptr_t)lambda & 15)) return fail(MGQ_EINVAL, "mgq_clover_vjp: lambda NULL or misaligned");
    if (!scratch || ((uintptr_t)scratch & 255)) return fail(MGQ_EINVAL, "mgq_clover_vjp: scratch NULL or not 256-byte aligned");
    if (scratch_bytes < clover_vjp_scratch(lat))
        return fail(MGQ_ENOMEM, "mgq_clover_vjp: scratch has %llu bytes, needs %llu", (unsigned long long)scratch_bytes,
                    (unsigned long long)clover_vjp_scratch(lat));
    const Geom g = make_geom(lat->dims);
    cudaStream_t st = as_stream(stream);
    dispatch_prec(lat->prec, [&]<class T, int NP>() {
        Planes6<T> C;
        C.p = reinterpret_cast<T*>(scratch);
        C.S = g.S;
        k_clover_cotangent<T, NP><<<dim3(nblk(g.V, 128), 3), 128, 0, st>>>(links_of<T, NP>(lat), g, observable, C);
        k_clover_vjp<T, NP><<<dim3(nblk(g.Vh, 128), 8), 128, 0, st>>>(links_of<T, NP>(lat), g, C, (T)scale,
                                                                   alg_at<T>(lambda, lat->dims));
    });
    return cuda_check("mgq_clover_vjp");
}

}  // extern "C"
