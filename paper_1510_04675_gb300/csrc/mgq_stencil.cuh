// Stencils shared by the libmgq kernels: the staple sum (Sec. III, Wilson
// action), the per-site plaquette sum, and the clover field strength.
#pragma once

#include "mgq_device.cuh"

namespace mgq {

// Rows 0 and 1 of op(a) op(b) (row 2 of the result is left unset): the callers
// rebuild it as conj(row0 x row1) because the product is in SU(3).  FP32: packed, or
// with single FMAs for FMA = true.
template <bool FMA, bool DA, bool DB> __device__ __forceinline__ M3<float> two_rows(const M3<float>& a, const M3<float>& b) {
    if constexpr (FMA) return fma_product<2, DA, DB>(a, b);
    else return x2_product<2, DA, DB>(a, b);
}
template <bool FMA = false> __device__ __forceinline__ M3<float> mul_nd_2(const M3<float>& a, const M3<float>& b) {
    return two_rows<FMA, false, true>(a, b);
}
template <bool FMA = false> __device__ __forceinline__ M3<float> mul_nn_2(const M3<float>& a, const M3<float>& b) {
    return two_rows<FMA, false, false>(a, b);
}
template <bool FMA = false> __device__ __forceinline__ M3<float> mul_dn_2(const M3<float>& a, const M3<float>& b) {
    return two_rows<FMA, true, false>(a, b);
}

// row 2 of a product of SU(3) factors, in either form
template <bool PACKED = false> __device__ __forceinline__ void complete(M3<float>& m) {
    if constexpr (PACKED) rebuild_row2_packed(m);
    else rebuild_row2(m);
}

// =============================================================== staple
// A_mu(x) = sum_{nu != mu} [ U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+
//                          + U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu) ]
// so that Re Tr(U_mu(x) A_mu(x)) sums the six plaquettes holding U_mu(x).
// x has parity par; x +- e_nu has parity 1 - par, x + e_mu - e_nu parity par.
//
// Staple in two-row form (FP32 links, 12- or 18-real); each half-term is added to A
// as it completes (A += up, A += dn), the order of staple_staged, so that staged and
// unstaged kernels agree bit for bit.  Each staple term is a product of three
// SU(3) links, hence in SU(3): only rows 0, 1 of every partial product are
// computed and row 2 is rebuilt, and a link that enters only through its rows
// (the left factor) is never completed.
//   up = (a b^+) c^+            a = U_nu(x+mu), b = U_mu(x+nu), c = U_nu(x)
//   dn = (e d)^+ f              d = U_nu(x+mu-nu), e = U_mu(x-nu), f = U_nu(x-nu)
template <class LinkField>
__device__ __forceinline__ M3<float> staple_two_row(const LinkField& U, const Geom& g, const int x[4], int h, int mu,
                                                int par) {
    M3<float> A;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) A.e[i][j] = mk(0.f, 0.f);
    const int op = par ^ 1;
    const Hops H = make_hops(g, x);
    const int fmu = pick(H.fwd, mu);
    const int hpm = (H.lex + fmu) >> 1;
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
        if (nu == mu) continue;
        const int hpn = (H.lex + H.fwd[nu]) >> 1;
        const int hmn = (H.lex + H.bwd[nu]) >> 1;
        const int hpm_mn = (H.lex + fmu + H.bwd[nu]) >> 1;
        M3<float> up, dn;
        {
            M3<float> t = mul_nd_2(U.load_rows(nu, op, hpm), U.template load<true>(mu, op, hpn));
            complete<true>(t);
            up = mul_nd_2(t, U.template load<true>(nu, par, h));
            complete<true>(up);
        }
        {
            M3<float> t = mul_nn_2(U.load_rows(mu, op, hmn), U.template load<true>(nu, par, hpm_mn));
            complete<true>(t);
            dn = mul_dn_2(t, U.template load<true>(nu, op, hmn));
            complete<true>(dn);
        }
        acc_add(A, up);
        acc_add(A, dn);
    }
    return A;
}

// ---- the two-row staple with its links staged through shared memory ----
// For FP32 12-real (paired) links.  The staple's six half-terms (the up and the
// down product of each direction nu != mu, in increasing nu) each need three
// links; the thread copies the links of half-term k+1 into its own
// shared-memory slots with cp.async while it computes half-term k from the
// other buffer, so those loads are in flight during the arithmetic without
// holding registers.  The updated link itself is staged with the first
// half-term and read back after the staple.  Each half-term is added to A as
// it completes (A += up, A += dn).  sm: (2 stages x 3 links + 1) x 3 pair-planes
// x STAGED_THREADS float4 (STAGED_SMEM bytes per block of STAGED_THREADS
// threads), each thread using its own column; the fixed block size keeps every
// slot address a constant offset from one base.
constexpr int STAGED_THREADS = 128;
constexpr int STAGED_SMEM = (2 * 3 + 1) * 3 * 16 * STAGED_THREADS;

__device__ __forceinline__ void cp_async16(float4* smem, const float4* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(__cvta_generic_to_global(gmem)) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// slot j of a stage (j = 0..2), or the updated link's slot (stage 2, j = 0)
__device__ __forceinline__ float4* staged_slot(float4* sm, int stage, int j, int k) {
    return sm + ((stage * 3 + j) * 3 + k) * STAGED_THREADS + threadIdx.x;
}
__device__ __forceinline__ void stage_link(float4* sm, int stage, int j, const Links<float, 6>& U, int mu, int par, int h) {
    const float4* q = reinterpret_cast<const float4*>(U.block(mu, par, h)) + (h & 31);
#pragma unroll
    for (int k = 0; k < 3; k++) cp_async16(staged_slot(sm, stage, j, k), q + (k << 5));
}
__device__ __forceinline__ M3<float> staged_rows(float4* sm, int stage, int j) {
    M3<float> m;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float4 v = *staged_slot(sm, stage, j, k);
        m.e[(2 * k) / 3][(2 * k) % 3] = mk(v.x, v.y);
        m.e[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk(v.z, v.w);
    }
    return m;
}
template <bool PACKED = false> __device__ __forceinline__ M3<float> staged_full(float4* sm, int stage, int j) {
    M3<float> m = staged_rows(sm, stage, j);
    complete<PACKED>(m);
    return m;
}
// the updated link staged by thread col of the block (slot (2, 0)), with the
// row 2 that thread wrote into its free slot (0, 2)
__device__ __forceinline__ M3<float> own_full_of(float4* sm, int col) {
    M3<float> m;
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float4 v = sm[((2 * 3 + 0) * 3 + k) * STAGED_THREADS + col];
        m.e[(2 * k) / 3][(2 * k) % 3] = mk(v.x, v.y);
        m.e[(2 * k + 1) / 3][(2 * k + 1) % 3] = mk(v.z, v.w);
    }
    const float4 r0 = sm[((0 * 3 + 2) * 3 + 0) * STAGED_THREADS + col];
    const float2 r1 = *reinterpret_cast<const float2*>(&sm[((0 * 3 + 2) * 3 + 1) * STAGED_THREADS + col]);
    m.e[2][0] = mk(r0.x, r0.y);
    m.e[2][1] = mk(r0.z, r0.w);
    m.e[2][2] = mk(r1.x, r1.y);
    return m;
}

// A = the staple of U_MU(x) (as staple_two_row, with the accumulation above);
// u = U_MU(x) (full, row 2 rebuilt).  MU may be a run-time direction; the
// sub-sweeps pass a compile-time one.
struct NoWork {
    __device__ void operator()() const {}
};
// early(): independent work that runs while the first loads are in flight; PACKED:
// the form of the row-2 rebuilds; FMA: that of a term's second product.  The first
// product of a term is packed, the second takes single FMAs: overrelaxation 44.5 ->
// 43.8 us per 32^4 launch, 16.0 -> 15.4 us at 24^4, against packed products throughout
// (single FMAs throughout 15.9 us at 24^4 but 50.3 us at 32^4).
template <bool PACKED = false, bool FMA = true, class Work = NoWork>
__device__ __forceinline__ M3<float> staple_staged(const Links<float, 6>& U, const Geom& g, const int x[4], int h,
                                                   const int MU, int par, float4* sm, M3<float>& u,
                                                   Work early = Work()) {
    const int op = par ^ 1;
    const Hops H = make_hops(g, x);
    const int fmu = pick(H.fwd, MU);
    const int hpm = (H.lex + fmu) >> 1;
    int hpn[3], hmn[3], hpm_mn[3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const int nu = i < MU ? i : i + 1;
        hpn[i] = (H.lex + pick(H.fwd, nu)) >> 1;
        hmn[i] = (H.lex + pick(H.bwd, nu)) >> 1;
        hpm_mn[i] = (H.lex + fmu + pick(H.bwd, nu)) >> 1;
    }
    // half-term k: nu = the (k/2)-th direction other than MU; even k: up = (a b^+) c^+
    // with a = U_nu(x+mu), b = U_mu(x+nu), c = U_nu(x); odd k: dn = (e d)^+ f with
    // d = U_nu(x+mu-nu), e = U_mu(x-nu), f = U_nu(x-nu)
    auto issue = [&](int k, int stage) {
        const int i = k >> 1, nu = i < MU ? i : i + 1;
        if ((k & 1) == 0) {
            stage_link(sm, stage, 0, U, nu, op, hpm);
            stage_link(sm, stage, 1, U, MU, op, hpn[i]);
            stage_link(sm, stage, 2, U, nu, par, h);
        } else {
            stage_link(sm, stage, 0, U, nu, par, hpm_mn[i]);
            stage_link(sm, stage, 1, U, MU, op, hmn[i]);
            stage_link(sm, stage, 2, U, nu, op, hmn[i]);
        }
    };
    stage_link(sm, 2, 0, U, MU, par, h);  // the updated link, with the first half-term
    issue(0, 0);
    cp_async_commit();
    issue(1, 1);
    cp_async_commit();
    early();
    M3<float> A;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) A.e[i][j] = mk(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 6; k++) {
        if (k < 5) cp_async_wait<1>();
        else cp_async_wait<0>();
        const int st = k & 1;
        M3<float> term;
        if ((k & 1) == 0) {
            const M3<float> t = mul_nd_2(staged_rows(sm, st, 0), staged_full<PACKED>(sm, st, 1));
            term = mul_nd_2<FMA>(t, staged_full<PACKED>(sm, st, 2));
        } else {
            M3<float> t = mul_nn_2(staged_rows(sm, st, 1), staged_full<PACKED>(sm, st, 0));
            complete<PACKED>(t);
            term = mul_dn_2<FMA>(t, staged_full<PACKED>(sm, st, 2));
        }
        complete<PACKED>(term);
        acc_add(A, term);
        if (k + 2 < 6) {
            issue(k + 2, st);
            cp_async_commit();
        }
    }
    u = staged_full<PACKED>(sm, 2, 0);
    return A;
}

// Full products, no use of unitarity (the FP64 parity path): the upper terms
// a (b^+ c^+) summed over nu, the lower terms d^+ (e^+ f) summed over nu, then
// added; the second product of each term accumulates onto the sum directly.
// Column k of every term needs column k of c^+ or f alone, which the kernels with
// one column per lane use (mgq_columns.cuh; same operations, same bits).
__device__ __forceinline__ M3<double> staple_full(const Links<double, 9>& U, const Geom& g, const int x[4], int h, int mu,
                                                  int par) {
    M3<double> A, D;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) A.e[i][j] = D.e[i][j] = mk(0.0, 0.0);
    const int op = par ^ 1;
    const Hops H = make_hops(g, x);
    const int fmu = pick(H.fwd, mu);
    const int hpm = (H.lex + fmu) >> 1;
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
        if (nu == mu) continue;
        const int hpn = (H.lex + H.fwd[nu]) >> 1;
        const M3<double> v = mul_dd(U.load(mu, op, hpn), U.load(nu, par, h));  // U_mu(x+nu)^+ U_nu(x)^+
        chain_product_add<false, false>(A, U.load(nu, op, hpm), v);            // U_nu(x+mu)
    }
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
        if (nu == mu) continue;
        const int hmn = (H.lex + H.bwd[nu]) >> 1;
        const int hpm_mn = (H.lex + fmu + H.bwd[nu]) >> 1;
        const M3<double> w = mul_dn(U.load(mu, op, hmn), U.load(nu, op, hmn));  // U_mu(x-nu)^+ U_nu(x-nu)
        chain_product_add<true, false>(D, U.load(nu, par, hpm_mn), w);          // U_nu(x+mu-nu)^+
    }
    acc_add(A, D);
    return A;
}

// FP32 (both formats): products of SU(3) factors in two-row form; FP64: full
// products.
template <class T, int NP>
__device__ __forceinline__ M3<T> staple(const Links<T, NP>& U, const Geom& g, const int x[4], int h, int mu, int par) {
    if constexpr (sizeof(T) == 4) return staple_two_row(U, g, x, h, mu, par);
    else return staple_full(U, g, x, h, mu, par);
}

// One upper term a b^+ c^+ and one lower term (e d)^+ f of the staple, the left factors'
// rows 0, 1 given: rows 0, 1 of every partial product, row 2 rebuilt; FMA as in two_rows.
template <bool FMA = false>
__device__ __forceinline__ M3<float> up_term(const M3<float>& a_rows, const M3<float>& b, const M3<float>& c) {
    M3<float> r = mul_nd_2<FMA>(mul_nd_2<FMA>(a_rows, b), c);
    rebuild_row2(r);
    return r;
}
template <bool FMA = false>
__device__ __forceinline__ M3<float> down_term(const M3<float>& e_rows, const M3<float>& d, const M3<float>& f) {
    M3<float> t = mul_nn_2<FMA>(e_rows, d);
    rebuild_row2(t);
    M3<float> r = mul_dn_2<FMA>(t, f);
    rebuild_row2(r);
    return r;
}

// =============================================================== plaquette
// Re Tr(a b^+) of a, b in SU(3) from their rows 0, 1: with s_ij = row_i(a) .
// conj(row_j(b)) it is s00 + s11 + conj(s00 s11 - s01 s10) (row 2 = conj(row0 x row1) and
// the Binet-Cauchy identity for the cross products).
__device__ __forceinline__ float retr_two_row(const M3<float>& a, const M3<float>& b) {
    Cx<float> sij[2][2];
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 2; j++)
            sij[i][j] = mulc(a.e[i][0], b.e[j][0]) + mulc(a.e[i][1], b.e[j][1]) + mulc(a.e[i][2], b.e[j][2]);
    const Cx<float> d = sij[0][0] * sij[1][1] - sij[0][1] * sij[1][0];
    return sij[0][0].re + sij[1][1].re + d.re;
}

// Per site: sum over mu < nu < ND of Re Tr[U_mu(x) U_nu(x+mu) (U_nu(x) U_mu(x+nu))^+]
// (ND = 4: all six planes; ND = 3: the planes of directions 0, 1, 2).
template <class T, int NP, int ND = 4>
__device__ __forceinline__ double site_plaquettes(const Links<T, NP>& U, const Geom& g, int par, int h) {
    int x[4];
    cb_coords(g, par, h, x);
    const int op = par ^ 1;
    const Hops H = make_hops(g, x);
    double acc = 0.0;
#pragma unroll
    for (int mu = 0; mu < ND - 1; mu++) {
        const int hpm = (H.lex + H.fwd[mu]) >> 1;
        if constexpr (sizeof(T) == 4) {
            // FP32: a = U_mu(x) U_nu(x+mu) and b = U_nu(x) U_mu(x+nu) are in SU(3)
            const M3<T> umu = U.load_rows(mu, par, h);
#pragma unroll
            for (int nu = mu + 1; nu < ND; nu++) {
                const int hpn = (H.lex + H.fwd[nu]) >> 1;
                const M3<T> a = mul_nn_2(umu, U.load(nu, op, hpm));
                const M3<T> b = mul_nn_2(U.load_rows(nu, par, h), U.load(mu, op, hpn));
                acc += (double)retr_two_row(a, b);
            }
        } else {
            const M3<T> umu = U.load(mu, par, h);
#pragma unroll
            for (int nu = mu + 1; nu < ND; nu++) {
                const int hpn = (H.lex + H.fwd[nu]) >> 1;
                const M3<T> a = mul_nn(umu, U.load(nu, op, hpm));
                const M3<T> b = mul_nn(U.load(nu, par, h), U.load(mu, op, hpn));
                acc += (double)retr_nd(a, b);
            }
        }
    }
    return acc;
}

// =============================================================== clover
// The three loops around the unit square of lines with sides A_mu, A_nu are
// written for a line field A_d(x) (the links, or products of m links) whose hops H
// are the lines' lengths; op is the parity one line away.

template <class T> __device__ __forceinline__ void acc_sub(M3<T>& a, const M3<T>& b) {
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) a.e[i][j] = a.e[i][j] - b.e[i][j];
}

// Clover leaves around x in the (mu,nu) plane, all starting and ending at x,
// counterclockwise; the algebra coefficients g of G = traceless part of
// (Q - Q^+)/8, i.e. g = t(TA(Q))/4.  TA(M^+) = -TA(M), so the leaves l1 and l4 that
// hold U_mu(x), and l2 and l3 that hold U_mu(x-mu), come in pairs with one product
// for that link:
//   l1 - l4^+ = U_mu(x) [U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+ - U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu)]
//   l2 - l3^+ = [U_nu(x) U_mu(x-mu+nu)^+ U_nu(x-mu)^+ - U_nu(x-nu)^+ U_mu(x-mu-nu)^+ U_nu(x-mu-nu)] U_mu(x-mu)
// ten products where four separate leaves take twelve.  All three rows are multiplied
// out: rows 0, 1 with row 2 = conj(row0 x row1) would be an eighth less work, but row 2
// then carries the roundings of the other two, and matrices off SU(3) another value.
template <class T, int NP>
__device__ __forceinline__ void clover_coeffs(const Links<T, NP>& U, const Hops& H, int par, int op, int mu, int nu, T out[8]) {
    const int fm = pick(H.fwd, mu), fn = pick(H.fwd, nu), bm = pick(H.bwd, mu), bn = pick(H.bwd, nu);
    const int x = H.lex;
    // a b^+ c^+ - (e d)^+ f
    auto sides = [](const M3<T>& a, const M3<T>& b, const M3<T>& c, const M3<T>& e, const M3<T>& d, const M3<T>& f) {
        M3<T> D = mul_nd(mul_nd(a, b), c);
        acc_sub(D, mul_dn(mul_nn(e, d), f));
        return D;
    };
    M3<T> Q = mul_nn(U.load(mu, par, x >> 1),
                     sides(U.load(nu, op, (x + fm) >> 1), U.load(mu, op, (x + fn) >> 1), U.load(nu, par, x >> 1),
                           U.load(mu, op, (x + bn) >> 1), U.load(nu, par, (x + fm + bn) >> 1), U.load(nu, op, (x + bn) >> 1)));
    acc_add(Q, mul_nn(sides(U.load(nu, par, x >> 1), U.load(mu, par, (x + bm + fn) >> 1), U.load(nu, op, (x + bm) >> 1),
                            U.load(mu, par, (x + bm + bn) >> 1), U.load(nu, op, (x + bn) >> 1), U.load(nu, par, (x + bm + bn) >> 1)),
                      U.load(mu, op, (x + bm) >> 1)));
    ta_coeffs(Q, out);
#pragma unroll
    for (int a = 0; a < 8; a++) out[a] *= T(0.25);
}

// The dual pairs of planes (01, 23), (02, 13), (03, 12): pair p's second plane.
__device__ __forceinline__ int dual_mu(int p) { return p == 0 ? 2 : 1; }
__device__ __forceinline__ int dual_nu(int p) { return p == 2 ? 2 : 3; }

// Re Tr of the loop A_mu(x) A_nu(x+mu) (A_nu(x) A_mu(x+nu))^+ of lines A.
template <class T, int NP>
__device__ __forceinline__ T loop_retr(const Links<T, NP>& U, const Hops& H, int par, int op, int mu, int nu) {
    const int x = H.lex >> 1, xm = (H.lex + pick(H.fwd, mu)) >> 1, xn = (H.lex + pick(H.fwd, nu)) >> 1;
    const M3<T> a = mul_nn(U.load(mu, par, x), U.load(nu, op, xm));
    return retr_nd(a, mul_nn(U.load(nu, par, x), U.load(mu, op, xn)));
}

// The plaquette of FP32 links in SU(3), as in site_plaquettes.
template <int NP>
__device__ __forceinline__ float plaquette_retr(const Links<float, NP>& U, const Hops& H, int par, int op, int mu, int nu) {
    const int x = H.lex >> 1, xm = (H.lex + pick(H.fwd, mu)) >> 1, xn = (H.lex + pick(H.fwd, nu)) >> 1;
    const M3<float> a = mul_nn_2<NP == 9>(U.load_rows(mu, par, x), U.load(nu, op, xm));
    return retr_two_row(a, mul_nn_2<NP == 9>(U.load_rows(nu, par, x), U.load(mu, op, xn)));
}

// =============================================================== SU(2) steps
// rows i, j of m <- R(r) rows i, j, restricted to the rows (do_i, do_j) and
// columns (bit masks ci, cj) that are read later; with the subgroup index a
// compile-time constant the unused updates vanish.
template <class T>
__device__ __forceinline__ void su2_rows(M3<T>& m, int i, int j, const T r[4], bool do_i, bool do_j, int ci, int cj) {
    const Cx<T> a = mk(r[0], r[3]), b = mk(r[2], r[1]), c = mk(-r[2], r[1]), d = mk(r[0], -r[3]);
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const Cx<T> mi = m.e[i][k], mj = m.e[j][k];
        if (do_i && ((ci >> k) & 1)) m.e[i][k] = a * mi + b * mj;
        if (do_j && ((cj >> k) & 1)) m.e[j][k] = c * mi + d * mj;
    }
}

// FP64: one column of the two rows as chains.
__device__ __forceinline__ void su2_pair(Cx<double>& mi, Cx<double>& mj, const double r[4]) {
    Cx<double> ni = cmul0(mk(r[0], r[3]), mi), nj = cmul0(mk(-r[2], r[1]), mi);
    cmac(ni, mk(r[2], r[1]), mj);
    cmac(nj, mk(r[0], -r[3]), mj);
    mi = ni;
    mj = nj;
}
template <>
__device__ __forceinline__ void su2_rows<double>(M3<double>& m, int i, int j, const double r[4], bool do_i, bool do_j,
                                                 int ci, int cj) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
        Cx<double> mi = m.e[i][k], mj = m.e[j][k];
        su2_pair(mi, mj, r);
        if (do_i && ((ci >> k) & 1)) m.e[i][k] = mi;
        if (do_j && ((cj >> k) & 1)) m.e[j][k] = mj;
    }
}

// FP32: a m_i + b m_j with a = r0 + i r3, b = r2 + i r1 (and c = -r2 + i r1,
// d = r0 - i r3 for row j) with single FMAs (32^4 overrelaxation launch 45.5 -> 45.1
// us against packed pairs, same bits).
template <>
__device__ __forceinline__ void su2_rows<float>(M3<float>& m, int i, int j, const float r[4], bool do_i, bool do_j,
                                                int ci, int cj) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const Cx<float> x = m.e[i][k], y = m.e[j][k];
        if (do_i && ((ci >> k) & 1)) {
            float re = __fmul_rn(r[0], x.re), im = __fmul_rn(r[0], x.im);
            re = __fmaf_rn(r[3], -x.im, re);
            im = __fmaf_rn(r[3], x.re, im);
            re = __fmaf_rn(r[2], y.re, re);
            im = __fmaf_rn(r[2], y.im, im);
            re = __fmaf_rn(r[1], -y.im, re);
            im = __fmaf_rn(r[1], y.re, im);
            m.e[i][k] = mk(re, im);
        }
        if (do_j && ((cj >> k) & 1)) {
            float re = __fmul_rn(-r[2], x.re), im = __fmul_rn(-r[2], x.im);
            re = __fmaf_rn(r[1], -x.im, re);
            im = __fmaf_rn(r[1], x.re, im);
            re = __fmaf_rn(r[0], y.re, re);
            im = __fmaf_rn(r[0], y.im, im);
            re = __fmaf_rn(-r[3], -y.im, re);
            im = __fmaf_rn(-r[3], y.re, im);
            m.e[j][k] = mk(re, im);
        }
    }
}

// The same as packed FMAs on (re, im) pairs.
__device__ __forceinline__ void su2_rows_packed(M3<float>& m, int i, int j, const float r[4], bool do_i, bool do_j, int ci,
                                                int cj) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const float2 MI = make_float2(m.e[i][k].re, m.e[i][k].im), iMI = make_float2(-m.e[i][k].im, m.e[i][k].re);
        const float2 MJ = make_float2(m.e[j][k].re, m.e[j][k].im), iMJ = make_float2(-m.e[j][k].im, m.e[j][k].re);
        if (do_i && ((ci >> k) & 1)) {
            float2 v = __fmul2_rn(bcast(r[0]), MI);
            v = __ffma2_rn(bcast(r[3]), iMI, v);
            v = __ffma2_rn(bcast(r[2]), MJ, v);
            v = __ffma2_rn(bcast(r[1]), iMJ, v);
            m.e[i][k] = from_f2(v);
        }
        if (do_j && ((cj >> k) & 1)) {
            float2 v = __fmul2_rn(bcast(-r[2]), MI);
            v = __ffma2_rn(bcast(r[1]), iMI, v);
            v = __ffma2_rn(bcast(r[0]), MJ, v);
            v = __ffma2_rn(bcast(-r[3]), iMJ, v);
            m.e[j][k] = from_f2(v);
        }
    }
}

template <bool PACKED, class T>
__device__ __forceinline__ void su2_rows_as(M3<T>& m, int i, int j, const T r[4], bool do_i, bool do_j, int ci, int cj) {
    if constexpr (PACKED && sizeof(T) == 4) su2_rows_packed(m, i, j, r, do_i, do_j, ci, cj);
    else su2_rows(m, i, j, r, do_i, do_j, ci, cj);
}
// V = U A
template <bool PACKED, class T> __device__ __forceinline__ M3<T> link_times_staple(const M3<T>& u, const M3<T>& A) {
    if constexpr (PACKED && sizeof(T) == 4) return x2_product<3, false, false>(u, A);
    else return mul_nn(u, A);
}

// After the update of subgroup s: U needs rows 0, 1 (the final
// reunitarisation rebuilds row 2) and, until s = 2, row 2 as an input; V only
// needs the entries the later subgroups read (s = 1 reads row 0 and
// V20, V22, s = 2 reads V11, V12, V21, V22).
template <bool PACKED = false, class T>
__device__ __forceinline__ void apply_subgroup(M3<T>& u, M3<T>& v, int s, const T R[4]) {
    if (s == 0) {
        su2_rows_as<PACKED>(u, 0, 1, R, true, true, 7, 7);
        su2_rows_as<PACKED>(v, 0, 1, R, true, true, 7, 6);
    } else if (s == 1) {
        su2_rows_as<PACKED>(u, 0, 2, R, true, true, 7, 7);
        su2_rows_as<PACKED>(v, 0, 2, R, false, true, 0, 6);
    } else {
        su2_rows_as<PACKED>(u, 1, 2, R, true, false, 7, 0);
    }
}

// Creutz's a0 and the direction (cos phi, sin phi), phi = 2 pi u3.  FP64 uses
// the accurate library functions (the oracle's operations); FP32 uses the
// hardware exponential, logarithm and sine/cosine where their absolute error
// (~1e-6) is harmless, and the accurate forms near their ill-conditioned ends.
__device__ __forceinline__ double creutz_a0(double k, double em, double u0) { return 1.0 + log1p((1.0 - u0) * em) / k; }
__device__ __forceinline__ float creutz_a0(float k, float em, float u0) {
    const float y = (1.f - u0) * em;
    return 1.f + (y < -0.1f ? __logf(1.f + y) : log1pf(y)) * __frcp_rn(k);
}
__device__ __forceinline__ double creutz_k(double beta, double xi) { return xi * (beta * (2.0 / 3.0)); }
__device__ __forceinline__ float creutz_k(float beta, float xi) { return xi * (beta * 0.666666667f); }
__device__ __forceinline__ double recip(double x) { return 1.0 / x; }
__device__ __forceinline__ float recip(float x) { return __frcp_rn(x); }
// sqrt of a positive argument (both uses above are > 0: rest >= u1^2 > 0 and
// |cos theta| < 1); FP32 takes x rsqrt(x)
__device__ __forceinline__ double sampler_sqrt(double x) { return sqrt(x); }
__device__ __forceinline__ float sampler_sqrt(float x) { return x * rsqrtf(x); }
__device__ __forceinline__ double creutz_em(double k) { return expm1(-2.0 * k); }
__device__ __forceinline__ float creutz_em(float k) { return k > 0.25f ? __expf(-2.f * k) - 1.f : expm1f(-2.f * k); }
__device__ __forceinline__ void creutz_phi(double u3, double* s, double* c) { sincospi(2.0 * u3, s, c); }
__device__ __forceinline__ void creutz_phi(float u3, float* s, float* c) {
    // 2 pi u3 - pi lies in (-pi, pi), where __sincosf is accurate; shift back by pi
    float sn, cs;
    __sincosf(fmaf(6.28318530718f, u3, -3.14159265359f), &sn, &cs);
    *s = -sn;
    *c = -cs;
}

// =============================================================== heat bath
// One link: V = U A; per subgroup (0,1), (0,2), (1,2): w from the block,
// k = 2 beta |w| / 3, up to n_hb Creutz attempts
//   a0 = 1 + log1p((1 - u0) expm1(-2k)) / k, accept iff u1^2 <= 1 - a0^2,
// direction cos(theta) = 2 u2 - 1, phi = 2 pi u3; R = X (w/|w|), U <- R U,
// V <- R V; reunitarise at the end.  dec[s] = accepted attempt or 255.

// |w|^2 of a subgroup's quaternion (FP64: a fixed chain)
template <class T> __device__ __forceinline__ T quat_norm2(const T w[4]) {
    return w[0] * w[0] + w[1] * w[1] + w[2] * w[2] + w[3] * w[3];
}
template <> __device__ __forceinline__ double quat_norm2<double>(const double w[4]) {
    return fma_rn(w[3], w[3], fma_rn(w[2], w[2], fma_rn(w[1], w[1], __dmul_rn(w[0], w[0]))));
}

// The direction of X from words z, w of a draw: cos, sin of theta and of phi.
template <class T> __device__ __forceinline__ void creutz_direction(uint4 r, T* ct, T* st, T* sp, T* cp) {
    const T u2 = u01<T>(r.z), u3 = u01<T>(r.w);
    *ct = T(2) * u2 - T(1);
    *st = sampler_sqrt(sub_rn(T(1), mul_rn(*ct, *ct)));
    creutz_phi(u3, sp, cp);
}

// One Creutz attempt from words x, y of its draw and its direction: R = X (w/|w|) and
// true on acceptance.
template <class T>
__device__ __forceinline__ bool creutz_rotation(const T w[4], T xi, T k, T em, uint32_t wx, uint32_t wy, T ct, T st, T sp, T cp,
                                                T R[4]) {
    const T u0 = u01<T>(wx), u1 = u01<T>(wy);
    const T a0 = creutz_a0(k, em, u0);
    const T rest = sub_rn(T(1), mul_rn(a0, a0));
    if (!(mul_rn(u1, u1) <= rest)) return false;
    const T rad = sampler_sqrt(rest);
    const T X[4] = {a0, rad * st * cp, rad * st * sp, rad * ct};
    const T inv = recip(xi);
    const T wh[4] = {w[0] * inv, w[1] * inv, w[2] * inv, w[3] * inv};
    qmul(X, wh, R);
    return true;
}

// The same with the four words r.
template <class T>
__device__ __forceinline__ bool creutz_draw(const T w[4], T xi, T k, T em, uint4 r, T R[4]) {
    const T u0 = u01<T>(r.x), u1 = u01<T>(r.y);
    const T a0 = creutz_a0(k, em, u0);
    const T rest = sub_rn(T(1), mul_rn(a0, a0));
    if (!(mul_rn(u1, u1) <= rest)) return false;
    const T rad = sampler_sqrt(rest);
    T ct, st, sp, cp;
    creutz_direction(r, &ct, &st, &sp, &cp);
    const T X[4] = {a0, rad * st * cp, rad * st * sp, rad * ct};
    const T inv = recip(xi);
    const T wh[4] = {w[0] * inv, w[1] * inv, w[2] * inv, w[3] * inv};
    qmul(X, wh, R);
    return true;
}

// the attempt on subgroup s, applied to u and v when accepted
template <bool PACKED = false, class T>
__device__ __forceinline__ bool creutz_attempt(M3<T>& u, M3<T>& v, int s, const T w[4], T xi, T k, T em, uint4 r) {
    T R[4];
    if (!creutz_draw(w, xi, k, em, r, R)) return false;
    apply_subgroup<PACKED>(u, v, s, R);
    return true;
}

// PACKED: the FP32 forms of V, the rotations and the rebuilds; the kernels that read
// their links straight into registers use it (24^4, 18-real: heat bath 24.4 us against
// 25.1 with single FMAs, overrelaxation 19.9 against 20.8), the staged ones and those
// with a term per warp do not.
template <bool PACKED = false, class T>
__device__ __forceinline__ void hb_link(M3<T>& u, const M3<T>& A, T beta, int n_hb, const RngKey& rk, uint32_t lex,
                                        uint32_t mu, uint8_t* dec) {
    M3<T> v = link_times_staple<PACKED>(u, A);
#pragma unroll
    for (int s = 0; s < 3; s++) {
        const int i = (s == 2) ? 1 : 0, j = (s == 0) ? 1 : 2;
        T w[4];
        block_w(v, i, j, w);
        const T xi = m_sqrt(quat_norm2(w));
        uint8_t d = 255;
        if (xi >= tiny_norm<T>()) {
            const T k = creutz_k(beta, xi);
            const T em = creutz_em(k);
            for (int att = 0; att < n_hb; att++) {
                if (creutz_attempt<PACKED>(u, v, s, w, xi, k, em, draw(rk, lex, mu, (uint32_t)s, (uint32_t)att, KIND_HB))) {
                    d = (uint8_t)att;
                    break;
                }
            }
        }
        if (dec) dec[s] = d;
    }
    reunitarize(u);
}

// The single-attempt heat bath with the three draws given (r[s]: subgroup s,
// attempt 0), so that a kernel can draw them while its loads are in flight.
template <class T>
__device__ __forceinline__ void hb_link_drawn(M3<T>& u, const M3<T>& A, T beta, const uint4 r[3]) {
    M3<T> v = mul_nn(u, A);
#pragma unroll
    for (int s = 0; s < 3; s++) {
        const int i = (s == 2) ? 1 : 0, j = (s == 0) ? 1 : 2;
        T w[4];
        block_w(v, i, j, w);
        const T xi = m_sqrt(quat_norm2(w));
        if (xi >= tiny_norm<T>()) {
            const T k = creutz_k(beta, xi);
            creutz_attempt(u, v, s, w, xi, k, creutz_em(k), r[s]);
        }
    }
    reunitarize(u);
}

// Overrelaxation's rotation (w/|w|)^2 = (w0^2 - |w_vec|^2, 2 w0 w_vec) / |w|^2;
// false when |w| is too small to divide by
template <class T> __device__ __forceinline__ bool or_rotation(const T w[4], T R[4]) {
    const T n2 = quat_norm2(w);
    if (!(m_sqrt(n2) >= tiny_norm<T>())) return false;
    const T inv2 = recip(n2);
    R[0] = (w[0] * w[0] - w[1] * w[1] - w[2] * w[2] - w[3] * w[3]) * inv2;
    R[1] = T(2) * w[0] * w[1] * inv2;
    R[2] = T(2) * w[0] * w[2] * inv2;
    R[3] = T(2) * w[0] * w[3] * inv2;
    return true;
}
// FP64, in fixed operations; |w| >= 1e-300 holds for every |w|^2 > 0
template <> __device__ __forceinline__ bool or_rotation<double>(const double w[4], double R[4]) {
    const double n2 = quat_norm2(w);
    if (!(n2 > 0.0)) return false;
    const double inv2 = 1.0 / n2, t = __dmul_rn(__dadd_rn(w[0], w[0]), inv2);
    const double v2 = fma_rn(w[3], w[3], fma_rn(w[2], w[2], __dmul_rn(w[1], w[1])));
    R[0] = __dmul_rn(fma_rn(w[0], w[0], -v2), inv2);
    R[1] = __dmul_rn(t, w[1]);
    R[2] = __dmul_rn(t, w[2]);
    R[3] = __dmul_rn(t, w[3]);
    return true;
}

// Overrelaxation of one link: per subgroup R = (w/|w|)^2; reunitarise.
template <bool PACKED = false, class T>
__device__ __forceinline__ void or_link(M3<T>& u, const M3<T>& A) {
    M3<T> v = link_times_staple<PACKED>(u, A);
#pragma unroll
    for (int s = 0; s < 3; s++) {
        const int i = (s == 2) ? 1 : 0, j = (s == 0) ? 1 : 2;
        T w[4], R[4];
        block_w(v, i, j, w);
        if (or_rotation(w, R)) apply_subgroup<PACKED>(u, v, s, R);
    }
    reunitarize(u);
}

}  // namespace mgq
