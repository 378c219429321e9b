// FP64 link updates with one matrix column per lane.
//
// An FP64 warp instruction occupies its SM sub-partition for 64 cycles on this
// part whatever lanes are active, so a launch is as fast as its longest chain of
// FP64 operations until there are warps for all 608 sub-partitions.  One thread
// per link takes about 2000 operations a link and needs 19456 links for that;
// smaller launches leave most of the chip idle behind the same chain.  Here a link
// is held by three lanes, one column each (LPL = 3), or by six, the upper and the
// lower staple terms apart (LPL = 6):
//   - column k of an upper term a (b^+ c^+) needs column k of c^+ only, of a lower
//     term d^+ (e^+ f) column k of f, and column k of V = U A column k of A: 18
//     complex multiply-adds a term and lane, no exchange (LPL = 6: one addition of
//     the two halves);
//   - the SU(2) rotations act on rows i, j of every column alike; the lanes
//     exchange the four entries of V's block, and the rotation's scalars are
//     computed by all lanes of a link;
//   - the reunitarisation exchanges norms, inner products and row entries.
// One compound sweep (1 heat bath + 4 overrelaxation) of 8^4: 3.75 -> 0.90 ms (an
// overrelaxation launch 94 -> 20 us, a heat bath 118 -> 38 us).
// Every operation and its order are those of the one-thread form (staple_full,
// hb_link, or_link), so both agree bit for bit.
#pragma once

#include "mgq_force_out.cuh"
#include "mgq_stencil.cuh"

namespace mgq {

// One warp per block: the blocks then spread over the SMs one warp at a time (8^4: 410
// warps, three to an SM, where blocks of four fill 103 SMs; four warps of an SM share
// its FP64 rate, 76 cycles an operation each instead of 64): 8^4 compound sweep 0.94 ->
// 0.90 ms, 10-step trajectory on 8^3x12 1.28 -> 1.18 ms.
constexpr int COL_THREADS = 32;

// the lanes of a link: k the lane's column, half its staple terms (0 upper, 1
// lower) when LPL = 6, base the lane of column 0 in its half
template <int LPL>
struct ColumnLane {
    static constexpr int kPerWarp = 32 / LPL;  // links per warp; 2 idle lanes
    static constexpr int kPerBlock = (COL_THREADS / 32) * kPerWarp;
    int grp, k, half, base;
    bool active;
    __device__ __forceinline__ ColumnLane() {
        const int lane = threadIdx.x & 31, sub = lane % LPL;
        grp = lane / LPL;
        active = grp < kPerWarp;  // the two lanes left over repeat the last link and store nothing
        if (!active) grp = kPerWarp - 1;
        half = sub / 3;
        k = sub - 3 * half;
        base = lane - k;
    }
    __device__ __forceinline__ int item(int block) const {
        return (block * (COL_THREADS / 32) + (threadIdx.x >> 5)) * kPerWarp + grp;
    }
};

__device__ __forceinline__ Cx<double> shfl_cx(Cx<double> v, int lane) {
    return mk(__shfl_sync(0xffffffffu, v.re, lane), __shfl_sync(0xffffffffu, v.im, lane));
}
// v with the sign of im turned for mask = 0x80000000
__device__ __forceinline__ Cx<double> flip_im(Cx<double> v, int mask) {
    return mk(v.re, __hiloint2double(__double2hiint(v.im) ^ mask, __double2loint(v.im)));
}
__device__ __forceinline__ Cx<double> elem(const Cx<double>* link, int e) { return ldg_cx(link + (e << 5)); }

// A += column k of one staple term: upper (dn = 0) or lower (dn = 1), direction
// nu; the same loads and operations either way, with the element order and the
// conjugations of the factors chosen per lane
__device__ __forceinline__ void staple_column_term(const Links<double, 9>& U, const Hops& H, int h, int mu, int nu, int par,
                                                   int dn, int k, Cx<double> A[3]) {
    const int op = par ^ 1, fmu = pick(H.fwd, mu);
    const int hn = (H.lex + (dn ? pick(H.bwd, nu) : pick(H.fwd, nu))) >> 1;             // x -+ nu
    const int ha = (H.lex + fmu + (dn ? pick(H.bwd, nu) : 0)) >> 1;                     // x + mu (- nu)
    const Cx<double>* m1 = U.base(mu, op, hn);                                          // b or e
    const Cx<double>* xs = dn ? U.base(nu, op, hn) : U.base(nu, par, h);                // f or c
    const Cx<double>* m2 = dn ? U.base(nu, par, ha) : U.base(nu, op, ha);               // d or a
    const int cflip = dn ? 0 : (int)0x80000000, dflip = dn ? (int)0x80000000 : 0;
    Cx<double> x[3], v[3];
#pragma unroll
    for (int l = 0; l < 3; l++) x[l] = flip_im(elem(xs, dn ? 3 * l + k : 3 * k + l), cflip);
#pragma unroll
    for (int j = 0; j < 3; j++)
        v[j] = dot3(conjg(elem(m1, j)), x[0], conjg(elem(m1, 3 + j)), x[1], conjg(elem(m1, 6 + j)), x[2]);
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) cmac(A[i], flip_im(elem(m2, dn ? 3 * j + i : 3 * i + j), dflip), v[j]);
}

// column k of the staple of U_mu(x) (as staple_full)
template <int LPL>
__device__ __forceinline__ void staple_column(const Links<double, 9>& U, const Geom& g, const int x[4], int h, int mu, int par,
                                              const ColumnLane<LPL>& c, Cx<double> A[3]) {
    const Hops H = make_hops(g, x);
    Cx<double> D[3];
#pragma unroll
    for (int i = 0; i < 3; i++) A[i] = D[i] = mk(0.0, 0.0);
#pragma unroll
    for (int n = 0; n < 3; n++) {
        const int nu = n < mu ? n : n + 1;
        if constexpr (LPL == 6) {
            staple_column_term(U, H, h, mu, nu, par, c.half, c.k, A);
        } else {
            staple_column_term(U, H, h, mu, nu, par, 0, c.k, A);
            staple_column_term(U, H, h, mu, nu, par, 1, c.k, D);
        }
    }
#pragma unroll
    for (int i = 0; i < 3; i++) {
        if constexpr (LPL == 6) D[i] = shfl_cx(A[i], c.base + c.k + (c.half ? -3 : 3));
        A[i] = A[i] + D[i];
    }
}

// column k of V = U A, and column k of U into u
__device__ __forceinline__ void left_column(const Cx<double>* link, const Cx<double> A[3], int k, Cx<double> u[3], Cx<double> v[3]) {
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const Cx<double> a = elem(link, 3 * i), b = elem(link, 3 * i + 1), c = elem(link, 3 * i + 2);
        v[i] = dot3(a, A[0], b, A[1], c, A[2]);
        u[i] = k == 0 ? a : (k == 1 ? b : c);
    }
}

// block_w of V's (i, j) block, V held by columns in the lanes from base on
__device__ __forceinline__ void column_block_w(const Cx<double> v[3], int i, int j, int base, double w[4]) {
    const Cx<double> vii = shfl_cx(v[i], base + i), vji = shfl_cx(v[j], base + i);
    const Cx<double> vij = shfl_cx(v[i], base + j), vjj = shfl_cx(v[j], base + j);
    w[0] = 0.5 * (vii.re + vjj.re);
    w[1] = -0.5 * (vij.im + vji.im);
    w[2] = 0.5 * (vji.re - vij.re);
    w[3] = 0.5 * (vjj.im - vii.im);
}

// reunitarize<double> with one column per lane
__device__ __forceinline__ void column_reunitarize(Cx<double> u[3], int k, int base) {
    auto sum = [&](double v) {
        return sum3(__shfl_sync(0xffffffffu, v, base), __shfl_sync(0xffffffffu, v, base + 1),
                    __shfl_sync(0xffffffffu, v, base + 2));
    };
    u[0] = scale(u[0], inv_norm(sum(norm2_rn(u[0]))));
    const Cx<double> q = cmul0(u[1], conjg(u[0]));
    const Cx<double> mip = mk(-sum(q.re), -sum(q.im));
    cmac(u[1], mip, u[0]);
    u[1] = scale(u[1], inv_norm(sum(norm2_rn(u[1]))));
    const int p = base + (k + 1) % 3, r = base + (k + 2) % 3;
    const Cx<double> r0p = shfl_cx(u[0], p), r0q = shfl_cx(u[0], r), r1p = shfl_cx(u[1], p), r1q = shfl_cx(u[1], r);
    u[2] = cross_conj(r0p, r0q, r1p, r1q);
}

// One (mu, par) sub-sweep.  HB: the heat bath of hb_link, else overrelaxation; with
// partials != nullptr (the direction-3 sub-sweeps that end an overrelaxation
// sweep) also the plaquettes of k_overrelax_last, lane k taking plane k of
// (0,1), (0,2), (1,2), summed per block.
// The links are those of block `block` of the lattice; partial receives the block's sum.
template <bool HB, int LPL>
__device__ __forceinline__ void update_columns(const Links<double, 9>& U, const Geom& g, int block, int mu, int par, double beta,
                                               const RngKey& rk, int n_hb, uint8_t* dec, double* partial) {
    const ColumnLane<LPL> c;
    const int h0 = c.item(block);
    const bool live = c.active && h0 < g.Vh && c.half == (LPL == 6 ? 1 : 0);  // the lanes that end with U
    const int h = h0 < g.Vh ? h0 : g.Vh - 1;
    int x[4];
    cb_coords(g, par, h, x);
    const int lex = lex_of(g, x);
    // heat bath: lane k draws subgroup k's first attempt and its direction for all
    uint4 words;
    double ct, st, sp, cp;
    if constexpr (HB) {
        words = draw(rk, (uint32_t)lex, (uint32_t)mu, (uint32_t)c.k, 0u, KIND_HB);
        creutz_direction(words, &ct, &st, &sp, &cp);
    }
    pdl_wait();
    Cx<double> A[3], u[3], v[3];
    staple_column<LPL>(U, g, x, h, mu, par, c, A);
    left_column(U.base(mu, par, h), A, c.k, u, v);
    double acc = 0.0;
    if (!HB && par == 1) acc = c.k == 0 ? v[0].re : (c.k == 1 ? v[1].re : v[2].re);  // Re Tr(U A), kept by the update
    // six lanes: the lower half carries V through the rotations, the upper half U
    if (LPL == 6 && c.half == 0) {
#pragma unroll
        for (int i = 0; i < 3; i++) u[i] = v[i];
    }
    const int vbase = c.base - 3 * c.half;
#pragma unroll
    for (int s = 0; s < 3; s++) {
        const int i = (s == 2) ? 1 : 0, j = (s == 0) ? 1 : 2;
        double w[4], R[4];
        column_block_w(LPL == 6 ? u : v, i, j, vbase, w);
        bool turn = false;
        if constexpr (HB) {
            const double xi = m_sqrt(quat_norm2(w));
            const int src = vbase + s;  // the lane that drew for this subgroup
            const uint32_t wx = __shfl_sync(0xffffffffu, words.x, src), wy = __shfl_sync(0xffffffffu, words.y, src);
            const double cts = __shfl_sync(0xffffffffu, ct, src), sts = __shfl_sync(0xffffffffu, st, src),
                         sps = __shfl_sync(0xffffffffu, sp, src), cps = __shfl_sync(0xffffffffu, cp, src);
            uint8_t d = 255;
            if (xi >= tiny_norm<double>()) {
                const double k = creutz_k(beta, xi), em = creutz_em(k);
                turn = creutz_rotation(w, xi, k, em, wx, wy, cts, sts, sps, cps, R);
                if (turn) d = 0;
                for (int att = 1; att < n_hb && !turn; att++) {
                    turn = creutz_draw(w, xi, k, em, draw(rk, (uint32_t)lex, (uint32_t)mu, (uint32_t)s, (uint32_t)att, KIND_HB), R);
                    if (turn) d = (uint8_t)att;
                }
            }
            if (dec && live && c.k == 0) dec[((size_t)lex * 4 + mu) * 3 + s] = d;
        } else {
            turn = or_rotation(w, R);
        }
        if (turn) {
            su2_pair(u[i], u[j], R);
            if (LPL == 3 && s < 2) su2_pair(v[i], v[j], R);
        }
    }
    column_reunitarize(u, c.k, c.base);
    // only now: blocks of the next launch that settle while these run find their
    // places on the idle SMs, two and three deep, and then run at half the rate
    pdl_launch_dependents();
    if (live) {
        Cx<double>* b = U.base(mu, par, h);
#pragma unroll
        for (int i = 0; i < 3; i++) b[(3 * i + c.k) << 5] = u[i];
    }
    if (partial) {
        if (live) {
            const int a = c.k == 2 ? 1 : 0, b = c.k == 0 ? 1 : 2;
            const int ha = lex_hop(g, x, a, +1) >> 1, hb = lex_hop(g, x, b, +1) >> 1;
            const M3<double> p = mul_nn(U.load(a, par, h), U.load(b, par ^ 1, ha));
            acc += retr_nd(p, mul_nn(U.load(b, par, h), U.load(a, par ^ 1, hb)));
        } else {
            acc = 0.0;
        }
        acc = block_sum(acc);
        if (threadIdx.x == 0) *partial = acc;
    }
}

template <bool HB, int LPL>
__global__ void __launch_bounds__(COL_THREADS) k_update_columns(Links<double, 9> U, Geom g, int mu, int par, double beta, RngKey rk,
                                                                int n_hb, uint8_t* __restrict__ dec, double* __restrict__ partials) {
    update_columns<HB, LPL>(U, g, blockIdx.x, mu, par, beta, rk, n_hb, dec, partials ? partials + blockIdx.x : nullptr);
}

// The force of every link (as k_force), block row y the (mu, parity) plane.  With M = U A by columns, lane k holds M_nk of the pair (k, n),
// n = k + 1 mod 3, and gets M_kn: two coefficients each, the diagonal ones by all.
template <int LPL, class Out>
__global__ void __launch_bounds__(COL_THREADS) k_force_columns(Links<double, 9> U, Geom g, Out out) {
    const ColumnLane<LPL> c;
    const int mu = blockIdx.y >> 1, par = blockIdx.y & 1, h0 = c.item(blockIdx.x), h = h0 < g.Vh ? h0 : g.Vh - 1;
    int x[4];
    cb_coords(g, par, h, x);
    pdl_wait();
    if (out.idle()) return;
    Cx<double> A[3], u[3], v[3];
    staple_column<LPL>(U, g, x, h, mu, par, c, A);
    left_column(U.base(mu, par, h), A, c.k, u, v);
    // v = column k of M.  Entry (k, n) sits in lane n, row k; lane n serves its
    // predecessor k = n - 1, so each lane offers the entry of that row
    const Cx<double> offer = c.k == 0 ? v[2] : (c.k == 1 ? v[0] : v[1]);
    const Cx<double> got = shfl_cx(offer, c.base + (c.k + 1) % 3);
    const Cx<double> has = c.k == 0 ? v[1] : (c.k == 1 ? v[2] : v[0]);
    const double dk = c.k == 0 ? v[0].im : (c.k == 1 ? v[1].im : v[2].im);
    const double d0 = __shfl_sync(0xffffffffu, dk, c.base), d1 = __shfl_sync(0xffffffffu, dk, c.base + 1),
                 d2 = __shfl_sync(0xffffffffu, dk, c.base + 2);
    pdl_launch_dependents();
    if (!c.active || h0 >= g.Vh || c.half) return;
    const double re = c.k == 2 ? has.re - got.re : got.re - has.re;  // t_1, t_6, t_4 = Re(M_ij - M_ji), i < j
    const double diag = c.k == 0 ? d0 - d1 : (d0 + d1 - 2.0 * d2) * 0.57735026918962576451;
    const int a = c.k == 0 ? 0 : (c.k == 1 ? 5 : 3);  // pairs 01, 12, 02
    out.put_one(mu, par, h, a, has.im + got.im);
    out.put_one(mu, par, h, a + 1, re);
    if (c.k < 2) out.put_one(mu, par, h, c.k == 0 ? 2 : 7, diag);
}

// Lanes per link (1: a thread for each; 3; 6) of a launch over n links, from the
// FP64 operations of a link's chain per lane and the warps that share one of the
// 608 sub-partitions: whichever ends first.
inline int lanes_per_link(long n, long ops1, long ops3, long ops6) {
    constexpr long kPartitions = 152 * 4;
    auto cost = [](long warps, long ops) { return (warps + kPartitions - 1) / kPartitions * ops; };
    const long one = cost((n + 31) / 32, ops1), three = cost((n + 9) / 10, ops3), six = cost((n + 4) / 5, ops6);
    return one <= three && one <= six ? 1 : (three <= six ? 3 : 6);
}
// a sub-sweep's link: staple 1296 and 108 of products, about 500 for V, the rotations
// and the reunitarisation; by columns about 300 of those, half the rotations' in six lanes
inline int update_lanes(long n) { return lanes_per_link(n, 1900, 740, 450); }
// the force's link: staple and product
inline int force_lanes(long n) { return lanes_per_link(n, 1420, 490, 275); }

}  // namespace mgq
