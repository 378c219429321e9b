// FP32 sub-sweeps of small lattices with a staple term per warp.
//
// A thread that does a whole link runs some 2000 instructions one after the other;
// a launch over fewer links than the chip has threads for is as slow as that chain
// and its six dependent rounds of loads.  Here a block of WARPS = 6 or 3 warps holds
// 32 links: the six half-terms of their staples (the upper or the lower product of
// one direction, all of its loads at once) are shared among the warps, left in
// shared memory, and warp 0 adds the six in staple_two_row's order and updates the
// links.  The products, the order of the additions and the update are those of the
// one-thread form, so both agree bit for bit.  FP32 12-real, heat bath and
// overrelaxation per launch: 8^4 6.6 and 3.8 -> 3.3 and 2.5 us, 12^4 8.0 and 6.3 -> 4.7
// and 3.7 us (six warps); 16^4 9.6 and 6.6 -> 6.7 and 6.0 us (three).
#pragma once

#include "mgq_stencil.cuh"

namespace mgq {

constexpr int TERMS_LINKS = 32;  // per block

// half-term w of the staple of U_mu(x), as in staple_two_row: direction w / 2 of
// those other than mu, upper (even w) or lower; FMA as in two_rows
template <bool FMA, int NP>
__device__ __forceinline__ M3<float> staple_half_term(const Links<float, NP>& U, const Hops& H, int mu, int par, int w) {
    const int op = par ^ 1, i = w >> 1, nu = i < mu ? i : i + 1;
    const int fmu = pick(H.fwd, mu);
    M3<float> r;
    if ((w & 1) == 0) {
        r = up_term<FMA>(U.load_rows(nu, op, (H.lex + fmu) >> 1), U.load(mu, op, (H.lex + pick(H.fwd, nu)) >> 1), U.load(nu, par, H.lex >> 1));
    } else {
        const int b = pick(H.bwd, nu), hmn = (H.lex + b) >> 1;
        r = down_term<FMA>(U.load_rows(mu, op, hmn), U.load(nu, par, (H.lex + fmu + b) >> 1), U.load(nu, op, hmn));
    }
    return r;
}

enum { TERMS_HEATBATH = 0, TERMS_OVERRELAX = 1, TERMS_OVERRELAX_LAST = 2 };

// One (mu, par) sub-sweep: the single-attempt heat bath (a subgroup's draws taken by
// each of warps 0 to 2 after its terms), overrelaxation, or the direction-3
// overrelaxation that also measures plaquettes as k_overrelax_last does (the planes
// of directions 0, 1, 2 shared among the warps from 1 on; one partial sum per block).
// The links are those of block `block` of the lattice; partial receives the block's sum.
template <int NP, int KIND, int WARPS, bool FMA>
__device__ __forceinline__ void update_terms(const Links<float, NP>& U, const Geom& g, int block, int mu, int par, float beta,
                                             const RngKey& rk, double* partial) {
    __shared__ float2 term[6][9][TERMS_LINKS];
    __shared__ uint4 words[3][TERMS_LINKS];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int h0 = block * TERMS_LINKS + lane, h = h0 < g.Vh ? h0 : g.Vh - 1;
    int x[4];
    cb_coords(g, par, h, x);
    const Hops H = make_hops(g, x);
    pdl_wait();
    M3<float> u;
    if (w == 0) u = U.load(mu, par, h);
#pragma unroll 1
    for (int k = w * (6 / WARPS); k < (w + 1) * (6 / WARPS); k++) {
        const M3<float> t = staple_half_term<FMA>(U, H, mu, par, k);
#pragma unroll
        for (int e = 0; e < 9; e++) term[k][e][lane] = make_float2(t.e[e / 3][e % 3].re, t.e[e / 3][e % 3].im);
    }
    if (KIND == TERMS_HEATBATH && w < 3)
        words[w][lane] = draw(rk, (uint32_t)H.lex, (uint32_t)mu, (uint32_t)w, 0u, KIND_HB);
    __syncthreads();
    // only now: blocks of the next launch that settle earlier crowd the SMs unevenly
    // (12^4 overrelaxation 4.2 -> 3.85 us)
    pdl_launch_dependents();
    double acc = 0.0;
    if (w == 0) {
        M3<float> A;
#pragma unroll
        for (int e = 0; e < 9; e++) {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < 6; k++) s = __fadd2_rn(s, term[k][e][lane]);
            A.e[e / 3][e % 3] = mk(s.x, s.y);
        }
        if (KIND == TERMS_OVERRELAX_LAST && par == 1 && h0 < g.Vh) acc = (double)retr_nn(u, A);
        if constexpr (KIND == TERMS_HEATBATH) {
            const uint4 r[3] = {words[0][lane], words[1][lane], words[2][lane]};
            hb_link_drawn(u, A, beta, r);
        } else {
            or_link(u, A);
        }
        if (h0 < g.Vh) U.store(mu, par, h, u);
    } else if (KIND == TERMS_OVERRELAX_LAST && h0 < g.Vh) {
        // planes 01, 02, 12
        for (int p = w - 1; p < 3; p += WARPS - 1)
            acc += (double)plaquette_retr(U, H, par, par ^ 1, p == 2 ? 1 : 0, p == 0 ? 1 : 2);
    }
    if constexpr (KIND == TERMS_OVERRELAX_LAST) {
        acc = block_sum(acc);
        if (threadIdx.x == 0) *partial = acc;
    }
}

template <int NP, int KIND, int WARPS, bool FMA>
__global__ void __launch_bounds__(WARPS * TERMS_LINKS, 24 / WARPS) k_update_terms(Links<float, NP> U, Geom g, int mu, int par, float beta, RngKey rk,
                                                                                  double* __restrict__ partials) {
    update_terms<NP, KIND, WARPS, FMA>(U, g, blockIdx.x, mu, par, beta, rk, KIND == TERMS_OVERRELAX_LAST ? partials + blockIdx.x : nullptr);
}

// Warps per 32 links of an FP32 launch over n links, 0 for the kernels with a thread per
// link.  Six warps give the shortest chain, three hold more links per SM, and a thread
// per link wins once it fills the SMs; heat bath and overrelaxation of one launch, us:
//               18-real: six      three      thread     12-real: six    three       thread (staged)
//   n = 14336    4.6  3.7    4.9  4.2    8.7  6.9       4.8  3.9    4.6   4.2     9.5  7.6
//       16384    5.0  3.9    5.0  4.3    8.9  7.0       5.0  4.0    4.7   4.3     8.8  7.1
//       20480    6.3  5.0    6.8  4.8    9.2  7.5       6.4  5.1    6.4   4.8    11.7  9.8
//       32768    8.1  6.1    6.7  5.6    9.5  7.2       8.1  6.4    6.8   6.1    10.8  8.6
//       36864    8.3  6.5    6.8  5.7    9.4  6.6       8.4  6.6    6.7   6.1    11.6  9.2
//       40960    9.2  7.2    9.8  7.2    9.5  7.7       9.3  7.5    9.5   7.1    11.6  9.1
//       45056    9.8  7.7   10.0  8.0    9.5  7.8       9.7  7.7    9.8   8.0    10.7  7.8
//       61440   12.5  9.6   11.4  9.5    9.8  7.9      12.3  9.8   11.2   9.0    11.9  9.5
//       65536   12.8 10.0   11.7  9.7    9.7  7.9      13.3 10.2   11.8   9.7    11.7  9.4
//       69632   13.6 10.6   11.8  9.8    9.7  7.9      13.7 10.9   12.5  10.2    11.7  9.4
// The lines lie where the neighbours meet: 16384; 40960 for 18-real links, one wave of
// their one-thread blocks; 65536 for 12-real ones.  Several attempts per subgroup, or
// recorded decisions, run a thread per link.
inline int term_warps(int prec, long n) {
    if (prec == MGQ_F64) return 0;
    if (n < 16384) return 6;
    return n < (prec == MGQ_F32 ? 40960 : 65536) ? 3 : 0;
}

// The products of such a launch: single FMAs, whose chain is shorter (12-real heat bath
// and overrelaxation of 16^4 7.3 and 6.2 -> 6.7 and 6.0 us, 18-real 6.9 and 6.0 -> 6.7
// and 5.5), except where the SMs hold a full wave of three-warp blocks and more:
// there issue counts and the packed forms have fewer (16^3x24: packed 10.1 and 8.1,
// single 10.3 and 8.6 us; 16^3x20: 9.6 and 7.1 against 9.4 and 7.0).  The bits are the same.
inline bool term_single_fma(long n) { return n < 49152; }

}  // namespace mgq
