// libmgq Wilson flow (Sec. IV.B; fixed step, Luscher's third-order
// Runge-Kutta integrator) and clover observables E(t), Q(t) (Sec. IV.B-C).
#include "mgq_internal.h"
#include "mgq_stencil.cuh"

namespace mgq {

// Per site: E(x) = -1/2 sum_{mu,nu} Tr G^2 = 1/2 sum_{mu<nu} |g_munu|^2 and
// q(x) = -1/(32 pi^2) eps Tr(G G) = 1/(8 pi^2) (g01.g23 - g02.g13 + g03.g12),
// using Tr(X_a X_b) = -delta_ab / 2, with G from the leaves of the line field A of
// m links a side (m = 1: the links).  One thread per site and dual pair of planes
// (block row y): its two field strengths stay in registers, and a small lattice
// has three times the threads of a thread per site (mgq_topo_charge on 24^3x48, FP32
// 12-real: 396 -> 291 us a call, 16^4: 83 -> 58 us; bound by the FMAs of its ten full
// products a plane and the twelve link loads that feed them).
template <class T, int NP>
__global__ void __launch_bounds__(128, sizeof(T) == 8 ? 1 : 4) k_clover(Links<T, NP> A, Geom g, int m, double* __restrict__ partials,
                                                                       const int* __restrict__ gate) {
    if (gate && !__ldg(gate)) return;  // grid-uniform: the whole launch skips
    const int p = blockIdx.y;
    double e = 0.0, q = 0.0;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < g.V; idx += gridDim.x * blockDim.x) {
        const int par = idx >= g.Vh, h = idx - par * g.Vh;
        int x[4];
        cb_coords(g, par, h, x);
        const Hops H = m == 1 ? make_hops(g, x) : make_hops(g, x, m);
        const int op = par ^ (m & 1);
        T Ga[8], Gb[8];
        clover_coeffs(A, H, par, op, 0, p + 1, Ga);
        clover_coeffs(A, H, par, op, dual_mu(p), dual_nu(p), Gb);
        // per-site sums in the link precision (FP64 arithmetic is slow on this
        // part), accumulated over sites in FP64
        T es = T(0), dot = T(0);
#pragma unroll
        for (int a = 0; a < 8; a++) {
            es += Ga[a] * Ga[a] + Gb[a] * Gb[a];
            dot += Ga[a] * Gb[a];
        }
        e += (double)es;
        q += (double)(p == 1 ? -dot : dot);
    }
    e = block_sum(0.5 * e);
    q = block_sum(q * (1.0 / (8.0 * 9.869604401089358)));
    if (threadIdx.x == 0) {
        const int b = blockIdx.y * gridDim.x + blockIdx.x, nb = 3 * gridDim.x;
        partials[b] = e;
        partials[nb + b] = q;
    }
}

int clover_partials(const mgq_lattice* lat, int m, double* partials, const int* gate, cudaStream_t st) {
    const Geom g = make_geom(lat->dims);
    const int nb = reduction_blocks(g.V, 128);  // at most 1184: 2 x 3 x 1184 partial sums
    dispatch_prec(lat->prec, [&]<class T, int NP>() {
        if (m == 1) k_clover<T, NP><<<dim3(nb, 3), 128, 0, st>>>(links_of<T, NP>(lat), g, 1, partials, gate);
        else k_clover<T, 9><<<dim3(nb, 3), 128, 0, st>>>(links_at<T, 9>(ws_lines(lat), lat->dims), g, m, partials, gate);
    });
    return 3 * nb;
}

mgq_status clover_into(const mgq_lattice* lat, double* partials, double* dev_out, cudaStream_t st) {
    const Geom g = make_geom(lat->dims);
    const int nb = clover_partials(lat, 1, partials, nullptr, st);
    launch_final_sum2(partials, nb, 1.0 / (double)g.V, 1.0, dev_out, st);
    return cuda_check("clover");
}

mgq_status improved_charge_into(const mgq_lattice* lat, double* partials, double* dev_out, cudaStream_t st);

// One RK3 step of size eps with the workspace's algebra buffer B:
// Z_i = eps Z(W_i), Z(W) = -TA(W A(W));
// W1 = exp(Z0/4) W0; W2 = exp(8/9 Z1 - 17/36 Z0) W1; W3 = exp(3/4 Z2 - 8/9 Z1 + 17/36 Z0) W2
static mgq_status flow_step(mgq_lattice* lat, void* B, double eps, cudaStream_t st) {
    mgq_status s;
    if ((s = force_accumulate(lat, B, -eps, 0.0, st))) return s;                       // B = Z0
    if ((s = exp_update(lat, B, 0.25, st))) return s;
    if ((s = force_accumulate(lat, B, -eps * 8.0 / 9.0, -17.0 / 36.0, st))) return s;  // B = 8/9 Z1 - 17/36 Z0
    if ((s = exp_update(lat, B, 1.0, st))) return s;
    if ((s = force_accumulate(lat, B, -eps * 0.75, -1.0, st))) return s;               // B = 3/4 Z2 - B
    return exp_update(lat, B, 1.0, st);
}

// E and Q of the current links into meas[0], meas[1] (device); charge 1 takes
// the three-loop improved Q (its four values pass through tmp[0..3]).
static mgq_status measure_EQ(const mgq_lattice* lat, int charge, double* meas, double* tmp, cudaStream_t st) {
    mgq_status s = clover_into(lat, ws_partials(lat), meas, st);
    if (s || !charge) return s;
    if ((s = improved_charge_into(lat, ws_partials(lat), tmp, st))) return s;
    if (cudaMemcpyAsync(meas + 1, tmp, sizeof(double), cudaMemcpyDeviceToDevice, st) != cudaSuccess)
        return cuda_check("measure_EQ");
    return MGQ_OK;
}

}  // namespace mgq

using namespace mgq;

extern "C" {

mgq_status mgq_topo_charge(const mgq_lattice* lat, double* E_out, double* Q_out, void* stream) {
    Trace trace("mgq_topo_charge");
    mgq_status s = check_lattice(lat, true, "mgq_topo_charge");
    if (s) return s;
    cudaStream_t st = as_stream(stream);
    double* sc = ws_scalars(lat);
    if ((s = clover_into(lat, ws_partials(lat), sc + 16, st))) return s;
    return deliver_pairs(sc + 16, E_out, Q_out, 1, st, "mgq_topo_charge");
}

mgq_status mgq_wilson_flow(mgq_lattice* lat, double eps, int n_steps, int meas_every, double* E_out, double* Q_out,
                           void* stream) {
    Trace trace("mgq_wilson_flow");
    mgq_status s = check_lattice(lat, true, "mgq_wilson_flow");
    if (s) return s;
    if (!(eps > 0.0) || n_steps < 0 || meas_every < 1)
        return fail(MGQ_EINVAL, "mgq_wilson_flow: need eps > 0, n_steps >= 0, meas_every >= 1");
    const int nm = n_steps / meas_every + 1;
    if (2 * nm + 32 > (int)WS_NSCALARS) return fail(MGQ_EINVAL, "mgq_wilson_flow: at most %d measurements", (int)(WS_NSCALARS - 32) / 2);
    cudaStream_t st = as_stream(stream);
    double* sc = ws_scalars(lat);
    double* meas = sc + 32;  // E at meas[2m], Q at meas[2m+1]
    void* B = ws_alg(lat);
    int m = 0;
    for (int k = 0; k <= n_steps; k++) {
        if (k % meas_every == 0) {
            if ((s = clover_into(lat, ws_partials(lat), meas + 2 * m, st))) return s;
            m++;
        }
        if (k == n_steps) break;
        if ((s = flow_step(lat, B, eps, st))) return s;
    }
    return deliver_pairs(meas, E_out, Q_out, (size_t)nm, st, "mgq_wilson_flow");
}

mgq_status mgq_wilson_flow_times(mgq_lattice* lat, double t_end, double eps, const double* t_meas, int n_meas,
                                 int charge, double* E_out, double* Q_out, void* stream) {
    Trace trace("mgq_wilson_flow_times");
    mgq_status s = check_lattice(lat, true, "mgq_wilson_flow_times");
    if (s) return s;
    if (!(eps > 0.0) || !(t_end >= 0.0) || n_meas < 0 || (n_meas > 0 && !t_meas) || charge < 0 || charge > 1)
        return fail(MGQ_EINVAL, "mgq_wilson_flow_times: need eps > 0, t_end >= 0, n_meas >= 0, t_meas, charge 0 or 1");
    if (2 * n_meas + 64 > (int)WS_NSCALARS)
        return fail(MGQ_EINVAL, "mgq_wilson_flow_times: at most %d measurements", (int)(WS_NSCALARS - 64) / 2);
    for (int i = 0; i < n_meas; i++)
        if (!(t_meas[i] >= 0.0) || t_meas[i] > t_end || (i > 0 && t_meas[i] < t_meas[i - 1]))
            return fail(MGQ_EINVAL, "mgq_wilson_flow_times: t_meas must be ascending within [0, t_end]");
    if (t_end / eps > 1e8) return fail(MGQ_EINVAL, "mgq_wilson_flow_times: more than 1e8 steps");
    cudaStream_t st = as_stream(stream);
    double* sc = ws_scalars(lat);
    double* meas = sc + 64;  // E at meas[2i], Q at meas[2i+1]
    void* B = ws_alg(lat);
    const double tiny = 1e-12 * (t_end > 1.0 ? t_end : 1.0);
    double t = 0.0;
    int i = 0;
    while (i < n_meas && t_meas[i] <= t + tiny) {
        if ((s = measure_EQ(lat, charge, meas + 2 * i, sc + 24, st))) return s;
        i++;
    }
    while (t < t_end - tiny) {
        // the next stop: the next measurement time below t_end, else t_end
        const double stop = (i < n_meas && t_meas[i] < t_end) ? t_meas[i] : t_end;
        const double h = stop - t < eps ? stop - t : eps;
        if ((s = flow_step(lat, B, h, st))) return s;
        t = h == stop - t ? stop : t + h;
        while (i < n_meas && t_meas[i] <= t + tiny) {
            if ((s = measure_EQ(lat, charge, meas + 2 * i, sc + 24, st))) return s;
            i++;
        }
    }
    return deliver_pairs(meas, E_out, Q_out, (size_t)n_meas, st, "mgq_wilson_flow_times");
}

}  // extern "C"
