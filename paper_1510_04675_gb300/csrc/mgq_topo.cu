// libmgq three-loop improved topological charge (Sec. IV.C; the gluonic
// operator of de Forcrand, Garcia Perez and Stamatescu, Nucl. Phys. B 499
// (1997) 409).  q_m(x) is the clover charge density built from the four m x m
// leaves around x in every plane (m = 1, 2, 3).  An m x m clover on spacing a
// is the 1 x 1 clover on spacing m a, so q_m / m^4 = a^4 [q + (m a)^2 X +
// (m a)^4 Y + ...] for a smooth field, and sum_m c_m q_m / m^4 with
// sum c_m = 1, sum c_m m^2 = 0, sum c_m m^4 = 0, i.e. c = (3/2, -3/5, 1/10),
// has no O(a^2) and O(a^4) terms at tree level.
#include "mgq_internal.h"
#include "mgq_stencil.cuh"

namespace mgq {

// The m x m leaves are the 1 x 1 leaves of the field of straight lines of m links,
// which one pass per m extends by a link (line_field, in the workspace): a leaf is four
// line loads instead of 4 m link products (24^3x48, FP32 12-real, the three charges:
// 4.92 ms with every leaf multiplied out, now 0.94 ms; 0.81 ms with rows 0, 1 of the
// products only, which left 10 to 40 % more rounding error in the flowed E and the
// charges).
// NPI: planes of the lines extended, those of the links for the first pass.
template <class T, int NP, int NPI>
__global__ void __launch_bounds__(128) k_line_extend(Links<T, NP> U, Links<T, NPI> in, Links<T, 9> out, Geom g, int len) {
    const int mu = blockIdx.y >> 1, par = blockIdx.y & 1, h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= g.Vh) return;
    int x[4];
    cb_coords(g, par, h, x);
    const Hops H = make_hops(g, x, len);
    const M3<T> u = U.load(mu, par ^ (len & 1), (H.lex + pick(H.fwd, mu)) >> 1);
    out.store(mu, par, h, mul_nn(in.load(mu, par, h), u));
}

void line_field(const mgq_lattice* lat, int m, cudaStream_t st) {
    const Geom g = make_geom(lat->dims);
    dispatch_prec(lat->prec, [&]<class T, int NP>() {
        const dim3 grid((g.Vh + 127) / 128, 8);
        const Links<T, NP> U = links_of<T, NP>(lat);
        const Links<T, 9> lines = links_at<T, 9>(ws_lines(lat), lat->dims);
        if (m == 2) k_line_extend<T, NP, NP><<<grid, 128, 0, st>>>(U, U, lines, g, 1);
        else k_line_extend<T, NP, 9><<<grid, 128, 0, st>>>(U, lines, lines, g, m - 1);
    });
}

// out[0] = 3/2 Q_1 - 3/5 Q_2 / 16 + 1/10 Q_3 / 81 from out[1..3]
__global__ void k_improved_combine(double* out) {
    out[0] = 1.5 * out[1] - 0.6 * out[2] / 16.0 + 0.1 * out[3] / 81.0;
}

// {Q_improved, Q_1x1, Q_2x2, Q_3x3} into dev_out[0..3] (device)
mgq_status improved_charge_into(const mgq_lattice* lat, double* partials, double* dev_out, cudaStream_t st) {
    for (int m = 1; m <= 3; m++) {
        if (m > 1) line_field(lat, m, st);
        const int nb = clover_partials(lat, m, partials, nullptr, st);
        launch_final_sum(partials + nb, nb, 1.0, dev_out + m, st);
    }
    k_improved_combine<<<1, 1, 0, st>>>(dev_out);
    return cuda_check("improved_charge");
}

}  // namespace mgq

using namespace mgq;

extern "C" {

mgq_status mgq_topo_charge_improved(const mgq_lattice* lat, double* Q_out, void* stream) {
    Trace trace("mgq_topo_charge_improved");
    mgq_status s = check_lattice(lat, true, "mgq_topo_charge_improved");
    if (s) return s;
    if (!Q_out) return fail(MGQ_EINVAL, "mgq_topo_charge_improved: Q_out is NULL");
    cudaStream_t st = as_stream(stream);
    double* sc = ws_scalars(lat);
    if ((s = improved_charge_into(lat, ws_partials(lat), sc + 20, st))) return s;
    return deliver(sc + 20, Q_out, 4, st, "mgq_topo_charge_improved");
}

}  // extern "C"
