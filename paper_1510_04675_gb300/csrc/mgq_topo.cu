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
// which one pass per m extends by a link (line_field, into the workspace's link
// copy): a leaf is four line loads instead of 4 m link products (24^3x48, FP32
// 12-real, the three charges: 4.83 ms -> 0.82 ms, of which 3 x 245 us for the
// clovers and 2 x 40 us for the lines).

template <class T, int NP>
__global__ void __launch_bounds__(128) k_line_extend(Links<T, NP> U, Links<T, NP> in, Links<T, NP> out, Geom g, int len) {
    const int mu = blockIdx.y >> 1, par = blockIdx.y & 1, h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= g.Vh) return;
    int x[4];
    cb_coords(g, par, h, x);
    const Hops H = make_hops(g, x, len);
    const M3<T> u = U.load(mu, par ^ (len & 1), (H.lex + pick(H.fwd, mu)) >> 1);
    M3<T> r;
    if constexpr (sizeof(T) == 4) {
        r = mul_nn_2(in.load_rows(mu, par, h), u);
        rebuild_row2(r);
    } else {
        r = mul_nn(in.load(mu, par, h), u);
    }
    out.store(mu, par, h, r);
}

void line_field(const mgq_lattice* lat, const void* lines_in, void* lines_out, int m, cudaStream_t st) {
    const Geom g = make_geom(lat->dims);
    dispatch_prec(lat->prec, [&]<class T, int NP>() {
        k_line_extend<T, NP><<<dim3((g.Vh + 127) / 128, 8), 128, 0, st>>>(
            links_of<T, NP>(lat), links_at<T, NP>(const_cast<void*>(lines_in), lat->dims), links_at<T, NP>(lines_out, lat->dims),
            g, m - 1);
    });
}

// out[0] = 3/2 Q_1 - 3/5 Q_2 / 16 + 1/10 Q_3 / 81 from out[1..3]
__global__ void k_improved_combine(double* out) {
    out[0] = 1.5 * out[1] - 0.6 * out[2] / 16.0 + 0.1 * out[3] / 81.0;
}

// {Q_improved, Q_1x1, Q_2x2, Q_3x3} into dev_out[0..3] (device)
mgq_status improved_charge_into(const mgq_lattice* lat, double* partials, double* dev_out, cudaStream_t st) {
    const void* lines = lat->links;
    for (int m = 1; m <= 3; m++) {
        if (m > 1) {
            line_field(lat, lines, ws_links(lat), m, st);
            lines = ws_links(lat);
        }
        const int nb = clover_partials(lat, lines, m, partials, nullptr, st);
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
