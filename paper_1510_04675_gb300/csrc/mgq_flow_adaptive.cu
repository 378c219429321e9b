// libmgq adaptive-step Wilson flow (Sec. IV.B: tolerance and maximal step as
// in Table II; the step controller follows the cited embedded Runge-Kutta
// scheme).  A trial step of size h runs the three stages of the third-order
// integrator and, from the same stage generators, the second-order solution
// W2 = exp(2 Z1 - Z0) W0.  d = max over links of |W3 - W2|_F / 3; the step is
// kept iff d <= tol and the next trial size is h min(2, 0.95 (tol/d)^(1/3)),
// capped by the maximal step and by the next measurement time.  A step that
// was cut short to land on a measurement time keeps the previous size.
//
// The controller lives on the device: each trial is a fixed sequence of
// launches whose kernels read the step size and their gate from a small
// control block, so the host never waits on a step.  It reads the finished
// flag once per chunk of trials.  The trial's kernels use programmatic
// dependent launch (see pdl_wait), so they read their predecessors' outputs
// with plain loads only.
#include "mgq_internal.h"
#include "mgq_stencil.cuh"

namespace mgq {

__global__ void k_adapt_init(FlowCtl* c, double eps0) {
    c->t = 0.0;
    c->eps = eps0;
    c->h = 0.0;
    c->t_next = 0.0;
    c->dbits = 0ull;
    c->active = 0;
    c->hits = 0;
    c->restore = 0;
    c->meas = 1;  // E, Q at t = 0
    c->m = 0;
    c->steps = 0;
    c->rejects = 0;
    c->status = 0;
}

// Sets up the next trial: its size, capped by the maximal step and the next
// measurement time, or the end of the flow.
__device__ __forceinline__ void adapt_begin(FlowCtl* c, double t_end, double eps_max, double dt_meas, int max_meas) {
    c->active = 0;
    c->restore = 0;
    c->meas = 0;
    if (c->status != 0) return;
    const double tiny = 1e-12 * dt_meas;
    if (!(c->t < t_end - tiny) || c->m >= max_meas) {
        c->status = 1;
        return;
    }
    const double t_next = fmin(dt_meas * (double)c->m, t_end);
    double h = fmin(c->eps, eps_max);
    int hits = 0;
    if (c->t + h >= t_next - tiny) {
        h = t_next - c->t;
        hits = 1;
    }
    c->t_next = t_next;
    c->h = h;
    c->hits = hits;
    c->dbits = 0ull;
    c->active = 1;
}

__global__ void k_adapt_end(FlowCtl* c, double tol, double eps_max) {
    pdl_launch_dependents();
    pdl_wait();
    if (!c->active) return;
    const double d = __longlong_as_double((long long)c->dbits);
    double fac = d > 0.0 ? 0.95 * cbrt(tol / d) : 2.0;
    if (fac > 2.0) fac = 2.0;
    if (d <= tol) {
        c->t = c->hits ? c->t_next : c->t + c->h;
        c->steps++;
        c->meas = c->hits;
        if (!c->hits) c->eps = c->h * fac;
    } else {
        c->restore = 1;
        c->rejects++;
        c->eps = c->h * fac;
        if (!(c->eps >= 1e-9 * eps_max)) c->status = 2;
    }
}

// W <- exp(s B) W, block row y the (mu, parity) plane.  SAVE: the old W goes to
// `start` first (the start of the trial, restored on rejection).  ERROR (the
// trial's last stage): also d = max over links of |W3 - exp(Y) W0|_F / 3, Y = 2 Z1 -
// Z0, with W3 at hand and W0 from `start`.
template <class T, int NP, bool SAVE, bool ERROR>
__global__ void __launch_bounds__(128) k_flow_exp(Links<T, NP> U, Geom g, Alg<T> B, T s, FlowCtl* c, Links<T, NP> start,
                                                  Alg<T> Y) {
    pdl_launch_dependents();
    const int mu = blockIdx.y >> 1, par = blockIdx.y & 1, h = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait();
    if (!c->active) return;
    double d = 0.0;
    if (h < g.Vh) {
        T q[8];
        B.load(mu, par, h, q);
        const M3<T> u0 = U.load(mu, par, h);
#pragma unroll
        for (int a = 0; a < 8; a++) q[a] *= s;
        if (SAVE) start.store(mu, par, h, u0);
        M3<T> u = mul_nn(exp_alg(q), u0);
        if (sizeof(T) == 4) reunitarize(u);
        U.store(mu, par, h, u);
        if constexpr (ERROR) {
            Y.load(mu, par, h, q);
            const M3<T> w2 = mul_nn(exp_alg(q), start.load(mu, par, h));
            // in the link precision: an FP32 estimate steers the step as well as
            // an FP64 one, and FP64 arithmetic is slow on this part
            T s2 = T(0);
#pragma unroll
            for (int i = 0; i < 3; i++)
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    const T dr = u.e[i][j].re - w2.e[i][j].re;
                    const T di = u.e[i][j].im - w2.e[i][j].im;
                    s2 += dr * dr + di * di;
                }
            d = (double)(m_sqrt(s2) / T(3));
        }
    }
    if constexpr (ERROR) {
        // Non-negative doubles order like their bit patterns, and a NaN compares
        // above every number, so a broken step is rejected.
        unsigned long long bits = (unsigned long long)__double_as_longlong(d);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_down_sync(0xffffffffu, bits, o);
            bits = other > bits ? other : bits;
        }
        if ((threadIdx.x & 31) == 0 && bits) atomicMax(&c->dbits, bits);
    }
}

__global__ void k_flow_restore(uint4* links, const uint4* backup, size_t nwords,
                               const FlowCtl* c) {
    pdl_launch_dependents();
    pdl_wait();
    if (!c->restore) return;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nwords; i += (size_t)gridDim.x * blockDim.x)
        links[i] = backup[i];
}

// After a trial (and before the first): the measurement it asked for, meas[2m] = E
// (site average), meas[2m+1] = Q from the clover partials, m++; then the next trial
// is set up.
__global__ void k_adapt_next(FlowCtl* c, const double* partials, int nb, double invV, double* meas, double t_end, double eps_max,
                             double dt_meas, int max_meas) {
    pdl_launch_dependents();
    pdl_wait();
    if (c->meas) {
        double e = 0.0, q = 0.0;
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
            e += partials[i];
            q += partials[nb + i];
        }
        e = block_sum(e);
        q = block_sum(q);
        if (threadIdx.x == 0) {
            meas[2 * c->m] = e * invV;
            meas[2 * c->m + 1] = q;
            c->m++;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) adapt_begin(c, t_end, eps_max, dt_meas, max_meas);
}

static inline int nblk(long n, int t) { return (int)((n + t - 1) / t); }

// Measurement times k dt_meas <= t_end, plus t_end when it is not one of them.
int adaptive_measurements(double t_end, double dt_meas) {
    const int k = (int)floor(t_end / dt_meas + 1e-9);
    return k + 1 + (t_end - k * dt_meas > 1e-12 * dt_meas ? 1 : 0);
}

}  // namespace mgq

using namespace mgq;

extern "C" {

uint64_t mgq_flow_adaptive_scratch_bytes(const mgq_lattice* lat) {
    if (!lat || !links_bytes(lat)) return 0;
    return round256(alg_bytes(lat));
}

int mgq_flow_adaptive_measurements(double t_end, double dt_meas) {
    if (!(t_end >= 0.0) || !(dt_meas > 0.0) || t_end / dt_meas > 1e6) return -1;
    return adaptive_measurements(t_end, dt_meas);
}

mgq_status mgq_wilson_flow_adaptive(mgq_lattice* lat, double t_end, double tol, double eps_max, double eps0,
                                    double dt_meas, double* E_out, double* Q_out, int* n_meas, int* n_steps,
                                    int* n_rejects, void* scratch, uint64_t scratch_bytes, void* stream) {
    Trace trace("mgq_wilson_flow_adaptive");
    mgq_status s = check_lattice(lat, true, "mgq_wilson_flow_adaptive");
    if (s) return s;
    if (!(t_end >= 0.0) || !(tol > 0.0) || !(eps_max > 0.0) || !(eps0 > 0.0) || !(dt_meas > 0.0))
        return fail(MGQ_EINVAL, "mgq_wilson_flow_adaptive: need t_end >= 0 and tol, eps_max, eps0, dt_meas > 0");
    const int nm = mgq_flow_adaptive_measurements(t_end, dt_meas);
    if (nm < 0 || 2 * nm + 32 > (int)WS_NSCALARS)
        return fail(MGQ_EINVAL, "mgq_wilson_flow_adaptive: at most %d measurements", (int)(WS_NSCALARS - 32) / 2);
    if (!scratch || ((uintptr_t)scratch & 255))
        return fail(MGQ_EINVAL, "mgq_wilson_flow_adaptive: scratch NULL or not 256-byte aligned");
    if (scratch_bytes < round256(alg_bytes(lat)))
        return fail(MGQ_ENOMEM, "mgq_wilson_flow_adaptive: scratch has %llu bytes, needs %llu",
                    (unsigned long long)scratch_bytes, (unsigned long long)round256(alg_bytes(lat)));
    const Geom g = make_geom(lat->dims);
    cudaStream_t st = as_stream(stream);
    double* sc = ws_scalars(lat);
    FlowCtl* c = reinterpret_cast<FlowCtl*>(sc);
    double* meas = sc + 32;
    double* partials = ws_partials(lat);
    const double invV = 1.0 / (double)g.V;
    void* Bp = ws_alg(lat);
    void* backup = ws_links(lat);
    const size_t nwords = links_bytes(lat) / 16;

    auto next = [&]() {
        const int nb = clover_partials(lat, 1, partials, &c->meas, st);
        launch_pdl(k_adapt_next, 1, 512, st, c, partials, nb, invV, meas, t_end, eps_max, dt_meas, nm);
    };
    auto trial = [&]() {
        dispatch_prec(lat->prec, [&]<class T, int NP>() {
            const Links<T, NP> U = links_of<T, NP>(lat), U0 = links_at<T, NP>(backup, lat->dims);
            const Alg<T> B = alg_at<T>(Bp, lat->dims), Y = alg_at<T>(scratch, lat->dims);
            const dim3 eb(nblk(g.Vh, 128), 8);
            // Z0: B = Z0, Y = -Z0
            flow_stage(lat, Bp, 1.0, 0.0, scratch, -1.0, 0.0, c, st);
            launch_pdl(k_flow_exp<T, NP, true, false>, eb, 128, st, U, g, B, T(0.25), c, U0, Y);
            // Z1: B = 8/9 Z1 - 17/36 B, Y = 2 Z1 + Y
            flow_stage(lat, Bp, 8.0 / 9.0, -17.0 / 36.0, scratch, 2.0, 1.0, c, st);
            launch_pdl(k_flow_exp<T, NP, false, false>, eb, 128, st, U, g, B, T(1), c, U0, Y);
            // Z2: B = 3/4 Z2 - B
            flow_stage(lat, Bp, 0.75, -1.0, scratch, 0.0, 0.0, c, st);
            launch_pdl(k_flow_exp<T, NP, false, true>, eb, 128, st, U, g, B, T(1), c, U0, Y);
        });
        launch_pdl(k_adapt_end, 1, 1, st, c, tol, eps_max);
        launch_pdl(k_flow_restore, 1184, 256, st, reinterpret_cast<uint4*>(lat->links),
                   reinterpret_cast<const uint4*>(backup), nwords, (const FlowCtl*)c);
        next();
    };

    k_adapt_init<<<1, 1, 0, st>>>(c, eps0);
    next();
    if ((s = cuda_check("mgq_wilson_flow_adaptive"))) return s;
    // Trials run in chunks between reads of the status word; a chunk that
    // finishes early leaves its remaining trials as gated no-op launches.
    constexpr int kChunk = 16, kMaxTrials = 1 << 20;
    int status = 0;
    for (int done = 0; status == 0; done += kChunk) {
        if (done >= kMaxTrials) return fail(MGQ_EINVAL, "mgq_wilson_flow_adaptive: more than %d trial steps", kMaxTrials);
        for (int i = 0; i < kChunk; i++) trial();
        if ((s = cuda_check("mgq_wilson_flow_adaptive"))) return s;
        if ((s = deliver_int(&c->status, &status, 1, st, "mgq_wilson_flow_adaptive"))) return s;
    }
    if (status == 2)
        return fail(MGQ_EINVAL, "mgq_wilson_flow_adaptive: step size underflow (tolerance below the precision floor)");
    int cnt[3];
    if ((s = deliver_int(&c->m, cnt, 3, st, "mgq_wilson_flow_adaptive"))) return s;
    if ((s = deliver_pairs(meas, E_out, Q_out, (size_t)cnt[0], st, "mgq_wilson_flow_adaptive"))) return s;
    if (n_meas) *n_meas = cnt[0];
    if (n_steps) *n_steps = cnt[1];
    if (n_rejects) *n_rejects = cnt[2];
    return MGQ_OK;
}

}  // extern "C"
