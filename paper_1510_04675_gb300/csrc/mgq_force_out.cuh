// What the force kernels do with the algebra coefficients t of TA(U A) of a link.
#pragma once

#include "mgq_internal.h"

namespace mgq {

// B <- aB B + cB t (aB == 0: written without being read).
template <class T>
struct ForceOut {
    Alg<T> B;
    T cB, aB;

    __device__ __forceinline__ bool idle() const { return false; }
    // coefficient a of link (mu, par, h)
    __device__ __forceinline__ void put_one(int mu, int par, int h, int a, T t) const {
        T* b = B.at(mu, par, h) + a * Alg<T>::kStep;
        *b = aB == T(0) ? cB * t : aB * *b + cB * t;
    }
    // what B holds of a link, read ahead of put() so that the loads run beside the
    // staple's arithmetic (32^4 P-step, FP32 12-real: 233 us, read at the end 245 us)
    struct Ahead {
        T b[8];
    };
    __device__ __forceinline__ void fetch(int mu, int par, int h, Ahead& f) const {
        if (aB != T(0)) B.load(mu, par, h, f.b);
    }
    // all eight coefficients
    __device__ __forceinline__ void put(int mu, int par, int h, const T t[8], Ahead& f) const {
        T* b = f.b;
        if (aB == T(0)) {
#pragma unroll
            for (int a = 0; a < 8; a++) b[a] = cB * t[a];
        } else {
#pragma unroll
            for (int a = 0; a < 8; a++) b[a] = aB * b[a] + cB * t[a];
        }
        B.store(mu, par, h, b);
    }
};

// The same with z = -h t in place of t, h the step size of an adaptive-flow trial
// (ctl == nullptr: z = t), and a second field: Y <- aY Y + cY z (cY == 0: Y untouched).
// With a control block the launch does nothing while its trial is not active.
template <class T>
struct StageOut {
    ForceOut<T> b, y;
    const FlowCtl* ctl;

    __device__ __forceinline__ bool idle() const { return ctl && !ctl->active; }  // grid-uniform
    __device__ __forceinline__ T step() const { return ctl ? (T)(-ctl->h) : T(1); }
    __device__ __forceinline__ void put_one(int mu, int par, int h, int a, T t) const {
        const T z = step() * t;
        b.put_one(mu, par, h, a, z);
        if (y.cB != T(0)) y.put_one(mu, par, h, a, z);
    }
    typedef typename ForceOut<T>::Ahead Ahead;
    __device__ __forceinline__ void fetch(int mu, int par, int h, Ahead& f) const { b.fetch(mu, par, h, f); }
    // the loads of both fields before the first store, which might alias them
    __device__ __forceinline__ void put(int mu, int par, int h, const T t[8], Ahead& f) const {
        const T s = step();
        T z[8], w[8];
        T* v = f.b;
        if (y.cB != T(0) && y.aB != T(0)) y.B.load(mu, par, h, w);
#pragma unroll
        for (int a = 0; a < 8; a++) {
            z[a] = s * t[a];
            v[a] = b.aB == T(0) ? b.cB * z[a] : b.aB * v[a] + b.cB * z[a];
            w[a] = y.aB == T(0) ? y.cB * z[a] : y.aB * w[a] + y.cB * z[a];
        }
        b.B.store(mu, par, h, v);
        if (y.cB != T(0)) y.B.store(mu, par, h, w);
    }
};

}  // namespace mgq
