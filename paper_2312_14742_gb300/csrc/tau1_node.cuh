// Equilibria of a node link by link, for the D2Q9, BGK and Zou-He kernels and for
// 16-bit boxes (links.cuh); the 3D kernels of FP32 and FP64 boxes sum them axis by
// axis (moments.cuh).
//
// Eq. (feq) with c_s^2 = 1/3, written as the deviation from the rest weight
// and divided by the weight w_k:
//     (f_k^eq - w_k) / w_k = drho + rho (3 c.v + 4.5 (c.v)^2 - 1.5 v.v)
//                          = A + p + p^2 H,   p = c_k . P,
// with the per-node moments A = drho - 1.5 rho v.v, P = 3 rho v, H = 1/(2 rho)
// and v = u + g (velocity-shift body force).
#pragma once

#include "common.cuh"

namespace lbm {

template <typename T> struct NodeMoments {
    T A, Px, Py, Pz, H;
};

template <typename T>
__device__ __forceinline__ NodeMoments<T> node_moments(T drho, T ux, T uy, T uz, T gx, T gy, T gz)
{
    // Every fused multiply-add is written out, so that no kernel depends on
    // the compiler's contraction choices.
    NodeMoments<T> m;
    const T rho = T(1) + drho;
    const T vx = ux + gx, vy = uy + gy, vz = uz + gz;
    const T vv = fma(vz, vz, fma(vy, vy, vx * vx));
    m.A = fma(T(-1.5) * rho, vv, drho);
    const T r3 = T(3) * rho;
    m.Px = r3 * vx;
    m.Py = r3 * vy;
    m.Pz = r3 * vz;
    m.H = T(0.5) * recip(rho);
    return m;
}

// p = c_k . P with compile-time velocity components (adds and subtractions in
// axis order x, y, z, so that p of inv(k) is exactly -p of k).
template <int K, typename T>
__device__ __forceinline__ T dir_dot(T Px, T Py, T Pz)
{
    constexpr int cx = cvel(K, 0), cy = cvel(K, 1), cz = cvel(K, 2);
    T p = T(0);
    bool any = false;
    if (cx != 0) { p = cx > 0 ? Px : -Px; any = true; }
    if (cy != 0) { p = any ? (cy > 0 ? p + Py : p - Py) : (cy > 0 ? Py : -Py); any = true; }
    if (cz != 0) { p = any ? (cz > 0 ? p + Pz : p - Pz) : (cz > 0 ? Pz : -Pz); any = true; }
    return p;
}

// (f_k^eq - w_k) / w_k from the source moments: A + p (1 + p H), evaluated as
// fma(p*H, p, A) + p. The value for inv(k) uses -p and is exact in sign.
template <typename T>
__device__ __forceinline__ T feq_scaled(T A, T H, T p)
{
    return fma(p * H, p, A) + p;
}

}  // namespace lbm
