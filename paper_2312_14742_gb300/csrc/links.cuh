// Link-by-link sums of a Tau1 node, the arithmetic of the 16-bit formats.
//
// Tau1 (Eq. LBMTau1) sums, over the directions k, the equilibrium that arrives
// from the source x - c_k, each formed as in tau1_node.cuh; a wall link takes the
// node's own equilibrium in direction inv(k) (Algorithm "Complete Tau1 ...
// halfway bounce-back"). FP32 and FP64 boxes take the cheaper sums of moments.cuh.
// A 16-bit state is rounded stochastically: a sum that differs in its last bit
// rounds another way somewhere, the flow goes along another path, and the mean
// velocity moves by some 1e-4 of itself. So that a 16-bit box gives the same
// statistics under every release, its links keep their operations and their order
// (acc_order()), in every kernel.
#pragma once

#include "pack2.cuh"
#include "static_for.cuh"
#include "tau1_node.cuh"

namespace lbm {

// Formats whose nodes are summed link by link.
constexpr bool by_links(int storage) { return storage == ST_F16S || storage == ST_BF16S; }

// Place of link K in the order in which a node is accumulated: the c_z = +1
// links, then c_z = 0, then c_z = -1, each group in k order.
__host__ __device__ constexpr int acc_order(int k) { return (cvel(k, 2) == 1 ? 0 : (cvel(k, 2) == 0 ? 1 : 2)) * 32 + k; }

// True when link K is the first, in that order, to add to accumulator comp
// (0: S, 1..3: J_x..J_z) of its class. The sum then starts from that term
// instead of from zero: one addition fewer, and only the sign of an all-zero
// sum can differ.
template <int Q> __host__ __device__ constexpr bool first_link(int K, int comp)
{
    for (int k = 1; k < Q; ++k)
        if (dir_class(k) == dir_class(K) && (comp == 0 || cvel(k, comp - 1) != 0) && acc_order(k) < acc_order(K))
            return false;
    return true;
}

// Accumulators of one node: per direction class, the sum of the scaled
// equilibria and of c times them. add<Q, K> must be called in acc_order.
template <typename T, int NC> struct NodeAcc {
    T S[NC];
    T Jx[NC], Jy[NC], Jz[NC];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int c = 0; c < NC; ++c) S[c] = Jx[c] = Jy[c] = Jz[c] = T(0);
    }
    template <int C, bool FIRST> __device__ static __forceinline__ void put(T& a, T f)
    {
        if constexpr (C > 0) {
            if constexpr (FIRST) a = f;
            else a = a + f;
        } else if constexpr (C < 0) {
            if constexpr (FIRST) a = -f;
            else a = a - f;
        }
    }
    template <int Q, int K> __device__ __forceinline__ void add(T f)
    {
        constexpr int cls = dir_class(K);
        put<1, first_link<Q>(K, 0)>(S[cls], f);
        put<cvel(K, 0), first_link<Q>(K, 1)>(Jx[cls], f);
        put<cvel(K, 1), first_link<Q>(K, 2)>(Jy[cls], f);
        put<cvel(K, 2), first_link<Q>(K, 3)>(Jz[cls], f);
    }
};

// Calls f for the links of acc_order's group CZ, in order.
template <int Q, int CZ, typename F> __device__ __forceinline__ void links_of(F&& f)
{
    static_for<1, Q>([&](auto kc) {
        if constexpr (cvel(decltype(kc)::value, 2) == CZ) f(kc);
    });
}

// Final step of Algorithm "Optimized Tau1 ... stores velocity": apply the
// class weights, then one reciprocal of rho for the three velocity components.
template <int Q, typename T>
__device__ __forceinline__ void node_finish(const NodeAcc<T, Weights<Q>::NCLASS>& a, T& drho, T& ux, T& uy, T& uz)
{
    constexpr int NC = Weights<Q>::NCLASS;
    T d = T(Weights<Q>::w(0)) * a.S[0];
    T jx = T(0), jy = T(0), jz = T(0);
#pragma unroll
    for (int c = 1; c < NC; ++c) {
        const T w = T(Weights<Q>::w(c));
        d = fma(w, a.S[c], d);
        jx = fma(w, a.Jx[c], jx);
        jy = fma(w, a.Jy[c], jy);
        jz = fma(w, a.Jz[c], jz);
    }
    const T r = recip(T(1) + d);
    drho = d;
    ux = jx * r;
    uy = jy * r;
    uz = jz * r;
}

// One node gathered by one thread from its record and load(k, solid, d, ux, uy, uz),
// which gives the record of the source x - c_k or says that it is a wall. SKIP:
// a wall's record is not evaluated at all, where that pays for the branch.
template <int Q, bool SKIP, typename T, typename F>
__device__ __forceinline__ void gather_links(const StepArgs& a, T d0, T ux0, T uy0, T uz0, F&& load, T& d, T& ux, T& uy, T& uz)
{
    const T gx = gcomp<T>(a, 0), gy = gcomp<T>(a, 1), gz = gcomp<T>(a, 2);
    const NodeMoments<T> own = node_moments<T>(d0, ux0, uy0, uz0, gx, gy, gz);
    NodeAcc<T, Weights<Q>::NCLASS> acc;
    acc.S[0] = own.A;  // rest direction: p = 0
    auto link = [&](auto kc) {
        constexpr int K = decltype(kc)::value;
        T sd, sx, sy, sz;
        bool solid = false;
        load(kc, solid, sd, sx, sy, sz);
        T v = T(0);
        if (!SKIP || !solid) {
            const NodeMoments<T> m = node_moments<T>(sd, sx, sy, sz, gx, gy, gz);
            v = feq_scaled(m.A, m.H, dir_dot<K, T>(m.Px, m.Py, m.Pz));
        }
        // reflected population: own state in direction inv(k), p(inv k) = -p(k)
        const T b = feq_scaled(own.A, own.H, -dir_dot<K, T>(own.Px, own.Py, own.Pz));
        acc.template add<Q, K>(solid ? b : v);
    };
    links_of<Q, 1>(link);
    links_of<Q, 0>(link);
    links_of<Q, -1>(link);
    node_finish<Q, T>(acc, d, ux, uy, uz);
}

}  // namespace lbm
