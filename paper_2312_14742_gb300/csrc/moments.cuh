// Arithmetic of one Tau1 node update in FP32 and FP64, shared by every 3D step
// kernel (the 16-bit formats take links.cuh).
//
// Tau1 (Eq. LBMTau1) sums, over the directions k, the equilibrium of the
// source x - c_k. With c_s^2 = 1/3 the equilibrium's deviation from its rest
// weight is (Eq. feq)
//     (f_k^eq - w_k) / w_k = A + c.P + c.Q.c,
// P = 3 rho (u + g), Q = 4.5 rho (u + g)(u + g), A = drho - tr(Q)/3 (velocity-shift
// body force g): no division.
//
// The destination needs only four sums over its sources: the density and the
// three momentum components. Both lattices are products or near-products of
// one-dimensional stencils, so the sums are taken axis by axis: along y (the
// values that rows send up and down, up[] and dn[]), then along z (what a
// plane sends to the plane above, P[], keeps, O[], and sends below, M[]), then
// along x (three values to each side). D3Q19 takes 89 operations per node and
// D3Q27 96, where summing link by link takes 134 and 196, and a node passes 6
// values along x instead of 10 or 18.
//
// Walls (Algorithm "Complete Tau1 ... halfway bounce-back"): a solid source
// has zero moments and adds nothing; bounce() returns what the wall links of a
// node add, the node's own equilibria in the directions inv(k), from a mask of
// its wall links. It is added to the finished sums, so a node without wall
// links needs no wall arithmetic at all.
//
// Every kernel that steps such a node calls these functions in this order, with
// every fused multiply-add written out, so all of them give the same bits. The
// assembler fuses a packed product into a packed sum even where contraction is
// off, so a product that feeds a sum is written product(): a fused operation
// already.
#pragma once

#include "common.cuh"
#include "pack2.cuh"
#include "static_for.cuh"

namespace lbm {

template <typename T, typename = void> struct IsFp64 : std::is_same<T, double> {};
template <typename T> struct IsFp64<T, std::void_t<typename T::elem>> : std::is_same<typename T::elem, double> {};

// Scales of the moments: v = V (u + g), r = R rho, so that with p = c.(r v) the
// linear term of a direction is L p and the quadratic one p (c.v). That asks for
// V R L = 3 and V^2 R = 4.5; V = 1.5, R = 2, L = 1 would do and costs the same,
// but 1.5 u has at most one bit more than u, so that rounding it, with the
// constant 1.5 g added, errs to the same side step after step: a channel's
// momentum was 1e-6 off after 100 steps. These V have full mantissas, and u V
// rounds as any number does: 1.3e-7. The two products hold to 5e-13 in FP32
// (constants with 24 bits) and to 2e-23 in FP64.
// A = drho - r vv / 3 takes back the trace of the quadratic terms, and what it
// leaves is lost or gained by every node in every step: a third rounded to 24 bits
// cost 4.5e-8 u.u of density a step. So R / 3 has 24 bits too, and r / 3 is
// rounded from drho by itself.
template <typename T> struct Scale {
    static constexpr double V = IsFp64<T>::value ? 1.544922908228737 : 1.5488158464431763;
    static constexpr double R = IsFp64<T>::value ? 1.885379965393459 : 1.8759140968322754;
    static constexpr double L = IsFp64<T>::value ? 1.0299486054858247 : 1.0325438976287842;
    static constexpr double R3 = R / 3.0;
    static_assert(3.0 * R3 == R && (IsFp64<T>::value || (double)(float)R3 == R3), "a third without rounding");
};

template <typename T> struct Moments {
    T A, r, vx, vy, vz;
};

// What a node's density leaves after the trace, from d = drho.
template <typename T> __device__ __forceinline__ T less_trace(T d, T vx, T vy, T vz)
{
    const T vv = fma(vz, vz, fma(vy, vy, vx * vx));
    return fma(fma(T(-Scale<T>::R3), d, T(-Scale<T>::R3)), vv, d);
}

// A product as one fused operation (+0 for a zero product of either sign): its
// result can feed a packed sum, see above.
template <typename T> __device__ __forceinline__ T product(T a, T b) { return fma(a, b, T(0)); }

// How a stored record enters its moments: V (u + g), R (1 + drho), drho.
template <int ST> struct Terms {
    using T = typename Storage<ST>::ctype;
    T gx, gy, gz;
    __device__ __forceinline__ explicit Terms(const StepArgs& a)
        : gx(T(Scale<T>::V) * gcomp<T>(a, 0)), gy(T(Scale<T>::V) * gcomp<T>(a, 1)), gz(T(Scale<T>::V) * gcomp<T>(a, 2))
    {
    }
    __device__ __forceinline__ T r(T d) const { return fma(T(Scale<T>::R), d, T(Scale<T>::R)); }
    __device__ __forceinline__ T vx(T u) const { return fma(T(Scale<T>::V), u, gx); }
    __device__ __forceinline__ T vy(T u) const { return fma(T(Scale<T>::V), u, gy); }
    __device__ __forceinline__ T vz(T u) const { return fma(T(Scale<T>::V), u, gz); }
};

// Values of a record as stored, in the compute type.
template <typename E> struct Rec {
    E d, ux, uy, uz;
};
template <int ST> __device__ __forceinline__ Rec<typename Storage<ST>::ctype> record(const void* base, uint32_t i)
{
    const float one[4] = {1.f, 1.f, 1.f, 1.f};
    Rec<typename Storage<ST>::ctype> r;
    Storage<ST>::load(base, i, one, r.d, r.ux, r.uy, r.uz);
    return r;
}
template <int ST> __device__ __forceinline__ Rec<typename Storage<ST>::ctype> record_at(const void* p)
{
    const float one[4] = {1.f, 1.f, 1.f, 1.f};
    Rec<typename Storage<ST>::ctype> r;
    Storage<ST>::load_at(p, one, r.d, r.ux, r.uy, r.uz);
    return r;
}

// Moments of one source record; a wall (solid) has none.
template <int ST, typename T>
__device__ __forceinline__ Moments<T> moments_of(const Rec<T>& c, const Terms<ST>& t, bool solid)
{
    const T vx = t.vx(c.ux), vy = t.vy(c.uy), vz = t.vz(c.uz), A = less_trace<T>(c.d, vx, vy, vz);
    return {solid ? T(0) : A, solid ? T(0) : t.r(c.d), vx, vy, vz};
}

// c.v for a constant direction c (axis order x, y, z).
template <int CX, int CY, int CZ, typename T> __device__ __forceinline__ T dir_sum(T Px, T Py, T Pz)
{
    T p = T(0);
    if constexpr (CX != 0) p = CX > 0 ? Px : -Px;
    if constexpr (CY != 0) {
        if constexpr (CX == 0) p = CY > 0 ? Py : -Py;
        else p = CY > 0 ? p + Py : p - Py;
    }
    if constexpr (CZ != 0) {
        if constexpr (CX == 0 && CY == 0) p = CZ > 0 ? Pz : -Pz;
        else p = CZ > 0 ? p + Pz : p - Pz;
    }
    return p;
}

// One plane of one column, by lattice.
//   NV: values a row sends to the row above (up) and below (dn);
//   Mid: what the y sum of the own row takes besides;
//   NP, NO: values a plane sends to the next plane (P) or the one before (M),
//   and keeps (O), after the y sum.
// Units: 1/36 (D3Q19: weights 12, 2, 1) and 1/216 (D3Q27: 64, 16, 4, 1).
template <int Q> struct Sums;

template <> struct Sums<19> {
    static constexpr int NV = 5, NP = 4, NO = 6;
    static constexpr double ONE = 36.0, UNIT = 1.0 / ONE;
    __host__ __device__ static constexpr int weight(int cls) { return cls == 0 ? 12 : (cls == 1 ? 2 : 1); }
    template <typename T> struct Mid {
        T A, fxp, fxm, fzp, fzm, xpp, xpm, xmp, xmm;
    };
    // up: (1,1,0) (-1,1,0) (0,1,0) (0,1,1) (0,1,-1); dn: the same with c_y = -1
    template <typename T>
    __device__ static __forceinline__ void in_plane(const Moments<T>& m, Mid<T>& c, T (&up)[NV], T (&dn)[NV])
    {
        c.A = m.A;
        // the values along +-c from q = c.v: A + p q + L p and A + p q - L p, p = r q
        auto along = [&](T q, T& fp, T& fm) {
            const T p = product(m.r, q), e = fma(p, q, m.A);
            fp = fma(T(Scale<T>::L), p, e);
            fm = fma(T(-Scale<T>::L), p, e);
        };
        along(m.vx, c.fxp, c.fxm);
        along(m.vy, up[2], dn[2]);
        along(m.vz, c.fzp, c.fzm);
        along(m.vx + m.vy, up[0], dn[1]);
        along(m.vx - m.vy, dn[0], up[1]);
        along(m.vx + m.vz, c.xpp, c.xmm);
        along(m.vx - m.vz, c.xpm, c.xmp);
        along(m.vy + m.vz, up[3], dn[4]);
        along(m.vy - m.vz, up[4], dn[3]);
    }
    // S: up values of row y - 1, N: dn values of row y + 1
    template <typename T>
    __device__ static __forceinline__ void y_sum(const Mid<T>& c, const T (&S)[NV], const T (&N)[NV], T (&P)[NP],
                                                 T (&O)[NO], T (&M)[NP])
    {
        O[0] = fma(T(2), c.fxp, S[0] + N[0]);
        O[1] = S[0] - N[0];
        O[2] = fma(T(2), c.fxm, S[1] + N[1]);
        O[3] = S[1] - N[1];
        O[4] = fma(T(6), c.A, S[2] + N[2]);
        O[5] = S[2] - N[2];
        P[0] = c.xpp;
        P[1] = c.xmp;
        P[2] = fma(T(2), c.fzp, S[3] + N[3]);
        P[3] = S[3] - N[3];
        M[0] = c.xpm;
        M[1] = c.xmm;
        M[2] = fma(T(2), c.fzm, S[4] + N[4]);
        M[3] = S[4] - N[4];
    }
    // z sums of plane z, begun with P of plane z - 1 and O of plane z, ended with
    // M of plane z + 1; X, Y: {density, y, z sums} sent to x + 1 and x - 1, C: those kept
    template <typename T>
    __device__ static __forceinline__ void z_begin(const T (&P)[NP], const T (&O)[NO], T (&Z)[9])
    {
        Z[0] = O[0] + P[0];
        Z[1] = O[1];
        Z[2] = P[0];
        Z[3] = O[2] + P[1];
        Z[4] = O[3];
        Z[5] = P[1];
        Z[6] = fma(T(2), O[4], P[2]);
        Z[7] = fma(T(2), O[5], P[3]);
        Z[8] = P[2];
    }
    template <typename T>
    __device__ static __forceinline__ void z_end(const T (&Z)[9], const T (&M)[NP], T (&X)[3], T (&Y)[3], T (&C)[3])
    {
        X[0] = Z[0] + M[0];
        X[1] = Z[1];
        X[2] = Z[2] - M[0];
        Y[0] = Z[3] + M[1];
        Y[1] = Z[4];
        Y[2] = Z[5] - M[1];
        C[0] = Z[6] + M[2];
        C[1] = Z[7] + M[3];
        C[2] = Z[8] - M[2];
    }
    template <typename T> __device__ static __forceinline__ T x_sum(T c, T x, T y) { return c + (x + y); }
};

template <> struct Sums<27> {
    static constexpr int NV = 7, NP = 6, NO = 6;
    static constexpr double ONE = 216.0, UNIT = 1.0 / ONE;
    __host__ __device__ static constexpr int weight(int cls)
    {
        return cls == 0 ? 64 : (cls == 1 ? 16 : (cls == 2 ? 4 : 1));
    }
    // per c_z (0, +1, -1) the part of c.P and c.Q.c that c_x = 0 and c_x = +-1 take
    template <typename T> struct Mid {
        T a[3], b[3], q;
    };
    template <typename T>
    __device__ static __forceinline__ void in_plane(const Moments<T>& m, Mid<T>& c, T (&up)[NV], T (&dn)[NV])
    {
        const T L = T(Scale<T>::L), mL = T(-Scale<T>::L);
        const T Px = product(m.r, m.vx), Py = product(m.r, m.vy), Pz = product(m.r, m.vz);
        const T Lx = product(L, Px), Ly = product(L, Py);
        const T ez = fma(Pz, m.vz, m.A), qx = product(Px, m.vx);
        const T qxy = Px * m.vy, qxz = Px * m.vz, qyz = Py * m.vz;
        c.a[0] = m.A;
        c.a[1] = fma(L, Pz, ez);
        c.a[2] = fma(mL, Pz, ez);
        c.b[0] = Lx;
        c.b[1] = fma(T(2), qxz, Lx);
        c.b[2] = fma(T(-2), qxz, Lx);
        const T y[3] = {Ly, fma(T(2), qyz, Ly), fma(T(-2), qyz, Ly)};
        c.q = qx;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const T e = fma(Py, m.vy, c.a[j]);
            up[2 * j] = e + y[j];
            dn[2 * j] = e - y[j];
            up[2 * j + 1] = fma(T(2), qxy, c.b[j]);
            dn[2 * j + 1] = fma(T(-2), qxy, c.b[j]);
        }
        up[6] = qx;
        dn[6] = qx;
    }
    template <typename T>
    __device__ static __forceinline__ void y_sum(const Mid<T>& c, const T (&S)[NV], const T (&N)[NV], T (&P)[NP],
                                                 T (&O)[NO], T (&M)[NP])
    {
        auto line = [&](int j, T (&R)[NP]) {
            R[0] = fma(T(4), c.a[j], S[2 * j] + N[2 * j]);
            R[1] = fma(T(4), c.b[j], S[2 * j + 1] + N[2 * j + 1]);
            R[2] = S[2 * j] - N[2 * j];
            R[3] = S[2 * j + 1] - N[2 * j + 1];
        };
        line(0, O);
        line(1, P);
        line(2, M);
        O[4] = P[4] = M[4] = fma(T(4), c.q, S[6] + N[6]);
        O[5] = P[5] = M[5] = S[6] - N[6];
    }
    template <typename T>
    __device__ static __forceinline__ void z_begin(const T (&P)[NP], const T (&O)[NO], T (&Z)[9])
    {
        Z[0] = fma(T(4), O[0], P[0]);
        Z[1] = fma(T(4), O[1], P[1]);
        Z[2] = fma(T(4), O[4], P[4]);
        Z[3] = fma(T(4), O[2], P[2]);
        Z[4] = fma(T(4), O[3], P[3]);
        Z[5] = fma(T(4), O[5], P[5]);
        Z[6] = P[0];
        Z[7] = P[1];
        Z[8] = P[4];
    }
    template <typename T>
    __device__ static __forceinline__ void z_end(const T (&Z)[9], const T (&M)[NP], T (&X)[3], T (&Y)[3], T (&C)[3])
    {
        auto side = [&](int j, T a, T b, T q) {
            const T e = a + q;
            X[j] = e + b;
            Y[j] = e - b;
            C[j] = a;
        };
        side(0, Z[0] + M[0], Z[1] + M[1], Z[2] + M[4]);
        side(1, Z[3] + M[2], Z[4] + M[3], Z[5] + M[5]);
        side(2, Z[6] - M[0], Z[7] - M[1], Z[8] - M[4]);
    }
    template <typename T> __device__ static __forceinline__ T x_sum(T c, T x, T y) { return fma(T(4), c, x + y); }
};

// The z march of one column: what the planes so far leave for the next ones.
template <int Q, typename T> struct March {
    using S = Sums<Q>;
    T Z[9];      // sums of the previous plane, all but the M of this one
    T P[S::NP];  // P of the previous plane
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int j = 0; j < 9; ++j) Z[j] = T(0);
#pragma unroll
        for (int j = 0; j < S::NP; ++j) P[j] = T(0);
    }
    // the sums of the previous plane from P, O and M of this one
    __device__ __forceinline__ void advance(const T (&p)[S::NP], const T (&o)[S::NO], const T (&m)[S::NP], T (&X)[3],
                                            T (&Y)[3], T (&C)[3])
    {
        S::z_end(Z, m, X, Y, C);
        S::z_begin(P, o, Z);
#pragma unroll
        for (int j = 0; j < S::NP; ++j) P[j] = p[j];
    }
};

// Density and momentum sums of a node: C its own, X those of column x - 1, Y those of x + 1.
template <int Q, typename T>
__device__ __forceinline__ void node_sums(const T (&C)[3], const T (&X)[3], const T (&Y)[3], T (&s)[4])
{
    s[0] = Sums<Q>::x_sum(C[0], X[0], Y[0]);
    s[1] = X[0] - Y[0];
    s[2] = Sums<Q>::x_sum(C[1], X[1], Y[1]);
    s[3] = Sums<Q>::x_sum(C[2], X[2], Y[2]);
}

// 1 / x for x near ONE. The hardware's FP32 approximation is one-sided there, and
// the same side every step: a channel's momentum drifted by 2e-6 in 100 steps.
// One Newton step takes the bias out.
template <typename T> __device__ __forceinline__ T recip_unbiased(T x, T minus_x)
{
    const T r = recip(x);
    if constexpr (IsFp64<T>::value) return r;
    else return fma(r, fma(minus_x, r, T(1)), r);
}

// The new (drho, u) from the sums: one reciprocal (Algorithm "Optimized Tau1
// ... stores velocity"), of rho in the sums' unit, so that the rounded unit
// enters no velocity.
template <int Q, typename T>
__device__ __forceinline__ void node_state(const T (&s)[4], T& d, T& ux, T& uy, T& uz)
{
    d = T(Sums<Q>::UNIT) * s[0];
    const T r = recip_unbiased(T(Sums<Q>::ONE) + s[0], T(-Sums<Q>::ONE) - s[0]);
    ux = s[1] * r;
    uy = s[2] * r;
    uz = s[3] * r;
}

// Moments of a pair of records in the lanes of L (f2 or d2, pack2.cuh), solid
// where sA or sB; MIRROR 1 (2) mirrors lane B in x (y), which gives the same
// values with the directions exchanged.
template <int MIRROR, int ST, typename L, typename E>
__device__ __forceinline__ Moments<L> pair_moments(const Rec<E>& a, const Rec<E>& b, const Terms<ST>& t, bool sA, bool sB)
{
    const L r = L(sA ? E(0) : t.r(a.d), sB ? E(0) : t.r(b.d));
    L vx = L(t.vx(a.ux), t.vx(b.ux));
    L vy = L(t.vy(a.uy), t.vy(b.uy));
    const L vz = L(t.vz(a.uz), t.vz(b.uz));
    if constexpr (MIRROR == 1) vx.v.y = -vx.v.y;
    if constexpr (MIRROR == 2) vy.v.y = -vy.v.y;
    const L A = less_trace<L>(L(a.d, b.d), vx, vy, vz);
    return {L(sA ? E(0) : A.v.x, sB ? E(0) : A.v.y), r, vx, vy, vz};
}

// Direction index of a velocity (-1: none).
__host__ __device__ constexpr int kdir(int cx, int cy, int cz)
{
    for (int k = 0; k < 27; ++k)
        if (cvel(k, 0) == cx && cvel(k, 1) == cy && cvel(k, 2) == cz) return k;
    return -1;
}

// Bit of the source at offset (dx, dy, dz) in a node's 27-bit neighbour mask
// (bit set: that neighbour is a wall).
__host__ __device__ constexpr int nbit(int dx, int dy, int dz) { return 9 * (dx + 1) + 3 * (dz + 1) + (dy + 1); }

// What the wall links of a node add to its sums: its own equilibria in
// direction inv(k), travelling along c_k. with(k, v, add) calls add(v) where
// link k is a wall, or add(0) or nothing elsewhere.
template <int Q, typename T, typename F>
__device__ __forceinline__ void bounce(const Moments<T>& m, F&& with, T (&B)[4])
{
    B[0] = B[1] = B[2] = B[3] = T(0);
    static_for<0, (Q - 1) / 2>([&](auto ic) {
        constexpr int K = 1 + 2 * decltype(ic)::value;  // K + 1 = inv(K)
        constexpr int cx = cvel(K, 0), cy = cvel(K, 1), cz = cvel(K, 2);
        constexpr int WI = Sums<Q>::weight(dir_class(K));
        const T q = dir_sum<cx, cy, cz>(m.vx, m.vy, m.vz), p = product(m.r, q), e = fma(p, q, m.A);
        // link K receives f(inv K) = e - L p, link inv(K) receives f(K) = e + L p
        auto add = [&](T b, auto sc) {
            constexpr int s = decltype(sc)::value;
            B[0] = fma(T(WI), b, B[0]);
            if constexpr (cx != 0) B[1] = fma(T(WI * cx * s), b, B[1]);
            if constexpr (cy != 0) B[2] = fma(T(WI * cy * s), b, B[2]);
            if constexpr (cz != 0) B[3] = fma(T(WI * cz * s), b, B[3]);
        };
        with(std::integral_constant<int, K>{}, fma(T(-Scale<T>::L), p, e), [&](T b) { add(b, std::integral_constant<int, 1>{}); });
        with(std::integral_constant<int, K + 1>{}, fma(T(Scale<T>::L), p, e), [&](T b) { add(b, std::integral_constant<int, -1>{}); });
    });
}

// Adds them where there are any.
template <int Q, typename T>
__device__ __forceinline__ void add_bounce(const Moments<T>& own, uint32_t wall, T (&s)[4])
{
    if (wall == 0u) return;
    T B[4];
    bounce<Q, T>(own, [&](auto kc, T v, auto&& add) {
        constexpr int K = decltype(kc)::value;
        if (wall & (1u << nbit(-cvel(K, 0), -cvel(K, 1), -cvel(K, 2)))) add(v);
    }, B);
#pragma unroll
    for (int f = 0; f < 4; ++f) s[f] = s[f] + B[f];
}

// The sums of one column of nine sources: at(dy, dz) gives their moments.
template <int Q, typename T, typename F>
__device__ __forceinline__ void column_sums(F&& at, T (&X)[3], T (&Y)[3], T (&C)[3])
{
    using S = Sums<Q>;
    T P[S::NP], O[S::NO], M[S::NP];
    static_for<0, 3>([&](auto zc) {
        constexpr int DZ = decltype(zc)::value - 1;
        using IZ = std::integral_constant<int, DZ>;
        typename S::template Mid<T> c, skip;
        T up[S::NV], dn[S::NV], none[S::NV];
        S::in_plane(at(std::integral_constant<int, 0>{}, IZ{}), c, none, none);
        S::in_plane(at(std::integral_constant<int, -1>{}, IZ{}), skip, up, none);
        S::in_plane(at(std::integral_constant<int, 1>{}, IZ{}), skip, none, dn);
        T p[S::NP], o[S::NO], m[S::NP];
        S::y_sum(c, up, dn, p, o, m);
#pragma unroll
        for (int j = 0; j < S::NP; ++j) {
            if (DZ == -1) P[j] = p[j];
            if (DZ == 1) M[j] = m[j];
        }
#pragma unroll
        for (int j = 0; j < S::NO; ++j)
            if (DZ == 0) O[j] = o[j];
    });
    T z[9];
    S::z_begin(P, O, z);
    S::z_end(z, M, X, Y, C);
}

// The same update gathered by one thread: fetch(k, solid) gives the record of the
// source x - c_k and whether it is a wall, own the moments of the node itself. In
// D3Q19 the columns on both sides share the lanes of packed arithmetic, the right
// one mirrored in x (9.9 M listed nodes 221 us, 231 without); D3Q27 has no
// registers for that (1.8 M sparse nodes 110 us, 74 without).
template <int Q, int ST, typename T, typename F>
__device__ __forceinline__ void gather_sums(const Terms<ST>& t, const Moments<T>& own, F&& fetch, T (&s)[4])
{
    T X[3], Y[3], C[3], skipA[3], skipB[3];
    auto column = [&](auto xc, T (&X)[3], T (&Y)[3], T (&C)[3]) {
        column_sums<Q, T>([&](auto yc, auto zc) -> Moments<T> {
            constexpr int K = kdir(-decltype(xc)::value, -decltype(yc)::value, -decltype(zc)::value);
            if constexpr (K == 0) {
                return own;
            } else if constexpr (K < Q) {
                bool w;
                const Rec<T> r = fetch(std::integral_constant<int, K>{}, w);
                return moments_of<ST, T>(r, t, w);
            } else {
                return Moments<T>{};  // no such link: its values are not used
            }
        }, X, Y, C);
    };
    if constexpr (Q == 19) {
        using L = typename Lanes<T>::type;
        L sides[3], skipX[3], skipC[3];
        column_sums<Q, L>([&](auto yc, auto zc) -> Moments<L> {
            constexpr int K = kdir(1, -decltype(yc)::value, -decltype(zc)::value);
            constexpr int KR = kdir(-1, -decltype(yc)::value, -decltype(zc)::value);
            if constexpr (K < Q) {
                bool sA, sB;
                const Rec<T> a = fetch(std::integral_constant<int, K>{}, sA);
                const Rec<T> b = fetch(std::integral_constant<int, KR>{}, sB);
                return pair_moments<1, ST, L>(a, b, t, sA, sB);
            } else {
                return Moments<L>{};
            }
        }, sides, skipX, skipC);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            X[j] = sides[j].v.x;
            Y[j] = sides[j].v.y;
        }
    } else {
        column(std::integral_constant<int, -1>{}, X, skipA, skipB);
    }
    T skip[3];
    column(std::integral_constant<int, 0>{}, skipA, skipB, C);
    if constexpr (Q != 19) column(std::integral_constant<int, 1>{}, skipA, Y, skip);
    node_sums<Q, T>(C, X, Y, s);
}

}  // namespace lbm
