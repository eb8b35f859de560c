// Tau1 step, one thread per node, neighbours read straight from global memory.
//
// The plain form of Algorithm "Tau1" (pull, AB layout) with the halfway
// bounce-back of Algorithm "Complete Tau1 ... halfway bounce-back": the node
// reads every source's record, forms its moments and takes the sums of
// moments.cuh, or of links.cuh; wall links bring the node's own equilibria. It serves any box
// shape and every storage format and is the cross-check of the tiled kernel,
// which evaluates the same functions in the same order: both give the same bits.
#include "kernels.h"
#include "links.cuh"
#include "moments.cuh"

namespace lbm {

template <int Q, int ST>
__global__ void __launch_bounds__(256) tau1_simple_kernel(StepArgs a)
{
    using T = typename Storage<ST>::ctype;
    const int64_t n = (int64_t)a.nx * a.ny * a.nz;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Scales sc(a.dscale);
    T d0, ux0, uy0, uz0;
    Storage<ST>::load(a.pre, (uint32_t)i, sc.inv, d0, ux0, uy0, uz0);
    if (isnan(d0)) return;  // solid node
    const int x = (int)(i % a.nx);
    const int y = (int)((i / a.nx) % a.ny);
    const int z = (int)(i / ((int64_t)a.nx * a.ny));
    auto load = [&](auto kc, bool& solid, T& d, T& ux, T& uy, T& uz) {
        constexpr int K = decltype(kc)::value;
        int sx = x - cvel(K, 0), sy = y - cvel(K, 1), sz = z - cvel(K, 2);
        bool inside = true;
        if (sx < 0 || sx >= a.nx) { if (a.periodic[0]) sx = sx < 0 ? sx + a.nx : sx - a.nx; else inside = false; }
        if (sy < 0 || sy >= a.ny) { if (a.periodic[1]) sy = sy < 0 ? sy + a.ny : sy - a.ny; else inside = false; }
        if (sz < 0 || sz >= a.nz) { if (a.periodic[2]) sz = sz < 0 ? sz + a.nz : sz - a.nz; else inside = false; }
        d = T(NAN);
        ux = uy = uz = T(0);
        if (inside) {
            const int64_t s = (int64_t)sx + (int64_t)a.nx * ((int64_t)sy + (int64_t)a.ny * sz);
            Storage<ST>::load(a.pre, (uint32_t)s, sc.inv, d, ux, uy, uz);
        }
        solid = isnan(d);
    };
    T d, ux, uy, uz;
    if constexpr (by_links(ST)) {
        gather_links<Q, false>(a, d0, ux0, uy0, uz0, load, d, ux, uy, uz);
    } else {
        const Terms<ST> t(a);
        const Moments<T> own = moments_of<ST, T>({d0, ux0, uy0, uz0}, t, false);
        uint32_t wall = 0;
        T sums[4];
        gather_sums<Q, ST>(t, own, [&](auto kc, bool& solid) {
            constexpr int K = decltype(kc)::value;
            Rec<T> c;
            load(kc, solid, c.d, c.ux, c.uy, c.uz);
            if (solid) wall |= 1u << nbit(-cvel(K, 0), -cvel(K, 1), -cvel(K, 2));
            return c;
        }, sums);
        add_bounce<Q, T>(own, wall, sums);
        node_state<Q, T>(sums, d, ux, uy, uz);
    }
    step_store<ST>(a.post, (uint32_t)i, d, ux, uy, uz, sc.s, a.seed);
}

template <int Q, int ST>
static cudaError_t launch_simple_t(const StepArgs& a, cudaStream_t s)
{
    const int64_t n = (int64_t)a.nx * a.ny * a.nz;
    const int64_t blocks = (n + 255) / 256;
    tau1_simple_kernel<Q, ST><<<(unsigned)blocks, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_tau1_simple(int q, int storage, const StepArgs& a, cudaStream_t s)
{
    switch (q * 10 + storage) {
    case 190 + ST_F64: return launch_simple_t<19, ST_F64>(a, s);
    case 190 + ST_F32: return launch_simple_t<19, ST_F32>(a, s);
    case 190 + ST_F16S: return launch_simple_t<19, ST_F16S>(a, s);
    case 190 + ST_BF16S: return launch_simple_t<19, ST_BF16S>(a, s);
    case 270 + ST_F64: return launch_simple_t<27, ST_F64>(a, s);
    case 270 + ST_F32: return launch_simple_t<27, ST_F32>(a, s);
    case 270 + ST_F16S: return launch_simple_t<27, ST_F16S>(a, s);
    case 270 + ST_BF16S: return launch_simple_t<27, ST_BF16S>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
