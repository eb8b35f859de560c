// Tau1 step kernel of one dense box: a warp per strip (strip.cuh), the strips in
// chunk-major order so that those of a chunk run side by side and read each
// other's outer rows from L2. Every size, periodicity and storage format takes
// this kernel; the compact layout runs it over a list of strips.
#include "strip.cuh"

namespace lbm {

namespace {

using namespace col;

// LIST: per strip 32 slots, negative (~slot) where the lane does not own its column,
// and the chunk; else the strips of the whole box, chunk-major.
template <int Q, int ST, int R, int MINB, bool LIST>
__global__ void __launch_bounds__(Cfg<Q, ST, R>::NT, 4 * MINB / Cfg<Q, ST, R>::W)
    tau1_strip_kernel(StepArgs a, int nstrips, int count, int chunk, const int* __restrict__ list)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = uniform((int)(threadIdx.x >> 5)), i = Cfg<Q, ST, R>::W * (int)blockIdx.x + warp;
    if constexpr (LIST) asm volatile("griddepcontrol.launch_dependents;");  // the node list of this step: other nodes
    if (i >= count) return;
    Place pl;
    int c;
    if constexpr (LIST) {
        const int* item = list + (size_t)i * STRIP_ITEM;
        const int v = item[threadIdx.x & 31];
        pl = place_of_slot<R>(a, (uint32_t)(v < 0 ? ~v : v), v >= 0);
        c = uniform(item[32]);
    } else {
        c = i / nstrips;
        pl = place_of_strip<R>(a, i - c * nstrips);
    }
    const int z0 = c * chunk, z1 = a.nz - z0 < chunk ? a.nz : z0 + chunk;
    unsigned char* const mine = smem + warp * Cfg<Q, ST, R>::WARP;
    if constexpr (by_links(ST)) {
        float amax[4];
        strip_links<Q, ST, R, false>(a, Scales(a.dscale), pl, z0, z1, mine, amax);
    } else {
        strip_step<Q, ST, R>(a, pl, z0, z1, mine);
    }
    // a launch that began before the node-list kernel had ended ends after it
    if constexpr (LIST) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// strip_plan.h prices the shapes that strip.cuh has
template <int Q, int ST, int V> constexpr bool priced()
{
    constexpr StripShapeCost c = strip_shape(Q, ST, V);
    return c.rows == StripShape<Q, ST, V>::R && c.minb == StripShape<Q, ST, V>::MINB;
}

template <int Q, int ST, int V, bool LIST>
cudaError_t launch_t(const StepArgs& a, int zchunk, cudaStream_t s, const int* list, int count, int after_list)
{
    using Sh = StripShape<Q, ST, V>;
    using C = Cfg<Q, ST, Sh::R>;
    static_assert(C::SMEM <= 227 * 1024, "shared memory of one block");
    static_assert(priced<Q, ST, V>(), "shape of the plan");
    auto kern = tau1_strip_kernel<Q, ST, Sh::R, Sh::MINB, LIST>;
    // the attribute is per device; setting it on every launch is cheap
    constexpr int MOST = LIST ? 226 * 1024 : C::SMEM;  // list: an SM's shared memory, less 2 KB
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, MOST);
    if (e != cudaSuccess) return e;
    const int64_t strips = strips_of(a.nx, a.ny, a.periodic[0], C::R);
    const int chunk = a.nz < zchunk ? a.nz : zchunk;
    const int64_t n = LIST ? (int64_t)count : strips * (((int64_t)a.nz + chunk - 1) / chunk);
    if (n > 0x7fffffffLL - C::W) return cudaErrorInvalidConfiguration;
    if (n == 0) return cudaSuccess;
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((n + C::W - 1) / C::W));
    cfg.blockDim = dim3(C::NT);
    cfg.dynamicSmemBytes = C::SMEM;
    // Blocks that start as the list's end would crowd on the SMs that come free
    // first: no more on an SM than an even share (192^3, 30% fluid 72.0 -> 61.6 us).
    if (LIST && ST == ST_F32 && after_list > 0) {
        const int share = (int)((cfg.gridDim.x + (unsigned)after_list - 1) / (unsigned)after_list);
        if (share < Sh::MINB) cfg.dynamicSmemBytes = (size_t)(MOST / share - 1024) / 16 * 16;
    }
    cfg.stream = s;
    cfg.attrs = &overlap;
    cfg.numAttrs = after_list ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, a, (int)strips, (int)n, chunk, list);
}

template <int Q, int ST>
cudaError_t launch_s(int shape, int zchunk, const StepArgs& a, cudaStream_t s, const int* list, int count, int after_list)
{
    auto go = [&](auto vc) {
        constexpr int V = decltype(vc)::value;
        // the compact layout takes shapes 0 and 1
        if constexpr (V < 2)
            if (list) return launch_t<Q, ST, V, true>(a, zchunk, s, list, count, after_list);
        return list ? cudaErrorInvalidValue : launch_t<Q, ST, V, false>(a, zchunk, s, nullptr, 0, 0);
    };
    if constexpr (ST == ST_F64) {
        return shape == 0 ? go(std::integral_constant<int, 0>{}) : cudaErrorInvalidValue;
    } else {
        switch (shape) {
        case 0: return go(std::integral_constant<int, 0>{});
        case 1: return go(std::integral_constant<int, 1>{});
        case 2: return go(std::integral_constant<int, 2>{});
        default: return cudaErrorInvalidValue;
        }
    }
}

cudaError_t launch(int q, int storage, int shape, int zchunk, const StepArgs& a, cudaStream_t s, const int* list,
                   int count, int after_list)
{
    switch (q * 10 + storage) {
    case 190 + ST_F64: return launch_s<19, ST_F64>(shape, zchunk, a, s, list, count, after_list);
    case 190 + ST_F32: return launch_s<19, ST_F32>(shape, zchunk, a, s, list, count, after_list);
    case 190 + ST_F16S: return launch_s<19, ST_F16S>(shape, zchunk, a, s, list, count, after_list);
    case 190 + ST_BF16S: return launch_s<19, ST_BF16S>(shape, zchunk, a, s, list, count, after_list);
    case 270 + ST_F64: return launch_s<27, ST_F64>(shape, zchunk, a, s, list, count, after_list);
    case 270 + ST_F32: return launch_s<27, ST_F32>(shape, zchunk, a, s, list, count, after_list);
    case 270 + ST_F16S: return launch_s<27, ST_F16S>(shape, zchunk, a, s, list, count, after_list);
    case 270 + ST_BF16S: return launch_s<27, ST_BF16S>(shape, zchunk, a, s, list, count, after_list);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// A strip counts its planes up to nz in 32 bits: not for 2^31 - 1 of them.
bool tau1_tiled_supported(int q, int storage, int64_t n)
{
    return (q == 19 || q == 27) && storage >= ST_F64 && storage <= ST_BF16S && n > 0 && n < ((int64_t)1 << 31) - 1;
}

int tau1_tile_shapes(int storage) { return strip_shapes(storage); }

int tau1_tiled_variants(int, int storage) { return 4 * strip_shapes(storage); }

cudaError_t launch_tau1_tiled(int q, int storage, const StripPlan& plan, const StepArgs& a, cudaStream_t s)
{
    return launch(q, storage, plan.shape, plan.chunk, a, s, nullptr, 0, 0);
}

cudaError_t launch_tau1_tiled_list(int q, int storage, int shape, int zchunk, const StepArgs& a, const int* list,
                                   int count, int after_list, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    if (!list) return cudaErrorInvalidValue;
    return launch(q, storage, shape, zchunk, a, s, list, count, after_list);
}

}  // namespace lbm
