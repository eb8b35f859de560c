// Tau1 step kernel of one dense box: a warp per strip (strip.cuh), the strips in
// chunk-major order so that those of a chunk run side by side and read each
// other's outer rows from L2. Every size, periodicity and storage format takes
// this kernel; the compact layout runs it over a list of strips.
#include "strip.cuh"

namespace lbm {

namespace {

using namespace col;

// list (or NULL): per strip 32 slots, negative (~slot) where the lane does not own
// its column, and the chunk; else the strips of the whole box, chunk-major.
template <int Q, int ST, int R, int MINB>
__global__ void __launch_bounds__(128, MINB)
    tau1_strip_kernel(StepArgs a, int nstrips, int count, int chunk, const int* __restrict__ list)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = uniform((int)(threadIdx.x >> 5)), i = 4 * (int)blockIdx.x + warp;
    if (i >= count) return;
    Place pl;
    int c;
    if (list) {
        const int* item = list + (size_t)i * STRIP_ITEM;
        const int v = item[threadIdx.x & 31];
        pl = place_of_slot<R>(a, (uint32_t)(v < 0 ? ~v : v), v >= 0);
        c = uniform(item[32]);
    } else {
        c = i / nstrips;
        pl = place_of_strip<R>(a, i - c * nstrips);
    }
    const int z0 = c * chunk, z1 = min(a.nz, z0 + chunk);
    const Scales sc(a.dscale);
    float amax[4];
    strip_step<Q, ST, R, false>(a, sc, pl, z0, z1, smem + warp * Cfg<Q, ST, R>::WARP, amax);
    // a launch that began before the node-list kernel had ended ends after it
    if (list) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Planes per block for a box of `tiles` tiles when the GPU holds `resident`
// blocks: the chunk with the least (waves of blocks) x (planes a block forms),
// a block forming two planes beside its own and about as much again to start.
int whole_waves(int nz, long long tiles, long long resident)
{
    int best = nz;
    long long best_cost = -1;
    for (int n = 1; n <= nz;) {
        const int chunk = (nz + n - 1) / n, used = (nz + chunk - 1) / chunk;
        const long long cost = ((tiles * used + resident - 1) / resident) * (chunk + 4);
        if (best_cost < 0 || cost < best_cost) {
            best = chunk;
            best_cost = cost;
        }
        n = chunk == 1 ? nz + 1 : (nz + chunk - 2) / (chunk - 1);  // the next smaller chunk
    }
    return best;
}

template <int Q, int ST, int V>
cudaError_t launch_t(const StepArgs& a, int zchunk, cudaStream_t s, const int* list, int count, bool after_list)
{
    using Sh = ColShape<Q, typename Storage<ST>::ctype, V>;
    using C = Cfg<Q, ST, Sh::R>;
    static_assert(C::SMEM <= 227 * 1024, "shared memory of one block");
    auto kern = tau1_strip_kernel<Q, ST, Sh::R, Sh::MINB>;
    // the attribute is per device; setting it on every launch is cheap
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    const long long strips = strips_of(a.nx, a.ny, a.periodic[0], C::R);
    int chunk = a.nz < zchunk ? a.nz : zchunk;
    if (zchunk == 0) {
        int dev = 0, sms = 0, per_sm = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::NT, C::SMEM);
        if (e != cudaSuccess) return e;
        chunk = whole_waves(a.nz, strips, (long long)sms * C::W * (per_sm > 0 ? per_sm : 1));
    }
    const int nchunks = (a.nz + chunk - 1) / chunk;
    const long long n = list ? (long long)count : strips * nchunks;
    if (n > 0x7fffffffLL - C::W) return cudaErrorInvalidConfiguration;
    if (n == 0) return cudaSuccess;
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((n + C::W - 1) / C::W));
    cfg.blockDim = dim3(C::NT);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = s;
    cfg.attrs = &overlap;
    cfg.numAttrs = after_list ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, a, (int)strips, (int)n, chunk, list);
}

template <int Q, int ST>
cudaError_t launch_s(int shape, int zchunk, const StepArgs& a, cudaStream_t s, const int* list, int count, bool after_list)
{
    if constexpr (ST == ST_F64) {
        return shape == 0 ? launch_t<Q, ST, 0>(a, zchunk, s, list, count, after_list) : cudaErrorInvalidValue;
    } else {
        switch (shape) {
        case 0: return launch_t<Q, ST, 0>(a, zchunk, s, list, count, after_list);
        case 1: return launch_t<Q, ST, 1>(a, zchunk, s, list, count, after_list);
        case 2: return launch_t<Q, ST, 2>(a, zchunk, s, list, count, after_list);
        case 3: return launch_t<Q, ST, 3>(a, zchunk, s, list, count, after_list);
        default: return cudaErrorInvalidValue;
        }
    }
}

cudaError_t launch(int q, int storage, int shape, int zchunk, const StepArgs& a, cudaStream_t s, const int* list,
                   int count, bool after_list)
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

constexpr int CHUNKS[4] = {0, 32, 16, 48};  // planes per block; 0: whole waves of blocks

}  // namespace

bool tau1_tiled_supported(int q, int storage, int64_t n)
{
    return (q == 19 || q == 27) && storage >= ST_F64 && storage <= ST_BF16S && n > 0 && n < ((int64_t)1 << 31);
}

int tau1_tile_shapes(int storage) { return storage == ST_F64 ? 1 : COL_SHAPES; }

int tau1_tiled_variants(int, int storage) { return 4 * tau1_tile_shapes(storage); }

int tau1_strip_rows(int storage, int shape)
{
    if (storage == ST_F64) return ColShape<19, double, 0>::R;
    return shape == 0 || shape == 2 ? ColShape<19, float, 0>::R : ColShape<19, float, 1>::R;
}

cudaError_t launch_tau1_tiled(int q, int storage, int variant, const StepArgs& a, cudaStream_t s)
{
    const int nr = tau1_tile_shapes(storage);
    if (variant < 0 || variant >= 4 * nr) return cudaErrorInvalidValue;
    return launch(q, storage, nr == 1 ? 0 : dense_shape(variant % nr), CHUNKS[variant / nr], a, s, nullptr, 0, false);
}

cudaError_t launch_tau1_tiled_list(int q, int storage, int shape, int zchunk, const StepArgs& a, const int* list,
                                   int count, bool after_list, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    if (!list) return cudaErrorInvalidValue;
    return launch(q, storage, shape, zchunk, a, s, list, count, after_list);
}

}  // namespace lbm
