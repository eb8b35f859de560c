// Tau1 step kernel of one dense box: a warp per strip (strip.cuh), the strips in
// chunk-major order so that those of a chunk run side by side and read each
// other's outer rows from L2. Every size, periodicity and storage format takes
// this kernel; the compact layout runs it over a list of strips.
#include <cmath>

#include "strip.cuh"

namespace lbm {

namespace {

using namespace col;

// list (or NULL): per strip 32 slots, negative (~slot) where the lane does not own
// its column, and the chunk; else the strips of the whole box, chunk-major.
template <int Q, int ST, int R, int MINB>
__global__ void __launch_bounds__(Cfg<Q, ST, R>::NT, 4 * MINB / Cfg<Q, ST, R>::W)
    tau1_strip_kernel(StepArgs a, int nstrips, int count, int chunk, const int* __restrict__ list)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = uniform((int)(threadIdx.x >> 5)), i = Cfg<Q, ST, R>::W * (int)blockIdx.x + warp;
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
    unsigned char* const mine = smem + warp * Cfg<Q, ST, R>::WARP;
    if constexpr (by_links(ST)) {
        float amax[4];
        strip_links<Q, ST, R, false>(a, Scales(a.dscale), pl, z0, z1, mine, amax);
    } else {
        strip_step<Q, ST, R>(a, pl, z0, z1, mine);
    }
    // a launch that began before the node-list kernel had ended ends after it
    if (list) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Time of a step of nz planes in strips of a shape and chunk, up to a factor. A
// chunk of c planes costs its strip c + 4 planes (two beside its own, and as
// much again to start). plane[n] is the time of a plane on an SM with n resident
// blocks: nearly n times one where the SM is full, latency below. In a wave or
// two the fullest SM decides, and strips differ (walls); many waves even out,
// but for the end of the last one.
double step_cost(int nz, long long strips, int chunk, int sms, int minb, const double* plane)
{
    const long long blocks = (strips * ((nz + chunk - 1) / chunk) + STRIP_WARPS - 1) / STRIP_WARPS;
    const double waves = (double)blocks / (sms * minb);
    if (waves <= 1) return (chunk + 4) * 1.15 * plane[(blocks + sms - 1) / sms];
    return (chunk + 4) * plane[minb] * (waves <= 2.5 ? 1.15 * std::ceil(waves) : waves + 0.4);
}

// Time of a plane with 0 .. 4 resident blocks, by format and shape, fitted to
// sweeps of shape and chunk over 11 boxes. Measured, in us, with four rows and
// two: D3Q19 FP32 96^3 16.6 and 14.6, 250 x 130 x 90 34.7 and 33.0, 128^3 24.8 and
// 26.3, 384^3 408 and 428; BF16 512 x 256 x 256 311 and 285; FP16 161 x 127 x 101
// 32.6 and 28.8. Chunks: BF16 512 x 256 x 256 in two rows takes 285 in chunks of
// 48 planes, 294 of 32, 312 of 16, 333 of 256 (one wave).
constexpr double PLANE_F32[STRIP_SHAPES][5] = {{0, 0.95, 1.3, 1.7, 2.1}, {0, 1.6, 2.3, 3.0, 0}, {0, 1.6, 2.3, 0, 0}};
constexpr double PLANE_16[STRIP_SHAPES][5] = {{0, 0.87, 1.2, 1.56, 1.93}, {0, 0.87, 1.2, 1.56, 0}, {0, 1.6, 2.3, 0, 0}};
constexpr double PLANE_F64[5] = {0, 1.2, 2.0, 0, 0};

// Rows per strip and resident blocks per SM of a shape.
struct Shape {
    int rows, minb;
};
template <int Q, int ST> constexpr Shape shape_t(int v)
{
    using S0 = StripShape<Q, ST, 0>;
    if constexpr (ST == ST_F64) {
        return {S0::R, S0::MINB};
    } else {
        using S1 = StripShape<Q, ST, 1>;
        using S2 = StripShape<Q, ST, 2>;
        return v == 0 ? Shape{S0::R, S0::MINB} : (v == 1 ? Shape{S1::R, S1::MINB} : Shape{S2::R, S2::MINB});
    }
}
Shape shape_of(int q, int storage, int v)
{
    if (storage == ST_F64) return q == 19 ? shape_t<19, ST_F64>(v) : shape_t<27, ST_F64>(v);
    if (storage == ST_F32) return q == 19 ? shape_t<19, ST_F32>(v) : shape_t<27, ST_F32>(v);
    return q == 19 ? shape_t<19, ST_F16S>(v) : shape_t<27, ST_F16S>(v);  // both 16-bit formats
}

struct Plan {
    int shape, chunk;
};

// The shape (of first, first - 1 .. last) and chunk of the least cost.
Plan plan_of(const StepArgs& a, int q, int storage, int sms, int first, int last, int chunk)
{
    Plan best{first, chunk};
    double least = -1;
    for (int v = first; v >= last; --v) {
        const Shape sh = shape_of(q, storage, v);
        const double* plane = storage == ST_F64 ? PLANE_F64 : (storage == ST_F32 ? PLANE_F32[v] : PLANE_16[v]);
        const long long strips = strips_of(a.nx, a.ny, a.periodic[0], sh.rows);
        auto take = [&](int c) {
            const double cost = step_cost(a.nz, strips, c, sms, sh.minb, plane);
            if (least < 0 || cost < least) {
                best = {v, c};
                least = cost;
            }
        };
        if (chunk > 0) {
            take(chunk);
            continue;
        }
        for (int n = 1; n <= a.nz;) {
            const int c = (a.nz + n - 1) / n;
            take(c);
            n = c == 1 ? a.nz + 1 : (a.nz + c - 2) / (c - 1);  // the next smaller chunk
        }
    }
    return best;
}

template <int Q, int ST, int V>
cudaError_t launch_t(const StepArgs& a, int zchunk, cudaStream_t s, const int* list, int count, bool after_list)
{
    using Sh = StripShape<Q, ST, V>;
    using C = Cfg<Q, ST, Sh::R>;
    static_assert(C::SMEM <= 227 * 1024, "shared memory of one block");
    auto kern = tau1_strip_kernel<Q, ST, Sh::R, Sh::MINB>;
    // the attribute is per device; setting it on every launch is cheap
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    const long long strips = strips_of(a.nx, a.ny, a.periodic[0], C::R);
    const int chunk = a.nz < zchunk ? a.nz : zchunk;
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

constexpr int CHUNKS[4] = {0, 32, 16, 48};  // planes per chunk; 0: by the box

}  // namespace

bool tau1_tiled_supported(int q, int storage, int64_t n)
{
    return (q == 19 || q == 27) && storage >= ST_F64 && storage <= ST_BF16S && n > 0 && n < ((int64_t)1 << 31);
}

int tau1_tile_shapes(int storage) { return storage == ST_F64 ? 1 : STRIP_SHAPES + 1; }

int tau1_tiled_variants(int, int storage) { return 4 * tau1_tile_shapes(storage); }

int tau1_strip_rows(int q, int storage, int shape) { return shape_of(q, storage, shape).rows; }

cudaError_t launch_tau1_tiled(int q, int storage, int variant, const StepArgs& a, cudaStream_t s)
{
    const int nr = tau1_tile_shapes(storage);
    if (variant < 0 || variant >= 4 * nr) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int v = variant % nr, chunk = CHUNKS[variant / nr];  // v 0: the shape by the box
    // two rows or four in FP32; FP64 has one shape, and link by link the first one
    // is the best or within 2% of it on 12 of 14 boxes
    const Plan p = v > 0 ? plan_of(a, q, storage, sms, v - 1, v - 1, chunk)
                         : plan_of(a, q, storage, sms, storage == ST_F32 ? 1 : 0, 0, chunk);
    return launch(q, storage, p.shape, p.chunk, a, s, nullptr, 0, false);
}

cudaError_t launch_tau1_tiled_list(int q, int storage, int shape, int zchunk, const StepArgs& a, const int* list,
                                   int count, bool after_list, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    if (!list) return cudaErrorInvalidValue;
    return launch(q, storage, shape, zchunk, a, s, list, count, after_list);
}

}  // namespace lbm
