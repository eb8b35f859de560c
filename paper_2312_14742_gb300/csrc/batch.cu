// Batched persistent Tau1 step: many dense boxes of different sizes advance
// one step in one launch.
//
// The work of a step is the list of strips of every live box (box-major, each
// box chunk-major as in the single-box kernel), `chunk` planes high; the host
// picks the chunk that fills whole waves of the grid. A node's result does not
// depend on the chunk. A grid of (SMs x resident blocks) works through the list:
// each warp takes its first item by its index and then the next unclaimed one
// (an atomic counter), so warps that drew small items (partial strips or chunks)
// take more of them. Each item is one strip_step() or strip_links() call with that
// box's arguments, read from the device table. Everything that changes from step to
// step lives in the table on the device: which copy holds a box's current
// state, its step count (the stochastic-rounding seed), its 16-bit scales.
// Boxes of every size take the same strips (strip.cuh). A launch therefore has the
// same arguments every step, and K steps can be captured once in a CUDA graph and
// replayed while boxes come and go (the host edits the table between replays).
//
// The last block to finish (an atomic count, no waiting) closes the step for
// every live box: swaps its copies, counts the step and, for FP16 storage,
// picks the scale of the next written copy by the headroom rule from the
// maxima that the blocks gathered while storing. The state written and the
// scales chosen depend only on the box's own state and step count, so a box
// gives the same bits alone and in any mix.
#include "batch.h"
#include "strip.cuh"

namespace lbm {

namespace {

using namespace col;

__device__ __forceinline__ uint32_t step_seed(int64_t step) { return (uint32_t)(step + 1) * 0x9E3779B9u; }

// Headroom rule of the 16-bit scales (FP16): reference magnitude
// r = max(m_f, max_f' m_f' / 16, 64 |g|_max); S = 2^(12 - e(r)) when
// m_f S > 2^13 or r S < 2^9.
__device__ float decide_scale(const float m[4], int f, float s_old, float gfloor)
{
    const float mall = fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
    const float ref = fmaxf(fmaxf(m[f], 0.0625f * mall), gfloor);
    if (!(ref > 0.f) || !isfinite(mall)) return s_old;
    if (m[f] * s_old <= 8192.f && ref * s_old >= 512.f) return s_old;
    int e;
    frexpf(ref, &e);
    e = 12 - e;
    e = e > 100 ? 100 : (e < -100 ? -100 : e);
    return ldexpf(1.f, e);
}

__device__ void finish_box(BatchDomain& R, int storage)
{
    const uint32_t c = R.cur;
    const int64_t step = R.step + 1;
    if (storage == ST_F16S || storage == ST_BF16S) {
        // buf[c ^ 1] was just written with scale[c ^ 1]; the next step writes buf[c]
        const bool check = storage == ST_F16S && step % BATCH_RESCALE_EVERY == 0;
        float m[4] = {0.f, 0.f, 0.f, 0.f};
        if (check)
#pragma unroll
            for (int f = 0; f < 4; ++f) m[f] = __uint_as_float(atomicExch(&R.amax[f], 0u));
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const float s = check ? decide_scale(m, f, R.scale[c ^ 1][f], R.gfloor) : R.scale[c ^ 1][f];
            R.scale[c][f] = s;
            R.scale[c][4 + f] = 1.f / s;
        }
    }
    R.cur = c ^ 1;
    R.step = step;
}

// The item's arguments, in uniform registers: they come from device memory, and
// in ordinary registers they would push the strip's values into local memory.
__device__ __forceinline__ StepArgs uniform_args(const BatchDomain& D, uint32_t c)
{
    StepArgs a;
    a.nx = uniform(D.a.nx);
    a.ny = uniform(D.a.ny);
    a.nz = uniform(D.a.nz);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        a.periodic[d] = uniform(D.a.periodic[d]);
        a.g[d] = uniform(D.a.g[d]);
        a.gf[d] = uniform(D.a.gf[d]);
    }
    a.pre = uniform(D.buf[c]);
    a.post = uniform(D.buf[c ^ 1]);
    a.seed = (uint32_t)uniform((int)step_seed(D.step));
    return a;
}

template <int Q, int ST, int R, int MINB>
__global__ void __launch_bounds__(Cfg<Q, ST, R>::NT, 4 * MINB / Cfg<Q, ST, R>::W) tau1_batch_kernel(BatchTable* T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int last;
    // FP16 only (BF16 keeps S = 1): maxima of the stored values, needed on the
    // step before each scale check
    constexpr bool AMAX = ST == ST_F16S;
    const int nitems = uniform(T->nitems), ndom = uniform(T->ndom), chunk = uniform(T->chunk);
    const int* __restrict__ begin = T->item_begin;
    const int warp = uniform((int)(threadIdx.x >> 5)), nwarps = Cfg<Q, ST, R>::W * (int)gridDim.x;
    // each warp takes its first item by its index, then the next free one
    // (items differ in size: partial strips, partial chunks, several boxes)
    for (int it = Cfg<Q, ST, R>::W * (int)blockIdx.x + warp; it < nitems;) {
        // box of this item: the last d with begin[d] <= it
        int lo = 0, hi = ndom - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (begin[mid] <= it) lo = mid;
            else hi = mid - 1;
        }
        const int slot = uniform(T->live[lo]);
        BatchDomain& D = T->dom[slot];
        const int local = uniform(it - begin[lo]);
        const uint32_t c = (uint32_t)uniform((int)D.cur);
        const StepArgs a = uniform_args(D, c);
        const int nstrips = uniform(D.nstrips), z0 = local / nstrips * chunk, z1 = a.nz - z0 < chunk ? a.nz : z0 + chunk;
        const Place pl = place_of_strip<R>(a, local % nstrips);
        unsigned char* const mine = smem + warp * Cfg<Q, ST, R>::WARP;
        [[maybe_unused]] float amax[4] = {0.f, 0.f, 0.f, 0.f};
        if constexpr (by_links(ST)) {
            const Scales sc(AMAX ? D.scale[c] : nullptr, AMAX ? D.scale[c ^ 1] : nullptr);
            strip_links<Q, ST, R, AMAX>(a, sc, pl, z0, z1, mine, amax);
        } else {
            strip_step<Q, ST, R>(a, pl, z0, z1, mine);
        }
        if (AMAX && (D.step + 1) % BATCH_RESCALE_EVERY == 0) {
#pragma unroll
            for (int f = 0; f < 4; ++f) {
                float m = amax[f];
                for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
                // non-negative floats order like their bit patterns
                if ((threadIdx.x & 31) == 0 && m > 0.f) atomicMax(&D.amax[f], __float_as_uint(m));
            }
        }
        if ((threadIdx.x & 31) == 0) it = nwarps + (int)atomicAdd(&T->next, 1u);
        it = uniform(it);
    }
    // close the step: the last block to arrive updates every live box
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&T->done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int d = threadIdx.x; d < ndom; d += blockDim.x) finish_box(T->dom[T->live[d]], ST);
    if (threadIdx.x == 0) {
        T->done = 0;
        T->next = 0;
    }
}

template <int Q, int ST, int V>
struct BatchKernel {
    using Sh = StripShape<Q, ST, V>;
    using C = Cfg<Q, ST, Sh::R>;
    static_assert(C::SMEM <= 227 * 1024, "shared memory of one block");
    static constexpr auto fn() { return tau1_batch_kernel<Q, ST, Sh::R, Sh::MINB>; }
    static cudaError_t prepare(int& grid, int& rows)
    {
        auto kern = fn();
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
        if (e != cudaSuccess) return e;
        int dev = 0, sms = 0, per_sm = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::NT, C::SMEM)) != cudaSuccess)
            return e;
        grid = sms * (per_sm > 0 ? per_sm : 1);
        rows = C::R;
        return cudaSuccess;
    }
    static cudaError_t launch(BatchTable* T, int grid, cudaStream_t s)
    {
        fn()<<<grid, C::NT, C::SMEM, s>>>(T);
        return cudaGetLastError();
    }
};

// Shape of variant 0; the others name one. The arguments come from the table and
// take registers, so that the formats summed link by link do not all take the shape
// of the single box. us per step of 12 boxes of 32^3 to 128^3, of 4 of 192^3 and of
// 3 of 96^3, with shape 0, 1 and 2: D3Q19 FP16 101, 117, 96; 273, 271, 274; 37, 40, 36;
// BF16 94, 108, 92; 256, 256, 263; 34, 38, 34; D3Q27 FP16 162, 145, 157; 377, 377, 419;
// 54, 49, 52; BF16 144, 138, 132; 347, 364, 364; 50, 47, 46.
constexpr int batch_shape(int q, int st)
{
    if (st == ST_F16S) return q == 19 ? 2 : 1;
    if (st == ST_BF16S) return q == 19 ? 0 : 2;
    return 1;
}

template <int Q, int ST>
cudaError_t dispatch_v(int variant, bool prep, BatchTable* T, int& grid, int& rows, cudaStream_t s)
{
    auto go = [&](auto k) {
        using K = decltype(k);
        return prep ? K::prepare(grid, rows) : K::launch(T, grid, s);
    };
    if constexpr (ST == ST_F64) {
        return variant == 0 ? go(BatchKernel<Q, ST, 0>{}) : cudaErrorInvalidValue;
    } else {
        switch (variant) {
        case 0: return go(BatchKernel<Q, ST, batch_shape(Q, ST)>{});
        case 1: return go(BatchKernel<Q, ST, 0>{});
        case 2: return go(BatchKernel<Q, ST, 1>{});
        case 3: return go(BatchKernel<Q, ST, 2>{});
        default: return cudaErrorInvalidValue;
        }
    }
}

cudaError_t dispatch(int q, int storage, int variant, bool prep, BatchTable* T, int& grid, int& rows,
                     cudaStream_t s)
{
    switch (q * 10 + storage) {
    case 190 + ST_F64: return dispatch_v<19, ST_F64>(variant, prep, T, grid, rows, s);
    case 190 + ST_F32: return dispatch_v<19, ST_F32>(variant, prep, T, grid, rows, s);
    case 190 + ST_F16S: return dispatch_v<19, ST_F16S>(variant, prep, T, grid, rows, s);
    case 190 + ST_BF16S: return dispatch_v<19, ST_BF16S>(variant, prep, T, grid, rows, s);
    case 270 + ST_F64: return dispatch_v<27, ST_F64>(variant, prep, T, grid, rows, s);
    case 270 + ST_F32: return dispatch_v<27, ST_F32>(variant, prep, T, grid, rows, s);
    case 270 + ST_F16S: return dispatch_v<27, ST_F16S>(variant, prep, T, grid, rows, s);
    case 270 + ST_BF16S: return dispatch_v<27, ST_BF16S>(variant, prep, T, grid, rows, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t batch_prepare(int q, int storage, int variant, int* grid, int* rows)
{
    int g = 0, r = 0;
    cudaError_t e = dispatch(q, storage, variant, true, nullptr, g, r, nullptr);
    *grid = g;
    *rows = r;
    return e;
}

cudaError_t launch_tau1_batch(int q, int storage, int variant, BatchTable* T, int grid, cudaStream_t s)
{
    int r = 0;
    return dispatch(q, storage, variant, false, T, grid, r, s);
}

}  // namespace lbm
