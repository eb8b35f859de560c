// Compact porous layout: the dense state records, with the work of a step
// split by tile column (a 32 x H tile of the x-y plane, a chunk of 24 or 32
// z planes).
//
// The paper's kernels skip solid chunks and treat mixed chunks through the
// node mask (Section 3.2); its bandwidth model for porous media charges a
// mixed chunk for all of its nodes (Section 4.3, B_est), and its outlook
// (Section 5) names indirect addressing of the fluid nodes. Here each tile
// column is classed by its fluid count c out of m nodes:
//   - c = 0: never visited (no record is read or written);
//   - c >= f* m: stepped by the tiled kernel, in strips cut from the runs of
//     such tiles (every node is loaded, as in the dense layout);
//   - 0 < c < f* m: its fluid nodes join a node list (4-byte box indices, in
//     z, y, x order of the tile), stepped one thread per node with the
//     neighbours read straight from the dense records (each state copy holds
//     one more record after the box: a solid sentinel for the sources that
//     lie outside a non-periodic face).
// Both kernels compute every node as the dense kernels do, and the node sets
// are disjoint, so a step gives the dense step's bits.
#include <algorithm>

#include "kernels.h"
#include "links.cuh"
#include "moments.cuh"

namespace lbm {

namespace {

// n / d for 0 <= n < 2^31 and a divisor d >= 1 fixed per launch, as a
// multiply-high, an add and a shift (Granlund and Montgomery, "Division by
// invariant integers using multiplication", 1994): with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1, n / d = (umulhi(m, n) + n) >> l; the sum
// stays below 2^32 because n < 2^31.
struct DivBy {
    uint32_t m, l;
    static DivBy make(uint32_t d)
    {
        DivBy r;
        r.l = 0;
        while ((1ull << r.l) < d) ++r.l;
        r.m = (uint32_t)((((1ull << 32) * ((1ull << r.l) - d)) / d) + 1);
        return r;
    }
    __device__ __forceinline__ uint32_t div(uint32_t n) const { return (__umulhi(m, n) + n) >> l; }
};

// Offsets, relative to a node at coordinate c of an axis of n nodes and
// stride st, of the source coordinate c - v for v = -1, 0, +1 (entry v + 1),
// and whether that source lies in the box (periodic axes wrap).
__device__ __forceinline__ void axis_sources(uint32_t c, uint32_t n, int st, bool per, int off[3], bool in[3])
{
    off[1] = 0;
    in[1] = true;
    // v = +1: source c - 1
    in[2] = c > 0 || per;
    off[2] = c > 0 ? -st : (per ? (int)(n - 1) * st : 0);
    // v = -1: source c + 1
    in[0] = c + 1 < n || per;
    off[0] = c + 1 < n ? st : (per ? -(int)(n - 1) * st : 0);
}

// One Tau1 step of the listed (fluid) box nodes, the neighbours' records
// gathered from the dense state. A source outside a non-periodic face is read
// from the sentinel record n (drho = NaN, u = 0) that follows the box in both
// state copies, so that every source is a plain load and a wall is recognised by
// its NaN alone. The sums are those of moments.cuh or links.cuh. One thread per
// node: two nodes per thread in packed arithmetic take a third fewer instructions
// but leave too few warps to hide the gathers (303 us against 256 on 9.9 M nodes).
// Warps matter more than loads in flight per thread: at 40 registers (D3Q19) a
// thread cannot hold 18 records, and the compiler spreads the loads that are
// written first; D3Q27 with all 26 records in registers takes 341 to 416 us.
// Away from the faces, where all nodes of a warp are as a rule, the sources lie at
// fixed distances: a third of the instructions went into finding them. 9.9 M nodes
// in D3Q19 take 204 us (221 without that case, 236 link by link), in D3Q27 321 (336,
// 339), in BF16 222 and 311 (244 and 331 before the strips); the default split of the
// same box (320^3, 30% fluid) 205 us and 249, 211 and 350 before the strips. D3Q27
// boxes that stay in L2 and go to the list altogether are slower than link by link:
// 161 x 127 x 101 at 40% 30.8 us against 28.8.
struct ListArgs {
    const int* nodes;
    int count;
    DivBy by_nx, by_nxy;
};

constexpr int LIST_THREADS = 128;

// What a node's sources need: the offsets per axis, and whether they are in the box.
struct Around {
    uint32_t i;
    int ox[3], oy[3], oz[3];
    bool ix[3], iy[3], iz[3];
    // true where no source lies on another side of the box
    __device__ __forceinline__ bool set(const StepArgs& a, const ListArgs& l, uint32_t node)
    {
        i = node;
        const uint32_t nx = (uint32_t)a.nx, nxy = nx * (uint32_t)a.ny;
        const uint32_t z = l.by_nxy.div(i), r = i - z * nxy, y = l.by_nx.div(r), x = r - y * nx;
        axis_sources(x, nx, 1, a.periodic[0], ox, ix);
        axis_sources(y, (uint32_t)a.ny, (int)nx, a.periodic[1], oy, iy);
        axis_sources(z, (uint32_t)a.nz, (int)nxy, a.periodic[2], oz, iz);
        return x - 1u < nx - 2u && y - 1u < (uint32_t)a.ny - 2u && z - 1u < (uint32_t)a.nz - 2u && nx > 2 && a.ny > 2 && a.nz > 2;
    }
    template <int K> __device__ __forceinline__ uint32_t source(uint32_t sentinel) const
    {
        constexpr int X = cvel(K, 0) + 1, Y = cvel(K, 1) + 1, Z = cvel(K, 2) + 1;
        return (ix[X] && iy[Y] && iz[Z]) ? i + (uint32_t)(ox[X] + oy[Y] + oz[Z]) : sentinel;
    }
};

// The step of the listed node of this thread.
template <int Q, int ST> __device__ __forceinline__ void list_node(const StepArgs& a, const ListArgs& l)
{
    using T = typename Storage<ST>::ctype;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const Scales sc(a.dscale);
    const uint32_t sentinel = (uint32_t)a.nx * (uint32_t)a.ny * (uint32_t)a.nz;
    if (t >= l.count) return;
    Around A;
    const bool inner = A.set(a, l, (uint32_t)__ldg(l.nodes + t));
    Rec<T> r[Q];
    auto load = [&](Rec<T>& c, uint32_t i) { Storage<ST>::load(a.pre, i, sc.inv, c.d, c.ux, c.uy, c.uz); };
    load(r[0], A.i);
    if (isnan(r[0].d)) return;  // a listed node is fluid; a NaN state is left as it is, as elsewhere
    auto step = [&](auto source) {
        constexpr bool FIRST = sizeof(T) == 4 && (Q == 19 || by_links(ST));
        if constexpr (FIRST)  // loads first (else as they are used)
            static_for<1, Q>([&](auto kc) { load(r[decltype(kc)::value], source(kc)); });
        auto fetch = [&](auto kc, bool& solid) -> const Rec<T>& {
            constexpr int K = decltype(kc)::value;
            if constexpr (!FIRST) load(r[K], source(kc));
            solid = isnan(r[K].d);
            return r[K];
        };
        T d, ux, uy, uz;
        if constexpr (by_links(ST)) {
            gather_links<Q, false>(a, r[0].d, r[0].ux, r[0].uy, r[0].uz, [&](auto kc, bool& solid, T& d, T& ux, T& uy, T& uz) {
                const Rec<T>& c = fetch(kc, solid);
                d = c.d;
                ux = c.ux;
                uy = c.uy;
                uz = c.uz;
            }, d, ux, uy, uz);
        } else {
            const Terms<ST> terms(a);
            const Moments<T> own = moments_of<ST, T>(r[0], terms, false);
            uint32_t wall = 0;
            T sums[4];
            gather_sums<Q, ST>(terms, own, [&](auto kc, bool& solid) {
                constexpr int K = decltype(kc)::value;
                const Rec<T>& c = fetch(kc, solid);
                if (solid) wall |= 1u << nbit(-cvel(K, 0), -cvel(K, 1), -cvel(K, 2));
                return c;
            }, sums);
            add_bounce<Q, T>(own, wall, sums);
            node_state<Q, T>(sums, d, ux, uy, uz);
        }
        step_store<ST>(a.post, A.i, d, ux, uy, uz, sc.s, a.seed);
    };
    // away from the faces the sources are at fixed distances
    if (__all_sync(__activemask(), inner)) {
        const uint32_t nx = (uint32_t)a.nx, nxy = nx * (uint32_t)a.ny;
        step([&](auto kc) {
            constexpr int K = decltype(kc)::value;
            return A.i - ((uint32_t)cvel(K, 0) + (uint32_t)cvel(K, 1) * nx + (uint32_t)cvel(K, 2) * nxy);
        });
    } else {
        step([&](auto kc) { return A.template source<decltype(kc)::value>(sentinel); });
    }
}

template <int Q, int ST>
__global__ void __launch_bounds__(LIST_THREADS, ST == ST_F64 ? 0 : (Q == 19 ? 12 : 8)) tau1_list_kernel(StepArgs a, ListArgs l)
{
    asm volatile("griddepcontrol.launch_dependents;");  // the tiled kernel of this step: other nodes
    list_node<Q, ST>(a, l);
    // a launch that began before the tiled kernel had ended ends after it
    if (blockIdx.x == gridDim.x - 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The sentinel record n of a state copy: drho = NaN, u = 0.
template <int ST>
__global__ void sentinel_kernel(void* buf, uint32_t n, const float* __restrict__ dscale)
{
    using T = typename Storage<ST>::ctype;
    const float one[4] = {1.f, 1.f, 1.f, 1.f};
    Storage<ST>::store(buf, n, T(NAN), T(0), T(0), T(0), dscale ? dscale : one);
}

template <int Q, int ST>
cudaError_t launch_list_t(const StepArgs& a, const int* nodes, int count, bool after_tiled, cudaStream_t s)
{
    const ListArgs l{nodes, count, DivBy::make((uint32_t)a.nx), DivBy::make((uint32_t)a.nx * (uint32_t)a.ny)};
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((count + LIST_THREADS - 1) / LIST_THREADS));
    cfg.blockDim = dim3(LIST_THREADS);
    cfg.stream = s;
    cfg.attrs = &overlap;
    cfg.numAttrs = after_tiled ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, tau1_list_kernel<Q, ST>, a, l);
}

constexpr int CT = 256;  // threads of the count and list kernels (8 warps)

struct TileGeo {
    int nx, ny, nz, h, chunk, ntx, ntiles;
    __device__ void origin(int b, int& x0, int& y0, int& z0, int& z1) const
    {
        const int tile = b % ntiles;
        z0 = (b / ntiles) * chunk;
        z1 = min(nz, z0 + chunk);
        x0 = (tile % ntx) * 32;
        y0 = (tile / ntx) * h;
    }
    // node of lane x of x-row r of the tile column (rows in z, y order), or -1
    __device__ int64_t node(int x0, int y0, int z0, int r, int lane) const
    {
        const int x = x0 + lane, y = y0 + r % h, z = z0 + r / h;
        if (x >= nx || y >= ny) return -1;
        return (int64_t)x + (int64_t)nx * ((int64_t)y + (int64_t)ny * z);
    }
};

__device__ __forceinline__ bool is_fluid(const uint8_t* flags, int64_t i)
{
    return i >= 0 && !(flags[i] & FLAG_SOLID);
}

// counts[b] = fluid nodes of tile column b; one block per tile column, one
// warp per x-row (coalesced flag bytes).
__global__ void __launch_bounds__(CT) tile_count_kernel(TileGeo g, const uint8_t* __restrict__ flags, int* counts)
{
    __shared__ int part[CT / 32];
    int x0, y0, z0, z1;
    g.origin(blockIdx.x, x0, y0, z0, z1);
    const int rows = g.h * (z1 - z0);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    int c = 0;
    for (int r = warp; r < rows; r += CT / 32) c += __popc(__ballot_sync(0xffffffffu, is_fluid(flags, g.node(x0, y0, z0, r, lane))));
    if (lane == 0) part[warp] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int w = 0; w < CT / 32; ++w) s += part[w];
        counts[blockIdx.x] = s;
    }
}

// The fluid nodes of the listed tile columns: tile column tiles[j] writes its
// fluid nodes, in row order, to nodes[offsets[j] ...]. One block per tile
// column; a round of 8 rows at a time, one per warp, numbered by a scan of
// the warps' ballot counts.
__global__ void __launch_bounds__(CT) tile_nodes_kernel(TileGeo g, const uint8_t* __restrict__ flags,
                                                        const int* __restrict__ tiles, const int* __restrict__ offsets,
                                                        int* __restrict__ nodes)
{
    __shared__ int part[CT / 32];
    int x0, y0, z0, z1;
    g.origin(tiles[blockIdx.x], x0, y0, z0, z1);
    const int rows = g.h * (z1 - z0);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    int base = offsets[blockIdx.x];
    for (int r0 = 0; r0 < rows; r0 += CT / 32) {
        const int r = r0 + warp;
        const int64_t i = r < rows ? g.node(x0, y0, z0, r, lane) : -1;
        const bool f = is_fluid(flags, i);
        const unsigned m = __ballot_sync(0xffffffffu, f);
        if (lane == 0) part[warp] = __popc(m);
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < CT / 32; ++w) {
            before += w < warp ? part[w] : 0;
            total += part[w];
        }
        if (f) nodes[base + before + __popc(m & ((1u << lane) - 1u))] = (int)i;
        base += total;
        __syncthreads();
    }
}

TileGeo geo_of(const CompactTiles& t, int nx, int ny, int nz)
{
    TileGeo g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.h = t.h;
    g.chunk = nz < t.zchunk ? nz : t.zchunk;
    g.ntx = (nx + 31) / 32;
    g.ntiles = g.ntx * ((ny + g.h - 1) / g.h);
    return g;
}

}  // namespace

CompactTiles compact_tiles(int q, int storage, int variant)
{
    const int nr = tau1_tile_shapes(storage);
    CompactTiles t;
    const int v = variant % nr;
    // two rows per strip, for v 2, 3 four (link by link another register budget): a list
    // of few strips is balanced by halves (D3Q19 FP32 at 30% fluid: 192^3 61.6 and 59.6 us
    // with four rows and two, 256^3 122.6 and 118.7, 320^3 206.0 and 204.7)
    t.shape = nr == 1 || v < 2 ? 0 : 1;
    t.zchunk = variant < nr ? 24 : 32;
    t.h = v == 1 ? 16 : (v == 3 ? 12 : 8);
    t.rows = strip_shape(q, storage, t.shape).rows;
    return t;
}

int64_t compact_tile_columns(const CompactTiles& t, int nx, int ny, int nz)
{
    const TileGeo g = geo_of(t, nx, ny, nz);
    if (g.h <= 0) return 0;
    return (int64_t)g.ntiles * ((nz + g.chunk - 1) / g.chunk);
}

int64_t compact_tile_nodes(const CompactTiles& t, int nx, int ny, int nz, int b)
{
    const TileGeo g = geo_of(t, nx, ny, nz);
    const int tile = b % g.ntiles;
    const int z0 = (b / g.ntiles) * g.chunk;
    const int x0 = (tile % g.ntx) * 32, y0 = (tile / g.ntx) * g.h;
    const int64_t w = nx - x0 < 32 ? nx - x0 : 32;
    const int64_t hh = ny - y0 < g.h ? ny - y0 : g.h;
    const int64_t d = nz - z0 < g.chunk ? nz - z0 : g.chunk;
    return w * hh * d;
}

void compact_strips(const CompactTiles& t, int nx, int ny, int nz, const std::vector<int>& tiles, int zstrip,
                    std::vector<int>& items)
{
    const TileGeo g = geo_of(t, nx, ny, nz);
    items.clear();
    int lanes = 32, chunk = -1;  // of the last item
    auto pad = [&] {
        for (; lanes < 32; ++lanes) items.push_back(items.back() < 0 ? items.back() : ~items.back());
        if (chunk >= 0) items.push_back(chunk);
    };
    for (size_t first = 0, last; first < tiles.size(); first = last) {
        // the tiles of one chunk of planes, once for each of its parts
        const int c = tiles[first] / g.ntiles, z1 = std::min(nz, (c + 1) * g.chunk);
        for (last = first; last < tiles.size() && tiles[last] / g.ntiles == c;) ++last;
        for (int z0 = c * g.chunk; z0 < z1; z0 += zstrip) {
            for (size_t i = first; i < last;) {
                // a run of tiles side by side, then each of its groups of rows
                const int tile = tiles[i] % g.ntiles, tx = tile % g.ntx;
                size_t e = i + 1;
                while (e < last && tiles[e] == tiles[e - 1] + 1 && tx + (int)(e - i) < g.ntx) ++e;
                for (int j = 0; j < t.h / t.rows; ++j) {
                    const int row = (tile / g.ntx * (t.h / t.rows) + j) * (nx + 2);  // slot of column -1
                    int x = 32 * tx;
                    const int end = std::min(nx, 32 * (tx + (int)(e - i)));
                    while (x < end) {
                        if (lanes > 29 || z0 / zstrip != chunk) {
                            pad();
                            lanes = 0;
                            chunk = z0 / zstrip;
                        }
                        const int n = std::min(end - x, 30 - lanes);
                        items.push_back(~(row + x));
                        for (int k = 1; k <= n; ++k) items.push_back(row + x + k);
                        items.push_back(~(row + x + n + 1));
                        lanes += n + 2;
                        x += n;
                    }
                }
                i = e;
            }
        }
    }
    pad();
}

cudaError_t launch_compact_count(const CompactTiles& t, int nx, int ny, int nz, const uint8_t* flags, int* counts,
                                 cudaStream_t s)
{
    const TileGeo g = geo_of(t, nx, ny, nz);
    const int64_t nb = compact_tile_columns(t, nx, ny, nz);
    if (nb <= 0 || nb > 0x7fffffffLL) return cudaErrorInvalidValue;
    tile_count_kernel<<<(unsigned)nb, CT, 0, s>>>(g, flags, counts);
    return cudaGetLastError();
}

cudaError_t launch_compact_nodes(const CompactTiles& t, int nx, int ny, int nz, const uint8_t* flags, const int* tiles,
                                 const int* offsets, int ntiles, int* nodes, cudaStream_t s)
{
    if (ntiles == 0) return cudaSuccess;
    const TileGeo g = geo_of(t, nx, ny, nz);
    tile_nodes_kernel<<<(unsigned)ntiles, CT, 0, s>>>(g, flags, tiles, offsets, nodes);
    return cudaGetLastError();
}

cudaError_t launch_compact_sentinel(int storage, void* buf, int64_t n, const float* dscale, cudaStream_t s)
{
    switch (storage) {
    case ST_F64: sentinel_kernel<ST_F64><<<1, 1, 0, s>>>(buf, (uint32_t)n, dscale); break;
    case ST_F32: sentinel_kernel<ST_F32><<<1, 1, 0, s>>>(buf, (uint32_t)n, dscale); break;
    case ST_F16S: sentinel_kernel<ST_F16S><<<1, 1, 0, s>>>(buf, (uint32_t)n, dscale); break;
    case ST_BF16S: sentinel_kernel<ST_BF16S><<<1, 1, 0, s>>>(buf, (uint32_t)n, dscale); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_tau1_list(int q, int storage, const StepArgs& a, const int* nodes, int64_t count, bool after_tiled,
                             cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    // node indices are int32 and nx ny z + y nx + x must not wrap in 32 bits
    if (count > 0x7fffffffLL || (int64_t)a.nx * a.ny * a.nz >= ((int64_t)1 << 31)) return cudaErrorInvalidValue;
    const int c = (int)count;
    switch (q * 10 + storage) {
    case 190 + ST_F64: return launch_list_t<19, ST_F64>(a, nodes, c, after_tiled, s);
    case 190 + ST_F32: return launch_list_t<19, ST_F32>(a, nodes, c, after_tiled, s);
    case 190 + ST_F16S: return launch_list_t<19, ST_F16S>(a, nodes, c, after_tiled, s);
    case 190 + ST_BF16S: return launch_list_t<19, ST_BF16S>(a, nodes, c, after_tiled, s);
    case 270 + ST_F64: return launch_list_t<27, ST_F64>(a, nodes, c, after_tiled, s);
    case 270 + ST_F32: return launch_list_t<27, ST_F32>(a, nodes, c, after_tiled, s);
    case 270 + ST_F16S: return launch_list_t<27, ST_F16S>(a, nodes, c, after_tiled, s);
    case 270 + ST_BF16S: return launch_list_t<27, ST_BF16S>(a, nodes, c, after_tiled, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
