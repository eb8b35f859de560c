// Tau1 step of one strip: 32 columns (30 of them its own) and R rows marched in z
// by one warp.
//
// A lane owns the R rows of one column, in pairs (y, y + R/2) in the lanes of
// its packed arithmetic (f32x2 for FP32, two FP64 values for FP64). Per plane
// (moments.cuh has the arithmetic):
//   - it reads its R records and those of the two rows around the strip, and
//     forms their moments; the y sums need no other lane (the two outer rows
//     give only what they send inwards);
//   - what passes along x goes by shuffle; the first and last lane hold the
//     columns beside the strip and store nothing (a periodic box of 32
//     columns needs none: they rotate);
//   - seven values per pair of nodes wait in registers for the next plane.
// A warp needs nothing from any other.
//
// Walls: solid sources add nothing to the sums. A warp that sees a solid node
// around its strip gathers its nodes next to a wall, a few percent, into a list
// and finishes 64 at a time, two per lane (bounce()), so that wall terms cost
// one pass over 64 nodes and not one over every node of the strip.
// Media crowded with walls pay for that list: 256^3 D3Q19 FP32 at 50% porosity takes 156
// us with spheres of radius 6 and 168 with radius 3, where the tile kernels, which
// carried wall terms for every node, took 155. (162 and 174 while nodes at solid
// corners, where D3Q19 has no links, were listed too and the list was written word
// by word; 138 instead of 134 at 90%, radius 8.)
//
// Records come by cp.async, each lane copying those it will read itself, one
// plane ahead: no alignment rule besides the record's own, periodic images and
// ragged boxes are just other addresses, and a cell that lies beyond a
// non-periodic face keeps a NaN record.
//
// The 16-bit formats march the same strips link by link (strip_links()): no list,
// and more values along x.
//
// 256^3, spheres of radius 8 at 90% porosity, us per step by default, and of the
// tile kernels before: D3Q19 FP32 134 (156), BF16 150 (183), D3Q27 FP32 144 (261), BF16
// 206 (315); 128^3 D3Q19 FP64 687 (934). FP32 is bound by issue and the latency of
// the 12 warps per SM of four-row strips, not by HBM (74 us for the state alone).
// Blocks whose four warps met at a barrier per plane and formed 32 own columns each
// took 10 to 23% more.
#pragma once

#include "kernels.h"
#include "links.cuh"
#include "mbarrier.cuh"
#include "moments.cuh"
#include "pack2.cuh"
#include "strip_plan.h"

namespace lbm {

namespace col {

template <int Q, int ST, int R_> struct Cfg {
    using E = typename Storage<ST>::ctype;
    using L = typename Lanes<E>::type;
    using S = Sums<Q>;
    static constexpr int W = STRIP_WARPS, NT = 32 * W;                  // strips (warps) per block
    static constexpr int R = R_, NP = R / 2;                  // rows and pairs of rows per strip
    static constexpr int REC = Storage<ST>::NODE_BYTES;
    static constexpr int NSTAGE = 3;                          // previous, current and next plane
    static constexpr int LINE = 32 * REC;                     // one staged row: 32 records
    static constexpr int B = R + 2;                           // solid bits of a plane: rows -1 .. R
    // nodes waiting for their wall terms: sums, own record, place and solid bits around
    static constexpr int FULL = 64, CAP = FULL - 1 + 32 * R;  // finished when FULL; the most there can be
    // offsets in a warp's part
    static constexpr int PART = NSTAGE * B * LINE;            // [CAP][4]
    static constexpr int RAW = PART + CAP * 4 * (int)sizeof(E);
    static constexpr int IDS = RAW + (CAP * REC + 15) / 16 * 16;  // [CAP] x 16 bytes
    static constexpr int WARP = by_links(ST) ? PART : IDS + CAP * 16;
    static constexpr int SMEM = W * WARP;
    static_assert(R % 2 == 0 && 3 * B <= 32, "rows");
    static_assert(PART % 16 == 0 && RAW % 16 == 0 && WARP % 16 == 0, "alignment");
};

template <int BYTES> __device__ __forceinline__ void cp_async(uint32_t dst, const void* src)
{
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
template <int REC> __device__ __forceinline__ void copy_record(uint32_t d, const unsigned char* src)
{
    if constexpr (REC == 32) {
        cp_async<16>(d, src);
        cp_async<16>(d + 16, src + 16);
    } else {
        cp_async<REC>(d, src);
    }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// a record of a wall: drho = NaN, u = 0
template <int ST> __device__ __forceinline__ void put_wall(unsigned char* dst)
{
    if constexpr (ST == ST_F64) {
        reinterpret_cast<uint4*>(dst)[0] = make_uint4(0xffffffffu, 0x7fffffffu, 0u, 0u);
        reinterpret_cast<uint4*>(dst)[1] = make_uint4(0u, 0u, 0u, 0u);
    } else if constexpr (ST == ST_F32) {
        *reinterpret_cast<uint4*>(dst) = make_uint4(0x7fffffffu, 0u, 0u, 0u);
    } else {
        *reinterpret_cast<uint2*>(dst) = make_uint2(0x7fffu, 0u);
    }
}

__device__ __forceinline__ f2 lanes_of(float a, float b) { return f2(a, b); }
__device__ __forceinline__ d2 lanes_of(double a, double b) { return d2(a, b); }

// A value that is the same in the whole warp, in a form that the compiler knows
// to be: it then lives in a uniform register.
__device__ __forceinline__ int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ float uniform(float v) { return __shfl_sync(0xffffffffu, v, 0); }
__device__ __forceinline__ double uniform(double v) { return __shfl_sync(0xffffffffu, v, 0); }
template <typename T> __device__ __forceinline__ T* uniform(T* v)
{
    return reinterpret_cast<T*>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(v), 0));
}

template <typename L> __device__ __forceinline__ L shfl_pair(const L& v, int src)
{
    return lanes_of(__shfl_sync(0xffffffffu, v.v.x, src), __shfl_sync(0xffffffffu, v.v.y, src));
}

__device__ __forceinline__ bool wrap_coord(int& c, int n, int periodic)
{
    if (c >= 0 && c < n) return true;
    if (!periodic) return false;
    c %= n;
    if (c < 0) c += n;
    return true;
}

__device__ __forceinline__ void track_amax(float (&m)[4], float d, float ux, float uy, float uz)
{
    m[0] = fmaxf(m[0], fabsf(d));
    m[1] = fmaxf(m[1], fabsf(ux));
    m[2] = fmaxf(m[2], fabsf(uy));
    m[3] = fmaxf(m[3], fabsf(uz));
}

// What a lane of a strip holds: the column at x and rows y0 .. y0 + R - 1; owner:
// it stores them (else the column only feeds its neighbours); the lanes that hold
// the columns to the left and right, where it is one.
struct Place {
    int x, y0;
    bool owner;
    int left, right;
};

// The columns of a box in one sequence of slots: per R rows the nx columns and
// the two beside them. A lane that owns its slot has both neighbours in the next
// lanes, so that any window of the sequence makes a strip, across the end of a
// row of columns as well.
template <int R> __device__ __forceinline__ Place place_of_slot(const StepArgs& a, uint32_t slot, bool owner)
{
    const uint32_t w = (uint32_t)a.nx + 2u, row = slot / w;
    const int lane = threadIdx.x & 31;
    Place p;
    p.x = (int)(slot - row * w) - 1;
    p.y0 = (int)min(row * R, (uint32_t)a.ny);
    p.owner = owner && p.x >= 0 && p.x < a.nx && p.y0 < a.ny;
    p.left = (lane + 31) & 31;
    p.right = (lane + 1) & 31;
    return p;
}

// Strip i of a box: 30 slots of the sequence, the first and last lane hold the
// ones before and after. A periodic box of 32 columns takes a lane per column
// and rotates them.
template <int R> __device__ __forceinline__ Place place_of_strip(const StepArgs& a, int i)
{
    const int lane = threadIdx.x & 31;
    if (strip_rotates(a.nx, a.periodic[0])) return {lane, i * R, true, (lane + 31) & 31, (lane + 1) & 31};
    return place_of_slot<R>(a, 30u * (uint32_t)i + (uint32_t)lane, lane >= 1 && lane <= 30);
}
// The planes of a strip as they pass through a warp's shared memory: R + 2 rows
// of 32 records, a slot per plane, each lane's cells copied by the lane itself.
// A cell beyond a non-periodic face holds a wall's record.
template <int Q, int ST, int R> struct Planes {
    using C = Cfg<Q, ST, R>;
    static constexpr int REC = C::REC, B = C::B;
    const StepArgs& a;
    unsigned char* mine;
    uint32_t nxy;
    size_t plane;
    // the lane's cells: rows 0 .. rows - 1 are the box's, one plane row after
    // the other; row `rows` (above the strip, or the first one beyond the box in
    // its last strip) and row -1 are images of others, or walls
    int rows;
    uint32_t xy, xy_below, xy_above;
    uint32_t ok = 0;      // bit r + 1: row r is copied
    uint32_t active = 0;  // bit r + 1: row r is a node this lane owns
    bool full;

    // in-plane index of a staged cell's image in the box; false for a wall
    __device__ __forceinline__ bool source(int x, int y, uint32_t& i) const
    {
        const bool in = wrap_coord(x, a.nx, a.periodic[0]) && wrap_coord(y, a.ny, a.periodic[1]);
        i = (uint32_t)x + (uint32_t)a.nx * (uint32_t)y;
        return in;
    }
    __device__ __forceinline__ unsigned char* cell(int slot, int row) const
    {
        return mine + slot * (B * C::LINE) + (row + 1) * C::LINE;
    }
    __device__ __forceinline__ Planes(const StepArgs& args, const Place& pl, unsigned char* smem)
        : a(args), mine(smem + (threadIdx.x & 31) * REC), nxy((uint32_t)args.nx * (uint32_t)args.ny),
          plane((size_t)nxy * REC), rows(min(R, args.ny - pl.y0))
    {
        if (rows > 0) {
            if (source(pl.x, pl.y0 - 1, xy_below)) ok |= 1u;
            if (source(pl.x, pl.y0, xy))
#pragma unroll
                for (int r = 0; r < R; ++r) ok |= r < rows ? 2u << r : 0u;
            if (source(pl.x, pl.y0 + rows, xy_above)) ok |= 2u << rows;
        }
        full = __all_sync(0xffffffffu, ok == (1u << B) - 1u);
#pragma unroll
        for (int r = 0; r < R; ++r) active |= pl.owner && r < rows ? 2u << r : 0u;
        __syncwarp();  // the previous call's last reads are done
#pragma unroll
        for (int s = 0; s < C::NSTAGE; ++s) {
#pragma unroll
            for (int r = 0; r < B; ++r)
                if (!(ok >> r & 1u)) put_wall<ST>(cell(s, r - 1));
        }
    }
    // starts the copy of plane p into a slot
    __device__ __forceinline__ void stage(int p, int slot) const
    {
        int gz = p;
        if (wrap_coord(gz, a.nz, a.periodic[2])) {
            const unsigned char* base = static_cast<const unsigned char*>(a.pre) + (size_t)gz * plane;
            const uint32_t d = smem_u32(cell(slot, -1));
            if (full) {
                copy_record<REC>(d, base + (size_t)xy_below * REC);
#pragma unroll
                for (int r = 0; r < R; ++r)
                    copy_record<REC>(d + (r + 1) * C::LINE, base + (size_t)(xy + (uint32_t)(r * a.nx)) * REC);
                copy_record<REC>(d + (R + 1) * C::LINE, base + (size_t)xy_above * REC);
            } else {
                if (ok & 1u) copy_record<REC>(d, base + (size_t)xy_below * REC);
                for (int r = 0; r <= R; ++r)
                    if (ok >> (r + 1) & 1u)
                        copy_record<REC>(d + (r + 1) * C::LINE,
                                         base + (size_t)(r == rows ? xy_above : xy + (uint32_t)(r * a.nx)) * REC);
            }
        } else {
#pragma unroll
            for (int r = 0; r < B; ++r) put_wall<ST>(cell(slot, r - 1));
        }
        cp_commit();
    }
};

// One strip of one step: planes z0 <= z < z1 of the columns at pl. All lanes of
// the warp call it together; smem holds Cfg::WARP bytes of this warp's own,
// 16-byte aligned.
template <int Q, int ST, int R_>
__device__ __forceinline__ void strip_step(const StepArgs& a, const Place& pl, int z0, int z1, unsigned char* smem)
{
    using C = Cfg<Q, ST, R_>;
    using E = typename C::E;
    using L = typename C::L;
    using S = Sums<Q>;
    constexpr int REC = C::REC, R = C::R, NP = C::NP, NV = S::NV;
    constexpr int B = C::B;

    const int lane = threadIdx.x & 31;
    const uint32_t nxy = (uint32_t)a.nx * (uint32_t)a.ny;
    Terms<ST> t(a);
    t.gx = uniform(t.gx);
    t.gy = uniform(t.gy);
    t.gz = uniform(t.gz);

    const Planes<Q, ST, R_> planes(a, pl, smem);
    auto read = [&](const unsigned char* p) { return record_at<ST>(p); };
    const uint32_t xy = planes.xy, active = planes.active;

    E* const part = reinterpret_cast<E*>(smem + C::PART);
    unsigned char* const raw = smem + C::RAW;
    uint4* const ids = reinterpret_cast<uint4*>(smem + C::IDS);
    int waiting = 0;  // nodes on the list
    // finishes the nodes first .. end - 1 of the list (at most FULL), two per
    // lane of the warp
    auto finish_listed = [&](int first, int end) {
        const int half = (end - first + 1) / 2;
        if (lane >= half) return;
        const int eA = first + lane, eB = eA + half < end ? eA + half : eA;
        const uint4 iA = ids[eA], iB = ids[eB];
        const Rec<E> rA = read(raw + eA * REC), rB = read(raw + eB * REC);
        const Moments<L> m = pair_moments<0, ST, L>(rA, rB, t, false, false);
        L s[4], Bn[4];
        bounce<Q, L>(m, [&](auto kc, L v, auto&& add) {
            // the source x - c_k: its column's word, its plane's bits, its row's bit
            constexpr int K = decltype(kc)::value, cz = cvel(K, 2);
            constexpr uint32_t bit = 1u << ((cz == -1 ? 0 : (cz == 0 ? B : 2 * B)) + 1 - cvel(K, 1));
            const uint32_t bA = cvel(K, 0) == 1 ? iA.y : (cvel(K, 0) == 0 ? iA.z : iA.w);
            const uint32_t bB = cvel(K, 0) == 1 ? iB.y : (cvel(K, 0) == 0 ? iB.z : iB.w);
            add(lanes_of(bA & bit ? v.v.x : E(0), bB & bit ? v.v.y : E(0)));
        }, Bn);
        const Rec<E> pA = read(reinterpret_cast<const unsigned char*>(part + 4 * eA)),
                     pB = read(reinterpret_cast<const unsigned char*>(part + 4 * eB));
        s[0] = lanes_of(pA.d, pB.d) + Bn[0];
        s[1] = lanes_of(pA.ux, pB.ux) + Bn[1];
        s[2] = lanes_of(pA.uy, pB.uy) + Bn[2];
        s[3] = lanes_of(pA.uz, pB.uz) + Bn[3];
        L d, ux, uy, uz;
        node_state<Q, L>(s, d, ux, uy, uz);
        step_store<ST>(a.post, iA.x, d.v.x, ux.v.x, uy.v.x, uz.v.x, nullptr, a.seed);
        if (eB != eA) {
            step_store<ST>(a.post, iB.x, d.v.y, ux.v.y, uy.v.y, uz.v.y, nullptr, a.seed);
        }
    };

    March<Q, L> z[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) z[j].clear();
    // solid bits of this column: rows -1 .. R of planes p, p - 1, p - 2 (B bits each)
    uint32_t hist = 0;
    constexpr uint32_t HMASK = (1u << (3 * B)) - 1u;
    int slot = 0;
    planes.stage(z0 - 1, 0);
#pragma unroll 2
    for (int p = z0 - 1; p <= z1; ++p) {
        const int next = slot == C::NSTAGE - 1 ? 0 : slot + 1;
        if (p < z1) planes.stage(p + 1, next);
        else cp_commit();
        cp_wait<1>();
        // y sums of the strip's pairs of rows, and the z sums of plane p - 1
        L X[NP][3], Y[NP][3], Cs[NP][3];
        uint32_t sb = 0;
        {
            L up[NP][NV], dn[NP][NV], h[NV];
            typename S::template Mid<L> mid[NP];
            {
                L skip[NV];
                typename S::template Mid<L> skipm;
                const Rec<E> ra = read(planes.cell(slot, -1)), rb = read(planes.cell(slot, R));
                const bool sA = isnan(ra.d), sB = isnan(rb.d);
                S::in_plane(pair_moments<2, ST, L>(ra, rb, t, sA, sB), skipm, h, skip);
                sb |= (sA ? 1u : 0u) | (sB ? 2u << R : 0u);
            }
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const Rec<E> ra = read(planes.cell(slot, j)), rb = read(planes.cell(slot, j + NP));
                const bool sA = isnan(ra.d), sB = isnan(rb.d);
                S::in_plane(pair_moments<0, ST, L>(ra, rb, t, sA, sB), mid[j], up[j], dn[j]);
                sb |= (sA ? 2u << j : 0u) | (sB ? 2u << (j + NP) : 0u);
            }
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                L So[NV], No[NV], P[S::NP], O[S::NO], M[S::NP];
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    So[k] = j > 0 ? up[j > 0 ? j - 1 : 0][k] : lanes_of(h[k].v.x, up[NP - 1][k].v.x);
                    No[k] = j < NP - 1 ? dn[j < NP - 1 ? j + 1 : 0][k] : lanes_of(dn[0][k].v.y, h[k].v.y);
                }
                S::y_sum(mid[j], So, No, P, O, M);
                z[j].advance(P, O, M, X[j], Y[j], Cs[j]);
            }
        }
        hist = (hist << B | sb) & HMASK;
        L s[NP][4];
#pragma unroll
        for (int j = 0; j < NP; ++j) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                X[j][k] = shfl_pair(X[j][k], pl.left);
                Y[j][k] = shfl_pair(Y[j][k], pl.right);
            }
            node_sums<Q, L>(Cs[j], X[j], Y[j], s[j]);
        }
        // rows of plane p - 1 to store: fluid nodes of the box and the chunk
        uint32_t store = p > z0 ? active & ~(hist >> B) : 0u;
        const uint32_t zoff = nxy * (uint32_t)(p - 1);
        if (__any_sync(0xffffffffu, hist != 0u)) {
            // solid bits of the columns left and right, and of all three together
            const uint32_t hl = __shfl_sync(0xffffffffu, hist, pl.left), hr = __shfl_sync(0xffffffffu, hist, pl.right);
            // rows next to a wall; D3Q19 has no links to the corners
            uint32_t lst;
            if constexpr (Q == 19) {
                const uint32_t side = hl | hr, own = hist | hist >> B | hist >> (2 * B), rows = own | side >> B;
                lst = store & (rows | rows << 1 | rows >> 1 | side | side >> (2 * B));
            } else {
                uint32_t n3 = hist | hl | hr;
                n3 |= n3 >> B | n3 >> (2 * B);
                lst = store & (n3 | n3 << 1 | n3 >> 1);
            }
            store &= ~lst;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool mineq = (lst >> (r + 1) & 1u) != 0u;
                const uint32_t m = __ballot_sync(0xffffffffu, mineq);
                if (mineq) {
                    const int e = waiting + __popc(m & ((1u << lane) - 1u));
                    E q[4];
#pragma unroll
                    for (int f = 0; f < 4; ++f) q[f] = r < NP ? s[r % NP][f].v.x : s[r % NP][f].v.y;
                    Storage<ST>::store(part, (uint32_t)e, q[0], q[1], q[2], q[3], nullptr);
                    const unsigned char* rec = planes.cell(slot == 0 ? C::NSTAGE - 1 : slot - 1, r);
#pragma unroll
                    for (int k = 0; k < REC / 16; ++k)
                        reinterpret_cast<uint4*>(raw + e * REC)[k] = reinterpret_cast<const uint4*>(rec)[k];
                    ids[e] = make_uint4(zoff + xy + (uint32_t)(r * a.nx), hl >> r, hist >> r, hr >> r);
                }
                waiting += __popc(m);
            }
            if (waiting >= C::FULL) {
                __syncwarp();
                do {
                    waiting -= C::FULL;
                    finish_listed(waiting, waiting + C::FULL);
                } while (waiting >= C::FULL);
                __syncwarp();
            }
        }
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            L d, ux, uy, uz;
            node_state<Q, L>(s[j], d, ux, uy, uz);
            if (store >> (j + 1) & 1u) {
                step_store<ST>(a.post, zoff + xy + (uint32_t)(j * a.nx), d.v.x, ux.v.x, uy.v.x, uz.v.x, nullptr, a.seed);
            }
            if (store >> (j + NP + 1) & 1u) {
                step_store<ST>(a.post, zoff + xy + (uint32_t)((j + NP) * a.nx), d.v.y, ux.v.y, uy.v.y, uz.v.y, nullptr, a.seed);
            }
        }
        slot = next;
    }
    __syncwarp();
    finish_listed(0, waiting);
}

// The same strip in the 16-bit formats, summed link by link (links.cuh). What a
// plane sends along x is shuffled per link. The sums of a node begin with the
// c_z = +1 links, whose values wait in registers for the node's own plane, and
// end with the c_z = -1 links, for which the node's own c_z = +1 values wait; wall
// links take the node's own value in their place in the order, where the warp sees
// any. With AMAX, amax[f] collects the largest |value| of field f among the
// nodes this lane stores.
template <int Q, int ST, int R_, bool AMAX>
__device__ __forceinline__ void strip_links(const StepArgs& a, const Scales& sc, const Place& pl, int z0, int z1,
                                            unsigned char* smem, float (&amax)[4])
{
    using C = Cfg<Q, ST, R_>;
    using E = typename C::E;
    using L = typename C::L;
    constexpr int R = C::R, NP = C::NP, B = C::B, NC = Weights<Q>::NCLASS;

    const uint32_t nxy = (uint32_t)a.nx * (uint32_t)a.ny;
    const L g0(uniform(gcomp<E>(a, 0))), g1(uniform(gcomp<E>(a, 1))), g2(uniform(gcomp<E>(a, 2)));
    float scale[4], inv[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        scale[f] = uniform(sc.s[f]);
        inv[f] = uniform(sc.inv[f]);
    }
    const Planes<Q, ST, R_> planes(a, pl, smem);
    const uint32_t xy = planes.xy, active = planes.active;

    // outgoing values of two records, those of direction k and inv(k) from one
    // product; none from a wall; MIRROR: the second record mirrored in y
    auto outgoing = [&](const unsigned char* pa, const unsigned char* pb, auto mirror, L (&out)[Q], bool& sA, bool& sB) {
        constexpr bool MIRROR = decltype(mirror)::value;
        Rec<E> ra, rb;
        Storage<ST>::load_at(pa, inv, ra.d, ra.ux, ra.uy, ra.uz);
        Storage<ST>::load_at(pb, inv, rb.d, rb.ux, rb.uy, rb.uz);
        sA = isnan(ra.d);
        sB = isnan(rb.d);
        const L d(sA ? E(0) : ra.d, sB ? E(0) : rb.d);
        const L rho = L(E(1)) + d, mass(sA ? E(0) : rho.v.x, sB ? E(0) : rho.v.y);
        const L vx = L(ra.ux, rb.ux) + g0, vz = L(ra.uz, rb.uz) + g2;
        L vy = L(ra.uy, rb.uy) + g1;
        if constexpr (MIRROR) vy.v.y = -vy.v.y;
        const L vv = fma(vz, vz, fma(vy, vy, vx * vx));
        const L A = fma(L(E(-1.5)) * mass, vv, d), r3 = L(E(3)) * mass, H = L(E(0.5)) * recip(rho);
        const L Px = product(r3, vx), Py = product(r3, vy), Pz = product(r3, vz);
        out[0] = A;
        static_for<0, (Q - 1) / 2>([&](auto ic) {
            constexpr int K = 1 + 2 * decltype(ic)::value;  // K + 1 = inv(K)
            const L p = dir_dot<K, L>(Px, Py, Pz), e = fma(p * H, p, A);
            out[K] = e + p;
            out[K + 1] = e - p;
        });
    };

    NodeAcc<L, NC> acc[NP];  // of plane p - 1, all but its c_z = -1 links
    L up[NP][Q];             // c_z = +1 links: what they bring to plane p
    L own[NP][Q];            // own c_z = +1 values of plane p - 1
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        acc[j].clear();
#pragma unroll
        for (int k = 0; k < Q; ++k) up[j][k] = own[j][k] = L(E(0));
    }
    // solid bits of this column and of those left and right: rows -1 .. R of planes p, p - 1, p - 2 (B bits each)
    uint32_t hist = 0, hl = 0, hr = 0;
    constexpr uint32_t HMASK = (1u << (3 * B)) - 1u;
    int slot = 0;
    planes.stage(z0 - 1, 0);
#pragma unroll 1
    for (int p = z0 - 1; p <= z1; ++p) {
        const int next = slot == C::NSTAGE - 1 ? 0 : slot + 1;
        if (p < z1) planes.stage(p + 1, next);
        else cp_commit();
        cp_wait<1>();
        L out[NP][Q], edge[Q];  // edge: rows -1 and R, the latter mirrored in y
        uint32_t sb = 0;
        {
            bool sA, sB;
            outgoing(planes.cell(slot, -1), planes.cell(slot, R), std::true_type{}, edge, sA, sB);
            sb |= (sA ? 1u : 0u) | (sB ? 2u << R : 0u);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                outgoing(planes.cell(slot, j), planes.cell(slot, j + NP), std::false_type{}, out[j], sA, sB);
                sb |= (sA ? 2u << j : 0u) | (sB ? 2u << (j + NP) : 0u);
            }
        }
        hist = (hist << B | sb) & HMASK;
        const bool walls = __any_sync(0xffffffffu, hist != 0u);
        if (walls) {
            hl = __shfl_sync(0xffffffffu, hist, pl.left);
            hr = __shfl_sync(0xffffffffu, hist, pl.right);
        }
        // what link k brings from plane p to the rows of pair j
        auto brings = [&](auto kc, int j) -> L {
            constexpr int K = decltype(kc)::value, cx = cvel(K, 0), cy = cvel(K, 1);
            constexpr int KM = kdir(cx, -cy, cvel(K, 2));
            L v = out[j][K];
            if constexpr (cy == 1) v = j > 0 ? out[j > 0 ? j - 1 : 0][K] : lanes_of(edge[K].v.x, out[NP - 1][K].v.x);
            if constexpr (cy == -1) v = j < NP - 1 ? out[j < NP - 1 ? j + 1 : 0][K] : lanes_of(out[0][K].v.y, edge[KM].v.y);
            if constexpr (cx != 0) v = shfl_pair(v, cx == 1 ? pl.left : pl.right);
            return v;
        };
        // v, or b where link k comes from a wall; PLANE: planes between its source and plane p
        auto or_wall = [&](auto kc, auto plane, int j, L v, L b) -> L {
            constexpr int K = decltype(kc)::value, cx = cvel(K, 0), PLANE = decltype(plane)::value;
            const uint32_t w = cx == 1 ? hl : (cx == 0 ? hist : hr);
            const uint32_t bit = 1u << (PLANE * B + 1 - cvel(K, 1));
            return lanes_of(w & bit << j ? b.v.x : v.v.x, w & bit << (j + NP) ? b.v.y : v.v.y);
        };
        using Here = std::integral_constant<int, 0>;
        using Below = std::integral_constant<int, 1>;
        // plane p - 1: its last links; rows to store: fluid nodes of the box and the chunk
        const uint32_t store = p > z0 ? active & ~(hist >> B) : 0u;
        const uint32_t zoff = nxy * (uint32_t)(p - 1);
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            L v[Q];
            links_of<Q, -1>([&](auto kc) { v[decltype(kc)::value] = brings(kc, j); });
            if (walls)
                links_of<Q, -1>([&](auto kc) {
                    constexpr int K = decltype(kc)::value;
                    v[K] = or_wall(kc, Here{}, j, v[K], own[j][inv_dir(K)]);
                });
            links_of<Q, -1>([&](auto kc) { acc[j].template add<Q, decltype(kc)::value>(v[decltype(kc)::value]); });
            L d, ux, uy, uz;
            node_finish<Q, L>(acc[j], d, ux, uy, uz);
            if (store >> (j + 1) & 1u) {
                step_store<ST>(a.post, zoff + xy + (uint32_t)(j * a.nx), d.v.x, ux.v.x, uy.v.x, uz.v.x, scale, a.seed);
                if constexpr (AMAX) track_amax(amax, d.v.x, ux.v.x, uy.v.x, uz.v.x);
            }
            if (store >> (j + NP + 1) & 1u) {
                step_store<ST>(a.post, zoff + xy + (uint32_t)((j + NP) * a.nx), d.v.y, ux.v.y, uy.v.y, uz.v.y, scale, a.seed);
                if constexpr (AMAX) track_amax(amax, d.v.y, ux.v.y, uy.v.y, uz.v.y);
            }
        }
        // plane p: the links from the plane below and from its own
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            L v[Q];
            links_of<Q, 0>([&](auto kc) { v[decltype(kc)::value] = brings(kc, j); });
            if (walls) {
                links_of<Q, 1>([&](auto kc) {
                    constexpr int K = decltype(kc)::value;
                    up[j][K] = or_wall(kc, Below{}, j, up[j][K], out[j][inv_dir(K)]);
                });
                links_of<Q, 0>([&](auto kc) {
                    constexpr int K = decltype(kc)::value;
                    v[K] = or_wall(kc, Here{}, j, v[K], out[j][inv_dir(K)]);
                });
            }
            acc[j].S[0] = out[j][0];
            links_of<Q, 1>([&](auto kc) { acc[j].template add<Q, decltype(kc)::value>(up[j][decltype(kc)::value]); });
            links_of<Q, 0>([&](auto kc) { acc[j].template add<Q, decltype(kc)::value>(v[decltype(kc)::value]); });
            links_of<Q, 1>([&](auto kc) {
                constexpr int K = decltype(kc)::value;
                up[j][K] = brings(kc, j);
                own[j][K] = out[j][K];
            });
        }
        slot = next;
    }
}

// Rows per strip, and resident blocks the register budget is sized for. Four rows
// form six rows' moments for four, two rows four for two, but two leave
// registers for more warps.
template <int Q, int ST, int V> struct StripShape;
template <int Q> struct StripShape<Q, ST_F32, 0> { static constexpr int R = 2, MINB = 4; };
template <int Q> struct StripShape<Q, ST_F32, 1> { static constexpr int R = 4, MINB = 3; };
template <int Q> struct StripShape<Q, ST_F32, 2> { static constexpr int R = 4, MINB = 2; };
template <int Q, int V> struct StripShape<Q, ST_F64, V> { static constexpr int R = 2, MINB = 2; };
// Link by link, two rows fill the registers: D3Q27 spills 200 bytes at 4 blocks
// (256^3 BF16 225 us per step, 206 at 3) and 90 with four rows.
template <int Q, int V> struct LinkShape;
template <int Q> struct LinkShape<Q, 0> { static constexpr int R = 2, MINB = Q == 19 ? 4 : 3; };
template <int Q> struct LinkShape<Q, 1> { static constexpr int R = 2, MINB = Q == 19 ? 3 : 2; };
template <int Q> struct LinkShape<Q, 2> { static constexpr int R = 4, MINB = 2; };
template <int Q, int V> struct StripShape<Q, ST_F16S, V> : LinkShape<Q, V> {};
template <int Q, int V> struct StripShape<Q, ST_BF16S, V> : LinkShape<Q, V> {};

}  // namespace col

}  // namespace lbm
