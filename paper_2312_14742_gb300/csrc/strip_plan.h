// How a box is cut into strips (strip.cuh): the strips of a plane, and the shape of
// a strip and the planes per chunk that a step of the box takes. Host code without
// CUDA, for any box of fewer than 2^31 nodes.
#pragma once

#include <cmath>
#include <cstdint>

namespace lbm {

constexpr int STRIP_WARPS = 4;  // warps per block of the dense and batched kernels, a strip each

// A periodic box of 32 columns takes a lane per column and rotates them.
constexpr bool strip_rotates(int nx, int periodic) { return nx == 32 && periodic; }

// Strips of a plane of nx x ny nodes.
constexpr int64_t strips_of(int nx, int ny, int periodic, int rows_per_strip)
{
    const int64_t rows = ((int64_t)ny + rows_per_strip - 1) / rows_per_strip;
    return strip_rotates(nx, periodic) ? rows : (rows * ((int64_t)nx + 2) - 2 + 29) / 30;
}

constexpr int STRIP_SHAPES = 3;  // per lattice and format; FP64 has one

// A shape of strips: its rows, the resident blocks per SM that its registers are
// sized for, and the time of a plane with 0 .. 4 blocks on an SM, and in many waves
// where that is not the last of them.
struct StripShapeCost {
    int rows, minb;
    double plane[5], many = 0;
};

// Storage 0 FP64, 1 FP32, 2 and 3 the 16-bit formats (lbm_storage). The times of a
// plane, up to a factor, are fitted to sweeps of shape and chunk over 18 boxes.
// Measured in FP32, in us, with two rows and four: D3Q19 256^3 138 and 135,
// 512 x 256 x 128 138 and 133, 384^3 416 and 400, 128^3 26.7 and 25.3, but
// 250 x 130 x 90 34.5 and 37.2, 96^3 14.4 and 16.4; D3Q27 256^3 147 and 163, 320^3 267
// and 296, 250 x 130 x 90 37.0 and 45, 200^3 92.5 and 90.4, 96 x 256 x 128 without
// walls 34.7 and 28.8. On 11 boxes left out of the fit the default is the faster of
// the two, or within 2% of it.
constexpr StripShapeCost strip_shape(int q, int storage, int v)
{
    if (storage == 0) return {2, 2, {0, 1.2, 2.0, 0, 0}};
    if (storage == 1)
        return v == 0 ? StripShapeCost{2, 4, {0, 0.95, 1.3, 1.7, 2.1}, q == 19 ? 2.2 : 2.1}
                      : (v == 1 ? StripShapeCost{4, 3, {0, 1.6, 2.3, 3.0, 0}, q == 19 ? 3.0 : 3.24}
                                : StripShapeCost{4, 2, {0, 1.6, 2.3, 0, 0}});
    if (q == 19)
        return v == 0 ? StripShapeCost{2, 4, {0, 0.87, 1.2, 1.56, 1.93}}
                      : (v == 1 ? StripShapeCost{2, 3, {0, 0.87, 1.2, 1.56, 0}} : StripShapeCost{4, 2, {0, 1.6, 2.3, 0, 0}});
    return v == 0 ? StripShapeCost{2, 3, {0, 0.87, 1.2, 1.56, 0}}
                  : (v == 1 ? StripShapeCost{2, 2, {0, 0.87, 1.2, 0, 0}} : StripShapeCost{4, 2, {0, 1.6, 2.3, 0, 0}});
}

// Time of a step of that many strips of a shape and of chunk planes each, up to a
// factor. A strip of c planes costs c + 4 planes (two beside its own, and as much
// again to start). plane[n] is nearly n times one where the SM is full, latency
// below. In a wave or two the fullest SM decides, and strips differ (walls); many
// waves even out, but for the end of the last one.
inline double strip_cost(int64_t strips, int64_t chunk, int sms, const StripShapeCost& s)
{
    const int64_t blocks = (strips + STRIP_WARPS - 1) / STRIP_WARPS;
    const double planes = (double)chunk + 4, waves = (double)blocks / ((double)sms * s.minb);
    if (waves <= 1) return planes * 1.15 * s.plane[(blocks + sms - 1) / sms];
    if (waves <= 2.5) return planes * s.plane[s.minb] * 1.15 * std::ceil(waves);
    return planes * (s.many > 0 ? s.many : s.plane[s.minb]) * (waves + 0.4);
}

struct StripPlan {
    int shape, chunk;
};

constexpr int strip_shapes(int storage) { return storage == 0 ? 1 : STRIP_SHAPES + 1; }  // 0: by the box
constexpr int STRIP_CHUNKS[4] = {0, 32, 16, 48};  // planes per chunk by variant / strip_shapes; 0: by the box

// Shape and chunk of a variant, of the least cost where the variant leaves them
// open. Chunks of equal height: of nz planes in n, for every n that lowers the
// height, some 2 sqrt(nz) candidates (16 us for 1e5 planes: once per handle and
// variant, not per step).
inline StripPlan strip_plan(int q, int storage, int variant, int nx, int ny, int nz, int periodic_x, int sms)
{
    const int v = variant % strip_shapes(storage), fixed = STRIP_CHUNKS[variant / strip_shapes(storage)];
    // two rows or four in FP32; FP64 has one shape, and link by link the first one
    // is the best or within 2% of it on 12 of 14 boxes
    const int first = v > 0 ? v - 1 : (storage == 1 ? 1 : 0), last = v > 0 ? v - 1 : 0;
    StripPlan best{first, 1};
    double least = -1;
    for (int shape = first; shape >= last; --shape) {
        const StripShapeCost s = strip_shape(q, storage, shape);
        const int64_t strips = strips_of(nx, ny, periodic_x, s.rows), planes = nz;
        auto take = [&](int64_t c) {
            const double cost = strip_cost(strips * ((planes + c - 1) / c), c, sms, s);
            if (least < 0 || cost < least) {
                best = {shape, (int)c};
                least = cost;
            }
        };
        if (fixed > 0) {
            take(fixed < nz ? fixed : nz);
            continue;
        }
        for (int64_t c = planes;;) {
            take(c);
            if (c == 1) break;
            const int64_t n = (planes + c - 2) / (c - 1);  // fewest chunks of less than c planes
            c = (planes + n - 1) / n;
        }
    }
    return best;
}

// Compact layout: how the strips of its tile columns (zchunk planes, `strips` strips
// of them; storage and shape as above) and its node list share a step.
//   planes: of a strip, a part of zchunk that divides it. Strips of whole columns
//   leave small boxes to the latency of 24 planes: 160 x 288 x 58 at 29% fluid 59 us per
//   step, 32 in parts (D3Q19 FP32). The list's blocks run beside the strips, so that
//   waves even out; FP64 strips are their own bound.
//   first: the strips are launched before the list and the list may start beside them.
//   That pays where they fill the GPU at most once (128^3 at 40% 33 and 25 us) and the list's
//   blocks are few, too: beside FP32 strips, which take nearly all shared memory, a
//   gather finds little L1 (192^3 at 30%, f* = 0.5: 61 us with the list first, 81 so). The
//   16-bit strips leave it its L1 (192^3 BF16 58 and 53 us).
struct CompactPlan {
    int planes;
    bool first;
};
inline CompactPlan compact_plan(int q, int storage, int shape, int zchunk, int64_t strips, int64_t listed, int sms)
{
    const StripShapeCost s = strip_shape(q, storage, shape);
    const double wave = (double)STRIP_WARPS * sms * s.minb;
    CompactPlan best{zchunk, false};
    double least = -1;
    for (int n = 1; n <= zchunk / 4; ++n) {
        if (zchunk % n != 0) continue;
        const int64_t count = strips * n, planes = zchunk / n;
        const double waves = (double)count / wave;
        const double cost = waves <= 1 || storage == 0 ? strip_cost(count, planes, sms, s)
                                                       : ((double)planes + 4) * s.plane[s.minb] * (waves + 0.4);
        if (least < 0 || cost < least) {
            best = {(int)planes, waves <= 1};
            least = cost;
        }
    }
    const int64_t resident = (int64_t)2 * 12 * 128 * sms;  // two waves of the list's threads (D3Q19)
    best.first = best.first && (storage >= 2 || listed <= resident);
    return best;
}

}  // namespace lbm
