// Launch plans of the plain sweep: host arithmetic, no CUDA needed.
#pragma once
#include <stddef.h>

namespace stg {

// Shared memory of an SM, and what the system reserves of it for each CTA.
constexpr size_t SM_SHARED = 228 << 10, CTA_SHARED = 1 << 10;

// Shape of a CTA of the prefetched sweep: vectors of a row, threads, shared memory.
struct PrefetchShape {
    int width, threads;
    size_t smem;
};
// nx columns in vectors of V, rows of a CTA, shared bytes a thread's slots take; alone: one CTA an SM.
//
// Rows of more than one CTA (32 vectors) are cut evenly, so that no CTA has its slots for a few
// lanes. Not rows of one CTA, where a narrower one only has fewer warps (25-point BF16, GLUP/s: 64^3 56 -> 39-45,
// 33 x 500 x 100 47 -> 44).
//
// alone (the 25-point sweeps): a CTA asks for half of the SM's shared memory at least. The CTAs of
// a cut row are small enough for two (25-point BF16: 160 or 192 threads of 560 bytes), whose slots leave
// 49 or 13 KB of L1 to the neighbour rows that each thread copies through it and up to nine rows share. GLUP/s,
// fields set and read back, T = 10, uncut / two CTAs / one: 176 x 256 x 200 104 / 60 / 116, 288^3 124 / 63 / 134,
// 270 x 256 x 141 115 / 64 / 124, 130 x 200 x 90 85 / 96 / 96, 140 x 64 x 300 86 / 100 / 99, 160 x 163 x 328
// - / 98 / 113, 203 x 250 x 141 (one either way) 112 / 116 / 116. The 7-point sweeps read one row on each side
// and gain from two.
inline PrefetchShape prefetch_shape(int nx, int V, int rows, size_t bytes, bool alone) {
    PrefetchShape p;
    const int ctas = (nx + 32 * V - 1) / (32 * V);
    p.width = ctas > 1 ? (nx + ctas * V - 1) / (ctas * V) : 32;
    p.threads = (p.width * rows + 31) / 32 * 32;
    p.smem = (size_t)p.threads * bytes;
    if (alone && ctas > 1 && p.smem < SM_SHARED / 2) p.smem = SM_SHARED / 2;
    return p;
}

// Whether an FP64 step of `ctas` CTAs, of which the GPU holds `slots`, with walks of `planes` planes is set up
// beside the step before it. FP64 sweeps are bound by the FP64 units, which CTAs that are set up early load
// unevenly: those of a second wave (1 % slower at 203 x 250 x 141), and those that find free slots
// beside a step that does not fill the GPU, on the SMs that have fewest of its CTAs, for the
// whole of a long walk. Speed with / without, fill of the slots and planes a walk: 7-point variable 469 x 230 x 29 0.76
// (0.51, 29), constant 600 x 300 x 30 0.82 (0.62, 30), 253 x 429 x 32 0.85 (0.71, 16), 328 x 461 x 19 0.93 (0.57, 19),
// 393 x 183 x 40 0.98 (0.79, 14); 186 x 332 x 83 0.99 (0.83, 21), 500 x 500 x 28 1.02 (0.83, 28), 81 x 99 x 44 1.15
// (0.75, 2), 64^3 1.24 (0.84, 1).
inline bool early_fp64(long long ctas, int slots, int planes) {
    return ctas <= slots && (5 * ctas >= 4LL * slots || planes < 12);
}

// How the interior copies cut their rows: a CTA of COPY_WARPS warps has 1 << lg neighbouring rows and
// COPY_WARPS >> lg segments of `seg` units of each; the CTAs of a group of rows (xblocks) follow one
// another. Rows are cut as far as there would be fewer than COPY_WANT warps (64 an SM), but not below one pass
// of a warp (32 lanes of COPY_UNITS units): a warp that moves a whole long row has 2 KB under way, and few such rows
// leave the GPU idle. A field set and read back and its sweep, FP32, T = 4, whole rows -> cut: 1000000 x 1 x 1 1099
// -> 43 us, 100000 x 8 x 4 193 -> 37, 20000 x 3 x 5 37 -> 26. Grids of 9728 rows or more are copied by whole rows.
constexpr int COPY_WARPS = 8, COPY_UNITS = 4;
constexpr long long COPY_WANT = 152 * 64;

struct CopySplit {
    int lg;
    unsigned xblocks;
    long long seg;
    // Whether the kernels need the split: not where a CTA has COPY_WARPS whole rows.
    bool cut() const { return lg != 3 || xblocks != 1; }
};
// ny rows a plane, rows in all, units a row.
inline CopySplit copy_split(int ny, long long rows, long long units) {
    CopySplit c;
    c.lg = ny >= 8 ? 3 : ny >= 4 ? 2 : ny >= 2 ? 1 : 0;
    const long long want = (COPY_WANT + rows - 1) / rows, pass = 32 * COPY_UNITS;
    c.seg = ((units + want - 1) / want + pass - 1) / pass * pass;
    const long long segs = (units + c.seg - 1) / c.seg, per = COPY_WARPS >> c.lg;
    c.xblocks = (unsigned)((segs + per - 1) / per);
    return c;
}

}  // namespace stg
