// Temporally blocked sweep with overlapped tiles (7-point stencils, FP32 field): one launch
// advances the whole grid by H steps, reading u_t once from one array and writing u_{t+H} to the
// other, so a step costs 1/H of the plain sweep's HBM traffic (Section III's code balance with
// the cache block held in registers).
//
// * A CTA owns an xy tile and streams it along z. A warp covers one row of 128 columns with
//   128-bit vectors; a thread keeps RB rows of its vector for all H time levels, so the z
//   neighbours of every level are in its registers: at iteration s the input plane s arrives
//   and level l computes plane s - l - 1 from the planes s - l - 2 .. s - l of level l - 1.
// * Of the values that threads share, x neighbours come by shuffle and y neighbours from the
//   own rows, or from one row above and below that the neighbouring warps published in shared
//   memory one iteration before: one CTA barrier per iteration, whatever H.
// * Input planes (and the planes of the coefficient arrays) arrive by tensor copies
//   (cp.async.bulk.tensor) several iterations ahead, one thread issuing them; level 0's y
//   neighbours are read from the copied plane. A thread reads its coefficient vectors from the
//   copied plane once and keeps them in registers for the H iterations in which the levels pass
//   it: read again by every level they took most of the shared-memory bandwidth (384^3 FP32 300 ->
//   425 GLUP/s, BF16, kept as stored and widened at each use, 363 -> 484).
// * Tiles overlap: a level's outermost columns / rows are wrong where the tile ends inside the
//   domain, one more per level, so neighbouring tiles recompute 4 columns (one vector) and
//   H - 1 rows on each side, and chunks of z recompute H planes. Tiles of one pass never wait for
//   each other.
// * All passes of a run are one persistent launch: (pass, tile) items are popped from a counter, and
//   a tile waits, bounded, until its 27 neighbours (itself among them) have finished the pass
//   before. At small grids there is no launch between passes, at large ones no last wave. The steps
//   that are left over (T % 3) are passes of one level.
// * The per-point operations and their order are those of common.cuh, so the results are
//   bit-identical to the plain sweep.
//
// What bounds it (GB300): a point costs about 5.5 instructions per lane (packed arithmetic, one
// shuffle per direction and row, no redundant shared-memory traffic), the diamond kernel of
// blocked_impl.cuh 24; HBM at 3 bytes per update is the next bound (about 2100 GLUP/s). Measured,
// 7-point constant, GLUP/s, AUTO before (diamonds) -> this: 1024^3 856 -> 1898, 512^3 727 -> 1610,
// 256^3 394 -> 1037, 301 x 257 x 199 241 -> 861, 64^3 16 -> 64 (plain sweep: 700, 682, 544, 503, 125; the
// rule of STENCIL_AUTO in api.cu has both sides from 64^3 to 160^3).
// 7-point variable 384^3: FP32 200 -> 425 (HBM at 5.2 TB/s, 13 bytes per update), BF16 253 -> 484
// (issue and latency of the widening).
#pragma once
#include <type_traits>

#include "internal.h"
#include "overlap.h"
#include "overlap_rings.h"
#include "tma.cuh"

namespace stg {

// Four consecutive x values as two packed pairs.
struct V4 {
    F2 a, b;
    static __device__ __forceinline__ V4 of(const float* v) { return V4{F2::pack(v[0], v[1]), F2::pack(v[2], v[3])}; }
    __device__ __forceinline__ void get(float* v) const {
        a.unpack(v[0], v[1]);
        b.unpack(v[2], v[3]);
    }
};

// Loads ordered only by the token tok of the barrier before them (the data was written before
// that barrier and is not rewritten until the next one): free to be scheduled within an iteration.
__device__ __forceinline__ V4 ov_lds(uint32_t a, uint32_t tok) {
    V4 r;
    asm("ld.shared.v2.b64 {%0, %1}, [%2];\n" : "=l"(r.a.r), "=l"(r.b.r) : "r"(a), "r"(tok));
    return r;
}
__device__ __forceinline__ void ov_sts(uint32_t a, const V4& x) {
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};\n" ::"r"(a), "l"(x.a.r), "l"(x.b.r));
}
__device__ __forceinline__ void ov_stg(float* p, const V4& x) {
    *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(x.a.r, x.b.r);
}
// One thread's coefficient vector as it is stored, and widened to FP32.
template <typename TC> struct OvCoef;
template <> struct OvCoef<float> {
    V4 v;
    __device__ __forceinline__ void ld(uint32_t a, uint32_t tok) { v = ov_lds(a, tok); }
    __device__ __forceinline__ V4 get() const { return v; }
};
template <> struct OvCoef<__nv_bfloat16> {
    uint32_t u0, u1;
    __device__ __forceinline__ void ld(uint32_t a, uint32_t tok) {
        asm("ld.shared.v2.u32 {%0, %1}, [%2];\n" : "=r"(u0), "=r"(u1) : "r"(a), "r"(tok));
    }
    __device__ __forceinline__ V4 get() const {
        // exact: a BF16 value is the upper half of its FP32 value
        return V4{F2::pack(__uint_as_float(u0 << 16), __uint_as_float(u0 & 0xffff0000u)),
                  F2::pack(__uint_as_float(u1 << 16), __uint_as_float(u1 & 0xffff0000u))};
    }
};
__device__ __forceinline__ uint32_t ov_bar(uint32_t x) {
    uint32_t t;
    asm volatile("bar.sync 0;\n\tmov.u32 %0, %1;\n" : "=r"(t) : "r"(x) : "memory");
    return t;
}
// Orders the loads that take the returned token after everything before it.
__device__ __forceinline__ uint32_t ov_order(uint32_t x) {
    uint32_t t;
    asm volatile("mov.u32 %0, %1;\n" : "=r"(t) : "r"(x) : "memory");
    return t;
}

// One grid of a launch: tile (bx, by, bz) of pass p reads f[(p0 + p) & 1] and writes the other
// array. The first `full` passes advance H steps, the others one.
struct OvGrid {
    CUtensorMap map[2];   // the field arrays, box (OV_X, NW RB + 2, 1)
    CUtensorMap cmap[7];  // the coefficient arrays, box (CXW, NW RB, 1)
    Layout L;
    float* f[2];
    float c0, c1, hv;
    int ntx, nty, ntz, zc;
    int p0, passes, full;
};

struct OvCtl {
    int* status;  // sticky: 1 once a wait gave up (may be null)
    int* never;   // a flag nothing sets (the stall hook waits on it)
    int* head;    // next item to pop
    int* done;    // per tile: passes finished
    unsigned spin_limit;
    int stall_item;
};

// Sizes of one instantiation. PD: field planes copied ahead; CR: coefficient planes held (the one
// being read and those in flight).
template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR>
struct OvCfg {
    static constexpr int NC = KindTraits<KIND>::NC;
    static constexpr int YT = NW * RB, YH = H - 1;
    static constexpr int ROWB = OV_X * 4;
    static constexpr int RING = PD + 2;                    // ahead, current, the one whose rows the neighbours read
    static constexpr int PLANEB = (YT + 2) * ROWB;         // rows -1 .. YT
    static constexpr int PR = RB == 1 ? 1 : 2;             // rows a warp publishes per level
    static constexpr int PUBL = (NW + 2) * PR * ROWB;      // one level's published rows
    // a copied coefficient row starts CX0 columns before the tile: its first element must lie on a
    // 16-byte boundary, and the tiles' first columns are odd multiples of 4 elements in the arrays
    static constexpr int CX0 = sizeof(TC) == 2 ? 4 : 0, CXW = OV_X + 2 * CX0;
    static constexpr int CROWB = CXW * (int)sizeof(TC);
    static constexpr int CARRB = (YT * CROWB + 127) / 128 * 128;  // one coefficient array's plane
    static constexpr int CPLANEB = NC * CARRB, CTXB = NC * YT * CROWB;
    static constexpr int COEF0 = RING * PLANEB;
    static constexpr int PUB0 = COEF0 + (NC > 0 ? CR * CPLANEB : 0);
    static constexpr int BAR0 = PUB0 + 2 * (H - 1) * PUBL;
    static constexpr int BYTES = BAR0 + (RING + CR) * 8;
    static_assert(PLANEB % 128 == 0 && PUB0 % 16 == 0, "box destinations stay 128-byte aligned");
};

// A value that is the same in every lane, told to the compiler (it then lives in uniform registers:
// 1892 against 1740 GLUP/s at 1024^3 for the warp index alone).
__device__ __forceinline__ int ov_uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// One tile of one pass, the whole CTA. HL: the levels it computes (H, or 1 in a short pass; the
// geometry is that of H either way). Thread 0 issues the copies.
// In a batch the grid's constants come from global memory: broadcast, so that they are uniform too.
template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR, int HL, bool BATCH>
__device__ __forceinline__ void overlap_tile(const OvGrid& A, const int src, const int bx, const int by, const int bz,
                                             const uint32_t s0, OvRings* ring, int* status) {
    using S = OvCfg<KIND, TC, NW, RB, H, PD, CR>;
    constexpr int YT = S::YT, YH = S::YH, NC = S::NC, PR = S::PR;
    const int lane = threadIdx.x & 31, w = ov_uniform((int)threadIdx.x >> 5);
    auto uni = [](int v) { return BATCH ? ov_uniform(v) : v; };
    const int nx = uni(A.L.nx), ny = uni(A.L.ny), nz = uni(A.L.nz), px = uni(A.L.px), py = uni(A.L.py), xo = uni(A.L.xo);
    const int ntx = uni(A.ntx), nty = uni(A.nty), zc = uni(A.zc);
    const float c0 = __int_as_float(uni(__float_as_int(A.c0))), c1 = __int_as_float(uni(__float_as_int(A.c1)));
    const int xs = ov_first(bx, OV_X, OV_V), ys = ov_first(by, YT, YH);  // first owned column and row
    const int xe = bx == ntx - 1 ? nx : ov_first(bx + 1, OV_X, OV_V);
    const int ye = by == nty - 1 ? ny : ov_first(by + 1, YT, YH);
    // the tile's first column and row; the last tile of several starts up to RB - 1 rows earlier,
    // so that the domain ends with a warp's last row
    const int xl = bx == 0 ? 0 : xs - OV_V;
    const int yl = by == 0 ? 0 : (by == nty - 1 ? ny - (ny - (ys - YH) + RB - 1) / RB * RB : ys - YH);
    const int x = xl + 4 * lane, y0 = yl + w * RB;  // this thread's first column and row
    const int z0 = bz * zc, z1 = min(nz, z0 + zc);
    const float hv = __int_as_float(uni(__float_as_int(A.hv)));
    const V4 hvv{F2::pack(hv, hv), F2::pack(hv, hv)};

    const bool live = y0 < ny;  // warp-uniform
    const int s_begin = max(z0 - HL, -1), s_end = z1 + HL;  // iterations [s_begin, s_end)
    const int zl = min(nz + 1, s_end);                      // field planes [s_begin, zl) are copied
    // coefficient planes [cb, ce) are copied (level 0 computes plane s - 1, usefully from z0 - HL + 1)
    const int cb = max(z0 - HL + 1, 0), ce = min(nz, s_end - 1);
    const uint32_t bar = s0 + S::BAR0, cbar = bar + 8 * S::RING;
    auto copy = [&](int z, int slot) {
        mbar_arrive_expect_tx(bar + 8 * slot, S::PLANEB);
        tma_load_3d(s0 + slot * S::PLANEB, &A.map[src], xo + xl, yl, z + 1, bar + 8 * slot);
    };
    auto ccopy = [&](int z, int slot) {
        if constexpr (NC > 0) {
            mbar_arrive_expect_tx(cbar + 8 * slot, S::CTXB);
#pragma unroll
            for (int m = 0; m < NC; ++m)
                tma_load_3d(s0 + S::COEF0 + slot * S::CPLANEB + m * S::CARRB, &A.cmap[m], xo + xl - S::CX0, yl + 1,
                            z + 1, cbar + 8 * slot);
        }
    };
    const OvRings r0{ov_uniform(ring->fs), ov_uniform(ring->cs), ov_uniform(ring->fp), ov_uniform(ring->cp), 0};
    if (threadIdx.x == 0) {
        for (int p = 0; p < PD; ++p)
            if (s_begin + p < zl) copy(s_begin + p, ov_slot(r0.fs, p, S::RING));
        if constexpr (NC > 0)
            for (int p = 0; p < CR - 1; ++p)
                if (cb + p < ce) ccopy(cb + p, ov_slot(r0.cs, p, CR));
    }
    const uint32_t own = s0 + (uint32_t)((w * RB + 1) * S::ROWB + lane * 16);
    const uint32_t cown = s0 + (uint32_t)(S::COEF0 + w * RB * S::CROWB + (S::CX0 + lane * 4) * (int)sizeof(TC));
    const uint32_t pub = s0 + (uint32_t)(S::PUB0 + w * PR * S::ROWB + lane * 16);  // entry of the warp above
    // rows outside the tile, and rows of warps outside the domain, hold the Dirichlet value
#pragma unroll 1
    for (int p = 0; p < 2 * (H - 1) && HL > 1; ++p) {
        const uint32_t o = pub + (uint32_t)(p * S::PUBL);
        if (w == 0) ov_sts(o + (PR - 1) * S::ROWB, hvv);
        if (w == NW - 1) ov_sts(o + 2 * PR * S::ROWB, hvv);
        if (!live) {
            ov_sts(o + PR * S::ROWB, hvv);
            if (PR == 2) ov_sts(o + 3 * S::ROWB, hvv);
        }
    }

    const size_t plane = (size_t)px * py;
    const bool xown = x >= xs && x < xe;
    float* dp = A.f[src ^ 1] + plane + (size_t)((live ? y0 : 0) + 1) * px + (xo + (xown ? x : 0));  // row y0, z = 0
    const bool xfull = x + 4 <= nx;
    bool st[RB];
#pragma unroll
    for (int i = 0; i < RB; ++i) st[i] = xown && y0 + i >= ys && y0 + i < ye;
    // CTA-uniform. 0: every column of the tile and its x neighbours are interior; 1: the domain
    // ends on a vector boundary; 2: some vector or warp straddles its end
    const bool straddle = (xl + OV_X > nx && nx % 4 != 0) || (yl + YT > ny && (ny - yl) % RB != 0);
    const int mode = straddle ? 2 : (bx == 0 || xl + OV_X >= nx ? 1 : 0);
    const bool ledge = lane == 0, redge = lane == 31 || x + 4 >= nx;

    V4 win[HL][3][RB];
#pragma unroll
    for (int l = 0; l < HL; ++l)
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int i = 0; i < RB; ++i) win[l][r][i] = hvv;

    OvCoef<TC> co[NC > 0 ? 3 : 1][NC > 0 ? NC : 1][RB];  // planes s - 1, s - 2, s - 3, rotating as the windows
    int sl = r0.fs, slf = (r0.fs + PD) % S::RING;      // ring slots of field planes s and s + PD
    uint32_t so = (uint32_t)(sl * S::PLANEB);          // byte offsets of field planes s and s - 1
    uint32_t sc = (uint32_t)((sl == 0 ? S::RING - 1 : sl - 1) * S::PLANEB);
    uint32_t ph = (uint32_t)r0.fp, par = 0, tok = 0;
    // coefficient slot of plane s - 1 (level 0's) and its phase, from plane cb on
    int cl = r0.cs;
    uint32_t cph = (uint32_t)r0.cp;
    // iteration in which a copy did not arrive in time (the results are invalid): no more copies
    // are issued and no more waits made, and the CTA walks no more tiles (overlap_rings.h)
    int lost = OV_NOT_LOST;
    auto arrived = [&](uint32_t b, uint32_t phase, int s) {
        if (!mbar_test(b, phase) && lost == OV_NOT_LOST && !mbar_wait(b, phase, status)) lost = s;
    };

    // STEADY: every plane of the iteration is a real plane and is stored. The other iterations
    // select instead of branching (1898 against 1776 GLUP/s at 1024^3, 1037 against 969 at 256^3:
    // the compiler then overlaps the levels).
    auto iter = [&](const int s, auto phase, auto edgec, auto steadyc) {
        constexpr int PH = decltype(phase)::value, EDGE = decltype(edgec)::value;
        constexpr bool STEADY = decltype(steadyc)::value;
        constexpr int ZM = PH % 3, ZC = (PH + 1) % 3, ZP = (PH + 2) % 3;
        const bool cnow = NC > 0 && (STEADY || (s - 1 >= cb && s - 1 < ce));
        if (threadIdx.x == 0 && lost == OV_NOT_LOST) {
            if (s + PD < zl) copy(s + PD, slf);
            if (NC > 0) {
                // the slot of plane s - 2, read in the iteration before: plane s - 2 + CR (those up to
                // cb + CR - 2 were copied at the start)
                const int z = s - 2 + CR;
                if (z >= cb + CR - 1 && z < ce) ccopy(z, cl >= 1 ? cl - 1 : CR - 1);
            }
        }
        if (STEADY || s < zl) arrived(bar + 8 * sl, ph, s);
        if (cnow) arrived(cbar + 8 * cl, cph, s);
        const uint32_t tw = ov_order(tok);
        if (live) {
            if (STEADY || s < zl) {
#pragma unroll
                for (int i = 0; i < RB; ++i) win[0][ZP][i] = ov_lds(own + so + (uint32_t)(i * S::ROWB), tw);
            }
            if constexpr (NC > 0) {
                // (a plane that was not copied feeds only points whose results are not used)
                const uint32_t cq = cown + (uint32_t)(cl * S::CPLANEB);
#pragma unroll
                for (int i = 0; i < RB; ++i)
#pragma unroll
                    for (int m = 0; m < NC; ++m) co[PH % 3][m][i].ld(cq + (uint32_t)(m * S::CARRB + i * S::CROWB), tw);
            }
            const uint32_t prd = pub + (par ^ (uint32_t)((H - 1) * S::PUBL));
            const uint32_t pwr = pub + par;
#pragma unroll
            for (int l = 0; l < HL; ++l) {
                const int z = s - l - 1;
                const bool zin = STEADY || (z >= 0 && z < nz);  // uniform
                V4 out[RB];
                V4 up, dn;
                if (l == 0) {
                    up = ov_lds(own + sc - (uint32_t)S::ROWB, tok);
                    dn = ov_lds(own + sc + (uint32_t)(RB * S::ROWB), tok);
                } else {
                    const uint32_t q = prd + (uint32_t)((l - 1) * S::PUBL);
                    up = ov_lds(q + (PR - 1) * S::ROWB, tok);  // last row of the warp above
                    dn = ov_lds(q + 2 * PR * S::ROWB, tok);    // first row of the warp below
                }
#pragma unroll
                for (int i = 0; i < RB; ++i) {
                    const V4 c = win[l][ZC][i];
                    const V4 ym = i == 0 ? up : win[l][ZC][i > 0 ? i - 1 : 0];
                    const V4 yp = i == RB - 1 ? dn : win[l][ZC][i < RB - 1 ? i + 1 : 0];
                    const V4 zm = win[l][ZM][i], zp = win[l][ZP][i];
                    float v[4];
                    c.get(v);
                    float xm0 = __shfl_up_sync(0xffffffffu, v[3], 1);
                    float xp3 = __shfl_down_sync(0xffffffffu, v[0], 1);
                    if constexpr (EDGE > 0) {
                        xm0 = ledge ? hv : xm0;
                        xp3 = redge ? hv : xp3;
                    }
                    if constexpr (KIND == K7C) {
                        // (one grid: read where they are used, from the parameter bank: 1905 GLUP/s at
                        // 1024^3, 1780 with both held in registers)
                        const float q0 = BATCH ? c0 : A.c0, q1 = BATCH ? c1 : A.c1;
                        const F2 c0p = F2::pack(q0, q0), c1p = F2::pack(q1, q1);
                        const F2 sxa = F2::pack(Ar<float>::add(v[1], xm0), Ar<float>::add(v[2], v[0]));
                        const F2 sxb = F2::pack(Ar<float>::add(v[3], v[1]), Ar<float>::add(xp3, v[2]));
                        out[i].a = upd7c_x2(c0p, c1p, c.a, sxa, yp.a, ym.a, zp.a, zm.a);
                        out[i].b = upd7c_x2(c0p, c1p, c.b, sxb, yp.b, ym.b, zp.b, zm.b);
                    } else {
                        // Listing 2's order; the x terms point by point (the neighbours are
                        // not register pairs), the others as packed pairs
                        const auto& k = co[NC > 0 ? (PH + 3 - l % 3) % 3 : 0];
                        V4 q = k[0][i].get();
                        V4 r{F2::mul(q.a, c.a), F2::mul(q.b, c.b)};
                        float o[4], kp[4], km[4];
                        r.get(o);
                        k[NC > 0 ? 1 : 0][i].get().get(kp);
                        k[NC > 0 ? 2 : 0][i].get().get(km);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            o[e] = Ar<float>::fma(kp[e], e < 3 ? v[e < 3 ? e + 1 : 0] : xp3, o[e]);
                            o[e] = Ar<float>::fma(km[e], e > 0 ? v[e > 0 ? e - 1 : 0] : xm0, o[e]);
                        }
                        r = V4::of(o);
                        auto term = [&](int m, const V4& u) {
                            q = k[NC > 0 ? m : 0][i].get();
                            r.a = F2::fma(q.a, u.a, r.a);
                            r.b = F2::fma(q.b, u.b, r.b);
                        };
                        term(3, yp);
                        term(4, ym);
                        term(5, zp);
                        term(6, zm);
                        out[i] = r;
                    }
                    if constexpr (EDGE == 2 || !STEADY) {
                        float o[4];
                        out[i].get(o);
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            o[e] = !zin || (EDGE == 2 && (x + e >= nx || y0 + i >= ny)) ? hv : o[e];
                        out[i] = V4::of(o);
                    }
                }
                if (l < HL - 1) {
                    const uint32_t q = pwr + (uint32_t)(l * S::PUBL + PR * S::ROWB);
                    ov_sts(q, out[0]);
                    if (PR == 2) ov_sts(q + S::ROWB, out[RB - 1]);
#pragma unroll
                    for (int i = 0; i < RB; ++i) win[l + 1 < HL ? l + 1 : 0][ZP][i] = out[i];
                } else if (STEADY || (z >= z0 && z < z1)) {
                    float* d = dp + (size_t)z * plane;
#pragma unroll
                    for (int i = 0; i < RB; ++i) {
                        if (EDGE < 2 || xfull) {
                            if (st[i]) ov_stg(d + (size_t)i * px, out[i]);
                        } else if (st[i]) {
                            float o[4];
                            out[i].get(o);
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (x + e < nx) d[(size_t)i * px + e] = o[e];
                        }
                    }
                }
            }
        }
        sc = so;
        so += S::PLANEB;
        if (++sl == S::RING) {
            sl = 0;
            so = 0;
            ph ^= 1u;
        }
        slf = slf + 1 == S::RING ? 0 : slf + 1;
        if (NC > 0 && (STEADY || s - 1 >= cb)) {
            if (++cl == CR) {
                cl = 0;
                cph ^= 1u;
            }
        }
        par ^= (uint32_t)((H - 1) * S::PUBL);
        tok = ov_bar(tok + 1);
    };
    // iterations whose planes s - HL .. s are all real and whose last level is stored
    const int t0 = z0 + HL, t1 = min(z1 + HL, nz);
    auto walk = [&](auto edgec) {
        int s = s_begin;
        auto gen = [&](int n) {  // iterations up to n, whole rotations
            for (; s < n; s += 3) {
                iter(s, std::integral_constant<int, 0>{}, edgec, std::false_type{});
                if (s + 1 < s_end) iter(s + 1, std::integral_constant<int, 1>{}, edgec, std::false_type{});
                if (s + 2 < s_end) iter(s + 2, std::integral_constant<int, 2>{}, edgec, std::false_type{});
            }
        };
        gen(min(t0, s_end));
        for (; s + 2 < t1; s += 3) {
            iter(s, std::integral_constant<int, 0>{}, edgec, std::true_type{});
            iter(s + 1, std::integral_constant<int, 1>{}, edgec, std::true_type{});
            iter(s + 2, std::integral_constant<int, 2>{}, edgec, std::true_type{});
        }
        gen(s_end);
    };
    tok = ov_bar(tok);
    if (HL < H || mode == 2) walk(std::integral_constant<int, 2>{});
    else if (mode == 1) walk(std::integral_constant<int, 1>{});
    else walk(std::integral_constant<int, 0>{});
    if (threadIdx.x == 0 && lost != OV_NOT_LOST) {
        ring->lost = 1;
        // the copies still in flight end before the CTA goes on (bounded): the last one of every slot
        const int fl = ov_last_field(s_begin, zl, lost, PD), cf = ov_last_coef(cb, ce, lost, CR);
        for (int p = max(0, fl - S::RING + 1); p <= fl; ++p)
            mbar_wait(bar + 8 * ov_slot(r0.fs, p, S::RING), (uint32_t)ov_phase(r0.fs, r0.fp, p, S::RING), status);
        for (int p = max(0, cf - CR + 1); NC > 0 && p <= cf; ++p)
            mbar_wait(cbar + 8 * ov_slot(r0.cs, p, CR), (uint32_t)ov_phase(r0.cs, r0.cp, p, CR), status);
    }
    // read by every thread after the barrier that follows the tile
    if (threadIdx.x == 0) ov_advance<(NC > 0)>(ring, r0, r0.fs + zl - s_begin, r0.cs + ce - cb, S::RING, CR);
}

__device__ __forceinline__ int ov_ld_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void ov_st_release(int* p, int v) {
    asm volatile("st.release.gpu.global.s32 [%0], %1;\n" ::"l"(p), "r"(v) : "memory");
}
// Bounded wait until *flag >= need; one that runs out sets the status word, after which no wait is made.
__device__ __forceinline__ void ov_wait_flag(const OvCtl& C, const int* flag, int need) {
    unsigned n = 0;
    while (ov_ld_acquire(flag) < need) {
        if (C.status && *(volatile const int*)C.status != 0) return;
        if (++n > C.spin_limit) {
            if (C.status) atomicCAS(C.status, 0, 1);
            return;
        }
        __nanosleep(64);
    }
}
// Lane n < 27 of a warp waits for neighbour n of tile (bx, by, bz), the tile itself among them, to
// have finished `need` passes: they hold what the tile reads, and have read what it overwrites.
__device__ __forceinline__ void ov_wait_tiles(const OvCtl& C, const int* done, int ntx, int nty, int ntz, int bx, int by,
                                              int bz, int need) {
    const int n = threadIdx.x & 31;
    const int x = bx + n % 3 - 1, y = by + n / 3 % 3 - 1, z = bz + n / 9 - 1;
    if (n < 27 && x >= 0 && x < ntx && y >= 0 && y < nty && z >= 0 && z < ntz)
        ov_wait_flag(C, done + x + ntx * (y + (size_t)nty * z), need);
    __syncwarp();
}

// Persistent launch over the (pass, tile) items of one grid in that order, popped from a counter:
// an item waits only for items before it, and every popped item is held by a running CTA that
// finishes the one before it first, so the launch ends with any number of resident CTAs.
template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR>
__global__ void __launch_bounds__(NW * 32, 1) overlap_kernel(const __grid_constant__ OvGrid G, const OvCtl C) {
    using S = OvCfg<KIND, TC, NW, RB, H, PD, CR>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_item;
    __shared__ OvRings s_ring;
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
    if (threadIdx.x == 0) {
        for (int p = 0; p < S::RING + CR; ++p) mbar_init(s0 + S::BAR0 + 8 * p, 1);
        mbar_init_fence();
        s_ring = OvRings{0, 0, 0, 0, 0};
    }
    const int tiles = G.ntx * G.nty * G.ntz, items = tiles * G.passes;
    int next = 0;  // thread 0: the item to do next
    if (threadIdx.x == 0) next = atomicAdd(C.head, 1);
    for (;;) {
        if (threadIdx.x < 32) {
            const int i = __shfl_sync(0xffffffffu, next, 0);
            if (i < items) {
                const int p = i / tiles, t = i - p * tiles;
                if (p > 0)
                    ov_wait_tiles(C, C.done, G.ntx, G.nty, G.ntz, t % G.ntx, t / G.ntx % G.nty, t / (G.ntx * G.nty), p);
                if (threadIdx.x == 0) {
                    if (i == C.stall_item) ov_wait_flag(C, C.never, 1);
                    next = atomicAdd(C.head, 1);
                    // what other CTAs stored (acquired above) is read by tensor copies next
                    fence_proxy_async_global();
                }
            }
            // (~i: published without being walked)
            if (threadIdx.x == 0) s_item = i < items && !ov_walks(s_ring) ? ~i : i;
        }
        __syncthreads();
        const int w = ov_uniform(s_item), i = w < 0 ? ~w : w;
        if (i >= items) break;
        const int p = i / tiles, t = i - p * tiles;
        const int bx = t % G.ntx, by = t / G.ntx % G.nty, bz = t / (G.ntx * G.nty), src = (G.p0 + p) & 1;
        if (w < 0) {
        } else if (p < G.full) overlap_tile<KIND, TC, NW, RB, H, PD, CR, H, false>(G, src, bx, by, bz, s0, &s_ring, C.status);
        else overlap_tile<KIND, TC, NW, RB, H, PD, CR, 1, false>(G, src, bx, by, bz, s0, &s_ring, C.status);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();  // with the barrier before it: the CTA's stores are visible GPU-wide
            ov_st_release(C.done + t, p + 1);
        }
    }
}

// The same over the items of many grids, in the order that the host planned (every item after those
// it waits for). Each grid's parity is read from and, once its last tile has finished, written to
// device memory, so that the launch can be replayed.
struct OvBatchArgs {
    const OvGrid* grids;
    const OvItem* items;
    int nitems;
    int* head;
    int* status;        // 1: a wait gave up
    int* never;
    int* gdone;         // per grid: items finished in this launch
    int* done;          // per tile (grid q from first[q]): passes finished
    const int* first;
    const int* ntiles;  // per grid: items per launch
    const int* parity_flip;  // per grid: T & 1
    int* parity;
    unsigned spin_limit;
};

template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR>
__global__ void __launch_bounds__(NW * 32, 1) overlap_batch_kernel(const OvBatchArgs B) {
    using S = OvCfg<KIND, TC, NW, RB, H, PD, CR>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_item, s_src;
    __shared__ OvRings s_ring;
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
    if (threadIdx.x == 0) {
        for (int p = 0; p < S::RING + CR; ++p) mbar_init(s0 + S::BAR0 + 8 * p, 1);
        mbar_init_fence();
        s_ring = OvRings{0, 0, 0, 0, 0};
    }
    const OvCtl C{B.status, B.never, B.head, B.done, B.spin_limit, -1};
    int next = 0;  // thread 0: the item to do next
    if (threadIdx.x == 0) next = atomicAdd(B.head, 1);
    for (;;) {
        if (threadIdx.x < 32) {
            const int i = __shfl_sync(0xffffffffu, next, 0);
            if (i < B.nitems) {
                const OvItem it = B.items[i];
                const bool stall = it.g < 0;
                const int g = stall ? ~it.g : it.g;
                const OvGrid& G = B.grids[g];
                const int ntx = G.ntx, nty = G.nty;
                if (it.p > 0)
                    ov_wait_tiles(C, B.done + B.first[g], ntx, nty, G.ntz, it.t % ntx, it.t / ntx % nty, it.t / (ntx * nty),
                                  it.p);
                if (threadIdx.x == 0) {
                    if (stall) ov_wait_flag(C, B.never, 1);
                    next = atomicAdd(B.head, 1);
                    const int p0 = *(volatile int*)(B.parity + g);
                    s_src = (p0 + it.p) & 1;
                    // what other CTAs stored (acquired above), and the grid's maps (written by the
                    // upload), are read through the copy engine next
                    fence_proxy_async_global();
                    tma_map_acquire(&G.map[s_src]);
                    for (int m = 0; m < S::NC; ++m) tma_map_acquire(&G.cmap[m]);
                }
            }
            // (~i: published without being walked)
            if (threadIdx.x == 0) s_item = i < B.nitems && !ov_walks(s_ring) ? ~i : i;
        }
        __syncthreads();
        const int w = ov_uniform(s_item), i = w < 0 ? ~w : w;
        if (i >= B.nitems) break;
        const int src = ov_uniform(s_src);
        const int ig = ov_uniform(B.items[i].g), g = ig < 0 ? ~ig : ig;
        const int p = ov_uniform(B.items[i].p), t = ov_uniform(B.items[i].t);
        const OvGrid& G = B.grids[g];
        const int ntx = ov_uniform(G.ntx), nty = ov_uniform(G.nty);
        const int bx = t % ntx, by = t / ntx % nty, bz = t / (ntx * nty);
        if (w < 0) {
        } else if (p < ov_uniform(G.full)) overlap_tile<KIND, TC, NW, RB, H, PD, CR, H, true>(G, src, bx, by, bz, s0, &s_ring, C.status);
        else overlap_tile<KIND, TC, NW, RB, H, PD, CR, 1, true>(G, src, bx, by, bz, s0, &s_ring, C.status);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();  // with the barrier before it: the CTA's stores are visible GPU-wide
            ov_st_release(B.done + B.first[g] + t, p + 1);
            // the last item of the grid: every other one has read the parity
            if (atomicAdd(B.gdone + g, 1) == B.ntiles[g] - 1) B.parity[g] ^= B.parity_flip[g];
        }
    }
}

// Host-side description of one grid (everything but the z chunk and the pass counts).
template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR>
cudaError_t overlap_grid(const SweepArgs& a, void* const field[2], OvGrid* G) {
    using S = OvCfg<KIND, TC, NW, RB, H, PD, CR>;
    const Layout& L = a.L;
    for (int i = 0; i < 2; ++i) {
        if (!tma_encode_3d(&G->map[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, field[i], L, OV_X, S::YT + 2))
            return cudaErrorNotSupported;
        G->f[i] = static_cast<float*>(field[i]);
    }
    for (int m = 0; m < S::NC; ++m)
        if (!tma_encode_3d(&G->cmap[m], sizeof(TC) == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                           (int)sizeof(TC), a.coef[m], L, S::CXW, S::YT))
            return cudaErrorNotSupported;
    G->L = L;
    G->c0 = (float)a.c0;
    G->c1 = (float)a.c1;
    G->hv = (float)a.halo;
    G->ntx = ov_tiles(L.nx, OV_X, OV_V);
    G->nty = ov_tiles(L.ny, S::YT, S::YH);
    return cudaSuccess;
}

template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR>
cudaError_t overlap_batch_go(const OvBatchArgs& B, int sms, cudaStream_t st) {
    using S = OvCfg<KIND, TC, NW, RB, H, PD, CR>;
    auto kfn = overlap_batch_kernel<KIND, TC, NW, RB, H, PD, CR>;
    cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, S::BYTES);
    if (e) return e;
    kfn<<<(unsigned)(B.nitems < sms ? B.nitems : sms), NW * 32, S::BYTES, st>>>(B);
    return cudaGetLastError();
}

// T steps in one launch: T / H passes of H steps and T % H of one. With an odd H every pass flips
// the parity as its steps do, so the result is in the array that T's parity names.
template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR>
cudaError_t overlap_launch(const SweepArgs& a, void* const field[2], int p0, int T, int chunks, int* ws, size_t ws_bytes,
                           const PersistCtl& ctl, cudaStream_t st, long long* launches) {
    using S = OvCfg<KIND, TC, NW, RB, H, PD, CR>;
    static_assert(H % 2 == 1, "a pass flips the parity once");
    const Layout& L = a.L;
    auto kfn = overlap_kernel<KIND, TC, NW, RB, H, PD, CR>;
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
    if ((e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, S::BYTES))) return e;
    OvGrid G{};
    if ((e = overlap_grid<KIND, TC, NW, RB, H, PD, CR>(a, field, &G))) return e;
    const long long columns = (long long)G.ntx * G.nty;
    G.zc = ov_chunk(columns, L.nz, H, sms, chunks);
    G.ntz = (L.nz + G.zc - 1) / G.zc;
    const long long tiles = columns * G.ntz;
    G.p0 = p0;
    G.full = T / H;
    G.passes = T / H + T % H;
    if (sizeof(int) * (size_t)(OV_WS_DONE + tiles) > ws_bytes || tiles * G.passes > INT_MAX / 2)
        return cudaErrorNotReady;
    if ((e = cudaMemsetAsync(ws + OV_WS_NEVER, 0, sizeof(int) * (size_t)(OV_WS_DONE - OV_WS_NEVER + tiles), st))) return e;
    OvCtl C{ws, ws + OV_WS_NEVER, ws + OV_WS_HEAD, ws + OV_WS_DONE, ctl.spin_limit, ctl.stall_item};
    const long long items = tiles * G.passes;
    kfn<<<(unsigned)(items < sms ? items : sms), NW * 32, S::BYTES, st>>>(G, C);
    if ((e = cudaGetLastError())) return e;
    if (launches) ++*launches;
    return cudaSuccess;
}

}  // namespace stg
