// Positions of the overlapped sweep's copy rings (overlap_impl.cuh), carried by a CTA from one tile
// to the next. Host and device code, no CUDA needed.
//
// A plane is copied into the slots of its ring in turn; slot q's barrier completes one phase per
// copy, so a reader waits for the phase that the number of earlier turns gives. If a copy does not
// arrive in time (the results are invalid then, and the status word says so), the CTA stops
// copying: it waits, bounded, for the copies that are under way, and walks none of the tiles that it
// takes from there on (they are published as finished, so that no other CTA waits for them). A later tile that
// copied again would meet barriers whose phases no longer follow from the positions: it could arm
// one whose copy has not landed, and leave the CTA with copies under way into its shared memory.
#pragma once
#include <limits.h>

#ifdef __CUDACC__
#define OV_FN __host__ __device__ __forceinline__
#else
#define OV_FN inline
#endif

namespace stg {

#ifndef __CUDACC__
inline int min(int a, int b) { return a < b ? a : b; }
inline int max(int a, int b) { return a > b ? a : b; }
#endif

// Slot and phase of the next field plane (fs, fp) and coefficient plane (cs, cp); lost: a copy did
// not arrive.
struct OvRings {
    int fs, cs, fp, cp, lost;
};

constexpr int OV_NOT_LOST = INT_MAX;

// Whether the CTA walks its next tile.
OV_FN bool ov_walks(const OvRings& r) { return r.lost == 0; }

// The last planes that a tile had issued when it stopped in iteration `lost`, counted from its first ones: field
// planes s_begin .. zl - 1 are copied PD ahead, coefficient planes cb .. ce - 1 into CR slots.
OV_FN int ov_last_field(int s_begin, int zl, int lost, int PD) { return min(zl, lost + PD + 1) - 1 - s_begin; }
OV_FN int ov_last_coef(int cb, int ce, int lost, int CR) { return min(ce, max(cb + CR - 1, lost + CR - 1)) - 1 - cb; }

// Slot and phase of plane p of a tile (counted from its first one) whose first plane has slot s and phase ph.
OV_FN int ov_slot(int s, int p, int ring) { return (s + p) % ring; }
OV_FN int ov_phase(int s, int ph, int p, int ring) { return ph ^ ((s + p) / ring & 1); }

// Positions after a tile; nf, nc: its first slots plus the planes that it copies (COEF: it has coefficient planes).
template <bool COEF>
OV_FN void ov_advance(OvRings* r, const OvRings& r0, int nf, int nc, int ring, int cr) {
    r->fs = nf % ring;
    r->fp = r0.fp ^ (nf / ring & 1);
    if (COEF) r->cs = nc % cr;
    if (COEF) r->cp = r0.cp ^ (nc / cr & 1);
}

}  // namespace stg
