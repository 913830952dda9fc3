// Positions of the overlapped sweep's copy rings (overlap_impl.cuh), carried by a CTA from one tile
// to the next. Host and device code, no CUDA needed.
//
// A plane is copied into the slots of its ring in turn; slot q's barrier completes one phase per
// copy, so a reader waits for the phase that the number of earlier turns gives. If a copy does not
// arrive in time (the results are invalid then, and the status word says so), the CTA stops
// copying: it waits, bounded, for the copies that are under way and issues none from there on, in
// that tile or in any later one. A later tile that copied again would meet barriers whose phases no
// longer follow from the positions: it could arm one whose copy has not landed, and leave the
// CTA with copies under way into its shared memory.
#pragma once
#include <limits.h>

#ifdef __CUDACC__
#define OV_FN __host__ __device__ __forceinline__
#else
#define OV_FN inline
#endif

namespace stg {

// Slot and phase of the next field plane (fs, fp) and coefficient plane (cs, cp); lost: a copy did
// not arrive.
struct OvRings {
    int fs, cs, fp, cp, lost;
};

constexpr int OV_NOT_LOST = INT_MAX;

// The iteration in which copies stopped, as a tile that begins at iteration s_begin finds it.
OV_FN int ov_lost_before(const OvRings& r, int s_begin) { return r.lost ? s_begin - 1 : OV_NOT_LOST; }

// Planes that a tile had issued when it stopped in iteration `lost` (not before s_begin): field planes
// from s_begin on (at most zl - s_begin, copied PD ahead), coefficient planes from cb on (at
// most ce - cb, copied into CR slots).
OV_FN int ov_issued_fields(int s_begin, int zl, int lost, int PD) {
    const int n = (zl < lost + PD + 1 ? zl : lost + PD + 1) - s_begin;
    return n > 0 ? n : 0;
}
OV_FN int ov_issued_coefs(int cb, int ce, int lost, int CR) {
    const int m = lost + CR - 1 > cb + CR - 1 ? lost + CR - 1 : cb + CR - 1;
    const int n = (ce < m ? ce : m) - cb;
    return n > 0 ? n : 0;
}

// Slot and phase of plane p of a tile (counted from its first one) whose first plane has slot s and phase ph.
OV_FN int ov_slot(int s, int p, int ring) { return (s + p) % ring; }
OV_FN int ov_phase(int s, int ph, int p, int ring) { return ph ^ ((s + p) / ring & 1); }

// After a tile of nf field planes and nc coefficient planes; lost: the CTA stopped copying.
OV_FN OvRings ov_rings_after(const OvRings& r, int nf, int nc, int ring, int cr, bool lost) {
    return OvRings{ov_slot(r.fs, nf, ring), ov_slot(r.cs, nc, cr), ov_phase(r.fs, r.fp, nf, ring),
                   ov_phase(r.cs, r.cp, nc, cr), lost ? 1 : 0};
}

}  // namespace stg
