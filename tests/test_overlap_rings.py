"""Copy rings of the overlapped sweep: a CTA's walk over its tiles, with a copy that arrives after the
wait for it has given up, played on the host with the functions that the kernel uses. In every tile that
has not lost a copy a wait returns only for the plane it waits for; no barrier is armed while its copy
is under way; and none is under way when the CTA ends."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "overlap_rings.h"
using namespace stg;
struct Ring {  // n slots, each with its barrier: completed phases, the copy under way, the plane held
    int n, done[16] = {}, held[16];
    bool flight[16] = {};
    int plane[16];
    int fault = 0;
    explicit Ring(int n_) : n(n_) { for (int q = 0; q < 16; ++q) held[q] = plane[q] = -1000; }
    void arm(int q, int z) { fault |= flight[q] ? 1 : 0; flight[q] = true; plane[q] = z; }
    void land(int q) { if (flight[q]) { flight[q] = false; held[q] = plane[q]; ++done[q]; } }
    void land_all(int but) { for (int q = 0; q < n; ++q) if (plane[q] != but) land(q); }
    bool test(int q, int phase) const { return (done[q] & 1) != phase; }
};
// One CTA's tiles: tile i has field planes [0, nf), coefficient planes [0, nc), iterations [0, its). In
// tile `bad` the copy of field plane `late` (of coefficient plane late, if coef) arrives only after the wait.
extern "C" int walk(int PD, int CR, const int* nfs, const int* ncs, int tiles, int bad, int late, int coef, int after) {
    const int RING = PD + 2;
    Ring F(RING), C(CR);
    OvRings r{0, 0, 0, 0, 0};
    int fault = 0, lost_seen = 0;
    for (int t = 0; t < tiles; ++t) {
        const int nf = nfs[t], nc = ncs[t], base = 100000 * (t + 1), its = nf + 3;
        if (!ov_walks(r)) continue;
        int lost = OV_NOT_LOST;
        const int lf = t == bad && !coef ? base + late : -1, lc = t == bad && coef ? base + late : -1;
        {
            for (int p = 0; p < PD && p < nf; ++p) F.arm(ov_slot(r.fs, p, RING), base + p);
            for (int p = 0; p < CR - 1 && p < nc; ++p) C.arm(ov_slot(r.cs, p, CR), base + p);
        }
        for (int s = 0; s < its; ++s) {
            // (coefficient plane s - 1 is read in iteration s, plane s - 2 + CR copied)
            if (lost == OV_NOT_LOST) {
                if (s + PD < nf) F.arm(ov_slot(r.fs, s + PD, RING), base + s + PD);
                const int z = s - 2 + CR;
                if (z >= CR - 1 && z < nc) C.arm(ov_slot(r.cs, z, CR), base + z);
            }
            F.land_all(lf);
            C.land_all(lc);
            auto read = [&](Ring& R, int p, int n, int s0, int ph, int size) {
                if (lost != OV_NOT_LOST || p < 0 || p >= n) return;
                const int q = ov_slot(s0, p, size);
                if (!R.test(q, ov_phase(s0, ph, p, size))) { lost = s; lost_seen = 1; }
                else if (R.held[q] != base + p) fault |= 2;  // let through, but another plane is there
            };
            read(F, s, nf, r.fs, r.fp, RING);
            read(C, s - 1, nc, r.cs, r.cp, CR);
        }
        const OvRings r0 = r;
        if (lost != OV_NOT_LOST) {
            const int mf = ov_last_field(0, nf, lost, PD) + 1, mc = ov_last_coef(0, nc, lost, CR) + 1;
            // the late copy lands now: the waits for the last copy of every slot see all of them end
            for (int q = 0; q < RING; ++q) F.land(q);
            for (int q = 0; q < CR; ++q) C.land(q);
            for (int p = mf > RING ? mf - RING : 0; p < mf; ++p) {
                const int q = ov_slot(r.fs, p, RING);
                if (!F.test(q, ov_phase(r.fs, r.fp, p, RING)) || F.held[q] != base + p) fault |= 4;
            }
            for (int p = mc > CR ? mc - CR : 0; p < mc; ++p) {
                const int q = ov_slot(r.cs, p, CR);
                if (!C.test(q, ov_phase(r.cs, r.cp, p, CR)) || C.held[q] != base + p) fault |= 4;
            }
        }
        if (lost != OV_NOT_LOST) r.lost = 1;
        ov_advance<true>(&r, r0, r0.fs + nf, r0.cs + nc, RING, CR);
        if (t > bad && bad >= 0 && lost_seen && lost == OV_NOT_LOST && after) fault |= 8;  // copied again
    }
    for (int q = 0; q < RING; ++q) fault |= F.flight[q] ? 16 : 0;
    for (int q = 0; q < CR; ++q) fault |= C.flight[q] ? 16 : 0;
    return (fault | F.fault | C.fault) + (lost_seen << 8);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rings")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1410_5561_gb300", "csrc"), str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _walk(lib, PD, CR, tiles, bad=-1, late=0, coef=0):
    n = len(tiles)
    nf = (ctypes.c_int * n)(*[t[0] for t in tiles])
    nc = (ctypes.c_int * n)(*[t[1] for t in tiles])
    return lib.walk(PD, CR, nf, nc, n, bad, late, coef, 1)


TILES = [(9, 7), (5, 4), (17, 15), (4, 2), (26, 24), (8, 6)]


@pytest.mark.parametrize("PD,CR", [(4, 3), (4, 2), (3, 3), (2, 4)])
def test_rings_with_every_copy_in_time(lib, PD, CR):
    for n in range(1, len(TILES) + 1):
        assert _walk(lib, PD, CR, TILES[:n]) == 0


@pytest.mark.parametrize("PD,CR", [(4, 3), (4, 2), (3, 3), (2, 4)])
@pytest.mark.parametrize("coef", [0, 1])
def test_rings_after_a_late_copy(lib, PD, CR, coef):
    for bad, t in enumerate(TILES):
        for late in range(t[coef]):
            assert _walk(lib, PD, CR, TILES, bad, late, coef) == 256, (bad, late)  # lost, and no fault
