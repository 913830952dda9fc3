// Overlapped-tile sweep: entry points (kernels and launcher in overlap_impl.cuh).
#include "overlap_impl.cuh"

namespace stg {

bool overlap_ok(const SweepArgs& a) {
    return (a.kind == K7C || a.kind == K7V) && a.fdt == DT_F32 && a.L.xo == OV_V;
}

cudaError_t overlap_run(const SweepArgs& a, void* const field[2], int p0, int T, int chunks, int* ws, size_t ws_bytes,
                        const PersistCtl& ctl, cudaStream_t st, long long* launches) {
    if (!overlap_ok(a)) return cudaErrorInvalidValue;
    // H = 3: an odd pass keeps the parity rule, and 16 warps of 2 rows hold three levels in 128
    // registers without spills. Measured at 1024^3 (7-point constant, GLUP/s): 16 x 2 rows H = 3 1751,
    // H = 4 1447 (spills), 12 x 3 H = 3 1656, 12 x 2 H = 4 1531, 8 x 4 H = 3 1722, H = 4 1573, 16 x 3 H = 2 1423.
    // Variable coefficients take 28 registers a plane and row in FP32 (14 in BF16), three planes deep: one
    // row a warp, 12 warps (BF16: 16; 384^3, GLUP/s: 16 warps 484, 12 warps 446, widened once 464, 8 x 2 388).
    constexpr int H = 3;
    if (a.kind == K7C)
        return overlap_launch<K7C, float, 16, 2, H, 4, 1>(a, field, p0, T, chunks, ws, ws_bytes, ctl, st, launches);
    if (a.cdt == DT_BF16)
        return overlap_launch<K7V, __nv_bfloat16, 16, 1, H, 4, 3>(a, field, p0, T, chunks, ws, ws_bytes, ctl, st, launches);
    return overlap_launch<K7V, float, 12, 1, H, 4, 3>(a, field, p0, T, chunks, ws, ws_bytes, ctl, st, launches);
}

}  // namespace stg
