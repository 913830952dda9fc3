// Overlapped-tile sweep: geometry shared by the host and the kernel, and the launcher.
#pragma once
#include "internal.h"

namespace stg {

// Along x a tile is one warp of vectors (OV_X columns), of which one vector (OV_V columns) per
// inner side is computed redundantly.
constexpr int OV_X = 128, OV_V = 4;

// Tiles that cover n cells with tiles of `span` cells of which `halo` on each inner side are
// redundant (none at the ends of the domain).
__host__ __device__ inline int ov_tiles(int n, int span, int halo) {
    if (n <= span) return 1;
    const int rest = n - 2 * (span - halo), inner = span - 2 * halo;
    return 2 + (rest > 0 ? (rest + inner - 1) / inner : 0);
}
// First cell that tile b owns.
__host__ __device__ inline int ov_first(int b, int span, int halo) {
    return b == 0 ? 0 : (span - halo) + (b - 1) * (span - 2 * halo);
}

// Workspace words (ints): the status word (shared with the other persistent schedules), a flag
// nothing sets, the item counter, then the passes finished per tile.
constexpr int OV_WS_STATUS = 0, OV_WS_NEVER = 1, OV_WS_HEAD = 2, OV_WS_DONE = 3;

// Planes per z chunk: the number of chunks that minimises waves of CTAs (one per SM) x iterations
// of a CTA (its planes, 2 H redundant ones, and about OV_START iterations to start), or the given
// number of chunks. A chunk has at least OV_MINZ planes unless it is the only one: a tile reads
// from, and is read by, the next tile on each side only.
constexpr int OV_START = 4, OV_MINZ = 4;
inline int ov_chunk(long long tiles, int nz, int H, int sms, int chunks) {
    const int most = nz / OV_MINZ > 1 ? nz / OV_MINZ : 1;
    if (chunks > 0) return (nz + (chunks < most ? chunks : most) - 1) / (chunks < most ? chunks : most);
    int best = nz;
    long long cost = -1;
    for (int n = 1; n <= most && n <= 8 * sms; ++n) {
        const int zc = (nz + n - 1) / n;
        const long long c = (tiles * ((nz + zc - 1) / zc) + sms - 1) / sms * (zc + 2 * H + OV_START);
        if (cost < 0 || c < cost) {
            cost = c;
            best = zc;
        }
    }
    return best;
}

}  // namespace stg
