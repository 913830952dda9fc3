// Overlapped-tile sweep: entry points for one grid and for a batch (kernels and launchers in
// overlap_impl.cuh).
#include <algorithm>
#include <queue>

#include "overlap_impl.cuh"

namespace stg {

bool overlap_ok(const SweepArgs& a) {
    return (a.kind == K7C || a.kind == K7V) && a.fdt == DT_F32 && a.L.xo == OV_V;
}

// Kernel configuration of a grid (overlap_ok): the template arguments KIND, TC, NW, RB, H, PD, CR.
//
// H = 3: an odd pass keeps the parity rule, and 16 warps of 2 rows hold three levels in 128
// registers without spills. Measured at 1024^3 (7-point constant, GLUP/s): 16 x 2 rows H = 3 1751,
// H = 4 1447 (spills), 12 x 3 H = 3 1656, 12 x 2 H = 4 1531, 8 x 4 H = 3 1722, H = 4 1573, 16 x 3 H = 2 1423.
// Variable coefficients take 28 registers a plane and row in FP32 (14 in BF16), three planes deep: one
// row a warp, 12 warps (BF16: 16; 384^3, GLUP/s: 16 warps 484, 12 warps 446, widened once 464, 8 x 2 388).
constexpr int OV_H = 3;
#define OV_7C K7C, float, 16, 2, OV_H, 4, 1
#define OV_7V K7V, float, 12, 1, OV_H, 4, 3
#define OV_7VB K7V, __nv_bfloat16, 16, 1, OV_H, 4, 3
#define OV_CALL(kind, cdt, fn, ...) \
    ((kind) == K7C ? fn<OV_7C>(__VA_ARGS__) : (cdt) == DT_BF16 ? fn<OV_7VB>(__VA_ARGS__) : fn<OV_7V>(__VA_ARGS__))

cudaError_t overlap_run(const SweepArgs& a, void* const field[2], int p0, int T, int chunks, int* ws, size_t ws_bytes,
                        const PersistCtl& ctl, cudaStream_t st, long long* launches) {
    if (!overlap_ok(a)) return cudaErrorInvalidValue;
    return OV_CALL(a.kind, a.cdt, overlap_launch, a, field, p0, T, chunks, ws, ws_bytes, ctl, st, launches);
}

// ------------------------------------------------------------------ batch

namespace {

template <int KIND, typename TC, int NW, int RB, int H, int PD, int CR>
long long columns_of(const Layout& L) {
    using S = OvCfg<KIND, TC, NW, RB, H, PD, CR>;
    return (long long)ov_tiles(L.nx, OV_X, OV_V) * ov_tiles(L.ny, S::YT, S::YH);
}

struct PlanGrid {
    long long columns;
    int nz, passes, full, chunks, zc, ntz;
    // iterations of one tile of pass p
    int cost(int p) const { return zc + 2 * (p < full ? OV_H : 1) + OV_START; }
    void cut(int n) {
        chunks = n;
        zc = (nz + n - 1) / n;
        ntz = (nz + zc - 1) / zc;
    }
};

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// The items in the order of a list schedule on the GPU's SMs: a tile of the ready pass with the
// longest remaining chain of passes first, a pass being ready when the one before it has been
// scheduled to end. So a CTA that pops an item seldom waits, and the grids with most steps do not
// run last on an empty GPU. A grid's columns are cut in z only as far as its chain of passes would
// otherwise outlast its share of the whole batch.
cudaError_t overlap_batch_plan(const BatchGrid* g, int n, size_t limit, BatchLaunch* bl) {
    bl->overlap = false;
    for (int q = 0; q < n; ++q)
        if (!overlap_ok(g[q].a)) return cudaSuccess;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return cudaErrorInvalidDevice;
    std::vector<PlanGrid> P(n);
    for (int q = 0; q < n; ++q) {
        const SweepArgs& a = g[q].a;
        P[q].columns = OV_CALL(a.kind, a.cdt, columns_of, a.L);
        P[q].nz = a.L.nz;
        P[q].full = g[q].T / OV_H;
        P[q].passes = g[q].T / OV_H + g[q].T % OV_H;
        P[q].cut(1);
    }
    auto chain = [&](const PlanGrid& p) { return (double)p.full * p.cost(0) + (double)(p.passes - p.full) * p.cost(p.full); };
    double work = 0;
    for (const PlanGrid& p : P) work += chain(p) * (double)(p.columns * p.ntz);
    std::priority_queue<std::pair<double, int>> longest;
    for (int q = 0; q < n; ++q)
        if (P[q].passes > 0) longest.push({chain(P[q]), q});
    while (!longest.empty()) {
        const int q = longest.top().second;
        PlanGrid& p = P[q];
        if (chain(p) <= 0.7 * work / sms || p.nz / (p.chunks + 1) < OV_MINZ) break;
        longest.pop();
        work -= chain(p) * (double)(p.columns * p.ntz);
        p.cut(p.chunks + 1);
        work += chain(p) * (double)(p.columns * p.ntz);
        longest.push({chain(p), q});
    }
    long long items = 0, counters = 0;
    bl->ov_zc.assign(n, 1);
    bl->ov_first.assign(n, 0);
    for (int q = 0; q < n; ++q) {
        bl->ov_zc[q] = P[q].zc;
        bl->ov_first[q] = (int)counters;
        counters += P[q].columns * P[q].ntz;
        items += P[q].columns * P[q].ntz * P[q].passes;
        if (items > (1 << 28) || counters > (1 << 28)) return cudaSuccess;
    }
    size_t off = 64;  // the tensor maps want 64-byte alignment, which the workspace need not have
    const size_t o_grids = off;
    off += up256(sizeof(OvGrid) * (size_t)n);
    const size_t o_items = off;
    off += up256(sizeof(OvItem) * (size_t)items);
    const size_t o_ntiles = off;
    off += up256(sizeof(int) * (size_t)n);
    const size_t o_parity = off;
    off += up256(sizeof(int) * (size_t)n);
    const size_t o_first = off;
    off += up256(sizeof(int) * (size_t)n);
    const size_t o_flip = off;
    off += up256(sizeof(int) * (size_t)n);
    const size_t o_counters = off;  // head, status, never, gdone[n], done[counters]
    const size_t counter_bytes = sizeof(int) * (size_t)(3 + n + counters);
    off += up256(counter_bytes);
    if (off > limit) return cudaSuccess;
    bl->off_grids = o_grids;
    bl->off_items = o_items;
    bl->off_ntiles = o_ntiles;
    bl->off_parity = o_parity;
    bl->off_first = o_first;
    bl->off_flip = o_flip;
    bl->off_counters = o_counters;
    bl->counter_bytes = counter_bytes;
    bl->bytes = std::max(bl->diamond_bytes, off);

    std::vector<OvItem>& out = bl->ov_items;
    out.clear();
    out.reserve((size_t)items);
    bl->ntiles.assign(n, 0);
    struct Next { int pass; long long tile, left; double rest; };
    std::vector<Next> st(n);
    auto shorter = [&](int a, int b) { return st[a].rest < st[b].rest || (st[a].rest == st[b].rest && a > b); };
    std::priority_queue<int, std::vector<int>, decltype(shorter)> ready(shorter);
    for (int q = 0; q < n; ++q) {
        st[q] = {0, 0, P[q].columns * P[q].ntz, chain(P[q])};
        bl->ntiles[q] = (int)(P[q].columns * P[q].ntz * P[q].passes);
        if (P[q].passes > 0) ready.push(q);
    }
    typedef std::pair<long long, int> Event;  // (end of a tile, its grid)
    std::priority_queue<Event, std::vector<Event>, std::greater<Event>> running;
    long long now = 0;
    while (!ready.empty() || !running.empty()) {
        while (!ready.empty() && (int)running.size() < sms) {
            const int q = ready.top();
            Next& s = st[q];
            out.push_back(OvItem{q, s.pass, (int)s.tile});
            running.push({now + P[q].cost(s.pass), q});
            if (++s.tile == P[q].columns * P[q].ntz) ready.pop();
        }
        const int q = running.top().second;
        now = running.top().first;
        running.pop();
        Next& s = st[q];
        if (--s.left == 0) {
            s.rest -= P[q].cost(s.pass);
            if (++s.pass < P[q].passes) {
                s.tile = 0;
                s.left = P[q].columns * P[q].ntz;
                ready.push(q);
            }
        }
    }
    bl->items.clear();
    bl->nitems = (int)out.size();
    bl->overlap = true;
    return cudaSuccess;
}

static size_t aligned64(const char* ws) { return (64 - ((uintptr_t)ws & 63u)) & 63u; }

cudaError_t overlap_batch_upload(const BatchGrid* g, int n, BatchLaunch* bl, char* ws, cudaStream_t s) {
    std::vector<OvGrid> G(n);
    std::vector<int> par(n), flip(n);
    cudaError_t e;
    for (int q = 0; q < n; ++q) {
        const SweepArgs& a = g[q].a;
        if ((e = OV_CALL(a.kind, a.cdt, overlap_grid, a, g[q].field, &G[q]))) return e;
        G[q].zc = bl->ov_zc[q];
        G[q].ntz = (a.L.nz + G[q].zc - 1) / G[q].zc;
        G[q].full = g[q].T / OV_H;
        G[q].passes = g[q].T / OV_H + g[q].T % OV_H;
        par[q] = g[q].parity;
        flip[q] = g[q].T & 1;
    }
    // (the maps move down to the first 64-byte boundary of the workspace: off_grids leaves 64 bytes)
    const std::pair<size_t, std::pair<const void*, size_t>> parts[] = {
        {bl->off_grids - 64 + aligned64(ws), {G.data(), sizeof(OvGrid) * (size_t)n}},
        {bl->off_items, {bl->ov_items.data(), sizeof(OvItem) * bl->ov_items.size()}},
        {bl->off_ntiles, {bl->ntiles.data(), sizeof(int) * (size_t)n}},
        {bl->off_parity, {par.data(), sizeof(int) * (size_t)n}},
        {bl->off_first, {bl->ov_first.data(), sizeof(int) * (size_t)n}},
        {bl->off_flip, {flip.data(), sizeof(int) * (size_t)n}},
    };
    for (const auto& p : parts)
        if (p.second.second > 0 &&
            (e = cudaMemcpyAsync(ws + p.first, p.second.first, p.second.second, cudaMemcpyHostToDevice, s)))
            return e;
    return cudaStreamSynchronize(s);  // host vectors are freed on return
}

cudaError_t overlap_batch_launch(const BatchLaunch& bl, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
    char* ws = bl.ws;
    int* cnt = reinterpret_cast<int*>(ws + bl.off_counters);
    if ((e = cudaMemsetAsync(cnt, 0, bl.counter_bytes, s))) return e;
    if (bl.nitems < 1) return cudaSuccess;
    OvBatchArgs B{};
    B.grids = reinterpret_cast<const OvGrid*>(ws + bl.off_grids - 64 + aligned64(ws));
    B.items = reinterpret_cast<const OvItem*>(ws + bl.off_items);
    B.nitems = bl.nitems;
    B.head = cnt;
    B.status = cnt + 1;
    B.never = cnt + 2;
    B.gdone = cnt + 3;
    B.done = cnt + 3 + bl.ngrids;
    B.first = reinterpret_cast<const int*>(ws + bl.off_first);
    B.ntiles = reinterpret_cast<const int*>(ws + bl.off_ntiles);
    B.parity_flip = reinterpret_cast<const int*>(ws + bl.off_flip);
    B.parity = reinterpret_cast<int*>(ws + bl.off_parity);
    B.spin_limit = bl.spin_limit;
    return OV_CALL(bl.kind, bl.cdt, overlap_batch_go, B, sms, s);
}

}  // namespace stg
