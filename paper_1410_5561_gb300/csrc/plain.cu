// Plain one-step-per-pass streaming sweep (the analog of the paper's spatially
// blocked baseline, Section IV, "Spt. Blk."): every launch reads u_t once and
// writes u_{t+1} once, so it moves 2*s_f + n_c*s_c bytes per LUP at best.
//
// Thread mapping: a warp covers 32 vectors of V = 16/sizeof(field) consecutive
// x values (128-bit accesses; FP64: fewer where a row is cut evenly, see launch_plain);
// a CTA stacks BY rows along y; each thread walks a chunk of z planes
// (sweep_column.cuh: register ring of the column's planes, neighbours through L1/L2,
// coefficients with evict-first loads). The number of z chunks is chosen from the
// kernel's occupancy so that the CTAs fill whole waves of the GPU.
#include <stdint.h>

#include "internal.h"
#include "occupancy.h"
#include "pdl.cuh"
#include "plain_plan.h"
#include "sweep_column.cuh"

namespace stg {

// Per stencil and element types: planes loaded ahead (PF) and the CTAs per SM the register
// allocation must allow (MINB), chosen by measurement on GB300. The constant-coefficient
// sweep has a single HBM stream per thread and wants loads in flight; the variable ones
// issue n_c + 1 streaming loads per plane already and are limited by the registers their
// coefficient vectors take (the 25-point BF16 / FP64 sweeps double their speed at 2 CTAs). The
// constant FP64 sweep is bound by the FP64 pipe and forms 3 of its 7 operations on the integer pipes
// (upd7c_soft): 512^3 79.6 -> 120 GLUP/s, 64^3 36 -> 52, 203 x 250 x 141 49 -> 88 (cut evenly, see
// launch_plain). GLUP/s at 512^3 by operations moved: the product 97, and one pair sum 102, two 120, three 97
// (more integer work than the pipe saved); registers: 4 CTAs 120, 3 118, 2 110, 5 (spills) 119.
// WARP_ROWS: a row per warp that the compiler knows of. With the width of a row as an argument the constant
// FP32 sweep, the one with the fewest operations a point, lost up to 19 % to the division and the registers that
// hold it (GLUP/s with the argument -> without, fields set and read back: 64^3 97 -> 110, 256^3 460 -> 534, 512^3
// 547 -> 594, 301 x 257 x 199 406 -> 488; run alone 512^3 615 -> 682, 1024^3 611 -> 700). The variable sweeps gain
// nothing from it from 192^3 on (7-point FP32 loses 1 %) and keep the argument.
template <int PF_, int MINB_, bool WARP_ROWS_ = false>
struct PlainCfgOf {
    static constexpr int PF = PF_, MINB = MINB_;
    static constexpr bool WARP_ROWS = WARP_ROWS_;
};
template <int KIND, typename TF, typename TC> struct PlainCfg : PlainCfgOf<1, 1> {};
template <> struct PlainCfg<K7C, float, float> : PlainCfgOf<3, 5, true> {};
template <> struct PlainCfg<K7C, double, double> : PlainCfgOf<1, 4> {};
template <> struct PlainCfg<K7V, float, float> : PlainCfgOf<0, 3> {};
template <> struct PlainCfg<K7V, double, double> : PlainCfgOf<0, 3> {};
template <> struct PlainCfg<K25V, float, float> : PlainCfgOf<0, 1> {};
template <> struct PlainCfg<K25V, float, __nv_bfloat16> : PlainCfgOf<1, 2> {};
template <> struct PlainCfg<K25V, double, double> : PlainCfgOf<1, 2> {};

template <int KIND, typename TF, typename TC, int BY, int PF>
__global__ void __launch_bounds__(32 * BY, (PlainCfg<KIND, TF, TC>::MINB))
plain_sweep_kernel(Layout L, const TF* __restrict__ src, TF* __restrict__ dst, CoefPtrs<TC> C,
                   TF c0, TF c1, int zchunk, int width) {
    constexpr int V = 16 / sizeof(TF);
    if (PlainCfg<KIND, TF, TC>::WARP_ROWS) width = 32;
    dependent_begin();
    const int ty = (int)threadIdx.x / width;
    const int i0 = (blockIdx.x * width + (threadIdx.x - ty * width)) * V;
    const int j = blockIdx.y * BY + ty;
    if (i0 >= L.nx || j >= L.ny || ty >= BY) return;
    const int k0 = blockIdx.z * zchunk;
    const int k1 = min(L.nz, k0 + zchunk);
    if (k0 >= k1) return;
    sweep_column<KIND, TF, TC, PF, true, false, KIND == K7C && sizeof(TF) == 8>(L, src, dst, C, c0, c1, i0, j, k0, k1);
}

// The plain sweep with every load of a plane copied D planes ahead into per-thread shared-memory
// slots (ColumnAsync): the copies in flight hold shared memory, not registers.
template <int KIND, typename TF, typename TC, int BY, int D>
__global__ void __launch_bounds__(32 * BY) plain_async_kernel(Layout L, const TF* __restrict__ src, TF* __restrict__ dst,
                                                              CoefPtrs<TC> C, TF c0, TF c1, int zchunk, int width) {
    constexpr int V = 16 / sizeof(TF);
    using Col = ColumnAsync<KIND, TF, TC, true, D>;
    extern __shared__ __align__(16) unsigned char plain_smem[];
    dependent_begin();
    const int ty = (int)threadIdx.x / width;
    const int i0 = (blockIdx.x * width + (threadIdx.x - ty * width)) * V;
    const int j = blockIdx.y * BY + ty;
    if (i0 >= L.nx || j >= L.ny || ty >= BY) return;
    const int k0 = blockIdx.z * zchunk;
    const int k1 = min(L.nz, k0 + zchunk);
    if (k0 >= k1) return;
    const int NT = (int)blockDim.x, tid = (int)threadIdx.x;
    const uint32_t s0 = (uint32_t)__cvta_generic_to_shared(plain_smem);
    Col col;
    col.begin(L, src, C, i0, j, k0, k1, s0 + (uint32_t)(tid * 16), (uint32_t)(NT * 16),
              s0 + (uint32_t)(D * Col::SF * NT * 16 + tid * Col::CB), (uint32_t)(NT * Col::CB));
    for (int k = k0; k < k1; ++k) col.plane(L, src, dst, C, c0, c1, i0, k);
}

// z chunks per column: minimise (waves of CTAs) x (planes per chunk + ring warm-up),
// with chunks of at least 16 planes, or of any size while those would not fill the GPU once: a thread
// walks its planes one memory latency after another (7-point constant FP64 64^3: 20.7 us a step in
// chunks of 16 planes, 7.4 in chunks of one). thin: the CTAs up to which chunks get thinner (0: slots; more
// CTAs than that fit where they are narrower, but thinner chunks then only repeat more first planes).
static int plain_chunks(long long xy, int nz, int R, int slots, int thin = 0) {
    if (slots <= 0) slots = 8 * 152;
    if (thin <= 0) thin = slots;
    int best = 1;
    long long best_cost = -1;
    int maxchunks = (nz + 15) / 16 > 0 ? (nz + 15) / 16 : 1;
    if (xy * maxchunks < thin) maxchunks = (int)(nz < thin / xy + 1 ? nz : thin / xy + 1);
    for (int n = 1; n <= maxchunks; ++n) {
        const int zc = (nz + n - 1) / n;
        const int nn = (nz + zc - 1) / zc;
        const long long waves = (xy * nn + slots - 1) / slots;
        const long long cost = waves * (zc + 2 * R);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = nn;
        }
    }
    return best;
}

template <int KIND, typename TF, typename TC>
static cudaError_t launch_plain(const SweepArgs& a, const void* src, void* dst, cudaStream_t s) {
    constexpr int BY = 8;
    constexpr int PF = PlainCfg<KIND, TF, TC>::PF;
    constexpr int V = 16 / sizeof(TF);
    const Layout& L = a.L;
    if (L.nx == 0 || L.ny == 0 || L.nz == 0) return cudaSuccess;
    CoefPtrs<TC> C{};
    for (int m = 0; m < KindTraits<KIND>::NC; ++m) C.c[m] = static_cast<const TC*>(a.coef[m]);
    unsigned gx = (unsigned)((L.nx + 32 * V - 1) / (32 * V));
    unsigned gy = (unsigned)((L.ny + BY - 1) / BY);
    if (a.plain_prefetch == 2) {
        constexpr int D = 2;
        using Col = ColumnAsync<KIND, TF, TC, true, D>;
        constexpr auto kernel = plain_async_kernel<KIND, TF, TC, BY, D>;
        constexpr size_t bytes = (size_t)D * (Col::SF * 16 + KindTraits<KIND>::NC * Col::CB);
        const PrefetchShape p = prefetch_shape(L.nx, V, BY, bytes, KIND == K25V);
        constexpr int FULL = 32 * BY * (int)bytes;
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, FULL);
        if (e != cudaSuccess) return e;
        const int slots = resident_ctas<kernel>(p.threads, p.smem);
        const int thin = resident_ctas<kernel>(32 * BY, FULL);
        const int nchunks = plain_chunks((long long)gx * gy, L.nz, KindTraits<KIND>::R, slots, thin);
        const int zchunk = (L.nz + nchunks - 1) / nchunks;
        return launch_dependent(true, kernel, dim3(gx, gy, (unsigned)nchunks), dim3((unsigned)p.threads), p.smem, s, L,
                                static_cast<const TF*>(src), static_cast<TF*>(dst), C, (TF)a.c0, (TF)a.c1, zchunk, p.width);
    }
    constexpr auto kernel = plain_sweep_kernel<KIND, TF, TC, BY, PF>;
    // Vectors of a row per CTA. FP64 (bound by its pipe, which idle lanes hold as well): the row is cut
    // evenly and the CTA's rows follow one another in its warps, GLUP/s at 203 x 250 x 141: 7-point
    // constant 46 -> 52, 7-point variable 59 -> 63, 25-point (130 x 200 x 162) 14.6 -> 19.0. FP32 (bound
    // by HBM): a row per warp; 25-point 303 x 150 x 141 92.0 GLUP/s, cut evenly 90.8.
    const int width = sizeof(TF) == 8 ? (L.nx + (int)gx * V - 1) / ((int)gx * V) : 32;
    // FP64 grids of fewer than BY rows have no threads for the others, so that more CTAs fit: 7-point constant 4096 x 1
    // x 4096, about 240 us a step, with 7 of 8 warps idle 750 (and 380 before it formed some operations on the
    // integer pipes, which one warp a scheduler does not hide).
    const int rows = sizeof(TF) == 8 && L.ny < BY ? L.ny : BY;
    const int threads = (width * rows + 31) / 32 * 32;
    const int slots = resident_ctas<kernel>(threads);
    const int nchunks = plain_chunks((long long)gx * gy, L.nz, KindTraits<KIND>::R, slots);
    const int zchunk = (L.nz + nchunks - 1) / nchunks;
    dim3 grid(gx, gy, (unsigned)nchunks);
    // Set up beside the step before it (pdl.cuh), 64^3, us per step: 7-point constant FP64 20.7 -> 7.4, FP32
    // 9.5 -> 2.8 (thinner chunks included), at 256^3 33.0 -> 31.0. Not every FP64 sweep (early_fp64).
    const bool early = sizeof(TF) == 4 || early_fp64((long long)gx * gy * nchunks, slots, zchunk);
    return launch_dependent(early, kernel, grid, dim3((unsigned)threads), 0, s, L, static_cast<const TF*>(src),
                            static_cast<TF*>(dst), C, (TF)a.c0, (TF)a.c1, zchunk, width);
}

cudaError_t plain_step(const SweepArgs& a, const void* src, void* dst, cudaStream_t s) {
    switch (a.kind) {
        case K7C:
            if (a.fdt == DT_F32) return launch_plain<K7C, float, float>(a, src, dst, s);
            if (a.fdt == DT_F64) return launch_plain<K7C, double, double>(a, src, dst, s);
            break;
        case K7V:
            if (a.fdt == DT_F32 && a.cdt == DT_F32) return launch_plain<K7V, float, float>(a, src, dst, s);
            if (a.fdt == DT_F32 && a.cdt == DT_BF16)
                return launch_plain<K7V, float, __nv_bfloat16>(a, src, dst, s);
            if (a.fdt == DT_F64 && a.cdt == DT_F64) return launch_plain<K7V, double, double>(a, src, dst, s);
            break;
        case K25V:
            if (a.fdt == DT_F32 && a.cdt == DT_F32) return launch_plain<K25V, float, float>(a, src, dst, s);
            if (a.fdt == DT_F32 && a.cdt == DT_BF16)
                return launch_plain<K25V, float, __nv_bfloat16>(a, src, dst, s);
            if (a.fdt == DT_F64 && a.cdt == DT_F64) return launch_plain<K25V, double, double>(a, src, dst, s);
            break;
    }
    return cudaErrorInvalidValue;
}

// ------------------------------------------------------------------ fill
template <typename T>
__global__ void fill_kernel(T* __restrict__ p, size_t n, T v) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        p[i] = v;
}

// ------------------------------------------------------------------ interior copy
// Dense (nz, ny, nx) rows <-> the padded layout's interior rows. Either side may be device
// memory or page-locked host memory mapped into the device's address space (read and written
// over the host link by the kernel's own loads and stores, which keeps many accesses in flight:
// faster than a pitched DMA of short rows). A warp moves a row in units of U, the widest type
// that divides both sides' addresses and the row length, four units per lane in flight; rows
// of an odd length so move by elements. Bound by HBM, or by the launch below 128^3: a CTA per row
// and single bytes for odd lengths took 170 us for 301 x 257 x 199 FP32, this 27 us (4.5 TB/s).
// Few long rows are cut into segments (copy_split), so that the GPU has warps for them.

// Row of this warp among ny, and the first unit of its segment. CUT: the rows are cut (without, the kernels know that a
// warp has a whole row: with the split's arithmetic a copy of 101 x 200 x 150 took 8.2 us, so 6.2).
template <bool CUT>
static __device__ __forceinline__ int copy_row(const CopySplit& c, size_t* first) {
    *first = 0;
    if (!CUT) return (int)(blockIdx.x * COPY_WARPS + threadIdx.y);
    const unsigned g = blockIdx.x / c.xblocks, xb = blockIdx.x - g * c.xblocks;
    *first = (size_t)(xb * (COPY_WARPS >> c.lg) + (threadIdx.y >> c.lg)) * (size_t)c.seg;
    return (int)((g << c.lg) + (threadIdx.y & ((1u << c.lg) - 1u)));
}
static dim3 copy_grid(const CopySplit& c, int ny, int nz, int arrays) {
    const unsigned groups = (unsigned)((ny + (1 << c.lg) - 1) >> c.lg);
    return dim3(groups * c.xblocks, (unsigned)(nz < 65535 ? nz : 65535), (unsigned)arrays);
}

template <typename U, bool CUT>
__global__ void __launch_bounds__(32 * COPY_WARPS) copy_rows_kernel(const char* __restrict__ src, char* __restrict__ dst,
                                                                   Layout L, int eb, int to_padded, CopySplit c) {
    size_t first;
    const int y = copy_row<CUT>(c, &first);
    if (y >= L.ny) return;
    const size_t rb = (size_t)L.nx * eb, all = rb / sizeof(U);
    const size_t n = CUT && first + (size_t)c.seg < all ? first + (size_t)c.seg : all;  // the segment's end
    for (int z = (int)blockIdx.y; z < L.nz; z += (int)gridDim.y) {
        const size_t pad = L.at(0, y, z) * (size_t)eb, den = ((size_t)z * L.ny + y) * rb;
        const U* a = reinterpret_cast<const U*>(src + (to_padded ? den : pad));
        U* b = reinterpret_cast<U*>(dst + (to_padded ? pad : den));
        for (size_t i = first + threadIdx.x; i < n; i += 32 * COPY_UNITS) {
            U v[COPY_UNITS];
#pragma unroll
            for (int u = 0; u < COPY_UNITS; ++u)
                if (i + 32 * u < n) v[u] = a[i + 32 * u];
#pragma unroll
            for (int u = 0; u < COPY_UNITS; ++u)
                if (i + 32 * u < n) b[i + 32 * u] = v[u];
        }
    }
}

// Widest unit (bytes) that divides every address and length in `bits` (or-ed together).
static int copy_unit(uintptr_t bits, int eb) {
    return (bits & 15u) == 0 ? 16 : (bits & 7u) == 0 ? 8 : (bits & 3u) == 0 ? 4 : (bits & 1u) == 0 && eb % 2 == 0 ? 2 : 1;
}

cudaError_t copy_rows(const Layout& L, int eb, const void* src, void* dst, bool to_padded, cudaStream_t s) {
    if (L.nx == 0 || L.ny == 0 || L.nz == 0) return cudaSuccess;
    const uintptr_t bits = (uintptr_t)src | (uintptr_t)dst | ((uintptr_t)L.nx * eb) | ((uintptr_t)L.xo * eb) |
                           ((uintptr_t)L.px * eb);
    const int unit = copy_unit(bits, eb);
    const CopySplit c = copy_split(L.ny, (long long)L.ny * L.nz, (long long)L.nx * eb / unit);
    const dim3 grid = copy_grid(c, L.ny, L.nz, 1), block(32, COPY_WARPS);
    const char* a = static_cast<const char*>(src);
    char* b = static_cast<char*>(dst);
    auto go = [&](auto u) {
        using U = decltype(u);
        if (c.cut()) copy_rows_kernel<U, true><<<grid, block, 0, s>>>(a, b, L, eb, to_padded, c);
        else copy_rows_kernel<U, false><<<grid, block, 0, s>>>(a, b, L, eb, to_padded, c);
    };
    switch (unit) {
        case 16: go(uint4{}); break;
        case 8: go(uint2{}); break;
        case 4: go(0u); break;
        case 2: go((unsigned short)0); break;
        default: go((unsigned char)0); break;
    }
    return cudaGetLastError();
}

// Dense arrays into padded ones with zeros in every other cell, all arrays in one launch and every
// padded byte written once (a fill and a copy of each array wrote the interior twice and took two
// launches an array).
struct PackArgs {
    const char* src[13];
    char* dst[13];
};

template <typename U, bool CUT>
__global__ void __launch_bounds__(32 * COPY_WARPS) pack_rows_kernel(const __grid_constant__ PackArgs P, Layout L, int eb,
                                                                   CopySplit c) {
    size_t first;
    const int r = copy_row<CUT>(c, &first);
    if (r >= L.py) return;
    const char* const src = P.src[blockIdx.z];
    char* const dst = P.dst[blockIdx.z];
    const long long lo = (long long)L.xo * eb / (int)sizeof(U), n = (long long)L.nx * eb / (int)sizeof(U);
    const long long all = (long long)L.px * eb / (int)sizeof(U);
    const long long np = CUT && (long long)first + c.seg < all ? (long long)first + c.seg : all;  // the segment's end
    const int y = r - L.R;
    for (int q = (int)blockIdx.y; q < L.pz; q += (int)gridDim.y) {
        const int z = q - L.R;
        const bool in = y >= 0 && y < L.ny && z >= 0 && z < L.nz;
        const U* a = reinterpret_cast<const U*>(src + (in ? ((size_t)z * L.ny + y) * ((size_t)L.nx * eb) : 0));
        U* b = reinterpret_cast<U*>(dst + ((size_t)q * L.py + r) * ((size_t)L.px * eb));
        for (long long i = (long long)first + threadIdx.x; i < np; i += 32 * COPY_UNITS) {
            U v[COPY_UNITS];
#pragma unroll
            for (int u = 0; u < COPY_UNITS; ++u) {
                const long long x = i + 32 * u - lo;
                v[u] = U{};
                if (in && x >= 0 && x < n) v[u] = a[x];
            }
#pragma unroll
            for (int u = 0; u < COPY_UNITS; ++u)
                if (i + 32 * u < np) b[i + 32 * u] = v[u];
        }
    }
}

cudaError_t pack_rows(const Layout& L, int eb, const void* const* src, void* const* dst, int n, cudaStream_t s) {
    PackArgs P{};
    uintptr_t bits = ((uintptr_t)L.nx * eb) | ((uintptr_t)L.xo * eb) | ((uintptr_t)L.px * eb);
    for (int m = 0; m < n; ++m) {
        P.src[m] = static_cast<const char*>(src[m]);
        P.dst[m] = static_cast<char*>(dst[m]);
        bits |= (uintptr_t)src[m] | (uintptr_t)dst[m];
    }
    const int unit = copy_unit(bits, eb);
    const CopySplit c = copy_split(L.py, (long long)L.py * L.pz * n, (long long)L.px * eb / unit);
    const dim3 grid = copy_grid(c, L.py, L.pz, n), block(32, COPY_WARPS);
    auto go = [&](auto u) {
        using U = decltype(u);
        if (c.cut()) pack_rows_kernel<U, true><<<grid, block, 0, s>>>(P, L, eb, c);
        else pack_rows_kernel<U, false><<<grid, block, 0, s>>>(P, L, eb, c);
    };
    switch (unit) {
        case 16: go(uint4{}); break;
        case 8: go(uint2{}); break;
        case 4: go(0u); break;
        case 2: go((unsigned short)0); break;
        default: go((unsigned char)0); break;
    }
    return cudaGetLastError();
}

// Dense copy by the SMs' own loads and stores, with few CTAs: each thread keeps DC_U
// independent 16-byte loads in flight, so a handful of SMs can stream host memory over the
// link while the other SMs run a sweep.
constexpr int DC_U = 8;
__global__ void __launch_bounds__(1024) dense_copy_kernel(const uint4* __restrict__ src, uint4* __restrict__ dst,
                                                          size_t n) {
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + (DC_U - 1) * stride < n; i += DC_U * stride) {
        uint4 v[DC_U];
#pragma unroll
        for (int u = 0; u < DC_U; ++u) v[u] = src[i + u * stride];
#pragma unroll
        for (int u = 0; u < DC_U; ++u) dst[i + u * stride] = v[u];
    }
    for (; i < n; i += stride) dst[i] = src[i];
}

cudaError_t dense_copy(void* dst, const void* src, size_t bytes, int ctas, cudaStream_t s) {
    if (bytes == 0) return cudaSuccess;
    dense_copy_kernel<<<(unsigned)ctas, 1024, 0, s>>>(static_cast<const uint4*>(src), static_cast<uint4*>(dst),
                                                      bytes / 16);
    return cudaGetLastError();
}

cudaError_t fill_value(void* p, size_t n, int dt, double v, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    unsigned blocks = (unsigned)((n + 255) / 256);
    if (blocks > 152u * 16u) blocks = 152u * 16u;
    if (dt == DT_F32) fill_kernel<float><<<blocks, 256, 0, s>>>((float*)p, n, (float)v);
    else if (dt == DT_F64) fill_kernel<double><<<blocks, 256, 0, s>>>((double*)p, n, v);
    else fill_kernel<__nv_bfloat16><<<blocks, 256, 0, s>>>((__nv_bfloat16*)p, n, __double2bfloat16(v));
    return cudaGetLastError();
}

}  // namespace stg
