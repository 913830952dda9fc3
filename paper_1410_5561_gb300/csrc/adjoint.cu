// Adjoint (reverse-mode) sweep of the variable-coefficient stencils.
//
// Forward (Listings 2 and 3): u_{t+1} = A(C) u_t on the interior, Dirichlet halo.
// For L = 0.5 ||u_T - target||^2 (or any cotangent lambda_T of u_T):
//   lambda_t = A^T lambda_{t+1},
//   (A^T l)(q) = sum over the terms of every point p that reads q of C(p) l(p):
//     7-point:  C0(q) l(q) + C1(q-x) l(q-x) + C2(q+x) l(q+x) + C3(q-y) l(q-y)
//               + C4(q+y) l(q+y) + C5(q-z) l(q-z) + C6(q+z) l(q+z)
//     25-point: C00(q) l(q) + sum_{d,a} [C_da(q - d e_a) l(q - d e_a) + C_da(q + d e_a) l(q + d e_a)]
//   dL/dC_m(p) = sum_t lambda_{t+1}(p) * (the field value that multiplies C_m(p) at step t),
//   dL/du_0 = lambda_0.
// Zero halos in lambda and in the coefficient arrays make the "p is interior"
// condition of the transpose automatic. Coefficient gradients accumulate in FP64.
#include "adjoint_column.cuh"
#include "internal.h"
#include "pdl.cuh"

namespace stg {

struct AdjGrad {
    double* g[13];
};

// One transposed step over the interior: lam_out = A^T lam_in (lambda_column). A warp covers
// 32 x vectors of V = 16/sizeof(field) points (128-bit loads), warps are stacked along y, and
// each thread walks a chunk of z planes.
template <int KIND, typename TF, typename TC, int BY>
__global__ void __launch_bounds__(32 * BY) adjoint_vec_kernel(Layout L, const TF* __restrict__ lam_in,
                                                              TF* __restrict__ lam_out, CoefPtrs<TC> C, int zchunk) {
    constexpr int V = 16 / sizeof(TF);
    dependent_begin();
    const int i0 = (blockIdx.x * 32 + threadIdx.x) * V;
    const int j = blockIdx.y * BY + threadIdx.y;
    if (i0 >= L.nx || j >= L.ny) return;
    const int k0 = blockIdx.z * zchunk;
    const int k1 = min(L.nz, k0 + zchunk);
    lambda_column<KIND, TF, TC, false>(L, lam_in, lam_out, C, i0, j, k0, k1);
}

// Coefficient gradients of several steps in one pass: for the steps t = t_hi, t_hi - 1,
// ..., t_lo (in that order, the order of the backward walk), gC_m(p) += lam_{t+1}(p) x
// (the field value(s) C_m(p) weighs in step t), one FP64 fma per step on an accumulator
// kept in registers, so each gradient array is read and written once per pass instead of
// once per step. The fma sequence per element is the one the one-step kernel performs, so
// the result is the same bit for bit. lam[g] = lam_{t_hi + 1 - g}, u[g] = u_{t_hi - g}.
constexpr int ADJ_GROUP = 16;  // steps per gradient pass

template <typename TF>
struct AdjSteps {
    const TF* lam[ADJ_GROUP];
    const TF* u[ADJ_GROUP];
};

// FP32 -> FP64 without the FP64 pipe, which also does the hardware conversion and already bounds
// this kernel: N values at once, by integer operations where all of them are normal numbers or, with ZEROS, zeros (the
// magnitude times 2^29 as a 64-bit integer is the FP64 significand and exponent field, short of
// the difference of the two exponent biases), else by the hardware conversion. Exact either way. Zeros
// are every cell next to the halo and every lane past a ragged row's end: left to the hardware they
// took whole warps there (training step, 25-point BF16 203 x 250 x 141 T = 12: 7.1 -> 5.8 ms, 7-point FP32
// 250 x 220 x 180 T = 20: 8.8 -> 7.2 ms). Not for the 25-point stencil on rows of whole vectors: its weights
// are pair sums, none of them zero for a halo alone, and the two operations more per value cost 1 %.
template <int N, bool ZEROS>
struct Widen {
    double d[N];
    __device__ __forceinline__ explicit Widen(const float* x) {
        unsigned a[N], lo = 0x7f800000u, hi = 0u;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            a[i] = __float_as_uint(x[i]) & 0x7fffffffu;
            lo = min(lo, ZEROS ? a[i] - 1u : a[i]);  // (zeros become the largest value)
            hi = max(hi, a[i]);
        }
        if (lo >= (ZEROS ? 0x007fffffu : 0x00800000u) && hi < 0x7f800000u) {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const unsigned long long w = (unsigned long long)a[i] * (1u << 29) + (896ull << 52);
                const unsigned h = !ZEROS || a[i] != 0u ? (unsigned)(w >> 32) : 0u;  // (the low half of a zero is zero)
                d[i] = __hiloint2double((int)(h | (__float_as_uint(x[i]) & 0x80000000u)), (int)(unsigned)w);
            }
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) d[i] = (double)x[i];
        }
    }
    __device__ __forceinline__ explicit Widen(const double* x) {
#pragma unroll
        for (int i = 0; i < N; ++i) d[i] = x[i];
    }
};

// Bound by the FP64 pipe: one fma per coefficient, point and step (14.3 ms at its peak for 13
// arrays, 256^3, 40 steps). With hardware conversions of the weights on the same pipe it took
// 34.0 ms, with Widen 19.4, at three CTAs per SM (168 registers, 24 bytes spilled) 17.6; vectors of
// two points (more warps, but twice the loads) 29.6.
template <int KIND, typename TF, int V, int NT, bool ZEROS>
__global__ void __launch_bounds__(NT, 3) adjoint_grad_kernel(Layout L, AdjSteps<TF> S, int nsteps, AdjGrad G, int zchunk) {
    constexpr int R = KindTraits<KIND>::R;
    constexpr int NC = KindTraits<KIND>::NC;
    constexpr int J = (R + V - 1) / V;
    constexpr int XL = (2 * J + 1) * V;
    using A = Ar<TF>;
    // threads over the plane's vectors in order, so that only its last warp has idle lanes
    const unsigned nv = (unsigned)(L.nx + V - 1) / V;
    const unsigned long long q = (unsigned long long)blockIdx.x * NT + threadIdx.x;
    if (q >= (unsigned long long)nv * (unsigned)L.ny) return;
    const int j = (int)(q / nv), i0 = (int)(q - (unsigned long long)j * nv) * V;
    const int k0 = blockIdx.y * zchunk;
    const int k1 = min(L.nz, k0 + zchunk);
    const size_t sy = (size_t)L.px, sz = L.plane();
    const bool full = i0 + V <= L.nx;
    for (int k = k0; k < k1; ++k) {
        const size_t p = L.at(i0, j, k);
        // all accumulators in registers: every gradient array read once and written once
        double gv[NC][V];
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            const double* gp = G.g[m] + p;
            if (full) {
#pragma unroll
                for (int h = 0; h < V; h += 2) {
                    const double2 g = *reinterpret_cast<const double2*>(gp + h);
                    gv[m][h] = g.x;
                    gv[m][h + 1] = g.y;
                }
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e) gv[m][e] = i0 + e < L.nx ? gp[e] : 0.0;
            }
        }
        // steps outermost: the neighbours of each state are loaded once per step
        for (int g = 0; g < nsteps; ++g) {
            const TF* u = S.u[g];
            const Vec<TF, V> lv = ldv_ro<TF, V>(S.lam[g] + p);
            TF ux[XL];
#pragma unroll
            for (int q = -J; q <= J; ++q) {
                const Vec<TF, V> wu = ldv_ro<TF, V>(u + p + (ptrdiff_t)q * V);
#pragma unroll
                for (int e = 0; e < V; ++e) ux[(q + J) * V + e] = wu.v[e];
            }
            const Widen<V, ZEROS> lam(lv.v);
            // weight of array m: 7-point C0 u(p), C(2a+1) u(p + e_a), C(2a+2) u(p - e_a);
            // 25-point C00 u(p), C(3(d-1)+a+1) (u(p + d e_a) + u(p - d e_a)), the pair sum
            // in the field precision as the forward step forms it
            {
                const Widen<V, ZEROS> w(ux + J * V);
#pragma unroll
                for (int e = 0; e < V; ++e) gv[0][e] = __fma_rn(lam.d[e], w.d[e], gv[0][e]);
            }
#pragma unroll
            for (int d = 1; d <= R; ++d) {
                TF up[3][V], um[3][V];
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    if (a == 0) {
#pragma unroll
                        for (int e = 0; e < V; ++e) {
                            up[a][e] = ux[J * V + e + d];
                            um[a][e] = ux[J * V + e - d];
                        }
                    } else {
                        const size_t o = (size_t)d * (a == 1 ? sy : sz);
                        const Vec<TF, V> vp = ldv_ro<TF, V>(u + p + o);
                        const Vec<TF, V> vm = ldv_ro<TF, V>(u + p - o);
#pragma unroll
                        for (int e = 0; e < V; ++e) {
                            up[a][e] = vp.v[e];
                            um[a][e] = vm.v[e];
                        }
                    }
                }
                if constexpr (KIND == K7V) {
                    // C(2a+1) weighs u(p + e_a), C(2a+2) weighs u(p - e_a)
                    const Widen<3 * V, ZEROS> wp(&up[0][0]), wm(&um[0][0]);
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int e = 0; e < V; ++e) {
                            gv[1 + 2 * a][e] = __fma_rn(lam.d[e], wp.d[a * V + e], gv[1 + 2 * a][e]);
                            gv[2 + 2 * a][e] = __fma_rn(lam.d[e], wm.d[a * V + e], gv[2 + 2 * a][e]);
                        }
                } else {
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int e = 0; e < V; ++e) up[a][e] = A::add(up[a][e], um[a][e]);
                    const Widen<3 * V, ZEROS> w(&up[0][0]);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const int m = 3 * (d - 1) + a + 1;
#pragma unroll
                        for (int e = 0; e < V; ++e) gv[m][e] = __fma_rn(lam.d[e], w.d[a * V + e], gv[m][e]);
                    }
                }
            }
        }
#pragma unroll
        for (int m = 0; m < NC; ++m) {
            double* gp = G.g[m] + p;
            if (full) {
#pragma unroll
                for (int h = 0; h < V; h += 2) *reinterpret_cast<double2*>(gp + h) = make_double2(gv[m][h], gv[m][h + 1]);
            } else {
#pragma unroll
                for (int e = 0; e < V; ++e)
                    if (i0 + e < L.nx) gp[e] = gv[m][e];
            }
        }
    }
}

// Planes a thread walks in the kernels of this file, which keep nothing from one plane to the next:
// as many as leave about 16 CTAs of 128 threads per SM (152), at most 16 (one plane after another
// costs its full latency: 96 x 70 x 83, 16 planes a thread, took 188 us per gradient pass, 7-point,
// and 36 us per transposed step). gridDim.z stays below its limit at any nz.
static int adj_chunk(long long xy, int nz) {
    long long c = xy * nz / (152 * 16);
    c = c < 1 ? 1 : (c > 16 ? 16 : c);
    const long long least = ((long long)nz + 65534) / 65535;
    return (int)(c < least ? least : c);
}

template <int KIND, typename TF>
static cudaError_t adj_grads(const Layout& L, const void* const* lam, const void* const* u, int n,
                             double* const* gC, cudaStream_t s) {
    constexpr int V = 16 / sizeof(TF), NT = 128;
    dim3 grid((unsigned)(((long long)((L.nx + V - 1) / V) * L.ny + NT - 1) / NT), 1);
    const int zchunk = adj_chunk(grid.x, L.nz);
    grid.y = (unsigned)((L.nz + zchunk - 1) / zchunk);
    AdjGrad G{};
    for (int m = 0; m < KindTraits<KIND>::NC; ++m) G.g[m] = gC[m];
    for (int g0 = 0; g0 < n; g0 += ADJ_GROUP) {
        AdjSteps<TF> S{};
        const int ng = n - g0 < ADJ_GROUP ? n - g0 : ADJ_GROUP;
        for (int g = 0; g < ng; ++g) {
            S.lam[g] = static_cast<const TF*>(lam[g0 + g]);
            S.u[g] = static_cast<const TF*>(u[g0 + g]);
        }
        if (KIND == K25V && L.nx % V == 0) adjoint_grad_kernel<KIND, TF, V, NT, KIND != K25V><<<grid, NT, 0, s>>>(L, S, ng, G, zchunk);
        else adjoint_grad_kernel<KIND, TF, V, NT, true><<<grid, NT, 0, s>>>(L, S, ng, G, zchunk);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t adjoint_grads(const SweepArgs& a, const void* const* lam, const void* const* u, int n, double* const* gC,
                          cudaStream_t s) {
    if (a.L.nx == 0 || a.L.ny == 0 || a.L.nz == 0 || n <= 0) return cudaSuccess;
    if (a.kind == K7V) {
        if (a.fdt == DT_F32) return adj_grads<K7V, float>(a.L, lam, u, n, gC, s);
        if (a.fdt == DT_F64) return adj_grads<K7V, double>(a.L, lam, u, n, gC, s);
    } else if (a.kind == K25V) {
        if (a.fdt == DT_F32) return adj_grads<K25V, float>(a.L, lam, u, n, gC, s);
        if (a.fdt == DT_F64) return adj_grads<K25V, double>(a.L, lam, u, n, gC, s);
    }
    return cudaErrorInvalidValue;
}

// dst(interior) = src(interior); every other cell of dst = 0.
template <typename TF>
__global__ void copy_interior_zero_halo_kernel(Layout L, const TF* __restrict__ src, TF* __restrict__ dst) {
    const size_t n = L.count();
    for (size_t q = (size_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (size_t)gridDim.x * blockDim.x) {
        const size_t row = q / (size_t)L.px;
        const int x = (int)(q - row * (size_t)L.px) - L.xo;
        const int y = (int)(row % (size_t)L.py) - L.R;
        const int z = (int)(row / (size_t)L.py) - L.R;
        const bool in = x >= 0 && x < L.nx && y >= 0 && y < L.ny && z >= 0 && z < L.nz;
        dst[q] = in ? src[q] : TF(0);
    }
}

template <int KIND, typename TF, typename TC>
static cudaError_t adj_step(const SweepArgs& a, const void* lam_in, void* lam_out, cudaStream_t s) {
    const Layout& L = a.L;
    CoefPtrs<TC> C{};
    for (int m = 0; m < KindTraits<KIND>::NC; ++m) C.c[m] = static_cast<const TC*>(a.coef[m]);
    constexpr int BY = 4;
    constexpr int V = 16 / sizeof(TF);
    dim3 block(32, BY, 1);
    dim3 grid((unsigned)((L.nx + 32 * V - 1) / (32 * V)), (unsigned)((L.ny + BY - 1) / BY), 1);
    const int zchunk = adj_chunk((long long)grid.x * grid.y, L.nz);
    grid.z = (unsigned)((L.nz + zchunk - 1) / zchunk);
    return launch_dependent(true, adjoint_vec_kernel<KIND, TF, TC, BY>, grid, block, 0, s, L, static_cast<const TF*>(lam_in),
                            static_cast<TF*>(lam_out), C, zchunk);
}

cudaError_t adjoint_step(const SweepArgs& a, const void* lam_in, void* lam_out, cudaStream_t s) {
    if (a.L.nx == 0 || a.L.ny == 0 || a.L.nz == 0) return cudaSuccess;
    if (a.kind == K7V) {
        if (a.fdt == DT_F32 && a.cdt == DT_F32) return adj_step<K7V, float, float>(a, lam_in, lam_out, s);
        if (a.fdt == DT_F32 && a.cdt == DT_BF16) return adj_step<K7V, float, __nv_bfloat16>(a, lam_in, lam_out, s);
        if (a.fdt == DT_F64) return adj_step<K7V, double, double>(a, lam_in, lam_out, s);
    } else if (a.kind == K25V) {
        if (a.fdt == DT_F32 && a.cdt == DT_F32) return adj_step<K25V, float, float>(a, lam_in, lam_out, s);
        if (a.fdt == DT_F32 && a.cdt == DT_BF16) return adj_step<K25V, float, __nv_bfloat16>(a, lam_in, lam_out, s);
        if (a.fdt == DT_F64) return adj_step<K25V, double, double>(a, lam_in, lam_out, s);
    }
    return cudaErrorInvalidValue;
}

cudaError_t copy_interior_zero_halo(const Layout& L, int dt, const void* src, void* dst, cudaStream_t s) {
    unsigned blocks = (unsigned)((L.count() + 255) / 256);
    if (blocks > 152u * 32u) blocks = 152u * 32u;
    if (dt == DT_F32)
        copy_interior_zero_halo_kernel<float><<<blocks, 256, 0, s>>>(L, (const float*)src, (float*)dst);
    else if (dt == DT_F64)
        copy_interior_zero_halo_kernel<double><<<blocks, 256, 0, s>>>(L, (const double*)src, (double*)dst);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

}  // namespace stg
