// The normal operator's G^H G as a stencil on the half-plane grid.
//
// G^H G couples the cells of one visibility's J x J footprint, so it is a
// real symmetric band matrix: with w_m the footprint weights of visibility m
// (folded into the half plane, see HalfPlane),
//   out[k] = sum_d T[k][d] X[k + d],  T[k][d] = sum_m w_m[k] w_m[k + d],
// |dx|, |dy| < J, and T[k + d][-d] = T[k][d], so one half of the offsets is
// kept: dy = 0 with dx >= 0, and 0 < dy < J with every dx, NC = J + (J-1)(2J-1)
// of them. T depends on the coverage alone and is built with the plan; an
// application then reads NC coefficients per grid cell however many
// visibilities there are, instead of walking the visibilities' runs.
//
// Layout: T[y][d][x], x < W (the row stride of the half plane): a warp reads
// the planes of a row segment as coalesced rows.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "internal.h"
#include "launch.h"

namespace purify {

PURIFY_HD constexpr int stencil_planes(int J) { return J + (J - 1) * (2 * J - 1); }
// plane of offset (dy, dx)
PURIFY_HD constexpr int stencil_plane(int J, int dy, int dx) {
    return dy == 0 ? dx : J + (dy - 1) * (2 * J - 1) + dx + J - 1;
}

// ------------------------------------------------------------------ build
// T from the half-plane runs, a warp per run. The products of a visibility's
// weights factor over the axes: lane i holds wx[a] wx[a'] of the i-th pair
// a <= a' (two pairs for J = 8), the y pairs b <= b' come by shuffle, and
// acc[j] sums the product of x pair i and y pair j over the run (at most 48
// visibilities). The run's sums are then added in double: the pair gives
// T[(b, a)][(b' - b, a' - a)] and, for b < b' and a < a', also
// T[(b, a')][(b' - b, a - a')].
template <typename T, int J>
__global__ void __launch_bounds__(128)
k_stencil_build(const int2* __restrict__ set_info, const int2* __restrict__ run_cl, const T* __restrict__ rec,
                int nruns, int width, typename KbOf<T>::type kp, int W, int Ky, double* __restrict__ out) {
    constexpr int NP = J * (J + 1) / 2, NI = (NP + 31) / 32, NC = stencil_planes(J);
    constexpr int DEG = sizeof(T) == 4 ? kb_poly_deg(J) : kb_poly_deg_d(J);
    const int lane = threadIdx.x & 31, axis = lane >> 4, tap = min(lane & 15, J - 1);
    // pair a <= a' of index i (row-major over the upper triangle)
    int pa[NI], pb[NI];
#pragma unroll
    for (int s = 0; s < NI; ++s) {
        int i = min(lane + 32 * s, NP - 1), a = 0;
        while (i >= J - a) { i -= J - a; ++a; }
        pa[s] = a;
        pb[s] = a + i;
    }
    T cf[DEG + 1];
#pragma unroll
    for (int i = 0; i <= DEG; ++i) cf[i] = kp.coef[tap][i];
    const int nw = gridDim.x * (blockDim.x >> 5);
    for (int q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < nruns; q += nw) {
        const int2 cl = run_cl[q];
        if (cl.y <= 0) continue;
        // this lane's axis of the run's records (see LaneWork), a row apart
        const T* z = rec + (size_t)set_info[q / width].x * 2 * width +
                     (width == 32 ? 2 * (q % 32) + axis : q % 16 + 16 * axis);
        T acc[NI][NP];
#pragma unroll
        for (int s = 0; s < NI; ++s)
#pragma unroll
            for (int j = 0; j < NP; ++j) acc[s][j] = T(0);
        for (int k = 0; k < cl.y; ++k) {
            const T zk = z[(size_t)k * 2 * width];
            // lane (axis, tap): this tap's weight
            T w = cf[DEG];
#pragma unroll
            for (int i = DEG - 1; i >= 0; --i) w = fma(w, zk, cf[i]);
            if constexpr (sizeof(T) == 8) {
                if (!kp.poly) w = kb_tap_exact(J, tap, kp.beta, kp.inv_i0beta, zk);
            }
            T px[NI], py[NI];
#pragma unroll
            for (int s = 0; s < NI; ++s) {
                px[s] = __shfl_sync(0xffffffffu, w, pa[s]) * __shfl_sync(0xffffffffu, w, pb[s]);
                py[s] = __shfl_sync(0xffffffffu, w, 16 + pa[s]) * __shfl_sync(0xffffffffu, w, 16 + pb[s]);
            }
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const T wy = __shfl_sync(0xffffffffu, py[j / 32], j % 32);
#pragma unroll
                for (int s = 0; s < NI; ++s) acc[s][j] = fma(px[s], wy, acc[s][j]);
            }
        }
        const int cx = cl.x & 0xFFFF, cy = (int)((unsigned)cl.x >> 16);
#pragma unroll
        for (int s = 0; s < NI; ++s) {
            if (lane + 32 * s >= NP) continue;
            const int a = pa[s], a2 = pb[s];
            int j = 0;
#pragma unroll
            for (int b = 0; b < J; ++b) {
                double* row = out + (size_t)((cy + b) & (Ky - 1)) * NC * W + cx;
#pragma unroll
                for (int b2 = b; b2 < J; ++b2, ++j) {
                    const double v = (double)acc[s][j];
                    atomicAdd(row + (size_t)stencil_plane(J, b2 - b, a2 - a) * W + a, v);
                    if (b2 > b && a2 > a) atomicAdd(row + (size_t)stencil_plane(J, b2 - b, a - a2) * W + a2, v);
                }
            }
        }
    }
}

__global__ void k_to_float(const double* __restrict__ in, float* __restrict__ out, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

// ------------------------------------------------------------------ apply
// out[k] = sum over the kept offsets d of T[k][d] X[k + d], and of
// T[k - d][d] X[k - d]: each coefficient is read at its own cell and again,
// shifted, by the cell it couples to (the second reading comes from L1 or
// L2: the rows of a block and of its neighbours run at the same time). A
// thread owns V neighbouring cells of a row (one 16-byte access of X), a warp
// 32 V cells, a block STENCIL_ROWS rows of them. Cells outside the stored
// columns have zero coefficients (the row stride leaves at least eight unused
// columns, which also follow the previous plane's), so the window loads only
// clamp their address. Blocks without any coefficient (`used`) store zeros.
// Bound by the coefficients: NC sizeof(T) bytes a cell from HBM, twice that
// from L2 (1024 x 1024, J = 6: 0.52 GB). A form that marches down the rows and
// reads each coefficient once (row accumulators in registers, a shift chain
// along x) took 130 us there against 120, and 45 against 12 at 256 x 256: too
// few warps in flight. By the runs (lane pairs): 226 and 21 us on the half
// plane, 278 and 26 on the whole one.
static constexpr int STENCIL_ROWS = 8;
template <typename T> struct StencilVec { static constexpr int V = 16 / sizeof(typename cplx_of<T>::type); };

__device__ __forceinline__ void s_load(const float* p, float (&v)[2]) {
    const float2 q = __ldg(reinterpret_cast<const float2*>(p));
    v[0] = q.x;
    v[1] = q.y;
}
__device__ __forceinline__ void s_load(const double* p, double (&v)[1]) { v[0] = __ldg(p); }
// two cells (float) or one (double) per 16-byte access
__device__ __forceinline__ void s_cells(const float2* p, float2* v) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = make_float2(q.x, q.y);
    v[1] = make_float2(q.z, q.w);
}
__device__ __forceinline__ void s_cells(const double2* p, double2* v) { v[0] = *p; }
__device__ __forceinline__ void s_store(float2* p, const float2 (&v)[2]) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
}
__device__ __forceinline__ void s_store(double2* p, const double2 (&v)[1]) { *p = v[0]; }
__device__ __forceinline__ float2 s_fma(float w, float2 x, float2 a) { return __ffma2_rn(make_float2(w, w), x, a); }
__device__ __forceinline__ double2 s_fma(double w, double2 x, double2 a) {
    return make_double2(fma(w, x.x, a.x), fma(w, x.y, a.y));
}

template <typename T, int J>
__global__ void __launch_bounds__(32 * STENCIL_ROWS, 2)
k_stencil(const T* __restrict__ coef, const typename cplx_of<T>::type* __restrict__ X,
          typename cplx_of<T>::type* __restrict__ out, const unsigned char* __restrict__ used, int W, int Ky,
          const int* __restrict__ skip) {
    using C = typename cplx_of<T>::type;
    constexpr int V = StencilVec<T>::V, NC = stencil_planes(J), E = J - 1;
    constexpr int EL = (E + V - 1) / V * V, XN = V + 2 * EL;   // window margin and width in whole accesses
    pdl_wait();
    if (skip && *skip) return;
    const int x = (blockIdx.x * 32 + (threadIdx.x & 31)) * V, y = blockIdx.y * STENCIL_ROWS + (threadIdx.x >> 5);
    if (x < W) {
        C acc[V];
#pragma unroll
        for (int v = 0; v < V; ++v) acc[v] = cmake<C>(T(0), T(0));
        if (used[blockIdx.y * gridDim.x + blockIdx.x]) {
            int xo[XN / V];
#pragma unroll
            for (int i = 0; i < XN; i += V) xo[i / V] = min(max(x - EL + i, 0), W - V);
            const T* own = coef + (size_t)y * NC * W + x;
            C xw[XN];
            auto window = [&](int yy) {
                const C* xr = X + (size_t)yy * W;
#pragma unroll
                for (int i = 0; i < XN; i += V) s_cells(xr + xo[i / V], &xw[i]);
            };
            // T[k][d] X[k + d]: plane pointer p at this cell, window of row y + dy
            auto add_own = [&](const T* p, int dx) {
                T t[V];
                s_load(p, t);
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] = s_fma(t[v], xw[EL + v + dx], acc[v]);
            };
            // T[k - d][d] X[k - d]: plane pointer p at column x of row y - dy
            auto add_shifted = [&](const T* p, int dx) {
                T t[V];
                if (dx % V == 0) {
                    s_load(p - dx, t);
                } else {
#pragma unroll
                    for (int v = 0; v < V; ++v) t[v] = __ldg(p - dx + v);
                }
#pragma unroll
                for (int v = 0; v < V; ++v) acc[v] = s_fma(t[v], xw[EL + v - dx], acc[v]);
            };
            window(y);
            add_own(own, 0);
#pragma unroll
            for (int dx = 1; dx <= E; ++dx) {
                add_own(own + dx * W, dx);
                add_shifted(own + dx * W, dx);
            }
            own += J * W;                       // plane (1, -E)
            int plane = J;
#pragma unroll 1
            for (int dy = 1; dy <= E; ++dy, own += (2 * J - 1) * W, plane += 2 * J - 1) {
                window((y + dy) & (Ky - 1));
#pragma unroll
                for (int dx = -E; dx <= E; ++dx) add_own(own + (dx + E) * W, dx);
                const int yy = (y - dy) & (Ky - 1);
                const T* nb = coef + ((size_t)yy * NC + plane) * W + x;
                window(yy);
#pragma unroll
                for (int dx = -E; dx <= E; ++dx) add_shifted(nb + (dx + E) * W, dx);
            }
        }
        s_store(out + (size_t)y * W + x, acc);
    }
    pdl_trigger();
}

// ------------------------------------------------------------- launchers
static dim3 stencil_grid(const purify_plan* p) {
    const int cols = 32 * (p->dtype == PURIFY_F32 ? StencilVec<float>::V : StencilVec<double>::V);
    return dim3((p->half.W + cols - 1) / cols, p->Ky / STENCIL_ROWS);
}

// Blocks that read a non-zero coefficient, from the runs' first-tap cells
// (row * W + column): coefficients lie in the footprint's cells, and a block
// reads those of its own cells and of the J - 1 rows above and columns beside.
static std::vector<unsigned char> stencil_used(const purify_plan* p, const std::vector<int>& cells) {
    const dim3 g = stencil_grid(p);
    const int E = p->J - 1, cols = 32 * (p->dtype == PURIFY_F32 ? StencilVec<float>::V : StencilVec<double>::V);
    std::vector<unsigned char> used((size_t)g.x * g.y, 0);
    for (int c : cells) {
        const int cy = c / p->half.W, cx = c % p->half.W;
        const int xa = std::max(0, cx - E) / cols, xb = std::min((cx + 2 * E) / cols, (int)g.x - 1);
        for (int dy = 0; dy <= 2 * E + STENCIL_ROWS; dy += STENCIL_ROWS) {
            const int yb = ((cy + std::min(dy, 2 * E)) & (p->Ky - 1)) / STENCIL_ROWS;
            for (int xbk = xa; xbk <= xb; ++xbk) used[(size_t)yb * g.x + xbk] = 1;
        }
    }
    return used;
}

template <typename T, int J> static void stencil_build_tj(purify_plan* p) {
    Stencil& s = p->stencil;
    const LaneWork& lw = p->half_lanes;
    const int64_t n = (int64_t)p->Ky * stencil_planes(J) * p->half.W;
    // the shifted readings of the last plane run up to J - 1 elements past it
    s.coef.alloc(sizeof(T) * (n + 16));
    PURIFY_CUDA(cudaMemsetAsync(s.coef.as<T>() + n, 0, sizeof(T) * 16, p->stream));
    DevBuf sum;
    double* acc = s.coef.as<double>();
    if (sizeof(T) == 4) {
        sum.alloc(sizeof(double) * n);
        acc = sum.as<double>();
    }
    PURIFY_CUDA(cudaMemsetAsync(acc, 0, sizeof(double) * n, p->stream));
    k_stencil_build<T, J><<<152 * 8, 128, 0, p->stream>>>(lw.set_info.as<int2>(), lw.run_cl.as<int2>(), lw.rec.as<T>(),
                                                          lw.nsets * lw.width, lw.width, kb_table<T>(p), p->half.W, p->Ky, acc);
    PURIFY_CUDA(cudaGetLastError());
    if (sizeof(T) == 4) {
        k_to_float<<<152 * 8, 256, 0, p->stream>>>(acc, s.coef.as<float>(), n);
        PURIFY_CUDA(cudaGetLastError());
    }
    PURIFY_CUDA(cudaStreamSynchronize(p->stream));   // `sum` is released here
    add_launches(sizeof(T) == 4 ? 2 : 1);
}
template <int J> static void stencil_build_j(purify_plan* p) {
    if (p->dtype == PURIFY_F32) stencil_build_tj<float, J>(p); else stencil_build_tj<double, J>(p);
}

int64_t stencil_bytes(const purify_plan* p) {
    return (int64_t)p->Ky * stencil_planes(p->J) * p->half.W * (p->dtype == PURIFY_F32 ? 4 : 8);
}

bool build_stencil(purify_plan* p, const std::vector<int>& cells) {
    const std::vector<unsigned char> used = stencil_used(p, cells);
    try {
        p->stencil.used.alloc(used.size());
        PURIFY_CUDA(cudaMemcpy(p->stencil.used.p, used.data(), used.size(), cudaMemcpyHostToDevice));
        settle_uploads();   // the build reads the run tables on the plan's stream
        PURIFY_J_DISPATCH(p->J, stencil_build_j, p);
    } catch (const Error& e) {
        // the memory that was free when it was chosen may be gone by now
        if (e.status != PURIFY_ENOMEM) throw;
        p->stencil.coef.release();
        p->stencil.used.release();
        return false;
    }
    p->stencil.on = true;
    return true;
}

template <typename T, int J> static void stencil_tj(purify_plan* p, const int* skip) {
    using C = typename cplx_of<T>::type;
    const Stencil& s = p->stencil;
    Launch L(p, "normal_gg");
    launch_dependent(k_stencil<T, J>, stencil_grid(p), 32 * STENCIL_ROWS, 0, p->stream, (const T*)s.coef.as<T>(),
                     (const C*)p->grid.as<C>(), p->gacc.as<C>(), (const unsigned char*)s.used.as<unsigned char>(),
                     p->half.W, p->Ky, skip);
    L.done();
}
template <int J> static void stencil_j(purify_plan* p, const int* skip) {
    if (p->dtype == PURIFY_F32) stencil_tj<float, J>(p, skip); else stencil_tj<double, J>(p, skip);
}
void launch_stencil(purify_plan* p, const int* skip) { PURIFY_J_DISPATCH(p->J, stencil_j, p, skip); }

}  // namespace purify
