// SARA dictionary: Psi^dagger (analysis) and Psi (synthesis).
//
// Sec. 1 of the paper builds Psi = [Psi_1, ..., Psi_q] from q coherent
// bases. The plan uses the Dirac basis plus Daubechies db1..db8 (selected by
// the basis mask), each an orthonormal periodic 2-D Mallat transform with L
// levels, scaled by 1/sqrt(q) so that Psi Psi^dagger = I.
//
// One analysis level maps an h x w low-pass band to four h/2 x w/2 sub-bands
//   a[k] = sum_n h[n] x[(2k + n) mod len],  d[k] = sum_n g[n] x[(2k + n) mod len]
// applied along rows, then along columns. A block owns a TH x TW tile of every
// sub-band of one basis: its threads filter the rows of the input tile (TH plus
// halo) straight from global memory, KX outputs of both filters from one
// register window, into shared memory, then the columns, RK outputs of the four
// sub-bands from two windows. Synthesis is the transpose: out[2i + par] = sum_j
// h[2j + par] a[i - j] + g[2j + par] d[i - j], rows first (from global
// memory), then columns; the finest level sums all bases in the block's
// registers, so the image is written once. All wavelet bases of a level run in
// one launch (blockIdx.z), filters with their compile-time lengths. The levels
// whose bands fit shared memory run in one launch, a block per basis (*_tail).
// The filters are a few multiply-adds per byte, so the register windows carry
// the weight: with every tap read from shared memory these kernels were bound
// by it (9 bases: analysis of 1024 x 1024 over 5 levels 58 us, now 32; synthesis
// of 512 x 1024 over 4 levels 72 us, now 31; the coefficients' 42 and 21 MB
// take 6 and 3 us).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "host_tables.h"
#include "launch.h"

namespace purify {

// Daubechies filters are the same for every plan: one constant-memory bank
// per precision, written once per device (init_filter_banks).
__constant__ FilterBank<float> c_bank_f;
__constant__ FilterBank<double> c_bank_d;
template <typename T> __device__ __forceinline__ const FilterBank<T>& fbank();
template <> __device__ __forceinline__ const FilterBank<float>& fbank<float>() { return c_bank_f; }
template <> __device__ __forceinline__ const FilterBank<double>& fbank<double>() { return c_bank_d; }

// Tile geometry. FP32: sub-band tiles of 32 columns, 256 threads. FP64 is
// bound by its arithmetic pipe (2 FMA per clock and SM): small tiles spread a
// level over all SMs. Band sizes are powers of two, so wrapping is a mask.
template <typename T> struct WaveTile;
template <> struct WaveTile<float> {
    static constexpr int TW = 32, KX = 4, THREADS = 256;
    // largest band area of the tails: one SM per basis; 128 x 128 (two levels
    // fewer launches) took 29 us where two launches of tiles take 10
    static constexpr int TAIL = 1024;
    static constexpr int SYN_RK = 4;
};
template <> struct WaveTile<double> {
    static constexpr int TW = 8, KX = 2, THREADS = 64, TAIL = 64;
    static constexpr int SYN_RK = 2;
};
// threads of a synthesis tile of TH sub-band rows: one per output column and
// SYN_RK sub-band rows
template <typename T, int TH> constexpr int syn_threads() { return 2 * WaveTile<T>::TW * TH / WaveTile<T>::SYN_RK; }
static constexpr int TAIL_THREADS = 512;

// The filter taps of basis pb in registers (unused entries are zero).
template <typename T, int L> struct Taps {
    T h[L], g[L];
    __device__ __forceinline__ void load(int pb) {
        const FilterBank<T>& fb = fbank<T>();
#pragma unroll
        for (int n = 0; n < L; ++n) { h[n] = fb.h[pb][n]; g[n] = fb.g[pb][n]; }
    }
};

// Runs STMT with the compile-time constant L equal to the filter length LEN
// (2, 4, ..., 16).
#define PURIFY_WITH_LENGTH(LEN, STMT)                                  \
    switch (LEN) {                                                     \
        case 2: { constexpr int L = 2; STMT; } break;                  \
        case 4: { constexpr int L = 4; STMT; } break;                  \
        case 6: { constexpr int L = 6; STMT; } break;                  \
        case 8: { constexpr int L = 8; STMT; } break;                  \
        case 10: { constexpr int L = 10; STMT; } break;                \
        case 12: { constexpr int L = 12; STMT; } break;                \
        case 14: { constexpr int L = 14; STMT; } break;                \
        default: { constexpr int L = 16; STMT; } break;                \
    }

// ------------------------------------------------------------- analysis
// Row filters: low- and high-pass outputs k0 .. k0 + KX - 1 of one input row
// (periodic, w columns) from a register window of 2 KX + L - 2 inputs; VEC:
// the row is 16-byte aligned, w >= 4 (the window then comes in 16-byte loads,
// which wrap as a whole).
template <typename T, int L, int KX, bool VEC>
__device__ __forceinline__ void row_filter(const Taps<T, L>& f, const T* __restrict__ row, int w, int k0, T (&a)[KX],
                                           T (&d)[KX]) {
    constexpr int V = 16 / sizeof(T), N = (2 * KX + L - 2 + V - 1) / V * V;
    alignas(16) T win[N];
    if constexpr (VEC) {
#pragma unroll
        for (int i = 0; i < N; i += V) {
            const uint4 q = *reinterpret_cast<const uint4*>(row + ((2 * k0 + i) & (w - 1)));
            *reinterpret_cast<uint4*>(win + i) = q;
        }
    } else {
#pragma unroll
        for (int i = 0; i < 2 * KX + L - 2; ++i) win[i] = row[(2 * k0 + i) & (w - 1)];
    }
#pragma unroll
    for (int j = 0; j < KX; ++j) {
        a[j] = d[j] = T(0);
#pragma unroll
        for (int n = 0; n < L; ++n) {
            a[j] += f.h[n] * win[2 * j + n];
            d[j] += f.g[n] * win[2 * j + n];
        }
    }
}

// Column filters: sub-band rows 0 .. RK - 1 of one column from rows 0 .. 2 RK +
// L - 3 (masked by rm) of the row-filtered columns ta, td (row stride ld).
template <typename T, int L, int RK>
__device__ __forceinline__ void col_filter(const Taps<T, L>& f, const T* ta, const T* td, int ld, int r0, int rm,
                                           T (&ll)[RK], T (&lh)[RK], T (&hl)[RK], T (&hh)[RK]) {
#pragma unroll
    for (int j = 0; j < RK; ++j) ll[j] = lh[j] = hl[j] = hh[j] = T(0);
#pragma unroll
    for (int i = 0; i < 2 * RK + L - 2; ++i) {
        const T av = ta[((r0 + i) & rm) * ld], dv = td[((r0 + i) & rm) * ld];
#pragma unroll
        for (int j = 0; j < RK; ++j) {
            const int n = i - 2 * j;
            if (n >= 0 && n < L) {
                ll[j] += f.h[n] * av;
                lh[j] += f.g[n] * av;
                hl[j] += f.h[n] * dv;
                hh[j] += f.g[n] * dv;
            }
        }
    }
}

// One analysis level of basis pb on the TH x TW sub-band tile at (ky0, kx0).
template <typename T, int L, int TH>
__device__ __forceinline__ void dwt_tile(const T* __restrict__ in, int src_ld, bool vec, T* __restrict__ out, int nx,
                                         T* __restrict__ llo, int h, int w, int ky0, int kx0, int pb, T inv_sqrt_q,
                                         T* smem) {
    using W = WaveTile<T>;
    constexpr int TW = W::TW, KX = W::KX, RK = TH * TW / W::THREADS, RG = TW / KX;
    Taps<T, L> f;
    f.load(pb);
    const int hs = h >> 1, wsub = w >> 1;
    const int th = min(TH, hs - ky0), tw = min(TW, wsub - kx0);
    const int rows = 2 * th + L - 2;
    T* ta = smem;                          // [2 TH + L - 2][TW] row low-pass
    T* td = ta + (2 * TH + L - 2) * TW;    // row high-pass
    for (int t = threadIdx.x; t < rows * RG; t += W::THREADS) {
        const int r = t / RG, k = (t - r * RG) * KX;
        if (k >= tw) continue;
        const T* row = in + (size_t)((2 * ky0 + r) & (h - 1)) * src_ld;
        alignas(16) T a[KX], d[KX];
        if (vec) row_filter<T, L, KX, true>(f, row, w, kx0 + k, a, d);
        else row_filter<T, L, KX, false>(f, row, w, kx0 + k, a, d);
        // KX outputs are 16 bytes; outputs past tw are not read
        *reinterpret_cast<uint4*>(ta + r * TW + k) = *reinterpret_cast<const uint4*>(a);
        *reinterpret_cast<uint4*>(td + r * TW + k) = *reinterpret_cast<const uint4*>(d);
    }
    __syncthreads();
    const int kx = threadIdx.x % TW, ky = threadIdx.x / TW * RK;
    if (kx < tw && ky < th) {
        T ll[RK], lh[RK], hl[RK], hh[RK];
        col_filter<T, L, RK>(f, ta + kx, td + kx, TW, 2 * ky, ~0, ll, lh, hl, hh);
        const int gx = kx0 + kx;
#pragma unroll
        for (int j = 0; j < RK; ++j) {
            const int gy = ky0 + ky + j;
            if (ky + j >= th) break;
            if (llo) llo[(size_t)gy * wsub + gx] = ll[j];
            else out[(size_t)gy * nx + gx] = ll[j] * inv_sqrt_q;
            out[(size_t)gy * nx + wsub + gx] = hl[j] * inv_sqrt_q;
            out[(size_t)(hs + gy) * nx + gx] = lh[j] * inv_sqrt_q;
            out[(size_t)(hs + gy) * nx + wsub + gx] = hh[j] * inv_sqrt_q;
        }
    }
}

// One analysis level for every wavelet basis (blockIdx.z < nw) and, at the
// first level, the Dirac plane (blockIdx.z == nw, the tile's 2 TH x 2 TW image
// pixels).
template <typename T, int TH>
__global__ void __launch_bounds__(WaveTile<T>::THREADS)
k_dwt_level(const T* __restrict__ src, int src_basis_stride, int src_ld, int vec, T* __restrict__ coef,
            const int* __restrict__ planes, int N, int nx, T* __restrict__ ll_out, int ll_basis_stride, int h, int w,
            const int* __restrict__ pids, int nw, int dirac_plane, T inv_sqrt_q) {
    constexpr int TW = WaveTile<T>::TW;
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int z = blockIdx.z;
    if (z == nw) {
        const int r0 = blockIdx.y * 2 * TH, c0 = blockIdx.x * 2 * TW;
        for (int t = threadIdx.x; t < 4 * TH * TW; t += blockDim.x) {
            int r = r0 + t / (2 * TW), c = c0 + t % (2 * TW);
            if (r < h && c < w) coef[(size_t)dirac_plane * N + (size_t)r * nx + c] = src[(size_t)r * src_ld + c] * inv_sqrt_q;
        }
        return;
    }
    const int pb = pids[z];              // db index 1..8
    const T* in = src + (size_t)z * src_basis_stride;
    T* out = coef + (size_t)planes[z] * N;
    T* llo = ll_out ? ll_out + (size_t)z * ll_basis_stride : nullptr;
    PURIFY_WITH_LENGTH(fbank<T>().len[pb],
                       (dwt_tile<T, L, TH>(in, src_ld, vec != 0, out, nx, llo, h, w, blockIdx.y * TH, blockIdx.x * TW, pb,
                                           inv_sqrt_q, reinterpret_cast<T*>(smem_raw))));
    pdl_trigger();
}
template <typename T> static size_t dwt_smem_bytes(int maxL, int TH) {
    return sizeof(T) * 2 * (size_t)(2 * TH + maxL - 2) * WaveTile<T>::TW;
}

// The last `levels` analysis levels of basis pb in shared memory, from the h x
// w band at `in` (row stride src_ld): a block per basis.
template <typename T, int L>
__device__ __forceinline__ void dwt_tail(const T* __restrict__ in, int src_ld, T* __restrict__ out, int nx, int h, int w,
                                         int levels, int pb, T inv_sqrt_q, T* smem) {
    constexpr int KX = WaveTile<T>::KX, RK = 2;
    Taps<T, L> f;
    f.load(pb);
    // odd row strides: the row filters' lanes take consecutive rows
    T* band = smem;                       // [h][w + 1]
    T* ta = band + h * (w + 1);           // [h][w / 2 + 1]
    T* td = ta + h * (w / 2 + 1);
    for (int t = threadIdx.x; t < h * w; t += blockDim.x) band[t / w * (w + 1) + t % w] = in[(size_t)(t / w) * src_ld + t % w];
    for (int lev = 0; lev < levels; ++lev) {
        __syncthreads();
        const int hs = h >> 1, wsub = w >> 1, rg = (wsub + KX - 1) / KX, ldt = wsub + 1;
        for (int t = threadIdx.x; t < h * rg; t += blockDim.x) {
            const int r = t & (h - 1), k = t / h * KX;
            T a[KX], d[KX];
            row_filter<T, L, KX, false>(f, band + r * (w + 1), w, k, a, d);
#pragma unroll
            for (int j = 0; j < KX; ++j)
                if (k + j < wsub) {
                    ta[r * ldt + k + j] = a[j];
                    td[r * ldt + k + j] = d[j];
                }
        }
        __syncthreads();
        const bool last = lev == levels - 1;
        const int kg = (hs + RK - 1) / RK;
        for (int t = threadIdx.x; t < kg * wsub; t += blockDim.x) {
            const int kx = t % wsub, ky = t / wsub * RK;
            T ll[RK], lh[RK], hl[RK], hh[RK];
            col_filter<T, L, RK>(f, ta + kx, td + kx, ldt, 2 * ky, h - 1, ll, lh, hl, hh);
#pragma unroll
            for (int j = 0; j < RK; ++j) {
                const int gy = ky + j;
                if (gy >= hs) break;
                if (last) out[(size_t)gy * nx + kx] = ll[j] * inv_sqrt_q;
                else band[gy * (wsub + 1) + kx] = ll[j];
                out[(size_t)gy * nx + wsub + kx] = hl[j] * inv_sqrt_q;
                out[(size_t)(hs + gy) * nx + kx] = lh[j] * inv_sqrt_q;
                out[(size_t)(hs + gy) * nx + wsub + kx] = hh[j] * inv_sqrt_q;
            }
        }
        h = hs;
        w = wsub;
    }
}
// blockIdx.x < nw: a wavelet basis; the blocks past them (when the tail holds
// the first level) copy the Dirac plane
template <typename T>
__global__ void __launch_bounds__(TAIL_THREADS)
k_dwt_tail(const T* __restrict__ src, int src_basis_stride, int src_ld, T* __restrict__ coef,
           const int* __restrict__ planes, int N, int nx, int h, int w, int levels, const int* __restrict__ pids, int nw,
           int dirac_plane, T inv_sqrt_q) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int z = blockIdx.x;
    if (z >= nw) {
        for (int t = threadIdx.x; t < h * w; t += blockDim.x)
            coef[(size_t)dirac_plane * N + (size_t)(t / w) * nx + t % w] = src[(size_t)(t / w) * src_ld + t % w] * inv_sqrt_q;
        return;
    }
    const int pb = pids[z];
    PURIFY_WITH_LENGTH(fbank<T>().len[pb],
                       (dwt_tail<T, L>(src + (size_t)z * src_basis_stride, src_ld, coef + (size_t)planes[z] * N, nx, h, w,
                                       levels, pb, inv_sqrt_q, reinterpret_cast<T*>(smem_raw))));
    pdl_trigger();
}

// ------------------------------------------------------------ synthesis
// Column synthesis of sub-band rows i0 .. i0 + RK - 1 of one column: output
// rows 2 i0 .. 2 i0 + 2 RK - 1 of lo(i) and hi(i), the low- and high-pass
// samples of row i (any i; the accessor wraps).
template <typename T, int L, int RK, typename Lo, typename Hi>
__device__ __forceinline__ void syn_filter(const Taps<T, L>& f, int i0, Lo lo, Hi hi, T (&o)[2 * RK]) {
#pragma unroll
    for (int m = 0; m < 2 * RK; ++m) o[m] = T(0);
#pragma unroll
    for (int i = 0; i < RK + L / 2 - 1; ++i) {
        const T a = lo(i0 - (L / 2 - 1) + i), d = hi(i0 - (L / 2 - 1) + i);
#pragma unroll
        for (int r = 0; r < RK; ++r) {
            const int j = r + L / 2 - 1 - i;   // tap pair of output row pair r
            if (j >= 0 && j < L / 2) {
                o[2 * r] += f.h[2 * j] * a + f.g[2 * j] * d;
                o[2 * r + 1] += f.h[2 * j + 1] * a + f.g[2 * j + 1] * d;
            }
        }
    }
}

// barrier of one group of N threads
template <int N> __device__ __forceinline__ void syn_sync(int group) {
    asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(N) : "memory");
}

// Row synthesis of 2 KX outputs from low-pass samples of `lo` and high-pass
// samples of `hi` (n columns each, periodic), sub-band columns k0 .. k0 + KX - 1
// (k0 a multiple of KX) and the L / 2 - 1 before them; VEC: both rows 16-byte
// aligned, n >= 4 (the window comes in whole 16-byte loads).
template <typename T, int L, int KX, bool VEC>
__device__ __forceinline__ void syn_row(const Taps<T, L>& f, const T* __restrict__ lo, const T* __restrict__ hi, int n,
                                        int k0, T* o) {
    constexpr int V = 16 / sizeof(T), E = L / 2 - 1, EB = (E + V - 1) / V * V, NW = EB + KX;
    alignas(16) T a[NW], d[NW];
    if constexpr (VEC) {
#pragma unroll
        for (int i = 0; i < NW; i += V) {
            const int c = (k0 - EB + i) & (n - 1);
            *reinterpret_cast<uint4*>(a + i) = *reinterpret_cast<const uint4*>(lo + c);
            *reinterpret_cast<uint4*>(d + i) = *reinterpret_cast<const uint4*>(hi + c);
        }
    } else {
#pragma unroll
        for (int i = EB - E; i < NW; ++i) {
            const int c = (k0 - EB + i) & (n - 1);
            a[i] = lo[c];
            d[i] = hi[c];
        }
    }
    T r[2 * KX];
    syn_filter<T, L, KX>(f, 0, [&](int i) { return a[i + EB]; }, [&](int i) { return d[i + EB]; }, r);
#pragma unroll
    for (int e = 0; e < 2 * KX; ++e) o[e] = r[e];
}

// Basis pb's part of the (2 TH) x (2 TW) output tile whose sub-band tile
// starts at (ky0, kx0): rows first (the four sub-bands in 16-byte loads, the low
// and the high rows to shared memory), then columns. Thread item (output
// column, group of RK sub-band rows) holds 2 RK outputs, added to acc. `ll`: the
// low-pass sub-band (row stride ll_ld); the details are in `det` (row stride
// nx); `vec`: both begin at a multiple of 16 bytes, w >= 8. Ends with the shared
// tile free for the next basis.
template <typename T, int L, int TH>
__device__ __forceinline__ void synth_tile(const T* __restrict__ ll, int ll_ld, const T* __restrict__ det, bool vec,
                                           int nx, int h, int w, int ky0, int kx0, int pb, T* smem, int group, int tid,
                                           T (&acc)[2 * WaveTile<T>::SYN_RK]) {
    using W = WaveTile<T>;
    constexpr int TW = W::TW, RK = W::SYN_RK, KX = W::KX, E = L / 2 - 1, RG = TW / KX, CW = 2 * TW;
    constexpr int NT = syn_threads<T, TH>();
    static_assert(E <= 7, "filter longer than the row margin");
    Taps<T, L> f;
    f.load(pb);
    const int hs = h >> 1, wsub = w >> 1;
    T* sL = smem;                    // [TH + 7][CW] rows of the low-pass (along y) half
    T* sH = sL + (TH + 7) * CW;      // and of the high-pass half
    for (int t = tid; t < (TH + E) * RG; t += NT) {
        const int r = t / RG, k = (t - r * RG) * KX;
        if (kx0 + k >= wsub) continue;
        const int ky = (ky0 - E + r) & (hs - 1);
        const T* const lo = det + (size_t)ky * nx + wsub;          // row-detail, column-approx
        const T* const hi = det + (size_t)(hs + ky) * nx;          // row-approx, column-detail
        alignas(16) T oL[2 * KX], oH[2 * KX];
        if (vec) {
            syn_row<T, L, KX, true>(f, ll + (size_t)ky * ll_ld, lo, wsub, kx0 + k, oL);
            syn_row<T, L, KX, true>(f, hi, hi + wsub, wsub, kx0 + k, oH);
        } else {
            syn_row<T, L, KX, false>(f, ll + (size_t)ky * ll_ld, lo, wsub, kx0 + k, oL);
            syn_row<T, L, KX, false>(f, hi, hi + wsub, wsub, kx0 + k, oH);
        }
        constexpr int V = 16 / sizeof(T);
#pragma unroll
        for (int e = 0; e < 2 * KX; e += V) {
            *reinterpret_cast<uint4*>(sL + r * CW + 2 * k + e) = *reinterpret_cast<const uint4*>(oL + e);
            *reinterpret_cast<uint4*>(sH + r * CW + 2 * k + e) = *reinterpret_cast<const uint4*>(oH + e);
        }
    }
    syn_sync<NT>(group);
    {
        const int x = tid % CW, g = tid / CW * RK;
        const T *cl = sL + (g + E) * CW + x, *ch = sH + (g + E) * CW + x;
        T o[2 * RK];
        syn_filter<T, L, RK>(f, 0, [&](int i) { return cl[i * CW]; }, [&](int i) { return ch[i * CW]; }, o);
#pragma unroll
        for (int m = 0; m < 2 * RK; ++m) acc[m] += o[m];
    }
    syn_sync<NT>(group);
}
// The same out of line, for the loop over bases (inlined there, the eight
// lengths' windows were kept live together and spilled).
template <typename T> struct SynthPart { T v[2 * WaveTile<T>::SYN_RK]; };
template <typename T, int L, int TH>
__device__ __noinline__ SynthPart<T> synth_part(const T* __restrict__ ll, int ll_ld, const T* __restrict__ det, bool vec,
                                                int nx, int h, int w, int ky0, int kx0, int pb, T* smem, int group,
                                                int tid) {
    SynthPart<T> p = {};
    synth_tile<T, L, TH>(ll, ll_ld, det, vec, nx, h, w, ky0, kx0, pb, smem, group, tid, p.v);
    return p;
}
template <int V> using Int = std::integral_constant<int, V>;
// tiles of TH sub-band rows that synthesise a w x h band
template <typename T> static int64_t synth_tiles(int w, int h, int TH) {
    return (int64_t)((w / 2 + WaveTile<T>::TW - 1) / WaveTile<T>::TW) * ((h / 2 + TH - 1) / TH);
}
template <typename T> static size_t synth_smem_bytes(int TH) { return sizeof(T) * 2 * (TH + 7) * 2 * WaveTile<T>::TW; }

// One synthesis level for every wavelet basis (blockIdx.z): the reconstructed
// h x w band of basis z into ll_out (row stride w).
template <typename T, int TH>
__global__ void __launch_bounds__(syn_threads<T, TH>())
k_idwt_level(const T* __restrict__ ll_in, int ll_basis_stride, int ll_ld, const T* __restrict__ coef, int vec,
             const int* __restrict__ planes, int N, int nx, T* __restrict__ ll_out, int out_basis_stride, int h,
             int w, const int* __restrict__ pids) {
    using W = WaveTile<T>;
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int z = blockIdx.z, pb = pids[z];
    const int ky0 = blockIdx.y * TH, kx0 = blockIdx.x * W::TW;
    const T* det = coef + (size_t)planes[z] * N;
    const T* ll = ll_in ? ll_in + (size_t)z * ll_basis_stride : det;
    T acc[2 * W::SYN_RK] = {};
    PURIFY_WITH_LENGTH(fbank<T>().len[pb],
                       (synth_tile<T, L, TH>(ll, ll_in ? ll_ld : nx, det, vec != 0, nx, h, w, ky0, kx0, pb,
                                         reinterpret_cast<T*>(smem_raw), 0, (int)threadIdx.x, acc)));
    constexpr int CW = 2 * W::TW;
    const int y = 2 * (ky0 + threadIdx.x / CW * W::SYN_RK), x = 2 * kx0 + threadIdx.x % CW;
    if (x < w) {
        T* out = ll_out + (size_t)z * out_basis_stride + x;
#pragma unroll
        for (int m = 0; m < 2 * W::SYN_RK; ++m)
            if (y + m < h) out[(size_t)(y + m) * w] = acc[m];
    }
    pdl_trigger();
}

// Finest synthesis level summed over all wavelet bases plus the Dirac plane:
// x = (c_dirac + sum_z W_z^T c_z) / sqrt(q). G groups of threads share a
// tile, group g takes bases g, g + G, ... in order (their column passes
// wait for global memory at different times). FP32 adds the even bases' parts
// and the odd ones' in two chains and then those two, whatever G (two short
// chains round less than one: 7.7e-8 against 8.2e-8 of the image); FP64 the
// groups' sums in group order. LEN > 0: all groups run the code of that filter length (see
// the rule in psi_t). When `ll_in` is null (L == 1) the low-pass bands come from
// the coefficient planes.
template <typename T, int TH, int G, int LEN>
__global__ void __launch_bounds__(syn_threads<T, TH>() * G, sizeof(T) == 4 && LEN == 0 ? 2 : 1)
k_idwt_final(const T* __restrict__ ll_in, int ll_basis_stride, const T* __restrict__ coef, int vec,
             const int* __restrict__ planes, int N, int nx, int ny, const int* __restrict__ pids, int nw,
             int dirac_plane, T inv_sqrt_q, T* __restrict__ x) {
    using W = WaveTile<T>;
    constexpr int NO = 2 * W::SYN_RK, NT = syn_threads<T, TH>(), CW = 2 * W::TW, GE = 2 * (TH + 7) * CW;
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* const smem = reinterpret_cast<T*>(smem_raw);
    const int ky0 = blockIdx.y * TH, kx0 = blockIdx.x * W::TW;
    const int group = threadIdx.x / NT, tid = threadIdx.x - group * NT;
    constexpr bool CHAINS = sizeof(T) == 4, OWN_ODD = CHAINS && G == 1;   // OWN_ODD: one group holds both chains
    T acc[NO] = {}, odd[OWN_ODD ? NO : 1] = {};
    for (int z = group; z < nw; z += G) {
        const int pb = pids[z];
        const T* det = coef + (size_t)planes[z] * N;
        const T* ll = ll_in ? ll_in + (size_t)z * ll_basis_stride : det;
        T* const tile = smem + group * GE;
        if constexpr (LEN > 0) {
            synth_tile<T, LEN, TH>(ll, ll_in ? (nx >> 1) : nx, det, vec != 0, nx, ny, nx, ky0, kx0, pb, tile, group, tid, acc);
        } else {
            SynthPart<T> part;
            PURIFY_WITH_LENGTH(fbank<T>().len[pb],
                               (part = synth_part<T, L, TH>(ll, ll_in ? (nx >> 1) : nx, det, vec != 0, nx, ny, nx, ky0,
                                                            kx0, pb, tile, group, tid)));
#pragma unroll
            for (int e = 0; e < NO; ++e) {
                if (OWN_ODD && z % 2 != 0) odd[OWN_ODD ? e : 0] += part.v[e];
                else acc[e] += part.v[e];
            }
        }
    }
    const int y = 2 * (ky0 + tid / CW * W::SYN_RK), xx = 2 * kx0 + tid % CW;
    auto put = [&](int e, T v) {
        if (xx >= nx || y + e >= ny) return;
        const size_t idx = (size_t)(y + e) * nx + xx;
        if (dirac_plane >= 0) v += coef[(size_t)dirac_plane * N + idx];
        x[idx] = v * inv_sqrt_q;
    };
    if constexpr (G == 1) {
#pragma unroll
        for (int e = 0; e < NO; ++e) put(e, OWN_ODD ? acc[e] + odd[OWN_ODD ? e : 0] : acc[e]);
    } else {
        // the groups' sums through shared memory (all are done with their
        // tiles), every G-th output row by one of the groups
        __syncthreads();
#pragma unroll
        for (int e = 0; e < NO; ++e) smem[(group * NO + e) * NT + tid] = acc[e];
        __syncthreads();
        for (int e = group; e < NO; e += G) {
            auto sum = [&](int g) { return smem[(g * NO + e) * NT + tid]; };
            T v = sum(0);
            if constexpr (CHAINS) {
                T w = sum(1);
#pragma unroll
                for (int g = 2; g + 1 < G; g += 2) {
                    v += sum(g);
                    w += sum(g + 1);
                }
                v += w;
            } else {
#pragma unroll
                for (int g = 1; g < G; ++g) v += sum(g);
            }
            put(e, v);
        }
    }
    pdl_trigger();
}

// The coarsest `levels` synthesis levels of a basis in shared memory, up to the
// h x w band, written to ll_out (row stride w): a block per basis.
template <typename T, int L>
__device__ __forceinline__ void idwt_tail(const T* __restrict__ det, int nx, T* __restrict__ out, int h, int w, int levels,
                                          int pb, T* smem) {
    constexpr int KX = WaveTile<T>::KX, RK = 2;
    Taps<T, L> f;
    f.load(pb);
    T* band = smem;                     // the low-pass band so far, [hs][wsub]
    T* sA = band + h * (w + 1);         // [h][wsub + 1]: an odd stride, the row passes' lanes take consecutive rows
    T* sD = sA + h * (w / 2 + 1);
    {
        const int hc = h >> levels, wc = w >> levels;
        for (int t = threadIdx.x; t < hc * wc; t += blockDim.x) band[t] = det[(size_t)(t / wc) * nx + t % wc];
    }
    for (int lev = levels - 1; lev >= 0; --lev) {
        __syncthreads();
        const int hl = h >> lev, wl = w >> lev, hs = hl >> 1, wsub = wl >> 1, rg = (hs + RK - 1) / RK;
        for (int t = threadIdx.x; t < rg * wsub; t += blockDim.x) {
            const int kx = t % wsub, i0 = t / wsub * RK;
            auto at = [&](const T* p) { return [=](int i) { return p[(size_t)(i & (hs - 1)) * nx + kx]; }; };
            T o[2 * RK], q[2 * RK];
            syn_filter<T, L, RK>(f, i0, [&](int i) { return band[(i & (hs - 1)) * wsub + kx]; }, at(det + (size_t)hs * nx), o);
            syn_filter<T, L, RK>(f, i0, at(det + wsub), at(det + (size_t)hs * nx + wsub), q);
#pragma unroll
            for (int m = 0; m < 2 * RK; ++m)
                if (2 * i0 + m < hl) {
                    sA[(2 * i0 + m) * (wsub + 1) + kx] = o[m];
                    sD[(2 * i0 + m) * (wsub + 1) + kx] = q[m];
                }
        }
        __syncthreads();
        T* dst = lev == 0 ? out : band;
        const int cg = (wsub + KX - 1) / KX;
        for (int t = threadIdx.x; t < hl * cg; t += blockDim.x) {
            const int m = t & (hl - 1), k = t / hl * KX;
            const T *ra = sA + m * (wsub + 1), *rd = sD + m * (wsub + 1);
            T o[2 * KX];
            syn_filter<T, L, KX>(f, k, [&](int i) { return ra[i & (wsub - 1)]; }, [&](int i) { return rd[i & (wsub - 1)]; }, o);
#pragma unroll
            for (int e = 0; e < 2 * KX; ++e)
                if (2 * k + e < wl) dst[(size_t)m * wl + 2 * k + e] = o[e];
        }
    }
}
template <typename T>
__global__ void __launch_bounds__(TAIL_THREADS)
k_idwt_tail(const T* __restrict__ coef, const int* __restrict__ planes, int N, int nx, T* __restrict__ ll_out,
            int out_basis_stride, int h, int w, int levels, const int* __restrict__ pids) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int z = blockIdx.x, pb = pids[z];
    PURIFY_WITH_LENGTH(fbank<T>().len[pb],
                       (idwt_tail<T, L>(coef + (size_t)planes[z] * N, nx, ll_out + (size_t)z * out_basis_stride, h, w,
                                        levels, pb, reinterpret_cast<T*>(smem_raw))));
    pdl_trigger();
}
// band and the two half-width columns, odd strides
template <typename T> static size_t tail_smem_bytes(int h, int w) { return sizeof(T) * (size_t)h * (2 * w + 3); }

// ------------------------------------------------------------- launchers
struct WaveletLayout {
    int nw = 0;            // wavelet bases
    int dirac_plane = -1;  // coefficient plane of the Dirac basis, or -1
};

static WaveletLayout layout(const purify_plan* p) {
    WaveletLayout l;
    for (size_t i = 0; i < p->bases.size(); ++i) {
        if (p->bases[i] == 0) l.dirac_plane = (int)i;
        else l.nw++;
    }
    return l;
}

// Device int meta array of a plan: pids[0..8) = db index of each wavelet
// basis, planes[8..16) = its coefficient plane.
static const int* pid_array(const purify_plan* p) { return p->wmeta.as<int>(); }
static const int* plane_array(const purify_plan* p) { return p->wmeta.as<int>() + 8; }

static bool g_bank_ready[64];
static std::mutex g_bank_mutex;

void init_filter_banks() {
    int dev = 0;
    PURIFY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) throw Error{PURIFY_ECUDA, "device index out of range"};
    // one upload per device, also when several host threads make their first call at once
    std::lock_guard<std::mutex> lock(g_bank_mutex);
    if (g_bank_ready[dev]) return;
    FilterBank<float> bf;
    FilterBank<double> bd;
    std::memset(&bf, 0, sizeof(bf));
    std::memset(&bd, 0, sizeof(bd));
    bf.len[0] = bd.len[0] = 0;
    for (int p = 1; p <= 8; ++p) {
        std::vector<double> h = daubechies(p);
        int L = (int)h.size();
        bf.len[p] = bd.len[p] = L;
        for (int n = 0; n < L; ++n) {
            double g = ((n & 1) ? -1.0 : 1.0) * h[L - 1 - n];
            bd.h[p][n] = h[n];
            bd.g[p][n] = g;
            bf.h[p][n] = (float)h[n];
            bf.g[p][n] = (float)g;
        }
    }
    PURIFY_CUDA(cudaMemcpyToSymbol(c_bank_f, &bf, sizeof(bf)));
    PURIFY_CUDA(cudaMemcpyToSymbol(c_bank_d, &bd, sizeof(bd)));
    settle_uploads();
    g_bank_ready[dev] = true;
}

template <typename K> static void wave_smem(K kernel, size_t bytes) {
    if (bytes > 48 * 1024) PURIFY_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
}

// Psi^dagger of an ny x nx image into coefficient planes c: `bufs` the two
// low-pass buffers with their per-basis strides; launched(name) brackets each
// launch (returns a callable run after it).
template <typename T, typename Launched>
static void analyse(const T* x, T* c, int nx, int ny, int levels, int nw, int dirac_plane, int q, int maxL,
                    const int* pids, const int* planes, T* const (&bufs)[2], const int (&strides)[2], cudaStream_t st,
                    Launched launched) {
    using W = WaveTile<T>;
    const T inv_sqrt_q = (T)(1.0 / std::sqrt((double)q));
    const int N = nx * ny;
    int h = ny, w = nx;
    const T* src = x;
    int src_stride = 0, src_ld = nx;
    if (nw == 0) levels = 1;   // the Dirac plane alone
    for (int lev = 0; lev < levels; ++lev) {
        const bool first = lev == 0;
        const int dirac = first && dirac_plane >= 0 ? 1 : 0;
        auto done = launched("dwt_level");
        if (nw > 0 && h * w <= W::TAIL && levels - lev >= 2) {   // (one level alone is faster by tiles: 10.4 us against 12.6 at 256 x 256)
            const size_t sm = tail_smem_bytes<T>(h, w);
            wave_smem(k_dwt_tail<T>, sm);
            launch_dependent(k_dwt_tail<T>, nw + dirac, TAIL_THREADS, sm, st, src, src_stride, src_ld, c, planes, N, nx, h,
                             w, levels - lev, pids, nw, dirac_plane, inv_sqrt_q);
            done();
            return;
        }
        const int hs = h / 2, wsub = w / 2;
        T* llo = lev == levels - 1 ? nullptr : bufs[lev & 1];
        auto go = [&](auto kern, int TH) {
            const size_t sm = dwt_smem_bytes<T>(maxL, TH);
            wave_smem(kern, sm);
            const dim3 g((wsub + W::TW - 1) / W::TW, (hs + TH - 1) / TH, nw + dirac);
            // the image may begin at any element of the caller's array
            const int vec = w >= 4 && (uintptr_t)src % 16 == 0;
            launch_dependent(kern, g, W::THREADS, sm, st, src, src_stride, src_ld, vec, c, planes, N, nx, llo,
                             strides[lev & 1], h, w, pids, nw, dirac_plane, inv_sqrt_q);
        };
        // tall tiles cost less halo; short ones while those do not fill the chip
        if constexpr (sizeof(T) == 4) {
            const int64_t cols = (wsub + W::TW - 1) / W::TW;
            if (cols * ((hs + 31) / 32) * std::max(nw, 1) >= 152 * 4) go(k_dwt_level<T, 32>, 32);
            else if (cols * ((hs + 15) / 16) * std::max(nw, 1) >= 152) go(k_dwt_level<T, 16>, 16);
            else go(k_dwt_level<T, 8>, 8);
        } else {
            go(k_dwt_level<T, 8>, 8);
        }
        done();
        src = llo;
        src_stride = strides[lev & 1];
        src_ld = wsub;
        h = hs;
        w = wsub;
    }
}

static int longest_filter(const purify_plan* p) {
    int maxL = 2;
    for (int b : p->bases) if (b > 0) maxL = std::max(maxL, 2 * b);
    return maxL;
}

template <typename T> static void psi_adj_t(purify_plan* p, const void* xv, void* cv) {
    const WaveletLayout wl = layout(p);
    T* const bufs[2] = {p->ll0.as<T>(), p->ll1.as<T>()};
    const int strides[2] = {(int)(p->N / 4), (int)(p->N / 4)};
    analyse<T>((const T*)xv, (T*)cv, p->nx, p->ny, p->levels, wl.nw, wl.dirac_plane, p->q, longest_filter(p),
               pid_array(p), plane_array(p), bufs, strides, p->stream, [&](const char* name) {
                   auto l = std::make_shared<Launch>(p, name);
                   return [l] { l->done(); };
               });
}

template <typename T> static void psi_t(purify_plan* p, const void* cv, void* xv) {
    using W = WaveTile<T>;
    const T* c = (const T*)cv;
    T* x = (T*)xv;
    const WaveletLayout wl = layout(p);
    const T inv_sqrt_q = (T)(1.0 / std::sqrt((double)p->q));
    const int N = (int)p->N, llstride = (int)(p->N / 4);
    T* bufs[2] = {p->ll0.as<T>(), p->ll1.as<T>()};
    const T* ll_in = nullptr;  // coarsest level reads LL from the coefficients
    const bool aligned = (uintptr_t)c % 16 == 0;   // the coefficients may begin at any element of the caller's array
    int ll_ld = p->nx;
    // levels L .. 2 reconstruct low-pass bands into scratch, the coarse ones
    // together
    int lev = p->levels - 1;
    if (wl.nw > 0) {
        int top = lev + 1;   // finest of the levels whose output fits the tail
        while (top > 1 && ((int64_t)(p->ny >> (top - 1)) * (p->nx >> (top - 1))) <= W::TAIL) --top;
        if (top < lev) {   // (one level alone is faster by tiles)
            const int h = p->ny >> top, w = p->nx >> top;
            T* out = bufs[top & 1];
            const size_t sm = tail_smem_bytes<T>(h, w);
            wave_smem(k_idwt_tail<T>, sm);
            Launch L(p, "idwt_level");
            launch_dependent(k_idwt_tail<T>, wl.nw, TAIL_THREADS, sm, p->stream, c, plane_array(p), N, p->nx, out, llstride, h,
                             w, lev - top + 1, pid_array(p));
            L.done();
            ll_in = out;
            ll_ld = w;
            lev = top - 1;
        }
        for (; lev >= 1; --lev) {
            const int h = p->ny >> lev, w = p->nx >> lev;
            T* out = bufs[lev & 1];
            auto go = [&](auto th) {
                constexpr int TH = decltype(th)::value;
                const dim3 g((w / 2 + W::TW - 1) / W::TW, (h / 2 + TH - 1) / TH, wl.nw);
                Launch L(p, "idwt_level");
                launch_dependent(k_idwt_level<T, TH>, g, syn_threads<T, TH>(), synth_smem_bytes<T>(TH), p->stream, ll_in,
                                 llstride, ll_ld, c, (int)(aligned && w >= 8), plane_array(p), N, p->nx, out, llstride, h,
                                 w, pid_array(p));
                L.done();
            };
            // tall tiles cost less halo; FP64 takes short ones where tall
            // ones are fewer than the SMs (Psi of 128 x 128: 59.7 us against
            // 61.0; of 512 x 512, where they are not: 247 against 240)
            if (sizeof(T) == 8 && synth_tiles<T>(w, h, 16) * wl.nw < 152) go(Int<8>());
            else go(Int<16>());
            ll_in = out;
            ll_ld = w;
        }
    }
    auto go = [&](auto th, auto groups, auto len) {
        constexpr int TH = decltype(th)::value, G = decltype(groups)::value, LEN = decltype(len)::value;
        const size_t sm = synth_smem_bytes<T>(TH) * G;
        wave_smem(k_idwt_final<T, TH, G, LEN>, sm);
        const dim3 g((p->nx / 2 + W::TW - 1) / W::TW, (p->ny / 2 + TH - 1) / TH, 1);
        Launch L(p, "idwt_final");
        launch_dependent(k_idwt_final<T, TH, G, LEN>, g, syn_threads<T, TH>() * G, sm, p->stream, ll_in, llstride, c,
                         (int)(aligned && p->nx >= 8), plane_array(p), N, p->nx, p->ny, pid_array(p), wl.nw,
                         wl.dirac_plane, inv_sqrt_q, x);
        L.done();
    };
    // One SM walks a tile's bases, so tiles are chosen by how many there are.
    // From 256 tall ones on the chip is full: one group of threads, the least
    // halo. With fewer, short tiles and more groups side by side; and where
    // even the short tiles are fewer than the SMs, a tile's time is a chain of
    // latencies, with the fetching of eight filter lengths' code among them:
    // eight groups run one code, of the longest filter's length (shorter
    // filters end in zeros, so an infinite coefficient reaches as far as the
    // longest). Psi over 4 levels (5 at 1024 x 1024), nine bases,
    // us, one group of tall tiles | two of short | eight of the same code:
    // 128 x 128 21.5 17.9 14.3, 256 x 256 24.7 20.2 15.2, 512 x 256 24.3 20.4
    // 19.6, 512 x 512 25.0 21.5 27.8, 1024 x 512 28.4 30.3 42.7, 1024 x 1024
    // 48.5 50.3 77.5. FP64 is bound by its arithmetic: the number of tiles alone
    // decides (64 x 64 51.8 with four groups of 8 rows, 48.2 with eight of 4;
    // 512 x 64 54.5 and 72.0, 67.1 with two of 16; 256 x 256 95.6, 134.8, 84.7).
    const int64_t tall = synth_tiles<T>(p->nx, p->ny, 16);
    if constexpr (sizeof(T) == 4) {
        if (tall >= 256) go(Int<16>(), Int<1>(), Int<0>());
        else if (tall >= 128) go(Int<8>(), Int<2>(), Int<0>());
        else PURIFY_WITH_LENGTH(longest_filter(p), (go(Int<4>(), Int<8>(), Int<L>())));
    } else {
        if (tall >= 128) go(Int<16>(), Int<2>(), Int<0>());
        else if (synth_tiles<T>(p->nx, p->ny, 8) >= 128) go(Int<8>(), Int<4>(), Int<0>());
        else go(Int<4>(), Int<8>(), Int<0>());
    }
}

void launch_psi_adj(purify_plan* p, const void* x, void* c) {
    if (p->dtype == PURIFY_F32) psi_adj_t<float>(p, x, c); else psi_adj_t<double>(p, x, c);
}
void launch_psi(purify_plan* p, const void* c, void* x) {
    if (p->dtype == PURIFY_F32) psi_t<float>(p, c, x); else psi_t<double>(p, c, x);
}

}  // namespace purify

// ------------------------------------------- allocation-free Psi^dagger
// A plan-free variant of the multilevel analysis for callers that must not
// allocate device memory. The low-pass ping-pong scratch of the level
// kernels lives in one file-scope device array instead of plan buffers; every
// device that loads this library holds it until the process exits.
namespace purify {

static const size_t kStaticScratchBytes = size_t(4) << 20;  // 4 MiB
// The two low-pass buffers: level 0 writes nw N / 4 values into the first,
// level 1 nw N / 16 into the second, deeper levels alternate and need less.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];
// the basis table of the current mask (pids, then coefficient planes)
static __device__ __align__(16) int g_static_meta[16];

// Host code cannot use the arrays' names as device addresses: their device
// addresses are looked up once per device (with that device current).
static std::mutex g_static_mutex;
static void* g_static_addr[64];
static void* g_static_meta_addr[64];

static void* symbol_address(const void* symbol, const char* what) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, symbol);
    if (e != cudaSuccess || ptr == nullptr) {
        cudaGetLastError();
        throw Error{PURIFY_ECUDA, std::string("cudaGetSymbolAddress of the ") + what + " failed: " +
                                      cudaGetErrorString(e)};
    }
    return ptr;
}

static void static_addresses(void** scratch, int** meta) {
    int dev = 0;
    PURIFY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) throw Error{PURIFY_ECUDA, "device index out of range"};
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_addr[dev]) {
        g_static_meta_addr[dev] = symbol_address(g_static_meta, "static basis table");
        g_static_addr[dev] = symbol_address(g_static_scratch, "static scratch");
    }
    *scratch = g_static_addr[dev];
    *meta = static_cast<int*>(g_static_meta_addr[dev]);
}

// Basis table of a mask: pids[z] = db index of wavelet z, planes[z] = its
// coefficient plane (written into the static scratch by the device).
__global__ void k_static_meta(unsigned mask, int* meta) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int z = 0, plane = 0;
    for (int b = 0; b < 9; ++b) {
        if (!(mask >> b & 1)) continue;
        if (b > 0) { meta[z] = b; meta[8 + z] = plane; ++z; }
        ++plane;
    }
    for (; z < 8; ++z) { meta[z] = 0; meta[8 + z] = 0; }
}

size_t psi_adj_static_bytes(int nx, int ny, unsigned mask, int dtype) {
    int nw = 0;
    for (int b = 1; b < 9; ++b) nw += (mask >> b & 1);
    size_t rb = dtype == PURIFY_F32 ? 4 : 8;
    size_t N = (size_t)nx * ny;
    return (size_t)nw * (N / 4 + N / 16) * rb;
}

size_t psi_adj_static_capacity() { return kStaticScratchBytes; }

template <typename T>
static void psi_adj_static_t(const T* x, T* c, int nx, int ny, int levels, unsigned mask, cudaStream_t st) {
    void* scratch = nullptr;
    int* meta = nullptr;
    static_addresses(&scratch, &meta);
    const size_t N = (size_t)nx * ny;
    int nw = 0, q = 0, dirac_plane = -1;
    for (int b = 0; b < 9; ++b) {
        if (!(mask >> b & 1)) continue;
        if (b == 0) dirac_plane = q; else ++nw;
        ++q;
    }
    // per-basis strides: N / 4 in the first buffer, N / 16 in the second
    T* const bufs[2] = {static_cast<T*>(scratch), static_cast<T*>(scratch) + (size_t)nw * (N / 4)};
    const int strides[2] = {(int)(N / 4), (int)(N / 16)};
    int maxL = 2;
    for (int b = 1; b < 9; ++b) if (mask >> b & 1) maxL = std::max(maxL, 2 * b);
    k_static_meta<<<1, 32, 0, st>>>(mask, meta);
    PURIFY_CUDA(cudaGetLastError());
    add_launches(1);
    analyse<T>(x, c, nx, ny, levels, nw, dirac_plane, q, maxL, meta, meta + 8, bufs, strides, st, [](const char*) {
        return [] {
            PURIFY_CUDA(cudaGetLastError());
            add_launches(1);
        };
    });
}

void psi_adj_static(const void* x, void* c, int nx, int ny, int levels, unsigned mask, int dtype,
                    cudaStream_t st) {
    init_filter_banks();
    if (dtype == PURIFY_F32) psi_adj_static_t<float>((const float*)x, (float*)c, nx, ny, levels, mask, st);
    else psi_adj_static_t<double>((const double*)x, (double*)c, nx, ny, levels, mask, st);
}

}  // namespace purify
