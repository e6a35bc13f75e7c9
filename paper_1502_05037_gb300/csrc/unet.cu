// Learned warm start: BF16 convolution layers on the fifth-generation tensor
// cores, plus the element-wise kernels of a U-Net (pooling, upsampling,
// masks, loss, Adam).
//
// A 3x3 or 1x1 convolution of an NHWC BF16 image is an implicit GEMM
//   D[pixel][co] = sum over (tap, ci) of A[pixel][(tap, ci)] * W[co][(tap, ci)]
// with M = pixels, N = output channels, K = taps x input channels. A block of
// 128 threads owns a 16 x 8 tile of one image's pixels and a range of the
// output channels. It stages the tile with its one-pixel halo once, channel
// group by channel group (8 channels = 16 bytes a pixel, pixels contiguous: a
// K-major core matrix is 8 pixels of a tile row), so the nine taps are nine
// start addresses into the same copy: tap (dy, dx) is (10 dy + dx) x 16 bytes
// further. The weights come through a ring of shared stages (cp.async), in
// the order of the accumulation (tap by tap, 16 channels an instruction); one
// thread issues tcgen05.mma (M = 128, K = 16) into tensor memory and commits
// each stage to an mbarrier, which frees its slot. The epilogue reads the FP32
// accumulators with tcgen05.ld, adds the bias, applies ReLU (or masks by an
// activation, for gradients) and stores BF16 and/or FP32 in 16-byte pieces.
// Weight gradients are the transposed product over the same tiles
// (k_dw_tc): M = output channels, N = input channels of a tap, K = pixels.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <string>
#include <vector>

#include "internal.h"
#include "tc.cuh"
#include "unet.h"

namespace purify {

static constexpr int CONV_KC = 64;          // K elements per chunk (wide inputs)
static constexpr uint32_t WAIT_LIMIT = 1u << 24;

// Spatial tile and its halo: channel group g of position (py, px) of the
// 18 x 10 halo tile at 16 bytes x (g * TP + py * 10 + px); TP = 181 puts the
// groups of a pixel on distinct banks.
static constexpr int T_ROWS = 16, T_COLS = 8, HALO_W = T_COLS + 2, HALO_N = (T_ROWS + 2) * HALO_W, TP = HALO_N + 1;
static constexpr int CONV_STAGE = 16384;    // bytes of weights per ring stage
static constexpr int CONV_SLOTS = 4;
static constexpr int CONV_THREADS = 256;   // two warps per 32 accumulator rows: each takes every other 16 columns

__device__ __forceinline__ void cp_async16z(uint32_t sdst, const void* gsrc, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sdst), "l"(gsrc), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait_pending() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The halo tile of channel groups [g0, g0 + ng) of image b at tile origin
// (y0, x0) into shared memory at sdst (zero outside the image and past Cin):
// input NHWC, channel stride cs, first channel co, read through a x2 nearest
// upsampling with up = 1. Consecutive threads take consecutive groups of a
// pixel. `vec`: the channels can be copied 8 at a time.
__device__ __forceinline__ void load_halo(unsigned char* sdst, const bf16* in, int b, int y0, int x0, int H, int W,
                                          int Cin, int cs, int co, int up, int g0, int ng, bool vec) {
    const int Hs = H >> up, Ws = W >> up;
    const bf16* const base = in + (size_t)b * Hs * Ws * cs + co + g0 * 8;
    const uint32_t sbase = tc::smem_u32(sdst);
    const int cmax = Cin - g0 * 8;
    // a thread takes channel group g of halo column px and every nr-th row of
    // it (the columns that do not fit the block's threads in further rounds)
    const int cols = ng * HALO_W, nr = max(1, min(T_ROWS + 2, CONV_THREADS / cols));
    for (int j = threadIdx.x; j < cols * nr; j += CONV_THREADS) {
        const int g = j % ng, q = j / ng, px = q % HALO_W, x = x0 + px - 1;
        const bool xin = (unsigned)x < (unsigned)W && g * 8 < cmax;
        const bf16* const col = base + (xin ? (size_t)(x >> up) * cs + g * 8 : 0);
        for (int py = q / HALO_W; py < T_ROWS + 2; py += nr) {
            const int y = y0 + py - 1;
            const bool inside = xin && (unsigned)y < (unsigned)H;
            const bf16* src = inside ? col + (size_t)((y >> up) * Ws) * cs : in;
            const int slot = (g * TP + py * HALO_W + px) * 16;
            if (vec) {
                cp_async16z(sbase + slot, src, inside);
            } else {
                bf16 v[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = inside && g * 8 + e < cmax ? src[e] : __float2bfloat16(0.f);
                *reinterpret_cast<uint4*>(sdst + slot) = *reinterpret_cast<const uint4*>(v);
            }
        }
    }
}

// 16 consecutive output channels c .. c + 15 of pixel q (row values v).
__device__ __forceinline__ void conv_store(const ConvArgs& a, size_t q, int c, float (&v)[16]) {
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        if (c + e < a.Cout) {
            v[e] += a.bias ? __ldg(a.bias + c + e) : 0.f;
            if (a.relu) v[e] = fmaxf(v[e], 0.f);
        }
    }
    // channels below f32_ch in FP32, the others (or all) in BF16
    if (a.out_f32 && c < a.f32_ch) {
        float* o = a.out_f32 + q * a.f32_ch + c;
        const int n = min(16, a.f32_ch - c);
        if (a.residual) {
            for (int e = 0; e < n; ++e) v[e] += a.residual[q * a.f32_ch + c + e];
        }
        if (n == 16 && a.vec_f32) {
#pragma unroll
            for (int e = 0; e < 16; e += 4) *reinterpret_cast<float4*>(o + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        } else {
#pragma unroll
            for (int e = 0; e < 16; ++e)
                if (e < n) o[e] = v[e];
        }
    }
    if (a.out && c + 15 >= a.bf_from) {
        bf16 r[16];
        const bf16* act = a.mask ? a.mask + q * a.mask_cs + a.mask_co + (c - a.bf_from) : nullptr;
        bf16* o = a.out + q * a.out_cs + a.out_co + (c - a.bf_from);
        const bool whole = c >= a.bf_from && c + 16 <= a.Cout && a.vec_out;
        if (whole) {
            if (act) {
                bf16 m[16];
                *reinterpret_cast<uint4*>(m) = *reinterpret_cast<const uint4*>(act);
                *reinterpret_cast<uint4*>(m + 8) = *reinterpret_cast<const uint4*>(act + 8);
#pragma unroll
                for (int e = 0; e < 16; ++e) v[e] = __bfloat162float(m[e]) > 0.f ? v[e] : 0.f;
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) r[e] = __float2bfloat16_rn(v[e]);
            *reinterpret_cast<uint4*>(o) = *reinterpret_cast<const uint4*>(r);
            *reinterpret_cast<uint4*>(o + 8) = *reinterpret_cast<const uint4*>(r + 8);
        } else {
#pragma unroll
            for (int e = 0; e < 16; ++e)
                if (c + e >= a.bf_from && c + e < a.Cout) {
                    float t = v[e];
                    if (act) t = __bfloat162float(act[e]) > 0.f ? t : 0.f;
                    o[e] = __float2bfloat16_rn(t);
                }
        }
    }
}

// Convolution by halo tiles with all of a block's weights in shared memory: a
// block keeps the weights of its output channels [blockIdx.y nsub, + nsub) and
// walks tiles blockIdx.x, + gridDim.x, ...; while the MMAs of a tile run (into
// one of two accumulators), the next tile's halo is copied into the other of
// two buffers and the previous tile's accumulator is stored.
// Eight warps load and store (two per quarter of the accumulator rows), so that
// the issue slots, not one warp's chain of address and conversion work, bound
// a tile: with four, a 32 -> 32 tile took 10 thousand cycles to store and 1.9
// to load beside 2.3 of MMA issue. A gradient (8 images, 256 x 256, 4 levels,
// base 32) took 4438 us and a forward pass of one 361 with a block per tile and
// one thread issuing, and 3402 and 271 now; with a block per tile and the rest
// as here, 3495 and 283.
__global__ void __launch_bounds__(CONV_THREADS) k_conv_tiles(ConvArgs a, int tiles_x, int tiles_y, int ntiles, int nsub) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t s_taddr;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int G8 = a.Cinp / 8, KT = a.k * a.k * G8;
    const int a_bytes = (G8 * TP * 16 + 127) / 128 * 128;
    unsigned char* const sB = smem + 2 * (size_t)a_bytes;
    uint32_t ncols = 32;
    while ((int)ncols < 2 * nsub) ncols <<= 1;
    if (warp == 0) {
        tc::tmem_alloc(&s_taddr, ncols);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        tc::mbar_init(&bar[0], 1);
        tc::mbar_init(&bar[1], 1);
    }
    const int n0 = blockIdx.y * nsub;
    const bool vec_in = a.in_cs % 8 == 0 && a.in_co % 8 == 0 && a.Cin % 8 == 0;
    auto origin = [&](int tile, int& b, int& y0, int& x0) {
        b = tile / (tiles_x * tiles_y);
        const int rem = tile - b * tiles_x * tiles_y;
        y0 = rem / tiles_x * T_ROWS;
        x0 = (rem - rem / tiles_x * tiles_x) * T_COLS;
    };
    auto load = [&](int tile, int buf) {
        int b, y0, x0;
        origin(tile, b, y0, x0);
        load_halo(smem + (size_t)buf * a_bytes, a.in, b, y0, x0, a.H, a.W, a.Cin, a.in_cs, a.in_co, a.up, 0, G8, vec_in);
    };
    // the weights, packed [tap][ci / 8][Npad][8]
    {
        const int dgr = CONV_THREADS / nsub, drow = CONV_THREADS - dgr * nsub;
        int g = tid / nsub, r = tid - g * nsub;
        uint32_t d = tc::smem_u32(sB) + tid * 16;
        while (g < KT) {
            cp_async16z(d, a.w + ((size_t)g * a.Npad + n0 + r) * 8, true);
            d += CONV_THREADS * 16;
            g += dgr;
            r += drow;
            if (r >= nsub) {
                r -= nsub;
                ++g;
            }
        }
    }
    const int first = blockIdx.x, step = gridDim.x;
    load(first, 0);
    cp_async_commit_group();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = s_taddr, idesc = tc::idesc_bf16_f32(128, nsub);
    const uint64_t ad0 = tc::smem_desc(tc::smem_u32(smem), TP * 16, HALO_W * 16);
    const uint64_t bd0 = tc::smem_desc(tc::smem_u32(sB), nsub * 16, 128);
    auto store = [&](int tile, int buf) {
        int b, y0, x0;
        origin(tile, b, y0, x0);
        const int row = (warp & 3) * 32 + lane, y = y0 + row / T_COLS, x = x0 + row % T_COLS;
        const bool ok = y < a.H && x < a.W;
        const size_t q = ((size_t)b * a.H + y) * a.W + x;
        for (int c = (warp >> 2) * 16; c < nsub; c += 32) {
            float v[16];
            tc::tmem_ld16(tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(buf * nsub + c), v);
            if (ok && n0 + c < a.Cout) conv_store(a, q, n0 + c, v);
        }
    };
    int fail = 0, i = 0;
    for (int tile = first; tile < ntiles; tile += step, ++i) {
        const int buf = i & 1;
        cp_async_wait_pending<0>();
        tc::fence_proxy_async();
        tc::fence_before_sync();
        if (__syncthreads_or(fail)) { fail = 1; break; }
        if (warp == 0) {
            tc::fence_after_sync();
            uint64_t bd = bd0;
            const uint64_t ad = ad0 + (uint32_t)(buf * (a_bytes / 16));
            int g = 0, tap = 0, sh = a.k == 3 ? 0 : HALO_W + 1;
            for (int s = 0; s < KT; s += 2) {
                tc::mma_bf16(tbase + (uint32_t)(buf * nsub), ad + (uint32_t)(g * TP + sh), bd, idesc, s > 0 ? 1u : 0u);
                bd += 2 * nsub;
                g += 2;
                if (g == G8) {
                    g = 0;
                    ++tap;
                    sh += tap % 3 == 0 ? HALO_W - 2 : 1;
                }
            }
            tc::mma_commit(&bar[buf]);
        }
        // the MMAs of the tile before are done: its buffer and accumulator are free to use
        if (i > 0 && !tc::mbar_wait(&bar[buf ^ 1], ((i - 1) >> 1) & 1, WAIT_LIMIT)) fail = 1;
        if (!fail && tile + step < ntiles) load(tile + step, buf ^ 1);
        cp_async_commit_group();
        if (!fail && i > 0) {
            tc::fence_after_sync();
            store(tile - step, buf ^ 1);
        }
    }
    if (!fail && !tc::mbar_wait(&bar[(i - 1) & 1], ((i - 1) >> 1) & 1, WAIT_LIMIT)) fail = 1;
    cp_async_wait_pending<0>();
    fail = __syncthreads_or(fail);
    tc::fence_after_sync();
    if (!fail) store(first + (i - 1) * step, (i - 1) & 1);
    else if (tid == 0) atomicExch(a.err, 1);
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, ncols);
}

// Convolution by halo tiles, the weights streamed (wide inputs). blockIdx.x: tile; blockIdx.y:
// output channels [blockIdx.y nsub, + nsub). kg: 8-channel groups of weights per
// ring stage (even).
// Bound by shared-memory bandwidth (a 128 x N x 16 MMA reads (128 + N) x 32
// bytes) and, for the narrow layers, by the copies into it; several blocks per
// SM overlap one's copies with another's MMAs and epilogue. The form before it
// gathered every tap's rows anew and waited for the MMAs after each 64 channels:
// 8 images of 32 x 32, 256 to 512 channels, took 154 us, now 44.
__global__ void __launch_bounds__(CONV_THREADS) k_conv_halo(ConvArgs a, int tiles_x, int tiles_y, int nsub, int kg, int slots) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar[CONV_SLOTS];
    __shared__ uint32_t s_taddr;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int G8 = a.Cinp / 8;                       // channel groups of the input
    const int KT = a.k * a.k * G8;                   // channel groups over all taps
    const int NS = (KT + kg - 1) / kg;               // stages
    unsigned char* const sA = smem;
    unsigned char* const sB = smem + ((size_t)G8 * TP * 16 + 127) / 128 * 128;
    const int slot_bytes = kg * nsub * 16;
    uint32_t ncols = 32;
    while ((int)ncols < nsub) ncols <<= 1;
    if (warp == 0) {
        tc::tmem_alloc(&s_taddr, ncols);
        tc::tmem_relinquish();
    }
    if (tid == 0)
        for (int i = 0; i < slots; ++i) tc::mbar_init(&bar[i], 1);
    const int tile = blockIdx.x;
    const int b = tile / (tiles_x * tiles_y), rem = tile - b * tiles_x * tiles_y;
    const int y0 = rem / tiles_x * T_ROWS, x0 = (rem % tiles_x) * T_COLS;
    const int n0 = blockIdx.y * nsub;
    const bool vec_in = a.in_cs % 8 == 0 && a.in_co % 8 == 0 && a.Cin % 8 == 0;
    load_halo(sA, a.in, b, y0, x0, a.H, a.W, a.Cin, a.in_cs, a.in_co, a.up, 0, G8, vec_in);
    // stage i of the weights: channel groups [i kg, (i + 1) kg) of the packed
    // order [tap][ci / 8][Npad][8], this block's output channels
    const int dgr = CONV_THREADS / nsub, drow = CONV_THREADS - dgr * nsub, g_first = tid / nsub, r_first = tid - g_first * nsub;
    const uint32_t b0 = tc::smem_u32(sB);
    auto load_stage = [&](int i) {
        const int k0 = i * kg, n = min(kg, KT - k0);
        uint32_t d = b0 + (uint32_t)((i % slots) * slot_bytes + tid * 16);
        const bf16* const src = a.w + ((size_t)k0 * a.Npad + n0) * 8;
        int g = g_first, r = r_first;
        while (g < n) {
            cp_async16z(d, src + (size_t)(g * a.Npad + r) * 8, true);
            d += CONV_THREADS * 16;
            g += dgr;
            r += drow;
            if (r >= nsub) {
                r -= nsub;
                ++g;
            }
        }
    };
#pragma unroll
    for (int i = 0; i < CONV_SLOTS - 1; ++i) {
        if (i < NS && i < slots) load_stage(i);
        cp_async_commit_group();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = s_taddr, idesc = tc::idesc_bf16_f32(128, nsub);
    // operand descriptors; a start address moves in units of 16 bytes
    const uint64_t ad0 = tc::smem_desc(tc::smem_u32(sA), TP * 16, HALO_W * 16);
    const uint64_t bd0 = tc::smem_desc(b0, nsub * 16, 128);
    int tap = 0, g = 0, fail = 0;   // of the next K step
    int sh = a.k == 3 ? 0 : HALO_W + 1;
    for (int i = 0; i < NS; ++i) {
        cp_async_wait_pending<CONV_SLOTS - 2>();
        tc::fence_proxy_async();
        tc::fence_before_sync();
        if (__syncthreads_or(fail)) { fail = 1; break; }
        if (warp == 0) {
            tc::fence_after_sync();
            const int n = min(kg, KT - i * kg);
            uint64_t bd = bd0 + (uint32_t)((i % slots) * (slot_bytes / 16));
            for (int s = 0; s < n; s += 2) {
                tc::mma_bf16(tbase, ad0 + (uint32_t)(g * TP + sh), bd, idesc, (i > 0 || s > 0) ? 1u : 0u);
                bd += 2 * nsub;
                g += 2;
                if (g == G8) {
                    g = 0;
                    ++tap;
                    sh += tap % 3 == 0 ? HALO_W - 2 : 1;
                }
            }
            tc::mma_commit(&bar[i % slots]);
        }
        // refill the slot of the stage before, once its MMAs are done
        const int nx = i + CONV_SLOTS - 1;
        if (nx < NS) {
            if (i > 0 && !tc::mbar_wait(&bar[(i - 1) % slots], ((i - 1) / slots) & 1, WAIT_LIMIT)) fail = 1;
            if (!fail) load_stage(nx);
        }
        cp_async_commit_group();
    }
    if (!fail && !tc::mbar_wait(&bar[(NS - 1) % slots], ((NS - 1) / slots) & 1, WAIT_LIMIT)) fail = 1;
    cp_async_wait_pending<0>();
    fail = __syncthreads_or(fail);
    tc::fence_after_sync();
    if (!fail) {
        // accumulator row of this lane: pixel (row / 8, row % 8) of the tile
        const int row = (warp & 3) * 32 + lane, y = y0 + row / T_COLS, x = x0 + row % T_COLS;
        const bool ok = y < a.H && x < a.W;
        const size_t q = ((size_t)b * a.H + y) * a.W + x;
        for (int c = (warp >> 2) * 16; c < nsub; c += 32) {
            float v[16];
            tc::tmem_ld16(tbase + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c, v);
            if (ok && n0 + c < a.Cout) conv_store(a, q, n0 + c, v);
        }
    } else if (tid == 0) {
        atomicExch(a.err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, ncols);
}

// The form for inputs too wide for a whole halo tile in shared memory: a block
// owns 128 consecutive pixels and all output channels and gathers each tap's
// rows, 64 channels at a time.
__global__ void __launch_bounds__(128) k_conv_tc(ConvArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    bf16* sA = reinterpret_cast<bf16*>(smem);                       // 128 x KC
    bf16* sB = sA + 128 * CONV_KC;                                  // Npad x KC
    uint64_t* bar = reinterpret_cast<uint64_t*>(sB + 256 * CONV_KC);
    uint32_t* s_taddr = reinterpret_cast<uint32_t*>(bar + 1);
    int* s_fail = reinterpret_cast<int*>(s_taddr + 1);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int Npad = a.Npad;
    uint32_t ncols = 32;
    while ((int)ncols < Npad) ncols <<= 1;
    if (warp == 0) {
        tc::tmem_alloc(s_taddr, ncols);
        tc::tmem_relinquish();
    }
    if (tid == 0) {
        tc::mbar_init(bar, 1);
        *s_fail = 0;
    }
    tc::fence_proxy_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = *s_taddr;
    const uint32_t idesc = tc::idesc_bf16_f32(128, Npad);

    const int HW = a.H * a.W;
    const int npix = a.B * HW;
    const int q = blockIdx.x * 128 + tid;
    const bool qok = q < npix;
    int pb = 0, py = 0, px = 0;
    if (qok) { pb = q / HW; int rem = q - pb * HW; py = rem / a.W; px = rem - py * a.W; }
    const bool vec_in = (a.in_cs % 8 == 0) && (a.in_co % 8 == 0) && (a.Cin % 8 == 0);
    const int half = a.k / 2;
    uint32_t phase = 0;
    int chunk = 0;
    bool failed = false;
    for (int tap = 0; tap < a.k * a.k && !failed; ++tap) {
        const int dy = tap / a.k - half, dx = tap % a.k - half;
        const int yy = py + dy, xx = px + dx;
        const bool inside = qok && yy >= 0 && yy < a.H && xx >= 0 && xx < a.W;
        const int sh = a.up ? 1 : 0;
        const int Hs = a.H >> sh, Ws = a.W >> sh;
        const bf16* src =
            inside ? a.in + ((size_t)(pb * Hs + (yy >> sh)) * Ws + (xx >> sh)) * a.in_cs + a.in_co : a.in;
        for (int c0 = 0; c0 < a.Cinp; c0 += CONV_KC) {
            const int kc = min(CONV_KC, a.Cinp - c0);        // multiple of 16
            const int kcu = kc / 8;                           // 16-byte units per row
            // A row `tid`: channels c0 .. c0 + kc of the tap's source pixel
            unsigned char* arow = reinterpret_cast<unsigned char*>(sA) + (size_t)(tid / 8) * kcu * 128 + (tid % 8) * 16;
            for (int j = 0; j < kcu; ++j) {
                uint4 v = make_uint4(0, 0, 0, 0);
                const int cbase = c0 + 8 * j;
                if (inside) {
                    if (vec_in && cbase + 8 <= a.Cin) {
                        v = *reinterpret_cast<const uint4*>(src + cbase);
                    } else if (cbase < a.Cin) {
                        bf16 tmp[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) tmp[e] = (cbase + e < a.Cin) ? src[cbase + e] : __float2bfloat16(0.f);
                        v = *reinterpret_cast<uint4*>(tmp);
                    }
                }
                *reinterpret_cast<uint4*>(arow + j * 128) = v;
            }
            // B rows: weights of every output channel for this chunk
            for (int n = tid; n < Npad; n += 128) {
                const bf16* wsrc = a.w + ((size_t)(tap * (a.Cinp / 8) + c0 / 8) * a.Npad + n) * 8;
                unsigned char* brow = reinterpret_cast<unsigned char*>(sB) + (size_t)(n / 8) * kcu * 128 + (n % 8) * 16;
                for (int j = 0; j < kcu; ++j)
                    *reinterpret_cast<uint4*>(brow + j * 128) = *reinterpret_cast<const uint4*>(wsrc + (size_t)8 * j * a.Npad);
            }
            tc::fence_proxy_async();
            tc::fence_before_sync();
            __syncthreads();
            if (warp == 0) {
                tc::fence_after_sync();
                const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
                for (int s = 0; s < kc / 16; ++s) {
                    uint64_t ad = tc::smem_desc(a0 + s * 256, 128, kcu * 128);
                    uint64_t bd = tc::smem_desc(b0 + s * 256, 128, kcu * 128);
                    tc::mma_bf16(tbase, ad, bd, idesc, (chunk > 0 || s > 0) ? 1u : 0u);
                }
                tc::mma_commit(bar);
            }
            // the shared buffers are reused by the next chunk: wait for the MMAs
            bool done = tc::mbar_wait(bar, phase, WAIT_LIMIT);
            phase ^= 1;
            if (!done) atomicExch(s_fail, 1);
            __syncthreads();
            if (*s_fail) failed = true;
            ++chunk;
            if (failed) break;
        }
    }
    tc::fence_after_sync();
    if (!failed) {
        // epilogue: lane of this warp = accumulator row = pixel q0 + 32*warp + lane
        const int row = warp * 32 + lane;
        const int qo = blockIdx.x * 128 + row;
        for (int c = 0; c < Npad; c += 16) {
            float v[16];
            tc::tmem_ld16(tbase + ((uint32_t)(warp * 32) << 16) + (uint32_t)c, v);
            if (qo < npix && c < a.Cout) conv_store(a, qo, c, v);
        }
    } else if (tid == 0) {
        atomicExch(a.err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, ncols);
}

static size_t conv_smem_bytes() { return sizeof(bf16) * (128 + 256) * CONV_KC + 64; }

// the shared-memory limit is a per-device setting: raised on a kernel's first
// launch on each device (threads racing on it set the same value)
template <typename K> static void raise_smem(std::atomic<bool> (&done)[64], K kernel, int bytes) {
    int dev = 0;
    PURIFY_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) throw Error{PURIFY_ECUDA, "device index out of range"};
    if (!done[dev].load(std::memory_order_relaxed)) {
        PURIFY_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
        done[dev].store(true, std::memory_order_relaxed);
    }
}
static constexpr int kConvSmemMax = 216 * 1024;   // largest request of the kernels here

void conv_tc_launch(const ConvArgs& args, cudaStream_t st) {
    ConvArgs a = args;
    if (a.Npad < 16 || a.Npad > 256 || a.Npad % 16 || a.Cinp % 16 || (a.k != 1 && a.k != 3))
        throw Error{PURIFY_EINVAL, "conv: unsupported shape"};
    if (a.out_f32 && a.f32_ch == 0) a.f32_ch = a.Cout;
    a.vec_out = a.out && a.out_cs % 8 == 0 && a.out_co % 8 == 0 && a.bf_from % 16 == 0 &&
                (!a.mask || (a.mask_cs % 8 == 0 && a.mask_co % 8 == 0)) && (uintptr_t)a.out % 16 == 0 &&
                (uintptr_t)a.mask % 16 == 0;
    // out_f32 may be a caller's array, aligned to its elements only
    a.vec_f32 = a.out_f32 && a.f32_ch % 4 == 0 && (uintptr_t)a.out_f32 % 16 == 0;
    const int tx = (a.W + T_COLS - 1) / T_COLS, ty = (a.H + T_ROWS - 1) / T_ROWS;
    const int64_t tiles = (int64_t)a.B * tx * ty;
    const int KT = a.k * a.k * a.Cinp / 8;
    const size_t halo = ((size_t)a.Cinp / 8 * TP * 16 + 127) / 128 * 128;
    if (tiles >= (int64_t)1 << 31) throw Error{PURIFY_EINVAL, "conv: image too large"};
    // output channels per block: all, or halves until a block's weights fit
    // shared memory beside two halo tiles (wider outputs repeat the copies
    // and read the tile for fewer channels: not below 32)
    int nsub = a.Npad;
    auto resident = [&](int n) { return 2 * halo + (size_t)KT * n * 16; };
    while (nsub % 64 == 0 && resident(nsub) > (size_t)200 * 1024) nsub /= 2;
    if (resident(nsub) <= (size_t)200 * 1024) {
        // and while the blocks do not fill the chip
        while (nsub % 32 == 0 && tiles * (a.Npad / nsub) < 152) nsub /= 2;
        const size_t sm = resident(nsub);
        const int per_sm = std::max(1, std::min((int)((size_t)220 * 1024 / (sm + 1024)), 256 / std::max(32, 2 * nsub)));
        const int gx = (int)std::min<int64_t>(tiles, std::max(1, 152 * per_sm / (a.Npad / nsub)));
        static std::atomic<bool> tiles_attr[64];
        raise_smem(tiles_attr, k_conv_tiles, kConvSmemMax);
        k_conv_tiles<<<dim3((unsigned)gx, a.Npad / nsub), CONV_THREADS, sm, st>>>(a, tx, ty, (int)tiles, nsub);
        PURIFY_CUDA(cudaGetLastError());
        add_launches(1);
        return;
    }
    nsub = a.Npad;
    while (nsub % 32 == 0 && tiles * (a.Npad / nsub) < 152) nsub /= 2;
    const int kg = std::min(std::max(2, CONV_STAGE / (nsub * 16) / 2 * 2), KT);
    const int slots = std::min(CONV_SLOTS, (KT + kg - 1) / kg);
    const size_t sm = halo + (size_t)slots * kg * nsub * 16;
    if (sm <= (size_t)200 * 1024) {
        static std::atomic<bool> halo_attr[64];
        raise_smem(halo_attr, k_conv_halo, kConvSmemMax);
        k_conv_halo<<<dim3((unsigned)tiles, a.Npad / nsub), CONV_THREADS, sm, st>>>(a, tx, ty, nsub, kg, slots);
    } else {
        static std::atomic<bool> attr[64];
        raise_smem(attr, k_conv_tc, (int)conv_smem_bytes());
        const int npix = a.B * a.H * a.W;
        k_conv_tc<<<(npix + 127) / 128, 128, conv_smem_bytes(), st>>>(a);
    }
    PURIFY_CUDA(cudaGetLastError());
    add_launches(1);
}

// ------------------------------------------------------- weight gradients
// dW[co][tap][ci] += sum over pixels of gz[p][co] x[p + tap][ci] on the tensor
// cores: D[co][(tap, ci)], M = 128 output channels (zero rows past Cout), N =
// nt input channels of one tap per MMA, K = 16 pixels (two rows of the tile).
// A block holds the accumulators of its taps side by side in tensor memory
// (taps x nt <= 512 columns) and walks pixel tiles tile0, tile0 + gridDim.y,
// ...; per tile it stages gz (16 x 8 pixels) and the halo of x, three tiles in
// flight. Pixels are the contiguous axis of neither operand, so both are
// MN-major: a core matrix is 8 pixels x 8 channels, 16 bytes a pixel, exactly
// what the copies write; a tap is again a start address.
// By register tiles on the CUDA cores this took 10.5 ms of a 19.7 ms gradient
// (8 images of 256 x 256, 4 levels, base 32), now 1.2 ms (1.6 with four warps a
// block and one thread issuing).
// The tensor core's own FP32 additions lose more than a rounded sum's: over
// the hundreds of MMAs of a block's tiles the error against 64 bits was 1.8e-6
// to 4e-6 where the CUDA cores had 3.5e-7 to 4.5e-7. The accumulators are
// therefore added up in rounded FP32 every DW_FLUSH tiles (8 MMAs each), which
// leaves 1.7e-7 to 3.7e-7 on the layers of the 8-image case, against 1.4e-7 to
// 4.5e-7 of the same sums by FP32 multiply-adds alone.
static constexpr int DW_SLOTS = 3;
static constexpr int DW_FLUSH = 3;
static constexpr int GP = T_ROWS * T_COLS + 1;   // gz group stride in pixels
__global__ void __launch_bounds__(CONV_THREADS)
k_dw_tc(const bf16* __restrict__ gz, int Cout, const bf16* __restrict__ x, int xcs, int xco, int Cin, int B, int H, int W,
        int up, int k, int tiles_x, int tiles_y, int nt, int ntap, int ci_tiles, int tap_groups,
        float* __restrict__ dW, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bar[DW_SLOTS];
    __shared__ uint32_t s_taddr;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int quarter = warp & 3;   // accumulator rows 32 quarter .. + 31
    int id = blockIdx.x;
    const int tg = id % tap_groups; id /= tap_groups;
    const int ci0 = (id % ci_tiles) * nt, co0 = id / ci_tiles * 128;
    const int tap0 = tg * ntap, taps = min(ntap, k * k - tap0);
    const int NG = nt / 8;
    const int a_bytes = 16 * GP * 16, slot_bytes = ((a_bytes + NG * TP * 16) + 127) / 128 * 128;
    const int ntiles = B * tiles_x * tiles_y;
    const int first = blockIdx.y, step = gridDim.y, NS = (ntiles - first + step - 1) / step;
    if (warp == 0) {
        tc::tmem_alloc(&s_taddr, 512);
        tc::tmem_relinquish();
    }
    if (tid == 0)
        for (int i = 0; i < DW_SLOTS; ++i) tc::mbar_init(&bar[i], 1);
    const int ng = min(16, (Cout - co0 + 7) / 8);   // channel groups of gz; those past them stay zero
    const int dpos = CONV_THREADS / ng, dgr = CONV_THREADS - dpos * ng, pos_first = tid / ng, g_first = tid - pos_first * ng;
    auto load_tile = [&](int i) {
        const int tile = first + i * step;
        const int b = tile / (tiles_x * tiles_y), rem = tile - b * tiles_x * tiles_y;
        const int y0 = rem / tiles_x * T_ROWS, x0 = (rem % tiles_x) * T_COLS;
        unsigned char* d = smem + (size_t)(i % DW_SLOTS) * slot_bytes;
        uint32_t sd = tc::smem_u32(d);
        const bf16* const base = gz + (size_t)b * H * W * Cout + co0;
        int pos = pos_first, g = g_first;
        while (pos < T_ROWS * T_COLS) {
            const int y = y0 + pos / T_COLS, xx = x0 + pos % T_COLS;
            const bool ok = y < H && xx < W;
            cp_async16z(sd + (uint32_t)(g * GP + pos) * 16, ok ? base + (size_t)(y * W + xx) * Cout + g * 8 : gz, ok);
            pos += dpos;
            g += dgr;
            if (g >= ng) {
                g -= ng;
                ++pos;
            }
        }
        load_halo(d + a_bytes, x, b, y0, x0, H, W, Cin, xcs, xco, up, ci0 / 8, NG, true);
    };
    // the zero rows of narrow outputs, written once
    for (int s = 0; s < DW_SLOTS; ++s)
        for (int t = tid; t < 16 * GP; t += CONV_THREADS)
            *reinterpret_cast<uint4*>(smem + (size_t)s * slot_bytes + (size_t)t * 16) = make_uint4(0, 0, 0, 0);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < DW_SLOTS - 1; ++i) {
        if (i < NS) load_tile(i);
        cp_async_commit_group();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = s_taddr;
    // both operands MN-major (bits 15, 16 of the instruction descriptor)
    const uint32_t idesc = tc::idesc_bf16_f32(128, nt) | (1u << 15) | (1u << 16);
    // channel groups GP (TP) pixels apart, tile rows 8 (10)
    const uint64_t ad0 = tc::smem_desc(tc::smem_u32(smem), T_COLS * 16, GP * 16);
    const uint64_t bd0 = tc::smem_desc(tc::smem_u32(smem) + a_bytes, HALO_W * 16, TP * 16);
    // the accumulators' sums so far added to dW; with at most 32 output
    // channels (one warp's rows) to the block's own sums in shared memory
    // until the last time
    const int co = co0 + quarter * 32 + lane;
    float* const sums = Cout <= 32 ? reinterpret_cast<float*>(smem + (size_t)DW_SLOTS * slot_bytes) + lane : nullptr;
    auto flush = [&](bool first_time, bool last) {
        if (co0 + quarter * 32 >= Cout) return;   // this warp's rows are the zero rows
        const int n = min(nt, Cin - ci0);
        for (int t = 0; t < taps; ++t) {
            float* row = dW + ((size_t)co * k * k + tap0 + t) * Cin + ci0;
            for (int c = (warp >> 2) * 16; c < nt; c += 32) {
                float v[16];
                tc::tmem_ld16(tbase + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(t * nt + c), v);
                if (co >= Cout) continue;
                if (sums) {
                    float* p = sums + (t * nt + c) * 32;
                    if (!first_time) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] += p[e * 32];
                    }
                    if (!last) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) p[e * 32] = v[e];
                        continue;
                    }
                }
                if (c + 16 <= n && (uintptr_t)(row + c) % 16 == 0) {
#pragma unroll
                    for (int e = 0; e < 16; e += 4)
                        asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(row + c + e), "f"(v[e]),
                                     "f"(v[e + 1]), "f"(v[e + 2]), "f"(v[e + 3])
                                     : "memory");
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e)
                        if (c + e < n) atomicAdd(row + c + e, v[e]);
                }
            }
        }
    };
    int fail = 0;
    for (int i = 0; i < NS; ++i) {
        cp_async_wait_pending<DW_SLOTS - 2>();
        tc::fence_proxy_async();
        tc::fence_before_sync();
        if (__syncthreads_or(fail)) { fail = 1; break; }
        if (warp == 0) {
            tc::fence_after_sync();
            const uint32_t slot = (uint32_t)((i % DW_SLOTS) * (slot_bytes / 16));
            for (int t = 0; t < taps; ++t) {
                const int tap = tap0 + t, sh = k == 3 ? tap / 3 * HALO_W + tap % 3 : HALO_W + 1;
                const uint64_t ad = ad0 + slot, bd = bd0 + slot + sh;
                const uint32_t d = tbase + (uint32_t)(t * nt);
#pragma unroll
                for (int s = 0; s < T_ROWS; s += 2)
                    tc::mma_bf16(d, ad + s * T_COLS, bd + s * HALO_W, idesc, (i % DW_FLUSH > 0 || s > 0) ? 1u : 0u);
            }
            tc::mma_commit(&bar[i % DW_SLOTS]);
        }
        const int nx = i + DW_SLOTS - 1;
        if (nx < NS) {
            if (i > 0 && !tc::mbar_wait(&bar[(i - 1) % DW_SLOTS], ((i - 1) / DW_SLOTS) & 1, WAIT_LIMIT)) fail = 1;
            if (!fail) load_tile(nx);
        }
        cp_async_commit_group();
        if ((i + 1) % DW_FLUSH == 0 && i + 1 < NS) {
            if (!fail && !tc::mbar_wait(&bar[i % DW_SLOTS], (i / DW_SLOTS) & 1, WAIT_LIMIT)) fail = 1;
            tc::fence_after_sync();
            if (!fail) flush(i < DW_FLUSH, false);
        }
    }
    if (!fail && NS > 0 && !tc::mbar_wait(&bar[(NS - 1) % DW_SLOTS], ((NS - 1) / DW_SLOTS) & 1, WAIT_LIMIT)) fail = 1;
    cp_async_wait_pending<0>();
    fail = __syncthreads_or(fail);
    tc::fence_after_sync();
    if (!fail) {
        flush(NS <= DW_FLUSH, true);
    } else if (tid == 0) {
        atomicExch(err, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 0) tc::tmem_dealloc(tbase, 512);
}

bool dw_tc_ok(int Cout, int Cin, int xcs, int xco) {
    return Cout % 8 == 0 && Cin % 8 == 0 && xcs % 8 == 0 && xco % 8 == 0;
}

void dw_tc_launch(const bf16* gz, int Cout, const bf16* x, int xcs, int xco, int Cin, int B, int H, int W, int up, int k,
                  float* dW, int* err, cudaStream_t st) {
    const int tx = (W + T_COLS - 1) / T_COLS, ty = (H + T_ROWS - 1) / T_ROWS;
    const int nt = Cin <= 32 ? (Cin <= 16 ? 16 : 32) : 64;
    const int ntap = k == 1 ? 1 : (nt == 64 ? 5 : 9);   // 512 accumulator columns hold 8 taps of 64
    const int tap_groups = (k * k + ntap - 1) / ntap, ci_tiles = (Cin + nt - 1) / nt, co_tiles = (Cout + 127) / 128;
    const int64_t tiles = (int64_t)B * tx * ty;
    // one block per SM (all of its tensor memory)
    const int blocks = tap_groups * ci_tiles * co_tiles;
    const int split = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, 152 / blocks));
    const int slot = ((16 * GP * 16 + nt / 8 * TP * 16) + 127) / 128 * 128;
    static std::atomic<bool> attr[64];
    raise_smem(attr, k_dw_tc, kConvSmemMax);
    const size_t sums = Cout <= 32 ? (size_t)ntap * nt * 32 * sizeof(float) : 0;
    k_dw_tc<<<dim3(blocks, split), CONV_THREADS, (size_t)DW_SLOTS * slot + sums, st>>>(gz, Cout, x, xcs, xco, Cin, B, H, W, up, k, tx, ty, nt,
                                                                      ntap, ci_tiles, tap_groups, dW, err);
    PURIFY_CUDA(cudaGetLastError());
    add_launches(1);
}

// ----------------------------------------------------------- conversions
__global__ void k_f32_to_bf16(const float* __restrict__ x, bf16* __restrict__ y, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = __float2bfloat16_rn(x[i]);
}

// FP32 weights [Cout][k][k][Cin] -> BF16 [k][k][Cinp / 8][Npad][8], zero padded
__global__ void k_pack_weights(const float* __restrict__ w, bf16* __restrict__ wp, int Cout, int k, int Cin,
                               int Npad, int Cinp) {
    const int64_t n = (int64_t)Npad * k * k * Cinp;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / 8;
        const int co = (int)(r % Npad), g = (int)(r / Npad), tap = g / (Cinp / 8);
        const int ci = (g - tap * (Cinp / 8)) * 8 + (int)(i % 8);
        float v = (co < Cout && ci < Cin) ? w[((int64_t)co * k * k + tap) * Cin + ci] : 0.f;
        wp[i] = __float2bfloat16_rn(v);
    }
}

int round16(int v) { return (v + 15) / 16 * 16; }

// Convolution of FP32 NHWC input through BF16 tensor cores (test and
// inference entry; allocates its staging buffers).
void conv2d_f32(const float* x, int B, int H, int W, int Cin, const float* w, const float* bias, int Cout, int k,
                int relu, float* out, cudaStream_t st) {
    const int Cinp = round16(Cin), Npad = std::max(16, round16(Cout));
    DevBuf xb, wb, err;
    xb.alloc(sizeof(bf16) * (size_t)B * H * W * Cin);
    wb.alloc(sizeof(bf16) * (size_t)Npad * k * k * Cinp);
    err.alloc(sizeof(int));
    PURIFY_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), st));
    const int64_t nx = (int64_t)B * H * W * Cin;
    k_f32_to_bf16<<<(int)std::min<int64_t>(4096, (nx + 255) / 256), 256, 0, st>>>(x, xb.as<bf16>(), nx);
    k_pack_weights<<<256, 256, 0, st>>>(w, wb.as<bf16>(), Cout, k, Cin, Npad, Cinp);
    PURIFY_CUDA(cudaGetLastError());
    add_launches(2);
    ConvArgs a{};
    a.in = xb.as<bf16>();
    a.B = B; a.H = H; a.W = W; a.Cin = Cin; a.in_cs = Cin; a.in_co = 0;
    a.w = wb.as<bf16>(); a.k = k; a.Cinp = Cinp; a.Npad = Npad;
    a.bias = bias; a.Cout = Cout; a.relu = relu;
    a.out = nullptr; a.out_f32 = out; a.residual = nullptr;
    a.err = err.as<int>();
    conv_tc_launch(a, st);
    int herr = 0;
    PURIFY_CUDA(cudaMemcpyAsync(&herr, err.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    PURIFY_CUDA(cudaStreamSynchronize(st));
    if (herr) throw Error{PURIFY_ETIMEOUT, "tensor-core convolution: a bounded wait gave up"};
}

}  // namespace purify
