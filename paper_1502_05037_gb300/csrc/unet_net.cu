// Learned warm start: the U-Net driver (forward, backward, Adam) on top of
// the tensor-core convolution of unet.cu. The network is not in the paper: it
// maps a normalised dirty image to a starting point for SDMM, which leaves the
// convex problem (3) and its solution unchanged.
//
// Layout NHWC; activations BF16 (the tensor-core operands), gradients and
// parameters FP32. Architecture (L levels, base width c):
//   encoder l < L-1: conv3x3+ReLU, conv3x3+ReLU (kept as the skip), maxpool 2x2
//   bottom:          conv3x3+ReLU, conv3x3+ReLU
//   decoder l:       x2 upsampling fused into conv3x3+ReLU (2c -> c), concat with
//                    the skip (channel offsets of one buffer), conv3x3+ReLU x 2
//   head:            conv1x1 (c -> 1) plus the input (residual), FP32.
// Backward: input gradients are convolutions with the flipped, transposed
// weights, weight gradients the transposed product, both on the tensor cores;
// the ReLU masks are applied where a gradient is produced (the convolution's
// epilogue, the pooling and upsampling kernels), which write the BF16 operand
// of the next step directly.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "internal.h"
#include "reduce.cuh"
#include "unet.h"

namespace purify {

// ------------------------------------------------------------ small kernels
static inline int eblocks(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 8192)); }

// 8 BF16 channels as floats, and back
struct Ch8 {
    float v[8];
    __device__ __forceinline__ void load(const bf16* p) {
        bf16 t[8];
        *reinterpret_cast<uint4*>(t) = *reinterpret_cast<const uint4*>(p);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = __bfloat162float(t[e]);
    }
    __device__ __forceinline__ void load(const float* p) {
        const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
    __device__ __forceinline__ void store(bf16* p) const {
        bf16 t[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] = __float2bfloat16_rn(v[e]);
        *reinterpret_cast<uint4*>(p) = *reinterpret_cast<const uint4*>(t);
    }
};
// pooled pixel and channel group of index i over [B][Ho][Wo][C / 8]
struct Pool8 {
    int c;
    size_t base;   // its 2 x 2 window's first pixel at full resolution
    __device__ __forceinline__ Pool8(int64_t i, int H, int W, int C) {
        const int G = C / 8, Ho = H / 2, Wo = W / 2;
        int r = (int)(i / G);
        c = (int)(i - (int64_t)r * G) * 8;
        const int x = r % Wo;
        r /= Wo;
        const int y = r % Ho, b = r / Ho;
        base = (size_t)(b * H + 2 * y) * W + 2 * x;
    }
    __device__ __forceinline__ size_t pix(int k, int W) const { return base + (k & 1) + (size_t)(k >> 1) * W; }
};

// All channel counts below are multiples of 8, one thread per 8 channels.
__global__ void k_maxpool_fwd(const bf16* __restrict__ in, int cs, int co, bf16* __restrict__ out, int B, int H, int W,
                              int C) {
    const int64_t n = (int64_t)B * (H / 2) * (W / 2) * (C / 8);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const Pool8 p(i, H, W, C);
        Ch8 m, t;
        m.load(in + p.base * cs + co + p.c);
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            t.load(in + p.pix(k, W) * cs + co + p.c);
#pragma unroll
            for (int e = 0; e < 8; ++e) m.v[e] = fmaxf(m.v[e], t.v[e]);
        }
        m.store(out + i * 8);
    }
}

// Through the pooling and the ReLU before it: gz[b][y][x][c] = in > 0 ?
// ((first maximum of its 2x2 window, row-major) ? gout : 0) + gadd : 0, BF16;
// gadd the skip's gradient [pixels][C].
__global__ void k_maxpool_bwd(const bf16* __restrict__ in, int cs, int co, const float* __restrict__ gout,
                              const float* __restrict__ gadd, bf16* __restrict__ gz, int B, int H, int W, int C) {
    const int64_t n = (int64_t)B * (H / 2) * (W / 2) * (C / 8);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const Pool8 p(i, H, W, C);
        Ch8 v[4], g;
        g.load(gout + i * 8);
        int arg[8] = {};
        float best[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) best[e] = -INFINITY;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k].load(in + p.pix(k, W) * cs + co + p.c);
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (v[k].v[e] > best[e]) { best[e] = v[k].v[e]; arg[e] = k; }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const size_t o = p.pix(k, W) * C + p.c;
            Ch8 r;
            r.load(gadd + o);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float t = (k == arg[e] ? g.v[e] : 0.f) + r.v[e];
                r.v[e] = v[k].v[e] > 0.f ? t : 0.f;
            }
            r.store(gz + o);
        }
    }
}

// Through the x2 upsampling and the ReLU before it: the sum of the 2x2 block
// of ghi, zero where act (channel stride C) is not positive, BF16.
__global__ void k_upsample_bwd(const float* __restrict__ ghi, const bf16* __restrict__ act, bf16* __restrict__ gz, int B,
                               int H, int W, int C) {
    const int64_t n = (int64_t)B * (H / 2) * (W / 2) * (C / 8);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const Pool8 p(i, H, W, C);
        Ch8 s, t, m;
        s.load(ghi + p.base * C + p.c);
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            t.load(ghi + p.pix(k, W) * C + p.c);
#pragma unroll
            for (int e = 0; e < 8; ++e) s.v[e] += t.v[e];
        }
        m.load(act + i * 8);
#pragma unroll
        for (int e = 0; e < 8; ++e) s.v[e] = m.v[e] > 0.f ? s.v[e] : 0.f;
        s.store(gz + i * 8);
    }
}

// out[c] += sum over pixels of w[p] v[p][c] (w = 1 when null; v has channel
// stride cs), and with w also wsum += sum of w[p]: the bias gradients, and the
// head's weight and bias gradient. A thread keeps 8 channels of every
// (blockDim / (C / 8))-th pixel of the block's chunk; the block's sums are
// combined in shared memory, one atomic per channel and block.
__global__ void __launch_bounds__(256) k_colsum(const bf16* __restrict__ v, int cs, int C, int64_t P, int pch,
                                                const bf16* __restrict__ w, float* __restrict__ out,
                                                float* __restrict__ wsum) {
    __shared__ float sh[256][9];
    const int G = C / 8, lanes = blockDim.x / G;
    const int g = threadIdx.x % G, l = threadIdx.x / G;
    float acc[9] = {};
    if (l < lanes) {
        const int64_t p1 = min(P, ((int64_t)blockIdx.x + 1) * pch);
        for (int64_t p = (int64_t)blockIdx.x * pch + l; p < p1; p += lanes) {
            Ch8 t;
            t.load(v + p * cs + g * 8);
            const float s = w ? __bfloat162float(w[p]) : 1.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = fmaf(s, t.v[e], acc[e]);
            acc[8] += s;
        }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) sh[threadIdx.x][e] = acc[e];
    __syncthreads();
    for (int c = threadIdx.x; c <= C; c += blockDim.x) {
        const int gg = c < C ? c / 8 : 0, e = c < C ? c % 8 : 8;
        if (c == C && !wsum) continue;
        float s = 0.f;
        for (int k = 0; k < lanes; ++k) s += sh[k * G + gg][e];
        atomicAdd(c < C ? out + c : wsum, s);
    }
}

// Weight gradient of a 3 x 3 convolution of one input channel: dW[co][tap] +=
// sum over pixels of gz[p][co] x[p + tap]. A thread owns one output channel and
// walks pixels of a row with the 3 x 3 window of x in registers.
__global__ void __launch_bounds__(256) k_dw_point(const bf16* __restrict__ gz, int Cout, const bf16* __restrict__ x,
                                                  int B, int H, int W, int seg, float* __restrict__ dW) {
    __shared__ float sh[256][9];
    const int lanes = blockDim.x / Cout, co = threadIdx.x % Cout, l = threadIdx.x / Cout;
    const int per_row = (W + seg - 1) / seg;
    const int64_t nseg = (int64_t)B * H * per_row;
    float acc[9] = {};
    if (l < lanes) {
        for (int64_t s = (int64_t)blockIdx.x * lanes + l; s < nseg; s += (int64_t)gridDim.x * lanes) {
            const int r = (int)(s / per_row), x0 = (int)(s - (int64_t)r * per_row) * seg, x1 = min(W, x0 + seg);
            const int b = r / H, y = r - b * H;
            auto at = [&](int dy, int xx) -> float {
                const int yy = y + dy;
                return yy >= 0 && yy < H && xx >= 0 && xx < W ? __bfloat162float(x[((size_t)b * H + yy) * W + xx]) : 0.f;
            };
            float w0[3], w1[3], w2[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                w0[d] = at(d - 1, x0 - 1);
                w1[d] = at(d - 1, x0);
            }
            for (int xx = x0; xx < x1; ++xx) {
#pragma unroll
                for (int d = 0; d < 3; ++d) w2[d] = at(d - 1, xx + 1);
                const float g = __bfloat162float(gz[(((size_t)b * H + y) * W + xx) * Cout + co]);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    acc[3 * d] = fmaf(g, w0[d], acc[3 * d]);
                    acc[3 * d + 1] = fmaf(g, w1[d], acc[3 * d + 1]);
                    acc[3 * d + 2] = fmaf(g, w2[d], acc[3 * d + 2]);
                    w0[d] = w1[d];
                    w1[d] = w2[d];
                }
            }
        }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) sh[threadIdx.x][e] = acc[e];
    __syncthreads();
    for (int i = threadIdx.x; i < 9 * Cout; i += blockDim.x) {
        const int c = i / 9, e = i - c * 9;
        float s = 0.f;
        for (int k = 0; k < lanes; ++k) s += sh[k * Cout + c][e];
        atomicAdd(&dW[i], s);
    }
}

// FP32 weights [Cout][k][k][Cin] -> flipped, transposed BF16
// [k][k][Cb / 8][Nb][8]: W'[ci][ky][kx][co] = W[co][k-1-ky][k-1-kx][ci] (zero
// padded)
__global__ void k_pack_weights_bwd(const float* __restrict__ w, bf16* __restrict__ wp, int Cout, int k, int Cin, int Nb,
                                   int Cb) {
    const int64_t n = (int64_t)Nb * k * k * Cb;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / 8;
        const int ci = (int)(r % Nb), g = (int)(r / Nb), tap = g / (Cb / 8);
        const int co = (g - tap * (Cb / 8)) * 8 + (int)(i % 8);
        int ky = tap / k, kx = tap % k;
        int ftap = (k - 1 - ky) * k + (k - 1 - kx);
        float v = (ci < Cin && co < Cout) ? w[((int64_t)co * k * k + ftap) * Cin + ci] : 0.f;
        wp[i] = __float2bfloat16_rn(v);
    }
}

// loss = mean (pred - t)^2 to *out (FP64, fixed order), g = 2 (pred - t) / n in BF16
__global__ void k_mse(const float* __restrict__ pred, const float* __restrict__ t, bf16* __restrict__ g, int64_t n,
                      double* part, unsigned* counter, double* out) {
    float acc = 0.f;
    const float s = 2.f / (float)n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float d = pred[i] - t[i];
        acc += d * d;
        g[i] = __float2bfloat16_rn(s * d);
    }
    double b = block_sum((double)acc);
    if (threadIdx.x == 0) part[blockIdx.x] = b;
    if (arrive_last(counter)) {
        double tot = ordered_sum(part, gridDim.x);
        if (threadIdx.x == 0) {
            *out = tot / (double)n;
            *counter = 0;
        }
    }
}

// Adam (Kingma & Ba 2015) with bias correction
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int64_t n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        float gi = g[i];
        float mi = b1 * m[i] + (1.f - b1) * gi;
        float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// ------------------------------------------------------------------ network
struct UnetLayer {
    std::string name;
    int cout, k, cin;
    int64_t woff, boff;      // into the flat parameter vector
    int Npad, Cinp, Nb, Cb;  // packed forward / backward weight shapes
    DevBuf wf, wb;           // packed BF16 weights
};

struct Unet {
    int H, W, L, base, maxB;
    cudaStream_t st;
    std::vector<UnetLayer> layers;
    int64_t nparams = 0;
    int64_t step = 0;
    DevBuf params, grads, m, v;
    // activations (BF16)
    DevBuf xbf;                                 // [B][H][W][1]
    std::vector<DevBuf> a, cat, pool, da, dbb;  // per level
    DevBuf bA, bB;
    DevBuf pred;                                // FP32 [B][H][W]
    // gradients (FP32) and BF16 staging
    std::vector<DevBuf> gcat;
    DevBuf g1, gz, gz2;
    DevBuf red_part, red_ctr, loss, err;
    int ch(int l) const { return base << l; }
    int64_t pix(int l, int B) const { return (int64_t)B * (H >> l) * (W >> l); }
    UnetLayer& layer(const std::string& n) {
        for (auto& x : layers) if (x.name == n) return x;
        throw Error{PURIFY_EINVAL, "unknown layer " + n};
    }
};

static void build_layers(Unet& u) {
    int cin = 1;
    auto add = [&](const std::string& n, int cout, int k, int ci) {
        UnetLayer l;
        l.name = n;
        l.cout = cout;
        l.k = k;
        l.cin = ci;
        l.woff = u.nparams;
        u.nparams += (int64_t)cout * k * k * ci;
        l.boff = u.nparams;
        u.nparams += cout;
        l.Npad = std::max(16, round16(cout));
        l.Cinp = round16(ci);
        l.Nb = std::max(16, round16(ci));
        l.Cb = round16(cout);
        u.layers.push_back(std::move(l));
    };
    for (int l = 0; l < u.L - 1; ++l) {
        int c = u.ch(l);
        add("e" + std::to_string(l) + "a", c, 3, cin);
        add("e" + std::to_string(l) + "b", c, 3, c);
        cin = c;
    }
    int cb = u.ch(u.L - 1);
    add("ba", cb, 3, cin);
    add("bb", cb, 3, cb);
    for (int l = u.L - 2; l >= 0; --l) {
        int c = u.ch(l);
        add("d" + std::to_string(l) + "u", c, 3, 2 * c);
        add("d" + std::to_string(l) + "a", c, 3, 2 * c);
        add("d" + std::to_string(l) + "b", c, 3, c);
    }
    add("head", 1, 1, u.base);
}

static void pack_all(Unet& u) {
    const float* P = u.params.as<float>();
    for (auto& l : u.layers) {
        int64_t nf = (int64_t)l.Npad * l.k * l.k * l.Cinp, nb = (int64_t)l.Nb * l.k * l.k * l.Cb;
        k_pack_weights<<<eblocks(nf), 256, 0, u.st>>>(P + l.woff, l.wf.as<bf16>(), l.cout, l.k, l.cin, l.Npad, l.Cinp);
        k_pack_weights_bwd<<<eblocks(nb), 256, 0, u.st>>>(P + l.woff, l.wb.as<bf16>(), l.cout, l.k, l.cin, l.Nb, l.Cb);
    }
    PURIFY_CUDA(cudaGetLastError());
    add_launches(2 * (int64_t)u.layers.size());
}

Unet* unet_create(int H, int W, int L, int base, int maxB, uint64_t seed, cudaStream_t st) {
    PURIFY_REQUIRE(L >= 2 && L <= 6 && base >= 8 && base % 8 == 0 && (base << (L - 1)) <= 256,
                   "unet: levels in [2, 6], base multiple of 8 with base * 2^(levels-1) <= 256");
    PURIFY_REQUIRE(H % (1 << (L - 1)) == 0 && W % (1 << (L - 1)) == 0 && H >= 8 && W >= 8,
                   "unet: H and W must be divisible by 2^(levels-1)");
    PURIFY_REQUIRE(maxB >= 1, "unet: max batch >= 1");
    Unet* u = new Unet();
    try {
        u->H = H; u->W = W; u->L = L; u->base = base; u->maxB = maxB; u->st = st;
        build_layers(*u);
        // He-normal initial weights from a seeded generator, zero biases
        std::vector<float> p(u->nparams, 0.f);
        uint64_t s = seed * 0x9E3779B97F4A7C15ull + 1;
        auto uni = [&]() {
            s ^= s << 13; s ^= s >> 7; s ^= s << 17;
            return ((double)(s >> 11) + 0.5) * (1.0 / 9007199254740992.0);
        };
        for (auto& l : u->layers) {
            double stdv = std::sqrt(2.0 / (l.k * l.k * l.cin));
            int64_t nw = (int64_t)l.cout * l.k * l.k * l.cin;
            for (int64_t i = 0; i < nw; ++i) {
                double r1 = uni(), r2 = uni();
                p[l.woff + i] = (float)(stdv * std::sqrt(-2.0 * std::log(r1)) * std::cos(6.283185307179586 * r2));
            }
            l.wf.alloc(sizeof(bf16) * (size_t)l.Npad * l.k * l.k * l.Cinp);
            l.wb.alloc(sizeof(bf16) * (size_t)l.Nb * l.k * l.k * l.Cb);
        }
        u->params.alloc(sizeof(float) * u->nparams);
        u->grads.alloc(sizeof(float) * u->nparams);
        u->m.alloc(sizeof(float) * u->nparams);
        u->v.alloc(sizeof(float) * u->nparams);
        PURIFY_CUDA(cudaMemcpy(u->params.p, p.data(), sizeof(float) * u->nparams, cudaMemcpyHostToDevice));
        PURIFY_CUDA(cudaMemset(u->m.p, 0, u->m.bytes));
        PURIFY_CUDA(cudaMemset(u->v.p, 0, u->v.bytes));
        // buffers
        u->xbf.alloc(sizeof(bf16) * u->pix(0, maxB));
        u->a.resize(L); u->cat.resize(L); u->pool.resize(L); u->da.resize(L); u->dbb.resize(L); u->gcat.resize(L);
        for (int l = 0; l < L - 1; ++l) {
            int64_t P = u->pix(l, maxB);
            int c = u->ch(l);
            u->a[l].alloc(sizeof(bf16) * P * c);
            u->cat[l].alloc(sizeof(bf16) * P * 2 * c);
            u->pool[l].alloc(sizeof(bf16) * u->pix(l + 1, maxB) * c);
            u->da[l].alloc(sizeof(bf16) * P * c);
            u->dbb[l].alloc(sizeof(bf16) * P * c);
            u->gcat[l].alloc(sizeof(float) * P * c);
        }
        int64_t Pb = u->pix(L - 1, maxB);
        u->bA.alloc(sizeof(bf16) * Pb * u->ch(L - 1));
        u->bB.alloc(sizeof(bf16) * Pb * u->ch(L - 1));
        u->pred.alloc(sizeof(float) * u->pix(0, maxB));
        int64_t gmax = 0;
        for (int l = 0; l < L; ++l) gmax = std::max(gmax, u->pix(l, maxB) * 2 * u->ch(l));
        u->g1.alloc(sizeof(float) * gmax);
        u->gz.alloc(sizeof(bf16) * gmax);
        u->gz2.alloc(sizeof(bf16) * gmax);
        u->red_part.alloc(sizeof(double) * 8192);
        u->red_ctr.alloc(sizeof(unsigned) * 4);
        u->loss.alloc(sizeof(double));
        u->err.alloc(sizeof(int));
        PURIFY_CUDA(cudaMemset(u->red_ctr.p, 0, u->red_ctr.bytes));
        PURIFY_CUDA(cudaMemset(u->err.p, 0, sizeof(int)));
        settle_uploads();
        pack_all(*u);
        PURIFY_CUDA(cudaStreamSynchronize(st));
    } catch (...) {
        delete u;
        throw;
    }
    return u;
}

void unet_destroy(Unet* u) {
    if (!u) return;
    cudaStreamSynchronize(u->st);
    delete u;
}

static ConvArgs conv_args(Unet& u, UnetLayer& l, bool backward) {
    ConvArgs a{};
    a.k = l.k;
    if (!backward) {
        a.w = l.wf.as<bf16>(); a.Cinp = l.Cinp; a.Npad = l.Npad; a.Cout = l.cout; a.Cin = l.cin;
        a.bias = u.params.as<float>() + l.boff;
    } else {
        a.w = l.wb.as<bf16>(); a.Cinp = l.Cb; a.Npad = l.Nb; a.Cout = l.cin; a.Cin = l.cout;
        a.bias = nullptr;
    }
    a.err = u.err.as<int>();
    return a;
}

// conv layer forward: input (buffer, channel stride, offset, resolution level, upsample) -> BF16 output slice
static void fwd_conv(Unet& u, const std::string& name, int B, const bf16* in, int in_cs, int in_co, int lev, int up,
                     bf16* out, int out_cs, int out_co) {
    UnetLayer& l = u.layer(name);
    ConvArgs a = conv_args(u, l, false);
    a.in = in; a.in_cs = in_cs; a.in_co = in_co; a.up = up;
    a.B = B; a.H = u.H >> lev; a.W = u.W >> lev;
    a.relu = 1;
    a.out = out; a.out_cs = out_cs; a.out_co = out_co;
    conv_tc_launch(a, u.st);
}

void unet_forward(Unet& u, const float* x, int B, float* out) {
    const int L = u.L;
    const int64_t P0 = u.pix(0, B);
    k_f32_to_bf16<<<eblocks(P0), 256, 0, u.st>>>(x, u.xbf.as<bf16>(), P0);
    add_launches(1);
    const bf16* in = u.xbf.as<bf16>();
    int in_cs = 1;
    for (int l = 0; l < L - 1; ++l) {
        int c = u.ch(l);
        std::string s = std::to_string(l);
        fwd_conv(u, "e" + s + "a", B, in, in_cs, 0, l, 0, u.a[l].as<bf16>(), c, 0);
        fwd_conv(u, "e" + s + "b", B, u.a[l].as<bf16>(), c, 0, l, 0, u.cat[l].as<bf16>(), 2 * c, 0);
        int64_t n = u.pix(l + 1, B) * c / 8;
        k_maxpool_fwd<<<eblocks(n), 256, 0, u.st>>>(u.cat[l].as<bf16>(), 2 * c, 0, u.pool[l].as<bf16>(), B, u.H >> l,
                                                   u.W >> l, c);
        add_launches(1);
        in = u.pool[l].as<bf16>();
        in_cs = c;
    }
    int cb = u.ch(L - 1);
    fwd_conv(u, "ba", B, in, in_cs, 0, L - 1, 0, u.bA.as<bf16>(), cb, 0);
    fwd_conv(u, "bb", B, u.bA.as<bf16>(), cb, 0, L - 1, 0, u.bB.as<bf16>(), cb, 0);
    const bf16* low = u.bB.as<bf16>();
    for (int l = L - 2; l >= 0; --l) {
        int c = u.ch(l);
        std::string s = std::to_string(l);
        fwd_conv(u, "d" + s + "u", B, low, 2 * c, 0, l, 1, u.cat[l].as<bf16>(), 2 * c, c);
        fwd_conv(u, "d" + s + "a", B, u.cat[l].as<bf16>(), 2 * c, 0, l, 0, u.da[l].as<bf16>(), c, 0);
        fwd_conv(u, "d" + s + "b", B, u.da[l].as<bf16>(), c, 0, l, 0, u.dbb[l].as<bf16>(), c, 0);
        low = u.dbb[l].as<bf16>();
    }
    UnetLayer& h = u.layer("head");
    ConvArgs a = conv_args(u, h, false);
    a.in = u.dbb[0].as<bf16>(); a.in_cs = u.base; a.in_co = 0; a.up = 0;
    a.B = B; a.H = u.H; a.W = u.W; a.relu = 0;
    a.out = nullptr; a.out_f32 = out ? out : u.pred.as<float>(); a.residual = x;
    conv_tc_launch(a, u.st);
}

// Where an input gradient goes: channels below f32_ch (all with out null) to
// f32 [P][f32_ch], the others masked by the activation they belong to (its
// ReLU) to BF16 `out` [P][cin - f32_ch].
struct GradOut {
    float* f32 = nullptr;
    int f32_ch = 0;
    bf16* out = nullptr;
    const bf16* act = nullptr;
    int act_cs = 0, act_co = 0;
};

// input gradient of a conv layer from gz (BF16 [P][cout]) at level lev
static void bwd_dx(Unet& u, UnetLayer& l, int B, int lev, const bf16* gz, const GradOut& g) {
    ConvArgs a = conv_args(u, l, true);
    a.in = gz; a.in_cs = l.cout; a.in_co = 0; a.up = 0;
    a.B = B; a.H = u.H >> lev; a.W = u.W >> lev; a.relu = 0;
    a.out_f32 = g.f32; a.f32_ch = g.f32_ch; a.residual = nullptr;
    a.out = g.out; a.out_cs = l.cin - g.f32_ch; a.out_co = 0; a.bf_from = g.f32_ch;
    a.mask = g.act; a.mask_cs = g.act_cs; a.mask_co = g.act_co;
    conv_tc_launch(a, u.st);
}

static void colsum(Unet& u, const bf16* v, int cs, int C, int64_t P, const bf16* w, float* out, float* wsum) {
    const int pch = (int)std::max<int64_t>(64, (P + 152 * 4 - 1) / (152 * 4));
    k_colsum<<<(int)((P + pch - 1) / pch), 256, 0, u.st>>>(v, cs, C, P, pch, w, out, wsum);
    PURIFY_CUDA(cudaGetLastError());
    add_launches(1);
}

// weight and bias gradients of a layer with input x (channel stride xcs)
static void bwd_dw(Unet& u, UnetLayer& l, int B, int lev, const bf16* gz, const bf16* x, int xcs, int up) {
    const int H = u.H >> lev, W = u.W >> lev;
    const int64_t P = (int64_t)B * H * W;
    float* dW = u.grads.as<float>() + l.woff;
    float* db = u.grads.as<float>() + l.boff;
    if (l.cout == 1 && l.k == 1) {
        // the head: both gradients in one pass
        colsum(u, x, xcs, l.cin, P, gz, dW, db);
        return;
    }
    if (l.cin == 1 && l.k == 3 && !up && xcs == 1) {
        k_dw_point<<<152 * 4, 256, 0, u.st>>>(gz, l.cout, x, B, H, W, 32, dW);
        PURIFY_CUDA(cudaGetLastError());
        add_launches(1);
    } else {
        PURIFY_REQUIRE(dw_tc_ok(l.cout, l.cin, xcs, 0), "unet: layer channels must be multiples of 8");
        dw_tc_launch(gz, l.cout, x, xcs, 0, l.cin, B, H, W, up, l.k, dW, u.err.as<int>(), u.st);
    }
    colsum(u, gz, l.cout, l.cout, P, nullptr, db, nullptr);
}

// forward + backward; gradients in u.grads, loss in u.loss (device)
void unet_gradients(Unet& u, const float* x, const float* target, int B) {
    PURIFY_REQUIRE(B >= 1 && B <= u.maxB, "unet: batch larger than the network was created for");
    const int L = u.L;
    unet_forward(u, x, B, nullptr);
    PURIFY_CUDA(cudaMemsetAsync(u.grads.p, 0, u.grads.bytes, u.st));
    const int64_t P0 = u.pix(0, B);
    // gz: gradient with respect to the current layer's pre-activation (BF16
    // [P][cout]); each step writes the next one's into the other buffer
    bf16 *gz = u.gz.as<bf16>(), *gn = u.gz2.as<bf16>();
    float* const t = u.g1.as<float>();
    auto masked = [&](const bf16* act, int cs, int co) {
        GradOut g;
        g.out = gn;
        g.act = act;
        g.act_cs = cs;
        g.act_co = co;
        return g;
    };
    GradOut plain;   // all channels in FP32
    plain.f32 = t;
    // head (1x1, no ReLU): gz = the loss gradient
    k_mse<<<256, 256, 0, u.st>>>(u.pred.as<float>(), target, gz, P0, u.red_part.as<double>(),
                                 u.red_ctr.as<unsigned>(), u.loss.as<double>());
    add_launches(1);
    UnetLayer& head = u.layer("head");
    bwd_dw(u, head, B, 0, gz, u.dbb[0].as<bf16>(), u.base, 0);
    bwd_dx(u, head, B, 0, gz, masked(u.dbb[0].as<bf16>(), u.base, 0));
    std::swap(gz, gn);
    for (int l = 0; l < L - 1; ++l) {
        const int c = u.ch(l);
        std::string s = std::to_string(l);
        UnetLayer& lb = u.layer("d" + s + "b");
        bwd_dw(u, lb, B, l, gz, u.da[l].as<bf16>(), c, 0);
        bwd_dx(u, lb, B, l, gz, masked(u.da[l].as<bf16>(), c, 0));
        std::swap(gz, gn);
        // the concatenation: channels [0, c) the skip (kept for the encoder),
        // [c, 2c) the up branch
        UnetLayer& la = u.layer("d" + s + "a");
        bwd_dw(u, la, B, l, gz, u.cat[l].as<bf16>(), 2 * c, 0);
        GradOut both = masked(u.cat[l].as<bf16>(), 2 * c, c);
        both.f32 = u.gcat[l].as<float>();
        both.f32_ch = c;
        bwd_dx(u, la, B, l, gz, both);
        std::swap(gz, gn);
        UnetLayer& lu = u.layer("d" + s + "u");
        const bf16* low = (l == L - 2) ? u.bB.as<bf16>() : u.dbb[l + 1].as<bf16>();
        bwd_dw(u, lu, B, l, gz, low, 2 * c, 1);
        bwd_dx(u, lu, B, l, gz, plain);   // [P][2c] at level l
        const int64_t nlo = u.pix(l + 1, B) * 2 * c / 8;
        k_upsample_bwd<<<eblocks(nlo), 256, 0, u.st>>>(t, low, gn, B, u.H >> l, u.W >> l, 2 * c);
        add_launches(1);
        std::swap(gz, gn);
    }
    const int cb = u.ch(L - 1);
    UnetLayer& lbb = u.layer("bb");
    bwd_dw(u, lbb, B, L - 1, gz, u.bA.as<bf16>(), cb, 0);
    bwd_dx(u, lbb, B, L - 1, gz, masked(u.bA.as<bf16>(), cb, 0));
    std::swap(gz, gn);
    UnetLayer& lba = u.layer("ba");
    bwd_dw(u, lba, B, L - 1, gz, u.pool[L - 2].as<bf16>(), u.ch(L - 2), 0);
    bwd_dx(u, lba, B, L - 1, gz, plain);   // gradient of pool[L-2]
    for (int l = L - 2; l >= 0; --l) {
        const int c = u.ch(l);
        std::string s = std::to_string(l);
        // through the max pooling, plus the skip gradient
        const int64_t npool = u.pix(l + 1, B) * c / 8;
        k_maxpool_bwd<<<eblocks(npool), 256, 0, u.st>>>(u.cat[l].as<bf16>(), 2 * c, 0, t, u.gcat[l].as<float>(), gz, B,
                                                        u.H >> l, u.W >> l, c);
        add_launches(1);
        UnetLayer& lb = u.layer("e" + s + "b");
        bwd_dw(u, lb, B, l, gz, u.a[l].as<bf16>(), c, 0);
        bwd_dx(u, lb, B, l, gz, masked(u.a[l].as<bf16>(), c, 0));
        std::swap(gz, gn);
        UnetLayer& la = u.layer("e" + s + "a");
        const bf16* xin = l == 0 ? u.xbf.as<bf16>() : u.pool[l - 1].as<bf16>();
        const int xcs = l == 0 ? 1 : u.ch(l - 1);
        bwd_dw(u, la, B, l, gz, xin, xcs, 0);
        if (l > 0) bwd_dx(u, la, B, l, gz, plain);
    }
}

double unet_read_loss(Unet& u) {
    double v = 0;
    PURIFY_CUDA(cudaMemcpyAsync(&v, u.loss.p, sizeof(double), cudaMemcpyDeviceToHost, u.st));
    int e = 0;
    PURIFY_CUDA(cudaMemcpyAsync(&e, u.err.p, sizeof(int), cudaMemcpyDeviceToHost, u.st));
    PURIFY_CUDA(cudaStreamSynchronize(u.st));
    if (e) throw Error{PURIFY_ETIMEOUT, "tensor-core convolution: a bounded wait gave up"};
    return v;
}

void unet_adam(Unet& u, float lr) {
    u.step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - std::pow(b1, (float)u.step), c2 = 1.f - std::pow(b2, (float)u.step);
    k_adam<<<eblocks(u.nparams), 256, 0, u.st>>>(u.params.as<float>(), u.grads.as<float>(), u.m.as<float>(),
                                                 u.v.as<float>(), u.nparams, lr, b1, b2, 1e-8f, c1, c2);
    add_launches(1);
    pack_all(u);
}

void unet_set_params(Unet& u, const float* p) {
    PURIFY_CUDA(cudaMemcpyAsync(u.params.p, p, sizeof(float) * u.nparams, cudaMemcpyDefault, u.st));
    pack_all(u);
    PURIFY_CUDA(cudaStreamSynchronize(u.st));
}

void unet_get(Unet& u, int what, float* out) {
    const DevBuf& b = what == 0 ? u.params : u.grads;
    PURIFY_CUDA(cudaMemcpyAsync(out, b.p, sizeof(float) * u.nparams, cudaMemcpyDefault, u.st));
    PURIFY_CUDA(cudaStreamSynchronize(u.st));
}

int64_t unet_nparams(Unet& u) { return u.nparams; }

}  // namespace purify
