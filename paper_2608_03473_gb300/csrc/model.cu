// model.cu -- the entry-context model of the speculative path: a byte-window
// network that reads the 64 bytes around a chunk start and scores every
// context (BOUNDARY or a DFA state), trained on the true contexts that the
// enumerative path resolves.  The lexer stays exact whatever it predicts: a
// wrong guess only costs a rescan.
//
//   h0[t]   = emb[x_t]                               x = w[p - 32, p + 32), pad byte 256 outside
//   a[t,f]  = bc[f] + sum_{k<5,d<8} Wc[f,k,d] h0[t+k-2,d]   (zero outside the window)
//   m[u,f]  = max_{t=4u..4u+3} relu(a[t,f])          (the first maximum takes the gradient)
//   h1      = relu(m W1 + b1),  z = h1 W2 + b2       W1: 512 x H, W2: H x C (C = states + 1)
//   loss    = mean over the batch of -log softmax(z)[y]
// 32 filters, H = 64 and the 211 contexts of the refused C-like set give
// 49 915 parameters.  Every product reads BF16 weights and accumulates in
// FP32 (activations stay FP32); FP32 master weights are updated by AdamW
// (decoupled weight decay on the weight matrices).  Inference takes the
// argmax of z over the candidate contexts of the byte before p.  The products
// are small (a few hundred MFLOP per 512 MiB of input) and run on the CUDA
// cores.

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "internal.h"
#include "runtime.h"

namespace lx {
namespace {

constexpr uint32_t MW = 64;          // window bytes
constexpr uint32_t MD = 8;           // embedding width
constexpr uint32_t MROWS = 257;      // 256 byte values + padding
constexpr uint32_t MF = 32;          // convolution filters
constexpr uint32_t MK = 5;           // filter width
constexpr uint32_t MPOOL = 4;        // max-pool width (and stride)
constexpr uint32_t MU = MW / MPOOL;  // pooled positions
constexpr uint32_t MIN_ = MU * MF;   // MLP input width (512)
constexpr int GT = 16;               // GEMM tile
constexpr uint32_t PRED_BATCH = 24576;
constexpr float WEIGHT_DECAY = 1e-2f;   // AdamW, on Wc, W1 and W2

}  // namespace
}  // namespace lx

struct lx_model {
    uint32_t C = 0, H = 0;
    uint64_t step = 0;
    // parameters in one FP32 block: emb | Wc | bc | W1 | b1 | W2 | b2, and Adam moments
    float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
    __nv_bfloat16 *w16 = nullptr;   // the BF16 weights every product reads
    size_t n_params = 0;
    size_t o_emb = 0, o_wc = 0, o_bc = 0, o_w1 = 0, o_b1 = 0, o_w2 = 0, o_b2 = 0;
    uint8_t *arg = nullptr;         // per (window, pooled position, filter): argmax | relu-active << 2
    size_t arg_bytes = 0;
    // activations for a batch, and windows for inference batches
    float *act = nullptr;
    size_t act_floats = 0;
    uint16_t *win = nullptr;
    bool mg_ready = false;          // k_mlp_grad may use its shared memory
    float *h_g = nullptr;           // pinned: the gradient and the loss on their way to the caller
    int device = -1;
};

namespace lx {
namespace {

__device__ __forceinline__ uint32_t window_byte(const uint8_t *in, uint64_t n, uint64_t p, uint32_t k)
{
    const int64_t q = (int64_t)p - (int64_t)(MW / 2) + (int64_t)k;
    return (q >= 0 && (uint64_t)q < n) ? (uint32_t)in[q] : 256u;
}

__device__ __forceinline__ float to_f(float x) { return x; }
__device__ __forceinline__ float to_f(__nv_bfloat16 x) { return __bfloat162float(x); }

// Convolution, ReLU and max pooling, one warp per window, lane = filter: the
// filter's 40 weights stay in registers, the window's embedded bytes in shared
// memory (two zero rows on either side), and each of them is read once per
// four outputs: 65 us per 16 384 windows (1.6 times its multiply-adds).  The convolution outputs t = 4u .. 4u+3 give the first maximum
// of their ReLU into m[b, u * MF + f], and its index (with whether it was
// positive) for the backward pass.  One thread per (window, u, f), reading
// embedding and weights from global memory for each, took 258 us per 16 384
// windows and 11.6 us for 512.
constexpr int CP_WARPS = 8;
constexpr uint32_t MPAD = MK / 2, MHR = MW + 2 * MPAD;   // rows of a window in shared memory

__device__ __forceinline__ void embed_row(const __nv_bfloat16 *emb, uint32_t byte, float (&v)[MD])
{
    const uint4 e = __ldg(reinterpret_cast<const uint4 *>(emb + (size_t)byte * MD));   // MD bf16
    const uint32_t p[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
    for (uint32_t i = 0; i < 4; i++) {
        v[2 * i] = __uint_as_float(p[i] << 16);
        v[2 * i + 1] = __uint_as_float(p[i] & 0xFFFF0000u);
    }
}

__device__ __forceinline__ bool nonfinite(float x) { return (__float_as_uint(x) & 0x7F800000u) == 0x7F800000u; }

// Returns whether the lane met an infinity or a NaN.
__device__ __forceinline__ bool load_window(const uint16_t *w, const __nv_bfloat16 *emb, float (*h)[MD], uint32_t lane)
{
    bool bad = false;
    for (uint32_t t = lane; t < MHR; t += 32) {
        float v[MD] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (t >= MPAD && t < MPAD + MW) embed_row(emb, w[t - MPAD], v);
        *reinterpret_cast<float4 *>(&h[t][0]) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4 *>(&h[t][4]) = make_float4(v[4], v[5], v[6], v[7]);
#pragma unroll
        for (uint32_t d = 0; d < MD; d++) bad |= nonfinite(v[d]);
    }
    return bad;
}

__global__ void __launch_bounds__(32 * CP_WARPS) k_conv_pool(const uint16_t *win, uint32_t B, const __nv_bfloat16 *emb,
                                                             const __nv_bfloat16 *wc, const __nv_bfloat16 *bc, float *mo,
                                                             uint8_t *arg)
{
    __shared__ __align__(16) float hs[CP_WARPS][MHR][MD];
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float w[MK][MD];
#pragma unroll
    for (uint32_t k = 0; k < MK; k++)
#pragma unroll
        for (uint32_t d = 0; d < MD; d++) w[k][d] = to_f(wc[((size_t)lane * MK + k) * MD + d]);
    const float bias = to_f(bc[lane]);
    float(*h)[MD] = hs[wid];
    for (uint32_t b = blockIdx.x * CP_WARPS + wid; b < B; b += gridDim.x * CP_WARPS) {
        __syncwarp();
        load_window(win + (size_t)b * MW, emb, h, lane);
        __syncwarp();
#pragma unroll 1
        for (uint32_t u = 0; u < MU; u++) {
            float a[MPOOL] = {bias, bias, bias, bias};
#pragma unroll
            for (uint32_t r = 0; r < MPOOL + MK - 1; r++) {   // row t = 4u + r - 2; every output sums k, d in order
                const float4 x = *reinterpret_cast<const float4 *>(&h[MPOOL * u + r][0]);
                const float4 y = *reinterpret_cast<const float4 *>(&h[MPOOL * u + r][4]);
                const float v[MD] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                for (uint32_t j = 0; j < MPOOL; j++)
                    if (r >= j && r - j < MK) {
#pragma unroll
                        for (uint32_t d = 0; d < MD; d++) a[j] = fmaf(w[r - j][d], v[d], a[j]);
                    }
            }
            float best = -1.0f;
            uint32_t bj = 0, pos = 0;
#pragma unroll
            for (uint32_t j = 0; j < MPOOL; j++) {
                const float rr = a[j] > 0.0f ? a[j] : 0.0f;
                if (rr > best) {
                    best = rr;
                    bj = j;
                    pos = a[j] > 0.0f ? 1u : 0u;
                }
            }
            const size_t i = (size_t)b * MIN_ + u * MF + lane;
            mo[i] = best;
            if (arg) arg[i] = (uint8_t)(bj | (pos << 2));
        }
    }
}

// Two float products at once, each as fmaf rounds.
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    return (unsigned long long)__float_as_uint(hi) << 32 | __float_as_uint(lo);
}

// k_conv_pool for prediction: a warp takes two windows at a time, each product
// of a filter with both in one instruction (their rows interleaved in shared
// memory), every output's sum in the same order.  24 576 windows 82 -> 73 us
// (their products alone: 54).  A training batch's few windows stay one a warp.
__global__ void __launch_bounds__(32 * CP_WARPS) k_conv_pool2(const uint16_t *win, uint32_t B, const __nv_bfloat16 *emb,
                                                              const __nv_bfloat16 *wc, const __nv_bfloat16 *bc, float *mo)
{
    __shared__ __align__(16) unsigned long long hs[CP_WARPS][MHR][MD];
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long w[MK][MD];
#pragma unroll
    for (uint32_t k = 0; k < MK; k++)
#pragma unroll
        for (uint32_t d = 0; d < MD; d++) {
            const float x = to_f(wc[((size_t)lane * MK + k) * MD + d]);
            w[k][d] = pack2(x, x);
        }
    const float bias = to_f(bc[lane]);
    unsigned long long(*h)[MD] = hs[wid];
    for (uint32_t b = 2 * (blockIdx.x * CP_WARPS + wid); b < B; b += 2 * gridDim.x * CP_WARPS) {
        const uint16_t *w0 = win + (size_t)b * MW, *w1 = b + 1 < B ? w0 + MW : w0;
        __syncwarp();
        for (uint32_t t = lane; t < MHR; t += 32) {
            float v[MD] = {0, 0, 0, 0, 0, 0, 0, 0}, x[MD] = {0, 0, 0, 0, 0, 0, 0, 0};
            if (t >= MPAD && t < MPAD + MW) {
                embed_row(emb, w0[t - MPAD], v);
                embed_row(emb, w1[t - MPAD], x);
            }
#pragma unroll
            for (uint32_t d = 0; d < MD; d += 2)
                *reinterpret_cast<float4 *>(&h[t][d]) = make_float4(v[d], x[d], v[d + 1], x[d + 1]);
        }
        __syncwarp();
#pragma unroll 1
        for (uint32_t u = 0; u < MU; u++) {
            unsigned long long a[MPOOL];
#pragma unroll
            for (uint32_t j = 0; j < MPOOL; j++) a[j] = pack2(bias, bias);
#pragma unroll
            for (uint32_t r = 0; r < MPOOL + MK - 1; r++) {   // row t = 4u + r - 2; every output sums k, d in order
                unsigned long long v[MD];
#pragma unroll
                for (uint32_t d = 0; d < MD; d += 2) {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&h[MPOOL * u + r][d]);
                    v[d] = x.x, v[d + 1] = x.y;
                }
#pragma unroll
                for (uint32_t j = 0; j < MPOOL; j++)
                    if (r >= j && r - j < MK) {
#pragma unroll
                        for (uint32_t d = 0; d < MD; d++) a[j] = fma2(w[r - j][d], v[d], a[j]);
                    }
            }
            float m0 = 0.0f, m1 = 0.0f;
#pragma unroll
            for (uint32_t j = 0; j < MPOOL; j++) {
                const float x = __uint_as_float((uint32_t)a[j]), y = __uint_as_float((uint32_t)(a[j] >> 32));
                if (x > m0) m0 = x;
                if (y > m1) m1 = y;
            }
            const size_t i = (size_t)b * MIN_ + u * MF + lane;
            mo[i] = m0;
            if (b + 1 < B) mo[i + MIN_] = m1;
        }
    }
}

// ---- one training batch: k_conv_pool, k_mlp_grad, k_outer ----
// Everything of a window but the weight gradients is its own: k_mlp_grad takes
// MG windows per CTA through both dense layers, the softmax and back through
// the convolution, with the activations in shared memory.  It replaces ten
// launches (products in 16 x 16 tiles that left most SMs idle, column sums by
// one thread per column, a thread per convolution weight): a gradient of 512
// windows 391 -> 88 us, 58 of them in the three kernels, which wait on
// shared and L2 loads with 16 warps per SM.
constexpr uint32_t MG = 4;            // windows per CTA
constexpr uint32_t MG_NT = 512;       // (256 left the SM's schedulers two warps each: 46 us for 512 windows)
constexpr uint32_t MG_KP = 8;         // parts of the first product's sum
constexpr uint32_t MG_MAXH = 256, MG_MAXC = 1024;
constexpr uint32_t DA_LD = MF + 1;    // row stride of the dense pooled gradient (bank spread)

struct MgSmem {   // float offsets of k_mlp_grad's shared memory
    uint32_t mo, a1, h1, z, dh, part, total;
    __host__ __device__ MgSmem(uint32_t H, uint32_t C)
    {
        uint32_t o = 0;
        auto take = [&](uint32_t n) { const uint32_t at = o; o += (n + 3) & ~3u; return at; };
        mo = take(MIN_ * MG);      // [k][window]; later the gradient of m
        a1 = take(H * MG);
        h1 = take(H * MG);
        dh = take(H * MG);
        z = take(C * MG);          // logits, then their gradient, [c][window]
        // partial sums of the first product, or the convolution's part: windows,
        // dense pooled gradients, per-warp weight sums, weights, embedding sums
        const uint32_t conv = MG * MHR * MD + MG * MHR * DA_LD + (MG_NT / 32) * MF * MK * MD + MF * MK * MD + MROWS * MD;
        const uint32_t p1 = MG_KP * H * MG, p2 = 2 * C * MG, p = p1 > p2 ? p1 : p2;
        part = take(conv > p ? conv : p);
        total = o;
    }
};

__global__ void __launch_bounds__(MG_NT) k_mlp_grad(const uint16_t *win, const uint16_t *y, uint32_t B, uint32_t H,
                                                    uint32_t C, const float *mo, const uint8_t *arg,
                                                    const __nv_bfloat16 *emb, const __nv_bfloat16 *wc,
                                                    const __nv_bfloat16 *w1, const __nv_bfloat16 *b1,
                                                    const __nv_bfloat16 *w2, const __nv_bfloat16 *b2, float *h1o,
                                                    float *dzo, float *dho, float *gemb, float *gwc, float *gbc,
                                                    float *lossw)
{
    extern __shared__ __align__(16) float sm[];
    const MgSmem L(H, C);
    const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, b0 = blockIdx.x * MG;
    float4 *smo = reinterpret_cast<float4 *>(sm + L.mo), *sa1 = reinterpret_cast<float4 *>(sm + L.a1);
    float4 *sh1 = reinterpret_cast<float4 *>(sm + L.h1), *sdh = reinterpret_cast<float4 *>(sm + L.dh);
    float4 *sz = reinterpret_cast<float4 *>(sm + L.z), *sp = reinterpret_cast<float4 *>(sm + L.part);
    const bool ok[MG] = {b0 < B, b0 + 1 < B, b0 + 2 < B, b0 + 3 < B};
    static_assert(MG == 4, "one float4 per (feature, four windows)");
    for (uint32_t i = tid; i < MIN_; i += MG_NT) {
        float4 v = make_float4(0, 0, 0, 0);
        if (ok[0]) v.x = mo[(size_t)(b0 + 0) * MIN_ + i];
        if (ok[1]) v.y = mo[(size_t)(b0 + 1) * MIN_ + i];
        if (ok[2]) v.z = mo[(size_t)(b0 + 2) * MIN_ + i];
        if (ok[3]) v.w = mo[(size_t)(b0 + 3) * MIN_ + i];
        smo[i] = v;
    }
    __syncthreads();
    auto fma4 = [](float4 &a, float w, const float4 &v) {
        a.x = fmaf(w, v.x, a.x);
        a.y = fmaf(w, v.y, a.y);
        a.z = fmaf(w, v.z, a.z);
        a.w = fmaf(w, v.w, a.w);
    };
    // NaN stays (fmaxf would make it 0, and a diverged model's loss finite)
    auto relu = [](float a) { return a <= 0.0f ? 0.0f : a; };
    auto add4 = [](float4 a, const float4 &v) { return make_float4(a.x + v.x, a.y + v.y, a.z + v.z, a.w + v.w); };
    // a1 = m W1 + b1, the sum over k in parts
    for (uint32_t q = tid; q < MG_KP * H; q += MG_NT) {
        const uint32_t j = q % H, part = q / H;
        float4 a = make_float4(0, 0, 0, 0);
#pragma unroll 32
        for (uint32_t k = part * (MIN_ / MG_KP); k < (part + 1) * (MIN_ / MG_KP); k++) fma4(a, to_f(w1[(size_t)k * H + j]), smo[k]);
        sp[q] = a;
    }
    __syncthreads();
    for (uint32_t j = tid; j < H; j += MG_NT) {
        float4 a = sp[j];
#pragma unroll
        for (uint32_t q = 1; q < MG_KP; q++) a = add4(a, sp[q * H + j]);
        const float b = to_f(b1[j]);
        a = make_float4(a.x + b, a.y + b, a.z + b, a.w + b);
        sa1[j] = a;
        a = make_float4(relu(a.x), relu(a.y), relu(a.z), relu(a.w));
        sh1[j] = a;
        if (ok[0]) h1o[(size_t)(b0 + 0) * H + j] = a.x;
        if (ok[1]) h1o[(size_t)(b0 + 1) * H + j] = a.y;
        if (ok[2]) h1o[(size_t)(b0 + 2) * H + j] = a.z;
        if (ok[3]) h1o[(size_t)(b0 + 3) * H + j] = a.w;
    }
    __syncthreads();
    // z = h1 W2 + b2, the sum over k in two halves
    for (uint32_t q = tid; q < 2 * C; q += MG_NT) {
        const uint32_t c = q % C, half = q / C;
        float4 a = make_float4(0, 0, 0, 0);
#pragma unroll 16
        for (uint32_t k = half ? H / 2 : 0; k < (half ? H : H / 2); k++) fma4(a, to_f(w2[(size_t)k * C + c]), sh1[k]);
        sp[q] = a;
    }
    __syncthreads();
    for (uint32_t c = tid; c < C; c += MG_NT) {
        const float b = to_f(b2[c]);
        const float4 a = add4(sp[c], sp[C + c]);
        sz[c] = make_float4(a.x + b, a.y + b, a.z + b, a.w + b);
    }
    __syncthreads();
    // softmax cross-entropy, a warp per window: dz = (softmax(z) - onehot(y)) / B
    if (wid < MG && b0 + wid < B) {
        float *zr = sm + L.z + wid;
        const uint32_t yb = y[b0 + wid];
        float mx = -INFINITY;
        for (uint32_t c = lane; c < C; c += 32) mx = fmaxf(mx, zr[MG * c]);
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float se = 0.0f;
        for (uint32_t c = lane; c < C; c += 32) se += expf(zr[MG * c] - mx);
        for (int o = 16; o; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
        const float lse = mx + logf(se);
        if (lane == 0) lossw[b0 + wid] = lse - (yb < C ? zr[MG * yb] : 0.0f);   // (k_outer takes the mean)
        __syncwarp();
        for (uint32_t c = lane; c < C; c += 32) {
            const float g = (expf(zr[MG * c] - lse) - (c == yb ? 1.0f : 0.0f)) / (float)B;
            zr[MG * c] = g;
            dzo[(size_t)(b0 + wid) * C + c] = g;
        }
    } else if (wid < MG) {
        for (uint32_t c = lane; c < C; c += 32) sm[L.z + MG * c + wid] = 0.0f;
    }
    __syncthreads();
    // dh1 = dz W2^T where a1 > 0 (or NaN): a warp per row of W2
    for (uint32_t j = wid; j < H; j += MG_NT / 32) {
        float4 a = make_float4(0, 0, 0, 0);
        for (uint32_t c = lane; c < C; c += 32) fma4(a, to_f(w2[(size_t)j * C + c]), sz[c]);
        for (int o = 16; o; o >>= 1) {
            a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
            a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
            a.z += __shfl_xor_sync(0xffffffffu, a.z, o);
            a.w += __shfl_xor_sync(0xffffffffu, a.w, o);
        }
        if (lane == 0) {
            const float4 s = sa1[j];
            a = make_float4(s.x <= 0.0f ? 0.0f : a.x, s.y <= 0.0f ? 0.0f : a.y, s.z <= 0.0f ? 0.0f : a.z,
                            s.w <= 0.0f ? 0.0f : a.w);
            sdh[j] = a;
            if (ok[0]) dho[(size_t)(b0 + 0) * H + j] = a.x;
            if (ok[1]) dho[(size_t)(b0 + 1) * H + j] = a.y;
            if (ok[2]) dho[(size_t)(b0 + 2) * H + j] = a.z;
            if (ok[3]) dho[(size_t)(b0 + 3) * H + j] = a.w;
        }
    }
    __syncthreads();
    // dm = dh1 W1^T, into the place of m
    for (uint32_t i = tid; i < MIN_; i += MG_NT) {
        float4 a = make_float4(0, 0, 0, 0);
        if (H % 8 == 0) {   // a row of W1 is a lane's own: 16 bytes at a time
            const uint4 *row = reinterpret_cast<const uint4 *>(w1 + (size_t)i * H);
#pragma unroll 4
            for (uint32_t j = 0; j < H / 8; j++) {
                const uint4 v = __ldg(row + j);
                const uint32_t p[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (uint32_t q = 0; q < 4; q++) {
                    fma4(a, __uint_as_float(p[q] << 16), sdh[8 * j + 2 * q]);
                    fma4(a, __uint_as_float(p[q] & 0xFFFF0000u), sdh[8 * j + 2 * q + 1]);
                }
            }
        } else {
            for (uint32_t j = 0; j < H; j++) fma4(a, to_f(w1[(size_t)i * H + j]), sdh[j]);
        }
        smo[i] = a;
    }
    // the convolution's part of shared memory
    float *hs = sm + L.part, *da = hs + MG * MHR * MD, *pw = da + MG * MHR * DA_LD;
    float *swc = pw + (MG_NT / 32) * MF * MK * MD, *ge = swc + MF * MK * MD;
    for (uint32_t i = tid; i < MG * MHR * DA_LD; i += MG_NT) da[i] = -0.0f;   // no maximum there
    bool bad = false;
    for (uint32_t i = tid; i < MF * MK * MD; i += MG_NT) {
        swc[i] = to_f(wc[i]);
        bad |= nonfinite(swc[i]);
    }
    for (uint32_t i = tid; i < MROWS * MD; i += MG_NT) ge[i] = 0.0f;
    __syncthreads();
    if (wid < MG && b0 + wid < B)
        bad |= load_window(win + (size_t)(b0 + wid) * MW, emb, reinterpret_cast<float(*)[MD]>(hs + wid * MHR * MD), lane);
    // the gradient of each pooled maximum at the position that gave it
    {
        uint32_t av[MG * MIN_ / MG_NT];   // all loads first
#pragma unroll
        for (uint32_t i = 0; i < MG * MIN_ / MG_NT; i++) {
            const uint32_t q = tid + i * MG_NT;
            av[i] = b0 + q / MIN_ < B ? arg[(size_t)b0 * MIN_ + q] : 0u;
        }
#pragma unroll
        for (uint32_t i = 0; i < MG * MIN_ / MG_NT; i++) {
            const uint32_t q = tid + i * MG_NT, w = q / MIN_, r = q % MIN_, u = r / MF, f = r % MF;
            if (av[i] & 4u) da[(w * MHR + MPAD + MPOOL * u + (av[i] & 3u)) * DA_LD + f] = sm[L.mo + MG * r + w] + 0.0f;   // (-0 -> 0)
        }
    }
    // Positions without a maximum count as zeros, which are left out where some
    // filter or embedding is infinite or NaN (0 times that is not 0).  (Leaving
    // them out always: 512 windows of random bytes 89 -> 95 us.)
    const bool careful = __syncthreads_or(bad);
    {   // weights and bias: lane = filter, some warps per window, each its share of the pooled positions
        constexpr uint32_t WPW = MG_NT / 32 / MG, UP = MU / WPW;
        const uint32_t w = wid / WPW, u0 = (wid % WPW) * UP;
        float acc[MK][MD], sb = 0.0f;
#pragma unroll
        for (uint32_t k = 0; k < MK; k++)
#pragma unroll
            for (uint32_t d = 0; d < MD; d++) acc[k][d] = 0.0f;
        uint32_t av[UP];
#pragma unroll
        for (uint32_t i = 0; i < UP; i++) av[i] = b0 + w < B ? arg[(size_t)(b0 + w) * MIN_ + (u0 + i) * MF + lane] : 0u;
        if (b0 + w < B)
#pragma unroll
            for (uint32_t i = 0; i < UP; i++) {
                const uint32_t u = u0 + i, ar = av[i];
                if (careful && !(ar & 4u)) continue;
                const float g = (ar & 4u) ? sm[L.mo + MG * (u * MF + lane) + w] : 0.0f;
                sb += g;
                const float *h = hs + (w * MHR + MPOOL * u + (ar & 3u)) * MD;   // row t - 2
#pragma unroll
                for (uint32_t k = 0; k < MK; k++) {
                    const float4 p = *reinterpret_cast<const float4 *>(h + k * MD);
                    const float4 q = *reinterpret_cast<const float4 *>(h + k * MD + 4);
                    const float v[MD] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
                    for (uint32_t d = 0; d < MD; d++) acc[k][d] = fmaf(g, v[d], acc[k][d]);
                }
            }
#pragma unroll
        for (uint32_t k = 0; k < MK; k++)
#pragma unroll
            for (uint32_t d = 0; d < MD; d++) pw[(wid * MK * MD + k * MD + d) * MF + lane] = acc[k][d];
        atomicAdd(&gbc[lane], sb);
    }
    float dx[MD] = {0, 0, 0, 0, 0, 0, 0, 0};
    constexpr uint32_t FP = MG_NT / (MG * MW);   // parts of the filters
    const uint32_t part = tid / (MG * MW), at = tid % (MG * MW);
    static_assert(FP == 2, "two places for the parts below");
    {   // dh0: a thread per position of a window and half of the filters
        const uint32_t w = at / MW, t = at % MW;
        for (uint32_t k = 0; k < MK; k++) {
            const float *g = da + (w * MHR + MPAD + t + MPAD - k) * DA_LD;   // output position t + 2 - k
            auto add = [&](uint32_t f, float gv) {
                const float4 p = *reinterpret_cast<const float4 *>(swc + (f * MK + k) * MD);
                const float4 q = *reinterpret_cast<const float4 *>(swc + (f * MK + k) * MD + 4);
                const float v[MD] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
                for (uint32_t d = 0; d < MD; d++) dx[d] = fmaf(gv, v[d], dx[d]);
            };
            const uint32_t f0 = part * (MF / FP), f1 = f0 + MF / FP;
            if (careful) {
                for (uint32_t f = f0; f < f1; f++)
                    if (__float_as_uint(g[f]) != 0x80000000u) add(f, g[f]);   // -0: no maximum
            } else {
#pragma unroll 4
                for (uint32_t f = f0; f < f1; f++) add(f, g[f]);
            }
        }
    }
    __syncthreads();
    // into the embedding's rows, eight lanes per position: the lanes of a warp
    // meet in a word at most four times, however often a byte repeats
    float *const half0 = hs, *const half1 = sm + L.mo;   // (windows and dm are done with)
    float *const mine = (part ? half1 : half0) + at * MD;
    *reinterpret_cast<float4 *>(mine) = make_float4(dx[0], dx[1], dx[2], dx[3]);
    *reinterpret_cast<float4 *>(mine + 4) = make_float4(dx[4], dx[5], dx[6], dx[7]);
    __syncthreads();
    for (uint32_t i = tid; i < MG * MW * MD; i += MG_NT) {
        const uint32_t t = i / MD;   // window * 64 + position
        if (b0 + t / MW >= B) break;   // past the batch there is no window (and 0 times an infinite weight is not 0)
        const float v = half0[i] + half1[i];
        if (v != 0.0f) atomicAdd(&ge[win[(size_t)b0 * MW + t] * MD + i % MD], v);
    }
    __syncthreads();
    for (uint32_t i = tid; i < MF * MK * MD; i += MG_NT) {   // i = (k, d) * MF + f
        float s = 0.0f;
#pragma unroll
        for (uint32_t q = 0; q < MG_NT / 32; q++) s += pw[q * MF * MK * MD + i];
        atomicAdd(&gwc[(i % MF) * MK * MD + i / MF], s);
    }
    for (uint32_t i = tid; i < MROWS * MD; i += MG_NT)
        if (ge[i] != 0.0f) atomicAdd(&gemb[i], ge[i]);
}

// Weight gradients: G[M x N] = A^T D, A [B][M], D [B][N], and the column sums of
// D (the bias) from the first row of tiles.  64 x 64 tiles, 4 x 4 per thread;
// blockIdx.z: which of the two layers.  One cluster of CTAs shares a tile, or
// two, each CTA one slice of the batch; a cluster adds its sums in the order of
// the slices, each CTA its part of the tile from all of them, and the clusters
// add theirs to the zeros in G, where the order of two does not matter: a
// gradient is the same each time (adding each slice's as it came was not).  A CTA past the tiles
// takes the mean of the windows' losses, in 64 bits.
constexpr uint32_t OT = 64, OK = 16, OSLICE = 64, OCLUSTER = 8;

// The address of this CTA's shared word `a` in the cluster's CTA `rank`.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 cluster_ld(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(256) k_outer(uint32_t B, uint32_t slice, const float *lossw,
                                               float *loss, const float *A0, const float *D0, uint32_t M0, uint32_t N0,
                                               float *G0, float *s0, const float *A1, const float *D1, uint32_t M1,
                                               uint32_t N1, float *G1, float *s1)
{
    const bool one = blockIdx.z != 0;
    const float *A = one ? A1 : A0, *D = one ? D1 : D0;
    float *G = one ? G1 : G0, *cs = one ? s1 : s0;
    const uint32_t M = one ? M1 : M0, N = one ? N1 : N0;
    const uint32_t nt = (N + OT - 1) / OT, m0 = (blockIdx.x / nt) * OT, n0 = (blockIdx.x % nt) * OT;
    const uint32_t tid = threadIdx.x;
    if (m0 >= M) {   // (the whole cluster)
        if (blockIdx.x == gridDim.x - 1 && blockIdx.y + blockIdx.z == 0) {
            __shared__ double red[8];
            double l = 0.0;
            for (uint32_t i = tid; i < B; i += 256) l += (double)lossw[i];
            for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
            if ((tid & 31u) == 0) red[tid >> 5] = l;
            __syncthreads();
            l = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
            if (tid == 0) *loss = (float)(l / (double)B);
        }
        return;
    }
    __shared__ __align__(16) float As[OK][OT], Ds[OK][OT], part[OT * OT + OT];
    const uint32_t tx = tid & 15u, ty = tid >> 4;
    const uint32_t k0 = min(B, blockIdx.y * slice), k1 = min(B, k0 + slice);
    float acc[4][4], sum = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0.0f;
    for (uint32_t k = k0; k < k1; k += OK) {
#pragma unroll
        for (uint32_t i = 0; i < OK * OT / 256; i++) {
            const uint32_t q = tid + 256 * i, r = q / OT, c = q % OT;
            As[r][c] = k + r < k1 && m0 + c < M ? A[(size_t)(k + r) * M + m0 + c] : 0.0f;
            Ds[r][c] = k + r < k1 && n0 + c < N ? D[(size_t)(k + r) * N + n0 + c] : 0.0f;
        }
        __syncthreads();
#pragma unroll
        for (uint32_t r = 0; r < OK; r++) {
            const float4 a = *reinterpret_cast<const float4 *>(&As[r][4 * ty]);
            const float4 d = *reinterpret_cast<const float4 *>(&Ds[r][4 * tx]);
            const float av[4] = {a.x, a.y, a.z, a.w}, dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[i][j] = fmaf(av[i], dv[j], acc[i][j]);
        }
        if (m0 == 0 && tid < OT)
            for (uint32_t r = 0; r < OK; r++) sum += Ds[r][tid];
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
        *reinterpret_cast<float4 *>(&part[(4 * ty + i) * OT + 4 * tx]) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    if (tid < OT) part[OT * OT + tid] = sum;
    cluster_sync();
    const uint32_t S = gridDim.y > OCLUSTER ? gridDim.y / 2 : gridDim.y, rank = blockIdx.y % S;   // the cluster's CTAs
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(part);
    const uint32_t words = OT * OT + (m0 == 0 ? OT : 0);
    for (uint32_t i = 4 * (rank * 256 + tid); i < words; i += S * 1024) {
        float4 x[OCLUSTER];   // all loads first
#pragma unroll
        for (uint32_t q = 0; q < OCLUSTER; q++)
            x[q] = q < S ? cluster_ld(cluster_addr(base + 4 * i, q)) : make_float4(0, 0, 0, 0);
        float v[4] = {0, 0, 0, 0};
#pragma unroll
        for (uint32_t q = 0; q < OCLUSTER; q++) v[0] += x[q].x, v[1] += x[q].y, v[2] += x[q].z, v[3] += x[q].w;
        float *to = i < OT * OT ? G + (size_t)(m0 + i / OT) * N : cs;
        if (i < OT * OT && m0 + i / OT >= M) continue;
#pragma unroll
        for (uint32_t j = 0; j < 4; j++)
            if (n0 + i % OT + j < N) atomicAdd(&to[n0 + i % OT + j], v[j]);
    }
    cluster_sync();   // (until the others have read this CTA's sums)
}

// Backward through pooling and the convolution's weights: each thread one
// (f, k, d) weight over a slice of the batch (and thread d == 0, k == 0 the
// bias), atomically accumulated.  dm: gradient of m.
template <class TW>
__global__ void k_conv_back_w(const uint16_t *win, uint32_t B, const TW *emb, const float *dm, const uint8_t *arg,
                              float *gwc, float *gbc, uint32_t per)
{
    const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= MF * MK * MD) return;
    const uint32_t f = q / (MK * MD), k = (q / MD) % MK, d = q % MD;
    const uint32_t b0 = blockIdx.y * per, b1 = min(B, b0 + per);
    float sw = 0.0f, sb = 0.0f;
    for (uint32_t b = b0; b < b1; b++)
        for (uint32_t u = 0; u < MU; u++) {
            const uint32_t i = b * MIN_ + u * MF + f;
            const uint32_t ar = arg[i];
            if (!(ar & 4u)) continue;
            const float da = dm[i];
            sb += da;
            const int t = (int)(u * MPOOL + (ar & 3u) + k) - (int)(MK / 2);
            if (t >= 0 && t < (int)MW) sw = fmaf(da, to_f(emb[(size_t)win[(size_t)b * MW + t] * MD + d]), sw);
        }
    atomicAdd(&gwc[q], sw);
    if (k == 0 && d == 0) atomicAdd(&gbc[f], sb);
}

// Backward through the convolution's input: dh0[b, t, d] from every pooled
// maximum whose filter touched t; one thread per (window, u, f).
template <class TW>
__global__ void k_conv_back_x(uint32_t B, const TW *wc, const float *dm, const uint8_t *arg, float *dh0)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * MIN_) return;
    const uint32_t ar = arg[i];
    if (!(ar & 4u)) return;
    const uint32_t b = i / MIN_, r = i % MIN_, u = r / MF, f = r % MF;
    const float da = dm[i];
    for (uint32_t k = 0; k < MK; k++) {
        const int t = (int)(u * MPOOL + (ar & 3u) + k) - (int)(MK / 2);
        if (t < 0 || t >= (int)MW) continue;
        for (uint32_t d = 0; d < MD; d++)
            atomicAdd(&dh0[((size_t)b * MW + t) * MD + d], da * to_f(wc[((size_t)f * MK + k) * MD + d]));
    }
}

// C[M x N] = alpha * op(A) op(B) (+ bias[N]) (+ C if accumulate): A is M x K
// (or K x M when ta), B is K x N (or N x K when tb), all row-major.
template <class TW>
__global__ void k_gemm(const float *A, const TW *Bm, float *Cm, const TW *bias, uint32_t M, uint32_t N,
                       uint32_t K, int ta, int tb, int relu_out)
{
    __shared__ float As[GT][GT + 1], Bs[GT][GT + 1];
    const uint32_t r = blockIdx.y * GT + threadIdx.y, c = blockIdx.x * GT + threadIdx.x;
    float acc = 0.0f;
    for (uint32_t k0 = 0; k0 < K; k0 += GT) {
        const uint32_t ka = k0 + threadIdx.x, kb = k0 + threadIdx.y;
        As[threadIdx.y][threadIdx.x] =
            (r < M && ka < K) ? (ta ? A[(size_t)ka * M + r] : A[(size_t)r * K + ka]) : 0.0f;
        Bs[threadIdx.y][threadIdx.x] =
            (kb < K && c < N) ? to_f(tb ? Bm[(size_t)c * K + kb] : Bm[(size_t)kb * N + c]) : 0.0f;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < GT; k++) acc = fmaf(As[threadIdx.y][k], Bs[k][threadIdx.x], acc);
        __syncthreads();
    }
    if (r < M && c < N) {
        if (bias) acc += to_f(bias[c]);
        if (relu_out) acc = acc > 0.0f ? acc : 0.0f;
        Cm[(size_t)r * N + c] = acc;
    }
}

// Inference products: C[M x N] = A[M x K] B[K x N] + bias (ReLU optional),
// each CTA a 64 x 64 tile of C, each thread 8 x 4 of it in registers (two rows
// to a product), K in steps of 16 through shared memory, the next step's loads
// under way during this one's products.  24 576 x 64 x 512: 71 us in tiles of
// 128 rows, whose 192 CTAs left most SMs one where others had two, 55 so.
constexpr int RB_M = 64, RB_N = 64, RB_K = 16, RB_NT = 128;

template <class TW>
__global__ void __launch_bounds__(RB_NT) k_gemm_rb(const float *A, const TW *Bm, float *Cm, const TW *bias, uint32_t M,
                                                 uint32_t N, uint32_t K, int relu_out)
{
    __shared__ __align__(16) float As[RB_K][RB_M + 4];   // A tile, k-major
    __shared__ __align__(16) float Bs[RB_K][RB_N];
    const uint32_t tid = threadIdx.x, tx = tid & 15u, ty = tid >> 4;
    const uint32_t m0 = blockIdx.y * RB_M, n0 = blockIdx.x * RB_N;
    const uint32_t ar = tid >> 1, ak = (tid & 1u) * 8u, br = tid >> 3, bc = (tid & 7u) * 8u;
    unsigned long long acc[4][4];   // rows 2 i, 2 i + 1
    float pa[8], pb[8];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] = 0;
    auto fetch = [&](uint32_t k0) {
        const uint32_t m = m0 + ar;
        const float *row = A + (size_t)m * K + k0 + ak;
        if (m < M && K % 4 == 0 && k0 + ak + 8 <= K) {   // rows on 16-byte boundaries
            const float4 x = *reinterpret_cast<const float4 *>(row), y = *reinterpret_cast<const float4 *>(row + 4);
            pa[0] = x.x, pa[1] = x.y, pa[2] = x.z, pa[3] = x.w, pa[4] = y.x, pa[5] = y.y, pa[6] = y.z, pa[7] = y.w;
        } else {
#pragma unroll
            for (uint32_t i = 0; i < 8; i++) pa[i] = m < M && k0 + ak + i < K ? row[i] : 0.0f;
        }
#pragma unroll
        for (uint32_t i = 0; i < 8; i++)
            pb[i] = k0 + br < K && n0 + bc + i < N ? to_f(Bm[(size_t)(k0 + br) * N + n0 + bc + i]) : 0.0f;
    };
    fetch(0);
    for (uint32_t k0 = 0; k0 < K; k0 += RB_K) {
#pragma unroll
        for (uint32_t i = 0; i < 8; i++) As[ak + i][ar] = pa[i];
        *reinterpret_cast<float4 *>(&Bs[br][bc]) = make_float4(pb[0], pb[1], pb[2], pb[3]);
        *reinterpret_cast<float4 *>(&Bs[br][bc + 4]) = make_float4(pb[4], pb[5], pb[6], pb[7]);
        __syncthreads();
        if (k0 + RB_K < K) fetch(k0 + RB_K);
#pragma unroll
        for (int k = 0; k < RB_K; k++) {
            const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(&As[k][ty * 8]);
            const ulonglong2 c = *reinterpret_cast<const ulonglong2 *>(&As[k][ty * 8 + 4]);
            const float4 b = *reinterpret_cast<const float4 *>(&Bs[k][tx * 4]);
            const unsigned long long av[4] = {a.x, a.y, c.x, c.y};
            const unsigned long long bv[4] = {pack2(b.x, b.x), pack2(b.y, b.y), pack2(b.z, b.z), pack2(b.w, b.w)};
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int j = 0; j < 4; j++) acc[i][j] = fma2(av[i], bv[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const uint32_t m = m0 + ty * 8 + i;
        if (m >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const uint32_t nn = n0 + tx * 4 + j;
            if (nn >= N) continue;
            float v = __uint_as_float((uint32_t)(acc[i / 2][j] >> (i & 1 ? 32 : 0)));
            if (bias) v += to_f(bias[nn]);
            if (relu_out) v = v > 0.0f ? v : 0.0f;
            Cm[(size_t)m * N + nn] = v;
        }
    }
}

// softmax cross-entropy per row: dz = (softmax(z) - onehot(y)) / B, loss sum
__global__ void k_softmax_ce(const float *z, const uint16_t *y, uint32_t B, uint32_t C, float *dz, float *loss)
{
    const uint32_t b = blockIdx.x;
    if (b >= B) return;
    const float *zr = z + (size_t)b * C;
    float mx = -INFINITY;
    for (uint32_t c = threadIdx.x; c < C; c += blockDim.x) mx = fmaxf(mx, zr[c]);
    for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float se = 0.0f;
    for (uint32_t c = threadIdx.x; c < C; c += blockDim.x) se += expf(zr[c] - mx);
    for (int o = 16; o; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
    const float lse = mx + logf(se);
    for (uint32_t c = threadIdx.x; c < C; c += blockDim.x) {
        const float pr = expf(zr[c] - lse);
        dz[(size_t)b * C + c] = (pr - (c == y[b] ? 1.0f : 0.0f)) / (float)B;
    }
    if (threadIdx.x == 0) atomicAdd(loss, (lse - zr[y[b]]) / (float)B);
}

// column sums: out[c] = sum_b M[b, c]
__global__ void k_colsum(const float *Mx, uint32_t B, uint32_t N, float *out)
{
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    float s = 0.0f;
    for (uint32_t b = 0; b < B; b++) s += Mx[(size_t)b * N + c];
    out[c] = s;
}

// dA1 = dH1 * (A1 > 0)
__global__ void k_relu_back(float *dh, const float *a, size_t n)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && a[i] <= 0.0f) dh[i] = 0.0f;
}

// demb[x, d] += dh0[b, t, d] for byte x at window position t
__global__ void k_emb_back(const uint16_t *win, uint32_t B, const float *dh0, float *demb)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * MW * MD) return;
    const uint32_t b = i / (MW * MD), r = i % (MW * MD), t = r / MD, d = r % MD;
    const float v = dh0[i];
    if (v != 0.0f) atomicAdd(&demb[(size_t)win[(size_t)b * MW + t] * MD + d], v);
}

// AdamW (beta 0.9 / 0.999, eps 1e-8): decoupled weight decay on the weight
// matrices [d0, d1), [d2, d3), [d4, d5), then the Adam step; the BF16 copy
// follows the FP32 master weights.
__global__ void k_adamw(float *w, float *m, float *v, const float *g, __nv_bfloat16 *w16, size_t n, float lr,
                        float b1c, float b2c, float wd, size_t d0, size_t d1, size_t d2, size_t d3, size_t d4,
                        size_t d5)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = 0.9f * m[i] + 0.1f * gi;
    const float vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    float wi = w[i];
    if ((i >= d0 && i < d1) || (i >= d2 && i < d3) || (i >= d4 && i < d5)) wi -= lr * wd * wi;
    wi -= lr * (mi / b1c) / (sqrtf(vi / b2c) + 1e-8f);
    w[i] = wi;
    w16[i] = __float2bfloat16(wi);
}

__global__ void k_to_bf16(const float *w, __nv_bfloat16 *w16, size_t n)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) w16[i] = __float2bfloat16(w[i]);
}

// windows of the chunk starts (pad where there is no start)
__global__ void k_windows(const uint8_t *in, uint64_t n, const uint64_t *start, uint32_t j0, uint32_t cnt,
                          uint16_t *win)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= cnt * MW) return;
    const uint32_t b = i / MW, k = i % MW;
    const uint64_t p = start[j0 + b];
    win[i] = p == ~0ull ? 256u : (uint16_t)window_byte(in, n, p, k);
}

// The argmax of the logits over the candidate contexts of the byte before
// each chunk start (BOUNDARY = class C-1 -> 0xFFFE); one warp per chunk.
__global__ void k_argmax(const float *z, uint32_t C, uint32_t j0, uint32_t cnt, const uint64_t *start,
                         const uint32_t *cinfo, const uint8_t *scan_blob, uint32_t cbeg_off, uint32_t cand_off,
                         uint16_t *guess)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b >= cnt) return;
    const uint32_t j = j0 + b;
    if (j == 0 || start[j] == ~0ull) {
        if (lane == 0) guess[j] = 0xFFFEu;
        return;
    }
    const uint16_t *cbeg = reinterpret_cast<const uint16_t *>(scan_blob + cbeg_off);
    const uint16_t *cand = reinterpret_cast<const uint16_t *>(scan_blob + cand_off);
    const uint32_t byte = cinfo[j] >> 8, lo = cbeg[byte], hi = cbeg[byte + 1];
    const float *zr = z + (size_t)b * C;
    float best = -INFINITY;
    uint32_t arg = C - 1;
    for (uint32_t t = lane; t < 1 + hi - lo; t += 32) {
        const uint32_t c = t == 0 ? C - 1 : cand[lo + t - 1];
        const float v = zr[c];
        if (v > best || (v == best && c < arg)) {
            best = v;
            arg = c;
        }
    }
    for (int o = 16; o; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const uint32_t oa = __shfl_xor_sync(0xffffffffu, arg, o);
        if (ob > best || (ob == best && oa < arg)) {
            best = ob;
            arg = oa;
        }
    }
    if (lane == 0) guess[j] = arg == C - 1 ? (uint16_t)0xFFFEu : (uint16_t)arg;
}

}  // namespace

uint32_t model_contexts(const lx_model *m) { return m ? m->C : 0; }

}  // namespace lx

using namespace lx;

namespace {

int ensure_act(lx_model *m, uint32_t B, bool predict = false)
{
    const size_t need = predict ? (size_t)B * (MIN_ + m->H + m->C) + 16
                                : (size_t)B * (MIN_ * 2 + MW * MD + m->H * 3 + m->C * 2) + 16;
    if (m->act_floats < need) {
        if (m->act) cudaFree(m->act);
        m->act = nullptr;
        m->act_floats = 0;
        if (cudaMalloc(&m->act, need * sizeof(float)) != cudaSuccess) return LX_E_NOMEM;
        m->act_floats = need;
    }
    const size_t abytes = predict ? 0 : (size_t)B * MIN_;
    if (m->arg_bytes < abytes) {
        if (m->arg) cudaFree(m->arg);
        m->arg = nullptr;
        m->arg_bytes = 0;
        if (cudaMalloc(&m->arg, abytes) != cudaSuccess) return LX_E_NOMEM;
        m->arg_bytes = abytes;
    }
    return LX_OK;
}

dim3 gemm_grid(uint32_t M, uint32_t N) { return dim3((N + GT - 1) / GT, (M + GT - 1) / GT); }
uint32_t conv_grid(uint32_t B) { return std::min<uint32_t>((B + CP_WARPS - 1) / CP_WARPS, 8 * 152); }
dim3 rb_grid(uint32_t M, uint32_t N) { return dim3((N + RB_N - 1) / RB_N, (M + RB_M - 1) / RB_M); }

// Forward (and with labels, backward into m->g) for a batch of windows, on
// the BF16 weights.  Activations: m | a1 | h1 | z | dz | dh1 | dm | dh0 | loss
int model_pass(lx_model *m, const uint16_t *d_win, const uint16_t *d_y, uint32_t B, float *d_logits_out,
               cudaStream_t s, float *h_loss)
{
    int rc = ensure_act(m, B);
    if (rc != LX_OK) return rc;
    const uint32_t H = m->H, C = m->C;
    float *mo = m->act, *a1 = mo + (size_t)B * MIN_, *h1 = a1 + (size_t)B * H, *z = h1 + (size_t)B * H;
    float *dz = z + (size_t)B * C, *dh1 = dz + (size_t)B * C, *dm = dh1 + (size_t)B * H;
    float *dh0 = dm + (size_t)B * MIN_, *loss = dh0 + (size_t)B * MW * MD;
    const __nv_bfloat16 *w = m->w16;
    const dim3 t2(GT, GT);
    const uint32_t nm = B * MIN_;
    k_conv_pool<<<conv_grid(B), 32 * CP_WARPS, 0, s>>>(d_win, B, w + m->o_emb, w + m->o_wc, w + m->o_bc, mo, m->arg);
    if (d_y && !d_logits_out && H <= MG_MAXH && C <= MG_MAXC) {
        const uint32_t smem = 4 * MgSmem(H, C).total;
        if (!m->mg_ready) {   // once per model; the largest sizes', which all models share
            rc = cuda_err(cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               4 * MgSmem(MG_MAXH, MG_MAXC).total));
            if (rc != LX_OK) return rc;
            m->mg_ready = true;
        }
        float *g = m->g;   // the loss follows the gradient
        cudaMemsetAsync(g, 0, sizeof(float) * (m->n_params + 1), s);
        k_mlp_grad<<<(B + MG - 1) / MG, MG_NT, smem, s>>>(d_win, d_y, B, H, C, mo, m->arg, w + m->o_emb, w + m->o_wc,
                                                         w + m->o_w1, w + m->o_b1, w + m->o_w2, w + m->o_b2, h1, dz, dh1,
                                                         g + m->o_emb, g + m->o_wc, g + m->o_bc, dm);   // dm: here the windows' losses
        const uint32_t t1 = (MIN_ / OT) * ((H + OT - 1) / OT), t2n = ((H + OT - 1) / OT) * ((C + OT - 1) / OT);
        // slices of 64 windows, of more where that makes over 16
        const uint32_t slice = std::max(OSLICE, ((B + 2 * OCLUSTER - 1) / (2 * OCLUSTER) + OK - 1) / OK * OK);
        const uint32_t ns = (B + slice - 1) / slice, cluster = ns > OCLUSTER ? (ns + 1) / 2 : ns;
        const uint32_t slices = ns > OCLUSTER ? 2 * cluster : cluster;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(std::max(t1, t2n) + 1, slices, 2);   // (the last: the loss)
        cfg.blockDim = dim3(256);
        cfg.stream = s;
        cudaLaunchAttribute at[1] = {};
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1;
        at[0].val.clusterDim.y = cluster;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        rc = cuda_err(cudaLaunchKernelEx(&cfg, k_outer, B, slice, (const float *)dm, g + m->n_params, (const float *)mo, (const float *)dh1, (uint32_t)MIN_, H,
                                         g + m->o_w1, g + m->o_b1, (const float *)h1, (const float *)dz, H, C, g + m->o_w2,
                                         g + m->o_b2));
        if (rc == LX_OK) rc = cuda_err(cudaGetLastError());
        if (rc == LX_OK && h_loss) {
            rc = cuda_err(cudaMemcpyAsync(h_loss, g + m->n_params, sizeof(float), cudaMemcpyDeviceToHost, s));
            if (rc == LX_OK) rc = cuda_err(cudaStreamSynchronize(s));
        }
        return rc;
    }
    k_gemm<__nv_bfloat16><<<gemm_grid(B, H), t2, 0, s>>>(mo, w + m->o_w1, a1, w + m->o_b1, B, H, MIN_, 0, 0, 0);
    cudaMemcpyAsync(h1, a1, sizeof(float) * B * H, cudaMemcpyDeviceToDevice, s);
    k_relu_back<<<(B * H + 255) / 256, 256, 0, s>>>(h1, a1, (size_t)B * H);   // h1 = relu(a1)
    k_gemm<__nv_bfloat16><<<gemm_grid(B, C), t2, 0, s>>>(h1, w + m->o_w2, z, w + m->o_b2, B, C, H, 0, 0, 0);
    if (d_logits_out)
        cudaMemcpyAsync(d_logits_out, z, sizeof(float) * B * C, cudaMemcpyDeviceToDevice, s);
    if (!d_y) return cuda_err(cudaGetLastError());
    float *g = m->g;
    cudaMemsetAsync(loss, 0, sizeof(float), s);
    cudaMemsetAsync(g, 0, sizeof(float) * m->n_params, s);
    cudaMemsetAsync(dh0, 0, sizeof(float) * B * MW * MD, s);
    k_softmax_ce<<<B, 32, 0, s>>>(z, d_y, B, C, dz, loss);
    k_gemm<float><<<gemm_grid(H, C), t2, 0, s>>>(h1, dz, g + m->o_w2, nullptr, H, C, B, 1, 0, 0);   // h1^T dz
    k_colsum<<<(C + 255) / 256, 256, 0, s>>>(dz, B, C, g + m->o_b2);
    k_gemm<__nv_bfloat16><<<gemm_grid(B, H), t2, 0, s>>>(dz, w + m->o_w2, dh1, nullptr, B, H, C, 0, 1, 0);  // dz W2^T
    k_relu_back<<<(B * H + 255) / 256, 256, 0, s>>>(dh1, a1, (size_t)B * H);
    k_gemm<float><<<gemm_grid(MIN_, H), t2, 0, s>>>(mo, dh1, g + m->o_w1, nullptr, MIN_, H, B, 1, 0, 0);  // m^T dh1
    k_colsum<<<(H + 255) / 256, 256, 0, s>>>(dh1, B, H, g + m->o_b1);
    k_gemm<__nv_bfloat16><<<gemm_grid(B, MIN_), t2, 0, s>>>(dh1, w + m->o_w1, dm, nullptr, B, MIN_, H, 0, 1, 0);
    const uint32_t per = 32;
    const dim3 gw((MF * MK * MD + 127) / 128, (B + per - 1) / per);
    k_conv_back_w<__nv_bfloat16><<<gw, 128, 0, s>>>(d_win, B, w + m->o_emb, dm, m->arg, g + m->o_wc, g + m->o_bc, per);
    k_conv_back_x<__nv_bfloat16><<<(nm + 255) / 256, 256, 0, s>>>(B, w + m->o_wc, dm, m->arg, dh0);
    k_emb_back<<<(B * MW * MD + 255) / 256, 256, 0, s>>>(d_win, B, dh0, g + m->o_emb);
    cudaMemcpyAsync(g + m->n_params, loss, sizeof(float), cudaMemcpyDeviceToDevice, s);
    rc = cuda_err(cudaGetLastError());
    if (rc == LX_OK && h_loss) {
        rc = cuda_err(cudaMemcpyAsync(h_loss, loss, sizeof(float), cudaMemcpyDeviceToHost, s));
        if (rc == LX_OK) rc = cuda_err(cudaStreamSynchronize(s));
    }
    return rc;
}

// splitmix64 -> uniform in [-a, a)
float init_value(uint64_t &st, float a)
{
    st += 0x9E3779B97F4A7C15ull;
    uint64_t z = st;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (float)((double)(z >> 11) / (double)(1ull << 53) * 2.0 - 1.0) * a;
}

}  // namespace

int lx::model_predict(lx_model *m, const uint8_t *in, uint64_t n, const uint64_t *start, const uint32_t *cinfo,
                      const uint8_t *scan_blob, uint32_t cbeg_off, uint32_t cand_off, uint32_t M, uint16_t *guess,
                      cudaStream_t s)
{
    const uint32_t parts = (M + PRED_BATCH - 1) / PRED_BATCH, B = (M + parts - 1) / parts;   // batches of equal size
    int rc = ensure_act(m, B, true);
    if (rc != LX_OK) return rc;
    if (!m->win && cudaMalloc(&m->win, sizeof(uint16_t) * PRED_BATCH * MW) != cudaSuccess) return LX_E_NOMEM;
    const uint32_t H = m->H, C = m->C;
    float *mo = m->act, *h1 = mo + (size_t)B * MIN_, *z = h1 + (size_t)B * H;
    const __nv_bfloat16 *w = m->w16;
    for (uint32_t j0 = 0; j0 < M; j0 += B) {
        const uint32_t cnt = std::min<uint32_t>(B, M - j0);
        k_windows<<<(cnt * MW + 255) / 256, 256, 0, s>>>(in, n, start, j0, cnt, m->win);
        k_conv_pool2<<<conv_grid((cnt + 1) / 2), 32 * CP_WARPS, 0, s>>>(m->win, cnt, w + m->o_emb, w + m->o_wc,
                                                                        w + m->o_bc, mo);
        // h1 = relu(m W1 + b1), z = h1 W2 + b2
        k_gemm_rb<__nv_bfloat16><<<rb_grid(cnt, H), RB_NT, 0, s>>>(mo, w + m->o_w1, h1, w + m->o_b1, cnt, H, MIN_, 1);
        k_gemm_rb<__nv_bfloat16><<<rb_grid(cnt, C), RB_NT, 0, s>>>(h1, w + m->o_w2, z, w + m->o_b2, cnt, C, H, 0);
        k_argmax<<<(cnt * 32 + 255) / 256, 256, 0, s>>>(z, C, j0, cnt, start, cinfo, scan_blob, cbeg_off, cand_off,
                                                        guess);
    }
    return cuda_err(cudaGetLastError());
}

extern "C" int lx_model_create(uint32_t n_contexts, uint32_t hidden, uint64_t seed, lx_model **out)
{
    if (!out || n_contexts < 2 || n_contexts > 0xFFFEu || hidden == 0 || hidden > 1024) return LX_E_INVAL;
    *out = nullptr;
    lx_model *m = new (std::nothrow) lx_model();
    if (!m) return LX_E_NOMEM;
    m->C = n_contexts;
    m->H = hidden;
    cudaGetDevice(&m->device);
    m->o_emb = 0;
    m->o_wc = m->o_emb + (size_t)MROWS * MD;
    m->o_bc = m->o_wc + (size_t)MF * MK * MD;
    m->o_w1 = m->o_bc + MF;
    m->o_b1 = m->o_w1 + (size_t)MIN_ * hidden;
    m->o_w2 = m->o_b1 + hidden;
    m->o_b2 = m->o_w2 + (size_t)hidden * n_contexts;
    m->n_params = m->o_b2 + n_contexts;
    std::vector<float> h(m->n_params, 0.0f);
    uint64_t st = seed;
    for (size_t i = m->o_emb; i < m->o_wc; i++) h[i] = init_value(st, 0.5f);
    const float ac = 1.0f / std::sqrt((float)(MK * MD)), a1 = 1.0f / std::sqrt((float)MIN_),
                a2 = 1.0f / std::sqrt((float)hidden);
    for (size_t i = m->o_wc; i < m->o_bc; i++) h[i] = init_value(st, ac);
    for (size_t i = m->o_w1; i < m->o_b1; i++) h[i] = init_value(st, a1);
    for (size_t i = m->o_w2; i < m->o_b2; i++) h[i] = init_value(st, a2);
    const size_t bytes = sizeof(float) * m->n_params;
    bool ok = cudaMalloc(&m->w, bytes) == cudaSuccess && cudaMalloc(&m->m, bytes) == cudaSuccess &&
              cudaMalloc(&m->v, bytes) == cudaSuccess &&
              cudaMalloc(&m->g, bytes + sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->w16, sizeof(__nv_bfloat16) * m->n_params) == cudaSuccess;
    ok = ok && cudaMemcpy(m->w, h.data(), bytes, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemset(m->m, 0, bytes) == cudaSuccess && cudaMemset(m->v, 0, bytes) == cudaSuccess;
    if (ok) {
        k_to_bf16<<<(unsigned)((m->n_params + 255) / 256), 256>>>(m->w, m->w16, m->n_params);
        ok = cudaDeviceSynchronize() == cudaSuccess;
    }
    if (!ok) {
        lx_model_free(m);
        return LX_E_NOMEM;
    }
    *out = m;
    return LX_OK;
}

extern "C" void lx_model_free(lx_model *m)
{
    if (!m) return;
    cudaFree(m->w);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->g);
    cudaFree(m->w16);
    cudaFree(m->act);
    cudaFree(m->arg);
    cudaFree(m->win);
    cudaFreeHost(m->h_g);
    delete m;
}

extern "C" int lx_model_info(const lx_model *m, uint32_t *n_contexts, uint32_t *hidden, uint32_t *window,
                             uint32_t *embed, uint64_t *n_params)
{
    if (!m) return LX_E_INVAL;
    if (n_contexts) *n_contexts = m->C;
    if (hidden) *hidden = m->H;
    if (window) *window = MW;
    if (embed) *embed = MD;
    if (n_params) *n_params = m->n_params;
    return LX_OK;
}

extern "C" int lx_model_get_params(const lx_model *m, float *host, uint64_t count)
{
    if (!m || !host || count != m->n_params) return LX_E_INVAL;
    return cuda_err(cudaMemcpy(host, m->w, sizeof(float) * count, cudaMemcpyDeviceToHost));
}

extern "C" int lx_model_set_params(lx_model *m, const float *host, uint64_t count)
{
    if (!m || !host || count != m->n_params) return LX_E_INVAL;
    int rc = cuda_err(cudaMemcpy(m->w, host, sizeof(float) * count, cudaMemcpyHostToDevice));
    if (rc != LX_OK) return rc;
    k_to_bf16<<<(unsigned)((m->n_params + 255) / 256), 256>>>(m->w, m->w16, m->n_params);
    return cuda_err(cudaDeviceSynchronize());
}

extern "C" int lx_model_windows(const uint8_t *d_in, uint64_t n, const uint64_t *d_pos, uint32_t count,
                                uint16_t *d_windows, void *stream)
{
    if ((count && (!d_pos || !d_windows)) || (n && !d_in)) return LX_E_INVAL;
    if (!count) return LX_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    k_windows<<<(count * MW + 255) / 256, 256, 0, s>>>(d_in, n, d_pos, 0, count, d_windows);
    return cuda_err(cudaGetLastError());
}

extern "C" int lx_model_forward(lx_model *m, const uint16_t *d_windows, uint32_t batch, float *d_logits,
                                void *stream)
{
    if (!m || !d_windows || !d_logits || batch == 0) return LX_E_INVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rc = model_pass(m, d_windows, nullptr, batch, d_logits, s, nullptr);
    if (rc == LX_OK) rc = cuda_err(cudaStreamSynchronize(s));
    return rc;
}

extern "C" int lx_model_gradient(lx_model *m, const uint16_t *d_windows, const uint16_t *d_labels, uint32_t batch,
                                 float *host_grad, uint64_t count, float *loss, void *stream)
{
    if (!m || !d_windows || !d_labels || batch == 0 || !host_grad || count != m->n_params) return LX_E_INVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the gradient and the loss behind it in one copy to pinned memory: a copy
    // to pageable memory of this size takes longer than the kernels
    if (!m->h_g && cudaMallocHost(&m->h_g, sizeof(float) * (count + 1)) != cudaSuccess) return LX_E_NOMEM;
    int rc = model_pass(m, d_windows, d_labels, batch, nullptr, s, nullptr);
    if (rc == LX_OK) rc = cuda_err(cudaMemcpyAsync(m->h_g, m->g, sizeof(float) * (count + 1), cudaMemcpyDeviceToHost, s));
    if (rc == LX_OK) rc = cuda_err(cudaStreamSynchronize(s));
    if (rc != LX_OK) return rc;
    std::memcpy(host_grad, m->h_g, sizeof(float) * count);
    if (loss) *loss = m->h_g[count];
    return rc;
}

extern "C" int lx_model_train_step(lx_model *m, const uint16_t *d_windows, const uint16_t *d_labels,
                                   uint32_t batch, float lr, float *loss, void *stream)
{
    if (!m || !d_windows || !d_labels || batch == 0 || !(lr > 0.0f)) return LX_E_INVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    float l = 0.0f;
    int rc = model_pass(m, d_windows, d_labels, batch, nullptr, s, &l);
    if (rc != LX_OK) return rc;
    m->step++;
    const float b1c = 1.0f - std::pow(0.9f, (float)m->step), b2c = 1.0f - std::pow(0.999f, (float)m->step);
    k_adamw<<<(unsigned)((m->n_params + 255) / 256), 256, 0, s>>>(m->w, m->m, m->v, m->g, m->w16, m->n_params, lr,
                                                                  b1c, b2c, WEIGHT_DECAY, m->o_wc, m->o_bc, m->o_w1,
                                                                  m->o_b1, m->o_w2, m->o_b2);
    rc = cuda_err(cudaGetLastError());
    if (loss) *loss = l;
    return rc;
}
