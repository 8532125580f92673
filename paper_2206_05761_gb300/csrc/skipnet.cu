// skipnet.cu -- the subtree CNN on the tensor cores: forward, backward and
// Adam, each convolution an implicit GEMM issued with tcgen05.mma (BF16
// operands staged in shared memory, FP32 accumulators in TMEM).
//
//   forward       Z[p][o]  = b[o] + sum_k Xcol[p][k] W[o][k]      M=128 pixels, N=16, K=48|144
//   grad input    dX[p][c] = sum_k dZcol[p][k] W'[c][k]           the same convolution of dZ with
//                            the taps reversed and W transposed over its channels
//   grad weights  dW[k][o] = sum_p Xcol[p][k] dZ[p][o]            M=128 k-rows, N=16, K=pixels
//
// k = tap * cin + c with tap = 3*(di+1) + (dj+1): the im2col of a 3x3 window
// with zero padding over channels-last images.  Parameters are kept in FP32
// (the CPU oracle's layout [cout][cin][3][3]) and packed to BF16 operand
// tiles after every update.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "../../include/hwfv1.h"
#include "skipnet.h"
#include "tcgen05.cuh"

namespace hwfv1 {
namespace {

using bf16 = __nv_bfloat16;

struct Layer {
    int cin, kpad, cout, offw, offb;
};
constexpr Layer kLayers[3] = {
    {4, 48, 16, 0, 576},
    {16, 144, 16, 592, 2896},
    {16, 144, 5, 2912, 3632},
};
__constant__ Layer c_layers[3] = {
    {4, 48, 16, 0, 576},
    {16, 144, 16, 592, 2896},
    {16, 144, 5, 2912, 3632},
};
constexpr uint32_t kWaitLimit = 1u << 24;   // polls of an mbarrier before giving up

// ---------------------------------------------------------------------------
// Weight packing: FP32 [cout][cin][3][3] -> the B tiles (N = 16 rows, K =
// kpad, core-matrix layout) of the forward GEMM (rows cout) and, where cin is
// 16, of the input gradient (rows cin, k = tap' * 16 + cout with tap' = 8 - tap).
// ---------------------------------------------------------------------------
__global__ void k_pack(const float* __restrict__ params, bf16* __restrict__ wf, bf16* __restrict__ wt) {
    const Layer ly = c_layers[blockIdx.y];
    bf16* f = wf + blockIdx.y * (16 * 144);
    bf16* t = wt + blockIdx.y * (16 * 144);
    for (int idx = threadIdx.x; idx < 16 * ly.kpad; idx += blockDim.x) {
        const int o = idx / ly.kpad, k = idx % ly.kpad;
        float v = 0.f;
        if (o < ly.cout && k < 9 * ly.cin) {
            const int tap = k / ly.cin, c = k % ly.cin;
            v = params[ly.offw + (o * ly.cin + c) * 9 + tap];
        }
        f[tc::core_off(o, k, ly.kpad / 8) / 2] = __float2bfloat16(v);
    }
    if (ly.cin != 16) return;
    for (int idx = threadIdx.x; idx < 16 * 144; idx += blockDim.x) {
        const int c = idx / 144, k = idx % 144, tap = 8 - k / 16, o = k % 16;
        const float v = o < ly.cout ? params[ly.offw + (o * ly.cin + c) * 9 + tap] : 0.f;
        t[tc::core_off(c, k, 18) / 2] = __float2bfloat16(v);
    }
}

struct Img {
    int B, H, W, cin;
};

// Which of the 9 taps of pixel p fall inside its image (none past the last
// pixel).  Tap t of pixel p is pixel p + tap_shift(t, W).
__device__ __forceinline__ uint32_t tap_mask(const Img& g, int p) {
    if (p >= g.B * g.H * g.W) return 0u;
    const int rem = p % (g.H * g.W), y = rem / g.W, x = rem % g.W;
    const uint32_t row = (x > 0 ? 1u : 0u) | 2u | (x + 1 < g.W ? 4u : 0u);
    return (y > 0 ? row : 0u) | (row << 3) | (y + 1 < g.H ? row << 6 : 0u);
}
__device__ __forceinline__ int tap_shift(int tap, int W) { return (tap / 3 - 1) * W + tap % 3 - 1; }

// The im2col row of pixel p (k = tap * CIN + c over the 3x3 taps, zero
// outside the image and for k >= 9 CIN) written to row `row` of the
// core-matrix operand: every load first (16 bytes a piece, 8 for CIN = 4),
// then the stores.
template <int CIN>
__device__ __forceinline__ void im2col_row(const bf16* __restrict__ X, const Img& g, int p, uint32_t row,
                                           uint8_t* sA) {
    const uint32_t m = tap_mask(g, p);
    if constexpr (CIN == 16) {
        uint4 v[9][2];
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            const uint4* src = reinterpret_cast<const uint4*>(X + ((int64_t)p + tap_shift(tap, g.W)) * 16);
            const bool ok = (m >> tap) & 1u;
            v[tap][0] = ok ? __ldg(src) : make_uint4(0u, 0u, 0u, 0u);
            v[tap][1] = ok ? __ldg(src + 1) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int tap = 0; tap < 9; ++tap)
#pragma unroll
            for (int cb = 0; cb < 2; ++cb)
                *reinterpret_cast<uint4*>(sA + tc::core_off(row, tap * 16 + cb * 8, 18)) = v[tap][cb];
    } else {
        uint2 v[12];
#pragma unroll
        for (int tap = 0; tap < 12; ++tap) {
            const bool ok = tap < 9 && ((m >> tap) & 1u);
            v[tap] = ok ? __ldg(reinterpret_cast<const uint2*>(X + ((int64_t)p + tap_shift(tap, g.W)) * 4))
                        : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int tap = 0; tap < 12; ++tap)
            *reinterpret_cast<uint2*>(sA + tc::core_off(row, tap * 4, 6)) = v[tap];
    }
}

// Shared TMEM/mbarrier bookkeeping of one CTA (128 threads).
struct TcCta {
    uint64_t bar;
    uint32_t tmem;
};

__device__ __forceinline__ void tc_begin(TcCta& s, uint32_t ncols) {
    if (threadIdx.x < 32) {
        tc::tmem_alloc(&s.tmem, ncols);
        tc::tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        tc::mbar_init(&s.bar, 1);
        tc::fence_mbar_init();
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
}

// Wait for the committed MMAs (bounded); on timeout flag the error and wait
// once more (bounded) so that TMEM is not freed under a running MMA.
__device__ __forceinline__ bool tc_wait(TcCta& s, uint32_t phase, int* err) {
    const bool ok = tc::mbar_wait_bounded(&s.bar, phase, kWaitLimit);
    if (!ok) {
        if (threadIdx.x == 0) atomicOr(err, 1);
        tc::mbar_wait_bounded(&s.bar, phase, kWaitLimit);
    }
    tc::fence_after_sync();
    return ok;
}

__device__ __forceinline__ void tc_end(TcCta& s, uint32_t ncols) {
    tc::fence_before_sync();
    __syncthreads();
    if (threadIdx.x < 32) {
        tc::fence_after_sync();
        tc::tmem_dealloc(s.tmem, ncols);
    }
}

// ---------------------------------------------------------------------------
// One convolution, 128 pixels per CTA, its epilogue in registers (thread t
// holds pixel t's 16 outputs).
//   kActivate  A = relu(Z + b), bf16
//   kLogits    Z + b, float (16 a pixel, zero from cout on)
//   kLoss      softmax cross-entropy of the logits: the summed loss and
//              dZ = (softmax - onehot) / npix, bf16
//   kInputGrad dZ of the layer below: the outputs where its activation is
//              positive (relu'), else 0, bf16
// ---------------------------------------------------------------------------
enum ConvOut { kActivate, kLogits, kLoss, kInputGrad };
struct ConvArgs {
    const bf16* X;                  // [npix][CIN]
    Img g;
    const bf16* w;                  // packed B tile, 16 x kpad
    const float* bias;              // (not kInputGrad)
    int cout;
    bf16* A;                        // bf16 output [npix][16]
    float* Z;                       // kLogits: output [npix][16]
    const uint8_t* labels;          // kLoss
    float inv_npix;
    double* loss;
    const bf16* act;                // kInputGrad: the layer below's activations [npix][16]
    int* err;
};

__device__ __forceinline__ uint32_t pack2(float a, float b) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ void store_bf16x16(bf16* dst, const float (&v)[16]) {
    uint4* d = reinterpret_cast<uint4*>(dst);
    d[0] = make_uint4(pack2(v[0], v[1]), pack2(v[2], v[3]), pack2(v[4], v[5]), pack2(v[6], v[7]));
    d[1] = make_uint4(pack2(v[8], v[9]), pack2(v[10], v[11]), pack2(v[12], v[13]), pack2(v[14], v[15]));
}

// Bound by the latency of its three parts (im2col gather, one MMA chain,
// epilogue), not by bytes or the tensor cores: 18-20 us for 131,072 pixels
// (8 images of 128 x 128) with 16 channels in.  What a pixel needs moves as
// 128-bit accesses (41 us with element-wise stores), and the input gradient is
// the same convolution with relu' in its epilogue (96 us for its columns, 43 to
// add them up and 12 for relu' as kernels of their own).
template <int CIN, int OUT>
__global__ void __launch_bounds__(128) k_conv(ConvArgs a) {
    constexpr int kpad = CIN == 16 ? 144 : 48, kb = kpad / 8;
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ TcCta s;
    uint8_t* sA = smem;                        // 128 x kpad
    uint8_t* sB = smem + 256 * kpad;           // 16 x kpad
    const int t = threadIdx.x;
    const int p = blockIdx.x * 128 + t;
    const int npix = a.g.B * a.g.H * a.g.W;
    im2col_row<CIN>(a.X, a.g, p, (uint32_t)t, sA);
    const uint4* src = reinterpret_cast<const uint4*>(a.w);
    for (int i = t; i < 2 * kpad; i += 128) reinterpret_cast<uint4*>(sB)[i] = src[i];
    tc_begin(s, 32);
    if (t == 0) {
        const uint32_t a0 = tc::smem_addr(sA), b0 = tc::smem_addr(sB);
        for (int kk = 0; kk < kpad / 16; ++kk)
            tc::mma_bf16(s.tmem, tc::sdesc(a0 + kk * 256, 128, kb * 128), tc::sdesc(b0 + kk * 256, 128, kb * 128),
                         tc::idesc_bf16(128, 16), kk > 0);
        tc::mma_commit(&s.bar);
    }
    tc_wait(s, 0, a.err);
    float v[16];
    tc::tmem_ld16(s.tmem + ((uint32_t)(32 * (t >> 5)) << 16), v);
    if constexpr (OUT == kInputGrad) {
        if (p < npix) {
            const uint4* m = reinterpret_cast<const uint4*>(a.act + (size_t)p * 16);
            const uint4 m0 = __ldg(m), m1 = __ldg(m + 1);
            const uint32_t w[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
            for (int o = 0; o < 16; ++o) {
                // activations are never negative: positive = not 0
                const uint32_t h = (o & 1) ? w[o / 2] >> 16 : w[o / 2] & 0xFFFFu;
                if ((h & 0x7FFFu) == 0u) v[o] = 0.f;
            }
            store_bf16x16(a.A + (size_t)p * 16, v);
        }
    } else {
        if (p < npix) {
#pragma unroll
            for (int o = 0; o < 16; ++o) v[o] = o < a.cout ? v[o] + __ldg(a.bias + o) : 0.f;
        }
        if constexpr (OUT == kActivate) {
            if (p < npix) {
#pragma unroll
                for (int o = 0; o < 16; ++o) v[o] = fmaxf(v[o], 0.f);
                store_bf16x16(a.A + (size_t)p * 16, v);
            }
        } else if constexpr (OUT == kLogits) {
            if (p < npix) {
                float4* z = reinterpret_cast<float4*>(a.Z + (size_t)p * 16);
#pragma unroll
                for (int j = 0; j < 4; ++j) z[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
        } else {
            double l = 0.0;
            if (p < npix) {
                float m = -INFINITY, se = 0.f;
#pragma unroll
                for (int o = 0; o < kSkipCls; ++o) m = fmaxf(m, v[o]);
                float e[kSkipCls];
#pragma unroll
                for (int o = 0; o < kSkipCls; ++o) {
                    e[o] = expf(v[o] - m);
                    se += e[o];
                }
                const int y = a.labels[p];
                float zy = v[0], d[16];
#pragma unroll
                for (int o = 0; o < 16; ++o) {
                    d[o] = o < kSkipCls ? (e[o < kSkipCls ? o : 0] / se - (o == y ? 1.f : 0.f)) * a.inv_npix : 0.f;
                    if (o < kSkipCls && o == y) zy = v[o];
                }
                store_bf16x16(a.A + (size_t)p * 16, d);
                l = (double)(logf(se) + m - zy);
            }
            for (int off = 16; off; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
            if ((t & 31) == 0) atomicAdd(a.loss, l);
        }
    }
    tc_end(s, 32);
}

// ---------------------------------------------------------------------------
// Weight gradient: D[k][o] = sum_p Xcol[p][k] dZ[p][o], and with a row of ones
// under the kpad rows of k the bias gradient sum_p dZ[p][o].  A CTA takes
// 128-pixel chunks b, b + grid, ... and adds them up in TMEM; its part goes to
// part + blockIdx.x * (16 kpad + 16) ([o][k], then [o]), and k_sum_grads adds
// the parts in block order (no float atomics: the same gradients on every
// run).
//
// Both operands have the pixels along K, while the images have the channels
// contiguous: a warp gathers 8 pixels x 8 channels (4 bytes a lane) and stores
// them transposed with stmatrix, four core matrices (512 contiguous bytes) at
// a time: 20 us for 131,072 pixels with 16 channels; 205 us element by
// element, with two divisions each.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void stmatrix_x4_trans(uint32_t addr, const uint32_t (&r)[4]) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3])
                 : "memory");
}

template <int CIN>
__global__ void __launch_bounds__(256) k_conv_bwd_weight(const bf16* __restrict__ X, Img g,
                                                         const bf16* __restrict__ dZ, int cout,
                                                         float* __restrict__ part, int* err) {
    constexpr int kpad = CIN == 16 ? 144 : 48, kb = kpad / 8;
    constexpr int mt = (kpad + 16 + 127) / 128;        // 128-row tiles of k and the row of ones
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ TcCta s;
    __shared__ uint16_t taps[128];
    uint8_t* sA = smem;                        // mt*128 x 128 (rows k, K = pixels)
    uint8_t* sB = smem + mt * 32768;           // 16 x 128 (rows o)
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int npix = g.B * g.H * g.W, nchunk = (npix + 127) / 128;
    tc_begin(s, 32);
    const uint32_t a0 = tc::smem_addr(sA), b0 = tc::smem_addr(sB);
    // rows of k past the ones' core row are never written: their D rows are
    // not read
    uint32_t phase = 0;
    bool ok = true;
    for (int ch = blockIdx.x; ch < nchunk && ok; ch += gridDim.x) {
        const int base = ch * 128;
        if (t < 128) taps[t] = (uint16_t)tap_mask(g, base + t);
        __syncthreads();
        // core row blocks: kb of X, one of ones, two of dZ; each is 16 pixel
        // groups, four per store
        for (int q = warp; q < 4 * (kb + 3); q += 8) {
            const int r = q >> 2, pg = (q & 3) * 4;
            const uint32_t c2 = 2u * (lane & 3);          // the lane's channel pair in the block
            uint32_t v[4];
            if (r < kb) {
                const int k = r * 8 + c2, tap = k / CIN, c = k % CIN;
                const int64_t sh = tap_shift(tap, g.W);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int i = (pg + m) * 8 + (lane >> 2);
                    const bool in = tap < 9 && ((taps[i] >> tap) & 1u);
                    v[m] = in ? __ldg(reinterpret_cast<const uint32_t*>(X + (base + i + sh) * CIN + c)) : 0u;
                }
            } else if (r == kb) {
#pragma unroll
                for (int m = 0; m < 4; ++m) v[m] = c2 == 0u ? 0x3F80u : 0u;      // (dZ is 0 past the last pixel)
            } else {
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int i = base + (pg + m) * 8 + (lane >> 2);
                    v[m] = i < npix ? __ldg(reinterpret_cast<const uint32_t*>(dZ + (int64_t)i * 16 + (r - kb - 1) * 8 + c2))
                                    : 0u;
                }
            }
            const uint32_t blk = r <= kb ? a0 + r * 2048 : b0 + (r - kb - 1) * 2048;
            stmatrix_x4_trans(blk + (pg + (lane >> 3)) * 128 + (lane & 7) * 16, v);
        }
        tc::fence_async_smem();
        tc::fence_before_sync();
        __syncthreads();
        if (t == 0) {
            tc::fence_after_sync();
            for (int m = 0; m < mt; ++m)
                for (int kk = 0; kk < 8; ++kk)
                    tc::mma_bf16(s.tmem + 16 * m, tc::sdesc(a0 + m * 32768 + kk * 256, 128, 2048),
                                 tc::sdesc(b0 + kk * 256, 128, 2048), tc::idesc_bf16(128, 16),
                                 (kk > 0 || ch != (int)blockIdx.x) ? 1u : 0u);
            tc::mma_commit(&s.bar);
        }
        ok = tc_wait(s, phase, err);            // the operands are read: the next chunk may replace them
        phase ^= 1u;
        ok = __syncthreads_and(ok ? 1 : 0) != 0;
    }
    float* const pw = part + (size_t)blockIdx.x * (16 * kpad + 16);
    if (warp < 4) {
        for (int m = 0; m < mt; ++m) {
            float v[16];
            tc::tmem_ld16(s.tmem + ((uint32_t)(32 * warp) << 16) + 16 * m, v);
            const int k = m * 128 + t;
            if (k < kpad) {
#pragma unroll
                for (int o = 0; o < 16; ++o) pw[(size_t)o * kpad + k] = v[o];
            } else if (k == kpad) {
#pragma unroll
                for (int o = 0; o < 16; ++o) pw[16 * kpad + o] = v[o];
            }
        }
    }
    tc_end(s, 32);
}

// The flat FP32 gradients of the three layers: the nb blocks' parts of every
// entry added in a fixed order (warp w of 32 adds parts w, w + 32, ..., the
// warps' sums follow in order), 32 entries per CTA so that the parts are read
// in full lines.  Entries of layer l: o * kpad + k, then 16 kpad + o.
struct GradParts {
    const float* part[3];
    int nb[3];
};
__global__ void __launch_bounds__(1024) k_sum_grads(GradParts a, float* __restrict__ grads) {
    const Layer ly = c_layers[blockIdx.y];
    const int per = 16 * ly.kpad + 16, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    __shared__ float sum[32][32];
    float acc = 0.f;
    if (e < per) {
        const int l = blockIdx.y, nb = l == 0 ? a.nb[0] : (l == 1 ? a.nb[1] : a.nb[2]);
        const float* src = (l == 0 ? a.part[0] : (l == 1 ? a.part[1] : a.part[2])) + e;
#pragma unroll 4
        for (int b = warp; b < nb; b += 32) acc += __ldg(src + (size_t)b * per);
    }
    sum[warp][lane] = acc;
    __syncthreads();
    if (warp != 0 || e >= per) return;
    acc = sum[0][lane];
#pragma unroll
    for (int w = 1; w < 32; ++w) acc += sum[w][lane];
    if (e < 16 * ly.kpad) {
        const int o = e / ly.kpad, k = e % ly.kpad, tap = k / ly.cin, c = k % ly.cin;
        if (o < ly.cout && tap < 9) grads[ly.offw + (o * ly.cin + c) * 9 + tap] = acc;
    } else if (e - 16 * ly.kpad < ly.cout) {
        grads[ly.offb + e - 16 * ly.kpad] = acc;
    }
}

__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        m[i] = b1 * m[i] + (1.f - b1) * g[i];
        v[i] = b2 * v[i] + (1.f - b2) * g[i] * g[i];
        w[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
    }
}

template <typename P>
bool dalloc(P** p, size_t bytes) {
    if (cudaMalloc(reinterpret_cast<void**>(p), bytes) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

size_t smem_conv(int kpad) { return 288u * kpad; }
size_t smem_bwd_weight(int kpad) { return ((kpad + 16 + 127) / 128) * 32768u + 4096u; }

}  // namespace

struct SkipNet {
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    bf16 *wf = nullptr, *wt = nullptr;      // 3 layers x (16 x 144): forward, input gradient
    // the weight gradients' per-block parts, one array per layer
    float* part = nullptr;
    int part_blocks = 0;                    // most blocks of one layer
    int* err = nullptr;
    double* loss = nullptr;
    int64_t adam_t = 0;
    SkipWork work;
};

static void pack(SkipNet* n, cudaStream_t st) {
    k_pack<<<dim3(1, 3), 256, 0, st>>>(n->params, n->wf, n->wt);
}

SkipNet* skipnet_create(uint32_t seed) {
    static bool attrs = false;
    if (!attrs) {
        cudaFuncSetAttribute(k_conv_bwd_weight<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem_bwd_weight(144));
        attrs = true;
    }
    SkipNet* n = new SkipNet;
    bool ok = dalloc(&n->params, sizeof(float) * kSkipParams) && dalloc(&n->grads, sizeof(float) * kSkipParams) &&
              dalloc(&n->m, sizeof(float) * kSkipParams) && dalloc(&n->v, sizeof(float) * kSkipParams) &&
              dalloc(&n->wf, sizeof(bf16) * 3 * 16 * 144) && dalloc(&n->wt, sizeof(bf16) * 3 * 16 * 144) &&
              dalloc(&n->err, sizeof(int)) && dalloc(&n->loss, sizeof(double));
    if (!ok) {
        skipnet_destroy(n);
        return nullptr;
    }
    cudaMemset(n->m, 0, sizeof(float) * kSkipParams);
    cudaMemset(n->v, 0, sizeof(float) * kSkipParams);
    cudaMemset(n->err, 0, sizeof(int));
    // He initialisation from a seeded xorshift + Box-Muller on the host
    std::vector<float> h(kSkipParams, 0.f);
    uint64_t s = 0x9E3779B97F4A7C15ull ^ seed;
    auto uni = [&]() {
        s ^= s << 13;
        s ^= s >> 7;
        s ^= s << 17;
        return ((s >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    };
    for (const Layer& ly : kLayers) {
        const double sd = std::sqrt(2.0 / (9.0 * ly.cin));
        for (int i = 0; i < ly.cout * ly.cin * 9; ++i) {
            const double u1 = uni(), u2 = uni();
            h[ly.offw + i] = (float)(sd * std::sqrt(-2.0 * std::log(u1)) * std::cos(6.283185307179586 * u2));
        }
    }
    skipnet_set_params(n, h.data(), kSkipParams);
    return n;
}

void skipnet_destroy(SkipNet* n) {
    if (!n) return;
    for (void* p : {(void*)n->params, (void*)n->grads, (void*)n->m, (void*)n->v, (void*)n->wf, (void*)n->wt,
                    (void*)n->err, (void*)n->loss, (void*)n->part})
        if (p) cudaFree(p);
    skipwork_free(&n->work);
    delete n;
}

bool skipnet_set_params(SkipNet* n, const float* host, int64_t cnt) {
    if (cnt != kSkipParams) return false;
    if (cudaMemcpy(n->params, host, sizeof(float) * kSkipParams, cudaMemcpyHostToDevice) != cudaSuccess) return false;
    pack(n, 0);
    return cudaDeviceSynchronize() == cudaSuccess;
}

bool skipnet_get_params(const SkipNet* n, float* host, int64_t cnt) {
    if (cnt != kSkipParams) return false;
    return cudaMemcpy(host, n->params, sizeof(float) * kSkipParams, cudaMemcpyDeviceToHost) == cudaSuccess;
}

int* skipnet_err(SkipNet* n) { return n->err; }

bool skipwork_reserve(SkipWork* w, int64_t npix) {
    if (w->cap >= npix) return true;
    skipwork_free(w);
    const size_t nf = sizeof(float) * 16 * npix, nb = sizeof(bf16) * 16 * npix;
    bool ok = dalloc(&w->A1, nb) && dalloc(&w->A2, nb) && dalloc(&w->Z3, nf) && dalloc(&w->dZ1, nb) &&
              dalloc(&w->dZ2, nb) && dalloc(&w->dZ3, nb);
    if (!ok) {
        skipwork_free(w);
        return false;
    }
    w->cap = npix;
    return true;
}

void skipwork_free(SkipWork* w) {
    for (void* p : {(void*)w->A1, (void*)w->A2, (void*)w->Z3, (void*)w->dZ1, (void*)w->dZ2, (void*)w->dZ3})
        if (p) cudaFree(p);
    *w = SkipWork();
}

// the two hidden layers: activations A1, A2
static ConvArgs hidden_layers(const SkipNet* n, const bf16* x, int nimg, int H, int W, SkipWork* w, cudaStream_t st) {
    const int nb = (nimg * H * W + 127) / 128;
    ConvArgs a = {};
    a.X = x;
    a.g = Img{nimg, H, W, 4};
    a.w = n->wf;
    a.bias = n->params + kLayers[0].offb;
    a.cout = 16;
    a.A = w->A1;
    a.err = n->err;
    k_conv<4, kActivate><<<nb, 128, smem_conv(48), st>>>(a);
    a.X = w->A1;
    a.g.cin = 16;
    a.w = n->wf + 16 * 144;
    a.bias = n->params + kLayers[1].offb;
    a.A = w->A2;
    k_conv<16, kActivate><<<nb, 128, smem_conv(144), st>>>(a);
    a.X = w->A2;
    a.w = n->wf + 2 * 16 * 144;
    a.bias = n->params + kLayers[2].offb;
    a.cout = kLayers[2].cout;
    return a;                                // the last layer's, its output left to the caller
}

cudaError_t skipnet_forward(const SkipNet* n, const bf16* x, int nimg, int H, int W, SkipWork* w,
                            cudaStream_t st) {
    const int npix = nimg * H * W;
    if (w->cap < npix) return cudaErrorInvalidValue;
    ConvArgs a = hidden_layers(n, x, nimg, H, W, w, st);
    a.A = nullptr;
    a.Z = w->Z3;
    k_conv<16, kLogits><<<(npix + 127) / 128, 128, smem_conv(144), st>>>(a);
    return cudaGetLastError();
}

// Forward + loss + backward; gradients (flat FP32) in n->grads, loss in n->loss.
static cudaError_t skipnet_backprop(SkipNet* n, const bf16* x, const uint8_t* labels, int nimg, int H, int W,
                                    cudaStream_t st) {
    SkipWork* w = &n->work;
    const int npix = nimg * H * W;
    if (!skipwork_reserve(w, npix)) return cudaErrorMemoryAllocation;
    const int nb = (npix + 127) / 128;
    // three CTAs of the widest weight gradient (70 KB of operands) per SM
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int nw = std::min(nb, 3 * nsm);
    constexpr size_t per = 16 * 144 + 16;
    if (n->part_blocks < nw) {
        if (n->part) cudaFree(n->part);
        n->part = nullptr;
        n->part_blocks = 0;
        if (!dalloc(&n->part, sizeof(float) * 3 * per * nw)) return cudaErrorMemoryAllocation;
        n->part_blocks = nw;
    }
    cudaMemsetAsync(n->loss, 0, sizeof(double), st);
    ConvArgs a = hidden_layers(n, x, nimg, H, W, w, st);
    a.A = w->dZ3;
    a.labels = labels;
    a.inv_npix = 1.f / npix;
    a.loss = n->loss;
    k_conv<16, kLoss><<<nb, 128, smem_conv(144), st>>>(a);
    const bf16* acts[3] = {x, w->A1, w->A2};
    bf16* dZ[3] = {w->dZ1, w->dZ2, w->dZ3};
    GradParts gp;
    for (int l = 2; l >= 0; --l) {
        const Layer ly = kLayers[l];
        const Img g{nimg, H, W, ly.cin};
        float* part = n->part + (size_t)l * per * n->part_blocks;
        gp.part[l] = part;
        gp.nb[l] = nw;
        if (l > 0) {
            k_conv_bwd_weight<16><<<nw, 256, smem_bwd_weight(144), st>>>(acts[l], g, dZ[l], ly.cout, part, n->err);
            // gradient w.r.t. this layer's input, through the layer below's relu
            ConvArgs b = {};
            b.X = dZ[l];
            b.g = Img{nimg, H, W, 16};
            b.w = n->wt + l * 16 * 144;
            b.A = dZ[l - 1];
            b.act = acts[l];
            b.err = n->err;
            k_conv<16, kInputGrad><<<nb, 128, smem_conv(144), st>>>(b);
        } else {
            k_conv_bwd_weight<4><<<nw, 256, smem_bwd_weight(48), st>>>(acts[l], g, dZ[l], ly.cout, part, n->err);
        }
    }
    k_sum_grads<<<dim3((unsigned)((per + 31) / 32), 3), 1024, 0, st>>>(gp, n->grads);
    return cudaGetLastError();
}

}  // namespace hwfv1

// ---------------------------------------------------------------------------
// C ABI of the network (include/hwfv1.h)
// ---------------------------------------------------------------------------
namespace {
hwfv1_status net_status(hwfv1::SkipNet* n, cudaError_t e) {
    if (e != cudaSuccess) return HWFV1_ERR_CUDA;
    int err = 0;
    if (cudaMemcpy(&err, hwfv1::skipnet_err(n), sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess)
        return HWFV1_ERR_CUDA;
    return err ? HWFV1_ERR_TIMEOUT : HWFV1_OK;
}
bool image_ok(int nimg, int H, int W) {
    return nimg >= 1 && H >= 1 && W >= 1 && (int64_t)nimg * H * W <= (1ll << 28);
}
}  // namespace

extern "C" {

int32_t hwfv1_skipnet_num_params(void) { return hwfv1::kSkipParams; }

hwfv1_status hwfv1_skipnet_create(uint32_t seed, hwfv1_skipnet** out) {
    if (!out) return HWFV1_ERR_INVALID_SPEC;
    *out = nullptr;
    hwfv1::SkipNet* n = hwfv1::skipnet_create(seed);
    if (!n) return HWFV1_ERR_OOM;
    *out = new hwfv1_skipnet{n};
    return cudaDeviceSynchronize() == cudaSuccess ? HWFV1_OK : HWFV1_ERR_CUDA;
}

hwfv1_status hwfv1_skipnet_set_params(hwfv1_skipnet* s, const float* host, int64_t n) {
    if (!s || !host) return HWFV1_ERR_INVALID_SPEC;
    return hwfv1::skipnet_set_params(s->net, host, n) ? HWFV1_OK : HWFV1_ERR_INVALID_SPEC;
}

hwfv1_status hwfv1_skipnet_get_params(hwfv1_skipnet* s, float* host, int64_t n) {
    if (!s || !host) return HWFV1_ERR_INVALID_SPEC;
    return hwfv1::skipnet_get_params(s->net, host, n) ? HWFV1_OK : HWFV1_ERR_INVALID_SPEC;
}

hwfv1_status hwfv1_skipnet_forward(hwfv1_skipnet* s, const uint16_t* x, int32_t nimg, int32_t H, int32_t W,
                                   float* logits) {
    if (!s || !x || !logits || !image_ok(nimg, H, W)) return HWFV1_ERR_INVALID_SPEC;
    hwfv1::SkipNet* n = s->net;
    const int64_t npix = (int64_t)nimg * H * W;
    if (!hwfv1::skipwork_reserve(&n->work, npix)) return HWFV1_ERR_OOM;
    cudaError_t e = hwfv1::skipnet_forward(n, reinterpret_cast<const __nv_bfloat16*>(x), nimg, H, W, &n->work, 0);
    if (e == cudaSuccess)
        e = cudaMemcpy(logits, n->work.Z3, sizeof(float) * 16 * npix, cudaMemcpyDeviceToDevice);
    return net_status(n, e);
}

hwfv1_status hwfv1_skipnet_gradients(hwfv1_skipnet* s, const uint16_t* x, const uint8_t* labels, int32_t nimg,
                                     int32_t H, int32_t W, double* loss, float* grads_host) {
    if (!s || !x || !labels || !image_ok(nimg, H, W)) return HWFV1_ERR_INVALID_SPEC;
    hwfv1::SkipNet* n = s->net;
    cudaError_t e = hwfv1::skipnet_backprop(n, reinterpret_cast<const __nv_bfloat16*>(x), labels, nimg, H, W, 0);
    if (e == cudaSuccess && loss) {
        double l = 0;
        e = cudaMemcpy(&l, n->loss, sizeof(double), cudaMemcpyDeviceToHost);
        *loss = l / ((double)nimg * H * W);
    }
    if (e == cudaSuccess && grads_host)
        e = cudaMemcpy(grads_host, n->grads, sizeof(float) * hwfv1::kSkipParams, cudaMemcpyDeviceToHost);
    return net_status(n, e);
}

hwfv1_status hwfv1_skipnet_train(hwfv1_skipnet* s, const uint16_t* x, const uint8_t* labels, int32_t nimg,
                                 int32_t H, int32_t W, int32_t batch, int32_t epochs, float lr, uint32_t seed,
                                 double* last_loss) {
    if (!s || !x || !labels || !image_ok(nimg, H, W) || batch < 1 || batch > nimg || epochs < 0 || !(lr > 0.f))
        return HWFV1_ERR_INVALID_SPEC;
    hwfv1::SkipNet* n = s->net;
    const int nbatch = nimg / batch;
    const int64_t per = (int64_t)batch * H * W;
    std::vector<int> order(nbatch);
    uint64_t r = 0x2545F4914F6CDD1Dull ^ seed;
    cudaError_t e = cudaSuccess;
    double ls = 0.0;
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        for (int i = 0; i < nbatch; ++i) order[i] = i;
        for (int i = nbatch - 1; i > 0; --i) {          // Fisher-Yates with xorshift
            r ^= r << 13;
            r ^= r >> 7;
            r ^= r << 17;
            const int j = (int)(r % (uint64_t)(i + 1));
            std::swap(order[i], order[j]);
        }
        for (int bi = 0; bi < nbatch && e == cudaSuccess; ++bi) {
            const int b = order[bi];
            const __nv_bfloat16* xb = reinterpret_cast<const __nv_bfloat16*>(x) + (size_t)b * per * 4;
            e = hwfv1::skipnet_backprop(n, xb, labels + (size_t)b * per, batch, H, W, 0);
            n->adam_t++;
            const float b1 = 0.9f, b2 = 0.999f;
            const float c1 = 1.f - std::pow(b1, (float)n->adam_t), c2 = 1.f - std::pow(b2, (float)n->adam_t);
            hwfv1::k_adam<<<(hwfv1::kSkipParams + 255) / 256, 256>>>(n->params, n->grads, n->m, n->v,
                                                                    hwfv1::kSkipParams, lr, b1, b2, 1e-8f, c1, c2);
            hwfv1::pack(n, 0);
            if (e == cudaSuccess) e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess && last_loss) {
        e = cudaMemcpy(&ls, n->loss, sizeof(double), cudaMemcpyDeviceToHost);
        *last_loss = ls / (double)per;
    }
    return net_status(n, e);
}

void hwfv1_skipnet_destroy(hwfv1_skipnet* s) {
    if (!s) return;
    hwfv1::skipnet_destroy(s->net);
    delete s;
}

}  // extern "C"
