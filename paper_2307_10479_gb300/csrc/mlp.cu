// Learned early stop of the search (not in the paper; the paper stops by the eps test only).
// A 12 -> 64 -> 64 -> 2 perceptron with ReLU scores, after every hop, whether the result list
// can still change; the search stops when the "stop" logit beats "continue" by a threshold, and
// the eps test of Alg. 1 still stops it no later than the plain method would.
//
// Training kernels (float32), all deterministic: one block runs forward and backward for up to
// 128 samples with every activation in shared memory, then sums each parameter's gradient over
// its samples in a fixed order; a second kernel sums the block partials in block order and a
// third applies Adam. Parameter layout (5,122 floats): W1 [64][12], b1, W2 [64][64], b2,
// W3 [2][64], b3 (logit 0 = continue, logit 1 = stop); loss = mean softmax cross-entropy.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <string>

#include "deg_internal.h"

namespace deg {
namespace {

constexpr int IN = kStopFeatures, H = 64, OUT = 2;
constexpr int OW1 = 0, OB1 = OW1 + H * IN, OW2 = OB1 + H, OB2 = OW2 + H * H, OW3 = OB2 + H, OB3 = OW3 + OUT * H;
constexpr int NP = OB3 + OUT;
static_assert(NP == kStopParams, "parameter count");
constexpr int BS = 128;       // samples per block
constexpr int kTrainThreads = 256;
constexpr int LD = BS + 4;    // row stride of the activation tiles [feature][sample]: float4 reads of 8 rows miss each other's banks
constexpr int LW = H + 4;     // of the transposed W2

// (out[4], 8 samples) += w4 (x) (a, b): one step of a 4 x 8 register tile.
__device__ __forceinline__ void outer(float (&acc)[4][8], const float4& w, const float4& a, const float4& b) {
    const float wv[4] = {w.x, w.y, w.z, w.w}, xv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(wv[i], xv[j], acc[i][j]);
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float s) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
}

// Forward and backward of one block's samples. The three 64 x 64 products (layer 2 forward, its input
// gradient, its weight gradient) are nearly all of the work; each runs from register tiles, three or eight float4
// reads of shared memory for 32 or 64 FMAs, where one thread per sample and per parameter read two values per FMA.
// Activations are stored feature by feature, so that a tile's samples are contiguous. Bound by the
// SMs that have a block (64 of 152 at 8,192 samples: 29 us, where a thread per sample took 74).
__global__ void __launch_bounds__(kTrainThreads) mlp_fwd_bwd_kernel(const float* __restrict__ w, const float* __restrict__ x,
                                                                    const int32_t* __restrict__ labels, int64_t count,
                                                                    float* __restrict__ partial, float* __restrict__ loss_partial) {
    extern __shared__ __align__(16) float sm[];
    float* w2 = sm;                       // [H][H]
    float* w2t = w2 + H * H;              // [H][LW], transposed
    float* rest = w2t + H * LW;           // W1, b1, b2, W3, b3
    float* w1 = rest;
    float* b1 = w1 + H * IN;
    float* b2 = b1 + H;
    float* w3 = b2 + H;
    float* b3 = w3 + OUT * H;
    float* xs = b3 + 4;                   // [IN][LD]
    float* h1 = xs + IN * LD;             // [H][LD] each
    float* h2 = h1 + H * LD;
    float* d1 = h2 + H * LD;
    float* d2 = d1 + H * LD;
    float* dz = d2 + H * LD;              // [OUT][LD]
    float* lsum = dz + OUT * LD;          // [BS]
    const int t = threadIdx.x;
    const int64_t s0 = (int64_t)blockIdx.x * BS;
    for (int i = t; i < H * H; i += kTrainThreads) {
        const float v = w[OW2 + i];
        w2[i] = v;
        w2t[(i % H) * LW + i / H] = v;
    }
    for (int i = t; i < H * IN; i += kTrainThreads) w1[i] = w[OW1 + i];
    for (int i = t; i < H; i += kTrainThreads) {
        b1[i] = w[OB1 + i];
        b2[i] = w[OB2 + i];
    }
    for (int i = t; i < OUT * H; i += kTrainThreads) w3[i] = w[OW3 + i];
    if (t < OUT) b3[t] = w[OB3 + t];
    for (int i = t; i < BS * IN; i += kTrainThreads) xs[(i % IN) * LD + i / IN] = s0 + i / IN < count ? x[s0 * IN + i] : 0.f;
    __syncthreads();
    const int s8 = (t & 15) * 8, r4 = (t >> 4) * 4;           // this thread's samples and features
    float acc[4][8];
    // layer 1
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = b1[r4 + i];
#pragma unroll
    for (int k = 0; k < IN; ++k)
        outer(acc, make_float4(w1[r4 * IN + k], w1[(r4 + 1) * IN + k], w1[(r4 + 2) * IN + k], w1[(r4 + 3) * IN + k]),
              *reinterpret_cast<const float4*>(xs + k * LD + s8), *reinterpret_cast<const float4*>(xs + k * LD + s8 + 4));
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) h1[(r4 + i) * LD + s8 + j] = fmaxf(acc[i][j], 0.f);
    __syncthreads();
    // layer 2
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = b2[r4 + i];
#pragma unroll 4
    for (int k = 0; k < H; ++k)
        outer(acc, *reinterpret_cast<const float4*>(w2t + k * LW + r4), *reinterpret_cast<const float4*>(h1 + k * LD + s8),
              *reinterpret_cast<const float4*>(h1 + k * LD + s8 + 4));
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) h2[(r4 + i) * LD + s8 + j] = fmaxf(acc[i][j], 0.f);
    __syncthreads();
    // layer 3 and the loss: a sample a thread. dz = softmax - onehot (the 1/count of the mean is applied at the
    // reduction)
    if (t < BS) {
        const bool live = s0 + t < count;
        float z[OUT];
        for (int o = 0; o < OUT; ++o) {
            float a = b3[o];
#pragma unroll 16
            for (int i = 0; i < H; ++i) a = fmaf(w3[o * H + i], h2[i * LD + t], a);
            z[o] = a;
        }
        const float m = fmaxf(z[0], z[1]);
        const float lse = m + logf(expf(z[0] - m) + expf(z[1] - m));
        const int y = live ? labels[s0 + t] : 0;
        lsum[t] = live ? lse - z[y] : 0.f;
        for (int o = 0; o < OUT; ++o) dz[o * LD + t] = live ? expf(z[o] - lse) - (o == y ? 1.f : 0.f) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float g = fmaf(w3[H + r4 + i], dz[LD + s8 + j], w3[r4 + i] * dz[s8 + j]);
            d2[(r4 + i) * LD + s8 + j] = h2[(r4 + i) * LD + s8 + j] > 0.f ? g : 0.f;
            acc[i][j] = 0.f;
        }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < H; ++k)
        outer(acc, *reinterpret_cast<const float4*>(w2 + k * H + r4), *reinterpret_cast<const float4*>(d2 + k * LD + s8),
              *reinterpret_cast<const float4*>(d2 + k * LD + s8 + 4));
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) d1[(r4 + i) * LD + s8 + j] = h1[(r4 + i) * LD + s8 + j] > 0.f ? acc[i][j] : 0.f;
    __syncthreads();
    // parameter gradients: sums over this block's samples, in sample order
    float* out = partial + (int64_t)blockIdx.x * NP;
    {
        const int i0 = t & 15, j0 = t >> 4;                   // W2[j][i], rows 16 apart
        float g[4][4] = {};
#pragma unroll 2
        for (int s = 0; s < BS; s += 4) {
            float4 a[4], b[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                a[e] = *reinterpret_cast<const float4*>(d2 + (j0 + 16 * e) * LD + s);
                b[e] = *reinterpret_cast<const float4*>(h1 + (i0 + 16 * e) * LD + s);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int f = 0; f < 4; ++f) g[e][f] = dot4(a[e], b[f], g[e][f]);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int f = 0; f < 4; ++f) out[OW2 + (j0 + 16 * e) * H + i0 + 16 * f] = g[e][f];
    }
    // W1 (768), W3 (128) and the biases (130): a dot product of two rows, or the sum of one
    for (int p = t; p < H * IN + OUT * H + 2 * H + OUT; p += kTrainThreads) {
        const float *a, *b = nullptr;
        int at = p;
        if (p < H * IN) {
            a = d1 + (p / IN) * LD;
            b = xs + (p % IN) * LD;
            at = OW1 + p;
        } else if ((at = p - H * IN) < OUT * H) {
            a = dz + (at / H) * LD;
            b = h2 + (at % H) * LD;
            at += OW3;
        } else if ((at -= OUT * H) < H) {
            a = d1 + at * LD;
            at += OB1;
        } else if ((at -= H) < H) {
            a = d2 + at * LD;
            at += OB2;
        } else {
            a = dz + (at - H) * LD;
            at += OB3 - H;
        }
        float g = 0.f;
        const float4 one = make_float4(1.f, 1.f, 1.f, 1.f);
#pragma unroll 8
        for (int s = 0; s < BS; s += 4) {
            const float4 u = *reinterpret_cast<const float4*>(a + s);
            g = dot4(u, b ? *reinterpret_cast<const float4*>(b + s) : one, g);
        }
        out[at] = g;
    }
    if (t < 32) {
        float l = (lsum[t] + lsum[t + 32]) + (lsum[t + 64] + lsum[t + 96]);
#pragma unroll
        for (int m = 16; m; m >>= 1) l += __shfl_xor_sync(0xffffffffu, l, m);
        if (t == 0) loss_partial[blockIdx.x] = l;
    }
}

__global__ void mlp_reduce_kernel(const float* __restrict__ partial, const float* __restrict__ loss_partial,
                                  int nblocks, int64_t count, float* __restrict__ grad, float* __restrict__ loss) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const float inv = 1.f / (float)count;
    if (p < NP) {
        float g = 0.f;
#pragma unroll 8
        for (int b = 0; b < nblocks; ++b) g += partial[(int64_t)b * NP + p];
        grad[p] = g * inv;
    }
    if (p == 0 && loss) {
        float l = 0.f;
        for (int b = 0; b < nblocks; ++b) l += loss_partial[b];
        *loss = l * inv;
    }
}

__global__ void mlp_adam_kernel(float* w, float* m, float* v, const float* g, int step, float lr) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NP) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float mp = b1 * m[p] + (1.f - b1) * g[p];
    const float vp = b2 * v[p] + (1.f - b2) * g[p] * g[p];
    m[p] = mp;
    v[p] = vp;
    const float mh = mp / (1.f - powf(b1, (float)step));
    const float vh = vp / (1.f - powf(b2, (float)step));
    w[p] -= lr * mh / (sqrtf(vh) + eps);
}

__global__ void mlp_predict_kernel(const float* __restrict__ w, const float* __restrict__ x, int64_t count,
                                   float* __restrict__ p_stop) {
    __shared__ float ws[NP];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) ws[i] = w[i];
    __syncthreads();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= count) return;
    float xi[IN], h1[H], z[OUT];
    for (int i = 0; i < IN; ++i) xi[i] = x[s * IN + i];
    for (int j = 0; j < H; ++j) {
        float a = ws[OB1 + j];
        for (int i = 0; i < IN; ++i) a = fmaf(ws[OW1 + j * IN + i], xi[i], a);
        h1[j] = fmaxf(a, 0.f);
    }
    for (int o = 0; o < OUT; ++o) z[o] = ws[OB3 + o];
    for (int j = 0; j < H; ++j) {
        float a = ws[OB2 + j];
        for (int i = 0; i < H; ++i) a = fmaf(ws[OW2 + j * H + i], h1[i], a);
        a = fmaxf(a, 0.f);
        for (int o = 0; o < OUT; ++o) z[o] = fmaf(ws[OW3 + o * H + j], a, z[o]);
    }
    p_stop[s] = 1.f / (1.f + expf(z[0] - z[1]));
}

// bfloat16 copy for inference inside the search, with W1 and W2 transposed ([in][out]) so the
// 32 lanes of a warp read consecutive outputs: W1t [12][64], b1, W2t [64][64], b2, W3, b3.
__global__ void pack_inference_kernel(const float* w, __nv_bfloat16* out) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NP) return;
    int src = p;
    if (p < OB1) {
        const int i = p / H, j = p % H;      // out position [i][j] <- W1[j][i]
        src = OW1 + j * IN + i;
    } else if (p >= OW2 && p < OB2) {
        const int i = (p - OW2) / H, j = (p - OW2) % H;
        src = OW2 + j * H + i;
    }
    out[p] = __float2bfloat16_rn(w[src]);
}

size_t fwd_bwd_smem() { return sizeof(float) * (H * H + H * LW + H * IN + 2 * H + OUT * H + 4 + (IN + 4 * H + OUT) * LD + BS); }

}  // namespace

int mlp_loss_grad(const float* w, const float* x, const int32_t* labels, int64_t count, float* grad, float* loss,
                  float* scratch, deg_stream_t stream, std::string* why) {
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const int nb = (int)((count + BS - 1) / BS);
    float* partial = scratch;
    float* lpart = scratch + (int64_t)nb * NP;
    cudaError_t e = cudaFuncSetAttribute(mlp_fwd_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)fwd_bwd_smem());
    if (e != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    mlp_fwd_bwd_kernel<<<nb, kTrainThreads, fwd_bwd_smem(), st>>>(w, x, labels, count, partial, lpart);
    mlp_reduce_kernel<<<(NP + 255) / 256, 256, 0, st>>>(partial, lpart, nb, count, grad, loss);
    if ((e = cudaGetLastError()) != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    return 0;
}

int64_t mlp_scratch_floats(int64_t count) {
    const int64_t nb = (count + BS - 1) / BS;
    return nb * NP + nb;
}

int mlp_adam(float* w, float* m, float* v, const float* g, int step, float lr, deg_stream_t stream, std::string* why) {
    mlp_adam_kernel<<<(NP + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(w, m, v, g, step, lr);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    return 0;
}

int mlp_predict(const float* w, const float* x, int64_t count, float* p_stop, deg_stream_t stream, std::string* why) {
    mlp_predict_kernel<<<(unsigned)((count + 127) / 128), 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(w, x, count, p_stop);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    return 0;
}

int mlp_pack_inference(const float* w, uint16_t* out, deg_stream_t stream, std::string* why) {
    pack_inference_kernel<<<(NP + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        w, reinterpret_cast<__nv_bfloat16*>(out));
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return *why = cudaGetErrorString(e), (int)e;
    return 0;
}

}  // namespace deg
