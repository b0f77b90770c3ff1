// Learned pivot: a small MLP g -> coefficients on a stored basis U of
// converged eigenvectors, trained on this library's own solves.  The paper
// has no learned component; this is the proposal step in front of the
// bootstrapped pivot, which stays the fallback.
//
//   h1 = gelu(W1 g + b1)   1 -> H     (gelu(x) = x/2 (1 + erf(x/sqrt 2)))
//   h2 = gelu(W2 h1 + b2)  H -> H
//   y  = W3 h2 + b3        H -> O  (O = nbasis * b, reshaped nbasis x b)
//
// Weights are used in BF16 (round-to-nearest-even copies of FP32 master
// weights), activations and accumulation are FP32.  Loss: mean squared error.
// Optimiser: Adam (Kingma & Ba 2015) on the FP32 masters.  One training epoch
// (forward, loss, backward, Adam) is captured once in a CUDA graph and
// replayed.  The pivot P = U C(g) reuses the Ritz-vector kernel.
#include <cuda_bf16.h>

#include <algorithm>
#include <vector>

#include "common.cuh"

struct bbl_mlp {
    int hidden = 0, out = 0, nparams = 0;
    int cap_batch = 0;
    bbl::DevBuf params, grads, m, v, wbf, act, tstep, lossbuf;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int graph_batch = -1;
    const void* graph_g = nullptr;
    const void* graph_t = nullptr;
    float graph_lr = 0.f;
    ~bbl_mlp() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }
    // packed offsets (FP32 params): W1[H], b1[H], W2[H*H], b2[H], W3[O*H], b3[O]
    int oW1() const { return 0; }
    int ob1() const { return hidden; }
    int oW2() const { return 2 * hidden; }
    int ob2() const { return 2 * hidden + hidden * hidden; }
    int oW3() const { return 3 * hidden + hidden * hidden; }
    int ob3() const { return 3 * hidden + hidden * hidden + out * hidden; }
};

namespace bbl {
namespace {

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}
__device__ __forceinline__ float bf(const __nv_bfloat16* w, int i) { return __bfloat162float(w[i]); }

// activations layout per sample: z1[H] h1[H] z2[H] h2[H] dz1[H] dz2[H] y[O] dy[O]
//
// A step is small (48 samples, hidden 128, 512 outputs: 8 MFLOP forward, 0.3 MB of
// parameters), so its kernels are bound by the latency of dependent loads:
// they spread the weight rows over the SMs, read them along their contiguous
// dimension and keep a tile of samples per weight in registers.  (One CTA per
// sample with a thread per output row read the weights with a stride of a row:
// 44 us forward, 21 us backward, 74 us a step; the step's five kernels now take 28 us:
// 4.2, 4.4, 10.7, 5.8 and 3.4.)
constexpr int kFwS = 16;          // samples per CTA, forward
constexpr int kFwThreads = 256;
constexpr int kFwWarps = kFwThreads / 32;
constexpr int kBwS = 4;           // samples per CTA, backward
constexpr int kBwThreads = 1024;

// v[s] summed over the warp for s = lane / 2 (16 values, 16 shuffles)
__device__ __forceinline__ float warp_sum16(float (&v)[kFwS]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int off = 16, h = kFwS / 2; off > 1; off >>= 1, h >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int x = 0; x < kFwS / 2; ++x)
            if (x < h) {
                const float send = up ? v[x] : v[x + h], keep = up ? v[x + h] : v[x];
                v[x] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// One layer for 16 samples, a warp per output row o: acc = sum_i W[o][i] in[s][i]
// (in: the samples' inputs in shared memory, rows of `in_dim`); the lane pair of
// sample s gets row o's sum for it.
__device__ __forceinline__ float row_dot16(const __nv_bfloat16* __restrict__ Wrow, const float* in, int in_dim) {
    const int lane = threadIdx.x & 31;
    float acc[kFwS];
#pragma unroll
    for (int q = 0; q < kFwS; ++q) acc[q] = 0.0f;
    for (int i0 = 0; i0 < in_dim; i0 += 128) {
        float w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u + lane;
            w[u] = i < in_dim ? __bfloat162float(Wrow[i]) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u + lane;
            if (i < in_dim) {
#pragma unroll
                for (int q = 0; q < kFwS; ++q) acc[q] = fmaf(w[u], in[q * in_dim + i], acc[q]);
            }
        }
    }
    return warp_sum16(acc);
}

// h1 of 16 samples (recomputed by every CTA; the first row of CTAs stores
// it), then z2 and h2 of 8 rows
__global__ void __launch_bounds__(kFwThreads) hidden_kernel(int batch, int H, int O, const float* __restrict__ P,
                                                            const __nv_bfloat16* __restrict__ Wb,
                                                            const float* __restrict__ g, float* __restrict__ act) {
    extern __shared__ float sh[];
    const int s0 = blockIdx.x * kFwS, ns = min(kFwS, batch - s0);
    const size_t st = 6 * H + 2 * O;
    const float* b1 = P + H;
    const float* b2 = P + 2 * H + H * H;
    for (int e = threadIdx.x; e < kFwS * H; e += kFwThreads) {
        const int q = e / H, i = e - q * H;
        float hv = 0.0f;
        if (q < ns) {
            const float z = fmaf(bf(Wb, i), g[s0 + q], b1[i]);
            hv = gelu(z);
            if (blockIdx.y == 0) {
                act[(s0 + q) * st + i] = z;
                act[(s0 + q) * st + H + i] = hv;
            }
        }
        sh[e] = hv;
    }
    __syncthreads();
    const int o = blockIdx.y * kFwWarps + (threadIdx.x >> 5);
    if (o >= H) return;
    const float z = row_dot16(Wb + H + (size_t)o * H, sh, H) + b2[o];
    const int q = (threadIdx.x & 31) >> 1;
    if ((threadIdx.x & 1) == 0 && q < ns) {
        act[(s0 + q) * st + 2 * H + o] = z;
        act[(s0 + q) * st + 3 * H + o] = gelu(z);
    }
}

// The squares are summed in units of the power of two above their number, which
// rounds nothing: their plain sum could overflow where the mean does not.
__device__ __forceinline__ float loss_unit(int batch, int O) {
    const int e = (__float_as_int((float)batch * (float)O) >> 23) - 127;  // the number is in [2^e, 2^(e+1))
    return __int_as_float((126 - e) << 23);
}

// y of 8 output rows for 16 samples; with a target also dy = 2 (y - t) / N and
// the CTA's sum of squares (in units of loss_unit)
__global__ void __launch_bounds__(kFwThreads) output_kernel(int batch, int H, int O, const float* __restrict__ P,
                                                            const __nv_bfloat16* __restrict__ Wb,
                                                            float* __restrict__ act, float* __restrict__ y_out,
                                                            const float* __restrict__ target,
                                                            float* __restrict__ lossp) {
    extern __shared__ float sh[];
    __shared__ float red[kFwWarps];
    const int s0 = blockIdx.x * kFwS, ns = min(kFwS, batch - s0);
    const size_t st = 6 * H + 2 * O;
    for (int e = threadIdx.x; e < kFwS * H; e += kFwThreads) {
        const int q = e / H, i = e - q * H;
        sh[e] = q < ns ? act[(s0 + q) * st + 3 * H + i] : 0.0f;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, o = blockIdx.y * kFwWarps + warp;
    float l = 0.0f;
    if (o < O) {
        const float y = row_dot16(Wb + H + H * H + (size_t)o * H, sh, H) + P[3 * H + H * H + O * H + o];
        const int q = (threadIdx.x & 31) >> 1;
        if ((threadIdx.x & 1) == 0 && q < ns) {
            float* a = act + (s0 + q) * st;
            a[6 * H + o] = y;
            if (y_out) y_out[(size_t)(s0 + q) * O + o] = y;
            if (target) {
                const float d = y - target[(size_t)(s0 + q) * O + o];
                const float inv = 1.0f / ((float)batch * (float)O);
                a[6 * H + O + o] = 2.0f * d * inv;
                l = d * d * loss_unit(batch, O);
            }
        }
    }
    if (!target) return;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
    if ((threadIdx.x & 31) == 0) red[warp] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int w = 0; w < kFwWarps; ++w) t += red[w];
        lossp[blockIdx.x * gridDim.y + blockIdx.y] = t;
    }
}

// The whole forward pass of one sample per CTA, for networks so small that the two
// kernels' launches count: the same sums in the same order as row_dot16's.
__device__ __forceinline__ float row_dot(const __nv_bfloat16* __restrict__ Wrow, const float* in, int in_dim) {
    float acc = 0.0f;
    for (int i = threadIdx.x & 31; i < in_dim; i += 32) acc = fmaf(__bfloat162float(Wrow[i]), in[i], acc);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    return acc;
}
constexpr int kSmallNet = 1024;  // H (H + O)
__global__ void __launch_bounds__(kFwThreads) forward_small_kernel(int H, int O, const float* __restrict__ P,
                                                                   const __nv_bfloat16* __restrict__ Wb,
                                                                   const float* __restrict__ g,
                                                                   float* __restrict__ y_out) {
    __shared__ float h1[32], h2[32];  // H (H + O) <= kSmallNet: H below 32
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const float* b2 = P + 2 * H + H * H;
    if (threadIdx.x < H) h1[threadIdx.x] = gelu(fmaf(bf(Wb, threadIdx.x), g[blockIdx.x], P[H + threadIdx.x]));
    __syncthreads();
    for (int o = warp; o < H; o += kFwWarps) {
        const float z = row_dot(Wb + H + (size_t)o * H, h1, H) + b2[o];
        if (lane == 0) h2[o] = gelu(z);
    }
    __syncthreads();
    for (int o = warp; o < O; o += kFwWarps) {
        const float y = row_dot(Wb + H + H * H + (size_t)o * H, h2, H) + P[3 * H + H * H + O * H + o];
        if (lane == 0) y_out[(size_t)blockIdx.x * O + o] = y;
    }
}

// out[q][i] = sum_o W[o][i] d[q][o] for the CTA's 4 samples (d: rows of n_out in
// shared memory): a warp takes 32 V columns i, V per lane (4, one 8-byte load,
// where H is a multiple of 4), and a share of the rows o; the shares are added in
// order.  A few CTAs walk all of W, so the chain of loads per warp is what counts:
// hidden 128, 512 outputs, 48 samples: V = 1 (8 shares) 18.1 us, V = 4 (32) 10.6.  part: 32 warps x
// 4 x 32 V floats.
template <int V, typename Put>
__device__ __forceinline__ void columns_dot(const __nv_bfloat16* __restrict__ W, int H, int n_out, const float* d,
                                            float* part, Put&& put) {
    constexpr int TW = 32 * V;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles = (H + TW - 1) / TW, shares = (kBwThreads / 32) / tiles;
    const int tile = warp % tiles, share = warp / tiles;
    const int i = TW * tile + V * lane;
    float acc[kBwS][V] = {};
    if (share < shares && i < H) {
#pragma unroll 8
        for (int o = share; o < n_out; o += shares) {
            float w[V];
            if constexpr (V == 4) {
                const uint2 x = __ldg(reinterpret_cast<const uint2*>(W + (size_t)o * H + i));
                w[0] = __uint_as_float(x.x << 16);
                w[1] = __uint_as_float(x.x & 0xffff0000u);
                w[2] = __uint_as_float(x.y << 16);
                w[3] = __uint_as_float(x.y & 0xffff0000u);
            } else {
                w[0] = __bfloat162float(W[(size_t)o * H + i]);
            }
#pragma unroll
            for (int q = 0; q < kBwS; ++q)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[q][v] = fmaf(w[v], d[q * n_out + o], acc[q][v]);
        }
    }
#pragma unroll
    for (int q = 0; q < kBwS; ++q)
#pragma unroll
        for (int v = 0; v < V; ++v) part[(warp * kBwS + q) * TW + V * lane + v] = acc[q][v];
    __syncthreads();
    for (int e = threadIdx.x; e < kBwS * H; e += kBwThreads) {
        const int q = e / H, c = e - q * H;
        float t = 0.0f;
#pragma unroll 8
        for (int k = 0; k < shares; ++k) t += part[((k * tiles + c / TW) * kBwS + q) * TW + c % TW];
        put(q, c, t);
    }
    __syncthreads();
}

// backward through the activations of 4 samples: dz2, dz1
template <int V>
__global__ void __launch_bounds__(kBwThreads) backward_act_kernel(int batch, int H, int O,
                                                                  const __nv_bfloat16* __restrict__ Wb,
                                                                  float* __restrict__ act) {
    extern __shared__ float sh[];
    float* part = sh;                           // (32 warps) x 4 x 32 V
    float* dz2 = part + kBwThreads * kBwS * V;  // 4 x H
    float* dy = dz2 + kBwS * H;                 // 4 x O
    const int s0 = blockIdx.x * kBwS, ns = min(kBwS, batch - s0);
    const size_t st = 6 * H + 2 * O;
    for (int e = threadIdx.x; e < kBwS * O; e += kBwThreads) {
        const int q = e / O, o = e - q * O;
        dy[e] = q < ns ? act[(s0 + q) * st + 6 * H + O + o] : 0.0f;
    }
    __syncthreads();
    columns_dot<V>(Wb + H + H * H, H, O, dy, part, [&](int q, int i, float t) {
        float v = 0.0f;
        if (q < ns) {
            float* a = act + (s0 + q) * st;
            v = t * gelu_grad(a[2 * H + i]);
            a[5 * H + i] = v;
        }
        dz2[q * H + i] = v;
    });
    columns_dot<V>(Wb + H, H, H, dz2, part, [&](int q, int i, float t) {
        if (q < ns) {
            float* a = act + (s0 + q) * st;
            a[4 * H + i] = t * gelu_grad(a[i]);
        }
    });
}

// weight gradients, one thread per parameter, summed over the batch in order;
// the last CTA adds the partial losses
__global__ void __launch_bounds__(256) backward_w_kernel(int batch, int H, int O, const float* __restrict__ g,
                                                         const float* __restrict__ act, float* __restrict__ G,
                                                         int nloss, const float* __restrict__ lossp,
                                                         float* __restrict__ loss) {
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ float red[256];
        float l = 0.0f;
        for (int e = threadIdx.x; e < nloss; e += 256) l += lossp[e];
        red[threadIdx.x] = l;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) *loss = red[0] * (1.0f / ((float)batch * (float)O) / loss_unit(batch, O));
        return;
    }
    const int np = 3 * H + H * H + O * H + O;
    const int p = blockIdx.x * 256 + threadIdx.x;
    if (p >= np) return;
    const size_t st = 6 * H + 2 * O;
    // dG = sum_s left[s] * right[s]; right is 1 for a bias
    const float *left, *right = nullptr;
    size_t rst = st;
    if (p < H) {  // W1[o]
        left = act + 4 * H + p;
        right = g;
        rst = 1;
    } else if (p < 2 * H) {  // b1
        left = act + 4 * H + (p - H);
    } else if (p < 2 * H + H * H) {  // W2[o][i]
        const int e = p - 2 * H, o = e / H, i = e % H;
        left = act + 5 * H + o;
        right = act + H + i;
    } else if (p < 3 * H + H * H) {  // b2
        left = act + 5 * H + (p - 2 * H - H * H);
    } else if (p < 3 * H + H * H + O * H) {  // W3[o][i]
        const int e = p - 3 * H - H * H, o = e / H, i = e % H;
        left = act + 6 * H + O + o;
        right = act + 3 * H + i;
    } else {  // b3
        left = act + 6 * H + O + (p - 3 * H - H * H - O * H);
    }
    // 16 samples' loads at once, two loops: with one loop and the choice inside, the
    // loads waited for one another (128 and 512, 48 samples: 8.9 us, now 5.8; 32 and 64, 5000
    // samples: 600, now 295).
    constexpr int U = 16;
    float acc = 0.0f;
    int s = 0;
    if (right) {
        for (; s + U <= batch; s += U, left += U * st, right += U * rst) {
            float l[U], r[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                l[u] = __ldg(left + u * st);
                r[u] = __ldg(right + u * rst);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) acc = fmaf(l[u], r[u], acc);
        }
        for (; s < batch; ++s, left += st, right += rst) acc = fmaf(__ldg(left), __ldg(right), acc);
    } else {
        for (; s + U <= batch; s += U, left += U * st) {
            float l[U];
#pragma unroll
            for (int u = 0; u < U; ++u) l[u] = __ldg(left + u * st);
#pragma unroll
            for (int u = 0; u < U; ++u) acc += l[u];
        }
        for (; s < batch; ++s, left += st) acc += __ldg(left);
    }
    G[p] = acc;
}

// the BF16 copy of parameter p (W1 | W2 | W3), -1 for a bias
__device__ __forceinline__ int bf16_index(int H, int O, int p) {
    if (p < H) return p;
    if (p >= 2 * H && p < 2 * H + H * H) return H + (p - 2 * H);
    if (p >= 3 * H + H * H && p < 3 * H + H * H + O * H) return H + H * H + (p - 3 * H - H * H);
    return -1;
}

// bf16 copies of the weight matrices
__global__ void to_bf16_kernel(int H, int O, const float* __restrict__ P, __nv_bfloat16* __restrict__ Wb) {
    const int np = 3 * H + H * H + O * H + O;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < np; p += gridDim.x * blockDim.x) {
        const int w = bf16_index(H, O, p);
        if (w >= 0) Wb[w] = __float2bfloat16_rn(P[p]);
    }
}

// one Adam step, the new BF16 weights, and (by the CTA that ends last: all have
// read the step count by then) the step count; tstep[1] counts the CTAs
__global__ void __launch_bounds__(256) adam_kernel(int H, int O, float lr, float b1, float b2, float eps,
                                                   float* __restrict__ P, const float* __restrict__ G,
                                                   float* __restrict__ M, float* __restrict__ V,
                                                   __nv_bfloat16* __restrict__ Wb, int* tstep) {
    const int t = *(volatile int*)tstep + 1;
    const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
    const int p = blockIdx.x * 256 + threadIdx.x;
    if (p < 3 * H + H * H + O * H + O) {
        const float gr = G[p];
        const float m = b1 * M[p] + (1.0f - b1) * gr;
        const float v = b2 * V[p] + (1.0f - b2) * gr * gr;
        M[p] = m;
        V[p] = v;
        const float np = P[p] - lr * (m / c1) / (sqrtf(v / c2) + eps);
        P[p] = np;
        const int w = bf16_index(H, O, p);
        if (w >= 0) Wb[w] = __float2bfloat16_rn(np);
    }
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(tstep + 1, 1) == (int)gridDim.x - 1) {
        tstep[1] = 0;
        tstep[0] = t;
    }
}

__global__ void widen_kernel(int count, const float* __restrict__ y, double* __restrict__ C) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < count) C[e] = (double)y[e];
}

int loss_parts(const bbl_mlp* M, int batch) {
    return (int)(ceil_div(M->out, kFwWarps) * ceil_div(batch, kFwS));
}

bbl_status ensure_batch(bbl_mlp* M, int batch) {
    if (batch <= M->cap_batch) return BBL_OK;
    // the buffers go before the larger ones come: until both are there, no
    // capacity and no captured graph that points to them
    M->cap_batch = 0;
    if (M->exec) {
        cudaGraphExecDestroy(M->exec);
        cudaGraphDestroy(M->graph);
        M->exec = nullptr;
        M->graph = nullptr;
        M->graph_batch = -1;
    }
    BBL_TRY(M->act.alloc(sizeof(float) * (size_t)batch * (6 * M->hidden + 2 * M->out)));
    BBL_TRY(M->lossbuf.alloc(sizeof(float) * (size_t)(loss_parts(M, batch) + 8)));  // the loss, then its parts
    M->cap_batch = batch;
    return BBL_OK;
}

bbl_status launch_forward(const bbl_mlp* M, int batch, const float* g, float* y, const float* target, cudaStream_t st) {
    const int H = M->hidden, O = M->out;
    // Only the output is wanted, of a small network and a batch that the GPU holds at once:
    // one launch (hidden 16, 32 outputs, 6 samples: 26 us a call, two kernels 29)
    if (!target && y && H * (H + O) <= kSmallNet && batch <= 512) {
        forward_small_kernel<<<(unsigned)batch, kFwThreads, 0, st>>>(H, O, M->params.as<float>(),
                                                                     M->wbf.as<__nv_bfloat16>(), g, y);
        BBL_LAUNCH_CHECK();
        return BBL_OK;
    }
    const size_t sm = sizeof(float) * kFwS * H;
    static OncePerDevice hidden_once, output_once;
    BBL_TRY(allow_smem(hidden_once, hidden_kernel, kFwS * 1024 * 4));
    BBL_TRY(allow_smem(output_once, output_kernel, kFwS * 1024 * 4));
    const unsigned groups = (unsigned)ceil_div(batch, kFwS);  // in x: any batch (y holds 65535 at most, rows 512)
    hidden_kernel<<<dim3(groups, (unsigned)ceil_div(H, kFwWarps)), kFwThreads, sm, st>>>(
        batch, H, O, M->params.as<float>(), M->wbf.as<__nv_bfloat16>(), g, M->act.as<float>());
    BBL_LAUNCH_CHECK();
    output_kernel<<<dim3(groups, (unsigned)ceil_div(O, kFwWarps)), kFwThreads, sm, st>>>(
        batch, H, O, M->params.as<float>(), M->wbf.as<__nv_bfloat16>(), M->act.as<float>(), y, target,
        M->lossbuf.as<float>() + 8);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

// forward, MSE loss (into lossbuf[0]) and backward into the gradient buffer
bbl_status launch_loss_grad(bbl_mlp* M, int batch, const float* g, const float* target, cudaStream_t st) {
    const int H = M->hidden, O = M->out;
    const int V = H % 4 == 0 ? 4 : 1;
    const auto backward_act = V == 4 ? backward_act_kernel<4> : backward_act_kernel<1>;
    static OncePerDevice once1, once4;
    BBL_TRY(allow_smem(once1, backward_act_kernel<1>, sizeof(float) * (kBwThreads * kBwS + kBwS * (1024 + 4096))));
    BBL_TRY(allow_smem(once4, backward_act_kernel<4>, sizeof(float) * (kBwThreads * kBwS * 4 + kBwS * (1024 + 4096))));
    BBL_TRY(launch_forward(M, batch, g, nullptr, target, st));
    backward_act<<<(unsigned)ceil_div(batch, kBwS), kBwThreads,
                   sizeof(float) * (kBwThreads * kBwS * V + kBwS * (H + O)), st>>>(
        batch, H, O, M->wbf.as<__nv_bfloat16>(), M->act.as<float>());
    BBL_LAUNCH_CHECK();
    backward_w_kernel<<<(unsigned)ceil_div(M->nparams, 256) + 1, 256, 0, st>>>(
        batch, H, O, g, M->act.as<float>(), M->grads.as<float>(), loss_parts(M, batch), M->lossbuf.as<float>() + 8,
        M->lossbuf.as<float>());
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

bbl_status launch_adam(bbl_mlp* M, float lr, cudaStream_t st) {
    adam_kernel<<<(unsigned)ceil_div(M->nparams, 256), 256, 0, st>>>(
        M->hidden, M->out, lr, 0.9f, 0.999f, 1e-8f, M->params.as<float>(), M->grads.as<float>(), M->m.as<float>(),
        M->v.as<float>(), M->wbf.as<__nv_bfloat16>(), M->tstep.as<int>());
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

}  // namespace
bbl_status ritz_vectors(int64_t n, int b, int nblocks, int dtype, const void* Q, int k, const double* S, double* X,
                        cudaStream_t st);
}  // namespace bbl

extern "C" {

bbl_status bbl_mlp_create(int hidden, int out_dim, bbl_mlp** out) {
    using namespace bbl;
    if (!out || hidden < 1 || hidden > 1024 || out_dim < 1 || out_dim > 4096)
        return set_error(BBL_ERR_INVALID_ARG, "mlp_create: bad arguments");
    bbl_mlp* M = new bbl_mlp();
    M->hidden = hidden;
    M->out = out_dim;
    M->nparams = 3 * hidden + hidden * hidden + out_dim * hidden + out_dim;
    const size_t pb = sizeof(float) * M->nparams;
    bbl_status s;
    if ((s = M->params.alloc(pb)) != BBL_OK || (s = M->grads.alloc(pb)) != BBL_OK || (s = M->m.alloc(pb)) != BBL_OK ||
        (s = M->v.alloc(pb)) != BBL_OK || (s = M->tstep.alloc(2 * sizeof(int))) != BBL_OK ||
        (s = M->wbf.alloc(sizeof(__nv_bfloat16) * (hidden + hidden * hidden + out_dim * hidden))) != BBL_OK) {
        delete M;
        return s;
    }
    cudaMemset(M->params.p, 0, pb);
    cudaMemset(M->m.p, 0, pb);
    cudaMemset(M->v.p, 0, pb);
    cudaMemset(M->tstep.p, 0, 2 * sizeof(int));
    cudaMemset(M->wbf.p, 0, M->wbf.bytes);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        delete M;
        return set_error(BBL_ERR_CUDA, "mlp_create: initialisation failed");
    }
    *out = M;
    return BBL_OK;
}

void bbl_mlp_destroy(bbl_mlp* M) {
    if (M) {
        cudaDeviceSynchronize();
        delete M;
    }
}

int bbl_mlp_num_params(const bbl_mlp* M) { return M ? M->nparams : 0; }

bbl_status bbl_mlp_set_params(bbl_mlp* M, const float* packed, void* stream) {
    using namespace bbl;
    if (!M || !packed) return set_error(BBL_ERR_INVALID_ARG, "mlp_set_params: NULL argument");
    cudaStream_t st = as_stream(stream);
    BBL_CUDA(cudaMemcpyAsync(M->params.p, packed, sizeof(float) * M->nparams, cudaMemcpyDefault, st));
    BBL_CUDA(cudaMemsetAsync(M->m.p, 0, M->m.bytes, st));
    BBL_CUDA(cudaMemsetAsync(M->v.p, 0, M->v.bytes, st));
    BBL_CUDA(cudaMemsetAsync(M->tstep.p, 0, 2 * sizeof(int), st));
    to_bf16_kernel<<<64, 256, 0, st>>>(M->hidden, M->out, M->params.as<float>(), M->wbf.as<__nv_bfloat16>());
    BBL_LAUNCH_CHECK();
    BBL_CUDA(cudaStreamSynchronize(st));
    return BBL_OK;
}

bbl_status bbl_mlp_get_params(const bbl_mlp* M, float* packed, float* grads, void* stream) {
    using namespace bbl;
    if (!M) return set_error(BBL_ERR_INVALID_ARG, "mlp_get_params: NULL model");
    cudaStream_t st = as_stream(stream);
    if (packed) BBL_CUDA(cudaMemcpyAsync(packed, M->params.p, sizeof(float) * M->nparams, cudaMemcpyDefault, st));
    if (grads) BBL_CUDA(cudaMemcpyAsync(grads, M->grads.p, sizeof(float) * M->nparams, cudaMemcpyDefault, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    return BBL_OK;
}

bbl_status bbl_mlp_forward(bbl_mlp* M, int batch, const float* g, float* y, void* stream) {
    using namespace bbl;
    if (!M || !g || !y || batch < 1) return set_error(BBL_ERR_INVALID_ARG, "mlp_forward: bad arguments");
    BBL_TRY(ensure_batch(M, batch));
    cudaStream_t st = as_stream(stream);
    BBL_TRY(launch_forward(M, batch, g, y, nullptr, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    return BBL_OK;
}

bbl_status bbl_mlp_loss_grad(bbl_mlp* M, int batch, const float* g, const float* target, float* loss, void* stream) {
    using namespace bbl;
    if (!M || !g || !target || batch < 1) return set_error(BBL_ERR_INVALID_ARG, "mlp_loss_grad: bad arguments");
    BBL_TRY(ensure_batch(M, batch));
    cudaStream_t st = as_stream(stream);
    BBL_TRY(launch_loss_grad(M, batch, g, target, st));
    float h = 0.f;
    BBL_CUDA(cudaMemcpyAsync(&h, M->lossbuf.p, sizeof(float), cudaMemcpyDeviceToHost, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    if (loss) *loss = h;
    return BBL_OK;
}

bbl_status bbl_mlp_adam_step(bbl_mlp* M, float lr, void* stream) {
    using namespace bbl;
    if (!M || !(lr > 0)) return set_error(BBL_ERR_INVALID_ARG, "mlp_adam_step: bad arguments");
    cudaStream_t st = as_stream(stream);
    BBL_TRY(launch_adam(M, lr, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    return BBL_OK;
}

bbl_status bbl_mlp_train(bbl_mlp* M, int batch, const float* g, const float* target, int epochs, float lr,
                         float* loss_hist, void* stream) {
    using namespace bbl;
    if (!M || !g || !target || batch < 1 || epochs < 0 || !(lr > 0))
        return set_error(BBL_ERR_INVALID_ARG, "mlp_train: bad arguments");
    BBL_TRY(ensure_batch(M, batch));
    cudaStream_t st = as_stream(stream);
    cudaStream_t cap = nullptr;
    if (!st) {  // graphs cannot be captured on the legacy stream
        BBL_CUDA(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
        st = cap;
    }
    if (!M->exec || M->graph_batch != batch || M->graph_g != g || M->graph_t != target || M->graph_lr != lr) {
        if (M->exec) {
            cudaGraphExecDestroy(M->exec);
            cudaGraphDestroy(M->graph);
            M->exec = nullptr;
            M->graph = nullptr;
        }
        BBL_CUDA(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
        bbl_status s = launch_loss_grad(M, batch, g, target, st);
        if (s == BBL_OK) s = launch_adam(M, lr, st);
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(st, &graph);
        if (s != BBL_OK) return s;
        if (e != cudaSuccess) return set_error(BBL_ERR_CUDA, "mlp_train: capture failed: %s", cudaGetErrorString(e));
        M->graph = graph;
        BBL_CUDA(cudaGraphInstantiate(&M->exec, graph, 0));
        M->graph_batch = batch;
        M->graph_g = g;
        M->graph_t = target;
        M->graph_lr = lr;
    }
    std::vector<float> hist;
    DevBuf lh;
    if (loss_hist) BBL_TRY(lh.alloc(sizeof(float) * (epochs + 1)));
    for (int e = 0; e < epochs; ++e) {
        BBL_CUDA(cudaGraphLaunch(M->exec, st));
        count_launch();
        if (loss_hist)
            BBL_CUDA(cudaMemcpyAsync(lh.as<float>() + e, M->lossbuf.p, sizeof(float), cudaMemcpyDeviceToDevice, st));
    }
    if (loss_hist && epochs > 0)
        BBL_CUDA(cudaMemcpyAsync(loss_hist, lh.p, sizeof(float) * epochs, cudaMemcpyDeviceToHost, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    if (cap) cudaStreamDestroy(cap);
    return BBL_OK;
}

bbl_status bbl_pivot_learned(bbl_mlp* M, float g, int64_t n, int b_U, int nblocks_U, const float* U, int b, double* P,
                             void* stream) {
    using namespace bbl;
    if (!M || !U || !P || n < 1 || b_U < 1 || b_U > kMaxB || nblocks_U < 1 || b < 1 || b > kMaxB ||
        (int64_t)nblocks_U * b_U * b != M->out)
        return set_error(BBL_ERR_INVALID_ARG, "pivot_learned: shapes do not match the network output");
    cudaStream_t st = as_stream(stream);
    BBL_TRY(ensure_batch(M, 1));
    DevBuf gb(st), y(st), C(st);
    BBL_TRY(gb.alloc(sizeof(float)));
    BBL_TRY(y.alloc(sizeof(float) * M->out));
    BBL_TRY(C.alloc(sizeof(double) * M->out));
    BBL_CUDA(cudaMemcpyAsync(gb.p, &g, sizeof(float), cudaMemcpyHostToDevice, st));
    BBL_TRY(launch_forward(M, 1, gb.as<float>(), y.as<float>(), nullptr, st));
    widen_kernel<<<(unsigned)ceil_div(M->out, 256), 256, 0, st>>>(M->out, y.as<float>(), C.as<double>());
    BBL_LAUNCH_CHECK();
    BBL_TRY(ritz_vectors(n, b_U, nblocks_U, BBL_FP32, U, b, C.as<double>(), P, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    return BBL_OK;
}

}  // extern "C"
