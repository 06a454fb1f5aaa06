// The reaction surrogate's network (8 -> 64 -> 64 -> 8, ReLU hidden layers)
// and its training on the GPU: forward and backward passes over blocks of
// samples, per-block partial gradients reduced in a fixed order (double
// accumulation), Adam, and the loss accumulated in double.  Not part of the
// paper: the learned replacement of the cell-model update.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <vector>

#include "bbx_mlp.cuh"

using namespace bbx;

namespace {

constexpr int kSB = 32;        // samples per training block
constexpr int kThreads = 256;  // threads per training block

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Row of sample i of a minibatch: the identity (seed 0) or a counter-based
// hash draw with replacement.
__device__ __forceinline__ long long sample_row(long long i, long long n, unsigned long long seed,
                                                unsigned long long step) {
    if (seed == 0) return i;
    return (long long)(splitmix64(seed ^ (step * 0x100000001B3ull + (unsigned long long)i)) % (unsigned long long)n);
}

// Forward and backward for kSB samples of the minibatch: per-block partial
// gradients (float, [gridDim.x][kMlpParams]) and partial loss (double).
//
// Every product is a tile of outputs per thread with its operands read from
// shared memory as float4: 32 multiply-adds for six 16-byte loads, where one
// output at a time took two 4-byte loads a multiply-add, the weights' at a
// stride of 64 floats (32 lanes on one bank).  Weight rows are padded to 68
// (12) floats, so that eight lanes' float4 of eight rows touch every bank once.  Each
// sum keeps its order (over inputs, outputs or samples ascending, from the
// bias or 0), so results are bitwise those of one output at a time.
// A step of 4096 samples: 84 us before, 21 by tiles, 13 with the weights' loads
// all in flight at once.
constexpr int kW1P = 12, kW2P = 68;  // padded row lengths
constexpr int kSmW1 = 0, kSmW2 = kSmW1 + 64 * kW1P, kSmW3 = kSmW2 + 64 * kW2P, kSmB1 = kSmW3 + 8 * kW2P,
              kSmB2 = kSmB1 + 64, kSmB3 = kSmB2 + 64, kSmX = kSmB3 + 8, kSmDy = kSmX + kSB * 8,
              kSmH1 = kSmDy + kSB * 8, kSmH2 = kSmH1 + kSB * 64, kSmD2 = kSmH2 + kSB * 64,
              kSmFloats = kSmD2 + kSB * 64;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float dot4(float4 a, float4 b, float z) {  // in order x, y, z, w
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, z))));
}

// Outputs of a layer with K inputs for rows j = jt + 16 i of the weights and
// samples s = st + 16 e (i < 4, e < 2): relu(b + W in).
template <int K, int WP>
__device__ __forceinline__ void layer_tile(const float* W, const float* bias, const float* in, float* out, int jt, int st) {
    float z[2][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) z[0][i] = z[1][i] = bias[jt + 16 * i];
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float4 a0 = ld4(in + st * K + k), a1 = ld4(in + (st + 16) * K + k);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 w = ld4(W + (jt + 16 * i) * WP + k);
            z[0][i] = dot4(w, a0, z[0][i]);
            z[1][i] = dot4(w, a1, z[1][i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        out[st * 64 + jt + 16 * i] = fmaxf(z[0][i], 0.0f);
        out[(st + 16) * 64 + jt + 16 * i] = fmaxf(z[1][i], 0.0f);
    }
}

__global__ void __launch_bounds__(kThreads) k_mlp_fwd_bwd(const float* __restrict__ P, const float* __restrict__ X,
                                                           const float* __restrict__ T, long long n, int batch,
                                                           unsigned long long seed, unsigned long long step,
                                                           const float* __restrict__ norm, float* __restrict__ gpart,
                                                           double* __restrict__ lpart) {
    extern __shared__ float4 sm4[];
    float* sm = reinterpret_cast<float*>(sm4);
    float *W1 = sm + kSmW1, *W2 = sm + kSmW2, *W3 = sm + kSmW3, *b1 = sm + kSmB1, *b2 = sm + kSmB2, *b3 = sm + kSmB3;
    float *xs = sm + kSmX, *dy = sm + kSmDy, *h1 = sm + kSmH1, *h2 = sm + kSmH2, *d2 = sm + kSmD2;
    __shared__ double lsum[kThreads / 32];
    static_assert(kSB == 32 && kThreads == 256, "thread tiles");
    const int tid = threadIdx.x;
    const int jt = tid & 15, st = tid >> 4;
    const int s0 = blockIdx.x * kSB;
    const int ns = min(kSB, batch - s0);
    // the weights, every load of a thread in flight at once (in a loop of loads
    // and stores each pass waited for its own round trip to L2)
    float4 w2[4], w13;
#pragma unroll
    for (int i = 0; i < 4; ++i) w2[i] = ld4(P + kOffW2 + 4 * (tid + kThreads * i));
    w13 = ld4(P + (tid < 128 ? kOffW1 + 4 * tid : kOffW3 + 4 * (tid - 128)));
    const float bv = P[tid < 64 ? kOffB1 + tid : (tid < 128 ? kOffB2 + tid - 64 : kOffB3 + (tid & 7))];
    // normalised inputs and targets: one value of each per thread (sample tid / 8, variable tid % 8)
    const int ts = tid >> 3, tv = tid & 7;
    float xv = 0.0f, tgt = 0.0f;
    if (ts < ns) {
        const long long r = sample_row(s0 + ts, n, seed, step);
        const float x = X[r * 8 + tv], t = T[r * 8 + tv];
        xv = (x - norm[kNormMuIn + tv]) / norm[kNormSdIn + tv];
        tgt = (t - norm[kNormMuOut + tv]) / norm[kNormSdOut + tv];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int e = 4 * (tid + kThreads * i);
        *reinterpret_cast<float4*>(W2 + (e >> 6) * kW2P + (e & 63)) = w2[i];
    }
    if (tid < 128) {
        *reinterpret_cast<float4*>(W1 + (tid >> 1) * kW1P + 4 * (tid & 1)) = w13;
        (tid < 64 ? b1 : b2)[tid & 63] = bv;
    } else {
        *reinterpret_cast<float4*>(W3 + ((tid - 128) >> 4) * kW2P + 4 * (tid & 15)) = w13;
        if (tid < 136) b3[tid - 128] = bv;
    }
    xs[tid] = xv;
    __syncthreads();
    layer_tile<8, kW1P>(W1, b1, xs, h1, jt, st);
    __syncthreads();
    layer_tile<64, kW2P>(W2, b2, h1, h2, jt, st);
    __syncthreads();
    // output, loss and dL/dy = 2 (y - t) / (batch * 8)
    double lacc = 0.0;
    {
        float g = 0.0f;
        if (ts < ns) {
            float y = b3[tv];
#pragma unroll 4
            for (int k = 0; k < 64; k += 4) y = dot4(ld4(W3 + tv * kW2P + k), ld4(h2 + ts * 64 + k), y);
            const float d = y - tgt;
            lacc = (double)d * (double)d;
            g = 2.0f / (float)(batch * 8) * d;
        }
        dy[tid] = g;
    }
    for (int off = 16; off > 0; off >>= 1) lacc += __shfl_xor_sync(0xffffffffu, lacc, off);
    if ((tid & 31) == 0) lsum[tid >> 5] = lacc;
    __syncthreads();
    // dL/dz2 = (dy W3) * relu'(z2): column k of samples s = tid / 64 + 4 i
    const int kc = tid & 63, sq = tid >> 6;
    {
        float w[8];
#pragma unroll
        for (int o = 0; o < 8; ++o) w[o] = W3[o * kW2P + kc];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int s = sq + 4 * i;
            const float4 a = ld4(dy + s * 8), b = ld4(dy + s * 8 + 4);
            float g = fmaf(a.x, w[0], 0.0f);
            g = fmaf(a.y, w[1], g);
            g = fmaf(a.z, w[2], g);
            g = fmaf(a.w, w[3], g);
            g = fmaf(b.x, w[4], g);
            g = fmaf(b.y, w[5], g);
            g = fmaf(b.z, w[6], g);
            g = fmaf(b.w, w[7], g);
            d2[s * 64 + kc] = h2[s * 64 + kc] > 0.0f ? g : 0.0f;
        }
    }
    __syncthreads();
    float* gp = gpart + (size_t)blockIdx.x * kMlpParams;
    // gradients of layer 3 (rows o = sq, sq + 4) and of the biases
    {
        float g0 = 0.0f, g1 = 0.0f;
#pragma unroll 8
        for (int s = 0; s < kSB; ++s) {
            const float h = h2[s * 64 + kc];
            g0 = fmaf(dy[s * 8 + sq], h, g0);
            g1 = fmaf(dy[s * 8 + sq + 4], h, g1);
        }
        gp[kOffW3 + sq * 64 + kc] = g0;
        gp[kOffW3 + (sq + 4) * 64 + kc] = g1;
    }
    if (tid < 64) {
        float g = 0.0f;
#pragma unroll 8
        for (int s = 0; s < kSB; ++s) g += d2[s * 64 + tid];
        gp[kOffB2 + tid] = g;
    } else if (tid < 72) {
        float g = 0.0f;
        for (int s = 0; s < kSB; ++s) g += dy[s * 8 + tid - 64];
        gp[kOffB3 + tid - 64] = g;
    }
    // gradients of layer 2: a 4 x 4 tile of (j, k) per thread
    {
        float g[4][4] = {};
#pragma unroll 4
        for (int s = 0; s < kSB; ++s) {
            const float4 a = ld4(d2 + s * 64 + 4 * st), h = ld4(h1 + s * 64 + 4 * jt);
            const float av[4] = {a.x, a.y, a.z, a.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int q = 0; q < 4; ++q) g[i][q] = fmaf(av[i], hv[q], g[i][q]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) gp[kOffW2 + (4 * st + i) * 64 + 4 * jt + q] = g[i][q];
    }
    __syncthreads();
    // dL/dz1 = (d2 W2) * relu'(z1), written over h2: columns 4 jt .. 4 jt + 3 of samples st, st + 16
    {
        float g[2][4] = {};
#pragma unroll 4
        for (int j = 0; j < 64; j += 4) {
            const float4 a0 = ld4(d2 + st * 64 + j), a1 = ld4(d2 + (st + 16) * 64 + j);
            const float av[2][4] = {{a0.x, a0.y, a0.z, a0.w}, {a1.x, a1.y, a1.z, a1.w}};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 w = ld4(W2 + (j + i) * kW2P + 4 * jt);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    g[e][0] = fmaf(av[e][i], w.x, g[e][0]);
                    g[e][1] = fmaf(av[e][i], w.y, g[e][1]);
                    g[e][2] = fmaf(av[e][i], w.z, g[e][2]);
                    g[e][3] = fmaf(av[e][i], w.w, g[e][3]);
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int i = (st + 16 * e) * 64 + 4 * jt + q;
                h2[i] = h1[i] > 0.0f ? g[e][q] : 0.0f;
            }
    }
    __syncthreads();
    for (int e = tid; e < 64 * 8; e += kThreads) {
        const int j = e / 8, k = e % 8;
        float g = 0.0f;
#pragma unroll 8
        for (int s = 0; s < kSB; ++s) g = fmaf(h2[s * 64 + j], xs[s * 8 + k], g);
        gp[kOffW1 + e] = g;
    }
    if (tid < 64) {
        float g = 0.0f;
#pragma unroll 8
        for (int s = 0; s < kSB; ++s) g += h2[s * 64 + tid];
        gp[kOffB1 + tid] = g;
    }
    if (tid == 0) {
        double l = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) l += lsum[w];
        lpart[blockIdx.x] = l;
    }
}

// Sum the per-block gradients in a fixed order (double accumulation: eight
// segments of the blocks, each in block order, then the segments in order),
// write the gradient, and (if lr > 0) apply one Adam step.  A block takes 32
// parameters; one more block sums the loss partials: loss = sum / (batch * 8).
// (One thread a parameter over all blocks' partials took 30 us for 128 of
// them: a chain of loads on 21 SMs.)
constexpr int kRedSeg = 8;
__global__ void __launch_bounds__(32 * kRedSeg) k_mlp_reduce_adam(
    const float* __restrict__ gpart, int nblk, const double* __restrict__ lpart, int batch, float* __restrict__ P,
    float* __restrict__ M, float* __restrict__ V, float* __restrict__ G, double* __restrict__ loss, int step, float lr,
    float beta1, float beta2, float eps) {
    __shared__ double part[kRedSeg][32];
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
    if (blockIdx.x == gridDim.x - 1) {  // the loss
        double l = 0.0;
        for (int b = threadIdx.x; b < nblk; b += 32 * kRedSeg) l += lpart[b];
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) part[seg][0] = l;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < kRedSeg; ++w) s += part[w][0];
            *loss = s / ((double)batch * 8.0);
        }
        return;
    }
    const int i = blockIdx.x * 32 + lane;
    const int per = (nblk + kRedSeg - 1) / kRedSeg, b0 = seg * per, b1 = min(nblk, b0 + per);
    double g = 0.0;
    if (i < kMlpParams) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) g += gpart[(size_t)b * kMlpParams + i];
    }
    part[seg][lane] = g;
    __syncthreads();
    if (seg != 0 || i >= kMlpParams) return;
    g = 0.0;
#pragma unroll
    for (int w = 0; w < kRedSeg; ++w) g += part[w][lane];
    G[i] = (float)g;
    if (lr > 0.0f) {
        const float gf = (float)g;
        const float m = beta1 * M[i] + (1.0f - beta1) * gf;
        const float v = beta2 * V[i] + (1.0f - beta2) * gf * gf;
        M[i] = m;
        V[i] = v;
        const float mh = m / (1.0f - powf(beta1, (float)step));
        const float vh = v / (1.0f - powf(beta2, (float)step));
        P[i] = P[i] - lr * mh / (sqrtf(vh) + eps);
    }
}

// Per-feature mean, standard deviation (of inputs and targets) and input
// min/max, accumulated in double by one block.
__global__ void k_mlp_stats(const float* __restrict__ X, const float* __restrict__ T, long long n,
                            double* __restrict__ out /* 8 x {sum_x, sumsq_x, min_x, max_x, sum_t, sumsq_t} */) {
    __shared__ double red[6][8][32];
    const int f = threadIdx.x % 8, lane = threadIdx.x / 8;  // 256 threads: 8 features x 32 lanes
    double sx = 0, sxx = 0, st = 0, stt = 0, mn = 1e300, mx = -1e300;
    for (long long r = lane; r < n; r += 32) {
        const double x = X[r * 8 + f], t = T[r * 8 + f];
        sx += x;
        sxx += x * x;
        st += t;
        stt += t * t;
        mn = fmin(mn, x);
        mx = fmax(mx, x);
    }
    red[0][f][lane] = sx;
    red[1][f][lane] = sxx;
    red[2][f][lane] = mn;
    red[3][f][lane] = mx;
    red[4][f][lane] = st;
    red[5][f][lane] = stt;
    __syncthreads();
    if (threadIdx.x < 8) {
        const int ff = threadIdx.x;
        double a[6] = {0, 0, 1e300, -1e300, 0, 0};
        for (int l = 0; l < 32; ++l) {
            a[0] += red[0][ff][l];
            a[1] += red[1][ff][l];
            a[2] = fmin(a[2], red[2][ff][l]);
            a[3] = fmax(a[3], red[3][ff][l]);
            a[4] += red[4][ff][l];
            a[5] += red[5][ff][l];
        }
        for (int q = 0; q < 6; ++q) out[ff * 6 + q] = a[q];
    }
}

__global__ void k_mlp_init(float* P, unsigned long long seed) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= kMlpParams) return;
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases
    float r = 0.0f;
    if (i < kOffB1) r = rsqrtf(8.0f);
    else if (i >= kOffW2 && i < kOffB2) r = 0.125f;
    else if (i >= kOffW3 && i < kOffB3) r = 0.125f;
    const unsigned long long h = splitmix64(seed ^ (unsigned long long)(i + 1) * 0xD1B54A32D192ED03ull);
    const float u = (float)((h >> 40) * (1.0 / 16777216.0));  // [0, 1)
    P[i] = r * (2.0f * u - 1.0f);
}

}  // namespace

struct bbx_mlp {
    cudaStream_t stream = nullptr;
    float* d_P = nullptr;     // parameters, packed W1 b1 W2 b2 W3 b3
    float* d_M = nullptr;     // Adam first moment
    float* d_V = nullptr;     // Adam second moment
    float* d_G = nullptr;     // last gradient
    float* d_gpart = nullptr;
    double* d_lpart = nullptr;
    double* d_loss = nullptr;
    float* d_norm = nullptr;  // kNormSize floats
    float h_norm[kNormSize];
    int cap_blocks = 0;
    int step = 0;
};

namespace {

int ensure_blocks(bbx_mlp* m, int nblk) {
    if (nblk <= m->cap_blocks) return BBX_OK;
    cudaFree(m->d_gpart);
    cudaFree(m->d_lpart);
    m->d_gpart = nullptr;
    m->d_lpart = nullptr;
    if (cudaMalloc(&m->d_gpart, sizeof(float) * kMlpParams * (size_t)nblk) != cudaSuccess ||
        cudaMalloc(&m->d_lpart, sizeof(double) * (size_t)nblk) != cudaSuccess) {
        cudaGetLastError();
        m->cap_blocks = 0;
        return BBX_ERR_NOMEM;
    }
    m->cap_blocks = nblk;
    return BBX_OK;
}

int run_batch(bbx_mlp* m, const float* X, const float* T, long long n, int batch, unsigned long long seed, float lr) {
    const int nblk = (batch + kSB - 1) / kSB;
    int rc = ensure_blocks(m, nblk);
    if (rc) return rc;
    if (lr > 0.0f) ++m->step;
    k_mlp_fwd_bwd<<<nblk, kThreads, sizeof(float) * kSmFloats, m->stream>>>(m->d_P, X, T, n, batch, seed, (unsigned long long)m->step,
                                                    m->d_norm, m->d_gpart, m->d_lpart);
    k_mlp_reduce_adam<<<(kMlpParams + 31) / 32 + 1, 32 * kRedSeg, 0, m->stream>>>(m->d_gpart, nblk, m->d_lpart, batch, m->d_P,
                                                                       m->d_M, m->d_V, m->d_G, m->d_loss, m->step,
                                                                       lr, 0.9f, 0.999f, 1e-8f);
    if (cudaGetLastError() != cudaSuccess) return BBX_ERR_CUDA;
    return BBX_OK;
}

}  // namespace

const float* bbx_mlp_device_params(const bbx_mlp* m) { return m->d_P; }
const float* bbx_mlp_device_norm(const bbx_mlp* m) { return m->d_norm; }

extern "C" {

int bbx_mlp_create(bbx_mlp** out, unsigned long long seed, void* cuda_stream) {
    if (!out) return BBX_ERR_ARG;
    *out = nullptr;
    bbx_mlp* m = new (std::nothrow) bbx_mlp();
    if (!m) return BBX_ERR_NOMEM;
    m->stream = static_cast<cudaStream_t>(cuda_stream);
    if (cudaMalloc(&m->d_P, sizeof(float) * kMlpParams) != cudaSuccess ||
        cudaMalloc(&m->d_M, sizeof(float) * kMlpParams) != cudaSuccess ||
        cudaMalloc(&m->d_V, sizeof(float) * kMlpParams) != cudaSuccess ||
        cudaMalloc(&m->d_G, sizeof(float) * kMlpParams) != cudaSuccess ||
        cudaMalloc(&m->d_loss, sizeof(double)) != cudaSuccess ||
        cudaMalloc(&m->d_norm, sizeof(float) * kNormSize) != cudaSuccess ||
        cudaFuncSetAttribute(k_mlp_fwd_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(float) * kSmFloats) !=
            cudaSuccess) {
        cudaGetLastError();
        bbx_mlp_destroy(m);
        return BBX_ERR_NOMEM;
    }
    for (int k = 0; k < 8; ++k) {
        m->h_norm[kNormMuIn + k] = 0.0f;
        m->h_norm[kNormSdIn + k] = 1.0f;
        m->h_norm[kNormMuOut + k] = 0.0f;
        m->h_norm[kNormSdOut + k] = 1.0f;
        m->h_norm[kNormLo + k] = -INFINITY;
        m->h_norm[kNormHi + k] = INFINITY;
    }
    k_mlp_init<<<(kMlpParams + 255) / 256, 256, 0, m->stream>>>(m->d_P, seed);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemsetAsync(m->d_M, 0, sizeof(float) * kMlpParams, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->d_V, 0, sizeof(float) * kMlpParams, m->stream) != cudaSuccess ||
        cudaMemcpyAsync(m->d_norm, m->h_norm, sizeof(m->h_norm), cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess) {
        cudaGetLastError();
        bbx_mlp_destroy(m);
        return BBX_ERR_CUDA;
    }
    *out = m;
    return BBX_OK;
}

void bbx_mlp_destroy(bbx_mlp* m) {
    if (!m) return;
    cudaStreamSynchronize(m->stream);
    cudaFree(m->d_P);
    cudaFree(m->d_M);
    cudaFree(m->d_V);
    cudaFree(m->d_G);
    cudaFree(m->d_gpart);
    cudaFree(m->d_lpart);
    cudaFree(m->d_loss);
    cudaFree(m->d_norm);
    cudaGetLastError();
    delete m;
}

int bbx_mlp_set_params(bbx_mlp* m, const float* params, size_t n) {
    if (!m || !params || n != (size_t)kMlpParams) return BBX_ERR_ARG;
    if (cudaMemcpyAsync(m->d_P, params, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->d_M, 0, sizeof(float) * kMlpParams, m->stream) != cudaSuccess ||
        cudaMemsetAsync(m->d_V, 0, sizeof(float) * kMlpParams, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess) {
        cudaGetLastError();
        return BBX_ERR_CUDA;
    }
    m->step = 0;
    return BBX_OK;
}

int bbx_mlp_get_params(bbx_mlp* m, float* params, size_t n) {
    if (!m || !params || n != (size_t)kMlpParams) return BBX_ERR_ARG;
    if (cudaMemcpyAsync(params, m->d_P, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess) {
        cudaGetLastError();
        return BBX_ERR_CUDA;
    }
    return BBX_OK;
}

int bbx_mlp_set_normalization(bbx_mlp* m, const float* norm, size_t n) {
    if (!m || !norm || n != (size_t)kNormSize) return BBX_ERR_ARG;
    for (int k = 0; k < 8; ++k)
        if (!(norm[kNormSdIn + k] > 0.0f) || !(norm[kNormSdOut + k] > 0.0f)) return BBX_ERR_ARG;
    memcpy(m->h_norm, norm, sizeof(m->h_norm));
    if (cudaMemcpyAsync(m->d_norm, m->h_norm, sizeof(m->h_norm), cudaMemcpyHostToDevice, m->stream) != cudaSuccess ||
        cudaStreamSynchronize(m->stream) != cudaSuccess) {
        cudaGetLastError();
        return BBX_ERR_CUDA;
    }
    return BBX_OK;
}

int bbx_mlp_get_normalization(bbx_mlp* m, float* norm, size_t n) {
    if (!m || !norm || n != (size_t)kNormSize) return BBX_ERR_ARG;
    memcpy(norm, m->h_norm, sizeof(m->h_norm));
    return BBX_OK;
}

int bbx_mlp_fit_normalization(bbx_mlp* m, const float* x_dev, const float* t_dev, long long n) {
    if (!m || !x_dev || !t_dev || n < 2) return BBX_ERR_ARG;
    double* d_out = nullptr;
    if (cudaMalloc(&d_out, sizeof(double) * 48) != cudaSuccess) {
        cudaGetLastError();
        return BBX_ERR_NOMEM;
    }
    double h[48];
    k_mlp_stats<<<1, 256, 0, m->stream>>>(x_dev, t_dev, n, d_out);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d_out, sizeof(h), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    cudaFree(d_out);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return BBX_ERR_CUDA;
    }
    float norm[kNormSize];
    for (int k = 0; k < 8; ++k) {
        const double* a = h + 6 * k;
        const double mx = a[0] / n, vx = a[1] / n - mx * mx;
        const double mt = a[4] / n, vt = a[5] / n - mt * mt;
        norm[kNormMuIn + k] = (float)mx;
        norm[kNormSdIn + k] = (float)std::sqrt(vx > 1e-30 ? vx : 1e-30);
        norm[kNormMuOut + k] = (float)mt;
        norm[kNormSdOut + k] = (float)std::sqrt(vt > 1e-30 ? vt : 1e-30);
        norm[kNormLo + k] = (float)a[2];
        norm[kNormHi + k] = (float)a[3];
    }
    return bbx_mlp_set_normalization(m, norm, kNormSize);
}

int bbx_mlp_gradients(bbx_mlp* m, const float* x_dev, const float* t_dev, int batch, float* grad, size_t n,
                      double* loss) {
    if (!m || !x_dev || !t_dev || batch <= 0 || !grad || n != (size_t)kMlpParams) return BBX_ERR_ARG;
    int rc = run_batch(m, x_dev, t_dev, batch, batch, 0ull, 0.0f);
    if (rc) return rc;
    if (cudaMemcpyAsync(grad, m->d_G, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
        (loss && cudaMemcpyAsync(loss, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess) ||
        cudaStreamSynchronize(m->stream) != cudaSuccess) {
        cudaGetLastError();
        return BBX_ERR_CUDA;
    }
    return BBX_OK;
}

int bbx_mlp_train(bbx_mlp* m, const float* x_dev, const float* t_dev, long long n, int batch, int steps, double lr,
                  unsigned long long seed, double* final_loss) {
    if (!m || !x_dev || !t_dev || n <= 0 || batch <= 0 || steps < 0 || !(lr > 0.0) || seed == 0) return BBX_ERR_ARG;
    for (int s = 0; s < steps; ++s) {
        int rc = run_batch(m, x_dev, t_dev, n, batch, seed, (float)lr);
        if (rc) return rc;
    }
    if (final_loss) {
        if (cudaMemcpyAsync(final_loss, m->d_loss, sizeof(double), cudaMemcpyDeviceToHost, m->stream) != cudaSuccess ||
            cudaStreamSynchronize(m->stream) != cudaSuccess) {
            cudaGetLastError();
            return BBX_ERR_CUDA;
        }
    }
    return BBX_OK;
}

}  // extern "C"
