// Cost model: a 37 -> 64 -> 64 -> 1 ReLU network that predicts log(seconds)
// of one fused-operator pass from (k, physical target mask, N, batch), trained
// on timings the library collects from its own kernels.  Forward, backward
// and Adam (Kingma & Ba 2015, Algorithm 1) run as CUDA kernels in FP32;
// batch reductions use a fixed order, so results are deterministic.
//
// Parameter layout (6657 floats): W1[64][37], b1[64], W2[64][64], b2[64],
// W3[1][64], b3[1].
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <string>
#include <vector>

#include "qsa.h"
#include "qsa_costmodel.h"
#include "qsa_internal.h"
#include "qsa_runtime.h"

namespace qsa {

namespace {

namespace cg = cooperative_groups;

constexpr int IN = kMlpIn, H = kMlpH;
constexpr int OFF_W1 = 0, OFF_B1 = H * IN, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H, OFF_W3 = OFF_B2 + H,
              OFF_B3 = OFF_W3 + H;

// The network on tiles of `S` samples per CTA, all of it in shared memory: the
// parameters once per CTA, the tile's activations, and with GRAD its gradients.
// The work is small (a minibatch of 64 is 0.4 MFLOP forward), so what it costs
// is launches and the memory between them; one launch does a whole minibatch:
// the CTAs of a cluster sum their gradients through distributed shared memory
// in rank order (each takes a share of the parameters), and only batches of
// more than one cluster write partial sums for a second launch.
// Loss, gradients and the Adam step of 64 samples, by the caller's clock: 73.7
// us in eleven launches (a thread per output looping over the batch), 21.1 us in
// two.
constexpr int kMlpThreads = 256, kMlpMaxS = 32, kMlpCluster = 8;
constexpr int kW2 = H + 1;   // padded row of W2 in shared memory (a warp reads 32 rows at a time)

struct MlpShared {
    float w1[H * IN], b1[H], w2[H * kW2], b2[H], w3[H], b3;
    float x[kMlpMaxS * IN], t[kMlpMaxS];
    alignas(16) float a1[kMlpMaxS * H];
    alignas(16) float a2[kMlpMaxS * H];
    alignas(16) float d2[kMlpMaxS * H];
    alignas(16) float d1[kMlpMaxS * H];
    float dy[kMlpMaxS];
    float g[kMlpParams];   // the tile's gradients, in the parameters' layout
    double sq;             // and its sum of squared errors
};

// Partial gradients of a cluster and its sum of squared errors (a double in two words).
constexpr size_t kMlpPartial = kMlpParams + 2;

template <bool GRAD>
__global__ void __launch_bounds__(kMlpThreads) k_mlp(const float* __restrict__ P, const float* __restrict__ X,
                                                     const float* __restrict__ t, size_t n, int S,
                                                     float* __restrict__ y, float* __restrict__ G,
                                                     float* __restrict__ loss, float* __restrict__ partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    MlpShared& sh = *reinterpret_cast<MlpShared*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < H * IN; i += kMlpThreads) sh.w1[i] = P[OFF_W1 + i];
    for (int i = tid; i < H * H; i += kMlpThreads) sh.w2[(i / H) * kW2 + i % H] = P[OFF_W2 + i];
    if (tid < H) {
        sh.b1[tid] = P[OFF_B1 + tid];
        sh.b2[tid] = P[OFF_B2 + tid];
        sh.w3[tid] = P[OFF_W3 + tid];
    }
    if (tid == 0) sh.b3 = P[OFF_B3];
    const size_t s0 = static_cast<size_t>(blockIdx.x) * S;
    const int ns = s0 >= n ? 0 : static_cast<int>(n - s0 < static_cast<size_t>(S) ? n - s0 : static_cast<size_t>(S));
    for (int i = tid; i < S * IN; i += kMlpThreads) sh.x[i] = i < ns * IN ? X[s0 * IN + i] : 0.f;
    if (GRAD && tid < S) sh.t[tid] = tid < ns ? t[s0 + tid] : 0.f;
    __syncthreads();
    // layers 1 and 2: thread -> unit tid % 64, samples tid / 64 + 4 j
    const int o = tid & (H - 1), q = tid >> 6;
    for (int s = q; s < ns; s += 4) {
        float z = sh.b1[o];
#pragma unroll
        for (int i = 0; i < IN; ++i) z = fmaf(sh.w1[o * IN + i], sh.x[s * IN + i], z);
        sh.a1[s * H + o] = z > 0.f ? z : 0.f;
    }
    __syncthreads();
    for (int s = q; s < ns; s += 4) {
        float z = sh.b2[o];
#pragma unroll 16
        for (int i = 0; i < H; ++i) z = fmaf(sh.w2[o * kW2 + i], sh.a1[s * H + i], z);
        sh.a2[s * H + o] = z > 0.f ? z : 0.f;
    }
    __syncthreads();
    // layer 3: a warp per sample
    double sq = 0.0;
    for (int s = warp; s < ns; s += kMlpThreads / 32) {
        float v = fmaf(sh.w3[lane], sh.a2[s * H + lane], sh.w3[lane + 32] * sh.a2[s * H + lane + 32]);
#pragma unroll
        for (int k = 16; k > 0; k >>= 1) v += __shfl_xor_sync(0xffffffffu, v, k);
        v += sh.b3;
        if (GRAD) {
            const float e = v - sh.t[s];
            if (lane == 0) sh.dy[s] = 2.f * e / static_cast<float>(n);
            sq += static_cast<double>(e * e);
        } else if (lane == 0) {
            y[s0 + s] = v;
        }
    }
    if constexpr (GRAD) {
        __shared__ double wsq[kMlpThreads / 32];
        if (lane == 0) wsq[warp] = sq;
        __syncthreads();
        if (tid == 0) {
            double a = 0.0;
            for (int k = 0; k < kMlpThreads / 32; ++k) a += wsq[k];
            sh.sq = a;
        }
        for (int s = q; s < ns; s += 4) sh.d2[s * H + o] = sh.a2[s * H + o] > 0.f ? sh.dy[s] * sh.w3[o] : 0.f;
        __syncthreads();
        // dW2: 4 x 4 outputs per thread; d1 = (d2 W2) masked
        {
            const int o0 = (tid >> 4) * 4, i0 = (tid & 15) * 4;
            float acc[4][4] = {};
            for (int s = 0; s < ns; ++s) {
                const float4 d = *reinterpret_cast<const float4*>(sh.d2 + s * H + o0);
                const float4 a = *reinterpret_cast<const float4*>(sh.a1 + s * H + i0);
                const float dd[4] = {d.x, d.y, d.z, d.w}, aa[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(dd[u], aa[v], acc[u][v]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) sh.g[OFF_W2 + (o0 + u) * H + i0 + v] = acc[u][v];
        }
        for (int s = q; s < ns; s += 4) {
            float a = 0.f;
#pragma unroll 16
            for (int u = 0; u < H; ++u) a = fmaf(sh.d2[s * H + u], sh.w2[u * kW2 + o], a);
            sh.d1[s * H + o] = sh.a1[s * H + o] > 0.f ? a : 0.f;
        }
        __syncthreads();
        for (int k = tid; k < H * IN; k += kMlpThreads) {
            const int u = k / IN, i = k % IN;
            float a = 0.f;
            for (int s = 0; s < ns; ++s) a = fmaf(sh.d1[s * H + u], sh.x[s * IN + i], a);
            sh.g[OFF_W1 + k] = a;
        }
        if (tid < H) {
            float b1 = 0.f, b2 = 0.f;
            for (int s = 0; s < ns; ++s) {
                b1 += sh.d1[s * H + tid];
                b2 += sh.d2[s * H + tid];
            }
            sh.g[OFF_B1 + tid] = b1;
            sh.g[OFF_B2 + tid] = b2;
        } else if (tid < 2 * H) {
            const int u = tid - H;
            float w = 0.f;
            for (int s = 0; s < ns; ++s) w = fmaf(sh.dy[s], sh.a2[s * H + u], w);
            sh.g[OFF_W3 + u] = w;
        } else if (tid == 2 * H) {
            float b = 0.f;
            for (int s = 0; s < ns; ++s) b += sh.dy[s];
            sh.g[OFF_B3] = b;
        }
        // the cluster's sum, in rank order
        cg::cluster_group cluster = cg::this_cluster();
        cluster.sync();
        const unsigned C = cluster.num_blocks(), r = cluster.block_rank();
        const unsigned nclusters = gridDim.x / C, c = blockIdx.x / C;
        float* out = nclusters == 1 ? G : partial + c * kMlpPartial;
        for (unsigned i = r * kMlpThreads + tid; i < static_cast<unsigned>(kMlpParams); i += C * kMlpThreads) {
            float a = 0.f;
            for (unsigned k = 0; k < C; ++k) a += cluster.map_shared_rank(sh.g, k)[i];
            out[i] = a;
        }
        if (r == 0 && tid == 0) {
            double a = 0.0;
            for (unsigned k = 0; k < C; ++k) a += *cluster.map_shared_rank(&sh.sq, k);
            if (nclusters > 1) {
                out[kMlpParams] = __int_as_float(__double2loint(a));
                out[kMlpParams + 1] = __int_as_float(__double2hiint(a));
            } else if (loss) {
                *loss = static_cast<float>(a / static_cast<double>(n));
            }
        }
        cluster.sync();   // no CTA leaves while another reads its gradients
    }
}

// Gradients (and the loss) from the clusters' partial sums, in order.
__global__ void k_mlp_reduce(const float* __restrict__ partial, int nclusters, size_t n, float* __restrict__ G,
                             float* __restrict__ loss) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < kMlpParams) {
        float a = 0.f;
        for (int c = 0; c < nclusters; ++c) a += partial[c * kMlpPartial + i];
        G[i] = a;
    } else if (i == kMlpParams && loss) {
        double a = 0.0;
        for (int c = 0; c < nclusters; ++c) {
            const float* p = partial + c * kMlpPartial + kMlpParams;
            a += __hiloint2double(__float_as_int(p[1]), __float_as_int(p[0]));
        }
        *loss = static_cast<float>(a / static_cast<double>(n));
    }
}

// Squared error of each sample.
__global__ void k_squares(const float* __restrict__ y, const float* __restrict__ t, size_t n, float* __restrict__ sq) {
    const size_t s = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const float e = y[s] - t[s];
    sq[s] = e * e;
}

// out[0] = mean of v[0..n-1] (one CTA, fixed order).
__global__ void k_mean(const float* __restrict__ v, size_t n, float* __restrict__ out) {
    __shared__ double sh[256];
    double a = 0.0;
    for (size_t i = threadIdx.x; i < n; i += blockDim.x) a += v[i];
    sh[threadIdx.x] = a;
    __syncthreads();
    for (int st = blockDim.x >> 1; st > 0; st >>= 1) {
        if (static_cast<int>(threadIdx.x) < st) sh[threadIdx.x] += sh[threadIdx.x + st];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = static_cast<float>(sh[0] / static_cast<double>(n));
}

// Adam: m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// p -= lr * (m / c1) / (sqrt(v / c2) + eps), with c1 = 1 - b1^t, c2 = 1 - b2^t.
// With wd > 0 the gradient of the L2 penalty (wd / 2) |p|^2 is added first.
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, size_t count, float lr, float b1, float b2, float eps, float c1,
                       float c2, float wd) {
    const size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= count) return;
    const float gi = g[i] + wd * p[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

inline unsigned blocks_for(size_t work, int threads) {
    return static_cast<unsigned>((work + threads - 1) / threads);
}

// Workspace per sample: room for a sample's activations and their gradients
// (6 x 64 + 3 floats); the partial sums of a cluster's 256 samples take less.
constexpr size_t kWsPerSample = 6 * H + 3;
static_assert(kMlpPartial * 2 <= kWsPerSample * (kMlpMaxS * kMlpCluster + 1), "partial sums fit the workspace");

cudaError_t forward(const float* P, const float* X, size_t n, float* y, cudaStream_t st) {
    cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(k_mlp<false>), static_cast<int>(sizeof(MlpShared)));
    if (e != cudaSuccess) return e;
    // as many CTAs as samples allow while the chip has room: eight samples each, then up to 32
    const int S = n > 16u * num_sms() ? kMlpMaxS : n > 8u * num_sms() ? 16 : 8;
    k_mlp<false><<<blocks_for(n, S), kMlpThreads, sizeof(MlpShared), st>>>(P, X, nullptr, n, S, y, nullptr, nullptr,
                                                                           nullptr);
    return cudaGetLastError();
}

cudaError_t loss_grad(const float* P, const float* X, const float* t, size_t n, float* ws, float* G, float* loss,
                      cudaStream_t st) {
    cudaError_t e = set_smem_attr(reinterpret_cast<const void*>(k_mlp<true>), static_cast<int>(sizeof(MlpShared)));
    if (e != cudaSuccess) return e;
    // one cluster while its CTAs take at most 32 samples each
    const int S = n <= 8 * kMlpCluster ? 8 : n <= 16 * kMlpCluster ? 16 : kMlpMaxS;
    const unsigned ctas = blocks_for(n, S);
    const unsigned C = std::min<unsigned>(ctas, kMlpCluster), nclusters = (ctas + C - 1) / C;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(nclusters * C);
    cfg.blockDim = dim3(kMlpThreads);
    cfg.dynamicSmemBytes = sizeof(MlpShared);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, k_mlp<true>, P, X, t, n, S, static_cast<float*>(nullptr), G, loss, ws);
    if (e == cudaSuccess && nclusters > 1)
        k_mlp_reduce<<<blocks_for(kMlpParams + 1, 256), 256, 0, st>>>(ws, static_cast<int>(nclusters), n, G, loss);
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// splitmix64 (Steele, Lea & Flood 2014) for initialisation and shuffling.
uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
double uniform01(uint64_t& s) { return static_cast<double>(splitmix(s) >> 11) * (1.0 / 9007199254740992.0); }

}  // namespace

}  // namespace qsa

using namespace qsa;

extern "C" {

size_t qsa_mlp_workspace_bytes(size_t n) { return sizeof(float) * kWsPerSample * n; }

qsa_status qsa_mlp_forward(const float* params_dev, const float* X_dev, size_t n, float* y_dev, float* workspace_dev,
                           void* stream) {
    if (!params_dev || !X_dev || !y_dev || !workspace_dev || n == 0) return fail(QSA_E_ARG, "NULL argument or n = 0");
    cudaError_t e = forward(params_dev, X_dev, n, y_dev, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return fail(QSA_E_CUDA, std::string("mlp forward: ") + cudaGetErrorString(e));
    return QSA_OK;
}

qsa_status qsa_mlp_loss_grad(const float* params_dev, const float* X_dev, const float* t_dev, size_t n,
                             float* grads_dev, float* loss_dev, float* workspace_dev, void* stream) {
    if (!params_dev || !X_dev || !t_dev || !grads_dev || !workspace_dev || n == 0)
        return fail(QSA_E_ARG, "NULL argument or n = 0");
    cudaError_t e = loss_grad(params_dev, X_dev, t_dev, n, workspace_dev, grads_dev, loss_dev,
                              static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return fail(QSA_E_CUDA, std::string("mlp backward: ") + cudaGetErrorString(e));
    return QSA_OK;
}

qsa_status qsa_mlp_adam_step(float* params_dev, const float* grads_dev, float* m_dev, float* v_dev, size_t count,
                             int step, float lr, float beta1, float beta2, float eps, void* stream) {
    if (!params_dev || !grads_dev || !m_dev || !v_dev || step < 1) return fail(QSA_E_ARG, "bad Adam arguments");
    const float c1 = static_cast<float>(1.0 - std::pow(static_cast<double>(beta1), step));
    const float c2 = static_cast<float>(1.0 - std::pow(static_cast<double>(beta2), step));
    k_adam<<<blocks_for(count, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(params_dev, grads_dev, m_dev, v_dev,
                                                                                  count, lr, beta1, beta2, eps, c1, c2,
                                                                                  0.f);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(QSA_E_CUDA, std::string("adam: ") + cudaGetErrorString(e));
    return QSA_OK;
}

qsa_status qsa_costmodel_init(uint64_t seed, float* params_host) {
    if (!params_host) return fail(QSA_E_ARG, "NULL argument");
    // He-uniform weights: U(-sqrt(6/fan_in), +sqrt(6/fan_in)); zero biases.
    uint64_t s = seed ^ 0x5DEECE66Dull;
    std::memset(params_host, 0, sizeof(float) * kMlpParams);
    auto fill = [&](int off, int count, int fan_in) {
        const double a = std::sqrt(6.0 / fan_in);
        for (int i = 0; i < count; ++i) params_host[off + i] = static_cast<float>((2.0 * uniform01(s) - 1.0) * a);
    };
    fill(OFF_W1, H * IN, IN);
    fill(OFF_W2, H * H, H);
    fill(OFF_W3, H, H);
    return QSA_OK;
}

qsa_status qsa_costmodel_train(const float* X_host, const float* y_host, size_t n, int epochs, int batch, float lr,
                               float weight_decay, uint64_t seed, float* params_inout_host, float* epoch_loss_host) {
    if (!X_host || !y_host || !params_inout_host || n == 0 || epochs < 1 || batch < 1 || weight_decay < 0.f)
        return fail(QSA_E_ARG, "bad training arguments");
    // Standardise the targets (log-seconds sit far from the network's initial
    // output): train on (y - mu) / sigma with the output layer rescaled to
    // match, then fold mu and sigma back into W3 and b3.
    double mu = 0.0, var = 0.0;
    for (size_t i = 0; i < n; ++i) mu += y_host[i];
    mu /= static_cast<double>(n);
    for (size_t i = 0; i < n; ++i) var += (y_host[i] - mu) * (y_host[i] - mu);
    const double sigma = std::max(1e-6, std::sqrt(var / static_cast<double>(n)));
    std::vector<float> yn(n);
    for (size_t i = 0; i < n; ++i) yn[i] = static_cast<float>((y_host[i] - mu) / sigma);
    for (int j = 0; j < H; ++j) params_inout_host[OFF_W3 + j] = static_cast<float>(params_inout_host[OFF_W3 + j] / sigma);
    params_inout_host[OFF_B3] = static_cast<float>((params_inout_host[OFF_B3] - mu) / sigma);
    y_host = yn.data();
    const size_t bsz = std::min<size_t>(static_cast<size_t>(batch), n);
    float *dX = nullptr, *dY = nullptr, *dP = nullptr, *dG = nullptr, *dM = nullptr, *dV = nullptr, *dWs = nullptr,
          *dLoss = nullptr, *dXb = nullptr, *dYb = nullptr, *dOut = nullptr;
    const size_t np = kMlpParams;
    cudaStream_t st = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    auto A = [&](float** p, size_t cnt) {
        if (e == cudaSuccess) e = dev_malloc(p, sizeof(float) * cnt);
    };
    A(&dX, n * IN);
    A(&dY, n);
    A(&dP, np);
    A(&dG, np);
    A(&dM, np);
    A(&dV, np);
    A(&dWs, kWsPerSample * n);
    A(&dLoss, 1);
    A(&dXb, bsz * IN);
    A(&dYb, bsz);
    A(&dOut, n);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dX, X_host, sizeof(float) * n * IN, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dY, y_host, sizeof(float) * n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dP, params_inout_host, sizeof(float) * np, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dM, 0, sizeof(float) * np, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dV, 0, sizeof(float) * np, st);
    std::vector<size_t> order(n);
    std::iota(order.begin(), order.end(), size_t(0));
    std::vector<float> xb(bsz * IN), yb(bsz);
    uint64_t rs = seed;
    int step = 0;
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        for (size_t i = n; i > 1; --i) std::swap(order[i - 1], order[splitmix(rs) % i]);  // Fisher-Yates
        for (size_t b0 = 0; b0 + bsz <= n && e == cudaSuccess; b0 += bsz) {
            for (size_t r = 0; r < bsz; ++r) {
                std::memcpy(&xb[r * IN], X_host + order[b0 + r] * IN, sizeof(float) * IN);
                yb[r] = y_host[order[b0 + r]];
            }
            e = cudaMemcpyAsync(dXb, xb.data(), sizeof(float) * bsz * IN, cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess) e = cudaMemcpyAsync(dYb, yb.data(), sizeof(float) * bsz, cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess) e = loss_grad(dP, dXb, dYb, bsz, dWs, dG, nullptr, st);
            ++step;
            if (e == cudaSuccess) {
                const float c1 = static_cast<float>(1.0 - std::pow(0.9, step));
                const float c2 = static_cast<float>(1.0 - std::pow(0.999, step));
                k_adam<<<blocks_for(np, 256), 256, 0, st>>>(dP, dG, dM, dV, np, lr, 0.9f, 0.999f, 1e-8f, c1, c2,
                                                            weight_decay);
                e = cudaGetLastError();
            }
            // the pageable staging vectors are reused: wait for the copies
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        }
        if (epoch_loss_host && e == cudaSuccess) {
            e = forward(dP, dX, n, dOut, st);
            if (e == cudaSuccess) {
                k_squares<<<blocks_for(n, 256), 256, 0, st>>>(dOut, dY, n, dWs);
                k_mean<<<1, 256, 0, st>>>(dWs, n, dLoss);
                e = cudaMemcpyAsync(&epoch_loss_host[ep], dLoss, sizeof(float), cudaMemcpyDeviceToHost, st);
            }
        }
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(params_inout_host, dP, sizeof(float) * np, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    for (float* p : {dX, dY, dP, dG, dM, dV, dWs, dLoss, dXb, dYb, dOut})
        if (p) dev_free(p);
    if (st) cudaStreamDestroy(st);
    // fold the standardisation back into the output layer (also on failure,
    // so the caller's parameters keep their meaning)
    for (int j = 0; j < H; ++j) params_inout_host[OFF_W3 + j] = static_cast<float>(params_inout_host[OFF_W3 + j] * sigma);
    params_inout_host[OFF_B3] = static_cast<float>(params_inout_host[OFF_B3] * sigma + mu);
    if (epoch_loss_host)
        for (int ep = 0; ep < epochs; ++ep) epoch_loss_host[ep] = static_cast<float>(epoch_loss_host[ep] * sigma * sigma);
    if (e != cudaSuccess) return fail(QSA_E_CUDA, std::string("cost-model training: ") + cudaGetErrorString(e));
    return QSA_OK;
}

// Time one fused-operator pass for n_samples random (k, physical targets)
// on the state (identity matrices, so the amplitudes are unchanged) and
// return the features and log(median seconds over reps launches).
qsa_status qsa_costmodel_collect(qsa_state s, size_t n_samples, int reps, int precision, uint64_t seed,
                                 float* X_host, float* y_host) {
    qsa_status stt = check_state(s);
    if (stt != QSA_OK) return stt;
    if (!X_host || !y_host || reps < 1 || precision < 0 || precision > 1) return fail(QSA_E_ARG, "bad arguments");
    const int n = s->n;
    const int kmax = std::min(QSA_MAX_K, n);
    // identity matrices for k = 1..kmax, uploaded once
    std::vector<float> hm;
    std::vector<size_t> off(kmax + 1, 0);
    for (int k = 1; k <= kmax; ++k) {
        off[k] = hm.size();
        const size_t D = size_t(1) << k;
        hm.resize(hm.size() + 2 * D * D, 0.f);
        for (size_t i = 0; i < D; ++i) hm[off[k] + 2 * (i * D + i)] = 1.f;
        while (hm.size() % 4) hm.push_back(0.f);
    }
    stt = ensure_dev(s, reinterpret_cast<void**>(&s->d_mat), &s->mat_cap, hm.size() * sizeof(float));
    if (stt != QSA_OK) return stt;
    cudaError_t e = cudaMemcpyAsync(s->d_mat, hm.data(), hm.size() * sizeof(float), cudaMemcpyHostToDevice, s->stream);
    if (e != cudaSuccess) return cuda_fail(s, e, "collect upload");
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    uint64_t rs = seed;
    std::vector<float> t(reps);
    for (size_t i = 0; i < n_samples; ++i) {
        const int k = 1 + static_cast<int>(splitmix(rs) % static_cast<uint64_t>(kmax));
        int perm[QSA_MAX_QUBITS];
        for (int q = 0; q < n; ++q) perm[q] = q;
        for (int q = n; q > 1; --q) std::swap(perm[q - 1], perm[splitmix(rs) % static_cast<uint64_t>(q)]);
        int phys[QSA_MAX_K];
        uint64_t mask = 0;
        for (int j = 0; j < k; ++j) {
            phys[j] = perm[j];
            mask |= 1ull << perm[j];
        }
        for (int r = 0; r < reps && e == cudaSuccess; ++r) {
            cudaEventRecord(a, s->stream);
            stt = apply_physical(s, phys, k, s->d_mat + off[k], precision, nullptr);
            if (stt != QSA_OK) break;
            cudaEventRecord(b, s->stream);
            e = cudaEventSynchronize(b);
            float ms = 0.f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, a, b);
            t[r] = ms;
        }
        if (stt != QSA_OK || e != cudaSuccess) break;
        std::sort(t.begin(), t.end());
        costmodel_features(k, mask, n, 1, X_host + i * kMlpIn);
        y_host[i] = static_cast<float>(std::log(std::max(1e-9, t[reps / 2] * 1e-3)));
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (stt != QSA_OK) return stt;
    if (e != cudaSuccess) return cuda_fail(s, e, "collect timing");
    return sync_and_check(s, "collect");
}

}  // extern "C"
