// k_mlp.cu -- the learned per-cell cost model: a 3 -> 32 -> 32 -> 1
// multilayer perceptron with ReLU, trained with mean-squared error and Adam
// (Kingma & Ba) on per-cell timings, and the contiguous equal-cost partition
// of cells over persistent CTAs that its predictions feed.  The paper
// balances uneven work with its cell-task schedule (Sec. 2.1) and reports the
// imbalance of inhomogeneous systems (Sec. 1); this model predicts that
// unevenness ahead of the force pass.
//
// Parameter layout (1217 float32): W1[32][3], b1[32], W2[32][32], b2[32],
// W3[32], b3[1].
#include <cmath>
#include <mutex>
#include <string>

#include "k_scan.cuh"

namespace mdg {

constexpr int kH = 32;
constexpr int kNP = kH * 3 + kH + kH * kH + kH + kH + 1;  // 1217
constexpr int kOffB1 = kH * 3, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH;
// Gradient kernel: warps of 32 samples; blocks of four warps, three per SM.
constexpr int kGradWarps = 4;
constexpr int kGradBlocks = 152 * 3;
constexpr int kRow = kH + 4;  // padded row of a sample's 32 activations (conflict-free float4s)

namespace {

__global__ void mlp_forward_kernel(const float *__restrict__ X, long long ns,
                                   const float *__restrict__ P, float *__restrict__ y,
                                   const DevStatus *ds, bool gated) {
    if (scan_off(ds, gated)) return;
    __shared__ float sP[kNP];
    for (int k = threadIdx.x; k < kNP; k += blockDim.x) sP[k] = P[k];
    __syncthreads();
    const float *W1 = sP, *b1 = sP + kOffB1, *W2 = sP + kOffW2, *b2 = sP + kOffB2,
                *W3 = sP + kOffW3;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < ns;
         s += (long long)gridDim.x * blockDim.x) {
        const float x0 = X[3 * s], x1 = X[3 * s + 1], x2 = X[3 * s + 2];
        float a1[kH];
#pragma unroll
        for (int u = 0; u < kH; ++u) {
            float z = b1[u] + W1[3 * u] * x0 + W1[3 * u + 1] * x1 + W1[3 * u + 2] * x2;
            a1[u] = z > 0.f ? z : 0.f;
        }
        float out = sP[kOffB3];
        for (int u = 0; u < kH; ++u) {
            float z = b2[u];
#pragma unroll
            for (int k = 0; k < kH; ++k) z += W2[kH * u + k] * a1[k];
            out += W3[u] * (z > 0.f ? z : 0.f);
        }
        y[s] = out;
    }
}

// Shared memory of the gradient kernel: the weights, the products
// V[u][k] = W2[u][k] W3[u], and per warp three arrays of 32 sample rows.
struct GradSmem {
    float P[(kNP + 3) & ~3];
    float V[kH * kH];
    float4 x[kGradWarps][32];  // a sample's inputs and dL/dyhat
    float a1[kGradWarps][32][kRow];
    float d2[kGradWarps][32][kRow];  // dL/dyhat where unit u of layer 2 is active, else 0
    float s1[kGradWarps][32][kRow];  // layer 2's activations, later dL/dz of layer 1
};

// Stage 1: partial gradient (a sum over the block's samples) and partial
// squared-error sum of every block.
//
// One warp takes 32 samples at a time.  First a lane is a sample: forward and
// backward pass in registers against weights broadcast from shared memory
// (one 16-byte read feeds four multiply-adds).  Then a lane is a tile of the
// gradient: the layer-2 gradient sum_s d2[s][u] a1[s][k] is a 32 x 32 x 32
// product, eight u by four k per lane, three 16-byte reads per 32
// multiply-adds, accumulated in registers over all of the warp's groups.  With
// d2[s][u] = dy_s W3[u] [z2_u > 0], W3[u] is a common factor of row u and is
// multiplied in once per block, not per sample.  About 3,400 multiply-adds per
// sample: FP32-bound.  One block holds 66 KB of shared memory, three run per SM, and
// the grid is at most one wave, so the second stage adds 456 partials at most
// (one block per 64 samples before: 8,457 partials of 41 MB, added by one
// serial thread per parameter in 0.92 ms at 541,199 samples).  The float32 sums grow
// with the groups a warp takes: at 541,199 and 4,000,037 samples (10 and 69 groups)
// the largest error is 2.6e-8 and 8.7e-8 of the gradient's largest entry.
__global__ void __launch_bounds__(32 * kGradWarps, 3)
mlp_grad_partial_kernel(const float *__restrict__ X, const float *__restrict__ Y, long long ns,
                        const float *__restrict__ P, float *__restrict__ partial,
                        float *__restrict__ lossp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GradSmem &sm = *reinterpret_cast<GradSmem *>(smem_raw);
    for (int k = threadIdx.x; k < kNP; k += blockDim.x) sm.P[k] = P[k];
    __syncthreads();
    for (int k = threadIdx.x; k < kH * kH; k += blockDim.x)
        sm.V[k] = sm.P[kOffW2 + k] * sm.P[kOffW3 + k / kH];
    __syncthreads();
    const float *W1 = sm.P, *b1 = sm.P + kOffB1, *W2 = sm.P + kOffW2, *b2 = sm.P + kOffB2,
                *W3 = sm.P + kOffW3;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int ti = (lane >> 3) * 8, tj = (lane & 7) * 4;  // the lane's tile of the layer-2 gradient
    float g2[8][4];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k) g2[u][k] = 0.f;
    float g1x = 0.f, g1y = 0.f, g1z = 0.f, gb1 = 0.f, gb2 = 0.f, g3 = 0.f, gb3 = 0.f, lsum = 0.f;
    const float inv2 = 2.f / (float)ns;
    const long long groups = (ns + 31) >> 5;
    const long long stride = (long long)gridDim.x * kGradWarps;
    for (long long gr = (long long)blockIdx.x * kGradWarps + wid; gr < groups; gr += stride) {
        const long long s = gr * 32 + lane;
        const bool ok = s < ns;
        const float x0 = ok ? X[3 * s] : 0.f, x1 = ok ? X[3 * s + 1] : 0.f,
                    x2 = ok ? X[3 * s + 2] : 0.f;
        float a1[kH];
        unsigned m1 = 0;  // active units of layer 1
#pragma unroll
        for (int u = 0; u < kH; ++u) {
            const float z = b1[u] + W1[3 * u] * x0 + W1[3 * u + 1] * x1 + W1[3 * u + 2] * x2;
            a1[u] = z > 0.f ? z : 0.f;
            m1 |= z > 0.f ? 1u << u : 0u;
        }
#pragma unroll
        for (int u = 0; u < kH; u += 4)
            *reinterpret_cast<float4 *>(&sm.a1[wid][lane][u]) =
                make_float4(a1[u], a1[u + 1], a1[u + 2], a1[u + 3]);
        float yh = sm.P[kOffB3];
        unsigned m2 = 0;  // active units of layer 2
#pragma unroll 1
        for (int u = 0; u < kH; u += 4) {
            float z[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) z[q] = b2[u + q];
#pragma unroll
            for (int k = 0; k < kH; k += 4)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float4 w = *reinterpret_cast<const float4 *>(W2 + kH * (u + q) + k);
                    z[q] += w.x * a1[k];
                    z[q] += w.y * a1[k + 1];
                    z[q] += w.z * a1[k + 2];
                    z[q] += w.w * a1[k + 3];
                }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                m2 |= z[q] > 0.f ? 1u << (u + q) : 0u;
                z[q] = z[q] > 0.f ? z[q] : 0.f;
                yh += W3[u + q] * z[q];
            }
            *reinterpret_cast<float4 *>(&sm.s1[wid][lane][u]) = make_float4(z[0], z[1], z[2], z[3]);
        }
        const float e = ok ? yh - Y[s] : 0.f;
        const float dy = e * inv2;
        lsum += e * e;
        sm.x[wid][lane] = make_float4(x0, x1, x2, dy);
#pragma unroll
        for (int u = 0; u < kH; u += 4)
            *reinterpret_cast<float4 *>(&sm.d2[wid][lane][u]) =
                make_float4((m2 >> u) & 1u ? dy : 0.f, (m2 >> (u + 1)) & 1u ? dy : 0.f,
                            (m2 >> (u + 2)) & 1u ? dy : 0.f, (m2 >> (u + 3)) & 1u ? dy : 0.f);
        __syncwarp();
        // output layer: lane k adds dy_s a2[s][k]
        for (int t = 0; t < 32; ++t) g3 += sm.x[wid][t].w * sm.s1[wid][t][lane];
        gb3 += dy;
        __syncwarp();
        // dL/da1[k] = dy sum_u [z2_u > 0] V[u][k]
        float acc[kH];
#pragma unroll
        for (int k = 0; k < kH; ++k) acc[k] = 0.f;
#pragma unroll 2
        for (int u = 0; u < kH; ++u) {
            const float on = (m2 >> u) & 1u ? 1.f : 0.f;
#pragma unroll
            for (int k = 0; k < kH; k += 4) {
                const float4 v = *reinterpret_cast<const float4 *>(sm.V + kH * u + k);
                acc[k] += on * v.x;
                acc[k + 1] += on * v.y;
                acc[k + 2] += on * v.z;
                acc[k + 3] += on * v.w;
            }
        }
#pragma unroll
        for (int k = 0; k < kH; k += 4)
            *reinterpret_cast<float4 *>(&sm.s1[wid][lane][k]) =
                make_float4((m1 >> k) & 1u ? dy * acc[k] : 0.f,
                            (m1 >> (k + 1)) & 1u ? dy * acc[k + 1] : 0.f,
                            (m1 >> (k + 2)) & 1u ? dy * acc[k + 2] : 0.f,
                            (m1 >> (k + 3)) & 1u ? dy * acc[k + 3] : 0.f);
        __syncwarp();
#pragma unroll 4
        for (int t = 0; t < 32; ++t) {
            const float4 da = *reinterpret_cast<const float4 *>(&sm.d2[wid][t][ti]);
            const float4 db = *reinterpret_cast<const float4 *>(&sm.d2[wid][t][ti + 4]);
            const float4 av = *reinterpret_cast<const float4 *>(&sm.a1[wid][t][tj]);
            const float d[8] = {da.x, da.y, da.z, da.w, db.x, db.y, db.z, db.w};
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                g2[u][0] += d[u] * av.x;
                g2[u][1] += d[u] * av.y;
                g2[u][2] += d[u] * av.z;
                g2[u][3] += d[u] * av.w;
            }
            const float4 xs = sm.x[wid][t];
            const float e1 = sm.s1[wid][t][lane];
            g1x += e1 * xs.x;
            g1y += e1 * xs.y;
            g1z += e1 * xs.z;
            gb1 += e1;
            gb2 += sm.d2[wid][t][lane];
        }
        __syncwarp();  // the rows are rewritten by the next group
    }
    // the warp's sums to shared memory, in the parameter layout, then a
    // fixed-order sum over the warps
    __syncthreads();
    float *red = &sm.a1[0][0][0];  // kGradWarps x kNP: fits in the a1 and d2 rows
    static_assert(kGradWarps * kNP <= 2 * kGradWarps * 32 * kRow, "block sums fit");
    float *w = red + wid * kNP;
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            w[kOffW2 + kH * (ti + u) + tj + k] = g2[u][k] * W3[ti + u];
    w[3 * lane] = g1x;
    w[3 * lane + 1] = g1y;
    w[3 * lane + 2] = g1z;
    w[kOffB1 + lane] = gb1;
    w[kOffB2 + lane] = gb2 * W3[lane];
    w[kOffW3 + lane] = g3;
    for (int o = 16; o > 0; o >>= 1) {
        gb3 += __shfl_down_sync(0xffffffffu, gb3, o);
        lsum += __shfl_down_sync(0xffffffffu, lsum, o);
    }
    float *wl = &sm.s1[0][0][0];
    if (lane == 0) {
        w[kOffB3] = gb3;
        wl[wid] = lsum;
    }
    __syncthreads();
    float *out = partial + (size_t)blockIdx.x * kNP;
    for (int p = threadIdx.x; p < kNP; p += blockDim.x) {
        float t = red[p];
#pragma unroll
        for (int q = 1; q < kGradWarps; ++q) t += red[q * kNP + p];
        out[p] = t;
    }
    if (threadIdx.x == 0) lossp[blockIdx.x] = (wl[0] + wl[1]) + (wl[2] + wl[3]);
    static_assert(kGradWarps == 4, "the sum above");
}

// Stage 2: fixed-order sums over the blocks' partials, in float64.  A block
// takes 32 parameters; its eight warps take every eighth partial.
__global__ void __launch_bounds__(256)
mlp_grad_reduce_kernel(const float *__restrict__ partial, const float *__restrict__ lossp,
                       int nblk, long long ns, float *__restrict__ G, float *__restrict__ loss) {
    __shared__ double part[8][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    const bool is_loss = p == kNP;
    double acc = 0.0;
    if (p < kNP)
        for (int b = wid; b < nblk; b += 8) acc += (double)partial[(size_t)b * kNP + p];
    else if (is_loss)
        for (int b = wid; b < nblk; b += 8) acc += (double)lossp[b];
    part[wid][lane] = acc;
    __syncthreads();
    if (wid != 0) return;
    for (int q = 1; q < 8; ++q) acc += part[q][lane];
    if (p < kNP) G[p] = (float)acc;
    else if (is_loss && loss) *loss = (float)(acc / (double)ns);
}

__global__ void adam_kernel(float *__restrict__ P, const float *__restrict__ G,
                            float *__restrict__ m, float *__restrict__ v, long long np, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= np) return;
    const float g = G[k];
    const float mk = b1 * m[k] + (1.f - b1) * g;
    const float vk = b2 * v[k] + (1.f - b2) * g * g;
    m[k] = mk;
    v[k] = vk;
    P[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

// bounds[b] = first k with inclusive_prefix[k] * nparts > b * total.
__global__ void partition_kernel(const long long *__restrict__ excl, long long ncells, int nparts,
                                 long long *__restrict__ bounds, const DevStatus *ds,
                                 bool gated) {
    if (scan_off(ds, gated)) return;
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > nparts) return;
    if (b == 0) { bounds[0] = 0; return; }
    if (b == nparts) { bounds[nparts] = ncells; return; }
    const long long total = excl[ncells];
    const long long target = (long long)b * total;
    long long lo = 0, hi = ncells;  // search in [lo, hi)
    while (lo < hi) {
        const long long mid = lo + (hi - lo) / 2;
        if (excl[mid + 1] * (long long)nparts > target) hi = mid;
        else lo = mid + 1;
    }
    bounds[b] = lo;
}

// He-uniform initial weights (bound sqrt(6 / fan_in)), zero biases.  The
// uniform deviates come from splitmix64 of (seed, parameter index).
__global__ void mlp_init_kernel(float *P, unsigned long long seed) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kNP) return;
    int fan_in = 0;
    if (k < kOffB1) fan_in = 3;
    else if (k >= kOffW2 && k < kOffB2) fan_in = kH;
    else if (k >= kOffW3 && k < kOffB3) fan_in = kH;
    if (fan_in == 0) {
        P[k] = 0.f;
        return;
    }
    unsigned long long z = seed + (unsigned long long)(k + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double u = ((double)(z >> 11) + 0.5) * (1.0 / 9007199254740992.0);
    const double b = sqrt(6.0 / fan_in);
    P[k] = (float)((2.0 * u - 1.0) * b);
}

}  // namespace

cudaError_t launch_mlp_init(float *P, unsigned long long seed, cudaStream_t s) {
    mlp_init_kernel<<<(kNP + kBlock - 1) / kBlock, kBlock, 0, s>>>(P, seed);
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const float *X, long long ns, const float *P, float *y,
                               cudaStream_t s, const DevStatus *ds, bool gated) {
    if (ns <= 0) return cudaSuccess;
    long long nb = (ns + kBlock - 1) / kBlock;
    int grid = (int)(nb < 152 * 16 ? nb : 152 * 16);
    mlp_forward_kernel<<<grid, kBlock, 0, s>>>(X, ns, P, y, ds, gated);
    return cudaGetLastError();
}

// scratch: at least mlp_grad_scratch_floats(ns) floats
static int mlp_grad_blocks(long long ns) {
    const long long nb = (ns + 32 * kGradWarps - 1) / (32 * kGradWarps);
    return (int)(nb < kGradBlocks ? nb : kGradBlocks);
}
size_t mlp_grad_scratch_floats(long long ns) {
    return (size_t)mlp_grad_blocks(ns) * (kNP + 1) + 1;
}

cudaError_t launch_mlp_loss_grad(const float *X, const float *Y, long long ns, const float *P,
                                 float *G, float *loss, float *scratch, cudaStream_t s) {
    const int nblk = mlp_grad_blocks(ns);
    float *partial = scratch;
    float *lossp = scratch + (size_t)nblk * kNP;
    // over 48 KB of shared memory: set on every call (a host-side attribute of
    // the function on the current device)
    cudaError_t e = cudaFuncSetAttribute(mlp_grad_partial_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(GradSmem));
    if (e != cudaSuccess) return e;
    mlp_grad_partial_kernel<<<nblk, 32 * kGradWarps, sizeof(GradSmem), s>>>(X, Y, ns, P, partial,
                                                                           lossp);
    mlp_grad_reduce_kernel<<<(kNP + 1 + 31) / 32, 256, 0, s>>>(partial, lossp, nblk, ns, G, loss);
    return cudaGetLastError();
}

cudaError_t launch_adam(float *P, const float *G, float *m, float *v, long long np, long long t,
                        float lr, float b1, float b2, float eps, cudaStream_t s) {
    const float c1 = (float)(1.0 - std::pow((double)b1, (double)t));
    const float c2 = (float)(1.0 - std::pow((double)b2, (double)t));
    adam_kernel<<<(int)((np + kBlock - 1) / kBlock), kBlock, 0, s>>>(P, G, m, v, np, lr, b1, b2,
                                                                    eps, c1, c2);
    return cudaGetLastError();
}

// scratch: at least ncells + 1 + ncells / kScanTile + 4 int64
cudaError_t launch_partition(const long long *cost, long long ncells, int nparts,
                             long long *bounds, long long *scratch, cudaStream_t s,
                             const DevStatus *ds, bool gated) {
    long long *excl = scratch;
    long long *bsum = scratch + ncells + 1;
    cudaError_t e = launch_scan<long long>(cost, excl, (int)ncells, bsum, ds, gated, s);
    if (e != cudaSuccess) return e;
    partition_kernel<<<(nparts + 1 + kBlock - 1) / kBlock, kBlock, 0, s>>>(excl, ncells, nparts,
                                                                          bounds, ds, gated);
    return cudaGetLastError();
}

}  // namespace mdg

// ---- C ABI of the cost-model building blocks --------------------------------

namespace {
thread_local std::string g_mlp_error;
}

extern "C" {

md_status md_mlp_forward(const float *X_dev, int64_t ns, const float *P_dev, float *y_dev,
                         void *cuda_stream) {
    if (ns < 0 || (ns > 0 && (!X_dev || !P_dev || !y_dev))) return MD_ERR_INVALID;
    return mdg::launch_mlp_forward(X_dev, ns, P_dev, y_dev, (cudaStream_t)cuda_stream) ==
                   cudaSuccess
               ? MD_OK
               : MD_ERR_CUDA;
}

md_status md_mlp_loss_grad(const float *X_dev, const float *y_dev, int64_t ns,
                           const float *P_dev, float *G_dev, float *loss_dev,
                           void *cuda_stream) {
    if (ns <= 0 || !X_dev || !y_dev || !P_dev || !G_dev) return MD_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    float *scratch = nullptr;
    const size_t bytes = mdg::mlp_grad_scratch_floats(ns) * sizeof(float);
    if (cudaMallocAsync((void **)&scratch, bytes, s) != cudaSuccess) return MD_ERR_OOM;
    cudaError_t e = mdg::launch_mlp_loss_grad(X_dev, y_dev, ns, P_dev, G_dev, loss_dev, scratch, s);
    cudaError_t e2 = cudaFreeAsync(scratch, s);
    return (e == cudaSuccess && e2 == cudaSuccess) ? MD_OK : MD_ERR_CUDA;
}

md_status md_mlp_adam(float *P_dev, const float *G_dev, float *m_dev, float *v_dev, int64_t np,
                      int64_t t, float lr, float beta1, float beta2, float epsilon,
                      void *cuda_stream) {
    if (np <= 0 || t < 1 || !P_dev || !G_dev || !m_dev || !v_dev) return MD_ERR_INVALID;
    return mdg::launch_adam(P_dev, G_dev, m_dev, v_dev, np, t, lr, beta1, beta2, epsilon,
                            (cudaStream_t)cuda_stream) == cudaSuccess
               ? MD_OK
               : MD_ERR_CUDA;
}

md_status md_partition(const int64_t *cost_dev, int64_t ncells, int32_t nparts,
                       int64_t *bounds_dev, void *cuda_stream) {
    if (ncells < 1 || ncells >= ((int64_t)1 << 31) || nparts < 1 || !cost_dev || !bounds_dev)
        return MD_ERR_INVALID;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    long long *scratch = nullptr;
    const size_t words = (size_t)ncells + 1 + (size_t)ncells / mdg::kScanTile + 8;
    if (cudaMallocAsync((void **)&scratch, words * sizeof(long long), s) != cudaSuccess)
        return MD_ERR_OOM;
    cudaError_t e = mdg::launch_partition((const long long *)cost_dev, ncells, nparts,
                                          (long long *)bounds_dev, scratch, s);
    cudaError_t e2 = cudaFreeAsync(scratch, s);
    return (e == cudaSuccess && e2 == cudaSuccess) ? MD_OK : MD_ERR_CUDA;
}

}  // extern "C"

// ---- md_partition without device allocation ----------------------------------
//
// Some callers cannot allocate device memory while they run: a simulation loop
// that fixed its memory budget at start-up, a host framework whose own
// allocator owns the device heap, or a driver setup without stream-ordered
// allocation (cudaMallocAsync unsupported).  md_partition takes its scan
// scratch from cudaMallocAsync; this variant uses a fixed array that lives in
// the library's device image instead.  Every GPU that loads the library holds
// the array (about 8.4 MB) until the process exits.

namespace mdg {
namespace {

constexpr long long kNoAllocMaxCells = 1ll << 20;  // largest ncells accepted
constexpr long long kNoAllocWords = kNoAllocMaxCells + 1 + kNoAllocMaxCells / kScanTile + 8;

// prefix sums of the costs (ncells + 1) followed by the scan's tile sums
static __device__ __align__(256) long long g_partition_scratch[kNoAllocWords];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
long long *g_scratch_addr[kMaxDevices] = {};

// Device address of g_partition_scratch on the current device.  In host code
// the array's name is only a stand-in, so the address is looked up once per
// device (with that device current) and cached.
cudaError_t scratch_address(long long **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_addr[dev]) {
        long long *p = nullptr;
        e = cudaGetSymbolAddress((void **)&p, g_partition_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = p;
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

}  // namespace
}  // namespace mdg

extern "C" md_status md_partition_noalloc(const int64_t *cost_dev, int64_t ncells, int32_t nparts,
                                          int64_t *bounds_dev, void *cuda_stream) {
    if (ncells < 1 || nparts < 1 || !cost_dev || !bounds_dev) {
        mdg::set_thread_error("md_partition_noalloc: bad argument");
        return MD_ERR_INVALID;
    }
    if (ncells > mdg::kNoAllocMaxCells) {
        mdg::set_thread_error("md_partition_noalloc: ncells = " + std::to_string(ncells) +
                              " exceeds the fixed scratch limit of " +
                              std::to_string(mdg::kNoAllocMaxCells) +
                              " cells (use md_partition, which allocates)");
        return MD_ERR_INVALID;
    }
    long long *scratch = nullptr;
    cudaError_t e = mdg::scratch_address(&scratch);
    if (e != cudaSuccess) {
        mdg::set_thread_error(std::string("md_partition_noalloc: cudaGetSymbolAddress: ") +
                              cudaGetErrorString(e));
        return MD_ERR_CUDA;
    }
    // The scan overwrites every scratch word it reads, so nothing needs clearing.
    e = mdg::launch_partition((const long long *)cost_dev, ncells, nparts, (long long *)bounds_dev,
                              scratch, (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) {
        mdg::set_thread_error(std::string("md_partition_noalloc: ") + cudaGetErrorString(e));
        return MD_ERR_CUDA;
    }
    return MD_OK;
}
