// The workers' side of Algorithm 1 on the device, so that a whole synchronous iteration (workers' gradients,
// failures, Zeno_b, update) can run on one GPU without a host round trip:
//   worker_grad_softmax_kernel / worker_grad_lsq_kernel   v_i = grad F_i(x) on worker i's own samples,
//                                                         for softmax regression and for least squares;
//                                                         a worker's labels may be flipped (the
//                                                         experiments' label-flipping failure);
//   inject_faults_kernel                                  the bit-flipping failure (negated gradient, the
//                                                         first faulty row copied over the others) and the
//                                                         failure model's scaled gradient eps * v.
// These kernels build the step's INPUT (the candidate matrix V); they are not on the scoring path.  The sizes
// they are meant for are the paper's (a hundred samples per worker, a model of a few thousand parameters).
#include <math.h>

#include "zeno_internal.h"

namespace zeno {

namespace {

constexpr int kWThreads = 256;
constexpr int kWMaxClasses = 32;
constexpr int kWMaxSmem = 224 * 1024;         // one class pads to four: 12,288 samples' delta and the sums need 200 KB

__device__ __forceinline__ float block_sum(float v, float *scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    float t = 0.f;
    for (int w = 0; w < kWThreads / 32; ++w) t += scratch[w];
    return t;
}

template <typename T> __device__ __forceinline__ void store_elem(T *p, float v);
template <> __device__ __forceinline__ void store_elem<float>(float *p, float v) { *p = v; }
template <> __device__ __forceinline__ void store_elem<__nv_bfloat16>(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

// Softmax regression, worker w = blockIdx.y: samples feats[w][n][in], labels[w][n].
//   delta[j][c] = (softmax(W a_j + b)[c] - [c == label_j]) / n;  dW[c][k] = sum_j delta[j][c] a_j[k];  db[c] = sum_j delta[j][c]
// A cluster of blocks works for one worker: block r takes its share of the samples' logits and leaves their delta in the
// shared memory of all of them, then every block takes its share of the input indices of dW.  Latency is all there is
// (20 workers of 100 samples x 784 inputs read 6 MB, 1 us): one block a worker, with its samples one after another in a
// warp, left 128 SMs idle and took 500 us for those sizes where this takes 22 us.  A block with fewer samples than its
// warps take at a time splits their input range over the warps (256 workers of one sample x 3072 inputs, 20 classes:
// 28 us, 1,750 before; one block a worker: 186).
// dynamic shared memory: delta [n][pitch] (pitch: classes rounded up to 4), then the sample groups' sums.
constexpr int kWCluster = 8;                  // blocks of a worker's cluster at most
constexpr int kWGradWarps = 8;
constexpr int kWSamples = 2;                  // samples a warp takes at a time: the weights are read once for both

// CM: classes the registers are sized for, a multiple of 4.  SPLIT: the kernel for few samples, whose clusters may be of
// fewer than kWCluster blocks.
template <typename T, int CM, bool SPLIT>
__global__ void __launch_bounds__(kWGradWarps * 32, 2)
worker_grad_softmax_kernel(const T *x, int in, int classes, int has_bias, const float *feats, const int32_t *labels, int n,
                           const int32_t *flip, T *V, int64_t ldv) {
    extern __shared__ __align__(16) float delta[];
    constexpr int S = kWSamples, CR = CM <= 4 ? 4 : CM <= 16 ? 16 : 32;
    const int w = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = (int)cluster_rank(), cluster = SPLIT ? (int)gridDim.x : kWCluster;
    const int pitch = (classes + 3) & ~3;
    float *sums = delta + (size_t)n * pitch;
    __shared__ float part_z[SPLIT ? kWGradWarps : 1][S][CR];
    pdl_wait();                               // no early trigger: what follows reads V through the read-only path
    const float *a = feats + (int64_t)w * n * in;
    const int32_t *lab = labels + (int64_t)w * n;
    const bool flipped = flip != nullptr && flip[w] != 0;
    T *out = V + (int64_t)w * ldv;
    const int cls = lane & (CR - 1);
    const float bias = has_bias && cls < classes ? load_elem(x + (int64_t)classes * in + cls) : 0.f;
    cluster_barrier();                        // every block of the cluster runs: their shared memory may be written
    // logits of this block's samples: a warp takes S of them, lanes stride the input index; with fewer of them than warps
    // a sample's warps (warp, warp + units, ..) deal the input range out
    const int per_block = (n + cluster - 1) / cluster;
    const int j_end = min(n, (rank + 1) * per_block);
    const int units = (per_block + S - 1) / S, parts = SPLIT && units < kWGradWarps ? kWGradWarps / units : 1;
    const int part = parts > 1 ? warp / units : 0;
    // one turn if warps share samples, and then all of them take it
    for (int u = parts > 1 ? warp % units : warp; u < units; u += kWGradWarps) {
        const int j0 = rank * per_block + u * S;
        if (!SPLIT && j0 >= j_end) break;
        float z[S][CM];
#pragma unroll
        for (int q = 0; q < S; ++q)
#pragma unroll
            for (int c = 0; c < CM; ++c) z[q][c] = 0.f;
        if (!SPLIT && CM <= 12) {
#pragma unroll 4
            for (int k = lane; k < in; k += 32) {
                float av[S];
#pragma unroll
                for (int q = 0; q < S; ++q) av[q] = __ldg(a + (int64_t)min(j0 + q, j_end - 1) * in + k);
#pragma unroll
                for (int c = 0; c < CM; ++c) {
                    if (c < classes) {
                        const float wv = load_elem(x + (int64_t)c * in + k);
#pragma unroll
                        for (int q = 0; q < S; ++q) z[q][c] = fmaf(wv, av[q], z[q][c]);
                    }
                }
            }
        } else if (!SPLIT || (j0 < j_end && part < parts)) {
            // of more classes the conditions become branches, each with a load to wait for: beyond the classes the last
            // one's weight again, its product dropped
#pragma unroll(CM <= 12 ? 4 : 1)
            for (int k = part * 32 + lane; k < in; k += parts * 32) {
                float av[S], wv[CM];
#pragma unroll
                for (int q = 0; q < S; ++q) av[q] = __ldg(a + (int64_t)min(j0 + q, j_end - 1) * in + k);
#pragma unroll
                for (int c = 0; c < CM; ++c) wv[c] = load_elem(x + (int64_t)min(c, classes - 1) * in + k);
#pragma unroll
                for (int c = 0; c < CM; ++c)
#pragma unroll
                    for (int q = 0; q < S; ++q) z[q][c] = fmaf(wv[c], av[q], z[q][c]);
            }
        }
        // lane c (and its copies CR lanes apart) collects class c, so that a class costs one exponential
        auto collect = [&](int q) {
            float v[CR];
#pragma unroll
            for (int c = 0; c < CR; ++c) v[c] = c < CM ? z[q][c < CM ? c : 0] : 0.f;
            return warp_transpose_reduce<CR>(v, lane);
        };
        if (SPLIT && parts > 1) {
#pragma unroll
            for (int q = 0; q < S; ++q) part_z[warp][q][cls] = collect(q);
            __syncthreads();
            if (part > 0) break;
        }
#pragma unroll
        for (int q = 0; q < S; ++q) {
            float zj;
            if (SPLIT && parts > 1) {
                zj = bias;
                for (int p = 0; p < parts; ++p) zj += part_z[warp + p * units][q][cls];
            } else {
                zj = collect(q) + bias;
            }
            const int j = j0 + q;
            if (j >= j_end) break;
            float zmax = cls < classes ? zj : -INFINITY;
#pragma unroll
            for (int s = CR / 2; s >= 1; s >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, s));
            const float e = cls < classes ? expf(zj - zmax) : 0.f;
            float se = e;
#pragma unroll
            for (int s = CR / 2; s >= 1; s >>= 1) se += __shfl_xor_sync(0xffffffffu, se, s);
            int label = __ldg(lab + j);
            if (flipped) label = classes - 1 - label;
            const float dj = cls < classes ? (e / se - (cls == label ? 1.f : 0.f)) / (float)n : 0.f;
            if (cls < pitch)                  // the copies share the cluster's blocks between them
                for (int r = lane / CR; r < cluster; r += 32 / CR) cluster_store(cluster_addr(delta + (size_t)j * pitch + cls, r), dj);
        }
    }
    cluster_barrier();
    // dW: this block's chunks of 32 input indices, a lane per index, all classes in registers.  With fewer chunks
    // than warps, groups of warps share a chunk and split the samples; their sums are added in group order.
    const int chunks = (in + 31) / 32, per = (chunks + cluster - 1) / cluster;
    const int first = rank * per, mine = min(per, chunks - first);
    const int groups = per >= kWGradWarps ? 1 : kWGradWarps / per;
    const int group = per >= kWGradWarps ? 0 : warp / per;
    const int step = groups > 1 ? per : kWGradWarps;
    const int js = (n + groups - 1) / groups;
    for (int t = groups > 1 ? warp % per : warp; t < per; t += step) {      // one turn if groups share the chunks
        const int k = (first + t) * 32 + lane;
        const bool ok = group < groups && t < mine && k < in;
        float g[CM];
#pragma unroll
        for (int c = 0; c < CM; ++c) g[c] = 0.f;
        if (ok) {
            const int j1 = min(n, (group + 1) * js);
#pragma unroll 8
            for (int j = group * js; j < j1; ++j) {
                const float av = __ldg(a + (int64_t)j * in + k);
                const float4 *dj = reinterpret_cast<const float4 *>(delta + (size_t)j * pitch);
#pragma unroll
                for (int c4 = 0; c4 < CM / 4; ++c4) {
                    if (4 * c4 < pitch) {
                        const float4 d4 = dj[c4];
                        g[4 * c4] = fmaf(d4.x, av, g[4 * c4]);
                        g[4 * c4 + 1] = fmaf(d4.y, av, g[4 * c4 + 1]);
                        g[4 * c4 + 2] = fmaf(d4.z, av, g[4 * c4 + 2]);
                        g[4 * c4 + 3] = fmaf(d4.w, av, g[4 * c4 + 3]);
                    }
                }
            }
        }
        if (groups > 1) {
            if (ok && group > 0) {
#pragma unroll
                for (int c = 0; c < CM; ++c)
                    if (c < classes) sums[(((group - 1) * per + t) * classes + c) * 32 + lane] = g[c];
            }
            __syncthreads();
            if (ok && group == 0) {
                for (int q = 0; q + 1 < groups; ++q)
#pragma unroll
                    for (int c = 0; c < CM; ++c)
                        if (c < classes) g[c] += sums[((q * per + t) * classes + c) * 32 + lane];
            }
        }
        if (ok && group == 0) {
#pragma unroll
            for (int c = 0; c < CM; ++c)
                if (c < classes) store_elem(out + (int64_t)c * in + k, g[c]);
        }
    }
    if (has_bias && rank == cluster - 1) {    // the block with the fewest input indices
        for (int c = warp; c < classes; c += kWGradWarps) {
            float g = 0.f;
            for (int j = lane; j < n; j += 32) g += delta[(size_t)j * pitch + c];
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1) g += __shfl_xor_sync(0xffffffffu, g, s);
            if (lane == 0) store_elem(out + (int64_t)classes * in + c, g);
        }
    }
}

inline size_t worker_grad_smem(int in, int classes, int n, int cluster) {
    const int per = ((in + 31) / 32 + cluster - 1) / cluster;
    const int groups = per >= kWGradWarps ? 1 : kWGradWarps / per;
    return ((size_t)n * ((classes + 3) & ~3) + (size_t)(groups - 1) * per * classes * 32) * sizeof(float);
}

template <typename T, int CM, bool SPLIT>
cudaError_t launch_softmax_split(Context &c, const T *x, int in, int classes, const float *feats, const int32_t *labels, int n,
                                 int m, const int32_t *flip, T *V, int64_t ldv, cudaStream_t s) {
    // fewer blocks a worker where two an SM do not hold them all and they would have no samples for their warps: further
    // waves of blocks with little to do cost more than they bring
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    int cluster = kWCluster;
    while (SPLIT && cluster > 1 && m * cluster > 2 * sms && n < kWGradWarps * kWSamples * cluster) cluster /= 2;
    const size_t smem = worker_grad_smem(in, classes, n, cluster);
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(worker_grad_softmax_kernel<T, CM, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kWMaxSmem);
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    return launch_clustered(worker_grad_softmax_kernel<T, CM, SPLIT>, cluster, dim3(cluster, m), dim3(kWGradWarps * 32), smem, s,
                            chain_launches(c), x, in, classes, (int)c.desc.has_bias, feats, labels, n, flip, V, ldv);
}

// up to 64 samples eight blocks leave at least every second warp without any
template <typename T, int CM>
cudaError_t launch_softmax(Context &c, const T *x, int in, int classes, const float *feats, const int32_t *labels, int n,
                           int m, const int32_t *flip, T *V, int64_t ldv, cudaStream_t s) {
    if (n <= kWCluster * kWGradWarps * kWSamples / 2) return launch_softmax_split<T, CM, true>(c, x, in, classes, feats, labels, n, m, flip, V, ldv, s);
    return launch_softmax_split<T, CM, false>(c, x, in, classes, feats, labels, n, m, flip, V, ldv, s);
}

template <typename T>
cudaError_t launch_softmax_classes(Context &c, const T *x, int in, int classes, const float *feats, const int32_t *labels, int n,
                                   int m, const int32_t *flip, T *V, int64_t ldv, cudaStream_t s) {
    if (classes <= 4) return launch_softmax<T, 4>(c, x, in, classes, feats, labels, n, m, flip, V, ldv, s);
    if (classes <= 12) return launch_softmax<T, 12>(c, x, in, classes, feats, labels, n, m, flip, V, ldv, s);
    if (classes <= 20) return launch_softmax<T, 20>(c, x, in, classes, feats, labels, n, m, flip, V, ldv, s);
    return launch_softmax<T, kWMaxClasses>(c, x, in, classes, feats, labels, n, m, flip, V, ldv, s);
}

// Least squares, worker w = blockIdx.x: A[w][n][d], y[w][n]:  r_j = a_j . x - y_j;  grad[k] = sum_j a_j[k] r_j / n.
// dynamic shared memory: r [n].
__global__ void __launch_bounds__(kWThreads) worker_grad_lsq_kernel(const float *x, int64_t d, const float *A, const float *y,
                                                                     int n, float *V, int64_t ldv) {
    extern __shared__ float r[];
    __shared__ float scratch[kWThreads / 32];
    const int w = blockIdx.x;
    const float *a = A + (int64_t)w * n * d;
    for (int j = 0; j < n; ++j) {
        float s = 0.f;
        for (int64_t k = threadIdx.x; k < d; k += kWThreads) s = fmaf(a[(int64_t)j * d + k], x[k], s);
        s = block_sum(s, scratch);
        if (threadIdx.x == 0) r[j] = s - y[(int64_t)w * n + j];
    }
    __syncthreads();
    float *out = V + (int64_t)w * ldv;
    for (int64_t k = threadIdx.x; k < d; k += kWThreads) {
        float g = 0.f;
        for (int j = 0; j < n; ++j) g = fmaf(a[(int64_t)j * d + k], r[j], g);
        out[k] = g / (float)n;
    }
}

// mode 0: V[faulty[f]] = -V[faulty[0]] for every f (the first faulty row is negated in place, after the
// others have copied it: blocks of columns are independent, a thread owns a column); mode 1: V[faulty[f]] *= eps.
template <typename T>
__global__ void __launch_bounds__(256) inject_faults_kernel(T *V, int64_t ldv, int64_t d, const int32_t *faulty, int n_faulty,
                                                            int m, int mode, float eps) {
    pdl_wait();                               // no early trigger: what follows reads V through the read-only path
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < d; k += (int64_t)gridDim.x * blockDim.x) {
        if (mode == 0) {
            const int f0 = __ldg(faulty);
            if (f0 < 0 || f0 >= m) continue;
            const float v = -load_elem(V + (int64_t)f0 * ldv + k);
#pragma unroll 4
            for (int f = 0; f < n_faulty; ++f) {
                const int row = __ldg(faulty + f);
                if (row >= 0 && row < m) store_elem(V + (int64_t)row * ldv + k, v);
            }
        } else {
            for (int f = 0; f < n_faulty; ++f) {
                const int row = faulty[f];
                if (row >= 0 && row < m) store_elem(V + (int64_t)row * ldv + k, eps * load_elem(V + (int64_t)row * ldv + k));
            }
        }
    }
}

}  // namespace

bool worker_gradients_supported(const Context &c, int n) {
    if (n < 1) return false;
    if (c.desc.kind == ZENO_LOSS_LEAST_SQUARES) return c.desc.param_dtype == ZENO_F32 && n <= 4096;
    if (c.desc.kind != ZENO_LOSS_SOFTMAX_MLP) return false;
    return c.desc.n_layers == 1 && c.desc.dims[1] <= kWMaxClasses && (int64_t)n * c.desc.dims[1] * 4 <= 48 * 1024;
}

cudaError_t launch_worker_gradients(Context &c, const void *x, const float *features, const void *targets, int n, int m,
                                    const int32_t *flip, void *V, int64_t ldv, cudaStream_t s, int *launches) {
    ++*launches;
    profile_mark(c, "worker_gradients", s);
    if (c.desc.kind == ZENO_LOSS_LEAST_SQUARES) {
        worker_grad_lsq_kernel<<<m, kWThreads, (size_t)n * sizeof(float), s>>>(static_cast<const float *>(x), c.d, features,
                                                                              static_cast<const float *>(targets), n,
                                                                              static_cast<float *>(V), ldv);
        return cudaGetLastError();
    }
    const int in = (int)c.desc.dims[0], classes = (int)c.desc.dims[1];
    const int32_t *labels = static_cast<const int32_t *>(targets);
    if (c.desc.param_dtype == ZENO_BF16)
        return launch_softmax_classes(c, static_cast<const __nv_bfloat16 *>(x), in, classes, features, labels, n, m, flip,
                                      static_cast<__nv_bfloat16 *>(V), ldv, s);
    return launch_softmax_classes(c, static_cast<const float *>(x), in, classes, features, labels, n, m, flip,
                                  static_cast<float *>(V), ldv, s);
}

cudaError_t launch_inject_faults(Context &c, void *V, int64_t ldv, int m, const int32_t *faulty, int n_faulty, int mode,
                                 float eps, cudaStream_t s, int *launches) {
    ++*launches;
    profile_mark(c, "inject_faults", s);
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    int64_t want = (c.d + 255) / 256;
    const int blocks = (int)(want < (int64_t)sms * 8 ? (want < 1 ? 1 : want) : (int64_t)sms * 8);
    if (c.desc.param_dtype == ZENO_BF16)
        return launch_chained(inject_faults_kernel<__nv_bfloat16>, dim3(blocks), dim3(256), 0, s, chain_launches(c),
                              static_cast<__nv_bfloat16 *>(V), ldv, c.d, faulty, n_faulty, m, mode, eps);
    return launch_chained(inject_faults_kernel<float>, dim3(blocks), dim3(256), 0, s, chain_launches(c), static_cast<float *>(V),
                          ldv, c.d, faulty, n_faulty, m, mode, eps);
}

}  // namespace zeno
