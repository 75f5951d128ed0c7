// The server loop of a small softmax regression in binary32 (Algorithm 1, server lines) in two launches.
//
// An iteration of such a model is a chain of latencies: two kernels that each wait for the other take 9 us for 0.6 MB.  The
// logits are linear in the parameters, X (x - gamma v)^T = X x^T - gamma X v^T, and X v^T does not depend on what the loop has
// done so far: loop_products_kernel takes the products and the norms of many iterations' candidates at once, on the whole
// device.  What is left to do in turn is small enough for one cluster of sixteen blocks.  Block r owns a stretch of the
// parameter vector: its entries of x stay in shared memory from the first iteration to the last, and its entries of the m
// candidates are there while an iteration lasts (the next iteration's on their way, where two copies fit).  An iteration:
//   1. the products of the block's entries of x with the batch's features go to all sixteen blocks;
//   2. every block adds them up and takes the cross-entropy of its models (model c: block c mod 16), which goes to all;
//   3. every block forms all scores and the ranking for itself, averages its own columns of the selected rows, in rank
//      order as the averaging kernel does, and updates its own entries of x.
// Two cluster barriers an iteration are all the waiting there is.  784 x 10, 20 candidates, 4 samples: 4.4 us an iteration where
// the step's kernels take 9.0; one launch that forms every candidate's logits in turn took 8.3.
#include <atomic>

#include "zeno_internal.h"

namespace zeno {

namespace {

constexpr int kLoopCluster = 16, kLoopThreads = 512, kLoopWarps = kLoopThreads / 32;
constexpr int kLoopMaxClasses = 32;              // a lane a class
constexpr int kLoopParts = 4;                    // parts of a block's stretch
constexpr int kLoopSamples = 4;                  // samples a warp takes at a time
constexpr size_t kLoopSmem = 220 * 1024;
constexpr int kLoopLosses = 5;                   // losses a warp takes one after another, at most
constexpr int kLoopBatch = 32;                   // iterations whose products a handle has room for, at least,
constexpr int64_t kLoopProducts = 1 << 20;       // but no more floats than this

// How a cluster divides a model, and where a block's shared memory holds what (bytes from its start; x at 0).
struct LoopPlan {
    int sl, n, G;                                // entries of a part and of a stretch; parts in all
    int each;                                    // every sample's loss is handed out, not their sum
    int ML, zslots;                              // models of a block; partial logits of a sample, at most
    int hw, whole;                               // staged columns of the features: their whole rows, or those of the stretch
    int bufs, copy, feature_copy;                // copies of an iteration's inputs; bytes of an asynchronous copy of V and of the features
    int at_loss, at_lossd, at_keys, at_v, at_h, at_lab, at_prod, at_norm, at_z, at_bias, at_rows;
    int v_bytes, h_bytes, prod_bytes, norm_bytes, bytes;
};

struct LoopArgs {
    float *x;
    const float *V;
    int64_t ldv, stride_v;
    const float *features;
    const int32_t *labels;
    const float *products, *norms;               // [steps][m][n_r][classes], [steps][m]
    int d, in, classes, m, n_r, steps, keep;
    float gamma, rho;
    float *scores;                               // [steps][m] or NULL
    int32_t *idx;                                // [steps][keep] or NULL
    LoopPlan p;
};

template <int BYTES>
__device__ __forceinline__ void loop_copy(void *dst, const void *src) { cp_async<BYTES>((uint32_t)__cvta_generic_to_shared(dst), src); }
__device__ __forceinline__ void cluster_store_double(uint32_t addr, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
// the largest of the lanes' values (a NaN with its sign clear counts as larger than all)
__device__ __forceinline__ float loop_warp_max(float v) {
    const int b = __float_as_int(v), k = __reduce_max_sync(0xffffffffu, b ^ ((b >> 31) & 0x7fffffff));
    return __int_as_float(k ^ ((k >> 31) & 0x7fffffff));
}
// the two halves of a cluster barrier
__device__ __forceinline__ void loop_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void loop_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// products[t][c][j][o] = sum_k features[t][j][k] V[t][c][o][k] + the candidate's bias entry o; norms[t][c] = ||v||^2.
// A block per candidate and iteration, a warp per class and part of the columns, lanes along the columns, NS samples at a time.
// A part has at most 2,048 columns: a lane's sums are of 64 products however wide the model is.
constexpr int kProductWarps = 8, kProductCols = 2048, kProductUnits = 128;
template <int NS>
__global__ void __launch_bounds__(kProductWarps * 32) loop_products_kernel(const float *V, int64_t ldv, int64_t stride_v, const float *features, int in,
                                                                          int classes, int has_bias, int parts, int m, int n_r, float *products, float *norms) {
    __shared__ float norm_part[kProductWarps], part[2][kProductUnits][NS];
    pdl_wait();
    pdl_launch_dependents();
    const int c = blockIdx.x, t = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float *v = V + (int64_t)t * stride_v + (int64_t)c * ldv;
    const float *f = features + (int64_t)t * n_r * in;
    float *out = products + ((int64_t)t * m + c) * n_r * classes;
    const int len = ((in + parts - 1) / parts + 31) / 32 * 32;
    float nrm = 0.f;
    auto bias_of = [&](int o) { return has_bias ? __ldg(v + (int64_t)classes * in + o) : 0.f; };
    for (int j0 = 0, b = 0; j0 < n_r; j0 += NS, b ^= 1) {
        for (int unit = warp; unit < classes * parts; unit += kProductWarps) {
            const int o = unit / parts, k0 = (unit - o * parts) * len, k1 = min(in, k0 + len);
            const float *row = v + (int64_t)o * in;
            float acc[NS];
            const float *h[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                acc[s] = 0.f;
                h[s] = f + (int64_t)min(j0 + s, n_r - 1) * in;
            }
#pragma unroll 4
            for (int k = k0 + lane; k < k1; k += 32) {
                const float vv = __ldg(row + k);
                if (j0 == 0) nrm = fmaf(vv, vv, nrm);
#pragma unroll
                for (int s = 0; s < NS; ++s) acc[s] = fmaf(vv, __ldg(h[s] + k), acc[s]);
            }
            const float z = warp_transpose_reduce<NS>(acc, lane);
            if (parts > 1) {
                if (lane < NS) part[b][unit][lane] = z;
            } else {
                const float bias = bias_of(o);
                if (lane == 0 && j0 == 0) nrm = fmaf(bias, bias, nrm);
                if (lane < NS && j0 + lane < n_r) out[(j0 + lane) * classes + o] = z + bias;
            }
        }
        if (parts == 1) continue;
        __syncthreads();             // the other buffer is written next
        for (int q = threadIdx.x; q < classes * NS; q += kProductWarps * 32) {
            const int o = q / NS, s = q - o * NS;
            float z = 0.f;
            for (int p = 0; p < parts; ++p) z += part[b][o * parts + p][s];
            const float bias = bias_of(o);
            if (j0 + s < n_r) out[(j0 + s) * classes + o] = z + bias;
            if (j0 == 0 && s == 0) nrm = fmaf(bias, bias, nrm);
        }
    }
    nrm = warp_sum(nrm);
    if (lane == 0) norm_part[warp] = nrm;
    __syncthreads();
    if (threadIdx.x == 0) {
        float n = 0.f;
        for (int w = 0; w < kProductWarps; ++w) n += norm_part[w];
        norms[(int64_t)t * m + c] = n;
    }
}

__global__ void __launch_bounds__(kLoopThreads, 1) softmax_loop_kernel(const __grid_constant__ LoopArgs a) {
    extern __shared__ __align__(16) uint8_t sm[];
    const LoopPlan &p = a.p;
    float *xs = reinterpret_cast<float *>(sm);
    double *loss_s = reinterpret_cast<double *>(sm + p.at_loss), *lossd = reinterpret_cast<double *>(sm + p.at_lossd);
    unsigned long long *keys = reinterpret_cast<unsigned long long *>(sm + p.at_keys);
    int *lab_s = reinterpret_cast<int *>(sm + p.at_lab), *rows = reinterpret_cast<int *>(sm + p.at_rows);
    float *zpart = reinterpret_cast<float *>(sm + p.at_z), *biasw = reinterpret_cast<float *>(sm + p.at_bias);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rank = (int)cluster_rank();
    const int p0 = rank * p.n, own = max(0, min(p.n, a.d - p0));            // this block's entries
    const int nw = a.in * a.classes;                                        // weights, before the bias
    const int k0 = p0 % a.in;                                               // column of the first one
    // what a lane adds up as class `lane`: the parts its weights lie in
    const int part_lo = lane * a.in / p.sl, part_hi = (lane * a.in + a.in - 1) / p.sl;
    const int mine = rank <= a.m ? (a.m - rank) / kLoopCluster + 1 : 0;     // models rank, rank + 16, ..
    const int sample_groups = (a.n_r + kLoopSamples - 1) / kLoopSamples;
    const double inv_n = 1.0 / (double)a.n_r;
    // integer divisions cost as much as everything else a phase does: what they give does not change from one iteration to the next
    const int split = a.n_r >= kLoopWarps ? 1 : kLoopWarps / a.n_r;         // warps that load a sample's features
    const int my_part = warp & (kLoopParts - 1), my_class = (p0 + my_part * p.sl) / a.in;
    const int lm0 = warp / a.n_r, j_first = warp - lm0 * a.n_r, lm_step = kLoopWarps / a.n_r, j_step = kLoopWarps - lm_step * a.n_r;
    const int f_sample = (kLoopWarps - 1 - warp) / split, f_part = (kLoopWarps - 1 - warp) - f_sample * split;
    // a lane's place in the other blocks when it hands out a warp's four sums: sample lane % 4, blocks lane / 4 and 8 on
    const uint32_t z_a = cluster_addr(zpart, lane >> 2), z_b = cluster_addr(zpart, 8 + (lane >> 2));

    pdl_wait();                      // no early trigger: x is written here and read through the read-only path elsewhere
    auto load = [&](int t, int buf) {            // the last warps first: the first ones have products to take
        const int w = kLoopWarps - 1 - warp;
        float *vs = reinterpret_cast<float *>(sm + p.at_v + buf * p.v_bytes);
        float *hs = reinterpret_cast<float *>(sm + p.at_h + buf * p.h_bytes);
        const float *src = a.V + (int64_t)t * a.stride_v + p0;
        for (int i = w; i < a.m; i += kLoopWarps) {
            const float *row = src + (int64_t)i * a.ldv;
            float *dst = vs + i * p.n;
            if (p.copy == 16) {
                for (int q = lane * 4; q < own; q += 128) loop_copy<16>(dst + q, row + q);
            } else {
                for (int q = lane; q < own; q += 32) loop_copy<4>(dst + q, row + q);
            }
        }
        const float *f = a.features + (int64_t)t * a.n_r * a.in;
        const int cols = p.whole ? a.in : own, first = p.whole ? 0 : k0;     // of a stretch that is shorter than a row
        const int E = p.feature_copy / 4;
        for (int j = f_sample; j < a.n_r; j += split > 1 ? a.n_r : kLoopWarps)
            for (int q = (f_part * 32 + lane) * E; q < cols; q += 32 * split * E) {
                const int k = first + q;
                const float *from = f + (int64_t)j * a.in + (k >= a.in ? k - a.in : k);
                if (E == 4) loop_copy<16>(hs + j * p.hw + q, from);
                else loop_copy<4>(hs + j * p.hw + q, from);
            }
        float *prod = reinterpret_cast<float *>(sm + p.at_prod + buf * p.prod_bytes);
        const int per_model = a.n_r * a.classes;
        for (int lm = rank == 0 ? 1 : 0; lm < mine; ++lm) {
            const float *from = a.products + ((int64_t)t * a.m + lm * kLoopCluster + rank - 1) * per_model;
            for (int q = tid; q < per_model; q += kLoopThreads) loop_copy<4>(prod + lm * per_model + q, from + q);
        }
        float *norm = reinterpret_cast<float *>(sm + p.at_norm + buf * p.norm_bytes);
        for (int i = tid; i < a.m; i += kLoopThreads) loop_copy<4>(norm + i, a.norms + (int64_t)t * a.m + i);
        for (int j = tid; j < a.n_r; j += kLoopThreads) loop_copy<4>(lab_s + buf * a.n_r + j, a.labels + (int64_t)t * a.n_r + j);
        cp_async_commit();
    };
    load(0, 0);
    for (int q = tid; q < own; q += kLoopThreads) xs[q] = a.x[p0 + q];
    if (tid < kLoopMaxClasses) biasw[tid] = 0.f;
    cluster_barrier();               // every block runs, its bias entries are cleared

    for (int t = 0; t < a.steps; ++t) {
        const int buf = p.bufs == 2 ? t & 1 : 0;
        cp_async_wait<0>();
        __syncthreads();             // x is updated and this iteration's inputs are here
        const float *vs = reinterpret_cast<const float *>(sm + p.at_v + buf * p.v_bytes);
        const float *hs = reinterpret_cast<const float *>(sm + p.at_h + buf * p.h_bytes);

        // ---- 1: X x^T of this block's entries
        for (int group = warp / kLoopParts; group < sample_groups; group += kLoopWarps / kLoopParts) {
            const int j0 = group * kLoopSamples, g = rank * kLoopParts + my_part;
            int q = my_part * p.sl;
            const int q_end = min(q + p.sl, own);
            for (int o = my_class; q < q_end && o < a.classes; ++o) {
                const int q_seg = min(q_end, (o + 1) * a.in - p0);
                const float *h = hs + j0 * p.hw + (p.whole ? p0 - o * a.in : 0);
                float acc[kLoopSamples] = {};
#pragma unroll 4
                for (int u = q + lane; u < q_seg; u += 32) {
                    const float w = xs[u];
#pragma unroll
                    for (int s = 0; s < kLoopSamples; ++s) acc[s] = fmaf(w, h[s * p.hw + u], acc[s]);
                }
                const float z = warp_transpose_reduce<kLoopSamples>(acc, lane);      // lane l: the sum of sample l % 4
                const int j = j0 + (lane & 3);
                if (j < a.n_r) {
                    cluster_store(z_a + 4 * ((g + o) * a.n_r + j), z);
                    cluster_store(z_b + 4 * ((g + o) * a.n_r + j), z);
                }
                q = q_seg;
            }
        }
        if (p0 + own > nw) {                                     // the bias entries
            for (int u = max(nw - p0, 0) + warp; u < own; u += kLoopWarps)
                if (lane < kLoopCluster) cluster_store(cluster_addr(biasw + p0 + u - nw, lane), xs[u]);
        }
        loop_arrive();               // what the others wait for is on its way
        if (t + 1 < a.steps) {
            if (p.bufs == 2) {
                load(t + 1, buf ^ 1);
            } else {                 // at least into L2
                const char *src = reinterpret_cast<const char *>(a.V + (int64_t)(t + 1) * a.stride_v + p0);
                for (int i = warp; i < a.m; i += kLoopWarps)
                    for (int q = lane * 128; q < own * 4; q += 32 * 128)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(src + (int64_t)i * a.ldv * 4 + q));
            }
        }
        loop_wait();

        // ---- 2: losses of this block's models
        const float *prod = reinterpret_cast<const float *>(sm + p.at_prod + buf * p.prod_bytes);
        for (int lm = lm0, j = j_first; lm < mine;) {
            double z = 0.0;
            if (lane < a.classes) {
                const float *zp = zpart + lane * a.n_r + j;
#pragma unroll 4
                for (int g = part_lo; g <= part_hi; ++g) z += (double)zp[g * a.n_r];
                z += (double)biasw[lane];
                if (lm > 0 || rank > 0) z -= (double)a.gamma * (double)prod[(lm * a.n_r + j) * a.classes + lane];
            }
            // what the exponentials are taken against: the largest logit's float, or, where a float is too coarse, itself
            double ref = (double)loop_warp_max(lane < a.classes ? (float)z : -INFINITY);
            if (!(fabs(ref) < 1e5)) {
                ref = lane < a.classes ? z : -INFINITY;
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) ref = fmax(ref, __shfl_xor_sync(0xffffffffu, ref, s));
            }
            const float se = warp_sum(lane < a.classes ? expf((float)(z - ref)) : 0.f);      // a NaN logit makes se NaN
            int l = lab_s[buf * a.n_r + j];
            if (l < 0 || l >= a.classes) l = 0;
            const double zl = __shfl_sync(0xffffffffu, z, l);
            const double loss = (ref - zl) + (double)logf(se);
            // few samples: every one's loss goes to all blocks, which add them up; else their sum
            if (p.each) {
                if (lane < kLoopCluster) cluster_store_double(cluster_addr(lossd + (lm * kLoopCluster + rank) * a.n_r + j, lane), loss);
            } else if (lane == 0) {
                loss_s[lm * a.n_r + j] = loss;
            }
            lm += lm_step;
            j += j_step;
            if (j >= a.n_r) { j -= a.n_r; ++lm; }
        }
        if (!p.each) {
            __syncthreads();
            for (int lm = warp; lm < mine; lm += kLoopWarps) {
                double l = 0.0;
                for (int j = lane; j < a.n_r; j += 32) l += loss_s[lm * a.n_r + j];
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) l += __shfl_xor_sync(0xffffffffu, l, s);
                if (lane < kLoopCluster) cluster_store_double(cluster_addr(lossd + lm * kLoopCluster + rank, lane), l);
            }
        }
        cluster_barrier();

        // ---- 3: scores, ranking, average, update
        const float *norm = reinterpret_cast<const float *>(sm + p.at_norm + buf * p.norm_bytes);
        for (int i = tid; i < a.m; i += kLoopThreads) {
            double diff = 0.0;
            if (p.each) {
                for (int j = 0; j < a.n_r; ++j) diff += lossd[j] - lossd[(1 + i) * a.n_r + j];
            } else {
                diff = lossd[0] - lossd[1 + i];
            }
            const float sc = (float)(diff * inv_n - (double)a.rho * (double)norm[i]);
            if (rank == 0 && a.scores) a.scores[(int64_t)t * a.m + i] = sc;
            keys[i] = rank_key(sc, i);
        }
        __syncthreads();
        for (int i = warp; i < a.m; i += kLoopWarps) {
            const unsigned long long key = keys[i];
            int better = 0;
            for (int j = lane; j - lane < a.m; j += 32) better += __popc(__ballot_sync(0xffffffffu, j < a.m && keys[j] > key));
            if (lane == 0 && better < a.keep) {
                rows[better] = i * p.n;
                if (rank == 0 && a.idx) a.idx[(int64_t)t * a.keep + better] = i;
            }
        }
        __syncthreads();
        for (int q = tid; q < own; q += kLoopThreads) {
            float acc = 0.f;
#pragma unroll 8
            for (int r = 0; r < a.keep; ++r) acc += vs[rows[r] + q];
            xs[q] = fmaf(-a.gamma, acc / (float)a.keep, xs[q]);
        }
        if (p.bufs == 1 && t + 1 < a.steps) {
            __syncthreads();         // the candidates have been read
            load(t + 1, 0);
        }
    }
    for (int q = tid; q < own; q += kLoopThreads) a.x[p0 + q] = xs[q];
}

// Parts of a class: as few of up to 2,048 columns as leave the eight warps even shares, a part's start and end counting as 384
// columns.  Iterations whose products fill a warp or two a block wait for them: 16384 x 2 of five candidates, one sample, four
// iterations take 35 us, with a warp a class 53; 0 where there would be more than a block has room for.
int product_parts(int in, int classes) {
    const int least = (in + kProductCols - 1) / kProductCols;
    int best = 0;
    int64_t cost = 0;
    for (int p = least; p < least + 8 && p * classes <= kProductUnits; ++p) {
        const int64_t len = ((in + p - 1) / p + 31) / 32 * 32, c = (classes * p + kProductWarps - 1) / kProductWarps * (len + 384);
        if (!best || c < cost) { best = p; cost = c; }
    }
    return best;
}

bool loop_plan(int64_t d, int in, int classes, int m, int n_r, LoopPlan *p) {
    if (!product_parts(in, classes)) return false;
    if (classes > kLoopMaxClasses || m > kRankMax || d > (int64_t)kLoopSmem * kLoopCluster || n_r > (int)kLoopSmem) return false;
    p->G = kLoopCluster * kLoopParts;
    p->sl = (int)(((d + p->G - 1) / p->G + 7) / 8 * 8);
    p->n = p->sl * kLoopParts;
    p->ML = m / kLoopCluster + 1;
    p->whole = p->n > in;
    p->hw = p->whole ? in : p->n;
    p->zslots = p->G + classes;
    p->each = n_r <= 8;
    const int64_t n_pad = (n_r + kLoopSamples - 1) / kLoopSamples * kLoopSamples;
    for (p->bufs = 2; p->bufs >= 1; --p->bufs) {
        int64_t at = 0;
        auto take = [&](int64_t bytes) {
            const int64_t here = at;
            at += (bytes + 15) / 16 * 16;
            return (int)here;
        };
        auto whole16 = [](int64_t bytes) { return (bytes + 15) / 16 * 16; };
        const int64_t v_bytes = whole16((int64_t)m * p->n * 4), h_bytes = whole16(n_pad * p->hw * 4);
        const int64_t prod_bytes = whole16((int64_t)p->ML * n_r * classes * 4), norm_bytes = whole16((int64_t)m * 4);
        take((int64_t)p->n * 4);                                   // x
        p->at_loss = take((int64_t)p->ML * n_r * 8);
        p->at_lossd = take((int64_t)p->ML * kLoopCluster * 8 * (p->each ? n_r : 1));
        p->at_keys = take((int64_t)m * 8);
        p->at_v = take(v_bytes * p->bufs);
        p->at_h = take(h_bytes * p->bufs);
        p->at_lab = take((int64_t)n_r * 4 * p->bufs);
        p->at_prod = take(prod_bytes * p->bufs);
        p->at_norm = take(norm_bytes * p->bufs);
        p->at_z = take((int64_t)p->zslots * n_r * 4);
        p->at_bias = take((int64_t)kLoopMaxClasses * 4);
        p->at_rows = take((int64_t)m * 4);
        if (at > (int64_t)kLoopSmem) continue;
        p->v_bytes = (int)v_bytes;
        p->h_bytes = (int)h_bytes;
        p->prod_bytes = (int)prod_bytes;
        p->norm_bytes = (int)norm_bytes;
        p->bytes = (int)at;
        return true;
    }
    return false;
}

cudaError_t set_attributes() {
    cudaError_t e = cudaFuncSetAttribute(softmax_loop_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLoopSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(softmax_loop_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// Whether the device, the current one, holds the cluster: asked once, by the first loop that could use it (the answer takes two
// milliseconds).  The functions' attributes are set on the way.
bool cluster_fits(int device) {
    static std::atomic<signed char> known[kMaxDevices];          // 0: not asked, 1: yes, -1: no
    const bool keep = device >= 0 && device < kMaxDevices;
    if (keep && known[device].load(std::memory_order_relaxed)) return known[device].load(std::memory_order_relaxed) > 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kLoopCluster);
    cfg.blockDim = dim3(kLoopThreads);
    cfg.dynamicSmemBytes = kLoopSmem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kLoopCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (set_attributes() != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, softmax_loop_kernel, &cfg) != cudaSuccess) {
        cudaGetLastError();          // no answer: the steps' kernels this time
        return false;
    }
    if (keep) known[device].store(n >= 1 ? 1 : -1, std::memory_order_relaxed);
    return n >= 1;
}

}  // namespace

// Floats of the products a handle keeps room for, 0 where it never takes this path: another model, sizes beyond the shared
// memory with the fewest candidates and samples.  They lie where Krum's partial sums do: a handle's calls are ordered.
int64_t loop_workspace(const zeno_model_desc &desc, int64_t d, int m_max, int n_r_max) {
    if (desc.kind != ZENO_LOSS_SOFTMAX_MLP || desc.n_layers != 1 || desc.param_dtype != ZENO_F32) return 0;
    LoopPlan p;
    if (desc.dims[0] > (1 << 20) || desc.dims[1] > kLoopMaxClasses || !loop_plan(d, (int)desc.dims[0], (int)desc.dims[1], 1, 1, &p)) return 0;
    // most of m n_r: the m candidates are less than a block's models times the blocks
    const int64_t most = kLoopLosses * kLoopWarps * kLoopCluster, rows = (int64_t)m_max * n_r_max < most ? (int64_t)m_max * n_r_max : most;
    const int64_t need = kLoopBatch * (rows * desc.dims[1] + m_max);
    return need < kLoopProducts ? need : kLoopProducts;
}

// iterations whose products fit the handle's room
static int64_t loop_batch(const Context &c, int m, int n_r) { return c.loop_floats / ((int64_t)m * ((int64_t)n_r * c.desc.dims[1] + 1)); }

bool loop_usable(const Context &c, int m, int n_r, int steps, bool aligned) {
    if (!c.loop_ws || steps < kLoopMinSteps) return false;
    LoopPlan p;
    if (!loop_plan(c.d, (int)c.desc.dims[0], (int)c.desc.dims[1], m, n_r, &p) || loop_batch(c, m, n_r) < kLoopMinSteps) return false;
    // sixteen blocks against all: up to five losses a warp, one after another, and so many products of a block.  Eight iterations
    // by the step's kernels and by these, us: 784 x 10 of 20 candidates 75 and 46 with 4 samples, 85 and 68 with 16, 97 and 125
    // with 32; 4096 x 4 of 12 candidates 70 and 69 with 8 samples, 81 and 106 with 16; 100 x 4 of 64 candidates 76 and 64 with
    // 16 samples, 109 and 130 with 32; 200 x 10 of 128 candidates, 8 samples: 103 and 67
    if ((p.ML * n_r + kLoopWarps - 1) / kLoopWarps > kLoopLosses || n_r * p.n > 8800) return false;
    // Wide models whose steps are quick, with loads of four columns and less than 12 us each: few iterations do not pay for the
    // products and the first candidates' copies, and copies that nothing overlaps take as long as a step.  us, steps and loop:
    // 4096 x 10 of 5 candidates, one sample, four iterations 31 and 38, eight 62 and 60; 4096 x 4 of 12, 8 samples 33 and 34, 64 and
    // 54; 1024 x 32 of 20, one copy of 166 KB, eight 73 and 89, twenty with 4 samples 181 and 186.  2395 x 9 of 15, no such loads: four
    // 52 and 44; 16384 x 2 of 20: four 56 and 51
    const bool quick_steps = (aligned || m < 3) && c.desc.dims[0] < 8192;
    if (quick_steps && steps < 8 && (p.n > 1250 || (p.bufs == 1 && n_r * p.n > 8000))) return false;
    return (!quick_steps || p.bufs == 2 || p.n <= 1400) && cluster_fits(c.device);
}

cudaError_t launch_loop(Context &c, float *x, const float *V, int64_t ldv, int64_t stride_v, int m, const float *features, const int32_t *labels,
                        int n_r, int steps, float gamma, float rho, int keep, float *scores, int32_t *idx, cudaStream_t s, int *launches) {
    LoopArgs a;
    a.x = x;
    a.ldv = ldv;
    a.stride_v = stride_v;
    a.d = (int)c.d;
    a.in = (int)c.desc.dims[0];
    a.classes = (int)c.desc.dims[1];
    a.m = m;
    a.n_r = n_r;
    a.keep = keep;
    a.gamma = gamma;
    a.rho = rho;
    if (!loop_plan(c.d, a.in, a.classes, m, n_r, &a.p)) return cudaErrorInvalidValue;
    // a block's stretch starts at a multiple of eight entries
    a.p.copy = reinterpret_cast<uintptr_t>(V) % 16 == 0 && ldv % 4 == 0 && stride_v % 4 == 0 ? 16 : 4;
    a.p.feature_copy = reinterpret_cast<uintptr_t>(features) % 16 == 0 && a.in % 4 == 0 ? 16 : 4;
    const int parts = product_parts(a.in, a.classes);
    const int batch = (int)(loop_batch(c, m, n_r) < 32768 ? loop_batch(c, m, n_r) : 32768);
    const int batches = (steps + batch - 1) / batch, each = (steps + batches - 1) / batches;
    profile_mark(c, "server_loop", s);
    for (int t0 = 0; t0 < steps; t0 += each) {
        a.steps = steps - t0 < each ? steps - t0 : each;
        a.V = V + (int64_t)t0 * stride_v;
        a.features = features + (int64_t)t0 * n_r * a.in;
        a.labels = labels + (int64_t)t0 * n_r;
        a.products = c.loop_ws;
        a.norms = c.loop_ws + (int64_t)a.steps * m * n_r * a.classes;
        a.scores = scores ? scores + (int64_t)t0 * m : nullptr;
        a.idx = idx ? idx + (int64_t)t0 * keep : nullptr;
        *launches += 2;
        const dim3 grid(m, a.steps);
        float *norms = c.loop_ws + (int64_t)a.steps * m * n_r * a.classes;
        cudaError_t e = n_r <= 4 ? launch_chained(loop_products_kernel<4>, grid, dim3(kProductWarps * 32), 0, s, chain_launches(c), a.V, ldv, stride_v, a.features, a.in,
                                                  a.classes, (int)c.desc.has_bias, parts, m, n_r, c.loop_ws, norms)
                                 : launch_chained(loop_products_kernel<8>, grid, dim3(kProductWarps * 32), 0, s, chain_launches(c), a.V, ldv, stride_v, a.features, a.in,
                                                  a.classes, (int)c.desc.has_bias, parts, m, n_r, c.loop_ws, norms);
        if (e != cudaSuccess) return e;
        e = launch_clustered(softmax_loop_kernel, kLoopCluster, dim3(kLoopCluster), dim3(kLoopThreads), (size_t)a.p.bytes, s, chain_launches(c), a);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace zeno
