// The paper's baseline aggregation rules on the same candidate matrix V (Experiments, "Baselines"): Krum_b here,
// the marginal Median in zeno_median.cu.
//
// Krum: the squared distances ||v_i - v_j||^2 of all pairs, taken as sums of squared differences (not
// from a Gram matrix: two honest candidates may differ by far less than their norms), then for every
// candidate the sum over its m - b - 2 nearest neighbours, the arg min of those sums, and a copy of the
// winning row.  The pair sums are accumulated per block over its share of the columns and added up
// afterwards in a fixed order, so the result does not depend on scheduling.  Three launches: the pairs; a block per
// candidate that adds its distances up and sums the nearest; the copy, whose blocks find the arg min themselves.
#include <math.h>

#include "zeno_internal.h"

namespace zeno {

namespace {

// ---- Krum -----------------------------------------------------------------------------------

constexpr int kKrumThreads = 256;
constexpr int kKrumCols = 128;                // columns staged per tile
constexpr int kKrumPitch = kKrumCols + 1;     // row pitch in floats: rows of a tile start in different banks

__host__ __device__ inline int krum_row_blocks(int m) { return (m + 3) / 4; }
__host__ __device__ inline int krum_tiles(int m) { const int mb = krum_row_blocks(m); return mb * (mb + 1) / 2; }
// groups of threads that share the pair tiles and split a tile's columns between them
__host__ __device__ inline int krum_groups(int m) { const int t = krum_tiles(m); return t >= kKrumThreads ? 1 : kKrumThreads / t; }
// shared memory of the pair kernel: the staged rows, or the groups' sums when those need more
inline size_t krum_pairs_smem(int m) {
    const size_t rows = (size_t)krum_row_blocks(m) * 4 * kKrumPitch, red = (size_t)krum_groups(m) * krum_tiles(m) * 16;
    return (rows > red ? rows : red) * sizeof(float);
}

// tile index -> (ib, jb) with ib <= jb, row by row of the upper triangle of blocks of four rows
__device__ __forceinline__ void krum_tile_of(int tile, int mb, int &ib, int &jb) {
    ib = 0;
    int left = tile;
    while (left >= mb - ib) { left -= mb - ib; ++ib; }
    jb = ib + left;
}

// part[block][tile][4][4]: sums of squared differences of the 4 x 4 pairs (i, j) of a tile over the
// columns this block took.  With fewer tiles than threads, groups of threads split a staged tile's
// columns and their sums are added in group order before they are written.
// kMaxMine: pair tiles a thread may hold (1 while the tiles are fewer than the threads; 528 tiles at m = 128
// over 256 threads need 3).
template <typename T, int kMaxMine>
__global__ void __launch_bounds__(kKrumThreads, kMaxMine == 1 ? 4 : 3) krum_pairs_kernel(const T *V, int64_t ldv, int64_t d, int m, float *part) {
    extern __shared__ float rows[];           // [m rounded up to 4][kKrumPitch], then [groups][tiles][16]
    pdl_wait();
    pdl_launch_dependents();
    const int mb = krum_row_blocks(m), tiles = krum_tiles(m), groups = krum_groups(m);
    const int m4 = mb * 4;
    const int tid = threadIdx.x;
    const bool shared_tiles = tiles < kKrumThreads;                 // one tile a thread, groups of threads
    const int group = tid / tiles < groups ? tid / tiles : -1;      // threads beyond groups * tiles idle
    const int n_mine = shared_tiles ? (group >= 0 ? 1 : 0) : (tiles - tid + kKrumThreads - 1) / kKrumThreads;
    float acc[kMaxMine][16];
#pragma unroll
    for (int q = 0; q < kMaxMine; ++q)
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[q][e] = 0.f;
    for (int64_t j0 = (int64_t)blockIdx.x * kKrumCols; j0 < d; j0 += (int64_t)gridDim.x * kKrumCols) {
        __syncthreads();
#pragma unroll 8
        for (int t = tid; t < m4 * kKrumCols; t += kKrumThreads) {
            const int r = t / kKrumCols, c = t - r * kKrumCols;
            rows[r * kKrumPitch + c] = (r < m && j0 + c < d) ? load_elem(V + (int64_t)r * ldv + j0 + c) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kMaxMine; ++q) {
            if (q >= n_mine) break;
            const int tile = shared_tiles ? tid - group * tiles : tid + q * kKrumThreads;
            int ib, jb;
            krum_tile_of(tile, mb, ib, jb);
            const float *ri = rows + ib * 4 * kKrumPitch, *rj = rows + jb * 4 * kKrumPitch;
            const int c0 = shared_tiles ? group : 0, cs = shared_tiles ? groups : 1;
#pragma unroll(kMaxMine == 1 ? 4 : 1)
            for (int c = c0; c < kKrumCols; c += cs) {
                float a[4], b[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    a[u] = ri[u * kKrumPitch + c];
                    b[u] = rj[u * kKrumPitch + c];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int w = 0; w < 4; ++w) {
                        const float df = a[u] - b[w];
                        acc[q][u * 4 + w] = fmaf(df, df, acc[q][u * 4 + w]);
                    }
            }
        }
    }
    float *dst = part + (int64_t)blockIdx.x * tiles * 16;
    if (!shared_tiles) {
#pragma unroll
        for (int q = 0; q < kMaxMine; ++q) {
            if (q >= n_mine) break;
            float *o = dst + (tid + q * kKrumThreads) * 16;
#pragma unroll
            for (int e = 0; e < 16; e += 4) *reinterpret_cast<float4 *>(o + e) = make_float4(acc[q][e], acc[q][e + 1], acc[q][e + 2], acc[q][e + 3]);
        }
        return;
    }
    __syncthreads();                          // the staged rows are done with: the groups' sums take their place
    if (group >= 0) {
#pragma unroll
        for (int e = 0; e < 16; ++e) rows[tid * 16 + e] = acc[0][e];       // tid = group * tiles + tile
    }
    __syncthreads();
    for (int t = tid; t < tiles * 16; t += kKrumThreads) {
        float sum = 0.f;
        for (int g = 0; g < groups; ++g) sum += rows[g * tiles * 16 + t];
        dst[t] = sum;
    }
}

// Candidate i = blockIdx.x: its distances to the others, the blocks' partial sums added in a fixed order (a warp an entry:
// lanes take every 32nd block and their sums meet in a butterfly, in double; a NaN distance counts as plus infinity),
// then the sum of the m - b - 2 smallest: a distance belongs to it if fewer than that many others are smaller, or equal
// and of a lower index.
constexpr int kSumsWarps = 32;                // one round of entries up to 32 candidates
__global__ void __launch_bounds__(kSumsWarps * 32) krum_sums_kernel(const float *part, int slabs, int m, int b, float *sums_out, float *sums_ws) {
    __shared__ float dist[ZENO_KRUM_MAX_M];
    __shared__ double warp_part[kSumsWarps];
    pdl_wait();
    pdl_launch_dependents();
    const int mb = krum_row_blocks(m), tiles = krum_tiles(m);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x;
    for (int j = warp; j < m; j += kSumsWarps) {
        const int lo = min(i, j), hi = max(i, j), ib = lo >> 2, jb = hi >> 2;
        const int tile = ib * mb - ib * (ib - 1) / 2 + (jb - ib);
        const float *src = part + tile * 16 + (lo & 3) * 4 + (hi & 3);
        double s = 0.0;
#pragma unroll 8
        for (int q = lane; q < slabs; q += 32) s += (double)__ldcg(src + (int64_t)q * tiles * 16);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) dist[j] = nan_to_inf((float)s);
    }
    __syncthreads();
    const int nn = m - b - 2;
    double mine = 0.0;
    for (int j = threadIdx.x; j < m; j += kSumsWarps * 32) {
        if (j == i) continue;
        const float v = dist[j];
        int rank = 0;
        for (int k = 0; k < m; ++k)
            if (k != i && k != j) rank += dist[k] < v || (dist[k] == v && k < j);
        if (rank < nn) mine += (double)v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0) warp_part[warp] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kSumsWarps; ++w) s += warp_part[w];
        sums_ws[i] = (float)s;
        if (sums_out) sums_out[i] = (float)s;
    }
}

// The arg min of the sums, lowest index first, found by every block for itself, and (out != NULL) the copy of its row.
template <typename T>
__global__ void __launch_bounds__(256) copy_row_kernel(const T *V, int64_t ldv, int64_t d, int m, const float *sums, int32_t *k_out,
                                                       float *out) {
    __shared__ int row_s;
    pdl_wait();
    pdl_launch_dependents();
    if (threadIdx.x < 32) {
        float best = INFINITY;
        int at = ZENO_KRUM_MAX_M;
        for (int i = threadIdx.x; i < m; i += 32) {
            const float v = __ldcg(sums + i);
            if (at == ZENO_KRUM_MAX_M || v < best) { best = v; at = i; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float v = __shfl_xor_sync(0xffffffffu, best, o);
            const int w = __shfl_xor_sync(0xffffffffu, at, o);
            if (w < ZENO_KRUM_MAX_M && (at == ZENO_KRUM_MAX_M || v < best || (v == best && w < at))) { best = v; at = w; }
        }
        if (threadIdx.x == 0) {
            row_s = at;
            if (blockIdx.x == 0) *k_out = at;
        }
    }
    __syncthreads();
    if (!out) return;
    const T *row = V + (int64_t)row_s * ldv;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < d; j += (int64_t)gridDim.x * blockDim.x) out[j] = load_elem(row + j);
}

template <typename T>
cudaError_t launch_krum_typed(Context &c, const T *V, int64_t ldv, int m, int b, float *out, int32_t *k, float *sums,
                              cudaStream_t s) {
    const int64_t d = c.d;
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    const int tiles = krum_tiles(m);
    const size_t smem = krum_pairs_smem(m);
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(krum_pairs_kernel<T, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)krum_pairs_smem(ZENO_KRUM_MAX_M));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(krum_pairs_kernel<T, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)krum_pairs_smem(ZENO_KRUM_MAX_M));
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    // as many blocks as stay resident (shared memory, 2048 threads an SM), within what the partials were sized for
    int per_sm = (int)((200u << 10) / smem);
    per_sm = per_sm > 8 ? 8 : (per_sm < 1 ? 1 : per_sm);
    const int64_t want = (d + kKrumCols - 1) / kKrumCols;
    int blocks = per_sm * sms < c.krum_blocks ? per_sm * sms : c.krum_blocks;
    if (want < blocks) blocks = (int)(want < 1 ? 1 : want);
    cudaError_t e = launch_chained(tiles < kKrumThreads ? krum_pairs_kernel<T, 1> : krum_pairs_kernel<T, 3>, dim3(blocks),
                                   dim3(kKrumThreads), smem, s, chain_launches(c), V, ldv, d, m, c.krum_part);
    if (e != cudaSuccess) return e;
    e = launch_chained(krum_sums_kernel, dim3(m), dim3(kSumsWarps * 32), 0, s, chain_launches(c), (const float *)c.krum_part, blocks, m, b, sums,
                       c.krum_sums);
    if (e != cudaSuccess) return e;
    const int64_t cw = (d + 255) / 256;
    const int cblocks = !out ? 1 : (int)(cw < (int64_t)sms * 8 ? (cw < 1 ? 1 : cw) : (int64_t)sms * 8);
    return launch_chained(copy_row_kernel<T>, dim3(cblocks), dim3(256), 0, s, chain_launches(c), V, ldv, d, m,
                          (const float *)c.krum_sums, k, out);
}

}  // namespace

// floats of Krum's workspace for up to m candidates and `blocks` blocks: the blocks' pair sums
size_t krum_part_floats(int m, int blocks) { return (size_t)blocks * krum_tiles(m) * 16; }

cudaError_t launch_krum(Context &c, const void *V, int64_t ldv, int m, int b, float *out, int32_t *k, float *sums,
                        cudaStream_t s, int *launches) {
    *launches += 3;
    profile_mark(c, "krum", s);
    if (c.desc.param_dtype == ZENO_BF16)
        return launch_krum_typed(c, static_cast<const __nv_bfloat16 *>(V), ldv, m, b, out, k, sums, s);
    return launch_krum_typed(c, static_cast<const float *>(V), ldv, m, b, out, k, sums, s);
}

}  // namespace zeno
