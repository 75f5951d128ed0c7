// The paper's baseline aggregation rules on the same candidate matrix V (Experiments, "Baselines"): Krum_b here,
// the marginal Median in zeno_median.cu.
//
// Krum: the squared distances ||v_i - v_j||^2 of all pairs, taken as sums of squared differences (not
// from a Gram matrix: two honest candidates may differ by far less than their norms), then for every
// candidate the sum over its m - b - 2 nearest neighbours, the arg min of those sums, and a copy of the
// winning row.  The pair sums are accumulated per block over its share of the columns and added up
// afterwards in a fixed order, so the result does not depend on scheduling.
#include <math.h>

#include "zeno_internal.h"

namespace zeno {

namespace {

__device__ __forceinline__ float nan_to_inf(float v) { return v != v ? INFINITY : v; }

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

// dist[i][j] = the blocks' partial sums added in block order (in double), one warp an entry: lanes take
// every 32nd block and their sums meet in a fixed butterfly.  A NaN distance counts as plus infinity.
__global__ void __launch_bounds__(256) krum_reduce_kernel(const float *part, int slabs, int m, float *dist) {
    const int mb = krum_row_blocks(m), tiles = krum_tiles(m);
    const int lane = threadIdx.x & 31;
    const int entry = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (entry >= tiles * 16) return;
    const int tile = entry >> 4, e = entry & 15;
    int ib, jb;
    krum_tile_of(tile, mb, ib, jb);
    const int i = ib * 4 + (e >> 2), j = jb * 4 + (e & 3);
    if (i >= m || j >= m) return;
    double s = 0.0;
    for (int q = lane; q < slabs; q += 32) s += (double)part[(int64_t)q * tiles * 16 + entry];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
        const float v = nan_to_inf((float)s);
        dist[i * m + j] = v;
        if (ib != jb) dist[j * m + i] = v;    // a diagonal tile holds both (i, j) and (j, i) itself
    }
}

// One block.  For every candidate the sum of its m - b - 2 smallest distances to the others (ascending,
// as a sorted sum); the arg min, lowest index first.
__global__ void __launch_bounds__(128) krum_finish_kernel(const float *dist, int m, int b, float *sums_out, int32_t *k_out,
                                                          float *sums_ws) {
    const int nn = m - b - 2;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        unsigned used[ZENO_KRUM_MAX_M / 32];
#pragma unroll
        for (int w = 0; w < ZENO_KRUM_MAX_M / 32; ++w) used[w] = 0u;
        used[i >> 5] |= 1u << (i & 31);
        float s = 0.f;
        for (int t = 0; t < nn; ++t) {
            int best = -1;
            float bv = INFINITY;
            for (int j = 0; j < m; ++j) {
                if (used[j >> 5] & (1u << (j & 31))) continue;
                const float v = dist[i * m + j];
                if (best < 0 || v < bv) { best = j; bv = v; }
            }
            used[best >> 5] |= 1u << (best & 31);
            s += bv;
        }
        sums_ws[i] = s;
        if (sums_out) sums_out[i] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int best = 0;
        for (int i = 1; i < m; ++i)
            if (sums_ws[i] < sums_ws[best]) best = i;
        *k_out = best;
    }
}

template <typename T>
__global__ void __launch_bounds__(256) copy_row_kernel(const T *V, int64_t ldv, int64_t d, int m, const int32_t *k, float *out) {
    const int row = *k;
    if (row < 0 || row >= m) return;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < d; j += (int64_t)gridDim.x * blockDim.x)
        out[j] = load_elem(V + (int64_t)row * ldv + j);
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
    if (tiles < kKrumThreads)
        krum_pairs_kernel<T, 1><<<blocks, kKrumThreads, smem, s>>>(V, ldv, d, m, c.krum_part);
    else
        krum_pairs_kernel<T, 3><<<blocks, kKrumThreads, smem, s>>>(V, ldv, d, m, c.krum_part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    float *dist = c.krum_part + (size_t)c.krum_blocks * krum_tiles(c.m_max) * 16;     // m_max <= ZENO_KRUM_MAX_M here
    krum_reduce_kernel<<<(tiles * 16 + 7) / 8, 256, 0, s>>>(c.krum_part, blocks, m, dist);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    krum_finish_kernel<<<1, 128, 0, s>>>(dist, m, b, sums, k, c.krum_sums);
    e = cudaGetLastError();
    if (e != cudaSuccess || !out) return e;
    int64_t cw = (d + 255) / 256;
    const int cblocks = (int)(cw < (int64_t)sms * 8 ? (cw < 1 ? 1 : cw) : (int64_t)sms * 8);
    copy_row_kernel<T><<<cblocks, 256, 0, s>>>(V, ldv, d, m, k, out);
    return cudaGetLastError();
}

}  // namespace

// floats of Krum's workspace for up to m candidates and `blocks` blocks: the blocks' pair sums, then dist[m][m]
size_t krum_part_floats(int m, int blocks) { return (size_t)blocks * krum_tiles(m) * 16 + (size_t)m * m; }

cudaError_t launch_krum(Context &c, const void *V, int64_t ldv, int m, int b, float *out, int32_t *k, float *sums,
                        cudaStream_t s, int *launches) {
    *launches += out ? 4 : 3;
    profile_mark(c, "krum", s);
    if (c.desc.param_dtype == ZENO_BF16)
        return launch_krum_typed(c, static_cast<const __nv_bfloat16 *>(V), ldv, m, b, out, k, sums, s);
    return launch_krum_typed(c, static_cast<const float *>(V), ldv, m, b, out, k, sums, s);
}

}  // namespace zeno
