// Candidate-model forward for the softmax-cross-entropy MLP, CUDA-core path: dense layers by columns, and the rule that says
// which of the two kernels for rows of any alignment takes a layer (the other one, by tiles: zeno_mlp.cu).
#include <type_traits>

#include "zeno_internal.h"

namespace zeno {

namespace {

// One dense layer of all models, rows of any alignment, by columns: a warp takes R rows of one model and N samples, a lane
// every 32nd column (W = 4: four columns of every 128, rows aligned to four elements).  The rows' entries of x and v come
// straight from memory into the lane that needs them, the next step's while this one's are multiplied; w = x - gamma v is
// formed there and meets the lane's columns of the N samples, staged in shared memory for the block's eight warps by
// asynchronous copies.  A lane's sums are those of every 32nd product; the lanes' are added at the end.  Where tiles are few
// a cluster of blocks deals the stretches of 256 columns out and meets in the first one's shared memory.
// LONG (a block has more than eight stretches): the lanes' sums are added after every eight, 64 products a lane, and those sums
// to a total, so that rounding errors stay those of short sums however long the row is (root mean square error of a sum of
// 4,095, 40,001 products of random signs: 1.5e-7, 1.8e-7 of it; 2.2e-7, 6.8e-7 in one run; by tiles 1.7e-7, 2.5e-7).  Shorter
// rows do without the code: with it the step of 1029-301-131-11 takes 2 % longer.
// Bound by the loads' latency while few are in flight, then by shared-memory reads and additions.  A whole scoring pass by
// columns and by tiles (zeno_mlp.cu): 65 models of 2500 x 2000, one sample, binary32 0.51 of the time, bfloat16 0.39; of
// 1345 x 1000 and 11 samples 0.87 and 0.54; of 1029 x 301 x 131 and 62 samples 0.94 and 0.64.
constexpr int kRowsAhead = 4;
constexpr int kRowsWarps = 8, kRowsThreads = kRowsWarps * 32, kRowsCols = 256;
__host__ __device__ constexpr int rows_red_floats(int R, int N) { return kRowsWarps * R * N; }
__host__ __device__ constexpr int rows_own_floats(int R, int N) {
    return 2 * N * kRowsCols > rows_red_floats(R, N) ? 2 * N * kRowsCols : rows_red_floats(R, N);
}
constexpr int kRowsRun = 8;                      // stretches of a run
inline size_t rows_smem(int R, int N, int cluster, bool async, bool runs) {
    return sizeof(float) * ((size_t)rows_own_floats(R, N) + (runs ? rows_red_floats(R, N) : 0) + (cluster > 1 ? (size_t)cluster * (rows_red_floats(R, N) + kRowsWarps) : 0) +
                            (async ? (size_t)kRowsWarps * kRowsAhead * 2 * R * 32 : 0));
}
template <typename T, int W> struct RowsRaw { using Type = typename RawOf<T>::One; };
template <typename T> struct RowsRaw<T, 4> { using Type = typename RawOf<T>::Four; };
template <typename Raw> __device__ __forceinline__ void raw_unpack(Raw v, float (&o)[1]) { o[0] = raw_to_float(v); }
template <typename Raw> __device__ __forceinline__ void raw_unpack(Raw v, float (&o)[4]) {
    const float4 f = raw_to_float4(v);
    o[0] = f.x; o[1] = f.y; o[2] = f.z; o[3] = f.w;
}

// ASYNC (binary32, W = 1): every lane's words come by asynchronous copies into words of shared memory that it alone reads,
// kRowsAhead steps ahead, where the sums leave no registers for more than one step's loads.
template <typename T, int R, int N, int W, bool ASYNC, bool LONG>
__global__ void __launch_bounds__(kRowsThreads, 2) mlp_rows_kernel(LayerArgs a, int sample_tiles, int cluster) {
    // steps whose entries of x and v are on their way: two where the registers hold them
    constexpr int U = W == 1 && !ASYNC && (R == 4 ? N <= 16 : N <= 4) ? 2 : 1;
    constexpr int C = kRowsCols, kSteps = C / (32 * W), kRows = kRowsWarps * R, kRed = rows_red_floats(R, N);
    constexpr int kTotals = rows_own_floats(R, N), kOwn = kTotals + (LONG ? kRed : 0), kBatch = R * N < 32 ? R * N : 32;
    static_assert(kRowsThreads % kRows == 0, "a thread finishes one row");
    using Raw = typename RowsRaw<T, W>::Type;
    extern __shared__ __align__(16) float smem_dyn[];
    if (a.first_in_call) pdl_wait();
    if (cluster > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = cluster > 1 ? (int)cluster_rank() : 0;
    const int c = blockIdx.y;                    // model: 0 = x, 1+i = x - gamma v_i
    const int tile = blockIdx.x / cluster, row_tile = tile / sample_tiles, sample_tile = tile - row_tile * sample_tiles;
    const int row0 = row_tile * kRows + warp * R, j0 = sample_tile * N;
    const int K = a.in, nrows = min(max(a.out - row0, 0), R);
    const bool has_v = c > 0;
    const T *xw = static_cast<const T *>(a.x) + a.offW;
    const T *vbase = static_cast<const T *>(a.V) + (has_v ? (int64_t)(c - 1) * a.ldv : 0);
    const T *vw = vbase + a.offW;
    const float *hin = a.Hin + (int64_t)c * a.hin_cand_stride;

    float acc[R][N], nr[R];
    uint32_t off[R];                             // bytes; rows beyond the layer: its last one again, dropped at the end
#pragma unroll
    for (int r = 0; r < R; ++r) {
        nr[r] = 0.f;
        off[r] = (uint32_t)min(row0 + r, a.out - 1) * (uint32_t)K * (uint32_t)sizeof(T);
#pragma unroll
        for (int n = 0; n < N; ++n) acc[r][n] = 0.f;
    }
    float *mine = smem_dyn + kOwn + (cluster > 1 ? cluster * (kRed + kRowsWarps) : 0) + (warp * kRowsAhead * 2 * R) * 32 + lane;
    int slot = 0;                                // ASYNC: of the next step
    Raw xr[U][R], vr[U][R];
    auto load = [&](int u, int k0) {             // columns beyond the row: its last ones again, taken for zero below
        const uint32_t k = (uint32_t)min(k0 + lane * W, K - W) * (uint32_t)sizeof(T);
        if constexpr (ASYNC) {
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(mine + u * 2 * R * 32);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                cp_async<4>(dst + r * 256, reinterpret_cast<const char *>(xw) + (off[r] + k));
                cp_async<4>(dst + r * 256 + 128, reinterpret_cast<const char *>(vw) + (off[r] + k));
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                xr[u][r] = __ldg(reinterpret_cast<const Raw *>(reinterpret_cast<const char *>(xw) + (off[r] + k)));
                vr[u][r] = __ldg(reinterpret_cast<const Raw *>(reinterpret_cast<const char *>(vw) + (off[r] + k)));    // of model 0 a row that is dropped
            }
        }
    };
    auto stage = [&](int chunk, int b) {
        constexpr int kLanes = C / W;            // threads along a sample's stretch
        const int q = tid % kLanes * W, k = chunk * C + q;
        const float *src = hin + (int64_t)(j0 + tid / kLanes) * K + k;
        uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem_dyn + b * N * C + tid / kLanes * C + q);
#pragma unroll 4
        for (int j = tid / kLanes; j < N; j += kRowsThreads / kLanes, src += (int64_t)(kRowsThreads / kLanes) * K, dst += 4 * (kRowsThreads / kLanes) * C) {
            const bool ok = k < K && j0 + j < a.n_r;
            cp_async<4 * W>(dst, ok ? src : hin, ok);
        }
        if (!ASYNC) cp_async_commit();          // else with the next step's words
    };
    const int chunks = (K + C - 1) / C;
    // the step `ahead` steps after step s of this stretch, in the stretches this block takes
    auto column_of = [&](int chunk, int s, int ahead) {
        return s + ahead < kSteps ? chunk * C + (s + ahead) * 32 * W : (chunk + cluster) * C + (s + ahead - kSteps) * 32 * W;
    };
    if (!ASYNC) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (rank * C + u * 32 * W < K) load(u, rank * C + u * 32 * W);
    }
    // the bias entries of the row this thread finishes
    const int frow = tid % kRows, fo = row_tile * kRows + frow;
    float bx = 0.f, bv = 0.f;
    if (rank == 0 && fo < a.out && a.offB >= 0) {
        bx = load_elem(static_cast<const T *>(a.x) + a.offB + fo);
        if (has_v) bv = load_elem(vbase + a.offB + fo);
    }
    if (!a.first_in_call) pdl_wait();
    pdl_launch_dependents();
    if (rank < chunks) stage(rank, 0);
    if (ASYNC) {
        for (int u = 0; u < kRowsAhead; ++u) {
            if (rank * C + u * 32 < K) load(u, rank * C + u * 32);
            cp_async_commit();
        }
    }
    // lane l: the lanes' sums of pair e0 + l of the warp's (row, sample) pairs
    auto batch_sum = [&](int e0) {
        float v[kBatch];
#pragma unroll
        for (int e = 0; e < kBatch; ++e) v[e] = e0 + e < R * N ? acc[(e0 + e) % R][(e0 + e) / R < N ? (e0 + e) / R : 0] : 0.f;
        return warp_transpose_reduce<kBatch>(v, lane);
    };
    float *totals = smem_dyn + kTotals + warp * R * N + lane;        // LONG: of the runs so far, a lane its own
    int b = 0, chunk = rank, runs = 0;
    while (true) {
        const int run_end = LONG ? min(chunks, chunk + kRowsRun * cluster) : chunks;
        for (; chunk < run_end; chunk += cluster, b ^= 1) {
            const bool more = chunk + cluster < chunks;
            cp_async_wait<ASYNC ? kRowsAhead - 1 : 0>();
            __syncthreads();                         // this stretch is here; the other buffer has been read
            if (more) stage(chunk + cluster, b ^ 1);
            const float *hs = smem_dyn + b * N * C + lane * W;
            auto steps = [&](auto tail) {            // tail: some lanes' columns may lie beyond the row
                constexpr bool kTail = decltype(tail)::value;
#pragma unroll 1
                for (int s0 = 0; s0 < kSteps; s0 += U) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int s = s0 + u, k0 = chunk * C + s * 32 * W;
                        if (kTail && k0 >= K) break;
                        float w[R][W];
                        const bool in = !kTail || k0 + lane * W < K;
                        if (ASYNC) cp_async_wait<kRowsAhead - 1>();
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            float x[W], v[W];
                            if constexpr (ASYNC) {
                                x[0] = mine[slot * 2 * R * 32 + r * 64];
                                v[0] = mine[slot * 2 * R * 32 + r * 64 + 32];
                            } else {
                                raw_unpack(xr[u][r], x);
                                raw_unpack(vr[u][r], v);
                            }
#pragma unroll
                            for (int e = 0; e < W; ++e) {
                                if (!has_v || !in) v[e] = 0.f;
                                w[r][e] = candidate_param<T>(in ? x[e] : 0.f, v[e], a.gamma);
                                nr[r] = fmaf(v[e], v[e], nr[r]);
                            }
                        }
                        const int next = column_of(chunk, s, ASYNC ? kRowsAhead : U);
                        if (next < K) load(ASYNC ? slot : u, next);
                        if (ASYNC) {
                            cp_async_commit();
                            if (++slot == kRowsAhead) slot = 0;
                        }
#pragma unroll
                        for (int n = 0; n < N; ++n) {
                            float h[W];
                            if constexpr (W == 4) {
                                const float4 t = *reinterpret_cast<const float4 *>(hs + n * C + s * 32 * W);
                                h[0] = t.x; h[1] = t.y; h[2] = t.z; h[3] = t.w;
                            } else {
                                h[0] = hs[n * C + s * 32];
                            }
#pragma unroll
                            for (int r = 0; r < R; ++r)
#pragma unroll
                                for (int e = 0; e < W; ++e) acc[r][n] = fmaf(w[r][e], h[e], acc[r][n]);
                        }
                    }
                }
            };
            if ((chunk + 1) * C <= K) steps(std::false_type{});
            else steps(std::true_type{});
        }
        if constexpr (!LONG) {
            break;
        } else {
            if (chunk >= chunks) break;
#pragma unroll
            for (int e0 = 0; e0 < R * N; e0 += kBatch) {
                const float z = batch_sum(e0);
                if (lane < kBatch && e0 + lane < R * N) totals[e0] = runs ? totals[e0] + z : z;
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int n = 0; n < N; ++n) acc[r][n] = 0.f;
            ++runs;
        }
    }
    // the lanes' sums as [sample][row] where the samples were staged
    if (ASYNC) cp_async_wait<0>();
    __syncthreads();
    float *red = smem_dyn;
#pragma unroll
    for (int e0 = 0; e0 < R * N; e0 += kBatch) {
        float z = batch_sum(e0);
        const int e = e0 + lane;
        if (LONG && lane < kBatch && e < R * N && runs) z += totals[e0];
        if (lane < kBatch && e < R * N) red[e / R * kRows + warp * R + e % R] = z;
    }
    float nrm = 0.f;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (r < nrows) nrm += nr[r];
    if (tid < kRows) nrm = fmaf(bv, bv, nrm);
    nrm = warp_sum(nrm);
    __syncthreads();
    float *parts = smem_dyn + kOwn;                                  // [cluster][kRed + warps], the first block's is used
    if (cluster > 1) {
        __syncwarp();
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        const uint32_t dst = cluster_addr(parts + rank * (kRed + kRowsWarps), 0);
        for (int t = tid; t < kRed; t += kRowsThreads) cluster_store(dst + 4 * t, red[t]);
        if (lane == 0) cluster_store(dst + 4 * (kRed + warp), nrm);
        cluster_barrier();
        if (rank != 0) return;
        nrm = 0.f;
        for (int r = 0; r < cluster; ++r) nrm += parts[r * (kRed + kRowsWarps) + kRed + warp];
    }
    const float bias = candidate_param<T>(bx, bv, a.gamma);
#pragma unroll
    for (int t = tid; t < kRed; t += kRowsThreads) {
        float z = 0.f;
        if (cluster > 1) {
            for (int r = 0; r < cluster; ++r) z += parts[r * (kRed + kRowsWarps) + t];
        } else {
            z = red[t];
        }
        if (a.offB >= 0) z += bias;
        if (a.relu) z = relu_keep_nan(z);
        const int j = j0 + t / kRows;
        if (fo < a.out && j < a.n_r) a.Hout[((int64_t)c * a.n_r + j) * a.out + fo] = z;
    }
    // partial ||v||^2 of the rows and bias entries; one slot per warp
    if (has_v && sample_tile == 0 && lane == 0)
        a.normpart[(int64_t)(c - 1) * a.np_slots + a.np_base + row_tile * kRowsWarps + warp] = nrm;
}

template <typename T, int R, int N, int W, bool ASYNC, bool LONG>
cudaError_t launch_rows_kernel(Context &c, const LayerArgs &a, int64_t tiles, int sample_tiles, int cluster, cudaStream_t s) {
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(mlp_rows_kernel<T, R, N, W, ASYNC, LONG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)rows_smem(R, N, kMaxCluster, ASYNC, LONG));
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    // the sample tiles of the same rows run side by side and find them in L2
    return launch_clustered(mlp_rows_kernel<T, R, N, W, ASYNC, LONG>, cluster, dim3((unsigned)(tiles * cluster), a.m + 1), dim3(kRowsThreads),
                            rows_smem(R, N, cluster, ASYNC, LONG), s, chain_launches(c), a, sample_tiles, cluster);
}

template <typename T, int R, int N, int W, bool ASYNC = false>
cudaError_t launch_rows_tiles(Context &c, const LayerArgs &a, cudaStream_t s) {
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    const int sample_tiles = (a.n_r + N - 1) / N;
    const int64_t tiles = (int64_t)((a.out + kRowsWarps * R - 1) / (kRowsWarps * R)) * sample_tiles;
    int cluster = 1;
    while (cluster < kMaxCluster && tiles * (a.m + 1) * 2 * cluster <= 2 * sms && a.in > kRowsCols * cluster) cluster *= 2;
    return a.in > kRowsRun * kRowsCols * cluster ? launch_rows_kernel<T, R, N, W, ASYNC, true>(c, a, tiles, sample_tiles, cluster, s)
                                                 : launch_rows_kernel<T, R, N, W, ASYNC, false>(c, a, tiles, sample_tiles, cluster, s);
}

// rows a warp takes: eight of few samples where no alignment asks for the registers, four of narrow layers, whose blocks
// would otherwise have no rows for most of their warps
__host__ __device__ constexpr int rows_of_warp(int out, int n_r, bool aligned) { return !aligned && n_r <= 8 && out > 32 ? 8 : 4; }

// Many samples in tiles of twelve and more, up to as many as the registers hold the sums of: the fewest padded samples, then the fewest tiles.
constexpr int kRowsSamples = 24, kRowsAsyncFrom = 512;       // samples of a tile; columns from which one tile's weights come by copies
int rows_samples(int n_r, int most) {
    int best = most, least = 1 << 30;
    for (int n = most; n >= 12; n -= 4) {
        const int padded = (n_r + n - 1) / n * n;
        if (padded < least) { least = padded; best = n; }
    }
    return best;
}

template <typename T, int W>
cudaError_t launch_rows(Context &c, const LayerArgs &a, cudaStream_t s) {
    if (rows_of_warp(a.out, a.n_r, W == 4) == 8) {
        if (a.n_r <= 1) return launch_rows_tiles<T, 8, 1, 1>(c, a, s);
        if (a.n_r <= 2) return launch_rows_tiles<T, 8, 2, 1>(c, a, s);
        if (a.n_r <= 4) return launch_rows_tiles<T, 8, 4, 1>(c, a, s);
        return launch_rows_tiles<T, 8, 8, 1>(c, a, s);
    }
    if (a.n_r <= 1) return launch_rows_tiles<T, 4, 1, W>(c, a, s);
    if (a.n_r <= 2) return launch_rows_tiles<T, 4, 2, W>(c, a, s);
    if (a.n_r <= 4) return launch_rows_tiles<T, 4, 4, W>(c, a, s);
    if (a.n_r <= 8) return launch_rows_tiles<T, 4, 8, W>(c, a, s);
    constexpr int kMost = W == 1 ? kRowsSamples : is_bf16<T>::value ? 16 : 12;
    const int best = rows_samples(a.n_r, kMost);
    // one tile of 20 or 24 samples and rows long enough to fill the pipeline: 38 models of 1029 x 301 with 19 samples take 44 us
    // with the copies and 50 without, of 301 x 131 16 and 14; with more tiles the copies and the reads of their words are too
    // many for the load units (65 models of 1345 x 1000, 62 samples: 794 us and 650).  40 layers of 17 to 24 samples, 512 to 6000 columns and
    // 5 to 128 candidates: 0.90 of the time without on average, 0.65 to 1.17 (none of them faster by tiles)
    if constexpr (W == 1 && !is_bf16<T>::value) {
        if (a.n_r <= 24 && best >= 20 && a.in >= kRowsAsyncFrom)
            return best == 20 ? launch_rows_tiles<T, 4, 20, 1, true>(c, a, s) : launch_rows_tiles<T, 4, 24, 1, true>(c, a, s);
    }
    if (best == 12) return launch_rows_tiles<T, 4, 12, W>(c, a, s);
    if (best == 16) return launch_rows_tiles<T, 4, kMost < 16 ? 12 : 16, W>(c, a, s);
    if (best == 20) return launch_rows_tiles<T, 4, kMost < 20 ? 12 : 20, W>(c, a, s);
    return launch_rows_tiles<T, 4, kMost < 24 ? 12 : 24, W>(c, a, s);
}

}  // namespace

// Whether a layer of many binary32 samples, rows of any alignment, is small enough for the kernel by columns.  The one by tiles reads its
// samples from shared memory half as often, and does better with more work than fills the device: 12 candidates of 3972 x 930, 94
// samples 518 us by tiles and 807 by columns; 32 of 4082 x 614, 86 893 and 1,282; 42 of 1166 x 33, 89 (1.2 waves of blocks by columns, one
// nearly full one by tiles) 63 and 79.  With less the shorter blocks win: 21 of 3512 x 72, 103 samples 225 and 131; 15 of 2288 x 333, 50
// 154 and 112; tiles of up to twenty samples, whose sums leave registers to load ahead, even of a few waves: 37 of 1049 x 152, 103
// samples 149 and 104, 125 of 829 x 57, 97 124 and 103, but of short rows not (11 of 168 x 1314, 32 27 and 31).  380 layers of 17 to 128 samples:
// 0.87 of the time of the kernel by tiles on average, the worst 1.20; by columns wherever rows are long 1.56.
static bool few_blocks(const Context &c, int in, int out, int n_r, int m) {
    const int places = 2 * (c.sm_count > 0 ? c.sm_count : 148);          // two blocks an SM of either kernel
    // narrow layers: 41 to 48 samples are the same tiles either way (73 candidates of 885 x 26, 47 samples: 28 us and 31)
    if (out <= 32 && n_r <= 48) return n_r <= 40;
    const LayerTiles t = layer_tiles(c, in, out, n_r, m);
    const int samples = rows_samples(n_r, kRowsSamples);
    if (samples <= 20 && in >= 320) return t.tiles * 2 <= 5 * (int64_t)places;
    if (samples <= 16) return t.tiles * 4 <= 3 * (int64_t)places;
    const int64_t blocks = (int64_t)(m + 1) * ((out + 31) / 32) * ((n_r + samples - 1) / samples);
    const int64_t tile_blocks = t.tiles * t.cluster;
    const bool one_full_wave = tile_blocks <= places && tile_blocks * 20 >= (int64_t)places * 17;
    return blocks <= places || (blocks <= 2 * places && !one_full_wave);
}

// Which of the two kernels takes a layer.  By columns: from 128 columns on, or 64 where few samples leave few sums to add up
// over the lanes at the end (the layers of 64 x 48 x 1000 of 64 candidates and 128 samples: 245 us by columns, 113 by
// tiles); of aligned rows, whose four columns a lane leave the registers for fewer samples a tile, many samples only
// where rows are long (300 x 260 in bfloat16 of 64 candidates, 128 samples: 1.15 times as long by columns, 2500 x 2000 of 21
// candidates 0.91); and within 32-bit offsets.
bool layer_by_columns(const Context &c, int in, int out, int n_r, int m, bool aligned) {
    const bool f32 = c.desc.param_dtype == ZENO_F32;
    if (in < (n_r <= 8 ? 64 : 128) || (aligned && n_r > 32 && in < 1024)) return false;
    // 21 to 24 samples, 25 to 32 and more than 40: 24 a tile, of long rows by asynchronous copies; sixteen; whatever pads least
    const bool many = n_r > 40 || (n_r > 24 && n_r <= 32) || (n_r > 20 && n_r <= 24 && in < kRowsAsyncFrom);
    if (f32 && !aligned && many && !few_blocks(c, in, out, n_r, m)) return false;
    return (int64_t)in * out * (f32 ? 4 : 2) < (int64_t)1 << 32;
}

// norm partials of a layer: a slot per warp of every row tile
int mlp_norm_slots(const Context &c, int in, int out, int n_r, int m, bool aligned) {
    const int rows = layer_by_columns(c, in, out, n_r, m, aligned) ? kRowsWarps * rows_of_warp(out, n_r, aligned) : 64;
    return (out + rows - 1) / rows * kRowsWarps;
}
int mlp_norm_slots_most(int out) { return (out + 31) / 32 * kRowsWarps; }

cudaError_t launch_layer_by_columns(Context &c, const LayerArgs &a, bool aligned, cudaStream_t s) {
    if (c.desc.param_dtype == ZENO_BF16)
        return aligned ? launch_rows<__nv_bfloat16, 4>(c, a, s) : launch_rows<__nv_bfloat16, 1>(c, a, s);
    return aligned ? launch_rows<float, 4>(c, a, s) : launch_rows<float, 1>(c, a, s);
}

}  // namespace zeno
