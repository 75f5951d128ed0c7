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

// The rows are taken in blocks of B, their number rounded up to even, and a warp holds one tile of pairs in registers: B x B
// pairs of two different blocks, or the 2 x B (B - 1) / 2 pairs inside the blocks 2 w and 2 w + 1.  A lane owns a column: it
// reads 2 B values of a staged tile of columns (neighbouring lanes, neighbouring words) for up to B x B differences and
// multiplications, and keeps its sums to the end.  Every tile's lanes take the same columns in the same order, so identical
// rows get identical distances.  With more tiles than a block has warps, gridDim.y blocks share a stretch of columns, each
// staging the row blocks its tiles name; with fewer, groups of warps split the columns.
// The rows come by asynchronous copies, three stages, 16 bytes at a time where rows are aligned, else 4.
// Bound by issue: of 20 rows a column costs 190 differences and 190 multiplications, 0.74 of the schedulers' slots are taken,
// 0.6 of them by these.  1.8 M columns: 20 rows 48 us (4 x 4 tiles a thread from shared memory: 104), 64 rows 401 (580), 100 rows
// 1,080 (1,280).  Two columns an instruction (packed additions and multiplications, blocks of 5 and 7 rows): 54, 810 and 2,240
// us; the packed instructions take the arithmetic pipe twice as long each.
constexpr int kKrumThreads = 256, kKrumWarps = kKrumThreads / 32;
constexpr int kKrumStages = 3;
constexpr int kKrumBlocksPerSm = 2;
constexpr int kKrumMaxBlocks = 16;            // row blocks
constexpr int kKrumMaxTiles = kKrumMaxBlocks * kKrumMaxBlocks / 2;
constexpr int kKrumPad = 8;                   // entries between staged rows: rows stay aligned to 16 bytes
// Rows staged by a block: 90 of any plan for up to ZENO_KRUM_MAX_M candidates.  The tables' 9 bytes a row come before the stages, which
// should start at a multiple of 128 bytes (20 candidates of 1.8 M columns: 58.7 us, with tables of 90 rows 60.6).
constexpr int kKrumMaxRows = 128;

struct KrumPlan {
    int B, nb;                                // rows of a block, blocks
    int tiles, ny, per_y;                     // tiles of pairs; blocks that share them; tiles of each
    unsigned used[kKrumMaxTiles / kKrumWarps];                 // row blocks a block of blocks y reads
    unsigned char ia[kKrumMaxTiles], ib[kKrumMaxTiles];        // a tile's blocks; diag: the pairs inside them
    unsigned char diag[kKrumMaxTiles];
    unsigned char at[kKrumMaxBlocks][kKrumMaxBlocks];          // the tile of two blocks
};

// columns staged at a time: as many as leave room for two blocks an SM (three stages of 28, 70 and 90 binary32 rows).
// bfloat16 rows always have room for 128 columns, the plans of blocks of three and five rows for 256
inline int krum_cols(int rows, int entry_bytes) { return rows * entry_bytes <= 28 * 4 ? 256 : rows * entry_bytes <= 70 * 4 ? 128 : 64; }

__device__ __forceinline__ float krum_value(const float *p) { return *p; }
__device__ __forceinline__ float krum_value(const __nv_bfloat16 *p) {
    return bf16_bits_to_float(*reinterpret_cast<const unsigned short *>(p));
}

// part[block][tile][B * B]: sums of squared differences of a tile's pairs over the columns this block took.
template <typename T, int B, int C, bool WIDE>
__global__ void __launch_bounds__(kKrumThreads, kKrumBlocksPerSm)
krum_pairs_kernel(const T *V, int64_t ldv, int64_t d, int m, const __grid_constant__ KrumPlan plan, float *part) {
    constexpr int kPitch = C + kKrumPad, kPairs = B * (B - 1) / 2;
    constexpr int E = (WIDE ? 16 : 4) / (int)sizeof(T), kChunks = C / E;          // entries of a copy, copies of a row
    constexpr bool kHalves = !WIDE && sizeof(T) == 2;             // rows may start in the second half of 4 bytes
    extern __shared__ __align__(16) uint8_t krum_smem[];
    __shared__ const T *row_at[kKrumMaxRows];                     // where a staged row's copies start, or NULL
    __shared__ unsigned char late[kKrumMaxRows];                  // entries of them before the row's first
    T *stage0 = reinterpret_cast<T *>(krum_smem);
    pdl_wait();
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned used = plan.used[blockIdx.y];
    const int rows = __popc(used) * B, stage = rows * kPitch;
    // this warp's tile and its share of the columns
    const int groups = plan.per_y <= kKrumWarps / 2 ? kKrumWarps / plan.per_y : 1;
    const int group = warp / plan.per_y, mine = warp - group * plan.per_y, tile = blockIdx.y * plan.per_y + mine;
    const bool busy = group < groups && tile < plan.tiles;
    const int ia = busy ? plan.ia[tile] : 0, ib = busy ? plan.ib[tile] : 0;
    const bool diag = busy && plan.diag[tile];
    const bool odd_base = kHalves && (reinterpret_cast<uintptr_t>(V) & 2), odd_pitch = kHalves && (ldv & 1);
    auto half = [&](int row) { return (int)(odd_base != (odd_pitch && (row & 1))); };

    for (int r = threadIdx.x; r < rows; r += kKrumThreads) {
        unsigned left = used;
        for (int skip = r / B; skip > 0; --skip) left &= left - 1;
        const int row = (__ffs(left) - 1) * B + r % B;
        row_at[r] = row < m ? V + (int64_t)row * ldv - half(row) : nullptr;
        late[r] = (unsigned char)half(row);
    }
    __syncthreads();
    for (int r = warp; r < rows; r += kKrumWarps)                 // rows beyond m are and stay zero
        if (!row_at[r])
            for (int s = 0; s < kKrumStages; ++s)
                for (int c = lane; c < kPitch; c += 32) stage0[s * stage + r * kPitch + c] = T(0.f);
    const int64_t tiles_c = (d + C - 1) / C;
    auto load = [&](int64_t ct, int s) {
        const int64_t j0 = ct * C;
        const bool last = j0 + C > d;
        const int q = threadIdx.x % kChunks * E, r0 = threadIdx.x / kChunks;      // kChunks divides the threads
        uint32_t dst = (uint32_t)__cvta_generic_to_shared(stage0 + s * stage + r0 * kPitch + q);
        for (int r = r0; r < rows; r += kKrumThreads / kChunks, dst += kKrumThreads / kChunks * kPitch * (int)sizeof(T)) {
            const T *row = row_at[r];
            if (!row) continue;
            const bool ok = !last || j0 + q - (kHalves ? late[r] : 0) < d;         // beyond the columns nothing is read
            cp_async<WIDE ? 16 : 4>(dst, ok ? row + j0 + q : row, ok);
        }
        if (kHalves && (int)threadIdx.x < rows && late[threadIdx.x]) {             // the last entry of rows that start half a word late
            const T *row = row_at[threadIdx.x];
            const bool ok = j0 + C - 1 < d;
            if (row) cp_async<4>((uint32_t)__cvta_generic_to_shared(stage0 + s * stage + threadIdx.x * kPitch + C), ok ? row + j0 + C : row, ok);
        }
    };
    float acc[B * B];
#pragma unroll
    for (int e = 0; e < B * B; ++e) acc[e] = 0.f;
    // the tile's two blocks of rows within a stage; of bfloat16 rows with an odd pitch every other one starts an entry later
    const int sa = __popc(used & ((1u << ia) - 1)) * B, sb = __popc(used & ((1u << ib) - 1)) * B;
    const int a_even = sa * kPitch + half(ia * B), a_odd = sa * kPitch + half(ia * B + 1);
    const int b_even = sb * kPitch + half(ib * B), b_odd = sb * kPitch + half(ib * B + 1);

    int64_t ct = blockIdx.x;
    for (int s = 0; s < kKrumStages - 1; ++s) {
        if (ct + (int64_t)s * gridDim.x < tiles_c) load(ct + (int64_t)s * gridDim.x, s);
        cp_async_commit();
    }
    int s = 0;
    for (; ct < tiles_c; ct += gridDim.x) {
        cp_async_wait<kKrumStages - 2>();
        __syncthreads();                      // the stage has landed for every thread; the one before is free
        const int64_t next = ct + (int64_t)(kKrumStages - 1) * gridDim.x;
        if (next < tiles_c) load(next, s == 0 ? kKrumStages - 1 : s - 1);
        cp_async_commit();
        T *st = stage0 + s * stage;
        if (ct * C + C > d) {                 // beyond the columns whatever the copies brought counts as zero
            const int left = (int)(d - ct * C);
            for (int r = warp; r < rows; r += kKrumWarps)
                for (int c = left + late[r] + lane; c < kPitch; c += 32) st[r * kPitch + c] = T(0.f);
            __syncthreads();
        }
        if (busy) {
#pragma unroll 1
            for (int c = group * 32 + lane; c < C; c += groups * 32) {
                auto value = [&](int even, int odd, int r) { return krum_value(st + (kHalves && (r & 1) ? odd : even) + r * kPitch + c); };
                float a[B];
#pragma unroll
                for (int r = 0; r < B; ++r) a[r] = value(a_even, a_odd, r);
                if (!diag) {
#pragma unroll
                    for (int q = 0; q < B; ++q) {
                        const float b = value(b_even, b_odd, q);
#pragma unroll
                        for (int r = 0; r < B; ++r) {
                            const float df = a[r] - b;
                            acc[q * B + r] = fmaf(df, df, acc[q * B + r]);
                        }
                    }
                } else {
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        if (t == 1) {
#pragma unroll
                            for (int r = 0; r < B; ++r) a[r] = value(b_even, b_odd, r);
                        }
#pragma unroll
                        for (int q = 1; q < B; ++q)
#pragma unroll
                            for (int r = 0; r < q; ++r) {
                                const float df = a[r] - a[q];
                                float &sum = acc[t * kPairs + q * (q - 1) / 2 + r];
                                sum = fmaf(df, df, sum);
                            }
                    }
                }
            }
        }
        if (++s == kKrumStages) s = 0;
    }
    // the lanes' sums, 32 pairs at a time (lane l receives pair l of the batch), then the groups'
    cp_async_wait<0>();
    __syncthreads();
    float *red = reinterpret_cast<float *>(krum_smem);             // [group][tile of the block][B * B]
    if (busy) {
#pragma unroll
        for (int e0 = 0; e0 < B * B; e0 += 32) {
            float v[32];
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = e0 + e < B * B ? acc[e0 + e < B * B ? e0 + e : 0] : 0.f;
            const float sum = warp_transpose_reduce<32>(v, lane);
            if (e0 + lane < B * B) red[warp * B * B + e0 + lane] = sum;
        }
    }
    __syncthreads();
    const int here = min(plan.per_y, plan.tiles - (int)blockIdx.y * plan.per_y) * B * B;
    float *dst = part + ((int64_t)blockIdx.x * plan.tiles + blockIdx.y * plan.per_y) * (B * B);
    for (int t = threadIdx.x; t < here; t += kKrumThreads) {
        float sum = 0.f;
        for (int g = 0; g < groups; ++g) sum += red[g * plan.per_y * B * B + t];
        dst[t] = sum;
    }
}

// The pairs of fewer columns, or of rows that only copies of 4 bytes bring: 4 x 4 pairs a thread, columns staged by loads of one
// entry, which need no alignment.  Bound by its reads of shared memory, eight for sixteen pairs, and by the loads, which nothing
// overlaps; but a block of little code that starts and ends quickly, and one for a stretch of 128 columns.
constexpr int kSquareCols = 128;              // columns staged per tile
constexpr int kSquarePitch = kSquareCols + 1; // row pitch in floats: rows of a tile start in different banks

__host__ __device__ inline int square_row_blocks(int m) { return (m + 3) / 4; }
__host__ __device__ inline int square_tiles(int m) { const int mb = square_row_blocks(m); return mb * (mb + 1) / 2; }
// groups of threads that share the pair tiles and split a tile's columns between them
__host__ __device__ inline int square_groups(int m) { const int t = square_tiles(m); return t >= kKrumThreads ? 1 : kKrumThreads / t; }
// shared memory of the kernel: the staged rows, or the groups' sums when those need more
inline size_t squares_smem(int m) {
    const size_t rows = (size_t)square_row_blocks(m) * 4 * kSquarePitch, red = (size_t)square_groups(m) * square_tiles(m) * 16;
    return (rows > red ? rows : red) * sizeof(float);
}

// tile index -> (ib, jb) with ib <= jb, row by row of the upper triangle of blocks of four rows
__device__ __forceinline__ void square_tile_of(int tile, int mb, int &ib, int &jb) {
    ib = 0;
    int left = tile;
    while (left >= mb - ib) { left -= mb - ib; ++ib; }
    jb = ib + left;
}

// part[block][tile][4][4]: sums of squared differences of the 4 x 4 pairs (i, j) of a tile over the
// columns this block took.  With fewer tiles than threads, groups of threads split a staged tile's
// columns and their sums are added in group order before they are written.
// kMaxMine: pair tiles a thread may hold (1 while the tiles are fewer than the threads, else 2).
template <typename T, int kMaxMine>
__global__ void __launch_bounds__(kKrumThreads, kMaxMine == 1 ? 4 : 3) krum_squares_kernel(const T *V, int64_t ldv, int64_t d, int m, float *part) {
    extern __shared__ float rows[];           // [m rounded up to 4][kSquarePitch], then [groups][tiles][16]
    pdl_wait();
    pdl_launch_dependents();
    const int mb = square_row_blocks(m), tiles = square_tiles(m), groups = square_groups(m);
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
    for (int64_t j0 = (int64_t)blockIdx.x * kSquareCols; j0 < d; j0 += (int64_t)gridDim.x * kSquareCols) {
        __syncthreads();
#pragma unroll 8
        for (int t = tid; t < m4 * kSquareCols; t += kKrumThreads) {
            const int r = t / kSquareCols, c = t - r * kSquareCols;
            rows[r * kSquarePitch + c] = (r < m && j0 + c < d) ? load_elem(V + (int64_t)r * ldv + j0 + c) : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kMaxMine; ++q) {
            if (q >= n_mine) break;
            const int tile = shared_tiles ? tid - group * tiles : tid + q * kKrumThreads;
            int ib, jb;
            square_tile_of(tile, mb, ib, jb);
            const float *ri = rows + ib * 4 * kSquarePitch, *rj = rows + jb * 4 * kSquarePitch;
            const int c0 = shared_tiles ? group : 0, cs = shared_tiles ? groups : 1;
#pragma unroll(kMaxMine == 1 ? 4 : 1)
            for (int c = c0; c < kSquareCols; c += cs) {
                float a[4], b[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    a[u] = ri[u * kSquarePitch + c];
                    b[u] = rj[u * kSquarePitch + c];
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
template <bool SQUARES>
__global__ void __launch_bounds__(kSumsWarps * 32) krum_sums_kernel(const float *part, int slabs, int m, int b,
                                                                    const __grid_constant__ KrumPlan plan, float *sums_out, float *sums_ws) {
    __shared__ float dist[ZENO_KRUM_MAX_M];
    __shared__ double warp_part[kSumsWarps];
    pdl_wait();
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x, B = SQUARES ? 4 : plan.B;
    const int tiles = SQUARES ? square_tiles(m) : plan.tiles;
    const int64_t slab = (int64_t)tiles * B * B;
    for (int j = warp; j < m; j += kSumsWarps) {
        const int lo = min(i, j), hi = max(i, j), ia = lo / B, ib = hi / B, r = lo - ia * B, q = hi - ib * B;
        int tile, e;
        if (SQUARES) {
            const int mb = square_row_blocks(m);
            tile = ia * mb - ia * (ia - 1) / 2 + (ib - ia);
            e = r * B + q;
        } else {
            tile = plan.at[ia][ib];
            e = ia != ib ? q * B + r : (ia & 1) * (B * (B - 1) / 2) + q * (q - 1) / 2 + r;
        }
        const float *src = part + (int64_t)tile * B * B + (i == j ? 0 : e);
        double s = 0.0;
#pragma unroll(SQUARES ? 8 : 4)
        for (int q = lane; q < slabs; q += 32) s += (double)__ldcg(src + q * slab);
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

int krum_grid_x(const KrumPlan &p, int sms) {
    const int x = kKrumBlocksPerSm * sms / p.ny;
    return x < 1 ? 1 : x;
}

// Rows in blocks of B: the B that pads m to an even number of blocks with the fewest rows, the largest of those that tie.
void krum_size(int m, KrumPlan *plan) {
    KrumPlan &p = *plan;
    int best = 1 << 30;
    for (int B : {3, 5, 7, 8, 10}) {
        const int nb = (m + 2 * B - 1) / (2 * B) * 2;
        if (nb > kKrumMaxBlocks || nb * B > best || (nb > 2 && B < 7)) continue;
        best = nb * B;
        p.B = B;
        p.nb = nb;
    }
    p.tiles = p.nb * p.nb / 2;
    p.ny = (p.tiles + kKrumWarps - 1) / kKrumWarps;
    p.per_y = (p.tiles + p.ny - 1) / p.ny;
}

KrumPlan krum_plan(int m) {
    KrumPlan p = {};
    krum_size(m, &p);
    // neighbouring tiles share row blocks: two of the one against four of the other
    int n = 0;
    for (int i0 = 0; i0 < p.nb; i0 += 2)
        for (int j0 = 0; j0 < p.nb; j0 += 4)
            for (int i = i0; i < i0 + 2 && i < p.nb; ++i)
                for (int j = j0; j < j0 + 4 && j < p.nb; ++j) {
                    if (i >= j) continue;
                    const bool diag = j == i + 1 && (i & 1) == 0;              // these two blocks have a tile of either kind
                    for (int k = 0; k < (diag ? 2 : 1); ++k) {
                        p.ia[n] = (unsigned char)i;
                        p.ib[n] = (unsigned char)j;
                        p.diag[n] = (unsigned char)k;
                        if (k) p.at[i][i] = p.at[j][j] = (unsigned char)n;
                        else p.at[i][j] = (unsigned char)n;
                        p.used[n / p.per_y] |= 1u << i | 1u << j;
                        ++n;
                    }
                }
    return p;
}

template <typename T, int B, int C, bool WIDE>
cudaError_t launch_pairs_cols(Context &c, const KrumPlan &p, int rows, const T *V, int64_t ldv, int m, cudaStream_t s, int *blocks) {
    auto smem = [](int r) {
        const size_t stages = (size_t)kKrumStages * r * (C + kKrumPad) * sizeof(T), red = sizeof(float) * kKrumWarps * B * B;
        return red > stages ? red : stages;
    };
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(krum_pairs_kernel<T, B, C, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem(C == 256 ? 28 * 4 / (int)sizeof(T) : C == 128 ? 70 * 4 / (int)sizeof(T) : kKrumMaxRows));
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    const int64_t want = (c.d + C - 1) / C;
    *blocks = krum_grid_x(p, c.sm_count > 0 ? c.sm_count : 148);
    if (want < *blocks) *blocks = (int)want;
    return launch_chained(krum_pairs_kernel<T, B, C, WIDE>, dim3(*blocks, p.ny), dim3(kKrumThreads), smem(rows), s, chain_launches(c), V, ldv,
                          c.d, m, p, c.krum_part);
}

template <typename T, int B, bool WIDE>
cudaError_t launch_pairs(Context &c, const KrumPlan &p, const T *V, int64_t ldv, int m, cudaStream_t s, int *blocks) {
    int rows = 0;
    for (int y = 0; y < p.ny; ++y) {
        int n = 0;
        for (unsigned u = p.used[y]; u; u &= u - 1) n += B;
        if (n > rows) rows = n;
    }
    const int cols = krum_cols(rows, sizeof(T));
    if constexpr (B >= 7) {
        if constexpr (B >= 8 && sizeof(T) == 4) {
            if (cols == 64) return launch_pairs_cols<T, B, 64, WIDE>(c, p, rows, V, ldv, m, s, blocks);
        }
        if (cols != 256) return launch_pairs_cols<T, B, 128, WIDE>(c, p, rows, V, ldv, m, s, blocks);
    }
    return launch_pairs_cols<T, B, 256, WIDE>(c, p, rows, V, ldv, m, s, blocks);
}

template <typename T, bool WIDE>
cudaError_t launch_pairs_of(Context &c, const KrumPlan &p, const T *V, int64_t ldv, int m, cudaStream_t s, int *blocks) {
    switch (p.B) {
        case 3: return launch_pairs<T, 3, WIDE>(c, p, V, ldv, m, s, blocks);
        case 5: return launch_pairs<T, 5, WIDE>(c, p, V, ldv, m, s, blocks);
        case 7: return launch_pairs<T, 7, WIDE>(c, p, V, ldv, m, s, blocks);
        case 8: return launch_pairs<T, 8, WIDE>(c, p, V, ldv, m, s, blocks);
        default: return launch_pairs<T, 10, WIDE>(c, p, V, ldv, m, s, blocks);
    }
}

// blocks of 4 x 4 pairs that are resident at once
int square_places(int m, int sms) {
    const int per_sm = (int)((200u << 10) / squares_smem(m));
    return (per_sm > 4 ? 4 : per_sm) * sms;   // four: what the registers let be resident
}

// Which of the two kernels takes the pairs.  Few columns are over sooner in little code than register tiles are filled and emptied.
// All three launches, 4 x 4 and register tiles, us: 20 candidates of 6,000 binary32 columns 8.7 and 10.0, of 400 k 42 and 23; 34 of 8,000, bfloat16
// rows of odd pitch 12.6 and 17.3; 12 of 1,074, bfloat16 7.1 and 8.4; up to six candidates fill register tiles of three rows as quickly.
// With 49 to 88 candidates that holds for as many columns as give every SM a block of 4 x 4 pairs, not for fewer, which either kernel leaves SMs
// without: 60 of 10,128 columns, rows not aligned 16.4 and 20.8, 67 of 11,828 21.2 and 26.1, of 2,616 18.3 and 15.5, 79 of 7,026 20.9 and 24.4, of
// 1,980 19.1 and 15.5; 61 to 64 are eight blocks of eight rows without a row too many (of 9,890 20.1 and 19.7, of 234 16.4 and 13.0).
// Many columns of more than 56 candidates, rows not aligned, where most threads have a tile: a block of the
// register tiles stages many rows there by copies of 4 bytes, up to nine times over (88 of 300 k: 187 us and 262, bfloat16 183 and
// 265; 112: 344 and 428, of 30 k 84 and 59; 102 of 111,840 133 and 167, 59 of 242,606
// in bfloat16 97 and 118; but 83 of 133,650 129 and 109, 80 of 223,762 142 and 130).  With few of the last round's threads busy, as at 92, it is the other way.
bool krum_by_squares(int m, int64_t d, int sms, int entry_bytes, bool wide) {
    if (m <= 6) return false;
    int more = 0, most = 0;                   // columns for every SM
    if (wide) {
        if (m <= 12) most = 16;
        else if (m <= (entry_bytes == 4 ? 48 : 42)) most = 96;
        else if (entry_bytes == 4 && m <= 60) { more = 44; most = 100; }
    } else {
        if (m <= 12) most = m <= 10 ? 48 : 80;
        else if (m <= 48) most = 128;
        else if (m <= 56) { more = 32; most = 88; }
        else if (m <= 60) most = 112;
        else if (m >= 65 && m <= 72) { more = 36; most = 84; }
        else if (m >= 73 && m <= 88) { more = 40; most = 64; }
    }
    if (d > (int64_t)more * sms && d <= (int64_t)most * sms) return true;
    const int rounds = (square_tiles(m) + kKrumThreads - 1) / kKrumThreads;
    const int64_t pairs = (int64_t)m * (m - 1) / 2, places = (int64_t)rounds * kKrumThreads * 16;
    const bool busy = rounds <= 2 && square_groups(m) * pairs * 100 >= places * 57;
    const int many = m > 96 && m <= 108 ? 640 : m >= 73 && m <= 80 ? 2048 : 1024;
    return !wide && m > 56 && busy && d > (int64_t)many * sms;
}
int square_blocks(int m, int64_t d, int sms) {
    const int64_t want = (d + kSquareCols - 1) / kSquareCols, most = square_places(m, sms);
    return (int)(want < most ? want : most);
}

template <typename T>
cudaError_t launch_squares(Context &c, const T *V, int64_t ldv, int m, cudaStream_t s, int *blocks) {
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(krum_squares_kernel<T, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)squares_smem(ZENO_KRUM_MAX_M));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(krum_squares_kernel<T, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)squares_smem(ZENO_KRUM_MAX_M));
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    *blocks = square_blocks(m, c.d, c.sm_count > 0 ? c.sm_count : 148);
    return launch_chained(square_tiles(m) < kKrumThreads ? krum_squares_kernel<T, 1> : krum_squares_kernel<T, 2>, dim3(*blocks), dim3(kKrumThreads),
                          squares_smem(m), s, chain_launches(c), V, ldv, c.d, m, c.krum_part);
}

template <typename T>
cudaError_t launch_krum_typed(Context &c, const T *V, int64_t ldv, int m, int b, float *out, int32_t *k, float *sums,
                              cudaStream_t s) {
    const int64_t d = c.d;
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    const KrumPlan p = krum_plan(m);
    int blocks = 0;
    const bool wide = reinterpret_cast<uintptr_t>(V) % 16 == 0 && (ldv * (int64_t)sizeof(T)) % 16 == 0;
    cudaError_t e;
    const bool squares = krum_by_squares(m, d, sms, (int)sizeof(T), wide);
    if (squares) e = launch_squares(c, V, ldv, m, s, &blocks);
    else e = wide ? launch_pairs_of<T, true>(c, p, V, ldv, m, s, &blocks) : launch_pairs_of<T, false>(c, p, V, ldv, m, s, &blocks);
    if (e != cudaSuccess) return e;
    e = launch_chained(squares ? krum_sums_kernel<true> : krum_sums_kernel<false>, dim3(m), dim3(kSumsWarps * 32), 0, s, chain_launches(c),
                       (const float *)c.krum_part, blocks, m, b, p, sums, c.krum_sums);
    if (e != cudaSuccess) return e;
    const int64_t cw = (d + 255) / 256;
    const int cblocks = !out ? 1 : (int)(cw < (int64_t)sms * 8 ? (cw < 1 ? 1 : cw) : (int64_t)sms * 8);
    return launch_chained(copy_row_kernel<T>, dim3(cblocks), dim3(256), 0, s, chain_launches(c), V, ldv, d, m,
                          (const float *)c.krum_sums, k, out);
}

}  // namespace

// floats of Krum's workspace for up to m_max candidates of d columns: the blocks' sums of every tile's pairs
size_t krum_part_floats(int m_max, int64_t d, int sms) {
    size_t most = 0;
    KrumPlan p;
    for (int m = 1; m <= m_max; ++m) {
        krum_size(m, &p);
        const size_t need = (size_t)krum_grid_x(p, sms) * p.tiles * p.B * p.B;
        if (need > most) most = need;
        if (krum_by_squares(m, d, sms, 4, false) || krum_by_squares(m, d, sms, 4, true)) {      // and with them the calls of bfloat16
            const size_t squares = (size_t)square_blocks(m, d, sms) * square_tiles(m) * 16;
            if (squares > most) most = squares;
        }
    }
    return most;
}

cudaError_t launch_krum(Context &c, const void *V, int64_t ldv, int m, int b, float *out, int32_t *k, float *sums,
                        cudaStream_t s, int *launches) {
    *launches += 3;
    profile_mark(c, "krum", s);
    if (c.desc.param_dtype == ZENO_BF16)
        return launch_krum_typed(c, static_cast<const __nv_bfloat16 *>(V), ldv, m, b, out, k, sums, s);
    return launch_krum_typed(c, static_cast<const float *>(V), ldv, m, b, out, k, sums, s);
}

}  // namespace zeno
