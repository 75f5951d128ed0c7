// Convolutional layers of the candidates' models on the 5th-generation tensor cores: a 3 x 3 layer of all m + 1
// models as one implicit GEMM per model, D[pixel][output plane] = sum over taps and input planes of
// A[pixel + tap][plane] W[plane, tap][output plane].
//
// Layout.  The input of a layer lies as [model][term][group of 4 planes][pixel][4 planes], its values split into
// two terms (a leading part of tf32 precision and the remainder).  Pixels are numbered in one line over all samples
// with ONE zero column after every row and ONE zero row after every sample (and zeros before the first), so the
// zero padding of every window falls on stored zeros and a tap is a fixed distance along the line.  A group's
// stretch of pixels is then contiguous 16-byte units: it comes by one untiled bulk copy, lands as the
// no-swizzle K-major operand (8 pixels x 16 bytes are a core matrix, the next 8 pixels follow at once), and a tap is
// an operand that starts so many 16-byte units later.  The nine taps read ONE copy of the pixels; fetching a shifted
// tile per tap would move nine times the bytes.  Lines through the padding are computed and dropped: (S + 1)^2 / S^2.
//
// A stage of the ring is eight input planes (two groups) of 256 neighbouring pixels and their reach, and the weights
// of these planes for all nine taps: per tile of 128 pixels 9 steps of K = 8.  A first layer of up to four planes has
// one group; its steps pair two neighbouring taps of a window row instead (the second core matrix along K starts
// one pixel later), six steps in all.
//
// Splitting fp32 for tf32 tensor cores: w = w_hi + w_lo, h = h_hi + h_lo; D1 += h_hi w_hi, D2 += h_hi w_lo + h_lo w_hi
// (a bfloat16 weight is exact in tf32: w_lo = 0 and its products are left out).  D1 and D2 are drained into fp32
// registers after every three steps, and the accumulator sets alternate.  The tensor core adds with truncation towards
// zero, so a drained sum comes out too small by a share that grows with the steps between drains, and an average share
// is added back at every drain.  These shares are measured, not derived: the mean relative error of the losses of
// four-layer networks without it, spread over the layers, was 2.75e-8, 6.1e-8 and 16.3e-8 of a drained sum for drains
// after 1, 3 and 9 steps (fp32 weights), 0.95e-8, 3.2e-8 and 10e-8 (bfloat16, whose products have fewer bits to lose); they
// move by about a sixth with the data (images of either sign, all positive, with a large mean, 8 to 256 planes).
// Relative errors of the losses against 64 bits over 26 networks and inputs, geometric mean of the rms, and of the
// mean: this kernel 4.0e-8 and 5.7e-9, the CUDA-core kernel 4.4e-8 and 3.8e-9 (a binary32 loss is itself rounded by up
// to 6e-8); with drains after nine steps 6.4e-8 and 1.3e-8.
//
// Warp roles: warp 0 producer, warps 1 and 2 MMA issuers for one of the two tiles each, warp 1 owner of TMEM, warps 4-7
// and 8-11 drain and finish one of the tiles each (thread = pixel: bias, ReLU, the split into two terms, 16-byte stores
// along the pixels).  Work items are (model, block of output planes, pair of tiles); a block takes every gridDim.x-th one.
// The number of output planes is a constant of the instantiation: with a run-time number the draining loop's branches
// made the drains, not the MMAs, what the kernel waited for (three drains a stage: second layer below 163 us against 130).
//
// Before the layers, cnn_pack_kernel forms w = x - gamma v of every model in the operand layout (and the sums of
// v^2); after every second layer cnn_pool_kernel takes the 2 x 2 maxima.  Measured on 21 models of
// 32 x 32 x 3 -> 32, 32, 64, 64 planes: a step of 4 samples 93 us (with the CUDA-core kernel 353), of 32 samples with
// bfloat16 weights 382 us (1,268).  What bounds it: an MMA fetches its 128 pixels from shared memory in about 60 cycles
// whatever it multiplies them with (the alignment of a tap makes no difference), and the first layer of 32 samples
// writes 190 MB in 80 us.
#include <algorithm>
#include <math.h>

#include "zeno_internal.h"
#include "zeno_tc.cuh"

namespace zeno {

namespace {

constexpr int kCThreads = 32 * 12;
constexpr int kCMaxStages = 6;
constexpr int kCTiles = 2;                   // tiles of 128 pixels per item
constexpr int kCSmem = 225 * 1024;
constexpr int kCTmemCols = 512;
constexpr int kCMaxN = 64;                   // output planes per item
constexpr int kCMaxSets = 4;                 // accumulator sets
constexpr int kCDrain = 3;                   // steps after which the accumulators are drained

struct CnnTcArgs {
    const float *in;                         // [models][2][groups][px][4] (the shared batch: model stride 0)
    int64_t in_model;                        // floats per model
    int64_t px;                              // pixels of the input's line
    const float *w;                          // packed weights of this layer, first model
    const float *bias;                       // [model][nblk * N]
    int64_t w_model, bias_model;             // floats per model
    float *out;                              // pool == 0: the next layer's input; pool == 1: unsplit, one term
    int64_t out_model, out_px;
    int out_groups;                          // groups of four output planes the next layer has
    int pool;
    int groups, stages_per_item;             // groups of input planes; stages of an item
    int nblk;                                // items along the output planes
    int side, n_r, models, tile_pairs, tiles;
    int lead, out_lead;
    float debias;                            // average share of a drained D1 that truncation has taken
    int ring, stage_bytes, plane_bytes, a_bytes, b_bytes;
    int *status;
    uint32_t spin_limit;
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void tc_mma_tf32_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// K-major operand without swizzle: core matrices of 8 rows x 16 bytes, the next 8 rows 128 bytes on.  The low word
// holds the address in 16-byte units and, from bit 16 on, the distance of a step's second core matrix.
__device__ __forceinline__ uint64_t desc_plain(uint32_t low) {
    return (uint64_t)low | (uint64_t)(128 >> 4) << 32 | (uint64_t)1 << 46;
}

// two binary32 values at a time
__device__ __forceinline__ uint64_t pack2(uint32_t a, uint32_t b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
    uint32_t a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
    return make_float2(__uint_as_float(a), __uint_as_float(b));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// NB: blocks of sixteen output planes of an item
template <bool BF16W, bool FIRST, int NB>
__global__ void __launch_bounds__(kCThreads, 1) cnn_conv_tc_kernel(CnnTcArgs a) {
    constexpr int N = 16 * NB, kSets = kCTmemCols / (kCTiles * 2 * N) < kCMaxSets ? kCTmemCols / (kCTiles * 2 * N) : kCMaxSets;
    extern __shared__ __align__(128) uint8_t ring_s[];
    // full, empty [kCMaxStages]; dfull, dempty [kCTiles][kCMaxSets]
    constexpr int kBars = 2 * kCMaxStages + 2 * kCTiles * kCMaxSets;
    constexpr int kSteps = FIRST ? 6 : 9, kDrain = kCDrain;
    __shared__ __align__(8) uint64_t bars[kBars];
    __shared__ __align__(8) uint64_t drain_bar[kCTiles];
    __shared__ __align__(8) uint64_t never_bar;
    __shared__ uint32_t tmem_base_slot;
    __shared__ int abort_state[kAbortWords];
    int &abort_flag = abort_state[0];
    __shared__ int issued[kCMaxStages];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto bar_full = [&](int s) { return smem_u32(&bars[s]); };
    auto bar_empty = [&](int s) { return smem_u32(&bars[kCMaxStages + s]); };
    auto bar_dfull = [&](int t, int q) { return smem_u32(&bars[2 * kCMaxStages + t * kCMaxSets + q]); };
    auto bar_dempty = [&](int t, int q) { return smem_u32(&bars[2 * kCMaxStages + (kCTiles + t) * kCMaxSets + q]); };
    if (tid == 0) {
        abort_flag = 0;
        abort_state[1] = (int)a.spin_limit;
        for (int s = 0; s < kCMaxStages; ++s) {
            mbar_init(bar_full(s), 1);
            mbar_init(bar_empty(s), kCTiles);  // the commits of the MMAs that read the stage
            issued[s] = 0;
        }
        for (int t = 0; t < kCTiles; ++t) {
            for (int q = 0; q < kCMaxSets; ++q) {
                mbar_init(bar_dfull(t, q), 1);
                mbar_init(bar_dempty(t, q), 4);
            }
            mbar_init(smem_u32(&drain_bar[t]), 1);
        }
        mbar_init(smem_u32(&never_bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_slot)), "r"(kCTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_wait();
    pdl_launch_dependents();
    const uint32_t tmem = tmem_base_slot;
    volatile int *abortp = &abort_flag;
    const int pitch = a.side + 1;
    const int n_items = a.models * a.nblk * a.tile_pairs;
    constexpr int tile_cols = 2 * N;                             // D1 and D2 of a tile
    // item -> (model, block of planes, pair of tiles): neighbouring blocks share a model's weights in L2
    auto get_item = [&](int li, int &model, int &nb, int &pair) {
        const int item = blockIdx.x + li * gridDim.x;
        const int mb = item / a.tile_pairs;
        pair = item - mb * a.tile_pairs;
        model = mb / a.nblk;
        nb = mb - model * a.nblk;
        return item < n_items;
    };

    int model, nb, pair;
    if (warp == 0) {
        // ------------------------------------------------------------------ producer
        wait_for_nothing(smem_u32(&never_bar), abortp);
        int s = 0;
        uint32_t round = 0;
        constexpr int terms_groups = FIRST ? 1 : 2;               // groups of planes a stage holds, of either term
        for (int li = 0;; ++li) {
            if (!__all_sync(0xffffffffu, get_item(li, model, nb, pair) && !*abortp)) break;
            const float *in = a.in + (int64_t)model * a.in_model + ((int64_t)a.lead + pair * (kCTiles * 128) - pitch - 1) * 4;
            const float *w = a.w + (int64_t)model * a.w_model + (int64_t)nb * a.stages_per_item * (a.b_bytes / 4);
            bool ok = true;
            for (int st = 0; st < a.stages_per_item; ++st) {
                ok = __all_sync(0xffffffffu, mbar_wait(bar_empty(s), (round & 1) ^ 1, abortp));
                if (!ok) break;
                if (elect_one()) {
                    mbar_expect_tx(bar_full(s), a.a_bytes + a.b_bytes);
                    issued[s] = (int)round + 1;
                    const uint32_t dst = smem_u32(ring_s) + s * a.stage_bytes;
                    for (int p = 0; p < 2 * terms_groups; ++p) {   // leading terms of the groups, then the remainders
                        const int term = p / terms_groups, g = st * 2 + p - term * terms_groups;
                        bulk_load(dst + p * a.plane_bytes, in + (int64_t)(term * a.groups + g) * a.px * 4, a.plane_bytes, bar_full(s));
                    }
                    bulk_load(dst + a.a_bytes, w + (int64_t)st * (a.b_bytes / 4), a.b_bytes, bar_full(s));
                }
                __syncwarp();
                if (++s == a.ring) {
                    s = 0;
                    ++round;
                }
            }
            if (!ok) break;
        }
    } else if (warp <= kCTiles) {
        // ------------------------------------------------------------------ MMA issuers, one for each tile
        const int t = warp - 1;
        const uint32_t idesc_base = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(128 >> 4) << 24);
        const uint32_t idesc_n = idesc_base | ((uint32_t)(N >> 3) << 17);
        const uint32_t idesc_2n = idesc_base | ((uint32_t)((2 * N) >> 3) << 17);
        const uint32_t k_a = FIRST ? 16u : (uint32_t)a.plane_bytes, k_b = (uint32_t)(BF16W ? N : 2 * N) * 16u;
        const uint32_t lo_off = (uint32_t)(FIRST ? 1 : 2) * a.plane_bytes, b_step = 2u * (BF16W ? N : 2 * N);
        int s = 0, set = 0;
        uint32_t round = 0, use = 0;
        for (int li = 0;; ++li) {
            if (!__all_sync(0xffffffffu, get_item(li, model, nb, pair) && !*abortp)) break;
            const bool have = pair * kCTiles + t < a.tiles;      // the last pair may hold one tile
            bool ok = true;
            for (int st = 0; st < a.stages_per_item; ++st) {
                ok = __all_sync(0xffffffffu, mbar_wait(bar_full(s), round & 1, abortp));
                if (!ok) break;
                // the descriptors' low words count 16-byte units, so a step is one addition: one lane that issued all 36
                // MMAs of a stage was what the kernel waited for while it built every descriptor anew
                const uint32_t ax = (smem_u32(ring_s) + s * a.stage_bytes) >> 4;
                const uint32_t a_hi = ax | (k_a >> 4) << 16, a_lo = a_hi + (lo_off >> 4);
                const uint32_t b_0 = (ax + (a.a_bytes >> 4)) | (k_b >> 4) << 16;
#pragma unroll
                for (int k0 = 0; k0 < kSteps; k0 += kDrain) {
                    ok = __all_sync(0xffffffffu, mbar_wait(bar_dempty(t, set), (use & 1) ^ 1, abortp));
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        const uint32_t d1 = tmem + set * (kCTiles * tile_cols) + t * tile_cols, d2 = d1 + N;
                        if (have) {
#pragma unroll
                            for (int ks = k0; ks < k0 + kDrain; ++ks) {
                                const int dy = FIRST ? ks / 2 : ks / 3, dx = FIRST ? (ks % 2) * 2 : ks % 3;
                                const uint32_t at = (uint32_t)(t * 128 + dx) + dy * pitch;
                                const uint64_t hi = desc_plain(a_hi + at), lo = desc_plain(a_lo + at), wd = desc_plain(b_0 + ks * b_step);
                                if (BF16W) {
                                    tc_mma_tf32_ss(d1, hi, wd, idesc_n, (uint32_t)(ks - k0));       // h_hi w
                                    tc_mma_tf32_ss(d2, lo, wd, idesc_n, (uint32_t)(ks - k0));       // h_lo w
                                } else {
                                    tc_mma_tf32_ss(d1, hi, wd, idesc_2n, (uint32_t)(ks - k0));      // h_hi [w_hi; w_lo]
                                    tc_mma_tf32_ss(d2, lo, wd, idesc_n, 1u);                        // h_lo w_hi
                                }
                            }
                        }
                        tc_commit(bar_dfull(t, set));
                        if (k0 + kDrain == kSteps) tc_commit(bar_empty(s));
                    }
                    __syncwarp();
                    if (++set == kSets) {
                        set = 0;
                        ++use;
                    }
                }
                if (!ok) break;
                if (++s == a.ring) {
                    s = 0;
                    ++round;
                }
            }
            if (!ok) break;
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ drain and finish
        const int t = (warp - 4) >> 2, quad = warp & 3;          // this warp's tile of the pair and its pixels of the tile
        const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
        const int per_sample = pitch * pitch, drains = a.stages_per_item * (kSteps / kDrain);
        const uint64_t debias = pack2(__float_as_uint(a.debias), __float_as_uint(a.debias));
        int set = 0;
        uint32_t use = 0;
        for (int li = 0;; ++li) {
            if (!__all_sync(0xffffffffu, get_item(li, model, nb, pair) && !*abortp)) break;
            const bool have = pair * kCTiles + t < a.tiles;      // the last pair may hold one tile
            // the sums start from the bias, asked for before the first accumulators are awaited (written two kernels ago:
            // not by the read-only path)
            const float4 *bias = reinterpret_cast<const float4 *>(a.bias + (int64_t)model * a.bias_model + nb * N);
            uint64_t acc[N / 2];
#pragma unroll
            for (int c = 0; c < N / 4; ++c) {
                const float4 b = __ldcg(bias + c);
                acc[2 * c] = pack2(__float_as_uint(b.x), __float_as_uint(b.y));
                acc[2 * c + 1] = pack2(__float_as_uint(b.z), __float_as_uint(b.w));
            }
            bool ok = true;
            for (int dr = 0; dr < drains; ++dr) {
                ok = __all_sync(0xffffffffu, mbar_wait(bar_dfull(t, set), use & 1, abortp));
                if (!ok) break;
                tc_fence_after();
                // a missing tile's accumulators are read as well: whatever they hold, nothing of it is stored
                const uint32_t d = tmem + lane_addr + set * (kCTiles * tile_cols) + t * tile_cols;
#pragma unroll
                for (int b0 = 0; b0 < NB; b0 += 2) {
                    constexpr int kMost = NB < 2 ? 1 : 2;
                    uint32_t big[kMost][16], small[kMost][16];
#pragma unroll
                    for (int b = 0; b < kMost; ++b)
                        if (b0 + b < NB) {
                            tc_ld16(d + (b0 + b) * 16, big[b]);
                            tc_ld16(d + N + (b0 + b) * 16, small[b]);
                        }
                    tc_wait_ld();
                    if (b0 + 2 >= NB) {                          // all of the set is in registers
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar_dempty(t, set));
                    }
#pragma unroll
                    for (int b = 0; b < kMost; ++b)
                        if (b0 + b < NB) {
#pragma unroll
                            for (int j = 0; j < 16; j += 2) {
                                uint64_t &sum = acc[(b0 + b) * 8 + j / 2];
                                const uint64_t v = pack2(big[b][j], big[b][j + 1]), l = pack2(small[b][j], small[b][j + 1]);
                                sum = add2(sum, add2(v, fma2(v, debias, l)));
                            }
                        }
                }
                if (++set == kSets) {
                    set = 0;
                    ++use;
                }
            }
            if (!ok) break;
            const int q = (pair * kCTiles + t) * 128 + quad * 32 + lane;        // this thread's pixel on the line
            const int sample = q / per_sample, r = q - sample * per_sample, y = r / pitch, x = r - y * pitch;
            if (have && sample < a.n_r && y < a.side && x < a.side) {           // not padding
                float4 *out = reinterpret_cast<float4 *>(a.out + (int64_t)model * a.out_model) + a.out_lead + q;
#pragma unroll
                for (int c = 0; c < N / 4; ++c) {
                    const int grp = nb * (N / 4) + c;
                    if (grp >= a.out_groups) break;
                    const float2 z01 = unpack2(acc[2 * c]), z23 = unpack2(acc[2 * c + 1]);
                    const float4 z = make_float4(relu_keep_nan(z01.x), relu_keep_nan(z01.y), relu_keep_nan(z23.x), relu_keep_nan(z23.y));
                    if (a.pool) {
                        out[(int64_t)grp * a.out_px] = z;
                    } else {
                        const float4 h = make_float4(tf32_hi(z.x), tf32_hi(z.y), tf32_hi(z.z), tf32_hi(z.w));
                        out[(int64_t)grp * a.out_px] = h;
                        out[(int64_t)(a.out_groups + grp) * a.out_px] = make_float4(z.x - h.x, z.y - h.y, z.z - h.z, z.w - h.w);
                    }
                }
            }
            __syncwarp();                                        // the next item's first tcgen05.ld is the whole warp's
        }
    }

    // ---------------------------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp >= 1 && warp <= kCTiles && abort_flag) drain_mmas(smem_u32(&drain_bar[warp - 1]));
    if (tid == 0 && abort_flag) {
        for (int s = 0; s < kCMaxStages; ++s)
            if (issued[s] > 0) {
                for (uint32_t i = 0; i < kSpinLimit; ++i) {
                    if (mbar_try_wait(bar_full(s), (uint32_t)(issued[s] - 1) & 1)) break;
                    __nanosleep(64);
                }
            }
        atomicCAS(a.status, 0, wait_code(4, abort_flag, smem_u32(bars)));
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCTmemCols) : "memory");
    }
}

// What the layers read: the batch split into two terms in the layout of a first layer, and w = x - gamma v of every
// model's convolutional layers as operands, with their biases and the sums of v^2.  Entries no plane or tap stands for
// are zero from the allocation on and never written.
struct CnnPackLayer {
    int64_t offW, offB;
    int cin, cout, first, nks, n, rows, stages, splits, blocks, np_base;
    float *w, *bias;
    int64_t w_model, bias_model;
};
struct CnnPackArgs {
    const void *x, *V;
    int64_t ldv;
    float gamma;
    const float *features;
    float *in0;                    // [2][groups][px][4]
    int64_t px;
    int lead, side, planes, groups, n_r, weight_blocks;
    int first_model;               // of this launch; the workspace counts from it
    float *normpart;
    int np_slots;
    CnnPackLayer layer[ZENO_MAX_LAYERS];
};

template <typename T>
__global__ void __launch_bounds__(256) cnn_pack_kernel(const __grid_constant__ CnnPackArgs a) {
    pdl_wait();
    pdl_launch_dependents();
    const int tid = threadIdx.x;
    if ((int)blockIdx.x >= a.weight_blocks) {                    // the batch, dealt over the rest of the grid
        const int pixels = a.side * a.side, pitch = a.side + 1, total = a.n_r * a.groups * pixels;
        const int nb = (gridDim.x - a.weight_blocks) * gridDim.y;
        const int first = ((blockIdx.x - a.weight_blocks) * gridDim.y + blockIdx.y) * 256 + tid;
        // A first layer's paired taps multiply a fourth column with zero weights.  For the last pixel of the last sample
        // that is the first pixel of the slot after the batch, the one position beyond it that is read into a pixel that
        // counts: an earlier call with more samples may have left a NaN or an infinity there, and 0 x NaN is NaN.
        if (a.groups == 1 && first < 2)                          // of either term
            reinterpret_cast<float4 *>(a.in0)[first * a.px + a.lead + (int64_t)a.n_r * pitch * pitch] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int t = first; t < total; t += nb * 256) {
            const int ng = t / pixels, pix = t - ng * pixels, n = ng / a.groups, g = ng - n * a.groups;
            const int y = pix / a.side, x = pix - y * a.side;
            float h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = 4 * g + e;
                const float v = c < a.planes ? __ldg(a.features + ((int64_t)n * a.planes + c) * pixels + pix) : 0.f;
                h[e] = tf32_hi(v);
                l[e] = v - h[e];
            }
            float4 *dst = reinterpret_cast<float4 *>(a.in0) + a.lead + ((int64_t)n * pitch + y) * pitch + x;
            dst[(int64_t)g * a.px] = make_float4(h[0], h[1], h[2], h[3]);
            dst[(int64_t)(a.groups + g) * a.px] = make_float4(l[0], l[1], l[2], l[3]);
        }
        return;
    }
    // sixteen output planes of one layer of one model and sixteen of its input planes: a pair a thread, so that no load waits for
    // another one's use (with all input planes in one block, in turn, the experiment's network took 10.7 us)
    int li = 0, blk = blockIdx.x;
    while (blk >= a.layer[li].blocks) blk -= a.layer[li++].blocks;
    const CnnPackLayer &L = a.layer[li];
    const int c = blockIdx.y, model = a.first_model + c;
    const bool has_v = model > 0;
    const T *xp = static_cast<const T *>(a.x);
    const T *vp = static_cast<const T *>(a.V) + (has_v ? (int64_t)(model - 1) * a.ldv : 0);
    float nrm = 0.f;
    const int oblk = blk / L.splits, split = blk - oblk * L.splits;
    // consecutive threads: the four planes of a group, then the output planes, so that the stores are contiguous
    const int t = split * 256 + tid, ci = (t >> 6) * 4 + (t & 3), o = oblk * 16 + ((t >> 2) & 15);
    if (ci < L.cin && o < L.cout) {
        const int nb = o / L.n, row = o - nb * L.n;
        const int64_t src = L.offW + ((int64_t)o * L.cin + ci) * 9;
        float xv[9], vv[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            xv[k] = load_elem(xp + src + k);
            vv[k] = has_v ? load_elem(vp + src + k) : 0.f;
        }
        float *dst = L.w + (int64_t)c * L.w_model + (int64_t)(nb * L.stages + (L.first ? 0 : ci >> 3)) * L.nks * 2 * L.rows * 4 +
                     row * 4 + (ci & 3);
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const float w = candidate_param<T>(xv[k], vv[k], a.gamma);
            nrm = fmaf(vv[k], vv[k], nrm);
            // step and core matrix along K of this tap and plane
            const int step = L.first ? (k / 3) * 2 + (k % 3) / 2 : k, half = L.first ? (k % 3) & 1 : (ci >> 2) & 1;
            float *d = dst + (int64_t)(step * 2 + half) * L.rows * 4;
            if (is_bf16<T>::value) {
                d[0] = w;
            } else {
                const float h = tf32_hi(w);
                d[0] = h;
                d[L.n * 4] = w - h;
            }
        }
    }
    if (split == 0 && tid < 16 && L.offB >= 0 && oblk * 16 + tid < L.cout) {
        const int o = oblk * 16 + tid;
        const float bv = has_v ? load_elem(vp + L.offB + o) : 0.f;
        nrm = fmaf(bv, bv, nrm);
        L.bias[(int64_t)c * L.bias_model + o] = candidate_param<T>(load_elem(xp + L.offB + o), bv, a.gamma);
    }
    if (has_v) {                                                 // one slot per warp
#pragma unroll
        for (int s = 16; s >= 1; s >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, s);
        if ((tid & 31) == 0) a.normpart[(int64_t)(model - 1) * a.np_slots + L.np_base + blk * 8 + (tid >> 5)] = nrm;
    }
}

__device__ __forceinline__ float max_nan(float a, float b) { return (a != a) ? a : ((b != b) ? b : fmaxf(a, b)); }

// 2 x 2 maxima of a layer's planes z [model][group][px][4]: into the next layer's input, split into its two terms, or
// (flat != NULL) as the dense layer's input [model][n_r][planes][side / 2]^2.
__global__ void __launch_bounds__(256) cnn_pool_kernel(const float *z, int64_t z_model, int64_t z_px, int lead, int side, int planes,
                                                       int groups, int n_r, float *out, int64_t out_model, int64_t out_px,
                                                       int out_groups, int out_lead, float *flat) {
    pdl_wait();
    pdl_launch_dependents();
    const int model = blockIdx.y, half = side / 2, pixels = half * half, pitch = side + 1;
    const int total = n_r * groups * pixels;
    const float4 *zm = reinterpret_cast<const float4 *>(z + (int64_t)model * z_model) + lead;
    for (int t = blockIdx.x * 256 + threadIdx.x; t < total; t += gridDim.x * 256) {
        const int ng = t / pixels, pix = t - ng * pixels, n = ng / groups, g = ng - n * groups;
        const int y = pix / half, x = pix - y * half;
        const float4 *p = zm + (int64_t)g * z_px + ((int64_t)n * pitch + 2 * y) * pitch + 2 * x;
        const float4 a = __ldcg(p), b = __ldcg(p + 1), c = __ldcg(p + pitch), d = __ldcg(p + pitch + 1);
        const float v[4] = {max_nan(max_nan(a.x, b.x), max_nan(c.x, d.x)), max_nan(max_nan(a.y, b.y), max_nan(c.y, d.y)),
                            max_nan(max_nan(a.z, b.z), max_nan(c.z, d.z)), max_nan(max_nan(a.w, b.w), max_nan(c.w, d.w))};
        if (flat) {
            float *f = flat + ((int64_t)model * n_r + n) * planes * pixels + (int64_t)4 * g * pixels + pix;
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (4 * g + e < planes) f[(int64_t)e * pixels] = v[e];
        } else {
            const int op = half + 1;
            float4 *o = reinterpret_cast<float4 *>(out + (int64_t)model * out_model) + out_lead + ((int64_t)n * op + y) * op + x;
            const float4 h = make_float4(tf32_hi(v[0]), tf32_hi(v[1]), tf32_hi(v[2]), tf32_hi(v[3]));
            o[(int64_t)g * out_px] = h;
            o[(int64_t)(out_groups + g) * out_px] = make_float4(v[0] - h.x, v[1] - h.y, v[2] - h.z, v[3] - h.w);
        }
    }
}

int round_up_int(int v, int q) { return (v + q - 1) / q * q; }

template <bool BF16W, bool FIRST, int NB>
cudaError_t launch_conv_nb(Context &c, const CnnTcArgs &a, int blocks, size_t smem, cudaStream_t s) {
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(cnn_conv_tc_kernel<BF16W, FIRST, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kCSmem);
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    return launch_chained(cnn_conv_tc_kernel<BF16W, FIRST, NB>, dim3(blocks), dim3(kCThreads), smem, s, chain_launches(c), a);
}
template <bool BF16W, bool FIRST>
cudaError_t launch_conv(Context &c, const CnnTcArgs &a, int nb, int blocks, size_t smem, cudaStream_t s) {
    static_assert(kCMaxN == 64, "one to four blocks of sixteen planes");
    if (nb == 1) return launch_conv_nb<BF16W, FIRST, 1>(c, a, blocks, smem, s);
    if (nb == 2) return launch_conv_nb<BF16W, FIRST, 2>(c, a, blocks, smem, s);
    if (nb == 3) return launch_conv_nb<BF16W, FIRST, 3>(c, a, blocks, smem, s);
    return launch_conv_nb<BF16W, FIRST, 4>(c, a, blocks, smem, s);
}

}  // namespace

// norm partials of a layer's weights: a slot per warp of every block that packs them
int cnn_tc_norm_slots(int cin, int cout) { return (cin + 15) / 16 * ((cout + 15) / 16) * 8; }

// Sizes of the layers of a handle's network, and where their parts lie in a workspace for `models` models (floats from
// its start).
static void layout_models(const Context &c, int models, CnnTcNet *net) {
    const zeno_model_desc &d = c.desc;
    const int lc = d.n_layers - 1;
    const bool bf16 = d.param_dtype == ZENO_BF16;
    int64_t off = 0;
    auto take = [&](int64_t floats) {
        const int64_t at = off;
        off += (floats + 63) / 64 * 64;
        return at;
    };
    int side = (int)d.dims[0];
    int64_t z_most = 0;
    net->layers = lc;
    net->models = models;
    for (int l = 0; l < lc; ++l) {
        CnnTcLayer &L = net->layer[l];
        L.side = side;
        L.cin = (int)d.dims[l + 1];
        L.cout = (int)d.dims[l + 2];
        L.first = l == 0 && L.cin <= 4;
        L.pool = l & 1;
        L.groups = L.first ? 1 : round_up_int(L.cin, 8) / 4;
        L.stages = L.first ? 1 : L.groups / 2;
        L.nks = L.first ? 6 : 9;
        L.nblk = (L.cout + kCMaxN - 1) / kCMaxN;
        L.n = round_up_int((L.cout + L.nblk - 1) / L.nblk, 16);
        L.rows = bf16 ? L.n : 2 * L.n;
        // the line of pixels: zeros before the first row, after it whole items and their reach
        L.lead = side + 2;
        L.px = L.lead + (int64_t)(c.n_r_max + 1) * (side + 1) * (side + 1) + kCTiles * 128 + side + 3;
        L.in_model = 2 * (int64_t)L.groups * L.px * 4;
        L.in = take(L.in_model * (l == 0 ? 1 : models));
        L.w_model = (int64_t)L.nblk * L.stages * L.nks * 2 * L.rows * 4;
        L.w = take(L.w_model * models);
        L.bias_model = (int64_t)L.nblk * L.n;
        L.bias = take(L.bias_model * models);
        if (L.pool) {
            const int64_t z = (int64_t)(L.cout + 3) / 4 * L.px * 4 * models;
            if (z > z_most) z_most = z;
            side /= 2;
        }
    }
    net->z = take(z_most);
    net->floats = off;
}

// As many models as 4 GiB hold, at least one, so that a large handle leaves the memory to the caller's candidates: 101
// models of 32 x 32 x 3 -> 32, 32, 64, 64 with 128 samples would take 8.4 GB (the CUDA-core layers' buffers: 3.4).  A
// group's uneven last wave and the gaps between its kernels are what it costs: their step takes 6.66 ms in two groups,
// with 512 MiB and groups of six models 7.76.
constexpr int64_t kCWorkspaceFloats = (int64_t)1 << 30;
void cnn_tc_layout(const Context &c, CnnTcNet *net) {
    layout_models(c, c.m_max + 1, net);
    if (net->floats <= kCWorkspaceFloats) return;
    CnnTcNet one, two;
    layout_models(c, 1, &one);
    layout_models(c, 2, &two);
    const int64_t more = (kCWorkspaceFloats - one.floats) / (two.floats - one.floats);
    const int most = more < 0 ? 1 : 1 + (int)more;
    if (most > c.m_max) return;
    const int groups = (c.m_max + most) / most;                      // of evenly many models
    layout_models(c, (c.m_max + groups) / groups, net);
}

cudaError_t launch_cnn_tc(Context &c, const CnnTcNet &net, const void *x, const void *V, int64_t ldv, const float *features,
                          int n_r, int m, float gamma, float *flat, cudaStream_t s, int *launches) {
    const bool bf16 = c.desc.param_dtype == ZENO_BF16;
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    CnnPackArgs p = {};
    p.x = x;
    p.V = V;
    p.ldv = ldv;
    p.gamma = gamma;
    p.features = features;
    p.in0 = c.cnn_ws + net.layer[0].in;
    p.px = net.layer[0].px;
    p.lead = net.layer[0].lead;
    p.side = net.layer[0].side;
    p.planes = net.layer[0].cin;
    p.groups = net.layer[0].groups;
    p.n_r = n_r;
    p.normpart = c.normpart;
    p.np_slots = c.np_slots;
    for (int l = 0; l < net.layers; ++l) {
        const CnnTcLayer &L = net.layer[l];
        CnnPackLayer &q = p.layer[l];
        q.offW = c.offW[l];
        q.offB = c.offB[l];
        q.cin = L.cin;
        q.cout = L.cout;
        q.first = L.first;
        q.nks = L.nks;
        q.n = L.n;
        q.rows = L.rows;
        q.stages = L.stages;
        q.splits = (L.cin + 15) / 16;
        q.blocks = (L.cout + 15) / 16 * q.splits;
        q.np_base = c.np_base[l];
        q.w = c.cnn_ws + L.w;
        q.bias = c.cnn_ws + L.bias;
        q.w_model = L.w_model;
        q.bias_model = L.bias_model;
        p.weight_blocks += q.blocks;
    }
    const int64_t batch = (int64_t)n_r * p.groups * p.side * p.side;
    const CnnTcLayer &last = net.layer[net.layers - 1];
    const int64_t flat_model = (int64_t)n_r * last.cout * (last.side / 2) * (last.side / 2);
    for (int first = 0; first <= m; first += net.models) {
        const int models = std::min(net.models, m + 1 - first);
        int fx = 0;                                  // the batch is packed once, with the first group's weights
        if (first == 0) {
            fx = (int)((batch + 256LL * models - 1) / (256LL * models));
            const int fx_cap = 8 * sms / models + 1;
            if (fx > fx_cap) fx = fx_cap;
        }
        p.first_model = first;
        ++*launches;
        profile_mark(c, "cnn_conv3x3", s);          // with the first layer
        const dim3 pack_grid(p.weight_blocks + fx, models);
        cudaError_t e = bf16 ? launch_chained(cnn_pack_kernel<__nv_bfloat16>, pack_grid, dim3(256), 0, s, chain_launches(c), p)
                             : launch_chained(cnn_pack_kernel<float>, pack_grid, dim3(256), 0, s, chain_launches(c), p);
        if (e != cudaSuccess) return e;
        for (int l = 0; l < net.layers; ++l) {
            const CnnTcLayer &L = net.layer[l];
            const CnnTcLayer *next = l + 1 < net.layers ? &net.layer[l + 1] : nullptr;
            CnnTcArgs a = {};
            a.in = c.cnn_ws + L.in;
            a.in_model = l == 0 ? 0 : L.in_model;
            a.px = L.px;
            a.w = c.cnn_ws + L.w;
            a.bias = c.cnn_ws + L.bias;
            a.w_model = L.w_model;
            a.bias_model = L.bias_model;
            a.pool = L.pool;
            const int z_groups = (L.cout + 3) / 4;
            if (L.pool) {
                a.out = c.cnn_ws + net.z;
                a.out_model = (int64_t)z_groups * L.px * 4;
                a.out_px = L.px;
                a.out_groups = z_groups;
                a.out_lead = L.lead;
            } else {
                a.out = c.cnn_ws + next->in;
                a.out_model = next->in_model;
                a.out_px = next->px;
                a.out_groups = next->groups;
                a.out_lead = next->lead;
            }
            a.groups = L.groups;
            a.stages_per_item = L.stages;
            a.debias = bf16 ? 3.2e-8f : 6.1e-8f;              // for kCDrain steps, see the top of the file
            a.nblk = L.nblk;
            a.side = L.side;
            a.n_r = n_r;
            a.models = models;
            a.tiles = (int)(((int64_t)n_r * (L.side + 1) * (L.side + 1) + 127) / 128);
            a.tile_pairs = (a.tiles + kCTiles - 1) / kCTiles;
            a.lead = L.lead;
            a.plane_bytes = (kCTiles * 128 + 2 * (L.side + 2) + 1) * 16;      // the paired taps of a first layer reach one further
            a.a_bytes = (L.first ? 2 : 4) * a.plane_bytes;
            a.b_bytes = L.nks * 2 * L.rows * 16;
            a.stage_bytes = round_up_int(a.a_bytes + a.b_bytes, 128);
            a.ring = (kCSmem - 1024) / a.stage_bytes;
            if (a.ring > kCMaxStages) a.ring = kCMaxStages;
            a.status = c.dev_status;
            a.spin_limit = c.spin_limit;
            const int items = a.models * a.nblk * a.tile_pairs;
            const int rounds = (items + sms - 1) / sms, blocks = (items + rounds - 1) / rounds;
            ++*launches;
            if (l > 0) profile_mark(c, "cnn_conv3x3", s);
            // more than half of an SM's shared memory, so that no SM holds two of the kernel's blocks, of which the second would
            // wait for the first one's tensor memory while other SMs idle (two layers of 16 planes, 640 images: 59 us against 51)
            const size_t smem = std::max((size_t)a.ring * a.stage_bytes, (size_t)116 * 1024);
            e = bf16 ? (L.first ? launch_conv<true, true>(c, a, L.n / 16, blocks, smem, s) : launch_conv<true, false>(c, a, L.n / 16, blocks, smem, s))
                     : (L.first ? launch_conv<false, true>(c, a, L.n / 16, blocks, smem, s) : launch_conv<false, false>(c, a, L.n / 16, blocks, smem, s));
            if (e != cudaSuccess) return e;
            if (!L.pool) continue;
            const int total = n_r * z_groups * (L.side / 2) * (L.side / 2);
            int bx = (total + 255) / 256;
            const int cap = 16 * sms / models + 1;
            if (bx > cap) bx = cap;
            ++*launches;
            e = launch_chained(cnn_pool_kernel, dim3(bx, models), dim3(256), 0, s, chain_launches(c), (const float *)a.out, a.out_model,
                               a.out_px, L.lead, L.side, L.cout, z_groups, n_r, next ? c.cnn_ws + next->in : nullptr,
                               next ? next->in_model : 0, next ? next->px : 0, next ? next->groups : 0, next ? next->lead : 0,
                               next ? nullptr : flat + first * flat_model);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace zeno
