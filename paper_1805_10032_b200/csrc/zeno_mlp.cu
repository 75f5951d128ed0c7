// Candidate-model forward for the softmax-cross-entropy MLP (Definition 2: f_r(x) and
// f_r(x - gamma v_i) on the same n_r samples), CUDA-core path.
//
// One launch per dense layer evaluates that layer for all m+1 models at once (model 0 is x itself); w = x - gamma v is
// formed from the loads of x and V (the perturbed model never exists in memory), and the same pass sums the squares of
// the V entries (the rho ||v||^2 term).
//
// A small last layer (mlp_head_kernel) runs as one cluster of blocks per model and also evaluates the
// cross-entropy.  In a step the averaging kernel forms the scores and the ranking from the losses; in a call that
// ends with the scores the block that finishes last (a ticket, no waiting) does, so neither costs a launch.
#include <type_traits>

#include "zeno_internal.h"
#include "zeno_tail.cuh"

namespace zeno {

namespace {

// One dense layer of all models, rows of any alignment, by tiles (the layers layer_by_columns in zeno_rows.cu does not take).  A block
// takes 8 R output rows of one model and 8 TN samples and
// stages slices of 64 input columns in shared memory -- w = x - gamma v formed on the way, v^2 accumulated, all of the
// next slice's loads in flight during the present one's arithmetic.  Its four groups of 64 threads take sixteen of the
// columns each and their sums are added at the end, so that few rows still have eight warps at work on every 8 R of
// them; a thread holds R rows x TN samples and reads four columns of each at a time (R + TN 16-byte reads for 4 R TN
// multiplications).  R = 8, or 4 for layers of up to 32 rows, which then take up to 64 samples at a time instead of 32.
// VEC (rows aligned to four elements): a load takes four columns of a row, half a warp a row's slice; else a warp loads
// 32 neighbouring columns of one row, which needs no alignment and touches two lines.
// The products are summed in runs of 64 columns that are then added to the total, so rounding errors stay those of
// short sums.  Where that leaves SMs idle a cluster of blocks deals the slices out and meets in the first one's
// shared memory.
// Bound by the loads' latency and the CUDA cores' rate: 38 models of 1029 x 301 with 19 samples take 61 us (one
// warp per four rows and one block an SM: 80).  A whole pass with VEC and without: 101 models of 2500 x 2000 in bfloat16,
// 4 samples, 892 us and 3,381; with R = 4 and 8: 61 models of 3001 x 20 x 3, 200 samples, 181 us and 309.
constexpr int kLK = 64, kLGroups = 4, kLPitch = kLK + 4;
constexpr int kLRun = 4;                         // slices of a run (a group's sixteen columns of each)
constexpr int kLFewRows = 32;                    // layers of up to so many rows: R = 4
__host__ __device__ constexpr int layer_stage_floats(int R, int TN) { return 2 * (8 * R + 8 * TN) * kLPitch; }
__host__ __device__ constexpr int layer_red_floats(int R, int TN) { return 8 * R * (8 * TN + 1); }
__host__ __device__ constexpr int layer_own_floats(int R, int TN) {
    return layer_stage_floats(R, TN) > kLGroups * layer_red_floats(R, TN) ? layer_stage_floats(R, TN) : kLGroups * layer_red_floats(R, TN);
}
inline size_t layer_smem(int R, int TN, int cluster) {
    return sizeof(float) * ((size_t)layer_own_floats(R, TN) + (cluster > 1 ? cluster * (layer_red_floats(R, TN) + 8) : 0));
}

template <typename T, int R, int TN, bool VEC>
__global__ void __launch_bounds__(kLGroups * 64, 2) mlp_layer_kernel(LayerArgs a, int sample_tiles, int cluster) {
    constexpr int kRows = 8 * R, BN = 8 * TN, kRed = layer_red_floats(R, TN), kOwn = layer_own_floats(R, TN);
    // Loads with no condition around them, entries beyond the rows or columns taken from elsewhere in the layer and dropped
    // when they are staged: every conditional bfloat16 load became a branch with a wait of its own (21 models of
    // 1345 x 1000, 4 samples: 217 us a pass against 102).  Binary32 loads stay conditional, and so do bfloat16 ones beside the
    // registers of more samples: the masks and the spills cost more there (10 to 20 %).
    constexpr bool kFree = VEC || (is_bf16<T>::value && TN <= 2);
    using Raw = typename std::conditional<VEC, typename RawOf<T>::Four, typename std::conditional<kFree, typename RawOf<T>::One, float>::type>::type;
    constexpr int kLoads = VEC ? R / 2 : 2 * R;  // of x and of v, a thread and slice
    extern __shared__ __align__(16) float smem_dyn[];
    pdl_wait();
    pdl_launch_dependents();
    if (cluster > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = tid >> 6, t = tid & 63;
    const int rank = cluster > 1 ? (int)cluster_rank() : 0;
    const int c = blockIdx.y;                    // model: 0 = x, 1+i = x - gamma v_i
    const int tile = blockIdx.x / cluster, row_tile = tile / sample_tiles, sample_tile = tile - row_tile * sample_tiles;
    const int row0 = row_tile * kRows, j0 = sample_tile * BN;
    const int K = a.in;
    const bool has_v = c > 0;
    const T *xw = static_cast<const T *>(a.x) + a.offW;
    const T *vbase = static_cast<const T *>(a.V) + (has_v ? (int64_t)(c - 1) * a.ldv : 0);
    const T *vw = vbase + a.offW;
    const float *hin = a.Hin + (int64_t)c * a.hin_cand_stride;
    const int tx = t & 7, ty = t >> 3;           // this thread's rows tx + 8 r and samples ty + 8 n

    float acc[R][TN], tot[R][TN];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < TN; ++n) acc[r][n] = tot[r][n] = 0.f;
    float nrm = 0.f;
    Raw xr[kLoads], vr[kLoads];
    float hr[2 * TN];
    // VEC: rows 2 warp + (lane >> 4) + 16 u, columns from 4 (lane & 15) on; else rows warp + 8 r, columns lane and lane + 32
    const int vrow = 2 * warp + (lane >> 4), vcol = 4 * (lane & 15);
    auto load = [&](int kt) {
        if constexpr (VEC) {
#pragma unroll
            for (int u = 0; u < R / 2; ++u) {
                const int k = kt * kLK + vcol;
                const int64_t at = (int64_t)min(row0 + vrow + 16 * u, a.out - 1) * K + (k < K ? k : 0);
                xr[u] = __ldg(reinterpret_cast<const Raw *>(xw + at));
                vr[u] = __ldg(reinterpret_cast<const Raw *>(vw + at));         // of model 0 a row that is dropped
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = kt * kLK + h * 32 + lane, o = row0 + warp + 8 * r;
                    if constexpr (kFree) {
                        const int64_t at = (int64_t)min(o, a.out - 1) * K + min(k, K - 1);
                        xr[2 * r + h] = __ldg(reinterpret_cast<const Raw *>(xw + at));
                        vr[2 * r + h] = __ldg(reinterpret_cast<const Raw *>(vw + at));
                    } else {
                        const bool ok = k < K && o < a.out;
                        xr[2 * r + h] = ok ? load_elem(xw + (int64_t)o * K + k) : 0.f;
                        vr[2 * r + h] = ok && has_v ? load_elem(vw + (int64_t)o * K + k) : 0.f;
                    }
                }
        }
#pragma unroll
        for (int r = 0; r < TN; ++r)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = kt * kLK + h * 32 + lane, j = j0 + warp + 8 * r;
                hr[2 * r + h] = k < K && j < a.n_r ? __ldg(hin + (int64_t)j * K + k) : 0.f;
            }
    };
    auto store = [&](int b, int kt) {
        float *ws = smem_dyn + b * (kRows + BN) * kLPitch, *hs = ws + kRows * kLPitch;
        if constexpr (VEC) {
#pragma unroll
            for (int u = 0; u < R / 2; ++u) {
                const bool ok = kt * kLK + vcol < K && row0 + vrow + 16 * u < a.out;
                const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 x = ok ? raw_to_float4(xr[u]) : zero, v = ok && has_v ? raw_to_float4(vr[u]) : zero;
                nrm = fmaf(v.x, v.x, nrm);
                nrm = fmaf(v.y, v.y, nrm);
                nrm = fmaf(v.z, v.z, nrm);
                nrm = fmaf(v.w, v.w, nrm);
                *reinterpret_cast<float4 *>(ws + (vrow + 16 * u) * kLPitch + vcol) =
                    make_float4(candidate_param<T>(x.x, v.x, a.gamma), candidate_param<T>(x.y, v.y, a.gamma),
                                candidate_param<T>(x.z, v.z, a.gamma), candidate_param<T>(x.w, v.w, a.gamma));
            }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float x, v;
                    if constexpr (kFree) {
                        const bool ok = kt * kLK + h * 32 + lane < K && row0 + warp + 8 * r < a.out;
                        x = ok ? raw_to_float(xr[2 * r + h]) : 0.f;
                        v = ok && has_v ? raw_to_float(vr[2 * r + h]) : 0.f;
                    } else {
                        x = xr[2 * r + h];
                        v = vr[2 * r + h];
                    }
                    nrm = fmaf(v, v, nrm);
                    ws[(warp + 8 * r) * kLPitch + h * 32 + lane] = candidate_param<T>(x, v, a.gamma);
                }
        }
#pragma unroll
        for (int r = 0; r < TN; ++r)
#pragma unroll
            for (int h = 0; h < 2; ++h) hs[(warp + 8 * r) * kLPitch + h * 32 + lane] = hr[2 * r + h];
    };
    const int slices = (K + kLK - 1) / kLK;
    if (rank < slices) {
        load(rank);
        store(0, rank);
        __syncthreads();
        int b = 0, run = 0;
        for (int kt = rank; kt < slices; kt += cluster, b ^= 1) {
            const bool more = kt + cluster < slices;
            if (more) load(kt + cluster);
            const float *ws = smem_dyn + b * (kRows + BN) * kLPitch + g * 16, *hs = ws + kRows * kLPitch;
#pragma unroll
            for (int k = 0; k < 16; k += 4) {
                float4 h[TN];
#pragma unroll
                for (int n = 0; n < TN; ++n) h[n] = *reinterpret_cast<const float4 *>(hs + (ty + 8 * n) * kLPitch + k);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4 w = *reinterpret_cast<const float4 *>(ws + (tx + 8 * r) * kLPitch + k);
#pragma unroll
                    for (int n = 0; n < TN; ++n) {
                        acc[r][n] = fmaf(w.x, h[n].x, acc[r][n]);
                        acc[r][n] = fmaf(w.y, h[n].y, acc[r][n]);
                        acc[r][n] = fmaf(w.z, h[n].z, acc[r][n]);
                        acc[r][n] = fmaf(w.w, h[n].w, acc[r][n]);
                    }
                }
            }
            if (++run == kLRun || !more) {
                run = 0;
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int n = 0; n < TN; ++n) {
                        tot[r][n] += acc[r][n];
                        acc[r][n] = 0.f;
                    }
            }
            if (more) {
                store(b ^ 1, kt + cluster);
                __syncthreads();
            }
        }
    }
    // the groups' sums, in group order
    __syncthreads();
    float *red = smem_dyn;                                           // [kLGroups][kRows][BN + 1]
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int n = 0; n < TN; ++n) red[g * kRed + (tx + 8 * r) * (BN + 1) + ty + 8 * n] = tot[r][n];
    __syncthreads();
    constexpr int kStep = kLGroups * 64 / kRows;                     // a thread finishes one row's samples n0, n0 + kStep, ..
    const int row = R == 8 ? t : tid % kRows, n0 = R == 8 ? g : tid / kRows, o = row0 + row;
    float bx = 0.f, bv = 0.f;
    if (rank == 0 && o < a.out && a.offB >= 0) {
        bx = load_elem(static_cast<const T *>(a.x) + a.offB + o);
        if (has_v) bv = load_elem(vbase + a.offB + o);
    }
    if (n0 == 0) nrm = fmaf(bv, bv, nrm);
    nrm = warp_sum(nrm);
    float *parts = smem_dyn + kOwn;                                  // [cluster][kRed + 8], the first block's is used
    if (cluster > 1) {
        __syncwarp();
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        const uint32_t dst = cluster_addr(parts + rank * (kRed + 8), 0);
        for (int n = n0; n < BN; n += kStep) {
            float z = 0.f;
#pragma unroll
            for (int u = 0; u < kLGroups; ++u) z += red[u * kRed + row * (BN + 1) + n];
            cluster_store(dst + 4 * (row * (BN + 1) + n), z);
        }
        if (lane == 0) cluster_store(dst + 4 * (kRed + warp), nrm);
        cluster_barrier();
        if (rank != 0) return;
        nrm = 0.f;
        for (int r = 0; r < cluster; ++r) nrm += parts[r * (kRed + 8) + kRed + warp];
    }
    const float bias = candidate_param<T>(bx, bv, a.gamma);
    for (int n = n0; n < BN; n += kStep) {
        float z = 0.f;
        if (cluster > 1) {
            for (int r = 0; r < cluster; ++r) z += parts[r * (kRed + 8) + row * (BN + 1) + n];
        } else {
#pragma unroll
            for (int u = 0; u < kLGroups; ++u) z += red[u * kRed + row * (BN + 1) + n];
        }
        if (a.offB >= 0) z += bias;
        if (a.relu) z = relu_keep_nan(z);
        if (o < a.out && j0 + n < a.n_r) a.Hout[((int64_t)c * a.n_r + j0 + n) * a.out + o] = z;
    }
    // partial ||v||^2 of the rows and bias entries; one slot per warp
    if (has_v && sample_tile == 0 && lane == 0)
        a.normpart[(int64_t)(c - 1) * a.np_slots + a.np_base + row_tile * (kLGroups * 2) + warp] = nrm;
}

// The last layer when it is small (out <= 32 classes and n_r <= 32 samples, or out <= 16 and
// n_r <= 64): a cluster of blocks per model computes all of the model's logits and its cross-entropy.
// Block r of the cluster takes a slice of the input range: it forms w = x - gamma v for its columns of the layer's
// rows in shared memory (coalesced loads, v^2 accumulated on the way), before it waits for the kernel that produces the
// activations; warp q then multiplies samples SPW q .. SPW q + SPW - 1, whose activations nobody else of the block needs and
// which come straight from memory, against all rows, lanes striding k; the partial logits go to the first block's shared
// memory, which adds them up and takes the loss, half a warp per sample where the classes fit.
// The work is a chain of latencies (784 x 10 of 21 models: 0.7 MB) and, with many samples, of shared-memory reads: every
// warp reads all rows.  65 models of 4096 x 10 in bfloat16, 64 samples: 30 us a scoring pass (43 with the activations through
// shared memory, sixteen rows for ten and a warp per sample in the loss); 1029 x 10, binary32: 22 (29).
// Blocks an SM has room for.  Clusters are sized for two an SM with up to 16 x 16 logits, but clusters of four and eight leave places of
// a GPC's SMs empty: 36 models in clusters of eight are 288 blocks, of which two an SM are 264 at a time and three 384.  Rows of
// any alignment, whose loads are of one entry, do with the registers for three (35 candidates of 7969 x 13, 5 samples: 27.0 us; with two
// 39.8; 73 of 10760 x 10, one sample: 55 and 85); of four entries they do not.
__host__ __device__ constexpr int head_blocks(int out_t, int spw, bool vec) {
    return out_t <= 16 && spw <= 2 ? (vec ? 2 : 3) : !vec && out_t * spw <= 64 ? 2 : 1;
}
// bytes of the staged rows, at most
__host__ __device__ constexpr int head_rows_bytes(int out_t, int spw, bool vec) { return (head_blocks(out_t, spw, vec) == 3 ? 56 : 96) * 1024; }
template <typename T, int OUT_T, int SPW, bool VEC>
__global__ void __launch_bounds__(256, head_blocks(OUT_T, SPW, VEC)) mlp_head_kernel(LayerArgs a, int cluster, int kslice, int KC) {
    constexpr int NS = 8 * SPW, W = 4;           // samples a cluster can hold; columns of a lane at a time
    constexpr int kAhead = SPW == 8 || (!VEC && OUT_T > 12 && SPW > 1) ? 1 : SPW == 4 ? 2 : 4;      // times 128 columns of the samples on their way
    constexpr int kRows = (OUT_T + 7) / 8;       // rows a warp stages
    constexpr int kLossLanes = OUT_T <= 16 ? 16 : 32, kLossAt = 256 / kLossLanes, kLossTurns = (NS + kLossAt - 1) / kLossAt;
    extern __shared__ __align__(16) float smem_dyn[];
    float *ws = smem_dyn;                                            // [OUT_T][KC]
    float *zp = ws + OUT_T * KC;                                     // [cluster][NS][OUT_T], the first block's is used
    float *np = zp + cluster * NS * OUT_T;                           // [cluster][8] sums of v^2, likewise
    __shared__ double loss_s[NS];

    // The weights are inputs of the whole call: unless this is the call's first kernel (what precedes it
    // on the stream may then still be producing x or V), they are read while the kernel that produces the
    // activations is still running.
    if (a.first_in_call) pdl_wait();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = (int)cluster_rank();
    const int c = blockIdx.x / cluster;
    const int K = a.in;
    const int k0 = rank * kslice, k1 = min(K, k0 + kslice);
    const bool has_v = c > 0;
    const T *xw = static_cast<const T *>(a.x) + a.offW;
    const T *vbase = static_cast<const T *>(a.V) + (has_v ? (int64_t)(c - 1) * a.ldv : 0);
    const T *vw = vbase + a.offW;
    const float *hin = a.Hin + (int64_t)c * a.hin_cand_stride;

    float acc[OUT_T][SPW];
#pragma unroll
    for (int o = 0; o < OUT_T; ++o)
#pragma unroll
        for (int q = 0; q < SPW; ++q) acc[o][q] = 0.f;
    float nrm = 0.f;
    // the first block's: a lane's bias entry and the labels of the samples it takes, requested now, used at the end
    const int cls = lane & (kLossLanes - 1), first_loss = threadIdx.x / kLossLanes;
    float bias_x = 0.f, bias_v = 0.f;
    int lab[kLossTurns];
#pragma unroll
    for (int q = 0; q < kLossTurns; ++q) lab[q] = 0;
    if (rank == 0) {
        if (a.offB >= 0 && cls < a.out) {
            bias_x = load_elem(static_cast<const T *>(a.x) + a.offB + cls);
            if (has_v) bias_v = load_elem(vbase + a.offB + cls);
            if (threadIdx.x < kLossLanes) nrm = bias_v * bias_v;
        }
#pragma unroll
        for (int q = 0; q < kLossTurns; ++q)
            if (first_loss + kLossAt * q < a.n_r) lab[q] = __ldg(a.labels + first_loss + kLossAt * q);
    }

    // w = x - gamma v of the layer's rows for the columns from kb on (zero beyond the rows and the slice)
    auto stage_weights = [&](int kb) {
        if constexpr (VEC) {
            constexpr int kBatch = 4;            // of 128 columns: all of a thread's loads of a batch before the first is used
            for (int k4 = 0; k4 < KC; k4 += kBatch * 128) {
                float xv[kRows * kBatch][4], vv[kRows * kBatch][4];
#pragma unroll
                for (int u = 0; u < kRows * kBatch; ++u) {
                    const int o = warp + 8 * (u / kBatch), kk = k4 + (u % kBatch) * 128 + 4 * lane;
#pragma unroll
                    for (int e = 0; e < 4; ++e) xv[u][e] = vv[u][e] = 0.f;
                    if (o < a.out && kk < KC && kb + kk < k1) {
                        load_vec4(xw + (int64_t)o * K + kb + kk, xv[u]);
                        if (has_v) load_vec4(vw + (int64_t)o * K + kb + kk, vv[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < kRows * kBatch; ++u) {
                    const int o = warp + 8 * (u / kBatch), kk = k4 + (u % kBatch) * 128 + 4 * lane;
                    if (o < OUT_T && kk < KC) {
                        float w4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            w4[e] = candidate_param<T>(xv[u][e], vv[u][e], a.gamma);
                            nrm = fmaf(vv[u][e], vv[u][e], nrm);
                        }
                        *reinterpret_cast<float4 *>(ws + o * KC + kk) = make_float4(w4[0], w4[1], w4[2], w4[3]);
                    }
                }
            }
        } else {
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const int o = warp + 8 * r;
                if (o >= OUT_T) break;
#pragma unroll 8
                for (int kk = lane; kk < KC; kk += 32) {
                    float xv = 0.f, vv = 0.f;
                    if (o < a.out && kb + kk < k1) {
                        xv = load_elem(xw + (int64_t)o * K + kb + kk);
                        if (has_v) vv = load_elem(vw + (int64_t)o * K + kb + kk);
                    }
                    ws[o * KC + kk] = candidate_param<T>(xv, vv, a.gamma);
                    nrm = fmaf(vv, vv, nrm);
                }
            }
        }
    };

    if (k0 < k1) stage_weights(k0);
    pdl_wait();
    pdl_launch_dependents();
    const float *hq[SPW];                        // this warp's samples; beyond the last one it again, its sums are dropped
#pragma unroll
    for (int q = 0; q < SPW; ++q) hq[q] = hin + (int64_t)min(warp * SPW + q, a.n_r - 1) * K;
    for (int kb = k0; kb < k1; kb += KC) {
        if (kb > k0) {
            __syncthreads();
            stage_weights(kb);
        }
        __syncthreads();
        if (warp * SPW < a.n_r) {
            const int len = min(KC, k1 - kb);
            // a lane's columns of 128: four neighbours (VEC), or every 32nd
            constexpr int kStep = VEC ? 1 : 32;
            const int at = VEC ? 4 * lane : lane;
            float h[kAhead][SPW][W];
            auto load = [&](int k, float (&to)[SPW][W]) {
#pragma unroll
                for (int q = 0; q < SPW; ++q) {
                    if constexpr (VEC) {
                        const float4 t = k + at < len ? __ldcg(reinterpret_cast<const float4 *>(hq[q] + kb + k + at)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        to[q][0] = t.x; to[q][1] = t.y; to[q][2] = t.z; to[q][3] = t.w;
                    } else {
#pragma unroll
                        for (int e = 0; e < W; ++e) to[q][e] = k + at + kStep * e < len ? __ldcg(hq[q] + kb + k + at + kStep * e) : 0.f;
                    }
                }
            };
#pragma unroll
            for (int d = 0; d < kAhead; ++d) load(128 * d, h[d]);
#pragma unroll 1
            for (int k = 0; k < len; k += 128 * kAhead) {
#pragma unroll
                for (int d = 0; d < kAhead; ++d) {
                    const int kd = k + 128 * d;
                    if (kd >= len) break;
#pragma unroll
                    for (int o = 0; o < OUT_T; ++o) {
                        float w[W];
                        if constexpr (VEC) {
                            const float4 t = *reinterpret_cast<const float4 *>(ws + o * KC + kd + at);
                            w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
                        } else {
#pragma unroll
                            for (int e = 0; e < W; ++e) w[e] = ws[o * KC + kd + at + kStep * e];
                        }
#pragma unroll
                        for (int q = 0; q < SPW; ++q)
#pragma unroll
                            for (int e = 0; e < W; ++e) acc[o][q] = fmaf(w[e], h[d][q][e], acc[o][q]);
                    }
                    load(kd + 128 * kAhead, h[d]);
                }
            }
        }
    }
    // the earlier layers' partial sums of v^2 of this candidate
    if (rank == 0 && has_v) {
        for (int l = 0; l + 1 < a.tail.used.layers; ++l) {
            const float *src = a.tail.normpart + (int64_t)(c - 1) * a.tail.np_slots + a.tail.used.base[l];
            const int count = a.tail.used.count[l];
            for (int t0 = threadIdx.x; t0 < count; t0 += 4 * 256) {
                float v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = t0 + u * 256 < count ? __ldcg(src + t0 + u * 256) : 0.f;
                nrm += (v[0] + v[1]) + (v[2] + v[3]);
            }
        }
    }

    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");     // every block runs: its shared memory may be written
    // lane totals, up to 32 (row, sample) pairs at a time; lane l receives pair l of the batch
    constexpr int kPairs = OUT_T * SPW, N = kPairs < 32 ? (kPairs <= 16 ? 16 : 32) : 32;
    if (warp * SPW < a.n_r) {
        const uint32_t dst = cluster_addr(zp + (size_t)rank * NS * OUT_T, 0);
#pragma unroll
        for (int e0 = 0; e0 < kPairs; e0 += N) {
            float v[N];
#pragma unroll
            for (int e = 0; e < N; ++e) v[e] = e0 + e < kPairs ? acc[e0 + e < kPairs ? (e0 + e) / SPW : 0][(e0 + e) % SPW] : 0.f;
            const float z = warp_transpose_reduce<N>(v, lane);
            const int e = e0 + lane, o = e / SPW, j = warp * SPW + e % SPW;
            if (lane < N && e < kPairs && o < a.out && j < a.n_r) cluster_store(dst + 4 * (j * OUT_T + o), z);
        }
    }
    nrm = warp_sum(nrm);
    if (lane == 0) cluster_store(cluster_addr(np + rank * 8 + warp, 0), nrm);
    cluster_barrier();
    if (rank != 0) return;
    // the samples' losses: a lane per class (logits and their differences in double: the score is a difference of losses that
    // agree in several digits)
    const double bias = a.offB >= 0 ? (double)candidate_param<T>(bias_x, bias_v, a.gamma) : 0.0;
#pragma unroll
    for (int q = 0; q < kLossTurns; ++q) {
        const int j = first_loss + kLossAt * q;
        if (j - (lane / kLossLanes) >= a.n_r) break;             // the whole warp's samples
        double z = 0.0;
        if (cls < a.out && j < a.n_r) {
            for (int r = 0; r < cluster; ++r) z += (double)zp[(r * NS + j) * OUT_T + cls];
            z += bias;
        }
        double zmax = cls < a.out ? z : -INFINITY;       // not rounded: a logit of 1e10 is 512 from its float
#pragma unroll
        for (int s = kLossLanes / 2; s >= 1; s >>= 1) zmax = fmax(zmax, __shfl_xor_sync(0xffffffffu, zmax, s));
        float se = cls < a.out ? expf((float)(z - zmax)) : 0.f;             // a NaN logit makes se NaN
#pragma unroll
        for (int s = kLossLanes / 2; s >= 1; s >>= 1) se += __shfl_xor_sync(0xffffffffu, se, s);
        int l = lab[q];
        if (l < 0 || l >= a.out) l = 0;
        const double zl = __shfl_sync(0xffffffffu, z, (lane & ~(kLossLanes - 1)) + l);
        if (cls == 0 && j < a.n_r) loss_s[j] = (zmax - zl) + (double)logf(se);
    }
    __syncthreads();
    if (warp == 0) {
        double l = 0.0;
        for (int j = lane; j < a.n_r; j += 32) l += loss_s[j];
        l = warp_sum(l);
        if (lane == 0) {
            a.tail.loss_sum[c] = l;
            a.losses[c] = (float)(l / (double)a.n_r);
        }
    } else if (warp == 1 && has_v) {
        float nv = 0.f;
        for (int t = lane; t < cluster * 8; t += 32) nv += np[t];
        nv = warp_sum(nv);
        if (lane == 0) a.tail.norm_tot[c - 1] = nv;
    }
    if (a.tail.defer) return;
    if (take_last_ticket(a.tail.ticket, gridDim.x / cluster)) finalize_and_select(a.tail);
}

// Per model: mean over the samples of log-sum-exp(z) - z[label].  G blocks per model (block g takes
// the samples j = g, g + G, ..), one warp per sample, fixed summation order: the blocks leave their
// sums in loss_part and the last block to finish adds them up, model by model, before it runs the
// tail.  G = 1 for small problems: the block writes the model's loss itself.
__global__ void __launch_bounds__(256) mlp_loss_kernel(const float *logits, const int32_t *labels,
                                                        int n_r, int classes, float *losses, double *loss_part,
                                                        int G, TailArgs tail) {
    __shared__ double per_warp[8];
    pdl_wait();
    pdl_launch_dependents();
    const int c = blockIdx.x / G, g = blockIdx.x - c * G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double mine = 0.0;
    for (int j = g + warp * G; j < n_r; j += 8 * G) {
        const float *z = logits + ((int64_t)c * n_r + j) * classes;
        float zmax = -INFINITY;
        for (int q = lane; q < classes; q += 32) zmax = fmaxf(zmax, z[q]);
#pragma unroll
        for (int s = 16; s >= 1; s >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, s));
        float se = 0.f;
        for (int q = lane; q < classes; q += 32) se += expf(z[q] - zmax);   // a NaN logit makes se NaN
        se = warp_sum(se);
        int lab = labels[j];
        if (lab < 0 || lab >= classes) lab = 0;
        mine += (double)((zmax - z[lab]) + logf(se));   // identical in every lane of the warp
    }
    if (lane == 0) per_warp[warp] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += per_warp[w];
        if (G == 1) {
            tail.loss_sum[c] = t;
            losses[c] = (float)(t / (double)n_r);
        } else {
            loss_part[blockIdx.x] = t;
        }
    }
    if (c > 0 && g == 0) block_norm_total(tail, c - 1);
    if (tail.defer) return;
    if (take_last_ticket(tail.ticket, gridDim.x)) {
        if (G > 1) {
            for (int i = threadIdx.x; i <= tail.m; i += blockDim.x) {
                double t = 0.0;
                for (int q = 0; q < G; ++q) t += __ldcg(loss_part + i * G + q);
                tail.loss_sum[i] = t;
                losses[i] = (float)(t / (double)n_r);
            }
            __threadfence();
            __syncthreads();
        }
        finalize_and_select(tail);
    }
}

// Blocks that share a tile's slices.  Two blocks fit an SM: with fewer than that, clusters, at least two slices a block
// (evening out a last wave with clusters as well made 190 tiles' kernel 10 % faster and its step 9 % slower).
int layer_cluster(const Context &c, int64_t tiles, int in) {
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    int cluster = 1;
    while (cluster < kMaxCluster && tiles * 2 * cluster <= 2 * sms && in >= 2 * kLK * 2 * cluster) cluster *= 2;
    return cluster;
}

// Samples in tiles of eight times this: one tile if it holds them all, else the width that pads them least (narrow layers, 33 to 48
// samples: two tiles of 24; a step of 21 models of 122-507-7-20-11 with 33 takes 39.5 us, with one tile of 64 52).
int layer_tile_width(int out, int n_r) {
    if (out <= kLFewRows) return n_r <= 8 ? 1 : n_r <= 16 ? 2 : n_r <= 32 ? 4 : n_r <= 48 ? 3 : 8;
    const bool by24 = n_r > 32 && (n_r + 23) / 24 <= (n_r + 31) / 32;
    return n_r <= 8 ? 1 : n_r <= 16 ? 2 : n_r <= 24 || by24 ? 3 : 4;
}

template <typename T, int R, int TN, bool VEC>
cudaError_t launch_layer_tiles(Context &c, const LayerArgs &a, cudaStream_t s) {
    const int sample_tiles = (a.n_r + 8 * TN - 1) / (8 * TN);
    const int64_t tiles = (int64_t)((a.out + 8 * R - 1) / (8 * R)) * sample_tiles;
    const int cluster = layer_cluster(c, tiles * (a.m + 1), a.in);
    // the limit is the function's, for every handle and thread of the process: the most any call asks for, set once
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(mlp_layer_kernel<T, R, TN, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)layer_smem(R, TN, kMaxCluster));
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    // the sample tiles of the same rows run side by side and find them in L2
    return launch_clustered(mlp_layer_kernel<T, R, TN, VEC>, cluster, dim3((unsigned)(tiles * cluster), a.m + 1), dim3(kLGroups * 64),
                            layer_smem(R, TN, cluster), s, chain_launches(c), a, sample_tiles, cluster);
}

template <typename T, bool VEC>
cudaError_t launch_layer(Context &c, const LayerArgs &a, cudaStream_t s) {
    const bool narrow = a.out <= kLFewRows;
    switch (layer_tile_width(a.out, a.n_r)) {
        case 1: return narrow ? launch_layer_tiles<T, 4, 1, VEC>(c, a, s) : launch_layer_tiles<T, 8, 1, VEC>(c, a, s);
        case 2: return narrow ? launch_layer_tiles<T, 4, 2, VEC>(c, a, s) : launch_layer_tiles<T, 8, 2, VEC>(c, a, s);
        case 3: return narrow ? launch_layer_tiles<T, 4, 3, VEC>(c, a, s) : launch_layer_tiles<T, 8, 3, VEC>(c, a, s);
        case 4: return narrow ? launch_layer_tiles<T, 4, 4, VEC>(c, a, s) : launch_layer_tiles<T, 8, 4, VEC>(c, a, s);
        default: return launch_layer_tiles<T, 4, 8, VEC>(c, a, s);
    }
}

}  // namespace

LayerTiles layer_tiles(const Context &c, int in, int out, int n_r, int m) {
    const int rows = out <= kLFewRows ? kLFewRows : 64, samples = 8 * layer_tile_width(out, n_r);
    const int64_t tiles = (int64_t)(m + 1) * ((out + rows - 1) / rows) * ((n_r + samples - 1) / samples);
    return {tiles, layer_cluster(c, tiles, in)};
}

// The cross-entropy can ride on the last layer's launch when one block sees all of a model's
// logits: every output row in one block, every sample in one tile.
bool mlp_can_fuse_loss(int out, int n_r) { return (out <= 32 && n_r <= 32) || (out <= 16 && n_r <= 64); }

template <typename T, int OUT_T, int SPW, bool VEC>
cudaError_t launch_head_sized(Context &c, const LayerArgs &a, cudaStream_t s) {
    constexpr int NS = 8 * SPW, kMostCols = head_rows_bytes(OUT_T, SPW, VEC) / 4 / OUT_T / 128 * 128;
    // blocks per model: as many as leave a slice of 128 columns and are resident at once (two to an SM up to 16 x 16
    // logits, one beyond: the accumulators).  A second wave costs more than the longer slice (101 models of 512 x 10,
    // 64 samples: 21 us with one block a model, 29 with two)
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    const int room = a.out <= 16 && a.n_r <= 16 ? 2 * sms : sms;
    int cluster = 1;                             // powers of two: clusters of seven leave a third of the SMs without one
    while (cluster < kMaxCluster && a.in / (2 * cluster) >= 128 && (a.m + 1) * 2 * cluster <= room) cluster *= 2;
    const int kslice = ((a.in + cluster - 1) / cluster + 3) / 4 * 4;
    const int turns = (kslice + kMostCols - 1) / kMostCols, KC = ((kslice + turns - 1) / turns + 127) / 128 * 128;
    auto smem = [](int cols, int blocks) { return sizeof(float) * ((size_t)OUT_T * cols + (size_t)blocks * (NS * OUT_T + 8)); };
    // the limit is the function's, for every handle and thread of the process: the most any call asks for, set once
    static PerDeviceOnce attr_set;
    if (attr_set.need(c.device)) {
        cudaError_t e = cudaFuncSetAttribute(mlp_head_kernel<T, OUT_T, SPW, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem(kMostCols, kMaxCluster));
        if (e != cudaSuccess) return e;
        attr_set.mark(c.device);
    }
    return launch_clustered(mlp_head_kernel<T, OUT_T, SPW, VEC>, cluster, dim3(cluster * (a.m + 1)), dim3(256), smem(KC, cluster), s,
                            chain_launches(c), a, cluster, kslice, KC);
}

template <typename T, bool VEC>
cudaError_t launch_head(Context &c, const LayerArgs &a, cudaStream_t s) {
    if (a.out <= 12) {
        if (a.n_r <= 8) return launch_head_sized<T, 12, 1, VEC>(c, a, s);
        if (a.n_r <= 16) return launch_head_sized<T, 12, 2, VEC>(c, a, s);
        if (a.n_r <= 32) return launch_head_sized<T, 12, 4, VEC>(c, a, s);
        return launch_head_sized<T, 12, 8, VEC>(c, a, s);
    }
    if (a.out <= 16) {
        if (a.n_r <= 8) return launch_head_sized<T, 16, 1, VEC>(c, a, s);
        if (a.n_r <= 16) return launch_head_sized<T, 16, 2, VEC>(c, a, s);
        if (a.n_r <= 32) return launch_head_sized<T, 16, 4, VEC>(c, a, s);
        return launch_head_sized<T, 16, 8, VEC>(c, a, s);
    }
    if (a.n_r <= 8) return launch_head_sized<T, 32, 1, VEC>(c, a, s);
    if (a.n_r <= 16) return launch_head_sized<T, 32, 2, VEC>(c, a, s);
    return launch_head_sized<T, 32, 4, VEC>(c, a, s);
}

cudaError_t launch_mlp_layer(Context &c, const LayerArgs &a, bool aligned, cudaStream_t s,
                             int *launches) {
    ++*launches;
    profile_mark(c, a.fuse_loss ? "mlp_head_loss_tail" : "mlp_layer", s);
    if (a.fuse_loss) {
        if (c.desc.param_dtype == ZENO_BF16)
            return aligned ? launch_head<__nv_bfloat16, true>(c, a, s) : launch_head<__nv_bfloat16, false>(c, a, s);
        return aligned ? launch_head<float, true>(c, a, s) : launch_head<float, false>(c, a, s);
    }
    if (layer_by_columns(c, a.in, a.out, a.n_r, a.m, aligned)) return launch_layer_by_columns(c, a, aligned, s);
    if (c.desc.param_dtype == ZENO_BF16)
        return aligned ? launch_layer<__nv_bfloat16, true>(c, a, s) : launch_layer<__nv_bfloat16, false>(c, a, s);
    return aligned ? launch_layer<float, true>(c, a, s) : launch_layer<float, false>(c, a, s);
}

// enough blocks to spread a large batch of wide logits over the SMs
int mlp_loss_groups(int n_r, int classes) {
    if ((int64_t)n_r * classes < 16384) return 1;
    return n_r >= 64 ? 8 : n_r >= 32 ? 4 : 2;
}

cudaError_t launch_mlp_loss(Context &c, const float *logits, const int32_t *labels, int n_r,
                            int m, int classes, float *losses, const TailArgs &tail, cudaStream_t s,
                            int *launches) {
    ++*launches;
    profile_mark(c, "mlp_loss_tail", s);
    const int G = mlp_loss_groups(n_r, classes);
    return launch_chained(mlp_loss_kernel, dim3((m + 1) * G), dim3(256), 0, s, chain_launches(c), logits, labels, n_r,
                          classes, losses, c.loss_part, G, tail);
}

}  // namespace zeno
