// The marginal Median (Experiments, "Baselines"): out[j] = the one-dimensional median of column j, the middle
// value of the m sorted entries, the mean of the two middle ones for even m; a NaN entry counts as plus
// infinity.  One pass over V.
//
// Up to 128 candidates one thread holds a whole column in registers as two halves of H values, sorts each
// half by an odd-even merge network whose indices are constants, and takes the middle of the two sorted
// halves without merging them: of two ascending lists a and b of H values the H smallest are
// min(a[i], b[H - 1 - i]), so the value of rank H - 1 is the largest of those and the value of rank H the
// smallest of max(a[i], b[H - 1 - i]).  A column of fewer than 2 H values is padded with equally many minus
// and plus infinities (one more plus infinity when the number is odd), which leaves the middle where it is.
// Up to 12 candidates, where the loads are what it waits for, bfloat16 columns go two to a thread, compared in pairs by
// the packed minimum and maximum (1.8 M columns of 5: 8.3 us against 10.8 with one); beyond, the packed comparisons are
// the slower ones (100: 717 us against 232, and 19.0 against 6.5 for 7,960 columns, which then fill half as many SMs).
//
// Beyond 128 candidates 8, 16 or 32 neighbouring lanes of a warp share a column, 32 values each, sorted by a
// bitonic network whose long-range stages exchange values by shuffles.
#include <math.h>

#include "zeno_internal.h"

namespace zeno {

namespace {

constexpr int kMedianThreads = 128;
constexpr int kMedianMaxHalf = 64;            // values in each half of a column one thread holds
constexpr int kMedianTwoColsHalf = 6;         // bfloat16: halves up to which a thread takes two columns

__host__ __device__ constexpr int ilog2(int v) { return v <= 1 ? 0 : 1 + ilog2(v >> 1); }

// What a register of the one-thread kernel holds: one column in binary32, or two bfloat16 columns.
template <typename T>
struct OneCol {
    using Elem = T;
    using Reg = float;
    static constexpr int kCols = 1;
    static __device__ __forceinline__ Reg load(const T *p, bool, bool) { return load_elem(p); }
    static __device__ __forceinline__ Reg all(float v) { return v; }
    static __device__ __forceinline__ Reg min(Reg a, Reg b) { return fminf(a, b); }
    static __device__ __forceinline__ Reg max(Reg a, Reg b) { return fmaxf(a, b); }
    // s stays zero while every value seen is finite
    static __device__ __forceinline__ Reg probe(Reg v, Reg s) { return fmaf(v, 0.f, s); }
    static __device__ __forceinline__ bool all_finite(Reg s) { return s == 0.f; }
    static __device__ __forceinline__ Reg clean(Reg v) { return nan_to_inf(v); }
    static __device__ __forceinline__ void store(float *out, Reg lo, Reg hi, bool odd, bool) {
        *out = odd ? lo : 0.5f * lo + 0.5f * hi;
    }
};
struct TwoCols {
    using Elem = __nv_bfloat16;
    using Reg = __nv_bfloat162;
    static constexpr int kCols = 2;
    // whole: both columns exist and their four bytes may be read at once
    static __device__ __forceinline__ Reg load(const __nv_bfloat16 *p, bool whole, bool second) {
        uint32_t u;
        if (whole) {
            u = __ldg(reinterpret_cast<const uint32_t *>(p));
        } else {
            const unsigned short *q = reinterpret_cast<const unsigned short *>(p);
            u = __ldg(q) | (second ? (uint32_t)__ldg(q + 1) << 16 : 0u);
        }
        return *reinterpret_cast<Reg *>(&u);
    }
    static __device__ __forceinline__ Reg all(float v) { return __float2bfloat162_rn(v); }
    static __device__ __forceinline__ Reg min(Reg a, Reg b) { return __hmin2(a, b); }
    static __device__ __forceinline__ Reg max(Reg a, Reg b) { return __hmax2(a, b); }
    static __device__ __forceinline__ Reg probe(Reg v, Reg s) { return __hfma2(v, all(0.f), s); }
    static __device__ __forceinline__ bool all_finite(Reg s) { return __low2float(s) == 0.f && __high2float(s) == 0.f; }
    static __device__ __forceinline__ Reg clean(Reg v) {
        return __floats2bfloat162_rn(nan_to_inf(__low2float(v)), nan_to_inf(__high2float(v)));
    }
    static __device__ __forceinline__ void store(float *out, Reg lo, Reg hi, bool odd, bool second) {
        out[0] = odd ? __low2float(lo) : 0.5f * __low2float(lo) + 0.5f * __low2float(hi);
        if (second) out[1] = odd ? __high2float(lo) : 0.5f * __high2float(lo) + 0.5f * __high2float(hi);
    }
};

// Ascending sort of n values held in registers: Batcher's odd-even merge sort.  A merge of sorted runs of p
// values compares, for k = p, p / 2, .. 1, the values k apart that belong to the same pair of runs; elements
// from n on would be plus infinity and never move, so their comparators are left out.
template <typename C, int n>
__device__ __forceinline__ void sort_registers(typename C::Reg (&a)[n]) {
    constexpr int kLog = n <= 1 ? 0 : ilog2(n - 1) + 1;
#pragma unroll
    for (int lp = 0; lp < kLog; ++lp) {
        const int p = 1 << lp;
#pragma unroll
        for (int lk = lp; lk >= 0; --lk) {
            const int k = 1 << lk, first = lk == lp ? 0 : k;
#pragma unroll
            for (int i = 0; i < n; ++i) {
                const bool compared = i >= first && ((i - first) & (2 * k - 1)) < k && i / (2 * p) == (i + k) / (2 * p);
                if (compared && i + k < n) {
                    const typename C::Reg lo = C::min(a[i], a[i + k]), hi = C::max(a[i], a[i + k]);
                    a[i] = lo;
                    a[i + k] = hi;
                }
            }
        }
    }
}

// Blocks that stay resident with the registers a half of H values needs.
__host__ __device__ constexpr int median_blocks_per_sm(int H) {
    const int b = 65536 / (kMedianThreads * (2 * H + 36));
    return b > 8 ? 8 : b;
}

// m candidates, 2 H - 8 < m <= 2 H.  A block takes kMedianThreads registers' worth of columns at a time; the
// rows' addresses are the same for the whole block and are added to the thread's own offset.
// Bound by the comparisons: minimum and maximum issue at half the rate of an addition, so a column of 100
// costs about 1,700 half-rate instructions where reading it costs 100 loads.  100 x 1.8 M binary32 values take
// 241 us (114 us of memory time); the whole column sorted over four lanes with shuffles took 934 us.
template <typename C, int H>
__global__ void __launch_bounds__(kMedianThreads, median_blocks_per_sm(H))
median_select_kernel(const typename C::Elem *V, int64_t ldv, int64_t d, int m, int pairs, float *out) {
    using T = typename C::Elem;
    using Reg = typename C::Reg;
    constexpr int kTile = kMedianThreads * C::kCols;
    constexpr int kSlack = H <= 16 ? 1 : 7;       // most padding values
    pdl_wait();
    pdl_launch_dependents();
    const int low_pad = (2 * H - m) / 2;
    for (int64_t j0 = (int64_t)blockIdx.x * kTile; j0 < d; j0 += (int64_t)gridDim.x * kTile) {
        const int64_t left = d - j0;              // columns from here on
        int off = threadIdx.x * C::kCols;
        const bool live = off < left, second = off + 1 < left;
        if (!live) off = 0;                       // computed on the tile's first column and dropped
        const bool whole = pairs && (live ? second : left > 1);
        const T *base = V + j0;
        Reg a[H], b[H], s = C::all(0.f);
#pragma unroll
        for (int i = 0; i < 2 * H; ++i) {
            Reg v;
            if (i < 2 * H - kSlack || i < m) {
                v = C::load(base + (int64_t)i * ldv + off, whole, second);
                s = C::probe(v, s);
            } else {
                v = C::all(i - m < low_pad ? -INFINITY : INFINITY);
            }
            if (i < H) a[i] = v; else b[i - H] = v;
        }
        if (!C::all_finite(s)) {                  // an infinity or a NaN among them: NaN becomes plus infinity
#pragma unroll
            for (int i = 0; i < H; ++i) {
                a[i] = C::clean(a[i]);
                b[i] = C::clean(b[i]);
            }
        }
        sort_registers<C, H>(a);
        sort_registers<C, H>(b);
        Reg lo = C::min(a[0], b[H - 1]), hi = C::max(a[0], b[H - 1]);
#pragma unroll
        for (int i = 1; i < H; ++i) {
            lo = C::max(lo, C::min(a[i], b[H - 1 - i]));
            hi = C::min(hi, C::max(a[i], b[H - 1 - i]));
        }
        if (live) C::store(out + j0 + off, lo, hi, m & 1, second);
    }
}

// ---- more than 128 candidates -----------------------------------------------------------------

constexpr int kMedianRegs = 32;               // values of a column one lane holds

// Ascending sort of the R * TPC values that TPC neighbouring lanes hold, element e = t * R + i in
// register i of lane t, by the bitonic network in the form whose comparators all point the same way: a
// merge of blocks of k elements first compares every element with its mirror image in the block
// (e ^ (k - 1)), then halves the distance from k / 4 down.  Every index below is a constant once the
// loops are unrolled, so the values stay in registers; partners R or more elements away sit in another
// lane and come by shuffle.
template <int R, int TPC>
__device__ __forceinline__ void bitonic_sort_lanes(float (&a)[R], int t) {
    constexpr int kLogN = ilog2(R) + ilog2(TPC);
#pragma unroll
    for (int lk = 1; lk <= kLogN; ++lk) {
        const int k = 1 << lk;
        if (k > R) {                          // mirror partner: register R - 1 - i of lane t ^ (k / R - 1)
            const bool keep_min = (t & (k / (2 * R))) == 0;
            float o[R];
#pragma unroll
            for (int i = 0; i < R; ++i) o[i] = __shfl_xor_sync(0xffffffffu, a[R - 1 - i], k / R - 1);
#pragma unroll
            for (int i = 0; i < R; ++i) a[i] = keep_min ? fminf(a[i], o[i]) : fmaxf(a[i], o[i]);
        } else {
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const int l = i ^ (k - 1);
                if (l > i) {
                    const float lo = fminf(a[i], a[l]), hi = fmaxf(a[i], a[l]);
                    a[i] = lo;
                    a[l] = hi;
                }
            }
        }
#pragma unroll
        for (int lj = lk - 2; lj >= 0; --lj) {
            const int j = 1 << lj;
            if (j >= R) {
                const bool keep_min = (t & (j / R)) == 0;
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const float o = __shfl_xor_sync(0xffffffffu, a[i], j / R);
                    a[i] = keep_min ? fminf(a[i], o) : fmaxf(a[i], o);
                }
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int l = i ^ j;
                    if (l > i) {
                        const float lo = fminf(a[i], a[l]), hi = fmaxf(a[i], a[l]);
                        a[i] = lo;
                        a[l] = hi;
                    }
                }
            }
        }
    }
}

// A warp takes 32 / TPC neighbouring columns at a time; lane = column * TPC + t holds rows t * R .. of it,
// padded with plus infinity, which leaves the middle ranks where they are.
template <typename T, int TPC>
__global__ void __launch_bounds__(kMedianThreads, 4) median_lanes_kernel(const T *V, int64_t ldv, int64_t d, int m, float *out) {
    constexpr int R = kMedianRegs, kCols = 32 / TPC;
    pdl_wait();
    pdl_launch_dependents();
    const int lane = threadIdx.x & 31, t = lane % TPC, c = lane / TPC;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int p0 = (m - 1) / 2, p1 = m / 2;   // ranks of the middle values
    for (int64_t j0 = warp * kCols; j0 < d; j0 += warps * kCols) {
        const int64_t j = j0 + c;
        const bool live = j < d;
        float a[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int row = t * R + i;
            a[i] = (live && row < m) ? nan_to_inf(load_elem(V + (int64_t)row * ldv + j)) : INFINITY;
        }
        bitonic_sort_lanes<R, TPC>(a, t);
        float lo = 0.f, hi = 0.f;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            if (t * R + i == p0) lo = a[i];
            if (t * R + i == p1) hi = a[i];
        }
        lo = __shfl_sync(0xffffffffu, lo, (lane & ~(TPC - 1)) | (p0 / R));
        hi = __shfl_sync(0xffffffffu, hi, (lane & ~(TPC - 1)) | (p1 / R));
        if (live && t == 0) out[j] = (m & 1) ? lo : 0.5f * lo + 0.5f * hi;
    }
}

template <typename T, int TPC>
cudaError_t launch_lanes(Context &c, const T *V, int64_t ldv, int m, float *out, cudaStream_t s) {
    const int sms = c.sm_count > 0 ? c.sm_count : 148;
    const int64_t d = c.d;
    const int per_block = (kMedianThreads / 32) * (32 / TPC);          // columns a block takes at a time
    const int64_t want = (d + per_block - 1) / per_block, cap = (int64_t)sms * 16;
    const int blocks = (int)(want < cap ? (want < 1 ? 1 : want) : cap);
    return launch_chained(median_lanes_kernel<T, TPC>, dim3(blocks), dim3(kMedianThreads), 0, s, chain_launches(c), V, ldv, d, m, out);
}

// the one-thread kernel whose halves hold just m values: every H up to 16, then steps of four (a finer step
// would save at most 6 % of the comparisons and quadruple the kernels)
template <typename C, int H>
struct MedianSelect {
    using T = typename C::Elem;
    static cudaError_t launch(Context &c, const T *V, int64_t ldv, int m, float *out, cudaStream_t s) {
        constexpr int kSmaller = H > 16 ? H - 4 : H - 1;
        if (m <= 2 * kSmaller) return MedianSelect<C, kSmaller>::launch(c, V, ldv, m, out, s);
        const int sms = c.sm_count > 0 ? c.sm_count : 148;
        const int64_t d = c.d, tile = kMedianThreads * C::kCols;
        const int64_t want = (d + tile - 1) / tile, cap = (int64_t)sms * median_blocks_per_sm(H) * 8;
        const int blocks = (int)(want < cap ? want : cap);
        const int pairs = ldv % 2 == 0 && reinterpret_cast<uintptr_t>(V) % 4 == 0;
        return launch_chained(median_select_kernel<C, H>, dim3(blocks), dim3(kMedianThreads), 0, s, chain_launches(c), V, ldv, d, m,
                              pairs, out);
    }
};
template <typename C>
struct MedianSelect<C, 0> {
    static cudaError_t launch(Context &, const typename C::Elem *, int64_t, int, float *, cudaStream_t) { return cudaErrorInvalidValue; }
};

cudaError_t launch_select(Context &c, const float *V, int64_t ldv, int m, float *out, cudaStream_t s) {
    return MedianSelect<OneCol<float>, kMedianMaxHalf>::launch(c, V, ldv, m, out, s);
}
cudaError_t launch_select(Context &c, const __nv_bfloat16 *V, int64_t ldv, int m, float *out, cudaStream_t s) {
    if (m <= 2 * kMedianTwoColsHalf) return MedianSelect<TwoCols, kMedianTwoColsHalf>::launch(c, V, ldv, m, out, s);
    return MedianSelect<OneCol<__nv_bfloat16>, kMedianMaxHalf>::launch(c, V, ldv, m, out, s);
}

template <typename T>
cudaError_t launch_typed(Context &c, const T *V, int64_t ldv, int m, float *out, cudaStream_t s) {
    static_assert(kMedianRegs * 32 >= ZENO_MAX_CANDIDATES, "a warp holds the longest column");
    if (m <= 2 * kMedianMaxHalf) return launch_select(c, V, ldv, m, out, s);
    if (m <= kMedianRegs * 8) return launch_lanes<T, 8>(c, V, ldv, m, out, s);
    if (m <= kMedianRegs * 16) return launch_lanes<T, 16>(c, V, ldv, m, out, s);
    return launch_lanes<T, 32>(c, V, ldv, m, out, s);
}

}  // namespace

cudaError_t launch_median(Context &c, const void *V, int64_t ldv, int m, float *out, cudaStream_t s, int *launches) {
    ++*launches;
    profile_mark(c, "median", s);
    if (c.desc.param_dtype == ZENO_BF16) return launch_typed(c, static_cast<const __nv_bfloat16 *>(V), ldv, m, out, s);
    return launch_typed(c, static_cast<const float *>(V), ldv, m, out, s);
}

}  // namespace zeno
