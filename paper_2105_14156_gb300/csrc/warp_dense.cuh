// Dense accumulator of one warp: the paper's "dense row" (values in an array
// indexed by column) for products whose B is narrow enough for a warp to own
// every column, shared by the batched kernel (k_batched.cu) and the narrow-B
// rows of the two phases (k_narrow.cu).
//
// A shared-memory float add has no native atomic on this GPU (a compare-and-swap
// loop: 3.4 op/clk/SM in float, 0.8 in double), but nobody else touches the warp's
// accumulator and few lanes of a step meet in a word: most rows simply add atomically,
// 32 products of any rows of B a step (dense_mode). In float, long rows of B, and shorter
// ones where copies cost nothing, take plain loads and stores: the columns inside one
// row of B are distinct, so the warp walks the rows of B that a row of A selects, W
// lanes to a row (W = 8, 16 or 32), each of the 32 / W lane groups with an accumulator
// copy of its own, and no two lanes of one step ever hit one word. That holds when
// every row of B ascends, which a pass over B's columns shows beforehand (descents_*,
// below; it checks their range too); else those products are added atomically as well,
// and checked one by one.
//
// Measured: 512 batched products of 256-column B (12.5 entries a row, float)
// 4.49 -> 1.63 ms a call and 24 of 3000 columns (double) 1.38 -> 0.33 ms,
// against a block's tables and accumulators with a lane's row found by search, and hash
// tables with a bitonic sort; the batched kernel now issues on 50 % of the cycles and
// waits for loads of B otherwise.
//
// Occupancy needs no bitmap: an unused word holds -0.0, which no sum of
// products reaches (a product that is -0.0 is added as +0.0, and a sum is -0.0
// only when both terms are) and which leaves no trace in a sum (-0.0 + x = x).
// The copies are added up, and their words returned to -0.0, while the row is
// written out in column order.
#pragma once

#include "device_common.cuh"

namespace smash {

// How a warp adds a row's products (mode). W lanes to a row of B with an
// accumulator copy per lane group: W by B's mean row length, the narrowest group
// that holds most rows in one step. Copies are cleared, added up and scanned with
// every row, and shared memory for them leaves fewer blocks resident, so they may
// take kDenseCopyBytes together; wider accumulators have one copy and take 32
// lanes a row of B from a mean of more than 16 entries on. Everything else adds
// atomically (kDenseFlat: 32 products of any rows of B a step), and so does double,
// where plain adds were nowhere faster.
// (Values of 40,000 rows times 1,024 columns in float, rows of A x rows of B: 18 x 4
// entries two copies 169 us, one with 32 lanes a row 134, flat 125; 25 x 12: 185, 144,
// 143; 59 x 20: 32 lanes 106, flat 116. Double, 512 columns, 74 x 4: 458, 433, 162.
// 256 columns in float, skewed graph of 50,021 rows: two copies 146 us, flat 170.)
// With rows for no more warps than one block an SM has, residency is no matter: the
// copies may take all of an accumulator's room (square of a skewed graph of 1,024
// rows, whose crowded columns make atomic adds wait: 79 us, flat 84).
enum : int { kDenseFlat = 0, kDenseW8 = 1, kDenseW16 = 2, kDenseW32 = 3 };
__host__ __device__ constexpr int dense_copies(int mode) { return mode == kDenseW8 ? 4 : mode == kDenseW16 ? 2 : 1; }
// Words of one accumulator copy.
__host__ __device__ constexpr int dense_stride(int ncols) { return (ncols + 31) & ~31; }
// Most bytes a warp's accumulator may take (eight warps of a block: 192 KB), and
// most that several copies may take.
constexpr int kDenseWarpBytes = 24 * 1024;
constexpr int kDenseCopyBytes = 2 * 1024;

// entries: of `rows` rows of B (all, or each as often as a product reads it). few:
// one block an SM has a warp for every row of the product.
__host__ __device__ inline int dense_mode(int64_t entries, int64_t rows, int ncols, int vsz, bool few) {
    if (vsz == 8 || entries < 3 * rows) return kDenseFlat;
    int m = entries <= 8 * rows ? kDenseW8 : entries <= 16 * rows ? kDenseW16 : kDenseW32;
    const int64_t copy = (int64_t)dense_stride(ncols) * vsz;
    if (!few) return dense_copies(m) == 1 || dense_copies(m) * copy <= kDenseCopyBytes ? m : kDenseFlat;
    while (dense_copies(m) > 1 && dense_copies(m) * copy > kDenseWarpBytes) ++m;
    return m;
}
__host__ __device__ inline size_t dense_warp_bytes(int mode, int ncols, int vsz) {
    return (size_t)dense_copies(mode) * dense_stride(ncols) * vsz;
}

__device__ __forceinline__ float dense_unused(float) { return __int_as_float((int)0x80000000); }
__device__ __forceinline__ double dense_unused(double) { return __hiloint2double((int)0x80000000, 0); }
__device__ __forceinline__ bool dense_used(float v) { return __float_as_uint(v) != 0x80000000u; }
__device__ __forceinline__ bool dense_used(double v) {
    return __double2hiint(v) != (int)0x80000000 || __double2loint(v) != 0;
}
// a * b, +0.0 for -0.0 (in double by the bits: a double add costs a warp 16
// cycles of the FP64 pipe).
__device__ __forceinline__ float dense_product(float a, float b) { return __fadd_rn(__fmul_rn(a, b), 0.f); }
__device__ __forceinline__ double dense_product(double a, double b) {
    const double p = __dmul_rn(a, b);
    return dense_used(p) ? p : 0.0;
}

template <typename V>
__device__ __forceinline__ void dense_clear(V *acc, int words) {
    for (int j = lane_id(); j < words; j += 32) acc[j] = dense_unused(V(0));
}

constexpr int kDenseUnroll = 4;   // steps whose loads of B are issued together

// Every product of the A entries in batches of 32 that start at first, first +
// step, ... below ae, with W lanes to a row of B: f(group, act, j, a, b) is
// called by all 32 lanes together once per step (act: the lane holds a product
// of its lane group's row; a, b: 0 when !NUM). Rows of up to 2 W entries take
// one or two steps of their lane group (the second steps of a batch packed
// together), longer ones all lanes as group 0. Columns are not checked.
template <typename V, int W, bool NUM, typename F>
__device__ __forceinline__ void dense_rows(const Operands<V> &op, int64_t first, int64_t ae, int64_t step, int *err,
                                           F &&f) {
    constexpr int S = 32 / W;
    const int lane = lane_id();
    const int sub = lane / W, sl = lane & (W - 1);
    for (int64_t base = first; base < ae; base += step) {
        int len = 0;
        int64_t bs = 0;
        V av = V(0);
        if (base + lane < ae) load_a_entry<V, NUM>(op, base + lane, len, bs, av, err);
        const int n = (int)(ae - base < 32 ? ae - base : 32);
        const int own = len > 2 * W ? 0 : len;   // entries added by the lane group
        for (int e = 0; e < n; e += S * kDenseUnroll) {
            int jv[kDenseUnroll];
            bool act[kDenseUnroll];
            V au[kDenseUnroll], bv[kDenseUnroll];
#pragma unroll
            for (int u = 0; u < kDenseUnroll; ++u) {
                const int src = e + u * S + sub;   // at most 31: n <= 32 and S * kDenseUnroll divides 32
                const int64_t st = __shfl_sync(kFull, bs, src) + sl;
                const int l = __shfl_sync(kFull, own, src);
                act[u] = sl < l;
                au[u] = V(0);
                bv[u] = V(0);
                if constexpr (NUM) au[u] = __shfl_sync(kFull, av, src);
                jv[u] = 0;
                if (act[u]) {
                    jv[u] = __ldg(op.b_ci + st);
                    if constexpr (NUM) bv[u] = __ldg(op.b_val + st);
                }
            }
#pragma unroll
            for (int u = 0; u < kDenseUnroll; ++u)
                if (u == 0 || e + u * S < n) f(sub, act[u], jv[u], au[u], bv[u]);
        }
        // second steps: the rows left over, S at a time
        for (unsigned todo = __ballot_sync(kFull, own > W); todo;) {
            int src = 0;
            bool have = false;
#pragma unroll
            for (int x = 0; x < S; ++x) {
                if (x == sub && todo) {
                    src = __ffs(todo) - 1;
                    have = true;
                }
                todo &= todo - 1;
            }
            __syncwarp();
            const int64_t st = __shfl_sync(kFull, bs, src) + W + sl;
            const int l = __shfl_sync(kFull, own, src);
            V a = V(0), b = V(0);
            if constexpr (NUM) a = __shfl_sync(kFull, av, src);
            const bool act = have && W + sl < l;
            int j = 0;
            if (act) {
                j = __ldg(op.b_ci + st);
                if constexpr (NUM) b = __ldg(op.b_val + st);
            }
            f(sub, act, j, a, b);
        }
        // long rows of B, all lanes: 32 entries of one row a step, the steps of
        // consecutive rows in flight together
        unsigned todo = __ballot_sync(kFull, len > 2 * W);
        int src = __ffs(todo) - 1, o = 0;
        while (src >= 0) {
            int jv[kDenseUnroll];
            bool act[kDenseUnroll];
            V au[kDenseUnroll], bv[kDenseUnroll];
#pragma unroll
            for (int u = 0; u < kDenseUnroll; ++u) {
                act[u] = false;
                jv[u] = 0;
                au[u] = V(0);
                bv[u] = V(0);
                if (src >= 0) {   // the same for all lanes
                    const int64_t st = __shfl_sync(kFull, bs, src) + o + lane;
                    const int l = __shfl_sync(kFull, len, src);
                    if constexpr (NUM) au[u] = __shfl_sync(kFull, av, src);
                    act[u] = o + lane < l;
                    if (act[u]) {
                        jv[u] = __ldg(op.b_ci + st);
                        if constexpr (NUM) bv[u] = __ldg(op.b_val + st);
                    }
                    o += 32;
                    if (o >= l) {
                        todo &= todo - 1;
                        src = __ffs(todo) - 1;
                        o = 0;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kDenseUnroll; ++u) f(0, act[u], jv[u], au[u], bv[u]);
        }
    }
}

// Adds the products to the warp's accumulator copies (ascend: every row of B
// ascends below op.ncols). All 32 lanes call it.
template <typename V>
__device__ __forceinline__ void dense_accumulate(const Operands<V> &op, int mode, bool ascend, int64_t first,
                                                 int64_t ae, int64_t step, V *acc, int *err) {
    const int stride = dense_stride(op.ncols);
    if (!ascend || sizeof(V) == 8) mode = kDenseFlat;
    // (the barrier orders a step before the next one's loads of the same words)
    auto add = [&](int group, bool act, int j, V a, V b) {
        if (act) acc[group * stride + j] += dense_product(a, b);
        __syncwarp();
    };
    if (mode == kDenseW8) {
        dense_rows<V, 8, true>(op, first, ae, step, err, add);
    } else if (mode == kDenseW16) {
        dense_rows<V, 16, true>(op, first, ae, step, err, add);
    } else if (mode == kDenseW32) {
        dense_rows<V, 32, true>(op, first, ae, step, err, add);
    } else {
        for (int64_t base = first; base < ae; base += step)
            warp_products<V, true>(op, base, ae - base < 32 ? ae : base + 32, err, [&](int j, V a, V b) {
                atomicAdd(acc + j, dense_product(a, b));
            });
    }
    __syncwarp();
}

// The accumulator's entries in column order: f(place, column, value), and
// every word back to -0.0. Returns the number of entries.
template <typename V, typename F>
__device__ __forceinline__ int dense_emit(V *acc, int mode, int ncols, F &&f) {
    const int lane = lane_id();
    const int stride = dense_stride(ncols), copies = dense_copies(mode);
    int run = 0;
    for (int j0 = lane; j0 < stride; j0 += 32 * kDenseUnroll) {
        V v[kDenseUnroll];
#pragma unroll
        for (int u = 0; u < kDenseUnroll; ++u) {
            const int j = j0 + 32 * u;
            v[u] = dense_unused(V(0));
            if (j < stride) {
                v[u] = acc[j];
                acc[j] = dense_unused(V(0));
                for (int s = 1; s < copies; ++s) {
                    v[u] += acc[s * stride + j];
                    acc[s * stride + j] = dense_unused(V(0));
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kDenseUnroll; ++u) {
            const bool used = dense_used(v[u]);
            const unsigned m = __ballot_sync(kFull, used);
            if (used) f(run + __popc(m & lanemask_lt()), j0 + 32 * u, v[u]);
            run += __popc(m);
        }
    }
    __syncwarp();
    return run;
}

// Whether every row of B ascends below cols(B), from two coalesced passes: the
// places e of the whole column array with col[e - 1] >= col[e]
// (descents_between, over any split of the entries), less those of them where a
// non-empty row starts (descents_at_starts, over any split of the rows), are
// none. A column outside [0, ncols), or a row of B that does not end at or after
// its start (two others may then start at one place), rules it out: `bad`.
__device__ __forceinline__ long long descents_between(const int32_t *ci, int64_t e0, int64_t e1, int ncols, int t,
                                                      int nt, bool &bad) {
    long long d = 0;
    for (int64_t e = e0 + t; e < e1; e += nt) {
        const int j = __ldg(ci + e);
        if (e > 0 && __ldg(ci + e - 1) >= j) ++d;
        if ((unsigned)j >= (unsigned)ncols) bad = true;
    }
    return d;
}
__device__ __forceinline__ long long descents_at_starts(const int64_t *rp, const int32_t *ci, int64_t nnz, int64_t r0,
                                                        int64_t r1, int t, int nt, bool &bad) {
    long long d = 0;
    for (int64_t r = r0 + t; r < r1; r += nt) {
        const int64_t s = __ldg(rp + r), e = __ldg(rp + r + 1);
        if (s < 0 || e < s || e > nnz) bad = true;
        else if (s > 0 && e > s && __ldg(ci + s - 1) >= __ldg(ci + s)) ++d;
    }
    return d;
}
// A warp's share of both added to a word that is 0 when B ascends: twice the
// places, and the lowest bit for `bad` (an even number of any sign never clears
// it, however many there are).
__device__ __forceinline__ void descents_add(unsigned long long *word, long long d, bool bad) {
    d = warp_sum(d);
    bad = __any_sync(kFull, bad);
    if (lane_id() == 0) {
        if (d) atomicAdd(word, (unsigned long long)(2 * d));
        if (bad) atomicOr(word, 1ull);
    }
}

}  // namespace smash
