// Dense accumulator of one warp: the paper's "dense row" (values in an array
// indexed by column) for products whose B is narrow enough for a warp to own
// every column, shared by the batched kernel (k_batched.cu) and the narrow-B
// rows of the two phases (k_narrow.cu).
//
// The shared-memory float add has no native atomic on this GPU (a
// compare-and-swap loop: 3.4 op/clk/SM in float, 0.8 in double), so the
// products are added with plain loads and stores. Nobody else touches the
// warp's accumulator, and the columns inside one row of B are distinct: the
// warp walks the rows of B that a row of A selects, W lanes to a row of B
// (W = 8, 16 or 32, by B's mean row length), each of the 32 / W lane groups
// with an accumulator copy of its own, so no two lanes of one step ever hit
// one word. That holds when every row of B ascends, which a pass over B's
// columns shows beforehand (descents_*, below; it checks their range too); for
// any other B the products are added atomically and checked one by one.
//
// Measured: 512 batched products of 256-column B (12.5 entries a row, float)
// 4.48 -> 1.69 ms a call and 24 of 3000 columns (double) 1.41 -> 0.38 ms,
// against atomic adds with a lane's row found by search, and hash tables with a
// bitonic sort; the batched kernel now issues on 55 % of the cycles and waits
// for loads of B otherwise.
//
// Occupancy needs no bitmap: an unused word holds -0.0, which no sum of
// products reaches (a product is formed as a * b + 0.0, and a sum that rounds
// to zero is +0.0 unless both terms are -0.0), and which adding leaves no
// trace (-0.0 + x = x). The copies are added up, and their words returned to
// -0.0, while the row is written out in column order.
#pragma once

#include "device_common.cuh"

namespace smash {

// Lane groups by B's mean row length: the narrowest group that holds most
// rows in one step keeps the most lanes busy; below 3 entries a row even eight
// lanes would mostly idle, and 32 products of many rows share a step instead
// (kDenseFlat, atomic adds). Copies that would not fit the accumulator's room
// take wider groups.
enum : int { kDenseFlat = 0, kDenseW8 = 1, kDenseW16 = 2, kDenseW32 = 3 };
__host__ __device__ constexpr int dense_copies(int mode) { return mode == kDenseW8 ? 4 : mode == kDenseW16 ? 2 : 1; }
// Words of one accumulator copy.
__host__ __device__ constexpr int dense_stride(int ncols) { return (ncols + 31) & ~31; }
// Most bytes a warp's accumulator may take (eight warps of a block: 192 KB).
constexpr int kDenseWarpBytes = 24 * 1024;

__host__ __device__ inline int dense_mode(int64_t b_nnz, int64_t b_rows, int ncols, int vsz) {
    int m = b_nnz < 3 * b_rows ? kDenseFlat : b_nnz <= 8 * b_rows ? kDenseW8 : b_nnz <= 16 * b_rows ? kDenseW16
                                                                                                       : kDenseW32;
    while (dense_copies(m) > 1 && (int64_t)dense_copies(m) * dense_stride(ncols) * vsz > kDenseWarpBytes) ++m;
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

// One step of W lanes per row of B: every active lane adds a * b to column j
// of its group's copy. (The barrier orders the step before the next one's
// loads of the same words.)
template <typename V>
__device__ __forceinline__ void dense_step(V *mine, bool act, int j, V a, V b) {
    if (act) mine[j] += dense_product(a, b);
    __syncwarp();
}

// Adds the products of A entries in batches of 32 that start at first, first
// + step, ... below ae, with W lanes to a row of B (ascending columns below
// op.ncols). Rows of up to 2 W entries take one or two steps of their lane
// group (the second steps of a batch packed together), longer ones all lanes.
template <typename V, int W>
__device__ __forceinline__ void dense_rows(const Operands<V> &op, int64_t first, int64_t ae, int64_t step, V *acc,
                                           int stride, int *err) {
    constexpr int S = 32 / W;
    const int lane = lane_id();
    const int sub = lane / W, sl = lane & (W - 1);
    V *mine = acc + sub * stride;
    for (int64_t base = first; base < ae; base += step) {
        int len = 0;
        int64_t bs = 0;
        V av = V(0);
        if (base + lane < ae) load_a_entry<V, true>(op, base + lane, len, bs, av, err);
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
                act[u] = sl < __shfl_sync(kFull, own, src);
                au[u] = __shfl_sync(kFull, av, src);
                jv[u] = 0;
                bv[u] = V(0);
                if (act[u]) {
                    jv[u] = __ldg(op.b_ci + st);
                    bv[u] = __ldg(op.b_val + st);
                }
            }
#pragma unroll
            for (int u = 0; u < kDenseUnroll; ++u)
                if (u == 0 || e + u * S < n) dense_step<V>(mine, act[u], jv[u], au[u], bv[u]);
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
            const V a = __shfl_sync(kFull, av, src);
            const bool act = have && W + sl < l;
            int j = 0;
            V b = V(0);
            if (act) {
                j = __ldg(op.b_ci + st);
                b = __ldg(op.b_val + st);
            }
            dense_step<V>(mine, act, j, a, b);
        }
        // long rows of B, all lanes on the first copy
        for (unsigned todo = __ballot_sync(kFull, len > 2 * W); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int64_t st = __shfl_sync(kFull, bs, src) + lane;
            const int l = __shfl_sync(kFull, len, src);
            const V a = __shfl_sync(kFull, av, src);
            for (int o = 0; o < l; o += 32 * kDenseUnroll) {
                int jv[kDenseUnroll];
                V bv[kDenseUnroll];
#pragma unroll
                for (int u = 0; u < kDenseUnroll; ++u) {
                    jv[u] = 0;
                    bv[u] = V(0);
                    if (o + 32 * u + lane < l) {
                        jv[u] = __ldg(op.b_ci + st + o + 32 * u);
                        bv[u] = __ldg(op.b_val + st + o + 32 * u);
                    }
                }
#pragma unroll
                for (int u = 0; u < kDenseUnroll; ++u) dense_step<V>(acc, o + 32 * u + lane < l, jv[u], a, bv[u]);
            }
        }
    }
}

// The same by mode (ascend: every row of B ascends below op.ncols). All 32
// lanes call it.
template <typename V>
__device__ __forceinline__ void dense_accumulate(const Operands<V> &op, int mode, bool ascend, int64_t first,
                                                 int64_t ae, int64_t step, V *acc, int *err) {
    const int stride = dense_stride(op.ncols);
    if (!ascend) mode = kDenseFlat;
    if (mode == kDenseW8) {
        dense_rows<V, 8>(op, first, ae, step, acc, stride, err);
    } else if (mode == kDenseW16) {
        dense_rows<V, 16>(op, first, ae, step, acc, stride, err);
    } else if (mode == kDenseW32) {
        dense_rows<V, 32>(op, first, ae, step, acc, stride, err);
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

// Whether every row of B ascends, from two coalesced passes: the places e of
// the whole column array with col[e - 1] >= col[e] (descents_between, over any
// split of the entries), less those of them where a non-empty row starts
// (descents_at_starts, over any split of the rows), are none. A column
// outside [0, ncols) counts as kDescentBad.
constexpr long long kDescentBad = 1ll << 40;
__device__ __forceinline__ long long descents_between(const int32_t *ci, int64_t e0, int64_t e1, int ncols, int t,
                                                      int nt) {
    long long d = 0;
    for (int64_t e = e0 + t; e < e1; e += nt) {
        const int j = __ldg(ci + e);
        if (e > 0 && __ldg(ci + e - 1) >= j) ++d;
        if ((unsigned)j >= (unsigned)ncols) d += kDescentBad;
    }
    return d;
}
__device__ __forceinline__ long long descents_at_starts(const int64_t *rp, const int32_t *ci, int64_t nnz, int64_t r0,
                                                        int64_t r1, int t, int nt) {
    long long d = 0;
    for (int64_t r = r0 + t; r < r1; r += nt) {
        const int64_t s = __ldg(rp + r), e = __ldg(rp + r + 1);
        if (s > 0 && e > s && e <= nnz && __ldg(ci + s - 1) >= __ldg(ci + s)) ++d;
    }
    return d;
}

}  // namespace smash
