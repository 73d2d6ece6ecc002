// Rows of products whose B is narrow: a warp owns all columns of a row, in
// both phases (the paper's "dense row" with a scratchpad array per thread
// group instead of one for the whole block).
//
// Symbolic: a byte per column, set by plain stores (lanes that set the same
// byte agree), counted and cleared word by word. Numeric: the dense
// accumulator of warp_dense.cuh.
//
// A warp claims a few rows at a time; lane l loads the bounds of row l. Rows
// with more than `heavy` entries of A (64 and a sixteenth of the words that the
// warps' accumulators have to be added up over, and a warp's share of all the
// bin's entries on a full grid: 40,000 rows of 147 entries, two a row of B, times 1,024
// columns in float took 418 us with every row a block's, 180 us so) would leave one
// warp running long after the others: every block first
// looks through its share of the bin (every gridDim.x-th row, so that the heavy
// rows of a skewed graph, which sit together, spread over the blocks) and
// serves the heavy ones with all its warps, each taking every eighth batch of
// 32 entries.
//
// Measured (50,021-row skewed graph times 256 columns at 5 %, float; before: a
// block of 256 threads per row): counts 0.31 -> 0.09 ms, values 0.28 -> 0.10 ms,
// the whole product 0.71 -> 0.35 ms; a 1024-row graph's square 235 -> 167 us
// (both with the fewer launches of small products).
// What is left waits for the chain of loads (row list, row of A, row pointer
// of B, row of B) of the heavy rows' blocks: 19 % of the issue slots are used by the
// counts, 35 % by the values. Fetching the next batch's row pointers ahead cost more
// instructions than the wait it hid (512 batched products 1.69 -> 1.94 ms).
#include <climits>

#include "device_common.cuh"
#include "kernels.h"
#include "launch_cache.h"
#include "warp_dense.cuh"
#include "writeout.cuh"

namespace smash {

constexpr int kNarrowNT = 256;
constexpr int kNarrowWarps = kNarrowNT / 32;

struct NarrowShare {
    int chunk;   // rows a warp claims at once
    int heavy;   // entries of A above which a row takes a block
};

// Heavy rows of the block's share of the bin: f(i) by all threads for each.
template <typename F>
__device__ __forceinline__ void narrow_heavy(const int64_t *a_rp, int64_t a_nnz, const int *rows, int count, int heavy,
                                             F &&f) {
    __shared__ int s_list[kNarrowNT], s_n;
    for (int64_t base = blockIdx.x; base < count; base += (int64_t)gridDim.x * kNarrowNT) {
        __syncthreads();
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const int64_t x = base + (int64_t)gridDim.x * threadIdx.x;
        if (x < count) {
            const int i = rows[x];
            const int64_t ab = __ldg(a_rp + i), ae = __ldg(a_rp + i + 1);
            if (ab >= 0 && ae - ab > heavy && ae <= a_nnz) s_list[atomicAdd(&s_n, 1)] = i;
        }
        __syncthreads();
        const int n = s_n;
        for (int q = 0; q < n; ++q) f(s_list[q]);
    }
    __syncthreads();
}

// ----- symbolic ----------------------------------------------------------------
template <int W>
__device__ __forceinline__ void narrow_flag(const Operands<float> &op, int64_t first, int64_t ae, int64_t step,
                                            unsigned char *fl, int *err) {
    bool bad = false;
    dense_rows<float, W, false>(op, first, ae, step, err, [&](int, bool act, int j, float, float) {
        if (act) {
            if ((unsigned)j < (unsigned)op.ncols) fl[j] = 1;
            else bad = true;
        }
    });
    if (bad) raise_err(err, kErrBadIndex);
}

__device__ __forceinline__ void narrow_flag_rows(const Operands<float> &op, int mode, int64_t first, int64_t ae,
                                                 int64_t step, unsigned char *fl, int *err) {
    if (mode == kDenseW8) narrow_flag<8>(op, first, ae, step, fl, err);
    else if (mode == kDenseW16) narrow_flag<16>(op, first, ae, step, fl, err);
    else narrow_flag<32>(op, first, ae, step, fl, err);
}

// words: 4-byte words of one warp's flags (cols(B) bytes, rounded up to 128).
__global__ void __launch_bounds__(kNarrowNT) k_narrow_count(Operands<float> op, const int *rows, int count, int *token,
                                                            int mode, int words, NarrowShare sh, int *nnz_out, int *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_tot;
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    unsigned *mine = (unsigned *)smem + (size_t)w * words;
    for (int x = lane; x < words; x += 32) mine[x] = 0u;
    narrow_heavy(op.a_rp, op.a_nnz, rows, count, sh.heavy, [&](int i) {
        const int64_t ab = __ldg(op.a_rp + i), ae = __ldg(op.a_rp + i + 1);
        if (threadIdx.x == 0) s_tot = 0;
        narrow_flag_rows(op, mode, ab + 32 * w, ae, 32 * kNarrowWarps, smem, err);   // the first warp's flags
        __syncthreads();
        int c = 0;
        for (int x = threadIdx.x; x < words; x += kNarrowNT) {
            c += __popc(((unsigned *)smem)[x]);
            ((unsigned *)smem)[x] = 0u;
        }
        c = warp_sum(c);
        if (lane == 0) atomicAdd(&s_tot, c);
        __syncthreads();
        if (threadIdx.x == 0) nnz_out[i] = s_tot;
        __syncthreads();
    });
    for (;;) {
        unsigned r0 = 0;   // (claims past the last of up to 2^31 - 1 rows stay below 2^32)
        if (lane == 0) r0 = atomicAdd((unsigned *)token, (unsigned)sh.chunk);
        r0 = __shfl_sync(kFull, r0, 0);
        if (r0 >= (unsigned)count) break;
        int il = 0;
        int64_t abl = 0, ael = 0;
        bool light = false;
        if (lane < sh.chunk && r0 + lane < (unsigned)count) {
            il = rows[r0 + lane];
            a_row_range(op, il, abl, ael, err);
            light = ael - abl <= sh.heavy;
        }
        for (unsigned todo = __ballot_sync(kFull, light); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int i = __shfl_sync(kFull, il, src);
            const int64_t ab = __shfl_sync(kFull, abl, src), ae = __shfl_sync(kFull, ael, src);
            narrow_flag_rows(op, mode, ab, ae, 32, (unsigned char *)mine, err);
            __syncwarp();
            int c = 0;
            for (int x = lane; x < words; x += 32) {
                c += __popc(mine[x]);
                mine[x] = 0u;
            }
            c = __reduce_add_sync(kFull, c);
            if (lane == 0) nnz_out[i] = c;
            __syncwarp();
        }
    }
}

// ----- numeric -----------------------------------------------------------------
// Whether every row of B ascends below cols(B): *descents becomes 0.
__global__ void __launch_bounds__(256) k_descents(const int64_t *rp, const int32_t *ci, int64_t rows, int64_t nnz,
                                                  int ncols, long long *descents) {
    constexpr int64_t kEnt = 8192, kRow = 2048;
    const int64_t eseg = (nnz + kEnt - 1) / kEnt, segs = eseg + (rows + kRow - 1) / kRow;
    long long d = 0;
    bool bad = false;
    for (int64_t q = blockIdx.x; q < segs; q += gridDim.x) {
        if (q < eseg) {
            const int64_t e0 = q * kEnt;
            d += descents_between(ci, e0, e0 + kEnt < nnz ? e0 + kEnt : nnz, ncols, threadIdx.x, 256, bad);
        } else {
            const int64_t r0 = (q - eseg) * kRow;
            d -= descents_at_starts(rp, ci, nnz, r0, r0 + kRow < rows ? r0 + kRow : rows, threadIdx.x, 256, bad);
        }
    }
    descents_add((unsigned long long *)descents, d, bad);
}

// Row i of C, room [c0, c0 + n_exp), from the accumulator.
template <typename V>
__device__ __forceinline__ void narrow_out(V *acc, int mode, int ncols, int i, int64_t c0, int n_exp,
                                           const NumOutT<V> &out, int *err) {
    int32_t *ci = out.c_ci + c0;
    V *val = out.c_val + c0;
    const int n = dense_emit(acc, mode, ncols, [&](int pos, int j, V v) {
        if (pos < n_exp) {
            __stcs(ci + pos, j);
            __stcs(val + pos, v);
        }
    });
    if (lane_id() == 0) {
        if (out.row_nnz) out.row_nnz[i] = n <= n_exp ? n : -1;
        else if (n != n_exp) raise_err(err, kErrCountMismatch);
    }
}

template <typename V>
__global__ void __launch_bounds__(kNarrowNT) k_narrow_num(Operands<V> op, const int *rows, int count, int *token,
                                                          int mode, int warp_words, NarrowShare sh,
                                                          const long long *descents, NumOutT<V> out, int *err) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = lane_id();
    const int w = threadIdx.x >> 5;
    V *all = (V *)smem;
    V *acc = all + (size_t)w * warp_words;
    const bool ascend = *descents == 0;   // (flat adds: of no account)
    dense_clear(acc, warp_words);
    __syncwarp();
    narrow_heavy(op.a_rp, op.a_nnz, rows, count, sh.heavy, [&](int i) {
        const int64_t ab = __ldg(op.a_rp + i), ae = __ldg(op.a_rp + i + 1);
        dense_accumulate(op, mode, ascend, ab + 32 * w, ae, 32 * kNarrowWarps, acc, err);
        __syncthreads();
        for (int x = threadIdx.x; x < warp_words; x += kNarrowNT) {
            V v = all[x];
            for (int q = 1; q < kNarrowWarps; ++q) {
                V *o = all + (size_t)q * warp_words + x;
                v += *o;
                *o = dense_unused(V(0));
            }
            all[x] = v;
        }
        __syncthreads();
        if (w == 0) {
            int64_t c0;
            int n_exp;
            out_range(out, i, c0, n_exp, err);
            narrow_out(acc, mode, op.ncols, i, c0, n_exp, out, err);
        }
        __syncthreads();
    });
    for (;;) {
        unsigned r0 = 0;
        if (lane == 0) r0 = atomicAdd((unsigned *)token, (unsigned)sh.chunk);
        r0 = __shfl_sync(kFull, r0, 0);
        if (r0 >= (unsigned)count) break;
        int il = 0, nl = 0;
        int64_t abl = 0, ael = 0, cl = 0;
        bool light = false;
        if (lane < sh.chunk && r0 + lane < (unsigned)count) {
            il = rows[r0 + lane];
            const int64_t s = out.c_rp[il], t = out.c_rp[il + 1];
            a_row_range(op, il, abl, ael, err);
            light = ael - abl <= sh.heavy;
            row_bounds_ok(s, t, out.c_nnz, cl, nl, err);
        }
        for (unsigned todo = __ballot_sync(kFull, light); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            const int i = __shfl_sync(kFull, il, src), n_exp = __shfl_sync(kFull, nl, src);
            const int64_t ab = __shfl_sync(kFull, abl, src), ae = __shfl_sync(kFull, ael, src);
            const int64_t c0 = __shfl_sync(kFull, cl, src);
            dense_accumulate(op, mode, ascend, ab, ae, 32, acc, err);
            narrow_out(acc, mode, op.ncols, i, c0, n_exp, out, err);
        }
    }
}

// ---------------------------------------------------------------------------
template <typename V>
static Operands<V> narrow_operands(const RawOperands &r) {
    Operands<V> o;
    o.a_rp = r.a_rp;
    o.a_ci = r.a_ci;
    o.a_val = (const V *)r.a_val;
    o.b_rp = r.b_rp;
    o.b_ci = r.b_ci;
    o.b_val = (const V *)r.b_val;
    o.a_nnz = r.a_nnz;
    o.b_nnz = r.b_nnz;
    o.b_rows = r.b_rows;
    o.ncols = r.ncols;
    return o;
}

// Blocks of a launch (one for each 8 rows or 256 entries of A, as many as are
// resident at most), the rows a warp claims at once (eight claims per warp of a
// full grid, at most eight rows) and the heavy rows' threshold.
template <typename K>
static int narrow_grid(K kernel, size_t smem, int sms, int count, long long entries, int words, NarrowShare &sh) {
    allow_smem((const void *)kernel);
    int per_sm = resident_per_sm((const void *)kernel, kNarrowNT, smem);
    const int64_t cap = (int64_t)(per_sm < 1 ? 1 : per_sm) * sms;
    const int64_t share = count / (cap * kNarrowWarps * 8);
    sh.chunk = share < 1 ? 1 : share > 8 ? 8 : (int)share;
    const int64_t share_entries = entries / (cap * kNarrowWarps);
    sh.heavy = 64 + words / 16;
    if (share_entries > sh.heavy) sh.heavy = share_entries < INT_MAX ? (int)share_entries : INT_MAX;
    int64_t want = ((int64_t)count + (int64_t)kNarrowWarps * sh.chunk - 1) / (kNarrowWarps * sh.chunk);
    if (want < entries / 256) want = entries / 256;
    if (want > count) want = count;
    return (int)(want < cap ? want : cap);
}

bool narrow_symbolic(int64_t ncols) { return ncols <= kNarrowSymCols; }
bool narrow_few(int64_t rows, int sms) { return rows <= (int64_t)sms * kNarrowWarps; }

// Which numeric rows a warp's accumulator serves, by the bytes of one. An
// accumulator is cleared and scanned for every row, and 8 of them decide how many
// blocks are resident; the alternatives are a table (rows below a quarter of the
// columns) and column windows with a block a row.
//   Up to 6 KB in float, 8 KB in double: every dense row, down to a sixteenth of the
// columns (us, accumulator and alternative, rows of a sixteenth / a quarter / all of
// the columns: float 1,024 columns 108 and 131 / 134 and 371 / 113 and 235, double 129
// and 137 / 164 and 587 / 148 and 414).
//   Up to 12 KB: from an eighth on (double 1,536 columns, a sixteenth 169 and 169, an
// eighth 211 and 245, a quarter 225 and 594; float 2,048 columns 176 and 174, 195 and
// 261, 170 and 320), where there is a row for more than one block's warps an SM and the
// rows' products are at most twice the columns (2,048-row skewed square, 300 rows:
// 145 and 120; 3,000 columns, products four times as many: 275 and 182).
//   Up to 24 KB in double: from a quarter on, where an entry of A has 8 products or more
// besides (2,048 columns, 49 entries of 12 products 347 and 493, 294 of 2 599 and 460).
// In float windows are better beyond 12 KB (4,000 columns, a quarter 310 and 270).
constexpr int narrow_short_bytes(int dtype) { return dtype ? 8 * 1024 : 6 * 1024; }
constexpr int kNarrowMediumBytes = 12 * 1024;

int narrow_ratio(int dtype, int64_t ncols) {
    const int64_t bytes = ncols * (dtype ? 8 : 4);
    return bytes <= narrow_short_bytes(dtype) ? 4 : bytes <= kNarrowMediumBytes ? 2 : 1;
}
bool narrow_numeric(int dtype, int64_t ncols, long long rows, long long entries, long long products, int sms) {
    const int64_t bytes = ncols * (dtype ? 8 : 4);
    if (bytes <= narrow_short_bytes(dtype)) return true;
    if (bytes > (dtype ? kDenseWarpBytes : kNarrowMediumBytes)) return false;
    if (narrow_few(rows, sms) || products > 2 * ncols * rows) return false;
    return bytes <= kNarrowMediumBytes || products >= 8 * entries;
}

void launch_narrow_count(const RawOperands &r, const int *rows, int count, long long entries, long long products,
                         int *token, int sms,
                         int *nnz_out, int *err, cudaStream_t s) {
    if (count <= 0) return;
    const int words = ((r.ncols + 127) & ~127) / 4;
    const size_t smem = (size_t)kNarrowWarps * words * 4;
    NarrowShare sh;
    const int grid = narrow_grid(k_narrow_count, smem, sms, count, entries, words, sh);
    // (no accumulator copies to fit: the lane group by the mean row length alone)
    const int mode = dense_mode(products, entries, 32, 4, true);
    k_narrow_count<<<grid, kNarrowNT, smem, s>>>(narrow_operands<float>(r), rows, count, token,
                                                 mode == kDenseFlat ? kDenseW8 : mode, words, sh, nnz_out, err);
}

template <typename V>
static int narrow_num_typed(const RawOperands &r, const int *rows, int count, long long entries, long long products,
                            int *token, int sms, long long *descents, const NumOut &o, int *err, cudaStream_t s) {
    const NumOutT<V> out{o.c_rp, o.c_ci, (V *)o.c_val, o.c_nnz, o.row_nnz};
    // plain adds need a pass over B, which fewer products than B has entries don't pay for
    const bool few = narrow_few(count, sms);
    const int mode = products < r.b_nnz ? kDenseFlat : dense_mode(products, entries, r.ncols, sizeof(V), few);
    if (mode != kDenseFlat) {
        cudaMemsetAsync(descents, 0, sizeof(long long), s);
        const int64_t segs = r.b_nnz / 8192 + r.b_rows / 2048 + 2;
        k_descents<<<(int)(segs < 8ll * sms ? segs : 8ll * sms), 256, 0, s>>>(r.b_rp, r.b_ci, r.b_rows, r.b_nnz,
                                                                            r.ncols, descents);
    }
    const size_t warp_bytes = dense_warp_bytes(mode, r.ncols, sizeof(V));
    const size_t smem = kNarrowWarps * warp_bytes;
    NarrowShare sh;
    const int grid = narrow_grid(k_narrow_num<V>, smem, sms, count, entries, (int)(warp_bytes / sizeof(V)), sh);
    k_narrow_num<V><<<grid, kNarrowNT, smem, s>>>(narrow_operands<V>(r), rows, count, token, mode,
                                                  (int)(warp_bytes / sizeof(V)), sh, descents, out, err);
    return mode != kDenseFlat ? 2 : 1;
}

int launch_narrow_num(int dtype, const RawOperands &r, const int *rows, int count, long long entries,
                      long long products, int *token, int sms, long long *descents, const NumOut &out, int *err,
                      cudaStream_t s) {
    if (count <= 0) return 0;
    if (dtype) return narrow_num_typed<double>(r, rows, count, entries, products, token, sms, descents, out, err, s);
    return narrow_num_typed<float>(r, rows, count, entries, products, token, sms, descents, out, err, s);
}

}  // namespace smash
