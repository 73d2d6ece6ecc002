// Batched SpGEMM: many independent products C_m = A_m * B_m in one persistent,
// work-stealing kernel.
//
// Not in the paper as such; it carries Version 2's tokenization (threads poll
// a shared token counter for the next piece of work instead of a static
// schedule) across products: every block repeatedly claims the next work item
// of a global list with one atomic add, so products of very different sizes
// keep all SMs busy. Items are (a) single large rows, processed by the whole
// block, listed first so they start early, (b) medium rows, one warp each, and
// (c) chunks of consecutive rows, claimed by a warp. A row's accumulator is
// a dense array over the columns of B when B is narrow (warp_dense.cuh), one
// per warp, else a hash table.
//
// Why three sizes: with all rows of narrow products in chunks of 32, the 32
// heaviest rows of a skewed graph fell to one warp, and every other block
// waited for it at the grid barrier (36 of 53 stall cycles per issue; 3 of 15
// now).
//
// One cooperative launch runs four phases separated by grid barriers (each
// wait bounded; a barrier that times out sets an error word and the kernel
// returns): counts (and the values of narrow products' rows), per-product
// row-pointer scans, product base offsets, numeric values with sorted write-out. Rows too large for one
// block's table are done around the kernel by the regular per-product path.
#include "device_common.cuh"
#include "kernels.h"
#include "launch_cache.h"
#include "writeout.cuh"
#include "batch_types.h"
#include "warp_dense.cuh"

namespace smash {


__device__ __forceinline__ int find_mat(const int64_t *start, int nmat, int64_t g) {
    int lo = 0, hi = nmat;   // last m with start[m] <= g
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (start[mid] <= g) lo = mid;
        else hi = mid;
    }
    return lo;
}

template <typename V>
__device__ __forceinline__ Operands<V> mat_ops(const BatchMat &m) {
    Operands<V> o;
    o.a_rp = m.a_rp;
    o.a_ci = m.a_ci;
    o.a_val = (const V *)m.a_val;
    o.b_rp = m.b_rp;
    o.b_ci = m.b_ci;
    o.b_val = (const V *)m.b_val;
    o.a_nnz = m.a_nnz;
    o.b_nnz = m.b_nnz;
    o.b_rows = m.b_rows;
    o.ncols = m.ncols;
    return o;
}

__device__ __forceinline__ int colbits(int n) {
    int b = 0;
    while ((1 << b) < n && b < 31) ++b;
    return b;
}

// Row classification over all products' rows. One thread per row, four
// entries in flight; rows of more than kLongBatchRow entries go to a list that
// k_batch_rowinfo_long spreads over all warps, a warp per row (the long rows of
// a skewed graph sit together: counted by the warp that finds them they took
// 0.24 ms of the 512-product batch). From 16, 48 and 192 entries on: 512 products 1.68,
// 1.66 and 1.72 ms, 24 products 0.32, 0.34 and 0.37 ms.
constexpr int kLongBatchRow = 48;

__device__ __forceinline__ long long batch_b_len(const BatchMat &M, int k, int *err) {
    if ((unsigned)k >= (unsigned)M.b_rows) {
        raise_err(err, kErrBadIndex);
        return 0;
    }
    const int64_t s = __ldg(M.b_rp + k), t = __ldg(M.b_rp + k + 1);
    if (s >= 0 && t >= s && t <= M.b_nnz) return t - s;
    raise_err(err, kErrBadRowPtr);
    return 0;
}

// Class, room and lists of row g with f products; returns its room.
__device__ __forceinline__ long long batch_classify(const BatchArgs &p, const BatchMat &M, int64_t g, long long f) {
    const long long ub = f < (long long)M.ncols ? f : (long long)M.ncols;
    uint8_t c;
    if (ub == 0) c = kRowEmpty;
    else if (M.mode >= 0) c = f <= kMedFlop ? kRowSmall : f <= kBigFlop ? kRowMed : kRowBig;
    else if (table_bits(ub, p.inv_load) <= p.warp_bits) c = kRowSmall;
    else if (table_bits(ub, p.inv_load) <= p.block_bits) c = kRowBig;
    else c = kRowHuge;
    p.cls[g] = c;
    p.ub[g] = (int)ub;
    p.nnz[g] = 0;
    if (c == kRowBig) p.big[atomicAdd(p.counters + 0, 1)] = (int)g;
    if (c == kRowHuge) p.huge[atomicAdd(p.counters + 1, 1)] = (int)g;
    if (c == kRowMed) p.med[atomicAdd(p.counters + 12, 1)] = (int)g;
    return ub;
}

// f, if row and accumulator are such that it speaks for accumulators (batched_modes).
__device__ __forceinline__ long long batch_long(const BatchArgs &p, const BatchMat &M, long long f) {
    return M.mode >= 0 && M.ncols > p.large_cols && f > kBatchLongRow ? f : 0;
}

// The first row_blocks blocks count rows, the others pass over the narrow
// products' B (whether its rows ascend).
__global__ void __launch_bounds__(256) k_batch_rowinfo(BatchArgs p, int row_blocks) {
    const int lane = lane_id();
    if ((int)blockIdx.x >= row_blocks) {
        for (int64_t q = blockIdx.x - row_blocks; q < p.nseg; q += gridDim.x - row_blocks) {
            int lo = 0, hi = p.nmat;   // last product whose segments start at or before q
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (p.mats[mid].seg_off <= q) lo = mid;
                else hi = mid;
            }
            const BatchMat &M = p.mats[lo];
            int64_t x = q - M.seg_off;
            const int64_t eseg = (M.b_nnz + kSegEntries - 1) / kSegEntries;
            long long d;
            bool bad = false;
            if (x < eseg) {
                const int64_t e0 = x * kSegEntries;
                const int64_t e1 = e0 + kSegEntries < M.b_nnz ? e0 + kSegEntries : M.b_nnz;
                d = descents_between(M.b_ci, e0, e1, M.ncols, threadIdx.x, 256, bad);
            } else {
                const int64_t r0 = (x - eseg) * kSegRows;
                const int64_t r1 = r0 + kSegRows < M.b_rows ? r0 + kSegRows : M.b_rows;
                d = -descents_at_starts(M.b_rp, M.b_ci, M.b_nnz, r0, r1, threadIdx.x, 256, bad);
            }
            descents_add((unsigned long long *)p.descents + lo, d, bad);
        }
        return;
    }
    const int64_t threads = (int64_t)row_blocks * blockDim.x;
    unsigned long long my_ub = 0, my_f = 0, my_long = 0;
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < p.nrows; g += threads) {
        const int mi = find_mat(p.row_start, p.nmat, g);
        const BatchMat &M = p.mats[mi];
        const int64_t r = g - p.row_start[mi];
        int64_t ab = __ldg(M.a_rp + r), ae = __ldg(M.a_rp + r + 1);
        if (ab < 0 || ae < ab || ae > M.a_nnz) {
            raise_err(p.err, kErrBadRowPtr);
            ab = ae = 0;
        }
        if (ae - ab > kLongBatchRow) {
            p.longs[atomicAdd(p.counters + 13, 1)] = (int)g;
            continue;
        }
        long long f = 0;
        for (int64_t e = ab; e < ae; e += 4) {
            int k[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) k[u] = e + u < ae ? __ldg(M.a_ci + e + u) : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (e + u < ae) f += batch_b_len(M, k[u], p.err);
        }
        my_ub += (unsigned long long)batch_classify(p, M, g, f);
        my_f += (unsigned long long)f;
        my_long += (unsigned long long)batch_long(p, M, f);
    }
    my_ub = warp_sum(my_ub);
    my_f = warp_sum(my_f);
    my_long = warp_sum(my_long);
    if (lane == 0) {
        atomicAdd(p.sums + 0, my_ub);
        atomicAdd(p.sums + 1, my_f);
        if (my_long) atomicAdd(p.sums + 2, my_long);
    }
}

__global__ void __launch_bounds__(256) k_batch_rowinfo_long(BatchArgs p) {
    const int lane = lane_id();
    const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int n = p.counters[13];
    unsigned long long my_ub = 0, my_f = 0, my_long = 0;
    for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < n; q += warps) {
        const int64_t g = p.longs[q];
        const int mi = find_mat(p.row_start, p.nmat, g);
        const BatchMat &M = p.mats[mi];
        const int64_t r = g - p.row_start[mi];
        const int64_t ab = __ldg(M.a_rp + r), ae = __ldg(M.a_rp + r + 1);   // checked by k_batch_rowinfo
        long long f = 0;
        for (int64_t e0 = ab + lane; e0 < ae; e0 += 128) {
            int k[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) k[u] = e0 + 32 * u < ae ? __ldg(M.a_ci + e0 + 32 * u) : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (e0 + 32 * u < ae) f += batch_b_len(M, k[u], p.err);
        }
        __syncwarp();
        f = warp_sum(f);
        if (lane == 0) {
            my_ub += (unsigned long long)batch_classify(p, M, g, f);
            my_f += (unsigned long long)f;
            my_long += (unsigned long long)batch_long(p, M, f);
        }
    }
    if (lane == 0 && my_f) {
        atomicAdd(p.sums + 0, my_ub);
        atomicAdd(p.sums + 1, my_f);
        if (my_long) atomicAdd(p.sums + 2, my_long);
    }
}

// Grid barrier for a cooperative launch; returns false after a timeout
// (wait_spins polls). missing > 0 makes the barrier wait for arrivals that
// never come, so that every block's wait runs out (a test of the time-out).
__device__ __forceinline__ bool grid_barrier(int *bar, int *err, long long wait_spins, int missing) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int *gen = bar + 1;
        const int g = *gen;
        __threadfence();
        const int arrived = atomicAdd(bar, 1);
        int ok = 1;
        if (arrived == (int)gridDim.x - 1 + missing) {
            atomicExch(bar, 0);
            __threadfence();
            atomicAdd(bar + 1, 1);
        } else {
            long long it = 0;
            while (*gen == g) {
                if (++it > wait_spins) {
                    raise_err(err, kErrTimeout);
                    ok = 0;
                    break;
                }
                __nanosleep(256);
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

template <typename V>
struct BatchSmem {
    unsigned char *tab;     // 8 warp tables (or one block table)
    ProdScratch<V> sc;      // block-wide product staging
};

// A row of a narrow product: values, count and the sorted row (staged), by one
// warp whose dense accumulator is acc.
template <typename V>
__device__ __forceinline__ void narrow_emit(const BatchArgs &p, const BatchMat &M, int64_t g, V *acc) {
    const int64_t so = p.stage_off[g];
    const int room = p.ub[g];
    int32_t *ci = p.stage_ci + so;
    V *val = (V *)p.stage_val + so;
    const int n = dense_emit(acc, M.mode, M.ncols, [&](int pos, int j, V v) {
        if (pos < room) {
            ci[pos] = j;
            val[pos] = v;
        }
    });
    if (lane_id() == 0) {
        p.nnz[g] = n < room ? n : room;
        if (n > room) raise_err(p.err, kErrTableFull);
    }
}

template <typename V>
__device__ __forceinline__ void narrow_row(const BatchArgs &p, const BatchMat &M, int mi, int64_t g, int64_t r,
                                           V *acc) {
    const Operands<V> op = mat_ops<V>(M);
    int64_t ab, ae;
    a_row_range(op, r, ab, ae, p.err);
    dense_accumulate(op, M.mode, p.descents[mi] == 0, ab, ae, 32, acc, p.err);
    narrow_emit(p, M, g, acc);
}

// The same by the whole block: every warp takes each kBW-th batch of 32
// entries of the row, the warps' accumulators are added up in the first
// warp's, which writes the row out.
template <typename V>
__device__ void narrow_block_row(const BatchArgs &p, const BatchMat &M, int mi, int64_t g, int64_t r,
                                 unsigned char *tab) {
    const Operands<V> op = mat_ops<V>(M);
    const int w = threadIdx.x >> 5;
    int64_t ab, ae;
    a_row_range(op, r, ab, ae, p.err);
    dense_accumulate(op, M.mode, p.descents[mi] == 0, ab + 32 * w, ae, 32 * kBW, (V *)(tab + (size_t)w * p.warp_bytes),
                     p.err);
    __syncthreads();
    const int words = dense_copies(M.mode) * dense_stride(M.ncols);
    for (int x = threadIdx.x; x < words; x += kBNT) {
        V v = ((V *)tab)[x];
        for (int q = 1; q < kBW; ++q) {
            V *o = (V *)(tab + (size_t)q * p.warp_bytes) + x;
            v += *o;
            *o = dense_unused(V(0));
        }
        ((V *)tab)[x] = v;
    }
    __syncthreads();
    if (w == 0) narrow_emit(p, M, g, (V *)tab);
    __syncthreads();
}

// One small row of a wide product by one warp: count (NUM = false) or values
// + write-out.
template <typename V, bool NUM>
__device__ void warp_row(const BatchArgs &p, const BatchMat &M, int64_t g, int64_t r, unsigned char *wtab, int64_t c0,
                         int n_exp, int64_t base) {
    const Operands<V> op = mat_ops<V>(M);
    const int lane = lane_id();
    int64_t ab, ae;
    a_row_range(op, r, ab, ae, p.err);
    const int T = 1 << p.tw_bits;
    // hash table of the warp
    const int tb = table_bits(p.ub[g], p.inv_load);
    const int Tr = 1 << tb;
    int *keys = (int *)wtab;
    V *vals = (V *)(wtab + (size_t)T * 4);
    for (int s = lane; s < Tr; s += 32) {
        keys[s] = kEmpty;
        if (NUM) vals[s] = V(0);
    }
    __syncwarp();
    HashCfg hc = p.hc;
    hc.colbits = colbits(M.ncols);
    int cnt = 0;
    warp_products<V, NUM>(op, ab, ae, p.err, [&](int j, V a, V bkj) {
        bool ins;
        const int h = hash_find_or_insert<false>(keys, tb, hc, j, ins);
        if (h < 0) {
            raise_err(p.err, kErrTableFull);
            return;
        }
        if (NUM) atomicAdd(vals + h, a * bkj);
        cnt += ins ? 1 : 0;
    });
    const int tot = warp_sum(cnt);
    __syncwarp();
    if (!NUM) {
        if (lane == 0) p.nnz[g] = tot;
    } else {
        if (lane == 0 && tot != n_exp) raise_err(p.err, kErrCountMismatch);
        NumOutT<V> out{nullptr, p.ci_pool + base, (V *)p.val_pool + base, 0, nullptr};
        unsigned places = 0u;   // (a table's columns are distinct)
        if (tot <= 32) writeout_warp_rank<V>(keys, vals, Tr, n_exp, out, c0, places);
        else writeout_bitonic<V, 32, kBNT>(keys, vals, Tr, n_exp, out, c0, nullptr);
    }
    __syncwarp();
}

// One big row by the whole block.
template <typename V, bool NUM>
__device__ void block_row(const BatchArgs &p, const BatchMat &M, int64_t g, int64_t r, const BatchSmem<V> &sm,
                          int64_t c0, int n_exp, int64_t base) {
    using G = Group<kBNT, kBNT>;
    const Operands<V> op = mat_ops<V>(M);
    int64_t ab, ae;
    a_row_range(op, r, ab, ae, p.err);
    const int Tall = kBW << p.tw_bits;
    const int tb = table_bits(p.ub[g], p.inv_load);
    const int Tr = 1 << tb;
    int *keys = (int *)sm.tab;
    V *vals = (V *)(sm.tab + (size_t)Tall * 4);
    for (int s = threadIdx.x; s < Tr; s += kBNT) {
        keys[s] = kEmpty;
        if (NUM) vals[s] = V(0);
    }
    __syncthreads();
    HashCfg hc = p.hc;
    hc.colbits = colbits(M.ncols);
    int cnt = 0;
    group_products<V, NUM, kBNT, kBNT>(op, ab, ae, sm.sc, p.err, [&](int j, V a, V bkj) {
        bool ins;
        const int h = hash_find_or_insert<false>(keys, tb, hc, j, ins);
        if (h < 0) {
            raise_err(p.err, kErrTableFull);
            return;
        }
        if (NUM) atomicAdd(vals + h, a * bkj);
        cnt += ins ? 1 : 0;
    });
    const int tot = G::template sum<int>(cnt, sm.sc.red);
    if (!NUM) {
        if (threadIdx.x == 0) p.nnz[g] = tot;
    } else {
        if (threadIdx.x == 0 && tot != n_exp) raise_err(p.err, kErrCountMismatch);
        NumOutT<V> out{nullptr, p.ci_pool + base, (V *)p.val_pool + base, 0, nullptr};
        writeout_bitonic<V, kBNT, kBNT>(keys, vals, Tr, n_exp, out, c0, sm.sc.red);
    }
    __syncthreads();
}

// Work of one phase: the big rows first, one per block, then the medium rows,
// one per warp (claimed with one counter each); then every warp claims chunks
// of consecutive rows of the flattened row space on its own (32, fewer when
// that would leave warps without work) and serves the small rows among them,
// with no block-wide wait between rows of unequal cost.
// The rows of narrow products are computed and staged in the first phase
// (NUM = false) and copied to their places in the last (NUM = true), a chunk's
// rows one after another, four loads per lane in flight.
template <typename V, bool NUM, bool WIDE>
__device__ void run_items(const BatchArgs &p, const BatchSmem<V> &sm) {
    __shared__ int s_item;
    const int w = threadIdx.x >> 5;
    const int lane = lane_id();
    const int nbig = p.counters[0];
    unsigned char *wtab = sm.tab + (size_t)w * p.warp_bytes;
    V *acc = (V *)wtab;
    bool clean = false;   // the dense accumulator's words are unused (a hash table shares its room)
    if (!NUM || WIDE) {
        for (;;) {
            if (threadIdx.x == 0) s_item = atomicAdd(p.counters + (NUM ? 3 : 2), 1);
            __syncthreads();
            const int it = s_item;
            __syncthreads();
            if (it >= nbig) break;
            const int64_t g = p.big[it];
            const int mi = find_mat(p.row_start, p.nmat, g);
            const BatchMat &M = p.mats[mi];
            const int64_t r = g - p.row_start[mi];
            if (M.mode >= 0) {
                if (!NUM) {
                    if (!clean) dense_clear(acc, p.dense_words);
                    clean = true;
                    __syncthreads();
                    narrow_block_row<V>(p, M, mi, g, r, sm.tab);
                }
            } else if constexpr (WIDE) {
                int64_t c0 = 0;
                int n_exp = 0;
                int64_t base = 0;
                if (NUM) {
                    const int64_t *rp = p.rp_pool + p.row_start[mi] + mi;
                    c0 = rp[r];
                    n_exp = (int)(rp[r + 1] - rp[r]);
                    base = p.base[mi];
                }
                clean = false;
                block_row<V, NUM>(p, M, g, r, sm, c0, n_exp, base);
            }
        }
    }
    if (!NUM) {
        const int nmed = p.counters[12];
        for (;;) {
            int it = 0;
            if (lane == 0) it = atomicAdd(p.counters + 4, 1);
            it = __shfl_sync(kFull, it, 0);
            if (it >= nmed) break;
            const int64_t g = p.med[it];
            const int mi = find_mat(p.row_start, p.nmat, g);
            if (!clean) dense_clear(acc, p.dense_words);
            clean = true;
            __syncwarp();
            narrow_row<V>(p, p.mats[mi], mi, g, g - p.row_start[mi], acc);
        }
    }
    for (;;) {
        int ch = 0;
        if (lane == 0) ch = atomicAdd(p.counters + (NUM ? 9 : 8), 1);
        ch = __shfl_sync(kFull, ch, 0);
        const int64_t g0 = (int64_t)ch * p.chunk;
        if (g0 >= p.nrows) break;
        // lane l: row g0 + l, its product and, in the last phase, its places
        const int64_t gl = g0 + lane;
        const int cls = lane < p.chunk && gl < p.nrows ? p.cls[gl] : kRowEmpty;
        int ml = 0, nl = 0;
        bool narrow = false;
        int64_t dl = 0, sl = 0;
        if (cls != kRowEmpty) {
            ml = find_mat(p.row_start, p.nmat, gl);
            narrow = p.mats[ml].mode >= 0;
            if (NUM && narrow) {
                dl = p.base[ml] + p.rp_pool[gl + ml];
                sl = p.stage_off[gl];
                nl = p.nnz[gl];
            }
        }
        if (NUM) {
            for (unsigned todo = __ballot_sync(kFull, narrow); todo; todo &= todo - 1) {
                const int x = __ffs(todo) - 1;
                const int n = __shfl_sync(kFull, nl, x);
                const int64_t d = __shfl_sync(kFull, dl, x), s = __shfl_sync(kFull, sl, x);
                for (int q0 = lane; q0 < n; q0 += 128) {
                    int32_t c[4];
                    V v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (q0 + 32 * u < n) {
                            c[u] = p.stage_ci[s + q0 + 32 * u];
                            v[u] = ((const V *)p.stage_val)[s + q0 + 32 * u];
                        }
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (q0 + 32 * u < n) {
                            p.ci_pool[d + q0 + 32 * u] = c[u];
                            ((V *)p.val_pool)[d + q0 + 32 * u] = v[u];
                        }
                    }
                }
            }
        }
        for (unsigned todo = __ballot_sync(kFull, cls == kRowSmall && (WIDE || !NUM) && !(NUM && narrow)); todo;
             todo &= todo - 1) {
            const int x = __ffs(todo) - 1;
            const int64_t g = g0 + x;
            const int mi = __shfl_sync(kFull, ml, x);
            const BatchMat &M = p.mats[mi];
            const int64_t r = g - p.row_start[mi];
            if (!WIDE || M.mode >= 0) {
                if (!clean) dense_clear(acc, p.dense_words);
                clean = true;
                __syncwarp();
                narrow_row<V>(p, M, mi, g, r, acc);
            } else if constexpr (WIDE) {
                int64_t c0 = 0;
                int n_exp = 0;
                int64_t base = 0;
                if (NUM) {
                    const int64_t *rp = p.rp_pool + p.row_start[mi] + mi;
                    c0 = rp[r];
                    n_exp = (int)(rp[r + 1] - rp[r]);
                    base = p.base[mi];
                }
                clean = false;
                warp_row<V, NUM>(p, M, g, r, wtab, c0, n_exp, base);
            }
        }
    }
}

template <typename V, bool WIDE>
__global__ void __launch_bounds__(kBNT) k_batched(const BatchArgs *pp) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ long long s_w[32];
    // the arguments live in device memory (a recorded launch is replayed with
    // new arguments copied there)
    __shared__ BatchArgs s_p;
    if (threadIdx.x == 0) s_p = *pp;
    __syncthreads();
    const BatchArgs &p = s_p;
    BatchSmem<V> sm;
    sm.tab = smem;
    sm.sc = carve_prod_scratch<V, kBNT>(smem + (size_t)kBW * p.warp_bytes);
    int *bar = p.counters + 6;
    // phase 1: counts (rows of narrow products: values too, staged)
    run_items<V, false, WIDE>(p, sm);
    if (!grid_barrier(bar, p.err, p.wait_spins, p.missing)) return;
    // phase 2: row pointers of each product (one product per block at a time)
    __shared__ int s_m;
    for (;;) {
        if (threadIdx.x == 0) s_m = atomicAdd(p.counters + 5, 1);
        __syncthreads();
        const int mi = s_m;
        __syncthreads();
        if (mi >= p.nmat) break;
        const int64_t r0 = p.row_start[mi], n = p.row_start[mi + 1] - r0;
        int64_t *rp = p.rp_pool + r0 + mi;
        long long carry = 0;
        for (int64_t b0 = 0; b0 < n; b0 += kBNT) {
            const int64_t i = b0 + threadIdx.x;
            const long long v = i < n ? p.nnz[r0 + i] : 0;
            const long long incl = warp_incl_scan64(v);
            if (lane_id() == 31) s_w[threadIdx.x >> 5] = incl;
            __syncthreads();
            long long off = carry, tot = 0;
            for (int k = 0; k < kBW; ++k) {
                if (k < (int)(threadIdx.x >> 5)) off += s_w[k];
                tot += s_w[k];
            }
            if (i < n) rp[i] = off + incl - v;
            carry += tot;
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            rp[n] = carry;
            p.totals[mi] = carry;
        }
    }
    if (!grid_barrier(bar, p.err, p.wait_spins, p.missing)) return;
    // phase 3: base offsets of the products in the pools
    if (blockIdx.x == 0) {
        long long carry = 0;
        for (int b0 = 0; b0 < p.nmat; b0 += kBNT) {
            const int i = b0 + threadIdx.x;
            const long long v = i < p.nmat ? p.totals[i] : 0;
            const long long incl = warp_incl_scan64(v);
            if (lane_id() == 31) s_w[threadIdx.x >> 5] = incl;
            __syncthreads();
            long long off = carry, tot = 0;
            for (int k = 0; k < kBW; ++k) {
                if (k < (int)(threadIdx.x >> 5)) off += s_w[k];
                tot += s_w[k];
            }
            if (i < p.nmat) p.base[i] = off + incl - v;
            carry += tot;
            __syncthreads();
        }
        if (threadIdx.x == 0) p.base[p.nmat] = carry;
    }
    if (!grid_barrier(bar, p.err, p.wait_spins, p.missing)) return;
    // phase 4: values
    run_items<V, true, WIDE>(p, sm);
}

// ---------------------------------------------------------------------------
size_t batched_table_bytes(int dtype, int tw_bits) { return ((size_t)1 << tw_bits) * (dtype ? 12 : 8); }

size_t batched_smem(int dtype, int warp_bytes, bool wide) {
    const size_t sc = dtype ? num_scratch_bytes<double, kBNT>() : num_scratch_bytes<float, kBNT>();
    return (size_t)kBW * warp_bytes + (wide ? sc : 0);
}

void launch_batch_rowinfo(const BatchArgs &p, int sms, cudaStream_t s) {
    if (p.nrows == 0) return;
    const int64_t blocks = (p.nrows + 255) / 256;
    const int64_t cap = (int64_t)sms * 8;
    const int rb = (int)(blocks < cap ? blocks : cap);
    const int64_t seg_cap = (int64_t)sms * 4;
    k_batch_rowinfo<<<rb + (int)(p.nseg < seg_cap ? p.nseg : seg_cap), 256, 0, s>>>(p, rb);
    k_batch_rowinfo_long<<<(int)(blocks < sms ? blocks : sms) * 4, 256, 0, s>>>(p);
}

using BatchKernel = void (*)(const BatchArgs *);
static BatchKernel batched_kernel(int dtype, bool wide) {
    if (dtype) return wide ? (BatchKernel)k_batched<double, true> : (BatchKernel)k_batched<double, false>;
    return wide ? (BatchKernel)k_batched<float, true> : (BatchKernel)k_batched<float, false>;
}

int batched_grid(int dtype, int warp_bytes, bool wide, int sms) {
    const size_t smem = batched_smem(dtype, warp_bytes, wide);
    BatchKernel k = batched_kernel(dtype, wide);
    int per = resident_per_sm((const void *)k, kBNT, smem);
    return per * sms;
}

int launch_batched(int dtype, const BatchArgs *p_dev, int warp_bytes, bool wide, int grid, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(kBNT, 1, 1);
    cfg.dynamicSmemBytes = batched_smem(dtype, warp_bytes, wide);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, batched_kernel(dtype, wide), p_dev);
    return e == cudaSuccess ? 0 : (int)e;
}

}  // namespace smash
