// Symbolic phase: the exact number of distinct columns of every row of C.
//
// Hashing Phase without values: every product's column tag is inserted into
// a per-row open-addressing table with compare-and-swap on EMPTY (= -1), +1
// linear probing on collision; the row's count is the number of successful
// inserts. Three table placements, by row size:
//   k_sym_hash   shared-memory table of 2^tbits int32 tags, one thread group
//                per row, rows claimed by atomic tokens (Version 2's
//                tokenization: a work counter instead of a static schedule);
//   k_sym_dense  the paper's "dense row": a bitmap over all columns of B in
//                shared memory (no probing), for rows whose bound is a large
//                fraction of cols(B);
//   k_sym_spill  the table in global memory (Version 3 moved it to DRAM), for
//                rows too large for shared memory when the bitmap does not fit.
#include "block_walk.cuh"
#include "device_common.cuh"
#include "kernels.h"
#include "launch_cache.h"

namespace smash {

template <int GS, int NT>
__global__ void __launch_bounds__(NT) k_sym_hash(Operands<float> op, const int *rows, int count, int *token,
                                                 int tbits, HashCfg hc, int *nnz_out, int *err) {
    using G = Group<GS, NT>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_row[2][G::kGroups];
    const int T = 1 << tbits;
    int *keys = (int *)smem + (size_t)G::gid() * T;
    // group scratch (GS > 32 only: warp rows enumerate from registers)
    unsigned char *scr = smem + (size_t)G::kGroups * T * 4 + (size_t)G::gid() * prod_scratch_bytes<float, GS>();
    const ProdScratch<float> sc = carve_prod_scratch<float, GS>(scr);
    const int t = G::tid();
    RowClaim<G> claim(token, s_row);
    for (;;) {
        const int r = claim.next(count);
        if (r >= count) break;
        const int i = rows[r];
        for (int s = t; s < T; s += GS) keys[s] = kEmpty;
        G::sync();
        int64_t ab, ae;
        a_row_range(op, i, ab, ae, err);
        int cnt = 0;
        // warp rows: the register-staged enumerator (measured faster here than
        // the shared-memory one, which the numeric warp rows use)
        auto ins_key = [&](int j, float, float) {
            bool ins;
            if (hash_find_or_insert<false>(keys, tbits, hc, j, ins) < 0) raise_err(err, kErrTableFull);
            cnt += ins ? 1 : 0;
        };
        if constexpr (GS == 32) warp_products<float, false>(op, ab, ae, err, ins_key);
        else group_products<float, false, GS, NT>(op, ab, ae, sc, err, ins_key);
        int tot;
        if constexpr (GS == 32) tot = warp_sum(cnt);
        else tot = G::template sum<int>(cnt, sc.red);
        if (t == 0) nnz_out[i] = tot;
        G::sync();
    }
}

// Size check of the numeric count pass (see NumCheck).
__device__ __forceinline__ void count_check(const NumCheck &nc, int i, int tot, int *err) {
    const int64_t s = nc.c_rp[i], t = nc.c_rp[i + 1];
    if (s < 0 || t < s || t > nc.c_nnz) {
        raise_err(err, kErrBadRowPtr);
        if (nc.row_nnz) nc.row_nnz[i] = -1;
        return;
    }
    if (nc.row_nnz) nc.row_nnz[i] = (int64_t)tot <= t - s ? tot : -1;
    else if ((int64_t)tot != t - s) raise_err(err, kErrCountMismatch);
}

// Word of a column's bit: an aligned group of 32 words keeps its place, the banks
// inside it are mixed with the bits above (the columns of skewed graphs crowd in
// words whose low bits are 0: 262,144-row square 3.64 -> 3.52 ms; a third field
// costs more instructions than it saves conflicts, 3.66 ms).
__device__ __forceinline__ unsigned bit_place(unsigned c) { return (c >> 5) ^ ((c >> 10) & 31u); }
constexpr int kSpareWords = 32;   // after the bitmap: hold the bit past the last column when it fills its words

// Dense rows: a bitmap over the columns of B; count = popcount. With wc.wcnt
// the row's distinct columns are also counted per block of kSubCols columns
// (slot = wc.slot_base + r), for the numeric dense kernel. The warps share the
// row's products (block_walk); a warp then takes every kWarps-th block of
// kSubCols columns, four words a lane, and counts and clears it in one pass.
// words: of the bitmap, a multiple of kSubCols / 32. Bound by the shared-memory
// pipe (71 % of the cycles: a test and mostly an atomic per product, the lanes'
// words spread over the banks at random) and instruction issue (61 %, some 27
// instructions per 32 products; 131,072-row skewed square, 1.10 ms).
// (Columns checked by a branch per product and steps of 32 products looked up
// with a vote each: 262,144-row square 4.04 ms, now 3.56; training samples and
// gradient at 65,536 rows 1.39 ms, now 1.19. No test before the atomic: 3.83 ms.)
template <int NT, typename IT>
__global__ void __launch_bounds__(NT) k_sym_dense(Operands<float> op, const int *rows, int count, int *token,
                                                  int words, int apart_from, WinCount wc, int *nnz_out, NumCheck nc,
                                                  int *err) {
    using G = Group<NT, NT>;
    constexpr int kWarps = NT / 32;
    constexpr int kSubWords = kSubCols / 32;
    static_assert(kSubWords == 128, "a warp counts a block of columns with one 16-byte load a lane");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_row[2][1];
    __shared__ int s_part[2][kWarps];   // the warps' counts of this row and of the one before
    unsigned *bm = (unsigned *)smem;
    const int t = threadIdx.x;
    const int lane = lane_id();
    const int wp = t >> 5;
    for (int x = t; x < words + kSpareWords; x += NT) bm[x] = 0u;
    RowClaim<G> claim(token, s_row);   // (its barrier ends the clearing)
    for (int par = 0;; par ^= 1) {
        const int r = claim.next(count);
        if (r >= count) break;
        const int i = rows[r];
        int64_t slot = -1;
        if (wc.wcnt && wc.skip_slotted) slot = wc.wslot[i];
        const bool counted = slot >= 0;   // counted before: only the size check
        int c = 0;
        if (counted) {
            for (int q = t; q < wc.nsub; q += NT) c += wc.wcnt[slot * wc.nsub + q];
            c = __reduce_add_sync(kFull, c);
        } else {
            int64_t ab, ae;
            a_row_range(op, i, ab, ae, err);
            // columns out of range share the bit past the last column: no
            // branch per product; the bits' words are read before any is set
            block_walk<float, IT, false, kWarps>(op, ab, ae, wp, ae - ab >= apart_from, err, [&](auto &j, auto &, auto &, auto &act) {
                constexpr int U = sizeof(act) / sizeof(act[0]);
                unsigned at[U], bit[U], had[U];   // (bits set meanwhile are set again)
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned c = min((unsigned)j[u], (unsigned)op.ncols);
                    at[u] = bit_place(c);
                    bit[u] = 1u << (c & 31);
                    had[u] = ~0u;
                    if (act[u]) had[u] = *(volatile unsigned *)(bm + at[u]);
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (!(had[u] & bit[u])) atomicOr(bm + at[u], bit[u]);
            });
            slot = wc.slot_base + r;
            __syncthreads();
            // the bit past the last column, by the warp that counts its word
            if (lane == 0 && wp == (op.ncols / kSubCols) % kWarps) {
                unsigned *w = bm + bit_place((unsigned)op.ncols);
                const unsigned bit = 1u << (op.ncols & 31);
                if (*w & bit) {
                    *w &= ~bit;
                    raise_err(err, kErrBadIndex);
                }
            }
            __syncwarp();
            for (int q = wp; q * kSubWords < words; q += kWarps) {
                uint4 *v = (uint4 *)(bm + q * kSubWords) + lane;
                const uint4 x = *v;
                *v = make_uint4(0u, 0u, 0u, 0u);
                const int n = __reduce_add_sync(kFull, __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w));
                c += n;
                if (wc.wcnt && lane == 0 && q < wc.nsub) wc.wcnt[slot * wc.nsub + q] = (uint16_t)n;
            }
            if (wc.wcnt && t == 0) wc.wslot[i] = (int)slot;
        }
        // A row counted before has this barrier alone: warp 0 may still read the
        // counts while the other warps write the next row's, into the other half.
        // They write this half again behind that row's barrier, which warp 0
        // reaches after its read.
        if (lane == 0) s_part[par][wp] = c;
        __syncthreads();
        if (wp == 0) {
            const int tot = __reduce_add_sync(kFull, lane < kWarps ? s_part[par][lane] : 0);
            if (lane == 0) {
                if (nnz_out) nnz_out[i] = tot;
                else count_check(nc, i, tot, err);
            }
        }
    }
}

// Spill rows: the key table lives in global memory, one slice per block.
template <int NT>
__global__ void __launch_bounds__(NT) k_sym_spill(Operands<float> op, const int *rows, int count, int *token,
                                                  HashCfg hc, float inv_load, const long long *bound,
                                                  int spill_tbits, int *tables, int *nnz_out, int *err) {
    using G = Group<NT, NT>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_row;
    const ProdScratch<float> sc = carve_prod_scratch<float, NT>(smem);
    int *keys = tables + ((size_t)blockIdx.x << spill_tbits);
    const int t = threadIdx.x;
    for (;;) {
        if (t == 0) s_row = atomicAdd(token, 1);
        __syncthreads();
        const int r = s_row;
        if (r >= count) break;
        const int i = rows[r];
        int tb = table_bits(bound[i], inv_load);
        if (tb > spill_tbits) {
            raise_err(err, kErrTableFull);
            tb = spill_tbits;
        }
        const int T = 1 << tb;
        for (int s = t; s < T; s += NT) __stcg(keys + s, kEmpty);
        __syncthreads();
        int64_t ab, ae;
        a_row_range(op, i, ab, ae, err);
        int cnt = 0;
        group_products<float, false, NT, NT>(op, ab, ae, sc, err, [&](int j, float, float) {
            bool ins;
            if (hash_find_or_insert<true>(keys, tb, hc, j, ins) < 0) raise_err(err, kErrTableFull);
            cnt += ins ? 1 : 0;
        });
        const int tot = G::template sum<int>(cnt, sc.red);
        if (t == 0) nnz_out[i] = tot;
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
static Operands<float> sym_operands(const RawOperands &r) {
    Operands<float> o;
    o.a_rp = r.a_rp;
    o.a_ci = r.a_ci;
    o.a_val = nullptr;
    o.b_rp = r.b_rp;
    o.b_ci = r.b_ci;
    o.b_val = nullptr;
    o.a_nnz = r.a_nnz;
    o.b_nnz = r.b_nnz;
    o.b_rows = r.b_rows;
    o.ncols = r.ncols;
    return o;
}


template <typename K>
static int resident_grid(K kernel, int nt, size_t smem, int sms, int want_blocks, int cap_per_sm = 64) {
    int per_sm = resident_per_sm((const void *)kernel, nt, smem);
    if (per_sm < 1) per_sm = 1;
    if (per_sm > cap_per_sm) per_sm = cap_per_sm;
    long long cap = (long long)per_sm * sms;
    return (int)(want_blocks < cap ? want_blocks : cap);
}

template <int GS, int NT>
static void sym_hash_launch(const Operands<float> &op, const int *rows, int count, int *token, int tbits,
                            HashCfg hc, int sms, int *nnz_out, int *err, cudaStream_t s) {
    constexpr int groups = NT / GS;
    const size_t smem = (size_t)groups * ((size_t)4 << tbits) +
                        (GS > 32 ? (size_t)groups * prod_scratch_bytes<float, GS>() : 0);
    auto kern = k_sym_hash<GS, NT>;
    allow_smem((const void *)kern);
    const int want = (count + groups - 1) / groups;
    const int grid = resident_grid(kern, NT, smem, sms, want);
    kern<<<grid, NT, smem, s>>>(op, rows, count, token, tbits, hc, nnz_out, err);
}

static int threads_per_row(int tbits, int shift) {
    int t = 1 << (tbits > shift ? tbits - shift : 0);
    if (t < 32) t = 32;
    if (t > 1024) t = 1024;
    return t;
}

void launch_sym_hash(const RawOperands &r, const int *rows, int count, int *token, const HashLaunch &hl,
                     int *nnz_out, int *err, cudaStream_t s) {
    if (count <= 0) return;
    const Operands<float> op = sym_operands(r);
    const HashCfg hc{hl.hash_kind, hl.colbits};
    switch (threads_per_row(hl.tbits, hl.group_shift)) {
        case 32: sym_hash_launch<32, 256>(op, rows, count, token, hl.tbits, hc, hl.sms, nnz_out, err, s); break;
        case 64: sym_hash_launch<64, 64>(op, rows, count, token, hl.tbits, hc, hl.sms, nnz_out, err, s); break;
        case 128: sym_hash_launch<128, 128>(op, rows, count, token, hl.tbits, hc, hl.sms, nnz_out, err, s); break;
        case 256: sym_hash_launch<256, 256>(op, rows, count, token, hl.tbits, hc, hl.sms, nnz_out, err, s); break;
        case 512: sym_hash_launch<512, 512>(op, rows, count, token, hl.tbits, hc, hl.sms, nnz_out, err, s); break;
        default: sym_hash_launch<1024, 1024>(op, rows, count, token, hl.tbits, hc, hl.sms, nnz_out, err, s); break;
    }
}

static size_t sym_dense_words(int64_t ncols) { return (size_t)((ncols + kSubCols - 1) / kSubCols) * (kSubCols / 32); }

// Block size and blocks per SM of the bitmap kernel: as many resident
// threads as the bitmaps allow, then as many rows in flight as possible (or
// the requested blocks per SM).
static void sym_dense_shape(const HashLaunch &hl, int64_t ncols, int &nt, int &per_sm) {
    const size_t words = sym_dense_words(ncols);
    const int sm_smem = max_smem_per_sm();
    const int nts[3] = {1024, 512, 256};
    int best_nt = 1024, best_b = 1, best_thr = 0;
    for (int q = 0; q < 3; ++q) {
        if (best_thr == (1 << 30)) break;
        const size_t per_block = (words + kSpareWords) * 4 + 320 + 1024;   // static variables, reserved by the driver
        if (per_block > (size_t)max_smem_per_block() + 1024) continue;
        int b = (int)((size_t)sm_smem / per_block);
        if (b > 2048 / nts[q]) b = 2048 / nts[q];
        if (b < 1) continue;
        if (hl.sym_dense_blocks > 0) {
            if (b >= hl.sym_dense_blocks && nts[q] * hl.sym_dense_blocks <= 2048) {
                best_nt = nts[q];
                best_b = hl.sym_dense_blocks;
                best_thr = 1 << 30;
            }
            continue;
        }
        if (b * nts[q] > best_thr || (b * nts[q] == best_thr && b > best_b)) {
            best_thr = b * nts[q];
            best_nt = nts[q];
            best_b = b;
        }
    }
    nt = best_nt;
    per_sm = best_b;
}

int sym_dense_threads(const HashLaunch &hl, int64_t ncols) {
    int nt, b;
    sym_dense_shape(hl, ncols, nt, b);
    return nt;
}

template <int NT>
static void sym_dense_go(const Operands<float> &op, const int *rows, int count, int apart_from, int *token, int per_sm,
                         const HashLaunch &hl, const WinCount &wc, int *nnz_out, const NumCheck &nc, int *err,
                         cudaStream_t s) {
    const int words = (int)sym_dense_words(op.ncols);
    const size_t smem = (size_t)(words + kSpareWords) * 4;
    auto kern = op.b_nnz < INT_MAX ? k_sym_dense<NT, int32_t> : k_sym_dense<NT, int64_t>;
    allow_smem((const void *)kern);
    const int grid = resident_grid(kern, NT, smem, hl.sms, count, per_sm);
    kern<<<grid, NT, smem, s>>>(op, rows, count, token, words, apart_from, wc, nnz_out, nc, err);
}

void launch_sym_dense(const RawOperands &r, const int *rows, int count, long long entries, long long products,
                      int *token, const HashLaunch &hl, const WinCount &wc, int *nnz_out, const NumCheck &nc, int *err,
                      cudaStream_t s) {
    if (count <= 0) return;
    const Operands<float> op = sym_operands(r);
    int nt, per_sm;
    sym_dense_shape(hl, r.ncols, nt, per_sm);
    const int apart_from = walk_apart_from(entries, products, nt / 32);
    if (nt == 256) sym_dense_go<256>(op, rows, count, apart_from, token, per_sm, hl, wc, nnz_out, nc, err, s);
    else if (nt == 512) sym_dense_go<512>(op, rows, count, apart_from, token, per_sm, hl, wc, nnz_out, nc, err, s);
    else sym_dense_go<1024>(op, rows, count, apart_from, token, per_sm, hl, wc, nnz_out, nc, err, s);
}

int sym_spill_grid(const HashLaunch &hl) {
    const int per = hl.blocks_per_sm > 0 ? hl.blocks_per_sm : 1;
    return hl.sms * per;
}

void launch_sym_spill(const RawOperands &r, const int *rows, int count, int *token, const HashLaunch &hl,
                      float inv_load, const long long *bound, int spill_tbits, int *tables, int *nnz_out,
                      int *err, cudaStream_t s) {
    if (count <= 0) return;
    const Operands<float> op = sym_operands(r);
    const HashCfg hc{hl.hash_kind, hl.colbits};
    const size_t smem = prod_scratch_bytes<float, 1024>();
    auto kern = k_sym_spill<1024>;
    int grid = sym_spill_grid(hl);
    if (grid > count) grid = count;
    kern<<<grid, 1024, smem, s>>>(op, rows, count, token, hc, inv_load, bound, spill_tbits, tables, nnz_out, err);
}

}  // namespace smash
