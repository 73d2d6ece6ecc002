// Shared definitions of the batched path (device kernel and host driver).
#pragma once

#include <cstdint>

#include "device_common.cuh"

namespace smash {

constexpr int kBW = 8;                 // warps per block
constexpr int kBNT = kBW * 32;

// Classification of a row.
enum : uint8_t { kRowEmpty = 0, kRowSmall = 1, kRowBig = 2, kRowHuge = 3, kRowMed = 4 };
// Products of a narrow row (its product's B fits a warp's dense accumulator):
// up to kMedFlop it is served with its neighbours (a warp claims 32 rows at
// once), up to kBigFlop by a warp that claims it alone, above by a block.
// (512 products of 256 columns, skewed, ms: kMedFlop 128 1.69, 512 1.66, 2,048 1.79;
// kBigFlop 2,048 1.76, 8,192 and 32,768 1.66; 24 products of 3,000 columns 0.36 with
// kBigFlop 2,048, 0.34 with 8,192, 0.35 with 32,768.)
constexpr int kMedFlop = 512;
constexpr int kBigFlop = 8192;
constexpr int kBatchLongRow = 512;   // products above which a row outgrows the default warp table
constexpr int kSegEntries = 8192;
constexpr int kSegRows = 2048;

struct BatchMat {
    const int64_t *a_rp;
    const int32_t *a_ci;
    const void *a_val;
    const int64_t *b_rp;
    const int32_t *b_ci;
    const void *b_val;
    int64_t a_nnz;
    int64_t b_nnz;
    int32_t a_rows;
    int32_t b_rows;
    int32_t ncols;
    int32_t mode;     // dense accumulator of a warp (warp_dense.cuh), -1: B too wide, hash tables
    int64_t row_off;  // first row of this product in the flattened row space
    int64_t seg_off;  // first of its segments in the pass over the narrow B (segments of kSegEntries
                      // entries, then of kSegRows rows)
};

struct BatchArgs {
    const BatchMat *mats;
    int nmat;
    int64_t nrows;          // all products' rows
    const int64_t *row_start;   // [nmat+1]
    uint8_t *cls;           // [nrows]
    int *ub;                // [nrows] min(flop, cols)
    int *nnz;               // [nrows]
    int *big;               // [nrows] list of big rows
    int *huge;              // [nrows] list of huge rows
    int *med;               // [nrows] list of narrow rows claimed one at a time
    int *longs;             // [nrows] list of rows counted by a warp (k_batch_rowinfo_long)
    int *counters;          // [16]: 0 nbig, 1 nhuge, 2..3 item tokens, 4 med token, 5 matrix token, 6..7 barrier,
                            // 8..9 row-chunk tokens of the two row phases, 12 nmed, 13 nlong
    unsigned long long *sums;   // [4]: sum ub, sum flop, flop of long rows (kBatchLongRow) of products with a large accumulator
    int large_cols;             // columns above which an accumulator is large
    long long *descents;    // [nmat] 0: every row of B ascends (warp_dense.cuh)
    int64_t nseg;           // segments of all products
    int chunk;              // rows a warp claims at once (1 .. 32)
    int64_t *rp_pool;       // row pointers: product m at row_start[m] + m
    int32_t *ci_pool;
    void *val_pool;
    int64_t *base;          // [nmat+1] first entry of product m in the pools
    int64_t *totals;        // [nmat]
    int *err;
    int tw_bits;            // per-warp table: 2^tw_bits slots
    int warp_bits;          // rows whose table needs at most 2^warp_bits slots: one warp (<= tw_bits)
    int block_bits;         // ... at most 2^block_bits slots: the whole block (<= tw_bits + 3); larger:
                            // the regular per-product path
    int warp_bytes;         // shared memory of one warp: its table or dense accumulator
    int dense_words;        // words of the widest dense accumulator
    HashCfg hc;             // colbits filled per product
    float inv_load;
    // narrow rows take one pass: the first phase computes their values and
    // stages each sorted row at stage_off[g] (room: min(flop, cols)); the last
    // phase copies it to its exact place
    const int64_t *stage_off;
    int32_t *stage_ci;
    void *stage_val;
    long long wait_spins;   // a grid barrier gives up after this many polls (~256 ns each)
    int missing;            // test hook: arrivals a barrier waits for beyond the grid (0: none)
};

// Shared memory of a block whose warps have warp_bytes each; wide: some B is
// too wide for a dense accumulator (its rows take hash tables).
size_t batched_smem(int dtype, int warp_bytes, bool wide);
size_t batched_table_bytes(int dtype, int tw_bits);   // a warp's table of 2^tw_bits slots
void launch_batch_rowinfo(const BatchArgs &p, int sms, cudaStream_t s);
int batched_grid(int dtype, int warp_bytes, bool wide, int sms);
// p_dev: the arguments in device memory (read by every block at start).
int launch_batched(int dtype, const BatchArgs *p_dev, int warp_bytes, bool wide, int grid, cudaStream_t s);

}  // namespace smash
