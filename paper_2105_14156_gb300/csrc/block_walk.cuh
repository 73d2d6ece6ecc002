// Products of one row of A shared out over the warps of a block without
// staging or barriers, for the kernels whose block owns one accumulator (the
// column windows of the numeric phase, the column bitmap of the symbolic one).
//
// Every warp loads each batch of 32 entries of the row for itself (lane l:
// where entry l's row of B starts, its length, a_ik; the warps' loads of the
// same words hit in L1), lays the batch's products on one line with a scan, and
// walks its own kWarps-th part of the line. Inside a row of B of which at least
// kWalkAlone products are left, up to four coalesced loads are issued per lane
// and round and nothing else is done per product; shorter pieces take steps of
// 32 products that may span several rows of B (a lane's entry is the number of
// entries that end at or before its product: some 12 instructions a step more,
// against the idle lanes of a piece's last step).
//
// Measured against staging the entries in shared memory with a block scan and
// three barriers a batch, and finding the entry in every step (group_products):
// the bitmap pass of the skewed 262,144-row square (2.8 G products) 5.9 -> 3.6 ms
// (61 -> 33 instructions per 32 products), the float64 windows of the 65,536-row
// one 4.0 -> 3.9 ms (bound by the adds), whole calls 6.06 -> 4.22 ms and 6.51 ->
// 6.03 ms. With whole rounds inside shorter rows of B (kWalkAlone 48 instead of
// 128; 33 and 80 are no better), steps that carry their first entry instead of
// looking it up with a vote, and fewer instructions per bit: 3.54 and 5.61 ms, and
// the one-pass float32 131,072-row square 11.05 -> 10.65 ms.
#pragma once

#include <climits>

#include "device_common.cuh"

namespace smash {

// Position of the n-th (0-based) set bit of x (n < popc(x)), by halving.
__device__ __forceinline__ int nth_set_bit(unsigned x, int n) {
    int pos = 0;
    int c = __popc(x & 0xffffu);
    if (n >= c) { n -= c; x >>= 16; pos += 16; }
    c = __popc(x & 0xffu);
    if (n >= c) { n -= c; x >>= 8; pos += 8; }
    c = __popc(x & 0xfu);
    if (n >= c) { n -= c; x >>= 4; pos += 4; }
    c = __popc(x & 0x3u);
    if (n >= c) { n -= c; x >>= 2; pos += 2; }
    if (n >= (int)(x & 1u)) pos += 1;
    return pos;
}

// Where a column's accumulator lies in shared memory. Columns of skewed graphs
// crowd at multiples of powers of two (a low bit of an R-MAT column is 0 with
// probability .76, so a quarter of them would share one of the 32 banks); the
// low five bits are mixed with the five above, which keeps every aligned group
// of 32 columns in its place. (Skewed squares, none / these five bits / ten bits
// and the bitmap's words as well: one-pass float32 131,072 rows 10.84 / 10.49 /
// 10.65 ms, float64 65,536 rows 5.62 / 5.58 / 5.61 ms.)
__device__ __forceinline__ unsigned column_place(unsigned off) { return off ^ ((off >> 5) & 31u); }

constexpr int kWalkUnroll = 4;
constexpr int kWalkAlone = 48;

// The least entries of A from which a row's warps take whole batches in turn
// (apart) instead of a part of each. entries, products: of the rows of a launch
// (entries once for each window); warps: of a block. Every warp loads and scans
// each batch that it has a part of, which costs more than walking the part where
// the rows of B are short: every row below 6 products an entry, the rows with three
// batches below kWalkShort, with one for every fourth warp below kWalkShort * 2, with
// one for every warp below kWalkMedium.
// (Values of 800 dense rows of 100,000 columns, 13,750 entries of 8 products, in
// parts and apart: float 6.21 and 1.13 ms, double 12.3 and 1.27 ms; 5,500 of 20: 2.65
// and 0.68, 5.18 and 0.84 ms. Counts of rows of 1,100 entries of 8: 154 and 110 us; of
// 59 entries of 50 products 121 us in parts, 145 us apart; values of 25,510 rows of 49
// entries of 12, 1,024 columns: 350 and 391 us. The skewed float64 square
// of 65,536 rows: 5.49 ms in parts, 5.52 so, 5.84 with a batch for every fourth
// warp below kWalkMedium, 9.6 with every row apart.)
constexpr int kWalkShort = 16, kWalkMedium = 128;
inline int walk_apart_from(long long entries, long long products, int warps) {
    if (products < 6 * entries) return 0;
    if (products < kWalkShort * entries) return 96;
    if (products < kWalkShort * 2 * entries) return 8 * warps > 128 ? 8 * warps : 128;
    return products < kWalkMedium * entries ? 32 * warps : INT_MAX;
}

// One round of S steps of 32 products from product q of the batch's line on (q to
// hi are the warp's): the entries that end inside a step are one OR-reduction of
// shifted bits, which also advances the first entry of the next step (c0). No
// step is skipped by a branch: past hi it only idles.
template <typename V, typename IT, bool NUM, int S, typename F>
__device__ __forceinline__ void walk_steps(const Operands<V> &op, int incl, IT start, V av, int q, int hi, int &c0,
                                           F &&f) {
    const int lane = lane_id();
    const unsigned lt = lanemask_lt();
    int jv[S];
    V a_u[S], b_u[S];
    bool act[S];
#pragma unroll
    for (int u = 0; u < S; ++u) {
        const int p = q + 32 * u;
        const unsigned ends = __reduce_or_sync(kFull, bit_or_none(incl - 1 - p));
        const int ci = (c0 + __popc(ends & lt)) & 31;   // (past the last product: any lane)
        c0 += __popc(ends);
        const IT idx = __shfl_sync(kFull, start, ci) + (IT)(p + lane);
        a_u[u] = V(0);
        b_u[u] = V(0);
        if constexpr (NUM) a_u[u] = __shfl_sync(kFull, av, ci);
        jv[u] = 0;
        act[u] = p + lane < hi;
        if (act[u]) {
            jv[u] = __ldg(op.b_ci + idx);
            if constexpr (NUM) b_u[u] = __ldg(op.b_val + idx);
        }
    }
    f(jv, a_u, b_u, act);
}

// f(j, a, b, act) for every product of A entries [ab, ae) in warp w's share, two
// or four a lane at a time (arrays; j: the columns, checked by f, 0 where the
// lane holds no product (act); a, b: 0 when !NUM). With a sliced B only the
// entries of op.slice. All 32 lanes call it; f may diverge. IT: type of the
// positions in B (int32_t when B has fewer than 2^31 entries).
// apart: the warps take whole batches in turn instead of a part of each.
template <typename V, typename IT, bool NUM, int kWarps, typename F>
__device__ __forceinline__ void block_walk(const Operands<V> &op, int64_t ab, int64_t ae, int w, bool apart, int *err,
                                           F &&f) {
    const int lane = lane_id();
    const int step = apart ? 32 * kWarps : 32;
    for (int64_t base = apart ? ab + 32 * w : ab; base < ae; base += step) {
        int len = 0;
        int64_t bs64 = 0;
        V av = V(0);
        if (base + lane < ae) load_a_entry<V, NUM>(op, base + lane, len, bs64, av, err);
        IT bs = (IT)bs64;
        const unsigned nz = __ballot_sync(kFull, len > 0);
        if (nz == 0u) continue;
        const int nv = __popc(nz);
        if (nv < 32 && nz != (1u << nv) - 1u) {
            // entries without products move out of the way
            const int src = lane < nv ? nth_set_bit(nz, lane) : 0;
            len = __shfl_sync(kFull, len, src);
            bs = __shfl_sync(kFull, bs, src);
            if constexpr (NUM) av = __shfl_sync(kFull, av, src);
            if (lane >= nv) len = 0;
        }
        const int incl = warp_incl_scan(len);
        const int total = __shfl_sync(kFull, incl, 31);
        const IT start = bs - (IT)(incl - len);   // product p of this entry reads B at start + p
        const int per = apart ? total : (total + kWarps - 1) / kWarps;
        int q = apart ? 0 : min(w * per, total);
        const int hi = min(q + per, total);
        int c0 = __popc(__ballot_sync(kFull, incl <= q));   // entry of product q (any past the last)
        while (q < hi) {
            const int last = __shfl_sync(kFull, incl, c0);
            const int end = last < hi ? last : hi;
            if (end - q >= kWalkAlone) {
                int jv[kWalkUnroll];
                V a_u[kWalkUnroll], b_u[kWalkUnroll];
                bool act[kWalkUnroll];
                const IT st = __shfl_sync(kFull, start, c0) + (IT)lane;
                V a = V(0);
                if constexpr (NUM) a = __shfl_sync(kFull, av, c0);
                const int32_t *pc = op.b_ci + st;
                const V *pv = op.b_val + st;
#pragma unroll
                for (int u = 0; u < kWalkUnroll; ++u) a_u[u] = a;
                for (; end - q >= 32 * kWalkUnroll; q += 32 * kWalkUnroll) {
#pragma unroll
                    for (int u = 0; u < kWalkUnroll; ++u) {
                        act[u] = true;
                        jv[u] = __ldg(pc + q + 32 * u);
                        b_u[u] = V(0);
                        if constexpr (NUM) b_u[u] = __ldg(pv + q + 32 * u);
                    }
                    f(jv, a_u, b_u, act);
                }
                if (end - q >= kWalkAlone) {
#pragma unroll
                    for (int u = 0; u < kWalkUnroll; ++u) {
                        act[u] = q + 32 * u + lane < end;
                        jv[u] = 0;
                        b_u[u] = V(0);
                        if (act[u]) {
                            jv[u] = __ldg(pc + q + 32 * u);
                            if constexpr (NUM) b_u[u] = __ldg(pv + q + 32 * u);
                        }
                    }
                    f(jv, a_u, b_u, act);
                    q = end;
                }
                if (q == last) ++c0;
            } else if (hi - q > 32 * (kWalkUnroll / 2)) {
                walk_steps<V, IT, NUM, kWalkUnroll>(op, incl, start, av, q, hi, c0, f);
                q += 32 * kWalkUnroll;
            } else {
                walk_steps<V, IT, NUM, kWalkUnroll / 2>(op, incl, start, av, q, hi, c0, f);
                q += 32 * (kWalkUnroll / 2);
            }
            __syncwarp();
        }
    }
    __syncwarp();
}

}  // namespace smash
