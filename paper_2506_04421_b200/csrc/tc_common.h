// Argument structures shared by the tensor-core kernels and their host-side dispatch (internal).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <algorithm>
#include "hmar_common.h"

namespace hmar {

// Device form of a forward work tile: query rows [row_begin, row_begin + row_count) and up to two key
// segments (second one used by the inference step only: previous scale, then current scale).
struct FwdWork {
    int32_t row_begin, row_count;
    int32_t s0_begin, s0_end;
    int32_t s1_begin, s1_end;
    int32_t uniform;
    int32_t pad;
};

// Division of numbers below 2^31 by a number that the host knows: q = (hi(n * mul) + n) >> shift with mul = 2^32 * (2^shift / d - 1)
// rounded up and shift = ceil(log2(d)) (Granlund and Montgomery, "Division by invariant integers using multiplication").
// A division by a variable is some forty instructions, and every block of the forward began with three of them, in all of its
// warps: 1 100 clocks of a block's 11 000 to 69 000.  Kernel times, taken as fwd_sm100.cu says: L = 680 960 heads 127 -> 121 us, L = 2240 384 heads 346 -> 338, L = 384 128
// heads 17.7 -> 16.6, inference step 13 -> 18 1536 heads 143 -> 139, 24 -> 32 384 heads 224 -> 219.5.
struct FastDiv {
    uint32_t mul = 0, shift = 0;
    FastDiv() = default;
    constexpr explicit FastDiv(uint32_t d) {
        shift = d > 1 ? 32 - __builtin_clz(d - 1) : 0;
        mul = (uint32_t)(((1ull << 32) * ((1ull << shift) - d) + d - 1) / d);
    }
    HMAR_HD constexpr int operator()(int n) const {
        return (int)(((uint32_t)(((uint64_t)(uint32_t)n * mul) >> 32) + (uint32_t)n) >> shift);
    }
};
static_assert(FastDiv(1)(0x7fffffff) == 0x7fffffff && FastDiv(2)(0x7fffffff) == 0x3fffffff && FastDiv(3)(0x7ffffffd) == 0x2aaaaaa9 &&
              FastDiv(7)(0x7ffffffe) == 306783378 && FastDiv(7)(306783378 * 7 - 1) == 306783377 && FastDiv(641)(640) == 0 &&
              FastDiv(0x7fffffff)(0x7fffffff) == 1 && FastDiv(0x7fffffff)(0x7ffffffe) == 0, "division at the ends of its range");

struct FwdArgs {
    const FwdWork* work;     // n_work tiles per head; nullptr = inference step (tiles derived in-kernel)
    int n_work;
    int n_q_rows;            // rows per head of q / out / lse
    size_t head_bytes;       // Q, K and V of one head
    int n_heads;             // set by the launcher, as group_heads: the blocks go group by group of this many heads, and
    int group_heads;         // tile by tile over the heads of a group
    int heads_per_batch;     // H: head bh is head bh % H of batch bh / H (the tensor maps are 4-D: D, rows, H, B)
    FastDiv by_group, by_group_heads, by_last_heads, by_batch;      // set by the launcher: group_heads * n_work (an inference step: n_work),
                             // heads of a group, heads of the last group, heads_per_batch
    long long out_row_stride, out_head_stride, out_batch_stride;   // of `out`, in elements (lse is always [B*H, rows])
    long long out_extent, lse_extent;   // elements reachable through out / lse (read by the checking build only)
    int n0, n1;              // inference step: rows of the previous / current scale's keys
    float scale_log2;        // softmax_scale * log2(e)
    __nv_bfloat16* out;
    float* lse;              // may be nullptr
    int* status;             // device status word {code, detail}, may be nullptr
    ScaleTable st;
};

// Backward work tile: key rows [row_begin, row_begin + row_count) and the query range that may see them.
struct BwdWork {
    int32_t row_begin, row_count;
    int32_t q_begin, q_end;
    int32_t uniform;
    int32_t class_count;     // tiles of the head that cost as much as this one; they follow one another (see bwd_fill_classes)
    int32_t pad[2];
};

// A head's tiles in classes of equal cost (equal numbers of 128-query steps), the costliest first; returns the sum of
// the steps.
inline int bwd_fill_classes(BwdWork* work, int n) {
    auto steps = [](const BwdWork& w) { return (w.q_end - w.q_begin + 127) / 128; };
    std::stable_sort(work, work + n, [&](const BwdWork& a, const BwdWork& b) { return steps(a) > steps(b); });
    for (int i = 0, first = 0; i <= n; ++i) {
        if (i < n && steps(work[i]) == steps(work[first])) continue;
        for (int k = first; k < i; ++k) work[k].class_count = i - first;
        first = i;
    }
    int total = 0;
    for (int i = 0; i < n; ++i) total += steps(work[i]);
    return total;
}

// Share, in thousandths, of a head's steps that belong to full tiles (128 key rows that all see the whole query
// range): those run without any mask code.
inline int bwd_plain_permille(const BwdWork* work, int n) {
    long long plain = 0, total = 0;
    for (int i = 0; i < n; ++i) {
        const int steps = (work[i].q_end - work[i].q_begin + 127) / 128;
        total += steps;
        if (work[i].uniform && work[i].row_count == 128) plain += steps;
    }
    return total > 0 ? (int)(plain * 1000 / total) : 1000;
}

constexpr size_t kL2Bytes = 126u << 20;      // L2 of the one part this library is built for

// Whether the backward's items go head by head instead of class by class.  Class by class a head's rows are read once per
// class.  Where its items are short (a mean of fewer than four steps) and the tensors do not stay in L2, that costs more than
// the balance gives: head by head L = 680 960 heads 311 -> 285 us, L = 395 768 heads 148 -> 132.  Otherwise it is the other
// way round: L = 680 128 heads 53.3 against 49.5, L = 1000 192 heads 100 against 96.6, L = 2240 96 heads 200 against 185.
inline bool bwd_by_head(int head_steps, int n_work, size_t n_rows) {
    const size_t row_bytes = 4 * kHeadDim * sizeof(__nv_bfloat16) + kHeadDim * sizeof(float);     // Q, K, V, dO and the dQ accumulator
    return head_steps < 4 * n_work && n_rows * row_bytes > kL2Bytes + kL2Bytes / 4;
}

// Whether the backward runs the instantiation whose code holds one variant of the softmax-gradient code, with a bit per column, and
// not three (none, rows only, columns).  It is the better one where few steps belong to full tiles, and the line lies higher where
// the items go head by head: tiles of all kinds follow one another there, and with them the variants of the code.  Whole backward, one
// variant / three.  Class by class, 25 000 to 190 000 rows: mean 0.94 (0.79 to 1.01) at shares of 330 to 400, 0.99 (0.83 to 1.04)
// from 400 to 500, 1.02 (0.95 to 1.07; a single list of 500: 0.94) from 515 to 570, 1.05 (0.98 to 1.12) above.  Head by head, 230 000 to
// 800 000 rows: 0.84 (0.74 to 0.95) up to 490, 0.93 (0.82 to 1.02) to 600, 0.94 (0.81 to 1.04) to 700, 0.98 (0.87 to 1.05) to
// 900, 1.04 (1.01 to 1.07) above.  (L = 680, share 421: 0.84 with 960 heads, 1.00 with 128.)
inline bool bwd_one_mask(int plain_permille, bool by_head) { return plain_permille < (by_head ? 700 : 500); }

// The item that a block takes in a round: returns its tile and sets its head, or returns -1 where there are no more.
// A head's tiles are ordered by cost; tiles of equal cost are one class.  The launch works class by class, head by head
// inside a class (by_head: all tiles are one class), and the items are dealt to the blocks round by round, back and forth.
// The blocks' sums then differ by 0.6 % (L = 9451, 192 heads) where a stretch or several runs of heads per block differed by
// 12 %, and the blocks work on few heads at a time: at L = 2240 18, whose dQ accumulators stay in L2.
HMAR_HD int bwd_deal(const BwdWork* work, int n_work, int n_heads, int by_head, int n_blocks, int block, int round, int& head) {
    int pos = round * n_blocks + ((round & 1) ? n_blocks - 1 - block : block);
    if (pos >= n_heads * n_work) return -1;
    int t = 0, count = by_head ? n_work : work[0].class_count;
    while (pos >= n_heads * count) {
        pos -= n_heads * count;
        t += count;
        count = work[t].class_count;
    }
    head = pos / count;
    return t + pos - head * count;
}

struct BwdArgs {
    const BwdWork* work;
    int n_work;
    int n_heads;             // B * H
    int plain_permille;      // from bwd_plain_permille: picks the instantiation of the main kernel, see bwd_one_mask
    int head_steps;          // steps of all tiles of a head (from bwd_fill_classes)
    int by_head;             // set by the launcher (bwd_by_head)
    int L;
    float scale_log2;        // softmax_scale * log2(e)
    float softmax_scale;
    const float* lse;        // [BH, L] from the forward
    const float* delta;      // [BH, L] rowsum(dO o O) (read by the main kernel)
    float* delta_w;          // same buffer, written by the preprocess kernel
    float* dq_acc;           // [BH, L, 64] fp32 accumulator
    // Layout of the bf16 tensors: head bh is head bh % heads_per_batch of batch bh / heads_per_batch, and element
    // (batch, head, row, d) sits at batch * *_batch + head * *_head + row * *_row + d (strides in elements).  q, k, v
    // share the `in` strides, out and dout the `od` strides, dq, dk, dv the `g` strides; lse, delta and the fp32 dQ
    // accumulator are always dense [BH, L(, 64)].
    int heads_per_batch;
    long long in_row, in_head, in_batch;
    long long od_row, od_head, od_batch;
    long long g_row, g_head, g_batch;
    long long in_extent, g_extent;      // elements reachable through v and through dk / dv (checking build only)
    const __nv_bfloat16* v;  // read directly for the rows that go to TMEM
    __nv_bfloat16* dk;
    __nv_bfloat16* dv;
    int* status;
    ScaleTable st;
};

// Whether the backward's tensors are all dense [B*H, L, 64]: the instantiation with compile-time strides.  It takes a head by its
// number alone, as the tensor maps of one batch of B*H heads do.  Maps of several batches want the head's number inside its batch,
// also where the batches follow one another: theirs would end before a head past the first batch, whose rows would be loaded as
// zeros and whose dK and dV would not be stored.
constexpr bool bwd_dense(const BwdArgs& a) {
    const long long row = kHeadDim, head = (long long)a.L * kHeadDim;
    return a.heads_per_batch == a.n_heads && a.in_row == row && a.od_row == row && a.g_row == row && a.in_head == head && a.od_head == head &&
           a.g_head == head;
}
constexpr BwdArgs bwd_layout_example(int heads_per_batch, int n_heads, int L, long long row, long long head, long long batch) {
    BwdArgs a{};
    a.heads_per_batch = heads_per_batch;
    a.n_heads = n_heads;
    a.L = L;
    a.in_row = a.od_row = a.g_row = row;
    a.in_head = a.od_head = a.g_head = head;
    a.in_batch = a.od_batch = a.g_batch = batch;
    return a;
}
static_assert(bwd_dense(bwd_layout_example(6, 6, 30, 64, 1920, 11520)) && !bwd_dense(bwd_layout_example(3, 6, 30, 64, 1920, 5760)) &&
              !bwd_dense(bwd_layout_example(3, 6, 30, 576, 64, 17280)) && !bwd_dense(bwd_layout_example(6, 6, 30, 64, 1984, 11904)),
              "one batch of dense heads; dense batches, the packed layout and heads apart are strided");

size_t fwd_tc_smem_bytes();
cudaError_t launch_selftest_wait(int* status, cudaStream_t stream);
cudaError_t launch_bwd_tc(const CUtensorMap& q, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& dout_map,
                          const CUtensorMap& dq_acc_map, const CUtensorMap& dk_map, const CUtensorMap& dv_map, const BwdArgs& args,
                          const __nv_bfloat16* out, const __nv_bfloat16* dout, __nv_bfloat16* dq, int BH, cudaStream_t stream);
cudaError_t launch_fwd_tc(const CUtensorMap& q, const CUtensorMap& k0, const CUtensorMap& v0, const CUtensorMap& k1,
                          const CUtensorMap& v1, const FwdArgs& args, int BH, cudaStream_t stream);

}  // namespace hmar
