// Backward kernels of HMAR's Markovian block-sparse attention for sm_100a.
//
// The gradient of exact softmax attention is recomputed from the forward's lse (the paper benchmarks
// this pass in App. B.4; Sec. 4.1 builds the kernel on FlashAttention, whose backward this follows):
//   P = exp(scale * Q K^T - lse),  dV = P^T dO,  dP = dO V^T,  dS = P o (dP - delta),
//   dQ = scale * dS K,  dK = scale * dS^T Q,  delta_i = sum_d dO_id O_id.
//
// Main kernel: persistent blocks, one per SM.  A work item is one tile of up to 128 key rows of one
// head; the block walks over the contiguous range of query rows that may see them under the mask
// (queries of the keys' own scale and of the next scale; paper Sec. 4.1, Fig. attn-mask), 128 queries
// (one step) at a time.  A step is split into two halves of 64 queries with their own TMEM columns and
// barriers; each half belongs to one compute warpgroup, so the two warpgroups and the tensor core work
// on different halves at the same time.  The steps of all items of a block form one pipeline: while the
// warpgroups work on an item's last step the tensor core already computes the next item's first scores.
//   warps 0-3   compute warpgroup of half 0: 32 key rows per warp, 64 query columns.  P^T and dS^T in
//               fp32 with packed two-float instructions; P^T (bf16) goes back to TMEM over S^T, dS^T
//               (bf16) goes to TMEM over dP^T (A operand of dK) and to shared memory (A operand of dQ)
//   warps 4-7   the same for half 1
//   warps 8-11  per step: drain dQ_i from TMEM through a staging buffer into the fp32 accumulator with
//               bulk tensor reductions (cp.reduce.async.bulk.tensor).  Per item: copy the next item's K
//               and V rows into TMEM as soon as the current item's last scores are done, and write the
//               finished dK, dV (scaled, bf16; by bulk tensor stores where a warp's 32 rows are all the tile's), V, dK and dV
//               as whole rows per instruction
//   warp 12     TMA producer: K per item (two buffers); Q_i, dO_i through a 3-stage ring
//   warp 13     issues tcgen05.mma.  K and V in TMEM are the A operands of S^T = K Q_i^T and
//               dP^T = V dO_i^T; dV += P^T dO_i and dK += dS^T Q_i read their A operand from TMEM too;
//               dQ_i = dS K reads dS from shared memory as an MN-major operand
//   warp 14     loads -lse_i * log2(e) and -delta_i with plain loads (their row offsets are not 16-byte
//               aligned) into an 8-deep ring
//   warp 15     works out the block's items and hands them to the other warps through an 8-slot ring
// TMEM columns: S^T [0,128) (half h at h*64; P^T of half h over its first 32 columns), dP^T [128,256)
// (dS^T likewise), dK [256,320), dV [320,384), dQ_i [384,448), K [448,480), V [480,512).
// dK and dV stay in TMEM for a whole item and are written once at its end.
// Registers: the block starts with 128 per thread; the compute warpgroups raise theirs and the other
// two warpgroups lower theirs (setmaxnreg) within the same total.
// The SMs of a cluster share the instruction cache behind the small per-partition one, and this kernel's
// speed depends on how much code it streams through it: changes that only add instructions (more unrolled
// variants, code that never runs) have cost up to a tenth of the time, so variants are kept few.  (96 to 97 % of the
// requests hit now, 67 to 92 % while each wait carried a timer and a report of its own.)
// What bounds it at L = 2240 is the 128-byte port of shared memory: per 128 x 128 step (2 780 clocks on average, item ends included;
// 2 450 in the steady loop) the tensor core takes 877 of its cycles, the LSU 961 (loads 326, stores 593, barriers 42),
// the copies of Q and dO 256 and the copy engine's reading of staged dQ 256: 2 350, averages of a whole launch like the 2 780.
// Hand-overs rearranged, more warps or more issuers leave that as it is, and none of them made the kernel faster.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>

#include "hmar_common.h"
#include "launchers.h"
#include "ptx_sm100.cuh"
#include "tc_common.h"

namespace hmar {
namespace {

using namespace ptx;

constexpr int BKV = 128;             // key rows per item
constexpr int BQ = 128;              // query rows per step
constexpr int HQ = 64;               // query rows per half step
constexpr int D = kHeadDim;
constexpr int NSTAGE = 3;
constexpr int AUX_STAGES = 8;        // ring of lse / delta rows, loaded this many steps ahead
constexpr int TILE_BYTES = 128 * D * 2;          // 16 KB
constexpr int ITEM_STAGES = 8;       // ring of items handed out by the scheduler warp
constexpr int ITEM_READERS = 15;     // warps that read every item: all but the scheduler
constexpr int NUM_COMPUTE_THREADS = 256;
constexpr int DRAIN_WARP0 = 8, PRODUCER_WARP = 12, MMA_WARP = 13, AUX_WARP = 14, SCHED_WARP = 15;
constexpr int NUM_THREADS = 512;
constexpr int REGS_COMPUTE = 152, REGS_DRAIN = 104, REGS_MISC = 104;
static_assert(2 * REGS_COMPUTE + REGS_DRAIN + REGS_MISC == 4 * 128, "register budget of the block");
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t COL_ST = 0, COL_DPT = 128, COL_DK = 256, COL_DV = 320, COL_DQ = 384, COL_K = 448, COL_V = 480;

// A work item as the roles see it: key rows [row_begin, row_begin + row_count) of head bh (head `head` of batch `batch`)
// and `steps` steps over the query rows [q_begin, q_end).  steps == 0: there are no more items.
struct Item {
    int bh, head, batch;
    int row_begin, row_count;
    int q_begin, q_end;
    int steps_uniform;                      // steps * 2 + uniform
    __device__ __forceinline__ int steps() const { return steps_uniform >> 1; }
    __device__ __forceinline__ bool uniform() const { return steps_uniform & 1; }
    // number of query columns of half h of step i handed to the tensor core (a multiple of 16)
    __device__ __forceinline__ int half_cols(int i, int h) const {
        const int n_eff = (min(BQ, q_end - (q_begin + i * BQ)) + 15) & ~15;
        return h == 0 ? min(n_eff, HQ) : max(n_eff - HQ, 0);
    }
};

struct __align__(1024) SharedStorage {
    uint8_t k[2][TILE_BYTES];               // K of the current item and of the next one (B operand of dQ)
    uint8_t q[NSTAGE][TILE_BYTES];
    uint8_t dout[NSTAGE][TILE_BYTES];
    uint8_t ds[2][2][TILE_BYTES];           // dS^T, double buffered: [step parity][64-query half][key row][64 queries], 128B swizzle
    uint8_t dq_stage[TILE_BYTES];           // per drain warp: 32 query rows x 32 fp32 columns of dQ_i on their way to the accumulator, 128B swizzle
    float lse2[AUX_STAGES][BQ];             // -lse * log2(e); -inf for query rows outside the range
    float delta[AUX_STAGES][BQ];            // -delta
    uint64_t k_full[2], k_free[2];          // [item parity]: K tile in shared memory / no longer read
    uint64_t kv_tmem, kv_free;              // K, V rows in TMEM / no longer read
    uint64_t qdo_full[NSTAGE], q_empty[NSTAGE], aux_full[AUX_STAGES], aux_empty[AUX_STAGES];
    uint64_t s_full[2], p_full[2];            // [half of the step]
    uint64_t dq_full, dq_empty, acc_full, acc_empty;
    Item item[ITEM_STAGES];
    uint64_t item_full[ITEM_STAGES], item_empty[ITEM_STAGES];
    uint32_t tmem_base;
    uint32_t gave_up;                       // offset of the barrier whose wait ran out (0: none did)
};
#define AT(field) (base + (uint32_t)offsetof(SharedStorage, field))     // shared-memory address

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Adds a [32 rows x 32 fp32] tile in shared memory (128-byte swizzle) to global memory at (column c0, row c1).
__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap* m, const void* smem_src, int c0, int c1) {
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(smem_src)), "r"(c0), "r"(c1)
                 : "memory");
}
// Writes [32 rows x 64 bf16] from shared memory (128-byte swizzle) to rows c1.. of head c2 of batch c3.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap* m, const void* smem_src, int c1, int c2, int c3) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(m)), "r"(smem_u32(smem_src)), "r"(0), "r"(c1), "r"(c2), "r"(c3)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

template <int N> __device__ __forceinline__ void reg_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N> __device__ __forceinline__ void reg_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// One row of a 128-byte-swizzled [128 rows x 64 bf16] tile, as 32 packed words in row order.
__device__ __forceinline__ void load_swizzled_row(const uint8_t* tile, int r, uint32_t (&dst)[32]) {
    const uint8_t* row = tile + r * 128;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const uint4 val = *reinterpret_cast<const uint4*>(row + ((c ^ (r & 7)) << 4));
        dst[4 * c] = val.x; dst[4 * c + 1] = val.y; dst[4 * c + 2] = val.z; dst[4 * c + 3] = val.w;
    }
}

// The 64 query columns of one half step for the 32 key rows of one warp:
// P^T = 2^(S^T * scale * log2e - lse * log2e) and dS^T = P^T o (dP^T - delta) in fp32.
// S^T and dP^T are read 16 key rows at a time in the layout in which a thread holds, of two rows, the
// column pairs 8k + 2(t % 4) + {0, 1}: a thread then needs lse and delta of 16 columns only (eight 8-byte
// loads each, two shared-memory wavefronts per load, counted: 256 of a step's 326; one key row per thread would need all 64 columns as
// broadcast loads, which were the largest share of the shared-memory traffic of the LSU).  A column pair
// packs into one bf16x2: P^T goes back to TMEM over S^T and dS^T over dP^T with the matching store layout
// (the 32 packed columns start at the half's first column, which this warp has already read for these
// rows), and dS^T also goes to shared memory, 4 bytes per pair (a warp's store covers 16 bytes of 8 rows,
// 128-byte swizzle on the key row: no bank conflicts).
// MODE 2: row i of this thread's four rows sees only columns [c_lo[i], c_hi[i]) of the step.
// MODE 1: every row either sees all columns or is past the end of the key tile (c_hi[i] <= 0).  Such a row
// holds another tile's keys; its P^T and dS^T only reach rows of dV and dK that are never written, but in
// dQ = dS K it would be summed over, so the copy of dS in shared memory gets zeros there.
// MODE 0: all rows see all columns.
// ROLLED: the two halves of the rows are iterations of a loop and not two copies of the code.  Less code, but the compiler
// no longer mixes one half's stores with the next half's loads: the instantiation for partial and packed tiles is bound
// by the code at its many item boundaries and gains (L = 680: 332 -> 295 us), the one for full tiles loses (L = 2240: 832 -> 849 us).
template <int MODE, bool ROLLED>
__device__ __forceinline__ void softmax_grad_half(uint32_t lane_base, int cbase, const uint64_t (&nls)[8], const uint64_t (&nde)[8],
                                                  float sl2, const int (&c_lo)[4], const int (&c_hi)[4], uint8_t* ds_tile,
                                                  int quarter, int lane) {
    const int tq = lane & 3, tr = lane >> 2;
    // nls, nde: -lse * log2(e) and -delta of this thread's column pairs; the arithmetic works on pairs of columns
    // with packed fp32 instructions (half as many instructions to issue and to fetch)
    const uint64_t sl2_2 = f32x2(sl2, sl2);
#pragma unroll (ROLLED ? 1 : 2)
    for (int hl = 0; hl < 2; ++hl) {                    // lanes 0-15, then 16-31 of the warp's quarter
        const int lo2[2] = {hl ? c_lo[2] : c_lo[0], hl ? c_lo[3] : c_lo[1]}, hi2[2] = {hl ? c_hi[2] : c_hi[0], hl ? c_hi[3] : c_hi[1]};
        // MODE 2: a bit per column of the half, moved so that this thread's pairs are the lowest two of each byte (bounds compared
        // column by column: L = 680 960 heads, main kernel 253 -> 245 us, L = 384 128 heads 31.3 -> 29.2)
        uint32_t seen[2][2];
        if (MODE == 2) {
#pragma unroll
            for (int rs = 0; rs < 2; ++rs) {
                visible_columns(lo2[rs] - cbase, hi2[rs] - cbase, seen[rs][0], seen[rs][1]);
                seen[rs][0] >>= 2 * tq;
                seen[rs][1] >>= 2 * tq;
            }
        }
        const uint32_t taddr = lane_base + ((uint32_t)(hl * 16) << 16);
        uint32_t s_buf[32], dp_buf[32];
        tmem_ld_16x256b_x8(taddr + COL_ST + cbase, s_buf);
        tmem_ld_16x256b_x8(taddr + COL_DPT + cbase, dp_buf);
        tmem_ld_wait();
        uint32_t p_pack[16], ds_pack[16];
        // key rows of this thread: quarter * 32 + hl * 16 + tr (+ 8); both have (row & 7) == tr
        uint8_t* ds_row = ds_tile + (quarter * 4 + hl * 2) * 1024 + tr * 128 + tq * 4;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
#pragma unroll
            for (int rs = 0; rs < 2; ++rs) {
                float x0, x1;
                f32x2_split(ffma2(f32x2(__uint_as_float(s_buf[4 * k + 2 * rs]), __uint_as_float(s_buf[4 * k + 2 * rs + 1])),
                                  sl2_2, nls[k]), x0, x1);
                float p0 = ex2(x0), p1 = ex2(x1);
                if (MODE == 2) {
                    if (!(seen[rs][k >> 2] >> (8 * (k & 3)) & 1u)) p0 = 0.f;
                    if (!(seen[rs][k >> 2] >> (8 * (k & 3)) & 2u)) p1 = 0.f;
                }
                float d0, d1;
                f32x2_split(fmul2(f32x2(p0, p1),
                                  fadd2(f32x2(__uint_as_float(dp_buf[4 * k + 2 * rs]), __uint_as_float(dp_buf[4 * k + 2 * rs + 1])),
                                        nde[k])), d0, d1);
                p_pack[2 * k + rs] = pack_bf16(p0, p1);
                ds_pack[2 * k + rs] = pack_bf16(d0, d1);
                // 8-row groups are 1024 bytes apart; 16-byte piece k of a row sits at position k ^ (row & 7)
                *reinterpret_cast<uint32_t*>(ds_row + rs * 1024 + ((k ^ tr) << 4)) =
                    (MODE == 1 && hi2[rs] <= 0) ? 0u : ds_pack[2 * k + rs];
            }
        }
        tmem_st_16x128b_x8(taddr + COL_ST + cbase, p_pack);
        tmem_st_16x128b_x8(taddr + COL_DPT + cbase, ds_pack);
    }
}

// STRIDED: the bf16 tensors have the strides given in the arguments (packed projection layouts); otherwise they are
// dense [BH, L, 64] and every address is formed with compile-time strides.  Dense tensors through the strided one, whole
// backward: L = 680 960 heads 381.6 -> 397.8 us, 128 heads 59.9 -> 60.6, 16 heads 16.6 -> 17.0, L = 2240 384 heads 829 -> 838; equal from
// L = 1600 with 39 heads to L = 9451 with 48.  (9 % in an earlier form of the kernel.)
// ONE_MASK: every tile goes through the variant of the softmax-gradient code with per-element bounds, so that the
// block's code holds one variant instead of three.  It is the instantiation for side lists whose tiles are mostly
// partial or packed (L = 680, 960 heads: whole backward 0.84 of the three variants' time); where most steps belong to full tiles
// the plain variant's shorter arithmetic wins (share 700, class by class: 4 to 10 %).  See bwd_one_mask.
template <bool STRIDED, bool ONE_MASK>
__global__ void __launch_bounds__(NUM_THREADS, 1)
hmar_bwd_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do,
                   const __grid_constant__ CUtensorMap map_dq, const __grid_constant__ CUtensorMap map_dk,
                   const __grid_constant__ CUtensorMap map_dv, const BwdArgs args) {
    // aligned by its declaration, so that every shared-memory address is a constant of the code (one added at run time
    // costs a register in every role and about 5 % of the code); checked below
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    SharedStorage& sm = *reinterpret_cast<SharedStorage*>(smem_raw);
    const uint32_t base = smem_u32(&sm);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if ((base & 1023u) != 0) {
        if (threadIdx.x == 0) report_gave_up(args.status, 0x3FF);
        return;
    }

    const int L = args.L;

    if (threadIdx.x == 0) {
        sm.gave_up = 0;
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sm.k_full[b], 1);
            mbar_init(&sm.k_free[b], 1);
        }
        mbar_init(&sm.kv_tmem, 128);
        mbar_init(&sm.kv_free, 1);
        for (int s = 0; s < NSTAGE; ++s) {
            mbar_init(&sm.qdo_full[s], 1);
            mbar_init(&sm.q_empty[s], 1);
        }
        for (int s = 0; s < AUX_STAGES; ++s) {
            mbar_init(&sm.aux_full[s], 32);
            mbar_init(&sm.aux_empty[s], NUM_COMPUTE_THREADS);
        }
        for (int h = 0; h < 2; ++h) {
            mbar_init(&sm.s_full[h], 1);
            mbar_init(&sm.p_full[h], NUM_COMPUTE_THREADS / 2);
        }
        mbar_init(&sm.dq_full, 1);
        mbar_init(&sm.dq_empty, 128);
        mbar_init(&sm.acc_full, 1);
        mbar_init(&sm.acc_empty, 128);
        for (int s = 0; s < ITEM_STAGES; ++s) {
            mbar_init(&sm.item_full[s], 1);
            mbar_init(&sm.item_empty[s], ITEM_READERS);
        }
        fence_mbar_init();
    }
    grid_wait();
    // From here on memory is read with plain loads: delta was written by the kernel before, lse, V and (where the call
    // allocates nothing) the work list by earlier ones, so none of it is read-only for the lifetime of this launch, which
    // a non-coherent load would ask for.
    // Whether an earlier block gave up: one answer for all threads, since the word may change between two of them and the
    // block's barriers and its tensor-memory allocation want whole warps.
    const int given_up = args.status != nullptr ? *reinterpret_cast<volatile int*>(args.status) : 0;
    if (__syncthreads_or(given_up)) return;
    if (warp == MMA_WARP) {
        tmem_alloc(&sm.tmem_base, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return warp_wait_or_give_up(bar, parity, &sm.gave_up, bar - base); };

    // The block's items go through a ring.  `look(n)` waits until item n is there; its fields are then read in place, and
    // `done(n)` gives the slot back (once per warp; items are looked at and done in order).
    auto look = [&](int n) -> bool { return wait(AT(item_full) + (n % ITEM_STAGES) * 8, (n / ITEM_STAGES) & 1); };
    auto done = [&](int n) {
        __syncwarp();
        if (lane == 0) bar_arrive(AT(item_empty) + (n % ITEM_STAGES) * 8);
    };
    auto item_at = [&](int n) -> const Item& { return sm.item[n % ITEM_STAGES]; };

    if (warp >= PRODUCER_WARP) {
        reg_dec<REGS_MISC>();
        if (warp == SCHED_WARP) {
            // ================================================================== item scheduler
            // The last records say that there are no more (the readers look up to two items ahead).
            int extra = 0;
            for (int n = 0; extra < 3; ++n) {
                const int slot = n % ITEM_STAGES;
                if (n >= ITEM_STAGES && !wait(AT(item_empty) + slot * 8, ((n / ITEM_STAGES) & 1) ^ 1)) break;
                Item it;
                it.steps_uniform = 0;
                const int tile = bwd_deal(args.work, args.n_work, args.n_heads, args.by_head, (int)gridDim.x, (int)blockIdx.x, n, it.bh);
                if (tile >= 0) {
                    const BwdWork w = args.work[tile];
                    it.batch = STRIDED ? it.bh / args.heads_per_batch : 0;
                    it.head = it.bh - it.batch * args.heads_per_batch * (STRIDED ? 1 : 0);
                    it.row_begin = w.row_begin;
                    it.row_count = w.row_count;
                    it.q_begin = w.q_begin;
                    it.q_end = w.q_end;
                    it.steps_uniform = ((w.q_end - w.q_begin + BQ - 1) / BQ) * 2 + (w.uniform != 0);
                } else {
                    ++extra;
                }
                if (lane == 0) {
                    sm.item[slot] = it;
                    bar_arrive(AT(item_full) + slot * 8);
                }
                __syncwarp();
            }
        } else if (warp == PRODUCER_WARP) {
            // ================================================================== producer
            // The whole warp runs the control flow; one elected lane issues the copies.
            const bool leader = elect_one();
            if (leader) {
                prefetch_tensormap(&map_q);
                prefetch_tensormap(&map_k);
                prefetch_tensormap(&map_v);
                prefetch_tensormap(&map_do);
            }
            bool ok = true;
            int gs = 0;                                     // steps issued so far, over all items
            for (int item = 0; ok; ++item) {
                ok = look(item);
                if (!ok) break;
                const Item w = item_at(item);
                done(item);
                const int n_steps = w.steps(), head = w.head, batch = w.batch;
                if (n_steps == 0) break;
                if (item >= 2) {
                    // the buffer held K of the item before the previous one, read by its dQ products
                    ok = wait(AT(k_free) + (item & 1) * 8, ((item >> 1) & 1) ^ 1);
                    if (!ok) break;
                }
                if (leader) {
                    bar_expect_tx(AT(k_full) + (item & 1) * 8, TILE_BYTES);
                    tma_load_4d_at(AT(k) + (item & 1) * TILE_BYTES, &map_k, AT(k_full) + (item & 1) * 8, 0, w.row_begin, head, batch);
                    // the V rows are read by the drain warps a few steps from now: bring them into L2
                    tma_prefetch_4d(&map_v, 0, w.row_begin, head, batch);
                }
                __syncwarp();
                for (int i = 0; i < n_steps; ++i, ++gs) {
                    const int slot = gs % NSTAGE;
                    const int q0 = w.q_begin + i * BQ;
                    if (gs >= NSTAGE) {
                        ok = wait(AT(q_empty) + (slot) * 8, ((gs / NSTAGE) & 1) ^ 1);
                        if (!ok) break;
                    }
                    if (leader) {
                        bar_expect_tx(AT(qdo_full) + (slot) * 8, 2 * TILE_BYTES);
                        tma_load_4d_at(AT(q) + slot * TILE_BYTES, &map_q, AT(qdo_full) + (slot) * 8, 0, q0, head, batch);
                        tma_load_4d_at(AT(dout) + slot * TILE_BYTES, &map_do, AT(qdo_full) + (slot) * 8, 0, q0, head, batch);
                    }
                    __syncwarp();
                }
            }
            if (!ok) {
                // give the copies already issued a bounded chance to land before the block exits
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 2000000ull) { }
            }
        } else if (warp == AUX_WARP) {
            // ================================================================== lse / delta loader
            // lse and delta rows of a step go to ring slot (step count) % AUX_STAGES, several steps ahead of
            // their use (plain loads: their row offsets are not 16-byte aligned, so TMA cannot fetch them).
            bool ok = true;
            int gs = 0;
            for (int item = 0; ok; ++item) {
                ok = look(item);
                if (!ok) break;
                const Item w = item_at(item);
                done(item);
                const int n_steps = w.steps(), bh = w.bh;
                if (n_steps == 0) break;
                for (int i = 0; i < n_steps; ++i, ++gs) {
                    const int aslot = gs % AUX_STAGES;
                    if (gs >= AUX_STAGES) {
                        ok = wait(AT(aux_empty) + (aslot) * 8, ((gs / AUX_STAGES) & 1) ^ 1);
                        if (!ok) break;
                    }
                    const int q0 = w.q_begin + i * BQ;
                    // all loads first, then the stores: stores to shared memory in between would serialise them
                    float lv[BQ / 32], dv[BQ / 32];
#pragma unroll
                    for (int t = 0; t < BQ / 32; ++t) {
                        const int row = q0 + t * 32 + lane;
                        const bool in = row < w.q_end &&
                                        HMAR_IN_BOUNDS(row >= 0 && row < L && bh >= 0 && bh < args.n_heads, args.status, 0xB201);
                        lv[t] = in ? args.lse[(size_t)bh * L + row] : INFINITY;
                        dv[t] = in ? args.delta[(size_t)bh * L + row] : 0.f;
                    }
#pragma unroll
                    for (int t = 0; t < BQ / 32; ++t) {
                        sm.lse2[aslot][t * 32 + lane] = lv[t] * -1.4426950408889634f;
                        sm.delta[aslot][t * 32 + lane] = -dv[t];
                    }
                    bar_arrive(AT(aux_full) + (aslot) * 8);
                }
            }
        } else if (warp == MMA_WARP) {
            // ================================================================== MMA issuer
            // The whole warp runs the control flow and one elected lane issues (a warp that has split into
            // one running lane and 31 parked ones issues far more slowly).  Descriptors are built once and
            // advanced by adding (byte offset >> 4) to them.
            // The tensor core's queue holds only a few products, and a product issued to an idle tensor core
            // costs about a hundred clocks before it starts, so a step is issued as two uninterrupted bursts:
            //   X_i = dV,dK of half 0 of step i, then S^T,dP^T of half 0 of step i+1
            //   Y_i = dV,dK of half 1 of step i, then S^T,dP^T of half 1 of step i+1, then dQ_i
            // each preceded by one look at the barriers it depends on (two at a time, both usually complete).
            const bool leader = elect_one();
            const uint64_t k_mn0 = smem_desc_sw128(AT(k), 1024);    // K as MN-major B of dQ
            // the ring slots and the dS buffers are 16 KB apart: descriptor of slot s = base + s * 1024
            const uint64_t q_kd0 = smem_desc_sw128(AT(q), 16), do_kd0 = smem_desc_sw128(AT(dout), 16);
            const uint64_t q_mn0 = smem_desc_sw128(AT(q), 1024), do_mn0 = smem_desc_sw128(AT(dout), 1024);
            const uint64_t ds_mn0 = smem_desc_sw128(AT(ds), TILE_BYTES);
            constexpr uint32_t idesc_acc = idesc_bf16_f32(BKV, D, false, true);    // A from TMEM, B MN-major
            constexpr uint32_t idesc_dq = idesc_bf16_f32(BQ, D, true, true);
            bool ok = true;
            int gs = 0;                                         // steps issued so far (ring slot, dQ parity)
            int ng[2] = {0, 0};                                 // gradient halves issued so far, per half
            // waits for barrier a and, if have_b, barrier b; the two first looks overlap
            auto wait2 = [&](uint32_t a, uint32_t pa, uint32_t b, uint32_t pb, bool have_b) -> bool {
                bool ra, rb;
                warp_try_wait2(a, pa, have_b ? b : a, have_b ? pb : pa, ra, rb);
                // a barrier seen complete is not looked at again: a look is a shared-memory round trip behind the
                // compute warps' stores, on the critical path of the step
                return (ra || wait(a, pa)) && (!have_b || rb || wait(b, pb));
            };
            // S^T_h = K Q_h^T,  dP^T_h = V dO_h^T : n query columns of half h, Q / dO tile in ring slot `slot`
            auto scores = [&](int h, int n, int slot) {
                const uint32_t idesc = idesc_bf16_f32(BKV, n, false, false);
                const uint64_t qd = q_kd0 + slot * 1024 + h * 512, dd = do_kd0 + slot * 1024 + h * 512;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    mma_ts(tmem + COL_ST + h * HQ, tmem + COL_K + ks * 8, qd + ks * 2, idesc, ks > 0);
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    mma_ts(tmem + COL_DPT + h * HQ, tmem + COL_V + ks * 8, dd + ks * 2, idesc, ks > 0);
                commit_at(AT(s_full) + (h) * 8);
            };
            // dV += P_h^T dO_h,  dK += dS_h^T Q_h : n query columns of half h
            auto grads = [&](int h, int n, int slot, bool first) {
                const int nk = n / 16;
                const uint64_t dod = do_mn0 + slot * 1024 + h * 512, qd = q_mn0 + slot * 1024 + h * 512;
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    if (ks < nk)
                        mma_ts(tmem + COL_DV, tmem + COL_ST + h * HQ + ks * 8, dod + ks * 128, idesc_acc, !first || (ks > 0));
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    if (ks < nk)
                        mma_ts(tmem + COL_DK, tmem + COL_DPT + h * HQ + ks * 8, qd + ks * 128, idesc_acc, !first || (ks > 0));
            };

            // The steps of all items form one sequence: while the compute warpgroups work on a step, the
            // tensor core gets the next step's S^T, dP^T even when that step belongs to the next item (whose
            // K, V rows the drain warps have put into TMEM by then).
            ok = look(0) && look(1);
            bool live = ok && item_at(0).steps() > 0;
            if (live) {
                const Item& w0 = item_at(0);
                ok = wait2(AT(kv_tmem), 0, AT(qdo_full), 0, true);
                if (ok) {
                    tc_fence_after();
                    if (leader) {
                        scores(0, w0.half_cols(0, 0), 0);
                        const int n1 = w0.half_cols(0, 1);
                        if (n1 > 0) scores(1, n1, 0);
                        if (w0.steps() == 1 && item_at(1).steps() > 0) commit_at(AT(kv_free));
                    }
                    __syncwarp();
                }
            }
            for (int item = 0; live && ok; ++item) {
                ok = look(item + 2);
                if (!ok) break;
                const Item w = item_at(item);
                const Item wn = item_at(item + 1);
                const int n_steps = w.steps(), n_steps_next = wn.steps();
                const bool next_item = n_steps_next > 0, item_after = item_at(item + 2).steps() > 0;
                const uint64_t k_mn = k_mn0 + (item & 1) * 1024;
                for (int i = 0; i < n_steps && ok; ++i, ++gs) {
                    const int slot = gs % NSTAGE, slot_next = (gs + 1) % NSTAGE;
                    const bool more = i + 1 < n_steps;          // the item has another step
                    const bool cross = !more && next_item;      // the next step is the next item's first
                    const bool any_next = more || cross;
                    const int n0 = w.half_cols(i, 0), n1 = w.half_cols(i, 1);
                    const int m0 = more ? w.half_cols(i + 1, 0) : cross ? wn.half_cols(0, 0) : 0;
                    const int m1 = more ? w.half_cols(i + 1, 1) : cross ? wn.half_cols(0, 1) : 0;
                    // the next step is the last one that reads its item's K, V rows in TMEM, and another item follows
                    const bool frees_kv = more ? (i + 2 == n_steps && next_item) : (cross && n_steps_next == 1 && item_after);
                    // ---- burst X: needs P^T, dS^T of half 0 and the next step's Q / dO tile
                    ok = wait2(AT(p_full) + (0) * 8, ng[0] & 1, AT(qdo_full) + (slot_next) * 8, ((gs + 1) / NSTAGE) & 1, any_next);
                    if (!ok) break;
                    ++ng[0];
                    if (cross) {                                // K, V of the next item in TMEM
                        ok = wait(AT(kv_tmem), (item + 1) & 1);
                        if (!ok) break;
                    }
                    if (i == 0 && item > 0) {                   // dK, dV of the previous item read out
                        ok = wait(AT(acc_empty), (item - 1) & 1);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    if (leader) {
                        grads(0, n0, slot, i == 0);
                        if (m0 > 0) scores(0, m0, slot_next);
                    }
                    __syncwarp();
                    // ---- burst Y: needs P^T, dS^T of half 1 (if the step has one) and dQ of the previous
                    // step drained from TMEM
                    if (n1 > 0) {
                        ok = wait2(AT(p_full) + (1) * 8, ng[1] & 1, AT(dq_empty), (gs - 1) & 1, gs > 0);
                        ++ng[1];
                    } else if (gs > 0) {
                        ok = wait(AT(dq_empty), (gs - 1) & 1);
                    }
                    if (!ok) break;
                    if (i == 0) {                               // K of this item in shared memory (B operand of dQ)
                        ok = wait(AT(k_full) + (item & 1) * 8, (item >> 1) & 1);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    if (leader) {
                        if (n1 > 0) grads(1, n1, slot, false);
                        commit_at(AT(q_empty) + (slot) * 8);           // Q_i, dO_i are not read again
                        if (!more) commit_at(AT(acc_full));     // dK, dV of the item are complete
                        // the next scores of half 1 go first: the compute warpgroup is waiting for them, dQ_i
                        // is not needed before the drain warps get to it
                        if (m1 > 0) scores(1, m1, slot_next);
                        if (frees_kv) commit_at(AT(kv_free));
                        // dQ_i = dS K over both halves: A = dS (queries x keys) read as an MN-major operand.  When
                        // the step has no second half its rows are stale data and are never drained.
                        const uint64_t dsd = ds_mn0 + (gs & 1) * 2048;
#pragma unroll
                        for (int ks = 0; ks < BKV / 16; ++ks)
                            mma_ss(tmem + COL_DQ, dsd + ks * 128, k_mn + ks * 128, idesc_dq, ks > 0);
                        commit_at(AT(dq_full));
                        if (!more) commit_at(AT(k_free) + (item & 1) * 8);
                    }
                    __syncwarp();
                }
                done(item);
                live = next_item;
            }
        }
    } else if (warp >= DRAIN_WARP0) {
        // ================================================================== dQ drain
        // One query row per thread, and every warp on its own: dQ_i leaves TMEM 32 columns at a time, is
        // staged in the warp's 4 KB of shared memory and added to the fp32 accumulator by one bulk tensor
        // reduction per 32 x 32 piece (whole cache lines, issued by the copy engine; per-thread reductions
        // would be 16-byte pieces of 32 different lines).  Rows past the end of the query range are staged
        // as zeros.
        reg_dec<REGS_DRAIN>();
        const int quarter = warp & 3;
        const int r = quarter * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        const int sub_row = lane >> 3, piece = lane & 7;      // whole rows: lane's row among four and its 16-byte piece
        uint8_t* stage = sm.dq_stage + quarter * 4096;
        uint8_t* stage_row = stage + (lane >> 3) * 1024 + (lane & 7) * 128;
        if (lane == 0) prefetch_tensormap(&map_dq);
        uint32_t buf[32];
        bool ok = true;
        int gs = 0;
        // K and V rows of item gc (the block's item number `item`) to TMEM, one key row per thread: the A
        // operands of S^T = K Q^T and dP^T = V dO^T.  The V rows come straight from global memory, four whole rows per
        // load instruction and through the staging buffer into the thread that owns the row, and wait in registers until
        // the previous item's last scores have been computed; the K row is read from the tile that the copy engine has put
        // into shared memory for the dQ products.  Rows past the end of the sequence are zeros.
        auto copy_kv = [&](int item, bool wait_free) -> bool {
            const Item& wc = item_at(item);
            const int row0 = wc.row_begin + quarter * 32 + sub_row;
            const __nv_bfloat16* vsrc = STRIDED ? args.v + wc.batch * args.in_batch + wc.head * args.in_head + row0 * args.in_row
                                                : args.v + ((size_t)wc.bh * L + row0) * D;
            const long long step = STRIDED ? 4 * args.in_row : 4 * D;
            uint4 rows[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const __nv_bfloat16* src = vsrc + c * step + piece * 8;
                const bool v_in = row0 + 4 * c < L && HMAR_IN_BOUNDS(src >= args.v && src - args.v + 8 <= args.in_extent, args.status, 0xB202);
                rows[c] = v_in ? *reinterpret_cast<const uint4*>(src) : make_uint4(0u, 0u, 0u, 0u);
            }
            if (lane == 0) bulk_wait_read_all();                // the last piece of dQ has been read out of the staging buffer
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 8; ++c)
                *reinterpret_cast<uint4*>(stage + (4 * c + sub_row) * 128 + ((piece ^ ((4 * c + sub_row) & 7)) << 4)) = rows[c];
            __syncwarp();
            load_swizzled_row(stage, lane, buf);
            __syncwarp();
            if (wait_free) {
                if (!wait(AT(kv_free), (item - 1) & 1)) return false;
                tc_fence_after();
            }
            tmem_st32(lane_base + COL_V, buf);
            if (!wait(AT(k_full) + (item & 1) * 8, (item >> 1) & 1)) return false;
            load_swizzled_row(sm.k[item & 1], r, buf);
            tmem_st32(lane_base + COL_K, buf);
            tmem_st_wait();
            tc_fence_before();
            bar_arrive(AT(kv_tmem));
            return true;
        };
        ok = look(0) && look(1);
        if (ok && item_at(0).steps() > 0) {
            ok = copy_kv(0, false);
            if (ok && item_at(0).steps() == 1 && item_at(1).steps() > 0) ok = copy_kv(1, true);
        }
        for (int item = 0; ok; ++item) {
            const Item w = item_at(item);
            const int n_steps = w.steps();
            if (n_steps == 0) break;
            ok = look(item + 2);
            if (!ok) break;
            const int bh = w.bh;
            const int n_steps_next = item_at(item + 1).steps();
            const bool next_item = n_steps_next > 0, item_after = item_at(item + 2).steps() > 0;
            for (int i = 0; i < n_steps; ++i, ++gs) {
                const bool more = i + 1 < n_steps;
                // the next step is the last one of its item and another item follows: that item's K, V rows
                // go to TMEM as soon as the next step's scores are complete
                if (more ? (i + 2 == n_steps && next_item) : (next_item && n_steps_next == 1 && item_after)) {
                    const int nc = more ? item + 1 : item + 2;
                    ok = copy_kv(nc, true);
                    if (!ok) break;
                }
                if (!more) {
                    // ---- end of the item: dK and dV, one key row per thread, scaled and rounded to bf16
                    ok = wait(AT(acc_full), item & 1);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int part = 0; part < 4; ++part) {
                        tmem_ld32(lane_base + (part < 2 ? COL_DK : COL_DV) + (part & 1) * 32, buf);
                        tmem_ld_wait();
                        if (part == 3) {
                            tc_fence_before();
                            bar_arrive(AT(acc_empty));         // the next item's products may overwrite dK / dV
                        }
                        // rows go through the staging buffer, so that a store instruction covers four whole rows (a thread
                        // storing its own row touches 32 lines per instruction, which L1 takes one by one)
                        const float mul = part < 2 ? args.softmax_scale : 1.f;
                        if ((part & 1) == 0) {
                            if (lane == 0) bulk_wait_read_all();
                            __syncwarp();
                        }
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            uint4 o;
                            o.x = pack_bf16(__uint_as_float(buf[8 * t + 0]) * mul, __uint_as_float(buf[8 * t + 1]) * mul);
                            o.y = pack_bf16(__uint_as_float(buf[8 * t + 2]) * mul, __uint_as_float(buf[8 * t + 3]) * mul);
                            o.z = pack_bf16(__uint_as_float(buf[8 * t + 4]) * mul, __uint_as_float(buf[8 * t + 5]) * mul);
                            o.w = pack_bf16(__uint_as_float(buf[8 * t + 6]) * mul, __uint_as_float(buf[8 * t + 7]) * mul);
                            *reinterpret_cast<uint4*>(stage_row + ((((part & 1) * 4 + t) ^ (lane & 7)) << 4)) = o;
                        }
                        // A warp whose 32 rows are all the tile's sends them with one copy; other rows belong to another tile.
                        // (Always with stores: packed layout, 96 heads of L = 2240, 215 -> 210 us; L = 680 960 heads 333.5 -> 331.)
                        if ((part & 1) == 1 && quarter * 32 + 32 <= w.row_count) {
                            fence_proxy_async_smem();
                            __syncwarp();
                            if (lane == 0) {
                                tma_store_4d(part < 2 ? &map_dk : &map_dv, stage, w.row_begin + quarter * 32, w.head, w.batch);
                                bulk_commit_group();
                            }
                        } else if ((part & 1) == 1) {
                            __syncwarp();
                            __nv_bfloat16* base = part < 2 ? args.dk : args.dv;
                            const int row0 = quarter * 32 + sub_row;
                            __nv_bfloat16* dst = base + piece * 8 + (STRIDED ? w.batch * args.g_batch + w.head * args.g_head + (w.row_begin + row0) * args.g_row
                                                                            : (long long)((size_t)bh * L + w.row_begin + row0) * D);
                            const long long step = STRIDED ? 4 * args.g_row : 4 * D;
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const uint4 o = *reinterpret_cast<const uint4*>(stage + (4 * c + sub_row) * 128 + ((piece ^ ((4 * c + sub_row) & 7)) << 4));
                                __nv_bfloat16* at = dst + c * step;
                                if (row0 + 4 * c < w.row_count && HMAR_IN_BOUNDS(at >= base && at - base + 8 <= args.g_extent, args.status, 0xB203))
                                    *reinterpret_cast<uint4*>(at) = o;
                            }
                            __syncwarp();
                        }
                    }
                }
                ok = wait(AT(dq_full), gs & 1);
                if (!ok) break;
                tc_fence_after();
                const int q0 = w.q_begin + i * BQ;
                const bool row_in = r < min(BQ, w.q_end - q0);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    tmem_ld32(lane_base + COL_DQ + c * 32, buf);
                    tmem_ld_wait();
                    if (c == 1) {
                        tc_fence_before();
                        bar_arrive(AT(dq_empty));
                    }
                    // the previous piece must have been read out of the staging buffer
                    if (lane == 0) bulk_wait_read_all();
                    __syncwarp();
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        const uint4 val = row_in ? make_uint4(buf[4 * t], buf[4 * t + 1], buf[4 * t + 2], buf[4 * t + 3])
                                                 : make_uint4(0u, 0u, 0u, 0u);
                        *reinterpret_cast<uint4*>(stage_row + ((t ^ (lane & 7)) << 4)) = val;
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_reduce_add_2d(&map_dq, stage, c * 32, bh * L + q0 + quarter * 32);
                        bulk_commit_group();
                    }
                }
            }
            if (ok) done(item);
        }
        if (lane == 0) bulk_wait_all();         // the staging buffer must outlive the last copy's read
    } else {
        // ================================================================== compute warpgroups
        reg_inc<REGS_COMPUTE>();
        const int quarter = warp & 3;
        const int h = warp >> 2;                            // the half of every step this warpgroup owns
        const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
        const float sl2 = args.scale_log2;
        bool ok = true;
        int gs = 0;                                         // steps seen so far (aux ring, dS buffer parity)
        int nsh = 0;                                        // non-empty halves of this warpgroup seen so far

        for (int item = 0; ok; ++item) {
            ok = look(item);
            if (!ok) break;
            const Item w = item_at(item);
            done(item);
            const int n_steps = w.steps();
            if (n_steps == 0) break;
            // the four key rows this thread works on in the softmax-gradient layout, and the queries that may see them
            const bool tile_masked = ONE_MASK || (!w.uniform()) || (w.row_count < BKV);
            const bool rows_only = !ONE_MASK && w.uniform();        // only rows past the end of the tile are hidden
            int qlo[4], qhi[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int rr = quarter * 32 + (i >> 1) * 16 + (lane >> 2) + (i & 1) * 8;
                qlo[i] = w.q_begin; qhi[i] = w.q_end;
                if (tile_masked && rr >= w.row_count) { qlo[i] = 0; qhi[i] = 0; }
            }
            if (!w.uniform()) {
                // Scale by scale and not row by row: the table lies in constant memory, where lanes that read different
                // entries are served one after the other (a packed tile's search took 3 000 clocks at L = 680; 960 heads
                // 346.0 -> 341.3 us, 128 heads 60.7 -> 59.3).
                for (int s = 0; s < args.st.n_scales; ++s) {
                    const int begin = args.st.start[s] - w.row_begin, end = args.st.start[s + 1] - w.row_begin;
                    if (end <= 0) continue;
                    if (begin >= w.row_count) break;
                    const int first = args.st.start[first_query_scale(args.st.window, s)];
                    const int last = args.st.start[last_query_scale(args.st.window, s, args.st.n_scales) + 1];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int rr = quarter * 32 + (i >> 1) * 16 + (lane >> 2) + (i & 1) * 8;
                        if (rr >= begin && rr < end && rr < w.row_count) { qlo[i] = first; qhi[i] = last; }
                    }
                }
            }

            for (int i = 0; i < n_steps && ok; ++i, ++gs) {
                const int q0 = w.q_begin + i * BQ;
                const int n_valid = min(BQ, w.q_end - q0);
                const int n_cols = w.half_cols(i, h);
                const int cbase = h * HQ;                   // first query column of this half inside the step

                const int aslot = gs % AUX_STAGES;
                ok = wait(AT(aux_full) + (aslot) * 8, (gs / AUX_STAGES) & 1);
                if (!ok) break;

                // The step's lse and delta are fetched while the scores are still being computed: behind the wait for the
                // scores, this look and these loads were 450 of the 2 975 clocks from one step of a warpgroup to the next.
                uint64_t nls[8], nde[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    nls[k] = *reinterpret_cast<const uint64_t*>(sm.lse2[aslot] + cbase + 8 * k + 2 * (lane & 3));
                    nde[k] = *reinterpret_cast<const uint64_t*>(sm.delta[aslot] + cbase + 8 * k + 2 * (lane & 3));
                }
                if (n_cols > 0) {
                    ok = wait(AT(s_full) + (h) * 8, nsh & 1);
                    if (!ok) break;
                    ++nsh;
                    tc_fence_after();
                    // tiles whose rows all see every column skip the mask code
                    if (tile_masked) {
                        int c_lo[4], c_hi[4];               // visible query columns of the four rows in this step
#pragma unroll
                        for (int r4 = 0; r4 < 4; ++r4) {
                            c_lo[r4] = max(qlo[r4] - q0, 0);
                            c_hi[r4] = min(qhi[r4] - q0, n_valid);
                        }
                        if (rows_only)
                            softmax_grad_half<1, ONE_MASK>(lane_base, cbase, nls, nde, sl2, c_lo, c_hi,
                                                 sm.ds[gs & 1][h], quarter, lane);
                        else
                            softmax_grad_half<2, ONE_MASK>(lane_base, cbase, nls, nde, sl2, c_lo, c_hi,
                                                 sm.ds[gs & 1][h], quarter, lane);
                    } else {
                        const int none[4] = {0, 0, 0, 0};
                        softmax_grad_half<0, ONE_MASK>(lane_base, cbase, nls, nde, sl2, none, none,
                                                 sm.ds[gs & 1][h], quarter, lane);
                    }
                    tmem_st_wait();
                    tc_fence_before();
                    fence_proxy_async_smem();
                    bar_arrive(AT(p_full) + (h) * 8);
                }
                bar_arrive(AT(aux_empty) + (aslot) * 8);      // this thread is done with the step's lse / delta
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0) report_gave_up(args.status, sm.gave_up);
}

// ------------------------------------------------------------------------------------------------
// Offset (elements) of row `row` (= bh * L + l) of a strided bf16 tensor.
struct RowLayout {
    int L, heads_per_batch;
    long long row, head, batch;
    FastDiv by_L, by_heads;
    template <bool STRIDED>
    __device__ __forceinline__ long long offset(size_t r) const {
        if (!STRIDED) return (long long)r * D;
        // (a tensor of 2^31 rows of 128 bytes would be larger than the memory)
        const int bh = by_L((int)r), l = (int)r - bh * L;
        const int b = by_heads(bh), h = bh - b * heads_per_batch;
        return b * batch + h * head + l * row;
    }
};

// delta_i = sum_d dO_id * O_id  (one warp per 4 rows: 8 lanes x 16 bytes cover a row).  The same pass
// clears the fp32 dQ accumulator (32 bytes per lane), which saves a separate pass over it.
template <bool STRIDED>
__global__ void __launch_bounds__(256)
hmar_bwd_delta_kernel(const __nv_bfloat16* out, const __nv_bfloat16* dout, float* delta, float* dq_acc, size_t n_rows, const RowLayout lay) {
    const size_t row = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    const int part = threadIdx.x & 7;
    float acc = 0.f;
    grid_wait();
    if (row < n_rows) {
        float4* z = reinterpret_cast<float4*>(dq_acc + row * D + part * 8);
        z[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
        const long long off = lay.template offset<STRIDED>(row) + part * 8;
        const uint4 a = *reinterpret_cast<const uint4*>(out + off);
        const uint4 b = *reinterpret_cast<const uint4*>(dout + off);
        const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
        const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float2 fa = __bfloat1622float2(pa[t]), fb = __bfloat1622float2(pb[t]);
            acc = fmaf(fa.x, fb.x, acc);
            acc = fmaf(fa.y, fb.y, acc);
        }
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    if (row < n_rows && part == 0) delta[row] = acc;
}

// dq = bf16(scale * dq_acc)
template <bool STRIDED>
__global__ void __launch_bounds__(256)
hmar_bwd_dq_convert_kernel(const float* acc, __nv_bfloat16* dq, float scale, size_t n8, const RowLayout lay) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n8) return;
    grid_wait();
    const float4 a = reinterpret_cast<const float4*>(acc)[2 * idx];
    const float4 b = reinterpret_cast<const float4*>(acc)[2 * idx + 1];
    uint4 o;
    o.x = pack_bf16(a.x * scale, a.y * scale);
    o.y = pack_bf16(a.z * scale, a.w * scale);
    o.z = pack_bf16(b.x * scale, b.y * scale);
    o.w = pack_bf16(b.z * scale, b.w * scale);
    *reinterpret_cast<uint4*>(dq + lay.template offset<STRIDED>(idx >> 3) + (idx & 7) * 8) = o;
}

}  // namespace

// Number of SMs of the current device (one persistent block each), looked up once per device.
static int sm_count() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 1;
    if (cached[dev] == 0) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
        cached[dev] = n;
    }
    return cached[dev];
}

template <bool STRIDED>
static cudaError_t launch_bwd_tc_layout(const CUtensorMap& q, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& dout_map,
                                        const CUtensorMap& dq_acc_map, const CUtensorMap& dk_map, const CUtensorMap& dv_map, const BwdArgs& args,
                                        const __nv_bfloat16* out, const __nv_bfloat16* dout, __nv_bfloat16* dq, int BH, cudaStream_t stream) {
    const size_t smem = sizeof(SharedStorage);
    const size_t n_rows = (size_t)BH * args.L;
    {
        KernelTimer timer("hmar_bwd_delta_kernel", stream);
        const RowLayout lay{args.L, args.heads_per_batch, args.od_row, args.od_head, args.od_batch, FastDiv(args.L), FastDiv(args.heads_per_batch)};
        const cudaError_t e = launch_overlapped(hmar_bwd_delta_kernel<STRIDED>, (unsigned)((n_rows * 8 + 255) / 256), 256, 0, stream, out, dout,
                                                args.delta_w, args.dq_acc, n_rows, lay);
        if (e != cudaSuccess) return e;
    }
    {
        KernelTimer timer("hmar_bwd_tc_kernel", stream);
        const long long items = (long long)BH * args.n_work;
        const unsigned grid = (unsigned)(items < sm_count() ? items : sm_count());
        BwdArgs a = args;
        a.by_head = bwd_by_head(args.head_steps, args.n_work, n_rows);
        static SmemOptIn opt_in[2];
        const bool one_mask = bwd_one_mask(args.plain_permille, a.by_head);
        auto kernel = one_mask ? hmar_bwd_tc_kernel<STRIDED, true> : hmar_bwd_tc_kernel<STRIDED, false>;
        cudaError_t e = opt_in[one_mask]((const void*)kernel, smem);
        if (e == cudaSuccess) e = launch_overlapped(kernel, grid, NUM_THREADS, smem, stream, q, k, v, dout_map, dq_acc_map, dk_map, dv_map, a);
        if (e != cudaSuccess) return e;
    }
    const size_t n8 = n_rows * D / 8;
    {
        KernelTimer timer("hmar_bwd_dq_convert_kernel", stream);
        const RowLayout lay{args.L, args.heads_per_batch, args.g_row, args.g_head, args.g_batch, FastDiv(args.L), FastDiv(args.heads_per_batch)};
        const cudaError_t e = launch_overlapped(hmar_bwd_dq_convert_kernel<STRIDED>, (unsigned)((n8 + 255) / 256), 256, 0, stream, args.dq_acc, dq,
                                                args.softmax_scale, n8, lay);
        if (e != cudaSuccess) return e;
    }
    count_launch(3);
    return cudaGetLastError();
}

cudaError_t launch_bwd_tc(const CUtensorMap& q, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& dout_map,
                          const CUtensorMap& dq_acc_map, const CUtensorMap& dk_map, const CUtensorMap& dv_map, const BwdArgs& args,
                          const __nv_bfloat16* out, const __nv_bfloat16* dout, __nv_bfloat16* dq, int BH, cudaStream_t stream) {
    return bwd_dense(args) ? launch_bwd_tc_layout<false>(q, k, v, dout_map, dq_acc_map, dk_map, dv_map, args, out, dout, dq, BH, stream)
                           : launch_bwd_tc_layout<true>(q, k, v, dout_map, dq_acc_map, dk_map, dv_map, args, out, dout, dq, BH, stream);
}

}  // namespace hmar
