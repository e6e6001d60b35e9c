// Forward kernel of HMAR's Markovian block-sparse attention for sm_100a, and the inference step.
//
// One block handles one work tile: up to 128 consecutive query rows of one head and the contiguous
// key range those rows may see under the mask (paper Sec. 4.1, Fig. attn-mask).  It is the usual
// IO-aware tiling with an online softmax (Sec. 4.1: the kernel extends FlashAttention), laid out for
// Blackwell.  The key range is walked 64 keys at a time, and a block is ONE softmax chain:
//   logits ready -> softmax warpgroup -> P ready -> tensor core (O += P V, next logits) -> ...
// A chain spends most of its time waiting for the other side (the round trip through the barriers and the
// tensor core's queue is longer than either side's work), so what keeps an SM busy is the number of
// independent chains on it: a block is kept small (256 threads, 128 TMEM columns, 50 KB of shared memory)
// and FOUR blocks share an SM.  Each block's set-up, first copies and epilogue, during which it computes
// nothing, are then overlapped by three running chains instead of being a quarter of its life.
//   warps 0-3   softmax: one query row per thread, 64 logits per tile read from TMEM once; the running
//               maximum is kept unless the tile exceeds it by more than 2^8 (then O and the row sum are
//               rescaled first), P = 2^(s - m) goes back to TMEM as bf16 over S; at the end O / l -> out
//   warp 4      TMA producer: K and V tiles of 64 keys through a shared-memory ring (Q and the first K, V
//               tiles are requested by thread 0 during the set-up).  The tensor maps are 4-D (64, rows,
//               heads, batches) with the tensor's own strides, so contiguous [B,H,L,64] tensors and the
//               packed [B,L,3,H,64] projection output go through the same code; the output address is
//               formed from three strides
//   warp 5      issues tcgen05.mma: S = Q K^T (both operands in shared memory), O += P V (P from TMEM, V an
//               MN-major shared-memory operand), one burst per tile: O += P V of tile j, then S of tile
//               j + 1 into the columns P has just left
//   warps 6-7   idle: setmaxnreg works on whole warpgroups (four warps), so the producer and the MMA warp
//               sit in a full second warpgroup (a block of 192 threads cannot redistribute its registers;
//               without the redistribution the softmax warps spill and the kernel is 4 % slower)
// TMEM columns: S/P [0,64), O [64,128).
// Registers: the block starts with 64 per thread (four blocks per SM); the softmax warpgroup raises its
// to 96 and the second warpgroup drops to 32 (setmaxnreg), the same total.  24 bytes are spilled then, 44 with 88 and 40 (L = 680
// 960 heads 114.4 -> 115.6 us, inference step 13 -> 18 1536 heads 138.2 -> 140.2), 60 with 104 and 24 (1 % slower).
// A time in these comments is that of the kernel in a row of some tens of launches, caches as the launch before leaves them, both sides
// of a pair in turn on one GPU.  Pairs of different dates do not add up: a block of the step 13 -> 18 lives 26 500 clocks, and the
// launch takes 123 us on a GPU that was idle before (SMs at 1.8 GHz inside the kernel) and 139 to 143 at the power limit (1.61 to 1.65).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>

#include "hmar_common.h"
#include "launchers.h"
#include "ptx_sm100.cuh"
#include "tc_common.h"

namespace hmar {
namespace {

using namespace ptx;

constexpr int BM = 128;              // query rows per block
constexpr int BN = 64;               // keys per tile
constexpr int D = kHeadDim;
constexpr int NSTAGE = 2;
constexpr int Q_BYTES = BM * D * 2;             // 16 KB
constexpr int TILE_BYTES = BN * D * 2;          // 8 KB
constexpr int NUM_THREADS = 256;
constexpr int NUM_SOFTMAX_THREADS = 128;
constexpr int PRODUCER_WARP = 4, MMA_WARP = 5;
constexpr int REGS_START = 64, REGS_SOFTMAX = 96, REGS_MISC = 32;
static_assert(4 * REGS_SOFTMAX + 4 * REGS_MISC == 8 * REGS_START, "register budget of the block");
constexpr uint32_t TMEM_COLS = 128;
constexpr uint32_t COL_S = 0, COL_O = 64;
constexpr float kRescaleThreshold = 8.0f;       // in log2 units

struct __align__(1024) SharedStorage {
    uint8_t q[Q_BYTES];
    uint8_t k[NSTAGE][TILE_BYTES];
    uint8_t v[NSTAGE][TILE_BYTES];
    uint64_t q_full;
    uint64_t k_full[NSTAGE], k_empty[NSTAGE], v_full[NSTAGE], v_empty[NSTAGE];
    uint64_t s_full, p_full, o_done;
    uint32_t tmem_base;
    int skip;
    uint32_t gave_up;                       // offset of the barrier whose wait ran out (0: none did)
};
#define AT(field) (base + (uint32_t)offsetof(SharedStorage, field))     // shared-memory address

struct KvTile {
    int seg;        // 0 or 1
    int coord;      // first row of the tile inside its tensor
    int n_valid;    // valid keys in the tile (1..64)
};

__device__ __forceinline__ KvTile kv_tile(const FwdWork& w, int tiles0, int j) {
    KvTile t;
    if (j < tiles0) {
        t.seg = 0;
        t.coord = w.s0_begin + j * BN;
        t.n_valid = min(BN, w.s0_end - t.coord);
    } else {
        t.seg = 1;
        t.coord = w.s1_begin + (j - tiles0) * BN;
        t.n_valid = min(BN, w.s1_end - t.coord);
    }
    return t;
}

// columns issued for a tile with n_valid keys (a multiple of 16)
__device__ __forceinline__ int tile_cols(int n_valid) { return (n_valid + 15) & ~15; }

template <int N> __device__ __forceinline__ void reg_inc() {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N> __device__ __forceinline__ void reg_dec() {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

__global__ void __launch_bounds__(NUM_THREADS, 4)
hmar_fwd_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k0,
                   const __grid_constant__ CUtensorMap map_v0, const __grid_constant__ CUtensorMap map_k1,
                   const __grid_constant__ CUtensorMap map_v1, const FwdArgs args) {
    // aligned by its declaration, so that every shared-memory address is a constant of the code; checked below
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    SharedStorage& sm = *reinterpret_cast<SharedStorage*>(smem_raw);
    const uint32_t base = smem_u32(&sm);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;

    if ((base & 1023u) != 0) {
        if (threadIdx.x == 0) report_gave_up(args.status, 0x3FF);
        return;
    }
    // ---- which tile of which head
    int bh, wi;
    const int group = args.by_group((int)blockIdx.x);
    if (args.work != nullptr) {
        const int first_head = group * args.group_heads, in_group = (int)blockIdx.x - first_head * args.n_work;
        const bool whole = first_head + args.group_heads <= args.n_heads;
        wi = whole ? args.by_group_heads(in_group) : args.by_last_heads(in_group);
        bh = first_head + in_group - wi * (whole ? args.group_heads : args.n_heads - first_head);
    } else {
        bh = group;
        wi = (int)blockIdx.x - bh * args.n_work;
    }
    const int batch = args.by_batch(bh), head = bh - batch * args.heads_per_batch;
    FwdWork w;
    if (args.work != nullptr) {
        w = args.work[wi];
    } else {   // inference step: dense window, previous scale then current scale
        w.row_begin = wi * BM;
        w.row_count = min(BM, args.n_q_rows - w.row_begin);
        w.s0_begin = 0; w.s0_end = args.n0;
        w.s1_begin = 0; w.s1_end = args.n1;
        w.uniform = 1;
    }
    const int tiles0 = (w.s0_end - w.s0_begin + BN - 1) / BN;
    const int tiles1 = (w.s1_end - w.s1_begin + BN - 1) / BN;
    const int n_tiles = tiles0 + tiles1;

    // ---- set-up
    int given_up = 0;
    if (threadIdx.x == 0) {
        sm.gave_up = 0;
        mbar_init(&sm.q_full, 1);
        for (int s = 0; s < NSTAGE; ++s) {
            mbar_init(&sm.k_full[s], 1);
            mbar_init(&sm.k_empty[s], 1);
            mbar_init(&sm.v_full[s], 1);
            mbar_init(&sm.v_empty[s], 1);
        }
        mbar_init(&sm.s_full, 1);
        mbar_init(&sm.p_full, NUM_SOFTMAX_THREADS);
        mbar_init(&sm.o_done, 1);
        fence_mbar_init();
        grid_wait();
        // whether a block of this launch (or an earlier one) already gave up on a wait: asked for now, looked at after the set-up
        if (args.status != nullptr) given_up = *reinterpret_cast<volatile int*>(args.status);
        // The block's first copies (Q, first K and V tiles) start here, before the TMEM allocation and the
        // block-wide barrier, so that their latency overlaps the rest of the set-up.
        const KvTile t0 = kv_tile(w, tiles0, 0);
        mbar_arrive_expect_tx(&sm.q_full, Q_BYTES);
        tma_load_4d(sm.q, &map_q, &sm.q_full, 0, w.row_begin, head, batch);
        mbar_arrive_expect_tx(&sm.k_full[0], TILE_BYTES);
        tma_load_4d(sm.k[0], t0.seg ? &map_k1 : &map_k0, &sm.k_full[0], 0, t0.coord, head, batch);
        mbar_arrive_expect_tx(&sm.v_full[0], TILE_BYTES);
        tma_load_4d(sm.v[0], t0.seg ? &map_v1 : &map_v0, &sm.v_full[0], 0, t0.coord, head, batch);
    }
    if (warp == MMA_WARP) {
        grid_wait();
        tmem_alloc(&sm.tmem_base, TMEM_COLS);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) sm.skip = given_up;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem_base;
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return warp_wait_or_give_up(bar, parity, &sm.gave_up, bar - base); };

    if (sm.skip != 0) {
        // do no further work; the first copies have to land before the block's shared memory is given back
        if (warp == 0) wait(AT(q_full), 0) && wait(AT(k_full), 0) && wait(AT(v_full), 0);
    } else if (warp >= PRODUCER_WARP) {
        reg_dec<REGS_MISC>();
        if (warp == PRODUCER_WARP) {
            // ================================================================== TMA producer
            // The whole warp runs the control flow; one elected lane issues the copies (a warp that has split
            // into one running lane and 31 parked ones issues far more slowly).
            const bool leader = elect_one();
            if (leader) {
                prefetch_tensormap(&map_q);
                prefetch_tensormap(&map_k0);
                prefetch_tensormap(&map_v0);
            }
            __syncwarp();
            bool ok = true;
            for (int j = 1; j < n_tiles && ok; ++j) {           // tile 0 was requested during the set-up
                const int slot = j % NSTAGE;
                const uint32_t par = ((j / NSTAGE) & 1) ^ 1;     // parity of the previous use of the slot
                const KvTile t = kv_tile(w, tiles0, j);
                if (j >= NSTAGE) ok = wait(AT(k_empty) + (slot) * 8, par);
                if (!ok) break;
                if (leader) {
                    bar_expect_tx(AT(k_full) + (slot) * 8, TILE_BYTES);
                    tma_load_4d_at(AT(k) + slot * TILE_BYTES, t.seg ? &map_k1 : &map_k0, AT(k_full) + (slot) * 8, 0, t.coord, head, batch);
                }
                __syncwarp();
                if (j >= NSTAGE) ok = wait(AT(v_empty) + (slot) * 8, par);
                if (!ok) break;
                if (leader) {
                    bar_expect_tx(AT(v_full) + (slot) * 8, TILE_BYTES);
                    tma_load_4d_at(AT(v) + slot * TILE_BYTES, t.seg ? &map_v1 : &map_v0, AT(v_full) + (slot) * 8, 0, t.coord, head, batch);
                }
                __syncwarp();
            }
            if (!ok) {
                // give the copies already issued a bounded chance to land before the block exits
                const uint64_t t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 2000000ull) { }
            }
        } else if (warp == MMA_WARP) {
            // ================================================================== MMA issuer
            // The whole warp runs the control flow; one elected lane issues.  Descriptors are built once and
            // advanced by adding (byte offset >> 4), so issuing an MMA costs a few instructions.
            const bool leader = elect_one();
            const uint64_t q_kd = smem_desc_sw128(AT(q), 16);
            const uint64_t k_kd0 = smem_desc_sw128(AT(k), 16);      // ring slots are 8 KB apart
            const uint64_t v_mn0 = smem_desc_sw128(AT(v), 1024);
            constexpr uint32_t idesc_pv = idesc_bf16_f32(BM, D, false, true);
            constexpr uint32_t SLOT_UNITS = TILE_BYTES >> 4;
            // S = Q K^T for n keys of the tile in ring slot `slot`
            auto issue_s = [&](int n, int slot) {
                const uint32_t idesc = idesc_bf16_f32(BM, n, false, false);
                const uint64_t kd = k_kd0 + slot * SLOT_UNITS;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    mma_ss(tmem + COL_S, q_kd + ks * 2, kd + ks * 2, idesc, ks > 0);
                commit_at(AT(s_full));
            };
            // O += P V for n keys
            auto issue_pv = [&](int n, int slot, bool first) {
                const int nk = n / 16;
                const uint64_t vd = v_mn0 + slot * SLOT_UNITS;
#pragma unroll
                for (int ks = 0; ks < BN / 16; ++ks)
                    if (ks < nk)
                        mma_ts(tmem + COL_O, tmem + COL_S + ks * 8, vd + ks * 128, idesc_pv, !first || (ks > 0));
            };

            bool ok = true;
            {
                bool rq, rk;
                warp_try_wait2(AT(q_full), 0, AT(k_full), 0, rq, rk);
                ok = (rq || wait(AT(q_full), 0)) && (rk || wait(AT(k_full), 0));
            }
            if (ok) {
                tc_fence_after();
                if (leader) {
                    issue_s(tile_cols(kv_tile(w, tiles0, 0).n_valid), 0);
                    if (NSTAGE < n_tiles) commit_at(AT(k_empty) + (0) * 8);
                }
                __syncwarp();
            }
            for (int j = 0; j < n_tiles && ok; ++j) {
                const int slot = j % NSTAGE, slot_next = (j + 1) % NSTAGE;
                const bool more = j + 1 < n_tiles;
                const int n = tile_cols(kv_tile(w, tiles0, j).n_valid);
                const int n_next = more ? tile_cols(kv_tile(w, tiles0, j + 1).n_valid) : 0;
                // one burst: O += P V of tile j, then S of tile j + 1 over the columns P leaves.  The copies are
                // looked at first (normally long complete), both looks sent before either answer is used: a look
                // at a barrier is a shared-memory round trip, and after the softmax warps' arrival every such trip
                // delays the products they are waiting for.
                {
                    const uint32_t v_bar = AT(v_full) + slot * 8, v_par = (j / NSTAGE) & 1;
                    const uint32_t k_bar = more ? AT(k_full) + slot_next * 8 : v_bar, k_par = more ? ((j + 1) / NSTAGE) & 1 : v_par;
                    bool rv, rk;
                    warp_try_wait2(v_bar, v_par, k_bar, k_par, rv, rk);
                    ok = (rv || wait(v_bar, v_par)) && (rk || wait(k_bar, k_par));
                }
                // The last tile of a key segment may be ragged: the rows between its last key and the next multiple of
                // 16 (the granularity of the product over keys) belong to another scale, or to nobody.  Their P is
                // exactly 0, but 0 x (Inf or NaN) is NaN, so these V rows are cleared before O += P V reads them:
                // a non-finite value outside a row's window cannot reach its output.  (Whole rows: the 128-byte swizzle
                // permutes 16-byte pieces inside a row only.)
                if (ok) {
                    const int n_valid = kv_tile(w, tiles0, j).n_valid;
                    if (n_valid < n) {
                        for (int idx = n_valid * 8 + lane; idx < n * 8; idx += 32)
                            *reinterpret_cast<uint4*>(sm.v[slot] + idx * 16) = make_uint4(0u, 0u, 0u, 0u);
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                    }
                }
                if (ok) ok = wait(AT(p_full), j & 1);
                if (!ok) break;
                tc_fence_after();
                if (leader) {
                    issue_pv(n, slot, j == 0);
                    if (n_next > 0) issue_s(n_next, slot_next);
                    // V of tile j and K of tile j + 1 have been handed to their last readers; a slot is signalled
                    // free only if a later tile will use it (the block may exit as soon as the softmax warps have
                    // seen o_done: an arrival that lands after that would hit the barriers of the next block on
                    // this SM)
                    if (j + NSTAGE < n_tiles) commit_at(AT(v_empty) + (slot) * 8);
                    if (j + 1 + NSTAGE < n_tiles) commit_at(AT(k_empty) + (slot_next) * 8);
                    if (!more) commit_at(AT(o_done));
                }
                __syncwarp();
            }
        }
    } else {
        // The registers move for a whole warpgroup: all of its threads execute this one instruction, and what tells its
        // warps apart comes after it.
        reg_inc<REGS_SOFTMAX>();
        if (warp * 32 >= w.row_count) {
            // ============================================================== softmax warp past the tile's last row
            // It only answers: its rows of P hold whatever S left there and reach its rows of O alone.  A scale of 324
            // tokens has one such warp in twelve, one of 169 two in eight.
#pragma unroll 1
            for (int j = 0; j < n_tiles; ++j) {
                if (!wait(AT(s_full), j & 1)) break;
                bar_arrive(AT(p_full));
            }
        } else {
            // ============================================================== softmax warps + epilogue
            const int r = warp * 32 + lane;                        // row inside the tile
            const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
            const int row = w.row_begin + r;
            const bool row_ok = r < w.row_count;
            int lo = w.s0_begin, hi = w.s0_end;                    // per-row key bounds (training, packed tiles)
            if (!w.uniform && row_ok) {
                const int s = scale_of_row(args.st, row);
                lo = args.st.start[first_key_scale(args.st.window, s)];
                hi = args.st.start[last_key_scale(args.st.window, s) + 1];
            }
            const float sl2 = args.scale_log2;
            const uint32_t s_addr = lane_base + COL_S;
            const uint32_t o_addr = lane_base + COL_O;
            float m_used = -INFINITY, l = 0.f;
            bool ok = true;
            uint32_t b0[32], b1[32];

            for (int j = 0; j < n_tiles && ok; ++j) {
                const KvTile t = kv_tile(w, tiles0, j);
                const int n = tile_cols(t.n_valid);
                // key c of the tile is visible to this row iff c in [c_lo, c_hi)
                const int c_lo = w.uniform ? 0 : max(lo - t.coord, 0);
                const int c_hi = w.uniform ? t.n_valid : min(hi - t.coord, t.n_valid);
                const bool two = n > 32;                           // second 32-column chunk present
                const bool need_mask = (!w.uniform) || (t.n_valid < (two ? 64 : 32));

                ok = wait(AT(s_full), j & 1);
                if (!ok) break;
                tc_fence_after();

                tmem_ld32(s_addr, b0);
                if (two) tmem_ld32(s_addr + 32, b1);
                tmem_ld_wait();

                // masked logits become -inf once, so the maximum and the exponentials treat them alike (columns the
                // tensor core did not write hold stale values and lie outside [c_lo, c_hi) too)
                if (need_mask) {
                    // A bit per column, and a test of one constant bit per logit: bounds compared logit by logit were four hundred
                    // instructions, run once or twice in a block and fetched for it (L = 680 960 heads 123 -> 116 us, 128 heads
                    // 25 -> 23, inference step 13 -> 18 1536 heads 142 -> 132.5, 9 -> 13 384 heads 25 -> 23).
                    uint32_t v0, v1;
                    visible_columns(c_lo, c_hi, v0, v1);
#pragma unroll
                    for (int i = 0; i < 32; ++i)
                        if (!(v0 >> i & 1u)) b0[i] = 0xff800000u;
                    if (two) {
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (!(v1 >> i & 1u)) b1[i] = 0xff800000u;
                    }
                }
                float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};     // four chains of maxima, not one of 64
#pragma unroll
                for (int i = 0; i < 32; ++i) mx4[i & 3] = fmaxf(mx4[i & 3], __uint_as_float(b0[i]));
                if (two) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) mx4[i & 3] = fmaxf(mx4[i & 3], __uint_as_float(b1[i]));
                }
                const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * sl2;     // softmax_scale > 0

                // Keep the running maximum unless this tile exceeds it by more than the threshold.  O is quiet
                // here: the product that precedes S of this tile in the tensor core's queue is the last one that
                // wrote it, and the next one waits for these warps.
                const bool grow = mx > m_used + kRescaleThreshold;  // false for -inf > -inf
                if (__any_sync(0xffffffffu, grow)) {
                    const float m_new = fmaxf(m_used, mx);
                    const float f = (m_used == -INFINITY) ? 0.f : ex2(m_used - m_new);
                    m_used = m_new;
                    l *= f;
                    if (j > 0) {
#pragma unroll 1
                        for (int piece = 0; piece < 4; ++piece) {
                            uint32_t o[16];
                            tmem_ld16(o_addr + piece * 16, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                            tmem_st16(o_addr + piece * 16, o);
                        }
                    }
                }
                const float m_sub = (m_used == -INFINITY) ? 0.f : m_used;

                // P = 2^(s * scale - m): fp32 row sum, bf16 P written over the S columns already read.  Pairs of logits share an
                // instruction but for the exponential: with the exponentials' pipe 85 % busy while four blocks are in their loops,
                // the issue slots between them count (one by one: L = 680 960 heads 114.1 -> 117.1 to 118.8 us, L = 2240 384 heads 2 to 8 %,
                // inference step 13 -> 18 1536 heads 138 -> 141, 24 -> 32 384 heads 239 -> 245.5).  The compiler takes the maxima above by
                // threes on its own, and O / l in pairs changes nothing.
                uint32_t packed[16];
                const uint64_t sl2_2 = f32x2(sl2, sl2), m_2 = f32x2(-m_sub, -m_sub);
                uint64_t l_2 = f32x2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < 32; i += 2) {
                    float x0, x1;
                    f32x2_split(ffma2(f32x2(__uint_as_float(b0[i]), __uint_as_float(b0[i + 1])), sl2_2, m_2), x0, x1);
                    const float p0 = ex2(x0), p1 = ex2(x1);
                    l_2 = fadd2(l_2, f32x2(p0, p1));
                    packed[i / 2] = pack_bf16(p0, p1);
                }
                tmem_st16(s_addr, packed);
                if (two) {
#pragma unroll
                    for (int i = 0; i < 32; i += 2) {
                        float x0, x1;
                        f32x2_split(ffma2(f32x2(__uint_as_float(b1[i]), __uint_as_float(b1[i + 1])), sl2_2, m_2), x0, x1);
                        const float p0 = ex2(x0), p1 = ex2(x1);
                        l_2 = fadd2(l_2, f32x2(p0, p1));
                        packed[i / 2] = pack_bf16(p0, p1);
                    }
                    tmem_st16(s_addr + 16, packed);
                }
                float l_a, l_b;
                f32x2_split(l_2, l_a, l_b);
                l += l_a + l_b;
                tmem_st_wait();
                tc_fence_before();
                bar_arrive(AT(p_full));
            }

            // ---- epilogue: out = O / l, lse = ln(l) + m (natural log of the scaled logits' sum)
            if (ok) ok = wait(AT(o_done), 0);
            if (ok) {
                tc_fence_after();
                const float inv = 1.f / l;
                tmem_ld32(o_addr, b0);
                tmem_ld32(o_addr + 32, b1);
                tmem_ld_wait();
                const long long lse_off = (long long)bh * args.n_q_rows + row;
                if (row_ok && args.lse != nullptr && HMAR_IN_BOUNDS(lse_off >= 0 && lse_off < args.lse_extent, args.status, 0xB102))
                    args.lse[lse_off] = (m_used + log2f(l)) * 0.6931471805599453f;
                // The warp's 32 rows go through the shared memory of its own query rows (read for the last time by the products
                // that o_done covers), 16-byte pieces swizzled by the row, so that a store instruction covers four whole rows and
                // not a piece of each of 32 (L1 takes a line at a time: 256 lines a warp, now 32).
                uint8_t* stage = sm.q + warp * 4096;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t* src = i < 4 ? b0 + 8 * i : b1 + 8 * (i - 4);
                    uint4 v4;
                    v4.x = pack_bf16(__uint_as_float(src[0]) * inv, __uint_as_float(src[1]) * inv);
                    v4.y = pack_bf16(__uint_as_float(src[2]) * inv, __uint_as_float(src[3]) * inv);
                    v4.z = pack_bf16(__uint_as_float(src[4]) * inv, __uint_as_float(src[5]) * inv);
                    v4.w = pack_bf16(__uint_as_float(src[6]) * inv, __uint_as_float(src[7]) * inv);
                    *reinterpret_cast<uint4*>(stage + lane * 128 + ((i ^ (lane & 7)) << 4)) = v4;
                }
                __syncwarp();
                // Two rounds at a time: a block runs this code once, so what it costs is largely the fetching of it (all eight
                // unrolled with their addresses worked out from scratch 1 to 2 % more: L = 680 960 heads 119.3 -> 121.8 us).
                const int piece = lane & 7, rr0 = lane >> 3;
                long long off = batch * args.out_batch_stride + head * args.out_head_stride + (w.row_begin + warp * 32 + rr0) * args.out_row_stride + piece * 8;
                const long long step = 4 * args.out_row_stride;
                const int rows = w.row_count - warp * 32;
#pragma unroll 2
                for (int rr = rr0; rr < 32; rr += 4, off += step) {
                    const uint4 v4 = *reinterpret_cast<const uint4*>(stage + rr * 128 + ((piece ^ (rr & 7)) << 4));
                    if (rr < rows && HMAR_IN_BOUNDS(off >= 0 && off + 8 <= args.out_extent, args.status, 0xB101))
                        *reinterpret_cast<uint4*>(args.out + off) = v4;
                }
            }
        }
    }

    // ---- tear-down
    tc_fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0) report_gave_up(args.status, sm.gave_up);
}

// Self-test of the bounded waits: a warp waits on a barrier that nothing ever arrives on, with a limit of about a
// millisecond, through the very wait and report functions the kernels use, and a second warp waits, three times as long,
// for the first.  Both give up; the block records HMAR_ERR_DEVICE_TIMEOUT with the first one's location, 0xD1A6, in the
// status word and returns; nothing traps.
__global__ void hmar_selftest_wait_kernel(int* status) {
    __shared__ uint64_t never, after;
    __shared__ uint32_t gave_up;
    if (threadIdx.x == 0) {
        gave_up = 0;
        mbar_init(&never, 1);
        mbar_init(&after, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        if (warp_wait_or_give_up(smem_u32(&never), 0, &gave_up, 0xD1A6, 2000000u) && threadIdx.x == 0) bar_arrive(smem_u32(&after));
    } else {
        warp_wait_or_give_up(smem_u32(&after), 0, &gave_up, 0xD1A7, 6000000u);
    }
    __syncthreads();
    if (threadIdx.x == 0) report_gave_up(status, gave_up);
}

}  // namespace

cudaError_t launch_selftest_wait(int* status, cudaStream_t stream) {
    hmar_selftest_wait_kernel<<<1, 64, 0, stream>>>(status);
    count_launch(1);
    return cudaGetLastError();
}

size_t fwd_tc_smem_bytes() { return sizeof(SharedStorage); }

cudaError_t launch_fwd_tc(const CUtensorMap& q, const CUtensorMap& k0, const CUtensorMap& v0, const CUtensorMap& k1,
                          const CUtensorMap& v1, const FwdArgs& args, int BH, cudaStream_t stream) {
    const size_t smem = fwd_tc_smem_bytes();
    static SmemOptIn opt_in;
    const cudaError_t e = opt_in((const void*)hmar_fwd_tc_kernel, smem);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)BH * (unsigned)args.n_work;
    // The blocks of a training pass go group by group of heads and, inside a group, costliest tiles first over its heads:
    // with all tiles of a head in turn, the last blocks to start hold costly tiles and the launch ends in a thin wave.
    // A group's Q, K and V are what L2 holds, since a head's rows are read once per tile of the head: one group of all
    // heads is slower where they exceed it (L = 2240, 384 heads: 425 us, head by head 412).  Head by head -> groups, us:
    // L = 2240 96 heads 115 -> 100, 192 heads 200 -> 186, 384 heads 365 -> 352; L = 9451 48 heads 675 -> 610, 192 heads
    // 2355 -> 2295; L = 680 128 heads 30 -> 26; L = 1000 192 heads 55 -> 49; L = 1300 39 heads 43 -> 34; L = 680 960
    // heads and L = 395 768 heads equal.  Groups of 48 MB are 1 to 4 % slower than these, of 96 or 160 MB equal.
    // The tiles of an inference step all cost the same, and stay head by head (groups: 0 to 15 % slower).
    FwdArgs a = args;
    const size_t groups = (BH * args.head_bytes + kL2Bytes - 1) / kL2Bytes;
    a.n_heads = BH;
    a.group_heads = (int)((BH + groups - 1) / groups);
    if (args.work != nullptr) {
        a.by_group = FastDiv((uint32_t)a.group_heads * (uint32_t)a.n_work);
        a.by_group_heads = FastDiv((uint32_t)a.group_heads);
        a.by_last_heads = FastDiv((uint32_t)((BH - 1) % a.group_heads + 1));
    } else {
        a.by_group = FastDiv((uint32_t)a.n_work);
    }
    a.by_batch = FastDiv((uint32_t)a.heads_per_batch);
    {
        KernelTimer timer(args.work != nullptr ? "hmar_fwd_tc_kernel" : "hmar_fwd_tc_kernel/scale_step", stream);
        const cudaError_t launched = launch_overlapped(hmar_fwd_tc_kernel, grid, NUM_THREADS, smem, stream, q, k0, v0, k1, v1, a);
        if (launched != cudaSuccess) return launched;
    }
    count_launch(1);
    return cudaGetLastError();
}

}  // namespace hmar
