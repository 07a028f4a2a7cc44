// Backward pass of the text rows on the sm_100a tensor cores (head_dim D = 128 or 64): dK / dV and dQ.
//
// Both kernels keep two 128 x D operand tiles resident in shared memory (A1, A2) and stream the tiles
// of the other two operands (B1: three TMA-filled stages, B2: two) past them.  Per streamed tile j the
// tensor pipe computes two products into TMEM, X_j = A1 B1_j^T and Y_j = A2 B2_j^T (128 x 128, fp32),
// and the row warps turn them into bf16 operands for the accumulating MMAs in two phases:
//   phase A (after X_j)   P = exp2(X scale - lse) on the visible pairs, kept in registers
//   phase B (after Y_j)   dS = P (Y - delta), written as bf16 over the first half of Y's own columns
// TMEM (512 columns): X [0,128), Y [128,256), accumulators from 256.
//
//   dK / dV  key-stationary and transposed: A1 = K tile, A2 = V tile (text or summary stream), B1 = Q tile,
//            B2 = dO tile of the (query tile, query head) pairs that see the keys; X = S^T, Y = dP^T.
//            The warps hand X back as soon as it is in their registers, so X_{j+1} runs beside the
//            exponentials of tile j; phase B goes through each warp's 32-column block of Y in two halves of
//            16 queries and writes dS^T over the first 8 and P^T over the other 8 columns of the half just
//            read, with one arrival per half: the accumulations over the first halves (k-steps 0, 2, 4, 6)
//            run beside the arithmetic of the second.  Pipe order per j: X_{j+1}, dV += P^T dO_j and
//            dK += dS^T Q_j (even k-steps, then odd), Y_{j+1}.  At the end each key row adds dV and
//            scale * dK to the fp32 accumulators of its stream: vector atomics where several segments cover a key
//            tile, plain stores where one CTA does (text keys, bwd_text_keys_stored).
//   dQ       query-stationary: A1 = Q tile, A2 = dO tile, B1 = K tile, B2 = V tile over the visible
//            summary tiles, then the visible text tiles (Eq. 3); X = S, Y = dP.  One accumulator leaves
//            room for a second Y buffer (columns from 384), so both products of tile j + 1 are issued
//            as soon as the warps have read X_j, and the warps never wait for the pipe: order per j:
//            X_{j+1}, Y_{j+1}, dQ += dS K_j.  At the end scale * dQ goes to the caller's tensor as bf16.
//
// A CTA (one per SM) works through many units -- a key tile with a segment of query tiles, or a query tile of one head -- one
// after the other; see "the units of a CTA" below.  The streams of tiles run on across units: stages, barriers and the Y buffers
// are counted over all tiles of the CTA, and the next unit's loads and first products run beside the last unit's epilogue.
//
// Warps 0-15: one accumulator row per thread, four warps per row quarter (warps w, w + 4, w + 8, w + 12
// share the lanes 32 (w % 4) ..; each takes 32 of the 128 columns: the element-wise work has no reduction
// across columns, and four warps per scheduler hide the TMEM load / store latencies); warp 16: TMA
// producer and the unit descriptors; warp 17: MMA issuer, a converged warp of which one lane issues; warps 18, 19 only make the
// fifth warpgroup whole, for the register hand-over.  Role, loop counts and waits are known to the compiler as the same in all
// lanes (votes and reductions of the warp), so that addresses, descriptors and loop control stay in uniform registers: with the
// warp number as threadIdx.x / 32 and waits of single lanes the two kernels took 12 - 14 % longer.  The
// tensor pipe works in order, so the completion of a product also tells which stage the accumulation before it
// has finished with: in the dQ kernel row warp 0, which sees every completion of X and Y, passes that on to
// the producer through one "empty" barrier per stage (except for the K stages, which the early products would
// otherwise release too late); in the dK / dV kernel the issuer commits to the "empty" barriers right behind
// each accumulation.  (The producer itself may fall several completions behind, which a parity wait on a
// shared barrier cannot follow: hence one barrier per stage.)  Every mbarrier wait is bounded (status word +
// CTA-wide abort flag).
//
// What bounds them: the row warps and the shared-memory reads of the products (X and Y read both operands from there: 160 KB a
// tile of dQ and 192 KB of dK / dV beside 64 KB that TMA writes, at 128 bytes a cycle).  Thousand cycles of 148 SMs, a CTA per
// unit -> CTAs that stay: 2 x 8,192 tokens in 64 + 8 chunks, 32/8 heads: dQ 961 -> 774, dK / dV 454 + 878 -> 386 + 751 (tensor pipe
// 73, 69 and 74 % active at 2 x 32,768); 7,942 ragged tokens, 16/16 heads, packed: 206 -> 155, 77 + 270 -> 70 + 217.  A training
// layer 2,107 -> 1,983 us, 585 -> 548 us; 2 x 32,768 tokens 14.5 -> 13.9 ms (power cap).  Full tiles read in place take these
// ragged launches 118 us of dQ where packed ones take 104, 191 of dK / dV where they take 185, and spare 52 us of pack.
// dK / dV spills 8 bytes (32 of loads) at head_dim 128, 4 (24) at 64; dQ nothing.
// A unit's end costs about 3,500 cycles (last product, epilogue, first loads of the next unit's scalars) where the end of a CTA
// and the start of the next took some 10,000.  The scalars of the next tile are negated when they are stored and not beside their
// load, which stalled every tile of dK / dV for it (5 - 7 %).
// Tried and taken back: a second issuing warp (dQ 811 -> 841), the Q / K stage checked a tile ahead (759 -> 943).
#include <cuda_bf16.h>

#include <algorithm>

#include "ksa_bwd.h"
#include "ksa_launch.h"
#include "ksa_ptx.cuh"

namespace ksa {

using namespace ptx;

constexpr int kBwdTcThreads = 640;              // five warpgroups
constexpr int kBwdTcRegs = 96;                  // five warps on a scheduler, 5 x 32 x 96 registers fit its file
constexpr int kBwdRegsRows = 104, kBwdRegsOther = 64;        // after the hand-over
static_assert(16 * kBwdRegsRows + 4 * kBwdRegsOther <= 20 * kBwdTcRegs, "register hand-over exceeds the CTA's allocation");
constexpr int kBwdSegPairs = 64;                // dK / dV: (query tile, query head) pairs per CTA, at least 16 query tiles
constexpr int kB1Stages = 3, kB2Stages = 2;

// shared memory map (bytes from the 1024-aligned base) for head_dim D
template <int D>
struct BtMap {
    static constexpr int kTile = 128 * D * 2;   // one 128 x D bf16 tile: [64-element half of d][128 rows][128 B]
    static constexpr int kOffA1 = 0, kOffA2 = kTile, kOffB1 = 2 * kTile, kOffB2 = kOffB1 + kB1Stages * kTile;
    static constexpr int kOffBars = kOffB2 + kB2Stages * kTile;                        // 25 barriers
    static constexpr int kOffMisc = kOffBars + 256;                                    // TMEM slot, abort flags, next block
    static constexpr int kOffRow = kOffMisc + 64;                                      // dK / dV: [2][lse, delta][128] per-query scalars
    static constexpr int kOffUnit = kOffRow + 2 * 2 * 128 * 4;                         // two unit descriptors of 64 bytes
    static constexpr int kLayoutBytes = kOffUnit + 128;
    // head_dim 128: the whole opt-in window (the layout needs all but 576 bytes of it); 64: the layout and the slack
    // for its 1024-byte alignment
    static constexpr int kSmem = D == 128 ? 232448 : kLayoutBytes + 1024;
    static_assert(kLayoutBytes <= kSmem, "shared memory layout");
};
enum : int { BB_AFULL = 0, BB_B1FULL = 1, BB_B2FULL = 4, BB_XFULL = 6, BB_YFULL = 7, BB_PA = 8, BB_PB = 9, BB_OFULL = 10,
             BB_B1EMPTY = 11, BB_B2EMPTY = 14, BB_YFULL2 = 16, BB_PB2 = 17,
             BB_AEMPTY = 18, BB_UFULL = 19, BB_UEMPTY = 21, BB_CLC = 23, BB_DRAIN = 24 };
// words of a unit descriptor
enum : int { U_J = 0, U_TEXT_OFF = 1, U_TILE = 2, U_HEAD = 3, U_A = 4, U_B = 5, U_C = 6, U_AUG = 8 };

__device__ __forceinline__ uint32_t bt_ld_shared(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void bt_st_shared(uint32_t addr, uint32_t v)
{
    asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ bool bt_wait(uint32_t bar, uint32_t parity, uint32_t abort_addr, int32_t* status, int code)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (uint32_t it = 1;; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0u) {
            if (bt_ld_shared(abort_addr) != 0u) return false;
            if (clock64() - t0 > (1ll << 31)) {
                atomicCAS(status, 0, code);
                bt_st_shared(abort_addr, 1u);
                return false;
            }
        }
    }
}
// A converged warp waits, every branch on a vote of the whole warp: after a wait of each lane, or of one lane, for itself the
// compiler no longer takes the warp for converged (dK / dV 822 -> 759 thousand cycles; cases of the head comment)
// progress: the address of a word that changes while somebody still works towards this barrier; the limit then starts again.
__device__ __forceinline__ bool bt_wait_converged(uint32_t bar, uint32_t parity, uint32_t abort_addr, int32_t* status, int code,
                                                  long long limit = 1ll << 31, uint32_t progress = 0)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    long long t0 = clock64();
    uint32_t seen = 0;
    for (uint32_t it = 1;; ++it) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if ((it & 63u) == 0u) {
            if (__any_sync(0xffffffffu, bt_ld_shared(abort_addr) != 0u)) return false;
            if (__any_sync(0xffffffffu, clock64() - t0 > limit)) {
                if (progress != 0u) {
                    const uint32_t now = __shfl_sync(0xffffffffu, bt_ld_shared(progress), 0);
                    if (now != seen) { seen = now; t0 = clock64(); continue; }
                }
                atomicCAS(status, 0, code);
                bt_st_shared(abort_addr, 1u);
                return false;
            }
        }
    }
}

// Shared-memory layout and barrier addresses of one CTA.
template <int D>
struct BtSmem {
    using M = BtMap<D>;
    uint32_t base;
    __device__ __forceinline__ uint32_t a1() const { return base + M::kOffA1; }
    __device__ __forceinline__ uint32_t a2() const { return base + M::kOffA2; }
    __device__ __forceinline__ uint32_t b1(int stage) const { return base + M::kOffB1 + (uint32_t)stage * M::kTile; }
    __device__ __forceinline__ uint32_t b2(int stage) const { return base + M::kOffB2 + (uint32_t)stage * M::kTile; }
    __device__ __forceinline__ uint32_t bar(int i) const { return base + M::kOffBars + 8u * (uint32_t)i; }
    __device__ __forceinline__ uint32_t tmem_slot() const { return base + M::kOffMisc; }
    __device__ __forceinline__ uint32_t abort_addr() const { return base + M::kOffMisc + 4; }
    __device__ __forceinline__ uint32_t blocks_taken() const { return base + M::kOffMisc + 12; }       // answered requests
    __device__ __forceinline__ uint32_t next_block() const { return base + M::kOffMisc + 16; }
    __device__ __forceinline__ uint32_t unit(int n, int word) const { return base + M::kOffUnit + (uint32_t)(n & 1) * 64u + 4u * (uint32_t)word; }
};

// The layout starts on the first 1024-byte boundary of the dynamic window; false (and a status code) if it
// does not fit behind it.  Uniform over the CTA: everybody returns before any barrier is touched.
template <int D>
__device__ __forceinline__ bool bt_layout(BtSmem<D>& sm, const uint8_t* raw, int32_t* status)
{
    const uint32_t raw_addr = smem_u32(raw);
    sm.base = (raw_addr + 1023u) & ~1023u;
    if (sm.base - raw_addr + (uint32_t)BtMap<D>::kLayoutBytes > (uint32_t)BtMap<D>::kSmem) {
        if (threadIdx.x == 0) atomicCAS(status, 0, (int)kStatusSmemLayout);
        return false;
    }
    return true;
}

// The barriers, by the producer's thread, which goes on to its first loads at once: they run beside the rest of the
// set-up (TMEM, the row warps' scalars).  bt_ready() is where everybody meets.
template <int D>
__device__ __forceinline__ void bt_init_barriers(const BtSmem<D>& sm)
{
    mbar_init(sm.bar(BB_AFULL), 1);
    for (int s = 0; s < kB1Stages; ++s) { mbar_init(sm.bar(BB_B1FULL + s), 1); mbar_init(sm.bar(BB_B1EMPTY + s), 1); }
    for (int s = 0; s < kB2Stages; ++s) { mbar_init(sm.bar(BB_B2FULL + s), 1); mbar_init(sm.bar(BB_B2EMPTY + s), 1); }
    mbar_init(sm.bar(BB_XFULL), 1);
    mbar_init(sm.bar(BB_YFULL), 1);
    mbar_init(sm.bar(BB_YFULL2), 1);
    mbar_init(sm.bar(BB_PA), 16);
    mbar_init(sm.bar(BB_PB), 16);
    mbar_init(sm.bar(BB_PB2), 16);
    mbar_init(sm.bar(BB_OFULL), 1);
    mbar_init(sm.bar(BB_AEMPTY), 1);
    for (int s = 0; s < 2; ++s) { mbar_init(sm.bar(BB_UFULL + s), 1); mbar_init(sm.bar(BB_UEMPTY + s), 17); }   // 16 row warps and the issuer
    mbar_init(sm.bar(BB_CLC), 1);
    mbar_init(sm.bar(BB_DRAIN), 1);
    bt_st_shared(sm.abort_addr(), 0u);
    bt_st_shared(sm.abort_addr() + 4, 0u);
    bt_st_shared(sm.blocks_taken(), 0u);
    fence_mbar_init();
}
template <int D>
__device__ __forceinline__ void bt_ready(const BtSmem<D>& sm, int warp)
{
    if (warp == 17) { tmem_alloc(sm.tmem_slot(), 512); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}

// ---- MMA issue helpers (a converged warp; `leader` != 0 in the issuing lane) -------------------------
// D[tmem_d] = A B^T, both 128 x D tiles K-major in shared memory ([64-element half of d][128 rows][128 B]).
template <int D>
__device__ __forceinline__ void bt_product(uint32_t leader, uint32_t tmem_d, uint32_t a_tile, uint32_t b_tile)
{
    constexpr uint32_t idesc = make_idesc_bf16(128, 128, false), hi = smem_desc_hi_sw128(1024);
    const uint32_t ad = smem_desc_lo(a_tile, 16), bd = smem_desc_lo(b_tile, 16);
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t off = (uint32_t)(((kk >> 2) * 16384 + (kk & 3) * 32) >> 4);
        mma_ss_warp(leader, tmem_d, ad + off, bd + off, hi, idesc, kk > 0 ? 1u : 0u);
    }
}
// D[tmem_d] (+)= A B: A = 128 x 128 bf16 in TMEM (16 packed columns at the start of every 32-column chunk of
// tmem_a), B = a 128 x D tile in shared memory read MN-major (64-element atoms of d 16384 bytes apart,
// 8-row groups 1024 bytes apart): D accumulator columns.
template <int D>
__device__ __forceinline__ void bt_accumulate(uint32_t leader, uint32_t tmem_d, uint32_t tmem_a, uint32_t b_tile, bool first)
{
    constexpr uint32_t idesc = make_idesc_bf16(128, D, true), hi = smem_desc_hi_sw128(1024);
    const uint32_t bd = smem_desc_lo(b_tile, 16384);
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
        mma_ts_warp(leader, tmem_d, tmem_a + (kk >> 1) * 32 + (kk & 1) * 8, bd + (uint32_t)((kk * 2048) >> 4), hi, idesc, (!first || kk > 0) ? 1u : 0u);
}

// Half of such an accumulation for the dK / dV kernel, whose row warps hand their 32-column blocks over in two
// halves of 16 query columns: the four k-steps 2 c + odd, whose 16 x bf16 operand stands in the 8 columns at
// tmem_a + 32 c + 16 odd (tmem_a already points at dS^T, or 8 columns further at P^T).
template <int D>
__device__ __forceinline__ void bt_accumulate_half(uint32_t leader, uint32_t tmem_d, uint32_t tmem_a, uint32_t b_tile, int odd, bool first)
{
    constexpr uint32_t idesc = make_idesc_bf16(128, D, true), hi = smem_desc_hi_sw128(1024);
    const uint32_t bd = smem_desc_lo(b_tile, 16384);
#pragma unroll
    for (int c = 0; c < 4; ++c)
        mma_ts_warp(leader, tmem_d, tmem_a + c * 32 + odd * 16, bd + (uint32_t)(((2 * c + odd) * 2048) >> 4), hi, idesc, (!first || c > 0) ? 1u : 0u);
}

// ---- producer helpers (one thread) ----------------------------------------------------------------
// Tile `tile` of a sequence's text (summary) rows, its two 64-column halves, as ReadMode says: rows of a 3-D map of a packed
// stream, or chunks of a 4-D (5-D) view [D, rows per chunk, (start,) chunk, head] of the caller's interleaved tensor, whose box
// lands in shared memory as the same dense tile.
struct BtPlace {
    int mode, per_text, per_summ;                                         // ReadMode, chunks of a text / a summary tile
    int chunk0, start, text_off, summ_off, n_text, n_summ;                // of the sequence
};
__device__ __forceinline__ BtPlace bt_place(const BwdArgs& a, const SeqInfo& sq)
{
    return BtPlace{a.direct, 128 / a.k, a.m > 0 ? 128 / a.m : 0, sq.chunk0, a.direct == kReadTails ? row_in_chunk(sq, a.k, a.m) : 0,
                   sq.text_off, sq.summ_off, sq.n_text, sq.n_summ};
}
template <int D>
__device__ __forceinline__ void bt_issue_tile(uint32_t dst, uint32_t bar, const CUtensorMap* map, const CUtensorMap* tail, const BtPlace& p, bool summ, int tile, int head)
{
    const int row = (summ ? p.summ_off : p.text_off) + tile * 128, chunk = p.chunk0 + tile * (summ ? p.per_summ : p.per_text);
#pragma unroll
    for (int h = 0; h < D / 64; ++h) {
        const uint32_t to = dst + h * 16384;
        if (p.mode == kReadInPlace) tma_load_4d(to, map, bar, h * 64, 0, chunk, head);
        else if (p.mode == kReadPacked) tma_load_3d(to, map, bar, h * 64, row, head);
        else if ((tile + 1) * 128 <= (summ ? p.n_summ : p.n_text)) tma_load_5d(to, map, bar, h * 64, 0, p.start, chunk, head);
        else tma_load_3d(to, tail, bar, h * 64, row, head);
    }
}
template <int D>
__device__ __forceinline__ void bt_load_tile(uint32_t dst, uint32_t bar, const CUtensorMap* map, const CUtensorMap* tail, const BtPlace& p, bool summ, int tile, int head)
{
    mbar_arrive_expect_tx(bar, (uint32_t)BtMap<D>::kTile);
    bt_issue_tile<D>(dst, bar, map, tail, p, summ, tile, head);
}
// After an abort: leave no copy in flight.  Bounded waits (the second flag is never set) for the last fill of
// every stage; filled_a / filled1 / filled2 = A pairs / B1 / B2 tiles whose load was issued; asked = requests for a block that
// were answered, pending: one more is on its way.
template <int D>
__device__ __forceinline__ void bt_drain(const BtSmem<D>& sm, int filled_a, int filled1, int filled2, bool pending, int asked, int32_t* status)
{
    const uint32_t never = sm.abort_addr() + 4;
    if (pending) bt_wait(sm.bar(BB_CLC), (uint32_t)(asked & 1), never, status, kStatusWaitNextBlock);
    if (filled_a > 0) bt_wait(sm.bar(BB_AFULL), (uint32_t)((filled_a - 1) & 1), never, status, kStatusWaitKvFull);
    for (int s = 0; s < kB1Stages; ++s) {
        const int fills = (filled1 + kB1Stages - 1 - s) / kB1Stages;     // tiles j < filled1 with j % 3 == s
        if (fills > 0) bt_wait(sm.bar(BB_B1FULL + s), (uint32_t)((fills - 1) & 1), never, status, kStatusWaitQFull);
    }
    for (int s = 0; s < kB2Stages; ++s) {
        const int fills = (filled2 + kB2Stages - 1 - s) / kB2Stages;
        if (fills > 0) bt_wait(sm.bar(BB_B2FULL + s), (uint32_t)((fills - 1) & 1), never, status, kStatusWaitQFull);
    }
}

// The issuer's end: no product is in flight when TMEM is freed (after an abort, too).
template <int D>
__device__ __forceinline__ void bt_drain_pipe(uint32_t leader, const BtSmem<D>& su, int32_t* status)
{
    tc_commit_warp(leader, su.bar(BB_DRAIN));
    bt_wait(su.bar(BB_DRAIN), 0, su.abort_addr() + 4, status, kStatusWaitOFull);
}

// A stage is about to take tile j of the CTA (tiles are counted over its units): wait until its previous tile was released.
template <int D>
__device__ __forceinline__ bool bt_stage_free(const BtSmem<D>& sm, int empty0, int stages, int j, int32_t* status)
{
    if (j < stages) return true;
    return bt_wait(sm.bar(empty0 + j % stages), (uint32_t)((j / stages - 1) & 1), sm.abort_addr(), status, kStatusWaitQEmpty);
}

// ---- the units of a CTA ---------------------------------------------------------------------------
// The grid has a block for every unit of work, and a CTA that is through with its own unit takes over the next block that has
// not started (cluster launch control: the block is cancelled, its index comes back through shared memory) until none is left.
// The producer's thread does that, works out what the unit is, and hands it to the other warps as a descriptor in shared memory
// (two slots); J = 0 ends the CTA.
struct BtBlock { int x, y, z; };
template <int D>
__device__ __forceinline__ void bt_request_block(const BtSmem<D>& sm)
{
    fence_proxy_async();                                                  // the slot was read by this thread
    mbar_arrive_expect_tx(sm.bar(BB_CLC), 16u);
    clc_try_cancel(sm.next_block(), sm.bar(BB_CLC));
}
// The answer to request number `n` of the CTA: 1 and the block, 0 if none was left (nothing is asked for after that), -1 if the
// wait gave up.
template <int D>
__device__ __forceinline__ int bt_take_block(const BtSmem<D>& sm, int n, BtBlock& blk, int32_t* status)
{
    if (!bt_wait(sm.bar(BB_CLC), (uint32_t)(n & 1), sm.abort_addr(), status, kStatusWaitNextBlock)) return -1;
    return clc_query(sm.next_block(), blk.x, blk.y, blk.z) ? 1 : 0;
}
// The other side for dK / dV: descriptor n is there.  The producer may have to pass any number of blocks without work on its way
// to the next unit (every tile has the segments that a tile of the longest sequence may need): a long sequence among 65,000 short
// ones has tens of millions of them in a row, at 2 us each on 148 SMs a second's worth, so the limit holds from one to the next.
#ifdef KSA_DEBUG
constexpr long long kUnitWaitCycles = 1ll << 19;        // (so that a test of milliseconds passes it)
#else
constexpr long long kUnitWaitCycles = 1ll << 31;
#endif
template <int D>
__device__ __forceinline__ bool bt_wait_unit(const BtSmem<D>& sm, int n, int32_t* status)
{
    return bt_wait_converged(sm.bar(BB_UFULL + (n & 1)), (uint32_t)((n >> 1) & 1), sm.abort_addr(), status, kStatusWaitUnit, kUnitWaitCycles, sm.blocks_taken());
}
// A word of descriptor n for a whole warp, known to the compiler as the same in every lane: loop counts and addresses that come
// of it stay in uniform registers.
template <int D>
__device__ __forceinline__ int bt_unit_word(const BtSmem<D>& sm, int n, int word)
{
    return (int)__reduce_or_sync(0xffffffffu, bt_ld_shared(sm.unit(n, word)));
}
// The producer's side of the slots: descriptor n may be written / has been written.
template <int D>
__device__ __forceinline__ bool bt_unit_free(const BtSmem<D>& sm, int n, int32_t* status)
{
    if (n < 2) return true;
    return bt_wait(sm.bar(BB_UEMPTY + (n & 1)), (uint32_t)(((n >> 1) - 1) & 1), sm.abort_addr(), status, kStatusWaitUnit);
}

// =====================================================================================================
// dK / dV
// =====================================================================================================
// A unit: one key tile, one KV head, a segment of the query tiles that see the keys.  Block (x, y): segment x % segs of key tile
// x / segs of the packed stream (its rows are numbered over all sequences), KV head y.  (Segments first: the units in flight
// then share their query tiles.  Tiles first, the launch over the summary keys at 32,768 tokens read them from memory again and
// again and took 4,060 instead of 3,390 us.)
struct BtDkvUnit { int J, kt, hk, seg0, n_keys, krow0; BtPlace at; };
__device__ __forceinline__ bool bt_dkv_unit(const BwdArgs& a, const BtBlock& blk, const int summ, const int seg_tiles, const int segs, BtDkvUnit& u)
{
    const int tile = blk.x / segs;
    const SeqInfo sq = a.seqs[seq_of_row(a.seqs, a.num_seqs, tile * 128, !summ)];
    u.krow0 = tile * 128;
    u.kt = tile - (summ ? sq.summ_off : sq.text_off) / 128;
    u.hk = blk.y;
    u.n_keys = summ ? sq.n_summ : sq.n_text;
    u.at = bt_place(a, sq);
    if (u.kt * 128 >= u.n_keys) return false;
    const int n_qt = (sq.n_text + 127) / 128;
    int qt_lo, qt_hi;                                                     // the query tiles that see the keys (Eq. 3)
    if (!summ) {
        const int key_last = min(u.n_keys, u.kt * 128 + 128) - 1;
        qt_lo = u.kt;
        const long long i_max = ((long long)(key_last / a.k) + a.C + 1) * a.k - 1;
        qt_hi = (int)min((long long)(n_qt - 1), i_max / 128);
    } else {
        const long long i_min = ((long long)(u.kt * 128) / a.m + 1 + a.C) * a.k;     // first row that sees summary kt*128
        if (i_min >= sq.n_text) return false;
        qt_lo = (int)(i_min / 128);
        qt_hi = n_qt - 1;
    }
    u.seg0 = qt_lo + (blk.x - tile * segs) * seg_tiles;
    if (u.seg0 > qt_hi) return false;
    u.J = (min(qt_hi + 1, u.seg0 + seg_tiles) - u.seg0) * (a.Hq / a.Hkv);            // streamed tiles: (query tile, query head) pairs
    return true;
}

template <int D>
__device__ __forceinline__ void bt_dkv_block(const BwdArgs& a, const BwdMaps& maps, const int summ, const int seg_tiles, const int segs, const int store)
{
    extern __shared__ uint8_t bsm_raw[];
    const int warp = (int)__reduce_or_sync(0xffffffffu, threadIdx.x >> 5), lane = threadIdx.x & 31;       // (uniform to the compiler)
    const int G = a.Hq / a.Hkv;
    BtSmem<D> sm;
    if (!bt_layout(sm, bsm_raw, a.status)) return;

    // ---- the producer's thread: descriptor and loads of a unit ------------------------------------
    BtDkvUnit u{};
    bool started = false;                                                 // unit 0: described, first tile on its way
    auto publish = [&](int n) {
        bt_st_shared(sm.unit(n, U_TEXT_OFF), (uint32_t)u.at.text_off); bt_st_shared(sm.unit(n, U_TILE), (uint32_t)u.kt);
        bt_st_shared(sm.unit(n, U_HEAD), (uint32_t)u.hk); bt_st_shared(sm.unit(n, U_A), (uint32_t)u.seg0);
        bt_st_shared(sm.unit(n, U_B), (uint32_t)u.n_keys); bt_st_shared(sm.unit(n, U_C), (uint32_t)u.krow0);
        bt_st_shared(sm.unit(n, U_J), (uint32_t)u.J);
        mbar_arrive(sm.bar(BB_UFULL + (n & 1)));
    };
    auto load_a = [&]() {                                                 // K and V tile
        mbar_arrive_expect_tx(sm.bar(BB_AFULL), 2u * BtMap<D>::kTile);
        bt_issue_tile<D>(sm.a1(), sm.bar(BB_AFULL), summ ? &maps.ks : &maps.kt, summ ? &maps.ks_tail : &maps.kt_tail, u.at, summ != 0, u.kt, u.hk);
        bt_issue_tile<D>(sm.a2(), sm.bar(BB_AFULL), summ ? &maps.vs : &maps.vt, summ ? &maps.vs_tail : &maps.vt_tail, u.at, summ != 0, u.kt, u.hk);
    };
    auto load_b = [&](int j, uint32_t dst, uint32_t bar, const CUtensorMap* map, const CUtensorMap* tail) {   // pair (query tile, head of the group) j
        bt_load_tile<D>(dst, bar, map, tail, u.at, false, u.seg0 + j / G, u.hk * G + j % G);
    };
    if (warp == 16 && lane == 0) {
        bt_init_barriers(sm);
        started = bt_dkv_unit(a, BtBlock{(int)blockIdx.x, (int)blockIdx.y, 0}, summ, seg_tiles, segs, u);
        if (started) {
            load_b(0, sm.b1(0), sm.bar(BB_B1FULL), &maps.qt, &maps.qt_tail);
            load_a();
            load_b(0, sm.b2(0), sm.bar(BB_B2FULL), &maps.dot, &maps.dot_tail);
            publish(0);
        }
    }
    bt_ready(sm, warp);
    const uint32_t tmem = bt_ld_shared(sm.tmem_slot());
    const uint32_t tX = tmem, tY = tmem + 128u, tDV = tmem + 256u, tDK = tmem + 384u;

    if (warp >= 16) {
        setmaxnreg_dec<kBwdRegsOther>();
        if (warp == 16) { if (lane == 0) {
            // =============================== TMA producer ===============================
            int na = started ? 1 : 0, g1 = na, g2 = na, asked = 0;        // A pairs, B1 and B2 tiles loaded; answered requests
            bool alive = true, pending = false, took_first = false;      // ... the grid's first block among them
            for (int n = 0; alive; ++n) {
                if (!started) {                                           // the next block that holds work
                    u.J = 0;
                    for (;;) {
                        if (!pending) { bt_request_block(sm); pending = true; }
                        BtBlock blk;
                        const int got = bt_take_block(sm, asked, blk, a.status);
                        if (got < 0) { alive = false; break; }
                        ++asked; pending = false;
                        bt_st_shared(sm.blocks_taken(), (uint32_t)asked);
                        took_first |= got > 0 && blk.x + blk.y == 0;
                        if (got == 0 || bt_dkv_unit(a, blk, summ, seg_tiles, segs, u)) break;
                        u.J = 0;
                    }
                    if (!alive || !bt_unit_free(sm, n, a.status)) { alive = false; break; }
                    publish(n);
                    if (u.J == 0) break;                                  // none left: the CTA ends
                }
                for (int j = started ? 1 : 0; j < u.J; ++j) {
                    if (j + 1 == u.J) { bt_request_block(sm); pending = true; }          // comes while the stages are waited for
                    if (!bt_stage_free(sm, BB_B1EMPTY, kB1Stages, g1, a.status)) { alive = false; break; }
                    load_b(j, sm.b1(g1 % kB1Stages), sm.bar(BB_B1FULL + g1 % kB1Stages), &maps.qt, &maps.qt_tail);
                    ++g1;
                    if (j == 0) {                                         // the unit before has formed its last products
                        if (na > 0 && !bt_wait(sm.bar(BB_AEMPTY), (uint32_t)((na - 1) & 1), sm.abort_addr(), a.status, kStatusWaitQEmpty)) { alive = false; break; }
                        load_a();
                        ++na;
                    }
                    if (!bt_stage_free(sm, BB_B2EMPTY, kB2Stages, g2, a.status)) { alive = false; break; }
                    load_b(j, sm.b2(g2 & 1), sm.bar(BB_B2FULL + (g2 & 1)), &maps.dot, &maps.dot_tail);
                    ++g2;
                }
                started = false;
            }
            if (bt_ld_shared(sm.abort_addr()) != 0u) bt_drain(sm, na, g1, g2, pending, asked, a.status);
            if (took_first) pdl_wait();                                    // (see the launches)
        } } else if (warp == 17) {
            // =============================== MMA issuer =================================
            // the whole warp walks the loop on warp-uniform values, one lane issues
            const uint32_t leader = elect_one();
            const uint32_t tm = __reduce_or_sync(0xffffffffu, tmem), base = __reduce_or_sync(0xffffffffu, sm.base);
            const BtSmem<D> su{base};
            const uint32_t uX = tm, uY = tm + 128u, uDV = tm + 256u, uDK = tm + 384u;
            auto wait = [&](uint32_t bar, uint32_t parity, int code) -> bool {
                return bt_wait_converged(bar, parity, su.abort_addr(), a.status, code);
            };
            bool alive = true;
            int g = 0, s1 = 0;                                            // tiles of the units before; the next tile's B1 stage ...
            uint32_t b1_phase = 0;                                        // ... and the parity of its fill
            for (int n = 0; alive; ++n) {
                if (!bt_wait_unit(su, n, a.status)) break;
                const int Ju = bt_unit_word(su, n, U_J);
                mbar_arrive_warp(leader, su.bar(BB_UEMPTY + (n & 1)));
                if (Ju == 0) break;
                alive = wait(su.bar(BB_AFULL), n & 1, kStatusWaitKvFull) && wait(su.bar(BB_B1FULL + s1), b1_phase, kStatusWaitQFull);
                if (!alive) break;
                // (X and Y are free: every row warp has handed over the last tile of the unit before)
                bt_product<D>(leader, uX, su.a1(), su.b1(s1));
                tc_commit_warp(leader, su.bar(BB_XFULL));
                if (!wait(su.bar(BB_B2FULL + (g & 1)), (g >> 1) & 1, kStatusWaitQFull)) break;
                bt_product<D>(leader, uY, su.a2(), su.b2(g & 1));
                tc_commit_warp(leader, su.bar(BB_YFULL));
                if (Ju == 1) tc_commit_warp(leader, su.bar(BB_AEMPTY));
                for (int j = 0; j < Ju; ++j, ++g) {
                    const int s1n = s1 + 1 == kB1Stages ? 0 : s1 + 1;
                    if (s1n == 0) b1_phase ^= 1u;
                    if (j + 1 < Ju && !(alive = wait(su.bar(BB_B1FULL + s1n), b1_phase, kStatusWaitQFull))) break;
                    // the warps hold X_j in registers: the next S^T product may overwrite it while they exponentiate
                    if (!(alive = wait(su.bar(BB_PA), g & 1, kStatusWaitPFull))) break;
                    tc_fence_after();
                    if (j + 1 < Ju) {
                        bt_product<D>(leader, uX, su.a1(), su.b1(s1n));
                        tc_commit_warp(leader, su.bar(BB_XFULL));
                    }
                    // dS^T and P^T of the first 16 queries of every block stand in Y's columns: the even k-steps
                    if (!(alive = wait(su.bar(BB_PB), g & 1, kStatusWaitPFull))) break;
                    tc_fence_after();
                    bt_accumulate_half<D>(leader, uDV, uY + 8, su.b2(g & 1), 0, j == 0);            // dV += P^T dO_j
                    bt_accumulate_half<D>(leader, uDK, uY, su.b1(s1), 0, j == 0);                   // dK += dS^T Q_j
                    // ... the other 16: the odd k-steps
                    if (j + 1 < Ju && !(alive = wait(su.bar(BB_B2FULL + ((g + 1) & 1)), ((g + 1) >> 1) & 1, kStatusWaitQFull))) break;
                    if (!(alive = wait(su.bar(BB_PB2), g & 1, kStatusWaitPFull))) break;
                    tc_fence_after();
                    bt_accumulate_half<D>(leader, uDV, uY + 8, su.b2(g & 1), 1, false);
                    tc_commit_warp(leader, su.bar(BB_B2EMPTY + (g & 1)));                           // ... then its dO stage is free
                    bt_accumulate_half<D>(leader, uDK, uY, su.b1(s1), 1, false);
                    tc_commit_warp(leader, su.bar(BB_B1EMPTY + s1));                                // ... then its Q stage is free
                    if (j + 1 < Ju) {
                        bt_product<D>(leader, uY, su.a2(), su.b2((g + 1) & 1));
                        tc_commit_warp(leader, su.bar(BB_YFULL));
                        if (j + 2 == Ju) tc_commit_warp(leader, su.bar(BB_AEMPTY));                 // K and V may make way for the next unit's
                    }
                    s1 = s1n;
                }
                if (alive) tc_commit_warp(leader, su.bar(BB_OFULL));
            }
            bt_drain_pipe(leader, su, a.status);
        }
    } else {
        setmaxnreg_inc<kBwdRegsRows>();
        // =============================== key rows ===================================
        uint8_t* base_ptr = bsm_raw + (sm.base - smem_u32(bsm_raw));
        // per-query scalars of the streamed tile, negated, double-buffered by tile: [tile & 1][lse, delta][128 columns]; every
        // row warp writes the 32 columns it reads itself, one tile ahead (the four warps of a column group write the same
        // values, and each relies on its own writes only), see below
        float* rows = reinterpret_cast<float*>(base_ptr + BtMap<D>::kOffRow);
        const int quarter = warp & 3, cg = warp >> 2;                        // lanes 32 quarter ..; columns 32 cg ..
        const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
        const uint32_t tXc = tX + lane_sel + cg * 32, tYc = tY + lane_sel + cg * 32;    // this warp's 32 x 32 block
        const int kdiv = summ ? a.m : a.k;
        // The streamed tiles walk the pairs (query tile, head of the group) in order; the chunk of the block's first
        // query, i0 = 128 qt + 32 cg, is kept as quotient and remainder by k and advanced by 128 per query tile
        // (integer divisions are slow, and this loop is the warps' critical path).
        const int step_q = 128 / a.k, step_r = 128 - step_q * a.k, q31 = 31 / a.k, r31 = 31 - q31 * a.k;
        int J = 0, kt = 0, hk = 0, qt = 0, text_off = 0, krow0 = 0, key = 0;       // the unit; the next pair's query tile
        bool alive = true;
        auto take_unit = [&](int n) -> bool {
            if (!bt_wait_unit(sm, n, a.status)) return false;
            __syncwarp();
            J = bt_unit_word(sm, n, U_J); text_off = bt_unit_word(sm, n, U_TEXT_OFF);
            kt = bt_unit_word(sm, n, U_TILE); hk = bt_unit_word(sm, n, U_HEAD);
            qt = bt_unit_word(sm, n, U_A); krow0 = bt_unit_word(sm, n, U_C);
            const int key_raw = kt * 128 + quarter * 32 + lane;
            key = key_raw < bt_unit_word(sm, n, U_B) ? key_raw : 0x3fffffff;      // rows past the stream: never visible
            __syncwarp();
            if (lane == 0) mbar_arrive(sm.bar(BB_UEMPTY + (n & 1)));
            return true;
        };
        // This lane's scalars for the next tile, untouched until they are stored: the negation beside the load would wait for it
        // there and then, in front of every tile.
        float n_lse = 0.f, n_dl = 0.f;
        auto fetch = [&](int qt_, int g_) {                               // pair (query tile, head of the group)
            const size_t r = (size_t)(hk * G + g_) * a.text_rows + text_off + (size_t)qt_ * 128 + 32 * cg + lane;
            n_lse = __ldcg(a.lse_t + r);                                 // +inf on padding rows: P = 0 there
            n_dl = __ldcg(a.delta_t + r);                                // (past L1: see the launches)
        };
        auto put_scalars = [&](int tile) {
            rows[(tile & 1) * 256 + 32 * cg + lane] = -n_lse;
            rows[(tile & 1) * 256 + 128 + 32 * cg + lane] = -n_dl;
        };
        alive = take_unit(0);
        if (alive && J > 0) { fetch(qt, 0); put_scalars(0); __syncwarp(); }
        int t = 0;                                                        // tile, counted over the units
        for (int n = 0; alive && J > 0; ++n) {
            const int kq = key / kdiv;                                    // the key's chunk
            const int kq_first = (kt * 128) / kdiv, kq_last = (kt * 128 + 127) / kdiv;
            int g = 0;
            int iq0 = (qt * 128 + 32 * cg) / a.k, ir0 = (qt * 128 + 32 * cg) - iq0 * a.k;
            const int t_end = t + J;
            for (; t < t_end; ++t) {
                if (t + 1 < t_end) fetch(g + 1 == G ? qt + 1 : qt, g + 1 == G ? 0 : g + 1);   // lands while this tile is worked on
                const float4* lse_c = reinterpret_cast<const float4*>(rows + (t & 1) * 256 + 32 * cg);     // this warp's 32 columns
                const float4* dl_c = lse_c + 32;
                const int i0 = qt * 128 + 32 * cg;                            // first query of the block
                const int iq1 = iq0 + q31 + (ir0 + r31 >= a.k ? 1 : 0);       // chunk of the block's last query
                // ---------------- phase A: P^T = exp2(S^T scale - lse), kept in registers ----------------
                if (!bt_wait_converged(sm.bar(BB_XFULL), t & 1, sm.abort_addr(), a.status, kStatusWaitSFull)) { alive = false; break; }
                tc_fence_after();
                // all pairs of the block visible / none (rows past the streams drop out by themselves: zero K / V
                // rows are discarded at the end, padding queries have lse = +inf)
                bool full, none;
                if (!summ) {
                    full = kt * 128 + 127 <= i0 && iq1 - kq_first <= a.C;
                    none = kt * 128 > i0 + 31 || iq0 - kq_last > a.C;
                } else {
                    full = iq0 - kq_last > a.C;
                    none = iq1 - kq_first <= a.C;
                }
                uint32_t x[32];                                               // S^T, then P^T in place (fp32 bits), kept for phase B
                if (none) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) x[c] = 0u;
                } else {
                    tmem_ld32(tXc, x);
                    tc_wait_ld();
                }
                // X_j is in registers: the issuer may start X_{j+1} while the exponentials run.  (This hand-over and those
                // below order TMEM accesses only, which the fences and waits around them cover: relaxed arrivals.)
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_relaxed(sm.bar(BB_PA));
                if (!none) {
                    if (full) {
                        const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
#pragma unroll
                        for (int c = 0; c < 32; c += 4) {
                            const float4 l4 = lse_c[c >> 2];
                            const float2 v = ffma2(make_float2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), sc2, make_float2(l4.x, l4.y));
                            const float2 w = ffma2(make_float2(__uint_as_float(x[c + 2]), __uint_as_float(x[c + 3])), sc2, make_float2(l4.z, l4.w));
                            x[c] = __float_as_uint(ex2_approx(v.x));
                            x[c + 1] = __float_as_uint(ex2_approx(v.y));
                            x[c + 2] = __float_as_uint(ex2_approx(w.x));
                            x[c + 3] = __float_as_uint(ex2_approx(w.y));
                        }
                    } else {
                        int iq = iq0, ir = ir0;                               // chunk of query i0 + c, counted up from i0's
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            const bool vis = summ ? (iq - kq > a.C) : (key <= i0 + c && iq - kq <= a.C);
                            const float v = fmaf(__uint_as_float(x[c]), a.scale_log2, reinterpret_cast<const float*>(lse_c)[c]);
                            x[c] = __float_as_uint(ex2_approx(vis ? v : -INFINITY));
                            if (++ir == a.k) { ir = 0; ++iq; }
                        }
                    }
                }
                // ---------------- phase B: dS^T = P^T (dP^T - delta); both as bf16 over Y's own columns ----------------
                if (!bt_wait_converged(sm.bar(BB_YFULL), t & 1, sm.abort_addr(), a.status, kStatusWaitSFull)) { alive = false; break; }
                tc_fence_after();
                // Y_j was issued after every warp's arrival for tile j - 1: that tile's scalars may be overwritten
                if (t + 1 < t_end) put_scalars(t + 1);
                // handed over in two halves of 16 queries, so that the accumulations of the first run beside the
                // arithmetic of the second: columns 16 half + 0 .. 7 take dS^T, 16 half + 8 .. 15 take P^T
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    uint32_t o[16];
                    if (none) {
#pragma unroll
                        for (int c = 0; c < 16; ++c) o[c] = 0u;
                    } else {
                        uint32_t ys[16];
                        tmem_ld16(tYc + half * 16, ys);
                        tc_wait_ld();
#pragma unroll
                        for (int c = 0; c < 16; c += 4) {
                            const int e = half * 16 + c;
                            const float4 d4 = dl_c[e >> 2];
                            const float2 p2 = make_float2(__uint_as_float(x[e]), __uint_as_float(x[e + 1]));
                            const float2 q2 = make_float2(__uint_as_float(x[e + 2]), __uint_as_float(x[e + 3]));
                            const float2 s2 = fmul2(p2, fadd2(make_float2(__uint_as_float(ys[c]), __uint_as_float(ys[c + 1])), make_float2(d4.x, d4.y)));
                            const float2 r2 = fmul2(q2, fadd2(make_float2(__uint_as_float(ys[c + 2]), __uint_as_float(ys[c + 3])), make_float2(d4.z, d4.w)));
                            o[c >> 1] = pack_bf16x2(s2.x, s2.y);
                            o[(c >> 1) + 1] = pack_bf16x2(r2.x, r2.y);
                            o[8 + (c >> 1)] = pack_bf16x2(p2.x, p2.y);
                            o[9 + (c >> 1)] = pack_bf16x2(q2.x, q2.y);
                        }
                    }
                    tmem_st16(tYc + half * 16, o);                            // over the block's own columns of dP^T
                    tc_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_relaxed(sm.bar(half ? BB_PB2 : BB_PB));
                }
                if (++g == G) {                                               // next query tile
                    g = 0; ++qt;
                    iq0 += step_q; ir0 += step_r;
                    if (ir0 >= a.k) { ir0 -= a.k; ++iq0; }
                }
            }
            if (!alive) break;
            // odd cg: scale * dK, even cg: dV; cg / 2 picks the half of the row (D / 2 elements)
            // (tcgen05.ld is warp-collective: rows past the stream load, too)
            const bool is_dk = (cg & 1) != 0, row_ok = key != 0x3fffffff;
            const int d0 = (cg >> 1) * (D / 2);
            const size_t arow = (size_t)hk * (summ ? a.summ_rows : a.text_rows) + (size_t)krow0 + quarter * 32 + lane;
            float* acc = (is_dk ? (summ ? a.dks : a.dkt) : (summ ? a.dvs : a.dvt)) + acc_at(arow, d0, D);
            // the next unit and its first scalars, beside the last products (every warp's tile before the last is done: see above)
            if (!take_unit(n + 1)) break;
            if (J > 0) fetch(qt, 0);
            if (!bt_wait_converged(sm.bar(BB_OFULL), n & 1, sm.abort_addr(), a.status, kStatusWaitOFull)) break;
            tc_fence_after();
            const float mul = is_dk ? a.scale : 1.f;
            const uint32_t tacc = (is_dk ? tDK : tDV) + lane_sel + d0;
#pragma unroll
            for (int c = 0; c < D / 64; ++c) {
                uint32_t o[32];
                tmem_ld32(tacc + c * 32, o);
                tc_wait_ld();
                if (row_ok) {
                    // store: this CTA is the only one of its launch for these keys and the first writer of their rows
#pragma unroll
                    for (int e = 0; e < 32; e += 4) {
                        const float4 val = make_float4(__uint_as_float(o[e]) * mul, __uint_as_float(o[e + 1]) * mul,
                                                       __uint_as_float(o[e + 2]) * mul, __uint_as_float(o[e + 3]) * mul);
                        float4* at = reinterpret_cast<float4*>(acc + (c * 32 + e) / 4 * 512);        // (acc_at)
                        if (store) *at = val;
                        else atomicAdd(at, val);
                    }
                }
            }
            // the accumulators are read before this warp's first hand-over of the next unit, behind which they are overwritten
            tc_fence_before();
            if (J > 0) { put_scalars(t); __syncwarp(); }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 17) tmem_dealloc(tmem, 512);
}

// =====================================================================================================
// dQ
// =====================================================================================================
// A unit: one query tile and one query head, over the visible summary tiles, then the visible text tiles (Eq. 3).  Block
// (x, y): x-th query tile of the packed stream from its end (a sequence's long rows first), head y.
struct BtDqUnit { int J, n_s, t_lo, qt, h; BtPlace at; long long aug_off; };
__device__ __forceinline__ void bt_dq_unit(const BwdArgs& a, const BtBlock& blk, BtDqUnit& u)
{
    const int row0 = (int)a.text_rows - 128 - blk.x * 128;
    const SeqInfo sq = a.seqs[seq_of_row(a.seqs, a.num_seqs, row0, true)];
    u.qt = (row0 - sq.text_off) / 128;
    u.h = blk.y;
    u.at = bt_place(a, sq); u.aug_off = sq.aug_off;
    const int i_first = u.qt * 128, i_last = min(sq.n_text, i_first + 128) - 1;
    const int far_first = max(0, i_first / a.k - a.C), far_last = max(0, i_last / a.k - a.C);
    u.n_s = a.m > 0 ? (min(sq.n_summ, far_last * a.m) + 127) / 128 : 0;               // summary tiles seen by the last row
    u.t_lo = (int)(((long long)far_first * a.k) / 128);                                // first text tile seen by the first row
    u.J = u.n_s + u.qt - u.t_lo + 1;
}

template <int D>
__device__ __forceinline__ void bt_dq_block(const BwdArgs& a, const BwdMaps& maps)
{
    extern __shared__ uint8_t bsm_raw[];
    const int warp = (int)__reduce_or_sync(0xffffffffu, threadIdx.x >> 5), lane = threadIdx.x & 31;       // (uniform to the compiler)
    const int G = a.Hq / a.Hkv;
    BtSmem<D> sm;
    if (!bt_layout(sm, bsm_raw, a.status)) return;

    // ---- the producer's thread: descriptor and loads of a unit ------------------------------------
    BtDqUnit u{};
    auto publish = [&](int n) {
        bt_st_shared(sm.unit(n, U_TEXT_OFF), (uint32_t)u.at.text_off); bt_st_shared(sm.unit(n, U_TILE), (uint32_t)u.qt);
        bt_st_shared(sm.unit(n, U_HEAD), (uint32_t)u.h); bt_st_shared(sm.unit(n, U_A), (uint32_t)u.n_s);
        bt_st_shared(sm.unit(n, U_B), (uint32_t)u.t_lo); bt_st_shared(sm.unit(n, U_C), (uint32_t)u.at.n_text);
        bt_st_shared(sm.unit(n, U_AUG), (uint32_t)u.aug_off); bt_st_shared(sm.unit(n, U_AUG + 1), (uint32_t)(u.aug_off >> 32));
        bt_st_shared(sm.unit(n, U_J), (uint32_t)u.J);
        mbar_arrive(sm.bar(BB_UFULL + (n & 1)));
    };
    auto load_a = [&]() {                                                 // Q and dO tile
        mbar_arrive_expect_tx(sm.bar(BB_AFULL), 2u * BtMap<D>::kTile);
        bt_issue_tile<D>(sm.a1(), sm.bar(BB_AFULL), &maps.qt, &maps.qt_tail, u.at, false, u.qt, u.h);
        bt_issue_tile<D>(sm.a2(), sm.bar(BB_AFULL), &maps.dot, &maps.dot_tail, u.at, false, u.qt, u.h);
    };
    auto load_b = [&](int j, uint32_t dst, uint32_t bar, const CUtensorMap* map_s, const CUtensorMap* map_t, const CUtensorMap* tail_s, const CUtensorMap* tail_t) {
        const bool is_summ = j < u.n_s;
        bt_load_tile<D>(dst, bar, is_summ ? map_s : map_t, is_summ ? tail_s : tail_t, u.at, is_summ, is_summ ? j : u.t_lo + j - u.n_s, u.h / G);
    };
    if (warp == 16 && lane == 0) {
        bt_init_barriers(sm);
        bt_dq_unit(a, BtBlock{(int)blockIdx.x, (int)blockIdx.y, 0}, u);
        load_b(0, sm.b1(0), sm.bar(BB_B1FULL), &maps.ks, &maps.kt, &maps.ks_tail, &maps.kt_tail);
        load_a();
        load_b(0, sm.b2(0), sm.bar(BB_B2FULL), &maps.vs, &maps.vt, &maps.vs_tail, &maps.vt_tail);
        publish(0);
    }
    bt_ready(sm, warp);
    const uint32_t tmem = bt_ld_shared(sm.tmem_slot());
    const uint32_t tX = tmem, tDQ = tmem + 256u;
    // dP of tile j (counted over the CTA's units), then dS in place
    auto tY = [&](int j) -> uint32_t { return tmem + ((j & 1) ? 384u : 128u); };
    auto y_full = [&](int j) -> uint32_t { return sm.bar((j & 1) ? BB_YFULL2 : BB_YFULL); };
    // likewise one phase B barrier per Y buffer: with both products of tile j + 1 issued early, a warp may finish
    // tile j + 1 before another has finished tile j, and must not arrive in its phase
    auto p_b = [&](int j) -> uint32_t { return sm.bar((j & 1) ? BB_PB2 : BB_PB); };

    if (warp >= 16) {
        setmaxnreg_dec<kBwdRegsOther>();
        if (warp == 16) { if (lane == 0) {
            // =============================== TMA producer ===============================
            int na = 1, g1 = 1, g2 = 1, asked = 0;                        // A pairs, B1 and B2 tiles loaded; answered requests
            bool alive = true, pending = false, took_first = false;      // ... the grid's first block among them
            for (int n = 0; alive; ++n) {
                if (n > 0) {                                              // the next block
                    if (!pending) { bt_request_block(sm); pending = true; }
                    BtBlock blk;
                    const int got = bt_take_block(sm, asked, blk, a.status);
                    if (got < 0) break;
                    ++asked; pending = false;
                    took_first |= got > 0 && blk.x + blk.y == 0;
                    if (got > 0) bt_dq_unit(a, blk, u); else u.J = 0;
                    if (!bt_unit_free(sm, n, a.status)) break;
                    publish(n);
                    if (u.J == 0) break;                                  // none left: the CTA ends
                }
                for (int j = n > 0 ? 0 : 1; j < u.J; ++j) {
                    if (j + 1 == u.J) { bt_request_block(sm); pending = true; }          // comes while the stages are waited for
                    if (!bt_stage_free(sm, BB_B1EMPTY, kB1Stages, g1, a.status)) { alive = false; break; }
                    load_b(j, sm.b1(g1 % kB1Stages), sm.bar(BB_B1FULL + g1 % kB1Stages), &maps.ks, &maps.kt, &maps.ks_tail, &maps.kt_tail);
                    ++g1;
                    if (j == 0) {                                         // the unit before has formed its last products
                        if (!bt_wait(sm.bar(BB_AEMPTY), (uint32_t)((na - 1) & 1), sm.abort_addr(), a.status, kStatusWaitQEmpty)) { alive = false; break; }
                        load_a();
                        ++na;
                    }
                    if (!bt_stage_free(sm, BB_B2EMPTY, kB2Stages, g2, a.status)) { alive = false; break; }
                    load_b(j, sm.b2(g2 & 1), sm.bar(BB_B2FULL + (g2 & 1)), &maps.vs, &maps.vt, &maps.vs_tail, &maps.vt_tail);
                    ++g2;
                }
            }
            if (bt_ld_shared(sm.abort_addr()) != 0u) bt_drain(sm, na, g1, g2, pending, asked, a.status);
            if (took_first) pdl_wait();                                    // (see the launches)
        } } else if (warp == 17) {
            // =============================== MMA issuer =================================
            // the whole warp walks the loop on warp-uniform values, one lane issues
            const uint32_t leader = elect_one();
            const uint32_t tm = __reduce_or_sync(0xffffffffu, tmem), base = __reduce_or_sync(0xffffffffu, sm.base);
            const BtSmem<D> su{base};
            const uint32_t uX = tm, uDQ = tm + 256u;
            auto uY = [&](int j) -> uint32_t { return tm + ((j & 1) ? 384u : 128u); };
            auto u_full = [&](int j) -> uint32_t { return su.bar((j & 1) ? BB_YFULL2 : BB_YFULL); };
            auto wait = [&](uint32_t bar, uint32_t parity, int code) -> bool {
                return bt_wait_converged(bar, parity, su.abort_addr(), a.status, code);
            };
            bool alive = true;
            int g = 0, s1 = 0;                                            // tiles of the units before; the next tile's B1 stage ...
            uint32_t b1_phase = 0;                                        // ... and the parity of its fill
            for (int n = 0; alive; ++n) {
                if (!wait(su.bar(BB_UFULL + (n & 1)), (n >> 1) & 1, kStatusWaitUnit)) break;
                const int Ju = bt_unit_word(su, n, U_J);
                mbar_arrive_warp(leader, su.bar(BB_UEMPTY + (n & 1)));
                if (Ju == 0) break;
                alive = wait(su.bar(BB_AFULL), n & 1, kStatusWaitKvFull) && wait(su.bar(BB_B1FULL + s1), b1_phase, kStatusWaitQFull);
                if (!alive) break;
                // (X is free: every row warp has handed over the last tile of the unit before)
                bt_product<D>(leader, uX, su.a1(), su.b1(s1));
                tc_commit_warp(leader, su.bar(BB_XFULL));
                if (!wait(su.bar(BB_B2FULL + (g & 1)), (g >> 1) & 1, kStatusWaitQFull)) break;
                bt_product<D>(leader, uY(g), su.a2(), su.b2(g & 1));
                tc_commit_warp(leader, u_full(g));
                if (Ju == 1) tc_commit_warp(leader, su.bar(BB_AEMPTY));
                for (int j = 0; j < Ju; ++j, ++g) {
                    const int s1n = s1 + 1 == kB1Stages ? 0 : s1 + 1;
                    if (s1n == 0) b1_phase ^= 1u;
                    if (j + 1 < Ju) {
                        if (!(alive = wait(su.bar(BB_B1FULL + s1n), b1_phase, kStatusWaitQFull))) break;
                        if (!(alive = wait(su.bar(BB_B2FULL + ((g + 1) & 1)), ((g + 1) >> 1) & 1, kStatusWaitQFull))) break;
                        // phase A of tile j has read X into registers; the other Y buffer was read by dQ += dS K_{j-1}
                        if (!(alive = wait(su.bar(BB_PA), g & 1, kStatusWaitPFull))) break;
                        tc_fence_after();
                        bt_product<D>(leader, uX, su.a1(), su.b1(s1n));
                        tc_commit_warp(leader, su.bar(BB_XFULL));
                        bt_product<D>(leader, uY(g + 1), su.a2(), su.b2((g + 1) & 1));
                        tc_commit_warp(leader, u_full(g + 1));
                        if (j + 2 == Ju) tc_commit_warp(leader, su.bar(BB_AEMPTY));                // Q and dO may make way for the next unit's
                    }
                    if (!(alive = wait(su.bar((g & 1) ? BB_PB2 : BB_PB), (g >> 1) & 1, kStatusWaitPFull))) break;
                    tc_fence_after();
                    bt_accumulate<D>(leader, uDQ, uY(g), su.b1(s1), j == 0);                       // dQ += dS K_j
                    tc_commit_warp(leader, su.bar(BB_B1EMPTY + s1));                               // K_j is free after that
                    s1 = s1n;
                }
                if (alive) tc_commit_warp(leader, su.bar(BB_OFULL));
            }
            bt_drain_pipe(leader, su, a.status);
        }
    } else {
        setmaxnreg_inc<kBwdRegsRows>();
        // =============================== query rows =================================
        const int quarter = warp & 3, cg = warp >> 2;                     // lanes 32 quarter ..; columns 32 cg ..
        const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
        const uint32_t tXc = tX + lane_sel + cg * 32;                     // this warp's 32 x 32 block
        int J = 0, n_s = 0, i_w0 = 0;
        float lse2 = 0.f, dl = 0.f;
        // (the slot is handed back when the unit's output rows have been worked out, see below)
        auto take_unit = [&](int n) -> bool {
            if (!bt_wait_converged(sm.bar(BB_UFULL + (n & 1)), (n >> 1) & 1, sm.abort_addr(), a.status, kStatusWaitUnit)) return false;
            __syncwarp();
            J = bt_unit_word(sm, n, U_J);
            if (J == 0) return true;
            n_s = bt_unit_word(sm, n, U_A);
            i_w0 = bt_unit_word(sm, n, U_TILE) * 128 + quarter * 32;
            const size_t r = (size_t)bt_unit_word(sm, n, U_HEAD) * a.text_rows + bt_unit_word(sm, n, U_TEXT_OFF) + i_w0 + lane;
            lse2 = __ldcg(a.lse_t + r);                                  // +inf / 0 on padding rows: P = 0 there
            dl = __ldcg(a.delta_t + r);                                  // (past L1: see the launches)
            return true;
        };
        bool alive = take_unit(0);
        int j = 0;                                                        // tile, counted over the units
        for (int n = 0; alive && J > 0; ++n) {
            const int i = i_w0 + lane;
            const int iq = i / a.k, iq_w0 = i_w0 / a.k, iq_w1 = (i_w0 + 31) / a.k;
            // The chunk of the block's first key, kc0 = key0 + 32 cg, is kept as quotient and remainder by the keys per
            // chunk of its stream and advanced by 128 per tile (kc0: the key); divisions only where the stream starts (integer
            // divisions are slow, and this loop is the warps' critical path).
            int cdiv = 0, kc0 = 32 * cg, kq0 = 0, kr0 = 0, step_q = 0, step_r = 0, q31 = 0, r31 = 0;
            const int j_text = j + n_s, j_end = j + J;                    // first text tile, first tile of the next unit
            for (; j < j_end; ++j, kc0 += 128) {
                const bool is_summ = j < j_text;
                if (cdiv == 0 || j == j_text) {                               // first tile of the summary / the text stream
                    if (!is_summ) kc0 = bt_unit_word(sm, n, U_B) * 128 + 32 * cg;
                    cdiv = is_summ ? a.m : a.k;                               // keys per chunk in this stream
                    kq0 = kc0 / cdiv; kr0 = kc0 - kq0 * cdiv;
                    step_q = 128 / cdiv; step_r = 128 - step_q * cdiv;
                    q31 = 31 / cdiv; r31 = 31 - q31 * cdiv;
                } else {
                    kq0 += step_q; kr0 += step_r;
                    if (kr0 >= cdiv) { kr0 -= cdiv; ++kq0; }
                }
                const int kq1 = kq0 + q31 + (kr0 + r31 >= cdiv ? 1 : 0);      // chunk of the block's last key
                // the warp's 32 x 32 block: all visible, none, or mixed (zero rows past a stream add nothing to dQ).
                // Text key t is visible to row i iff t <= i and chunk(i) - chunk(t) <= C; summary key s iff
                // chunk(i) - chunk(s) > C (Eq. 3)
                bool full, none;
                if (is_summ) {
                    full = iq_w0 - kq1 > a.C;
                    none = iq_w1 - kq0 <= a.C;
                } else {
                    full = kc0 + 31 <= i_w0 && iq_w1 - kq0 <= a.C;
                    none = kc0 > i_w0 + 31 || iq_w0 - kq1 > a.C;
                }
                // ---------------- phase A: P = exp2(S scale - lse) ----------------
                if (!bt_wait_converged(sm.bar(BB_XFULL), j & 1, sm.abort_addr(), a.status, kStatusWaitSFull)) { alive = false; break; }
                tc_fence_after();
                uint32_t x[32];                                               // S, then P in place (fp32 bits)
                if (!none) {
                    tmem_ld32(tXc, x);
                    tc_wait_ld();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_relaxed(sm.bar(BB_PA));            // X may be overwritten from here on
                if (!none) {
                    if (full) {
                        const float2 sc2 = make_float2(a.scale_log2, a.scale_log2), nl2 = make_float2(-lse2, -lse2);
#pragma unroll
                        for (int c = 0; c < 32; c += 2) {
                            const float2 v = ffma2(make_float2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])), sc2, nl2);
                            x[c] = __float_as_uint(ex2_approx(v.x));
                            x[c + 1] = __float_as_uint(ex2_approx(v.y));
                        }
                    } else {
                        int kq = kq0, kr = kr0;                               // chunk of key kc0 + c, counted up from kc0's
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            const bool vis = is_summ ? (iq - kq > a.C) : (kc0 + c <= i && iq - kq <= a.C);
                            const float v = fmaf(__uint_as_float(x[c]), a.scale_log2, -lse2);
                            x[c] = __float_as_uint(ex2_approx(vis ? v : -INFINITY));
                            if (++kr == cdiv) { kr = 0; ++kq; }
                        }
                    }
                }
                // ---------------- phase B: dS = P (dP - delta) ----------------
                // one barrier per Y buffer: Y_{j+1} may be complete before a warp gets here for Y_j
                if (!bt_wait_converged(y_full(j), (j >> 1) & 1, sm.abort_addr(), a.status, kStatusWaitSFull)) { alive = false; break; }
                tc_fence_after();
                if (warp == 0 && lane == 0) mbar_arrive_relaxed(sm.bar(BB_B2EMPTY + (j & 1)));          // Y_j is complete: its V stage is free
                const uint32_t tYc = tY(j) + lane_sel + cg * 32;
                uint32_t dd[16];
                if (none) {
#pragma unroll
                    for (int c = 0; c < 16; ++c) dd[c] = 0u;
                } else {
                    uint32_t ys[32];
                    tmem_ld32(tYc, ys);
                    tc_wait_ld();
                    const float2 nd2 = make_float2(-dl, -dl);
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        const float2 d2 = fmul2(make_float2(__uint_as_float(x[c]), __uint_as_float(x[c + 1])),
                                                fadd2(make_float2(__uint_as_float(ys[c]), __uint_as_float(ys[c + 1])), nd2));
                        dd[c >> 1] = pack_bf16x2(d2.x, d2.y);
                    }
                }
                tmem_st16(tYc, dd);                                           // over the block's own first 16 columns
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_relaxed(p_b(j));
            }
            if (!alive) break;
            // scale * dQ as bf16 to the row's augmented position (Eq. 1); warp group cg writes elements 32 cg ..
            int64_t off = -1;                                             // -1: a padding row
            const int n_text = bt_unit_word(sm, n, U_C), h = bt_unit_word(sm, n, U_HEAD);
            const int64_t aug_off = (int64_t)(((unsigned long long)(uint32_t)bt_unit_word(sm, n, U_AUG + 1) << 32) | (uint32_t)bt_unit_word(sm, n, U_AUG));
            if (i < n_text) off = (aug_off + (int64_t)iq * (a.k + a.m) + (i - iq * a.k)) * a.dq_st + (int64_t)h * a.dq_sh + cg * 32;
            __syncwarp();
            if (lane == 0) mbar_arrive(sm.bar(BB_UEMPTY + (n & 1)));
            // the next unit and its rows' scalars, beside the last product
            if (!take_unit(n + 1)) break;
            if (!bt_wait_converged(sm.bar(BB_OFULL), n & 1, sm.abort_addr(), a.status, kStatusWaitOFull)) break;
            tc_fence_after();
            if (cg * 32 < D) {                                            // warp-uniform: the row has D elements
                uint32_t o[32];
                tmem_ld32(tDQ + lane_sel + cg * 32, o);
                tc_wait_ld();
                // (the accumulators are read before this warp's first hand-over of the next unit, behind which they are overwritten)
                tc_fence_before();
                uint4 w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    w[e].x = pack_bf16x2(__uint_as_float(o[8 * e]) * a.scale, __uint_as_float(o[8 * e + 1]) * a.scale);
                    w[e].y = pack_bf16x2(__uint_as_float(o[8 * e + 2]) * a.scale, __uint_as_float(o[8 * e + 3]) * a.scale);
                    w[e].z = pack_bf16x2(__uint_as_float(o[8 * e + 4]) * a.scale, __uint_as_float(o[8 * e + 5]) * a.scale);
                    w[e].w = pack_bf16x2(__uint_as_float(o[8 * e + 6]) * a.scale, __uint_as_float(o[8 * e + 7]) * a.scale);
                }
                quad_transpose(w, lane);                                  // w[e]: 16 bytes of the group's row e
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int64_t at = __shfl_sync(0xffffffffu, off, (lane & 28) + e);
                    if (at >= 0) *reinterpret_cast<uint4*>(a.dq + at + (lane & 3) * 8) = w[e];
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 17) tmem_dealloc(tmem, 512);
}

// The three launches -- dK / dV of the summary keys, of the text keys, dQ -- do not depend on each other: each one's CTAs take
// the SMs that the one in front leaves (programmatic dependent launches), longest CTAs first (64, about 40 and 9 + 16 tiles
// each at 32,768 tokens), so that the tails of the first two are filled (training layer of 7,942 ragged tokens, 16/16 heads
// 619 -> 590 us, 2 x 8,192 tokens 2,132 -> 2,064 us; nothing at 2 x 32,768).
// Nothing here waits for the launch in front, which was itself started behind the preparation; only the CTA that has the first
// block of each waits for its end when it is through, so that the kernel behind the three, an ordinary launch, finds all of them
// done.  What the preparation and the pack wrote stands in L2 by then, but without a wait of its own (pdl_wait) a kernel has no
// promise that its L1 has dropped those addresses' old contents: the tiles come by TMA, lse and delta by loads that bypass L1,
// the sums are added in L2.  A fence.acq_rel.gpu at the start of each CTA instead costs 0.7 - 1.6 % of a training layer.
// (The sequence table needs none of that: no kernel writes it, and the host has waited for its upload before it launches any
// kernel of the call, so the upload happens before all of them.  Read past L1, 1,000 short sequences beside one of 65,536 tokens
// took 8.46 -> 9.19 ms backward and, with the summary rows' kernel behind the text kernel, 2.88 -> 4.59 ms forward.)
// The CTA that started as the grid's first block; the producer's thread of a CTA that took that block over waits there.
__device__ __forceinline__ void bt_end_behind_front()
{
    if (blockIdx.x + blockIdx.y == 0) pdl_wait();
}
template <int D>
__global__ void __maxnreg__(kBwdTcRegs)
ksa_bwd_dkv_tc_kernel(const __grid_constant__ BwdArgs a, const __grid_constant__ BwdMaps maps, const int summ, const int seg_tiles, const int segs, const int store)
{
    pdl_launch_dependents();
    bt_dkv_block<D>(a, maps, summ, seg_tiles, segs, store);
    bt_end_behind_front();
}
template <int D>
__global__ void __maxnreg__(kBwdTcRegs)
ksa_bwd_dq_tc_kernel(const __grid_constant__ BwdArgs a, const __grid_constant__ BwdMaps maps)
{
    bt_dq_block<D>(a, maps);
    bt_end_behind_front();
}

cudaError_t setup_bwd_tc()
{
    cudaError_t e = cudaFuncSetAttribute(ksa_bwd_dkv_tc_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, BtMap<128>::kSmem);
    if (e != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(ksa_bwd_dq_tc_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, BtMap<128>::kSmem)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(ksa_bwd_dkv_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, BtMap<64>::kSmem)) != cudaSuccess) return e;
    return cudaFuncSetAttribute(ksa_bwd_dq_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, BtMap<64>::kSmem);
}

// Query tiles that see a text key tile (an upper bound), and the query tiles a CTA of the dK / dV kernel walks.
static long long bwd_text_span(const BwdArgs& a)
{
    return std::min<long long>(a.max_text_pad / 128, ((long long)a.C + 1) * a.k / 128 + 2);
}
static int bwd_seg_tiles(const BwdArgs& a) { return std::max(16, kBwdSegPairs / (a.Hq / a.Hkv)); }

// True if one CTA covers every query tile that sees a text key tile: then the text-key launch writes its rows of the
// accumulators with plain stores -- it must be their first writer (no clear needed; the summary rows' kernel adds later).
bool bwd_text_keys_stored(const BwdArgs& a) { return bwd_text_span(a) <= bwd_seg_tiles(a); }

cudaError_t launch_bwd_tc(const BwdArgs& a, const BwdMaps& maps, cudaStream_t stream)
{
    const size_t smem = a.D == 128 ? BtMap<128>::kSmem : BtMap<64>::kSmem;
    bool first = true;                                                    // behind the preparation: an ordinary launch
    for (int summ = 1; summ >= 0; --summ) {
        if (summ && (a.m <= 0 || a.max_n_summ <= 0)) continue;
        const long long span = summ ? a.max_text_pad / 128 : bwd_text_span(a);
        // a unit walks seg query tiles x G heads: 16 tiles with four or more heads per KV head, more with fewer (the
        // final atomics of a unit are spread over about 64 streamed tiles either way)
        const int seg = bwd_seg_tiles(a);
        const int store = (!summ && bwd_text_keys_stored(a)) ? 1 : 0;
        const long long segs = (span + seg - 1) / seg, blocks = (summ ? a.summ_rows : a.text_rows) / 128 * segs;
        if (blocks > 0x7fffffffll) return cudaErrorInvalidConfiguration;
        const dim3 grid((unsigned)blocks, (unsigned)a.Hkv);
        auto* kernel = a.D == 128 ? ksa_bwd_dkv_tc_kernel<128> : ksa_bwd_dkv_tc_kernel<64>;
        cudaError_t e;
        if (first) {
            kernel<<<grid, kBwdTcThreads, smem, stream>>>(a, maps, summ, seg, (int)segs, store);
            e = cudaGetLastError();
        } else {
            e = launch_dependent(kernel, grid, kBwdTcThreads, smem, stream, a, maps, summ, seg, (int)segs, store);
        }
        if (e != cudaSuccess) return e;
        first = false;
    }
    return launch_dependent(a.D == 128 ? ksa_bwd_dq_tc_kernel<128> : ksa_bwd_dq_tc_kernel<64>,
                            dim3((unsigned)(a.text_rows / 128), (unsigned)a.Hq), kBwdTcThreads, smem, stream, a, maps);
}

}  // namespace ksa
