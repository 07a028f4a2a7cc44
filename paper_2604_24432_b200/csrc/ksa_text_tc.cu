// Text-row KSA attention on the sm_100a tensor cores.
//
// One persistent CTA per SM walks its share of the work list.  A work item is one tile of
// 128 text query rows for one or two query heads that share a KV head, plus the key/value
// tiles Eq. 3 makes visible to it: tiles of the packed summary stream first, then tiles of
// the packed text stream (the sliding-chunk band up to the diagonal).
//
// Warp roles (384 threads = three warpgroups):
//   warps 0-3   softmax of query tile 0 (one row per thread), O rescale, epilogue
//   warps 4-7   softmax of query tile 1
//   warp  8     TMA: Q tiles and K tiles (a ring of shared-memory stages)
//   warp  9     issues S = Q K^T (smem x smem, tcgen05.mma)
//   warp 10     issues O += P V (P from TMEM)
//   warp 11     TMA: V tiles (a ring of their own)
// TMEM (512 columns): one score slot S [0,128) that the two query tiles take in turns, the bf16
// probabilities P0 [128,192) and P1 [192,256), O0 [256,256+D), O1 [384,384+D).
//
// Pipeline per key/value tile j and query tile t:
//   warp 9:  once the slot is free (loaded[] of the scores before): S_t(j) = Q_t K(j)^T -> s_full[t]
//   softmax: load S_t into registers, hand the slot on                                  -> loaded[t]
//            mask (only on tiles flagged partial), running max with lazy rescale,
//            p = 2^(s*scale*log2e - m), row sum; wait for O_t += P_t V(j-1), rescale O_t
//            if the max moved, write P_t                                                -> p_full[t]
//   warp 10: O_t += P_t V(j)                                                            -> pv_done[t]
// A score row only has to stand in TMEM between its product and its load: the exponentials (most of a
// tile's time) work from registers.  So one slot serves both query tiles, and the scores of a query
// tile's next key tile are formed while its softmax still works on the one before: neither the
// products nor the two hand-overs stand between one softmax and the next.  (With a slot per query tile
// and P over it, every tile went through softmax, hand-over, 16 products, hand-over one after the other.)
// The two products have an issuing warp each, so that neither waits in the other's instruction stream:
// an issuing warp executes about one instruction in seven cycles beside the softmax warps, so the eight
// MMAs of a product take it as long to issue as the tensor pipe needs for them, and every barrier check
// on top left the pipe idle.  One sequence of 32,768 tokens, 32/8 heads, whole call: 1.532 ms with a slot per query
// tile, 1.477 ms with the shared slot and one issuing thread, 1.466 ms with a converged issuing warp, 1.328 ms with
// two.  131,072 tokens, 32/4 heads: 18.9 -> 16.6 ms a call (the clock falls from 1,700 to 1,430 MHz under the
// power limit as the pipes fill), 8,192 tokens: 258 -> 229 us.
// What bounds it now: the round trip of the score slot (product 560 cycles, hand-over 300, load 300 - 400, hand-over 100, for
// each query tile in turn) and the softmax warps' own loop (1,700 - 1,900 cycles of maximum and exponentials while the other
// group's run beside them, 300 for each hand-over).  A key tile and pair of query tiles takes 2,850 cycles.  One to three of
// eight exponential pairs as polynomials on the FMA pipe: 317 -> 319, 317, 343 thousand cycles (8,192 tokens, 32/8 heads), so
// the special-function unit is not what it waits for.  A work item's start and end cost 5,000 more: its entry and divisions
// (KV head and division by k come prepared: 325 -> 318), O's last product and the epilogue.  The epilogue in four warps of
// its own (208 / 48 registers) took 6,400 cycles a tile beside the softmax and held up the next item's first product: 353.
//
// Every mbarrier wait is bounded: on timeout the thread records which wait gave up in the
// status word, raises a CTA-wide abort flag, all roles leave their loops, the producer
// waits (bounded) for its copies in flight, TMEM is freed and the kernel returns.
#include <cuda_bf16.h>

#include "ksa_launch.h"
#include "ksa_ptx.cuh"
#include "ksa_wait.cuh"

namespace ksa {

using namespace ptx;

constexpr int kThreadsTc = 384;           // three warpgroups
constexpr int kRegsSoftmax = 216;         // registers per thread of the softmax warpgroups after the hand-over
constexpr int kRegsOther = 72;            // ... of the TMA / MMA warpgroup
// The CTA's register allocation is fixed at launch (65,536 / 384 threads = 170 -> 168 per thread): the softmax warps
// can only gain what the third warpgroup gives up; a larger setmaxnreg.inc would wait forever.
static_assert(8 * kRegsSoftmax + 4 * kRegsOther <= 12 * ((65536 / 384) / 8 * 8), "register hand-over exceeds the CTA's allocation");
constexpr int kLoadQkWarp = 8, kQkWarp = 9, kLoadVWarp = 11;         // (10: the PV products)
// log2 units: P stays below 2^12.  A small threshold costs rescales of O: with 1 % of the keys four times larger (the 128k
// workload) some row of nearly every warp outgrew 2^8 once or twice per work item.  Measured at 128k: 8 -> 1,032,
// 12 -> 1,047, 20 -> 1,058 TFLOP/s, but the error against the fp64 oracle grows with it (mean |err| 5.6e-4, 5.9e-4,
// 6.2e-4; at 20 one sampled element of the 64 + 8 layout left the 2e-2 bound), so 12 it is.
constexpr float kRescaleThreshold = 12.0f;

// barrier slots; then K full, K empty, V full, V empty per stage
enum : int { BAR_QFULL = 0, BAR_QEMPTY = 2, BAR_SFULL = 4, BAR_LOADED = 6, BAR_PFULL = 8, BAR_PVDONE = 10, BAR_DRAIN = 12, kBarKv = 14 };

template <int D>
struct TcCfg {
    static constexpr int kTileBytes = 128 * D * 2;
    static constexpr int kHalves = D / 64;                       // 64-column (128-byte) swizzle panels
    // Ring depths (tiles).  A K stage is taken up early (scores are formed a tile ahead), a V stage as its
    // probabilities are ready: with five stages beside the two Q tiles (all that fits at D = 128) K gets three.
    static constexpr int kStagesK = (D == 128) ? 3 : 5, kStagesV = (D == 128) ? 2 : 5;
    static constexpr int kQOff = 0;
    static constexpr int kKOff = 2 * kTileBytes;
    static constexpr int kVOff = kKOff + kStagesK * kTileBytes;
    static constexpr int kBarOff = kVOff + kStagesV * kTileBytes;
    static constexpr int kNumBars = kBarKv + 2 * (kStagesK + kStagesV);
    static constexpr int kSmemBytes = kBarOff + 8 * kNumBars + 64 + 1024;   // + slack for 1024-byte alignment
    // MN-major V operand: the two 64-column panels of a D = 128 tile are 16 KB apart,
    // groups of 8 keys are 1 KB apart.
    static constexpr uint32_t kVLbo = 16384;
    static constexpr uint32_t kVSbo = 1024;
};

template <int D>
__global__ void __launch_bounds__(kThreadsTc, 1)
ksa_text_tc_kernel(const __grid_constant__ KernelArgs a, const __grid_constant__ TextMaps maps)
{
    using Cfg = TcCfg<D>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sQ = smem_base + Cfg::kQOff;
    const uint32_t sK = smem_base + Cfg::kKOff, sV = smem_base + Cfg::kVOff;
    const uint32_t bars = smem_base + Cfg::kBarOff;
    const uint32_t tmem_slot = bars + 8 * Cfg::kNumBars;
    const uint32_t abort_addr = tmem_slot + 4;
    auto bar = [&](int i) -> uint32_t { return bars + 8u * (uint32_t)i; };
    auto k_full = [&](int st) -> uint32_t { return bar(kBarKv + st); };
    auto k_empty = [&](int st) -> uint32_t { return bar(kBarKv + Cfg::kStagesK + st); };
    auto v_full = [&](int st) -> uint32_t { return bar(kBarKv + 2 * Cfg::kStagesK + st); };
    auto v_empty = [&](int st) -> uint32_t { return bar(kBarKv + 2 * Cfg::kStagesK + Cfg::kStagesV + st); };

    const int tid = threadIdx.x;
    const int warp = (int)__reduce_or_sync(0xffffffffu, (unsigned)tid >> 5);     // (uniform to the compiler: 330 -> 325 thousand cycles)
    const int lane = tid & 31;

    if (tid == 0) {
        for (int t = 0; t < 2; ++t) {
            mbar_init(bar(BAR_QFULL + t), 1);
            mbar_init(bar(BAR_QEMPTY + t), 1);
            mbar_init(bar(BAR_SFULL + t), 1);
            mbar_init(bar(BAR_LOADED + t), 4);     // one arrival per softmax warp
            mbar_init(bar(BAR_PFULL + t), 4);
            mbar_init(bar(BAR_PVDONE + t), 1);
            mbar_init(bar(BAR_DRAIN + t), 1);
        }
        for (int st = 0; st < Cfg::kStagesK; ++st) { mbar_init(k_full(st), 1); mbar_init(k_empty(st), 1); }
        for (int st = 0; st < Cfg::kStagesV; ++st) { mbar_init(v_full(st), 1); mbar_init(v_empty(st), 1); }
        st_shared_u32(abort_addr, 0u);
        st_shared_u32(abort_addr + 4, 0u);     // never raised: lets the teardown waits run while aborting
        fence_mbar_init();
    }
    if (warp == kLoadQkWarp) {            // one warp allocates all 512 TMEM columns (1 CTA per SM)
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ld_shared_u32(tmem_slot);
    // Launched while the kernel in front (the pack) drains: nothing is read before it has finished.  From then on -- not
    // before: it does not wait for that kernel itself -- the summary rows' kernel behind may start as soon as every CTA is
    // resident; it takes the SMs that this kernel leaves.
    pdl_wait();
    pdl_launch_dependents();

    const int grid = (int)gridDim.x;
    const int cta = (int)blockIdx.x;
    // items are taken in snake order over the longest-first list: round r gives this CTA
    // item r*grid + cta (even r) or r*grid + grid-1-cta (odd r)
    auto item_index = [&](int r) -> int { return r * grid + ((r & 1) ? (grid - 1 - cta) : cta); };

    if (warp >= 8) {
        // register hand-over: this warpgroup gives most of its registers to the softmax warpgroups,
        // which keep a whole 128-column score row per thread
        setmaxnreg_dec<kRegsOther>();
        if (warp == kLoadQkWarp || warp == kLoadVWarp) {
            // =============================== TMA producers ===============================
            // warp 8: the Q tiles of an item and its K tiles; warp 11: its V tiles.  The two query heads of an item share
            // a KV head (one K and one V tile per key tile) or, where a pair straddles two KV heads (multi-head attention,
            // odd group sizes), each has its own: then a key tile takes two stages of each ring, head 0 first.
            if (lane == 0) {
                const bool is_v = warp == kLoadVWarp;
                const CUtensorMap* map_t = is_v ? &maps.vt : &maps.kt;
                const CUtensorMap* map_s = is_v ? &maps.vs : &maps.ks;
                const CUtensorMap* tail_t = is_v ? &maps.vt_tail : &maps.kt_tail;
                const CUtensorMap* tail_s = is_v ? &maps.vs_tail : &maps.ks_tail;
                const bool tails = a.direct == kReadTails;
                prefetch_tensormap(map_t); prefetch_tensormap(map_s);
                if (!is_v) prefetch_tensormap(&maps.qt);
                const int stages = is_v ? Cfg::kStagesV : Cfg::kStagesK;
                const uint32_t ring = is_v ? sV : sK, full0 = is_v ? v_full(0) : k_full(0), empty0 = is_v ? v_empty(0) : k_empty(0);
                uint32_t q_phase = 0, ring_phase = 0;        // q_phase: bit t for query tile t
                int stage = 0;
                uint32_t armed_mask = 0, armed_parity = 0;   // per stage: a load was issued / with which parity
                uint32_t q_armed = 0;                        // per query tile: a load was issued
                bool alive = true;
                for (int r = 0; alive; ++r) {
                    const int idx = item_index(r);
                    if (idx >= a.num_work) break;
                    const WorkItem w = a.work[idx];
                    const SeqInfo sq = a.seqs[w.seq];
                    const int hk = w.kv_head, nsplit = w.kv_per_tile;
                    const int T = w.ns_tiles + (w.band_hi - w.band_lo + 1);
                    const int start = tails ? row_in_chunk(sq, a.k, a.m) : 0;
                    // Half h of a tile: `tile` of the text (summary) rows of this sequence
                    auto load = [&](uint32_t dst, const CUtensorMap* map, const CUtensorMap* tail, uint32_t full, int h, bool summ, int tile, int head) {
                        const int per = kTileN / (summ ? max(a.m, 1) : a.k);                     // chunks of a tile
                        const int row = (summ ? sq.summ_off : sq.text_off) + tile * kTileN;
                        if (a.direct == kReadInPlace) tma_load_4d(dst, map, full, h * 64, 0, sq.chunk0 + tile * per, head);
                        else if (!tails) tma_load_3d(dst, map, full, h * 64, row, head);
                        else if ((tile + 1) * kTileN <= (summ ? sq.n_summ : sq.n_text)) tma_load_5d(dst, map, full, h * 64, 0, start, sq.chunk0 + tile * per, head);
                        else tma_load_3d(dst, tail, full, h * 64, row, head);
                    };
                    auto load_q = [&](int t) {
                        if (!bounded_wait(bar(BAR_QEMPTY + t), ((q_phase >> t) & 1u) ^ 1u, abort_addr, a.status, kStatusWaitQEmpty)) { alive = false; return; }
                        q_phase ^= 1u << t;
                        mbar_arrive_expect_tx(bar(BAR_QFULL + t), (uint32_t)Cfg::kTileBytes);
                        q_armed |= 1u << t;
                        for (int h = 0; h < Cfg::kHalves; ++h)
                            load(sQ + t * Cfg::kTileBytes + h * 16384, &maps.qt, &maps.qt_tail, bar(BAR_QFULL + t), h, false, w.q_tile, w.head0 + t);
                    };
                    if (!is_v) load_q(0);
                    for (int j = 0; j < T && alive; ++j) {
                        const bool summ = j < w.ns_tiles;
                        const int tile = summ ? j : w.band_lo + j - w.ns_tiles;
                        for (int u = 0; u < nsplit; ++u) {
                            if (!bounded_wait(empty0 + 8u * stage, ring_phase ^ 1u, abort_addr, a.status, kStatusWaitKvEmpty)) { alive = false; break; }
                            mbar_arrive_expect_tx(full0 + 8u * stage, (uint32_t)Cfg::kTileBytes);
                            armed_mask |= 1u << stage;
                            armed_parity = (armed_parity & ~(1u << stage)) | (ring_phase << stage);
                            for (int h = 0; h < Cfg::kHalves; ++h)
                                load(ring + stage * Cfg::kTileBytes + h * 16384, summ ? map_s : map_t, summ ? tail_s : tail_t, full0 + 8u * stage, h, summ, tile, hk + u);
                            if (++stage == stages) { stage = 0; ring_phase ^= 1u; }
                            if (j == 0 && u == 0 && !is_v && w.n_heads == 2) { load_q(1); if (!alive) break; }
                        }
                    }
                }
                if (ld_shared_u32(abort_addr) != 0u) {
                    // leave no copy in flight behind: wait (bounded) for every load that was issued
                    for (int t = 0; t < 2; ++t)
                        if (q_armed & (1u << t)) bounded_wait(bar(BAR_QFULL + t), ((q_phase >> t) & 1u) ^ 1u, abort_addr + 4, a.status, kStatusWaitQFull);
                    for (int st = 0; st < stages; ++st)
                        if (armed_mask & (1u << st))
                            bounded_wait(full0 + 8u * st, (armed_parity >> st) & 1u, abort_addr + 4, a.status, kStatusWaitKvFull);
                }
            }
        } else {
            // =============================== MMA issuers =================================
            // the whole warp walks the loop on warp-uniform values, one lane issues
            constexpr uint32_t hi = smem_desc_hi_sw128(1024);
            const uint32_t leader = elect_one();
            const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
            bool alive = true;
            auto wait = [&](uint32_t b, uint32_t parity, int code) {
                if (alive) alive = __all_sync(0xffffffffu, bounded_wait(b, parity, abort_addr, a.status, code));
            };
            uint32_t stage = 0, ring_phase = 0, phase0 = 0, phase1 = 0;
            if (warp == kQkWarp) {
                constexpr uint32_t idesc = make_idesc_bf16(128, 128, false);
                const uint32_t q_lo = smem_desc_lo(sQ, 16), k_lo = smem_desc_lo(sK, 16);
                uint32_t q_phase0 = 0, q_phase1 = 0;
                int before = -1;                            // query tile whose scores stand in the slot
                for (int r = 0; alive; ++r) {
                    const int idx = item_index(r);
                    if (idx >= a.num_work) break;
                    const WorkItem w = a.work[idx];
                    const int T = __shfl_sync(0xffffffffu, w.ns_tiles + (w.band_hi - w.band_lo + 1), 0);
                    const int nh = __shfl_sync(0xffffffffu, w.n_heads, 0);
                    const bool split = __shfl_sync(0xffffffffu, w.kv_per_tile, 0) == 2;
                    for (int j = 0; j < T && alive; ++j) {
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            if (t == 1 && nh == 1) break;
                            if (j == 0) {
                                wait(bar(BAR_QFULL + t), t ? q_phase1 : q_phase0, kStatusWaitQFull);
                                if (t) q_phase1 ^= 1u; else q_phase0 ^= 1u;
                            }
                            if (t == 0 || split) wait(k_full(0) + 8u * stage, ring_phase, kStatusWaitKvFull);
                            // the slot: the scores before are in their group's registers
                            if (before == 0) { wait(bar(BAR_LOADED), phase0, kStatusWaitPFull); phase0 ^= 1u; }
                            else if (before == 1) { wait(bar(BAR_LOADED + 1), phase1, kStatusWaitPFull); phase1 ^= 1u; }
                            if (!alive) break;
                            before = t;
                            tc_fence_after();
                            const uint32_t qd = q_lo + (uint32_t)(t * (Cfg::kTileBytes >> 4)), kd = k_lo + stage * (uint32_t)(Cfg::kTileBytes >> 4);
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk) {
                                const uint32_t off = (uint32_t)((kk >> 2) * 16384 + (kk & 3) * 32) >> 4;
                                mma_ss_warp(leader, tm, qd + off, kd + off, hi, idesc, kk > 0 ? 1u : 0u);
                            }
                            tc_commit_warp(leader, bar(BAR_SFULL + t));
                            if ((t == nh - 1 || split) && ++stage == (uint32_t)Cfg::kStagesK) { stage = 0; ring_phase ^= 1u; }
                        }
                    }
                }
            } else {
                constexpr uint32_t idesc = make_idesc_bf16(128, D, true);
                const uint32_t v_lo = smem_desc_lo(sV, Cfg::kVLbo);
                for (int r = 0; alive; ++r) {
                    const int idx = item_index(r);
                    if (idx >= a.num_work) break;
                    const WorkItem w = a.work[idx];
                    const int T = __shfl_sync(0xffffffffu, w.ns_tiles + (w.band_hi - w.band_lo + 1), 0);
                    const int nh = __shfl_sync(0xffffffffu, w.n_heads, 0);
                    const bool split = __shfl_sync(0xffffffffu, w.kv_per_tile, 0) == 2;
                    for (int j = 0; j < T && alive; ++j) {
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            if (t == 1 && nh == 1) break;
                            if (t == 0 || split) wait(v_full(0) + 8u * stage, ring_phase, kStatusWaitKvFull);
                            wait(bar(BAR_PFULL + t), t ? phase1 : phase0, kStatusWaitPFull);
                            if (t) phase1 ^= 1u; else phase0 ^= 1u;
                            if (!alive) break;
                            tc_fence_after();
                            const uint32_t vd = v_lo + stage * (uint32_t)(Cfg::kTileBytes >> 4);
#pragma unroll
                            for (int kk = 0; kk < kTileN / 16; ++kk)
                                mma_ts_warp(leader, tm + 256u + t * 128u, tm + 128u + t * 64u + kk * 8u, vd + (uint32_t)((kk * 2048) >> 4), hi, idesc,
                                            (j > 0 || kk > 0) ? 1u : 0u);
                            tc_commit_warp(leader, bar(BAR_PVDONE + t));
                            if ((t == nh - 1 || split) && ++stage == (uint32_t)Cfg::kStagesV) { stage = 0; ring_phase ^= 1u; }
                        }
                    }
                }
            }
            // drain the tensor pipe before TMEM is released
            const uint32_t drain = bar(BAR_DRAIN + (warp == kQkWarp ? 0 : 1));
            tc_commit_warp(leader, drain);
            bounded_wait(drain, 0, abort_addr + 4, a.status, kStatusWaitOFull);
        }
    } else {
        setmaxnreg_inc<kRegsSoftmax>();
        // =============================== softmax warpgroups =========================
        const int t = warp >> 2;
        const int row = tid & 127;
        const uint32_t lane_sel = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_sel;                                   // the score slot
        const uint32_t tP = tmem + lane_sel + 128u + (uint32_t)(t * 64);
        const uint32_t tO = tmem + lane_sel + 256u + (uint32_t)(t * 128);
        const float scale_log2 = a.scale_log2;
        uint32_t sf_phase = 0, pv_phase = 0;
        const int s_len = a.k + a.m;
        bool alive = true;
        // Shared-memory stages are handed back to the producers by the first thread of a warpgroup: of the item's LAST
        // query tile where both share the K / V tiles (the products of an issuing warp complete in order, so its s_full
        // for key tile j says that both have read K(j), its pv_done that both have read V(j)), of each query tile for
        // its own stages where the pair straddles two KV heads.
        int k_base = 0, v_base = 0;                        // ring stages of the item's first tiles
        for (int r = 0; alive; ++r) {
            const int idx = item_index(r);
            if (idx >= a.num_work) break;
            const WorkItem w = a.work[idx];
            const int nsplit = w.kv_per_tile;                // ring stages per K / V tile
            // the next stage this thread hands back, and how far on the one after it stands
            int rel_k = (k_base + (nsplit - 1) * t) % Cfg::kStagesK, rel_v = (v_base + (nsplit - 1) * t) % Cfg::kStagesV;
            k_base = (k_base + nsplit * (w.ns_tiles + (w.band_hi - w.band_lo + 1))) % Cfg::kStagesK;
            v_base = (v_base + nsplit * (w.ns_tiles + (w.band_hi - w.band_lo + 1))) % Cfg::kStagesV;
            if (t >= w.n_heads) continue;
            const bool first_thread = (tid & 127) == 0;
            const bool releaser = first_thread && (nsplit == 2 || t == w.n_heads - 1);
            auto release_k = [&]() {
                mbar_arrive_relaxed(k_empty(rel_k));
                if ((rel_k += nsplit) >= Cfg::kStagesK) rel_k -= Cfg::kStagesK;
            };
            auto release_v = [&]() {
                mbar_arrive_relaxed(v_empty(rel_v));
                if ((rel_v += nsplit) >= Cfg::kStagesV) rel_v -= Cfg::kStagesV;
            };
            const SeqInfo sq = a.seqs[w.seq];
            const int T = w.ns_tiles + (w.band_hi - w.band_lo + 1);
            const int i_raw = w.q_tile * kTileM + row;
            const bool valid = i_raw < sq.n_text;
            const int i = valid ? i_raw : sq.n_text - 1;     // padding rows mimic the last row; never stored
            const int chunk = a.k_inverse ? (int)__umul64hi((unsigned long long)i, a.k_inverse) : i;      // i / k
            const int far = max(0, chunk - a.C);
            const int lo_i = far * a.k;                      // Eq. 3: first visible text token
            const int cnt_i = far * a.m;                     // Eq. 3: summaries [0, cnt_i) visible
            float m_used = -INFINITY, l_run = 0.f;

            // Both barriers of a tile are asked for ahead of their waits: a passed wait costs some 300 cycles beside the other
            // group's exponentials (8,192 tokens, 32/8 heads: 317 -> 312 thousand cycles; 32,413 ragged tokens 1,304 -> 1,287).
            bool s_ok = false;                               // the scores of this tile are known to be there
            for (int j = 0; j < T; ++j) {
                bool ok;
                if (!__all_sync(0xffffffffu, s_ok)) {
                    ok = bounded_wait(bar(BAR_SFULL + t), sf_phase, abort_addr, a.status, kStatusWaitSFull);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) { alive = false; break; }
                }
                sf_phase ^= 1u;
                tc_fence_after();
                uint32_t s[128];
                {
                    uint32_t (&c0)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[0]);
                    uint32_t (&c1)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[32]);
                    uint32_t (&c2)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[64]);
                    uint32_t (&c3)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[96]);
                    tmem_ld32(tS + 0, c0); tmem_ld32(tS + 32, c1); tmem_ld32(tS + 64, c2); tmem_ld32(tS + 96, c3);
                }
                // the stage hand-backs ride on the latency of the loads
                if (releaser) release_k();                   // K(j)
                if (first_thread && j == T - 1) mbar_arrive_relaxed(bar(BAR_QEMPTY + t));
                tc_wait_ld();
                // the scores are in registers: the slot may take the next ones
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_relaxed(bar(BAR_LOADED + t));
                // in-tile mask, only where the schedule says the tile is partial
                bool masked;
                int ca, cb;                                   // visible columns [ca, cb)
                if (j < w.ns_tiles) {
                    masked = j >= w.ns_nomask;
                    ca = 0; cb = cnt_i - j * kTileN;
                } else {
                    const int bt = w.band_lo + (j - w.ns_tiles);
                    masked = !(bt >= w.band_nomask_lo && bt < w.band_nomask_hi);
                    ca = lo_i - bt * kTileN; cb = i + 1 - bt * kTileN;
                }
                if (masked) {
                    const uint32_t width = (uint32_t)max(cb - ca, 0);
#pragma unroll
                    for (int c = 0; c < 128; ++c)
                        if ((uint32_t)(c - ca) >= width) s[c] = 0xff800000u;   // -inf
                }
                // row maximum, two new scores per instruction
                float mx0 = fmax3(__uint_as_float(s[0]), __uint_as_float(s[1]), __uint_as_float(s[2]));
                float mx1 = fmax3(__uint_as_float(s[3]), __uint_as_float(s[4]), __uint_as_float(s[5]));
                float mx2 = fmax3(__uint_as_float(s[6]), __uint_as_float(s[7]), __uint_as_float(s[8]));
                float mx3 = fmax3(__uint_as_float(s[9]), __uint_as_float(s[10]), __uint_as_float(s[11]));
#pragma unroll
                for (int c = 12; c < 124; c += 8) {
                    mx0 = fmax3(mx0, __uint_as_float(s[c]), __uint_as_float(s[c + 1]));
                    mx1 = fmax3(mx1, __uint_as_float(s[c + 2]), __uint_as_float(s[c + 3]));
                    mx2 = fmax3(mx2, __uint_as_float(s[c + 4]), __uint_as_float(s[c + 5]));
                    mx3 = fmax3(mx3, __uint_as_float(s[c + 6]), __uint_as_float(s[c + 7]));
                }
                mx0 = fmax3(mx0, __uint_as_float(s[124]), __uint_as_float(s[125]));
                mx1 = fmax3(mx1, __uint_as_float(s[126]), __uint_as_float(s[127]));
                const float mx_sc = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * scale_log2;
                // lazy rescale: the reference max only moves when some row of the warp outgrew it
                const bool need = mx_sc > m_used + kRescaleThreshold;
                const bool need_any = __any_sync(0xffffffffu, need);
                float alpha = 1.f;
                if (need_any) {
                    const float m_new = fmaxf(m_used, mx_sc);
                    alpha = (m_new == -INFINITY) ? 1.f : ex2_approx(m_used - m_new);
                    m_used = m_new;
                    l_run *= alpha;
                }
                const float neg_m = (m_used == -INFINITY) ? 0.f : -m_used;
                const float2 sc2 = make_float2(scale_log2, scale_log2);
                const float2 nm2 = make_float2(neg_m, neg_m);
                bool pv_ok = false;                           // the product before is known to be done
                float2 la = make_float2(0.f, 0.f), lb = make_float2(0.f, 0.f);
                // probabilities of the column pair (2q, 2q+1), packed into s[q]; the scale-and-shift
                // and the row sum work on packed pairs (half the FMA-pipe instructions)
#pragma unroll
                for (int q = 0; q < 64; ++q) {
                    const float2 x = ffma2(make_float2(__uint_as_float(s[2 * q]), __uint_as_float(s[2 * q + 1])), sc2, nm2);
                    float2 pr;
                    pr.x = ex2_approx(x.x); pr.y = ex2_approx(x.y);
                    if (q & 1) lb = fadd2(lb, pr); else la = fadd2(la, pr);
                    if (q == 48 && j > 0) pv_ok = mbar_test_wait(bar(BAR_PVDONE + t), pv_phase);
                    s[q] = pack_bf16x2(pr.x, pr.y);
                }
                l_run += (la.x + la.y) + (lb.x + lb.y);
                if (j > 0) {
                    // O_t += P_t V(j-1) has read P_t and written O_t
                    if (!__all_sync(0xffffffffu, pv_ok)) {
                        ok = bounded_wait(bar(BAR_PVDONE + t), pv_phase, abort_addr, a.status, kStatusWaitPvDone);
                        ok = __all_sync(0xffffffffu, ok);
                        if (!ok) { alive = false; break; }
                    }
                    pv_phase ^= 1u;
                    if (releaser) release_v();               // V(j-1)
                    tc_fence_after();
                }
                s_ok = j + 1 < T && mbar_test_wait(bar(BAR_SFULL + t), sf_phase);
                {
                    uint32_t (&p0)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[0]);
                    uint32_t (&p1)[32] = *reinterpret_cast<uint32_t (*)[32]>(&s[32]);
                    tmem_st32(tP + 0, p0); tmem_st32(tP + 32, p1);
                }
                if (need_any && j > 0) {
#pragma unroll
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t o[32];
                        tmem_ld32(tO + c * 32, o);
                        tc_wait_ld();
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                        tmem_st32(tO + c * 32, o);
                    }
                }
                tc_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_relaxed(bar(BAR_PFULL + t));
            }
            if (!alive) break;
            // ---- epilogue: O / l -> bf16 at the row's augmented position (Eq. 1), LSE ----
            bool ok = bounded_wait(bar(BAR_PVDONE + t), pv_phase, abort_addr, a.status, kStatusWaitOFull);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            pv_phase ^= 1u;
            if (releaser) release_v();                       // V(T-1)
            tc_fence_after();
            const float inv_l = 1.f / l_run;
            const int h = w.head0 + t;
            const int64_t aug = sq.aug_off + (int64_t)chunk * s_len + (i - chunk * a.k);
            const bool store = valid && ksa_out_row_ok(a, aug, h);
            // a row stands in one lane: four lanes exchange 64 bytes of their rows, so that a store touches 8 lines, not 32
            // (the epilogues took 246 of 3,207 cycles a key tile at 32,768 tokens: the store path takes a line per cycle)
            const int64_t off = store ? aug * a.o_st + (int64_t)h * a.o_sh : -1;
#pragma unroll
            for (int c = 0; c < D / 32; ++c) {
                uint32_t o[32];
                tmem_ld32(tO + c * 32, o);
                tc_wait_ld();
                uint4 pk[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    pk[e].x = pack_bf16x2(__uint_as_float(o[8 * e]) * inv_l, __uint_as_float(o[8 * e + 1]) * inv_l);
                    pk[e].y = pack_bf16x2(__uint_as_float(o[8 * e + 2]) * inv_l, __uint_as_float(o[8 * e + 3]) * inv_l);
                    pk[e].z = pack_bf16x2(__uint_as_float(o[8 * e + 4]) * inv_l, __uint_as_float(o[8 * e + 5]) * inv_l);
                    pk[e].w = pack_bf16x2(__uint_as_float(o[8 * e + 6]) * inv_l, __uint_as_float(o[8 * e + 7]) * inv_l);
                }
                quad_transpose(pk, lane);                             // pk[e]: 16 bytes of the group's row e
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int64_t at = __shfl_sync(0xffffffffu, off, (lane & 28) + e);
                    if (at >= 0) *reinterpret_cast<uint4*>(a.out + at + c * 32 + (lane & 3) * 8) = pk[e];
                }
            }
            if (store) a.lse[(int64_t)h * a.total_aug + aug] = (m_used + log2f(l_run)) * 0.6931471805599453f;
            tc_fence_before();
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == kLoadQkWarp) tmem_dealloc(tmem, 512);
}

cudaError_t setup_text_tc()
{
    cudaError_t e = cudaFuncSetAttribute(ksa_text_tc_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         TcCfg<128>::kSmemBytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(ksa_text_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                TcCfg<64>::kSmemBytes);
}

cudaError_t launch_text_tc(const KernelArgs& a, const TextMaps& maps, int num_sms, cudaStream_t stream)
{
    if (a.num_work <= 0) return cudaSuccess;
    const int grid = a.num_work < num_sms ? a.num_work : num_sms;
    KernelArgs ka = a;
    // exact for the rows of a sequence: the product is off by less than i / 2^64, and i / k by 1 / k or more from the next integer
    ka.k_inverse = a.k > 1 ? ~0ull / (uint64_t)a.k + 1 : 0;
    return a.D == 128 ? launch_dependent(ksa_text_tc_kernel<128>, dim3((unsigned)grid), kThreadsTc, TcCfg<128>::kSmemBytes, stream, ka, maps)
                      : launch_dependent(ksa_text_tc_kernel<64>, dim3((unsigned)grid), kThreadsTc, TcCfg<64>::kSmemBytes, stream, ka, maps);
}

}  // namespace ksa
