// Second kernel of the grouped INT4 formats for calls with few token rows: w4a4_gemm.cu's computation (same formats, same exact group
// sums, same order of additions, same bits) in tiles of 128 rows x 64 columns, or 32 with groups of 64.
//
// With few tiles a tile's k-blocks are a chain of hand-overs between the tensor core and the epilogue, so the call takes as
// long as the chain: more, narrower tiles on more SMs, and a short chain.  A tensor-memory buffer holds the accumulator tiles
// of ALL groups of a k-block of 128 codes, so there is one hand-over per k-block where w4a4_gemm.cu has one per group; the
// two unpack warps take k-blocks in turn (half of a turn is waiting); the epilogue asks for a unit's scales with the unit.
// With groups of 64 a k-block takes 590 cycles: the expansion, the MMA warp's chain of waits, MMAs and commits and the epilogue's chain per
// buffer are each busy for 80 to 95 % of them.  It took 780 with barriers and tests of their own for the scales (now they land with the operands),
// the next buffer's first unit requested at one of two places, and addresses that were not known to be uniform, and 1060 with one hand-over
// per group: us alone, 256 x 1152 -> 1152 7.0 -> 6.0, 16 x 12288 -> 3072 41.0 -> 29.8, 64 x 3072 -> 9216 13.3 -> 10.4.  Tried: a whole buffer
// per tensor-memory wait 0 to 6 % slower, three expanding warps in a block of 16 warps 4 to 13 %.
// 32-column tiles halve the expansion and the epilogue of a k-block and leave the MMA warp's chain: second kernel 256 x 1152 -> 1152 6.2 -> 5.7 us, 16 x 3072 ->
// 3072 9.4 -> 8.4, 16 x 12288 -> 3072 28.5 -> 24.5.  Only where they keep at most half of the SMs busy: 512 x 1152 -> 1152, 144 tiles, gains 0.4 us alone and loses
// as much behind the rotation, whose 72 CTAs leave it no room to start early.
//
// Roles (384 threads = 3 warpgroups):
//   warpgroup 0: warp 0 TMA producer, warp 1 MMA issuer + TMEM owner, warps 2-3 nibble -> byte unpack (k-blocks in turn)
//   warpgroups 1-2: epilogue; warp%4 selects the TMEM lane quadrant (token rows), the warpgroup
//                   selects the half of the tile's columns.
//
// SPLITK: clusters of up to four CTAs cut the K-groups of one tile into contiguous ranges; each CTA rescales its
// range into its own fp32 accumulators, the others store theirs into the last CTA's shared memory (distributed shared
// memory), and that CTA adds them in rank order, adds the rank-r branch and the bias, and stores.
#include "w4a4.cuh"

#include <atomic>

namespace dirotq {
namespace {

constexpr int SPLIT_MAX = 4;          // CTAs per cluster of the split plan
constexpr int NUM_EPI_WARPS = 8, NUM_THREADS = 384;
constexpr int EPI_REGS = 224, AUX_REGS = 56;  // setmaxnreg budgets: 256 x EPI + 128 x AUX <= 384 x 168
constexpr int RED_BYTES = 128 * 64 * 4;  // one CTA's partial tile: 128 rows x 64 columns fp32
constexpr int SC_SLOTS = 11;          // scale records, one per k-block
template <bool SPLITK, int BN>
struct Plan {
    static constexpr int BU_BYTES = BN * BKC;         // unpacked weight codes / bf16 W~_h chunk
    static constexpr int BP_BYTES = BN * BKC / 2;     // packed weight codes (TMA staging)
    static constexpr int STAGE_BYTES = A_BYTES + BU_BYTES + BP_BYTES;  // 28 KB, or 22
    static constexpr int SC_SW_BYTES = 2 * BN * 4;    // up to two groups per k-block
    static constexpr int SC_SX_BYTES = 2 * BM * 4;    // activation scales of up to two groups
    static constexpr int SC_BYTES = SC_SW_BYTES + SC_SX_BYTES;
    static constexpr int STAGES = SPLITK ? 4 : 6;
    // (Even: then an unpack warp, which takes every second k-block, has itself seen the previous one of a stage land, and cannot take that
    // one's missing phase for its own: a barrier is waited on by parity.)
    static_assert(STAGES % 2 == 0, "see above");
    static constexpr int BAR_OFFSET = STAGES * STAGE_BYTES + SC_SLOTS * SC_BYTES;
    static constexpr int RED_OFFSET = BAR_OFFSET + 512;  // split plan: the other CTAs' partial tiles land here (last CTA)
    static constexpr int SMEM_BYTES = BAR_OFFSET + 512 + 1024 + (SPLITK ? (SPLIT_MAX - 1) * RED_BYTES : 0);
    static_assert(SMEM_BYTES <= 232448 && STAGE_BYTES % 1024 == 0 && SC_BYTES % 128 == 0, "shared memory plan");
    static_assert(8 * (4 * STAGES + 11) <= 400, "barriers end below the words at +400");
    // A k-block's scales land with its operands, on the same barrier, in a ring of their own that has no "empty" barriers: the producer
    // loads k-block j when the MMAs of j - STAGES are done, those had waited until the epilogue was through with the buffer four before.
    static_assert(SC_SLOTS >= STAGES + 5, "scale records");
};

template <int G, bool SPLITK, int BN>
__global__ void __launch_bounds__(NUM_THREADS, 1)
w4a4_narrow_kernel(const __grid_constant__ CUtensorMap tmap_codes, const __grid_constant__ CUtensorMap tmap_wpacked,
                 const __grid_constant__ CUtensorMap tmap_wscale, const __grid_constant__ CUtensorMap tmap_xscale,
                 const __grid_constant__ CUtensorMap tmap_xh, const __grid_constant__ CUtensorMap tmap_wh,
                 const GemmKernelParams p) {
    using P = Plan<SPLITK, BN>;
    static_assert(BN == 64 || (BN == 32 && G == 64 && !SPLITK), "32-column tiles: groups of 64, not split");
    constexpr int STAGES = P::STAGES, BAR_OFFSET = P::BAR_OFFSET, STAGE_BYTES = P::STAGE_BYTES, BU_BYTES = P::BU_BYTES, BP_BYTES = P::BP_BYTES;
    constexpr int SC_SW_BYTES = P::SC_SW_BYTES, SC_BYTES = P::SC_BYTES;
    constexpr int HB = BN / 2;         // columns per epilogue warp: the warpgroup selects the half of the tile
    constexpr int GPK = BKC / G;       // groups per k-block: 2 (G = 64) or 1 (G = 128)
    constexpr int MMA_PER_G = G / 32;  // 8-bit MMA instructions (K = 32) per group
    constexpr int BUF_COLS = GPK * BN;  // a tensor-memory buffer: the accumulator tiles of a k-block's groups
    constexpr int NBUF = 4;             // (the barrier map has four slots)
    // The epilogue works through a buffer in two units per warp: its 32 columns of the two groups, or two halves of them.
    constexpr int UC = GPK * HB / 2, NU = 2, UPG = NU / GPK;  // columns per unit, units per buffer, per group

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sc_base = smem_base + STAGES * STAGE_BYTES;
    const uint32_t bar_base = smem_base + BAR_OFFSET;
    // barriers: full[S], unpacked[S], empty[S], tmem_full[NBUF], tmem_empty[NBUF], spare, split plan's two
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto unp_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
    auto empty_bar = [&](int s) { return bar_base + 8u * (2 * STAGES + s); };
    auto tfull_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + a); };
    auto tempty_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + 4 + a); };
    auto pre_bar = [&](int s) { return bar_base + 8u * (3 * STAGES + 11 + s); };  // see early_weights below
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + BAR_OFFSET + 400);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + BAR_OFFSET + 404);

    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);  // (known to be uniform)
    const int lane = threadIdx.x & 31;
    // Trace build (TRACE_CLK): slot 9 entry, 10 set-up done, 11 previous grid ended, 12 / 13 producer has issued its first k-block /
    // everything, 14 / 15 first unpack warp sees / has expanded the first stage, 16 / 17 / 18 MMA warp starts the first / fifth / last
    // k-block, 19 it has committed the last tile, 20 first epilogue warp sees its first accumulator, 21 starts its ninth K-group, 22 has
    // folded in the last group, 23 the rank-r tile, 24 has stored its last outputs.
    if (threadIdx.x == 0) TRACE_CLK(p.status, 9);

    const int num_m_blocks = (p.M + BM - 1) / BM;
    const int num_n_blocks = (p.N + BN - 1) / BN;
    const int num_tiles = num_m_blocks * num_n_blocks;
    // Split plan: this CTA's range of k-blocks [kb0, kb1) of the cluster's tile (the first ranks take
    // one k-block more when the division leaves a rest); the LAST rank gathers the partial tiles and has the rank-r branch.
    // (Without the split every one of these is the constant or the parameter it stands for.)
    const uint32_t csize = SPLITK ? cluster_nctarank() : 1u, crank = SPLITK ? cluster_ctarank() : 0u;
    const bool gathers = !SPLITK || crank == csize - 1;
    const int split_base = SPLITK ? p.num_kb / static_cast<int>(csize) : 0, split_rest = SPLITK ? p.num_kb % static_cast<int>(csize) : 0;
    const int kb0 = SPLITK ? static_cast<int>(crank) * split_base + min(static_cast<int>(crank), split_rest) : 0;
    const int kb1 = SPLITK ? kb0 + split_base + (static_cast<int>(crank) < split_rest ? 1 : 0) : p.num_kb;
    const int lr_here = gathers ? p.lr_chunks : 0;
    // (tile loops read these where they are needed, like blockIdx.x and gridDim.x themselves, not held in registers across the
    // roles' loops)
    auto first_tile = [&]() { return SPLITK ? static_cast<int>(blockIdx.x / csize) : static_cast<int>(blockIdx.x); };
    auto tile_stride = [&]() { return SPLITK ? static_cast<int>(gridDim.x / csize) : static_cast<int>(gridDim.x); };
    const uint32_t red_bar = bar_base + 8u * (3 * STAGES + 9);  // split plan: "partial tiles landed" (last CTA)

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(unp_bar(s), 32);  // every thread of the unpack warp whose turn it is arrives for itself
            mbar_init(empty_bar(s), 1);
            mbar_init(pre_bar(s), 1);
        }
        for (int a = 0; a < NBUF; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), NUM_EPI_WARPS * 32);
        }
        mbar_init(bar_base + 8u * (3 * STAGES + 8), 1);  // spare: see umma_drain
        if constexpr (SPLITK) {
            mbar_init(red_bar, 1);  // counts the bytes of the other CTAs' partial tiles
            mbar_init(red_bar + 8u, NUM_EPI_WARPS * 32);  // this CTA's partial tile is in its shared memory (every epilogue thread arrives)
            if (gathers) mbar_arrive_expect_tx(red_bar, (csize - 1) * RED_BYTES);
        }
        *abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmap_codes);
        tma_prefetch_desc(&tmap_wpacked);
        tma_prefetch_desc(&tmap_wscale);
        tma_prefetch_desc(&tmap_xscale);
        tma_prefetch_desc(&tmap_xh);
        tma_prefetch_desc(&tmap_wh);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    if constexpr (SPLITK) cluster_sync_all();  // the gathering CTA's barrier is initialised before anything arrives on it
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // everything above touched only this CTA's own shared and tensor memory; what follows reads the first kernel's output
    if (threadIdx.x == 0) TRACE_CLK(p.status, 10);
    // Weights and their scales may be loaded, and expanded, while the previous kernel is still running (GemmArgs::early_weights): those of the
    // first tile's first stages land on barriers of their own, the stage's barrier then counts the activations only.
    const int pre = p.early_weights && first_tile() < num_tiles ? min(STAGES, kb1 - kb0) : 0;
    if (warp == 0 && pre > 0 && elect_one()) {
        const int n0 = (first_tile() / num_m_blocks) * BN;
        for (int j = 0; j < pre; ++j) {
            mbar_arrive_expect_tx(pre_bar(j), BP_BYTES + GPK * BN * 4);
            tma_load_2d(smem_base + j * STAGE_BYTES + A_BYTES + BU_BYTES, &tmap_wpacked, pre_bar(j), (kb0 + j) * (BKC / 2), n0);
            tma_load_2d(sc_base + j * SC_BYTES, &tmap_wscale, pre_bar(j), n0, (kb0 + j) * GPK);
        }
    }
    __syncwarp();
    if (pre == 0 || (warp != 2 && warp != 3)) {  // (otherwise the unpack warps wait when they are through with the early weights)
        grid_dependency_wait();
        if (threadIdx.x == 0) TRACE_CLK(p.status, 11);
        // the next layer's first kernel may be scheduled as this grid's CTAs leave their SMs (it waits for this whole grid)
        grid_launch_dependents();
    }

    if (warp < 4) {
        reg_dealloc<AUX_REGS>();

        if (warp == 0) {
            // -------------------------------------------------------- TMA producer
            // (the whole warp walks the loops and waits, one elected lane issues: counters, addresses and coordinates stay
            // warp-uniform, which shortens the chain of instructions per stage)
            {
                RingPos<STAGES> at;
                uint32_t slot = 0;
                long long w_empty = 0;
                bool ok = true;
                for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                    const int m0 = (tile % num_m_blocks) * BM;
                    const int n0 = (tile / num_m_blocks) * BN;
                    for (int kb = kb0; kb < kb1; ++kb, at.next()) {
                        const uint32_t s = at.s;
                        if (!timed_wait(empty_bar(s), at.ph ^ 1, abort_flag, p.status, DEV_TIMEOUT_PRODUCER, w_empty)) { ok = false; break; }
                        const uint32_t st = smem_base + s * STAGE_BYTES;
                        if (elect_one()) {
                            const uint32_t sc = sc_base + slot * SC_BYTES;
                            const bool weights = at.it >= static_cast<uint32_t>(pre);
                            mbar_arrive_expect_tx(full_bar(s), p.x_rows * BKC + GPK * BM * 4 + (weights ? BP_BYTES + GPK * BN * 4 : 0));
                            tma_load_2d(st, &tmap_codes, full_bar(s), kb * BKC, m0);
                            if (weights) {
                                tma_load_2d(st + A_BYTES + BU_BYTES, &tmap_wpacked, full_bar(s), kb * (BKC / 2), n0);
                                tma_load_2d(sc, &tmap_wscale, full_bar(s), n0, kb * GPK);
                            }
                            tma_load_2d(sc + SC_SW_BYTES, &tmap_xscale, full_bar(s), m0, kb * GPK);
                            if (at.it == 0) TRACE_CLK(p.status, 12);
                        }
                        if (++slot == SC_SLOTS) slot = 0;
                    }
                    if (!ok) break;
                    for (int lr = 0; lr < lr_here; ++lr, at.next()) {
                        const uint32_t s = at.s;
                        if (!mbar_wait(empty_bar(s), at.ph ^ 1, abort_flag, p.status, DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
                        const uint32_t st = smem_base + s * STAGE_BYTES;
                        if (elect_one()) {
                            mbar_arrive_expect_tx(full_bar(s), p.x_rows * BKC + BU_BYTES);
                            tma_load_2d(st, &tmap_xh, full_bar(s), lr * 64, m0);
                            tma_load_2d(st + A_BYTES, &tmap_wh, full_bar(s), lr * 64, n0);
                        }
                    }
                }
                if (lane == 0) TRACE_CLK(p.status, 13);
                if (lane == 0) flush_wait(p.status, WS_PROD_EMPTY, w_empty);
                if (!ok && lane == 0) {
                    const uint32_t first = at.it > STAGES ? at.it - STAGES : 0;
                    for (uint32_t j = first; j < at.it; ++j) {
                        const unsigned long long t0 = globaltimer_ns();
                        while (!mbar_try_wait(full_bar(j % STAGES), (j / STAGES) & 1) &&
                               globaltimer_ns() - t0 < 100000000ull) {}
                    }
                }
            }
        } else if (warp == 1) {
            // -------------------------------------------------------- MMA issuer
            // One thread, and every instruction it executes waits its turn behind the two epilogue warps of its
            // scheduler, so its loop is kept short: stage index, parities and the operand descriptors are carried
            // along instead of recomputed (a descriptor differs between stages only in the address field of its low
            // word, which cannot overflow: shared-memory addresses have 18 bits, the field holds address / 16).
            // (whole warp in the loops, one elected lane issues, as in the producer)
            {
                constexpr uint32_t idesc_f8 = umma_idesc(1 /*f32*/, 0 /*E4M3*/, BM, BN);
                constexpr uint32_t idesc_i8 = umma_idesc(2 /*s32*/, 1 /*s8*/, BM, BN);  // integer-path build only
                constexpr uint32_t idesc_bf = umma_idesc(1 /*f32*/, 1 /*bf16*/, BM, BN);
                const uint64_t desc0 = umma_desc_sw128(smem_base);
                const uint32_t desc_hi = static_cast<uint32_t>(desc0 >> 32), desc_lo0 = static_cast<uint32_t>(desc0);
                auto desc = [&](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
                uint32_t s = 0, ph = 0;        // stage of the operand ring and its parity
                uint32_t b = 0, bph = 1;       // accumulator tile and the parity its "empty" barrier is waited with
                int pre_left = pre;
                long long w_ops = 0, w_tempty = 0;
                const long long t_kernel = clock64();
                bool ok = true;
                for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                    for (int kb = kb0; ok && kb < kb1; ++kb) {
                        // the unpack warps arrive after they have seen the stage's loads land (one barrier for both operands), so
                        // their barrier covers the activation codes as well
                        if (!timed_wait(unp_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_ops)) { ok = false; break; }
                        if (pre_left > 0) {  // (these were expanded before their activations had been asked for)
                            --pre_left;
                            // (timed in the diagnostic build: the clock reads cost a short call up to 2 %, 1500 x 512 -> 512 10.05 -> 10.28 us)
                            if (!(kTraceBuild ? timed_wait(full_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_ops)
                                              : mbar_wait(full_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA))) { ok = false; break; }
                        }
                        if (lane == 0) { if (kb == kb0) TRACE_CLK(p.status, 16); if (kb == 4) TRACE_CLK(p.status, 17); if (kb == kb1 - 1) TRACE_CLK(p.status, 18); }
                        if (!timed_wait(tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_tempty)) { ok = false; break; }
                        tc_fence_after_sync();
                        if (elect_one()) {
                            const uint32_t a_lo = desc_lo0 + s * (STAGE_BYTES >> 4), b_lo = a_lo + (A_BYTES >> 4), d = tmem_base + b * BUF_COLS;
#pragma unroll
                            for (int kk = 0; kk < 4; ++kk) {  // 32-byte step inside the 128-byte row
                                const int gi = kk / MMA_PER_G, k = kk % MMA_PER_G;
                                // (an odd number of groups: the last k-block's second one is zeros, codes and scales)
                                if constexpr (kI8Path)
                                    umma_i8(d + gi * BN, desc(a_lo + 2 * kk), desc(b_lo + 2 * kk), idesc_i8, k != 0);
                                else
                                    umma_f8f6f4(d + gi * BN, desc(a_lo + 2 * kk), desc(b_lo + 2 * kk), idesc_f8, k != 0);
                            }
                            umma_commit(tfull_bar(b));
                            umma_commit(empty_bar(s));
                        }
                        if (++b == NBUF) { b = 0; bph ^= 1; }
                        if (++s == STAGES) { s = 0; ph ^= 1; }
                    }
                    if (!ok) break;
                    if (SPLITK && lr_here == 0) continue;  // split plan: only the gathering CTA has the rank-r branch
                    // rank-r bf16 branch: one more accumulator tile, fp32
                    if (!mbar_wait(tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA)) { ok = false; break; }
                    tc_fence_after_sync();
                    for (int lr = 0; lr < lr_here; ++lr) {
                        if (!mbar_wait(unp_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA)) { ok = false; break; }
                        tc_fence_after_sync();
                        const uint32_t a_lo = desc_lo0 + s * (STAGE_BYTES >> 4), b_lo = a_lo + (A_BYTES >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                umma_bf16(tmem_base + b * BUF_COLS, desc(a_lo + 2 * k), desc(b_lo + 2 * k), idesc_bf, (lr | k) != 0);
                            umma_commit(empty_bar(s));
                        }
                        if (++s == STAGES) { s = 0; ph ^= 1; }
                    }
                    if (!ok) break;
                    if (elect_one()) umma_commit(tfull_bar(b));
                    if (lane == 0) TRACE_CLK(p.status, 19);
                    if (++b == NBUF) { b = 0; bph ^= 1; }
                }
                if (lane == 0) {
                    flush_wait(p.status, WS_MMA_OPERANDS, w_ops);
                    flush_wait(p.status, WS_MMA_TEMPTY, w_tempty);
                    flush_wait(p.status, WS_KERNEL, clock64() - t_kernel);
                }
            }
        } else {
            // -------------------------------------------------------- nibble -> byte unpack (warps 2, 3)
            // The two warps take k-blocks in turn, each expands a whole one: half of a turn is waiting (the stage's barrier, the loads, the
            // proxy fence), which one warp does while the other works.  Together on every k-block they took 900 cycles for one.
            const int u = lane;
            long long w_full = 0;
            bool ok = true;
            uint32_t s = warp - 2, ph = 0, first_it = 0;  // (s, ph: stage and parity of this warp's next item)
            for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                const int items = (kb1 - kb0) + lr_here;
                for (int i = static_cast<int>((warp - 2 + first_it) & 1); i < items; i += 2) {
                    const uint32_t it = first_it + i;
                    // (before this warp's first wait on what the previous kernel leaves: how long that one runs is no part of a bounded wait, nor of
                    // w_full; a warp's items are two apart)
                    if (it - static_cast<uint32_t>(pre) < 2u) grid_dependency_wait();
                    // A barrier is waited on by its phase's parity, and of a stage expanded early this warp has not seen the activations land: they have when
                    // the stage's MMAs are done.  (Not a wait for the landing itself: the barrier may be two phases on by now.)
                    if (it - STAGES < static_cast<uint32_t>(pre) && !mbar_wait(empty_bar(s), ph ^ 1, abort_flag, p.status, DEV_TIMEOUT_UNPACK)) { ok = false; break; }
                    ok = timed_wait(it < static_cast<uint32_t>(pre) ? pre_bar(s) : full_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_UNPACK, w_full);
                    if (!ok) break;
                    if (first_it == 0 && i == 0 && u == 0) TRACE_CLK(p.status, 14);
                    if (i < kb1 - kb0) {
                        // 16-byte piece idx = u + 32 j of the packed tile: row = idx/4 = u/4 + 8 j, piece c = u%4.
                        // The swizzle phase row%8 = u/4 and the piece do not depend on j, so every address is
                        // a per-thread base plus a compile-time offset.
                        uint8_t* st = smem_gen + s * STAGE_BYTES;
                        const uint4* src = reinterpret_cast<const uint4*>(st + A_BYTES + BU_BYTES) + u;
                        const int c = u & 3, sw = u >> 2;
                        uint8_t* d0 = st + A_BYTES + (u >> 2) * 128 + (((2 * c) ^ sw) << 4);
                        uint8_t* d1 = st + A_BYTES + (u >> 2) * 128 + (((2 * c + 1) ^ sw) << 4);
                        // The loads of a batch are issued before any of its stores: the compiler cannot prove that the
                        // staging buffer and the operand tile do not overlap, so a load written after a store would wait
                        // for it and the whole unpack would run as one dependent chain.
                        constexpr int PIECES = (BN * 4) / 32, BATCH = PIECES < 8 ? PIECES : 8;
#pragma unroll
                        for (int jb = 0; jb < PIECES; jb += BATCH) {
                            uint4 pk[BATCH];
#pragma unroll
                            for (int j = 0; j < BATCH; ++j) pk[j] = src[32 * (jb + j)];
#pragma unroll
                            for (int j = 0; j < BATCH; ++j) {
                                // a word holds codes k..k+3 in bits 7, 2..0 of its bytes and codes k+4..k+7 four bit
                                // positions further up, wrapping around (see prepare.cu): mask, rotate, mask
                                uint4 o0, o1;
                                o0.x = code_bytes(pk[j].x & kSignMag); o0.y = code_bytes(__funnelshift_r(pk[j].x, pk[j].x, 4) & kSignMag);
                                o0.z = code_bytes(pk[j].y & kSignMag); o0.w = code_bytes(__funnelshift_r(pk[j].y, pk[j].y, 4) & kSignMag);
                                o1.x = code_bytes(pk[j].z & kSignMag); o1.y = code_bytes(__funnelshift_r(pk[j].z, pk[j].z, 4) & kSignMag);
                                o1.z = code_bytes(pk[j].w & kSignMag); o1.w = code_bytes(__funnelshift_r(pk[j].w, pk[j].w, 4) & kSignMag);
                                *reinterpret_cast<uint4*>(d0 + (jb + j) * 1024) = o0;  // 8 rows of 128 bytes further down
                                *reinterpret_cast<uint4*>(d1 + (jb + j) * 1024) = o1;
                            }
                        }
                        fence_proxy_async_smem();  // generic-proxy writes -> visible to the tensor core
                    }
                    // each thread signs off its own writes (a warp-wide barrier followed by one lane's arrival costs about
                    // a hundred cycles more on this part than 32 arrivals)
                    mbar_arrive(unp_bar(s));
                    if (first_it == 0 && i == 0 && u == 0) TRACE_CLK(p.status, 15);
                    s += 2;
                    if (s >= STAGES) { s -= STAGES; ph ^= 1; }
                }
                first_it += items;
            }
            grid_dependency_wait();
            if (warp == 2 && u == 0) flush_wait(p.status, WS_UNPACK_FULL, w_full);
        }
    } else {
        reg_alloc<EPI_REGS>();
        // ------------------------------------------------------------ epilogue (warps 4..11)
        // A warp owns 32 token rows (its TMEM lane quadrant) x BN/2 columns.  The accumulators are read with the
        // 16x256b shape: a thread then holds 4 rows (l/4 + 8 i) x the column pairs 2 (l%4) + {0, 1} of every block
        // of 8 columns, so one load of weight scales serves four rows (with the 32x32b shape, one row per thread,
        // every thread would need all column scales of every group and the shared-memory pipe, not the FMA
        // pipe, would bound the kernel).  The weight scales of the thread's columns of a 32-column run lie side by side
        // (see wscale_index in common.h).
        //
        // The buffers of an output tile (one per k-block, then the rank-r one) are one stream of units in two register sets: while
        // one is folded in, the next and its column scales are on their way.  When a buffer's last unit has arrived, the buffer
        // goes back to the MMA warp, the next buffer is waited for (it is there in the steady state) and its first
        // unit requested, all before the last unit is folded in; so neither the hand-over nor a round
        // trip to tensor or shared memory is paid, and there is one hand-over per 128 codes.
        const int q = warp & 3;
        const int half = (warp - 4) >> 2;
        const int lr4 = lane >> 2;        // row inside a group of 8
        const int lc2 = (lane & 3) * 2;   // first of this thread's two columns inside a block of 8
        uint32_t b = 0, bph = 0;          // accumulator tile read next, parity its "full" barrier is waited with
        uint32_t slot = 0;                // scale record of the current k-block
        long long w_tfull = 0;
        const long long t_epi = clock64();
        const uint32_t taddr0 = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + half * HB;
        // No vote after a wait: the warp is converged there, so the barrier test, the abort flag and the clock are read
        // by one instruction for all lanes and every lane gets the same answer.
        bool ok = true;
        uint32_t raw[2][UC];     // [0..UC/2-1]: TMEM lanes 0..15 of the quadrant (rows i = 0, 1), then lanes 16..31 (rows 2, 3)
        uint64_t w2[2][UC / 8];  // a unit's column scales, two adjacent columns each
        float sxv[2][4];         // a group's token scales of the thread's rows (groups of 128: in use, requested)
        auto request_unit = [&](uint32_t buf, int u, uint32_t (&dst)[UC]) {
            const uint32_t t = taddr0 + buf * BUF_COLS + u / UPG * BN + u % UPG * UC;
            if constexpr (UC == 32) {
                tmem_ld_16x256b_x2(t, dst);
                tmem_ld_16x256b_x2(t + 16, dst + 8);
                tmem_ld_16x256b_x2(t + (16u << 16), dst + 16);
                tmem_ld_16x256b_x2(t + (16u << 16) + 16, dst + 24);
            } else {
                tmem_ld_16x256b_x2(t, dst);
                tmem_ld_16x256b_x2(t + (16u << 16), dst + 8);
            }
        };
        // (volatile: requested here, not where they are used)
        auto request_scales = [&](uint32_t sc_slot, int u) {
            const uint32_t sc = sc_base + sc_slot * SC_BYTES;
            const int gi = u / UPG, col = half * HB + u % UPG * UC;  // first column of the unit in the tile
            const uint32_t a = sc + 4u * (gi * BN + (col & ~31) + 4 * lc2 + (col & 31) / 4);
#pragma unroll
            for (int e = 0; e < UC / 8; e += 2)
                asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(w2[u & 1][e]), "=l"(w2[u & 1][e + 1]) : "r"(a + 8u * e) : "memory");
            if (u % UPG == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(sxv[GPK == 2 ? gi : 1][i]) : "r"(sc + 4u * (2 * BN + gi * BM + q * 32 + lr4 + 8 * i)) : "memory");
            }
        };
        auto unit_arrived = [&](uint32_t (&v)[UC]) {
            tmem_ld_wait();
#pragma unroll
            for (int c = 0; c < UC; c += 16) tmem_ld_fence(*reinterpret_cast<uint32_t(*)[16]>(v + c));
            if constexpr (kI8Path) {
#pragma unroll
                for (int i = 0; i < UC; ++i) v[i] = __float_as_uint(__int2float_rn(static_cast<int>(v[i])));  // |P| < 2^24: exact
            }
        };
        // element of a unit: block of 8 columns cb (0 .. UC / 8 - 1), row i, first of the two columns
        auto element = [](int cb, int i) { return UC / 2 * (i >> 1) + 4 * cb + 2 * (i & 1); };
        auto pair_index = [](int u, int cb, int i) { return (u % UPG * (UC / 8) + cb) * 4 + i; };  // its accumulator pair
        auto release_tile = [&](uint32_t buf) {  // every tcgen05.ld of this thread on the tile has completed
            tc_fence_before_sync();
            mbar_arrive(tempty_bar(buf));  // all lanes arrive (see the unpack warps' note on the cost of electing one)
        };
        for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
            const int m0 = (tile % num_m_blocks) * BM;
            const int n0 = (tile / num_m_blocks) * BN;
            if (!SPLITK && m0 + q * 32 >= p.M) {  // a warp without token rows only hands the buffers back
                for (int i = kb0; i <= kb1; ++i) {
                    ok = mbar_wait(tfull_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE);
                    if (!ok) break;
                    release_tile(b);
                    if (++b == NBUF) { b = 0; bph ^= 1; }
                    if (i < kb1 && ++slot == SC_SLOTS) slot = 0;
                }
                continue;
            }
            const int rbase = m0 + q * 32 + lr4;  // this thread's rows: rbase + 8 i, i = 0..3
            const int colbase = n0 + half * HB;
            uint64_t acc2[HB / 2];  // two adjacent columns per 64-bit register: [(block of 8 columns) * 4 + row i]
#pragma unroll
            for (int j = 0; j < HB / 2; ++j) acc2[j] = 0ull;

            // Folds a unit in.  The scale of an element is t = s_x * (2^18 s_w): two bf16-valued factors (and a power of two), so
            // the fp32 product is EXACT.  It is formed for two adjacent columns at a time with one packed multiply whose operands
            // are 64-bit registers as they come (the pair of column scales straight from a shared-memory load, the token's
            // scale duplicated once per group); then acc = fma(S, t, acc), again packed (the accumulator's two adjacent columns are
            // consecutive registers of the tensor-memory load): one rounding per element and group, two instructions per two elements.
            auto fold_unit = [&](int u) {
                uint32_t (&v)[UC] = raw[u & 1];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    // the accumulator holds S = 2^-18 P (integer-path build: P as int32, and 2^-18 goes into the token scale)
                    const float sx = sxv[u / UPG][i] * (kI8Path ? 1.0f / kWScaleFold : 1.0f);
                    const uint64_t sx2 = pack_f32x2(sx, sx);
#pragma unroll
                    for (int cb = 0; cb < UC / 8; ++cb) {
                        const int x = element(cb, i), a = pair_index(u, cb, i);
                        acc2[a] = fma_f32x2(pack_u32x2(v[x], v[x + 1]), mul_f32x2(w2[u & 1][cb], sx2), acc2[a]);
                    }
                }
            };

            // first buffer and scales of this output tile (split plan: of this CTA's range, which may be empty, and only the gathering
            // CTA has a rank-r tile)
            if (!SPLITK || kb1 > kb0 || lr_here > 0) {
                ok = timed_wait(tfull_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_tfull);
                if (!ok) break;
                if (warp == 4 && lane == 0) TRACE_CLK(p.status, 20);
                tc_fence_after_sync();
                request_unit(b, 0, raw[0]);
                if (!SPLITK || kb1 > kb0) request_scales(slot, 0);  // (they landed with the operands the buffer was made from)
            }

            for (int kb = kb0; kb < kb1; ++kb) {
                if (warp == 4 && lane == 0 && kb * GPK == 8) TRACE_CLK(p.status, 21);
                // what comes after this buffer: the next k-block's, or the rank-r tile
                const uint32_t nb = b + 1 == NBUF ? 0 : b + 1, nbph = b + 1 == NBUF ? bph ^ 1 : bph;
                const uint32_t nslot = slot + 1 == SC_SLOTS ? 0 : slot + 1;
                const bool new_scales = kb + 1 < kb1;
                const bool more = !SPLITK || new_scales || lr_here > 0;  // another buffer follows (always, unless split)
#pragma unroll
                for (int u = 0; u < NU; ++u) {
                    unit_arrived(raw[u & 1]);
                    if constexpr (GPK == 1) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) sxv[0][i] = u == 0 ? sxv[1][i] : sxv[0][i];
                    }
                    if (u + 1 < NU) {
                        request_unit(b, u + 1, raw[(u + 1) & 1]);
                        request_scales(slot, u + 1);
                    } else {
                        // the whole buffer is in registers: hand it back to the MMA warp, and request the next one's first unit
                        release_tile(b);
                        if (more) {
                            ok = timed_wait(tfull_bar(nb), nbph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_tfull);
                            if (!ok) break;
                            tc_fence_after_sync();
                            request_unit(nb, 0, raw[0]);  // (NU is even: the last unit sits in raw[1])
                            if (new_scales) request_scales(nslot, 0);
                        }
                    }
                    fold_unit(u);
                }
                if (!ok) break;
                slot = nslot;
                b = nb;
                bph = nbph;
            }
            if (!ok) break;
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 22);
            // rank-r branch: an fp32 tile whose first unit is already on its way
            if (!SPLITK || lr_here > 0) {
#pragma unroll
                for (int u = 0; u < UPG; ++u) {
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < UC; c += 16) tmem_ld_fence(*reinterpret_cast<uint32_t(*)[16]>(raw[u & 1] + c));
                    if (u + 1 < UPG) request_unit(b, u + 1, raw[(u + 1) & 1]);
                    else release_tile(b);
#pragma unroll
                    for (int cb = 0; cb < UC / 8; ++cb)
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int x = element(cb, i), a = pair_index(u, cb, i);
                            acc2[a] = add_f32x2(acc2[a], pack_u32x2(raw[u & 1][x], raw[u & 1][x + 1]));
                        }
                }
                if (++b == NBUF) { b = 0; bph ^= 1; }
            }
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 23);
            if constexpr (SPLITK) {
                // The partial tiles meet in the last CTA of the cluster.  Every other CTA's epilogue threads put their 16
                // register pairs into their own shared memory (the operand ring, idle by now: every MMA of this CTA has
                // completed), word j of thread t at [j][t]; one thread then sends the 32 KB to the gathering CTA with a bulk
                // copy that counts its bytes on that CTA's barrier.  The gathering thread t holds the same rows and columns
                // in every CTA and adds the partial tiles in rank order.
                const uint32_t et = threadIdx.x - 128u;
                const uint32_t red_base = smem_base + P::RED_OFFSET;
                if (!gathers) {
#pragma unroll
                    for (int j = 0; j < HB / 2; ++j) st_shared_u64(smem_base + j * (NUM_EPI_WARPS * 256u) + et * 8u, acc2[j]);
                    fence_proxy_async_smem();       // these writes -> visible to the copy engine
                    mbar_arrive(red_bar + 8u);
                    if (et == 0 && mbar_wait(red_bar + 8u, 0, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE))  // a bounded wait, like all
                        bulk_copy_to_cluster(map_to_cta(red_base + crank * RED_BYTES, csize - 1), smem_base, RED_BYTES,
                                             map_to_cta(red_bar, csize - 1));
                    continue;  // one tile per cluster: nothing else to do (the cluster meets once more before anyone leaves)
                }
                if (!mbar_wait(red_bar, 0, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE)) { ok = false; break; }
                for (uint32_t r = 0; r + 1 < csize; ++r) {
#pragma unroll
                    for (int j = 0; j < HB / 2; ++j)
                        acc2[j] = add_f32x2(acc2[j], ld_shared_u64(red_base + r * RED_BYTES + j * (NUM_EPI_WARPS * 256u) + et * 8u));
                }
            }
            if constexpr (HB < 32) {
                // two blocks of 8 columns: four bytes of each per lane
#pragma unroll
                for (int t = 0; t < HB / 8; ++t) {
                    const int col = colbase + t * 8 + lc2;
                    const float2 bv = col < p.N ? __ldg(reinterpret_cast<const float2*>(p.bias + col)) : make_float2(0.f, 0.f);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        float y_lo, y_hi;
                        unpack_f32x2(acc2[t * 4 + i], y_lo, y_hi);
                        const int row = rbase + 8 * i;
                        if (row < p.M && col < p.N)
                            *reinterpret_cast<uint32_t*>(p.y + static_cast<size_t>(row) * p.N + col) = pack_bf16x2(y_lo + bv.x, y_hi + bv.y);
                    }
                }
            } else {
                // A lane holds 2 of the 8 columns of every block; four blocks are transposed inside the quad of lanes
                // (two exchange steps) so that each lane ends up with all 8 columns = 16 bytes of one block and the
                // warp writes 64 contiguous bytes per row.
                const int j = lane & 3;
#pragma unroll
                for (int m = 0; m < HB / 32; ++m) {
                    float2 bv[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const int col = colbase + (4 * m + t) * 8 + lc2;
                        bv[t] = col < p.N ? __ldg(reinterpret_cast<const float2*>(p.bias + col)) : make_float2(0.f, 0.f);
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t v[4];
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            float y_lo, y_hi;
                            unpack_f32x2(acc2[(4 * m + t) * 4 + i], y_lo, y_hi);
                            v[t] = pack_bf16x2(y_lo + bv[t].x, y_hi + bv[t].y);
                        }
                        const bool odd = (j & 1) != 0, upper = (j & 2) != 0;
                        const uint32_t r01 = __shfl_xor_sync(0xffffffffu, odd ? v[0] : v[1], 1);
                        const uint32_t r23 = __shfl_xor_sync(0xffffffffu, odd ? v[2] : v[3], 1);
                        const uint32_t u0 = odd ? r01 : v[0], u1 = odd ? v[1] : r01;  // block (j & 1), lanes 2 (j / 2) + {0, 1}
                        const uint32_t p0 = odd ? r23 : v[2], p1 = odd ? v[3] : r23;  // block 2 + (j & 1)
                        const uint32_t x0 = __shfl_xor_sync(0xffffffffu, upper ? u0 : p0, 2);
                        const uint32_t x1 = __shfl_xor_sync(0xffffffffu, upper ? u1 : p1, 2);
                        const uint4 o = upper ? make_uint4(x0, x1, p0, p1) : make_uint4(u0, u1, x0, x1);  // block j
                        const int row = rbase + 8 * i;
                        const int col = colbase + (4 * m + j) * 8;
                        if (row < p.M && col < p.N)
                            *reinterpret_cast<uint4*>(p.y + static_cast<size_t>(row) * p.N + col) = o;
                    }
                }
            }
        }
        if (warp == 4 && lane == 0) TRACE_CLK(p.status, 24);
        if (warp == 4 && lane == 0) {
            flush_wait(p.status, WS_EPI_TFULL, w_tfull);
            flush_wait(p.status, WS_EPI_TOTAL, clock64() - t_epi);
        }
    }

    // ---------------------------------------------------------------- teardown
    if (warp == 1 && lane == 0 && *abort_flag != 0) umma_drain(bar_base + 8u * (3 * STAGES + 8));  // a wait gave up: let issued MMAs finish first
    tc_fence_before_sync();
    __syncthreads();
    if constexpr (SPLITK) cluster_sync_all();  // no CTA of the cluster leaves while another may still write into it or signal it
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, 512);
    }
}

}  // namespace

dirotq_status_t launch_w4a4_narrow(const dirotq_layer* L, const GemmArgs& a, int columns, bool may_split, cudaStream_t stream) {
    const Geometry& g = L->geo;
    CUtensorMap tmap_codes, tmap_xscale, tmap_xh;
    dirotq_status_t st;
    st = encode_tmap_2d(&tmap_codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a.codes, (uint64_t)g.K_lp, (uint64_t)a.M,
                        (uint64_t)g.K_lp, BKC, box_rows(a.M), CU_TENSOR_MAP_SWIZZLE_128B);
    if (st != DIROTQ_OK) return st;
    st = encode_tmap_2d(&tmap_xscale, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.xscale, (uint64_t)a.ldm, (uint64_t)g.n_g,
                        (uint64_t)a.ldm * 4, BM, BKC / g.G, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (st != DIROTQ_OK) return st;
    st = encode_tmap_2d(&tmap_xh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.xh, (uint64_t)g.r_pad, (uint64_t)a.M,
                        (uint64_t)g.r_pad * 2, 64, box_rows(a.M), CU_TENSOR_MAP_SWIZZLE_128B);
    if (st != DIROTQ_OK) return st;

    GemmKernelParams p;
    p.M = a.M; p.N = g.N; p.n_g = g.n_g;
    p.num_kb = (g.K_lp + BKC - 1) / BKC;
    p.lr_chunks = g.r_pad / 64;
    p.bias = reinterpret_cast<const float*>(L->blob + L->lay.off_bias);
    p.y = a.y; p.partials = a.partials; p.status = a.status; p.early_weights = a.early_weights; p.x_rows = box_rows(a.M);

    const int num_tiles = ((a.M + BM - 1) / BM) * ((g.N + columns - 1) / columns), sms = sm_count(L->device), which = g.G == 64 ? 0 : 1;
    using KernelFn = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap,
                              const CUtensorMap, const CUtensorMap, const GemmKernelParams);
    if (may_split) {
        // The split plan: the largest cluster (4, 3 or 2 CTAs over the k-blocks of a tile) that leaves every CTA at least two
        // k-blocks and whose clusters, one per tile, are all resident at once (asked of the runtime once per device and size).
        // Only on request (knob value 66): the partial tiles are added in another order than one CTA adds the groups, and by
        // default a token's output bits do not depend on how many other tokens the call has.
        const KernelFn kern = g.G == 64 ? w4a4_narrow_kernel<64, true, 64> : w4a4_narrow_kernel<128, true, 64>;
        constexpr int smem = Plan<true, 64>::SMEM_BYTES;
        static SmemOptIn<2> opt_in;
        static std::atomic<int> resident[64][SPLIT_MAX + 1];  // 0: not asked yet; else clusters resident at once + 1
        if (!opt_in.ensure(kern, which, L->device, smem)) return DIROTQ_ERR_CUDA;
        for (int c = SPLIT_MAX; c >= 2; --c) {
            if (p.num_kb / c < 2) continue;
            const int dev = L->device;
            int have = dev >= 0 && dev < 64 ? resident[dev][c].load() : 0;
            if (have == 0) {
                have = 1 + max_active_clusters(kern, c, NUM_THREADS, smem);  // (both group sizes have the same footprint)
                if (dev >= 0 && dev < 64) resident[dev][c].store(have);
            }
            if (num_tiles > have - 1) continue;
            const cudaError_t err = launch_kernel_clusters(kern, num_tiles * c, c, NUM_THREADS, smem, stream, true, tmap_codes, L->tmap_wpacked64,
                                                           L->tmap_wscale64, tmap_xscale, tmap_xh, L->tmap_wh64, p);
            return err == cudaSuccess ? DIROTQ_OK : DIROTQ_ERR_CUDA;
        }
    }
    const bool half = columns == 32;
    const KernelFn kern = half ? w4a4_narrow_kernel<64, false, 32> : g.G == 64 ? w4a4_narrow_kernel<64, false, 64> : w4a4_narrow_kernel<128, false, 64>;
    const int smem = half ? Plan<false, 32>::SMEM_BYTES : Plan<false, 64>::SMEM_BYTES;
    static SmemOptIn<3> opt_in;
    if (!opt_in.ensure(kern, half ? 2 : which, L->device, smem)) return DIROTQ_ERR_CUDA;
    const cudaError_t err = launch_kernel(kern, num_tiles < sms ? num_tiles : sms, NUM_THREADS, smem, stream, true, tmap_codes,
                                          half ? L->tmap_wpacked32 : L->tmap_wpacked64, half ? L->tmap_wscale32 : L->tmap_wscale64, tmap_xscale, tmap_xh,
                                          half ? L->tmap_wh32 : L->tmap_wh64, p);
    return err == cudaSuccess ? DIROTQ_OK : DIROTQ_ERR_CUDA;
}

}  // namespace dirotq
