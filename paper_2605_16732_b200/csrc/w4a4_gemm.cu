// Kernels (b)+(c): W4A4 group GEMM with per-group rescale, bf16 rank-r branch and bias.
//
//   y[m,n] = bf16( sum_g s_x[m,g] s_w[g,n] P_g[m,n]  +  sum_{i<r} x~_h[m,i] W~_h[i,n]  +  bias[n] )
//   P_g[m,n] = sum_{j in group g} q_x[m,j] q_w[j,n]                              (paper Eq. 5)
//
// sm_100a has no INT4 MMA, and an int32 accumulator costs a conversion per element and group before it
// can be scaled.  The integer products are therefore computed EXACTLY on the 8-bit float path
// (tcgen05.mma kind::f8f6f4, E4M3 operands, fp32 accumulation):
//   * an E4M3 byte s0000mmm is (-1)^s m * 2^-9 for m = 0..7 (subnormals; with a fourth magnitude bit, 0..15: the
//     first binade continues the same line), so a code stored as sign + magnitude IS an E4M3 number;
//   * activation codes arrive from kernel (a) one per byte in that form: q_x * 2^-9 (the asymmetric variant
//     stores u = 0..15 as 0000uuuu = u * 2^-9);
//   * weight codes stay packed (two per byte: sign + 3-bit magnitude each) in HBM and in the TMA staging
//     buffer; two "unpack" warps split every 32-bit word of eight codes into two words of four bytes
//     s0000mmm = q_w * 2^-9 (one mask, one rotate and one mask: the nibble order of prepare.cu is chosen for
//     that) in the 128-byte-swizzled layout the MMA reads;
//   * every product is an integer times 2^-18 and a group's sum is below 2^24 in magnitude, so the fp32
//     accumulator holds S_g = 2^-18 P_g without rounding.  The weight scales are stored as 2^18 s_w (exact), so
//         t = s_x * (2^18 s_w)            -- exact: two bf16-valued factors and a power of two --
//         acc = fma(S_g, t, acc)          -- one rounding per element and group --
//     folds a group in with one (packed, two columns at a time) multiply and one fused multiply-add per element and
//     no integer conversion.
// The exactness of the accumulation is a property of the tensor core that the parity tests pin: the
// group sums exported by the debug entry equal the CPU checker's int32 sums bit for bit, on random
// codes and on patterns built to lose low bits (long runs of +-49 followed by +-1).
//
// Every K-group gets its own accumulator tile in tensor memory (two tiles, ping-pong): the MMA warp
// fills tile g%2 while the epilogue warps drain tile (g-1)%2 into per-thread fp32 accumulators.  The
// bf16 rank-r branch is issued as one more "group" (kind::f16 into the same ping-pong tile) and added
// unscaled.
//
// Tiles of 256, 192 or 128 columns here; w4a4_narrow.cu has the same computation in 64- and 32-column tiles.
//
// What bounds it: the issue slots of the schedulers.  The rescale's packed multiply and multiply-add hold a scheduler's issue port for two
// cycles each and nothing issues beside them: of the 1125 cycles a K-group of a 128 x 256 tile took, 660 were these, and everything else that
// is issued on the same schedulers (the epilogue's own loads, barriers and counters, the weight expansion, the MMA warp) came on top, in no
// pipe's peak but in the sum.  So what helps is fewer instructions per group:
//   * CTA pairs (PAIRED): each CTA loads its own activation codes and loads AND expands half of the tile's weights, half the expansion.  With groups of
//     128 the two expanding warps had set the pace (1430 of 1509 cycles per k-block busy).  One tile of 256 rows in one CTA (TALL) halves it too.
//   * a group's scales in a record of their own that lands with the operands: no barriers, tests and arrivals for scales, one offset to step on;
//   * the next tile's first chunk requested after a plain wait, at one place (the tile is practically always there);
//   * warp numbers known to be uniform, so that addresses and barriers are worked out on the uniform path;
//   * row and column numbers worked out at the end of a tile, not held: with 128 accumulators and 64 values in flight a thread
//     has 30 registers left, and every one too many turned into moves on the port that is the bound.
// 4608 x 3072 -> 9216, us alone, groups of 64 / 128: 256 columns 278 -> 252 / 190 -> 185, pairs 236 / 153 (266 / 164 before the others), tall
// 241 / 157, 192 columns 311 -> 267 / 211 -> 200, 128 columns 328 -> 290 / 222 -> 224.
//
// Roles (384 threads = 3 warpgroups):
//   warpgroup 0: warp 0 TMA producer, warp 1 MMA issuer + TMEM owner, warps 2-3 nibble -> byte unpack
//   warpgroups 1-2: epilogue; warp%4 selects the TMEM lane quadrant (token rows), the warpgroup
//                   selects the half of the tile's columns.
#include "w4a4.cuh"
#include "w4a4_plan.h"

#include <atomic>

namespace dirotq {
namespace {

// Plan for tiles of BN output columns.
//   256: two epilogue warpgroups, 128 columns (128 fp32 accumulators) per thread; an accumulator tile can only be read in
//        pieces between the arithmetic and is held for three quarters of a group.
//   192: three epilogue warpgroups, 64 columns per thread: a thread's share of an accumulator tile fits its two chunk
//        buffers, so the tile goes back to the tensor core after the first quarter of a group, and three warps per scheduler
//        hide each other's waits.  16 warps: 152 registers for the epilogue threads, 56 for the others.
//   128: two warpgroups, 64 columns per thread, four accumulator tiles; for layers whose wider tiles would leave SMs idle.
// and of how many token rows:
//   ONE:  128.
//   PAIRED: 128 in each of two CTAs that share every MMA (tcgen05.mma.cta_group::2, 256 columns): each loads its own activation codes and loads and
//         expands half of the tile's weights.
//   TALL: 256 in one CTA, a warpgroup for each half (128 columns): a warp's share is that of the 256-column tile, the weights to expand are half.
enum Rows : int { ONE, PAIRED, TALL };
template <int BN, Rows ROWS = ONE>
struct Plan {
    static constexpr int EPI_WG = BN == 192 ? 3 : 2;  // epilogue warpgroups
    static constexpr int EPI_WARPS = 4 * EPI_WG;
    static constexpr int THREADS = 128 + 128 * EPI_WG;
    // setmaxnreg budgets: 128 * AUX + 128 * EPI_WG * EPI at most what the block is launched with
    static constexpr int HB = ROWS == TALL ? BN : BN / EPI_WG;  // columns per epilogue warp
    static constexpr int EPI_REGS = EPI_WG == 3 ? 152 : HB == 128 ? 224 : 216;
    static constexpr int AUX_REGS = EPI_WG == 3 ? 56 : HB == 128 ? 56 : 64;
    static constexpr int SC_SLOTS = BN == 192 ? 13 : BN == 128 && ROWS == ONE ? 18 : 14;  // scale records, one per group
    static constexpr int STAGES = ROWS == PAIRED ? 5 : ROWS == TALL ? 3 : BN == 256 ? 3 : BN == 192 ? 4 : 5;
    static constexpr int CTA_ROWS = ROWS == TALL ? 2 * BM : BM;   // token rows of a CTA
    static constexpr int TILE_ROWS = ROWS == ONE ? BM : 2 * BM;   // ... of a tile
    static constexpr int BUF_COLS = ROWS == TALL ? 2 * BN : BN;   // tensor-memory columns of an accumulator tile
    static constexpr int WROWS = ROWS == PAIRED ? BN / 2 : BN;    // weight rows this CTA loads and expands
    static constexpr int AC_BYTES = CTA_ROWS * BKC;   // activation codes / bf16 x~_h chunk
    static constexpr int BU_BYTES = WROWS * BKC;      // unpacked weight codes / bf16 W~_h chunk (32 KB at BN = 256)
    static constexpr int BP_BYTES = WROWS * BKC / 2;  // packed weight codes (TMA staging)
    static constexpr int STAGE_BYTES = AC_BYTES + BU_BYTES + BP_BYTES;  // KB: 256 columns 64, 192 52, 128 40; tall 56, a pair's CTA 40
    static constexpr int SC_SW_BYTES = BN * 4, SC_BYTES = SC_SW_BYTES + CTA_ROWS * 4;  // weight scales, activation scales
    static constexpr int BAR_OFFSET = STAGES * STAGE_BYTES + SC_SLOTS * SC_BYTES;
    static constexpr int SMEM_BYTES = BAR_OFFSET + 512 + 1024;
    static_assert(SMEM_BYTES <= 232448, "shared memory plan too large");
    static_assert(STAGE_BYTES % 1024 == 0 && SC_BYTES % 128 == 0, "tile alignment");
    static_assert(8 * (4 * STAGES + 11) <= 400, "barriers end below the words at +400");
};

template <int G, bool kPartials, int BN, Rows ROWS>
__global__ void __launch_bounds__(Plan<BN, ROWS>::THREADS, 1)
w4a4_gemm_kernel(const __grid_constant__ CUtensorMap tmap_codes, const __grid_constant__ CUtensorMap tmap_wpacked,
                 const __grid_constant__ CUtensorMap tmap_wscale, const __grid_constant__ CUtensorMap tmap_xscale,
                 const __grid_constant__ CUtensorMap tmap_xh, const __grid_constant__ CUtensorMap tmap_wh,
                 const GemmKernelParams p) {
    using P = Plan<BN, ROWS>;
    constexpr bool PAIR = ROWS == PAIRED;
    constexpr int STAGES = P::STAGES, STAGE_BYTES = P::STAGE_BYTES, BU_BYTES = P::BU_BYTES, BP_BYTES = P::BP_BYTES;
    constexpr int SC_SW_BYTES = P::SC_SW_BYTES, SC_BYTES = P::SC_BYTES, BAR_OFFSET = P::BAR_OFFSET;
    constexpr int SC_SLOTS = P::SC_SLOTS, NUM_EPI_WARPS = P::EPI_WARPS;
    constexpr int HB = P::HB;          // columns per epilogue warp: the warpgroup selects the slice of the tile (TALL: the half of its rows)
    constexpr int AC_BYTES = P::AC_BYTES, BUF_COLS = P::BUF_COLS, TILE_ROWS = P::TILE_ROWS;
    constexpr int CHUNKS = HB / 32;    // 32-column chunks per epilogue warp and accumulator tile
    constexpr int GPK = BKC / G;       // groups per k-block: 2 (G = 64) or 1 (G = 128)
    constexpr int MMA_PER_G = G / 32;  // 8-bit MMA instructions (K = 32) per group
    constexpr int NBUF = 512 / BUF_COLS;  // accumulator tiles in tensor memory: 2 of 256 columns, 4 of 128 (the barrier map has four slots)
    // A group's scales land with its k-block's operands, on the same barrier, in a ring of records that has no "empty" barriers: the
    // producer loads k-block j when the MMAs of j - STAGES are done, those had waited until the epilogue was through with the group
    // NBUF accumulator tiles before their last one, so of the groups before k-block j only the last STAGES * GPK + NBUF may still be read.
    static_assert(SC_SLOTS >= (STAGES + 1) * GPK + NBUF, "scale records");

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sc_base = smem_base + STAGES * STAGE_BYTES;
    const uint32_t bar_base = smem_base + BAR_OFFSET;
    // barriers: full[S], unpacked[S], empty[S], tmem_full[4], tmem_empty[4], spare, the other CTA's tmem_empty[2]
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto unp_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
    auto empty_bar = [&](int s) { return bar_base + 8u * (2 * STAGES + s); };
    auto tfull_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + a); };
    auto tempty_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + 4 + a); };
    auto peer_tempty_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + 9 + a); };  // pairs: in the leader, the other CTA's
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

    const uint32_t crank = PAIR ? blockIdx.x & 1u : 0u;  // (the rank in the cluster, known to be uniform)
    const int num_m_blocks = (p.M + TILE_ROWS - 1) / TILE_ROWS;
    const int num_n_blocks = (p.N + BN - 1) / BN;
    auto first_tile = [&]() { return static_cast<int>(PAIR ? blockIdx.x >> 1 : blockIdx.x); };
    auto tile_stride = [&]() { return static_cast<int>(PAIR ? gridDim.x >> 1 : gridDim.x); };
    auto tile_row = [&](int tile) { return (tile % num_m_blocks) * TILE_ROWS + static_cast<int>(crank) * BM; };  // this CTA's first row
    const int num_tiles = num_m_blocks * num_n_blocks;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full_bar(s), 1);
            // every thread of the two unpack warps arrives for itself; of a pair's four, one lane each, on the leader's barrier
            mbar_init(unp_bar(s), PAIR ? 4 : 64);
            mbar_init(empty_bar(s), 1);
            mbar_init(pre_bar(s), 1);
        }
        for (int a = 0; a < NBUF; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), NUM_EPI_WARPS * 32);
            if (PAIR) mbar_init(peer_tempty_bar(a), 1);
        }
        mbar_init(bar_base + 8u * (3 * STAGES + 8), 1);  // spare: see umma_drain
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
        if constexpr (PAIR) {
            tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
            tmem_relinquish_pair();
        } else {
            tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
            tmem_relinquish();
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();  // the other CTA's barriers are initialised before anything arrives on them
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // everything above touched only this CTA's own shared and tensor memory; what follows reads the first kernel's output
    if (threadIdx.x == 0) TRACE_CLK(p.status, 10);
    // Weights and their scales may be loaded, and expanded, while the previous kernel is still running (GemmArgs::early_weights): those of the
    // first tile's first stages land on barriers of their own, the stage's barrier then counts the activations only.
    // (Not in pairs, where one barrier tells the leader of both operands.)
    const int pre = !PAIR && p.early_weights && first_tile() < num_tiles ? min(STAGES, p.num_kb) : 0;
    if (warp == 0 && pre > 0 && elect_one()) {
        const int n0 = (first_tile() / num_m_blocks) * BN;
        for (int j = 0; j < pre; ++j) {
            const int groups = min(GPK, p.n_g - j * GPK);
            mbar_arrive_expect_tx(pre_bar(j), BP_BYTES + groups * SC_SW_BYTES);
            tma_load_2d(smem_base + j * STAGE_BYTES + AC_BYTES + BU_BYTES, &tmap_wpacked, pre_bar(j), j * (BKC / 2), n0);
            for (int gi = 0; gi < groups; ++gi)
                tma_load_2d(sc_base + (j * GPK + gi) * SC_BYTES, &tmap_wscale, pre_bar(j), n0, j * GPK + gi);
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
        reg_dealloc<P::AUX_REGS>();

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
                    const int m0 = tile_row(tile);
                    const int n0 = (tile / num_m_blocks) * BN, w0 = n0 + static_cast<int>(crank) * P::WROWS;
                    for (int kb = 0; kb < p.num_kb; ++kb, at.next()) {
                        const uint32_t s = at.s;
                        if (!timed_wait(empty_bar(s), at.ph ^ 1, abort_flag, p.status, DEV_TIMEOUT_PRODUCER, w_empty)) { ok = false; break; }
                        const uint32_t st = smem_base + s * STAGE_BYTES;
                        const int groups = min(GPK, p.n_g - kb * GPK);  // (an odd number of groups: the last k-block has one)
                        const bool weights = at.it >= static_cast<uint32_t>(pre);
                        if (elect_one()) {
                            mbar_arrive_expect_tx(full_bar(s), (ROWS == ONE ? p.x_rows * BKC : AC_BYTES) + (weights ? BP_BYTES : 0) + groups * (weights ? SC_BYTES : SC_BYTES - SC_SW_BYTES));
                            tma_load_2d(st, &tmap_codes, full_bar(s), kb * BKC, m0);
                            if (ROWS == TALL) tma_load_2d(st + A_BYTES, &tmap_codes, full_bar(s), kb * BKC, m0 + BM);
                            if (weights) tma_load_2d(st + AC_BYTES + BU_BYTES, &tmap_wpacked, full_bar(s), kb * (BKC / 2), w0);
                        }
#pragma unroll
                        for (int gi = 0; gi < GPK; ++gi) {
                            if (gi < groups) {
                                if (elect_one()) {
                                    const uint32_t sc = sc_base + slot * SC_BYTES;
                                    if (weights) tma_load_2d(sc, &tmap_wscale, full_bar(s), n0, kb * GPK + gi);
                                    tma_load_2d(sc + SC_SW_BYTES, &tmap_xscale, full_bar(s), m0, kb * GPK + gi);
                                    if (at.it == 0) TRACE_CLK(p.status, 12);
                                }
                                if (++slot == SC_SLOTS) slot = 0;
                            }
                        }
                    }
                    if (!ok) break;
                    for (int lr = 0; lr < p.lr_chunks; ++lr, at.next()) {
                        const uint32_t s = at.s;
                        if (!mbar_wait(empty_bar(s), at.ph ^ 1, abort_flag, p.status, DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
                        const uint32_t st = smem_base + s * STAGE_BYTES;
                        if (elect_one()) {
                            mbar_arrive_expect_tx(full_bar(s), (ROWS == ONE ? p.x_rows * BKC : AC_BYTES) + BU_BYTES);
                            tma_load_2d(st, &tmap_xh, full_bar(s), lr * 64, m0);
                            if (ROWS == TALL) tma_load_2d(st + A_BYTES, &tmap_xh, full_bar(s), lr * 64, m0 + BM);
                            tma_load_2d(st + AC_BYTES, &tmap_wh, full_bar(s), lr * 64, w0);
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
        } else if (PAIR && warp == 1 && crank != 0) {
            // -------------------------------------------------------- pairs: "accumulator tile drained", passed on to the leader
            // (one arrival over the cluster for the 256 of this CTA's epilogue threads, which do not wait for it)
            uint32_t b = 0, bph = 0;
            bool ok = true;
            for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                for (int g = 0; g <= p.n_g; ++g) {
                    ok = mbar_wait(tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA);
                    if (!ok) break;
                    if (elect_one()) mbar_arrive_cluster(map_to_cta(peer_tempty_bar(b), 0));
                    if (++b == NBUF) { b = 0; bph ^= 1; }
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
                constexpr uint32_t MMA_ROWS = PAIR ? 2 * BM : BM;
                constexpr uint32_t idesc_f8 = umma_idesc(1 /*f32*/, 0 /*E4M3*/, MMA_ROWS, BN);
                constexpr uint32_t idesc_i8 = umma_idesc(2 /*s32*/, 1 /*s8*/, MMA_ROWS, BN);  // integer-path build only
                constexpr uint32_t idesc_bf = umma_idesc(1 /*f32*/, 1 /*bf16*/, MMA_ROWS, BN);
                const uint64_t desc0 = umma_desc_sw128(smem_base);
                const uint32_t desc_hi = static_cast<uint32_t>(desc0 >> 32), desc_lo0 = static_cast<uint32_t>(desc0);
                auto desc = [&](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
                auto commit = [&](uint32_t bar) {
                    if constexpr (PAIR) umma_commit_pair(bar, 3);  // the same barrier of both CTAs
                    else umma_commit(bar);
                };
                uint32_t s = 0, ph = 0;        // stage of the operand ring and its parity
                uint32_t b = 0, bph = 1;       // accumulator tile and the parity its "empty" barrier is waited with
                int pre_left = pre;
                long long w_ops = 0, w_tempty = 0;
                const long long t_kernel = clock64();
                bool ok = true;
                for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                    int groups_left = p.n_g;
                    for (int kb = 0; ok && kb < p.num_kb; ++kb) {
                        // the unpack warps arrive after they have seen the stage's loads land (one barrier for both operands), so
                        // their barrier covers the activation codes as well
                        if (!timed_wait(unp_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_ops)) { ok = false; break; }
                        if (!PAIR && pre_left > 0) {  // (these were expanded before their activations had been asked for)
                            --pre_left;
                            // (timed in the diagnostic build: the clock reads cost a short call up to 2 %, 1500 x 512 -> 512 10.05 -> 10.28 us)
                            if (!(kTraceBuild ? timed_wait(full_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_ops)
                                              : mbar_wait(full_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA))) { ok = false; break; }
                        }
                        if (lane == 0) { if (kb == 0) TRACE_CLK(p.status, 16); if (kb == 4) TRACE_CLK(p.status, 17); if (kb == p.num_kb - 1) TRACE_CLK(p.status, 18); }
                        tc_fence_after_sync();
                        const uint32_t a_lo = desc_lo0 + s * (STAGE_BYTES >> 4), b_lo = a_lo + (AC_BYTES >> 4);
#pragma unroll
                        for (int gi = 0; gi < GPK; ++gi) {
                            if (gi < groups_left) {
                                if (!timed_wait(tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_tempty) ||
                                    (PAIR && !timed_wait(peer_tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_tempty))) { ok = false; break; }
                                tc_fence_after_sync();
                                if (elect_one()) {
#pragma unroll
                                    for (int k = 0; k < MMA_PER_G * (ROWS == TALL ? 2 : 1); ++k) {
                                        const int kk = gi * MMA_PER_G + k % MMA_PER_G;  // 32-byte step inside the 128-byte row
                                        const int half = k / MMA_PER_G;                 // (TALL: the second 128 token rows)
                                        const uint32_t d = tmem_base + b * BUF_COLS + half * BN;
                                        const uint64_t ad = desc(a_lo + half * (A_BYTES >> 4) + 2 * kk), bd = desc(b_lo + 2 * kk);
                                        const uint32_t acc = k % MMA_PER_G != 0;
                                        if constexpr (PAIR && kI8Path)
                                            umma_i8_pair(d, ad, bd, idesc_i8, acc);
                                        else if constexpr (PAIR)
                                            umma_f8f6f4_pair(d, ad, bd, idesc_f8, acc);
                                        else if constexpr (kI8Path)
                                            umma_i8(d, ad, bd, idesc_i8, acc);
                                        else
                                            umma_f8f6f4(d, ad, bd, idesc_f8, acc);
                                    }
                                    commit(tfull_bar(b));
                                }
                                if (++b == NBUF) { b = 0; bph ^= 1; }
                            }
                        }
                        if (!ok) break;
                        groups_left -= GPK;
                        if (elect_one()) commit(empty_bar(s));
                        if (++s == STAGES) { s = 0; ph ^= 1; }
                    }
                    if (!ok) break;
                    // rank-r bf16 branch: one more accumulator tile, fp32
                    if (!mbar_wait(tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA) ||
                        (PAIR && !mbar_wait(peer_tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA))) { ok = false; break; }
                    tc_fence_after_sync();
                    for (int lr = 0; lr < p.lr_chunks; ++lr) {
                        if (!mbar_wait(unp_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA)) { ok = false; break; }
                        tc_fence_after_sync();
                        const uint32_t a_lo = desc_lo0 + s * (STAGE_BYTES >> 4), b_lo = a_lo + (AC_BYTES >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const uint32_t d = tmem_base + b * BUF_COLS;
                                if constexpr (PAIR) umma_bf16_pair(d, desc(a_lo + 2 * k), desc(b_lo + 2 * k), idesc_bf, (lr | k) != 0);
                                else umma_bf16(d, desc(a_lo + 2 * k), desc(b_lo + 2 * k), idesc_bf, (lr | k) != 0);
                                if (ROWS == TALL) umma_bf16(d + BN, desc(a_lo + (A_BYTES >> 4) + 2 * k), desc(b_lo + 2 * k), idesc_bf, (lr | k) != 0);
                            }
                            commit(empty_bar(s));
                        }
                        if (++s == STAGES) { s = 0; ph ^= 1; }
                    }
                    if (!ok) break;
                    if (elect_one()) commit(tfull_bar(b));
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
            const int u = threadIdx.x - 64;  // 0..63
            RingPos<STAGES> at;
            long long w_full = 0;
            bool ok = true;
            for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                const int items = p.num_kb + p.lr_chunks;
                for (int i = 0; i < items; ++i, at.next()) {
                    const uint32_t s = at.s;
                    // (before the first wait on what the previous kernel leaves: how long that one runs is no part of a bounded wait, nor of w_full)
                    if (!PAIR && at.it == static_cast<uint32_t>(pre)) grid_dependency_wait();
                    // A barrier is waited on by its phase's parity, and of a stage expanded early this warp has not seen the activations land: they have when
                    // the stage's MMAs are done.  (Not a wait for the landing itself: the barrier may be two phases on by now.)
                    if (at.it - STAGES < static_cast<uint32_t>(pre) && !mbar_wait(empty_bar(s), at.ph ^ 1, abort_flag, p.status, DEV_TIMEOUT_UNPACK)) { ok = false; break; }
                    ok = timed_wait(at.it < static_cast<uint32_t>(pre) ? pre_bar(s) : full_bar(s), at.ph, abort_flag, p.status, DEV_TIMEOUT_UNPACK, w_full);
                    if (!ok) break;
                    if (at.it == 0 && u == 0) TRACE_CLK(p.status, 14);
                    if (i < p.num_kb) {
                        // 16-byte piece idx = u + 64 j of the packed tile: row = idx/4 = u/4 + 16 j, piece c = u%4.
                        // The swizzle phase row%8 = (u/4)%8 and the piece do not depend on j, so every address is
                        // a per-thread base plus a compile-time offset.
                        uint8_t* st = smem_gen + s * STAGE_BYTES;
                        const uint4* src = reinterpret_cast<const uint4*>(st + AC_BYTES + BU_BYTES) + u;
                        const int c = u & 3, sw = (u >> 2) & 7;
                        uint8_t* d0 = st + AC_BYTES + (u >> 2) * 128 + (((2 * c) ^ sw) << 4);
                        uint8_t* d1 = st + AC_BYTES + (u >> 2) * 128 + (((2 * c + 1) ^ sw) << 4);
                        // The loads of a batch are issued before any of its stores: the compiler cannot prove that the
                        // staging buffer and the operand tile do not overlap, so a load written after a store would wait
                        // for it and the whole unpack would run as one dependent chain.
                        constexpr int PIECES = (P::WROWS * 4) / 64, BATCH = PIECES % 8 == 0 ? 8 : 4;
#pragma unroll
                        for (int jb = 0; jb < PIECES; jb += BATCH) {
                            uint4 pk[BATCH];
#pragma unroll
                            for (int j = 0; j < BATCH; ++j) pk[j] = src[64 * (jb + j)];
#pragma unroll
                            for (int j = 0; j < BATCH; ++j) {
                                // a word holds codes k..k+3 in bits 7, 2..0 of its bytes and codes k+4..k+7 four bit
                                // positions further up, wrapping around (see prepare.cu): mask, rotate, mask
                                uint4 o0, o1;
                                o0.x = code_bytes(pk[j].x & kSignMag); o0.y = code_bytes(__funnelshift_r(pk[j].x, pk[j].x, 4) & kSignMag);
                                o0.z = code_bytes(pk[j].y & kSignMag); o0.w = code_bytes(__funnelshift_r(pk[j].y, pk[j].y, 4) & kSignMag);
                                o1.x = code_bytes(pk[j].z & kSignMag); o1.y = code_bytes(__funnelshift_r(pk[j].z, pk[j].z, 4) & kSignMag);
                                o1.z = code_bytes(pk[j].w & kSignMag); o1.w = code_bytes(__funnelshift_r(pk[j].w, pk[j].w, 4) & kSignMag);
                                *reinterpret_cast<uint4*>(d0 + (jb + j) * 2048) = o0;  // 16 rows of 128 bytes further down
                                *reinterpret_cast<uint4*>(d1 + (jb + j) * 2048) = o1;
                            }
                        }
                        fence_proxy_async_smem();  // generic-proxy writes -> visible to the tensor core
                    }
                    // each thread signs off its own writes (a warp-wide barrier followed by one lane's arrival costs about
                    // a hundred cycles more on this part than 32 arrivals)
                    if constexpr (PAIR) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(map_to_cta(unp_bar(s), 0));
                    } else {
                        mbar_arrive(unp_bar(s));
                    }
                    if (at.it == 0 && u == 0) TRACE_CLK(p.status, 15);
                }
            }
            grid_dependency_wait();
            if (u == 0) flush_wait(p.status, WS_UNPACK_FULL, w_full);
        }
    } else {
        reg_alloc<P::EPI_REGS>();
        // ------------------------------------------------------------ epilogue (warps 4..11)
        // A warp owns 32 token rows (its TMEM lane quadrant) x BN/2 columns.  The accumulators are read with the
        // 16x256b shape: a thread then holds 4 rows (l/4 + 8 i) x the column pairs 2 (l%4) + {0, 1} of every block
        // of 8 columns, so one load of weight scales serves four rows (with the 32x32b shape, one row per thread,
        // every thread would need all 128 column scales of every group and the shared-memory pipe, not the FMA
        // pipe, would bound the kernel).  A chunk is 32 columns: TMEM lanes 0..15 and 16..31 of the quadrant, 32 values
        // per thread (see request_chunk), and the 8 weight scales of the thread's columns, which the layer stores
        // side by side (see wscale_index in common.h), in two 16-byte loads.
        //
        // The accumulator tiles of an output tile (one per K-group, then the rank-r one) are one stream: before the last chunk
        // of a tile is folded in, the next tile is waited for (it is there in the steady state: the MMAs of a group take a third
        // of the rescale) and its first chunk requested, so that neither the hand-over nor the first tensor-memory round trip is
        // paid between groups.
        const int q = warp & 3;
        const int half = (warp - 4) >> 2;
        const int lr4 = lane >> 2;        // row inside a group of 8
        const int lc2 = (lane & 3) * 2;   // first of this thread's two columns inside a block of 8
        uint32_t sc_off = 0;              // the current group's scale record
        long long w_tfull = 0;
        const long long t_epi = clock64();
        const int cta_row = (ROWS == TALL ? half * BM : 0) + q * 32 + lr4, tile_col = ROWS == TALL ? 0 : half * HB;  // this thread's first row, warp's first column
        const uint32_t taddr0 = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + half * HB;
        // The accumulator tile read next (its tensor-memory address and its "full" barrier, the "empty" one lies a fixed distance behind it),
        // that barrier's parity and the next tile's.
        uint32_t tcur = taddr0, bcur = tfull_bar(0), pcur = 0, pnxt = 0;
        auto tnext = [&]() { return NBUF == 2 ? 2 * taddr0 + BUF_COLS - tcur : tcur == taddr0 + (NBUF - 1) * BUF_COLS ? taddr0 : tcur + BUF_COLS; };
        auto bnext = [&]() { return NBUF == 2 ? 2 * tfull_bar(0) + 8u - bcur : bcur == tfull_bar(NBUF - 1) ? tfull_bar(0) : bcur + 8u; };
        auto advance = [&](uint32_t t, uint32_t b) {
            tcur = t;
            bcur = b;
            const uint32_t p1 = pcur;
            pcur = pnxt;
            // the tile after the next one: two tiles, the one just left, a phase later; four, a phase later than the next one where that is the last
            pnxt = NBUF == 2 ? p1 ^ 1 : b == tfull_bar(NBUF - 1) ? pnxt ^ 1 : pnxt;
        };
        const uint8_t* sw_base = smem_gen + STAGES * STAGE_BYTES + 4 * (tile_col + 4 * lc2);
        const uint8_t* sx_base = smem_gen + STAGES * STAGE_BYTES + SC_SW_BYTES + 4 * cta_row;
        // (worked out where they are needed, not held in registers across the groups)
        auto first_row = [&](int tile) { return tile_row(tile) + cta_row; };  // this thread's rows: first_row + 8 i, i = 0..3
        auto first_col = [&](int tile) { return (tile / num_m_blocks) * BN + tile_col; };
        // No vote after a wait: the warp is converged there, so the barrier test, the abort flag and the clock are read
        // by one instruction for all lanes and every lane gets the same answer.
        bool ok = true;
        uint32_t raw[2][32];  // [0..15]: TMEM lanes 0..15 of the quadrant (rows i = 0, 1), [16..31]: lanes 16..31
        auto request_chunk = [&](uint32_t tile_addr, int c, uint32_t* dst) {
            // 32 columns move in 32 cycles as two .x2 loads and in 64 as one .x4, which is half the instructions.  Measured on 18 layers, .x2 is
            // ahead by up to 4 %, except in 128-column tiles with groups of 128, where .x4 is by 1 to 2 %.  .x2 / .x4 in us, 4608 -> 1152
            // at 4096 tokens: 256 columns 91.5 / 92.4 (groups of 64), 64.2 / 65.3 (of 128); 128 columns 55.7 / 55.9, 39.7 / 39.0.
            const uint32_t t = tile_addr + c * 32;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if constexpr (BN == 128 && G == 128) {
                    tmem_ld_16x256b_x4(t + (static_cast<uint32_t>(h) << 20), dst + 16 * h);
                } else {
                    tmem_ld_16x256b_x2(t + (static_cast<uint32_t>(h) << 20), dst + 16 * h);
                    tmem_ld_16x256b_x2(t + (static_cast<uint32_t>(h) << 20) + 16, dst + 16 * h + 8);
                }
            }
        };
        auto release_tile = [&]() {  // every tcgen05.ld of this thread on the current tile has completed
            tc_fence_before_sync();
            mbar_arrive(bcur + (tempty_bar(0) - tfull_bar(0)));  // all lanes arrive (see the unpack warps' note on the cost of electing one)
        };
        for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
            uint64_t acc2[HB / 2];  // two adjacent columns per 64-bit register: [(block of 8 columns) * 4 + row i]
#pragma unroll
            for (int j = 0; j < HB / 2; ++j) acc2[j] = 0ull;

            // first accumulator tile of this output tile (its scales landed with the operands it was made from)
            ok = timed_wait(bcur, pcur, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_tfull);
            if (!ok) break;
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 20);
            tc_fence_after_sync();
            request_chunk(tcur, 0, raw[0]);

            for (int g = 0; g < p.n_g; ++g) {
                if (warp == 4 && lane == 0 && g == 8) TRACE_CLK(p.status, 21);
                const float* s_sx = reinterpret_cast<const float*>(sx_base + sc_off);
                const ulonglong2* swp = reinterpret_cast<const ulonglong2*>(sw_base + sc_off);
                sc_off = sc_off == (SC_SLOTS - 1) * SC_BYTES ? 0 : sc_off + SC_BYTES;
                // the accumulator holds S = 2^-18 P (integer-path build: P as int32, and 2^-18 goes into the token scale)
                uint64_t sx2[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float sx = s_sx[8 * i] * (kI8Path ? 1.0f / kWScaleFold : 1.0f);
                    sx2[i] = pack_f32x2(sx, sx);
                }
                const uint32_t tn = tnext(), bn = bnext();  // what comes after this tile: the next group's, or the rank-r tile
#pragma unroll
                for (int c = 0; c < CHUNKS; ++c) {
                    uint32_t (&cur)[32] = raw[c & 1];
                    // this chunk's weight scales, two adjacent columns per 64-bit register: requested before the wait so
                    // that their latency hides behind it
                    uint64_t w2[4];
                    if constexpr (!kPartials) {
                        const ulonglong2 wa = swp[c * 8], wb = swp[c * 8 + 1];
                        w2[0] = wa.x; w2[1] = wa.y; w2[2] = wb.x; w2[3] = wb.y;
                    }
                    tmem_ld_wait();  // waits for every outstanding load, hence a look-ahead of one chunk
                    tmem_ld_fence(cur);
                    if constexpr (kI8Path) {
#pragma unroll
                        for (int i = 0; i < 32; ++i) cur[i] = __float_as_uint(__int2float_rn(static_cast<int>(cur[i])));  // |P| < 2^24: exact
                    }
                    if (c < CHUNKS - 1) {
                        request_chunk(tcur, c + 1, raw[(c + 1) & 1]);
                    } else {
                        // the whole tile is in registers: hand it back to the MMA warp, and request the next one's first chunk
                        release_tile();
                        ok = timed_wait(bn, pnxt, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_tfull);
                        if (!ok) break;
                        tc_fence_after_sync();
                        request_chunk(tn, 0, raw[0]);  // CHUNKS is even: the last chunk sits in raw[1]
                    }
                    if constexpr (kPartials) {
                        // unit scales here: 2^18 S = P, an integer
                        const int rbase = first_row(tile), colbase = first_col(tile);
#pragma unroll
                        for (int i = 0; i < 4; ++i)
#pragma unroll
                            for (int cb = 0; cb < 4; ++cb) {
                                const int pidx = 16 * (i >> 1) + 4 * cb + 2 * (i & 1);
                                const int row = rbase + 8 * i;
                                const int col = colbase + c * 32 + cb * 8 + lc2;
                                if (row < p.M && col < p.N)
                                    *reinterpret_cast<int2*>(p.partials + (static_cast<size_t>(g) * p.M + row) * p.N + col) =
                                        make_int2(__float2int_rn(__uint_as_float(cur[pidx]) * kAccUnit),
                                                  __float2int_rn(__uint_as_float(cur[pidx + 1]) * kAccUnit));
                            }
                    } else {
                        // The scale of an element is t = s_x * (2^18 s_w): two bf16-valued factors (and a power of two), so
                        // the fp32 product is EXACT.  It is formed for two adjacent columns at a time with one packed
                        // multiply whose operands are 64-bit registers as they come (the pair of column scales straight
                        // from a shared-memory load, the token's scale duplicated once per group), so no register moves
                        // are spent on packing; then acc = fma(S, t, acc), again packed (the accumulator's two adjacent
                        // columns are consecutive registers of the tensor-memory load): one rounding per element and group,
                        // two instructions per two elements.
#pragma unroll
                        for (int cb = 0; cb < 4; ++cb)
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const int pidx = 16 * (i >> 1) + 4 * cb + 2 * (i & 1);
                                const int a = (c * 4 + cb) * 4 + i;
                                acc2[a] = fma_f32x2(pack_u32x2(cur[pidx], cur[pidx + 1]), mul_f32x2(w2[cb], sx2[i]), acc2[a]);
                            }
                    }
                }
                if (!ok) break;
                advance(tn, bn);
            }
            if (!ok) break;
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 22);
            // rank-r branch: an fp32 tile whose first chunk is already on its way
#pragma unroll
            for (int c = 0; c < CHUNKS; ++c) {
                uint32_t (&cur)[32] = raw[c & 1];
                tmem_ld_wait();
                tmem_ld_fence(cur);
                if (c < CHUNKS - 1) request_chunk(tcur, c + 1, raw[(c + 1) & 1]);
                else release_tile();
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int cb = 0; cb < 4; ++cb) {
                        const int pidx = 16 * (i >> 1) + 4 * cb + 2 * (i & 1);
                        const int a = (c * 4 + cb) * 4 + i;
                        acc2[a] = add_f32x2(acc2[a], pack_u32x2(cur[pidx], cur[pidx + 1]));
                    }
            }
            advance(tnext(), bnext());
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 23);
            if constexpr (!kPartials) {
                // A lane holds 2 of the 8 columns of every block; four blocks are transposed inside the quad of lanes
                // (two exchange steps) so that each lane ends up with all 8 columns = 16 bytes of one block and the
                // warp writes 64 contiguous bytes per row.
                const int j = lane & 3;
                const int rbase = first_row(tile), colbase = first_col(tile);
#pragma unroll
                for (int m = 0; m < CHUNKS; ++m) {
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
    if (warp == 1 && lane == 0 && crank == 0 && *abort_flag != 0) umma_drain<PAIR>(bar_base + 8u * (3 * STAGES + 8));  // a wait gave up: let issued MMAs finish first
    tc_fence_before_sync();
    if constexpr (PAIR) cluster_sync_all();  // neither CTA leaves while the other may still read its operands or signal its barriers
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after_sync();
        if constexpr (PAIR) tmem_dealloc_pair(tmem_base, 512);
        else tmem_dealloc(tmem_base, 512);
    }
}

template <int BN, Rows ROWS = ONE>
static dirotq_status_t launch_w4a4_gemm_bn(const dirotq_layer* L, const GemmArgs& a, cudaStream_t stream) {
    using P = Plan<BN, ROWS>;
    constexpr bool PAIR = ROWS == PAIRED;
    const Geometry& g = L->geo;
    CUtensorMap tmap_codes, tmap_xscale, tmap_xh;
    dirotq_status_t st;
    st = encode_tmap_2d(&tmap_codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a.codes, (uint64_t)g.K_lp, (uint64_t)a.M,
                        (uint64_t)g.K_lp, BKC, ROWS == ONE ? box_rows(a.M) : BM, CU_TENSOR_MAP_SWIZZLE_128B);
    if (st != DIROTQ_OK) return st;
    st = encode_tmap_2d(&tmap_xscale, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.xscale, (uint64_t)a.ldm, (uint64_t)g.n_g,
                        (uint64_t)a.ldm * 4, P::CTA_ROWS, 1, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (st != DIROTQ_OK) return st;
    st = encode_tmap_2d(&tmap_xh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.xh, (uint64_t)g.r_pad, (uint64_t)a.M,
                        (uint64_t)g.r_pad * 2, 64, ROWS == ONE ? box_rows(a.M) : BM, CU_TENSOR_MAP_SWIZZLE_128B);
    if (st != DIROTQ_OK) return st;

    GemmKernelParams p;
    p.M = a.M; p.N = g.N; p.n_g = g.n_g;
    p.num_kb = (g.K_lp + BKC - 1) / BKC;
    p.lr_chunks = g.r_pad / 64;
    p.bias = reinterpret_cast<const float*>(L->blob + L->lay.off_bias);
    p.y = a.y; p.partials = a.partials; p.status = a.status; p.early_weights = a.early_weights; p.x_rows = ROWS == ONE ? box_rows(a.M) : BM;

    constexpr int CTAS = PAIR ? 2 : 1;
    const int num_tiles = ((a.M + P::TILE_ROWS - 1) / P::TILE_ROWS) * ((g.N + BN - 1) / BN), slots = sm_count(L->device) / CTAS;
    const int grid = CTAS * (num_tiles < slots ? num_tiles : slots);
    using KernelFn = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap,
                              const CUtensorMap, const CUtensorMap, const GemmKernelParams);
    KernelFn kern;
    const bool dbg = a.partials != nullptr;
    if constexpr (ROWS != ONE) {  // (the debug entry's group sums come from the other plans)
        kern = g.G == 64 ? w4a4_gemm_kernel<64, false, BN, ROWS> : w4a4_gemm_kernel<128, false, BN, ROWS>;
    } else {
        if (g.G == 64) kern = dbg ? w4a4_gemm_kernel<64, true, BN, ONE> : w4a4_gemm_kernel<64, false, BN, ONE>;
        else           kern = dbg ? w4a4_gemm_kernel<128, true, BN, ONE> : w4a4_gemm_kernel<128, false, BN, ONE>;
    }
    static SmemOptIn<4> opt_in;  // one per instantiation of this launcher, i.e. per tile width
    const int vi = (g.G == 64 ? 0 : 2) + (dbg ? 1 : 0);
    if (!opt_in.ensure(kern, vi, L->device, P::SMEM_BYTES)) return DIROTQ_ERR_CUDA;
    auto launch = [&](const auto&... args) {
        return PAIR ? launch_kernel_pairs(kern, grid, P::THREADS, P::SMEM_BYTES, stream, true, args...)
                    : launch_kernel(kern, grid, P::THREADS, P::SMEM_BYTES, stream, true, args...);
    };
    const cudaError_t err = launch(tmap_codes, P::WROWS == 128 ? L->tmap_wpacked128 : P::WROWS == 192 ? L->tmap_wpacked192 : L->tmap_wpacked,
                                   BN == 128 ? L->tmap_wscale128 : BN == 192 ? L->tmap_wscale192 : L->tmap_wscale, tmap_xscale, tmap_xh,
                                   P::WROWS == 128 ? L->tmap_wh128 : P::WROWS == 192 ? L->tmap_wh192 : L->tmap_wh, p);
    return err == cudaSuccess ? DIROTQ_OK : DIROTQ_ERR_CUDA;
}

}  // namespace

static std::atomic<int> g_forced_plan{0};  // 0: chosen per call

dirotq_status_t set_w4a4_tile_columns(int columns) {
    const int plan = w4a4_forced_plan(columns);
    if (plan < 0) return DIROTQ_ERR_INVALID_ARG;
    g_forced_plan.store(plan);
    return DIROTQ_OK;
}

dirotq_status_t launch_w4a4_gemm(const dirotq_layer* L, const GemmArgs& a, cudaStream_t stream) {
    const int forced = g_forced_plan.load();
    const int plan = forced ? forced : choose_w4a4_plan(a.M, L->geo.N, L->geo.K_lp, L->geo.G, sm_count(L->device));
    if (a.partials == nullptr && plan <= 66) return launch_w4a4_narrow(L, a, plan == 32 && L->geo.G == 64 ? 32 : 64, plan == 66, stream);
    if (plan == 258 && a.partials == nullptr) return launch_w4a4_gemm_bn<256, PAIRED>(L, a, stream);
    if (plan == 130 && a.partials == nullptr) return launch_w4a4_gemm_bn<128, TALL>(L, a, stream);
    if (plan == 192) return launch_w4a4_gemm_bn<192>(L, a, stream);
    return plan >= 256 ? launch_w4a4_gemm_bn<256>(L, a, stream) : launch_w4a4_gemm_bn<128>(L, a, stream);
}

}  // namespace dirotq
