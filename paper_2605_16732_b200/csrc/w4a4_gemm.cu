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
// Tiles of 256, 128 or (on request) 192 columns here; w4a4_narrow.cu has the same computation in 64-column tiles.
//
// CTA pairs (PAIR; 256 token rows x 256 columns per cluster of two, tcgen05.mma.cta_group::2): each CTA loads its own activation codes and
// loads AND expands half of the tile's weights.  A K-group of a 128 x 256 tile keeps the schedulers of an SM busy for most of its time (the
// rescale's packed multiply and multiply-add take two issue cycles each: 660 of 1125 cycles), so what a pair saves is
// what the expansion takes from them and from shared memory: half.  4608 x 3072 -> 9216, us alone: groups of 64 278 -> 266, of 128 190 -> 164
// (there the two expanding warps had no time left: 1430 of 1509 cycles per k-block).
//
// Roles (384 threads = 3 warpgroups):
//   warpgroup 0: warp 0 TMA producer, warp 1 MMA issuer + TMEM owner, warps 2-3 nibble -> byte unpack
//   warpgroups 1-2: epilogue; warp%4 selects the TMEM lane quadrant (token rows), the warpgroup
//                   selects the half of the tile's columns.
#include "w4a4.cuh"

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
template <int BN, bool PAIR = false>
struct Plan {
    static constexpr int EPI_WG = BN == 192 ? 3 : 2;  // epilogue warpgroups
    static constexpr int EPI_WARPS = 4 * EPI_WG;
    static constexpr int THREADS = 128 + 128 * EPI_WG;
    static constexpr int EPI_REGS = EPI_WG == 3 ? 152 : 216;  // setmaxnreg budgets: 128 * AUX + 128 * EPI_WG * EPI <= 65536
    static constexpr int AUX_REGS = EPI_WG == 3 ? 56 : 64;
    static constexpr int SC_SLOTS = BN == 192 ? 6 : 8;
    static constexpr int STAGES = PAIR ? 5 : BN == 256 ? 3 : BN == 192 ? 4 : 5;
    static constexpr int WROWS = PAIR ? BN / 2 : BN;  // weight rows this CTA loads and expands
    static constexpr int BU_BYTES = WROWS * BKC;      // unpacked weight codes / bf16 W~_h chunk (32 KB at BN = 256)
    static constexpr int BP_BYTES = WROWS * BKC / 2;  // packed weight codes (TMA staging)
    static constexpr int STAGE_BYTES = A_BYTES + BU_BYTES + BP_BYTES;  // 64 KB / 40 KB
    static constexpr int SC_SW_BYTES = 2 * BN * 4;    // up to two groups per k-block
    static constexpr int SC_SX_BYTES = 2 * BM * 4;    // activation scales of up to two groups
    static constexpr int SC_BYTES = SC_SW_BYTES + SC_SX_BYTES;  // 3 KB / 2 KB
    static constexpr int BAR_OFFSET = STAGES * STAGE_BYTES + SC_SLOTS * SC_BYTES;
    static constexpr int SMEM_BYTES = BAR_OFFSET + 512 + 1024;
};
static_assert(Plan<256>::SMEM_BYTES <= 232448 && Plan<256, true>::SMEM_BYTES <= 232448 && Plan<192>::SMEM_BYTES <= 232448 && Plan<128>::SMEM_BYTES <= 232448, "shared memory plan too large");
static_assert(Plan<128>::STAGE_BYTES % 1024 == 0 && Plan<128>::SC_BYTES % 128 == 0, "tile alignment");
static_assert(Plan<192>::STAGE_BYTES % 1024 == 0 && Plan<192>::SC_BYTES % 128 == 0, "tile alignment");
static_assert(8 * (3 * Plan<256, true>::STAGES + 2 * 8 + 11) <= 400 && 8 * (3 * Plan<128>::STAGES + 2 * 8 + 9) <= 400 && 8 * (3 * Plan<192>::STAGES + 2 * 6 + 9) <= 400,
              "barriers end below the words at +400");

template <int G, bool kPartials, int BN, bool PAIR>
__global__ void __launch_bounds__(Plan<BN, PAIR>::THREADS, 1)
w4a4_gemm_kernel(const __grid_constant__ CUtensorMap tmap_codes, const __grid_constant__ CUtensorMap tmap_wpacked,
                 const __grid_constant__ CUtensorMap tmap_wscale, const __grid_constant__ CUtensorMap tmap_xscale,
                 const __grid_constant__ CUtensorMap tmap_xh, const __grid_constant__ CUtensorMap tmap_wh,
                 const GemmKernelParams p) {
    using P = Plan<BN, PAIR>;
    constexpr int STAGES = P::STAGES, STAGE_BYTES = P::STAGE_BYTES, BU_BYTES = P::BU_BYTES, BP_BYTES = P::BP_BYTES;
    constexpr int SC_SW_BYTES = P::SC_SW_BYTES, SC_BYTES = P::SC_BYTES, BAR_OFFSET = P::BAR_OFFSET;
    constexpr int SC_SLOTS = P::SC_SLOTS, NUM_EPI_WARPS = P::EPI_WARPS;
    constexpr int HB = BN / P::EPI_WG;  // columns per epilogue warp: the warpgroup selects the slice of the tile
    constexpr int CHUNKS = HB / 32;    // 32-column chunks per epilogue warp and accumulator tile
    constexpr int GPK = BKC / G;       // groups per k-block: 2 (G = 64) or 1 (G = 128)
    constexpr int MMA_PER_G = G / 32;  // 8-bit MMA instructions (K = 32) per group
    constexpr int NBUF = 512 / BN;     // accumulator tiles in tensor memory: 2 of 256 columns, 4 of 128 (the barrier map has four slots)

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sc_base = smem_base + STAGES * STAGE_BYTES;
    const uint32_t bar_base = smem_base + BAR_OFFSET;
    // barriers: full[S], unpacked[S], empty[S], sc_full[SC], sc_empty[SC], tmem_full[NBUF], tmem_empty[NBUF]
    auto full_bar = [&](int s) { return bar_base + 8u * s; };
    auto unp_bar = [&](int s) { return bar_base + 8u * (STAGES + s); };
    auto empty_bar = [&](int s) { return bar_base + 8u * (2 * STAGES + s); };
    auto scfull_bar = [&](int s) { return bar_base + 8u * (3 * STAGES + s); };
    auto scempty_bar = [&](int s) { return bar_base + 8u * (3 * STAGES + SC_SLOTS + s); };
    auto tfull_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + 2 * SC_SLOTS + a); };
    auto tempty_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + 2 * SC_SLOTS + 4 + a); };
    auto peer_tempty_bar = [&](int a) { return bar_base + 8u * (3 * STAGES + 2 * SC_SLOTS + 9 + a); };  // pairs: in the leader, the other CTA's
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + BAR_OFFSET + 400);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + BAR_OFFSET + 404);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    // Trace build (TRACE_CLK): slot 9 entry, 10 set-up done, 11 previous grid ended, 12 / 13 producer has issued its first k-block /
    // everything, 14 / 15 first unpack warp sees / has expanded the first stage, 16 / 17 / 18 MMA warp starts the first / fifth / last
    // k-block, 19 it has committed the last tile, 20 first epilogue warp sees its first accumulator, 21 starts its ninth K-group, 22 has
    // folded in the last group, 23 the rank-r tile, 24 has stored its last outputs.
    if (threadIdx.x == 0) TRACE_CLK(p.status, 9);

    // a tile is BM token rows of one CTA, or of each CTA of a pair
    const uint32_t crank = PAIR ? cluster_ctarank() : 0u;
    constexpr int TILE_ROWS = PAIR ? 2 * BM : BM;
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
        }
        for (int s = 0; s < SC_SLOTS; ++s) {
            mbar_init(scfull_bar(s), 1);
            mbar_init(scempty_bar(s), NUM_EPI_WARPS * 32);
        }
        for (int a = 0; a < NBUF; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), NUM_EPI_WARPS * 32);
            if (PAIR) mbar_init(peer_tempty_bar(a), 1);
        }
        mbar_init(bar_base + 8u * (3 * STAGES + 2 * SC_SLOTS + 8), 1);  // spare: see umma_drain
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
    grid_dependency_wait();
    if (threadIdx.x == 0) TRACE_CLK(p.status, 11);
    // the next layer's first kernel may be scheduled as this grid's CTAs leave their SMs (it waits for this whole grid)
    grid_launch_dependents();

    if (warp < 4) {
        reg_dealloc<P::AUX_REGS>();

        if (warp == 0) {
            // -------------------------------------------------------- TMA producer
            // (the whole warp walks the loops and waits, one elected lane issues: counters, addresses and coordinates stay
            // warp-uniform, which shortens the chain of instructions per stage)
            {
                uint32_t it = 0, sc_it = 0;
                long long w_empty = 0;
                bool ok = true;
                for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                    const int m0 = tile_row(tile);
                    const int n0 = (tile / num_m_blocks) * BN, w0 = n0 + static_cast<int>(crank) * P::WROWS;
                    for (int kb = 0; kb < p.num_kb; ++kb, ++it, ++sc_it) {
                        const int s = it % STAGES;
                        if (!timed_wait(empty_bar(s), ((it / STAGES) & 1) ^ 1, abort_flag, p.status, DEV_TIMEOUT_PRODUCER, w_empty)) { ok = false; break; }
                        const uint32_t st = smem_base + s * STAGE_BYTES;
                        if (elect_one()) {
                            mbar_arrive_expect_tx(full_bar(s), A_BYTES + BP_BYTES);
                            tma_load_2d(st, &tmap_codes, full_bar(s), kb * BKC, m0);
                            tma_load_2d(st + A_BYTES + BU_BYTES, &tmap_wpacked, full_bar(s), kb * (BKC / 2), w0);
                        }
                        const int slot = sc_it % SC_SLOTS;
                        if (!mbar_wait(scempty_bar(slot), ((sc_it / SC_SLOTS) & 1) ^ 1, abort_flag, p.status, DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
                        const uint32_t sc = sc_base + slot * SC_BYTES;
                        if (elect_one()) {
                            mbar_arrive_expect_tx(scfull_bar(slot), GPK * (BN + BM) * 4);
                            tma_load_2d(sc, &tmap_wscale, scfull_bar(slot), n0, kb * GPK);
                            tma_load_2d(sc + SC_SW_BYTES, &tmap_xscale, scfull_bar(slot), m0, kb * GPK);
                            if (it == 0) TRACE_CLK(p.status, 12);
                        }
                    }
                    if (!ok) break;
                    for (int lr = 0; lr < p.lr_chunks; ++lr, ++it) {
                        const int s = it % STAGES;
                        if (!mbar_wait(empty_bar(s), ((it / STAGES) & 1) ^ 1, abort_flag, p.status, DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
                        const uint32_t st = smem_base + s * STAGE_BYTES;
                        if (elect_one()) {
                            mbar_arrive_expect_tx(full_bar(s), A_BYTES + BU_BYTES);
                            tma_load_2d(st, &tmap_xh, full_bar(s), lr * 64, m0);
                            tma_load_2d(st + A_BYTES, &tmap_wh, full_bar(s), lr * 64, w0);
                        }
                    }
                }
                if (lane == 0) TRACE_CLK(p.status, 13);
                if (lane == 0) flush_wait(p.status, WS_PROD_EMPTY, w_empty);
                if (!ok && lane == 0) {
                    const uint32_t first = it > STAGES ? it - STAGES : 0;
                    for (uint32_t j = first; j < it; ++j) {
                        const unsigned long long t0 = globaltimer_ns();
                        while (!mbar_try_wait(full_bar(j % STAGES), (j / STAGES) & 1) &&
                               globaltimer_ns() - t0 < 100000000ull) {}
                    }
                    const uint32_t sfirst = sc_it > SC_SLOTS ? sc_it - SC_SLOTS : 0;
                    for (uint32_t j = sfirst; j < sc_it; ++j) {
                        const unsigned long long t0 = globaltimer_ns();
                        while (!mbar_try_wait(scfull_bar(j % SC_SLOTS), (j / SC_SLOTS) & 1) &&
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
                constexpr uint32_t idesc_f8 = umma_idesc(1 /*f32*/, 0 /*E4M3*/, TILE_ROWS, BN);
                constexpr uint32_t idesc_i8 = umma_idesc(2 /*s32*/, 1 /*s8*/, TILE_ROWS, BN);  // integer-path build only
                constexpr uint32_t idesc_bf = umma_idesc(1 /*f32*/, 1 /*bf16*/, TILE_ROWS, BN);
                const uint64_t desc0 = umma_desc_sw128(smem_base);
                const uint32_t desc_hi = static_cast<uint32_t>(desc0 >> 32), desc_lo0 = static_cast<uint32_t>(desc0);
                auto desc = [&](uint32_t lo) { return (static_cast<uint64_t>(desc_hi) << 32) | lo; };
                auto commit = [&](uint32_t bar) {
                    if constexpr (PAIR) umma_commit_pair(bar, 3);  // the same barrier of both CTAs
                    else umma_commit(bar);
                };
                uint32_t s = 0, ph = 0;        // stage of the operand ring and its parity
                uint32_t b = 0, bph = 1;       // accumulator tile and the parity its "empty" barrier is waited with
                long long w_ops = 0, w_tempty = 0;
                const long long t_kernel = clock64();
                bool ok = true;
                for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                    int groups_left = p.n_g;
                    for (int kb = 0; ok && kb < p.num_kb; ++kb) {
                        // the unpack warps arrive after they have seen the stage's loads land (one barrier for both operands), so
                        // their barrier covers the activation codes as well
                        if (!timed_wait(unp_bar(s), ph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_ops)) { ok = false; break; }
                        if (lane == 0) { if (kb == 0) TRACE_CLK(p.status, 16); if (kb == 4) TRACE_CLK(p.status, 17); if (kb == p.num_kb - 1) TRACE_CLK(p.status, 18); }
                        tc_fence_after_sync();
                        const uint32_t a_lo = desc_lo0 + s * (STAGE_BYTES >> 4), b_lo = a_lo + (A_BYTES >> 4);
#pragma unroll
                        for (int gi = 0; gi < GPK; ++gi) {
                            if (gi < groups_left) {
                                if (!timed_wait(tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_tempty) ||
                                    (PAIR && !timed_wait(peer_tempty_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_MMA, w_tempty))) { ok = false; break; }
                                tc_fence_after_sync();
                                if (elect_one()) {
#pragma unroll
                                    for (int k = 0; k < MMA_PER_G; ++k) {
                                        const int kk = gi * MMA_PER_G + k;  // 32-byte step inside the 128-byte row
                                        if constexpr (PAIR && kI8Path)
                                            umma_i8_pair(tmem_base + b * BN, desc(a_lo + 2 * kk), desc(b_lo + 2 * kk), idesc_i8, k != 0);
                                        else if constexpr (PAIR)
                                            umma_f8f6f4_pair(tmem_base + b * BN, desc(a_lo + 2 * kk), desc(b_lo + 2 * kk), idesc_f8, k != 0);
                                        else if constexpr (kI8Path)
                                            umma_i8(tmem_base + b * BN, desc(a_lo + 2 * kk), desc(b_lo + 2 * kk), idesc_i8, k != 0);
                                        else
                                            umma_f8f6f4(tmem_base + b * BN, desc(a_lo + 2 * kk), desc(b_lo + 2 * kk), idesc_f8, k != 0);
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
                        const uint32_t a_lo = desc_lo0 + s * (STAGE_BYTES >> 4), b_lo = a_lo + (A_BYTES >> 4);
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                if constexpr (PAIR) umma_bf16_pair(tmem_base + b * BN, desc(a_lo + 2 * k), desc(b_lo + 2 * k), idesc_bf, (lr | k) != 0);
                                else umma_bf16(tmem_base + b * BN, desc(a_lo + 2 * k), desc(b_lo + 2 * k), idesc_bf, (lr | k) != 0);
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
            uint32_t it = 0;
            long long w_full = 0;
            bool ok = true;
            for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
                const int items = p.num_kb + p.lr_chunks;
                for (int i = 0; i < items; ++i, ++it) {
                    const int s = it % STAGES;
                    ok = timed_wait(full_bar(s), (it / STAGES) & 1, abort_flag, p.status, DEV_TIMEOUT_UNPACK, w_full);
                    if (!ok) break;
                    if (it == 0 && u == 0) TRACE_CLK(p.status, 14);
                    if (i < p.num_kb) {
                        // 16-byte piece idx = u + 64 j of the packed tile: row = idx/4 = u/4 + 16 j, piece c = u%4.
                        // The swizzle phase row%8 = (u/4)%8 and the piece do not depend on j, so every address is
                        // a per-thread base plus a compile-time offset.
                        uint8_t* st = smem_gen + s * STAGE_BYTES;
                        const uint4* src = reinterpret_cast<const uint4*>(st + A_BYTES + BU_BYTES) + u;
                        const int c = u & 3, sw = (u >> 2) & 7;
                        uint8_t* d0 = st + A_BYTES + (u >> 2) * 128 + (((2 * c) ^ sw) << 4);
                        uint8_t* d1 = st + A_BYTES + (u >> 2) * 128 + (((2 * c + 1) ^ sw) << 4);
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
                    if (it == 0 && u == 0) TRACE_CLK(p.status, 15);
                }
            }
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
        // The accumulator tiles of an output tile (one per K-group, then the rank-r one) are one stream: while the
        // last chunk of a tile is folded in, the next tile's barrier is tested (not waited for) and, if it has
        // completed, its first chunk is requested, so that in the steady state neither the hand-over nor the first
        // tensor-memory round trip is paid between groups.
        const int q = warp & 3;
        const int half = (warp - 4) >> 2;
        const int lr4 = lane >> 2;        // row inside a group of 8
        const int lc2 = (lane & 3) * 2;   // first of this thread's two columns inside a block of 8
        uint32_t b = 0, bph = 0;          // accumulator tile read next, parity its "full" barrier is waited with
        uint32_t slot = 0, sph = 0;       // scale slot of the current k-block, parity of its "full" barrier
        long long w_tfull = 0, w_sc = 0;
        const long long t_epi = clock64();
        const uint32_t taddr0 = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + half * HB;
        const float* sc0 = reinterpret_cast<const float*>(smem_gen + STAGES * STAGE_BYTES);
        // No vote after a wait: the warp is converged there, so the barrier test, the abort flag and the clock are read
        // by one instruction for all lanes and every lane gets the same answer.
        bool ok = true;
        uint32_t raw[2][32];  // [0..15]: TMEM lanes 0..15 of the quadrant (rows i = 0, 1), [16..31]: lanes 16..31
        auto request_chunk = [&](uint32_t buf, int c, uint32_t* dst) {
            // 32 columns move in 32 cycles as two .x2 loads and in 64 as one .x4, which is half the instructions.  Measured on 18 layers, .x2 is
            // ahead by up to 4 %, except in 128-column tiles with groups of 128, where .x4 is by 1 to 2 %.  .x2 / .x4 in us, 4608 -> 1152
            // at 4096 tokens: 256 columns 91.5 / 92.4 (groups of 64), 64.2 / 65.3 (of 128); 128 columns 55.7 / 55.9, 39.7 / 39.0.
            const uint32_t t = taddr0 + buf * BN + c * 32;
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
        auto release_tile = [&](uint32_t buf) {  // every tcgen05.ld of this thread on the tile has completed
            tc_fence_before_sync();
            mbar_arrive(tempty_bar(buf));  // all lanes arrive (see the unpack warps' note on the cost of electing one)
        };
        for (int tile = first_tile(); ok && tile < num_tiles; tile += tile_stride()) {
            const int m0 = tile_row(tile);
            const int n0 = (tile / num_m_blocks) * BN;
            const int rbase = m0 + q * 32 + lr4;  // this thread's rows: rbase + 8 i, i = 0..3
            const int colbase = n0 + half * HB;
            uint64_t acc2[HB / 2];  // two adjacent columns per 64-bit register: [(block of 8 columns) * 4 + row i]
#pragma unroll
            for (int j = 0; j < HB / 2; ++j) acc2[j] = 0ull;

            // first scales and first accumulator tile of this output tile
            ok = timed_wait(scfull_bar(slot), sph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_sc) &&
                 timed_wait(tfull_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_tfull);
            if (!ok) break;
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 20);
            tc_fence_after_sync();
            request_chunk(b, 0, raw[0]);

            for (int g = 0; g < p.n_g; ++g) {
                if (warp == 4 && lane == 0 && g == 8) TRACE_CLK(p.status, 21);
                const int gi = g & (GPK - 1);
                const bool last_of_kb = gi == GPK - 1 || g == p.n_g - 1;
                const float* s_sw = sc0 + slot * (SC_BYTES / 4);
                // the accumulator holds S = 2^-18 P (integer-path build: P as int32, and 2^-18 goes into the token scale)
                float sxv[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    sxv[i] = s_sw[2 * BN + gi * BM + q * 32 + lr4 + 8 * i] * (kI8Path ? 1.0f / kWScaleFold : 1.0f);
                uint64_t sx2[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) sx2[i] = pack_f32x2(sxv[i], sxv[i]);
                const ulonglong2* swp = reinterpret_cast<const ulonglong2*>(s_sw + gi * BN + half * HB + 4 * lc2);
                // what comes after this tile: the next group's, or the rank-r tile
                const uint32_t nb = b + 1 == NBUF ? 0 : b + 1, nbph = b + 1 == NBUF ? bph ^ 1 : bph;
                const uint32_t nslot = slot + 1 == SC_SLOTS ? 0 : slot + 1, nsph = slot + 1 == SC_SLOTS ? sph ^ 1 : sph;
                const bool new_scales = last_of_kb && g + 1 < p.n_g;
                bool ahead = false;
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
                        request_chunk(b, c + 1, raw[(c + 1) & 1]);
                    } else {
                        // the whole tile is in registers: hand it back to the MMA warp, and look at the next one
                        release_tile(b);
                        ahead = mbar_test_wait(tfull_bar(nb), nbph) && (!new_scales || mbar_test_wait(scfull_bar(nslot), nsph));
                        if (ahead) {
                            tc_fence_after_sync();
                            request_chunk(nb, 0, raw[0]);  // CHUNKS is even: the last chunk sits in raw[1]
                        }
                    }
                    if constexpr (kPartials) {
                        // unit scales here: 2^18 S = P, an integer
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
                if (last_of_kb) {
                    // this k-block's scales have all been read (the multiply-adds that consumed them were issued above)
                    mbar_arrive(scempty_bar(slot));
                    slot = nslot;
                    sph = nsph;
                }
                b = nb;
                bph = nbph;
                if (!ahead) {
                    if (new_scales) ok = timed_wait(scfull_bar(slot), sph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_sc);
                    ok = ok && timed_wait(tfull_bar(b), bph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE, w_tfull);
                    if (!ok) break;
                    tc_fence_after_sync();
                    request_chunk(b, 0, raw[0]);
                }
            }
            if (!ok) break;
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 22);
            // rank-r branch: an fp32 tile whose first chunk is already on its way
#pragma unroll
            for (int c = 0; c < CHUNKS; ++c) {
                uint32_t (&cur)[32] = raw[c & 1];
                tmem_ld_wait();
                tmem_ld_fence(cur);
                if (c < CHUNKS - 1) request_chunk(b, c + 1, raw[(c + 1) & 1]);
                else release_tile(b);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int cb = 0; cb < 4; ++cb) {
                        const int pidx = 16 * (i >> 1) + 4 * cb + 2 * (i & 1);
                        const int a = (c * 4 + cb) * 4 + i;
                        acc2[a] = add_f32x2(acc2[a], pack_u32x2(cur[pidx], cur[pidx + 1]));
                    }
            }
            if (++b == NBUF) { b = 0; bph ^= 1; }
            if (warp == 4 && lane == 0) TRACE_CLK(p.status, 23);
            if constexpr (!kPartials) {
                // A lane holds 2 of the 8 columns of every block; four blocks are transposed inside the quad of lanes
                // (two exchange steps) so that each lane ends up with all 8 columns = 16 bytes of one block and the
                // warp writes 64 contiguous bytes per row.
                const int j = lane & 3;
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
            flush_wait(p.status, WS_EPI_SCALES, w_sc);
            flush_wait(p.status, WS_EPI_TOTAL, clock64() - t_epi);
        }
    }

    // ---------------------------------------------------------------- teardown
    if (warp == 1 && lane == 0 && crank == 0 && *abort_flag != 0) umma_drain<PAIR>(bar_base + 8u * (3 * STAGES + 2 * SC_SLOTS + 8));  // a wait gave up: let issued MMAs finish first
    tc_fence_before_sync();
    if constexpr (PAIR) cluster_sync_all();  // neither CTA leaves while the other may still read its operands or signal its barriers
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after_sync();
        if constexpr (PAIR) tmem_dealloc_pair(tmem_base, 512);
        else tmem_dealloc(tmem_base, 512);
    }
}

template <int BN, bool PAIR = false>
static dirotq_status_t launch_w4a4_gemm_bn(const dirotq_layer* L, const GemmArgs& a, cudaStream_t stream) {
    const Geometry& g = L->geo;
    CUtensorMap tmap_codes, tmap_xscale, tmap_xh;
    dirotq_status_t st;
    st = encode_tmap_2d(&tmap_codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a.codes, (uint64_t)g.K_lp, (uint64_t)a.M,
                        (uint64_t)g.K_lp, BKC, BM, CU_TENSOR_MAP_SWIZZLE_128B);
    if (st != DIROTQ_OK) return st;
    st = encode_tmap_2d(&tmap_xscale, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.xscale, (uint64_t)a.ldm, (uint64_t)g.n_g,
                        (uint64_t)a.ldm * 4, BM, BKC / g.G, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (st != DIROTQ_OK) return st;
    st = encode_tmap_2d(&tmap_xh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.xh, (uint64_t)g.r_pad, (uint64_t)a.M,
                        (uint64_t)g.r_pad * 2, 64, BM, CU_TENSOR_MAP_SWIZZLE_128B);
    if (st != DIROTQ_OK) return st;

    GemmKernelParams p;
    p.M = a.M; p.N = g.N; p.n_g = g.n_g;
    p.num_kb = (g.K_lp + BKC - 1) / BKC;
    p.lr_chunks = g.r_pad / 64;
    p.bias = reinterpret_cast<const float*>(L->blob + L->lay.off_bias);
    p.y = a.y; p.partials = a.partials; p.status = a.status;

    using P = Plan<BN, PAIR>;
    constexpr int TILE_ROWS = PAIR ? 2 * BM : BM, CTAS = PAIR ? 2 : 1;
    const int num_tiles = ((a.M + TILE_ROWS - 1) / TILE_ROWS) * ((g.N + BN - 1) / BN), slots = sm_count(L->device) / CTAS;
    const int grid = CTAS * (num_tiles < slots ? num_tiles : slots);
    using KernelFn = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap,
                              const CUtensorMap, const CUtensorMap, const GemmKernelParams);
    KernelFn kern;
    const bool dbg = a.partials != nullptr;
    if constexpr (PAIR) {  // (the debug entry's group sums come from single CTAs)
        kern = g.G == 64 ? w4a4_gemm_kernel<64, false, BN, true> : w4a4_gemm_kernel<128, false, BN, true>;
    } else {
        if (g.G == 64) kern = dbg ? w4a4_gemm_kernel<64, true, BN, false> : w4a4_gemm_kernel<64, false, BN, false>;
        else           kern = dbg ? w4a4_gemm_kernel<128, true, BN, false> : w4a4_gemm_kernel<128, false, BN, false>;
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

static std::atomic<int> g_tile_columns{0};  // 0: chosen per call; 64 / 128 / 192 / 256: forced; 66: 64 columns, split plan where it applies

dirotq_status_t set_w4a4_tile_columns(int columns) {
    if (columns != 0 && columns != 64 && columns != 66 && columns != 128 && columns != 192 && columns != 256 && columns != 512) return DIROTQ_ERR_INVALID_ARG;
    g_tile_columns.store(columns);
    return DIROTQ_OK;
}

dirotq_status_t launch_w4a4_gemm(const dirotq_layer* L, const GemmArgs& a, cudaStream_t stream) {
    // The plan with the shortest schedule: turns of the SMs x what one tile of the plan costs.  Costs relative to a 256-column tile, from
    // the cycles per 128 codes of a tile: 2360, 1390 and 780 with groups of 64, 1600, 990 and 620 with groups of 128 (the
    // activation tile, the rank-r branch, the pipeline fill and the hand-overs are paid per tile whatever its width).
    // A turn of pair tiles takes 0.957 of a turn of 256-column tiles with groups of 64, 0.86 with groups of 128; a pair covers two row blocks, which can
    // cost it a turn (4173 x 3072 -> 12288: 12 turns against 11, 349 us against 339).
    const int forced = g_tile_columns.load(), sms = sm_count(L->device);
    const long m_blocks = (a.M + BM - 1) / BM;
    auto turns = [&](int columns) { return static_cast<double>((m_blocks * ((L->geo.N + columns - 1) / columns) + sms - 1) / sms); };
    const double c256 = turns(256), c128 = (L->geo.G == 64 ? 0.60 : 0.64) * turns(128), c64 = (L->geo.G == 64 ? 0.34 : 0.40) * turns(64);
    const double c512 = (L->geo.G == 64 ? 0.957 : 0.86) * static_cast<double>(((m_blocks + 1) / 2 * ((L->geo.N + 255) / 256) + sms / 2 - 1) / (sms / 2));
    const int plan = forced ? forced : c512 < c256 && c512 <= c128 && c512 <= c64 ? 512 : c64 <= c128 && c64 <= c256 ? 64 : c128 < c256 ? 128 : 256;
    if (a.partials == nullptr && (plan == 64 || plan == 66)) return launch_w4a4_narrow(L, a, plan == 66, stream);
    if (plan == 512 && a.partials == nullptr) return launch_w4a4_gemm_bn<256, true>(L, a, stream);
    if (plan == 192) return launch_w4a4_gemm_bn<192>(L, a, stream);
    return plan >= 256 ? launch_w4a4_gemm_bn<256>(L, a, stream) : launch_w4a4_gemm_bn<128>(L, a, stream);
}

}  // namespace dirotq
