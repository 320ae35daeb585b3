// W4A8 second kernel for calls with many token rows: the contraction of w4a8_gemm.cu in CTA pairs.
//
//   y[m,n] = bf16( s_x[m] s_w[n] P[m,n]  +  sum_{i<r} x~_h[m,i] W~_h[i,n]  +  bias[n] ),   P exact in int32
//
// Clusters of two CTAs (tcgen05.mma.cta_group::2): a pair owns 256 token rows x 256 output columns; each CTA loads its own 128 rows of
// activation codes, and loads AND expands half of the tile's weight rows, so an expanded weight serves 256 token rows.
// What paced single CTAs (w4a8_gemm.cu, there once with 256-column tiles too) is the path of the weights through shared memory:
// per 256 columns and k-block of 128 codes 24 KB arrive, the unpack reads 16 and writes 32 KB, the tensor core reads 48, in
// 1000 cycles where the MMAs need 512, with the load -> unpack -> MMA round trip spread over four stages.  Here it is 24 KB
// arriving, 8 + 16 for the expansion and 32 for the tensor core per CTA, on three rings with depths of their own (codes, packed
// weights, expanded weights), the expansion done by three teams of two warps that take k-blocks in turn (one team's turn is
// mostly waiting).  A k-block takes 650 cycles, of which the MMAs 512.  Second kernel, before -> after: 4608 x 3072 -> 9216 165 ->
// 100 us (2.6 POP/s), 1024 x 3072 -> 3072 17.7 -> 16.4, 2048 x 1152 -> 4608 16.9 -> 15.4.
// Ring slots and parities are carried along (a division by the ring depth per item and role cost more than it looks: 4096 x 4608 -> 1152 29.8 -> 22.5 us,
// 256 x 1152 -> 1152 8.0 -> 6.6).
// An output tile is two accumulator passes, the int32 one over K and the fp32 one of the rank-r branch, in two tensor-memory
// buffers; the epilogue warps take the first into registers while the second runs, so the next tile's MMAs start at once.
#include "common.h"
#include "ptx.cuh"

#include <cuda_bf16.h>

namespace dirotq {
namespace {

constexpr int BM = 128;
constexpr int BKC = 128;                 // codes per k-block
constexpr int NUM_THREADS = 512;
constexpr int TEAMS = 3, TEAM_WARPS = 2, NUM_EPI_WARPS = 8;

// Shared-memory plan for tiles of BN output columns: 256, or 128 where those would leave SMs idle.
template <int BN>
struct Plan {
    static constexpr int ROWS = BN / 2;  // weight rows of one CTA
    // ring depths: code tiles, packed weights, expanded weights
    static constexpr int NA = BN == 256 ? 6 : 8, NP = BN == 256 ? 6 : 8, NW = BN == 256 ? 3 : 5;
    // A barrier is waited on by its phase's parity, so whoever skips phases must know the one before last to be complete.  A team
    // that comes to item i has finished i - TEAMS, hence the MMAs of i - TEAMS - NW are done and everything up to there has
    // landed: NP >= NW + TEAMS and NW >= TEAMS.  The producer, which waits for an operand slot at rank-r items only, has a
    // code slot first: the MMAs of i - NA are done, so NA <= 2 NW.
    static_assert(NP >= NW + TEAMS && NW >= TEAMS && NA <= 2 * NW, "ring depths");
    static constexpr int A_BYTES = BM * BKC, W_BYTES = ROWS * BKC, P_BYTES = ROWS * BKC / 2;
    static constexpr int W_OFFSET = NA * A_BYTES, P_OFFSET = W_OFFSET + NW * W_BYTES, BAR_OFFSET = P_OFFSET + NP * P_BYTES;
    static constexpr int COL_OFFSET = BAR_OFFSET + 512;  // per epilogue warp: scale and bias of its BN / 2 columns
    static constexpr int COL_BYTES = BN / 2 * 8;
    static constexpr int STORE_OFFSET = (COL_OFFSET + NUM_EPI_WARPS * COL_BYTES + 1023) / 1024 * 1024;
    static constexpr int SMEM_BYTES = STORE_OFFSET + NUM_EPI_WARPS * 2048 + 1024;
    static_assert(8 * (2 * (NA + NP + NW) + 4) <= 448, "barriers end below the words at +448");
    static_assert(SMEM_BYTES <= 232448, "shared memory plan");
};

struct PairParams {
    int M, N, num_kb, lr_chunks;
    const float* xscale;     // [M]
    const float* wscale;     // [N]
    const float* bias;       // [N]
    int* status;
};

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {  // no arrival
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

template <int BN>
__global__ void __launch_bounds__(NUM_THREADS, 1)
w4a8_pair_kernel(const __grid_constant__ CUtensorMap tmap_codes, const __grid_constant__ CUtensorMap tmap_wpacked,
                 const __grid_constant__ CUtensorMap tmap_xh, const __grid_constant__ CUtensorMap tmap_wh, const __grid_constant__ CUtensorMap tmap_y, const PairParams p) {
    using P = Plan<BN>;
    constexpr int NA = P::NA, NP = P::NP, NW = P::NW, ROWS = P::ROWS, HB = BN / 2;
    constexpr int A_BYTES = P::A_BYTES, W_BYTES = P::W_BYTES, P_BYTES = P::P_BYTES, W_OFFSET = P::W_OFFSET, P_OFFSET = P::P_OFFSET;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t bar_base = smem_base + P::BAR_OFFSET;
    auto a_full = [&](uint32_t s) { return bar_base + 8u * s; };                     // leader: both CTAs' A tiles have landed
    auto a_empty = [&](uint32_t s) { return bar_base + 8u * (NA + s); };
    auto p_full = [&](uint32_t s) { return bar_base + 8u * (2 * NA + s); };          // this CTA's packed weights have landed
    auto p_empty = [&](uint32_t s) { return bar_base + 8u * (2 * NA + NP + s); };
    auto w_full = [&](uint32_t s) { return bar_base + 8u * (2 * NA + 2 * NP + s); };  // leader: both CTAs' weights are expanded
    auto w_empty = [&](uint32_t s) { return bar_base + 8u * (2 * NA + 2 * NP + NW + s); };
    auto tfull_bar = [&](uint32_t a) { return bar_base + 8u * (2 * (NA + NP + NW) + a); };
    auto tempty_bar = [&](uint32_t a) { return bar_base + 8u * (2 * (NA + NP + NW) + 2 + a); };
    const uint32_t spare_bar = bar_base + 456u;
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + P::BAR_OFFSET + 448);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + P::BAR_OFFSET + 452);

    const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;  // (the warp known to be uniform)
    // Trace build (TRACE_CLK), k-blocks 18..20 of the block's first tile: slots 9..11 producer has issued the packed weights, 12..14 a
    // team sees them landed, 15..17 it has an operand slot, 18..20 it has expanded them, 21..23 MMA warp sees them, 24..26 it
    // has issued; slot 30 entry, 31 previous grid ended.
    if (threadIdx.x == 0) TRACE_CLK(p.status, 30);
    const uint32_t cta_rank = blockIdx.x & 1u;  // (the rank in the cluster)
    const int tile_first = static_cast<int>(blockIdx.x >> 1), tile_step = static_cast<int>(gridDim.x >> 1);
    const int num_m_blocks = (p.M + 2 * BM - 1) / (2 * BM), num_n_blocks = (p.N + BN - 1) / BN;
    const int num_tiles = num_m_blocks * num_n_blocks;
    const int items = p.num_kb + p.lr_chunks;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NA; ++s) {
            mbar_init(a_full(s), 1);
            mbar_init(a_empty(s), 1);
        }
        for (int s = 0; s < NP; ++s) {
            mbar_init(p_full(s), 1);
            mbar_init(p_empty(s), TEAM_WARPS);
        }
        for (int s = 0; s < NW; ++s) {
            mbar_init(w_full(s), 2 * TEAM_WARPS);
            mbar_init(w_empty(s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(tfull_bar(a), 1);
            mbar_init(tempty_bar(a), 2 * NUM_EPI_WARPS * 32);
        }
        mbar_init(spare_bar, 1);  // see the teardown
        *abort_flag = 0;
        fence_mbar_init();
        tma_prefetch_desc(&tmap_codes);
        tma_prefetch_desc(&tmap_wpacked);
        tma_prefetch_desc(&tmap_xh);
        tma_prefetch_desc(&tmap_wh);
        tma_prefetch_desc(&tmap_y);
    }
    if (warp == 1) {
        tmem_alloc_pair(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();  // the other CTA's barriers are initialised before anything arrives on them
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    grid_dependency_wait();
    grid_launch_dependents();
    if (threadIdx.x == 0) TRACE_CLK(p.status, 31);

    if (warp < 8) {
        reg_dealloc<64>();
        if (warp == 0) {
            // -------------------------------------------------------- TMA producer (whole warp in the loops, one lane issues)
            // Its chain of instructions per k-block is on the critical path: slots, parities and addresses are carried along.
            uint32_t sa = 0, pha = 1, sp = 0, php = 1, sw = 0, phw = 1, it = 0;
            bool ok = true;
            for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step) {
                const int m0 = (tile % num_m_blocks) * 2 * BM + static_cast<int>(cta_rank) * BM;
                const int n0 = (tile / num_m_blocks) * BN + static_cast<int>(cta_rank) * ROWS;
                for (int i = 0; i < items; ++i, ++it) {
                    if (!mbar_wait(p_empty(sp), php, abort_flag, p.status, DEV_TIMEOUT_PRODUCER) ||
                        !mbar_wait(a_empty(sa), pha, abort_flag, p.status, DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
                    if (i < p.num_kb) {
                        if (elect_one()) {
                            mbar_arrive_expect_tx(p_full(sp), P_BYTES);  // (columns past N read as zero bytes and are not stored)
                            tma_load_2d(smem_base + P_OFFSET + sp * P_BYTES, &tmap_wpacked, p_full(sp), i * (BKC / 2), n0);
                            if (it >= 18 && it <= 20) TRACE_CLK(p.status, it - 9);
                        }
                    } else {
                        // the bf16 weights of the rank-r branch go straight into an operand slot; only when their bytes are expected
                        // are the expanding warps let through, whose arrivals complete the slot's phase
                        if (!mbar_wait(w_empty(sw), phw, abort_flag, p.status, DEV_TIMEOUT_PRODUCER)) { ok = false; break; }
                        if (elect_one()) {
                            if (cta_rank == 0) mbar_expect_tx(w_full(sw), 2 * W_BYTES);
                            tma_load_2d_pair(smem_base + W_OFFSET + sw * W_BYTES, &tmap_wh, map_to_cta(w_full(sw), 0), (i - p.num_kb) * 64, n0);
                            mbar_arrive(p_full(sp));
                        }
                    }
                    if (elect_one()) {
                        if (cta_rank == 0) mbar_arrive_expect_tx(a_full(sa), 2 * A_BYTES);  // counts both CTAs' bytes
                        if (i < p.num_kb) tma_load_2d_pair(smem_base + sa * A_BYTES, &tmap_codes, map_to_cta(a_full(sa), 0), i * BKC, m0);
                        else tma_load_2d_pair(smem_base + sa * A_BYTES, &tmap_xh, map_to_cta(a_full(sa), 0), (i - p.num_kb) * 64, m0);
                    }
                    if (++sa == NA) { sa = 0; pha ^= 1; }
                    if (++sp == NP) { sp = 0; php ^= 1; }
                    if (++sw == NW) { sw = 0; phw ^= 1; }
                }
            }
            if (!ok && lane == 0) {  // give the loads in flight, some of which report to the other CTA, a fixed time
                const unsigned long long t0 = globaltimer_ns();
                while (globaltimer_ns() - t0 < 1000000ull) {}
            }
        } else if (warp == 1) {
            if (cta_rank == 0) {
                // ---------------------------------------------------- MMA issuer
                constexpr uint32_t idesc_i8 = umma_idesc(2 /*s32*/, 1 /*s8*/, 2 * BM, BN);
                constexpr uint32_t idesc_bf = umma_idesc(1 /*f32*/, 1 /*bf16*/, 2 * BM, BN);
                uint32_t sa = 0, pha = 0, sw = 0, phw = 0, tph = 1;
                const uint64_t desc0 = umma_desc_sw128(smem_base);  // (slots differ in the low word's address field, which cannot overflow)
                bool ok = true;
                for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step) {
                    for (int pass = 0; ok && pass < 2; ++pass) {  // the integer pass over K, the rank-r one
                        const uint32_t d = tmem_base + pass * BN;
                        if (!mbar_wait(tempty_bar(pass), tph, abort_flag, p.status, DEV_TIMEOUT_MMA)) { ok = false; break; }
                        tc_fence_after_sync();
                        const int len = pass == 0 ? p.num_kb : p.lr_chunks;
                        for (int i = 0; i < len; ++i) {
                            if (!mbar_wait(w_full(sw), phw, abort_flag, p.status, DEV_TIMEOUT_MMA) ||
                                !mbar_wait(a_full(sa), pha, abort_flag, p.status, DEV_TIMEOUT_MMA)) { ok = false; break; }
                            tc_fence_after_sync();
                            if (elect_one()) {
                                if (pass == 0 && tile == tile_first && i >= 18 && i <= 20) TRACE_CLK(p.status, i + 3);
                                const uint64_t adesc = desc0 + sa * (A_BYTES >> 4), bdesc = desc0 + ((W_OFFSET + sw * W_BYTES) >> 4);
#pragma unroll
                                for (int k = 0; k < 4; ++k) {  // 32 bytes of every row per instruction
                                    if (pass == 0) umma_i8_pair(d, adesc + 2 * k, bdesc + 2 * k, idesc_i8, (i | k) != 0);
                                    else umma_bf16_pair(d, adesc + 2 * k, bdesc + 2 * k, idesc_bf, (i | k) != 0);
                                }
                                umma_commit_pair(w_empty(sw), 3);  // both CTAs' slots are free again
                                umma_commit_pair(a_empty(sa), 3);
                                if (pass == 0 && tile == tile_first && i >= 18 && i <= 20) TRACE_CLK(p.status, i + 6);
                            }
                            __syncwarp();
                            if (++sa == NA) { sa = 0; pha ^= 1; }
                            if (++sw == NW) { sw = 0; phw ^= 1; }
                        }
                        if (ok && elect_one()) umma_commit_pair(tfull_bar(pass), 3);  // both CTAs' epilogue warps
                        __syncwarp();
                    }
                    tph ^= 1;
                }
            }
        } else {
            // -------------------------------------------------------- expansion (warps 2..7: three teams of two)
            // A row's k-block is 64 bytes of packed codes; thread u takes the 16-byte quarter u % 4 of rows u / 4 + 16 j and writes two of the
            // row's eight 16-byte pieces.  Piece c of row r of a 128-byte-swizzled tile lies at r * 128 + ((c ^ (r & 7)) << 4).
            constexpr int PIECES = ROWS / 16;
            const int team = (warp - 2) >> 1, u = threadIdx.x & 63, part = u & 3, r0 = u >> 2, swz = r0 & 7;
            uint32_t first_it = 0;  // items before this tile
            uint32_t sp = team % NP, php = 0, sw = team % NW, phw = 1;  // slots and parities of this team's next item (NP, NW >= TEAMS)
            bool ok = true;
            for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step, first_it += items) {
                for (int i = (team + TEAMS - static_cast<int>(first_it % TEAMS)) % TEAMS; i < items; i += TEAMS) {
                    const uint32_t it = first_it + i;
                    if (!mbar_wait(p_full(sp), php, abort_flag, p.status, DEV_TIMEOUT_UNPACK)) { ok = false; break; }
                    if (i < p.num_kb) {
                        if (u == 0 && it >= 18 && it <= 20) TRACE_CLK(p.status, it - 6);
                        uint4 pk[PIECES];
                        const uint4* src = reinterpret_cast<const uint4*>(smem_gen + P_OFFSET + sp * P_BYTES) + u;
#pragma unroll
                        for (int j = 0; j < PIECES; ++j) pk[j] = src[64 * j];
                        if (!mbar_wait(w_empty(sw), phw, abort_flag, p.status, DEV_TIMEOUT_UNPACK)) { ok = false; break; }
                        if (u == 0 && it >= 18 && it <= 20) TRACE_CLK(p.status, it - 3);
                        uint8_t* dst = smem_gen + W_OFFSET + sw * W_BYTES + r0 * 128;
#pragma unroll
                        for (int j = 0; j < PIECES; ++j) {
                            // nibble q + 8 (low: codes 0..3 of a word's eight, high: 4..7) -> the int8 value 16 q (into the high half, then
                            // flip bit 7: 16 (q + 8) - 128); the epilogue shifts the sums back
                            uint4 o0, o1;
                            o0.x = ((pk[j].x << 4) & 0xF0F0F0F0u) ^ 0x80808080u; o0.y = (pk[j].x & 0xF0F0F0F0u) ^ 0x80808080u;
                            o0.z = ((pk[j].y << 4) & 0xF0F0F0F0u) ^ 0x80808080u; o0.w = (pk[j].y & 0xF0F0F0F0u) ^ 0x80808080u;
                            o1.x = ((pk[j].z << 4) & 0xF0F0F0F0u) ^ 0x80808080u; o1.y = (pk[j].z & 0xF0F0F0F0u) ^ 0x80808080u;
                            o1.z = ((pk[j].w << 4) & 0xF0F0F0F0u) ^ 0x80808080u; o1.w = (pk[j].w & 0xF0F0F0F0u) ^ 0x80808080u;
                            *reinterpret_cast<uint4*>(dst + j * 2048 + (((2 * part) ^ swz) << 4)) = o0;
                            *reinterpret_cast<uint4*>(dst + j * 2048 + (((2 * part + 1) ^ swz) << 4)) = o1;
                        }
                        fence_proxy_async_smem();  // these writes -> visible to the tensor core
                    }
                    __syncwarp();
                    if (u == 0 && it >= 18 && it <= 20) TRACE_CLK(p.status, it);
                    if (lane == 0) {
                        mbar_arrive(p_empty(sp));
                        mbar_arrive_cluster(map_to_cta(w_full(sw), 0));
                    }
                    sp += TEAMS;
                    if (sp >= NP) { sp -= NP; php ^= 1; }
                    sw += TEAMS;
                    if (sw >= NW) { sw -= NW; phw ^= 1; }
                }
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 8..15): one token row per thread, BN / 2 columns
        reg_alloc<192>();
        const int q = warp & 3, half = (warp - 8) >> 2;
        float* s_sw = reinterpret_cast<float*>(smem_gen + P::COL_OFFSET + (warp - 8) * P::COL_BYTES);
        float* s_bias = s_sw + HB;
        const uint32_t sbuf = smem_base + P::STORE_OFFSET + static_cast<uint32_t>(warp - 8) * 2048u;
        uint32_t tph = 0;
        bool ok = true;
        for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step, tph ^= 1) {
            const int m0 = (tile % num_m_blocks) * 2 * BM + static_cast<int>(cta_rank) * BM + q * 32;
            const int col0 = (tile / num_m_blocks) * BN + half * HB;
            const int row = m0 + lane;
            __syncwarp();  // every lane has read the previous tile's scales
            for (int e = lane; e < HB; e += 32) {
                s_sw[e] = col0 + e < p.N ? __ldg(p.wscale + col0 + e) : 0.f;
                s_bias[e] = col0 + e < p.N ? __ldg(p.bias + col0 + e) : 0.f;
            }
            const float sx = row < p.M ? p.xscale[row] : 0.f;
            __syncwarp();
            const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + half * HB;
            float t[HB];  // P s_x
            if (!mbar_wait(tfull_bar(0), tph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE)) { ok = false; break; }
            tc_fence_after_sync();
#pragma unroll
            for (int c = 0; c < HB / 32; ++c) {
                uint32_t raw[32];
                tmem_ld_32x32b_x32(taddr + c * 32, raw);
                tmem_ld_wait();
                tmem_ld_fence(raw);
                // the accumulator holds 16 P (exact); |P| < 2^24, so the conversion is exact too
#pragma unroll
                for (int j = 0; j < 32; ++j) t[c * 32 + j] = static_cast<float>(static_cast<int32_t>(raw[j]) >> 4) * sx;
            }
            tc_fence_before_sync();
            mbar_arrive_cluster(map_to_cta(tempty_bar(0), 0));
            if (!mbar_wait(tfull_bar(1), tph, abort_flag, p.status, DEV_TIMEOUT_EPILOGUE)) { ok = false; break; }
            tc_fence_after_sync();
#pragma unroll
            for (int c = 0; c < HB / 32; ++c) {
                uint32_t lr[32], packed[16];
                tmem_ld_32x32b_x32(taddr + BN + c * 32, lr);
                tmem_ld_wait();
                tmem_ld_fence(lr);
                if (c == HB / 32 - 1) {
                    tc_fence_before_sync();
                    mbar_arrive_cluster(map_to_cta(tempty_bar(1), 0));
                }
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 sw = *reinterpret_cast<const float4*>(s_sw + c * 32 + j), b = *reinterpret_cast<const float4*>(s_bias + c * 32 + j);
                    const float* tc = t + c * 32 + j;
                    packed[j >> 1] = pack_bf16x2(fmaf(tc[0], sw.x, __uint_as_float(lr[j])) + b.x, fmaf(tc[1], sw.y, __uint_as_float(lr[j + 1])) + b.y);
                    packed[(j >> 1) + 1] =
                        pack_bf16x2(fmaf(tc[2], sw.z, __uint_as_float(lr[j + 2])) + b.z, fmaf(tc[3], sw.w, __uint_as_float(lr[j + 3])) + b.w);
                }
                // 32 columns of the warp's 32 rows through its staging tile into a TMA store (as in w4a8_gemm.cu)
                if (lane == 0) bulk_wait_group_read_all();  // the staging tile's previous contents have been read
                __syncwarp();
#pragma unroll
                for (int pc = 0; pc < 4; ++pc) {
                    const uint32_t dst = sbuf + static_cast<uint32_t>(lane) * 64u + (static_cast<uint32_t>(pc ^ ((lane >> 1) & 3)) << 4);
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(packed[4 * pc]), "r"(packed[4 * pc + 1]),
                                 "r"(packed[4 * pc + 2]), "r"(packed[4 * pc + 3])
                                 : "memory");
                }
                fence_proxy_async_smem();  // these writes -> visible to the copy engine
                __syncwarp();
                if (lane == 0 && m0 < p.M && col0 + c * 32 < p.N) {
                    tma_store_2d(&tmap_y, sbuf, col0 + c * 32, m0);
                    bulk_commit_group();
                }
            }
        }
        if (lane == 0) bulk_wait_group_all();  // this warp's stores are performed before the CTA leaves
    }

    if (warp == 1 && lane == 0 && cta_rank == 0 && *abort_flag != 0) {  // a wait gave up: let issued MMAs finish first
        umma_commit_pair(spare_bar, 1);
        const unsigned long long t0 = globaltimer_ns();
        while (!mbar_try_wait(spare_bar, 0) && globaltimer_ns() - t0 < 100000000ull) {}
    }
    tc_fence_before_sync();
    cluster_sync_all();  // neither CTA leaves while the other may still read its operands or signal its barriers
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

template <int BN>
dirotq_status_t launch_bn(const dirotq_layer* L, const A8GemmArgs& a, cudaStream_t stream) {
    const Geometry& g = L->geo;
    CUtensorMap tmap_codes, tmap_xh, tmap_y;
    dirotq_status_t st = encode_tmap_2d(&tmap_codes, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a.codes, (uint64_t)g.K_lp, (uint64_t)a.M,
                                        (uint64_t)g.K_lp, BKC, BM, CU_TENSOR_MAP_SWIZZLE_128B);
    if (st == DIROTQ_OK)
        st = encode_tmap_2d(&tmap_xh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.xh, (uint64_t)g.r_pad, (uint64_t)a.M, (uint64_t)g.r_pad * 2, 64,
                            BM, CU_TENSOR_MAP_SWIZZLE_128B);
    if (st == DIROTQ_OK)
        st = encode_tmap_2d(&tmap_y, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.y, (uint64_t)g.N, (uint64_t)a.M, (uint64_t)g.N * 2, 32, 32,
                            CU_TENSOR_MAP_SWIZZLE_64B);
    if (st != DIROTQ_OK) return st;
    PairParams p;
    p.M = a.M; p.N = g.N;
    p.num_kb = g.K_lp / BKC;
    p.lr_chunks = g.r_pad / 64;
    p.xscale = a.xscale;
    p.wscale = reinterpret_cast<const float*>(L->blob + L->lay.off_wscale);
    p.bias = reinterpret_cast<const float*>(L->blob + L->lay.off_bias);
    p.status = a.status;
    static SmemOptIn<1> opt_in;
    if (!opt_in.ensure(w4a8_pair_kernel<BN>, 0, L->device, Plan<BN>::SMEM_BYTES)) return DIROTQ_ERR_CUDA;
    const int tiles = ((a.M + 2 * BM - 1) / (2 * BM)) * ((g.N + BN - 1) / BN), pairs = sm_count(L->device) / 2;
    const cudaError_t err = launch_kernel_pairs(w4a8_pair_kernel<BN>, 2 * (tiles < pairs ? tiles : pairs), NUM_THREADS, Plan<BN>::SMEM_BYTES, stream, true,
                                                tmap_codes, BN == 256 ? L->tmap_wpacked128 : L->tmap_wpacked64, tmap_xh,
                                                BN == 256 ? L->tmap_wh128 : L->tmap_wh64, tmap_y, p);
    return err == cudaSuccess ? DIROTQ_OK : DIROTQ_ERR_CUDA;
}

}  // namespace

dirotq_status_t launch_w4a8_pair(const dirotq_layer* L, int columns, const A8GemmArgs& a, cudaStream_t stream) {
    return columns == 256 ? launch_bn<256>(L, a, stream) : launch_bn<128>(L, a, stream);
}

}  // namespace dirotq
