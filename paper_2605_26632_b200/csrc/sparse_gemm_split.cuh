// 2:4 sparse x dense GEMM, K split over the CTA pairs (or single CTAs) of a thread-block cluster:
//     Y[m, n] = bf16( s_m * sum_k X~[m,k] W[n,k] + bias[n] + Yr[m,n] )
//
// Why a third kernel.  A problem of few tiles leaves most of the SMs without one, and its time is one tile's: 256 x 12288
// x 3072 ran on 24 of 74 CTA pairs for 96 K blocks, 30.0 us; here 20.2.  Here the `splits` members of a cluster share one
// output tile, each takes a contiguous range of its K blocks, and the fp32 accumulators are added in the
// cluster's shared memory: no global partials, no ticket, and the order of the additions is fixed.
//
// What bounds it (256 x K x 3072 in two splits, 96 SMs): 5.5 us that no K block is in -- launch, first loads, the exchange (~1.1
// us), epilogue -- and 0.30 us per K block of a split, W out of HBM at 5.2 TB/s (80 % of the copy rate): 12288 is 20.0 us, of which
// the stream alone would be 11.5.  With W in the L2 a K block takes 0.20 us, the operand stream of an SM.
// Measured and not built: two row tiles per W stage, as in sparse_gemm_rt2_kernel (an exchange of 123 KB per CTA costs ~5 us: 1024 x
// 12288 x 3072 44 us against 39.4 unsplit); 240- and 256-wide tiles (within 4 % of the 192-wide one).
//
// One tile per cluster, not persistent.  Roles per CTA as in sparse_gemm_kernel: warp 0 TMA producer, warp 1 MMA issuer (of
// a CTA pair's leader), warps 4..11 epilogue.
//
// The exchange.  The accumulator of a CTA is eight units, one per epilogue warp: the 32 rows of the
// warp's tensor-memory quarter x its share of the columns.  Unit u belongs to split u * splits / 8.  When
// every member's MMAs are done (first cluster barrier: the rings are free) each warp whose unit is not its split's copies it,
// in the register layout of the tensor-memory loads, to the owner's ring (512 contiguous bytes per store); after the second
// barrier the owners' warps add what they received to their own accumulators, own first, then the others in ascending
// order, and finish as the other kernels' epilogues do.
#pragma once

#include "epilogue.cuh"
#include "ptx.cuh"
#include "prune_compress.cuh"  // row_scale_from_partials
#include "sparse_gemm.cuh"     // instruction descriptors

namespace lynx {

struct SplitGemmParams {
    int64_t M, N, K;
    const float* row_scale;      // [M] or nullptr
    const float* scale_partial;  // or: per-K-split row sums of a deferred prune launch
    int scale_ks;
    const float* col_scale;    // [N] FP8 weight scales or nullptr
    const uint16_t* bias;      // [N] bf16 or nullptr
    const uint16_t* residual;  // [M x N] bf16 (ld = ldr) or nullptr
    int64_t ldr;
    uint32_t* dev_error;
    int tiles_m;     // tiles of CG * 128 rows; consecutive clusters take the row tiles of one column tile
    int splits;      // members of a cluster: cluster size = CG * splits
    int lora_steps;  // R / 64 dense stages behind the last split's K blocks (0 = no low-rank branch)
    int w_prefetch;  // layer calls: W tiles of the first stages are fetched before the wait for the prune launch
    int trigger;     // the next kernel's CTAs may be placed while this grid works (enough SMs are left for them)
};

template <int BN_, int CG_, int STAGES_, bool FP8_ = false>
struct SplitCfg {
    static constexpr int BN = BN_, CG = CG_, STAGES = STAGES_;
    static constexpr bool FP8 = FP8_;
    static constexpr int BM = 128;
    static constexpr int BK = FP8 ? 256 : 128;      // logical K per stage
    static constexpr int BOX_X = FP8 ? 128 : 64;    // elements of a 128-byte row of A or W
    static constexpr int BN_CTA = BN / CG;
    static constexpr int A_BYTES = BM * 128;
    static constexpr int E_BYTES = FP8 ? 4096 : 2048;
    static constexpr int E_COLS = E_BYTES / 512;
    static constexpr int B_HALF_BYTES = BN_CTA * 128;
    static constexpr int B_BYTES = 2 * B_HALF_BYTES;
    static constexpr int STAGE_BYTES = A_BYTES + E_BYTES + B_BYTES;
    static constexpr int RING_BYTES = STAGES * STAGE_BYTES;
    static constexpr int CH = (BN % 64 == 0) ? 64 : 48;  // epilogue column chunk
    static constexpr int NCH = BN / CH;
    static constexpr int SLOTS = (NCH + 1) / 2;          // most chunks of a unit
    static constexpr int UNITS = 8;                      // one per epilogue warp
    static constexpr int UNIT_BYTES = SLOTS * CH * 128;  // a unit's accumulators: 32 lanes x SLOTS * CH registers
    static constexpr int E_COL0 = BN;
    static constexpr int TMEM_COLS = 512;
    static constexpr int STRIP_BYTES = BN * 4 * (FP8 ? 2 : 1);
    static constexpr int NUM_BARS = 2 * STAGES + 1;
    static constexpr int SMEM_BYTES = 1024 /*align slack*/ + RING_BYTES + STRIP_BYTES + 256;
    static constexpr int THREADS = GEMM_THREADS;
    // units an owner receives from the other splits have to fit into its ring
    static constexpr bool splits_fit(int s) {
        return s >= 2 && CG * s <= 8 && (UNITS + s - 1) / s * (s - 1) * UNIT_BYTES <= RING_BYTES;
    }
    static_assert(BN % CH == 0 && NCH >= 2 && BN % 16 == 0 && BN_CTA % 8 == 0, "tile N");
    static_assert(B_HALF_BYTES % 1024 == 0 && UNIT_BYTES % 1024 == 0, "swizzled tiles and staging boxes stay 1024-byte aligned");
    static_assert(E_COL0 % 4 == 0 && E_COL0 + E_COLS * STAGES <= TMEM_COLS, "tensor memory budget");
    static_assert(8 * NUM_BARS + 16 <= 256, "barrier area");
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
    static_assert(splits_fit(2), "exchange area");
};

template <class Cfg, bool LORA>
__global__ void __launch_bounds__(Cfg::THREADS, 1)
sparse_gemm_split_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                         const __grid_constant__ CUtensorMap tmap_e, const __grid_constant__ CUtensorMap tmap_y,
                         const __grid_constant__ CUtensorMap tmap_t, const __grid_constant__ CUtensorMap tmap_la,
                         const SplitGemmParams p) {
    constexpr int CG = Cfg::CG, STAGES = Cfg::STAGES, BN = Cfg::BN;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sA = smem_base;                   // [stage] A_BYTES
    const uint32_t sB = sA + STAGES * Cfg::A_BYTES;  // [stage] B_BYTES
    const uint32_t sE = sB + STAGES * Cfg::B_BYTES;  // [stage] E_BYTES
    const uint32_t sStrip = sE + STAGES * Cfg::E_BYTES;
    const uint32_t sBar = sStrip + Cfg::STRIP_BYTES;
    const uint32_t bar_full = sBar, bar_empty = sBar + 8 * STAGES, bar_tfull = sBar + 16 * STAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_gen + (sBar - smem_base) + 8 * Cfg::NUM_BARS);
    volatile uint32_t* cta_abort = tmem_slot + 1;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int crank = (int)cluster_ctarank();
    const int sub = crank % CG, split = crank / CG;  // CTA of the pair, split of the cluster
    const bool leader = sub == 0;
    const int cluster_id = blockIdx.x / (CG * p.splits);
    const int tm = cluster_id % p.tiles_m, tn = cluster_id / p.tiles_m;
    const int kblocks = (int)(p.K / Cfg::BK);
    const int kb0 = split * kblocks / p.splits, nkb = (split + 1) * kblocks / p.splits - kb0;
    const int lora_steps = (LORA && split == p.splits - 1) ? p.lora_steps : 0;
    const int steps = nkb + lora_steps;
    const int rb = tm * CG + sub;  // this CTA's 128-row block
    const int n0_cta = tn * BN + sub * Cfg::BN_CTA;

    if (threadIdx.x == 0) {
        *cta_abort = 0;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar_full + 8 * s, 1);   // leader's producer arrives once (+ transaction bytes)
            mbar_init(bar_empty + 8 * s, 1);  // one tcgen05.commit
        }
        mbar_init(bar_tfull, 1);  // one tcgen05.commit
        fence_mbar_init();
        prefetch_tmap(&tmap_a);
        prefetch_tmap(&tmap_b);
        prefetch_tmap(&tmap_e);
        prefetch_tmap(&tmap_y);
        if (lora_steps) {
            prefetch_tmap(&tmap_t);
            prefetch_tmap(&tmap_la);
        }
    }
    if (warp == 1) {
        tmem_alloc<CG>(smem_u32(tmem_slot), Cfg::TMEM_COLS);
        tmem_relinquish<CG>();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_relaxed();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    const uint32_t full0 = (CG == 2) ? mapa(bar_full, (uint32_t)(crank - sub)) : bar_full;  // the pair's leader's barriers
    // W tiles of the first stages, before the wait for the previous kernel (W is not its output in a layer call)
    int npre = 0;
    if (warp == 0 && p.w_prefetch) {
        npre = nkb < STAGES ? nkb : STAGES;
        if (elect_one()) for (int s = 0; s < npre; ++s) {
            const uint32_t b_dst = sB + s * Cfg::B_BYTES;
            const int x = (kb0 + s) * Cfg::BK;
            if (leader) mbar_arrive_expect_tx(bar_full + 8 * s, CG * Cfg::STAGE_BYTES);
            if constexpr (CG == 1) {
                tma_load_2d(b_dst, &tmap_b, x, n0_cta, bar_full + 8 * s);
                tma_load_2d(b_dst + Cfg::B_HALF_BYTES, &tmap_b, x + Cfg::BOX_X, n0_cta, bar_full + 8 * s);
            } else {
                tma_load_2d_pair(b_dst, &tmap_b, x, n0_cta, full0 + 8 * s);
                tma_load_2d_pair(b_dst + Cfg::B_HALF_BYTES, &tmap_b, x + Cfg::BOX_X, n0_cta, full0 + 8 * s);
            }
        }
    }
    // everything above overlapped the previous kernel's tail; its results are needed from here on
    griddep_wait();
    if (p.trigger) griddep_launch_dependents();

    if (warp < GEMM_EPI_WARP0) {
        setmaxnreg_dec<GEMM_REGS_ISSUE>();
        if (warp == 0) {
            // -------------------------------------------------------------- producer ----------
            auto load = [&](uint32_t dst, const CUtensorMap* m, int x, int y, uint32_t bar) {
                if constexpr (CG == 1) tma_load_2d(dst, m, x, y, bar);
                else tma_load_2d_pair(dst, m, x, y, bar);
            };
            constexpr int E_ROWS = Cfg::E_BYTES / 1024;  // 1024-byte rows of the metadata tensor map per stage
            uint32_t stage = 0, phase = 0;
            bool ok = true;
            int issued = 0;
            for (int i = 0; i < steps; ++i) {
                ok = mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1, cta_abort, p.dev_error);
                if (!ok) break;
                const uint32_t a_dst = sA + stage * Cfg::A_BYTES, b_dst = sB + stage * Cfg::B_BYTES;
                const uint32_t e_dst = sE + stage * Cfg::E_BYTES;
                const uint32_t bar = full0 + 8 * stage;
                if (!elect_one()) {
                } else if (i < nkb) {
                    const int kb = kb0 + i;
                    const bool pre = i < npre;  // W tile and byte count went out before the wait
                    // the leader announces the bytes of both CTAs; the peer's bytes may land first
                    if (leader && !pre) mbar_arrive_expect_tx(bar_full + 8 * stage, CG * Cfg::STAGE_BYTES);
                    load(a_dst, &tmap_a, kb * Cfg::BOX_X, rb * Cfg::BM, bar);
                    load(e_dst, &tmap_e, 0, E_ROWS * (rb * kblocks + kb), bar);
                    if (!pre) {
                        load(b_dst, &tmap_b, kb * Cfg::BK, n0_cta, bar);
                        load(b_dst + Cfg::B_HALF_BYTES, &tmap_b, kb * Cfg::BK + Cfg::BOX_X, n0_cta, bar);
                    }
                } else {
                    // low-rank stages: T box in the A slot, L_A box in the first half of the W slot
                    const int j = i - nkb;
                    if (leader) mbar_arrive_expect_tx(bar_full + 8 * stage, CG * (Cfg::A_BYTES + Cfg::B_HALF_BYTES));
                    load(a_dst, &tmap_t, j * 64, rb * Cfg::BM, bar);
                    load(b_dst, &tmap_la, j * 64, n0_cta, bar);
                }
                ++issued;
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            for (int s = 0; s < STAGES && ok; ++s) {  // the last releases of the stages (see epilogue.cuh)
                ok = mbar_wait_warp(bar_empty + 8 * stage, phase ^ 1, cta_abort, p.dev_error);
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
            if (!ok && issued) bounded_delay_ns(200000);  // let the copies in flight land before teardown
        } else if (warp == 1 && leader) {
            // -------------------------------------------------------------- MMA issuer --------
            constexpr uint32_t idesc0 = make_idesc_sp_bf16(Cfg::BM * CG, BN), idesc1 = idesc0 | 1u;
            constexpr uint32_t idesc_dense = idesc0 & ~(1u << 2);
            constexpr uint32_t idesc8 = make_idesc_sp_e4m3(Cfg::BM * CG, BN);
            const uint64_t d0 = make_desc_sw128(sA);
            const uint32_t desc_hi = (uint32_t)(d0 >> 32);
            const uint32_t a_lo0 = (uint32_t)d0, b_lo0 = (uint32_t)make_desc_sw128(sB);
            const uint64_t e_d0 = make_desc_rows16(sE);
            constexpr uint32_t BH = Cfg::B_HALF_BYTES >> 4;
            const uint16_t pair = (uint16_t)(0x3u << (crank - sub));
            auto commit = [&](uint32_t bar) {
                if constexpr (CG == 1) tc_commit(bar);
                else tc_commit_pair(bar, pair);
            };
            uint32_t stage = 0, phase = 0, accumulate = 0;
            for (int i = 0; i < steps; ++i) {
                if (!mbar_wait_warp(bar_full + 8 * stage, phase, cta_abort, p.dev_error)) break;
                tc_fence_after();
                const uint32_t b_lo = b_lo0 + stage * (Cfg::B_BYTES >> 4);
                const bool sparse = !LORA || i < nkb;
                if (elect_one()) {
                    const uint32_t a_lo = a_lo0 + stage * (Cfg::A_BYTES >> 4);
                    const uint32_t e = tmem_base + Cfg::E_COL0 + stage * Cfg::E_COLS;
                    const uint64_t e_desc = e_d0 + (uint64_t)(stage * (Cfg::E_BYTES >> 4));
                    if (sparse) {
                        tmem_cp_128x128b<CG>(e, e_desc);
                        if constexpr (Cfg::FP8) {
                            tmem_cp_128x128b<CG>(e + 4, e_desc + (uint64_t)(2048 >> 4));
                            mma_sp_f8_lh<CG>(tmem_base, a_lo, b_lo, desc_hi, e, idesc8, accumulate);
                            mma_sp_f8_lh<CG>(tmem_base, a_lo + 2, b_lo + 4, desc_hi, e + 2, idesc8, 1u);
                            mma_sp_f8_lh<CG>(tmem_base, a_lo + 4, b_lo + BH, desc_hi, e + 4, idesc8, 1u);
                            mma_sp_f8_lh<CG>(tmem_base, a_lo + 6, b_lo + BH + 4, desc_hi, e + 6, idesc8, 1u);
                        } else {
                            mma_sp_bf16_lh<CG>(tmem_base, a_lo, b_lo, desc_hi, e, idesc0, accumulate);
                            mma_sp_bf16_lh<CG>(tmem_base, a_lo + 2, b_lo + 4, desc_hi, e, idesc1, 1u);
                            mma_sp_bf16_lh<CG>(tmem_base, a_lo + 4, b_lo + BH, desc_hi, e + 2, idesc0, 1u);
                            mma_sp_bf16_lh<CG>(tmem_base, a_lo + 6, b_lo + BH + 4, desc_hi, e + 2, idesc1, 1u);
                        }
                    } else {
                        mma_bf16_lh<CG>(tmem_base, a_lo, b_lo, desc_hi, idesc_dense, accumulate);
                        mma_bf16_lh<CG>(tmem_base, a_lo + 2, b_lo + 2, desc_hi, idesc_dense, 1u);
                        mma_bf16_lh<CG>(tmem_base, a_lo + 4, b_lo + 4, desc_hi, idesc_dense, 1u);
                        mma_bf16_lh<CG>(tmem_base, a_lo + 6, b_lo + 6, desc_hi, idesc_dense, 1u);
                    }
                    if (i == steps - 1) commit(bar_tfull);
                    commit(bar_empty + 8 * stage);
                }
                accumulate = 1u;
                if (++stage == STAGES) { stage = 0; phase ^= 1; }
            }
        }
        __syncwarp();
        cluster_arrive_relaxed();  // every member's MMAs are done (what the epilogue warps wait for before they arrive)
        cluster_wait();
        cluster_arrive_relaxed();  // the accumulators are where they belong
        cluster_wait();
    } else {
        setmaxnreg_inc<GEMM_REGS_EPI>();
        // ------------------------------------------------------------------ epilogue ----------
        constexpr int CH = Cfg::CH, NCH = Cfg::NCH, SLOTS = Cfg::SLOTS;
        const int ew = warp - GEMM_EPI_WARP0, q = warp & 3, h = ew >> 2;  // quarter, which of its two warps
        const uint32_t sc = sStrip + BN * 4;
        if (const int c = (int)threadIdx.x - 32 * GEMM_EPI_WARP0; c < BN) {
            const int n = tn * BN + c;
            sts32f(sStrip + c * 4, (p.bias != nullptr && n < p.N) ? __uint_as_float((uint32_t)p.bias[n] << 16) : 0.0f);
            if constexpr (Cfg::FP8) sts32f(sc + c * 4, (p.col_scale != nullptr && n < p.N) ? p.col_scale[n] : 1.0f);
        }
        bar_sync_named(GEMM_EPI_BARRIER, 32 * GEMM_EPI_WARPS);
        // This warp's unit: chunks [c_own, c_own + n_own) of the accumulator; the odd chunk goes to the first warp of the quarter.
        const int c_own = h == 0 ? 0 : SLOTS, n_own = h == 0 ? SLOTS : NCH - SLOTS, m0 = rb * Cfg::BM + q * 32;
        const int owner = ew * p.splits / Cfg::UNITS;
        const bool own = owner == split;
        // where split `from` leaves the unit in its owner's ring
        auto inbox = [&](int from) {
            const int local = ew - (owner * Cfg::UNITS + p.splits - 1) / p.splits;
            return smem_base + (uint32_t)((local * (p.splits - 1) + (from < owner ? from : from - 1)) * Cfg::UNIT_BYTES);
        };
        float s[4];
        uint32_t packed[SLOTS][2][CH / 4];
        if (own) {
            const int64_t row = m0 + lane;
            float sl = 1.0f;
            if (row < p.M) {
                if (p.scale_partial != nullptr) sl = row_scale_from_partials(p.scale_partial, row, p.scale_ks);
                else if (p.row_scale != nullptr) sl = p.row_scale[row];
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) s[i] = __shfl_sync(0xffffffffu, sl, 8 * i + (lane >> 2));
            if (p.residual != nullptr) {  // arrives during the main loop, in the registers of the results
#pragma unroll
                for (int slot = 0; slot < SLOTS; ++slot)
                    if (slot < n_own)
                        epi_load_residual<CH>(p.residual, p.ldr, m0, p.M, tn * BN + (c_own + slot) * CH, p.N, lane, packed[slot]);
            }
        }
        const bool alive = mbar_wait_warp(bar_tfull, 0, cta_abort, p.dev_error);
        tc_fence_after();
        __syncwarp();
        cluster_arrive_release();
        cluster_wait();  // every member's MMAs are done: the rings are free
        const uint32_t t_row = tmem_base + ((uint32_t)(q * 32) << 16);
        if (alive && !own) {
            const uint32_t dst = mapa(inbox(split), (uint32_t)(owner * CG + sub)) + lane * 16;
#pragma unroll
            for (int slot = 0; slot < SLOTS; ++slot) {
                if (slot >= n_own) break;
                uint32_t v[2][CH / 2];
                epi_tmem_ld<CH>(t_row + (c_own + slot) * CH, v);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < CH / 4; ++i) {
                    const uint32_t* x = &v[i / (CH / 8)][4 * (i % (CH / 8))];
                    sts128_cluster(dst + (slot * (CH / 4) + i) * 512, x[0], x[1], x[2], x[3]);
                }
            }
        }
        __syncwarp();
        cluster_arrive_release();
        cluster_wait();
        if (alive && own) {
            auto finish = [&](auto has_residual) {
                constexpr bool RES = decltype(has_residual)::value;
#pragma unroll
                for (int slot = 0; slot < SLOTS; ++slot) {
                    if (slot >= n_own) break;
                    const int c = c_own + slot;
                    uint32_t v[2][CH / 2];
                    epi_tmem_ld<CH>(t_row + c * CH, v);
                    tmem_ld_wait();
                    for (int from = 0; from < p.splits; ++from) {
                        if (from == split) continue;
                        const uint32_t src = inbox(from) + lane * 16;
#pragma unroll
                        for (int i = 0; i < CH / 4; ++i) {
                            uint32_t a[4];
                            lds128(src + (slot * (CH / 4) + i) * 512, a[0], a[1], a[2], a[3]);
                            uint32_t* x = &v[i / (CH / 8)][4 * (i % (CH / 8))];
#pragma unroll
                            for (int e = 0; e < 4; ++e) x[e] = __float_as_uint(__uint_as_float(x[e]) + __uint_as_float(a[e]));
                        }
                    }
                    epi_convert<CH, Cfg::FP8, RES>(v, s, sStrip + c * (CH * 4), sc + c * (CH * 4), lane, packed[slot]);
                }
            };
            if (p.residual != nullptr) finish(std::true_type{});
            else finish(std::false_type{});
            __syncwarp();  // the unit's inbox has been read: its memory stages the results, a box per chunk
            const uint32_t box = inbox(split == 0 ? 1 : 0);
#pragma unroll
            for (int slot = 0; slot < SLOTS; ++slot) {
                if (slot >= n_own) break;
                const int n0 = tn * BN + (c_own + slot) * CH;
                if (n0 < p.N)  // rows past M and columns past N are clipped by the store
                    epi_store<CH, 32>(&tmap_y, packed[slot], n0, m0, box + slot * (32 * CH * 2), true, lane);
            }
        }
        if (lane == 0) tma_store_wait_read<0>();  // (the end of the grid makes the stores visible)
        __syncwarp();
    }

    // ---------------------------------------------------------------------- teardown ----------
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) cluster_sync_relaxed();  // both CTAs of a pair have read their accumulators
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc<CG>(tmem_base, Cfg::TMEM_COLS);
    }
}

}  // namespace lynx
