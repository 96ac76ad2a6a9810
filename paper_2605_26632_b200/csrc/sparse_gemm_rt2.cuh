// 2:4 sparse x dense GEMM, "two row tiles per W stage" form (Algorithm 1 lines 5-6):
//     Y[m, n] = bf16( s_m * sum_k X~[m,k] W[n,k] + bias[n] + Yr[m,n] )
//
// Why a second kernel.  A CTA pair works on TWO 256-row tiles of the same 240 columns at once
// ("double"): a ring stage holds two compressed-A tiles and two metadata blocks per CTA but ONE W
// tile, 66 KB for twice the MMAs of the single-tile kernel's 48 KB stage (-31 % bytes per flop).  The
// eight MMAs of a stage take 960 cycles and the loop runs at 950-1050 per stage; a single's four take
// 480 and its loop runs at 530-650, because 48 KB per 480 cycles is more than a CTA gets (84 B/clk with no
// MMAs at all).  Under the power cap, which launches of this size reach within milliseconds, the bytes
// not moved count again: 4096 x 3072 x 12288 runs 121.7 us in doubles, 127.1 us in singles
// (sustained 140.8 against 148.1).
// The two accumulators fill all of tensor memory (2 x 240 columns + metadata), so the epilogue
// of a double is not hidden behind a following main loop: the eight epilogue warps read the first accumulator as
// soon as its last MMA is done, then the second, and the issuer starts the next item on the first while
// the second is read.  What remains is about 2500 cycles per double (24000 of MMAs at K = 3072).
//
// Work items of a cluster: "doubles" (512 x 240) first, then "singles" (256 x 240, the tile of
// sparse_gemm_kernel; consecutive singles alternate between the two accumulators, so their
// epilogues overlap the next single's main loop).  How many doubles a launch uses is the host's
// choice (PairSchedule, a cost model): doubles cost less per unit, singles fill the clusters that
// would otherwise idle in the last round.
//
// FP8 operands (Gemm2Cfg<.., true>): the same with 256 logical K per stage, 70 KB and twice the metadata columns, for which
// tensor memory has two slots (E_SLOTS).  The board's power cap bounds these launches, too (994 W, 1180 MHz): what counts is
// the bytes not moved.  16384 x 12288 x 3072 307 -> 288 us in blocks of seconds, 4096 x 3072 x 12288 78.0 -> 72.7 in short ones.
//
// Roles per CTA (384 threads): warp 0 TMA producer, warp 1 MMA issuer (leader CTA), both converged with
// one elected lane issuing (see sparse_gemm.cuh), warps 2 and 3 idle, warps 4-11 epilogue.  Every wait is
// bounded (mbar_wait): on expiry the kernel raises the error word and all roles leave.
#pragma once

#include "ptx.cuh"
#include "prune_compress.cuh"  // row_scale_from_partials
#include "epilogue.cuh"
#include "sparse_gemm.cuh"     // make_idesc_sp_bf16

namespace lynx {

// Distribution of the output over C clusters.  Units are 256 x BN tiles (tm, tn).  Double slot i
// pairs the row tiles 2d and 2d + 1 of column tile tn; inside a group of `gd` double rows the row
// index runs fastest (the clusters of a round then share gd * 2 blocks of A and C / gd tiles of W).
// The first D slots are run as doubles, dealt round-robin: cluster c gets slots c, c + C, ...
// Every other unit is a single: the two halves of the slots D .. Dmax - 1 and, when the number of
// row tiles is odd, the last row tile.  Singles are dealt so that clusters with one double fewer
// ("light", index >= D % C) get one first, then round-robin over all clusters starting there.
struct PairSchedule {
    int TM, TN, C;
    int DM, gd, D, Dmax, S, b, L;

    __host__ __device__ void init(int tiles_m, int tiles_n, int clusters, int doubles, int group_double_rows) {
        TM = tiles_m; TN = tiles_n; C = clusters;
        DM = TM / 2;
        gd = group_double_rows;
        if (gd <= 0 || gd > DM) gd = DM > 0 ? DM : 1;
        if (DM > 0) {  // groups of nearly equal size
            const int groups = (DM + gd - 1) / gd;
            gd = (DM + groups - 1) / groups;
        }
        Dmax = DM * TN;
        D = doubles < 0 ? 0 : (doubles > Dmax ? Dmax : doubles);
        S = 2 * (Dmax - D) + ((TM & 1) ? TN : 0);
        b = D % C;
        L = C - b;
    }
    __host__ __device__ void slot_coords(int i, int& d, int& tn) const {
        const int per_group = gd * TN;
        const int g = i / per_group, r = i - g * per_group;
        const int rows = (DM - g * gd < gd) ? DM - g * gd : gd;
        tn = r / rows;
        d = g * gd + (r - tn * rows);
    }
    __host__ __device__ int position(int c) const { return (c - b + C) % C; }
    __host__ __device__ int num_doubles(int c) const { return (D > c) ? (D - c + C - 1) / C : 0; }
    __host__ __device__ int num_singles(int c) const {
        const int p = position(c);
        const int first = (p < L && p < S) ? 1 : 0;
        const int rest = (S > L + p) ? (S - L - p + C - 1) / C : 0;
        return first + rest;
    }
    // k-th single of cluster c -> index in the list of singles
    __host__ __device__ int single_index(int c, int k) const {
        const int p = position(c);
        if (p < L) return k == 0 ? p : L + p + (k - 1) * C;
        return L + p + k * C;
    }
    __host__ __device__ void single_unit(int j, int& tm, int& tn) const {
        const int broken = 2 * (Dmax - D);
        if (j < broken) {
            int d;
            slot_coords(D + (j >> 1), d, tn);
            tm = 2 * d + (j & 1);
        } else {
            tm = TM - 1;
            tn = j - broken;
        }
    }
    __host__ __device__ int num_items(int c) const { return num_doubles(c) + num_singles(c); }
    // item i of cluster c: first row tile, column tile, row tiles (1 or 2); for a single also its
    // ordinal among the cluster's singles (which accumulator it uses)
    __host__ __device__ void item(int c, int i, int& tm0, int& tn, int& rows, int& ordinal) const {
        const int nd = num_doubles(c);
        if (i < nd) {
            int d;
            slot_coords(c + i * C, d, tn);
            tm0 = 2 * d;
            rows = 2;
            ordinal = 0;
        } else {
            ordinal = i - nd;
            single_unit(single_index(c, ordinal), tm0, tn);
            rows = 1;
        }
    }
};

struct Gemm2Params {
    int64_t M, N, K;
    const float* row_scale;      // [M] or nullptr
    const float* scale_partial;  // or: per-K-split row sums of a deferred prune launch
    int scale_ks;
    const float* col_scale;    // [N] FP8 weight scales or nullptr
    const uint16_t* bias;      // [N] bf16 or nullptr
    const uint16_t* residual;  // [M x N] bf16 (ld = ldr) or nullptr
    int64_t ldr;
    uint32_t* dev_error;
    PairSchedule sched;
    int lora_steps;  // R / 64 extra dense stages per item (0 = no low-rank branch)
    int w_prefetch;  // layer calls: W tiles of the first stages are fetched before the wait for the prune launch
};

// FP8_ = true: E4M3 operands, in the byte geometry of a stage as in GemmCfg (256 logical K, twice the metadata).
template <int BN_, int STAGES_, bool FP8_ = false>
struct Gemm2Cfg {
    static constexpr int BN = BN_, STAGES = STAGES_, CG = 2;
    static constexpr bool FP8 = FP8_;
    static constexpr int BM = 128, BK = FP8 ? 256 : 128;
    static constexpr int BOX_X = FP8 ? 128 : 64;       // elements of a 128-byte row of A or W
    static constexpr int BN_CTA = BN / CG;
    static constexpr int A_BYTES = BM * 128;           // one row tile of compressed A: 16 KB
    static constexpr int E_BYTES = FP8 ? 4096 : 2048;  // its metadata
    static constexpr int B_HALF_BYTES = BN_CTA * 128;  // one 128-byte K slice of this CTA's W rows
    static constexpr int B_BYTES = 2 * B_HALF_BYTES;
    static constexpr int STAGE_BYTES = 2 * A_BYTES + 2 * E_BYTES + B_BYTES;
    static constexpr int SINGLE_TX = A_BYTES + E_BYTES + B_BYTES;
    static constexpr int CH = 48;                      // epilogue column chunk
    static constexpr int NCH = BN / CH;
    static constexpr int E_COL0 = 2 * BN;              // metadata columns behind the two accumulators
    static constexpr int E_COLS = 2 * E_BYTES / 512;   // per stage: half of them per row tile
    // Slots of a stage's metadata in tensor memory.  FP8 stages have 16 columns, and beside two 240-column accumulators
    // there is room for two of them: the issuer waits for the MMAs of the stage before the last, whose columns it
    // overwrites.  (The last stage's eight MMAs run meanwhile: nothing stalls.)
    static constexpr int E_SLOTS = FP8 ? 2 : STAGES;
    static constexpr int TMEM_COLS = 512;
    static constexpr int EPI_WARPS = GEMM_EPI_WARPS;
    static constexpr int THREADS = GEMM_THREADS;
    // the single-tile items run on a ring of their own over the same shared memory: four stages of
    // 48 KB (A 16 KB, metadata 2 KB, W 30 KB) instead of three of 66 KB
    static constexpr int STAGES1 = 4;
    static constexpr int RING1_A = 0, RING1_B = STAGES1 * A_BYTES, RING1_E = RING1_B + STAGES1 * B_BYTES;
    static constexpr int NUM_BARS = 2 * STAGES + 2 * STAGES1 + 4;
    static constexpr int C_BOX_BYTES = 32 * CH * 2;    // a chunk of 32 rows x 48 columns
    static constexpr int BOX_ROWS = FP8 ? 16 : 32;     // rows of an epilogue warp's own staging box
    static constexpr int C_BYTES = EPI_WARPS * BOX_ROWS * CH * 2;
    static constexpr int BIAS_BYTES = BN * 4 * (FP8 ? 2 : 1);  // the item's bias values (and weight scales, fp32), two items' worth
    static constexpr int SMEM_BYTES = 1024 /*align slack*/ + STAGES * STAGE_BYTES + C_BYTES + 2 * BIAS_BYTES + 256;
    // Cycles from one chunk store of a CTA to the next.  The stores compete with the operand stream of the next main
    // loop, whose ring is too short to ride out 122 KB leaving at once: a double's 40 chunks go one after the other,
    // spread over 500 cycles per K block (a K block of a double takes 960, of a single 530-650), at most 16000 in
    // all: 4096 x 3072 x 12288 122.1 -> 120.0 us, 4352 x 3072 x 9216 100.2 -> 98.7 (over 100 cycles per K block: 122.5
    // and 99.7); without a limit the last stores at K = 12288 delay what follows (layer + 1 %).
    // With a residual they go at once: a warp fetches the next item's only behind its last store, and fetched late
    // it holds up that item's epilogue: 4352 x 3072 x 9216 115.1 -> 112.1 us, 4352 x 3072 x 3072 40.6 -> 39.7.
    __host__ __device__ static constexpr int store_pace(int kblocks, bool residual) {
        return residual ? 0 : (kblocks < 32 ? kblocks : 32) * 100 / EPI_WARPS;
    }
    static_assert(store_pace(24, false) * NCH * EPI_WARPS == 500 * 24 && store_pace(96, false) * NCH * EPI_WARPS == 16000 &&
                      store_pace(24, true) == 0, "spread of a double's chunk stores");
    static_assert(NCH == 5 && BN % CH == 0 && BN_CTA % 8 == 0, "tile N: the epilogue deals five chunks per accumulator");
    static_assert(EPI_WARPS * 5 * C_BOX_BYTES <= STAGES * STAGE_BYTES, "last item: a staging box per chunk in the ring");
    static_assert(B_HALF_BYTES % 1024 == 0, "swizzle atoms need 1024-byte aligned tiles");
    static_assert(E_COL0 + E_COLS * E_SLOTS <= TMEM_COLS && E_COLS / 2 * STAGES1 <= E_COLS * E_SLOTS, "tensor memory budget");
    static_assert(E_SLOTS == STAGES || (E_SLOTS == 2 && STAGES == 3), "the issuer looks two stages back");
    static_assert(RING1_E + STAGES1 * E_BYTES <= STAGES * STAGE_BYTES, "the single-tile ring fits into the double ring's memory");
    static_assert(8 * NUM_BARS + 16 <= 256, "barrier area");
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
};

template <class Cfg, bool LORA>
__global__ void __launch_bounds__(Cfg::THREADS, 1)
sparse_gemm_rt2_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                       const __grid_constant__ CUtensorMap tmap_e, const __grid_constant__ CUtensorMap tmap_y,
                       const __grid_constant__ CUtensorMap tmap_t, const __grid_constant__ CUtensorMap tmap_la,
                       const Gemm2Params p) {
    constexpr int STAGES = Cfg::STAGES, BN = Cfg::BN;
    const int lora_steps = LORA ? p.lora_steps : 0;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t sA = smem_base;                              // [stage][row tile] A_BYTES
    const uint32_t sB = sA + STAGES * 2 * Cfg::A_BYTES;         // [stage] B_BYTES
    const uint32_t sE = sB + STAGES * Cfg::B_BYTES;             // [stage][row tile] E_BYTES
    const uint32_t sC = sE + STAGES * 2 * Cfg::E_BYTES;         // [epilogue warp] C_BOX_BYTES
    const uint32_t sBias = sC + Cfg::C_BYTES;                   // [item parity] BIAS_BYTES
    const uint32_t sBar = sBias + 2 * Cfg::BIAS_BYTES;
    const uint32_t bar_full = sBar, bar_empty = sBar + 8 * STAGES;
    const uint32_t bar_tfull = sBar + 16 * STAGES, bar_tempty = bar_tfull + 16;
    const uint32_t bar_full1 = bar_tempty + 16, bar_empty1 = bar_full1 + 8 * Cfg::STAGES1;  // single-tile ring
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_gen + (sBar - smem_base) + 8 * Cfg::NUM_BARS);
    volatile uint32_t* cta_abort = tmem_slot + 1;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    const int cluster_id = blockIdx.x / 2;
    const int kblocks = (int)(p.K / Cfg::BK);
    const PairSchedule& sched = p.sched;
    const int num_items = sched.num_items(cluster_id);

    if (threadIdx.x == 0) {
        *cta_abort = 0;
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar_full + 8 * s, 1);   // leader's producer arrives once (+ transaction bytes)
            mbar_init(bar_empty + 8 * s, 1);  // one tcgen05.commit
        }
        for (int s = 0; s < Cfg::STAGES1; ++s) {
            mbar_init(bar_full1 + 8 * s, 1);
            mbar_init(bar_empty1 + 8 * s, 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(bar_tfull + 8 * a, 1);   // one tcgen05.commit
            mbar_init(bar_tempty + 8 * a, 2 * Cfg::EPI_WARPS);  // the epilogue warps of both CTAs
        }
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
        tmem_alloc<2>(smem_u32(tmem_slot), Cfg::TMEM_COLS);
        tmem_relinquish<2>();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_relaxed();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    // W tiles of the first stages of the first item, before the wait for the previous kernel (W is
    // not its output in a layer call); the producer below skips them
    int npre = 0;
    if (warp == 0 && p.w_prefetch && num_items > 0) {
        int tm0, tn, rows, ordinal;
        sched.item(cluster_id, 0, tm0, tn, rows, ordinal);
        const bool r1 = rows == 1;
        const int nst = r1 ? Cfg::STAGES1 : STAGES;
        npre = kblocks < nst ? kblocks : nst;
        const uint32_t bfull = r1 ? bar_full1 : bar_full;
        const uint32_t full0 = mapa(bfull, 0);
        const int n0 = tn * BN + (int)rank * Cfg::BN_CTA;
        const uint32_t tx = r1 ? (uint32_t)Cfg::SINGLE_TX : (uint32_t)Cfg::STAGE_BYTES;
        if (elect_one()) for (int s = 0; s < npre; ++s) {
            const uint32_t b_dst = r1 ? sA + Cfg::RING1_B + s * Cfg::B_BYTES : sB + s * Cfg::B_BYTES;
            if (leader) mbar_arrive_expect_tx(bfull + 8 * s, 2 * tx);
            tma_load_2d_pair(b_dst, &tmap_b, s * Cfg::BK, n0, full0 + 8 * s);
            tma_load_2d_pair(b_dst + Cfg::B_HALF_BYTES, &tmap_b, s * Cfg::BK + Cfg::BOX_X, n0, full0 + 8 * s);
        }
    }
    // everything above overlapped the previous kernel's tail; its results are needed from here on
    griddep_wait();

    if (warp < GEMM_EPI_WARP0) {
    setmaxnreg_dec<GEMM_REGS_ISSUE>();
    if (warp == 0) {
        // ------------------------------------------------------------------ producer ----------
        {
            constexpr int E_ROWS = Cfg::E_BYTES / 1024;  // 1024-byte rows of the metadata tensor map per stage and row tile
            uint32_t stage = 0, phase = 0, issued = 0;
            bool ok = true;
            bool ring1 = false;  // false: the 3 x 66 KB ring of the doubles, true: the 4 x 48 KB ring of the singles
            for (int it = 0; it < num_items && ok; ++it) {
                int tm0, tn, rows, ordinal;
                sched.item(cluster_id, it, tm0, tn, rows, ordinal);
                if (rows == 1 && !ring1) {
                    // First single-tile item: the rings overlap in memory, so every stage of the doubles'
                    // ring has to be released first (the stages below `stage` were last used in this
                    // round of the ring, the others in the round before; a fresh barrier passes).
                    for (int s = 0; s < STAGES && ok; ++s)
                        ok = mbar_wait_warp(bar_empty + 8 * s, ((uint32_t)s < stage) ? phase : (phase ^ 1u), cta_abort, p.dev_error);
                    if (!ok) break;
                    ring1 = true;
                    stage = 0;
                    phase = 0;
                }
                const uint32_t nst = ring1 ? (uint32_t)Cfg::STAGES1 : (uint32_t)STAGES;
                const uint32_t bfull = ring1 ? bar_full1 : bar_full, bempty = ring1 ? bar_empty1 : bar_empty;
                const uint32_t full0 = mapa(bfull, 0);  // the leader's barriers
                const int rb0 = tm0 * 2 + (int)rank;  // 128-row block of this CTA in the first row tile; the second: + 2
                const int n0 = tn * BN + (int)rank * Cfg::BN_CTA;
                const uint32_t tx = (rows == 2) ? (uint32_t)Cfg::STAGE_BYTES : (uint32_t)Cfg::SINGLE_TX;
                for (int kb = 0; kb < kblocks + lora_steps; ++kb) {
                    if (!mbar_wait_warp(bempty + 8 * stage, phase ^ 1, cta_abort, p.dev_error)) {
                        ok = false;
                        break;
                    }
                    const uint32_t a_dst = ring1 ? sA + Cfg::RING1_A + stage * Cfg::A_BYTES : sA + stage * 2 * Cfg::A_BYTES;
                    const uint32_t b_dst = ring1 ? sA + Cfg::RING1_B + stage * Cfg::B_BYTES : sB + stage * Cfg::B_BYTES;
                    const uint32_t e_dst = ring1 ? sA + Cfg::RING1_E + stage * Cfg::E_BYTES : sE + stage * 2 * Cfg::E_BYTES;
                    const uint32_t bar = full0 + 8 * stage;
                    if (!elect_one()) {
                    } else if (kb < kblocks) {
                        const bool pre = it == 0 && kb < npre;  // W tile and byte count went out before the wait
                        // the leader announces the bytes of both CTAs; the peer's bytes may land first
                        if (leader && !pre) mbar_arrive_expect_tx(bfull + 8 * stage, 2 * tx);
                        tma_load_2d_pair(a_dst, &tmap_a, kb * Cfg::BOX_X, rb0 * Cfg::BM, bar);
                        tma_load_2d_pair(e_dst, &tmap_e, 0, E_ROWS * (rb0 * kblocks + kb), bar);
                        if (!pre) {
                            tma_load_2d_pair(b_dst, &tmap_b, kb * Cfg::BK, n0, bar);
                            tma_load_2d_pair(b_dst + Cfg::B_HALF_BYTES, &tmap_b, kb * Cfg::BK + Cfg::BOX_X, n0, bar);
                        }
                        if (rows == 2) {
                            tma_load_2d_pair(a_dst + Cfg::A_BYTES, &tmap_a, kb * Cfg::BOX_X, (rb0 + 2) * Cfg::BM, bar);
                            tma_load_2d_pair(e_dst + Cfg::E_BYTES, &tmap_e, 0, E_ROWS * ((rb0 + 2) * kblocks + kb), bar);
                        }
                    } else {
                        // low-rank stages: T boxes in the A slots, L_A box in the first half of the W slot
                        const int j = kb - kblocks;
                        if (leader) mbar_arrive_expect_tx(bfull + 8 * stage, 2u * (uint32_t)(rows * Cfg::A_BYTES + Cfg::B_HALF_BYTES));
                        tma_load_2d_pair(a_dst, &tmap_t, j * 64, rb0 * Cfg::BM, bar);
                        if (rows == 2) tma_load_2d_pair(a_dst + Cfg::A_BYTES, &tmap_t, j * 64, (rb0 + 2) * Cfg::BM, bar);
                        tma_load_2d_pair(b_dst, &tmap_la, j * 64, n0, bar);
                    }
                    ++issued;
                    if (++stage == nst) { stage = 0; phase ^= 1; }
                }
            }
            // the last releases of the stages (see epilogue.cuh; a switch of the rings has waited for the other one's)
            const uint32_t nst = ring1 ? (uint32_t)Cfg::STAGES1 : (uint32_t)STAGES, bempty = ring1 ? bar_empty1 : bar_empty;
            for (uint32_t s = 0; s < nst && ok; ++s) {
                ok = mbar_wait_warp(bempty + 8 * stage, phase ^ 1, cta_abort, p.dev_error);
                if (++stage == nst) { stage = 0; phase ^= 1; }
            }
            if (!ok && issued) bounded_delay_ns(200000);  // let the copies in flight land before teardown
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer --------
        if (leader) {
            constexpr uint32_t idesc0 = make_idesc_sp_bf16(Cfg::BM * 2, BN), idesc1 = idesc0 | 1u;
            constexpr uint32_t idesc_dense = idesc0 & ~(1u << 2);
            const uint64_t d0 = make_desc_sw128(sA);
            const uint32_t desc_hi = (uint32_t)(d0 >> 32);
            const uint32_t ring_lo0 = (uint32_t)d0;                             // descriptor word of the ring's first byte
            const uint32_t b_lo0 = (uint32_t)make_desc_sw128(sB);
            const uint64_t e_d0 = make_desc_rows16(sE), e1_d0 = make_desc_rows16(sA + Cfg::RING1_E);
            constexpr uint32_t BH = Cfg::B_HALF_BYTES >> 4;
            constexpr uint32_t idesc8 = make_idesc_sp_e4m3(Cfg::BM * 2, BN);
            constexpr int E_HALF = Cfg::E_COLS / 2;  // metadata columns of one row tile
            uint32_t stage = 0, phase = 0;
            uint32_t e_slot = 0;  // FP8 doubles: the stage's metadata slot
            bool ring1 = false;
            AccTurns turns;
            bool ok = true;
            for (int it = 0; it < num_items && ok; ++it) {
                int tm0, tn, rows, ordinal;
                sched.item(cluster_id, it, tm0, tn, rows, ordinal);
                if (rows == 1 && !ring1) {  // the producer switches rings at the same item
                    ring1 = true;
                    stage = 0;
                    phase = 0;
                }
                const uint32_t nst = ring1 ? (uint32_t)Cfg::STAGES1 : (uint32_t)STAGES;
                const uint32_t bfull = ring1 ? bar_full1 : bar_full, bempty = ring1 ? bar_empty1 : bar_empty;
                // accumulators of this item: a double fills both, the k-th single accumulator k % 2
                const int acc0 = (rows == 2) ? 0 : (ordinal & 1);
                // (a double's second accumulator is waited for behind the first one's MMAs: the epilogue
                // hands them back one after the other)
                ok = mbar_wait_warp(bar_tempty + 8 * acc0, turns.fill(acc0), cta_abort, p.dev_error);
                if (!ok) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc0 * BN;
                const int ksteps = kblocks + lora_steps;
                uint32_t accumulate = 0;
                for (int kb = 0; kb < ksteps; ++kb) {
                    if (!mbar_wait_warp(bfull + 8 * stage, phase, cta_abort, p.dev_error)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a_lo = ring1 ? ring_lo0 + ((Cfg::RING1_A + stage * Cfg::A_BYTES) >> 4)
                                                : ring_lo0 + stage * (2 * Cfg::A_BYTES >> 4);
                    const uint32_t b_lo = ring1 ? ring_lo0 + ((Cfg::RING1_B + stage * Cfg::B_BYTES) >> 4)
                                                : b_lo0 + stage * (Cfg::B_BYTES >> 4);
                    if constexpr (Cfg::E_SLOTS < STAGES) {
                        if (!ring1) {
                            // the stage before the last one: with three stages the next one of the ring, a round back
                            // (a fresh barrier passes)
                            const uint32_t older = stage == STAGES - 1 ? 0u : stage + 1;
                            if (!mbar_wait_warp(bempty + 8 * older, older ? phase ^ 1u : phase, cta_abort, p.dev_error)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                            e_slot ^= 1u;
                        }
                    }
                    const uint32_t e_tmem = tmem_base + Cfg::E_COL0 +
                                            (ring1 ? E_HALF * stage : Cfg::E_COLS * (Cfg::E_SLOTS < STAGES ? e_slot : stage));
                    const uint64_t e_desc = ring1 ? e1_d0 + (uint64_t)(stage * (Cfg::E_BYTES >> 4))
                                                  : e_d0 + (uint64_t)(stage * (2 * Cfg::E_BYTES >> 4));
                    const bool sparse = kb < kblocks;
                    // one row tile's MMAs of this stage
                    auto issue = [&](int r) {
                        const uint32_t dt = d_tmem + r * BN, al = a_lo + r * (Cfg::A_BYTES >> 4), et = e_tmem + E_HALF * r;
                        if constexpr (Cfg::FP8) {
                            // four K steps of 64 logical elements: A advances 32 bytes, W 64 bytes, metadata two columns
                            mma_sp_f8_lh<2>(dt, al, b_lo, desc_hi, et, idesc8, accumulate);
                            mma_sp_f8_lh<2>(dt, al + 2, b_lo + 4, desc_hi, et + 2, idesc8, 1u);
                            mma_sp_f8_lh<2>(dt, al + 4, b_lo + BH, desc_hi, et + 4, idesc8, 1u);
                            mma_sp_f8_lh<2>(dt, al + 6, b_lo + BH + 4, desc_hi, et + 6, idesc8, 1u);
                        } else if (sparse) {
                            // four K steps of 32 logical elements: A advances 32 bytes, W 64 bytes (steps 2, 3 in
                            // the second 64-element slice); metadata column pair + step parity
                            mma_sp_bf16_lh<2>(dt, al, b_lo, desc_hi, et, idesc0, accumulate);
                            mma_sp_bf16_lh<2>(dt, al + 2, b_lo + 4, desc_hi, et, idesc1, 1u);
                            mma_sp_bf16_lh<2>(dt, al + 4, b_lo + BH, desc_hi, et + 2, idesc0, 1u);
                            mma_sp_bf16_lh<2>(dt, al + 6, b_lo + BH + 4, desc_hi, et + 2, idesc1, 1u);
                        } else {
                            // low-rank stage: dense K steps of 16 elements, both operands advance 32 bytes
                            mma_bf16_lh<2>(dt, al, b_lo, desc_hi, idesc_dense, accumulate);
                            mma_bf16_lh<2>(dt, al + 2, b_lo + 2, desc_hi, idesc_dense, 1u);
                            mma_bf16_lh<2>(dt, al + 4, b_lo + 4, desc_hi, idesc_dense, 1u);
                            mma_bf16_lh<2>(dt, al + 6, b_lo + 6, desc_hi, idesc_dense, 1u);
                        }
                    };
                    if (elect_one()) {
                        if (sparse) {
                            // (a row tile's 128 x 128 metadata blocks, one or two: four columns each)
#pragma unroll
                            for (int j = 0; j < E_HALF / 4; ++j) tmem_cp_128x128b<2>(e_tmem + 4 * j, e_desc + (uint64_t)(j * (2048 >> 4)));
                            if (rows == 2) {
#pragma unroll
                                for (int j = 0; j < E_HALF / 4; ++j)
                                    tmem_cp_128x128b<2>(e_tmem + E_HALF + 4 * j, e_desc + (uint64_t)((Cfg::E_BYTES + j * 2048) >> 4));
                            }
                        }
                        issue(0);
                        if (kb == ksteps - 1) tc_commit_pair(bar_tfull + 8 * acc0, 0x3);
                    }
                    if (rows == 2) {
                        if (kb == 0) {
                            if (!mbar_wait_warp(bar_tempty + 8, turns.fill(1), cta_abort, p.dev_error)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                        }
                        if (elect_one()) {
                            issue(1);
                            if (kb == ksteps - 1) tc_commit_pair(bar_tfull + 8, 0x3);
                        }
                    }
                    if (elect_one()) tc_commit_pair(bempty + 8 * stage, 0x3);
                    accumulate = 1u;
                    if (++stage == nst) { stage = 0; phase ^= 1; }
                }
            }
            for (int a = 0; a < 2 && ok; ++a)  // the last hand-backs (see epilogue.cuh)
                ok = mbar_wait_warp(bar_tempty + 8 * a, turns.fill(a), cta_abort, p.dev_error);
        }
    }
    } else {
        setmaxnreg_inc<GEMM_REGS_EPI>();
        // ------------------------------------------------------------------ epilogue ----------
        // Both warps of a lane quarter drain every accumulator.  An accumulator's five chunks are dealt
        // 3 + 2, a double's second accumulator 2 + 3, so a warp holds at most five chunks.
        const int h = (warp - GEMM_EPI_WARP0) >> 2;  // which of the quarter's two warps
        const int q = warp & 3;         // tensor-memory lane quarter this warp may read
        const uint32_t tempty0 = mapa(bar_tempty, 0);
        const uint32_t own_box = sC + (warp - GEMM_EPI_WARP0) * (Cfg::C_BYTES / Cfg::EPI_WARPS);
        constexpr int CH = Cfg::CH, NCH = Cfg::NCH;
        const int n_first = h == 0 ? 3 : 2;  // chunks of the item's first accumulator
        AccTurns turns;
        bool alive = true;
        for (int it = 0; it < num_items; ++it) {
            int tm0, tn, rows, ordinal;
            sched.item(cluster_id, it, tm0, tn, rows, ordinal);
            const bool last = it == num_items - 1;
            const int acc0 = (rows == 2) ? 0 : (ordinal & 1);
            // the item's bias values as fp32, for all epilogue warps (the other parity's may still be read)
            const uint32_t sb = sBias + (it & 1) * Cfg::BIAS_BYTES, sc = sb + BN * 4;
            if (const int c = (int)threadIdx.x - 32 * GEMM_EPI_WARP0; c < BN) {
                const int n = tn * BN + c;
                sts32f(sb + c * 4, (p.bias != nullptr && n < p.N) ? __uint_as_float((uint32_t)p.bias[n] << 16) : 0.0f);
                if constexpr (Cfg::FP8) sts32f(sc + c * 4, (p.col_scale != nullptr && n < p.N) ? p.col_scale[n] : 1.0f);
            }
            bar_sync_named(GEMM_EPI_BARRIER, 32 * Cfg::EPI_WARPS);  // every warp passes it once per item, whatever became of its waits
            if (!alive) continue;
            // the rows' scales (or their sums from the prune launch's partial sums) are fetched while
            // the main loop still runs
            const int m0 = (tm0 * 2 + (int)rank) * Cfg::BM + q * 32;  // this warp's rows in the first row tile; the second: + 256
            float s[2][4];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int64_t row = m0 + r * 256 + lane;
                float sl = 1.0f;
                if (r < rows && row < p.M) {
                    if (p.scale_partial != nullptr) sl = row_scale_from_partials(p.scale_partial, row, p.scale_ks);
                    else if (p.row_scale != nullptr) sl = p.row_scale[row];
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) s[r][i] = __shfl_sync(0xffffffffu, sl, 8 * i + (lane >> 2));
            }
            const int slots = rows == 2 ? NCH : n_first;
            // slot -> row tile of the item and chunk
            auto chunk_of = [&](int slot, int& r, int& c) {
                r = slot >= n_first;
                c = h == 0 ? (r ? slot - 3 : slot) : (r ? slot : 3 + slot);
            };
            // All chunks are converted to packed bf16 first, so an accumulator goes back after its
            // tensor-memory reads; the stores follow while the next main loop already runs.
            uint32_t packed[NCH][2][CH / 4];
            auto convert = [&](auto has_residual) {
                constexpr bool RES = decltype(has_residual)::value;
                if constexpr (RES) {  // the residual arrives during the main loop, in the registers of the results
#pragma unroll
                    for (int slot = 0; slot < NCH; ++slot) {
                        if (slot >= slots) break;
                        int r, c;
                        chunk_of(slot, r, c);
                        epi_load_residual<CH>(p.residual, p.ldr, m0 + r * 256, p.M, tn * BN + c * CH, p.N, lane, packed[slot]);
                    }
                }
#pragma unroll
                for (int slot = 0; slot < NCH; ++slot) {
                    if (slot >= slots || !alive) break;
                    int r, c;
                    chunk_of(slot, r, c);
                    const int acc = acc0 + r;
                    if (slot == 0 || slot == n_first) {
                        alive = mbar_wait_warp(bar_tfull + 8 * acc, turns.drain(acc), cta_abort, p.dev_error);
                        if (!alive) break;
                        tc_fence_after();
                    }
                    uint32_t v[2][CH / 2];
                    epi_tmem_ld<CH>(tmem_base + ((uint32_t)(q * 32) << 16) + acc * BN + c * CH, v);
                    tmem_ld_wait();
                    if (slot == n_first - 1 || slot == slots - 1) {
                        // this warp's share of the accumulator is read: hand it back to the MMA issuer
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(tempty0 + 8 * acc);
                    }
                    float sr[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) sr[i] = r ? s[1][i] : s[0][i];
                    epi_convert<CH, Cfg::FP8, RES>(v, sr, sb + c * (CH * 4), sc + c * (CH * 4), lane, packed[slot]);
                }
            };
            if (p.residual != nullptr) convert(std::true_type{});
            else convert(std::false_type{});
            if (!alive) continue;
            const long long t_store = clock64();
            const int pace = Cfg::store_pace(kblocks, p.residual != nullptr);
#pragma unroll
            for (int slot = 0; slot < NCH; ++slot) {
                if (slot >= slots) break;
                int r, c;
                chunk_of(slot, r, c);
                if (pace > 0 && !last) {
                    const long long at = t_store + (long long)(slot * Cfg::EPI_WARPS + warp - GEMM_EPI_WARP0) * pace;
                    for (int i = 0; i < 1000 && clock64() < at; ++i) __nanosleep(100);
                }
                const int n0 = tn * BN + c * CH;
                // rows past M and columns past N are clipped by the store.  The last item stages in the ring:
                // its MMAs are done (the wait above) and nothing is loaded any more.
                if (n0 < p.N)
                    epi_store<CH, Cfg::BOX_ROWS>(&tmap_y, packed[slot], n0, m0 + r * 256,
                                      last ? smem_base + ((warp - GEMM_EPI_WARP0) * NCH + slot) * Cfg::C_BOX_BYTES : own_box, last, lane);
            }
        }
        if (lane == 0) tma_store_wait_read<0>();  // (the end of the grid makes the stores visible)
    }

    // ---------------------------------------------------------------------- teardown ----------
    tc_fence_before();
    __syncthreads();
    cluster_sync_relaxed();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc<2>(tmem_base, Cfg::TMEM_COLS);
    }
}

}  // namespace lynx
