// Epilogue pieces shared by the two sparse GEMM kernels: accumulator chunk -> scale, bias, residual ->
// packed bf16 registers -> staging box -> TMA store.
//
// What bounds it.  A launch's last tile has nothing left to hide its epilogue behind, and the 512-row
// items of the two-row-tile kernel hold both accumulators until theirs are read.  With four warps per
// tile, a shuffle per bias value and one staging box per warp, the epilogue of a 128 x 192 tile took
// 5300 cycles on an idle GPU and 8100 with every SM storing (13500 with a residual, whose loads were
// fetched chunk by chunk).  Hence: eight warps per tile (two per tensor-memory lane quarter); all chunks of
// a warp converted to packed bf16 registers before the first is stored (the accumulator goes back
// after the tensor-memory reads); packed fp32 multiply-adds; the residual fetched into the output registers
// during the main loop and replaced there; and for the last item a staging box per chunk in the ring's
// memory, which nothing uses any more, so that no store waits for another.
//
// Layout.  The accumulators are read in the 16 x 256-bit shape: of a 16-row x 8-column block lane t holds rows
// t / 4 and t / 4 + 8, columns 2 (t % 4) and + 1.  A lane then needs two bias values per eight columns
// for its four rows; in the row-per-lane shape every lane needs every column's value, and those broadcast
// loads alone occupied the shared memory for 1900 cycles per 512 x 240 item.  The blocks go to the
// staging box with stmatrix.
//
// The next launch.  The single-tile kernel lets it begin (griddepcontrol.launch_dependents) when its last tile's MMAs are done, in
// the layer calls whose own prune kernel has one block per SM: what follows, in a chain of them, is such a kernel, and its
// prologue then runs as the SMs become free, under the last epilogues.  These are the low-rank layers (rank 64: 299 x 3840 x 3840
// 21.6 -> 21.1 us, 936 x 3072 x 3072 22.2 -> 21.5) and FP8 layers of K >= 2048 (299 x 2048 x 3840 10.3 -> 9.8, 936 x 2816 x
// 3072 13.2 -> 12.7, 936 x 2304 x 9216 19.4 -> 18.9).  Shorter FP8 rows are pruned in blocks of 16 rows, which, like the small
// blocks of the plain layer's prune kernel, pile up on the SMs that leave first: 936 x 1792 x 3072 12.1 -> 14.2, 600 x 1024 x 3072
// 9.1 -> 10.1, 4352 x 1536 x 3072 22.7 -> 23.7, plain 936 x 3072 x 3072 16.1 -> 17.0.  Nor is it used in the two-row-tile kernel
// (low-rank: no difference; FP8 4096 x 12288 x 3072 105.0 -> 106.2).
#pragma once

#include "ptx.cuh"

namespace lynx {

constexpr int GEMM_EPI_WARPS = 8;
constexpr int GEMM_EPI_WARP0 = 4;         // first epilogue warp: the producer, the issuer and two idle warps come before
constexpr uint32_t GEMM_EPI_BARRIER = 1;  // named barrier of the epilogue warps
constexpr int GEMM_THREADS = 32 * (GEMM_EPI_WARP0 + GEMM_EPI_WARPS);
// Register shares (per thread) of the two kinds of warpgroups; 128 * 72 + 256 * 216 = the 384 * 168 the block is
// launched with.  An epilogue warp holds up to five packed chunks beside the one it converts.
constexpr int GEMM_REGS_ISSUE = 72, GEMM_REGS_EPI = 216;
// Do the shares fit what a block launched with `regs` registers per thread owns?  If not, the epilogue's
// setmaxnreg.inc waits for ever; how many a kernel is launched with is the compiler's choice, so the host asks
// the built kernel before its first launch.
constexpr bool gemm_register_shares_fit(int regs) {
    return 128 * GEMM_REGS_ISSUE + 32 * GEMM_EPI_WARPS * GEMM_REGS_EPI <= GEMM_THREADS * regs;
}
static_assert(gemm_register_shares_fit(65536 / GEMM_THREADS / 8 * 8), "register pool of the block");

// Whose turn an accumulator buffer is: the issuer fills it once its previous contents were handed back, the
// epilogue drains it once it is filled, and each of its two barriers completes one phase per use.  fill() is the parity
// of the hand-back barrier that lets the issuer fill the buffer (a fresh barrier passes), drain() that of the barrier
// that tells the epilogue that it is filled.
//
// After its last item the issuer waits for every buffer once more, as if it were to fill it again.  The hand-backs
// of CTA 1's epilogue warps are remote arrives on a barrier of CTA 0; without that wait nothing orders the last
// of them before CTA 0 leaves and its shared memory is given away.  The producers do the same with the ring's stages,
// whose release is a commit that arrives on both CTAs' barriers.  What they wait for comes before the epilogue's last
// stores: 6302 x 640 x 3496 GEMM 26.2 us without, 26.0 with.  (Only the launches that compute the down projection
// themselves feel it: the rank-64 GROUP layer of that size 38.4 -> 38.9.)

// Buffers in turn, item i uses i % BUFFERS: the single-tile kernel.
template <int BUFFERS>
struct CyclicTurn {
    int buffer;
    uint32_t odd;  // uses of the buffer before this item, mod 2
    __host__ __device__ explicit CyclicTurn(int item)
        : buffer(BUFFERS == 2 ? (item & 1) : 0), odd((uint32_t)(BUFFERS == 2 ? (item >> 1) : item) & 1u) {}
    __host__ __device__ uint32_t fill() const { return odd ^ 1u; }
    __host__ __device__ uint32_t drain() const { return odd; }
};

// Any order of use: the two-row-tile kernel.  Bit a of the word is the number of uses of buffer a so far, mod 2 (a bit
// each: an array with a run-time index lives in local memory).
struct AccTurns {
    uint32_t odd = 0;
    __host__ __device__ uint32_t fill(int a) {
        const uint32_t parity = ((odd >> a) & 1u) ^ 1u;
        odd ^= 1u << a;
        return parity;
    }
    __host__ __device__ uint32_t drain(int a) {
        const uint32_t parity = (odd >> a) & 1u;
        odd ^= 1u << a;
        return parity;
    }
};

// One 32-row x CH-column chunk: v[half][4 g + 2 k + e] = row 16 half + 8 k + lane / 4, column 8 g + 2 (lane % 4) + e
template <int CH>
__device__ __forceinline__ void epi_tmem_ld(uint32_t taddr, uint32_t (&v)[2][CH / 2]) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        const uint32_t t = taddr + ((uint32_t)(16 * half) << 16);
        if constexpr (CH == 64) {
            tmem_ld_16x256b_x8(t, v[half]);
        } else {
            tmem_ld_16x256b_x4(t, *reinterpret_cast<uint32_t(*)[16]>(&v[half][0]));
            tmem_ld_16x256b_x2(t + 32, *reinterpret_cast<uint32_t(*)[8]>(&v[half][16]));
        }
    }
}

// The chunk's residual values in the layout of the packed results (columns past N and rows past M: zero)
template <int CH>
__device__ __forceinline__ void epi_load_residual(const uint16_t* residual, int64_t ldr, int64_t row0, int64_t M, int n0, int64_t N,
                                                  int lane, uint32_t (&out)[2][CH / 4]) {
#pragma unroll
    for (int half = 0; half < 2; ++half)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int64_t row = row0 + 16 * half + 8 * k + (lane >> 2);
            const uint16_t* src = residual + row * ldr + n0 + 2 * (lane & 3);
#pragma unroll
            for (int g = 0; g < CH / 8; ++g)
                out[half][2 * g + k] = (row < M && n0 + 8 * g < N) ? *reinterpret_cast<const uint32_t*>(src + 8 * g) : 0u;
        }
}

// out[half][2 g + k] = bf16(fma(s [* col_scale], v, bias) [+ the residual that `out` holds]); s[2 half + k]: the
// lane's rows' scales; sb / sc: shared-memory addresses of the chunk's fp32 bias values and weight scales.
template <int CH, bool COL_SCALE, bool RES>
__device__ __forceinline__ void epi_convert(const uint32_t (&v)[2][CH / 2], const float (&s)[4], uint32_t sb, uint32_t sc, int lane,
                                            uint32_t (&out)[2][CH / 4]) {
    const uint32_t col = 8 * (lane & 3);
#pragma unroll
    for (int g = 0; g < CH / 8; ++g) {
        const uint64_t b = lds64(sb + g * 32 + col);
        uint64_t c = 0;
        if constexpr (COL_SCALE) c = lds64(sc + g * 32 + col);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int half = i >> 1, k = i & 1;
            uint64_t m = pack_f32x2(s[i], s[i]);
            if constexpr (COL_SCALE) m = mul_f32x2(m, c);
            uint64_t y = fma_f32x2(m, pack_b32x2(v[half][4 * g + 2 * k], v[half][4 * g + 2 * k + 1]), b);
            if constexpr (RES) {
                const uint32_t r = out[half][2 * g + k];
                y = add_f32x2(y, pack_f32x2(bf16_lo_f(r), bf16_hi_f(r)));
            }
            out[half][2 * g + k] = pack_bf16x2_of(y);
        }
    }
}

// One chunk to the output through a staging box of shared memory (64-column boxes: 128-byte rows with the
// 128-byte swizzle; 48: dense 96-byte rows).  BOX_ROWS: rows of the tensor map's box and of the warp's own box.
// fresh: `box` holds 32 rows and nothing has used it; else it is the warp's own, whose previous store must have read it.
template <int CH, int BOX_ROWS>
__device__ __forceinline__ void epi_store(const CUtensorMap* tmap, const uint32_t (&o)[2][CH / 4], int n0, int m0, uint32_t box,
                                          bool fresh, int lane) {
    constexpr int ROW_BYTES = CH * 2;
    // lane l addresses row l % 8 of 8 x 8 matrix l / 8: rows 0-7 and 8-15 of column group g, then of g + 1
    const uint32_t r = (lane & 7) + (lane & 8), gl = lane >> 4;
    auto put = [&](const uint32_t (&h)[CH / 4], uint32_t base) {
#pragma unroll
        for (int g = 0; g < CH / 8; g += 2)
            stmatrix_x4(base + r * ROW_BYTES + ((CH == 64 ? ((g + gl) ^ (r & 7)) : (g + gl)) << 4), h[2 * g], h[2 * g + 1], h[2 * g + 2],
                        h[2 * g + 3]);
    };
    if (fresh || BOX_ROWS == 32) {
        if (!fresh) {
            if (lane == 0) tma_store_wait_read<0>();
            __syncwarp();
        }
        put(o[0], box);
        put(o[1], box + 16 * ROW_BYTES);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < 32; i += BOX_ROWS) tma_store_2d(tmap, n0, m0 + i, box + i * ROW_BYTES);
            tma_store_commit();
        }
        return;
    }
#pragma unroll
    for (int half = 0; half < 2; ++half) {  // 16-row boxes
        if (lane == 0) tma_store_wait_read<0>();
        __syncwarp();
        put(o[half], box);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
            tma_store_2d(tmap, n0, m0 + 16 * half, box);
            tma_store_commit();
        }
    }
}

}  // namespace lynx
