// The contractions of the codebook step (Section 4.2, Eq. 8) and their sums by level, one tensor-core kernel:
//
//     G^(j) = P^T H_k P   (m x m),     r^(j) = P^T H_k w_j        for every channel j of every group k,
//
// P the channel's one-hot assignment matrix, with nothing between the products and their sums by level.  A unit is (256 rows
// r of H, 256 columns (channel, level) of P) and computes D[column][r] = sum_c P[c][column] H[c][r] with the one-hot columns
// as the M side.  The tensor-memory load that hands a warp 16 accumulator rows in the layout of an m16n8k16 A operand then
// lets the sum over the rows of each level be a small product of its own: D (three bf16 terms, 24 bits, 16 rows r at a time,
// smallest term first) times the one-hot codes of r, added up in fp32 over 128 rows and in fp64 beyond.
// The one-hot operand never exists in global memory: one warp per stage writes it there.  A stage's previous ones are
// known to the lanes that wrote them, so a k-step costs two 2-byte stores per code (clear, set) instead of 16 KB.
// r comes from units of the same shape with A = W^T (by TMA) whose epilogue sums D[channel][r] by the code of r; these units
// come first.
//
// H and W enter as bf16 hi + lo (16 significant bits): H hi, then H lo, over the whole contraction for the one-hot columns;
// hi hi, lo hi (W lo), hi lo (H lo) for W.  What is dropped is below 2^-16 of each entry.  (Contracting over one triangle of
// H only, G = F + F^T, halves the work and was measured: 1.85 ms an update.  It was not kept: the tensor core's fp32
// accumulation truncates, with half as many additions the levels come out 1e-5 different, and 11 % of the codes of the next
// descent cycles with them.)
// Stage: [A | B], 16 KB each per CTA, of which only B comes through the L2.  What bounds the kernel is the tensor core and
// the thread that feeds it (695 clocks a k-step with the one-hot stores left out, 512 at the nominal rate) and shared-memory
// bandwidth (807 with them).  Measured, 4096 x 4096, 4 groups, 16 levels, one update: 3.7 ms = 1300 TFLOP/s with the issuing
// thread on warp 1, a tenth of a millisecond less on warp 3.  With the one-hot matrix, H P and H W^T in
// global memory it was 0.17 (one-hot) + 2.88 (H P) + 0.40 (H W^T) + 0.55 (sums by level) = 4.00 ms and 0.5 GB of scratch.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "gq_codebook.cuh"
#include "gq_pipeline.cuh"

namespace gq {

constexpr int CG_STAGES = 6;
constexpr int CG_SLOT_BYTES = (CTA_ROWS / BOX_FEATURES) * BOX_BYTES;      // one operand block: 16 KB
constexpr int CG_STAGE_BYTES = 2 * CG_SLOT_BYTES;                         // [A | B]
constexpr int CG_HOT_WARPS = CG_STAGES;                                   // write the one-hot operand, a stage each
constexpr int CG_EPI_WARPS = 8;
constexpr int CG_THREADS = 32 * (4 + CG_HOT_WARPS + CG_EPI_WARPS);
constexpr int CG_LEVEL_SUMS = CG_EPI_WARPS * CB_MAX_LEVELS * 32;          // fp32 [warp][level][lane]
constexpr int CG_SMEM_BYTES = CG_STAGES * CG_STAGE_BYTES + CG_LEVEL_SUMS * 4 + 1024;

struct CodebookGemmParams {
    const uint8_t *Q;        // [d_out][d]
    double *G;               // [d_out][16][16], added to
    double *R;               // [d_out][16], added to
    int d, d_out, g, mk, m;
    int row_blocks;          // ceil(d / 256)
    int w_tiles;             // ceil(mk / 256): tiles of 256 channels per group
    int hot_tiles;           // ceil(mk * MP / 256): tiles of 256 one-hot columns per group
    int w_units;             // row_blocks * g * w_tiles
    int units;               // w_units + row_blocks * g * hot_tiles
    int pairs;
    uint32_t *status;
    unsigned long long wait_budget_ns;
};

struct CodebookUnit {
    int ti;          // row block of H
    int k;           // group
    int tile;        // tile of one-hot columns / channels
    bool hot;        // one-hot columns (else W)
    int passes;      // over the contraction: one-hot: H hi, H lo; W: (W hi, H hi), (W lo, H hi), (W hi, H lo)
};

// The it-th unit of a pair: row blocks outermost, so that the pairs share a block of H in L2.
__device__ __forceinline__ bool codebook_unit(const CodebookGemmParams &p, int pair, int it, CodebookUnit &u)
{
    const int unit = it * p.pairs + pair;
    if (unit >= p.units) return false;
    u.hot = unit >= p.w_units;
    const int v = u.hot ? unit - p.w_units : unit, tiles = u.hot ? p.hot_tiles : p.w_tiles, per = p.g * tiles;
    u.ti = v / per;
    const int rest = v - u.ti * per;
    u.k = rest / tiles;
    u.tile = rest - u.k * tiles;
    u.passes = u.hot ? 2 : 3;
    return true;
}

// Tensor memory, 16 lanes x 32 columns: register 4 b + e of thread t holds lane t / 4 + (e >= 2 ? 8 : 0), column
// 8 b + 2 (t % 4) + (e & 1): for two neighbouring b the A operand of an m16n8k16 product.
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void mma_m16n8k16_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// x (low half) and y rounded to bf16; x and y become what is left of them.
__device__ __forceinline__ uint32_t take_bf16x2(float &x, float &y)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    const uint32_t bits = *reinterpret_cast<const uint32_t *>(&h);
    x -= __uint_as_float(bits << 16);
    y -= __uint_as_float(bits & 0xffff0000u);
    return bits;
}

// MP: one-hot columns per channel (4, 8 or 16, at least m; columns m .. MP - 1 stay zero).
// mapH0/1: H as bf16 hi / lo [g][d][d]; mapW0/1: W^T as bf16 hi / lo [d][d_out].
template <int MP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(CG_THREADS, 1)
codebook_gemm_kernel(const __grid_constant__ CUtensorMap mapH0, const __grid_constant__ CUtensorMap mapH1,
                     const __grid_constant__ CUtensorMap mapW0, const __grid_constant__ CUtensorMap mapW1,
                     const CodebookGemmParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[CG_STAGES];     // first CTA: bytes of both CTAs + the one-hot warps of both
    __shared__ __align__(8) uint64_t bar_empty[CG_STAGES];    // both CTAs: signalled by the MMA commits
    __shared__ __align__(8) uint64_t bar_acc_full[2];         // both CTAs, one per accumulator
    __shared__ __align__(8) uint64_t bar_acc_empty[2];        // first CTA, one per accumulator: 16 epilogue warps arrive
    __shared__ __align__(8) uint64_t bar_drain;
    __shared__ uint32_t tmem_base_smem;
    __shared__ volatile uint32_t abort_flag;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = static_cast<int>(blockIdx.x >> 1);
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;

    if (threadIdx.x == 0) {
        for (int s = 0; s < CG_STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1 + 2);         // bytes, and the stage's one-hot warp of either CTA
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&bar_acc_full[b]), 1);
            mbar_init(smem_u32(&bar_acc_empty[b]), 2 * CG_EPI_WARPS);
        }
        mbar_init(smem_u32(&bar_drain), 1);
        abort_flag = 0u;
        fence_mbar_init();
        prefetch_tensormap(&mapH0);
        prefetch_tensormap(&mapH1);
        prefetch_tensormap(&mapW0);
        prefetch_tensormap(&mapW1);
    }
    griddep_launch();
    if (warp == 2) {
        tmem_alloc(smem_u32(&tmem_base_smem), TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    cluster_sync_all();
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_base_smem;
    const WaitCtx wc{&abort_flag, p.status, p.wait_budget_ns};
    griddep_wait();
    const int kblocks = (p.d + TILE_K - 1) / TILE_K;

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------------------------ TMA producer (both CTAs)
        int s = 0;
        uint32_t ph = 0;
        uint32_t issued = 0;
        bool ok = true;
        CodebookUnit u;
        for (int it = 0; ok && codebook_unit(p, pair, it, u); ++it) {
            const int b0 = u.ti * TILE_N + static_cast<int>(rank) * CTA_ROWS;
            const int a0 = u.k * p.mk + u.tile * TILE_M + static_cast<int>(rank) * CTA_ROWS;      // W units: first channel
            for (int pass = 0; ok && pass < u.passes; ++pass) {
                const void *bmap = (pass == u.passes - 1) ? &mapH1 : &mapH0;
                const void *amap = (pass == 1) ? &mapW1 : &mapW0;
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!bounded_wait(smem_u32(&bar_empty[s]), ph ^ 1u, wc, 1u, it)) { ok = false; break; }
                    const uint32_t full_local = smem_u32(&bar_full[s]);
                    if (rank == 0) mbar_arrive_expect_tx(full_local, (u.hot ? 2 : 4) * CG_SLOT_BYTES);      // both CTAs' bytes
                    const uint32_t full = map_to_cta(full_local, 0);
                    const uint32_t stage = ring + s * CG_STAGE_BYTES;
#pragma unroll
                    for (int q = 0; q < CTA_ROWS / BOX_FEATURES; ++q) {
                        tma_load_3d_pair(stage + CG_SLOT_BYTES + q * BOX_BYTES, bmap, full, b0 + q * BOX_FEATURES, kb * TILE_K, u.k);
                        if (!u.hot) tma_load_3d_pair(stage + q * BOX_BYTES, amap, full, a0 + q * BOX_FEATURES, kb * TILE_K, 0);
                    }
                    ++issued;
                    if (++s == CG_STAGES) { s = 0; ph ^= 1u; }
                }
            }
        }
        // Stay until every stage has been released again: the release is an arrival on this CTA's barriers,
        // which must not come after the CTA has gone.
        for (int q = 0; ok && issued != 0u && q < CG_STAGES; ++q) {
            if (!bounded_wait(smem_u32(&bar_empty[s]), ph ^ 1u, wc, 5u, 0u)) ok = false;
            if (++s == CG_STAGES) { s = 0; ph ^= 1u; }
        }
        if (!ok) spin_ns(1000000ull);
    } else if (warp == 3 && lane == 0 && rank == 0) {
        // ------------------------------------------------------------------ MMA issuer (first CTA)
        // Warp 3: what this thread does between two k-steps the tensor core waits for, and warps 4 w + 1 on its scheduler include
        // two of the one-hot warps, warps 4 w + 3 one.  gq_lnq with two updates, 4096 x 4096, 16 levels: 10.11 -> 9.89 ms with
        // warp 1 -> 3, both sides in turn; six other layers 0 to 2.4 % faster.
        constexpr uint32_t idesc = umma_idesc_bf16_mn(TILE_M, TILE_N);
        int s = 0;
        uint32_t ph = 0;
        uint32_t acc_ph = 0u;                           // bit b: phase of accumulator b
        int buf = 0;
        bool ok = true;
        CodebookUnit u;
        for (int it = 0; ok && codebook_unit(p, pair, it, u); ++it) {
            if (!bounded_wait_hot(smem_u32(&bar_acc_empty[buf]), ((acc_ph >> buf) & 1u) ^ 1u, wc, 2u, it)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * TILE_N);
            const int ksteps = u.passes * kblocks;
            for (int ks = 0; ks < ksteps; ++ks) {
                if (!bounded_wait_hot(smem_u32(&bar_full[s]), ph, wc, 3u, it)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t sa = ring + s * CG_STAGE_BYTES;
                const uint32_t sb = sa + CG_SLOT_BYTES;
#pragma unroll
                for (int k16 = 0; k16 < TILE_K / 16; ++k16) {
                    const uint64_t adesc = umma_smem_desc_mn_sw128(sa + k16 * 16 * 128, BOX_BYTES, 1024);
                    const uint64_t bdesc = umma_smem_desc_mn_sw128(sb + k16 * 16 * 128, BOX_BYTES, 1024);
                    umma_bf16(d_tmem, adesc, bdesc, idesc, (ks != 0 || k16 != 0) ? 1u : 0u);
                }
                umma_commit_pair(smem_u32(&bar_empty[s]));
                if (++s == CG_STAGES) { s = 0; ph ^= 1u; }
            }
            if (!ok) break;
            umma_commit_pair(smem_u32(&bar_acc_full[buf]));
            acc_ph ^= 1u << buf;
            buf ^= 1;
        }
        if (!ok) {
            // Make sure no MMA is still writing TMEM when it is released.
            umma_commit_local(smem_u32(&bar_drain));
            const uint64_t t0 = global_timer_ns();
            while (!mbar_try_wait(smem_u32(&bar_drain), 0u) && global_timer_ns() - t0 < 5000000ull) {}
        }
    } else if (warp >= 4 && warp < 4 + CG_HOT_WARPS) {
        // ------------------------------------------------------------------ one-hot operand
        // One warp per stage: it waits for its stage, clears the ones it set there last (their codes stay in registers), sets
        // the new ones and signals.  A lane owns one channel and MY_ROWS of the 64 contraction rows; codes are read when the
        // previous ones have been used, six k-steps ahead.  (One set of four warps working on every stage in turn took
        // 1700 clocks a k-step, most of it waiting for its own stores to be visible: 5.3 ms an update.)
        constexpr int CHANNELS = CTA_ROWS / MP;                 // channels of this CTA's 128 columns
        constexpr int MY_ROWS = TILE_K * CHANNELS / 32;         // 16, 32 or 64
        constexpr int WORDS = MY_ROWS / 4;
        const int stage = warp - 4;
        const int ch = lane % CHANNELS, rloc = (lane / CHANNELS) * MY_ROWS;
        const uint32_t sa = ring + stage * CG_STAGE_BYTES;
        const uint32_t flip = static_cast<uint32_t>(lane >> 3) & 3u;         // lanes of a bank start on different rows
        const uint32_t top = static_cast<uint32_t>(p.m - 1) * 0x01010101u;
        // 2-byte element (row, column) of the block, swizzled as a TMA load would have left it
        auto at = [&](int row, int col) {
            return sa + static_cast<uint32_t>((col >> 6) * BOX_BYTES + row * 128 + ((((col >> 3) & 7) ^ (row & 7)) << 4) + (col & 7) * 2);
        };
        uint32_t old[WORDS], cur[WORDS];
        bool fresh = true;                                      // the stage has not held one-hot columns yet
        uint32_t ph = 0;
        int offset = stage;                                     // this warp's first k-step of the next unit
        bool ok = true;
        CodebookUnit u;
        for (int it = 0; ok && codebook_unit(p, pair, it, u); ++it) {
            const int jl = u.tile * (TILE_M / MP) + static_cast<int>(rank) * CHANNELS + ch;      // channel in the group
            const bool have = u.hot && jl < p.mk;
            const uint8_t *q_row = p.Q + static_cast<size_t>(u.k * p.mk + (have ? jl : 0)) * p.d;
            const int ksteps = u.passes * kblocks;
            // codes of a k-step, eight at a time (rows are a multiple of 8); 0xff where there is none, others at most m - 1
            auto fetch = [&](int ks) {
                const int row0 = (ks % kblocks) * TILE_K + rloc;
#pragma unroll
                for (int w = 0; w < WORDS; w += 2) {
                    uint2 v = make_uint2(0xffffffffu, 0xffffffffu);
                    if (have && ks < ksteps && row0 + 4 * w < p.d) {
                        v = ld_u32x2(q_row + row0 + 4 * w);
                        v.x = __vminu4(v.x, top);
                        v.y = __vminu4(v.y, top);
                    }
                    cur[w] = v.x;
                    cur[w + 1] = v.y;
                }
            };
            fetch(offset);
            int ks = offset;
            for (; ks < ksteps; ks += CG_STAGES) {
                bool got = true;
                if (lane == 0) got = bounded_wait(smem_u32(&bar_empty[stage]), ph ^ 1u, wc, 6u, it);
                got = __any_sync(0xffffffffu, got && lane == 0);
                if (!got) { ok = false; break; }
                (void)mbar_try_wait(smem_u32(&bar_empty[stage]), ph ^ 1u);       // every lane observes the completed phase
                ph ^= 1u;
                if (u.hot) {
                    auto put = [&](uint32_t word, int w, int r, unsigned short v) {
                        const uint32_t rr = static_cast<uint32_t>(r) ^ flip, code = (word >> (8u * rr)) & 0xffu;
                        if (code < static_cast<uint32_t>(MP))
                            asm volatile("st.shared.u16 [%0], %1;" ::"r"(at(rloc + 4 * w + static_cast<int>(rr), ch * MP + static_cast<int>(code))),
                                         "h"(v) : "memory");
                    };
                    if (fresh) {
                        // the whole block: 512 bytes per lane
                        fresh = false;
#pragma unroll 4
                        for (int i = lane; i < CG_SLOT_BYTES / 16; i += 32) st_shared_16(sa + 16u * i, make_uint4(0u, 0u, 0u, 0u));
                        __syncwarp();
                    } else {
#pragma unroll
                        for (int w = 0; w < WORDS; ++w)
#pragma unroll
                            for (int r = 0; r < 4; ++r) put(old[w], w, r, 0);
                    }
#pragma unroll
                    for (int w = 0; w < WORDS; ++w) {
#pragma unroll
                        for (int r = 0; r < 4; ++r) put(cur[w], w, r, 0x3F80);
                        old[w] = cur[w];
                    }
                    fetch(ks + CG_STAGES);
                    fence_proxy_async_smem();        // make the stores visible to the tensor core's reads
                }
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_full[stage]), 0));
            }
            offset = ks - ksteps;
        }
    } else if (warp >= 4 + CG_HOT_WARPS) {
        // ------------------------------------------------------------------ epilogue: sums by level
        const int ew = warp - (4 + CG_HOT_WARPS);       // 0..7; four consecutive warps cover the four lane quarters
        const int q = warp & 3;                         // TMEM lane quarter this warp may access
        const int half = ew >> 2;                       // which 128 of the 256 rows of H
        const int t4 = lane & 3, g8 = lane >> 2;
        float *level_sums = reinterpret_cast<float *>(smem_raw + (ring - smem_u32(smem_raw)) + CG_STAGES * CG_STAGE_BYTES) +
                            ew * CB_MAX_LEVELS * 32 + lane;
        uint32_t full_ph = 0u;                          // bit b: phase of accumulator b
        int buf = 0;
        bool ok = true;
        CodebookUnit u;
        for (int it = 0; ok && codebook_unit(p, pair, it, u); ++it) {
            if (lane == 0) ok = bounded_wait(smem_u32(&bar_acc_full[buf]), (full_ph >> buf) & 1u, wc, 4u, it);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            (void)mbar_try_wait(smem_u32(&bar_acc_full[buf]), (full_ph >> buf) & 1u);     // every lane observes the completed phase
            full_ph ^= 1u << buf;
            tc_fence_after_sync();
            const uint32_t tmem_tile = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                                       static_cast<uint32_t>(buf * TILE_N + half * 128);
            const int row0 = u.ti * TILE_N + half * 128;                         // first row of H of this warp
            if (u.hot) {
#pragma unroll 1
                for (int hh = 0; hh < 2; ++hh) {                                 // 16 accumulator rows: 16 / MP channels
                    const int col0 = u.tile * TILE_M + static_cast<int>(rank) * CTA_ROWS + q * 32 + hh * 16;
                    const int j0 = col0 / MP;                                    // first of their channels, in the group
                    // channel and level of operand column g8 in the two blocks of eight
                    const int jb[2] = {j0 + (MP == 16 ? 0 : MP == 8 ? 0 : g8 >> 2), j0 + (MP == 16 ? 0 : MP == 8 ? 1 : 2 + (g8 >> 2))};
                    const uint32_t lv[2] = {static_cast<uint32_t>(g8 & (MP - 1)),
                                            static_cast<uint32_t>(MP == 16 ? g8 + 8 : g8 & (MP - 1))};
                    const uint8_t *qb[2];
#pragma unroll
                    for (int b = 0; b < 2; ++b) qb[b] = p.Q + static_cast<size_t>(u.k * p.mk + (jb[b] < p.mk ? jb[b] : 0)) * p.d;
                    float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 1
                    for (int n0 = 0; n0 < 128; n0 += 32) {
                        uint32_t raw[16];
                        tmem_ld_16x256b_x4(tmem_tile + (static_cast<uint32_t>(hh * 16) << 16) + static_cast<uint32_t>(n0), raw);
                        // codes of the rows this thread's registers stand for (rows past the matrix: D is 0)
                        uint32_t code[2][4];
#pragma unroll
                        for (int x = 0; x < 4; ++x) {
                            const int row = row0 + n0 + 8 * x + 2 * t4;
                            const bool in = row < p.d;
#pragma unroll
                            for (int b = 0; b < 2; ++b) {
                                code[b][x] = in ? ld_u16(qb[b] + row) : 0u;
                            }
                        }
                        tmem_ld_wait();
                        const uint32_t top = static_cast<uint32_t>(p.m - 1);
#pragma unroll
                        for (int x = 0; x < 4; x += 2) {                         // 16 rows: one contraction step
                            float v[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(raw[4 * x + e]);
                            uint32_t b0[2], b1[2];
#pragma unroll
                            for (int b = 0; b < 2; ++b) {
                                auto hot = [&](uint32_t two) {                   // two codes -> two bf16 0 / 1
                                    const uint32_t c0 = min(two & 0xffu, top), c1 = min(two >> 8, top);
                                    return (c0 == lv[b] ? 0x3F80u : 0u) | (c1 == lv[b] ? 0x3F800000u : 0u);
                                };
                                b0[b] = hot(code[b][x]);
                                b1[b] = hot(code[b][x + 1]);
                            }
                            uint32_t a[3][4];
#pragma unroll
                            for (int term = 0; term < 3; ++term)
#pragma unroll
                                for (int e = 0; e < 4; ++e) a[term][e] = take_bf16x2(v[2 * e], v[2 * e + 1]);
#pragma unroll
                            for (int b = 0; b < 2; ++b) {
                                float s16[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                                for (int term = 2; term >= 0; --term) mma_m16n8k16_bf16(s16, a[term], b0[b], b1[b]);
#pragma unroll
                                for (int e = 0; e < 4; ++e) c[b][e] += s16[e];
                            }
                        }
                    }
                    if (hh == 1) {
                        // This warp holds all it needs from the accumulator: hand it back to the MMA issuer (first CTA).
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_acc_empty[buf]), 0));
                    }
#pragma unroll
                    for (int b = 0; b < 2; ++b)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int arow = g8 + (e >= 2 ? 8 : 0), n = 2 * t4 + (e & 1);
                            const int chan = MP == 16 ? 0 : MP == 8 ? b : 2 * b + (n >> 2);
                            const int level = MP == 16 ? n + 8 * b : n & (MP - 1);
                            const int j = j0 + chan;
                            if (arow / MP == chan && j < p.mk)
                                atomicAdd(p.G + (static_cast<size_t>(u.k * p.mk + j) * CB_MAX_LEVELS + level) * CB_MAX_LEVELS +
                                              (arow & (MP - 1)), static_cast<double>(c[b][e]));
                        }
                }
            } else {
                // lane = channel; D[channel][row] added to the channel's sum for the code of the row
                const int jl = u.tile * TILE_M + static_cast<int>(rank) * CTA_ROWS + q * 32 + lane;
                const bool have = jl < p.mk;
                const size_t j = static_cast<size_t>(u.k * p.mk + (have ? jl : 0));
                const uint8_t *q_row = p.Q + j * p.d;
#pragma unroll
                for (int l = 0; l < CB_MAX_LEVELS; ++l) level_sums[l * 32] = 0.0f;
#pragma unroll 1
                for (int n0 = 0; n0 < 128; n0 += 32) {
                    uint32_t r[32];
                    tmem_ld_32x32(tmem_tile + static_cast<uint32_t>(n0), r);
                    uint2 codes[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int row = row0 + n0 + 8 * x;
                        codes[x] = row < p.d ? ld_u32x2(q_row + row) : make_uint2(0u, 0u);
                    }
                    tmem_ld_wait();
#pragma unroll
                    for (int x = 0; x < 4; ++x)
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            const uint32_t raw = ((e < 4 ? codes[x].x : codes[x].y) >> (8 * (e & 3))) & 0xffu;
                            const uint32_t code = min(raw, static_cast<uint32_t>(p.m - 1));
                            level_sums[code * 32] += __uint_as_float(r[8 * x + e]);
                        }
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_acc_empty[buf]), 0));
                if (have)
                    for (int l = 0; l < p.m; ++l) atomicAdd(p.R + j * CB_MAX_LEVELS + l, static_cast<double>(level_sums[l * 32]));
            }
            buf ^= 1;
        }
    }

    __syncwarp();
    tc_fence_before_sync();
    cluster_sync_all();
    if (warp == 2) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

}  // namespace gq
