// Cyclic coordinate descent with fixed codebooks on the guided layer objective
// (Section 4.2, Eq. 10; Appendix B.2, Algorithms 3 and 4): the kernels around the tensor-core panel product.
//
// For every group k and channel j in J_k, coordinates i = 0 .. d_in - 1 in order are set to
//     Round_j( W_ij - (1 / H_ii) * sum_{c != i} H_ic * E_cj ),     E = What - W  (current values),
// all channels in parallel.  The coordinates are processed in blocks of CD_BLOCK = 256 (the lazy batch of
// Algorithm 4).  For a block starting at s0 the sum splits into
//   - c outside the block: one tensor-core product per block, P = H[block rows, outside] * E[outside]
//     (pair_gemm_kernel<MODE_PANEL>); rows before the block already hold this cycle's values, rows after it
//     the previous cycle's - exactly what Algorithm 4's B holds for these rows when the block is reached;
//   - c inside the block: done here, sequentially, by cd_block_kernel.
// (Algorithm 4 pushes a finished block's correction to all later rows; here every block pulls the
// contributions of all other rows just before it is processed.  The sums are the same; only their order
// differs, and B never has to exist for more than one block.)
//
// Work arrays are coordinate-major ([d_in][d_out], the paper's orientation) so that one coordinate of all
// channels is contiguous; W, What and the codes are transposed on the way in and out.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "gq_pipeline.cuh"

namespace gq {

constexpr int CD_BLOCK = 256;           // coordinates per block
constexpr int CD_BAND = 32;             // coordinates whose running sums one chain thread holds
constexpr int CD_BANDS = CD_BLOCK / CD_BAND;
constexpr int CD_THREADS = 256;
constexpr int CD_MAX_LEVELS = 16;       // codebook entries per channel (m = 2^b, b <= 4)
constexpr int CD_LEVEL_LD = CD_MAX_LEVELS + 1;   // padded per-channel rows of the level tables
constexpr int CD_H_BUFS = 3;
constexpr int CD_H_FLOATS = CD_BLOCK * CD_BAND;          // one [256][32] tile of H: 32 KB
constexpr int CD_PARTS = 6;             // pieces of the contraction range of a band's pulled sums
// CH: channels per CTA of the block kernel, 32 or 16; a lane of the chain warp each
constexpr int cd_smem_bytes(int CH)
{
    return (3 * CD_BLOCK * CH + CD_H_BUFS * CD_H_FLOATS + CD_PARTS * CD_BAND * CH + CD_BLOCK + 3 * CH * CD_LEVEL_LD) * 4 + 1024;
}

__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16 &hi, __nv_bfloat16 &lo)
{
    hi = __float2bfloat16_rn(v);
    lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// Wt = W^T, E = (What - W)^T (fp32 and as bf16 hi + lo), all [d_in][d_out].  Tiles of 32 coordinates x 64 channels: whole
// 128-byte segments on both sides (4096 x 4096: 51 us; one value per lane and 64-byte segments 73).
__global__ void __launch_bounds__(256)
cd_prepare_kernel(const float *W, const float *What, int d_in, int d_out, float *Wt, float *Et, __nv_bfloat16 *Ehi, __nv_bfloat16 *Elo)
{
    __shared__ float tw[64][33], th[64][33];
    griddep_launch();
    griddep_wait();
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 64;          // coordinate / channel origin
#pragma unroll
    for (int r = 0; r < 64; r += 8) {
        const int j = j0 + r + ty, i = i0 + tx;
        const bool ok = j < d_out && i < d_in;
        tw[r + ty][tx] = ok ? W[static_cast<size_t>(j) * d_in + i] : 0.0f;
        th[r + ty][tx] = ok ? What[static_cast<size_t>(j) * d_in + i] : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 32; r += 8) {
        const int i = i0 + r + ty, j = j0 + 2 * tx;                // d_out is a multiple of 8: pairs are inside or outside
        if (i < d_in && j < d_out) {
            const float w0 = tw[2 * tx][r + ty], w1 = tw[2 * tx + 1][r + ty];
            const float e0 = th[2 * tx][r + ty] - w0, e1 = th[2 * tx + 1][r + ty] - w1;
            const size_t o = static_cast<size_t>(i) * d_out + j;
            *reinterpret_cast<float2 *>(Wt + o) = make_float2(w0, w1);
            *reinterpret_cast<float2 *>(Et + o) = make_float2(e0, e1);
            const __nv_bfloat162 hi = __floats2bfloat162_rn(e0, e1);
            *reinterpret_cast<__nv_bfloat162 *>(Ehi + o) = hi;
            *reinterpret_cast<__nv_bfloat162 *>(Elo + o) = __floats2bfloat162_rn(e0 - __low2float(hi), e1 - __high2float(hi));
        }
    }
}

// H -> bf16 hi + lo and rdiag[k][i] = 1 / H_k[i][i] (0 where H_ii <= 0), for the panel products here and for the codebook
// step (gq_codebook_gemm.cuh).  One block per row of a group's matrix, 16-byte loads (d_in is a multiple of 8): bound by the
// 8 bytes per entry it moves.  With one entry per thread and a 64-bit modulo each to find the diagonal it took 342 us for
// four 4096 x 4096 matrices, now 79.
__global__ void __launch_bounds__(256)
split_h_kernel(const float *H, int d_in, __nv_bfloat16 *Hhi, __nv_bfloat16 *Hlo,
                  float *rdiag)
{
    griddep_launch();
    griddep_wait();
    const int i = static_cast<int>(blockIdx.x);
    const size_t row = static_cast<size_t>(blockIdx.y) * d_in + i;
    const float4 *src = reinterpret_cast<const float4 *>(H + row * d_in);
    uint2 *hi = reinterpret_cast<uint2 *>(Hhi + row * d_in), *lo = reinterpret_cast<uint2 *>(Hlo + row * d_in);
    for (int c = threadIdx.x; c < d_in / 4; c += 256) {
        const float4 v = src[c];
        const float f[4] = {v.x, v.y, v.z, v.w};
        __align__(8) __nv_bfloat16 h[4], l[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            split_bf16(f[e], h[e], l[e]);
            if (4 * c + e == i) rdiag[row] = f[e] > 0.0f ? 1.0f / f[e] : 0.0f;
        }
        hi[c] = *reinterpret_cast<uint2 *>(h);
        lo[c] = *reinterpret_cast<uint2 *>(l);
    }
}

// Q = Qt^T back to [d_out][d_in] and What = codebook[Q].  64 x 64 tiles, four codes per thread; `bytes`: Q is not 4-byte
// aligned and is written byte by byte.  (4096 x 4096: 19 us; 51 with one code per thread, 32-byte segments and W_hat carried through every block.)
__global__ void __launch_bounds__(256)
cd_finish_kernel(const float *codebook, const uint8_t *Qt, int d_in, int d_out, int m, float *What, uint8_t *Q, bool bytes)
{
    __shared__ __align__(4) uint8_t tq[64][68];                    // stored to in words
    griddep_launch();
    griddep_wait();
    const int c4 = (threadIdx.x & 15) * 4, r0 = threadIdx.x >> 4;
    const int i0 = blockIdx.x * 64, j0 = blockIdx.y * 64;
#pragma unroll
    for (int r = r0; r < 64; r += 16) {                            // d_in and d_out are multiples of 8: fours are inside or outside
        const int i = i0 + r, j = j0 + c4;
        *reinterpret_cast<uint32_t *>(&tq[r][c4]) =
            (i < d_in && j < d_out) ? *reinterpret_cast<const uint32_t *>(Qt + static_cast<size_t>(i) * d_out + j) : 0u;
    }
    __syncthreads();
#pragma unroll
    for (int r = r0; r < 64; r += 16) {
        const int j = j0 + r, i = i0 + c4;
        if (j >= d_out || i >= d_in) continue;
        const float *cb = codebook + static_cast<size_t>(j) * m;
        const size_t o = static_cast<size_t>(j) * d_in + i;
        const uint8_t top = static_cast<uint8_t>(m - 1);             // no code leads past the channel's levels
        const uchar4 q = make_uchar4(min(tq[c4][r], top), min(tq[c4 + 1][r], top), min(tq[c4 + 2][r], top), min(tq[c4 + 3][r], top));
        *reinterpret_cast<float4 *>(What + o) = make_float4(cb[q.x], cb[q.y], cb[q.z], cb[q.w]);
        if (bytes) {
            Q[o] = q.x; Q[o + 1] = q.y; Q[o + 2] = q.z; Q[o + 3] = q.w;
        } else {
            *reinterpret_cast<uchar4 *>(Q + o) = q;
        }
    }
}

struct CdBlockParams {
    const float *rdiag;      // [g][d_in]
    const float *codebook;   // [d_out][m]
    float *P;                // [CD_BLOCK][d_out] pulled sums; zeroed again once read
    float *Et;               // [d_in][d_out]
    __nv_bfloat16 *Ehi, *Elo;
    uint8_t *Qt;             // [d_in][d_out]
    int d_in, d_out, g, mk, m;
    int s0;                  // first coordinate of the block
    int rows;                // coordinates in the block (<= CD_BLOCK)
    int slices;              // ceil(mk / CH): CTAs per group
    bool last_cycle;         // write the codes
    uint32_t *status;
    unsigned long long wait_budget_ns;
};

__device__ __forceinline__ void bar_sync_named(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive_named(int id, int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// The nearest of LEV sorted levels, ties already decided by the thresholds between neighbours: the number of thresholds
// below the target is the position of the level.  A tree of compares and selects: no table read, no exchange between lanes.
template <int LEV>
__device__ __forceinline__ float nearest_level(float target, const float (&lev)[LEV], const float (&thr)[LEV])
{
    float v[LEV];
#pragma unroll
    for (int q = 0; q < LEV; ++q) v[q] = lev[q];
#pragma unroll
    for (int width = 1; width < LEV; width *= 2)
#pragma unroll
        for (int k = 0; k < LEV / (2 * width); ++k)
            v[k] = target > thr[2 * width * k + width - 1] ? v[2 * k + 1] : v[2 * k];
    return v[0];
}

// What step I of a band reads from shared memory: H[I][rows after I], W_I of the lane's channel, 1 / H_II.
struct ChainOperands {
    float4 h[CD_BAND / 4];
    float w, rd;
    template <int I, int CH>
    __device__ __forceinline__ void load(const float *hd, const float *wb, const float *rb)
    {
#pragma unroll
        for (int q = (I + 1) / 4; q < CD_BAND / 4; ++q) h[q] = *reinterpret_cast<const float4 *>(hd + I * CD_BAND + 4 * q);
        w = wb[I * CH];
        rd = rb[I];
    }
};

// Steps I .. RUN - 1 of a run (a band is CD_BAND / RUN of them).  Bu is a window of 32 sums that starts with the run's rows;
// every step updates what comes after it in the window.  In the second run of a band the window's upper half lies past the
// band: those sums are formed from whatever follows in shared memory and never used.  Operands are read two steps ahead (the
// product warps keep the shared-memory pipe busy, so a read takes longer than a step).  Written as a recursion because the
// compiler does not unroll the loop, and the sums have to stay in registers.
template <int LEV, int CH, int RUN, int I>
__device__ __forceinline__ void chain_steps(const ChainOperands &cur, const ChainOperands &nxt, const float *hd, const float *rb,
                                            float *wb, float *eb, float (&Bu)[CD_BAND], const float (&lev)[LEV],
                                            const float (&thr)[LEV])
{
    ChainOperands after;
    if constexpr (I + 2 < RUN) after.load<I + 2, CH>(hd, wb, rb);
    const float val = nearest_level<LEV>(cur.w - cur.rd * Bu[I], lev, thr);
    const float e_new = val - cur.w;
#pragma unroll
    for (int r = I + 1; r < CD_BAND; ++r) {
        const float4 hq = cur.h[r >> 2];
        Bu[r] = fmaf((r & 3) == 0 ? hq.x : (r & 3) == 1 ? hq.y : (r & 3) == 2 ? hq.z : hq.w, e_new, Bu[r]);
    }
    eb[I * CH] = e_new;
    wb[I * CH] = val;                                 // W_i is not needed any more: What of the block takes its place
    if constexpr (I + 1 < RUN) chain_steps<LEV, CH, RUN, I + 1>(nxt, after, hd, rb, wb, eb, Bu, lev, thr);
}

// Where four rows (quad rq of a band) of channel ch stand in a part of the pulled sums, in floats: the swizzle keeps both
// the products' stores (a quarter warp: channels 4 j + b, one quad) and the chain's loads (one quad of 32 channels) free
// of bank conflicts.
__device__ __forceinline__ int sums_at(int ch, int rq)
{
    return ch * CD_BAND + ((rq ^ (ch >> 2) ^ ch) & 7) * 4;
}

// One block of coordinates for CH channels of one group.
//
// The running sums  Bu[r] = sum_{c != r} H[r][c] E_c  (current E: this cycle's values for c < r, last cycle's for c > r)
// are needed one coordinate after the other, each after a rounding decision on the one before it: 256 dependent steps.
// What bounds the kernel is the length of one step, so everything that is not part of it is moved to other warps:
//   chain warp (0)       one lane per channel.  A band of 32 coordinates at a time, its 32 running sums in registers: round
//                        (nearest_level: compares and selects only), E_i = val - W_i, add H[i][r] E_i to the sums of the
//                        rows after i inside the band.  No shuffle, vote or table read lies on the path.
//   product warps (6, with 16 channels 3 of two parts each)   while the chain works on band t they form the sums of band t + 1 over every coordinate of the block
//                        outside bands t and t + 1, plus last cycle's values of band t + 1 above its diagonal; when the chain
//                        is through with band t they add its new values (32 x 32 x CH) and hand the sums over.  Every part
//                        forms all of the 32 x CH sums, 8 rows x 4 channels per thread, over a share of the contraction;
//                        all of them on the three schedulers that the chain warp does not use.  A value loaded from shared
//                        memory costs a lane-register write whether or not lanes share it (measured: a 16-byte load takes
//                        4 clocks of the SM's load pipe, 2 if all lanes read the same address), hence 12 loaded values
//                        per 32 multiply-adds.
//   loader warp (4)      TMA: the tiles of W, E and P (256 coordinates x CH channels), and H[all 256][band] (32 KB) per
//                        band into one of three buffers, two bands ahead.
// Two named barriers per band: sums ready (products -> chain), band done (chain -> products, loader).
// Measured for one block of 4096 channels, 16 levels: 33.9 us (8 levels, 1408 channels: 22.8 by itself, 19 from the end of the
// panel product to its own, 27 with 32 channels per CTA); 1.2 us more with the excluded coordinates multiplied by zero instead of
// left out;
// with eight threads per channel that did all updates themselves and two votes and a table read per step it was 81 us (78).
template <int LEV, int CH>
__global__ void __launch_bounds__(CD_THREADS, 1)
cd_block_kernel(const __grid_constant__ CUtensorMap mapH, const __grid_constant__ CUtensorMap mapW,
                const __grid_constant__ CUtensorMap mapE, const __grid_constant__ CUtensorMap mapP, const CdBlockParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_tiles;
    __shared__ __align__(8) uint64_t bar_h[CD_H_BUFS];
    __shared__ volatile uint32_t abort_flag;
    // aligned by an offset: rounding the pointer itself would make every access below a generic one
    float *Ws = reinterpret_cast<float *>(smem_raw + ((0u - smem_u32(smem_raw)) & 1023u));
    float *Es = Ws + CD_BLOCK * CH;                      // [256][CH] E of the block, updated in place
    float *Ps = Es + CD_BLOCK * CH;                      // [256][CH] P
    float *Hs = Ps + CD_BLOCK * CH;                      // [CD_H_BUFS][256][32] H[c][rows of a band]
    float *Ss = Hs + CD_H_BUFS * CD_H_FLOATS;            // [CD_PARTS][CH][32 rows] pulled sums of a band (sums_at)
    float *rds = Ss + CD_PARTS * CD_BAND * CH;           // [256]
    float *srt = rds + CD_BLOCK;                         // [CH][CD_LEVEL_LD] sorted levels
    float *thr_s = srt + CH * CD_LEVEL_LD;               // [CH][CD_LEVEL_LD] thresholds between neighbours
    int *sidx = reinterpret_cast<int *>(thr_s + CH * CD_LEVEL_LD);      // [CH][CD_LEVEL_LD] given index by sorted position

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int k = blockIdx.x / p.slices;
    const int ch0 = k * p.mk + (blockIdx.x % p.slices) * CH;             // first channel of this CTA
    const int ch_n = min(CH, (k + 1) * p.mk - ch0);                   // valid channels (a multiple of 8)
    const WaitCtx wc{&abort_flag, p.status, p.wait_budget_ns};

    auto load_band = [&](int t) {                        // H[block coordinates][band t] (zero outside the matrix)
        const uint32_t bar = smem_u32(&bar_h[t % CD_H_BUFS]);
        mbar_arrive_expect_tx(bar, CD_H_FLOATS * 4);
        tma_load_3d(smem_u32(Hs + (t % CD_H_BUFS) * CD_H_FLOATS), &mapH, bar, p.s0 + t * CD_BAND, p.s0, k);
    };
    // A wait that ran out is recorded; the warps go on (with wrong values) so that every barrier completes.
    auto wait_band = [&](int t) {
        (void)bounded_wait(smem_u32(&bar_h[t % CD_H_BUFS]), static_cast<uint32_t>(t / CD_H_BUFS) & 1u, wc, 21u, blockIdx.x);
    };
    griddep_launch();
    if (tid == 128) {
        mbar_init(smem_u32(&bar_tiles), 1);
        for (int b = 0; b < CD_H_BUFS; ++b) mbar_init(smem_u32(&bar_h[b]), 1);
        abort_flag = 0u;
        fence_mbar_init();
        fence_proxy_async_smem();
        griddep_wait();
        load_band(0);
        const uint32_t bar = smem_u32(&bar_tiles);
        mbar_arrive_expect_tx(bar, 3 * CD_BLOCK * CH * 4);
        tma_load_3d(smem_u32(Es), &mapE, bar, ch0, p.s0, 0);
        tma_load_3d(smem_u32(Ps), &mapP, bar, ch0, 0, 0);
        tma_load_3d(smem_u32(Ws), &mapW, bar, ch0, p.s0, 0);
        for (int b = 1; b < CD_H_BUFS; ++b) load_band(b);
    }
    griddep_wait();
    rds[tid] = tid < p.rows ? p.rdiag[static_cast<size_t>(k) * p.d_in + p.s0 + tid] : 0.0f;
    // ---- the channel's levels, sorted (eight threads per channel), and the thresholds between neighbours: their midpoints,
    // lowered by one ulp where the upper level has the smaller given index, so that a tie goes to the smaller index.
    // Sorted means a total order, so that every position is written: numbers ascending, then NaN, equal ones by index.  A
    // threshold beside a NaN is a NaN and never exceeded: no target is rounded to it while the channel has a number.  The
    // positions past the channel's levels hold NaN as well, with the highest indices.
    if (tid < 8 * CH) {
        const int cidx = tid >> 3, l = tid & 7;
        const bool chan = cidx < ch_n;
        const float v0 = (l < p.m && chan) ? p.codebook[static_cast<size_t>(ch0 + cidx) * p.m + l] : CUDART_NAN_F;
        const float v1 = (l + 8 < p.m && chan) ? p.codebook[static_cast<size_t>(ch0 + cidx) * p.m + l + 8] : CUDART_NAN_F;
        auto key = [](float v) {                         // unsigned, ascending with v; -0 as 0, NaN above infinity
            const uint32_t b = __float_as_uint(v + 0.0f);
            return isnan(v) ? 0xff800001u : (b ^ (static_cast<uint32_t>(static_cast<int32_t>(b) >> 31) | 0x80000000u));
        };
        const uint32_t k0 = key(v0), k1 = key(v1);
        int rank0 = 0, rank1 = 0;                        // positions of (v0, l) and (v1, l + 8) among the 16 pairs
#pragma unroll
        for (int r = 0; r < CD_MAX_LEVELS; ++r) {
            const uint32_t kr = __shfl_sync(0xffffffffu, r < 8 ? k0 : k1, r & 7, 8);
            rank0 += kr < k0 + (r < l ? 1u : 0u) ? 1 : 0;
            rank1 += kr < k1 + (r < l + 8 ? 1u : 0u) ? 1 : 0;
        }
        float *ms = srt + cidx * CD_LEVEL_LD;
        int *mi = sidx + cidx * CD_LEVEL_LD;
        ms[rank0] = v0;
        mi[rank0] = l;
        ms[rank1] = v1;
        mi[rank1] = l + 8;
        __syncwarp();
        auto threshold = [&](int q) {                    // between sorted levels q and q + 1
            const float mid = 0.5f * (ms[q] + ms[q + 1]);
            return (mi[q] < mi[q + 1] || !(fabsf(mid) < CUDART_INF_F)) ? mid : nextafterf(mid, -CUDART_INF_F);
        };
        thr_s[cidx * CD_LEVEL_LD + 2 * l] = threshold(2 * l);
        thr_s[cidx * CD_LEVEL_LD + 2 * l + 1] = 2 * l + 2 < CD_MAX_LEVELS ? threshold(2 * l + 1) : CUDART_INF_F;
    }
    __syncthreads();
    (void)bounded_wait(smem_u32(&bar_tiles), 0u, wc, 20u, blockIdx.x);

    constexpr int BAR_SUMS = 1, BAR_BAND = 2;
    constexpr int SHARE = 32 / CH;                       // parts a product warp forms, CH lanes each
    constexpr int PRODUCTS = CD_PARTS / SHARE;           // product warps: 1 .. 3 and, with CH = 32, 5 .. 7
    constexpr int SUMS_THREADS = (1 + PRODUCTS) * 32, BAND_THREADS = SUMS_THREADS + 32;
    if (warp == 0) {
        // ------------------------------------------------------------------ chain: the coordinates in order
        // With 16 levels the 32 unrolled steps of a band (30 KB of code) and the products' loops do not fit the instruction
        // cache together: 39.6 us a block against 34.8 with 16 steps twice.  With 8 they do (31.4 against 33.2), but where a
        // block is short the first band, which fetches all code, counts for more: with 16 channels 1181 against 1191 us for the
        // descent named below.  With 4 levels 32 steps stay the better (2320 x 2032, two cycles: 740 against 747).
        constexpr int RUN = LEV > 8 || (LEV == 8 && CH == 16) ? CD_BAND / 2 : CD_BAND;
        const int ch = lane % CH;                        // lanes past the channels read along until the steps begin
        float lev[LEV], thr[LEV];
#pragma unroll
        for (int q = 0; q < LEV; ++q) {
            lev[q] = srt[ch * CD_LEVEL_LD + q];
            thr[q] = thr_s[ch * CD_LEVEL_LD + q];
        }
#pragma unroll 1
        for (int t = 0; t < CD_BANDS; ++t) {
            wait_band(t);
            const float *hd = Hs + (t % CD_H_BUFS) * CD_H_FLOATS + t * CD_BAND * CD_BAND;      // H[band][band]
            float *wb = Ws + t * CD_BAND * CH + ch, *eb = Es + t * CD_BAND * CH + ch;
            const float *rb = rds + t * CD_BAND;
            ChainOperands first, second;                 // not written by the products: read while the sums are awaited
            first.load<0, CH>(hd, wb, rb);
            second.load<1, CH>(hd, wb, rb);
            bar_sync_named(BAR_SUMS, SUMS_THREADS);
            if (lane < CH) {                             // one lane per channel, or two would share its words of W and E
                float Bu[CD_BAND];
#pragma unroll
                for (int q = 0; q < CD_BAND / 4; ++q) {
                    const float *sp = Ss + sums_at(ch, q);
                    float4 v[CD_PARTS];
#pragma unroll
                    for (int n = 0; n < CD_PARTS; ++n) v[n] = *reinterpret_cast<const float4 *>(sp + n * CD_BAND * CH);
                    Bu[4 * q + 0] = ((v[0].x + v[1].x) + (v[2].x + v[3].x)) + (v[4].x + v[5].x);
                    Bu[4 * q + 1] = ((v[0].y + v[1].y) + (v[2].y + v[3].y)) + (v[4].y + v[5].y);
                    Bu[4 * q + 2] = ((v[0].z + v[1].z) + (v[2].z + v[3].z)) + (v[4].z + v[5].z);
                    Bu[4 * q + 3] = ((v[0].w + v[1].w) + (v[2].w + v[3].w)) + (v[4].w + v[5].w);
                }
#pragma unroll 1
                for (int run = 0; run < CD_BAND / RUN; ++run) {
                    if (run > 0) {
                        hd += RUN * (CD_BAND + 1);         // the same number of rows and columns on
                        rb += RUN;
                        wb += RUN * CH;
                        eb += RUN * CH;
                        first.load<0, CH>(hd, wb, rb);
                        second.load<1, CH>(hd, wb, rb);
#pragma unroll
                        for (int r = 0; r + RUN < CD_BAND; ++r) Bu[r] = Bu[r + RUN];
                    }
                    chain_steps<LEV, CH, RUN, 0>(first, second, hd, rb, wb, eb, Bu, lev, thr);
                }
            }
            __syncwarp();
            if (t + 1 < CD_BANDS) bar_arrive_named(BAR_BAND, BAND_THREADS);
        }
    } else if (warp == 4) {
        // ------------------------------------------------------------------ loader
        for (int t = 0; t + 1 < CD_BANDS; ++t) {
            bar_sync_named(BAR_BAND, BAND_THREADS);      // band t's buffer is free
            if (lane == 0 && t + CD_H_BUFS < CD_BANDS) load_band(t + CD_H_BUFS);
        }
    } else if ((warp < 4 ? warp - 1 : warp - 2) < PRODUCTS) {
        // ------------------------------------------------------------------ products: sums of band t
        const int part = (warp < 4 ? warp - 1 : warp - 2) * SHARE + lane / CH;                 // 0..5
        const int r0 = (lane % CH) / (CH / 4) * 8, c0 = (lane % (CH / 4)) * 4;                 // 8 rows x 4 channels
#pragma unroll 1
        for (int t = 0; t < CD_BANDS; ++t) {
            wait_band(t);
            const float *hb = Hs + (t % CD_H_BUFS) * CD_H_FLOATS + r0;
            const float *eb = Es + c0;
            float acc[8][4];
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                const float4 v = part == 0 ? *reinterpret_cast<const float4 *>(Ps + (t * CD_BAND + r0 + a) * CH + c0)
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
                acc[a][0] = v.x; acc[a][1] = v.y; acc[a][2] = v.z; acc[a][3] = v.w;
            }
            auto add_row = [&](int a, float h, const float4 &e) {
                acc[a][0] = fmaf(h, e.x, acc[a][0]);
                acc[a][1] = fmaf(h, e.y, acc[a][1]);
                acc[a][2] = fmaf(h, e.z, acc[a][2]);
                acc[a][3] = fmaf(h, e.w, acc[a][3]);
            };
            auto load_h = [&](int c, float (&h)[8]) {
                const float4 lo = *reinterpret_cast<const float4 *>(hb + c * CD_BAND);
                const float4 hi = *reinterpret_cast<const float4 *>(hb + c * CD_BAND + 4);
                h[0] = lo.x; h[1] = lo.y; h[2] = lo.z; h[3] = lo.w;
                h[4] = hi.x; h[5] = hi.y; h[6] = hi.z; h[7] = hi.w;
            };
            auto load_e = [&](int c) { return *reinterpret_cast<const float4 *>(eb + c * CH); };
            // (coordinates at a time: four with 16 channels, 1250 -> 1191 us for 2056 x 1408, 8 levels, four cycles; two 1238; with 32
            // channels eight, 1275 against 1280 for 1400 x 2480, 16 levels, two rounds)
            constexpr int UNROLL = CH == 16 ? 4 : 8;
            // one band for each part, neither the one the chain is working on (t - 1) nor this one
            {
                const int first = (t == 0 ? part + 1 : part >= t - 1 ? part + 2 : part) * CD_BAND;
#pragma unroll UNROLL
                for (int c = first; c < first + CD_BAND; ++c) {
                    float h[8];
                    load_h(c, h);
                    const float4 e = load_e(c);
#pragma unroll
                    for (int a = 0; a < 8; ++a) add_row(a, h[a], e);
                }
            }
            // bands that all six share, 5 or 6 coordinates each.  n = 0: last cycle's values inside the band, coordinates after
            // the row only; n = 1 (t = 0 only): the band left over; n = 2: band t - 1 once the chain is through with it.
            const int k0 = part * CD_BAND / CD_PARTS, k1 = (part + 1) * CD_BAND / CD_PARTS;
#pragma unroll 1
            for (int n = 0; n < 3; ++n) {
                if (n == 2 && t > 0) bar_sync_named(BAR_BAND, BAND_THREADS);
                const int band = n == 0 ? t : n == 1 ? (t == 0 ? 7 : -1) : t - 1;
                if (band < 0) continue;
#pragma unroll
                for (int i = 0; i < (CD_BAND + CD_PARTS - 1) / CD_PARTS; ++i) {
                    const int kc = k0 + i, at = band * CD_BAND + min(kc, CD_BAND - 1);
                    const int rows = kc >= k1 ? 0 : n == 0 ? kc - r0 : 8;      // of this thread's eight
                    float h[8];
                    load_h(at, h);
                    const float4 e = load_e(at);
                    // left out and not multiplied by zero: last cycle's value may be no number
#pragma unroll
                    for (int a = 0; a < 8; ++a)
                        if (a < rows) add_row(a, h[a], e);
                }
            }
#pragma unroll
            for (int b = 0; b < 4; ++b)
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    *reinterpret_cast<float4 *>(Ss + part * CD_BAND * CH + sums_at(c0 + b, r0 / 4 + q)) =
                        make_float4(acc[4 * q][b], acc[4 * q + 1][b], acc[4 * q + 2][b], acc[4 * q + 3][b]);
            bar_arrive_named(BAR_SUMS, SUMS_THREADS);
        }
    }
    __syncthreads();

    // ---- tiles out, four channels per thread; P is left zero for the next block's panel product
    for (int idx = tid; idx < CD_BLOCK * CH / 4; idx += CD_THREADS) {
        const int r = idx / (CH / 4), c = idx % (CH / 4) * 4;
        if (c >= ch_n) continue;
        *reinterpret_cast<float4 *>(p.P + static_cast<size_t>(r) * p.d_out + ch0 + c) = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r >= p.rows) continue;
        const size_t o = static_cast<size_t>(p.s0 + r) * p.d_out + ch0 + c;
        const float4 e4 = *reinterpret_cast<const float4 *>(Es + r * CH + c);
        const float e[4] = {e4.x, e4.y, e4.z, e4.w};
        __align__(8) __nv_bfloat16 hi[4], lo[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) split_bf16(e[b], hi[b], lo[b]);
        *reinterpret_cast<float4 *>(p.Et + o) = e4;
        *reinterpret_cast<uint2 *>(p.Ehi + o) = *reinterpret_cast<uint2 *>(hi);
        *reinterpret_cast<uint2 *>(p.Elo + o) = *reinterpret_cast<uint2 *>(lo);
        if (!p.last_cycle) continue;                     // the codes of earlier cycles are never read
        const float4 v4 = *reinterpret_cast<const float4 *>(Ws + r * CH + c);
        const float v[4] = {v4.x, v4.y, v4.z, v4.w};
        uint32_t codes = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float *ms = srt + (c + b) * CD_LEVEL_LD;
            int pos = 0;                                 // first sorted level that is not below val: among equal ones the
#pragma unroll
            for (int step = LEV / 2; step > 0; step >>= 1)      // one with the smallest given index
                if (ms[pos + step - 1] < v[b]) pos += step;
            codes |= static_cast<uint32_t>(min(sidx[(c + b) * CD_LEVEL_LD + pos], p.m - 1)) << (8 * b);
        }
        *reinterpret_cast<uint32_t *>(p.Qt + o) = codes;
    }
}

}  // namespace gq
