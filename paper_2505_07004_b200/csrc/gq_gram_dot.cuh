// The objective of Eq. 7 on the tensor cores:
//
//     loss_k = sum_{j in J_k} delta_j^T H_k delta_j = < H_k , Delta_k^T Delta_k >,     Delta_k = rows J_k of W - W_hat,
//
// evaluated on the upper triangle, sum_{a <= b} (2 - [a == b]) D_k[a][b] H_k[a][b] with D_k = Delta_k^T Delta_k.
// D_k is never written: a CTA pair forms one 256 x 256 tile of it in tensor memory and contracts it with the
// matching entries of H_k straight out of tensor memory.
//
// Operands.  Delta is prepared once per call as ONE fp16 matrix (delta_half_kernel): delta * 2^e with a single
// power of two e for the whole layer, such that the largest finite entry rounds to [2^14, 2^16), but for the clamps.
// fp16 carries 11 significant bits at any magnitude above 2^-14, i.e. down to 2^-28 of the largest entry at least (what is
// smaller is off by at most 2^-39 of the largest), and the
// scaling is undone exactly (2^-2e in the final fp64 reduction).  One product at the
// 16-bit rate replaces three bf16 products (hi hi + hi lo + lo hi): the contraction then costs about as much as
// streaming H from HBM, which is what the kernel below is built around.  Rounding: both factors of every
// product carry a relative error of at most 2^-12 (round to nearest), unbiased, so the objective is good to
// 2^-11 = 4.9e-4 in the worst case of all errors aligned and to ~1e-6 for errors of random sign.
//
// Units.  A unit is one 256 x 256 tile (i <= j) of one group; a pair's tensor memory holds two such accumulators,
// so the tile of unit n + 1 is being computed while the tile of unit n is contracted with H: the tensor core
// never waits for a read-out.  (Units of two column tiles sharing their row operand, as in gq_hessian.cuh, need
// a quarter less operand traffic from L2 but fill tensor memory with one unit: measured on the 4096 x 4096 layer
// the tensor core then idled for a third of every unit, waiting for H.)  The stage is [A | B], 16 KB each, 64
// channels of the contraction, six stages.  Units are numbered group-major and, inside a group, in the
// super-block tile order of gq_pipeline.cuh, so that the pairs working at the same time share operand blocks.
//
// H.  The entries of H_k that go with a tile (256 KB per pair) do not depend on the accumulators; what limits
// their delivery is the number of requests an SM can have in flight (a lane needs 32 consecutive floats of ITS
// row, tensor memory dictates lane = row, so a warp's 32-byte load is 32 separate sector requests).  So the
// requests are spread over the whole time the tile is being computed: as soon as an epilogue warp has finished a
// tile it requests the four 32 x 32 blocks of its next tile into registers (128 KB per CTA: with that the eight
// epilogue warps hold all of the CTA's share), and they have a full unit of MMAs (4 - 7 us) to arrive.  (An extra
// warp that asked for the same rows earlier still with bulk L2 prefetches changed nothing measurable on any of
// the layer shapes and was taken out again.)  Once the accumulator is complete the contraction itself takes well
// under a microsecond: tensor-memory columns of block j + 1 are requested before block j is used, blocks above
// the diagonal take a branch without per-entry weights, and the accumulator is handed back as soon as its last
// block sits in registers.
//
// Roles: warp 0 (one lane) TMA producer, warp 1 (one lane, first CTA) MMA issuer, warp 2 TMEM allocation,
// warp 3 idle, warps 4..11 epilogue (registers: the service warpgroup gives up all but 40, the two
// epilogue warpgroups take 232).  Whole units only: one fp64 partial per (unit, CTA, warp), reduced in a fixed
// order, so the result is reproducible.  Every mbarrier wait is bounded (gq_pipeline.cuh).
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "gq_pipeline.cuh"

namespace gq {

constexpr int GD_STAGES = 6;
constexpr int GD_SLOT_BYTES = (CTA_ROWS / BOX_FEATURES) * BOX_BYTES;      // one operand block: 16 KB
constexpr int GD_STAGE_BYTES = 2 * GD_SLOT_BYTES;                         // [A | B]
constexpr int GD_EPI_WARPS = 8;
constexpr int GD_THREADS = 32 * (4 + GD_EPI_WARPS);
constexpr int GD_SMEM_BYTES = GD_STAGES * GD_STAGE_BYTES + 1024;
constexpr int GD_PARTIALS_PER_UNIT = 2 * GD_EPI_WARPS;       // one fp64 per (CTA of the pair, epilogue warp)
constexpr int GD_SAMPLE_EXP = 14;                            // the largest sampled |delta| * 2^e lies in [2^14, 2^15);
constexpr int GD_FITS_EXP = 15;                              // the largest of all has to round to a finite value, 65504 at most
constexpr unsigned int GD_FITS_ROUND = 0x1000;               // carries into the exponent what fp16 rounds up to 2^16: 65520 on
constexpr int GD_MAX_SHIFT = 100;                            // |e| is kept below this (the scale stays a normal float)

// Header of the objective workspace, written by the preparation kernels and read by the reduction.
struct GramDotHeader {
    int guess;                  // e of the first preparation pass
    int shift;                  // e: the fp16 matrix holds (W - W_hat) * 2^e
    unsigned int blocks_done;   // groups whose loss has been written (the last one forms the total)
};

struct GramDotParams {
    int d;                   // d_in
    int rows;                // channels per group (contraction length)
    int g;
    int nj;                  // ceil(d / 256)
    int tiles;               // nj (nj + 1) / 2: 256 x 256 tiles on the upper triangle
    int raster;              // edge (in tiles) of the super-blocks of the tile order (gq_pipeline.cuh)
    Schedule sched;          // units = tiles * g (group-major: unit = k * tiles + tile slot), ksteps = ceil(rows / 64)
    const float *H;          // [g][d][d], only a <= b is read
    double *partials;        // [units][GD_PARTIALS_PER_UNIT]
    uint32_t *status;
    unsigned long long wait_budget_ns;
};

// Instruction descriptor for kind::f16 with fp16 A and B (both MN-major), fp32 accumulator: as
// umma_idesc_bf16_mn with the operand format fields [7,10) and [10,13) left at 0 (= f16).
__host__ __device__ constexpr uint32_t umma_idesc_f16_mn(uint32_t m, uint32_t n)
{
    return (1u << 4) | (1u << 15) | (1u << 16) | ((n >> 3) << 17) | ((m >> 4) << 24);
}

// Eight consecutive floats (32 bytes, 32-byte aligned) that are read once: no L1 allocation.
__device__ __forceinline__ void ld_stream_f32x8(const float *p, float (&v)[8])
{
    asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
}

// 16 bytes of fp32 input, loaded by volatile asm so that a thread's loads are all issued before the first use.
__device__ __forceinline__ float4 ld_f32x4(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_f32x4_last_use(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.cs.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

constexpr int DELTA_VEC_PER_THREAD = 4;      // float4 pairs a thread of the first preparation kernel handles
constexpr unsigned DELTA_BLOCK_VECS = 256u * DELTA_VEC_PER_THREAD;
constexpr unsigned DELTA_REDO_VECS = 256u * DELTA_VEC_PER_THREAD;      // of eight fp16 values, a block of the second one at a time

// The power of two that takes a value of biased exponent `biased` (0: zero or subnormal) to [2^target, 2^(target + 1)).
__device__ __forceinline__ int delta_shift(unsigned int biased, int target)
{
    int k = static_cast<int>(biased) - 127;                        // floor(log2(value)) for normal values
    if (k < -126) k = -126;
    int e = target - k;
    if (e > GD_MAX_SHIFT) e = GD_MAX_SHIFT;
    if (e < -GD_MAX_SHIFT) e = -GD_MAX_SHIFT;
    return e;
}
__device__ __forceinline__ float delta_scale(int e)
{
    return __uint_as_float(static_cast<unsigned int>(127 + e) << 23);
}
__device__ __forceinline__ float delta_max(float m, const float4 &w, const float4 &q)      // a NaN never wins fmaxf
{
    return fmaxf(m, fmaxf(fmaxf(fabsf(w.x - q.x), fabsf(w.y - q.y)), fmaxf(fabsf(w.z - q.z), fabsf(w.w - q.w))));
}
// The same over finite differences only.  One without a size says nothing about the scale of the others, and stays what it is in
// fp16 whatever the scale.  (For a thread's own sixteen values only where infinity shows: the comparisons cost a call on a
// 3152 x 296 layer a quarter of a microsecond.)
__device__ __forceinline__ float delta_max_finite(float m, const float4 &w, const float4 &q)
{
    auto size = [](float d) { return fabsf(d) < CUDART_INF_F ? fabsf(d) : 0.0f; };
    return fmaxf(m, fmaxf(fmaxf(size(w.x - q.x), size(w.y - q.y)), fmaxf(size(w.z - q.z), size(w.w - q.w))));
}
__device__ __forceinline__ uint2 delta_half4(const float4 &w, const float4 &q, float scale)
{
    uint2 o;
    __half2 *h = reinterpret_cast<__half2 *>(&o);
    h[0] = __floats2half2_rn((w.x - q.x) * scale, (w.y - q.y) * scale);
    h[1] = __floats2half2_rn((w.z - q.z) * scale, (w.w - q.w) * scale);
    return o;
}
// Maximum over the 256 threads of a block; `red` holds eight words.
__device__ __forceinline__ unsigned int block_max(unsigned int v, unsigned int *red)
{
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
#pragma unroll
    for (int w8 = 0; w8 < 8; ++w8) v = max(v, red[w8]);
    return v;
}

// out = fp16((W - W_hat) * 2^e), round to nearest (the differences are formed in fp32, as everywhere in the objective), and
// the biased exponent of every block's largest finite |W - W_hat| (one more where fp16 would round it up to the next power of
// two).  e has to be known before the first
// value is stored and depends on the largest, so it is guessed: every block looks at the same 1024 values, spread over the
// layer, and leaves room for values 2 to 4 times as large.  delta_redo_kernel takes care of layers that need more.
// A block goes over DELTA_BLOCK_VECS pairs of float4, or several times as many where there is no room for a byte from each.
// HBM-bound: W and W_hat are read once.  The sample is 64 runs of 64 bytes and not 256 of 16, each a request of its own in every
// block.  Three candidates of a 4096 x 4096 layer, whole calls: 324 us, with a pass over both matrices for the maximum before the
// pass that converts 371; with the sample of 256 places 348 and 380 in another run.  Two candidates of 3152 x 296, where all is in
// the L2: 4 % slower than two passes with 256 places, layers of 0.2 to 2 million weights with 64 none.
__global__ void __launch_bounds__(256)
delta_half_kernel(const float *W, const float *What, unsigned count4, GramDotHeader *header, uint8_t *block_exp, __half *out)
{
    __shared__ unsigned int red[2][8];
    griddep_launch();
    griddep_wait();
    unsigned base = blockIdx.x * DELTA_BLOCK_VECS + threadIdx.x;
    float4 w[DELTA_VEC_PER_THREAD], q[DELTA_VEC_PER_THREAD];
    // four pairs of float4 side by side, somewhere in each 64th of the layer (the same for every block)
    const unsigned part = max(count4 / 64u, 4u), spot = threadIdx.x / 4u;
    const unsigned sidx = min(((spot * part + __umulhi(spot * 2654435761u, part)) & ~3u) + threadIdx.x % 4u, count4 - 1u);
    const float4 sw = ld_f32x4(reinterpret_cast<const float4 *>(W) + sidx);
    const float4 sq = ld_f32x4(reinterpret_cast<const float4 *>(What) + sidx);
    auto load = [&] {
#pragma unroll
        for (int t = 0; t < DELTA_VEC_PER_THREAD; ++t) {
            const unsigned idx = base + t * 256u;
            const bool in = idx < count4;
            w[t] = in ? ld_f32x4_last_use(reinterpret_cast<const float4 *>(W) + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
            q[t] = in ? ld_f32x4_last_use(reinterpret_cast<const float4 *>(What) + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    load();
    const int e = delta_shift(block_max(__float_as_uint(delta_max_finite(0.0f, sw, sq)), red[0]) >> 23, GD_SAMPLE_EXP);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        header->guess = e;
        header->blocks_done = 0u;
    }
    const float scale = delta_scale(e);
    float largest = 0.0f;
    for (;;) {
        float m = 0.0f;
#pragma unroll
        for (int t = 0; t < DELTA_VEC_PER_THREAD; ++t) {
            const unsigned idx = base + t * 256u;
            m = delta_max(m, w[t], q[t]);
            if (idx < count4) reinterpret_cast<uint2 *>(out)[idx] = delta_half4(w[t], q[t], scale);
        }
        if (!(m < CUDART_INF_F)) {
            m = 0.0f;
#pragma unroll
            for (int t = 0; t < DELTA_VEC_PER_THREAD; ++t) m = delta_max_finite(m, w[t], q[t]);
        }
        largest = fmaxf(largest, m);
        base += gridDim.x * DELTA_BLOCK_VECS;
        if (base - threadIdx.x >= count4) break;
        load();
    }
    const unsigned int bits = block_max(__float_as_uint(largest), red[1]);
    if (threadIdx.x == 0) block_exp[blockIdx.x] = static_cast<uint8_t>((bits + GD_FITS_ROUND) >> 23);
}

// Eight fp16 values of scale 2^guess at the scale 2^(guess - down), in place.  Where the results are normal, or zero to begin with,
// that is `down` less in their exponents: the bits that rounding at the smaller scale gives.  False where a value is not finite
// or would lose bits that it has.
__host__ __device__ __forceinline__ bool delta_lower(uint4 &v, unsigned down)
{
    const unsigned least = down < 30u ? (down + 1u) << 10 : 0x7c00u, span = 0x7c00u - least;      // magnitudes in [least, 0x7c00)
    bool ok = true;
    auto two = [&](uint32_t &w) {
        const unsigned lo = w & 0x7fffu, hi = (w >> 16) & 0x7fffu;
        ok = ok && (lo == 0u || lo - least < span) && (hi == 0u || hi - least < span);
        w -= (lo ? down << 10 : 0u) + (hi ? down << 26 : 0u);
    };
    two(v.x);
    two(v.y);
    two(v.z);
    two(v.w);
    return ok;
}

// Decides on e: the guess where the largest finite |W - W_hat| is a finite fp16 with it (all blocks return at once), else the
// power of two that takes it to [2^15, 65520), or just below where it rounds up to 2^15, to which the matrix is then brought:
// the values that have their bits by lowering the exponent, a quarter of the bytes of W and W_hat and most of them in the L2,
// the others (among them what has overflowed) from W and W_hat.  blocks: of delta_half_kernel.
// One row 20 times as wide as the others, a call: 113 us for 4096 x 4096 and 250 for 4096 x 11008 with one group; 131 and 294 with
// all values from W and W_hat again, 123 and 273 with a pass over both for the maximum before one that converts.  A million
// times as wide, where 3 % of the threads' values are formed again: 115 and 258, 131 and 292, 121 and 271.
__global__ void __launch_bounds__(256)
delta_redo_kernel(const float *W, const float *What, unsigned count4, GramDotHeader *header, const uint8_t *block_exp,
                  unsigned blocks, __half *out)
{
    __shared__ unsigned int red[8];
    griddep_launch();
    griddep_wait();
    unsigned int biased = 0u;
    const unsigned words = blocks / 16u;
    for (unsigned i = threadIdx.x; i < words; i += 256u) {         // block_exp is 16-byte aligned
        const uint4 v = reinterpret_cast<const uint4 *>(block_exp)[i];
        const uint32_t four = __vmaxu4(__vmaxu4(v.x, v.y), __vmaxu4(v.z, v.w));
        biased = max(biased, max(max(four & 0xffu, (four >> 8) & 0xffu), max((four >> 16) & 0xffu, four >> 24)));
    }
    if (threadIdx.x < blocks % 16u) biased = max(biased, static_cast<unsigned int>(block_exp[words * 16u + threadIdx.x]));
    biased = block_max(biased, red);
    const int guess = header->guess, exact = delta_shift(biased, GD_FITS_EXP);
    const bool fits = static_cast<int>(biased) - 127 + guess <= GD_FITS_EXP || exact == guess;
    if (blockIdx.x == 0 && threadIdx.x == 0) header->shift = fits ? guess : exact;
    if (fits) return;
    const float scale = delta_scale(exact);
    const unsigned down = static_cast<unsigned>(guess - exact);    // positive: what does not fit is too large
    const unsigned count8 = count4 / 2u, stride = gridDim.x * DELTA_REDO_VECS;
    uint4 *o = reinterpret_cast<uint4 *>(out);
    // from the end: what delta_half_kernel has written last is still in the L2
    for (unsigned base = blockIdx.x * DELTA_REDO_VECS + threadIdx.x; base < count8; base += stride) {
        uint4 v[DELTA_VEC_PER_THREAD];
#pragma unroll
        for (int t = 0; t < DELTA_VEC_PER_THREAD; ++t) {
            const unsigned idx = base + t * 256u;
            v[t] = idx < count8 ? o[count8 - 1u - idx] : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int t = 0; t < DELTA_VEC_PER_THREAD; ++t) {
            const unsigned idx = base + t * 256u, at = count8 - 1u - idx;
            if (idx >= count8) continue;
            if (!delta_lower(v[t], down)) {
                const float4 *w = reinterpret_cast<const float4 *>(W) + 2 * static_cast<size_t>(at);
                const float4 *q = reinterpret_cast<const float4 *>(What) + 2 * static_cast<size_t>(at);
                const uint2 a = delta_half4(ld_f32x4(w), ld_f32x4(q), scale), b = delta_half4(ld_f32x4(w + 1), ld_f32x4(q + 1), scale);
                v[t] = make_uint4(a.x, a.y, b.x, b.y);
            }
            o[at] = v[t];
        }
    }
}

// loss[k] = 2^(-2e) * sum over the group's partial sums (block k), loss[g] = sum_k loss[k] (formed, in group order,
// by whichever block finishes last).  Every sum is formed in a fixed order (strided per thread, butterfly per warp,
// warp results in order), so the result does not vary from run to run.  partials: [g][slots][per_unit] (units are
// numbered group-major).  header->blocks_done is 0 before the launch (delta_half_kernel).
// (1024 threads: two groups of 6441 tiles take 20 us; 256 took 58.)
constexpr int GD_REDUCE_THREADS = 1024;
__global__ void __launch_bounds__(GD_REDUCE_THREADS)
gram_dot_reduce_kernel(const double *partials, int slots, int g, int per_unit, GramDotHeader *header, double *loss)
{
    __shared__ double warp_sum[GD_REDUCE_THREADS / 32];
    __shared__ bool last;
    griddep_launch();
    griddep_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k = blockIdx.x;
    const double *pk = partials + static_cast<size_t>(k) * slots * per_unit;
    const int count = slots * per_unit;
    double acc0 = 0.0, acc1 = 0.0, acc2 = 0.0, acc3 = 0.0;
    int idx = threadIdx.x;
    constexpr int T = GD_REDUCE_THREADS;
    for (; idx + 3 * T < count; idx += 4 * T) {            // four independent loads in flight
        acc0 += pk[idx];
        acc1 += pk[idx + T];
        acc2 += pk[idx + 2 * T];
        acc3 += pk[idx + 3 * T];
    }
    for (; idx < count; idx += T) acc0 += pk[idx];
    double acc = (acc0 + acc1) + (acc2 + acc3);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if (lane == 0) warp_sum[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = 0.0;
        for (int w = 0; w < T / 32; ++w) v += warp_sum[w];
        loss[k] = v * ldexp(1.0, -2 * header->shift);
        __threadfence();
        last = atomicAdd(&header->blocks_done, 1u) == static_cast<unsigned int>(g) - 1u;
        if (last) {
            __threadfence();
            double total = 0.0;
            for (int kk = 0; kk < g; ++kk) total += *const_cast<volatile double *>(loss + kk);
            loss[g] = total;
        }
    }
}

struct GramUnit {
    int ti, tj;      // tile (row block, column block), ti <= tj
    int k;           // group
};

__device__ __forceinline__ GramUnit gram_unit(const GramDotParams &p, int unit)
{
    GramUnit u;
    u.k = unit / p.tiles;
    tile_of_slot_blocked(unit - u.k * p.tiles, p.nj, p.raster, u.ti, u.tj);
    return u;
}

// mapD: fp16 [g][rows][d] (64-feature x 64-row boxes, 128-byte swizzle), the prepared Delta of every group.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GD_THREADS, 1)
gram_dot_kernel(const __grid_constant__ CUtensorMap mapD, const GramDotParams p)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bar_full[GD_STAGES];     // first CTA: bytes of both CTAs
    __shared__ __align__(8) uint64_t bar_empty[GD_STAGES];    // both CTAs: signalled by the MMA commits
    __shared__ __align__(8) uint64_t bar_acc_full[2];         // both CTAs, one per accumulator: signalled by the MMA commit
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
        for (int s = 0; s < GD_STAGES; ++s) {
            mbar_init(smem_u32(&bar_full[s]), 1);
            mbar_init(smem_u32(&bar_empty[s]), 1);
        }
        for (int kk = 0; kk < 2; ++kk) {
            mbar_init(smem_u32(&bar_acc_full[kk]), 1);
            mbar_init(smem_u32(&bar_acc_empty[kk]), 2 * GD_EPI_WARPS);
        }
        mbar_init(smem_u32(&bar_drain), 1);
        abort_flag = 0u;
        fence_mbar_init();
        prefetch_tensormap(&mapD);
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

    if (warp < 4) {
        // The service warpgroup keeps 40 registers per thread; the rest goes to the epilogue warpgroups.
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == 0 && lane == 0) {
            // -------------------------------------------------------------- TMA producer (both CTAs)
            int s = 0;
            uint32_t ph = 0;
            uint32_t issued = 0;
            bool ok = true;
            WorkItem w;
            for (int it = 0; ok && whole_unit(p.sched, pair, it, w); ++it) {
                const GramUnit u = gram_unit(p, w.unit);
                const int a0 = u.ti * TILE_M + static_cast<int>(rank) * CTA_ROWS;
                const int b0 = u.tj * TILE_N + static_cast<int>(rank) * CTA_ROWS;
                for (int ks = w.ks0; ks < w.ks1; ++ks) {
                    const int row = ks * TILE_K;
                    if (!bounded_wait(smem_u32(&bar_empty[s]), ph ^ 1u, wc, 1u, w.unit)) { ok = false; break; }
                    const uint32_t full_local = smem_u32(&bar_full[s]);
                    if (rank == 0) mbar_arrive_expect_tx(full_local, 2 * GD_STAGE_BYTES);      // both CTAs' bytes
                    const uint32_t full = map_to_cta(full_local, 0);
                    const uint32_t stage = ring + s * GD_STAGE_BYTES;
#pragma unroll
                    for (int q = 0; q < CTA_ROWS / BOX_FEATURES; ++q) {
                        tma_load_3d_pair(stage + q * BOX_BYTES, &mapD, full, a0 + q * BOX_FEATURES, row, u.k);
                        tma_load_3d_pair(stage + GD_SLOT_BYTES + q * BOX_BYTES, &mapD, full, b0 + q * BOX_FEATURES, row, u.k);
                    }
                    ++issued;
                    if (++s == GD_STAGES) { s = 0; ph ^= 1u; }
                }
            }
            // Stay until every stage has been released again: the release is an arrival on this CTA's barriers,
            // which must not come after the CTA has gone.
            for (int q = 0; ok && issued != 0u && q < GD_STAGES; ++q) {
                if (!bounded_wait(smem_u32(&bar_empty[s]), ph ^ 1u, wc, 5u, 0u)) ok = false;
                if (++s == GD_STAGES) { s = 0; ph ^= 1u; }
            }
            if (!ok) spin_ns(1000000ull);
        } else if (warp == 1 && lane == 0 && rank == 0) {
            // -------------------------------------------------------------- MMA issuer (first CTA)
            constexpr uint32_t idesc = umma_idesc_f16_mn(TILE_M, TILE_N);
            int s = 0;
            uint32_t ph = 0;
            uint32_t acc_ph[2] = {0u, 0u};
            bool ok = true;
            WorkItem w;
            for (int it = 0; ok && whole_unit(p.sched, pair, it, w); ++it) {
                const int buf = it & 1;
                // the accumulator of unit it - 2 must have been read out
                if (!bounded_wait_hot(smem_u32(&bar_acc_empty[buf]), acc_ph[buf] ^ 1u, wc, 2u, w.unit)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * TILE_N);
                for (int ks = w.ks0; ks < w.ks1; ++ks) {
                    if (!bounded_wait_hot(smem_u32(&bar_full[s]), ph, wc, 3u, w.unit)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t sa = ring + s * GD_STAGE_BYTES;
                    const uint32_t sb = sa + GD_SLOT_BYTES;
#pragma unroll
                    for (int k16 = 0; k16 < TILE_K / 16; ++k16) {
                        const uint64_t adesc = umma_smem_desc_mn_sw128(sa + k16 * 16 * 128, BOX_BYTES, 1024);
                        const uint64_t bdesc = umma_smem_desc_mn_sw128(sb + k16 * 16 * 128, BOX_BYTES, 1024);
                        umma_bf16(d_tmem, adesc, bdesc, idesc, (ks != w.ks0 || k16 != 0) ? 1u : 0u);
                    }
                    umma_commit_pair(smem_u32(&bar_empty[s]));
                    if (++s == GD_STAGES) { s = 0; ph ^= 1u; }
                }
                if (!ok) break;
                umma_commit_pair(smem_u32(&bar_acc_full[buf]));
                acc_ph[buf] ^= 1u;
            }
            if (!ok) {
                // Make sure no MMA is still writing TMEM when it is released.
                umma_commit_local(smem_u32(&bar_drain));
                const uint64_t t0 = global_timer_ns();
                while (!mbar_try_wait(smem_u32(&bar_drain), 0u) && global_timer_ns() - t0 < 5000000ull) {}
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
        // ------------------------------------------------------------------ epilogue: partial = <accumulator, H>
        const int ew = warp - 4;                        // 0..7
        const int q = warp & 3;                         // TMEM lane quarter this warp may access
        const int half = ew >> 2;                       // which 128 of the 256 accumulator columns
        uint32_t full_ph[2] = {0u, 0u};
        bool ok = true;
        WorkItem w;
        for (int it = 0; ok && whole_unit(p.sched, pair, it, w); ++it) {
            const int buf = it & 1;
            const GramUnit u = gram_unit(p, w.unit);
            const int row0 = u.ti * TILE_M + static_cast<int>(rank) * CTA_ROWS + q * 32;
            const int row = row0 + lane;
            // sum_{a <= b} (2 - [a == b]) D[a][b] H_k[a][b] over this warp's four 32 x 32 blocks of the tile:
            // block j covers columns tj * 256 + (half * 4 + j) * 32 .. + 31.
            const bool row_ok = row < p.d;
            const float *hrow = p.H + (static_cast<size_t>(u.k) * p.d + (row_ok ? row : 0)) * static_cast<size_t>(p.d);
            const int colw = u.tj * TILE_N + half * 128;
            // uniform over the warp: does block j hold entries on or above the diagonal inside the matrix?
            auto block_active = [&](int j) { return colw + j * 32 < p.d && row0 < p.d && colw + j * 32 + 32 > row0; };
            // All four blocks of H are requested now, while the tensor core is still working on this tile.
            float hq[4][4][8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const bool act = row_ok && block_active(j);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int c = colw + j * 32 + v * 8;
                    if (act && c < p.d && c + 7 >= row) {
                        ld_stream_f32x8(hrow + c, hq[j][v]);
                    } else {
#pragma unroll
                        for (int e = 0; e < 8; ++e) hq[j][v][e] = 0.0f;
                    }
                }
            }
            if (lane == 0) ok = bounded_wait(smem_u32(&bar_acc_full[buf]), full_ph[buf], wc, 4u, w.unit);
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            (void)mbar_try_wait(smem_u32(&bar_acc_full[buf]), full_ph[buf]);     // every lane observes the completed phase
            full_ph[buf] ^= 1u;
            tc_fence_after_sync();
            const uint32_t tmem_tile = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                                       static_cast<uint32_t>(buf * TILE_N + half * 128);
            double dsum = 0.0;
            uint32_t r[2][32];
            tmem_ld_32x32(tmem_tile, r[0]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                tmem_ld_wait();
                if (j < 3) {
                    tmem_ld_32x32(tmem_tile + static_cast<uint32_t>((j + 1) * 32), r[(j + 1) & 1]);
                } else {
                    // This warp holds all it needs from the accumulator: hand it back to the MMA issuer (first CTA).
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&bar_acc_empty[buf]), 0));
                }
                if (block_active(j)) {
                    const int col0 = colw + j * 32;
                    float part = 0.0f;
                    if (col0 > row0 + 31) {
                        // the whole block lies above the diagonal: every entry counts twice
#pragma unroll
                        for (int v = 0; v < 4; ++v)
#pragma unroll
                            for (int e = 0; e < 8; ++e)
                                part = fmaf(__uint_as_float(r[j & 1][v * 8 + e]), hq[j][v][e], part);
                        part *= 2.0f;
                    } else {
#pragma unroll
                        for (int v = 0; v < 4; ++v)
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                const int c = col0 + v * 8 + e;
                                const float wgt = (c > row) ? 2.0f : ((c == row) ? 1.0f : 0.0f);
                                part = fmaf(wgt * __uint_as_float(r[j & 1][v * 8 + e]), hq[j][v][e], part);
                            }
                    }
                    dsum += static_cast<double>(part);
                }
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, off);
            if (lane == 0)
                p.partials[static_cast<size_t>(w.unit) * GD_PARTIALS_PER_UNIT + rank * GD_EPI_WARPS + ew] = dsum;
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
