// mlp.cu -- BF16 tensor-core kernels of the learned surrogate: a multilayer
// perceptron (SiLU hidden layers) trained with AdamW and evaluated in batches.
// The paper has no learned component; this is the surrogate that maps scenario
// parameters to the aggregate's fractal dimension and RDF.
//
// GEMM: C[M x N] = A[M x K] * B[N x K]^T, A and B row-major BF16 (both
// "K-major"), FP32 accumulation in tensor memory, on the 5th-generation
// tensor cores of sm_100+ (tcgen05):
//  * one CTA of 256 threads computes a 128 x n_tile block (n_tile <= 256,
//    multiple of 16); the FP32 accumulator lives in TMEM (allocated per CTA);
//  * operands arrive by TMA (cp.async.bulk.tensor, 2-D tensor maps, boxes of
//    64 K-columns x rows) into a ring of up to four stages of 64 K-columns each,
//    in the K-major 128-byte swizzle of the tensor maps and the tcgen05 matrix
//    descriptors: a row's 64 columns are one 128-byte line, 8 rows an atom of
//    1024 bytes, atoms adjacent along M/N.  Rows beyond M or N and columns beyond
//    K are zero-filled by the TMA.  (In boxes of 8 columns, the layout without a
//    swizzle, the copies went out in 16-byte pieces:
//    training 4 networks took 147 us per minibatch of 256, now 133; 4096
//    predictions 106 us, now 103);
//  * one thread issues the loads (mbarrier expect_tx per stage), one thread
//    issues tcgen05.mma (M = 128, N = n_tile, K = 16 per instruction) and
//    releases each stage with tcgen05.commit; every wait is bounded (clock64
//    budget) and reports FLAG_TIMEOUT instead of hanging;
//  * the epilogue (8 warps) reads the accumulator with tcgen05.ld (32 lanes x
//    32 bit, 16 columns per load; warps w and w + 4 share TMEM lanes
//    32(w mod 4) .. +31 and split the 16-column groups), stages the tile in
//    shared memory and writes it row by row (one warp per row, lanes along the
//    columns), applying bias, SiLU, the SiLU derivative for back-propagation,
//    or a plain FP32 store.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include "npsim_internal.cuh"

namespace npsim {

namespace {

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// tcgen05 shared-memory matrix descriptor, no swizzle: start address, leading
// (K-direction) and stride (M/N-direction) byte offsets, each encoded >> 4;
// bits 46-47 carry the descriptor version (1) required by tcgen05.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo & 0x3FFFFu) >> 4) << 16;
    d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// The same of an operand in the 128-byte swizzle (bits 61-63 = 2): 64 K-columns per
// row, atoms of 8 rows (1024 bytes) one after the other; the start moves along K
// inside the atom, 32 bytes per 16 columns.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    return smem_desc(addr, 16, 1024) | (uint64_t)2 << 61;
}

// Instruction descriptor of tcgen05.mma kind::f16: D = F32 (bits 4-5 = 1),
// A = B = BF16 (bits 7-9 = 1, bits 10-12 = 1), both K-major (bits 15, 16 = 0),
// N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__device__ __forceinline__ uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return ok != 0;
}

// Default bound of every mbarrier wait: 2^32 SM cycles, ~2 s at 2 GHz.
constexpr long long kWaitCycles = 1ll << 32;

// Bounded wait for the completion of the mbarrier phase with the given parity:
// false once `budget` SM cycles have passed without it.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity,
                                                  long long budget = kWaitCycles)
{
    const long long t0 = clock64();
    while (!mbar_try(bar, parity)) {
        if (clock64() - t0 > budget)
            return false;
    }
    return true;
}

// SiLU and its derivative with the fast exponential and division intrinsics:
// their ~1e-6 relative error lies far below the BF16 rounding (2^-9) applied to
// every activation and gradient.  A huge exp(-z) gives a quotient of exactly 0.
__device__ __forceinline__ float silu(float z) { return __fdividef(z, 1.0f + __expf(-z)); }

__device__ __forceinline__ float dsilu(float z)
{
    const float s = __fdividef(1.0f, 1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

constexpr int kChunkK = 64;    // K columns per pipeline stage
constexpr int kTileM = 128;    // rows per CTA
constexpr int kMaxTileN = 256;
constexpr int kMaxStages = 4;
constexpr int kStageBudget = 200 * 1024; // shared memory for the operand ring

__host__ __device__ __forceinline__ int stage_bytes(int n_tile)
{
    return (kTileM + n_tile) * kChunkK * 2;
}

// Shared memory of one CTA: the operand ring, reused by the epilogue for the
// FP32 output tile (row pitch n_tile + 1 floats: conflict-free both ways).
__host__ __device__ __forceinline__ int dyn_smem_bytes(int n_tile, int stages)
{
    const int ring = stages * stage_bytes(n_tile);
    const int tile = kTileM * (n_tile + 1) * 4;
    return ring > tile ? ring : tile;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// 2-D TMA load of the box at (x = K column, y = row) into shared memory,
// completing `bytes` of the barrier's transaction count.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y,
                                            uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
                 "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
                 : "memory");
}

// The tensor map into the descriptor cache, before its first use.
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     bar)
                 : "memory");
}

constexpr int kGemmThreads = 256;

// Tile (bm, bn) of product z.
__device__ __forceinline__ void gemm_tile(const CUtensorMap *tmA, const CUtensorMap *tmB,
                                          const GemmArgs &g, int stages, int bm, int bn, int z)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages], done;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort, s_issued;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int m0 = bm * kTileM, n0 = bn * g.n_tile;
    const int nt = min(g.n_tile, g.N - n0); // multiple of 16 (N and n_tile are)
    const int nchunks = (g.K + kChunkK - 1) / kChunkK;
    const uint32_t base = smem_addr(smem);
    const uint32_t sbytes = (uint32_t)stage_bytes(g.n_tile);
    const uint32_t a_bytes = kTileM * kChunkK * 2;
    const uint32_t done_bar = smem_addr(&done);
    // bound of the main loop's waits (a test may shorten it); the drain after an
    // abort always waits with the default bound, so copies and MMAs in flight
    // land before the CTA frees its tensor memory and leaves
    const long long wb = g.wait_cycles > 0 ? g.wait_cycles : kWaitCycles;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(&s_tmem)),
                     "r"(g.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        prefetch_map(tmA);
        prefetch_map(tmB);
        for (int s = 0; s < stages; ++s) {
            mbar_init(smem_addr(&full[s]), 1);
            mbar_init(smem_addr(&empty[s]), 1);
        }
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
        s_abort = 0;
        s_issued = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;
    const int zero = after_previous();
    m0 += zero;
    n0 += zero;
    const int ya = z * g.za + m0, yb = z * g.zb + n0; // operand rows

    if (warp == 0) {
        if (lane == 0) { // TMA producer
            int c = 0;
            for (; c < nchunks; ++c) {
                const int s = c % stages, u = c / stages;
                if (u > 0 &&
                    !mbar_wait_bounded(smem_addr(&empty[s]), (uint32_t)((u - 1) & 1), wb)) {
                    atomicExch(&s_abort, 1);
                    break;
                }
                const uint32_t sa = base + (uint32_t)s * sbytes, sb = sa + a_bytes;
                const uint32_t fb = smem_addr(&full[s]);
                mbar_expect_tx(fb, sbytes); // columns and rows out of range arrive as zeros
                tma_load_2d(sa, tmA, c * kChunkK, ya, fb);
                tma_load_2d(sb, tmB, c * kChunkK, yb, fb);
            }
            s_issued = c;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) { // MMA issuer
            const uint32_t idesc = idesc_bf16(kTileM, nt);
            for (int c = 0; c < nchunks; ++c) {
                const int s = c % stages, u = c / stages;
                if (!mbar_wait_bounded(smem_addr(&full[s]), (uint32_t)(u & 1), wb)) {
                    atomicExch(&s_abort, 1);
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const int kc = min(kChunkK, g.K - c * kChunkK);
                const uint32_t sa = base + (uint32_t)s * sbytes, sb = sa + a_bytes;
                for (int ks = 0; ks < kc; ks += 16) {
                    const uint64_t ad = smem_desc_sw128(sa + (uint32_t)(ks * 2));
                    const uint64_t bd = smem_desc_sw128(sb + (uint32_t)(ks * 2));
                    const uint32_t acc = (c > 0 || ks > 0) ? 1u : 0u;
                    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                                     tmem),
                                 "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
                }
                mma_commit(smem_addr(&empty[s])); // stage s may be refilled
            }
            // fires once every MMA issued so far has completed (also after an abort)
            mma_commit(done_bar);
        }
        __syncwarp();
    }

    // the epilogue's share of the previous layer's pre-activations, on its way while
    // the products run: a thread handles two columns of every eighth row (in
    // tiles of at most 32 or 16 columns of every 16th or 32nd).  (Read in the row loop, one column per
    // lane, each row's load waited behind the previous row's stores: a backward
    // launch of 4 networks, 256 rows and 256 columns took 26 us, now 8; a forward one
    // 14.5, now 8.5, cold caches)
    constexpr int kWarps = kGemmThreads / 32;
    const int rows = min(kTileM, g.M - m0);
    const bool pairs = nt <= 64 && g.ldc % 2 == 0 && n0 % 2 == 0 && g.zc % 2 == 0;
    // a tile of at most 32 (16) columns: half (a quarter of) a warp per row
    const int lpr = nt <= 16 ? 8 : nt <= 32 ? 16 : 32, rpw = 32 / lpr;
    const int col = 2 * (lane & (lpr - 1));
    const int row_in = warp * rpw + lane / lpr;
    const bool mine = col < nt;
    constexpr int kRowGroup = 4; // rows per pass of the row loop
    const size_t pair0 = (size_t)z * g.zc + (size_t)(m0 + row_in) * g.ldc + n0 + col;
    const size_t row_step = (size_t)(kWarps * rpw) * g.ldc;
    const int passes = kTileM / (kWarps * rpw);
    float2 zreg[kRowGroup];
    auto load_z = [&](int q0) {
#pragma unroll
        for (int u = 0; u < kRowGroup; ++u)
            zreg[u] = mine && (q0 + u) * kWarps * rpw + row_in < rows
                          ? *reinterpret_cast<const float2 *>(g.Z + pair0 + (q0 + u) * row_step)
                          : make_float2(0.f, 0.f);
    };
    if (pairs && g.mode == GEMM_DACT)
        load_z(0);

    // wait for the accumulator (bounded), then the epilogue
    if (!mbar_wait_bounded(done_bar, 0, wb))
        atomicExch(&s_abort, 1);
    __syncthreads();
    const bool abort = s_abort != 0;
    if (abort) {
        if (tid == 0) {
            atomicOr(g.flags, FLAG_TIMEOUT);
            // let the copies still in flight land before the CTA leaves: at most
            // one outstanding load per stage (the last one issued)
            const int issued = s_issued;
            for (int s = 0; s < stages && s < issued; ++s) {
                const int u_last = (issued - 1 - s) / stages;
                mbar_wait_bounded(smem_addr(&full[s]), (uint32_t)(u_last & 1));
            }
            mbar_wait_bounded(done_bar, 0);
        }
    } else {
        asm volatile("tcgen05.fence::after_thread_sync;");
        float *S = reinterpret_cast<float *>(smem);
        const int pitch = g.n_tile + 1;
        const int quad = warp & 3, half = warp >> 2;
        const int rl = quad * 32 + lane;
        for (int j = half * 16; j < nt; j += 32) {
            uint32_t r[16];
            const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)j;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                         "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                           "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
                           "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                         : "r"(taddr));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int q = 0; q < 16; ++q)
                S[rl * pitch + j + q] = __uint_as_float(r[q]);
        }
        __syncthreads();
        // one warp per output row, lanes along the columns (coalesced)
        const float *bias = g.bias ? g.bias + (size_t)z * g.zbias + n0 : nullptr;
        if (pairs) { // two columns per lane
            const float2 b2 = bias && mine ? make_float2(bias[col], bias[col + 1])
                                   : make_float2(0.f, 0.f);
#pragma unroll 1
            for (int q0 = 0; q0 < passes; q0 += kRowGroup) {
                float2 zc[kRowGroup];
#pragma unroll
                for (int u = 0; u < kRowGroup; ++u)
                    zc[u] = zreg[u];
                if (g.mode == GEMM_DACT && q0 + kRowGroup < passes)
                    load_z(q0 + kRowGroup);
#pragma unroll
                for (int u = 0; u < kRowGroup; ++u) {
                    const int rr = (q0 + u) * kWarps * rpw + row_in;
                    if (!mine || rr >= rows)
                        break;
                    const size_t o = pair0 + (q0 + u) * row_step;
                    float *Sr = S + rr * pitch + col;
                    float2 v = make_float2(Sr[0], Sr[1]);
                    if (g.mode == GEMM_DACT) {
                        v = make_float2(v.x * dsilu(zc[u].x), v.y * dsilu(zc[u].y));
                    } else if (bias) {
                        v = make_float2(v.x + b2.x, v.y + b2.y);
                    }
                    if (g.mode == GEMM_ACT) {
                        if (g.Z)
                            *reinterpret_cast<float2 *>(g.Z + o) = v;
                        if (g.act)
                            v = make_float2(silu(v.x), silu(v.y));
                    }
                    if (g.mode != GEMM_F32)
                        *reinterpret_cast<__nv_bfloat162 *>(g.Cb + o) = __floats2bfloat162_rn(v.x, v.y);
                    if (g.Cf)
                        *reinterpret_cast<float2 *>(g.Cf + o) = v;
                    if (g.CbT) {
                        Sr[0] = v.x;
                        Sr[1] = v.y;
                    }
                }
            }
        } else {
            for (int rr = warp; rr < rows; rr += kWarps) {
                const size_t ro = (size_t)z * g.zc + (size_t)(m0 + rr) * g.ldc + n0;
                float *Sr = S + rr * pitch;
                for (int cc = lane; cc < nt; cc += 32) {
                    const size_t o = ro + cc;
                    float v = Sr[cc];
                    if (g.mode == GEMM_F32) {
                        if (bias)
                            v += bias[cc];
                        g.Cf[o] = v;
                    } else if (g.mode == GEMM_ACT) {
                        if (bias)
                            v += bias[cc];
                        if (g.Z)
                            g.Z[o] = v;
                        const float act = g.act ? silu(v) : v;
                        g.Cb[o] = __float2bfloat16_rn(act);
                        if (g.Cf)
                            g.Cf[o] = act;
                        Sr[cc] = act;
                    } else { // GEMM_DACT: gradient through the SiLU of the previous layer
                        const float d = v * dsilu(g.Z[o]);
                        g.Cb[o] = __float2bfloat16_rn(d);
                        if (g.Cf)
                            g.Cf[o] = d;
                        Sr[cc] = d;
                    }
                }
            }
        }
        if (g.CbT) { // the transposed copy: one warp per column, lanes along the rows
            __syncthreads();
            for (int cc = warp; cc < nt; cc += kWarps) {
                __nv_bfloat16 *o = g.CbT + (size_t)z * g.zt + (size_t)(n0 + cc) * g.ldt + m0;
                if (rows == kTileM && g.ldt % 2 == 0 && g.zt % 2 == 0) {
#pragma unroll
                    for (int rr = 2 * lane; rr < kTileM; rr += 64)
                        *reinterpret_cast<__nv_bfloat162 *>(o + rr) = __floats2bfloat162_rn(
                            S[rr * pitch + cc], S[(rr + 1) * pitch + cc]);
                } else {
                    for (int rr = lane; rr < rows; rr += 32)
                        o[rr] = __float2bfloat16_rn(S[rr * pitch + cc]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(g.tmem_cols));
}

// Products g0 (tiles 0 .. nb0 - 1 of blockIdx.x) and g1 (the rest) for the
// networks blockIdx.y.  The training passes are chains of small products (a few
// tiles each): what they cost is the launches, so all networks share one, and the
// weight gradient of a layer runs beside the gradient handed to the layer below.
__global__ void __launch_bounds__(kGemmThreads, 1)
k_gemm_bf16(const __grid_constant__ CUtensorMap tA0, const __grid_constant__ CUtensorMap tB0,
            const __grid_constant__ CUtensorMap tA1, const __grid_constant__ CUtensorMap tB1,
            const __grid_constant__ GemmArgs g0, const __grid_constant__ GemmArgs g1, int stages0,
            int stages1, int nb0)
{
    // one copy of the tile's code for both products: with two, their row loops
    // unrolled, a backward launch on cold caches took 15 us, half of it waiting for
    // instructions (now 10; 512 rows in the running chain 170 -> 165 us a minibatch)
    const bool second = (int)blockIdx.x >= nb0;
    const GemmArgs &g = second ? g1 : g0;
    const int x = blockIdx.x - (second ? nb0 : 0), mb = (g.M + kTileM - 1) / kTileM;
    gemm_tile(second ? &tA1 : &tA0, second ? &tB1 : &tB0, g, second ? stages1 : stages0, x % mb,
              x / mb, blockIdx.y);
}

// ---------------------------------------------------------------------------
// Fused inference of the whole network: one CTA runs every layer of one
// network on 128 rows of the batch, so activations never leave the SM.
//  * the A operand of every layer lives in shared memory (`abuf`, canonical
//    no-swizzle K-major layout): layer 0's input arrives by TMA, the epilogue
//    of layer l writes the BF16 activations of layer l + 1 into the same
//    buffer once layer l's MMAs have completed;
//  * weights stream by TMA through a ring of kInferStages stages of up to
//    N x 64 BF16 (one producer thread, running ahead across layers);
//  * one thread issues tcgen05.mma (M = 128, N = layer width, K = 16) into
//    one TMEM accumulator that every layer reuses;
//  * 8 epilogue warps read the accumulator (tcgen05.ld), add the bias, apply
//    SiLU and write BF16 activations (hidden layers) or FP32 outputs (last
//    layer, to the network's slice of y); they release the next layer with
//    an mbarrier after a proxy fence (generic writes -> tensor-core reads).
// The arithmetic is that of the layer-by-layer GEMM path (same MMA sequence,
// same epilogue operations), so both give the same bits.
constexpr int kInferThreads = 320; // warp 0 producer, warp 1 MMA, warps 2-9 epilogue
constexpr int kInferStages = 3;

// Tensor maps of the fused inference: the batch input (rows x in_p) and, per
// layer, the weights of every network stacked along the rows (n_nets * N x K).
struct MlpMaps {
    CUtensorMap x;
    CUtensorMap w[kMaxMlpLayers + 1];
};

struct MlpDev {
    int NL, in_p, H, out_p, bp, tmem_cols, abuf_bytes, stage_bytes;
    const float *bias[kMaxMlpLayers + 1]; // per layer, network k at k bias_stride
    int bias_stride;
    float *y;                              // [n_nets][bp][out_p]
    int *flags;
};

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ int infer_k(const MlpDev &d, int l) { return l == 0 ? d.in_p : d.H; }
__device__ __forceinline__ int infer_n(const MlpDev &d, int l) { return l == d.NL ? d.out_p : d.H; }

__global__ void __launch_bounds__(kInferThreads, 1)
k_mlp_infer(const __grid_constant__ MlpMaps maps, MlpDev d)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t full[kInferStages], empty[kInferStages], x_full, acc_full,
        act_ready, drain, bias_ready;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort, s_issued, s_x_issued;
    __shared__ float s_bias[2][256]; // the epilogue's bias, by layer parity

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int net = blockIdx.y;
    const int m0 = blockIdx.x * kTileM;
    const uint32_t abuf = smem_addr(smem);
    const uint32_t ring = abuf + (uint32_t)d.abuf_bytes;
    const uint32_t sbytes = (uint32_t)d.stage_bytes;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(&s_tmem)),
                     "r"(d.tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int s = 0; s < kInferStages; ++s) {
            mbar_init(smem_addr(&full[s]), 1);
            mbar_init(smem_addr(&empty[s]), 1);
        }
        mbar_init(smem_addr(&x_full), 1);
        mbar_init(smem_addr(&acc_full), 1);
        mbar_init(smem_addr(&act_ready), 8); // one arrival per epilogue warp
        mbar_init(smem_addr(&drain), 1);
        mbar_init(smem_addr(&bias_ready), kInferThreads - 64); // every epilogue thread
        asm volatile("fence.mbarrier_init.release.cluster;");
        s_abort = 0;
        s_issued = 0;
        s_x_issued = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = s_tmem;
    net += after_previous();

    if (warp == 0) {
        if (lane == 0) { // TMA producer: the input tile, then every layer's weights
            const uint32_t xb = smem_addr(&x_full);
            mbar_expect_tx(xb, (uint32_t)(kTileM * d.in_p * 2));
            for (int kg = 0; kg < d.in_p / 8; ++kg)
                tma_load_2d(abuf + (uint32_t)(kg * kTileM * 16), &maps.x, kg * 8, m0, xb);
            s_x_issued = 1;
            int c = 0;
            bool ok = true;
            for (int l = 0; l <= d.NL && ok; ++l) {
                const int K = infer_k(d, l), N = infer_n(d, l);
                const int row0 = net * N;
                for (int k0 = 0; k0 < K; k0 += kChunkK, ++c) {
                    const int s = c % kInferStages, u = c / kInferStages;
                    if (u > 0 && !mbar_wait_bounded(smem_addr(&empty[s]), (uint32_t)((u - 1) & 1))) {
                        atomicExch(&s_abort, 1);
                        ok = false;
                        break;
                    }
                    const uint32_t sb = ring + (uint32_t)s * sbytes, fb = smem_addr(&full[s]);
                    mbar_expect_tx(fb, (uint32_t)(N * kChunkK * 2));
                    tma_load_2d(sb, &maps.w[l], k0, row0, fb);
                }
            }
            s_issued = c;
        }
        __syncwarp();
    } else if (warp == 1) {
        if (lane == 0) { // MMA issuer
            int c = 0;
            bool ok = true;
            for (int l = 0; l <= d.NL && ok; ++l) {
                const uint32_t gate = l == 0 ? smem_addr(&x_full) : smem_addr(&act_ready);
                const uint32_t par = l == 0 ? 0u : (uint32_t)((l - 1) & 1);
                if (!mbar_wait_bounded(gate, par)) {
                    atomicExch(&s_abort, 1);
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;");
                const int K = infer_k(d, l), N = infer_n(d, l);
                const uint32_t idesc = idesc_bf16(kTileM, N);
                for (int k0 = 0; k0 < K; k0 += kChunkK, ++c) {
                    const int s = c % kInferStages, u = c / kInferStages;
                    if (!mbar_wait_bounded(smem_addr(&full[s]), (uint32_t)(u & 1))) {
                        atomicExch(&s_abort, 1);
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    const int kc = min(kChunkK, K - k0);
                    const uint32_t sb = ring + (uint32_t)s * sbytes;
                    for (int ks = 0; ks < kc; ks += 16) {
                        const int k = k0 + ks;
                        const uint64_t ad = smem_desc(abuf + (uint32_t)((k / 8) * kTileM * 16),
                                                      kTileM * 16, 128);
                        const uint64_t bd = smem_desc_sw128(sb + (uint32_t)(ks * 2));
                        const uint32_t acc = k > 0 ? 1u : 0u;
                        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(
                                         tmem),
                                     "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
                    }
                    mma_commit(smem_addr(&empty[s]));
                }
                mma_commit(smem_addr(&acc_full)); // this layer's accumulator is complete
            }
            mma_commit(smem_addr(&drain)); // every MMA issued has completed (also after an abort)
        }
        __syncwarp();
    } else { // epilogue warps 2..9: TMEM lanes 32 (warp mod 4) .. +31, alternate 16-column groups
        const int quad = warp & 3, half = (warp - 2) >> 2;
        const int r = quad * 32 + lane; // row inside the tile
        for (int l = 0; l <= d.NL; ++l) {
            const int N = infer_n(d, l);
            // this layer's bias into shared memory while its MMAs run.  Every
            // epilogue thread arrives after its store and waits for all 256
            // (bounded): the completed phase also shows that every thread has
            // left the previous layer, so the other parity's buffer is free
            float *bias = s_bias[l & 1];
            if (tid - 64 < N)
                bias[tid - 64] = d.bias[l][(size_t)net * d.bias_stride + (tid - 64)];
            mbar_arrive(smem_addr(&bias_ready));
            if (!mbar_wait_bounded(smem_addr(&bias_ready), (uint32_t)(l & 1)) ||
                !mbar_wait_bounded(smem_addr(&acc_full), (uint32_t)(l & 1))) {
                atomicExch(&s_abort, 1);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const bool last = l == d.NL;
            float *yrow = last ? d.y + ((size_t)net * d.bp + m0 + r) * d.out_p : nullptr;
            for (int j = half * 16; j < N; j += 32) {
                uint32_t v[16];
                const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)j;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 "
                             "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                             : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]),
                               "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                               "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                               "=r"(v[15])
                             : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (last) {
#pragma unroll
                    for (int q = 0; q < 16; q += 4)
                        *reinterpret_cast<float4 *>(yrow + j + q) = make_float4(
                            __uint_as_float(v[q]) + bias[j + q],
                            __uint_as_float(v[q + 1]) + bias[j + q + 1],
                            __uint_as_float(v[q + 2]) + bias[j + q + 2],
                            __uint_as_float(v[q + 3]) + bias[j + q + 3]);
                } else {
#pragma unroll
                    for (int h8 = 0; h8 < 2; ++h8) { // two 8-column core-matrix rows
                        uint32_t p[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int q = h8 * 8 + 2 * e;
                            const float a0 = silu(__uint_as_float(v[q]) + bias[j + q]);
                            const float a1 = silu(__uint_as_float(v[q + 1]) + bias[j + q + 1]);
                            const __nv_bfloat162 b2 = __floats2bfloat162_rn(a0, a1);
                            p[e] = *reinterpret_cast<const uint32_t *>(&b2);
                        }
                        const int col = j + h8 * 8;
                        uint8_t *dst = smem + (size_t)(col / 8) * kTileM * 16 + (size_t)r * 16;
                        *reinterpret_cast<uint4 *>(dst) = make_uint4(p[0], p[1], p[2], p[3]);
                    }
                }
            }
            if (!last) { // the activations are the next layer's A operand
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;");
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(smem_addr(&act_ready));
            }
        }
    }

    __syncthreads();
    if (s_abort) {
        if (tid == 0) {
            atomicOr(d.flags, FLAG_TIMEOUT);
            // copies still in flight land before the CTA leaves (at most the
            // last one issued per stage, and the input tile)
            const int issued = s_issued;
            for (int s = 0; s < kInferStages && s < issued; ++s) {
                const int u_last = (issued - 1 - s) / kInferStages;
                mbar_wait_bounded(smem_addr(&full[s]), (uint32_t)(u_last & 1));
            }
            if (s_x_issued)
                mbar_wait_bounded(smem_addr(&x_full), 0);
            mbar_wait_bounded(smem_addr(&drain), 0);
        }
        __syncthreads();
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(d.tmem_cols));
}

// out[c][r] = in[r][c] for an R x C BF16 matrix (32 x 32 tiles in shared memory).
__global__ void k_transpose_bf16(const __nv_bfloat16 *__restrict__ in, int R, int C, int ldi,
                                 __nv_bfloat16 *__restrict__ out, int ldo)
{
    __shared__ __nv_bfloat16 t[32][33];
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int r = r0 + k, c = c0 + threadIdx.x;
        t[k][threadIdx.x] = (r < R && c < C) ? in[(size_t)r * ldi + c] : __float2bfloat16_rn(0.f);
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int c = c0 + k, r = r0 + threadIdx.x;
        if (c < C && r < R)
            out[(size_t)c * ldo + r] = t[threadIdx.x][k];
    }
}

// Mean-squared error over rows < m_valid and the first n_valid columns of a
// padded M x ldy output: dL/dy = 2 w_c (y - t) / (m_valid * n_valid) (FP32, BF16
// and its transpose); loss accumulated (sum of w_c (y - t)^2 / (m_valid n_valid)).
// Network blockIdx.y.
__global__ void k_mse_grad(const float *__restrict__ y, const float *__restrict__ t,
                           const float *__restrict__ w, int M, int m_valid, int n_valid,
                           int ldy, float *__restrict__ gf, __nv_bfloat16 *__restrict__ gb,
                           __nv_bfloat16 *__restrict__ gbT, float *__restrict__ loss)
{
    const size_t z = (size_t)blockIdx.y * M * ldy;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x + after_previous();
    const int r = idx / ldy, c = idx - r * ldy;
    float g = 0.f, l = 0.f;
    if (r < M) {
        if (r < m_valid && c < n_valid) {
            const float e = y[z + idx] - t[z + (size_t)r * ldy + c];
            const float wc = w ? w[c] : 1.f;
            const float s = 1.0f / ((float)m_valid * (float)n_valid);
            g = 2.f * wc * e * s;
            l = wc * e * e * s;
        }
        gf[z + idx] = g;
        gb[z + idx] = __float2bfloat16_rn(g);
        gbT[z + (size_t)c * M + r] = __float2bfloat16_rn(g);
    }
    // warp reduction of the loss, one atomic per warp
    for (int o = 16; o > 0; o >>= 1)
        l += __shfl_down_sync(0xffffffffu, l, o);
    if ((threadIdx.x & 31) == 0 && l != 0.f)
        atomicAdd(loss + blockIdx.y, l);
}

// Column sums of M x out_p FP32 matrices (bias gradients of layer blockIdx.y,
// network blockIdx.z), 32 columns per CTA, rows in fixed order (deterministic): the
// CTA brings 256 rows at a time into shared memory, and one warp adds them, so that
// the chain of adds and not the loads' latency sets the time (4 networks, 256 rows,
// 1104 columns: 8.5 us; one warp per 32 columns reading 16 rows ahead took 13.4).
__global__ void __launch_bounds__(256)
k_colsum(const __grid_constant__ ColsumArgs a, const __grid_constant__ NetDims d, float *__restrict__ grads)
{
    __shared__ float t[256][32];
    const int l = blockIdx.y, N = d.out_p[l];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane + after_previous();
    if ((int)blockIdx.x * 32 >= N)
        return;
    const float *G = a.G[l] + (size_t)blockIdx.z * a.M * N + c;
    float s = 0.f;
    for (int r0 = 0; r0 < a.M; r0 += 256) {
        const int rows = min(256, a.M - r0);
        if (c < N) {
#pragma unroll 8
            for (int r = warp; r < rows; r += 8)
                t[r][lane] = G[(size_t)(r0 + r) * N];
        }
        __syncthreads();
        if (warp == 0 && c < N) {
#pragma unroll 16
            for (int r = 0; r < rows; ++r)
                s += t[r][lane];
        }
        __syncthreads();
    }
    if (warp == 0 && c < N)
        grads[(size_t)blockIdx.z * d.n_params + d.off[l] + d.out_p[l] * d.in_p[l] + c] = s;
}

// The 32 x 32 tiles of every layer's weights, then its biases, counted through the
// layers (blockIdx.x of the kernels below).
struct ParamTile {
    int l, r0, c0; // r0 < 0: the biases
};

__host__ __device__ inline int layer_tiles(const NetDims &d, int l)
{
    return ((d.out_p[l] + 31) / 32) * ((d.in_p[l] + 31) / 32) + 1;
}

__device__ __forceinline__ ParamTile param_tile(const NetDims &d, int x)
{
    int l = 0;
    for (; l + 1 < d.n_layers && x >= layer_tiles(d, l); ++l)
        x -= layer_tiles(d, l);
    const int tc = (d.in_p[l] + 31) / 32;
    return x == layer_tiles(d, l) - 1 ? ParamTile{l, -1, 0} : ParamTile{l, x / tc * 32, x % tc * 32};
}

// The BF16 copy of a 32 x 32 tile of weights (thread (tx, ty): column tx, rows ty,
// ty + 8, ...) and its transpose, which goes through shared memory: written weight
// by weight, each two bytes touched a sector of their own (AdamW of 4 networks of
// 222 k parameters: 8.7 us, before 13.4).
__device__ __forceinline__ void put_tile(const NetDims &d, int k, const ParamTile &p,
                                         const float (&w)[4], __nv_bfloat16 (&t)[32][33])
{
    const int rows = d.out_p[p.l], cols = d.in_p[p.l];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const size_t base = (size_t)k * rows * cols;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = p.r0 + ty + 8 * q, c = p.c0 + tx;
        const __nv_bfloat16 b = __float2bfloat16_rn(w[q]);
        t[ty + 8 * q][tx] = b;
        if (r < rows && c < cols)
            d.Wb[p.l][base + (size_t)r * cols + c] = b;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int c = p.c0 + ty + 8 * q, r = p.r0 + tx;
        if (r < rows && c < cols)
            d.Wt[p.l][base + (size_t)c * rows + r] = t[tx][ty + 8 * q];
    }
}

// AdamW (I. Loshchilov, F. Hutter, "Decoupled weight decay regularization"):
// m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2; w -= lr (m_hat / (sqrt(v_hat) + eps) + wd w),
// with m_hat = m / (1 - b1^t), v_hat = v / (1 - b2^t).  The mask keeps padded
// entries at zero; biases do not decay.
__device__ __forceinline__ float adamw_one(size_t idx, unsigned char mk, float *__restrict__ w,
                                           const float *__restrict__ g, float *__restrict__ m,
                                           float *__restrict__ v, const AdamArgs &a)
{
    float wi = w[idx];
    if (mk & 1) {
        const float wd = mk & 2 ? a.wd : 0.f;
        const float gi = g[idx];
        const float mi = a.b1 * m[idx] + (1.f - a.b1) * gi;
        const float vi = a.b2 * v[idx] + (1.f - a.b2) * gi * gi;
        m[idx] = mi;
        v[idx] = vi;
        const float mh = mi / a.bc1, vh = vi / a.bc2;
        wi -= a.lr * (mh / (sqrtf(vh) + a.eps) + wd * wi);
        w[idx] = wi;
    }
    return wi;
}

// AdamW and the BF16 copies, one tile per CTA.  Network k0 + blockIdx.y.
__global__ void __launch_bounds__(256)
k_adamw(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m,
        float *__restrict__ v, const unsigned char *__restrict__ mask,
        const __grid_constant__ NetDims d, int k0, AdamArgs a)
{
    __shared__ __nv_bfloat16 t[32][33];
    const ParamTile p = param_tile(d, blockIdx.x);
    const int k = k0 + blockIdx.y, rows = d.out_p[p.l], cols = d.in_p[p.l];
    const size_t net = (size_t)k * d.n_params + after_previous();
    if (p.r0 < 0) {
        for (int c = threadIdx.x; c < rows; c += blockDim.x) {
            const int e = d.off[p.l] + rows * cols + c;
            adamw_one(net + e, mask[e], w, g, m, v, a);
        }
        return;
    }
    float wt[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = p.r0 + (threadIdx.x >> 5) + 8 * q, c = p.c0 + (threadIdx.x & 31);
        const int e = d.off[p.l] + r * cols + c;
        wt[q] = r < rows && c < cols ? adamw_one(net + e, mask[e], w, g, m, v, a) : 0.f;
    }
    put_tile(d, k, p, wt, t);
}

// BF16 copies of the flat parameters of network k.
__global__ void __launch_bounds__(256)
k_weights_bf16(const float *__restrict__ w, const __grid_constant__ NetDims d, int k)
{
    __shared__ __nv_bfloat16 t[32][33];
    const ParamTile p = param_tile(d, blockIdx.x);
    if (p.r0 < 0)
        return;
    const int rows = d.out_p[p.l], cols = d.in_p[p.l];
    float wt[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = p.r0 + (threadIdx.x >> 5) + 8 * q, c = p.c0 + (threadIdx.x & 31);
        wt[q] = r < rows && c < cols ? w[(size_t)k * d.n_params + d.off[p.l] + r * cols + c] : 0.f;
    }
    put_tile(d, k, p, wt, t);
}

} // namespace

namespace {

// cuTensorMapEncodeTiled from the driver, looked up once through the runtime.
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool looked = false;
    if (!looked) {
        looked = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// Tensor map of a row-major BF16 matrix (rows x K, leading dimension ld elements)
// read in boxes of 64 K-columns x box_rows rows in the 128-byte swizzle, or of 8
// K-columns without (`plain`); out-of-range rows and columns read as zero.
bool encode_operand(CUtensorMap *m, const __nv_bfloat16 *ptr, int rows, int K, int ld,
                    int box_rows, bool plain = false)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc)
        return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {plain ? 8u : (cuuint32_t)kChunkK, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void *)ptr, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE,
               plain ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

} // namespace

namespace {
bool gemm_ok(const GemmArgs &g)
{
    return !(g.M <= 0 || g.N <= 0 || g.K <= 0 || (g.N % 16) || (g.K % 16) || (g.n_tile % 16) ||
             g.n_tile < 16 || g.n_tile > kMaxTileN || (g.lda % 8) || (g.ldb % 8) || g.lda < g.K ||
             g.ldb < g.K || ((uintptr_t)g.A % 16) || ((uintptr_t)g.B % 16) || g.nz < 1);
}

int gemm_stages(const GemmArgs &g)
{
    const int nchunks = (g.K + kChunkK - 1) / kChunkK;
    int stages = kStageBudget / stage_bytes(g.n_tile);
    stages = stages < kMaxStages ? stages : kMaxStages;
    return stages < nchunks ? stages : nchunks;
}

int gemm_tiles(const GemmArgs &g)
{
    return ((g.M + kTileM - 1) / kTileM) * ((g.N + g.n_tile - 1) / g.n_tile);
}

bool gemm_maps(const GemmArgs &g, CUtensorMap *ta, CUtensorMap *tb)
{
    return encode_operand(ta, g.A, (g.nz - 1) * g.za + g.M, g.K, g.lda, kTileM) &&
           encode_operand(tb, g.B, (g.nz - 1) * g.zb + g.N, g.K, g.ldb, g.n_tile);
}
} // namespace

cudaError_t launch_gemm(const GemmArgs &g0, const GemmArgs *g1, cudaStream_t st)
{
    if (!gemm_ok(g0) || (g1 && (!gemm_ok(*g1) || g1->nz != g0.nz)))
        return cudaErrorInvalidValue;
    static bool attr_done = false;
    if (!attr_done) {
        cudaError_t e = cudaFuncSetAttribute(k_gemm_bf16, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             dyn_smem_bytes(kMaxTileN, kMaxStages));
        if (e != cudaSuccess)
            return e;
        attr_done = true;
    }
    CUtensorMap ta0, tb0, ta1{}, tb1{};
    if (!gemm_maps(g0, &ta0, &tb0) || (g1 && !gemm_maps(*g1, &ta1, &tb1)))
        return cudaErrorInvalidValue;
    const int s0 = gemm_stages(g0), s1 = g1 ? gemm_stages(*g1) : 0;
    const int nb0 = gemm_tiles(g0), nb1 = g1 ? gemm_tiles(*g1) : 0;
    int smem = dyn_smem_bytes(g0.n_tile, s0);
    if (g1 && dyn_smem_bytes(g1->n_tile, s1) > smem)
        smem = dyn_smem_bytes(g1->n_tile, s1);
    return launch_after(k_gemm_bf16, dim3(nb0 + nb1, g0.nz), kGemmThreads, smem, st, ta0, tb0, ta1, tb1,
                        g0, g1 ? *g1 : g0, s0, s1, nb0);
}

bool mlp_infer_supported(int NL, int in_p, int H, int out_p)
{
    return NL >= 1 && NL <= kMaxMlpLayers && H >= 16 && H <= 256 && H % 16 == 0 &&
           out_p >= 16 && out_p <= 256 && out_p % 16 == 0 && in_p >= 16 && in_p <= 256 &&
           in_p % 16 == 0;
}

cudaError_t launch_mlp_infer(const MlpInferArgs &a, cudaStream_t st)
{
    if (!mlp_infer_supported(a.NL, a.in_p, a.H, a.out_p) || a.bp < kTileM || a.bp % kTileM ||
        a.n_nets < 1 || !a.X || !a.y)
        return cudaErrorInvalidValue;
    const int kmax = a.in_p > a.H ? a.in_p : a.H;
    const int nmax = a.H > a.out_p ? a.H : a.out_p;
    MlpDev d{};
    d.NL = a.NL;
    d.in_p = a.in_p;
    d.H = a.H;
    d.out_p = a.out_p;
    d.bp = a.bp;
    d.tmem_cols = 32;
    while (d.tmem_cols < nmax) // TMEM columns: a power of two >= 32
        d.tmem_cols *= 2;
    d.abuf_bytes = (kTileM * kmax * 2 + 1023) / 1024 * 1024;
    d.stage_bytes = nmax * kChunkK * 2;
    d.y = a.y;
    d.flags = a.flags;
    MlpMaps maps{};
    if (!encode_operand(&maps.x, a.X, a.bp, a.in_p, a.in_p, kTileM, true))
        return cudaErrorInvalidValue;
    for (int l = 0; l <= a.NL; ++l) {
        const int K = l == 0 ? a.in_p : a.H, N = l == a.NL ? a.out_p : a.H;
        if (!a.W[l] || !a.b[l] || ((uintptr_t)a.W[l] % 16) ||
            !encode_operand(&maps.w[l], a.W[l], a.n_nets * N, K, K, N))
            return cudaErrorInvalidValue;
        d.bias[l] = a.b[l];
        d.bias_stride = a.b_stride;
    }
    const int smem = d.abuf_bytes + kInferStages * d.stage_bytes;
    static bool attr_done = false;
    if (!attr_done) {
        cudaError_t e = cudaFuncSetAttribute(k_mlp_infer, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kTileM * 256 * 2 + kInferStages * 256 * kChunkK * 2);
        if (e != cudaSuccess)
            return e;
        attr_done = true;
    }
    dim3 grid(a.bp / kTileM, a.n_nets);
    return launch_after(k_mlp_infer, grid, kInferThreads, smem, st, maps, d);
}

cudaError_t launch_transpose_bf16(const void *in, int R, int C, int ldi, void *out, int ldo,
                                  cudaStream_t st)
{
    dim3 grid((C + 31) / 32, (R + 31) / 32);
    k_transpose_bf16<<<grid, dim3(32, 8), 0, st>>>((const __nv_bfloat16 *)in, R, C, ldi,
                                                   (__nv_bfloat16 *)out, ldo);
    return cudaGetLastError();
}

cudaError_t launch_mse_grad(const float *y, const float *t, const float *w, int M, int m_valid,
                            int n_valid, int ldy, int nz, float *gf, void *gb, void *gbT,
                            float *loss, cudaStream_t st)
{
    const int n = M * ldy;
    return launch_after(k_mse_grad, dim3((n + 255) / 256, nz), 256, 0, st, y, t, w, M, m_valid, n_valid,
                        ldy, gf, (__nv_bfloat16 *)gb, (__nv_bfloat16 *)gbT, loss);
}

cudaError_t launch_colsum(const ColsumArgs &c, const NetDims &d, float *grads, cudaStream_t st)
{
    int w = 0;
    for (int l = 0; l < d.n_layers; ++l)
        w = d.out_p[l] > w ? d.out_p[l] : w;
    return launch_after(k_colsum, dim3((w + 31) / 32, d.n_layers, c.nz), 256, 0, st, c, d, grads);
}

static int param_tiles(const NetDims &d)
{
    int n = 0;
    for (int l = 0; l < d.n_layers; ++l)
        n += layer_tiles(d, l);
    return n;
}

cudaError_t launch_adamw(float *w, const float *g, float *m, float *v, const unsigned char *mask,
                         const NetDims &d, int k0, int nz, const AdamArgs &a, cudaStream_t st)
{
    return launch_after(k_adamw, dim3(param_tiles(d), nz), 256, 0, st, w, g, m, v, mask, d, k0, a);
}

cudaError_t launch_weights_bf16(const float *w, const NetDims &d, int k, cudaStream_t st)
{
    k_weights_bf16<<<param_tiles(d), 256, 0, st>>>(w, d, k);
    return cudaGetLastError();
}

} // namespace npsim
