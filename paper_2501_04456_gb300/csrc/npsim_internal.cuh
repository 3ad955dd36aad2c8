// npsim_internal.cuh -- device-side types and helpers shared by the library's
// CUDA translation units (never by the CPU oracle).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include "../../include/npsim.h"

namespace npsim {

// ---------------------------------------------------------------------------
// The kernels of a surrogate's training pass or prediction, queued one after another,
// start before the kernel in front has ended (programmatic dependent launch): the
// launch and the CTAs' setup (barriers, tensor memory) go on during its last wave.  A
// kernel launched by launch_after calls after_previous() and reads or writes nothing
// that a kernel writes before that; from there on every kernel queued before it is
// complete (each one in the chain has waited for the one in front, so that none can be
// overtaken), and only then may the next one start early.  The value returned, zero,
// goes into the indices of all loads that follow: the compiler, which takes loads
// through read-only pointers to be movable across the wait, sees that they depend on
// it.  Fourteen launches of a minibatch of 256 for 4 networks: 133 -> 97 us.  The steps of
// a simulation are captured graphs, whose kernels follow each other closely as it is:
// there the early CTAs gave nothing (ensembles, all pairs: within 0.5 %) or took
// (list steps of 250 k NPs: 19.0 -> 19.5 us).
__device__ __forceinline__ int after_previous()
{
    int zero;
    asm volatile("griddepcontrol.wait;\n\t"
                 "mov.u32 %0, 0;\n\t"
                 "griddepcontrol.launch_dependents;"
                 : "=r"(zero)
                 :
                 : "memory");
    return zero;
}

template <class... P, class... A>
cudaError_t launch_after(void (*fn)(P...), dim3 grid, int block, size_t smem, cudaStream_t st,
                         const A &...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}


// ---------------------------------------------------------------------------
// Error word bits (device int, read once per npsim_step).
enum : int {
    FLAG_NONFINITE = 1,
    FLAG_TIMEOUT = 2,
    FLAG_BAD_CELL = 4,
    FLAG_NBR_OVERFLOW = 8, // some NP had more list partners than the list holds (not an error)
    FLAG_ESCAPED = 16,     // an NP farther than 2 max(R0, R(t)) from the centre, full spring on
};

// ---------------------------------------------------------------------------
// Philox4x32-10 (J. K. Salmon et al., "Parallel random numbers: as easy as
// 1, 2, 3", SC'11): ten rounds of two 32x32->64 multiplies mixing the counter,
// with the key advanced by the two Weyl increments between rounds.
struct U4 {
    uint32_t x, y, z, w;
};

__device__ __forceinline__ U4 philox10(U4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t m0 = 0xD2511F53u, m1 = 0xCD9E8D57u;
        uint32_t lo0 = c.x * m0, hi0 = __umulhi(c.x, m0);
        uint32_t lo1 = c.z * m1, hi1 = __umulhi(c.z, m1);
        c = U4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// Three standard normals of particle i at step `step` (counter (i, step_lo,
// step_hi, purpose), key = seed).  Uniforms u = (k + 1/2) 2^-32, rounded to
// float; Box-Muller in float32 with the accurate logf, sincospif and cospif.
__device__ __forceinline__ void normals3(uint64_t seed, uint32_t i, int64_t step,
                                         uint32_t purpose, float &n0, float &n1, float &n2)
{
    const uint64_t s = (uint64_t)step;
    U4 r = philox10(U4{i, (uint32_t)s, (uint32_t)(s >> 32), purpose}, (uint32_t)seed,
                    (uint32_t)(seed >> 32));
    const float sc = 2.3283064365386963e-10f; // 2^-32
    float u0 = fmaf(__uint2float_rn(r.x), sc, 0.5f * sc);
    float u1 = fmaf(__uint2float_rn(r.y), sc, 0.5f * sc);
    float u2 = fmaf(__uint2float_rn(r.z), sc, 0.5f * sc);
    float u3 = fmaf(__uint2float_rn(r.w), sc, 0.5f * sc);
    // the radii sqrt(-2 ln u) as x rsqrt(x) (within two ulp of sqrt; 0 at u = 1)
    const float x1 = -2.0f * logf(u0), x2 = -2.0f * logf(u2);
    const float rho1 = x1 > 0.0f ? x1 * rsqrtf(x1) : 0.0f;
    const float rho2 = x2 > 0.0f ? x2 * rsqrtf(x2) : 0.0f;
    float s1, c1;
    sincospif(2.0f * u1, &s1, &c1);
    const float c3 = cospif(2.0f * u3); // the sine of this angle is not used
    n0 = rho1 * c1;
    n1 = rho1 * s1;
    n2 = rho2 * c3;
}

// Knuth's TwoSum: hi + lo accumulates a with the rounding error of hi + a
// carried in lo (compensated float32 accumulation).
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float a)
{
    float s = __fadd_rn(hi, a);
    float bp = __fsub_rn(s, hi);
    float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(a, bp));
    hi = s;
    lo = __fadd_rn(lo, err);
}

// ---------------------------------------------------------------------------
// Pair sums over grouped (padded) orders.
constexpr float kPairSelfEps = 1e-20f; // added to r^2; the self pair has r_ij = 0 exactly
constexpr float kPairSelfMin = 1e-12f; // LJ: r^2 below this is the self pair
constexpr float kPairPad = 1.0e18f;    // padding position: every term with it underflows to 0
// Smallest |C q_a q_b| in whose units sym_row_segment keeps its sums: below it
// the division of the LJ depth by it would bring the overflow of s^12 closer.
constexpr float kSymMinScale = 1e-4f;

// One j-tile of the packed LJ + Coulomb pair sum: KI rows per thread, JP
// partner pairs staged in shared memory as negated coordinates, s_a = (-x0,
// -x1, -y0, -y1), s_b = (-z0, -z1); cst[k] = (sigma_ab^2, 24 eps_ab, rc_ab^2,
// C q_a q_b) of row k and the tile's type.  Per pair:
//   d = x_i - x_j; r^2 = d.d (+ kPairSelfEps); 1/r = rsqrt(r^2); s^6 = (sigma_ab^2/r^2)^3;
//   f = [C q_a q_b / r + [r^2 < rc_ab^2] s^6 (48 eps_ab s^6 - 24 eps_ab)] / r^2,
//   a += f d
// (the bracket is 24 eps_ab (2 s^12 - s^6) r^2 / r^2, the LJ force over r),
// on the packed float32x2 instructions, two partners per register pair: 17
// packed instructions per two pairs, two MUFU.RSQ, two cutoff selects.  DIAG
// (a tile that holds a row's own column) also masks the self pair out of the
// LJ term, whose r^-14 would overflow there.
template <int KI, bool DIAG>
__device__ __forceinline__ void ljc_tile_sweep(const float4 *__restrict__ s_a,
                                               const float2 *__restrict__ s_b, int JP,
                                               const float2 (&xi)[KI], const float2 (&yi)[KI],
                                               const float2 (&zi)[KI], const float4 (&cst)[KI],
                                               float2 (&ax)[KI], float2 (&ay)[KI],
                                               float2 (&az)[KI])
{
    const float2 eps2 = make_float2(kPairSelfEps, kPairSelfEps);
    float2 sig2[KI], e48[KI], em24[KI], cqq[KI];
#pragma unroll
    for (int k = 0; k < KI; ++k) {
        sig2[k] = make_float2(cst[k].x, cst[k].x);
        e48[k] = make_float2(2.0f * cst[k].y, 2.0f * cst[k].y);
        em24[k] = make_float2(-cst[k].y, -cst[k].y);
        cqq[k] = make_float2(cst[k].w, cst[k].w);
    }
#pragma unroll 2
    for (int m = 0; m < JP; ++m) {
        const float4 a = s_a[m];
        const float2 nz = s_b[m];
        const float2 nx = make_float2(a.x, a.y), ny = make_float2(a.z, a.w);
#pragma unroll
        for (int k = 0; k < KI; ++k) {
            const float2 dx = __fadd2_rn(xi[k], nx);
            const float2 dy = __fadd2_rn(yi[k], ny);
            const float2 dz = __fadd2_rn(zi[k], nz);
            float2 r2 = __ffma2_rn(dz, dz, eps2);
            r2 = __ffma2_rn(dy, dy, r2);
            r2 = __ffma2_rn(dx, dx, r2);
            const float2 ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
            const float2 ri2 = __fmul2_rn(ri, ri);
            const float2 s2 = __fmul2_rn(sig2[k], ri2);
            const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
            float2 t = __fmul2_rn(s6, __ffma2_rn(e48[k], s6, em24[k]));
            if (DIAG) {
                t.x = (r2.x < cst[k].z && r2.x > kPairSelfMin) ? t.x : 0.0f;
                t.y = (r2.y < cst[k].z && r2.y > kPairSelfMin) ? t.y : 0.0f;
            } else {
                t.x = r2.x < cst[k].z ? t.x : 0.0f;
                t.y = r2.y < cst[k].z ? t.y : 0.0f;
            }
            const float2 f = __fmul2_rn(__ffma2_rn(cqq[k], ri, t), ri2);
            ax[k] = __ffma2_rn(f, dx, ax[k]);
            ay[k] = __ffma2_rn(f, dy, ay[k]);
            az[k] = __ffma2_rn(f, dz, az[k]);
        }
    }
}

// One j-tile of the Coulomb-only sum with the charge factored out: a += sum_j
// d / r^3 (the caller multiplies by the tile's C q_a q_b or q_t): 11 packed
// lanes per pair (3 sub, 3 for r^2, 2 for 1/r^3, 3 accumulate), one MUFU.RSQ.
// The self pair contributes exactly 0 (d = 0, r^2 = kPairSelfEps).
template <int KI>
__device__ __forceinline__ void coul_tile_sweep(const float4 *__restrict__ s_a,
                                                const float2 *__restrict__ s_b, int JP,
                                                const float2 (&xi)[KI], const float2 (&yi)[KI],
                                                const float2 (&zi)[KI], float2 (&ax)[KI],
                                                float2 (&ay)[KI], float2 (&az)[KI])
{
    const float2 eps2 = make_float2(kPairSelfEps, kPairSelfEps);
#pragma unroll 2
    for (int m = 0; m < JP; ++m) {
        const float4 a = s_a[m];
        const float2 nz = s_b[m];
        const float2 nx = make_float2(a.x, a.y), ny = make_float2(a.z, a.w);
#pragma unroll
        for (int k = 0; k < KI; ++k) {
            const float2 dx = __fadd2_rn(xi[k], nx);
            const float2 dy = __fadd2_rn(yi[k], ny);
            const float2 dz = __fadd2_rn(zi[k], nz);
            float2 r2 = __ffma2_rn(dz, dz, eps2);
            r2 = __ffma2_rn(dy, dy, r2);
            r2 = __ffma2_rn(dx, dx, r2);
            const float2 ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
            const float2 f = __fmul2_rn(__fmul2_rn(ri, ri), ri);
            ax[k] = __ffma2_rn(f, dx, ax[k]);
            ay[k] = __ffma2_rn(f, dy, ay[k]);
            az[k] = __ffma2_rn(f, dz, az[k]);
        }
    }
}

// Axis-aligned box of points: lo = +inf, hi = -inf when empty.
struct Box3 {
    float lx, ly, lz, hx, hy, hz;
};

__device__ __forceinline__ Box3 box_empty()
{
    return Box3{INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
}

__device__ __forceinline__ void box_add(Box3 &b, float x, float y, float z)
{
    b.lx = fminf(b.lx, x);
    b.ly = fminf(b.ly, y);
    b.lz = fminf(b.lz, z);
    b.hx = fmaxf(b.hx, x);
    b.hy = fmaxf(b.hy, y);
    b.hz = fmaxf(b.hz, z);
}

// Box of the points of the whole warp, in every lane.
__device__ __forceinline__ Box3 box_warp_reduce(Box3 b)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        b.lx = fminf(b.lx, __shfl_xor_sync(0xffffffffu, b.lx, o));
        b.ly = fminf(b.ly, __shfl_xor_sync(0xffffffffu, b.ly, o));
        b.lz = fminf(b.lz, __shfl_xor_sync(0xffffffffu, b.lz, o));
        b.hx = fmaxf(b.hx, __shfl_xor_sync(0xffffffffu, b.hx, o));
        b.hy = fmaxf(b.hy, __shfl_xor_sync(0xffffffffu, b.hy, o));
        b.hz = fmaxf(b.hz, __shfl_xor_sync(0xffffffffu, b.hz, o));
    }
    return b;
}

// Squared distance between two boxes (0 if they overlap; +inf if one is empty).
__device__ __forceinline__ float box_gap2(const Box3 &a, const Box3 &b)
{
    if (a.lx > a.hx || b.lx > b.hx)
        return INFINITY;
    const float gx = fmaxf(0.0f, fmaxf(b.lx - a.hx, a.lx - b.hx));
    const float gy = fmaxf(0.0f, fmaxf(b.ly - a.hy, a.ly - b.hy));
    const float gz = fmaxf(0.0f, fmaxf(b.lz - a.hz, a.lz - b.hz));
    return gx * gx + gy * gy + gz * gz;
}

// 16-byte asynchronous copy global -> shared (cp.async, L2 only), and its
// completion by the issuing thread.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}

__device__ __forceinline__ void cp_async_wait_own()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Shared memory of ljc_row_segment: two staged j-tiles (negated coordinates,
// two partners per entry, and the box of each 64-partner segment) -- one
// swept while the next is filled -- and the raw partner records of the next
// tile as gathered by cp.async.
template <int JT>
struct LjcSmem {
    float4 raw[JT];      // (x, y, z, q) of the next tile's partners, grouped order
    float4 a[2][JT / 2]; // (-x0, -x1, -y0, -y1)
    float2 b[2][JT / 2]; // (-z0, -z1)
    Box3 seg[2][JT / 64];
};

// Staging of entry m (partners 2m, 2m + 1) of a j-tile from its raw records:
// negated, paired coordinates and, by a warp reduction (whole warps stage), the
// box of the warp's 64 partners.  vmask bit k: partner 2m + k is a particle
// (not padding).
template <int JT>
__device__ __forceinline__ void ljc_stage_entry(LjcSmem<JT> &sm, int buf, int m, float4 a,
                                                float4 b, int vmask)
{
    sm.a[buf][m] = make_float4(-a.x, -b.x, -a.y, -b.y);
    sm.b[buf][m] = make_float2(-a.z, -b.z);
    Box3 pb = box_empty();
    if (vmask & 1)
        box_add(pb, a.x, a.y, a.z);
    if (vmask & 2)
        box_add(pb, b.x, b.y, b.z);
    pb = box_warp_reduce(pb); // the 32 entries m of this warp = one segment
    if ((threadIdx.x & 31) == 0)
        sm.seg[buf][m >> 5] = pb;
}

// Row tile r (rows r*ITILE .. of a grouped order occupying positions [gbase,
// gbase + glen) of perm / tblk) against its j-tiles jt0 .. jt1-1 of the same
// order; writes the row partials, as compensated (hi, lo) pairs, to slot
// [6][ITILE].  For every (warp, 64-partner segment) pair the LJ term is
// evaluated only when the box of the warp's rows and the box of the segment
// come within sqrt(rc2_lim); elsewhere the Coulomb-only sweep runs (the charge
// product applied once per tile), or nothing when has_coul is 0.  s_tab: the
// 8 x 8 type-pair table (sigma^2, 24 eps, rc^2, C q q) in shared memory.
//
// Staging is software-pipelined: while tile jt is swept, the first JT/2
// threads have the partner records of tile jt + 1 in flight (cp.async into
// sm.raw, the partner indices read one tile earlier still) and turn them into
// the other staged buffer after the sweep, so one barrier per tile remains and
// the gather's latency hides behind the sweep.
template <int BLOCK, int KI, int JT>
__device__ __forceinline__ void ljc_row_segment(const float4 *__restrict__ xq,
                                                const int *__restrict__ perm,
                                                const int *__restrict__ tblk, int gbase,
                                                int glen, const float4 *__restrict__ s_tab,
                                                float rc2_lim, int has_coul, int r, int jt0,
                                                int jt1, LjcSmem<JT> &sm, float *__restrict__ slot)
{
    constexpr int ITILE = BLOCK * KI;
    constexpr int JP = JT / 2;
    constexpr int NSEG = JT / 64;
    static_assert(JP <= BLOCK && JP % 32 == 0, "one staged entry per thread of whole warps");
    float2 xi[KI], yi[KI], zi[KI];
    int trow[KI];
    float hx[KI], hy[KI], hz[KI], lx[KI], ly[KI], lz[KI];
    Box3 wb = box_empty();
#pragma unroll
    for (int k = 0; k < KI; ++k) {
        const int lpos = r * ITILE + k * BLOCK + threadIdx.x;
        const bool in = lpos < glen;
        const int i = in ? perm[gbase + lpos] : -1;
        float4 q = make_float4(kPairPad, kPairPad, kPairPad, 0.0f);
        if (i >= 0) {
            q = xq[i];
            box_add(wb, q.x, q.y, q.z);
        }
        xi[k] = make_float2(q.x, q.x);
        yi[k] = make_float2(q.y, q.y);
        zi[k] = make_float2(q.z, q.z);
        trow[k] = (in ? tblk[(gbase + lpos) >> 8] : 0) * NPSIM_MAX_TYPES;
        hx[k] = hy[k] = hz[k] = lx[k] = ly[k] = lz[k] = 0.0f;
    }
    wb = box_warp_reduce(wb); // the box of this warp's rows

    const bool stager = threadIdx.x < JP;
    const int m = threadIdx.x;
    const float4 pad = make_float4(-kPairPad, -kPairPad, -kPairPad, 0.0f);
    int pn0 = -1, pn1 = -1; // partner indices of the tile after the one staged next
    if (stager) {           // tile jt0 staged synchronously (glen is a multiple of JT)
        const int k0 = gbase + jt0 * JT + 2 * m;
        const int j0 = perm[k0], j1 = perm[k0 + 1];
        if (jt0 + 1 < jt1) {
            pn0 = perm[k0 + JT];
            pn1 = perm[k0 + JT + 1];
        }
        ljc_stage_entry<JT>(sm, 0, m, j0 >= 0 ? xq[j0] : pad, j1 >= 0 ? xq[j1] : pad,
                            (j0 >= 0) | ((j1 >= 0) << 1));
    }
    __syncthreads();

    for (int jt = jt0; jt < jt1; ++jt) {
        const int cur = (jt - jt0) & 1;
        const bool next = jt + 1 < jt1; // uniform over the block
        int vmask = 0;
        if (stager && next) { // gather tile jt + 1 while this one is swept
            vmask = (pn0 >= 0) | ((pn1 >= 0) << 1);
            if (pn0 >= 0)
                cp_async16(&sm.raw[2 * m], xq + pn0);
            else
                sm.raw[2 * m] = pad;
            if (pn1 >= 0)
                cp_async16(&sm.raw[2 * m + 1], xq + pn1);
            else
                sm.raw[2 * m + 1] = pad;
            cp_async_commit();
            if (jt + 2 < jt1) {
                const int k2 = gbase + (jt + 2) * JT + 2 * m;
                pn0 = perm[k2];
                pn1 = perm[k2 + 1];
            }
        }

        const int tt = tblk[(gbase + jt * JT) >> 8]; // one type per tile
        float4 cst[KI];
        float2 ax[KI], ay[KI], az[KI], cx[KI], cy[KI], cz[KI];
#pragma unroll
        for (int k = 0; k < KI; ++k) {
            cst[k] = s_tab[trow[k] + tt];
            ax[k] = ay[k] = az[k] = cx[k] = cy[k] = cz[k] = make_float2(0.0f, 0.0f);
        }
        const bool diag = jt * JT < (r + 1) * ITILE && (jt + 1) * JT > r * ITILE;
        for (int sg = 0; sg < NSEG; ++sg) { // warp-uniform choice per segment
            const bool lj = rc2_lim > 0.0f && box_gap2(wb, sm.seg[cur][sg]) <= rc2_lim;
            const float4 *sa = sm.a[cur] + 32 * sg;
            const float2 *sb = sm.b[cur] + 32 * sg;
            if (lj && diag)
                ljc_tile_sweep<KI, true>(sa, sb, 32, xi, yi, zi, cst, ax, ay, az);
            else if (lj)
                ljc_tile_sweep<KI, false>(sa, sb, 32, xi, yi, zi, cst, ax, ay, az);
            else if (has_coul)
                coul_tile_sweep<KI>(sa, sb, 32, xi, yi, zi, cx, cy, cz);
        }
#pragma unroll
        for (int k = 0; k < KI; ++k) {
            const float qq = cst[k].w; // C q_a q_b of the Coulomb-only segments
            two_sum_acc(hx[k], lx[k], fmaf(qq, cx[k].x + cx[k].y, ax[k].x + ax[k].y));
            two_sum_acc(hy[k], ly[k], fmaf(qq, cy[k].x + cy[k].y, ay[k].x + ay[k].y));
            two_sum_acc(hz[k], lz[k], fmaf(qq, cz[k].x + cz[k].y, az[k].x + az[k].y));
        }

        if (stager && next) { // this thread's copies have landed: stage tile jt + 1
            cp_async_wait_own();
            ljc_stage_entry<JT>(sm, cur ^ 1, m, sm.raw[2 * m], sm.raw[2 * m + 1], vmask);
        }
        __syncthreads(); // tile jt + 1 staged; tile jt's buffer free again
    }

#pragma unroll
    for (int k = 0; k < KI; ++k) {
        const int idx = k * BLOCK + threadIdx.x;
        slot[idx] = hx[k];
        slot[ITILE + idx] = hy[k];
        slot[2 * ITILE + idx] = hz[k];
        slot[3 * ITILE + idx] = lx[k];
        slot[4 * ITILE + idx] = ly[k];
        slot[5 * ITILE + idx] = lz[k];
    }
}

// ---------------------------------------------------------------------------
// Each unordered pair once (Newton's third law): the pair force is added to the
// row's sum and, with the other sign, to the partner's.
//
// A warp holds 32 KI rows in registers (KI per lane) and meets 64 partners (32
// staged entries of two) in 32 steps: at step s lane l takes entry (l + s) mod
// 32, so the lanes read 32 consecutive entries of shared memory without bank
// conflicts, and the sum of an entry's partners travels with the entry from
// lane to lane (three float2 shuffles per step, shared by KI rows).  After 32
// steps every row has met every partner, each entry's sums are complete over
// the warp's rows and back in lane (entry).  Per unordered pair 14 packed lanes
// (3 sub, 3 for r^2, 2 for 1/r^3, 3 + 3 accumulate) where the one-sided sweep
// spends 2 x 11.  Measured on one full chip of warps (synthetic tiles, 1e10
// ordered pairs): one-sided 3.43 ms; each pair once 2.53 ms with KI = 4 (96-128
// registers), 2.29 with KI = 8 (168 registers, 12 warps per SM, steps unrolled
// eight times), 2.22 with the shuffles left out: the FP32 pipe is the bound
// (76-79 % of its lanes issue in every one of these forms), and the more rows
// share a step's shuffles and shared-memory reads the nearer it is.  The sums of
// two rows or two partners per register pair, folded before the shuffle (three
// shuffles for six), measured no better (2.38).

// One rotation of an entry's sums: lane l takes lane l + 1's.
__device__ __forceinline__ void sym_rotate(float2 &g, int src)
{
    g.x = __shfl_sync(0xffffffffu, g.x, src);
    g.y = __shfl_sync(0xffffffffu, g.y, src);
}

// Steps after which a lane starts an entry's sums anew (FOLD): at most 128 rows' terms
// in one float32 chain, as many as the one-sided kernels add in each half of a pair of a
// 256-partner tile.  One chain over the 256 rows of KI = 8 rounds more than that: LJ +
// Coulomb, 16384 charges, rms error against float64 6.0e-8, of the last third of the NPs
// 7.3e-8; folded 4.4e-8 and 4.8e-8.  The fold costs 0.8 % of an LJ + Coulomb launch
// (60000 NPs, 0.989 -> 0.997 ms) and 2.9 % of a Coulomb one (100000: 2.345 -> 2.414),
// which goes without: autotune() leaves KI = 8 to lengths at which 512-partner tiles, no
// better than one chain of 256, were the best one-sided choice.
template <int KI, bool FOLD>
constexpr int kSymFoldSteps = FOLD && KI * 32 > 128 ? 128 / KI : 32;

// The sums of an entry over one run of steps join those of the runs before, which are
// still at the lane that held the entry when the run began.
template <int STEPS>
__device__ __forceinline__ void sym_fold(float2 &h, const float2 &g, int lane)
{
    if (STEPS == 32) {
        h = g;
    } else {
        const int src = (lane + STEPS) & 31;
        h.x = __shfl_sync(0xffffffffu, h.x, src) + g.x;
        h.y = __shfl_sync(0xffffffffu, h.y, src) + g.y;
    }
}

// Coulomb-only: ax += d / r^3 for the rows, g = sum of d / r^3 for the partners (the
// caller applies the charges and the partners' sign).
template <int KI, bool FOLD>
__device__ __forceinline__ void coul_sym_sweep(const float4 *__restrict__ s_a,
                                               const float2 *__restrict__ s_b, int lane,
                                               const float2 (&xi)[KI], const float2 (&yi)[KI],
                                               const float2 (&zi)[KI], float2 (&ax)[KI],
                                               float2 (&ay)[KI], float2 (&az)[KI], float2 &hx,
                                               float2 &hy, float2 &hz)
{
    const float2 eps2 = make_float2(kPairSelfEps, kPairSelfEps);
    constexpr int STEPS = kSymFoldSteps<KI, FOLD>;
    constexpr int UNROLL = KI == 4 && !FOLD ? 16 : 8; // 13824 NPs 0.065, with 16 0.064 ms
    const int src = (lane + 1) & 31;
    hx = hy = hz = make_float2(0.0f, 0.0f);
#pragma unroll 1
    for (int s0 = 0; s0 < 32; s0 += STEPS) {
        float2 gx = make_float2(0.0f, 0.0f), gy = gx, gz = gx;
#pragma unroll UNROLL
        for (int s = s0; s < s0 + STEPS; ++s) {
            const int m = (lane + s) & 31;
            const float4 a = s_a[m];
            const float2 nz = s_b[m];
            const float2 nx = make_float2(a.x, a.y), ny = make_float2(a.z, a.w);
#pragma unroll
            for (int k = 0; k < KI; ++k) {
                const float2 dx = __fadd2_rn(xi[k], nx);
                const float2 dy = __fadd2_rn(yi[k], ny);
                const float2 dz = __fadd2_rn(zi[k], nz);
                float2 r2 = __ffma2_rn(dz, dz, eps2);
                r2 = __ffma2_rn(dy, dy, r2);
                r2 = __ffma2_rn(dx, dx, r2);
                const float2 ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
                const float2 f = __fmul2_rn(__fmul2_rn(ri, ri), ri);
                ax[k] = __ffma2_rn(f, dx, ax[k]);
                ay[k] = __ffma2_rn(f, dy, ay[k]);
                az[k] = __ffma2_rn(f, dz, az[k]);
                gx = __ffma2_rn(f, dx, gx);
                gy = __ffma2_rn(f, dy, gy);
                gz = __ffma2_rn(f, dz, gz);
            }
            sym_rotate(gx, src);
            sym_rotate(gy, src);
            sym_rotate(gz, src);
        }
        sym_fold<STEPS>(hx, gx, lane);
        sym_fold<STEPS>(hy, gy, lane);
        sym_fold<STEPS>(hz, gz, lane);
    }
}

// LJ + Coulomb with one set of pair constants (a warp's rows have one type and a
// tile's partners another): cst = (sigma_ab^2, 24 eps_ab, rc_ab^2, C q_a q_b),
// as in ljc_tile_sweep without the self pair.
template <int KI>
__device__ __forceinline__ void ljc_sym_sweep(const float4 *__restrict__ s_a,
                                              const float2 *__restrict__ s_b, int lane,
                                              const float2 (&xi)[KI], const float2 (&yi)[KI],
                                              const float2 (&zi)[KI], const float4 cst,
                                              float2 (&ax)[KI], float2 (&ay)[KI],
                                              float2 (&az)[KI], float2 &hx, float2 &hy, float2 &hz)
{
    const float2 eps2 = make_float2(kPairSelfEps, kPairSelfEps);
    const float2 sig2 = make_float2(cst.x, cst.x);
    const float2 e48 = make_float2(2.0f * cst.y, 2.0f * cst.y);
    const float2 em24 = make_float2(-cst.y, -cst.y);
    const float2 cqq = make_float2(cst.w, cst.w);
    constexpr int STEPS = kSymFoldSteps<KI, true>;
    const int src = (lane + 1) & 31;
    hx = hy = hz = make_float2(0.0f, 0.0f);
#pragma unroll 1
    for (int s0 = 0; s0 < 32; s0 += STEPS) {
        float2 gx = make_float2(0.0f, 0.0f), gy = gx, gz = gx;
        for (int s = s0; s < s0 + STEPS; ++s) {
            const int m = (lane + s) & 31;
            const float4 a = s_a[m];
            const float2 nz = s_b[m];
            const float2 nx = make_float2(a.x, a.y), ny = make_float2(a.z, a.w);
#pragma unroll
            for (int k = 0; k < KI; ++k) {
                const float2 dx = __fadd2_rn(xi[k], nx);
                const float2 dy = __fadd2_rn(yi[k], ny);
                const float2 dz = __fadd2_rn(zi[k], nz);
                float2 r2 = __ffma2_rn(dz, dz, eps2);
                r2 = __ffma2_rn(dy, dy, r2);
                r2 = __ffma2_rn(dx, dx, r2);
                const float2 ri = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
                const float2 ri2 = __fmul2_rn(ri, ri);
                const float2 s2 = __fmul2_rn(sig2, ri2);
                const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
                float2 t = __fmul2_rn(s6, __ffma2_rn(e48, s6, em24));
                t.x = r2.x < cst.z ? t.x : 0.0f;
                t.y = r2.y < cst.z ? t.y : 0.0f;
                const float2 f = __fmul2_rn(__ffma2_rn(cqq, ri, t), ri2);
                ax[k] = __ffma2_rn(f, dx, ax[k]);
                ay[k] = __ffma2_rn(f, dy, ay[k]);
                az[k] = __ffma2_rn(f, dz, az[k]);
                gx = __ffma2_rn(f, dx, gx);
                gy = __ffma2_rn(f, dy, gy);
                gz = __ffma2_rn(f, dz, gz);
            }
            sym_rotate(gx, src);
            sym_rotate(gy, src);
            sym_rotate(gz, src);
        }
        sym_fold<STEPS>(hx, gx, lane);
        sym_fold<STEPS>(hy, gy, lane);
        sym_fold<STEPS>(hz, gz, lane);
    }
}

// Shared memory of sym_row_segment: the staged tiles of LjcSmem and the
// partners' sums of one tile per warp (two buffers: one is summed over the warps
// while the next tile fills the other).
template <int BLOCK, int KI>
constexpr int sym_min_ctas()
{
    // 168, 96 (128 with 256 threads or more) or 80 registers per thread
    return KI >= 8 ? 384 / BLOCK : KI >= 4 ? (BLOCK <= 128 ? 640 : 512) / BLOCK : 768 / BLOCK;
}

template <int BLOCK, int KI, int JT>
struct SymSmem {
    LjcSmem<JT> st;
    float2 g[2][3][BLOCK / 32][JT / 2];
    float hl[6][KI * BLOCK]; // the rows' compensated sums (hi x, y, z, lo x, y, z)
};

// Row tile r of the grouped order [gbase, gbase + glen) against its j-tiles
// jt0 .. jt1 - 1 (all at or beyond the row's own diagonal block, jt >= r ITILE /
// JT).  In the diagonal block (columns below (r + 1) ITILE) the tile holds both
// orders of its pairs and is swept one-sided; beyond it each pair is evaluated
// once for both sides.  Writes
//  * the rows' sums over these tiles to row_slot [6][ITILE] as compensated (hi,
//    lo) pairs, one TwoSum per tile, as ljc_row_segment does;
//  * the partners' sums over the ITILE rows of every two-sided tile to
//    col[c * col_ld + position - (r + 1) ITILE], c = x, y, z: one float32 per
//    ITILE rows (a lane adds 32 KI terms, with LJ 128 at a time, then the warps'
//    sums are added pairwise), which the reduction adds compensated.
// A warp's rows are consecutive positions (32 KI divides the groups' 256-block
// padding), so they have one type.  The sums are kept in units of `scale`, the
// charge product when it is not small (the Coulomb-only sweep then needs no
// multiply by it), else 1 with the LJ + Coulomb sweep on every segment.  has_coul 0: no
// Coulomb term; 1: type pairs without a charge product, whose terms are exactly zero, are
// passed over where LJ does not act either; 2: they are swept too (sum_neutral).  With LJ
// false the tables hold no LJ term: no boxes, always the Coulomb sweep.
template <int BLOCK, int KI, int JT, bool LJ>
__device__ __forceinline__ void sym_row_segment(const float4 *__restrict__ xq,
                                                const int *__restrict__ perm,
                                                const int *__restrict__ tblk, int gbase,
                                                int glen, const float4 *__restrict__ s_tab,
                                                int has_coul, int r, int jt0, int jt1,
                                                SymSmem<BLOCK, KI, JT> &smem,
                                                float *__restrict__ row_slot,
                                                float *__restrict__ col, size_t col_ld)
{
    constexpr int ITILE = BLOCK * KI;
    constexpr int JP = JT / 2;
    constexpr int NSEG = JT / 64;
    constexpr int NW = BLOCK / 32;
    constexpr int RT = ITILE / JT;
    static_assert(JP <= BLOCK && JP % 32 == 0 && ITILE % JT == 0 && 256 % (32 * KI) == 0, "shape");
    LjcSmem<JT> &sm = smem.st;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int row0 = r * ITILE + warp * (32 * KI); // the warp's first row
    const bool active = row0 < glen;               // a warp's rows are all in or all out
    const int trow = (active ? tblk[(gbase + row0) >> 8] : 0) * NPSIM_MAX_TYPES;
    float2 xi[KI], yi[KI], zi[KI];
    Box3 wb = box_empty();
#pragma unroll
    for (int k = 0; k < KI; ++k) {
        const int i = active ? perm[gbase + row0 + k * 32 + lane] : -1;
        float4 q = make_float4(kPairPad, kPairPad, kPairPad, 0.0f);
        if (i >= 0) {
            q = xq[i];
            if (LJ)
                box_add(wb, q.x, q.y, q.z);
        }
        xi[k] = make_float2(q.x, q.x);
        yi[k] = make_float2(q.y, q.y);
        zi[k] = make_float2(q.z, q.z);
#pragma unroll
        for (int c = 0; c < 6; ++c)
            smem.hl[c][k * BLOCK + threadIdx.x] = 0.0f;
    }
    if (LJ)
        wb = box_warp_reduce(wb); // the box of this warp's rows

    const bool stager = threadIdx.x < JP;
    const int m = threadIdx.x;
    const float4 pad = make_float4(-kPairPad, -kPairPad, -kPairPad, 0.0f);
    auto stage = [&](int buf, const float4 a, const float4 b, int vmask) {
        if (LJ) {
            ljc_stage_entry<JT>(sm, buf, m, a, b, vmask);
        } else {
            sm.a[buf][m] = make_float4(-a.x, -b.x, -a.y, -b.y);
            sm.b[buf][m] = make_float2(-a.z, -b.z);
        }
    };
    int pn0 = -1, pn1 = -1; // partner indices of the tile after the one staged next
    if (stager) {           // tile jt0 staged synchronously (glen is a multiple of JT)
        const int k0 = gbase + jt0 * JT + 2 * m;
        const int j0 = perm[k0], j1 = perm[k0 + 1];
        if (jt0 + 1 < jt1) {
            pn0 = perm[k0 + JT];
            pn1 = perm[k0 + JT + 1];
        }
        stage(0, j0 >= 0 ? xq[j0] : pad, j1 >= 0 ? xq[j1] : pad, (j0 >= 0) | ((j1 >= 0) << 1));
    }
    __syncthreads();

    for (int jt = jt0; jt < jt1; ++jt) {
        const int cur = (jt - jt0) & 1;
        const bool next = jt + 1 < jt1; // uniform over the block
        int vmask = 0;
        if (stager && next) { // gather tile jt + 1 while this one is swept
            vmask = (pn0 >= 0) | ((pn1 >= 0) << 1);
            if (pn0 >= 0)
                cp_async16(&sm.raw[2 * m], xq + pn0);
            else
                sm.raw[2 * m] = pad;
            if (pn1 >= 0)
                cp_async16(&sm.raw[2 * m + 1], xq + pn1);
            else
                sm.raw[2 * m + 1] = pad;
            cp_async_commit();
            if (jt + 2 < jt1) {
                const int k2 = gbase + (jt + 2) * JT + 2 * m;
                pn0 = perm[k2];
                pn1 = perm[k2 + 1];
            }
        }

        float4 cst = s_tab[trow + tblk[(gbase + jt * JT) >> 8]]; // one type per tile
        // LJ between this warp's rows and a segment only when their boxes come
        // within the type pair's own cutoff (with a margin for float rounding)
        const float lj2 = LJ && cst.y != 0.0f ? cst.z * 1.0001f : -1.0f;
        float scale = cst.w;
        bool general = false; // LJ + Coulomb sweep on every segment
        if (LJ) {
            const bool unit = fabsf(cst.w) < kSymMinScale;
            general = unit && (cst.w != 0.0f ? has_coul != 0 : has_coul > 1);
            scale = unit ? 1.0f : cst.w;
            cst.y = unit ? cst.y : cst.y / cst.w;
            cst.w = unit ? cst.w : 1.0f;
        }
        float2 ax[KI], ay[KI], az[KI];
#pragma unroll
        for (int k = 0; k < KI; ++k)
            ax[k] = ay[k] = az[k] = make_float2(0.0f, 0.0f);
        const bool two_sided = jt >= (r + 1) * RT; // uniform over the block
        if (two_sided) {
            for (int sg = 0; sg < NSEG; ++sg) { // warp-uniform choice per segment
                const float4 *sa = sm.a[cur] + 32 * sg;
                const float2 *sb = sm.b[cur] + 32 * sg;
                float2 gx = make_float2(0.0f, 0.0f), gy = gx, gz = gx;
                const bool lj = LJ && active &&
                                (general || box_gap2(wb, sm.seg[cur][sg]) <= lj2);
                if (lj)
                    ljc_sym_sweep<KI>(sa, sb, lane, xi, yi, zi, cst, ax, ay, az, gx, gy, gz);
                else if (active && (!LJ || (has_coul && cst.w != 0.0f)))
                    coul_sym_sweep<KI, LJ>(sa, sb, lane, xi, yi, zi, ax, ay, az, gx, gy, gz);
                smem.g[cur][0][warp][32 * sg + lane] = make_float2(-scale * gx.x, -scale * gx.y);
                smem.g[cur][1][warp][32 * sg + lane] = make_float2(-scale * gy.x, -scale * gy.y);
                smem.g[cur][2][warp][32 * sg + lane] = make_float2(-scale * gz.x, -scale * gz.y);
            }
        } else if (active) {
            float4 csts[KI];
#pragma unroll
            for (int k = 0; k < KI; ++k)
                csts[k] = cst;
            for (int sg = 0; sg < NSEG; ++sg) {
                const float4 *sa = sm.a[cur] + 32 * sg;
                const float2 *sb = sm.b[cur] + 32 * sg;
                if (LJ && (general || box_gap2(wb, sm.seg[cur][sg]) <= lj2))
                    ljc_tile_sweep<KI, true>(sa, sb, 32, xi, yi, zi, csts, ax, ay, az);
                else if (!LJ || (has_coul && cst.w != 0.0f))
                    coul_tile_sweep<KI>(sa, sb, 32, xi, yi, zi, ax, ay, az);
            }
        }
#pragma unroll
        for (int k = 0; k < KI; ++k) {
            const int e = k * BLOCK + threadIdx.x; // this thread's own words
            two_sum_acc(smem.hl[0][e], smem.hl[3][e], scale * (ax[k].x + ax[k].y));
            two_sum_acc(smem.hl[1][e], smem.hl[4][e], scale * (ay[k].x + ay[k].y));
            two_sum_acc(smem.hl[2][e], smem.hl[5][e], scale * (az[k].x + az[k].y));
        }

        if (stager && next) { // this thread's copies have landed: stage tile jt + 1
            cp_async_wait_own();
            stage(cur ^ 1, sm.raw[2 * m], sm.raw[2 * m + 1], vmask);
        }
        // tile jt + 1 staged, tile jt's buffer free again, the warps' partner sums
        // complete (their buffer is filled again after the next tile's barrier)
        __syncthreads();
        if (two_sided && threadIdx.x < JP) {
            float *o = col + (size_t)(jt * JT - (r + 1) * ITILE) + 2 * threadIdx.x;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float2 t[NW];
#pragma unroll
                for (int w = 0; w < NW; ++w)
                    t[w] = smem.g[cur][c][w][threadIdx.x];
#pragma unroll
                for (int h = NW / 2; h > 0; h >>= 1)
#pragma unroll
                    for (int w = 0; w < h; ++w)
                        t[w] = __fadd2_rn(t[w], t[w + h]);
                *reinterpret_cast<float2 *>(o + c * col_ld) = t[0];
            }
        }
    }

#pragma unroll
    for (int k = 0; k < KI; ++k) {
        const int idx = warp * (32 * KI) + k * 32 + lane;
#pragma unroll
        for (int c = 0; c < 6; ++c)
            row_slot[c * ITILE + idx] = smem.hl[c][k * BLOCK + threadIdx.x];
    }
}

// ---------------------------------------------------------------------------
// Per-type coefficients used by the integrator (computed on the host in
// float64 from npsim_type_t and the scenario).
struct TypeCoef {
    double mass, inv_mass, half_sigma, k_wall;
    double c1, sd_o;    // BAOAB O step: v <- c1 v + sd_o xi
    double mob, sd_bd;  // overdamped: x += F dt mob + sd_bd xi
    double charge_c;    // C * q (Coulomb-only all-pairs kernel returns the field)
    // float32 copies used by the integrator (all of its arithmetic is float32 or
    // compensated float32): dt/(2m), c1 as hi + lo (its rounding error would
    // otherwise compound over the 1/(gamma dt) steps a velocity remembers),
    // sd_o, dt*mob, sd_bd, C q, m g, m w^2, k_wall, sigma/2; for the printed
    // step (vi) dt/m, gamma dt and the kick magnitude
    float hdt_m, c1f, c1lo, sd_of, dt_mob, sd_bdf, qc, mg, mw2, kw, hs;
    float dt_m, gdt, kick;
};

// ---------------------------------------------------------------------------
// Compensated float32 ("double-float") arithmetic: a value is an unevaluated
// sum hi + lo of two floats with |lo| <= ulp(hi)/2, about 48 significant bits.
// Every operation is rounded separately (no fused multiply-add contraction).

// Knuth's TwoSum: s + e == a + b exactly.
__device__ __forceinline__ float2 df_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
    return make_float2(s, e);
}

// Dekker's Fast2Sum (|a| >= |b| or a == 0): s + e == a + b exactly.
__device__ __forceinline__ float2 df_fast_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}

// (h, l) += b, renormalised.
__device__ __forceinline__ void df_add(float &h, float &l, float b)
{
    const float2 t = df_two_sum(h, b);
    const float2 u = df_fast_two_sum(t.x, __fadd_rn(t.y, l));
    h = u.x;
    l = u.y;
}

// (h, l) += (bh, bl), renormalised.
__device__ __forceinline__ void df_add_df(float &h, float &l, float bh, float bl)
{
    const float2 t = df_two_sum(h, bh);
    const float2 u = df_fast_two_sum(t.x, __fadd_rn(__fadd_rn(t.y, l), bl));
    h = u.x;
    l = u.y;
}

// (h, l) *= b (float), renormalised; the product of h and b is exact via FMA.
__device__ __forceinline__ void df_mul(float &h, float &l, float b)
{
    const float p = __fmul_rn(h, b);
    const float e = __fmaf_rn(h, b, -p);
    const float2 u = df_fast_two_sum(p, __fmaf_rn(l, b, e));
    h = u.x;
    l = u.y;
}

// Equilibrium radius of the interface spring for a particle of half-diameter
// hs at t = step dt: R_eff = R(t) - hs with R(t)^2 = R0^2 - k t (radius-square
// law, 0 once the droplet has gone).  Returned as (R_eff^2 hi, R_eff^2 lo,
// R_eff, 2 hs = the width of the band (-r, r) about the surface) from one
// float64 evaluation.  Host and device both call this (the
// explicit fma fixes the rounding), so a table set by the host equals the one
// the integrator writes for the same step bit for bit.
__host__ __device__ inline float4 spring_entry(double R0, double k_evap, double dt,
                                               long long step, double hs)
{
    const double t = (double)step * dt;
    const double R2 = fma(-k_evap, t, R0 * R0);
    const double R = R2 > 0.0 ? sqrt(R2) : 0.0;
    const double re = R - hs;
    const double re2 = re * re;
    const float h = (float)re2;
    return make_float4(h, (float)(re2 - (double)h), (float)re, (float)(2.0 * hs));
}

// External forces (interface spring, gravity, centrifugal) on a particle at
// x = xh + xl (float hi / lo words).  The spring needs s = |x| - R_eff, the
// difference of two nearly equal numbers; it is formed as
// (|x|^2 - R_eff^2) / (|x| + R_eff) with |x|^2 from exact products and sums
// (the lo^2 terms lie below the precision kept), so s keeps float32 relative
// precision however large |x| is.  wall = 2 limits the spring to the band
// (-r, r) about the surface, 0 < s < 2 r (spring.w = 2 r).
//
// With flags given, the failure check of the interface (no counterpart in the
// paper, whose runs rely on strong damping for stability) runs on the NPs near
// or beyond the surface: with the full spring on (wall 1) no NP gets farther
// than twice the larger of R0 and R(t) from the centre unless a step went
// unstable (twice R(t) alone is not a bound: under a fast compression a heavy
// NP can lag the moving interface by more than R(t) itself); R(t) = R_eff +
// sigma/2 from the spring entry.  Sets FLAG_ESCAPED.
__device__ __forceinline__ void external_force(const float4 &xh, float lx, float ly, float lz,
                                               float kw, float mg, float mw2, float4 spring,
                                               int wall, int rot_mode, float &fx,
                                               float &fy, float &fz, float R0 = 0.0f,
                                               int *flags = nullptr)
{
    fx = fy = fz = 0.0f;
    // the spring acts only beyond R_eff (s > 0): an NP whose float32 |x|^2 from
    // the hi words lies below (R_eff - 0.01)^2 is certainly inside (the lo words
    // and the rounding of that sum move |x| by far less than 0.01), so the
    // exact distance is formed only near the surface
    const float reff_in = spring.z - 0.01f;
    const float r2_cheap = __fmaf_rn(xh.x, xh.x, __fmaf_rn(xh.y, xh.y, __fmul_rn(xh.z, xh.z)));
    if (wall && !(reff_in > 0.0f && r2_cheap < reff_in * reff_in)) {
        if (flags && wall == 1) {
            const float R = fmaxf(__fmaf_rn(0.5f, spring.w, spring.z), R0);
            if (r2_cheap > __fmul_rn(4.0f, __fmul_rn(R, R)))
                atomicOr(flags, FLAG_ESCAPED);
        }
        float r2h = 0.0f, r2l = 0.0f;
        const float hh[3] = {xh.x, xh.y, xh.z}, ll[3] = {lx, ly, lz};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const float p = __fmul_rn(hh[d], hh[d]);
            const float e = __fmaf_rn(hh[d], hh[d], -p);
            df_add_df(r2h, r2l, p, __fmaf_rn(2.0f * hh[d], ll[d], e));
        }
        // |x| and 1/|x| from one rsqrt (a few ulp: far below the force tolerance);
        // every operation below is rounded explicitly, so the force does not
        // depend on how the compiler fuses operations in each kernel that
        // inlines this (the integrator's modes must agree bit for bit)
        const float rinv = rsqrtf(r2h);
        const float reff = spring.z;
        float s;
        if (reff > 0.0f) {
            float dh = r2h, dl = r2l;
            df_add_df(dh, dl, -spring.x, -spring.y);
            s = __fdividef(dh, __fmaf_rn(r2h, rinv, reff)); // (|x|^2 - R_eff^2) / (|x| + R_eff)
        } else {
            s = __fmaf_rn(r2h, rinv, -reff);
        }
        if (s > 0.0f && r2h > 0.0f && (wall != 2 || s < spring.w)) {
            const float f = __fmul_rn(__fmul_rn(-kw, s), rinv);
            fx = __fmul_rn(f, xh.x);
            fy = __fmul_rn(f, xh.y);
            fz = __fmul_rn(f, xh.z);
        }
    }
    fz = __fsub_rn(fz, mg);
    if (rot_mode == 1) {
        fx = __fmaf_rn(mw2, xh.x, fx);
        fy = __fmaf_rn(mw2, xh.y, fy);
    } else if (rot_mode == 2) {
        fx = __fmaf_rn(mw2, xh.x, fx);
        fy = __fmaf_rn(mw2, xh.y, fy);
        fz = __fmaf_rn(mw2, xh.z, fz);
    }
}

struct StepParams {
    int n;
    int n_types;
    int rot_mode;
    int wall;
    int integrator;
    int pad_;
    uint64_t seed;
    double dt, R0, k_evap, g, omega2;
    TypeCoef tc[NPSIM_MAX_TYPES];
};

// Stream-K decomposition of the all-pairs sum: W = n_it * n_jt work units
// (i-tile x j-tile) split evenly into `grid` ranges; range c covers units
// [W c / grid, W (c+1) / grid).  The part of i-tile row r computed in range c
// is written to partial slot r + c (unique: rows and ranges both advance
// along the unit order).  A static launch runs range c on CTA c; a dynamic
// launch (the grouped kernels) starts `ctas` CTAs on ranges 0 .. ctas - 1 and
// hands out the rest from a device counter, so a CTA that runs ahead of the
// others on its SM takes more ranges.  Slots depend only on the range, so the
// sums do not depend on which CTA ran which range.
struct StreamK {
    int itile;   // i per CTA tile = block * ki
    int jtile;   // j per shared-memory tile
    int n_it;    // number of i tiles
    int n_jt;    // number of j tiles
    int grid;    // ranges (= CTAs of a static launch)
    int ctas;    // CTAs of a dynamic launch (<= grid; 0 for static launches)
    long long W; // n_it * n_jt
    // tri > 0: the triangular form of the kernels that evaluate each pair once
    // (allpairs_sym.cu): row r has the j-tiles tri r .. n_jt - 1 only (tri =
    // itile / jtile), len = positions covered (a multiple of jtile)
    int tri;
    int len;
};

// First unit of row r of the triangular form (row r has n_jt - tri r units).
__host__ __device__ __forceinline__ long long tri_row_begin(const StreamK &s, int r)
{
    return (long long)r * s.n_jt - (long long)s.tri * r * (r - 1) / 2;
}

// Row of unit p of the triangular form: the root of the quadratic, then exact.
__device__ __forceinline__ int tri_row_of(const StreamK &s, long long p)
{
    const float b = (float)s.n_jt + 0.5f * (float)s.tri;
    const float disc = fmaxf(b * b - 2.0f * (float)s.tri * (float)p, 0.0f);
    int r = min(max((int)((b - sqrtf(disc)) / (float)s.tri), 0), s.n_it - 1);
    while (r + 1 < s.n_it && tri_row_begin(s, r + 1) <= p)
        ++r;
    while (r > 0 && tri_row_begin(s, r) > p)
        --r;
    return r;
}

// Floats before row r's column partials (see sym_row_segment): rows k < r hold
// 3 planes of len - (k + 1) itile floats each.
__host__ __device__ __forceinline__ size_t sym_col_offset(int len, int itile, int r)
{
    return 3 * ((size_t)r * (size_t)len - (size_t)itile * ((size_t)r * ((size_t)r + 1) / 2));
}

// Floats of all column partials of a grouped order of `len` positions.
__host__ __device__ __forceinline__ size_t sym_col_floats(int len, int itile)
{
    const int rows = len / itile; // rows k with len - (k + 1) itile > 0 (the last may be 0)
    return rows > 0 ? sym_col_offset(len, itile, rows) : 0;
}

__host__ __device__ __forceinline__ long long sk_begin(const StreamK &s, int c)
{
    return s.W * (long long)c / s.grid;
}

// First CTA whose range contains unit p.
__host__ __device__ __forceinline__ int sk_cta_of(const StreamK &s, long long p)
{
    int c = (int)(p * s.grid / s.W);
    while (c + 1 < s.grid && sk_begin(s, c + 1) <= p)
        ++c;
    while (c > 0 && sk_begin(s, c) > p)
        --c;
    return c;
}

// ---------------------------------------------------------------------------
// Sum of a position's partials of the kernels that evaluate each pair once
// (sym_row_segment): its row's n_rows slots [6][itile] from row_slots on, then
// the column partials of the first n_cols row tiles (those before its own, r' =
// 0 .. r - 1; none in a one-sided sum).  Four
// threads share a position (64 positions per CTA of 256 threads, so the reads
// are coalesced and a long column has four times the loads in flight): thread
// `part` takes every fourth slot, compensated; sym_finish adds the four in a
// fixed order.
__device__ __forceinline__ void sym_sum_partials(const float *__restrict__ row_slots, int n_rows,
                                                 const float *__restrict__ cols, int itile,
                                                 int len, int r, int n_cols, int p, int part,
                                                 float (&h)[3], float (&l)[3])
{
    const float *rs = row_slots + (p - r * itile);
    for (int c = part; c < n_rows; c += 4) {
        const float *q = rs + (size_t)c * 6 * itile;
#pragma unroll
        for (int d = 0; d < 3; ++d)
            df_add_df(h[d], l[d], __ldcs(q + d * itile), __ldcs(q + (3 + d) * itile));
    }
    int k = part;
    for (; k + 4 < n_cols; k += 8) { // two row tiles' loads before their adds
        const float *q0 = cols + sym_col_offset(len, itile, k) + (p - (k + 1) * itile);
        const float *q1 = cols + sym_col_offset(len, itile, k + 4) + (p - (k + 5) * itile);
        const size_t l0 = (size_t)(len - (k + 1) * itile), l1 = (size_t)(len - (k + 5) * itile);
        float w[6];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            w[d] = __ldcs(q0 + d * l0);
            w[3 + d] = __ldcs(q1 + d * l1);
        }
#pragma unroll
        for (int d = 0; d < 3; ++d)
            df_add(h[d], l[d], w[d]);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            df_add(h[d], l[d], w[3 + d]);
    }
    for (; k < n_cols; k += 4) {
        const float *q = cols + sym_col_offset(len, itile, k) + (p - (k + 1) * itile);
        const size_t ld = (size_t)(len - (k + 1) * itile);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            df_add(h[d], l[d], __ldcs(q + d * ld));
    }
}

// Parts 1 .. 3 added to part 0 in order; the 32-byte record of particle i
// (hi x, y, z, lo x | lo y, z, 0, 0), none for padding (i < 0).
__device__ __forceinline__ void sym_finish(float (&s_part)[3][6][64], int part, float (&h)[3],
                                           float (&l)[3], int i, float *__restrict__ F_pair)
{
    const int x = threadIdx.x & 63;
    if (part > 0) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            s_part[part - 1][d][x] = h[d];
            s_part[part - 1][3 + d][x] = l[d];
        }
    }
    __syncthreads();
    if (part == 0 && i >= 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
            for (int d = 0; d < 3; ++d)
                df_add_df(h[d], l[d], s_part[q][d][x], s_part[q][3 + d][x]);
        float4 *o = reinterpret_cast<float4 *>(F_pair + 8 * (size_t)i);
        o[0] = make_float4(h[0], h[1], h[2], l[0]);
        o[1] = make_float4(l[1], l[2], 0.0f, 0.0f);
    }
}

// LJ / Coulomb type-pair table entry: (sigma_ab^2, 24 eps_ab, rc_ab^2, C q_a q_b).
// Stored 8 x 8 (row a, column b).
struct PairTab {
    float4 e[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
};

// Cell grid for the LJ cutoff path.
struct CellGrid {
    int dim;        // cells per axis
    int n_cells;    // dim^3
    float inv_h;    // 1 / cell edge
    float L;        // grid covers [-L, L)^3; coordinates outside are clamped
    int tb;         // type blocks of the sort key: key = type * n_cells + cell when
                    // tb > 1 (cell order grouped by type first), key = cell when tb == 1
    // stencil half-width (in cells) per type pair: partners of type b of an NP of
    // type a within its list radius lie within ext[a * 8 + b] cells along each
    // axis (1 when the edge is at least every radius)
    unsigned char ext[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
};

// Record a message for npsim_last_error() on this thread and return `code`
// (defined in capi.cu).
int report_error(int code, const char *fmt, ...);

// One copy into host arrays that lie back to back.  cudaErrorInvalidValue, with the error
// cleared: they are page-locked one by one and no copy may span them; the caller copies
// them one by one.
inline cudaError_t copy_joined(void *host, const void *dev, size_t bytes, cudaStream_t st)
{
    const cudaError_t e = cudaMemcpyAsync(host, dev, bytes, cudaMemcpyDeviceToHost, st);
    if (e == cudaErrorInvalidValue)
        cudaGetLastError();
    return e;
}

// An NVTX range named after the C-ABI entry point it is declared in, for the
// length of the call: the calls show on Nsight Systems timelines above the
// kernels they launch (the NVTX calls do nothing when no tool is attached).
struct TraceRange {
    explicit TraceRange(const char *name) { nvtxRangePushA(name); }
    ~TraceRange() { nvtxRangePop(); }
    TraceRange(const TraceRange &) = delete;
    TraceRange &operator=(const TraceRange &) = delete;
};
#define NP_TRACE() ::npsim::TraceRange np_trace_range_(__func__)

// ---------------------------------------------------------------------------
// Launchers (host functions defined in the .cu files).

struct ApConfig {
    int block, ki, jt, occ;
};

// All-pairs kernels (allpairs.cu)
int ap_num_configs();
ApConfig ap_config(int idx);
int ap_occupancy(int idx, bool lj);
bool ap_packed(int idx); // float32x2 Coulomb-only kernel
// Charge-grouped packed Coulomb kernel (allpairs_grouped.cu): rows and columns
// follow perm (grouped by charge, groups padded to 512), qblk = charge of each
// 256-position block.
int grp_num_configs();
ApConfig grp_config(int idx);
int grp_occupancy(int idx);
// work: two zeroed device counters (ranges handed out, CTAs done), reset to 0
// by the last CTA of each launch; launches sharing one pair must not overlap.
cudaError_t launch_allpairs_grouped(int idx, const StreamK &sk, const float4 *xq,
                                    const int *perm, int n_perm, const float *qblk,
                                    unsigned *work, float *slots, cudaStream_t st);
// Type-grouped packed LJ + Coulomb kernel (allpairs_grouped.cu): rows and
// columns follow perm (grouped by type, groups padded to 512), tblk = type of
// each 256-position block; the table selects LJ + Coulomb, LJ or Coulomb.
int ljg_num_configs();
ApConfig ljg_config(int idx);
int ljg_occupancy(int idx);
// rc2_lim: LJ is evaluated only between tiles whose boxes come within
// sqrt(rc2_lim) (0: no LJ); has_coul = 0 skips the other tiles entirely.
cudaError_t launch_allpairs_ljgrp(int idx, const StreamK &sk, const float4 *xq,
                                  const int *perm, int n_perm, const int *tblk,
                                  const PairTab *tab, float rc2_lim, int has_coul,
                                  unsigned *work, float *slots, cudaStream_t st);
// Each pair once (allpairs_sym.cu): the type-grouped order, triangular StreamK,
// row and column partials in one array (sym_slots_floats floats), summed into
// one 32-byte record per NP by launch_sym_reduce (F_pair [n][8]: hi x, y, z, lo
// x, y, z, 0, 0).  Configurations [0, sym_num_configs(false)) sum Coulomb only,
// those of lj = true LJ + Coulomb as the table says.
int sym_num_configs(bool lj);
ApConfig sym_config(bool lj, int idx);
int sym_occupancy(bool lj, int idx);
size_t sym_slots_floats(const StreamK &sk);
cudaError_t launch_allpairs_sym(bool lj, int idx, const StreamK &sk, const float4 *xq,
                                const int *perm, const int *tblk, const PairTab *tab,
                                int has_coul, unsigned *work, float *slots, cudaStream_t st);
cudaError_t launch_sym_reduce(const StreamK &sk, const float *slots, const int *perm,
                              float *F_pair, cudaStream_t st);
cudaError_t launch_allpairs(int cfg_idx, bool lj, const StreamK &sk, const float4 *xq,
                            const int *typ, int n, const PairTab *tab, float *slots,
                            cudaStream_t st);

// Integrator (integrate.cu)
enum IntMode : int {
    MODE_FORCES = 0, // assemble F from partials + external, write F
    MODE_A = 1,      // BAOA (or overdamped update) from the stored F; step += 1
    MODE_BA = 2,     // assemble F, finish the step (B), then BAOA of the next; step += 1
    MODE_B = 3,      // assemble F, finish the step (B), write F and v
};

// State of the integrator: position = xq.xyz (float32, the word the pair kernels
// read) + x_lo (float32 SoA [3][n]); velocity float32 SoA [3][n]; force as
// float32 hi/lo SoA [6][n] (hi x, y, z, then lo x, y, z).  Stream-K partial
// slots use the same hi/lo split; the cell-list LJ forces are one 32-byte
// (hi x, y, z, lo x, y, z, 0, 0) record per NP, indexed by particle.
struct IntArgs {
    float *x_lo, *v, *F;     // see above
    const int *typ;
    float4 *xq;              // (x hi, y hi, z hi, q)
    const float *slots;      // stream-K partials [slot][6][itile] (or NULL)
    StreamK sk;
    const float *F_lj;       // cell-list LJ forces [n][8] (hi x, y, z, lo x, y, z, 0, 0) (or NULL)
    const float *F_pair;     // summed all-pairs forces [n][8] of the kernels that
                             // evaluate each pair once (or NULL): in place of slots
    const int *row_pos;      // grouped layout: position of particle i in the rows (-1:
                             // no Coulomb partial); NULL: row position = i
    const float4 *x_ref;     // positions at the last neighbour-list build (or NULL)
    float4 *sxq;             // cell-ordered current positions of the neighbour-list
    const int *cell_pos;     // kernel, and the slot of NP i (both NULL without one)
    int *nbr_gate;           // set to 1 when an NP has moved more than half the skin
    float half_skin2;        // (skin / 2)^2, with margin
    float4 *spring;          // spring radius per type (spring_entry), two buffers
                             // [2][NPSIM_MAX_TYPES]: buffer (step & 1) holds the
                             // current step's; modes that advance the step write
                             // the other one for step + 1
    int ext_on;              // add external forces
    int field_slots;         // slots hold sum_j q_j r_ij/r^3 (Coulomb-only kernel): scale by C q_i
    long long *step;         // device step counter: the first step of the current chunk
    int step_ofs;            // this launch's step = *step + step_ofs
    int step_commit;         // last launch of a chunk: set *step to this launch's step
                             // (+ 1 in the modes that take the A part) once every CTA
                             // has read it
    int *flags;
    unsigned *done;          // CTAs counted in by the committing launch (zero between)
};

// Velocity and position of one particle through the closing half kick B and / or
// the B-A-O-A part of the next step (or the overdamped update, or step (vi) as
// printed), from the force f and the step's normals nz (A part).
template <bool DO_B, bool DO_A>
__device__ __forceinline__ void kick_drift(const TypeCoef &tc, int integrator, float hdt,
                                           const float (&nz)[3], const float (&f)[3],
                                           float (&v)[3], float (&xhi)[3], float (&xlo)[3])
{
    const bool baoab = integrator == 0;
    if (DO_B && baoab) {
#pragma unroll
        for (int d = 0; d < 3; ++d)
            v[d] = __fmaf_rn(tc.hdt_m, f[d], v[d]);
    }
    if (DO_A) {
        if (baoab) {
            // the two A half steps around the O step add dt/2 (v' + v'') to the
            // position (the O step does not depend on x): one compensated add
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                v[d] = __fmaf_rn(tc.hdt_m, f[d], v[d]);               // B
                const float va = v[d];                                // A (first half)
                v[d] = __fmaf_rn(tc.c1f, v[d],
                                 __fmaf_rn(tc.c1lo, v[d], __fmul_rn(tc.sd_of, nz[d]))); // O
                df_add(xhi[d], xlo[d], __fmul_rn(hdt, __fadd_rn(va, v[d]))); // A + A
            }
        } else if (integrator == 1) {
#pragma unroll
            for (int d = 0; d < 3; ++d)
                df_add(xhi[d], xlo[d], __fmaf_rn(f[d], tc.dt_mob, __fmul_rn(tc.sd_bdf, nz[d])));
        } else { // step (vi) as printed: drag and force, a kick of fixed size, drift
            const float nn = sqrtf(__fmaf_rn(nz[0], nz[0], __fmaf_rn(nz[1], nz[1],
                                                                     __fmul_rn(nz[2], nz[2]))));
            const float a = nn > 0.0f ? __fdiv_rn(tc.kick, nn) : 0.0f; // kick / |n|
            const float dt = 2.0f * hdt;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                v[d] = __fmaf_rn(tc.dt_m, f[d], __fmaf_rn(-tc.gdt, v[d], v[d]));
                v[d] = __fmaf_rn(a, nz[d], v[d]);
                df_add(xhi[d], xlo[d], __fmul_rn(dt, v[d]));
            }
        }
    }
}

// One particle's update after its force (Fh + Fl) has been assembled: store F
// (MODE_FORCES, MODE_B), the closing half kick B (MODE_BA, MODE_B) and the
// B-A-O-A part of the next step, or the overdamped update (MODE_A, MODE_BA).
// Arrays are SoA over n particles: x_lo [3][n], v_ [3][n], F [6][n]; xq holds
// the hi words of the position.  Noise is drawn for particle noise_idx.
template <int MODE>
__device__ __forceinline__ void advance_particle(int i, int n, uint32_t noise_idx,
                                                 const TypeCoef &tc, int integrator, float hdt,
                                                 uint64_t seed, long long step, const float4 &xh,
                                                 float lx, float ly, float lz, const float Fh[3],
                                                 const float Fl[3], const float (&v0)[3],
                                                 float *x_lo, float *v_, float *F, float4 *xq,
                                                 int *flags,
                                                 const float4 *x_ref = nullptr,
                                                 int *nbr_gate = nullptr, float half_skin2 = 0.f,
                                                 float4 *sxq = nullptr,
                                                 const int *cell_pos = nullptr, int ti = 0)
{
    constexpr bool DO_B = (MODE == MODE_BA || MODE == MODE_B);
    constexpr bool DO_A = (MODE == MODE_A || MODE == MODE_BA);
    if (MODE == MODE_FORCES || MODE == MODE_B) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            F[d * n + i] = Fh[d];
            F[(3 + d) * n + i] = Fl[d];
        }
    }
    if (MODE == MODE_FORCES)
        return;
    const float f[3] = {__fadd_rn(Fh[0], Fl[0]), __fadd_rn(Fh[1], Fl[1]),
                        __fadd_rn(Fh[2], Fl[2])};
    float v[3] = {v0[0], v0[1], v0[2]}; // v_ at i, read by the caller
    float xhi[3] = {xh.x, xh.y, xh.z}, xlo[3] = {lx, ly, lz};
    float nz[3] = {0.f, 0.f, 0.f};
    if (DO_A)
        normals3(seed, noise_idx, step, 0u, nz[0], nz[1], nz[2]);
    kick_drift<DO_B, DO_A>(tc, integrator, hdt, nz, f, v, xhi, xlo);
    if (DO_A) {
        xq[i] = make_float4(xhi[0], xhi[1], xhi[2], xh.w);
        if (sxq) // the neighbour-list kernel's cell-ordered copy
            sxq[cell_pos[i]] = make_float4(xhi[0], xhi[1], xhi[2], __int_as_float(ti));
        x_lo[i] = xlo[0];
        x_lo[n + i] = xlo[1];
        x_lo[2 * n + i] = xlo[2];
        if (!(isfinite(xhi[0]) && isfinite(xhi[1]) && isfinite(xhi[2])))
            atomicOr(flags, FLAG_NONFINITE);
        if (x_ref) { // moved more than half the skin since the list was built: rebuild
            const float4 r = x_ref[i];
            const float ex = xhi[0] - r.x, ey = xhi[1] - r.y, ez = xhi[2] - r.z;
            if (!(fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= half_skin2))
                *nbr_gate = 1;
        }
    }
    v_[i] = v[0];
    v_[n + i] = v[1];
    v_[2 * n + i] = v[2];
}

// `steps` steps (at most kMaxFreeSteps) of a simulation without pair forces, from the
// device step counter on, in one launch.
constexpr int kMaxFreeSteps = 64;
cudaError_t launch_free_steps(const IntArgs &a, const StepParams &p, int steps, cudaStream_t st);
cudaError_t launch_integrate(int mode, const IntArgs &a, const StepParams &p,
                             cudaStream_t st);
// The integrator's sum of the all-pairs partial slots alone, for positions
// 0 .. n_pos - 1 of the stream-K order, to out (6 n_pos floats: hi x, y, z,
// lo x, y, z planes).
cudaError_t launch_slot_sum(const float *slots, const StreamK &sk, int n_pos, float *out,
                            cudaStream_t st);

// Ensemble of droplets (ensemble.cu).  Each droplet's particles are listed in a
// type-grouped order (groups padded to 256 positions) at positions [gpos0,
// gpos0 + npad) of the ensemble's grouped order.  The all-pairs work is a list of
// items (a row tile of a droplet against up to `chunk` of its consecutive
// j-tiles); the column partials of droplet d (sym_row_segment) start at float
// col0 of theirs, and its row tiles at row0 of row_first.
struct EnsDrop {
    int offset, n, rot_mode, wall, integrator;
    int gpos0, npad;
    float rc2_lim;  // LJ only between tiles within this squared distance (0: no LJ)
    int has_coul;   // 0: tiles out of LJ range add nothing
    int row0;
    long long col0;
    uint64_t seed;
    double dt, R0, k_evap, g, omega2;
    TypeCoef tc[NPSIM_MAX_TYPES];
};

struct EnsItem {
    int drop, row, jt0, jt1; // row tile of the droplet, its j-tiles jt0 .. jt1 - 1
    int slot;                // where the rows' sums go
};

struct EnsAllpairsArgs {
    const float4 *xq;
    const int *perm;        // grouped position -> particle (-1: padding)
    const int *tblk;        // type of each 256-position block
    const int *dblk;        // droplet of each 256-position block
    const EnsDrop *drops;
    const PairTab *tabs;    // one table per droplet
    const EnsItem *items;   // longest first
    const int *row_first;   // first slot of every row tile, slots in row order; one past the end
    int n_items;
    int n_pos;              // grouped length
    int itile;
    int sym;                // kernels that evaluate each pair once (column partials)
    unsigned *work;         // [0] next item, [1] CTAs done (both 0 between launches)
    float *slots;           // one [6][itile] slot per work item, then the column partials
    float *F_pair;          // [n_total][8] (hi x, y, z, lo x, y, z, 0, 0): the summed forces
};

struct EnsIntArgs {
    float *x_lo, *v, *F;     // layouts as in IntArgs, over the concatenation
    const int *typ;
    float4 *xq;
    const int *drop_of;
    const EnsDrop *drops;
    const float *F_pair;     // all-pairs forces [n_total][8], as in IntArgs (or NULL)
    float4 *spring;          // [2][n_drops][NPSIM_MAX_TYPES], as in IntArgs
    int ext_on;
    int pad_;
    long long *step;
    int *flags;
    unsigned *done;
};

int ens_num_configs();
ApConfig ens_config(int idx);
int ens_occupancy(int idx);
bool ens_sym(int idx); // evaluates each pair once
// The all-pairs launch on `ctas` CTAs and the reduction of its partials into
// a.F_pair.
cudaError_t launch_ens_allpairs(int idx, int ctas, const EnsAllpairsArgs &a, cudaStream_t st);
cudaError_t launch_ens_integrate(int mode, const EnsIntArgs &a, int n_total, int n_drops,
                                 cudaStream_t st);

// BF16 tensor-core MLP kernels (mlp.cu).
enum : int {
    GEMM_F32 = 0,  // C (FP32) = A B^T (+ bias)
    GEMM_ACT = 1,  // z = A B^T + bias -> Z (FP32, optional); C (BF16) = SiLU(z) or z
    GEMM_DACT = 2, // C (BF16, and FP32 if Cf) = (A B^T) * SiLU'(Z)
};

struct GemmArgs {
    const __nv_bfloat16 *A; // M x K, row-major, lda
    const __nv_bfloat16 *B; // N x K, row-major, ldb
    int M, N, K, lda, ldb, ldc;
    int n_tile;    // columns per CTA (multiple of 16, <= 256)
    int tmem_cols; // power of two >= max(32, n_tile)
    int mode, act;
    const float *bias;      // N or NULL
    float *Cf;              // FP32 output (M x N, ldc) or NULL
    __nv_bfloat16 *Cb;      // BF16 output or NULL
    float *Z;               // pre-activation (GEMM_ACT writes, GEMM_DACT reads), ldc
    __nv_bfloat16 *CbT;     // transposed copy of Cb (N x M, ldt) or NULL
    int ldt;
    int *flags;             // FLAG_TIMEOUT on a bounded wait that expired
    long long wait_cycles;  // bound of the main loop's waits in SM cycles (0: 2^32)
    // nz products of one shape (networks), product z's operands z za / z zb rows
    // further, its outputs z zc (Cf, Cb, Z), z zt (CbT), z zbias elements further
    int nz, za, zb;
    size_t zc, zt, zbias;
};

struct AdamArgs {
    float lr, b1, b2, eps, wd, bc1, bc2; // bc = 1 - beta^t
};

// The parameters of one network as a flat vector: layer l's weights (out_p x in_p)
// at off[l], its biases right behind; Wb / Wt: the BF16 copy and its transpose of
// all networks, network k at k out_p in_p.
constexpr int kMaxLayers = 9; // 8 hidden and the output layer
struct NetDims {
    int n_layers, n_params;
    int off[kMaxLayers], out_p[kMaxLayers], in_p[kMaxLayers];
    __nv_bfloat16 *Wb[kMaxLayers], *Wt[kMaxLayers];
};

// One product (g1 NULL), or two independent ones of the same nz in one launch.
cudaError_t launch_gemm(const GemmArgs &g0, const GemmArgs *g1, cudaStream_t st);

// Fused inference of a whole MLP (mlp.cu): every layer of every network in one
// launch, activations kept in shared memory, one CTA per (128 rows, network).
// W[l] / b[l]: layer l's BF16 weights (N_l x K_l, K-major) and FP32 biases of
// all networks stacked (network k at rows k N_l); y: [n_nets][bp][out_p].
constexpr int kMaxMlpLayers = 6; // hidden layers the fused kernel takes
struct MlpInferArgs {
    const __nv_bfloat16 *X;                    // bp x in_p
    const __nv_bfloat16 *W[kMaxMlpLayers + 1]; // layer l: n_nets * N_l x K_l
    const float *b[kMaxMlpLayers + 1];         // layer l of network 0; network k at k b_stride
    int b_stride;
    int NL, in_p, H, out_p, bp, n_nets;
    float *y;
    int *flags;
};
bool mlp_infer_supported(int NL, int in_p, int H, int out_p);
cudaError_t launch_mlp_infer(const MlpInferArgs &a, cudaStream_t st);
cudaError_t launch_transpose_bf16(const void *in, int R, int C, int ldi, void *out, int ldo,
                                  cudaStream_t st);
// Mean-squared error and its gradient for nz networks, y and gf / gb / gbT (the
// transposed BF16 gradient, ldy x M) of network z M ldy elements further, loss[z].
cudaError_t launch_mse_grad(const float *y, const float *t, const float *w, int M, int m_valid,
                            int n_valid, int ldy, int nz, float *gf, void *gb, void *gbT,
                            float *loss, cudaStream_t st);
// Bias gradients of every layer: column sums over the M rows of G[l] (width
// out_p[l], network z M out_p[l] further) into the flat gradients.
struct ColsumArgs {
    const float *G[kMaxLayers];
    int M, nz;
};
cudaError_t launch_colsum(const ColsumArgs &c, const NetDims &d, float *grads, cudaStream_t st);
// AdamW on the flat parameters of nz networks from network k0 on; mask bit 0: a
// parameter (padding keeps 0), bit 1: decays.
cudaError_t launch_adamw(float *w, const float *g, float *m, float *v, const unsigned char *mask,
                         const NetDims &d, int k0, int nz, const AdamArgs &a, cudaStream_t st);
// BF16 copies of the flat parameters of network k.
cudaError_t launch_weights_bf16(const float *w, const NetDims &d, int k, cudaStream_t st);

// Cell list (celllist.cu).  The sort key of NP i is its cell (tb == 1) or
// type * n_cells + cell (tb = the number of types): the cell order lists all NPs
// of type 0 cell by cell, then those of type 1, and so on.  count and start
// cover the tb * n_cells keys.
struct CellBufs {
    int *key, *rank, *count, *start, *arrived, *sorted, *tile_sum;
    int *pos;    // cell-ordered position of NP i (the inverse of sorted)
    float4 *sxq; // cell-ordered (x, y, z, type as int bits): the positions of the
                 // build, and with a neighbour list the current positions (the
                 // integrator writes each new position to its NP's slot);
                 // sxq[n] is a record far from every NP (type 0) that pads the
                 // neighbour lists
};
// Build the cell list of positions xq.
cudaError_t launch_cell_build(const CellGrid &g, const float4 *xq, const int *typ, int n,
                              CellBufs &b, cudaStream_t st);
// Rewrite the cell-ordered records from positions xq in the order of the last build.
cudaError_t launch_cell_refresh(const CellBufs &b, const float4 *xq, const int *typ, int n,
                                cudaStream_t st);
// Verlet neighbour list over the cells (celllist.cu): entries are cell-order
// slots; entry k of the NP at cell-order slot p at nbr[nbr_index(k, p, n)]
// -- blocks of four entries, block j of all slots contiguous, so that a thread
// reads its next four entries with one 16-byte load and a warp reads 512
// contiguous bytes; cap (a multiple of 4) entries per slot; a list's last block
// is padded with entries n naming the far record sxq[n].  nnbr [n] the full
// counts by slot; x_ref [n] the positions of the last build by particle index.
__host__ __device__ __forceinline__ size_t nbr_index(int k, int p, int n)
{
    return ((size_t)(k >> 2) * (size_t)n + (size_t)p) * 4 + (size_t)(k & 3);
}
struct NbrList {
    unsigned *nbr; // partner slots
    int *nnbr;
    float4 *x_ref;
    unsigned long long *builds; // number of builds run (device counter)
    int cap;
};
// rcc2 (or NULL): squared cutoffs of the truncated Coulomb term per type pair
// (8 x 8); with it the lists cover both cutoffs and the list force kernel adds
// C q_a q_b r_ij / r^3 within the Coulomb cutoff to the LJ term.
// Cell list and neighbour lists of positions xq in one cooperative launch (gate:
// NULL = always, else only when *gate != 0).  bar: kBarWords words, all but the bound
// zero between launches (cleared by the host after FLAG_TIMEOUT).  While FLAG_TIMEOUT is
// set the list kernels return without touching anything (wait_expired).
enum : int {
    kBarArrived = 0, // CTAs arrived at the grid barrier
    kBarDone = 1,    // CTAs done
    kBarDrawn = 2,   // slots drawn by the build's warps
    kBarGates = 3,   // gates inside a launch of many steps (three)
    kBarPolls = 6,   // bound of a barrier wait in polls, set by the host
    kBarWords = 7,
};
cudaError_t launch_list_build(const CellGrid &g, const CellBufs &b, const float4 *xq,
                              const int *typ, int n, const PairTab *tab, const float *rcc2,
                              float skin, const NbrList &l, int *flags, const int *gate,
                              unsigned *bar, cudaStream_t st);
// `steps` steps (at most kMaxFusedSteps) from the device step counter on, of a
// simulation of n <= kMaxFusedNps whose pair forces all come from the lists, in one
// cooperative launch; I as for the integrator, bar as above, sxq2 a second array of
// cell-ordered records like b.sxq (its record n far from every NP), F_lj [n][8] scratch.
constexpr int kMaxFusedSteps = 256;
constexpr int kMaxFusedNps = 65536;
int list_steps_capacity(); // NPs one launch can hold on the current device
cudaError_t launch_list_steps(const CellGrid &g, const CellBufs &b, int n, const PairTab *tab,
                              const float *rcc2, float skin, const NbrList &l, unsigned *bar,
                              const IntArgs &I, const StepParams &p, float4 *sxq2, float *F_lj,
                              int steps, cudaStream_t st);
cudaError_t launch_lj_nbr(const CellGrid &g, const CellBufs &b, const float4 *xq,
                          const int *typ, int n, const PairTab *tab, const float *rcc2,
                          const NbrList &l, float *F_lj, int *gate, const int *flags,
                          cudaStream_t st);
int cell_scan_tiles(int n_cells);

// Stats (stats.cu)
double pair_hist_cell_edge(double r_max, double L); // cell edge of the histogram's grid
cudaError_t launch_pair_hist(const double *x, int n, double r_max, int n_bins,
                             const CellGrid &g, const CellBufs &b,
                             unsigned long long *hist, cudaStream_t st);
cudaError_t launch_radial_hist(const double *x, int n, double r_max, int n_bins,
                               unsigned long long *hist, cudaStream_t st);
// mode 0: per-CTA sums of x; 1: sums of |x - c|^2; 2: componentwise minima;
// 3: componentwise maxima of |x_d|.  part holds 3 doubles per CTA of 256 threads.
// I(q) of Sec. 3.3 for a piecewise-constant g on [0, r_max), and its fractal form
// N_surf^2 (q R_g)^(-D_f) into out_frac (or NULL); device arrays.
cudaError_t launch_scattering(const double *g, int n_bins, double r_max, const double *q, int n_q,
                              double n_surf, double Rg, double Df, double *out,
                              double *out_frac, cudaStream_t st);
// Half diameter of every type (surface band of N_surf).
struct SurfHalf {
    double h[NPSIM_MAX_TYPES];
};
cudaError_t launch_surface_count(const double *x, const int *typ, int n, double R,
                                 const SurfHalf &hs, unsigned long long *count, cudaStream_t st);
cudaError_t launch_block_reduce(int mode, const double *x, int n, const double *c,
                                double *part, cudaStream_t st);
// Boxes of edge eps0 2^k with a particle, k = k0 .. k0 + n_scales - 1, added to
// counts[k]; tables: n_scales of table_size keys (a power of two >= 2n).
cudaError_t launch_boxcount(const double *x, int n, const double *origin, double eps0, int k0,
                            int n_scales, unsigned long long *tables,
                            unsigned long long table_size, unsigned long long *counts, int *flags,
                            cudaStream_t st);
// Split float64 positions (SoA) into the integrator's hi (mirror) / lo words,
// and back (x = hi + lo in float64, for statistics).
cudaError_t launch_mirror(const double *x, const int *typ, const float *charge_by_type,
                          int n, float4 *xq, float *x_lo, cudaStream_t st);
cudaError_t launch_positions_f64(const float4 *xq, const float *x_lo, int n, double *x,
                                 cudaStream_t st);
// The same for n NPs whose lo words are rows of a [3][ld] array (one droplet of
// an ensemble); x is [3][n].
cudaError_t launch_positions_f64_ld(const float4 *xq, const float *x_lo, int n, int ld,
                                    double *x, cudaStream_t st);
// The state as host-facing AoS float64 (n x 3 each; NULL outputs are skipped):
// position hi + lo, velocity, force hi + lo.  x_lo, v and F are rows of [3][ld],
// [3][ld] and [6][ld] arrays (ld = n, or one droplet's part of an ensemble's).
cudaError_t launch_state_aos(const float4 *xq, const float *x_lo, const float *v, const float *F,
                             int n, size_t ld, double *xo, double *vo, double *Fo,
                             cudaStream_t st);

} // namespace npsim
