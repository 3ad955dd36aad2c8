// ensemble.cu -- many independent droplets of uneven size advanced together:
// one all-pairs launch, one sum of its partials and one integrator launch per
// step cover every droplet.
//
// Each droplet d is the system of arXiv 2501.04456 Sec. 2 (its own NP types,
// charges, LJ table, radius law, seed).  Particles of all droplets are stored
// back to back (structure of arrays over the concatenation).  Inside the
// ensemble each droplet's particles are listed in a type-grouped order (each
// type's group padded to 256 positions), so every j-tile holds partners of one
// type.  The all-pairs work of a droplet is the triangle of its (row tile x
// j-tile) units at or beyond the diagonal (each pair once, sym_row_segment) or,
// for the one-sided kernel, the whole square; every row is cut into work items
// of at most `chunk` j-tiles.  The host lists the items of all droplets once,
// longest first and among equals those nearest the diagonal (48 droplets: 1.95 ms a
// launch in row order, 1.88 so), and the CTAs of one launch draw them from a device counter
// until none are left, so a 512-NP and a 32768-NP droplet share the GPU in
// proportion to their work within one launch and items rich in LJ segments
// (which cost more than Coulomb-only ones) are balanced as they run.  An item
// writes one compensated (hi, lo) float32 partial per row into its own slot and
// its partners' sums to their own places; k_ens_reduce adds them in a fixed
// order, so the result does not depend on which CTA ran which item.  The
// reduction runs along the grouped order, in which partials are contiguous, and
// hands the integrator one 32-byte record per particle (read in particle order;
// the integrator's own gathers of 24-byte slots by grouped position used to
// fetch a 32-byte sector per float).
//
// The integrator is the fused BAOAB / overdamped pass of integrate.cu with the
// droplet's own coefficients.  Noise is keyed by the droplet's seed and counted
// by the particle's index inside its droplet, so a droplet draws the same
// normals here as in a single-droplet run.
#include "npsim_internal.cuh"

namespace npsim {

namespace {

// Draws the CTA's next item (n_items: none left).  Called by every thread.
__device__ __forceinline__ int next_item(unsigned *work, int *s_item)
{
    __syncthreads(); // every thread has read *s_item and finished the last item
    if (threadIdx.x == 0)
        *s_item = (int)atomicAdd(work, 1u);
    __syncthreads();
    return *s_item;
}

// The last CTA out resets the counters for the next launch (every CTA has drawn
// its last item by the time it counts itself out).
__device__ __forceinline__ void items_done(unsigned *work)
{
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(work + 1, 1u) == gridDim.x - 1) {
            work[0] = 0u;
            work[1] = 0u;
            __threadfence();
        }
    }
}

// One-sided: at least 1024 threads resident per SM, whose register cap (64)
// holds the sweeps without spills.
template <int BLOCK, int KI, int JT>
__global__ void __launch_bounds__(BLOCK, 1024 / BLOCK)
k_ens_ljc(EnsAllpairsArgs a)
{
    constexpr int ITILE = BLOCK * KI;
    __shared__ LjcSmem<JT> sm;
    __shared__ float4 s_tab[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ int s_item;
    int cur = -1;
    for (int it = next_item(a.work, &s_item); it < a.n_items; it = next_item(a.work, &s_item)) {
        const EnsItem item = a.items[it];
        const EnsDrop &D = a.drops[item.drop];
        if (item.drop != cur) { // ordered before use by the staging barrier
            for (int k = threadIdx.x; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; k += BLOCK)
                s_tab[k] = a.tabs[item.drop].e[k];
            cur = item.drop;
        }
        ljc_row_segment<BLOCK, KI, JT>(a.xq, a.perm, a.tblk, D.gpos0, D.npad, s_tab, D.rc2_lim,
                                       D.has_coul, item.row, item.jt0, item.jt1, sm,
                                       a.slots + (size_t)item.slot * 6 * ITILE);
    }
    items_done(a.work);
}

// Each pair once (see sym_row_segment).
template <int BLOCK, int KI, int JT>
__global__ void __launch_bounds__(BLOCK, (sym_min_ctas<BLOCK, KI>()))
k_ens_sym(EnsAllpairsArgs a)
{
    constexpr int ITILE = BLOCK * KI;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    SymSmem<BLOCK, KI, JT> &sm = *reinterpret_cast<SymSmem<BLOCK, KI, JT> *>(s_dyn);
    __shared__ float4 s_tab[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ int s_item;
    int cur = -1;
    for (int it = next_item(a.work, &s_item); it < a.n_items; it = next_item(a.work, &s_item)) {
        const EnsItem item = a.items[it];
        const EnsDrop &D = a.drops[item.drop];
        if (item.drop != cur) { // ordered before use by the staging barrier
            for (int k = threadIdx.x; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; k += BLOCK)
                s_tab[k] = a.tabs[item.drop].e[k];
            cur = item.drop;
        }
        float *col = a.slots + (size_t)a.n_items * 6 * ITILE + (size_t)D.col0 +
                     sym_col_offset(D.npad, ITILE, item.row);
        sym_row_segment<BLOCK, KI, JT, true>(a.xq, a.perm, a.tblk, D.gpos0, D.npad, s_tab,
                                             D.has_coul, item.row, item.jt0, item.jt1, sm,
                                             a.slots + (size_t)item.slot * 6 * ITILE, col,
                                             (size_t)(D.npad - (item.row + 1) * ITILE));
    }
    items_done(a.work);
}

// The partials of every grouped position, 64 positions per CTA (they share a
// droplet and a row tile: both are multiples of 64 long).
__global__ void __launch_bounds__(256)
k_ens_reduce(EnsAllpairsArgs a)
{
    __shared__ float s_part[3][6][64];
    const int g0 = blockIdx.x * 64;
    const EnsDrop &D = a.drops[a.dblk[g0 >> 8]];
    const int p = g0 - D.gpos0 + (threadIdx.x & 63); // position in the droplet's order
    const int part = threadIdx.x >> 6;
    const int r = (g0 - D.gpos0) / a.itile;
    const int s0 = a.row_first[D.row0 + r], s1 = a.row_first[D.row0 + r + 1];
    float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
    sym_sum_partials(a.slots + (size_t)s0 * 6 * a.itile, s1 - s0,
                     a.slots + (size_t)a.n_items * 6 * a.itile + (size_t)D.col0, a.itile, D.npad, r,
                     a.sym ? r : 0, p, part, h, l);
    sym_finish(s_part, part, h, l, a.perm[D.gpos0 + p], a.F_pair);
}

template <int MODE>
__global__ void __launch_bounds__(256)
k_ens_integrate(EnsIntArgs a, int n_total, int n_drops)
{
    constexpr bool ASSEMBLE = (MODE != MODE_A);
    constexpr bool DO_A = (MODE == MODE_A || MODE == MODE_BA);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    // this thread's state first (in flight during the barrier below)
    int d = 0, ti = 0;
    float4 xh = make_float4(0.f, 0.f, 0.f, 0.f);
    float lx = 0.f, ly = 0.f, lz = 0.f;
    float v[3] = {0.f, 0.f, 0.f};
    if (i < n_total) {
        d = a.drop_of[i];
        ti = a.typ[i];
        xh = a.xq[i];
        lx = a.x_lo[i];
        ly = a.x_lo[n_total + i];
        lz = a.x_lo[2 * n_total + i];
        if (MODE != MODE_FORCES) {
            v[0] = a.v[i];
            v[1] = a.v[n_total + i];
            v[2] = a.v[2 * n_total + i];
        }
    }
    // the device step counter: read by thread 0 before the CTA's one barrier,
    // the CTA counted in right after, and the last CTA to count advances it
    __shared__ long long s_step;
    if (threadIdx.x == 0)
        s_step = *a.step;
    __syncthreads();
    const long long step = s_step;
    if (DO_A && threadIdx.x == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(a.done, 1u);
        if (prev == gridDim.x - 1) {
            *a.step = step + 1;
            *a.done = 0u;
            __threadfence();
        }
    }
    if (DO_A) {
        // spring radii of step + 1 for every (droplet, type), spread over the
        // first CTAs of the launch (one entry per thread)
        for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_drops * NPSIM_MAX_TYPES;
             e += gridDim.x * blockDim.x) {
            const EnsDrop &D = a.drops[e / NPSIM_MAX_TYPES];
            a.spring[(size_t)((step + 1) & 1) * n_drops * NPSIM_MAX_TYPES + e] =
                spring_entry(D.R0, D.k_evap, D.dt, step + 1,
                             D.tc[e % NPSIM_MAX_TYPES].half_sigma);
        }
    }
    const float4 *spring = a.spring + (size_t)(step & 1) * n_drops * NPSIM_MAX_TYPES;

    if (i < n_total) {
        const int n = n_total;
        const EnsDrop &D = a.drops[d];
        const int li = i - D.offset;
        const TypeCoef tc = D.tc[ti];
        float Fh[3] = {0.f, 0.f, 0.f}, Fl[3] = {0.f, 0.f, 0.f};
        if (ASSEMBLE) {
            if (a.F_pair) {
                const float4 *q = reinterpret_cast<const float4 *>(a.F_pair + 8 * (size_t)i);
                const float4 q0 = q[0], q1 = q[1];
                Fh[0] = q0.x;
                Fh[1] = q0.y;
                Fh[2] = q0.z;
                Fl[0] = q0.w;
                Fl[1] = q1.x;
                Fl[2] = q1.y;
            }
            if (a.ext_on) {
                float ex, ey, ez;
                external_force(xh, lx, ly, lz, tc.kw, tc.mg, tc.mw2,
                               spring[d * NPSIM_MAX_TYPES + ti], D.wall, D.rot_mode, ex, ey,
                               ez, (float)D.R0,
                               MODE == MODE_FORCES ? nullptr : a.flags); // steps only
                df_add(Fh[0], Fl[0], ex);
                df_add(Fh[1], Fl[1], ey);
                df_add(Fh[2], Fl[2], ez);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                Fh[k] = a.F[k * n + i];
                Fl[k] = a.F[(3 + k) * n + i];
            }
        }
        advance_particle<MODE>(i, n, (uint32_t)li, tc, D.integrator, 0.5f * (float)D.dt, D.seed,
                               step, xh, lx, ly, lz, Fh, Fl, v, a.x_lo, a.v, a.F, a.xq, a.flags);
    }
}

struct EEntry {
    ApConfig cfg;
    const void *fn;
    int smem;
    bool sym;
};

#define NPSIM_ENS_SYM(B, K, J)                                                              \
    EEntry                                                                                  \
    {                                                                                       \
        ApConfig{B, K, J, 0}, (const void *)k_ens_sym<B, K, J>, (int)sizeof(SymSmem<B, K, J>), \
            true                                                                            \
    }

// j-tiles of at most 256 partners: the droplets' type groups are padded to 256.
// Launch + reduction (ms; the one-sided kernel in brackets): <64,8,128> 48 droplets of
// 512 to 32768 NPs 1.87 [2.70], 128 of 512 to 8192 0.633 [0.787], 4 of 32768 to 65536
// 2.50 [3.72]; <128,4,128> 8 of 4000 to 8000 0.132 [0.159]; <128,2,128> 16 of 512 to 4096
// 0.054 [0.061]; <64,2,64> 3 of 300 to 600 0.019 [0.020].  The three others are within 1 to
// 4 % of the best beside them: <128,8,128> 2 of 100000 to 200000 12.1, <64,4,64> 128 of 512
// to 8192 0.639, <64,8,64> 48 of 512 to 32768 1.95.
// The last shape is the one-sided kernel, for ensembles whose column partials
// (6 n^2 / itile bytes per droplet) do not fit; each pair once is faster on all
// others.
const EEntry kEns[] = {
    NPSIM_ENS_SYM(128, 8, 128), NPSIM_ENS_SYM(64, 8, 128), NPSIM_ENS_SYM(128, 4, 128),
    NPSIM_ENS_SYM(64, 8, 64),   NPSIM_ENS_SYM(64, 4, 64),  NPSIM_ENS_SYM(128, 2, 128),
    NPSIM_ENS_SYM(64, 2, 64),
    EEntry{ApConfig{256, 1, 256, 0}, (const void *)k_ens_ljc<256, 1, 256>, 0, false},
};

} // namespace

int ens_num_configs() { return (int)(sizeof(kEns) / sizeof(kEns[0])); }

ApConfig ens_config(int idx) { return kEns[idx].cfg; }

bool ens_sym(int idx) { return kEns[idx].sym; }

int ens_occupancy(int idx)
{
    const EEntry &e = kEns[idx];
    int occ = 0;
    if ((e.smem && cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        e.smem) != cudaSuccess) ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, e.fn, e.cfg.block, e.smem) !=
            cudaSuccess)
        return 0;
    return occ;
}

cudaError_t launch_ens_allpairs(int idx, int ctas, const EnsAllpairsArgs &a, cudaStream_t st)
{
    const EEntry &e = kEns[idx];
    if (e.smem) {
        const cudaError_t rc =
            cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, e.smem);
        if (rc != cudaSuccess)
            return rc;
    }
    EnsAllpairsArgs b = a;
    void *args[] = {(void *)&b};
    const cudaError_t rc =
        cudaLaunchKernel(e.fn, dim3(ctas), dim3(e.cfg.block), args, (size_t)e.smem, st);
    if (rc != cudaSuccess)
        return rc;
    k_ens_reduce<<<a.n_pos / 64, 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_ens_integrate(int mode, const EnsIntArgs &a, int n_total, int n_drops,
                                 cudaStream_t st)
{
    const int grid = (n_total + 255) / 256;
    switch (mode) {
    case MODE_FORCES: k_ens_integrate<MODE_FORCES><<<grid, 256, 0, st>>>(a, n_total, n_drops); break;
    case MODE_A: k_ens_integrate<MODE_A><<<grid, 256, 0, st>>>(a, n_total, n_drops); break;
    case MODE_BA: k_ens_integrate<MODE_BA><<<grid, 256, 0, st>>>(a, n_total, n_drops); break;
    case MODE_B: k_ens_integrate<MODE_B><<<grid, 256, 0, st>>>(a, n_total, n_drops); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

} // namespace npsim
