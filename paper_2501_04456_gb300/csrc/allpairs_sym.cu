// allpairs_sym.cu -- all-pairs forces (step (ii) of the loop in arXiv 2501.04456
// Sec. 2.2) with each unordered pair evaluated once: the force on the row goes
// to the row's sum, its opposite to the partner's (Newton's third law).
//
// What bounds the pair sum is the FP32 pipe.  The one-sided kernels
// (allpairs_grouped.cu) spend 11 packed lanes on every ordered pair, 22 on a
// pair of particles; here the pair costs 14 (20 against 34 where LJ acts), see
// coul_sym_sweep / sym_row_segment for the warp's rotation that adds the
// partners' sums without atomics and in a fixed order.
//
// Rows and columns follow the type-grouped order.  Row tile r meets the j-tiles
// at or beyond its own diagonal block only; these units (a triangle) are cut
// into equal ranges handed out at run time as in the other grouped kernels.  A
// range writes its rows' sums to slot row + range, and every unit beyond the
// diagonal its partners' sums to its own place in the column partials, 12 bytes
// per partner and row tile: N^2 / (2 ITILE) x 12 bytes a launch.  k_sym_reduce
// then adds both kinds of partials of every position in a fixed order, reading
// them along the grouped order (coalesced even where the particles' indices are
// in no spatial order), and writes one 32-byte record per particle, which the
// integrator reads in particle order.
#include "npsim_internal.cuh"

namespace npsim {

namespace {

template <int BLOCK, int KI, int JT, bool LJ>
__global__ void __launch_bounds__(BLOCK, (sym_min_ctas<BLOCK, KI>()))
k_pairs_sym(const float4 *__restrict__ xq, const int *__restrict__ perm,
            const int *__restrict__ tblk, const PairTab *__restrict__ tab, int has_coul, StreamK sk, unsigned *__restrict__ work, float *__restrict__ slots)
{
    constexpr int ITILE = BLOCK * KI;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    SymSmem<BLOCK, KI, JT> &sm = *reinterpret_cast<SymSmem<BLOCK, KI, JT> *>(s_dyn);
    __shared__ float4 s_tab[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ int s_range;
    for (int k = threadIdx.x; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; k += BLOCK)
        s_tab[k] = tab->e[k]; // ordered before use by the first tile's barrier
    float *cols = slots + (size_t)(sk.n_it + sk.grid) * 6 * ITILE;

    for (int c = blockIdx.x; c < sk.grid;) {
        const long long p_end = sk_begin(sk, c + 1);
        long long p = sk_begin(sk, c);
        int r = tri_row_of(sk, p);
        while (p < p_end) {
            const long long r0 = tri_row_begin(sk, r), r1 = tri_row_begin(sk, r + 1);
            const int jt0 = sk.tri * r + (int)(p - r0);
            const int jt1 = (int)min((long long)sk.n_jt, jt0 + (p_end - p));
            sym_row_segment<BLOCK, KI, JT, LJ>(
                xq, perm, tblk, 0, sk.len, s_tab, has_coul, r, jt0, jt1, sm,
                slots + (size_t)(r + c) * 6 * ITILE, cols + sym_col_offset(sk.len, ITILE, r),
                (size_t)(sk.len - (r + 1) * ITILE));
            p += jt1 - jt0;
            r += p == r1;
        }
        // the next free range (see next_range in allpairs_grouped.cu)
        __syncthreads();
        if (threadIdx.x == 0)
            s_range = (int)gridDim.x + (int)atomicAdd(work, 1u);
        __syncthreads();
        c = s_range;
    }
    if (threadIdx.x == 0) { // the last CTA out resets the counters
        __threadfence();
        if (atomicAdd(work + 1, 1u) == gridDim.x - 1) {
            work[0] = 0u;
            work[1] = 0u;
            __threadfence();
        }
    }
}

__global__ void __launch_bounds__(256)
k_sym_reduce(StreamK sk, const float *__restrict__ slots, const int *__restrict__ perm,
             float *__restrict__ F_pair)
{
    __shared__ float s_part[3][6][64];
    const int p = blockIdx.x * 64 + (threadIdx.x & 63);
    const int part = threadIdx.x >> 6;
    const int r = blockIdx.x * 64 / sk.itile; // itile is a multiple of 64
    const int c0 = sk_cta_of(sk, tri_row_begin(sk, r));
    const int c1 = sk_cta_of(sk, tri_row_begin(sk, r + 1) - 1);
    float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
    sym_sum_partials(slots + (size_t)(r + c0) * 6 * sk.itile, c1 - c0 + 1,
                     slots + (size_t)(sk.n_it + sk.grid) * 6 * sk.itile, sk.itile, sk.len, r, r,
                     p, part, h, l);
    sym_finish(s_part, part, h, l, perm[p], F_pair);
}

struct SEntry {
    ApConfig cfg;
    const void *fn;
    int smem;
};

#define NPSIM_SYM(B, K, J, LJ)                                                              \
    SEntry                                                                                  \
    {                                                                                       \
        ApConfig{B, K, J, 0}, (const void *)k_pairs_sym<B, K, J, LJ>, (int)sizeof(SymSmem<B, K, J>) \
    }

// Where each shape is the best, launch + reduction by grouped length (ms; the best
// one-sided kernel in brackets).  Coulomb: <128,8,128> 24576 0.168 [0.219], 100352 2.34
// [3.26], 300032 20.4 [28.8]; <64,8,128> 34304 0.299; <128,4,128> 5120 0.023 [0.025],
// 16384 0.086 [0.113]; <64,4,64> 7680 0.035, 11776 0.054; <64,2,64> 1024 0.015 [0.017],
// 2560 0.017 [0.019].  (Eight rows above 20480 only: kSymLongRows.)  LJ + Coulomb:
// <128,8,128> 30208 0.298 [0.382], 300032 21.7 [32.0]; <64,8,128> 60416 0.994 [1.39];
// <128,4,128> 16384 0.111 [0.134]; <64,4,64> 8192 0.045 [0.056]; <128,2,128> 4096 0.025
// [0.029], as the next; <64,2,64> 1024 0.019 [0.023], 2560 0.021 [0.025]: long rows want
// many rows per thread, short ones many small units.
const SEntry kSym[] = {
    NPSIM_SYM(128, 8, 128, false), NPSIM_SYM(64, 8, 128, false), NPSIM_SYM(128, 4, 128, false),
    NPSIM_SYM(64, 4, 64, false),   NPSIM_SYM(64, 2, 64, false),
};

const SEntry kSymLj[] = {
    NPSIM_SYM(128, 8, 128, true), NPSIM_SYM(64, 8, 128, true), NPSIM_SYM(128, 4, 128, true),
    NPSIM_SYM(64, 4, 64, true),   NPSIM_SYM(128, 2, 128, true), NPSIM_SYM(64, 2, 64, true),
};

const SEntry &entry(bool lj, int idx) { return lj ? kSymLj[idx] : kSym[idx]; }

} // namespace

int sym_num_configs(bool lj)
{
    return (int)(lj ? sizeof(kSymLj) : sizeof(kSym)) / (int)sizeof(SEntry);
}

ApConfig sym_config(bool lj, int idx) { return entry(lj, idx).cfg; }

int sym_occupancy(bool lj, int idx)
{
    const SEntry &e = entry(lj, idx);
    int occ = 0;
    if (cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, e.smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, e.fn, e.cfg.block, e.smem) !=
            cudaSuccess)
        return 0;
    return occ;
}

size_t sym_slots_floats(const StreamK &sk)
{
    return (size_t)(sk.n_it + sk.grid) * 6 * (size_t)sk.itile + sym_col_floats(sk.len, sk.itile);
}

cudaError_t launch_allpairs_sym(bool lj, int idx, const StreamK &sk, const float4 *xq,
                                const int *perm, const int *tblk, const PairTab *tab,
                                int has_coul, unsigned *work, float *slots, cudaStream_t st)
{
    const SEntry &e = entry(lj, idx);
    StreamK a = sk;
    void *args[] = {(void *)&xq,       (void *)&perm, (void *)&tblk, (void *)&tab,
                    (void *)&has_coul, (void *)&a,    (void *)&work, (void *)&slots};
    cudaError_t rc = cudaFuncSetAttribute(e.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, e.smem);
    if (rc != cudaSuccess)
        return rc;
    return cudaLaunchKernel(e.fn, dim3(sk.ctas > 0 ? min(sk.ctas, sk.grid) : sk.grid),
                            dim3(e.cfg.block), args, (size_t)e.smem, st);
}

cudaError_t launch_sym_reduce(const StreamK &sk, const float *slots, const int *perm,
                              float *F_pair, cudaStream_t st)
{
    if (sk.len <= 0)
        return cudaSuccess;
    k_sym_reduce<<<sk.len / 64, 256, 0, st>>>(sk, slots, perm, F_pair);
    return cudaGetLastError();
}

} // namespace npsim
