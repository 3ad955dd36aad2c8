// celllist.cu -- cell binning (step (i) of the loop in arXiv 2501.04456 Sec. 2.2:
// NPs are sorted into spatial cells so that near neighbours are found quickly)
// and the truncated, unshifted Lennard-Jones force over the neighbouring cells
// (step (ii)):
//   F_i = sum_{j != i, r < rc_ij} 24 eps_ij (2 (s_ij/r)^12 - (s_ij/r)^6) r_ij / r^2.
//
// Binning is a counting sort: hash (sort key of each NP, its arrival rank from
// an atomic counter), exclusive scan of the per-key counts, scatter, then every
// NP is placed at its rank by index inside its key (one thread per NP counts
// the members of its key with a smaller index) so that the order inside a
// cell -- and therefore the float summation order of the LJ kernel -- does not
// depend on the atomic arrival order (runs are bit-reproducible).  For the LJ
// lists the key is type * n_cells + cell: the cell order lists the NPs of one
// type cell by cell, then the next type, so that consecutive threads of the
// list kernels hold NPs of one type (lists of similar length, read coalesced)
// in nearby cells (their partners lie in the same few cells).  The NP records
// (position, type in the fourth word) are written in cell order too, so the
// kernels read neighbours from contiguous memory; with a neighbour list the
// integrator keeps these records current, so the per-step list kernel reads
// every position in cell order and never gathers by particle index.
//
// The simulation keeps a Verlet neighbour list on top of the cells: the cell
// edge is the largest cutoff plus a skin, a build lists for every NP the
// partners within its pair cutoff plus the skin and records the positions it
// saw; the integrator raises a gate when some NP has moved more than half the
// skin since then, and only then does the next build kernel do its work.  A
// pair within its cutoff now was within cutoff + skin at the build, so the
// list (or, for an NP whose list overflowed, the cells of the build) holds
// every pair that can interact: the forces are those of a rebuild every step.  The
// cell edge is at least the largest cutoff (times 1 + 1e-5, so float rounding
// of the cell index can never separate two NPs within the cutoff by more than
// one cell); coordinates beyond the grid are clamped into the edge cells,
// which keeps every pair within the cutoff in neighbouring cells.
#include "npsim_internal.cuh"

namespace npsim {

namespace {

__device__ __forceinline__ int cell_coord(float x, const CellGrid &g)
{
    int c = (int)floorf((x + g.L) * g.inv_h);
    return min(max(c, 0), g.dim - 1);
}

// The phases of the counting sort, grid-stride over the launch that runs them: as
// kernels of their own (statistics) or one after the other between the grid
// barriers of k_list_build.  Arrays that a phase writes and a later one reads are
// plain pointers: a phase of the same kernel must not take them through the
// read-only path.

__device__ __forceinline__ void cell_zero(int *count, int m)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < m; c += gridDim.x * blockDim.x)
        count[c] = 0;
}

__device__ __forceinline__ void cell_hash(const CellGrid &g, const float4 *xq, const int *typ,
                                          int n, int *key, int *rank, int *count)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float4 p = xq[i];
        int c = (cell_coord(p.z, g) * g.dim + cell_coord(p.y, g)) * g.dim + cell_coord(p.x, g);
        if (g.tb > 1)
            c += typ[i] * g.n_cells;
        key[i] = c;
        rank[i] = atomicAdd(&count[c], 1);
    }
}

// Exclusive scan of count[0..m) into start[0..m], start[m] = total, in three
// passes: each CTA scans a tile of kScanTile counts and records the tile total;
// one CTA scans the tile totals; every CTA then adds its tile's offset.
constexpr int kScanThreads = 256;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

// Exclusive scan of one value per thread over a CTA of kScanThreads threads;
// *total receives the sum of all values.
__device__ __forceinline__ int cta_exclusive_scan(int v, int *s_warp, int *total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += u;
    }
    if (lane == 31)
        s_warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int x = lane < kScanThreads / 32 ? s_warp[lane] : 0;
        int ix = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, ix, o);
            if (lane >= o)
                ix += u;
        }
        if (lane < kScanThreads / 32)
            s_warp[lane] = ix - x;
        if (lane == kScanThreads / 32 - 1)
            s_warp[kScanThreads / 32] = ix;
    }
    __syncthreads();
    const int r = s_warp[w] + incl - v;
    *total = s_warp[kScanThreads / 32];
    __syncthreads(); // s_warp may be reused by the caller
    return r;
}

// With `local` the tile-local scans are left in count as well.
__device__ __forceinline__ void scan_tiles(int *count, int *start, int *tile_sum, int m,
                                           int *s_warp, bool local)
{
    const int n_tiles = (m + kScanTile - 1) / kScanTile;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int base = t * kScanTile + threadIdx.x * kScanItems;
        int a[kScanItems];
        int s = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            a[k] = base + k < m ? count[base + k] : 0;
            s += a[k];
        }
        int total;
        int run = cta_exclusive_scan(s, s_warp, &total);
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            if (base + k < m) {
                start[base + k] = run;
                if (local)
                    count[base + k] = run;
            }
            run += a[k];
        }
        if (threadIdx.x == 0)
            tile_sum[t] = total;
    }
}

// One CTA: exclusive scan of the tile totals in place; start[m] = grand total.
__device__ __forceinline__ void scan_totals(int *tile_sum, int n_tiles, int *start, int m,
                                            int *s_warp)
{
    int carry = 0;
    for (int b0 = 0; b0 < n_tiles; b0 += kScanTile) {
        const int base = b0 + threadIdx.x * kScanItems;
        int a[kScanItems];
        int s = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            a[k] = base + k < n_tiles ? tile_sum[base + k] : 0;
            s += a[k];
        }
        int total;
        int run = carry + cta_exclusive_scan(s, s_warp, &total);
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            if (base + k < n_tiles)
                tile_sum[base + k] = run;
            run += a[k];
        }
        carry += total;
    }
    if (threadIdx.x == 0)
        start[m] = carry;
}

__device__ __forceinline__ void scan_add(int *start, const int *tile_sum, int m)
{
    const int n_tiles = (m + kScanTile - 1) / kScanTile;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const int off = tile_sum[t];
        const int base = t * kScanTile + threadIdx.x;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const int i = base + k * kScanThreads;
            if (i < m)
                start[i] += off;
        }
    }
}

__device__ __forceinline__ void cell_scatter(const int *key, const int *rank, const int *start,
                                             int *arrived, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        arrived[start[key[i]] + rank[i]] = i;
}

// Members of every cell in index order: the NP at arrival slot q goes to its
// cell's start plus the number of members with a smaller index (O(m) per NP for
// a cell of m members, all NPs in parallel), with its record (x, y, z, type as
// int bits).
__device__ __forceinline__ void cell_order(const int *arrived, const int *key, const int *start,
                                           const float4 *xq, const int *typ, int *sorted, int *pos,
                                           float4 *sxq, int n)
{
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const int i = arrived[q];
        const int c = key[i];
        const int b = start[c], e = start[c + 1];
        int rank = 0;
        for (int k = b; k < e; ++k)
            rank += arrived[k] < i;
        const float4 x = xq[i];
        sorted[b + rank] = i;
        pos[i] = b + rank;
        sxq[b + rank] = make_float4(x.x, x.y, x.z, __int_as_float(typ[i]));
    }
}

__global__ void k_cell_zero(int *count, int m) { cell_zero(count, m); }

__global__ void k_cell_hash(CellGrid g, const float4 *xq, const int *typ, int n, int *key,
                            int *rank, int *count)
{
    cell_hash(g, xq, typ, n, key, rank, count);
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_tiles(int *count, int *start, int *tile_sum, int m)
{
    __shared__ int s_warp[kScanThreads / 32 + 1];
    scan_tiles(count, start, tile_sum, m, s_warp, false);
}

__global__ void __launch_bounds__(kScanThreads)
k_scan_totals(int *tile_sum, int n_tiles, int *start, int m)
{
    __shared__ int s_warp[kScanThreads / 32 + 1];
    scan_totals(tile_sum, n_tiles, start, m, s_warp);
}

__global__ void __launch_bounds__(kScanThreads) k_scan_add(int *start, const int *tile_sum, int m)
{
    scan_add(start, tile_sum, m);
}

__global__ void k_cell_scatter(const int *key, const int *rank, const int *start, int *arrived,
                               int n)
{
    cell_scatter(key, rank, start, arrived, n);
}

__global__ void k_cell_order(const int *arrived, const int *key, const int *start,
                             const float4 *xq, const int *typ, int *sorted, int *pos, float4 *sxq,
                             int n)
{
    cell_order(arrived, key, start, xq, typ, sorted, pos, sxq, n);
}

// Cell-ordered records of other positions in the order of the last build.
__global__ void k_cell_gather(const int *__restrict__ sorted, const float4 *__restrict__ xq,
                              const int *__restrict__ typ, float4 *__restrict__ sxq, int n)
{
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        const int i = sorted[p];
        const float4 q = xq[i];
        sxq[p] = make_float4(q.x, q.y, q.z, __int_as_float(typ[i]));
    }
}

// Per-row-type tables in shared memory: the pair table and, per row type, its
// largest squared cutoff (force kernels) or cutoff-plus-skin (list build).
// rcc2 (or NULL): squared cutoffs of the truncated Coulomb term per type pair
// (coulomb mode 2); a pair is listed within max(LJ cutoff, Coulomb cutoff) +
// skin, counting only the terms that act (eps_ab != 0, C q_a q_b != 0).
__device__ __forceinline__ void load_tables(const PairTab *__restrict__ tab,
                                            const float *__restrict__ rcc2, float skin,
                                            float4 *s_tab, float *s_rl2, float *s_rmax,
                                            float *s_rcc2 = nullptr)
{
    for (int k = threadIdx.x; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; k += blockDim.x) {
        const float4 t = tab->e[k];
        s_tab[k] = t;
        const float rcc = rcc2 ? rcc2[k] : 0.0f;
        if (s_rcc2)
            s_rcc2[k] = rcc;
        const float r_lj = t.y != 0.0f ? sqrtf(t.z) : 0.0f;
        const float r_c = (rcc > 0.0f && t.w != 0.0f) ? sqrtf(rcc) : 0.0f;
        const float r = fmaxf(r_lj, r_c);
        s_rl2[k] = r > 0.0f ? (r + skin) * (r + skin) : 0.0f; // 0: never listed
    }
    __syncthreads();
    if (threadIdx.x < NPSIM_MAX_TYPES) {
        float m = 0.0f;
        for (int b = 0; b < NPSIM_MAX_TYPES; ++b)
            m = fmaxf(m, skin > 0.0f ? s_rl2[threadIdx.x * NPSIM_MAX_TYPES + b]
                                     : s_tab[threadIdx.x * NPSIM_MAX_TYPES + b].z);
        s_rmax[threadIdx.x] = m;
    }
    __syncthreads();
}

// Arguments of the list build: the cell grid and buffers, the positions it reads,
// the lists it writes and its grid barrier.
struct ListBuildArgs {
    CellGrid g;
    CellBufs b;
    const float4 *xq;
    const int *typ;
    int n, cap;
    const PairTab *tab;
    const float *rcc2;
    float skin;
    unsigned *nbr;
    int *nnbr;
    float4 *x_ref;
    unsigned long long *builds;
    int *flags;
    const int *gate;
    unsigned *bar; // kBar* words
};

// The neighbour list of the NP at cell-order slot p: the partners within (rc_ab +
// skin) in the cells its list radii reach, type block by type block in scan
// order, as their cell-order slots (the partner's type is the fourth word of its
// record), in blocks of four at nbr[nbr_index(k, p, n)] for k < cap; nnbr[p] =
// the full count (an NP with more than cap partners is summed from the cells
// instead).  Lists are written by slot so that the per-step force kernel, which
// runs in the same order, reads them coalesced.  Records the position of this
// build in x_ref (by particle).
__device__ __forceinline__ void nbr_slot(const ListBuildArgs &A, const float4 *sxq, int p,
                                         unsigned *__restrict__ nbr, const float *s_rl2,
                                         const float *s_rmax)
{
    const CellGrid &g = A.g;
    const int *start = A.b.start;
    const int n = A.n, cap = A.cap;
    const int tb = g.tb > 1 ? g.tb : 1;
    const float4 pi = sxq[p];
    const int i = A.b.sorted[p];
    const int ti = __float_as_int(pi.w);
    const int row = ti * NPSIM_MAX_TYPES;
    const float rmax = s_rmax[ti];
    const int cx = cell_coord(pi.x, g), cy = cell_coord(pi.y, g), cz = cell_coord(pi.z, g);
    int cnt = 0;
    for (int t = 0; t < tb; ++t) {
        if (tb > 1 && s_rl2[row + t] == 0.0f)
            continue; // no term acts between these types
        const int kofs = t * g.n_cells;
        // the cells this type pair's list radius can reach (with tb == 1, the
        // widest stencil of the row type); with type blocks every candidate
        // of block t has type t, so its squared list radius is fixed
        int w = g.ext[row + t];
        if (tb == 1)
            for (int b = 1; b < NPSIM_MAX_TYPES; ++b)
                w = max(w, (int)g.ext[row + b]);
        const float rl2_t = tb > 1 ? s_rl2[row + t] : rmax;
        for (int dz = -w; dz <= w; ++dz) {
            const int z = cz + dz;
            if (z < 0 || z >= g.dim)
                continue;
            for (int dy = -w; dy <= w; ++dy) {
                const int y = cy + dy;
                if (y < 0 || y >= g.dim)
                    continue;
                const int base = kofs + (z * g.dim + y) * g.dim;
                const int b = start[base + max(cx - w, 0)];
                const int e = start[base + min(cx + w, g.dim - 1) + 1];
                for (int q = b; q < e; ++q) {
                    const float4 pj = sxq[q];
                    const float dx = pi.x - pj.x, dy2 = pi.y - pj.y, dz2 = pi.z - pj.z;
                    const float r2 = fmaf(dx, dx, fmaf(dy2, dy2, dz2 * dz2));
                    if (r2 >= rl2_t || q == p)
                        continue;
                    const int tj = __float_as_int(pj.w);
                    if (tb > 1 || r2 < s_rl2[row + tj]) {
                        if (cnt < cap)
                            nbr[nbr_index(cnt, p, n)] = (unsigned)q;
                        ++cnt;
                    }
                }
            }
        }
    }
    // pad the last block with the far record (whole blocks of four
    // partners); an empty list gets one block of it, so that the first
    // block, which the force kernel reads before the count, always names
    // valid records
    for (int k = cnt; k < cap && (k < 4 || (k & 3)); ++k)
        nbr[nbr_index(k, p, n)] = (unsigned)n;
    A.nnbr[p] = cnt;
    if (cnt > cap)
        atomicOr(A.flags, FLAG_NBR_OVERFLOW);
    A.x_ref[i] = make_float4(pi.x, pi.y, pi.z, 0.0f);
}

// Shared memory of the list build.
struct ListBuildSmem {
    int warp[kScanThreads / 32 + 1];
    int ok;
    int off[kScanTile]; // prefix of the scan tiles' totals (when they are few enough)
    float4 tab[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    float rl2[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    float rmax[NPSIM_MAX_TYPES];
};

// True in every thread while FLAG_TIMEOUT is set.  A launch whose barrier wait gave up
// leaves the barrier's counters, the sort counts and the lists half done: until the host
// has put them right (read_flags), the list kernels queued behind it must not touch
// them -- a build would pass its barriers early and scatter past its arrays.
__device__ __forceinline__ bool wait_expired(const int *flags)
{
    return __syncthreads_or(threadIdx.x == 0 && (*(volatile const int *)flags & FLAG_TIMEOUT)) != 0;
}

// Barrier over the CTAs of a cooperative launch (all resident): phase = barriers
// passed so far, the same in every thread.  A wait is bounded (`polls`, used by the
// first thread: read once per launch, a read at every barrier took 1 % of a step of 1000
// NPs); one that
// gives up sets FLAG_TIMEOUT and returns false in every thread of its CTA, which
// then leaves the kernel.  Nobody passes a later barrier without its arrival, so the
// other CTAs give up there in turn.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned &phase, unsigned polls,
                                             int *flags, int *s_ok)
{
    __syncthreads();
    ++phase;
    if (threadIdx.x == 0) {
        const unsigned target = phase * gridDim.x;
        __threadfence();
        atomicAdd(bar + kBarArrived, 1u);
        int ok = 0;
        for (unsigned it = 0; it < polls && !ok; ++it) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar + kBarArrived) : "memory");
            ok = v >= target;
            if (!ok && it > 64)
                __nanosleep(100);
        }
        if (!ok)
            atomicOr(flags, FLAG_TIMEOUT);
        __threadfence();
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// The phases of a build by every CTA of a cooperative launch, between grid barriers
// (false: one gave up), the records going to sxq.  The counts are zero on entry and
// left zero.  With up to
// kScanTile scan tiles (a million sort keys) every CTA scans their totals itself,
// and the offsets are added while the NPs are scattered: four barriers; beyond,
// one CTA scans the totals: six.
__device__ __forceinline__ bool list_build(const ListBuildArgs &A, float4 *sxq, ListBuildSmem &S,
                                           unsigned &phase, unsigned polls)
{
    const CellBufs &B = A.b;
    const int n = A.n;
    const int m = (A.g.tb > 1 ? A.g.tb : 1) * A.g.n_cells; // sort keys
    const int n_tiles = (m + kScanTile - 1) / kScanTile;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    auto barrier = [&]() { return grid_barrier(A.bar, phase, polls, A.flags, &S.ok); };

    if (tid == 0) {
        if (A.builds)
            ++*A.builds;
        A.bar[kBarDrawn] = 0u;
    }
    cell_hash(A.g, A.xq, A.typ, n, B.key, B.rank, B.count);
    if (!barrier())
        return false;
    const bool few = n_tiles <= kScanTile;
    scan_tiles(B.count, B.start, B.tile_sum, m, S.warp, few);
    if (!barrier())
        return false;
    if (few) {
        int a[kScanItems], sum = 0, total;
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            const int t = threadIdx.x * kScanItems + k;
            a[k] = t < n_tiles ? B.tile_sum[t] : 0;
            sum += a[k];
        }
        int run = cta_exclusive_scan(sum, S.warp, &total);
#pragma unroll
        for (int k = 0; k < kScanItems; ++k) {
            S.off[threadIdx.x * kScanItems + k] = run;
            run += a[k];
        }
        __syncthreads();
        for (int c = tid; c < m; c += stride)
            B.start[c] = B.count[c] + S.off[c / kScanTile];
        if (tid == 0)
            B.start[m] = total;
        for (int i = tid; i < n; i += stride) {
            const int c = B.key[i];
            B.arrived[B.count[c] + S.off[c / kScanTile] + B.rank[i]] = i;
        }
    } else {
        if (blockIdx.x == 0)
            scan_totals(B.tile_sum, n_tiles, B.start, m, S.warp);
        if (!barrier())
            return false;
        scan_add(B.start, B.tile_sum, m);
        if (!barrier())
            return false;
        cell_scatter(B.key, B.rank, B.start, B.arrived, n);
    }
    if (!barrier())
        return false;
    cell_order(B.arrived, B.key, B.start, A.xq, A.typ, B.sorted, B.pos, sxq, n);
    cell_zero(B.count, m);
    if (!barrier())
        return false;
    // warps draw batches of 32 slots for the lists from the last slot back: the cell
    // order lists the types one after another, so the largest NPs, whose lists are
    // the longest, go first
    const int lane = threadIdx.x & 31;
    for (;;) {
        unsigned first = 0;
        if (lane == 0)
            first = atomicAdd(A.bar + kBarDrawn, 32u);
        const int left = n - (int)__shfl_sync(0xffffffffu, first, 0); // slots not drawn yet
        if (left <= 0)
            break;
        const int p = left - 1 - lane;
        if (p >= 0)
            nbr_slot(A, sxq, p, A.nbr, S.rl2, S.rmax);
    }
    return true;
}

// The last CTA out resets the barrier's counters for the next launch; true in its
// first thread.
__device__ __forceinline__ bool barrier_done(unsigned *bar)
{
    __syncthreads();
    if (threadIdx.x != 0)
        return false;
    __threadfence();
    if (atomicAdd(bar + kBarDone, 1u) != gridDim.x - 1)
        return false;
    bar[kBarArrived] = bar[kBarDone] = 0u;
    __threadfence();
    return true;
}

// The list build in one cooperative launch: counting sort of the NPs into cells,
// then the lists.  Every step launches it, and unless the integrator has raised the
// gate (some NP has moved more than half the skin) it returns at once: as nine gated
// kernels (zero, hash, three scan passes, scatter, order, gather, lists) the closed
// gate cost nine launches a step, 16 of the 33 us of a 250000-NP step of the
// truncated model; this way 8.  Six CTAs per SM (at most 42 registers): the scans of the
// cells wait for their loads, with five the builds of a dense 4.2 M-NP aggregate take 0.328
// instead of 0.312 ms per step.
__global__ void __launch_bounds__(kScanThreads, 6)
k_list_build(const __grid_constant__ ListBuildArgs A)
{
    __shared__ ListBuildSmem S;
    if (A.gate && *A.gate == 0) // nobody writes it while this kernel runs
        return;
    unsigned phase = 0;
    const unsigned polls = A.bar[kBarPolls];
    load_tables(A.tab, A.rcc2, A.skin, S.tab, S.rl2, S.rmax);
    if (wait_expired(A.flags))
        return;
    if (list_build(A, A.b.sxq, S, phase, polls))
        barrier_done(A.bar);
}

// The forces of the NP at slot p whose list overflowed: every NP of the cells of
// its build (the NP's sort key holds its build cell; a superset of its list),
// summed pair by pair into the compensated totals.  Kept out of line so that
// it takes no registers from the list loops.  Plain pointers: k_list_steps writes
// all of these arrays in the launch that reads them here.
template <bool COUL>
__device__ __noinline__ void cell_slot_forces(int p, const CellGrid g, const int *start,
                                              const int *sorted, const int *key,
                                              const float4 *sxq, float *F_lj,
                                              const float4 *s_tab, const float *s_rcc2)
{
    const float4 pi = sxq[p];
    const int i = sorted[p];
    const int ti = __float_as_int(pi.w);
    const int row = ti * NPSIM_MAX_TYPES;
    float hx = 0.f, hy = 0.f, hz = 0.f, lx = 0.f, ly = 0.f, lz = 0.f;
    const int tb = g.tb > 1 ? g.tb : 1;
    const int c = key[i] - (g.tb > 1 ? ti * g.n_cells : 0);
    const int cx = c % g.dim, cy = (c / g.dim) % g.dim, cz = c / (g.dim * g.dim);
    for (int t = 0; t < tb; ++t) {
        const int kofs = t * g.n_cells;
        int w = g.ext[row + t];
        if (tb == 1)
            for (int b = 1; b < NPSIM_MAX_TYPES; ++b)
                w = max(w, (int)g.ext[row + b]);
        for (int dz = -w; dz <= w; ++dz) {
            const int z = cz + dz;
            if (z < 0 || z >= g.dim)
                continue;
            for (int dy = -w; dy <= w; ++dy) {
                const int y = cy + dy;
                if (y < 0 || y >= g.dim)
                    continue;
                const int base = kofs + (z * g.dim + y) * g.dim;
                const int b = start[base + max(cx - w, 0)];
                const int e = start[base + min(cx + w, g.dim - 1) + 1];
                for (int q = b; q < e; ++q)
                    if (q != p) {
                        const float4 pj = sxq[q];
                        const float dx = pi.x - pj.x, dy2 = pi.y - pj.y, dz2 = pi.z - pj.z;
                        const float r2 = fmaf(dx, dx, fmaf(dy2, dy2, dz2 * dz2));
                        const int tj = __float_as_int(pj.w);
                        const float4 tt = s_tab[row + tj];
                        const float ri = rsqrtf(r2);
                        const float rinv2 = ri * ri;
                        const float s2 = tt.x * rinv2;
                        const float s6 = s2 * s2 * s2;
                        float f = r2 < tt.z ? tt.y * rinv2 * s6 * fmaf(2.0f, s6, -1.0f) : 0.0f;
                        if (COUL && r2 < s_rcc2[row + tj])
                            f = fmaf(tt.w * ri, rinv2, f);
                        two_sum_acc(hx, lx, f * dx);
                        two_sum_acc(hy, ly, f * dy2);
                        two_sum_acc(hz, lz, f * dz2);
                    }
            }
        }
    }
    float4 *o = reinterpret_cast<float4 *>(F_lj + 8 * (size_t)i);
    o[0] = make_float4(hx, hy, hz, lx);
    o[1] = make_float4(ly, lz, 0.0f, 0.0f);
}

// LJ forces (and, with rcc2, the truncated Coulomb term) from the neighbour
// lists at the current positions for the NP at cell-order slot p: its own
// record sxq[p] (kept current by the integrator), its list column and its
// partners' records are read in cell order -- coalesced over consecutive
// slots, and for the partners from the nearby cells -- and the 32-byte force
// record goes to the NP's index i = sorted[p], where the integrator reads it.
// An NP whose list overflowed sums over the cells of that build instead (a
// superset of its list).  pi: its record, cur: its first list block, cnt: its count.
// Returns the (hi x, y, z, lo x | lo y, z, 0, 0) record in o0, o1.
template <bool COUL>
__device__ __forceinline__ void slot_forces(int p, int i, const float4 pi, uint4 cur, int cnt,
                                            const CellGrid &g, const int *start,
                                            const int *sorted, const int *key,
                                            const float4 *sxq, int n, int cap,
                                            const unsigned *nbr, float *F_lj, const float4 *s_tab,
                                            const float *s_rcc2, float4 &o0, float4 &o1)
{
    const int ti = __float_as_int(pi.w);
    const int row = ti * NPSIM_MAX_TYPES;
    float hx = 0.f, hy = 0.f, hz = 0.f, lx = 0.f, ly = 0.f, lz = 0.f;
    // One pair's force added into (sx, sy, sz); 1/r^2 as rsqrt(r^2)^2, as in
    // the all-pairs kernels.  The block sums go into the compensated (hi, lo)
    // totals by flush(), once per block of up to four partners.
    auto pair = [&](const float4 pj, float &sx, float &sy, float &sz) {
        const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const int tj = __float_as_int(pj.w);
        const float4 t = s_tab[row + tj];
        const float ri = rsqrtf(r2);
        const float rinv2 = ri * ri;
        const float s2 = t.x * rinv2;
        const float s6 = s2 * s2 * s2;
        // LJ (r < rc_ab) plus, with COUL, Coulomb truncated at its own cutoff
        float f = r2 < t.z ? t.y * rinv2 * s6 * fmaf(2.0f, s6, -1.0f) : 0.0f;
        if (COUL && r2 < s_rcc2[row + tj])
            f = fmaf(t.w * ri, rinv2, f); // C q_a q_b / r^3
        sx = fmaf(f, dx, sx);
        sy = fmaf(f, dy, sy);
        sz = fmaf(f, dz, sz);
    };
    auto flush = [&](float sx, float sy, float sz) {
        two_sum_acc(hx, lx, sx);
        two_sum_acc(hy, ly, sy);
        two_sum_acc(hz, lz, sz);
    };
    // List entries arrive four at a time (one 16-byte load per block of four,
    // contiguous over consecutive slots), two blocks ahead of their use, and a
    // block's partner records are gathered one block ahead, so that each thread
    // keeps the next block's gathers and the entries after it in flight while
    // it computes.  A list's last block is padded with the far record, whose
    // terms are exactly zero, so every block is four whole pairs.  Pairs are
    // summed in list order, each block of four in float32 and then into the
    // compensated (hi, lo) total.  The first block is read before the count is
    // known (cap >= 4 entries exist for every slot).  Entries are the
    // partners' slots; a partner's type is the fourth word of its record.
    // The lists stream through once per step: they are read with the
    // evict-first (streaming) policy so that they do not push the partner
    // records out of L1 and L2.
    const uint4 *nb4 = reinterpret_cast<const uint4 *>(nbr);
    const uint4 far4 = make_uint4((unsigned)n, (unsigned)n, (unsigned)n, (unsigned)n);
    if (cnt > cap) {
        cell_slot_forces<COUL>(p, g, start, sorted, key, sxq, F_lj, s_tab, s_rcc2);
        const float4 *o = reinterpret_cast<const float4 *>(F_lj + 8 * (size_t)i);
        o0 = o[0];
        o1 = o[1];
        return;
    }
    {
        const int nblk = (cnt + 3) >> 2;
        uint4 nxt = nblk > 1 ? __ldcs(nb4 + (size_t)n + p) : far4;
        float4 pj[4];
        pj[0] = sxq[cur.x];
        pj[1] = sxq[cur.y];
        pj[2] = sxq[cur.z];
        pj[3] = sxq[cur.w];
        for (int j = 0; j < nblk; ++j) {
            const uint4 nn = j + 2 < nblk ? __ldcs(nb4 + (size_t)(j + 2) * n + p) : far4;
            float4 pn[4];
            if (j + 1 < nblk) {
                pn[0] = sxq[nxt.x];
                pn[1] = sxq[nxt.y];
                pn[2] = sxq[nxt.z];
                pn[3] = sxq[nxt.w];
            }
            float sx = 0.f, sy = 0.f, sz = 0.f;
            pair(pj[0], sx, sy, sz);
            pair(pj[1], sx, sy, sz);
            pair(pj[2], sx, sy, sz);
            pair(pj[3], sx, sy, sz);
            flush(sx, sy, sz);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                pj[u] = pn[u];
            cur = nxt;
            nxt = nn;
        }
    }
    o0 = make_float4(hx, hy, hz, lx);
    o1 = make_float4(ly, lz, 0.0f, 0.0f);
}

// List forces, one thread per cell-order slot (slot_forces), and closes the
// rebuild gate.  The CTAs take the 128-slot tiles from the last one back: the
// cell order lists the types one after another, so the last tiles hold the
// largest NPs, whose lists are the longest (several times the mean in a
// polydisperse aggregate); started first, they no longer run alone at the end
// of the launch while the short ones fill the tail.  8 CTAs of 128 per SM (64
// registers: each thread keeps two blocks of partner records and entries in
// flight).  Lists within L2 (262144 NPs of a dried aggregate, 62 partners each): 42 us,
// L1 data pipe 81 % of the active cycles: the k-th partners of a warp lie in 14 lines.
// Two or four threads per NP touch fewer (43, 47 us against 45 in the step) but do the
// work per NP as often (3 partners per NP: 16, 22 against 12).
template <bool COUL>
__global__ void __launch_bounds__(128, 8)
k_lj_nbr(const __grid_constant__ CellGrid g, const int *__restrict__ start, const int *__restrict__ sorted,
         const int *__restrict__ key, const float4 *__restrict__ sxq, int n,
         const PairTab *__restrict__ tab, const float *__restrict__ rcc2, int cap,
         const unsigned *__restrict__ nbr, const int *__restrict__ nnbr,
         float *__restrict__ F_lj, int *__restrict__ gate, const int *__restrict__ flags)
{
    __shared__ float4 s_tab[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ float s_rl2[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ float s_rcc2[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ float s_rmax[NPSIM_MAX_TYPES];
    const int p = (int)(gridDim.x - 1 - blockIdx.x) * (int)blockDim.x + (int)threadIdx.x;
    const bool expired = *flags & FLAG_TIMEOUT; // nobody sets it while this kernel runs
    int i = 0, cnt = 0;
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
    uint4 cur = make_uint4(0u, 0u, 0u, 0u);
    if (p < n) { // on their way with the tables and the flags
        i = sorted[p];
        cnt = nnbr[p];
        pi = sxq[p];
        cur = __ldcs(reinterpret_cast<const uint4 *>(nbr) + p);
    }
    load_tables(tab, COUL ? rcc2 : nullptr, 0.0f, s_tab, s_rl2, s_rmax, s_rcc2);
    if (expired) // unfinished lists (wait_expired); the gate stays open
        return;
    if (gate && blockIdx.x == 0 && threadIdx.x == 0)
        *gate = 0; // every build kernel of this step has run; the integrator may reopen it
    if (p < n) {
        float4 o0, o1;
        slot_forces<COUL>(p, i, pi, cur, cnt, g, start, sorted, key, sxq, n, cap, nbr, F_lj, s_tab,
                          s_rcc2, o0, o1);
        // one 32-byte record per NP, a whole DRAM sector
        float4 *o = reinterpret_cast<float4 *>(F_lj + 8 * (size_t)i);
        o[0] = o0;
        o[1] = o1;
    }
}

// Up to kMaxFusedSteps steps of a droplet whose pair forces all come from the lists,
// in one cooperative launch.  A step of a small droplet is three short kernels
// (gated build, list forces, integrator), 9.2 us at 1000 NPs, of which their work is
// perhaps two; here a step is one pass over the NPs and one grid barrier (1000 NPs
// 5.2 us, 30000 8.3, warps mostly waiting at the barrier):
//   A part of the first step; then per step: [barrier; build if the gate is open];
//   list forces, external forces, B and the next step's A part of each NP by the
//   thread that holds its slot; after the last step's B the counters move on.
// Arithmetic and order are those of the separate kernels (the same functions), so a
// run that mixes both is bit-identical.  Every thread holds at most one NP, whose
// state, first list block and count stay in its registers between builds, and draws
// the next step's noise before it waits at the barrier: after the barrier only the
// partners' records are on the way to its force.  While some threads still read
// their partners' records of the current positions others already write new ones, so
// the cell-ordered records alternate between two arrays; the last step's pass, which
// moves nothing, leaves them in the first.
struct FusedStepArgs {
    ListBuildArgs L;
    IntArgs I;          // xq, x_lo, v, F, typ, spring, step, flags, half_skin2, x_ref
    float4 *sxq2;       // the other cell-ordered records (n + 1, the last one far)
    float *F_lj;        // scratch of the overflow path
    const int *gate;    // set on entry: build in the first pass
    // Gates inside the launch, zero between launches: pass j reads word j mod 3,
    // raises word (j + 1) mod 3 and clears word (j + 2) mod 3, so no word is written
    // in a pass in which a CTA may still read it.
    unsigned *gates;
    int steps;
};

// The NP of one slot between builds.
struct SlotNp {
    int i, ti, cnt;
    uint4 first;               // first list block
    float q, xhi[3], xlo[3], v[3], ref[3];
};

__device__ __forceinline__ void slot_load(const FusedStepArgs &a, int n, int p, SlotNp &s)
{
    const IntArgs &I = a.I;
    s.i = a.L.b.sorted[p];
    s.cnt = a.L.nnbr[p];
    s.first = __ldcs(reinterpret_cast<const uint4 *>(a.L.nbr) + p);
    s.ti = I.typ[s.i];
    const float4 x = I.xq[s.i], r = a.L.x_ref[s.i];
    s.q = x.w;
    s.xhi[0] = x.x;
    s.xhi[1] = x.y;
    s.xhi[2] = x.z;
    s.ref[0] = r.x;
    s.ref[1] = r.y;
    s.ref[2] = r.z;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        s.xlo[d] = I.x_lo[d * n + s.i];
        s.v[d] = I.v[d * n + s.i];
    }
}

__device__ __forceinline__ void slot_store(const FusedStepArgs &a, int n, const SlotNp &s)
{
    const IntArgs &I = a.I;
    I.xq[s.i] = make_float4(s.xhi[0], s.xhi[1], s.xhi[2], s.q);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        I.x_lo[d * n + s.i] = s.xlo[d];
        I.v[d * n + s.i] = s.v[d];
    }
}

template <bool COUL>
__global__ void __launch_bounds__(kScanThreads, 2)
k_list_steps(const __grid_constant__ FusedStepArgs a, const __grid_constant__ StepParams p)
{
    __shared__ ListBuildSmem S;
    __shared__ float4 s_tab[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ float s_rl2[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ float s_rcc2[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    __shared__ float s_rmax[NPSIM_MAX_TYPES];
    __shared__ TypeCoef s_tc[NPSIM_MAX_TYPES];
    const ListBuildArgs &L = a.L;
    const int n = p.n;
    load_tables(L.tab, L.rcc2, L.skin, S.tab, S.rl2, S.rmax);
    load_tables(L.tab, COUL ? L.rcc2 : nullptr, 0.0f, s_tab, s_rl2, s_rmax, s_rcc2);
    if (threadIdx.x < NPSIM_MAX_TYPES)
        s_tc[threadIdx.x] = p.tc[threadIdx.x];
    const unsigned polls = L.bar[kBarPolls];
    if (wait_expired(L.flags)) // its barrier orders the tables, too
        return;
    const long long step0 = *a.I.step;
    const float R0f = (float)p.R0;
    unsigned phase = 0;
    // spring radii of step s + 1, by the first CTA in a pass that takes the A part of s
    auto next_spring = [&](long long s) {
        if (blockIdx.x == 0 && threadIdx.x < p.n_types)
            a.I.spring[((s + 1) & 1) * NPSIM_MAX_TYPES + threadIdx.x] =
                spring_entry(p.R0, p.k_evap, p.dt, s + 1, p.tc[threadIdx.x].half_sigma);
    };
    const float hdt = 0.5f * (float)p.dt;
    next_spring(step0);
    // the first step's A part, by particle (the slots may be those of no build yet)
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float4 x = a.I.xq[i];
        const float v[3] = {a.I.v[i], a.I.v[n + i], a.I.v[2 * n + i]};
        float Fh[3], Fl[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            Fh[d] = a.I.F[d * n + i];
            Fl[d] = a.I.F[(3 + d) * n + i];
        }
        const int ti = a.I.typ[i];
        advance_particle<MODE_A>(i, n, (uint32_t)i, s_tc[ti], p.integrator, hdt, p.seed, step0, x,
                                 a.I.x_lo[i], a.I.x_lo[n + i], a.I.x_lo[2 * n + i], Fh, Fl, v,
                                 a.I.x_lo, a.I.v, a.I.F, a.I.xq, a.I.flags, a.I.x_ref,
                                 reinterpret_cast<int *>(a.gates) + 1, a.I.half_skin2, L.b.sxq,
                                 L.b.pos, ti);
    }
    // slots spread over the CTAs a warp at a time (the launch has a thread for each)
    const int slot = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
    const bool mine = slot < n;
    SlotNp s{};
    float nz[3] = {0.f, 0.f, 0.f};
    for (int j = 1; j <= a.steps; ++j) {
        const bool last = j == a.steps;
        if (!grid_barrier(L.bar, phase, polls, L.flags, &S.ok))
            return;
        float4 *cur = (j & 1) ? L.b.sxq : a.sxq2, *nxt = (j & 1) ? a.sxq2 : L.b.sxq;
        volatile unsigned *w = a.gates;
        const bool build = w[j % 3] != 0u || (j == 1 && *(volatile int *)a.gate != 0);
        if (build) {
            if (mine && j > 1)
                slot_store(a, n, s);
            if (!grid_barrier(L.bar, phase, polls, L.flags, &S.ok) ||
                !list_build(L, cur, S, phase, polls) ||
                !grid_barrier(L.bar, phase, polls, L.flags, &S.ok))
                return;
        }
        if (mine && (build || j == 1)) {
            slot_load(a, n, slot, s);
            if (!last)
                normals3(p.seed, (uint32_t)s.i, step0 + j, 0u, nz[0], nz[1], nz[2]);
        }
        if (blockIdx.x == 0 && threadIdx.x == 0)
            w[(j + 2) % 3] = 0u;
        if (!last)
            next_spring(step0 + j);
        if (!mine)
            continue;
        const float4 spring = a.I.spring[((step0 + j) & 1) * NPSIM_MAX_TYPES + s.ti];
        const float4 pi = make_float4(s.xhi[0], s.xhi[1], s.xhi[2], __int_as_float(s.ti));
        float4 o0, o1;
        slot_forces<COUL>(slot, s.i, pi, s.first, s.cnt, L.g, L.b.start, L.b.sorted, L.b.key, cur, n,
                          L.cap, L.nbr, a.F_lj, s_tab, s_rcc2, o0, o1);
        const TypeCoef &tc = s_tc[s.ti];
        float Fh[3] = {0.f, 0.f, 0.f}, Fl[3] = {0.f, 0.f, 0.f};
        df_add_df(Fh[0], Fl[0], o0.x, o0.w);
        df_add_df(Fh[1], Fl[1], o0.y, o1.x);
        df_add_df(Fh[2], Fl[2], o0.z, o1.y);
        float ex, ey, ez;
        external_force(make_float4(s.xhi[0], s.xhi[1], s.xhi[2], s.q), s.xlo[0], s.xlo[1], s.xlo[2],
                       tc.kw, tc.mg, tc.mw2, spring, p.wall, p.rot_mode, ex, ey, ez, R0f, a.I.flags);
        df_add(Fh[0], Fl[0], ex);
        df_add(Fh[1], Fl[1], ey);
        df_add(Fh[2], Fl[2], ez);
        const float f[3] = {__fadd_rn(Fh[0], Fl[0]), __fadd_rn(Fh[1], Fl[1]), __fadd_rn(Fh[2], Fl[2])};
        if (!last) {
            kick_drift<true, true>(tc, p.integrator, hdt, nz, f, s.v, s.xhi, s.xlo);
            nxt[slot] = make_float4(s.xhi[0], s.xhi[1], s.xhi[2], __int_as_float(s.ti));
            if (!(isfinite(s.xhi[0]) && isfinite(s.xhi[1]) && isfinite(s.xhi[2])))
                atomicOr(a.I.flags, FLAG_NONFINITE);
            // moved more than half the skin since the list was built: build
            const float dx = s.xhi[0] - s.ref[0], dy = s.xhi[1] - s.ref[1], dz = s.xhi[2] - s.ref[2];
            if (!(fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= a.I.half_skin2))
                a.gates[(j + 1) % 3] = 1u;
            if (j + 1 < a.steps)
                normals3(p.seed, (uint32_t)s.i, step0 + j + 1, 0u, nz[0], nz[1], nz[2]);
        } else {
            kick_drift<true, false>(tc, p.integrator, hdt, nz, f, s.v, s.xhi, s.xlo);
            if (cur != L.b.sxq)
                L.b.sxq[slot] = pi;
            slot_store(a, n, s);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                a.I.F[d * n + s.i] = Fh[d];
                a.I.F[(3 + d) * n + s.i] = Fl[d];
            }
        }
    }
    if (barrier_done(L.bar)) { // every thread is past its use of the step and the gates
        *a.I.step = step0 + a.steps;
        for (int k = 0; k < 3; ++k)
            a.gates[k] = 0u;
        *a.I.nbr_gate = 0; // the last pass has built what the one before it asked for
    }
}

} // namespace

int cell_scan_tiles(int n_cells) { return (n_cells + kScanTile - 1) / kScanTile; }

namespace {
constexpr int kMaxGrid = 1216; // 8 CTAs on each of 152 SMs (grid-stride kernels)

int sm_count()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return sms;
}

int grid_for(int n, int block)
{
    const int g = (n + block - 1) / block;
    return g < 1 ? 1 : (g < kMaxGrid ? g : kMaxGrid);
}
} // namespace

cudaError_t launch_cell_build(const CellGrid &g, const float4 *xq, const int *typ, int n,
                              CellBufs &b, cudaStream_t st)
{
    const int B = 256;
    const int m = (g.tb > 1 ? g.tb : 1) * g.n_cells; // sort keys
    const int gn = grid_for(n, B), gc = grid_for(m, B);
    k_cell_zero<<<gc, B, 0, st>>>(b.count, m);
    k_cell_hash<<<gn, B, 0, st>>>(g, xq, typ, n, b.key, b.rank, b.count);
    const int nt = cell_scan_tiles(m);
    const int gt = nt < kMaxGrid ? nt : kMaxGrid;
    k_scan_tiles<<<gt, kScanThreads, 0, st>>>(b.count, b.start, b.tile_sum, m);
    k_scan_totals<<<1, kScanThreads, 0, st>>>(b.tile_sum, nt, b.start, m);
    k_scan_add<<<gt, kScanThreads, 0, st>>>(b.start, b.tile_sum, m);
    k_cell_scatter<<<gn, B, 0, st>>>(b.key, b.rank, b.start, b.arrived, n);
    k_cell_order<<<gn, B, 0, st>>>(b.arrived, b.key, b.start, xq, typ, b.sorted, b.pos, b.sxq, n);
    return cudaGetLastError();
}

cudaError_t launch_cell_refresh(const CellBufs &b, const float4 *xq, const int *typ, int n,
                                cudaStream_t st)
{
    k_cell_gather<<<grid_for(n, 256), 256, 0, st>>>(b.sorted, xq, typ, b.sxq, n);
    return cudaGetLastError();
}

namespace {
ListBuildArgs list_build_args(const CellGrid &g, const CellBufs &b, const float4 *xq,
                              const int *typ, int n, const PairTab *tab, const float *rcc2,
                              float skin, const NbrList &l, int *flags, const int *gate,
                              unsigned *bar)
{
    ListBuildArgs A{};
    A.g = g;
    A.b = b;
    A.xq = xq;
    A.typ = typ;
    A.n = n;
    A.cap = l.cap;
    A.tab = tab;
    A.rcc2 = rcc2;
    A.skin = skin;
    A.nbr = l.nbr;
    A.nnbr = l.nnbr;
    A.x_ref = l.x_ref;
    A.builds = l.builds;
    A.flags = flags;
    A.gate = gate;
    A.bar = bar;
    return A;
}

// A cooperative launch of `want` CTAs of kScanThreads, or as many as the device
// holds at once.
template <class... P>
cudaError_t launch_coop(void (*fn)(P...), int want, cudaStream_t st, const P &...args)
{
    int occ = 0;
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kScanThreads, 0);
    if (e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(max(1, min(want, occ * sm_count())));
    cfg.blockDim = dim3(kScanThreads);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, args...);
}
} // namespace

cudaError_t launch_list_build(const CellGrid &g, const CellBufs &b, const float4 *xq,
                              const int *typ, int n, const PairTab *tab, const float *rcc2,
                              float skin, const NbrList &l, int *flags, const int *gate,
                              unsigned *bar, cudaStream_t st)
{
    const ListBuildArgs A =
        list_build_args(g, b, xq, typ, n, tab, rcc2, skin, l, flags, gate, bar);
    // a thread per four NPs or keys
    const int m = (g.tb > 1 ? g.tb : 1) * g.n_cells;
    return launch_coop<ListBuildArgs>(k_list_build, max((n + 63) / 64, cell_scan_tiles(m)), st, A);
}

int list_steps_capacity()
{
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_list_steps<true>, kScanThreads, 0) !=
        cudaSuccess)
        return 0;
    return min(kMaxFusedNps, min(occ, 2) * sm_count() * kScanThreads); // as launch_list_steps cuts it
}

cudaError_t launch_list_steps(const CellGrid &g, const CellBufs &b, int n, const PairTab *tab,
                              const float *rcc2, float skin, const NbrList &l, unsigned *bar,
                              const IntArgs &I, const StepParams &p, float4 *sxq2, float *F_lj,
                              int steps, cudaStream_t st)
{
    FusedStepArgs a{};
    a.L = list_build_args(g, b, I.xq, I.typ, n, tab, rcc2, skin, l, I.flags, I.nbr_gate, bar);
    a.I = I;
    a.sxq2 = sxq2;
    a.F_lj = F_lj;
    a.gate = I.nbr_gate;
    a.gates = bar + kBarGates;
    a.steps = steps;
    // a warp's 32 slots per CTA while that leaves SMs free (the other warps help the
    // builds), then one CTA per SM, two when their threads do not reach n
    const int warps = (n + 31) / 32;
    const int sms = sm_count();
    const int want = n <= sms * kScanThreads ? min(warps, sms) : 2 * sms;
    if (n > list_steps_capacity())
        return cudaErrorInvalidValue; // every slot needs a thread
    return rcc2 ? launch_coop<FusedStepArgs, StepParams>(k_list_steps<true>, want, st, a, p)
                : launch_coop<FusedStepArgs, StepParams>(k_list_steps<false>, want, st, a, p);
}

cudaError_t launch_lj_nbr(const CellGrid &g, const CellBufs &b, const float4 *xq,
                          const int *typ, int n, const PairTab *tab, const float *rcc2,
                          const NbrList &l, float *F_lj, int *gate, const int *flags,
                          cudaStream_t st)
{
    (void)xq; // the current positions are the cell-ordered records b.sxq
    (void)typ;
    const int B = 128;
    const int grid = (n + B - 1) / B;
    if (rcc2)
        k_lj_nbr<true><<<grid, B, 0, st>>>(g, b.start, b.sorted, b.key, b.sxq, n, tab, rcc2,
                                           l.cap, l.nbr, l.nnbr, F_lj, gate, flags);
    else
        k_lj_nbr<false><<<grid, B, 0, st>>>(g, b.start, b.sorted, b.key, b.sxq, n, tab, nullptr,
                                            l.cap, l.nbr, l.nnbr, F_lj, gate, flags);
    return cudaGetLastError();
}

} // namespace npsim
