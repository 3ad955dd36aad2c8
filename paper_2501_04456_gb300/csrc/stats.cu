// stats.cu -- post-processing statistics of arXiv 2501.04456 Sec. 3 on the GPU:
//  * pair-distance histogram for the RDF of Sec. 3.2 (ordered pairs, bins of
//    width r_max/n_bins over [0, r_max)); candidates come from a cell grid, a
//    float32 distance test discards far pairs and settles the bin of all but those
//    near a bin boundary, whose bin is decided in float64 from the float64
//    positions with the operations sqrt(dx*dx + dy*dy + dz*dz) and floor(r / dr)
//    rounded one by one (no fused multiply-add), so integer counts are exact;
//  * radial histogram of |x| for the concentration C_NPs(r) of Sec. 3.2;
//  * the scattered intensity I(q) of Sec. 3.3 as the transform of g(r);
//  * N_surf, the number of NPs at the droplet surface (Sec. 1: the scattered
//    intensity grows with N_surf^2), counted as the NPs whose centre lies in
//    the band (-r_i, r_i) about the surface, | |x_i| - R(t) | < r_i, the band
//    in which Sec. 2.2 step (iv) applies the interface force;
//  * per-CTA partial sums (centre of mass, squared deviations) and minima,
//    finished on the host in CTA order (deterministic);
//  * box counting: the number of distinct integer triples floor((x - o)/eps)
//    via an open-addressing hash set in device memory (the count does not
//    depend on insertion order).
#include "npsim_internal.cuh"

namespace npsim {

namespace {

__device__ __forceinline__ int cell_coord_s(float x, const CellGrid &g)
{
    int c = (int)floorf((x + g.L) * g.inv_h);
    return min(max(c, 0), g.dim - 1);
}

__device__ __forceinline__ double dist_rn(double ax, double ay, double az, double bx,
                                          double by, double bz)
{
    const double dx = __dsub_rn(ax, bx), dy = __dsub_rn(ay, by), dz = __dsub_rn(az, bz);
    return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)),
                                __dmul_rn(dz, dz)));
}

constexpr int kMaxSmemBins = 4096;

// Parameters of the pair histogram: the candidate cells (edge about a third of
// the prefilter radius, stencil half-width w) and the float32 classification.
struct PairHistArgs {
    int n, n_bins, w, copies; // copies: histogram copies per CTA (power of two; 0: global atomics)
    double dr;
    float r_cut;  // prefilter radius: r_max plus the error of a float32 distance
    float inv_dr; // bins per unit length
    float tol;    // bound of the error of a float32 distance, in bins
};

// One thread per NP at cell-order slot p and layer dz of its stencil (blockIdx.y),
// each unordered pair once: layers above its own, in its own layer the rows
// behind its own, in its own row the slots behind p -- whose slots are all larger
// than p.  Rows and cells that r_cut cannot reach from the NP's own coordinates
// are left out.
//
// What bounds it is the work per candidate.  In float64 (1/64 of the float32 rate
// here) the square root and the division of every pair within r_max take the
// time: 33 ms for 200000 NPs of an aggregate (3e8 pairs).  A bin is nearly always
// certain in float32: with t the float32 distance in bins and tol the bound of its
// error (positions rounded to their hi words, the rounding of the difference, of
// r^2 and of the square root), floor(t) is the bin unless t lies within tol of a
// boundary; only those pairs (about 0.2 % at r_max = 10, 128 bins) are decided in
// float64 as before, so the counts are the same.  Counts go to `copies` copies of
// the histogram in shared memory (neighbouring lanes to different copies).
__global__ void __launch_bounds__(128)
k_pair_hist(const double *__restrict__ x, PairHistArgs a, CellGrid g,
            const int *__restrict__ start, const int *__restrict__ sorted,
            const float4 *__restrict__ sxq, unsigned long long *__restrict__ hist)
{
    extern __shared__ unsigned int s_h[];
    const int n_h = a.n_bins * a.copies;
    for (int b = threadIdx.x; b < n_h; b += blockDim.x)
        s_h[b] = 0u;
    __syncthreads();
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int dz = blockIdx.y;
    const int copy = a.copies ? (int)threadIdx.x & (a.copies - 1) : 0;
    if (p < a.n) {
        const float4 pi = sxq[p];
        const int cx = cell_coord_s(pi.x, g), cy = cell_coord_s(pi.y, g),
                  cz = cell_coord_s(pi.z, g);
        const float rc2 = a.r_cut * a.r_cut;
        const float h = 1.0f / g.inv_h, slack = 1e-3f * h; // cell coordinates are rounded
        const int z = cz + dz;
        const float gz = dz > 0 ? fmaxf(0.0f, (float)z * h - g.L - pi.z - slack) : 0.0f;
        if (z < g.dim && !(gz * gz > rc2)) {
            for (int dy = dz > 0 ? -a.w : 0; dy <= a.w; ++dy) {
                const int y = cy + dy;
                if (y < 0 || y >= g.dim)
                    continue;
                const float gy = dy > 0   ? fmaxf(0.0f, (float)y * h - g.L - pi.y - slack)
                                 : dy < 0 ? fmaxf(0.0f, pi.y + g.L - (float)(y + 1) * h - slack)
                                          : 0.0f;
                const float left = rc2 - gz * gz - gy * gy;
                if (left < 0.0f)
                    continue;
                const float ext = sqrtf(left) + slack;
                const int base = (z * g.dim + y) * g.dim;
                const bool own = dz == 0 && dy == 0;
                const int x0 = max(cell_coord_s(pi.x - ext, g), max(cx - a.w, 0));
                const int x1 = min(cell_coord_s(pi.x + ext, g), min(cx + a.w, g.dim - 1));
                const int q0 = own ? p + 1 : start[base + x0];
                const int q1 = start[base + x1 + 1];
                for (int q = q0; q < q1; ++q) {
                    const float4 pj = sxq[q];
                    const float ex = pi.x - pj.x, ey = pi.y - pj.y, ez = pi.z - pj.z;
                    const float r2 = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                    if (!(r2 <= rc2))
                        continue;
                    const float t = r2 * rsqrtf(r2) * a.inv_dr;
                    int bin = (int)t;
                    const float fr = t - (float)bin;
                    if (!(fr > a.tol && fr < 1.0f - a.tol)) { // near a boundary
                        const int i = sorted[p], j = sorted[q];
                        const double r =
                            dist_rn(x[i], x[a.n + i], x[2 * (size_t)a.n + i], x[j], x[a.n + j],
                                    x[2 * (size_t)a.n + j]);
                        const double bb = floor(__ddiv_rn(r, a.dr));
                        bin = bb < (double)a.n_bins ? (int)bb : a.n_bins;
                    }
                    if (bin < a.n_bins) {
                        if (a.copies)
                            atomicAdd(&s_h[bin * a.copies + copy], 1u);
                        else
                            atomicAdd(&hist[bin], 2ull);
                    }
                }
            }
        }
    }
    __syncthreads();
    if (a.copies)
        for (int b = threadIdx.x; b < a.n_bins; b += blockDim.x) {
            unsigned long long c = 0;
            for (int k = 0; k < a.copies; ++k)
                c += s_h[b * a.copies + k];
            if (c)
                atomicAdd(&hist[b], 2ull * c); // ordered pairs
        }
}

__global__ void __launch_bounds__(256)
k_radial_hist(const double *__restrict__ x, int n, double dr, int n_bins,
              unsigned long long *__restrict__ hist)
{
    __shared__ unsigned int s_h[kMaxSmemBins];
    const bool smem = n_bins <= kMaxSmemBins;
    if (smem)
        for (int b = threadIdx.x; b < n_bins; b += blockDim.x)
            s_h[b] = 0u;
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const double r = dist_rn(x[i], x[n + i], x[2 * n + i], 0.0, 0.0, 0.0);
        const double bb = floor(__ddiv_rn(r, dr));
        if (bb < (double)n_bins) {
            if (smem)
                atomicAdd(&s_h[(int)bb], 1u);
            else
                atomicAdd(&hist[(int)bb], 1ull);
        }
    }
    __syncthreads();
    if (smem)
        for (int b = threadIdx.x; b < n_bins; b += blockDim.x)
            if (s_h[b])
                atomicAdd(&hist[b], (unsigned long long)s_h[b]);
}

// NPs with | |x_i| - R | < half_sigma[type_i] (|x| and the difference in
// float64, rounded operation by operation as in the radial histogram).
__global__ void __launch_bounds__(256)
k_surface_count(const double *__restrict__ x, const int *__restrict__ typ, int n, double R,
                SurfHalf hs, unsigned long long *__restrict__ count)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    int in = 0;
    if (i < n) {
        const double r = dist_rn(x[i], x[n + i], x[2 * n + i], 0.0, 0.0, 0.0);
        in = fabs(__dsub_rn(r, R)) < hs.h[typ[i]];
    }
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if ((threadIdx.x & 31) == 0 && m)
        atomicAdd(count, (unsigned long long)__popc(m));
}

// G(u) = sin u - u cos u (the antiderivative of u sin u): by its series below
// u = 0.5, where the difference of the two terms would cancel.
__device__ __forceinline__ double scat_G(double u)
{
    if (u < 0.5) {
        const double u2 = u * u;
        // u^3/3 - u^5/30 + u^7/840 - u^9/45360 + u^11/3991680 - u^13/518918400
        double s = -1.0 / 518918400.0;
        s = s * u2 + 1.0 / 3991680.0;
        s = s * u2 - 1.0 / 45360.0;
        s = s * u2 + 1.0 / 840.0;
        s = s * u2 - 1.0 / 30.0;
        s = s * u2 + 1.0 / 3.0;
        return s * u2 * u;
    }
    return sin(u) - u * cos(u);
}

// One warp per q: I(q) = N_surf^2 4 pi sum_b g_b [G(q r_{b+1}) - G(q r_b)] / q^3
// (q = 0: N_surf^2 4 pi sum_b g_b (r_{b+1}^3 - r_b^3) / 3); lane l sums bins l,
// l + 32, ... and the lanes are combined in a fixed butterfly order.  out_frac
// (or NULL): the fractal form N_surf^2 (q R_g)^(-D_f).
__global__ void k_scattering(const double *__restrict__ g, int n_bins, double dr,
                             const double *__restrict__ q, int n_q, double n_surf, double Rg,
                             double Df, double *__restrict__ out, double *__restrict__ out_frac)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= n_q)
        return;
    const double qq = q[w];
    double acc = 0.0;
    for (int b = lane; b < n_bins; b += 32) {
        const double r0 = b * dr, r1 = (b + 1) * dr;
        const double t = qq > 0.0 ? scat_G(qq * r1) - scat_G(qq * r0)
                                  : (r1 * r1 * r1 - r0 * r0 * r0) / 3.0;
        acc += g[b] * t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
        const double four_pi = 12.566370614359172953850573533118;
        const double n2 = n_surf * n_surf;
        out[w] = n2 * (qq > 0.0 ? four_pi * acc / (qq * qq * qq) : four_pi * acc);
        if (out_frac)
            out_frac[w] = n2 * pow(qq * Rg, -Df);
    }
}

// Per-CTA partials: mode 0 -> sum of x (3 values), 1 -> sum of |x - c|^2
// (1 value), 2 -> componentwise minimum (3 values), 3 -> componentwise maximum
// of |x_d| (3 values).  Tree reduction in a fixed order inside the CTA.
template <int MODE>
__global__ void __launch_bounds__(256)
k_block_reduce(const double *__restrict__ x, int n, const double *__restrict__ c,
               double *__restrict__ part)
{
    __shared__ double s[3][256];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double a0, a1, a2;
    if (MODE == 2) {
        a0 = a1 = a2 = INFINITY;
        if (i < n) {
            a0 = x[i];
            a1 = x[n + i];
            a2 = x[2 * n + i];
        }
    } else if (MODE == 3) {
        a0 = a1 = a2 = 0.0;
        if (i < n) {
            a0 = fabs(x[i]);
            a1 = fabs(x[n + i]);
            a2 = fabs(x[2 * n + i]);
        }
    } else if (MODE == 0) {
        a0 = a1 = a2 = 0.0;
        if (i < n) {
            a0 = x[i];
            a1 = x[n + i];
            a2 = x[2 * n + i];
        }
    } else {
        a0 = a1 = a2 = 0.0;
        if (i < n) {
            const double e0 = __dsub_rn(c[0], x[i]), e1 = __dsub_rn(c[1], x[n + i]),
                         e2 = __dsub_rn(c[2], x[2 * n + i]);
            a0 = __dadd_rn(__dadd_rn(__dmul_rn(e0, e0), __dmul_rn(e1, e1)),
                           __dmul_rn(e2, e2));
        }
    }
    s[0][threadIdx.x] = a0;
    s[1][threadIdx.x] = a1;
    s[2][threadIdx.x] = a2;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            for (int d = 0; d < 3; ++d) {
                const double u = s[d][threadIdx.x], w = s[d][threadIdx.x + o];
                s[d][threadIdx.x] = (MODE == 2) ? fmin(u, w)
                                    : (MODE == 3) ? fmax(u, w) : __dadd_rn(u, w);
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[3 * blockIdx.x + 0] = s[0][0];
        part[3 * blockIdx.x + 1] = s[1][0];
        part[3 * blockIdx.x + 2] = s[2][0];
    }
}

constexpr unsigned long long kEmpty = ~0ull;

__device__ __forceinline__ unsigned long long mix64(unsigned long long k)
{
    // SplitMix64 finaliser (S. Vigna): spreads keys over the table.
    k ^= k >> 30;
    k *= 0xBF58476D1CE4E5B9ull;
    k ^= k >> 27;
    k *= 0x94D049BB133111EBull;
    k ^= k >> 31;
    return k;
}

// Scale k = k0 + blockIdx.y (box edge eps0 2^k) in its own table of mask + 1 keys
// and counter.  A key that is there already is seen by a plain read: at the
// coarse scales most particles find theirs, and a compare-and-swap each would
// queue on a handful of addresses.
__global__ void k_box_insert(const double *__restrict__ x, int n, const double *__restrict__ o,
                             double eps0, int k0, unsigned long long *__restrict__ tables,
                             unsigned long long mask, unsigned long long *__restrict__ counts,
                             int *__restrict__ flags)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const double eps = ldexp(eps0, k0 + (int)blockIdx.y);
    unsigned long long *table = tables + (size_t)blockIdx.y * (mask + 1);
    long long b[3];
    for (int k = 0; k < 3; ++k)
        b[k] = (long long)floor(__ddiv_rn(__dsub_rn(x[(size_t)k * n + i], o[k]), eps));
    // triples are non-negative (o is the minimum corner); 21 bits per axis
    if (b[0] >= (1 << 21) || b[1] >= (1 << 21) || b[2] >= (1 << 21)) {
        atomicOr(flags, FLAG_BAD_CELL);
        return;
    }
    const unsigned long long key = ((unsigned long long)b[2] << 42) |
                                   ((unsigned long long)b[1] << 21) | (unsigned long long)b[0];
    unsigned long long h = mix64(key) & mask;
    for (unsigned long long probe = 0; probe <= mask; ++probe) {
        if (*(volatile unsigned long long *)&table[h] == key)
            return;
        const unsigned long long prev = atomicCAS(&table[h], kEmpty, key);
        if (prev == kEmpty) {
            atomicAdd(&counts[k0 + blockIdx.y], 1ull);
            return;
        }
        if (prev == key)
            return;
        h = (h + 1) & mask;
    }
    atomicOr(flags, FLAG_BAD_CELL); // table full (cannot happen: size >= 2n)
}

} // namespace

// float32 prefilter radius: r_max plus a margin far above float32 rounding of
// positions of magnitude <= L
static float pair_hist_r_cut(double r_max, double L)
{
    return (float)(r_max * (1.0 + 1e-4) + 1e-5 * L + 1e-6);
}

// The cell edge the histogram wants (make_grid may enlarge it): a third of the
// prefilter radius leaves about 2.3 candidates per pair within it (27 cells of its
// own size: 6.4); the margin covers float32 rounding of the cell coordinates.
double pair_hist_cell_edge(double r_max, double L)
{
    return (double)pair_hist_r_cut(r_max, L) / 3.0 * (1.0 + 1e-3);
}

cudaError_t launch_pair_hist(const double *x, int n, double r_max, int n_bins,
                             const CellGrid &g, const CellBufs &b,
                             unsigned long long *hist, cudaStream_t st)
{
    PairHistArgs a{};
    a.n = n;
    a.n_bins = n_bins;
    a.dr = r_max / (double)n_bins;
    a.r_cut = pair_hist_r_cut(r_max, (double)g.L);
    a.inv_dr = (float)(1.0 / a.dr);
    a.w = (int)ceil((double)a.r_cut * (double)g.inv_h * (1.0 + 1e-6));
    a.w = a.w < 1 ? 1 : a.w > g.dim ? g.dim : a.w;
    // a float32 distance is off by the positions' lo words (2 x 2^-24 L per
    // component, less than 2.1e-7 L in all) and a few roundings of relative 2^-24;
    // four times the first, 1e-6 of the largest distance for the second
    a.tol = (float)((8.4e-7 * (double)g.L + 1e-6 * (double)a.r_cut) / a.dr);
    a.copies = n_bins <= 1024 ? 4 : n_bins <= 2048 ? 2 : n_bins <= kMaxSmemBins ? 1 : 0;
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * n_bins, st);
    if (e != cudaSuccess)
        return e;
    k_pair_hist<<<dim3((n + 127) / 128, a.w + 1), 128, sizeof(unsigned) * n_bins * a.copies, st>>>(
        x, a, g, b.start, b.sorted, b.sxq, hist);
    return cudaGetLastError();
}

cudaError_t launch_radial_hist(const double *x, int n, double r_max, int n_bins,
                               unsigned long long *hist, cudaStream_t st)
{
    const double dr = r_max / (double)n_bins;
    cudaError_t e = cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * n_bins, st);
    if (e != cudaSuccess)
        return e;
    k_radial_hist<<<(n + 255) / 256, 256, 0, st>>>(x, n, dr, n_bins, hist);
    return cudaGetLastError();
}

cudaError_t launch_scattering(const double *g, int n_bins, double r_max, const double *q, int n_q,
                              double n_surf, double Rg, double Df, double *out,
                              double *out_frac, cudaStream_t st)
{
    const int threads = 128;
    const int grid = (n_q * 32 + threads - 1) / threads;
    k_scattering<<<grid, threads, 0, st>>>(g, n_bins, r_max / (double)n_bins, q, n_q, n_surf, Rg,
                                           Df, out, out_frac);
    return cudaGetLastError();
}

cudaError_t launch_surface_count(const double *x, const int *typ, int n, double R,
                                 const SurfHalf &hs, unsigned long long *count, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess)
        return e;
    k_surface_count<<<(n + 255) / 256, 256, 0, st>>>(x, typ, n, R, hs, count);
    return cudaGetLastError();
}

cudaError_t launch_block_reduce(int mode, const double *x, int n, const double *c,
                                double *part, cudaStream_t st)
{
    const int grid = (n + 255) / 256;
    if (mode == 0)
        k_block_reduce<0><<<grid, 256, 0, st>>>(x, n, c, part);
    else if (mode == 1)
        k_block_reduce<1><<<grid, 256, 0, st>>>(x, n, c, part);
    else if (mode == 2)
        k_block_reduce<2><<<grid, 256, 0, st>>>(x, n, c, part);
    else
        k_block_reduce<3><<<grid, 256, 0, st>>>(x, n, c, part);
    return cudaGetLastError();
}

cudaError_t launch_boxcount(const double *x, int n, const double *origin, double eps0, int k0,
                            int n_scales, unsigned long long *tables,
                            unsigned long long table_size, unsigned long long *counts, int *flags,
                            cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(
        tables, 0xFF, sizeof(unsigned long long) * table_size * (size_t)n_scales, st);
    if (e != cudaSuccess)
        return e;
    k_box_insert<<<dim3((n + 255) / 256, n_scales), 256, 0, st>>>(x, n, origin, eps0, k0, tables,
                                                                  table_size - 1, counts, flags);
    return cudaGetLastError();
}

} // namespace npsim
