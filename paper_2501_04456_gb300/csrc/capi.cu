// capi.cu -- runtime behind the C ABI of include/npsim.h: owns the device
// buffers of one simulation, picks the all-pairs launch shape with a timing
// autotuner, captures chunks of steps into CUDA graphs, and implements state
// I/O, force queries, statistics, checkpoints and the test hooks.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "npsim_internal.cuh"

using namespace npsim;

namespace {

thread_local std::string g_err;

int set_err(int code, const char *fmt, ...)
{
    char buf[1024];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}

#define NP_CUDA(call)                                                                   \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return set_err(e_ == cudaErrorMemoryAllocation ? NPSIM_ERR_OOM : NPSIM_ERR_CUDA, \
                           "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_),    \
                           __FILE__, __LINE__);                                         \
    } while (0)

#define NP_REQUIRE(cond, ...)                                                           \
    do {                                                                                \
        if (!(cond))                                                                    \
            return set_err(NPSIM_ERR_INVALID_ARG, __VA_ARGS__);                         \
    } while (0)

constexpr int kChunk = 16;      // steps per captured graph
constexpr double kKf = 1.593;   // fractal prefactor, Sec. 3.1
constexpr size_t kBoxTableKeys = (size_t)8 << 20; // box-counting tables of one launch: 64 MiB

template <class T> cudaError_t dalloc(T **p, size_t count)
{
    *p = nullptr;
    return cudaMalloc((void **)p, sizeof(T) * (count ? count : 1));
}

template <class T> void dfree(T *&p)
{
    if (p)
        cudaFree((void *)p);
    p = nullptr;
}

void free_cells(CellBufs &b)
{
    dfree(b.key);
    dfree(b.rank);
    dfree(b.count);
    dfree(b.start);
    dfree(b.arrived);
    dfree(b.sorted);
    dfree(b.pos);
    dfree(b.sxq);
    dfree(b.tile_sum);
}

// Scratch of the statistics of Sec. 3 (allocated on first use, grown as needed):
// float64 positions, the cell list of the pair histogram, the results and the
// box-counting hash tables.
struct StatsWork {
    double *x = nullptr; // [3][n] float64 positions (hi + lo), when the owner has none
    int x_cap = 0;
    CellGrid grid{};
    CellBufs cb{};
    int cells_cap = 0, cells_n = 0; // cells and NPs the cell buffers hold
    // results of one call, read back in as few copies as its steps allow: 8-byte
    // words, 6 per CTA of 256 threads (reductions), the histograms, N_surf, boxes
    unsigned long long *res = nullptr;
    size_t res_cap = 0;
    double *vec = nullptr;  // centre of mass [3], box origin [3]
    unsigned long long *table = nullptr;
    size_t table_cap = 0;   // keys
};
void free_stats(StatsWork &w)
{
    dfree(w.x);
    free_cells(w.cb);
    dfree(w.res);
    dfree(w.vec);
    dfree(w.table);
    w = StatsWork{};
}

int check_device(int *sms)
{
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || count < 1)
        return set_err(NPSIM_ERR_NO_DEVICE, "no CUDA device visible");
    int dev = 0;
    NP_CUDA(cudaGetDevice(&dev));
    int major = 0, minor = 0;
    NP_CUDA(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
    NP_CUDA(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev));
    if (!(major == 10 && minor == 3))
        return set_err(NPSIM_ERR_NO_DEVICE,
                       "device %d is sm_%d%d; this library is built for sm_103a only", dev,
                       major, minor);
    if (sms)
        NP_CUDA(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
    return NPSIM_OK;
}

std::mutex g_tune_mu;
// (n, lj, grouped length, neutral NPs elided) -> (launch shape, ranges per CTA)
std::map<std::array<long long, 4>, std::pair<int, int>> g_tune_cache;
// Ranges per CTA the autotuner tries for the grouped kernels (dynamic
// launches), and the one a forced shape gets by default.
constexpr int kRangesPerCta[] = {1, 4, 16};
constexpr int kDefaultRangesPerCta = 4;
// ensembles: (grouped length, LJ on, Coulomb on) of every droplet -> launch shape
std::map<std::vector<long long>, int> g_ens_tune_cache;

void fill_streamk(StreamK &sk, int n, const ApConfig &c, int grid_target)
{
    sk.itile = c.block * c.ki;
    sk.jtile = c.jt;
    sk.n_it = (n + sk.itile - 1) / sk.itile;
    sk.n_jt = (n + c.jt - 1) / c.jt;
    sk.W = (long long)sk.n_it * sk.n_jt;
    sk.grid = (int)std::min<long long>(std::max(grid_target, 1), sk.W);
    sk.ctas = 0;
    sk.tri = 0;
    sk.len = 0;
}

// Floats of stream-K partial slots: one slot per (i-tile row, range) pair a
// row can meet, each (hi x, y, z, lo x, y, z) x itile.
// Verlet skin of the LJ neighbour lists (sigma units of the smallest type = 1),
// and the squared displacement (half the skin, less 1 % for rounding) that
// triggers a rebuild.
constexpr float kSkin = 0.3f;
constexpr float kHalfSkin2 = (0.5f * kSkin * 0.99f) * (0.5f * kSkin * 0.99f);

size_t slots_floats(const StreamK &sk)
{
    return (size_t)(sk.n_it + sk.grid) * 6 * (size_t)sk.itile;
}

} // namespace

namespace npsim {
int report_error(int code, const char *fmt, ...)
{
    char buf[1024];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return code;
}
} // namespace npsim

struct npsim_sim {
    int n = 0, T = 0, sms = 0;
    npsim_params_t P{};
    npsim_type_t types[NPSIM_MAX_TYPES]{};
    double eps_ov[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES]{};
    bool has_ov = false;
    std::vector<int32_t> h_type;
    std::vector<int32_t> h_rank; // order of each NP inside its type group (grouped kernels)
    double d_mean = 1.0;
    float charge_f[NPSIM_MAX_TYPES]{};

    cudaStream_t user = nullptr, cap = nullptr;

    // State: position = xq.xyz (hi words) + x_lo; velocity and force in float32,
    // forces as (hi, lo) pairs.  x is float64 scratch for uploads and statistics.
    double *x = nullptr;                  // [3][n]
    double *stage = nullptr;              // host-facing AoS copies [x | v | F], 9 n (lazy)
    float *x_lo = nullptr, *v = nullptr;  // [3][n]
    float *F = nullptr, *F_tmp = nullptr; // [6][n]
    float4 *xq = nullptr;
    int *typ = nullptr;
    float *slots = nullptr;
    float *F_pair = nullptr;              // [n][8] all-pairs forces (each-pair-once shapes)
    unsigned *ap_work = nullptr;          // range counters of the grouped kernels [2]
    float *F_lj = nullptr;                // [n][8]: (hi x, y, z, lo x | lo y, z, -, -)
    PairTab *tab_full = nullptr, *tab_lj = nullptr, *tab_coul = nullptr;
    float rc2_lim = 0.0f; // largest LJ rc^2 of the table (x 1.0001): tile-culling bound
    int any_charge = 0;   // Coulomb on and some type charged
    float *d_rcc2 = nullptr; // coulomb mode 2: squared Coulomb cutoff per type pair (8 x 8)
    long long *d_step = nullptr;
    float4 *d_spring = nullptr; // [2][NPSIM_MAX_TYPES] spring radius table (spring_entry)
    int *d_flags = nullptr;
    unsigned *d_done = nullptr;

    CellGrid grid{};
    CellBufs cb{};
    bool cell = false;
    double rlist[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES]{}; // list radius per type pair (0: none)
    double cell_h_min = 0.0; // smallest list radius (the cell edge the grid aims at)
    double cell_rc = 0.0;    // largest cutoff of the cell-list terms
    size_t cells_alloc = 0;  // sort keys the cell buffers hold
    NbrList nl{};          // Verlet list over the cells (cell-list LJ)
    int *d_gate = nullptr; // 1: rebuild the cell and neighbour lists at the next pass
    bool gate_open = false;    // the host has set it since the last list pass
    bool flags_unread = false; // lists may have been built since the flags were read
    unsigned *list_bar = nullptr; // words of the list kernels' grid barrier (kBarWords)
    int fused_cap = 0;            // largest n that takes fused steps
    float4 *sxq2 = nullptr;       // the other cell-ordered records of fused steps (lazy)

    bool ap = false, ap_lj = false;
    int ap_idx = 0;
    int ap_per_cta = kDefaultRangesPerCta; // stream-K ranges per CTA (grouped kernels)

    // type-grouped order for the grouped kernels (built when pair sums are on)
    int *perm = nullptr;    // [n_perm] particle at each grouped position, -1 = padding
    float *qblk = nullptr;  // [n_perm / 256] charge of each 256-position block
    int *tblk = nullptr;    // [n_perm / 256] type of each 256-position block
    int *row_pos = nullptr; // [n] grouped position of particle i (-1: no pair row)
    int n_perm = 0;         // grouped length (multiple of 512)
    int grp_len = 0;        // rows and columns the grouped kernels cover
    StreamK sk{};
    StepParams sp{};

    std::map<int, cudaGraphExec_t> graphs;
    int64_t step = 0;
    int last_chunk = 0;

    // per-kernel timing: events around each kernel group of each step of a chunk
    bool profiling = false;
    cudaEvent_t ev[kChunk][4][2]{};
    // frame recorder: device staging ring, copy stream, per-slot events
    static constexpr int kRecSlots = 3;
    float4 *rec_ring = nullptr;
    cudaStream_t rec_stream = nullptr;
    cudaEvent_t rec_ready[kRecSlots]{}, rec_done[kRecSlots]{};

    // statistics (allocated on first use)
    StatsWork sw{};

    ~npsim_sim()
    {
        for (auto &g : graphs)
            cudaGraphExecDestroy(g.second);
        graphs.clear();
        for (int k = 0; k < kRecSlots; ++k) {
            if (rec_ready[k])
                cudaEventDestroy(rec_ready[k]);
            if (rec_done[k])
                cudaEventDestroy(rec_done[k]);
        }
        if (rec_stream)
            cudaStreamDestroy(rec_stream);
        dfree(rec_ring);
        for (int j = 0; j < kChunk; ++j)
            for (int k = 0; k < 4; ++k)
                for (int e = 0; e < 2; ++e)
                    if (ev[j][k][e])
                        cudaEventDestroy(ev[j][k][e]);
        dfree(x);
        dfree(stage);
        dfree(x_lo);
        dfree(v);
        dfree(F);
        dfree(F_tmp);
        dfree(xq);
        dfree(typ);
        dfree(slots);
        dfree(F_pair);
        dfree(ap_work);
        dfree(perm);
        dfree(qblk);
        dfree(tblk);
        dfree(row_pos);
        dfree(F_lj);
        dfree(tab_full);
        dfree(tab_lj);
        dfree(tab_coul);
        dfree(d_step);
        dfree(d_spring);
        dfree(d_flags);
        dfree(d_done);
        dfree(d_gate);
        dfree(list_bar);
        dfree(sxq2);
        dfree(nl.nbr);
        dfree(nl.nnbr);
        dfree(nl.x_ref);
        dfree(nl.builds);
        free_cells(cb);
        free_stats(sw);
        dfree(d_rcc2);
        if (cap)
            cudaStreamDestroy(cap);
    }
};

namespace {

// List radius (largest acting cutoff + skin) of every type pair of a pair table,
// as the list kernels form it in float32 (0: the pair is never listed), for
// LJ (t.z = rc^2 where 24 eps = t.y != 0) and, with rcc2, the truncated
// Coulomb term (where C q_a q_b = t.w != 0).
void list_radii(const PairTab &tab, const float *rcc2, float skin, double *rl)
{
    for (int k = 0; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; ++k) {
        const float4 t = tab.e[k];
        const float r_lj = t.y != 0.0f ? std::sqrt(t.z) : 0.0f;
        const float r_c = (rcc2 && rcc2[k] > 0.0f && t.w != 0.0f) ? std::sqrt(rcc2[k]) : 0.0f;
        const float r = std::max(r_lj, r_c);
        rl[k] = r > 0.0f ? (double)r + (double)skin : 0.0;
    }
}

// Stencil half-widths of a grid for the list radii rl: a partner within r of an
// NP lies at most ceil(r / h) cells away along each axis (clamping coordinates
// beyond the grid into the edge cells only shortens distances); a relative
// margin of 1e-5 covers float32 rounding of the cell coordinates.
void set_extents(CellGrid &g, const double *rl)
{
    const double h = 1.0 / (double)g.inv_h;
    for (int k = 0; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; ++k) {
        const double e = rl[k] > 0.0 ? std::ceil(rl[k] * (1.0 + 1e-5) / h) : 1.0;
        g.ext[k] = (unsigned char)std::min(std::max(e, 1.0), 60.0);
    }
}

// Buffers of a cell list of n NPs over the g.tb * g.n_cells sort keys.  pos, sorted
// and key start at 0 so that what they name is in range before the first build.
int alloc_cells(CellGrid &g, CellBufs &b, int n)
{
    const size_t m = (size_t)std::max(g.tb, 1) * (size_t)g.n_cells;
    NP_CUDA(dalloc(&b.key, n));
    NP_CUDA(dalloc(&b.rank, n));
    NP_CUDA(dalloc(&b.count, m));
    NP_CUDA(dalloc(&b.start, m + 1));
    NP_CUDA(dalloc(&b.arrived, n));
    NP_CUDA(dalloc(&b.sorted, n));
    NP_CUDA(dalloc(&b.pos, n));
    for (int *q : {b.pos, b.sorted, b.key})
        NP_CUDA(cudaMemset(q, 0, sizeof(int) * (size_t)(n > 0 ? n : 1)));
    // one record past the NPs: a position far from every NP (type 0), the
    // partner that pads each neighbour list to whole blocks of four
    NP_CUDA(cudaMemset(b.count, 0, sizeof(int) * m)); // the list build leaves them zero
    NP_CUDA(dalloc(&b.sxq, (size_t)n + 1));
    const float4 far = make_float4(kPairPad, kPairPad, kPairPad, 0.0f);
    NP_CUDA(cudaMemcpy(b.sxq + n, &far, sizeof(far), cudaMemcpyHostToDevice));
    NP_CUDA(dalloc(&b.tile_sum, cell_scan_tiles((int)m)));
    return NPSIM_OK;
}

// Cell grid over [-L, L)^3 with edge >= h_min, at most max_cells cells.
CellGrid make_grid(double L, double h_min, long long max_cells)
{
    CellGrid g{};
    double h = h_min * (1.0 + 1e-5);
    long long dim = (long long)std::ceil(2.0 * L / h);
    if (dim < 1)
        dim = 1;
    while (dim * dim * dim > max_cells && dim > 1) {
        h *= 1.1;
        dim = (long long)std::ceil(2.0 * L / h);
    }
    g.dim = (int)dim;
    g.n_cells = (int)(dim * dim * dim);
    g.inv_h = (float)(1.0 / h);
    g.L = (float)L;
    g.tb = 1;
    for (auto &e : g.ext)
        e = 1;
    return g;
}

// The LJ cell list's grid over [-L, L)^3: edge = the smallest list radius of
// the acting type pairs (each pair scans as many cells as its own radius
// needs), sort keys (types x cells) capped at about two per NP so that the
// cell ranges stay in L2 (the edge grows until the grid fits), cell order
// grouped by type.
CellGrid lj_grid(const npsim_sim *s, double L)
{
    CellGrid g = make_grid(L, s->cell_h_min, std::max<long long>(2LL * s->n / s->T + 4096, 1 << 16));
    g.tb = s->T; // cell order grouped by type (uniform list lengths per warp)
    set_extents(g, s->rlist);
    return g;
}

// Cell buffers large enough for grid g (reallocated only when it has more keys).
int ensure_cells(npsim_sim *s, CellGrid &g)
{
    const size_t keys = (size_t)std::max(g.tb, 1) * (size_t)g.n_cells;
    if (keys > s->cells_alloc || !s->cb.key) {
        free_cells(s->cb);
        s->cells_alloc = 0;
        int rc = alloc_cells(g, s->cb, s->n);
        if (rc)
            return rc;
        s->cells_alloc = keys;
    }
    return NPSIM_OK;
}


// Launch shapes of the all-pairs sum in one index space: the identity-order
// kernels of allpairs.cu (scalar and packed), the charge-grouped Coulomb kernels
// of allpairs_grouped.cu, the Coulomb kernels of allpairs_sym.cu (each pair
// once), then the LJ + Coulomb kernels of allpairs_grouped.cu and of
// allpairs_sym.cu.
enum ShapeFamily { SF_PLAIN, SF_GRP, SF_SYM, SF_LJG, SF_SYMLJ };

int family_size(int f)
{
    switch (f) {
    case SF_PLAIN: return ap_num_configs();
    case SF_GRP: return grp_num_configs();
    case SF_SYM: return sym_num_configs(false);
    case SF_LJG: return ljg_num_configs();
    default: return sym_num_configs(true);
    }
}

int shape_count()
{
    int n = 0;
    for (int f = SF_PLAIN; f <= SF_SYMLJ; ++f)
        n += family_size(f);
    return n;
}

// Family of shape k; *local receives its index inside the family.
int shape_family(int k, int *local = nullptr)
{
    int f = SF_PLAIN;
    while (f < SF_SYMLJ && k >= family_size(f))
        k -= family_size(f++);
    if (local)
        *local = k;
    return f;
}

bool shape_grouped(int k) { return shape_family(k) != SF_PLAIN; }

// LJ + Coulomb kernels over the grouped order
bool shape_ljg(int k) { return shape_family(k) >= SF_LJG; }

// kernels that evaluate each pair once
bool shape_sym(int k)
{
    const int f = shape_family(k);
    return f == SF_SYM || f == SF_SYMLJ;
}

ApConfig shape_config(int k)
{
    int l = 0;
    switch (shape_family(k, &l)) {
    case SF_PLAIN: return ap_config(l);
    case SF_GRP: return grp_config(l);
    case SF_LJG: return ljg_config(l);
    case SF_SYM: return sym_config(false, l);
    default: return sym_config(true, l);
    }
}

// Column partials of the kernels that evaluate each pair once take 6 bytes x
// N^2 / itile (of an ensemble: summed over its droplets): allowed up to 8 GiB (1.2
// million grouped NPs with the largest row tile); beyond it the one-sided kernels,
// whose scratch grows with N, remain.  Tiles of fewer than 512 rows are candidates up to
// 512 MiB (151000 NPs at 256 rows): there they lost long before (best of 256 rows
// against best of 512 or 1024, ms: Coulomb 24500 0.183, 0.168, 100000 2.65, 2.35; LJ
// 60000 1.06, 0.99; 48 droplets of up to 32768 2.02, 1.89), and their scratch alone made
// the tuning of 400000 NPs take 7.5 GB.
size_t sym_max_bytes(int itile) { return itile < 512 ? (size_t)512 << 20 : (size_t)8 << 30; }

// The largest of the candidates' scratch sizes (floats) that can be had, with `extra`
// floats behind it: where the largest does not fit, the shapes that need it drop out and
// the next is tried.  *all: every candidate has its place.  NPSIM_TUNE_BYTES bounds what
// a tuner may take (for a GPU that others share).
int alloc_tune_scratch(std::vector<size_t> needs, size_t extra, float **tmp, size_t *need, bool *all)
{
    const char *env = getenv("NPSIM_TUNE_BYTES");
    const size_t most = env ? (size_t)strtoull(env, nullptr, 10) : SIZE_MAX;
    std::sort(needs.begin(), needs.end(), std::greater<size_t>());
    for (size_t f : needs) {
        cudaError_t e = cudaErrorMemoryAllocation;
        if ((f + extra) * sizeof(float) <= most) {
            e = dalloc(tmp, f + extra);
            if (e != cudaSuccess && e != cudaErrorMemoryAllocation)
                NP_CUDA(e);
            cudaGetLastError(); // a failed allocation
        }
        if (e == cudaSuccess) {
            *need = f;
            *all = f == needs[0];
            return NPSIM_OK;
        }
    }
    return set_err(NPSIM_ERR_OOM, "no room for the scratch of any launch shape");
}

// Coulomb kernels with eight rows per thread add 256 terms to a partner's sum before it
// is compensated.  Beyond this grouped length the best one-sided kernels had tiles of
// 512 partners, the same chain (60000 NPs, rms error against float64 4.0e-8, one-sided
// 4.8e-8); up to it some had 256 (16384, 20480), and four rows per thread, or the LJ +
// Coulomb kernels, whose chains are half as long, keep to theirs (16384 NPs 3.1e-8,
// one-sided 3.4e-8, eight rows 3.8e-8).  Launch and sum, four against eight rows, ms:
// 13824 NPs 0.064, 0.070; 15360 0.080, 0.080; 16384 0.086, 0.084; 18432 0.104, 0.098;
// 20480 0.126, 0.127; 24576 0.172, 0.168; 32256 0.287, 0.268.
constexpr int kSymLongRows = 20480;

int shape_occupancy(const npsim_sim *s, int k, bool lj)
{
    int l = 0;
    const int f = shape_family(k, &l);
    if (f != SF_PLAIN && (!s->perm || s->grp_len == 0))
        return 0;
    if (f == SF_SYM || f == SF_SYMLJ) {
        const ApConfig c = shape_config(k);
        const int itile = c.block * c.ki;
        if (sym_col_floats(s->grp_len, itile) * sizeof(float) > sym_max_bytes(itile))
            return 0;
        return f == SF_SYMLJ ? sym_occupancy(true, l) : lj ? 0 : sym_occupancy(false, l);
    }
    if (f == SF_LJG)
        return ljg_occupancy(l);
    if (f == SF_GRP)
        return lj ? 0 : grp_occupancy(l);
    return ap_occupancy(l, lj);
}

// Stream-K split of shape k on `ctas` CTAs; the grouped kernels cut the
// units into per_cta ranges per CTA and hand them out at run time.
void shape_streamk(const npsim_sim *s, int k, int ctas, int per_cta, StreamK &sk)
{
    const ApConfig c = shape_config(k);
    if (!shape_grouped(k)) {
        fill_streamk(sk, s->n, c, ctas);
        return;
    }
    // rows and columns over the grouped order (grp_len is a multiple of 512)
    sk.itile = c.block * c.ki;
    sk.jtile = c.jt;
    sk.n_it = (s->grp_len + sk.itile - 1) / sk.itile;
    sk.n_jt = s->grp_len / c.jt;
    sk.W = (long long)sk.n_it * sk.n_jt;
    sk.tri = 0;
    sk.len = s->grp_len;
    if (shape_sym(k)) {
        sk.tri = sk.itile / sk.jtile;
        sk.W = tri_row_begin(sk, sk.n_it);
    }
    ctas = std::max(ctas, 1);
    sk.grid = (int)std::min<long long>((long long)ctas * std::max(per_cta, 1), sk.W);
    sk.ctas = std::min(ctas, sk.grid);
}

// Type-pair table of a pair sum: LJ + Coulomb, LJ only or Coulomb only.
const PairTab *pair_table(const npsim_sim *s, bool lj, bool coul)
{
    return lj ? (coul ? s->tab_full : s->tab_lj) : s->tab_coul;
}

size_t shape_slots_floats(const StreamK &sk)
{
    return sk.tri ? sym_slots_floats(sk) : slots_floats(sk);
}

cudaError_t shape_launch(const npsim_sim *s, int k, bool lj, bool coul, const StreamK &sk,
                         float *slots, cudaStream_t st)
{
    int l = 0;
    const int f = shape_family(k, &l);
    if (f == SF_SYM || f == SF_SYMLJ)
        return launch_allpairs_sym(f == SF_SYMLJ, l, sk, s->xq, s->perm, s->tblk,
                                   pair_table(s, lj, coul),
                                   !coul || !s->any_charge ? 0 : s->P.sum_neutral ? 2 : 1,
                                   s->ap_work, slots, st);
    if (f == SF_LJG)
        return launch_allpairs_ljgrp(l, sk, s->xq, s->perm, s->n_perm, s->tblk,
                                     pair_table(s, lj, coul), lj ? s->rc2_lim : 0.0f,
                                     coul ? s->any_charge : 0, s->ap_work, slots, st);
    if (f == SF_GRP)
        return launch_allpairs_grouped(l, sk, s->xq, s->perm, s->n_perm, s->qblk, s->ap_work,
                                       slots, st);
    return launch_allpairs(l, lj, sk, s->xq, s->typ, s->n, lj ? pair_table(s, lj, coul) : nullptr,
                           slots, st);
}

// The sum of shape k's partials that a step pays for beside its all-pairs
// launch: the reduction into F_pair, or the integrator's read of the slots.
cudaError_t shape_sum(const npsim_sim *s, int k, const StreamK &sk, const float *slots, float *out,
                      cudaStream_t st)
{
    if (sk.tri)
        return launch_sym_reduce(sk, slots, s->perm, out, st);
    return launch_slot_sum(slots, sk, shape_grouped(k) ? s->grp_len : s->n, out, st);
}

// Queue the pair forces of the current positions and one integrator pass at
// step (device counter) + step_ofs; step_commit: this pass ends a chunk of
// steps and moves the counter on.  Kernel groups timed by npsim_kernel_times.
enum { KG_ALLPAIRS = 0, KG_CELL_BUILD = 1, KG_CELL_LJ = 2, KG_INTEGRATE = 3 };

int enqueue_pass(npsim_sim *s, int mode, bool want_lj, bool want_coul, bool ext, float *Fout,
                 cudaStream_t st, int prof_slot = -1, int step_ofs = 0, bool step_commit = false)
{
    const bool ap_lj = want_lj && s->P.lj_mode == 1;
    // with the neutral NPs left out and no type charged, the grouped Coulomb
    // sum is empty
    const bool ap_coul = want_coul && s->P.coulomb == 1 &&
                         !(shape_grouped(s->ap_idx) && s->grp_len == 0);
    // coulomb mode 2: Coulomb truncated at its cutoff, summed with LJ from the lists
    const bool cell_coul = want_coul && s->P.coulomb == 2;
    const bool lj_cell = s->cell && (want_lj || cell_coul);
    const bool ap = ap_lj || ap_coul;
    const bool ljg = shape_ljg(s->ap_idx);
    // the ungrouped kernels also serve a Coulomb-only pass of an LJ simulation
    // whose tuned shape is charge-grouped (never: LJ excludes it) or type-grouped
    const bool grouped = ap && shape_grouped(s->ap_idx) && (ljg || !ap_lj);
    const bool prof = prof_slot >= 0 && s->profiling;
    auto mark = [&](int group, int edge) -> cudaError_t {
        // inside stream capture a plain cudaEventRecord only orders the capture;
        // the External flag makes it a real event-record node of the graph
        return prof ? cudaEventRecordWithFlags(s->ev[prof_slot][group][edge], st,
                                               cudaEventRecordExternal)
                    : cudaSuccess;
    };
    if (lj_cell) {
        // builds (past its gate check) only after an NP has moved more than half the
        // skin since the last build
        NP_CUDA(mark(KG_CELL_BUILD, 0));
        NP_CUDA(launch_list_build(s->grid, s->cb, s->xq, s->typ, s->n, s->tab_full, s->d_rcc2,
                                  kSkin, s->nl, s->d_flags, s->d_gate, s->list_bar, st));
        NP_CUDA(mark(KG_CELL_BUILD, 1));
        NP_CUDA(mark(KG_CELL_LJ, 0));
        NP_CUDA(launch_lj_nbr(s->grid, s->cb, s->xq, s->typ, s->n,
                              want_lj ? s->tab_full : s->tab_coul,
                              cell_coul ? s->d_rcc2 : nullptr, s->nl, s->F_lj, s->d_gate, s->d_flags,
                              st));
        NP_CUDA(mark(KG_CELL_LJ, 1));
    }
    if (ap) {
        NP_CUDA(mark(KG_ALLPAIRS, 0));
        NP_CUDA(shape_launch(s, s->ap_idx, ap_lj, ap_coul, s->sk, s->slots, st));
        if (s->sk.tri)
            NP_CUDA(launch_sym_reduce(s->sk, s->slots, s->perm, s->F_pair, st));
        NP_CUDA(mark(KG_ALLPAIRS, 1));
    }
    IntArgs a{};
    a.x_lo = s->x_lo;
    a.v = s->v;
    a.F = Fout;
    a.typ = s->typ;
    a.xq = s->xq;
    a.slots = ap && !s->sk.tri ? s->slots : nullptr;
    a.F_pair = ap && s->sk.tri ? s->F_pair : nullptr;
    a.sk = s->sk;
    a.F_lj = lj_cell ? s->F_lj : nullptr;
    a.ext_on = ext ? 1 : 0;
    a.field_slots = (a.slots && !ap_lj && !ljg) ? 1 : 0; // ljg sums C q_a q_b from its table
    a.row_pos = grouped ? s->row_pos : nullptr;
    a.spring = s->d_spring;
    a.x_ref = s->cell ? s->nl.x_ref : nullptr;
    a.sxq = s->cell ? s->cb.sxq : nullptr;
    a.cell_pos = s->cell ? s->cb.pos : nullptr;
    a.nbr_gate = s->d_gate;
    a.half_skin2 = kHalfSkin2;
    a.step = s->d_step;
    a.step_ofs = step_ofs;
    a.step_commit = step_commit ? 1 : 0;
    a.flags = s->d_flags;
    a.done = s->d_done;
    NP_CUDA(mark(KG_INTEGRATE, 0));
    NP_CUDA(launch_integrate(mode, a, s->sp, st));
    NP_CUDA(mark(KG_INTEGRATE, 1));
    return NPSIM_OK;
}

// Queue k >= 1 steps from the step in the device counter: A, (pairs, BA) x
// (k - 1), pairs, B; the launches carry their offsets from the counter, and
// the last one moves it on by k.
int enqueue_chunk(npsim_sim *s, int k, cudaStream_t st)
{
    IntArgs a{};
    a.x_lo = s->x_lo;
    a.v = s->v;
    a.F = s->F;
    a.typ = s->typ;
    a.xq = s->xq;
    a.sk = s->sk;
    a.spring = s->d_spring;
    a.x_ref = s->cell ? s->nl.x_ref : nullptr;
    a.sxq = s->cell ? s->cb.sxq : nullptr;
    a.cell_pos = s->cell ? s->cb.pos : nullptr;
    a.nbr_gate = s->d_gate;
    a.half_skin2 = kHalfSkin2;
    a.step = s->d_step; // the chunk's first step; launch j + 1 below is at step + j + 1
    a.step_ofs = 0;
    a.step_commit = 0;
    a.flags = s->d_flags;
    a.done = s->d_done;
    NP_CUDA(launch_integrate(MODE_A, a, s->sp, st));
    for (int j = 0; j < k; ++j) {
        // the last pass (B at step + k) moves the counter on to step + k
        int rc = enqueue_pass(s, j + 1 < k ? MODE_BA : MODE_B, true, true, true, s->F, st, j,
                              j + 1, j + 1 == k);
        if (rc)
            return rc;
    }
    return NPSIM_OK;
}

int get_graph(npsim_sim *s, int k, cudaGraphExec_t *out)
{
    auto it = s->graphs.find(k);
    if (it != s->graphs.end()) {
        *out = it->second;
        return NPSIM_OK;
    }
    NP_CUDA(cudaStreamBeginCapture(s->cap, cudaStreamCaptureModeThreadLocal));
    int rc = enqueue_chunk(s, k, s->cap);
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamEndCapture(s->cap, &g);
    if (rc) {
        if (g)
            cudaGraphDestroy(g);
        return rc;
    }
    if (e != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "graph capture failed: %s", cudaGetErrorString(e));
    cudaGraphExec_t ex = nullptr;
    e = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "graph instantiate failed: %s", cudaGetErrorString(e));
    s->graphs[k] = ex;
    *out = ex;
    return NPSIM_OK;
}

int set_gate(npsim_sim *s, int v)
{
    s->gate_open = v != 0;
    if (s->d_gate) {
        NP_CUDA(cudaMemcpyAsync(s->d_gate, &v, sizeof(int), cudaMemcpyHostToDevice, s->user));
        NP_CUDA(cudaStreamSynchronize(s->user)); // v lives on this stack frame
    }
    return NPSIM_OK;
}

// A neighbour list overflowed (those NPs were summed from the cells, so the
// forces were exact): grow the list to 1.25 x the longest count plus 8, drop
// the graphs (they hold the old buffer) and rebuild at the next pass.
int grow_neighbour_list(npsim_sim *s)
{
    std::vector<int> cnt((size_t)s->n);
    NP_CUDA(cudaMemcpy(cnt.data(), s->nl.nnbr, sizeof(int) * cnt.size(), cudaMemcpyDeviceToHost));
    const int mx = *std::max_element(cnt.begin(), cnt.end());
    if (mx <= s->nl.cap)
        return NPSIM_OK;
    const int cap = ((mx + mx / 4 + 8) + 3) & ~3; // whole blocks of four entries
    unsigned *nb = nullptr;
    cudaError_t e = dalloc(&nb, (size_t)cap * s->n);
    if (e != cudaSuccess)
        return set_err(NPSIM_ERR_OOM, "neighbour list of %d x %d entries: %s", cap, s->n,
                       cudaGetErrorString(e));
    NP_CUDA(cudaMemsetAsync(nb, 0, sizeof(unsigned) * (size_t)cap * s->n, s->user));
    dfree(s->nl.nbr);
    s->nl.nbr = nb;
    s->nl.cap = cap;
    for (auto &g : s->graphs)
        cudaGraphExecDestroy(g.second);
    s->graphs.clear();
    return set_gate(s, 1);
}

// Bound of a wait at the list kernels' grid barrier in polls (about a microsecond
// each): 2^22, and beyond 2^21 NPs in proportion to n^2, because a build compares each NP
// with every member of its cell -- all of them when one far NP stretches the grid or the
// positions are not finite (by count of its loads 2 s at 4 million NPs, bound 16 s).
unsigned list_wait_polls(int n)
{
    const double f = (double)n / (1 << 21);
    return (unsigned)std::min(4294967295.0, std::ldexp(std::max(1.0, f * f), 22));
}

int set_list_wait(npsim_sim *s, unsigned polls)
{
    NP_CUDA(cudaMemcpyAsync(s->list_bar + kBarPolls, &polls, sizeof(polls), cudaMemcpyHostToDevice,
                            s->user));
    NP_CUDA(cudaStreamSynchronize(s->user)); // polls lives on this stack frame
    return NPSIM_OK;
}

// A list kernel's barrier wait has given up and the launches behind it have left the
// lists alone: its counters and the sort counts back to zero, the lists to be built
// anew, and the host's step count to the device's, which steps that were not finished
// have not moved on.
int recover_lists(npsim_sim *s)
{
    if (s->list_bar) {
        NP_CUDA(cudaMemsetAsync(s->list_bar, 0, kBarPolls * sizeof(unsigned), s->user));
        NP_CUDA(cudaMemsetAsync(s->cb.count, 0, sizeof(int) * s->cells_alloc, s->user));
    }
    long long step = 0;
    NP_CUDA(cudaMemcpyAsync(&step, s->d_step, sizeof(step), cudaMemcpyDeviceToHost, s->user));
    NP_CUDA(cudaStreamSynchronize(s->user));
    s->step = step;
    return set_gate(s, 1);
}

int read_flags(npsim_sim *s)
{
    int h = 0;
    NP_CUDA(cudaMemcpyAsync(&h, s->d_flags, sizeof(int), cudaMemcpyDeviceToHost, s->user));
    NP_CUDA(cudaStreamSynchronize(s->user));
    s->flags_unread = false;
    if (h & FLAG_TIMEOUT) { // before all else: the other bits may come of it
        NP_CUDA(cudaMemsetAsync(s->d_flags, 0, sizeof(int), s->user));
        int rc = recover_lists(s);
        return rc ? rc : set_err(NPSIM_ERR_TIMEOUT, "a bounded device wait expired");
    }
    if (h & FLAG_NBR_OVERFLOW) {
        const int rest = h & ~FLAG_NBR_OVERFLOW;
        NP_CUDA(cudaMemcpyAsync(s->d_flags, &rest, sizeof(int), cudaMemcpyHostToDevice, s->user));
        NP_CUDA(cudaStreamSynchronize(s->user));
        int rc = grow_neighbour_list(s);
        if (rc)
            return rc;
        h = rest;
    }
    if (h) {
        NP_CUDA(cudaMemsetAsync(s->d_flags, 0, sizeof(int), s->user));
        if (h & FLAG_NONFINITE)
            return set_err(NPSIM_ERR_NONFINITE, "a position became non-finite");
        if (h & FLAG_ESCAPED)
            return set_err(NPSIM_ERR_ESCAPED,
                           "an NP was farther than 2 max(R0, R(t)) from the droplet centre");
        return set_err(NPSIM_ERR_CUDA, "device error word 0x%x", h);
    }
    return NPSIM_OK;
}

// Pick the all-pairs launch shape (and, for the grouped kernels, the ranges
// per CTA): time each candidate on the current positions, together with the
// integrator's sum over its partial slots (more ranges mean more slots per
// row: the all-pairs launch can gain less than the sum loses).
int autotune(npsim_sim *s)
{
    const bool lj = s->ap_lj;
    const int nc = shape_count();
    // NPSIM_AUTOTUNE=0 takes the first shape; NPSIM_AUTOTUNE=1:<index>[:<ranges per
    // CTA>] forces one (ignored if that shape cannot run this sum); neither
    // touches the cache.
    const char *env = getenv("NPSIM_AUTOTUNE");
    if (env && env[0] == '0') {
        s->ap_idx = 0;
        s->ap_per_cta = kDefaultRangesPerCta;
        return NPSIM_OK;
    }
    if (env && env[0] == '1' && env[1] == ':') {
        const int idx = atoi(env + 2);
        const char *m = strchr(env + 2, ':');
        if (idx >= 0 && idx < nc && shape_occupancy(s, idx, lj) > 0) {
            s->ap_idx = idx;
            s->ap_per_cta = m ? std::max(1, atoi(m + 1)) : kDefaultRangesPerCta;
            return NPSIM_OK;
        }
    }
    const std::array<long long, 4> key{s->n, lj ? 1 : 0, s->grp_len,
                                       s->P.sum_neutral ? 0 : 1};
    {
        std::lock_guard<std::mutex> g(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            s->ap_idx = it->second.first;
            s->ap_per_cta = it->second.second;
            return NPSIM_OK;
        }
    }
    const int n_m = (int)(sizeof(kRangesPerCta) / sizeof(kRangesPerCta[0]));
    int best = 0, best_m = kDefaultRangesPerCta;
    bool all = true;
    {
        const size_t out_floats = 8 * (size_t)std::max(s->n, s->grp_len);
        float *tmp = nullptr;
        size_t need = 0;
        std::vector<size_t> needs;
        for (int c = 0; c < nc; ++c) {
            const int occ = shape_occupancy(s, c, lj);
            if (occ <= 0)
                continue;
            StreamK sk;
            shape_streamk(s, c, occ * s->sms, kRangesPerCta[n_m - 1], sk);
            needs.push_back((shape_slots_floats(sk) + 3) & ~(size_t)3); // 16-byte records follow
        }
        int rc = alloc_tune_scratch(needs, out_floats, &tmp, &need, &all);
        if (rc)
            return rc;
        float *sum_out = tmp + need;
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        float best_ms = 1e30f;
        const bool coul = s->P.coulomb == 1;
        const bool log = getenv("NPSIM_AUTOTUNE_LOG") != nullptr; // per-shape times to stderr
        for (int c = 0; c < nc; ++c) {
            const int occ = shape_occupancy(s, c, lj);
            // for the full sum of neutral NPs the LJ + Coulomb kernels have only their
            // dearer sweep (no charge product to take as the unit of the sums)
            if (occ <= 0 || (s->P.sum_neutral && !lj && shape_ljg(c)))
                continue;
            if (!lj && shape_family(c) == SF_SYM && shape_config(c).ki > 4 &&
                s->grp_len <= kSymLongRows)
                continue;
            for (int mi = 0; mi < (shape_grouped(c) ? n_m : 1); ++mi) {
                const int m = shape_grouped(c) ? kRangesPerCta[mi] : 1;
                StreamK sk;
                shape_streamk(s, c, occ * s->sms, m, sk);
                if (shape_grouped(c) && mi > 0 && sk.grid == sk.ctas)
                    break; // no more ranges than CTAs: the same launch as m = 1
                if (shape_slots_floats(sk) > need)
                    break; // the scratch did not fit
                if (shape_launch(s, c, lj, coul, sk, tmp, s->user) != cudaSuccess ||
                    shape_sum(s, c, sk, tmp, sum_out, s->user) != cudaSuccess)
                    continue;
                const int reps = s->n > 100000 ? 2 : 5;
                cudaEventRecord(e0, s->user);
                for (int r = 0; r < reps; ++r) {
                    shape_launch(s, c, lj, coul, sk, tmp, s->user);
                    shape_sum(s, c, sk, tmp, sum_out, s->user);
                }
                cudaEventRecord(e1, s->user);
                if (cudaEventSynchronize(e1) != cudaSuccess)
                    continue;
                float ms = 0.f;
                cudaEventElapsedTime(&ms, e0, e1);
                if (log) {
                    const ApConfig cf = shape_config(c);
                    fprintf(stderr,
                            "npsim autotune n=%d shape %d <%d,%d,%d> grid %d ranges %d: "
                            "%.4f ms\n",
                            s->n, c, cf.block, cf.ki, cf.jt, sk.ctas > 0 ? sk.ctas : sk.grid,
                            sk.grid, ms / reps);
                }
                if (ms < best_ms) {
                    best_ms = ms;
                    best = c;
                    best_m = m;
                }
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        cudaFree(tmp);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess)
            return set_err(NPSIM_ERR_CUDA, "autotune: %s", cudaGetErrorString(e));
    }
    s->ap_idx = best;
    s->ap_per_cta = best_m;
    if (all) { // the best of what memory was free is not kept for later simulations
        std::lock_guard<std::mutex> g(g_tune_mu);
        g_tune_cache[key] = std::make_pair(best, best_m);
    }
    return NPSIM_OK;
}

// Spatially compact order of the particles `idx` (AoS positions x): a k-d tree
// whose cuts halve a range across the longest side of its bounding box at a whole
// number of blocks, so that every aligned run of 64, 128 or 256 positions is one
// box of the tree, as compact as its count allows.  The pair kernels choose
// between the LJ and the Coulomb-only sweep by the boxes of 64 partners and of a
// warp's rows (64 to 256): along the Z-order curve, whose runs jump, the boxes of
// 256 rows and 64 partners of a dilute 16384-NP droplet lie within the LJ cutoff
// for 35 % of the pairs of boxes, here for 17 % (60000 NPs: 13 and 5 %).
struct KdPoint {
    float c[3];
    int i;
};

template <int AX> void kd_cut(KdPoint *p, size_t half, size_t n)
{
    // ties by index: the halves are functions of the positions alone
    std::nth_element(p, p + half, p + n, [](const KdPoint &u, const KdPoint &v) {
        return u.c[AX] < v.c[AX] || (u.c[AX] == v.c[AX] && u.i < v.i);
    });
}

// lo, hi: a box that holds the points (cut along, not measured again)
void kd_order(KdPoint *p, size_t n, std::array<float, 3> lo, std::array<float, 3> hi)
{
    constexpr size_t kLeaf = 64, kBlock = 256;
    while (n > kLeaf) {
        int ax = 0;
        for (int d = 1; d < 3; ++d)
            if (hi[d] - lo[d] > hi[ax] - lo[ax])
                ax = d;
        // the cut: the multiple of b nearest the middle, b the largest of 64, 128,
        // 256 that leaves something on both sides
        size_t b = kLeaf;
        while (b < kBlock && 2 * b < n)
            b *= 2;
        const size_t half = std::max<size_t>(1, (n / 2 + b / 2) / b) * b;
        if (ax == 0)
            kd_cut<0>(p, half, n);
        else if (ax == 1)
            kd_cut<1>(p, half, n);
        else
            kd_cut<2>(p, half, n);
        const float cut = p[half].c[ax];
        std::array<float, 3> left_hi = hi;
        left_hi[ax] = cut;
        kd_order(p, half, lo, left_hi);
        lo[ax] = cut;
        p += half;
        n -= half;
    }
}

void spatial_sort(std::vector<int> &idx, const double *x)
{
    std::vector<KdPoint> p(idx.size());
    std::array<float, 3> lo{INFINITY, INFINITY, INFINITY}, hi{-INFINITY, -INFINITY, -INFINITY};
    for (size_t k = 0; k < idx.size(); ++k) {
        const double *c = x + 3 * (size_t)idx[k];
        for (int d = 0; d < 3; ++d) { // any place will do for what has none
            const float v = (float)c[d];
            p[k].c[d] = std::isfinite(v) ? v : 0.0f;
            lo[d] = std::min(lo[d], p[k].c[d]);
            hi[d] = std::max(hi[d], p[k].c[d]);
        }
        p[k].i = idx[k];
    }
    kd_order(p.data(), p.size(), lo, hi);
    for (size_t k = 0; k < idx.size(); ++k)
        idx[k] = p[k].i;
}

// Type-grouped order: the charged types first (in type order), then the
// neutral ones; inside a group NPs follow a spatially compact order of their
// positions at creation when LJ is in the pair sum (tiles of nearby NPs let the LJ kernel
// skip tile pairs beyond the cutoff), else their index order; every group is
// padded with -1 to a multiple of 512, so each
// 256-position block has one type (and one charge).  Unless sum_neutral is
// set, and with no LJ in the pair sum, the grouped kernels cover only the
// charged groups and neutral NPs have no pair row (their Coulomb terms are
// exactly zero).
int build_grouping(npsim_sim *s, const int32_t *type, const double *x0, const int32_t *rank)
{
    std::vector<int> order;
    for (int t = 0; t < s->T; ++t)
        if (s->types[t].charge != 0.0)
            order.push_back(t);
    const int n_charged_types = (int)order.size();
    for (int t = 0; t < s->T; ++t)
        if (s->types[t].charge == 0.0)
            order.push_back(t);
    std::vector<std::vector<int>> members(s->T);
    for (int i = 0; i < s->n; ++i)
        members[type[i]].push_back(i);
    for (auto &m : members) {
        if (rank) // an order saved with a checkpoint: resume in the same summation order
            std::stable_sort(m.begin(), m.end(), [&](int a, int b) { return rank[a] < rank[b]; });
        else if (s->P.lj_mode == 1) // LJ in the pair sum: spatially compact tiles
            spatial_sort(m, x0);
        // Coulomb only: index order keeps the integrator's partial reads coalesced
    }
    std::vector<int> perm, tb;
    std::vector<float> qb;
    std::vector<int> pos(s->n, -1);
    int charged_len = 0;
    for (int g = 0; g < (int)order.size(); ++g) {
        const int t = order[g];
        if (members[t].empty())
            continue;
        for (int i : members[t]) {
            pos[i] = (int)perm.size();
            perm.push_back(i);
        }
        while (perm.size() % 512)
            perm.push_back(-1);
        while (qb.size() < perm.size() / 256) {
            qb.push_back((float)s->types[t].charge);
            tb.push_back(t);
        }
        if (g < n_charged_types)
            charged_len = (int)perm.size();
    }
    s->n_perm = (int)perm.size();
    s->h_rank.assign(pos.begin(), pos.end());
    const bool skip = !s->P.sum_neutral && s->P.lj_mode != 1;
    if (skip) {
        s->grp_len = charged_len;
        for (int i = 0; i < s->n; ++i)
            if (s->types[type[i]].charge == 0.0)
                pos[i] = -1;
    } else {
        s->grp_len = s->n_perm;
    }
    NP_CUDA(dalloc(&s->perm, perm.size()));
    NP_CUDA(dalloc(&s->qblk, qb.size()));
    NP_CUDA(dalloc(&s->tblk, tb.size()));
    NP_CUDA(dalloc(&s->row_pos, (size_t)s->n));
    NP_CUDA(cudaMemcpy(s->perm, perm.data(), sizeof(int) * perm.size(), cudaMemcpyHostToDevice));
    NP_CUDA(cudaMemcpy(s->qblk, qb.data(), sizeof(float) * qb.size(), cudaMemcpyHostToDevice));
    NP_CUDA(cudaMemcpy(s->tblk, tb.data(), sizeof(int) * tb.size(), cudaMemcpyHostToDevice));
    NP_CUDA(cudaMemcpy(s->row_pos, pos.data(), sizeof(int) * pos.size(),
                       cudaMemcpyHostToDevice));
    return NPSIM_OK;
}

void to_soa(const double *aos, int n, std::vector<double> &soa)
{
    soa.resize(3 * (size_t)n);
    for (int i = 0; i < n; ++i)
        for (int d = 0; d < 3; ++d)
            soa[(size_t)d * n + i] = aos[3 * (size_t)i + d];
}

// Device-side AoS float64 copies of the requested parts of the state of n NPs (any
// pointer NULL) in `stage` (9 n doubles), then the copies to the host arrays --
// one for parts that lie back to back on both sides -- on the stream, waited for.
int state_to_host(const float4 *xq, const float *x_lo, const float *vel, const float *F_src, int n,
                  size_t ld, double *stage, double *x, double *v, double *F, cudaStream_t st)
{
    const size_t n3 = 3 * (size_t)n;
    double *dx = x ? stage : nullptr, *dv = v ? stage + n3 : nullptr,
           *dF = F ? stage + 2 * n3 : nullptr;
    NP_CUDA(launch_state_aos(xq, x_lo, vel, F_src, n, ld, dx, dv, dF, st));
    cudaError_t e = cudaErrorInvalidValue;
    if (x && v == x + n3 && F == v + n3)
        e = copy_joined(x, dx, sizeof(double) * 3 * n3, st);
    if (e != cudaErrorInvalidValue) {
        NP_CUDA(e);
    } else {
        if (x)
            NP_CUDA(cudaMemcpyAsync(x, dx, sizeof(double) * n3, cudaMemcpyDeviceToHost, st));
        if (v)
            NP_CUDA(cudaMemcpyAsync(v, dv, sizeof(double) * n3, cudaMemcpyDeviceToHost, st));
        if (F)
            NP_CUDA(cudaMemcpyAsync(F, dF, sizeof(double) * n3, cudaMemcpyDeviceToHost, st));
    }
    NP_CUDA(cudaStreamSynchronize(st));
    return NPSIM_OK;
}

int copy_state_out(npsim_sim *s, const float *F_src, double *x, double *v, double *F)
{
    if (!s->stage)
        NP_CUDA(dalloc(&s->stage, 9 * (size_t)s->n));
    return state_to_host(s->xq, s->x_lo, s->v, F_src, s->n, (size_t)s->n, s->stage, x, v, F, s->user);
}

// Host float64 SoA -> device float32 (rounded to nearest).
int put_f32(const std::vector<double> &src, float *d, cudaStream_t st)
{
    std::vector<float> h(src.begin(), src.end());
    NP_CUDA(cudaMemcpyAsync(d, h.data(), sizeof(float) * h.size(), cudaMemcpyHostToDevice, st));
    NP_CUDA(cudaStreamSynchronize(st));
    return NPSIM_OK;
}

// Positions in float64 (hi + lo of every coordinate) into s->x.
int positions_f64(npsim_sim *s)
{
    NP_CUDA(launch_positions_f64(s->xq, s->x_lo, s->n, s->x, s->user));
    return NPSIM_OK;
}

// Set the step counter and recompute the forces of the current state.
int finish_upload(npsim_sim *s, int64_t step, bool rebuild = true)
{
    if (rebuild) {
        int rc = set_gate(s, 1); // new positions: rebuild the lists at the next pass
        if (rc)
            return rc;
    }
    long long st = step;
    NP_CUDA(cudaMemcpyAsync(s->d_step, &st, sizeof(long long), cudaMemcpyHostToDevice,
                            s->user));
    float4 tab[NPSIM_MAX_TYPES] = {};
    for (int t = 0; t < s->T; ++t)
        tab[t] = spring_entry(s->P.R0, s->P.k_evap, s->P.dt, st, 0.5 * s->types[t].sigma);
    NP_CUDA(cudaMemcpyAsync(s->d_spring + (st & 1) * NPSIM_MAX_TYPES, tab, sizeof(tab),
                            cudaMemcpyHostToDevice, s->user));
    NP_CUDA(cudaStreamSynchronize(s->user)); // tab lives on this stack frame
    int rc = enqueue_pass(s, MODE_FORCES, true, true, true, s->F, s->user);
    if (rc)
        return rc;
    s->gate_open = false;
    NP_CUDA(cudaStreamSynchronize(s->user));
    s->step = step;
    return read_flags(s);
}

int upload_state(npsim_sim *s, const double *x, const double *v, int64_t step)
{
    std::vector<double> buf;
    to_soa(x, s->n, buf);
    NP_CUDA(cudaMemcpyAsync(s->x, buf.data(), sizeof(double) * buf.size(),
                            cudaMemcpyHostToDevice, s->user));
    NP_CUDA(cudaStreamSynchronize(s->user));
    if (v) {
        to_soa(v, s->n, buf);
        int rc = put_f32(buf, s->v, s->user);
        if (rc)
            return rc;
    } else {
        NP_CUDA(cudaMemsetAsync(s->v, 0, sizeof(float) * 3 * (size_t)s->n, s->user));
    }
    NP_CUDA(launch_mirror(s->x, s->typ, s->charge_f, s->n, s->xq, s->x_lo, s->user));
    return finish_upload(s, step);
}

// Replace the state by raw words (hi [3][n], lo [3][n], v [3][n], float32 SoA).
int upload_words(npsim_sim *s, const float *words, int64_t step)
{
    const size_t n = (size_t)s->n;
    std::vector<float4> xq(n);
    for (size_t i = 0; i < n; ++i)
        xq[i] = make_float4(words[i], words[n + i], words[2 * n + i],
                            s->charge_f[s->h_type[i]]);
    NP_CUDA(cudaStreamSynchronize(s->user));
    NP_CUDA(cudaMemcpy(s->xq, xq.data(), sizeof(float4) * n, cudaMemcpyHostToDevice));
    NP_CUDA(cudaMemcpy(s->x_lo, words + 3 * n, sizeof(float) * 3 * n, cudaMemcpyHostToDevice));
    NP_CUDA(cudaMemcpy(s->v, words + 6 * n, sizeof(float) * 3 * n, cudaMemcpyHostToDevice));
    return finish_upload(s, step);
}

// Per-type integrator coefficients (float64 on the host): BAOAB O-step factors
// c1 = exp(-gamma dt), sqrt((1 - c1^2) kT / m); overdamped mobility 1/(m gamma)
// and noise sqrt(2 kT dt / (m gamma)); C q for the Coulomb field.
void fill_coefs(const npsim_type_t *types, const npsim_params_t *params, TypeCoef *tc,
                float *charge_f)
{
    const double C = params->bjerrum;
    for (int t = 0; t < params->n_types; ++t) {
        const npsim_type_t &ty = types[t];
        TypeCoef &c = tc[t];
        c.mass = ty.mass;
        c.inv_mass = 1.0 / ty.mass;
        c.half_sigma = 0.5 * ty.sigma;
        c.k_wall = ty.k_wall;
        c.c1 = std::exp(-ty.gamma * params->dt);
        c.sd_o = std::sqrt((1.0 - c.c1 * c.c1) * params->kT / ty.mass);
        c.mob = ty.gamma > 0 ? 1.0 / (ty.mass * ty.gamma) : 0.0;
        c.sd_bd = std::sqrt(2.0 * params->kT * params->dt * c.mob);
        c.charge_c = C * ty.charge;
        c.hdt_m = (float)(0.5 * params->dt / ty.mass);
        c.c1f = (float)c.c1;
        c.c1lo = (float)(c.c1 - (double)c.c1f);
        c.sd_of = (float)c.sd_o;
        c.dt_mob = (float)(params->dt * c.mob);
        c.sd_bdf = (float)c.sd_bd;
        c.qc = (float)c.charge_c;
        c.mg = (float)(ty.mass * params->g);
        c.mw2 = (float)(ty.mass * params->omega * params->omega);
        c.kw = (float)ty.k_wall;
        c.hs = (float)c.half_sigma;
        c.dt_m = (float)(params->dt / ty.mass);
        c.gdt = (float)(ty.gamma * params->dt);
        c.kick = (float)params->v_kick;
        if (charge_f)
            charge_f[t] = (float)ty.charge;
    }
}

// Type-pair tables (sigma_ab^2, 24 eps_ab, rc_ab^2, C q_a q_b) with Lorentz-Berthelot
// mixing unless eps_ov (T x T) is given; tl is the same with the Coulomb column 0.
// Returns the largest cutoff.
double fill_tabs(const npsim_type_t *types, const npsim_params_t *params, const double *eps_ov,
                 PairTab *tf, PairTab *tl)
{
    const int T = params->n_types;
    const double C = params->bjerrum;
    double rc_max = 0.0;
    for (int a = 0; a < T; ++a)
        for (int b = 0; b < T; ++b) {
            const double sig = 0.5 * (types[a].sigma + types[b].sigma);
            const double eps = eps_ov ? eps_ov[a * T + b] : std::sqrt(types[a].eps * types[b].eps);
            const double rc = params->lj_cut * sig;
            rc_max = std::max(rc_max, rc);
            const float4 e = make_float4(
                (float)(sig * sig), (float)(24.0 * eps), (float)(rc * rc),
                (float)(params->coulomb ? C * types[a].charge * types[b].charge : 0.0));
            tf->e[a * NPSIM_MAX_TYPES + b] = e;
            if (tl)
                tl->e[a * NPSIM_MAX_TYPES + b] = make_float4(e.x, e.y, e.z, 0.0f);
        }
    return rc_max;
}

int validate(const npsim_type_t *types, const npsim_params_t *p, int64_t n)
{
    NP_REQUIRE(types && p, "types and params are required");
    NP_REQUIRE(n >= 1 && n <= (1ll << 29), "n = %lld out of range [1, 2^29]", (long long)n);
    NP_REQUIRE(p->n_types >= 1 && p->n_types <= NPSIM_MAX_TYPES, "n_types = %d",
               p->n_types);
    NP_REQUIRE(p->dt > 0 && std::isfinite(p->dt), "dt must be positive");
    NP_REQUIRE(p->kT >= 0, "kT must be >= 0");
    NP_REQUIRE(p->rot_mode >= 0 && p->rot_mode <= 2, "rot_mode must be 0, 1 or 2");
    NP_REQUIRE(p->lj_mode >= 0 && p->lj_mode <= 2, "lj_mode must be 0, 1 or 2");
    NP_REQUIRE(p->integrator >= 0 && p->integrator <= 2, "integrator must be 0, 1 or 2");
    NP_REQUIRE(p->wall >= 0 && p->wall <= 2, "wall must be 0, 1 or 2");
    NP_REQUIRE(p->coulomb >= 0 && p->coulomb <= 2, "coulomb must be 0, 1 or 2");
    NP_REQUIRE(p->coulomb != 2 || p->lj_mode == 2,
               "coulomb 2 (truncated, through the cell list) needs lj_mode 2");
    NP_REQUIRE(p->coulomb != 2 || (p->coulomb_cut > 0 && std::isfinite(p->coulomb_cut)),
               "coulomb 2 needs coulomb_cut > 0");
    NP_REQUIRE(p->R0 > 0 || !p->wall, "R0 must be positive when the wall is on");
    NP_REQUIRE(p->integrator != 2 || (p->v_kick >= 0 && std::isfinite(p->v_kick)),
               "v_kick must be finite and >= 0");
    NP_REQUIRE(p->lj_mode == 0 || p->lj_cut > 0, "lj_cut must be positive");
    for (int t = 0; t < p->n_types; ++t) {
        NP_REQUIRE(types[t].sigma > 0 && types[t].mass > 0, "type %d: sigma, mass > 0", t);
        NP_REQUIRE(types[t].gamma >= 0 && types[t].eps >= 0 && types[t].k_wall >= 0,
                   "type %d: gamma, eps, k_wall >= 0", t);
        NP_REQUIRE(p->integrator != 1 || types[t].gamma > 0,
                   "type %d: the overdamped integrator needs gamma > 0", t);
    }
    return NPSIM_OK;
}

} // namespace

extern "C" {

const char *npsim_last_error(void) { return g_err.c_str(); }

int npsim_device_info(int *sm_count, int *clock_khz, int *cc_major, int *cc_minor)
{
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || count < 1)
        return set_err(NPSIM_ERR_NO_DEVICE, "no CUDA device visible");
    int dev = 0;
    NP_CUDA(cudaGetDevice(&dev));
    if (sm_count)
        NP_CUDA(cudaDeviceGetAttribute(sm_count, cudaDevAttrMultiProcessorCount, dev));
    if (clock_khz)
        NP_CUDA(cudaDeviceGetAttribute(clock_khz, cudaDevAttrClockRate, dev));
    if (cc_major)
        NP_CUDA(cudaDeviceGetAttribute(cc_major, cudaDevAttrComputeCapabilityMajor, dev));
    if (cc_minor)
        NP_CUDA(cudaDeviceGetAttribute(cc_minor, cudaDevAttrComputeCapabilityMinor, dev));
    return NPSIM_OK;
}

} // extern "C"

namespace {

// npsim_create with an optional saved grouping order (rank, n entries: the
// order of each NP inside its type group, from a checkpoint).
int create_impl(const npsim_type_t *types, const npsim_params_t *params, int64_t n,
                const double *x0, const double *v0, const int32_t *type, void *stream,
                const int32_t *rank, npsim_sim_t *out)
{
    if (!out)
        return set_err(NPSIM_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    int rc = validate(types, params, n);
    if (rc)
        return rc;
    NP_REQUIRE(x0 && type, "x0 and type are required");
    int sms = 0;
    rc = check_device(&sms);
    if (rc)
        return rc;
    for (int64_t i = 0; i < n; ++i) {
        NP_REQUIRE(type[i] >= 0 && type[i] < params->n_types, "type[%lld] = %d out of range",
                   (long long)i, type[i]);
        NP_REQUIRE(std::isfinite(x0[3 * i]) && std::isfinite(x0[3 * i + 1]) &&
                       std::isfinite(x0[3 * i + 2]),
                   "x0[%lld] is not finite", (long long)i);
    }

    npsim_sim *s = new npsim_sim();
    s->n = (int)n;
    s->T = params->n_types;
    s->sms = sms;
    s->P = *params;
    for (int t = 0; t < s->T; ++t)
        s->types[t] = types[t];
    if (params->eps_override) {
        s->has_ov = true;
        for (int k = 0; k < s->T * s->T; ++k)
            s->eps_ov[k] = params->eps_override[k];
    }
    s->P.eps_override = nullptr;
    s->h_type.assign(type, type + n);
    s->user = (cudaStream_t)stream;

    auto bail = [&](int code) {
        delete s;
        return code;
    };
    cudaError_t ce = cudaStreamCreateWithFlags(&s->cap, cudaStreamNonBlocking);
    if (ce != cudaSuccess)
        return bail(set_err(NPSIM_ERR_CUDA, "stream create: %s", cudaGetErrorString(ce)));

    // per-type coefficients and pair tables (float64 on the host)
    std::vector<long long> tcount(s->T, 0);
    for (int64_t i = 0; i < n; ++i)
        tcount[type[i]]++;
    double dsum = 0.0;
    for (int t = 0; t < s->T; ++t)
        dsum += (double)tcount[t] * types[t].sigma;
    s->d_mean = dsum / (double)n;

    StepParams &sp = s->sp;
    sp.n = s->n;
    sp.n_types = s->T;
    sp.rot_mode = params->rot_mode;
    sp.wall = params->wall;
    sp.integrator = params->integrator;
    sp.seed = params->seed;
    sp.dt = params->dt;
    sp.R0 = params->R0;
    sp.k_evap = params->k_evap;
    sp.g = params->g;
    sp.omega2 = params->omega * params->omega;
    fill_coefs(types, params, sp.tc, s->charge_f);
    PairTab tf{}, tl{}, tc{};
    const double rc_max = fill_tabs(types, params, s->has_ov ? s->eps_ov : nullptr, &tf, &tl);
    for (int k = 0; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; ++k) { // Coulomb only: no LJ pair in range
        tc.e[k] = make_float4(0.0f, 0.0f, 0.0f, tf.e[k].w);
        if (params->lj_mode != 0 && tf.e[k].y != 0.0f)
            s->rc2_lim = std::max(s->rc2_lim, tf.e[k].z * 1.0001f);
        if (tf.e[k].w != 0.0f)
            s->any_charge = 1;
    }

#define BAIL_CUDA(call)                                                                 \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return bail(set_err(e_ == cudaErrorMemoryAllocation ? NPSIM_ERR_OOM         \
                                                                 : NPSIM_ERR_CUDA,      \
                                "%s failed: %s", #call, cudaGetErrorString(e_)));       \
    } while (0)

    const size_t n3 = 3 * (size_t)n;
    BAIL_CUDA(dalloc(&s->x, n3));
    BAIL_CUDA(dalloc(&s->x_lo, n3));
    BAIL_CUDA(dalloc(&s->v, n3));
    BAIL_CUDA(dalloc(&s->F, 2 * n3));
    BAIL_CUDA(dalloc(&s->F_tmp, 2 * n3));
    BAIL_CUDA(dalloc(&s->xq, (size_t)n));
    BAIL_CUDA(dalloc(&s->typ, (size_t)n));
    BAIL_CUDA(dalloc(&s->tab_full, 1));
    BAIL_CUDA(dalloc(&s->tab_lj, 1));
    BAIL_CUDA(dalloc(&s->tab_coul, 1));
    BAIL_CUDA(dalloc(&s->d_step, 1));
    BAIL_CUDA(dalloc(&s->d_spring, 2 * NPSIM_MAX_TYPES));
    BAIL_CUDA(cudaMemsetAsync(s->d_spring, 0, sizeof(float4) * 2 * NPSIM_MAX_TYPES, s->user));
    BAIL_CUDA(dalloc(&s->d_flags, 1));
    BAIL_CUDA(dalloc(&s->d_done, 1));
    BAIL_CUDA(cudaMemsetAsync(s->d_flags, 0, sizeof(int), s->user));
    BAIL_CUDA(cudaMemsetAsync(s->d_done, 0, sizeof(unsigned), s->user));
    BAIL_CUDA(cudaMemcpyAsync(s->tab_full, &tf, sizeof(PairTab), cudaMemcpyHostToDevice,
                              s->user));
    BAIL_CUDA(cudaMemcpyAsync(s->tab_lj, &tl, sizeof(PairTab), cudaMemcpyHostToDevice,
                              s->user));
    BAIL_CUDA(cudaMemcpyAsync(s->tab_coul, &tc, sizeof(PairTab), cudaMemcpyHostToDevice,
                              s->user));
    BAIL_CUDA(cudaMemcpyAsync(s->typ, type, sizeof(int) * (size_t)n, cudaMemcpyHostToDevice,
                              s->user));
    BAIL_CUDA(cudaStreamSynchronize(s->user));

    s->cell = params->lj_mode == 2;
    double rc_cell = rc_max; // largest cutoff of the cell-list terms
    if (params->coulomb == 2) {
        // truncated Coulomb: cutoff coulomb_cut * sigma_ab for every charged pair
        float rcc2[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES] = {};
        const int T = params->n_types;
        for (int a = 0; a < T; ++a)
            for (int b = 0; b < T; ++b) {
                if (types[a].charge == 0.0 || types[b].charge == 0.0)
                    continue;
                const double rcc = params->coulomb_cut * 0.5 * (types[a].sigma + types[b].sigma);
                rcc2[a * NPSIM_MAX_TYPES + b] = (float)(rcc * rcc);
                rc_cell = std::max(rc_cell, rcc);
            }
        BAIL_CUDA(dalloc(&s->d_rcc2, (size_t)NPSIM_MAX_TYPES * NPSIM_MAX_TYPES));
        BAIL_CUDA(cudaMemcpy(s->d_rcc2, rcc2, sizeof(rcc2), cudaMemcpyHostToDevice));
    }
    if (s->cell) {
        double L = params->R0;
        for (int64_t i = 0; i < 3 * n; ++i)
            L = std::max(L, std::fabs(x0[i]));
        L += rc_cell + kSkin;
        // cell edge: the smallest list radius of the acting type pairs (each pair
        // scans as many cells as its own radius needs), the sort keys (types x
        // cells) capped at about two per NP, so that the cell ranges stay in L2
        // (the edge grows until the grid fits)
        float rcc2h[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES] = {};
        if (s->d_rcc2)
            BAIL_CUDA(cudaMemcpy(rcc2h, s->d_rcc2, sizeof(rcc2h), cudaMemcpyDeviceToHost));
        list_radii(tf, s->d_rcc2 ? rcc2h : nullptr, kSkin, s->rlist);
        double h_min = rc_cell + kSkin;
        for (int a = 0; a < s->T; ++a)
            for (int b = 0; b < s->T; ++b)
                if (s->rlist[a * NPSIM_MAX_TYPES + b] > 0.0)
                    h_min = std::min(h_min, s->rlist[a * NPSIM_MAX_TYPES + b]);
        s->cell_h_min = h_min;
        s->cell_rc = rc_cell;
        s->grid = lj_grid(s, L);
        rc = ensure_cells(s, s->grid);
        if (rc)
            return bail(rc);
        BAIL_CUDA(dalloc(&s->F_lj, 8 * (size_t)n)); // one 32-byte record per NP
        s->nl.cap = 32; // grown after the first build if some NP has more partners
        BAIL_CUDA(dalloc(&s->nl.nbr, (size_t)s->nl.cap * n));
        BAIL_CUDA(dalloc(&s->nl.nnbr, (size_t)n));
        BAIL_CUDA(dalloc(&s->nl.x_ref, (size_t)n));
        BAIL_CUDA(dalloc(&s->nl.builds, 1));
        BAIL_CUDA(cudaMemsetAsync(s->nl.builds, 0, sizeof(unsigned long long), s->user));
        BAIL_CUDA(dalloc(&s->d_gate, 1));
        s->fused_cap = list_steps_capacity();
        BAIL_CUDA(dalloc(&s->list_bar, kBarWords));
        BAIL_CUDA(cudaMemsetAsync(s->list_bar, 0, kBarWords * sizeof(unsigned), s->user));
        BAIL_CUDA(cudaMemsetAsync(s->nl.nnbr, 0, sizeof(int) * (size_t)n, s->user));
        BAIL_CUDA(cudaMemsetAsync(s->nl.nbr, 0, sizeof(unsigned) * (size_t)s->nl.cap * n, s->user));
    }
    if (s->cell) {
        rc = set_list_wait(s, list_wait_polls(s->n));
        if (rc)
            return bail(rc);
    }
    s->ap_lj = params->lj_mode == 1;
    s->ap = params->coulomb == 1 || s->ap_lj;

    // positions for the mirror (needed before tuning)
    {
        std::vector<double> buf;
        to_soa(x0, s->n, buf);
        BAIL_CUDA(cudaMemcpy(s->x, buf.data(), sizeof(double) * n3, cudaMemcpyHostToDevice));
        BAIL_CUDA(launch_mirror(s->x, s->typ, s->charge_f, s->n, s->xq, s->x_lo, s->user));
    }
    if (s->ap) {
        rc = build_grouping(s, type, x0, rank);
        if (rc)
            return bail(rc);
        BAIL_CUDA(dalloc(&s->ap_work, 2));
        BAIL_CUDA(cudaMemsetAsync(s->ap_work, 0, 2 * sizeof(unsigned), s->user));
        rc = autotune(s);
        if (rc)
            return bail(rc);
        int occ = std::max(1, shape_occupancy(s, s->ap_idx, s->ap_lj));
        shape_streamk(s, s->ap_idx, occ * s->sms, s->ap_per_cta, s->sk);
        ce = dalloc(&s->slots, shape_slots_floats(s->sk));
        if (ce == cudaSuccess && s->sk.tri)
            ce = dalloc(&s->F_pair, 8 * (size_t)n);
        if (ce == cudaErrorMemoryAllocation && s->sk.tri) {
            // no room for the column partials: a one-sided shape, whose scratch
            // grows with N only
            cudaGetLastError();
            dfree(s->slots);
            s->ap_idx = 0;
            while (shape_family(s->ap_idx) != (s->ap_lj ? SF_LJG : SF_GRP))
                ++s->ap_idx;
            occ = std::max(1, shape_occupancy(s, s->ap_idx, s->ap_lj));
            shape_streamk(s, s->ap_idx, occ * s->sms, s->ap_per_cta, s->sk);
            ce = dalloc(&s->slots, shape_slots_floats(s->sk));
        }
        BAIL_CUDA(ce);
    } else {
        s->sk = StreamK{};
        s->sk.itile = 1;
        s->sk.n_jt = 1;
        s->sk.grid = 1;
        s->sk.W = 1;
    }
#undef BAIL_CUDA
    rc = upload_state(s, x0, v0, 0);
    if (rc)
        return bail(rc);
    *out = s;
    return NPSIM_OK;
}

} // namespace

extern "C" {

int npsim_create(const npsim_type_t *types, const npsim_params_t *params, int64_t n,
                 const double *x0, const double *v0, const int32_t *type, void *stream,
                 npsim_sim_t *out)
{
    NP_TRACE();
    return create_impl(types, params, n, x0, v0, type, stream, nullptr, out);
}

void npsim_destroy(npsim_sim_t sim)
{
    NP_TRACE();
    if (!sim)
        return;
    cudaStreamSynchronize(sim->user);
    delete sim;
}

} // extern "C"

namespace {
// Queue n_steps steps as graph chunks of at most kChunk steps (no host wait).
// The LJ cell grid follows the droplet.  With the interface spring on, the NPs
// stay within about R(t) of the centre; at every step that is a multiple of
// kRegridPeriod the grid's half-width L is compared with R(t) plus the largest
// cutoff and the skin, and when that differs from L by more than a quarter
// (the droplet has shrunk or grown) a new grid replaces the old one: the cell
// buffers are resized if needed, the lists are rebuilt at the next pass and
// the step graphs are captured again.  The decision depends on the step count
// alone, and the steps are cut at those multiples whatever the calls' sizes,
// so runs stay bit-reproducible (npsim_step(37) = 5 + 16 + 1 + 15 steps).
constexpr int64_t kRegridPeriod = 1024;

// Only the spring on every NP beyond its equilibrium point (wall 1) keeps the
// NPs inside R(t); without a spring or with the band-only one they may leave.
bool follows_droplet(const npsim_sim *s) { return s->cell && s->P.wall == 1; }

int regrid_if_needed(npsim_sim *s)
{
    if (!follows_droplet(s) || s->step % kRegridPeriod != 0)
        return NPSIM_OK;
    const double t = (double)s->step * s->P.dt;
    const double R2 = s->P.R0 * s->P.R0 - s->P.k_evap * t;
    const double R = R2 > 0.0 ? std::sqrt(R2) : 0.0;
    const double L_want = std::max(R, 1.0) + s->cell_rc + kSkin;
    const double L = (double)s->grid.L;
    if (L_want >= 0.75 * L && L_want <= L)
        return NPSIM_OK;
    NP_CUDA(cudaStreamSynchronize(s->user)); // nothing of the old grid in flight
    CellGrid g = lj_grid(s, L_want);
    int rc = ensure_cells(s, g);
    if (rc)
        return rc;
    s->grid = g;
    for (auto &e : s->graphs)
        cudaGraphExecDestroy(e.second);
    s->graphs.clear();
    return set_gate(s, 1);
}

// Small droplets whose pair forces all come from the lists take many steps per
// launch (not while the kernels are timed apart).
bool fused_steps(const npsim_sim *s)
{
    return s->cell && !s->ap && s->n <= s->fused_cap && !s->profiling;
}

// No pair force at all: every NP's steps are its own.
bool free_steps(const npsim_sim *s) { return !s->cell && !s->ap && !s->profiling; }

int enqueue_free(npsim_sim *s, int k)
{
    IntArgs a{};
    a.x_lo = s->x_lo;
    a.v = s->v;
    a.F = s->F;
    a.typ = s->typ;
    a.xq = s->xq;
    a.spring = s->d_spring;
    a.step = s->d_step;
    a.flags = s->d_flags;
    a.done = s->d_done;
    NP_CUDA(launch_free_steps(a, s->sp, k, s->user));
    return NPSIM_OK;
}

int enqueue_fused(npsim_sim *s, int k)
{
    if (!s->sxq2) {
        NP_CUDA(dalloc(&s->sxq2, (size_t)s->n + 1));
        const float4 far = make_float4(kPairPad, kPairPad, kPairPad, 0.0f);
        NP_CUDA(cudaMemcpyAsync(s->sxq2 + s->n, &far, sizeof(far), cudaMemcpyHostToDevice, s->user));
        NP_CUDA(cudaStreamSynchronize(s->user)); // far lives on this stack frame
    }
    IntArgs a{};
    a.x_lo = s->x_lo;
    a.v = s->v;
    a.F = s->F;
    a.typ = s->typ;
    a.xq = s->xq;
    a.spring = s->d_spring;
    a.x_ref = s->nl.x_ref;
    a.nbr_gate = s->d_gate;
    a.half_skin2 = kHalfSkin2;
    a.step = s->d_step;
    a.flags = s->d_flags;
    NP_CUDA(launch_list_steps(s->grid, s->cb, s->n, s->tab_full, s->d_rcc2, kSkin, s->nl,
                              s->list_bar, a, s->sp, s->sxq2, s->F_lj, k, s->user));
    return NPSIM_OK;
}

int enqueue_steps(npsim_sim *s, int64_t n_steps)
{
    int64_t rem = n_steps;
    if (rem > 0 && s->cell)
        s->flags_unread = true;
    while (rem > 0) {
        int rc0 = regrid_if_needed(s);
        if (rc0)
            return rc0;
        if (free_steps(s)) {
            const int k = (int)std::min<int64_t>(rem, kMaxFreeSteps);
            int rc = enqueue_free(s, k);
            if (rc)
                return rc;
            rem -= k;
            s->step += k;
            continue;
        }
        if (fused_steps(s)) {
            int k = (int)std::min<int64_t>(rem, kMaxFusedSteps);
            if (follows_droplet(s)) // stop at the next multiple of kRegridPeriod
                k = (int)std::min<int64_t>(k, kRegridPeriod - s->step % kRegridPeriod);
            int rc = enqueue_fused(s, k);
            if (rc)
                return rc;
            rem -= k;
            s->step += k;
            continue;
        }
        int k = (int)std::min<int64_t>(rem, kChunk);
        if (follows_droplet(s)) // stop at the next multiple of kRegridPeriod
            k = (int)std::min<int64_t>(k, kRegridPeriod - s->step % kRegridPeriod);
        cudaGraphExec_t ex = nullptr;
        int rc = get_graph(s, k, &ex);
        if (rc)
            return rc;
        NP_CUDA(cudaGraphLaunch(ex, s->user));
        s->last_chunk = k;
        rem -= k;
        s->step += k;
    }
    if (n_steps > 0)
        s->gate_open = false; // their last pass leaves the gate closed
    return NPSIM_OK;
}
} // namespace

extern "C" {

int npsim_step(npsim_sim_t s, int64_t n_steps)
{
    NP_TRACE();
    NP_REQUIRE(s, "sim is NULL");
    NP_REQUIRE(n_steps >= 0, "n_steps must be >= 0");
    int rc = enqueue_steps(s, n_steps);
    if (rc)
        return rc;
    return read_flags(s);
}

int npsim_step_record(npsim_sim_t s, int64_t n_steps, int64_t every, float *frames,
                      int64_t n_frames)
{
    NP_TRACE();
    NP_REQUIRE(s && frames, "sim and frames are required");
    NP_REQUIRE(n_steps >= 0 && every >= 1, "n_steps >= 0 and every >= 1 are required");
    const int64_t nf = n_steps / every;
    NP_REQUIRE(n_frames >= nf, "frames holds %lld frames, %lld are recorded",
               (long long)n_frames, (long long)nf);
    const size_t bytes = sizeof(float4) * (size_t)s->n;
    constexpr int R = npsim_sim::kRecSlots;
    if (!s->rec_ring) {
        NP_CUDA(dalloc(&s->rec_ring, (size_t)R * s->n));
        NP_CUDA(cudaStreamCreateWithFlags(&s->rec_stream, cudaStreamNonBlocking));
        for (int k = 0; k < R; ++k) {
            NP_CUDA(cudaEventCreateWithFlags(&s->rec_ready[k], cudaEventDisableTiming));
            NP_CUDA(cudaEventCreateWithFlags(&s->rec_done[k], cudaEventDisableTiming));
        }
    }
    // copies are asynchronous only into page-locked memory: register the
    // caller's buffer for the call unless it already is
    bool registered = false;
    if (nf > 0) {
        cudaPointerAttributes at{};
        const bool locked = cudaPointerGetAttributes(&at, frames) == cudaSuccess &&
                            at.type == cudaMemoryTypeHost;
        cudaGetLastError(); // a plain host pointer may leave an error behind
        if (!locked) {
            NP_CUDA(cudaHostRegister(frames, bytes * (size_t)nf, cudaHostRegisterDefault));
            registered = true;
        }
    }
    int rc = NPSIM_OK;
    cudaError_t e = cudaSuccess;
    for (int64_t f = 0; f < nf && rc == NPSIM_OK && e == cudaSuccess; ++f) {
        rc = enqueue_steps(s, every);
        if (rc)
            break;
        const int slot = (int)(f % R);
        if (f >= R) // the slot's previous frame has reached the host
            e = cudaStreamWaitEvent(s->user, s->rec_done[slot], 0);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(s->rec_ring + (size_t)slot * s->n, s->xq, bytes,
                                cudaMemcpyDeviceToDevice, s->user);
        if (e == cudaSuccess)
            e = cudaEventRecord(s->rec_ready[slot], s->user);
        if (e == cudaSuccess)
            e = cudaStreamWaitEvent(s->rec_stream, s->rec_ready[slot], 0);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(frames + (size_t)f * 4 * s->n, s->rec_ring + (size_t)slot * s->n,
                                bytes, cudaMemcpyDeviceToHost, s->rec_stream);
        if (e == cudaSuccess)
            e = cudaEventRecord(s->rec_done[slot], s->rec_stream);
    }
    if (rc == NPSIM_OK && e == cudaSuccess)
        rc = enqueue_steps(s, n_steps - nf * every);
    const cudaError_t e2 = cudaStreamSynchronize(s->rec_stream);
    if (registered)
        cudaHostUnregister(frames);
    if (rc)
        return rc;
    if (e != cudaSuccess || e2 != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "frame recorder: %s",
                       cudaGetErrorString(e != cudaSuccess ? e : e2));
    return read_flags(s);
}

int npsim_get_state(npsim_sim_t s, double *x, double *v, double *F, int64_t *step)
{
    NP_TRACE();
    NP_REQUIRE(s, "sim is NULL");
    if (x || v || F) {
        int rc = copy_state_out(s, s->F, x, v, F);
        if (rc)
            return rc;
    }
    if (step)
        *step = s->step;
    return NPSIM_OK;
}

int npsim_set_state(npsim_sim_t s, const double *x, const double *v, int64_t step)
{
    NP_REQUIRE(s && x, "sim and x are required");
    NP_REQUIRE(step >= 0, "step must be >= 0");
    return upload_state(s, x, v, step);
}

int npsim_forces(npsim_sim_t s, int what, double *F)
{
    NP_TRACE();
    NP_REQUIRE(s && F, "sim and F are required");
    NP_REQUIRE(what >= 0 && what <= 3, "what must be 0..3");
    const bool lj = what == 0 || what == 1 || what == 2;
    const bool coul = what == 0 || what == 1 || what == 3;
    // the lists are built in this pass only if the host has opened the gate; a build may
    // give up, and reading the flags takes 12 us
    const bool lists = s->cell && (lj || (coul && s->P.coulomb == 2));
    if (lists && s->gate_open)
        s->flags_unread = true;
    int rc = enqueue_pass(s, MODE_FORCES, lj, coul, what == 0, s->F_tmp, s->user);
    if (rc)
        return rc;
    if (lists)
        s->gate_open = false;
    rc = copy_state_out(s, s->F_tmp, nullptr, nullptr, F);
    return rc || !s->flags_unread ? rc : read_flags(s);
}

int npsim_test_list_wait(npsim_sim_t s, int64_t polls)
{
    NP_REQUIRE(s && s->cell, "a simulation with neighbour lists is required");
    NP_REQUIRE(polls >= -1 && polls <= 0xffffffffll, "polls must be -1 .. 2^32 - 1");
    return set_list_wait(s, polls < 0 ? list_wait_polls(s->n) : (unsigned)polls);
}

int npsim_positions_device(npsim_sim_t s, float *dev_xyzq)
{
    NP_REQUIRE(s && dev_xyzq, "sim and buffer are required");
    NP_CUDA(cudaMemcpyAsync(dev_xyzq, s->xq, sizeof(float4) * (size_t)s->n,
                            cudaMemcpyDeviceToDevice, s->user));
    return NPSIM_OK;
}

int npsim_allpairs_config(npsim_sim_t s, int *block, int *i_per_thread, int *j_tile,
                          int *grid, int *index, int *packed)
{
    NP_REQUIRE(s, "sim is NULL");
    const ApConfig c = shape_config(s->ap_idx);
    if (block)
        *block = s->ap ? c.block : 0;
    if (i_per_thread)
        *i_per_thread = s->ap ? c.ki : 0;
    if (j_tile)
        *j_tile = s->ap ? c.jt : 0;
    if (grid)
        *grid = !s->ap ? 0 : s->sk.ctas > 0 ? s->sk.ctas : s->sk.grid;
    if (index)
        *index = s->ap ? s->ap_idx : -1;
    if (packed)
        *packed = !s->ap                  ? 0
                  : shape_ljg(s->ap_idx)     ? 3
                  : shape_grouped(s->ap_idx) ? 2
                  : ap_packed(s->ap_idx)     ? 1
                                             : 0;
    return NPSIM_OK;
}

int npsim_allpairs_ranges(npsim_sim_t s, int *ranges)
{
    NP_REQUIRE(s && ranges, "sim and ranges are required");
    *ranges = s->ap ? s->sk.grid : 0;
    return NPSIM_OK;
}

int npsim_allpairs_num_configs(int *count)
{
    NP_REQUIRE(count, "count is NULL");
    *count = shape_count();
    return NPSIM_OK;
}

int npsim_launches_per_step(npsim_sim_t s, int *launches)
{
    NP_REQUIRE(s && launches, "sim and launches are required");
    // integrator, all-pairs (and the sum of its partials), the gated list build, the
    // list LJ forces; one launch where it takes many steps
    *launches = 1;
    if (!fused_steps(s) && !free_steps(s))
        *launches += (s->ap ? (s->sk.tri ? 2 : 1) : 0) + (s->cell ? 2 : 0);
    return NPSIM_OK;
}

int npsim_cell_grid(npsim_sim_t s, int *dim, int64_t *n_cells)
{
    NP_REQUIRE(s, "sim is NULL");
    if (dim)
        *dim = s->cell ? s->grid.dim : 0;
    if (n_cells)
        *n_cells = s->cell ? s->grid.n_cells : 0;
    return NPSIM_OK;
}

int npsim_nbr_info(npsim_sim_t s, int *cap, double *mean_len, int64_t *builds)
{
    NP_REQUIRE(s, "sim is NULL");
    if (cap)
        *cap = s->cell ? s->nl.cap : 0;
    if (mean_len)
        *mean_len = 0.0;
    if (builds)
        *builds = 0;
    if (!s->cell)
        return NPSIM_OK;
    NP_CUDA(cudaStreamSynchronize(s->user));
    if (mean_len) {
        std::vector<int> cnt((size_t)s->n);
        NP_CUDA(cudaMemcpy(cnt.data(), s->nl.nnbr, sizeof(int) * cnt.size(),
                           cudaMemcpyDeviceToHost));
        double sum = 0.0;
        for (int c : cnt)
            sum += c;
        *mean_len = sum / (double)s->n;
    }
    if (builds) {
        unsigned long long b = 0;
        NP_CUDA(cudaMemcpy(&b, s->nl.builds, sizeof(b), cudaMemcpyDeviceToHost));
        *builds = (int64_t)b;
    }
    return NPSIM_OK;
}

int npsim_chunk_steps(npsim_sim_t s, int *chunk)
{
    NP_REQUIRE(s && chunk, "sim and chunk are required");
    *chunk = kChunk;
    return NPSIM_OK;
}

int npsim_profile(npsim_sim_t s, int enable)
{
    NP_REQUIRE(s, "sim is NULL");
    NP_CUDA(cudaStreamSynchronize(s->user));
    if (enable && !s->ev[0][0][0]) {
        for (int j = 0; j < kChunk; ++j)
            for (int k = 0; k < 4; ++k)
                for (int e = 0; e < 2; ++e)
                    NP_CUDA(cudaEventCreate(&s->ev[j][k][e]));
    }
    if ((enable != 0) != s->profiling) {
        for (auto &g : s->graphs)
            cudaGraphExecDestroy(g.second);
        s->graphs.clear();
        s->profiling = enable != 0;
        s->last_chunk = 0;
    }
    return NPSIM_OK;
}

int npsim_kernel_times(npsim_sim_t s, double *ms, int *samples)
{
    NP_REQUIRE(s && ms, "sim and ms are required");
    NP_REQUIRE(s->profiling, "profiling is not enabled (npsim_profile)");
    NP_CUDA(cudaStreamSynchronize(s->user));
    const bool used[4] = {s->ap, s->cell, s->cell, true};
    const int k = s->last_chunk;
    for (int g = 0; g < 4; ++g) {
        double tot = 0.0;
        if (used[g])
            for (int j = 0; j < k; ++j) {
                float t = 0.f;
                NP_CUDA(cudaEventElapsedTime(&t, s->ev[j][g][0], s->ev[j][g][1]));
                tot += t;
            }
        ms[g] = (k > 0 && used[g]) ? tot / k : 0.0;
    }
    if (samples)
        *samples = k;
    return NPSIM_OK;
}

// ---------------------------------------------------------------------------
// Statistics

} // extern "C"

namespace {

// The statistics of Sec. 3 of one droplet of n NPs whose float64 positions
// ([3][n]) are x, float32 hi words xq and types typ (all device), at droplet
// radius R: the RDF (Sec. 3.2), the radial concentration C_NPs, N_surf, the
// centre of mass and R_g (Eqs. r0, Rg), D_f from the fractal equation (Eq. N)
// and by box counting.  Shared by npsim_stats and npsim_ens_stats.
int stats_core(StatsWork &w, const double *x, const float4 *xq, const int *typ, int n, double R,
               double d_mean, const npsim_type_t *types, int T, int *d_flags,
               const npsim_stats_cfg_t *cfg, int64_t *rdf_counts, double *rdf_g,
               int64_t *radial_counts, double *radial_c, npsim_stats_t *out, cudaStream_t st)
{
    memset(out, 0, sizeof(*out));
    out->R = R;
    out->d_mean = d_mean;
    const double pi = 3.14159265358979323846;

    const int nblk = (n + 255) / 256;
    const bool rdf = cfg->n_bins > 0 && rdf_counts, radial = cfg->radial_bins > 0 && radial_counts;
    if (!w.vec)
        NP_CUDA(dalloc(&w.vec, 8));
    // words of the results: [3 nblk] and [3 nblk] of a reduction, RDF bins,
    // radial bins, N_surf, box counts
    const size_t o_hist = 6 * (size_t)nblk, o_rhist = o_hist + (rdf ? cfg->n_bins : 0),
                 o_surf = o_rhist + (radial ? cfg->radial_bins : 0), o_box = o_surf + 1,
                 n_res = o_box + NPSIM_MAX_SCALES;
    if (n_res > w.res_cap) {
        dfree(w.res);
        w.res_cap = 0;
        NP_CUDA(dalloc(&w.res, n_res));
        w.res_cap = n_res;
    }
    std::vector<unsigned long long> res(n_res);
    double *d_part = reinterpret_cast<double *>(w.res);
    const double *part = reinterpret_cast<const double *>(res.data());
    // words [0, count) of the results to the host, after everything queued so far
    auto fetch = [&](size_t first, size_t count) -> cudaError_t {
        cudaError_t e = cudaMemcpyAsync(res.data() + first, w.res + first,
                                        sizeof(unsigned long long) * count,
                                        cudaMemcpyDeviceToHost, st);
        return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
    };
    // extent of the cloud: minimum corner (box-counting origin), largest |x_d|
    NP_CUDA(launch_block_reduce(2, x, n, nullptr, d_part, st));
    NP_CUDA(launch_block_reduce(3, x, n, nullptr, d_part + 3 * (size_t)nblk, st));
    NP_CUDA(fetch(0, 6 * (size_t)nblk));
    double o[3] = {INFINITY, INFINITY, INFINITY};
    double L = R;
    for (int b = 0; b < nblk; ++b)
        for (int d = 0; d < 3; ++d) {
            o[d] = std::min(o[d], part[3 * (size_t)b + d]);
            L = std::max(L, part[3 * (size_t)(nblk + b) + d]);
        }

    int rc = NPSIM_OK;
    if (rdf) {
        // cell grid over the cloud (positions are needed in float32 only to choose
        // candidates and for the bins that float32 settles)
        L += cfg->r_max + 1.0;
        CellGrid g = make_grid(L, pair_hist_cell_edge(cfg->r_max, L),
                               std::max<long long>(4 * (long long)n + 4096, 1 << 16));
        if (g.n_cells > w.cells_cap || n > w.cells_n) {
            // grow to hold both this droplet and the largest one seen so far
            CellGrid ga = g;
            ga.n_cells = std::max(g.n_cells, w.cells_cap);
            const int na = std::max(n, w.cells_n);
            free_cells(w.cb);
            w.cells_cap = w.cells_n = 0;
            rc = alloc_cells(ga, w.cb, na);
            if (rc)
                return rc;
            w.cells_cap = ga.n_cells;
            w.cells_n = na;
        }
        w.grid = g;
        NP_CUDA(launch_cell_build(g, xq, typ, n, w.cb, st));
        NP_CUDA(launch_pair_hist(x, n, cfg->r_max, cfg->n_bins, g, w.cb, w.res + o_hist, st));
    }
    if (radial)
        NP_CUDA(launch_radial_hist(x, n, R, cfg->radial_bins, w.res + o_rhist, st));
    // N_surf: NPs in the band (-r_i, r_i) about the surface
    SurfHalf hs{};
    for (int t = 0; t < T; ++t)
        hs.h[t] = 0.5 * types[t].sigma;
    NP_CUDA(launch_surface_count(x, typ, n, R, hs, w.res + o_surf, st));
    NP_CUDA(launch_block_reduce(0, x, n, nullptr, d_part, st));
    NP_CUDA(fetch(0, o_surf + 1));
    out->n_surf = (int64_t)res[o_surf];
    const double V = 4.0 / 3.0 * pi * R * R * R;
    if (rdf) {
        const double dr = cfg->r_max / (double)cfg->n_bins;
        for (int b = 0; b < cfg->n_bins; ++b) {
            rdf_counts[b] = (int64_t)res[o_hist + b];
            if (rdf_g) {
                const double r0 = b * dr, r1 = (b + 1) * dr;
                const double dV = 4.0 / 3.0 * pi * (r1 * r1 * r1 - r0 * r0 * r0);
                rdf_g[b] = ((double)rdf_counts[b] / (double)n) / ((double)(n - 1) * dV / V);
            }
        }
    }
    if (radial) {
        const double dr = R / (double)cfg->radial_bins;
        for (int b = 0; b < cfg->radial_bins; ++b) {
            radial_counts[b] = (int64_t)res[o_rhist + b];
            if (radial_c) {
                const double r0 = b * dr, r1 = (b + 1) * dr;
                const double dV = 4.0 / 3.0 * pi * (r1 * r1 * r1 - r0 * r0 * r0);
                radial_c[b] = ((double)radial_counts[b] / (double)n) / (dV / V);
            }
        }
    }
    // centre of mass and radius of gyration (Eqs. r0, Rg), fractal equation (Eq. N)
    double c[3] = {0, 0, 0};
    for (int b = 0; b < nblk; ++b)
        for (int d = 0; d < 3; ++d)
            c[d] += part[3 * (size_t)b + d];
    for (int d = 0; d < 3; ++d)
        c[d] /= (double)n;
    NP_CUDA(cudaMemcpyAsync(w.vec, c, sizeof(c), cudaMemcpyHostToDevice, st));
    NP_CUDA(launch_block_reduce(1, x, n, w.vec, d_part, st));
    NP_CUDA(fetch(0, 3 * (size_t)nblk));
    double ss = 0.0;
    for (int b = 0; b < nblk; ++b)
        ss += part[3 * (size_t)b];
    const double Rg = std::sqrt(ss / (double)n);
    out->Rg = Rg;
    out->Df_rg = std::log((double)n / kKf) / std::log(2.0 * Rg / d_mean);
    for (int d = 0; d < 3; ++d)
        out->center[d] = c[d];

    out->Df_box = NAN;
    if (cfg->boxcount) {
        size_t tsz = 1;
        while (tsz < 2 * (size_t)n)
            tsz <<= 1;
        int ns = 0;
        while (ns < cfg->max_scales && d_mean * std::ldexp(1.0, ns) <= 2.0 * Rg)
            ++ns;
        // one table per scale, as many scales per launch as fit kBoxTableKeys (one
        // at least)
        const int group = (int)std::max<size_t>(1, std::min<size_t>(ns, kBoxTableKeys / tsz));
        if (group * tsz > w.table_cap) {
            dfree(w.table);
            w.table_cap = 0;
            NP_CUDA(dalloc(&w.table, group * tsz));
            w.table_cap = group * tsz;
        }
        NP_CUDA(cudaMemcpyAsync(w.vec + 3, o, sizeof(o), cudaMemcpyHostToDevice, st));
        if (ns > 0) {
            NP_CUDA(cudaMemsetAsync(w.res + o_box, 0, sizeof(unsigned long long) * ns, st));
            for (int k = 0; k < ns; k += group)
                NP_CUDA(launch_boxcount(x, n, w.vec + 3, d_mean, k, std::min(group, ns - k),
                                        w.table, tsz, w.res + o_box, d_flags, st));
            NP_CUDA(fetch(o_box, ns));
        }
        for (int k = 0; k < ns; ++k)
            out->nbox[k] = (int64_t)res[o_box + k];
        out->n_scales = ns;
        if (ns - 1 >= 2) {
            // least squares of ln N_box on ln eps over scales k >= 1
            const int m = ns - 1;
            double mx = 0, my = 0;
            for (int k = 1; k < ns; ++k) {
                mx += std::log(d_mean * std::ldexp(1.0, k));
                my += std::log((double)out->nbox[k]);
            }
            mx /= m;
            my /= m;
            double sxy = 0, sxx = 0;
            for (int k = 1; k < ns; ++k) {
                const double ex = std::log(d_mean * std::ldexp(1.0, k)) - mx;
                sxy += ex * (std::log((double)out->nbox[k]) - my);
                sxx += ex * ex;
            }
            out->Df_box = -sxy / sxx;
        }
    }
    return NPSIM_OK;
}

int check_stats_cfg(const npsim_stats_cfg_t *cfg)
{
    NP_REQUIRE(cfg->n_bins >= 0 && cfg->radial_bins >= 0, "bins must be >= 0");
    NP_REQUIRE(cfg->n_bins == 0 || cfg->r_max > 0, "r_max must be positive");
    NP_REQUIRE(cfg->max_scales >= 0 && cfg->max_scales <= NPSIM_MAX_SCALES,
               "max_scales must be in [0, %d]", NPSIM_MAX_SCALES);
    return NPSIM_OK;
}

} // namespace

extern "C" {

int npsim_stats(npsim_sim_t s, const npsim_stats_cfg_t *cfg, int64_t *rdf_counts,
                double *rdf_g, int64_t *radial_counts, double *radial_c, npsim_stats_t *out)
{
    NP_TRACE();
    NP_REQUIRE(s && cfg && out, "sim, cfg and out are required");
    int rc = check_stats_cfg(cfg);
    if (rc)
        return rc;
    const double t = (double)s->step * s->P.dt;
    const double R2 = s->P.R0 * s->P.R0 - s->P.k_evap * t;
    const double R = R2 > 0 ? std::sqrt(R2) : 0.0;
    rc = positions_f64(s);
    if (rc)
        return rc;
    rc = stats_core(s->sw, s->x, s->xq, s->typ, s->n, R, s->d_mean, s->types, s->P.n_types,
                    s->d_flags, cfg, rdf_counts, rdf_g, radial_counts, radial_c, out, s->user);
    if (rc)
        return rc;
    return read_flags(s);
}

// ---------------------------------------------------------------------------
// Checkpoints

namespace {
// Layout: header, then the raw state words so that a resumed run is
// bit-identical: position hi words [3][n], lo words [3][n], velocities [3][n]
// (float32 SoA), the types (int32[n]) and the order of the NPs inside their
// type groups (int32[n], the pair kernels' summation order); with a cell list
// also the neighbour-list state: the cell grid and list capacity (header), the
// positions of the last build (float4[n]) and the rebuild gate (header), from
// which a resumed run rebuilds exactly the list the saved run was using.
const char kMagic[8] = {'N', 'P', 'S', 'I', 'M', 'C', 'K', '5'};

struct CkptHeader {
    char magic[8];
    int32_t version, n_types;
    int64_t n, step;
    int32_t rot_mode, lj_mode, coulomb, wall, integrator, has_ov, sum_neutral, pad_;
    uint64_t seed;
    double dt, kT, R0, k_evap, g, omega, bjerrum, lj_cut, v_kick, coulomb_cut;
    double eps_ov[NPSIM_MAX_TYPES * NPSIM_MAX_TYPES];
    npsim_type_t types[NPSIM_MAX_TYPES];
    int32_t cell, grid_dim, grid_cells, nbr_cap, gate, pad2_;
    float grid_inv_h, grid_L;
};

// Put the neighbour-list state of a checkpoint back: the saved grid and list
// capacity, a build from the saved build positions (which writes the same
// lists and x_ref), and the saved gate.
int restore_lists(npsim_sim *s, const CkptHeader &h, const float4 *x_ref_host)
{
    if (!s->cell || !h.cell)
        return NPSIM_OK;
    CellGrid g{};
    g.dim = h.grid_dim;
    g.n_cells = h.grid_cells;
    g.inv_h = h.grid_inv_h;
    g.L = h.grid_L;
    g.tb = s->T;
    set_extents(g, s->rlist);
    int rc0 = ensure_cells(s, g);
    if (rc0)
        return rc0;
    s->grid = g;
    if (h.nbr_cap != s->nl.cap) {
        dfree(s->nl.nbr);
        NP_CUDA(dalloc(&s->nl.nbr, (size_t)h.nbr_cap * s->n));
        NP_CUDA(cudaMemsetAsync(s->nl.nbr, 0, sizeof(unsigned) * (size_t)h.nbr_cap * s->n, s->user));
        s->nl.cap = h.nbr_cap;
    }
    for (auto &e : s->graphs)
        cudaGraphExecDestroy(e.second);
    s->graphs.clear();
    NP_CUDA(cudaMemcpy(s->nl.x_ref, x_ref_host, sizeof(float4) * (size_t)s->n,
                       cudaMemcpyHostToDevice));
    NP_CUDA(launch_list_build(s->grid, s->cb, s->nl.x_ref, s->typ, s->n, s->tab_full, s->d_rcc2,
                              kSkin, s->nl, s->d_flags, nullptr, s->list_bar, s->user));
    // the list kernel reads the current positions from the cell-ordered records
    NP_CUDA(launch_cell_refresh(s->cb, s->xq, s->typ, s->n, s->user));
    NP_CUDA(cudaStreamSynchronize(s->user));
    return set_gate(s, h.gate);
}
} // namespace

int npsim_scattering(const double *g, int32_t n_bins, double r_max, double n_surf, double Rg,
                     double Df, const double *q, int32_t n_q, double *I, double *I_frac)
{
    NP_TRACE();
    NP_REQUIRE(g && q && I, "g, q and I are required");
    NP_REQUIRE(n_bins >= 1 && n_q >= 1, "n_bins and n_q must be >= 1");
    NP_REQUIRE(r_max > 0 && std::isfinite(r_max), "r_max must be positive");
    for (int k = 0; k < n_q; ++k)
        NP_REQUIRE(q[k] >= 0 && std::isfinite(q[k]), "q[%d] must be finite and >= 0", k);
    int count = 0;
    if (cudaGetDeviceCount(&count) != cudaSuccess || count < 1)
        return set_err(NPSIM_ERR_NO_DEVICE, "no CUDA device visible");
    double *dg = nullptr, *dq = nullptr, *dI = nullptr, *dF = nullptr;
    auto release = [&]() {
        dfree(dg);
        dfree(dq);
        dfree(dI);
        dfree(dF);
    };
    cudaError_t e = dalloc(&dg, (size_t)n_bins);
    if (e == cudaSuccess)
        e = dalloc(&dq, (size_t)n_q);
    if (e == cudaSuccess)
        e = dalloc(&dI, (size_t)n_q);
    if (e == cudaSuccess && I_frac)
        e = dalloc(&dF, (size_t)n_q);
    if (e == cudaSuccess)
        e = cudaMemcpy(dg, g, sizeof(double) * n_bins, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(dq, q, sizeof(double) * n_q, cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = launch_scattering(dg, n_bins, r_max, dq, n_q, n_surf, Rg, Df, dI, dF, 0);
    if (e == cudaSuccess)
        e = cudaMemcpy(I, dI, sizeof(double) * n_q, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && I_frac)
        e = cudaMemcpy(I_frac, dF, sizeof(double) * n_q, cudaMemcpyDeviceToHost);
    release();
    if (e != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "npsim_scattering: %s", cudaGetErrorString(e));
    return NPSIM_OK;
}

int npsim_save(npsim_sim_t s, const char *path)
{
    NP_TRACE();
    NP_REQUIRE(s && path, "sim and path are required");
    CkptHeader h{};
    memcpy(h.magic, kMagic, 8);
    h.version = 5;
    h.n_types = s->T;
    h.n = s->n;
    h.step = s->step;
    h.rot_mode = s->P.rot_mode;
    h.lj_mode = s->P.lj_mode;
    h.coulomb = s->P.coulomb;
    h.wall = s->P.wall;
    h.integrator = s->P.integrator;
    h.has_ov = s->has_ov ? 1 : 0;
    h.sum_neutral = s->P.sum_neutral;
    h.seed = s->P.seed;
    h.dt = s->P.dt;
    h.kT = s->P.kT;
    h.R0 = s->P.R0;
    h.k_evap = s->P.k_evap;
    h.g = s->P.g;
    h.omega = s->P.omega;
    h.bjerrum = s->P.bjerrum;
    h.lj_cut = s->P.lj_cut;
    h.v_kick = s->P.v_kick;
    h.coulomb_cut = s->P.coulomb_cut;
    memcpy(h.eps_ov, s->eps_ov, sizeof(h.eps_ov));
    memcpy(h.types, s->types, sizeof(h.types));
    const size_t n = (size_t)s->n;
    NP_CUDA(cudaStreamSynchronize(s->user));
    std::vector<float4> xq(n);
    std::vector<float> words(9 * n);
    NP_CUDA(cudaMemcpy(xq.data(), s->xq, sizeof(float4) * n, cudaMemcpyDeviceToHost));
    NP_CUDA(cudaMemcpy(words.data() + 3 * n, s->x_lo, sizeof(float) * 3 * n,
                       cudaMemcpyDeviceToHost));
    NP_CUDA(cudaMemcpy(words.data() + 6 * n, s->v, sizeof(float) * 3 * n,
                       cudaMemcpyDeviceToHost));
    for (size_t i = 0; i < n; ++i) {
        words[i] = xq[i].x;
        words[n + i] = xq[i].y;
        words[2 * n + i] = xq[i].z;
    }
    FILE *f = fopen(path, "wb");
    if (!f)
        return set_err(NPSIM_ERR_IO, "cannot open %s for writing", path);
    std::vector<int32_t> rank(s->h_rank);
    rank.resize(n, 0);
    std::vector<float4> xref;
    if (s->cell) {
        h.cell = 1;
        h.grid_dim = s->grid.dim;
        h.grid_cells = s->grid.n_cells;
        h.grid_inv_h = s->grid.inv_h;
        h.grid_L = s->grid.L;
        h.nbr_cap = s->nl.cap;
        NP_CUDA(cudaMemcpy(&h.gate, s->d_gate, sizeof(int), cudaMemcpyDeviceToHost));
        xref.resize(n);
        NP_CUDA(cudaMemcpy(xref.data(), s->nl.x_ref, sizeof(float4) * n, cudaMemcpyDeviceToHost));
    }
    bool ok = fwrite(&h, sizeof(h), 1, f) == 1 &&
              fwrite(words.data(), sizeof(float), words.size(), f) == words.size() &&
              fwrite(s->h_type.data(), sizeof(int32_t), s->h_type.size(), f) ==
                  s->h_type.size() &&
              fwrite(rank.data(), sizeof(int32_t), rank.size(), f) == rank.size() &&
              fwrite(xref.data(), sizeof(float4), xref.size(), f) == xref.size();
    ok = (fclose(f) == 0) && ok;
    if (!ok)
        return set_err(NPSIM_ERR_IO, "short write to %s", path);
    return NPSIM_OK;
}

int npsim_load(const char *path, const npsim_type_t *types_override,
               const npsim_params_t *params_override, void *stream, npsim_sim_t *out)
{
    NP_TRACE();
    NP_REQUIRE(path && out, "path and out are required");
    *out = nullptr;
    FILE *f = fopen(path, "rb");
    if (!f)
        return set_err(NPSIM_ERR_IO, "cannot open %s", path);
    CkptHeader h{};
    if (fread(&h, sizeof(h), 1, f) != 1 || memcmp(h.magic, kMagic, 8) != 0 || h.version != 5 ||
        h.n < 1 || h.n > (1ll << 29) || h.n_types < 1 || h.n_types > NPSIM_MAX_TYPES) {
        fclose(f);
        return set_err(NPSIM_ERR_IO, "%s is not an npsim checkpoint", path);
    }
    const size_t n = (size_t)h.n;
    std::vector<float> words(9 * n);
    std::vector<int32_t> ty(n), rank(n);
    std::vector<float4> xref(h.cell ? n : 0);
    bool ok = fread(words.data(), sizeof(float), words.size(), f) == words.size() &&
              fread(ty.data(), sizeof(int32_t), ty.size(), f) == ty.size() &&
              fread(rank.data(), sizeof(int32_t), rank.size(), f) == rank.size() &&
              fread(xref.data(), sizeof(float4), xref.size(), f) == xref.size();
    fclose(f);
    if (!ok)
        return set_err(NPSIM_ERR_IO, "%s is truncated", path);
    // float64 values (AoS) for creation: x = hi + lo, v
    std::vector<double> x(3 * n), v(3 * n);
    for (size_t i = 0; i < n; ++i)
        for (int d = 0; d < 3; ++d) {
            x[3 * i + d] = (double)words[d * n + i] + (double)words[(3 + d) * n + i];
            v[3 * i + d] = (double)words[(6 + d) * n + i];
        }
    npsim_params_t p{};
    p.n_types = h.n_types;
    p.rot_mode = h.rot_mode;
    p.lj_mode = h.lj_mode;
    p.coulomb = h.coulomb;
    p.wall = h.wall;
    p.integrator = h.integrator;
    p.sum_neutral = h.sum_neutral;
    p.seed = h.seed;
    p.dt = h.dt;
    p.kT = h.kT;
    p.R0 = h.R0;
    p.k_evap = h.k_evap;
    p.g = h.g;
    p.omega = h.omega;
    p.bjerrum = h.bjerrum;
    p.lj_cut = h.lj_cut;
    p.v_kick = h.v_kick;
    p.coulomb_cut = h.coulomb_cut;
    p.eps_override = h.has_ov ? h.eps_ov : nullptr;
    if (params_override) {
        p = *params_override;
        NP_REQUIRE(p.n_types == h.n_types, "params_override changes n_types");
    }
    const npsim_type_t *tys = types_override ? types_override : h.types;
    npsim_sim_t s = nullptr;
    int rc = create_impl(tys, &p, h.n, x.data(), v.data(), ty.data(), stream, rank.data(), &s);
    if (rc)
        return rc;
    rc = upload_words(s, words.data(), h.step);
    if (!rc && h.cell) { // the saved list state, then the forces from it
        rc = restore_lists(s, h, xref.data());
        if (!rc)
            rc = finish_upload(s, h.step, false);
    }
    if (rc) {
        npsim_destroy(s);
        return rc;
    }
    *out = s;
    return NPSIM_OK;
}

} // extern "C"

// ---------------------------------------------------------------------------
// Ensemble of independent droplets

struct npsim_ens {
    int D = 0, n_total = 0, sms = 0;
    std::vector<int> off, cnt;
    std::vector<EnsDrop> h_drops;
    std::vector<PairTab> h_tabs;
    std::vector<npsim_params_t> P;
    std::vector<std::vector<npsim_type_t>> types;
    std::vector<std::vector<double>> eps_ov;
    std::vector<int32_t> h_type;

    cudaStream_t user = nullptr, cap = nullptr;
    // state layouts as in npsim_sim, over the concatenation of the droplets
    float *x_lo = nullptr, *v = nullptr;  // [3][n_total]
    float *F = nullptr, *F_tmp = nullptr; // [6][n_total]
    float4 *xq = nullptr;
    int *typ = nullptr, *drop_of = nullptr;
    int *perm = nullptr, *tblk = nullptr, *dblk = nullptr; // type-grouped order
    int n_pos = 0;               // its length
    EnsDrop *drops = nullptr;
    PairTab *tabs = nullptr;
    EnsItem *items = nullptr;    // work items of the all-pairs launch
    int *row_first = nullptr;    // first slot of every row tile
    unsigned *d_work = nullptr;  // work-item counters of the all-pairs launch
    float *slots = nullptr;      // one [6][itile] slot per work item, then column partials
    float *F_pair = nullptr;     // [n_total][8] all-pairs forces
    long long *d_step = nullptr;
    float4 *d_spring = nullptr; // [2][D][NPSIM_MAX_TYPES]
    int *d_flags = nullptr;
    unsigned *d_done = nullptr;

    int shape = 0;
    int ctas = 1;           // CTAs of the all-pairs launch
    int n_items = 0;        // its work items
    std::map<int, cudaGraphExec_t> graphs;
    int64_t step = 0;
    // kernel timing (npsim_ens_profile): events around the all-pairs launch
    // (group 0) and the integrator launch (group 1) of every pass of a chunk
    bool profiling = false;
    int last_chunk = 0;
    cudaEvent_t ev[kChunk][2][2]{};

    double *stage = nullptr;    // host-facing copy of one droplet's state (lazy)
    size_t stage_cap = 0;       // NPs it holds
    std::vector<double> d_mean; // number-mean NP diameter of each droplet
    StatsWork sw{};             // statistics of one droplet at a time (lazy)

    ~npsim_ens()
    {
        free_stats(sw);
        for (auto &g : graphs)
            cudaGraphExecDestroy(g.second);
        for (auto &a : ev)
            for (auto &b : a)
                for (auto &x : b)
                    if (x)
                        cudaEventDestroy(x);
        dfree(x_lo);
        dfree(v);
        dfree(F);
        dfree(F_tmp);
        dfree(xq);
        dfree(typ);
        dfree(drop_of);
        dfree(perm);
        dfree(tblk);
        dfree(dblk);
        dfree(drops);
        dfree(tabs);
        dfree(stage);
        dfree(items);
        dfree(row_first);
        dfree(d_work);
        dfree(slots);
        dfree(F_pair);
        dfree(d_step);
        dfree(d_spring);
        dfree(d_flags);
        dfree(d_done);
        if (cap)
            cudaStreamDestroy(cap);
    }
};

namespace {

// Work items per CTA that the chunk size aims at: enough that the last items
// drawn (the only imbalance of dynamic scheduling, longest items first) are
// short, few enough that the per-item slots stay small.
constexpr int kItemsPerCta = 12;

// The all-pairs work of an ensemble for one launch shape: work items (longest
// first, slots numbered in row order), first slot of every row tile, floats of
// the row slots and column partials.
struct EnsGeometry {
    std::vector<EnsItem> items;
    std::vector<int> row_first;
    size_t floats = 0;
    int ctas = 1;
};

// Geometry for launch shape `shape` on grid_target CTAs; sets the droplets'
// row0 and col0.
EnsGeometry ens_geometry(npsim_ens *e, int shape, int grid_target)
{
    const ApConfig c = ens_config(shape);
    const int itile = c.block * c.ki;
    const bool sym = ens_sym(shape);
    const int tri = sym ? itile / c.jt : 0; // first j-tile of row r: tri r
    long long W = 0;
    for (const EnsDrop &g : e->h_drops) { // npad is a multiple of 256, jt divides 256
        const long long n_it = (g.npad + itile - 1) / itile, n_jt = g.npad / c.jt;
        W += n_it * n_jt - tri * n_it * (n_it - 1) / 2;
    }
    const long long target = (long long)std::max(grid_target, 1) * kItemsPerCta;
    // items are counted in int: a chunk that keeps them below 2^30
    const int chunk = (int)std::max<long long>({1, (W + target - 1) / target, W >> 28});
    EnsGeometry G;
    long long col = 0;
    for (int d = 0; d < e->D; ++d) {
        EnsDrop &g = e->h_drops[d];
        const int n_it = (g.npad + itile - 1) / itile, n_jt = g.npad / c.jt;
        g.row0 = (int)G.row_first.size();
        g.col0 = col;
        if (sym)
            col += (long long)sym_col_floats(g.npad, itile);
        for (int r = 0; r < n_it; ++r) {
            G.row_first.push_back((int)G.items.size());
            for (int j = tri * r; j < n_jt; j += chunk)
                G.items.push_back(EnsItem{d, r, j, std::min(n_jt, j + chunk), (int)G.items.size()});
        }
    }
    G.row_first.push_back((int)G.items.size());
    // longest first, those nearest the diagonal (rich in LJ) before others
    std::stable_sort(G.items.begin(), G.items.end(), [tri](const EnsItem &a, const EnsItem &b) {
        const int la = a.jt1 - a.jt0, lb = b.jt1 - b.jt0;
        return la != lb ? la > lb : a.jt0 - tri * a.row < b.jt0 - tri * b.row;
    });
    G.floats = G.items.size() * 6 * (size_t)itile + (size_t)col;
    G.ctas = (int)std::min<size_t>((size_t)std::max(grid_target, 1), G.items.size());
    return G;
}

int ens_upload_geometry(npsim_ens *e, int shape, const EnsGeometry &G)
{
    dfree(e->items);
    dfree(e->row_first);
    NP_CUDA(dalloc(&e->items, G.items.size()));
    NP_CUDA(dalloc(&e->row_first, G.row_first.size()));
    NP_CUDA(cudaMemcpyAsync(e->drops, e->h_drops.data(), sizeof(EnsDrop) * e->D,
                            cudaMemcpyHostToDevice, e->user));
    NP_CUDA(cudaMemcpyAsync(e->items, G.items.data(), sizeof(EnsItem) * G.items.size(),
                            cudaMemcpyHostToDevice, e->user));
    NP_CUDA(cudaMemcpyAsync(e->row_first, G.row_first.data(), sizeof(int) * G.row_first.size(),
                            cudaMemcpyHostToDevice, e->user));
    NP_CUDA(cudaStreamSynchronize(e->user));
    e->shape = shape;
    e->n_items = (int)G.items.size();
    e->ctas = G.ctas;
    return NPSIM_OK;
}

EnsAllpairsArgs ens_ap_args(npsim_ens *e, float *slots)
{
    const ApConfig c = ens_config(e->shape);
    EnsAllpairsArgs a{};
    a.xq = e->xq;
    a.perm = e->perm;
    a.tblk = e->tblk;
    a.dblk = e->dblk;
    a.drops = e->drops;
    a.tabs = e->tabs;
    a.items = e->items;
    a.row_first = e->row_first;
    a.n_items = e->n_items;
    a.n_pos = e->n_pos;
    a.itile = c.block * c.ki;
    a.sym = ens_sym(e->shape) ? 1 : 0;
    a.work = e->d_work;
    a.slots = slots;
    a.F_pair = e->F_pair;
    return a;
}

int ens_pass(npsim_ens *e, int mode, bool ext, float *Fout, cudaStream_t st,
             int prof_slot = -1)
{
    const bool prof = prof_slot >= 0 && e->profiling;
    // inside stream capture the External flag makes each record a real
    // event-record node of the graph
    auto mark = [&](int group, int edge) -> cudaError_t {
        return prof ? cudaEventRecordWithFlags(e->ev[prof_slot][group][edge], st,
                                               cudaEventRecordExternal)
                    : cudaSuccess;
    };
    NP_CUDA(mark(0, 0));
    NP_CUDA(launch_ens_allpairs(e->shape, e->ctas, ens_ap_args(e, e->slots), st));
    NP_CUDA(mark(0, 1));
    EnsIntArgs a{};
    a.x_lo = e->x_lo;
    a.v = e->v;
    a.F = Fout;
    a.typ = e->typ;
    a.xq = e->xq;
    a.drop_of = e->drop_of;
    a.drops = e->drops;
    a.F_pair = e->F_pair;
    a.spring = e->d_spring;
    a.ext_on = ext ? 1 : 0;
    a.step = e->d_step;
    a.flags = e->d_flags;
    a.done = e->d_done;
    NP_CUDA(mark(1, 0));
    NP_CUDA(launch_ens_integrate(mode, a, e->n_total, e->D, st));
    NP_CUDA(mark(1, 1));
    return NPSIM_OK;
}

int ens_chunk(npsim_ens *e, int k, cudaStream_t st)
{
    EnsIntArgs a{};
    a.x_lo = e->x_lo;
    a.v = e->v;
    a.F = e->F;
    a.typ = e->typ;
    a.xq = e->xq;
    a.drop_of = e->drop_of;
    a.drops = e->drops;
    a.spring = e->d_spring;
    a.step = e->d_step;
    a.flags = e->d_flags;
    a.done = e->d_done;
    NP_CUDA(launch_ens_integrate(MODE_A, a, e->n_total, e->D, st));
    for (int j = 0; j < k; ++j) {
        int rc = ens_pass(e, j + 1 < k ? MODE_BA : MODE_B, true, e->F, st, j);
        if (rc)
            return rc;
    }
    return NPSIM_OK;
}

int ens_graph(npsim_ens *e, int k, cudaGraphExec_t *out)
{
    auto it = e->graphs.find(k);
    if (it != e->graphs.end()) {
        *out = it->second;
        return NPSIM_OK;
    }
    NP_CUDA(cudaStreamBeginCapture(e->cap, cudaStreamCaptureModeThreadLocal));
    int rc = ens_chunk(e, k, e->cap);
    cudaGraph_t g = nullptr;
    cudaError_t ce = cudaStreamEndCapture(e->cap, &g);
    if (rc) {
        if (g)
            cudaGraphDestroy(g);
        return rc;
    }
    if (ce != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "graph capture failed: %s", cudaGetErrorString(ce));
    cudaGraphExec_t ex = nullptr;
    ce = cudaGraphInstantiate(&ex, g, 0);
    cudaGraphDestroy(g);
    if (ce != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "graph instantiate failed: %s", cudaGetErrorString(ce));
    e->graphs[k] = ex;
    *out = ex;
    return NPSIM_OK;
}

// The requested parts of droplet d's state on the host (one conversion kernel and
// up to three copies; the parts used to be copied row by row of the device arrays
// and put together here: 16 droplets of 512 to 4096 NPs took 2.3 ms, now 0.5).
int ens_state_out(npsim_ens *e, int d, const float *F_src, double *x, double *v, double *F)
{
    const size_t n = (size_t)e->cnt[d], off = (size_t)e->off[d];
    if (n > e->stage_cap) {
        dfree(e->stage);
        e->stage_cap = 0;
        const size_t most = (size_t)*std::max_element(e->cnt.begin(), e->cnt.end());
        NP_CUDA(dalloc(&e->stage, 9 * most));
        e->stage_cap = most;
    }
    return state_to_host(e->xq + off, e->x_lo + off, e->v + off, F_src + off, (int)n,
                         (size_t)e->n_total, e->stage, x, v, F, e->user);
}

// Whether the ensemble's column partials are small enough for launch shape c.
bool ens_shape_fits(const npsim_ens *e, int c)
{
    if (!ens_sym(c))
        return true;
    const ApConfig cf = ens_config(c);
    const int itile = cf.block * cf.ki;
    size_t col = 0;
    for (const EnsDrop &g : e->h_drops)
        col += sym_col_floats(g.npad, itile);
    return col * sizeof(float) <= sym_max_bytes(itile);
}

// Time every ensemble launch shape on the current positions; keep the fastest.
int ens_autotune(npsim_ens *e)
{
    const int nc = ens_num_configs();
    const char *env = getenv("NPSIM_ENS_SHAPE");
    int best = -1;
    if (env) {
        const int idx = atoi(env);
        if (idx >= 0 && idx < nc && ens_occupancy(idx) > 0)
            best = idx;
    }
    // the same ensemble geometry gets the same shape within a process (so
    // that repeated runs of one ensemble sum in the same order)
    std::vector<long long> key;
    for (int d = 0; d < e->D; ++d) {
        const EnsDrop &g = e->h_drops[d];
        key.push_back(((long long)g.npad << 2) | (g.rc2_lim > 0.0f ? 2 : 0) |
                      (g.has_coul ? 1 : 0));
    }
    const bool pinned = best >= 0;
    if (!pinned) {
        std::lock_guard<std::mutex> g(g_tune_mu);
        auto it = g_ens_tune_cache.find(key);
        if (it != g_ens_tune_cache.end())
            best = it->second;
    }
    const bool cached = !pinned && best >= 0;
    bool all = true;
    if (best < 0) {
        float *tmp = nullptr;
        size_t need = 0;
        std::vector<size_t> needs;
        for (int c = 0; c < nc; ++c) {
            const int occ = ens_occupancy(c);
            if (occ > 0 && ens_shape_fits(e, c))
                needs.push_back(ens_geometry(e, c, occ * e->sms).floats);
        }
        int rc = alloc_tune_scratch(needs, 0, &tmp, &need, &all);
        if (rc)
            return rc;
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        float best_ms = 1e30f;
        for (int c = 0; c < nc; ++c) {
            const int occ = ens_occupancy(c);
            if (occ <= 0 || !ens_shape_fits(e, c))
                continue;
            const EnsGeometry G = ens_geometry(e, c, occ * e->sms);
            if (G.floats > need)
                continue;
            rc = ens_upload_geometry(e, c, G);
            if (rc) {
                cudaFree(tmp);
                return rc;
            }
            if (launch_ens_allpairs(c, e->ctas, ens_ap_args(e, tmp), e->user) != cudaSuccess)
                continue;
            cudaEventRecord(e0, e->user);
            for (int r = 0; r < 2; ++r)
                launch_ens_allpairs(c, e->ctas, ens_ap_args(e, tmp), e->user);
            cudaEventRecord(e1, e->user);
            if (cudaEventSynchronize(e1) != cudaSuccess)
                continue;
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (getenv("NPSIM_AUTOTUNE_LOG")) {
                const ApConfig cf = ens_config(c);
                fprintf(stderr,
                        "npsim ensemble autotune shape %d <%d,%d,%d> grid %d items %d: %.4f ms\n",
                        c, cf.block, cf.ki, cf.jt, e->ctas, e->n_items, ms / 2);
            }
            if (ms < best_ms) {
                best_ms = ms;
                best = c;
            }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        cudaFree(tmp);
        cudaError_t ce = cudaGetLastError();
        if (ce != cudaSuccess)
            return set_err(NPSIM_ERR_CUDA, "ensemble autotune: %s", cudaGetErrorString(ce));
        if (best < 0)
            best = 0;
    }
    if (!pinned && !cached && all) {
        std::lock_guard<std::mutex> g(g_tune_mu);
        g_ens_tune_cache[key] = best;
    }
    EnsGeometry G = ens_geometry(e, best, std::max(1, ens_occupancy(best)) * e->sms);
    cudaError_t ce = dalloc(&e->slots, G.floats);
    if (ce == cudaErrorMemoryAllocation && ens_sym(best)) {
        // no room for the column partials: the one-sided shape
        cudaGetLastError();
        while (ens_sym(best))
            best = (best + 1) % nc;
        G = ens_geometry(e, best, std::max(1, ens_occupancy(best)) * e->sms);
        ce = dalloc(&e->slots, G.floats);
    }
    NP_CUDA(ce);
    return ens_upload_geometry(e, best, G);
}

} // namespace

extern "C" {

int npsim_ens_create(const npsim_droplet_t *drops, int32_t n_drops, void *stream,
                     npsim_ens_t *out)
{
    NP_TRACE();
    NP_REQUIRE(out, "out is NULL");
    *out = nullptr;
    NP_REQUIRE(drops && n_drops >= 1, "need at least one droplet");
    long long total = 0;
    for (int d = 0; d < n_drops; ++d) {
        const npsim_droplet_t &dr = drops[d];
        int rc = validate(dr.types, &dr.params, dr.n);
        if (rc)
            return set_err(rc, "droplet %d: %s", d, g_err.c_str());
        NP_REQUIRE(dr.params.lj_mode != 2, "droplet %d: the ensemble sums LJ inside the all-pairs "
                                           "kernel (lj_mode 0 or 1)", d);
        NP_REQUIRE(dr.x0 && dr.type, "droplet %d: x0 and type are required", d);
        for (int64_t i = 0; i < dr.n; ++i)
            NP_REQUIRE(dr.type[i] >= 0 && dr.type[i] < dr.params.n_types,
                       "droplet %d: type[%lld] out of range", d, (long long)i);
        total += dr.n;
    }
    NP_REQUIRE(total <= (1ll << 29), "too many particles in the ensemble");
    int sms = 0;
    int rc = check_device(&sms);
    if (rc)
        return rc;

    npsim_ens *e = new npsim_ens();
    auto bail = [&](int code) {
        delete e;
        return code;
    };
    e->D = n_drops;
    e->n_total = (int)total;
    e->sms = sms;
    e->user = (cudaStream_t)stream;
    e->off.resize(n_drops);
    e->cnt.resize(n_drops);
    e->h_drops.assign(n_drops, EnsDrop{});
    e->h_tabs.assign(n_drops, PairTab{});
    e->P.resize(n_drops);
    e->types.resize(n_drops);
    e->eps_ov.resize(n_drops);
    e->d_mean.assign(n_drops, 1.0);
    std::vector<double> xs(3 * (size_t)total), vs(3 * (size_t)total, 0.0);
    std::vector<int> dof((size_t)total);
    std::vector<float4> xq0((size_t)total);
    e->h_type.resize((size_t)total);
    int off = 0;
    for (int d = 0; d < n_drops; ++d) {
        const npsim_droplet_t &dr = drops[d];
        const int n = (int)dr.n;
        e->off[d] = off;
        e->cnt[d] = n;
        e->P[d] = dr.params;
        e->types[d].assign(dr.types, dr.types + dr.params.n_types);
        if (dr.params.eps_override)
            e->eps_ov[d].assign(dr.params.eps_override,
                                dr.params.eps_override + dr.params.n_types * dr.params.n_types);
        e->P[d].eps_override = nullptr;
        EnsDrop &g = e->h_drops[d];
        g.offset = off;
        g.n = n;
        g.rot_mode = dr.params.rot_mode;
        g.wall = dr.params.wall;
        g.integrator = dr.params.integrator;
        g.seed = dr.params.seed;
        g.dt = dr.params.dt;
        g.R0 = dr.params.R0;
        g.k_evap = dr.params.k_evap;
        g.g = dr.params.g;
        g.omega2 = dr.params.omega * dr.params.omega;
        float qf[NPSIM_MAX_TYPES] = {};
        fill_coefs(dr.types, &dr.params, g.tc, qf);
        npsim_params_t pc = dr.params;
        if (pc.lj_mode == 0) { // no LJ: zero the LJ columns of the table
            pc.lj_cut = 0.0;
        }
        fill_tabs(dr.types, &pc, e->eps_ov[d].empty() ? nullptr : e->eps_ov[d].data(),
                  &e->h_tabs[d], nullptr);
        if (pc.lj_mode == 0)
            for (int k = 0; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; ++k) {
                e->h_tabs[d].e[k].y = 0.0f;
                e->h_tabs[d].e[k].z = 0.0f;
            }
        g.rc2_lim = 0.0f;
        g.has_coul = 0;
        for (int k = 0; k < NPSIM_MAX_TYPES * NPSIM_MAX_TYPES; ++k) {
            const float4 t = e->h_tabs[d].e[k];
            if (t.y != 0.0f)
                g.rc2_lim = std::max(g.rc2_lim, t.z * 1.0001f);
            if (t.w != 0.0f)
                g.has_coul = 1;
        }
        double dsum = 0.0;
        for (int i = 0; i < n; ++i)
            dsum += dr.types[dr.type[i]].sigma;
        e->d_mean[d] = dsum / (double)n;
        for (int i = 0; i < n; ++i) {
            for (int k = 0; k < 3; ++k) {
                xs[(size_t)k * total + off + i] = dr.x0[3 * (size_t)i + k];
                if (dr.v0)
                    vs[(size_t)k * total + off + i] = dr.v0[3 * (size_t)i + k];
            }
            dof[off + i] = d;
            e->h_type[off + i] = dr.type[i];
        }
        off += n;
    }
    // type-grouped order of every droplet: its types in order, each group in a
    // spatially compact order of the initial positions and padded with -1 to a multiple of 256
    std::vector<int> gperm, gtblk, gdblk;
    for (int d = 0; d < n_drops; ++d) {
        EnsDrop &g = e->h_drops[d];
        g.gpos0 = (int)gperm.size();
        for (int t = 0; t < drops[d].params.n_types; ++t) {
            std::vector<int> mem;
            for (int i = 0; i < e->cnt[d]; ++i)
                if (drops[d].type[i] == t)
                    mem.push_back(i);
            if (mem.empty())
                continue;
            spatial_sort(mem, drops[d].x0);
            for (int i : mem)
                gperm.push_back(e->off[d] + i);
            while (gperm.size() % 256)
                gperm.push_back(-1);
            while (gtblk.size() < gperm.size() / 256) {
                gtblk.push_back(t);
                gdblk.push_back(d);
            }
        }
        g.npad = (int)gperm.size() - g.gpos0;
    }
    e->n_pos = (int)gperm.size();
#define EBAIL(call)                                                                     \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return bail(set_err(e_ == cudaErrorMemoryAllocation ? NPSIM_ERR_OOM         \
                                                                 : NPSIM_ERR_CUDA,      \
                                "%s failed: %s", #call, cudaGetErrorString(e_)));       \
    } while (0)
    EBAIL(cudaStreamCreateWithFlags(&e->cap, cudaStreamNonBlocking));
    const size_t n3 = 3 * (size_t)total;
    EBAIL(dalloc(&e->x_lo, n3));
    EBAIL(dalloc(&e->v, n3));
    EBAIL(dalloc(&e->F, 2 * n3));
    EBAIL(dalloc(&e->F_tmp, 2 * n3));
    EBAIL(dalloc(&e->xq, (size_t)total));
    EBAIL(dalloc(&e->typ, (size_t)total));
    EBAIL(dalloc(&e->drop_of, (size_t)total));
    EBAIL(dalloc(&e->drops, (size_t)n_drops));
    EBAIL(dalloc(&e->tabs, (size_t)n_drops));
    EBAIL(dalloc(&e->F_pair, 8 * (size_t)total));
    EBAIL(dalloc(&e->d_work, 2));
    EBAIL(cudaMemsetAsync(e->d_work, 0, 2 * sizeof(unsigned), e->user));
    EBAIL(dalloc(&e->d_step, 1));
    EBAIL(dalloc(&e->d_spring, (size_t)2 * n_drops * NPSIM_MAX_TYPES));
    EBAIL(dalloc(&e->d_flags, 1));
    EBAIL(dalloc(&e->d_done, 1));
    {
        // position = hi (nearest float, in xq) + lo (the float nearest the rest)
        std::vector<float> lo(n3), vf(vs.begin(), vs.end());
        for (size_t k = 0; k < n3; ++k)
            lo[k] = (float)(xs[k] - (double)(float)xs[k]);
        EBAIL(cudaMemcpy(e->x_lo, lo.data(), sizeof(float) * n3, cudaMemcpyHostToDevice));
        EBAIL(cudaMemcpy(e->v, vf.data(), sizeof(float) * n3, cudaMemcpyHostToDevice));
    }
    EBAIL(cudaMemcpy(e->typ, e->h_type.data(), sizeof(int) * (size_t)total,
                     cudaMemcpyHostToDevice));
    EBAIL(cudaMemcpy(e->drop_of, dof.data(), sizeof(int) * (size_t)total,
                     cudaMemcpyHostToDevice));
    EBAIL(dalloc(&e->perm, gperm.size()));
    EBAIL(dalloc(&e->tblk, gtblk.size()));
    EBAIL(dalloc(&e->dblk, gdblk.size()));
    EBAIL(cudaMemcpy(e->perm, gperm.data(), sizeof(int) * gperm.size(), cudaMemcpyHostToDevice));
    EBAIL(cudaMemcpy(e->tblk, gtblk.data(), sizeof(int) * gtblk.size(), cudaMemcpyHostToDevice));
    EBAIL(cudaMemcpy(e->dblk, gdblk.data(), sizeof(int) * gdblk.size(), cudaMemcpyHostToDevice));
    EBAIL(cudaMemcpy(e->tabs, e->h_tabs.data(), sizeof(PairTab) * (size_t)n_drops,
                     cudaMemcpyHostToDevice));
    for (int i = 0; i < (int)total; ++i) {
        const int d = dof[i];
        const float q = (float)e->types[d][e->h_type[i]].charge;
        xq0[i] = make_float4((float)xs[i], (float)xs[total + i], (float)xs[2 * total + i], q);
    }
    EBAIL(cudaMemcpy(e->xq, xq0.data(), sizeof(float4) * (size_t)total, cudaMemcpyHostToDevice));
    EBAIL(cudaMemsetAsync(e->d_step, 0, sizeof(long long), e->user));
    {
        // spring radii of step 0 (buffer 0)
        std::vector<float4> sp((size_t)2 * n_drops * NPSIM_MAX_TYPES, make_float4(0, 0, 0, 0));
        for (int d = 0; d < n_drops; ++d)
            for (int t = 0; t < drops[d].params.n_types; ++t)
                sp[(size_t)d * NPSIM_MAX_TYPES + t] =
                    spring_entry(drops[d].params.R0, drops[d].params.k_evap, drops[d].params.dt,
                                 0, 0.5 * drops[d].types[t].sigma);
        EBAIL(cudaMemcpy(e->d_spring, sp.data(), sizeof(float4) * sp.size(),
                         cudaMemcpyHostToDevice));
    }
    EBAIL(cudaMemsetAsync(e->d_flags, 0, sizeof(int), e->user));
    EBAIL(cudaMemsetAsync(e->d_done, 0, sizeof(unsigned), e->user));
#undef EBAIL
    rc = ens_autotune(e);
    if (rc)
        return bail(rc);
    rc = ens_pass(e, MODE_FORCES, true, e->F, e->user);
    if (rc)
        return bail(rc);
    if (cudaStreamSynchronize(e->user) != cudaSuccess)
        return bail(set_err(NPSIM_ERR_CUDA, "initial forces failed"));
    *out = e;
    return NPSIM_OK;
}

void npsim_ens_destroy(npsim_ens_t e)
{
    NP_TRACE();
    if (!e)
        return;
    cudaStreamSynchronize(e->user);
    delete e;
}

int npsim_ens_step(npsim_ens_t e, int64_t n_steps)
{
    NP_TRACE();
    NP_REQUIRE(e, "ensemble is NULL");
    NP_REQUIRE(n_steps >= 0, "n_steps must be >= 0");
    int64_t rem = n_steps;
    while (rem > 0) {
        const int k = (int)std::min<int64_t>(rem, kChunk);
        cudaGraphExec_t ex = nullptr;
        int rc = ens_graph(e, k, &ex);
        if (rc)
            return rc;
        NP_CUDA(cudaGraphLaunch(ex, e->user));
        rem -= k;
        e->step += k;
        e->last_chunk = k;
    }
    int h = 0;
    NP_CUDA(cudaMemcpyAsync(&h, e->d_flags, sizeof(int), cudaMemcpyDeviceToHost, e->user));
    NP_CUDA(cudaStreamSynchronize(e->user));
    if (h) {
        NP_CUDA(cudaMemsetAsync(e->d_flags, 0, sizeof(int), e->user));
        if (!(h & FLAG_NONFINITE) && (h & FLAG_ESCAPED))
            return set_err(NPSIM_ERR_ESCAPED,
                           "an NP was farther than 2 max(R0, R(t)) from its droplet's centre");
        return set_err(NPSIM_ERR_NONFINITE, "a position became non-finite");
    }
    return NPSIM_OK;
}

int npsim_ens_profile(npsim_ens_t e, int enable)
{
    NP_REQUIRE(e, "ensemble is NULL");
    NP_CUDA(cudaStreamSynchronize(e->user));
    if (enable && !e->ev[0][0][0]) {
        for (auto &a : e->ev)
            for (auto &b : a)
                for (auto &x : b)
                    NP_CUDA(cudaEventCreate(&x));
    }
    if ((enable != 0) != e->profiling) {
        for (auto &g : e->graphs)
            cudaGraphExecDestroy(g.second);
        e->graphs.clear();
        e->profiling = enable != 0;
        e->last_chunk = 0;
    }
    return NPSIM_OK;
}

int npsim_ens_kernel_times(npsim_ens_t e, double *ms, int *samples)
{
    NP_REQUIRE(e && ms, "ensemble and ms are required");
    NP_REQUIRE(e->profiling, "profiling is not enabled (npsim_ens_profile)");
    NP_CUDA(cudaStreamSynchronize(e->user));
    const int k = e->last_chunk;
    for (int g = 0; g < 2; ++g) {
        double tot = 0.0;
        for (int j = 0; j < k; ++j) {
            float t = 0.f;
            NP_CUDA(cudaEventElapsedTime(&t, e->ev[j][g][0], e->ev[j][g][1]));
            tot += t;
        }
        ms[g] = k > 0 ? tot / k : 0.0;
    }
    if (samples)
        *samples = k;
    return NPSIM_OK;
}

int npsim_ens_get_state(npsim_ens_t e, int32_t d, double *x, double *v, double *F,
                        int64_t *step)
{
    NP_TRACE();
    NP_REQUIRE(e && d >= 0 && d < e->D, "bad ensemble or droplet index");
    if (x || v || F) {
        int rc = ens_state_out(e, d, e->F, x, v, F);
        if (rc)
            return rc;
    }
    if (step)
        *step = e->step;
    return NPSIM_OK;
}

int npsim_ens_forces(npsim_ens_t e, int32_t d, double *F)
{
    NP_TRACE();
    NP_REQUIRE(e && F && d >= 0 && d < e->D, "bad ensemble, droplet index or F");
    int rc = ens_pass(e, MODE_FORCES, true, e->F_tmp, e->user);
    if (rc)
        return rc;
    return ens_state_out(e, d, e->F_tmp, nullptr, nullptr, F);
}

int npsim_ens_stats(npsim_ens_t e, int32_t d, const npsim_stats_cfg_t *cfg, int64_t *rdf_counts,
                    double *rdf_g, int64_t *radial_counts, double *radial_c, npsim_stats_t *out)
{
    NP_TRACE();
    NP_REQUIRE(e && cfg && out && d >= 0 && d < e->D,
               "bad ensemble, droplet index, cfg or out");
    int rc = check_stats_cfg(cfg);
    if (rc)
        return rc;
    const int n = e->cnt[d], off = e->off[d];
    if (n > e->sw.x_cap) {
        dfree(e->sw.x);
        e->sw.x_cap = 0;
        NP_CUDA(dalloc(&e->sw.x, 3 * (size_t)n));
        e->sw.x_cap = n;
    }
    const npsim_params_t &p = e->P[d];
    const double t = (double)e->step * p.dt;
    const double R2 = p.R0 * p.R0 - p.k_evap * t;
    const double R = R2 > 0 ? std::sqrt(R2) : 0.0;
    // droplet d's positions (hi + lo) from the ensemble's state, on the device
    NP_CUDA(launch_positions_f64_ld(e->xq + off, e->x_lo + off, n, e->n_total, e->sw.x,
                                    e->user));
    rc = stats_core(e->sw, e->sw.x, e->xq + off, e->typ + off, n, R, e->d_mean[d],
                    e->types[d].data(), p.n_types, e->d_flags, cfg, rdf_counts, rdf_g,
                    radial_counts, radial_c, out, e->user);
    if (rc)
        return rc;
    int h = 0;
    NP_CUDA(cudaMemcpyAsync(&h, e->d_flags, sizeof(int), cudaMemcpyDeviceToHost, e->user));
    NP_CUDA(cudaStreamSynchronize(e->user));
    if (h) {
        NP_CUDA(cudaMemsetAsync(e->d_flags, 0, sizeof(int), e->user));
        return set_err(NPSIM_ERR_CUDA, "device error word 0x%x", h);
    }
    return NPSIM_OK;
}

int npsim_ens_config(npsim_ens_t e, int *block, int *i_per_thread, int *j_tile, int *grid,
                     int *index)
{
    NP_REQUIRE(e, "ensemble is NULL");
    const ApConfig c = ens_config(e->shape);
    if (block)
        *block = c.block;
    if (i_per_thread)
        *i_per_thread = c.ki;
    if (j_tile)
        *j_tile = c.jt;
    if (grid)
        *grid = e->ctas;
    if (index)
        *index = e->shape;
    return NPSIM_OK;
}

int npsim_ens_work(npsim_ens_t e, int64_t *n_items, int32_t *itile)
{
    NP_REQUIRE(e, "ensemble is NULL");
    if (n_items)
        *n_items = e->n_items;
    const ApConfig c = ens_config(e->shape);
    if (itile)
        *itile = c.block * c.ki;
    return NPSIM_OK;
}

int npsim_ens_info(npsim_ens_t e, int64_t *n_total, double *pairs_per_step)
{
    NP_REQUIRE(e, "ensemble is NULL");
    if (n_total)
        *n_total = e->n_total;
    if (pairs_per_step) {
        double p = 0.0;
        for (int d = 0; d < e->D; ++d)
            p += (double)e->cnt[d] * (double)(e->cnt[d] - 1);
        *pairs_per_step = p;
    }
    return NPSIM_OK;
}

} // extern "C"

// ---------------------------------------------------------------------------
// Test hooks

namespace {

__global__ void k_philox(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                         long long n_blocks, uint32_t *out)
{
    const long long b = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (b >= n_blocks)
        return;
    const unsigned long long lo = (unsigned long long)c0 + (unsigned long long)b;
    const U4 r = philox10(U4{(uint32_t)lo, c1 + (uint32_t)(lo >> 32), c2, c3}, (uint32_t)seed,
                          (uint32_t)(seed >> 32));
    out[4 * b + 0] = r.x;
    out[4 * b + 1] = r.y;
    out[4 * b + 2] = r.z;
    out[4 * b + 3] = r.w;
}

__global__ void k_normals(uint64_t seed, long long step, int n, double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    float a, b, c;
    normals3(seed, (uint32_t)i, step, 0u, a, b, c);
    out[3 * i + 0] = a;
    out[3 * i + 1] = b;
    out[3 * i + 2] = c;
}

} // namespace

extern "C" int npsim_philox(uint64_t seed, const uint32_t ctr[4], int64_t n_blocks,
                            uint32_t *out)
{
    NP_REQUIRE(ctr && out, "ctr and out are required");
    NP_REQUIRE(n_blocks >= 0 && n_blocks <= (1ll << 28), "n_blocks out of range");
    int rc = check_device(nullptr);
    if (rc)
        return rc;
    if (n_blocks == 0)
        return NPSIM_OK;
    uint32_t *d = nullptr;
    NP_CUDA(dalloc(&d, 4 * (size_t)n_blocks));
    k_philox<<<(unsigned)((n_blocks + 255) / 256), 256>>>(seed, ctr[0], ctr[1], ctr[2], ctr[3],
                                                          n_blocks, d);
    cudaError_t e = cudaMemcpy(out, d, sizeof(uint32_t) * 4 * (size_t)n_blocks,
                               cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "philox: %s", cudaGetErrorString(e));
    return NPSIM_OK;
}

extern "C" int npsim_normals(uint64_t seed, int64_t step, int64_t n, double *out)
{
    NP_REQUIRE(out, "out is required");
    NP_REQUIRE(n >= 0 && n <= (1ll << 29), "n out of range");
    int rc = check_device(nullptr);
    if (rc)
        return rc;
    if (n == 0)
        return NPSIM_OK;
    double *d = nullptr;
    NP_CUDA(dalloc(&d, 3 * (size_t)n));
    k_normals<<<(unsigned)((n + 255) / 256), 256>>>(seed, step, (int)n, d);
    cudaError_t e = cudaMemcpy(out, d, sizeof(double) * 3 * (size_t)n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess)
        return set_err(NPSIM_ERR_CUDA, "normals: %s", cudaGetErrorString(e));
    return NPSIM_OK;
}
