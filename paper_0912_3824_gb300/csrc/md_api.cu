// md_api.cu -- host implementation of the C ABI declared in include/md.h.
//
// The handle carves every device array out of the caller's workspace, keeps
// the per-replica tables there, and drives the kernels on the caller's stream.
// md_step() is one cooperative launch of the run kernel (md_kernels.cuh): the
// half kick and drift that open it, the MD steps, and the list rebuilds that
// the displacements call for, all decided on the device, so a whole md_step of
// n steps needs no host round trip.  With use_graph = 0 the same kernel is
// launched once per phase (each step, each rebuild) with its time taken (the
// results are bitwise identical).
#include <cuda.h>
#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "md.h"
#include "md_bench.h"
#include "md_tables.h"
#include "md_common.cuh"
#include "md_corr.cuh"

static_assert(sizeof(md_params) == 192, "md_params layout is part of the ABI");

using mdk::KArgs;
using mdk::KernelSet;

// md_noalloc.cu: message of the calling thread's last failed handle-free call
const char *md_noalloc_message();

namespace {
// A named range on a profiler's host timeline for the duration of one API call
// (NVTX; costs nothing when no tool is attached).
struct ApiRange {
    explicit ApiRange(const char *name) { nvtxRangePushA(name); }
    ~ApiRange() { nvtxRangePop(); }
    ApiRange(const ApiRange &) = delete;
    ApiRange &operator=(const ApiRange &) = delete;
};
}  // namespace

namespace {

constexpr size_t kAlign = 256;
constexpr int kIntBlock = 256, kForceBlock = 128;
constexpr int kMaxRunGroups = 4096;    // bound on the run kernel's groups (entries of KArgs::slice)
constexpr int kNbWarpCellsPerSm = 8;                     // warp-per-cell build from this many cells per SM
constexpr double kCellMargin = 1e-3;   // cell edge exceeds the largest list radius by this
constexpr int kUnroll = 16;            // largest check interval
constexpr int kCheck = 4;              // automatic check interval below kCheckLargeN particles
constexpr int64_t kCheckLargeN = 262144;   // from here a check after every step

size_t align_up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// Everything that follows from the parameters and the replica sizes.
struct Geometry {
    int R = 0;
    int64_t n = 0;
    int K = 0, Kmax = 0, tpp = 8, ppb_f = 32;   // starting list capacity, its cap
    int check = kCheck;                 // MD steps between rebuild checks
    bool nb_block = false;              // neighbour build by groups of threads
    int nblk_i = 0, nblk_f = 0, ncell = 0;
    bool sweep = false;                 // step_form as reported: more chunks than groups
    int groups = 1, nwork = 0, cpb = 1; // run kernel: groups per block, groups with chunks, chunks per group
    double rl_max = 0.0;
    std::vector<mdk::Rep> rep;
    std::vector<int4> blk_i, blk_f;
    std::vector<int> crank;
    std::vector<int4> cxyz;
};

struct Layout {
    size_t off_ctl, off_rep, off_blk_i, off_blk_r, off_crank, off_cxyz;
    size_t off_pa, off_pb, off_va, off_vb, off_pa2, off_pb2, off_va2, off_vb2, off_qa, off_qb, off_force;
    size_t off_rref, off_image, off_image2, off_key, off_tmpidx;
    size_t off_ccount, off_ccursor, off_cstart, off_nbr, off_nnbr, off_part_f, off_part_i, off_part_e;
    size_t off_ring, off_totals, off_scale, off_st_pos, off_st_vel, off_st_img, off_st_code;
    size_t off_epot, off_epot_step, off_rs, off_slice;
    size_t off_st_f, off_st_e, total;
};

int prec_pos_bytes(int prec) { return prec == MD_PREC_FP64 ? 32 : 16; }

// Index of cell (x, y, z) along the Hilbert curve through a 2^b cube: the
// coordinates are transformed in place (Skilling's transposition method,
// "Programming the Hilbert curve", AIP Conf. Proc. 707, 2004), then their bits
// are interleaved, most significant first.
uint32_t hilbert3(uint32_t x, uint32_t y, uint32_t z, int b)
{
    uint32_t X[3] = {x, y, z};
    const uint32_t top = 1u << (b - 1);
    for (uint32_t q = top; q > 1; q >>= 1) {
        const uint32_t low = q - 1;
        for (int i = 0; i < 3; ++i) {
            if (X[i] & q) {
                X[0] ^= low;                          // reflect the lower bits of axis 0
            } else {
                const uint32_t t = (X[0] ^ X[i]) & low;   // exchange them with axis i
                X[0] ^= t;
                X[i] ^= t;
            }
        }
    }
    X[1] ^= X[0];                                     // Gray code across the axes
    X[2] ^= X[1];
    uint32_t t = 0;
    for (uint32_t q = top; q > 1; q >>= 1)
        if (X[2] & q)
            t ^= q - 1;
    for (int i = 0; i < 3; ++i)
        X[i] ^= t;
    uint32_t h = 0;
    for (int k = b - 1; k >= 0; --k)
        for (int i = 0; i < 3; ++i)
            h = (h << 1) | ((X[i] >> k) & 1u);
    return h;
}

uint32_t spread3(uint32_t v)
{
    uint32_t r = 0;
    for (int b = 0; b < 10; ++b)
        r |= ((v >> b) & 1u) << (3 * b);
    return r;
}

int auto_capacity(const md_params *p, const Geometry &g, const std::vector<double> &box,
                  const std::vector<int64_t> &nrep)
{
    double rho = 0.0;
    for (size_t r = 0; r < box.size(); ++r)
        rho = std::max(rho, (double)nrep[r] / (box[r] * box[r] * box[r]));
    const double nl = 4.18879020478639 * g.rl_max * g.rl_max * g.rl_max * rho;   // 4/3 pi r^3 rho
    int k = (int)std::ceil(1.35 * nl + 24.0);
    k = (k + 31) / 32 * 32;
    (void)p;
    return std::max(k, 32);
}

// Automatic lanes per particle.  From ~12,000 particles on (FP64: ~6,500) the
// work fills the GPU and 2 lanes (4) lose least to combining them; fewer particles
// leave it idle, and more lanes shorten the chain of a row's entries, as long as
// rows are long enough to share.  Measured on GB300, us per MD step:
//   KA mixed, N = 1000: 9.57 (2 lanes) 8.60 (4) 7.30 (8) 7.28 (16); 6000: 10.48 10.56
//     8.81 9.26; 10,000: 11.25 11.20 9.93 -; 12,000: 11.15 11.83 10.78 -; 14,000: 11.30
//     11.78 11.54 -; 16,384: 11.43 11.67 11.92 -; 20,000: 13.19 13.35 16.18 -
//     (so the lines of 2 and 8 lanes cross between 12,000 and 14,000)
//   LJ 0.8442 mixed, N = 2000: 9.51 9.49 9.13 9.06; 8000: 11.21 11.30 11.12 12.00
//   LJ 0.3 mixed (~28 entries a row), N = 2000: 7.98 8.65 8.56 8.38
//   KA smoothed, N = 1000: 12.90 9.89 7.68 (8); 12,000: 14.88 12.47 12.04; 24,000: 17.26 16.52 -
//   KA FP64, N = 1000: 68.8 36.5 23.5 18.5; 4000: 69.4 37.4 33.6 43.5; 8000: 69.8 54.6 59.1 70.8
//   KA FP64 smoothed, N = 1000: 138 74.8 43.0 (8); 4000: 138 74.8 63.8; 8000: 140 115 115
//     (4 lanes at every size: 8 would be faster below ~6,000)
int auto_lanes(const md_params *p, int R, const int64_t *nrep, const double *box, double rl)
{
    double n = 0.0, vol = 0.0;
    for (int r = 0; r < R; ++r) {
        n += (double)nrep[r];
        vol += box[r] * box[r] * box[r];
    }
    const bool longrow = 4.18879020478639 * rl * rl * rl * n > 48.0 * vol;   // entries a row on average
    if (p->precision == MD_PREC_FP64)
        return p->smooth_h > 0.0 || !longrow || n > 6500 ? 4 : n > 1200 ? 8 : 16;
    if (p->step_form == 2 || !longrow)
        return 2;
    if (p->smooth_h > 0.0)
        return n > 24000 ? 2 : n > 12000 ? 4 : 8;
    return n > 12000 ? 2 : n > 2048 ? 8 : 16;
}

// Returns MD_OK or MD_E_INVAL with *msg set.
int make_geometry(const md_params *p, int R, const int64_t *nrep, const double *box, Geometry &g,
                  std::string &msg)
{
    if (!p || R < 1 || !nrep || !box) {
        msg = "null argument or n_replicas < 1";
        return MD_E_INVAL;
    }
    if (p->n_species < 1 || p->n_species > 2) { msg = "n_species must be 1 or 2"; return MD_E_INVAL; }
    if (!(p->dt > 0.0) || !std::isfinite(p->dt)) { msg = "dt must be positive"; return MD_E_INVAL; }
    if (!(p->skin >= 0.0)) { msg = "skin must be >= 0"; return MD_E_INVAL; }
    if (p->precision < 0 || p->precision > 2) { msg = "unknown precision mode"; return MD_E_INVAL; }
    if (p->sample_interval < 1) { msg = "sample_interval must be >= 1"; return MD_E_INVAL; }
    const int tpp = p->threads_per_particle;
    if (tpp != 0 && (tpp < 1 || tpp > 32 || (tpp & (tpp - 1)))) {
        msg = "threads_per_particle must be 0 or a power of two in [1, 32]";
        return MD_E_INVAL;
    }
    if (p->step_form < 0 || p->step_form > 2) {
        msg = "step_form must be 0 (automatic), 1 or 2";
        return MD_E_INVAL;
    }
    if (p->build_form < 0 || p->build_form > 2) {
        msg = "build_form must be 0 (automatic), 1 (warp per cell) or 2 (groups of threads per cell)";
        return MD_E_INVAL;
    }
    if (p->neigh_capacity < 0 || p->neigh_capacity_max < 0) {
        msg = "neigh_capacity and neigh_capacity_max must be >= 0";
        return MD_E_INVAL;
    }
    if (p->step_budget < 0) { msg = "step_budget must be >= 0"; return MD_E_INVAL; }
    {
        const int ci = p->check_interval;
        if (ci != 0 && (ci < 1 || ci > kUnroll || (ci & (ci - 1)) || kUnroll % ci)) {
            msg = "check_interval must be 0 (automatic) or 1, 2, 4, 8 or 16";
            return MD_E_INVAL;
        }
    }
    if (!(p->smooth_h >= 0.0) || !std::isfinite(p->smooth_h)) {
        msg = "smooth_h must be finite and >= 0";
        return MD_E_INVAL;
    }
    if (p->reorder < 0 || p->reorder > 2) {
        msg = "reorder must be 0 (x-fastest), 1 (Morton) or 2 (Hilbert)";
        return MD_E_INVAL;
    }
    if (p->smooth_h > 0.0 && tpp > 8) {
        msg = "threads_per_particle above 8 is not available with the smoothed potential";
        return MD_E_INVAL;
    }
    const int ns = p->n_species;
    double rcmax = 0.0;
    for (int a = 0; a < ns; ++a) {
        if (!(p->mass[a] > 0.0)) { msg = "masses must be positive"; return MD_E_INVAL; }
        for (int b = 0; b < ns; ++b) {
            if (p->eps[a][b] != p->eps[b][a] || p->sigma[a][b] != p->sigma[b][a] ||
                p->rcut[a][b] != p->rcut[b][a]) {
                msg = "pair parameters must be symmetric";
                return MD_E_INVAL;
            }
            if (!(p->sigma[a][b] > 0.0) || !(p->rcut[a][b] > 0.0)) {
                msg = "sigma and rcut must be positive";
                return MD_E_INVAL;
            }
            rcmax = std::max(rcmax, p->rcut[a][b]);
        }
    }
    g.R = R;
    g.rl_max = rcmax + p->skin + (double)mdk::kListMargin;
    g.tpp = tpp ? tpp : auto_lanes(p, R, nrep, box, g.rl_max);
    g.ppb_f = kForceBlock / g.tpp;
    if (p->step_form == 2 && (p->precision == MD_PREC_FP64 || g.tpp > 2)) {
        msg = "step_form 2 needs MIXED or FP32 and 1 or 2 threads per particle";
        return MD_E_INVAL;
    }
    g.n = 0;
    g.rep.assign(R, mdk::Rep{});
    g.blk_i.clear();
    g.blk_f.clear();
    g.crank.clear();
    g.cxyz.clear();
    int cell0 = 0;
    for (int r = 0; r < R; ++r) {
        const double L = box[r];
        if (nrep[r] < 2) { msg = "every replica needs at least 2 particles"; return MD_E_INVAL; }
        if (!(L > 2.0 * g.rl_max)) {
            char b[160];
            snprintf(b, sizeof b, "box %d (L = %g) must exceed twice the largest cutoff plus skin (%g)",
                     r, L, 2.0 * g.rl_max);
            msg = b;
            return MD_E_INVAL;
        }
        if (g.n + nrep[r] > (int64_t)(1 << 30)) { msg = "too many particles"; return MD_E_INVAL; }
        mdk::Rep &q = g.rep[r];
        q.start = (int)g.n;
        q.n = (int)nrep[r];
        int nc = (int)std::floor(L / (g.rl_max + kCellMargin));
        if (nc < 3)
            nc = 1;
        if (nc > 1024)
            nc = 1024;
        q.nc = nc;
        q.cell0 = cell0;
        q.L = L;
        q.invL = 1.0 / L;
        q.cscale = nc / L;
        q.invLf = (float)(1.0 / L);
        q.cscalef = (float)(nc / L);
        q.qunit = (float)(L / 4294967296.0);
        q.qscale = (float)(4294967296.0 / L);
        // anchoring grid: smallest power of two with 2L < 2^24 * grid
        int e = (int)std::ceil(std::log2(2.0 * L)) - 24;
        double grid = std::ldexp(1.0, e);
        while (2.0 * L >= grid * 16777216.0)
            grid *= 2.0;
        q.grid = (float)grid;
        q.inv_grid = (float)(1.0 / grid);
        // grid * 2^32 / L lies in (2^9, 2^10]: times 2^28 it fits 38 bits, and times the
        // anchored high word's grid index (< 2^24) 62 bits
        q.qgrid = (unsigned long long)std::llround(grid * 4294967296.0 / L * 268435456.0);
        if (p->precision == MD_PREC_MIXED) {
            const double lh = std::rint(L / grid) * grid;
            q.Lhi = (float)lh;
            q.Llo = (float)(L - lh);
        } else {
            q.Lhi = (float)L;
            q.Llo = (float)(L - (double)(float)L);
        }
        // integrate-kernel blocks
        q.bi0 = (int)g.blk_i.size();
        for (int s = 0; s < q.n; s += kIntBlock)
            g.blk_i.push_back(make_int4(q.start + s, q.start + std::min(q.n, s + kIntBlock), r, 0));
        q.bi1 = (int)g.blk_i.size();
        q.bf0 = (int)g.blk_f.size();
        for (int s = 0; s < q.n; s += g.ppb_f)
            g.blk_f.push_back(make_int4(q.start + s, q.start + std::min(q.n, s + g.ppb_f), r, 0));
        q.bf1 = (int)g.blk_f.size();
        // cells, ordered along a Morton curve, a Hilbert curve (the curve of the
        // paper's reorder, Sec. 2.2) through the enclosing 2^b cube, or x-fastest
        const int nc3 = nc * nc * nc;
        int bits = 1;
        while ((1 << bits) < nc)
            ++bits;
        std::vector<std::pair<uint32_t, int>> order(nc3);
        for (int lin = 0; lin < nc3; ++lin) {
            const int cx = lin % nc, cy = (lin / nc) % nc, cz = lin / (nc * nc);
            uint32_t code = (uint32_t)lin;
            if (p->reorder == 1)
                code = spread3(cx) | (spread3(cy) << 1) | (spread3(cz) << 2);
            else if (p->reorder == 2)
                code = hilbert3(cx, cy, cz, bits);
            order[lin] = {code, lin};
        }
        std::sort(order.begin(), order.end());
        g.crank.resize(cell0 + nc3);
        g.cxyz.resize(cell0 + nc3);
        for (int rank = 0; rank < nc3; ++rank) {
            const int lin = order[rank].second;
            g.crank[cell0 + lin] = cell0 + rank;
            g.cxyz[cell0 + rank] = make_int4(lin % nc, (lin / nc) % nc, lin / (nc * nc), r);
        }
        cell0 += nc3;
        g.n += nrep[r];
    }
    g.ncell = cell0;
    g.nblk_i = (int)g.blk_i.size();
    g.nblk_f = (int)g.blk_f.size();
    std::vector<double> bx(box, box + R);
    std::vector<int64_t> nr(nrep, nrep + R);
    g.K = p->neigh_capacity > 0 ? (p->neigh_capacity + 7) / 8 * 8 : auto_capacity(p, g, bx, nr);
    g.Kmax = p->neigh_capacity_max > 0 ? (p->neigh_capacity_max + 7) / 8 * 8 : 2 * g.K;
    if (g.Kmax < g.K) {
        msg = "neigh_capacity_max must be 0 or at least neigh_capacity";
        return MD_E_INVAL;
    }
    if ((double)g.n * (double)g.Kmax > 4.0e12) { msg = "neighbour-list cap too large"; return MD_E_INVAL; }
    g.check = p->check_interval > 0 ? p->check_interval : (g.n >= kCheckLargeN ? 1 : kCheck);
    return MD_OK;
}

Layout make_layout(const md_params *p, const Geometry &g)
{
    Layout L;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + std::max<size_t>(bytes, 1)); return r; };
    const size_t n = (size_t)g.n;
    const size_t pb = prec_pos_bytes(p->precision);
    const bool mixed = p->precision == MD_PREC_MIXED;
    const int cap = p->obs_capacity > 0 ? p->obs_capacity : 4096;
    L.off_ctl = take(sizeof(mdk::Ctl));
    L.off_rep = take(sizeof(mdk::Rep) * g.R);
    L.off_blk_i = take(sizeof(int4) * g.nblk_i);
    L.off_blk_r = take(sizeof(int4) * 2 * (size_t)g.nblk_f);   // < nblk_f + groups rows
    L.off_rs = take(sizeof(mdk::RunSync));
    L.off_slice = take(sizeof(int) * kMaxRunGroups);
    L.off_crank = take(sizeof(int) * g.ncell);
    L.off_cxyz = take(sizeof(int4) * g.ncell);
    L.off_pa = take(pb * n);
    L.off_pb = take(mixed ? 16 * n : 0);
    L.off_va = take(pb * n);
    L.off_vb = take(mixed ? 16 * n : 0);
    L.off_pa2 = take(pb * n);
    L.off_pb2 = take(mixed ? 16 * n : 0);
    L.off_qa = take(mixed ? 16 * n : 0);
    L.off_qb = take(mixed ? 16 * n : 0);
    L.off_va2 = take(pb * n);
    L.off_vb2 = take(mixed ? 16 * n : 0);
    L.off_force = take(pb * n);
    L.off_rref = take(16 * n);
    L.off_image = take(16 * n);
    L.off_image2 = take(16 * n);
    L.off_key = take(8 * n);
    L.off_tmpidx = take(8 * n);
    L.off_ccount = take(4 * (size_t)g.ncell);
    L.off_ccursor = take(4 * (size_t)g.ncell);
    L.off_cstart = take(4 * ((size_t)g.ncell + 1));
    L.off_nbr = take(4 * n * (size_t)g.Kmax);       // room for the cap: K grows in place
    L.off_nnbr = take(4 * n);
    L.off_part_f = take(2 * 8 * 12 * (size_t)g.nblk_f);        // (2 parities)
    L.off_part_i = take(8 * 4 * (size_t)g.nblk_i);
    L.off_part_e = take(2 * 8 * (size_t)g.nblk_f);
    L.off_ring = take(sizeof(mdk::Obs) * (size_t)cap * g.R);
    L.off_epot = take(sizeof(double) * (size_t)cap * g.R);
    L.off_epot_step = take(sizeof(long long) * (size_t)cap);
    L.off_totals = take(sizeof(mdk::Obs) * g.R);
    L.off_scale = take(8 * (size_t)g.R);
    L.off_st_pos = take(24 * n);
    L.off_st_vel = take(24 * n);
    L.off_st_img = take(12 * n + 4);                // (and a word: is the state lost)
    L.off_st_code = take(4 * n);
    L.off_st_f = take(24 * n);
    L.off_st_e = take(8 * n);
    L.total = o;
    return L;
}

const KernelSet &kernel_set(int prec)
{
    if (prec == MD_PREC_FP64)
        return mdk::kernels_fp64();
    if (prec == MD_PREC_FP32)
        return mdk::kernels_fp32();
    return mdk::kernels_mixed();
}

int force_index(int tpp)
{
    int k = 0;
    while ((1 << k) < tpp)
        ++k;
    return k;
}

}  // namespace

struct md_handle {
    md_params p;
    Geometry g;
    Layout lay;
    cudaStream_t s = nullptr;
    char *ws = nullptr;
    KArgs a;
    const KernelSet *ks = nullptr;
    int nsm = 0;                     // blocks of the run kernel: one per SM that the stream can have
    const void *runk = nullptr;      // the run kernel in use: precision, lanes per particle, smoothing
    int cap = 4096;
    // pinned host staging
    char *pin = nullptr;
    size_t pin_bytes = 0;
    cudaEvent_t ev_stage = nullptr;
    // timing of the run kernel's phases (use_graph = 0)
    cudaEvent_t ev_f0 = nullptr, ev_f1 = nullptr, ev_i1 = nullptr;
    double step_ms = 0.0, rebuild_ms = 0.0;
    int64_t step_launches = 0, rebuild_checks = 0;
    int64_t obs_read = 0;
    int64_t epot_read = -1;          // newest step returned by md_epot_series
    int64_t n_species[2] = {0, 0};   // particles per species over all replicas
    bool stale = false, lost = false;   // reported with a status and not mended yet: Ctl::stale
    std::string err;
};

namespace {

int fail(md_handle *h, int code, const std::string &m)
{
    if (h)
        h->err = m;
    return code;
}

int cuda_fail(md_handle *h, cudaError_t e, const char *what)
{
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    return fail(h, MD_E_CUDA, m);
}

#define CK(h, expr)                                   \
    do {                                              \
        cudaError_t e_ = (expr);                      \
        if (e_ != cudaSuccess)                        \
            return cuda_fail((h), e_, #expr);         \
    } while (0)

int launch(md_handle *h, const void *f, int grid, int block, const KArgs &a)
{
    if (grid <= 0)
        return MD_OK;
    void *pp[1] = {(void *)&a};
    CK(h, cudaLaunchKernel(f, dim3((unsigned)grid), dim3((unsigned)block), pp, 0, h->s));
    return MD_OK;
}

// SMs that launches on stream s can have: all of the device's, or those of the
// green context that the stream (or, for a default stream, the current context)
// belongs to.  The run kernel's blocks must all be resident, one per SM.
int stream_sms(cudaStream_t s, int device_sms)
{
    const auto entry = [](const char *name) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion(name, &fn, 12040, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        return fn;
    };
    CUdevResource r;
    memset(&r, 0, sizeof r);
    CUgreenCtx green = nullptr;
    CUcontext ctx = nullptr;
    bool known = false;
    if (s && s != cudaStreamLegacy && s != cudaStreamPerThread) {
        const auto of_stream = (CUresult(*)(CUstream, CUgreenCtx *))entry("cuStreamGetGreenCtx");
        const auto of_green = (CUresult(*)(CUgreenCtx, CUdevResource *, CUdevResourceType))entry("cuGreenCtxGetDevResource");
        if (of_stream && of_green && of_stream(s, &green) == CUDA_SUCCESS && green)
            known = of_green(green, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS;
    }
    if (!green) {
        const auto current = (CUresult(*)(CUcontext *))entry("cuCtxGetCurrent");
        const auto of_ctx = (CUresult(*)(CUcontext, CUdevResource *, CUdevResourceType))entry("cuCtxGetDevResource");
        known = current && of_ctx && current(&ctx) == CUDA_SUCCESS && ctx &&
                of_ctx(ctx, &r, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS;
    }
    const int n = known ? (int)r.sm.smCount : 0;
    return n > 0 && n < device_sms ? n : device_sms;
}

int grid_n(int64_t n, int per) { return (int)((n + per - 1) / per); }

// One launch of the run kernel: what it does (mdk::RUN_*), steps and their
// place in the md_step.
int launch_run(md_handle *h, int what, int64_t nsteps = 0, int64_t budget = 0, int pos0 = 0, bool last = true)
{
    KArgs a = h->a;
    a.what = what;
    a.nsteps = nsteps;
    a.budget = budget;
    a.pos0 = pos0;
    a.last = last ? 1 : 0;
    void *pp[1] = {(void *)&a};
    CK(h, cudaLaunchCooperativeKernel(h->runk, dim3((unsigned)h->nsm), dim3((unsigned)(kForceBlock * h->g.groups)), pp,
                                      (size_t)h->g.groups * (size_t)h->ks->group_smem, h->s));
    return MD_OK;
}

int launch_kinetic(md_handle *h, int mode)
{
    KArgs a = h->a;
    a.imode = mode;
    return launch(h, h->ks->kinetic, h->g.nblk_i, kIntBlock, a);
}

int stage_wait(md_handle *h)
{
    CK(h, cudaEventSynchronize(h->ev_stage));
    return MD_OK;
}

int ensure_pinned(md_handle *h, size_t bytes)
{
    if (bytes <= h->pin_bytes)
        return MD_OK;
    int rc = stage_wait(h);
    if (rc)
        return rc;
    CK(h, cudaStreamSynchronize(h->s));
    if (h->pin)
        cudaFreeHost(h->pin);
    h->pin = nullptr;
    h->pin_bytes = 0;
    CK(h, cudaMallocHost((void **)&h->pin, bytes));
    h->pin_bytes = bytes;
    return MD_OK;
}

int read_ctl(md_handle *h, mdk::Ctl *out)
{
    int rc = ensure_pinned(h, sizeof(mdk::Ctl));
    if (rc)
        return rc;
    if ((rc = stage_wait(h)))
        return rc;
    CK(h, cudaMemcpyAsync(h->pin, h->a.ctl, sizeof(mdk::Ctl), cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaStreamSynchronize(h->s));
    memcpy(out, h->pin, sizeof(mdk::Ctl));
    return MD_OK;
}

// Stream-launch mode: launch the rebuild if the device flag asks for it (waits
// for the stream); adds its CUDA-event time to *ms when given.
int rebuild_if_flagged(md_handle *h, float *ms)
{
    mdk::Ctl c;
    int rc = read_ctl(h, &c);
    if (rc)
        return rc;
    if (!c.rebuild || c.status)
        return MD_OK;
    CK(h, cudaEventRecord(h->ev_f1, h->s));
    if ((rc = launch_run(h, mdk::RUN_REBUILD)))
        return rc;
    CK(h, cudaEventRecord(h->ev_i1, h->s));
    CK(h, cudaEventSynchronize(h->ev_i1));
    if (ms)
        CK(h, cudaEventElapsedTime(ms, h->ev_f1, h->ev_i1));
    h->rebuild_checks += 1;
    return MD_OK;
}

int status_code(unsigned st)
{
    if (st & mdk::ST_NONFINITE) return MD_E_NONFINITE;
    if (st & mdk::ST_UNSTABLE) return MD_E_UNSTABLE;
    if (st & mdk::ST_OVERFLOW) return MD_E_CAPACITY;
    if (st & mdk::ST_TIMEOUT) return MD_E_TIMEOUT;
    if (st & mdk::ST_BOUNDS) return MD_E_BOUNDS;
    return MD_OK;
}

const char *status_message(int code)
{
    switch (code) {
    case MD_E_NONFINITE: return "a position became non-finite; the step loop stopped";
    case MD_E_UNSTABLE: return "a particle moved more than a quarter box in one step; the step loop stopped";
    case MD_E_CAPACITY: return "a neighbour list exceeded neigh_capacity_max; the step loop stopped";
    case MD_E_BOUNDS: return "an index left its array (bounds-checked build); the access was redirected";
    case MD_E_TIMEOUT: return "the device step loop exceeded its iteration bound";
    default: return "";
    }
}

constexpr const char *kLostMessage = "a wait of the step kernel for its other blocks gave up: the state is lost "
                                     "until md_set_state";

// Synchronise, report (once) and clear a device status.  (A launch that gave up
// may have left counts of a binning that never ended.)
int check_device(md_handle *h)
{
    mdk::Ctl c;
    int rc = read_ctl(h, &c);
    if (rc)
        return rc;
    const int code = status_code(c.status);
    if (code != MD_OK) {
        KArgs a = h->a;
        if ((rc = launch(h, h->ks->reset, 1, 1, a)))
            return rc;
        CK(h, cudaMemsetAsync(h->a.ccount, 0, 4 * (size_t)h->g.ncell, h->s));
        CK(h, cudaStreamSynchronize(h->s));
        h->stale = (c.stale & mdk::STALE_LISTS) != 0;
        h->lost = (c.stale & mdk::STALE_STATE) != 0;
        return fail(h, code, h->lost ? kLostMessage : status_message(code));
    }
    return MD_OK;
}

int lost(md_handle *h) { return h->lost ? fail(h, MD_E_TIMEOUT, kLostMessage) : MD_OK; }

// After a failure that left lists of another order or a state loaded while the
// failure was pending: lists and forces of the current state.
int refresh(md_handle *h)
{
    if (!h->stale)
        return MD_OK;
    h->stale = false;
    return launch_run(h, mdk::RUN_REBUILD | mdk::RUN_FORCES);
}

// Copies between the caller's arrays and the pinned staging area, shared out
// over a few threads where they are large: one core moves ~15 GB/s into fresh
// pages (first touch) and ~28 GB/s into warm ones, well below the link to the
// GPU.  (get_state at N = 1,048,576, 63 MB: 4.9 ms by one thread.)
struct CopyJob { void *dst; const void *src; size_t bytes; };

constexpr size_t kCopyShare = 1u << 20;    // bytes a thread is worth starting for
constexpr int kCopyThreads = 8;

void copy_jobs(const CopyJob *job, int njob)
{
    size_t total = 0;
    for (int k = 0; k < njob; ++k)
        total += job[k].bytes;
    const unsigned hw = std::thread::hardware_concurrency();
    const size_t nt = std::min<size_t>({total / kCopyShare, (size_t)kCopyThreads, (size_t)std::max(1u, hw / 2)});
    // part t of n: bytes [total t / n, total (t + 1) / n) of the jobs laid end to end
    const auto part = [&](size_t t, size_t n) {
        const size_t b0 = total / n * t, b1 = t + 1 == n ? total : total / n * (t + 1);
        size_t at = 0;
        for (int k = 0; k < njob; ++k) {
            const size_t lo = std::max(b0, at), hi = std::min(b1, at + job[k].bytes);
            if (lo < hi)
                memcpy((char *)job[k].dst + (lo - at), (const char *)job[k].src + (lo - at), hi - lo);
            at += job[k].bytes;
        }
    };
    if (nt < 2) {
        part(0, 1);
        return;
    }
    std::thread th[kCopyThreads];
    size_t started = 1;
    try {
        for (; started < nt; ++started)
            th[started] = std::thread(part, started, nt);
    } catch (...) {                        // (no more threads to be had: their parts are done here)
    }
    part(0, nt);
    for (size_t t = started; t < nt; ++t)
        part(t, nt);
    for (size_t t = 1; t < started; ++t)
        th[t].join();
}

// Copy the caller's state into pinned staging, upload it, load it into the
// working layout, rebuild, evaluate forces and record them as a sample.
int upload_state(md_handle *h, const int32_t *species, const double *pos, const double *vel,
                 const int32_t *image)
{
    const size_t n = (size_t)h->g.n;
    const size_t bytes = 24 * n + 24 * n + 12 * n + 4 * n;
    int rc = ensure_pinned(h, bytes);
    if (rc)
        return rc;
    if ((rc = stage_wait(h)))
        return rc;
    char *q = h->pin;
    const CopyJob in[4] = {{q, pos, 24 * n},
                           {q + 24 * n, vel, vel ? 24 * n : 0},
                           {q + 48 * n, image, image ? 12 * n : 0},
                           {q + 60 * n, species, 4 * n}};
    copy_jobs(in, 4);
    if (!vel)
        memset(q + 24 * n, 0, 24 * n);
    if (!image)
        memset(q + 48 * n, 0, 12 * n);
    CK(h, cudaMemcpyAsync(h->a.st_pos, q, 24 * n, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaMemcpyAsync(h->a.st_vel, q + 24 * n, 24 * n, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaMemcpyAsync(h->a.st_img, q + 48 * n, 12 * n, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaMemcpyAsync(h->a.st_code, q + 60 * n, 4 * n, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaEventRecord(h->ev_stage, h->s));
    if ((rc = launch(h, h->ks->load, h->g.nblk_i, kIntBlock, h->a)))
        return rc;
    return launch_run(h, mdk::RUN_REBUILD | mdk::RUN_SAMPLE);
}

}  // namespace

extern "C" {

int md_params_default(md_params *p)
{
    if (!p)
        return MD_E_INVAL;
    memset(p, 0, sizeof *p);
    p->n_species = 1;
    p->shift = 1;
    for (int a = 0; a < 2; ++a) {
        for (int b = 0; b < 2; ++b) {
            p->eps[a][b] = 1.0;
            p->sigma[a][b] = 1.0;
            p->rcut[a][b] = 2.5;
        }
        p->mass[a] = 1.0;
    }
    p->dt = 0.005;
    p->skin = 0.3;
    p->precision = MD_PREC_MIXED;
    p->sample_interval = 100;
    p->use_graph = 1;
    p->reorder = 1;
    return MD_OK;
}

int md_cell_order(const md_params *p, int32_t n_replicas, const int64_t *n_per_replica, const double *box,
                  int32_t *rank, int32_t *cells_per_edge)
{
    Geometry g;
    std::string msg;
    int rc = make_geometry(p, n_replicas, n_per_replica, box, g, msg);
    if (rc)
        return rc;
    const int nc = g.rep[0].nc;
    if (cells_per_edge)
        *cells_per_edge = nc;
    if (rank)
        for (int lin = 0; lin < nc * nc * nc; ++lin)
            rank[lin] = g.crank[lin];
    return MD_OK;
}

int md_workspace_size(const md_params *p, int32_t n_replicas, const int64_t *n_per_replica,
                      const double *box, size_t *bytes)
{
    if (!bytes)
        return MD_E_INVAL;
    Geometry g;
    std::string msg;
    int rc = make_geometry(p, n_replicas, n_per_replica, box, g, msg);
    if (rc)
        return rc;
    *bytes = make_layout(p, g).total;
    return MD_OK;
}

static int create_impl(md_handle *h, const md_params *p, const int32_t *species, const double *pos,
                       const double *vel, const int32_t *image, void *workspace, size_t workspace_bytes,
                       void *cuda_stream)
{
    int rc;
    h->p = *p;
    h->lay = make_layout(p, h->g);
    if (!species || !pos || !workspace || ((uintptr_t)workspace % kAlign) != 0)
        return fail(h, MD_E_INVAL, "null array or workspace not 256-byte aligned");
    if (workspace_bytes < h->lay.total)
        return fail(h, MD_E_NOMEM, "workspace smaller than md_workspace_size()");
    for (int64_t i = 0; i < h->g.n; ++i)
        if (species[i] < 0 || species[i] >= p->n_species)
            return fail(h, MD_E_INVAL, "species out of range");
    for (int64_t i = 0; i < h->g.n; ++i)
        h->n_species[species[i]] += 1;
    for (auto &q : h->g.rep) {
        double m = 0.0;
        for (int i = q.start; i < q.start + q.n; ++i)
            m += p->mass[species[i]];
        q.mtot = m;
    }
    h->s = (cudaStream_t)cuda_stream;
    h->ws = (char *)workspace;
    h->ks = &kernel_set(p->precision);
    h->cap = p->obs_capacity > 0 ? p->obs_capacity : 4096;
    const Geometry &g = h->g;
    const Layout &L = h->lay;
    KArgs &a = h->a;
    memset(&a, 0, sizeof a);
    char *w = h->ws;
    a.n = (int)g.n;
    a.nrep = g.R;
    a.ncell = g.ncell;
    a.Kstride = g.Kmax;
    a.si = p->sample_interval;
    a.obs_cap = h->cap;
    a.epot_cap = h->cap;
    a.nblk_i = g.nblk_i;
    a.pa = w + L.off_pa; a.pb = w + L.off_pb; a.va = w + L.off_va; a.vb = w + L.off_vb;
    a.pa2 = w + L.off_pa2; a.pb2 = w + L.off_pb2; a.va2 = w + L.off_va2; a.vb2 = w + L.off_vb2;
    a.qa = (int4 *)(w + L.off_qa); a.qb = (int4 *)(w + L.off_qb);
    a.force = w + L.off_force;
    a.rref = (float4 *)(w + L.off_rref);
    a.image = (int4 *)(w + L.off_image);
    a.image2 = (int4 *)(w + L.off_image2);
    a.key = (int2 *)(w + L.off_key);
    a.tmpidx = (int2 *)(w + L.off_tmpidx);
    a.ccount = (int *)(w + L.off_ccount);
    a.ccursor = (int *)(w + L.off_ccursor);
    a.cstart = (int *)(w + L.off_cstart);
    a.crank = (const int *)(w + L.off_crank);
    a.cxyz = (const int4 *)(w + L.off_cxyz);
    a.nbr = (int *)(w + L.off_nbr);
    a.nnbr = (int *)(w + L.off_nnbr);
    a.blk_i = (const int4 *)(w + L.off_blk_i);
    a.blk_r = (const int4 *)(w + L.off_blk_r);
    a.rs = (mdk::RunSync *)(w + L.off_rs);
    a.slice = (int *)(w + L.off_slice);
    a.check = g.check;
    a.part_f = (double *)(w + L.off_part_f);
    a.part_i = (double *)(w + L.off_part_i);
    a.part_e = w + L.off_part_e;
    a.ring = (mdk::Obs *)(w + L.off_ring);
    a.epot = (double *)(w + L.off_epot);
    a.epot_step = (long long *)(w + L.off_epot_step);
    a.totals = (mdk::Obs *)(w + L.off_totals);
    a.ctl = (mdk::Ctl *)(w + L.off_ctl);
    a.rep = (const mdk::Rep *)(w + L.off_rep);
    a.st_pos = (double *)(w + L.off_st_pos);
    a.st_vel = (double *)(w + L.off_st_vel);
    a.st_img = (int *)(w + L.off_st_img);
    a.st_code = (int *)(w + L.off_st_code);
    a.st_f = (double *)(w + L.off_st_f);
    a.st_e = (double *)(w + L.off_st_e);
    a.scale = (double *)(w + L.off_scale);
    // pair table (Sec. 3 potential, Sec. 5 parameters)
    for (int x = 0; x < 2; ++x)
        for (int y = 0; y < 2; ++y) {
            const int k = x * 2 + y;
            const int xs = std::min(x, p->n_species - 1), ys = std::min(y, p->n_species - 1);
            const double eps = p->eps[xs][ys], sig = p->sigma[xs][ys], rc = p->rcut[xs][ys];
            const double sr6 = std::pow(sig / rc, 6.0);
            const double shift = p->shift ? 4.0 * eps * (sr6 * sr6 - sr6) : 0.0;
            const double rl = rc + p->skin + (double)mdk::kListMargin;
            a.tab.rc2d[k] = rc * rc;
            a.tab.sig2d[k] = sig * sig;
            a.tab.eps4d[k] = 4.0 * eps;
            a.tab.eps48d[k] = 48.0 * eps;
            a.tab.shiftd[k] = shift;
            a.tab.rc2[k] = (float)(rc * rc);
            a.tab.rl2[k] = (float)(rl * rl);
            a.tab.sig2[k] = (float)(sig * sig);
            a.tab.eps4[k] = (float)(4.0 * eps);
            a.tab.eps48[k] = (float)(48.0 * eps);
            a.tab.shift[k] = (float)shift;
            // smoothing of Sec. 4: x = (r - r_c) / (h sigma_ab)
            const double ihs = p->smooth_h > 0.0 ? 1.0 / (p->smooth_h * sig) : 0.0;
            a.tab.rcd[k] = rc;
            a.tab.ihsd[k] = ihs;
            a.tab.rc[k] = (float)rc;
            a.tab.ihs[k] = (float)ihs;
            a.tab.vcd[k] = eps != 0.0 ? shift / (4.0 * eps) : 0.0;
            a.tab.vc[k] = (float)a.tab.vcd[k];
            a.tab.e48vcd[k] = a.tab.eps48d[k] * a.tab.vcd[k];
        }
    for (int s = 0; s < 2; ++s) {
        const int ss = std::min(s, p->n_species - 1);
        const double m = p->mass[ss];
        const double hk = 0.5 * p->dt / m;
        a.mass[s] = m;
        a.hdtm[s] = hk;
        a.hdtm_hi[s] = (float)hk;
        a.hdtm_lo[s] = (float)(hk - (double)(float)hk);
    }
    a.dt = p->dt;
    a.dt_hi = (float)p->dt;
    a.dt_lo = (float)(p->dt - (double)(float)p->dt);
    const double thr = std::max(0.5 * p->skin - (double)mdk::kDispMargin, 0.0);
    a.disp_thr = (float)thr;
    a.spin_max = mdk::kSpinMax;
    for (int s = 0; s < 2; ++s)
        a.inv_mass[s] = (float)(1.0 / a.mass[s]);
    if (a.hdtm_hi[0] == 0.0f)
        return fail(h, MD_E_INVAL, "dt / (2 m) underflows single precision");

    int dev = 0, nsm = 0, per_sm = 0, resident = 0;
    CK(h, cudaGetDevice(&dev));
    CK(h, cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    nsm = stream_sms(h->s, nsm);
    h->runk = h->ks->run[h->p.smooth_h > 0.0][force_index(g.tpp)];
    const int most = std::min(h->ks->groups[h->p.smooth_h > 0.0], kMaxRunGroups / std::max(nsm, 1));
    if (most < 1)
        return fail(h, MD_E_CUDA, "the run kernel does not fit the device");
    CK(h, cudaFuncSetAttribute(h->runk, cudaFuncAttributeMaxDynamicSharedMemorySize, most * h->ks->group_smem));
    CK(h, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, h->runk, kForceBlock * most,
                                                        (size_t)most * (size_t)h->ks->group_smem));
    if (resident < 1)
        return fail(h, MD_E_CUDA, "the run kernel does not fit the device");
    per_sm = most;
    h->nsm = nsm;
    const bool one_each = g.nblk_f <= nsm * per_sm;   // a group for every chunk
    h->g.sweep = p->step_form == 2 || (p->step_form == 0 && !one_each && p->precision != MD_PREC_FP64 && g.tpp <= 2);
    // the build takes a warp per cell when there are at least kNbWarpCellsPerSm cells per SM
    // and a cell's particles fit one batch of lanes on average; groups of threads otherwise
    // (measured on GB300: LJ at 729 cells or fewer and dense cells of ~40 are faster with
    // groups, LJ from 1331 cells and KA N=65,536 with a warp per cell)
    h->g.nb_block = p->build_form == 2 ||
                    (p->build_form == 0 && ((int64_t)g.ncell < (int64_t)kNbWarpCellsPerSm * nsm ||
                                            (double)g.n > 32.0 * (double)g.ncell));
    h->a.nb_warp = h->g.nb_block ? 0 : 1;
    // pinned staging, events
    CK(h, cudaEventCreateWithFlags(&h->ev_stage, cudaEventDisableTiming));
    CK(h, cudaEventCreate(&h->ev_f0));
    CK(h, cudaEventCreate(&h->ev_f1));
    CK(h, cudaEventCreate(&h->ev_i1));
    CK(h, cudaEventRecord(h->ev_stage, h->s));
    size_t tbytes = sizeof(mdk::Rep) * g.R + sizeof(int4) * (g.nblk_i + 3 * (size_t)g.nblk_f) +
                    sizeof(int) * g.ncell + sizeof(int4) * g.ncell;
    size_t sbytes = 64 * (size_t)g.n;
    if ((rc = ensure_pinned(h, std::max(tbytes, sbytes) + 4096)))
        return rc;
    // tables
    {
        char *q = h->pin;
        auto put = [&](size_t off, const void *src, size_t bytes) -> int {
            memcpy(q, src, bytes);
            cudaError_t e = cudaMemcpyAsync(w + off, q, bytes, cudaMemcpyHostToDevice, h->s);
            q += align_up(bytes);
            return e == cudaSuccess ? MD_OK : cuda_fail(h, e, "table upload");
        };
        const std::vector<int4> bf = mdt::sm_block_order(g.blk_f, nsm, nsm * per_sm);
        const std::vector<int4> br =
            mdt::step_table(bf, g.blk_f, !one_each, nsm, per_sm, h->g.nwork, h->g.cpb);
        h->a.cpb = h->g.cpb;
        h->a.nrow = (int)br.size();
        h->a.nslot = g.R == 1 ? h->g.nwork : g.nblk_f;
        // groups without chunks, where the GPU holds more than there are chunks, add up the
        // steps' partial sums, a replica each; in a rebuild a group takes a cell (or a share of
        // one where cells are few).  Where the chunks' groups outnumber the cells, shares ask for
        // 2 groups per SM at most: the launch occupies every SM, and up to 3 groups (2 of the
        // kernels that hold 5) leave room for another handle's on another stream.  us per MD
        // step and handle, 1 / 2 / 4 / 8 handles, with up to 4 groups for shares and with 2:
        // KA N = 2000 8.4 8.5 8.4 8.4 and 8.4 4.6 4.6 3.6; 4000 9.5 9.5 9.5 9.4 and 9.5 5.2 5.1
        // 4.1; FP64 N = 4000 33.9 33.7 33.7 - and 33.9 29.2 29.0 -.  (Cells that outnumber the
        // chunks do need groups: N = 16,384, 512 cells, 13.1 with 4 and 14.2 with 3, which
        // would let two handles take 8.7 each.  One group at N = 864 would let seven handles in,
        // 2.2 for 3.1 of eight, but costs a single one 1 to 3 %.)
        const int base = h->g.nwork + std::min(g.R, nsm), parts = std::max(1, std::min(8, 4 * nsm / g.ncell));
        const int cells = g.ncell < kMaxRunGroups ? g.ncell * parts : kMaxRunGroups;
        const int want = std::max(base, g.ncell <= base ? std::min(cells, 2 * nsm) : cells);
        h->g.groups = std::min(per_sm, (want + nsm - 1) / nsm);
        h->a.nb_parts = std::max(1, std::min(8, nsm * h->g.groups / g.ncell));
        if ((rc = put(L.off_rep, g.rep.data(), sizeof(mdk::Rep) * g.R)) ||
            (rc = put(L.off_blk_i, g.blk_i.data(), sizeof(int4) * g.nblk_i)) ||
            (rc = put(L.off_blk_r, br.data(), sizeof(int4) * br.size())) ||
            (rc = put(L.off_crank, g.crank.data(), sizeof(int) * g.ncell)) ||
            (rc = put(L.off_cxyz, g.cxyz.data(), sizeof(int4) * g.ncell)))
            return rc;
        mdk::Ctl c0;
        memset(&c0, 0, sizeof c0);
        c0.K = g.K;
        c0.Kmax = g.Kmax;
        if ((rc = put(L.off_ctl, &c0, sizeof c0)))
            return rc;
        cudaError_t e = cudaMemsetAsync(a.ccount, 0, 4 * (size_t)g.ncell, h->s);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(a.slice, 0, sizeof(int) * kMaxRunGroups, h->s);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(a.rs, 0, sizeof(mdk::RunSync), h->s);
        if (e == cudaSuccess)   // every slot of the per-step series empty (step -1)
            e = cudaMemsetAsync(a.epot_step, 0xff, sizeof(long long) * (size_t)h->cap, h->s);
        if (e == cudaSuccess)
            e = cudaEventRecord(h->ev_stage, h->s);
        if (e != cudaSuccess)
            return cuda_fail(h, e, "initialisation");
    }
    if ((rc = upload_state(h, species, pos, vel, image)))
        return rc;
    return check_device(h);
}

int md_create(md_handle **out, const md_params *p, int32_t n_replicas, const int64_t *n_per_replica,
              const double *box, const int32_t *species, const double *pos, const double *vel,
              const int32_t *image, void *workspace, size_t workspace_bytes, void *cuda_stream)
{
    ApiRange range_("md_create");
    if (!out)
        return MD_E_INVAL;
    *out = nullptr;
    md_handle *h = new (std::nothrow) md_handle();
    if (!h)
        return MD_E_NOMEM;
    std::string msg;
    int rc = make_geometry(p, n_replicas, n_per_replica, box, h->g, msg);
    if (rc == MD_OK)
        rc = create_impl(h, p, species, pos, vel, image, workspace, workspace_bytes, cuda_stream);
    if (rc != MD_OK) {
        md_destroy(h);
        return rc;
    }
    *out = h;
    return MD_OK;
}

int md_step(md_handle *h, int64_t nsteps)
{
    ApiRange range_("md_step");
    if (!h)
        return MD_E_INVAL;
    if (nsteps < 1)
        return fail(h, MD_E_INVAL, "nsteps must be >= 1");
    int rc;
    if ((rc = lost(h)) || (rc = refresh(h)))
        return rc;
    // bound on the steps executed (a device loop that could not end would hold the GPU)
    const int64_t budget = h->p.step_budget > 0 ? h->p.step_budget : nsteps + 64;
    if (h->p.use_graph)
        return launch_run(h, mdk::RUN_FIRST | mdk::RUN_STEPS, nsteps, budget);
    // The same phases as launches of their own, with their times.  At each check
    // point the host reads the device's rebuild flag and launches the rebuild
    // when it is set, so exactly the same work runs (results are bitwise equal).
    if ((rc = launch_run(h, mdk::RUN_FIRST | mdk::RUN_DEFER)) || (rc = rebuild_if_flagged(h, nullptr)))
        return rc;
    const int ci = h->g.check;
    for (int64_t k = 0; k < nsteps && k < budget; ++k) {
        CK(h, cudaEventRecord(h->ev_f0, h->s));
        if ((rc = launch_run(h, mdk::RUN_STEPS, 1, budget - k, (int)(k % ci), k == nsteps - 1)))
            return rc;
        CK(h, cudaEventRecord(h->ev_f1, h->s));
        CK(h, cudaEventSynchronize(h->ev_f1));
        float ms = 0.f;
        CK(h, cudaEventElapsedTime(&ms, h->ev_f0, h->ev_f1));
        h->step_ms += ms;
        h->step_launches += 1;
        if (k % ci == ci - 1 && k < nsteps - 1) {
            float mr = 0.f;
            if ((rc = rebuild_if_flagged(h, &mr)))
                return rc;
            h->rebuild_ms += mr;
        }
    }
    return MD_OK;
}

int md_rescale_velocities(md_handle *h, const double *T_target)
{
    ApiRange range_("md_rescale_velocities");
    if (!h || !T_target)
        return MD_E_INVAL;
    int rc;
    for (int r = 0; r < h->g.R; ++r)
        if (!(T_target[r] >= 0.0))
            return fail(h, MD_E_INVAL, "target temperatures must be >= 0");
    if ((rc = lost(h)) || (rc = stage_wait(h)))
        return rc;
    memcpy(h->pin, T_target, 8 * (size_t)h->g.R);
    CK(h, cudaMemcpyAsync(h->a.scale, h->pin, 8 * (size_t)h->g.R, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaEventRecord(h->ev_stage, h->s));
    if ((rc = launch_kinetic(h, mdk::IM_KE)))
        return rc;
    return launch(h, h->ks->scale, h->g.nblk_i, kIntBlock, h->a);
}

// Andersen heat bath (Sec. 2.3): one collision of every particle.
int md_andersen(md_handle *h, const double *T_target, uint64_t seed, int64_t event)
{
    ApiRange range_("md_andersen");
    if (!h || !T_target)
        return MD_E_INVAL;
    if (event < 0)
        return fail(h, MD_E_INVAL, "event index must be >= 0");
    const unsigned long long n = (unsigned long long)h->g.n;
    if ((unsigned long long)event > (~0ull >> 1) / 4 / (n + 1))
        return fail(h, MD_E_INVAL, "event index too large");
    int rc;
    for (int r = 0; r < h->g.R; ++r)
        if (!(T_target[r] >= 0.0) || !std::isfinite(T_target[r]))
            return fail(h, MD_E_INVAL, "target temperatures must be finite and >= 0");
    if ((rc = lost(h)) || (rc = stage_wait(h)))
        return rc;
    memcpy(h->pin, T_target, 8 * (size_t)h->g.R);
    CK(h, cudaMemcpyAsync(h->a.scale, h->pin, 8 * (size_t)h->g.R, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaEventRecord(h->ev_stage, h->s));
    // rand48 (a = 0x5DEECE66D, c = 0xB, modulo 2^48), seeded as srand48; leapfrog over n threads
    const unsigned long long A = 0x5DEECE66DULL, Cc = 0xBULL, mask = 0xFFFFFFFFFFFFULL;
    unsigned long long AN = 1, CN = 0, Ab = A, Cb = Cc;
    for (unsigned long long p = n; p; p >>= 1) {
        if (p & 1ull) {
            AN = (Ab * AN) & mask;
            CN = (Ab * CN + Cb) & mask;
        }
        Cb = (Ab * Cb + Cb) & mask;
        Ab = (Ab * Ab) & mask;
    }
    mdk::KArgs a = h->a;
    a.r48_x0 = ((seed & 0xFFFFFFFFull) << 16) | 0x330Eull;
    a.r48_AN = AN;
    a.r48_CN = CN;
    a.r48_base = (long long)(4ull * (unsigned long long)event * n);
    if ((rc = launch(h, h->ks->andersen, h->g.nblk_i, kIntBlock, a)) ||
        (rc = launch_kinetic(h, mdk::IM_TOTALS)))
        return rc;
    return launch(h, h->ks->andersen_fix, h->g.nblk_i, kIntBlock, h->a);
}

// ---------------------------------------------------------------------------
// Blocking scheme for time-correlation functions (Sec. 2.5).  Block n holds at
// most l samples spaced l^n samples apart; when it is full its first entry is
// correlated with the others and dropped.  Snapshots live in a pool of k l
// slots shared by the blocks (a sample that enters several blocks is stored
// once); the host keeps the bookkeeping, the device the data and the sums.
// ---------------------------------------------------------------------------
struct md_corr {
    md_handle *h = nullptr;
    int k = 0, l = 0, nq = 0, nblocks = 0;
    int64_t m = 0;                            // samples taken
    double *pool = nullptr;                   // [k l][n][3]
    int *species = nullptr;                   // [n]
    double *q = nullptr;                      // [nq][3]
    double *part = nullptr;                   // [nblocks][l-1][4]
    double *acc = nullptr;                    // [k][l-1][4]
    std::vector<std::vector<int>> blocks;     // slot ids, oldest first
    std::vector<int> refs;                    // blocks referring to each slot
    std::vector<int64_t> origins;             // [k][l-1]
};

namespace {

size_t corr_layout(int64_t n, int k, int l, int nq, size_t off[6])
{
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o = align_up(o + std::max<size_t>(bytes, 1)); return r; };
    const size_t nb = (size_t)((n + mdk::kCorrBlock - 1) / mdk::kCorrBlock);
    off[0] = take(sizeof(double) * 3 * (size_t)n * (size_t)k * (size_t)l);
    off[1] = take(sizeof(int) * (size_t)n);
    off[2] = take(sizeof(double) * 3 * (size_t)nq);
    off[3] = take(sizeof(double) * 4 * nb * (size_t)(l - 1));
    off[4] = take(sizeof(double) * 4 * (size_t)k * (size_t)(l - 1));
    off[5] = o;
    return o;
}

int corr_check(const md_handle *h, int k, int l, int nq)
{
    if (!h || k < 1 || l < 2 || l - 1 > mdk::kCorrMaxJ || nq < 1 || nq > mdk::kCorrMaxQ)
        return MD_E_INVAL;
    double span = 1.0;                         // l^k must stay a valid sample index
    for (int n = 0; n < k; ++n)
        span *= l;
    return span < 9e15 ? MD_OK : MD_E_INVAL;
}

}  // namespace

int md_corr_workspace_size(const md_handle *h, int32_t k, int32_t l, int32_t n_q, size_t *bytes)
{
    if (!bytes || corr_check(h, k, l, n_q))
        return MD_E_INVAL;
    size_t off[6];
    *bytes = corr_layout(h->g.n, k, l, n_q, off);
    return MD_OK;
}

int md_corr_create(md_corr **out, md_handle *h, int32_t k, int32_t l, int32_t n_q, const double *q,
                   void *workspace, size_t workspace_bytes)
{
    ApiRange range_("md_corr_create");
    if (!out || !q || corr_check(h, k, l, n_q))
        return h ? fail(h, MD_E_INVAL, "md_corr_create: bad arguments (1 <= k, 2 <= l <= 32, "
                                       "1 <= n_q <= 64, non-null q)") : MD_E_INVAL;
    *out = nullptr;
    size_t off[6];
    const size_t need = corr_layout(h->g.n, k, l, n_q, off);
    if (!workspace || ((uintptr_t)workspace % kAlign) != 0)
        return fail(h, MD_E_INVAL, "md_corr_create: workspace missing or not 256-byte aligned");
    if (workspace_bytes < need)
        return fail(h, MD_E_NOMEM, "md_corr_create: workspace smaller than md_corr_workspace_size()");
    for (int t = 0; t < 3 * n_q; ++t)
        if (!std::isfinite(q[t]))
            return fail(h, MD_E_INVAL, "md_corr_create: non-finite wavevector");
    md_corr *c = new (std::nothrow) md_corr;
    if (!c)
        return fail(h, MD_E_NOMEM, "md_corr_create: host allocation failed");
    char *w = (char *)workspace;
    c->h = h;
    c->k = k;
    c->l = l;
    c->nq = n_q;
    c->nblocks = (int)((h->g.n + mdk::kCorrBlock - 1) / mdk::kCorrBlock);
    c->pool = (double *)(w + off[0]);
    c->species = (int *)(w + off[1]);
    c->q = (double *)(w + off[2]);
    c->part = (double *)(w + off[3]);
    c->acc = (double *)(w + off[4]);
    c->blocks.assign(k, std::vector<int>());
    c->refs.assign((size_t)k * l, 0);
    c->origins.assign((size_t)k * (l - 1), 0);
    int rc;
    if ((rc = stage_wait(h)) || (rc = ensure_pinned(h, sizeof(double) * 3 * n_q))) {
        delete c;
        return rc;
    }
    memcpy(h->pin, q, sizeof(double) * 3 * n_q);
    cudaError_t e = cudaMemcpyAsync(c->q, h->pin, sizeof(double) * 3 * n_q, cudaMemcpyHostToDevice, h->s);
    if (e == cudaSuccess)
        e = cudaEventRecord(h->ev_stage, h->s);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(c->acc, 0, sizeof(double) * 4 * (size_t)k * (l - 1), h->s);
    if (e != cudaSuccess) {
        delete c;
        return cuda_fail(h, e, "md_corr_create");
    }
    *out = c;
    return MD_OK;
}

int md_corr_sample(md_corr *c)
{
    ApiRange range_("md_corr_sample");
    if (!c)
        return MD_E_INVAL;
    md_handle *h = c->h;
    if (const int rl = lost(h))
        return rl;
    int slot = -1;
    for (size_t s = 0; s < c->refs.size(); ++s)
        if (c->refs[s] == 0) {
            slot = (int)s;
            break;
        }
    if (slot < 0)
        return fail(h, MD_E_INVAL, "md_corr_sample: no free snapshot slot");   // cannot happen: k l slots
    const size_t n = (size_t)h->g.n;
    mdk::KArgs a = h->a;
    a.snap = c->pool + 3 * n * (size_t)slot;
    a.snap_species = c->species;
    int rc;
    if ((rc = launch(h, h->ks->snapshot, h->g.nblk_i, kIntBlock, a)))
        return rc;
    int64_t spacing = 1;
    for (int b = 0; b < c->k; ++b, spacing *= c->l) {
        if (c->m % spacing)
            break;
        std::vector<int> &blk = c->blocks[b];
        blk.push_back(slot);
        c->refs[slot] += 1;
        if ((int)blk.size() < c->l)
            continue;
        mdk::CorrArgs ca;
        ca.s0 = c->pool + 3 * n * (size_t)blk[0];
        for (int j = 1; j < c->l; ++j)
            ca.sj[j - 1] = c->pool + 3 * n * (size_t)blk[j];
        for (int j = c->l; j <= mdk::kCorrMaxJ; ++j)
            ca.sj[j - 1] = nullptr;
        ca.nj = c->l - 1;
        ca.n = (int)n;
        ca.nq = c->nq;
        ca.species = c->species;
        ca.q = c->q;
        ca.part = c->part;
        ca.acc = c->acc + (size_t)b * (c->l - 1) * 4;
        ca.nblocks = c->nblocks;
        mdk::k_corr<<<c->nblocks, mdk::kCorrBlock, 0, h->s>>>(ca);
        mdk::k_corr_reduce<<<1, mdk::kCorrReduce, 0, h->s>>>(ca);
        CK(h, cudaGetLastError());
        for (int j = 0; j < c->l - 1; ++j)
            c->origins[(size_t)b * (c->l - 1) + j] += 1;
        c->refs[blk[0]] -= 1;
        blk.erase(blk.begin());
    }
    c->m += 1;
    return MD_OK;
}

int md_corr_result(md_corr *c, int64_t *lags, double *msd, double *fs, int64_t *origins)
{
    ApiRange range_("md_corr_result");
    if (!c)
        return MD_E_INVAL;
    md_handle *h = c->h;
    const size_t nl = (size_t)c->k * (c->l - 1);
    std::vector<double> acc(4 * nl);
    CK(h, cudaStreamSynchronize(h->s));
    CK(h, cudaMemcpy(acc.data(), c->acc, sizeof(double) * 4 * nl, cudaMemcpyDeviceToHost));
    int64_t spacing = 1;
    for (int b = 0; b < c->k; ++b, spacing *= c->l)
        for (int j = 1; j < c->l; ++j) {
            const size_t t = (size_t)b * (c->l - 1) + (j - 1);
            const int64_t no = c->origins[t];
            if (lags)
                lags[t] = (int64_t)j * spacing;
            if (origins)
                origins[t] = no;
            for (int a = 0; a < 2; ++a) {
                const double cnt = (double)no * (double)h->n_species[a];
                const double nan = std::nan("");
                if (msd)
                    msd[2 * t + a] = cnt > 0 ? acc[4 * t + 2 * a] / cnt : nan;
                if (fs)
                    fs[2 * t + a] = cnt > 0 ? acc[4 * t + 2 * a + 1] / cnt : nan;
            }
        }
    return MD_OK;
}

int md_corr_destroy(md_corr *c)
{
    delete c;
    return MD_OK;
}

int md_compute_forces(md_handle *h, double *f, double *e, md_obs *totals)
{
    ApiRange range_("md_compute_forces");
    if (!h)
        return MD_E_INVAL;
    int rc;
    const size_t n = (size_t)h->g.n;
    if ((rc = lost(h)))
        return rc;
    h->stale = false;
    if ((rc = launch_run(h, mdk::RUN_REBUILD | mdk::RUN_TOTALS)) ||
        (rc = launch(h, h->ks->expforce, grid_n(h->g.n, kIntBlock), kIntBlock, h->a)))
        return rc;
    if ((rc = check_device(h)))
        return rc;
    const size_t tb = sizeof(md_obs) * h->g.R;
    if ((rc = ensure_pinned(h, 32 * n + tb + 512)))
        return rc;
    char *q = h->pin;
    CK(h, cudaMemcpyAsync(q, h->a.st_f, 24 * n, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaMemcpyAsync(q + 24 * n, h->a.st_e, 8 * n, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaMemcpyAsync(q + 32 * n, h->a.totals, tb, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaStreamSynchronize(h->s));
    const CopyJob out[3] = {{f, q, f ? 24 * n : 0}, {e, q + 24 * n, e ? 8 * n : 0}, {totals, q + 32 * n, totals ? tb : 0}};
    copy_jobs(out, 3);
    return MD_OK;
}

int md_observables(md_handle *h, md_obs *out, int32_t max_samples, int32_t *n_samples)
{
    ApiRange range_("md_observables");
    if (!h || !n_samples || (max_samples > 0 && !out))
        return MD_E_INVAL;
    *n_samples = 0;
    mdk::Ctl c;
    int rc = read_ctl(h, &c);
    if (rc)
        return rc;
    const int64_t avail = c.obs_count - h->obs_read;
    int64_t m = std::min<int64_t>(avail, h->cap);
    m = std::min<int64_t>(m, max_samples);
    const int64_t first = c.obs_count - m;
    const size_t rec = sizeof(md_obs) * h->g.R;
    if (m > 0) {
        if ((rc = ensure_pinned(h, rec * (size_t)m)))
            return rc;
        int64_t done = 0;
        while (done < m) {
            const int64_t slot = (first + done) % h->cap;
            const int64_t cnt = std::min<int64_t>(m - done, h->cap - slot);
            CK(h, cudaMemcpyAsync(h->pin + rec * done, (char *)h->a.ring + rec * slot, rec * cnt,
                                  cudaMemcpyDeviceToHost, h->s));
            done += cnt;
        }
        CK(h, cudaStreamSynchronize(h->s));
        memcpy(out, h->pin, rec * (size_t)m);
    }
    h->obs_read = c.obs_count;
    *n_samples = (int32_t)m;
    const int code = status_code(c.status);
    if (code != MD_OK)
        return check_device(h);
    return MD_OK;
}

int md_epot_series(md_handle *h, int64_t *steps, double *e_pot, int32_t max_steps, int32_t *n_steps)
{
    ApiRange range_("md_epot_series");
    if (!h || !n_steps || (max_steps > 0 && (!steps || !e_pot)))
        return MD_E_INVAL;
    *n_steps = 0;
    mdk::Ctl c;
    int rc = read_ctl(h, &c);
    if (rc)
        return rc;
    const size_t cap = (size_t)h->cap, R = (size_t)h->g.R;
    const size_t sb = align_up(sizeof(long long) * cap);
    if ((rc = ensure_pinned(h, sb + sizeof(double) * cap * R)) || (rc = stage_wait(h)))
        return rc;
    CK(h, cudaMemcpyAsync(h->pin, h->a.epot_step, sizeof(long long) * cap, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaMemcpyAsync(h->pin + sb, h->a.epot, sizeof(double) * cap * R, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaStreamSynchronize(h->s));
    const long long *st = (const long long *)h->pin;
    const double *ev = (const double *)(h->pin + sb);
    std::vector<std::pair<long long, size_t>> got;       // (step, slot) not yet returned
    for (size_t k = 0; k < cap; ++k)
        if (st[k] > h->epot_read)
            got.push_back({st[k], k});
    std::sort(got.begin(), got.end());
    const size_t m = std::min<size_t>(got.size(), (size_t)std::max(max_steps, 0));
    const size_t first = got.size() - m;                  // the newest m
    for (size_t t = 0; t < m; ++t) {
        steps[t] = got[first + t].first;
        memcpy(e_pot + t * R, ev + got[first + t].second * R, sizeof(double) * R);
    }
    if (!got.empty())
        h->epot_read = got.back().first;
    *n_steps = (int32_t)m;
    if (status_code(c.status) != MD_OK)
        return check_device(h);
    return MD_OK;
}

int md_get_state(md_handle *h, double *pos, double *vel, int32_t *image)
{
    ApiRange range_("md_get_state");
    if (!h)
        return MD_E_INVAL;
    int rc;
    const size_t n = (size_t)h->g.n;
    if ((rc = lost(h)) || (rc = launch(h, h->ks->getstate, grid_n(h->g.n, kIntBlock), kIntBlock, h->a)))
        return rc;
    if ((rc = ensure_pinned(h, 60 * n + 4)) || (rc = stage_wait(h)))
        return rc;
    char *q = h->pin;
    CK(h, cudaMemcpyAsync(q, h->a.st_pos, 24 * n, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaMemcpyAsync(q + 24 * n, h->a.st_vel, 24 * n, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaMemcpyAsync(q + 48 * n, h->a.st_img, 12 * n + 4, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaStreamSynchronize(h->s));
    int32_t gone;
    memcpy(&gone, q + 60 * n, 4);
    if (gone)                                            // (not reported yet)
        return check_device(h);
    const CopyJob out[3] = {{pos, q, pos ? 24 * n : 0},
                            {vel, q + 24 * n, vel ? 24 * n : 0},
                            {image, q + 48 * n, image ? 12 * n : 0}};
    copy_jobs(out, 3);
    return MD_OK;
}

int md_set_state(md_handle *h, const double *pos, const double *vel, const int32_t *image)
{
    ApiRange range_("md_set_state");
    if (!h || !pos || !vel)
        return MD_E_INVAL;
    int rc;
    // species are kept: read them back from the working layout is not needed,
    // the staging area still holds the codes uploaded at creation
    const size_t n = (size_t)h->g.n;
    if ((rc = ensure_pinned(h, 64 * n)) || (rc = stage_wait(h)))
        return rc;
    char *q = h->pin;
    const CopyJob in[3] = {{q, pos, 24 * n}, {q + 24 * n, vel, 24 * n}, {q + 48 * n, image, image ? 12 * n : 0}};
    copy_jobs(in, 3);
    if (!image)
        memset(q + 48 * n, 0, 12 * n);
    CK(h, cudaMemcpyAsync(h->a.st_pos, q, 24 * n, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaMemcpyAsync(h->a.st_vel, q + 24 * n, 24 * n, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaMemcpyAsync(h->a.st_img, q + 48 * n, 12 * n, cudaMemcpyHostToDevice, h->s));
    CK(h, cudaEventRecord(h->ev_stage, h->s));
    h->stale = h->lost = false;
    if ((rc = launch(h, h->ks->load, h->g.nblk_i, kIntBlock, h->a)))
        return rc;
    return launch_run(h, mdk::RUN_REBUILD | mdk::RUN_FORCES);
}

int md_get_neighbours(md_handle *h, int32_t *counts, int32_t *lists, int32_t kmax)
{
    ApiRange range_("md_get_neighbours");
    if (!h || !counts || (lists && kmax < 1))
        return MD_E_INVAL;
    const size_t n = (size_t)h->g.n;
    int rc;
    mdk::Ctl c;
    if ((rc = lost(h)) || (rc = refresh(h)) || (rc = read_ctl(h, &c)))
        return rc;
    if (c.stale & mdk::STALE_STATE)                      // (not reported yet)
        return check_device(h);
    const size_t K = (size_t)h->g.Kmax;                  // row stride of the lists (the cap)
    if ((rc = ensure_pinned(h, align_up(4 * n) + align_up(16 * n) + 4 * n * K)) || (rc = stage_wait(h)))
        return rc;
    char *q = h->pin;
    int *nn = (int *)q;
    int4 *img = (int4 *)(q + align_up(4 * n));
    int *nb = (int *)(q + align_up(4 * n) + align_up(16 * n));
    const int4 *dimg = c.state_par ? h->a.image2 : h->a.image;   // tags of the current order
    CK(h, cudaMemcpyAsync(nn, h->a.nnbr, 4 * n, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaMemcpyAsync(img, dimg, 16 * n, cudaMemcpyDeviceToHost, h->s));
    if (lists)
        CK(h, cudaMemcpyAsync(nb, h->a.nbr, 4 * n * K, cudaMemcpyDeviceToHost, h->s));
    CK(h, cudaStreamSynchronize(h->s));
    for (size_t s = 0; s < n; ++s) {
        const int t = img[s].w;
        counts[t] = nn[s];
        if (lists) {
            for (int k = 0; k < kmax; ++k)
                lists[(size_t)t * kmax + k] = (k < nn[s] && (size_t)k < K) ? img[nb[s * K + k]].w : -1;
        }
    }
    return MD_OK;
}

int md_info(md_handle *h, md_info_t *out)
{
    if (!h || !out)
        return MD_E_INVAL;
    mdk::Ctl c;
    int rc = read_ctl(h, &c);
    if (rc)
        return rc;
    memset(out, 0, sizeof *out);
    out->n_total = h->g.n;
    out->n_replicas = h->g.R;
    out->neigh_capacity = c.K;
    out->neigh_capacity_max = h->g.Kmax;
    out->regrows = c.regrows;
    out->build_form = h->g.nb_block ? 2 : 1;
    out->step_form = h->g.sweep ? 2 : 1;
    out->threads_per_particle = h->g.tpp;
    out->check_interval = h->g.check;
    out->cells_per_edge = h->g.rep[0].nc;
    out->step = c.step;
    out->rebuilds = c.rebuilds;
    out->kernel_launches = c.n_kernels;
    out->max_neighbours = c.max_nbr;
    out->status = status_code(c.status);
    out->step_ms = h->step_ms;
    out->step_launches = h->step_launches;
    out->rebuild_ms = h->rebuild_ms;
    out->rebuild_checks = h->rebuild_checks;
    out->step_device_ms = (double)c.dev_ns * 1e-6;
    out->step_device_launches = c.dev_launches;
    return MD_OK;
}

int md_sync(md_handle *h)
{
    if (!h)
        return MD_E_INVAL;
    return check_device(h);
}

int md_set_wait_limit(md_handle *h, uint32_t polls)
{
    if (!h)
        return MD_E_INVAL;
    h->a.spin_max = polls ? polls : mdk::kSpinMax;
    return MD_OK;
}

int md_destroy(md_handle *h)
{
    ApiRange range_("md_destroy");
    if (!h)
        return MD_E_INVAL;
    if (h->ws)
        cudaStreamSynchronize(h->s);
    if (h->pin)
        cudaFreeHost(h->pin);
    if (h->ev_stage)
        cudaEventDestroy(h->ev_stage);
    if (h->ev_f0)
        cudaEventDestroy(h->ev_f0);
    if (h->ev_f1)
        cudaEventDestroy(h->ev_f1);
    if (h->ev_i1)
        cudaEventDestroy(h->ev_i1);
    delete h;
    return MD_OK;
}

const char *md_last_error(const md_handle *h)
{
    if (!h)
        return md_noalloc_message();
    return h->err.c_str();
}

const char *md_status_string(int code)
{
    switch (code) {
    case MD_OK: return "MD_OK";
    case MD_E_INVAL: return "MD_E_INVAL";
    case MD_E_NOMEM: return "MD_E_NOMEM";
    case MD_E_CUDA: return "MD_E_CUDA";
    case MD_E_NONFINITE: return "MD_E_NONFINITE";
    case MD_E_UNSTABLE: return "MD_E_UNSTABLE";
    case MD_E_TIMEOUT: return "MD_E_TIMEOUT";
    case MD_E_CAPACITY: return "MD_E_CAPACITY";
    case MD_E_BOUNDS: return "MD_E_BOUNDS";
    default: return "MD_E_UNKNOWN";
    }
}

}  // extern "C"
