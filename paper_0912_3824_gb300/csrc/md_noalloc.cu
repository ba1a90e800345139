// md_noalloc.cu -- force evaluation that allocates no device memory.
//
// Some callers cannot allocate device memory at the moment they need forces:
// an out-of-memory handler that must still evaluate a configuration after an
// allocation has failed, a host application whose memory manager owns the
// whole device and forbids cudaMalloc / cudaFree outside its own pool, or
// code that is certified to allocate nothing after start-up.  For them,
// md_forces_noalloc() evaluates forces, per-particle energies and the
// energy / virial totals of one periodic configuration by a direct sum over
// all pairs, using only the caller's input and output arrays plus a fixed
// scratch area that lives in this library's own device memory.
//
// That scratch is a file-scope __device__ array, reserved on every GPU that
// loads the library for the life of the process.  Host code cannot pass the
// array's name to a kernel (on the host it only names a stand-in), so its
// device address is looked up once per device with cudaGetSymbolAddress().
#include <cuda_runtime.h>

#include <cmath>
#include <cstddef>
#include <cstdio>
#include <mutex>

#include "md.h"

namespace {

constexpr int kMaxBlocks = 8192;   // blocks of a call: the scratch holds a partial sum of each
constexpr int kRows = 4;           // particles per warp at a time
constexpr int kTile = 512;         // partners staged at a time
constexpr int kPart = 8;           // e_pot, virial, w_xx, w_yy, w_zz, w_xy, w_xz, w_yz
constexpr int kMaxDevices = 64;


// Per-block partial sums, the ticket that elects the block finishing the
// totals, and a flag raised by any block that met a species outside
// [0, n_species) (512 KiB + 256 B).  ticket and bad are cleared by every call.
struct Scratch {
    double part[kMaxBlocks * kPart];
    unsigned int ticket;
    unsigned int bad;
    unsigned int pad[62];
};

static __device__ __align__(256) Scratch g_noalloc_scratch;

struct Pot {
    double rc2[4], sig2[4], eps4[4], eps48[4], shift[4];
    float rc2u[4];                 // (r_c + margin)^2 in units of (L / 2^32)^2
};

// Species code of a particle, clamped into [0, nsp) so that it always indexes
// the pair table; an out-of-range code raises the call's bad flag.
__device__ __forceinline__ int species_in_range(int t, int nsp, Scratch *s)
{
    if (t < 0 || t >= nsp) {
        atomicOr(&s->bad, 1u);
        return t < 0 ? 0 : nsp - 1;
    }
    return t;
}

// Number of boxes nearest to d / L, as a double: adding 1.5 2^52 rounds.
__device__ __forceinline__ double boxes(double d, double invL)
{
    constexpr double big = 6755399441055744.0;
    return fma(d, invL, big) - big;
}

// x / L modulo 1 in units of 2^-32: the low word of x 2^32 / L + 1.5 2^52.  Off
// by less than 1 1/4 units for |x| < 2^18 L; beyond (or not finite), `far` is set.
__device__ __forceinline__ int circle(double x, double scale, unsigned int far_hi, bool &far)
{
    far |= (unsigned int)(__double2hiint(x) & 0x7fffffff) >= far_hi;
    return __double2loint(fma(x, scale, 6755399441055744.0));
}

// Direct sum over all pairs.  A warp takes kRows particles, its lanes the
// partners, staged by the block as 32-bit fractions of the box: their wrapped
// differences are the nearest images, so the test that lets a pair through (with
// a margin for the rounding) is single precision and integers only.  The FP64
// pipe, narrow on this GPU, sees only the pairs let through: they wait in a
// queue per particle and are evaluated 32 at a time, one per lane, from the
// caller's coordinates, in double (FP64 mode) or in single precision on
// separations formed in double (the other modes).  Coordinates so far from the
// box that the fractions are not safe let every pair through.
//
// Bound by the tests for large n (about 13 instructions per 32 partners and
// particle) and by the FP64 sums for small n.  KA mixture, mixed: 0.14 ms at
// n = 6000, 0.55 at 16,384, 5.5 at 65,536; one thread per particle doing every test
// in FP64 took 4.5, 10.3 and 154 ms.
template <bool FP64MATH, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_forces_allpairs(Pot pot, int n, int nsp, double L, const int *species,
                                                                const double *pos, double *force, double *energy,
                                                                double *totals, Scratch *s)
{
    __shared__ int4 tile[kTile];
    __shared__ int queue[WARPS][kRows][64];
    __shared__ double red[WARPS][kPart];
    __shared__ double tot[32][kPart];
    __shared__ int is_last, tile_far;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt_mask = (1u << lane) - 1u;
    const double invL = 1.0 / L, scale = 4294967296.0 / L;
    const unsigned int far_hi = (unsigned int)__double2hiint(262144.0 * L);
    double acc[kPart] = {0, 0, 0, 0, 0, 0, 0, 0};         // totals of the lane's pairs, each seen from both sides

    for (long long base = (long long)blockIdx.x * WARPS * kRows; base < n; base += (long long)gridDim.x * WARPS * kRows) {
        const int i0 = (int)base + w * kRows;             // the warp's particles i0 .. i0 + kRows - 1
        int4 qi[kRows];
        float lim[kRows][2];
        double f[kRows][4];                               // force, energy
        int cnt[kRows];
        bool own_far = false;
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            const size_t i = (size_t)min(i0 + r, n - 1);
            qi[r].x = circle(pos[3 * i], scale, far_hi, own_far);
            qi[r].y = circle(pos[3 * i + 1], scale, far_hi, own_far);
            qi[r].z = circle(pos[3 * i + 2], scale, far_hi, own_far);
            qi[r].w = species_in_range(species[i], nsp, s);
            lim[r][0] = i0 + r < n ? pot.rc2u[qi[r].w * 2] : 0.0f;
            lim[r][1] = i0 + r < n ? pot.rc2u[qi[r].w * 2 + 1] : 0.0f;
            f[r][0] = f[r][1] = f[r][2] = f[r][3] = 0.0;
            cnt[r] = 0;
        }
        // evaluates the first m (up to 32) queued partners of particle i0 + r
        const auto flush = [&](int r, int m) {
            const int i = i0 + r, j = lane < m ? queue[w][r][lane] : i;
            if (j != i) {
                double dx = pos[3 * (size_t)i] - pos[3 * (size_t)j];
                double dy = pos[3 * (size_t)i + 1] - pos[3 * (size_t)j + 1];
                double dz = pos[3 * (size_t)i + 2] - pos[3 * (size_t)j + 2];
                dx = fma(-L, boxes(dx, invL), dx);
                dy = fma(-L, boxes(dy, invL), dy);
                dz = fma(-L, boxes(dz, invL), dz);
                const double r2 = dx * dx + dy * dy + dz * dz;
                const int tj = species[j];
                const int ab = qi[r].w * 2 + (tj < 0 ? 0 : (tj >= nsp ? nsp - 1 : tj));
                if (r2 < pot.rc2[ab]) {
                    double fr, v;
                    if (FP64MATH) {
                        const double ir2 = 1.0 / r2;
                        const double s2 = pot.sig2[ab] * ir2;
                        const double s6 = s2 * s2 * s2;
                        fr = pot.eps48[ab] * ir2 * s6 * (s6 - 0.5);
                        v = pot.eps4[ab] * s6 * (s6 - 1.0) - pot.shift[ab];
                    } else {
                        const float ir2 = 1.0f / (float)r2;
                        const float s2 = (float)pot.sig2[ab] * ir2;
                        const float s6 = s2 * s2 * s2;
                        fr = (double)((float)pot.eps48[ab] * ir2 * s6 * (s6 - 0.5f));
                        v = (double)((float)pot.eps4[ab] * s6 * (s6 - 1.0f) - (float)pot.shift[ab]);
                    }
                    const double px = fr * dx, py = fr * dy, pz = fr * dz;
                    f[r][0] += px;
                    f[r][1] += py;
                    f[r][2] += pz;
                    f[r][3] += v;
                    acc[1] += fr * r2;
                    acc[2] += px * dx;
                    acc[3] += py * dy;
                    acc[4] += pz * dz;
                    acc[5] += px * dy;
                    acc[6] += px * dz;
                    acc[7] += py * dz;
                }
            }
        };

        for (int j0 = 0; j0 < n; j0 += kTile) {
            __syncthreads();
            if (threadIdx.x == 0)
                tile_far = 0;
            __syncthreads();
            for (int t = threadIdx.x; t < kTile && j0 + t < n; t += 32 * WARPS) {
                const size_t j = (size_t)(j0 + t);
                bool far = own_far;
                int4 q;
                q.x = circle(pos[3 * j], scale, far_hi, far);
                q.y = circle(pos[3 * j + 1], scale, far_hi, far);
                q.z = circle(pos[3 * j + 2], scale, far_hi, far);
                q.w = species_in_range(species[j], nsp, s);
                tile[t] = q;
                if (far)
                    tile_far = 1;
            }
            __syncthreads();
            const int m = min(kTile, n - j0);
            const bool all = tile_far != 0 || own_far;
            for (int t0 = 0; t0 < m; t0 += 32) {
                const int t = t0 + lane;
                const bool ok = t < m;
                const int4 q = tile[ok ? t : 0];
#pragma unroll
                for (int r = 0; r < kRows; ++r) {
                    const float x = __int2float_rn((int)((unsigned)qi[r].x - (unsigned)q.x));
                    const float y = __int2float_rn((int)((unsigned)qi[r].y - (unsigned)q.y));
                    const float z = __int2float_rn((int)((unsigned)qi[r].z - (unsigned)q.z));
                    const float r2 = fmaf(x, x, fmaf(y, y, z * z));
                    const unsigned b =
                        __ballot_sync(0xffffffffu, ok && (r2 < (q.w ? lim[r][1] : lim[r][0]) || all) && i0 + r < n);
                    if (b == 0u)
                        continue;
                    if (b >> lane & 1u)
                        queue[w][r][cnt[r] + __popc(b & lt_mask)] = j0 + t;
                    cnt[r] += __popc(b);
                    if (cnt[r] >= 32) {
                        __syncwarp();
                        flush(r, 32);
                        __syncwarp();
                        // the rest moves to the front: by its own lanes only, and ordered before the
                        // next partners, which other lanes add behind it
                        const bool rest = lane < cnt[r] - 32;
                        const int next = rest ? queue[w][r][32 + lane] : 0;
                        __syncwarp();
                        if (rest)
                            queue[w][r][lane] = next;
                        __syncwarp();
                        cnt[r] -= 32;
                    }
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            flush(r, cnt[r]);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                for (int o = 16; o > 0; o >>= 1)
                    f[r][k] += __shfl_xor_sync(0xffffffffu, f[r][k], o);
            const int i = i0 + r;
            if (lane == 0 && i < n) {
                // a species code out of range: NaN
                const bool bad = species[i] < 0 || species[i] >= nsp;
                const double poison = bad ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
                force[3 * (size_t)i] = f[r][0] + poison;
                force[3 * (size_t)i + 1] = f[r][1] + poison;
                force[3 * (size_t)i + 2] = f[r][2] + poison;
                if (energy)
                    energy[i] = 0.5 * f[r][3] + poison;
                acc[0] += f[r][3];
            }
        }
    }
    // block sums in a fixed order, then the last block adds the blocks' sums
#pragma unroll
    for (int k = 0; k < kPart; ++k) {
        double v = 0.5 * acc[k];
        for (int o = 16; o > 0; o >>= 1)
            v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0)
            red[w][k] = v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 0; k < kPart; ++k) {
            double v = 0.0;
            for (int q = 0; q < WARPS; ++q)
                v += red[q][k];
            s->part[(size_t)blockIdx.x * kPart + k] = v;
        }
        __threadfence();
        is_last = atomicAdd(&s->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last)
        return;
    __threadfence();
    // (a slice of the blocks per 8 threads, then the slices in order)
    constexpr int kSlices = 32 * WARPS / kPart;
    const int c = threadIdx.x % kPart, sl = threadIdx.x / kPart;
    double v = 0.0;
#pragma unroll 4
    for (unsigned int b = sl; b < gridDim.x; b += kSlices)
        v += __ldcg(&s->part[(size_t)b * kPart + c]);
    tot[sl][c] = v;
    __syncthreads();
    if (threadIdx.x < kPart) {
        v = 0.0;
        for (int q = 0; q < kSlices; ++q)
            v += tot[q][threadIdx.x];
        // a species code out of range makes every total NaN
        if (atomicOr(&s->bad, 0u) != 0u)
            v = __longlong_as_double(0x7ff8000000000000ll);
        totals[threadIdx.x] = v;
    }
}

template <int WARPS>
void launch(bool fp64, cudaStream_t st, const Pot &pot, int n, int nsp, double box, const int *species, const double *pos,
            double *force, double *energy, double *totals, Scratch *s)
{
    const int per = WARPS * kRows, need = (n + per - 1) / per, grid = need < kMaxBlocks ? need : kMaxBlocks;
    if (fp64)
        k_forces_allpairs<true, WARPS><<<grid, 32 * WARPS, 0, st>>>(pot, n, nsp, box, species, pos, force, energy, totals, s);
    else
        k_forces_allpairs<false, WARPS><<<grid, 32 * WARPS, 0, st>>>(pot, n, nsp, box, species, pos, force, energy, totals, s);
}

std::mutex g_lock;
Scratch *g_addr[kMaxDevices] = {};

// Message of the calling thread's last failed call (a fixed buffer: nothing is
// allocated to report a failure); md_last_error(NULL) returns it.
thread_local char t_msg[256] = "";

int fail(int code, const char *m)
{
    snprintf(t_msg, sizeof t_msg, "%s", m);
    return code;
}

}  // namespace

// The message of the calling thread's last md_forces_noalloc failure ("" if
// its last call succeeded); md_api.cu returns it from md_last_error(NULL).
const char *md_noalloc_message() { return t_msg; }

extern "C" int md_forces_noalloc(const md_params *p, int64_t n, double box, const int32_t *species,
                                 const double *pos, double *force, double *energy, double *totals,
                                 void *cuda_stream)
{
    t_msg[0] = '\0';
    if (!p || !species || !pos || !force || !totals)
        return fail(MD_E_INVAL, "md_forces_noalloc: null argument");
    if (!(p->precision >= MD_PREC_FP64 && p->precision <= MD_PREC_FP32))
        return fail(MD_E_INVAL, "md_forces_noalloc: unknown precision mode");
    if (n < 2)
        return fail(MD_E_INVAL, "md_forces_noalloc: need at least 2 particles");
    if (n > MD_NOALLOC_MAX_N)
        return fail(MD_E_INVAL, "md_forces_noalloc: n exceeds MD_NOALLOC_MAX_N (1048576), the size of its "
                                "fixed scratch area; use md_create / md_compute_forces instead");
    if (p->n_species < 1 || p->n_species > 2)
        return fail(MD_E_INVAL, "md_forces_noalloc: n_species must be 1 or 2");
    if (p->smooth_h != 0.0)
        return fail(MD_E_INVAL, "md_forces_noalloc: the smoothed potential (smooth_h > 0) is not supported; "
                                "use md_create / md_compute_forces");
    Pot pot;
    double rcmax = 0.0;
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b) {
            const int x = a < p->n_species ? a : p->n_species - 1, y = b < p->n_species ? b : p->n_species - 1;
            const double eps = p->eps[x][y], sig = p->sigma[x][y], rc = p->rcut[x][y];
            if (!(sig > 0.0) || !(rc > 0.0))
                return fail(MD_E_INVAL, "md_forces_noalloc: sigma and rcut must be positive");
            const double sr2 = sig * sig / (rc * rc), sr6 = sr2 * sr2 * sr2;
            const int k = a * 2 + b;
            pot.rc2[k] = rc * rc;
            pot.sig2[k] = sig * sig;
            pot.eps4[k] = 4.0 * eps;
            pot.eps48[k] = 48.0 * eps;
            pot.shift[k] = p->shift ? 4.0 * eps * (sr6 * sr6 - sr6) : 0.0;
            rcmax = rc > rcmax ? rc : rcmax;
        }
    if (!(box > 2.0 * rcmax) || !(box < 1e300))
        return fail(MD_E_INVAL, "md_forces_noalloc: box must be finite and exceed twice the largest cutoff");

    // once per device, with that device current: the scratch array's address
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
        return fail(MD_E_CUDA, "md_forces_noalloc: no usable current device");
    Scratch *s;
    {
        std::lock_guard<std::mutex> lk(g_lock);
        if (!g_addr[dev]) {
            void *ptr = nullptr;
            if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr)
                return fail(MD_E_CUDA, "md_forces_noalloc: cudaGetSymbolAddress of the scratch area failed");
            g_addr[dev] = (Scratch *)ptr;
        }
        s = g_addr[dev];
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    static_assert(offsetof(Scratch, bad) == offsetof(Scratch, ticket) + sizeof(unsigned int), "adjacent words");
    if (cudaMemsetAsync(&s->ticket, 0, 2 * sizeof(unsigned int), st) != cudaSuccess)
        return fail(MD_E_CUDA, "md_forces_noalloc: clearing the scratch ticket failed");
    // margin of the single-precision test: the fractions are off by 2.5 units in a difference,
    // its conversion and the sum of squares by a few 2^-24 of it
    const double unit = box / 4294967296.0;
    for (int k = 0; k < 4; ++k) {
        const double rc = sqrt(pot.rc2[k]) * (1.0 + 1e-6) / unit + 8.0;
        pot.rc2u[k] = (float)(rc * rc * (1.0 + 1e-6));
    }
    // few particles: smaller blocks, to spread over the SMs
    const int nsp = p->n_species;
    const bool fp64 = p->precision == MD_PREC_FP64;
    if (n <= 16384)
        launch<4>(fp64, st, pot, (int)n, nsp, box, species, pos, force, energy, totals, s);
    else
        launch<8>(fp64, st, pot, (int)n, nsp, box, species, pos, force, energy, totals, s);
    if (cudaGetLastError() != cudaSuccess)
        return fail(MD_E_CUDA, "md_forces_noalloc: kernel launch failed");
    return MD_OK;
}
