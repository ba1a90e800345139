// md_kernels.cuh -- the MD step kernels, templated on the precision mode.
//
// Included by one translation unit per precision (md_kernels_{fp64,mixed,fp32}.cu),
// each of which instantiates every kernel for its mode and exports a table of
// kernel entry addresses.  All kernels take one KArgs by value.
//
// State layout in device memory (slot order = cell order after each rebuild):
//   MIXED  pos: float4 (H.x, H.y, H.z, species bits) + float4 (l.x, l.y, l.z, 0);
//               position = H + l with H on a power-of-two grid (see anchor_wrap)
//          vel: float4 high words + float4 low words (normalised double-single)
//   FP64   pos: d4 (x, y, z, species bits), vel: d4
//   FP32   pos: float4 (x, y, z, species bits), vel: float4
//   force: float4 (MIXED, FP32) or d4 (FP64): (Fx, Fy, Fz, e_i)
//   image: int4 (nx, ny, nz, original index)
// Positions are double-buffered (Ctl::pos_par): the step kernel reads the
// current buffer for every neighbour and writes the drifted positions into the
// other one.  Velocities and images are double-buffered by Ctl::state_par,
// which changes only when a rebuild permutes the particles.
//
// One kernel, k_run, does all of md_step in one cooperative launch (one block
// per SM): the opening half kick and drift, the MD steps -- pair forces over
// the neighbour list, then, per particle, the velocity-Verlet half kick that
// completes v(t), the kinetic sample, the half kick that starts the next step
// and the drift (Sec. 2.2) --, and the list rebuilds that the displacement
// criterion of Sec. 2.2 calls for.  Force evaluations outside md_step are
// launches of the same kernel.
#pragma once

#include <type_traits>

#include "md_common.cuh"

namespace mdk {

constexpr int kIntBlock = 256;   // per-particle kernels: one thread per particle
constexpr int kForceBlock = 128; // run kernel: threads of a group (tpp threads per particle)
constexpr int kPartF = 12;       // doubles per partial sum of a sample step
constexpr int kUnr = 8;          // list entries per lane and iteration of the FP32 pair loops
                                 // (a multiple of 4, at most 8: lists are padded to 8)
constexpr int kPfDepth = 1;      // iterations ahead at which the list indices are loaded

// Bounds-checked build (compile with -DMD_CHECK_BOUNDS=1; off in the product
// library): every index read from device memory (list entries, cell keys,
// permutation slots) is tested against its array before use.
#ifndef MD_CHECK_BOUNDS
#define MD_CHECK_BOUNDS 0
#endif
constexpr bool kCheckBounds = MD_CHECK_BOUNDS != 0;

// i unchanged if 0 <= i < n; otherwise (checked builds) ST_BOUNDS is recorded
// and `safe` returned, so that the access stays inside the array.
__device__ __forceinline__ int checked(const KArgs &a, int i, int n, int safe)
{
    if constexpr (kCheckBounds) {
        if ((unsigned int)i >= (unsigned int)n) {
            atomicOr(&a.ctl->status, ST_BOUNDS);
            return safe;
        }
    }
    return i;
}

// ---------------------------------------------------------------------------
// Groups of kForceBlock threads.  The run kernel launches one block per SM and
// splits it into groups that work like blocks of their own (a chunk of particles
// or a cell each), synchronised by a named barrier each; only the grid barrier
// joins them, so it has one arrival and one poller per SM.
// ---------------------------------------------------------------------------
struct Grp {
    int id, vb, nvb;                   // group of the block, of the grid, groups in the grid
    __device__ __forceinline__ static int tid() { return threadIdx.x & (kForceBlock - 1); }
    __device__ __forceinline__ void sync() const
    {
        asm volatile("bar.sync %0, %1;" ::"r"(id + 1), "n"(kForceBlock) : "memory");
    }
};

// ---------------------------------------------------------------------------
// small helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// maximum of non-negative floats (NaN counts as 0): their bits order like them
__device__ __forceinline__ float warp_max(float v)
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(v, 0.f))));
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum NV doubles over the block in a fixed order; thread 0 ends with the sums.
// sh: shared scratch of 32*NV doubles.  Every thread of the block must call it.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double *sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k)
        v[k] = warp_sum(v[k]);
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k)
            sh[w * NV + k] = v[k];
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double x = lane < nw ? sh[lane * NV + k] : 0.0;
            v[k] = warp_sum(x);
        }
    }
    __syncthreads();
}

// Sums of 12 doubles over a group in a fixed order; valid in its thread 0.  Each
// butterfly step halves the values a lane still holds, so a warp takes 16 FP64
// additions, where 12 butterflies take 60: on this GPU a warp-wide FP64 addition
// keeps its pipe for ~18 cycles of the SM (the reductions of a sample step at KA
// N=65536 took 15 us that way).  sh: kGrpWarps*kPartF doubles.  Every thread of
// the group must call it.
constexpr int kGrpWarps = kForceBlock / 32;

__device__ __forceinline__ void grp_sum(const Grp &g, double (&v)[kPartF], double *sh)
{
    const int lane = threadIdx.x & 31, w = g.tid() >> 5;
    double x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {                        // lanes 16..31 go on with values 8..15 (12..15: 0)
        const double up = k + 8 < kPartF ? v[k + 8] : 0.0;
        const double give = lane & 16 ? v[k] : up, keep = lane & 16 ? up : v[k];
        x[k] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int o = 8, n = 4; n >= 1; o >>= 1, n >>= 1)
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const double give = lane & o ? x[k] : x[k + n], keep = lane & o ? x[k + n] : x[k];
            x[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
    // value of the lane: bit 16 -> 8, 8 -> 4, 4 -> 2, 2 -> 1
    const int k = (lane >> 1) & 15;
    if (!(lane & 1) && k < kPartF)
        sh[w * kPartF + k] = x[0];
    g.sync();
    if (g.tid() == 0) {
#pragma unroll
        for (int q = 0; q < kPartF; ++q) {
            double y = sh[q];
#pragma unroll
            for (int u = 1; u < kGrpWarps; ++u)
                y += sh[u * kPartF + q];
            v[q] = y;
        }
    }
    g.sync();
}

// Maxima of three non-negative floats over a group; valid in its thread 0.
__device__ __forceinline__ void grp_max3(const Grp &g, float &a, float &b, float &c, float *sh)
{
    const int lane = threadIdx.x & 31, w = g.tid() >> 5;
    a = warp_max(a);
    b = warp_max(b);
    c = warp_max(c);
    if (lane == 0) {
        sh[3 * w] = a;
        sh[3 * w + 1] = b;
        sh[3 * w + 2] = c;
    }
    g.sync();
    if (g.tid() == 0) {
#pragma unroll
        for (int u = 1; u < kGrpWarps; ++u) {
            a = fmaxf(a, sh[3 * u]);
            b = fmaxf(b, sh[3 * u + 1]);
            c = fmaxf(c, sh[3 * u + 2]);
        }
    }
}

// Sum of the energies over a group, in double or double-single (FP32
// arithmetic): warps by shuffles in a fixed butterfly order, then the warps'
// sums in order; valid in thread 0.  shf: 2 floats per warp (8-byte aligned).
__device__ __forceinline__ double e_warp(double e) { return warp_sum(e); }
__device__ __forceinline__ ds e_warp(ds e)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        e = ds_add(e, ds_from(__shfl_xor_sync(0xffffffffu, e.hi, o), __shfl_xor_sync(0xffffffffu, e.lo, o)));
    return e;
}
__device__ __forceinline__ double e_add(double x, double y) { return x + y; }
__device__ __forceinline__ ds e_add(ds x, ds y) { return ds_add(x, y); }

template <class E>
__device__ __forceinline__ void grp_esum(const Grp &g, E &e, float *shf)
{
    E *sh = reinterpret_cast<E *>(shf);
    e = e_warp(e);
    if ((threadIdx.x & 31) == 0)
        sh[g.tid() >> 5] = e;
    g.sync();
    if (g.tid() == 0) {
#pragma unroll
        for (int u = 1; u < kGrpWarps; ++u)
            e = e_add(e, sh[u]);
    }
}

__device__ __forceinline__ int species_of(float w) { return __float_as_int(w) & 15; }
__device__ __forceinline__ int species_of(double w) { return (int)(__double_as_longlong(w) & 15); }

// buffer selection by parity
__device__ __forceinline__ void *pos_a(const KArgs &a, int par) { return par ? a.pa2 : a.pa; }
__device__ __forceinline__ void *pos_b(const KArgs &a, int par) { return par ? a.pb2 : a.pb; }
__device__ __forceinline__ void *vel_a(const KArgs &a, int par) { return par ? a.va2 : a.va; }
__device__ __forceinline__ void *vel_b(const KArgs &a, int par) { return par ? a.vb2 : a.vb; }
__device__ __forceinline__ int4 *img_of(const KArgs &a, int par) { return par ? a.image2 : a.image; }

// Re-anchor a double-single coordinate so that its high word lies on the grid
// of spacing `grid` (a power of two chosen so that every coordinate in
// [-L, 2L) is exactly representable on it), then wrap it into [0, L).
// Shifting an anchored high word by the anchored box edge Lhi is exact in
// single precision, so the wrap loses nothing; differences of high words are
// exact too (the displacement check uses them).  The pair loops read the
// fixed-point copy instead (fixq).  Returns the change of the image counter
// (-1, 0, 1).
__device__ __forceinline__ int anchor_wrap(ds x, float grid, float inv_grid, float Lhi, float Llo,
                                           float &H, float &l)
{
    float h = __fmul_rn(rintf(__fmul_rn(x.hi, inv_grid)), grid);  // power-of-two scalings: exact
    float r = __fadd_rn(__fsub_rn(x.hi, h), x.lo);                 // x.hi - h is exact
    int img = 0;
    if (h > Lhi || (h == Lhi && r >= Llo)) {
        h = __fsub_rn(h, Lhi);
        r = __fsub_rn(r, Llo);
        img = 1;
    } else if (h < 0.0f || (h == 0.0f && r < 0.0f)) {
        h = __fadd_rn(h, Lhi);
        r = __fadd_rn(r, Llo);
        img = -1;
    }
    H = h;
    l = r;
    return img;
}

__device__ __forceinline__ float sep_f(float xi, float xj, float L, float invL)
{
    float d = xi - xj;
    return fmaf(-rintf(d * invL), L, d);
}

__device__ __forceinline__ double sep_d(double xi, double xj, double L, double invL)
{
    double d = xi - xj;
    return fma(-rint(d * invL), L, d);
}

// Fixed-point position (MIXED): x / L in units of 2^-32, modulo 2^32, from
// the exact double value of a double-single coordinate.  The periodic box is
// the full 32-bit circle, so the 32-bit wrapped difference of two coordinates
// is the minimum-image separation, exact in integers; only its conversion to
// single precision rounds.  One unit is L / 2^32 (8.8e-9 sigma at L = 38).
//
// Without FP64 (whose pipe is narrow on this GPU): the high word is an
// integer number m of grid steps (0 <= m < 2^24, exact), so x 2^32 / L =
// m C + l 2^32 / L with C = grid 2^32 / L in (2^9, 2^10].  m C is formed in
// 64-bit integers from C in units of 2^-28 (error < 2^-5 units) and rounded;
// |l| <= grid, so l 2^32 / L (at most C, single precision, error < 2^-13
// units) is rounded on its own.  The result is within 1 + 2^-5 units of the
// exact value (two roundings), the same in every kernel.
__device__ __forceinline__ unsigned int fixq(float H, float l, const Rep &rp)
{
    const unsigned int m = (unsigned int)__float2int_rn(__fmul_rn(H, rp.inv_grid));   // exact
    const unsigned long long hi = ((unsigned long long)m * rp.qgrid + (1ull << 27)) >> 28;
    return (unsigned int)hi + (unsigned int)__float2int_rn(__fmul_rn(l, rp.qscale));
}

__device__ __forceinline__ float sep_q(unsigned int qi, unsigned int qj, float unit)
{
    return __int2float_rn((int)(qi - qj)) * unit;
}

// two at a time
__device__ __forceinline__ float2 sep_q2(int qi, int qa, int qb, float unit)
{
    return __fmul2_rn(make_float2(__int2float_rn((int)((unsigned int)qi - (unsigned int)qa)),
                                  __int2float_rn((int)((unsigned int)qi - (unsigned int)qb))),
                      make_float2(unit, unit));
}

// minimum-image separations of one coordinate from two others (FP32 mode): the
// rounding to a whole number of boxes adds and takes away 1.5 2^23
__device__ __forceinline__ float2 sep_f2(float xi, float2 xj, float L, float invL)
{
    const float2 d = __fadd2_rn(make_float2(xi, xi), make_float2(-xj.x, -xj.y));
    const float2 big = make_float2(12582912.0f, 12582912.0f);
    const float2 t = __ffma2_rn(d, make_float2(invL, invL), big);
    const float2 k = __fadd2_rn(t, make_float2(-12582912.0f, -12582912.0f));
    return __ffma2_rn(k, make_float2(-L, -L), d);
}

// reciprocal of a normal number by the hardware's approximation (1 ulp)
__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int4 *q_of(const KArgs &a, int par) { return par ? a.qb : a.qa; }

// Kahan-compensated accumulation: the running sum is s - c.
__device__ __forceinline__ void kahan_add(float &s, float &c, float x)
{
    float y = __fsub_rn(x, c);
    float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
}

// Smoothing of Sec. 4: U = V g(x), g(x) = x^4 / (1 + x^4), x = (r - r_c) / (h sigma_ab).
// On entry fr = -V'(r)/r and v = V(r); on exit fr = -U'(r)/r and v = U(r):
//   -U'/r = (-V'/r) g - V g'(x) / (h sigma r),  g'(x) = 4 x^3 / (1 + x^4)^2.
__device__ __forceinline__ void smooth_pair(float r2, float rc, float ihs, float &fr, float &v)
{
    const float rinv = rsqrtf(r2);
    const float x = (r2 * rinv - rc) * ihs;
    const float x2 = x * x, x4 = x2 * x2;
    const float den = __fdividef(1.0f, 1.0f + x4);
    const float g = x4 * den;
    const float dg = 4.0f * x2 * x * den * den;
    fr = fr * g - v * dg * ihs * rinv;
    v = v * g;
}

__device__ __forceinline__ void smooth_pair(double r2, double rc, double ihs, double &fr, double &v)
{
    const double r = sqrt(r2);
    const double x = (r - rc) * ihs;
    const double x2 = x * x, x4 = x2 * x2;
    const double den = 1.0 / (1.0 + x4);
    const double g = x4 * den;
    const double dg = 4.0 * x2 * x * den * den;
    fr = fr * g - v * dg * ihs / r;
    v = v * g;
}

template <int P> using FT = typename std::conditional<P == FP64, double, float>::type;

// Per-particle potential energy and its block sums: double in FP64 mode,
// double-single (FP32 arithmetic) otherwise, so that the every-step energy
// reduction adds no FP64 instruction to the single-precision modes.
template <int P> using ET = typename std::conditional<P == FP64, double, ds>::type;
__device__ __forceinline__ double e_value(double e) { return e; }
__device__ __forceinline__ double e_value(ds e) { return ds_to_double(e); }
__device__ __forceinline__ float e_float(double e) { return (float)e; }
__device__ __forceinline__ float e_float(ds e) { return __fadd_rn(e.hi, e.lo); }
template <int P> __device__ __forceinline__ ET<P> e_zero()
{
    if constexpr (P == FP64)
        return 0.0;
    else
        return ds_from(0.f, 0.f);
}

// ---------------------------------------------------------------------------
// Per-particle velocity-Verlet pieces (Sec. 2.2), in the precision's state
// representation: MIXED updates velocities and positions in double-single
// (Sec. 2.4), FP64 in double, FP32 in float.
// ---------------------------------------------------------------------------
template <int P> struct PState;
template <> struct PState<MIXED> { float4 H, l; ds vx, vy, vz; int sp; };
template <> struct PState<FP64> { d4 x; double vx, vy, vz; int sp; };
template <> struct PState<FP32> { float4 x; float vx, vy, vz; int sp; };

template <int P>
__device__ __forceinline__ void load_pos(const KArgs &a, int pp, int i, PState<P> &s)
{
    if constexpr (P == MIXED) {
        s.H = ((const float4 *)pos_a(a, pp))[i];
        s.l = ((const float4 *)pos_b(a, pp))[i];
        s.sp = species_of(s.H.w);
    } else if constexpr (P == FP64) {
        s.x = ((const d4 *)pos_a(a, pp))[i];
        s.sp = species_of(s.x.w);
    } else {
        s.x = ((const float4 *)pos_a(a, pp))[i];
        s.sp = species_of(s.x.w);
    }
}

template <int P>
__device__ __forceinline__ void load_vel(const KArgs &a, int sp, int i, PState<P> &s)
{
    if constexpr (P == MIXED) {
        const float4 h = ((const float4 *)vel_a(a, sp))[i], l = ((const float4 *)vel_b(a, sp))[i];
        s.vx = ds_from(h.x, l.x);
        s.vy = ds_from(h.y, l.y);
        s.vz = ds_from(h.z, l.z);
    } else if constexpr (P == FP64) {
        const d4 v = ((const d4 *)vel_a(a, sp))[i];
        s.vx = v.x; s.vy = v.y; s.vz = v.z;
    } else {
        const float4 v = ((const float4 *)vel_a(a, sp))[i];
        s.vx = v.x; s.vy = v.y; s.vz = v.z;
    }
}

template <int P>
__device__ __forceinline__ void store_vel(const KArgs &a, int sp, int i, const PState<P> &s)
{
    if constexpr (P == MIXED) {
        ((float4 *)vel_a(a, sp))[i] = make_float4(s.vx.hi, s.vy.hi, s.vz.hi, 0.f);
        ((float4 *)vel_b(a, sp))[i] = make_float4(s.vx.lo, s.vy.lo, s.vz.lo, 0.f);
    } else if constexpr (P == FP64) {
        d4 v;
        v.x = s.vx; v.y = s.vy; v.z = s.vz; v.w = 0.0;
        ((d4 *)vel_a(a, sp))[i] = v;
    } else {
        ((float4 *)vel_a(a, sp))[i] = make_float4(s.vx, s.vy, s.vz, 0.f);
    }
}

// v += dt/(2m) f
template <int P>
__device__ __forceinline__ void half_kick(const KArgs &a, PState<P> &s, FT<P> fx, FT<P> fy, FT<P> fz)
{
    if constexpr (P == MIXED) {
        const ds hk = ds_from(a.hdtm_hi[s.sp], a.hdtm_lo[s.sp]);
        s.vx = ds_add(s.vx, ds_mul_f(hk, fx));
        s.vy = ds_add(s.vy, ds_mul_f(hk, fy));
        s.vz = ds_add(s.vz, ds_mul_f(hk, fz));
    } else if constexpr (P == FP64) {       // (roundings spelled out: the same in every kernel)
        const double hk = a.hdtm[s.sp];
        s.vx = fma(hk, fx, s.vx);
        s.vy = fma(hk, fy, s.vy);
        s.vz = fma(hk, fz, s.vz);
    } else {
        const float hk = a.hdtm_hi[s.sp];
        s.vx = fmaf(hk, fx, s.vx);
        s.vy = fmaf(hk, fy, s.vy);
        s.vz = fmaf(hk, fz, s.vz);
    }
}

// kinetic energy and momentum of the particle in FP64: kin[0..3]
template <int P>
__device__ __forceinline__ void kinetic(const KArgs &a, const PState<P> &s, double *kin)
{
    double vx, vy, vz;
    if constexpr (P == MIXED) {
        vx = ds_to_double(s.vx); vy = ds_to_double(s.vy); vz = ds_to_double(s.vz);
    } else {
        vx = s.vx; vy = s.vy; vz = s.vz;
    }
    const double m = a.mass[s.sp];
    kin[0] = __dmul_rn(0.5 * m, fma(vz, vz, fma(vy, vy, __dmul_rn(vx, vx))));
    kin[1] = m * vx;
    kin[2] = m * vy;
    kin[3] = m * vz;
}

// |v|^2 and |d|^2 feed the rebuild decision, which sets the particle order and
// so the summation order: their roundings are spelled out, so that every
// kernel that computes them decides alike.
__device__ __forceinline__ float norm2f(float x, float y, float z)
{
    return fmaf(z, z, fmaf(y, y, __fmul_rn(x, x)));
}
__device__ __forceinline__ float norm2(float x, float y, float z) { return norm2f(x, y, z); }
__device__ __forceinline__ float norm2(double x, double y, double z)
{
    return (float)fma(z, z, fma(y, y, __dmul_rn(x, x)));
}
__device__ __forceinline__ float speed2(const PState<MIXED> &s) { return norm2f(s.vx.hi, s.vy.hi, s.vz.hi); }
__device__ __forceinline__ float speed2(const PState<FP64> &s) { return norm2(s.vx, s.vy, s.vz); }
__device__ __forceinline__ float speed2(const PState<FP32> &s) { return norm2f(s.vx, s.vy, s.vz); }

// r += dt v, wrapped into [0, L) with image counting; writes the new position
// into buffer `dst`, updates the image counter in the state buffers `spar`,
// returns the squared displacement since the last list build (if wanted: `track`).
template <int P>
__device__ __forceinline__ float drift(const KArgs &a, const Rep &rp, PState<P> &s, int dst, int spar, int i, bool track,
                                       unsigned int &bad)
{
    int ix, iy, iz;
    float dd = 0.f;
    if constexpr (P == MIXED) {
        const ds dt = ds_from(a.dt_hi, a.dt_lo);
        const ds sx = ds_mul(dt, s.vx), sy = ds_mul(dt, s.vy), sz = ds_mul(dt, s.vz);
        const float lim = 0.25f * rp.Lhi;
        if (fabsf(sx.hi) > lim || fabsf(sy.hi) > lim || fabsf(sz.hi) > lim)
            bad |= ST_UNSTABLE;
        const ds nx = ds_add(ds_from(s.H.x, s.l.x), sx);
        const ds ny = ds_add(ds_from(s.H.y, s.l.y), sy);
        const ds nz = ds_add(ds_from(s.H.z, s.l.z), sz);
        ix = anchor_wrap(nx, rp.grid, rp.inv_grid, rp.Lhi, rp.Llo, s.H.x, s.l.x);
        iy = anchor_wrap(ny, rp.grid, rp.inv_grid, rp.Lhi, rp.Llo, s.H.y, s.l.y);
        iz = anchor_wrap(nz, rp.grid, rp.inv_grid, rp.Lhi, rp.Llo, s.H.z, s.l.z);
        if (!isfinite(s.H.x) || !isfinite(s.H.y) || !isfinite(s.H.z))
            bad |= ST_NONFINITE;
        ((float4 *)pos_a(a, dst))[i] = s.H;
        ((float4 *)pos_b(a, dst))[i] = s.l;
        q_of(a, dst)[i] = make_int4((int)fixq(s.H.x, s.l.x, rp), (int)fixq(s.H.y, s.l.y, rp),
                                    (int)fixq(s.H.z, s.l.z, rp), s.sp);
        if (track) {
            const float4 rr = a.rref[i];
            const float ex = __fadd_rn(sep_f(s.H.x, rr.x, rp.Lhi, rp.invLf), s.l.x);
            const float ey = __fadd_rn(sep_f(s.H.y, rr.y, rp.Lhi, rp.invLf), s.l.y);
            const float ez = __fadd_rn(sep_f(s.H.z, rr.z, rp.Lhi, rp.invLf), s.l.z);
            dd = norm2f(ex, ey, ez);
        }
    } else if constexpr (P == FP64) {
        const double sx = __dmul_rn(a.dt, s.vx), sy = __dmul_rn(a.dt, s.vy), sz = __dmul_rn(a.dt, s.vz);
        const double lim = 0.25 * rp.L;
        if (fabs(sx) > lim || fabs(sy) > lim || fabs(sz) > lim)
            bad |= ST_UNSTABLE;
        double x = __dadd_rn(s.x.x, sx), y = __dadd_rn(s.x.y, sy), z = __dadd_rn(s.x.z, sz);
        ix = iy = iz = 0;
        if (x >= rp.L) { x -= rp.L; ix = 1; } else if (x < 0.0) { x += rp.L; ix = -1; }
        if (y >= rp.L) { y -= rp.L; iy = 1; } else if (y < 0.0) { y += rp.L; iy = -1; }
        if (z >= rp.L) { z -= rp.L; iz = 1; } else if (z < 0.0) { z += rp.L; iz = -1; }
        if (!isfinite(x) || !isfinite(y) || !isfinite(z))
            bad |= ST_NONFINITE;
        s.x.x = x; s.x.y = y; s.x.z = z;
        ((d4 *)pos_a(a, dst))[i] = s.x;
        if (track) {
            const float4 rr = a.rref[i];
            const float ex = sep_f(__double2float_rn(x), rr.x, rp.Lhi, rp.invLf);
            const float ey = sep_f(__double2float_rn(y), rr.y, rp.Lhi, rp.invLf);
            const float ez = sep_f(__double2float_rn(z), rr.z, rp.Lhi, rp.invLf);
            dd = norm2f(ex, ey, ez);
        }
    } else {
        const float dt = a.dt_hi;
        const float sx = __fmul_rn(dt, s.vx), sy = __fmul_rn(dt, s.vy), sz = __fmul_rn(dt, s.vz);
        const float L = rp.Lhi;
        if (fabsf(sx) > 0.25f * L || fabsf(sy) > 0.25f * L || fabsf(sz) > 0.25f * L)
            bad |= ST_UNSTABLE;
        float x = __fadd_rn(s.x.x, sx), y = __fadd_rn(s.x.y, sy), z = __fadd_rn(s.x.z, sz);
        ix = iy = iz = 0;
        if (x >= L) { x -= L; ix = 1; } else if (x < 0.f) { x += L; ix = -1; }
        if (y >= L) { y -= L; iy = 1; } else if (y < 0.f) { y += L; iy = -1; }
        if (z >= L) { z -= L; iz = 1; } else if (z < 0.f) { z += L; iz = -1; }
        // a coordinate just below 0 can round to L when wrapped: it is 0 of the
        // original image
        if (x >= L) { x = 0.f; ix += 1; }
        if (y >= L) { y = 0.f; iy += 1; }
        if (z >= L) { z = 0.f; iz += 1; }
        if (!isfinite(x) || !isfinite(y) || !isfinite(z))
            bad |= ST_NONFINITE;
        s.x.x = x; s.x.y = y; s.x.z = z;
        ((float4 *)pos_a(a, dst))[i] = s.x;
        if (track) {
            const float4 rr = a.rref[i];
            const float ex = sep_f(x, rr.x, L, rp.invLf);
            const float ey = sep_f(y, rr.y, L, rp.invLf);
            const float ez = sep_f(z, rr.z, L, rp.invLf);
            dd = norm2f(ex, ey, ez);
        }
    }
    if (ix | iy | iz) {
        int4 *im = img_of(a, spar);
        int4 q = im[i];
        q.x += ix;
        q.y += iy;
        q.z += iz;
        im[i] = q;
    }
    return dd;
}

// ---------------------------------------------------------------------------
// Per-step reductions.  Every block of the run kernel leaves one partial per
// slot: the potential energy of the step (part_e: double in FP64 mode,
// double-single elsewhere, so that the every-step sum costs no FP64 arithmetic
// in the single-precision modes) and, on sample steps, the virial, kinetic and
// momentum sums (part_f).  A slot is a block for a handle of one replica and a
// chunk otherwise (a block may hold chunks of several replicas).  Two sets, by
// the parity of the step, so that one block can add up a step's partials while
// the others already write the next step's.
// ---------------------------------------------------------------------------
__device__ __forceinline__ size_t part_index(const KArgs &a, long long step, int slot)
{
    return (size_t)(step & 1) * (size_t)a.nslot + (size_t)slot;
}

template <int P>
__device__ __forceinline__ void put_epart(const KArgs &a, size_t k, ET<P> e)
{
    if constexpr (P == FP64)
        ((double *)a.part_e)[k] = e;
    else
        ((float2 *)a.part_e)[k] = make_float2(e.hi, e.lo);
}

template <int P>
__device__ __forceinline__ ET<P> get_epart(const KArgs &a, size_t k)
{
    if constexpr (P == FP64) {
        return ((const double *)a.part_e)[k];
    } else {
        const float2 x = ((const float2 *)a.part_e)[k];
        return ds_from(x.x, x.y);
    }
}

// The reductions of replica r at `step` from its slots' partials, by one
// group, in a fixed order (thread t adds partials t, t + 128, ..., then the
// group's tree): the potential energy into the per-step series and, for a
// sample, the record into the ring or (totals) into the totals array.
template <int P>
__device__ void finish_replica(const KArgs &a, const Grp &g, int r, long long step, bool sample, bool totals, long long slot,
                               float md2, long long rebuilds, double *sh, float *shf)
{
    const int s0 = a.nrep == 1 ? 0 : a.rep[r].bf0, s1 = a.nrep == 1 ? a.nslot : a.rep[r].bf1;
    ET<P> e = e_zero<P>();
    int b = s0 + g.tid();
    const int st = kForceBlock;
    for (; b + 7 * st < s1; b += 8 * st) {
        ET<P> x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            x[u] = get_epart<P>(a, part_index(a, step, b + u * st));
#pragma unroll
        for (int u = 0; u < 8; ++u)
            e = e_add(e, x[u]);
    }
    for (; b < s1; b += st)
        e = e_add(e, get_epart<P>(a, part_index(a, step, b)));
    grp_esum(g, e, shf);
    const double epot = e_value(e);
    if (g.tid() == 0 && !totals)
        a.epot[(step % a.epot_cap) * a.nrep + r] = epot;
    if (!sample) {
        g.sync();                                    // (shf is written again)
        return;
    }
    double v[kPartF];
#pragma unroll
    for (int k = 0; k < kPartF; ++k)
        v[k] = 0.0;
    for (int b2 = s0 + g.tid(); b2 < s1; b2 += st) {
        const double *p = a.part_f + part_index(a, step, b2) * kPartF;
#pragma unroll
        for (int k = 1; k < kPartF; ++k)
            v[k] += p[k];
    }
    grp_sum(g, v, sh);
    if (g.tid() == 0) {
        Obs o;
        o.step = step;
        o.e_pot = epot;
        o.virial = v[1];
        for (int k = 0; k < 6; ++k)
            o.w[k] = v[2 + k];
        o.e_kin = v[8];
        o.p[0] = v[9];
        o.p[1] = v[10];
        o.p[2] = v[11];
        o.max_disp = sqrt((double)md2);
        o.rebuilds = rebuilds;
        if (totals)
            a.totals[r] = o;
        else
            a.ring[slot * a.nrep + r] = o;
    }
}

// Rebuild decision: the list built at the last rebuild holds every pair
// within r_c + skin, so it stays complete while no particle has moved more
// than skin/2.  The next check comes after `look` further drifts, each at
// most dt (v + look dt a) per particle: rebuild now if the largest
// displacement plus that bound could exceed skin/2 (with a rounding margin).
__device__ __forceinline__ bool need_rebuild(const KArgs &a, int lookahead, float md2, float mv2, float ma2)
{
    const float look = (float)lookahead * (float)a.dt;
    const float d = sqrtf(md2) + look * (sqrtf(mv2) + 2.0f * look * sqrtf(ma2));
    return d > a.disp_thr;
}

// ---------------------------------------------------------------------------
// pair forces over the neighbour list (Sec. 2.2), 12-6 potential cut (and
// shifted) at r_c,ab (Sec. 3, Sec. 5).  TPP threads share one particle; each
// lane takes groups of consecutive list entries (16-byte index loads) and
// issues their gathers together.  List rows are padded with the particle
// itself to whole groups of 8 (r^2 = 0 exactly: never inside), so the loops
// carry no end-of-row masks.  Single precision: a group's contributions are
// summed branch-free (zero factor outside the cutoff) and the group sum enters
// a Kahan accumulator (MIXED; plain sum for FP32); lanes are combined in
// double-single.  The pair potential is summed alongside, every step (the
// potential energy is a per-step reduction of Sec. 2.2).  On return every lane
// of the particle holds the total force and ep, half the sum of its pair
// energies; the virial comes from pair_energy on sample steps.
// ---------------------------------------------------------------------------
// 1/24 as a double-single pair (the accumulated energies are 12 V; a particle
// takes half of each pair)
constexpr float kE24hi = (float)(1.0 / 24.0);
constexpr float kE24lo = (float)(1.0 / 24.0 - (double)(float)(1.0 / 24.0));

// FP64 mode: the FP64 pipe is narrow on this GPU (a warp-wide instruction keeps
// it for ~18 cycles of the SM whatever the number of active lanes), so it sees
// nothing but pairs inside the cutoff, spread evenly over the lanes.  A warp
// takes its particles' rows in rounds of kPairQ entries: a single-precision test
// with a margin (on coordinates cut to float by integer operations) queues the
// partners that can be inside, then every lane takes an equal run of the queue,
// whatever particles it belongs to, and leaves one partial sum per particle of
// its run; each particle adds its partials in lane order.  The reciprocal of r^2
// is one third-order Newton step on the hardware's 20-bit estimate.  22 FP64
// instructions per pair instead of ~40 per list entry with an IEEE division and
// a product and rounding per nearest image: KA N=16384, 4 lanes, 159 -> 102 us a
// step.
constexpr int kPairQ = 512;          // queued entries per round and warp: 16 list entries a lane
constexpr int kPairLane = kPairQ / 32;

struct PairQueue {
    double x[32][4];                 // the warp's particles: position and species bits
    double slot[64][4];              // partial sums (force, 12 V) by lane + particle
    int q[kPairQ];
    int first[33];                   // first queue entry of each particle
};

// A double's value cut to float precision, by integer operations (values below
// 2^-127 become tiny ones; infinities and NaN become ordinary numbers: a particle
// with such a coordinate is in nobody's list or fails the FP64 test, and its next
// drift reports it).
__device__ __forceinline__ float cut_float(double x)
{
    const unsigned int hi = (unsigned int)__double2hiint(x), lo = (unsigned int)__double2loint(x);
    const unsigned int e = max(hi & 0x7fffffffu, 896u << 20) - (896u << 20);
    return __uint_as_float((hi & 0x80000000u) | (e << 3) | (lo >> 29));
}

// 1/x of a normal number: y (1 + e + e^2) with e = 1 - x y, from the hardware's estimate
// y, whose relative error is below 2^-19.  The terms left out are below 2^-57, so
// the error is that of the last rounding, at most 2^-53 (1 + 2^-4).
__device__ __forceinline__ double rcp_newton(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

template <int TPP, bool SM>
__device__ __forceinline__ void pair_forces_d(const KArgs &a, const Rep &rp, int pp, int ii, int nn, PairQueue &Q,
                                              double &fx, double &fy, double &fz, double &ep)
{
    constexpr int PPW = 32 / TPP;                        // particles of the warp
    const int wl = threadIdx.x & 31, lane = wl & (TPP - 1), me = wl / TPP;
    const int *lst = a.nbr + (size_t)ii * (size_t)a.Kstride;
    const d4 *pos = (const d4 *)pos_a(a, pp);
    const d4 xi = pos[ii];
    const float L = (float)rp.L, half = 0.5f * L;
    const float xf = cut_float(xi.x), yf = cut_float(xi.y), zf = cut_float(xi.z);
    // cutoffs with the margin of the single-precision test.  A coordinate cut to 24 bits
    // is off by less than L 2^-23, always downwards, so a difference by as much; its
    // rounding, L in single precision and a shift on the wrong side of half a box add at
    // most twice that again: d = 3 L 2^-23 per component, 2 sqrt(3) r_c d + 3 d^2 in r^2,
    // and four roundings of r_c^2.  Taken: (16 r_c L + 4 r_c^2) 2^-23 + (8 L 2^-23)^2.
    float rc2f[2];
#pragma unroll
    for (int tj = 0; tj < 2; ++tj) {
        const int ab = species_of(xi.w) * 2 + tj;
        const float dl = L * 0x1p-20f;
        rc2f[tj] = a.tab.rc2[ab] + (fmaf(a.tab.rc[ab], 2.0f * dl, a.tab.rc2[ab] * 0x1p-21f) + dl * dl);
    }
    __syncwarp();
    if (lane == 0) {
        Q.x[me][0] = xi.x;
        Q.x[me][1] = xi.y;
        Q.x[me][2] = xi.z;
        Q.x[me][3] = xi.w;
    }
    double sx = 0.0, sy = 0.0, sz = 0.0, se = 0.0;       // of the lane's own particle; se: sum of 12 V
    const int rows = (int)__reduce_max_sync(0xffffffffu, (unsigned)nn);
    for (int r0 = 0; r0 < rows; r0 += kPairLane * TPP) {
        // queue the entries [r0, r0 + kPairLane TPP) of every row that can be inside
        const int k0 = r0 + kPairLane * lane;
        int jj[kPairLane];
        unsigned int keep = 0u;
#pragma unroll
        for (int b = 0; b < kPairLane; b += 4) {
            const bool in = k0 + b < nn;                 // (rows are padded to whole groups of 8)
            const int4 j4 = in ? *(const int4 *)(lst + k0 + b) : make_int4(ii, ii, ii, ii);
            jj[b] = j4.x;
            jj[b + 1] = j4.y;
            jj[b + 2] = j4.z;
            jj[b + 3] = j4.w;
            if (in) {
                d4 xs[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    xs[u] = pos[checked(a, jj[b + u], a.n, ii)];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    float dx = xf - cut_float(xs[u].x), dy = yf - cut_float(xs[u].y), dz = zf - cut_float(xs[u].z);
                    dx = fabsf(dx);
                    dy = fabsf(dy);
                    dz = fabsf(dz);
                    dx = dx > half ? dx - L : dx;
                    dy = dy > half ? dy - L : dy;
                    dz = dz > half ? dz - L : dz;
                    const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                    // (the padding is the particle itself)
                    if (!(r2 >= (species_of(xs[u].w) ? rc2f[1] : rc2f[0])) && jj[b + u] != ii)
                        keep |= 1u << (b + u);
                }
            }
        }
        const int n = __popc(keep);
        int incl = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (wl >= o)
                incl += y;
        }
        const int W = __shfl_sync(0xffffffffu, incl, 31);
        int at = incl - n;
        if (lane == 0)
            Q.first[me] = at;
        if (wl == 31)
            Q.first[PPW] = W;
#pragma unroll
        for (int b = 0; b < kPairLane; ++b)
            if (keep >> b & 1u)
                Q.q[at++] = jj[b];
        __syncwarp();

        // every lane takes m entries of the queue
        const int m = (W + 31) / 32;
        int t = wl * m;
        const int end = min(t + m, W);
        int p = 0;
        while (p + 1 < PPW && Q.first[p + 1] <= t)
            ++p;
        double ox = Q.x[p][0], oy = Q.x[p][1], oz = Q.x[p][2];
        int to = species_of(Q.x[p][3]) * 2;
        double gx = 0.0, gy = 0.0, gz = 0.0, ge = 0.0;
        d4 xn = pos[checked(a, t < end ? Q.q[t] : ii, a.n, ii)];   // one entry ahead
        for (int it = 0; it < m; ++it, ++t) {
            const bool on = t < end;
            const d4 xj = xn;
            xn = pos[checked(a, t + 1 < end ? Q.q[t + 1] : ii, a.n, ii)];
            if (on && t >= Q.first[p + 1]) {             // the next particle's entries
                double *s = Q.slot[wl + p];
                s[0] = gx; s[1] = gy; s[2] = gz; s[3] = ge;
                gx = gy = gz = ge = 0.0;
                do
                    ++p;
                while (t >= Q.first[p + 1]);
                ox = Q.x[p][0]; oy = Q.x[p][1]; oz = Q.x[p][2];
                to = species_of(Q.x[p][3]) * 2;
            }
            const int ab = to + species_of(xj.w);
            double dx = ox - xj.x, dy = oy - xj.y, dz = oz - xj.z;
            // nearest image: within the cutoff it is a shift by one box or none, told from
            // the high words
            const float ex = cut_float(dx), ey = cut_float(dy), ez = cut_float(dz);
            if (__any_sync(0xffffffffu, fabsf(ex) > half || fabsf(ey) > half || fabsf(ez) > half)) {
                dx = ex > half ? dx - rp.L : (ex < -half ? dx + rp.L : dx);
                dy = ey > half ? dy - rp.L : (ey < -half ? dy + rp.L : dy);
                dz = ez > half ? dz - rp.L : (ez < -half ? dz + rp.L : dz);
            }
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            // 0 < r2 < rc2, on the bits (neither is negative; a NaN is above)
            const long long bits = __double_as_longlong(r2);
            const bool in = on && bits > 0 && bits < __double_as_longlong(a.tab.rc2d[ab]);
            const double ir2 = rcp_newton(in ? r2 : 1.0);
            const double s2 = a.tab.sig2d[ab] * ir2;
            const double s6 = s2 * s2 * s2;
            const double w = s6 - 0.5;
            const double e6 = (in ? a.tab.eps48d[ab] : 0.0) * s6;
            double fr = e6 * ir2 * w;
            if (SM) {
                double v = in ? a.tab.eps4d[ab] * s6 * (s6 - 1.0) - a.tab.shiftd[ab] : 0.0;
                smooth_pair(in ? r2 : 1.0, a.tab.rcd[ab], a.tab.ihsd[ab], fr, v);
                ge = fma(12.0, v, ge);
            } else {
                ge += fma(e6, s6 - 1.0, in ? -a.tab.e48vcd[ab] : 0.0);
            }
            gx = fma(fr, dx, gx);
            gy = fma(fr, dy, gy);
            gz = fma(fr, dz, gz);
        }
        if (wl * m < end) {
            double *s = Q.slot[wl + p];
            s[0] = gx; s[1] = gy; s[2] = gz; s[3] = ge;
        }
        __syncwarp();
        // the particle's partials, in lane order
        const int q0 = Q.first[me], q1 = Q.first[me + 1];
        if (q0 < q1)
            for (int s = q0 / m + me; s <= (q1 - 1) / m + me; ++s) {
                sx += Q.slot[s][0];
                sy += Q.slot[s][1];
                sz += Q.slot[s][2];
                se += Q.slot[s][3];
            }
        __syncwarp();
    }
    fx = sx; fy = sy; fz = sz;
    ep = se * (1.0 / 24.0);
}

template <int P, int TPP, bool SM>
__device__ __forceinline__ void pair_forces(const KArgs &a, const Rep &rp, int pp, int ii, int nn, PairQueue *Q,
                                            FT<P> &fx, FT<P> &fy, FT<P> &fz, ET<P> &ep)
{
    const int lane = threadIdx.x & (TPP - 1);
    const int *lst = a.nbr + (size_t)ii * (size_t)a.Kstride;
    if constexpr (P == FP64) {
        pair_forces_d<TPP, SM>(a, rp, pp, ii, nn, *Q, fx, fy, fz, ep);
    } else {
        // MIXED reads the fixed-point copy (16 B per neighbour), FP32 the positions
        const float4 *pos = (const float4 *)pos_a(a, pp);
        const int4 *qp = q_of(a, pp);
        float4 Hi = make_float4(0.f, 0.f, 0.f, 0.f);
        int4 Qi = make_int4(0, 0, 0, 0);
        int ti;
        if constexpr (P == MIXED) {
            Qi = qp[ii];
            ti = Qi.w;
        } else {
            Hi = pos[ii];
            ti = species_of(Hi.w);
        }
        float rc2[2], sig2[2], eps48[2], vc[2];
#pragma unroll
        for (int tj = 0; tj < 2; ++tj) {
            rc2[tj] = a.tab.rc2[ti * 2 + tj];
            sig2[tj] = a.tab.sig2[ti * 2 + tj];
            eps48[tj] = a.tab.eps48[ti * 2 + tj];
            vc[tj] = a.tab.vc[ti * 2 + tj];
        }
        // the energy is accumulated as 12 V = eps48_ab (s6^2 - s6 - c_ab), c_ab = S_ab / (4 eps_ab):
        // eps48, masked by the cutoff test, serves the force and the energy alike
        float sx = 0.f, sy = 0.f, sz = 0.f, cx = 0.f, cy = 0.f, cz = 0.f, se = 0.f, ce = 0.f;
        // list indices are loaded kPfDepth iterations ahead, so that only the
        // position gathers remain on each iteration's critical path
        // (K is a multiple of 8: every 16-byte index load is in bounds and aligned)
        // (8 or more lanes: groups of 4, so that a row of ~80 entries fills the lanes evenly)
        constexpr int U = TPP >= 8 ? 4 : kUnr, kStride = U * TPP;
        int4 pf[kPfDepth][U / 4];
#pragma unroll
        for (int d = 0; d < kPfDepth; ++d)
#pragma unroll
            for (int w = 0; w < U / 4; ++w) {
                const int k = U * lane + d * kStride;
                // (the first ones without waiting for the row's length)
                pf[d][w] = k < (d == 0 ? a.Kstride : nn) ? *(const int4 *)(lst + k + 4 * w) : make_int4(0, 0, 0, 0);
            }
        for (int k0 = U * lane; k0 < nn; k0 += kStride) {
            int jj[U];
#pragma unroll
            for (int w = 0; w < U / 4; ++w) {
                const int4 q = pf[0][w];
                jj[4 * w] = q.x;
                jj[4 * w + 1] = q.y;
                jj[4 * w + 2] = q.z;
                jj[4 * w + 3] = q.w;
            }
#pragma unroll
            for (int d = 0; d + 1 < kPfDepth; ++d)
#pragma unroll
                for (int w = 0; w < U / 4; ++w)
                    pf[d][w] = pf[d + 1][w];
            if (k0 + kPfDepth * kStride < nn)
#pragma unroll
                for (int w = 0; w < U / 4; ++w)
                    pf[kPfDepth - 1][w] = *(const int4 *)(lst + k0 + kPfDepth * kStride + 4 * w);
            float4 Hs[U];
            int4 Qs[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                // rows are padded with the particle itself up to a multiple of kUnr
                const int j = checked(a, jj[u], a.n, ii);
                if constexpr (P == MIXED)
                    Qs[u] = qp[j];
                else
                    Hs[u] = pos[j];
            }
            // two entries at a time: the single-precision arithmetic of a pair of
            // entries is one packed instruction each
            float gx = 0.f, gy = 0.f, gz = 0.f, gv = 0.f;
#pragma unroll
            for (int u = 0; u < U; u += 2) {
                float2 dx, dy, dz;
                bool bj[2];
                if constexpr (P == MIXED) {
                    dx = sep_q2(Qi.x, Qs[u].x, Qs[u + 1].x, rp.qunit);
                    dy = sep_q2(Qi.y, Qs[u].y, Qs[u + 1].y, rp.qunit);
                    dz = sep_q2(Qi.z, Qs[u].z, Qs[u + 1].z, rp.qunit);
                    bj[0] = Qs[u].w != 0;
                    bj[1] = Qs[u + 1].w != 0;
                } else {
                    dx = sep_f2(Hi.x, make_float2(Hs[u].x, Hs[u + 1].x), rp.Lhi, rp.invLf);
                    dy = sep_f2(Hi.y, make_float2(Hs[u].y, Hs[u + 1].y), rp.Lhi, rp.invLf);
                    dz = sep_f2(Hi.z, make_float2(Hs[u].z, Hs[u + 1].z), rp.Lhi, rp.invLf);
                    bj[0] = species_of(Hs[u].w) != 0;
                    bj[1] = species_of(Hs[u + 1].w) != 0;
                }
                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                const float rca = bj[0] ? rc2[1] : rc2[0], rcb = bj[1] ? rc2[1] : rc2[0];
                // (the particle itself, r2 = 0 exactly, is never inside)
                const bool ina = r2.x > 0.0f && r2.x < rca, inb = r2.y > 0.0f && r2.y < rcb;
                const float2 sg = make_float2(bj[0] ? sig2[1] : sig2[0], bj[1] ? sig2[1] : sig2[0]);
                const float2 e48 = make_float2(ina ? (bj[0] ? eps48[1] : eps48[0]) : 0.0f,
                                               inb ? (bj[1] ? eps48[1] : eps48[0]) : 0.0f);
                const float2 ir2 = make_float2(rcp_approx(ina ? r2.x : rca), rcp_approx(inb ? r2.y : rcb));
                const float2 s2 = __fmul2_rn(sg, ir2);
                const float2 s6 = __fmul2_rn(__fmul2_rn(s2, s2), s2);
                float2 fr = __fmul2_rn(__fmul2_rn(__fmul2_rn(e48, ir2), s6),
                                       __fadd2_rn(s6, make_float2(-0.5f, -0.5f)));
                if (SM) {
                    float fs[2] = {fr.x, fr.y}, vs[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const bool in = h ? inb : ina;
                        const int ab = ti * 2 + (bj[h] ? 1 : 0);
                        const float q6 = h ? s6.y : s6.x, rr = h ? (inb ? r2.y : rcb) : (ina ? r2.x : rca);
                        vs[h] = in ? fmaf(a.tab.eps4[ab], q6 * q6 - q6, -a.tab.shift[ab]) : 0.0f;
                        smooth_pair(rr, a.tab.rc[ab], a.tab.ihs[ab], fs[h], vs[h]);
                    }
                    fr = make_float2(fs[0], fs[1]);
                    gv = fmaf(12.0f, vs[1], fmaf(12.0f, vs[0], gv));
                } else {
                    const float2 c = make_float2(bj[0] ? vc[1] : vc[0], bj[1] ? vc[1] : vc[0]);
                    const float2 t = __fadd2_rn(s6, c);
                    const float2 w = __ffma2_rn(s6, s6, make_float2(-t.x, -t.y));
                    gv = fmaf(e48.y, w.y, fmaf(e48.x, w.x, gv));
                }
                gx = fmaf(fr.y, dx.y, fmaf(fr.x, dx.x, gx));
                gy = fmaf(fr.y, dy.y, fmaf(fr.x, dy.x, gy));
                gz = fmaf(fr.y, dz.y, fmaf(fr.x, dz.x, gz));
            }
            if constexpr (P == MIXED) {
                kahan_add(sx, cx, gx);
                kahan_add(sy, cy, gy);
                kahan_add(sz, cz, gz);
                kahan_add(se, ce, gv);
            } else {
                sx += gx;
                sy += gy;
                sz += gz;
                se += gv;
            }
        }
        if constexpr (P == MIXED) {
            ds ax = ds_from(sx, -cx), ay = ds_from(sy, -cy), az = ds_from(sz, -cz), ae = ds_from(se, -ce);
#pragma unroll
            for (int o = TPP / 2; o > 0; o >>= 1) {
                ds bx = ds_from(__shfl_xor_sync(0xffffffffu, ax.hi, o), __shfl_xor_sync(0xffffffffu, ax.lo, o));
                ds by = ds_from(__shfl_xor_sync(0xffffffffu, ay.hi, o), __shfl_xor_sync(0xffffffffu, ay.lo, o));
                ds bz = ds_from(__shfl_xor_sync(0xffffffffu, az.hi, o), __shfl_xor_sync(0xffffffffu, az.lo, o));
                ds be = ds_from(__shfl_xor_sync(0xffffffffu, ae.hi, o), __shfl_xor_sync(0xffffffffu, ae.lo, o));
                ax = ds_add(ax, bx);
                ay = ds_add(ay, by);
                az = ds_add(az, bz);
                ae = ds_add(ae, be);
            }
            fx = __fadd_rn(ax.hi, ax.lo);
            fy = __fadd_rn(ay.hi, ay.lo);
            fz = __fadd_rn(az.hi, az.lo);
            ep = ds_mul(ae, ds_from(kE24hi, kE24lo));         // half of the sum of V = (12 V) / 24
        } else {
#pragma unroll
            for (int o = TPP / 2; o > 0; o >>= 1) {
                sx += __shfl_xor_sync(0xffffffffu, sx, o);
                sy += __shfl_xor_sync(0xffffffffu, sy, o);
                sz += __shfl_xor_sync(0xffffffffu, sz, o);
                se += __shfl_xor_sync(0xffffffffu, se, o);
            }
            fx = sx; fy = sy; fz = sz;
            ep = ds_from(se * (1.0f / 24.0f), 0.f);
        }
    }
}

// Virial and virial tensor of particle ii (half of each pair, the less
// frequent reductions of Sec. 2.2), as a separate pass over the list on sample
// steps so that the every-step loop carries no virial accumulators.
// acc[1..7] = W, W_xx, W_yy, W_zz, W_xy, W_xz, W_yz; acc[0] is left as it is.
template <int P, int TPP, bool SM>
__device__ __forceinline__ void pair_virial(const KArgs &a, const Rep &rp, int pp, int ii, int nn, double *acc)
{
    const int lane = threadIdx.x & (TPP - 1);
    const int *lst = a.nbr + (size_t)ii * (size_t)a.Kstride;
    FT<P> d7[7] = {0, 0, 0, 0, 0, 0, 0};
    if constexpr (P == FP64) {
        const d4 *pos = (const d4 *)pos_a(a, pp);
        const d4 xi = pos[ii];
        const int ti = species_of(xi.w);
        for (int k = lane; k < nn; k += TPP) {
            const d4 xj = pos[checked(a, lst[k], a.n, ii)];
            const int ab = ti * 2 + species_of(xj.w);
            const double dx = sep_d(xi.x, xj.x, rp.L, rp.invL);
            const double dy = sep_d(xi.y, xj.y, rp.L, rp.invL);
            const double dz = sep_d(xi.z, xj.z, rp.L, rp.invL);
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (r2 < a.tab.rc2d[ab] && r2 > 0.0) {
                const double ir2 = 1.0 / r2;
                const double s2 = a.tab.sig2d[ab] * ir2;
                const double s6 = s2 * s2 * s2;
                double fr = a.tab.eps48d[ab] * ir2 * s6 * (s6 - 0.5);
                if (SM) {
                    double v = a.tab.eps4d[ab] * s6 * (s6 - 1.0) - a.tab.shiftd[ab];
                    smooth_pair(r2, a.tab.rcd[ab], a.tab.ihsd[ab], fr, v);
                }
                d7[0] += fr * r2;
                d7[1] += fr * dx * dx; d7[2] += fr * dy * dy; d7[3] += fr * dz * dz;
                d7[4] += fr * dx * dy; d7[5] += fr * dx * dz; d7[6] += fr * dy * dz;
            }
        }
    } else {
        const int4 *qp = q_of(a, pp);
        const float4 *pos = (const float4 *)pos_a(a, pp);
        int4 Qi = make_int4(0, 0, 0, 0);
        float4 Hi = make_float4(0.f, 0.f, 0.f, 0.f);
        int ti;
        if constexpr (P == MIXED) {
            Qi = qp[ii];
            ti = Qi.w;
        } else {
            Hi = pos[ii];
            ti = species_of(Hi.w);
        }
        // groups of 4 entries, their gathers in flight together (rows are padded with the
        // particle itself, r2 = 0, to whole groups)
        for (int k0 = 4 * lane; k0 < nn; k0 += 4 * TPP) {
            const int4 j4 = *(const int4 *)(lst + k0);
            const int jj[4] = {j4.x, j4.y, j4.z, j4.w};
            int4 Qs[4];
            float4 Hs[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = checked(a, jj[u], a.n, ii);
                if constexpr (P == MIXED)
                    Qs[u] = qp[j];
                else
                    Hs[u] = pos[j];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float dx, dy, dz;
                int ab;
                if constexpr (P == MIXED) {
                    ab = ti * 2 + Qs[u].w;
                    dx = sep_q(Qi.x, Qs[u].x, rp.qunit);
                    dy = sep_q(Qi.y, Qs[u].y, rp.qunit);
                    dz = sep_q(Qi.z, Qs[u].z, rp.qunit);
                } else {
                    ab = ti * 2 + species_of(Hs[u].w);
                    dx = sep_f(Hi.x, Hs[u].x, rp.Lhi, rp.invLf);
                    dy = sep_f(Hi.y, Hs[u].y, rp.Lhi, rp.invLf);
                    dz = sep_f(Hi.z, Hs[u].z, rp.Lhi, rp.invLf);
                }
                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                if (r2 < a.tab.rc2[ab] && r2 > 0.0f) {
                    const float ir2 = __fdividef(1.0f, r2);
                    const float s2 = a.tab.sig2[ab] * ir2;
                    const float s6 = s2 * s2 * s2;
                    float fr = a.tab.eps48[ab] * ir2 * s6 * (s6 - 0.5f);
                    if (SM) {
                        float v = a.tab.eps4[ab] * s6 * (s6 - 1.0f) - a.tab.shift[ab];
                        smooth_pair(r2, a.tab.rc[ab], a.tab.ihs[ab], fr, v);
                    }
                    d7[0] += fr * r2;
                    d7[1] += fr * dx * dx; d7[2] += fr * dy * dy; d7[3] += fr * dz * dz;
                    d7[4] += fr * dx * dy; d7[5] += fr * dx * dz; d7[6] += fr * dy * dz;
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        double v = (double)d7[k];
#pragma unroll
        for (int o = TPP / 2; o > 0; o >>= 1)
            v += __shfl_xor_sync(0xffffffffu, v, o);
        acc[1 + k] = 0.5 * v;
    }
}

template <int P, typename E>
__device__ __forceinline__ void store_force(const KArgs &a, int i, FT<P> fx, FT<P> fy, FT<P> fz, E e)
{
    if constexpr (P == FP64) {
        d4 f;
        f.x = fx; f.y = fy; f.z = fz; f.w = e_value(e);
        ((d4 *)a.force)[i] = f;
    } else {
        ((float4 *)a.force)[i] = make_float4(fx, fy, fz, e_float(e));
    }
}

// ---------------------------------------------------------------------------
// One MD step of a chunk of particles.  Positions r(t) (current buffer), forces
// f(t) from the list, then per particle: v(t) = v(t-1/2) + dt/2m f(t) [sample],
// and unless this is the last step of md_step: v(t+1/2) = v(t) + dt/2m f(t),
// r(t+1) = r(t) + dt v(t+1/2) into the other buffer.  Without `kick` the forces
// and reductions alone, the state left as it is.
// ---------------------------------------------------------------------------
// One Cartesian component of the velocity-Verlet update, done by lane c of
// the particle's group: half kick(s), drift, re-anchor / wrap, displacement
// from the build position.  vh/vl: velocity component (hi/lo for MIXED, vh
// alone otherwise); returns the squared displacement component.
template <int P>
__device__ __forceinline__ void component_update(const KArgs &a, const Rep &rp, int pp, int spar, int i, int c,
                                                 int sp, float f_c, double f_cd, bool sample, bool kick, bool last,
                                                 float &vh, float &vl, double &vd, float rr,
                                                 double &ke, double &pc, float &dd, float &vv, unsigned int &bad)
{
    const size_t e = 4 * (size_t)i + c;
    if constexpr (P == MIXED) {
        const ds hk = ds_from(a.hdtm_hi[sp], a.hdtm_lo[sp]);
        ds v = ds_from(vh, vl);
        if (kick)
            v = ds_add(v, ds_mul_f(hk, f_c));
        if (sample) {
            const double x = ds_to_double(v);
            ke = 0.5 * a.mass[sp] * x * x;
            pc = a.mass[sp] * x;
        }
        if (!last) {
            v = ds_add(v, ds_mul_f(hk, f_c));
            const ds s = ds_mul(ds_from(a.dt_hi, a.dt_lo), v);
            if (fabsf(s.hi) > 0.25f * rp.Lhi)
                bad |= ST_UNSTABLE;
            const float H = ((const float *)pos_a(a, pp))[e], l = ((const float *)pos_b(a, pp))[e];
            float Hn, ln;
            const int dimg = anchor_wrap(ds_add(ds_from(H, l), s), rp.grid, rp.inv_grid, rp.Lhi, rp.Llo, Hn, ln);
            if (!isfinite(Hn))
                bad |= ST_NONFINITE;
            ((float *)pos_a(a, pp ^ 1))[e] = Hn;
            ((float *)pos_b(a, pp ^ 1))[e] = ln;
            ((unsigned int *)q_of(a, pp ^ 1))[e] = fixq(Hn, ln, rp);
            const float dx = __fadd_rn(sep_f(Hn, rr, rp.Lhi, rp.invLf), ln);
            dd = dx * dx;
            vv = v.hi * v.hi;
            if (dimg)
                ((int *)img_of(a, spar))[e] += dimg;
        }
        vh = v.hi;
        vl = v.lo;
    } else if constexpr (P == FP64) {
        const double hk = a.hdtm[sp];            // (roundings spelled out, as in half_kick / drift)
        double v = vd;
        if (kick)
            v = fma(hk, f_cd, v);
        if (sample) {
            ke = 0.5 * a.mass[sp] * v * v;
            pc = a.mass[sp] * v;
        }
        if (!last) {
            v = fma(hk, f_cd, v);
            const double s = __dmul_rn(a.dt, v);
            if (fabs(s) > 0.25 * rp.L)
                bad |= ST_UNSTABLE;
            double x = __dadd_rn(((const double *)pos_a(a, pp))[e], s);
            int dimg = 0;
            if (x >= rp.L) { x -= rp.L; dimg = 1; } else if (x < 0.0) { x += rp.L; dimg = -1; }
            if (!isfinite(x))
                bad |= ST_NONFINITE;
            ((double *)pos_a(a, pp ^ 1))[e] = x;
            const float dx = sep_f(__double2float_rn(x), rr, rp.Lhi, rp.invLf);
            dd = dx * dx;
            vv = (float)(v * v);
            if (dimg)
                ((int *)img_of(a, spar))[e] += dimg;
        }
        vd = v;
    } else {
        const float hk = a.hdtm_hi[sp];
        float v = vh;
        if (kick)
            v = fmaf(hk, f_c, v);
        if (sample) {
            ke = 0.5 * a.mass[sp] * (double)v * (double)v;
            pc = a.mass[sp] * (double)v;
        }
        if (!last) {
            v = fmaf(hk, f_c, v);
            const float s = __fmul_rn(a.dt_hi, v);
            const float L = rp.Lhi;
            if (fabsf(s) > 0.25f * L)
                bad |= ST_UNSTABLE;
            float x = __fadd_rn(((const float *)pos_a(a, pp))[e], s);
            int dimg = 0;
            if (x >= L) { x -= L; dimg = 1; } else if (x < 0.f) { x += L; dimg = -1; }
            if (x >= L) { x = 0.f; dimg += 1; }
            if (!isfinite(x))
                bad |= ST_NONFINITE;
            ((float *)pos_a(a, pp ^ 1))[e] = x;
            const float dx = sep_f(x, rr, L, rp.invLf);
            dd = dx * dx;
            vv = v * v;
            if (dimg)
                ((int *)img_of(a, spar))[e] += dimg;
        }
        vh = v;
    }
}

// Step body from 4 lanes per particle on: after the pair loop its lanes share the
// update.  Lanes c = 0..2 do one Cartesian component each of the double-single
// kick-drift-kick, lane 3 carries the species word to the new position buffer.
// The operands of the update are loaded before the neighbour loop so that their
// latency is hidden.
template <int P, int TPP, bool SAMPLE, bool SM>
__device__ __forceinline__ void step_body_split(const KArgs &a, const Rep &rep, PairQueue *Q, const int4 b, bool kick, bool last,
                                                int pp, int spar, double *part, ET<P> &eo, float &d2, float &v2, float &a2,
                                                unsigned int &bad)
{
    const Rep rp = rep;
    const int lane = threadIdx.x & (TPP - 1);
    const int i = b.x + Grp::tid() / TPP;
    const bool valid = i < b.y;
    const int ii = valid ? i : b.x;
    const int nn = valid ? a.nnbr[ii] : 0;
    float vh = 0.f, vl = 0.f, rr = 0.f;
    double vd = 0.0;
    if (valid && lane < 3) {
        const size_t e = 4 * (size_t)ii + lane;
        if constexpr (P == FP64) {
            vd = ((const double *)vel_a(a, spar))[e];
        } else {
            vh = ((const float *)vel_a(a, spar))[e];
            if constexpr (P == MIXED)
                vl = ((const float *)vel_b(a, spar))[e];
        }
        rr = ((const float *)a.rref)[e];
    }
    FT<P> fx = 0, fy = 0, fz = 0;
    ET<P> ep = e_zero<P>();
#pragma unroll
    for (int k = 0; k < kPartF; ++k)
        part[k] = 0.0;
    eo = e_zero<P>();
    pair_forces<P, TPP, SM>(a, rp, pp, ii, nn, Q, fx, fy, fz, ep);
    if (SAMPLE)
        pair_virial<P, TPP, SM>(a, rp, pp, ii, nn, part);
    // Every lane of the warp must reach the shuffles below, including the
    // lanes of padding particles past the end of a replica's range: they skip
    // the update and contribute zeros.
    int sp = 0;
    if (valid) {
        if constexpr (P == FP64)
            sp = species_of(((const double *)pos_a(a, pp))[4 * (size_t)i + 3]);
        else
            sp = species_of(((const float *)pos_a(a, pp))[4 * (size_t)i + 3]);
    }
    if (valid && lane == 0)
        store_force<P>(a, i, fx, fy, fz, ep);
    double ke = 0.0, p3[3] = {0.0, 0.0, 0.0};
    float dd = 0.f, vv = 0.f;
    if (!valid) {
        // no update
    } else if (lane < 3) {
        const size_t e = 4 * (size_t)i + lane;
        const FT<P> f_c = lane == 0 ? fx : (lane == 1 ? fy : fz);
        double pc = 0.0;
        component_update<P>(a, rp, pp, spar, i, lane, sp, (float)f_c, (double)f_c, SAMPLE, kick, last, vh, vl, vd, rr, ke, pc,
                            dd, vv, bad);
        p3[0] = lane == 0 ? pc : 0.0;
        p3[1] = lane == 1 ? pc : 0.0;
        p3[2] = lane == 2 ? pc : 0.0;
        if constexpr (P == FP64) {
            ((double *)vel_a(a, spar))[e] = vd;
        } else {
            ((float *)vel_a(a, spar))[e] = vh;
            if constexpr (P == MIXED)
                ((float *)vel_b(a, spar))[e] = vl;
        }
    } else if (lane == 3 && !last) {
        // the species word travels with the position
        if constexpr (P == FP64)
            ((double *)pos_a(a, pp ^ 1))[4 * (size_t)i + 3] = ((const double *)pos_a(a, pp))[4 * (size_t)i + 3];
        else
            ((float *)pos_a(a, pp ^ 1))[4 * (size_t)i + 3] = ((const float *)pos_a(a, pp))[4 * (size_t)i + 3];
        if constexpr (P == MIXED)
            ((int *)q_of(a, pp ^ 1))[4 * (size_t)i + 3] = sp;
    }
    // combine the component lanes (the first 4 of the particle)
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
        dd += __shfl_xor_sync(0xffffffffu, dd, o);
        vv += __shfl_xor_sync(0xffffffffu, vv, o);
        if (SAMPLE) {
            ke += __shfl_xor_sync(0xffffffffu, ke, o);
            p3[0] += __shfl_xor_sync(0xffffffffu, p3[0], o);
            p3[1] += __shfl_xor_sync(0xffffffffu, p3[1], o);
            p3[2] += __shfl_xor_sync(0xffffffffu, p3[2], o);
        }
    }
    if (!valid || lane != 0) {
#pragma unroll
        for (int k = 0; k < kPartF; ++k)
            part[k] = 0.0;
        return;
    }
    eo = ep;
    if (SAMPLE) {
        part[8] = ke;
        part[9] = p3[0];
        part[10] = p3[1];
        part[11] = p3[2];
    }
    if (!last) {
        d2 = dd;
        v2 = vv;
        const float im = a.inv_mass[sp];
        a2 = __fmul_rn(__fmul_rn(norm2(fx, fy, fz), im), im);
    }
}

template <int P, int TPP, bool SAMPLE, bool SM>
__device__ __forceinline__ void step_body(const KArgs &a, const Rep &rep, PairQueue *Q, const int4 b, bool kick, bool last, bool track,
                                          int pp, int spar, double *part, ET<P> &eo, float &d2, float &v2, float &a2,
                                          unsigned int &bad)
{
    if constexpr (TPP >= 4) {                        // (below 4 lanes one lane updates: measured faster)
        step_body_split<P, TPP, SAMPLE, SM>(a, rep, Q, b, kick, last, pp, spar, part, eo, d2, v2, a2, bad);
        return;
    }
    const Rep rp = rep;
    const int lane = threadIdx.x & (TPP - 1);
    const int i = b.x + Grp::tid() / TPP;
    const bool valid = i < b.y;
    const int ii = valid ? i : b.x;
    const int nn = valid ? a.nnbr[ii] : 0;
    FT<P> fx = 0, fy = 0, fz = 0;
    ET<P> ep = e_zero<P>();
#pragma unroll
    for (int k = 0; k < kPartF; ++k)
        part[k] = 0.0;
    eo = e_zero<P>();
    pair_forces<P, TPP, SM>(a, rp, pp, ii, nn, Q, fx, fy, fz, ep);
    if (SAMPLE)
        pair_virial<P, TPP, SM>(a, rp, pp, ii, nn, part);
    if (!(valid && lane == 0)) {
#pragma unroll
        for (int k = 0; k < kPartF; ++k)
            part[k] = 0.0;
        return;
    }
    eo = ep;
    store_force<P>(a, i, fx, fy, fz, ep);
    PState<P> s;
    load_pos<P>(a, pp, i, s);
    load_vel<P>(a, spar, i, s);
    if (kick)
        half_kick<P>(a, s, fx, fy, fz);             // completes v(t)
    if (SAMPLE)
        kinetic<P>(a, s, part + 8);
    if (!last) {
        half_kick<P>(a, s, fx, fy, fz);             // v(t + 1/2)
        d2 = drift<P>(a, rp, s, pp ^ 1, spar, i, track, bad);
        v2 = speed2(s);
        const float im = a.inv_mass[s.sp];
        a2 = __fmul_rn(__fmul_rn(norm2(fx, fy, fz), im), im);
    }
    store_vel<P>(a, spar, i, s);
}

// ---------------------------------------------------------------------------
// Cell binning by counting sort (Sec. 2.2: integer cell index per particle,
// particles sorted by cell, start index of each cell) with the cells ordered
// along a space-filling curve (the periodic reorder of Sec. 2.2).  Phases of a
// rebuild, each ending at a grid barrier of the run kernel: bin (cell key,
// histogram) -> scan (cell starts) -> scatter -> permute (deterministic order
// inside a cell; gather of the state into the other buffers) -> neighbour build
// (lists from the permuted positions).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int cell_coord(double x, double cscale, int nc)
{
    int c = (int)floor(x * cscale);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

__device__ __forceinline__ int cell_coord_f(float x, float cscale, int nc)
{
    int c = (int)floorf(x * cscale);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

// Octant of a coordinate inside its cell (0 or 1 per axis); the three
// interleave into the particle's sub-cell code along a Morton curve, the order
// of the particles inside a cell after each rebuild, so that the particles a
// warp holds are close in space (their neighbours overlap).  (A 4 x 4 x 4
// grid measured 0.25 % slower per MD step.)
__device__ __forceinline__ unsigned int sub2(double x, double cscale, int c)
{
    const int s = (int)floor((x * cscale - (double)c) * 2.0);
    return (unsigned int)(s < 0 ? 0 : (s > 1 ? 1 : s));
}

__device__ __forceinline__ unsigned int sub2f(float x, float cscale, int c)
{
    const int s = (int)floorf((x * cscale - (float)c) * 2.0f);
    return (unsigned int)(s < 0 ? 0 : (s > 1 ? 1 : s));
}

__device__ __forceinline__ int morton6(unsigned int x, unsigned int y, unsigned int z)
{
    return (int)((x & 1u) | ((y & 1u) << 1) | ((z & 1u) << 2) | ((x & 2u) << 2) | ((y & 2u) << 3) |
                 ((z & 2u) << 4));
}

// Cell key and sub-cell code of particle i from the positions in buffer pp.
template <int P>
__device__ __forceinline__ int cell_of(const KArgs &a, const Rep &rp, int pp, int i, int &sub)
{
    int cx, cy, cz;
    if constexpr (P == FP64) {
        const d4 x = ((const d4 *)pos_a(a, pp))[i];
        cx = cell_coord(x.x, rp.cscale, rp.nc);
        cy = cell_coord(x.y, rp.cscale, rp.nc);
        cz = cell_coord(x.z, rp.cscale, rp.nc);
        sub = morton6(sub2(x.x, rp.cscale, cx), sub2(x.y, rp.cscale, cy), sub2(x.z, rp.cscale, cz));
    } else {
        const float4 x = ((const float4 *)pos_a(a, pp))[i];
        cx = cell_coord_f(x.x, rp.cscalef, rp.nc);
        cy = cell_coord_f(x.y, rp.cscalef, rp.nc);
        cz = cell_coord_f(x.z, rp.cscalef, rp.nc);
        sub = morton6(sub2f(x.x, rp.cscalef, cx), sub2f(x.y, rp.cscalef, cy), sub2f(x.z, rp.cscalef, cz));
    }
    return checked(a, a.crank[rp.cell0 + (cz * rp.nc + cy) * rp.nc + cx], a.ncell, 0);
}

// Phase 1: cell keys and histogram.
template <int P>
__device__ __forceinline__ void rebuild_bin(const KArgs &a, const Grp &g, int pp)
{
    for (int row = g.vb; row < a.nblk_i; row += g.nvb) {
        const int4 b = a.blk_i[row];
        const Rep &rp = a.rep[b.z];
        for (int i = b.x + g.tid(); i < b.y; i += kForceBlock) {
            int sub;
            const int key = cell_of<P>(a, rp, pp, i, sub);
            a.key[i] = make_int2(key, sub);
            atomicAdd(&a.ccount[key], 1);
        }
    }
}

// Exclusive prefix sum of one value per thread over the group; `total` gets the
// sum.  sh: one int per warp.
__device__ __forceinline__ int grp_scan(const Grp &g, int v, int &total, int *sh)
{
    const int lane = threadIdx.x & 31, w = g.tid() >> 5, nw = kGrpWarps;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += y;
    }
    if (lane == 31)
        sh[w] = incl;
    g.sync();
    int before = 0, sum = 0;
    for (int k = 0; k < nw; ++k) {
        before += k < w ? sh[k] : 0;
        sum += sh[k];
    }
    g.sync();
    total = sum;
    return before + incl - v;
}

// Phase 2: first particle of every cell.  Each group scans a slice of
// slice_cells consecutive cells, after the particles of the cells before it,
// added up from the counts themselves, or beyond kScanDirect cells from the
// slices' sums (a barrier more); the counts are
// cleared for the next binning in the phase after.
constexpr int kScanDirect = 8192;

__device__ __forceinline__ void rebuild_slices(const KArgs &a, const Grp &g, int slice_cells, int *sh)
{
    const int c0 = g.vb * slice_cells, c1 = min(c0 + slice_cells, a.ncell);
    int v = 0, sum;
    for (int c = c0 + g.tid(); c < c1; c += kForceBlock)
        v += a.ccount[c];
    grp_scan(g, v, sum, sh);
    if (g.tid() == 0)
        a.slice[g.vb] = sum;
}

__device__ __forceinline__ void rebuild_scan(const KArgs &a, const Grp &g, int slice_cells, int *sh)
{
    const int c0 = g.vb * slice_cells, c1 = min(c0 + slice_cells, a.ncell);
    if (c0 >= a.ncell)
        return;
    int before = 0, carry;
    const int *from = a.ncell > kScanDirect ? a.slice : a.ccount;
    const int upto = a.ncell > kScanDirect ? g.vb : c0;
#pragma unroll 8
    for (int b = g.tid(); b < upto; b += kForceBlock)
        before += from[b];
    grp_scan(g, before, carry, sh);
    for (int base = c0; base < c1; base += kForceBlock) {
        const int c = base + g.tid();
        const int v = c < c1 ? a.ccount[c] : 0;
        int sum;
        const int at = carry + grp_scan(g, v, sum, sh);
        if (c < c1) {
            a.cstart[c] = at;
            a.ccursor[c] = 0;
        }
        carry += sum;
    }
    if (g.tid() == 0 && c1 == a.ncell)
        a.cstart[a.ncell] = carry;
}

// Phase 3: particles into their cells, in any order.
__device__ __forceinline__ void rebuild_scatter(const KArgs &a, const Grp &g)
{
    for (int i = g.vb * kForceBlock + g.tid(); i < a.n; i += g.nvb * kForceBlock) {
        const int2 key = a.key[i];
        const int k = checked(a, key.x, a.ncell, 0);
        const int slot = checked(a, a.cstart[k] + atomicAdd(&a.ccursor[k], 1), a.n, 0);
        a.tmpidx[slot] = make_int2(i, key.y);
    }
    for (int c = g.vb * kForceBlock + g.tid(); c < a.ncell; c += g.nvb * kForceBlock)
        a.ccount[c] = 0;                                 // ready for the next binning
}

// Phase 4: final slot of each particle: its cell's start plus the number of
// particles of the same cell that come before it in (sub-cell code, current
// index) order (deterministic), then gather of the whole state into the other
// buffers.
template <int P>
__device__ __forceinline__ void rebuild_permute(const KArgs &a, const Grp &g, int pp, int spar)
{
    for (int s = g.vb * kForceBlock + g.tid(); s < a.n; s += g.nvb * kForceBlock) {
        const int2 me = a.tmpidx[s];
        const int i = checked(a, me.x, a.n, 0);
        const int k = checked(a, a.key[i].x, a.ncell, 0);
        const int b0 = a.cstart[k], b1 = a.cstart[k + 1];
        int rank = 0;
#pragma unroll 8
        for (int t = b0; t < b1; ++t) {
            const int2 other = a.tmpidx[t];
            rank += (other.y < me.y || (other.y == me.y && other.x < i)) ? 1 : 0;
        }
        const int d = checked(a, b0 + rank, a.n, 0);
        if constexpr (P == FP64) {
            const d4 x = ((const d4 *)pos_a(a, pp))[i];
            ((d4 *)pos_a(a, pp ^ 1))[d] = x;
            ((d4 *)vel_a(a, spar ^ 1))[d] = ((const d4 *)vel_a(a, spar))[i];
            a.rref[d] = make_float4(__double2float_rn(x.x), __double2float_rn(x.y), __double2float_rn(x.z), 0.f);
        } else {
            const float4 x = ((const float4 *)pos_a(a, pp))[i];
            ((float4 *)pos_a(a, pp ^ 1))[d] = x;
            ((float4 *)vel_a(a, spar ^ 1))[d] = ((const float4 *)vel_a(a, spar))[i];
            if constexpr (P == MIXED) {
                ((float4 *)pos_b(a, pp ^ 1))[d] = ((const float4 *)pos_b(a, pp))[i];
                q_of(a, pp ^ 1)[d] = q_of(a, pp)[i];
                ((float4 *)vel_b(a, spar ^ 1))[d] = ((const float4 *)vel_b(a, spar))[i];
            }
            a.rref[d] = make_float4(x.x, x.y, x.z, 0.f);
        }
        img_of(a, spar ^ 1)[d] = img_of(a, spar)[i];
    }
}

// ---------------------------------------------------------------------------
// Neighbour-list build (Sec. 2.2), one group of threads per cell (or several, each
// taking a share of the cell's particles, where cells are few).  The group
// stages the particles of the 27 surrounding cells (all cells of the replica
// when fewer than three fit along its edge) in shared memory, in a fixed order
// (stencil order, then slot order inside a cell), as single-precision
// coordinates relative to the cell's centre, dropping those farther than the
// largest list radius from the cell's own box.  Each warp then takes its
// particles two at a time, its lanes the candidates, two per lane and
// iteration: the distance test of two candidates is six packed instructions,
// and one ballot per 32 candidates places the entries kept in the row, in
// candidate order, with stores that run along the row.  Rows are particle-major,
// nbr[i*Kstride + k], and hold every partner closer than r_c,ab + skin (plus a
// rounding margin: the list only has to contain every pair within r_c + skin,
// and the margin covers the rounding).  Reads the permuted positions (other
// buffer).  More candidates or own particles than fit are processed in rounds.
//
// Measured against a warp per cell with the particles as lanes (every lane
// testing the same candidate, a scattered store per entry kept): the test loop
// takes half the instructions per particle, and the stores are coalesced.
// ---------------------------------------------------------------------------
constexpr int kNbCap = 896;      // staged candidates per round (a multiple of 64)
constexpr int kNbGrp = 7;        // groups of up to 32 candidates a warp stages at once
constexpr int kNbOwn = 256;      // own-cell particles per batch
constexpr int kNbPass = 2;       // own-cell particles tested per warp pass over the candidates
constexpr int kNbChunks = 256;   // groups of up to 32 particles of one stencil cell per round of staging

struct NbBlock {
    float2 x[kNbCap / 2], y[kNbCap / 2], z[kNbCap / 2];   // candidates c, c + 32 side by side
    int2 w[kNbCap / 2];                                   // index | species << 31
    int cnt[kNbOwn];
    int c0[kNbChunks], c1[kNbChunks];
    int nchunk, max_nbr;
    int wsum[kForceBlock / 32];
};

// Word of particle j for the build: coordinates relative to `ctr` (nearest
// image) and index with the species in the sign bit.  The rounding is that of the
// small difference: MIXED and FP64 subtract on the fixed-point circle, to which
// one FP64 instruction takes a coordinate (as the conversion to single precision
// would; subtracting in double cost 1.3 % of a step at KA N=16384).  FP32 rounds once
// more where it shifts by the box, by half an ulp of L for each of a pair: 8.9e-5 at
// L = 1500, within the list margin (an exact shift cost 1 to 2 % of a step).
struct NbCentre { float x, y, z; unsigned int qx, qy, qz; double qscale; };

// x / L in units of 2^-32 modulo 2^32, to the nearest, for |x| <= 2^18 L
__device__ __forceinline__ unsigned int circle_d(double x, double qscale)
{
    return (unsigned int)__double2loint(fma(x, qscale, 6755399441055744.0));   // 1.5 2^52
}

template <int P>
__device__ __forceinline__ NbCentre nb_centre(const Rep &rp, const int4 &cc)
{
    NbCentre c;
    const float edge = rp.Lhi / (float)rp.nc;
    c.x = ((float)cc.x + 0.5f) * edge;
    c.y = ((float)cc.y + 0.5f) * edge;
    c.z = ((float)cc.z + 0.5f) * edge;
    c.qscale = rp.invL * 4294967296.0;
    // the same on the fixed-point circle
    c.qx = (unsigned int)((((unsigned long long)(2 * cc.x + 1)) << 31) / (unsigned int)rp.nc);
    c.qy = (unsigned int)((((unsigned long long)(2 * cc.y + 1)) << 31) / (unsigned int)rp.nc);
    c.qz = (unsigned int)((((unsigned long long)(2 * cc.z + 1)) << 31) / (unsigned int)rp.nc);
    return c;
}

template <int P>
__device__ __forceinline__ float3 nb_rel(const KArgs &a, const Rep &rp, const NbCentre &c, int pn, int j, int &sp)
{
    if constexpr (P == MIXED) {
        const int4 q = q_of(a, pn)[j];
        sp = q.w;
        return make_float3(sep_q((unsigned int)q.x, c.qx, rp.qunit), sep_q((unsigned int)q.y, c.qy, rp.qunit),
                           sep_q((unsigned int)q.z, c.qz, rp.qunit));
    } else if constexpr (P == FP64) {
        const d4 x = ((const d4 *)pos_a(a, pn))[j];
        sp = species_of(x.w);
        return make_float3(sep_q(circle_d(x.x, c.qscale), c.qx, rp.qunit), sep_q(circle_d(x.y, c.qscale), c.qy, rp.qunit),
                           sep_q(circle_d(x.z, c.qscale), c.qz, rp.qunit));
    } else {
        const float4 x = ((const float4 *)pos_a(a, pn))[j];
        sp = species_of(x.w);
        return make_float3(sep_f(x.x, c.x, rp.Lhi, rp.invLf), sep_f(x.y, c.y, rp.Lhi, rp.invLf),
                           sep_f(x.z, c.z, rp.Lhi, rp.invLf));
    }
}

// Particle range of the lane's stencil cell (lanes beyond the stencil: empty).
__device__ __forceinline__ void nb_stencil(const KArgs &a, const Rep &rp, const int4 &cc, int nst, int &s0, int &s1)
{
    const int lane = threadIdx.x & 31, nc = rp.nc;
    s0 = s1 = 0;
    if (lane < nst) {
        int x = cc.x, y = cc.y, z = cc.z;
        if (nst == 27) {
            x += lane % 3 - 1;
            y += (lane / 3) % 3 - 1;
            z += lane / 9 - 1;
            x += x < 0 ? nc : (x >= nc ? -nc : 0);
            y += y < 0 ? nc : (y >= nc ? -nc : 0);
            z += z < 0 ? nc : (z >= nc ? -nc : 0);
        }
        const int k = a.crank[rp.cell0 + (z * nc + y) * nc + x];
        s0 = a.cstart[k];
        s1 = a.cstart[k + 1];
    }
}

// Test of the staged candidates against the batch's particles.  WRAP: fewer
// than three cells along the edge, where the nearest image relative to the
// centre need not be the nearest image relative to a particle (from three cells
// on, a pair within the list radius lies less than half a box from the centre).
template <int P, bool WRAP>
__device__ __forceinline__ void nbuild_scan(const KArgs &a, const Grp &g, const Rep &rp, const NbCentre &ctr, int pn, int ob, int nown,
                                            int staged, int K, NbBlock &S)
{
    constexpr int NW = kForceBlock / 32;
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    for (int o0 = (g.tid() >> 5) * kNbPass; o0 < nown; o0 += NW * kNbPass) {
        float2 hx[kNbPass], hy[kNbPass], hz[kNbPass];
        float rl0[kNbPass], rl1[kNbPass];
        int cnt[kNbPass], wi[kNbPass];
        int *row[kNbPass];
#pragma unroll
        for (int p = 0; p < kNbPass; ++p) {
            const bool ok = o0 + p < nown;
            const int i = ob + (ok ? o0 + p : o0);
            int sp;
            const float3 r = nb_rel<P>(a, rp, ctr, pn, i, sp);
            hx[p] = make_float2(-r.x, -r.x);
            hy[p] = make_float2(-r.y, -r.y);
            hz[p] = make_float2(-r.z, -r.z);
            rl0[p] = ok ? a.tab.rl2[sp * 2] : -1.0f;              // -1: nothing passes
            rl1[p] = ok ? a.tab.rl2[sp * 2 + 1] : -1.0f;
            cnt[p] = S.cnt[ok ? o0 + p : o0];
            wi[p] = i | (sp << 31);
            row[p] = a.nbr + (size_t)i * (size_t)a.Kstride;
        }
        for (int s = lane; s < staged / 2; s += 32) {             // (staged is a multiple of 64 here)
            const float2 X = S.x[s], Y = S.y[s], Z = S.z[s];
            const int2 W = S.w[s];
#pragma unroll
            for (int p = 0; p < kNbPass; ++p) {
                float2 dx = __fadd2_rn(X, hx[p]), dy = __fadd2_rn(Y, hy[p]), dz = __fadd2_rn(Z, hz[p]);
                if (WRAP) {
                    dx.x = fmaf(-rintf(dx.x * rp.invLf), rp.Lhi, dx.x);
                    dx.y = fmaf(-rintf(dx.y * rp.invLf), rp.Lhi, dx.y);
                    dy.x = fmaf(-rintf(dy.x * rp.invLf), rp.Lhi, dy.x);
                    dy.y = fmaf(-rintf(dy.y * rp.invLf), rp.Lhi, dy.y);
                    dz.x = fmaf(-rintf(dz.x * rp.invLf), rp.Lhi, dz.x);
                    dz.y = fmaf(-rintf(dz.y * rp.invLf), rp.Lhi, dz.y);
                }
                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                const bool in0 = r2.x < (W.x < 0 ? rl1[p] : rl0[p]) && W.x != wi[p];
                const bool in1 = r2.y < (W.y < 0 ? rl1[p] : rl0[p]) && W.y != wi[p];
                const unsigned m0 = __ballot_sync(0xffffffffu, in0), m1 = __ballot_sync(0xffffffffu, in1);
                const int at0 = cnt[p] + __popc(m0 & lt_mask);
                const int at1 = cnt[p] + __popc(m0) + __popc(m1 & lt_mask);
                if (in0 && at0 < K)
                    row[p][at0] = W.x & 0x7fffffff;
                if (in1 && at1 < K)
                    row[p][at1] = W.y & 0x7fffffff;
                cnt[p] += __popc(m0) + __popc(m1);
            }
        }
        if (lane == 0)
#pragma unroll
            for (int p = 0; p < kNbPass; ++p)
                if (o0 + p < nown)
                    S.cnt[o0 + p] = cnt[p];
    }
}

// Lists of the share [part, part + 1) / nparts of the particles of cell c, from
// the positions in buffer pn (the permuted copy being built): row i holds at
// most K entries (the capacity in use).  The longest full count is recorded in
// max_nbr; entries beyond K are dropped (K then grows and the build is redone).
template <int P>
__device__ __forceinline__ void nbuild_cell(const KArgs &a, const Grp &g, int pn, int c, int part, int nparts, int K, NbBlock &S)
{
    const int tid = g.tid(), lane = tid & 31, warp = tid >> 5;
    constexpr int NW = kForceBlock / 32;
    const int4 cc = a.cxyz[c];
    const int first = a.cstart[c], ncell = a.cstart[c + 1] - first;
    const int lo = first + (int)((long long)ncell * part / nparts);
    const int hi = first + (int)((long long)ncell * (part + 1) / nparts);
    if (lo == hi)
        return;
    const Rep rp = a.rep[cc.w];
    const int nc = rp.nc;
    const int nst = nc >= 3 ? 27 : 1;
    const NbCentre ctr = nb_centre<P>(rp, cc);
    const float hx = 0.5f * rp.Lhi / (float)nc + 1e-3f;           // half edge of the cell's box
    const float rlmax2 = fmaxf(fmaxf(a.tab.rl2[0], a.tab.rl2[1]), fmaxf(a.tab.rl2[2], a.tab.rl2[3]));
    const unsigned lt_mask = (1u << lane) - 1u;

    int s0, s1;
    nb_stencil(a, rp, cc, nst, s0, s1);

    for (int ob = lo; ob < hi; ob += kNbOwn) {
        const int nown = min(kNbOwn, hi - ob);
        for (int t = tid; t < nown; t += kForceBlock)
            S.cnt[t] = 0;
        if (tid == 0)
            S.max_nbr = 0;
        int staged = 0;
        // groups of up to 32 particles of one stencil cell, in stencil order; the table
        // holds kNbChunks of them at a time (a cell of more than 32 kNbChunks / 27
        // particles is taken in several rounds)
        int at = s0;                                              // next particle of the lane's cell
        bool more = true;
        while (more) {
            const int want = min((s1 - at + 31) / 32, kNbChunks / 32);
            // in order: a lane's cell is complete before a later one's begins
            const unsigned left = __ballot_sync(0xffffffffu, (s1 - at + 31) / 32 > want);
            const int stop = left ? __ffs(left) - 1 : 31;         // lanes up to this one take part
            const int mine = lane <= stop ? want : 0;
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o)
                    incl += y;
            }
            const int nchunk = __shfl_sync(0xffffffffu, incl, 31);
            if (warp == 0)
                for (int k = 0; k < mine; ++k) {
                    S.c0[incl - mine + k] = at + 32 * k;
                    S.c1[incl - mine + k] = min(at + 32 * k + 32, s1);
                }
            at += 32 * mine;
            at = min(at, s1);
            more = left != 0u;
            g.sync();
            // the block's warps take kNbGrp consecutive groups each, all loads in flight, and
            // write what they keep behind what the warps before them keep
            for (int m0 = 0; m0 < nchunk; m0 += NW * kNbGrp) {
                float3 r[kNbGrp];
                int wj[kNbGrp];
                unsigned keep[kNbGrp];
                int n = 0;
#pragma unroll
                for (int u = 0; u < kNbGrp; ++u) {
                    const int m = m0 + warp * kNbGrp + u;
                    bool ok = false;
                    wj[u] = 0;
                    if (m < nchunk) {
                        const int j = S.c0[m] + lane;
                        if (j < S.c1[m]) {
                            int sp;
                            r[u] = nb_rel<P>(a, rp, ctr, pn, checked(a, j, a.n, 0), sp);
                            wj[u] = j | (sp << 31);
                            ok = true;
                        }
                    }
                    if (!ok)
                        r[u] = make_float3(1e9f, 0.f, 0.f);       // (never kept)
                }
#pragma unroll
                for (int u = 0; u < kNbGrp; ++u) {
                    bool ok = r[u].x < 1e8f;
                    if (nst == 27) {
                        const float gx = fmaxf(fabsf(r[u].x) - hx, 0.f), gy = fmaxf(fabsf(r[u].y) - hx, 0.f),
                                    gz = fmaxf(fabsf(r[u].z) - hx, 0.f);
                        ok = fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < rlmax2;
                    }
                    keep[u] = __ballot_sync(0xffffffffu, ok);
                    n += __popc(keep[u]);
                }
                if (lane == 0)
                    S.wsum[warp] = n;
                g.sync();
                int off = staged, add = 0;
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    off += w < warp ? S.wsum[w] : 0;
                    add += S.wsum[w];
                }
#pragma unroll
                for (int u = 0; u < kNbGrp; ++u) {
                    if (keep[u] >> lane & 1u) {
                        const int s = off + __popc(keep[u] & lt_mask);
                        const int t = (s >> 6) * 32 + (s & 31), h = (s >> 5) & 1;
                        (&S.x[t].x)[h] = r[u].x;
                        (&S.y[t].x)[h] = r[u].y;
                        (&S.z[t].x)[h] = r[u].z;
                        (&S.w[t].x)[h] = wj[u];
                    }
                    off += __popc(keep[u]);
                }
                staged += add;
                if (staged <= kNbCap - 32 * NW * kNbGrp && (more || m0 + NW * kNbGrp < nchunk)) {
                    g.sync();
                    continue;
                }
                // fill up to a multiple of 64 with candidates that fail every test
                const int full = (staged + 63) / 64 * 64;
                for (int s = staged + tid; s < full; s += kForceBlock) {
                    const int t = (s >> 6) * 32 + (s & 31), h = (s >> 5) & 1;
                    (&S.x[t].x)[h] = (&S.y[t].x)[h] = (&S.z[t].x)[h] = __int_as_float(0x7fc00000);   // NaN
                    (&S.w[t].x)[h] = 0;
                }
                g.sync();
                if (nst == 27)
                    nbuild_scan<P, false>(a, g, rp, ctr, pn, ob, nown, full, K, S);
                else
                    nbuild_scan<P, true>(a, g, rp, ctr, pn, ob, nown, full, K, S);
                staged = 0;
                g.sync();
            }
            g.sync();                                      // (the table is written again)
        }
        for (int o = tid; o < nown; o += kForceBlock) {
            const int cnt = S.cnt[o], kept = cnt < K ? cnt : K;
            a.nnbr[ob + o] = kept;
            // pad the row with the particle itself to a multiple of kUnr entries, so the
            // pair loop reads whole groups without masking (K is a multiple of 8)
            for (int k = kept; k < (kept + kUnr - 1) / kUnr * kUnr && k < K; ++k)
                a.nbr[(size_t)(ob + o) * (size_t)a.Kstride + k] = ob + o;
            atomicMax(&S.max_nbr, cnt);
        }
        g.sync();
        if (tid == 0)
            atomicMax(&a.ctl->max_nbr, S.max_nbr);
        g.sync();
    }
}

// ---------------------------------------------------------------------------
// The same lists in the same order by one warp per cell, its lanes the cell's
// particles (batches of 32), where there are cells enough to give every warp
// one: each lane tests the staged candidates one after the other (every read a
// broadcast of two candidates), and stores the ones kept straight into its row.
// About ten instructions per candidate and warp, whatever number of lanes is in
// use, against about two per candidate and particle of the form above: fewer
// from ~6 particles a cell on, and no barrier; but a cell's time is a serial
// chain of its ~400 candidates, so few cells are better shared out as above.
// ---------------------------------------------------------------------------
constexpr int kNbStage = 224;    // staged candidates per round and warp (a multiple of 32)
constexpr int kNbBatch = 4;      // stencil cells whose particles are loaded at once

struct NbWarp {
    float4 a[kNbStage / 2], b[kNbStage / 2];   // two candidates: (x, x', y, y'), (z, z', w, w')
};

// Tests of the staged candidates [0, n): lane's particle at (hx, hy, hz) negated;
// the entries kept go to `row` (bytes) + off, cnt counts them.  Blocks of 32
// candidates that cannot overflow a row take the loop without that test.
template <bool WRAP>
__device__ __forceinline__ void nbuild_scan_warp(const NbWarp &S, int n, const Rep &rp, float2 hx, float2 hy, float2 hz,
                                                 float rl0, float rl1, int wi, int K, char *row, int &cnt)
{
    for (int p0 = 0; p0 < n / 2; p0 += 16) {
        const int p1 = min(p0 + 16, n / 2);
        if (!WRAP && (int)__reduce_max_sync(0xffffffffu, (unsigned)cnt) + 32 <= K) {
            unsigned off = 4u * (unsigned)cnt;
#pragma unroll 4
            for (int p = p0; p < p1; ++p) {
                const float4 A = S.a[p], B = S.b[p];
                const float2 dx = __fadd2_rn(make_float2(A.x, A.y), hx), dy = __fadd2_rn(make_float2(A.z, A.w), hy),
                             dz = __fadd2_rn(make_float2(B.x, B.y), hz);
                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                const int w0 = __float_as_int(B.z), w1 = __float_as_int(B.w);
                if (r2.x < (w0 < 0 ? rl1 : rl0) && w0 != wi) {
                    *(int *)(row + off) = w0 & 0x7fffffff;
                    off += 4u;
                }
                if (r2.y < (w1 < 0 ? rl1 : rl0) && w1 != wi) {
                    *(int *)(row + off) = w1 & 0x7fffffff;
                    off += 4u;
                }
            }
            cnt = (int)(off >> 2);
        } else {
            for (int p = p0; p < p1; ++p) {
                const float4 A = S.a[p], B = S.b[p];
                float2 dx = __fadd2_rn(make_float2(A.x, A.y), hx), dy = __fadd2_rn(make_float2(A.z, A.w), hy),
                       dz = __fadd2_rn(make_float2(B.x, B.y), hz);
                if (WRAP) {
                    dx.x = fmaf(-rintf(dx.x * rp.invLf), rp.Lhi, dx.x);
                    dx.y = fmaf(-rintf(dx.y * rp.invLf), rp.Lhi, dx.y);
                    dy.x = fmaf(-rintf(dy.x * rp.invLf), rp.Lhi, dy.x);
                    dy.y = fmaf(-rintf(dy.y * rp.invLf), rp.Lhi, dy.y);
                    dz.x = fmaf(-rintf(dz.x * rp.invLf), rp.Lhi, dz.x);
                    dz.y = fmaf(-rintf(dz.y * rp.invLf), rp.Lhi, dz.y);
                }
                const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
                const int w0 = __float_as_int(B.z), w1 = __float_as_int(B.w);
                if (r2.x < (w0 < 0 ? rl1 : rl0) && w0 != wi) {
                    if (cnt < K)
                        *(int *)(row + 4u * (unsigned)cnt) = w0 & 0x7fffffff;
                    ++cnt;
                }
                if (r2.y < (w1 < 0 ? rl1 : rl0) && w1 != wi) {
                    if (cnt < K)
                        *(int *)(row + 4u * (unsigned)cnt) = w1 & 0x7fffffff;
                    ++cnt;
                }
            }
        }
    }
}

template <int P>
__device__ __forceinline__ void nbuild_cell_warp(const KArgs &a, int pn, int c, int K, NbWarp &S, int &longest)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int c0 = a.cstart[c], c1 = a.cstart[c + 1];
    const int4 cc = a.cxyz[c];
    if (c0 == c1)
        return;
    const Rep &rp = a.rep[cc.w];
    const int nst = rp.nc >= 3 ? 27 : 1;
    const NbCentre ctr = nb_centre<P>(rp, cc);
    const float hx = 0.5f * rp.Lhi / (float)rp.nc + 1e-3f;        // half edge of the cell's box
    const float rlmax2 = fmaxf(fmaxf(a.tab.rl2[0], a.tab.rl2[1]), fmaxf(a.tab.rl2[2], a.tab.rl2[3]));
    const unsigned lt_mask = (1u << lane) - 1u;
    int s0, s1;
    nb_stencil(a, rp, cc, nst, s0, s1);

    for (int ob = c0; ob < c1; ob += 32) {
        const bool own = ob + lane < c1;
        const int i = own ? ob + lane : ob;
        int sp;
        const float3 h = nb_rel<P>(a, rp, ctr, pn, i, sp);
        const float rl0 = own ? a.tab.rl2[sp * 2] : -1.0f;        // -1: nothing passes
        const float rl1 = own ? a.tab.rl2[sp * 2 + 1] : -1.0f;
        char *row = (char *)(a.nbr + (size_t)i * (size_t)a.Kstride);
        int cnt = 0, staged = 0;

        const auto scan = [&]() {
            if (staged & 1) {                                     // (a candidate that fails every test)
                if (lane == 0) {
                    float *f = (float *)&S.a[staged >> 1], *e = (float *)&S.b[staged >> 1];
                    f[1] = f[3] = e[1] = __int_as_float(0x7fc00000);
                    e[3] = 0.f;
                }
                ++staged;
            }
            __syncwarp();
            if (nst == 27)
                nbuild_scan_warp<false>(S, staged, rp, make_float2(-h.x, -h.x), make_float2(-h.y, -h.y),
                                        make_float2(-h.z, -h.z), rl0, rl1, i | (sp << 31), K, row, cnt);
            else
                nbuild_scan_warp<true>(S, staged, rp, make_float2(-h.x, -h.x), make_float2(-h.y, -h.y),
                                       make_float2(-h.z, -h.z), rl0, rl1, i | (sp << 31), K, row, cnt);
            __syncwarp();
            staged = 0;
        };
        // stage the lanes' particles r (index and species in w), in lane order
        const auto stage = [&](const float3 &r, int w, bool ok) {
            if (nst == 27) {
                const float gx = fmaxf(fabsf(r.x) - hx, 0.f), gy = fmaxf(fabsf(r.y) - hx, 0.f),
                            gz = fmaxf(fabsf(r.z) - hx, 0.f);
                ok = ok && fmaf(gx, gx, fmaf(gy, gy, gz * gz)) < rlmax2;
            }
            const unsigned m = __ballot_sync(FULL, ok);
            if (staged + 32 > kNbStage)
                scan();
            if (ok) {
                const int s = staged + __popc(m & lt_mask);
                float *f = (float *)&S.a[s >> 1] + (s & 1), *e = (float *)&S.b[s >> 1] + (s & 1);
                f[0] = r.x;
                f[2] = r.y;
                e[0] = r.z;
                e[2] = __int_as_float(w);
            }
            staged += __popc(m);
        };
        for (int k0 = 0; k0 < nst; k0 += kNbBatch) {
            float3 r[kNbBatch];
            int w[kNbBatch];
#pragma unroll
            for (int u = 0; u < kNbBatch; ++u) {
                const int k = min(k0 + u, 31);
                const int t = __shfl_sync(FULL, s0, k) + lane, e = __shfl_sync(FULL, s1, k);
                int tsp = 0;
                w[u] = -1;
                r[u] = make_float3(0.f, 0.f, 0.f);
                if (t < e) {
                    r[u] = nb_rel<P>(a, rp, ctr, pn, checked(a, t, a.n, 0), tsp);
                    w[u] = t;
                }
                if (tsp)
                    w[u] |= 1 << 31;
                else if (w[u] < 0)
                    w[u] = 0x7fffffff;                            // (no particle)
            }
#pragma unroll
            for (int u = 0; u < kNbBatch; ++u) {
                const int k = min(k0 + u, 31);
                const int t0 = __shfl_sync(FULL, s0, k), e = __shfl_sync(FULL, s1, k);
                if (t0 < e)
                    stage(r[u], w[u], w[u] != 0x7fffffff);
                for (int t = t0 + 32; t < e; t += 32) {           // (a cell of more than 32 particles)
                    float3 q = make_float3(0.f, 0.f, 0.f);
                    int tsp = 0;
                    if (t + lane < e)
                        q = nb_rel<P>(a, rp, ctr, pn, checked(a, t + lane, a.n, 0), tsp);
                    stage(q, (t + lane) | (tsp << 31), t + lane < e);
                }
            }
        }
        scan();

        if (own) {
            // padding with the particle itself to a multiple of kUnr entries, so the pair
            // loop reads whole groups without masking
            const int kept = cnt < K ? cnt : K;
            for (int k = kept; k < (kept + kUnr - 1) / kUnr * kUnr && k < K; ++k)
                ((int *)row)[k] = i;
            a.nnbr[i] = kept;
            longest = max(longest, cnt);
        }
        __syncwarp();
    }
}

// List capacity after a build whose longest list held mx > K entries (the
// fixed-size list of Sec. 2.2 grown in place): a quarter more than needed,
// rounded up to whole groups of 8, at most the cap Kmax (a multiple of 8, so
// the result still holds mx entries whenever mx <= Kmax).
__device__ __forceinline__ int grown_capacity(int mx, int Kmax)
{
    const int want = (mx + (mx + 3) / 4 + 7) / 8 * 8;
    return want < Kmax ? want : Kmax;
}

// ---------------------------------------------------------------------------
// k_run: md_step and force evaluations as one cooperative launch.  Its blocks
// are all resident; each MD step is one sweep over the block's chunks of
// particles and one barrier of the grid, whose last arriver decides, with a
// bound on how far particles can move before the next check, whether the lists
// must be rebuilt (the displacement criterion of Sec. 2.2); the rebuild runs in
// the same launch, a grid barrier after each of its phases.
//
// What bounds a step of a small system is latency: the launches, conditional
// nodes and idle steps of a graph of one kernel per step cost more than the
// forces.  The barrier (one atomic per block, then polling one word) replaces
// all of them.
//
// What every block must know alike (step, buffer parities, list capacity, what
// to do next) is kept per block in shared memory and follows from the flags
// that a barrier returns, so no block reads control words that another one may
// be changing.
// ---------------------------------------------------------------------------
enum RunFlag : unsigned int {
    RF_REBUILD = 1u,   // step: the lists must be rebuilt; build: redo it with the raised capacity
    RF_STOP = 2u,      // nothing follows
    RF_BAD = 4u,       // the phase failed (Ctl::status): its results are not made current
    RF_ABORT = 8u      // a barrier gave up waiting: leave at once
};

struct RunState {
    long long step, left, obs, rebuilds, regrows, budget;
    long long pend;                // step whose partial sums await their sum (-1: none)
    long long pend_obs, pend_rebuilds;
    unsigned long long t0, ns;
    int pp, spar, K, pos;
    int pend_sample;
    int last, sample, check, track; // of the running step: ends md_step, is a sample, is checked, needs maxima
    int to_sample;                 // steps until the next sample step
    int bad;                       // something went wrong in this block
    int unit;                      // next unit (cell or share of one) of the block's in the build

    Rep rep;                       // of a handle of one replica
    long long done;
    unsigned int count, flags;     // barriers passed (thread 0), flags of the last one
};

// Shared scratch of a group.  Of a step: sums, and what a thread keeps between
// its chunks (registers are scarce in the pair loop).
template <int P> struct PairScratch { __device__ PairQueue *queue(int) { return nullptr; } };
template <> struct PairScratch<FP64> {
    PairQueue q[kGrpWarps];
    __device__ PairQueue *queue(int w) { return q + w; }
};

template <int P>
struct RunSums {
    PairScratch<P> pair;
    double sh[kGrpWarps * kPartF];
    double tot[kPartF];                              // sums of a one-replica sample
    double e[kForceBlock];                           // energy (ET) and maxima so far, per thread
    float d2[kForceBlock], v2[kForceBlock], a2[kForceBlock];
};

template <int P>
struct RunGroup {
    union {
        NbBlock nb;
        NbWarp nbw[kGrpWarps];
        RunSums<P> step;
        int scan[kGrpWarps];
    };
    int4 row;                                        // the group's first chunk
    __align__(16) float es[4 * kGrpWarps];
    float mx[3 * kGrpWarps];
    int unit;                                        // the group's unit of the build
};

// Every block arrives; `decide` runs in thread 0 of the last one, sees the
// writes of all blocks and returns the flags that every block gets; `after` runs
// in thread 0 of every block with these flags.
template <class F, class G>
__device__ __forceinline__ unsigned int grid_barrier(const KArgs &a, RunState &S, F &&decide, G &&after)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        RunSync *rs = a.rs;
        const unsigned int next = (S.count + 1u) & 0x0fffffffu;
        unsigned int t, w;
        // (the high half counts the blocks with something wrong)
        const unsigned int add = S.bad ? 0x10001u : 1u;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;"
                     : "=r"(t) : "l"(&rs->arrive), "r"(add) : "memory");
        t += add;
        if ((t & 0xffffu) == gridDim.x) {
            rs->arrive = 0u;
            w = (next << 4) | decide((t >> 16) != 0u);
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&rs->word), "r"(w) : "memory");
        } else {
            unsigned int n = 0;
            // (polls without acquire: an acquire empties the SM's L1, which its other
            // blocks still use)
            do {
                asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(&rs->word) : "memory");
            } while ((w >> 4) != next && ++n < a.spin_max);
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            if ((w >> 4) != next) {
                atomicOr(&a.ctl->stale, STALE_LISTS | STALE_STATE);
                atomicOr(&a.ctl->status, ST_TIMEOUT);
                a.ctl->halted = 1u;
                w = RF_STOP | RF_BAD | RF_ABORT;
            }
        }
        S.count = next;
        S.flags = w & 15u;
        after(w & 15u);
    }
    __syncthreads();
    return S.flags;
}

__device__ __forceinline__ unsigned int grid_barrier(const KArgs &a, RunState &S)
{
    return grid_barrier(a, S, [](bool) -> unsigned int { return 0u; }, [](unsigned int) {});
}

// Maxima of this group's displacements, speeds and accelerations into the step's,
// thread 0.
__device__ __forceinline__ void put_maxima(const KArgs &a, long long step, float d2, float v2, float a2)
{
    unsigned int *m = a.rs->m[step & 1];
    if (d2 > 0.f)
        atomicMax(&m[0], __float_as_uint(d2));
    if (v2 > 0.f)
        atomicMax(&m[1], __float_as_uint(v2));
    if (a2 > 0.f)
        atomicMax(&m[2], __float_as_uint(a2));
}

__device__ __forceinline__ void put_bad(const KArgs &a, RunState &S, unsigned int bad)
{
    atomicOr(&a.ctl->status, bad);
    S.bad = 1;
}

// The whole grid's maxima, cleared for the step after the next (last arriver of
// the step's barrier).  The displacement is kept by the parity of the step it
// leads to (of the positions it belongs to).
struct Maxima { float d2, v2, a2; };

__device__ __forceinline__ Maxima take_maxima(const KArgs &a, long long step)
{
    uint4 *m = reinterpret_cast<uint4 *>(a.rs->m[step & 1]);
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(m) : "memory");
    *m = make_uint4(0u, 0u, 0u, 0u);
    a.rs->md2[(step + 1) & 1] = __uint_as_float(v.x);
    Maxima r;
    r.d2 = __uint_as_float(v.x);
    r.v2 = __uint_as_float(v.y);
    r.a2 = __uint_as_float(v.z);
    return r;
}

// Rebuild of the lists; returns the flags of its last barrier (the state's
// parities and capacity are those of the new lists unless RF_BAD).
template <int P>
__device__ __forceinline__ unsigned int run_rebuild(const KArgs &a, const Grp &g, RunState &S, RunGroup<P> &X)
{
    Ctl *ctl = a.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        ctl->max_nbr = 0;
    rebuild_bin<P>(a, g, S.pp);
    if (grid_barrier(a, S) & RF_ABORT)
        return S.flags;
    // cells per block of the scan; few cells: every block adds up the counts before its own
    const int slice_cells = (a.ncell + g.nvb - 1) / g.nvb;
    if (a.ncell > kScanDirect) {
        rebuild_slices(a, g, slice_cells, X.scan);
        if (grid_barrier(a, S) & RF_ABORT)
            return S.flags;
    }
    rebuild_scan(a, g, slice_cells, X.scan);
    if (grid_barrier(a, S) & RF_ABORT)
        return S.flags;
    rebuild_scatter(a, g);
    if (grid_barrier(a, S) & RF_ABORT)
        return S.flags;
    rebuild_permute<P>(a, g, S.pp, S.spar);
    const auto reset_units = [&](bool) -> unsigned int {
        a.rs->unit = g.nvb;
        return 0u;
    };
    if (grid_barrier(a, S, reset_units, [&](unsigned int) { S.unit = 0; }) & RF_ABORT)
        return S.flags;
    for (int retry = 0;; ++retry) {
        // the lists: at most K entries a row; the longest list decides.  Every SM has a run of
        // neighbouring cells, whose particles its L1 then holds; its warps or groups take them
        // in turns (the time per cell differs)
        const int pn = S.pp ^ 1, K = S.K;
        if (a.nb_warp) {
            const int u0 = (int)((long long)a.ncell * blockIdx.x / gridDim.x),
                      u1 = (int)((long long)a.ncell * (blockIdx.x + 1) / gridDim.x);
            int longest = 0;
            for (;;) {
                int u = 0;
                if ((threadIdx.x & 31) == 0)
                    u = u0 + atomicAdd(&S.unit, 1);
                u = __shfl_sync(0xffffffffu, u, 0);
                if (u >= u1)
                    break;
                nbuild_cell_warp<P>(a, pn, u, K, X.nbw[g.tid() >> 5], longest);
            }
            longest = (int)__reduce_max_sync(0xffffffffu, (unsigned)longest);
            if ((threadIdx.x & 31) == 0 && longest > 0)
                atomicMax(&ctl->max_nbr, longest);
        } else {
            // (ensembles have few, uneven cells: one counter for the whole grid, read ahead)
            const int nparts = a.nb_parts, nunit = a.ncell * nparts;
            for (int u = g.vb; u < nunit;) {
                unsigned int nu = 0;
                if (g.tid() == 0)
                    nu = atomicAdd(&a.rs->unit, 1u);
                nbuild_cell<P>(a, g, pn, u / nparts, u % nparts, nparts, K, X.nb);
                if (g.tid() == 0)
                    X.unit = (int)nu;
                g.sync();
                u = X.unit;
                g.sync();
            }
        }
        const unsigned int f = grid_barrier(a, S, [&](bool) -> unsigned int {
            a.rs->unit = g.nvb;
            atomicOr(&ctl->stale, STALE_LISTS);      // (rref and the rows are those of the new order)
            if (atomicOr(&ctl->status, 0u))
                return RF_STOP | RF_BAD;
            const int mx = atomicMax(&ctl->max_nbr, 0);
            if (mx <= K) {
                a.rs->md2[S.step & 1] = 0.f;         // the lists start from these positions
                atomicAnd(&ctl->stale, ~(unsigned int)STALE_LISTS);
                return 0u;
            }
            if (mx <= ctl->Kmax && retry == 0) {
                // grow the capacity and redo the build: same positions, so the
                // same counts, and they fit
                ctl->K = grown_capacity(mx, ctl->Kmax);
                return RF_REBUILD;
            }
            atomicOr(&ctl->status, ST_OVERFLOW);
            return RF_STOP | RF_BAD;
        }, [&](unsigned int flags) {
            if (retry == 0)
                S.rebuilds += 1;
            S.unit = 0;
            if (flags & RF_REBUILD) {
                S.K = ctl->K;
                S.regrows += 1;
            } else if (!(flags & RF_BAD)) {
                S.pp ^= 1;
                S.spar ^= 1;
            }
        });
        if (!(f & RF_REBUILD))
            return f;
    }
}

// The half kick and drift that open md_step.
template <int P>
__device__ __forceinline__ void run_first(const KArgs &a, const Grp &g, RunState &S, RunGroup<P> &X)
{
    const int pp = S.pp, spar = S.spar;
    float d2 = 0.f, v2 = 0.f, a2 = 0.f;
    unsigned int bad = 0u;
    for (int row = g.vb; row < a.nblk_i; row += g.nvb) {
        const int4 b = a.blk_i[row];
        const Rep rp = a.rep[b.z];
        for (int i = b.x + g.tid(); i < b.y; i += kForceBlock) {
            PState<P> s;
            load_pos<P>(a, pp, i, s);
            load_vel<P>(a, spar, i, s);
            FT<P> f[3];
            if constexpr (P == FP64) {
                const d4 q = ((const d4 *)a.force)[i];
                f[0] = q.x; f[1] = q.y; f[2] = q.z;
            } else {
                const float4 q = ((const float4 *)a.force)[i];
                f[0] = q.x; f[1] = q.y; f[2] = q.z;
            }
            half_kick<P>(a, s, f[0], f[1], f[2]);
            d2 = fmaxf(d2, drift<P>(a, rp, s, pp ^ 1, spar, i, true, bad));
            v2 = fmaxf(v2, speed2(s));
            const float im = a.inv_mass[s.sp];
            a2 = fmaxf(a2, __fmul_rn(__fmul_rn(norm2(f[0], f[1], f[2]), im), im));
            store_vel<P>(a, spar, i, s);
        }
    }
    if (bad)
        put_bad(a, S, bad);
    grp_max3(g, d2, v2, a2, X.mx);
    if (g.tid() == 0)
        put_maxima(a, S.step, d2, v2, a2);
}

// One sweep over the group's chunks: forces, the particles' update, and the
// partial sums and maxima.
template <int P, int TPP, bool SM, bool SAMPLE>
__device__ __forceinline__ void run_chunks(const KArgs &a, const Grp &g, RunState &S, RunGroup<P> &G)
{
    RunSums<P> &X = G.step;
    PairQueue *Q = X.pair.queue(g.tid() >> 5);
    X.d2[g.tid()] = X.v2[g.tid()] = X.a2[g.tid()] = 0.f;
    ET<P> *xe = reinterpret_cast<ET<P> *>(X.e);
    xe[g.tid()] = e_zero<P>();
    if (SAMPLE && g.tid() < kPartF)
        X.tot[g.tid()] = 0.0;
    if (g.vb * a.cpb >= a.nrow)
        return;                                      // (a group without chunks)
    for (int q = 0; q < a.cpb; ++q) {
        const int4 b = q == 0 ? G.row : a.blk_r[g.vb * a.cpb + q];
        if (b.w < 0)                                 // (padding rows: the same for the whole group)
            break;
        double part[kPartF];
        ET<P> eo;
        float d2 = 0.f, v2 = 0.f, a2 = 0.f;
        unsigned int bad = 0u;
        step_body<P, TPP, SAMPLE, SM>(a, a.nrep == 1 ? S.rep : a.rep[b.z], Q, b, (a.what & RUN_STEPS) != 0, S.last != 0,
                                      S.track != 0, S.pp, S.spar, part, eo, d2, v2, a2, bad);
        if (bad)
            put_bad(a, S, bad);
        X.d2[g.tid()] = fmaxf(X.d2[g.tid()], d2);
        X.v2[g.tid()] = fmaxf(X.v2[g.tid()], v2);
        X.a2[g.tid()] = fmaxf(X.a2[g.tid()], a2);
        if (SAMPLE) {
            grp_sum(g, part, X.sh);
            if (g.tid() == 0) {
                double *p = a.nrep == 1 ? X.tot : a.part_f + part_index(a, S.step, b.w) * kPartF;
#pragma unroll
                for (int k = 1; k < kPartF; ++k)
                    p[k] = a.nrep == 1 ? p[k] + part[k] : part[k];
            }
        }
        if (a.nrep == 1) {
            xe[g.tid()] = e_add(xe[g.tid()], eo);
        } else {
            grp_esum(g, eo, G.es);
            if (g.tid() == 0)
                put_epart<P>(a, part_index(a, S.step, b.w), eo);
            g.sync();                                // (G.es is written again)
        }
    }
    if (S.track) {
        float d2 = X.d2[g.tid()], v2 = X.v2[g.tid()], a2 = X.a2[g.tid()];
        grp_max3(g, d2, v2, a2, G.mx);
        if (g.tid() == 0)
            put_maxima(a, S.step, d2, v2, a2);
    }
    ET<P> e = xe[g.tid()];
    if (a.nrep == 1)
        grp_esum(g, e, G.es);
    if (g.tid() == 0) {
        if (a.nrep == 1) {
            put_epart<P>(a, part_index(a, S.step, g.vb), e);
            if (SAMPLE) {
                double *p = a.part_f + part_index(a, S.step, g.vb) * kPartF;
#pragma unroll
                for (int k = 1; k < kPartF; ++k)
                    p[k] = X.tot[k];
            }
        }
    }
}

// Sums of the step that awaits them, one group per replica, the last groups of
// the grid first: they have the fewest chunks (none, where groups are to spare).
template <int P>
__device__ __forceinline__ void run_service(const KArgs &a, const Grp &g, RunState &S, bool totals, RunGroup<P> &X)
{
    if (S.pend < 0)
        return;
    for (int r = g.nvb - 1 - g.vb; r < a.nrep; r += g.nvb) {
        finish_replica<P>(a, g, r, S.pend, S.pend_sample != 0, totals, S.pend_obs % (long long)a.obs_cap,
                          a.rs->md2[S.pend & 1], S.pend_rebuilds, X.step.sh, X.es);
        if (r == 0 && g.tid() == 0 && !totals)
            a.epot_step[S.pend % a.epot_cap] = S.pend;
    }
}

// Groups per SM: 7 at <= 72 registers a thread for the unsmoothed single-precision
// kernels, so that 1024 chunks (KA N=65536 at 2 lanes per particle) are one per
// group on 152 SMs (1064 blocks of 128 threads took 26.5 us a step there, 7 groups
// 23.3); 5 at <= 96 for FP64 and the smoothed kernels.  The kernels of 7 groups spill
// (`-Xptxas -v`, bytes stored at 1 / 2 / 4 / 8 or more lanes: mixed 276 / 232 / 304 / 128,
// FP32 184 / 200 / 184 / 120), FP64 smoothed 180 to 192, the others 40 at most.  6 or 8
// groups were not measured at other sizes.
template <int P, bool SM> constexpr int run_groups() { return P == FP64 || SM ? 5 : 7; }

// What the step at S.step, position S.pos between checks, has to do (thread 0).
// The maxima are needed where a check follows and where the positions that the
// drift leads to are sampled.
__device__ __forceinline__ void run_plan(const KArgs &a, RunState &S)
{
    const bool steps = (a.what & RUN_STEPS) != 0;
    S.last = !steps || (S.left == 1 && a.last);
    S.sample = steps ? S.to_sample == 0 : (a.what & RUN_FORCES) == 0;
    S.check = !S.last && S.pos == a.check - 1;
    S.track = S.check || (!S.last && (S.to_sample == 1 || a.si == 1));
}

template <int P, int TPP, bool SM>
__global__ void __launch_bounds__(kForceBlock * run_groups<P, SM>(), 1) k_run(KArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ RunState S;
    Grp g;
    g.id = threadIdx.x / kForceBlock;
    g.vb = blockIdx.x + g.id * gridDim.x;            // (groups p, p + gridDim, ... share an SM)
    g.nvb = gridDim.x * (blockDim.x / kForceBlock);
    RunGroup<P> &X = reinterpret_cast<RunGroup<P> *>(smem)[g.id];
    Ctl *ctl = a.ctl;
    if (a.nrep == 1)
        for (int k = threadIdx.x; k < (int)(sizeof(Rep) / 4); k += blockDim.x)
            reinterpret_cast<int *>(&S.rep)[k] = reinterpret_cast<const int *>(a.rep)[k];
    if (g.tid() == 0)
        X.row = g.vb * a.cpb < a.nrow ? a.blk_r[g.vb * a.cpb] : make_int4(0, 0, 0, -1);
    if (threadIdx.x == 0) {
        S.step = ctl->step;
        S.left = a.nsteps;
        S.budget = a.budget;
        S.obs = ctl->obs_count;
        S.rebuilds = ctl->rebuilds;
        S.regrows = ctl->regrows;
        S.pend = -1;
        S.pp = ctl->pos_par;
        S.spar = ctl->state_par;
        S.K = ctl->K;
        S.pos = a.pos0;
        S.to_sample = (int)((a.si - S.step % a.si) % a.si);
        S.count = a.rs->word >> 4;
        S.ns = 0ull;
        S.done = 0;
        S.bad = 0;
        S.flags = ctl->halted;
        run_plan(a, S);
    }
    __syncthreads();
    // A status pending from before: nothing is done until it has been reported.  (Every
    // block sees the same word: a launch writes it after its last barrier, or when a
    // barrier gave up, and then a block that starts late has nothing to add.)
    if (S.flags) {
        if (blockIdx.x == 0 && threadIdx.x == 0)
            ctl->n_kernels += 1;
        return;
    }
    unsigned int f = 0u;
    if (a.what & RUN_REBUILD)
        f = run_rebuild<P>(a, g, S, X);
    if (!(f & RF_STOP) && (a.what & RUN_FIRST)) {
        run_first<P>(a, g, S, X);
        f = grid_barrier(a, S, [&](bool bad) -> unsigned int {
            const Maxima m = take_maxima(a, S.step);
            if (bad)
                return RF_STOP | RF_BAD;
            return need_rebuild(a, a.check - 1, m.d2, m.v2, m.a2) ? RF_REBUILD : 0u;
        }, [&](unsigned int flags) {
            if (!(flags & RF_BAD)) {
                S.step += 1;
                S.to_sample = S.to_sample == 0 ? a.si - 1 : S.to_sample - 1;
                S.pp ^= 1;
                run_plan(a, S);
            }
        });
        if ((f & RF_REBUILD) && !(a.what & RUN_DEFER))
            f = run_rebuild<P>(a, g, S, X);
    }
    const bool steps = (a.what & RUN_STEPS) != 0;
    if (!(f & RF_STOP) && (a.what & (RUN_STEPS | RUN_SAMPLE | RUN_TOTALS | RUN_FORCES))) {
        if (threadIdx.x == 0)
            S.t0 = global_ns();
        for (;;) {
            // the previous step's sums (its partials were complete at the last barrier)
            run_service<P>(a, g, S, false, X);
            if (S.sample)
                run_chunks<P, TPP, SM, true>(a, g, S, X);
            else
                run_chunks<P, TPP, SM, false>(a, g, S, X);
            f = grid_barrier(a, S, [&](bool bad) -> unsigned int {
                Maxima m = {0.f, 0.f, 0.f};
                if (S.track)
                    m = take_maxima(a, S.step);
                if (bad)
                    return RF_STOP | RF_BAD;
                unsigned int fl = 0u;
                if (S.check && need_rebuild(a, a.check - 1, m.d2, m.v2, m.a2))
                    fl |= RF_REBUILD;
                if (!S.last && S.budget == 1) {
                    atomicOr(&ctl->status, ST_TIMEOUT);
                    fl |= RF_STOP;
                }
                if (!steps || S.left == 1)
                    fl |= RF_STOP;
                return fl;
            }, [&](unsigned int flags) {
                S.pend = -1;
                if (!(flags & RF_BAD)) {
                    // this step's sums: by the service blocks during the next one
                    S.pend = (a.what & RUN_FORCES) ? -1 : S.step;
                    S.pend_sample = S.sample;
                    S.pend_obs = S.obs;
                    S.pend_rebuilds = S.rebuilds;
                    if (S.sample && !(a.what & RUN_TOTALS))
                        S.obs += 1;
                    if (!S.last) {
                        S.step += 1;
                        S.to_sample = S.to_sample == 0 ? a.si - 1 : S.to_sample - 1;
                        S.pp ^= 1;
                    }
                    S.left -= 1;
                    S.budget -= 1;
                    S.pos = S.pos == a.check - 1 ? 0 : S.pos + 1;
                    run_plan(a, S);
                }
                S.done += 1;
                if (blockIdx.x == 0) {
                    const unsigned long long t = global_ns();
                    S.ns += t > S.t0 ? t - S.t0 : 0ull;
                    S.t0 = t;
                }
            });
            if (f & RF_ABORT)
                return;
            if (f & RF_STOP) {
                run_service<P>(a, g, S, (a.what & RUN_TOTALS) != 0, X);
                break;
            }
            if (f & RF_REBUILD) {
                f = run_rebuild<P>(a, g, S, X);
                if (f & RF_ABORT)
                    return;
                if (f & RF_STOP) {
                    run_service<P>(a, g, S, false, X);
                    break;
                }
                if (threadIdx.x == 0)
                    S.t0 = global_ns();
            }
        }
    }
    if (f & RF_ABORT)
        return;
    // the state of the handle, by one thread: the other blocks have passed their last barrier
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->step = S.step;
        ctl->obs_count = S.obs;
        ctl->rebuilds = S.rebuilds;
        ctl->regrows = S.regrows;
        ctl->pos_par = S.pp;
        ctl->state_par = S.spar;
        ctl->rebuild = (f & (RF_REBUILD | RF_BAD)) == RF_REBUILD;
        if (atomicOr(&ctl->status, 0u))
            ctl->halted = 1u;
        ctl->n_kernels += 1;
        if (steps) {
            ctl->dev_ns += S.ns;
            ctl->dev_launches += S.done;
        }
    }
}

// Kinetic energy and momentum of the current velocities per replica: into the
// totals record (IM_TOTALS), or as rescale factors (IM_KE) in scale[], which
// holds the target temperatures.  The last block adds up the blocks' sums, a
// block per replica up to 8 replicas, a warp per replica beyond.
__device__ __forceinline__ void put_kinetic(const KArgs &a, int r, const double *v)
{
    if (a.imode == IM_TOTALS) {
        Obs o;
        o.step = a.ctl->step;
        o.e_pot = o.virial = 0.0;
        for (int k = 0; k < 6; ++k)
            o.w[k] = 0.0;
        o.e_kin = v[0];
        o.p[0] = v[1];
        o.p[1] = v[2];
        o.p[2] = v[3];
        o.max_disp = 0.0;
        o.rebuilds = a.ctl->rebuilds;
        a.totals[r] = o;
    } else {
        const double dof = 3.0 * (double)a.rep[r].n - 3.0;
        const double target = a.scale[r];
        a.scale[r] = (v[0] > 0.0) ? sqrt(target * dof / (2.0 * v[0])) : 1.0;
    }
}

template <int P>
__global__ void __launch_bounds__(kIntBlock) k_kinetic(KArgs a)
{
    __shared__ double sh[32 * 4];
    __shared__ int s_last;
    Ctl *ctl = a.ctl;
    const bool halted = ctl->status != 0u;
    const int4 b = a.blk_i[blockIdx.x];
    const int i = b.x + threadIdx.x;
    double kin[4] = {0.0, 0.0, 0.0, 0.0};
    if (i < b.y && !halted) {
        PState<P> s;
        load_pos<P>(a, ctl->pos_par, i, s);
        load_vel<P>(a, ctl->state_par, i, s);
        kinetic<P>(a, s, kin);
    }
    block_sum<4>(kin, sh);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            a.part_i[(size_t)blockIdx.x * 4 + k] = kin[k];
        __threadfence();
        s_last = atomicAdd(&ctl->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last)
        return;
    __threadfence();
    const bool block_each = a.nrep <= 8;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (!halted)
        for (int r = block_each ? 0 : w; r < a.nrep; r += block_each ? 1 : nw) {
            const int b0 = a.rep[r].bi0, b1 = a.rep[r].bi1;
            double v[4] = {0.0, 0.0, 0.0, 0.0};
            for (int q = b0 + (block_each ? (int)threadIdx.x : lane); q < b1; q += block_each ? (int)blockDim.x : 32)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    v[k] += a.part_i[(size_t)q * 4 + k];
            if (block_each) {
                block_sum<4>(v, sh);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    v[k] = warp_sum(v[k]);
            }
            if (block_each ? threadIdx.x == 0 : lane == 0)
                put_kinetic(a, r, v);
        }
    if (threadIdx.x == 0) {
        ctl->ticket = 0u;
        ctl->n_kernels += 1;
    }
}

template <int P>
__global__ void __launch_bounds__(kIntBlock) k_load(KArgs a)
{
    Ctl *ctl = a.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        atomicAdd((unsigned long long *)&ctl->n_kernels, 1ull);
        ctl->stale = STALE_LISTS;
    }
    const int4 b = a.blk_i[blockIdx.x];
    const int i = b.x + threadIdx.x;
    if (i >= b.y)
        return;
    const int pp = ctl->pos_par, spar = ctl->state_par;
    const Rep rp = a.rep[b.z];
    const int sp = a.st_code[i];
    double x[3];
    int im[3];
    for (int k = 0; k < 3; ++k) {
        const double v = a.st_pos[3 * (size_t)i + k];
        const double q = floor(v * rp.invL);
        double w = v - q * rp.L;
        int m = a.st_img[3 * (size_t)i + k] + (int)q;
        if (w >= rp.L) { w -= rp.L; m += 1; }
        if (w < 0.0) { w += rp.L; m -= 1; }
        x[k] = w;
        im[k] = m;
    }
    const double *vv = a.st_vel + 3 * (size_t)i;
    if constexpr (P == FP64) {
        d4 p, v;
        p.x = x[0]; p.y = x[1]; p.z = x[2]; p.w = __longlong_as_double((long long)sp);
        v.x = vv[0]; v.y = vv[1]; v.z = vv[2]; v.w = 0.0;
        ((d4 *)pos_a(a, pp))[i] = p;
        ((d4 *)vel_a(a, spar))[i] = v;
    } else if constexpr (P == MIXED) {
        float H[3], l[3];
        for (int k = 0; k < 3; ++k) {
            // high word on the grid: multiples of rp.grid are exact in float for |x| < 2L
            const double h = rint(x[k] * (double)rp.inv_grid) * (double)rp.grid;
            H[k] = (float)h;
            l[k] = __double2float_rn(x[k] - h);
        }
        ((float4 *)pos_a(a, pp))[i] = make_float4(H[0], H[1], H[2], __int_as_float(sp));
        ((float4 *)pos_b(a, pp))[i] = make_float4(l[0], l[1], l[2], 0.f);
        q_of(a, pp)[i] = make_int4((int)fixq(H[0], l[0], rp), (int)fixq(H[1], l[1], rp),
                                   (int)fixq(H[2], l[2], rp), sp);
        ds vx = ds_from_double(vv[0]), vy = ds_from_double(vv[1]), vz = ds_from_double(vv[2]);
        ((float4 *)vel_a(a, spar))[i] = make_float4(vx.hi, vy.hi, vz.hi, 0.f);
        ((float4 *)vel_b(a, spar))[i] = make_float4(vx.lo, vy.lo, vz.lo, 0.f);
    } else {
        float fx = __double2float_rn(x[0]), fy = __double2float_rn(x[1]), fz = __double2float_rn(x[2]);
        const float L = rp.Lhi;
        // a coordinate just below L can round to L: it is 0 of the next image
        if (fx >= L) { fx = 0.f; im[0] += 1; }
        if (fy >= L) { fy = 0.f; im[1] += 1; }
        if (fz >= L) { fz = 0.f; im[2] += 1; }
        ((float4 *)pos_a(a, pp))[i] = make_float4(fx, fy, fz, __int_as_float(sp));
        ((float4 *)vel_a(a, spar))[i] = make_float4((float)vv[0], (float)vv[1], (float)vv[2], 0.f);
    }
    img_of(a, spar)[i] = make_int4(im[0], im[1], im[2], i);
}

// Write the state back to the staging area in the original order.
template <int P>
__global__ void __launch_bounds__(kIntBlock) k_getstate(KArgs a)
{
    const Ctl *ctl = a.ctl;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        atomicAdd((unsigned long long *)&a.ctl->n_kernels, 1ull);
        a.st_img[3 * (size_t)a.n] = (int)(ctl->stale & STALE_STATE);   // (read back with the images)
    }
    if (s >= a.n)
        return;
    const int pp = ctl->pos_par, spar = ctl->state_par;
    const int4 im = img_of(a, spar)[s];
    const size_t t = (size_t)im.w;
    double x[3], v[3];
    if constexpr (P == FP64) {
        const d4 p = ((const d4 *)pos_a(a, pp))[s], w = ((const d4 *)vel_a(a, spar))[s];
        x[0] = p.x; x[1] = p.y; x[2] = p.z;
        v[0] = w.x; v[1] = w.y; v[2] = w.z;
    } else if constexpr (P == MIXED) {
        const float4 H = ((const float4 *)pos_a(a, pp))[s], l = ((const float4 *)pos_b(a, pp))[s];
        const float4 vh = ((const float4 *)vel_a(a, spar))[s], vl = ((const float4 *)vel_b(a, spar))[s];
        x[0] = (double)H.x + (double)l.x; x[1] = (double)H.y + (double)l.y; x[2] = (double)H.z + (double)l.z;
        v[0] = (double)vh.x + (double)vl.x; v[1] = (double)vh.y + (double)vl.y; v[2] = (double)vh.z + (double)vl.z;
    } else {
        const float4 p = ((const float4 *)pos_a(a, pp))[s], w = ((const float4 *)vel_a(a, spar))[s];
        x[0] = p.x; x[1] = p.y; x[2] = p.z;
        v[0] = w.x; v[1] = w.y; v[2] = w.z;
    }
    for (int k = 0; k < 3; ++k) {
        a.st_pos[3 * t + k] = x[k];
        a.st_vel[3 * t + k] = v[k];
    }
    a.st_img[3 * t + 0] = im.x;
    a.st_img[3 * t + 1] = im.y;
    a.st_img[3 * t + 2] = im.z;
}

template <int P>
__global__ void __launch_bounds__(kIntBlock) k_expforce(KArgs a)
{
    const Ctl *ctl = a.ctl;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd((unsigned long long *)&a.ctl->n_kernels, 1ull);
    if (s >= a.n)
        return;
    const size_t t = (size_t)img_of(a, ctl->state_par)[s].w;
    double f[4];
    if constexpr (P == FP64) {
        const d4 q = ((const d4 *)a.force)[s];
        f[0] = q.x; f[1] = q.y; f[2] = q.z; f[3] = q.w;
    } else {
        const float4 q = ((const float4 *)a.force)[s];
        f[0] = q.x; f[1] = q.y; f[2] = q.z; f[3] = q.w;
    }
    a.st_f[3 * t + 0] = f[0];
    a.st_f[3 * t + 1] = f[1];
    a.st_f[3 * t + 2] = f[2];
    a.st_e[t] = f[3];
}

// v <- v * scale[replica]  (exact rescale, Sec. 2.3)
template <int P>
__global__ void __launch_bounds__(kIntBlock) k_scale(KArgs a)
{
    const Ctl *ctl = a.ctl;
    if (ctl->status)
        return;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd((unsigned long long *)&a.ctl->n_kernels, 1ull);
    const int4 b = a.blk_i[blockIdx.x];
    const int i = b.x + threadIdx.x;
    if (i >= b.y)
        return;
    const int spar = ctl->state_par;
    const double f = a.scale[b.z];
    if constexpr (P == FP64) {
        d4 v = ((d4 *)vel_a(a, spar))[i];
        v.x *= f; v.y *= f; v.z *= f;
        ((d4 *)vel_a(a, spar))[i] = v;
    } else if constexpr (P == MIXED) {
        const ds fs = ds_from_double(f);
        float4 vh = ((float4 *)vel_a(a, spar))[i], vl = ((float4 *)vel_b(a, spar))[i];
        ds x = ds_mul(ds_from(vh.x, vl.x), fs), y = ds_mul(ds_from(vh.y, vl.y), fs),
           z = ds_mul(ds_from(vh.z, vl.z), fs);
        ((float4 *)vel_a(a, spar))[i] = make_float4(x.hi, y.hi, z.hi, 0.f);
        ((float4 *)vel_b(a, spar))[i] = make_float4(x.lo, y.lo, z.lo, 0.f);
    } else {
        float4 v = ((float4 *)vel_a(a, spar))[i];
        const float ff = (float)f;
        v.x *= ff; v.y *= ff; v.z *= ff;
        ((float4 *)vel_a(a, spar))[i] = v;
    }
}

// clear a reported status so that the handle can be inspected and reused
template <int P>
__global__ void k_reset(KArgs a)
{
    a.ctl->status = 0u;
    a.ctl->halted = 0u;
    a.ctl->ticket = 0u;
    a.rs->arrive = 0u;
    for (int k = 0; k < 8; ++k)
        a.rs->m[k >> 2][k & 3] = 0u;
    a.ctl->n_kernels += 1;
}

// ---------------------------------------------------------------------------
// Andersen heat bath (Sec. 2.3): every particle draws a Maxwell-Boltzmann
// velocity from the rand48 sequence (x_{n+1} = a x_n + c mod 2^48; deviate n is
// x_{n+1} / 2^48).  Particle i (original index) is thread i of a leapfrog over
// the n particles: collision e uses its deviates (4e + k) n + i, k = 0..3.
// The first is reached by jumping ahead (the affine map raised to a power by
// squaring, exact in 64-bit integer arithmetic modulo 2^48), the others by the
// leapfrog x -> A_n x + C_n.  Box-Muller turns them into three normals; then
// k_andersen_fix removes the mean velocity and rescales to the target
// temperature exactly, per replica, from the FP64 totals.
// ---------------------------------------------------------------------------
constexpr unsigned long long kR48A = 0x5DEECE66DULL, kR48C = 0xBULL, kR48Mask = 0xFFFFFFFFFFFFULL;

__device__ __forceinline__ unsigned long long r48_jump(unsigned long long x, unsigned long long p)
{
    unsigned long long A = 1, C = 0, Ab = kR48A, Cb = kR48C;   // result map, map^(2^k)
    while (p) {
        if (p & 1ull) {
            A = (Ab * A) & kR48Mask;
            C = (Ab * C + Cb) & kR48Mask;
        }
        Cb = (Ab * Cb + Cb) & kR48Mask;
        Ab = (Ab * Ab) & kR48Mask;
        p >>= 1;
    }
    return (A * x + C) & kR48Mask;
}

template <int P>
__global__ void __launch_bounds__(kIntBlock) k_andersen(KArgs a)
{
    const Ctl *ctl = a.ctl;
    if (ctl->status)
        return;
    const int4 b = a.blk_i[blockIdx.x];
    const int i = b.x + threadIdx.x;
    if (i >= b.y)
        return;
    const int spar = ctl->state_par;
    const int orig = img_of(a, spar)[i].w;
    int sp;
    if constexpr (P == FP64)
        sp = species_of(((const d4 *)pos_a(a, ctl->pos_par))[i].w);
    else
        sp = species_of(((const float4 *)pos_a(a, ctl->pos_par))[i].w);
    unsigned long long x = r48_jump(a.r48_x0, (unsigned long long)a.r48_base + (unsigned long long)orig + 1ull);
    double u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        u[k] = (double)x * 0x1p-48;
        x = (a.r48_AN * x + a.r48_CN) & kR48Mask;
    }
    const double s = sqrt(a.scale[b.z] / a.mass[sp]);
    const double r1 = s * sqrt(-2.0 * log(1.0 - u[0])), r2 = s * sqrt(-2.0 * log(1.0 - u[2]));
    double s1, c1, s3, c3;
    sincospi(2.0 * u[1], &s1, &c1);
    sincospi(2.0 * u[3], &s3, &c3);
    const double v[3] = {r1 * c1, r1 * s1, r2 * c3};
    if constexpr (P == FP64) {
        d4 w;
        w.x = v[0]; w.y = v[1]; w.z = v[2]; w.w = 0.0;
        ((d4 *)vel_a(a, spar))[i] = w;
    } else if constexpr (P == MIXED) {
        const ds x0 = ds_from_double(v[0]), y0 = ds_from_double(v[1]), z0 = ds_from_double(v[2]);
        ((float4 *)vel_a(a, spar))[i] = make_float4(x0.hi, y0.hi, z0.hi, 0.f);
        ((float4 *)vel_b(a, spar))[i] = make_float4(x0.lo, y0.lo, z0.lo, 0.f);
    } else {
        ((float4 *)vel_a(a, spar))[i] = make_float4((float)v[0], (float)v[1], (float)v[2], 0.f);
    }
}

// v <- (v - P/M) s with s = sqrt(T (3N - 3) / (2 E_kin')), E_kin' = E_kin - |P|^2 / 2M,
// from the per-replica totals (E_kin, P) of the drawn velocities
template <int P>
__global__ void __launch_bounds__(kIntBlock) k_andersen_fix(KArgs a)
{
    const Ctl *ctl = a.ctl;
    if (ctl->status)
        return;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd((unsigned long long *)&a.ctl->n_kernels, 1ull);
    const int4 b = a.blk_i[blockIdx.x];
    const int i = b.x + threadIdx.x;
    if (i >= b.y)
        return;
    const Rep &rp = a.rep[b.z];
    const Obs &t = a.totals[b.z];
    const double M = rp.mtot;
    const double cx = t.p[0] / M, cy = t.p[1] / M, cz = t.p[2] / M;
    const double ek = t.e_kin - 0.5 * (t.p[0] * t.p[0] + t.p[1] * t.p[1] + t.p[2] * t.p[2]) / M;
    const double T = a.scale[b.z];
    const double f = (rp.n > 1 && T > 0.0 && ek > 0.0) ? sqrt(T * (3.0 * rp.n - 3.0) / (2.0 * ek)) : 0.0;
    const int spar = ctl->state_par;
    if constexpr (P == FP64) {
        d4 v = ((d4 *)vel_a(a, spar))[i];
        v.x = (v.x - cx) * f; v.y = (v.y - cy) * f; v.z = (v.z - cz) * f;
        ((d4 *)vel_a(a, spar))[i] = v;
    } else if constexpr (P == MIXED) {
        const float4 vh = ((float4 *)vel_a(a, spar))[i], vl = ((float4 *)vel_b(a, spar))[i];
        const ds x = ds_from_double((ds_to_double(ds_from(vh.x, vl.x)) - cx) * f);
        const ds y = ds_from_double((ds_to_double(ds_from(vh.y, vl.y)) - cy) * f);
        const ds z = ds_from_double((ds_to_double(ds_from(vh.z, vl.z)) - cz) * f);
        ((float4 *)vel_a(a, spar))[i] = make_float4(x.hi, y.hi, z.hi, 0.f);
        ((float4 *)vel_b(a, spar))[i] = make_float4(x.lo, y.lo, z.lo, 0.f);
    } else {
        float4 v = ((float4 *)vel_a(a, spar))[i];
        v.x = (float)((v.x - cx) * f); v.y = (float)((v.y - cy) * f); v.z = (float)((v.z - cz) * f);
        ((float4 *)vel_a(a, spar))[i] = v;
    }
}

// Snapshot for the time-correlation functions (Sec. 2.5): unwrapped positions
// r + L n (FP64) and species, stored by original particle index.
template <int P>
__global__ void __launch_bounds__(kIntBlock) k_snapshot(KArgs a)
{
    const Ctl *ctl = a.ctl;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd((unsigned long long *)&a.ctl->n_kernels, 1ull);
    const int4 b = a.blk_i[blockIdx.x];
    const int i = b.x + threadIdx.x;
    if (i >= b.y)
        return;
    const double L = a.rep[b.z].L;
    const int pp = ctl->pos_par, spar = ctl->state_par;
    const int4 im = img_of(a, spar)[i];
    double x[3];
    int sp;
    if constexpr (P == FP64) {
        const d4 p = ((const d4 *)pos_a(a, pp))[i];
        x[0] = p.x; x[1] = p.y; x[2] = p.z;
        sp = species_of(p.w);
    } else if constexpr (P == MIXED) {
        const float4 H = ((const float4 *)pos_a(a, pp))[i], l = ((const float4 *)pos_b(a, pp))[i];
        x[0] = (double)H.x + (double)l.x; x[1] = (double)H.y + (double)l.y; x[2] = (double)H.z + (double)l.z;
        sp = species_of(H.w);
    } else {
        const float4 p = ((const float4 *)pos_a(a, pp))[i];
        x[0] = p.x; x[1] = p.y; x[2] = p.z;
        sp = species_of(p.w);
    }
    const size_t t = (size_t)im.w;
    a.snap[3 * t + 0] = __dadd_rn(x[0], __dmul_rn(L, (double)im.x));
    a.snap[3 * t + 1] = __dadd_rn(x[1], __dmul_rn(L, (double)im.y));
    a.snap[3 * t + 2] = __dadd_rn(x[2], __dmul_rn(L, (double)im.z));
    a.snap_species[t] = sp;
}

template <int P>
KernelSet make_kernel_set()
{
    KernelSet k;
    k.kinetic = (const void *)k_kinetic<P>;
    k.groups[0] = run_groups<P, false>();
    k.groups[1] = run_groups<P, true>();
    k.group_smem = (int)sizeof(RunGroup<P>);
    k.run[0][0] = (const void *)k_run<P, 1, false>;
    k.run[0][1] = (const void *)k_run<P, 2, false>;
    k.run[0][2] = (const void *)k_run<P, 4, false>;
    k.run[0][3] = (const void *)k_run<P, 8, false>;
    k.run[0][4] = (const void *)k_run<P, 16, false>;
    k.run[0][5] = (const void *)k_run<P, 32, false>;
    // smoothed potential (Sec. 4): the common lane counts only
    k.run[1][0] = (const void *)k_run<P, 1, true>;
    k.run[1][1] = (const void *)k_run<P, 2, true>;
    k.run[1][2] = (const void *)k_run<P, 4, true>;
    k.run[1][3] = (const void *)k_run<P, 8, true>;
    k.run[1][4] = nullptr;
    k.run[1][5] = nullptr;
    k.load = (const void *)k_load<P>;
    k.getstate = (const void *)k_getstate<P>;
    k.expforce = (const void *)k_expforce<P>;
    k.scale = (const void *)k_scale<P>;
    k.reset = (const void *)k_reset<P>;
    k.andersen = (const void *)k_andersen<P>;
    k.andersen_fix = (const void *)k_andersen_fix<P>;
    k.snapshot = (const void *)k_snapshot<P>;
    return k;
}

}  // namespace mdk
