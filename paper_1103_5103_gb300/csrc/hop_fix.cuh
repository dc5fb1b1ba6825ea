// FP64 hop in block fixed point on the integer pipes (device code).
//
// GB300 executes FP64 at 1/57 of its FP32 rate (1.7 FMA per clock and SM
// measured) but a 32 x 32 + 64 bit integer multiply-add at 53-62 per clock
// and SM, so this hop carries an FP64 spinor through the stencil as 64-bit
// integers: exact adds, products of two 32-bit limbs each, one rounding back
// to FP64 at the end.
//
//  - Scale.  A component x becomes q = floor(x / 2^(E-58)), E the largest
//    exponent of the components that the thread has met so far; when a
//    neighbour raises E, the accumulators are shifted.
//  - Links are integers in units of 2^-62, packed once per gauge handle.
//  - A product keeps hi*hi in one 64-bit sum and hi*lo + lo*hi in another
//    (limbs are balanced: lo is signed, hi carries); the low word of the
//    second sum is rounded away once per colour row, lo*lo is dropped.  The
//    result is in units of 2^(E-56).
//  - Range: |q| < 2^59, the shrink doubles it, and a row of a link has unit
//    norm: a transported component is below 2.45 * 2^60 / 4 units of
//    2^(E-56), the sum of eight below 2^62.3.  Nothing overflows 63 bits.
//  - Error: a few units of 2^(E-56) per output component (below 2^(E-51)),
//    where one FP64 rounding of a value of the neighbours' size is 2^(E-53):
//    in norm the result is closer to the exact sum than that of eight FP64
//    transporters.  It is relative to the largest neighbour component, not to
//    each one: an input 2^-k of it counts with 58 - k bits, a result of that
//    size with about 53 - k.  Handles whose links keep colours apart, where
//    results of one colour can be small throughout, don't come here
//    (kMixingExp in layout.cu).
//  - A site with a neighbour component that is not finite, of 2^878 or more,
//    or whose components are not all zero and all below 2^-823 goes through
//    the FP64 transporters (the exponent range of the scale; infinities, NaN).
//
// Two threads per site, lanes l and l + 16 of a warp, one for each of the
// two colour vectors that the projector leaves: thread s takes spin s and
// the spin coupled to it (3 - s in x and y, 2 + s in z and t).  A whole site
// in one thread needs 168 registers (12 warps per SM) and ran 10% slower;
// small lattices get twice the threads.  The links and the spinor of a
// transporter are requested together before either is used (volatile loads:
// left to the compiler, the links came row by row, 2400 cycles of load
// latency per transporter).  Two bodies (phases +-i and +-1) serve the eight
// transporters: unrolled, 81 KB of code stalled on instruction fetch.
//
// 24^3x64, 3 rhs: 1998 -> 698 us (0.88 -> 2.51 TFLOP/s at 1320 flop per site
// and rhs); 1 rhs 674 -> 244 us; 8^4 34.8 -> 14.0 us.  Bound by the integer
// pipes: multiply-add pipe 70%, ALU 52%, FP64 pipe (conversion back and
// epilogue) 29% busy, issue 57%.  Also measured: spinors converted in a pass
// of their own (a hop 0.09 ns per site and rhs cheaper than its 0.53, the
// pass 0.07), three-product complex arithmetic with 27-real links (no
// faster), the shrink on the FP64 pipe (26% slower: its latency).
#pragma once

#include "hop.cuh"

namespace wl {

constexpr int kFixMinExp = 200;   // biased exponents the fixed-point path takes
constexpr int kFixMaxExp = 1900;
constexpr int kFixFrac = 58;      // q = x / 2^(E - kFixFrac)

typedef long long i64;
typedef unsigned long long u64;

// Shifts by any count >= 0 (PTX defines larger counts: all bits leave).
__device__ __forceinline__ u64 fix_shr(u64 v, int s)
{
    u64 r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
__device__ __forceinline__ i64 fix_sar(i64 v, int s)
{
    i64 r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}

// Loads that stay where they are written, ahead of the arithmetic: of links
// through the read-only path, of fields coherent (ld_field).
__device__ __forceinline__ int4 fix_ld_link(const int4 *p)
{
    int4 v;
    asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 fix_ld(const double2 *p)
{
    double2 v;
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

// Component x in units of 2^(E-58): q = result - mask, with the sign mask
// (0 or -1) added to neg.  flip (0 or -1) negates x.
__device__ __forceinline__ i64 fix_conv(double x, int E, int flip, int &neg)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi & 0x7fffffffu) >> 20);
    const unsigned mh = (hi & 0xfffffu) | 0x100000u;
    const u64 m = fix_shr((((u64)mh << 32) | lo) << (kFixFrac - 52), E - e);
    const int mask = ((int)hi >> 31) ^ flip;
    neg += mask;
    return (i64)(m ^ (u64)(i64)mask);
}

__device__ __forceinline__ int fix_absmax(int m, double2 v)
{
    return max(max(m, __double2hiint(v.x) & 0x7fffffff), __double2hiint(v.y) & 0x7fffffff);
}
__device__ __forceinline__ int fix_lobits(double2 v) { return __double2loint(v.x) | __double2loint(v.y); }

// v (-1)^m for m = 0 or -1
__device__ __forceinline__ i64 fix_neg(i64 v, i64 m) { return (v ^ m) - m; }

// High limb of the balanced split v = hi 2^32 + lo, lo = (int)v.
__device__ __forceinline__ int fix_hi(i64 v) { return (int)(v >> 32) + (int)((unsigned)v >> 31); }

// Offset of link (mu, site) in the integer links, int4 [4][stride / 32][9][32]
// (re.lo, re.hi, im.lo, im.hi): a link's nine entries are 32 apart.
__host__ __device__ __forceinline__ size_t fix_link(const Geom &g, int mu, int i)
{
    return (size_t)mu * 9 * g.stride + (size_t)(i >> 5) * (9 * 32) + (i & 31);
}

// The components of one neighbour that a thread takes: its own spin (a) and
// the spin that the direction couples to it (b).
struct FixRaw {
    double2 a[3], b[3];
};

__device__ __forceinline__ void fix_load(FixRaw &x, const void *in, size_t j, unsigned off_u, unsigned off_l, int stride)
{
    const double2 *q = static_cast<const double2 *>(in) + j;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        x.a[k] = fix_ld(q + (off_u + (unsigned)(k * stride)));
        x.b[k] = fix_ld(q + (off_l + (unsigned)(k * stride)));
    }
}

// A link, or with cj = -1 its transpose: u^dag h = conj(u^T conj(h)).
__device__ __forceinline__ void fix_load_link(int4 (&u)[9], const int4 *p, int cj)
{
    const int row = cj ? 32 : 96, col = cj ? 96 : 32;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int k = 0; k < 3; ++k) u[3 * r + k] = fix_ld_link(p + (r * row + k * col));
}

// One transporter of one colour vector: adds L psi (1 -/+ gamma_mu) for the
// thread's spin to up and to low (the spin coupled to it).  SWAP: the phases
// are +-i (x, z) instead of +-1 (y, t).  f: sign (0 or -1) of the phase; cj:
// -1 for u^dag (u then holds its transpose); neg: the time boundary.
template <bool SWAP>
__device__ __forceinline__ void fix_transport(const FixRaw &x, const int4 (&lk)[9], int f, int cj, bool neg, int &E,
                                              bool &special, i64 (&up)[6], i64 (&low)[6])
{
    int A = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) A = fix_absmax(fix_absmax(A, x.a[k]), x.b[k]);
    const int e = A >> 20;
    if (e > E) {
        const int sh = e - E;
        E = e;
        if (e > kFixMaxExp) special = true;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            up[k] = fix_sar(up[k], sh);
            low[k] = fix_sar(low[k], sh);
        }
    } else if (e < kFixMinExp) {   // zeros, or too small for the scale
        int z = A;
#pragma unroll
        for (int k = 0; k < 3; ++k) z |= fix_lobits(x.a[k]) | fix_lobits(x.b[k]);
        if (z != 0) special = true;
    }
    // shrink: h = a + phase b (its conjugate for u^dag), as limbs of re, im
    // and -im
    const int ts = neg ? -1 : 0, tc = ts ^ cj;
    int rh[3], rl[3], ih[3], il[3], nh[3], nl[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int n0 = 0, n1 = 0;
        i64 re = fix_conv(x.a[k].x, E, ts, n0), im = fix_conv(x.a[k].y, E, tc, n1);
        if constexpr (SWAP) {   // a + i sigma b
            re += fix_conv(x.b[k].y, E, ~f ^ ts, n0);
            im += fix_conv(x.b[k].x, E, f ^ tc, n1);
        } else {
            re += fix_conv(x.b[k].x, E, f ^ ts, n0);
            im += fix_conv(x.b[k].y, E, f ^ tc, n1);
        }
        re -= n0;
        im -= n1;
        rl[k] = (int)re;
        rh[k] = fix_hi(re);
        il[k] = (int)im;
        ih[k] = fix_hi(im);
        nl[k] = (int)-im;
        nh[k] = fix_hi(-im);
    }
    const i64 f64 = f, c64 = cj;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        i64 h0 = 0, h1 = 0, x0 = 1ll << 31, x1 = 1ll << 31;   // 2^31 rounds the dropped low word
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int4 u = lk[3 * r + k];
            h0 += (i64)u.y * rh[k];
            x0 += (i64)u.y * rl[k];
            x0 += (i64)u.x * rh[k];
            h1 += (i64)u.y * ih[k];
            x1 += (i64)u.y * il[k];
            x1 += (i64)u.x * ih[k];
            h0 += (i64)u.w * nh[k];
            x0 += (i64)u.w * nl[k];
            x0 += (i64)u.z * nh[k];
            h1 += (i64)u.w * rh[k];
            x1 += (i64)u.w * rl[k];
            x1 += (i64)u.z * rh[k];
        }
        const i64 re = h0 + (x0 >> 32), im = h1 + (x1 >> 32);   // w = (re, im), its conjugate for u^dag
        up[2 * r] += re;
        up[2 * r + 1] += fix_neg(im, c64);
        if constexpr (SWAP) {   // conj(i sigma) w = sigma (w.im, -w.re)
            low[2 * r] += fix_neg(im, f64 ^ c64);
            low[2 * r + 1] -= fix_neg(re, f64);
        } else {
            low[2 * r] += fix_neg(re, f64);
            low[2 * r + 1] += fix_neg(im, f64 ^ c64);
        }
    }
}

// FP64 value of an accumulator times scale: the integer rounded once to FP64
// (its halves as offset doubles, whose sum is exact up to that rounding),
// then the power of two of its scale.
__device__ __forceinline__ double fix_out(i64 v, double scale)
{
    const double lo = __hiloint2double(0x43300000, (int)v);                             // 2^52 + low word
    const double hi = __hiloint2double(0x45300000, (int)(v >> 32) ^ (int)0x80000000);   // 2^84 + 2^63 + high part
    return ((hi - (0x1p84 + 0x1p63 + 0x1p52)) + lo) * scale;
}

// The thread's accumulators and their scale.
struct FixAcc {
    i64 up[6], low[6];   // spin s; the spin that the direction couples to it
    int E;
    bool special;
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int k = 0; k < 6; ++k) up[k] = low[k] = 0;
        E = kFixMinExp;
        special = false;
    }
};

// What the transporters need of the output site.
struct FixSite {
    Coord c;
    int i;            // even-odd index (links)
    int nb[8];        // neighbours: forward, backward in x, y, z, t
    bool nf, nbk;     // time boundary
};

__device__ __forceinline__ FixSite fix_site(const HopArgs &a, int i)
{
    const Geom &g = a.g;
    FixSite q;
    q.c = site_coord(g, i, a.out_parity);
    const int rowbase = i - (q.c.x >> 1);
    bool f0, f1;
    neighbours<0>(g, i, q.c, rowbase, q.nb[0], q.nb[1], f0, f1);
    neighbours<1>(g, i, q.c, rowbase, q.nb[2], q.nb[3], f0, f1);
    neighbours<2>(g, i, q.c, rowbase, q.nb[4], q.nb[5], f0, f1);
    neighbours<3>(g, i, q.c, rowbase, q.nb[6], q.nb[7], q.nf, q.nbk);
#pragma unroll
    for (int k = 0; k < 8; ++k) q.nb[k] = WL_LOAD_IDX(q.nb[k], g.stride, 1);
    q.i = WL_LOAD_IDX(i, g.stride, 3);
    return q;
}

// Both transporters of directions x, z (SWAP) or y, t, by m = 0, 1.  CANON:
// the input is a canonical field ([site][12]) instead of an internal one.
template <bool DAG, bool CANON, bool SWAP>
__device__ __forceinline__ void fix_direction(const HopArgs &a, const void *in, const FixSite &q, int m, int s,
                                              FixAcc &A)
{
    const Geom &g = a.g;
    const int mu = (SWAP ? 0 : 1) + 2 * m;
    // signs of the phase of spin s in 1 - gamma: x (+, +), z (+, -); y (-, +), t (+, +)
    constexpr int PF = DAG ? -1 : 0;   // 1 + gamma in the forward hops of the adjoint
    const int f = (SWAP ? (m ? -s : 0) : (m ? 0 : s - 1)) ^ PF;
    const int cs = CANON ? 1 : g.stride;
    const unsigned off_u = (unsigned)(3 * s * cs), off_l = (unsigned)(3 * (m ? 2 + s : 3 - s) * cs);
    const int4 *lo = static_cast<const int4 *>(a.fix_out), *li = static_cast<const int4 *>(a.fix_in);
    FixRaw x;
    int4 u[9];
#pragma unroll 1
    for (int cj = 0; cj >= -1; --cj) {   // forward, backward
        const int j = m ? (cj ? (SWAP ? q.nb[5] : q.nb[7]) : (SWAP ? q.nb[4] : q.nb[6]))
                        : (cj ? (SWAP ? q.nb[1] : q.nb[3]) : (SWAP ? q.nb[0] : q.nb[2]));
        fix_load(x, in, CANON ? 12 * canon_site(q.c, a.out_parity, mu, j) : (size_t)j, off_u, off_l, cs);
        fix_load_link(u, (cj ? li : lo) + fix_link(g, mu, cj ? j : q.i), cj);
        fix_transport<SWAP>(x, u, f ^ cj, cj, !SWAP && m && (cj ? q.nbk : q.nf), A.E, A.special, A.up, A.low);
    }
}

// FP64 values of the accumulators (acc[0..2] spin s, acc[3..5] spin 3 - s),
// or those of the FP64 transporters for a special site.
template <bool DAG, bool CANON>
__device__ __forceinline__ void fix_values(const HopArgs &a, const void *in, int i, int s, const FixAcc &A,
                                           cx<double> (&acc)[6])
{
    if (!A.special) {
        const double scale = __hiloint2double((A.E + 2 - kFixFrac) << 20, 0);   // 2^(E - 1023 - 56)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            acc[k] = {fix_out(A.up[2 * k], scale), fix_out(A.up[2 * k + 1], scale)};
            acc[3 + k] = {fix_out(A.low[2 * k], scale), fix_out(A.low[2 * k + 1], scale)};
        }
    } else {
        HopArgs b = a;
        b.in = in;
        cx<double> full[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) full[k] = acc_zero<double>();
        hop_accumulate_rolled<WL_F64, DAG, CANON>(b, i, full);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            acc[k] = s ? full[3 + k] : full[k];
            acc[3 + k] = s ? full[6 + k] : full[9 + k];
        }
    }
}

// D in at site i by its two threads: thread s gets spin s in acc[0..2] and
// spin 3 - s in acc[3..5].  Every lane of the warp takes part.
template <bool DAG, bool CANON>
__device__ __forceinline__ void hop_half(const HopArgs &a, const void *in, int i, int s, cx<double> (&acc)[6])
{
    const FixSite q = fix_site(a, i);
    FixAcc A;
    A.clear();
#pragma unroll 1
    for (int m = 0; m < 2; ++m) {   // x, y, then z, t
        fix_direction<DAG, CANON, true>(a, in, q, m, s, A);
        fix_direction<DAG, CANON, false>(a, in, q, m, s, A);
        // the pair moves to the larger of its two scales and exchanges the
        // lower spins: after x, y thread s holds spin 3 - s and goes on with
        // 2 + s; after z, t it gets 3 - s back
        const int Eo = __shfl_xor_sync(0xffffffffu, A.E, 16);
        const int sh = max(0, Eo - A.E);
        A.E = max(A.E, Eo);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            A.up[k] = fix_sar(A.up[k], sh);
            A.low[k] = __shfl_xor_sync(0xffffffffu, fix_sar(A.low[k], sh), 16);
        }
    }
    A.special = __shfl_xor_sync(0xffffffffu, A.special ? 1 : 0, 16) || A.special;
    fix_values<DAG, CANON>(a, in, i, s, A, acc);
}

// Load and store of a thread's half of a site: spins s and 3 - s.
__device__ __forceinline__ void half_load(const void *base, int stride, int s, int i, cx<double> (&v)[6])
{
    i = WL_LOAD_IDX(i, stride, 1);
    const double2 *p = static_cast<const double2 *>(base) + i;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double2 x = ld_field(p + (size_t)(3 * s + k) * stride), y = ld_field(p + (size_t)(3 * (3 - s) + k) * stride);
        v[k] = {x.x, x.y};
        v[3 + k] = {y.x, y.y};
    }
}
__device__ __forceinline__ void half_store(void *base, int stride, int s, int i, const cx<double> (&v)[6])
{
    if (!WL_STORE_OK(i, stride, 2)) return;
    double2 *p = static_cast<double2 *>(base) + i;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[(size_t)(3 * s + k) * stride] = make_double2(v[k].re, v[k].im);
        p[(size_t)(3 * (3 - s) + k) * stride] = make_double2(v[3 + k].re, v[3 + k].im);
    }
}

// o = a1 x1 + a2 x2 + coef acc, stored, as EpiStore on the other hops.
__device__ __forceinline__ void half_epilogue(const EpiStore &e, int stride, int r, int s, int i,
                                              const cx<double> (&acc)[6], cx<double> (&o)[6])
{
    const size_t off = (size_t)r * e.rhs_bytes;
    if (e.out_raw) half_store(static_cast<char *>(e.out_raw) + off, stride, s, i, acc);
#pragma unroll
    for (int k = 0; k < 6; ++k) o[k] = e.coef * acc[k];
    if (e.x1) {
        cx<double> x[6];
        half_load(static_cast<const char *>(e.x1) + off, stride, s, i, x);
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = o[k] + e.a1 * x[k];
    }
    if (e.x2) {
        cx<double> x[6];
        half_load(static_cast<const char *>(e.x2) + off, stride, s, i, x);
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = o[k] + e.a2 * x[k];
    }
    half_store(static_cast<char *>(e.out) + off, stride, s, i, o);
}

// out = a1 x1 + a2 x2 + coef D in, as EpiStore on the other hops, for task
// `task`: 16 sites of one rhs.  The rhs of the same sites are consecutive
// tasks, taken by neighbouring warps, which share the links through L1.
template <bool DAG>
__device__ __forceinline__ void hop_fix_task(const HopArgs &a, const EpiStore &e, unsigned task, int lane)
{
    const int s = lane >> 4;
    const int r = (int)(task % (unsigned)a.nrhs);
    const int i0 = (int)(task / (unsigned)a.nrhs) * 16 + (lane & 15);
    if (i0 - (lane & 15) >= a.g.Vh || rhs_done(a, r)) return;   // the whole warp
    const bool active = i0 < a.g.Vh;
    const int i = active ? i0 : a.g.Vh - 1;
    cx<double> acc[6], o[6];
    hop_half<DAG, false>(a, static_cast<const char *>(a.in) + (size_t)r * a.rhs_bytes, i, s, acc);
    if (active) half_epilogue(e, a.g.stride, r, s, i, acc, o);
}

inline __host__ __device__ unsigned fix_tasks(const HopArgs &a)
{
    return (unsigned)((a.g.Vh + 15) / 16) * (unsigned)a.nrhs;
}

template <bool DAG>
__global__ void __launch_bounds__(128, 4) k_hop_fix(HopArgs a, EpiStore e)
{
    hop_fix_task<DAG>(a, e, blockIdx.x * 4 + (threadIdx.x >> 5) + chain_begin(), threadIdx.x & 31);
}

// The same with a fixed number of blocks that loop over the tasks: leaves
// the rest of each SM to work on other streams.
template <bool DAG>
__global__ void __launch_bounds__(128, 4) k_hop_fix_gs(HopArgs a, EpiStore e)
{
    const unsigned n = fix_tasks(a);
    for (unsigned t = blockIdx.x * 4 + (threadIdx.x >> 5) + chain_begin(); t < n; t += gridDim.x * 4) {
        hop_fix_task<DAG>(a, e, t, threadIdx.x & 31);
        __syncwarp();   // lanes past the last site rejoin
    }
}

// blocks_per_sm > 0: the looping form.
template <bool DAG>
void launch_k_hop_fix(const HopArgs &a, const EpiStore &e, int blocks_per_sm, cudaStream_t s)
{
    if (blocks_per_sm > 0) launch_chained(k_hop_fix_gs<DAG>, blocks_per_sm * sm_count(), 128, s, a, e);
    else launch_chained(k_hop_fix<DAG>, (fix_tasks(a) + 3) / 4, 128, s, a, e);
}

// The same with ||out_r||^2 into norms[r] for the rhs that are not skipped:
// the residual hop of an outer check and its norm in one pass (the norm's own
// pass reads the residual again: 294 us of 3.2 ms, 12 rhs on 24^3x64).  Blocks of
// 64 sites of one rhs.
template <bool DAG>
__global__ void __launch_bounds__(128, 4) k_hop_fix_norm(HopArgs a, EpiStore e, double *norms, double *partials,
                                                         unsigned *tickets)
{
    const int z = chain_begin();
    const int r = blockIdx.x % a.nrhs + z, sb = blockIdx.x / a.nrhs + z;
    if (rhs_done(a, r)) return;   // uniform over every block of this rhs
    const int lane = threadIdx.x & 31, s = lane >> 4;
    const int i0 = sb * 64 + (threadIdx.x >> 5) * 16 + (lane & 15);
    double red[1] = {0.0};
    if (i0 - (lane & 15) < a.g.Vh) {   // the whole warp
        const int i = min(i0, a.g.Vh - 1);
        cx<double> acc[6], o[6];
        hop_half<DAG, false>(a, static_cast<const char *>(a.in) + (size_t)r * a.rhs_bytes, i, s, acc);
        if (i0 < a.g.Vh) {
            half_epilogue(e, a.g.stride, r, s, i, acc, o);
#pragma unroll
            for (int k = 0; k < 6; ++k) red[0] = fma(o[k].re, o[k].re, fma(o[k].im, o[k].im, red[0]));
        }
    }
    double tot[1];
    if (site_sum<1>(red, a.g, partials, r, &tickets[r], sb, gridDim.x / a.nrhs, tot) && threadIdx.x == 0)
        norms[r] = tot[0];
}

// The reduction-fused hop (EpiReduce): blocks of 64 sites of one rhs.
template <bool DAG, int KIND>
__global__ void __launch_bounds__(128, 4) k_hop_fix_reduce(HopArgs a, EpiReduce<KIND> e)
{
    const int z = chain_begin();
    const int r = blockIdx.x % a.nrhs + z, sb = blockIdx.x / a.nrhs + z;
    BiState &st = e.st[r];
    if (__ldcg(&st.done)) return;   // uniform over every block of this rhs
    const int lane = threadIdx.x & 31, s = lane >> 4;
    const int i0 = sb * 64 + (threadIdx.x >> 5) * 16 + (lane & 15);
    const bool active = i0 < a.g.Vh;
    const double coef = e.coef_dev ? __ldcg(e.coef_dev) : e.coef;
    double red[EpiReduce<KIND>::NV] = {0.0, 0.0, 0.0};
    if (i0 - (lane & 15) < a.g.Vh) {   // the whole warp
        const int i = active ? i0 : a.g.Vh - 1;
        cx<double> acc[6];
        hop_half<DAG, false>(a, static_cast<const char *>(a.in) + (size_t)r * a.rhs_bytes, i, s, acc);
        if (active) {
            const size_t off = (size_t)r * e.rhs_bytes;
            cx<double> x[6], o[6];
            half_load(static_cast<const char *>(e.xin) + off, a.g.stride, s, i, x);
#pragma unroll
            for (int k = 0; k < 6; ++k) o[k] = e.a1 * x[k] + coef * acc[k];
            half_store(static_cast<char *>(e.out) + off, a.g.stride, s, i, o);
            cx<double> d = {0.0, 0.0};
            double n = 0.0;
            if constexpr (KIND == 0) {
                cx<double> rh[6];
                half_load(static_cast<const char *>(e.rhat) + off, a.g.stride, s, i, rh);
#pragma unroll
                for (int k = 0; k < 6; ++k) d = conjmad(rh[k], o[k], d);
            } else if constexpr (KIND == 1) {
#pragma unroll
                for (int k = 0; k < 6; ++k) d = conjmad(o[k], x[k], d);
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) n = fma(o[k].re, o[k].re, fma(o[k].im, o[k].im, n));
            red[0] = d.re;
            red[1] = d.im;
            red[2] = n;
        }
    }
    hop_reduce_finish<KIND>(a.g, e, st, r, sb, red);
}

template <bool DAG, int KIND>
void launch_k_hop_fix_reduce(const HopArgs &a, const EpiReduce<KIND> &e, cudaStream_t s)
{
    launch_chained(k_hop_fix_reduce<DAG, KIND>, (a.g.Vh + 63) / 64 * a.nrhs, 128, s, a, e);
}

// ------------------------------------------- canonical operator application
// wilson_dslash in FP64 without the layout passes: the hops read and write
// the canonical fields.
//   STAGE 0: out = add in + coef D in on both parities in one launch
//   STAGE 1: tmp_o = D_oe in_e (internal);  STAGE 2: out_e = in_e + coef D_eo
//   tmp_o, out_o = 0  (M_prec)
struct DslashArgs {
    HopArgs a[2];         // by output parity
    const double2 *in;    // canonical
    double2 *out;         // canonical
    void *tmp;            // internal, odd sites (stages 1, 2)
    double coef;
    int add;
};

// Store of a thread's half of a site, by stage.  active threads only.
template <int STAGE>
__device__ __forceinline__ void dslash_finish(const DslashArgs &d, const HopArgs &a, int i, int s, cx<double> (&acc)[6])
{
    if constexpr (STAGE == 1) {
        half_store(d.tmp, a.g.stride, s, i, acc);
    } else {
        const Coord c = site_coord(a.g, i, a.out_parity);
        const size_t bit = c.x & 1, n = 2 * (size_t)i + bit;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const size_t e = 12 * n + 3 * (h ? 3 - s : s) + k;
                // product, then sum, each rounded: the internal hops' epilogue
                cx<double> o = {__dmul_rn(d.coef, acc[3 * h + k].re), __dmul_rn(d.coef, acc[3 * h + k].im)};
                if (STAGE == 2 || d.add) {
                    const double2 x = d.in[e];
                    o = {__dadd_rn(o.re, x.x), __dadd_rn(o.im, x.y)};
                }
                d.out[e] = make_double2(o.re, o.im);
                if (STAGE == 2) d.out[12 * (n ^ 1) + 3 * (h ? 3 - s : s) + k] = make_double2(0.0, 0.0);
            }
    }
}

template <bool DAG, int STAGE>
__global__ void __launch_bounds__(128, 4) k_dslash_fix(DslashArgs d)
{
    const int lane = threadIdx.x & 31, s = lane >> 4;
    const unsigned task = blockIdx.x * 4 + (threadIdx.x >> 5) + chain_begin();
    const int p = STAGE == 0 ? (int)(task & 1) : STAGE == 1 ? 1 : 0;
    const HopArgs &a = d.a[p];
    const int i0 = (int)(STAGE == 0 ? task >> 1 : task) * 16 + (lane & 15);
    if (i0 - (lane & 15) >= a.g.Vh) return;   // the whole warp
    const int i = min(i0, a.g.Vh - 1);
    cx<double> acc[6];
    hop_half<DAG, STAGE != 2>(a, STAGE == 2 ? d.tmp : static_cast<const void *>(d.in), i, s, acc);
    if (i0 < a.g.Vh) dslash_finish<STAGE>(d, a, i, s, acc);
}

// The same with the four directions of 16 sites on the four warps of a
// block: a quarter of the serial work per thread, for lattices that do not
// fill the GPU.  The warps' sums meet in shared memory.
template <bool DAG, int STAGE>
__global__ void __launch_bounds__(128, 4) k_dslash_fix_split(DslashArgs d)
{
    __shared__ i64 sum[4][12][32];
    __shared__ int exps[4][32];
    const int lane = threadIdx.x & 31, s = lane >> 4, w = threadIdx.x >> 5;
    const unsigned task = blockIdx.x + chain_begin();
    const int p = STAGE == 0 ? (int)(task & 1) : STAGE == 1 ? 1 : 0;
    const HopArgs &a = d.a[p];
    const int i0 = (int)(STAGE == 0 ? task >> 1 : task) * 16 + (lane & 15);
    const int i = min(i0, a.g.Vh - 1);
    const void *in = STAGE == 2 ? d.tmp : static_cast<const void *>(d.in);
    const FixSite q = fix_site(a, i);
    FixAcc A;
    A.clear();
    if (w & 1) fix_direction<DAG, STAGE != 2, false>(a, in, q, w >> 1, s, A);   // y, t
    else fix_direction<DAG, STAGE != 2, true>(a, in, q, w >> 1, s, A);          // x, z
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        sum[w][k][lane] = A.up[k];
        sum[w][6 + k][lane] = A.low[k];
    }
    exps[w][lane] = A.special ? -1 : A.E;
    __syncthreads();
    if (w != 0) return;
    // thread s: spin s from its own sums, spin 3 - s from its own in x, y and
    // from its partner's in z, t
    A.special = false;
    int Ew[4], Eo[4];
    A.E = kFixMinExp;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Ew[k] = exps[k][lane];
        Eo[k] = exps[k][lane ^ 16];
        A.special |= Ew[k] < 0 || Eo[k] < 0;
        A.E = max(A.E, max(Ew[k], Eo[k]));
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        A.up[k] = A.low[k] = 0;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            A.up[k] += fix_sar(sum[v][k][lane], A.E - Ew[v]);
            A.low[k] += fix_sar(sum[v][6 + k][v < 2 ? lane : lane ^ 16], A.E - (v < 2 ? Ew[v] : Eo[v]));
        }
    }
    if (i0 >= a.g.Vh) return;
    cx<double> acc[6];
    fix_values<DAG, STAGE != 2>(a, in, i, s, A, acc);
    dslash_finish<STAGE>(d, a, i, s, acc);
}

template <bool DAG, int STAGE>
cudaError_t launch_dslash_fix(const DslashArgs &d, bool split, cudaStream_t s)
{
    const unsigned chunks = (unsigned)((d.a[0].g.Vh + 15) / 16) * (STAGE == 0 ? 2u : 1u);
    return split ? launch_chained(k_dslash_fix_split<DAG, STAGE>, chunks, 128, s, d)
                 : launch_chained(k_dslash_fix<DAG, STAGE>, (chunks + 3) / 4, 128, s, d);
}

}  // namespace wl
