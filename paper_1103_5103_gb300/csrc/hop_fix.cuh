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
//  - Error: a few units of 2^(E-56) per output component, where one FP64
//    rounding of a value of the neighbours' size is 2^(E-53): the result is
//    closer to the exact sum than that of eight FP64 transporters.
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

// Loads that stay where they are written, ahead of the arithmetic.
__device__ __forceinline__ int4 fix_ld(const int4 *p)
{
    int4 v;
    asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 fix_ld(const double2 *p)
{
    double2 v;
    asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
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

__device__ __forceinline__ void fix_load(FixRaw &x, const void *in, int j, unsigned off_u, unsigned off_l, int stride)
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
        for (int k = 0; k < 3; ++k) u[3 * r + k] = fix_ld(p + (r * row + k * col));
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

// D in at site i by its two threads: thread s gets spin s in acc[0..2] and
// spin 3 - s in acc[3..5].  Every lane of the warp takes part.
template <bool DAG>
__device__ __forceinline__ void hop_half(const HopArgs &a, const void *in, int i, int s, cx<double> (&acc)[6])
{
    const Geom &g = a.g;
    const Coord q = site_coord(g, i, a.out_parity);
    const int rowbase = i - (q.x >> 1);
    int nb[8];
    bool f0, f1, nf, nbk;
    neighbours<0>(g, i, q, rowbase, nb[0], nb[1], f0, f1);
    neighbours<1>(g, i, q, rowbase, nb[2], nb[3], f0, f1);
    neighbours<2>(g, i, q, rowbase, nb[4], nb[5], f0, f1);
    neighbours<3>(g, i, q, rowbase, nb[6], nb[7], nf, nbk);
#pragma unroll
    for (int k = 0; k < 8; ++k) nb[k] = WL_LOAD_IDX(nb[k], g.stride, 1);
    const int il = WL_LOAD_IDX(i, g.stride, 3);
    bool special = false;
    int E = kFixMinExp;
    // spin s, and the spin coupled to it: 3 - s in x and y, 2 + s in z and t
    i64 up[6], low[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) up[k] = low[k] = 0;
    const int4 *lo = static_cast<const int4 *>(a.fix_out), *li = static_cast<const int4 *>(a.fix_in);
    constexpr int PF = DAG ? -1 : 0;   // 1 + gamma in the forward hops of the adjoint
    const unsigned off_u = (unsigned)(3 * s * g.stride);
    unsigned off_l = (unsigned)(3 * (3 - s) * g.stride);
#pragma unroll 1
    for (int m = 0; m < 2; ++m) {   // x, y, then z, t
        // signs of the phase of spin s in 1 - gamma: x (+, +), z (+, -); y (-, +), t (+, +)
        const int fx = (m ? -s : 0) ^ PF, fy = (m ? 0 : s - 1) ^ PF;
        FixRaw x;
        int4 u[9];
#pragma unroll 1
        for (int cj = 0; cj >= -1; --cj) {   // forward, backward
            const int j = m ? (cj ? nb[5] : nb[4]) : (cj ? nb[1] : nb[0]);
            fix_load(x, in, j, off_u, off_l, g.stride);
            fix_load_link(u, (cj ? li : lo) + fix_link(g, 2 * m, cj ? j : il), cj);
            fix_transport<true>(x, u, fx ^ cj, cj, false, E, special, up, low);
        }
#pragma unroll 1
        for (int cj = 0; cj >= -1; --cj) {
            const int j = m ? (cj ? nb[7] : nb[6]) : (cj ? nb[3] : nb[2]);
            fix_load(x, in, j, off_u, off_l, g.stride);
            fix_load_link(u, (cj ? li : lo) + fix_link(g, 1 + 2 * m, cj ? j : il), cj);
            fix_transport<false>(x, u, fy ^ cj, cj, m && (cj ? nbk : nf), E, special, up, low);
        }
        off_l = (unsigned)(3 * (2 + s) * g.stride);
        // the pair moves to the larger of its two scales and exchanges the
        // lower spins: after x, y thread s holds spin 3 - s and goes on with
        // 2 + s; after z, t it gets 3 - s back
        const int Eo = __shfl_xor_sync(0xffffffffu, E, 16);
        const int sh = max(0, Eo - E);
        E = max(E, Eo);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            up[k] = fix_sar(up[k], sh);
            low[k] = __shfl_xor_sync(0xffffffffu, fix_sar(low[k], sh), 16);
        }
    }
    special = __shfl_xor_sync(0xffffffffu, special ? 1 : 0, 16) || special;
    if (!special) {
        const double scale = __hiloint2double((E + 2 - kFixFrac) << 20, 0);   // 2^(E - 1023 - 56)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            acc[k] = {fix_out(up[2 * k], scale), fix_out(up[2 * k + 1], scale)};
            acc[3 + k] = {fix_out(low[2 * k], scale), fix_out(low[2 * k + 1], scale)};
        }
    } else {
        HopArgs b = a;
        b.in = in;
        cx<double> full[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) full[k] = acc_zero<double>();
        hop_accumulate_rolled<WL_F64, DAG>(b, i, full);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            acc[k] = s ? full[3 + k] : full[k];
            acc[3 + k] = s ? full[6 + k] : full[9 + k];
        }
    }
}

// Load and store of a thread's half of a site: spins s and 3 - s.
__device__ __forceinline__ void half_load(const void *base, int stride, int s, int i, cx<double> (&v)[6])
{
    i = WL_LOAD_IDX(i, stride, 1);
    const double2 *p = static_cast<const double2 *>(base) + i;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double2 x = __ldg(p + (size_t)(3 * s + k) * stride), y = __ldg(p + (size_t)(3 * (3 - s) + k) * stride);
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
    cx<double> acc[6];
    hop_half<DAG>(a, static_cast<const char *>(a.in) + (size_t)r * a.rhs_bytes, i, s, acc);
    if (!active) return;
    const size_t off = (size_t)r * e.rhs_bytes;
    if (e.out_raw) half_store(static_cast<char *>(e.out_raw) + off, a.g.stride, s, i, acc);
    cx<double> o[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) o[k] = e.coef * acc[k];
    if (e.x1) {
        cx<double> x[6];
        half_load(static_cast<const char *>(e.x1) + off, a.g.stride, s, i, x);
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = o[k] + e.a1 * x[k];
    }
    if (e.x2) {
        cx<double> x[6];
        half_load(static_cast<const char *>(e.x2) + off, a.g.stride, s, i, x);
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = o[k] + e.a2 * x[k];
    }
    half_store(static_cast<char *>(e.out) + off, a.g.stride, s, i, o);
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
        hop_half<DAG>(a, static_cast<const char *>(a.in) + (size_t)r * a.rhs_bytes, i, s, acc);
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

}  // namespace wl
