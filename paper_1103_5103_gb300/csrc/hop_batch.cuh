// FP32 and FP16 hops with their loads issued a transporter ahead (device
// code): the link and the spinor of direction d + 1 are requested, as raw
// words, before direction d is computed.  The loads are volatile, so they
// stay in this order; left to the compiler they sink towards their uses.
//
// FP32 at 128 registers (four blocks per SM): 12 rhs on 24^3x64 386 -> 376 us,
// 1 rhs 51.0 -> 49.3 us, 16^3x32 10.4 -> 9.8 us against the best of the other
// kernels.  What bounds it on the large lattices is the latency of loads from
// L2 under their own traffic: 4.5 GB from L2 to L1 in 0.38 ms, 11.8 TB/s,
// where a plain read of 64 MB out of L2 reaches 14.5 TB/s (L2 to crossbar 43%
// and 60% busy), with long-scoreboard stalls ahead of all others.  Sharing
// links between rhs in neighbouring warps (L1 hits 19 -> 43%) and other depths
// and occupancies ended within 5%.
#pragma once

#include "hop.cuh"

namespace wl {

// Links through the read-only path, fields through coherent loads (ld_field in
// common.cuh says why).
__device__ __forceinline__ float4 ldv4_link(const void *p)
{
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ldv4_field(const void *p)
{
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint4 ldvu4_field(const void *p)
{
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned ldvu_field(const void *p)
{
    unsigned v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 ldvu2_link(const void *p)
{
    uint2 v;
    asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned ldvu_link(const void *p)
{
    unsigned v;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// The raw words of one transporter's link and neighbour spinor; get() unpacks
// them and returns the spinor's scale.
template <int P> struct RawDir;
template <> struct RawDir<WL_F32> {
    float4 u[3], s[6];
    __device__ __forceinline__ void load(const char *lk, const char *sp, int stride, int li, int j)
    {
        const float4 *l = reinterpret_cast<const float4 *>(lk) + WL_LOAD_IDX(li, stride, 3);
        const float4 *q = reinterpret_cast<const float4 *>(sp) + WL_LOAD_IDX(j, stride, 1);
#pragma unroll
        for (int k = 0; k < 3; ++k) u[k] = ldv4_link(l + (size_t)k * stride);
#pragma unroll
        for (int k = 0; k < 6; ++k) s[k] = ldv4_field(q + (size_t)k * stride);
    }
    __device__ __forceinline__ float get(cx<float> (&U)[9], cx<float> (&psi)[12]) const
    {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            U[2 * k] = {u[k].x, u[k].y};
            U[2 * k + 1] = {u[k].z, u[k].w};
        }
        reconstruct_row2(U);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            psi[2 * k] = {s[k].x, s[k].y};
            psi[2 * k + 1] = {s[k].z, s[k].w};
        }
        return 1.f;
    }
};
template <> struct RawDir<WL_F16> {
    uint2 u[4];
    unsigned u8;
    uint4 s[3];
    unsigned n;
    __device__ __forceinline__ void load(const char *lk, const char *sp, int stride, int li, int j)
    {
        li = WL_LOAD_IDX(li, stride, 3);
        j = WL_LOAD_IDX(j, stride, 1);
        const uint2 *l = reinterpret_cast<const uint2 *>(lk) + li;
        const uint4 *q = reinterpret_cast<const uint4 *>(sp) + j;
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = ldvu2_link(l + (size_t)k * stride);
        u8 = ldvu_link(reinterpret_cast<const unsigned *>(reinterpret_cast<const uint2 *>(lk) + (size_t)4 * stride) + li);
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k] = ldvu4_field(q + (size_t)k * stride);
        n = ldvu_field(SpinorIO<WL_F16>::norms(sp, stride) + j);
    }
    __device__ __forceinline__ float get(cx<float> (&U)[9], cx<float> (&psi)[12]) const
    {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 a = unpack_half2(u[k].x), b = unpack_half2(u[k].y);
            U[2 * k] = {a.x, a.y};
            U[2 * k + 1] = {b.x, b.y};
        }
        const float2 c = unpack_half2(u8);
        U[8] = {c.x, c.y};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float2 a = unpack_half2(s[k].x), b = unpack_half2(s[k].y), d = unpack_half2(s[k].z), e = unpack_half2(s[k].w);
            psi[4 * k + 0] = {a.x, a.y};
            psi[4 * k + 1] = {b.x, b.y};
            psi[4 * k + 2] = {d.x, d.y};
            psi[4 * k + 3] = {e.x, e.y};
        }
        return __uint_as_float(n);
    }
};

template <int P, int D>
__device__ __forceinline__ void batch_load(RawDir<P> &x, const HopArgs &a, const char *in, int i, const int (&nb)[8])
{
    constexpr int MU = D >> 1;
    constexpr bool FWD = (D & 1) == 0;
    const char *lk = static_cast<const char *>(FWD ? a.links_out : a.links_in) + (size_t)MU * link_dir_bytes(P, a.g.stride);
    x.load(lk, in, a.g.stride, FWD ? i : nb[D], nb[D]);
}
template <int P, bool DAG, int D>
__device__ __forceinline__ void batch_compute(const RawDir<P> &x, bool neg, cx<float> (&acc)[12])
{
    constexpr int MU = D >> 1;
    constexpr bool FWD = (D & 1) == 0;
    cx<float> U[9], psi[12];
    const float n = x.get(U, psi);
    if constexpr (FWD) transport<MU, DAG ? 1 : 0, false>(acc, psi, U, neg ? -n : n);
    else transport<MU, DAG ? 0 : 1, true>(acc, psi, U, neg ? -n : n);
}

// acc += D in at site i (in: the rhs's first spinor).
template <int P, bool DAG>
__device__ __forceinline__ void hop_accumulate_batch(const HopArgs &a, const void *base, int i, cx<float> (&acc)[12])
{
    const char *in = static_cast<const char *>(base);
    const Geom &g = a.g;
    const Coord c = site_coord(g, i, a.out_parity);
    const int rowbase = i - (c.x >> 1);
    int nb[8];
    bool f0, f1, nf, nbk;
    neighbours<0>(g, i, c, rowbase, nb[0], nb[1], f0, f1);
    neighbours<1>(g, i, c, rowbase, nb[2], nb[3], f0, f1);
    neighbours<2>(g, i, c, rowbase, nb[4], nb[5], f0, f1);
    neighbours<3>(g, i, c, rowbase, nb[6], nb[7], nf, nbk);
    RawDir<P> x, y;
    batch_load<P, 0>(x, a, in, i, nb);
    batch_load<P, 1>(y, a, in, i, nb);
    batch_compute<P, DAG, 0>(x, false, acc);
    batch_load<P, 2>(x, a, in, i, nb);
    batch_compute<P, DAG, 1>(y, false, acc);
    batch_load<P, 3>(y, a, in, i, nb);
    batch_compute<P, DAG, 2>(x, false, acc);
    batch_load<P, 4>(x, a, in, i, nb);
    batch_compute<P, DAG, 3>(y, false, acc);
    batch_load<P, 5>(y, a, in, i, nb);
    batch_compute<P, DAG, 4>(x, false, acc);
    batch_load<P, 6>(x, a, in, i, nb);
    batch_compute<P, DAG, 5>(y, false, acc);
    batch_load<P, 7>(y, a, in, i, nb);
    batch_compute<P, DAG, 6>(x, nf, acc);
    batch_compute<P, DAG, 7>(y, nbk, acc);
}

template <int P, bool DAG, int MINB>
__global__ void __launch_bounds__(128, MINB) k_hop_batch(HopArgs a, EpiStore epi)
{
    const int z = chain_begin();
    const int r = blockIdx.x % a.nrhs + z;
    const int i = (blockIdx.x / a.nrhs) * 128 + threadIdx.x + z;
    if (i >= a.g.Vh || rhs_done(a, r)) return;
    cx<float> acc[1][12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[0][k] = acc_zero<float>();
    hop_accumulate_batch<P, DAG>(a, static_cast<const char *>(a.in) + (size_t)r * a.rhs_bytes, i, acc[0]);
    epi.template operator()<P, 1>(a, i, true, r, acc);
}

template <int P, bool DAG, int MINB>
void launch_k_hop_batch(const HopArgs &a, const EpiStore &e, cudaStream_t s)
{
    launch_chained(k_hop_batch<P, DAG, MINB>, (a.g.Vh + 127) / 128 * a.nrhs, 128, s, a, e);
}

}  // namespace wl
