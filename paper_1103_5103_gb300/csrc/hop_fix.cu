// Instantiations of the fixed-point FP64 hop (hop_fix.cuh).
#include "hop_fix.cuh"

namespace wl {

int hop_fix_launch(int dagger, const HopArgs &a, const EpiStore &e, int blocks_per_sm, cudaStream_t s)
{
    if (dagger) launch_k_hop_fix<true>(a, e, blocks_per_sm, s);
    else launch_k_hop_fix<false>(a, e, blocks_per_sm, s);
    WL_CUDA_TRY(cudaGetLastError());
    return WL_OK;
}

int hop_fix_norm_launch(const HopArgs &a, const EpiStore &e, double *norms, double *partials, unsigned *tickets,
                        cudaStream_t s)
{
    WL_CUDA_TRY(launch_chained(k_hop_fix_norm<false>, (unsigned)((a.g.Vh + 63) / 64 * a.nrhs), 128, s, a, e, norms,
                               partials, tickets));
    return WL_OK;
}

template <int KIND>
static void reduce_kind(int dagger, const HopArgs &a, const void *epi, cudaStream_t s)
{
    const auto &e = *static_cast<const EpiReduce<KIND> *>(epi);
    if (dagger) launch_k_hop_fix_reduce<true, KIND>(a, e, s);
    else launch_k_hop_fix_reduce<false, KIND>(a, e, s);
}

int hop_fix_reduce_launch(int kind, int dagger, const HopArgs &a, const void *epi, cudaStream_t s)
{
    switch (kind) {
    case 0: reduce_kind<0>(dagger, a, epi, s); break;
    case 1: reduce_kind<1>(dagger, a, epi, s); break;
    case 2: reduce_kind<2>(dagger, a, epi, s); break;
    default: reduce_kind<3>(dagger, a, epi, s); break;
    }
    WL_CUDA_TRY(cudaGetLastError());
    return WL_OK;
}

// Canonical operator application; tmp: one internal FP64 spinor (M_prec).
int dslash_fix(wl_gauge *g, const void *in, void *out, double kappa, int op, int dagger, void *tmp, cudaStream_t s)
{
    DslashArgs d;
    for (int p = 0; p < 2; ++p) {
        HopArgs &a = d.a[p];
        a = HopArgs{};
        a.g = g->lat->geom;
        a.out_parity = p;
        a.nrhs = a.ngroups = 1;
        a.links_out = g->links[prec_index(WL_F64)][p];
        a.links_in = g->links[prec_index(WL_F64)][1 - p];
        a.fix_out = g->fix_links[p];
        a.fix_in = g->fix_links[1 - p];
    }
    d.in = static_cast<const double2 *>(in);
    d.out = static_cast<double2 *>(out);
    d.tmp = tmp;
    // four warps per 16 sites while the chunks do not fill the SMs: 8^4 8.9
    // against 12.6 us (M), 12.7 against 23.1 (M_prec), 20x12x6x14 M_prec 29.9
    // against 32.2; from two waves on the extra pass through shared memory
    // costs more (16^4 59 against 44)
    const unsigned chunks = (unsigned)((g->lat->geom.Vh + 15) / 16) * (op == WL_OP_MPREC ? 1u : 2u);
    const bool split = chunks <= 5u * (unsigned)sm_count();
    if (op == WL_OP_MPREC) {
        d.coef = -kappa * kappa;
        d.add = 1;
        WL_CUDA_TRY((dagger ? launch_dslash_fix<true, 1>(d, split, s) : launch_dslash_fix<false, 1>(d, split, s)));
        note_launch(s);
        WL_CUDA_TRY((dagger ? launch_dslash_fix<true, 2>(d, split, s) : launch_dslash_fix<false, 2>(d, split, s)));
    } else {
        d.add = op == WL_OP_M;
        d.coef = d.add ? -kappa : 1.0;
        WL_CUDA_TRY((dagger ? launch_dslash_fix<true, 0>(d, split, s) : launch_dslash_fix<false, 0>(d, split, s)));
    }
    note_launch(s);
    return WL_OK;
}

}  // namespace wl
