// Host dispatch of the hop kernels and the dslash entry points of the C ABI.
#include "hop.cuh"

namespace wl {

// ------------------------------------------------------------------ launch

static const void *links_of(wl_gauge *g, int prec, int parity) { return g->links[prec_index(prec)][parity]; }

// SM count of the current device (grid-stride launches).
int sm_count()
{
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
        v > 0)
        return v;
    return 1;
}

static int check_links(wl_gauge *g, int prec)
{
    if (!(g->prec_mask & prec) || !links_of(g, prec, 0)) {
        set_error("gauge handle holds no links of the requested precision");
        return WL_ERR_ARG;
    }
    return WL_OK;
}

// Arguments of a hop from in to sites of parity out_parity.
static HopArgs hop_args(wl_gauge *g, const Vec &in, int out_parity)
{
    HopArgs a;
    a.g = g->lat->geom;
    a.out_parity = out_parity;
    a.nrhs = in.nrhs;
    a.ngroups = in.nrhs;
    a.in = in.ptr;
    a.rhs_bytes = in.rhs_bytes;
    a.links_out = links_of(g, in.prec, out_parity);
    a.links_in = links_of(g, in.prec, 1 - out_parity);
    a.fix_out = g->fix_links[out_parity];
    a.fix_in = g->fix_links[1 - out_parity];
    a.skip = nullptr;
    a.skip_stride = 0;
    return a;
}

int hop_ex(wl_gauge *g, const Vec &in, const Vec &out, const Vec *x1, double a1, const Vec *x2, double a2,
           double coef, int out_parity, int dagger, int rhs_block, const int *skip, int skip_stride, cudaStream_t s,
           const Vec *out_raw, const NormOut *norm)
{
    WL_TRY(check_links(g, in.prec));
    if (in.prec != out.prec || (x1 && x1->prec != in.prec) || (x2 && x2->prec != in.prec)) {
        set_error("hop: precision mismatch");
        return WL_ERR_ARG;
    }
    HopArgs a = hop_args(g, in, out_parity);
    a.skip = skip;
    a.skip_stride = skip_stride;
    EpiStore e;
    e.out = out.ptr;
    e.out_raw = out_raw ? out_raw->ptr : nullptr;
    e.x1 = x1 ? x1->ptr : nullptr;
    e.x2 = x2 ? x2->ptr : nullptr;
    e.a1 = a1;
    e.a2 = a2;
    e.coef = coef;
    e.rhs_bytes = out.rhs_bytes;
    if (out.rhs_bytes != in.rhs_bytes) { set_error("hop: rhs stride mismatch"); return WL_ERR_ARG; }
    const int variant = hop_variant_for(g, in.prec, in.nrhs, rhs_block);
    if (norm && variant == 6000 && !dagger) {
        WL_TRY(hop_fix_norm_launch(a, e, norm->norms, norm->partials, norm->tickets, s));
        note_launch(s);
        return WL_OK;
    }
    int st = WL_ERR_ARG;
    switch (in.prec) {
    case WL_F64: st = hop_launch_prec<WL_F64>(variant, dagger, a, e, s); break;
    case WL_F32: st = hop_launch_prec<WL_F32>(variant, dagger, a, e, s); break;
    case WL_F16: st = hop_launch_prec<WL_F16>(variant, dagger, a, e, s); break;
    case WL_DF: st = hop_launch_prec<WL_DF>(variant, dagger, a, e, s); break;
    default: set_error("hop: bad precision"); return WL_ERR_ARG;
    }
    if (st == WL_VARIANT_NA) return WL_ERR_ARG;
    WL_TRY(st);
    WL_CUDA_TRY(cudaGetLastError());
    note_launch(s);
    if (norm) return blas_norm2(a.g, out, norm->norms, norm->partials, norm->tickets, s);
    return WL_OK;
}

int hop(wl_gauge *g, const Vec &in, const Vec &out, const Vec *x, double coef, int out_parity, int dagger,
        int rhs_block, cudaStream_t s)
{
    return hop_ex(g, in, out, x, 1.0, nullptr, 0.0, coef, out_parity, dagger, rhs_block, nullptr, 0, s);
}

// Blocks of a reduction-fused hop over one parity: 128 sites each, 64 in the
// fixed-point FP64 hop (two threads per site).
static int reduce_blocks(const wl_gauge *g, int prec)
{
    const Geom &geo = g->lat->geom;
    return prec == WL_F64 && g->fixed_point() ? (geo.Vh + 63) / 64 : site_blocks(geo);
}

template <int KIND>
static int hop_reduce_k(wl_gauge *g, const Vec &tmp, const Vec &xin, double a1, const Vec &out, const Vec &rhat,
                        double coef, const double *coef_dev, int out_parity, int dagger, BiState *state,
                        double *partials, int part, int parts, cudaStream_t s)
{
    WL_TRY(check_links(g, tmp.prec));
    HopArgs a = hop_args(g, tmp, out_parity);
    if (!g->fixed_point()) a.fix_out = a.fix_in = nullptr;   // (hop_reduce_launch_prec)
    a.skip = &state[0].done;
    a.skip_stride = sizeof(BiState) / sizeof(int);
    EpiReduce<KIND> e;
    e.out = out.ptr;
    e.xin = xin.ptr;
    e.rhat = rhat.ptr;
    e.a1 = a1;
    e.coef = coef;
    e.coef_dev = coef_dev;
    const int nblk = reduce_blocks(g, tmp.prec);
    e.blk_off = part * nblk;
    e.blk_total = parts * nblk;
    e.rhs_bytes = out.rhs_bytes;
    e.st = state;
    e.partials = partials;
    int st = WL_ERR_ARG;
    switch (tmp.prec) {
    case WL_F64: st = hop_reduce_launch_prec<WL_F64>(KIND, dagger, a, &e, s); break;
    case WL_F32: st = hop_reduce_launch_prec<WL_F32>(KIND, dagger, a, &e, s); break;
    case WL_F16: st = hop_reduce_launch_prec<WL_F16>(KIND, dagger, a, &e, s); break;
    case WL_DF: st = hop_reduce_launch_prec<WL_DF>(KIND, dagger, a, &e, s); break;
    default: set_error("hop_reduce: bad precision"); return WL_ERR_ARG;
    }
    WL_TRY(st);
    WL_CUDA_TRY(cudaGetLastError());
    note_launch(s);
    return WL_OK;
}

int hop_reduce(wl_gauge *g, int kind, const Vec &tmp, const Vec &xin, double a1, const Vec &out, const Vec &rhat,
               double coef, const double *coef_dev, int out_parity, int dagger, BiState *state, double *partials,
               int part, int parts, cudaStream_t s)
{
    switch (kind) {
    case 0: return hop_reduce_k<0>(g, tmp, xin, a1, out, rhat, coef, coef_dev, out_parity, dagger, state, partials,
                                   part, parts, s);
    case 1: return hop_reduce_k<1>(g, tmp, xin, a1, out, rhat, coef, coef_dev, out_parity, dagger, state, partials,
                                   part, parts, s);
    case 2: return hop_reduce_k<2>(g, tmp, xin, a1, out, rhat, coef, coef_dev, out_parity, dagger, state, partials,
                                   part, parts, s);
    case 3: return hop_reduce_k<3>(g, tmp, xin, a1, out, rhat, coef, coef_dev, out_parity, dagger, state, partials,
                                   part, parts, s);
    default: set_error("hop_reduce: bad kind"); return WL_ERR_ARG;
    }
}

}  // namespace wl

using namespace wl;

// ---------------------------------------------------------------- C ABI

// In the bounds-checked build the dslash calls synchronise the stream and
// report a recorded out-of-range index.
static int dslash_checked(int st, void *stream)
{
#ifdef WL_CHECKED
    if (st == WL_OK) WL_CUDA_TRY(cudaStreamSynchronize(as_stream(stream)));
    return checked_result(st);
#else
    (void)stream;
    return st;
#endif
}

extern "C" int wilson_hop(wl_gauge *g, const void *in, void *out, const void *x, double coef, int prec,
                          int out_parity, int dagger, void *stream)
{
    if (!g || !in || !out || !valid_prec(prec) || (out_parity != 0 && out_parity != 1) || in == out) {
        set_error("wilson_hop: bad argument");
        return WL_ERR_ARG;
    }
    Vec vi, vo, vx;
    vi.ptr = const_cast<void *>(in);
    vi.prec = vo.prec = vx.prec = prec;
    vi.rhs_bytes = vo.rhs_bytes = vx.rhs_bytes = spinor_bytes(g->lat->geom, prec);
    vo.ptr = out;
    vx.ptr = const_cast<void *>(x);
    std::lock_guard<std::mutex> lock(g->hop_mu);
    const int st = hop(g, vi, vo, x ? &vx : nullptr, coef, out_parity, dagger ? 1 : 0, 1, as_stream(stream));
    note_link_use(g, prec);
    return dslash_checked(st, stream);
}

extern "C" int wilson_hop_multi(wl_gauge *g, const void *in, void *out, const void *x, double coef, int prec,
                                int out_parity, int dagger, int n_rhs, size_t rhs_stride, int rhs_block,
                                void *stream)
{
    bool known_variant = rhs_block >= 0;
    if (rhs_block < 0 && valid_prec(prec))
        for (int v : hop_variants(prec)) known_variant |= (v == -rhs_block);
    if (!g || !in || !out || !valid_prec(prec) || (out_parity != 0 && out_parity != 1) || in == out || n_rhs < 1 ||
        !known_variant || rhs_block > 4 || rhs_block == 3 || (rhs_stride & 255) ||
        rhs_stride < spinor_bytes(g->lat->geom, prec)) {
        set_error("wilson_hop_multi: bad argument");
        return WL_ERR_ARG;
    }
    Vec vi, vo, vx;
    vi.ptr = const_cast<void *>(in);
    vo.ptr = out;
    vx.ptr = const_cast<void *>(x);
    vi.prec = vo.prec = vx.prec = prec;
    vi.nrhs = vo.nrhs = vx.nrhs = n_rhs;
    vi.rhs_bytes = vo.rhs_bytes = vx.rhs_bytes = rhs_stride;
    std::lock_guard<std::mutex> lock(g->hop_mu);
    const int st = hop(g, vi, vo, x ? &vx : nullptr, coef, out_parity, dagger ? 1 : 0, rhs_block, as_stream(stream));
    note_link_use(g, prec);
    return dslash_checked(st, stream);
}

namespace wl {

static bool device_fields(const void *in, const void *out);

// FP64 operator applications read and write the canonical fields in the hop
// itself (8^4 28.5 -> 8.9 us, 24^3x64 612 -> 499 us).  Page-locked host fields
// keep the layout passes, which read each site over the host link once.
bool dslash_direct(const wl_gauge *g, const void *in, const void *out, int prec)
{
    return prec == WL_F64 && g->fixed_point() && device_fields(in, out);
}

static bool device_fields(const void *in, const void *out)
{
    for (const void *p : {in, out}) {
        cudaPointerAttributes pa{};
        if (cudaPointerGetAttributes(&pa, p) != cudaSuccess || pa.type != cudaMemoryTypeDevice) {
            (void)cudaGetLastError();
            return false;
        }
    }
    return true;
}

}  // namespace wl

// FP32, FP16 and double-float: whether the last hop stores to the canonical
// field (device memory).  D and M, both parities in one launch, gain at every
// size (FP32 8^4 15.2 -> 12.0 us, 16^4 28.7 -> 18.0, 24^3x64 211 -> 167; DF
// 24^3x64 786 -> 619); M_prec, one parity after another, on lattices of up to
// 16384 sites of one parity, in double-float 8192 (us, layout passes ->
// canonical store, 8192 / 12288 / 16384 / 24576 / 32768 sites: FP32 16.8 ->
// 14.7, 18.6 -> 17.4, 18.6 -> 18.3, 22.6 -> 22.1, 26.7 -> 29.2; FP16 16.8 ->
// 13.9, 18.6 -> 16.5, 18.7 -> 17.8, 22.5 -> 19.6, 24.8 -> 30.8; DF 45.1 ->
// 44.5, 51.3 -> 52.1, 53.3 -> 59.4, 65.9 -> 73.4, 75.8 -> 83.4).
constexpr int canon_prec_sites(int prec) { return prec == WL_DF ? 8192 : 16384; }

static int dslash_common(wl_gauge *g, const void *in, void *out, double kappa, int prec, int op, int dagger,
                         void *stream)
{
    if (!g || !in || !out || in == out || !valid_prec(prec) || op < WL_OP_HOP || op > WL_OP_MPREC) {
        set_error("wilson_dslash: bad argument");
        return WL_ERR_ARG;
    }
    WL_TRY(check_links(g, prec));
    std::lock_guard<std::mutex> lock(g->mu);
    cudaStream_t s = as_stream(stream);
    const Geom &geo = g->lat->geom;
    Vec ie, io, oe, oo;
    // (an allocation may release the integer links: it comes before the choice)
    if (op == WL_OP_MPREC) WL_TRY(make_vec(g, "dslash_oo", prec, 1, &oo));
    if (dslash_direct(g, in, out, prec)) {
        const int st = dslash_fix(g, in, out, kappa, op, dagger, oo.ptr, s);
        note_link_use(g, prec);
        return st;
    }
    WL_TRY(make_vec(g, "dslash_ie", prec, 1, &ie));
    WL_TRY(make_vec(g, "dslash_io", prec, 1, &io));
    const bool canon = prec != WL_F64 && (op != WL_OP_MPREC || geo.Vh <= canon_prec_sites(prec)) && device_fields(in, out);
    if (!canon) {
        WL_TRY(make_vec(g, "dslash_oe", prec, 1, &oe));
        WL_TRY(make_vec(g, "dslash_oo", prec, 1, &oo));
    }
    const void *cin[1] = {in};
    void *cout[1] = {out};
    WL_TRY(import_full(geo, cin, ie, io, s));
    if (canon) {
        CanonHop h{};
        for (int p = 0; p < 2; ++p) {
            h.a[p] = hop_args(g, op == WL_OP_MPREC ? oo : p ? ie : io, p);
            if (op != WL_OP_HOP) h.x[p] = p ? io.ptr : ie.ptr;
        }
        h.a1 = 1.0;
        h.coef = op == WL_OP_HOP ? 1.0 : op == WL_OP_M ? -kappa : -kappa * kappa;
        h.out = static_cast<double2 *>(out);
        h.both = op != WL_OP_MPREC;
        if (op == WL_OP_MPREC) WL_TRY(hop(g, ie, oo, nullptr, 1.0, WL_ODD, dagger, 1, s));
        switch (prec) {
        case WL_F32: return hop_canon_launch_prec<WL_F32>(dagger, h, s);
        case WL_F16: return hop_canon_launch_prec<WL_F16>(dagger, h, s);
        default: return hop_canon_launch_prec<WL_DF>(dagger, h, s);
        }
    }
    if (op == WL_OP_HOP) {
        WL_TRY(hop(g, io, oe, nullptr, 1.0, WL_EVEN, dagger, 1, s));
        WL_TRY(hop(g, ie, oo, nullptr, 1.0, WL_ODD, dagger, 1, s));
    } else if (op == WL_OP_M) {
        WL_TRY(hop(g, io, oe, &ie, -kappa, WL_EVEN, dagger, 1, s));
        WL_TRY(hop(g, ie, oo, &io, -kappa, WL_ODD, dagger, 1, s));
    } else {
        // out_e = in_e - kappa^2 D_eo D_oe in_e.  With dagger hops this is
        // 1 - kappa^2 g5 D_eo D_oe g5 = M_prec^dag.
        WL_TRY(hop(g, ie, oo, nullptr, 1.0, WL_ODD, dagger, 1, s));
        WL_TRY(hop(g, oo, oe, &ie, -kappa * kappa, WL_EVEN, dagger, 1, s));
        WL_CUDA_TRY(cudaMemsetAsync(oo.ptr, 0, spinor_bytes(geo, prec), s));
    }
    WL_TRY(export_full(geo, oe, oo, cout, s));
    note_link_use(g, prec);
    return WL_OK;
}

extern "C" int wilson_dslash(wl_gauge *g, const void *in, void *out, double kappa, int prec, int op, void *stream)
{
    return dslash_checked(dslash_common(g, in, out, kappa, prec, op, 0, stream), stream);
}

extern "C" int wilson_dslash_dag(wl_gauge *g, const void *in, void *out, double kappa, int prec, int op,
                                 void *stream)
{
    return dslash_checked(dslash_common(g, in, out, kappa, prec, op, 1, stream), stream);
}
