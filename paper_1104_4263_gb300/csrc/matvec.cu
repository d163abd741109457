// FP64 products: the passes of fx_kernels.cuh for every transform length, and the operator
// views.
#include "fx_launch.cuh"
#include "op.cuh"
#include "prof.cuh"

namespace die {

static FxDev view_d(const dieop_s* op) {
    FxDev v{};
    v.n1 = op->n1; v.n2 = op->n2; v.M1 = op->M1; v.M2 = op->M2; v.Q1 = op->Q1; v.Q2 = op->Q2;
    v.q1 = fx_plan(op->M1).q; v.q2 = fx_plan(op->M2).q;
    v.fx1 = op->fx1; v.fx2 = op->fx2;
    v.gx = op->gx; v.ge = op->ge;
    v.chim = op->chim_d;
    v.planes = op->planes;
    v.apart = op->pol == DIE_TM;
    v.xs = (long)op->planes * op->n1 * op->n2;
    v.ws = (long)op->planes * op->M1 * op->n2;
    return v;
}
OpDev<float> view_f(const dieop_s* op) {
    OpDev<float> v{};
    v.n1 = op->n1; v.n2 = op->n2; v.M1 = op->M1; v.M2 = op->M2; v.Q1 = op->Q1; v.Q2 = op->Q2;
    v.f1 = op->f1; v.i1 = op->i1; v.f2 = op->f2; v.i2 = op->i2;
    v.planes = op->planes;
    v.xs = (long)op->planes * op->n1 * op->n2;
    v.ws = (long)op->planes * op->M1 * op->n2;
    v.tw1 = op->tw1_f; v.tw2 = op->tw2_f; v.gq = op->gq_f;
    v.twx1 = op->tw1_f + op->M1; v.twx2 = op->tw2_f + op->M2;
    v.gx1 = op->tw1_f + 3 * (size_t)op->M1; v.gx2 = op->tw2_f + 3 * (size_t)op->M2;
    v.tr = op->tile_rows_c64;
    v.chim = op->chim_f;
    return v;
}

// Calls f with the launchers of a transform length.
template <typename F> static void fx_for_length(int L, F&& f) {
    switch (L) {
        case 16: f(FxLaunch2<16>{}); return;
        case 32: f(FxLaunch2<32>{}); return;
        case 64: f(FxLaunch2<64>{}); return;
        case 128: f(FxLaunch2<128>{}); return;
        case 256: f(FxLaunch2<256>{}); return;
        case 512: f(FxLaunch2<512>{}); return;
        case 1024: f(FxLaunch2<1024>{}); return;
        case 2048: f(FxLaunch2<2048>{}); return;
        case 4096: f(FxLaunch2<4096>{}); return;
        case 48: f(FxLaunch2<48>{}); return;
        case 96: f(FxLaunch2<96>{}); return;
        case 192: f(FxLaunch2<192>{}); return;
        case 384: f(FxLaunch2<384>{}); return;
        case 768: f(FxLaunch2<768>{}); return;
        case 1536: f(FxLaunch2<1536>{}); return;
        default: break;
    }
    if (fx_plan(L).r0 == 6) f(FxLaunch3<6>{});
    else f(FxLaunch3<12>{});
}

static const double2* chi_of(const dieop_s* op, Contrast c) { return c == Contrast::Chi ? op->chi_d : op->chir_d; }

// nb products (reg: A(chi') A(chi), else A(contrast)) over consecutive vectors.
static die_status fx_product(dieop_s* op, bool reg, Contrast which, const double2* x, double2* y, double2* W,
                             double2* vb, const int* skip, cudaStream_t st, int nb, const FxNormalise& nrm = {}) {
    const FxDev v = view_d(op);
    const double2* chi = chi_of(op, reg ? Contrast::Chi : which);
    auto cols = [&] {
        DIE_PROF(PK_COLS, st, fx_for_length(v.M2, [&](auto l) { l.k2(v, W, skip, st, nb); }));
    };
    DIE_PROF(PK_ROWS_FWD, st, fx_for_length(v.M1, [&](auto l) { l.k1(v, x, chi, W, nrm, skip, st, nb); }));
    cols();
    if (reg) {
        DIE_PROF(PK_ROWS_INV_FWD, st,
                 fx_for_length(v.M1, [&](auto l) { l.k3k1(v, W, x, chi_of(op, Contrast::ChiReg), vb, skip, st, nb); }));
        cols();
    }
    DIE_PROF(PK_ROWS_INV, st, fx_for_length(v.M1, [&](auto l) { l.k3(v, W, reg ? vb : x, y, skip, st, nb); }));
    DIE_LAUNCH_CHECK();
    return DIE_OK;
}

template <>
die_status apply_op_skip<double, double2>(dieop_s* op, Contrast which, const double2* x, double2* y, const int* skip,
                                          cudaStream_t st, const Workspace* ws) {
    if (!ws) ws = &op->ws;
    return fx_product(op, false, which, x, y, (double2*)ws->W, nullptr, skip, st, 1);
}
template <>
die_status apply_reg_skip<double, double2>(dieop_s* op, const double2* x, double2* y, const int* skip,
                                           cudaStream_t st, const Workspace* ws) {
    if (!ws) ws = &op->ws;
    return fx_product(op, true, Contrast::Chi, x, y, (double2*)ws->W, (double2*)ws->v, skip, st, 1);
}
die_status apply_normalised(dieop_s* op, bool reg, double2* x, const double* inv, double* xm, double2* y,
                            const int* skip, cudaStream_t st, const Workspace* ws) {
    if (!ws) ws = &op->ws;
    return fx_product(op, reg, Contrast::Chi, x, y, (double2*)ws->W, (double2*)ws->v, skip, st, 1, {x, inv, xm});
}
template <>
die_status apply_op<double, double2>(dieop_s* op, Contrast c, const double2* x, double2* y, cudaStream_t st,
                                     const Workspace* ws) {
    return apply_op_skip<double, double2>(op, c, x, y, nullptr, st, ws);
}
template <>
die_status apply_reg<double, double2>(dieop_s* op, const double2* x, double2* y, cudaStream_t st,
                                      const Workspace* ws) {
    return apply_reg_skip<double, double2>(op, x, y, nullptr, st, ws);
}
template <>
die_status apply_batch<double, double2>(dieop_s* op, bool reg, const double2* x, double2* y, int nb, void* Wws,
                                        void* vws, cudaStream_t st) {
    return fx_product(op, reg, Contrast::Chi, x, y, (double2*)Wws, (double2*)vws, nullptr, st, nb);
}

}  // namespace die
