// Host run of the fixed-point transforms of the FP64 products (fx.cuh): every thread of a
// transform group executes its stages in turn, with the scale rule of the kernels, forward
// on half-zero inputs and inverse (re and im exchanged) on full ones.  Prints
// "L dir kind err" with err the 2-norm error against the plain DFT sum in long double,
// relative to the result, for random, single-value and constant inputs.
#include <cmath>
#include <complex>
#include <cstdio>
#include <vector>

#include "../paper_1104_4263_gb300/csrc/fx.cuh"

using namespace die;
using cl = std::complex<long double>;

template <int EPT, int R0, int R1> double error(int L, bool inv, int kind) {
    const int q = fx_plan(L).q, G = L / EPT;
    const long double tp = 6.283185307179586476925286766559005768L;
    std::vector<fxw> tw(L);
    for (int s = 1, ns = R0; s <= q; s++, ns *= R1)
        for (int r = 1; r < R1; r++)
            for (int k = 0; k < ns; k++) {
                const long double a = tp * (long double)(r * k) / (long double)(ns * R1);
                tw[r * ns + k - 1] = fx_factor(cosl(a), -sinl(a));
            }
    std::vector<double> re(L), im(L);
    unsigned s = 20110421u + L;
    auto rnd = [&] { s = s * 1103515245u + 12345u; return (s >> 8) / 16777216.0 - 0.5; };
    const int nz = inv ? L : L / 2;
    for (int i = 0; i < nz; i++) {
        re[i] = kind == 0 ? rnd() : kind == 1 ? (i == nz / 3 ? 0.7 : 0.0) : 1.0;
        im[i] = kind == 0 ? rnd() : kind == 1 ? (i == nz / 3 ? -0.1 : 0.0) : -1.0;
    }
    double m = 0, sum = 0;
    for (int i = 0; i < L; i++) {
        const double a = std::fabs(re[i]) + std::fabs(im[i]);
        m = std::fmax(m, a);
        sum += a;
    }
    const float lm = (float)std::log2(m), ls = (float)std::log2(sum);
    int e = fx_room(R0, R1, q, !inv, lm, ls, 0), room = e;
    std::vector<fxc> x((size_t)L), buf(padded_len(L));
    using Regs = fxc[EPT];
    auto regs = [&](int t) -> Regs& { return *reinterpret_cast<Regs*>(&x[(size_t)t * EPT]); };
    bool fits = true;
    auto check = [&] {
        for (const fxc& v : x) fits = fits && std::abs(cl(v.x, v.y)) <= ldexpl(1.0L, kFxLimit);
    };
    for (int t = 0; t < G; t++)
        for (int k = 0; k < EPT; k++) {
            const int i = t + fx_slot<EPT, R0>(k) * G;
            const fxc v{llrint(std::ldexp(re[i], e)), llrint(std::ldexp(im[i], e))};
            regs(t)[k] = inv ? fxc{v.y, v.x} : v;
        }
    for (int t = 0; t < G; t++) {
        fx_first<EPT, R0>(regs(t));
        stage_store<fxc, EPT, R0>(buf.data(), regs(t), L, 1, t, G);
    }
    check();
    for (int st = 1, ns = R0; st <= q; st++, ns *= R1) {
        for (int t = 0; t < G; t++) stage_load<fxc, EPT, R1>(buf.data(), regs(t), L, t, G);
        int up = 0;
        if (st > 1) {
            const int to = fx_room(R0, R1, q, !inv, lm, ls, st - 1);
            up = to - room;
            room = to;
        }
        for (fxc& v : x) v = fxc{v.x * (1ll << up), v.y * (1ll << up)};
        e += up;
        check();
        for (int t = 0; t < G; t++) {
            fx_stage<EPT, R1>(regs(t), ns, t, G, tw.data());
            stage_store<fxc, EPT, R1>(buf.data(), regs(t), L, ns, t, G);
        }
        check();
    }
    if (!fits) return 1e9;
    e -= 2 * q;
    long double err = 0, nrm = 0;
    for (int k = 0; k < L; k++) {
        cl acc = 0;
        for (int j = 0; j < nz; j++) {
            const long double a = (inv ? tp : -tp) * (long double)((long)j * k % L) / L;
            acc += cl(re[j], im[j]) * cl(cosl(a), sinl(a));
        }
        const fxc v = buf[pidx(k)];
        const cl got = inv ? cl(v.y, v.x) : cl(v.x, v.y);
        err += std::norm(got * ldexpl(1.0L, -e) - acc);
        nrm += std::norm(acc);
    }
    return (double)sqrtl(err / nrm);
}

template <int EPT, int R0, int R1> void report(int L) {
    for (int kind = 0; kind < 3; kind++) {
        std::printf("%d fwd %d %.3e\n", L, kind, error<EPT, R0, R1>(L, false, kind));
        std::printf("%d inv %d %.3e\n", L, kind, error<EPT, R0, R1>(L, true, kind));
    }
}

int main() {
    report<16, fx_plan(16).r0, fx_plan(16).r1>(16);
    report<16, fx_plan(32).r0, fx_plan(32).r1>(32);
    report<16, fx_plan(64).r0, fx_plan(64).r1>(64);
    report<16, fx_plan(128).r0, fx_plan(128).r1>(128);
    report<16, fx_plan(256).r0, fx_plan(256).r1>(256);
    report<16, fx_plan(512).r0, fx_plan(512).r1>(512);
    report<16, fx_plan(1024).r0, fx_plan(1024).r1>(1024);
    report<16, fx_plan(2048).r0, fx_plan(2048).r1>(2048);
    report<16, fx_plan(4096).r0, fx_plan(4096).r1>(4096);
    for (int L : {24, 96, 384, 1536}) report<12, 6, 4>(L);
    for (int L : {48, 192, 768, 3072}) report<12, 12, 4>(L);
    return 0;
}
