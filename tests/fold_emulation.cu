// CPU emulation of the folded passes: every thread of a CTA runs each phase in
// turn (the phases are what lies between two CTA barriers), on every wall
// pair, both layouts, odd line counts and all modes, against the operators as
// direct FP64 sums over the symmetric-periodic extension.  Prints the largest
// relative L2 error; compiled and run by test_fold_cpu.py.
#include <cstdio>
#include <cmath>
#include <complex>
#include <vector>
#include <random>
#include "pstd_fold.cuh"
#include "pstd_foldplan.h"
using namespace pstd;
typedef std::complex<double> cd;
template <class C, bool STR, int MODE>
void run_all(const FoldArgs& a, unsigned grid, int nthr) {
    std::vector<char> mem(fold::smem_bytes(a.ax, STR) + 64, 0x7f);
    for (unsigned b = 0; b < grid; ++b) {
        std::vector<fold::Pass<C, STR, MODE>> ps;
        ps.reserve(nthr);
        for (int t = 0; t < nthr; ++t) ps.emplace_back(a, b, mem.data(), t, nthr);
        if constexpr (MODE == FOLD_CONV) {
            for (auto& p : ps) p.template p1<FOLD_GRAD_P>();
            for (auto& p : ps) p.template p2<FOLD_GRAD_P>();
            for (auto& p : ps) p.template p3<FOLD_GRAD_P>();
            for (auto& p : ps) p.template p4<FOLD_GRAD_P>();
            for (auto& p : ps) p.mid();
            for (auto& p : ps) { p.finish_u(); p.template p2<FOLD_GRAD_U>(); }
            for (auto& p : ps) { p.template p3<FOLD_GRAD_U>(); p.fetch_acc(); }
            for (auto& p : ps) p.template p4<FOLD_GRAD_U>();
            for (auto& p : ps) p.p5();
            for (auto& p : ps) p.finish();
            continue;
        }
        for (auto& p : ps) p.fetch_u();
        for (auto& p : ps) { p.p1(); }
        for (auto& p : ps) p.p2();
        for (auto& p : ps) { p.p3(); p.fetch_acc(); }
        for (auto& p : ps) p.p4();
        for (auto& p : ps) p.p5();
        for (auto& p : ps) p.finish();
    }
}
template <bool STR, int MODE>
void run_cfg(const FoldArgs& a, unsigned grid, int nthr) {
    if (MODE == -1 && a.mode == FOLD_ORDER2 && a.ax.R == 8 && a.ax.A == 8 && a.ax.B == 8 && a.ax.P == 4) run_all<fold::Cfg<8, 8, 8, 4>, STR, FOLD_ORDER2>(a, grid, nthr);
    else if (MODE == -1 && a.mode == FOLD_ORDER2 && a.ax.R == 8 && a.ax.A == 5 && a.ax.B == 10 && a.ax.P == 4) run_all<fold::Cfg<8, 5, 10, 4>, STR, FOLD_ORDER2>(a, grid, nthr);
    else if (a.ax.R == 8 && a.ax.A == 5 && a.ax.B == 10 && a.ax.P == 4) run_all<fold::Cfg<8, 5, 10, 4>, STR, MODE>(a, grid, nthr);
    else if (a.ax.R == 8 && a.ax.A == 8 && a.ax.B == 8 && a.ax.P == 4) run_all<fold::Cfg<8, 8, 8, 4>, STR, MODE>(a, grid, nthr);
    else run_all<fold::AnyCfg, STR, MODE>(a, grid, nthr);
}
// operators in FP64 by modes through long sums: D_p (node -> half), D_u (half -> node)
// compiled and run-time radices of the convolution pass
template <bool STR>
void run_conv(const FoldArgs& a, unsigned grid, int nthr) {
    if (a.ax.R == 8 && a.ax.A == 5 && a.ax.B == 8 && a.ax.P <= 2) run_all<fold::Cfg<8, 5, 8, STR ? 2 : 1>, STR, FOLD_CONV>(a, grid, nthr);
    else if (a.ax.R == 8 && a.ax.A == 8 && a.ax.B == 10 && a.ax.P != 2) run_all<fold::Cfg<8, 8, 10, STR ? 4 : 1>, STR, FOLD_CONV>(a, grid, nthr);
    else run_all<fold::AnyCfg, STR, FOLD_CONV>(a, grid, nthr);
}
static void dft(std::vector<cd>& x) {
    const size_t n = x.size();
    std::vector<cd> w(n), y(n, 0.0);
    for (size_t i = 0; i < n; ++i) w[i] = std::polar(1.0, -2.0 * M_PI * (double)i / (double)n);
    for (size_t k = 0; k < n; ++k)
        for (size_t j = 0, e = 0; j < n; ++j, e = (e + k) % n) y[k] += x[j] * w[e];
    x.swap(y);
}
static double rel(const std::vector<float>& x, const std::vector<double>& y) {
    double n = 0, d = 0;
    for (size_t i = 0; i < x.size(); ++i) { d += (x[i] - y[i]) * (x[i] - y[i]); n += y[i] * y[i]; }
    return std::sqrt(d / (n > 0 ? n : 1));
}
int main() {
    double worst = 0;
    int cases = 0, skipped = 0;
    for (int N : {1,2,3,4,5,6,7,8,9,10,11,12,13,15,16,18,20,24,25,27,32,36,40,45,48,60,64,67,73,75,79,89,97,96,100,125,128,135,180,192,200,223,243,250,251,256,375,384,499,500,512})
        for (int w = 0; w < 4; ++w)
            for (int lay = 0; lay < 2; ++lay) {
                const int l = w >> 1, r = w & 1;   // 0 N, 1 D
                const int lo = l, hi = r ? N - 1 : N, lp = hi - lo + 1;
                if (lp < 1) continue;
                const int L = 2 * N, g = l != r;
                FoldChoice ch{};
                FoldAxis ax{};
                FoldTables tb;
                const bool conv = !fold_choose(L, ch);
                if (conv) {
                    if (!conv_choose(N, ch)) {
                        ++skipped;
                        continue;
                    }
                    fold_axis_conv(N, l, r, ch, ax, tb);
                } else {
                    fold_axis(N, l, r, ch, ax, tb);
                }
                ax.tw = tb.tw.data(); ax.tc = tb.tc.data(); ax.th = tb.th.data();
                const int outer = lay ? 2 : 1, inner = lay ? 11 : 1;
                const int nl = lay ? outer * inner : 7;
                ax.P = conv ? (lay ? 2 << (N & 1) : 1) : 4; ax.lgP = conv ? (lay ? 1 + (N & 1) : 0) : 2;
                ax.inner = inner; ax.nlines = nl;
                const unsigned grid = lay ? outer * ((inner + 2 * ax.P - 1) / (2 * ax.P)) : (nl + 2 * ax.P - 1) / (2 * ax.P);
                const int nthr = fold_threads(ax);
                std::mt19937 rng(N * 8 + w * 2 + lay);
                std::normal_distribution<double> nd;
                auto idx = [&](int line, int pos, int len) { return lay ? (size_t)(line / inner) * len * inner + (size_t)pos * inner + line % inner : (size_t)line * len + pos; };
                std::vector<float> p((size_t)nl * lp), u((size_t)nl * N);
                for (auto& x : p) x = nd(rng);
                for (auto& x : u) x = nd(rng);
                // D_p, D_u by spectral definition on the extension (dx = 1)
                std::vector<double> Dp((size_t)N * lp), Du((size_t)lp * N);
                std::vector<double> KP(4 * L), KU(4 * L);   // sum over n at half-integer offsets d/2
                for (int d = -2 * L; d < 2 * L; ++d) { double kp = 0; for (int n = 0; n < L; ++n) { int nn = g ? (n < N ? n : n - L) : (n <= N ? n : n - L); const double k = M_PI * (2.0 * nn + g) / L; kp += (cd(0, k) * std::polar(1.0, k * (d + 0.5))).real(); } KP[d + 2 * L] = kp / L; }
                auto sgn = [&](int wl) { return wl ? -1.0 : 1.0; };
                for (int i = 0; i < N; ++i) for (int j = 0; j < lp; ++j) {
                    double acc = 0; const int q = j + lo;
                    for (int img = 0; img < 2; ++img) {
                        if (img && (q == 0 || q == N)) continue;
                        const double s = img ? sgn(r) : 1.0; const int pos = img ? L - q : q;
                        acc += s * KP[i - pos + 2 * L];
                    }
                    Dp[(size_t)i * lp + j] = acc;
                }
                for (int i = 0; i < lp; ++i) for (int j = 0; j < N; ++j) {
                    double acc = 0;
                    for (int img = 0; img < 2; ++img) {
                        const double s = img ? -sgn(r) : 1.0; const double pos = img ? L - 1 - j + 0.5 : j + 0.5;
                        acc += s * KP[(int)std::floor(i + lo - pos) + 2 * L];
                    }
                    Du[(size_t)i * N + j] = acc;
                }
                auto apply = [&](const std::vector<double>& D, int no, int ni, const std::vector<float>& x) {
                    std::vector<double> y((size_t)nl * no, 0.0);
                    for (int ln = 0; ln < nl; ++ln) for (int i = 0; i < no; ++i) { double s = 0; for (int j = 0; j < ni; ++j) s += D[(size_t)i * ni + j] * x[idx(ln, j, ni)]; y[idx(ln, i, no)] = s; }
                    return y;
                };
                const double sP = -0.3, sU = -0.7;
                auto go = [&](int mode, FoldArgs& a) {
                    a.mode = mode;
                    if (lay) { if (mode == FOLD_STEP) run_cfg<true, FOLD_STEP>(a, grid, nthr); else run_cfg<true, -1>(a, grid, nthr); }
                    else { if (mode == FOLD_STEP) run_cfg<false, FOLD_STEP>(a, grid, nthr); else run_cfg<false, -1>(a, grid, nthr); }
                };
                std::vector<float2> coef; fold_step_coef(ax, 1.0, sP, sU, coef);
                auto check = [&](const char* what, double e) { ++cases; if (e > worst) worst = e; if (!(e < 1e-6)) printf("N=%d walls %d%d lay %d R%d A%d B%d %s: %g\n", N, l, r, lay, ax.R, ax.A, ax.B, what, e); };
                auto coef_of = [&](std::vector<float>& f, double scale) {
                    if (!conv) return fold_grad_coef(ax, 1.0, scale, f);
                    const std::vector<double> f1 = conv_coef(ax, g, 1.0, dft);
                    f.resize(f1.size());
                    for (size_t i = 0; i < f.size(); ++i) f[i] = (float)(f1[i] * scale);
                };
                if (conv) {
                    std::vector<float> f1, f2, U = u, out(p.size()), S(p.size());
                    for (auto& x : S) x = nd(rng);
                    coef_of(f1, sP);
                    coef_of(f2, sU);
                    FoldArgs b{}; b.ax = ax; b.mode = FOLD_CONV; b.f = f1.data(); b.f2 = f2.data(); b.in = p.data(); b.u = U.data(); b.acc_in = S.data(); b.out = out.data();
                    if (lay) run_conv<true>(b, grid, nthr); else run_conv<false>(b, grid, nthr);
                    auto y = apply(Dp, N, lp, p); std::vector<float> un(u.size()); std::vector<double> ud(u.size());
                    for (size_t i = 0; i < y.size(); ++i) { ud[i] = u[i] + sP * y[i]; un[i] = ud[i]; }
                    check("conv u", rel(U, ud));
                    auto z = apply(Du, lp, N, un); for (size_t i = 0; i < z.size(); ++i) z[i] = sU * z[i] + S[i];
                    check("conv p", rel(out, z));
                }
                // grad p
                { std::vector<float> f, out(u.size()); coef_of(f, 1.0); FoldArgs a{}; a.ax = ax; a.f = f.data(); a.in = p.data(); a.out = out.data(); go(FOLD_GRAD_P, a); check("gradp", rel(out, apply(Dp, N, lp, p))); }
                { std::vector<float> f, out(p.size()); coef_of(f, 1.0); FoldArgs a{}; a.ax = ax; a.f = f.data(); a.in = u.data(); a.out = out.data(); go(FOLD_GRAD_U, a); if (!(N == 1)) check("gradu", rel(out, apply(Du, lp, N, u))); }
                if (conv) continue;
                { std::vector<float> f, out(p.size(), 0.25f), q(p.size()); fold_order2_coef(ax, 1.0, 0.1, f); FoldArgs a{}; a.ax = ax; a.f = f.data(); a.in = p.data(); a.out = out.data(); a.accumulate = 1; a.pout = q.data(); go(FOLD_ORDER2, a);
                  auto y = apply(Dp, N, lp, p); std::vector<float> yf(y.begin(), y.end()); auto z = apply(Du, lp, N, yf); for (auto& v : z) v = v * 0.1 + 0.25; check("order2", rel(out, z)); for (size_t i = 0; i < z.size(); ++i) z[i] += p[i]; check("order2 p", rel(q, z)); }
                // step: to spec, pass, from spec
                { std::vector<float> U = u, out(p.size()), P = p, S(p.size());
                  for (auto& x : S) x = nd(rng);
                  FoldArgs a{}; a.ax = ax; a.in = U.data(); a.u = U.data(); go(FOLD_TO_SPEC, a);
                  FoldArgs b{}; b.ax = ax; b.coef = coef.data(); b.in = P.data(); b.u = U.data(); b.acc_in = lay ? S.data() : P.data(); b.out = out.data(); go(FOLD_STEP, b);
                  FoldArgs c{}; c.ax = ax; c.u = U.data(); c.out = U.data(); go(FOLD_FROM_SPEC, c);
                  auto y = apply(Dp, N, lp, p); std::vector<float> un(u.size()); std::vector<double> ud(u.size());
                  for (size_t i = 0; i < y.size(); ++i) { ud[i] = u[i] + sP * y[i]; un[i] = ud[i]; }
                  check("step u", rel(U, ud));
                  auto z = apply(Du, lp, N, un); for (size_t i = 0; i < z.size(); ++i) z[i] = sU * z[i] + (lay ? S[i] : P[i]);
                  check("step p", rel(out, z)); }
            }
    printf("%d checks, worst %g, %d without schedule\n", cases, worst, skipped);
    return 0;
}
