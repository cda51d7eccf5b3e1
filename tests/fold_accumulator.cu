// CPU emulation (fold_emulation.cu) of the compiled leapfrog pass with every
// accumulator it may be given -- p itself, another field, none -- and with the
// pressure as one field or as a sum of two, on contiguous and strided lines,
// against the run-time radices.  Prints the number of comparisons and of
// failures, after the output of fold_emulation.cu's own run; compiled and run by
// test_fold_forms_cpu.py.
#define main emulation_main
#include "fold_emulation.cu"
#undef main

static int compared = 0, failed = 0;

template <class C, bool STR>
void forms(int l, int r) {
    constexpr int L = C::R * C::A * C::B, N = L / 2;
    FoldAxis ax{};
    FoldTables tb;
    fold_axis(N, l, r, FoldChoice{C::R, C::A, C::B, C::P, C::P}, ax, tb);
    ax.tw = tb.tw.data();
    ax.tc = tb.tc.data();
    ax.th = tb.th.data();
    ax.P = C::P;
    while ((1 << ax.lgP) < C::P) ++ax.lgP;
    // one full and one ragged CTA
    const int lines = 3 * C::P + 1, outer = STR ? 2 : 1;
    ax.inner = STR ? lines : 1;
    ax.nlines = (int64_t)outer * lines;
    const unsigned grid = outer * ((lines + 2 * C::P - 1) / (2 * C::P));
    const int nthr = fold_threads(ax);
    std::mt19937 rng(L + 4 * l + 2 * r + STR);
    std::normal_distribution<double> nd;
    const size_t np = (size_t)ax.nlines * ax.lp, nu = (size_t)ax.nlines * N;
    std::vector<float> p(np), c(np), x(np), S(np), zero(np, 0.0f), V(nu);
    for (size_t i = 0; i < np; ++i) {
        p[i] = nd(rng);
        c[i] = nd(rng);
        S[i] = nd(rng);
    }
    for (auto& v : V) v = nd(rng);
    std::vector<float2> coef;
    fold_step_coef(ax, 1.0, -0.3, -0.7, coef);
    for (int two = 0; two < 2; ++two) {
        for (size_t i = 0; i < np; ++i) x[i] = two ? p[i] + c[i] : p[i];
        for (int acc = 0; acc < 3; ++acc) {
            std::vector<float> Va = V, Vb = V, a(np), b(np);
            FoldArgs w{};
            w.ax = ax;
            w.mode = FOLD_STEP;
            w.coef = coef.data();
            w.in = p.data();
            w.in2 = two ? c.data() : nullptr;
            w.u = Va.data();
            w.acc_in = acc == 0 ? w.in : acc == 1 ? S.data() : nullptr;
            w.out = a.data();
            // "p itself" is the pressure the pass reads, p + c where two fields
            // hold it; on strided lines that sum is not at hand (callers pass none)
            if (STR && two && acc == 0) continue;
            run_all<C, STR, FOLD_STEP>(w, grid, nthr);
            w.in = x.data();
            w.in2 = nullptr;
            w.u = Vb.data();
            w.acc_in = acc == 0 ? x.data() : acc == 1 ? S.data() : zero.data();
            w.out = b.data();
            run_all<fold::AnyCfg, STR, FOLD_STEP>(w, grid, nthr);
            double num = 0, den = 0;
            for (size_t i = 0; i < np; ++i) {
                num += ((double)a[i] - b[i]) * ((double)a[i] - b[i]);
                den += (double)b[i] * b[i];
            }
            for (size_t i = 0; i < nu; ++i) {
                num += ((double)Va[i] - Vb[i]) * ((double)Va[i] - Vb[i]);
                den += (double)Vb[i] * Vb[i];
            }
            ++compared;
            if (!(std::sqrt(num / den) < 1e-7)) {     // (a NaN fails)
                ++failed;
                std::printf("R%d A%d B%d P%d strided %d walls %d%d two fields %d accumulator %d: %g\n", C::R, C::A, C::B,
                            C::P, (int)STR, l, r, two, acc, std::sqrt(num / den));
            }
        }
    }
}
template <int R, int A, int B, int PS, int PC>
void all_forms() {
    for (int w = 0; w < 4; ++w) {
        forms<fold::Cfg<R, A, B, PC>, false>(w >> 1, w & 1);
        forms<fold::Cfg<R, A, B, 1>, false>(w >> 1, w & 1);
        forms<fold::Cfg<R, A, B, PS>, true>(w >> 1, w & 1);
        forms<fold::Cfg<R, A, B, 2>, true>(w >> 1, w & 1);
    }
}
int main() {
    emulation_main();
    all_forms<8, 2, 3, 8, 8>();
    all_forms<6, 5, 9, 8, 4>();
    all_forms<4, 8, 8, 8, 4>();
    all_forms<10, 5, 15, 4, 2>();
    all_forms<8, 8, 16, 4, 2>();
    all_forms<20, 10, 10, 4, 2>();
    std::printf("%d compared, %d failed\n", compared, failed);
    return failed != 0;
}
