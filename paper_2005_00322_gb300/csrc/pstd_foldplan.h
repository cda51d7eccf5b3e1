// pstd_foldplan.h -- host side of the folded passes (pstd_fold.cuh): the radix
// schedule of a length and its FP64-built, FP32-stored tables.
#pragma once

#include <cmath>
#include <complex>
#include <vector>

#include "pstd_fold.cuh"
#include "pstd_fold_list.h"

namespace pstd {

struct FoldChoice {
    int R, A, B;
    int PS, PC;              // pairs per CTA of a compiled schedule (0: run-time form)
};

// Real operations of one radix-n butterfly (adds, multiplies and fused
// multiply-adds of fold::Dft), to compare schedules.
inline double fold_radix_cost(int n) {
    switch (n) {
        case 1: return 0;
        case 2: return 4;
        case 3: return 16;
        case 4: return 16;
        case 5: return 40;
        case 7: return 84;
        case 8: return 52;
        case 11: return 220;
        case 13: return 312;
        default: break;
    }
    const int p = fold::small_factor(n), h = n / p;
    return p * fold_radix_cost(h) + h * fold_radix_cost(p) + 4.0 * (p - 1) * (h - 1);
}

// Schedule of length L: a compiled one, else L = R A B with the least work: R/2 + 1 sub-transforms of length A B and
// (A B)/2 + 1 butterflies of radix R, each element also costing a shared-memory
// round trip, a twiddle and its share of index arithmetic (about 12
// instructions).  Radices up to 10 keep a thread within 64 registers; larger
// ones are taken only where no such schedule exists or the work falls by
// more than their lost occupancy (a quarter).
inline bool fold_choose(int L, FoldChoice& best) {
    static const FoldChoice fixed[] = {
#define ENTRY(R, A, B, PS, PC) {R, A, B, PS, PC},
        PSTD_FOLD_ALL(ENTRY)
#undef ENTRY
    };
    for (const FoldChoice& f : fixed)
        if (f.R * f.A * f.B == L) {
            best = f;
            return true;
        }
    static const int even[] = {2, 4, 6, 8, 10, 12, 14, 16, 18, 20};
    static const int any[] = {1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 15, 16};
    double least = 0;
    best.R = 0;
    for (int R : even) {
        if (L % R) continue;
        const int M = L / R;
        for (int A : any) {
            if (M % A) continue;
            const int B = M / A;
            bool ok = false;
            for (int b : any) ok = ok || b == B;
            if (!ok) continue;
            const int NR = R / 2 + 1;
            double c = NR * (B * (fold_radix_cost(A) + 14.0 * A) + A * (fold_radix_cost(B) + 6.0 * B)) +
                       (M / 2 + 1) * (2 * fold_radix_cost(R) + 24.0 * R) / 2;
            int big = R;
            if (A > big) big = A;
            if (B > big) big = B;
            if (big > 10) c *= 1.25;
            if (big > 16) c *= 1.25;
            if (best.R == 0 || c < least) {
                least = c;
                best = FoldChoice{R, A, B, 0, 0};
            }
        }
    }
    return best.R > 0;
}

// Embedding of a line of N cells: the smallest compiled length L >= 4N.
inline bool conv_choose(int N, FoldChoice& best) {
    static const FoldChoice all[] = {
#define ENTRY(R, A, B) {R, A, B, 2, 1},
        PSTD_CONV_ALL(ENTRY)
#undef ENTRY
    };
    int least = 0;
    for (const FoldChoice& f : all) {
        const int L = f.R * f.A * f.B;
        if (L >= 4 * N && (least == 0 || L < least)) {
            least = L;
            best = f;
        }
    }
    return least > 0;
}

struct FoldTables {
    std::vector<float2> tw, tc, th;
};

// Geometry (without lines, pairs per CTA and device pointers) and twiddles of
// an axis of N cells; left / right: 0 Neumann, 1 Dirichlet.
inline void fold_axis(int N, int left, int right, const FoldChoice& ch, FoldAxis& x, FoldTables& t) {
    x.N = N;
    x.L = 2 * N;
    x.lo = left;
    x.lp = (right ? N - 1 : N) - left + 1;
    x.g = left != right;
    x.R = ch.R;
    x.A = ch.A;
    x.B = ch.B;
    x.M = ch.A * ch.B;
    x.nk = x.g ? (x.M + 1) / 2 : x.M / 2 + 1;
    x.s0 = !left && !right;
    x.sg = left ? -1.0f : 1.0f;
    x.rho = right ? -1.0f : 1.0f;
    // exp(-i pi num / den)
    auto unit = [](long num, long den) {
        const double a = M_PI * (double)(num % (2 * den)) / (double)den;
        return make_float2((float)std::cos(a), (float)-std::sin(a));
    };
    t.tw.resize((size_t)x.M);
    for (int k1 = 0; k1 < x.A; ++k1)
        for (int b = 0; b < x.B; ++b) t.tw[(size_t)k1 * x.B + b] = unit((long)b * (2 * k1 + x.g), x.M);
    const int H = x.R / 2;
    t.tc.resize((size_t)H * x.nk);
    t.th.resize((size_t)H * x.nk);
    for (int r = 0; r < H; ++r)
        for (int k = 0; k < x.nk; ++k) {
            t.tc[(size_t)r * x.nk + k] = unit((long)(r + 1) * (2 * k + x.g), x.L);
            t.th[(size_t)r * x.nk + k] = unit((long)(2 * r + 1) * (2 * k + x.g), 2L * x.L);
        }
}

// The embedding of an axis of N cells (walls as above) on choice `ch`: a
// folded axis of N' = L / 2 cells between two walls of the left wall's kind,
// storing the line's own nodes and half-nodes only.
inline void fold_axis_conv(int N, int left, int right, const FoldChoice& ch, FoldAxis& x, FoldTables& t) {
    fold_axis(ch.R * ch.A * ch.B / 2, left, left, ch, x, t);
    x.cN = N;
    x.lp = (right ? N - 1 : N) - left + 1;
}
// The staggered derivative's kernel at lag t = m + 1/2 (unit spacing), the
// derivative of the period-L interpolation kernel (Nyquist bin included once):
// group I sin(pi t) cot(pi t / L) / L, group II sin(pi t) / sin(pi t / L) / L.
inline double stagger_kernel(int N, int g, int m) {
    const double L = 2.0 * N, a = M_PI * (m + 0.5) / L, sn = std::sin(a);
    return -(m & 1 ? -1.0 : 1.0) * M_PI / (L * L) * (g ? std::cos(a) : 1.0) / (sn * sn);
}
// Multiplier per bin of an embedded derivative, C = i f X: the spectrum of the
// kernel cut off at |t| < 2N, over L; `fft` is a forward FP64 DFT in place.
template <class Fft>
std::vector<double> conv_coef(const FoldAxis& x, int g, double dx, Fft&& fft) {
    const int N = x.cN, L = x.L;
    std::vector<std::complex<double>> h((size_t)L, 0.0);
    for (int m = 0; m < 2 * N; ++m) {
        const double v = stagger_kernel(N, g, m);
        h[(size_t)m] += v;
        h[(size_t)(L - 1 - m)] -= v;         // odd: lag -(m + 1/2)
    }
    fft(h);
    std::vector<double> f((size_t)x.N + 1);
    for (int b = 0; b <= x.N; ++b) f[b] = (h[(size_t)b] * std::polar(1.0, -M_PI * b / L)).imag() / (L * dx);
    return f;
}

// Threads of a CTA: one per element group of the widest phase.
inline int fold_lanes(const FoldAxis& x) {
    const int NR = x.R / 2 + 1, m = x.A > x.B ? x.A : x.B;
    return NR * m > x.nk ? NR * m : x.nk;
}
inline int fold_threads(const FoldAxis& x) { return (fold_lanes(x) * x.P + 31) / 32 * 32; }

// Wavenumber of bin b, 0 <= b <= N - g; zero for a bin whose modes vanish
// (bin N between Dirichlet walls).
inline double fold_kappa(const FoldAxis& x, double dx, int b) {
    if (x.g ? b >= x.N : (b == x.N && x.sg < 0)) return 0.0;
    return M_PI * (2.0 * b + x.g) / (x.L * dx);
}
// Step coefficients per bin: V += c.x X, C = c.y V with c.x c.y =
// -kappa^2 sP sU / L.  c.y is divided by the rounded c.x, so that the product,
// which sets the mode's frequency, carries one rounding instead of two.  The
// second N + 1 entries are the first ones times the left wall's sign.
inline void fold_step_coef(const FoldAxis& x, double dx, double sP, double sU, std::vector<float2>& c) {
    c.assign(2 * ((size_t)x.N + 1), make_float2(0.0f, 0.0f));
    for (int b = 0; b <= x.N; ++b) {
        const double k = fold_kappa(x, dx, b);
        if (k == 0.0) continue;
        c[b].x = (float)(k * sP);
        c[b].y = (float)(-k * k * sP * sU / x.L / (double)c[b].x);
        c[x.N + 1 + b] = make_float2(x.sg * c[b].x, x.sg * c[b].y);
    }
}
inline void fold_grad_coef(const FoldAxis& x, double dx, double scale, std::vector<float>& f) {
    f.resize((size_t)x.N + 1);
    for (int b = 0; b <= x.N; ++b) f[b] = (float)(fold_kappa(x, dx, b) * scale / x.L);
}
inline void fold_order2_coef(const FoldAxis& x, double dx, double s2, std::vector<float>& f) {
    f.resize((size_t)x.N + 1);
    for (int b = 0; b <= x.N; ++b) {
        const double k = fold_kappa(x, dx, b);
        f[b] = (float)(-k * k * s2 / x.L);
    }
}

}  // namespace pstd
