// pstd_fold.cuh -- axis passes on symmetry-folded FFTs (walled axes).
//
// A pair of real lines rides in one complex sequence x (real and imaginary
// parts) whose symmetric-periodic extension (Section 3.2, Fig. 3) has length
// L = 2N and obeys x[-j] = s x[j] (s = +1 Neumann, -1 Dirichlet left wall),
// periodic (group I) or antiperiodic (group II, g = 1) in L.  Its spectrum
//     X[k] = sum_{j<L} x[j] exp(-i pi j (2k + g) / L)
// is a DTT of the pair (Table 1: types I and III) up to a constant phase, and
// X[-k-g] = s X[k], so N + 1 - g bins carry it.  A plain length-L FFT
// computes both halves of the sequence and both halves of the spectrum; this
// file computes one of each.
//
// Decimation by R (even): with j = R m + r and L = R M,
//     Y_r[k] = sum_{m<M} x[Rm + r] exp(-i pi m (2k + g) / M),
//     X[k + M q] = sum_r exp(-2 pi i r q / R) W_r,  W_r = t_r Y_r[k],
//     t_r = exp(-i pi r (2k + g) / L),
// and the symmetry gives W_{R-r} = s conj(t_r) Y_r[M - g - k].  So only the
// R/2 + 1 sub-sequences r <= R/2 are transformed, and only one radix-R
// butterfly of each pair (k, M - g - k) is run; it holds 2 x R/2 distinct bins.
// The inverse transform is the transpose: butterflies of the same pairs, then
// sub-transforms of the residues r <= R/2, which are the N + 1 nodes (each
// once, the residues 1 <= r < R/2 through the reflection too).  On the half-nodes
// (positions j + 1/2) the residues pair as r <-> R - 1 - r and R/2
// sub-transforms do.  A sub-transform of length M = A B is two register
// radices with one exchange.
//
// In these bins the staggered derivative's multiplier is real: with the
// velocity held as V = -i (its half-node spectrum), a leapfrog pass is
// V += (kappa scale) X, C = -(kappa scale) V, and one inverse transform of C
// (Eq. dtt_pstd_solution in transform space), with no conjugate-symmetric
// bookkeeping: N real coefficients per line, stored in the velocity's own
// buffer (slot b - 1 for NN walls, whose bin 0 vanishes, else slot b).
//
// A line of any other length N (convolution passes, cN = N below) is embedded:
// the derivative is the convolution of the extension with an odd kernel at
// half-integer lags, and N half-node outputs of the nodes |j| <= N (or the
// reverse) only need its lags |t| < 2N.  Cutting the kernel off there and laying
// both on a circle of L = 2 N' >= 4N positions keeps every symmetry (even or
// odd about 0, hence also about N'), so each derivative is a folded transform
// of length L with zeros beyond N, a real multiplier and a folded inverse.
//
// A pass runs as five phases with a CTA barrier between them, in place in one
// shared-memory buffer (element (r, k1, t) of the first radix, (r, k = k1 + A k2)
// of the second and (r, k) of the combination share addresses):
//   p1  input nodes -> radix A, twiddle      p4  radix B (inverse)
//   p2  radix B                              p5  twiddle, radix A -> output nodes
//   p3  radix R, spectral update, radix R
// What bounds it and why: see the kernels in pstd_fkernels.cuh.
#pragma once

#include <type_traits>
#include <utility>

#include "pstd_wcta.cuh"

namespace pstd {

// One walled axis (left and right wall at nodes).
struct FoldAxis {
    int N, L, lp, lo, g;
    int R, A, B, M;
    int P, lgP;              // line pairs per CTA (a power of two)
    int wide;                // a CTA's lines span 4 GiB or more: 64-bit offsets
    int nk;                  // butterflies: pairs {k, M - g - k}
    int s0;                  // velocity slot of bin b is b - s0
    int cN;                  // convolution passes: cells of the line (N = L / 2 is the embedding's); else 0
    float sg, rho;           // sign of p reflected about the left / right wall
    const float2* tw;        // [k1][t] exp(-i pi t (2 k1 + g) / M), A B entries
    const float2* tc;        // [r - 1][k] exp(-i pi r (2k + g) / L), r = 1..R/2
    const float2* th;        // [r][k] exp(-i pi (r + 1/2)(2k + g) / L), r < R/2
    int64_t nlines, inner;
};

enum { FOLD_STEP = 0, FOLD_GRAD_P = 1, FOLD_GRAD_U = 2, FOLD_TO_SPEC = 3, FOLD_FROM_SPEC = 4, FOLD_ORDER2 = 5,
       FOLD_CONV = 7,        // leapfrog pass of an embedded line: p -> u, u += , u -> p, p +=
       // kernels that loop over FOLD_STEP passes: a 1-D run, a cooperative run
       FOLD_LINE = 6, FOLD_PERSIST = 8,
       FOLD_MISC = -2 };     // kernels for GRAD_P, GRAD_U, TO_SPEC or FROM_SPEC, chosen at run time (-1: for any mode)

struct FoldArgs {
    FoldAxis ax;
    int mode;
    const float2* coef;      // FOLD_STEP: per bin b <= N (p -> V, V -> p); zero where a bin has no slot
    const float* f;          // FOLD_GRAD_*, FOLD_ORDER2, FOLD_CONV p -> u: per bin multiplier (without the factor i)
    const float* f2;         // FOLD_CONV u -> p
    const float* in;         // p (STEP, GRAD_P, ORDER2) or u
    const float* in2;        // STEP: p is in + in2 where given
    float* u;                // velocity spectrum (STEP, TO_SPEC, FROM_SPEC)
    const float* acc_in;     // STEP: out = acc_in + contribution; null (fixed schedules only): out = contribution.
                             // acc_in == in on contiguous lines: out = in (+ in2) + contribution
    float* out;
    int accumulate;          // GRAD_*, ORDER2: out += instead of out =
    float* pout;             // ORDER2: also write in + (the new out) here (may be `in`)
};

namespace fold {

// ---- radix-n DFTs in registers, natural order in and out ---------------------
// forward: y_k = sum_j a_j exp(-2 pi i j k / n); inverse: exp(+...).  Every
// operation is explicitly rounded (pstd_ops.cuh), so the per-axis kernels and
// the cooperative one round identically.
template <int n, int k>
struct Root {  // exp(+2 pi i k / n)
    static constexpr double ang = wf::unit_angle(k, n);
    static constexpr float c = (float)wf::taylor_cos(ang);
    static constexpr float s = (float)wf::taylor_sin(ang);
};
// a * exp(sgn 2 pi i k / n), sgn = +1 (INV) or -1
template <int n, int k, bool INV>
PSTD_HD float2 mul_root(float2 a) {
    constexpr int kk = ((k % n) + n) % n;
    if constexpr (kk == 0) {
        return a;
    } else if constexpr (2 * kk == n) {
        return make_float2(-a.x, -a.y);
    } else if constexpr (4 * kk == n) {
        return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
    } else if constexpr (4 * kk == 3 * n) {
        return INV ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
    } else {
        constexpr float c = Root<n, kk>::c;
        constexpr float s = INV ? Root<n, kk>::s : -Root<n, kk>::s;
        return make_float2(rfma(a.x, c, -rmul(a.y, s)), rfma(a.x, s, rmul(a.y, c)));
    }
}
constexpr int small_factor(int n) {
    for (int p : {4, 2, 3, 5, 7, 11, 13})
        if (n % p == 0) return p;
    return n;
}

template <int n, bool INV>
struct Dft;
template <bool INV>
struct Dft<1, INV> {
    static PSTD_HD void run(float2*) {}
};
template <bool INV>
struct Dft<2, INV> {
    static PSTD_HD void run(float2* a) { dft2(a); }
};
template <bool INV>
struct Dft<4, INV> {
    static PSTD_HD void run(float2* a) {
        const float2 s02 = cadd(a[0], a[2]), d02 = csub(a[0], a[2]);
        const float2 s13 = cadd(a[1], a[3]), d13 = csub(a[1], a[3]);
        const float2 r = INV ? make_float2(-d13.y, d13.x) : make_float2(d13.y, -d13.x);
        a[0] = cadd(s02, s13);
        a[2] = csub(s02, s13);
        a[1] = cadd(d02, r);
        a[3] = csub(d02, r);
    }
};
// 8 = 2 x 4 with the eighth roots folded into fused multiply-adds
template <bool INV>
struct Dft<8, INV> {
    static PSTD_HD void run(float2* a) {
        float2 e[4] = {a[0], a[2], a[4], a[6]};
        float2 o[4] = {a[1], a[3], a[5], a[7]};
        Dft<4, INV>::run(e);
        Dft<4, INV>::run(o);
        constexpr float h = 0.70710678118654752440f;  // sqrt(1/2)
        const float2 o2 = INV ? make_float2(-o[2].y, o[2].x) : make_float2(o[2].y, -o[2].x);
        // o1 w = h (x + y, y - x), o3 w^3 = h (y - x, -(x + y)) forward; conjugated roots inverse
        const float2 q1 = INV ? make_float2(rsub(o[1].x, o[1].y), radd(o[1].x, o[1].y))
                              : make_float2(radd(o[1].x, o[1].y), rsub(o[1].y, o[1].x));
        const float2 q3 = INV ? make_float2(-radd(o[3].x, o[3].y), rsub(o[3].x, o[3].y))
                              : make_float2(rsub(o[3].y, o[3].x), -radd(o[3].x, o[3].y));
        a[0] = cadd(e[0], o[0]);
        a[4] = csub(e[0], o[0]);
        a[1] = make_float2(rfma(h, q1.x, e[1].x), rfma(h, q1.y, e[1].y));
        a[5] = make_float2(rfma(-h, q1.x, e[1].x), rfma(-h, q1.y, e[1].y));
        a[2] = cadd(e[2], o2);
        a[6] = csub(e[2], o2);
        a[3] = make_float2(rfma(h, q3.x, e[3].x), rfma(h, q3.y, e[3].y));
        a[7] = make_float2(rfma(-h, q3.x, e[3].x), rfma(-h, q3.y, e[3].y));
    }
};
// odd primes: the pairs a_j +- a_{n-j} against cosines and sines
template <int n, bool INV, int k, int j>
PSTD_HD void prime_term(const float2* s, const float2* d, float2& c, float2& q) {
    if constexpr (j <= (n - 1) / 2) {
        constexpr float cs = Root<n, (j * k) % n>::c, sn = Root<n, (j * k) % n>::s;
        c = make_float2(rfma(cs, s[j].x, c.x), rfma(cs, s[j].y, c.y));
        q = make_float2(rfma(sn, d[j].x, q.x), rfma(sn, d[j].y, q.y));
        prime_term<n, INV, k, j + 1>(s, d, c, q);
    }
}
template <int n, bool INV, int k>
PSTD_HD void prime_out(float2* a, float2 a0, const float2* s, const float2* d) {
    if constexpr (k <= (n - 1) / 2) {
        float2 c = a0;
        constexpr float s1 = Root<n, k % n>::s, c1 = Root<n, k % n>::c;
        c = make_float2(rfma(c1, s[1].x, c.x), rfma(c1, s[1].y, c.y));
        float2 q = make_float2(rmul(s1, d[1].x), rmul(s1, d[1].y));
        prime_term<n, INV, k, 2>(s, d, c, q);
        // forward: y_k = c - i q, y_{n-k} = c + i q
        const float2 iq = INV ? make_float2(q.y, -q.x) : make_float2(-q.y, q.x);
        a[k] = csub(c, iq);
        a[n - k] = cadd(c, iq);
        prime_out<n, INV, k + 1>(a, a0, s, d);
    }
}
template <int n, bool INV>
PSTD_HD void prime_dft(float2* a) {
    constexpr int H = (n - 1) / 2;
    float2 s[H + 1], d[H + 1];
    const float2 a0 = a[0];
    float2 sum = a0;
#pragma unroll
    for (int j = 1; j <= H; ++j) {
        s[j] = cadd(a[j], a[n - j]);
        d[j] = csub(a[j], a[n - j]);
        sum = cadd(sum, s[j]);
    }
    prime_out<n, INV, 1>(a, a0, s, d);
    a[0] = sum;
}
// composite n = p H: p sub-transforms of length H over a[p i + q], twiddles,
// radix p across them
template <int n, int H, bool INV, int q, int... K>
PSTD_HD void twiddle_row(float2* b, std::integer_sequence<int, K...>) {
    ((b[K] = mul_root<n, q * K, INV>(b[K])), ...);
}
template <int n, int p, bool INV, int q>
PSTD_HD void sub_rows(const float2* a, float2 (*b)[n / p]) {
    if constexpr (q < p) {
        constexpr int H = n / p;
#pragma unroll
        for (int i = 0; i < H; ++i) b[q][i] = a[p * i + q];
        Dft<H, INV>::run(b[q]);
        twiddle_row<n, H, INV, q>(b[q], std::make_integer_sequence<int, H>{});
        sub_rows<n, p, INV, q + 1>(a, b);
    }
}
template <int n, bool INV>
struct Dft {
    static PSTD_HD void run(float2* a) {
        constexpr int p = small_factor(n);
        if constexpr (p == n) {
            prime_dft<n, INV>(a);
        } else {
            constexpr int H = n / p;
            float2 b[p][H];
            sub_rows<n, p, INV, 0>(a, b);
#pragma unroll
            for (int k = 0; k < H; ++k) {
                float2 c[p];
#pragma unroll
                for (int q = 0; q < p; ++q) c[q] = b[q][k];
                Dft<p, INV>::run(c);
#pragma unroll
                for (int q = 0; q < p; ++q) a[k + H * q] = c[q];
            }
        }
    }
};
// a[e] *= exp(-+ i pi e / n)
template <int n, bool INV, int... E>
PSTD_HD void half_twiddle(float2* a, std::integer_sequence<int, E...>) {
    ((a[E] = mul_root<2 * n, E, INV>(a[E])), ...);
}

// ---- geometry: radices and pairs per CTA fixed at compile time, or of the plan -
template <int R_, int A_, int B_, int P_>
struct Cfg {
    static constexpr int R = R_, A = A_, B = B_, P = P_;
    static constexpr bool fixed = R_ > 0;
    static constexpr bool resident = false;
    static constexpr bool onto_p_only = false;
};
using AnyCfg = Cfg<0, 0, 0, 0>;
// contiguous step passes of a last axis alone: acc_in == in
template <class C>
struct OntoP : C {
    static constexpr bool onto_p_only = true;
};
// tables that may lie in shared memory (a cooperative run's)
template <class C>
struct Resident : C {
    static constexpr bool resident = true;
};

PSTD_HD int padded(int A) { return A | 1; }   // odd stride of k2 / t: no bank conflicts between lanes
PSTD_HD int sub_words(int A, int B) { return padded(A) * B; }
PSTD_HD size_t buffer_words(const FoldAxis& x) { return (size_t)x.P * (x.R / 2 + 1) * sub_words(x.A, x.B); }
// Output rows of contiguous lines are gathered in shared memory: position i
// at word row_word(i), 4 spare words after each 32, so that the stride-R
// writes of p5 (R = 8, 16) spread over all banks.
PSTD_HD int row_word(int i) { return i + 4 * (i >> 5); }
PSTD_HD int row_pitch(const FoldAxis& x) { return row_word((x.lp > x.N ? x.lp : x.N) + 1) | 1; }
PSTD_HD size_t smem_bytes(const FoldAxis& x, bool strided) {
    return buffer_words(x) * sizeof(float2) + (strided ? 0 : (size_t)2 * x.P * row_pitch(x) * sizeof(float));
}

template <int V>
using Int = std::integral_constant<int, V>;

// run f with the radix as a compile-time constant
template <int FIX, class F>
PSTD_HD void with_radix(int r, F&& f) {
    if constexpr (FIX > 0) {
        f(Int<FIX>{});
    } else {
        switch (r) {
            case 1: f(Int<1>{}); break;
            case 2: f(Int<2>{}); break;
            case 3: f(Int<3>{}); break;
            case 4: f(Int<4>{}); break;
            case 5: f(Int<5>{}); break;
            case 6: f(Int<6>{}); break;
            case 7: f(Int<7>{}); break;
            case 8: f(Int<8>{}); break;
            case 9: f(Int<9>{}); break;
            case 10: f(Int<10>{}); break;
            case 11: f(Int<11>{}); break;
            case 12: f(Int<12>{}); break;
            case 13: f(Int<13>{}); break;
            case 15: f(Int<15>{}); break;
            case 16: f(Int<16>{}); break;
            default: break;
        }
    }
}
template <int FIX, class F>
PSTD_HD void with_even(int r, F&& f) {
    if constexpr (FIX > 0) {
        f(Int<FIX>{});
    } else {
        switch (r) {
            case 2: f(Int<2>{}); break;
            case 4: f(Int<4>{}); break;
            case 6: f(Int<6>{}); break;
            case 8: f(Int<8>{}); break;
            case 10: f(Int<10>{}); break;
            case 12: f(Int<12>{}); break;
            case 14: f(Int<14>{}); break;
            case 16: f(Int<16>{}); break;
            case 18: f(Int<18>{}); break;
            case 20: f(Int<20>{}); break;
            default: break;
        }
    }
}

PSTD_HD float2 ldc2(const float2* p) {   // read-only table entry
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}
PSTD_HD float ldc(const float* p) {
#ifdef __CUDA_ARCH__
    return __ldg(p);
#else
    return *p;
#endif
}

// One pass of one CTA: P line pairs.  STR: strided axis (lines adjacent in
// memory: neighbouring lanes hold neighbouring pairs, so global accesses are
// runs of 2P words, straight between memory and registers); otherwise
// contiguous lines, read in place (the R residues share their sectors in L1)
// and written through rows in shared memory.  MODE < 0: the mode is a
// run-time value (FOLD_MISC: of four).  Byte offsets from a CTA-uniform base are 32-bit in the fixed
// schedules (the plan takes the run-time form for fields beyond 4 GiB): with
// 64-bit ones the address arithmetic cost more than the FFT (40 integer against
// 36 floating-point instructions per point on 256^3).
template <class C, bool STR, int MODE>
struct Pass {
    using Off = typename std::conditional<C::fixed, uint32_t, int64_t>::type;
    const FoldArgs& a;
    float2* sm;
    float* st;
    int tid, nthr;
    int64_t line0;           // contiguous: first line of the CTA
    int64_t o, i0;           // strided: outer block, first inner index
    int nv;                  // lines of this CTA
    // Fixed schedules request what a phase needs from memory ahead of it, so
    // that the latency passes behind the barriers and the radices between:
    // the velocity slots after p1 (contiguous: before it), the accumulator
    // after p3.  A contiguous leapfrog pass mostly accumulates onto p itself
    // (acc_in == in, the last axis), which p5's thread has read in p1; the
    // second-order pass keeps that p for pout.
    static constexpr bool ahead = C::fixed && (MODE == FOLD_STEP || MODE == FOLD_ORDER2 || MODE == FOLD_CONV);
    static constexpr bool ahead_u = C::fixed && MODE == FOLD_STEP;
    static constexpr bool onto_p = ahead_u && !STR;
    static constexpr bool keep_p = ahead && MODE == FOLD_ORDER2 && STR;
    float2 uw[ahead_u ? C::R : 1];
    float2 ac[ahead ? C::A : 1];
    float2 pk[keep_p ? C::A : 1];

    static PSTD_HD float2 tab(const float2* p) { if constexpr (C::resident) return *p; else return ldc2(p); }
    PSTD_HD int R() const { if constexpr (C::fixed) return C::R; else return a.ax.R; }
    PSTD_HD int A() const { if constexpr (C::fixed) return C::A; else return a.ax.A; }
    PSTD_HD int B() const { if constexpr (C::fixed) return C::B; else return a.ax.B; }
    PSTD_HD int M() const { if constexpr (C::fixed) return C::A * C::B; else return a.ax.M; }
    PSTD_HD int L() const { if constexpr (C::fixed) return C::A * C::B * C::R; else return a.ax.L; }
    PSTD_HD int N() const { if constexpr (C::fixed) return C::A * C::B * C::R / 2; else return a.ax.N; }
    PSTD_HD int P() const { if constexpr (C::fixed) return C::P; else return a.ax.P; }
    PSTD_HD int Ap() const { return padded(A()); }
    PSTD_HD int S1() const { return Ap() * B(); }
    PSTD_HD int NRmax() const { return R() / 2 + 1; }
    // PM: the mode a phase runs in; a convolution pass runs a FOLD_GRAD_P and a
    // FOLD_GRAD_U
    template <int PM = MODE>
    PSTD_HD int mode() const { if constexpr (PM >= 0) return PM; else return a.mode; }
    template <int PM = MODE>
    PSTD_HD bool in_half() const { return mode<PM>() == FOLD_GRAD_U || mode<PM>() == FOLD_TO_SPEC; }
    template <int PM = MODE>
    PSTD_HD bool out_half() const { return mode<PM>() == FOLD_GRAD_P || mode<PM>() == FOLD_FROM_SPEC; }
    // (constant false in FOLD_MISC kernels)
    template <int PM = MODE>
    PSTD_HD bool stepping() const { if constexpr (MODE == FOLD_MISC) return false; else return mode<PM>() == FOLD_STEP; }
    template <int PM = MODE>
    PSTD_HD bool order2() const { if constexpr (MODE == FOLD_MISC) return false; else return mode<PM>() == FOLD_ORDER2; }
    PSTD_HD bool conv() const {
        if constexpr (MODE == FOLD_CONV) return true;
        else if constexpr (MODE != -1) return false;
        else return a.ax.cN > 0;
    }
    PSTD_HD int nhalf() const { return conv() ? a.ax.cN : N(); }     // stored half-nodes
    template <int PM = MODE>
    PSTD_HD int nin() const { return in_half<PM>() ? nhalf() : a.ax.lp; }
    template <int PM = MODE>
    PSTD_HD int nout() const { return out_half<PM>() ? nhalf() : a.ax.lp; }

    // f(pair p, work w) for this thread's items of W per pair
    template <class F>
    PSTD_HD void items(int W, F&& f) const {
        if constexpr (C::fixed) {
            if (tid >= W * C::P) return;
            if constexpr (STR) f(tid & (C::P - 1), tid / C::P);
            else f(tid / W, tid % W);
        } else {
            for (int idx = tid; idx < W * P(); idx += nthr) {
                if constexpr (STR) {
                    f(idx & (a.ax.P - 1), idx >> a.ax.lgP);
                } else {
                    const int p = idx / W;
                    f(p, idx - p * W);
                }
            }
        }
    }
    // address of element `loc` of residue r of pair p; step between locs
    PSTD_HD float2* at(int r, int p) const {
        if constexpr (STR) return sm + r * S1() * P() + p;
        else return sm + (p * NRmax() + r) * S1();
    }
    PSTD_HD int ls() const { if constexpr (STR) return P(); else return 1; }
    PSTD_HD int kloc(int k) const {
        if constexpr (C::fixed) return k + (k / C::A) * (padded(C::A) - C::A);
        else return a.ax.A & 1 ? k : k + k / a.ax.A;
    }
    // pair p holds lines 2p and 2p + 1, so that a line's partner, and with it
    // every rounding, does not depend on P (lines p and p + P of a strided tile
    // would touch each sector once instead of twice: 251 against 254 us per
    // 256^3 step)
    PSTD_HD bool va(int p) const { return 2 * p < nv; }
    PSTD_HD bool vb(int p) const { return 2 * p + 1 < nv; }

    PSTD_HD Pass(const FoldArgs& args, unsigned item, void* smem, int tid_, int nthr_)
        : a(args), sm((float2*)smem), tid(tid_), nthr(nthr_) {
        st = (float*)(sm + (size_t)P() * NRmax() * S1());
        if constexpr (STR) {
            const unsigned G = 2 * P();
            const unsigned per = ((unsigned)a.ax.inner + G - 1) / G;
            const unsigned blk = item / per;
            o = blk;
            i0 = (item - blk * per) * G;
            const int64_t left = a.ax.inner - i0;
            nv = (int)(left < G ? left : G);
        } else {
            line0 = (int64_t)item * 2 * P();
            const int64_t left = a.ax.nlines - line0;
            nv = (int)(left < 2 * P() ? left : 2 * P());
        }
    }
    // the CTA's first line at position 0 in a field of `len` entries along the
    // axis (uniform over the CTA), and a thread's byte offsets from it
    template <class T>
    PSTD_HD T* base(T* f, int len) const {
        if constexpr (STR) return f + (o * (int64_t)len * a.ax.inner + i0);
        else return f + line0 * (int64_t)len;
    }
    PSTD_HD Off line_off(int p, int len) const { return STR ? (Off)(8 * p) : (Off)(8 * p) * (Off)len; }
    PSTD_HD Off pos_step() const { return STR ? (Off)(4 * a.ax.inner) : (Off)4; }
    PSTD_HD int line_step(int len) const { return STR ? 1 : len; }
    static PSTD_HD float ld(const float* b, Off off) { return *(const float*)((const char*)b + off); }
    static PSTD_HD void put(float* b, Off off, float v) { *(float*)((char*)b + off) = v; }

    // f(true) for a CTA all of whose lines exist, else f(false): the common
    // case carries no per-line tests
    template <class F>
    PSTD_HD void by_full(F&& f) const {
        if (nv == 2 * P()) f(std::true_type{});
        else f(std::false_type{});
    }

    // p1: residue r, lane t: elements m = t + B e, radix A over e, twiddle.
    // The extension value at position j is node j (reflected about the right
    // wall beyond it) or half-node j.  For even A the positions below e = A/2
    // lie before the right wall, so which elements are reflected is known at
    // compile time, and only node 0 and node N may be absent.
    template <int PM = MODE>
    PSTD_HD void p1() {
        if (mode<PM>() == FOLD_FROM_SPEC) return;
        by_full([&](auto full) {
        with_radix<C::A>(A(), [&](auto RA) {
            constexpr int a_ = decltype(RA)::value;
            constexpr bool even = a_ % 2 == 0;
            const bool half = in_half<PM>();
            const int n = N(), lo = half ? 0 : a.ax.lo, len = nin<PM>();
            const int refl = half ? 2 * n - 1 : 2 * n;   // position j reflects to refl - j
            const float rsg = half ? -a.ax.rho : a.ax.rho;
            const float* xa = base(a.in, len);
            const float* xb = xa + line_step(len);
            items((half ? R() / 2 : R() / 2 + 1) * B(), [&](int p, int w) {
                const int r = w / B(), t = w - r * B();
                const int j0 = R() * t + r, dj = R() * B();
                const bool la = full || va(p), lb = full || vb(p);
                const Off ps = pos_step(), lof = line_off(p, len);
                const Off od = lof + (Off)(j0 - lo) * ps;          // position j0 + dj e: + e step
                const Off om = lof + (Off)(refl - j0 - lo) * ps;   // its reflection: - e step
                const Off step = (Off)dj * ps;
                float2 x[a_];
#pragma unroll
                for (int e = 0; e < a_; ++e) {
                    const int j = j0 + dj * e;
                    const bool mir = even ? 2 * e >= a_ : (half ? j >= n : j > n);
                    const Off off = mir ? om - (Off)e * step : od + (Off)e * step;
                    bool ok = true;
                    const int i = (mir ? refl - j : j) - lo;
                    if (conv() || (!half && (!even || e == 0 || 2 * e == a_))) ok = i >= 0 && i < len;
                    x[e] = make_float2(ok && la ? ld(xa, off) : 0.0f, ok && lb ? ld(xb, off) : 0.0f);
                    // node N of an embedded line stands at both ends of its window
                    if (conv() && !half && i + lo == a.ax.cN) x[e] = cscale(x[e], 0.5f);
                }
                // (after all loads of the first field are under way)
                if constexpr (ahead_u) {
                    if (a.in2) {
                        const float* za = base(a.in2, len);
                        const float* zb = za + line_step(len);
#pragma unroll
                        for (int e = 0; e < a_; ++e) {
                            const int j = j0 + dj * e;
                            const bool mir = even ? 2 * e >= a_ : j > n;
                            const Off off = mir ? om - (Off)e * step : od + (Off)e * step;
                            bool ok = true;
                            const int i = (mir ? refl - j : j) - lo;
                            if (!even || e == 0 || 2 * e == a_) ok = i >= 0 && i < len;
                            x[e].x = radd(x[e].x, ok && la ? ld(za, off) : 0.0f);
                            x[e].y = radd(x[e].y, ok && lb ? ld(zb, off) : 0.0f);
                        }
                    }
                }
#pragma unroll
                for (int e = 0; e < a_; ++e) {
                    const bool mir = even ? 2 * e >= a_ : (half ? j0 + dj * e >= n : j0 + dj * e > n);
                    if constexpr (onto_p) ac[e] = x[e];
                    if constexpr (keep_p) pk[e] = x[e];
                    if (mir) x[e] = cscale(x[e], rsg);
                }
                if (a.ax.g) half_twiddle<a_, false>(x, std::make_integer_sequence<int, a_>{});
                Dft<a_, false>::run(x);
                float2* d = at(r, p) + Ap() * t * ls();
#pragma unroll
                for (int k = 0; k < a_; ++k) {
                    if (k > 0 || a.ax.g) x[k] = cmul(x[k], tab(&a.ax.tw[k * B() + t]));
                    d[k * ls()] = x[k];
                }
            });
        });
        });
    }
    // p2 / p4: residue r, lane k1: radix B over the second index, in place
    template <bool INV>
    PSTD_HD void inner_radix(int NR) {
        with_radix<C::B>(B(), [&](auto RB) {
            constexpr int b_ = decltype(RB)::value;
            if constexpr (b_ > 1) {
                items(NR * A(), [&](int p, int w) {
                    const int r = w / A(), k1 = w - r * A();
                    float2* s = at(r, p) + k1 * ls();
                    float2 x[b_];
#pragma unroll
                    for (int t = 0; t < b_; ++t) x[t] = s[t * Ap() * ls()];
                    Dft<b_, INV>::run(x);
#pragma unroll
                    for (int t = 0; t < b_; ++t) s[t * Ap() * ls()] = x[t];
                });
            }
        });
    }
    template <int PM = MODE>
    PSTD_HD void p2() {
        if (mode<PM>() == FOLD_FROM_SPEC) return;
        inner_radix<false>(in_half<PM>() ? R() / 2 : R() / 2 + 1);
    }
    template <int PM = MODE>
    PSTD_HD void p4() {
        if (mode<PM>() == FOLD_TO_SPEC) return;
        inner_radix<true>(out_half<PM>() ? R() / 2 : R() / 2 + 1);
    }

    // velocity slots of pair p: x = the spectrum's real part, y = its
    // imaginary part.  A Dirichlet left wall turns the spectrum by -i, so there
    // the real part belongs to the second line.
    struct Slots {
        float* x;            // uniform bases of the real / imaginary part's lines
        float* y;
        Off up, down;        // byte offsets of bin k (output q: + q M) and bin L - g - k (- q M), from bin s0
        Off step;
        bool okx, oky;
    };
    PSTD_HD Slots slots(int p, int k, bool full) const {
        float* b = base(a.u, N());
        float* c = b + line_step(N());
        const bool A_ = full || va(p), B_ = full || vb(p);
        const bool swap = a.ax.sg < 0.0f;
        Slots s;
        s.x = swap ? c : b;
        s.y = swap ? b : c;
        s.okx = swap ? B_ : A_;
        s.oky = swap ? A_ : B_;
        const Off ps = pos_step(), lof = line_off(p, N());
        s.up = lof + (Off)(k - a.ax.s0) * ps;
        s.down = lof + (Off)(L() - a.ax.g - k - a.ax.s0) * ps;
        s.step = (Off)M() * ps;
        return s;
    }
    // canonical bin of output q of butterfly k
    PSTD_HD int bin(int k, int q) const {
        return 2 * q < R() ? k + M() * q : L() - a.ax.g - k - M() * q;
    }
    // only bin 0 (q = 0) and bin N (q = R/2) may have no slot
    PSTD_HD bool has_slot(int k, int q) const {
        if (q != 0 && 2 * q != R()) return true;
        const int i = bin(k, q) - a.ax.s0;
        return i >= 0 && i < N();
    }
    PSTD_HD Off slot_off(const Slots& s, int q) const {
        return 2 * q < R() ? s.up + (Off)q * s.step : s.down - (Off)q * s.step;
    }
    PSTD_HD float2 load_slot(const Slots& s, int k, int q) const {
        const bool ok = has_slot(k, q);
        const Off off = slot_off(s, q);
        return make_float2(ok && s.okx ? ld(s.x, off) : 0.0f, ok && s.oky ? ld(s.y, off) : 0.0f);
    }
    PSTD_HD void fetch_u() {
        if constexpr (ahead_u) {
            by_full([&](auto full) {
                items(a.ax.nk, [&](int p, int k) {
                    const Slots s = slots(p, k, full);
#pragma unroll
                    for (int q = 0; q < C::R; ++q) uw[q] = load_slot(s, k, q);
                });
            });
        }
    }

    // p3: butterfly k of pair p: radix R, spectral update, radix R
    template <int PM = MODE>
    PSTD_HD void p3() {
        with_even<C::R>(R(), [&](auto RR) {
            constexpr int r_ = decltype(RR)::value;
            constexpr int H = r_ / 2;
            const int nk = a.ax.nk, g = a.ax.g;
            const float sg = a.ax.sg;
            items(nk, [&](int p, int k) {
                const int kb = k + g == 0 ? 0 : M() - g - k;
                const int lk = kloc(k) * ls(), lkb = kloc(kb) * ls();
                const int rs = STR ? S1() * P() : S1();   // next residue
                float2* s = at(0, p);
                float2 w[r_];
                if (mode<PM>() != FOLD_FROM_SPEC) {
                    if (in_half<PM>()) {
#pragma unroll
                        for (int r = 0; r < H; ++r) {
                            const float2 t = tab(&a.ax.th[r * nk + k]);
                            w[r] = cmul(s[r * rs + lk], t);
                            w[r_ - 1 - r] = cscale(cmulc(s[r * rs + lkb], t), -sg);
                        }
                    } else {
                        w[0] = s[lk];
#pragma unroll
                        for (int r = 1; r < H; ++r) {
                            const float2 t = tab(&a.ax.tc[(r - 1) * nk + k]);
                            w[r] = cmul(s[r * rs + lk], t);
                            w[r_ - r] = cscale(cmulc(s[r * rs + lkb], t), sg);
                        }
                        w[H] = cmul(s[H * rs + lk], tab(&a.ax.tc[(H - 1) * nk + k]));
                    }
                    Dft<r_, false>::run(w);
                    if (in_half<PM>()) half_twiddle<r_, false>(w, std::make_integer_sequence<int, r_>{});
                }
                // spectral update; outputs q >= R/2 hold sg x (canonical bin)
                if (stepping<PM>()) {
                    const Slots sl = slots(p, k, nv == 2 * P());
                    if constexpr (!ahead_u) {
                        // all slots are read before any is written (bins of a
                        // self-paired butterfly appear twice)
                        float2 uv[r_];
#pragma unroll
                        for (int q = 0; q < r_; ++q) uv[q] = load_slot(sl, k, q);
                        update(w, uv, sl, k, kb);
                    } else {
                        update(w, uw, sl, k, kb);
                    }
                } else if (mode<PM>() == FOLD_TO_SPEC) {
                    const Slots sl = slots(p, k, false);
#pragma unroll
                    for (int q = 0; q < r_; ++q) {
                        // V = -i X
                        const float sq = 2 * q < r_ ? 1.0f : sg;
                        store_slot(sl, k, kb, q, make_float2(rmul(sq, w[q].y), -rmul(sq, w[q].x)));
                    }
                } else if (mode<PM>() == FOLD_FROM_SPEC) {
                    const Slots sl = slots(p, k, false);
                    const float sc = 1.0f / (float)L();
#pragma unroll
                    for (int q = 0; q < r_; ++q) {
                        const float2 v = load_slot(sl, k, q);
                        const float sq = 2 * q < r_ ? sc : sg * sc;
                        w[q] = make_float2(-rmul(sq, v.y), rmul(sq, v.x));
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < r_; ++q) {
                        // the signs of the canonical bin's two uses cancel
                        const float f = ldc(&(MODE == FOLD_CONV && PM == FOLD_GRAD_U ? a.f2 : a.f)[bin(k, q)]);
                        w[q] = order2<PM>() ? cscale(w[q], f)
                                                     : make_float2(-rmul(f, w[q].y), rmul(f, w[q].x));
                    }
                }
                if (mode<PM>() == FOLD_TO_SPEC) return;
                if (out_half<PM>()) {
                    half_twiddle<r_, true>(w, std::make_integer_sequence<int, r_>{});
                    Dft<r_, true>::run(w);
#pragma unroll
                    for (int r = 0; r < H; ++r) {
                        const float2 t = tab(&a.ax.th[r * nk + k]);
                        s[r * rs + lk] = cmulc(w[r], t);
                        if (k != kb) s[r * rs + lkb] = cscale(cmul(w[r_ - 1 - r], t), -sg);
                    }
                } else {
                    Dft<r_, true>::run(w);
                    s[lk] = w[0];
                    if (k != kb) s[lkb] = cscale(w[0], sg);
#pragma unroll
                    for (int r = 1; r < H; ++r) {
                        const float2 t = tab(&a.ax.tc[(r - 1) * nk + k]);
                        s[r * rs + lk] = cmulc(w[r], t);
                        if (k != kb) s[r * rs + lkb] = cscale(cmul(w[r_ - r], t), sg);
                    }
                    const float2 t = tab(&a.ax.tc[(H - 1) * nk + k]);
                    s[H * rs + lk] = cmulc(w[H], t);
                    if (k != kb) s[H * rs + lkb] = cscale(cmul(w[H], t), sg);
                }
            });
        });
    }
    // V of canonical bin (k, q), written once
    PSTD_HD void store_slot(const Slots& s, int k, int kb, int q, float2 v) const {
        const bool own = 2 * q < R() || k != kb || (2 * q == R() && k == 0);
        const bool ok = own && has_slot(k, q);
        const Off off = slot_off(s, q);
        if (ok && s.okx) put(s.x, off, v.x);
        if (ok && s.oky) put(s.y, off, v.y);
    }
    template <int r_>
    PSTD_HD void update(float2 (&w)[r_], const float2 (&uv)[r_], const Slots& sl, int k, int kb) const {
#pragma unroll
        for (int q = 0; q < r_; ++q) {
            // outputs q >= R/2 take the coefficients times sg (the second half
            // of the table)
            const float2 cf = tab(&a.coef[bin(k, q) + (2 * q < r_ ? 0 : N() + 1)]);
            const float2 v = make_float2(rfma(cf.x, w[q].x, uv[q].x), rfma(cf.x, w[q].y, uv[q].y));
            store_slot(sl, k, kb, q, v);
            w[q] = cscale(v, cf.y);
        }
    }

    // stored output index of position j (element e of residue r): whether it
    // is written, whether through the reflection.  The residues 0 and R/2
    // reflect onto themselves, so only their direct positions are written.
    template <int a_>
    PSTD_HD bool out_index(int e, bool self, int j, bool half, int& i, bool& mir) const {
        const int n = N();
        constexpr bool even = a_ % 2 == 0;
        if (half) {
            mir = even ? 2 * e >= a_ : j >= n;
            i = mir ? 2 * n - 1 - j : j;
            return !conv() || i < a.ax.cN;
        }
        mir = even ? 2 * e >= a_ : j > n;
        i = (mir ? 2 * n - j : j) - a.ax.lo;
        bool ok = !(mir && self);
        if (even ? 2 * e == a_ : j == n) {
            // node N itself is a direct position
            if (j == n) {
                ok = true;
                mir = false;
            }
        }
        if (conv() || !even || e == 0 || 2 * e == a_) ok = ok && i >= 0 && i < a.ax.lp;
        return ok;
    }
    PSTD_HD void fetch_acc() {
        if constexpr (ahead) {
            // (contiguous lines of an axis that is not the last -- the later axes
            // store one node -- add onto the accumulator like strided ones)
            if constexpr (onto_p) {
                if (C::onto_p_only || a.acc_in == a.in) return;
            }
            by_full([&](auto full) {
                const float* xa = base(MODE == FOLD_ORDER2 ? (const float*)a.out : a.acc_in, nout());
                const float* xb = xa + line_step(nout());
                const bool acc = MODE == FOLD_ORDER2 ? a.accumulate != 0 : a.acc_in != nullptr;
                items((C::R / 2 + 1) * C::B, [&](int p, int w) {
                    const int r = w / C::B, t = w - r * C::B, j0 = C::R * t + r;
                    const bool la = full || va(p), lb = full || vb(p);
                    const OutOff oo = out_off(p, j0, false);
#pragma unroll
                    for (int e = 0; e < C::A; ++e) {
                        int i;
                        bool mir;
                        const bool ok =
                            acc && out_index<C::A>(e, r == 0 || 2 * r == C::R, j0 + C::R * C::B * e, false, i, mir);
                        const Off off = oo.at(e, mir);
                        ac[e] = make_float2(ok && la ? ld(xa, off) : 0.0f, ok && lb ? ld(xb, off) : 0.0f);
                    }
                });
            });
        }
    }
    // byte offsets of the output positions j0 + R B e of pair p
    struct OutOff {
        Off direct, mirrored, step;
        PSTD_HD Off at(int e, bool mir) const { return mir ? mirrored - (Off)e * step : direct + (Off)e * step; }
    };
    PSTD_HD OutOff out_off(int p, int j0, bool half) const {
        const Off ps = pos_step(), lof = line_off(p, nout());
        const int lo = half ? 0 : a.ax.lo, refl = half ? 2 * N() - 1 : 2 * N();
        return OutOff{lof + (Off)(j0 - lo) * ps, lof + (Off)(refl - j0 - lo) * ps, (Off)(R() * B()) * ps};
    }
    // p5: residue r, lane t: twiddle, radix A over k1, output positions
    PSTD_HD void p5() {
        if (mode() == FOLD_TO_SPEC) return;
        with_radix<C::A>(A(), [&](auto RA) {
            constexpr int a_ = decltype(RA)::value;
            const bool half = out_half();
            const float rsg = half ? -a.ax.rho : a.ax.rho;
            float* ya = base(a.out, nout());
            float* yb = ya + line_step(nout());
            items((half ? R() / 2 : R() / 2 + 1) * B(), [&](int p, int w) {
                const int r = w / B(), t = w - r * B(), j0 = R() * t + r;
                const float2* s = at(r, p) + Ap() * t * ls();
                float2 x[a_];
#pragma unroll
                for (int k = 0; k < a_; ++k) {
                    x[k] = s[k * ls()];
                    if (k > 0 || a.ax.g) x[k] = cmulc(x[k], tab(&a.ax.tw[k * B() + t]));
                }
                Dft<a_, true>::run(x);
                if (a.ax.g) half_twiddle<a_, true>(x, std::make_integer_sequence<int, a_>{});
                const bool self = !half && (r == 0 || 2 * r == R());
                by_full([&](auto full) {
                    const bool la = full || va(p), lb = full || vb(p);
                    const OutOff oo = out_off(p, j0, half);
                    // Derivatives and the like: the values that outputs are added to,
                    // requested before the first store (which may alias them: one load
                    // after another took 9 us of a 512^2 half-step start).  Run-time
                    // radices above 8 have no registers for it, nor has their step.
                    constexpr bool early = STR && MODE < 0 && (C::fixed || a_ <= 8);
                    float2 old[early ? a_ : 1];
                    if constexpr (early) {
                        if (const float* za = added(ya)) {
                            const float* zb = za + line_step(nout());
#pragma unroll
                            for (int e = 0; e < a_; ++e) {
                                int i;
                                bool mir;
                                const bool ok = out_index<a_>(e, self, j0 + R() * B() * e, half, i, mir);
                                const Off off = oo.at(e, mir);
                                old[e] = make_float2(ok && la ? ld(za, off) : 0.0f, ok && lb ? ld(zb, off) : 0.0f);
                            }
                        }
                    }
#pragma unroll
                    for (int e = 0; e < a_; ++e) {
                        int i;
                        bool mir;
                        const bool ok = out_index<a_>(e, self, j0 + R() * B() * e, half, i, mir);
                        const float sgn = mir ? rsg : 1.0f;
                        if constexpr (STR) {
                            const Off off = oo.at(e, mir);
                            if constexpr (ahead) {
                                const float2 v = make_float2(rfma(sgn, x[e].x, ac[e].x), rfma(sgn, x[e].y, ac[e].y));
                                if (ok && la) put(ya, off, v.x);
                                if (ok && lb) put(yb, off, v.y);
                                if constexpr (keep_p) {
                                    if (a.pout) {
                                        float* qa = base(a.pout, nout());
                                        if (ok && la) put(qa, off, radd(pk[e].x, v.x));
                                        if (ok && lb) put(qa + line_step(nout()), off, radd(pk[e].y, v.y));
                                    }
                                }
                            } else if constexpr (early) {
                                emit(ya + off / 4, ok && la, rmul(sgn, x[e].x), old[e].x);
                                emit(yb + off / 4, ok && lb, rmul(sgn, x[e].y), old[e].y);
                            } else {
                                emit(ya + off / 4, ok && la, rmul(sgn, x[e].x));
                                emit(yb + off / 4, ok && lb, rmul(sgn, x[e].y));
                            }
                        } else {
                            // row position of node (lo + i) or half-node i
                            const int pt = row_pitch(a.ax);
                            float* q = st + 2 * p * pt + row_word(half ? i : i + a.ax.lo);
                            const float2 c = ahead ? make_float2(rfma(sgn, x[e].x, ac[e].x), rfma(sgn, x[e].y, ac[e].y))
                                                   : make_float2(rmul(sgn, x[e].x), rmul(sgn, x[e].y));
                            if (ok) q[0] = c.x;
                            if (ok) q[pt] = c.y;
                        }
                    }
                });
            });
        });
    }
    // Convolution pass, between its two derivatives: residue r, lane t of the
    // half-nodes: the inverse's last radix, u += , and the first radix of the
    // transform of the new u (the same positions).  The new u goes straight to
    // memory (strided) or to the rows.
    PSTD_HD void mid() {
        with_radix<C::A>(A(), [&](auto RA) {
            constexpr int a_ = decltype(RA)::value;
            const float rsg = -a.ax.rho;
            float* ua = base(a.u, nhalf());
            float* ub = ua + line_step(nhalf());
            items(R() / 2 * B(), [&](int p, int w) {
                const int r = w / B(), t = w - r * B(), j0 = R() * t + r, dj = R() * B();
                float2* s = at(r, p) + Ap() * t * ls();
                const bool la = va(p), lb = vb(p);
                const Off ps = pos_step(), lof = line_off(p, nhalf());
                const Off od = lof + (Off)j0 * ps, om = lof + (Off)(2 * N() - 1 - j0) * ps, step = (Off)dj * ps;
                float2 x[a_], u[a_];
#pragma unroll
                for (int e = 0; e < a_; ++e) {
                    int i;
                    bool mir;
                    const bool ok = out_index<a_>(e, false, j0 + dj * e, true, i, mir);
                    const Off off = mir ? om - (Off)e * step : od + (Off)e * step;
                    u[e] = make_float2(ok && la ? ld(ua, off) : 0.0f, ok && lb ? ld(ub, off) : 0.0f);
                }
#pragma unroll
                for (int k = 0; k < a_; ++k) {
                    x[k] = s[k * ls()];
                    if (k > 0) x[k] = cmulc(x[k], tab(&a.ax.tw[k * B() + t]));
                }
                Dft<a_, true>::run(x);
#pragma unroll
                for (int e = 0; e < a_; ++e) {
                    int i;
                    bool mir;
                    const bool ok = out_index<a_>(e, false, j0 + dj * e, true, i, mir);
                    const Off off = mir ? om - (Off)e * step : od + (Off)e * step;
                    const float sgn = mir ? rsg : 1.0f;
                    const float2 v = make_float2(rfma(sgn, x[e].x, u[e].x), rfma(sgn, x[e].y, u[e].y));
                    if constexpr (STR) {
                        if (ok && la) put(ua, off, v.x);
                        if (ok && lb) put(ub, off, v.y);
                    } else if (ok) {
                        float* q = st + 2 * p * row_pitch(a.ax) + row_word(i);
                        q[0] = v.x;
                        q[row_pitch(a.ax)] = v.y;
                    }
                    x[e] = make_float2(ok && la ? rmul(sgn, v.x) : 0.0f, ok && lb ? rmul(sgn, v.y) : 0.0f);
                }
                Dft<a_, false>::run(x);
#pragma unroll
                for (int k = 0; k < a_; ++k) {
                    if (k > 0) x[k] = cmul(x[k], tab(&a.ax.tw[k * B() + t]));
                    s[k * ls()] = x[k];
                }
            });
        });
    }
    // the new u of contiguous lines from their rows
    PSTD_HD void finish_u() {
        if constexpr (!STR) {
            const int len = nhalf(), pitch = row_pitch(a.ax);
            float* y = base(a.u, len);
            const int wid = tid >> 5, lane = tid & 31, nw = (nthr + 31) >> 5;
            for (int l = wid; l < nv; l += nw)
                for (int i = lane; i < len; i += 32) y[l * (int64_t)len + i] = st[l * pitch + row_word(i)];
        }
    }
    // *y = its new value from contribution c
    PSTD_HD void emit(float* y, bool ok, float c) const {
        if (!ok) return;
        const int64_t off = y - a.out;
        if (stepping() || mode() == FOLD_CONV) {
            *y = radd(a.acc_in[off], c);
            return;
        }
        const float v = a.accumulate ? radd(*y, c) : c;
        *y = v;
        if (order2() && a.pout) a.pout[off] = radd(a.in[off], v);
    }
    // what contributions to `y`, in a.out, are added to; null: nothing
    PSTD_HD const float* added(const float* y) const {
        if (stepping() || mode() == FOLD_CONV) return a.acc_in + (y - a.out);
        return a.accumulate ? y : nullptr;
    }
    // the same with that value at hand
    PSTD_HD void emit(float* y, bool ok, float c, float old) const {
        if (!ok) return;
        const float v = stepping() || mode() == FOLD_CONV || a.accumulate ? radd(old, c) : c;
        *y = v;
        if (order2() && a.pout) {
            const int64_t off = y - a.out;
            a.pout[off] = radd(a.in[off], v);
        }
    }
    // contiguous lines from their rows
    PSTD_HD void finish() {
        if constexpr (!STR) {
            if (mode() == FOLD_TO_SPEC) return;
            const int len = nout(), pitch = row_pitch(a.ax), lo = out_half() ? 0 : a.ax.lo;
            float* y = base(a.out, len);
            const int wid = tid >> 5, lane = tid & 31, nw = (nthr + 31) >> 5;
            for (int l = wid; l < nv; l += nw) {
                const float* q = st + l * pitch + row_word(lane + lo);   // + 36 words per 32 positions
                float* z = y + l * (int64_t)len + lane;
                int i = lane;
                if constexpr (MODE < 0) {
                    // (four at a time: loads before stores, as in p5)
                    const float* o = added(z);
                    for (; i + 96 < len; i += 128, q += 144, z += 128) {
                        float old[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) old[k] = o ? o[i - lane + 32 * k] : 0.0f;
#pragma unroll
                        for (int k = 0; k < 4; ++k) emit(z + 32 * k, true, q[36 * k], old[k]);
                    }
                }
                for (; i < len; i += 32, q += 36, z += 32) {
                    if constexpr (ahead) {
                        *z = *q;
                        if (mode() == FOLD_ORDER2 && a.pout) a.pout[z - a.out] = radd(a.in[z - a.out], *q);
                    } else emit(z, true, *q);
                }
            }
        }
    }
    // bring the tables to this SM's L1 before the fields may be touched
    PSTD_HD void warm() const {
#ifdef __CUDA_ARCH__
        if constexpr (C::resident) {
            if (__isShared(a.ax.tw)) return;
        }
        auto touch = [&](const void* p, int bytes) {
            for (int i = tid * 128; i < bytes; i += nthr * 128)
                asm volatile("prefetch.global.L1 [%0];" ::"l"((const char*)p + i));
        };
        touch(a.ax.tw, M() * 8);
        if (in_half() || out_half() || MODE == FOLD_CONV) touch(a.ax.th, R() / 2 * a.ax.nk * 8);
        if (!in_half() || !out_half()) touch(a.ax.tc, R() / 2 * a.ax.nk * 8);
        if (a.coef) touch(a.coef, (N() + 1) * 8);
#endif
    }
};

#ifdef __CUDACC__
template <class C, bool STR, int MODE>
__device__ __forceinline__ void fold_pass(const FoldArgs& a, unsigned item, void* smem, int tid, int nthr) {
#ifdef __CUDA_ARCH__
    Pass<C, STR, MODE> ps(a, item, smem, tid, nthr);
    ps.warm();
    // a pass launched while the previous one drains waits here, before it
    // touches a field; the next one may be scheduled from now on (it waits in
    // turn for this grid to end)
    pdl_wait();
    pdl_trigger();
    if constexpr (MODE == FOLD_CONV) {
        ps.template p1<FOLD_GRAD_P>();
        __syncthreads();
        ps.template p2<FOLD_GRAD_P>();
        __syncthreads();
        ps.template p3<FOLD_GRAD_P>();
        __syncthreads();
        ps.template p4<FOLD_GRAD_P>();
        __syncthreads();
        ps.mid();
        __syncthreads();
        ps.finish_u();
        ps.template p2<FOLD_GRAD_U>();
        __syncthreads();
        ps.template p3<FOLD_GRAD_U>();
        ps.fetch_acc();
        __syncthreads();
        ps.template p4<FOLD_GRAD_U>();
        __syncthreads();
        ps.p5();
        if constexpr (!STR) {
            __syncthreads();
            ps.finish();
        }
        return;
    }
    if constexpr (!STR) ps.fetch_u();
    ps.p1();
    if constexpr (STR) ps.fetch_u();
    __syncthreads();
    ps.p2();
    __syncthreads();
    ps.p3();
    ps.fetch_acc();
    __syncthreads();
    ps.p4();
    __syncthreads();
    ps.p5();
    if constexpr (!STR) {
        __syncthreads();
        ps.finish();
    }
#endif
}
#endif

}  // namespace fold
}  // namespace pstd
