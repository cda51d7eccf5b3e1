// pstd_fold_list.h -- schedules of the folded passes compiled with fixed
// radices: every extension length L = 2N with prime factors 2, 3 and 5 from
// N = 24 to 1024 (but 25 and 625) as X(R, A, B, PS, PC), L = R A B, PS / PC
// line pairs per CTA of the strided / contiguous passes where an axis has many
// lines (2 / 1 otherwise).
//
// One rule gives every entry (test_fold_schedules_cpu.py computes it).  With ops(n)
// the real operations of a radix-n butterfly, NR = R/2 + 1 sub-transforms and nk =
// A B / 2 + 1 butterflies, a thread's share of the phases is
//     p1 = ops(A) + 10 A,  p2 = ops(B) + 10 B,  p3 = 2 ops(R) + 20 R
// (a shared-memory round trip, a twiddle and index arithmetic beside the
// butterfly), and the CTA's lanes per pair are the items of the widest phase,
// max(NR max(A, B), nk).  The schedule with the least
//     0.33 lanes (2 p1 + 2 p2 + p3) + 0.67 (2 NR B p1 + 2 NR A p2 + nk p3)
// is taken: idle lanes count a third (a 128^3 step takes 39.0 us with (4, 8, 8),
// whose phases have 24, 24 and 33 items, 41.7 with (8, 4, 8) and its 40, 20 and 17;
// 48^3 7.9 with (6, 4, 4), 9.4 with (8, 3, 4); 810 x 810 x 32 437 with (12, 9, 15), 505
// with (18, 9, 10); 320^2 is the one grid measured where the runner-up is faster, 6.0
// against 6.2 us).  R = 10 competes only where no smaller R stays within 48 lanes:
// at 150 and 180 cells it would cost planes 4 to 10 percent (180 x 512 6.6 us, 6.0 with
// (8, 5, 9)).  R above 10 costs a tenth more (p3 is the longest
// serial phase: a 512^2 step takes 9.5 us with (8, 8, 16), 10.2 with (16, 8, 8)), any
// radix above 10 a fifth more and above 16 twice that (registers).  PS = 8 makes
// each global access of a strided pass a run of 16 words (256^3: 254 us per step
// against 288 with PS = 4); schedules wider than 48 lanes take 4, so that two
// CTAs fit an SM.  PC = 8 up to 20 lanes, 4 below 60, 2 from there (432 cells along
// the contiguous axis of 128 x 128 lines: 109 us per step with 2, 115 with 4; 384^3:
// 1067 against 1120).  Grouped by translation unit (pstd_fold_u*.cu), of like
// compile time.
#pragma once

#define PSTD_FOLD_U0(X) \
    X(6, 3, 3, 8, 8) \
    X(4, 4, 4, 8, 8) \
    X(8, 5, 6, 8, 4) \
    X(10, 5, 5, 8, 4) \
    X(6, 9, 10, 8, 4) \
    X(8, 10, 10, 4, 4) \
    X(10, 9, 12, 4, 2) \
    X(20, 10, 10, 4, 2)
#define PSTD_FOLD_U1(X) \
    X(6, 3, 6, 8, 4) \
    X(6, 3, 9, 8, 4) \
    X(4, 8, 8, 8, 4) \
    X(8, 8, 8, 8, 4) \
    X(10, 5, 15, 4, 2) \
    X(12, 9, 9, 4, 2) \
    X(8, 16, 16, 4, 2)
#define PSTD_FOLD_U2(X) \
    X(8, 3, 3, 8, 8) \
    X(8, 4, 6, 8, 4) \
    X(6, 5, 9, 8, 4) \
    X(8, 8, 9, 8, 4) \
    X(10, 9, 9, 4, 4) \
    X(10, 10, 12, 4, 2) \
    X(18, 9, 12, 4, 2)
#define PSTD_FOLD_U3(X) \
    X(6, 3, 5, 8, 8) \
    X(8, 4, 4, 8, 8) \
    X(10, 5, 8, 8, 4) \
    X(6, 8, 9, 8, 4) \
    X(10, 10, 10, 4, 2) \
    X(8, 12, 12, 4, 2) \
    X(10, 12, 16, 4, 2)
#define PSTD_FOLD_U4(X) \
    X(4, 5, 5, 8, 8) \
    X(8, 5, 5, 8, 4) \
    X(8, 6, 6, 8, 4) \
    X(8, 9, 9, 8, 4) \
    X(8, 9, 10, 4, 4) \
    X(10, 12, 12, 4, 2) \
    X(12, 9, 15, 4, 2)
#define PSTD_FOLD_U5(X) \
    X(4, 3, 4, 8, 8) \
    X(6, 5, 6, 8, 4) \
    X(8, 5, 9, 8, 4) \
    X(10, 5, 9, 4, 4) \
    X(8, 10, 12, 4, 2) \
    X(8, 8, 16, 4, 2) \
    X(10, 12, 15, 4, 2)
#define PSTD_FOLD_U6(X) \
    X(6, 4, 5, 8, 8) \
    X(6, 5, 5, 8, 8) \
    X(6, 8, 8, 8, 4) \
    X(6, 10, 10, 4, 4) \
    X(10, 8, 8, 8, 4) \
    X(18, 9, 9, 4, 2) \
    X(10, 10, 15, 4, 2)
#define PSTD_FOLD_U7(X) \
    X(4, 3, 5, 8, 8) \
    X(6, 6, 6, 8, 4) \
    X(6, 5, 10, 8, 4) \
    X(6, 8, 10, 8, 4) \
    X(8, 9, 12, 4, 2) \
    X(8, 10, 16, 4, 2) \
    X(8, 12, 16, 4, 2)
#define PSTD_FOLD_U8(X) \
    X(4, 4, 5, 8, 8) \
    X(4, 6, 6, 8, 8) \
    X(8, 5, 8, 8, 4) \
    X(6, 9, 9, 8, 4) \
    X(10, 9, 10, 4, 2) \
    X(16, 9, 9, 4, 2) \
    X(10, 10, 16, 4, 2)
#define PSTD_FOLD_U9(X) \
    X(6, 4, 4, 8, 8) \
    X(8, 4, 5, 8, 4) \
    X(6, 6, 9, 8, 4) \
    X(10, 5, 10, 4, 2) \
    X(8, 8, 12, 4, 2) \
    X(10, 9, 15, 4, 2) \
    X(12, 12, 12, 4, 2)
// Embeddings of the convolution passes (lines of N cells with no schedule of
// their own, 65 <= N <= 1280): the smallest length that is at least 4N (two
// neighbours differ by 7 to 17 percent), as X(R, A, B); 2 or 4 line pairs per CTA on strided axes, 1
// on contiguous ones.
#define PSTD_CONV_U0(X) X(8, 6, 6) X(6, 8, 9) X(8, 8, 10) X(10, 10, 10) X(10, 12, 12) X(8, 16, 16) X(12, 15, 16) X(18, 16, 16)
#define PSTD_CONV_U1(X) X(8, 5, 8) X(6, 8, 10) X(8, 9, 10) X(8, 9, 15) X(10, 10, 16) X(10, 15, 15) X(12, 16, 16) X(20, 16, 16)
#define PSTD_CONV_U2(X) X(8, 5, 9) X(8, 8, 8) X(8, 10, 10) X(10, 10, 12) X(12, 12, 12) X(10, 15, 16) X(16, 15, 15)
#define PSTD_CONV_U3(X) X(8, 5, 10) X(8, 8, 9) X(10, 9, 10) X(8, 10, 16) X(10, 12, 16) X(10, 16, 16) X(16, 16, 16)
#define PSTD_CONV_ALL(X) PSTD_CONV_U0(X) PSTD_CONV_U1(X) PSTD_CONV_U2(X) PSTD_CONV_U3(X)
#define PSTD_CONV_UNITS(X) X(0) X(1) X(2) X(3)
#define PSTD_FOLD_ALL(X) PSTD_FOLD_U0(X) PSTD_FOLD_U1(X) PSTD_FOLD_U2(X) PSTD_FOLD_U3(X) PSTD_FOLD_U4(X) PSTD_FOLD_U5(X) PSTD_FOLD_U6(X) PSTD_FOLD_U7(X) PSTD_FOLD_U8(X) PSTD_FOLD_U9(X)
#define PSTD_FOLD_UNITS(X) X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9)
