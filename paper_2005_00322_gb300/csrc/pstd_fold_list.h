// pstd_fold_list.h -- schedules of the folded passes compiled with fixed
// radices: every extension length L = 2N with prime factors 2, 3 and 5 from
// N = 24 to 1024 (but 25 and 625) as X(R, A, B, PS, PC), L = R A B, PS / PC
// line pairs per CTA of the strided / contiguous passes where an axis has many
// lines (2 / 1 otherwise).  The radices minimise butterfly operations plus
// shared-memory round trips, with a penalty on a large R (p3 is the longest
// serial phase: a 512^2 step takes 9.5 us with (8, 8, 16) and 10.2 with
// (16, 8, 8), 512 x 512 x 16 196 and 221), on radices above 10 (registers) and
// on phases that leave lanes idle.  PS = 8 makes each global access of a
// strided pass a run of 16 words (256^3: 254 us per step against 288 with
// PS = 4); schedules wider than 48 lanes per pair take 4, so that two CTAs fit
// an SM.  Measured choices against the rule: 256 (128^3: 39.0 us per step with
// (4, 8, 8), whose phases have 24, 24 and 33 lanes, 41.7 with (8, 4, 8) and its
// 40, 20 and 17), 400 (200 x 180 x 150: 110 against 116 with (8, 5, 10)) and
// PC = 2 at 768 (384^3: 1067 against 1120).  Grouped by translation unit (pstd_fold_u*.cu), of like compile time.
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
    X(12, 9, 9, 4, 4) \
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
    X(10, 10, 10, 4, 4) \
    X(8, 12, 12, 4, 2) \
    X(10, 12, 16, 4, 2)
#define PSTD_FOLD_U4(X) \
    X(4, 5, 5, 8, 8) \
    X(8, 5, 5, 8, 4) \
    X(8, 6, 6, 8, 4) \
    X(8, 9, 9, 8, 4) \
    X(8, 9, 10, 4, 4) \
    X(10, 12, 12, 4, 2) \
    X(18, 9, 10, 4, 2)
#define PSTD_FOLD_U5(X) \
    X(8, 2, 3, 8, 8) \
    X(6, 5, 6, 8, 4) \
    X(8, 5, 9, 8, 4) \
    X(10, 5, 9, 4, 4) \
    X(8, 10, 12, 4, 4) \
    X(8, 8, 16, 4, 2) \
    X(10, 12, 15, 4, 2)
#define PSTD_FOLD_U6(X) \
    X(8, 3, 5, 8, 4) \
    X(6, 5, 5, 8, 8) \
    X(6, 8, 8, 8, 4) \
    X(6, 10, 10, 4, 4) \
    X(8, 8, 10, 4, 4) \
    X(18, 9, 9, 4, 2) \
    X(10, 10, 15, 4, 2)
#define PSTD_FOLD_U7(X) \
    X(6, 2, 5, 8, 8) \
    X(6, 6, 6, 8, 4) \
    X(6, 5, 10, 8, 4) \
    X(6, 8, 10, 8, 4) \
    X(8, 9, 12, 4, 4) \
    X(8, 10, 16, 4, 2) \
    X(8, 12, 16, 4, 2)
#define PSTD_FOLD_U8(X) \
    X(8, 2, 5, 8, 4) \
    X(8, 3, 6, 8, 4) \
    X(8, 5, 8, 8, 4) \
    X(6, 9, 9, 8, 4) \
    X(10, 9, 10, 4, 4) \
    X(16, 9, 9, 4, 2) \
    X(10, 10, 16, 4, 2)
#define PSTD_FOLD_U9(X) \
    X(8, 3, 4, 8, 8) \
    X(8, 4, 5, 8, 4) \
    X(6, 6, 9, 8, 4) \
    X(10, 5, 10, 4, 4) \
    X(8, 8, 12, 4, 2) \
    X(10, 9, 15, 4, 2) \
    X(12, 12, 12, 4, 2)
// Embeddings of the convolution passes (lines of N cells with no schedule of
// their own, 65 <= N <= 1280): the smallest length that is at least 4N, 4 to
// 12 percent apart, as X(R, A, B); 2 or 4 line pairs per CTA on strided axes, 1
// on contiguous ones.
#define PSTD_CONV_U0(X) X(8, 6, 6) X(6, 8, 9) X(8, 8, 10) X(10, 10, 10) X(10, 12, 12) X(8, 16, 16) X(12, 15, 16) X(18, 16, 16)
#define PSTD_CONV_U1(X) X(8, 5, 8) X(6, 8, 10) X(8, 9, 10) X(8, 9, 15) X(10, 10, 16) X(10, 15, 15) X(12, 16, 16) X(20, 16, 16)
#define PSTD_CONV_U2(X) X(8, 5, 9) X(8, 8, 8) X(8, 10, 10) X(10, 10, 12) X(12, 12, 12) X(10, 15, 16) X(16, 15, 15)
#define PSTD_CONV_U3(X) X(8, 5, 10) X(8, 8, 9) X(10, 9, 10) X(8, 10, 16) X(10, 12, 16) X(10, 16, 16) X(16, 16, 16)
#define PSTD_CONV_ALL(X) PSTD_CONV_U0(X) PSTD_CONV_U1(X) PSTD_CONV_U2(X) PSTD_CONV_U3(X)
#define PSTD_CONV_UNITS(X) X(0) X(1) X(2) X(3)
#define PSTD_FOLD_ALL(X) PSTD_FOLD_U0(X) PSTD_FOLD_U1(X) PSTD_FOLD_U2(X) PSTD_FOLD_U3(X) PSTD_FOLD_U4(X) PSTD_FOLD_U5(X) PSTD_FOLD_U6(X) PSTD_FOLD_U7(X) PSTD_FOLD_U8(X) PSTD_FOLD_U9(X)
#define PSTD_FOLD_UNITS(X) X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9)
