// pstd_fkernels.cuh -- kernels of the folded passes (pstd_fold.cuh).
//
// Two forms share one source: radices and line pairs per CTA fixed at compile
// time (Cfg, the lengths of the power-of-two and 3 x 2^k grids), or read from
// the plan (AnyCfg, every other length with a schedule).  pstd_fold_*.cu
// instantiate them; fold_kernel finds the one of a schedule.
#pragma once

#include "pstd_fold.cuh"
#include "pstd_fold_list.h"
#include "pstd_gridsync.cuh"

namespace pstd {

struct FoldLaunch {
    unsigned grid;
    int threads;
    size_t smem;
};

// A whole run as one cooperative kernel: the passes of pstd_persist.cuh's
// schedule (a step's axis passes, last axis first, a grid barrier after each).
struct FoldPersistArgs {
    FoldArgs ax[3];
    int strided[3];
    unsigned items[3];
    int ndim;
    int64_t nsteps;
    GridSync sync;
    int members;             // > 0: a batch, passes and prefix sums in device memory
    const FoldArgs* mem;     // [members][3]
    const int64_t* prefix;   // [3][members + 1]
};

namespace fold {

// threads of a fixed schedule's CTA: one per element group of the widest phase
template <class C>
constexpr int cfg_threads() {
    constexpr int nr = C::R / 2 + 1, m = C::A > C::B ? C::A : C::B, nk = C::A * C::B / 2 + 1;
    return ((nr * m > nk ? nr * m : nk) * C::P + 31) / 32 * 32;
}
// Resident CTAs a schedule is compiled for.  p3 of a step holds a radix-R
// butterfly and the 2R fetched velocity words, p5 a radix-A one and 2A words of
// the accumulator: about 4 max(R, A) + 64 registers.  256^3 (R = A = B = 8,
// 320 threads): 96 registers and 2 CTAs 254 us per step, 64 registers and 3
// CTAs 306 (it spills), 112 and one CTA 313.
template <class C>
constexpr int cfg_blocks() {
    constexpr int m = C::R > C::A ? C::R : C::A, t = cfg_threads<C>();
    constexpr int regs = 4 * m + 64;
    constexpr int b = 65536 / (regs * t);
    return b > 16 ? 16 : (b >= 2 ? b : (t * 2 * 72 <= 65536 ? 2 : 1));
}
constexpr int kAnyThreads = 384;

// One axis pass on fixed radices.  Bound by latency: 256^3 (8, 8, 8) takes 84 to
// 86 us a pass (160 to 250 us on the length-512 complex FFTs before), DRAM 31 to
// 42%, issue 48 to 58%, L1 wavefronts 61% at 20 warps per SM; per point 36
// floating-point, 20 (strided) or 30 (contiguous) integer and 15 memory
// instructions.  Length 768 (8, 8, 12): 384^3 2.23 -> 1.08 ms per step.
// Convolution passes (FOLD_CONV) are bound by instructions, four transforms of
// 4N points and more per pair: 20 uneven 2-D grids 963 -> 300 us per step.
template <class C, bool STR, int MODE>
__global__ void __launch_bounds__(cfg_threads<C>(), cfg_blocks<C>()) k_fold(const __grid_constant__ FoldArgs a) {
    extern __shared__ float4 wsm4[];
    fold_pass<C, STR, MODE>(a, blockIdx.x, wsm4, threadIdx.x, blockDim.x);
}
// All steps of a 1-D run in one CTA: its one line pair is only ever touched by
// this CTA, so a CTA barrier replaces the kernel boundary and p and the slots
// stay in its L1 (line of 256 cells: 2.4 us per step as separate launches, 2.1
// here; bound by one CTA's chain of five phases).
template <class C>
__global__ void __launch_bounds__(cfg_threads<C>()) k_fold_line(const __grid_constant__ FoldArgs a, int64_t nsteps) {
#ifdef __CUDA_ARCH__
    extern __shared__ float4 wsm4[];
    for (int64_t s = 0; s < nsteps; ++s) {
        fold_pass<C, false, FOLD_STEP>(a, 0, wsm4, threadIdx.x, blockDim.x);
        __syncthreads();
    }
#endif
}
// Run-time radices: every phase holds a switch over them, so registers are those
// of the largest (it spills above radix 10) and offsets are 64-bit; about three
// times slower per point than fixed radices (224^3 477 us per step), still twice
// as fast as the routes these lengths had (112 x 70: 57 -> 22 us).
template <bool STR, int MODE>
__global__ void __launch_bounds__(kAnyThreads, 2) k_fold_any(const __grid_constant__ FoldArgs a) {
    extern __shared__ float4 wsm4[];
    fold_pass<AnyCfg, STR, MODE>(a, blockIdx.x, wsm4, threadIdx.x, blockDim.x);
}

}  // namespace fold

// Kernel of a schedule (mode FOLD_STEP, FOLD_ORDER2 or FOLD_LINE) with P pairs
// per CTA, or null where it is not compiled; one function per translation unit.
template <class C, bool STR>
const void* fold_mode(int mode) {
    if (mode == FOLD_STEP) return (const void*)fold::k_fold<C, STR, FOLD_STEP>;
    if (mode == FOLD_ORDER2) return (const void*)fold::k_fold<C, STR, FOLD_ORDER2>;
    return nullptr;
}
template <int R, int A, int B, int PS, int PC>
const void* fold_fixed(int P, bool strided, int mode) {
    if (mode == FOLD_LINE) return P == 1 && !strided ? (const void*)fold::k_fold_line<fold::Cfg<R, A, B, 1>> : nullptr;
    if (strided) {
        if (P == PS) return fold_mode<fold::Cfg<R, A, B, PS>, true>(mode);
        if (P == 2) return fold_mode<fold::Cfg<R, A, B, 2>, true>(mode);
        return nullptr;
    }
    if (P == PC) return fold_mode<fold::Cfg<R, A, B, PC>, false>(mode);
    if (P == 1) return fold_mode<fold::Cfg<R, A, B, 1>, false>(mode);
    return nullptr;
}
#define PSTD_FOLD_CASE(RR, AA, BB, PS, PC) \
    if (R == RR && A == AA && B == BB) return fold_fixed<RR, AA, BB, PS, PC>(P, strided, mode);
#define PSTD_FOLD_UNIT(U)                                                              \
    const void* fold_unit_##U(int R, int A, int B, int P, bool strided, int mode) {    \
        PSTD_FOLD_U##U(PSTD_FOLD_CASE)                                                 \
        return nullptr;                                                                \
    }

// Convolution pass on an embedding's radices (2 or 4 pairs per CTA strided, 1
// contiguous), or null.
template <int R, int A, int B>
const void* conv_fixed(int P, bool strided) {
    if (!strided) return (const void*)fold::k_fold<fold::Cfg<R, A, B, 1>, false, FOLD_CONV>;
    return P == 4 ? (const void*)fold::k_fold<fold::Cfg<R, A, B, 4>, true, FOLD_CONV>
                  : (const void*)fold::k_fold<fold::Cfg<R, A, B, 2>, true, FOLD_CONV>;
}
#define PSTD_CONV_CASE(RR, AA, BB) \
    if (R == RR && A == AA && B == BB) return conv_fixed<RR, AA, BB>(P, strided);
#define PSTD_CONV_UNIT(U)                                                \
    const void* conv_unit_##U(int R, int A, int B, int P, bool strided) {       \
        PSTD_CONV_U##U(PSTD_CONV_CASE)                                   \
        return nullptr;                                                  \
    }

// pstd_fold_any*.cu: the run-time schedules.  mode < 0: one kernel for the
// derivative, conversion and second-order modes.
const void* fold_any_step(bool strided);
const void* fold_any_misc(bool strided);
const void* fold_any_persist();

// Kernel of axis x in `mode`; whether it is a fixed schedule's.
const void* fold_kernel(const FoldAxis& x, bool strided, int mode, bool& fixed);
// overlap: a step's pass may start while the previous launch of its stream
// drains (programmatic stream serialisation)
cudaError_t fold_launch(const FoldArgs& a, bool strided, const FoldLaunch& g, cudaStream_t st, bool overlap = true);
// `nsteps` steps of a 1-D run as one launch; false where its schedule has no
// such kernel.
bool fold_has_line(const FoldAxis& x);
cudaError_t fold_launch_line(const FoldArgs& a, int64_t nsteps, const FoldLaunch& g, cudaStream_t st);
// Raise the dynamic shared-memory limit of the kernels of axis x.
cudaError_t fold_set_smem(const FoldAxis& x, bool strided, int bytes);

}  // namespace pstd
