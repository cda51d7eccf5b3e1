// pstd_fkernels.cuh -- kernels of the folded passes (pstd_fold.cuh).
//
// Two forms share one source: radices and line pairs per CTA fixed at compile
// time (Cfg, the lengths of pstd_fold_list.h), or read from the plan (AnyCfg,
// every other length with a schedule).  pstd_fold_*.cu
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
    unsigned items[3];
    int ndim;
    int64_t nsteps;
    GridSync sync;
    unsigned tables;         // > 0: a plan's tables are copied to this offset (bytes) of shared memory
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
        fold_pass<OntoP<C>, false, FOLD_STEP>(a, 0, wsm4, threadIdx.x, blockDim.x);
        __syncthreads();
    }
#endif
}
// Run-time radices: every phase holds a switch over them, so registers are those
// of the largest (it spills above radix 10) and offsets are 64-bit; about three
// times slower per point than fixed radices (224^3 442 us per step), still twice
// as fast as the routes these lengths had (112 x 70: 57 -> 22 us).
template <bool STR, int MODE>
__global__ void __launch_bounds__(kAnyThreads, 2) k_fold_any(const __grid_constant__ FoldArgs a) {
    extern __shared__ float4 wsm4[];
    fold_pass<AnyCfg, STR, MODE>(a, blockIdx.x, wsm4, threadIdx.x, blockDim.x);
}

// A whole run as one cooperative kernel (grid and barrier as in
// pstd_persist.cuh), for one plan or a batch: CS and CC are the passes of
// strided and contiguous lines.  Bound by the barrier's round trips (about 3 us a
// pass) and a pass' own chain.  Per step, against run-time radices for every
// length, and the register FFTs before: 512^2 15.4, 42.7, 18.1 us; 256^2 11.6, 29.7,
// 11.3; 128^3 62, 161, 107; 256^3 422, 805, 622; a line of 256 cells 3.1, 11.4, 4.3.
template <class CS, class CC>
constexpr int persist_threads() {
    if (!CS::fixed) return kAnyThreads;
    const int s = cfg_threads<CS>(), c = cfg_threads<CC>();
    return s > c ? s : c;
}
template <class CS, class CC>
constexpr int persist_blocks() {
    if (!CS::fixed) return 2;
    // 32 registers above cfg_blocks' for the loops and the two passes' addresses
    constexpr int m = CS::R > CS::A ? CS::R : CS::A, b = 65536 / ((4 * m + 96) * persist_threads<CS, CC>());
    return b > 8 ? 8 : (b >= 2 ? b : (m <= 10 && persist_threads<CS, CC>() * 2 * 96 <= 65536 ? 2 : 1));
}
template <class CS, class CC>
__global__ void __launch_bounds__(persist_threads<CS, CC>(), persist_blocks<CS, CC>())
    k_fold_persist(const __grid_constant__ FoldPersistArgs a) {
#ifdef __CUDA_ARCH__
    extern __shared__ float4 wsm4[];
    // The passes' arguments in shared memory: through a reference into the
    // parameters or global memory every field is a load of its own (a line of 256
    // cells: 7.9 us per step).  A batch keeps each pass' last member, which for a
    // CTA of one item per pass is found and fetched once a run.
    __shared__ FoldArgs args[3];
    auto fetch = [&](FoldArgs& d, const FoldArgs& src) {
        for (int i = threadIdx.x; i < (int)(sizeof(FoldArgs) / 4); i += blockDim.x)
            ((int*)&d)[i] = ((const int*)&src)[i];
    };
    __shared__ int64_t items[3];
    __shared__ int first[3], own[3];     // members of the first item and of args[k]
    if (!a.members)
        for (int k = 0; k < a.ndim; ++k) fetch(args[k], a.ax[a.ndim - 1 - k]);
    if (threadIdx.x < a.ndim) {
        const int k = threadIdx.x;
        const int64_t* pre = a.prefix + (size_t)k * (a.members + 1);
        items[k] = a.members ? pre[a.members] : (int64_t)a.items[a.ndim - 1 - k];
        first[k] = a.members && blockIdx.x < items[k] ? member_of(pre, a.members, blockIdx.x) : 0;
        own[k] = -1;
    }
    __syncthreads();
    // A barrier's acquire empties L1, so tables read through it arrive from L2 in
    // every pass (256^2: 15.8 us per step).
    if (a.tables) {
        char* to = (char*)wsm4 + a.tables;
        auto keep = [&](const float2*& t, int n) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) ((float2*)to)[i] = t[i];
            __syncthreads();
            if (threadIdx.x == 0) t = (const float2*)to;
            to += n * sizeof(float2);
        };
        for (int k = 0; k < a.ndim; ++k) {
            FoldAxis& x = args[k].ax;
            keep(x.tw, x.M);
            keep(x.tc, x.R / 2 * x.nk);
            keep(args[k].coef, 2 * (x.N + 1));
        }
        __syncthreads();
    }
    unsigned gen = threadIdx.x == 0 ? ld_acquire(a.sync.gen) : 0;
    for (int64_t s = 0; s < a.nsteps; ++s) {
        for (int k = 0; k < a.ndim; ++k) {
            const int64_t* pre = a.prefix + (size_t)k * (a.members + 1);
            const int64_t n = items[k];
            for (int64_t it = blockIdx.x; it < n; it += gridDim.x) {
                unsigned item = (unsigned)it;
                if (a.members) {
                    const int m = it == blockIdx.x ? first[k] : member_of(pre, a.members, it);
                    item = (unsigned)(it - pre[m]);
                    if (m != own[k]) {
                        __syncthreads();         // (every thread has read own)
                        fetch(args[k], a.mem[(size_t)m * 3 + k]);
                        if (threadIdx.x == 0) own[k] = m;
                        __syncthreads();
                    }
                }
                const FoldArgs& w = args[k];
                if (w.ax.inner > 1) fold_pass<Resident<CS>, true, FOLD_STEP>(w, item, wsm4, threadIdx.x, blockDim.x);
                else fold_pass<Resident<CC>, false, FOLD_STEP>(w, item, wsm4, threadIdx.x, blockDim.x);
                __syncthreads();     // shared memory is reused by the next item
            }
            if (!grid_sync(a.sync, gen)) return;
        }
    }
#endif
}

}  // namespace fold

// Lengths 2^k and 3 2^k: those that had kernels of every kind on the register
// FFTs.  Their derivatives and velocity conversions are compiled (256^3: 61 to 65
// us a pass, 115 to 120 on run-time radices, 84 to 133 on the register FFTs; on
// other lengths the run-time radices stand against the shared-memory program:
// 200 x 180 x 150 47 to 57 against 111 to 136), and their cooperative run has a form
// for many lines too (the form for few, 2 and 1 pairs, took 807 us per 256^3 step
// and 145 per 128^3 step).
constexpr bool fold_dyadic(int L) {
    while (L % 2 == 0) L /= 2;
    return L == 1 || L == 3;
}
// Kernel of a schedule (any mode but FOLD_CONV)
// with P pairs per CTA, or null where it is not compiled; one function per
// translation unit.
template <class C, bool STR>
const void* fold_mode(int mode) {
    if (mode == FOLD_STEP) return (const void*)fold::k_fold<C, STR, FOLD_STEP>;
    if (mode == FOLD_ORDER2) return (const void*)fold::k_fold<C, STR, FOLD_ORDER2>;
    if constexpr (fold_dyadic(C::R * C::A * C::B)) return (const void*)fold::k_fold<C, STR, FOLD_MISC>;
    return nullptr;
}
template <int R, int A, int B, int PS, int PC>
const void* fold_fixed(int P, bool strided, int mode) {
    if (mode == FOLD_PERSIST) {
        if (P == 1) return (const void*)fold::k_fold_persist<fold::Cfg<R, A, B, 2>, fold::Cfg<R, A, B, 1>>;
        if constexpr (fold_dyadic(R * A * B))
            return (const void*)fold::k_fold_persist<fold::Cfg<R, A, B, PS>, fold::Cfg<R, A, B, PC>>;
        return nullptr;
    }
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
const void* fold_any_misc_s();
const void* fold_any_misc_c();
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
// The cooperative kernel of an axis and its CTA.  Compiled schedules (`fixed`)
// run 2 line pairs per CTA on strided lines and 1 on contiguous ones or, where
// `many` is set and compiled, the schedule's own PS and PC; the run-time one the
// plan's pairs.
struct FoldPersist {
    const void* kernel;
    int threads;
    bool fixed;
    int PS, PC;
};
FoldPersist fold_persist(const FoldAxis& x, bool many, int PS, int PC);
// CTAs of a pass with p line pairs each
inline int64_t fold_tiles(const FoldAxis& x, bool strided, int p) {
    if (!strided) return (x.nlines + 2 * p - 1) / (2 * p);
    return (x.nlines / x.inner) * ((x.inner + 2 * p - 1) / (2 * p));
}
// Raise the dynamic shared-memory limit of the kernels of axis x.
cudaError_t fold_set_smem(const FoldAxis& x, bool strided, int bytes);

}  // namespace pstd
