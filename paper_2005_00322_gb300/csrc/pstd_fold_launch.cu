// pstd_fold_launch.cu -- kernel choice and launch of the folded passes.
#include "pstd_fkernels.cuh"

namespace pstd {

#define DECL(U) const void* fold_unit_##U(int R, int A, int B, int P, bool strided, int mode);
PSTD_FOLD_UNITS(DECL)
#undef DECL
#define DECL(U) const void* conv_unit_##U(int R, int A, int B, int P, bool strided);
PSTD_CONV_UNITS(DECL)
#undef DECL

const void* fold_kernel(const FoldAxis& x, bool strided, int mode, bool& fixed) {
    fixed = true;
    if (mode == FOLD_CONV) {
#define TRY(U) \
    if (const void* k = conv_unit_##U(x.R, x.A, x.B, x.P, strided)) return k;
        PSTD_CONV_UNITS(TRY)
#undef TRY
        return nullptr;
    }
    if (!x.wide && !x.cN) {
#define TRY(U) \
    if (const void* k = fold_unit_##U(x.R, x.A, x.B, x.P, strided, mode)) return k;
        PSTD_FOLD_UNITS(TRY)
#undef TRY
    }
    fixed = false;
    if (mode == FOLD_LINE) return nullptr;
    if (mode == FOLD_PERSIST) return fold_any_persist();
    if (mode == FOLD_STEP) return fold_any_step(strided);
    return strided ? fold_any_misc_s() : fold_any_misc_c();
}

cudaError_t fold_launch(const FoldArgs& a, bool strided, const FoldLaunch& g, cudaStream_t st, bool overlap) {
    bool fixed = false;
    const void* k = fold_kernel(a.ax, strided, a.mode, fixed);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(g.grid);
    // the run-time form loops over its work, so it takes no more threads than
    // it is compiled for
    cfg.blockDim = dim3(fixed || g.threads < fold::kAnyThreads ? g.threads : fold::kAnyThreads);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = st;
    // passes and conversions follow one another: one may start (and fetch its tables)
    // while the previous one drains; it waits before touching fields.  A derivative
    // is mostly a call of its own with nothing to overlap (512^2 half-step start: 26 us
    // with the attribute and without).
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap && a.mode != FOLD_GRAD_P && a.mode != FOLD_GRAD_U ? 1 : 0;
    void* args[] = {(void*)&a};
    return cudaLaunchKernelExC(&cfg, k, args);
}

bool fold_has_line(const FoldAxis& x) {
    bool fixed = false;
    return x.nlines == 1 && fold_kernel(x, false, FOLD_LINE, fixed) != nullptr;
}
cudaError_t fold_launch_line(const FoldArgs& a, int64_t nsteps, const FoldLaunch& g, cudaStream_t st) {
    bool fixed = false;
    const void* k = fold_kernel(a.ax, false, FOLD_LINE, fixed);
    void* args[] = {(void*)&a, (void*)&nsteps};
    return cudaLaunchKernel(k, dim3(1), dim3(g.threads), args, g.smem, st);
}

FoldPersist fold_persist(const FoldAxis& x, bool many, int PS, int PC) {
    FoldPersist p{};
    FoldAxis y = x;
    y.P = 2;
    if (many) p.kernel = fold_kernel(y, false, FOLD_PERSIST, p.fixed);
    if (many && p.fixed) {
        p.PS = PS;
        p.PC = PC;
    } else {
        y.P = 1;
        p.kernel = fold_kernel(y, false, FOLD_PERSIST, p.fixed);
        p.PS = 2;
        p.PC = 1;
    }
    const int NR = x.R / 2 + 1, nk = x.A * x.B / 2 + 1, m = NR * (x.A > x.B ? x.A : x.B);
    const int P = p.PS > p.PC ? p.PS : p.PC;
    p.threads = p.fixed ? ((m > nk ? m : nk) * P + 31) / 32 * 32 : fold::kAnyThreads;
    return p;
}

cudaError_t fold_set_smem(const FoldAxis& x, bool strided, int bytes) {
    for (int mode : {(int)(x.cN ? FOLD_CONV : FOLD_STEP), (int)FOLD_ORDER2, (int)FOLD_GRAD_P}) {
        if (x.cN && mode == FOLD_ORDER2) continue;
        bool fixed = false;
        const void* k = fold_kernel(x, strided, mode, fixed);
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    if (fold_has_line(x)) {
        bool fixed = false;
        const cudaError_t e = cudaFuncSetAttribute(fold_kernel(x, false, FOLD_LINE, fixed),
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    cudaFuncAttributes fa{};
    const void* k = fold_any_persist();
    cudaError_t e = cudaFuncGetAttributes(&fa, k);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes - (int)fa.sharedSizeBytes);
}

}  // namespace pstd
