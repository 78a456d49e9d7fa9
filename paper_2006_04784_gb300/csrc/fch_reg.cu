// The passes built for one grid size and precision (fch_reg.cuh). Compiled once per
// (precision, size) with FCH_T, FCH_SUFFIX and FCH_LOGN set (build.py), so that the many
// kernels build in parallel.
#include "fch_reg.cuh"

static_assert(fch::RegCfg<FCH_T, FCH_LOGN, false>::col_blocks == fch_reg_col_blocks(1 << FCH_LOGN, sizeof(FCH_T) == 4),
              "a partial sum for every block of the columns");

namespace {

typedef void (*pass_fn)(const fch_kparams);

inline cudaError_t launch_reg(pass_fn f, int blocks, int threads, int smem, bool &set, cudaStream_t s,
                              const fch_kparams &kp)
{
    if (!set) { // first launch: before any stream capture, like the other passes
        const cudaError_t e = cudaFuncSetAttribute((const void *)f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        set = true;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    fch_pdl_config(cfg, at, dim3((unsigned)blocks, kp.npairs > 1 ? (unsigned)kp.npairs : 1u), dim3((unsigned)threads),
                   (size_t)smem, s, kp.pdl != 0);
    return cudaLaunchKernelEx(&cfg, f, kp);
}

template <typename T, int M, int LOGN> cudaError_t col(const fch_kparams &kp, cudaStream_t s)
{
    typedef fch::RegCfg<T, LOGN, fch::col_xf(M)> G;
    static bool set = false;
    pass_fn f;
    if constexpr (G::cl)
        f = fch::col_pass_rcl<T, M, LOGN>;
    else
        f = fch::col_pass_r<T, M, LOGN>;
    return launch_reg(f, G::col_blocks, G::col_threads, G::col_smem, set, s, kp);
}

template <typename T, int M, int LOGN> cudaError_t row(const fch_kparams &kp, cudaStream_t s)
{
    typedef fch::RegCfg<T, LOGN, fch::row_xf(M)> G;
    static bool set = false;
    return launch_reg(fch::row_pass_r<T, M, LOGN>, G::N / G::rpb, G::row_threads, G::row_smem, set, s, kp);
}

} // namespace

#define FCH_CAT2(a, b, c) a##b##_##c
#define FCH_CAT(a, b, c) FCH_CAT2(a, b, c)
#define FCH_COL(M) \
    case M: return col<FCH_T, M, FCH_LOGN>(kp, s)
#define FCH_ROW(M) \
    case M: return row<FCH_T, M, FCH_LOGN>(kp, s)

cudaError_t FCH_CAT(fch_reg_col_, FCH_SUFFIX, FCH_LOGN)(int mode, const fch_kparams &kp, cudaStream_t s)
{
    switch (mode) {
        FCH_COL(CM_FWD_STORE);
        FCH_COL(CM_INV_LOAD);
        FCH_COL(CM_START);
        FCH_COL(CM_IMEX_SOLVE);
        FCH_COL(CM_F_FINISH);
        FCH_COL(CM_SAV_PQ);
        FCH_COL(CM_SAV_COMBINE);
        FCH_COL(CM_PSD_ITER);
        FCH_COL(CM_ETD_STAGE1);
        FCH_COL(CM_ETD_STAGE2);
    }
    return cudaErrorInvalidValue;
}

cudaError_t FCH_CAT(fch_reg_row_, FCH_SUFFIX, FCH_LOGN)(int mode, const fch_kparams &kp, cudaStream_t s)
{
    switch (mode) {
        FCH_ROW(RM_R2C_LOAD);
        FCH_ROW(RM_C2R_STORE);
        FCH_ROW(RM_NIMEX);
        FCH_ROW(RM_F);
        FCH_ROW(RM_SAV);
        FCH_ROW(RM_ENERGY);
        FCH_ROW(RM_NIMEX_DIRECT);
        FCH_ROW(RM_SAV_DIRECT);
    }
    return cudaErrorInvalidValue;
}
