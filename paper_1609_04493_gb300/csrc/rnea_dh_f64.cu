// rnea_dh_f64.cu -- double instantiations of the common-normal-frame RNEA kernels.
#include "rnea_dh_launch.cuh"
#include "rnea_wide.cuh"

int rd_rnea_dh_f64(const rd_model *m, int B, const void *q, const void *qd, const void *qdd,
                   void *tau, const double *base18, int stored, int block, int fast,
                   int kfull, int tmem, int reg_links, int stages, cudaStream_t s)
{
    return rdyn::dh_launch<double>(m, B, q, qd, qdd, tau, base18, stored != 0, block, false, kfull, tmem != 0, reg_links, stages, s);
}

bool rd_rnea_dhp_f64_fits(const rd_model *m) { return rdyn::dhp_f64_k<double>(m) >= 0; }

int rd_rnea_wide_f64(const rd_model *m, int B, const void *q, const void *qd, const void *qdd,
                     void *tau, const double *base18, cudaStream_t s)
{
    using namespace rdyn;
    static std::atomic<uint64_t> configured{0};
    const uint64_t bit = 1ull << (m->device & 63);
    if (!(configured.load() & bit)) {
        cudaError_t e = cudaFuncSetAttribute(rnea_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)wide_smem(RD_MAX_LINKS));
        if (e != cudaSuccess) return rd_cuda_fail(e, "cudaFuncSetAttribute");
        configured.fetch_or(bit);
    }
    double b[18];
    rd_convert_base_dh(m, base18, b);
    BaseParams<double> base;
    for (int k = 0; k < 6; ++k) {
        base.V0[k] = b[k];
        base.dV0[k] = b[6 + k];
        base.Fn[k] = b[12 + k];
    }
    rd_note_rnea(RD_RNEA_KERNEL_WIDE, 32, m->n);
    const unsigned grid = (unsigned)((B + kWidePerWarp - 1) / kWidePerWarp);
    rnea_wide_kernel<<<grid, 32, wide_smem(m->n), s>>>(
        m->d_dh64, m->n, B, static_cast<const double *>(q), static_cast<const double *>(qd),
        static_cast<const double *>(qdd), static_cast<double *>(tau), base);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return rd_cuda_fail(e, "rnea sixteen-lane kernel launch");
    return RD_OK;
}
