// aba_trio_f32.cu -- instantiations of the forward-dynamics kernel with three
// lanes per instance (aba_trio.cuh).
#include "aba_pair_launch.cuh"

int rd_aba_trio_f32(const rd_model *m, int B, const void *q, const void *qd, const void *tau,
                    void *qdd, int *status, void *ws, const double *base18, bool extended_bias,
                    cudaStream_t s)
{
    using rdyn::DF;
    using rdyn::launch_aba_multi;
    return extended_bias
               ? launch_aba_multi<float, DF, DF, 4>(m, B, q, qd, tau, qdd, status, ws, base18, s)
               : launch_aba_multi<float, DF, float, 4>(m, B, q, qd, tau, qdd, status, ws, base18, s);
}
