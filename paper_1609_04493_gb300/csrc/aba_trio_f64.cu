// aba_trio_f64.cu -- the forward-dynamics kernel with three lanes per instance
// (aba_trio.cuh) for FP64 data.
#include "aba_pair_launch.cuh"

int rd_aba_trio_f64(const rd_model *m, int B, const void *q, const void *qd, const void *tau,
                    void *qdd, int *status, void *ws, const double *base18, cudaStream_t s)
{
    return rdyn::launch_aba_multi<double, double, double, 4>(m, B, q, qd, tau, qdd, status, ws,
                                                             base18, s);
}
