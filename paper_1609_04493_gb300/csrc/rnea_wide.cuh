// rnea_wide.cuh -- FP64 inverse dynamics of small batches: sixteen lanes per instance,
// the recursions by component, the per-link work by link.
//
// A warp's FP64 instruction holds GB300's FP64 unit for 64 cycles alone and 76 beside
// the other three schedulers', however many of its lanes are active. A batch too small
// to fill the SMs is therefore bound by the number of FP64 instructions of one warp:
// 123 a link with one thread per instance, about 136 a link for the scans of
// rnea_scan.cuh with their combines. Here, per instance (common-normal frames,
// spatial_dh.cuh):
//   1. lane = link: cos, sin and the rotation R_i (12 instructions for 16 links);
//   2. base to tip, lane = component of v, w, a, al (Eq. id-forward): 7 a link;
//   3. lane = link: the bias wrench F_hat_i (51 for 16 links);
//   4. tip to base, lane = component of f, n (Eq. id-backward): 5 a link.
// That is 147 FP64 instructions at n = 7 and 510 at n = 32, counted in the source.
// Exchanges are shuffles and shared memory; profiled at n = 7, B = 1024 they are what
// the warps wait for (short scoreboard 3.4 per issue), the FP64 unit 41% busy. Two instances per warp, one warp per block
// so that blocks spread over the SMs. us, scans / this at B = 1024: n = 7: 29.5 / 10.2,
// n = 16: 36.4 / 17.2, n = 32: 49.6 / 32.6; at B = 4096: 55 / 22, 134 / 38, 181 / 74. From
// about 44 instances per SM the one-thread kernel does the work in fewer
// instructions.
#pragma once
#include "rnea_dhp.cuh"

namespace rdyn {

constexpr int kWideLanes = 16;
constexpr int kWidePerWarp = 32 / kWideLanes;
// doubles per link and instance: R (9), v w a al (12), F_hat (6)
constexpr int kWideScalars = 27;

inline size_t wide_smem(int n) { return (size_t)n * kWideScalars * kWidePerWarp * sizeof(double); }

__device__ __forceinline__ double wide_get(double x, int src)
{
    return __shfl_sync(0xffffffffu, x, src, kWideLanes);
}

// Three values by axis
__device__ __forceinline__ double wide_sel(int k, double a, double b, double c)
{
    return k == 0 ? a : (k == 1 ? b : c);
}

__global__ void __launch_bounds__(32)
rnea_wide_kernel(const double *__restrict__ consts, int n, int B, const double *__restrict__ q,
                 const double *__restrict__ qd, const double *__restrict__ qdd,
                 double *__restrict__ tau, BaseParams<double> base)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & (kWideLanes - 1), slot = threadIdx.x / kWideLanes;
    int b = blockIdx.x * kWidePerWarp + slot;
    const bool live = b < B;
    if (!live) b = B - 1;  // its work again, no output
    double *R = reinterpret_cast<double *>(smem) + (size_t)slot * n * kWideScalars;
    double *mot = R + 9 * n;   // [link][12]: v, w, a, al
    double *wr = mot + 12 * n; // [link][6]: f, n
    const size_t row = (size_t)b * (size_t)n;
    const double *qr = q + row, *qdr = qd + row, *qddr = qdd + row;

    // ---- 1. rotations
    for (int i = lane; i < n; i += kWideLanes) {
        const double *L = consts + i * kDhConsts;
        double s, c;
        sincos_fixed(__ldg(qr + i) + L[5], &s, &c);
        const DhRot<double> r = dh_rot(L[0], L[1], c, s);
        double *o = R + 9 * i;
        o[0] = c;     o[1] = -s;    o[2] = 0.0;
        o[3] = r.sca; o[4] = r.cca; o[5] = -r.sa;
        o[6] = r.ssa; o[7] = r.csa; o[8] = r.ca;
    }
    __syncwarp();

    // ---- 2. motion: lane 4 u + k carries component k of vector u (v, w, a, al)
    const int u = lane >> 2, k = lane & 3, kk = k == 3 ? 0 : k;  // k = 3: idle, repeats 0
    const int k1 = kk == 2 ? 0 : kk + 1, k2 = kk == 0 ? 2 : kk - 1;
    const bool linear = !(u & 1);          // v, a: + (angular) x b
    const int own = 4 * u, ang = 4 * (u | 1);
    double x = u == 0   ? wide_sel(kk, base.V0[0], base.V0[1], base.V0[2])
               : u == 1 ? wide_sel(kk, base.V0[3], base.V0[4], base.V0[5])
               : u == 2 ? wide_sel(kk, base.dV0[0], base.dV0[1], base.dV0[2])
                        : wide_sel(kk, base.dV0[3], base.dV0[4], base.dV0[5]);
    for (int i = 0; i < n; ++i) {
        const double *L = consts + i * kDhConsts;
        const double b1 = linear ? __ldg(L + 2 + k1) : 0.0, b2 = linear ? __ldg(L + 2 + k2) : 0.0;
        const double r0 = R[9 * i + 4 * kk], r1 = R[9 * i + 3 * k1 + kk], r2 = R[9 * i + 3 * k2 + kk];
        const double jd = __ldg(qdr + i), jdd = __ldg(qddr + i);
        // t = x + y x b, then R^T t: column kk of R
        const double y1 = wide_get(x, ang + k1), y2 = wide_get(x, ang + k2);
        const double t = fma(y1, b2, fma(-y2, b1, x));
        double o = fma(r0, t, fma(r1, wide_get(t, own + k1), r2 * wide_get(t, own + k2)));
        // S qd, S qdd; then a, al += qd (v, w) x e_z
        o += kk != 2 || linear ? 0.0 : (u == 1 ? jd : jdd);
        const double z = wide_get(o, 4 * (u & 1) + (kk == 0 ? 1 : 0));
        const double cz = u < 2 || kk == 2 ? 0.0 : (kk == 0 ? jd : -jd);
        x = fma(cz, u < 2 || kk == 2 ? 0.0 : z, o);
        if (k < 3) mot[12 * i + 3 * u + k] = x;
    }
    __syncwarp();

    // ---- 3. bias wrenches
    for (int i = lane; i < n; i += kWideLanes) {
        DhLink<double> L;
        load_dh(consts + i * kDhConsts, L);
        const double *m = mot + 12 * i;
        Motion<double> y;
        y.v = mk3(m[0], m[1], m[2]);
        y.w = mk3(m[3], m[4], m[5]);
        y.a = mk3(m[6], m[7], m[8]);
        y.al = mk3(m[9], m[10], m[11]);
        const Wrench<double> F = bias_wrench(L.m, L.c, L.I, y);
        double *o = wr + 6 * i;
        o[0] = F.f.x; o[1] = F.f.y; o[2] = F.f.z;
        o[3] = F.n.x; o[4] = F.n.y; o[5] = F.n.z;
    }
    __syncwarp();

    // ---- 4. wrenches: lanes 0..2 f, 4..6 n (the others repeat them)
    const int h = u & 1;  // 0: f, 1: n
    double F = h == 0 ? wide_sel(kk, base.Fn[0], base.Fn[1], base.Fn[2])
                      : wide_sel(kk, base.Fn[3], base.Fn[4], base.Fn[5]);
    for (int i = n - 1; i >= 0; --i) {
        const double Fh = wr[6 * i + 3 * h + kk];
        if (i == n - 1) {
            F += Fh;
        } else {
            const double *r = R + 9 * (i + 1) + 3 * kk;  // row kk of R_{i+1}
            const double *L = consts + (i + 1) * kDhConsts;
            const double b1 = __ldg(L + 2 + k1), b2 = __ldg(L + 2 + k2);
            // R f, R n + n_hat
            const double t = fma(r[kk], F, fma(r[k1], wide_get(F, 4 * h + k1),
                                               fma(r[k2], wide_get(F, 4 * h + k2), h ? Fh : 0.0)));
            const double f1 = wide_get(t, k1), f2 = wide_get(t, k2);
            // f: + f_hat; n: + b x (R f)
            F = fma(h ? b1 : 1.0, h ? f2 : Fh, t);
            F = fma(h ? -b2 : 0.0, h ? f1 : 0.0, F);
        }
        if (live && lane == 6) tau[row + i] = F;
    }
}

}  // namespace rdyn
