// aba_trio.cuh -- forward dynamics (aba_dh.cuh) with three lanes per instance, one
// per axis, for the articulated-inertia recursion and the solves, beside a warp
// (or a second set of lanes) for the bias sweeps.
//
// With J_hat = [[A, Bm], [Bm^T, C]], lane k of an instance holds column k of A,
// row k of Bm and column k of C: nine values. The update of Eq. (abi),
//     J_hat_i = J_i + X^T P X,   P = J_hat_{i+1} - U U^T / Omega_{i+1},
// X = Ad_{f^-1}, f = (R, b), then runs the same instructions on every lane:
//   P        each lane corrects its own nine values (its own U_v[k], U_w[k]
//            against the others');
//   A_r      = R A R^T as R (R A)^T: two 3x3 products of the lane's column with
//            one transpose between them;
//   B_r      = R Bm R^T: R times the lane's row, then its own row of R against
//            all rows;
//   C_r      as A_r, on P's xy part;
//   shift    row k of PT = ([b] A_r)^T is b x (column k of A_r); with
//            Bh = B_r + PT / 2 and Y = [b] Bh,
//            Bm' = B_r + PT - [m c],  C' = C_r + Y + Y^T + C_o,  A' = A_r + m I
//            (Y + Y^T = [b]B_r + ([b]B_r)^T - [b] A_r [b], as the last is
//            symmetric).
// The solves (z_hat and c_hat tip to base, lambda and qdd base to tip) follow in
// the same lanes, each with its component of z_hat and lambda.
// Exchanges (transposes, broadcasts) go through shared memory, each value
// written once by its owner, in rows of 33 so that the gathers do not conflict;
// a lane group never leaves its warp, so __syncwarp orders them. Sums of products
// in D are formed as one: in double-float every product's error and every partial
// sum's error are added up and renormalised once (df.cuh).
//
// The bias sweeps (motion, wrenches, tau_hat) depend on no inertia, so another
// warp runs them at the same time; one __syncthreads hands tau_hat over before the
// solves. No thread spins on another.
//
// What bounds it: FP32 issue and, below one block per SM, the dependent chains of
// the double-float updates (1.57 k warp instructions a link for ten instances, bias
// included, of which 1.1 k on the FMA pipe; issue 65% with 3.1 warps per scheduler, few
// instruction-fetch stalls: 0.09 per issue against 0.97 with two warps per 32
// instances; one thread per instance runs 2.2 k straight-line instructions a link).
// Splitting by axis costs
// half as many instructions again per instance, but three times as many warps
// run half the code each. us, GB300, FP32 data, two or three warps per 32
// instances before / now: n = 7: B = 1024 17.6 / 13.2, 16384 28.8 / 23.7; n = 64:
// B = 64 160 / 108, 1024 164 / 110, 4096 233 / 110, 16384 286 / 216; n = 100
// (double-float bias): B = 64 321 / 224, 4096 516 / 291, 16384 822 / 704. The
// records are staged in shared memory (n = 64, B = 4096: 112 against 144 us from
// global memory), the solves' inputs through a ring (112 against 126 with a ring
// of two links).
//   Bias in T: one thread per instance, operation for operation the sweeps of
//   aba_pair.cuh; block of four warps, 0..2 with ten instances each, 3 with the
//   bias of the thirty.
//   Bias in double-float (chains beyond RD_ABA_EXTENDED_BIAS_LINKS): three lanes
//   per instance there too; block of four warps, 0 and 1 with ten instances each, 2
//   and 3 with their bias.
// Lanes 30 and 31 of a three-lane warp repeat the work of lanes 27 and 28 and
// write nothing.
//
#pragma once
#include <cuda_pipeline.h>

#include "aba_pair.cuh"

namespace rdyn {

constexpr int kTrioPerWarp = 10;
constexpr int kTrioInstances = 3 * kTrioPerWarp;  // per block
constexpr int kTrioStride = 33;
constexpr int kTrioSlots = 17;

// Exchange rows of one warp.
template <typename D>
struct TrioShared {
    D x[kTrioSlots * kTrioStride];
};

// Ring of the solves' per-link inputs, each lane its own: U_v[k], U_w[k],
// 1 / Omega, tau_hat or c_hat, cos, sin. Filled by asynchronous copies
// kTrioRing - 1 links ahead, since the values come from L2 and a link's step is
// shorter than that latency.
constexpr int kTrioRing = 4;

template <typename D, typename TB>
struct TrioRing {
    D v[kTrioRing][4][32];
    TB cs[kTrioRing][2][32];
};

template <typename V>
__device__ __forceinline__ void trio_copy(V *dst, const V *src)
{
    static_assert(sizeof(V) == 4 || sizeof(V) == 8, "4- and 8-byte copies");
    __pipeline_memcpy_async(dst, src, sizeof(V));
}

template <typename D>
__device__ __forceinline__ D sel3(int k, D a, D b, D c)
{
    return k == 0 ? a : (k == 1 ? b : c);
}

// R = Rx(alpha) Rz(theta) as two plane rotations. S: type of cos and sin of theta
// (float when they carry no low part).
template <typename D, typename S>
struct TrioRot {
    S c, s;
    D ca, sa;
};

// R x, and R x for x_2 = 0 (unnormalised)
template <typename D, typename S>
__device__ __forceinline__ void trio_mul(const TrioRot<D, S> &R, const D x[3], D y[3])
{
    const D u = ddot2_raw(R.s, x[0], R.c, x[1]);
    y[0] = ddot2_raw(R.c, x[0], -R.s, x[1]);
    y[1] = ddot2_raw(R.ca, u, -R.sa, x[2]);
    y[2] = ddot2_raw(R.sa, u, R.ca, x[2]);
}

template <typename D, typename S>
__device__ __forceinline__ void trio_mul_xy(const TrioRot<D, S> &R, D x0, D x1, D y[3])
{
    const D u = ddot2_raw(R.s, x0, R.c, x1);
    y[0] = ddot2_raw(R.c, x0, -R.s, x1);
    y[1] = dmul_raw(R.ca, u);
    y[2] = dmul_raw(R.sa, u);
}

// Row k of R: (c, -s, 0), (s ca, c ca, -sa), (s sa, c sa, ca).
template <typename D, typename S>
__device__ __forceinline__ void trio_row(int k, D ca, D sa, S c, S s, D row[3])
{
    const D ax = k == 1 ? ca : sa;
    const D p = dmul_raw(s, ax), q = dmul_raw(c, ax);
    row[0] = k == 0 ? dcvt<D>(c) : p;
    row[1] = k == 0 ? dcvt<D>(-s) : q;
    row[2] = sel3(k, D(0), -sa, ca);
}

// Component k of a x b for a lane that holds (or reads) the others': k1 and k2 are
// the axes after and before k.
template <typename D>
__device__ __forceinline__ D trio_cross(D a1, D a2, D b1, D b2)
{
    return ddot2_raw(a1, b2, -a2, b1);
}

// A lane's place: its axis k, the next and the previous axis, its group's first
// lane, and whether it writes results.
struct TrioLane {
    int k, k1, k2, base;
    bool live;
};

__device__ __forceinline__ TrioLane trio_lane(int lane)
{
    TrioLane t;
    const int g = lane < 30 ? lane / 3 : kTrioPerWarp - 1;
    t.base = 3 * g;
    t.k = lane < 30 ? lane - t.base : lane - 30;
    t.k1 = t.k == 2 ? 0 : t.k + 1;
    t.k2 = t.k == 0 ? 2 : t.k - 1;
    t.live = lane < 30;
    return t;
}

// tau_hat_i in the bias workspace: T with D = T one scalar, FP32 two (the exact
// difference of two floats, or a rounded double-float); with double-float bias
// state the pair in slot 0, whose F_hat the carry has consumed.
template <typename D, typename T, typename TB>
__device__ __forceinline__ void trio_tau_put(T *ws, int B, int b, int i, TB F_nz, T tau)
{
    if constexpr (!std::is_same<TB, T>::value) {
        bias_put<TB>(ws, B, b, i, 0, DF(tau) - F_nz);
    } else if constexpr (sizeof(T) == 4) {
        const DF t = df_two_sum(tau, -F_nz);
        aba_put(ws, B, b, i, 6, t.hi);
        aba_put(ws, B, b, i, 7, t.lo);
    } else {
        aba_put(ws, B, b, i, 6, tau - F_nz);
    }
}

// Address of component k of link i's bias state; k = -1, -2: tau_hat's scalars
// of trio_tau_put.
template <typename TB, typename T>
__device__ __forceinline__ const TB *bias_at(const T *ws, int B, int b, int i, int k)
{
    if constexpr (std::is_same<TB, T>::value)
        return &ws[((size_t)i * kAbaStateScalars + (k < 0 ? 5 - k : k < 6 ? k : k + 2)) * (size_t)B + b];
    else
        return reinterpret_cast<const TB *>(ws) + ((size_t)i * kAbaBiasPairs + k) * (size_t)B + b;
}

// The inertia recursion of one warp's ten instances. sc, sd, sdf, qr: this lane's
// instance's constants, records and joint angles; n: its links; (wsz, B, b): its
// solve slots; L: its place. nmax: the longest chain of the warp (the loop bound,
// the same for every lane; RAGGED: chains of different lengths). U_i and
// 1 / Omega_i go to the workspace. Returns 1 if some Omega_i was not positive.
template <typename T, typename D, typename TB, int TRIG, bool RAGGED>
__device__ __forceinline__ int aba_trio_j(const T *__restrict__ sc, const D *__restrict__ sd,
                                          const DF *__restrict__ sdf, int n, int nmax,
                                          const T *__restrict__ qr, D *__restrict__ wsz, int B,
                                          int b, const TrioLane &L, TrioShared<D> &sh)
{
    const int k = L.k, k1 = L.k1, k2 = L.k2, base = L.base;
    const bool live = L.live;
    D *const own = &sh.x[threadIdx.x & 31];  // slot s of this lane: own[s * kTrioStride]
    const D *const grp = &sh.x[base];        // slot s of lane l of the group: grp[s * stride + l]
    const int co[3] = {19 + sel3(k, 0, 3, 4), 19 + sel3(k, 3, 1, 5), 19 + sel3(k, 4, 5, 2)};
    const D zero = D(0);
    D a[3], be[3], c[3], uv = zero, uw = zero, invOm = zero;
    TB ts = TB(0), tc = TB(0);
    T qv = T(0);
    int bad = 0, tg = 3;
    // J_i's own contributions: -[m c] row k, C_o column k
    auto mc_row = [&](const D *ri, D e[3]) {
        const D p = ri[16 + k2], m = -ri[16 + k1];  // row k: +mc_{k+2} at k+1, -mc_{k+1} at k+2
        e[0] = sel3(k, zero, m, p);
        e[1] = sel3(k, p, zero, m);
        e[2] = sel3(k, m, p, zero);
    };
#pragma unroll
    for (int j = 0; j < 3; ++j) a[j] = be[j] = c[j] = zero;
#pragma unroll 1
    for (int i = nmax - 1; i >= 0; --i) {
        const bool in = !RAGGED || i < n;
        const int ii = !RAGGED || in ? i : n - 1;  // clamped: loads stay in the chain
        const D *ri = sd + ii * kAbaDh64;
        if (RAGGED && ii > 0) {
            prefetch_l1(sd + (ii - 1) * kAbaDh64);
            prefetch_l1(sd + (ii - 1) * kAbaDh64 + kAbaDh64 / 2);
        }
        const T qn = __ldg(qr + ii);  // for the next step
        const D m = ri[6];
        D e[3];
        mc_row(ri, e);
        const D C0 = ri[co[0]], C1 = ri[co[1]], C2 = ri[co[2]];
        if (i != nmax - 1) {
            const int iu = !RAGGED || i + 1 < n ? i + 1 : n - 1;
            const D *r = sd + iu * kAbaDh64;
            TB s1, c1;
            if constexpr (std::is_same<TB, T>::value) {
                dh_trig<T, TRIG>(qv + sc[iu * kDhConsts + 5], &s1, &c1);
            } else {
                // double-float sin/cos: each lane of the group evaluates one
                // link's for the next three steps
                if (tg == 3) {
                    const int u = i + 1 - k > 0 ? i + 1 - k : 0;
                    const int it = !RAGGED || u < n ? u : n - 1;
                    aba_trig_tb<T, TB, TRIG>(sc, sdf, qr, it, ts, tc);
                    tg = 0;
                }
                s1 = df_shfl(ts, base + tg);
                c1 = df_shfl(tc, base + tg);
                ++tg;
            }
            using S = decltype(dscalar<D>(c1));
            const TrioRot<D, S> R{dscalar<D>(c1), dscalar<D>(s1), r[0], r[1]};
            const D b0 = r[2], b1 = r[3], b2 = r[4];
            // P: U_{i+1} of the three lanes is in slots 15, 16
            const D U0 = grp[15 * kTrioStride], U1 = grp[15 * kTrioStride + 1],
                    U2 = grp[15 * kTrioStride + 2];
            const D W0 = grp[16 * kTrioStride], W1 = grp[16 * kTrioStride + 1];
            const D nu = -dmul_raw(uv, invOm), nw = -dmul_raw(uw, invOm);
            a[0] = dfma_raw(nu, U0, a[0]);
            a[1] = dfma_raw(nu, U1, a[1]);
            a[2] = dfma_raw(nu, U2, a[2]);
            be[0] = dfma_raw(nu, W0, be[0]);
            be[1] = dfma_raw(nu, W1, be[1]);
            c[0] = k == 2 ? zero : dfma_raw(nw, W0, c[0]);  // P's w_z column vanishes
            c[1] = k == 2 ? zero : dfma_raw(nw, W1, c[1]);
            // first products: R A, Bm R^T (by rows), R C
            D t[3], u[3], v[3];
            trio_mul(R, a, t);
            trio_mul_xy(R, be[0], be[1], u);
            trio_mul_xy(R, c[0], c[1], v);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                own[j * kTrioStride] = t[j];
                own[(3 + j) * kTrioStride] = u[j];
                own[(6 + j) * kTrioStride] = v[j];
            }
            __syncwarp();
            // second products
#pragma unroll
            for (int l = 0; l < 3; ++l) t[l] = grp[k * kTrioStride + l];
            trio_mul(R, t, a);
            D Rk[3];
            trio_row(k, R.ca, R.sa, R.c, R.s, Rk);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const D *g = grp + (3 + j) * kTrioStride;
                be[j] = ddot3_raw(Rk[0], g[0], Rk[1], g[1], Rk[2], g[2]);
            }
            trio_mul_xy(R, grp[(6 + k) * kTrioStride], grp[(6 + k) * kTrioStride + 1], c);
            // shift: PT row k, Bh row k
            const D h[3] = {dhalf(ddot2_raw(b1, a[2], -b2, a[1])),
                            dhalf(ddot2_raw(b2, a[0], -b0, a[2])),
                            dhalf(ddot2_raw(b0, a[1], -b1, a[0]))};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                be[j] = dsum2_raw(be[j], h[j]);
                own[(9 + j) * kTrioStride] = be[j];
            }
            __syncwarp();
#pragma unroll
            for (int l = 0; l < 3; ++l) t[l] = grp[(9 + k) * kTrioStride + l];  // Bh column k
            const D y[3] = {ddot2_raw(b1, t[2], -b2, t[1]), ddot2_raw(b2, t[0], -b0, t[2]),
                            ddot2_raw(b0, t[1], -b1, t[0])};
#pragma unroll
            for (int j = 0; j < 3; ++j) own[(12 + j) * kTrioStride] = y[j];
            __syncwarp();
            const D C[3] = {C0, C1, C2};
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                c[l] = df_renorm(dsum4_raw(c[l], y[l], grp[(12 + k) * kTrioStride + l], C[l]));
                be[l] = df_renorm(dsum3_raw(be[l], h[l], e[l]));
                a[l] = df_renorm(a[l]);
            }
            const D ak = sel3(k, a[0], a[1], a[2]) + m;
            a[0] = k == 0 ? ak : a[0];
            a[1] = k == 1 ? ak : a[1];
            a[2] = k == 2 ? ak : a[2];
        }
        if (i == nmax - 1 || (RAGGED && i >= n - 1)) {  // the tip: J_i alone
            a[0] = k == 0 ? m : zero;
            a[1] = k == 1 ? m : zero;
            a[2] = k == 2 ? m : zero;
            be[0] = e[0]; be[1] = e[1]; be[2] = e[2];
            c[0] = C0; c[1] = C1; c[2] = C2;
        }
        qv = qn;
        // U_i = J_hat_i S: the last column of Bm, of C
        uv = be[2];
        uw = c[2];
        own[15 * kTrioStride] = uv;
        own[16 * kTrioStride] = uw;
        __syncwarp();
        const D Om = grp[16 * kTrioStride + 2];
        if (in && !dpositive(Om)) bad = 1;
        invOm = drecip(Om);
        if (live && in) {
            aba_zput(wsz, B, b, i, k, uv);
            aba_zput(wsz, B, b, i, 3 + k, uw);
            if (k == 0) aba_zput(wsz, B, b, i, 7, invOm);
        }
    }
    return bad;
}

// The solves of one warp's ten instances, after the inertia recursion and the bias
// sweeps: z_hat and c_hat tip to base, lambda and qdd base to tip (Eq.
// recursive-fd), each lane with its component. Returns 1 on a NaN.
template <typename T, typename D, typename TB, bool RAGGED>
__device__ __forceinline__ int aba_trio_solve(const D *__restrict__ sd, int n, int nmax,
                                              T *__restrict__ qddr, const T *ws, D *wsz, int B,
                                              int b, const TrioLane &L, TrioShared<D> &sh,
                                              TrioRing<D, TB> &rg)
{
    static_assert(std::is_same<D, DF>::value || std::is_same<D, T>::value, "FP32 data: double-float");
    using S = decltype(dscalar<D>(TB(0)));
    const int k = L.k, k1 = L.k1, k2 = L.k2;
    D *const own = &sh.x[threadIdx.x & 31];
    const D *const grp = &sh.x[L.base];
    const D zero = D(0);
    auto at = [&](int slot, int l) -> D { return grp[slot * kTrioStride + l]; };
    const int lane = threadIdx.x & 31;
    // step u of a sweep reads link i(u) and, SECOND, c_hat instead of tau_hat
    auto fetch = [&](int u, int i, bool second) {
        if (u < nmax) {
            const int ii = !RAGGED || i < n ? i : n - 1, slot = u % kTrioRing;
            auto zsrc = [&](int c) { return &wsz[((size_t)ii * kAbaSolveScalars + c) * (size_t)B + b]; };
            trio_copy(&rg.v[slot][0][lane], zsrc(k));
            trio_copy(&rg.v[slot][1][lane], zsrc(3 + k));
            trio_copy(&rg.v[slot][2][lane], zsrc(7));
            if (second) {
                trio_copy(&rg.v[slot][3][lane], zsrc(6));
            } else if constexpr (!std::is_same<TB, T>::value) {
                trio_copy(reinterpret_cast<TB *>(&rg.v[slot][3][lane]), bias_at<TB>(ws, B, b, ii, 0));
            } else {
                T *t = reinterpret_cast<T *>(&rg.v[slot][3][lane]);
                trio_copy(t, bias_at<TB>(ws, B, b, ii, -1));
                if (sizeof(T) == 4) trio_copy(t + 1, bias_at<TB>(ws, B, b, ii, -2));
            }
            trio_copy(&rg.cs[slot][0][lane], bias_at<TB>(ws, B, b, ii, 6));
            trio_copy(&rg.cs[slot][1][lane], bias_at<TB>(ws, B, b, ii, 7));
        }
        __pipeline_commit();
    };
    struct SolveIn {
        D uv, uw, iom, t;  // t: tau_hat, then c_hat
        S c, s;
    };
    auto take = [&](int u) -> SolveIn {
        __pipeline_wait_prior(kTrioRing - 2);
        const int slot = u % kTrioRing;
        SolveIn r;
        r.uv = rg.v[slot][0][lane];
        r.uw = rg.v[slot][1][lane];
        r.iom = rg.v[slot][2][lane];
        r.t = rg.v[slot][3][lane];
        r.c = dscalar<D>(rg.cs[slot][0][lane]);
        r.s = dscalar<D>(rg.cs[slot][1][lane]);
        return r;
    };
    // ---- z_hat_i = X^T (z_hat_{i+1} + U_{i+1} c_hat_{i+1}),
    //      c_hat_i = (tau_hat_i - S^T z_hat_i) / Omega_i
    D zf = zero, zn = zero, uv = zero, uw = zero, chat = zero;
    D Rk[3] = {zero, zero, zero}, bk1 = zero, bk2 = zero;  // row k of R, b of link i+1
#pragma unroll
    for (int u = 0; u < kTrioRing - 1; ++u) fetch(u, nmax - 1 - u, false);
#pragma unroll 1
    for (int i = nmax - 1; i >= 0; --i) {
        const bool in = !RAGGED || i < n;
        const int ii = !RAGGED || in ? i : n - 1;
        const D *r = sd + ii * kAbaDh64;
        const int u = nmax - 1 - i;
        if (RAGGED && ii > 0) prefetch_l1(sd + (ii - 1) * kAbaDh64);
        const SolveIn cur = take(u);
        fetch(u + kTrioRing - 1, i - (kTrioRing - 1), false);
        const S c = cur.c, s = cur.s;
        const D ca = r[0], sa = r[1];
        const D nb1 = r[2 + k1], nb2 = r[2 + k2];
        if (i != nmax - 1) {
            own[0] = dfma_raw(uv, chat, zf);
            own[kTrioStride] = dfma_raw(uw, chat, zn);
            __syncwarp();
            zf = df_renorm(ddot3_raw(Rk[0], at(0, 0), Rk[1], at(0, 1), Rk[2], at(0, 2)));
            own[2 * kTrioStride] = zf;
            const D g = ddot3_raw(Rk[0], at(1, 0), Rk[1], at(1, 1), Rk[2], at(1, 2));
            __syncwarp();
            zn = g + trio_cross(bk1, bk2, at(2, k1), at(2, k2));
            own[3 * kTrioStride] = zn;
            __syncwarp();
            chat = (cur.t - at(3, 2)) * cur.iom;
        } else {
            chat = cur.t * cur.iom;
        }
        if (RAGGED && !in) chat = zero;
        if (L.live && in && k == 0) aba_zput(wsz, B, b, i, 6, chat);
        uv = RAGGED && !in ? zero : cur.uv;
        uw = RAGGED && !in ? zero : cur.uw;
        // row k of R = Rx(alpha) Rz(theta) and b of link i for the next step
        trio_row(k, ca, sa, c, s, Rk);
        bk1 = nb1;
        bk2 = nb2;
    }
    __syncwarp();  // c_hat is read by all three lanes
    // ---- a = Ad_{f^-1} lambda_{i-1}; qdd_i = c_hat_i - U_i^T a / Omega_i;
    //      lambda_i = a + S qdd_i
    int bad = 0;
    D lv = zero, lw = zero;
    __pipeline_wait_prior(0);
#pragma unroll
    for (int u = 0; u < kTrioRing - 1; ++u) fetch(u, u, true);
#pragma unroll 1
    for (int i = 0; i < nmax; ++i) {
        const bool in = !RAGGED || i < n;
        const int ii = !RAGGED || in ? i : n - 1;
        const D *r = sd + ii * kAbaDh64;
        if (RAGGED && ii + 1 < n) prefetch_l1(sd + (ii + 1) * kAbaDh64);
        const SolveIn cur = take(i);
        fetch(i + kTrioRing - 1, i + kTrioRing - 1, true);
        const S c = cur.c, s = cur.s;
        const D ca = r[0], sa = r[1];
        // column k of R: (c, sca, ssa), (-s, cca, csa), (0, -sa, ca)
        const S t = k == 0 ? s : c;
        const D q1 = dmul_raw(t, ca), q2 = dmul_raw(t, sa);
        const D C0 = sel3(k, dcvt<D>(c), dcvt<D>(-s), zero);
        const D C1 = k == 2 ? -sa : q1, C2 = k == 2 ? ca : q2;
        own[0] = lw;
        __syncwarp();
        own[kTrioStride] = dsum2_raw(lv, trio_cross(at(0, k1), at(0, k2), r[2 + k1], r[2 + k2]));
        __syncwarp();
        const D av = df_renorm(ddot3_raw(C0, at(1, 0), C1, at(1, 1), C2, at(1, 2)));
        D aw = df_renorm(ddot3_raw(C0, at(0, 0), C1, at(0, 1), C2, at(0, 2)));
        own[2 * kTrioStride] = ddot2_raw(cur.uv, av, cur.uw, aw);
        __syncwarp();
        const D ua = dsum3_raw(at(2, 0), at(2, 1), at(2, 2));
        const D qdd = fma(-cur.iom, ua, cur.t);
        aw = k == 2 ? aw + qdd : aw;
        lv = av;
        lw = aw;
        if (in && disnan(qdd)) bad = 1;
        if (L.live && in && k == 0) qddr[i] = dcvt<T>(qdd);
    }
    return bad;
}

// The bias sweeps of one instance in T, one thread: those of aba_pair.cuh's warp
// Z, up to tau_hat. PF: constants in global memory, prefetched a link ahead.
template <typename T, typename D, int TRIG, bool PF = false>
__device__ __forceinline__ void aba_trio_bias(const T *__restrict__ sc, int n,
                                              const T *__restrict__ qr,
                                              const T *__restrict__ qdr,
                                              const T *__restrict__ taur, T *ws, int B, int b,
                                              const BaseParams<T> &base)
{
    Motion<T> x;
    x.v = mk3(base.V0[0], base.V0[1], base.V0[2]);
    x.w = mk3(base.V0[3], base.V0[4], base.V0[5]);
    x.a = mk3(base.dV0[0], base.dV0[1], base.dV0[2]);
    x.al = mk3(base.dV0[3], base.dV0[4], base.dV0[5]);
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        if (PF && i + 1 < n) prefetch_l1(sc + (i + 1) * kDhConsts);
        T s, c;
        DhLink<T> L;
        load_dh(sc + i * kDhConsts, L);
        dh_trig<T, TRIG>(__ldg(qr + i) + L.th0, &s, &c);
        x = dh_forward(dh_rot(L.ca, L.sa, c, s), L.b, __ldg(qdr + i), T(0), x);
        const Wrench<T> Fh = bias_wrench(L.m, L.c, L.I, x);
        const T vals[8] = {Fh.f.x, Fh.f.y, Fh.f.z, Fh.n.x, Fh.n.y, Fh.n.z, c, s};
#pragma unroll
        for (int k = 0; k < 8; ++k) bias_put<T>(ws, B, b, i, k, vals[k]);
    }
    Wrench<T> F;
    F.f = mk3(base.Fn[0], base.Fn[1], base.Fn[2]);
    F.n = mk3(base.Fn[3], base.Fn[4], base.Fn[5]);
    DhRot<T> Rn = dh_rot(T(1), T(0), T(1), T(0));
    V3<T> bn = mk3(T(0), T(0), T(0));
#pragma unroll 1
    for (int i = n - 1; i >= 0; --i) {
        Wrench<T> Fh;
        Fh.f = mk3(bias_get<T>(ws, B, b, i, 0), bias_get<T>(ws, B, b, i, 1),
                   bias_get<T>(ws, B, b, i, 2));
        Fh.n = mk3(bias_get<T>(ws, B, b, i, 3), bias_get<T>(ws, B, b, i, 4),
                   bias_get<T>(ws, B, b, i, 5));
        const T c = bias_get<T>(ws, B, b, i, 6), s = bias_get<T>(ws, B, b, i, 7);
        if (i == n - 1) {
            F.f = add3(F.f, Fh.f);
            F.n = add3(F.n, Fh.n);
        } else {
            F = dh_carry(Rn, bn, F, Fh);
        }
        trio_tau_put<D>(ws, B, b, i, F.n.z, __ldg(taur + i));
        const T *Lt = sc + i * kDhConsts;
        Rn = dh_rot(Lt[0], Lt[1], c, s);
        bn = mk3(Lt[2], Lt[3], Lt[4]);
    }
}

// The bias sweeps of one warp's ten instances in double-float (FP32 data), three
// lanes each: lane k carries component k of the motion and of the wrench
// (spatial_dh.cuh's dh_forward, bias_wrench and dh_carry by components).
template <bool RAGGED>
__device__ __forceinline__ void aba_trio_bias_df(const DF *__restrict__ sdf, int n, int nmax,
                                                 const float *__restrict__ qr,
                                                 const float *__restrict__ qdr,
                                                 const float *__restrict__ taur, float *ws, int B,
                                                 int b, const BaseParams<float> &base,
                                                 const TrioLane &L, TrioShared<DF> &sh)
{
    const int k = L.k, k1 = L.k1, k2 = L.k2;
    DF *const own = &sh.x[threadIdx.x & 31];
    const DF *const grp = &sh.x[L.base];
    const DF zero = DF(0.0f);
    auto at = [&](int slot, int l) -> DF { return grp[slot * kTrioStride + l]; };
    auto put = [&](int slot, DF v) { own[slot * kTrioStride] = v; };
    const int ci[3] = {10 + sel3(k, 0, 3, 4), 10 + sel3(k, 3, 1, 5), 10 + sel3(k, 4, 5, 2)};
    auto comp = [&](const float *u) { return DF(sel3(k, u[0], u[1], u[2])); };
    DF v = comp(base.V0), w = comp(base.V0 + 3), a = comp(base.dV0), al = comp(base.dV0 + 3);
    DF ts = zero, tc = zero;
#pragma unroll 1
    for (int i = 0; i < nmax; ++i) {
        const bool in = !RAGGED || i < n;
        const int ii = !RAGGED || in ? i : n - 1;
        const DF *r = sdf + ii * kAbaDh64;
        if (RAGGED && ii + 1 < n) {
            prefetch_l1(r + kAbaDh64);
            prefetch_l1(r + kAbaDh64 + kAbaDh64 / 2);
        }
        // sin/cos: each lane of the group evaluates one of the next three links
        const int ph = i % 3;
        if (ph == 0) {
            const int it = i + k < n ? i + k : n - 1;
            df_sincos((double)__ldg(qr + it) + df_to_double(sdf[it * kAbaDh64 + 5]), &ts, &tc);
        }
        const DF s = df_shfl(ts, L.base + ph), c = df_shfl(tc, L.base + ph);
        const DF ca = r[0], sa = r[1];
        const DF b1 = r[2 + k1], b2 = r[2 + k2];
        const DF t = k == 0 ? s : c;
        const DF C0 = sel3(k, c, -s, zero), C1 = k == 2 ? -sa : dmul_raw(t, ca),
                 C2 = k == 2 ? ca : dmul_raw(t, sa);
        put(0, w);
        put(1, al);
        __syncwarp();
        put(2, dsum2_raw(v, trio_cross(at(0, k1), at(0, k2), b1, b2)));
        put(3, dsum2_raw(a, trio_cross(at(1, k1), at(1, k2), b1, b2)));
        __syncwarp();
        const float qd = __ldg(qdr + ii);
        v = df_renorm(ddot3_raw(C0, at(2, 0), C1, at(2, 1), C2, at(2, 2)));
        a = ddot3_raw(C0, at(3, 0), C1, at(3, 1), C2, at(3, 2));
        w = ddot3_raw(C0, at(0, 0), C1, at(0, 1), C2, at(0, 2)) + DF(k == 2 ? qd : 0.0f);
        al = ddot3_raw(C0, at(1, 0), C1, at(1, 1), C2, at(1, 2));
        put(4, v);
        put(5, w);
        __syncwarp();
        // a -= qd (e_z x v), al -= qd (e_z x w): components x and y
        const float qk = k == 0 ? qd : (k == 1 ? -qd : 0.0f);
        const int ko = k == 0 ? 1 : 0;
        a = a + dmul_raw(qk, at(4, ko));
        al = al + dmul_raw(qk, at(5, ko));
        const DF c1 = r[7 + k1], c2 = r[7 + k2];
        const DF w1 = at(5, k1), w2 = at(5, k2);
        const DF I0 = r[ci[0]], I1 = r[ci[1]], I2 = r[ci[2]];
        put(6, al);
        put(7, dsum2_raw(v, trio_cross(w1, w2, c1, c2)));                      // velocity of the centre of mass
        put(8, ddot3_raw(I0, at(5, 0), I1, at(5, 1), I2, at(5, 2)));  // I w
        __syncwarp();
        const DF ac = dsum3_raw(a, trio_cross(at(6, k1), at(6, k2), c1, c2),
                            trio_cross(w1, w2, at(7, k1), at(7, k2)));
        const DF f = r[6] * ac;
        put(9, f);
        const DF n0 = dsum2_raw(ddot3_raw(I0, at(6, 0), I1, at(6, 1), I2, at(6, 2)),
                                trio_cross(w1, w2, at(8, k1), at(8, k2)));
        __syncwarp();
        const DF nn = n0 + trio_cross(c1, c2, at(9, k1), at(9, k2));
        if (L.live && in) {
            bias_put<DF>(ws, B, b, i, k, f);
            bias_put<DF>(ws, B, b, i, 3 + k, nn);
            if (k == 0) bias_put<DF>(ws, B, b, i, 6, c);
            if (k == 1) bias_put<DF>(ws, B, b, i, 7, s);
        }
    }
    __syncwarp();
    // wrench carry and tau_hat, tip to base
    const DF F0 = comp(base.Fn), N0 = comp(base.Fn + 3);
    DF Ff = F0, Fn = N0;
    DF Rk[3] = {zero, zero, zero}, b1 = zero, b2 = zero;
#pragma unroll 1
    for (int i = nmax - 1; i >= 0; --i) {
        const bool in = !RAGGED || i < n;
        const int ii = !RAGGED || in ? i : n - 1;
        const DF *r = sdf + ii * kAbaDh64;
        const DF fh = bias_get<DF>(ws, B, b, ii, k), nh = bias_get<DF>(ws, B, b, ii, 3 + k);
        const DF c = bias_get<DF>(ws, B, b, ii, 6), s = bias_get<DF>(ws, B, b, ii, 7);
        if (RAGGED && ii > 0) prefetch_l1(sdf + (ii - 1) * kAbaDh64);
        const DF ca = r[0], sa = r[1];
        const DF nb1 = r[2 + k1], nb2 = r[2 + k2];
        const float tau = __ldg(taur + ii);
        put(10, Ff);
        put(11, Fn);
        __syncwarp();
        const DF rf = ddot3_raw(Rk[0], at(10, 0), Rk[1], at(10, 1), Rk[2], at(10, 2));
        put(12, rf);
        const DF rn = ddot3_raw(Rk[0], at(11, 0), Rk[1], at(11, 1), Rk[2], at(11, 2));
        __syncwarp();
        const DF nx = dsum2_raw(rn, trio_cross(b1, b2, at(12, k1), at(12, k2)));
        const bool tip = i == nmax - 1 || (RAGGED && i >= n - 1);
        // the tip adds F_{n+1} as it is
        Ff = (tip ? F0 : rf) + fh;
        Fn = (tip ? N0 : nx) + nh;
        if (L.live && in && k == 2) trio_tau_put<DF>(ws, B, b, i, Fn, tau);
        trio_row(k, ca, sa, c, s, Rk);
        b1 = nb1;
        b2 = nb2;
    }
}

// The chain's records (D) and constants (T) into shared memory, for the block.
template <typename V>
__device__ __forceinline__ void trio_stage(V *dst, const V *__restrict__ src, int count)
{
    static_assert(sizeof(V) == 4 || sizeof(V) == 8, "");
    const int n16 = count * (int)sizeof(V) / 16;
    for (int t = threadIdx.x; t < n16; t += blockDim.x)
        reinterpret_cast<float4 *>(dst)[t] = __ldg(reinterpret_cast<const float4 *>(src) + t);
}

// A block's share of the workspace: its instances' scalars together, [link]
// [component][instance of the block], so that a link's values lie within a few
// lines. (With the whole batch as the instance stride, batches of a power of two
// put every component of every link on the same few cache sets: n = 64, B =
// 16384: 239 us against 227 at B = 16390.) per: bias scalars of T per link.
template <typename T, typename D>
__device__ __forceinline__ void trio_block_ws(T *&ws, D *&wsz, int n, int b0, int per)
{
    ws += (size_t)b0 * (size_t)n * (size_t)per;
    wsz += (size_t)b0 * (size_t)n * (size_t)kAbaSolveScalars;
}

// Bias in T: warps 0..2 ten instances each, warp 3 the bias of the thirty.
// Dynamic shared memory: n records, n constants.
template <typename T, typename D, int TRIG>
__global__ void __launch_bounds__(128, 4)
aba_trio_kernel(const T *__restrict__ sc, const D *__restrict__ sd, int n, int B,
                const T *__restrict__ q, const T *__restrict__ qd, const T *__restrict__ tau,
                T *__restrict__ qdd_out, int *__restrict__ status, T *ws, D *wsz,
                BaseParams<T> base)
{
    __shared__ TrioShared<D> sh[3];
    __shared__ TrioRing<D, T> rg[3];
    extern __shared__ __align__(16) unsigned char smem[];
    D *rec = reinterpret_cast<D *>(smem);
    T *con = reinterpret_cast<T *>(rec + n * kAbaDh64);
    trio_stage(rec, sd, n * kAbaDh64);
    trio_stage(con, sc, n * kDhConsts);
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b0 = blockIdx.x * kTrioInstances;
    const int nb = B - b0 < kTrioInstances ? B - b0 : kTrioInstances;
    trio_block_ws(ws, wsz, n, b0, kAbaStateScalars);
    if (warp == 3) {
        if (lane < nb) {
            const size_t row = (size_t)(b0 + lane) * (size_t)n;
            aba_trio_bias<T, D, TRIG>(con, n, q + row, qd + row, tau + row, ws, nb, lane, base);
        }
        __syncthreads();
        return;
    }
    // A warp without an instance (in the batch's last block) leaves: repeating the last
    // instance's work beside the warp that has it held the block up (n = 64, B =
    // 16384: 232 us against 216).
    if (warp * kTrioPerWarp >= nb) {
        __syncthreads();
        return;
    }
    TrioLane L = trio_lane(lane);
    int b = warp * kTrioPerWarp + L.base / 3;
    if (b >= nb) {  // beyond the batch: the last instance's work, no output
        b = nb - 1;
        L.live = false;
    }
    const size_t row = (size_t)(b0 + b) * (size_t)n;
    int bad = aba_trio_j<T, D, T, TRIG, false>(con, rec, nullptr, n, n, q + row, wsz, nb, b, L,
                                               sh[warp]);
    __syncthreads();
    bad |= aba_trio_solve<T, D, T, false>(rec, n, n, qdd_out + row, ws, wsz, nb, b, L, sh[warp],
                                          rg[warp]);
    if (status && L.live && L.k == 0) status[b0 + b] = bad ? RD_WARN_SINGULAR : 0;
}

// Bias in double-float: warps 0 and 1 the inertias and solves of ten instances
// each, warps 2 and 3 their bias. Dynamic shared memory: n records.
constexpr int kTrioExtInstances = 2 * kTrioPerWarp;

template <int TRIG>
__global__ void __launch_bounds__(128, 4)
aba_trio_ext_kernel(const float *__restrict__ sc, const DF *__restrict__ sdf, int n, int B,
                    const float *__restrict__ q, const float *__restrict__ qd,
                    const float *__restrict__ tau, float *__restrict__ qdd_out,
                    int *__restrict__ status, float *ws, DF *wsz, BaseParams<float> base)
{
    __shared__ TrioShared<DF> sh[4];
    __shared__ TrioRing<DF, DF> rg[2];
    extern __shared__ __align__(16) unsigned char smem[];
    DF *rec = reinterpret_cast<DF *>(smem);
    trio_stage(rec, sdf, n * kAbaDh64);
    __syncthreads();
    const int warp = threadIdx.x >> 5, pair = warp & 1;
    const int b0 = blockIdx.x * kTrioExtInstances;
    const int nb = B - b0 < kTrioExtInstances ? B - b0 : kTrioExtInstances;
    trio_block_ws(ws, wsz, n, b0, aba_bias_ws_scalars<float, DF>());
    if (pair * kTrioPerWarp >= nb) {
        __syncthreads();
        return;
    }
    TrioLane L = trio_lane(threadIdx.x & 31);
    int b = pair * kTrioPerWarp + L.base / 3;
    if (b >= nb) {
        b = nb - 1;
        L.live = false;
    }
    const size_t row = (size_t)(b0 + b) * (size_t)n;
    if (warp >= 2) {
        aba_trio_bias_df<false>(rec, n, n, q + row, qd + row, tau + row, ws, nb, b, base, L,
                                sh[warp]);
        __syncthreads();
        return;
    }
    int bad = aba_trio_j<float, DF, DF, TRIG, false>(sc, rec, rec, n, n, q + row, wsz, nb, b, L,
                                                     sh[warp]);
    __syncthreads();
    bad |= aba_trio_solve<float, DF, DF, false>(rec, n, n, qdd_out + row, ws, wsz, nb, b, L,
                                                sh[warp], rg[warp]);
    if (status && L.live && L.k == 0) status[b0 + b] = bad ? RD_WARN_SINGULAR : 0;
}

}  // namespace rdyn
