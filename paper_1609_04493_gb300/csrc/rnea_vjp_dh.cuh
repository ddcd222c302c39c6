// rnea_vjp_dh.cuh -- the adjoint of the two scans (rnea_vjp.cuh) in the
// common-normal frames of spatial_dh.cuh, with the link constants passed as a
// __grid_constant__ kernel parameter and FP32 sin/cos from trig_poly.cuh.
//
// The recursions are those of rnea_vjp.cuh; only the frames change. In a frame
// D_i the joint twist is still e_z (angular) and q_i enters the link transform
// as its last factor Rz(q_i), so d Ad_{f_i^-1} / dq_i = -ad_S Ad_{f_i^-1} and the
// gradient formulas carry over unchanged:
//   gqdd_i = S^T dVbar_i,
//   gqd_i  = S^T Vbar_i - <dVbar_i, ad_S V_i>,
//   gq_i   = -<Vbar_i, ad_S V_i> - <dVbar_i, ad_S dV_i> - <F_i, ad_S Fb_i>.
// Joint values and weights are read into registers one chunk ahead. For
// n % 4 == 0, n <= NMAX and 16-byte aligned rows.
#pragma once
#include "rnea_dhp.cuh"
#include "rnea_vjp.cuh"

namespace rdyn {

// Fb_i = Ad_{f^-1} Fb_{i-1} + S w  (the velocity step without the ad term)
template <typename T>
__device__ __forceinline__ void fb_forward_dh(const DhRot<T> &R, V3<T> b, T w, V3<T> &fv,
                                              V3<T> &fw)
{
    fv = dh_mulT(R, cross_add(fw, b, fv));
    fw = dh_mulT(R, fw);
    fw.z += w;
}

// inverse: Fb_{i-1} = Ad_f (Fb_i - S w)
template <typename T>
__device__ __forceinline__ void fb_backward_dh(const DhRot<T> &R, V3<T> b, T w, V3<T> &fv,
                                               V3<T> &fw)
{
    V3<T> ww = fw;
    ww.z -= w;
    const V3<T> pw = dh_mul(R, ww);
    fv = cross_add(b, pw, dh_mul(R, fv));
    fw = pw;
}

// The aligned pieces of chunk c of a row (ragged_row), read no further than the row's
// end.
template <typename T>
__device__ __forceinline__ Chunk<T> ld_pieces(const RaggedRow<T> &row, int n, int c)
{
    Chunk<T> v;
    const int left = row.off + n - 4 * c;
    const T *p = row.p + 4 * c;
    if (left >= 4) {
        ld_row_chunk(p, 0, v);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v.v[j] = j < left ? __ldg(p + j) : T(0);
    }
    return v;
}

// VEC: n % 4 == 0 and 16-byte aligned rows; without it rows of any length and
// alignment, each array streamed in aligned 16-byte pieces and shifted in registers
// (rnea_dhp.cuh), the gradients stored by the warp together through shared memory,
// eight rows' 16 bytes an instruction, and the last, shorter chunk as code of its own.
template <typename T, int NMAX, int BLOCK, int MODE, int TRIG, bool VEC = true>
__global__ void __launch_bounds__(BLOCK)
rnea_vjp_dh_kernel(const __grid_constant__ DhParamConsts<T, NMAX> pc, int n, int B,
                   const T *__restrict__ q, const T *__restrict__ qd, const T *__restrict__ qdd,
                   const T *__restrict__ wv, T *__restrict__ gq, T *__restrict__ gqd,
                   T *__restrict__ gqdd, T *__restrict__ ws, BaseParams<T> base)
{
    const T *sc = pc.c;
    // kVjpStoreShared: the per-link state in shared memory, [link][k][thread]
    extern __shared__ __align__(16) unsigned char vjp_smem[];
    T *sst = reinterpret_cast<T *>(vjp_smem);
    constexpr bool kStored = MODE == kVjpStore || MODE == kVjpStoreShared;
    // the instance; ragged rows: lanes beyond the batch repeat the last one's work (and
    // write its state again, the same values)
    const int b = blockIdx.x * BLOCK + threadIdx.x;
    const int bw = VEC || b < B ? b : B - 1;
    auto st_put = [&](int i, int k, T v) {
        if constexpr (MODE == kVjpStoreShared)
            sst[((size_t)i * kVjpStateScalars + k) * BLOCK + threadIdx.x] = v;
        else
            ws_put(ws, B, bw, i, k, v);
    };
    auto st_get = [&](int i, int k) -> T {
        if constexpr (MODE == kVjpStoreShared)
            return sst[((size_t)i * kVjpStateScalars + k) * BLOCK + threadIdx.x];
        else
            return ws_get(ws, B, bw, i, k);
    };
    if (VEC && b >= B) return;  // ragged rows: every lane stores for others
    const size_t row = (size_t)bw * (size_t)n;
    const T *qr = q + row, *qdr = qd + row, *qddr = qdd + row, *wr = wv + row;
    const RaggedRow<T> rr[4] = {ragged_row(qr), ragged_row(qdr), ragged_row(qddr), ragged_row(wr)};
    Chunk<T> plo[4], phi[4], pnx[4];  // ragged rows: pieces of neighbouring chunks
    __shared__ __align__(16) T stage[VEC ? 1 : BLOCK / 32][3][VEC ? 1 : 128];

    Motion<T> x;
    x.v = mk3(base.V0[0], base.V0[1], base.V0[2]);
    x.w = mk3(base.V0[3], base.V0[4], base.V0[5]);
    x.a = mk3(base.dV0[0], base.dV0[1], base.dV0[2]);
    x.al = mk3(base.dV0[3], base.dV0[4], base.dV0[5]);
    V3<T> fbv = mk3(T(0), T(0), T(0)), fbw = mk3(T(0), T(0), T(0));

    // ---- sweep 1: base -> tip
    const int nchunks = VEC ? n / 4 : (n + 3) / 4, nfull = n / 4;
    Chunk<T> cq, cqd, cqdd, cw, nq = {}, nqd = {}, nqdd = {}, nw = {};
    if constexpr (VEC) {
        ld_row_chunk(qr, 0, cq);
        ld_row_chunk(qdr, 0, cqd);
        ld_row_chunk(qddr, 0, cqdd);
        ld_row_chunk(wr, 0, cw);
    } else {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            plo[a] = ld_pieces(rr[a], n, 0);
            phi[a] = ld_pieces(rr[a], n, 1);
        }
    }
    // ragged: the chunk's values from its pieces and the next chunk's
    auto window = [&]() {
        cq = shift_pieces(plo[0], phi[0], rr[0].off);
        cqd = shift_pieces(plo[1], phi[1], rr[1].off);
        cqdd = shift_pieces(plo[2], phi[2], rr[2].off);
        cw = shift_pieces(plo[3], phi[3], rr[3].off);
    };
    auto forward_chunk = [&](int kc, auto full) {
        constexpr bool FULL = decltype(full)::value;
        const int i0 = 4 * kc;
        if constexpr (!VEC) {
#pragma unroll
            for (int a = 0; a < 4; ++a) pnx[a] = ld_pieces(rr[a], n, kc + 2);
            window();
        } else if (kc + 1 < nchunks) {
            ld_row_chunk(qr, i0 + 4, nq);
            ld_row_chunk(qdr, i0 + 4, nqd);
            ld_row_chunk(qddr, i0 + 4, nqdd);
            ld_row_chunk(wr, i0 + 4, nw);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = i0 + j;
            if (!FULL && i >= n) break;
            DhXf<T> X;
            load_dh_xf(sc + i * kDhConsts, X);
            T s, c;
            dh_trig<T, TRIG>(cq.v[j] + X.th0, &s, &c);
            const DhRot<T> R = dh_rot(X.ca, X.sa, c, s);
            x = dh_forward(R, X.b, cqd.v[j], cqdd.v[j], x);
            fb_forward_dh(R, X.b, cw.v[j], fbv, fbw);
            if constexpr (kStored) {
                const T vals[kVjpStateScalars] = {x.v.x,  x.v.y,  x.v.z,  x.w.x,  x.w.y,
                                                  x.w.z,  x.a.x,  x.a.y,  x.a.z,  x.al.x,
                                                  x.al.y, x.al.z, fbv.x,  fbv.y,  fbv.z,
                                                  fbw.x,  fbw.y,  fbw.z,  c,      s};
#pragma unroll
                for (int k = 0; k < kVjpStateScalars; ++k) st_put(i, k, vals[k]);
            }
        }
        if constexpr (VEC) {
            cq = nq;
            cqd = nqd;
            cqdd = nqdd;
            cw = nw;
        } else {
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                plo[a] = phi[a];
                phi[a] = pnx[a];
            }
        }
    };
    for (int kc = 0; kc < nfull; ++kc) forward_chunk(kc, std::true_type());
    if (!VEC && nfull < nchunks) forward_chunk(nfull, std::false_type());

    // ---- sweep 2: tip -> base
    Wrench<T> F;
    F.f = mk3(base.Fn[0], base.Fn[1], base.Fn[2]);
    F.n = mk3(base.Fn[3], base.Fn[4], base.Fn[5]);
    Wrench<T> Vb, dVb;  // adjoints of V_{i+1}, dV_{i+1} (covectors)
    DhRot<T> Rn = dh_rot(T(1), T(0), T(1), T(0));
    V3<T> bn = mk3(T(0), T(0), T(0));
    T qdn = T(0);
    const int last0 = n - 4;
    if constexpr (!VEC) {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            plo[a] = ld_pieces(rr[a], n, nchunks - 1);
            phi[a] = ld_pieces(rr[a], n, nchunks);
        }
    } else {
        ld_row_chunk(qdr, last0, cqd);
        if constexpr (MODE == kVjpRecompute) {
            ld_row_chunk(qr, last0, cq);
            ld_row_chunk(qddr, last0, cqdd);
            ld_row_chunk(wr, last0, cw);
        }
    }
    auto backward_chunk = [&](int i0, auto full) {
        constexpr bool FULL = decltype(full)::value;
        if constexpr (!VEC) {
            if (i0 > 0) {
#pragma unroll
                for (int a = 0; a < 4; ++a) pnx[a] = ld_pieces(rr[a], n, i0 / 4 - 1);
            }
            window();
        } else if (i0 > 0) {
            ld_row_chunk(qdr, i0 - 4, nqd);
            if constexpr (MODE == kVjpRecompute) {
                ld_row_chunk(qr, i0 - 4, nq);
                ld_row_chunk(qddr, i0 - 4, nqdd);
                ld_row_chunk(wr, i0 - 4, nw);
            }
        }
        Chunk<T> oq = {}, oqd = {}, oqdd = {};
#pragma unroll
        for (int j = 3; j >= 0; --j) {
            const int i = i0 + j;
            if (!FULL && i >= n) continue;
            DhLink<T> L;
            load_dh(sc + i * kDhConsts, L);
            T s, c;
            if constexpr (kStored) {
                x.v = mk3(st_get(i, 0), st_get(i, 1), st_get(i, 2));
                x.w = mk3(st_get(i, 3), st_get(i, 4), st_get(i, 5));
                x.a = mk3(st_get(i, 6), st_get(i, 7), st_get(i, 8));
                x.al = mk3(st_get(i, 9), st_get(i, 10), st_get(i, 11));
                fbv = mk3(st_get(i, 12), st_get(i, 13), st_get(i, 14));
                fbw = mk3(st_get(i, 15), st_get(i, 16), st_get(i, 17));
                c = st_get(i, 18);
                s = st_get(i, 19);
            } else {
                dh_trig<T, TRIG>(cq.v[j] + L.th0, &s, &c);
            }
            const DhRot<T> R = dh_rot(L.ca, L.sa, c, s);
            const Wrench<T> Fh = bias_wrench(L.m, L.c, L.I, x);
            if (i == n - 1) {
                F.f = add3(F.f, Fh.f);
                F.n = add3(F.n, Fh.n);
            } else {
                F = dh_carry(Rn, bn, F, Fh);
            }
            // local seeds from F_hat = J dV - ad^T_V (J V)
            Wrench<T> dVl, Vl;
            J_apply(L.m, L.c, L.I, fbv, fbw, dVl.f, dVl.n);           // J Fb
            V3<T> jvf, jvn;
            J_apply(L.m, L.c, L.I, x.v, x.w, jvf, jvn);               // J V
            const V3<T> adv = cross_add(x.v, fbw, cross3(x.w, fbv));   // ad_V Fb
            const V3<T> adw = cross3(x.w, fbw);
            V3<T> jaf, jan;
            J_apply(L.m, L.c, L.I, adv, adw, jaf, jan);               // J ad_V Fb
            Vl.f = sub3(scale3(T(-1), cross3(fbw, jvf)), jaf);
            Vl.n = sub3(scale3(T(-1), cross_add(fbv, jvf, cross3(fbw, jvn))), jan);
            if (i == n - 1) {
                Vb = Vl;
                dVb = dVl;
            } else {
                Wrench<T> Yb = Vb;  // Vbar_{i+1} - ad^T_{S qd_{i+1}} dVbar_{i+1}
                Yb.f.x = fma(-qdn, dVb.f.y, Yb.f.x);
                Yb.f.y = fma(qdn, dVb.f.x, Yb.f.y);
                Yb.n.x = fma(-qdn, dVb.n.y, Yb.n.x);
                Yb.n.y = fma(qdn, dVb.n.x, Yb.n.y);
                Vb = dh_carry(Rn, bn, Yb, Vl);
                dVb = dh_carry(Rn, bn, dVb, dVl);
            }
            oqdd.v[j] = dVb.n.z;
            oqd.v[j] = Vb.n.z - (dot_ez_cross(dVb.f, x.v) + dot_ez_cross(dVb.n, x.w));
            oq.v[j] = -(dot_ez_cross(Vb.f, x.v) + dot_ez_cross(Vb.n, x.w)) -
                      (dot_ez_cross(dVb.f, x.a) + dot_ez_cross(dVb.n, x.al)) -
                      (dot_ez_cross(F.f, fbv) + dot_ez_cross(F.n, fbw));
            if constexpr (MODE == kVjpRecompute) {
                if (i > 0) {
                    x = dh_recover(R, L.b, cqd.v[j], cqdd.v[j], x);
                    fb_backward_dh(R, L.b, cw.v[j], fbv, fbw);
                }
            }
            Rn = R;
            bn = L.b;
            qdn = cqd.v[j];
        }
        if constexpr (VEC) {
            st_chunk<T, true>(gq + row, i0, n, oq);
            st_chunk<T, true>(gqd + row, i0, n, oqd);
            st_chunk<T, true>(gqdd + row, i0, n, oqdd);
            cqd = nqd;
            if constexpr (MODE == kVjpRecompute) {
                cq = nq;
                cqdd = nqdd;
                cw = nw;
            }
        } else {
            const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
            __syncwarp();  // the chunk before has left
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                stage[wp][0][4 * lane + j] = oq.v[j];
                stage[wp][1][4 * lane + j] = oqd.v[j];
                stage[wp][2][4 * lane + j] = oqdd.v[j];
            }
            __syncwarp();
            const int e = lane & 3;
            const int b0 = blockIdx.x * BLOCK + 32 * wp + (lane >> 2);
            if (i0 + e < n) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (b0 + 8 * j < B) {
                        const size_t o = (size_t)(b0 + 8 * j) * (size_t)n + i0 + e;
                        gq[o] = stage[wp][0][lane + 32 * j];
                        gqd[o] = stage[wp][1][lane + 32 * j];
                        gqdd[o] = stage[wp][2][lane + 32 * j];
                    }
                }
            }
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                phi[a] = plo[a];
                plo[a] = pnx[a];
            }
        }
    };
    int top = 4 * (nchunks - 1);
    if (!VEC && nfull < nchunks) {
        backward_chunk(top, std::false_type());
        top -= 4;
    }
    for (int i0 = top; i0 >= 0; i0 -= 4) backward_chunk(i0, std::true_type());
}

}  // namespace rdyn
