// rnea_dhp.cuh -- the common-normal-frame RNEA of rnea_dh.cuh with the link
// constants passed as a __grid_constant__ kernel parameter, and a per-link
// backward-sweep state that is full for the first K links only.
//
// * Constants. Their index is the same for every thread of a warp, so they are
//   read through the uniform data path and take no slot in the per-thread
//   memory pipeline, which then carries only the joint values (a cp.async ring,
//   two chunks ahead) and the state.
// * State. Links 0..K-1 keep F_hat_i, cos and sin (8 scalars); links K..n-1
//   keep cos and sin only (2 scalars), and the backward sweep re-derives their
//   motion by inverting the forward step (the forward operands form a group,
//   Sec. III-B) and recomputes F_hat_i. K trades shared memory, and with it the
//   number of resident warps, against arithmetic; K = n is the plain stored
//   sweep, K = 0 the stateless one.
// * Trigonometry (FP32). The default evaluates sin/cos of q_i + theta0_i with
//   the FMA-pipe polynomials of trig_poly.cuh (error under one ulp); TRIG = 1
//   selects the special-function-unit approximation (RD_FLAG_FAST_TRIG). FP64
//   takes trig_fixed.cuh.
// For chains of at most NMAX links. Rows of whole 16-byte chunks (n % 4 == 0, 16-byte
// aligned) are staged by each thread for itself; others by the warp together
// (stage_chunk_ragged).
#pragma once
#include <type_traits>

#include "rnea_dh.cuh"
#include "trig_poly.cuh"

namespace rdyn {

// The 16 common-normal constants per link; for rnea_dhp_kernel with the second
// moments of kin_wrench in place of the rotational inertia.
template <typename T, int NMAX>
struct DhParamConsts {
    T c[NMAX * kDhConsts];
};

// S = tr(I)/2 E - I of one link's (xx, yy, zz, xy, xz, yz)
inline void dh_second_moments(const double I[6], double S[6])
{
    const double h = 0.5 * (I[0] + I[1] + I[2]);
    for (int k = 0; k < 3; ++k) {
        S[k] = h - I[k];
        S[3 + k] = -I[3 + k];
    }
}

enum DhTrig { kTrigPoly = 0, kTrigSfu = 1 };

template <typename T, int TRIG>
__device__ __forceinline__ void dh_trig(T x, T *s, T *c)
{
    if constexpr (sizeof(T) == 8) sincos_fixed(x, s, c);
    else if constexpr (TRIG == kTrigSfu) sincos_fast(x, s, c);
    else sincos_poly(x, s, c);
}

// Four joint values of a row (16-byte aligned) into registers.
template <typename T>
__device__ __forceinline__ void ld_row_chunk(const T *__restrict__ p, int i0, Chunk<T> &c)
{
    if constexpr (sizeof(T) == 4) {
        float4 t = __ldg(reinterpret_cast<const float4 *>(p + i0));
        c.v[0] = t.x; c.v[1] = t.y; c.v[2] = t.z; c.v[3] = t.w;
    } else {
        double2 a = __ldg(reinterpret_cast<const double2 *>(p + i0));
        double2 b = __ldg(reinterpret_cast<const double2 *>(p + i0 + 2));
        c.v[0] = a.x; c.v[1] = a.y; c.v[2] = b.x; c.v[3] = b.y;
    }
}

// The backward sweep needs qd and qdd only; they sit at positions 1 and 2 of
// the forward ring's slots.
template <typename T, int BLOCK>
__device__ __forceinline__ void stage_chunk2(unsigned char *ring, int slot, int tid,
                                             const T *qdr, const T *qddr, int i0)
{
    constexpr int P = vec16_per_chunk<T>();
    float4 *r = reinterpret_cast<float4 *>(ring);
    const T *src[2] = {qdr, qddr};
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int h = 0; h < P; ++h)
            cp_async16_cg(&r[((slot * 3 + a + 1) * P + h) * BLOCK + tid],
                          src[a] + i0 + h * (16 / (int)sizeof(T)));
}

template <typename T, int BLOCK>
__device__ __forceinline__ void read_chunk2(const unsigned char *ring, int slot, int tid,
                                            Chunk<T> &cqd, Chunk<T> &cqdd)
{
    constexpr int P = vec16_per_chunk<T>();
    const float4 *r = reinterpret_cast<const float4 *>(ring);
    Chunk<T> *dst[2] = {&cqd, &cqdd};
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int h = 0; h < P; ++h) {
            float4 v = r[((slot * 3 + a + 1) * P + h) * BLOCK + tid];
            if constexpr (sizeof(T) == 4) {
                dst[a]->v[0] = v.x; dst[a]->v[1] = v.y; dst[a]->v[2] = v.z; dst[a]->v[3] = v.w;
            } else {
                double2 d = *reinterpret_cast<double2 *>(&v);
                dst[a]->v[2 * h] = d.x;
                dst[a]->v[2 * h + 1] = d.y;
            }
        }
}

// ---- rows of any length and alignment: each thread streams the aligned 16-byte
// pieces that cover its row through the same ring, and shifts its four values of a
// chunk out of two neighbouring pieces' worth of registers (10 selects a chunk and
// array in FP32). A piece is read only up to the row's end; the first may begin with
// the values before the row, in the same aligned 16 bytes. Copying element by element
// instead was bound by the shared-memory copies themselves (n = 99, B = 65536: 135 us,
// 20 four-byte copies a chunk against 5). Torques go back through the ring,
// element by element but eight rows' 16 bytes an instruction instead of 32 rows' 4.

// Element e of row r (within the block) in the ring.
template <typename T, int BLOCK>
__device__ __forceinline__ T *ring_at(unsigned char *ring, int slot, int a, int r, int e)
{
    constexpr int V = 16 / (int)sizeof(T);  // elements per 16-byte piece
    return reinterpret_cast<T *>(ring) +
           (((slot * 3 + a) * (4 / V) + e / V) * BLOCK + r) * V + e % V;
}

// A thread's row of one array: its first piece, and where the row begins in it.
template <typename T>
struct RaggedRow {
    const T *p;
    int off;
};

template <typename T>
__device__ __forceinline__ RaggedRow<T> ragged_row(const T *row)
{
    const unsigned long long a = reinterpret_cast<unsigned long long>(row);
    return RaggedRow<T>{reinterpret_cast<const T *>(a & ~15ull), (int)(a & 15) / (int)sizeof(T)};
}

// Chunk c's pieces (elements 4 c .. 4 c + 3 from the first piece's start).
template <typename T, int BLOCK>
__device__ __forceinline__ void stage_pieces(unsigned char *ring, int slot, int a,
                                             const RaggedRow<T> &row, int n, int c)
{
    constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
    for (int h = 0; h < 4; h += V) {
        const int left = (row.off + n - (4 * c + h)) * (int)sizeof(T);  // bytes to the row's end
        if (left > 0) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(ring_at<T, BLOCK>(ring, slot, a, threadIdx.x, h));
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst),
                         "l"(row.p + 4 * c + h), "r"(left < 16 ? left : 16)
                         : "memory");
        }
    }
}

template <typename T, int BLOCK>
__device__ __forceinline__ Chunk<T> read_pieces(unsigned char *ring, int slot, int a)
{
    Chunk<T> c;
    if constexpr (sizeof(T) == 4) {
        const float4 v = *reinterpret_cast<float4 *>(ring_at<T, BLOCK>(ring, slot, a, threadIdx.x, 0));
        c.v[0] = v.x; c.v[1] = v.y; c.v[2] = v.z; c.v[3] = v.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
            const double2 v = *reinterpret_cast<double2 *>(ring_at<T, BLOCK>(ring, slot, a, threadIdx.x, j));
            c.v[j] = v.x;
            c.v[j + 1] = v.y;
        }
    }
    return c;
}

// The four values that begin `off` elements into lo followed by hi.
template <typename T>
__device__ __forceinline__ Chunk<T> shift_pieces(const Chunk<T> &lo, const Chunk<T> &hi, int off)
{
    T x[7] = {lo.v[0], lo.v[1], lo.v[2], lo.v[3], hi.v[0], hi.v[1], hi.v[2]};
    Chunk<T> c;
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int j = 0; j < 6; ++j) x[j] = off & 1 ? x[j + 1] : x[j];
#pragma unroll
        for (int j = 0; j < 4; ++j) c.v[j] = off & 2 ? x[j + 2] : x[j];
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) c.v[j] = off & 1 ? x[j + 1] : x[j];
    }
    return c;
}

// The warp's torques of chunk i0 out through the q part of slot `slot` (0 and 1 in
// turn: one barrier a chunk then suffices).
template <typename T, int BLOCK>
__device__ __forceinline__ void st_chunk_ragged(unsigned char *ring, int slot, T *tau, int n, int B,
                                                int i0, const Chunk<T> &c)
{
    const int lane = threadIdx.x & 31, w0 = threadIdx.x & ~31;
    if constexpr (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(ring_at<T, BLOCK>(ring, slot, 0, threadIdx.x, 0)) =
            make_float4(c.v[0], c.v[1], c.v[2], c.v[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; j += 2)
            *reinterpret_cast<double2 *>(ring_at<T, BLOCK>(ring, slot, 0, threadIdx.x, j)) =
                make_double2(c.v[j], c.v[j + 1]);
    }
    __syncwarp();
    const int e = lane & 3;
    if (i0 + e >= n) return;
    const int r0 = w0 + (lane >> 2);
    T *t = tau + (size_t)(blockIdx.x * BLOCK + r0) * (size_t)n + i0 + e;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if ((int)blockIdx.x * BLOCK + r0 + 8 * j < B) *t = *ring_at<T, BLOCK>(ring, slot, 0, r0 + 8 * j, e);
        t += 8 * n;
    }
}

// RL: how many of the K stored links (the first ones) keep their state in
// registers instead of shared memory
// STG: depth of the joint-value staging ring (3, or 2 to save shared memory)
template <typename T>
__host__ __device__ constexpr size_t dhp_smem_per_thread(int n, int K, int RL = 0, int STG = kStages)
{
    return (size_t)STG * 3 * 4 * sizeof(T) + (size_t)(K - RL) * 8 * sizeof(T) +
           (size_t)(n - K) * 2 * sizeof(T);
}

// Shared memory: the staging ring, then links RL..K-1 x 8 scalars, then
// (n - K) links x 2 scalars, each interleaved over the block's threads. The
// state of links 0..RL-1 (RL a multiple of 4, K >= RL) stays in registers: the
// chunks that hold them run as unrolled copies of the loop body, first in the
// forward sweep and last in the backward sweep, so every register index is a
// compile-time constant. With less shared memory per block more blocks are
// resident.
// VEC: n % 4 == 0 and 16-byte aligned rows; without it any n (K = n, or a multiple of
// 4) and any rows.
template <typename T, int NMAX, int BLOCK, int TRIG, int RL = 0, int STG = kStages, bool VEC = true>
__global__ void __launch_bounds__(BLOCK)
rnea_dhp_kernel(const __grid_constant__ DhParamConsts<T, NMAX> pc, int n, int K, int B,
                const T *__restrict__ q, const T *__restrict__ qd, const T *__restrict__ qdd,
                T *__restrict__ tau, BaseParams<T> base)
{
    static_assert(RL % 4 == 0 && RL >= 0 && RL <= 16, "register links: 0, 4, 8, 12 or 16");
    static_assert(STG == 2 || STG == 3, "staging ring of 2 or 3 chunks");
    constexpr int kRegChunks = RL / 4;
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned char *ring = smem;
    unsigned char *stf = ring + (size_t)STG * 3 * 4 * sizeof(T) * BLOCK;
    unsigned char *stc = stf + (size_t)(K - RL) * 8 * sizeof(T) * BLOCK;
    LinkState<T> rs[kRegChunks > 0 ? RL : 1];
    const T *sc = pc.c;

    const int tid = threadIdx.x;
    const int b = blockIdx.x * BLOCK + tid;
    if (VEC && b >= B) return;  // ragged rows: every lane stores for others
    const size_t row = (size_t)(VEC || b < B ? b : B - 1) * (size_t)n;
    const T *qr = q + row, *qdr = qd + row, *qddr = qdd + row;
    T *taur = tau + row;
    const RaggedRow<T> rr[3] = {ragged_row(qr), ragged_row(qdr), ragged_row(qddr)};
    Chunk<T> pc0[3], pc1[3];  // ragged rows: the pieces of two neighbouring chunks

    Kin<T> x = kin_base(base.V0, base.dV0);
    WMat<T> W = kin_wmat(x.w, x.al);

    // ---- forward sweep: base -> tip
    const int nchunks = VEC ? n / 4 : (n + 3) / 4, kchunks = VEC || K < n ? K / 4 : nchunks;
    Chunk<T> cq, cqd, cqdd;
    // Ragged rows need chunk kc's and chunk kc + 1's pieces at step kc (the last, of
    // index nchunks, exists where the row's offset pushes it over): a step reads the
    // pieces of kc + 1, keeps them in registers for the next, and fills the slot that
    // it emptied one step before with those of kc + STG.
    auto stage = [&](int kc) {
        if constexpr (VEC) {
            if (kc < nchunks) stage_chunk<T, BLOCK>(ring, kc % STG, tid, qr, qdr, qddr, 4 * kc);
        } else {
#pragma unroll
            for (int a = 0; a < 3; ++a) stage_pieces<T, BLOCK>(ring, kc % STG, a, rr[a], n, kc);
        }
        __pipeline_commit();
    };
#pragma unroll
    for (int k = 0; k < (VEC ? STG - 1 : STG); ++k) stage(k);
    if constexpr (!VEC) {
        __pipeline_wait_prior(STG - 1);
#pragma unroll
        for (int a = 0; a < 3; ++a) pc0[a] = read_pieces<T, BLOCK>(ring, 0, a);
    }
    // chunk kc into cq, cqd, cqdd
    auto fetch = [&](int kc) {
        if constexpr (VEC) {
            stage(kc + STG - 1);
            __pipeline_wait_prior(STG - 1);
            read_chunk<T, BLOCK>(ring, kc % STG, tid, cq, cqd, cqdd);
        } else {
            __pipeline_wait_prior(STG - 2);
#pragma unroll
            for (int a = 0; a < 3; ++a) pc1[a] = read_pieces<T, BLOCK>(ring, (kc + 1) % STG, a);
            stage(kc + STG);
            cq = shift_pieces(pc0[0], pc1[0], rr[0].off);
            cqd = shift_pieces(pc0[1], pc1[1], rr[1].off);
            cqdd = shift_pieces(pc0[2], pc1[2], rr[2].off);
#pragma unroll
            for (int a = 0; a < 3; ++a) pc0[a] = pc1[a];
        }
    };
    auto store = [&](int kc, const Chunk<T> &c) {
        if constexpr (VEC) st_chunk<T, true>(taur, 4 * kc, n, c);
        else st_chunk_ragged<T, BLOCK>(ring, kc & 1, tau, n, B, 4 * kc, c);
    };
    // one stored link of the forward sweep: motion, bias wrench, cos, sin
    auto forward_stored = [&](int i, T qi, T qdi, T qddi) -> LinkState<T> {
        DhLink<T> L;
        load_dh(sc + i * kDhConsts, L);
        T s, c;
        dh_trig<T, TRIG>(qi + L.th0, &s, &c);
        x = kin_forward(dh_rot(L.ca, L.sa, c, s), L.b, qdi, qddi, x, W);
        W = kin_wmat(x.w, x.al);
        LinkState<T> ls;
        ls.Fh = kin_wrench(L.m, L.c, L.I, W, x.a);
        ls.c = c;
        ls.s = s;
        return ls;
    };
    // the chunks whose state stays in registers
#pragma unroll
    for (int kc = 0; kc < kRegChunks; ++kc) {
        fetch(kc);
#pragma unroll
        for (int j = 0; j < 4; ++j) rs[4 * kc + j] = forward_stored(4 * kc + j, cq.v[j], cqd.v[j], cqdd.v[j]);
    }
    // The last chunk of a ragged chain is shorter; it runs as code of its own
    // (FULL = false), so that the whole chunks' links stay free of branches and their
    // loads and arithmetic interleave.
    auto forward_chunk = [&](int kc, auto full) {
        constexpr bool FULL = decltype(full)::value;
        const int i0 = 4 * kc;
        fetch(kc);
        if (kc < kchunks) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = i0 + j;
                if (FULL || i < n)
                    put_state<T>(stf, i - RL, tid, BLOCK,
                                 forward_stored(i, cq.v[j], cqd.v[j], cqdd.v[j]));
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = i0 + j;
                if (!FULL && i >= n) break;
                DhXf<T> X;
                load_dh_xf(sc + i * kDhConsts, X);
                T s, c;
                dh_trig<T, TRIG>(cq.v[j] + X.th0, &s, &c);
                x = kin_forward(dh_rot(X.ca, X.sa, c, s), X.b, cqd.v[j], cqdd.v[j], x, W);
                W = kin_wmat(x.w, x.al);
                put_cs<T>(stc, i - K, tid, BLOCK, c, s);
            }
        }
    };
    const int nfull = VEC ? nchunks : n / 4;
    for (int kc = kRegChunks; kc < nfull; ++kc) forward_chunk(kc, std::true_type());
    if (!VEC && nfull < nchunks) forward_chunk(nfull, std::false_type());

    // ---- backward sweep: tip -> base; first the links without full state
    Wrench<T> F;
    F.f = mk3(base.Fn[0], base.Fn[1], base.Fn[2]);
    F.n = mk3(base.Fn[3], base.Fn[4], base.Fn[5]);
    DhRot<T> Rn = dh_rot(T(1), T(0), T(1), T(0));  // rotation of link i+1
    V3<T> bn = mk3(T(0), T(0), T(0));
    if (!VEC) __syncwarp();  // the ring's q parts now take torques
    const int nrc = nchunks - kchunks;
    // Forward chunk c was staged in slot c % STG and is only overwritten by
    // chunk c + STG, so the ring still holds the last STG chunks: the
    // backward sweep reads those in place and stages older ones STG - 1
    // steps ahead, each into the slot of the chunk read one step before.
    // Ragged rows start over, from the tip's pieces down.
    auto stage_back = [&](int c) {
        if (c >= nchunks - nrc) {
#pragma unroll
            for (int a = 1; a < 3; ++a)
                stage_pieces<T, BLOCK>(ring, c % STG, a, rr[a], n, c);
        }
        __pipeline_commit();
    };
    if (!VEC && nrc) {
        __pipeline_wait_prior(0);
#pragma unroll
        for (int k = 0; k < STG; ++k) stage_back(nchunks - k);
        __pipeline_wait_prior(STG - 1);
#pragma unroll
        for (int a = 1; a < 3; ++a) pc1[a] = read_pieces<T, BLOCK>(ring, nchunks % STG, a);
    }
    auto rederived_chunk = [&](int kb, auto full) {
        constexpr bool FULL = decltype(full)::value;
        const int kc = nchunks - 1 - kb, i0 = 4 * kc;
        if constexpr (VEC) {
            const int ahead = kb + STG - 1;
            if (ahead >= STG && ahead < nrc) {
                const int c = nchunks - 1 - ahead;
                stage_chunk2<T, BLOCK>(ring, c % STG, tid, qdr, qddr, 4 * c);
            }
            __pipeline_commit();
            __pipeline_wait_prior(STG - 1);
            read_chunk2<T, BLOCK>(ring, kc % STG, tid, cqd, cqdd);
        } else {
            __pipeline_wait_prior(STG - 2);
#pragma unroll
            for (int a = 1; a < 3; ++a) pc0[a] = read_pieces<T, BLOCK>(ring, kc % STG, a);
            stage_back(kc + 1 - STG);
            cqd = shift_pieces(pc0[1], pc1[1], rr[1].off);
            cqdd = shift_pieces(pc0[2], pc1[2], rr[2].off);
#pragma unroll
            for (int a = 1; a < 3; ++a) pc1[a] = pc0[a];
        }
        Chunk<T> ct = {};
#pragma unroll
        for (int j = 3; j >= 0; --j) {
            const int i = i0 + j;
            if (!FULL && i >= n) continue;
            DhLink<T> L;
            load_dh(sc + i * kDhConsts, L);
            T s, c;
            get_cs<T>(stc, i - K, tid, BLOCK, c, s);
            const DhRot<T> R = dh_rot(L.ca, L.sa, c, s);
            const Wrench<T> Fh = kin_wrench(L.m, L.c, L.I, W, x.a);
            if (i == n - 1) {
                F.f = add3(F.f, Fh.f);
                F.n = add3(F.n, Fh.n);
            } else {
                F = dh_carry(Rn, bn, F, Fh);
            }
            if (i > K) x = kin_recover(R, L.b, cqd.v[j], cqdd.v[j], x, W);
            Rn = R;
            bn = L.b;
            ct.v[j] = F.n.z;
        }
        store(kc, ct);
    };
    int kb = 0;
    if (!VEC && nfull < nchunks && nrc) rederived_chunk(kb++, std::false_type());
    for (; kb < nrc; ++kb) rederived_chunk(kb, std::true_type());
    // ---- then the links with full state: shared memory, then registers
    auto backward_stored = [&](int i, const LinkState<T> &ls) -> T {
        if (i == n - 1) {
            F.f = add3(F.f, ls.Fh.f);
            F.n = add3(F.n, ls.Fh.n);
        } else {
            F = dh_carry(Rn, bn, F, ls.Fh);
        }
        DhXf<T> X;
        load_dh_xf(sc + i * kDhConsts, X);
        Rn = dh_rot(X.ca, X.sa, ls.c, ls.s);
        bn = X.b;
        return F.n.z;
    };
    auto stored_chunk = [&](int kc, auto full) {
        constexpr bool FULL = decltype(full)::value;
        const int i0 = 4 * kc;
        Chunk<T> ct = {};
#pragma unroll
        for (int j = 3; j >= 0; --j) {
            const int i = i0 + j;
            if (!FULL && i >= n) continue;
            LinkState<T> ls;
            get_state<T>(stf, i - RL, tid, BLOCK, ls);
            ct.v[j] = backward_stored(i, ls);
        }
        store(kc, ct);
    };
    if (!VEC && !nrc && nfull < nchunks) stored_chunk(nchunks - 1 - kb++, std::false_type());
    for (; kb < nchunks - kRegChunks; ++kb) stored_chunk(nchunks - 1 - kb, std::true_type());
#pragma unroll
    for (int kc = kRegChunks - 1; kc >= 0; --kc) {
        Chunk<T> ct;
#pragma unroll
        for (int j = 3; j >= 0; --j) ct.v[j] = backward_stored(4 * kc + j, rs[4 * kc + j]);
        store(kc, ct);
    }
}

}  // namespace rdyn
