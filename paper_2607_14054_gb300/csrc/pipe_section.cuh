// One section of the cascade over one group of 32 N samples held as lane
// chunks in registers: S3 non-recursive stage, S4-PH (particular solution,
// lane scan, re-run from the true lane state), the group's outgoing DF2T
// state, and S8 (zf) for the lane holding the channel's last sample.  Used by the
// warp-segment and streaming kernels and the section pipeline (pipe_section,
// pipe_section_dfx, pipe_section_cr), by the backward (lane_section) and, on
// time-reversed data, by its adjoint (pipe_section_dual).
#pragma once

#include "sos_f2.cuh"
#include "sos_pipe.cuh"

namespace sosf {

// v[mq] and v[mq - 1] (0 when mq = 0) by compile-time-indexed selects, for
// a run-time mq: no dynamic register indexing, no scratch memory.
template <int N>
__device__ __forceinline__ void pick_pair(const float (&v)[N], int mq, float& q0, float& q1) {
    q0 = v[0];
    q1 = 0.f;
#pragma unroll
    for (int m = 1; m < N; ++m) {
        q0 = m == mq ? v[m] : q0;
        q1 = m == mq ? v[m - 1] : q1;
    }
}

// Chunk v[] <-> the lane's row (N floats, 16-byte aligned).
template <int N>
__device__ __forceinline__ void chunk_to_row(const float (&v)[N], float* row) {
#pragma unroll
    for (int q = 0; q < N / 4; ++q)
        *reinterpret_cast<float4*>(row + 4 * q) =
            make_float4(v[4 * q + 0], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}

template <int N>
__device__ __forceinline__ void row_to_chunk(float (&v)[N], const float* row) {
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
        const float4 t = *reinterpret_cast<const float4*>(row + 4 * q);
        v[4 * q + 0] = t.x;
        v[4 * q + 1] = t.y;
        v[4 * q + 2] = t.z;
        v[4 * q + 3] = t.w;
    }
}


// A lane's chunk of N samples as packed pairs of quarter chunks (Q = N/4):
// u[m] = (v[m], v[m + Q]), w[m] = (v[m + 2Q], v[m + 3Q]).
template <int N>
struct QChunk {
    f2x u[N / 4], w[N / 4];
};

template <int N>
__device__ __forceinline__ void row_to_q(QChunk<N>& v, const float* row) {
    constexpr int Q = N / 4;
#pragma unroll
    for (int q = 0; q < Q; q += 4) {
        const float4 a = *reinterpret_cast<const float4*>(row + q);
        const float4 b = *reinterpret_cast<const float4*>(row + Q + q);
        const float4 c = *reinterpret_cast<const float4*>(row + 2 * Q + q);
        const float4 d = *reinterpret_cast<const float4*>(row + 3 * Q + q);
        v.u[q + 0] = f2_pack(a.x, b.x);
        v.u[q + 1] = f2_pack(a.y, b.y);
        v.u[q + 2] = f2_pack(a.z, b.z);
        v.u[q + 3] = f2_pack(a.w, b.w);
        v.w[q + 0] = f2_pack(c.x, d.x);
        v.w[q + 1] = f2_pack(c.y, d.y);
        v.w[q + 2] = f2_pack(c.z, d.z);
        v.w[q + 3] = f2_pack(c.w, d.w);
    }
}

// The chunk to the lane's row, every sample times `scale` (SC).
template <int N, bool SC>
__device__ __forceinline__ void q_to_row(const QChunk<N>& v, float* row, float scale = 1.f) {
    constexpr int Q = N / 4;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const f2x* t = h ? v.w : v.u;
#pragma unroll
        for (int q = 0; q < Q; q += 4) {
            float4 a, b;
            f2_unpack(t[q + 0], a.x, b.x);
            f2_unpack(t[q + 1], a.y, b.y);
            f2_unpack(t[q + 2], a.z, b.z);
            f2_unpack(t[q + 3], a.w, b.w);
            if (SC) {
                a = make_float4(a.x * scale, a.y * scale, a.z * scale, a.w * scale);
                b = make_float4(b.x * scale, b.y * scale, b.z * scale, b.w * scale);
            }
            *reinterpret_cast<float4*>(row + 2 * Q * h + q) = a;
            *reinterpret_cast<float4*>(row + 2 * Q * h + Q + q) = b;
        }
    }
}

// v[mq] and v[mq - 1] (0 when mq = 0) for a run-time mq, through the lane's
// row as scratch (N floats, 16-byte aligned).
template <int N>
__device__ __forceinline__ void pick_q(const QChunk<N>& v, int mq, float* row, float& q0,
                                       float& q1) {
    q_to_row<N, false>(v, row);
    q0 = row[mq];
    q1 = mq >= 1 ? row[mq - 1] : 0.f;
}

// The DF2T states entering a lane's quarters (zu: quarters 0 and 1, zw: 2 and
// 3) from the quarters' zero-state outgoing states (e*u, e*w) and, with ST,
// the group's incoming state (Z1, Z2) (zero otherwise): the quarters joined
// into halves and lanes, the lanes scanned (S4 (ii), z_{l+1} = Phi z_l + s_l),
// the lane's incoming state passed on from quarter to quarter, all in the
// basis s1 = z1, s2 = (z2 - t z1) / w (t = a1/2, cpl = (w, 1/w)) that phi is
// given in.  Lane 0 starts the scan from the group's state, which so reaches
// every lane without a table of Phi^lane.
template <bool ST>
__device__ __forceinline__ void join_states(f2x e1u, f2x e2u, f2x e1w, f2x e2w, float Z1, float Z2,
                                            float t, const float2 cpl, const float4* phi, f2x& zu1,
                                            f2x& zu2, f2x& zw1, f2x& zw2) {
    const int lane = threadIdx.x & 31;
    const f2x nt = f2_dup(-t), iw = f2_dup(cpl.y);
    e2u = f2_mul(f2_fma(nt, e1u, e2u), iw);
    e2w = f2_mul(f2_fma(nt, e1w, e2w), iw);
    float s01, s11, s02, s12, s21, s31, s22, s32;
    f2_unpack(e1u, s01, s11);
    f2_unpack(e2u, s02, s12);
    f2_unpack(e1w, s21, s31);
    f2_unpack(e2w, s22, s32);
    const float4 hp = phi[5], qp = phi[6];
    const float A1 = fmaf(qp.x, s01, fmaf(qp.y, s02, s11));
    const float A2 = fmaf(qp.z, s01, fmaf(qp.w, s02, s12));
    const float B1 = fmaf(qp.x, s21, fmaf(qp.y, s22, s31));
    const float B2 = fmaf(qp.z, s21, fmaf(qp.w, s22, s32));
    float S1 = fmaf(hp.x, A1, fmaf(hp.y, A2, B1));
    float S2 = fmaf(hp.z, A1, fmaf(hp.w, A2, B2));
    const float C2 = ST ? fmaf(-t, Z1, Z2) * cpl.y : 0.f;
    if (ST && lane == 0) {
        const float4 h = phi[0];
        S1 = fmaf(h.x, Z1, fmaf(h.y, C2, S1));
        S2 = fmaf(h.z, Z1, fmaf(h.w, C2, S2));
    }
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int d = 1 << j;
        const float t1 = __shfl_up_sync(0xffffffffu, S1, d);
        const float t2 = __shfl_up_sync(0xffffffffu, S2, d);
        const float4 h = phi[j];
        if (lane >= d) {
            S1 = fmaf(h.x, t1, fmaf(h.y, t2, S1));
            S2 = fmaf(h.z, t1, fmaf(h.w, t2, S2));
        }
    }
    float q01 = __shfl_up_sync(0xffffffffu, S1, 1);
    float q02 = __shfl_up_sync(0xffffffffu, S2, 1);
    if (lane == 0) {
        q01 = ST ? Z1 : 0.f;
        q02 = C2;
    }
    const float q21 = fmaf(hp.x, q01, fmaf(hp.y, q02, A1));
    const float q22 = fmaf(hp.z, q01, fmaf(hp.w, q02, A2));
    const float q11 = fmaf(qp.x, q01, fmaf(qp.y, q02, s01));
    const float q12 = fmaf(qp.z, q01, fmaf(qp.w, q02, s02));
    const float q31 = fmaf(qp.x, q21, fmaf(qp.y, q22, s21));
    const float q32 = fmaf(qp.z, q21, fmaf(qp.w, q22, s22));
    // z2 = t s1 + w s2
    const f2x pt = f2_dup(t), pw = f2_dup(cpl.x);
    zu1 = f2_pack(q01, q11);
    zw1 = f2_pack(q21, q31);
    zu2 = f2_fma(pt, zu1, f2_mul(pw, f2_pack(q02, q12)));
    zw2 = f2_fma(pt, zw1, f2_mul(pw, f2_pack(q22, q32)));
}

// One section over one group, from the group's incoming DF2T state (Z1, Z2)
// (scaled by 1/G_k when b0 is factored); leaves the group's outgoing state in
// (Z1, Z2).  The lane's chunk is filtered as four quarters side by side, two
// packed chains of N/4 steps each from zero state; their outgoing states are
// joined into the lane's by A^(N/4) (phi[6]) and A^(N/2) (phi[5]), the lane
// states scanned, and the quarters re-run side by side from their true
// incoming states.  What bounds it is the FMA pipe (6 FMAs per sample) once
// the dependent chains and the scan are covered; measured alone (compute
// only, 12 warps per SM, clock64), samples per clock and SM: one scalar chain
// per lane 8.1 (N = 32), two half chunks packed 13.0 (N = 32) and 16.8
// (N = 64), four quarters 14.3 and 20.0 -- 0.94 of the pipe at N = 64, where
// one scan serves 2048 samples.
// The states are joined, scanned and passed on in a basis of their own, s1 =
// z1, s2 = (z2 - (a1/2) z1) / w (Coef32::cpl), in which A is a scaled rotation
// (or symmetric) and no entry of its powers much exceeds 1: in the DF2T basis
// they grow to about 1 / sin(pole angle) and the FP32 products cancel at every
// step of the scan.
// phi: the powers in that basis, Phi^(2^j), j = 0..4, A^(N/2), A^(N/4).
// cpl: w, 1/w.  ZF: the group holds the channel's last sample (at element mq
// of the chunk of the lane where zf_owner is set), whose DF2T state goes to
// zf_dst; a separate instantiation, so that other groups carry none of it.
// s_own: the lane's row (N floats, 16-byte aligned), scratch for ZF.
// AL: the in-lane recursions add the low parts alo of a1, a2 (a section
// whose poles FP32 coefficients would displace noticeably).
template <int N, bool FACT, bool ZF = false, bool AL = false>
__device__ __forceinline__ void pipe_section(QChunk<N>& v, const float4 ab, const float b0,
                                             const float4* phi, const float2 cpl, float& Z1,
                                             float& Z2, bool zf_owner, int mq, float* s_own,
                                             float* zf_dst, float G, float2 alo = {0.f, 0.f}) {
    constexpr int Q = N / 4;
    const float b1 = ab.z, b2 = ab.w;
    const f2x na1 = f2_dup(-ab.x), na2 = f2_dup(-ab.y), pb1 = f2_dup(b1), pb2 = f2_dup(b2);
    const f2x nl1 = f2_dup(AL ? -alo.x : 0.f), nl2 = f2_dup(AL ? -alo.y : 0.f);
    f2x(&u)[Q] = v.u;
    f2x(&w)[Q] = v.w;
    // the all-pole terms, with a_i = ab + alo for AL (the low-part products
    // go first, into the smaller terms), FP32 a_i otherwise:
    // ap2 = t - a1 y1 - a2 y2, ap1 = t - a1 y1, st2 = -a1 y1 - a2 y2, st1 = -a2 y
    auto ap2 = [&](f2x y1, f2x y2, f2x t) {
        return f2_fma(na1, y1, f2_fma(na2, y2, AL ? f2_fma(nl1, y1, f2_fma(nl2, y2, t)) : t));
    };
    auto ap1 = [&](f2x y1, f2x t) { return f2_fma(na1, y1, AL ? f2_fma(nl1, y1, t) : t); };
    auto st2 = [&](f2x y1, f2x y2) {
        return f2_fma(na1, y1,
                      AL ? f2_fma(na2, y2, f2_fma(nl1, y1, f2_mul(nl2, y2))) : f2_mul(na2, y2));
    };
    auto st1 = [&](f2x y) { return AL ? f2_fma(na2, y, f2_mul(nl2, y)) : f2_mul(na2, y); };

    // S8 support: the section input at the channel's last sample
    float xq = 0.f, xqm1 = 0.f;
    if (ZF) pick_q<N>(v, mq, s_own, xq, xqm1);

    // S3: non-recursive stage with zero history inside each quarter
    const f2x ux1 = u[Q - 1], ux2 = u[Q - 2], wx1 = w[Q - 1], wx2 = w[Q - 2];
    const f2x pb0 = f2_dup(b0);
#pragma unroll
    for (int m = Q - 1; m >= 2; --m) {
        u[m] = f2_fma(pb2, u[m - 2], f2_fma(pb1, u[m - 1], FACT ? u[m] : f2_mul(pb0, u[m])));
        w[m] = f2_fma(pb2, w[m - 2], f2_fma(pb1, w[m - 1], FACT ? w[m] : f2_mul(pb0, w[m])));
    }
    u[1] = f2_fma(pb1, u[0], FACT ? u[1] : f2_mul(pb0, u[1]));
    w[1] = f2_fma(pb1, w[0], FACT ? w[1] : f2_mul(pb0, w[1]));
    if (!FACT) {
        u[0] = f2_mul(pb0, u[0]);
        w[0] = f2_mul(pb0, w[0]);
    }

    // S4 (i): particular solutions from zero state, terminal values only
    f2x p0 = u[0], p1 = ap1(p0, u[1]), r0 = w[0], r1 = ap1(r0, w[1]);
#pragma unroll
    for (int m = 2; m < Q; ++m) {
        const f2x p2 = ap2(p1, p0, u[m]), r2 = ap2(r1, r0, w[m]);
        p0 = p1;
        p1 = p2;
        r0 = r1;
        r1 = r2;
    }
    // the quarters' zero-state outgoing states, and from them the quarters'
    // incoming ones
    const f2x e1u = f2_fma(pb1, ux1, f2_fma(pb2, ux2, st2(p1, p0)));
    const f2x e2u = f2_fma(pb2, ux1, st1(p1));
    const f2x e1w = f2_fma(pb1, wx1, f2_fma(pb2, wx2, st2(r1, r0)));
    const f2x e2w = f2_fma(pb2, wx1, st1(r1));
    f2x zu1, zu2, zw1, zw2;
    join_states<true>(e1u, e2u, e1w, e2w, Z1, Z2, 0.5f * ab.x, cpl, phi, zu1, zu2, zw1, zw2);

    // S4 (iii): re-run the recursions from the true incoming states
    u[0] = f2_add(u[0], zu1);
    w[0] = f2_add(w[0], zw1);
    u[1] = ap1(u[0], f2_add(u[1], zu2));
    w[1] = ap1(w[0], f2_add(w[1], zw2));
#pragma unroll
    for (int m = 2; m < Q; ++m) {
        u[m] = ap2(u[m - 1], u[m - 2], u[m]);
        w[m] = ap2(w[m - 1], w[m - 2], w[m]);
    }

    // the group's outgoing state, from lane 31's last two inputs and outputs
    const float o1 = f2_b(f2_fma(pb1, wx1, f2_fma(pb2, wx2, st2(w[Q - 1], w[Q - 2]))));
    const float o2 = f2_b(f2_fma(pb2, wx1, st1(w[Q - 1])));
    Z1 = __shfl_sync(0xffffffffu, o1, 31);
    Z2 = __shfl_sync(0xffffffffu, o2, 31);

    // S8: final state at the channel's last sample
    if (ZF) {
        float yq, yqm1;
        pick_q<N>(v, mq, s_own, yq, yqm1);
        const f2x y1 = f2_dup(yq), y2 = f2_dup(yqm1);
        float f1;
        if (mq >= 1) f1 = fmaf(b1, xq, fmaf(b2, xqm1, f2_a(st2(y1, y2))));
        else f1 = fmaf(b1, xq, f2_a(ap1(y1, zu2)));
        const float f2 = fmaf(b2, xq, f2_a(st1(y1)));
        if (zf_owner) {
            zf_dst[0] = f1 * G;
            zf_dst[1] = f2 * G;
        }
    }
}

// One section over one group with one scalar chain per lane, for the
// backward's recomputation of the section signals: its gradient sums are held
// to the rounding of this order of operations (the coefficient gradients of
// cascades whose sections cancel each other amplify any other order's).
// Arguments as above, FP32 throughout, no final state.
// INJ: a DF2T state (zi1, zi2) enters at group-relative sample pinj instead
// of the group start (the inputs before it being zero): added to the
// all-pole input at pinj and pinj + 1 (a channel's first group, whose grid is
// anchored elsewhere).
template <int N, bool FACT, bool INJ>
__device__ __forceinline__ void lane_section(float (&v)[N], const float4 ab, const float b0,
                                             const float4* phi, const float4 lp, float& Z1,
                                             float& Z2, int pinj = -1, float zi1 = 0.f,
                                             float zi2 = 0.f) {
    const int lane = threadIdx.x & 31;
    const float a1 = ab.x, a2 = ab.y, b1 = ab.z, b2 = ab.w;
    // S3: non-recursive stage with zero history inside the lane
    const float xl1 = v[N - 1], xl2 = v[N - 2];
#pragma unroll
    for (int m = N - 1; m >= 2; --m)
        v[m] = fmaf(b2, v[m - 2], fmaf(b1, v[m - 1], FACT ? v[m] : b0 * v[m]));
    v[1] = fmaf(b1, v[0], FACT ? v[1] : b0 * v[1]);
    if (!FACT) v[0] = b0 * v[0];
    if (INJ) {
#pragma unroll
        for (int m = 0; m < N; ++m) {
            const int pos = lane * N + m;
            v[m] += pos == pinj ? zi1 : (pos == pinj + 1 ? zi2 : 0.f);
        }
    }

    // S4 (i): particular solution from zero state, terminal values only
    float w0 = v[0], w1 = fmaf(-a1, w0, v[1]);
#pragma unroll
    for (int m = 2; m < N; ++m) {
        const float w2 = fmaf(-a1, w1, fmaf(-a2, w0, v[m]));
        w0 = w1;
        w1 = w2;
    }
    float S1 = fmaf(b1, xl1, fmaf(b2, xl2, fmaf(-a1, w1, -a2 * w0)));
    float S2 = fmaf(b2, xl1, -a2 * w1);

    // S4 (ii): inclusive scan over lanes, z_{l+1} = Phi z_l + s_l
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int d = 1 << j;
        float t1 = __shfl_up_sync(0xffffffffu, S1, d);
        float t2 = __shfl_up_sync(0xffffffffu, S2, d);
        t1 = lane >= d ? t1 : 0.f;
        t2 = lane >= d ? t2 : 0.f;
        S1 = fmaf(phi[j].x, t1, fmaf(phi[j].y, t2, S1));
        S2 = fmaf(phi[j].z, t1, fmaf(phi[j].w, t2, S2));
    }
    float E1 = __shfl_up_sync(0xffffffffu, S1, 1);
    float E2 = __shfl_up_sync(0xffffffffu, S2, 1);
    if (lane == 0) {
        E1 = 0.f;
        E2 = 0.f;
    }
    // fold the group's incoming state into this lane's: Phi^lane Z + E
    const float zin1 = fmaf(lp.x, Z1, fmaf(lp.y, Z2, E1));
    const float zin2 = fmaf(lp.z, Z1, fmaf(lp.w, Z2, E2));

    // S4 (iii): re-run the recursion from the true incoming state
    v[0] = v[0] + zin1;
    v[1] = fmaf(-a1, v[0], v[1] + zin2);
#pragma unroll
    for (int m = 2; m < N; ++m) v[m] = fmaf(-a1, v[m - 1], fmaf(-a2, v[m - 2], v[m]));

    // the group's outgoing state, from lane 31's last two inputs and outputs
    const float o1 = fmaf(b1, xl1, fmaf(b2, xl2, fmaf(-a1, v[N - 1], -a2 * v[N - 2])));
    const float o2 = fmaf(b2, xl1, -a2 * v[N - 1]);
    Z1 = __shfl_sync(0xffffffffu, o1, 31);
    Z2 = __shfl_sync(0xffffffffu, o2, 31);
    // a state injected at the group's last sample: its second component
    // belongs to the next group
    if (INJ && pinj == 32 * N - 1) Z1 += zi2;
}

// Coefficients of one section in double-float, for channels run in extended
// precision throughout (normalised by a0, never factored).
struct SecDF {
    df a1, a2, b0, b1, b2;
    int rounds;  // of refinement (pipe_section_dfx)
};

__device__ __forceinline__ f2x f2_neg1() { return f2_dup(-1.f); }

// The all-pole solve of one group in FP32 (a_i = hi + lo parts): y_m = v_m -
// a1 y_{m-1} - a2 y_{m-2} over the group from zero state, by quarters as in
// pipe_section (particular solutions, joins, lane scan, re-run); y may be v.
template <int N>
__device__ __forceinline__ void pole_solve(const QChunk<N>& v, QChunk<N>& y, const f2x na1,
                                           const f2x na2, const f2x nl1, const f2x nl2,
                                           const float4* phi, const float2 cpl) {
    constexpr int Q = N / 4;
    auto ap2 = [&](f2x y1, f2x y2, f2x t) {
        return f2_fma(na1, y1, f2_fma(na2, y2, f2_fma(nl1, y1, f2_fma(nl2, y2, t))));
    };
    auto ap1 = [&](f2x y1, f2x t) { return f2_fma(na1, y1, f2_fma(nl1, y1, t)); };
    f2x p0 = v.u[0], p1 = ap1(p0, v.u[1]), r0 = v.w[0], r1 = ap1(r0, v.w[1]);
#pragma unroll
    for (int m = 2; m < Q; ++m) {
        const f2x p2 = ap2(p1, p0, v.u[m]), r2 = ap2(r1, r0, v.w[m]);
        p0 = p1;
        p1 = p2;
        r0 = r1;
        r1 = r2;
    }
    f2x zu1, zu2, zw1, zw2;
    join_states<false>(f2_fma(na1, p1, f2_mul(na2, p0)), f2_mul(na2, p1),
                       f2_fma(na1, r1, f2_mul(na2, r0)), f2_mul(na2, r1), 0.f, 0.f,
                       -0.5f * f2_a(na1), cpl, phi, zu1, zu2, zw1, zw2);
    y.u[0] = f2_add(v.u[0], zu1);
    y.w[0] = f2_add(v.w[0], zw1);
    y.u[1] = ap1(y.u[0], f2_add(v.u[1], zu2));
    y.w[1] = ap1(y.w[0], f2_add(v.w[1], zw2));
#pragma unroll
    for (int m = 2; m < Q; ++m) {
        y.u[m] = ap2(y.u[m - 1], y.u[m - 2], v.u[m]);
        y.w[m] = ap2(y.w[m - 1], y.w[m - 2], v.w[m]);
    }
}

// The values at m = -j (j = 1, 2) of both pairs of quarters: quarter q's are
// the last of quarter q - 1, the first quarter's the previous lane's (zero
// for lane 0).
template <int N>
__device__ __forceinline__ void q_history(const QChunk<N>& v, int j, f2x& hu, f2x& hw) {
    constexpr int Q = N / 4;
    float ua, ub, wa, wb;
    f2_unpack(v.u[Q - j], ua, ub);
    f2_unpack(v.w[Q - j], wa, wb);
    float prev = __shfl_up_sync(0xffffffffu, wb, 1);
    if ((threadIdx.x & 31) == 0) prev = 0.f;
    hu = f2_pack(prev, ua);
    hw = f2_pack(ub, wa);
}

// The largest magnitude in the lane's chunk (NaN skipped).
template <int N>
__device__ __forceinline__ float q_max(const QChunk<N>& v) {
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
        float a, b, c, d;
        f2_unpack(v.u[i], a, b);
        f2_unpack(v.w[i], c, d);
        m = fmaxf(fmaxf(m, fmaxf(fabsf(a), fabsf(b))), fmaxf(fabsf(c), fabsf(d)));
    }
    return m;
}

// q_max of a group with infinite samples: a lane that has one takes the largest
// of the others, so that the samples before it keep the digits that their own
// magnitude gives them.
__device__ __forceinline__ float finite_max(float m) {
    float f = m < INFINITY ? m : 0.f;
    for (int o = 16; o > 0; o >>= 1) f = fmaxf(f, __shfl_xor_sync(0xffffffffu, f, o));
    return m < INFINITY ? m : f;
}

// 1.5 * 2^e such that sums of terms up to `bound` in absolute value, added to
// it one by one, stay in its binade (then each addition's rounding error is
// itself an FP32 number, recovered by two more operations).
__device__ __forceinline__ float sum_anchor(float bound) {
    const int e = min((__float_as_int(bound) >> 23) & 0xff, 251) + 2;
    return __int_as_float((e << 23) | 0x400000);
}

// One section over one group with the samples in double-float (about 44
// bits): hi and lo parts in registers, for cascades in which later sections
// attenuate what earlier ones pass (poles next to the unit circle), where FP32
// rounding of an intermediate signal reaches the output amplified many times.
// The section's banded system is solved by iterative refinement (Wilkinson;
// Higham, Accuracy and Stability of Numerical Algorithms, ch. 12): its
// right-hand side, the FIR's output, is formed to about 2^-46 of its terms;
// an FP32 solve (pole_solve) gives y0; the residual u - A y0 is formed to the
// same 2^-46, where its terms cancel; a second FP32 solve gives the
// correction, and y = y0 + correction as hi and lo parts.  Each round divides
// the error by the FP32 solve's own relative error, and the rounding of y0
// needs no compensated recursion: every chain of dependent steps is an FP32
// one, and the long sums are independent from sample to sample and packed.
// (Solving the recursions step by step in double-float takes about 27
// dependent operations per sample, twice, and a double-float scan; 16 channels
// of 100,003 samples, two sections: 203 us that way, 88 this way, segments
// included.)
// The long sums add their products one by one to an anchor far larger than
// the sum (sum_anchor): each addition's error comes back exactly from two
// more FMAs, and the errors are summed beside the low parts.
// xh, xl: the section's input, replaced by its output.  mx: max |x| of the
// lane, replaced by max |y|; wild: the group's input has infinite samples.  Z1, Z2: the group's incoming DF2T state in
// double-float, left outgoing.  refine: rounds of refinement.  ZF: the group
// holds the channel's last sample (element mq of the chunk of the lane where
// zf_owner is set), whose state goes to zf_dst; row: scratch for it.
template <int N, bool ZF = false>
__device__ __forceinline__ void pipe_section_dfx(QChunk<N>& xh, QChunk<N>& xl, float& mx,
                                                 bool wild, const SecDF& q, const float4* phi,
                                                 const float2 cpl, int refine, df& Z1, df& Z2,
                                                 bool zf_owner, int mq, float* row,
                                                 float* zf_dst) {
    constexpr int Q = N / 4;
    const int lane = threadIdx.x & 31;
    const f2x m1 = f2_neg1();
    // c += the rounding error of t = T + b x, T <- t
    auto term = [&](f2x b, f2x x, f2x& T, f2x& c) {
        const f2x t = f2_fma(b, x, T);
        c = f2_add(c, f2_fma(b, x, f2_fma(t, m1, T)));
        T = t;
    };
    // the same for t = T + v
    auto term1 = [&](f2x v, f2x& T, f2x& c) {
        const f2x t = f2_add(v, T);
        c = f2_add(c, f2_add(v, f2_fma(t, m1, T)));
        T = t;
    };
    df xq{0.f, 0.f}, xqm1{0.f, 0.f}, xp1{0.f, 0.f};
    if (ZF) {
        pick_q<N>(xh, mq, row, xq.hi, xqm1.hi);
        pick_q<N>(xl, mq, row, xq.lo, xqm1.lo);
        xp1.hi = __shfl_up_sync(0xffffffffu, f2_b(xh.w[Q - 1]), 1);
        xp1.lo = __shfl_up_sync(0xffffffffu, f2_b(xl.w[Q - 1]), 1);
    }
    // the inputs that the outgoing state is formed from
    const df xe1{f2_b(xh.w[Q - 1]), f2_b(xl.w[Q - 1])}, xe2{f2_b(xh.w[Q - 2]), f2_b(xl.w[Q - 2])};

    // S3 in double-float: u = b0 x + b1 x' + b2 x'', plus the group's state on
    // its first two samples; in place, top down
    float mu;
    {
        const float cb = fabsf(q.b0.hi) + fabsf(q.b1.hi) + fabsf(q.b2.hi);
        mu = fmaxf(mx, __shfl_up_sync(0xffffffffu, mx, 1)) * cb;
        if (lane == 0) mu += fabsf(Z1.hi) + fabsf(Z2.hi);
        mu *= 1.001f;
        const f2x M = f2_dup(sum_anchor(mu));
        const f2x b0 = f2_dup(q.b0.hi), b1 = f2_dup(q.b1.hi), b2 = f2_dup(q.b2.hi);
        const f2x l0 = f2_dup(q.b0.lo), l1 = f2_dup(q.b1.lo), l2 = f2_dup(q.b2.lo);
        f2x hu1, hw1, hu2, hw2, gu1, gw1, gu2, gw2;
        q_history<N>(xh, 1, hu1, hw1);
        q_history<N>(xh, 2, hu2, hw2);
        q_history<N>(xl, 1, gu1, gw1);
        q_history<N>(xl, 2, gu2, gw2);
        auto fir = [&](f2x& h0, f2x& g0, f2x h1, f2x g1, f2x h2, f2x g2, f2x zh, f2x zl, bool z) {
            f2x T = f2_fma(b0, h0, M);
            f2x c = f2_fma(b0, h0, f2_fma(T, m1, M));
            term(b1, h1, T, c);
            term(b2, h2, T, c);
            if (z) {
                term1(zh, T, c);
                c = f2_add(c, zl);
            }
            c = f2_fma(b0, g0, f2_fma(l0, h0, c));
            c = f2_fma(b1, g1, f2_fma(l1, h1, c));
            c = f2_fma(b2, g2, f2_fma(l2, h2, c));
            h0 = f2_fma(M, m1, T);
            g0 = c;
        };
        const bool l0z = lane == 0;
        const f2x zh1 = f2_pack(l0z ? Z1.hi : 0.f, 0.f), zl1 = f2_pack(l0z ? Z1.lo : 0.f, 0.f);
        const f2x zh2 = f2_pack(l0z ? Z2.hi : 0.f, 0.f), zl2 = f2_pack(l0z ? Z2.lo : 0.f, 0.f);
#pragma unroll
        for (int m = Q - 1; m >= 2; --m) {
            fir(xh.u[m], xl.u[m], xh.u[m - 1], xl.u[m - 1], xh.u[m - 2], xl.u[m - 2], 0, 0, false);
            fir(xh.w[m], xl.w[m], xh.w[m - 1], xl.w[m - 1], xh.w[m - 2], xl.w[m - 2], 0, 0, false);
        }
        fir(xh.u[1], xl.u[1], xh.u[0], xl.u[0], hu1, gu1, zh2, zl2, true);
        fir(xh.w[1], xl.w[1], xh.w[0], xl.w[0], hw1, gw1, 0, 0, false);
        fir(xh.u[0], xl.u[0], hu1, gu1, hu2, gu2, zh1, zl1, true);
        fir(xh.w[0], xl.w[0], hw1, gw1, hw2, gw2, 0, 0, false);
    }

    // S4: the FP32 solve, then refinement; xh, xl hold the right-hand side
    const f2x na1 = f2_dup(-q.a1.hi), na2 = f2_dup(-q.a2.hi);
    const f2x nl1 = f2_dup(-q.a1.lo), nl2 = f2_dup(-q.a2.lo);
    QChunk<N> y, d;
    pole_solve<N>(xh, y, na1, na2, nl1, nl2, phi, cpl);
    mx = q_max<N>(y);
    if (wild) mx = finite_max(mx);
#pragma unroll 1
    for (int it = 0;; ++it) {
        const float my = fmaxf(mx, __shfl_up_sync(0xffffffffu, mx, 1));
        const f2x M = f2_dup(sum_anchor(1.001f * fmaf(4.f, my, mu)));
        f2x hu1, hw1, hu2, hw2;
        q_history<N>(y, 1, hu1, hw1);
        q_history<N>(y, 2, hu2, hw2);
        auto res = [&](f2x h, f2x g, f2x y0, f2x y1, f2x y2) -> f2x {
            f2x T = f2_add(h, M);
            f2x c = f2_add(g, f2_add(h, f2_fma(T, m1, M)));
            term(na1, y1, T, c);
            term(na2, y2, T, c);
            term(m1, y0, T, c);
            c = f2_fma(nl1, y1, f2_fma(nl2, y2, c));
            return f2_add(f2_fma(M, m1, T), c);
        };
#pragma unroll
        for (int m = 0; m < Q; ++m) {
            d.u[m] = res(xh.u[m], xl.u[m], y.u[m], m >= 1 ? y.u[m >= 1 ? m - 1 : 0] : hu1,
                         m >= 2 ? y.u[m >= 2 ? m - 2 : 0] : (m == 1 ? hu1 : hu2));
            d.w[m] = res(xh.w[m], xl.w[m], y.w[m], m >= 1 ? y.w[m >= 1 ? m - 1 : 0] : hw1,
                         m >= 2 ? y.w[m >= 2 ? m - 2 : 0] : (m == 1 ? hw1 : hw2));
        }
        pole_solve<N>(d, d, na1, na2, nl1, nl2, phi, cpl);
        if (it + 1 >= refine) break;
        // another round from the corrected solution, rounded
#pragma unroll
        for (int m = 0; m < Q; ++m) {
            y.u[m] = f2_add(y.u[m], d.u[m]);
            y.w[m] = f2_add(y.w[m], d.w[m]);
        }
        mx = q_max<N>(y);
        if (wild) mx = finite_max(mx);
    }
    // y + d as hi and lo parts
#pragma unroll
    for (int m = 0; m < Q; ++m) {
        xh.u[m] = f2_add(y.u[m], d.u[m]);
        xl.u[m] = f2_add(d.u[m], f2_fma(xh.u[m], m1, y.u[m]));
        xh.w[m] = f2_add(y.w[m], d.w[m]);
        xl.w[m] = f2_add(d.w[m], f2_fma(xh.w[m], m1, y.w[m]));
    }

    // S8 support: the state's second component entering this lane
    df zin2{0.f, 0.f};
    const df na1d = df_neg(q.a1);
    if (ZF) {
        const df yp{__shfl_up_sync(0xffffffffu, f2_b(xh.w[Q - 1]), 1),
                    __shfl_up_sync(0xffffffffu, f2_b(xl.w[Q - 1]), 1)};
        zin2 = lane == 0 ? Z2 : df_rec1(df_mul(q.b2, xp1), q.a2, yp);
    }
    // the group's outgoing state, from lane 31's last two inputs and outputs
    const df ye1{f2_b(xh.w[Q - 1]), f2_b(xl.w[Q - 1])}, ye2{f2_b(xh.w[Q - 2]), f2_b(xl.w[Q - 2])};
    const df o1 = df_rec1(df_dot3(q.b1, xe1, q.b2, xe2, na1d, ye1), q.a2, ye2);
    const df o2 = df_rec1(df_mul(q.b2, xe1), q.a2, ye1);
    Z1 = df{__shfl_sync(0xffffffffu, o1.hi, 31), __shfl_sync(0xffffffffu, o1.lo, 31)};
    Z2 = df{__shfl_sync(0xffffffffu, o2.hi, 31), __shfl_sync(0xffffffffu, o2.lo, 31)};
    // S8: final state at the channel's last sample
    if (ZF) {
        df yq, yqm1;
        pick_q<N>(xh, mq, row, yq.hi, yqm1.hi);
        pick_q<N>(xl, mq, row, yq.lo, yqm1.lo);
        df f1;
        if (mq >= 1) f1 = df_rec1(df_dot3(q.b1, xq, q.b2, xqm1, na1d, yq), q.a2, yqm1);
        else f1 = df_add(df_dot3(q.b1, xq, na1d, yq, df{0.f, 0.f}, df{0.f, 0.f}), zin2);
        const df f2 = df_rec1(df_mul(q.b2, xq), q.a2, yq);
        if (zf_owner) {
            zf_dst[0] = df_to_float(f1);
            zf_dst[1] = df_to_float(f2);
        }
    }
}

// The same section solved by cyclic reduction (Sec. VI-C) instead of PH.
// Register m across the 32 lanes is the strided block y_m of Eq.
// cr_permuted_system, and S_R (the shift onto the previous lane) is a
// one-lane shuffle, zero for lane 0: the group's incoming DF2T state enters
// as the corrections to lane 0's v_0 and v_1 (Eq. feedforward_block_uniform).
//   reduction (Eq. cr_elim_step2), level i, s = 2^i, kept blocks m = 2s-1,
//     4s-1, ..: v_m <- v_m - e_i v_{m-s} + f_i v_{m-2s}, and the eliminated
//     block keeps v~_{m-s} = v_{m-s} - g_i v_{m-2s} (g_i = f_i / e_i);
//   terminal block (Eq. cr_terminal_block): Y_l + e_n Y_{l-1} + f_n Y_{l-2}
//     = V_l across lanes, by a 5-round scan;
//   back substitution (Eqs. cr_backsub_penultimate, cr_backsub_final):
//     y_{m-s} = v~_{m-s} - c_i y_{m-2s} - d_i y_{m-4s}, indices below 0
//     taken from the previous lane (S_R) or the one before (S_R^2).
// Sequential depth log2 N per stage instead of N.
template <int N, bool FACT, bool ZF = false>
__device__ __forceinline__ void pipe_section_cr(float (&v)[N], const float4 ab, const float b0,
                                                const float4* cr, float& Z1, float& Z2,
                                                bool zf_owner, int mq, float* s_own,
                                                float* zf_dst, float G) {
    // cr: cr_lv[6], cr_d[2], cr_tpow[5], cr_misc (the Coef32 fields, staged)
    const float4* lv = cr;
    const float* dd = reinterpret_cast<const float*>(cr + 6);
    const float4* tp = cr + 8;
    const int lane = threadIdx.x & 31;
    const float a1 = ab.x, a2 = ab.y, b1 = ab.z, b2 = ab.w;
    const float zi1 = Z1, zi2 = Z2;

    float xq = 0.f, xqm1 = 0.f;
    if (ZF) pick_pair<N>(v, mq, xq, xqm1);

    // S3 with the true history: the previous lane's last two inputs (lane 0's
    // history is inside the group state)
    const float xl1 = v[N - 1], xl2 = v[N - 2];
    float px1 = __shfl_up_sync(0xffffffffu, xl1, 1);
    float px2 = __shfl_up_sync(0xffffffffu, xl2, 1);
    if (lane == 0) {
        px1 = 0.f;
        px2 = 0.f;
    }
#pragma unroll
    for (int m = N - 1; m >= 2; --m)
        v[m] = fmaf(b2, v[m - 2], fmaf(b1, v[m - 1], FACT ? v[m] : b0 * v[m]));
    v[1] = fmaf(b2, px1, fmaf(b1, v[0], FACT ? v[1] : b0 * v[1]));
    v[0] = fmaf(b2, px2, fmaf(b1, px1, FACT ? v[0] : b0 * v[0]));
    if (lane == 0) {
        v[0] += zi1;
        v[1] += zi2;
    }

    // reduction
#pragma unroll
    for (int i = 0; (1 << i) < N; ++i) {
        const int s = 1 << i;
        const float4 q = lv[i];  // e, f, g, c
        float pv = __shfl_up_sync(0xffffffffu, v[N - 1], 1);
        if (lane == 0) pv = 0.f;
#pragma unroll
        for (int m = N - 1; m >= 2 * s - 1; m -= 2 * s) {
            const float vms = v[m - s];
            const float vm2s = m - 2 * s >= 0 ? v[m - 2 * s] : pv;
            v[m] = fmaf(q.y, vm2s, fmaf(-q.x, vms, v[m]));
            v[m - s] = fmaf(-q.z, vm2s, vms);
        }
    }

    // terminal recurrence across lanes: inclusive scan of (Y_l, Y_{l-1})
    float S1 = v[N - 1], S2 = 0.f;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int d = 1 << j;
        float t1 = __shfl_up_sync(0xffffffffu, S1, d);
        float t2 = __shfl_up_sync(0xffffffffu, S2, d);
        t1 = lane >= d ? t1 : 0.f;
        t2 = lane >= d ? t2 : 0.f;
        S1 = fmaf(tp[j].x, t1, fmaf(tp[j].y, t2, S1));
        S2 = fmaf(tp[j].z, t1, fmaf(tp[j].w, t2, S2));
    }
    v[N - 1] = S1;
    const float Y1 = S2;  // S_R y_{N-1}: the previous lane's (0 for lane 0)
    float Y2 = __shfl_up_sync(0xffffffffu, S2, 1);  // S_R^2 y_{N-1}
    if (lane == 0) Y2 = 0.f;

    // back substitution
    constexpr int kLv = N == 16 ? 4 : N == 32 ? 5 : 6;
#pragma unroll
    for (int ii = 0; ii < kLv; ++ii) {
        const int lvl = kLv - 1 - ii;
        const int s = 1 << lvl;
        const float c = lv[lvl].w, d = dd[lvl];
        float sh4 = Y2;  // S_R y_{N-2s-1}, or S_R^2 y_{N-1} when 2s = N
        if (2 * s + 1 <= N) {
            sh4 = __shfl_up_sync(0xffffffffu, v[(N - 2 * s - 1) >= 0 ? N - 2 * s - 1 : 0], 1);
            if (lane == 0) sh4 = 0.f;
        }
#pragma unroll
        for (int m = 2 * s - 1; m < N; m += 2 * s) {
            const float ym2s = m - 2 * s >= 0 ? v[m - 2 * s >= 0 ? m - 2 * s : 0] : Y1;
            const int q = m - 4 * s;
            const float ym4s = q >= 0 ? v[q >= 0 ? q : 0] : (q == -1 ? Y1 : sh4);
            v[m - s] = fmaf(-d, ym4s, fmaf(-c, ym2s, v[m - s]));
        }
    }

    // the group's outgoing state, from lane 31's last two inputs and outputs
    const float o1 = fmaf(b1, xl1, fmaf(b2, xl2, fmaf(-a1, v[N - 1], -a2 * v[N - 2])));
    const float o2 = fmaf(b2, xl1, -a2 * v[N - 1]);
    Z1 = __shfl_sync(0xffffffffu, o1, 31);
    Z2 = __shfl_sync(0xffffffffu, o2, 31);

    // S8: final state at the channel's last sample
    if (ZF) {
        // DF2T z2 entering this lane: b2 x_{-1} - a2 y_{-1}
        const float zin2 = lane == 0 ? zi2 : fmaf(b2, px1, -a2 * Y1);
        float yq, yqm1;
        pick_pair<N>(v, mq, yq, yqm1);
        float f1;
        if (mq >= 1) f1 = fmaf(b1, xq, fmaf(b2, xqm1, fmaf(-a1, yq, -a2 * yqm1)));
        else f1 = fmaf(b1, xq, fmaf(-a1, yq, zin2));
        const float f2 = fmaf(b2, xq, -a2 * yq);
        if (zf_owner) {
            zf_dst[0] = f1 * G;
            zf_dst[1] = f2 * G;
        }
    }
}

// The adjoint's two runs of one section on the same reversed input g, fused
// so that their recursions interleave (two independent chains per lane): l
// gets the all-pole part (lambda, from state (L1, L2)), u the whole section
// with coefficients (b0, b1, b2) (dL/du, from state (U1, U2)).  Both share
// the poles, hence Phi^(2^j) and Phi^lane.  Same arithmetic as two
// lane_section calls (in DF2T states).
template <int N>
__device__ __forceinline__ void pipe_section_dual(float (&l)[N], float (&u)[N], const float a1,
                                                  const float a2, const float b0, const float b1,
                                                  const float b2, const float4* phi,
                                                  const float4 lp, float& L1, float& L2,
                                                  float& U1, float& U2) {
    const int lane = threadIdx.x & 31;
    // S3 for u (l has no FIR)
    const float xl1 = u[N - 1], xl2 = u[N - 2];
#pragma unroll
    for (int m = N - 1; m >= 2; --m) u[m] = fmaf(b2, u[m - 2], fmaf(b1, u[m - 1], b0 * u[m]));
    u[1] = fmaf(b1, u[0], b0 * u[1]);
    u[0] = b0 * u[0];

    // S4 (i): both particular solutions, interleaved
    float lw0 = l[0], lw1 = fmaf(-a1, lw0, l[1]);
    float uw0 = u[0], uw1 = fmaf(-a1, uw0, u[1]);
#pragma unroll
    for (int m = 2; m < N; ++m) {
        const float lw2 = fmaf(-a1, lw1, fmaf(-a2, lw0, l[m]));
        const float uw2 = fmaf(-a1, uw1, fmaf(-a2, uw0, u[m]));
        lw0 = lw1;
        lw1 = lw2;
        uw0 = uw1;
        uw1 = uw2;
    }
    float LS1 = fmaf(-a1, lw1, -a2 * lw0);
    float LS2 = -a2 * lw1;
    float US1 = fmaf(b1, xl1, fmaf(b2, xl2, fmaf(-a1, uw1, -a2 * uw0)));
    float US2 = fmaf(b2, xl1, -a2 * uw1);

    // S4 (ii): both lane scans
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int d = 1 << j;
        float t1 = __shfl_up_sync(0xffffffffu, LS1, d);
        float t2 = __shfl_up_sync(0xffffffffu, LS2, d);
        float t3 = __shfl_up_sync(0xffffffffu, US1, d);
        float t4 = __shfl_up_sync(0xffffffffu, US2, d);
        t1 = lane >= d ? t1 : 0.f;
        t2 = lane >= d ? t2 : 0.f;
        t3 = lane >= d ? t3 : 0.f;
        t4 = lane >= d ? t4 : 0.f;
        const float4 ph = phi[j];
        LS1 = fmaf(ph.x, t1, fmaf(ph.y, t2, LS1));
        LS2 = fmaf(ph.z, t1, fmaf(ph.w, t2, LS2));
        US1 = fmaf(ph.x, t3, fmaf(ph.y, t4, US1));
        US2 = fmaf(ph.z, t3, fmaf(ph.w, t4, US2));
    }
    float LE1 = __shfl_up_sync(0xffffffffu, LS1, 1);
    float LE2 = __shfl_up_sync(0xffffffffu, LS2, 1);
    float UE1 = __shfl_up_sync(0xffffffffu, US1, 1);
    float UE2 = __shfl_up_sync(0xffffffffu, US2, 1);
    if (lane == 0) {
        LE1 = 0.f;
        LE2 = 0.f;
        UE1 = 0.f;
        UE2 = 0.f;
    }
    const float lz1 = fmaf(lp.x, L1, fmaf(lp.y, L2, LE1));
    const float lz2 = fmaf(lp.z, L1, fmaf(lp.w, L2, LE2));
    const float uz1 = fmaf(lp.x, U1, fmaf(lp.y, U2, UE1));
    const float uz2 = fmaf(lp.z, U1, fmaf(lp.w, U2, UE2));

    // S4 (iii): both re-runs, interleaved
    l[0] = l[0] + lz1;
    l[1] = fmaf(-a1, l[0], l[1] + lz2);
    u[0] = u[0] + uz1;
    u[1] = fmaf(-a1, u[0], u[1] + uz2);
#pragma unroll
    for (int m = 2; m < N; ++m) {
        l[m] = fmaf(-a1, l[m - 1], fmaf(-a2, l[m - 2], l[m]));
        u[m] = fmaf(-a1, u[m - 1], fmaf(-a2, u[m - 2], u[m]));
    }

    // the group's outgoing states, from lane 31
    const float lo1 = fmaf(-a1, l[N - 1], -a2 * l[N - 2]);
    const float lo2 = -a2 * l[N - 1];
    const float uo1 = fmaf(b1, xl1, fmaf(b2, xl2, fmaf(-a1, u[N - 1], -a2 * u[N - 2])));
    const float uo2 = fmaf(b2, xl1, -a2 * u[N - 1]);
    L1 = __shfl_sync(0xffffffffu, lo1, 31);
    L2 = __shfl_sync(0xffffffffu, lo2, 31);
    U1 = __shfl_sync(0xffffffffu, uo1, 31);
    U2 = __shfl_sync(0xffffffffu, uo2, 31);
}


}  // namespace sosf
