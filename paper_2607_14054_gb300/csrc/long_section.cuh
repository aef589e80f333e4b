// Sections of long-memory channels (horizon above kLongHorizon) in sos_filter,
// sos_apply and sos_filtfilt with PH: one scalar chain per lane, ill-conditioned
// sections with the lane scan in double-float, and sections with double-float
// samples step by step.  The rounding errors of poles this close to the unit
// circle add up over 1e4 and more samples to 1e-5..1e-3 of a channel's output, in
// any order of operations, but other ones in each: this one is kept for its
// digits.  (Streams and plans for cyclic reduction run the same channels by
// pipe_section and pipe_section_dfx, whose errors are no larger: 64 channels of 8
// sections, radius 0.999..0.9999, by class: level 2 at most 1.6e-3 here and 4.4e-4
// there, class 3 4.9e-4 and 2.1e-4.)  The latency of the dependent steps is what
// bounds a segment; a team of warps takes its sections as stages of a pipeline
// (ws_long_phase in warpseg.cuh).
#pragma once

#include "pipe_section.cuh"

namespace sosf {

// One section over one group, lane chunk v[] in registers, from the group's
// incoming DF2T state (Z1, Z2), left outgoing: FIR with zero in-lane history,
// particular solution's terminal pair, lane scan, fold, re-run.  AL: the in-lane
// recursions add the low parts alo of a1, a2.  DFS: AL, and the scan and
// the fold in double-float (powers' low parts phi_lo, lpl; the chunk waits in the
// lane's row s_own).  ZF: the group holds the channel's last sample (element mq
// of the chunk of the lane where zf_owner is set), whose state times G goes to
// zf_dst.
template <int N, bool ZF, bool AL, bool DFS>
__device__ __forceinline__ void long_section(float (&v)[N], const float4 ab, const float b0,
                                             const float4* phi, const float4 lp, float& Z1,
                                             float& Z2, bool zf_owner, int mq, float* s_own,
                                             float* zf_dst, float G, const float2 alo,
                                             const float4* phi_lo, const float4 lpl) {
    const int lane = threadIdx.x & 31;
    const float a1 = ab.x, a2 = ab.y, b1 = ab.z, b2 = ab.w;
    // the all-pole terms, with a_i = ab + alo for AL (the low-part products go
    // first, into the smaller terms), FP32 a_i otherwise:
    // ap2 = t - a1 y1 - a2 y2, ap1 = t - a1 y1, st2 = -a1 y1 - a2 y2, st1 = -a2 y
    auto ap2 = [&](float y1, float y2, float t) {
        return fmaf(-a1, y1, fmaf(-a2, y2, AL ? fmaf(-alo.x, y1, fmaf(-alo.y, y2, t)) : t));
    };
    auto ap1 = [&](float y1, float t) { return fmaf(-a1, y1, AL ? fmaf(-alo.x, y1, t) : t); };
    auto st2 = [&](float y1, float y2) {
        return fmaf(-a1, y1, AL ? fmaf(-a2, y2, fmaf(-alo.x, y1, -alo.y * y2)) : -a2 * y2);
    };
    auto st1 = [&](float y) { return AL ? fmaf(-a2, y, -alo.y * y) : -a2 * y; };

    // S8 support: the section input at the channel's last sample (element mq
    // of the owner's chunk), picked by compile-time-indexed selects
    float xq = 0.f, xqm1 = 0.f;
    if (ZF) pick_pair<N>(v, mq, xq, xqm1);

    // S3: non-recursive stage with zero history inside the lane
    const float xl1 = v[N - 1], xl2 = v[N - 2];
#pragma unroll
    for (int m = N - 1; m >= 2; --m)
        v[m] = fmaf(b2, v[m - 2], fmaf(b1, v[m - 1], b0 * v[m]));
    v[1] = fmaf(b1, v[0], b0 * v[1]);
    v[0] = b0 * v[0];
    // S4 (i): particular solution from zero state, terminal values only
    float w0 = v[0], w1 = ap1(w0, v[1]);
#pragma unroll
    for (int m = 2; m < N; ++m) {
        const float w2 = ap2(w1, w0, v[m]);
        w0 = w1;
        w1 = w2;
    }
    float S1 = fmaf(b1, xl1, fmaf(b2, xl2, st2(w1, w0)));
    float S2 = fmaf(b2, xl1, st1(w1));

    float zin1, zin2;
    if (DFS) {
        // S4 (ii) and the fold in double-float; the chunk waits in the lane's
        // row (s_own) meanwhile, so that its registers serve the scan
        chunk_to_row<N>(v, s_own);
        df s1 = df_from(S1), s2 = df_from(S2);
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            const int d = 1 << j;
            df t1{__shfl_up_sync(0xffffffffu, s1.hi, d), __shfl_up_sync(0xffffffffu, s1.lo, d)};
            df t2{__shfl_up_sync(0xffffffffu, s2.hi, d), __shfl_up_sync(0xffffffffu, s2.lo, d)};
            if (lane < d) {
                t1 = df_from(0.f);
                t2 = df_from(0.f);
            }
            const float4 h = phi[j], l = phi_lo[j];
            s1 = df_add_fast(s1, df_add_fast(df_mul(df{h.x, l.x}, t1), df_mul(df{h.y, l.y}, t2)));
            s2 = df_add_fast(s2, df_add_fast(df_mul(df{h.z, l.z}, t1), df_mul(df{h.w, l.w}, t2)));
        }
        df e1{__shfl_up_sync(0xffffffffu, s1.hi, 1), __shfl_up_sync(0xffffffffu, s1.lo, 1)};
        df e2{__shfl_up_sync(0xffffffffu, s2.hi, 1), __shfl_up_sync(0xffffffffu, s2.lo, 1)};
        if (lane == 0) {
            e1 = df_from(0.f);
            e2 = df_from(0.f);
        }
        const df z1 = df_from(Z1), z2 = df_from(Z2);
        zin1 = df_to_float(df_add_fast(
            e1, df_add_fast(df_mul(df{lp.x, lpl.x}, z1), df_mul(df{lp.y, lpl.y}, z2))));
        zin2 = df_to_float(df_add_fast(
            e2, df_add_fast(df_mul(df{lp.z, lpl.z}, z1), df_mul(df{lp.w, lpl.w}, z2))));
        row_to_chunk<N>(v, s_own);
    } else {
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
        zin1 = fmaf(lp.x, Z1, fmaf(lp.y, Z2, E1));
        zin2 = fmaf(lp.z, Z1, fmaf(lp.w, Z2, E2));
    }

    // S4 (iii): re-run the recursion from the true incoming state
    v[0] = v[0] + zin1;
    v[1] = ap1(v[0], v[1] + zin2);
#pragma unroll
    for (int m = 2; m < N; ++m) v[m] = ap2(v[m - 1], v[m - 2], v[m]);

    // the group's outgoing state, from lane 31's last two inputs and outputs
    const float o1 = fmaf(b1, xl1, fmaf(b2, xl2, st2(v[N - 1], v[N - 2])));
    const float o2 = fmaf(b2, xl1, st1(v[N - 1]));
    Z1 = __shfl_sync(0xffffffffu, o1, 31);
    Z2 = __shfl_sync(0xffffffffu, o2, 31);
    // S8: final state at the channel's last sample
    if (ZF) {
        float yq, yqm1;
        pick_pair<N>(v, mq, yq, yqm1);
        float f1;
        if (mq >= 1) f1 = fmaf(b1, xq, fmaf(b2, xqm1, st2(yq, yqm1)));
        else f1 = fmaf(b1, xq, ap1(yq, zin2));
        const float f2 = fmaf(b2, xq, st1(yq));
        if (zf_owner) {
            zf_dst[0] = f1 * G;
            zf_dst[1] = f2 * G;
        }
    }
}

// One section over one group with the samples in double-float, step by step:
// the high parts in the lane's chunk vh[], the low parts in the lane's row
// lo[] (shared memory, 16-byte aligned, read and written four at a time).  The
// same steps as long_section, every one in double-float (about 44 bits).
template <int N, bool ZF>
__device__ __forceinline__ void long_section_dfx(float (&vh)[N], float* lo, const SecDF& q,
                                                 const float4* phi, const float4* phi_lo,
                                                 const float4 lp, const float4 lpl, df& Z1,
                                                 df& Z2, bool zf_owner, int mq, float* zf_dst) {
    const int lane = threadIdx.x & 31;
    const df na1 = df_neg(q.a1);
    float4* lo4 = reinterpret_cast<float4*>(lo);
    df xq{0.f, 0.f}, xqm1{0.f, 0.f};
    if (ZF) {
        pick_pair<N>(vh, mq, xq.hi, xqm1.hi);
        xq.lo = lo[mq];
        xqm1.lo = mq >= 1 ? lo[mq - 1] : 0.f;
    }
    const float4 top = lo4[N / 4 - 1];
    const df xl1{vh[N - 1], top.w}, xl2{vh[N - 2], top.z};
    // S3, top down (block q of four samples reads the inputs of blocks q and
    // q - 1, which the steps below it have not overwritten yet)
#pragma unroll
    for (int b = N / 4 - 1; b >= 0; --b) {
        const float4 c = lo4[b];
        const float4 d = b > 0 ? lo4[b > 0 ? b - 1 : 0] : make_float4(0.f, 0.f, 0.f, 0.f);
        const float l[6] = {d.z, d.w, c.x, c.y, c.z, c.w};  // lo of x_{4b-2} .. x_{4b+3}
        float h[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            const int m = 4 * b - 2 + i;
            h[i] = m >= 0 ? vh[m >= 0 ? m : 0] : 0.f;
        }
        float out[4];
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            const int m = 4 * b + i;
            df u;
            if (m >= 2)
                u = df_dot3(q.b0, df{h[i + 2], l[i + 2]}, q.b1, df{h[i + 1], l[i + 1]}, q.b2,
                            df{h[i], l[i]});
            else if (m == 1)
                u = df_dot3(q.b0, df{h[i + 2], l[i + 2]}, q.b1, df{h[i + 1], l[i + 1]},
                            df{0.f, 0.f}, df{0.f, 0.f});
            else
                u = df_mul(q.b0, df{h[i + 2], l[i + 2]});
            vh[m] = u.hi;
            out[i] = u.lo;
        }
        lo4[b] = make_float4(out[0], out[1], out[2], out[3]);
    }
    // S4 (i): the particular solution from zero state, its terminal pair
    df w0{0.f, 0.f}, w1{0.f, 0.f};
#pragma unroll
    for (int b = 0; b < N / 4; ++b) {
        const float4 c = lo4[b];
        const float l[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int m = 4 * b + i;
            const df u{vh[m], l[i]};
            df w2;
            if (m == 0) w2 = u;
            else if (m == 1) w2 = df_rec1(u, q.a1, w1);
            else w2 = df_rec(u, q.a1, w1, q.a2, w0);
            w0 = w1;
            w1 = w2;
        }
    }
    df s1 = df_rec1(df_dot3(q.b1, xl1, q.b2, xl2, na1, w1), q.a2, w0);
    df s2 = df_rec1(df_mul(q.b2, xl1), q.a2, w1);
    // S4 (ii): lane scan, z_{l+1} = Phi z_l + s_l, in double-float
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const int d = 1 << j;
        df t1{__shfl_up_sync(0xffffffffu, s1.hi, d), __shfl_up_sync(0xffffffffu, s1.lo, d)};
        df t2{__shfl_up_sync(0xffffffffu, s2.hi, d), __shfl_up_sync(0xffffffffu, s2.lo, d)};
        if (lane < d) {
            t1 = df{0.f, 0.f};
            t2 = df{0.f, 0.f};
        }
        const float4 h = phi[j], l = phi_lo[j];
        s1 = df_add(s1, df_add(df_mul(df{h.x, l.x}, t1), df_mul(df{h.y, l.y}, t2)));
        s2 = df_add(s2, df_add(df_mul(df{h.z, l.z}, t1), df_mul(df{h.w, l.w}, t2)));
    }
    df e1{__shfl_up_sync(0xffffffffu, s1.hi, 1), __shfl_up_sync(0xffffffffu, s1.lo, 1)};
    df e2{__shfl_up_sync(0xffffffffu, s2.hi, 1), __shfl_up_sync(0xffffffffu, s2.lo, 1)};
    if (lane == 0) {
        e1 = df{0.f, 0.f};
        e2 = df{0.f, 0.f};
    }
    // fold the group's incoming state into this lane's: Phi^lane Z + E
    const df zin1 = df_add(e1, df_add(df_mul(df{lp.x, lpl.x}, Z1), df_mul(df{lp.y, lpl.y}, Z2)));
    const df zin2 = df_add(e2, df_add(df_mul(df{lp.z, lpl.z}, Z1), df_mul(df{lp.w, lpl.w}, Z2)));
    // S4 (iii): the re-run from the true lane state
    df y1{0.f, 0.f}, y2{0.f, 0.f};  // y_{m-1}, y_{m-2}
#pragma unroll
    for (int b = 0; b < N / 4; ++b) {
        const float4 c = lo4[b];
        const float l[4] = {c.x, c.y, c.z, c.w};
        float out[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int m = 4 * b + i;
            const df u{vh[m], l[i]};
            df y;
            if (m == 0) y = df_add(u, zin1);
            else if (m == 1) y = df_rec1(df_add(u, zin2), q.a1, y1);
            else y = df_rec(u, q.a1, y1, q.a2, y2);
            vh[m] = y.hi;
            out[i] = y.lo;
            y2 = y1;
            y1 = y;
        }
        lo4[b] = make_float4(out[0], out[1], out[2], out[3]);
    }
    // the group's outgoing state, from lane 31's last two inputs and outputs
    const df o1 = df_rec1(df_dot3(q.b1, xl1, q.b2, xl2, na1, y1), q.a2, y2);
    const df o2 = df_rec1(df_mul(q.b2, xl1), q.a2, y1);
    Z1 = df{__shfl_sync(0xffffffffu, o1.hi, 31), __shfl_sync(0xffffffffu, o1.lo, 31)};
    Z2 = df{__shfl_sync(0xffffffffu, o2.hi, 31), __shfl_sync(0xffffffffu, o2.lo, 31)};
    // S8: final state at the channel's last sample
    if (ZF) {
        df yq, yqm1;
        pick_pair<N>(vh, mq, yq.hi, yqm1.hi);
        yq.lo = lo[mq];
        yqm1.lo = mq >= 1 ? lo[mq - 1] : 0.f;
        df f1;
        if (mq >= 1) f1 = df_rec1(df_dot3(q.b1, xq, q.b2, xqm1, na1, yq), q.a2, yqm1);
        else f1 = df_add(df_dot3(q.b1, xq, na1, yq, df{0.f, 0.f}, df{0.f, 0.f}), zin2);
        const df f2 = df_rec1(df_mul(q.b2, xq), q.a2, yq);
        if (zf_owner) {
            zf_dst[0] = df_to_float(f1);
            zf_dst[1] = df_to_float(f2);
        }
    }
}

}  // namespace sosf
