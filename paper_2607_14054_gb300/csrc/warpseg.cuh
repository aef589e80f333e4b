// Warp-segment forward kernel for channels within their memory horizon.
//
// The alternative to the section pipeline (pipe.cu) for the same segments:
// one warp runs all K sections of its own segment, group after group, each
// section carrying its DF2T state from one group to the next in registers
// (the paper's group chaining, Sec. V).  A GPU holds a few thousand such
// independent streams and none waits on another warp: there are no
// hand-overs and no pipeline fill, at the price of segments short enough to
// give every warp work, and so a larger share of warm-up (the memory horizon
// P, run from zero state before every segment but a channel's first).
//
// Per warp: two shared-memory slots of one group each (rows padded to N + 4
// floats).  While the sections run on one group in registers, cp.async fills
// the other slot with the next group (of this segment, or the first of the
// warp's next one).  The stride-N permutation in and out is paid once per
// group for the whole cascade (Sec. VII-B).
#pragma once

#include <type_traits>

#include "long_section.cuh"
#include "sos_pipe.cuh"

namespace sosf {

constexpr int kWsWarps = 4;  // warps per CTA
constexpr int kWsThreads = kWsWarps * 32;

// CTAs per SM the register budget is sized for.  N = 64: two, 255 registers
// per thread.  The FMA pipe is what bounds the section code and two packed
// chains per lane keep it busy, so more warps bring little, while at three
// (168 registers) the loops around the section spilled and the shared memory of
// three left too little L1 for what they spilled: 2^24 samples, K = 8, 71
// against 63 us; 4096 uneven channels 6.3 against 5.7 ms; 64 channels in
// double-float 20.1 against 14.5 ms.  N = 16 and 32 have shorter chunks.
template <int N>
__host__ __device__ constexpr int ws_ctas_per_sm() {
    return N == 64 ? 2 : 3;
}

template <int N>
struct WsCfg {
    static constexpr int kGroup = 32 * N;
    static constexpr int kGran = kGroup / 4;
    static constexpr int kSlot = 32 * (N + 4);  // floats per slot
    // two slots per warp; the long-memory teams share twelve for ext_n(N)
    static constexpr int kLongSlot = 32 * (ext_n(N) + 4);
    static constexpr int kFloats =
        kSlot * 2 * kWsWarps > 12 * kLongSlot ? kSlot * 2 * kWsWarps : 12 * kLongSlot;
    static constexpr size_t kSmem = sizeof(float) * kFloats;
};

// the asynchronous copies of one group (rem samples left in the channel)
template <int N>
__device__ __forceinline__ void ws_load(const float* src, int64_t rem, float* slot, int lane) {
    using SL = SlotLayout<N>;
    using WC = WsCfg<N>;
    if (rem >= WC::kGroup && ((reinterpret_cast<uintptr_t>(src) & 15u) == 0)) {
        const float4* s4 = reinterpret_cast<const float4*>(src);
#pragma unroll
        for (int q = 0; q < WC::kGran / 32; ++q)
            cp_async16(slot + SL::gran(q * 32 + lane), s4 + q * 32 + lane);
    } else {
        const int r = (int)(rem < WC::kGroup ? rem : WC::kGroup);
        for (int j = lane; j < WC::kGroup; j += 32)
            cp_async4(slot + SL::elem(j), j < r ? src + j : src, j < r);
    }
    cp_async_commit();
}

// One warp's segment, in shared memory: what the groups' loads and stores
// need, read where they need it, so that nothing of it is live in registers
// through the section loop (at N = 64 the chunk alone takes 64 of the 255).
struct WsSeg {
    int64_t base;   // packed index of the first computed sample (off + cstart)
    int64_t rbase;  // packed index of that sample's mirror image in the channel
    int64_t nbase;  // of the warp's next segment's, -1 if there is none to prefetch
    int rem, nrem;  // samples of the channel from there on (capped)
    int a, b;       // the segment's own outputs, relative to base
    int c, K, ngroups;
    int zrel;       // the channel's last sample relative to base where the segment
                    // holds it and the call asks for final states, else -1
    int first;      // the segment starts at the channel's start, from zi
    int cur;        // the slot that holds the segment's first group
    int64_t next, total;  // the warp's next segment, and where they end
};

__device__ __forceinline__ int ws_cap(int64_t n) {
    return (int)(n < 0x40000000 ? n : 0x40000000);
}

// What every group reads of a section's coefficients (Coef32's ab, misc, phi_c
// and cpl, in that order), kept by each warp in shared memory for the channel
// of its segment: read from global memory they would be evicted from the
// little L1 that the group slots leave by the streaming stores, a round trip
// to L2 in every section (N = 64, measured with 12 warps per SM, compute only:
// 1,214 against 1,098 cycles per section of a 2048-sample group, before any
// store; the kernel runs eight).
struct WsCoef {
    float4 ab, misc, phi[7], cpl;
};

// Everything of a CTA in shared memory besides the slots.
struct WsShared {
    float4 z[kWsWarps][kMaxSections];     // the sections' DF2T states
    WsCoef cf[kWsWarps][kMaxSections];
    WsSeg seg[kWsWarps];
    Params p;                             // the call's parameters
    int64_t item[kWsWarps];               // the segment a long-memory team works on
};
static __shared__ WsShared s_ws;
extern __shared__ float4 s_ws_slots[];

__device__ __forceinline__ int ws_warp() { return threadIdx.x >> 5; }
// the warp's slots in a kernel for N samples per lane, as a float offset
template <int N>
__device__ __forceinline__ int ws_slot_base() {
    return ws_warp() * 2 * WsCfg<N>::kSlot;
}
__device__ __forceinline__ float* ws_slots(int base) {
    return reinterpret_cast<float*>(s_ws_slots) + base;
}

// Precision class of a channel (ChanInfo::ext), which selects the
// instantiation of the segment code that runs it.
enum WsPrec {
    kPrecF32 = 0,  // every section in FP32
    kPrecAL = 1,   // sections flagged in Coef32::misc.w: coefficient low parts in the in-lane
                   // recursions
    kPrecDF = 2    // a range of sections with double-float samples (ChanInfo::dflo..dfhi),
                   // the others as kPrecAL
};

// The section coefficients of a channel run with double-float samples.
__device__ __forceinline__ SecDF load_secdf(const Coef32* cf) {
    const float4 ab = cf->ab, alo = cf->alo, br = cf->braw, bl = cf->blo;
    return SecDF{df{ab.x, alo.x}, df{ab.y, alo.y}, df{br.x, bl.x}, df{br.y, bl.y},
                 df{br.z, bl.z}, br.w > 1.5f ? 2 : 1};
}

// the copies of a channel's K sections, one cp.async group; cx: where the
// channel's powers for other than the plan's N samples per lane are, else null
__device__ __forceinline__ void ws_stage(const Coef32* cf0, const CoefDF* cx, int K, WsCoef* sc,
                                         int lane) {
    for (int i = lane; i < 10 * K; i += 32) {
        const int k = i / 10, f = i % 10;
        const float4* src = f == 0 ? &cf0[k].ab : f == 1 ? &cf0[k].misc : &cf0[k].phi_c[0] + f - 2;
        if (cx && f >= 2 && f < 9)
            src = &reinterpret_cast<const LongCoef*>(cx + k)->phi_x[0] + f - 2;
        cp_async16(reinterpret_cast<float4*>(sc) + i, src);
    }
    cp_async_commit();
}

// Sections [k0, k1) of a channel run with double-float samples over one
// group (kPrecDF): on entry the lane's row holds its chunk of the range's
// FP32 input, on exit the chunk of its output, rounded once.
template <int N, bool ZF>
__device__ __forceinline__ void dfx_group(int k0, int k1, int c, int row_at, int owner, int mq) {
    const Params& p = s_ws.p;
    const int lane = threadIdx.x & 31;
    float4* zs = s_ws.z[ws_warp()];
    const WsCoef* sc = s_ws.cf[ws_warp()];
    const Coef32* cf0 = p.c32 + (int64_t)c * p.kmax;
    float* row = ws_slots(row_at);
    QChunk<N> xh, xl;
    row_to_q<N>(xh, row);
#pragma unroll
    for (int m = 0; m < N / 4; ++m) {
        xl.u[m] = 0;
        xl.w[m] = 0;
    }
    float mx = q_max<N>(xh);
    const bool wild = __any_sync(0xffffffffu, mx == INFINITY);
    if (wild) mx = finite_max(mx);
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        const SecDF sd = load_secdf(cf0 + k);
        float* zf_dst = ZF ? p.zf + ((int64_t)c * p.kmax + k) * 2 : nullptr;
        const float4 zz = zs[k];
        df z1{zz.x, zz.y}, z2{zz.z, zz.w};
        pipe_section_dfx<N, ZF>(xh, xl, mx, wild, sd, sc[k].phi,
                                make_float2(sc[k].cpl.x, sc[k].cpl.y),
                                sd.rounds, z1, z2, lane == owner, mq, row,
                                zf_dst);
        if (lane == 0) zs[k] = make_float4(z1.hi, z1.lo, z2.hi, z2.lo);
    }
#pragma unroll
    for (int m = 0; m < N / 4; ++m) {
        xh.u[m] = f2_add(xh.u[m], xl.u[m]);
        xh.w[m] = f2_add(xh.w[m], xl.w[m]);
    }
    q_to_row<N, false>(xh, row);
}

// Sections [k0, k1) of a channel over one group in FP32, the chunk in
// registers; zs: their DF2T states (lo parts left zero), sc: their staged
// coefficients.  One copy of the section code (a rolled loop keeps the
// kernel's instruction footprint inside the instruction cache).
// PREC = kPrecAL: each section's level (Coef32::misc.w) picks the coefficient
// low parts.
// RAW: b0, b1, b2 normalised by a0 only (the double-float range's
// neighbours, whose states are not scaled by the factored gains).
template <int N, bool FACT, bool ZF, int PREC, bool RAW>
__device__ __forceinline__ void ws_sections(const Params& p, int c, const Coef32* cf0, int k0,
                                            int k1, QChunk<N>& v, float* row, float4* zs,
                                            const WsCoef* sc, int lane, int owner, int mq) {
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        const Coef32* cf = cf0 + k;
        float4 ab = sc[k].ab;
        float b0 = FACT ? 1.f : sc[k].misc.x;
        if (RAW) {
            const float4 br = cf->braw;
            ab.z = br.y;
            ab.w = br.z;
            b0 = br.x;
        }
        const float G = (ZF && FACT) ? sc[k].misc.y : 1.f;
        float* zf_dst = ZF ? p.zf + ((int64_t)c * p.kmax + k) * 2 : nullptr;
        const float4 zz = zs[k];
        float2 z = make_float2(zz.x, zz.z);
        const float2 cpl = make_float2(sc[k].cpl.x, sc[k].cpl.y);
        if (PREC != kPrecF32 && sc[k].misc.w > 0.5f) {
            const float4 alo = cf->alo;
            pipe_section<N, FACT, ZF, true>(v, ab, b0, sc[k].phi, cpl, z.x, z.y, lane == owner, mq,
                                            row, zf_dst, G, make_float2(alo.x, alo.y));
        } else {
            pipe_section<N, FACT, ZF>(v, ab, b0, sc[k].phi, cpl, z.x, z.y, lane == owner, mq, row,
                                      zf_dst, G);
        }
        // every lane holds the outgoing state; the writes agree
        if (lane == 0) zs[k] = make_float4(z.x, 0.f, z.y, 0.f);
    }
}

// The same by cyclic reduction (whole channels only, FP32).
template <int N, bool FACT, bool ZF>
__device__ __forceinline__ void ws_sections_cr(const Params& p, int c, const Coef32* cf0, int K,
                                               float (&v)[N], float* row, float4* zs, int lane,
                                               int owner, int mq) {
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        const Coef32* cf = cf0 + k;
        const float4 ab = cf->ab, zz = zs[k];
        const float b0 = FACT ? 1.f : cf->misc.x;
        const float G = (ZF && FACT) ? cf->misc.y : 1.f;
        float* zf_dst = ZF ? p.zf + ((int64_t)c * p.kmax + k) * 2 : nullptr;
        float2 z = make_float2(zz.x, zz.z);
        pipe_section_cr<N, FACT, ZF>(v, ab, b0, &cf->cr_lv[0], z.x, z.y, lane == owner, mq, row,
                                     zf_dst, G);
        if (lane == 0) zs[k] = make_float4(z.x, 0.f, z.y, 0.f);
    }
}

// One group through all K sections: the lane's chunk from its row into
// registers, filtered, and back.  ZF: the group holding the channel's last sample, element mq of lane owner's
// chunk; instantiated apart so that the hot loop holds no zf code.  PREC: the
// channel's precision class (WsPrec), apart for the same reason.
template <int N, bool FACT, bool CR, bool ZF, int PREC>
__device__ __forceinline__ void ws_filter(int row_at, int c, int K, int owner, int mq) {
    const Params& p = s_ws.p;
    const int lane = threadIdx.x & 31, w = ws_warp();
    float4* zs = s_ws.z[w];
    const WsCoef* sc = s_ws.cf[w];
    float* row = ws_slots(row_at);
    const Coef32* cf0 = p.c32 + (int64_t)c * p.kmax;
    if constexpr (CR) {
        float v[N];
        row_to_chunk<N>(v, row);
        ws_sections_cr<N, FACT, ZF>(p, c, cf0, K, v, row, zs, lane, owner, mq);
        if (FACT) {
            const float Gk = cf0[K - 1].misc.y;
#pragma unroll
            for (int m = 0; m < N; ++m) v[m] *= Gk;
        }
        chunk_to_row<N>(v, row);
    } else {
        QChunk<N> v;
        row_to_q<N>(v, row);
        if (PREC == kPrecDF) {
            // FP32 sections before and after the double-float range (their b
            // coefficients unfactored, like the range's), the range itself
            // with double-float samples
            const ChanInfo& ci = p.chan[c];
            const int dlo = ci.dflo, dhi = ci.dfhi;
            ws_sections<N, false, ZF, kPrecAL, true>(p, c, cf0, 0, dlo, v, row, zs, sc,
                                                       lane, owner, mq);
            q_to_row<N, false>(v, row);
            dfx_group<N, ZF>(dlo, dhi + 1, c, row_at, owner, mq);
            row_to_q<N>(v, row);
            ws_sections<N, false, ZF, kPrecAL, true>(p, c, cf0, dhi + 1, K, v, row, zs,
                                                       sc, lane, owner, mq);
        } else {
            ws_sections<N, FACT, ZF, PREC, false>(p, c, cf0, 0, K, v, row, zs, sc, lane, owner,
                                                  mq);
        }
        q_to_row<N, FACT>(v, row, FACT ? sc[K - 1].misc.y : 1.f);
    }
}

// Coalesced stores of samples [lo, hi) of the group in `slot`, whose first
// sample is number `at` of the packed output and whose mirror image (p.rev:
// the zero-phase filter's passes write time-reversed, where a pass for the
// reversal took 27 us for 64 channels of 100,003 beside a filtering kernel of
// 32) is number `rat`.
template <int N>
__device__ __forceinline__ void ws_store(const Params& p, const float* slot, int lane, int lo,
                                         int hi, int64_t at, int64_t rat) {
    using SL = SlotLayout<N>;
    using WC = WsCfg<N>;
    if (p.rev) {
        float* dst = p.y + rat;  // sample j goes to dst[-j]
        if (((lo | hi) & 3) == 0 && (reinterpret_cast<uintptr_t>(dst - 3) & 15u) == 0) {
            for (int i = (lo >> 2) + lane; i < (hi >> 2); i += 32) {
                const float4 t = *reinterpret_cast<const float4*>(slot + SL::gran(i));
                __stcs(reinterpret_cast<float4*>(dst - 4 * i - 3), make_float4(t.w, t.z, t.y, t.x));
            }
        } else {
            for (int j = lo + lane; j < hi; j += 32) __stcs(dst - j, slot[SL::elem(j)]);
        }
    } else {
        float* dst = p.y + at;
        const bool aligned = (reinterpret_cast<uintptr_t>(dst) & 15u) == 0;
        if (lo == 0 && hi == WC::kGroup && aligned) {
            float4* d4 = reinterpret_cast<float4*>(dst);
#pragma unroll
            for (int i = 0; i < WC::kGran / 32; ++i)
                __stcs(d4 + i * 32 + lane,
                       *reinterpret_cast<const float4*>(slot + SL::gran(i * 32 + lane)));
        } else if (((lo | hi) & 3) == 0 && aligned) {
            float4* d4 = reinterpret_cast<float4*>(dst);
            for (int i = (lo >> 2) + lane; i < (hi >> 2); i += 32)
                __stcs(d4 + i, *reinterpret_cast<const float4*>(slot + SL::gran(i)));
        } else {
            for (int j = lo + lane; j < hi; j += 32) __stcs(dst + j, slot[SL::elem(j)]);
        }
    }
    __syncwarp();
}

// Group g of a segment: prefetch the next group, filter this one (ws_filter),
// store the segment's own outputs.  base: the warp's two group slots, `cur`
// holding this group.
template <int N, bool FACT, bool CR, bool ZF, int PREC>
__device__ __forceinline__ void ws_group(const Params& p, const volatile WsSeg& sg, int base,
                                         int lane, int cur, int g) {
    using SL = SlotLayout<N>;
    using WC = WsCfg<N>;
    float* slots = ws_slots(base);
    // prefetch: the segment's next group, or the next segment's first
    float* nxt = slots + (cur ^ 1) * WC::kSlot;
    if (g + 1 < sg.ngroups) {
        ws_load<N>(p.x + sg.base + (int64_t)(g + 1) * WC::kGroup, sg.rem - (g + 1) * WC::kGroup,
                   nxt, lane);
        cp_async_wait1();
    } else if (sg.nbase >= 0) {
        ws_load<N>(p.x + sg.nbase, sg.nrem, nxt, lane);
        cp_async_wait1();
    } else {
        asm volatile("cp.async.wait_all;" ::: "memory");
    }
    __syncwarp();
    float* slot = slots + cur * WC::kSlot;
    ws_filter<N, FACT, CR, ZF, PREC>(base + cur * WC::kSlot + lane * SL::kRow, sg.c, sg.K,
                                     ZF ? (sg.zrel % WC::kGroup) / N : 0, ZF ? sg.zrel % N : 0);
    __syncwarp();
    const int a = sg.a - g * WC::kGroup, b = sg.b - g * WC::kGroup;
    ws_store<N>(p, slot, lane, a > 0 ? a : 0, b < WC::kGroup ? b : WC::kGroup,
                sg.base + (int64_t)g * WC::kGroup, sg.rbase - (int64_t)g * WC::kGroup);
}

// All groups of one segment through all K sections (one warp).  On return
// sg.cur is the slot of the next segment's first group (in flight where
// sg.nbase >= 0).
template <int N, bool FACT, bool CR, int PREC>
__device__ __forceinline__ void ws_segment(const Params& p, volatile WsSeg& sg, int base,
                                           int lane) {
    float4* zs = s_ws.z[ws_warp()];
    // the state entering the segment (zs[k], the same in every lane): zi
    // (scaled by 1/G_k when b0 is factored) on the channel's first segment,
    // zero state after a warm-up
    __syncwarp();
    if (!CR) {
        const int64_t at = (int64_t)sg.c * p.kmax;
        ws_stage(p.c32 + at, PREC == kPrecDF && p.N != N ? p.cdf + at : nullptr, sg.K,
                 s_ws.cf[ws_warp()], lane);
    }
    if (lane < sg.K) {
        const int c = sg.c;
        float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        if (sg.first && p.zi) {
            const float gi = FACT ? __ldg(&p.c32[(int64_t)c * p.kmax + lane].misc.z) : 1.f;
            z.x = __ldg(p.zi + ((int64_t)c * p.kmax + lane) * p.zstep + 0) * gi;
            z.z = __ldg(p.zi + ((int64_t)c * p.kmax + lane) * p.zstep + 1) * gi;
        }
        zs[lane] = z;
    }
    __syncwarp();
    // the channel's last sample is in the segment's last group when the
    // segment ends the channel: that group takes the zf path
    int g = 0, cur = sg.cur;
#pragma unroll 1
    for (; g < sg.ngroups - (sg.zrel >= 0 ? 1 : 0); ++g, cur ^= 1)
        ws_group<N, FACT, CR, false, PREC>(p, sg, base, lane, cur, g);
    if (sg.zrel >= 0) {
        ws_group<N, FACT, CR, true, PREC>(p, sg, base, lane, cur, g);
        cur ^= 1;
    }
    if (lane == 0) sg.cur = cur;
    __syncwarp();
}

// A segment of a channel of precision class 3; its first group is in slot 0
// and no other segment's is to be prefetched.  N: the channel's samples per
// lane.
template <int N>
__device__ __forceinline__ void ws_segment_df(const Params& p, int base, int lane) {
    volatile WsSeg& sg = s_ws.seg[ws_warp()];
    if (lane == 0) {
        sg.nbase = -1;
        sg.cur = 0;
    }
    __syncwarp();
    ws_segment<N, false, false, kPrecDF>(p, sg, base, lane);
}

// A segment's shared-memory record (lane 0 writes).
__device__ __forceinline__ void ws_set(const Params& p, volatile WsSeg& ws, const SegGeom& sg,
                                       int lane) {
    if (lane == 0) {
        ws.base = sg.off + sg.cstart;
        ws.rbase = sg.off + sg.len - 1 - sg.cstart;
        ws.rem = ws_cap(sg.len - sg.cstart);
        ws.a = (int)(sg.out_lo - sg.cstart);
        ws.b = (int)(sg.out_hi - sg.cstart);
        ws.c = sg.c;
        ws.K = sg.K;
        ws.ngroups = sg.ngroups;
        ws.zrel = p.zf && sg.out_hi == sg.len ? (int)(sg.len - 1 - sg.cstart) : -1;
        ws.first = sg.cstart == 0;
    }
    __syncwarp();
}

// One segment of a channel of precision class 0 to 2, in the instantiation it
// needs (identity, cyclic reduction, FP32 PH with or without coefficient low
// parts).
template <int N, bool CRK>
__device__ __forceinline__ void ws_run_segment(const Params& p, int base, int lane) {
    volatile WsSeg& sg = s_ws.seg[ws_warp()];
    float* slots = ws_slots(base);
    const int K = sg.K, c = sg.c;
    if (K == 0) {
        // identity channel: copy the segment's own samples (nothing of it is
        // in the slots, but the next segment's first group is due)
        for (int i = sg.a + lane; i < sg.b; i += 32)
            p.y[p.rev ? sg.rbase - i : sg.base + i] = __ldg(p.x + sg.base + i);
        const int nxt = sg.cur ^ 1;
        __syncwarp();
        if (sg.nbase >= 0)
            ws_load<N>(p.x + sg.nbase, sg.nrem, slots + nxt * WsCfg<N>::kSlot, lane);
        if (lane == 0) sg.cur = nxt;
        __syncwarp();
        return;
    }
    const ChanInfo& ci = p.chan[c];
    const bool fact = ci.mode != 0;
    const int ext = ci.ext;
    // cyclic reduction when the call asks for it and every section of the
    // channel is well conditioned for it (FP32 channels only), PH otherwise
    bool cr = CRK && ext == 0;
    for (int k = 0; k < K && cr; ++k)
        cr = __ldg(&p.c32[(int64_t)c * p.kmax + k].cr_misc.w) != 0.f;
    if (CRK && cr) {
        if (fact) ws_segment<N, true, CRK, kPrecF32>(p, sg, base, lane);
        else ws_segment<N, false, CRK, kPrecF32>(p, sg, base, lane);
    } else if (ext) {
        if (fact) ws_segment<N, true, false, kPrecAL>(p, sg, base, lane);
        else ws_segment<N, false, false, kPrecAL>(p, sg, base, lane);
    } else {
        if (fact) ws_segment<N, true, false, kPrecF32>(p, sg, base, lane);
        else ws_segment<N, false, false, kPrecF32>(p, sg, base, lane);
    }
}

// ---- long-memory channels (long_section.cuh) ----

__device__ __forceinline__ void team_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Sections [k0, k1) of a long-memory channel over the group in `hi` (and, in
// the double-float range, `lo`: the low parts), lane rows of N samples; the
// last stage multiplies the split-off gain in.  ZF: the group holds the
// channel's last sample (element mq of lane owner's chunk).
template <int N, bool ZF>
__device__ __forceinline__ void long_stage(const Params& p, const ChanInfo& ci, int c, int k0,
                                           int k1, bool last, float* hi, float* lo, float4* zs,
                                           int lane, int owner, int mq) {
    constexpr int R = SlotLayout<N>::kRow;
    const Coef32* cf0 = p.c32 + (int64_t)c * p.kmax;
    float* row = hi + lane * R;
    float* lrow = lo + lane * R;
    const bool df3 = ci.ext >= 3, fact = !df3 && ci.mode != 0;
    const int dlo = df3 ? ci.dflo : 8, dhi = df3 ? ci.dfhi : -1;
    float v[N];
    row_to_chunk<N>(v, row);
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
        const Coef32* cf = cf0 + k;
        const LongCoef* lc =
            reinterpret_cast<const LongCoef*>(p.cdf + (int64_t)c * p.kmax + k);
        float* zf_dst = ZF ? p.zf + ((int64_t)c * p.kmax + k) * 2 : nullptr;
        const float4 zz = zs[k];
        const float4 lp = cf->lane_pow[lane];
        float4 zo;
        if (k >= dlo && k <= dhi) {
            if (k == dlo) {
                // the range's input is FP32: its low parts start at zero
#pragma unroll
                for (int b = 0; b < N / 4; ++b)
                    reinterpret_cast<float4*>(lrow)[b] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            df z1{zz.x, zz.y}, z2{zz.z, zz.w};
            long_section_dfx<N, ZF>(v, lrow, load_secdf(cf), cf->phi_pow, lc->phi_lo, lp,
                                    lc->lane_lo[lane], z1, z2, lane == owner, mq, zf_dst);
            zo = make_float4(z1.hi, z1.lo, z2.hi, z2.lo);
            if (k == dhi) {
                // the range's output, rounded once
#pragma unroll
                for (int b = 0; b < N / 4; ++b) {
                    const float4 l = reinterpret_cast<const float4*>(lrow)[b];
                    v[4 * b + 0] += l.x;
                    v[4 * b + 1] += l.y;
                    v[4 * b + 2] += l.z;
                    v[4 * b + 3] += l.w;
                }
            }
        } else {
            float4 ab = cf->ab;
            float b0 = fact ? 1.f : cf->misc.x;
            if (df3) {
                const float4 br = cf->braw;
                ab.z = br.y;
                ab.w = br.z;
                b0 = br.x;
            }
            const float G = ZF && fact ? cf->misc.y : 1.f, lvl = cf->misc.w;
            const float4 al = cf->alo;
            const float2 alo = make_float2(al.x, al.y);
            const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
            float z1 = zz.x, z2 = zz.z;
            if (lvl > 1.5f)
                long_section<N, ZF, true, true>(v, ab, b0, cf->phi_pow, lp, z1, z2, lane == owner,
                                                mq, row, zf_dst, G, alo, lc->phi_lo,
                                                lc->lane_lo[lane]);
            else if (lvl > 0.5f)
                long_section<N, ZF, true, false>(v, ab, b0, cf->phi_pow, lp, z1, z2, lane == owner,
                                                 mq, row, zf_dst, G, alo, nullptr, none);
            else
                long_section<N, ZF, false, false>(v, ab, b0, cf->phi_pow, lp, z1, z2,
                                                  lane == owner, mq, row, zf_dst, G, alo, nullptr,
                                                  none);
            zo = make_float4(z1, 0.f, z2, 0.f);
        }
        __syncwarp();
        if (lane == 0) zs[k] = zo;
    }
    if (last && fact) {
        const float Gk = cf0[ci.K - 1].misc.y;
#pragma unroll
        for (int m = 0; m < N; ++m) v[m] *= Gk;
    }
    chunk_to_row<N>(v, row);
    __syncwarp();
}

// The segments of the long-memory channels.  A segment is a sequential walk of
// up to a thousand groups, most of it latency of dependent steps, and such a
// channel has few segments, so a team of q warps (q = 1, 2 or 4 for up to 2, 4
// and 8 sections) shares one: stage w of the team runs its share of the
// sections on group s - w while the stages before it run theirs on the groups
// after it, one team barrier per step; every section sees the same groups in
// the same order as if one warp ran them all (64 channels of 2^22 samples, K =
// 8: 20.7 ms, 34.2 with a warp per segment; 9 channels of 300,007, K = 3, the
// same digits).  The shares are cut by cost (double-float 6, double-float scan 2).
// N: samples per lane.
template <int N>
__device__ __forceinline__ void ws_long_phase(const Params& p, int lane) {
    constexpr int G = 32 * N, kSlot = 32 * SlotLayout<N>::kRow;
    const int64_t total = p.hdr->long_segs;
    if (total <= 0) return;
    const int q = p.hdr->long_team;
    const int w = ws_warp(), team = w / q, stage = w % q;
    // the team's 3 q slots: groups in flight, then their low parts
    const int nh = q == 1 ? 2 : q == 2 ? 3 : 6, nl = 3 * q - nh;
    float* slots = ws_slots(team * 3 * q * kSlot);
    float4* zs = s_ws.z[team];
    const int bar = 1 + team, threads = 32 * q;
    for (;;) {
        if (stage == 0 && lane == 0)
            s_ws.item[team] = (int64_t)atomicAdd(&p.hdr->long_next, 1ull);
        team_sync(bar, threads);
        const int64_t item = s_ws.item[team];
        if (item >= total) break;
        const SegGeom sg = seg_geom<G>(p, item);
        const ChanInfo ci = p.chan[sg.c];
        const int K = sg.K, ng = sg.ngroups;
        const Coef32* cf0 = p.c32 + (int64_t)sg.c * p.kmax;
        // this stage's sections
        int k0 = 0, k1 = 0;
        {
            auto cost = [&](int k) {
                return ci.ext >= 3 && k >= ci.dflo && k <= ci.dfhi ? 6
                                                                   : (cf0[k].misc.w > 1.5f ? 2 : 1);
            };
            int sum = 0, acc = 0;
            for (int k = 0; k < K; ++k) sum += cost(k);
            for (int k = 0; k < K; ++k) {
                // section k goes to the stage its middle falls into
                const int ck = cost(k), st = (2 * acc + ck) * q / (2 * sum);
                acc += ck;
                if (st < stage) k0 = k + 1;
                if (st <= stage) k1 = k + 1;
            }
        }
        const float* src = p.x + sg.off + sg.cstart;
        const int rem = ws_cap(sg.len - sg.cstart);
        const int zrel =
            p.zf && sg.out_hi == sg.len ? (int)(sg.len - 1 - sg.cstart) : -1;
        if (stage == 0) {
            if (lane < K) {
                float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                if (sg.cstart == 0 && p.zi) {
                    const float gi = ci.mode != 0 && ci.ext < 3 ? cf0[lane].misc.z : 1.f;
                    z.x = p.zi[((int64_t)sg.c * p.kmax + lane) * p.zstep + 0] * gi;
                    z.z = p.zi[((int64_t)sg.c * p.kmax + lane) * p.zstep + 1] * gi;
                }
                zs[lane] = z;
            }
            ws_load<N>(src, rem, slots, lane);
        }
        team_sync(bar, threads);
#pragma unroll 1
        for (int s = 0; s < ng + q - 1; ++s) {
            const int g = s - stage;
            if (stage == 0 && s < ng) {
                if (s + 1 < ng) {
                    ws_load<N>(src + (int64_t)(s + 1) * G, rem - (s + 1) * G,
                               slots + (s + 1) % nh * kSlot, lane);
                    cp_async_wait1();
                } else {
                    asm volatile("cp.async.wait_all;" ::: "memory");
                }
                __syncwarp();
            }
            if (g >= 0 && g < ng) {
                float* hi = slots + g % nh * kSlot;
                float* lo = slots + (nh + g % nl) * kSlot;
                const bool last = stage == q - 1;
                if (k0 < k1 || last) {
                    if (zrel >= 0 && g == ng - 1)
                        long_stage<N, true>(p, ci, sg.c, k0, k1, last, hi, lo, zs, lane,
                                            zrel % G / N, zrel % N);
                    else
                        long_stage<N, false>(p, ci, sg.c, k0, k1, last, hi, lo, zs, lane, 0, 0);
                }
                if (last) {
                    const int64_t at = sg.off + sg.cstart + (int64_t)g * G;
                    const int64_t a = sg.out_lo - sg.cstart - (int64_t)g * G;
                    const int64_t b = sg.out_hi - sg.cstart - (int64_t)g * G;
                    ws_store<N>(p, hi, lane, (int)(a > 0 ? a : 0), (int)(b < G ? b : G), at,
                                2 * sg.off + sg.len - 1 - at);
                }
            }
            team_sync(bar, threads);
        }
    }
    // the last team to finish resets the hand-out for the next launch
    if (stage == 0 && lane == 0) {
        __threadfence();
        const unsigned prev = atomicAdd(&p.hdr->long_done, 1u);
        if (prev + 1 == gridDim.x * (kWsWarps / q)) {
            p.hdr->long_next = 0;
            p.hdr->long_done = 0;
            __threadfence();
        }
    }
    __syncthreads();  // the slots go to the warps again
}

// The call's parameters to shared memory (whole CTA).
__device__ __forceinline__ void ws_params(const Params& pc) {
    static_assert(sizeof(Params) % 8 == 0 && sizeof(Params) / 8 <= kWsThreads, "one word per thread");
    if (threadIdx.x < sizeof(Params) / 8)
        reinterpret_cast<unsigned long long*>(&s_ws.p)[threadIdx.x] =
            reinterpret_cast<const unsigned long long*>(&pc)[threadIdx.x];
    __syncthreads();
}

// CRK: the cyclic-reduction instantiation (algo 2).  The PH one carries no
// cyclic-reduction code, so its register allocation does not pay for it.
template <int N, bool CRK>
__global__ void __launch_bounds__(kWsThreads, ws_ctas_per_sm<N>())
    sos_warpseg_kernel(const __grid_constant__ Params pc) {
    using WC = WsCfg<N>;
    // the look-back kernel queued behind this one may be launched now (it
    // waits for this kernel's completion before it starts work)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // launched early behind the plan kernel: wait for its completion (and
    // its writes) before the first read of the plan's tables
    asm volatile("griddepcontrol.wait;" ::: "memory");
    ws_params(pc);
    const Params& p = s_ws.p;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int base = ws_slot_base<N>();
    float* slots = ws_slots(base);
    volatile WsSeg& ws = s_ws.seg[w];
    ws_long_phase<ext_n(N)>(p, lane);
    const int64_t skip = p.hdr->long_segs;
    const int64_t total = p.hdr->total_pipe - skip;  // the other segments of the latest plan
    // segments: the first gridDim.x kWsWarps one per warp, the rest handed out
    // in order as warps come free (segments differ in length across uneven
    // channels).  The first round goes across the CTAs, and so the SMs, before
    // it goes into them, starting at another warp in each CTA of an SM (CTA i
    // and i + grid/3 usually share one), so that few segments, or the first and
    // costly ones, spread over all schedulers
    const unsigned per = (gridDim.x + ws_ctas_per_sm<N>() - 1) / ws_ctas_per_sm<N>();
    int64_t d = (int64_t)((w + blockIdx.x / per) % kWsWarps) * gridDim.x + blockIdx.x;
    if (lane == 0) ws.total = total;
    // the next segment of the hand-out (none when the first round had them all)
    auto next = [&]() -> int64_t {
        const int64_t nw = (int64_t)gridDim.x * kWsWarps, end = ws.total;
        if (end <= nw) return end;
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(&p.hdr->seg_next, 1ull);
        return nw + (int64_t)__shfl_sync(0xffffffffu, t, 0);
    };
    // ---- the segments of precision class 3, which come first ----
    constexpr int NX = ext_n(N);
#pragma unroll 1
    while (d < p.hdr->ext_segs - skip) {
        const SegGeom sg = seg_geom<WsCfg<NX>::kGroup>(p, skip + d);
        ws_load<NX>(p.x + sg.off + sg.cstart, sg.len - sg.cstart, slots, lane);
        ws_set(p, ws, sg, lane);
        ws_segment_df<NX>(p, base, lane);
        d = next();
    }
    // ---- the others ----
    if (d < total) {
        {
            const SegGeom sg = seg_geom<WC::kGroup>(p, skip + d);
            // the first group is on its way while the next segment is looked up
            if (sg.K > 0) ws_load<N>(p.x + sg.off + sg.cstart, sg.len - sg.cstart, slots, lane);
            if (lane == 0) ws.cur = 0;
            ws_set(p, ws, sg, lane);
        }
#pragma unroll 1
        for (;;) {
            // the warp's next segment, taken one ahead for the prefetch of its
            // first group (its geometry is looked up again)
            {
                const int64_t dn = next();
                SegGeom nx;
                nx.K = 0;
                if (dn < ws.total) nx = seg_geom<WC::kGroup>(p, skip + dn);
                if (lane == 0) {
                    ws.next = dn;
                    ws.nbase = nx.K > 0 ? nx.off + nx.cstart : -1;
                    ws.nrem = nx.K > 0 ? ws_cap(nx.len - nx.cstart) : 0;
                }
                __syncwarp();
            }
            ws_run_segment<N, CRK>(p, base, lane);
            const int64_t dn = ws.next;
            if (dn >= ws.total) break;
            const SegGeom sg = seg_geom<WC::kGroup>(p, skip + dn);
            __syncwarp();
            ws_set(p, ws, sg, lane);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    // the last warp to finish resets the hand-out for the next launch (every
    // warp's last atomicAdd on seg_next precedes its arrival here)
    const int64_t nw = (int64_t)gridDim.x * kWsWarps;
    if (lane == 0 && ws.total > nw) {
        __threadfence();
        const unsigned prev = atomicAdd(&p.hdr->seg_done, 1u);
        if (prev + 1 == (unsigned)nw) {
            p.hdr->seg_next = 0;
            p.hdr->seg_done = 0;
            __threadfence();
        }
    }
}

// Low-latency streaming: the next block of `chunk` samples of every channel
// (x, y: [C][chunk]) through all K sections, from the state `p.zi` into the
// state `p.zf`, in one launch with the coefficient tables of an earlier
// sos_prepare.  Warp w takes segment w % maxseg of channel w / maxseg: a
// channel within its memory horizon is cut into segments of
// max(seg_len, its shortest allowed segment) samples, each warmed up over the
// horizon from zero state (the first from the incoming state), so that a
// long block is not one warp's sequential walk; other channels are one
// segment.  No plan launch, no hand-out counter, no waits on other warps.
// The paper's real-time scenario: a signal arriving in blocks, the state
// carried from one block to the next (Sec. V's group chaining across calls).
template <int N>
__global__ void __launch_bounds__(kWsThreads, ws_ctas_per_sm<N>())
    sos_stream_kernel(const __grid_constant__ Params pc, int64_t chunk, int64_t seg_len,
                      int32_t maxseg, int32_t foreign) {
    using WC = WsCfg<N>;
    ws_params(pc);
    const Params& p = s_ws.p;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t gw = (int64_t)blockIdx.x * kWsWarps + w;
    const int c = (int)(gw / maxseg);
    const int si = (int)(gw % maxseg);
    if (c >= p.C || chunk <= 0) return;
    const ChanInfo ci = p.chan[c];
    int64_t seg = chunk;
    if (ci.horizon >= 0 && ci.K > 0) {
        // the incoming state of a stream is what earlier samples of the same
        // signal left, so its response is part of the impulse-response tail
        // the horizon bounds; a foreign initial state also has to die out
        const int64_t least = foreign ? ci.minseg_z : ci.minseg;
        seg = seg_len > least ? seg_len : least;
        if (seg > chunk) seg = chunk;
    }
    const int nseg = (int)((chunk + seg - 1) / seg);
    if (si >= nseg) return;
    // the channel's coefficient tables into L1 now, all sections at once
    // (each is otherwise a round trip to L2 at the section's first use, one
    // after another: most of a short block's latency)
    {
        const char* cb = reinterpret_cast<const char*>(p.c32 + (int64_t)c * p.kmax);
        const int lines = (int)((sizeof(Coef32) * (size_t)ci.K + 127) / 128);
        for (int i = lane; i < lines; i += 32)
            asm volatile("prefetch.global.L1 [%0];" ::"l"(cb + 128 * (size_t)i));
    }
    // state rows past K (or a channel without sections) pass through
    if (si == 0 && p.zf)
        for (int i = ci.K * 2 + lane; i < p.kmax * 2; i += 32)
            p.zf[(int64_t)c * p.kmax * 2 + i] = p.zi ? p.zi[(int64_t)c * p.kmax * 2 + i] : 0.f;
    const int base = ws_slot_base<N>();
    float* slots = ws_slots(base);
    SegGeom sg;
    sg.c = c;
    sg.si = si;
    sg.off = (int64_t)c * chunk;
    sg.len = chunk;
    sg.out_lo = (int64_t)si * seg;
    sg.out_hi = sg.out_lo + seg < chunk ? sg.out_lo + seg : chunk;
    sg.cstart = si == 0 ? 0 : sg.out_lo - ci.horizon;
    sg.horizon = ci.horizon;
    sg.K = ci.K;
    if (lane == 0) {
        s_ws.seg[w].nbase = -1;
        s_ws.seg[w].cur = 0;
    }
    auto set = [&](auto nn) {
        constexpr int M = decltype(nn)::value;
        sg.ngroups = (int)((sg.out_hi - sg.cstart + 32 * M - 1) / (32 * M));
        if (sg.K > 0) ws_load<M>(p.x + sg.off + sg.cstart, sg.len - sg.cstart, slots, lane);
        ws_set(p, s_ws.seg[w], sg, lane);
    };
    if (ci.ext < 3) {
        set(std::integral_constant<int, N>{});
        ws_run_segment<N, false>(p, base, lane);
    } else {
        set(std::integral_constant<int, ext_n(N)>{});
        ws_segment_df<ext_n(N)>(p, base, lane);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

}  // namespace sosf
