// The nonlocal (Kleinman-Bylander) part of the fused Chebyshev step on one unit of consecutive grid
// points held in shared memory (an xy plane, a group of x rows, or a CTA's rows of a cluster plane):
// the projections staged per slot, the apply colour by colour, and the per-slot partial projections
// of the step's output.  Unit point o (0 <= o < rows * N) is at sm[unit_pos(o)], by default
// sm[(o / N) * P + (o % N)].
// The tables are those of KBDev (slots, colours and entries per unit).
#pragma once
#include "fft_smem.cuh"
#include "grid_common.cuh"
#include "sgw_internal.cuh"

namespace sgw {

constexpr int KB_B = 3;    // KB entries per lane whose loads are in flight together, in units of a plane or many rows

// Position in shared memory of unit point o = y N + x (row y, column x) at row pitch P.  LAYOUT 0:
// natural, y P + x.  LAYOUT 1 (N = 288, the two-stage row transforms): a row is 16 groups of 19
// slots, column x at 19 (x mod 16) + x div 16, the order in which the 16 x 18 transforms leave it.
// LAYOUT 2: the tables hold the positions themselves.
template <int N, int P, int LAYOUT>
__device__ __forceinline__ int unit_pos_yx(int y, int x) {
    if constexpr (LAYOUT == 1) {
        static_assert(N == 288 && P >= 304, "layout 1 is the 288-point row in 16 groups of 19");
        return y * P + 19 * (x & 15) + (x >> 4);
    } else {
        return y * P + x;
    }
}
template <int N, int P, int LAYOUT>
__device__ __forceinline__ int unit_pos(int o) {
    if constexpr (LAYOUT == 2) return o;
    else return unit_pos_yx<N, P, LAYOUT>(o / N, o % N);
}

// kbc[b][k][p] = E_ap dV sum_{slots of a} kbp[b][slot][p] for every slot k of atom a, by one warp: lane l
// takes projector p = l % 4 of the atom's slots l / 4, l / 4 + 8, ... (in increasing unit), then the
// eight lanes of each p are summed by a fixed shuffle tree.  The result is stored once per slot, so
// that a unit's coefficients are one contiguous run (through the slot's atom they would be two more
// dependent loads away).  The whole warp calls it with one (a, b); a >= n_atoms does nothing.
__device__ __forceinline__ void kb_reduce_warp(const KbReduceArgs& kr, int a, int b, int lane) {
    if (a >= kr.n_atoms) return;
    const int p = lane & 3;
    const int q0 = __ldg(kr.atom_pos_off + a), q1 = __ldg(kr.atom_pos_off + a + 1);
    const float2* kb = kr.kbp + (size_t)b * kr.total_slots * 4;
    float2 acc = make_float2(0.f, 0.f);
    for (int q = q0 + (lane >> 2); q < q1; q += 8) {
        const float2 v = ld2_written(kb + (size_t)__ldg(kr.atom_pos + q) * 4 + p);
        acc.x += v.x;
        acc.y += v.y;
    }
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
    }
    const float4 e = __ldg(kr.atom_e + a);
    const float ep = (p == 0 ? e.x : (p == 1 ? e.y : (p == 2 ? e.z : e.w))) * kr.dV;
    const float2 r = make_float2(ep * acc.x, ep * acc.y);
    float2* kc = kr.kbc + (size_t)b * kr.total_slots * 4;
    for (int q = q0 + (lane >> 2); q < q1; q += 8) kc[(size_t)__ldg(kr.atom_pos + q) * 4 + p] = r;
}

// What a block needs to know of its unit before it can load anything else: the unit's slots s0 .. s1
// and the bounds of its colours, lane c of every warp holding the begin of colour c and `end` the
// end of the last (at most 32 colours).  Loaded together, first of all.
struct KbHead {
    int s0 = 0, s1 = 0, col = 0, end = 0;
    // begin of colour c (c <= max_colors); the whole warp calls it with one c
    __device__ __forceinline__ int begin(int c, int max_colors) const {
        const int v = __shfl_sync(0xffffffffu, col, c & 31);
        return c >= max_colors ? end : v;
    }
};
__device__ __forceinline__ KbHead kb_head(const StepArgs& a, int u) {
    KbHead h;
    const int lane = threadIdx.x & 31;
    const int* col = a.kbe_col + (size_t)u * (a.max_colors + 1);
    h.s0 = __ldg(a.plane_off + u);
    h.s1 = __ldg(a.plane_off + u + 1);
    h.end = __ldg(col + a.max_colors);
    h.col = __ldg(col + min(lane, a.max_colors));
    return h;
}

// E-weighted projector coefficients of the unit's slots into shared memory: kcs[4 s + p] for the
// unit's s-th slot and projector p (kc: the vector's coefficients, [slot][4]).
template <int NT>
__device__ __forceinline__ void kb_stage_coeffs(const KbHead& h, const float2* kc, float2* kcs) {
    const float2* src = kc + (size_t)4 * h.s0;
    for (int i = threadIdx.x; i < 2 * (h.s1 - h.s0); i += NT) reinterpret_cast<float4*>(kcs)[i] = ld4_written(src + 2 * i);
}

// B entries of a lane (at eb, eb + stride, ...; past e1 the last one again, to be skipped by the
// reader), all their loads in flight at once.
template <int B>
struct KbBatch {
    unsigned os[B];
    float4 be[B];
    __device__ __forceinline__ void load(const StepArgs& a, int eb, int stride, int e1) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int e = min(eb + i * stride, e1 - 1);
            os[i] = __ldg(a.kbe_os + e);
            be[i] = __ldg(a.kbe_beta + e);
        }
    }
};

// sm += sum_ap beta_ap E_ap <beta_ap|b1> over the unit, colour by colour (slots of one colour touch
// disjoint points, so each point is updated by one thread at a time; no atomics, fixed order).
// The entries' loads run one batch ahead, over the ends of the colours and past the barriers: the
// tables come from L2, and a batch's latency would otherwise be paid once per colour and remainder.
// (Two and three batches ahead, or larger ones, cost more registers than the latency they hid.)
// meanwhile() runs after the first loads are on their way; a barrier before the first update of sm
// makes its stores (and the caller's) visible; returns after a barrier.
template <int N, int P, int NT, int LAYOUT = 0, int B = KB_B, class F>
__device__ __forceinline__ void kb_apply_unit(const StepArgs& a, const KbHead& h, const float2* kcs, float2* sm,
                                              F&& meanwhile) {
    int c = 1, e0 = h.begin(0, a.max_colors), e1 = h.begin(1, a.max_colors);   // e0 .. e1 the rest of colour c - 1
    KbBatch<B> cur;
    if (e0 < e1) cur.load(a, e0 + threadIdx.x, NT, e1);
    meanwhile();
    __syncthreads();
    while (e0 < e1) {                     // a unit's colours are used from 0 upwards
        KbBatch<B> nxt;
        const int en = e0 + B * NT;
        const bool last = en >= e1;
        const int e2 = h.begin(c + 1, a.max_colors);
        if (!last) nxt.load(a, en + threadIdx.x, NT, e1);
        else if (e1 < e2) nxt.load(a, e1 + threadIdx.x, NT, e2);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if (e0 + (int)threadIdx.x + i * NT >= e1) break;
            const float4 be = cur.be[i];
            const int o = (int)(cur.os[i] & 0xffffu), sl = (int)(cur.os[i] >> 16);
            const float4 c01 = *reinterpret_cast<const float4*>(kcs + 4 * sl);
            const float4 c23 = *reinterpret_cast<const float4*>(kcs + 4 * sl + 2);
            float2& hv = sm[unit_pos<N, P, LAYOUT>(o)];
            hv.x += be.x * c01.x + be.y * c01.z + be.z * c23.x + be.w * c23.z;
            hv.y += be.x * c01.y + be.y * c01.w + be.z * c23.y + be.w * c23.w;
        }
        cur = nxt;
        if (!last) {
            e0 = en;
        } else {
            e0 = e1;
            e1 = e2;
            ++c;
            __syncthreads();
        }
    }
}

// Partial projections of the unit's values in sm (positions by unit_pos): kbp[b][slot][p] = sum over the
// slot's points of beta_ap(r) sm(r); one warp per slot, lanes strided over the points, fixed-order warp
// reduction.  The loads run one batch ahead here too, over the ends of the slots; kb_project_begin
// finds the warp's first two slots and can be called long before.
struct KbSlots {
    int k = 0, e0 = 0, e1 = 0, f0 = 0, f1 = 0;      // slot k's entries e0 .. e1, the warp's next slot's f0 .. f1
};
template <int NT>
__device__ __forceinline__ KbSlots kb_project_begin(const StepArgs& a, const KbHead& h) {
    constexpr int NW = NT / 32;
    KbSlots s;
    s.k = h.s0 + (threadIdx.x >> 5);
    if (s.k < h.s1) {
        s.e0 = __ldg(a.kbe_slot_beg + s.k);
        s.e1 = __ldg(a.kbe_slot_end + s.k);
        if (s.k + NW < h.s1) {
            s.f0 = __ldg(a.kbe_slot_beg + s.k + NW);
            s.f1 = __ldg(a.kbe_slot_end + s.k + NW);
        }
    }
    return s;
}
// Meets a barrier before it reads sm.
template <int N, int P, int NT, int LAYOUT = 0, int B = KB_B>
__device__ __forceinline__ void kb_project_unit(const StepArgs& a, const KbHead& h, const KbSlots& sl, int b, const float2* sm) {
    constexpr int NW = NT / 32;
    const int s1 = h.s1, lane = threadIdx.x & 31;
    int k = sl.k, e0 = sl.e0, e1 = sl.e1, f0 = sl.f0, f1 = sl.f1;
    KbBatch<B> cur;
    if (k < s1) cur.load(a, e0 + lane, 32, e1);
    __syncthreads();
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    while (k < s1) {                      // a slot has at least one entry
        KbBatch<B> nxt;
        const int en = e0 + B * 32;
        const bool last = en >= e1;
        if (!last) nxt.load(a, en + lane, 32, e1);
        else if (k + NW < s1) nxt.load(a, f0 + lane, 32, f1);
#pragma unroll
        for (int i = 0; i < B; ++i) {
            if (e0 + lane + 32 * i >= e1) break;
            const float2 v = sm[unit_pos<N, P, LAYOUT>((int)(cur.os[i] & 0xffffu))];
            const float4 be = cur.be[i];
            acc[0] += be.x * v.x; acc[1] += be.x * v.y;
            acc[2] += be.y * v.x; acc[3] += be.y * v.y;
            acc[4] += be.z * v.x; acc[5] += be.z * v.y;
            acc[6] += be.w * v.x; acc[7] += be.w * v.y;
        }
        cur = nxt;
        if (!last) {
            e0 = en;
            continue;
        }
        const float r = warp_reduce_scatter8(acc, lane);
        if ((lane & 3) == 0) reinterpret_cast<float*>(a.kbp + ((size_t)b * a.total_slots + k) * 4)[lane >> 2] = r;
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = 0.f;
        k += NW;
        e0 = f0;
        e1 = f1;
        if (k + NW < s1) {
            f0 = __ldg(a.kbe_slot_beg + k + NW);
            f1 = __ldg(a.kbe_slot_end + k + NW);
        }
    }
}

// The pointwise part of the fused step on ROWS x N unit points starting at global offset `off`
// (vector b's unit; sm holds H_kin b1 + V_NL b1 at pitch P): out = cpsi psi + ch alpha (h + (V - Ebar) b1
// [+ dv b1_partner]) + c2 b2, written to global memory and back into sm.  STREAM: b1, psi, b2 read and
// out written with evict-first caching.
template <int N, int ROWS, int P, int NT, int UNROLL = 2, int LAYOUT = 0, bool STREAM = false>
__device__ __forceinline__ void step_pointwise(const StepArgs& a, const VecInfo& inf, size_t off, size_t uoff,
                                               float2* sm) {
    constexpr size_t NG = (size_t)N * N * N;
    const float* V = a.vpot + (size_t)inf.vrow * NG + uoff;
    const float* dV = (a.dvpot != nullptr && inf.dvrow >= 0) ? a.dvpot + (size_t)inf.dvrow * NG + uoff : nullptr;
    const float2* bp = (dV != nullptr) ? a.b1 + (size_t)inf.partner * NG + uoff : nullptr;
    const float2 cpsi = a.coef.cpsi[inf.cset], ch = a.coef.ch[inf.cset], c2 = a.coef.c2[inf.cset];
    const float ebar = a.ebar, alpha = a.alpha;
#pragma unroll UNROLL
    for (int q = threadIdx.x; q < ROWS * N / 2; q += NT) {
        const int y = q / (N / 2), x = 2 * (q % (N / 2));
        const int o = y * N + x;
        // x is even: x + 1 sits one slot further (layout 0) or one group of 19 further (layout 1)
        const int sp = unit_pos_yx<N, P, LAYOUT>(y, x), sp1 = sp + (LAYOUT == 1 ? 19 : 1);
        float2 h0 = sm[sp], h1 = sm[sp1];
        const float4 bb = STREAM ? ldcs4(a.b1 + off + o) : ld4(a.b1 + off + o);
        const float2 v = __ldg(reinterpret_cast<const float2*>(V + o));
        h0.x += (v.x - ebar) * bb.x;
        h0.y += (v.x - ebar) * bb.y;
        h1.x += (v.y - ebar) * bb.z;
        h1.y += (v.y - ebar) * bb.w;
        if (dV != nullptr) {
            const float2 d = __ldg(reinterpret_cast<const float2*>(dV + o));
            const float4 pb = ld4(bp + o);            // the partner's b1: another vector's launch reads it too
            h0.x += d.x * pb.x;
            h0.y += d.x * pb.y;
            h1.x += d.y * pb.z;
            h1.y += d.y * pb.w;
        }
        float2 o0 = cmul(ch, cscale(h0, alpha)), o1 = cmul(ch, cscale(h1, alpha));
        if (a.psi != nullptr) {
            const float4 pp = STREAM ? ldcs4(a.psi + off + o) : ld4(a.psi + off + o);
            o0 = cadd(o0, cmul(cpsi, make_float2(pp.x, pp.y)));
            o1 = cadd(o1, cmul(cpsi, make_float2(pp.z, pp.w)));
        }
        if (a.b2 != nullptr) {
            const float4 b2 = STREAM ? ldcs4(a.b2 + off + o) : ld4(a.b2 + off + o);
            o0 = cadd(o0, cmul(c2, make_float2(b2.x, b2.y)));
            o1 = cadd(o1, cmul(c2, make_float2(b2.z, b2.w)));
        }
        if (STREAM)
            stcs4(a.out + off + o, o0, o1);
        else
            st4(a.out + off + o, o0, o1);
        sm[sp] = o0;
        sm[sp1] = o1;
    }
}

}  // namespace sgw
