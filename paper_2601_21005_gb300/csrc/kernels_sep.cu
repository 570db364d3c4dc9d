// The Chebyshev term with a separable kinetic energy.
//
// Without an energy cutoff T(k) = |k|^2 / 2 is a sum of one-dimensional symbols, so T psi is the sum
// of three line operations: along each axis a forward transform, times k_a^2 / 2, an inverse
// transform.  None of them needs another axis transformed, so a term reads and writes only
// real-space arrays and carries no transformed copy of its vector:
//   n <= 128:  z lines   W = T_z b                                          (16 B per vector-point)
//              planes    out = c psi + 2 H~ b - b2, H b = W + (T_x + T_y + V + V_NL) b     (40 B)
//   n = 288:   z lines   W = T_z b (16 B),  y lines  W += T_y b (24 B),  rows of x: the rest (40 B)
// against 64 B and 96 B when the vector's 3D transform is carried through the passes.  With a
// cutoff T is not separable: those contexts keep the transforms of the other grid kernels.
//
// Traffic bounds both passes at batches larger than L2; below that the planes' serial phases.  Every
// line is held in the registers of 2 or 4 lanes (reg_dft.cuh), so a transform takes no barrier; a
// plane's block meets one barrier per axis and per KB colour, where radix stages through shared
// memory take two per stage.  Measured per term of a degree-16 step with the KB parts of h = 0.5 clusters, the
// transform path -> this one: 64^3 x 64 240 -> 181 us (without KB 213 -> 148; the kernels by themselves, not
// overlapped: z lines 44 us, planes 148, 118 without KB), 64^3 x 8 40 -> 29 us, 96^3 x 8 218 -> 108 us, 128^3 x 12
// 594 -> 452 us, 48^3 x 64 213 -> 79 us, 32^3 x 64 38 -> 24 us, 288^3 x 16 (1963 KB atoms) 9.4 -> 6.6 ms.
#include <algorithm>

#include "dependent_launch.cuh"
#include "grid_common.cuh"
#include "kb_unit.cuh"
#include "reg_dft.cuh"
#include "sgw_internal.cuh"

namespace sgw {

// ------------------------------------------------------------------ shared pieces

__device__ __forceinline__ void sep_cp16(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
}

// The kernels of a term are launched by launch_dependent.  The z lines let the planes in at once: those load
// b and transform their rows and columns beside them, and wait only for the KB coefficients and W
// (per term, with the launches of a term in order, overlapped at their ends only, and so: 16^3 x 2 8.3, 3.9,
// 3.3 us; 32^3 x 12 16.5, 9.9, 8.5; 48^3 x 6 18.5, 12.8, 11.7; 64^3 x 8 36.1, 31.0, 29.2; 64^3 x 64 195, 188,
// 182).
// The plane pass lets the next term in after the pointwise part: at its start the z lines' blocks, which can
// do nothing yet, would take the places of planes.

// c m^2 for k = k1 + (N / T) i, m the signed frequency of k
template <int N, int T>
__device__ __forceinline__ float axis_factor(int k1, int i, float c) {
    const float m = (float)(k1 + (N / T) * i - (2 * i >= T ? N : 0));
    return c * m * m;
}

// The step's pointwise part on ROWS x N points of the unit at global offset `off` (unit points o = y N +
// x at sm[y PITCH + x], which holds H b but for W and the local potential):
//   out = cpsi psi + ch alpha (sm + W + (V - Ebar) b1 [+ dv b1_partner]) + c2 b2,
// to global memory and back into sm.  A thread takes U pairs of points at a time and loads all their
// operands before it uses one: absent ones are predicated off, since a branch around each would keep
// the loads of a group from being in flight together.  REAL: ch and c2 are real (every term but the
// last of a complex sum).
template <int N, int ROWS, int PITCH, int NT, int U, bool TAN, bool REAL>
__device__ __forceinline__ void sep_points(const StepArgs& a, const VecInfo& inf, size_t off, size_t uoff, float2* sm,
                                           const float2* bs) {
    static_assert(PITCH % 2 == 0, "rows start on 16 bytes");
    static_assert(ROWS * N / 2 % (U * NT) == 0, "whole groups");
    constexpr size_t NG = (size_t)N * N * N;
    const float* V = a.vpot + (size_t)inf.vrow * NG + uoff;
    const float* dV = TAN ? a.dvpot + (size_t)inf.dvrow * NG + uoff : nullptr;
    const float2* bp = TAN ? a.b1 + (size_t)inf.partner * NG + uoff : nullptr;
    const float2 cpsi = a.coef.cpsi[inf.cset], ch = cscale(a.coef.ch[inf.cset], a.alpha), c2 = a.coef.c2[inf.cset];
    const float ebar = a.ebar;
    const bool hp = a.psi != nullptr, hb = a.b2 != nullptr;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int q0 = threadIdx.x; q0 < ROWS * N / 2; q0 += U * NT) {
        float4 b1[U], w[U], ps[U], b2[U], pb[TAN ? U : 1];
        float2 v[U], d[TAN ? U : 1];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int o = 2 * (q0 + i * NT);              // pairs of points are contiguous over the unit's rows
            if (bs == nullptr) b1[i] = ld4(a.b1 + off + o);
            w[i] = ldcs4_written(a.W + off + o);
            ps[i] = hp ? ldcs4(a.psi + off + o) : zero;
            b2[i] = hb ? ldcs4(a.b2 + off + o) : zero;
            v[i] = __ldg(reinterpret_cast<const float2*>(V + o));
            if constexpr (TAN) {
                d[i] = __ldg(reinterpret_cast<const float2*>(dV + o));
                pb[i] = ld4(bp + o);
            }
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int q = q0 + i * NT, o = 2 * q;
            const int sp = (q / (N / 2)) * PITCH + 2 * (q % (N / 2));
            float4& sv = *reinterpret_cast<float4*>(sm + sp);
            if (bs != nullptr) b1[i] = *reinterpret_cast<const float4*>(bs + sp);
            float2 h[2] = {make_float2(sv.x + w[i].x, sv.y + w[i].y), make_float2(sv.z + w[i].z, sv.w + w[i].w)};
            const float2 bb[2] = {make_float2(b1[i].x, b1[i].y), make_float2(b1[i].z, b1[i].w)};
            const float2 pp[2] = {make_float2(ps[i].x, ps[i].y), make_float2(ps[i].z, ps[i].w)};
            const float2 b2v[2] = {make_float2(b2[i].x, b2[i].y), make_float2(b2[i].z, b2[i].w)};
            const float vv[2] = {v[i].x - ebar, v[i].y - ebar};
            float2 r[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                // the kinetic parts were summed first: (V - Ebar) b is the largest term, and this way one
                // rounding of its size is made, in the multiply-add
                h[j] = make_float2(fmaf(vv[j], bb[j].x, h[j].x), fmaf(vv[j], bb[j].y, h[j].y));
                if constexpr (TAN) {
                    const float dd = j == 0 ? d[i].x : d[i].y;
                    const float2 pbv = j == 0 ? make_float2(pb[i].x, pb[i].y) : make_float2(pb[i].z, pb[i].w);
                    h[j] = make_float2(fmaf(dd, pbv.x, h[j].x), fmaf(dd, pbv.y, h[j].y));
                }
                r[j] = REAL ? cscale(h[j], ch.x) : cmul(ch, h[j]);
                r[j] = cadd(r[j], cmul(cpsi, pp[j]));
                r[j] = REAL ? make_float2(fmaf(c2.x, b2v[j].x, r[j].x), fmaf(c2.x, b2v[j].y, r[j].y))
                            : cadd(r[j], cmul(c2, b2v[j]));
            }
            st4(a.out + off + o, r[0], r[1]);
            sv = make_float4(r[0].x, r[0].y, r[1].x, r[1].y);
        }
    }
}

template <int N, int ROWS, int PITCH, int NT, int U>
__device__ __forceinline__ void sep_pointwise(const StepArgs& a, const VecInfo& inf, size_t off, size_t uoff, float2* sm,
                                              const float2* bs = nullptr) {
    const bool tan = a.dvpot != nullptr && inf.dvrow >= 0;
    const bool real = a.coef.ch[inf.cset].y == 0.f && a.coef.c2[inf.cset].y == 0.f;
    if (tan && real) sep_points<N, ROWS, PITCH, NT, U, true, true>(a, inf, off, uoff, sm, bs);
    else if (tan) sep_points<N, ROWS, PITCH, NT, U, true, false>(a, inf, off, uoff, sm, bs);
    else if (real) sep_points<N, ROWS, PITCH, NT, U, false, true>(a, inf, off, uoff, sm, bs);
    else sep_points<N, ROWS, PITCH, NT, U, false, false>(a, inf, off, uoff, sm, bs);
}

// L2 prefetch of a unit's pointwise operands but W (one thread), PTS points at offset off
template <int N, int PTS>
__device__ __forceinline__ void sep_prefetch(const StepArgs& a, const VecInfo& inf, size_t off, size_t uoff) {
    constexpr size_t NG = (size_t)N * N * N;
    constexpr unsigned CB = PTS * sizeof(float2), VB = PTS * sizeof(float);
    if (a.psi != nullptr) l2_prefetch(a.psi + off, CB);
    if (a.b2 != nullptr) l2_prefetch(a.b2 + off, CB);
    l2_prefetch(a.vpot + (size_t)inf.vrow * NG + uoff, VB);
    if (a.dvpot != nullptr && inf.dvrow >= 0) {
        l2_prefetch(a.dvpot + (size_t)inf.dvrow * NG + uoff, VB);
        l2_prefetch(a.b1 + (size_t)inf.partner * NG + uoff, CB);
    }
}

// ------------------------------------------------------------------ z lines, n <= 128
// W = T_z b: a warp takes CPW neighbouring columns, each in the registers of T lanes (two lanes up to
// 64 points: four measured the same, 43 us at 64^3 x 64).  The blocks
// past the columns' reduce the vector's KB partials (k_kb_reduce's work, which the plane pass needs
// and which nothing here depends on), so that the term has no launch of its own for it.
constexpr int ZS_NT = 128;
template <int N> struct ZsCfg {
    static constexpr int T = N <= 64 ? 2 : 4;
    static constexpr int BLOCKS = N * N / (32 / T * (ZS_NT / 32));
    static constexpr int MINB = N <= 32 ? 8 : (N == 64 || N == 128 ? 4 : 5);
};

template <int N>
__global__ void __launch_bounds__(ZS_NT, (ZsCfg<N>::MINB))
k_sep_z(const float2* in, float2* W, float c, const float2* __restrict__ tw, KbReduceArgs kr) {
    constexpr int T = ZsCfg<N>::T, P = N / T, CPW = 32 / T;
    __shared__ float2 tws[N];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // vectors in descending order: the plane pass before left the last ones in L2, and this pass
    // leaves the first ones there for the plane pass after it
    const int b = gridDim.y - 1 - blockIdx.y;
    if (blockIdx.x >= ZsCfg<N>::BLOCKS) {
        dependents_wait();
        dependents_launch();
        kb_reduce_warp(kr, (blockIdx.x - ZsCfg<N>::BLOCKS) * (ZS_NT / 32) + warp, b, lane);
        return;
    }
    for (int i = threadIdx.x; i < N; i += ZS_NT) tws[i] = __ldg(tw + i);
    const int t = lane / CPW;
    const size_t off = (size_t)b * N * N * N + (blockIdx.x * (ZS_NT / 32) + warp) * CPW + lane % CPW + (size_t)t * N * N;
    dependents_wait();                       // the step before wrote `in`
    dependents_launch();
    float2 v[P];
#pragma unroll
    for (int a = 0; a < P; ++a) v[a] = ld2_written(in + off + (size_t)(T * a) * N * N);
    __syncthreads();
    line_op<N, T>(v, lane, tws, [&](int k1, int i) { return axis_factor<N, T>(k1, i, c); });
#pragma unroll
    for (int a = 0; a < P; ++a) W[off + (size_t)(T * a) * N * N] = v[a];
}

// ------------------------------------------------------------------ planes, n <= 128
// A block per plane.  Up to 64^2 the plane of b is copied to shared memory and T_x of the rows and T_y of
// the columns go to a second plane; the KB apply and the pointwise part follow on that one (64^3 x 36: 111 us
// per term with the KB apply first, which then waits for the z lines, and 106 so).  Two planes of 96^2 or
// 128^2 leave room for one block at best: there the rows are transformed in place, the KB apply comes
// before the columns, and b is read again from L2 (96^3 x 7: 91 us, against 102 with the KB apply first).
// Four lanes per line: two lanes hold twice the points and half the warps, and the same pass took
// 195 us instead of 169 at 64^3 x 64.  The operands of the pointwise part are asked into L2 once the
// plane has landed, and read evict-first: asked at the block's start they were evicted before use (a
// third more DRAM traffic than the algorithm's).
template <int N> struct SpCfg {
    static constexpr int T = 4;
    static constexpr int NT = N * T;
    // row pitch of the plane in shared memory: a half-warp reads 8 rows at two neighbouring points
    // without bank conflicts, and rows start on 16 bytes
    static constexpr int PITCH = N + 2;
    static constexpr bool KEEP = N <= 64;    // the plane of b stays in shared memory
    static constexpr size_t POINTS = (size_t)N * PITCH * (KEEP ? 2 : 1);
    static constexpr int MINB = N == 16 ? 16 : (N == 32 ? 8 : (N == 48 ? 5 : (N == 64 ? 3 : (N == 96 ? 2 : 1))));
};

template <int N>
__global__ void __launch_bounds__(SpCfg<N>::NT, (SpCfg<N>::MINB)) k_sep_plane(StepArgs a, float c, const float2* __restrict__ tw) {
    constexpr int T = SpCfg<N>::T, P = N / T, CPW = 32 / T, NT = SpCfg<N>::NT, PITCH = SpCfg<N>::PITCH;
    constexpr bool KEEP = SpCfg<N>::KEEP;
    extern __shared__ __align__(16) float2 sm[];
    float2* bs = sm + N * PITCH;
    float2* tws = bs + (KEEP ? N * PITCH : 0);
    float2* kcs = tws + N;
    const int z = blockIdx.x, b = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t uoff = (size_t)z * N * N, off = (size_t)b * N * N * N + uoff;
    const VecInfo inf = a.info[b];
    KbHead kh;
    if (a.kbc != nullptr || a.kbp != nullptr) kh = kb_head(a, z);
    if constexpr (KEEP) {
        const float2* src = a.b1 + off;
#pragma unroll 4
        for (int q = threadIdx.x; q < N * N / 2; q += NT) sep_cp16(bs + (q / (N / 2)) * PITCH + 2 * (q % (N / 2)), src + 2 * q);
        asm volatile("cp.async.commit_group;" ::: "memory");
    } else {
        const float2* src = a.b1 + off;
#pragma unroll 4
        for (int q = threadIdx.x; q < N * N / 2; q += NT) sep_cp16(sm + (q / (N / 2)) * PITCH + 2 * (q % (N / 2)), src + 2 * q);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (KEEP && threadIdx.x == 0) {
        // the plane of the block half a wave of resident blocks later, into L2 (162 -> 157 us at 64^3 x 64;
        // at 96 and 128, with one or two blocks per SM, it gained nothing)
        const long nxt = (long)b * N + z + SpCfg<N>::MINB * 152 / 2;
        if (nxt < (long)gridDim.y * N) l2_prefetch(a.b1 + nxt * N * N, N * N * sizeof(float2));
    }
    for (int i = threadIdx.x; i < N; i += NT) tws[i] = __ldg(tw + i);
    const float2* kc = a.kbc != nullptr ? a.kbc + (size_t)b * a.total_slots * 4 : nullptr;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (KEEP && threadIdx.x == 0) sep_prefetch<N, N * N>(a, inf, off, uoff);
    const int l = warp * CPW + lane % CPW, t = lane / CPW;
    const auto f = [&](int k1, int i) { return axis_factor<N, T>(k1, i, c); };
    {
        // T_x b of row l, in place in the one-plane form (a lane writes the points it has read)
        float2 v[P];
        float2* row = sm + l * PITCH + t;
        const float2* src = (KEEP ? bs : sm) + l * PITCH + t;
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = src[T * i];
        line_op<N, T>(v, lane, tws, f);
#pragma unroll
        for (int i = 0; i < P; ++i) row[T * i] = v[i];
    }
    const auto staged = [&] {
        dependents_wait();                   // the z lines wrote W and the coefficients
        if (threadIdx.x == 0) {
            if (!KEEP) sep_prefetch<N, N * N>(a, inf, off, uoff);
            l2_prefetch(a.W + off, N * N * sizeof(float2));
        }
        if (kc != nullptr) kb_stage_coeffs<NT>(kh, kc, kcs);
    };
    if (!KEEP && kc != nullptr) {
        kb_apply_unit<N, PITCH, NT, 2>(a, kh, kcs, sm, staged);
    } else {
        if (!KEEP) staged();
        __syncthreads();
    }
    {
        // + T_y b of column l
        float2 v[P];
        float2* col = sm + t * PITCH + l;
        if constexpr (KEEP) {
#pragma unroll
            for (int i = 0; i < P; ++i) v[i] = bs[(t + T * i) * PITCH + l];
        } else {
            const float2* src = a.b1 + off + (size_t)t * N + l;
#pragma unroll
            for (int i = 0; i < P; ++i) v[i] = __ldg(src + T * i * N);
        }
        line_op<N, T>(v, lane, tws, f);
#pragma unroll
        for (int i = 0; i < P; ++i) col[T * i * PITCH] = cadd(col[T * i * PITCH], v[i]);
    }
    if constexpr (KEEP) {
        if (kc != nullptr) kb_apply_unit<N, PITCH, NT, 2>(a, kh, kcs, sm, staged);
        else staged();
    }
    KbSlots ks;
    if (a.kbp != nullptr) ks = kb_project_begin<NT>(a, kh);
    __syncthreads();
    sep_pointwise<N, N, PITCH, NT, 1>(a, inf, off, uoff, sm, KEEP ? bs : nullptr);
    dependents_launch();
    if (a.kbp == nullptr) return;
    kb_project_unit<N, PITCH, NT, 2>(a, kh, ks, b, sm);
}

// ------------------------------------------------------------------ split-operator passes
// e^{-i T dt} is a product over the axes: planes W = e^{-i (T_x + T_y) dt} e^{-i V dt/2} psi (16 B per
// vector-point), then z lines psi = e^{-i V dt/2} e^{-i T_z dt} W (16 B), where the 3D transform took three
// passes.  The half-step phases e^{-i V dt/2} come from a table per potential row, which the vectors
// share (backward vectors take the conjugate); the factors along an axis depend on |m| only and are
// computed once per block.  Along an axis the line gains IDFT((e^{-i T_a dt} - 1) DFT(line)): the rounding
// of the transforms and of the factor, which is the same in every step, is then in proportion to what
// the step changes (three factors of modulus 1 +- 2^-25 would add up over the steps).
// Measured, ten steps of 27 vectors at 64^3 with KB: 1.40 -> 0.94 ms, of which the two passes 0.66 (at two
// blocks of 256 threads per SM; three or four spill the second line operation: 1.03, 1.04); the error
// against 64 bits went from 1.3e-6 to 3.7e-7.  Started early as the kernels of a term are, the two passes
// were slower (1.01 ms): they have little to do before they wait.
template <int N>
__device__ __forceinline__ void axis_phases(float2* ph, float ks, float dt, int nt) {
    for (int m = threadIdx.x; m <= N / 2; m += nt) {
        float sn, cs;                          // e^{-i w} - 1 = -2 sin^2(w/2) - 2 i sin(w/2) cos(w/2), over N
        sincosf(0.25f * ks * (float)(m * m) * dt, &sn, &cs);
        ph[m] = make_float2(sn * sn * (-2.0f / N), sn * cs * (-2.0f / N));
    }
}
template <int N, int T>
__device__ __forceinline__ float2 axis_phase(const float2* ph, int k1, int i) {
    return ph[abs(k1 + (N / T) * i - (2 * i >= T ? N : 0))];
}

template <int N>
__global__ void __launch_bounds__(SpCfg<N>::NT, (N == 128 ? 1 : (N == 64 ? 2 : 8)))
k_split_plane(const float2* __restrict__ psi, const float2* __restrict__ phase, const float* __restrict__ dvpot,
              const VecInfo* __restrict__ info, float dt, float ks, float2* __restrict__ W, const float2* __restrict__ tw) {
    constexpr int T = SpCfg<N>::T, P = N / T, CPW = 32 / T, NT = SpCfg<N>::NT, PITCH = SpCfg<N>::PITCH;
    constexpr size_t NG = (size_t)N * N * N;
    extern __shared__ __align__(16) float2 sm[];
    float2* tws = sm + N * PITCH;
    float2* ph = tws + N;
    const int z = blockIdx.x, b = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t uoff = (size_t)z * N * N, off = (size_t)b * NG + uoff;
    const VecInfo inf = info[b];
    const float sg = inf.cset == 0 ? 1.f : -1.f;
    const float2* E = phase + (size_t)inf.vrow * NG + uoff;
    const bool tan = dvpot != nullptr && inf.dvrow >= 0;
    const float* dV = tan ? dvpot + (size_t)inf.dvrow * NG + uoff : nullptr;
    const float2* pp = tan ? psi + (size_t)inf.partner * NG + uoff : nullptr;
#pragma unroll 2
    for (int q = threadIdx.x; q < N * N / 2; q += NT) {
        const int o = 2 * q;
        const float4 v = ld4(psi + off + o), e = ld4(E + o);
        float2 a0 = make_float2(v.x, v.y), a1 = make_float2(v.z, v.w);
        if (tan) {
            // the derivative of the half-step along V -> V + lam dv: psi - i s (dt/2) dv psi_partner
            const float4 pa = ld4(pp + o);
            const float2 d = __ldg(reinterpret_cast<const float2*>(dV + o));
            const float h = 0.5f * sg * dt;
            a0 = make_float2(a0.x + h * d.x * pa.y, a0.y - h * d.x * pa.x);
            a1 = make_float2(a1.x + h * d.y * pa.w, a1.y - h * d.y * pa.z);
        }
        a0 = cmul(a0, make_float2(e.x, sg * e.y));
        a1 = cmul(a1, make_float2(e.z, sg * e.w));
        *reinterpret_cast<float4*>(sm + (q / (N / 2)) * PITCH + 2 * (q % (N / 2))) = make_float4(a0.x, a0.y, a1.x, a1.y);
    }
    for (int i = threadIdx.x; i < N; i += NT) tws[i] = __ldg(tw + i);
    axis_phases<N>(ph, ks, sg * dt, NT);
    __syncthreads();
    const int l = warp * CPW + lane % CPW, t = lane / CPW;
    const auto f = [&](int k1, int i) { return axis_phase<N, T>(ph, k1, i); };
    float2 v[P];
    float2* row = sm + l * PITCH + t;
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = row[T * i];
    line_op<N, T>(v, lane, tws, f);
    asm volatile("" ::: "memory");           // the line is read again, not held in registers meanwhile
#pragma unroll
    for (int i = 0; i < P; ++i) row[T * i] = cadd(row[T * i], v[i]);
    __syncthreads();
    const float2* col = sm + t * PITCH + l;
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = col[T * i * PITCH];
    line_op<N, T>(v, lane, tws, f);
    asm volatile("" ::: "memory");
    float2* dst = W + off + (size_t)t * N + l;
#pragma unroll
    for (int i = 0; i < P; ++i) dst[T * i * N] = cadd(col[T * i * PITCH], v[i]);
}

template <int N>
__global__ void __launch_bounds__(ZS_NT, 4)
k_split_z(const float2* __restrict__ W, const float2* __restrict__ phase, const VecInfo* __restrict__ info, float dt,
          float ks, float2* __restrict__ psi, const float2* __restrict__ tw) {
    constexpr int T = ZsCfg<N>::T, P = N / T, CPW = 32 / T;
    constexpr size_t NG = (size_t)N * N * N, NN = (size_t)N * N;
    __shared__ float2 tws[N], ph[N / 2 + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b = gridDim.y - 1 - blockIdx.y;       // the last vectors' W is still in L2
    const VecInfo inf = info[b];
    const float sg = inf.cset == 0 ? 1.f : -1.f;
    for (int i = threadIdx.x; i < N; i += ZS_NT) tws[i] = __ldg(tw + i);
    const size_t at = (blockIdx.x * (ZS_NT / 32) + warp) * CPW + lane % CPW + (size_t)(lane / CPW) * NN;
    const float2* src = W + (size_t)b * NG + at;
    float2 v[P];
#pragma unroll
    for (int a = 0; a < P; ++a) v[a] = __ldg(src + (size_t)(T * a) * NN);
    axis_phases<N>(ph, ks, sg * dt, ZS_NT);
    __syncthreads();
    line_op<N, T>(v, lane, tws, [&](int k1, int i) { return axis_phase<N, T>(ph, k1, i); });
    const float2* E = phase + (size_t)inf.vrow * NG + at;
    float2* dst = psi + (size_t)b * NG + at;
#pragma unroll
    for (int a = 0; a < P; ++a) {
        const float2 e = __ldg(E + (size_t)(T * a) * NN), w = __ldg(src + (size_t)(T * a) * NN);
        dst[(size_t)(T * a) * NN] = cmul(cadd(w, v[a]), make_float2(e.x, sg * e.y));
    }
}

// e^{-i V dt/2} of `pairs` pairs of potential values.  TDH has one in every step, behind the kernel that writes V:
// started while that one ends (three TDH steps, 16^3 x 32 orbitals 113.8 -> 109.9 us, 64^3 x 4 211.6 -> 207.5).
__global__ void __launch_bounds__(256) k_split_phase(int64_t pairs, const float2* V, float hdt, float4* __restrict__ e) {
    dependents_wait();                       // the kernel before may have written V
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < pairs; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 v = ld2_written(V + i);
        float4 p;
        sincosf(v.x * hdt, &p.y, &p.x);
        sincosf(v.y * hdt, &p.w, &p.z);
        e[i] = make_float4(p.x, -p.y, p.z, -p.w);
    }
}

// ------------------------------------------------------------------ n = 288
// A 288-point line in the registers of 12 threads, 24 points each: x[t + 12 a] -> DFT24 over a,
// exchange through shared memory, two DFT12 over t for k1 = t' + 12 i (times W288^(t k1) on the way
// in and its conjugate on the way out), the factor between the DFT12 and its inverse, exchange back
// in place, inverse DFT24.  One round trip through shared memory each way.
constexpr int S2N = 288, S2T = 12, S2P = 24;

// slot(k1, t): position of stage-1 output k1 of thread t in the line's exchange buffer
template <class SLOT, class SYNC>
__device__ __forceinline__ void line288(float2 (&v)[S2P], int t, float c, const float2* tws, float2* ex, SLOT slot, SYNC sync) {
    RegDft<S2P, -1>::run(v);
#pragma unroll
    for (int k = 0; k < S2P; ++k) ex[slot(k, t)] = v[k];
    sync();
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int k1 = t + S2T * i;
        float2 r[S2T];
        r[0] = ex[slot(k1, 0)];
#pragma unroll
        for (int s = 1; s < S2T; ++s) r[s] = cmul(ex[slot(k1, s)], tws[s * k1]);
        RegDft<S2T, -1>::run(r);
#pragma unroll
        for (int k2 = 0; k2 < S2T; ++k2) {
            const float m = (float)(k1 + S2P * k2 - (k2 >= S2T / 2 ? S2N : 0));
            r[k2] = cscale(r[k2], c * m * m);
        }
        RegDft<S2T, +1>::run(r);
        ex[slot(k1, 0)] = r[0];
#pragma unroll
        for (int s = 1; s < S2T; ++s) ex[slot(k1, s)] = cmul(r[s], cconj(tws[s * k1]));
    }
    sync();
#pragma unroll
    for (int k = 0; k < S2P; ++k) v[k] = ex[slot(k, t)];
    RegDft<S2P, +1>::run(v);
}

// z lines (AXIS 0: W = T_z b) and y lines (AXIS 1: W += T_y b) of tiles of 16 x-columns; AXIS 0's
// blocks past the columns' reduce the KB partials.  Five blocks to an SM at 64 registers (8 vectors, z and y:
// 645 and 876 us, 4.76 and 5.24 TB/s; four at 80 registers 681 and 911; tiles of 8 columns, which are two
// sectors to a row, 828 and 1284, of 32 columns 707 and 893).
constexpr int SL_TX = 16, SL_NT = SL_TX * S2T;
template <int AXIS>
__global__ void __launch_bounds__(SL_NT, 5)
k_sep_lines288(const float2* in, float2* W, float c, const float2* __restrict__ tw, KbReduceArgs kr) {
    constexpr int NXT = S2N / SL_TX, BLOCKS = NXT * S2N;
    constexpr size_t NN = (size_t)S2N * S2N, ST = AXIS == 0 ? NN : S2N;
    extern __shared__ __align__(16) float2 sm[];
    float2* tws = sm + S2N * SL_TX;
    const int b = blockIdx.y;
    if (AXIS == 0 && blockIdx.x >= BLOCKS) {
        dependents_wait();
        dependents_launch();
        kb_reduce_warp(kr, (blockIdx.x - BLOCKS) * (SL_NT / 32) + (threadIdx.x >> 5), b, threadIdx.x & 31);
        return;
    }
    for (int i = threadIdx.x; i < S2N; i += SL_NT) tws[i] = __ldg(tw + i);
    const int l = threadIdx.x % SL_TX, t = threadIdx.x / SL_TX;
    const int xt = blockIdx.x % NXT, o = blockIdx.x / NXT;
    const size_t off = (size_t)b * S2N * NN + (size_t)o * (AXIS == 0 ? S2N : NN) + xt * SL_TX + l + (size_t)t * ST;
    if (AXIS == 0) dependents_wait();        // the step before wrote `in`
    float2 v[S2P];
#pragma unroll
    for (int a = 0; a < S2P; ++a) v[a] = ld2_written(in + off + (size_t)(S2T * a) * ST);
    if (AXIS == 1) dependents_wait();        // the z lines wrote W
    line288(v, t, c, tws, sm + l, [](int k, int s) { return (k * S2T + s) * SL_TX; }, [] { __syncthreads(); });
    dependents_launch();
    if constexpr (AXIS == 1) {
        float2 w[S2P];
#pragma unroll
        for (int a = 0; a < S2P; ++a) w[a] = ld2_written(W + off + (size_t)(S2T * a) * ST);
#pragma unroll
        for (int a = 0; a < S2P; ++a) v[a] = cadd(v[a], w[a]);
    }
#pragma unroll
    for (int a = 0; a < S2P; ++a) W[off + (size_t)(S2T * a) * ST] = v[a];
}

// The rows of x: units of 16 rows (192 threads, four blocks per SM), vectors fastest in launch
// order so that a unit's potential rows and KB entries come from DRAM once for all of them.  The
// exchange buffer's pitches (13 per k1, 316 per row) keep every half-warp access free of bank
// conflicts: 12 is the row pitch mod 16 and 13 x 12 mod 16, so the lanes of the next row continue
// the banks of this one.
constexpr int SR_R = 16, SR_NT = SR_R * S2T, SR_PITCH = 316;
__global__ void __launch_bounds__(SR_NT, 4) k_sep_rows288(StepArgs a, float c, const float2* __restrict__ tw) {
    constexpr size_t NG = (size_t)S2N * S2N * S2N;
    extern __shared__ __align__(16) float2 sm[];
    float2* tws = sm + SR_R * SR_PITCH;
    float2* kcs = tws + S2N;
    const int b = blockIdx.x, u = blockIdx.y;
    const size_t uoff = (size_t)u * SR_R * S2N, off = (size_t)b * NG + uoff;
    const VecInfo inf = a.info[b];
    const int r = threadIdx.x / S2T, t = threadIdx.x % S2T;
    KbHead kh;
    if (a.kbc != nullptr || a.kbp != nullptr) kh = kb_head(a, u);
    float2 v[S2P];
    const float2* src = a.b1 + off + (size_t)r * S2N + t;
#pragma unroll
    for (int i = 0; i < S2P; ++i) v[i] = __ldg(src + S2T * i);
    if (threadIdx.x == 0) {
        // the unit of the block half a wave later, into L2
        const long nxt = (long)u * gridDim.x + b + 304;
        if (nxt < (long)gridDim.x * gridDim.y)
            l2_prefetch(a.b1 + (nxt % gridDim.x) * NG + (nxt / gridDim.x) * SR_R * S2N, SR_R * S2N * sizeof(float2));
    }
    for (int i = threadIdx.x; i < S2N; i += SR_NT) tws[i] = __ldg(tw + i);
    const float2* kc = a.kbc != nullptr ? a.kbc + (size_t)b * a.total_slots * 4 : nullptr;
    float2* row = sm + r * SR_PITCH;
    line288(v, t, c, tws, row, [](int k, int s) { return k * 13 + s; }, [] { __syncthreads(); });
    __syncthreads();
#pragma unroll
    for (int i = 0; i < S2P; ++i) row[t + S2T * i] = v[i];
    dependents_wait();                       // the y lines wrote W, and the coefficients are older
    if (threadIdx.x == 0) {
        sep_prefetch<S2N, SR_R * S2N>(a, inf, off, uoff);
        l2_prefetch(a.W + off, SR_R * S2N * sizeof(float2));
    }
    if (kc != nullptr) kb_stage_coeffs<SR_NT>(kh, kc, kcs);
    if (kc != nullptr) kb_apply_unit<S2N, SR_PITCH, SR_NT, 2>(a, kh, kcs, sm, [] {});
    else __syncthreads();
    KbSlots ks;
    if (a.kbp != nullptr) ks = kb_project_begin<SR_NT>(a, kh);
    sep_pointwise<S2N, SR_R, SR_PITCH, SR_NT, 1>(a, inf, off, uoff, sm);
    dependents_launch();
    if (a.kbp == nullptr) return;
    kb_project_unit<S2N, SR_PITCH, SR_NT, 2>(a, kh, ks, b, sm);
}

// ------------------------------------------------------------------ launchers
#define SGW_DISPATCH_SEP(n, ...)                         \
    switch (n) {                                         \
        case 16: { constexpr int N = 16; __VA_ARGS__; } break;   \
        case 32: { constexpr int N = 32; __VA_ARGS__; } break;   \
        case 48: { constexpr int N = 48; __VA_ARGS__; } break;   \
        case 64: { constexpr int N = 64; __VA_ARGS__; } break;   \
        case 96: { constexpr int N = 96; __VA_ARGS__; } break;   \
        case 128: { constexpr int N = 128; __VA_ARGS__; } break; \
        default: break;                                  \
    }

#define SGW_DISPATCH_SPLIT(n, ...)                       \
    switch (n) {                                         \
        case 16: { constexpr int N = 16; __VA_ARGS__; } break;   \
        case 32: { constexpr int N = 32; __VA_ARGS__; } break;   \
        case 64: { constexpr int N = 64; __VA_ARGS__; } break;   \
        case 128: { constexpr int N = 128; __VA_ARGS__; } break; \
        default: break;                                  \
    }

int sep_unit_pos(int n, int o) {
    int pitch = SR_PITCH;
    SGW_DISPATCH_SEP(n, pitch = SpCfg<N>::PITCH);
    return (o / n) * pitch + o % n;
}

int64_t sep_unit_points(int n) { return n == S2N ? (int64_t)SR_R * S2N : (int64_t)n * n; }

size_t sep_step_smem(int n, int max_unit_slots) {
    size_t pts = (size_t)SR_R * SR_PITCH;
    SGW_DISPATCH_SEP(n, pts = SpCfg<N>::POINTS);
    return sizeof(float2) * (pts + n + 4 * (size_t)max_unit_slots);
}

static size_t sep_lines_smem() { return sizeof(float2) * ((size_t)S2N * SL_TX + S2N); }

// Every step kernel may use all the shared memory a block can have: the limit does not depend on
// one context's KB slots, so contexts with different potentials do not disturb each other.
template <class K> static cudaError_t sep_attr(K kern, int bytes) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         (int)cudaSharedmemCarveoutMaxShared);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

template <class K>
static cudaError_t sep_carveout(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}

cudaError_t sep_init_attributes(int n) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if (n == S2N) {
        if ((e = sep_attr(k_sep_lines288<0>, (int)sep_lines_smem()))) return e;
        if ((e = sep_attr(k_sep_lines288<1>, (int)sep_lines_smem()))) return e;
        return sep_attr(k_sep_rows288, optin);
    }
    SGW_DISPATCH_SEP(n, e = sep_attr(k_sep_plane<N>, optin));
    // Small planes' blocks start beside the z lines' (see spread_smem), and an SM that changes between the two
    // kernels' shares of shared memory and L1 has to run dry first: both take the largest share (48^3 x 6:
    // 11.8 -> 11.4 us per term; above, where the z lines use L1, it cost 1 to 4 %).
    if (e == cudaSuccess && n <= 48)
        SGW_DISPATCH_SEP(n, e = sep_carveout(k_sep_plane<N>); if (e == cudaSuccess) e = sep_carveout(k_sep_z<N>));
    return e;
}

void sep_z(int n, const float2* in, float2* W, int batch, float kscale, const float2* tw, const KbReduceArgs& kr,
           cudaStream_t st) {
    if (batch == 0) return;
    const float c = 0.5f * kscale / (float)n;
    if (n == S2N) {
        const unsigned kb = (unsigned)((kr.n_atoms + SL_NT / 32 - 1) / (SL_NT / 32));
        launch_dependent(k_sep_lines288<0>, dim3((S2N / SL_TX) * S2N + kb, batch), SL_NT, sep_lines_smem(), 1, st, in, W, c, tw, kr);
        return;
    }
    const unsigned kb = (unsigned)((kr.n_atoms + ZS_NT / 32 - 1) / (ZS_NT / 32));
    SGW_DISPATCH_SEP(n, launch_dependent(k_sep_z<N>, dim3(ZsCfg<N>::BLOCKS + kb, batch), ZS_NT, 0, 1, st, in, W, c, tw, kr));
}

void sep_y288(const float2* in, float2* W, int batch, float kscale, const float2* tw, cudaStream_t st) {
    if (batch == 0) return;
    launch_dependent(k_sep_lines288<1>, dim3((S2N / SL_TX) * S2N, batch), SL_NT, sep_lines_smem(), 1, st, in, W,
                     0.5f * kscale / S2N, tw, KbReduceArgs{});
}

// Shared memory for a block of the plane pass.  The z lines let the planes in early, and blocks take the
// first free places: without a limit up to MINB crowd on the SMs that run few z lines, and these finish
// last.  A grid of less than MINB blocks to an SM asks for so much that only an even share fits (32^3 x 12:
// 13.2 us per term without, 9.2 with; 48^3 x 6: 17.7, 11.8).
template <int N>
static size_t spread_smem(size_t sm, long blocks) {
    const long per = (blocks + 151) / 152;
    if (per >= SpCfg<N>::MINB) return sm;
    return std::max(sm, ((size_t)228 * 1024 / (per + 1) - 1024 + 255) / 128 * 128);
}

void sep_step(int n, const StepArgs& a, int batch, float kscale, const float2* tw, cudaStream_t st) {
    if (batch == 0) return;
    const float c = 0.5f * kscale / (float)n;
    const size_t sm = sep_step_smem(n, a.kbc != nullptr ? a.max_plane_slots : 0);
    if (n == S2N) {
        launch_dependent(k_sep_rows288, dim3(batch, S2N * S2N / SR_R), SR_NT, sm, 1, st, a, c, tw);
        return;
    }
    SGW_DISPATCH_SEP(n, launch_dependent(k_sep_plane<N>, dim3(N, batch), SpCfg<N>::NT, spread_smem<N>(sm, (long)N * batch), 1, st,
                                         a, c, tw));
}

static size_t split_plane_smem(int n) {
    size_t pts = 0;
    SGW_DISPATCH_SEP(n, pts = (size_t)N * SpCfg<N>::PITCH);
    return sizeof(float2) * (pts + n + n / 2 + 1);
}

cudaError_t sep_split_init_attributes(int n) {
    cudaError_t e = cudaSuccess;
    SGW_DISPATCH_SPLIT(n, e = sep_attr(k_split_plane<N>, (int)split_plane_smem(n)));
    return e;
}

void sep_split_phase(int64_t count, const float* V, float dt, float2* phase, cudaStream_t st) {
    const int64_t pairs = count / 2;         // a row is n^3 values, n even
    launch_dependent(k_split_phase, dim3((unsigned)std::min<int64_t>((pairs + 255) / 256, 152 * 16)), 256, 0, 1, st, pairs,
                     reinterpret_cast<const float2*>(V), 0.5f * dt, reinterpret_cast<float4*>(phase));
}

void sep_split_core(int n, float2* psi, const float2* phase, const float* dvpot, const VecInfo* info, float dt, float kscale,
                    float2* W, int batch, const float2* tw, cudaStream_t st) {
    if (batch == 0) return;
    SGW_DISPATCH_SPLIT(n, {
        k_split_plane<N><<<dim3(N, batch), SpCfg<N>::NT, split_plane_smem(n), st>>>(psi, phase, dvpot, info, dt, kscale, W,
                                                                                   tw);
        k_split_z<N><<<dim3(ZsCfg<N>::BLOCKS, batch), ZS_NT, 0, st>>>(W, phase, info, dt, kscale, psi, tw);
    });
}

}  // namespace sgw
