// Non-FFT kernels of the sGW hot path: Philox white noise, the TDH kick, power-iteration
// reductions, the Sigma(t) reductions (Eq. 5), time ordering of u^R, the
// damped transform (Eq. 7) and the QP root (Eq. 6).
#include <cmath>
#include <mutex>
#include <string>

#include "../../include/sgw.h"
#include "fft_smem.cuh"
#include "sgw_internal.cuh"

namespace sgw {

// ------------------------------------------------------------------ Philox4x32-10
// Written from the published definition (Salmon et al., SC'11): per round
// (c0,c1,c2,c3) <- (hi(M1 c2) ^ c1 ^ k0, lo(M1 c2), hi(M0 c0) ^ c3 ^ k1, lo(M0 c0)),
// key bumped by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k0 += W0;
            k1 += W1;
        }
        const uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        const uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}

__global__ void k_noise(int64_t ng, int64_t nblk, uint32_t k0, uint32_t k1, uint32_t stream_id, int sample0, int n_vec,
                        int64_t total, float amp, float2* __restrict__ out) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t blk = t % nblk;
        const int64_t sv = t / nblk;
        const int v = (int)(sv % n_vec);
        const int s = (int)(sv / n_vec);
        const uint4 w = philox4x32_10(make_uint4((uint32_t)blk, (uint32_t)v, (uint32_t)(sample0 + s), stream_id), k0, k1);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
        float2* o = out + sv * ng;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t g = blk * 4 + u;
            if (g < ng) o[g] = make_float2((ws[u] >> 31) ? -amp : amp, 0.f);
        }
    }
}

void launch_noise(int ng, uint64_t seed, uint32_t stream_id, int sample0, int n_samples, int n_vec, float amp,
                  float2* out, cudaStream_t st) {
    const int64_t nblk = (ng + 3) / 4;
    const int64_t total = nblk * n_samples * n_vec;
    if (total == 0) return;
    const int threads = 256;
    const int64_t blocks = std::min<int64_t>((total + threads - 1) / threads, 152 * 32);
    k_noise<<<(unsigned)blocks, threads, 0, st>>>(ng, nblk, (uint32_t)(seed & 0xFFFFFFFFu), (uint32_t)(seed >> 32),
                                                  stream_id, sample0, n_vec, total, amp, out);
}

// ------------------------------------------------------------------ small elementwise kernels
__global__ void k_real_to_c64(int64_t count, const float* __restrict__ in, float2* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = make_float2(in[i], 0.f);
}

void launch_real_to_c64(int64_t count, const float* in, float2* out, cudaStream_t st) {
    if (count == 0) return;
    const int64_t blocks = std::min<int64_t>((count + 255) / 256, 152 * 32);
    k_real_to_c64<<<(unsigned)blocks, 256, 0, st>>>(count, in, out);
}

// psi[s][l] = eta[s][l];  psi[s][n_eta + l] = -i v_p[s] eta[s][l]   (derivative of e^{-i lam v_p} eta)
__global__ void k_kick(int64_t ng, const float2* __restrict__ eta, const float* __restrict__ vp, int n_samples, int n_eta,
                       float2* __restrict__ psi) {
    const int64_t total = ng * n_samples * n_eta;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = i % ng;
        const int64_t sl = i / ng;
        const int64_t s = sl / n_eta, l = sl % n_eta;
        const float2 e = eta[i];
        const float v = vp[s * ng + g];
        psi[(s * 2 * n_eta + l) * ng + g] = e;
        psi[(s * 2 * n_eta + n_eta + l) * ng + g] = make_float2(v * e.y, -v * e.x);
    }
}

void launch_kick(int ng, const float2* eta, const float* vp, int n_samples, int n_eta, float2* psi, cudaStream_t st) {
    const int64_t total = (int64_t)ng * n_samples * n_eta;
    if (total == 0) return;
    const int64_t blocks = std::min<int64_t>((total + 255) / 256, 152 * 32);
    k_kick<<<(unsigned)blocks, 256, 0, st>>>(ng, eta, vp, n_samples, n_eta, psi);
}

// out[i] = phi[i mod ng] * eta[i]
__global__ void k_scale_mul(int64_t count, const float* __restrict__ phi, int64_t ng, const float2* __restrict__ eta,
                            float2* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        const float f = phi[i % ng];
        const float2 e = eta[i];
        out[i] = make_float2(f * e.x, f * e.y);
    }
}

void launch_scale_mul(int64_t count, const float* phi, int ng, const float2* eta, float2* out, cudaStream_t st) {
    if (count == 0) return;
    const int64_t blocks = std::min<int64_t>((count + 255) / 256, 152 * 32);
    k_scale_mul<<<(unsigned)blocks, 256, 0, st>>>(count, phi, ng, eta, out);
}

// Split one filtered batch per sample (vector 0 = zeta, 1..n_eta = eta_l):
//   eta[s][l] = filt[s][1 + l]; zeta[s] = (zeta_occ = filt[s][0], zeta_unocc = noise[s][0] - filt[s][0]);
//   source[s] = Re noise[s][0] * phi   (the source zeta-bar phi of the TDH kick).
__global__ void k_prepare(int64_t ng, const float2* __restrict__ noise, const float2* __restrict__ filt,
                          const float* __restrict__ phi, int n_samples, int n_eta, float2* __restrict__ eta,
                          float2* __restrict__ zeta, float* __restrict__ source) {
    const int64_t per = (int64_t)(n_eta + 1) * ng;
    const int64_t total = per * n_samples;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = i / per, r = i % per;
        const int64_t v = r / ng, g = r % ng;
        const float2 f = filt[i];
        if (v == 0) {
            const float2 z = noise[i];
            zeta[(2 * s) * ng + g] = f;
            zeta[(2 * s + 1) * ng + g] = make_float2(z.x - f.x, z.y - f.y);
            source[s * ng + g] = z.x * phi[g];
        } else {
            eta[(s * n_eta + v - 1) * ng + g] = f;
        }
    }
}

void launch_prepare(int ng, const float2* noise, const float2* filt, const float* phi, int n_samples, int n_eta,
                    float2* eta, float2* zeta, float* source, cudaStream_t st) {
    const int64_t total = (int64_t)ng * (n_eta + 1) * n_samples;
    if (total == 0) return;
    const int64_t blocks = std::min<int64_t>((total + 255) / 256, 152 * 32);
    k_prepare<<<(unsigned)blocks, 256, 0, st>>>(ng, noise, filt, phi, n_samples, n_eta, eta, zeta, source);
}

// ------------------------------------------------------------------ block reductions
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* sh /*[32*NV]*/) {
#pragma unroll
    for (int i = 0; i < NV; ++i)
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int i = 0; i < NV; ++i) sh[w * NV + i] = v[i];
    __syncthreads();
    if (threadIdx.x < 32) {
        for (int i = 0; i < NV; ++i) {
            double t = threadIdx.x < nw ? sh[threadIdx.x * NV + i] : 0.0;
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            v[i] = t;
        }
    }
}

template <int NV>
__device__ __forceinline__ void block_sumf(float (&v)[NV], float* sh /*[32*NV]*/) {
#pragma unroll
    for (int i = 0; i < NV; ++i)
        for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int i = 0; i < NV; ++i) sh[w * NV + i] = v[i];
    __syncthreads();
    if (threadIdx.x < 32) {
        for (int i = 0; i < NV; ++i) {
            float t = threadIdx.x < nw ? sh[threadIdx.x * NV + i] : 0.f;
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            v[i] = t;
        }
    }
}

// ------------------------------------------------------------------ power iteration (Sec. 2.1)
// scal[0] = Re <v|w>/dV, scal[1] = <w|w>/dV, scal[2] = <v|v>/dV  (the dV factors cancel).  One
// block, so that the sums have a fixed order (the iteration runs once per setup).
__global__ void __launch_bounds__(1024) k_dot2(int64_t ng, const float2* __restrict__ v, const float2* __restrict__ w,
                                               double* scal) {
    __shared__ double sh[32 * 3];
    double a[3] = {0.0, 0.0, 0.0};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ng; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 x = v[i], y = w[i];
        a[0] += (double)x.x * y.x + (double)x.y * y.y;
        a[1] += (double)y.x * y.x + (double)y.y * y.y;
        a[2] += (double)x.x * x.x + (double)x.y * x.y;
    }
    block_sum<3>(a, sh);
    if (threadIdx.x == 0) {
        scal[0] = a[0];
        scal[1] = a[1];
        scal[2] = a[2];
    }
}

void launch_dot2(int ng, const float2* v, const float2* w, double* scal, cudaStream_t st) {
    k_dot2<<<1, 1024, 0, st>>>(ng, v, w, scal);
}

// With sigma = *shift (0 if null): est = (S0 - sigma S2)/S2 (Rayleigh quotient of A = H - sigma);
// v <- (w - sigma v) / |w - sigma v|.
__global__ void k_power_update(int64_t ng, const float2* __restrict__ w, float2* __restrict__ v,
                               const double* __restrict__ scal, double* est_out, const double* shift) {
    const double sig = shift ? *shift : 0.0;
    const double s0 = scal[0], s1 = scal[1], s2 = scal[2];
    const double nrm2 = s1 - 2.0 * sig * s0 + sig * sig * s2;
    const float inv = (float)(1.0 / sqrt(nrm2));
    const float sg = (float)sig;
    if (blockIdx.x == 0 && threadIdx.x == 0 && est_out) *est_out = (s0 - sig * s2) / s2;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ng; i += (int64_t)gridDim.x * blockDim.x) {
        const float2 a = w[i], b = v[i];
        v[i] = make_float2((a.x - sg * b.x) * inv, (a.y - sg * b.y) * inv);
    }
}

void launch_power_update(int ng, const float2* w, float2* v, const double* scal, double* est_out, const double* shift,
                         float /*dV*/, cudaStream_t st) {
    const int blocks = std::min<int>((ng + 255) / 256, 152 * 4);
    k_power_update<<<blocks, 256, 0, st>>>(ng, w, v, scal, est_out, shift);
}

// ------------------------------------------------------------------ Sigma(t) accumulation (Eq. 5)
// zeta: [n_samples][2] (occ, unocc).  partial[((s*(n_steps+1) + j)*2 + pm) * nblk + blk]:
// pm = 0: sum phi zeta_unocc u ; pm = 1: sum phi zeta_occ u.

// A sum kept as three floats, s0 + s1 + s2: what rounding s0 loses goes to s1 without loss, what s1 loses
// to s2 (Knuth's two-sum).  72 bits to FP64's 53.
struct Sum3 {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    static __device__ __forceinline__ float two_sum(float& s, float x) {     // s + x exactly: the new s and what is returned
        const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z));
        s = t;
        return e;
    }
    // adds x (h + l), h + l a product's two halves; m: the largest leading product so far
    __device__ __forceinline__ void add(float x, float h, float l, float& m) {
        const float a = __fmul_rn(x, h), b = __fmaf_rn(x, h, -a), c = __fmul_rn(x, l), d = __fmaf_rn(x, l, -c);
        m = fmaxf(m, fabsf(a));
        const float e = two_sum(s0, a);
        const float e1 = two_sum(s1, b), e2 = two_sum(s1, c), e3 = two_sum(s1, e);
        s2 = __fadd_rn(s2, __fadd_rn(__fadd_rn(e1, e2), __fadd_rn(e3, d)));
    }
    __device__ __forceinline__ void add(const Sum3& o) {
        const float e = two_sum(s0, o.s0), e1 = two_sum(s1, o.s1), e2 = two_sum(s1, e);
        s2 = __fadd_rn(s2, __fadd_rn(o.s2, __fadd_rn(e1, e2)));
    }
    __device__ __forceinline__ double value() const { return (double)s0 + ((double)s1 + (double)s2); }
};

// f zeta u summed over this thread's points (complex products, no conjugation) in T
template <typename T>
__device__ __forceinline__ void sigma_points(int64_t ng, const float2* zu, const float2* zo, const float* phi,
                                             const float2* uj, T (&a)[4]) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ng; i += (int64_t)gridDim.x * blockDim.x) {
        const float f = phi[i];
        const float2 uu = uj[i];
        const float2 p = zu[i], m = zo[i];
        const T ur = (T)uu.x * f, ui = (T)uu.y * f;
        a[0] += (T)p.x * ur - (T)p.y * ui;
        a[1] += (T)p.x * ui + (T)p.y * ur;
        a[2] += (T)m.x * ur - (T)m.y * ui;
        a[3] += (T)m.x * ui + (T)m.y * ur;
    }
}

// T = double: the FP64 units do one or two operations a clock and SM, and the 17 that a point takes and
// those of the block's sums made this 58 us at 64^3 x 4 (0.45 TB/s).  Threads and warps sum instead as
// Sum3 on the FP32 units, 300 operations a point, with less rounding than FP64's: 20 us.  The
// halves of the products are exact while they are normal numbers: each product may lose 2^-149 where they
// are not, and |x| 2^-150 with x = zeta, whose factor u phi has halves of its own.  A block has at most 2^18
// points and a sum two products of each, so the losses stay below 2^-53 of the largest product while that is
// above 2^-76 and above 2^-77 |x|.  A block where it is not, or is above 2^100, or whose sums are not numbers,
// does its points again in FP64.
template <typename T>
__global__ void __launch_bounds__(256)
k_sigma_accum(int64_t ng, const float2* __restrict__ zeta, const float* __restrict__ phi, const float2* __restrict__ u,
              int64_t u_ss, int j, int n_steps, double2* __restrict__ partial) {
    __shared__ T sh[32 * 4];
    const int s = blockIdx.y;
    const float2* zo = zeta + (size_t)(2 * s) * ng;
    const float2* zu = zeta + (size_t)(2 * s + 1) * ng;
    const float2* uj = u + (size_t)s * u_ss + (size_t)j * ng;
    const size_t base = ((size_t)s * (n_steps + 1) + j) * 2;
    T a[4] = {0, 0, 0, 0};
    if constexpr (sizeof(T) == 8) {
        __shared__ double w[8][4];
        __shared__ float wbig[8], wx[8];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        Sum3 q[4];
        float big = 0.f, xs = 0.f;           // the largest product's and the largest zeta's magnitude
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < ng; i += (int64_t)gridDim.x * blockDim.x) {
            const float f = phi[i];
            const float2 uu = uj[i];
            const float2 p = zu[i], m = zo[i];
            xs = fmaxf(fmaxf(xs, fmaxf(fabsf(p.x), fabsf(p.y))), fmaxf(fabsf(m.x), fabsf(m.y)));
            const float rh = __fmul_rn(uu.x, f), rl = __fmaf_rn(uu.x, f, -rh);
            const float ih = __fmul_rn(uu.y, f), il = __fmaf_rn(uu.y, f, -ih);
            q[0].add(p.x, rh, rl, big); q[0].add(-p.y, ih, il, big);
            q[1].add(p.x, ih, il, big); q[1].add(p.y, rh, rl, big);
            q[2].add(m.x, rh, rl, big); q[2].add(-m.y, ih, il, big);
            q[3].add(m.x, ih, il, big); q[3].add(m.y, rh, rl, big);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
            xs = fmaxf(xs, __shfl_xor_sync(0xffffffffu, xs, o));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                Sum3 x;
                x.s0 = __shfl_down_sync(0xffffffffu, q[k].s0, o);
                x.s1 = __shfl_down_sync(0xffffffffu, q[k].s1, o);
                x.s2 = __shfl_down_sync(0xffffffffu, q[k].s2, o);
                q[k].add(x);
            }
        }
        if (lane == 0) {
            bool finite = true;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                w[warp][k] = q[k].value();
                finite = finite && fabsf(q[k].s0) <= 0x1p120f;
            }
            wbig[warp] = finite ? big : __int_as_float(0x7f800000);
            wx[warp] = xs;
        }
        __syncthreads();
        big = xs = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            big = fmaxf(big, wbig[i]);
            xs = fmaxf(xs, wx[i]);
        }
        if (big >= 0x1p-76f && big >= 0x1p-77f * xs && big <= 0x1p100f) {
            if (threadIdx.x < 2) {
                double re = 0, im = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    re += w[i][2 * threadIdx.x];
                    im += w[i][2 * threadIdx.x + 1];
                }
                partial[(base + threadIdx.x) * gridDim.x + blockIdx.x] = make_double2(re, im);
            }
            return;
        }
    }
    sigma_points<T>(ng, zu, zo, phi, uj, a);
    if constexpr (sizeof(T) == 8) block_sum<4>(a, sh);
    else block_sumf<4>(a, sh);
    if (threadIdx.x == 0) {
        partial[(base + 0) * gridDim.x + blockIdx.x] = make_double2((double)a[0], (double)a[1]);
        partial[(base + 1) * gridDim.x + blockIdx.x] = make_double2((double)a[2], (double)a[3]);
    }
}

void launch_sigma_accum(int ng, const float2* zeta, const float* phi, const float2* u, int n_samples,
                        int64_t u_sample_stride, int j, int n_steps, float /*dV*/, int fp64, double2* partial, int nblk,
                        cudaStream_t st) {
    const dim3 grid(nblk, n_samples);
    if (fp64)
        k_sigma_accum<double><<<grid, 256, 0, st>>>(ng, zeta, phi, u, u_sample_stride, j, n_steps, partial);
    else
        k_sigma_accum<float><<<grid, 256, 0, st>>>(ng, zeta, phi, u, u_sample_stride, j, n_steps, partial);
}

// ------------------------------------------------------------------ xi compression (Sec. 2.3)
// Draw k of xi_m of sample `sample`: Philox counter (k, m, sample, stream): segment p = floor(w0
// n_seg / 2^32) (the L points from L p), sign of point l = bit l of w1 (set -> -1).
__device__ __forceinline__ void xi_draw(uint32_t k, uint32_t m, uint32_t sample, uint32_t stream, uint32_t k0,
                                        uint32_t k1, uint32_t n_seg, uint32_t* pos, uint32_t* signs) {
    const uint4 w = philox4x32_10(make_uint4(k, m, sample, stream), k0, k1);
    *pos = (uint32_t)(((uint64_t)w.x * n_seg) >> 32);
    *signs = w.y;
}

// U[s][m] (row stride u_ss per sample) = c dV sum_r xi_m(r) f_s(r) for real rows f_s (stride f_ss):
// one warp per (m, s), lane l < L on point l of each draw; warp sums in a fixed order.
__global__ void __launch_bounds__(256)
k_xi_project(const float* __restrict__ f, int64_t f_ss, int n_samples, int n_xi, int K, int L, uint32_t n_seg,
             uint32_t k0, uint32_t k1, uint32_t stream, int sample0, float cdv, float* __restrict__ U, int64_t u_ss) {
    const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= (int64_t)n_xi * n_samples) return;
    const int m = (int)(w % n_xi), s = (int)(w / n_xi);
    const float* fs = f + (size_t)s * f_ss;
    float acc = 0.f;
    for (int kb = 0; kb < K; kb += 32) {
        // lane i draws segment kb + i once; the warp walks the draws in order through shuffles
        uint32_t pl = 0, sgl = 0;
        if (kb + lane < K) xi_draw((uint32_t)(kb + lane), (uint32_t)m, (uint32_t)(sample0 + s), stream, k0, k1, n_seg, &pl, &sgl);
        const int kn = min(32, K - kb);
        for (int i = 0; i < kn; ++i) {
            const uint32_t p = __shfl_sync(0xffffffffu, pl, i), sg = __shfl_sync(0xffffffffu, sgl, i);
            if (lane < L) {
                const float v = fs[(size_t)p * L + lane];
                acc += ((sg >> lane) & 1u) ? -v : v;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) U[(size_t)s * u_ss + m] = cdv * acc;
}

void launch_xi_project(const float* f, int64_t f_ss, int n_samples, int n_xi, int K, int L, int64_t ng, uint64_t seed,
                       uint32_t stream, int sample0, float cdv, float* U, int64_t u_ss, cudaStream_t st) {
    const int64_t warps = (int64_t)n_xi * n_samples;
    if (warps == 0) return;
    k_xi_project<<<(unsigned)((warps * 32 + 255) / 256), 256, 0, st>>>(
        f, f_ss, n_samples, n_xi, K, L, (uint32_t)(ng / L), (uint32_t)(seed & 0xFFFFFFFFu), (uint32_t)(seed >> 32),
        stream, sample0, cdv, U, u_ss);
}

// Sigma accumulation in the xi basis: partial sums of sum_m U_m(j) c sum_r xi_m(r)... written as
// sum_m U_m(j) [c sum_k sum_l sign phi zeta] for zeta_unocc (pm 0) and zeta_occ (pm 1), same partial
// layout as k_sigma_accum (the dV and the signs of Sigma(-t) are applied by k_sigma_reduce).
// Block b of sample s takes xi functions m = warp index + b * warps_per_block, strided by the grid.
template <typename T>
__global__ void __launch_bounds__(256)
k_sigma_accum_xi(const float2* __restrict__ zeta, const float* __restrict__ phi, const float2* __restrict__ Uxi,
                 int64_t u_ss, int j, int n_steps, int n_xi, int K, int L, uint32_t n_seg, uint32_t k0, uint32_t k1,
                 uint32_t stream, int sample0, float c, int64_t ng, double2* __restrict__ partial) {
    __shared__ T sh[32 * 4];
    const int s = blockIdx.y;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const float2* zo = zeta + (size_t)(2 * s) * ng;
    const float2* zu = zeta + (size_t)(2 * s + 1) * ng;
    const float2* Uj = Uxi + (size_t)s * u_ss + (size_t)j * n_xi;
    T a[4] = {0, 0, 0, 0};
    for (int m = blockIdx.x * wpb + wib; m < n_xi; m += gridDim.x * wpb) {
        float b[4] = {0.f, 0.f, 0.f, 0.f};     // sum over the support of sign phi zeta_unocc / zeta_occ
        for (int kb = 0; kb < K; kb += 32) {
            uint32_t pl = 0, sgl = 0;
            if (kb + lane < K)
                xi_draw((uint32_t)(kb + lane), (uint32_t)m, (uint32_t)(sample0 + s), stream, k0, k1, n_seg, &pl, &sgl);
            const int kn = min(32, K - kb);
            for (int i = 0; i < kn; ++i) {
                const uint32_t p = __shfl_sync(0xffffffffu, pl, i), sg = __shfl_sync(0xffffffffu, sgl, i);
                if (lane < L) {
                    const size_t r = (size_t)p * L + lane;
                    const float f = ((sg >> lane) & 1u) ? -phi[r] : phi[r];
                    const float2 pu = zu[r], po = zo[r];
                    b[0] += f * pu.x; b[1] += f * pu.y;
                    b[2] += f * po.x; b[3] += f * po.y;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            for (int o = 16; o > 0; o >>= 1) b[i] += __shfl_xor_sync(0xffffffffu, b[i], o);
        if (lane == 0) {
            const float2 u = Uj[m];
            const T ur = (T)u.x * c, ui = (T)u.y * c;
            a[0] += (T)b[0] * ur - (T)b[1] * ui;
            a[1] += (T)b[0] * ui + (T)b[1] * ur;
            a[2] += (T)b[2] * ur - (T)b[3] * ui;
            a[3] += (T)b[2] * ui + (T)b[3] * ur;
        }
    }
    if constexpr (sizeof(T) == 8) block_sum<4>(a, sh);
    else block_sumf<4>(a, sh);
    if (threadIdx.x == 0) {
        const size_t base = ((size_t)s * (n_steps + 1) + j) * 2;
        partial[(base + 0) * gridDim.x + blockIdx.x] = make_double2((double)a[0], (double)a[1]);
        partial[(base + 1) * gridDim.x + blockIdx.x] = make_double2((double)a[2], (double)a[3]);
    }
}

void launch_sigma_accum_xi(const float2* zeta, const float* phi, const float2* Uxi, int n_samples, int64_t u_ss, int j,
                           int n_steps, int n_xi, int K, int L, int64_t ng, uint64_t seed, uint32_t stream, int sample0,
                           float c, int fp64, double2* partial, int nblk, cudaStream_t st) {
    const dim3 grid(nblk, n_samples);
    const uint32_t k0 = (uint32_t)(seed & 0xFFFFFFFFu), k1 = (uint32_t)(seed >> 32), ns = (uint32_t)(ng / L);
    if (fp64)
        k_sigma_accum_xi<double><<<grid, 256, 0, st>>>(zeta, phi, Uxi, u_ss, j, n_steps, n_xi, K, L, ns, k0, k1, stream,
                                                       sample0, c, ng, partial);
    else
        k_sigma_accum_xi<float><<<grid, 256, 0, st>>>(zeta, phi, Uxi, u_ss, j, n_steps, n_xi, K, L, ns, k0, k1, stream,
                                                      sample0, c, ng, partial);
}

// sigma[s][n + j] = dV S+ ; sigma[s][n - j] = -dV S- ; sigma[s][n] = (dV S+ - dV S-)/2 at j = 0.
// The cross-block sums run in the accumulation precision, one warp to a time (one thread to a time waited
// for 128 loads in turn: 37 us at 13 times, now 5).
constexpr int SR_RED_NT = 128;
template <typename T>
__global__ void __launch_bounds__(SR_RED_NT)
k_sigma_reduce(const double2* __restrict__ partial, int n_samples, int n_steps, int nblk, double dV,
               double2* __restrict__ sigma) {
    const int t = (int)((blockIdx.x * (int64_t)SR_RED_NT + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (t >= n_samples * (n_steps + 1)) return;
    const int s = t / (n_steps + 1), j = t % (n_steps + 1);
    T r[4] = {0, 0, 0, 0};
    for (int b = lane; b < nblk; b += 32) {
        const double2 p = partial[(size_t)t * 2 * nblk + b], m = partial[((size_t)t * 2 + 1) * nblk + b];
        r[0] += (T)p.x; r[1] += (T)p.y; r[2] += (T)m.x; r[3] += (T)m.y;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        for (int o = 16; o > 0; o >>= 1) r[k] += __shfl_xor_sync(0xffffffffu, r[k], o);
    if (lane != 0) return;
    double2* row = sigma + (size_t)s * (2 * n_steps + 1);
    const double2 sp = make_double2(dV * r[0], dV * r[1]);
    const double2 sm = make_double2(-dV * r[2], -dV * r[3]);
    if (j == 0) {
        row[n_steps] = make_double2(0.5 * (sp.x + sm.x), 0.5 * (sp.y + sm.y));
    } else {
        row[n_steps + j] = sp;
        row[n_steps - j] = sm;
    }
}

void launch_sigma_reduce(const double2* partial, int n_samples, int n_steps, int nblk, double dV, int fp64,
                            double* sigma, cudaStream_t st) {
    const int64_t total = (int64_t)n_samples * (n_steps + 1);
    const unsigned blocks = (unsigned)((total * 32 + SR_RED_NT - 1) / SR_RED_NT);
    double2* out = reinterpret_cast<double2*>(sigma);
    if (fp64) k_sigma_reduce<double><<<blocks, SR_RED_NT, 0, st>>>(partial, n_samples, n_steps, nblk, dV, out);
    else k_sigma_reduce<float><<<blocks, SR_RED_NT, 0, st>>>(partial, n_samples, n_steps, nblk, dV, out);
}

// ------------------------------------------------------------------ time ordering
// u of one point is y_t = (1/M) sum_m X_|m| e^{-2 pi i t m / M} with X the length-M transform (e^{+}) of
// its real, causal, zero-padded u^R.  The real part of X is the transform of u^R's even part, so
//   Re y_0 = x_0, Re y_t = x_t / 2   (t > 0; the padding keeps t and -t apart),
// and the odd imaginary part, made even, gives
//   Im y_t = sum_j G(t, j) x_j, G(t, j) = (g(j + t) + g(j - t)) / M, g(n) = cot(pi n / M) for odd n, 0 for
// even n.  G couples times of opposite parity only, so the ordering of all points is two real matrix
// products with half the times each: 80 k multiply-adds per point at 400 steps, fewer operations than
// the point's three length-2048 transforms, in one pass over u^R and u and without their 9 KB of
// shared memory per point.  Bound by FP32 multiply-adds and the shared-memory reads that feed them.
// Measured at 64^3 points x 401 times: 4.72 ms by transforms, 1.24 ms (34 T multiply-add operations/s,
// 0.42 of the FP32 rate; smaller tiles of 7 or 10 rows a warp 1.42-1.50 ms, 4 rows 1.71).
// Sums run over chunks of CH terms whose totals are added up, which keeps the rounding below the
// transforms' (8e-8 against 1.0e-7 relative at 400 steps; one long sum would have 2.2e-7).
constexpr int TO_BK = 16, TO_BN = 128, TO_NT = 128, TO_STAGES = 3;
constexpr int TO_R = TO_NT / 32;     // a warp's lanes take 4 points each and share their rows
constexpr int TO_TM = 13;            // rows of a warp at most

// Row tiles: TO_R warps of TM rows each, held in TMP = TM rounded up to even slots.
struct ToShape {
    int tm, tiles, kpad;      // TM, row tiles per parity, padded K
};
static ToShape to_shape(int n_steps) {
    const int rows = n_steps / 2 + 1;                 // the even times; the odd ones are at most as many
    const int cand[] = {1, 2, 4, 7, 10, TO_TM};
    ToShape s;
    s.tiles = (rows + TO_R * TO_TM - 1) / (TO_R * TO_TM);
    s.tm = TO_TM;
    for (int c : cand)
        if (TO_R * c * s.tiles >= rows) {
            s.tm = c;
            break;
        }
    s.kpad = (rows + TO_BK - 1) / TO_BK * TO_BK;
    return s;
}
static int to_tmp(int tm) { return (tm + 1) & ~1; }

size_t time_order_matrix_bytes(int n_steps) {
    const ToShape s = to_shape(n_steps);
    return sizeof(float2) * 2 * (size_t)s.tiles * s.kpad * TO_R * to_tmp(s.tm);
}

// G in the order the product reads it, each value twice (the packed multiply-adds take pairs):
// [parity of t][tile][k][warp][slot], row t = 2 (TO_R TM tile + TM warp + slot) + parity, column
// j = 2 k + 1 - parity; 0 outside the times.  A block has TO_BK columns of a tile, whose j + t and j - t
// take as many values as it has rows and columns: so many FP64 cotangents it computes.
__global__ void __launch_bounds__(TO_NT)
k_time_order_matrix(int n_steps, int M, int tm, int tmp, int tiles, int kpad, float2* __restrict__ G) {
    __shared__ double cs[TO_R * TO_TM + TO_BK], cd[TO_R * TO_TM + TO_BK];        // cot(pi (j + t) / M), cot(pi (j - t) / M)
    const int nk = kpad / TO_BK, k0 = (int)(blockIdx.x % nk) * TO_BK, tile = (int)(blockIdx.x / nk) % tiles;
    const int par = (int)(blockIdx.x / nk) / tiles, R = TO_R * tm, r0 = R * tile;
    for (int i = threadIdx.x; i < R + TO_BK - 1; i += TO_NT) {
        const double a = (double)(2 * (k0 + r0 + i) + 1) / M, b = (double)(2 * (k0 - r0 + i - (R - 1)) + 1 - 2 * par) / M;
        cs[i] = cospi(a) / sinpi(a);                                             // j + t and j - t are odd
        cd[i] = cospi(b) / sinpi(b);
    }
    __syncthreads();
    float2* g = G + (((size_t)par * tiles + tile) * kpad + k0) * TO_R * tmp;
    for (int i = threadIdx.x; i < TO_BK * TO_R * tmp; i += TO_NT) {
        const int slot = i % tmp, r = tm * (i / tmp % TO_R) + slot, q = i / (TO_R * tmp);
        const bool in = slot < tm && 2 * (r0 + r) + par <= n_steps && 2 * (k0 + q) + 1 - par <= n_steps;
        const float v = in ? (float)((cs[q + r] + cd[q - r + R - 1]) / M) : 0.f;
        g[i] = make_float2(v, v);
    }
}

__device__ __forceinline__ void to_cp(void* smem, const void* gmem, int bytes, int valid) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    if (bytes == 16) asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(gmem), "r"(valid) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(s), "l"(gmem), "r"(valid) : "memory");
}
// Pairs of floats in 64-bit registers, for the packed operations (one instruction issued for two)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
}

// One (parity, row tile) of 128 points of a sample.  Warp tm: rows TM tm .. + TM, of which the block takes TS (all,
// or an even number of slots: a tile has NSUB blocks then); lane tn: points 4 tn .. + 4.
// VEC: rows of u^R and u start on 16 bytes (the number of points is a multiple of 4).  G may be the matrix of more
// steps, which has a parity every g_par elements and a tile every g_tile of it; K is padded to kpad here.
template <int TM, int TS, bool VEC>
__global__ void __launch_bounds__(TO_NT, 3)
k_time_order(int64_t np, const float* __restrict__ uR, float2* __restrict__ u, int n_steps, int tiles, int kpad, int ch,
             const float2* __restrict__ G, int g_par, int g_tile) {
    constexpr int TMP = (TM + 1) & ~1, NSUB = (TM + TS - 1) / TS, TSP = (TS + 1) & ~1, AM = TO_R * TSP;
    static_assert(NSUB == 1 || TS % 2 == 0, "slots are copied in pairs");
    extern __shared__ __align__(16) unsigned char to_sm[];
    float2* As = reinterpret_cast<float2*>(to_sm);                                  // [stage][k][TO_R][TSP]
    float* Bs = reinterpret_cast<float*>(As + TO_STAGES * TO_BK * AM);              // [stage][k][TO_BN]
    // the blocks of one group of points run together: they read the same rows of u^R
    const int which = blockIdx.x / NSUB % (2 * tiles), par = which / tiles, tile = which % tiles;
    const int slot0 = TS * (blockIdx.x % NSUB);
    const int64_t p0 = (int64_t)(blockIdx.x / (2 * NSUB * tiles)) * TO_BN;
    const size_t row0 = (size_t)blockIdx.y * (n_steps + 1);
    const int tn = threadIdx.x % 32, tm = threadIdx.x / 32;
    const float2* A = G + (par * g_par + tile * g_tile) + slot0;
    const int nk = kpad / TO_BK;
    const auto load = [&](int s, int kt) {
        const float2* a = A + (size_t)kt * TO_BK * TO_R * TMP;
        float2* as = As + s * TO_BK * AM;
        for (int i = threadIdx.x; i < TO_BK * AM / 2; i += TO_NT) {
            if constexpr (NSUB == 1) {
                to_cp(as + 2 * i, a + 2 * i, 16, 16);
            } else {
                const int row = i / (TSP / 2), slot = i % (TSP / 2) * 2;
                const bool ok = slot0 + slot < TMP;
                to_cp(as + 2 * i, ok ? a + row * TMP + slot : a, 16, ok ? 16 : 0);
            }
        }
        float* bs = Bs + s * TO_BK * TO_BN;
        constexpr int V = VEC ? 4 : 1;
        for (int i = threadIdx.x; i < TO_BK * TO_BN / V; i += TO_NT) {
            const int k = i / (TO_BN / V), p = i % (TO_BN / V) * V;
            const int j = 2 * (kt * TO_BK + k) + 1 - par;
            const bool ok = j <= n_steps && p0 + p < np;
            to_cp(bs + k * TO_BN + p, ok ? uR + (row0 + j) * np + p0 + p : uR, 4 * V, ok ? 4 * V : 0);
        }
    };
    f32x2 acc[TS][2], tot[TS][2];
#pragma unroll
    for (int i = 0; i < TS; ++i) acc[i][0] = acc[i][1] = tot[i][0] = tot[i][1] = 0ull;
#pragma unroll
    for (int s = 0; s < TO_STAGES - 1; ++s) {
        if (s < nk) load(s, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int kt = 0; kt < nk; ++kt) {
        asm volatile("cp.async.wait_group %0;" ::"n"(TO_STAGES - 2) : "memory");
        __syncthreads();                                  // stage kt has landed; stage kt - 1 is free
        if (kt + TO_STAGES - 1 < nk) load((kt + TO_STAGES - 1) % TO_STAGES, kt + TO_STAGES - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const ulonglong2* as = reinterpret_cast<const ulonglong2*>(As + (kt % TO_STAGES) * TO_BK * AM + tm * TSP);
        const float* bs = Bs + (kt % TO_STAGES) * TO_BK * TO_BN + 4 * tn;
#pragma unroll
        for (int k = 0; k < TO_BK; ++k) {
            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(bs + k * TO_BN);
#pragma unroll
            for (int i = 0; i < TSP / 2; ++i) {
                const ulonglong2 a = as[k * (AM / 2) + i];
                acc[2 * i][0] = fma2(a.x, b.x, acc[2 * i][0]);
                acc[2 * i][1] = fma2(a.x, b.y, acc[2 * i][1]);
                if (2 * i + 1 < TS) {
                    acc[(2 * i + 1) % TS][0] = fma2(a.y, b.x, acc[(2 * i + 1) % TS][0]);
                    acc[(2 * i + 1) % TS][1] = fma2(a.y, b.y, acc[(2 * i + 1) % TS][1]);
                }
            }
        }
        if (((kt + 1) * TO_BK) % ch == 0) {
#pragma unroll
            for (int i = 0; i < TS; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    tot[i][h] = add2(tot[i][h], acc[i][h]);
                    acc[i][h] = 0ull;
                }
        }
    }
    const int64_t p = p0 + 4 * tn;
#pragma unroll
    for (int i = 0; i < TS; ++i) {
        const int t = 2 * (TO_R * TM * tile + TM * tm + slot0 + i) + par;
        if (t > n_steps || p >= np || (NSUB > 1 && slot0 + i >= TM)) continue;
        const float* x = uR + (row0 + t) * np + p;
        float2* y = u + (row0 + t) * np + p;
        const float half = t == 0 ? 1.f : 0.5f;
        const float2 i0 = unpack2(add2(tot[i][0], acc[i][0])), i1 = unpack2(add2(tot[i][1], acc[i][1]));
        const float im[4] = {i0.x, i0.y, i1.x, i1.y};
        if constexpr (VEC) {
            const float4 r = __ldg(reinterpret_cast<const float4*>(x));
            reinterpret_cast<float4*>(y)[0] = make_float4(half * r.x, im[0], half * r.y, im[1]);
            reinterpret_cast<float4*>(y)[1] = make_float4(half * r.z, im[2], half * r.w, im[3]);
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (p + q < np) y[q] = make_float2(half * __ldg(x + q), im[q]);
        }
    }
}

template <int TM, int TS, bool VEC>
static void tlaunch(int64_t np, const float* uR, float2* u, int n_samples, int n_steps, int tiles, const ToShape& g,
                    const float2* G, cudaStream_t st) {
    constexpr int TMP = (TM + 1) & ~1, TSP = (TS + 1) & ~1, NSUB = (TM + TS - 1) / TS;
    const size_t smem = TO_STAGES * TO_BK * (sizeof(float2) * TO_R * TSP + sizeof(float) * TO_BN);
    const dim3 grid((unsigned)(2 * NSUB * tiles * ((np + TO_BN - 1) / TO_BN)), n_samples);
    const int kpad = (n_steps / 2 + TO_BK) / TO_BK * TO_BK;
    // chunks of 16 terms, 32 above 256: as many chunks as terms in one, about
    const int ch = kpad > 256 ? 2 * TO_BK : TO_BK;
    const int g_tile = g.kpad * TO_R * TMP, g_par = g.tiles * g_tile;
    cudaFuncSetAttribute(k_time_order<TM, TS, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_time_order<TM, TS, VEC><<<grid, TO_NT, smem, st>>>(np, uR, u, n_steps, tiles, kpad, ch, G, g_par, g_tile);
}
// Few points leave most of the chip idle: below a tile to every other SM a block takes four of its warps' TM rows.
// (100 steps of 1000 points, 16 tiles: 11.0 -> 6.9 us; 400 of 1000, 64: 22.9 -> 17.1; 400 of 2000, 128: 22.9 with
// whole tiles, 27.5 so.)
template <int TM> static void tlaunch(int64_t np, const float* uR, float2* u, int n_samples, int n_steps, const ToShape& g,
                                      const float2* G, cudaStream_t st) {
    constexpr int TS = TM > 4 ? 4 : TM;
    const int tiles = (n_steps / 2 + TO_R * TM) / (TO_R * TM);
    const bool few = 2 * tiles * ((np + TO_BN - 1) / TO_BN) * n_samples < 76;
    if (np % 4 == 0) few ? tlaunch<TM, TS, true>(np, uR, u, n_samples, n_steps, tiles, g, G, st)
                         : tlaunch<TM, TM, true>(np, uR, u, n_samples, n_steps, tiles, g, G, st);
    else few ? tlaunch<TM, TS, false>(np, uR, u, n_samples, n_steps, tiles, g, G, st)
             : tlaunch<TM, TM, false>(np, uR, u, n_samples, n_steps, tiles, g, G, st);
}

void launch_time_order_matrix(int n_steps, int M, float2* G, cudaStream_t st) {
    const ToShape s = to_shape(n_steps);
    k_time_order_matrix<<<2 * s.tiles * (s.kpad / TO_BK), TO_NT, 0, st>>>(n_steps, M, s.tm, to_tmp(s.tm), s.tiles, s.kpad, G);
}

void launch_time_order(int np, const float* uR, float2* u, int n_samples, int n_steps, const float2* G, int g_steps,
                       cudaStream_t st) {
    const ToShape s = to_shape(g_steps);
    switch (s.tm) {
        case 1: tlaunch<1>(np, uR, u, n_samples, n_steps, s, G, st); break;
        case 2: tlaunch<2>(np, uR, u, n_samples, n_steps, s, G, st); break;
        case 4: tlaunch<4>(np, uR, u, n_samples, n_steps, s, G, st); break;
        case 7: tlaunch<7>(np, uR, u, n_samples, n_steps, s, G, st); break;
        case 10: tlaunch<10>(np, uR, u, n_samples, n_steps, s, G, st); break;
        default: tlaunch<TO_TM>(np, uR, u, n_samples, n_steps, s, G, st); break;
    }
}

// ------------------------------------------------------------------ Sigma(omega) (Eq. 7)
template <typename T>
__device__ __forceinline__ void damped_term(const double2* __restrict__ sigma, int n_samples, int n_steps, int jj,
                                            double dt, double gamma, T& re, T& im, T& t) {
    // mean over samples of Sigma(t_j), times dt w_j e^{-gamma^2 t^2 / 2}
    double sx = 0, sy = 0;
    for (int s = 0; s < n_samples; ++s) {
        const double2 v = sigma[(size_t)s * (2 * n_steps + 1) + jj];
        sx += v.x;
        sy += v.y;
    }
    const int j = jj - n_steps;
    const T tj = (T)(dt * j);
    const T w = (jj == 0 || jj == 2 * n_steps) ? (T)0.5 : (T)1.0;
    const T damp = (T)dt * w * exp(-(T)0.5 * (T)gamma * (T)gamma * tj * tj) / (T)n_samples;
    re = (T)sx * damp;
    im = (T)sy * damp;
    t = tj;
}

template <typename T>
__global__ void k_sigma_omega(const double2* __restrict__ sigma, int n_samples, int n_steps, double dt, double gamma,
                              const double* __restrict__ omega, int n_omega, double2* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_omega) return;
    const T w = (T)omega[i];
    T ax = 0, ay = 0;
    for (int jj = 0; jj <= 2 * n_steps; ++jj) {
        T re, im, t;
        damped_term<T>(sigma, n_samples, n_steps, jj, dt, gamma, re, im, t);
        T sn, cs;
        sincos(w * t, &sn, &cs);
        ax += re * cs - im * sn;
        ay += re * sn + im * cs;
    }
    out[i] = make_double2((double)ax, (double)ay);
}

void launch_sigma_omega(const double* sigma, int n_samples, int n_steps, double dt, double gamma, const double* omega,
                        int n_omega, int fp64, double* out, cudaStream_t st) {
    if (n_omega == 0) return;
    const int blocks = (n_omega + 127) / 128;
    if (fp64)
        k_sigma_omega<double><<<blocks, 128, 0, st>>>(reinterpret_cast<const double2*>(sigma), n_samples, n_steps, dt,
                                                      gamma, omega, n_omega, reinterpret_cast<double2*>(out));
    else
        k_sigma_omega<float><<<blocks, 128, 0, st>>>(reinterpret_cast<const double2*>(sigma), n_samples, n_steps, dt,
                                                     gamma, omega, n_omega, reinterpret_cast<double2*>(out));
}

// ------------------------------------------------------------------ QP equation (Eq. 6)
// damped[jj] = mean_s Sigma_s(t_j) * dt w_j e^{-gamma^2 t_j^2/2}  (complex), jj = 0..2n
template <typename T>
__global__ void k_qp_damped(const double2* __restrict__ sigma, int n_samples, int n_steps, double dt, double gamma,
                            double2* __restrict__ damped) {
    const int jj = blockIdx.x * blockDim.x + threadIdx.x;
    if (jj > 2 * n_steps) return;
    T re, im, t;
    damped_term<T>(sigma, n_samples, n_steps, jj, dt, gamma, re, im, t);
    damped[jj] = make_double2((double)re, (double)im);
}

// Re Sigma(w) over the times +-dt j, j = j0, j0 + js, ...: a pair has one sine and cosine.
template <typename T>
__device__ __forceinline__ T re_sigma_at(const double2* __restrict__ damped, int n_steps, double dt, T w, int j0, int js) {
    T acc = 0;
    for (int j = j0; j <= n_steps; j += js) {
        const T t = (T)(dt * j);
        T sn, cs;
        sincos(w * t, &sn, &cs);
        const double2 p = damped[n_steps + j], m = damped[n_steps - j];
        acc += (T)p.x * cs - (T)p.y * sn;
        if (j > 0) acc += (T)m.x * cs + (T)m.y * sn;
    }
    return acc;
}

// scan[i] = f(w_i) = w_i - eps - X - Re Sigma(w_i) + vxc, w_i = eps - window + i step.  Bound by the latency
// and then the rate of FP64 sines: QP_SCAN_L lanes share a point's times, in blocks of one warp, so that every
// SM has some (4001 points x 25 times: 31 us with one thread to a point in 32 blocks, now 9.6).
constexpr int QP_SCAN_L = 4, QP_SCAN_P = 32 / QP_SCAN_L;
template <typename T>
__global__ void __launch_bounds__(32)
k_qp_scan(const double2* __restrict__ damped, int n_steps, double dt, double eps, const double* __restrict__ x,
          int n_samples, double vxc, double window, double step, int n_scan, double* __restrict__ scan) {
    const int i = blockIdx.x * QP_SCAN_P + threadIdx.x / QP_SCAN_L;
    const double w = eps - window + step * i;
    double r = (double)re_sigma_at<T>(damped, n_steps, dt, (T)w, threadIdx.x % QP_SCAN_L, QP_SCAN_L);
    for (int o = QP_SCAN_L / 2; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (i >= n_scan || threadIdx.x % QP_SCAN_L != 0) return;
    double xm = 0.0;
#pragma unroll 8
    for (int s = 0; s < n_samples; ++s) xm += x[s];
    xm /= n_samples;
    scan[i] = w - eps - xm - r + vxc;
}

// Re Sigma(w) by the block: one barrier, the warps' sums in two halves of sh[2 * 8] in turn
constexpr int QP_NT = 256;
template <typename T>
__device__ __forceinline__ double block_re_sigma(const double2* damped, int n_steps, double dt, double w, double* sh,
                                                 int& turn) {
    double v = (double)re_sigma_at<T>(damped, n_steps, dt, (T)w, threadIdx.x, QP_NT);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    double* h = sh + (turn ^= QP_NT / 32);
    if ((threadIdx.x & 31) == 0) h[threadIdx.x >> 5] = v;
    __syncthreads();
    double r = 0.0;
#pragma unroll
    for (int i = 0; i < QP_NT / 32; ++i) r += h[i];
    return r;
}

// One block: bracket nearest eps, bisection to 1e-10, standard error with the Z factor.  It is a chain of
// some 30 sums over the times, so what counts is the latency of each: the bracket is searched by all
// threads (one thread walking the 4001 points of the default scan took most of 1417 us at 25 times;
// now 93 us in all), a sum has one barrier, and the samples of the standard error go to the warps.
// result = (eps_qp, se, Re Sigma(eps_qp), Z); all NaN: no root.
template <typename T>
__global__ void __launch_bounds__(QP_NT)
k_qp_solve(const double2* __restrict__ sigma, const double* __restrict__ x, const double2* __restrict__ damped,
           int n_samples, int n_steps, double dt, double gamma, double eps, double vxc, double window, double step,
           const double* __restrict__ scan, int n_scan, double* __restrict__ result) {
    constexpr int NW = QP_NT / 32;
    __shared__ double sh[2 * NW], bds[NW], xm_s;
    __shared__ int bis[NW];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        double xs = 0;
#pragma unroll 8
        for (int s = 0; s < n_samples; ++s) xs += x[s];
        xm_s = xs / n_samples;
    }
    // bracket whose midpoint is nearest eps (first on ties)
    int best = -1;
    double bd = 1e300;
#pragma unroll 4
    for (int i = threadIdx.x; i < n_scan - 1; i += QP_NT) {
        const double a = scan[i], b = scan[i + 1];
        const int sa = (a > 0) - (a < 0), sb = (b > 0) - (b < 0);
        if (sa * sb <= 0) {
            const double mid = 0.5 * ((eps - window + step * i) + (eps - window + step * (i + 1)));
            const double d = fabs(mid - eps);
            if (d < bd) { bd = d; best = i; }
        }
    }
    auto nearer = [&](double d, int i) {
        if (i >= 0 && (best < 0 || d < bd || (d == bd && i < best))) { bd = d; best = i; }
    };
    for (int o = 16; o > 0; o >>= 1) {
        const double d = __shfl_xor_sync(0xffffffffu, bd, o);
        const int i = __shfl_xor_sync(0xffffffffu, best, o);
        nearer(d, i);
    }
    if (lane == 0) { bds[warp] = bd; bis[warp] = best; }
    __syncthreads();
    best = -1;
    bd = 1e300;
    for (int i = 0; i < NW; ++i) nearer(bds[i], bis[i]);
    if (best < 0) {
        if (threadIdx.x == 0) { result[0] = nan(""); result[1] = nan(""); result[2] = nan(""); result[3] = nan(""); }
        return;
    }
    const double xm = xm_s;
    int turn = 0;
    double a = eps - window + step * best, b = eps - window + step * (best + 1);
    double fa = scan[best];
    while (b - a > 1e-10) {
        const double c = 0.5 * (a + b);
        const double fc = c - eps - xm - block_re_sigma<T>(damped, n_steps, dt, c, sh, turn) + vxc;
        const int sfc = (fc > 0) - (fc < 0), sfa = (fa > 0) - (fa < 0);
        if (sfc == sfa && fc != 0.0) { a = c; fa = fc; }
        else b = c;
    }
    const double e = 0.5 * (a + b);
    const double rs = block_re_sigma<T>(damped, n_steps, dt, e, sh, turn);
    const double d = 1e-4;
    const double slope = (block_re_sigma<T>(damped, n_steps, dt, e + d, sh, turn) -
                          block_re_sigma<T>(damped, n_steps, dt, e - d, sh, turn)) / (2 * d);
    const double z = 1.0 / (1.0 - slope);
    // per-sample X_i + Re Sigma_i(e): Sigma_i(t) damped the same way (no sample mean)
    double m1 = 0, m2 = 0;
    for (int s = warp; s < n_samples; s += NW) {
        double acc = 0;
        for (int jj = lane; jj <= 2 * n_steps; jj += 32) {
            const int j = jj - n_steps;
            const T t = (T)(dt * j);
            const T w = (jj == 0 || jj == 2 * n_steps) ? (T)0.5 : (T)1.0;
            const T damp = (T)dt * w * exp(-(T)0.5 * (T)gamma * (T)gamma * t * t);
            const double2 v = sigma[(size_t)s * (2 * n_steps + 1) + jj];
            T sn, cs;
            sincos((T)e * t, &sn, &cs);
            acc += (double)(((T)v.x * cs - (T)v.y * sn) * damp);
        }
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const double per = x[s] + acc;
        m1 += per;
        m2 += per * per;
    }
    __syncthreads();
    if (lane == 0) { sh[warp] = m1; sh[NW + warp] = m2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        m1 = m2 = 0;
        for (int i = 0; i < NW; ++i) { m1 += sh[i]; m2 += sh[NW + i]; }
        double se = nan("");
        if (n_samples > 1) {
            const double mean = m1 / n_samples;
            const double var = (m2 - n_samples * mean * mean) / (n_samples - 1);
            se = fabs(z) * sqrt(fmax(var, 0.0) / n_samples);
        }
        result[0] = e;
        result[1] = se;
        result[2] = rs;
        result[3] = z;
    }
}

void launch_qp(const double* sigma, const double* x, int n_samples, int n_steps, double dt, double gamma, double eps_ks,
               double vxc, double window, double step, int fp64, double* scan, int n_scan, double* result,
               cudaStream_t st) {
    // scan[] holds n_scan doubles followed by the 2 n_steps + 1 damped complex terms
    double2* damped = reinterpret_cast<double2*>(scan + ((n_scan + 1) & ~1));
    const double2* sg = reinterpret_cast<const double2*>(sigma);
    const int nt = 2 * n_steps + 1;
    if (fp64) {
        k_qp_damped<double><<<(nt + 127) / 128, 128, 0, st>>>(sg, n_samples, n_steps, dt, gamma, damped);
        k_qp_scan<double><<<(n_scan + QP_SCAN_P - 1) / QP_SCAN_P, 32, 0, st>>>(damped, n_steps, dt, eps_ks, x, n_samples, vxc, window,
                                                              step, n_scan, scan);
        k_qp_solve<double><<<1, QP_NT, 0, st>>>(sg, x, damped, n_samples, n_steps, dt, gamma, eps_ks, vxc, window, step,
                                              scan, n_scan, result);
    } else {
        k_qp_damped<float><<<(nt + 127) / 128, 128, 0, st>>>(sg, n_samples, n_steps, dt, gamma, damped);
        k_qp_scan<float><<<(n_scan + QP_SCAN_P - 1) / QP_SCAN_P, 32, 0, st>>>(damped, n_steps, dt, eps_ks, x, n_samples, vxc, window,
                                                             step, n_scan, scan);
        k_qp_solve<float><<<1, QP_NT, 0, st>>>(sg, x, damped, n_samples, n_steps, dt, gamma, eps_ks, vxc, window, step,
                                             scan, n_scan, result);
    }
}

}  // namespace sgw

// ------------------------------------------------------------------ QP solve without allocation
// Some callers cannot let a library allocate device memory at all: a host application that has
// reserved the device's memory for its own pool allocator, or a plugin host that forbids
// allocations while it runs, would see cudaMalloc fail or have its memory accounting broken.
// For them sgw_qp_energy_noalloc runs the QP solve with its scratch in this fixed, statically
// sized device array instead of a context work area.  Every GPU that loads the library holds
// the array until the process exits.
namespace {
constexpr int kQpScratchDoubles = 131072;   // 1 MiB
static __device__ __align__(256) double g_qp_scratch[kQpScratchDoubles];

// Device address of g_qp_scratch on each device, looked up once per device with that device
// current (the host-side name is only a stand-in, not a device address).
constexpr int kMaxDevices = 64;
double* g_qp_scratch_dev[kMaxDevices] = {nullptr};
std::mutex g_qp_scratch_mu;
}  // namespace

extern "C" sgw_status sgw_qp_energy_noalloc(const double* sigma_dev, const double* x_dev, int n_samples,
                                            int n_steps, double dt, double gamma, double eps_ks, double vxc,
                                            double window, double step, int fp64, double* result_host,
                                            void* stream) {
    if (n_samples < 1 || n_steps < 0 || !(window > 0) || !(step > 0) || !sigma_dev || !x_dev || !result_host) {
        sgw::set_global_error("sgw_qp_energy_noalloc: bad arguments");
        return SGW_EINVAL;
    }
    // the scan size is checked as a double first: a huge window or a tiny step would overflow the
    // integer conversion
    const double r = 2.0 * window / step;
    if (!std::isfinite(r) || r + 1.0 > (double)kQpScratchDoubles) {
        sgw::set_global_error("sgw_qp_energy_noalloc: 2 window/step + 1 scan points exceed the 1 MiB static scratch "
                              "(131072 doubles)");
        return SGW_EINVAL;
    }
    const long long n_scan = std::llround(r) + 1;
    const long long need = ((n_scan + 1) & ~1LL) + 2LL * (2LL * n_steps + 1) + 4;
    if (need > kQpScratchDoubles) {
        sgw::set_global_error("sgw_qp_energy_noalloc: window/step and n_steps need more than the 1 MiB static "
                              "scratch (even(2 window/step + 1) + 2 (2 n_steps + 1) + 4 <= 131072 doubles)");
        return SGW_EINVAL;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        sgw::set_global_error("sgw_qp_energy_noalloc: no usable current device");
        return SGW_ECUDA;
    }
    cudaStream_t st = (cudaStream_t)stream;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if ((e = cudaStreamIsCapturing(st, &cap)) != cudaSuccess) {
        sgw::set_global_error((std::string("sgw_qp_energy_noalloc: ") + cudaGetErrorString(e)).c_str());
        return SGW_ECUDA;
    }
    double* scratch = nullptr;
    {
        // Outside a capture the address is looked up on every call (cheap), so a context that the
        // application reset and re-created gets the new one; during a capture the address cached
        // by an earlier call on this device is used.
        std::lock_guard<std::mutex> lk(g_qp_scratch_mu);
        if (cap == cudaStreamCaptureStatusNone) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_qp_scratch);
            if (e != cudaSuccess || !p) {
                sgw::set_global_error((std::string("sgw_qp_energy_noalloc: cudaGetSymbolAddress: ") +
                                       cudaGetErrorString(e)).c_str());
                return SGW_ECUDA;
            }
            g_qp_scratch_dev[dev] = static_cast<double*>(p);
        } else if (!g_qp_scratch_dev[dev]) {
            sgw::set_global_error("sgw_qp_energy_noalloc: the first call on a device must come before any stream "
                                  "capture");
            return SGW_ESTATE;
        }
        scratch = g_qp_scratch_dev[dev];
    }
    // scan values, then the damped terms, then the 4 result doubles; every element read in
    // this call is written first in this call, so nothing needs clearing between calls.
    double* result = scratch + (need - 4);
    sgw::launch_qp(sigma_dev, x_dev, n_samples, n_steps, dt, gamma, eps_ks, vxc, window, step, fp64, scratch,
                   (int)n_scan, result, st);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(result_host, result, 4 * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        sgw::set_global_error((std::string("sgw_qp_energy_noalloc: ") + cudaGetErrorString(e)).c_str());
        return SGW_ECUDA;
    }
    if (std::isnan(result_host[0])) {
        sgw::set_global_error("sgw_qp_energy_noalloc: no sign change of the QP equation in the window");
        return SGW_ENOCONV;
    }
    return SGW_OK;
}
