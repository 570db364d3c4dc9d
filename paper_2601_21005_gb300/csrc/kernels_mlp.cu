// Learned control variate: features of a sample's random vector, a 4-layer MLP trained and
// evaluated on the GPU (BF16 operands on the tensor cores, FP32 accumulate, FP32 master
// weights and Adam state), and the FP64 standardisation / control-variate rows.
//
// Network: h1 = tanh(x W1 + b1), h2 = tanh(h1 W2 + b2), h3 = tanh(h2 W3 + b3), y = h3 W4 + b4.
// Loss: mean over samples and outputs of (y - t)^2.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/sgw.h"
#include "dependent_launch.cuh"
#include "fft_smem.cuh"
#include "sgw_internal.cuh"

namespace sgw {

// ------------------------------------------------------------------ BF16 tensor-core GEMM
// C[m][n] = sum_k A(m, k) B(k, n),  A(m, k) = TA ? A[k lda + m] : A[m lda + k],
//                                   B(k, n) = TB ? B[n ldb + k] : B[k ldb + n].
// The products are small (M <= some hundreds of rows, N and K 20 to 1603), so a call is a chain of
// short kernels and the latency of each is what counts.  A block has a TM x 64 tile (4 warps of
// TM/2 x 32, mma.m16n8k16); four K steps of 64 are in flight by cp.async, which for K <= 256 is the
// whole slab at once, and the weights' share of them is requested before the kernel waits for the one
// before it.  BF16 matrices have rows padded with zeros to multiples of 8 elements, so every copy is
// 16 bytes and only rows are checked.  Where the backward pass's dZ has a K of 384 and more and few tiles, its K is
// split over the blocks of a cluster: up to eight, as long as three steps of 64 are left to each on
// average (a rank has a whole number of them, the last ones fewer or none: 26 steps over 8 ranks are
// 4 4 4 4 4 4 2 0).  The partial tiles are summed in rank order through distributed shared memory.
// 148-256-256-256-1603, gradients of 32 rows and the forward of 512: 292 and 92 us per call with 64 x 64
// tiles, one scalar load per element and a kernel for each sum; now 53 and 25.
enum { EPI_STORE = 0, EPI_BIAS_TANH = 1, EPI_BIAS = 2, EPI_DTANH = 3, EPI_LOSS = 4 };

struct GemmEpi {
    int mode;
    const float* bias;      // [N] (EPI_BIAS*, EPI_LOSS)
    float* out;             // [M][ldo] fp32 result (pre-activation for EPI_BIAS_TANH, dZ for EPI_DTANH, dY for
    int64_t ldo;            //  EPI_LOSS); null for a pre-activation nothing reads
    __nv_bfloat16* out_bf;  // [M][ldb] bf16 copy of tanh(z) (BIAS_TANH) or of out (DTANH, LOSS)
    int ldb;
    const float* aux;       // [M][ldo] the pre-activation whose tanh' multiplies (DTANH), or the targets (LOSS)
    const float* w;         // [N] loss weights (LOSS), null: all 1
    float scale;            // LOSS: out = scale w (y - aux)
    float* y;               // [M][ldo] the output itself (LOSS)
};

struct Gemm {
    int M, N, K;
    const __nv_bfloat16* A;
    int lda;
    const __nv_bfloat16* B;
    int ldb;
    GemmEpi ep;
};

constexpr int GN = 64, GK = 64, GS = 4, G_NT = 128;
template <int TM> struct GemmCfg {
    static constexpr int A_EL = TM * (GK + 8) > GK * (TM + 8) ? TM * (GK + 8) : GK * (TM + 8);
    static constexpr int ST_EL = A_EL + GK * (GN + 8);                 // bf16 elements of one stage
    static constexpr int SMEM = 2 * ST_EL * GS;
    static_assert(4 * TM * (GN + 4) <= SMEM, "the split's partial tile fits in the stages");
};

int64_t gemm_tiles(int tm, int M, int N) { return ((M + tm - 1) / tm) * (int64_t)((N + GN - 1) / GN); }

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ float ldf_written(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
template <bool TRANS>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    if (TRANS)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
    else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// One K step of an operand into shared memory: R x C elements at (r0, c0) of a row-major matrix of `rows`
// rows and a padded row length ld.
template <int R, int C>
__device__ __forceinline__ void gemm_stage(uint32_t dst, const __nv_bfloat16* src, int ld, int rows, int r0, int c0) {
    static_assert(R * C / 8 % G_NT == 0, "whole passes");
#pragma unroll
    for (int i = 0; i < R * C / 8 / G_NT; ++i) {
        const int e = threadIdx.x + i * G_NT, r = e / (C / 8), c = e % (C / 8) * 8;
        const bool ok = r0 + r < rows && c0 + c < ld;
        cp16(dst + 2 * (r * (C + 8) + c), ok ? src + (size_t)(r0 + r) * ld + c0 + c : src, ok);
    }
}

__device__ __forceinline__ void gemm_finish(const GemmEpi& ep, int row, int col, float v, float aux) {
    const size_t o = (size_t)row * ep.ldo + col;
    if (ep.mode == EPI_STORE) {
        ep.out[o] = v;
    } else if (ep.mode == EPI_BIAS_TANH) {
        v += ep.bias[col];
        if (ep.out) ep.out[o] = v;
        ep.out_bf[(size_t)row * ep.ldb + col] = __float2bfloat16(tanhf(v));
    } else if (ep.mode == EPI_BIAS) {
        ep.out[o] = v + ep.bias[col];
    } else if (ep.mode == EPI_DTANH) {
        const float th = tanhf(aux);
        v *= 1.f - th * th;
        ep.out[o] = v;
        ep.out_bf[(size_t)row * ep.ldb + col] = __float2bfloat16(v);
    } else {
        v += ep.bias[col];
        ep.y[o] = v;
        v = ep.scale * (ep.w ? ep.w[col] : 1.f) * (v - aux);
        ep.out[o] = v;
        ep.out_bf[(size_t)row * ep.ldb + col] = __float2bfloat16(v);
    }
}

// One tile of a product, by a block that is rank `rank` of `splits` for it.  WEIGHTS: B was written
// before the kernel directly before this one started.
template <int TM, int TA, int TB, bool WEIGHTS>
__device__ __forceinline__ void gemm_tile(const Gemm& g, int64_t tile, int rank, int splits) {
    extern __shared__ __align__(16) __nv_bfloat16 gsm[];
    typedef GemmCfg<TM> C;
    constexpr int MT = TM / 32;                                        // m16 tiles of a warp
    constexpr int LA = TA ? TM + 8 : GK + 8, LB = TB ? GK + 8 : GN + 8;
    const int nt = (g.N + GN - 1) / GN;
    const int m0 = (int)(tile / nt) * TM, n0 = (int)(tile % nt) * GN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * (TM / 2), wn = (warp & 1) * 32;
    const int chunk = ((g.K + GK - 1) / GK + splits - 1) / splits;
    const int s0 = min(rank * chunk, (g.K + GK - 1) / GK);
    const int steps = min(chunk, (g.K + GK - 1) / GK - s0);
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(gsm);
    auto stage_a = [&](int s) {
        const uint32_t d = base + 2 * C::ST_EL * (s % GS);
        const int k0 = (s0 + s) * GK;
        if (TA) gemm_stage<GK, TM>(d, g.A, g.lda, g.K, k0, m0);
        else gemm_stage<TM, GK>(d, g.A, g.lda, g.M, m0, k0);
    };
    auto stage_b = [&](int s) {
        const uint32_t d = base + 2 * C::ST_EL * (s % GS) + 2 * C::A_EL;
        const int k0 = (s0 + s) * GK;
        if (TB) gemm_stage<GN, GK>(d, g.B, g.ldb, g.N, n0, k0);
        else gemm_stage<GK, GN>(d, g.B, g.ldb, g.K, k0, n0);
    };
    if (WEIGHTS)
        for (int s = 0; s < min(GS, steps); ++s) stage_b(s);
    dependents_wait();
    dependents_launch();
    // the stages' groups are committed in order; B of the first GS, if early, belongs to the first group
#pragma unroll
    for (int s = 0; s < GS; ++s) {
        if (s < steps) {
            stage_a(s);
            if (!WEIGHTS) stage_b(s);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // the epilogue's operands, requested ahead
    const bool with_aux = g.ep.mode == EPI_DTANH || g.ep.mode == EPI_LOSS;
    float aux[MT][4][4];
    if (with_aux && splits == 1) {
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int row = m0 + wm + 16 * i + (lane >> 2) + (r >= 2 ? 8 : 0);
                    const int col = n0 + wn + 8 * j + 2 * (lane & 3) + (r & 1);
                    aux[i][j][r] = row < g.M && col < g.N ? ldf_written(g.ep.aux + (size_t)row * g.ep.ldo + col) : 0.f;
                }
    }
    float acc[MT][4][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int r = 0; r < 4; ++r) acc[i][j][r] = 0.f;
    for (int s = 0; s < steps; ++s) {
        asm volatile("cp.async.wait_group %0;" ::"n"(GS - 1) : "memory");
        __syncthreads();
        const uint32_t sa = base + 2 * C::ST_EL * (s % GS), sb = sa + 2 * C::A_EL;
#pragma unroll
        for (int ks = 0; ks < GK; ks += 16) {
            uint32_t af[MT][4], bf[2][4];
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                const int m = wm + 16 * i;
                if (TA) ldsm4<true>(af[i], sa + 2 * ((ks + (lane & 7) + (lane >> 4) * 8) * LA + m + (lane >> 3 & 1) * 8));
                else ldsm4<false>(af[i], sa + 2 * ((m + (lane & 15)) * LA + ks + (lane >> 4) * 8));
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int n = wn + 16 * j;
                if (TB) ldsm4<false>(bf[j], sb + 2 * ((n + (lane & 7) + (lane >> 4) * 8) * LB + ks + (lane >> 3 & 1) * 8));
                else ldsm4<true>(bf[j], sb + 2 * ((ks + (lane & 15)) * LB + n + (lane >> 4) * 8));
            }
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float* c = acc[i][j];
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                        "{%8,%9}, {%0,%1,%2,%3};\n"
                        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                        : "r"(af[i][0]), "r"(af[i][1]), "r"(af[i][2]), "r"(af[i][3]), "r"(bf[j >> 1][2 * (j & 1)]),
                          "r"(bf[j >> 1][2 * (j & 1) + 1]));
                }
        }
        __syncthreads();
        if (s + GS < steps) {
            stage_a(s + GS);
            stage_b(s + GS);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (splits == 1) {
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int row = m0 + wm + 16 * i + (lane >> 2) + (r >= 2 ? 8 : 0);
                    const int col = n0 + wn + 8 * j + 2 * (lane & 3) + (r & 1);
                    if (row < g.M && col < g.N) gemm_finish(g.ep, row, col, acc[i][j][r], aux[i][j][r]);
                }
    } else {
        constexpr int LP = GN + 4;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        float* part = reinterpret_cast<float*>(gsm);
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int r = 0; r < 4; r += 2)
                    *reinterpret_cast<float2*>(part + (wm + 16 * i + (lane >> 2) + 4 * r) * LP + wn + 8 * j + 2 * (lane & 3)) =
                        make_float2(acc[i][j][r], acc[i][j][r + 1]);
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        for (int e = rank * (TM * GN / splits) + threadIdx.x; e < (rank + 1) * (TM * GN / splits); e += G_NT) {
            const int r = e / GN, c = e % GN;
            const uint32_t at = base + 4 * (r * LP + c);
            float v = 0.f;
            for (int q = 0; q < splits; ++q) {
                uint32_t ra;
                float p;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(at), "r"(q));
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(p) : "r"(ra) : "memory");
                v += p;
            }
            if (m0 + r < g.M && n0 + c < g.N)
                gemm_finish(g.ep, m0 + r, n0 + c, v,
                            with_aux ? ldf_written(g.ep.aux + (size_t)(m0 + r) * g.ep.ldo + n0 + c) : 0.f);
        }
        // no block leaves while another may still read its partial tile
        asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// a layer's forward product
template <int TM>
__global__ void __launch_bounds__(G_NT) k_mlp_forward(Gemm g) {
    gemm_tile<TM, 0, 0, true>(g, blockIdx.x, 0, 1);
}

// out[n] = sum_m d[m][n] for 32 columns, fixed order: each warp a quarter of the rows in turn
__device__ __forceinline__ void colsum_block(int M, int N, int64_t ld, const float* d, float* out, int block) {
    __shared__ float sh[G_NT / 32][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n = block * 32 + lane;
    float s = 0.f;
    if (n < N) {
        int m = warp;
        for (; m + 28 < M; m += 32) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = ldf_written(d + (size_t)(m + 4 * i) * ld + n);
#pragma unroll
            for (int i = 0; i < 8; ++i) s += v[i];
        }
        for (; m < M; m += 4) s += ldf_written(d + (size_t)m * ld + n);
    }
    sh[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && n < N) out[n] = (sh[0][lane] + sh[1][lane]) + (sh[2][lane] + sh[3][lane]);
}

// The loss sum_o w_o (y - t)^2 in FP64 and a fixed order: partials loss[1 + block] in the launch that follows
// the output (its other blocks have more to do, and FP64 is slow), their sum in the one after it.
struct Loss {
    int64_t n;
    int O, blocks;
    const float *y, *t, *w;
    double* loss;
};

__device__ __forceinline__ void loss_block(const Loss& l, int block) {
    __shared__ double sh[G_NT / 32];
    double a = 0.0;
    for (int64_t i = block * (int64_t)G_NT + threadIdx.x; i < l.n; i += (int64_t)l.blocks * G_NT) {
        const float e = ldf_written(l.y + i) - l.t[i];
        const float wo = l.w ? l.w[i % l.O] : 1.f;
        a += (double)wo * e * e;
    }
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < G_NT / 32; ++i) s += sh[i];
        l.loss[1 + block] = s;
    }
}

__device__ __forceinline__ void loss_sum(const Loss& l) {
    if (threadIdx.x >= 32) return;
    double s = 0.0;
    for (int i = threadIdx.x; i < l.blocks; i += 32) s += *(const volatile double*)(l.loss + 1 + i);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) l.loss[0] = s;
}

// A layer's backward pass in one launch, all of it from dZ of the layer: the clusters of dZ of the layer
// below (d, absent for the first layer: d_tiles = 0) come first, then the blocks of dW, of the bias
// gradient and of the loss (partials after the last layer, their sum one launch later).
struct Backward {
    Gemm d, w;
    int64_t d_tiles, w_tiles;
    int splits, db_blocks, loss_blocks, loss_sums;
    const float* dz;
    float* db;
    int64_t ldz;
    Loss loss;
};

__global__ void __launch_bounds__(G_NT) k_mlp_backward(Backward b) {
    constexpr int TM = 32;
    int64_t i = blockIdx.x;
    if (i < b.d_tiles * b.splits) {
        gemm_tile<TM, 0, 1, true>(b.d, i / b.splits, (int)(i % b.splits), b.splits);
        return;
    }
    i -= b.d_tiles * b.splits;
    if (i < b.w_tiles) {
        gemm_tile<TM, 1, 0, false>(b.w, i, 0, 1);
        return;
    }
    i -= b.w_tiles;
    dependents_wait();
    dependents_launch();
    if (i < b.db_blocks) {
        colsum_block(b.w.K, b.w.N, b.ldz, b.dz, b.db, (int)i);
        return;
    }
    i -= b.db_blocks;
    if (i < b.loss_blocks) loss_block(b.loss, (int)i);
    else if (i == b.loss_blocks && b.loss_sums) loss_sum(b.loss);
}

// ------------------------------------------------------------------ small MLP kernels
// x [rows][cols] -> y [rows][ld] in BF16 (the columns beyond cols stay zero)
__global__ void k_mlp_input(int64_t n, int cols, int ld, const float* __restrict__ x, __nv_bfloat16* __restrict__ y) {
    dependents_launch();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i / cols * ld + i % cols] = __float2bfloat16(x[i]);
}

// Where the parameters of the layers start, and where the BF16 copy of each matrix lies, as a kernel over
// them all wants it: in rows, of which a block takes a piece of MLP_PC elements, MLP_U to a thread.  A matrix
// whose copy is padded has its rows and then the bias; one whose copy is not is a single row with the bias at
// its end.  Bound by the blocks' latency and L2 traffic: 64-1024-1024-1024-64 14.9 us with an element to a
// thread, 2000-64-64-64-64 6.7 with its short rows by themselves; with four and flat rows 10.4 and 4.3;
// 16-2048-2048-2048-16 59.5 -> 41 us, 148-256-256-256-1603 6.3 either way.
constexpr int MLP_NT = 256, MLP_U = 4, MLP_PC = MLP_NT * MLP_U;
struct MlpLayout {
    int64_t woff[4], poff[4], mat[4], first[5];     // mat: elements of the matrix; first: of the layer's blocks
    int len[4], ld[4], pieces[4];                   // len: of a row; ld: of the copy's; pieces: of a row
};

// The elements of this block: i, i + 1, .. below i + n (the first parameter's index), of which those before
// i + copied have a BF16 copy, from at on.
struct MlpPiece {
    int64_t i, at;
    int n, copied;
};
__device__ __forceinline__ MlpPiece mlp_piece(const MlpLayout& L) {
    const int64_t b = blockIdx.x;
    int64_t first = L.first[0], woff = L.woff[0], poff = L.poff[0], mat = L.mat[0];
    int len = L.len[0], ld = L.ld[0], pieces = L.pieces[0];
#pragma unroll
    for (int l = 1; l < 4; ++l)
        if (b >= L.first[l]) {
            first = L.first[l]; woff = L.woff[l]; poff = L.poff[l]; mat = L.mat[l];
            len = L.len[l]; ld = L.ld[l]; pieces = L.pieces[l];
        }
    const unsigned u = (unsigned)(b - first), r = u / (unsigned)pieces;
    const int c = (int)(u - r * (unsigned)pieces) * MLP_PC;
    const int64_t k = (int64_t)r * len + c;
    MlpPiece p;
    p.i = woff + k;
    p.at = poff + (int64_t)r * ld + c;
    p.n = min(len - c, MLP_PC);
    p.copied = (int)min((int64_t)p.n, max(mat - k, (int64_t)0));
    return p;
}

__global__ void __launch_bounds__(MLP_NT) k_mlp_weights(const float* __restrict__ w, __nv_bfloat16* __restrict__ wbf,
                                                        MlpLayout L) {
    const MlpPiece p = mlp_piece(L);
    for (int c = threadIdx.x; c < p.copied; c += MLP_NT) wbf[p.at + c] = __float2bfloat16(w[p.i + c]);
}

// Adam (Kingma & Ba) on FP32 master weights; writes the BF16 copies of the matrices.
__global__ void __launch_bounds__(MLP_NT) k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                                                 float* __restrict__ v, __nv_bfloat16* __restrict__ wbf, MlpLayout L,
                                                 float lr, float b1, float b2, float c1, float c2, float eps) {
    const MlpPiece p = mlp_piece(L);
    g += p.i; m += p.i; v += p.i; w += p.i; wbf += p.at;
    float g0[MLP_U], m0[MLP_U], v0[MLP_U], w0[MLP_U];
#pragma unroll
    for (int q = 0; q < MLP_U; ++q) {
        const int c = threadIdx.x + q * MLP_NT;
        if (c < p.n) { g0[q] = g[c]; m0[q] = m[c]; v0[q] = v[c]; w0[q] = w[c]; }
    }
#pragma unroll
    for (int q = 0; q < MLP_U; ++q) {
        const int c = threadIdx.x + q * MLP_NT;
        if (c >= p.n) break;
        const float gi = g0[q];
        const float mi = b1 * m0[q] + (1.f - b1) * gi;
        const float vi = b2 * v0[q] + (1.f - b2) * gi * gi;
        m[c] = mi;
        v[c] = vi;
        const float wi = w0[q] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[c] = wi;
        if (c < p.copied) wbf[c] = __float2bfloat16(wi);
    }
}

// ------------------------------------------------------------------ features
// feat[s][f]: for wave vector f = (mx, my, mz) of the list, sqrt(4 pi)/|k| dV sum_z W[s][z][my][mx] e^{-2 pi i mz z/n}
// (W = forward xy transform of zeta-bar * phi); real parts, then imaginary parts, then F(0) real.
__global__ void k_cv_gather(int n, const float2* __restrict__ W, int nk, const int4* __restrict__ ks, float kscale,
                            float dV, const float2* __restrict__ tw, float* __restrict__ feat) {
    const int s = blockIdx.x;
    const int nf = 2 * nk + 1;
    const size_t ng = (size_t)n * n * n;
    for (int f = threadIdx.x; f <= nk; f += blockDim.x) {
        const int4 m = f < nk ? ks[f] : make_int4(0, 0, 0, 0);
        const int ix = (m.x % n + n) % n, iy = (m.y % n + n) % n, iz = (m.z % n + n) % n;
        float re = 0.f, im = 0.f;
        for (int z = 0; z < n; ++z) {
            const float2 v = W[(size_t)s * ng + ((size_t)z * n + iy) * n + ix];
            const float2 w = tw[(iz * z) % n];          // e^{-2 pi i mz z / n}
            re += v.x * w.x - v.y * w.y;
            im += v.x * w.y + v.y * w.x;
        }
        if (f < nk) {
            const float k2 = kscale * (float)(m.x * m.x + m.y * m.y + m.z * m.z);
            const float wgt = dV * 3.5449077018110318f / sqrtf(k2);    // sqrt(4 pi)/|k|
            feat[(size_t)s * nf + f] = re * wgt;
            feat[(size_t)s * nf + nk + f] = im * wgt;
        } else {
            feat[(size_t)s * nf + 2 * nk] = re * dV;
        }
    }
}

// feat[s] = [|F_{s,0}(k)|^2 (nk), F_{s,0}(0)^2, sum_{v>=1} |F_{s,v}(k)|^2 (nk), sum_{v>=1} F_{s,v}(0)^2]
// from the per-vector coefficients raw[s][v] = [Re F(k) (nk), Im F(k) (nk), F(0)].
__global__ void k_cv_combine(int n_samples, int nv, int nk, const float* __restrict__ raw, float* __restrict__ feat) {
    const int s = blockIdx.x;
    const int nr = 2 * nk + 1, nf = 2 * (nk + 1);
    for (int f = threadIdx.x; f <= nk; f += blockDim.x) {
        float z = 0.f, e = 0.f;
        for (int v = 0; v < nv; ++v) {
            const float* r = raw + ((size_t)s * nv + v) * nr;
            const float q = f < nk ? r[f] * r[f] + r[nk + f] * r[nk + f] : r[2 * nk] * r[2 * nk];
            if (v == 0) z = q;
            else e += q;
        }
        feat[(size_t)s * nf + f] = z;
        feat[(size_t)s * nf + nk + 1 + f] = e;
    }
}

// float columns standardised in place with FP64 statistics (computed when compute != 0)
__global__ void k_cv_stats_f32(int n, int O, const float* __restrict__ y, double* __restrict__ mu,
                               double* __restrict__ sd) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= O) return;
    double m = 0.0;
    for (int i = 0; i < n; ++i) m += y[(size_t)i * O + o];
    m /= n;
    double v = 0.0;
    for (int i = 0; i < n; ++i) {
        const double d = y[(size_t)i * O + o] - m;
        v += d * d;
    }
    v = n > 1 ? v / (n - 1) : 0.0;
    mu[o] = m;
    sd[o] = v > 0.0 ? sqrt(v) : 1.0;
}

__global__ void k_cv_apply_f32(int64_t total, int O, float* __restrict__ y, const double* __restrict__ mu,
                               const double* __restrict__ sd) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(i % O);
        y[i] = (float)(((double)y[i] - mu[o]) / sd[o]);
    }
}

// source s = Re(zeta-bar) * phi as c64, zeta-bar taken with a sample stride
__global__ void k_cv_source(int64_t ng, const float2* __restrict__ zb, int64_t stride, const float* __restrict__ phi,
                            int n_samples, float2* __restrict__ out) {
    const int64_t total = ng * n_samples;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = i / ng, g = i % ng;
        out[i] = make_float2(zb[s * stride + g].x * phi[g], 0.f);
    }
}

// ------------------------------------------------------------------ FP64 standardisation and CV rows
// mu[o], sd[o] over n rows of y (double [n][O]); t = (y - mu)/sd in float.
__global__ void k_cv_stats(int n, int O, const double* __restrict__ y, double* __restrict__ mu, double* __restrict__ sd) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= O) return;
    double m = 0.0;
    for (int i = 0; i < n; ++i) m += y[(size_t)i * O + o];
    m /= n;
    double v = 0.0;
    for (int i = 0; i < n; ++i) {
        const double d = y[(size_t)i * O + o] - m;
        v += d * d;
    }
    v = n > 1 ? v / (n - 1) : 0.0;
    mu[o] = m;
    sd[o] = v > 0.0 ? sqrt(v) : 1.0;
}

__global__ void k_cv_standardize(int64_t total, int O, const double* __restrict__ y, const double* __restrict__ mu,
                                 const double* __restrict__ sd, float* __restrict__ t) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(i % O);
        t[i] = (float)((y[i] - mu[o]) / sd[o]);
    }
}

// rows[i][o] = mean_j f_c[j][o] + y[i][o] - f_p[i][o], with f = mu + sd * net (FP64).
__global__ void k_cv_rows(int Mc, int n, int O, const float* __restrict__ fc, const float* __restrict__ fp,
                          const double* __restrict__ y, const double* __restrict__ mu, const double* __restrict__ sd,
                          double* __restrict__ rows) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= O) return;
    double mc = 0.0;
    for (int j = 0; j < Mc; ++j) mc += mu[o] + sd[o] * (double)fc[(size_t)j * O + o];
    if (Mc > 0) mc /= Mc;
    for (int i = 0; i < n; ++i) {
        const double f = Mc > 0 ? mu[o] + sd[o] * (double)fp[(size_t)i * O + o] : 0.0;
        rows[(size_t)i * O + o] = (Mc > 0 ? mc : 0.0) + y[(size_t)i * O + o] - f;
    }
}

}  // namespace sgw

// ================================================================== host side
namespace sgw {
// ---------------------------------------------------------------- shell sums and the linear part
// out[i][c]: c < S: sum of the zeta-bar features of shell c, c = S: the zeta-bar k = 0 feature,
// then the same for the eta-bar block (S = n_shells); fixed k order, FP64 accumulation.
__global__ void k_cv_shells(int n, int nk, int n_shells, const int* __restrict__ shell_of_k,
                            const float* __restrict__ feat, float* __restrict__ out) {
    const int per = 2 * (n_shells + 1);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * per) return;
    const int i = t / per, c = t % per, half = c / (n_shells + 1), sh = c % (n_shells + 1);
    const float* f = feat + (size_t)i * 2 * (nk + 1) + (size_t)half * (nk + 1);
    double acc = 0.0;
    if (sh == n_shells) {
        acc = f[nk];
    } else {
        for (int k = 0; k < nk; ++k)
            if (__ldg(shell_of_k + k) == sh) acc += f[k];
    }
    out[t] = (float)acc;
}

__global__ void k_f32_to_f64(int64_t n, const float* __restrict__ a, double* __restrict__ b) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (double)a[i];
}

// G[a][b] = sum_r xs[r][a] xs[r][b], xs = (x - mu) / sd  (rows in increasing order)
__global__ void k_cv_gram(int n, int p, const double* __restrict__ x, const double* __restrict__ mu,
                          const double* __restrict__ sd, double* __restrict__ G) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= p * p) return;
    const int a = t / p, b = t % p;
    double acc = 0.0;
    for (int r = 0; r < n; ++r)
        acc += ((x[(size_t)r * p + a] - mu[a]) / sd[a]) * ((x[(size_t)r * p + b] - mu[b]) / sd[b]);
    G[t] = acc;
}

// C[a][j] = sum_r xs[r][a] (y[r][j] - ybar[j])
__global__ void k_cv_xty(int n, int p, int o, const double* __restrict__ x, const double* __restrict__ mu,
                         const double* __restrict__ sd, const double* __restrict__ y, const double* __restrict__ ybar,
                         double* __restrict__ C) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)p * o) return;
    const int a = (int)(t / o), j = (int)(t % o);
    double acc = 0.0;
    for (int r = 0; r < n; ++r) acc += ((x[(size_t)r * p + a] - mu[a]) / sd[a]) * (y[(size_t)r * o + j] - ybar[j]);
    C[t] = acc;
}

// Linear model m = [mu p][sd p][ybar o][B p x o]; f(x)_j = ybar_j + sum_a ((x_a - mu_a) / sd_a) B_aj
__device__ __forceinline__ double lin_eval(const double* __restrict__ m, int p, int o, const float* x, int j) {
    const double* mu = m;
    const double* sd = m + p;
    const double* ybar = m + 2 * p;
    const double* B = m + 2 * p + o;
    double acc = ybar[j];
    for (int a = 0; a < p; ++a) acc += (((double)x[a] - mu[a]) / sd[a]) * B[(size_t)a * o + j];
    return acc;
}

// out = f(x), or y - f(x) when y is given
__global__ void k_cv_lin_apply(int n, int p, int o, const double* __restrict__ m, const float* __restrict__ x,
                               const double* __restrict__ y, double* __restrict__ out) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * o) return;
    const int i = (int)(t / o), j = (int)(t % o);
    const double f = lin_eval(m, p, o, x + (size_t)i * p, j);
    out[t] = y != nullptr ? y[t] - f : f;
}

// xbar[a] = mean over the m cheap samples of x[.][a] (fixed order)
__global__ void k_cv_lin_mean(int mc, int p, const float* __restrict__ x, double* __restrict__ xbar) {
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= p) return;
    double acc = 0.0;
    for (int r = 0; r < mc; ++r) acc += (double)x[(size_t)r * p + a];
    xbar[a] = acc / mc;
}

// yout[i][j] = y[i][j] - f(x_i)_j + f(xbar)_j  (the mean of a linear f over the cheap samples)
__global__ void k_cv_lin_rows(int n, int p, int o, const double* __restrict__ m, const double* __restrict__ xbar,
                              const float* __restrict__ xp, const double* __restrict__ y, double* __restrict__ yout) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * o) return;
    const int i = (int)(t / o), j = (int)(t % o);
    const double* mu = m;
    const double* sd = m + p;
    const double* B = m + 2 * p + o;
    double d = 0.0;     // f(x_i) - f(xbar) = sum_a (x_ia - xbar_a) / sd_a B_aj
    for (int a = 0; a < p; ++a) d += (((double)xp[(size_t)i * p + a] - mu[a]) / sd[a] - (xbar[a] - mu[a]) / sd[a]) *
                                     B[(size_t)a * o + j];
    yout[t] = y[t] - d;
}

void launch_cv_source(int64_t ng, const float2* zb, int64_t stride, const float* phi, int n_samples, float2* out,
                      cudaStream_t st) {
    const int64_t total = ng * n_samples;
    if (total == 0) return;
    const int64_t blocks = std::min<int64_t>((total + 255) / 256, 152 * 32);
    k_cv_source<<<(unsigned)blocks, 256, 0, st>>>(ng, zb, stride, phi, n_samples, out);
}
void launch_cv_gather(int n, const float2* W, int n_samples, int nk, const int4* ks, float kscale, float dV,
                      const float2* tw, float* feat, cudaStream_t st) {
    if (n_samples == 0) return;
    k_cv_gather<<<n_samples, 128, 0, st>>>(n, W, nk, ks, kscale, dV, tw, feat);
}
void launch_cv_combine(int n_samples, int nv, int nk, const float* raw, float* feat, cudaStream_t st) {
    if (n_samples == 0) return;
    k_cv_combine<<<n_samples, 128, 0, st>>>(n_samples, nv, nk, raw, feat);
}
void launch_cv_standardize_f32(int n, int O, float* y, double* mu, double* sd, int compute, cudaStream_t st) {
    if (compute) k_cv_stats_f32<<<(O + 127) / 128, 128, 0, st>>>(n, O, y, mu, sd);
    const int64_t total = (int64_t)n * O;
    if (total == 0) return;
    const int64_t blocks = std::min<int64_t>((total + 255) / 256, 152 * 32);
    k_cv_apply_f32<<<(unsigned)blocks, 256, 0, st>>>(total, O, y, mu, sd);
}
void launch_cv_stats(int n, int O, const double* y, double* mu, double* sd, cudaStream_t st) {
    k_cv_stats<<<(O + 127) / 128, 128, 0, st>>>(n, O, y, mu, sd);
}
void launch_cv_standardize(int64_t total, int O, const double* y, const double* mu, const double* sd, float* t,
                           cudaStream_t st) {
    if (total == 0) return;
    const int64_t blocks = std::min<int64_t>((total + 255) / 256, 152 * 32);
    k_cv_standardize<<<(unsigned)blocks, 256, 0, st>>>(total, O, y, mu, sd, t);
}
void launch_cv_rows(int Mc, int n, int O, const float* fc, const float* fp, const double* y, const double* mu,
                    const double* sd, double* rows, cudaStream_t st) {
    k_cv_rows<<<(O + 127) / 128, 128, 0, st>>>(Mc, n, O, fc, fp, y, mu, sd, rows);
}

void launch_cv_shells(int n, int nk, int n_shells, const int* shell_of_k, const float* feat, float* out, cudaStream_t st) {
    const int total = n * 2 * (n_shells + 1);
    if (total > 0) k_cv_shells<<<(total + 127) / 128, 128, 0, st>>>(n, nk, n_shells, shell_of_k, feat, out);
}

void launch_f32_to_f64(int64_t n, const float* a, double* b, cudaStream_t st) {
    if (n > 0) k_f32_to_f64<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, st>>>(n, a, b);
}

void launch_cv_gram(int n, int p, const double* x, const double* mu, const double* sd, double* G, cudaStream_t st) {
    k_cv_gram<<<(p * p + 127) / 128, 128, 0, st>>>(n, p, x, mu, sd, G);
}

void launch_cv_xty(int n, int p, int o, const double* x, const double* mu, const double* sd, const double* y,
                   const double* ybar, double* C, cudaStream_t st) {
    const int64_t total = (int64_t)p * o;
    k_cv_xty<<<(unsigned)((total + 127) / 128), 128, 0, st>>>(n, p, o, x, mu, sd, y, ybar, C);
}

void launch_cv_lin_apply(int n, int p, int o, const double* m, const float* x, const double* y, double* out,
                         cudaStream_t st) {
    const int64_t total = (int64_t)n * o;
    if (total > 0) k_cv_lin_apply<<<(unsigned)((total + 127) / 128), 128, 0, st>>>(n, p, o, m, x, y, out);
}

void launch_cv_lin_rows(int mc, int n, int p, int o, const double* m, const float* xc, const float* xp,
                        const double* y, double* xbar, double* yout, cudaStream_t st) {
    k_cv_lin_mean<<<(p + 63) / 64, 64, 0, st>>>(mc, p, xc, xbar);
    const int64_t total = (int64_t)n * o;
    if (total > 0) k_cv_lin_rows<<<(unsigned)((total + 127) / 128), 128, 0, st>>>(n, p, o, m, xbar, xp, y, yout);
}

}  // namespace sgw

struct sgw_mlp {
    int n_in = 0, width = 0, n_out = 0, max_batch = 0, device = 0;
    cudaStream_t stream = nullptr;
    sgw::MlpLayout lay{};
    int64_t boff[4] = {0};          // where the biases start
    int ldw[4] = {0};               // padded row lengths of the BF16 weight matrices
    int ldx = 0, ldh = 0, ldo = 0;  // padded row lengths of the BF16 matrices with n_in, width, n_out columns
    int64_t np = 0;
    float* P = nullptr;            // FP32 master parameters: W1, b1, W2, b2, W3, b3, W4, b4
    float* G = nullptr;            // gradients (same layout)
    float* Ma = nullptr;           // Adam first moments
    float* Va = nullptr;           // Adam second moments
    __nv_bfloat16* Pbf = nullptr;  // BF16 copies of the weight matrices, rows padded (used by the GEMMs)
    int step = 0;
    __nv_bfloat16 *Xbf = nullptr, *Abf[3] = {nullptr}, *dYbf = nullptr, *dZbf[2] = {nullptr};
    float *Z[3] = {nullptr}, *Y = nullptr, *dY = nullptr, *dZ[2] = {nullptr};
    double* loss = nullptr;
    float* lw = nullptr;           // per-output loss weights (nullptr: all 1)
    std::string err;
};

namespace {
sgw_status mfail(sgw_mlp* m, sgw_status s, const std::string& msg) {
    if (m) m->err = msg;
    else sgw::set_global_error(msg.c_str());
    return s;
}
#define MCK(call)                                                                                         \
    do {                                                                                                  \
        cudaError_t e_ = (call);                                                                          \
        if (e_ != cudaSuccess) return mfail(m, SGW_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

uint64_t splitmix64(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

unsigned grid1(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16); }

constexpr int MAX_LOSS_BLOCKS = 304;       // partial sums of the loss: two blocks to an SM at most

// Rows of 32 or 64 to a tile: 64 reads the weights half as often and pays once its tiles fill the chip.
bool wide_tiles(int M, int N) { return sgw::gemm_tiles(64, M, N) >= 152; }

void forward_gemm(sgw_mlp* m, const sgw::Gemm& g) {
    if (wide_tiles(g.M, g.N))
        sgw::launch_dependent(sgw::k_mlp_forward<64>, dim3((unsigned)sgw::gemm_tiles(64, g.M, g.N)), sgw::G_NT,
                              sgw::GemmCfg<64>::SMEM, 1, m->stream, g);
    else
        sgw::launch_dependent(sgw::k_mlp_forward<32>, dim3((unsigned)sgw::gemm_tiles(32, g.M, g.N)), sgw::G_NT,
                              sgw::GemmCfg<32>::SMEM, 1, m->stream, g);
}

// The three hidden layers (their pre-activations kept when `keep`), then `last` for the output.
sgw_status mlp_forward(sgw_mlp* m, const float* x, int M, bool keep, const sgw::GemmEpi& last) {
    const int H = m->width, I = m->n_in, O = m->n_out;
    const int64_t n = (int64_t)M * I;
    sgw::k_mlp_input<<<grid1(n), 256, 0, m->stream>>>(n, I, m->ldx, x, m->Xbf);
    const __nv_bfloat16* in = m->Xbf;
    int K = I, ld = m->ldx;
    for (int l = 0; l < 3; ++l) {
        sgw::GemmEpi ep{};
        ep.mode = sgw::EPI_BIAS_TANH; ep.bias = m->P + m->boff[l];
        ep.out = keep ? m->Z[l] : nullptr; ep.ldo = H; ep.out_bf = m->Abf[l]; ep.ldb = m->ldh;
        forward_gemm(m, sgw::Gemm{M, H, K, in, ld, m->Pbf + m->lay.poff[l], m->ldw[l], ep});
        in = m->Abf[l];
        K = H;
        ld = m->ldh;
    }
    forward_gemm(m, sgw::Gemm{M, O, H, in, ld, m->Pbf + m->lay.poff[3], m->ldw[3], last});
    MCK(cudaGetLastError());
    return SGW_OK;
}

// Loss sum_o w_o (y - t)^2 / (M O) and its gradient.
sgw_status mlp_gradients(sgw_mlp* m, const float* x, const float* t, int M) {
    const int H = m->width, I = m->n_in, O = m->n_out;
    sgw::GemmEpi le{};
    le.mode = sgw::EPI_LOSS; le.bias = m->P + m->boff[3]; le.out = m->dY; le.ldo = O;
    le.out_bf = m->dYbf; le.ldb = m->ldo; le.aux = t; le.w = m->lw; le.scale = 2.0f / (float)((int64_t)M * O);
    le.y = m->Y;
    sgw_status s = mlp_forward(m, x, M, true, le);
    if (s) return s;
    const float* dz = m->dY;
    const __nv_bfloat16* dzbf = m->dYbf;
    int N = O, ldz = m->ldo;
    for (int l = 3; l >= 0; --l) {
        const int K_in = l > 0 ? H : I, to = l & 1;
        sgw::Backward b{};
        sgw::GemmEpi ew{};
        ew.mode = sgw::EPI_STORE; ew.out = m->G + m->lay.woff[l]; ew.ldo = N;
        b.w = sgw::Gemm{K_in, N, M, l > 0 ? m->Abf[l - 1] : m->Xbf, l > 0 ? m->ldh : m->ldx, dzbf, ldz, ew};
        b.splits = 1;
        if (l > 0) {
            sgw::GemmEpi ed{};
            ed.mode = sgw::EPI_DTANH; ed.out = m->dZ[to]; ed.ldo = H; ed.out_bf = m->dZbf[to]; ed.ldb = m->ldh;
            ed.aux = m->Z[l - 1];
            b.d = sgw::Gemm{M, H, N, dzbf, ldz, m->Pbf + m->lay.poff[l], m->ldw[l], ed};
        }
        b.d_tiles = l > 0 ? sgw::gemm_tiles(32, M, H) : 0;
        while (b.splits < 8 && N >= 2 * b.splits * 3 * sgw::GK && b.d_tiles * b.splits * 2 <= 152) b.splits *= 2;
        b.w_tiles = sgw::gemm_tiles(32, K_in, N);
        b.db_blocks = (N + 31) / 32;
        b.dz = dz; b.db = m->G + m->boff[l]; b.ldz = N;
        const int64_t ny = (int64_t)M * O;
        b.loss = sgw::Loss{ny, O, (int)std::min<int64_t>((ny + sgw::G_NT - 1) / sgw::G_NT, MAX_LOSS_BLOCKS), m->Y, t, m->lw, m->loss};
        b.loss_blocks = l == 3 ? b.loss.blocks : 0;
        b.loss_sums = l == 2;
        int64_t blocks = b.d_tiles * b.splits + b.w_tiles + b.db_blocks + b.loss_blocks + b.loss_sums;
        blocks = (blocks + b.splits - 1) / b.splits * b.splits;
        sgw::launch_dependent(sgw::k_mlp_backward, dim3((unsigned)blocks), sgw::G_NT, sgw::GemmCfg<32>::SMEM,
                              (unsigned)b.splits, m->stream, b);
        dz = m->dZ[to]; dzbf = m->dZbf[to];
        N = H; ldz = m->ldh;
    }
    MCK(cudaGetLastError());
    return SGW_OK;
}

int pad8(int n) { return (n + 7) / 8 * 8; }

template <class K>
bool gemm_attributes(K kern, int smem) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
}

sgw_status mlp_check(sgw_mlp* m, int M) {
    if (!m) return mfail(nullptr, SGW_EINVAL, "null mlp");
    if (M < 1 || M > m->max_batch) return mfail(m, SGW_EINVAL, "batch out of range (1..max_batch)");
    MCK(cudaSetDevice(m->device));
    return SGW_OK;
}
}  // namespace

extern "C" {

sgw_status sgw_mlp_create(sgw_mlp** out, int n_in, int width, int n_out, int max_batch, uint64_t seed, int device,
                          void* stream) {
    sgw_mlp* m = nullptr;
    if (!out || n_in < 1 || width < 1 || n_out < 1 || max_batch < 1) return mfail(nullptr, SGW_EINVAL, "bad mlp sizes");
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return mfail(nullptr, SGW_ECUDA, "cudaSetDevice failed");
    m = new (std::nothrow) sgw_mlp();
    if (!m) return mfail(nullptr, SGW_ENOMEM, "host allocation failed");
    m->n_in = n_in; m->width = width; m->n_out = n_out; m->max_batch = max_batch;
    m->device = device; m->stream = (cudaStream_t)stream;
    const int d[5] = {n_in, width, width, width, n_out};
    int64_t off = 0, bf = 0;
    for (int l = 0; l < 4; ++l) {
        const int ld = pad8(d[l + 1]);
        const bool one = ld == d[l + 1] && (d[l] + (int64_t)1) * d[l + 1] < (1 << 30);     // (a row's length is an int)
        m->ldw[l] = ld;
        m->lay.woff[l] = off;
        m->lay.mat[l] = (int64_t)d[l] * d[l + 1]; off += m->lay.mat[l];
        m->boff[l] = off; off += d[l + 1];
        m->lay.poff[l] = bf; bf += (int64_t)d[l] * ld;
        m->lay.len[l] = one ? (d[l] + 1) * d[l + 1] : d[l + 1];
        m->lay.ld[l] = ld;
        m->lay.pieces[l] = (m->lay.len[l] + sgw::MLP_PC - 1) / sgw::MLP_PC;
        m->lay.first[l + 1] = m->lay.first[l] + (int64_t)(one ? 1 : d[l] + 1) * m->lay.pieces[l];
    }
    m->ldx = pad8(n_in); m->ldh = pad8(width); m->ldo = pad8(n_out);
    m->np = off;
    const size_t B = max_batch;
    // the BF16 matrices are zeroed: what pads their rows is never written again
    auto get = [](auto** p, size_t bytes) { return cudaMalloc(p, bytes) == cudaSuccess; };
    auto get_bf = [&](__nv_bfloat16** p, int64_t el) { return get(p, 2 * el) && cudaMemset(*p, 0, 2 * el) == cudaSuccess; };
    bool ok = get(&m->P, 4 * off) && get(&m->G, 4 * off) && get(&m->Ma, 4 * off) && get(&m->Va, 4 * off) &&
              get_bf(&m->Pbf, bf) && get_bf(&m->Xbf, B * m->ldx) && get(&m->Y, 4 * B * n_out) &&
              get(&m->dY, 4 * B * n_out) && get_bf(&m->dYbf, B * m->ldo) &&
              get(&m->loss, sizeof(double) * (1 + MAX_LOSS_BLOCKS));
    for (int l = 0; l < 3 && ok; ++l) ok = get_bf(&m->Abf[l], B * m->ldh) && get(&m->Z[l], 4 * B * width);
    for (int l = 0; l < 2 && ok; ++l) ok = get(&m->dZ[l], 4 * B * width) && get_bf(&m->dZbf[l], B * m->ldh);
    ok = ok && gemm_attributes(sgw::k_mlp_forward<32>, sgw::GemmCfg<32>::SMEM) &&
         gemm_attributes(sgw::k_mlp_forward<64>, sgw::GemmCfg<64>::SMEM) &&
         gemm_attributes(sgw::k_mlp_backward, sgw::GemmCfg<32>::SMEM);
    if (!ok) {
        cudaGetLastError();
        sgw_mlp_destroy(m);
        return mfail(nullptr, SGW_ENOMEM, "mlp device allocation failed");
    }
    // uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights from splitmix64, zero biases
    std::vector<float> h(off, 0.f);
    uint64_t s = seed;
    for (int l = 0; l < 4; ++l) {
        const double a = 1.0 / std::sqrt((double)d[l]);
        for (int64_t i = 0; i < (int64_t)d[l] * d[l + 1]; ++i) {
            const double u = (double)(splitmix64(s) >> 11) * (1.0 / 9007199254740992.0);
            h[m->lay.woff[l] + i] = (float)(a * (2.0 * u - 1.0));
        }
    }
    sgw_status st = sgw_mlp_set_params(m, h.data(), off);
    if (st != SGW_OK) {
        std::string e = m->err;
        sgw_mlp_destroy(m);
        return mfail(nullptr, st, e);
    }
    *out = m;
    return SGW_OK;
}

void sgw_mlp_destroy(sgw_mlp* m) {
    if (!m) return;
    cudaSetDevice(m->device);
    void* p[] = {m->P, m->G, m->Ma, m->Va, m->Pbf, m->Xbf, m->Y, m->dY, m->dYbf, m->loss, m->lw, m->Abf[0], m->Abf[1],
                 m->Abf[2], m->Z[0], m->Z[1], m->Z[2], m->dZ[0], m->dZ[1], m->dZbf[0], m->dZbf[1]};
    for (void* q : p)
        if (q) cudaFree(q);
    delete m;
}

const char* sgw_mlp_last_error(const sgw_mlp* m) { return m ? m->err.c_str() : sgw_last_error(nullptr); }

int64_t sgw_mlp_param_count(const sgw_mlp* m) { return m ? m->np : 0; }

sgw_status sgw_mlp_set_params(sgw_mlp* m, const float* params_host, int64_t n) {
    if (!m || !params_host || n != m->np) return mfail(m, SGW_EINVAL, "parameter count mismatch");
    MCK(cudaSetDevice(m->device));
    MCK(cudaMemcpy(m->P, params_host, 4 * n, cudaMemcpyHostToDevice));
    MCK(cudaMemset(m->Ma, 0, 4 * n));
    MCK(cudaMemset(m->Va, 0, 4 * n));
    m->step = 0;
    sgw::k_mlp_weights<<<(unsigned)m->lay.first[4], sgw::MLP_NT, 0, m->stream>>>(m->P, m->Pbf, m->lay);
    MCK(cudaGetLastError());
    MCK(cudaStreamSynchronize(m->stream));
    return SGW_OK;
}

sgw_status sgw_mlp_get_params(sgw_mlp* m, float* params_host, int64_t n) {
    if (!m || !params_host || n != m->np) return mfail(m, SGW_EINVAL, "parameter count mismatch");
    MCK(cudaSetDevice(m->device));
    MCK(cudaStreamSynchronize(m->stream));
    MCK(cudaMemcpy(params_host, m->P, 4 * n, cudaMemcpyDeviceToHost));
    return SGW_OK;
}

sgw_status sgw_mlp_set_loss_weights(sgw_mlp* m, const float* w_host, int n_out) {
    if (!m || n_out != m->n_out) return mfail(m, SGW_EINVAL, "loss weights need n_out entries");
    MCK(cudaSetDevice(m->device));
    if (!w_host) {
        if (m->lw) cudaFree(m->lw);
        m->lw = nullptr;
        return SGW_OK;
    }
    if (!m->lw) MCK(cudaMalloc(&m->lw, sizeof(float) * n_out));
    MCK(cudaMemcpy(m->lw, w_host, sizeof(float) * n_out, cudaMemcpyHostToDevice));
    return SGW_OK;
}

sgw_status sgw_mlp_forward(sgw_mlp* m, const float* x_dev, int M, float* y_dev) {
    sgw_status s = mlp_check(m, M);
    if (s) return s;
    if (!x_dev || !y_dev) return mfail(m, SGW_EINVAL, "null pointers");
    // a y that floats can't be stored to goes by way of Y and a copy
    const bool direct = reinterpret_cast<uintptr_t>(y_dev) % alignof(float) == 0;
    sgw::GemmEpi ep{};
    ep.mode = sgw::EPI_BIAS; ep.bias = m->P + m->boff[3]; ep.out = direct ? y_dev : m->Y; ep.ldo = m->n_out;
    if ((s = mlp_forward(m, x_dev, M, false, ep))) return s;
    if (!direct) MCK(cudaMemcpyAsync(y_dev, m->Y, sizeof(float) * (size_t)M * m->n_out, cudaMemcpyDeviceToDevice, m->stream));
    return SGW_OK;
}

sgw_status sgw_mlp_gradients(sgw_mlp* m, const float* x_dev, const float* t_dev, int M, double* loss_host,
                             float* grads_host) {
    sgw_status s = mlp_check(m, M);
    if (s) return s;
    if (!x_dev || !t_dev) return mfail(m, SGW_EINVAL, "null pointers");
    if ((s = mlp_gradients(m, x_dev, t_dev, M))) return s;
    if (loss_host) {
        double l;
        MCK(cudaMemcpyAsync(&l, m->loss, 8, cudaMemcpyDeviceToHost, m->stream));
        MCK(cudaStreamSynchronize(m->stream));
        *loss_host = l / ((double)M * m->n_out);
    }
    if (grads_host) {
        MCK(cudaStreamSynchronize(m->stream));
        MCK(cudaMemcpy(grads_host, m->G, 4 * m->np, cudaMemcpyDeviceToHost));
    }
    return SGW_OK;
}

sgw_status sgw_mlp_adam_step(sgw_mlp* m, float lr) {
    if (!m) return mfail(nullptr, SGW_EINVAL, "null mlp");
    MCK(cudaSetDevice(m->device));
    m->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - (float)std::pow(0.9, m->step), c2 = 1.f - (float)std::pow(0.999, m->step);
    sgw::k_adam<<<(unsigned)m->lay.first[4], sgw::MLP_NT, 0, m->stream>>>(m->P, m->G, m->Ma, m->Va, m->Pbf, m->lay, lr, b1,
                                                                          b2, c1, c2, 1e-8f);
    MCK(cudaGetLastError());
    return SGW_OK;
}

sgw_status sgw_mlp_train_epoch(sgw_mlp* m, const float* x_dev, const float* t_dev, int n_rows, int batch, float lr,
                               double* mean_loss_host) {
    if (!m || !x_dev || !t_dev || n_rows < 1 || batch < 1 || batch > m->max_batch)
        return mfail(m, SGW_EINVAL, "bad training arguments");
    double tot = 0.0;
    for (int r0 = 0; r0 < n_rows; r0 += batch) {
        const int M = std::min(batch, n_rows - r0);
        double l = 0.0;
        sgw_status s = sgw_mlp_gradients(m, x_dev + (size_t)r0 * m->n_in, t_dev + (size_t)r0 * m->n_out, M,
                                          mean_loss_host ? &l : nullptr, nullptr);
        if (s) return s;
        if ((s = sgw_mlp_adam_step(m, lr))) return s;
        tot += l * M;
    }
    if (mean_loss_host) *mean_loss_host = tot / n_rows;
    return SGW_OK;
}

}  // extern "C"
