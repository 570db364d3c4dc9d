// DFTs of short lengths held in one thread's registers, with compile-time twiddles, and the
// "line operator": forward transform of a line, a diagonal factor in k, inverse transform, for a
// line split over T neighbouring lanes (no shared memory, no barrier).
#pragma once
#include "fft_smem.cuh"

namespace sgw {

// cos and sin of 2 pi k / n by their Taylor series in double, at compile time (argument reduced to
// [-pi/4, pi/4] by symmetry, so that the series is exact to rounding)
constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr double ct_sin_small(double x) {
    double t = x, s = x;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i) * (2 * i + 1));
        s += t;
    }
    return s;
}
constexpr double ct_cos_small(double x) {
    double t = 1.0, s = 1.0;
    for (int i = 1; i < 12; ++i) {
        t *= -x * x / ((2 * i - 1) * (2 * i));
        s += t;
    }
    return s;
}
// k / n of a turn: octant by octant
constexpr double ct_cos(int k, int n) {
    k = ((k % n) + n) % n;
    if (2 * k > n) k = n - k;                                         // cos is even
    if (4 * k > n) return -ct_cos(n - 2 * k, 2 * n);                  // cos(pi - x) = -cos x
    if (8 * k > n) return ct_sin_small(kTwoPi * (n - 4 * k) / (4.0 * n));
    return ct_cos_small(kTwoPi * k / n);
}
constexpr double ct_sin(int k, int n) { return ct_cos(4 * k - n, 4 * n); }   // sin x = cos(x - pi/2)

template <int K, int N> struct Turn {
    static constexpr float c = (float)ct_cos(K, N);
    static constexpr float s = (float)ct_sin(K, N);
};

// v exp(DIR 2 pi i K / N), K and N known at compile time (multiples of an eighth turn are cheaper)
template <int K, int N, int DIR>
__device__ __forceinline__ float2 rotc(float2 v) {
    constexpr int k = (DIR * K % N + N) % N;
    if constexpr (k == 0) return v;
    else if constexpr (4 * k == N) return make_float2(-v.y, v.x);
    else if constexpr (2 * k == N) return make_float2(-v.x, -v.y);
    else if constexpr (4 * k == 3 * N) return make_float2(v.y, -v.x);
    else if constexpr ((8 * k) % N == 0) {
        constexpr float r = 0.70710678118654752440f;
        constexpr float sc = Turn<k, N>::c > 0 ? 1.f : -1.f, ss = Turn<k, N>::s > 0 ? 1.f : -1.f;
        return make_float2(r * (sc * v.x - ss * v.y), r * (ss * v.x + sc * v.y));
    } else return cmul(v, make_float2(Turn<k, N>::c, Turn<k, N>::s));
}

template <int I> struct Ic { static constexpr int value = I; };
template <int B, int E, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (B < E) {
        f(Ic<B>{});
        static_for<B + 1, E>(f);
    }
}

// In-place DFT of v[0..N-1] with exp(DIR 2 pi i n k / N), natural order in and out.
template <int N, int DIR> struct RegDft;
template <int DIR> struct RegDft<1, DIR> { __device__ __forceinline__ static void run(float2*) {} };
template <int DIR> struct RegDft<2, DIR> : Dft<2, DIR> {};
template <int DIR> struct RegDft<3, DIR> : Dft<3, DIR> {};
template <int DIR> struct RegDft<4, DIR> : Dft<4, DIR> {};
template <int DIR> struct RegDft<8, DIR> : Dft<8, DIR> {};
// Cooley-Tukey, N = A B: n = b + B a, k = ka + A kb
template <int N, int A, int DIR> struct RegDftAB {
    static constexpr int B = N / A;
    __device__ __forceinline__ static void run(float2* v) {
        float2 u[B][A];
        static_for<0, B>([&](auto bi) {
            constexpr int b = decltype(bi)::value;
#pragma unroll
            for (int a = 0; a < A; ++a) u[b][a] = v[b + B * a];
            RegDft<A, DIR>::run(u[b]);
            static_for<1, A>([&](auto ki) {
                constexpr int k = decltype(ki)::value;
                u[b][k] = rotc<(b * k) % N, N, DIR>(u[b][k]);
            });
        });
#pragma unroll
        for (int k = 0; k < A; ++k) {
            float2 s[B];
#pragma unroll
            for (int b = 0; b < B; ++b) s[b] = u[b][k];
            RegDft<B, DIR>::run(s);
#pragma unroll
            for (int q = 0; q < B; ++q) v[k + A * q] = s[q];
        }
    }
};
template <int DIR> struct RegDft<6, DIR> : RegDftAB<6, 3, DIR> {};
template <int DIR> struct RegDft<12, DIR> : RegDftAB<12, 4, DIR> {};
template <int DIR> struct RegDft<16, DIR> : RegDftAB<16, 4, DIR> {};
template <int DIR> struct RegDft<24, DIR> : RegDftAB<24, 8, DIR> {};
template <int DIR> struct RegDft<32, DIR> : RegDftAB<32, 8, DIR> {};

// v = IDFT(f . DFT(v)) of N-point lines, unnormalised, a line on T lanes: lane l + (32 / T) t of a warp
// holds points t + T a of line l in v[a], a < P.  N = P T, n = t + T a, k = k1 + P k2:
//   X[k1 + P k2] = sum_t W_T^(t k2) W_N^(t k1) sum_a W_P^(a k1) x[t + T a].
// Lane t transforms its P points and hands block q of k1 (P / T values) to lane t + q: multiplying
// its inputs by W_T^(a t) first rotates its outputs by t blocks, so that slot block q always holds
// what lane t + q needs and no value is selected at run time.  The T-point transforms then act on
// sources t' - q; the phase W_T^(t' k2) by which that order differs cancels between the forward
// and the inverse transform (f is diagonal in k), so it is never applied.
// f(k1, i) with k1 a run-time int < P and k2 = i compile-time gives the factor (float or float2).
// tws: exp(-2 pi i m / N), m < N, in shared memory.  All lanes of the warp call it together.
template <class S> __device__ __forceinline__ float2 kmul(float2 v, S s);
template <> __device__ __forceinline__ float2 kmul<float>(float2 v, float s) { return cscale(v, s); }
template <> __device__ __forceinline__ float2 kmul<float2>(float2 v, float2 s) { return cmul(v, s); }

template <int T, int P, int DIR>
__device__ __forceinline__ void line_rotate(float2 (&v)[P], int t) {
    if constexpr (T == 2) {
        const float s = t ? -1.f : 1.f;
#pragma unroll
        for (int a = 1; a < P; a += 2) v[a] = cscale(v[a], s);
    } else {
        static_assert(T == 4, "two or four lanes per line");
        // exp(DIR 2 pi i a t / 4), a mod 4 = 1, 2, 3
        const float c1 = t == 0 ? 1.f : (t == 2 ? -1.f : 0.f);
        const float s1 = DIR * (t == 1 ? 1.f : (t == 3 ? -1.f : 0.f));
        const float c2 = (t & 1) ? -1.f : 1.f;
#pragma unroll
        for (int a = 0; a < P; ++a) {
            if ((a & 3) == 1) v[a] = cmul(v[a], make_float2(c1, s1));
            if ((a & 3) == 2) v[a] = cscale(v[a], c2);
            if ((a & 3) == 3) v[a] = cmul(v[a], make_float2(c1, -s1));
        }
    }
}

template <int N, int T, class F>
__device__ __forceinline__ void line_op(float2 (&v)[N / T], int lane, const float2* tws, F&& f) {
    constexpr int P = N / T, CPW = 32 / T, Q = P / T;
    static_assert(P % T == 0, "every lane takes P / T of the T-point transforms");
    const int t = lane / CPW, l = lane % CPW;
    line_rotate<T, P, -1>(v, t);
    RegDft<P, -1>::run(v);
#pragma unroll
    for (int j = 0; j < Q; ++j) {
        float2 w[T], r[T];
        // slot q Q + j of lane t holds k1 = ((q + t) mod T) Q + j
#pragma unroll
        for (int q = 0; q < T; ++q) {
            const int k1 = ((q + t) & (T - 1)) * Q + j;
            w[q] = tws[t * k1];
            r[q] = cmul(v[q * Q + j], w[q]);
        }
#pragma unroll
        for (int q = 1; q < T; ++q) {
            const int src = l + CPW * ((t - q) & (T - 1));
            r[q].x = __shfl_sync(0xffffffffu, r[q].x, src);
            r[q].y = __shfl_sync(0xffffffffu, r[q].y, src);
        }
        RegDft<T, +1>::run(r);
#pragma unroll
        for (int i = 0; i < T; ++i) r[i] = kmul(r[i], f(t * Q + j, i));
        RegDft<T, -1>::run(r);
#pragma unroll
        for (int q = 1; q < T; ++q) {
            const int src = l + CPW * ((t + q) & (T - 1));
            r[q].x = __shfl_sync(0xffffffffu, r[q].x, src);
            r[q].y = __shfl_sync(0xffffffffu, r[q].y, src);
        }
#pragma unroll
        for (int q = 0; q < T; ++q) v[q * Q + j] = cmul(r[q], cconj(w[q]));
    }
    RegDft<P, +1>::run(v);
    line_rotate<T, P, +1>(v, t);
}

}  // namespace sgw
