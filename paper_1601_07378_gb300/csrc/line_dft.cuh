// line_dft.cuh -- DFTs of up to 72 points held entirely in one thread's
// registers, for the line kernels of kernels_line.cuh.
//
// X[k] = sum_n x[n] exp(S 2 pi i n k / M), natural order in and out, every
// index a compile-time constant.  FP32 lane operations are what bounds these
// kernels (one instruction a cycle and scheduler, a paired instruction two),
// so the factorisations are chosen for the fewest of them:
//  * coprime factors by the prime-factor map (no twiddles between them);
//  * repeated factors by a last stage whose twiddles are folded into its
//    butterflies: w = g (1 + i t) with g = cos, t = tan (or g = sin and the
//    cotangent where |sin| > |cos|), so that w x costs two fused
//    multiply-adds and its scale g rides on the butterfly's own adds, now
//    fused multiply-adds by a constant.  A twiddled 4-point butterfly costs
//    22 lane operations instead of 28, a 48-point DFT 630 instead of 704.
//  * multiplications by +-i are operand swaps of scalar instructions.
#pragma once

#include "fft_core.cuh"

namespace vloc {
namespace line {

// a + S i b, and a + S i s b (s real)
template <int S> __device__ __forceinline__ float2 caddi(float2 a, float2 b) {
    return S > 0 ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, a.y - b.x);
}
template <int S> __device__ __forceinline__ float2 cfmai(float2 a, float s, float2 b) {
    const float t = S > 0 ? s : -s;
    return make_float2(fmaf(-t, b.y, a.x), fmaf(t, b.x, a.y));
}
// a + s b, one paired instruction (two scalar ones, which need no register
// pair of s, measured 4 % slower in the y/x pass: it is as short of issue slots
// as of lanes)
__device__ __forceinline__ float2 cfmar(float2 a, float s, float2 b) { return __ffma2_rn(make_float2(s, s), b, a); }

// x exp(S 2 pi i m / R) = g v: v by two fused multiply-adds, g the scale
template <int R, int S, int m_> struct Tw {
    static constexpr int m = ((S * m_) % R + R) % R;
    static constexpr double c = ct::cos_turn(m, R), s = ct::sin_turn(m, R);
    static constexpr bool unit = (4 * m) % R == 0;  // a power of i
    static constexpr bool by_cos = c * c >= s * s;
    static constexpr double g = unit ? 1.0 : by_cos ? c : s;
    __device__ __forceinline__ static float2 v(float2 x) {
        if constexpr (m == 0) return x;
        else if constexpr (4 * m == R) return make_float2(-x.y, x.x);
        else if constexpr (2 * m == R) return make_float2(-x.x, -x.y);
        else if constexpr (4 * m == 3 * R) return make_float2(x.y, -x.x);
        else if constexpr (by_cos) {
            constexpr float t = (float)(s / c);
            return make_float2(fmaf(-t, x.y, x.x), fmaf(t, x.x, x.y));
        } else {
            constexpr float t = (float)(c / s);
            return make_float2(fmaf(t, x.x, -x.y), fmaf(t, x.y, x.x));
        }
    }
    __device__ __forceinline__ static float2 mul(float2 x) {  // the whole product
        if constexpr (unit) return v(x);
        else {
            constexpr float cc = (float)c, ss = (float)s;
            return make_float2(x.x * cc - x.y * ss, x.x * ss + x.y * cc);
        }
    }
};

// B-point DFT of t[n] w^n, w = exp(S 2 pi i K / R), B = 2, 3, 4, 5
template <int B, int S, int R, int K> struct TDft;
template <int S, int R, int K> struct TDft<2, S, R, K> {
    __device__ __forceinline__ static void run(float2 (&t)[2]) {
        using W = Tw<R, S, K>;
        const float2 a = t[0], v = W::v(t[1]);
        if constexpr (W::unit) {
            t[0] = cadd(a, v);
            t[1] = csub(a, v);
        } else {
            t[0] = cfmar(a, (float)W::g, v);
            t[1] = cfmar(a, (float)-W::g, v);
        }
    }
};
template <int S, int R, int K> struct TDft<3, S, R, K> {
    __device__ __forceinline__ static void run(float2 (&t)[3]) {
        constexpr double h = 0.866025403784438646763723170752936183;  // sqrt(3) / 2
        using W1 = Tw<R, S, K>;
        using W2 = Tw<R, S, 2 * K>;
        const float2 a = t[0];
        if constexpr (K == 0) {
            const float2 p = cadd(t[1], t[2]), d = csub(t[1], t[2]), m = cfma(a, -0.5f, p);
            t[0] = cadd(a, p);
            t[1] = cfmai<S>(m, (float)h, d);
            t[2] = cfmai<S>(m, (float)-h, d);
        } else {
            constexpr double g = W1::g, r = W2::g / W1::g;
            const float2 v1 = W1::v(t[1]), v2 = W2::v(t[2]);
            const float2 p = cfmar(v1, (float)r, v2), d = cfmar(v1, (float)-r, v2), m = cfmar(a, (float)(-0.5 * g), p);
            t[0] = cfmar(a, (float)g, p);
            t[1] = cfmai<S>(m, (float)(g * h), d);
            t[2] = cfmai<S>(m, (float)(-g * h), d);
        }
    }
};
template <int S, int R, int K> struct TDft<4, S, R, K> {
    __device__ __forceinline__ static void run(float2 (&t)[4]) {
        if constexpr (K == 0) {
            const float2 t0 = cadd(t[0], t[2]), t1 = csub(t[0], t[2]), t2 = cadd(t[1], t[3]), t3 = csub(t[1], t[3]);
            t[0] = cadd(t0, t2);
            t[2] = csub(t0, t2);
            t[1] = caddi<S>(t1, t3);
            t[3] = caddi<-S>(t1, t3);
        } else {
            using W1 = Tw<R, S, K>;
            using W2 = Tw<R, S, 2 * K>;
            using W3 = Tw<R, S, 3 * K>;
            constexpr double g1 = W1::g, g2 = W2::g, r = W3::g / W1::g;
            const float2 v1 = W1::v(t[1]), v2 = W2::v(t[2]), v3 = W3::v(t[3]);
            const float2 a0 = cfmar(t[0], (float)g2, v2), a1 = cfmar(t[0], (float)-g2, v2);
            const float2 b0 = cfmar(v1, (float)r, v3), b1 = cfmar(v1, (float)-r, v3);
            t[0] = cfmar(a0, (float)g1, b0);
            t[2] = cfmar(a0, (float)-g1, b0);
            t[1] = cfmai<S>(a1, (float)g1, b1);
            t[3] = cfmai<S>(a1, (float)-g1, b1);
        }
    }
};
template <int S, int R, int K> struct TDft<5, S, R, K> {
    __device__ __forceinline__ static void run(float2 (&t)[5]) {
        constexpr float c1 = (float)ct::cos_turn(1, 5), c2 = (float)ct::cos_turn(2, 5);
        constexpr float s1 = (float)ct::sin_turn(1, 5), s2 = (float)ct::sin_turn(2, 5);
        const float2 x0 = t[0], x1 = Tw<R, S, K>::mul(t[1]), x2 = Tw<R, S, 2 * K>::mul(t[2]),
                     x3 = Tw<R, S, 3 * K>::mul(t[3]), x4 = Tw<R, S, 4 * K>::mul(t[4]);
        const float2 a1 = cadd(x1, x4), b1 = csub(x1, x4), a2 = cadd(x2, x3), b2 = csub(x2, x3);
        const float2 p1 = cfmar(cfmar(x0, c1, a1), c2, a2), p2 = cfmar(cfmar(x0, c2, a1), c1, a2);
        t[0] = cadd(cadd(x0, a1), a2);
        t[1] = cfmai<S>(cfmai<S>(p1, s1, b1), s2, b2);
        t[4] = cfmai<S>(cfmai<S>(p1, -s1, b1), -s2, b2);
        t[2] = cfmai<S>(cfmai<S>(p2, s2, b1), -s1, b2);
        t[3] = cfmai<S>(cfmai<S>(p2, -s2, b1), s1, b2);
    }
};

template <int M, int S> struct RDft;
// M = A B, n = B n1 + n2, k = k1 + A k2: A-point DFTs, then twiddled B-point
// butterflies
template <int A, int B, int S> struct DftTw {
    __device__ __forceinline__ static void run(float2* v) {
        float2 y[A * B];
        sfor<B>([&](auto n2) {
            float2 t[A];
            sfor<A>([&](auto n1) { t[n1] = v[B * n1 + n2]; });
            RDft<A, S>::run(t);
            sfor<A>([&](auto k1) { y[n2 * A + k1] = t[k1]; });
        });
        sfor<A>([&](auto k1) {
            float2 t[B];
            sfor<B>([&](auto n2) { t[n2] = y[n2 * A + k1]; });
            TDft<B, S, A * B, decltype(k1)::value>::run(t);
            sfor<B>([&](auto k2) { v[k1 + A * k2] = t[k2]; });
        });
    }
};
// M = A B with A, B coprime (Good-Thomas): n = B n1 + A n2, k = k1 mod A and
// k2 mod B by the Chinese remainder theorem, both mod M
constexpr int inv_mod(int a, int m) {
    for (int i = 1; i < m; ++i)
        if ((a * i) % m == 1 % m) return i;
    return 1;
}
template <int A, int B, int S> struct DftPfa {
    __device__ __forceinline__ static void run(float2* v) {
        constexpr int M = A * B, ea = B * inv_mod(B % A, A), eb = A * inv_mod(A % B, B);
        float2 y[M];
        sfor<B>([&](auto n2) {
            float2 t[A];
            sfor<A>([&](auto n1) { t[n1] = v[(B * n1 + A * n2) % M]; });
            RDft<A, S>::run(t);
            sfor<A>([&](auto k1) { y[n2 * A + k1] = t[k1]; });
        });
        sfor<A>([&](auto k1) {
            float2 t[B];
            sfor<B>([&](auto n2) { t[n2] = y[n2 * A + k1]; });
            RDft<B, S>::run(t);
            sfor<B>([&](auto k2) { v[(ea * k1 + eb * k2) % M] = t[k2]; });
        });
    }
};
template <int B, int S> struct DftPrime {
    __device__ __forceinline__ static void run(float2* v) {
        float2 t[B];
        sfor<B>([&](auto n) { t[n] = v[n]; });
        TDft<B, S, 1, 0>::run(t);
        sfor<B>([&](auto n) { v[n] = t[n]; });
    }
};
template <int S> struct RDft<2, S> : DftPrime<2, S> {};
template <int S> struct RDft<3, S> : DftPrime<3, S> {};
template <int S> struct RDft<4, S> : DftPrime<4, S> {};
template <int S> struct RDft<5, S> : DftPrime<5, S> {};
template <int S> struct RDft<6, S> : DftPfa<2, 3, S> {};
template <int S> struct RDft<8, S> : DftTw<4, 2, S> {};
template <int S> struct RDft<9, S> : DftTw<3, 3, S> {};
template <int S> struct RDft<10, S> : DftPfa<2, 5, S> {};
template <int S> struct RDft<12, S> : DftPfa<4, 3, S> {};
template <int S> struct RDft<15, S> : DftPfa<3, 5, S> {};
template <int S> struct RDft<16, S> : DftTw<4, 4, S> {};
template <int S> struct RDft<18, S> : DftPfa<9, 2, S> {};
template <int S> struct RDft<20, S> : DftPfa<4, 5, S> {};
template <int S> struct RDft<24, S> : DftPfa<8, 3, S> {};
template <int S> struct RDft<25, S> : DftTw<5, 5, S> {};
template <int S> struct RDft<27, S> : DftTw<9, 3, S> {};
template <int S> struct RDft<30, S> : DftPfa<6, 5, S> {};
template <int S> struct RDft<32, S> : DftTw<8, 4, S> {};
template <int S> struct RDft<36, S> : DftPfa<9, 4, S> {};
template <int S> struct RDft<40, S> : DftPfa<8, 5, S> {};
template <int S> struct RDft<45, S> : DftPfa<9, 5, S> {};
template <int S> struct RDft<48, S> : DftPfa<16, 3, S> {};
template <int S> struct RDft<50, S> : DftPfa<25, 2, S> {};
template <int S> struct RDft<54, S> : DftPfa<27, 2, S> {};
template <int S> struct RDft<60, S> : DftPfa<12, 5, S> {};
template <int S> struct RDft<64, S> : DftTw<16, 4, S> {};
template <int S> struct RDft<72, S> : DftPfa<9, 8, S> {};

}  // namespace line
}  // namespace vloc
