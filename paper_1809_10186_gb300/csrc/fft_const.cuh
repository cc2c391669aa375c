// FFT lines in registers with compile-time twiddles, for the lengths of the velocity grid
// (8, 16, 32 and 12, 24 = 3 * 2^m). Decimation in time: element k of a line goes into slot
// line_slot<N>(k) (fourier_dev.cuh), the result is in natural order, unnormalised.
//
// A butterfly with a twiddle w other than 1 and -+i takes six fused multiply-adds,
//   s = u + w v (two chains of two),  d = 2 u - s,
// instead of two products, two FMAs and four additions; d carries the rounding of s, which is of
// the size of its own. The twiddles are immediate operands, so a line loads nothing but its data:
// 388 instructions for N = 32.
#pragma once

#include "fourier_dev.cuh"

namespace dgfs {
namespace cfft {

using fdev::add;
using fdev::bitrev;
using fdev::cos_of;
using fdev::line_slot;
using fdev::pack;
using fdev::sin_of;
using fdev::sub;
using fdev::unpack;

// 2 u - s, packed in FP32
template <typename T>
__device__ __forceinline__ Cplx<T> twice_minus(Cplx<T> u, Cplx<T> s) {
    return Cplx<T>{fma(T(2), u.x, -s.x), fma(T(2), u.y, -s.y)};
}
template <>
__device__ __forceinline__ Cplx<float> twice_minus<float>(Cplx<float> u, Cplx<float> s) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack(u)), "l"(pack(Cplx<float>{2.f, 2.f})),
        "l"(pack(Cplx<float>{-s.x, -s.y})));
    return unpack(r);
}

// a + sqrt(1/2) x with the constant in two FP32 terms (the first a multiple of 1/128): in one term it is 1.7e-8 short,
// and the lines of N = 24, which meet it in every transform of length 8, lose 2.2e-8 a round trip instead of 1.4e-8.
__device__ __forceinline__ float plus_half_root(float a, float x) {
    constexpr double c = cos_of<8>(1), head = (double)(int)(c * 128.0) / 128.0;
    return fma((float)(c - head), x, fma((float)head, x, a));
}
__device__ __forceinline__ double plus_half_root(double a, double x) { return fma(cos_of<8>(1), x, a); }

// c + w x with a constant w; nothing for w = 0
template <typename T>
__device__ __forceinline__ T madd(T w, T x, T c) { return w == T(0) ? c : fma(w, x, c); }

// radix-2 stages of a length-S transform in a[OFF .. OFF + S), spans LEN, 2 LEN, ..., S
template <typename T, int NA, int OFF, int S, int LEN, bool FWD>
__device__ __forceinline__ void stages(Cplx<T> (&a)[NA]) {
    constexpr int half = LEN / 2;
#pragma unroll
    for (int i = 0; i < S; i += LEN)
#pragma unroll
        for (int j = 0; j < half; ++j) {
            const Cplx<T> u = a[OFF + i + j], v = a[OFF + i + j + half];
            Cplx<T> s, d;
            if (j == 0) {
                s = add(u, v);
                d = sub(u, v);
            } else if (4 * j == LEN) {                         // twiddle -i (forward), +i (inverse)
                const T sg = FWD ? T(1) : T(-1);
                s = Cplx<T>{u.x + sg * v.y, u.y - sg * v.x};
                d = Cplx<T>{u.x - sg * v.y, u.y + sg * v.x};
            } else if (sizeof(T) == 4 && NA % 3 == 0 && LEN == 8) {   // (+-1 +- i) sqrt(1/2), exact to 1e-10
                const T sr = cos_of<8>(j) > 0 ? T(1) : T(-1), si = FWD ? T(-1) : T(1);
                const Cplx<T> t{sr * v.x - si * v.y, si * v.x + sr * v.y};
                s = Cplx<T>{plus_half_root(u.x, t.x), plus_half_root(u.y, t.y)};
                d = twice_minus(u, s);
            } else {
                const T wr = (T)cos_of<LEN>(j), wi = FWD ? (T)(-sin_of<LEN>(j)) : (T)sin_of<LEN>(j);
                s = Cplx<T>{fma(-wi, v.y, fma(wr, v.x, u.x)), fma(wi, v.x, fma(wr, v.y, u.y))};
                d = twice_minus(u, s);
            }
            a[OFF + i + j] = s;
            a[OFF + i + j + half] = d;
        }
    if constexpr (LEN < S) stages<T, NA, OFF, S, 2 * LEN, FWD>(a);
}

template <typename T, int N, bool FWD>
__device__ __forceinline__ void line(Cplx<T> (&a)[N]) {
    if constexpr ((N & (N - 1)) == 0) {
        stages<T, N, 0, N, 2, FWD>(a);
    } else {
        constexpr int S = N / 3;
        static_assert(N == 12 || N == 24, "lengths 8, 12, 16, 24 and 32");
        stages<T, N, 0, S, 2, FWD>(a);
        stages<T, N, S, S, 2, FWD>(a);
        stages<T, N, 2 * S, S, 2, FWD>(a);
#pragma unroll
        for (int q = 0; q < S; ++q) {
            const Cplx<T> y0 = a[q], y1 = a[S + q], y2 = a[2 * S + q];
            if constexpr (sizeof(T) == 4) {
                // X[q + m S] = y0 + w^k y1 + w^2k y2, k = q + m S, four chained FMAs a part: as many instructions as a
                // radix-3 butterfly on twiddled y1, y2, and fewer roundings on the way to each result (N = 24:
                // 6.8e-8 of a line's norm, the butterfly 7.1e-8)
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const int k = q + m * S;
                    const T r1 = (T)cos_of<N>(k), i1 = FWD ? (T)(-sin_of<N>(k)) : (T)sin_of<N>(k);
                    const T r2 = (T)cos_of<N>(2 * k), i2 = FWD ? (T)(-sin_of<N>(2 * k)) : (T)sin_of<N>(2 * k);
                    a[k] = Cplx<T>{madd(-i2, y2.y, madd(r2, y2.x, madd(-i1, y1.y, madd(r1, y1.x, y0.x)))),
                                   madd(i2, y2.x, madd(r2, y2.y, madd(i1, y1.x, madd(r1, y1.y, y0.y))))};
                }
            } else {   // FP64, bound by its instructions: one radix-3 butterfly
                constexpr double c3 = FWD ? -cos_of<12>(1) : cos_of<12>(1);   // -+ sin(2 pi / 3)
                Cplx<T> t1 = y1, t2 = y2;
                if (q > 0) {
                    const T r1 = (T)cos_of<N>(q), i1 = FWD ? (T)(-sin_of<N>(q)) : (T)sin_of<N>(q);
                    const T r2 = (T)cos_of<N>(2 * q), i2 = FWD ? (T)(-sin_of<N>(2 * q)) : (T)sin_of<N>(2 * q);
                    t1 = Cplx<T>{fma(-i1, y1.y, r1 * y1.x), fma(i1, y1.x, r1 * y1.y)};
                    t2 = Cplx<T>{fma(-i2, y2.y, r2 * y2.x), fma(i2, y2.x, r2 * y2.y)};
                }
                const Cplx<T> p{t1.x + t2.x, t1.y + t2.y}, d{t1.x - t2.x, t1.y - t2.y};
                const Cplx<T> m{fma(T(-0.5), p.x, y0.x), fma(T(-0.5), p.y, y0.y)};
                a[q] = Cplx<T>{y0.x + p.x, y0.y + p.y};
                a[S + q] = Cplx<T>{fma((T)-c3, d.y, m.x), fma((T)c3, d.x, m.y)};
                a[2 * S + q] = Cplx<T>{fma((T)c3, d.y, m.x), fma((T)-c3, d.x, m.y)};
            }
        }
    }
}

}  // namespace cfft
}  // namespace dgfs
