// Device helpers of the shared-shift kernels (k_shift.cu, k_shift_sum.cu): half-spectrum fields
// [x][ky][kz], kz = 0 .. N/2 - 1, with the spectra of kz = 0 and kz = N/2 in the two parts of slot kz = 0.
#pragma once

#include "fft_const.cuh"
#include "shift.h"

namespace dgfs {
namespace shdev {

using fdev::line_slot;

template <typename T> struct Pair2;
template <> struct Pair2<float> { using type = float2; };
template <> struct Pair2<double> { using type = double2; };
template <typename T>
__device__ __forceinline__ Cplx<T> ld(const Cplx<T>* p) {
    const typename Pair2<T>::type v = *reinterpret_cast<const typename Pair2<T>::type*>(p);
    return Cplx<T>{v.x, v.y};
}
template <typename T>
__device__ __forceinline__ Cplx<T> ldg(const Cplx<T>* p) {
    const typename Pair2<T>::type v = __ldg(reinterpret_cast<const typename Pair2<T>::type*>(p));
    return Cplx<T>{v.x, v.y};
}
template <typename T>
__device__ __forceinline__ void st(Cplx<T>* p, Cplx<T> c) {
    typename Pair2<T>::type v;
    v.x = c.x;
    v.y = c.y;
    *reinterpret_cast<typename Pair2<T>::type*>(p) = v;
}

// two consecutive complex values from an even index (one 16-byte access in FP32)
template <bool GLOBAL>
__device__ __forceinline__ void ld_two(const Cplx<float>* p, Cplx<float>& a, Cplx<float>& b) {
    const float4 v = GLOBAL ? __ldg(reinterpret_cast<const float4*>(p)) : *reinterpret_cast<const float4*>(p);
    a = Cplx<float>{v.x, v.y};
    b = Cplx<float>{v.z, v.w};
}
template <bool GLOBAL>
__device__ __forceinline__ void ld_two(const Cplx<double>* p, Cplx<double>& a, Cplx<double>& b) {
    a = GLOBAL ? ldg(p) : ld(p);
    b = GLOBAL ? ldg(p + 1) : ld(p + 1);
}

template <typename T>
__device__ __forceinline__ Cplx<T> cmul(Cplx<T> a, T br, T bi) {
    return Cplx<T>{fma(-a.y, bi, a.x * br), fma(a.x, bi, a.y * br)};
}

// Row pitch (complex elements) of the y-translated fields in shared memory: a thread's kz row starts
// 16-byte aligned and eight consecutive rows fall into different 16-byte bank groups.
template <typename T, int N>
__host__ __device__ constexpr int row_pitch() {
    if (sizeof(T) == 8) return N / 2 + 1;
    return N == 32 ? 18 : N == 24 ? 14 : N == 16 ? 10 : 6;
}

// A y line of a half-spectrum plane (element ky at src[ky N/2]) times the y multiplier of a shift: row of the
// shift table (-1: no shift), neg: the opposite shift.
template <typename T, int N>
__device__ __forceinline__ void load_y_line(const Cplx<T>* src, const Cplx<T>* mu_r, int row, int neg, Cplx<T> (&v)[N]) {
    constexpr int NH = N / 2, MP = shift_mu_pitch(N);
#pragma unroll
    for (int k = 0; k < N; ++k) v[line_slot<N>(k)] = ldg(src + k * NH);
    if (row >= 0) {
        const Cplx<T>* m = mu_r + (int64_t) row * MP;
        const T sg = neg ? T(-1) : T(1);
#pragma unroll
        for (int k2 = 0; k2 < NH; k2 += 2) {
            Cplx<T> w2[2];
            ld_two<true>(m + k2, w2[0], w2[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int k = k2 + h;
                if (k == 0) continue;
                const T wi = sg * w2[h].y;
                v[line_slot<N>(k)] = cmul(v[line_slot<N>(k)], w2[h].x, wi);
                v[line_slot<N>(N - k)] = cmul(v[line_slot<N>(N - k)], w2[h].x, -wi);
            }
        }
        const T wn = ldg(m + NH).x;
        v[line_slot<N>(NH)].x *= wn;
        v[line_slot<N>(NH)].y *= wn;
    }
}

// The z line of T_s f + i T_-s g from the half spectra at zp (+s) and zm (-s, the conjugate phase).
template <typename T, int N>
__device__ __forceinline__ void load_z_line(const Cplx<T>* zp, const Cplx<T>* zm, const Cplx<T>* mu_r, int row, int neg,
                                            Cplx<T> (&v)[N]) {
    constexpr int NH = N / 2, MP = shift_mu_pitch(N);
    const bool zs = row >= 0;
    const Cplx<T>* m = mu_r + (int64_t) (zs ? row : 0) * MP;
    const T sg = neg ? T(-1) : T(1);
#pragma unroll
    for (int k2 = 0; k2 < NH; k2 += 2) {
        Cplx<T> a2[2], b2[2], w2[2];
        ld_two<false>(zp + k2, a2[0], a2[1]);
        ld_two<false>(zm + k2, b2[0], b2[1]);
        if (zs) ld_two<true>(m + k2, w2[0], w2[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = k2 + h;
            Cplx<T> a = a2[h], b = b2[h];
            if (k == 0) {   // kz = 0 and kz = N/2, both real
                const T wn = zs ? ldg(m + NH).x : T(1);
                v[0] = Cplx<T>{a.x, b.x};
                v[line_slot<N>(NH)] = Cplx<T>{wn * a.y, wn * b.y};
            } else {
                if (zs) {
                    const T wi = sg * w2[h].y;
                    a = cmul(a, w2[h].x, wi);
                    b = cmul(b, w2[h].x, -wi);
                }
                v[line_slot<N>(k)] = Cplx<T>{a.x - b.y, a.y + b.x};
                v[line_slot<N>(N - k)] = Cplx<T>{a.x + b.y, b.x - a.y};
            }
        }
    }
}

// half spectra of the two real lines that v's parts carried through a forward transform; put takes
// the real part's, then the imaginary part's
template <typename T, int N, typename F>
__device__ __forceinline__ void split_line(const Cplx<T> (&v)[N], F put) {
    constexpr int NH = N / 2;
    put(0, Cplx<T>{v[0].x, v[NH].x}, Cplx<T>{v[0].y, v[NH].y});
#pragma unroll
    for (int k = 1; k < NH; ++k) {
        const Cplx<T> p = v[k], m = v[N - k];
        put(k, Cplx<T>{T(0.5) * (p.x + m.x), T(0.5) * (p.y - m.y)}, Cplx<T>{T(0.5) * (p.y + m.y), T(0.5) * (m.x - p.x)});
    }
}

// A forward-transformed y line of a real field's half spectrum (slot kz) into the field at o (element ky at
// o[ky N/2]); the plane kz = 0 folded: ky = 0 .. N/2 - 1 of kz = 0, then of kz = N/2, the real values at ky = 0 and N/2
// packed in the slots ky = 0, so that a multiplier by k acts on every slot but those two by itself.
template <typename T, int N>
__device__ __forceinline__ void store_folded(const Cplx<T> (&w)[N], int kz, Cplx<T>* o) {
    constexpr int NH = N / 2;
    if (kz > 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) st(o + k * NH, w[k]);
    } else {
        split_line<T, N>(w, [&](int k, Cplx<T> a, Cplx<T> b) {
            st(o + k * NH, a);
            st(o + (NH + k) * NH, b);
        });
    }
}

}  // namespace shdev
}  // namespace dgfs
