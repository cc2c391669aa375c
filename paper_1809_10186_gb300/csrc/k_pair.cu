// Translate products with a transform per sphere pair (arXiv:1809.10186, Appendix eq. lowrank1): the FP32 form of
// dgfs_ssprk and dgfs_collide_dgamma, which keep its rounding bit for bit (every other call takes the shared
// translates of k_shift.cu). T_s f = IDFT(mu_s f^) with the separable multiplier mu_s; one complex inverse transform
// carries both translates of a pair, IDFT(mu_s f^ + i mu_-s f^) = T_s f + i T_-s f. Fields are plane-major ([kz][kx][ky]):
//   k_pair_load    f into a plane-major complex field (launch_dft3 transforms it)
//   k_pair_planes  per (node, r, pair, KZ planes): translate spectra formed while the x lines load, inverse
//                  transforms along x and y                                                        -> Z
//   k_pair_sum     per (x, y) line: inverse z transform of every pair's line, products summed in registers -> P_r
// Lines are transformed in registers (fourier_dev.cuh). All radial points of a batch go in one launch of each
// kernel: an SSP-RK3 step of 37 nodes at N = 16 takes 0.35 ms (0.96 ms with two launches per radial point).
#include <cstdint>

#include "fourier_dev.cuh"
#include "launchers.h"

namespace dgfs {

namespace {

using fdev::line_fft;
using fdev::line_slot;
using fdev::mul_rn;

// X[n][z][x][y] = {f[n][x][y][z], 0}: a real field into a plane-major complex field
template <typename T>
__global__ void __launch_bounds__(256) k_pair_load(const T* __restrict__ f, int N, int64_t n3, Cplx<T>* __restrict__ X) {
    const int64_t n = blockIdx.y;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // plane-major index
    if (e >= n3) return;
    const int64_t n2 = (int64_t)N * N;
    const int z = (int)(e / n2), x = (int)((e / N) % N), y = (int)(e % N);
    const int64_t base = n * n3;
    X[n * n3 + e] = Cplx<T>{f[base + ((int64_t)x * N + y) * N + z], T(0)};
}

// the largest divisor of N with KZ N <= 128 threads
constexpr int planes_per_cta(int N) {
    int kz = 1;
    for (int d = 1; d <= N; ++d)
        if (N % d == 0 && d * N <= 128) kz = d;
    return kz;
}

template <typename T, int N>
struct PlaneGeo {
    static constexpr int KZ = planes_per_cta(N);               // planes per CTA (4 at N = 32 and 24, 8 at 16)
    static constexpr int NT = KZ * N;                          // one line per thread per pass
    static constexpr int P = N + 1;                            // padded row (complex elements)
    static constexpr size_t smem = (size_t)KZ * N * P * sizeof(Cplx<T>);
};

// Planes kz0 .. kz0 + KZ - 1 of the translate spectra mu f^ + i conj(mu) f^ of pair blockIdx.y, then inverse
// transforms along x and y; output Z[n][r][pair] plane-major for nr radial points (item n nr + r in blockIdx.z). grid
// (N / KZ, npairs, nodes nr). The x lines are read straight from global memory (consecutive threads take consecutive
// ky: coalesced), the y lines go through shared memory.
template <typename T, int N>
__global__ void __launch_bounds__(PlaneGeo<T, N>::NT)
    k_pair_planes(const Cplx<T>* __restrict__ Fh, const Cplx<T>* __restrict__ mu_r, const Cplx<T>* __restrict__ dftw, int nr,
                  Cplx<T>* __restrict__ X) {
    using G = PlaneGeo<T, N>;
    constexpr int KZ = G::KZ, NT = G::NT, P = G::P;
    constexpr int64_t n2 = (int64_t)N * N, n3 = n2 * N;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    Cplx<T>* S = reinterpret_cast<Cplx<T>*>(sm_raw);   // [KZ][N][P]
    __shared__ Cplx<T> tw[N];
    __shared__ Cplx<T> m[3 * N];
    const int tid = threadIdx.x, kz0 = blockIdx.x * KZ, p = blockIdx.y, npairs = gridDim.y;
    const unsigned node = nr > 1 ? blockIdx.z / (unsigned)nr : blockIdx.z;
    const int rl = (int)(blockIdx.z - node * (unsigned)nr);   // radial point of the item
    const int64_t item = blockIdx.z;
    const int pl = tid / N, ln = tid % N;
    if (tid < N) tw[tid] = dftw[N + tid];
    Cplx<T>* Xf = X + (item * npairs + p) * n3 + (int64_t)kz0 * n2;
    Cplx<T> v[N];
    for (int i = tid; i < 3 * N; i += NT) m[i] = mu_r[((int64_t)rl * npairs + p) * 3 * N + i];
    __syncthreads();
    const Cplx<T>* Fp = Fh + (int64_t)node * n3 + (int64_t)(kz0 + pl) * n2 + ln;
    // which product of a sum is rounded by itself is written out: it is part of the rounding that is kept
    const Cplx<T> my = m[N + ln], mz = m[2 * N + kz0 + pl];
    const Cplx<T> myz{fma(my.x, mz.x, -mul_rn(my.y, mz.y)), fma(my.y, mz.x, mul_rn(my.x, mz.y))};
#pragma unroll
    for (int kx = 0; kx < N; ++kx) {
        const Cplx<T> mx = m[kx], fv = Fp[kx * N];
        const T a = fma(mx.x, myz.x, -mul_rn(mx.y, myz.y)), b = fma(mx.x, myz.y, mul_rn(mx.y, myz.x));
        v[line_slot<N>(kx)] = Cplx<T>{fma(b, fv.x, fma(-a, fv.y, fma(a, fv.x, -mul_rn(b, fv.y)))),
                                      fma(b, fv.y, fma(a, fv.x, fma(a, fv.y, mul_rn(b, fv.x))))};
    }
    // x lines (fixed ky = ln)
    line_fft<T, N>(v, tw, false);
#pragma unroll
    for (int k = 0; k < N; ++k) S[(pl * N + k) * P + ln] = v[k];
    __syncthreads();
    // y lines (fixed x = ln)
#pragma unroll
    for (int k = 0; k < N; ++k) v[line_slot<N>(k)] = S[(pl * N + ln) * P + k];
    line_fft<T, N>(v, tw, false);
#pragma unroll
    for (int k = 0; k < N; ++k) S[(pl * N + ln) * P + k] = v[k];
    __syncthreads();
    for (int e = tid; e < KZ * N * N; e += NT) {
        const int q = e / (N * N), x = (e / N) % N, y = e % N;
        Xf[e] = S[(q * N + x) * P + y];
    }
}

// VHS radial products with a transform per pair (dgfs_ssprk and dgfs_collide_dgamma of FP32 plans, which
// keep this arithmetic bit for bit; every other call takes the shared translates of k_shift.cu): for
// z-line (x, y) of node n, the inverse z transforms of every sphere point's translate lines give
//   P_r(x, y, z) = sum_p 2 w_p (T_s f)(T_-s f)
// summed in registers; P_r is written in the standard layout [x][y][z] through shared memory.
// grid (N^2 / 128, nodes, nr); Z plane-major [n][r][p][kz][x][y]; P_r = P + n stride + r N^3. All radial
// points of a batch in one launch: one launch per r left 74 CTAs at N = 16 and 37 nodes.
template <typename T, int N>
__global__ void __launch_bounds__(128) k_pair_sum(const Cplx<T>* __restrict__ Z, const Cplx<T>* __restrict__ dftw,
                                                       const T* __restrict__ wsig, int npairs,
                                                       int64_t node_stride, T* __restrict__ P) {
    constexpr int64_t n2 = (int64_t)N * N, n3 = n2 * N;
    constexpr int LINES = 128;
    __shared__ Cplx<T> tw[N];
    __shared__ T tile[LINES * (N + 1)];
    if (threadIdx.x < N) tw[threadIdx.x] = dftw[N + threadIdx.x];
    __syncthreads();
    const int64_t l0 = (int64_t)blockIdx.x * LINES, l = l0 + threadIdx.x;
    const int64_t n = blockIdx.y, item = n * gridDim.z + blockIdx.z;
    T acc[N];
#pragma unroll
    for (int k = 0; k < N; ++k) acc[k] = T(0);
    Cplx<T> v[N];
    if (l < n2) {
        for (int p = 0; p < npairs; ++p) {
            const T w = wsig[p] * T(2);
            const Cplx<T>* z = Z + (item * npairs + p) * n3 + l;
#pragma unroll
            for (int k = 0; k < N; ++k) v[line_slot<N>(k)] = z[k * n2];
            line_fft<T, N>(v, tw, false);
#pragma unroll
            for (int k = 0; k < N; ++k) acc[k] = fma(w * v[k].x, v[k].y, acc[k]);
        }
#pragma unroll
        for (int k = 0; k < N; ++k) tile[threadIdx.x * (N + 1) + k] = acc[k];
    }
    __syncthreads();
    const int nl = (int)((n2 - l0) < LINES ? (n2 - l0) : LINES);
    T* out = P + n * node_stride + blockIdx.z * n3 + l0 * N;
    for (int e = threadIdx.x; e < nl * N; e += LINES) out[e] = tile[(e / N) * (N + 1) + e % N];
}

template <int N>
cudaError_t planes_n(const Cplx<float>* Fh, const Cplx<float>* mu_r, const Cplx<float>* dftw, int npairs, int nr, int64_t nodes,
                     Cplx<float>* Z, cudaStream_t s) {
    using G = PlaneGeo<float, N>;
    static_assert(G::smem <= 48 * 1024, "static shared memory limit");
    k_pair_planes<float, N><<<dim3(N / G::KZ, (unsigned)npairs, (unsigned)(nodes * nr)), G::NT, G::smem, s>>>(Fh, mu_r, dftw, nr, Z);
    return cudaGetLastError();
}

template <int N>
cudaError_t sum_n(const Cplx<float>* Z, const Cplx<float>* dftw, const float* wsig, int npairs, int nr, int64_t nodes,
                  int64_t node_stride, float* P, cudaStream_t s) {
    k_pair_sum<float, N><<<dim3((N * N + 127) / 128, (unsigned)nodes, (unsigned)nr), 128, 0, s>>>(Z, dftw, wsig, npairs, node_stride,
                                                                                             P);
    return cudaGetLastError();
}

}  // namespace

#define DGFS_BY_N(CALL)                                   \
    if (nodes <= 0) return cudaSuccess;                   \
    if (nodes * nr > 65535) return cudaErrorInvalidValue; \
    if (N == 8) return CALL(8);                           \
    if (N == 12) return CALL(12);                         \
    if (N == 16) return CALL(16);                         \
    if (N == 24) return CALL(24);                         \
    if (N == 32) return CALL(32);                         \
    return cudaErrorInvalidValue

cudaError_t launch_pair_load(const float* f, int N, int64_t nodes, Cplx<float>* X, cudaStream_t s) {
    if (nodes <= 0) return cudaSuccess;
    if (nodes > 65535) return cudaErrorInvalidValue;
    const int64_t n3 = (int64_t)N * N * N;
    k_pair_load<float><<<dim3((unsigned)((n3 + 255) / 256), (unsigned)nodes), 256, 0, s>>>(f, N, n3, X);
    return cudaGetLastError();
}

cudaError_t launch_pair_planes(const Cplx<float>* Fh, const Cplx<float>* mu_r, const Cplx<float>* dftw, int N, int npairs, int nr,
                               int64_t nodes, Cplx<float>* Z, cudaStream_t s) {
#define CALL(n) planes_n<n>(Fh, mu_r, dftw, npairs, nr, nodes, Z, s)
    DGFS_BY_N(CALL);
#undef CALL
}

cudaError_t launch_pair_sum(const Cplx<float>* Z, const Cplx<float>* dftw, const float* wsig, int N, int npairs, int nr, int64_t nodes,
                            int64_t node_stride, float* P, cudaStream_t s) {
#define CALL(n) sum_n<n>(Z, dftw, wsig, npairs, nr, nodes, node_stride, P, s)
    DGFS_BY_N(CALL);
#undef CALL
}

}  // namespace dgfs
