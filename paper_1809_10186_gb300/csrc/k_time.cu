// Space-homogeneous time stepping and velocity moments (arXiv:1809.10186, Sec. 3.3 eq. moments1
// and Sec. 3.5 eqs. SSPRK2, SSPRK3).
//
// k_rk_combine forms one SSP-RK stage, out = a u + b v + c q, elementwise over a batch of fields;
// k_moments reduces every node's field to its mid-point-rule moments n, u, T, P, q and Boltzmann's
// H = int f ln f (over f > 0) in FP64, one cluster of eight CTAs per node.
#include <cstdint>

#include <cooperative_groups.h>

#include "launchers.h"

namespace dgfs {

namespace {

template <typename T>
__global__ void k_rk_combine(int64_t n, double a, const T* __restrict__ u, double b, const T* __restrict__ v,
                             double c, const T* __restrict__ q, T* __restrict__ out, int* __restrict__ flags) {
    const T ta = (T)a, tb = (T)b, tc = (T)c;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        T r = ta * u[i] + tc * q[i];
        if (v) r += tb * v[i];
        if (!isfinite(r)) atomicOr(flags, 2);
        out[i] = r;
    }
}

// sum over the block of NV doubles per thread (blockDim.x = 256); the result is in s[0..NV) for thread 0
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV], double* s) {
#pragma unroll
    for (int k = 0; k < NV; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();   // s may hold the previous reduction
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < NV; ++k) s[warp * NV + k] = v[k];
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < 8; ++w)
#pragma unroll
            for (int k = 0; k < NV; ++k) s[k] += s[w * NV + k];
    __syncthreads();
}

// The sums of the CTAs of a cluster: s[0..NV) of every CTA becomes the total (ranks added in order).
template <int NV>
__device__ __forceinline__ void cluster_total(double* s, double* total) {
    auto cl = cooperative_groups::this_cluster();
    cl.sync();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (unsigned r = 0; r < cl.num_blocks(); ++r) t += cl.map_shared_rank(s, r)[threadIdx.x];
        total[threadIdx.x] = t;
    }
    cl.sync();   // every CTA has read the partial sums before they are overwritten or their CTA exits
}

// FP64 arithmetic and latency bound this (2 FP64 FMAs per clock and SM, a logarithm per point), so a node is
// spread over a cluster of eight CTAs and a thread takes four points of one z line at a time: their sums
// over z first, then one step per sum for the x and y factors. 37 nodes at N = 16: 84 us (one CTA per
// node, every sum at every point: 103 us); what is left is the logarithm.
constexpr int kMomentCtas = 8;
template <typename T>
__global__ void __cluster_dims__(kMomentCtas, 1, 1) __launch_bounds__(256)
k_moments(const T* __restrict__ f, int N, double L, double* __restrict__ out) {
    __shared__ double s[8 * 11], tot[11];
    const int64_t node = blockIdx.x / kMomentCtas, n3 = (int64_t)N * N * N;
    const int rank = blockIdx.x % kMomentCtas, quads = (int)(n3 / 4), zq = N / 4;
    const T* fn = f + node * n3;
    const double dc = 2.0 * L / N, dv = dc * dc * dc;
    double a[4] = {0, 0, 0, 0};   // sum f, f c_x, f c_y, f c_z
    for (int q = rank * 256 + threadIdx.x; q < quads; q += kMomentCtas * 256) {
        const int x = q / (zq * N), y = (q / zq) % N, z = 4 * (q % zq);
        double t0 = 0.0, t1 = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double fv = (double)fn[4 * (int64_t)q + k];
            t0 += fv;
            t1 = fma(fv, -L + (z + k + 0.5) * dc, t1);
        }
        a[0] += t0;
        a[1] = fma(t0, -L + (x + 0.5) * dc, a[1]);
        a[2] = fma(t0, -L + (y + 0.5) * dc, a[2]);
        a[3] += t1;
    }
    block_sum<4>(a, s);
    cluster_total<4>(s, tot);
    const double n = tot[0] * dv, ux = tot[1] * dv / n, uy = tot[2] * dv / n, uz = tot[3] * dv / n;
    // sum f d^2, f dx dx, f dy dy, f dz dz, f dx dy, f dx dz, f dy dz, f dx d^2, f dy d^2, f dz d^2, f ln f
    double b[11] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int q = rank * 256 + threadIdx.x; q < quads; q += kMomentCtas * 256) {
        const int x = q / (zq * N), y = (q / zq) % N, z = 4 * (q % zq);
        double t0 = 0.0, t1 = 0.0, t2 = 0.0, t3 = 0.0;   // sum over z of f dz^k
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double fv = (double)fn[4 * (int64_t)q + k], dz = -L + (z + k + 0.5) * dc - uz;
            const double g = fv * dz, h = g * dz;
            t0 += fv;
            t1 += g;
            t2 += h;
            t3 = fma(h, dz, t3);
            if (fv > 0.0) b[10] = fma(fv, log(fv), b[10]);
        }
        const double dx = -L + (x + 0.5) * dc - ux, dy = -L + (y + 0.5) * dc - uy, r2 = dx * dx + dy * dy;
        const double d2 = fma(t0, r2, t2);               // sum over z of f d^2
        b[0] += d2;
        b[1] = fma(t0, dx * dx, b[1]);
        b[2] = fma(t0, dy * dy, b[2]);
        b[3] += t2;
        b[4] = fma(t0, dx * dy, b[4]);
        b[5] = fma(t1, dx, b[5]);
        b[6] = fma(t1, dy, b[6]);
        b[7] = fma(d2, dx, b[7]);
        b[8] = fma(d2, dy, b[8]);
        b[9] += fma(t1, r2, t3);
    }
    block_sum<11>(b, s);
    cluster_total<11>(s, tot);
    __syncthreads();
    if (rank == 0 && threadIdx.x == 0) {
        double* o = out + node * 15;
        o[0] = n;
        o[1] = ux;
        o[2] = uy;
        o[3] = uz;
        o[4] = 2.0 / (3.0 * n) * tot[0] * dv;
        for (int k = 0; k < 6; ++k) o[5 + k] = 2.0 * tot[1 + k] * dv;
        for (int k = 0; k < 3; ++k) o[11 + k] = tot[7 + k] * dv;
        o[14] = tot[10] * dv;
    }
}

}  // namespace

template <typename T>
cudaError_t launch_rk_combine(int64_t n, double a, const T* u, double b, const T* v, double c, const T* q, T* out,
                              int* flags, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = (n + 255) / 256;
    k_rk_combine<T><<<(unsigned)(blocks < 152 * 16 ? blocks : 152 * 16), 256, 0, s>>>(n, a, u, b, v, c, q, out, flags);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_moments(const T* f, int N, double L, int64_t B, double* out, cudaStream_t s) {
    for (int64_t b0 = 0; b0 < B; b0 += 1 << 27) {
        const int64_t nb = B - b0 < (1 << 27) ? B - b0 : (1 << 27);
        k_moments<T><<<(unsigned)(nb * kMomentCtas), 256, 0, s>>>(f + b0 * (int64_t)N * N * N, N, L, out + b0 * 15);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template cudaError_t launch_rk_combine<float>(int64_t, double, const float*, double, const float*, double,
                                              const float*, float*, int*, cudaStream_t);
template cudaError_t launch_rk_combine<double>(int64_t, double, const double*, double, const double*, double,
                                               const double*, double*, int*, cudaStream_t);
template cudaError_t launch_moments<float>(const float*, int, double, int64_t, double*, cudaStream_t);
template cudaError_t launch_moments<double>(const double*, int, double, int64_t, double*, cudaStream_t);

}  // namespace dgfs
