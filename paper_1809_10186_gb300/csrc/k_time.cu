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

// Sums of NV <= 16 doubles per thread over the block (blockDim.x = 256) into out[0..NV). Lanes exchange halves of their
// values (sums with lane ^ 16, ^ 8, ..): 16 additions and shuffles a warp, five steps of all NV would take 5 NV.
template <int NV>
__device__ __forceinline__ void block_sum(const double (&v)[NV], double* s, double* out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double w[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) w[k] = k < NV ? v[k < NV ? k : 0] : 0.0;
#pragma unroll
    for (int h = 8; h > 0; h >>= 1) {   // value k ends on the lanes 2 k and 2 k + 1
        const bool up = lane & (2 * h);
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const double give = up ? w[k] : w[k + h], keep = up ? w[k + h] : w[k];
            w[k] = keep + __shfl_xor_sync(0xffffffffu, give, 2 * h);
        }
    }
    w[0] += __shfl_xor_sync(0xffffffffu, w[0], 1);
    __syncthreads();   // s may hold the previous reduction
    const int k = lane >> 1;
    if ((lane & 1) == 0 && k < NV) s[warp * NV + k] = w[0];
    __syncthreads();
    if (threadIdx.x < NV) {
        double t = s[threadIdx.x];
        for (int q = 1; q < 8; ++q) t += s[q * NV + threadIdx.x];
        out[threadIdx.x] = t;
    }
}

constexpr int kMomentSlices = 8;
// The sums of all slices (slice r of the cluster's CTA r mod its CTAs, part[r NV ..]), added in order.
template <int NV>
__device__ __forceinline__ void cluster_total(cooperative_groups::cluster_group& cl, double* part, int slices, double* total) {
    cl.sync();
    if (threadIdx.x < NV) {
        double t = 0.0;
        for (int r = 0; r < slices; ++r) t += cl.map_shared_rank(part, r % cl.num_blocks())[r * NV + threadIdx.x];
        total[threadIdx.x] = t;
    }
    cl.sync();   // every CTA has read the partial sums before they are overwritten or their CTA exits
}

// FP64 arithmetic and latency bound this (2 FP64 FMAs per clock and SM, a logarithm per point). A node's points fall into
// up to eight slices, whose sums are formed alike whichever CTA has them: a thread takes four points of one z line
// at a time, their sums over z first, then one step per sum for the x and y factors. With few nodes the slices go to
// the CTAs of a cluster, with many to one CTA (launch_moments).
// 37 nodes at N = 16 52 us, 1000 546 us, 4000 at N = 8 374 us (a cluster of eight CTAs for every node: 89, 1450 and 3713 us;
// one CTA for every node and every sum at every point: 106, 660 and 551 us). What is left is the logarithm.
template <typename T>
__global__ void __launch_bounds__(256) k_moments(const T* __restrict__ f, int N, double L, int slices, double* __restrict__ out) {
    __shared__ double s[8 * 11], part[kMomentSlices * 11], tot[11];
    auto cl = cooperative_groups::this_cluster();
    const int ctas = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int64_t node = blockIdx.x / ctas, n3 = (int64_t)N * N * N;
    const int quads = (int)(n3 / 4), zq = N / 4;
    const T* fn = f + node * n3;
    const double dc = 2.0 * L / N, dv = dc * dc * dc;
    for (int r = rank; r < slices; r += ctas) {
        double a[4] = {0, 0, 0, 0};   // sum f, f c_x, f c_y, f c_z
        for (int q = r * 256 + threadIdx.x; q < quads; q += kMomentSlices * 256) {
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
        block_sum<4>(a, s, part + r * 4);
    }
    cluster_total<4>(cl, part, slices, tot);
    const double n = tot[0] * dv, ux = tot[1] * dv / n, uy = tot[2] * dv / n, uz = tot[3] * dv / n;
    for (int r = rank; r < slices; r += ctas) {
        // sum f d^2, f dx dx, f dy dy, f dz dz, f dx dy, f dx dz, f dy dz, f dx d^2, f dy d^2, f dz d^2, f ln f
        double b[11] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
        for (int q = r * 256 + threadIdx.x; q < quads; q += kMomentSlices * 256) {
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
        block_sum<11>(b, s, part + r * 11);
    }
    cluster_total<11>(cl, part, slices, tot);
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
    // slices with points, a power of two. CTAs per node: the rounds over the 152 SMs that the nodes take, and 15 % for a
    // cluster (150 nodes at N = 24, which fill the SMs once: 350 us in clusters of eight, 254 with one CTA
    // each; 37 nodes: 122 us in clusters of eight, 154 of four)
    const int quads = N * N * N / 4, slices = quads >= 256 * kMomentSlices ? kMomentSlices : (quads + 255) / 256;
    int ctas = 1;
    double best = (double)((B + 151) / 152);
    for (int c = 2; c <= slices; c *= 2)
        if (const double t = 1.15 * (double)((B * c + 151) / 152) / c; t <= best) {
            best = t;
            ctas = c;
        }
    for (int64_t b0 = 0; b0 < B; b0 += 1 << 27) {
        const int64_t nb = B - b0 < (1 << 27) ? B - b0 : (1 << 27);
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(nb * ctas));
        cfg.blockDim = dim3(256);
        cfg.stream = s;
        cudaLaunchAttribute cluster{};
        cluster.id = cudaLaunchAttributeClusterDimension;
        cluster.val.clusterDim.x = (unsigned)ctas;
        cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
        cfg.attrs = &cluster;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k_moments<T>, f + b0 * (int64_t)N * N * N, N, L, slices, out + b0 * 15);
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
