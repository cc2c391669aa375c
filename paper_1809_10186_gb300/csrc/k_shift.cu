// Translate products of the CUDA-core plans (FP32, FP64; arXiv:1809.10186, Appendix eq. lowrank1):
//   P_r = sum_p w_p [(T_s f)(T_-s g) + (T_-s f)(T_s g)],   s = c_r sigma_p / 2,
// with the translates taken in Fourier space, one axis after the other, and every translate that
// several sphere points share taken once. T_s is separable, T_s = X(s_x) Y(s_y) Z(s_z), and the points
// of a symmetric rule have few distinct components: the 38 points of M = 38 have 8 nonzero signed s_x
// and 25 distinct (s_x, s_y). Per radial point, in lines of one axis (complex, N points; the spectra of
// real fields are kept for kz >= 0 only), a separate transform per pair took 57 N^2 lines; this takes
// 4 N^2 (x) + 12.5 N^2 (y) + 19 N^2 (z; T_s f + i T_-s g share one line).
//
//   k_shift_forward   (y, z) spectra of every x plane of f                                  -> G
//   k_shift_x         x spectra, then per r and signed s_x: phase, inverse x transform      -> H
//   k_shift_products  per (node, r, XC planes x): per (s_x, s_y): phase, inverse y transform into
//                     shared memory; per pair: phase, inverse z transform of one line per thread,
//                     product summed in registers; P_r (or its (y, z) spectra, for a stage in spectra) written once
//
// Measured (GB300, FP32, N = 32, M = 38, 256 nodes, whole Q): 8.35 ms, 22.2 ms with a transform of its own
// per pair (two launches per radial point, 9.5 MB of spectra through DRAM per radial point and node
// against 2.2 MB here); N = 16, M = 6, FP64, one node: 0.17 ms, 0.97 ms before. k_shift_products takes 77 %
// of the FP32 step: 2.45 instructions a cycle (61 % of the issue slots), 49 % of the FMA pipe (ncu, 40 nodes); k_shift_x
// 15 %, at 82 % of the DRAM throughput.
//
// Half spectra: kz = 0 .. N/2 - 1, with the spectra of kz = 0 and kz = N/2 (both of real (x, y)
// fields, which x and y translates keep real) in the real and imaginary part of slot kz = 0.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdint>
#include <map>

#include "shift.h"
#include "shift_dev.cuh"

namespace dgfs {

namespace {

// The relative loss of a round trip through FP32 lines of N points, 1 - (mean diagonal of inverse times forward
// line / N), from the rounding of their twiddles alone (fft_const.cuh): |w| of the rounded ones is below 1 on
// average. 0.8e-8 (N = 8), 1.2e-8, 2.7e-8, 1.4e-8, 4.6e-8 (N = 32).
double line_loss(int N) {
    using C = std::complex<double>;
    auto w = [N](int k, int n) {   // e^{-2 pi i k / n} in FP32 (the inverse takes the conjugate)
        const double a = 2.0 * 3.14159265358979323846 * (k % n) / n;
        const bool exact = n == 8 && N == 24;   // plus_half_root
        auto f32 = [&](double v) { return std::fabs(v) < 1e-9 ? 0.0 : exact ? v : (double)(float)v; };
        return C(f32(std::cos(a)), -f32(std::sin(a)));
    };
    // the lines' linear map on x, decimation in time
    auto line = [&](auto&& self, const std::vector<C>& x, bool fwd) -> std::vector<C> {
        const int n = (int)x.size(), R = n % 3 == 0 ? 3 : 2, S = n / R;
        if (n == 1) return x;
        std::vector<std::vector<C>> y(R);
        for (int j = 0; j < R; ++j) {
            std::vector<C> s(S);
            for (int i = 0; i < S; ++i) s[i] = x[R * i + j];
            y[j] = self(self, s, fwd);
        }
        std::vector<C> out(n);
        for (int k = 0; k < n; ++k)
            for (int j = 0; j < R; ++j) {
                // radix 2 takes +- the twiddle of k < n / 2
                const C t = R == 2 ? (j && k >= S ? -1.0 : 1.0) * w(j * (k % S), n) : w(j * k, n);
                out[k] += (fwd ? t : std::conj(t)) * y[j][k % S];
            }
        return out;
    };
    double d = 0.0;
    for (int j = 0; j < N; ++j) {
        std::vector<C> e(N);
        e[j] = 1.0;
        d += line(line, line(line, e, true), false)[j].real() / N;
    }
    return 1.0 - d / N;
}

// FP32: constants that make the rounding of the tables, scales and twiddles a common factor of gain and loss, which
// cancel to a tenth of their size in Q (1e-7 of difference shows as 1e-6 of ||Q||). Against exact arithmetic
//   - an operand carries the FP32 forward scale 1/N^2 and, when it is translated along x, 1/N; 1 - line_loss per
//     axis that it went forward and back; the loss's operand always all three;
//   - the weights are rounded, |mu| of the rounded phases is not 1, and the loss weight is rounded.
// The first line goes into the weights, pair by pair; the factor by which what is left changes the gain of a Maxwellian of
// thermal speed L / sqrt(1.5 N) (3.5 of them at N = 8, 7 at N = 32), against the one of its loss, into p.balance, a
// factor of the radial tables. The weights take a common factor in [1, 2) by which all of them round well.
void balance_constants(const HostPlan& h, ShiftProgram& p) {
    auto f32 = [](double v) { return (double)(float)v; };
    const int N = h.N, Nr = h.Nrho, np = h.npairs, NH = N / 2;
    const size_t n3 = (size_t)N * N * N;
    const double ll = line_loss(N), syz = f32(1.0 / ((double)N * N)) * N * N, sx = f32(1.0 / N) * N;
    std::vector<double> a2(N);
    auto sk = [N](int q) { return q < N / 2 ? q : q - N; };
    for (int q = 0; q < N; ++q) {
        const double t = 3.14159265358979323846 * sk(q);
        a2[q] = std::exp(-0.5 * t * t / (1.5 * N));   // |f^|^2
    }
    std::vector<double> rho(Nr);
    for (int r = 0; r < Nr; ++r) rho[r] = 4.0 * 3.14159265358979323846 * h.b * std::pow(h.cr[r], h.gamma + 2.0);
    double lw = 0.0, lr = 0.0;   // loss: exact, with the FP32 weight
    for (size_t i = 0; i < n3; ++i) {
        double g = h.aniso ? h.GLa[i] : 0.0;
        for (int r = 0; r < Nr && !h.aniso; ++r) g += rho[r] * h.Lr[(size_t)r * n3 + i];
        const double m = a2[i / ((size_t)N * N)] * a2[(i / N) % N] * a2[i % N];
        lw += m * g;
        lr += m * f32(g);
    }
    for (int q = 0; q < np; ++q) {
        const bool tx = h.sig[3 * q] != 0.0;
        const double s = syz * (tx ? sx : 1.0);
        p.excess[q] = syz * sx / (s * s) * (1.0 + 2.0 * (tx ? 3 : 2) * ll);
    }
    double common = 1.0, best = -1.0;
    for (int i = 0; i < 4096 && !h.aniso; ++i) {   // (VSS: the weight is part of the kernel factor)
        const double c = 1.0 + i / 4096.0;
        double e = 0.0;
        for (int q = 0; q < np; ++q) {
            const double w = c * h.wsig[q] * p.excess[q], d = f32(w) / w - 1.0;
            e += h.wsig[q] * d * d;
        }
        if (best < 0.0 || e < best) {
            best = e;
            common = c;
        }
    }
    // gain of the Maxwellian at X^3 points of an octant (even along each axis): exact (g), with the rounded constants
    // (gr), and those on the compressed radial kernel with its factors at k = 0 rounded (gp)
    constexpr int X = 6;
    std::vector<double> g(X * X * X, 0.0), gr(g), gp(g), cosx(X * (size_t)N), sinx(cosx);
    for (int i = 0; i < X; ++i)
        for (int k = 0; k < N; ++k) {
            const double ang = 3.14159265358979323846 * sk(k) * (0.15 + 0.3 * i) / std::sqrt(1.5 * N), a = std::sqrt(a2[k]);
            cosx[i * N + k] = a * std::cos(ang);
            sinx[i * N + k] = k == NH ? 0.0 : a * std::sin(ang);
        }
    // the compressed radial kernel at k = 0, and with its factors rounded (either may pass zero at a low rank)
    std::vector<double> rad(Nr, 1.0), proj(Nr, 1.0);
    for (int r = 0; r < Nr && !h.aniso; ++r) {
        rad[r] = proj[r] = 0.0;
        for (int s = 0; s < h.rank; ++s) {
            const double u = h.Uk[(size_t)s * n3], c = h.Vr[(size_t)s * Nr + r];
            rad[r] += u * c;
            proj[r] += f32(u) * f32(c);
        }
    }
    for (int q = 0; q < np; ++q) {
        p.wsig[q] = common * h.wsig[q] * p.excess[q];
        const double rounded = h.aniso ? 1.0 : common * f32(p.wsig[q]) / p.wsig[q];
        for (int r = 0; r < Nr; ++r) {
            const double mass = h.aniso ? h.Fa[((size_t)r * np + q) * n3] : h.wsig[q] * h.wr[r] * rho[r];
            double ex[3][X], rd[3][X];   // (T_s f)(T_-s f) along each axis
            for (int ax = 0; ax < 3; ++ax) {
                const double* m = &h.mu[(((size_t)r * np + q) * 3 + ax) * N * 2];
                for (int i = 0; i < X; ++i) {
                    double c = 0.0, d = 0.0, cr = 0.0, dr = 0.0;
                    for (int k = 0; k < N; ++k) {
                        const double re = m[2 * k], im = k == NH ? 0.0 : m[2 * k + 1];
                        c += cosx[i * N + k] * re;
                        d += sinx[i * N + k] * im;
                        cr += cosx[i * N + k] * f32(re);
                        dr += sinx[i * N + k] * f32(im);
                    }
                    ex[ax][i] = (c - d) * (c + d);
                    rd[ax][i] = (cr - dr) * (cr + dr);
                }
            }
            for (int i = 0; i < X * X * X; ++i) {
                const int x = i / (X * X), y = i / X % X, z = i % X;
                g[i] += rad[r] * mass * ex[0][x] * ex[1][y] * ex[2][z];
                const double v = mass * rounded * rd[0][x] * rd[1][y] * rd[2][z];
                gr[i] += rad[r] * v;
                gp[i] += proj[r] * v;
            }
        }
    }
    double gg = 0.0, ggr = 0.0, ggp = 0.0;
    for (size_t i = 0; i < g.size(); ++i) {
        gg += g[i] * g[i];
        ggr += g[i] * gr[i];
        ggp += g[i] * gp[i];
    }
    // rounded constants move it by 1e-7; anything else (a kernel without a gain or a loss) is left alone
    auto factor = [&](double gain) {
        const double x = lr / lw * (gg / gain) * common;
        return (std::fabs(x - 1.0) < 1e-4 ? x : 1.0) / common;
    };
    p.balance = factor(ggr);
    p.project = factor(ggp);
}

}  // namespace

void build_shift_program(const HostPlan& h, bool fp32, ShiftProgram& p) {
    const int N = h.N, np = h.npairs, MP = shift_mu_pitch(N);
    p = ShiftProgram();
    p.wsig = h.wsig;
    p.excess.assign(np, 1.0);
    if (fp32) balance_constants(h, p);
    // FP32 results leave the last transform by a power of two; the tables carry the rest of 1 / N^3
    const double n3d = (double)N * N * N, exact = fp32 ? 1.0 / (n3d * shift_result_scale(N, false)) : 1.0;
    std::map<double, int> rows, xs;
    std::vector<std::pair<int, int>> at;   // a (pair, axis) that carries each row
    for (int q = 0; q < np; ++q)
        for (int a = 0; a < 3; ++a) {
            const double v = std::fabs(h.sig[3 * q + a]);
            if (v == 0.0) continue;
            if (rows.emplace(v, (int)rows.size()).second) at.push_back({q, a});
            if (a == 0 && xs.emplace(v, (int)xs.size()).second) p.xrows.push_back(rows[v]);
        }
    p.nrows = (int)rows.size();
    p.nx = (int)xs.size();
    p.mu.assign((size_t)h.Nrho * p.nrows * MP * 2, 0.0);
    for (int r = 0; r < h.Nrho; ++r)
        for (int d = 0; d < p.nrows; ++d) {
            const double* m = &h.mu[(((size_t)r * np + at[d].first) * 3 + at[d].second) * N * 2];
            const double sg = h.sig[3 * at[d].first + at[d].second] < 0 ? -1.0 : 1.0;
            double* o = &p.mu[((size_t)r * p.nrows + d) * MP * 2];
            for (int k = 0; k <= N / 2; ++k) {
                o[2 * k] = m[2 * k];
                o[2 * k + 1] = k == N / 2 ? 0.0 : sg * m[2 * k + 1];
            }
        }
    if (!h.aniso) {
        const int nq2 = 3 * (N / 2) * (N / 2) + 1;
        const size_t n3 = (size_t)N * N * N;
        for (auto* t : {&p.sq, &p.kq, &p.kqd, &p.st, &p.kt}) t->assign((size_t)h.Nrho * nq2, 0.0);
        const double gain = exact * p.balance;
        std::vector<int64_t> at_q(nq2, -1);   // a mode of each |k|^2
        auto sk = [N](int q) { return q < N / 2 ? q : q - N; };
        for (size_t i = 0; i < n3; ++i) {
            const int kx = sk((int)(i / ((size_t)N * N))), ky = sk((int)((i / N) % N)), kz = sk((int)(i % N));
            at_q[kx * kx + ky * ky + kz * kz] = (int64_t)i;
        }
        for (int r = 0; r < h.Nrho; ++r) {
            const double wr = h.wr[r] * 4.0 * 3.14159265358979323846 * h.b * std::pow(h.cr[r], h.gamma + 2.0);
            for (int q = 0; q < nq2; ++q) {
                if (at_q[q] < 0) continue;
                double v = 0.0;
                for (int s = 0; s < h.rank; ++s) v += h.Uk[(size_t)s * n3 + at_q[q]] * h.Vr[(size_t)s * h.Nrho + r];
                p.sq[(size_t)r * nq2 + q] = gain * v;
                p.kq[(size_t)r * nq2 + q] = gain * wr * v;
                p.kqd[(size_t)r * nq2 + q] = gain * std::log(h.cr[r]) * wr * v;
                p.st[(size_t)r * nq2 + q] = exact * v;
                p.kt[(size_t)r * nq2 + q] = exact * wr * v;
            }
        }
    }
    if (h.aniso)
        for (double& e : p.excess) e *= exact * p.balance;
    struct Key { double x, y, z; int q; };
    auto program = [&](bool both) {
        std::vector<Key> keys;
        for (int q = 0; q < np; ++q)
            for (int sg = 1; sg >= (both ? -1 : 1); sg -= 2)
                keys.push_back({sg * h.sig[3 * q], sg * h.sig[3 * q + 1], sg * h.sig[3 * q + 2], q});
        std::stable_sort(keys.begin(), keys.end(),
                         [](const Key& a, const Key& b) { return a.x != b.x ? a.x < b.x : a.y < b.y; });
        std::vector<ShiftEntry> out;
        for (size_t i = 0; i < keys.size(); ++i) {
            const Key& k = keys[i];
            auto row = [&](double v) { return v == 0.0 ? -1 : rows[std::fabs(v)]; };
            const int fx = k.x == 0.0 ? -1 : 2 * xs[std::fabs(k.x)], neg = k.x < 0;
            out.push_back({fx < 0 ? -1 : fx + neg, fx < 0 ? -1 : fx + 1 - neg, row(k.y), k.y < 0, row(k.z), k.z < 0, k.q,
                           i == 0 || k.x != keys[i - 1].x || k.y != keys[i - 1].y});
        }
        return out;
    };
    p.quad = program(false);
    p.bil = program(true);
}

namespace {

using namespace shdev;

// ---- forward (y, z) spectra ------------------------------------------------------------------

template <int N>
struct ForwardGeo {
    // planes per CTA, N/2 lines each: about one warp, so that one node already spreads over many SMs
    static constexpr int PX = N == 32 ? 2 : N == 12 ? 6 : N == 8 ? 8 : 4;
    static constexpr int NT = PX * N / 2;
    static constexpr int PITCH = N / 2 + 1;
};

// grid (N / PX, nodes). Lines along z of rows y and y + N/2 as real and imaginary part, separated into
// half spectra; then lines along y of every slot kz. Blocks y >= nodes: the fields P to folded spectra W.
// Bound by its loads and stores: 4-byte loads (64 per thread) left it at 4.1 TB/s over the P_r of 230 nodes at N = 32;
// with 16-byte loads, all in flight, the ragged batch of 1152 F16S nodes takes 8716 us (8905 before), FP32 calls 0.5 % less.
template <typename T, int N>
__global__ void __launch_bounds__(ForwardGeo<N>::NT)
k_shift_forward(const T* __restrict__ f, const T* __restrict__ b, const int64_t* __restrict__ offs, int nodes,
                const T* __restrict__ P, Cplx<T>* __restrict__ W, Cplx<T>* __restrict__ G) {
    using Geo = ForwardGeo<N>;
    constexpr int NH = N / 2, PX = Geo::PX, NT = Geo::NT, PITCH = Geo::PITCH;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T* rows = reinterpret_cast<T*>(sm_raw);                // [PX][N][N + 1], then S overwrites it
    Cplx<T>* S = reinterpret_cast<Cplx<T>*>(sm_raw);       // [PX][N][PITCH]
    const int tid = threadIdx.x, x0 = blockIdx.x * PX, pl = tid / NH, j = tid % NH;
    const int64_t n3 = (int64_t)N * N * N;
    const bool folded = (int)blockIdx.y >= nodes;
    const int64_t node = (int)blockIdx.y - (folded ? nodes : 0);
    const T* src = folded ? P : f;
    const int64_t base = (offs && !folded ? offs[node] : node * n3) + (int64_t)x0 * N * N;
    constexpr int V = 16 / (int)sizeof(T);   // values of one 16-byte load
    static_assert(N % V == 0 && PX * N * N % (V * NT) == 0, "whole vectors per thread");
    if (!(b && !folded) && (reinterpret_cast<uintptr_t>(src + base) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < PX * N * N / (V * NT); ++i) {
            const int e = (i * NT + tid) * V;
            alignas(16) T q[V];
            *reinterpret_cast<uint4*>(q) = __ldg(reinterpret_cast<const uint4*>(src + base + e));
#pragma unroll
            for (int k = 0; k < V; ++k) rows[(e / N) * (N + 1) + e % N + k] = q[k];
        }
    } else {   // a product, or a pointer off a 16-byte boundary
        for (int e = tid; e < PX * N * N; e += NT) rows[(e / N) * (N + 1) + e % N] = b && !folded ? src[base + e] * b[base + e] : src[base + e];
    }
    __syncthreads();
    Cplx<T> v[N];
#pragma unroll
    for (int z = 0; z < N; ++z)
        v[line_slot<N>(z)] = Cplx<T>{rows[(pl * N + j) * (N + 1) + z], rows[(pl * N + j + NH) * (N + 1) + z]};
    __syncthreads();
    cfft::line<T, N, true>(v);
    Cplx<T>* ra = S + (pl * N + j) * PITCH;
    Cplx<T>* rb = ra + NH * PITCH;
    st(ra, Cplx<T>{v[0].x, v[NH].x});
    st(rb, Cplx<T>{v[0].y, v[NH].y});
#pragma unroll
    for (int k = 1; k < NH; ++k) {
        const Cplx<T> p = v[k], m = v[N - k];
        st(ra + k, Cplx<T>{T(0.5) * (p.x + m.x), T(0.5) * (p.y - m.y)});
        st(rb + k, Cplx<T>{T(0.5) * (p.y + m.y), T(0.5) * (m.x - p.x)});
    }
    __syncthreads();
#pragma unroll
    for (int y = 0; y < N; ++y) v[line_slot<N>(y)] = ld(S + (pl * N + y) * PITCH + j);   // slot kz = j
    cfft::line<T, N, true>(v);
    const T sc = T(1) / (T(N) * T(N));
    Cplx<T>* g = (folded ? W : G) + node * (n3 / 2) + (int64_t)(x0 + pl) * N * NH + j;
    if (folded) {
        store_folded<T, N>(v, j, g);
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) st(g + k * NH, Cplx<T>{sc * v[k].x, sc * v[k].y});
    }
}

// ---- x translates ----------------------------------------------------------------------------

// One thread per column (ky, kz): the x spectrum of its line once, then for r = r0 + blockIdx.z RG .. and
// every signed x shift the phase and the inverse transform. grid (ceil(N^2 / 2 / NT), nodes, ceil(nr / RG)).
// Bound by its stores of H (1 MB per radial point and node at N = 32, M = 38).
template <typename T, int N, int NT>
__global__ void __launch_bounds__(NT)
k_shift_x(const Cplx<T>* __restrict__ G, const Cplx<T>* __restrict__ mu, const int* __restrict__ xrows, int nrows, int nx,
          int r0, int nr, int RG, Cplx<T>* __restrict__ H) {
    constexpr int NH = N / 2, COLS = N * NH, MP = shift_mu_pitch(N);
    constexpr int64_t FS = (int64_t)N * COLS;                // one half-spectrum field
    const int c = blockIdx.x * NT + threadIdx.x;
    if (c >= COLS) return;
    const int64_t node = blockIdx.y;
    Cplx<T> F[N];
    const Cplx<T>* g = G + node * FS + c;
#pragma unroll
    for (int x = 0; x < N; ++x) F[line_slot<N>(x)] = ldg(g + (int64_t)x * COLS);
    cfft::line<T, N, true>(F);
    const T sc = T(1) / T(N);
#pragma unroll
    for (int k = 0; k < N; ++k) F[k] = Cplx<T>{sc * F[k].x, sc * F[k].y};
    const int rl1 = min(nr, (int)(blockIdx.z + 1) * RG);
    for (int rl = blockIdx.z * RG; rl < rl1; ++rl) {
        Cplx<T>* h = H + (node * nr + rl) * (2 * nx) * FS + c;
        for (int fi = 0; fi < 2 * nx; ++fi, h += FS) {
            const Cplx<T>* m = mu + ((int64_t)(r0 + rl) * nrows + __ldg(xrows + (fi >> 1))) * MP;
            const T sg = fi & 1 ? T(-1) : T(1);
            Cplx<T> v[N];
            v[0] = F[0];
#pragma unroll
            for (int k = 1; k < NH; ++k) {
                const Cplx<T> w = ldg(m + k);
                v[line_slot<N>(k)] = cmul(F[k], w.x, sg * w.y);
                v[line_slot<N>(N - k)] = cmul(F[N - k], w.x, -sg * w.y);
            }
            const T wn = ldg(m + NH).x;
            v[line_slot<N>(NH)] = Cplx<T>{F[NH].x * wn, F[NH].y * wn};
            cfft::line<T, N, false>(v);
#pragma unroll
            for (int x = 0; x < N; ++x) st(h + (int64_t)x * COLS, v[x]);
        }
    }
}

// ---- y and z translates, products ------------------------------------------------------------

template <typename T, int N, int XC>
struct ProductGeo {
    static constexpr int NT = XC * N;                        // z lines; y lines: 2 XC N / 2
    static constexpr int PITCH = row_pitch<T, N>();
    static constexpr size_t smem = (size_t)2 * XC * N * PITCH * sizeof(Cplx<T>);
    // resident CTAs the registers are budgeted for (a line and its sums are 96 values at N = 32: with four
    // CTAs of 128 threads it spilled 100 bytes and measured 1 % slower than with three)
    static constexpr int MINB = sizeof(T) == 8 ? 1 : N == 32 ? 384 / NT : N == 24 ? 480 / NT : 768 / NT;
};

// grid (N / XC, nr, nodes); H [node][r][2 nx fields][x][ky][kz], G [node][x][ky][kz]
template <typename T, int N, int XC, bool FOLD>
__global__ void __launch_bounds__(ProductGeo<T, N, XC>::NT, ProductGeo<T, N, XC>::MINB)
k_shift_products(const Cplx<T>* __restrict__ Gf, const Cplx<T>* __restrict__ Hf, const Cplx<T>* __restrict__ Gg,
                 const Cplx<T>* __restrict__ Hg, const Cplx<T>* __restrict__ mu, const ShiftEntry* __restrict__ prog,
                 int nprog, T wscale, const T* __restrict__ wsig, int nrows, int nx, int r0, int64_t node_stride, T* __restrict__ P) {
    using Geo = ProductGeo<T, N, XC>;
    constexpr int NH = N / 2, PITCH = Geo::PITCH, NT = Geo::NT, MP = shift_mu_pitch(N);
    constexpr int64_t FS = (int64_t)N * N * NH, n3 = (int64_t)N * N * N;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    Cplx<T>* Y = reinterpret_cast<Cplx<T>*>(sm_raw);         // [sign][XC][y][PITCH]
    const int tid = threadIdx.x, x0 = blockIdx.x * XC, rl = blockIdx.y, nr = gridDim.y;
    const int64_t node = blockIdx.z;
    // this thread's y line: operand (0: +s of f, 1: -s of g), plane, kz
    const int op = tid / (XC * NH), ypl = (tid / NH) % XC, ykz = tid % NH;
    const int64_t ybase = (int64_t)(x0 + ypl) * N * NH + ykz;
    const Cplx<T>* Gy = (op ? Gg : Gf) + node * FS + ybase;
    const Cplx<T>* Hy = (op ? Hg : Hf) + (node * nr + rl) * (2 * nx) * FS + ybase;
    Cplx<T>* ydst = Y + ((op * XC + ypl) * N) * PITCH + ykz;
    // this thread's z line: plane tid / N, y = tid % N
    const Cplx<T>* zp = Y + tid * PITCH;
    const Cplx<T>* zm = Y + (NT + tid) * PITCH;
    const Cplx<T>* mu_r = mu + (int64_t)(r0 + rl) * nrows * MP;
    T acc[N];
#pragma unroll
    for (int z = 0; z < N; ++z) acc[z] = T(0);
    Cplx<T> v[N];
    for (int i = 0; i < nprog; ++i) {
        const ShiftEntry e = prog[i];
        if (e.newy) {
            const int fi = op ? e.fm : e.fp;
            load_y_line<T, N>(fi < 0 ? Gy : Hy + fi * FS, mu_r, e.yrow, e.yneg ^ op, v);
            cfft::line<T, N, false>(v);
            __syncthreads();   // the previous (s_x, s_y) has been read
#pragma unroll
            for (int y = 0; y < N; ++y) st(ydst + y * PITCH, v[y]);
            __syncthreads();
        }
        // z line of T_s f + i T_-s g from the half spectra a (+s) and b (-s, the conjugate phase)
        const T wgt = wscale * __ldg(wsig + e.pair);
        load_z_line<T, N>(zp, zm, mu_r, e.zrow, e.zneg, v);
        cfft::line<T, N, false>(v);
#pragma unroll
        for (int z = 0; z < N; ++z) acc[z] = fma(wgt * v[z].x, v[z].y, acc[z]);
    }
    T* tile = reinterpret_cast<T*>(sm_raw);                  // [NT][N + 1]
    __syncthreads();
#pragma unroll
    for (int z = 0; z < N; ++z) tile[tid * (N + 1) + z] = acc[z];
    __syncthreads();
    T* out = P + node * node_stride + rl * n3 + (int64_t)x0 * N * N;
    if constexpr (!FOLD) {   // P_r of the planes x0 .. x0 + XC - 1 (coalesced)
        for (int e = tid; e < NT * N; e += NT) out[e] = tile[(e / N) * (N + 1) + e % N];
        return;
    }
    // the (y, z) spectra of P_r, what the radial sum takes (k_shift_sum.cu): forward z of two rows (y, y + N/2) at a
    // time, forward y; half of the threads, 2 % of the kernel
    const int hpl = tid / NH, hj = tid % NH;
    const bool half = tid < NT / 2;
    if (half) {
        const T* ra = tile + (hpl * N + hj) * (N + 1);
        const T* rb = ra + NH * (N + 1);
#pragma unroll
        for (int z = 0; z < N; ++z) v[line_slot<N>(z)] = Cplx<T>{ra[z], rb[z]};
        cfft::line<T, N, true>(v);
    }
    __syncthreads();
    if (half)
        split_line<T, N>(v, [&](int k, Cplx<T> a, Cplx<T> b) {
            st(Y + (hpl * N + hj) * PITCH + k, a);
            st(Y + (hpl * N + hj + NH) * PITCH + k, b);
        });
    __syncthreads();
    if (half) {
#pragma unroll
        for (int y = 0; y < N; ++y) v[line_slot<N>(y)] = ld(Y + (hpl * N + y) * PITCH + hj);
        cfft::line<T, N, true>(v);
        store_folded<T, N>(v, hj, reinterpret_cast<Cplx<T>*>(out) + hpl * N * NH + hj);
    }
}

template <typename T, int N>
cudaError_t forward_n(const T* f, const T* b, const int64_t* offs, int64_t nodes, const T* P, int64_t fields, Cplx<T>* W, Cplx<T>* G,
                      cudaStream_t s) {
    using Geo = ForwardGeo<N>;
    constexpr size_t sm = (size_t)Geo::PX * N * Geo::PITCH * sizeof(Cplx<T>);
    k_shift_forward<T, N><<<dim3(N / Geo::PX, (unsigned)(nodes + fields)), Geo::NT, sm, s>>>(f, b, offs, (int)nodes, P, W, G);
    return cudaGetLastError();
}

template <typename T, int N>
cudaError_t shift_x_n(const ShiftDev<T>& d, const Cplx<T>* G, int r0, int nr, int64_t nodes, Cplx<T>* H, cudaStream_t s) {
    if (d.nx == 0 || nr == 0) return cudaSuccess;
    constexpr int COLS = N * N / 2, NT = COLS < 128 ? COLS : COLS % 128 ? 96 : 128;
    static_assert(COLS % NT == 0, "whole column blocks");
    // radial points per CTA (the x spectrum is formed once for them) while the launch fills the GPU
    // several times; a small batch takes one each, in one-warp CTAs, to reach more SMs
    const int64_t blocks = (int64_t)(COLS / NT) * nodes * nr;
    if (blocks >= 8192) {
        k_shift_x<T, N, NT><<<dim3(COLS / NT, (unsigned)nodes, (unsigned)((nr + 3) / 4)), NT, 0, s>>>(
            G, d.mu, d.xrows, d.nrows, d.nx, r0, nr, 4, H);
    } else {
        k_shift_x<T, N, 32><<<dim3((COLS + 31) / 32, (unsigned)nodes, (unsigned)nr), 32, 0, s>>>(
            G, d.mu, d.xrows, d.nrows, d.nx, r0, nr, 1, H);
    }
    return cudaGetLastError();
}

template <typename T, int N, int XC, bool FOLD>
cudaError_t products_x(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg, const Cplx<T>* Hg,
                       int r0, int nr, int64_t nodes, int64_t node_stride, T* P, cudaStream_t s) {
    using Geo = ProductGeo<T, N, XC>;
    auto kern = k_shift_products<T, N, XC, FOLD>;
    if (Geo::smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Geo::smem);
        if (e != cudaSuccess) return e;
    }
    const bool bil = Gg != nullptr;
    kern<<<dim3(N / XC, (unsigned)nr, (unsigned)nodes), Geo::NT, Geo::smem, s>>>(
        Gf, Hf, bil ? Gg : Gf, bil ? Hg : Hf, d.mu, bil ? d.bil : d.quad, bil ? d.nbil : d.nquad, bil ? T(1) : T(2), d.wsig,
        d.nrows, d.nx, r0, node_stride, P);
    return cudaGetLastError();
}

template <typename T, int N, bool FOLD>
cudaError_t products_n(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg, const Cplx<T>* Hg,
                       int r0, int nr, int64_t nodes, int64_t node_stride, T* P, cudaStream_t s) {
    constexpr int XC = N == 32 || N == 24 ? 4 : N == 12 ? 12 : 8;
    // two planes per CTA while whole CTAs of XC planes would not fill the 152 SMs about four deep
    if ((int64_t)(N / XC) * nr * nodes < 608)
        return products_x<T, N, 2, FOLD>(d, Gf, Hf, Gg, Hg, r0, nr, nodes, node_stride, P, s);
    return products_x<T, N, XC, FOLD>(d, Gf, Hf, Gg, Hg, r0, nr, nodes, node_stride, P, s);
}

}  // namespace

#define DGFS_BY_N(CALL)                       \
    if (nodes <= 0) return cudaSuccess;       \
    if (nodes > 65535) return cudaErrorInvalidValue; \
    if (N == 8) return CALL(8);               \
    if (N == 12) return CALL(12);             \
    if (N == 16) return CALL(16);             \
    if (N == 24) return CALL(24);             \
    if (N == 32) return CALL(32);             \
    return cudaErrorInvalidValue

template <typename T>
cudaError_t launch_shift_forward(const T* f, const T* b, const int64_t* offs, int N, int64_t nodes, Cplx<T>* G,
                                 cudaStream_t s) {
#define CALL(n) forward_n<T, n>(f, b, offs, nodes, nullptr, 0, nullptr, G, s)
    DGFS_BY_N(CALL);
#undef CALL
}

template <typename T>
cudaError_t launch_shift_folded(const T* P, int64_t fields, const T* f, const int64_t* offs, int N, int64_t nodes, Cplx<T>* W,
                                Cplx<T>* G, cudaStream_t s) {
    const int64_t n3 = (int64_t)N * N * N;
    int64_t f0 = 0;
    auto part = [&](int64_t lead, int64_t n) {
#define CALL(k) forward_n<T, k>(f, nullptr, offs, lead, P + f0 * n3, n, W + f0 * (n3 / 2), G, s)
        DGFS_BY_N(CALL);
#undef CALL
    };
    for (int64_t lead = nodes; f0 < fields; lead = 0) {   // grid.y limit
        const int64_t n = std::min<int64_t>(65535 - lead, fields - f0);
        const cudaError_t e = part(lead, n);
        if (e != cudaSuccess) return e;
        f0 += n;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_shift_x(const ShiftDev<T>& d, const Cplx<T>* G, int N, int r0, int nr, int64_t nodes, Cplx<T>* H,
                           cudaStream_t s) {
#define CALL(n) shift_x_n<T, n>(d, G, r0, nr, nodes, H, s)
    DGFS_BY_N(CALL);
#undef CALL
}

template <typename T>
cudaError_t launch_shift_products(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg,
                                  const Cplx<T>* Hg, int N, int r0, int nr, int64_t nodes, bool folded, int64_t node_stride,
                                  T* P, cudaStream_t s) {
#define CALL(n) (folded ? products_n<T, n, true> : products_n<T, n, false>)(d, Gf, Hf, Gg, Hg, r0, nr, nodes, node_stride, P, s)
    DGFS_BY_N(CALL);
#undef CALL
}

#define DGFS_SHIFT_INST(T)                                                                                            \
    template cudaError_t launch_shift_forward<T>(const T*, const T*, const int64_t*, int, int64_t, Cplx<T>*,               \
                                                 cudaStream_t);                                                       \
    template cudaError_t launch_shift_folded<T>(const T*, int64_t, const T*, const int64_t*, int, int64_t, Cplx<T>*,   \
                                                Cplx<T>*, cudaStream_t);                                              \
    template cudaError_t launch_shift_x<T>(const ShiftDev<T>&, const Cplx<T>*, int, int, int, int64_t, Cplx<T>*,      \
                                           cudaStream_t);                                                             \
    template cudaError_t launch_shift_products<T>(const ShiftDev<T>&, const Cplx<T>*, const Cplx<T>*, const Cplx<T>*, \
                                                  const Cplx<T>*, int, int, int, int64_t, bool, int64_t,    \
                                                  T*, cudaStream_t);
DGFS_SHIFT_INST(float)
DGFS_SHIFT_INST(double)
#undef DGFS_SHIFT_INST

}  // namespace dgfs
