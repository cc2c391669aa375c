// Shared-shift translate products of the CUDA-core plans (k_shift.cu): the host side of the
// program that the product kernel walks, and the launchers.
#pragma once

#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "launchers.h"
#include "plan_host.h"

namespace dgfs {

// One product term w (T_s f)(T_-s g). Its x translates are two fields of the x pass (-1: shift 0), its
// y and z multipliers rows of the shift table (-1: shift 0) with a sign.
struct ShiftEntry {
    int fp, fm;      // x-pass fields of +s_x (of f) and -s_x (of g)
    int yrow, yneg;  // |s_y|, 1 when s_y < 0
    int zrow, zneg;  // |s_z|, 1 when s_z < 0
    int pair;        // sphere pair (weight)
    int newy;        // 1: another (s_x, s_y) than the entry before it
};

// Entries sorted by (s_x, s_y), so that equal x and (x, y) translates are neighbours: M = 38 has 19 pairs
// but 8 nonzero signed x shifts and 13 (x, y) shifts up to sign; a rule without coinciding components
// gets an entry of its own for each.
struct ShiftProgram {
    int nrows = 0;                       // distinct nonzero |component| over all pairs and axes
    int nx = 0;                          // distinct nonzero |s_x|; fields 2i (+) and 2i + 1 (-)
    std::vector<int> xrows;              // [nx] row of the shift table
    std::vector<ShiftEntry> quad, bil;   // g = f: one entry per pair (weight 2 w_p); f, g: both signs (w_p)
    std::vector<double> sq, kq, kqd, st, kt;   // [Nrho][3 (N/2)^2 + 1] (VHS, see ShiftDev)
    std::vector<double> wsig;            // [npairs] weights; FP32: times excess (balance_constants)
    std::vector<double> excess;          // [npairs] VSS: factor of the pair's kernel factors (fill_vss_tables)
    double balance = 1.0, project = 1.0; // FP32: factor of the gain's radial multipliers, of the projection's coefficients
    std::vector<double> mu;              // [Nrho][nrows][MP][2] e^{i pi k s / L}, k = 0 .. N/2 (Nyquist cos)
};

// Row pitch of the shift table: N/2 + 1 modes, padded to an even count (16-byte FP32 rows).
constexpr int shift_mu_pitch(int N) { return N / 2 + 2; }

// fp32: for FP32 arithmetic
void build_shift_program(const HostPlan& h, bool fp32, ShiftProgram& p);
// scale of a result after its inverse transforms: 1 / N^3, FP32: the nearest power of two
double shift_result_scale(int N, bool fp64);

// Device side of the program, in the compute type.
template <typename T>
struct ShiftDev {
    int nrows = 0, nx = 0, nquad = 0, nbil = 0;
    const int* xrows = nullptr;
    const ShiftEntry *quad = nullptr, *bil = nullptr;
    const Cplx<T>* mu = nullptr;
    const T* wsig = nullptr;
    // VHS, [Nrho][3 (N/2)^2 + 1] by |k|^2: S(|k|, r) of the compressed radial kernel, w_r rho_r S (the multiplier of
    // K_r) and its derivative by gamma; st, kt: S and w_r rho_r S for P_r of the tensor cores, which carry the sphere
    // rule's own weights
    const T *sq = nullptr, *kq = nullptr, *kqd = nullptr, *st = nullptr, *kt = nullptr;
};

// G[node][x][ky][kz], kz = 0 .. N/2 - 1: the (y, z) spectra (times 1/N^2) of every x plane of the real
// field f; the real spectra of kz = 0 and kz = N/2 share the complex slot kz = 0. offs: element offset of
// every node (nullptr: node N^3).
// b: the field f b instead (nullptr: f).
template <typename T>
cudaError_t launch_shift_forward(const T* f, const T* b, const int64_t* offs, int N, int64_t nodes, Cplx<T>* G,
                                 cudaStream_t s);
// H[node][r - r0][field][x][ky][kz] for r in [r0, r0 + nr): the x translates of G by every signed x shift
template <typename T>
cudaError_t launch_shift_x(const ShiftDev<T>& d, const Cplx<T>* G, int N, int r0, int nr, int64_t nodes, Cplx<T>* H,
                           cudaStream_t s);
// P_r = the sum of the program's terms over the fields Hf/Gf (operand f) and Hg/Gg (operand g; Gg == nullptr: g = f);
// P + node node_stride + (r - r0) N^3. folded: its (y, z) spectra [x][ky][kz] (plane kz = 0 folded, shift_dev.cuh), as
// large as P_r.
template <typename T>
cudaError_t launch_shift_products(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg,
                                  const Cplx<T>* Hg, int N, int r0, int nr, int64_t nodes, bool folded, int64_t node_stride,
                                  T* P, cudaStream_t s);
// W: the same (folded) spectra of real fields P[fields][N^3] (a tensor-core plan's P_r); G: launch_shift_forward of f
template <typename T>
cudaError_t launch_shift_folded(const T* P, int64_t fields, const T* f, const int64_t* offs, int N, int64_t nodes, Cplx<T>* W,
                                Cplx<T>* G, cudaStream_t s);
// The radial sums (k_shift_sum.cu). gain: parts = sum_groups(Nrho), part [nodes][parts], or 1, part [2][nodes] (totals,
// then a group that a batch left unfinished); sum: part [nodes][kSumParts].
constexpr int kSumParts = 4, kSumGroups = 8;
constexpr int sum_group(int Nrho) { return (Nrho + kSumGroups - 1) / kSumGroups; }   // radial points per group
constexpr int sum_groups(int Nrho) { return Nrho < 1 ? 1 : (Nrho + sum_group(Nrho) - 1) / sum_group(Nrho); }
// part (+)= sum over r of tab[r0 + r][|k|^2] (times coef[node][r0 + r]) times the x spectra of W[node][r]
template <typename T>
cudaError_t launch_shift_gain(const ShiftDev<T>& d, const Cplx<T>* W, const T* tab, const T* coef, int Nrho, int N, int r0,
                              int nr, int parts, int64_t nodes, Cplx<T>* part, cudaStream_t s);
// per node: coef[node][r] = w_r rho_r, and with t.Lq the loss multiplier GLq[node][|k|^2]
template <typename T>
cudaError_t launch_shift_coef(const DevTables<T>& t, NodeParams np, int64_t nodes, T* coef, T* GLq, cudaStream_t s);

// VSS kernel and adjoint (k_shift_sum.cu). W [node][r][entry][x][ky][kz]: (y, z) spectra of every product of the
// quad (Gg == nullptr) or bil program.
template <typename T>
cudaError_t launch_shift_vss(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg, const Cplx<T>* Hg,
                             int N, int r0, int nr, int64_t nodes, Cplx<T>* W, cudaStream_t s);
// V [node][r][2 nx + 2][x][ky][kz]: the back-translated adjoint products before their x phases; Ur [node][r]: K_r u
template <typename T>
cudaError_t launch_shift_adj(const ShiftDev<T>& d, const Cplx<T>* G, const Cplx<T>* H, const Cplx<T>* Ur, int N,
                             int r0, int nr, int64_t nodes, Cplx<T>* V, cudaStream_t s);
// part (+)= the x spectra of the nf fields F[node][r] times A (VSS: [Nrho][npairs] half tables of
// N^3/2 + 2 N values, fill_vss_tables) or, A == nullptr, times the x phases of the adjoint's fields; summed over fields and r
template <typename T>
cudaError_t launch_shift_sum(const ShiftDev<T>& d, const Cplx<T>* F, int nf, const T* A, bool bil, int npairs, int N, int r0,
                             int nr, int64_t nodes, Cplx<T>* part, cudaStream_t s);
// out[node][r - r0] = the field G under the multiplier of K_r (d.kq)
template <typename T>
cudaError_t launch_shift_filter(const ShiftDev<T>& d, const Cplx<T>* G, int N, int r0, int nr, int64_t nodes, Cplx<T>* out,
                                cudaStream_t s);
// A real even multiplier: tab[k] (full grid, DFT index order), tab[node][|k|^2] (by_node) or, with Lr,
// sum_r rho_r(node) Lr[r][k].
template <typename T>
struct FilterTable {
    const T* tab = nullptr;
    int by_node = 0;
    const T* Lr = nullptr;
    const double* cr = nullptr;
    NodeParams np{};
    int Nrho = 0;
};
// F[field][nodes]: F_0 = scale times the inverse x transform of the sum of the parts, F_1 (F_2) = the field G1 (G2, or
// nullptr) under the multiplier m
template <typename T>
cudaError_t launch_shift_finish(const Cplx<T>* part, int parts, T scale, const Cplx<T>* G1, const Cplx<T>* G2,
                                const FilterTable<T>& m, int N, int64_t nodes, Cplx<T>* F, cudaStream_t s);
// out = F_0 - a F_1 - c F_2 on the grid (nf fields, field_stride complex elements apart; nullptr factors: 1; folded:
// the plane kz = 0 of F_0 as the VSS sums leave it)
template <typename T>
cudaError_t launch_shift_out(const Cplx<T>* F, int nf, int64_t field_stride, bool folded, const T* a, const T* c,
                             const int64_t* offs, int N, int64_t nodes, T* out, int* flags, cudaStream_t s);

}  // namespace dgfs
