// The calls that transform every product forward again, on the shared translates of k_shift.cu:
//
//   VSS kernel (alpha != 1): gain^ = sum_r sum_p A_rp(k) DFT[(T_s f)(T_-s g) + (T_-s f)(T_s g)]_k
//   adjoint (VJP):  gain = sum_r sum_p 2 w_p [T_-s(U_r T_-s f) + T_s(U_r T_s f)],  U_r = K_r u
//   VHS gain of the Fourier stage in spectra (capi.cu stage_in_spectra):  gain^ = sum_r K_r(k) DFT[P_r]_k
//
//   k_shift_vss     per (node, r, XC planes x): the product lines of two sphere points share one forward z
//                   transform (real and imaginary part, separated per line into half spectra), forward y  -> W
//   k_shift_adj     the same for U_r T_-s f and U_r T_s f; the back-translates are phases, so what shares
//                   (s_x, s_y) is summed after the z phases, what shares s_x after the y phases         -> V
//   k_shift_sum     per (ky, kz) column: forward x of every field of W (V), times A_rp (the x phase, K_r), summed
//                   over a part of the fields (VHS: of the radial points) in registers      -> partial spectra
//   k_shift_filter  K_r u: forward x, multiplier, inverse x
//   k_shift_finish  sum of the parts, inverse x; K_L f as k_shift_filter, in blocks of the same launch
//   k_shift_out     inverse y and z of the gain and the loss fields, the result
//
// Measured (GB300, FP32, N = 32, M = 38): VSS Q of 40 nodes 3.1 ms (6.5 ms with a three-axis transform of its own for
// every translate and product), VJP of 48 nodes 3.9 ms (11 ms). k_shift_vss is 65 % of the first (1.75 instructions a cycle
// at 11 warps per SM, waiting on its loads), k_shift_sum 27 % (its products from DRAM); k_shift_adj 79 % of the second (2.1
// instructions a cycle at 8 warps per SM: a line and its sums fill the registers). VHS, N = 24, 144 nodes: k_shift_sum 41 us
// (192 MB: 4.7 TB/s), k_shift_finish about 20 us, in the 655 us of the call; at a few nodes the launches
// bound it, which is why gain and loss share k_shift_finish (five nodes, F16S, N = 32, M = 12: 169 -> 144 us with it and P_r
// and f in one forward launch).
//
// Everything stays in half spectra (kz >= 0): A_rp and the loss weight act on real fields, so only their part
// even in k counts. A multiplier on the packed slot kz = 0 needs the spectra of kz = 0 and kz = N/2 apart.
// k_shift_vss separates them along y, where its threads hold whole lines: their plane kz = 0 of W carries
// ky = 0 .. N/2 - 1 of the first, then of the second, with the real ky = 0 and N/2 packed in the two slots
// ky = 0 (a "folded" plane); only those two columns are separated along x, in registers. k_shift_filter takes the
// plane as it is: one warp holds it, kx in registers and ky along the lanes.
#include <algorithm>
#include <cmath>

#include "shift.h"
#include "shift_dev.cuh"

namespace dgfs {

namespace {

using namespace shdev;

template <typename T, int N, int XC>
struct SumGeo {
    static constexpr int NT = XC * N;
    static constexpr int PITCH = row_pitch<T, N>();
    static constexpr int BUF = 2 * XC * N * PITCH;           // complex elements of one buffer
    static constexpr size_t smem = (size_t)2 * BUF * sizeof(Cplx<T>);
    // k_shift_vss keeps a line and one product line, k_shift_adj a line, its sum and U's line
    static constexpr int MINV = sizeof(T) == 8 ? 1 : N == 32 ? 384 / NT : N == 24 ? 480 / NT : 768 / NT;
    static constexpr int MINA = sizeof(T) == 8 ? 1 : N == 32 ? 256 / NT : N == 24 ? 384 / NT : 512 / NT;
};

// grid (N / XC, nr parts, nodes): part q of a radial point takes its share of the program, whole pairs of entries, so that
// the bits do not depend on it. W [node][r][entry][x][ky][kz].
template <typename T, int N, int XC>
__global__ void __launch_bounds__(SumGeo<T, N, XC>::NT, SumGeo<T, N, XC>::MINV)
k_shift_vss(const Cplx<T>* __restrict__ Gf, const Cplx<T>* __restrict__ Hf, const Cplx<T>* __restrict__ Gg,
            const Cplx<T>* __restrict__ Hg, const Cplx<T>* __restrict__ mu, const ShiftEntry* __restrict__ prog, int nprog,
            int nrows, int nx, int r0, int parts, Cplx<T>* __restrict__ W) {
    using Geo = SumGeo<T, N, XC>;
    const int shares = XC == 2 ? parts : 1;   // the wide blocks take it all (and spare the registers of a share)
    constexpr int NH = N / 2, PITCH = Geo::PITCH, NT = Geo::NT, MP = shift_mu_pitch(N);
    constexpr int64_t FS = (int64_t)N * N * NH;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    Cplx<T>* Y = reinterpret_cast<Cplx<T>*>(sm_raw);         // [sign][XC][y][PITCH] inverse y lines
    Cplx<T>* S = Y + Geo::BUF;                               // [field][XC][y][PITCH] forward z lines
    const int tid = threadIdx.x, x0 = blockIdx.x * XC, rl = blockIdx.y / shares, nr = gridDim.y / shares;
    const int64_t node = blockIdx.z;
    const int op = tid / (XC * NH), ypl = (tid / NH) % XC, ykz = tid % NH;
    const int64_t ybase = (int64_t)(x0 + ypl) * N * NH + ykz;
    const Cplx<T>* Gy = (op ? Gg : Gf) + node * FS + ybase;
    const Cplx<T>* Hy = (op ? Hg : Hf) + (node * nr + rl) * (2 * nx) * FS + ybase;
    const int yrow = ((op * XC + ypl) * N) * PITCH + ykz;     // this thread's y line in a buffer
    const Cplx<T>* mu_r = mu + (int64_t)(r0 + rl) * nrows * MP;
    Cplx<T>* Wn = W + (node * nr + rl) * nprog * FS + ybase;
    if constexpr (XC == 2) {   // this block's share
        const int pq = blockIdx.y % parts, pairs = (nprog + 1) / 2, i0 = 2 * (pairs * pq / parts);
        nprog = min(nprog, 2 * (pairs * (pq + 1) / parts)) - i0;
        prog += i0;
        Wn += i0 * FS;
    }
    T first[N];                                              // products of the even entry
    Cplx<T> v[N];
    for (int i = 0; i < nprog; ++i) {
        const ShiftEntry e = prog[i];
        if (e.newy || i == 0) {
            const int fi = op ? e.fm : e.fp;
            load_y_line<T, N>(fi < 0 ? Gy : Hy + fi * FS, mu_r, e.yrow, e.yneg ^ op, v);
            cfft::line<T, N, false>(v);
            __syncthreads();   // the previous (s_x, s_y) has been read
#pragma unroll
            for (int y = 0; y < N; ++y) st(Y + yrow + y * PITCH, v[y]);
            __syncthreads();
        }
        load_z_line<T, N>(Y + tid * PITCH, Y + (NT + tid) * PITCH, mu_r, e.zrow, e.zneg, v);
        cfft::line<T, N, false>(v);
        if ((i & 1) == 0) {
#pragma unroll
            for (int z = 0; z < N; ++z) first[z] = v[z].x * v[z].y;
            if (i + 1 < nprog) continue;
#pragma unroll
            for (int z = 0; z < N; ++z) v[z] = Cplx<T>{T(0), T(0)};
        }
        Cplx<T> w[N];
#pragma unroll
        for (int z = 0; z < N; ++z) w[line_slot<N>(z)] = Cplx<T>{first[z], v[z].x * v[z].y};
        cfft::line<T, N, true>(w);
        __syncthreads();       // the previous pair's half spectra have been read
        split_line<T, N>(w, [&](int k, Cplx<T> a, Cplx<T> b) {
            st(S + tid * PITCH + k, a);
            st(S + (NT + tid) * PITCH + k, b);
        });
        __syncthreads();
        const int j = (i & ~1) + op;
        if (j < nprog) {
#pragma unroll
            for (int y = 0; y < N; ++y) w[line_slot<N>(y)] = ld(S + yrow + y * PITCH);
            cfft::line<T, N, true>(w);
            store_folded<T, N>(w, ykz, Wn + j * FS);
        }
    }
}

// grid (N / XC, nr, nodes). Ur [node][r][x][ky][kz]: x-space half spectra of K_r u. V [node][r][2 nx + 2][x][ky][kz]:
// field fi collects what takes the x phase of x field fi, the last two what takes none.
template <typename T, int N, int XC>
__global__ void __launch_bounds__(SumGeo<T, N, XC>::NT, SumGeo<T, N, XC>::MINA)
k_shift_adj(const Cplx<T>* __restrict__ G, const Cplx<T>* __restrict__ H, const Cplx<T>* __restrict__ Ur,
            const Cplx<T>* __restrict__ mu, const ShiftEntry* __restrict__ prog, int nprog, const T* __restrict__ wsig,
            int nrows, int nx, int r0, Cplx<T>* __restrict__ V) {
    using Geo = SumGeo<T, N, XC>;
    constexpr int NH = N / 2, PITCH = Geo::PITCH, NT = Geo::NT, MP = shift_mu_pitch(N);
    constexpr int64_t FS = (int64_t)N * N * NH;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    Cplx<T>* Y = reinterpret_cast<Cplx<T>*>(sm_raw);         // [sign][XC][y][PITCH] inverse y lines
    Cplx<T>* S = Y + Geo::BUF;                               // [sign][XC][y][PITCH] sums over s_z
    const int tid = threadIdx.x, x0 = blockIdx.x * XC, rl = blockIdx.y, nr = gridDim.y;
    const int64_t node = blockIdx.z, item = node * nr + rl;
    const int op = tid / (XC * NH), ypl = (tid / NH) % XC, ykz = tid % NH;
    const int64_t ybase = (int64_t)(x0 + ypl) * N * NH + ykz;
    const Cplx<T>* Gy = G + node * FS + ybase;
    const Cplx<T>* Hy = H + item * (2 * nx) * FS + ybase;
    const int yrow = ((op * XC + ypl) * N) * PITCH + ykz;
    const Cplx<T>* mu_r = mu + (int64_t)(r0 + rl) * nrows * MP;
    Cplx<T>* Vn = V + item * (2 * nx + 2) * FS + ybase;
    Cplx<T> v[N];
    T u[N];   // U_r on this thread's z line
    if (op == 0) {
        load_y_line<T, N>(Ur + item * FS + ybase, mu_r, -1, 0, v);
        cfft::line<T, N, false>(v);
#pragma unroll
        for (int y = 0; y < N; ++y) st(Y + yrow + y * PITCH, v[y]);
    }
    __syncthreads();
    {
        const Cplx<T>* zr = Y + tid * PITCH;
        const Cplx<T> a0 = ld(zr);
        v[0] = Cplx<T>{a0.x, T(0)};
        v[line_slot<N>(NH)] = Cplx<T>{a0.y, T(0)};
#pragma unroll
        for (int k = 1; k < NH; ++k) {
            const Cplx<T> a = ld(zr + k);
            v[line_slot<N>(k)] = a;
            v[line_slot<N>(N - k)] = Cplx<T>{a.x, -a.y};
        }
        cfft::line<T, N, false>(v);
#pragma unroll
        for (int z = 0; z < N; ++z) u[z] = v[z].x;
    }
    Cplx<T> acc[N];   // this thread's (sign, plane, kz) line over ky: sum over the s_y of one s_x
#pragma unroll
    for (int k = 0; k < N; ++k) acc[k] = Cplx<T>{T(0), T(0)};
    ShiftEntry g{};   // first entry of the group in hand
    bool zero_seen = false; // a group without x shift
    uint64_t written = 0;   // x fields (the first 64) that hold a sum already: rules with points on both sides of x = 0
    for (int i = 0; i <= nprog; ++i) {
        const ShiftEntry e = prog[i < nprog ? i : 0];
        const bool next = i == nprog || e.newy;
        if (next && i > 0) {
            __syncthreads();   // the group's sums over s_z are complete
#pragma unroll
            for (int y = 0; y < N; ++y) v[line_slot<N>(y)] = ld(S + yrow + y * PITCH);
            cfft::line<T, N, true>(v);
            const Cplx<T>* m = mu_r + (int64_t)(g.yrow >= 0 ? g.yrow : 0) * MP;
            const T sg = (g.yneg ^ op) ? T(-1) : T(1);
#pragma unroll
            for (int k = 0; k <= NH; ++k) {
                Cplx<T> w{T(1), T(0)};
                if (g.yrow >= 0) w = ldg(m + k);
                const T wi = k == 0 || k == NH ? T(0) : sg * w.y;
                acc[k] = Cplx<T>{fma(v[k].x, w.x, fma(-v[k].y, wi, acc[k].x)), fma(v[k].y, w.x, fma(v[k].x, wi, acc[k].y))};
                if (k > 0 && k < NH) {
                    Cplx<T>& a = acc[N - k];
                    const Cplx<T> q = v[N - k];
                    a = Cplx<T>{fma(q.x, w.x, fma(q.y, wi, a.x)), fma(q.y, w.x, fma(-q.x, wi, a.y))};
                }
            }
            if (i == nprog || e.fp != g.fp) {   // the next s_x
                const int fi = g.fp < 0 ? 2 * nx + op : op ? g.fm : g.fp, xi = g.fp < 0 ? -1 : g.fp >> 1;
                Cplx<T>* o = Vn + fi * FS;
                // both fields of an |s_x| are written together; a second visit (the opposite s_x) adds
                bool add = false;
                zero_seen |= xi < 0;
                if (xi >= 0) {
                    if (xi < 64) {
                        add = (written >> xi) & 1;
                        written |= uint64_t(1) << xi;
                    } else {
                        for (int q = 0; q < i && !add; ++q) add = prog[q].fp >= 0 && (prog[q].fp >> 1) == xi && prog[q].fp != g.fp;
                    }
                }
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    Cplx<T> s = acc[k];
                    if (add) {
                        const Cplx<T> b = ld(o + k * NH);
                        s.x += b.x;
                        s.y += b.y;
                    }
                    st(o + k * NH, s);
                    acc[k] = Cplx<T>{T(0), T(0)};
                }
            }
        }
        if (i == nprog) {
            if (!zero_seen)
                for (int k = 0; k < N; ++k) st(Vn + (2 * nx + op) * FS + k * NH, Cplx<T>{T(0), T(0)});
            break;
        }
        if (e.newy) {
            const int fi = op ? e.fm : e.fp;
            load_y_line<T, N>(fi < 0 ? Gy : Hy + fi * FS, mu_r, e.yrow, e.yneg ^ op, v);
            cfft::line<T, N, false>(v);
            if (i == 0) __syncthreads();   // U's lines have been read (later groups: the barrier above)
#pragma unroll
            for (int y = 0; y < N; ++y) st(Y + yrow + y * PITCH, v[y]);
            __syncthreads();
            g = e;
        }
        load_z_line<T, N>(Y + tid * PITCH, Y + (NT + tid) * PITCH, mu_r, e.zrow, e.zneg, v);
        cfft::line<T, N, false>(v);
        Cplx<T> w[N];   // U T_-s f + i U T_s f
#pragma unroll
        for (int z = 0; z < N; ++z) w[line_slot<N>(z)] = Cplx<T>{u[z] * v[z].y, u[z] * v[z].x};
        cfft::line<T, N, true>(w);
        const T wgt = T(2) * __ldg(wsig + e.pair), sg = e.zneg ? T(-1) : T(1);
        const bool zs = e.zrow >= 0, set = e.newy;
        const Cplx<T>* m = mu_r + (int64_t)(zs ? e.zrow : 0) * MP;
        Cplx<T>* sp = S + tid * PITCH;          // T_s(U T_s f)
        Cplx<T>* sm = S + (NT + tid) * PITCH;   // T_-s(U T_-s f)
        split_line<T, N>(w, [&](int k, Cplx<T> b, Cplx<T> a) {
            if (k == 0) {
                const T wn = zs ? wgt * ldg(m + NH).x : wgt;
                a = Cplx<T>{wgt * a.x, wn * a.y};
                b = Cplx<T>{wgt * b.x, wn * b.y};
            } else {
                Cplx<T> p{wgt, T(0)};
                if (zs) {
                    const Cplx<T> q = ldg(m + k);
                    p = Cplx<T>{wgt * q.x, wgt * sg * q.y};
                }
                a = cmul(a, p.x, p.y);
                b = cmul(b, p.x, -p.y);
            }
            if (!set) {
                const Cplx<T> ao = ld(sp + k), bo = ld(sm + k);
                a = Cplx<T>{a.x + ao.x, a.y + ao.y};
                b = Cplx<T>{b.x + bo.x, b.y + bo.y};
            }
            st(sp + k, a);
            st(sm + k, b);
        });
    }
}

// ---- columns (ky, kz): x lines ----------------------------------------------------------------

// The packed plane kz = 0 (kx in registers, ky = lane < N): real multipliers m0 on the spectrum of kz = 0 and mn on
// that of kz = N/2. Every lane of the warp takes part.
template <typename T, int N, typename M>
__device__ __forceinline__ void packed_plane(const Cplx<T> (&v)[N], int ky, M mult, Cplx<T> (&out)[N]) {
    const int src = ky == 0 ? 0 : N - ky;
#pragma unroll
    for (int kx = 0; kx < N; ++kx) {
        const Cplx<T> a = v[kx], q = v[(N - kx) % N];
        const Cplx<T> b{__shfl_sync(0xffffffffu, q.x, src), __shfl_sync(0xffffffffu, q.y, src)};   // the mirror
        T m0, mn;
        mult(kx, m0, mn);
        const T h0 = T(0.5) * m0, hn = T(0.5) * mn;
        // m0 (a + conj b) / 2 + i mn (a - conj b) / 2i
        out[kx] = Cplx<T>{h0 * (a.x + b.x) + hn * (a.x - b.x), h0 * (a.y - b.y) + hn * (a.y + b.y)};
    }
}

constexpr int kColThreads = 128;

// blocks of all columns, or of the ones with kz > 0
template <int N, bool NONZERO>
constexpr int col_blocks() { return (N * (N / 2 - (NONZERO ? 1 : 0)) + kColThreads - 1) / kColThreads; }

// F [node][r][nf fields][x][ky][kz]; part [node][parts][kx][ky][kz]. VSS: the plane kz = 0 folded, times A[(r0 + r)
// npairs + pair of the field] in the same order, [kx][ky][kz] and the second multipliers of the two packed columns
// [2][kx]; else the x phase of field fi (fields 2 nx, 2 nx + 1: none). VSS reads 2.5 MB of products per radial point
// and node at N = 32, M = 38 and is bound by that.
// Its rounding depends neither on the batch of nodes nor on the batch of radial points of a launch:
// Adjoint, Vss: block z of kSumParts takes its share of the fields, their sum at a radial point added to the total in
// order, on top of part [node][kSumParts] of the batch before; k_shift_finish adds the parts in order. (One running sum
// over radial points and fields, up to 300 FP32 additions at M = 38, lost accuracy: the VSS JVP of 32 nodes at N = 24 was
// 2.6e-6 of its norm off, 1.9e-6 with the sums taken apart.)
// Radial: groups of RP = ceil(Nrho / kSumGroups) radial points, each group's sum added to the total in order: grid
// (col_blocks, nodes, 1) keeps the totals in shared memory (part [node]); grid (col_blocks, nodes, sum_groups) takes a
// group each (part [node][group]) where one block per column leaves SMs idle.
// Radial (VHS gain, nf = 1): times tab[r0 + r][|k|^2], and coef[node][r0 + r] when the kernel varies by node.
enum class Sum { Adjoint, Vss, Radial };
// REGS: the totals of Adjoint and Vss in registers (sum_launch).
template <typename T, int N, Sum MODE, bool REGS>
__global__ void __launch_bounds__(kColThreads, REGS ? 1 : 0)
k_shift_sum(const Cplx<T>* __restrict__ F, int nf, const T* __restrict__ A, const T* __restrict__ coef, int Nrho,
            const ShiftEntry* __restrict__ prog, int npairs,
            const Cplx<T>* __restrict__ mu, const int* __restrict__ xrows, int nrows, int nx, int r0, int nr, int RP,
            Cplx<T>* __restrict__ part) {
    constexpr int NH = N / 2, COLS = N * NH, MP = shift_mu_pitch(N), NQ = 3 * NH * NH + 1;
    constexpr int64_t FS = (int64_t)N * COLS, AS = FS + 2 * N;
    const int64_t node = blockIdx.y;
    const int col = blockIdx.x * kColThreads + threadIdx.x;
    if (col >= COLS) return;
    const bool pair = MODE != Sum::Adjoint && (col == 0 || col == NH * NH);   // ky = 0 and N/2 of one plane in a column
    // |ky|^2 + |kz|^2 of the column (folded plane kz = 0)
    const int cky = col / NH, ckz = col % NH;
    const int fy = ckz ? (cky < NH ? cky : N - cky) : cky % NH, fz = ckz ? ckz : cky < NH ? 0 : NH, q0 = fy * fy + fz * fz;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    Cplx<T>* total = reinterpret_cast<Cplx<T>*>(sm_raw) + threadIdx.x;   // [kx][thread] (one block per column)
    const bool whole = MODE == Sum::Radial && gridDim.z == 1, by_r = MODE != Sum::Radial && sizeof(T) == 4, totals = by_r || whole;
    Cplx<T>* pc = part + (node * gridDim.z + blockIdx.z) * FS + col;
    // the batch's radial points of this block: all, or the ones of its group
    const int lo = MODE != Sum::Radial || whole ? 0 : max(0, (int)blockIdx.z * RP - r0);
    const int hi = MODE != Sum::Radial || whole ? nr : min(nr, (int)(blockIdx.z + 1) * RP - r0);
    if (lo >= hi) return;
    const int f0 = MODE == Sum::Radial ? 0 : nf * (int)blockIdx.z / (int)gridDim.z;   // its fields
    const int f1 = MODE == Sum::Radial ? 1 : nf * (int)(blockIdx.z + 1) / (int)gridDim.z;
    Cplx<T> acc[N];
    // a group under way from the batch before: its sum (whole: kept behind the totals)
    const bool started = MODE == Sum::Radial ? (r0 + lo) % RP != 0 : !by_r && r0 > 0;
    Cplx<T> reg[REGS ? N : 1];
    if (totals) {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const Cplx<T> t = r0 >= RP ? ld(pc + (int64_t)k * COLS) : Cplx<T>{T(0), T(0)};
            if constexpr (REGS) reg[k] = t;
            else total[k * kColThreads] = t;
        }
    }
    const Cplx<T>* open = whole ? part + (gridDim.y + node) * FS + col : pc;
#pragma unroll
    for (int k = 0; k < N; ++k) acc[k] = started ? ld(open + (int64_t)k * COLS) : Cplx<T>{T(0), T(0)};
    for (int rl = lo; rl < hi; ++rl) {
        if (totals && rl > lo && (r0 + rl) % RP == 0) {   // the group is complete
#pragma unroll
            for (int k = 0; k < N; ++k) {
                Cplx<T>& t = REGS ? reg[REGS ? k : 0] : total[k * kColThreads];
                t = fdev::add(t, acc[k]);
                acc[k] = Cplx<T>{T(0), T(0)};
            }
        }
        const Cplx<T>* f = F + ((node * nr + rl) * nf + f0) * FS + col;
        for (int j = f0; j < f1; ++j, f += FS) {
            Cplx<T> v[N];
#pragma unroll
            for (int x = 0; x < N; ++x) v[line_slot<N>(x)] = ldg(f + (int64_t)x * COLS);
            cfft::line<T, N, true>(v);
            if constexpr (MODE == Sum::Radial) {
                const T* t = A + (r0 + rl) * NQ + q0;
                const T c = coef ? __ldg(coef + node * Nrho + r0 + rl) : T(1);
#pragma unroll
                for (int k = 0; k <= NH; ++k) {
                    const T m = c * __ldg(t + k * k);
                    acc[k] = Cplx<T>{fma(m, v[k].x, acc[k].x), fma(m, v[k].y, acc[k].y)};
                    if (k > 0 && k < NH) acc[N - k] = Cplx<T>{fma(m, v[N - k].x, acc[N - k].x), fma(m, v[N - k].y, acc[N - k].y)};
                }
                if (pair) {   // m a so far; m (a + conj b) / 2 + m' (a - conj b) / 2, b the mirror along x
#pragma unroll
                    for (int k = 0; k < N; ++k) {
                        const int k2 = k <= NH ? k * k : (N - k) * (N - k);
                        const T h = T(0.5) * c * (__ldg(t + k2 + NH * NH) - __ldg(t + k2));
                        const Cplx<T> b = v[(N - k) % N];
                        acc[k] = Cplx<T>{fma(h, v[k].x - b.x, acc[k].x), fma(h, v[k].y + b.y, acc[k].y)};
                    }
                }
            } else if constexpr (MODE == Sum::Vss) {
                const T* a = A + ((int64_t)(r0 + rl) * npairs + __ldg(&prog[j].pair)) * AS;
#pragma unroll
                for (int k = 0; k < N; ++k) {
                    const T m = __ldg(a + (int64_t)k * COLS + col);
                    acc[k] = Cplx<T>{fma(m, v[k].x, acc[k].x), fma(m, v[k].y, acc[k].y)};
                }
                if (pair) {   // m a so far; m (a + conj b) / 2 + m' (a - conj b) / 2, b the mirror along x
                    const T* a2 = a + FS + (col ? N : 0);
#pragma unroll
                    for (int k = 0; k < N; ++k) {
                        const T h = T(0.5) * (__ldg(a2 + k) - __ldg(a + (int64_t)k * COLS + col));
                        const Cplx<T> b = v[(N - k) % N];
                        acc[k] = Cplx<T>{fma(h, v[k].x - b.x, acc[k].x), fma(h, v[k].y + b.y, acc[k].y)};
                    }
                }
            } else {
                const bool shifted = j < 2 * nx;
                const Cplx<T>* m = mu + ((int64_t)(r0 + rl) * nrows + (shifted ? __ldg(xrows + (j >> 1)) : 0)) * MP;
                const T sg = j & 1 ? T(-1) : T(1);
#pragma unroll
                for (int k = 0; k <= NH; ++k) {
                    Cplx<T> w{T(1), T(0)};
                    if (shifted) w = ldg(m + k);
                    const T wi = k == 0 || k == NH ? T(0) : sg * w.y;
                    acc[k] = Cplx<T>{fma(v[k].x, w.x, fma(-v[k].y, wi, acc[k].x)), fma(v[k].y, w.x, fma(v[k].x, wi, acc[k].y))};
                    if (k > 0 && k < NH) {
                        Cplx<T>& b = acc[N - k];
                        const Cplx<T> q = v[N - k];
                        b = Cplx<T>{fma(q.x, w.x, fma(q.y, wi, b.x)), fma(q.y, w.x, fma(-q.x, wi, b.y))};
                    }
                }
            }
        }
    }
    if (totals) {
        const bool done = (r0 + nr) % RP == 0 || r0 + nr == Nrho;   // the last group is complete
        Cplx<T>* rest = part + (gridDim.y + node) * FS + col;       // (whole; the other sums have groups of one radial point)
#pragma unroll
        for (int k = 0; k < N; ++k) {
            Cplx<T> t = REGS ? reg[REGS ? k : 0] : total[k * kColThreads];
            if (done) t = Cplx<T>{t.x + acc[k].x, t.y + acc[k].y};
            else st(rest + (int64_t)k * COLS, acc[k]);
            st(pc + (int64_t)k * COLS, t);
        }
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) st(pc + (int64_t)k * COLS, acc[k]);
    }
}

// out[node][x][ky][kz] = scale * inverse x of the sum of the parts; blocks bx < col_blocks
template <typename T, int N>
__device__ __forceinline__ void reduce_columns(const Cplx<T>* __restrict__ part, int parts, T scale, int bx, int64_t node,
                                               Cplx<T>* __restrict__ out) {
    constexpr int COLS = N * N / 2;
    constexpr int64_t FS = (int64_t)N * COLS;
    const int c = bx * kColThreads + threadIdx.x;
    if (c >= COLS) return;
    Cplx<T> v[N];
#pragma unroll
    for (int k = 0; k < N; ++k) v[line_slot<N>(k)] = Cplx<T>{T(0), T(0)};
    for (int q = 0; q < parts; ++q) {
        const Cplx<T>* p = part + (node * parts + q) * FS + c;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const Cplx<T> a = ldg(p + (int64_t)k * COLS);
            Cplx<T>& b = v[line_slot<N>(k)];
            b = Cplx<T>{b.x + a.x, b.y + a.y};
        }
    }
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = Cplx<T>{scale * v[k].x, scale * v[k].y};
    cfft::line<T, N, false>(v);
#pragma unroll
    for (int x = 0; x < N; ++x) st(out + node * FS + (int64_t)x * COLS + c, v[x]);
}

// out = inverse x of M(k) times the x spectrum of G (fields of one node): M = t[k] (nq2 == 0, standard mode index),
// t[|k|^2], or (Lr) sum_r rho_r Lr[r][k], summed in FP64 (the loss weight of the sphere rule with a kernel that varies
// by node). Blocks bx < filter_blocks, the last one warp for the packed plane kz = 0
template <int N>
constexpr int filter_blocks() { return col_blocks<N, true>() + 1; }
template <typename T, int N>
__device__ __forceinline__ void filter_columns(const Cplx<T>* __restrict__ G, const T* __restrict__ t, int nq2,
                                               const T* __restrict__ Lr, const double* __restrict__ cr, const NodeParams& np,
                                               int Nrho, int bx, int64_t node, Cplx<T>* __restrict__ out) {
    constexpr int NH = N / 2, COLS = N * NH;
    constexpr int64_t FS = (int64_t)N * COLS;
    const bool packed = bx == filter_blocks<N>() - 1;
    __shared__ double rho[64];
    if (Lr) {
        const double gam = np.gamma ? np.gamma[node] : np.gamma0, bb = np.b ? np.b[node] : np.b0;
        for (int r = threadIdx.x; r < Nrho; r += kColThreads) rho[r] = fdev::radial_rho<double>(bb, gam, cr[r], np.dlog);
        __syncthreads();
    }
    int ky, kz;
    if (packed) {
        if (threadIdx.x >= 32) return;
        ky = threadIdx.x < N ? threadIdx.x : 0;
        kz = 0;
    } else {
        const int c = bx * kColThreads + threadIdx.x;
        if (c >= N * (NH - 1)) return;
        ky = c / (NH - 1);
        kz = c % (NH - 1) + 1;
    }
    const int col = ky * NH + kz;
    auto sq = [](int q) { const int k = q < NH ? q : q - N; return k * k; };
    auto mult = [&](int kx, int kzz) -> T {
        const int k = (kx * N + ky) * N + kzz;
        if (Lr) return fdev::loss_multiplier<T>(nullptr, nullptr, Lr, rho, true, 0, Nrho, 2 * FS, k);
        return __ldg(nq2 ? t + sq(kx) + sq(ky) + kzz * kzz : t + k);
    };
    Cplx<T> v[N], w[N];
#pragma unroll
    for (int x = 0; x < N; ++x) v[line_slot<N>(x)] = ldg(G + (int64_t)x * COLS + col);
    cfft::line<T, N, true>(v);
    const T sc = T(1) / T(N);
    if (packed) {
        Cplx<T> q[N];
        packed_plane<T, N>(v, ky, [&](int kx, T& m0, T& mn) {
            m0 = mult(kx, 0);
            mn = mult(kx, NH);
        }, q);
#pragma unroll
        for (int k = 0; k < N; ++k) w[line_slot<N>(k)] = Cplx<T>{sc * q[k].x, sc * q[k].y};
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const T m = sc * mult(k, kz);
            w[line_slot<N>(k)] = Cplx<T>{m * v[k].x, m * v[k].y};
        }
    }
    cfft::line<T, N, false>(w);
    if (packed && threadIdx.x >= N) return;
#pragma unroll
    for (int x = 0; x < N; ++x) st(out + (int64_t)x * COLS + col, w[x]);
}

// out[node][r]: K_r of every radial point. grid (filter_blocks, nodes, nr)
template <typename T, int N>
__global__ void __launch_bounds__(kColThreads)
k_shift_filter(const Cplx<T>* __restrict__ G, const T* __restrict__ tab, int r0, Cplx<T>* __restrict__ out) {
    constexpr int64_t FS = (int64_t)N * N * N / 2;
    constexpr int NQ = 3 * (N / 2) * (N / 2) + 1;
    const int64_t node = blockIdx.y;
    filter_columns<T, N>(G + node * FS, tab + (int64_t)(r0 + blockIdx.z) * NQ, NQ, nullptr, nullptr, NodeParams{}, 0, blockIdx.x, node,
                         out + (node * gridDim.z + blockIdx.z) * FS);
}

// The gain (F_0) and the loss fields (F_1 from G1, F_2 from G2, F [field][nodes]) in one launch.
// grid (col_blocks + filter_blocks (1 or 2), nodes)
template <typename T, int N>
__global__ void __launch_bounds__(kColThreads)
k_shift_finish(const Cplx<T>* __restrict__ part, int parts, T scale, const Cplx<T>* __restrict__ G1, const Cplx<T>* __restrict__ G2,
               FilterTable<T> m, Cplx<T>* __restrict__ F) {
    constexpr int64_t FS = (int64_t)N * N * N / 2;
    constexpr int NQ = 3 * (N / 2) * (N / 2) + 1, CB = col_blocks<N, false>(), FB = filter_blocks<N>();
    const int64_t node = blockIdx.y, nodes = gridDim.y;
    if (blockIdx.x < CB) {
        reduce_columns<T, N>(part, parts, scale, blockIdx.x, node, F);
        return;
    }
    const int k = (blockIdx.x - CB) / FB;
    filter_columns<T, N>((k ? G2 : G1) + node * FS, m.by_node ? m.tab + node * NQ : m.tab, m.by_node ? NQ : 0, m.Lr, m.cr, m.np, m.Nrho,
                         (blockIdx.x - CB) % FB, node, F + ((k + 1) * nodes + node) * FS);
}

// w_r rho_r(node), and (Lq) the loss multiplier by |k|^2 of each node, summed over r in FP64. One block per node.
template <typename T>
__global__ void k_shift_coef(const double* __restrict__ cr, const double* __restrict__ wr, NodeParams np, int Nrho,
                             const T* __restrict__ Lq, int nq2, T* __restrict__ coef, T* __restrict__ GLq) {
    __shared__ double rho[64];
    const int64_t node = blockIdx.x;
    const double gam = np.gamma ? np.gamma[node] : np.gamma0, bb = np.b ? np.b[node] : np.b0;
    for (int r = threadIdx.x; r < Nrho; r += blockDim.x) {
        rho[r] = fdev::radial_rho<double>(bb, gam, cr[r], np.dlog);
        coef[node * Nrho + r] = (T)(wr[r] * rho[r]);
    }
    __syncthreads();
    if (!Lq) return;
    for (int q = threadIdx.x; q < nq2; q += blockDim.x) {
        double g = 0.0;
        for (int r = 0; r < Nrho; ++r) g = fma(rho[r], (double)Lq[r * nq2 + q], g);
        GLq[node * nq2 + q] = (T)g;
    }
}

// ---- result ------------------------------------------------------------------------------------

template <int N>
struct OutGeo {
    static constexpr int PX = N == 32 ? 2 : N == 12 ? 6 : N == 8 ? 8 : 4;   // planes per CTA
    static constexpr int NT = PX * N / 2;
    static constexpr int PITCH = N / 2 + 1;
};

// out = F_0 - a F_1 - c F_2 (nf fields; a, c nullptr: 1), F [field][node][x][ky][kz]; folded: the plane kz = 0 of F_0
// is. grid (N / PX, nodes). A thread owns whole rows z, so its factors and results go by 16 bytes (fields are 16-byte
// aligned at every entry point): a value at a time cost 1.3 % of the DG term (667 -> 658 us) and 0.7 % of Q at N = 32.
template <typename T, int N>
__global__ void __launch_bounds__(OutGeo<N>::NT)
k_shift_out(const Cplx<T>* __restrict__ F, int nf, int64_t field_stride, int folded, const T* __restrict__ a,
            const T* __restrict__ c, const int64_t* __restrict__ offs, T* __restrict__ out, int* __restrict__ flags) {
    using Geo = OutGeo<N>;
    constexpr int NH = N / 2, PITCH = Geo::PITCH, V = 16 / (int)sizeof(T);   // values of one 16-byte access
    constexpr int64_t FS = (int64_t)N * N * NH, n3 = 2 * FS;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    Cplx<T>* S = reinterpret_cast<Cplx<T>*>(sm_raw);       // [PX][y][PITCH]
    const int tid = threadIdx.x, pl = tid / NH, j = tid % NH, x = blockIdx.x * Geo::PX + pl;
    const int64_t node = blockIdx.y;
    const int64_t row0 = (offs ? offs[node] : node * n3) + ((int64_t)x * N + j) * N, row1 = row0 + (int64_t)NH * N;   // rows y = j, j + N/2
    T q0[N], q1[N];
#pragma unroll
    for (int z = 0; z < N; ++z) q0[z] = q1[z] = T(0);
    for (int fo = 0; fo < nf; ++fo) {
        Cplx<T> v[N];
        const Cplx<T>* src = F + fo * field_stride + node * FS + (int64_t)x * N * NH + j;   // slot kz = j
        if (j > 0 || fo > 0 || !folded) {
#pragma unroll
            for (int k = 0; k < N; ++k) v[line_slot<N>(k)] = ldg(src + k * NH);
        } else {
            const Cplx<T> p = ldg(src), q = ldg(src + NH * NH);
            v[0] = Cplx<T>{p.x, q.x};
            v[line_slot<N>(NH)] = Cplx<T>{p.y, q.y};
#pragma unroll
            for (int k = 1; k < NH; ++k) {
                const Cplx<T> b = ldg(src + k * NH), h = ldg(src + (NH + k) * NH);
                v[line_slot<N>(k)] = Cplx<T>{b.x - h.y, b.y + h.x};
                v[line_slot<N>(N - k)] = Cplx<T>{b.x + h.y, h.x - b.y};
            }
        }
        cfft::line<T, N, false>(v);
        __syncthreads();
#pragma unroll
        for (int y = 0; y < N; ++y) st(S + (pl * N + y) * PITCH + j, v[y]);
        __syncthreads();
        const Cplx<T>* ra = S + (pl * N + j) * PITCH;
        const Cplx<T>* rb = ra + NH * PITCH;
        {
            const Cplx<T> p = ld(ra), q = ld(rb);
            v[0] = Cplx<T>{p.x, q.x};
            v[line_slot<N>(NH)] = Cplx<T>{p.y, q.y};
        }
#pragma unroll
        for (int k = 1; k < NH; ++k) {
            const Cplx<T> p = ld(ra + k), q = ld(rb + k);
            v[line_slot<N>(k)] = Cplx<T>{p.x - q.y, p.y + q.x};
            v[line_slot<N>(N - k)] = Cplx<T>{p.x + q.y, q.x - p.y};
        }
        cfft::line<T, N, false>(v);
        const T* mul = fo == 1 ? a : fo == 2 ? c : nullptr;
#pragma unroll
        for (int z = 0; z < N; z += V) {
            alignas(16) T m0[V], m1[V];
            if (mul) {
                *reinterpret_cast<uint4*>(m0) = *reinterpret_cast<const uint4*>(mul + row0 + z);
                *reinterpret_cast<uint4*>(m1) = *reinterpret_cast<const uint4*>(mul + row1 + z);
            }
#pragma unroll
            for (int k = 0; k < V; ++k) {
                q0[z + k] = fo ? q0[z + k] - (mul ? m0[k] : T(1)) * v[z + k].x : v[z + k].x;
                q1[z + k] = fo ? q1[z + k] - (mul ? m1[k] : T(1)) * v[z + k].y : v[z + k].y;
            }
        }
    }
    bool bad = false;
#pragma unroll
    for (int z = 0; z < N; z += V) {
        alignas(16) T r0[V], r1[V];
#pragma unroll
        for (int k = 0; k < V; ++k) {
            bad |= !isfinite(q0[z + k]) || !isfinite(q1[z + k]);
            r0[k] = q0[z + k];
            r1[k] = q1[z + k];
        }
        *reinterpret_cast<uint4*>(out + row0 + z) = *reinterpret_cast<const uint4*>(r0);
        *reinterpret_cast<uint4*>(out + row1 + z) = *reinterpret_cast<const uint4*>(r1);
    }
    if (bad) atomicOr(flags, 2);
}

// ---- launches ------------------------------------------------------------------------------------

template <typename K>
cudaError_t allow_smem(K kern, size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename T, int N, int XC>
cudaError_t vss_x(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg, const Cplx<T>* Hg, int r0,
                  int nr, int64_t nodes, Cplx<T>* W, cudaStream_t s) {
    using Geo = SumGeo<T, N, XC>;
    const cudaError_t e = allow_smem(k_shift_vss<T, N, XC>, Geo::smem);
    if (e != cudaSuccess) return e;
    const bool bil = Gg != nullptr;
    const int nprog = bil ? d.nbil : d.nquad;
    // shares of the program while the (x, r, node) blocks have fewer than eight warps for each of the 152 SMs (narrow blocks
    // only, see narrow()): the JVP of one node in FP64, N = 8, M = 26 took 514 us with one share, 336 with 13
    const int64_t threads = (int64_t)(N / XC) * nr * nodes * Geo::NT;
    const int parts = XC == 2 ? (int)std::max<int64_t>(1, std::min<int64_t>((nprog + 1) / 2, 152 * 256 / threads)) : 1;
    k_shift_vss<T, N, XC><<<dim3(N / XC, (unsigned)(nr * parts), (unsigned)nodes), Geo::NT, Geo::smem, s>>>(
        Gf, Hf, bil ? Gg : Gf, bil ? Hg : Hf, d.mu, bil ? d.bil : d.quad, nprog, d.nrows, d.nx, r0, parts, W);
    return cudaGetLastError();
}

template <typename T, int N, int XC>
cudaError_t adj_x(const ShiftDev<T>& d, const Cplx<T>* G, const Cplx<T>* H, const Cplx<T>* Ur, int r0, int nr,
                  int64_t nodes, Cplx<T>* V, cudaStream_t s) {
    using Geo = SumGeo<T, N, XC>;
    const cudaError_t e = allow_smem(k_shift_adj<T, N, XC>, Geo::smem);
    if (e != cudaSuccess) return e;
    k_shift_adj<T, N, XC><<<dim3(N / XC, (unsigned)nr, (unsigned)nodes), Geo::NT, Geo::smem, s>>>(
        G, H, Ur, d.mu, d.quad, d.nquad, d.wsig, d.nrows, d.nx, r0, V);
    return cudaGetLastError();
}

// planes per CTA: as in k_shift.cu (two while wide CTAs would not fill the SMs about four deep)
template <int N>
constexpr int wide() { return N == 32 || N == 24 ? 4 : N == 12 ? 12 : 8; }
template <int N>
bool narrow(int nr, int64_t nodes) { return (int64_t)(N / wide<N>()) * nr * nodes < 608; }

template <typename T, int N>
cudaError_t vss_n(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg, const Cplx<T>* Hg, int r0,
                  int nr, int64_t nodes, Cplx<T>* W, cudaStream_t s) {
    return narrow<N>(nr, nodes) ? vss_x<T, N, 2>(d, Gf, Hf, Gg, Hg, r0, nr, nodes, W, s)
                                : vss_x<T, N, wide<N>()>(d, Gf, Hf, Gg, Hg, r0, nr, nodes, W, s);
}

template <typename T, int N>
cudaError_t adj_n(const ShiftDev<T>& d, const Cplx<T>* G, const Cplx<T>* H, const Cplx<T>* Ur, int r0, int nr,
                  int64_t nodes, Cplx<T>* V, cudaStream_t s) {
    return narrow<N>(nr, nodes) ? adj_x<T, N, 2>(d, G, H, Ur, r0, nr, nodes, V, s)
                                : adj_x<T, N, wide<N>()>(d, G, H, Ur, r0, nr, nodes, V, s);
}

template <typename T, int N, Sum MODE>
cudaError_t sum_launch(const ShiftDev<T>& d, const Cplx<T>* F, int nf, const T* A, const T* coef, const ShiftEntry* prog, int npairs,
                       int Nrho, int r0, int nr, int parts, int64_t nodes, Cplx<T>* part, cudaStream_t s) {
    const bool by_r = MODE != Sum::Radial && sizeof(T) == 4;
    const dim3 grid(col_blocks<N, false>(), (unsigned)nodes, (unsigned)parts);
    auto go = [&](auto kern, bool regs) {
        const size_t sm = (by_r && !regs) || (MODE == Sum::Radial && parts == 1) ? sizeof(Cplx<T>) * N * kColThreads : 0;
        const cudaError_t e = allow_smem(kern, sm);
        if (e != cudaSuccess) return e;
        kern<<<grid, kColThreads, sm, s>>>(F, nf, A, coef, Nrho, prog, npairs, d.mu, d.xrows, d.nrows, d.nx, r0, nr,
                                           MODE == Sum::Radial ? sum_group(Nrho) : 1, part);
        return cudaGetLastError();
    };
    // Totals in registers (two thirds of the resident warps) or in shared memory (a read and a write of them per radial
    // point): registers for launches that leave SMs idle (VSS Q of one node, N = 32, M = 26: 358 us, 507 in shared memory)
    // and for VSS at N <= 12 and 32 (M = 26, 500 nodes at N = 12: 526 / 594 us; 40 nodes at N = 32: 2223 / 2312 us); at
    // N = 16, 24 and for the adjoint shared memory is level or ahead (VJP of 300 nodes, N = 24: 5317 / 5515 us)
    if constexpr (MODE != Sum::Radial && sizeof(T) == 4)
        if ((MODE == Sum::Vss && N != 16 && N != 24) || (int64_t)grid.x * grid.y * grid.z < 304)
            return go(k_shift_sum<T, N, MODE, true>, true);
    return go(k_shift_sum<T, N, MODE, false>, false);
}

template <typename T, int N>
cudaError_t sum_n(const ShiftDev<T>& d, const Cplx<T>* F, int nf, const T* A, bool bil, int npairs, int r0, int nr, int64_t nodes,
                  Cplx<T>* part, cudaStream_t s) {
    if (A) return sum_launch<T, N, Sum::Vss>(d, F, nf, A, nullptr, bil ? d.bil : d.quad, npairs, 0, r0, nr, kSumParts, nodes, part, s);
    return sum_launch<T, N, Sum::Adjoint>(d, F, nf, nullptr, nullptr, d.quad, npairs, 0, r0, nr, kSumParts, nodes, part, s);
}

template <typename T, int N>
cudaError_t gain_n(const ShiftDev<T>& d, const Cplx<T>* W, const T* tab, const T* coef, int Nrho, int r0, int nr, int parts,
                   int64_t nodes, Cplx<T>* part, cudaStream_t s) {
    return sum_launch<T, N, Sum::Radial>(d, W, 1, tab, coef, d.quad, 0, Nrho, r0, nr, parts, nodes, part, s);
}

template <typename T, int N>
cudaError_t filter_n(const ShiftDev<T>& d, const Cplx<T>* G, int r0, int nr, int64_t nodes, Cplx<T>* out, cudaStream_t s) {
    k_shift_filter<T, N><<<dim3(filter_blocks<N>(), (unsigned)nodes, (unsigned)nr), kColThreads, 0, s>>>(G, d.kq, r0, out);
    return cudaGetLastError();
}

template <typename T, int N>
cudaError_t finish_n(const Cplx<T>* part, int parts, T scale, const Cplx<T>* G1, const Cplx<T>* G2, const FilterTable<T>& m,
                     int64_t nodes, Cplx<T>* F, cudaStream_t s) {
    const int blocks = col_blocks<N, false>() + filter_blocks<N>() * (G2 ? 2 : 1);
    k_shift_finish<T, N><<<dim3((unsigned)blocks, (unsigned)nodes), kColThreads, 0, s>>>(part, parts, scale, G1, G2, m, F);
    return cudaGetLastError();
}

template <typename T, int N>
cudaError_t out_n(const Cplx<T>* F, int nf, int64_t field_stride, bool folded, const T* a, const T* c, const int64_t* offs, int64_t nodes,
                  T* out, int* flags, cudaStream_t s) {
    using Geo = OutGeo<N>;
    constexpr size_t sm = (size_t)Geo::PX * N * Geo::PITCH * sizeof(Cplx<T>);
    k_shift_out<T, N><<<dim3(N / Geo::PX, (unsigned)nodes), Geo::NT, sm, s>>>(F, nf, field_stride, folded, a, c, offs, out, flags);
    return cudaGetLastError();
}

}  // namespace

double shift_result_scale(int N, bool fp64) {
    const double n3 = (double)N * N * N;
    return fp64 ? 1.0 / n3 : std::exp2(-std::round(std::log2(n3)));
}

#define DGFS_BY_N(CALL)                              \
    if (nodes <= 0) return cudaSuccess;              \
    if (nodes > 65535) return cudaErrorInvalidValue; \
    if (N == 8) return CALL(8);                      \
    if (N == 12) return CALL(12);                    \
    if (N == 16) return CALL(16);                    \
    if (N == 24) return CALL(24);                    \
    if (N == 32) return CALL(32);                    \
    return cudaErrorInvalidValue

template <typename T>
cudaError_t launch_shift_vss(const ShiftDev<T>& d, const Cplx<T>* Gf, const Cplx<T>* Hf, const Cplx<T>* Gg, const Cplx<T>* Hg,
                             int N, int r0, int nr, int64_t nodes, Cplx<T>* W, cudaStream_t s) {
#define CALL(n) vss_n<T, n>(d, Gf, Hf, Gg, Hg, r0, nr, nodes, W, s)
    DGFS_BY_N(CALL);
#undef CALL
}
template <typename T>
cudaError_t launch_shift_adj(const ShiftDev<T>& d, const Cplx<T>* G, const Cplx<T>* H, const Cplx<T>* Ur, int N,
                             int r0, int nr, int64_t nodes, Cplx<T>* V, cudaStream_t s) {
#define CALL(n) adj_n<T, n>(d, G, H, Ur, r0, nr, nodes, V, s)
    DGFS_BY_N(CALL);
#undef CALL
}
template <typename T>
cudaError_t launch_shift_sum(const ShiftDev<T>& d, const Cplx<T>* F, int nf, const T* A, bool bil, int npairs, int N, int r0,
                             int nr, int64_t nodes, Cplx<T>* part, cudaStream_t s) {
#define CALL(n) sum_n<T, n>(d, F, nf, A, bil, npairs, r0, nr, nodes, part, s)
    DGFS_BY_N(CALL);
#undef CALL
}
template <typename T>
cudaError_t launch_shift_filter(const ShiftDev<T>& d, const Cplx<T>* G, int N, int r0, int nr, int64_t nodes, Cplx<T>* out,
                                cudaStream_t s) {
#define CALL(n) filter_n<T, n>(d, G, r0, nr, nodes, out, s)
    DGFS_BY_N(CALL);
#undef CALL
}
template <typename T>
cudaError_t launch_shift_finish(const Cplx<T>* part, int parts, T scale, const Cplx<T>* G1, const Cplx<T>* G2,
                                const FilterTable<T>& m, int N, int64_t nodes, Cplx<T>* F, cudaStream_t s) {
#define CALL(n) finish_n<T, n>(part, parts, scale, G1, G2, m, nodes, F, s)
    DGFS_BY_N(CALL);
#undef CALL
}
template <typename T>
cudaError_t launch_shift_gain(const ShiftDev<T>& d, const Cplx<T>* W, const T* tab, const T* coef, int Nrho, int N, int r0,
                              int nr, int parts, int64_t nodes, Cplx<T>* part, cudaStream_t s) {
#define CALL(n) gain_n<T, n>(d, W, tab, coef, Nrho, r0, nr, parts, nodes, part, s)
    DGFS_BY_N(CALL);
#undef CALL
}
template <typename T>
cudaError_t launch_shift_coef(const DevTables<T>& t, NodeParams np, int64_t nodes, T* coef, T* GLq, cudaStream_t s) {
    if (nodes <= 0) return cudaSuccess;
    k_shift_coef<T><<<(unsigned)nodes, 128, 0, s>>>(t.cr, t.wr, np, t.Nrho, t.Lq, 3 * (t.N / 2) * (t.N / 2) + 1, coef, GLq);
    return cudaGetLastError();
}
template <typename T>
cudaError_t launch_shift_out(const Cplx<T>* F, int nf, int64_t field_stride, bool folded, const T* a, const T* c,
                             const int64_t* offs, int N, int64_t nodes, T* out, int* flags, cudaStream_t s) {
#define CALL(n) out_n<T, n>(F, nf, field_stride, folded, a, c, offs, nodes, out, flags, s)
    DGFS_BY_N(CALL);
#undef CALL
}

#define DGFS_SHIFT_INST(T)                                                                                              \
    template cudaError_t launch_shift_vss<T>(const ShiftDev<T>&, const Cplx<T>*, const Cplx<T>*, const Cplx<T>*,        \
                                             const Cplx<T>*, int, int, int, int64_t, Cplx<T>*, cudaStream_t);           \
    template cudaError_t launch_shift_adj<T>(const ShiftDev<T>&, const Cplx<T>*, const Cplx<T>*, const Cplx<T>*,        \
                                             int, int, int, int64_t, Cplx<T>*, cudaStream_t);                 \
    template cudaError_t launch_shift_sum<T>(const ShiftDev<T>&, const Cplx<T>*, int, const T*, bool, int, int, int,    \
                                             int, int64_t, Cplx<T>*, cudaStream_t);                                    \
    template cudaError_t launch_shift_filter<T>(const ShiftDev<T>&, const Cplx<T>*, int, int, int, int64_t, Cplx<T>*, \
                                                cudaStream_t);                                                        \
    template cudaError_t launch_shift_finish<T>(const Cplx<T>*, int, T, const Cplx<T>*, const Cplx<T>*,               \
                                                const FilterTable<T>&, int, int64_t, Cplx<T>*, cudaStream_t);         \
    template cudaError_t launch_shift_out<T>(const Cplx<T>*, int, int64_t, bool, const T*, const T*, const int64_t*,    \
                                             int, int64_t, T*, int*, cudaStream_t);                                     \
    template cudaError_t launch_shift_gain<T>(const ShiftDev<T>&, const Cplx<T>*, const T*, const T*, int, int, int,    \
                                              int, int, int64_t, Cplx<T>*, cudaStream_t);                                    \
    template cudaError_t launch_shift_coef<T>(const DevTables<T>&, NodeParams, int64_t, T*, T*, cudaStream_t);
DGFS_SHIFT_INST(float)
DGFS_SHIFT_INST(double)
#undef DGFS_SHIFT_INST

}  // namespace dgfs
