// K1 / K2: the space-time predictor of Biot's system, one element per CTA, by
// the degree-block back-substitution of the paper (Section "Block-wise
// back-substitution", Algorithm 3), in binary64 (FP64 contexts, and mixed
// contexts with two refinement sweeps) or in double-binary32 (mixed contexts
// with one).
//
// GB300's binary64 pipe issues 2 lanes a clock and SM, so what it costs is the
// number of binary64 operations.  Three things keep it small:
//
// 1. The Khat products are integer sums over fixed-point rows (fixed_device.cuh),
//    each row (k, u) of X with one power-of-two scale per degree block.
// 2. The star products use the structure of the isotropic Jacobians instead of
//    their 162 entries per mode.  With n^j = -mu dt grad xi_j, the products
//    are formed with these 13 "primitive" rows, 25 operations a direction:
//      0 D = n.v   1 Df = n.vf   2 n_x u   9 n_y v   3..5 shear
//      6..8 S = sigma n          10..12 n p
//    Khat acts on the primitives, and the material constants combine the 13
//    sums to the 13 quantities once per mode, when its block is solved.
// 3. Z^{-1} is tridiagonal: time integration maps P_s to P_{s+-1}.  Two
//    products a row instead of N + 1 (only the fluid velocities, with
//    (Z - e I)^{-1}, are dense).
//
// The CTA keeps C[mode][13][T] in shared memory: the primitive sums of a mode
// until its block is solved, its predictor Q afterwards.  For g = N .. 0:
//   solve   a warp takes T lanes (u) of 32 / T modes and one of 4 groups of
//           quantities: b = S^{-1}w q0 - combinations of C, time solves with
//           the neighbours' u by warp shuffles; Q into C and to the outputs
//   scale   one power of two per (k, u) row of X from max |Q| over the block
//   star    lanes (j, mode, u): primitives, quantised into X
//   Khat    one warp per row l < o_g, lanes over (k, u): C[l] += Khat X
// (block 6 in two halves of its modes, so that two CTAs fit an SM).  The small
// blocks leave few independent operations, so what binds beside the binary64 pipe
// (72 % busy at N = 6) is latency: the work of each phase is cut fine and the CTA
// at N = 6 has 16 warps.  Against star products entry by entry, dense Z^{-1} and
// Khat in binary64, 20,000 elements at N = 6 take 5.73 instead of 22.45 ms; in
// double-binary32, against a binary32 tensor-core sweep, an exact residual and a
// correction sweep, 40,009 take 7.09 instead of 16.56 (N = 4, 20,011: 0.91 instead
// of 3.67).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <numeric>
#include <set>
#include <utility>

#include "chain.cuh"
#include "fixed_device.cuh"
#include "pair_device.cuh"
#include "poro_internal.h"
#include "tc_device.cuh"

namespace poro {
namespace {

// ------------------------------------------------------------ tables
// Per degree N in constant memory (they depend only on N): the Khat entries
// (offset of the column of X, numerator) pass by pass, and for 2, 4, 8 and 16
// warps the rows of each pass dealt to them, [warps + 1] list starts, then words
// l << 21 | entries << 13 | first entry.
constexpr int X_COLUMNS = 63;  // columns (direction, mode) of X a pass can hold
constexpr int khat_entries(int N) {
    return N == 1 ? 4 : N == 2 ? 29 : N == 3 ? 119 : N == 4 ? 364 : N == 5 ? 924 : 2058;
}
constexpr int entry_base(int N) { return N <= 1 ? 0 : entry_base(N - 1) + khat_entries(N - 1); }
PORO_HD constexpr int n_passes(int N) { return N == 0 ? 0 : pass_count(N, X_COLUMNS) + n_passes(N - 1); }
constexpr int pass_rows(int N) { return N == 0 ? 0 : pass_count(N, X_COLUMNS) * block_offset(N) + pass_rows(N - 1); }
// the lists of one warp count, and where those of 2 << v warps start
PORO_HD constexpr int list_part(int N, int v) { return pass_rows(N) + n_passes(N) * ((2 << v) + 1); }
PORO_HD constexpr int list_start(int N, int v) { return v == 0 ? 0 : list_start(N, v - 1) + list_part(N, v - 1); }
constexpr int list_base(int N) { return N <= 1 ? 0 : list_base(N - 1) + list_start(N - 1, 4); }
__constant__ int2 c_ent[entry_base(MAX_N) + khat_entries(MAX_N)];
__constant__ int32_t c_list[list_base(MAX_N) + list_start(MAX_N, 4)];

// terms of the 13 primitives: |row k| <= sum_i max_j |n^j_d| max |Q_q|
__constant__ int8_t c_prim_q[NQ][3] = {{QU, QV, QW},    {QUF, QVF, QWF}, {QU, -1, -1},     {QV, QU, -1},     {QW, QV, -1},
                                       {QW, QU, -1},    {SXX, SXY, SXZ}, {SXY, SYY, SYZ}, {SXZ, SYZ, SZZ}, {QV, -1, -1},
                                       {QP, -1, -1},    {QP, -1, -1},    {QP, -1, -1}};
__constant__ int8_t c_prim_d[NQ][3] = {{0, 1, 2}, {0, 1, 2}, {0, 0, 0}, {0, 1, 0}, {1, 2, 0}, {0, 2, 0}, {0, 1, 2},
                                       {0, 1, 2}, {0, 1, 2}, {1, 0, 0}, {0, 0, 0}, {1, 0, 0}, {2, 0, 0}};

// Z^{-1}: row u is z_lo on u - 1 (u = 0: on u itself) and z_hi on u + 1 (the
// last row: z_end on itself)
__constant__ double c_z_lo[MAX_N + 1] = {0.5, 0.5 / 1, 0.5 / 3, 0.5 / 5, 0.5 / 7, 0.5 / 9, 0.5 / 11};
__constant__ double c_z_hi[MAX_N + 1] = {-0.5 / 3, -0.5 / 5, -0.5 / 7, -0.5 / 9, -0.5 / 11, -0.5 / 13, -0.5 / 15};
__constant__ double c_z_end[MAX_N + 1] = {0.5, 0.5 / 3, 0.5 / 5, 0.5 / 7, 0.5 / 9, 0.5 / 11, 0.5 / 13};

struct DirectParams {
    const int32_t* elems;  // optional element index list (LTS clusters)
    const double* q0;
    const double* econst;
    double* qt;
    double* iout;
    double* qend;           // Q~(1) [ne][13][B], may be q0 (in double-binary32: q0 and its change, added in binary64)
    int64_t count;
    int stride;
    const double* inv_d;    // [B] 1 / d_l
    const float2* inv_d2;   // the same as (hi, lo)
    int32_t* status;        // double-binary32: set to 1 if the bounded wait gave up
    long long wait_limit;
    int whole_nan;          // a non-finite value makes the element's whole result NaN
    const RunPtrs* runs;    // items of several runs (nullptr: the pointers above)
    const int32_t* item_run;
};

// ------------------------------------------------------------ arithmetic
struct Bin64 : Bin64Base {
    using Low = long long;
    __device__ static R add_fixed(R a, long long hi, Low lo, int sc, const DirectParams& A, int l) {
        return ::fma(fixed_sum(hi, lo, sc), __ldg(A.inv_d + l), a);
    }
};
struct Bin32x2 : Bin32x2Base {
    using Low = float;
    __device__ static R add_fixed(R a, long long hi, Low lo, int sc, const DirectParams& A, int l) {
        const float2 inv = __ldg(A.inv_d2 + l), v = fixed_to_pair(hi, lo);
        const float f = pow2f(-sc);
        dw_mac(a.x, a.y, inv.x, inv.y, __fmul_rn(v.x, f), __fmul_rn(v.y, f));
        return a;
    }
};

// ------------------------------------------------------------ shape
// CTA sizes the autotuner chooses from (index 0 is the default), and the
// largest one that a small launch gains from.  Default and alternative for 2,000
// elements, microseconds, binary64 (double-binary32): N = 3 103, 101 (55, 63),
// N = 4 182, 221 (107, 154), N = 5 339, 492 (207, 354), N = 6 654, 676 (394, 438).
template <int N>
struct DirectSizes {
    static constexpr int WIDEST = N <= 2 ? 128 : N == 3 ? 256 : 512;
    static constexpr int NT0 = N == 6 ? 512 : N == 5 ? 256 : N == 4 ? 128 : 64;
    static constexpr int NT1 = N == 6 ? 256 : N == 5 ? 512 : N == 4 ? 256 : 128;
    // CTAs an SM that the default size's registers leave room for: what shared memory
    // allows from N = 3 on.  Against 8 CTAs, 40,000 elements, microseconds, binary64
    // (double-binary32): N = 3 1,554 -> 1,555 (937 -> 897), N = 2 780 -> 758 (499 ->
    // 468), N = 1 455 -> 438 (305 -> 272).  Narrower passes over X for still more CTAs
    // cost more at their barriers (N = 4, 24 columns, 6 CTAs: 1,551 -> 1,603, 927 -> 968;
    // N = 5, 30 columns, 4 CTAs: 2,456 -> 2,593, 1,505 -> 1,567 for 16,384).
    static constexpr int MIN_BLOCKS = N == 6 ? 2 : N == 5 ? 3 : N == 4 ? 5 : N == 3 ? 10 : 14;
};

template <int N, int NT_>
struct DirectShape {
    static constexpr int NT = NT_, NW = NT_ / 32;
    static constexpr int B = n_modes(N), T = N + 1, PT = NQ * T, PUL = (PT + 31) / 32;
    static constexpr int G = 32 / T;               // modes a warp solves at a time, one lane per (mode, u)
    // columns of X held: the widest pass is block N's, or at N = 6 block 5's
    static constexpr int XC = N == 6 ? X_COLUMNS : 3 * block_size(N);
    // element constants from the time matrices on: zuf[T][T], (e, g, dt), iso[16]
    static constexpr int EC0 = ec_zinv(N), EC = elem_const_stride(N) - EC0;
    // shared layout in 8-byte words
    static constexpr int OFF_X = B * PT;
    static constexpr int OFF_K = (OFF_X + XC * PT + 32 + 1) & ~1;   // raw constants (16-byte aligned for the bulk copy)
    static constexpr int OFF_R = OFF_K + EC;                        // the same as R (double-binary32)
    static constexpr int OFF_I = OFF_R + EC;                        // 32-bit words from here
    // max |Q| of two blocks, row scales, max_j |n_d|, flags, barrier, wait limit
    static constexpr int I_SC = 2 * PT, I_NM = 3 * PT, I_FLAG = (I_NM + 8 + 1) & ~1, I_BAR = I_FLAG + 2, I_END = I_BAR + 4;
    static constexpr int SMEM_BYTES = 8 * OFF_I + 4 * I_END;
    static_assert(XC <= X_COLUMNS, "columns of X");
    static_assert((8 * OFF_I) % 8 == 0 && EC % 2 == 0 && EC0 % 2 == 0, "alignment");
};

// ------------------------------------------------------------ kernel
// STEP: a time step's, which writes Q~(1).  With that part in one kernel for both, calls
// without it took longer, microseconds in binary64 (double-binary32): 40,000 elements at
// N = 2 758 (468) -> 741 (437), N = 3 1,543 (887) -> 1,513 (876), 20,000 at N = 6 5,821
// (3,576) -> 5,753 (3,568).
template <int N, int NT_, class P, bool STEP>
__global__ void __launch_bounds__(NT_, NT_ == DirectSizes<N>::NT0 ? DirectSizes<N>::MIN_BLOCKS : 1)
    stp_direct_kernel(const DirectParams A) {
    using S = DirectShape<N, NT_>;
    using R = typename P::R;
    constexpr int B = S::B, T = S::T, PT = S::PT, PUL = S::PUL, NT = S::NT, NW = S::NW, G = S::G;
    extern __shared__ __align__(16) double smd[];
    R* C = reinterpret_cast<R*>(smd);
    int2* X = reinterpret_cast<int2*>(smd + S::OFF_X);
    double* raw = smd + S::OFF_K;
    R* K = reinterpret_cast<R*>(smd + (P::DW ? S::OFF_R : S::OFF_K));
    int* si = reinterpret_cast<int*>(smd + S::OFF_I);
    uint32_t* qmax = reinterpret_cast<uint32_t*>(si);
    int* scale = si + S::I_SC;
    using NM = typename std::conditional<P::DW, float, double>::type;
    NM* nmax = reinterpret_cast<NM*>(si + ((S::I_NM + 1) & ~1));
    int* flag = si + S::I_FLAG;  // [0] non-finite value met, [1] the bounded wait gave up
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    chain_wait();
    if (chain_early(N)) chain_go();
    const int64_t it0 = blockIdx.x;
    const int64_t e = A.elems ? (int64_t)A.elems[it0] : it0;
    RunPtrs run{A.q0, A.econst, A.qt, A.iout, A.qend};
    if (A.runs) run = A.runs[A.item_run[it0]];
    const double* q0 = run.q0 + e * (int64_t)(NQ * B);
    const double* ec = run.econst + e * (int64_t)A.stride + S::EC0;

    // q0 on its way to L1 while the set-up runs
    for (int i = tid; i <= NQ * B / 16; i += NT)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(q0 + min(16 * i, NQ * B - 1)));
    // the element's constants: a bulk copy that lands while C is cleared
    // (double-binary32), or plain loads
    const uint32_t bar = tc::smem_addr(si + S::I_BAR);
    if (P::DW) {
        if (tid == 0) {
            // a wait of another CTA of this context gave up: skip (the
            // launch's results are reported as failed anyway)
            flag[1] = A.status ? *reinterpret_cast<volatile const int32_t*>(A.status) : 0;
            if (!flag[1]) {
                tc::mbar_init(bar, 1);
                tc::mbar_init_fence();
                tc::fence_async_smem();
                tc::mbar_expect_tx(bar, 8u * S::EC);
                tc::bulk_g2s(tc::smem_addr(raw), ec, 8u * S::EC, bar);
                *reinterpret_cast<long long*>(si + S::I_BAR + 2) = A.wait_limit;
                if (!tc::mbar_wait_s(bar, 0, bar + 8)) {
                    tc::mbar_wait(bar, 0);  // the copy lands before the CTA exits
                    if (A.status) atomicExch(A.status, 1);
                    flag[1] = 1;
                }
            }
        }
    } else {
        for (int i = tid; i < S::EC; i += NT) raw[i] = ec[i];
    }
    for (int i = tid; i < B * PT; i += NT) C[i] = P::zero();
    for (int i = tid; i < 2 * PT; i += NT) qmax[i] = 0u;
    if (tid == 0) flag[0] = 0;
    if (P::DW) {
        __syncthreads();
        if (flag[1]) return;
        for (int i = tid; i < S::EC; i += NT) K[i] = P::of(raw[i]);
    }
    __syncthreads();
    const R* zuf = K;
    const R* iso = K + T * T + (((3 * STAR_NNZ + T * T + 4) & 1) ? 5 : 4);
    if (tid < 3) {
        // max_j |n^j_d|; read after the next barriers
        double m = 0.0;
        const double* n = raw + (iso - K);
#pragma unroll
        for (int j = 0; j < 3; ++j) m = fmax(m, fabs(n[3 * j + tid]));
        nmax[tid] = P::DW ? (NM)__double2float_ru(m) : (NM)m;
    }
    // this lane's (mode, u) of the solves: group grp of T lanes
    const int grp = lane / T, u = lane - grp * T, base = grp * T;
    const float sw = (float)((2 * u + 1) * ((u & 1) ? -1 : 1));
    const R z_lo = P::of(c_z_lo[u]), z_hi = P::of(u == T - 1 ? c_z_end[u] : c_z_hi[u]);

    const int2* ent = c_ent + entry_base(N);
    constexpr int WV = NW == 2 ? 0 : NW == 4 ? 1 : NW == 8 ? 2 : 3;
    static_assert(NW == 2 || NW == 4 || NW == 8 || NW == 16, "2, 4, 8 or 16 warps");
    const int32_t* lists = c_list + list_base(N) + list_start(N, WV);
    const double dt = raw[T * T + 2];
    double* qo = run.qt ? run.qt + e * (int64_t)(B * PT) : nullptr;
    double* io = run.iout ? run.iout + e * (int64_t)(NQ * B) : nullptr;
    double* qe = STEP && run.qend ? run.qend + e * (int64_t)(NQ * B) : nullptr;
    int buf = 0;
#pragma unroll 1
    for (int g = N; g >= 0; --g) {
        const int o = block_offset(g), d = block_size(g);
        // ---- time solves of block g: 4 groups of quantities per G modes
#pragma unroll 1
        for (int t = warp; t < 4 * ((d + G - 1) / G); t += NW) {
            const int mb = t / 4 * G, kind = t % 4;
            const bool act = grp < G && mb + grp < d;
            const int m = o + min(mb + min(grp, G - 1), d - 1);
            R* c = C + m * PT + u;
            // lane u of a group loads entry u of the task's q0
            auto load = [&](int q) { return q0[q * B + m]; };
            // b = S^{-1}w q0 + a, with entry i of the task's q0
            auto rhs = [&](R ql, int i, R a) { return P::fma1(sw, P::shfl(ql, base + i), a); };
            auto plain = [&](R b) {
                const R lo = P::shfl(b, lane - 1), hi = P::shfl(b, lane + 1);
                return P::fma(z_hi, P::select(u == T - 1, b, hi), P::mul(z_lo, P::select(u == 0, b, lo)));
            };
            // x: row q of Q; returns it in binary64
            auto put = [&](int q, R x) {
                x = P::normal(x);
                const double v64 = P::value(x);
                if (act) {
                    atomicMax(qmax + buf * PT + q * T + u, P::abs_bits(x));
                    c[q * T] = x;
                    // outputs (global layout [p][l][u], dense)
                    if (qo) qo[(q * B + m) * T + u] = v64;
                }
                return v64;
            };
            // the time integrals and Q~(1) of the task's rows, entry i in lane i of
            // the group, from lane 0's value of the row and of b + E* Q (the columns
            // of Z^{-1} but the first sum to zero).  In double-binary32 `ends` leaves
            // q0 out of b, and what remains, the step's change, is added to q0 in
            // binary64, so that a field carried from step to step keeps its bits.
            // `old`: the lane's entry of q0.  q0 may be the array written: its entries
            // read by this task are the ones it writes.
            auto finish = [&](auto row, const auto& v, const double* old, auto ends) {
                constexpr int M = sizeof(v) / sizeof(double);
                if (io) {
#pragma unroll
                    for (int i = 0; i < M; i += T) {
                        double w = __shfl_sync(0xffffffffu, v[i], base);
#pragma unroll
                        for (int k = 1; k < T && i + k < M; ++k) {
                            const double wk = __shfl_sync(0xffffffffu, v[i + k], base);
                            w = u == k ? wk : w;
                        }
                        if (act && i + u < M) io[row(i + u) * B + m] = dt * w;
                    }
                }
                if (qe) {
                    R end[M];
                    ends(end);
#pragma unroll
                    for (int i = 0; i < M; i += T) {
                        R w = P::shfl(end[i], base);
#pragma unroll
                        for (int k = 1; k < T && i + k < M; ++k) w = P::select(u == k, P::shfl(end[i + k], base), w);
                        if (act && i + u < M) {
                            const double x = P::value(P::normal(w));
                            qe[row(i + u) * B + m] = P::DW ? old[i / T] + x : x;
                        }
                    }
                }
            };
            if (kind == 0) {
                // normal stresses and pressure from D, Df, n_x u, n_y v
                double old[(4 + T - 1) / T];
                R q[(4 + T - 1) / T];
#pragma unroll
                for (int i = 0; i < 4; i += T) q[i / T] = P::of(old[i / T] = load(i + u < 3 ? i + u : QP));
                const R D = c[0], Df = c[T], gx = c[2 * T], gy = c[9 * T];
                const R gz = P::sub(P::sub(D, gx), gy);
                const R Lm = P::neg(P::fma(iso[10], Df, P::mul(iso[9], D)));
                R a[4], b[4];
                b[0] = rhs(q[0], 0, a[0] = P::fma1(-2.f, gx, Lm));
                b[1] = rhs(q[1 / T], 1 % T, a[1] = P::fma1(-2.f, gy, Lm));
                b[2] = rhs(q[2 / T], 2 % T, a[2] = P::fma1(-2.f, gz, Lm));
                b[3] = rhs(q[3 / T], 3 % T, a[3] = P::fma(iso[11], Df, P::mul(iso[10], D)));
                const double v[4] = {put(SXX, plain(b[0])), put(SXX + 1, plain(b[1])), put(SXX + 2, plain(b[2])),
                                     put(QP, plain(b[3]))};
                finish([](int r) { return r < 3 ? SXX + r : QP; }, v, old, [&](R* end) {
#pragma unroll
                    for (int r = 0; r < 4; ++r) end[r] = P::DW ? a[r] : b[r];
                });
            } else {
                // one pair (u, u_f) of velocities and one shear stress
                const int i = kind - 1;
                const double old[2] = {load(u == 0 ? QU + i : u == 1 ? QUF + i : SXY + i), T > 2 ? 0.0 : load(SXY + i)};
                const R q = P::of(old[0]), qs = T > 2 ? q : P::of(old[1]);
                const R as = P::neg(c[(SXY + i) * T]);
                const R bs = rhs(qs, T > 2 ? 2 : 0, as);
                const R Sg = c[(QU + i) * T], Gp = c[(QUF + i) * T];
                const R au = P::neg(P::fma(iso[13], Gp, P::mul(iso[12], Sg)));
                const R af = P::fma(iso[14], Gp, P::mul(iso[13], Sg));
                const R bu = rhs(q, 0, au), bf = rhs(q, 1, af);
                R xf = P::mul(zuf[u * T], P::shfl(bf, base));
#pragma unroll
                for (int s = 1; s < T; ++s) xf = P::fma(zuf[u * T + s], P::shfl(bf, base + s), xf);
                xf = P::normal(xf);
                const R by = P::fma(K[T * T + 1], xf, bu);  // + g Q_uf
                const double v[3] = {put(QU + i, plain(by)), put(QUF + i, xf), put(SXY + i, plain(bs))};
                finish([i](int r) { return (r == 0 ? QU : r == 1 ? QUF : SXY) + i; }, v, old, [&](R* end) {
                    end[0] = P::DW ? P::fma(K[T * T + 1], xf, au) : by;
                    end[1] = P::fma(K[T * T], xf, P::DW ? af : bf);
                    end[2] = P::DW ? as : bs;
                });
            }
        }
        __syncthreads();
        if (g == 0) break;
        // ---- scale of every row (k, u) of X
        for (int r = tid; r < PT; r += NT) {
            const int k = r / T, uu = r - k * T;
            NM b = 0;
            if (qmax[buf * PT + r] >= P::INF) flag[0] = 1;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int q = c_prim_q[k][i];
                if (q >= 0) b += nmax[c_prim_d[k][i]] * bound_of(qmax[buf * PT + q * T + uu], NM(0));
            }
            scale[r] = row_scale(b);
            qmax[(buf ^ 1) * PT + r] = 0u;
        }
        buf ^= 1;
        __syncthreads();
        const int dm = pass_modes(g, X_COLUMNS);
#pragma unroll 1
        for (int m0 = 0; m0 < d; m0 += dm) {
            const int nm = min(dm, d - m0);
            // ---- primitives of modes o + m0 .., quantised: column j * dm + ml
            for (int it = tid; it < 3 * nm * T; it += NT) {
                const int j = it / (nm * T), r = it - j * (nm * T), ml = r / T, uu = r - ml * T;
                const R* q = C + (o + m0 + ml) * PT + uu;
                int2* x = X + (j * dm + ml) * PT + uu;
                const int* sc = scale + uu;
                const R nx = iso[3 * j], ny = iso[3 * j + 1], nz = iso[3 * j + 2];
                auto put = [&](int k, R v) { x[k * T] = quantise(v, sc[k * T]); };
                {
                    const R v0 = q[QU * T], v1 = q[QV * T], v2 = q[QW * T];
                    const R gx = P::mul(nx, v0), gy = P::mul(ny, v1);
                    put(2, gx);
                    put(9, gy);
                    put(0, P::fma(nz, v2, P::fma(ny, v1, gx)));
                    put(3, P::fma(ny, v0, P::mul(nx, v1)));
                    put(4, P::fma(nz, v1, P::mul(ny, v2)));
                    put(5, P::fma(nz, v0, P::mul(nx, v2)));
                }
                put(1, P::fma(nz, q[QWF * T], P::fma(ny, q[QVF * T], P::mul(nx, q[QUF * T]))));
                {
                    const R xx = q[SXX * T], xy = q[SXY * T], xz = q[SXZ * T];
                    put(6, P::fma(nz, xz, P::fma(ny, xy, P::mul(nx, xx))));
                    const R yy = q[SYY * T], yz = q[SYZ * T];
                    put(7, P::fma(nz, yz, P::fma(ny, yy, P::mul(nx, xy))));
                    put(8, P::fma(nz, q[SZZ * T], P::fma(ny, yz, P::mul(nx, xz))));
                }
                const R p = q[QP * T];
                put(10, P::mul(nx, p));
                put(11, P::mul(ny, p));
                put(12, P::mul(nz, p));
            }
            __syncthreads();
            // ---- C[l] += Khat X over the pass's columns; this warp's rows
            const int i1 = lists[warp + 1];
            const int32_t* rows = lists + NW + 1;
#pragma unroll 1
            for (int i = lists[warp]; i < i1; ++i) {
                const int w = rows[i], l = w >> 21, n0 = w & 8191, n1 = n0 + ((w >> 13) & 255);
                const int2* xl = X + lane;
                long long hi[PUL];
                typename P::Low lo[PUL];
#pragma unroll
                for (int k = 0; k < PUL; ++k) {
                    hi[k] = 0;
                    lo[k] = 0;
                }
#pragma unroll 4
                for (int n = n0; n < n1; ++n) {
                    const int2 en = ent[n];
                    const int2* xc = xl + en.x;
#pragma unroll
                    for (int k = 0; k < PUL; ++k) fixed_mac(en.y, xc[32 * k], hi[k], lo[k]);
                }
#pragma unroll
                for (int k = 0; k < PUL; ++k) {
                    const int r = lane + 32 * k;
                    if (r < PT) {
                        R* c = C + l * PT + r;
                        *c = P::add_fixed(*c, hi[k], lo[k], scale[r], A, l);
                    }
                }
            }
            // the next pass's lists: this pass's rows follow its starts
            lists = rows + lists[NW];
            __syncthreads();
        }
    }
    if (!A.whole_nan) return;
    for (int r = tid; r < PT; r += NT)
        if (qmax[buf * PT + r] >= P::INF) flag[0] = 1;
    __syncthreads();
    if (flag[0]) {
        const double nan = __longlong_as_double(0x7FF8000000000000LL);
        for (int i = tid; i < NQ * B; i += NT) {
            if (io) io[i] = nan;
            if (qe) qe[i] = nan;
        }
        if (qo)
            for (int i = tid; i < B * PT; i += NT) qo[i] = nan;
    }
}

template <int N, int NT_, class P>
int launch_nt(const DirectParams& A, void* stream) {
    using S = DirectShape<N, NT_>;
    auto* kern = A.qend || A.runs ? stp_direct_kernel<N, NT_, P, true> : stp_direct_kernel<N, NT_, P, false>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM_BYTES);
    if (err != cudaSuccess) return (int)err;
    return (int)launch_chained(kern, (unsigned)A.count, NT_, S::SMEM_BYTES, stream, A);
}

// The default size is for launches that fill the chip several times over.  One
// that leaves every CTA resident at once takes as long as one element, and the
// phases of an element go faster on more warps: so the widest CTA is taken that
// leaves at most 512 threads an SM.  Binary64 (double-binary32), microseconds a
// launch, default size -> this rule, 152 SMs:
//   100 elements   N = 2 13.8 -> 10.7 (13.3 -> 10.2)   N = 3 25.6 -> 15.5 (21.1 -> 13.3)
//                  N = 4 31.0 -> 23.8 (25.8 -> 19.5)   N = 5 41.9 -> 37.0 (31.7 -> 27.5)
//   304            N = 2 14.1 -> 12.5 (13.4 -> 10.8)   N = 3 26.4 -> 19.7 (21.3 -> 14.9)
//   608            N = 2 17.9 -> 17.3 (14.9 -> 12.3)   N = 3 34.3 -> 31.3 (24.2 -> 18.6)
// and one CTA more an SM turns it round (N = 3, 912 elements on 128 threads: 45.1
// -> 62.5; 384 on 256: 28.8 -> 37.1).
// Variant 1 is the alternative size for every launch, variant 2 only for those that
// the rule leaves to the default size.
template <int N>
int cta_size(int variant, int64_t count, int64_t sms) {
    using D = DirectSizes<N>;
    if (variant == 1) return D::NT1;
    if (D::WIDEST >= 512 && D::NT0 < 512 && count <= sms) return 512;
    if (D::WIDEST >= 256 && D::NT0 < 256 && count <= 2 * sms) return 256;
    if (D::WIDEST >= 128 && D::NT0 < 128 && count <= 4 * sms) return 128;
    return variant == 2 ? D::NT1 : D::NT0;
}

int sm_count(int& sms) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (int)err;
}

template <int N, class P>
int launch_p(const DirectParams& A, int variant, void* stream) {
    using D = DirectSizes<N>;
    int sms = 0;
    if (const int err = sm_count(sms)) return err;
    const int nt = cta_size<N>(variant, A.count, sms);
    if constexpr (D::NT0 == 64)
        if (nt == 64) return launch_nt<N, 64, P>(A, stream);
    if constexpr (D::NT0 <= 128 && D::WIDEST >= 128)
        if (nt == 128) return launch_nt<N, 128, P>(A, stream);
    if constexpr (D::WIDEST >= 256)
        if (nt == 256) return launch_nt<N, 256, P>(A, stream);
    if constexpr (D::WIDEST >= 512)
        if (nt == 512) return launch_nt<N, 512, P>(A, stream);
    return (int)cudaErrorInvalidValue;
}

template <int N>
int launch_n(const DirectParams& A, bool dw, int variant, void* stream) {
    return dw ? launch_p<N, Bin32x2>(A, variant, stream) : launch_p<N, Bin64>(A, variant, stream);
}

}  // namespace

bool khat_tables(const ReferenceData& R, int columns, int stride, int warps, std::vector<int32_t>& ent,
                 std::vector<int32_t>& list, std::vector<double>& inv_d, std::string& err) {
    const int N = R.N, B = R.B;
    // The derivatives along xi, eta - xi / 2 and zeta - eta: the Dubiner basis is
    // even or odd in the direction that collapses first, so these three matrices
    // have 2,058 entries at N = 6 where those along xi, eta, zeta have 3,920
    // (adapted_directions maps the coefficients).
    std::vector<double> kh((size_t)3 * B * B);
    for (size_t i = 0; i < (size_t)B * B; ++i) {
        const double x = R.khat[i], y = R.khat[(size_t)B * B + i], z = R.khat[(size_t)2 * B * B + i];
        const double v[3] = {x, y - 0.5 * x, z - y};
        for (int j = 0; j < 3; ++j) kh[(size_t)j * B * B + i] = std::fabs(v[j]) < 1e-10 ? 0.0 : v[j];
    }
    // integer rows over one denominator per row
    std::vector<int32_t> c((size_t)3 * B * B, 0);
    inv_d.assign(B, 1.0);
    for (int l = 0; l < B; ++l) {
        int64_t d = 1, sum = 0;
        for (int j = 0; j < 3; ++j)
            for (int m = 0; m < B; ++m) {
                int64_t num = 0, den = 1;
                const double v = kh[((size_t)j * B + l) * B + m];
                if (v == 0.0) continue;
                if (!rational_of(v, num, den) || (d = std::lcm(d, den)) > (1 << 30)) {
                    err = "Khat row has no small common denominator";
                    return false;
                }
            }
        for (int j = 0; j < 3; ++j)
            for (int m = 0; m < B; ++m) {
                const double v = kh[((size_t)j * B + l) * B + m] * (double)d;
                const int64_t ci = std::llround(v);
                sum += std::llabs(ci);
                // the kernels' 64-bit sums need sum |c| < 2^23, their binary32 numerators |c| <= 2^22
                if (std::fabs(v - (double)ci) > 1e-6 || std::llabs(ci) > (1 << 22) || sum >= (1 << 23)) {
                    err = "Khat numerator out of range";
                    return false;
                }
                c[((size_t)j * B + l) * B + m] = (int32_t)ci;
            }
        inv_d[l] = 1.0 / (double)d;
    }
    // entries pass by pass, rows in order
    struct Row { int l, n0, n; };
    std::vector<std::vector<Row>> passes;
    ent.clear();
    for (int g = N; g >= 1; --g) {
        const int o = block_offset(g), d = block_size(g), dm = pass_modes(g, columns);
        for (int m0 = 0; m0 < d; m0 += dm) {
            passes.emplace_back();
            for (int l = 0; l < o; ++l) {
                const int n0 = (int)ent.size() / 2;
                for (int j = 0; j < 3; ++j)
                    for (int m = m0; m < std::min(d, m0 + dm); ++m)
                        if (const int32_t v = c[((size_t)j * B + l) * B + o + m])
                            ent.insert(ent.end(), {(j * dm + m - m0) * stride, v});
                const int n = (int)ent.size() / 2 - n0;
                if (n > 0) passes.back().push_back({l, n0, n});
            }
        }
    }
    // rows of every pass dealt to the warps: longest first, each to the least
    // loaded warp; a row costs its entries and about 14 entries' time for the
    // conversion at its end
    for (const auto& pass : passes) {
        std::vector<Row> order = pass;
        std::stable_sort(order.begin(), order.end(), [](const Row& a, const Row& b) { return a.n > b.n; });
        std::vector<std::vector<int32_t>> dealt(warps);
        std::vector<int> load(warps, 0);
        for (const Row& r : order) {
            const int w = (int)(std::min_element(load.begin(), load.end()) - load.begin());
            load[w] += r.n + 14;
            dealt[w].push_back((int32_t)((uint32_t)r.l << 21 | (uint32_t)r.n << 13 | (uint32_t)r.n0));
        }
        int32_t at = 0;
        list.push_back(0);
        for (const auto& w : dealt) list.push_back(at += (int32_t)w.size());
        for (const auto& w : dealt) list.insert(list.end(), w.begin(), w.end());
    }
    return true;
}

bool direct_tables(const ReferenceData& R, std::vector<int32_t>& ent, std::vector<int32_t>& list,
                   std::vector<double>& inv_d, std::string& err) {
    list.clear();
    for (int v = 0; v < 4; ++v) {
        const size_t start = list.size();
        if (!khat_tables(R, X_COLUMNS, NQ * R.T, 2 << v, ent, list, inv_d, err)) return false;
        // the kernel finds the next warp count's lists at a fixed place
        list.resize(start + list_part(R.N, v), 0);
    }
    return true;
}

int upload_direct_tables(int N, const std::vector<int32_t>& ent, const std::vector<int32_t>& list) {
    if (N < 1 || N > MAX_N || (int)ent.size() != 2 * khat_entries(N) ||
        (int)list.size() != list_start(N, 4))
        return (int)cudaErrorInvalidValue;
    // once per (device, N): later contexts find the same data in place
    static std::mutex mu;
    static std::set<std::pair<int, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return (int)e;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({dev, N})) return 0;
    e = cudaMemcpyToSymbol(c_ent, ent.data(), sizeof(int32_t) * ent.size(), sizeof(int2) * entry_base(N));
    if (e == cudaSuccess)
        e = cudaMemcpyToSymbol(c_list, list.data(), sizeof(int32_t) * list.size(), sizeof(int32_t) * list_base(N));
    if (e == cudaSuccess) done.insert({dev, N});
    return (int)e;
}

int direct_cta_size(int N, int variant, int64_t count) {
    int sms = 0;
    if (sm_count(sms)) return 0;
    switch (N) {
        case 1: return cta_size<1>(variant, count, sms);
        case 2: return cta_size<2>(variant, count, sms);
        case 3: return cta_size<3>(variant, count, sms);
        case 4: return cta_size<4>(variant, count, sms);
        case 5: return cta_size<5>(variant, count, sms);
        case 6: return cta_size<6>(variant, count, sms);
        default: return 0;
    }
}

int64_t direct_default_count() {
    int sms = 0;
    sm_count(sms);
    return 4 * (int64_t)sms + 1;
}

int launch_stp_direct(const DeviceReference& ref, bool dw, bool whole_nan, int32_t* status, long long wait_limit,
                      const int32_t* elems, int64_t count, const double* q0, const double* econst, double* qt,
                      double* iout, double* qend, void* stream, int variant, const RunPtrs* runs,
                      const int32_t* item_run) {
    if (count <= 0) return 0;
    DirectParams A;
    A.elems = elems;
    A.q0 = q0;
    A.econst = econst;
    A.qt = qt;
    A.iout = iout;
    A.qend = qend;
    A.count = count;
    A.stride = elem_const_stride(ref.N);
    A.inv_d = ref.inv_d;
    A.inv_d2 = reinterpret_cast<const float2*>(ref.inv_d2);
    A.status = status;
    A.wait_limit = wait_limit > 0 ? wait_limit : tc::WAIT_LIMIT_CYCLES;
    A.whole_nan = whole_nan ? 1 : 0;
    A.runs = runs;
    A.item_run = item_run;
    switch (ref.N) {
        case 1: return launch_n<1>(A, dw, variant, stream);
        case 2: return launch_n<2>(A, dw, variant, stream);
        case 3: return launch_n<3>(A, dw, variant, stream);
        case 4: return launch_n<4>(A, dw, variant, stream);
        case 5: return launch_n<5>(A, dw, variant, stream);
        case 6: return launch_n<6>(A, dw, variant, stream);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace poro
