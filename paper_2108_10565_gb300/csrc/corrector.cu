// Corrector of the ADER-DG scheme (Eq. semi_discrete integrated over one time
// step, Section "Temporal discretisation with ADER"), point source and
// receivers, in binary64 or (mixed-precision contexts) double-binary32.
//
// With I the time-integrated predictor, A_n the normal Jacobian and the Godunov
// flux F^- q_L + F^+ q_R of the paper's weak form, integration by parts gives
//   dQ = E I - sum_j Khat^j A^j I                          volume and source
//      + M^{-1} sum_f c_f Pf^T [ (A_n - F^-) tL - F^+ tR ]    faces
// with c_f = 2 |S_f| / |J| and tL, tR the traces of both sides (Floc^f = Pf^T Pf).
// The volume line is the predictor's own equation tested with 1, whose left
// side is Q~(1) - Q: a time step's predictor therefore writes Q~(1) over Q and
// the corrector adds the faces alone.  (After poro_correct's separate predictor,
// and for the unrefined binary32 predictor, volume_kernel adds the line.)
//
// Only the 4 waves that enter the element enter the face term: A_n - F^- and
// (interior) F^+ are the same matrix W V, W 13 x 4, V 4 x 13.  So each side is
// reduced to 4 rows V I before its trace.  The traces use the Dubiner basis of
// the triangle on each face with its vertices in increasing order, in which Pf
// is sparse (N = 6: 3,060 of 9,408 entries); the neighbour's trace is taken on
// its own face and then turned by the vertex permutation, block-diagonal by
// degree.  Per element at N = 5 this is 55 thousand multiply-adds, against 246
// thousand with dense traces, two 13 x 13 flux matrices and the volume term.
//
// One CTA per element; neighbours are read only through I (or, for another
// cluster, the buffered sub-step sums or the predictor), so Q is updated in
// place.  What bounds it: binary64, the FP64 pipe (N = 5: 96 % busy, 6,000
// elements in 684 microseconds); double-binary32, load and barrier latency (N = 6,
// 5,184 elements: 405 microseconds).  Double-binary32 sums run on the packed
// binary32 operations, a lane per two of the 4 columns: half the instructions, and
// a table entry is read by 2 lanes instead of 4 (a run of 5,184 elements at N = 6:
// 6.49 -> 6.33 ms a pass; 12,288 in three clusters at N = 3: 15.33 -> 15.06).  In
// binary64 that only leaves fewer lanes for the FP64 pipe (N = 5, 6,000 elements:
// 3.54 -> 3.68 ms), so there a lane has one column.  Dense traces, flux matrices and
// the volume term took 29.5 ms (binary64) and 14.6 ms (double-binary32) for 48,000
// elements at N = 5; the faces alone now take 5.5 ms in binary64.
#include <cuda_runtime.h>

#include "chain.cuh"
#include "pair_device.cuh"
#include "poro_internal.h"

namespace poro {
namespace {

// 4 steps of a row's table entries: values (binary64, or (hi, lo) binary32)
// and columns, a byte each
template <class R>
struct Entries {
    R v[4];
    uint32_t col;
};
__device__ __forceinline__ void load_values(const int4& a, const int4& b, double* v) {
    v[0] = __hiloint2double(a.y, a.x);
    v[1] = __hiloint2double(a.w, a.z);
    v[2] = __hiloint2double(b.y, b.x);
    v[3] = __hiloint2double(b.w, b.z);
}
__device__ __forceinline__ void load_values(const int4& a, const int4& b, float2* v) {
    v[0] = make_float2(__int_as_float(a.x), __int_as_float(a.y));
    v[1] = make_float2(__int_as_float(a.z), __int_as_float(a.w));
    v[2] = make_float2(__int_as_float(b.x), __int_as_float(b.y));
    v[3] = make_float2(__int_as_float(b.z), __int_as_float(b.w));
}
template <int WIDTH, class R>
__device__ __forceinline__ Entries<R> load_entries(const int4* at, int row) {
    Entries<R> e;
    load_values(__ldg(at + row), __ldg(at + WIDTH + row), e.v);
    e.col = __ldg(reinterpret_cast<const uint32_t*>(at + 2 * WIDTH) + row);
    return e;
}

// sum over one row's entries of value times PACK columns of x [][4]; the rows of
// a group of WIDTH lie side by side, and the next 4 steps load while 4 are used
template <class P, int WIDTH>
__device__ __forceinline__ typename P::V row_sum(const int4* ent, int steps, int row, const typename P::V* x) {
    using R = typename P::R;
    constexpr int C = 4 / P::PACK;
    typename P::V a = P::zeros(), b = P::zeros();
    if (steps == 0) return a;
    Entries<R> e = load_entries<WIDTH, R>(ent, row);
    for (int n = 4; n <= steps; n += 4) {
        if (n < steps) ent += face_block_words(WIDTH);
        const Entries<R> next = load_entries<WIDTH, R>(ent, row);
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            a = P::vfma(P::all(e.v[i]), x[(e.col >> 8 * i & 255) * C], a);
            b = P::vfma(P::all(e.v[i + 1]), x[(e.col >> (8 * i + 8) & 255) * C], b);
        }
        e = next;
    }
    return P::vadd(a, b);
}

template <int N>
struct FaceShape {
    static constexpr int NT = N == 1 ? 32 : N == 2 ? 96 : N <= 4 ? 128 : 256;
    static constexpr int MIN_BLOCKS = 1152 / NT;  // 1024 resident threads: 15.30 instead of 15.06 ms at N = 3
    static constexpr int PG = NT / n_modes(N) < NQ ? NT / n_modes(N) : NQ;  // threads that share a mode in the last step
    static constexpr int B = n_modes(N), DF = face_modes(N), T = N + 1, TG = (DF + 7) / 8, BG = (B + 7) / 8;
    // shared layout in 8-byte words: the factors V [13][4], W [13][4] of the
    // four faces; Y [2 sides][4 faces][B][4]; traces [2][4][DF][4]
    static constexpr int OFF_Y = 4 * FACE_FACTORS, OFF_T = OFF_Y + 2 * 4 * B * 4, END = OFF_T + 2 * 4 * DF * 4;
    static constexpr int SMEM_BYTES = 8 * END;
};

// the neighbour across one face: where its time integral over this element's
// interval comes from
struct FaceSide {
    const double* src;  // I or the buffered sum [13][B] (mode 1), or the predictor [13][B][T] (mode 2)
    int mode;           // 0: boundary
    int face, perm;     // its local face, the vertex permutation
    double w[MAX_N + 1];  // mode 2: dt_r int_a^b chi_s
};

template <int N>
__device__ void face_side(const CorrectorData& D, int64_t e, int f, FaceSide& S) {
    constexpr int B = n_modes(N), QB = NQ * B, T = N + 1;
    const int64_t nbr = D.nb[e * 4 + f];
    S.mode = 0;
    if (nbr < 0) return;
    const int tab = D.tab[e * 4 + f];
    S.face = (tab / 6) & 3;
    S.perm = tab % 6;
    const int c = D.cl ? D.cl[e] : 0, cr = D.cl ? D.cl[nbr] : 0;
    S.mode = 1;
    if (cr == c) {
        S.src = D.iout + nbr * QB;
    } else if (cr < c) {
        S.src = D.buf + (int64_t)D.slot[nbr * D.C + c] * QB;
    } else {
        // larger neighbour: dt_r sum_s Qt_s int_a^b chi_s over the sub-interval
        S.mode = 2;
        S.src = D.qt + nbr * (int64_t)(QB * T);
        const double dtr = D.econst[nbr * elem_const_stride(N) + ec_scalars(N) + 2];
        const int64_t ks = D.tick + 1 - ((int64_t)1 << c);
        const int64_t m = (ks >> cr) << cr;
        const double h = __hiloint2double((1023 - cr) << 20, 0);  // 2^-cr
        const double a = (double)(ks - m) * h, b = (double)(D.tick + 1 - m) * h;
        // int_a^b P_s(2 tau - 1) dtau = (1/2) [ (P_{s+1} - P_{s-1}) / (2s+1) ]_{2a-1}^{2b-1}
        const double x0 = 2 * a - 1, x1 = 2 * b - 1;
        double p0 = 1, p1 = 1, q0 = x0, q1 = x1;  // P_{s-1}, P_s at both ends
        S.w[0] = dtr * (0.5 * (x1 - x0));
#pragma unroll
        for (int s = 1; s < T; ++s) {
            const double r0 = ((2 * s + 1) * x0 * q0 - s * p0) * (1.0 / (s + 1)),
                         r1 = ((2 * s + 1) * x1 * q1 - s * p1) * (1.0 / (s + 1));
            S.w[s] = dtr * (((r1 - p1) - (r0 - p0)) * (0.5 / (2 * s + 1)));
            p0 = q0;
            p1 = q1;
            q0 = r0;
            q1 = r1;
        }
    }
}

template <int N, class P, bool BATCH>
__global__ void __launch_bounds__(FaceShape<N>::NT, FaceShape<N>::MIN_BLOCKS)
    face_kernel(const CorrectorData D1, const int32_t* elems, const CorrectorData* runs, const int32_t* item_run) {
    using S = FaceShape<N>;
    using R = typename P::R;
    using V = typename P::V;
    constexpr int B = S::B, DF = S::DF, T = S::T, NT = S::NT;
    constexpr int C = 4 / P::PACK, FACE = C * 2 * NQ;  // V's to 4 columns, and in one face's factors
    extern __shared__ __align__(16) double smf[];
    V* VW = reinterpret_cast<V*>(smf);
    V* Y = reinterpret_cast<V*>(smf + S::OFF_Y);
    V* tr = reinterpret_cast<V*>(smf + S::OFF_T);
    __shared__ FaceSide side[4];
    const int tid = threadIdx.x;
    // one run's data (D1), or the item's run of a batched launch over several
    // runs (their tables in global memory)
    const CorrectorData& D = BATCH ? runs[item_run[blockIdx.x]] : D1;
    const int64_t e = elems ? elems[blockIdx.x] : (int64_t)blockIdx.x;
    if (tid < 4) face_side<N>(D, e, tid, side[tid]);
    {
        const V* g = reinterpret_cast<const V*>(D.fvw) + e * (int64_t)(FACE * 4);
        for (int i = tid; i < FACE * 4; i += NT) VW[i] = g[i];
    }
    chain_wait();
    if (chain_early(N)) chain_go();
    __syncthreads();
    // Y[k][c] = sum_p V[p][c] I[p][k] of both sides of every face
    for (int it = tid; it < 8 * B; it += NT) {
        const int sf = it / B, k = it - sf * B, f = sf & 3;
        const FaceSide& F = side[f];
        if (sf >= 4 && F.mode == 0) continue;
        const double* I = sf < 4 ? D.iout + e * (int64_t)(NQ * B) : F.src;
        R v[NQ];
        if (sf < 4 || F.mode == 1) {
#pragma unroll
            for (int p = 0; p < NQ; ++p) v[p] = P::of(I[p * B + k]);
        } else {
#pragma unroll
            for (int p = 0; p < NQ; ++p) {
                double a = 0.0;
#pragma unroll
                for (int s = 0; s < T; ++s) a = ::fma(I[(p * B + k) * T + s], F.w[s], a);
                v[p] = P::of(a);
            }
        }
        const V* Vf = VW + f * FACE;
        V a[C];
#pragma unroll
        for (int c = 0; c < C; ++c) a[c] = P::vmul(Vf[c], P::all(v[0]));
#pragma unroll
        for (int p = 1; p < NQ; ++p)
#pragma unroll
            for (int c = 0; c < C; ++c) a[c] = P::vfma(Vf[C * p + c], P::all(v[p]), a[c]);
#pragma unroll
        for (int c = 0; c < C; ++c) Y[(sf * B + k) * C + c] = a[c];
    }
    __syncthreads();
    // traces of the 4 rows: 8 C lanes take 8 rows of a face (ordered by length),
    // one per row and PACK columns
    const int grp = tid / (8 * C), rs = tid / C % 8, c = tid % C;
    constexpr int GROUPS = NT / (8 * C);
    for (int t = grp; t < 8 * S::TG; t += GROUPS) {
        const int sf = t & 7, f = t & 3;  // faces of side 0: own, 1: the neighbour's; long groups first
        if (sf >= 4 && side[f].mode == 0) continue;
        const int ft = sf < 4 ? f : side[f].face;
        const int4 row = __ldg(D.ftab + face_trace_slots(N) + (ft * S::TG + (t >> 3)) * 8 + rs);
        const V a = row_sum<P, 8>(D.ftab + row.x, row.y, rs, Y + sf * B * C + c);
        if (row.z >= 0) tr[(sf * DF + row.z) * C + c] = a;
    }
    __syncthreads();
    // difference of the sides, the neighbour's turned by its permutation
    for (int it = tid; it < 4 * C * DF; it += NT) {
        const int f = it / (C * DF), ac = it - f * (C * DF);
        if (side[f].mode == 0) continue;
        const int4 row = __ldg(D.ftab + face_turn_slots(N) + side[f].perm * DF + ac / C);
        V* o = tr + f * DF * C + ac;
        *o = P::vsub(*o, row_sum<P, 1>(D.ftab + row.x, row.y, 0, tr + (4 + f) * DF * C + ac % C));
    }
    __syncthreads();
    // M^{-1} Pf^T of the 4 rows, into the own side of Y
    for (int t = grp; t < 4 * S::BG; t += GROUPS) {
        const int f = t & 3;
        const int4 row = __ldg(D.ftab + face_back_slots(N) + (f * S::BG + (t >> 2)) * 8 + rs);
        const V a = row_sum<P, 8>(D.ftab + row.x, row.y, rs, tr + f * DF * C + c);
        if (row.z >= 0) Y[(f * B + row.z) * C + c] = a;
    }
    __syncthreads();
    // Q[p][k] += sum_f sum_c (c_f W_f)[p][c] Y[f][k][c]: a thread keeps its mode's
    // Y for every PG-th quantity
    if (tid < S::PG * B) {
        const int p0 = tid / B, k = tid - p0 * B;
        double* q = D.q + e * (int64_t)(NQ * B) + k;
        V y[4 * C];
#pragma unroll
        for (int i = 0; i < 4 * C; ++i) y[i] = Y[(i / C * B + k) * C + i % C];
        for (int p = p0; p < NQ; p += S::PG) {
            const double q0 = q[p * B];
            V a[2] = {P::zeros(), P::zeros()};
#pragma unroll
            for (int i = 0; i < 4 * C; ++i)
                a[i & (2 / P::PACK - 1)] = P::vfma(VW[i / C * FACE + C * (NQ + p) + i % C], y[i], a[i & (2 / P::PACK - 1)]);
            q[p * B] = q0 + P::value(P::normal(P::sum(P::PACK == 1 ? P::vadd(a[0], a[1]) : a[0])));
        }
    }
}

// Q += E I - sum_j Khat^j A^j I in binary64: the volume line for a predictor
// that did not write Q~(1) itself (poro_correct after a separate predictor, the
// unrefined form).  A thread takes a mode's star product in one direction, then one
// row and mode of the sum.  What bounds it: the binary64 pipe, so the division by dt
// comes once, at the end.  poro_correct, this kernel and the faces, milliseconds in
// binary64 (double-binary32): 48,000 elements at N = 2 1.71 (1.22), N = 3 3.93 (3.02);
// 16,464 at N = 5 5.10 (4.06), 10,368 at N = 6 5.44 (4.39).  One thread a mode for all
// three directions, with divisions there: 4.83 (4.34), 6.83 (5.91), 6.02 (4.98), 6.23 (5.16).
constexpr int volume_threads(int N) { return NQ * n_modes(N) < 256 ? (NQ * n_modes(N) + 31) / 32 * 32 : 256; }
template <bool BATCH>
__global__ void __launch_bounds__(256) volume_kernel(int N, const CorrectorData D1, const int32_t* elems,
                                                     const CorrectorData* runs, const int32_t* item_run) {
    extern __shared__ double smv[];
    chain_wait();
    chain_go();
    const int B = n_modes(N), QB = NQ * B, NT = blockDim.x;
    double* I = smv;           // [13][B]
    double* X = I + QB;        // [3][13][B]: dt A^j I
    double* star = X + 3 * QB;
    const int tid = threadIdx.x;
    const CorrectorData& D = BATCH ? runs[item_run[blockIdx.x]] : D1;
    const int64_t e = elems ? elems[blockIdx.x] : (int64_t)blockIdx.x;
    const double* ec = D.econst + e * elem_const_stride(N);
    const double* sc = ec + ec_scalars(N);
    for (int i = tid; i < QB; i += NT) I[i] = D.iout[e * QB + i];
    for (int i = tid; i < 3 * STAR_NNZ; i += NT) star[i] = ec[i];
    __syncthreads();
    for (int i = tid; i < 3 * B; i += NT) {
        const int j = i / B, l = i - j * B;
        const double* sj = star + j * STAR_NNZ;
        double acc[NQ];
#pragma unroll
        for (int p = 0; p < NQ; ++p) acc[p] = 0.0;
#pragma unroll
        for (int n = 0; n < STAR_NNZ; ++n) acc[star_row(n)] = fma(sj[n], I[star_col(n) * B + l], acc[star_row(n)]);
#pragma unroll
        for (int p = 0; p < NQ; ++p) X[j * QB + p * B + l] = acc[p];
    }
    __syncthreads();
    const double ev = sc[0], gv = sc[1], dt = sc[2];
    double* q = D.q + e * QB;
    for (int i = tid; i < QB; i += NT) {
        const int p = i / B, k = i - p * B;
        double acc = 0.0;
        for (int j = 0; j < 3; ++j) {
            const int32_t* kr = D.krow + j * (B + 1) + k;
            const double* x = X + j * QB + p * B;
            for (int n = kr[0]; n < kr[1]; ++n) acc = fma(D.kval[n], x[D.kcol[n]], acc);
        }
        // Darcy source term E I: u rows from u_f, u_f rows from u_f
        if (p >= QU && p <= QW) acc = fma(-gv, I[(p + QUF - QU) * B + k], acc);
        if (p >= QUF) acc = fma(-ev, I[i], acc);
        q[i] -= acc / dt;
    }
}

// buffers of the sub-step integrals for larger neighbours, one CTA per buffer:
// one of level L restarts at ticks that are multiples of 2^L.  (A CTA per element
// of the cluster, most of them without a buffer, took 9 microseconds for 4,676.)
__global__ void lts_buffer_kernel(int QB, const int4* items, const double* iout, double* buf, int64_t tick) {
    const int4 it = items[blockIdx.x];
    chain_wait();
    chain_go();
    const bool reset = (tick & (((int64_t)1 << it.z) - 1)) == 0;
    const double* I = iout + (int64_t)it.x * QB;
    double* b = buf + (int64_t)it.y * QB;
    for (int i = threadIdx.x; i < QB; i += blockDim.x) b[i] = reset ? I[i] : b[i] + I[i];
}

// q[elem] += (S(t1) - S(t0)) vec over the step [(k+1-len) dt, (k+1) dt] with S the
// antiderivative of the Ricker wavelet, S(t) = (t - tc) exp(-(pi f0 (t - tc))^2), k = *tick
// + k_rel + k_add; one CTA
__device__ void add_source(int QB, const TickItem& it, int64_t k_add) {
    __shared__ double S[2];
    if (threadIdx.x < 2) {  // S(t0), S(t1)
        const int64_t k = *it.tick + it.k_rel + k_add;
        const double t = (double)(threadIdx.x == 0 ? k + 1 - it.len : k + 1) * it.dt;
        const double a = 3.14159265358979323846 * it.f0 * (t - it.tc);
        S[threadIdx.x] = (t - it.tc) * exp(-a * a);
    }
    __syncthreads();
    const double amp = S[1] - S[0];
    double* q = it.q + it.elem * QB;
    for (int i = threadIdx.x; i < QB; i += blockDim.x) q[i] += amp * it.vec[i];
}

__global__ void tick_advance_kernel(int64_t* tick, int64_t n) {
    chain_wait();
    chain_go();
    *tick += n;
}

__global__ void ticks_advance_kernel(int64_t* const* ticks, int count, int64_t n) {
    chain_wait();
    chain_go();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) *ticks[i] += n;
}

// The source items of several runs, those of one element side by side: its first
// item's CTA adds them all, in order.  Or one CTA for a run's list.
__global__ void source_items_kernel(int QB, const TickItem* items) {
    chain_wait();
    chain_go();
    const TickItem* it = items + blockIdx.x;
    const TickItem* end = items + gridDim.x;
    const double* q = it->q;
    const int64_t elem = it->elem;
    auto same = [&](const TickItem& o) { return o.q == q && o.elem == elem; };
    if (it > items && same(it[-1])) return;
    for (; it < end && same(*it); ++it) {
        add_source(QB, *it, 0);
        __syncthreads();
    }
}
__global__ void source_list_kernel(int QB, const TickItem* items, int count, int64_t k_add) {
    chain_wait();
    chain_go();
    for (int i = 0; i < count; ++i) {
        add_source(QB, items[i], k_add);
        __syncthreads();
    }
}

// one CTA per receiver item: out[*counter] = Q[elem] phi, then ++*counter.  A warp
// per quantity, lanes over the modes: all that it costs is one pass through the
// load, shuffle and store latencies (4 warps, each taking 3 or 4 quantities in
// turn: a cycle of 384 elements at N = 2 took 46.5 microseconds, now 43.6).
constexpr int RNT = 32 * NQ;
__global__ void __launch_bounds__(RNT) receiver_items_kernel(int B, const TickItem* items) {
    const TickItem& it = items[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    chain_wait();
    chain_go();
    const int32_t idx = *it.counter;
    const double* q = it.q + it.elem * (int64_t)(NQ * B) + warp * B;
    double acc = 0.0;
    for (int l = lane; l < B; l += 32) acc = fma(q[l], it.vec[l], acc);
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
    if (lane == 0) it.out[(int64_t)idx * NQ + warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) *it.counter = idx + 1;
}

template <int N, class P>
int launch_faces_p(const CorrectorData& d, const int32_t* elems, int64_t count, void* stream, const CorrectorData* runs,
                   const int32_t* item_run) {
    using S = FaceShape<N>;
    auto* kern = runs ? face_kernel<N, P, true> : face_kernel<N, P, false>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM_BYTES);
    if (err != cudaSuccess) return (int)err;
    return (int)launch_chained(kern, (unsigned)count, S::NT, S::SMEM_BYTES, stream, d, elems, runs, item_run);
}

template <int N>
int launch_faces_n(const CorrectorData& d, const int32_t* elems, int64_t count, void* stream, const CorrectorData* runs,
                   const int32_t* item_run) {
    return d.dw ? launch_faces_p<N, Bin32x2Base>(d, elems, count, stream, runs, item_run)
                : launch_faces_p<N, Bin64Base>(d, elems, count, stream, runs, item_run);
}

}  // namespace

int launch_corrector(const CorrectorData& d, bool volume, const int32_t* elems, int64_t count, void* stream,
                     const CorrectorData* runs, const int32_t* item_run) {
    if (count <= 0) return 0;
    if (volume) {
        const size_t smem = sizeof(double) * (4 * NQ * n_modes(d.N) + 3 * STAR_NNZ);  // 36 KB at N = 6
        auto* kern = runs ? volume_kernel<true> : volume_kernel<false>;
        if (const cudaError_t err = launch_chained(kern, (unsigned)count, volume_threads(d.N), smem, stream, d.N, d, elems,
                                                   runs, item_run))
            return (int)err;
    }
    switch (d.N) {
        case 1: return launch_faces_n<1>(d, elems, count, stream, runs, item_run);
        case 2: return launch_faces_n<2>(d, elems, count, stream, runs, item_run);
        case 3: return launch_faces_n<3>(d, elems, count, stream, runs, item_run);
        case 4: return launch_faces_n<4>(d, elems, count, stream, runs, item_run);
        case 5: return launch_faces_n<5>(d, elems, count, stream, runs, item_run);
        case 6: return launch_faces_n<6>(d, elems, count, stream, runs, item_run);
        default: return (int)cudaErrorInvalidValue;
    }
}

int launch_lts_buffers(int N, const int4* items, int64_t count, const double* iout, double* buf, int64_t tick,
                       void* stream) {
    if (count <= 0) return 0;
    return (int)launch_chained(lts_buffer_kernel, (unsigned)count, 128, 0, stream, NQ * n_modes(N), items, iout, buf, tick);
}

int launch_tick_sources(int N, const TickItem* items, int64_t count, void* stream) {
    if (count <= 0) return 0;
    return (int)launch_chained(source_items_kernel, (unsigned)count, 256, 0, stream, NQ * n_modes(N), items);
}

int launch_source_list(int N, const TickItem* items, int count, int64_t k_add, void* stream) {
    if (count <= 0) return 0;
    return (int)launch_chained(source_list_kernel, 1u, 256, 0, stream, NQ * n_modes(N), items, count, k_add);
}

int launch_tick_receivers(int N, const TickItem* items, int64_t count, void* stream) {
    if (count <= 0) return 0;
    return (int)launch_chained(receiver_items_kernel, (unsigned)count, RNT, 0, stream, n_modes(N), items);
}

int launch_ticks_advance(int64_t* const* ticks, int count, int64_t n, void* stream) {
    if (count <= 0) return 0;
    return (int)launch_chained(ticks_advance_kernel, (unsigned)((count + 127) / 128), 128, 0, stream, ticks, count, n);
}

int launch_tick_advance(int64_t* tick, int64_t n, void* stream) {
    return (int)launch_chained(tick_advance_kernel, 1u, 1, 0, stream, tick, n);
}

}  // namespace poro
