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
// place.  What bounds it: binary64, the FP64 pipe; double-binary32, issue slots.
#include <cuda_runtime.h>

#include "pair_device.cuh"
#include "poro_internal.h"

namespace poro {
namespace {

// a table entry: value (binary64, or (hi, lo) binary32) and column
template <class P>
__device__ __forceinline__ void load_entry(const int4* at, typename P::R& v, int& col);
template <>
__device__ __forceinline__ void load_entry<Bin64Base>(const int4* at, double& v, int& col) {
    const int4 e = __ldg(at);
    v = __hiloint2double(e.y, e.x);
    col = e.z;
}
template <>
__device__ __forceinline__ void load_entry<Bin32x2Base>(const int4* at, float2& v, int& col) {
    const int4 e = __ldg(at);
    v = make_float2(__int_as_float(e.x), __int_as_float(e.y));
    col = e.z;
}

// sum over one row's entries of value times x[4 column], `width` rows a step;
// the next 4 entries load while 4 are used
template <class P>
__device__ __forceinline__ typename P::R row_sum(const int4* ent, int steps, int width, const typename P::R* x) {
    typename P::R a = P::zero(), b = P::zero(), v[4];
    int k[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) load_entry<P>(ent + i * width, v[i], k[i]);
    for (int n = 4; n <= steps; n += 4) {
        typename P::R w[4];
        int m[4];
        const int4* next = ent + (n < steps ? n : 0) * width;
#pragma unroll
        for (int i = 0; i < 4; ++i) load_entry<P>(next + i * width, w[i], m[i]);
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            a = P::fma(v[i], x[k[i] * 4], a);
            b = P::fma(v[i + 1], x[k[i + 1] * 4], b);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i] = w[i];
            k[i] = m[i];
        }
    }
    return P::add(a, b);
}

template <int N>
struct FaceShape {
    // a thread takes whole columns of the first step (8 B of them)
    static constexpr int NT = N == 1 ? 32 : N == 2 ? 96 : N <= 4 ? 160 : 224, NW = NT / 32;
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
__global__ void __launch_bounds__(FaceShape<N>::NT)
    face_kernel(const CorrectorData D1, const int32_t* elems, const CorrectorData* runs, const int32_t* item_run) {
    using S = FaceShape<N>;
    using R = typename P::R;
    constexpr int B = S::B, DF = S::DF, T = S::T, NT = S::NT, NW = S::NW;
    extern __shared__ __align__(16) double smf[];
    R* VW = reinterpret_cast<R*>(smf);
    R* Y = reinterpret_cast<R*>(smf) + S::OFF_Y;
    R* tr = reinterpret_cast<R*>(smf) + S::OFF_T;
    __shared__ FaceSide side[4];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // one run's data (D1), or the item's run of a batched launch over several
    // runs (their tables in global memory)
    const CorrectorData& D = BATCH ? runs[item_run[blockIdx.x]] : D1;
    const int64_t e = elems ? elems[blockIdx.x] : (int64_t)blockIdx.x;
    if (tid < 4) face_side<N>(D, e, tid, side[tid]);
    {
        const R* g = reinterpret_cast<const R*>(D.fvw) + e * (int64_t)(4 * FACE_FACTORS);
        for (int i = tid; i < 4 * FACE_FACTORS; i += NT) VW[i] = g[i];
    }
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
            for (int p = 0; p < NQ; ++p) v[p] = P::of(__ldg(I + p * B + k));
        } else {
#pragma unroll
            for (int p = 0; p < NQ; ++p) {
                double a = 0.0;
#pragma unroll
                for (int s = 0; s < T; ++s) a = ::fma(__ldg(I + (p * B + k) * T + s), F.w[s], a);
                v[p] = P::of(a);
            }
        }
        const R* V = VW + f * FACE_FACTORS;
        R a[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) a[c] = P::mul(V[c], v[0]);
#pragma unroll
        for (int p = 1; p < NQ; ++p)
#pragma unroll
            for (int c = 0; c < 4; ++c) a[c] = P::fma(V[4 * p + c], v[p], a[c]);
        R* y = Y + (sf * B + k) * 4;
#pragma unroll
        for (int c = 0; c < 4; ++c) y[c] = a[c];
    }
    __syncthreads();
    // traces of the 4 rows: a warp takes 8 rows of a face (ordered by length),
    // lanes (row, c)
    const int rs = lane >> 2, c = lane & 3;
    for (int t = warp; t < 8 * S::TG; t += NW) {
        const int sf = t / S::TG, f = sf & 3;  // sides 0: own, 1: the neighbour's
        if (sf >= 4 && side[f].mode == 0) continue;
        const int ft = sf < 4 ? f : side[f].face;
        const int4 row = __ldg(D.ftab + face_trace_slots(N) + (ft * S::TG + t % S::TG) * 8 + rs);
        const R a = row_sum<P>(D.ftab + row.x + rs, row.y, 8, Y + sf * B * 4 + c);
        if (row.z >= 0) tr[(sf * DF + row.z) * 4 + c] = a;
    }
    __syncthreads();
    // difference of the sides, the neighbour's turned by its permutation
    for (int it = tid; it < 16 * DF; it += NT) {
        const int f = it / (4 * DF), ac = it - f * (4 * DF);
        if (side[f].mode == 0) continue;
        const int4 row = __ldg(D.ftab + face_turn_slots(N) + side[f].perm * DF + (ac >> 2));
        R* o = tr + f * DF * 4 + ac;
        *o = P::sub(*o, row_sum<P>(D.ftab + row.x, row.y, 1, tr + (4 + f) * DF * 4 + (ac & 3)));
    }
    __syncthreads();
    // M^{-1} Pf^T of the 4 rows, into the own side of Y
    for (int t = warp; t < 4 * S::BG; t += NW) {
        const int f = t / S::BG;
        const int4 row = __ldg(D.ftab + face_back_slots(N) + t * 8 + rs);
        const R a = row_sum<P>(D.ftab + row.x + rs, row.y, 8, tr + f * DF * 4 + c);
        if (row.z >= 0) Y[(f * B + row.z) * 4 + c] = a;
    }
    __syncthreads();
    // Q[p][k] += sum_f sum_c (c_f W_f)[p][c] Y[f][k][c]
    double* q = D.q + e * (int64_t)(NQ * B);
    for (int it = tid; it < NQ * B; it += NT) {
        const int p = it / B, k = it - p * B;
        const double q0 = q[it];
        R a[2] = {P::zero(), P::zero()};
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            const R* W = VW + f * FACE_FACTORS + 4 * NQ + 4 * p;
            const R* y = Y + (f * B + k) * 4;
#pragma unroll
            for (int cc = 0; cc < 4; ++cc) a[cc & 1] = P::fma(W[cc], y[cc], a[cc & 1]);
        }
        q[it] = q0 + P::value(P::normal(P::add(a[0], a[1])));
    }
}

// Q += E I - sum_j Khat^j A^j I in binary64: the volume line for a predictor
// that did not write Q~(1) itself
constexpr int VNT = 128;
template <bool BATCH>
__global__ void __launch_bounds__(VNT) volume_kernel(int N, const CorrectorData D1, const int32_t* elems,
                                                     const CorrectorData* runs, const int32_t* item_run) {
    extern __shared__ double smv[];
    const int B = n_modes(N), QB = NQ * B;
    double* I = smv;      // [13][B]
    double* X = I + QB;   // [13][B]
    const int tid = threadIdx.x;
    const CorrectorData& D = BATCH ? runs[item_run[blockIdx.x]] : D1;
    const int64_t e = elems ? elems[blockIdx.x] : (int64_t)blockIdx.x;
    const double* ec = D.econst + e * elem_const_stride(N);
    const double* sc = ec + ec_scalars(N);
    const double ev = sc[0] / sc[2], gv = sc[1] / sc[2];
    double* q = D.q + e * QB;
    for (int i = tid; i < QB; i += VNT) I[i] = D.iout[e * QB + i];
    for (int j = 0; j < 3; ++j) {
        __syncthreads();
        const double* sj = ec + j * STAR_NNZ;
        for (int l = tid; l < B; l += VNT) {
            double acc[NQ];
#pragma unroll
            for (int p = 0; p < NQ; ++p) acc[p] = 0.0;
#pragma unroll
            for (int n = 0; n < STAR_NNZ; ++n) acc[star_row(n)] = fma(sj[n], I[star_col(n) * B + l], acc[star_row(n)]);
#pragma unroll
            for (int p = 0; p < NQ; ++p) X[p * B + l] = acc[p] / sc[2];
        }
        __syncthreads();
        const int32_t* kr = D.krow + j * (B + 1);
        for (int i = tid; i < QB; i += VNT) {
            const int p = i / B, k = i - p * B;
            double acc = 0.0;
            for (int n = kr[k]; n < kr[k + 1]; ++n) acc = fma(D.kval[n], X[p * B + D.kcol[n]], acc);
            if (j == 0) {
                // Darcy source term E I: u rows from u_f, u_f rows from u_f
                if (p >= QU && p <= QW) acc = fma(-gv, I[(p + QUF - QU) * B + k], acc);
                if (p >= QUF) acc = fma(-ev, I[i], acc);
            }
            q[i] -= acc;
        }
    }
}

// buffers of the sub-step integrals for larger neighbours: level L restarts
// at ticks that are multiples of 2^L
__global__ void lts_buffer_kernel(int QB, int C, const int32_t* elems, int64_t count, const int32_t* slot,
                                  const double* iout, double* buf, int64_t tick) {
    for (int64_t it = blockIdx.x; it < count; it += gridDim.x) {
        const int64_t e = elems[it];
        for (int L = 0; L < C; ++L) {
            const int sl = slot[e * C + L];
            if (sl < 0) continue;
            const bool reset = (tick & (((int64_t)1 << L) - 1)) == 0;
            double* b = buf + (int64_t)sl * QB;
            const double* I = iout + e * QB;
            for (int i = threadIdx.x; i < QB; i += blockDim.x) b[i] = reset ? I[i] : b[i] + I[i];
        }
    }
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

__global__ void tick_advance_kernel(int64_t* tick, int64_t n) { *tick += n; }

__global__ void ticks_advance_kernel(int64_t* const* ticks, int count, int64_t n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) *ticks[i] += n;
}

// one CTA per source item (of several runs), or one CTA for a run's list (its
// sources may share an element)
__global__ void source_items_kernel(int QB, const TickItem* items) { add_source(QB, items[blockIdx.x], 0); }
__global__ void source_list_kernel(int QB, const TickItem* items, int count, int64_t k_add) {
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
    kern<<<(unsigned)count, S::NT, S::SMEM_BYTES, (cudaStream_t)stream>>>(d, elems, runs, item_run);
    return (int)cudaGetLastError();
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
        const size_t smem = sizeof(double) * 2 * NQ * n_modes(d.N);
        auto* kern = runs ? volume_kernel<true> : volume_kernel<false>;
        kern<<<(unsigned)count, VNT, smem, (cudaStream_t)stream>>>(d.N, d, elems, runs, item_run);
        if (const cudaError_t err = cudaGetLastError()) return (int)err;
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

int launch_lts_buffers(int N, int C, const int32_t* elems, int64_t count, const int32_t* slot, const double* iout,
                       double* buf, int64_t tick, void* stream) {
    if (count <= 0) return 0;
    const int64_t grid = count < 65536 ? count : 65536;
    lts_buffer_kernel<<<(unsigned)grid, 128, 0, (cudaStream_t)stream>>>(NQ * n_modes(N), C, elems, count, slot, iout,
                                                                       buf, tick);
    return (int)cudaGetLastError();
}

int launch_tick_sources(int N, const TickItem* items, int64_t count, void* stream) {
    if (count <= 0) return 0;
    source_items_kernel<<<(unsigned)count, 256, 0, (cudaStream_t)stream>>>(NQ * n_modes(N), items);
    return (int)cudaGetLastError();
}

int launch_source_list(int N, const TickItem* items, int count, int64_t k_add, void* stream) {
    if (count <= 0) return 0;
    source_list_kernel<<<1, 256, 0, (cudaStream_t)stream>>>(NQ * n_modes(N), items, count, k_add);
    return (int)cudaGetLastError();
}

int launch_tick_receivers(int N, const TickItem* items, int64_t count, void* stream) {
    if (count <= 0) return 0;
    receiver_items_kernel<<<(unsigned)count, RNT, 0, (cudaStream_t)stream>>>(n_modes(N), items);
    return (int)cudaGetLastError();
}

int launch_ticks_advance(int64_t* const* ticks, int count, int64_t n, void* stream) {
    if (count <= 0) return 0;
    ticks_advance_kernel<<<(unsigned)((count + 127) / 128), 128, 0, (cudaStream_t)stream>>>(ticks, count, n);
    return (int)cudaGetLastError();
}

int launch_tick_advance(int64_t* tick, int64_t n, void* stream) {
    tick_advance_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(tick, n);
    return (int)cudaGetLastError();
}

}  // namespace poro
