// K11: the space-time predictor with sub-cell material variation (Section
// "Limitations": material varying inside an element turns the stiffness
// matrices into 3-tensors), in binary64, one element per CTA.
//
// The element's Jacobians and source matrix vary linearly inside it:
// A^{j*}(xi) = sum_r A^{j*}_r phi_r(xi), E*(xi) = sum_r E*_r phi_r(xi) over the
// four Dubiner modes of degree <= 1.  With the M^{-1}-scaled mass 3-tensor
// Mh3_r[k, l] = int phi_k phi_r phi_l / M_kk, the weighted derivative tensor is
// Mh3_r Khat^j (d_j phi_l lies in the basis), so the system is
//   Y Q = Y_0 Q + sum_{r>=1} Mh3_r (sum_j Khat^j (A^{j*}_r Q) - E*_r Q) = b0,
// Y_0 the constant-material operator of the mode-0 (mean) Jacobians, which
// Algorithm 3 solves.  A material of degree 1 couples modes of equal degree,
// so Lemma 1's block structure does not hold for Y itself; the kernel iterates
//   Q_{k+1} = Y_0^{-1} (b0 - Delta Q_k),  Delta = Y - Y_0,
// (Richardson iteration preconditioned by Algorithm 3 on the mean material)
// until max |Q_{k+1} - Q_k| <= tol max |Q_{k+1}|, at most max_iter times.
// The contraction factor is about the relative variation of the material
// inside the element.
//
// The three variation terms share their derivatives: isotropic Jacobians act
// through 13 primitive rows of the geometry alone (those of stp_direct.cu, here with
// n^j = dt grad xi_j), so W = sum_j Khat^j prim^j(Q_k) is formed once an iteration
// and every mode's term is W combined with 9 of its Jacobians' entries.  That is 2
// passes of Khat products (integer sums) an iteration, one over W and one in the
// sweep, instead of 4, and 26 instead of 162 multiply-adds a mode, time mode and
// direction for the variations.  N = 4, 500 elements: 3.90 -> 2.61 ms a pass, the
// binary64 pipe 65 % busy.  What bounds it beside that: latency, of the sweep's small
// blocks and of the barriers between them (2 elements an SM at N = 4, 1 from N = 5 on).
//
// Shared memory: U (iterate), V (right-hand side, then the next iterate) and W
// in the b / Q layout of the sweep, its fixed-point X (whose place takes a mode's
// combined term in between), the mean element constants, those of the variation and
// the reduction words.
#include <cuda_runtime.h>

#include "alg3_device.cuh"

namespace poro {
namespace {

struct SubParams {
    const double* q0;
    const double* econst;  // mean-material constants (the layout of the FP64 predictor)
    const double* evar;    // per element: dt grad xi_j on the primitive rows, 11 words per variation mode
    double* qt;
    double* iout;
    int32_t* iters;        // per element: iterations, negative if not converged
    int64_t count;
    int stride, vstride;
    KhatRows khat;
    const int32_t* m3_row;  // [3][B + 1], absolute into m3_col / m3_val
    const int32_t* m3_col;
    const double* m3_val;
    double tol;
    int max_iter;
};

constexpr int NVAR = 3;  // variation modes r = 1..3

// the 13 primitive rows, in the form that khat_block takes
struct Primitives {
    static constexpr int NQ = poro::NQ, NNZ = PRIM_NNZ;
    PORO_HD static constexpr int row(int n) { return prim_row(n); }
    PORO_HD static constexpr int col(int n) { return prim_col(n); }
};

template <int N, int NT_>
struct SubShape : SweepShape<N, BiotSystem, subcell_columns(N)> {
    using S = SweepShape<N, BiotSystem, subcell_columns(N)>;
    static constexpr int NT = NT_, NW = NT_ / 32;
    static constexpr int OFF_V = S::SQ;
    static constexpr int OFF_W = 2 * S::SQ;
    static constexpr int OFF_X = 3 * S::SQ;
    static constexpr int OFF_STAR = OFF_X + S::X_WORDS;            // mean constants: star, zuf, sc (EC words)
    static constexpr int EC = 3 * STAR_NNZ + S::T * S::T + 4;
    static constexpr int OFF_VAR = OFF_STAR + EC;                   // constants of the variation
    static constexpr int VAR = 3 * PRIM_NNZ + NVAR * SUBCELL_MODE;
    static constexpr int OFF_MAX = OFF_VAR + VAR;                   // max_j of the mean's star, of the primitives'
    static constexpr int OFF_RED = OFF_MAX + STAR_NNZ + PRIM_NNZ;   // 2 NW reduction words
    static constexpr int OFF_I = OFF_RED + 2 * NW;
    static constexpr int SMEM_BYTES = 8 * OFF_I + 4 * (S::I_WORDS + NQ + 1);
    // rows of a combined term that X's place holds: all of them up to N = 5
    static constexpr int CHUNK = S::X_WORDS / S::QS < NQ ? S::X_WORDS / S::QS : NQ;
    static_assert(CHUNK >= 1, "room for a row of a combined term");
};

// row p of sum_j Khat^j A^{j*}_r U - E*_r U at one (mode, time mode), from the
// primitive sums w and the iterate u (both [13], stride QS), with the
// x-direction entries k of the Jacobians and k[9] = e, k[10] = g of E*
template <int QS>
__device__ __forceinline__ double combine_row(int p, const double* w, const double* u, const double* k) {
    const double D = w[0], Df = w[QS];
    if (p <= SZZ) {  // normal stresses: k1 D + k2 Df + 2 k0 n_p u_p
        const double gx = w[2 * QS], gy = w[9 * QS];
        const double gp = p == SXX ? gx : p == SYY ? gy : D - gx - gy;
        return fma(2.0 * k[0], gp, fma(k[2], Df, k[1] * D));
    }
    if (p < QU) return k[0] * w[p * QS];
    if (p == QP) return fma(k[4], Df, k[3] * D);
    const int i = p < QP ? p - QU : p - QUF;
    const double Sg = w[(QU + i) * QS], G = w[(QUF + i) * QS], f = u[(QUF + i) * QS];
    return p < QP ? fma(-k[10], f, fma(k[6], G, k[5] * Sg)) : fma(-k[9], f, fma(k[8], G, k[7] * Sg));
}

// W = sum_j Khat^j prim^j(U) over all degree blocks (strictly upper in degree:
// rows l < o_g take column block g); begins after and ends with a barrier
template <int N, int NT, class S>
__device__ void flux_term(double* W, const double* U, const double* prim, const KhatRows& K, const SweepScratch<S>& X) {
    constexpr int T = S::T;
    const int32_t* list = K.list;
    for (int i = threadIdx.x; i < S::SQ; i += NT) W[i] = 0.0;
#pragma unroll 1
    for (int g = N; g >= 1; --g) {
        const int o = block_offset(g), d = block_size(g);
        for (int it = threadIdx.x; it < NQ * d * T; it += NT) {
            const int q = it / (d * T), mu = it - q * (d * T);
            atomicMax(X.qmax(0) + q * T + mu % T, (uint32_t)__double2hiint(U[q * S::QS + o * T + mu]) & 0x7FFFFFFFu);
        }
        __syncthreads();
        khat_block<N, NT, Primitives, S, 1>(W, U, g, prim, K, list, X, X.qmax(0), X.qmax(1));
        for (int i = threadIdx.x; i < S::PT; i += NT) X.qmax(0)[i] = 0u;
        __syncthreads();
    }
}

// V -= Mh3_r W for the rows [p0, p0 + np) of quantities, W their place; ends with
// a barrier
template <int NT, class S, int CHUNK>
__device__ void mass_term(double* V, const double* W, int p0, int np, const int32_t* row, const int32_t* col,
                          const double* val) {
    constexpr int B = S::B, T = S::T, QS = S::QS, PUL = (CHUNK * T + 31) / 32, NW = NT / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = warp; k < B; k += NW) {
        const int n0 = __ldg(row + k), n1 = __ldg(row + k + 1);
        double acc[PUL];
#pragma unroll
        for (int q = 0; q < PUL; ++q) acc[q] = 0.0;
        for (int n = n0; n < n1; ++n) {
            const double v = __ldg(val + n);
            const int l = __ldg(col + n) * T;
#pragma unroll
            for (int q = 0; q < PUL; ++q) {
                const int pu = lane + 32 * q;
                if (pu < np * T) acc[q] = fma(v, W[(pu / T) * QS + l + pu % T], acc[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < PUL; ++q) {
            const int pu = lane + 32 * q;
            if (pu < np * T) V[(p0 + pu / T) * QS + k * T + pu % T] -= acc[q];
        }
    }
    __syncthreads();
}

template <int N, int NT_>
__global__ void __launch_bounds__(NT_) stp_subcell_kernel(const SubParams P) {
    using S = SubShape<N, NT_>;
    constexpr int B = S::B, T = S::T, NT = S::NT, NW = S::NW, QS = S::QS, BT = B * T;
    extern __shared__ double sm[];
    double* bufs[2] = {sm, sm + S::OFF_V};
    double* W = sm + S::OFF_W;
    double* star = sm + S::OFF_STAR;
    double* zuf = star + 3 * STAR_NNZ;
    double* sc = zuf + T * T;
    double* var = sm + S::OFF_VAR;
    double* smax = sm + S::OFF_MAX;
    unsigned long long* red = reinterpret_cast<unsigned long long*>(sm + S::OFF_RED);
    using Sweep = typename S::S;
    int* ints = reinterpret_cast<int*>(sm + S::OFF_I);
    const SweepScratch<Sweep> X{reinterpret_cast<int2*>(sm + S::OFF_X), ints, smax, ints + S::I_ROW};
    const SweepScratch<Sweep> Xp{X.X, ints, smax + STAR_NNZ, ints + S::I_WORDS};
    double* term = sm + S::OFF_X;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    for (int64_t e = blockIdx.x; e < P.count; e += gridDim.x) {
        const double* q0 = P.q0 + e * (int64_t)(NQ * B);
        const double* ec = P.econst + e * (int64_t)P.stride;
        const double* ev = P.evar + e * (int64_t)P.vstride;
        for (int i = tid; i < S::EC; i += NT) star[i] = ec[i];
        for (int i = tid; i < S::VAR; i += NT) var[i] = ev[i];
        double* U = bufs[0];
        double* V = bufs[1];
        init_rhs<NT, Sweep>(U, q0);
        __syncthreads();
        sweep_setup<NT, Sweep, BiotSystem>(X, smax, star);
        star_setup<NT, Primitives>(Xp.row, smax + STAR_NNZ, var);
        __syncthreads();
        alg3_sweep<N, NT, BiotSystem, Sweep>(U, star, zuf, sc[1], P.khat, X);  // Q_0 = Y_0^{-1} b0
        int it = 0;
        bool converged = false, stop = false;
        while (it < P.max_iter && !stop) {
            ++it;
            init_rhs<NT, Sweep>(V, q0);
            flux_term<N, NT, Sweep>(W, U, var, P.khat, Xp);
            for (int r = 0; r < NVAR; ++r)
                for (int p0 = 0; p0 < NQ; p0 += S::CHUNK) {
                    const int np = min(S::CHUNK, NQ - p0);
                    const double* kr = var + 3 * PRIM_NNZ + r * SUBCELL_MODE;
                    for (int i = tid; i < np * BT; i += NT) {
                        const int p = i / BT, m = i - p * BT;
                        term[p * QS + m] = combine_row<QS>(p0 + p, W + m, U + m, kr);
                    }
                    __syncthreads();
                    mass_term<NT, Sweep, S::CHUNK>(V, term, p0, np, P.m3_row + r * (B + 1), P.m3_col, P.m3_val);
                }
            alg3_sweep<N, NT, BiotSystem, Sweep>(V, star, zuf, sc[1], P.khat, X);  // Q_{k+1}
            // max |Q_{k+1} - Q_k| and max |Q_{k+1}| over the element, as bit patterns:
            // the integer maximum of magnitudes is theirs, with NaN above infinity
            // (fmax would drop a NaN, and its comparisons run on the binary64 pipe)
            using Bits = unsigned long long;
            Bits dmax = 0, vmax = 0;
            for (int i = tid; i < NQ * BT; i += NT) {
                const int p = i / BT, m = i - p * BT;
                const double v = V[p * QS + m];
                dmax = max(dmax, (Bits)__double_as_longlong(fabs(v - U[p * QS + m])));
                vmax = max(vmax, (Bits)__double_as_longlong(fabs(v)));
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, s));
                vmax = max(vmax, __shfl_xor_sync(0xffffffffu, vmax, s));
            }
            if (lane == 0) {
                red[warp] = dmax;
                red[NW + warp] = vmax;
            }
            __syncthreads();
            dmax = vmax = 0;
            for (int w = 0; w < NW; ++w) {
                dmax = max(dmax, red[w]);
                vmax = max(vmax, red[NW + w]);
            }
            // a non-finite iterate stops the loop unconverged (and is written out as it is)
            const bool finite = max(dmax, vmax) < 0x7FF0000000000000ull;
            converged = finite && __longlong_as_double(dmax) <= P.tol * __longlong_as_double(vmax);
            stop = converged || !finite;
            double* t = U;
            U = V;
            V = t;
            __syncthreads();
        }
        const double dt = sc[2];
        double* io = P.iout ? P.iout + e * (int64_t)(NQ * B) : nullptr;
        double* qo = P.qt ? P.qt + e * (int64_t)(NQ * BT) : nullptr;
        if (io)
            for (int i = tid; i < NQ * B; i += NT) io[i] = dt * U[(i / B) * QS + (i % B) * T];
        if (qo)
            for (int i = tid; i < NQ * BT; i += NT) qo[i] = U[(i / BT) * QS + i % BT];
        if (tid == 0 && P.iters) P.iters[e] = converged ? it : -it;
        __syncthreads();
    }
}

template <int N, int NT_>
int launch_sub(const DeviceReference& ref, const SubcellReference& sub, int64_t count, const double* q0,
               const double* econst, const double* evar, double* qt, double* iout, int32_t* iters, double tol,
               int max_iter, void* stream) {
    using S = SubShape<N, NT_>;
    SubParams P;
    P.q0 = q0;
    P.econst = econst;
    P.evar = evar;
    P.qt = qt;
    P.iout = iout;
    P.iters = iters;
    P.count = count;
    P.stride = elem_const_stride(N);
    P.vstride = subcell_var_stride();
    P.khat = {reinterpret_cast<const int2*>(ref.sweep_ent), ref.sweep_list, ref.inv_d};
    P.m3_row = sub.m3_row;
    P.m3_col = sub.m3_col;
    P.m3_val = sub.m3_val;
    P.tol = tol;
    P.max_iter = max_iter;
    const size_t smem = S::SMEM_BYTES;
    cudaError_t err = cudaFuncSetAttribute(stp_subcell_kernel<N, NT_>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)smem);
    if (err != cudaSuccess) return (int)err;
    if (count <= 0) return 0;
    const int64_t grid = count < (int64_t)(1u << 30) ? count : (int64_t)(1u << 30);
    stp_subcell_kernel<N, NT_><<<(unsigned)grid, NT_, smem, (cudaStream_t)stream>>>(P);
    return (int)cudaGetLastError();
}

}  // namespace

int launch_stp_subcell(const DeviceReference& ref, const SubcellReference& sub, int64_t count, const double* q0,
                       const double* econst, const double* evar, double* qt, double* iout, int32_t* iters,
                       double tol, int max_iter, void* stream) {
    switch (ref.N) {
        case 1: return launch_sub<1, subcell_threads(1)>(ref, sub, count, q0, econst, evar, qt, iout, iters, tol, max_iter, stream);
        case 2: return launch_sub<2, subcell_threads(2)>(ref, sub, count, q0, econst, evar, qt, iout, iters, tol, max_iter, stream);
        case 3: return launch_sub<3, subcell_threads(3)>(ref, sub, count, q0, econst, evar, qt, iout, iters, tol, max_iter, stream);
        case 4: return launch_sub<4, subcell_threads(4)>(ref, sub, count, q0, econst, evar, qt, iout, iters, tol, max_iter, stream);
        case 5: return launch_sub<5, subcell_threads(5)>(ref, sub, count, q0, econst, evar, qt, iout, iters, tol, max_iter, stream);
        case 6: return launch_sub<6, subcell_threads(6)>(ref, sub, count, q0, econst, evar, qt, iout, iters, tol, max_iter, stream);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace poro
