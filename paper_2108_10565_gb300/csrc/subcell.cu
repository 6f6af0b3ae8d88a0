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
// Shared memory: U (iterate), V (right-hand side, then the next iterate) and W
// (one variation term) in the b / Q layout of the sweep, its fixed-point X (the
// Khat products are integer sums, in the sweep and in the variation terms), the
// mean element constants, the variation stars and the reduction words.
#include <cuda_runtime.h>

#include "alg3_device.cuh"

namespace poro {
namespace {

struct SubParams {
    const double* q0;
    const double* econst;  // mean-material constants (the layout of the FP64 predictor)
    const double* evar;    // per element: star_r[3][3][54] for r = 1..3, then (e_r, g_r) for r = 1..3
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

template <int N, int NT_>
struct SubShape : SweepShape<N, BiotSystem, subcell_columns(N)> {
    using S = SweepShape<N, BiotSystem, subcell_columns(N)>;
    static constexpr int NT = NT_, NW = NT_ / 32;
    static constexpr int OFF_V = S::SQ;
    static constexpr int OFF_W = 2 * S::SQ;
    static constexpr int OFF_X = 3 * S::SQ;
    static constexpr int OFF_STAR = OFF_X + S::X_WORDS;            // mean constants: star, zuf, sc (EC words)
    static constexpr int EC = 3 * STAR_NNZ + S::T * S::T + 4;
    static constexpr int OFF_VAR = OFF_STAR + EC;                   // variation stars and (e_r, g_r)
    static constexpr int VAR = NVAR * 3 * STAR_NNZ + 2 * NVAR;
    static constexpr int OFF_MAX = OFF_VAR + VAR;                   // max_j |star| of the mean, of the variations
    static constexpr int OFF_RED = OFF_MAX + (1 + NVAR) * STAR_NNZ; // 2 NW reduction words
    static constexpr int OFF_I = OFF_RED + 2 * NW;
    static constexpr int SMEM_BYTES = 8 * OFF_I + 4 * S::I_WORDS;
};

// W <- -E*_r U (source variation): u_f rows e_r U_uf, u rows g_r U_uf
template <int NT, class S>
__device__ void source_term(double* W, const double* U, double e, double g) {
    constexpr int QS = S::QS, BT = S::B * S::T;
    for (int i = threadIdx.x; i < NQ * BT; i += NT) {
        const int p = i / BT, m = i - p * BT;
        double v = 0.0;
        if (p >= QUF) v = -e * U[p * QS + m];
        else if (p >= QU && p <= QW) v = -g * U[(p + QUF - QU) * QS + m];
        W[p * QS + m] = v;
    }
}

// W += sum_j Khat^j (A^{j*}_r U) over all degree blocks (strictly upper in
// degree: rows l < o_g take column block g); begins after and ends with a barrier
template <int N, int NT, class S>
__device__ void flux_term(double* W, const double* U, const double* starr, const KhatRows& K, const SweepScratch<S>& X) {
    constexpr int T = S::T;
    const int32_t* list = K.list;
#pragma unroll 1
    for (int g = N; g >= 1; --g) {
        const int o = block_offset(g), d = block_size(g);
        for (int it = threadIdx.x; it < NQ * d * T; it += NT) {
            const int q = it / (d * T), mu = it - q * (d * T);
            atomicMax(X.qmax(0) + q * T + mu % T, (uint32_t)__double2hiint(U[q * S::QS + o * T + mu]) & 0x7FFFFFFFu);
        }
        __syncthreads();
        khat_block<N, NT, BiotSystem, S, 1>(W, U, g, starr, K, list, X, X.qmax(0), X.qmax(1));
        for (int i = threadIdx.x; i < S::PT; i += NT) X.qmax(0)[i] = 0u;
        __syncthreads();
    }
}

// V -= Mh3_r W (all rows k); ends with a barrier
template <int NT, class S>
__device__ void mass_term(double* V, const double* W, const int32_t* row, const int32_t* col, const double* val) {
    constexpr int B = S::B, T = S::T, QS = S::QS, PT = S::PT, PUL = S::PUL, NW = NT / 32;
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
                if (pu < PT) acc[q] = fma(v, W[(pu / T) * QS + l + pu % T], acc[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < PUL; ++q) {
            const int pu = lane + 32 * q;
            if (pu < PT) V[(pu / T) * QS + k * T + pu % T] -= acc[q];
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
    double* red = sm + S::OFF_RED;
    using Sweep = typename S::S;
    const SweepScratch<Sweep> X{reinterpret_cast<int2*>(sm + S::OFF_X), reinterpret_cast<int*>(sm + S::OFF_I), smax};
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
        for (int r = 0; r < NVAR; ++r)
            adapt_star<NT, STAR_NNZ>(var + r * 3 * STAR_NNZ, smax + (1 + r) * STAR_NNZ);
        __syncthreads();
        alg3_sweep<N, NT, BiotSystem, Sweep>(U, star, zuf, sc[1], P.khat, X);  // Q_0 = Y_0^{-1} b0
        int it = 0;
        bool converged = false, stop = false;
        while (it < P.max_iter && !stop) {
            ++it;
            init_rhs<NT, Sweep>(V, q0);
            for (int r = 0; r < NVAR; ++r) {
                source_term<NT, Sweep>(W, U, var[NVAR * 3 * STAR_NNZ + 2 * r], var[NVAR * 3 * STAR_NNZ + 2 * r + 1]);
                __syncthreads();
                SweepScratch<Sweep> Xr = X;
                Xr.smax = smax + (1 + r) * STAR_NNZ;
                flux_term<N, NT, Sweep>(W, U, var + r * 3 * STAR_NNZ, P.khat, Xr);
                mass_term<NT, Sweep>(V, W, P.m3_row + r * (B + 1), P.m3_col, P.m3_val);
            }
            alg3_sweep<N, NT, BiotSystem, Sweep>(V, star, zuf, sc[1], P.khat, X);  // Q_{k+1}
            // max |Q_{k+1} - Q_k| and max |Q_{k+1}| over the element
            double dmax = 0.0, vmax = 0.0;
            for (int i = tid; i < NQ * BT; i += NT) {
                const int p = i / BT, m = i - p * BT;
                const double v = V[p * QS + m];
                dmax = fmax(dmax, fabs(v - U[p * QS + m]));
                vmax = fmax(vmax, fabs(v));
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, s));
                vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, s));
            }
            if (lane == 0) {
                red[warp] = dmax;
                red[NW + warp] = vmax;
            }
            __syncthreads();
            dmax = 0.0;
            vmax = 0.0;
            for (int w = 0; w < NW; ++w) {
                dmax = fmax(dmax, red[w]);
                vmax = fmax(vmax, red[NW + w]);
            }
            // a non-finite iterate stops the loop unconverged (and is written out as it is)
            const bool finite = isfinite(dmax) && isfinite(vmax);
            converged = finite && dmax <= P.tol * vmax;
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
