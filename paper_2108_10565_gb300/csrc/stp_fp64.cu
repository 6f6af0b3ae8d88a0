// The space-time predictor of one element per CTA, in IEEE binary64, by the
// degree-block back-substitution of the paper (Section "Block-wise
// back-substitution", Algorithm 3), for the damped Maxwell system (Biot's
// kernel is in stp_direct.cu, the viscoelastic one in stp_visco.cu).
//
// Per element the CTA keeps b (quantities x B x T) in shared memory and overwrites
// it in place with the predictor Qt: once the modes of degree block g are solved,
// their b entries are dead.  For g = N .. 0:
//   S3  time solves: Q[p,m,:] = Zinv_p b[p,m,:] for the modes m of block g,
//       Zinv_p = (Z - E*_pp I)^{-1} (tridiagonal where E*_pp = 0), after the
//       couplings of E*'s strictly upper part
//   S4  green update (g > 0): X^j[p,m,u] = sum_q A^{j*}_pq Q[q,m,u] (the system's
//       star pattern), b[p,l,u] -= sum_j sum_m Khat^j_lm X^j[p,m,u], l < o_g, in
//       exact integers (fixed_device.cuh)
// then the time integration I = dt Qt[:, :, 0] (int_0^1 chi_s = delta_s0).
//
// What bounds it: the binary64 pipe (2 lanes a clock and SM) carries the star
// products and time solves, the integer pipes the Khat products, which were 60 to
// 75 % of the binary64 operations.  20,000 elements at N = 4: 0.65 ms, the binary64
// pipe 85 % busy (1.59 ms with the Khat products on it).
#include <cuda_runtime.h>

#include "alg3_device.cuh"

namespace poro {
namespace {

struct SweepParams {
    const double* q0;
    const double* econst;
    double* qt;
    double* iout;
    int stride;
    KhatRows khat;
};

template <int N, class Sys, int XC>
struct Shape : SweepShape<N, Sys, XC> {
    using S = SweepShape<N, Sys, XC>;
    // shared layout (8-byte words): bq | X | star[3 NNZ] | zsh[NSHM T T] |
    // sc[NSC] | smax[NNZ] | scratch; star .. sc are the element's constants in
    // their global order (EC words)
    static constexpr int OFF_X = S::SQ, OFF_STAR = OFF_X + S::X_WORDS;
    static constexpr int OFF_ZSH = OFF_STAR + 3 * Sys::NNZ, OFF_SC = OFF_ZSH + Sys::NSHM * S::T * S::T;
    static constexpr int EC = OFF_SC + Sys::NSC - OFF_STAR;
    static constexpr int OFF_MAX = OFF_SC + Sys::NSC, OFF_I = OFF_MAX + Sys::NNZ;
    static constexpr int SMEM_BYTES = 8 * OFF_I + 4 * S::I_WORDS;
};

template <int N, int NT, class Sys, int XC>
__global__ void __launch_bounds__(NT) stp_fp64_kernel(const SweepParams P) {
    using S = Shape<N, Sys, XC>;
    constexpr int NQ = Sys::NQ, B = S::B, T = S::T, QS = S::QS;
    extern __shared__ double sm[];
    double* bq = sm;
    double* star = sm + S::OFF_STAR;
    double* sc = sm + S::OFF_SC;
    double* smax = sm + S::OFF_MAX;
    int* ints = reinterpret_cast<int*>(sm + S::OFF_I);
    const SweepScratch<S> W{reinterpret_cast<int2*>(sm + S::OFF_X), ints, smax, ints + S::I_ROW};
    const int tid = threadIdx.x;
    const int64_t e = blockIdx.x;
    // element constants: stars, shifted time matrices and scalars are contiguous
    const double* ec = P.econst + e * (int64_t)P.stride;
    for (int i = tid; i < S::EC; i += NT) star[i] = ec[i];
    init_rhs<NT, S>(bq, P.q0 + e * (int64_t)(NQ * B));
    __syncthreads();
    sweep_setup<NT, S, Sys>(W, smax, star);
    __syncthreads();
    alg3_sweep<N, NT, Sys, S>(bq, star, sm + S::OFF_ZSH, sc[1], P.khat, W);
    // time integration and outputs (global layout [p][l][u], dense)
    const double dt = sc[Sys::DT_SC];
    if (P.iout) {
        double* io = P.iout + e * (int64_t)(NQ * B);
        for (int i = tid; i < NQ * B; i += NT) io[i] = dt * bq[(i / B) * QS + (i % B) * T];
    }
    if (P.qt) {
        double* qo = P.qt + e * (int64_t)(NQ * B * T);
        for (int i = tid; i < NQ * B * T; i += NT) qo[i] = bq[(i / (B * T)) * QS + i % (B * T)];
    }
}

template <int N, int NT, class Sys, int XC>
int launch_nt(const DeviceReference& ref, int stride, int64_t count, const double* q0, const double* econst, double* qt,
              double* iout, void* stream) {
    using S = Shape<N, Sys, XC>;
    if (count <= 0) return 0;
    const SweepParams P{q0, econst, qt, iout, stride,
                        {reinterpret_cast<const int2*>(ref.sweep_ent), ref.sweep_list, ref.inv_d}};
    auto* kern = stp_fp64_kernel<N, NT, Sys, XC>;
    const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM_BYTES);
    if (err != cudaSuccess) return (int)err;
    kern<<<(unsigned)count, NT, S::SMEM_BYTES, (cudaStream_t)stream>>>(P);
    return (int)cudaGetLastError();
}

template <int N>
int launch_maxwell(const DeviceReference& ref, int64_t count, const double* q0, const double* econst, double* qt,
                   double* iout, void* stream) {
    return launch_nt<N, maxwell::threads(N), MaxwellSystem, maxwell::columns(N)>(ref, maxwell::elem_const_stride(N), count,
                                                                                 q0, econst, qt, iout, stream);
}

}  // namespace

int launch_stp_fp64_maxwell(const DeviceReference& ref, int64_t count, const double* q0, const double* econst,
                            double* qt, double* iout, void* stream) {
    switch (ref.N) {
        case 1: return launch_maxwell<1>(ref, count, q0, econst, qt, iout, stream);
        case 2: return launch_maxwell<2>(ref, count, q0, econst, qt, iout, stream);
        case 3: return launch_maxwell<3>(ref, count, q0, econst, qt, iout, stream);
        case 4: return launch_maxwell<4>(ref, count, q0, econst, qt, iout, stream);
        case 5: return launch_maxwell<5>(ref, count, q0, econst, qt, iout, stream);
        case 6: return launch_maxwell<6>(ref, count, q0, econst, qt, iout, stream);
        default: return (int)cudaErrorInvalidValue;
    }
}

int launch_stp_fp64(const DeviceReference& ref, const int32_t* elems, int64_t count, const double* q0,
                    const double* econst, double* qt, double* iout, double* qend, void* stream, int variant,
                    const RunPtrs* runs, const int32_t* item_run) {
    return launch_stp_direct(ref, false, false, nullptr, 0, elems, count, q0, econst, qt, iout, qend, stream, variant,
                             runs, item_run);
}

}  // namespace poro
