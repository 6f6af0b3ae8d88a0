// The viscoelastic space-time predictor (3 relaxation mechanisms, 27 quantities), one
// element per CTA, in IEEE binary64, by the degree-block back-substitution of the
// paper (Section "Block-wise back-substitution", Algorithm 3; Section "Other
// applications").
//
// As Biot's kernel (stp_direct.cu) it works on primitive rows: with n^j = -dt grad
// xi_j, the star products of all 27 quantities are combinations of 9,
//   0..2 n_d v_d   3..5 shear n_b v_a + n_a v_b   6..8 S = sigma n,
// because every mechanism's anelastic functions follow the same strain rate.
// Khat acts on the 9 rows as exact integer sums (fixed_device.cuh), and the moduli
// combine the sums once per mode, when its block is solved.  Only stresses and
// velocities feed the star products, so shared memory holds 9 rows a mode: the
// primitive sums until the mode is solved, its stresses and velocities
// afterwards; the anelastic functions go from registers to the output.
//
// A warp solves T lanes (u) of 32 / T modes' normal stresses with their 9 anelastic
// functions, or of 32 / T pairs of a mode and a shear stress with its 3 and one
// velocity; at N <= 2, where blocks have few modes, a mode's normal stresses are three
// groups of lanes (8,000 elements at N = 1: 142 microseconds undivided, 89 so; with
// each shear stress a task of its own besides 196, and 357 instead of 284, now 215,
// at N = 2).  b = S^{-1}w q0 -
// combinations; th with (Z - e_l I)^{-1} (dense), then the couplings of E*'s strictly
// upper part into the stresses, which like the velocities take the tridiagonal
// Z^{-1}.
//
// What bounds it: the binary64 pipe, 94 thousand operations an element at N = 5, over
// half of them the dense solves of the anelastic functions; with star products and
// Khat on all 27 rows they were 128 thousand, and the integer sums three times as
// many.  4,001 elements at N = 5: 1.03 ms, the pipe 83 % busy (1.13 with a task per shear
// stress, 81 %; 2.22 on 27 rows, 4.01 with the Khat products in binary64).
#include <cuda_runtime.h>

#include "fixed_device.cuh"
#include "poro_internal.h"

namespace poro {
namespace {

using visco::NMECH;
constexpr int NP = 9;  // primitive rows

struct ViscoParams {
    const double* q0;
    const double* econst;
    double* qt;
    double* iout;
    const int2* ent;
    const int32_t* list;
    const double* inv_d;
};

template <int N>
struct ViscoShape {
    static constexpr int NT = visco::threads(N), NW = NT / 32;
    static constexpr int B = n_modes(N), T = N + 1, PT = NP * T, PUL = (PT + 31) / 32, G = 32 / T;
    static constexpr int XC = visco::columns(N);
    // normal stresses: a group of lanes per component where a warp holds three groups
    // for several modes with few left over; modes a warp takes
    static constexpr bool SPLIT = N <= 2;
    static constexpr int GN = SPLIT ? G / 3 : G;
    // constants from the time matrices on: Zs[NMECH][T][T], scalars, iso[16]
    static constexpr int EC0 = 3 * visco::STAR_NNZ, EC = visco::elem_const_stride(N) - EC0;
    static constexpr int SC = NMECH * T * T, ISO = visco::ec_iso(N) - EC0;
    // shared layout in 8-byte words
    static constexpr int OFF_X = B * PT, OFF_K = OFF_X + XC * PT + 32, OFF_N = OFF_K + EC, OFF_I = OFF_N + 4;
    static constexpr int I_WORDS = (3 * PT + 1) & ~1;  // max |Q| of two blocks, row scales
    static constexpr int SMEM_BYTES = 8 * OFF_I + 4 * I_WORDS;
    static constexpr int MIN_BLOCKS = N == 6 ? 3 : N == 5 ? 4 : N == 4 ? 5 : 8;
};

template <int N>
__global__ void __launch_bounds__(ViscoShape<N>::NT, ViscoShape<N>::MIN_BLOCKS) stp_visco_kernel(const ViscoParams A) {
    using S = ViscoShape<N>;
    constexpr int NQ = visco::NQ, B = S::B, T = S::T, PT = S::PT, PUL = S::PUL, NT = S::NT, NW = S::NW, G = S::G;
    extern __shared__ double sm[];
    double* C = sm;
    int2* X = reinterpret_cast<int2*>(sm + S::OFF_X);
    double* K = sm + S::OFF_K;
    const double* sc = K + S::SC;
    const double* iso = K + S::ISO;  // n[3][3], lambda, 2 mu, mu, 1 / rho, omega[3]
    double* nmax = sm + S::OFF_N;
    uint32_t* qmax = reinterpret_cast<uint32_t*>(sm + S::OFF_I);
    int* scale = reinterpret_cast<int*>(qmax) + 2 * PT;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int64_t e = blockIdx.x;
    const double* q0 = A.q0 + e * (int64_t)(NQ * B);
    for (int i = tid; i <= NQ * B / 16; i += NT)
        asm volatile("prefetch.global.L1 [%0];" ::"l"(q0 + min(16 * i, NQ * B - 1)));
    const double* ec = A.econst + e * (int64_t)visco::elem_const_stride(N) + S::EC0;
    for (int i = tid; i < S::EC; i += NT) K[i] = ec[i];
    for (int i = tid; i < B * PT; i += NT) C[i] = 0.0;
    for (int i = tid; i < 2 * PT; i += NT) qmax[i] = 0u;
    __syncthreads();
    if (tid < 3) nmax[tid] = fmax(fabs(iso[tid]), fmax(fabs(iso[3 + tid]), fabs(iso[6 + tid])));
    const int grp = lane / T, u = lane - grp * T, base = grp * T;
    const double sw = (double)((2 * u + 1) * ((u & 1) ? -1 : 1));
    // row u of Z^{-1} (tridiagonal): on u - 1 (u = 0: on itself) and on u + 1 (the last: on itself)
    double z_lo = 0.5, z_hi = 0.0;
#pragma unroll
    for (int s = 0; s < T; ++s)
        if (u == s) {
            z_lo = s == 0 ? 0.5 : 0.5 / (2 * s - 1);
            z_hi = s == T - 1 ? 0.5 / (2 * s + 1) : -0.5 / (2 * s + 3);
        }
    const double dt = sc[visco::sc_dt()];
    double* qo = A.qt ? A.qt + e * (int64_t)(NQ * B * T) : nullptr;
    double* io = A.iout ? A.iout + e * (int64_t)(NQ * B) : nullptr;
    const int32_t* list = A.list;
    int buf = 0;
#pragma unroll 1
    for (int g = N; g >= 0; --g) {
        const int o = block_offset(g), d = block_size(g);
        // ---- time solves of block g
#pragma unroll 1
        for (int t = warp, nn = (d + S::GN - 1) / S::GN; t < nn + (3 * d + G - 1) / G; t += NW) {
            // GN modes' normal stresses (SPLIT: three groups of lanes a mode, one for
            // component i), or G (shear component i, mode) pairs
            const bool normal = t < nn;
            const int per = normal && S::SPLIT ? 3 : 1, first = normal ? t * S::GN * per : (t - nn) * G;
            const int count = normal ? min(d * per, first + S::GN * per) : 3 * d;
            const bool act = grp < G && first + grp < count;
            const int item = min(first + min(grp, G - 1), count - 1);
            const int i = normal ? (S::SPLIT ? item % 3 : 0) : item / d, m = o + (normal ? item / per : item - i * d);
            double* c = C + m * PT + u;
            auto rhs = [&](int q, double a) { return fma(sw, q0[q * B + m], a); };  // S^{-1}w q0 + a
            auto plain = [&](double b) {
                const double lo = __shfl_sync(0xffffffffu, b, lane - 1), hi = __shfl_sync(0xffffffffu, b, lane + 1);
                return fma(z_hi, u == T - 1 ? b : hi, z_lo * (u == 0 ? b : lo));
            };
            auto out = [&](int q, double x) {
                if (!act) return;
                if (qo) qo[(q * B + m) * T + u] = x;
                if (io && u == 0) io[q * B + m] = dt * x;
            };
            auto keep = [&](int q, double x) {  // a stress or velocity
                out(q, x);
                if (!act) return;
                c[q * T] = x;
                atomicMax(qmax + buf * PT + q * T + u, (uint32_t)__double2hiint(x) & 0x7FFFFFFFu);
            };
            // anelastic function k of mechanism l from its strain-rate sum s
            auto anelastic = [&](int l, int k, double s) {
                const int q = 9 + 6 * l + k;
                const double b = rhs(q, -iso[13 + l] * s);
                const double* Z = K + l * T * T + u * T;
                double x0 = Z[0] * __shfl_sync(0xffffffffu, b, base), x1 = 0.0;
#pragma unroll
                for (int i = 1; i < T; ++i) {
                    const double bi = __shfl_sync(0xffffffffu, b, base + i);
                    if (i & 1) x1 = fma(Z[i], bi, x1);
                    else x0 = fma(Z[i], bi, x0);
                }
                const double x = x0 + x1;
                out(q, x);
                return x;
            };
            if (S::SPLIT && normal) {
                const double g0 = c[0], g1 = c[T], g2 = c[2 * T], gi = i == 0 ? g0 : i == 1 ? g1 : g2;
                double b = rhs(i, fma(-iso[10], gi, -iso[9] * ((g0 + g1) + g2)));
                const int lane0 = lane - i * T;  // this u in component 0's group
#pragma unroll 1
                for (int l = 0; l < NMECH; ++l) {
                    const double th = anelastic(l, i, gi);
                    const double t0 = __shfl_sync(0xffffffffu, th, lane0), t1 = __shfl_sync(0xffffffffu, th, lane0 + T),
                                 t2 = __shfl_sync(0xffffffffu, th, lane0 + 2 * T);
                    // (Ylam + 2 Ymu) on the own component, Ylam on the other two
                    const double off = sc[3 * l + 1], own = sc[3 * l] - off;
                    b += fma(own, th, off * ((t0 + t1) + t2));
                }
                keep(i, plain(b));
            } else if (normal) {
                const double gd[3] = {c[0], c[T], c[2 * T]};
                const double Lm = -iso[9] * ((gd[0] + gd[1]) + gd[2]);
                double b[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) b[k] = rhs(k, fma(-iso[10], gd[k], Lm));
#pragma unroll 1
                for (int l = 0; l < NMECH; ++l) {
                    double th[3];
#pragma unroll
                    for (int k = 0; k < 3; ++k) th[k] = anelastic(l, k, gd[k]);
                    const double off = sc[3 * l + 1], own = sc[3 * l] - off, s = off * ((th[0] + th[1]) + th[2]);
#pragma unroll
                    for (int k = 0; k < 3; ++k) b[k] += fma(own, th[k], s);
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) keep(k, plain(b[k]));
            } else {
                const double s = c[(3 + i) * T];
                double b = rhs(3 + i, -iso[11] * s);
#pragma unroll 1
                for (int l = 0; l < NMECH; ++l) b = fma(sc[3 * l + 2], anelastic(l, 3 + i, 0.5 * s), b);
                const double v = plain(rhs(6 + i, -iso[12] * c[(6 + i) * T]));
                keep(3 + i, plain(b));
                keep(6 + i, v);
            }
        }
        __syncthreads();
        if (g == 0) break;
        // ---- scale of every row (k, u) of X
        for (int r = tid; r < PT; r += NT) {
            const int k = r / T, uu = r - k * T;
            const uint32_t* qm = qmax + buf * PT + uu;
            auto term = [&](int dd, int q) { return nmax[dd] * bound_of(qm[q * T], 0.0); };
            double b;
            if (k < 3) b = term(k, 6 + k);
            else if (k < 6) b = k == 3 ? term(1, 6) + term(0, 7) : k == 4 ? term(2, 7) + term(1, 8) : term(2, 6) + term(0, 8);
            else b = term(0, k == 6 ? 0 : k == 7 ? 3 : 5) + term(1, k == 6 ? 3 : k == 7 ? 1 : 4) + term(2, k == 6 ? 5 : k == 7 ? 4 : 2);
            scale[r] = row_scale(b);
            qmax[(buf ^ 1) * PT + r] = 0u;
        }
        buf ^= 1;
        __syncthreads();
        const int dm = pass_modes(g, S::XC);
#pragma unroll 1
        for (int m0 = 0; m0 < d; m0 += dm) {
            const int nm = min(dm, d - m0);
            // ---- primitives of modes o + m0 .., quantised: column j * dm + ml
            for (int it = tid; it < 3 * nm * T; it += NT) {
                const int j = it / (nm * T), r = it - j * (nm * T), ml = r / T, uu = r - ml * T;
                const double* q = C + (o + m0 + ml) * PT + uu;
                int2* x = X + (j * dm + ml) * PT + uu;
                const int* s = scale + uu;
                const double nx = iso[3 * j], ny = iso[3 * j + 1], nz = iso[3 * j + 2];
                auto put = [&](int k, double v) { x[k * T] = quantise(v, s[k * T]); };
                const double v0 = q[6 * T], v1 = q[7 * T], v2 = q[8 * T];
                put(0, nx * v0);
                put(1, ny * v1);
                put(2, nz * v2);
                put(3, fma(ny, v0, nx * v1));
                put(4, fma(nz, v1, ny * v2));
                put(5, fma(nz, v0, nx * v2));
                const double xx = q[0], yy = q[T], zz = q[2 * T], xy = q[3 * T], yz = q[4 * T], xz = q[5 * T];
                put(6, fma(nz, xz, fma(ny, xy, nx * xx)));
                put(7, fma(nz, yz, fma(ny, yy, nx * xy)));
                put(8, fma(nz, zz, fma(ny, yz, nx * xz)));
            }
            __syncthreads();
            // ---- C[l] += Khat X over the pass's columns; this warp's rows
            const int i1 = __ldg(list + warp + 1);
            const int32_t* rows = list + NW + 1;
#pragma unroll 1
            for (int i = __ldg(list + warp); i < i1; ++i) {
                const int w = __ldg(rows + i), l = w >> 21, n0 = w & 8191, n1 = n0 + ((w >> 13) & 255);
                const int2* xl = X + lane;
                long long hi[PUL], lo[PUL];
#pragma unroll
                for (int k = 0; k < PUL; ++k) hi[k] = lo[k] = 0;
#pragma unroll 4
                for (int n = n0; n < n1; ++n) {
                    const int2 en = __ldg(A.ent + n);
                    const int2* xc = xl + en.x;
#pragma unroll
                    for (int k = 0; k < PUL; ++k) fixed_mac(en.y, xc[32 * k], hi[k], lo[k]);
                }
                const double inv = __ldg(A.inv_d + l);
#pragma unroll
                for (int k = 0; k < PUL; ++k) {
                    const int r = lane + 32 * k;
                    if (r < PT) C[l * PT + r] = fma(fixed_sum(hi[k], lo[k], scale[r]), inv, C[l * PT + r]);
                }
            }
            list = rows + __ldg(list + NW);
            __syncthreads();
        }
    }
}

template <int N>
int launch_n(const DeviceReference& ref, int64_t count, const double* q0, const double* econst, double* qt, double* iout,
             void* stream) {
    using S = ViscoShape<N>;
    const ViscoParams A{q0, econst, qt, iout, reinterpret_cast<const int2*>(ref.sweep_ent), ref.sweep_list, ref.inv_d};
    const cudaError_t err =
        cudaFuncSetAttribute(stp_visco_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM_BYTES);
    if (err != cudaSuccess) return (int)err;
    stp_visco_kernel<N><<<(unsigned)count, S::NT, S::SMEM_BYTES, (cudaStream_t)stream>>>(A);
    return (int)cudaGetLastError();
}

}  // namespace

int launch_stp_fp64_visco(const DeviceReference& ref, int64_t count, const double* q0, const double* econst, double* qt,
                          double* iout, void* stream) {
    if (count <= 0) return 0;
    switch (ref.N) {
        case 1: return launch_n<1>(ref, count, q0, econst, qt, iout, stream);
        case 2: return launch_n<2>(ref, count, q0, econst, qt, iout, stream);
        case 3: return launch_n<3>(ref, count, q0, econst, qt, iout, stream);
        case 4: return launch_n<4>(ref, count, q0, econst, qt, iout, stream);
        case 5: return launch_n<5>(ref, count, q0, econst, qt, iout, stream);
        case 6: return launch_n<6>(ref, count, q0, econst, qt, iout, stream);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace poro
