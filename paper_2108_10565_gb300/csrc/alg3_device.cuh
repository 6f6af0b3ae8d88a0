// Device building blocks of the degree-block back-substitution (Section
// "Block-wise back-substitution", Algorithm 3): the binary64 sweep of
// the Maxwell system and of the sub-cell iteration, and the layout that
// the binary32 sweep of stp_mixed.cu shares.
//
// Shared-memory layout of one element's b / Q tensor: quantity p at offset
// p * QS, mode l at l * T, time mode u at u, where the quantity stride QS is
// B * T padded so that the T lanes (p, u) of neighbouring quantities fall on
// consecutive banks: QS = T (mod 32) in 4-byte, (mod 16) in 8-byte words.
#pragma once

#include <cuda_runtime.h>

#include "fixed_device.cuh"
#include "poro_internal.h"

namespace poro {

__host__ __device__ constexpr int bank_stride(int n, int T) { return n + ((T - n % 32) + 32) % 32; }

// row <- Z^{-1} row, tridiagonal: row u is 1 / (2 (2u - 1)) on u - 1 (u = 0: 1/2
// on itself) and -1 / (2 (2u + 3)) on u + 1 (the last: 1 / (2 (2u + 1)) on
// itself); the high words of the result go to qmax[u] (a maximum)
template <int T>
__device__ __forceinline__ void solve_plain(double* row, uint32_t* qmax) {
    double x[T];
#pragma unroll
    for (int s = 0; s < T; ++s) x[s] = row[s];
#pragma unroll
    for (int u = 0; u < T; ++u) {
        const double lo = u == 0 ? 0.5 : 0.5 / (2 * u - 1), hi = u == T - 1 ? 0.5 / (2 * u + 1) : -0.5 / (2 * u + 3);
        const double y = fma(hi, x[u == T - 1 ? u : u + 1], lo * x[u == 0 ? 0 : u - 1]);
        row[u] = y;
        atomicMax(qmax + u, (uint32_t)__double2hiint(y) & 0x7FFFFFFFu);
    }
}
// row <- Zi row, dense
template <int T>
__device__ __forceinline__ void solve_row(double* row, const double* Zi, uint32_t* qmax) {
    double x[T];
#pragma unroll
    for (int s = 0; s < T; ++s) x[s] = row[s];
#pragma unroll
    for (int u = 0; u < T; ++u) {
        double y = 0.0;
#pragma unroll
        for (int s = 0; s < T; ++s) y = fma(Zi[u * T + s], x[s], y);
        row[u] = y;
        atomicMax(qmax + u, (uint32_t)__double2hiint(y) & 0x7FFFFFFFu);
    }
}

// The linear system of the predictor: its quantities, the union pattern of
// its reference Jacobians and the structure of its source matrix E (upper
// triangular, Section "Block-wise back-substitution"): per mode the time
// solves are NPLAIN rows with Z^{-1} (E_pp = 0), NSHIFT rows with
// (Z - e I)^{-1} and no coupling, and NPAIR pairs: src solved with
// (Z - e I)^{-1}, then b_dst += g Q_src, then dst with Z^{-1}.
// Per-element constants (in this order): star[3][NNZ], NSHM shifted time
// matrices (Z - e I)^{-1}, NSC scalars with dt at DT_SC.
struct BiotSystem {  // Biot's equations: G couples u_f -> u, v_f -> v, w_f -> w
    static constexpr int NQ = poro::NQ, NNZ = STAR_NNZ, NPLAIN = 7, NSHIFT = 0, NPAIR = 3;
    static constexpr int NSHM = 1, NSC = 4, DT_SC = 2;
    PORO_HD static constexpr int row(int n) { return star_row(n); }
    PORO_HD static constexpr int col(int n) { return star_col(n); }
    PORO_HD static constexpr int plain(int k) { return k < 6 ? k : QP; }
    PORO_HD static constexpr int shifted(int) { return 0; }
    PORO_HD static constexpr int pair_src(int i) { return QUF + i; }
    PORO_HD static constexpr int pair_dst(int i) { return QU + i; }
};
struct MaxwellSystem {  // damped Maxwell: E diagonal, -sigma/eps on the electric rows
    static constexpr int NQ = maxwell::NQ, NNZ = maxwell::STAR_NNZ, NPLAIN = 3, NSHIFT = 3, NPAIR = 0;
    static constexpr int NSHM = 1, NSC = 4, DT_SC = 2;
    PORO_HD static constexpr int row(int n) { return maxwell::star_row(n); }
    PORO_HD static constexpr int col(int n) { return maxwell::star_col(n); }
    PORO_HD static constexpr int plain(int k) { return 3 + k; }
    PORO_HD static constexpr int shifted(int k) { return k; }
    PORO_HD static constexpr int pair_src(int) { return 0; }
    PORO_HD static constexpr int pair_dst(int) { return 0; }
};
template <int N, int NQ_ = NQ>
struct Alg3Shape {
    static constexpr int B = n_modes(N);
    static constexpr int T = N + 1;
    static constexpr int QBT = NQ_ * B * T;                // dense size (global layout)
    static constexpr int QS = bank_stride(B * T, T);       // shared quantity stride
    static constexpr int SQ = NQ_ * QS;                    // shared size of b / Q
    static constexpr int PT = NQ_ * T;                     // (p, u) pairs of one mode
    static constexpr int PUL = (PT + 31) / 32;             // pairs per lane
};

// The binary64 sweep's layout: quantity stride for 8-byte words, and the
// integer X with room for XC columns (direction, mode) of PT rows (p, u)
template <int N, class Sys, int XC_>
struct SweepShape {
    static constexpr int NQ = Sys::NQ, B = n_modes(N), T = N + 1, XC = XC_;
    static constexpr int QS = B * T + ((T - B * T % 16) + 16) % 16, SQ = NQ * QS;
    static constexpr int PT = NQ * T, PUL = (PT + 31) / 32;
    static constexpr int X_WORDS = XC * PT + 32;      // 8-byte words (slack read by idle lanes)
    // scratch in 32-bit words: max |Q| of two blocks, row scales, row starts of the star pattern
    static constexpr int I_SCALE = 2 * PT, I_ROW = 3 * PT, I_WORDS = (3 * PT + NQ + 1 + 1) & ~1;
};

// Integer Khat rows (khat_tables with stride PT and this kernel's XC and warps)
struct KhatRows {
    const int2* ent;
    const int32_t* list;
    const double* inv_d;
};

// Scratch of the sweep in shared memory
template <class S>
struct SweepScratch {
    int2* X;
    int* w;              // I_WORDS
    const double* smax;  // [NNZ] max_j |star_j|
    int* row;            // [NQ + 1] row starts of the star pattern
    __device__ uint32_t* qmax(int buf) const { return reinterpret_cast<uint32_t*>(w) + buf * S::PT; }
    __device__ int* scale() const { return w + S::I_SCALE; }
};
// star[3][NNZ] into the directions of the integer Khat rows, and smax; entries
// are a thread's own, so no barrier is needed inside
template <int NT, int NNZ>
__device__ void adapt_star(double* star, double* smax) {
    for (int i = threadIdx.x; i < NNZ; i += NT) {
        double s0 = star[i], s1 = star[NNZ + i];
        const double s2 = star[2 * NNZ + i];
        adapted_directions(s0, s1, s2);
        star[i] = s0;
        star[NNZ + i] = s1;
        smax[i] = fmax(fabs(s0), fmax(fabs(s1), fabs(s2)));
    }
}
// fills the row starts and adapts the star (loaded before the caller's last
// barrier); the caller's barrier follows
template <int NT, class Sys>
__device__ void star_setup(int* row, double* smax, double* star) {
    for (int i = threadIdx.x; i <= Sys::NQ; i += NT) {
        int n = 0;
        while (n < Sys::NNZ && Sys::row(n) < i) ++n;
        row[i] = n;
    }
    adapt_star<NT, Sys::NNZ>(star, smax);
}
// the same, and clears the maxima
template <int NT, class S, class Sys>
__device__ void sweep_setup(const SweepScratch<S>& W, double* smax, double* star) {
    for (int i = threadIdx.x; i < 2 * S::PT; i += NT) W.w[i] = 0;
    star_setup<NT, Sys>(W.row, smax, star);
}

// dst[p, l, u] += SIGN sum_j sum_m Khat^j[l, o_g + m] X^j[p, m, u] for l < o_g with
// X^j[p, m, u] = sum_q A^{j*}_pq src[q, o_g + m, u], X in fixed point: one scale per
// row (p, u) from the block's max |src| in qmax.  Lanes run over the rows; the
// l are dealt to the warps.  Clears qmax_next; `list` moves to the next
// block's lists.  Begins after and ends with a barrier.
template <int N, int NT, class Sys, class S, int SIGN>
__device__ void khat_block(double* dst, const double* src, int g, const double* star, const KhatRows& K,
                           const int32_t*& list, const SweepScratch<S>& W, const uint32_t* qmax, uint32_t* qmax_next) {
    constexpr int NQ = Sys::NQ, NNZ = Sys::NNZ, T = S::T, QS = S::QS, PT = S::PT, PUL = S::PUL, NW = NT / 32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int o = block_offset(g), d = block_size(g), dm = pass_modes(g, S::XC);
    for (int r = tid; r < PT; r += NT) {
        const int p = r / T, u = r - p * T;
        double b = 0.0;
        for (int n = W.row[p]; n < W.row[p + 1]; ++n) b += W.smax[n] * bound_of(qmax[Sys::col(n) * T + u], 0.0);
        W.scale()[r] = row_scale(b);
        qmax_next[r] = 0u;
    }
    __syncthreads();
#pragma unroll 1
    for (int m0 = 0; m0 < d; m0 += dm) {
        const int nm = min(dm, d - m0);
        // X, quantised: column j * dm + ml
        for (int it = tid; it < 3 * nm * T; it += NT) {
            const int j = it / (nm * T), r = it - j * (nm * T), ml = r / T, u = r - ml * T;
            const double* q = src + (o + m0 + ml) * T + u;
            const double* sj = star + j * NNZ;
            double qv[NQ], acc[NQ];
#pragma unroll
            for (int p = 0; p < NQ; ++p) {
                qv[p] = q[p * QS];
                acc[p] = 0.0;
            }
#pragma unroll
            for (int n = 0; n < NNZ; ++n) acc[Sys::row(n)] = fma(sj[n], qv[Sys::col(n)], acc[Sys::row(n)]);
            int2* x = W.X + (j * dm + ml) * PT + u;
            const int* sc = W.scale() + u;
#pragma unroll
            for (int p = 0; p < NQ; ++p) x[p * T] = quantise(acc[p], sc[p * T]);
        }
        __syncthreads();
        const int i1 = __ldg(list + warp + 1);
        const int32_t* rows = list + NW + 1;
#pragma unroll 1
        for (int i = __ldg(list + warp); i < i1; ++i) {
            const int w = __ldg(rows + i), l = w >> 21, n0 = w & 8191, n1 = n0 + ((w >> 13) & 255);
            const int2* xl = W.X + lane;
            long long hi[PUL];
            long long lo[PUL];
#pragma unroll
            for (int k = 0; k < PUL; ++k) {
                hi[k] = 0;
                lo[k] = 0;
            }
#pragma unroll 4
            for (int n = n0; n < n1; ++n) {
                const int2 en = __ldg(K.ent + n);
                const int2* xc = xl + en.x;
#pragma unroll
                for (int k = 0; k < PUL; ++k)
                    fixed_mac(en.y, xc[32 * k], hi[k], lo[k]);
            }
            const double inv = SIGN * __ldg(K.inv_d + l);
#pragma unroll
            for (int k = 0; k < PUL; ++k) {
                const int r = lane + 32 * k;
                if (r < PT) {
                    double* b = dst + (r / T) * QS + l * T + r % T;
                    *b = fma(fixed_sum(hi[k], lo[k], W.scale()[r]), inv, *b);
                }
            }
        }
        list = rows + __ldg(list + NW);
        __syncthreads();
    }
}

// b[p,l,u] = (S^{-1} w)_u q0[p,l] with (S^{-1} w)_u = (2u+1)(-1)^u
template <int NT, class S>
__device__ __forceinline__ void init_rhs(double* bq, const double* q0) {
    for (int i = threadIdx.x; i < S::NQ * S::B; i += NT) {
        const double v = q0[i];
        const int p = i / S::B, l = i % S::B;
        double* row = bq + p * S::QS + l * S::T;
#pragma unroll
        for (int u = 0; u < S::T; ++u) row[u] = (double)((2 * u + 1) * ((u & 1) ? -1 : 1)) * v;
    }
}

// In-place sweep: on entry bq holds b, on exit the solution Q.  star[3][NNZ]:
// the element's reference Jacobians on the union pattern; zsh: its NSHM shifted
// matrices (Z - e I)^{-1}; gcoup = the coupling entry g of E* (Biot: E*_{u,uf}).
// Begins after and ends with a barrier; both maxima are clear at its ends.
template <int N, int NT, class Sys, class S>
__device__ void alg3_sweep(double* bq, const double* star, const double* zsh, const double gcoup, const KhatRows& K,
                           const SweepScratch<S>& W) {
    constexpr int T = S::T, QS = S::QS;
    const int tid = threadIdx.x;
    const int32_t* list = K.list;
    int buf = 0;
#pragma unroll 1
    for (int g = N; g >= 0; --g) {
        const int o = block_offset(g), d = block_size(g);
        uint32_t* qm = W.qmax(buf);
        // time solves of block g, per mode: the plain rows, the shifted rows,
        // and the coupled pairs (Biot: 6 stresses and p; u_f then u, v_f
        // then v, w_f then w)
        constexpr int NKIND = Sys::NPLAIN + Sys::NSHIFT + Sys::NPAIR;
        for (int it = tid; it < NKIND * d; it += NT) {
            const int kind = it / d, m = o + it % d;
            if (kind < Sys::NPLAIN) {
                const int q = Sys::plain(kind);
                solve_plain<T>(bq + q * QS + m * T, qm + q * T);
            } else if (kind < Sys::NPLAIN + Sys::NSHIFT) {
                const int q = Sys::shifted(kind - Sys::NPLAIN);
                solve_row<T>(bq + q * QS + m * T, zsh, qm + q * T);
            } else {
                const int i = kind - Sys::NPLAIN - Sys::NSHIFT, qf = Sys::pair_src(i), qv = Sys::pair_dst(i);
                double* rf = bq + qf * QS + m * T;
                double* rv = bq + qv * QS + m * T;
                solve_row<T>(rf, zsh, qm + qf * T);
#pragma unroll
                for (int u = 0; u < T; ++u) rv[u] = fma(gcoup, rf[u], rv[u]);
                solve_plain<T>(rv, qm + qv * T);
            }
        }
        __syncthreads();
        if (g == 0) break;
        khat_block<N, NT, Sys, S, -1>(bq, bq, g, star, K, list, W, qm, W.qmax(buf ^ 1));
        buf ^= 1;
    }
    for (int i = tid; i < 2 * S::PT; i += NT) W.w[i] = 0;
    __syncthreads();
}

}  // namespace poro
