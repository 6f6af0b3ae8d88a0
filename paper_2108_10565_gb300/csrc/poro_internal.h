// Internal declarations shared by the host set-up, the C ABI and the kernels
// of libporoader.  Not part of the public interface (include/poroader.h).
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "../../include/poroader.h"

// the CUDA runtime's graph-exec handle (cudaGraphExec_t points to it),
// declared here for the host translation units built without CUDA headers
struct CUgraphExec_st;
struct int4;

namespace poro {

constexpr int NQ = 13;
constexpr int MAX_N = 6;
// quantity indices, paper order (Section "Governing equations")
enum { SXX, SYY, SZZ, SXY, SYZ, SXZ, QU, QV, QW, QP, QUF, QVF, QWF };

constexpr int n_modes(int N) { return (N + 1) * (N + 2) * (N + 3) / 6; }
constexpr int block_size(int g) { return (g + 1) * (g + 2) / 2; }
constexpr int block_offset(int g) { return g * (g + 1) * (g + 2) / 6; }
// tensor-core tile of degree block g's Khat product: N extent (rows l < o_g,
// a multiple of 16, at least 16) and K extent (columns of the block, a
// multiple of the MMA's K step: 8 for tf32 words, 16 for bf16)
constexpr int tc_np(int g) { return block_offset(g) <= 16 ? 16 : (block_offset(g) + 15) / 16 * 16; }
constexpr int tc_kp(int g, bool bf16 = false) {
    return bf16 ? (block_size(g) + 15) / 16 * 16 : (block_size(g) + 7) / 8 * 8;
}

// Union sparsity pattern of A*, B*, C* (54 entries): for every row p the
// columns q with a structurally non-zero Jacobian entry.  Rows are stored
// contiguously; star_row_ptr(p) .. star_row_ptr(p+1) index star_col().
#ifdef __CUDACC__
#define PORO_HD __host__ __device__
#else
#define PORO_HD
#endif
constexpr int STAR_NNZ = 54;
PORO_HD constexpr int star_row_ptr(int p) {
    constexpr int t[NQ + 1] = {0, 6, 12, 18, 20, 22, 24, 28, 32, 36, 42, 46, 50, 54};
    return t[p];
}
PORO_HD constexpr int star_row(int n) {
    return n < 18 ? n / 6 : n < 24 ? 3 + (n - 18) / 2 : n < 36 ? 6 + (n - 24) / 4 : n < 42 ? 9 : 10 + (n - 42) / 4;
}
PORO_HD constexpr int star_col(int n) {
    constexpr int t[STAR_NNZ] = {
        QU, QV, QW, QUF, QVF, QWF,   // s_xx
        QU, QV, QW, QUF, QVF, QWF,   // s_yy
        QU, QV, QW, QUF, QVF, QWF,   // s_zz
        QU, QV,                      // s_xy
        QV, QW,                      // s_yz
        QU, QW,                      // s_xz
        SXX, SXY, SXZ, QP,           // u
        SYY, SXY, SYZ, QP,           // v
        SZZ, SXZ, SYZ, QP,           // w
        QU, QV, QW, QUF, QVF, QWF,   // p
        SXX, SXY, SXZ, QP,           // u_f
        SYY, SXY, SYZ, QP,           // v_f
        SZZ, SXZ, SYZ, QP};          // w_f
    return t[n];
}

// Damped Maxwell equations (Section "Other applications"): 6 quantities
// (E_x, E_y, E_z, H_x, H_y, H_z), eps E_t = curl H - sigma E, mu H_t =
// -curl E.  Union pattern of the reference Jacobians: row p couples the two
// field components of the other kind that its curl row involves.
namespace maxwell {
constexpr int NQ = 6;
constexpr int STAR_NNZ = 12;
PORO_HD constexpr int star_row(int n) { return n / 2; }
PORO_HD constexpr int star_col(int n) {
    constexpr int t[STAR_NNZ] = {4, 5, 3, 5, 3, 4, 1, 2, 0, 2, 0, 1};
    return t[n];
}
// per-element constants: star[3][12], (Z - e I)^{-1} [T][T], e, 0, dt, pad
PORO_HD constexpr int elem_const_stride(int N) { return (3 * STAR_NNZ + (N + 1) * (N + 1) + 4 + 1) & ~1; }
// CTA size of the predictor and the columns of X it holds
constexpr int threads(int N) { return N >= 4 ? 128 : 64; }
constexpr int columns(int N) { return 3 * block_size(N); }
}  // namespace maxwell

// Viscoelastic attenuation (Section "Other applications": upper-triangular
// source matrix), anelastic-function form with NMECH relaxation mechanisms:
// 27 quantities (6 stresses xx yy zz xy yz xz, velocities u v w, then six
// anelastic functions per mechanism in the stress order).  E* holds
// -omega_l dt on the diagonal of mechanism l's functions and the couplings
// -(Ylam_l + 2 Ymu_l) dt, -Ylam_l dt (normal block) and -2 Ymu_l dt (shear)
// from them into the stresses.  Union pattern of the reference Jacobians
// (51 entries a direction): normal stresses <- u v w, shear stresses <- their
// two velocities, velocities <- the three stresses of their row of sigma,
// anelastic functions <- the velocities of their strain-rate component.
namespace visco {
constexpr int NMECH = 3;
constexpr int NQ = 9 + 6 * NMECH;
constexpr int STAR_NNZ = 15 + 9 + 9 * NMECH;
// row-major pattern of the first 24 (stress and velocity rows) and of one
// mechanism's 9 (functions xx yy zz xy yz xz), columns as quantity indices
PORO_HD constexpr int star_row(int n) {
    constexpr int r[24] = {0, 0, 0, 1, 1, 1, 2, 2, 2, 3, 3, 4, 4, 5, 5, 6, 6, 6, 7, 7, 7, 8, 8, 8};
    constexpr int m[9] = {0, 1, 2, 3, 3, 4, 4, 5, 5};
    return n < 24 ? r[n] : 9 + 6 * ((n - 24) / 9) + m[(n - 24) % 9];
}
PORO_HD constexpr int star_col(int n) {
    constexpr int c[24] = {6, 7, 8, 6, 7, 8, 6, 7, 8, 6, 7, 7, 8, 6, 8, 0, 3, 5, 3, 1, 4, 5, 4, 2};
    constexpr int m[9] = {6, 7, 8, 6, 7, 7, 8, 6, 8};
    return n < 24 ? c[n] : m[(n - 24) % 9];
}
// per-element constants: star[3][51], (Z - e_l I)^{-1} [NMECH][T][T], then
// 14 scalars: per mechanism (-(Ylam+2Ymu) dt, -Ylam dt, -2 Ymu dt), e_l
// (NMECH), dt, pad
constexpr int NSC = 3 * NMECH + NMECH + 2;
PORO_HD constexpr int sc_dt() { return 4 * NMECH; }
// ..., then (from an even offset) iso[16], the factors of the star products:
// n^j = -dt grad xi_j [3][3], lam_u, 2 mu_u, mu_u, 1 / rho, omega[3]
PORO_HD constexpr int ec_iso(int N) { return (3 * STAR_NNZ + NMECH * (N + 1) * (N + 1) + NSC + 1) & ~1; }
PORO_HD constexpr int elem_const_stride(int N) { return ec_iso(N) + 16; }
// CTA size of the predictor and the columns of X it holds (N = 6: block 6 in
// two passes, so that three CTAs fit an SM)
constexpr int threads(int N) { return N >= 4 ? 256 : N == 3 ? 128 : 64; }
constexpr int columns(int N) { return N == 6 ? 63 : 3 * block_size(N); }
constexpr int ROWS = 9;  // primitive rows the predictor's integer sums run over
}  // namespace visco

// Per-element constants, in doubles, in this order:
//   star[3][54]       A^{j*} = dt A^j on the union pattern
//   zinv_uf[T][T]     (Z - e I)^{-1}, e = E*_{uf,uf} (row-major, [u][s])
//   e, g, dt, pad     E*_{uf,uf}, E*_{u,uf}, time step
//   iso[16]           (from an even offset) the star products of the isotropic
//                     Jacobians in factored form: n^j = -mu dt grad xi_j
//                     [3][3], then lambda_c / mu, M alpha / mu, M / mu,
//                     m / (D mu), rho_F / (D mu), rho / (D mu), pad
PORO_HD constexpr int ec_zinv(int) { return 3 * STAR_NNZ; }
PORO_HD constexpr int ec_scalars(int N) { return 3 * STAR_NNZ + (N + 1) * (N + 1); }
PORO_HD constexpr int ec_iso(int N) { return (ec_scalars(N) + 4 + 1) & ~1; }
PORO_HD constexpr int elem_const_stride(int N) { return ec_iso(N) + 16; }  // keeps every element's block 16-byte aligned

// Khat^j restricted to the columns of one degree block g, in CSR over the
// rows l < o_g (the only rows Lemma 1 leaves non-zero); entries
// (m_local, value) with m_local < d_g.
struct KhatBlockCSR {
    std::vector<int32_t> row_ptr;    // [o_g + 1]
    std::vector<int32_t> col;        // m_local
    std::vector<double> val;
};

struct ReferenceData {
    int N = 0, B = 0, T = 0;
    std::vector<double> mass_diag;     // [B]
    std::vector<double> khat;          // [3][B][B]
    std::vector<double> zinv;          // [T][T]  Z^{-1}
    std::vector<double> z;             // [T][T]  Z = S^{-1}(W - K^tau)
    std::vector<double> sinv_w;        // [T]     S^{-1} w
    std::vector<KhatBlockCSR> blocks;  // [(N+1)*3], index g*3 + j (block 0 empty)
    int64_t khat_block_nnz = 0;        // structural non-zeros of all Khat blocks
};

// ----- host set-up (setup.cpp) -----
bool reference_data(int N, ReferenceData& out, std::string& err);
bool material_jacobians(const poro_material& m, double abc[3][NQ][NQ], double e[NQ][NQ],
                        std::string& err);
bool max_wave_speed(const poro_material& m, double& v, std::string& err);
bool tet_geometry(const double* v12, double jinv[3][3], double& volume, double& insphere_d,
                  std::string& err);
bool invert_small(int n, const double* a, double* ainv);
// fills one element's constants block (elem_const_stride(N) doubles)
bool element_constants(const ReferenceData& ref, const double* v12, const poro_material& mat,
                       double dt, double* out, std::string& err);
// the same for a damped-Maxwell element, mat = (eps, mu, sigma)
// (maxwell::elem_const_stride(N) doubles)
bool maxwell_element_constants(const ReferenceData& ref, const double* v12, const double mat[3], double dt,
                               double* out, std::string& err);
// One viscoelastic element: mat = rho, lam_u, mu_u, omega[3], Ylam[3],
// Ymu[3]; out gets visco::elem_const_stride(N) doubles
bool visco_element_constants(const ReferenceData& ref, const double* v12, const double mat[12], double dt,
                             double* out, std::string& err);

// ----- sub-cell material (setup.cpp, subcell.cu) -----
// Per element, besides the mean-material constants (elem_const_stride
// layout, from the mode-0 Jacobians): dt grad xi_j on the pattern of the 13
// primitive rows, [3][26], then for the variation modes r = 1..3 of the
// linearly interpolated Jacobians their 9 entries k0..k8 in x-direction
// (subcell.cu, combine_row) and (e_r, g_r) of E*_r.
// (N = 1, 100 and 2,000 elements: 165 and 468 microseconds on 128 threads, 197 and 421 on
// 64; N = 2 525 and 1,616, on 64 676 and 1,822; N = 3, 500 elements: 1.60 ms on 256, 1.79
// on 128; N = 4, where two CTAs fit an SM, 3.73 on 256, 4.69 on 512; N = 5, 100 and 2,000:
// 3.22 and 24.9 ms on 512, 3.48 and 27.0 on 256; N = 6, 100: 5.97 on 512, 6.95 on 256)
constexpr int subcell_threads(int N) { return N >= 5 ? 512 : N >= 3 ? 256 : 128; }
constexpr int subcell_columns(int N) { return N == 6 ? 30 : 3 * block_size(N); }
constexpr int PRIM_NNZ = 26, SUBCELL_MODE = 11;
PORO_HD constexpr int subcell_var_stride() { return (3 * PRIM_NNZ + 3 * SUBCELL_MODE + 1) & ~1; }
// entry n of the primitive rows: row, quantity, component of n
PORO_HD constexpr int prim_row(int n) {
    constexpr int t[PRIM_NNZ] = {0, 0, 0, 1, 1, 1, 2, 3, 3, 4, 4, 5, 5, 6, 6, 6, 7, 7, 7, 8, 8, 8, 9, 10, 11, 12};
    return t[n];
}
PORO_HD constexpr int prim_col(int n) {
    constexpr int t[PRIM_NNZ] = {QU,  QV,  QW,  QUF, QVF, QWF, QU,  QU,  QV,  QV,  QW, QU, QW,
                                 SXX, SXY, SXZ, SXY, SYY, SYZ, SXZ, SYZ, SZZ, QV,  QP, QP, QP};
    return t[n];
}
PORO_HD constexpr int prim_dir(int n) {
    constexpr int t[PRIM_NNZ] = {0, 1, 2, 0, 1, 2, 0, 1, 0, 2, 1, 2, 0, 0, 1, 2, 0, 1, 2, 0, 1, 2, 1, 0, 1, 2};
    return t[n];
}
// Mh3_r = M^{-1} int phi_k phi_r phi_l, r = 1..3, as CSR over all rows k:
// row pointers [3][B + 1] absolute into col / val (device)
struct SubcellReference {
    int32_t* m3_row = nullptr;
    int32_t* m3_col = nullptr;
    double* m3_val = nullptr;
};
// host: the three tensors by the collapsed Gauss rule of reference_data
bool subcell_mass_tensors(const ReferenceData& R, std::vector<int32_t>& row, std::vector<int32_t>& col,
                          std::vector<double>& val, std::string& err);
// host: P[r][v], the modal coefficients f_r = sum_v P[r][v] f_v of the linear
// field with values f_v at the reference vertices
bool subcell_projection(double P[4][4], std::string& err);
// host: one element with vertex materials mats[4] (vertex v of v12 carries
// mats[v]); mean constants into mean_out, variation block into var_out
bool subcell_element_constants(const ReferenceData& ref, const double P[4][4], const double* v12,
                               const poro_material mats[4], double dt, double* mean_out, double* var_out,
                               std::string& err);

// ----- corrector set-up (mesh.cpp) -----
// Godunov flux solver matrices of one face: A_n^L q* = Fm q_L + Fp q_R.
// kind: PORO_FACE_INTERIOR (mR required), PORO_FACE_FREE_SURFACE, PORO_FACE_ABSORBING.
bool flux_solver(const poro_material& mL, const poro_material* mR, const double n[3], int kind, double* Fm,
                 double* Fp, std::string& err);
// phi_l(xi) for all l (singularity-free homogenised recurrences)
void basis_at(int N, const double xi[3], double* phi);
// one face in factors: A_n^L - F^- = W V (every kind) and, on interior
// faces, F^+ = W V; V and W as [13][4]
bool flux_factors(const poro_material& mL, const poro_material* mR, const double n[3], int kind, double* V, double* W,
                  std::string& err);
// Pf[4][df][B], df = (N+1)(N+2)/2: traces in the normalised Dubiner basis of the
// reference triangle on each face (its vertices in increasing local order), so
// that int_face f phi_k phi_l is Pf^T Pf; turn[6][df][df]: with the neighbour's
// trace on its face h under vertex permutation s, Pf[f]^T turn[s] Pf[h]
void face_traces(int N, std::vector<double>& Pf, std::vector<double>& turn);
// The corrector's table of 16-byte words: first the slots (first word, steps, row;
// row -1: none) of the traces, rows of Pf[f] in groups of 8, longest first; of
// M^{-1} Pf^T, likewise; of the turns, one row each; then their entries in blocks
// of 4 steps of a group's rows, padded with zeros: the values of steps 0 and 1 (as
// binary64 or (hi, lo) binary32), row by row, those of steps 2 and 3, and 4 columns
// a row, a byte each.
PORO_HD constexpr int face_modes(int N) { return (N + 1) * (N + 2) / 2; }
PORO_HD constexpr int face_trace_slots(int) { return 0; }
PORO_HD constexpr int face_back_slots(int N) { return 4 * ((face_modes(N) + 7) / 8) * 8; }
PORO_HD constexpr int face_turn_slots(int N) { return face_back_slots(N) + 4 * ((n_modes(N) + 7) / 8) * 8; }
PORO_HD constexpr int face_block_words(int width) { return 2 * width + (width + 3) / 4; }
constexpr int FACE_FACTORS = 2 * 4 * NQ;  // V and W of one face
void face_tables(int N, const std::vector<double>& mass, bool dw, std::vector<int32_t>& words);
int face_permutation_index(const int p[3]);

// ----- device side (kernels) -----
struct DeviceReference {
    int N = 0;
    // the integer Khat rows (khat_tables): 1 / d_l [B] and the same as (hi, lo)
    // binary32 words [B][2]; entries and lists of the binary64 sweep of the
    // context's system (Biot: of the sub-cell iteration)
    double* inv_d = nullptr;
    float* inv_d2 = nullptr;
    int32_t* sweep_ent = nullptr;
    int32_t* sweep_list = nullptr;
};

// Extra device data of the mixed-precision path (the unrefined sweeps).
struct MixedReference {
    const DeviceReference* base = nullptr;
    bool bf16 = false;              // sweeps' split products in bf16 (else tf32)
    float* zinv_f32 = nullptr;      // [T][T]
    // tensor-core images of Khat^j restricted to block g (rows l < o_g, columns
    // of the block), K-major core-matrix layout of tc_np(g) x tc_kp(g) words
    // (tf32 in 32-bit words, or bf16), hi image then lo image; tc_off[g][j] in
    // bytes
    float* khat_tc = nullptr;
    int32_t tc_off[MAX_N + 1][3] = {};
    int32_t* status = nullptr;      // device word: 1 after a bounded wait gave up
    long long wait_limit = 0;       // SM clocks a wait of the sweeps may take (0: about 1 s)
};

// Per-run buffers of a predictor launch that covers the elements of several
// simulations of the same degree and precision (the server's batched mode):
// item i of the launch is element elems[i] of run item_run[i], read from and
// written to that run's buffers.
struct RunPtrs {
    const double* q0;      // [ne][13][B]
    const double* econst;  // [ne][stride]
    double* qt;            // [ne][13][B][T] or nullptr
    double* iout;          // [ne][13][B] or nullptr
    double* qend;          // [ne][13][B] or nullptr: Q~(1), the sum over the time modes (may be q0)
};

// Launch the mixed-precision predictor for `count` elements: binary32 sweeps
// (refine 0), double-binary32 (1) or binary64 (2).  With `runs`
// (device array) and `item_run`, the items come from several runs and q0,
// econst, qt, iout are ignored.
int launch_stp_mixed(const MixedReference& ref, int refine, const int32_t* elems, int64_t count,
                     const double* q0, const double* econst, double* qt, double* iout, double* qend, void* stream,
                     int variant = 0, const RunPtrs* runs = nullptr, const int32_t* item_run = nullptr);

// Dense-LU comparator: reference data and per-batch scratch (factors,
// pivots, permutation, equilibration factors, singularity flag).
struct LUReference {
    int N = 0;
    double* z = nullptr;       // [T][T] Z = S^{-1}(W - K^tau)
    int32_t* krow = nullptr;   // [3][B+1] full-row CSR of Khat^j, absolute offsets
    int32_t* kcol = nullptr;
    double* kval = nullptr;
};
struct LUScratch {
    double* A = nullptr;       // [count][s][s] factors L\U of P R Y' C
    int32_t* piv = nullptr;    // [count][s]
    int32_t* perm = nullptr;   // [count][s]
    double* R = nullptr;       // [count][s]
    double* C = nullptr;       // [count][s]
    int32_t* bad = nullptr;    // 1 if a zero pivot occurred
    double* x = nullptr;       // [count][s] solution scratch of the blocked solve (nullable: one CTA per element)
    // the blocked solve's launches captured as a CUDA graph, valid for the
    // pointers and counts in key
    CUgraphExec_st* exec = nullptr;  // a cudaGraphExec_t
    const void* key[10] = {};
};
size_t lu_scratch_bytes(int N, int64_t count);
int launch_lu_factor(const LUReference& ref, int64_t count, const double* econst, LUScratch& w, void* stream);
int launch_lu_solve(const LUReference& ref, int64_t count, LUScratch& w, int64_t offset, const double* q0,
                    const double* econst, double* qt, double* iout, void* stream);

// Read-only view of the context fields the allocation-free LU entry point
// needs (defined in api.cu).
struct CtxView {
    int device = 0, N = 0;
    int64_t n_elem = 0;
    int stride = 0;
    const double* econst = nullptr;
    const LUReference* lref = nullptr;
    void* stream = nullptr;
};
bool ctx_view(const poro_ctx* c, CtxView& v);
void ctx_set_error(poro_ctx* c, const std::string& msg);

// Corrector (Eq. semi_discrete integrated over one step) for `count`
// elements starting at `first` of the mesh.
struct CorrectorData {
    int N = 0;
    const double* econst = nullptr;   // [ne][stride] (stars with dt, e, g, dt)
    const double* iout = nullptr;     // [ne][13][B] time-integrated predictor
    double* q = nullptr;              // [ne][13][B] DOFs, updated in place
    const int32_t* nb = nullptr;      // [ne][4]
    const int32_t* tab = nullptr;     // [ne][4] neighbour table index f*24 + h*6 + s, or -1
    bool dw = false;                  // double-binary32 (mixed-precision contexts), else binary64
    // [ne][4][2][13][4]: V, then c_f W (c_f = 2 |S_f| / |J|), of each face in 8-byte
    // words: binary64, or in double-binary32 two entries in 16 bytes, both high words
    // and then both low ones (the layout of a packed pair)
    const void* fvw = nullptr;
    const int4* ftab = nullptr;       // face_tables
    const int32_t* krow = nullptr;    // full-row CSR of Khat^j [3][B+1] (absolute)
    const int32_t* kcol = nullptr;
    const double* kval = nullptr;
    // clustered local time stepping (all nullptr / 1 for global time stepping)
    int C = 1;                        // number of clusters
    const int32_t* cl = nullptr;      // [ne] cluster of each element
    const int32_t* slot = nullptr;    // [ne][C] buffer slot of (element, larger level) or -1
    const double* buf = nullptr;      // [slots][13][B] buffered sub-step integrals
    const double* qt = nullptr;       // [ne][13][B][T] full predictors (larger neighbours)
    int64_t tick = 0;                 // tick k of the correction (interval ends at k + 1)
};
// one cluster's sub-step buffers, items (element, slot, level, -)
int launch_lts_buffers(int N, const int4* items, int64_t count, const double* iout, double* buf, int64_t tick,
                       void* stream);
// The faces' part of the corrector; with `volume` first the volume and source
// part (for a predictor that did not write Q~(1)).  `runs` (device array,
// nullable) / `item_run`: a launch over several runs; item i is element
// elems[i] of the run whose data is runs[item_run[i]] (d then only selects the
// precision and degree)
int launch_corrector(const CorrectorData& d, bool volume, const int32_t* elems, int64_t count, void* stream,
                     const CorrectorData* runs = nullptr, const int32_t* item_run = nullptr);
// One point source or receiver of one run.  Source: q[elem] += (S(t1) - S(t0)) vec
// over the step [(k+1-len) dt, (k+1) dt], k = *tick + k_rel (+ the launch's tick);
// receiver: out[*counter] = Q[elem] vec, then ++*counter.  One launch takes the
// sources (then one the receivers) of a cluster, or of all runs of a batched group.
struct TickItem {
    double* q = nullptr;
    const double* vec = nullptr;     // coef (source) or phi (receiver)
    double* out = nullptr;           // receiver samples
    int32_t* counter = nullptr;      // receiver sample counter
    const int64_t* tick = nullptr;   // the run's tick counter (source)
    int64_t elem = 0, len = 1, k_rel = 0;
    double f0 = 0.0, tc = 0.0, dt = 0.0;
};
// (items of one element side by side)
int launch_tick_sources(int N, const TickItem* items, int64_t count, void* stream);
// one run's list, in order, at tick k_add of the cycle
int launch_source_list(int N, const TickItem* items, int count, int64_t k_add, void* stream);
int launch_tick_receivers(int N, const TickItem* items, int64_t count, void* stream);
// *ticks[i] += n for i < count (the tick counters of a group's runs)
int launch_ticks_advance(int64_t* const* ticks, int count, int64_t n, void* stream);
int launch_tick_advance(int64_t* tick, int64_t n, void* stream);

// Batched advance of several simulations (the server): runs of one degree,
// precision, refinement, CTA variant and cluster count, each at the end of a
// cycle.  Every tick's predictors of all runs are one launch; each run's
// results are those it gets when advanced alone.  group_enqueue queues
// n_cycles cycles on the group's own stream; group_finish waits for them and
// appends the receiver samples.  The runs must not be used otherwise while
// the group exists.
struct RunGroup;
RunGroup* group_create(poro_ctx* const* runs, int n, std::string& err);
int group_enqueue(RunGroup* g, int64_t n_cycles, std::string& err);
poro_status group_finish(RunGroup* g, std::string& err);
void group_destroy(RunGroup* g);

// x = num / den with den <= 10^6 if x is such a rational to 1e-14 relative
bool rational_of(double x, int64_t& num, int64_t& den);
// Coefficients of the derivatives along xi, eta, zeta -> along xi, eta - xi / 2,
// zeta - eta, the directions of the integer Khat rows: sum_j n_j d_j is the same
PORO_HD inline void adapted_directions(double& n0, double& n1, double n2) {
    n1 += n2;
    n0 += 0.5 * n1;
}
// Integer Khat rows in passes of at most `columns` columns (direction, mode) of
// X: entries (column * stride, numerator) pass by pass, 1 / d_l per row, and
// (appended to list) per pass the rows dealt to `warps` warps, [warps + 1]
// starts, then words l << 21 | entries << 13 | first entry.
bool khat_tables(const ReferenceData& R, int columns, int stride, int warps, std::vector<int32_t>& ent,
                 std::vector<int32_t>& list, std::vector<double>& inv_d, std::string& err);
// The same for Biot's predictor kernel (stp_direct.cu), lists of all its warp
// counts; then their upload (once per device and degree).
bool direct_tables(const ReferenceData& R, std::vector<int32_t>& ent, std::vector<int32_t>& list,
                   std::vector<double>& inv_d, std::string& err);
int upload_direct_tables(int N, const std::vector<int32_t>& ent, const std::vector<int32_t>& list);
// Biot's predictor in binary64 or (dw) double-binary32, arguments as for
// launch_stp_fp64.  whole_nan: a non-finite value makes the element's whole
// result NaN; status, wait_limit: the bounded wait of the double-binary32 form.
int launch_stp_direct(const DeviceReference& ref, bool dw, bool whole_nan, int32_t* status, long long wait_limit,
                      const int32_t* elems, int64_t count, const double* q0, const double* econst, double* qt,
                      double* iout, double* qend, void* stream, int variant, const RunPtrs* runs,
                      const int32_t* item_run);
// the CTA size it takes for `count` elements (variant 0, 1 or 2), and a count from
// which on variant 0 takes the default size at every degree
int direct_cta_size(int N, int variant, int64_t count);
int64_t direct_default_count();

// Launch the FP64 Algorithm-3 predictor for `count` elements.
// q0[count][13][B], econst[count][stride], qt, iout, qend (Q~(1), may be q0) nullable.
// `elems` (nullable): element index list; outputs are indexed by element.
// `variant` selects the CTA size (0: default, wider for launches of few elements;
// 1: the alternative; 2: the alternative in place of the default, for launches of
// more elements, which the autotuners may pick).  `runs` / `item_run`: items of several runs, as for
// launch_stp_mixed.
int launch_stp_fp64(const DeviceReference& ref, const int32_t* elems, int64_t count, const double* q0,
                    const double* econst, double* qt, double* iout, double* qend, void* stream, int variant = 0,
                    const RunPtrs* runs = nullptr, const int32_t* item_run = nullptr);
// The same kernel for the damped Maxwell system (q0 [count][6][B], econst
// [count][maxwell::elem_const_stride(N)], qt [count][6][B][T]).
int launch_stp_fp64_maxwell(const DeviceReference& ref, int64_t count, const double* q0, const double* econst,
                            double* qt, double* iout, void* stream);
// Sub-cell material predictor (subcell.cu): evar [count][subcell_var_stride()],
// iters [count] (iterations of each element, negative if not converged).
int launch_stp_subcell(const DeviceReference& ref, const SubcellReference& sub, int64_t count, const double* q0,
                       const double* econst, const double* evar, double* qt, double* iout, int32_t* iters,
                       double tol, int max_iter, void* stream);
// ... and for the viscoelastic system (q0 [count][27][B], econst
// [count][visco::elem_const_stride(N)], qt [count][27][B][T]).
int launch_stp_fp64_visco(const DeviceReference& ref, int64_t count, const double* q0, const double* econst,
                            double* qt, double* iout, void* stream);

}  // namespace poro
