// K2: the unrefined form of the mixed-precision space-time predictor (mixed
// contexts with no refinement sweep; with one or two the predictor is
// stp_direct.cu's).
//
// One binary32 sweep of Algorithm 3 (degree blocks, time solves with
// (Z - E*_pp I)^{-1}, G coupling, star and Khat products).  The dominant step,
// b[p, l, u] -= sum_j sum_m Khat^j[l, m] X^j[p, m, u] over the rows l < o_g of
// degree block g, is a dense contraction whose left operand Khat is the same
// for every element: it runs on the tensor cores (tcgen05.mma, accumulator in
// TMEM) with both operands split into hi + lo words (tf32, or bf16 for the bf16
// form) and the three products hi*hi + hi*lo + lo*hi accumulated.  One MMA
// tile per (g, j): M = 128 rows (p, u) of the element, N = rows l (o_g rounded
// up to 16), K = columns m of the block.  X^j (A operand) is written by the
// star-product threads straight into shared memory in the K-major core-matrix
// layout; the Khat^j block images (B operand, prebuilt on the host in the same
// layout) arrive by bulk copy, prefetched during the previous block (tc_layout
// says which buffers fit per block).
#include <cuda_runtime.h>

#include "alg3_device.cuh"
#include "dw_device.cuh"
#include "tc_device.cuh"

namespace poro {
namespace {

struct K2Params {
    const int32_t* elems;     // optional element index list (LTS clusters)
    const double* q0;
    const double* econst;
    double* qt;
    double* iout;
    int64_t count;
    int stride;
    const float* zinv;        // Z^{-1} [T][T] binary32
    const float* khat_tc;     // tensor-core images of the Khat^j blocks (hi then lo)
    int32_t tc_off[MAX_N + 1][3];
    int32_t* status;          // set to 1 if a bounded wait gave up
    long long wait_limit;     // SM clocks after which a wait of the sweeps gives up (> 0)
    const RunPtrs* runs;      // items of several runs (nullptr: q0, econst, qt, iout above)
    const int32_t* item_run;
};

// CTA sizes the autotuner chooses from (index 0 is the default)
template <int N>
struct K2Sizes {
    static constexpr int NT0 = N >= 5 ? 256 : (N == 4 ? 128 : 64);
    static constexpr int NT1 = N >= 5 ? 128 : (N == 4 ? 256 : 128);
};

template <int N, int NT_, int BF = 0>
struct K2Shape : Alg3Shape<N> {
    using A = Alg3Shape<N>;
    static constexpr int NT = NT_;
    static constexpr int NW = NT / 32;
    static constexpr int T_ = N + 1;
    static constexpr int R4(int x) { return (x + 3) & ~3; }
    static constexpr int R32(int x) { return (x + 31) & ~31; }
    static constexpr int MAX2(int a, int b) { return a > b ? a : b; }
    // tensor-core operand tiles: A (X^j, hi and lo) with ceil(13 T / 8) row
    // groups of the widest block, then the Khat^j image (hi and lo).  The MMA
    // reads 16 row groups of each A tile; the rows past 13 T only feed
    // accumulator rows that are never read, so they may overlap what follows.
    // (sizes in floats; operand words are 4 bytes for tf32, 2 for bf16)
    static constexpr int ES = BF ? 2 : 4;
    static constexpr int KPM = tc_kp(N, BF != 0);
    static constexpr int SBOMAX = KPM * 8 * ES / 4;
    static constexpr int AH = (A::PT + 7) / 8 * SBOMAX;
    static constexpr int BIMG = 2 * tc_np(N) * KPM * ES / 4;
    // at least one A tile pair and one Khat image; the bf16 form gets the
    // room of the tf32 form, where the Khat images of all three directions fit
    // beside one A pair at every degree (tf32: up to degree 4)
    static constexpr int TC1 = MAX2(2 * AH + BIMG, AH + 16 * SBOMAX);
    static constexpr int TC_SIZE = BF ? MAX2(TC1, 2 * AH + 3 * BIMG) : TC1;
    // shared layout in floats
    static constexpr int OFF_XY = 0;
    static constexpr int XY_SIZE = R32(TC_SIZE);
    static constexpr int OFF_W = OFF_XY + XY_SIZE;
    static constexpr int OFF_SH = OFF_W + R4(A::SQ);
    static constexpr int OFF_ZIN = OFF_SH + R4(3 * STAR_NNZ);  // [T][8]
    static constexpr int OFF_ZUF = OFF_ZIN + 8 * T_;            // [T][8]
    static constexpr int OFF_BAR = OFF_ZUF + 8 * T_;  // 5 mbarriers, wait limit, TMEM slot, abort, dirty, drain mask
    static constexpr int SMEM_FLOATS = OFF_BAR + 16;
    static constexpr int TMEM_COLS = tc_np(N) <= 32 ? 32 : (tc_np(N) <= 64 ? 64 : 128);
    static_assert(A::PT <= 32 * (NW < 4 ? NW : 4), "every accumulator row (p, u) needs a reading warp");
    static_assert(NW == 2 || NW == 4 || NW == 8, "2, 4 or 8 warps");
};

// row[0..T) <- Zi row[0..T), Zi stored with row stride 8 (two 16-byte loads a row)
template <int T>
__device__ __forceinline__ void solve_row8(float* row, const float* Zi) {
    float x[T];
#pragma unroll
    for (int s = 0; s < T; ++s) x[s] = row[s];
#pragma unroll
    for (int u = 0; u < T; ++u) {
        const float4 a = *reinterpret_cast<const float4*>(Zi + 8 * u);
        float z[8] = {a.x, a.y, a.z, a.w, 0.f, 0.f, 0.f, 0.f};
        if constexpr (T > 4) {
            const float4 b = *reinterpret_cast<const float4*>(Zi + 8 * u + 4);
            z[4] = b.x;
            z[5] = b.y;
            z[6] = b.z;
            z[7] = b.w;
        }
        float acc = 0.f;
#pragma unroll
        for (int s = 0; s < T; ++s) acc = fmaf(z[s], x[s], acc);
        row[u] = acc;
    }
}

// Tensor-core state of one CTA (shared addresses, barrier phases).  Thread 0
// issues every MMA commit and the Khat copies needed inside a block; thread
// 96 (a warp with no epilogue rows) issues the next block's copies once the
// block's MMAs are done.  An issuing thread issues only while all of its own
// waits have succeeded.  Thread 0 waits for every copy before the MMAs that
// read it, and thread 96's copies follow MMAs that thread 0 issued only after
// such waits, so no barrier ever gets a second operation while an earlier one
// may still be in flight.
// Each thread keeps in `pend` the barriers it gave work that it has not seen
// complete: bits 0, 1 MMA commits (cleared by the successful wait), bits 2-4
// Khat copies into slots 0-2 (cleared by thread 0's wait on the copy, and by
// every thread once the block's last MMAs are done, which implies that every
// copy of the block was consumed); bit 31 records that one of the thread's
// waits gave up.  The abort path merges the masks of threads 0 and 96.
struct TcState {
    float* xy;      // operand region: A tiles (tf32 words, or bf16 values in the same bytes), then Khat images
    uint32_t xy_s;  // its shared address
    int xy_floats;  // its size
    uint32_t bar_s;     // mbarriers: MMAs done reading A buffer 0, 1; Khat image in slot 0, 1, 2
    uint32_t tmem;
    uint32_t mph, lph;  // phase parity of each barrier (bit b for MMA barrier b, bit 2 + s for slot s)
    uint32_t pend;      // barriers given work not seen complete; bit 31: a wait gave up
    volatile int* abort;
};
constexpr uint32_t GAVE_UP = 1u << 31;

// A wait that gives up keeps its phase, so that the abort path can still
// wait (with the full limit) for the operation it was waiting for
__device__ __forceinline__ void tc_wait(TcState& S, uint32_t bit) {
    const uint32_t par = ((bit < 2 ? S.mph : S.lph) >> bit) & 1u;
    // the wait limit is the 64-bit word after the five mbarriers
    if (tc::mbar_wait_s(S.bar_s + 8u * bit, par, S.bar_s + 40u)) {
        if (bit < 2)
            S.mph ^= 1u << bit;
        else
            S.lph ^= 1u << bit;
        S.pend &= ~(1u << bit);
    } else {
        *S.abort = 1;
        S.pend |= GAVE_UP;
    }
}

// abort path (thread 0, after a CTA barrier, with `mask` the union of the
// issuing threads' records): a wait with the full limit on every barrier
// given work not seen complete, so that copies and MMAs still in flight have
// landed before the CTA frees its TMEM and exits.  Barriers with nothing in
// flight are skipped.  (A copy of thread 96 that thread 0 consumed before an
// MMA wait gave up stays in thread 96's record; its barrier then has no
// pending phase and the wait runs out its limit: bounded, and only on this
// path.)
__device__ __forceinline__ void tc_drain(TcState& S, uint32_t mask) {
    for (uint32_t bit = 0; bit < 5; ++bit)
        if ((mask >> bit) & 1u) tc::mbar_wait(S.bar_s + 8u * bit, ((bit < 2 ? S.mph : S.lph) >> bit) & 1u);
}

// Operand layout of degree block g in the region (floats): nA A buffers (hi
// tile, lo tile), then nB Khat image slots (hi image, lo image).  Direction j
// uses A buffer j % nA and slot j % nB.  An MMA reads 16 row groups of an A
// tile; the rows past 13 T feed accumulator rows that are never read and
// stay inside the region.  As many slots as fit (all three directions' images
// can then be in flight before the block starts), then a second A buffer if
// it fits (the star products of direction j overlap the MMAs of j - 1).
struct TcLayout {
    int KP, NP, ahf, bif, nA, nB;
    uint32_t sbo, half;  // bytes: 8-row group stride; one Khat image (hi or lo)
};
template <int PT, int BF>
__device__ __forceinline__ TcLayout tc_layout(int g, int xy_floats) {
    constexpr int ES = BF ? 2 : 4;
    TcLayout L;
    L.KP = tc_kp(g, BF != 0);
    L.NP = tc_np(g);
    L.sbo = (uint32_t)L.KP * 8u * ES;
    L.half = (uint32_t)(L.NP * L.KP) * ES;
    L.ahf = (PT + 7) / 8 * (int)(L.sbo / 4);
    L.bif = (int)(2u * L.half / 4u);
    const int over = 16 * (int)(L.sbo / 4) - L.ahf;
    auto fits = [&](int na, int nb) { return 2 * na * L.ahf + nb * L.bif <= xy_floats && (2 * na - 1) * L.ahf + 16 * (int)(L.sbo / 4) <= xy_floats && over >= 0; };
    L.nB = fits(1, 3) ? 3 : (fits(1, 2) ? 2 : 1);
    // direction j >= nB loads once the MMAs of j - nB are done, known at step
    // j - nB + nA: that is no later than step j only if nA <= nB.  With three
    // A buffers (and three slots) the block runs all directions in one pass.
    L.nA = (L.nB == 3 && fits(3, 3)) ? 3 : ((L.nB >= 2 && fits(2, L.nB)) ? 2 : 1);
    return L;
}

// bulk copy of direction j's Khat image of block g into its slot (one
// thread, unless one of its waits gave up)
template <int PT, int BF>
__device__ __forceinline__ void tc_load_khat(TcState& S, const TcLayout& L, const K2Params& P, int g, int j) {
    if (S.pend & GAVE_UP) return;
    const int slot = j % L.nB;
    S.pend |= 4u << slot;
    const uint32_t bar = S.bar_s + 16u + 8u * (uint32_t)slot;
    const uint32_t dst = S.xy_s + 4u * (uint32_t)(2 * L.nA * L.ahf + slot * L.bif);
    tc::fence_async_smem();
    tc::mbar_expect_tx(bar, 2u * L.half);
    tc::bulk_g2s(dst, reinterpret_cast<const char*>(P.khat_tc) + P.tc_off[g][j], 2u * L.half, bar);
}

// star products of one item (ml, u) of block g (modes o + ml) for direction
// j's 54 coefficients: acc[p] = sum_q A^{j*}_pq Q[q, o+ml, u]
template <int T, int QS>
__device__ __forceinline__ void star_item(const float* bq, const float* sj, int o, int it, float acc[NQ]) {
    const int ml = it / T, u = it % T;
    float qv[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        qv[q] = bq[q * QS + (o + ml) * T + u];
        acc[q] = 0.f;
    }
#pragma unroll
    for (int n = 0; n < STAR_NNZ; ++n) acc[star_row(n)] = fmaf(sj[n], qv[star_col(n)], acc[star_row(n)]);
}

// store one item's 13 values as hi + lo (tf32 words, or bf16) into the A tiles
template <int T, int BF>
__device__ __forceinline__ void store_item(float* ah, float* al, int it, int KP, const float acc[NQ]) {
    const int ml = it / T, u = it % T;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        if (BF) {
            const int at = tc::kmajor_offset16(q * T + u, ml, KP);
            const uint16_t h = tc::bf16_bits(acc[q]);
            reinterpret_cast<uint16_t*>(ah)[at] = h;
            reinterpret_cast<uint16_t*>(al)[at] = tc::bf16_bits(acc[q] - tc::bf16_value(h));
        } else {
            const int at = tc::kmajor_offset(q * T + u, ml, KP);
            const float h = tc::to_tf32(acc[q]);
            ah[at] = h;
            al[at] = acc[q] - h;
        }
    }
}

// One binary32 sweep of Algorithm 3 with the Khat products on the tensor
// cores.  On entry bq holds b, on exit Q.  Returns false (uniformly across the
// CTA) if a bounded wait gave up.
template <int N, int NT, int BF>
__device__ bool alg3_sweep_tc(float* bq, const float* star, const float* zuf, const float* zin, const float gcoup,
                              const K2Params& P, TcState& S) {
    using A = Alg3Shape<N>;
    constexpr int T = A::T, QS = A::QS, PT = A::PT, NW = NT / 32;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the first block's Khat images load while its time solves run
    if (tid == 0 && N >= 1) {
        const TcLayout L0 = tc_layout<PT, BF>(N, S.xy_floats);
        for (int j = 0; j < L0.nB; ++j) tc_load_khat<PT, BF>(S, L0, P, N, j);
    }
#pragma unroll 1
    for (int g = N; g >= 0; --g) {
        const int o = block_offset(g), d = block_size(g);
        // time solves of block g: 7 plain rows (6 stresses, p) and 3 coupled
        // pairs (u_f then u, v_f then v, w_f then w) per mode
        for (int it = tid; it < 10 * d; it += NT) {
            const int kind = it / d, m = o + it % d;
            if (kind < 7) {
                const int p = kind < 6 ? kind : QP;
                solve_row8<T>(bq + p * QS + m * T, zin);
            } else {
                const int i = kind - 7;
                float* rf = bq + (QUF + i) * QS + m * T;
                float* rv = bq + (QU + i) * QS + m * T;
                solve_row8<T>(rf, zuf);
#pragma unroll
                for (int u = 0; u < T; ++u) rv[u] = fmaf(gcoup, rf[u], rv[u]);
                solve_row8<T>(rv, zin);
            }
        }
        __syncthreads();
        if (g == 0) break;
        constexpr int KSTEP = BF ? 16 : 8;
        const TcLayout L = tc_layout<PT, BF>(g, S.xy_floats);
        const int KP = L.KP, NP = L.NP;
        const uint32_t sbo = L.sbo, half = L.half;
        if (L.nA == 3) {
            // small block: the star products of all three directions in one
            // pass, one barrier, then every direction's MMAs and one commit
            for (int it = tid; it < 3 * d * T; it += NT) {
                const int j = it / (d * T), r = it - j * (d * T);
                float acc[NQ];
                star_item<T, QS>(bq, star + j * STAR_NNZ, o, r, acc);
                store_item<T, BF>(S.xy + 2 * j * L.ahf, S.xy + (2 * j + 1) * L.ahf, r, KP, acc);
            }
            tc::fence_async_smem();
            __syncthreads();
            if (*S.abort) return false;
            if (tid == 0) {
                for (int j = 0; j < 3; ++j) tc_wait(S, 2u + (uint32_t)j);
            }
            if (tid == 0 && !(S.pend & GAVE_UP)) {
                tc::fence_after_sync();
                const uint32_t id = BF ? tc::idesc_bf16(128, NP) : tc::idesc_tf32(128, NP);
                const int nk = KP / KSTEP;
                constexpr int MAXK = tc_kp(N, BF != 0) / KSTEP;
                for (int j = 0; j < 3; ++j) {
                    const uint32_t ah_s = S.xy_s + 4u * (uint32_t)(2 * j * L.ahf), al_s = ah_s + 4u * (uint32_t)L.ahf;
                    const uint32_t b_s = S.xy_s + 4u * (uint32_t)(6 * L.ahf + j * L.bif);
                    const uint64_t dal = tc::smem_desc(al_s, sbo), dah = tc::smem_desc(ah_s, sbo);
                    const uint64_t dbh = tc::smem_desc(b_s, sbo), dbl = tc::smem_desc(b_s + half, sbo);
#pragma unroll
                    for (int kk = 0; kk < MAXK; ++kk) {
                        if (kk < nk) {
                            const uint64_t k16 = 16ull * (uint64_t)kk;
                            if (BF) {
                                tc::mma_bf16(S.tmem, dal + k16, dbh + k16, id, (j | kk) != 0);
                                tc::mma_bf16(S.tmem, dah + k16, dbl + k16, id, 1u);
                                tc::mma_bf16(S.tmem, dah + k16, dbh + k16, id, 1u);
                            } else {
                                tc::mma_tf32(S.tmem, dal + k16, dbh + k16, id, (j | kk) != 0);
                                tc::mma_tf32(S.tmem, dah + k16, dbl + k16, id, 1u);
                                tc::mma_tf32(S.tmem, dah + k16, dbh + k16, id, 1u);
                            }
                        }
                    }
                }
                tc::mma_commit(S.bar_s);
                S.pend |= 1u;
            }
            tc_wait(S, 0u);
            // the block's MMAs are done: every copy of the block was consumed
            if (!(S.pend & GAVE_UP)) S.pend &= ~0x1Cu;
        } else {
#pragma unroll 1
        for (int j = 0; j < 3; ++j) {
            const int abuf = j % L.nA, slot = j % L.nB;
            const uint32_t mma_bar = S.bar_s + 8u * (uint32_t)abuf;
            if (j >= L.nA) {  // the MMAs of direction j - nA (and all before) are done
                tc_wait(S, (uint32_t)abuf);
                // their slots are free: load the images not yet in flight
                if (tid == 0)
                    for (int k = L.nB; k < 3; ++k)
                        if (k - L.nB <= j - L.nA && k - L.nB > j - 1 - L.nA) tc_load_khat<PT, BF>(S, L, P, g, k);
            }
            float* ah = S.xy + 2 * abuf * L.ahf;
            float* al = ah + L.ahf;
            const uint32_t ah_s = S.xy_s + 4u * (uint32_t)(2 * abuf * L.ahf), al_s = ah_s + 4u * (uint32_t)L.ahf;
            const uint32_t b_s = S.xy_s + 4u * (uint32_t)(2 * L.nA * L.ahf + slot * L.bif);
            // X^j[p, ml, u] = sum_q A^{j*}_pq Q[q, o+ml, u], stored as hi + lo
            // (tf32 words, or bf16)
            const float* sj = star + j * STAR_NNZ;
            for (int it = tid; it < d * T; it += NT) {
                float acc[NQ];
                star_item<T, QS>(bq, sj, o, it, acc);
                store_item<T, BF>(ah, al, it, KP, acc);
            }
            tc::fence_async_smem();
            __syncthreads();
            if (*S.abort) return false;
            if (tid == 0) tc_wait(S, 2u + (uint32_t)slot);
            if (tid == 0 && !(S.pend & GAVE_UP)) {
                tc::fence_after_sync();
                const uint32_t id = BF ? tc::idesc_bf16(128, NP) : tc::idesc_tf32(128, NP);
                // one K step = two core matrices along K, 256 B further: 16
                // units of the descriptors' start-address field (no carry,
                // shared addresses are below 2^18)
                const uint64_t dal = tc::smem_desc(al_s, sbo), dah = tc::smem_desc(ah_s, sbo);
                const uint64_t dbh = tc::smem_desc(b_s, sbo), dbl = tc::smem_desc(b_s + half, sbo);
                const int nk = KP / KSTEP;
                constexpr int MAXK = tc_kp(N, BF != 0) / KSTEP;
#pragma unroll
                for (int kk = 0; kk < MAXK; ++kk) {
                    if (kk < nk) {
                        const uint64_t k16 = 16ull * (uint64_t)kk;
                        if (BF) {
                            tc::mma_bf16(S.tmem, dal + k16, dbh + k16, id, (j | kk) != 0);
                            tc::mma_bf16(S.tmem, dah + k16, dbl + k16, id, 1u);
                            tc::mma_bf16(S.tmem, dah + k16, dbh + k16, id, 1u);
                        } else {
                            tc::mma_tf32(S.tmem, dal + k16, dbh + k16, id, (j | kk) != 0);
                            tc::mma_tf32(S.tmem, dah + k16, dbl + k16, id, 1u);
                            tc::mma_tf32(S.tmem, dah + k16, dbh + k16, id, 1u);
                        }
                    }
                }
                tc::mma_commit(mma_bar);
                S.pend |= 1u << abuf;
            }
        }
        // wait for the commits not yet waited for (directions 3 - nA .. 2);
        // the last one covers every MMA of the block
#pragma unroll 1
        for (int j = 3 - L.nA; j < 3; ++j) {
            tc_wait(S, (uint32_t)(j % L.nA));
        }
        // the block's MMAs are done: every copy of the block was consumed
        if (!(S.pend & GAVE_UP)) S.pend &= ~0x1Cu;
        }
        // the region is free: the next block's Khat images load during this
        // block's epilogue and the next time solves (issued by lane 0 of warp
        // 3, whose TMEM lane quarter holds no rows: 13 T <= 96)
        if (tid == (NW >= 4 ? 96 : 0) && g > 1) {
            const TcLayout Ln = tc_layout<PT, BF>(g - 1, S.xy_floats);
            for (int j = 0; j < Ln.nB; ++j) tc_load_khat<PT, BF>(S, Ln, P, g - 1, j);
        }
        tc::fence_after_sync();
        // b[p, l, u] -= D[(p, u), l]: warp w reads TMEM lanes 32 (w % 4) ...,
        // with 8 warps the two warps of a lane quarter split the columns
        {
            const int sp = warp & 3;
            const int ncol = NW == 8 ? NP / 2 : NP;
            const int c_begin = NW == 8 ? (warp >> 2) * ncol : 0;
            // a warp with a lane whose wait gave up reads no TMEM (the MMAs
            // may still be writing it); the CTA leaves the sweep below
            const bool skip = __any_sync(0xffffffffu, (S.pend & GAVE_UP) != 0u);
            if (sp * 32 < PT && !skip) {
                const int r = sp * 32 + lane;
                const int p = r / T, u = r - (r / T) * T;
                float* dst = bq + p * QS + u;
                const int c_end = min(c_begin + ncol, o);
#pragma unroll 1
                for (int c0 = c_begin; c0 < c_end; c0 += 16) {
                    float v[16];
                    tc::tmem_ld16(S.tmem + ((uint32_t)(sp * 32) << 16) + (uint32_t)c0, v);
                    if (r < PT) {
#pragma unroll
                        for (int q = 0; q < 16; ++q)
                            if (c0 + q < c_end) dst[(c0 + q) * T] -= v[q];
                    }
                }
            }
        }
        tc::fence_before_sync();
        __syncthreads();
        if (*S.abort) return false;
    }
    return true;
}

template <int N, int NT_, int BF>
__global__ void __launch_bounds__(NT_, 2) stp_mixed_kernel(const K2Params P) {
    using S = K2Shape<N, NT_, BF>;
    constexpr int B = S::B, T = S::T, NT = S::NT, QBT = S::QBT, QS = S::QS;
    extern __shared__ __align__(1024) float smf[];
    float* W = smf + S::OFF_W;
    float* sh = smf + S::OFF_SH;
    float* zin = smf + S::OFF_ZIN;
    float* zuf = smf + S::OFF_ZUF;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smf + S::OFF_BAR);
    long long* wlimit = reinterpret_cast<long long*>(smf + S::OFF_BAR + 10);  // wait limit (SM clocks)
    uint32_t* tslot = reinterpret_cast<uint32_t*>(smf + S::OFF_BAR + 12);
    volatile int* abort = reinterpret_cast<volatile int*>(smf + S::OFF_BAR + 13);
    int* dirty = reinterpret_cast<int*>(smf + S::OFF_BAR + 14);  // a result was not finite
    uint32_t* drain_mask = reinterpret_cast<uint32_t*>(smf + S::OFF_BAR + 15);  // thread 96's record, at exit
    const int tid = threadIdx.x;

    TcState tcs;
    tcs.xy = smf + S::OFF_XY;
    tcs.xy_s = tc::smem_addr(tcs.xy);
    tcs.xy_floats = S::XY_SIZE;
    tcs.bar_s = tc::smem_addr(bars);
    tcs.mph = tcs.lph = 0;
    tcs.pend = 0;
    tcs.abort = abort;

    // operand region starts finite (K padding of A meets zeros of B)
    for (int i = tid; i < S::XY_SIZE; i += NT) smf[S::OFF_XY + i] = 0.f;
    for (int i = tid; i < T * T; i += NT) {
        const int u = i / T, s = i % T;
        zin[8 * u + s] = P.zinv[i];
    }
    if (tid == 0) {
        *wlimit = P.wait_limit;
        *abort = 0;
        *dirty = 0;
        for (int b = 0; b < 5; ++b) tc::mbar_init(tcs.bar_s + 8u * (uint32_t)b, 1);
        tc::mbar_init_fence();
    }
    if (tid < 32) tc::tmem_alloc(tc::smem_addr(tslot), S::TMEM_COLS);
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    tcs.tmem = *tslot;

    for (int64_t it = blockIdx.x; it < P.count; it += gridDim.x) {
        const int64_t e = P.elems ? (int64_t)P.elems[it] : it;
        const double* q0 = (P.runs ? P.runs[P.item_run[it]].q0 : P.q0) + e * (int64_t)(NQ * B);
        const double* ec = (P.runs ? P.runs[P.item_run[it]].econst : P.econst) + e * (int64_t)P.stride;
        // a wait of another CTA of this context gave up: skip the remaining
        // elements (the launch's results are reported as failed anyway)
        const int failed = (tid == 0 && P.status) ? *reinterpret_cast<volatile const int32_t*>(P.status) : 0;
        for (int i = tid; i < 3 * STAR_NNZ; i += NT) sh[i] = (float)ec[i];
        for (int i = tid; i < T * T; i += NT) zuf[8 * (i / T) + i % T] = (float)ec[ec_zinv(N) + i];
        const double* scal = ec + 3 * STAR_NNZ + T * T;
        const float gcoup = (float)scal[1];
        const double dt = scal[2];
        // Q = Alg3_f32(b0), b0[p, l, u] = (S^{-1} w)_u q0[p, l]
        for (int i = tid; i < NQ * B; i += NT) {
            const float v = (float)q0[i];
            float* row = W + (i / B) * QS + (i % B) * T;
#pragma unroll
            for (int u = 0; u < T; ++u) row[u] = (float)((2 * u + 1) * ((u & 1) ? -1 : 1)) * v;
        }
        if (failed) *abort = 1;
        __syncthreads();
        if (*abort) break;
        if (!alg3_sweep_tc<N, NT, BF>(W, sh, zuf, zin, gcoup, P, tcs)) break;
        // Q in binary64; time integration
        double* qtb = P.runs ? P.runs[P.item_run[it]].qt : P.qt;
        double* iob = P.runs ? P.runs[P.item_run[it]].iout : P.iout;
        if (qtb || iob) {
            double* qo = qtb ? qtb + e * (int64_t)QBT : nullptr;
            double* io = iob ? iob + e * (int64_t)(NQ * B) : nullptr;
            // one (p, l) row of T time modes per thread
            bool bad = false;
            for (int i = tid; i < NQ * B; i += NT) {
                const int p = i / B, l = i - (i / B) * B;
                const float* w = W + p * QS + l * T;
#pragma unroll
                for (int u = 0; u < T; ++u) {
                    bad |= (__float_as_uint(w[u]) & 0x7F800000u) == 0x7F800000u;
                    const double v = __longlong_as_double((long long)f2d_bits(w[u]));
                    if (qo) qo[(int64_t)i * T + u] = v;
                    if (io && u == 0) io[i] = dt * v;
                }
            }
            if (bad) *dirty = 1;
        }
        __syncthreads();
        // a non-finite result may have left non-finite words in the operand
        // region, where the next element's A-tile padding (multiplied by the
        // zero padding of the Khat images) would turn them into NaN: clear it
        if (*dirty) {
            for (int i = tid; i < S::XY_SIZE; i += NT) smf[S::OFF_XY + i] = 0.f;
            tc::fence_async_smem();  // before the bulk copies into the region
            __syncthreads();
            if (tid == 0) *dirty = 0;
        }
    }
    // the issuing threads' records of work not seen complete (empty unless a
    // wait gave up: every copy and commit is waited for otherwise)
    if (tid == (S::NW >= 4 ? 96 : 0)) *drain_mask = tcs.pend & 0x1Fu;
    __syncthreads();
    if (tid == 0) {
        const uint32_t mask = (tcs.pend | *drain_mask) & 0x1Fu;
        if (mask) tc_drain(tcs, mask);
    }
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0 && *abort && P.status) atomicExch(P.status, 1);
    if (tid < 32) tc::tmem_dealloc(tcs.tmem, S::TMEM_COLS);
}

template <int N, int NT_, int BF>
int launch_nr(const MixedReference& ref, const int32_t* elems, int64_t count, const double* q0, const double* econst,
              double* qt, double* iout, void* stream, const RunPtrs* runs, const int32_t* item_run) {
    using S = K2Shape<N, NT_, BF>;
    K2Params P;
    P.elems = elems;
    P.q0 = q0;
    P.econst = econst;
    P.qt = qt;
    P.iout = iout;
    P.count = count;
    P.stride = elem_const_stride(N);
    P.zinv = ref.zinv_f32;
    P.khat_tc = ref.khat_tc;
    for (int g = 0; g <= MAX_N; ++g)
        for (int j = 0; j < 3; ++j) P.tc_off[g][j] = ref.tc_off[g][j];
    P.status = ref.status;
    P.wait_limit = ref.wait_limit > 0 ? ref.wait_limit : tc::WAIT_LIMIT_CYCLES;
    P.runs = runs;
    P.item_run = item_run;
    // one CTA per element; every resident CTA holds TMEM_COLS columns of the
    // SM's 512, so the shared-memory request is raised where needed to keep
    // at most 512 / TMEM_COLS CTAs of this kernel resident on an SM (so no
    // CTA of this kernel waits for TMEM behind another one of it).  Kernels
    // of different degrees running concurrently on other streams (the
    // server's requests) can together ask for more than 512 columns; a CTA
    // then waits in tcgen05.alloc until a CTA of the other kernel exits and
    // frees its columns.  That CTA depends on nothing of this one and all of
    // its waits are bounded, so the allocation wait ends too.
    int dev = 0, sm_smem = 0, reserved = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (err != cudaSuccess) return (int)err;
    size_t smem = sizeof(float) * S::SMEM_FLOATS;
    const size_t floor_smem = (size_t)sm_smem / (512 / S::TMEM_COLS + 1) + 64;
    if (smem + (size_t)reserved < floor_smem) smem = floor_smem - (size_t)reserved;
    auto* kern = stp_mixed_kernel<N, NT_, BF>;
    err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return (int)err;
    if (count <= 0) return 0;
    const int64_t grid = count < (int64_t)(1u << 30) ? count : (int64_t)(1u << 30);
    kern<<<(unsigned)grid, S::NT, smem, (cudaStream_t)stream>>>(P);
    return (int)cudaGetLastError();
}

template <int N>
int launch_n(const MixedReference& ref, int variant, const int32_t* elems, int64_t count, const double* q0,
             const double* econst, double* qt, double* iout, void* stream, const RunPtrs* runs,
             const int32_t* item_run) {
    // the bf16 form is built for the default CTA size only
    if (ref.bf16)
        return launch_nr<N, K2Sizes<N>::NT0, 1>(ref, elems, count, q0, econst, qt, iout, stream, runs, item_run);
    if (variant != 0)
        return launch_nr<N, K2Sizes<N>::NT1, 0>(ref, elems, count, q0, econst, qt, iout, stream, runs, item_run);
    return launch_nr<N, K2Sizes<N>::NT0, 0>(ref, elems, count, q0, econst, qt, iout, stream, runs, item_run);
}

}  // namespace

int launch_stp_mixed(const MixedReference& ref, int refine, const int32_t* elems, int64_t count, const double* q0,
                     const double* econst, double* qt, double* iout, double* qend, void* stream, int variant, const RunPtrs* runs,
                     const int32_t* item_run) {
    if (refine == 1)
        return launch_stp_direct(*ref.base, true, true, ref.status, ref.wait_limit, elems, count, q0, econst, qt, iout,
                                 qend, stream, variant, runs, item_run);
    if (refine == 2)
        return launch_stp_direct(*ref.base, false, true, nullptr, 0, elems, count, q0, econst, qt, iout, qend, stream,
                                 variant, runs, item_run);
    switch (ref.base->N) {
        case 1: return launch_n<1>(ref, variant, elems, count, q0, econst, qt, iout, stream, runs, item_run);
        case 2: return launch_n<2>(ref, variant, elems, count, q0, econst, qt, iout, stream, runs, item_run);
        case 3: return launch_n<3>(ref, variant, elems, count, q0, econst, qt, iout, stream, runs, item_run);
        case 4: return launch_n<4>(ref, variant, elems, count, q0, econst, qt, iout, stream, runs, item_run);
        case 5: return launch_n<5>(ref, variant, elems, count, q0, econst, qt, iout, stream, runs, item_run);
        case 6: return launch_n<6>(ref, variant, elems, count, q0, econst, qt, iout, stream, runs, item_run);
        default: return (int)cudaErrorInvalidValue;
    }
}

}  // namespace poro
