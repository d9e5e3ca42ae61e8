// ks_steady.cuh -- the settled path of time-invariant models (nx <= 8).
//
// With constant parameters the covariances of Theorems 1 and 2 do not depend
// on the measurements: P_k follows from the matrix parts (A, C, J) of the
// Lemma 3 element alone, and P_k -> P as the element powers' A_{2^i} -> 0.
// Doubling Lemma 4 on one element (the structure-preserving doubling of the
// Riccati equation, Anderson 1978) gives a^(2^i) in i combines, and
//   * i doublings give the fixed point P, its gain K and Phi = (I - K H) F;
//   * the transient is exact in closed form: with O_n = sum_{j<n} (Phi^j)^T
//     F^T H^T S^{-1} H F Phi^j and D_0 = P_1 - P,
//     P_{1+k} = P + D_k,  D_k = Phi^k (I + D_0 O_k)^{-1} D_0 (Phi^k)^T,
//     and a row with n later measurements has the smoothed covariance
//     (I - P O_n) (I + D_k O_n)^{-1} P_k: a product, since the difference from
//     P_k loses the digits by which a wide prior's P_k exceeds it (Wiener
//     velocity, q = r = 1, P_0 = 1000 I: 1.4e-4 off by that difference, 1.4e-5
//     in the scans, 9e-7 here).  The tables Phi^n, O_n of the first
//     128 n (the head of a sequence, and its end) take log2 levels of plain
//     products and each row one inverse, with no scan over the rows;
//   * after the head every covariance is P, every gain constant, and only the
//     means are left: m_k = F m_{k-1} + u + K e_k, whose chunks compose with
//     the powers of one matrix Phi = (I - K H) F, and, in the adjoint form of
//     Bryson and Frazier (1963), s_k = m_k + P_k l_k with
//     l_k = Phi^T l_{k+1} + F^T H^T S^{-1} e_{k+1};
//   * Phi^256 is negligible, so a block computes its rows from a window that
//     starts 256 steps earlier and ends 256 steps later: no block waits for
//     another one.
// The plan (ks_steady_kernels.cuh::plan_body, in the preparation kernel) builds
// the powers and checks that this holds for the model: every doubling combine
// well conditioned (the estimate below the refinement threshold), the
// transient of the actual P_1 below an ulp of P after 128 steps, and |Phi^256|
// negligible in units of the posterior sd.  A model that does not pass, and a
// sequence that meets a non-finite mean, goes through the general scans: the
// call launches them too, and they return at once unless the header word
// HDR_GENERAL (or a bad offsets table) asks for them.
//
// What bounds it: the moments are written once (168 B/step at nx = 4 with the
// measurements), the arithmetic is ~140 FMAs per step instead of ~1100, and
// the constant covariance rows go out as bulk copies of a shared-memory
// pattern, so a long call sits on the HBM writes.  Measured per call, the
// scans before and this after: nx = 4, 2^20 steps 229 -> 70 us (2.6 TB/s of the
// 6.8 a copy reaches; the rest is the plan's and the head's latency, 13 and 20
// us); 1024 steps 50 -> 41 us; nx = 6, 100003 steps filtered 177 -> 59 us; 24 nx
// = 8 sequences 1071 -> 217 us; 4096 mixed sequences 5.4 -> 1.0 ms.  Every length
// takes it: at 1024 steps it is the plan and one block, still less than the
// scans.  A head of 128 rows: one thread per row, seven doublings; 2048-row
// windows give 16 steps per thread, a quarter of them halo.
#pragma once

#include "ks_scan.cuh"
#include "ks_window.h"

namespace ks {

constexpr int kStLev = 7;                         // doublings to 128 steps
constexpr int kStPow = 5;                         // Phi^16 .. Phi^256
static_assert(kStHead == 1 << kStLev && (kStCH << (kStPow - 1)) == kStHalo, "levels");

// Thresholds of the settled check.  kStCovTol: the transient left in P, one
// FP32 ulp of it.  A window's means start from a guess whose distance from the
// truth, in posterior sd, is like that of every other chunk's guess, which the
// block has at hand: |Phi^256| times the largest of them has to stay below
// kStMeanTol sd (the same for the adjoint at the window's end), and the plan
// asks for kStPowTol before any measurement is looked at.
constexpr float kStCovTol = 1.2e-7f;              // 2^-23
constexpr float kStMeanTol = 2.4e-7f;             // 2^-22
constexpr float kStPowTol = 9.5e-7f;              // 2^-20

// From a start known far better than P (a known initial state), P + D_k would
// leave P_k the rounding of P: below an eighth of it in some variance the head
// takes P_1 through the element powers of the bits of k instead, sums of
// non-negative parts, up to seven inverses for
// one: 5 us more at nx = 4 (1000 steps, P_0 = 1e-6 I: 63 -> 68 us, the scans 90), and
// the filtered variances 4.4e-6 -> 2.4e-7 off (q = r = 1, dt = 0.1, P_0 = 1e-4 I).
constexpr float kStNarrow = 0.125f;

template <int N, int M>
struct alignas(16) SteadyCore {
    // what every window needs
    float F[N * N], Ph[N * N], H[M * N], K[N * M], B[N * M], Lf[N * M], u[N], d[M];
    float Pf[N * N], Ps[N * N];                   // settled filtered and smoothed covariance
    float FP[kStPow][N * N];                      // Phi^(16 2^i)
    float sd[N], rsd[N], nphi, ndual;             // sqrt(P_aa), 1 / it; |Phi^256| and |Phi^256^T| in these units
    int ok;
    // what the head and the end of a sequence need besides
    alignas(16) float W[sym_size(N)], On[sym_size(N)];   // F^T H^T S^-1 H F; O_128
    float Q[sym_size(N)], R[sym_size(M)], C1[sym_size(N)], b1[N];
    int narrow;                                   // P_1 lies far below P somewhere: see kStNarrow
};

// A plan in memory: what the blocks copy, and the element powers a^(2^i).
template <int N, int M>
struct alignas(16) SteadyPlan : SteadyCore<N, M> {
    float EA[kStLev][N * N], EC[kStLev][sym_size(N)], EJ[kStLev][sym_size(N)];
};

// Arguments of the preparation with the plan: one block per sequence.
template <int N, int M>
struct PlanArgs {
    const float *F, *u, *Q, *H, *d, *R;
    const double *m0, *P0;
    const float* y;
    ModelConst<N, M>* out;
    uint32_t* status;
    uint32_t* zero = nullptr;                  // words the scans want zeroed
    int nzero = 0;
    const int64_t* off = nullptr;              // first steps [B + 1]; null: one sequence of T steps
    int B = 1;
    int64_t T = 0;
    const uint32_t* first_tile = nullptr;
    BlockCoef<N, M>* coef = nullptr;           // block-fold coefficients for the general scans, steps ch
    int ch = 0;
    SteadyPlan<N, M>* plan = nullptr;
};

// Arguments of the settled path.
template <int N, int M>
struct SteadyArgs {
    const SteadyPlan<N, M>* plan;   // one per sequence
    const int64_t* off;             // first steps [B + 1]; null: one sequence of T steps
    int B;
    int64_t T;
    const float* y;
    float *fm, *fc, *sm, *sc;       // sm, sc null: the filter alone
    int keep;                       // 0: fm, fc are scratch (only the head's rows are written)
    uint32_t* status;
};

// Blocks of a launch over B sequences of T steps in all: sequence b has the
// slots from off[b] / kStOut + b on, at least as many as its windows.
inline int64_t steady_blocks(int64_t T, int B) { return T / kStOut + B; }

// Host launches (instantiated for every size in ks_steady*.cu).
template <int N, int M>
int launch_plan_kernel(const PlanArgs<N, M>& g, cudaStream_t st);
template <int N, int M>
int launch_steady_kernel(const SteadyArgs<N, M>& g, cudaStream_t st);

}  // namespace ks
