// ks_steady32.cuh -- the settled path (ks_steady.cuh) at nx = 32, one sequence.
//
// The same algebra with one warp per vector recursion (lane a holds component
// a) and thread blocks for the 32 x 32 products:
//   plan     the doubling to P, the powers Phi^(2^i), O_(2^i) (block 0) and the
//            FP64 first element beside it (block 1: at FP64 rates it is as long
//            as the doubling);
//   rows     block k < 128: head row k's P_k, smoothed covariance and the next
//            row's gain, and the sequence's k-th row from the end, each from the
//            tables' closed forms (its Phi^k, O_k from the bits of k); the other
//            blocks run the chunks of 32 rows once from a guess and fill the
//            constant filtered covariances;
//   forward  a chunk's true start is a sum over the eight chunks before it
//            (Phi^256 is negligible), so no chunk waits for another; the means,
//            the chunk's adjoint from zero, the constant smoothed covariances;
//   reverse  the same for the adjoint, and the smoothed means.
// The head's own rows (gains of their own) run in eight chunks of 16 in one
// block, joined by Psi = Phi^16 (I + D_a O_16)^{-1}, the closed form of their
// transition.  A general Kalman combine costs ~10 products and a pivoted
// inverse per step (1.08 MFLOP); here a step is three matrix-vector products,
// and a long call sits on writing the 8.4 KB of moments per step.
#pragma once

#include "ks_impl.cuh"

namespace ks {

constexpr int kS32Head = 128;       // rows with gains of their own
constexpr int kS32Chunk = 32;       // rows of a chunk
constexpr int kS32Back = 8;         // chunks that reach 256 rows
// Head and end rows apart need 256 rows; shorter sequences go through the
// scans.  At the line, 256 steps: 2262 us in the scans, 213 here; 65536
// steps 3406 -> 350 us.
constexpr int kS32MinT = 256;

struct Plan32 {
    float F[1024], Ph[1024], PhT[1024], P32[1024], P32T[1024], Pf[1024], Ps[1024];
    float PW[7][1024], OW[8][1024];                 // Phi^(2^i), O_(2^i)
    float EA[7][1024], EC[7][1024], EJ[7][1024];    // the element powers a^(2^i), for a narrow start (kStNarrow)
    float Q[1024], C1[1024];
    float H[256], K[256], B[256], Lf[256], HF[256], R[64], u[32], d[8], b1[32], sd[32], rsd[32];
    float nphi, ndual, nA;
    int ok, ok1;
};

// Scratch in the workspace beside the plan: the head rows' gains, B = F^T H^T
// S^{-1} and Psi, per-chunk misses of both recursions, innovations.
struct Scratch32 {
    Plan32* plan;
    float *Kr, *Br, *Psi, *miss, *mu, *eps;
};
inline int64_t s32_chunks(int64_t T) { return (T - kS32Head + kS32Chunk - 1) / kS32Chunk; }
inline size_t s32_bytes(int64_t T) {
    if (T < kS32MinT) return 0;
    return align_up(sizeof(Plan32), 256) +
           4 * ((size_t)kS32Head * 512 + 8 * 1024 + (size_t)s32_chunks(T) * 64 + 8 * (size_t)T) + 256;
}
inline Scratch32 s32_at(void* p, int64_t T) {
    Scratch32 s;
    s.plan = static_cast<Plan32*>(p);
    float* f = reinterpret_cast<float*>(static_cast<char*>(p) + align_up(sizeof(Plan32), 256));
    s.Kr = f; f += kS32Head * 256;
    s.Br = f; f += kS32Head * 256;
    s.Psi = f; f += 8 * 1024;
    s.miss = f; f += s32_chunks(T) * 32;
    s.mu = f; f += s32_chunks(T) * 32;
    s.eps = f;
    return s;
}

struct Args32 {
    const float *F, *u, *Q, *H, *d, *R;
    const double *m0, *P0;
    const float* y;
    int64_t T;
    ModelConst<32, 8>* mconst;
    uint32_t* status;
    uint32_t* zero;
    int nzero;
    float *fm, *fc, *sm, *sc;   // sm, sc null: the filter alone
    int keep;                   // 0: fc is scratch (only the head's rows are written)
    Scratch32 s;
};

// Launches the four kernels (ks_steady32.cu); T >= kS32MinT.
int launch_steady32_plan(const Args32& g, cudaStream_t st);
int launch_steady32(const Args32& g, cudaStream_t st);

}  // namespace ks
