// ks_loglik.cu -- marginal log-likelihood by one extra parallel pass over the
// filtered moments (Section III-C: Theorem 1's prefix also carries p(y_1:k)).
//
// p(y_1:n) = prod_k p(y_k | y_1:k-1) and, for the linear/Gaussian model,
//   p(y_k | y_1:k-1) = N(y_k; mu_k, S_k),  mu_k = G xbar_{k-1} + c0,
//   S_k = G P_{k-1} G^T + S0,  G = H F,  S0 = H Q H^T + R,  c0 = H u + d,
// with (xbar_{k-1}, P_{k-1}) the filtered posterior of the previous step and
// (m0, P0) in place of it at k = 1.  One thread (nx <= 6) or lane group (nx >=
// 8) per step forms S_k, then one thread its factor, the quadratic form and log
// det S_k; the per-step values are written in FP32 and summed in FP64 (block
// sums, one atomic per block).
#include <cuda_runtime.h>

#include "../../include/ks.h"

namespace ks {
namespace {

constexpr int kLLThreads = 128;
constexpr double kLog2Pi = 1.8378770664093453;

template <int N, int M>
struct LLConst {
    float G[M * N];      // H F
    float S0[M * M];     // H Q H^T + R
    float c0[M];         // H u + d
};

template <int N, int M>
__device__ void build_llconst(const float* __restrict__ F, const float* __restrict__ u, const float* __restrict__ Q,
                              const float* __restrict__ H, const float* __restrict__ d, const float* __restrict__ R,
                              LLConst<N, M>& c, float* HQ) {
    const int t = threadIdx.x, nt = blockDim.x;
    for (int e = t; e < M * N; e += nt) {
        const int q = e / N, a = e % N;
        float g = 0.f, h = 0.f;
        for (int k = 0; k < N; ++k) {
            g = fmaf(H[q * N + k], F[k * N + a], g);
            h = fmaf(H[q * N + k], Q[k * N + a], h);
        }
        c.G[e] = g;
        HQ[e] = h;
    }
    for (int q = t; q < M; q += nt) {
        float s = d ? d[q] : 0.f;
        if (u)
            for (int k = 0; k < N; ++k) s = fmaf(H[q * N + k], u[k], s);
        c.c0[q] = s;
    }
    __syncthreads();
    for (int e = t; e < M * M; e += nt) {
        const int q = e / M, p = e % M;
        float s = 0.5f * (R[q * M + p] + R[p * M + q]);
        for (int k = 0; k < N; ++k) s = fmaf(HQ[q * N + k], H[p * N + k], s);
        c.S0[e] = s;
    }
    __syncthreads();
}

// log N(r; 0, S) for an M x M SPD matrix S (row-major, lower triangle read);
// returns false when the Cholesky factorisation fails.
template <int M, class Real>
__device__ bool log_gauss(Real (&S)[M][M], Real (&r)[M], Real& out) {
    Real ld = 0;
#pragma unroll
    for (int j = 0; j < M; ++j) {
        Real s = S[j][j];
#pragma unroll
        for (int k = 0; k < j; ++k) s -= S[j][k] * S[j][k];
        if (!(s > Real(0))) return false;
        const Real l = sqrt(s);
        S[j][j] = l;
        ld += log(l);
#pragma unroll
        for (int i = j + 1; i < M; ++i) {
            Real t = S[i][j];
#pragma unroll
            for (int k = 0; k < j; ++k) t -= S[i][k] * S[j][k];
            S[i][j] = t / l;
        }
    }
    Real q = 0;                                     // || L^{-1} r ||^2
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Real t = r[i];
#pragma unroll
        for (int k = 0; k < i; ++k) t -= S[i][k] * r[k];
        r[i] = t / S[i][i];
        q += r[i] * r[i];
    }
    out = Real(-0.5) * (q + Real(M) * Real(kLog2Pi)) - ld;
    return true;
}

// The same from the lower triangle of S in packed rows and the residual r, in
// FP64 throughout and without square roots: S = L D L^T.  Pivots are paired
// under one logarithm (a product of two stays in range).
template <int M, class In>
__device__ bool log_gauss_ldl(const In* __restrict__ Sp, const In* __restrict__ r, double& out) {
    static_assert(M % 2 == 0, "paired pivots");
    double L[M][M], z[M], q = 0.0, ld = 0.0, pair = 1.0;   // below the diagonal: L D, then L
#pragma unroll
    for (int j = 0; j < M; ++j) {
        double s = Sp[j * (j + 1) / 2 + j], t = r[j];
#pragma unroll
        for (int k = 0; k < j; ++k) {
            double l = Sp[j * (j + 1) / 2 + k];
#pragma unroll
            for (int p = 0; p < k; ++p) l = fma(-L[j][p], L[k][p], l);
            L[j][k] = l;                                   // L_jk D_k
            const double w = l * L[k][k];                  // L_jk
            s = fma(-w, l, s);
            t = fma(-w, z[k], t);
            L[k][j] = w;
        }
        if (!(s > 0.0)) return false;
#pragma unroll
        for (int k = 0; k < j; ++k) L[j][k] = L[k][j];
        L[j][j] = 1.0 / s;
        z[j] = t;
        q = fma(t * t, L[j][j], q);
        pair *= s;
        if (j & 1) {
            ld += log(pair);
            pair = 1.0;
        }
    }
    out = -0.5 * (q + M * kLog2Pi + ld);
    return true;
}

// log p(y_1) from the prior, in FP64.
template <int N, int M>
__device__ bool prior_density(const LLConst<N, M>& c, const double* __restrict__ m0, const double* __restrict__ P0,
                              const float* __restrict__ y, double& val) {
    double S[M][M], r[M];
    for (int q = 0; q < M; ++q) {
        double gm = c.c0[q];
        for (int a = 0; a < N; ++a) gm += (double)c.G[q * N + a] * m0[a];
        r[q] = (double)y[q] - gm;
    }
    for (int q = 0; q < M; ++q) {
        double gp[N];
        for (int b = 0; b < N; ++b) {
            double s = 0.0;
            for (int a = 0; a < N; ++a) s += (double)c.G[q * N + a] * P0[a * N + b];
            gp[b] = s;
        }
        for (int p = 0; p <= q; ++p) {
            double s = c.S0[q * M + p];
            for (int b = 0; b < N; ++b) s += gp[b] * (double)c.G[p * N + b];
            S[q][p] = s;
        }
    }
    double v = 0.0;
    const bool ok = log_gauss<M, double>(S, r, v);
    val = v;
    return ok;
}

// Store a step's value; FP64 block sum, one atomic per block; failures.
template <int THREADS>
__device__ void finish(int64_t k, int64_t T, double val, bool bad, float* ll, double* total, uint32_t* bad_out,
                       double* red) {
    if (k < T) {
        if (ll) ll[k] = (float)val;
        bad = bad || !isfinite(val);
    }
    for (int off = 16; off > 0; off >>= 1) val += __shfl_down_sync(0xffffffffu, val, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = val;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < THREADS / 32; ++i) s += red[i];
        if (total) atomicAdd(total, s);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(bad_out, 1u);
}

template <int N, int M>
__global__ void __launch_bounds__(kLLThreads) loglik_kernel(
    const float* __restrict__ F, const float* __restrict__ u, const float* __restrict__ Q,
    const float* __restrict__ H, const float* __restrict__ d, const float* __restrict__ R,
    const double* __restrict__ m0, const double* __restrict__ P0, const float* __restrict__ y, int64_t T,
    const float* __restrict__ fmean, const float* __restrict__ fcov, float* __restrict__ ll,
    double* __restrict__ total, uint32_t* __restrict__ bad_out) {
    __shared__ LLConst<N, M> c;
    __shared__ float HQ[M * N];
    __shared__ double red[kLLThreads / 32];
    build_llconst<N, M>(F, u, Q, H, d, R, c, HQ);
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double val = 0.0;
    bool bad = false;
    if (k == 0) {
        bad = !prior_density<N, M>(c, m0, P0, y, val);
    } else if (k < T) {
        const float* xb = fmean + (k - 1) * N;
        const float* P = fcov + (k - 1) * N * N;
        float S[M][M], r[M];
#pragma unroll
        for (int q = 0; q < M; ++q) {
            float gm = c.c0[q];
#pragma unroll 8
            for (int a = 0; a < N; ++a) gm = fmaf(c.G[q * N + a], __ldg(xb + a), gm);
            r[q] = __ldg(y + k * M + q) - gm;
        }
#pragma unroll 1
        for (int q = 0; q < M; ++q) {
            float gp[N];
#pragma unroll
            for (int b = 0; b < N; ++b) gp[b] = 0.f;
#pragma unroll 4
            for (int a = 0; a < N; ++a) {
                const float g = c.G[q * N + a];
#pragma unroll
                for (int b = 0; b < N; ++b) gp[b] = fmaf(g, __ldg(P + a * N + b), gp[b]);
            }
#pragma unroll
            for (int p = 0; p < M; ++p) {
                if (p > q) break;
                float s = c.S0[q * M + p];
#pragma unroll
                for (int b = 0; b < N; ++b) s = fmaf(gp[b], c.G[p * N + b], s);
                S[q][p] = s;
            }
        }
        float v;
        bad = !log_gauss<M, float>(S, r, v);
        val = v;
    }
    finish<kLLThreads>(k, T, val, bad, ll, total, bad_out, red);
}

// nx >= 8: N lanes per step form S_k and y_k - mu_k (lane b holds column b of
// P, so a row is one coalesced read), kTileSteps steps a block; then one thread
// per step takes the step's density in FP64.  One thread per step, its P a row
// of 4 N^2 bytes of its own and step 0 in FP64 on one of them, was bound by
// uncoalesced loads and, in short calls, by step 0: 2128 us at nx = 32, 62861
// steps (849 us at 3001), 261 us at nx = 8, 262144 steps; this: 187 us (59 us) and
// 92 us.  At nx = 32 a warp's steps follow one another, so that a tile of 128
// keeps a short call waiting: 32 steps, 8 a warp.
// The FP64 tail (an LDL^T of the FP32 S) is there for the total: an FP32 log
// det has the same rounding error at every step of a settled filter, so the
// sum of T of them was up to 2e-8 off however long the sequence; now 7e-9 at 300
// steps and below 1e-9 from 30000 on.
constexpr int kTile = 128;                          // threads
template <int N>
constexpr int kTileSteps = N == 32 ? 32 : 128;
template <int N, int M>
__global__ void __launch_bounds__(kTile) loglik_tile_kernel(
    const float* __restrict__ F, const float* __restrict__ u, const float* __restrict__ Q,
    const float* __restrict__ H, const float* __restrict__ d, const float* __restrict__ R,
    const double* __restrict__ m0, const double* __restrict__ P0, const float* __restrict__ y, int64_t T,
    const float* __restrict__ fmean, const float* __restrict__ fcov, float* __restrict__ ll,
    double* __restrict__ total, uint32_t* __restrict__ bad_out) {
    constexpr int STEPS = kTileSteps<N>, NG = kTile / N, NE = M * (M + 1) / 2, PITCH = (NE + M) | 1;
    __shared__ LLConst<N, M> c;
    __shared__ float HQ[M * N];
    __shared__ __align__(16) float Gt[N * M];
    __shared__ float gps[NG][M][N + 1], xs[NG][N];
    __shared__ float tile[STEPS][PITCH];            // a step's S (lower triangle) and residual
    __shared__ double red[kTile / 32], gp0[M * N], first[NE + M];
    build_llconst<N, M>(F, u, Q, H, d, R, c, HQ);
    for (int e = threadIdx.x; e < M * N; e += kTile) Gt[e] = c.G[(e % M) * N + e / M];
    __syncthreads();
    const int g = threadIdx.x / N, b = threadIdx.x % N;
    const unsigned mask = N == 32 ? 0xffffffffu : ((1u << N) - 1u) << ((threadIdx.x & 31) / N * N);
    const int64_t k0 = (int64_t)blockIdx.x * STEPS;
    if (k0 == 0) {                                  // step 0, from the prior in FP64
        for (int e = threadIdx.x; e < M * N; e += kTile) {
            const int q = e / N, j = e % N;
            double s = 0.0;
#pragma unroll 8
            for (int a = 0; a < N; ++a) s += (double)Gt[a * M + q] * P0[a * N + j];
            gp0[e] = s;
        }
        __syncthreads();
        for (int e = threadIdx.x; e < NE + M; e += kTile) {
            double s;
            if (e < NE) {
                int q = 0;
                while ((q + 1) * (q + 2) / 2 <= e) ++q;
                const int p = e - q * (q + 1) / 2;
                s = c.S0[q * M + p];
#pragma unroll 8
                for (int j = 0; j < N; ++j) s += gp0[q * N + j] * (double)c.G[p * N + j];
            } else {
                const int q = e - NE;
                double gm = c.c0[q];
#pragma unroll 8
                for (int a = 0; a < N; ++a) gm += (double)c.G[q * N + a] * m0[a];
                s = (double)y[q] - gm;
            }
            first[e] = s;
        }
    }
#pragma unroll 1
    for (int i = 0; i < STEPS / NG; ++i) {
        const int64_t k = k0 + i * NG + g;
        if (k >= 1 && k < T) {                      // the same for a step's lanes
            const float* P = fcov + (k - 1) * N * N + b;
            float pa[N], acc[M];
#pragma unroll
            for (int a = 0; a < N; ++a) pa[a] = __ldg(P + a * N);
            xs[g][b] = __ldg(fmean + (k - 1) * N + b);
#pragma unroll
            for (int q = 0; q < M; ++q) acc[q] = 0.f;
#pragma unroll
            for (int a = 0; a < N; ++a)
#pragma unroll
                for (int q = 0; q < M; ++q) acc[q] = fmaf(Gt[a * M + q], pa[a], acc[q]);
#pragma unroll
            for (int q = 0; q < M; ++q) gps[g][q][b] = acc[q];   // G P
            __syncwarp(mask);
            float* out = tile[i * NG + g];
            for (int e = b; e < NE + M; e += N) {
                if (e < NE) {
                    int q = 0;
                    while ((q + 1) * (q + 2) / 2 <= e) ++q;
                    const int p = e - q * (q + 1) / 2;
                    float s = c.S0[q * M + p];
#pragma unroll 8
                    for (int j = 0; j < N; ++j) s = fmaf(gps[g][q][j], c.G[p * N + j], s);
                    out[e] = s;
                } else {
                    const int q = e - NE;
                    float gm = c.c0[q];
#pragma unroll 8
                    for (int j = 0; j < N; ++j) gm = fmaf(c.G[q * N + j], xs[g][j], gm);
                    out[e] = __ldg(y + k * M + q) - gm;
                }
            }
            __syncwarp(mask);
        }
    }
    __syncthreads();
    const int64_t k = threadIdx.x < STEPS ? k0 + threadIdx.x : T;
    double val = 0.0;
    bool bad = false;
    if (k == 0) {
        bad = !log_gauss_ldl<M>(first, first + NE, val);
    } else if (k < T) {
        bad = !log_gauss_ldl<M>(tile[threadIdx.x], tile[threadIdx.x] + NE, val);
    }
    finish<kTile>(k, T, val, bad, ll, total, bad_out, red);
}

template <int N, int M>
int launch(const ks_model* m, const float* y, int64_t T, const float* fm, const float* fc, float* ll, double* total,
           uint32_t* bad, cudaStream_t st) {
    constexpr int steps = N >= 8 ? kTileSteps<N> : kLLThreads;
    const int64_t blocks = (T + steps - 1) / steps;
    if constexpr (N >= 8)
        loglik_tile_kernel<N, M><<<(unsigned)blocks, kTile, 0, st>>>(m->F, m->u, m->Q, m->H, m->d, m->R, m->m0, m->P0,
                                                                     y, T, fm, fc, ll, total, bad);
    else
        loglik_kernel<N, M><<<(unsigned)blocks, kLLThreads, 0, st>>>(m->F, m->u, m->Q, m->H, m->d, m->R, m->m0, m->P0,
                                                                     y, T, fm, fc, ll, total, bad);
    return cudaGetLastError() == cudaSuccess ? KS_OK : KS_ECUDA;
}

}  // namespace
}  // namespace ks

extern "C" int ks_loglik(const ks_model* m, const float* y, int64_t T, const float* fmean, const float* fcov,
                         float* ll, double* total, uint32_t* status, void* stream) {
    using namespace ks;
    if (!m || !m->F || !m->Q || !m->H || !m->R || !m->m0 || !m->P0 || !y) return KS_EINVAL;
    if (m->time_varying != 0) return KS_EUNSUPPORTED;
    if (T < 1 || T > 0x7fffffffLL || (T > 1 && (!fmean || !fcov)) || !status) return KS_EINVAL;
    if (!ll && !total) return KS_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (total && cudaMemsetAsync(total, 0, sizeof(double), st) != cudaSuccess) return KS_ECUDA;
    if (cudaMemsetAsync(status, 0, sizeof(uint32_t), st) != cudaSuccess) return KS_ECUDA;
    const int nx = m->nx, ny = m->ny;
    if (nx == 2 && ny == 1) return launch<2, 1>(m, y, T, fmean, fcov, ll, total, status, st);
    if (nx == 4 && ny == 2) return launch<4, 2>(m, y, T, fmean, fcov, ll, total, status, st);
    if (nx == 6 && ny == 3) return launch<6, 3>(m, y, T, fmean, fcov, ll, total, status, st);
    if (nx == 8 && ny == 4) return launch<8, 4>(m, y, T, fmean, fcov, ll, total, status, st);
    if (nx == 32 && ny == 8) return launch<32, 8>(m, y, T, fmean, fcov, ll, total, status, st);
    return KS_EUNSUPPORTED;
}
