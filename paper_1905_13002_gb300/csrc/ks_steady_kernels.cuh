// ks_steady_kernels.cuh -- device code of the settled path (ks_steady.cuh).
#pragma once

#include <cstddef>
#include <type_traits>

#include "ks_impl.cuh"

namespace ks {

// ---------------------------------------------------------------- plan
// Gauss-Jordan inverse with partial pivoting by one warp: lane c < 2N holds
// column c of [X | I].  Returns false on a failed pivot; cond = the 1-norm
// condition number.
template <int N>
KS_DEV bool warp_inverse(const float* __restrict__ X, float* __restrict__ Xi, int lane, float& cond) {
    static_assert(2 * N <= 32, "one lane per column of [X | I]");
    float col[N];
    float nrm = 0.f;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        col[r] = lane < N ? X[r * N + lane] : (lane - N == r ? 1.f : 0.f);
        nrm += fabsf(col[r]);
    }
    if (lane >= N) nrm = 0.f;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        float pc[N];
#pragma unroll
        for (int r = 0; r < N; ++r) pc[r] = __shfl_sync(0xffffffffu, col[r], k);
        int p = k;
        float best = fabsf(pc[k]);
#pragma unroll
        for (int r = k + 1; r < N; ++r) {
            const float v = fabsf(pc[r]);
            if (v > best) { best = v; p = r; }
        }
#pragma unroll
        for (int r = k + 1; r < N; ++r) {
            const bool s = (p == r);
            const float a = pc[k], b = col[k];
            pc[k] = s ? pc[r] : a;
            pc[r] = s ? a : pc[r];
            col[k] = s ? col[r] : b;
            col[r] = s ? b : col[r];
        }
        ok = ok && (best > 1e-30f) && isfinite(best);
        col[k] *= __frcp_rn(pc[k]);
#pragma unroll
        for (int r = 0; r < N; ++r)
            if (r != k) col[r] = fmaf(-pc[r], col[k], col[r]);
    }
    float ni = 0.f;
#pragma unroll
    for (int r = 0; r < N; ++r) ni += fabsf(col[r]);
    if (lane < N || lane >= 2 * N) ni = 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nrm = fmaxf(nrm, __shfl_xor_sync(0xffffffffu, nrm, o));
        ni = fmaxf(ni, __shfl_xor_sync(0xffffffffu, ni, o));
    }
    cond = nrm * ni;
    if (lane >= N && lane < 2 * N) {
#pragma unroll
        for (int r = 0; r < N; ++r) Xi[r * N + lane - N] = col[r];
    }
    return ok;
}

template <int N, int M>
struct PlanSmem {
    float A[2][N * N], C[2][N * N], J[2][N * N];
    float Mx[N * N], Mi[N * N], X[N * N], W[N * N], V[N * N], Y[N * N], Z[N * N];
    float HP[M * N], S[M * M], Si[M * M], Hh[M * M], Hi[M * M], K[N * M];
    float sd[N];
    int ok, settled, narrow;
};

// Threads of the preparation with the plan: warps 0-3 the FP32 constants and
// the plan's chain, warps 4-6 the FP64 first element beside it.
constexpr int kChainThreads = 128;
constexpr int kPlanThreads = kChainThreads + kFirstThreads;
KS_DEV void chain_sync() { asm volatile("bar.sync 2, %0;" ::"n"(kChainThreads) : "memory"); }

// Largest row sum of |X| in units of sd, max_a sum_b |X_ab| sd_b / sd_a, or
// the largest column sum of the same scaled matrix (one warp).
template <int N, bool COL = false>
KS_DEV float scaled_norm(const float* __restrict__ X, const float* __restrict__ sd, int lane) {
    float s = 0.f;
    if (lane < N) {
        for (int b = 0; b < N; ++b)
            s = COL ? fmaf(fabsf(X[b * N + lane]), 1.f / sd[b], s) : fmaf(fabsf(X[lane * N + b]), sd[b], s);
        s = COL ? s * sd[lane] : s / sd[lane];
        if (!(s < 1e18f)) s = 1e18f;   // also when sd is not a number
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = fmaxf(s, __shfl_xor_sync(0xffffffffu, s, o));
    return s;
}

template <int N>
KS_DEV float dot_rr(const float* a, const float* b) {   // row . row
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < N; ++c) s = fmaf(a[c], b[c], s);
    return s;
}
template <int N>
KS_DEV float dot_rc(const float* a, const float* b) {   // row . column (stride N)
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < N; ++c) s = fmaf(a[c], b[c * N], s);
    return s;
}
template <int N>
KS_DEV float dot_cc(const float* a, const float* b) {   // column . column (stride N)
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < N; ++c) s = fmaf(a[c * N], b[c * N], s);
    return s;
}

// The element of Lemma 3 doubled kStLev times, by the chain's threads, from the
// FP32 constants mc; returns the buffer of the last one.  One output entry per
// thread and stage; a doubling combine is four stages (M, M^-1 by one warp, the
// three products with M^-1, the outer products).  powers: null, or where the
// elements before each doubling go.
template <int N, int M>
KS_DEV int element_powers(PlanSmem<N, M>& s, const ModelConst<N, M>& mc, SteadyPlan<N, M>* __restrict__ powers) {
    constexpr int NN = N * N, NT = kChainThreads;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    for (int e = t; e < NN; e += NT) {
        const int a = e / N, b = e % N;
        s.A[0][e] = mc.A[e];
        s.C[0][e] = mc.C[sidx(a, b)];
        float j = 0.f;
        for (int q = 0; q < M; ++q) j = fmaf(mc.U[q * N + a], mc.U[q * N + b], j);
        s.J[0][e] = j;
    }
    chain_sync();
    int cur = 0;
#pragma unroll 1
    for (int lev = 0; lev < kStLev; ++lev, cur ^= 1) {
        const float *A = s.A[cur], *C = s.C[cur], *J = s.J[cur];
        float *A2 = s.A[cur ^ 1], *C2 = s.C[cur ^ 1], *J2 = s.J[cur ^ 1];
        for (int e = t; e < NN; e += NT) {
            const int a = e / N, b = e % N;
            s.Mx[e] = dot_rr<N>(C + a * N, J + b * N) + (a == b ? 1.f : 0.f);
        }
        chain_sync();
        if (warp == 0) {
            float cond;
            const bool ok = warp_inverse<N>(s.Mx, s.Mi, lane, cond);
            if (lane == 0 && !(ok && cond <= kRefineCond)) s.ok = 0;
        } else if (powers != nullptr) {
            for (int e = t - 32; e < NN; e += NT - 32) {
                const int a = e / N, b = e % N;
                powers->EA[lev][e] = A[e];
                if (b <= a) {
                    powers->EC[lev][sidx(a, b)] = C[e];
                    powers->EJ[lev][sidx(a, b)] = J[e];
                }
            }
        }
        chain_sync();
        for (int e = t; e < 3 * NN; e += NT) {
            const int k = e / NN, f = e % NN, a = f / N, b = f % N;
            if (k == 0) s.X[f] = dot_rc<N>(A + a * N, s.Mi + b);           // A M^-1
            else if (k == 1) s.W[f] = dot_rr<N>(s.Mi + a * N, C + b * N);  // M^-1 C
            else s.V[f] = dot_cc<N>(s.Mi + a, J + b);                      // M^-T J
        }
        chain_sync();
        for (int e = t; e < 3 * NN; e += NT) {
            const int k = e / NN, f = e % NN, a = f / N, b = f % N;
            if (k == 0) A2[f] = dot_rc<N>(s.X + a * N, A + b);             // A M^-1 A
            else if (k == 1) s.Y[f] = dot_rc<N>(A + a * N, s.W + b);
            else s.Z[f] = dot_rc<N>(s.V + a * N, A + b);
        }
        chain_sync();
        for (int e = t; e < 2 * NN; e += NT) {                             // lower triangles, mirrored
            const int k = e / NN, f = e % NN, a = f / N, b = f % N;
            if (b > a) continue;
            float* D = k == 0 ? C2 : J2;
            const float v = k == 0 ? C[f] + dot_rr<N>(s.Y + a * N, A + b * N) : J[f] + dot_cc<N>(A + a, s.Z + b);
            D[f] = v;
            D[b * N + a] = v;
        }
        chain_sync();
    }
    return cur;
}

// The plan of one model, by the chain's threads, from the FP32 constants mc and
// the inputs in shared memory.
template <int N, int M, class PS>
KS_DEV void plan_body(PlanSmem<N, M>& s, const PS& p, const ModelConst<N, M>& mc, SteadyPlan<N, M>* __restrict__ out) {
    constexpr int NN = N * N, NT = kChainThreads;
    static_assert(NN <= 64 && N * M <= 32, "entries per warp of the single-warp stages");
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    for (int e = t; e < NN; e += NT) out->F[e] = mc.F[e];
    for (int e = t; e < M * N; e += NT) out->H[e] = p.H[e / N][e % N];
    for (int e = t; e < sym_size(N); e += NT) out->Q[e] = mc.Q[e];
    for (int e = t; e < sym_size(M); e += NT) {
        int a, b;
        tri_rc(e, a, b);
        out->R[e] = 0.5f * (p.R[a][b] + p.R[b][a]);
    }
    for (int e = t; e < N; e += NT) out->u[e] = mc.u[e];
    for (int e = t; e < M; e += NT) out->d[e] = p.d[e];
    const int cur = element_powers<N, M>(s, mc, nullptr);
    // ---- settled covariances, gains and Phi
    const float *A = s.A[cur], *P = s.C[cur], *J = s.J[cur];
    float *FPm = s.X, *Pm = s.Y, *Ph0 = s.A[cur ^ 1];
    for (int e = t; e < NN; e += NT) {
        const int a = e / N, b = e % N;
        FPm[e] = dot_rc<N>(mc.F + a * N, P + b);
        s.Mx[e] = dot_rr<N>(P + a * N, J + b * N) + (a == b ? 1.f : 0.f);
        out->Pf[e] = P[e];
    }
    for (int e = t; e < M * M; e += NT) s.Hh[e] = dot_rr<N>(&p.H[e / M][0], &p.H[e % M][0]);
    chain_sync();
    if (t < NN) {
        const int a = t / N, b = t % N, hi = a >= b ? a : b, lo = a >= b ? b : a;
        Pm[t] = dot_rr<N>(FPm + hi * N, mc.F + lo * N) + mc.Q[sidx(a, b)];
    }
    if (warp == 2) {
        float cond;
        const bool ok = warp_inverse<N>(s.Mx, s.Mi, lane, cond);
        if (lane == 0 && !(ok && cond <= kRefineCond)) s.ok = 0;
    } else if (warp == 3) {
        float cond;
        const bool ok = warp_inverse<M>(s.Hh, s.Hi, lane, cond);
        __syncwarp();
        if (!(ok && cond <= kRefineCond) && lane < M * M) s.Hi[lane] = 0.f;   // no lift: the guess is zero
    }
    chain_sync();
    if (warp == 0) {   // S, its inverse, the gains and Phi
        if (lane < M * N) s.HP[lane] = dot_rc<N>(&p.H[lane / N][0], Pm + lane % N);
        __syncwarp();
        if (lane < M * M) {
            const int a = lane / M, b = lane % M;
            s.S[lane] = dot_rr<N>(s.HP + a * N, &p.H[b][0]) + 0.5f * (p.R[a][b] + p.R[b][a]);
        }
        __syncwarp();
        float cond;
        const bool ok = warp_inverse<M>(s.S, s.Si, lane, cond);
        if (lane == 0 && !(ok && cond <= kRefineCond)) s.ok = 0;
        __syncwarp();
        float kv = 0.f, bv = 0.f;
        if (lane < N * M) {
            const int a = lane / M, q = lane % M;
            for (int r = 0; r < M; ++r) {
                kv = fmaf(s.HP[r * N + a], s.Si[r * M + q], kv);
                bv = fmaf(p.HF[r][a], s.Si[r * M + q], bv);
            }
        }
        __syncwarp();
        if (lane < N * M) {
            s.K[lane] = kv;
            s.HP[lane] = bv;                         // B, [N][M]
            out->K[lane] = kv;
            out->B[lane] = bv;
        }
        __syncwarp();
        for (int e = lane; e < NN; e += 32) {
            const int a = e / N, b = e % N;
            if (b <= a) {
                float w = 0.f;
                for (int q = 0; q < M; ++q) w = fmaf(s.HP[a * M + q], p.HF[q][b], w);
                out->W[sidx(a, b)] = w;
            }
            float v = mc.F[e];
            for (int q = 0; q < M; ++q) v = fmaf(-s.K[a * M + q], p.HF[q][b], v);
            Ph0[e] = v;
            out->Ph[e] = v;
        }
    } else if (warp == 1) {
        if (lane < N * M) {   // lift H^T (H H^T)^-1
            const int a = lane / M, q = lane % M;
            float v = 0.f;
            for (int r = 0; r < M; ++r) v = fmaf(p.H[r][a], s.Hi[r * M + q], v);
            out->Lf[lane] = v;
        }
        if (lane < N) {
            const float v = sqrtf(P[lane * N + lane]);
            s.sd[lane] = v;
            out->sd[lane] = v;
            out->rsd[lane] = 1.f / v;
        }
    } else {
        for (int e = t - 64; e < NN; e += 64) {   // Ps = (I + P J)^-1 P
            const int a = e / N, b = e % N, hi = a >= b ? a : b, lo = a >= b ? b : a;
            out->Ps[e] = dot_rr<N>(s.Mi + hi * N, P + lo * N);
            if (b <= a) out->On[sidx(a, b)] = dot_cc<N>(s.Mi + a, J + b);   // (I + J P)^-1 J
        }
    }
    chain_sync();
    if (warp == 3) {   // what is left of a unit transient after 128 steps (kept for the check against P_1)
        const float n = scaled_norm<N>(A, s.sd, lane);
        if (lane == 0) s.Hh[0] = n;
    }
    // ---- powers of Phi
    float *f0 = Ph0, *f1 = s.C[cur ^ 1];
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        if (t < NN) {
            const float v = dot_rc<N>(f0 + t / N * N, f0 + t % N);
            f1[t] = v;
            if (i >= 3) out->FP[i - 3][t] = v;
        }
        chain_sync();
        float* x = f0;
        f0 = f1;
        f1 = x;
    }
    if (warp == 1) {
        const float nf = scaled_norm<N>(f0, s.sd, lane);
        if (lane == 0) {
            out->nphi = nf;
            if (!(nf <= kStPowTol)) s.settled = 0;
        }
    } else if (warp == 2) {
        const float nd = scaled_norm<N, true>(f0, s.sd, lane);
        if (lane == 0) {
            out->ndual = nd;
            if (!(nd <= kStPowTol)) s.settled = 0;
        }
    }
}

// Preparation of the fused smooth calls: the model constants and the plan.  A
// single sequence whose model does not pass also gets the block fold's
// coefficients (`coef`), which only the general scans read; a segmented batch
// that folds has them built for every sequence.
template <int N, int M>
__host__ __device__ constexpr size_t plan_off() {   // PlanSmem after the preparation's
    return (((sizeof(PrepSmem<N, M>) + 15) / 16) * 16 + sizeof(ModelConst<N, M>) + 31) / 16 * 16;
}
template <int N, int M>
constexpr size_t plan_dyn_smem() {
    return plan_off<N, M>() + sizeof(PlanSmem<N, M>);
}

template <int N, int M, bool FOLD>
KS_DEV void plan_block(char* dsm, int sg, const PlanArgs<N, M>& g) {
    PrepSmem<N, M>& p = *reinterpret_cast<PrepSmem<N, M>*>(dsm);
    ModelConst<N, M>& mc =
        *reinterpret_cast<ModelConst<N, M>*>(dsm + ((sizeof(PrepSmem<N, M>) + 15) / 16) * 16);
    PlanSmem<N, M>& s = *reinterpret_cast<PlanSmem<N, M>*>(dsm + plan_off<N, M>());
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) {
        if (sg == 0) g.status[HDR_GENERAL] = 0u;
        s.ok = 1;
        s.settled = 1;
    }
    const float* y1 = prep_inputs<N, M>(p, sg, g.B, g.F, g.u, g.Q, g.H, g.d, g.R, g.m0, g.P0, g.y, g.status, g.zero,
                                        g.nzero, g.off, g.T, g.first_tile);
    if (t < kChainThreads) {
        if (warp == 0) prep_consts<N, M>(p, mc, lane);
        chain_sync();
        plan_body<N, M>(s, p, mc, g.plan + sg);
    } else if (y1 != nullptr) {
        first_element_fp64<N, M>(p, mc, t - kChainThreads);
    } else {
        for (int e = t - kChainThreads; e < N; e += kFirstThreads) mc.b1[e] = 0.f;
        for (int e = t - kChainThreads; e < sym_size(N); e += kFirstThreads) mc.C1[e] = 0.f;
    }
    __syncthreads();
    prep_store<N, M>(p, mc, g.out + sg, g.status);
    SteadyPlan<N, M>* out = g.plan + sg;
    for (int e = t; e < sym_size(N); e += kPlanThreads) out->C1[e] = mc.C1[e];
    for (int e = t; e < N; e += kPlanThreads) out->b1[e] = mc.b1[e];
    bool ok = false;
    if (warp == 0) {
        float f = lane < N ? mc.C1[sidx(lane, lane)] / (s.sd[lane] * s.sd[lane]) : 0.f;
        const bool narrow = __any_sync(0xffffffffu, lane < N && !(f >= kStNarrow));
        if (!(f < 1e18f)) f = 1e18f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) f = fmaxf(f, __shfl_xor_sync(0xffffffffu, f, o));
        if (lane == 0) out->narrow = s.narrow = narrow ? 1 : 0;
        const float n = s.Hh[0];
        // at every length: the head's closed forms hold for a fixed point P only
        const bool settled = s.settled != 0 && fmaxf(f, 1.f) * n * n <= kStCovTol;
        // wait settings of the look-back are a test's: it wants the scans
        ok = s.ok != 0 && p.ok0 != 0 && p.ok1 != 0 && settled && g.status[HDR_WAIT] == 0u &&
             g.status[HDR_FIRST_TILE] == 0u;
        if (lane == 0) out->ok = ok ? 1 : 0;
        if constexpr (FOLD) {
            if (g.coef != nullptr && (g.off != nullptr || !ok))
                block_coef_warp<N, M>(mc, &p.H[0][0], g.ch, g.coef + sg);
        }
    }
    // the powers, for a head from a narrow start only (stored beside the first
    // doubling they cost every plan: 20 us of 1000 for 4096 sequences)
    __syncthreads();
    if (s.narrow && t < kChainThreads) element_powers<N, M>(s, mc, out);
}

template <int N, int M, bool FOLD>
__global__ void __launch_bounds__(kPlanThreads) plan_kernel(PlanArgs<N, M> g) {
    extern __shared__ __align__(16) char prep_dsm[];
    pdl_trigger();   // the windows' blocks may take their places; they wait for the plan
    plan_block<N, M, FOLD>(prep_dsm, (int)blockIdx.x, g);
}

// ---------------------------------------------------------------- windows
template <int N, int M>
struct SteadySmem {
    static constexpr int MP = kStCH * N + 4, YP = kStCH * M + 4;   // floats per thread: distinct banks for float4
    static constexpr int SY = sym_size(N);
    static constexpr int PR = N * N * 4 >= 256 ? 16 : 4096 / (N * N * 4);   // rows of a covariance pattern
    float ms[kStNT * MP];                      // window means; before that the tables Phi^n, O_n
    float ys[kStNT * YP];                      // measurements, then innovations
    SteadyCore<N, M> pl;
    alignas(128) float pat[2][PR * N * N];
    float hd[kStHead * (N * M + N)];           // head rows: P_k, then their gains and adjoint inputs
    float lam[kStHead * N];                    // means, then adjoint, of the head rows
    float wd[2][4 * N];                        // per-warp exchange of the window scans
    float tot[4 * (N * N + N)];                // per-warp totals of the head's scans
    float mlast[N], lin[N];
    int seq;
    static_assert(kStHead * (N * N + SY) <= kStNT * MP && SY <= N * M + N, "the tables fit");
};

// Mi = (I + X J)^-1 (X, J symmetric).  What it may cost is told by its Skeel
// condition max |Mi| |I + X J| 1, which the scale of a row does not enter: a prior
// that is wide along a coordinate (an unknown velocity, say) makes rows large
// and loses nothing (30 for a Wiener velocity model with P_0 = 1e5 I, whose 1-norm
// condition is 1e5), one that is wide across coordinates loses about that many
// ulps.  Beyond kHeadCond the scans are as good.
constexpr float kHeadCond = 256.f;
template <int N>
KS_DEV void inverse_ixj(const float (&X)[sym_size(N)], const float (&J)[sym_size(N)], float (&Mi)[N][N], Flags& bad) {
    float Mx[N][N], e[N];
#pragma unroll
    for (int a = 0; a < N; ++a) {
        e[a] = 0.f;
#pragma unroll
        for (int b = 0; b < N; ++b) {
            float s = (a == b) ? 1.f : 0.f;
#pragma unroll
            for (int l = 0; l < N; ++l) s = fmaf(X[sidx(a, l)], J[sidx(l, b)], s);
            Mx[a][b] = s;
            e[a] += fabsf(s);
        }
    }
    bool ok = inverse_pp<N>(Mx, Mi);
#pragma unroll
    for (int a = 0; a < N; ++a) {
        float s = 0.f;
#pragma unroll
        for (int b = 0; b < N; ++b) s = fmaf(fabsf(Mi[a][b]), e[b], s);
        ok = ok && s <= kHeadCond;
    }
    if (!ok) bad |= FL_NEED;
}

// X <- A Mi X A^T with Mi = (I + X J)^-1 (Mi X is symmetric).
template <int N>
KS_DEV void congruence(float (&X)[sym_size(N)], const float* __restrict__ A, const float (&Mi)[N][N]) {
    float W[sym_size(N)];
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int b = 0; b <= a; ++b) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < N; ++c) s = fmaf(Mi[a][c], X[sidx(c, b)], s);
            W[sidx(a, b)] = s;
        }
#pragma unroll
    for (int a = 0; a < N; ++a) {
        float y[N];
#pragma unroll
        for (int b = 0; b < N; ++b) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < N; ++c) s = fmaf(A[a * N + c], W[sidx(c, b)], s);
            y[b] = s;
        }
#pragma unroll
        for (int b = 0; b <= a; ++b) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < N; ++c) s = fmaf(y[c], A[b * N + c], s);
            X[sidx(a, b)] = s;
        }
    }
}

// The smoothed covariance (I - P O) Mi P_k of a row, Mi = (I + D_k O)^-1, to dst.
template <int N>
KS_DEV void smoothed_cov(const float (&Pk)[sym_size(N)], const float (&Mi)[N][N], const float (&O)[sym_size(N)],
                         const float* __restrict__ P, float* __restrict__ dst) {
#pragma unroll
    for (int b = 0; b < N; ++b) {
        float w[N], o[N];
#pragma unroll
        for (int a = 0; a < N; ++a) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < N; ++c) s = fmaf(Mi[a][c], Pk[sidx(c, b)], s);
            w[a] = s;
        }
#pragma unroll
        for (int a = 0; a < N; ++a) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < N; ++c) s = fmaf(O[sidx(a, c)], w[c], s);
            o[a] = s;
        }
#pragma unroll
        for (int a = b; a < N; ++a) {
            float s = w[a];
#pragma unroll
            for (int c = 0; c < N; ++c) s = fmaf(-P[a * N + c], o[c], s);
            dst[a * N + b] = s;
            if (a != b) dst[b * N + a] = s;
        }
    }
}

template <int N>
KS_DEV void matvec(const float* __restrict__ X, const float (&v)[N], float (&o)[N]) {
#pragma unroll
    for (int a = 0; a < N; ++a) {
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < N; ++c) s = fmaf(X[a * N + c], v[c], s);
        o[a] = s;
    }
}

template <int N>
KS_DEV void matvec_t(const float* __restrict__ X, const float (&v)[N], float (&o)[N]) {   // X^T v
#pragma unroll
    for (int a = 0; a < N; ++a) {
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < N; ++c) s = fmaf(X[c * N + a], v[c], s);
        o[a] = s;
    }
}

// Inclusive scan of the affine maps x -> A x + b over the block's threads, in
// thread order (UP) or against it: on return (A, b) maps what enters the first
// (last) thread of the warp, and `in` is what enters the warp, given what
// enters the block.  tot: the warps' totals.
template <int N, bool UP>
KS_DEV void affine_scan(float (&A)[N * N], float (&b)[N], float (&in)[N], float* tot, int warp, int lane) {
#pragma unroll 1
    for (int h = 1; h < 32; h <<= 1) {
        float Al[N * N], bl[N];
#pragma unroll
        for (int i = 0; i < N * N; ++i)
            Al[i] = UP ? __shfl_up_sync(0xffffffffu, A[i], h) : __shfl_down_sync(0xffffffffu, A[i], h);
#pragma unroll
        for (int i = 0; i < N; ++i)
            bl[i] = UP ? __shfl_up_sync(0xffffffffu, b[i], h) : __shfl_down_sync(0xffffffffu, b[i], h);
        if (UP ? lane >= h : lane + h < 32) {
            float o[N];
            matvec<N>(A, bl, o);
#pragma unroll
            for (int a = 0; a < N; ++a) b[a] += o[a];
#pragma unroll
            for (int a = 0; a < N; ++a) {
                float r[N];
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    float s = 0.f;
#pragma unroll
                    for (int l = 0; l < N; ++l) s = fmaf(A[a * N + l], Al[l * N + c], s);
                    r[c] = s;
                }
#pragma unroll
                for (int c = 0; c < N; ++c) A[a * N + c] = r[c];
            }
        }
    }
    constexpr int TS = N * N + N;
    if (lane == (UP ? 31 : 0)) {
#pragma unroll
        for (int i = 0; i < N * N; ++i) tot[warp * TS + i] = A[i];
#pragma unroll
        for (int i = 0; i < N; ++i) tot[warp * TS + N * N + i] = b[i];
    }
    __syncthreads();
#pragma unroll 1
    for (int w = UP ? 0 : 3; UP ? w < warp : w > warp; w += UP ? 1 : -1) {
        float o[N];
        matvec<N>(tot + w * TS, in, o);
#pragma unroll
        for (int a = 0; a < N; ++a) in[a] = o[a] + tot[w * TS + N * N + a];
    }
}

// One filter step with gain K: x <- F x + u + K e, e = y - d - H (F x + u).
template <int N, int M>
KS_DEV void mean_step(const float* __restrict__ F, const float* __restrict__ u, const float* __restrict__ H,
                      const float* __restrict__ d, const float* __restrict__ K, const float (&y)[M], float (&x)[N],
                      float (&e)[M]) {
    float mp[N];
#pragma unroll
    for (int a = 0; a < N; ++a) {
        float s = u[a];
#pragma unroll
        for (int c = 0; c < N; ++c) s = fmaf(F[a * N + c], x[c], s);
        mp[a] = s;
    }
#pragma unroll
    for (int q = 0; q < M; ++q) {
        float s = y[q] - d[q];
#pragma unroll
        for (int c = 0; c < N; ++c) s = fmaf(-H[q * N + c], mp[c], s);
        e[q] = s;
    }
#pragma unroll
    for (int a = 0; a < N; ++a) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < M; ++q) s = fmaf(K[a * M + q], e[q], s);
        x[a] = mp[a] + s;
    }
}

// Phi = F - K H F.
template <int N, int M>
KS_DEV void phi_of(const SteadyCore<N, M>& pl, const float (&K)[N * M], float (&A)[N * N]) {
    float HF[M][N];
#pragma unroll
    for (int q = 0; q < M; ++q)
#pragma unroll
        for (int a = 0; a < N; ++a) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < N; ++c) s = fmaf(pl.H[q * N + c], pl.F[c * N + a], s);
            HF[q][a] = s;
        }
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int c = 0; c < N; ++c) {
            float s = pl.F[a * N + c];
#pragma unroll
            for (int q = 0; q < M; ++q) s = fmaf(-K[a * M + q], HF[q][c], s);
            A[a * N + c] = s;
        }
}

// A state that observes y: the lift L (y - d).  The chunks' start guess, so
// that their scan runs on small differences from it and not on positions.
template <int N, int M>
KS_DEV void lift(const float* __restrict__ Lf, const float* __restrict__ d, const float (&y)[M], float (&x)[N]) {
#pragma unroll
    for (int a = 0; a < N; ++a) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < M; ++q) s = fmaf(Lf[a * M + q], y[q] - d[q], s);
        x[a] = s;
    }
}

// Largest |x_a| in posterior sd.
template <int N>
KS_DEV float in_sd(const float (&x)[N], const float* __restrict__ rsd) {
    float m = 0.f;
#pragma unroll
    for (int a = 0; a < N; ++a) m = fmaxf(m, fabsf(x[a]) * rsd[a]);
    return m;
}

// Whether every component is a number below 1e30: beyond that the scans decide
// (their products overflow earlier than a matrix-vector recursion's).
template <int N>
KS_DEV bool all_finite(const float (&x)[N]) {
    float s = 0.f;
#pragma unroll
    for (int a = 0; a < N; ++a) s = fabsf(x[a]) < 1e30f ? s : 1.f;
    return s == 0.f;
}

// Rows [r0, r1) of the window (first row w0) from shared memory to the means
// at `dst` (row 0 of the sequence), coalesced.
template <int N>
KS_DEV void copy_rows(const float* __restrict__ ms, int w0, int r0, int r1, float* __restrict__ dst, int tid) {
    constexpr int MP = kStCH * N + 4;
    using V = typename std::conditional<N % 4 == 0, float4, float2>::type;
    constexpr int VN = sizeof(V) / 4, PER = N / VN;
    V* __restrict__ out = reinterpret_cast<V*>(dst + (int64_t)r0 * N);
    const int n = (r1 - r0) * PER;
    for (int i = tid; i < n; i += kStNT) {
        const int w = r0 - w0 + i / PER, k = i % PER;
        out[i] = *reinterpret_cast<const V*>(ms + (w / kStCH) * MP + (w % kStCH) * N + k * VN);
    }
}

// The covariances of a head (rows 0..127) and of the end of a sequence (its
// last 128 rows after the head): the tables Phi^n, O_n for n = 1..128, thread
// n - 1 its n, rows h+1..2h from the rows before by
//     Phi^{h+m} = Phi^m Phi^h,  O_{h+m} = O_h + (Phi^h)^T O_m Phi^h,
// then D_k and the smoothed rows by one copy of the inverse (a block runs this
// code once a launch, and fetching it is a large part of its time).  The rows'
// P_k are left in sm.hd for head_forward.
template <int N, int M>
KS_DEV void head_covs(SteadySmem<N, M>& sm, const SteadyPlan<N, M>* __restrict__ gp, bool head, bool tail, int len,
                      int o0, float* __restrict__ fc, float* __restrict__ sc, Flags& bad) {
    constexpr int SY = sym_size(N), NN = N * N, TS = NN + SY;
    const SteadyCore<N, M>& pl = sm.pl;
    const int k = threadIdx.x;
    const bool smooth = sc != nullptr;
    float* tab = sm.ms;                                    // entry n - 1: Phi^n, O_n
    {
        float* own = tab + k * TS;
        if (k == 0) {
#pragma unroll
            for (int i = 0; i < NN; ++i) own[i] = pl.Ph[i];
#pragma unroll
            for (int i = 0; i < SY; ++i) own[NN + i] = pl.W[i];
        }
        __syncthreads();
#pragma unroll 1
        for (int h = 1; h < kStHead; h *= 2) {
            if (k >= h && k < 2 * h) {
                const float *m = tab + (k - h) * TS, *p = tab + (h - 1) * TS;   // Phi^m, O_m; Phi^h, O_h
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    float r[N];
#pragma unroll
                    for (int c = 0; c < N; ++c) r[c] = m[a * N + c];
#pragma unroll
                    for (int c = 0; c < N; ++c) {
                        float s = 0.f;
#pragma unroll
                        for (int l = 0; l < N; ++l) s = fmaf(r[l], p[l * N + c], s);
                        own[a * N + c] = s;
                    }
                }
                float T[N][N];                             // O_m Phi^h
#pragma unroll
                for (int a = 0; a < N; ++a)
#pragma unroll
                    for (int c = 0; c < N; ++c) {
                        float s = 0.f;
#pragma unroll
                        for (int l = 0; l < N; ++l) s = fmaf(m[NN + sidx(a, l)], p[l * N + c], s);
                        T[a][c] = s;
                    }
#pragma unroll
                for (int a = 0; a < N; ++a)
#pragma unroll
                    for (int c = 0; c <= a; ++c) {
                        float s = p[NN + sidx(a, c)];
#pragma unroll
                        for (int l = 0; l < N; ++l) s = fmaf(p[l * N + a], T[l][c], s);
                        own[NN + sidx(a, c)] = s;
                    }
            }
            __syncthreads();
        }
    }
    // rounds: D_k of the head, its smoothed rows, the smoothed rows of the end;
    // from a narrow start, before these, P_1 through the powers of the bits of k
    const bool narrow = head && pl.narrow != 0;
    float P[SY], D[SY];
#pragma unroll
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int c = 0; c <= a; ++c) {
            P[sidx(a, c)] = narrow ? pl.C1[sidx(a, c)] : pl.Pf[a * N + c];
            D[sidx(a, c)] = 0.f;
        }
#pragma unroll 1
    for (int it = narrow ? -kStLev : 0; it < 3; ++it) {
        float X[SY], J[SY];
        bool run;
        int n = 0;                                         // later measurements of the row
        if (it < 0) {
            run = (k >> (it + kStLev)) & 1;
        } else if (it == 0) {
            run = head && !narrow;
            if (narrow) {
#pragma unroll
                for (int a = 0; a < N; ++a)
#pragma unroll
                    for (int c = 0; c <= a; ++c) D[sidx(a, c)] = P[sidx(a, c)] - pl.Pf[a * N + c];
            }
        } else if (it == 1) {
            run = head && smooth && k < len;
            n = len - 1 - k;
        } else {
            run = smooth && tail && len - 1 - k >= o0;
            n = k;
        }
        if (run) {
            const float* e = tab + max(k - 1, 0) * TS;     // Phi^k, O_k
            const float* A = it < 0 ? gp->EA[it + kStLev] : e;
            if (it <= 0) {
                const float* j = it < 0 ? gp->EJ[it + kStLev] : e + NN;
#pragma unroll
                for (int i = 0; i < SY; ++i) { X[i] = it < 0 ? P[i] : pl.C1[i] - P[i]; J[i] = j[i]; }
            } else {
                const float* o = n >= kStHead ? pl.On : tab + max(n - 1, 0) * TS + NN;
                if (it == 2) {
#pragma unroll
                    for (int a = 0; a < N; ++a)
#pragma unroll
                        for (int c = 0; c <= a; ++c) { P[sidx(a, c)] = pl.Pf[a * N + c]; D[sidx(a, c)] = 0.f; }
                }
#pragma unroll
                for (int i = 0; i < SY; ++i) { X[i] = D[i]; J[i] = n > 0 ? o[i] : 0.f; }
            }
            float Mi[N][N];
            if (it < 2) {
                inverse_ixj<N>(X, J, Mi, bad);
            } else {                                       // D = 0
#pragma unroll
                for (int a = 0; a < N; ++a)
#pragma unroll
                    for (int c = 0; c < N; ++c) Mi[a][c] = a == c ? 1.f : 0.f;
            }
            if (it > 0) {
                smoothed_cov<N>(P, Mi, J, pl.Pf, sc + (int64_t)(it == 1 ? k : len - 1 - k) * NN);
            } else if (it == 0 && k == 0) {
#pragma unroll
                for (int i = 0; i < SY; ++i) { D[i] = X[i]; P[i] = pl.C1[i]; }
            } else {
                congruence<N>(X, A, Mi);
#pragma unroll
                for (int i = 0; i < SY; ++i) {
                    D[i] = X[i];
                    P[i] = X[i] + (it < 0 ? gp->EC[it + kStLev][i] : P[i]);
                }
            }
        }
        if (it == 0 && head) {
#pragma unroll
            for (int i = 0; i < SY; ++i) sm.hd[k * SY + i] = P[i];
            if (k < len) {
#pragma unroll
                for (int a = 0; a < N; ++a)
#pragma unroll
                    for (int c = 0; c < N; ++c) fc[(int64_t)k * NN + a * N + c] = P[sidx(a, c)];
            }
        }
    }
}

// The head's means: thread k has row k (k < 128).  Its gain from the predicted
// covariance of the row before, its mean by a scan of the affine maps
// x_k = Phi_k x_{k-1} + ... in differences from the lifted measurements.
// Writes rows 0..min(len, 128)-1 of fm; leaves the gains and the adjoint's
// inputs for head_reverse.
template <int N, int M>
KS_DEV void head_forward(SteadySmem<N, M>& sm, const float* __restrict__ y, int len, float* __restrict__ fm,
                         Flags& bad) {
    constexpr int SY = sym_size(N);
    const SteadyCore<N, M>& pl = sm.pl;
    const int k = threadIdx.x, warp = k >> 5, lane = k & 31;
    const float* ptab = sm.hd;
    const bool on = k < len;
    __syncthreads();                                       // P_k of every row (head_covs)
    float yk[M], yg[M];
#pragma unroll
    for (int q = 0; q < M; ++q) yk[q] = on ? y[(int64_t)k * M + q] : 0.f;
#pragma unroll
    for (int q = 0; q < M; ++q) yg[q] = (k > 0 && k <= len) ? y[(int64_t)(k - 1) * M + q] : 0.f;
    float K[N * M], A[N * N], b[N], xg[N], Si[M][M];
    lift<N, M>(pl.Lf, pl.d, yk, xg);
    if (k == 0) {
#pragma unroll
        for (int i = 0; i < N * N; ++i) A[i] = 0.f;
#pragma unroll
        for (int i = 0; i < N * M; ++i) K[i] = 0.f;
#pragma unroll
        for (int a = 0; a < N; ++a) b[a] = pl.b1[a] - xg[a];
    } else {
        float HP[M][N], S[sym_size(M)];
        {
            float Pm[SY];
#pragma unroll
            for (int a = 0; a < N; ++a) {
                float r[N];
#pragma unroll
                for (int c = 0; c < N; ++c) {
                    float s = 0.f;
#pragma unroll
                    for (int l = 0; l < N; ++l) s = fmaf(pl.F[a * N + l], ptab[(k - 1) * SY + sidx(l, c)], s);
                    r[c] = s;
                }
#pragma unroll
                for (int c = 0; c <= a; ++c) {
                    float s = pl.Q[sidx(a, c)];
#pragma unroll
                    for (int l = 0; l < N; ++l) s = fmaf(r[l], pl.F[c * N + l], s);
                    Pm[sidx(a, c)] = s;
                }
            }
#pragma unroll
            for (int q = 0; q < M; ++q)
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    float s = 0.f;
#pragma unroll
                    for (int c = 0; c < N; ++c) s = fmaf(pl.H[q * N + c], Pm[sidx(c, a)], s);
                    HP[q][a] = s;
                }
        }
#pragma unroll
        for (int q = 0; q < M; ++q)
#pragma unroll
            for (int r = 0; r <= q; ++r) {
                float s = pl.R[sidx(q, r)];
#pragma unroll
                for (int c = 0; c < N; ++c) s = fmaf(HP[q][c], pl.H[r * N + c], s);
                S[sidx(q, r)] = s;
            }
        float Li[M][M];
        if (!chol_inv_lower<M>(S, Li)) bad |= FL_BAD;
#pragma unroll
        for (int q = 0; q < M; ++q)
#pragma unroll
            for (int r = 0; r <= q; ++r) {
                float s = 0.f;
#pragma unroll
                for (int l = q; l < M; ++l) s = fmaf(Li[l][q], Li[l][r], s);
                Si[q][r] = s;
                Si[r][q] = s;
            }
#pragma unroll
        for (int a = 0; a < N; ++a)
#pragma unroll
            for (int q = 0; q < M; ++q) {
                float s = 0.f;
#pragma unroll
                for (int r = 0; r < M; ++r) s = fmaf(HP[r][a], Si[r][q], s);
                K[a * M + q] = s;
            }
        phi_of<N, M>(pl, K, A);
        float x[N], e[M];
        lift<N, M>(pl.Lf, pl.d, yg, x);
        mean_step<N, M>(pl.F, pl.u, pl.H, pl.d, K, yk, x, e);
#pragma unroll
        for (int a = 0; a < N; ++a) b[a] = x[a] - xg[a];
    }
    float din[N], x[N];
#pragma unroll
    for (int a = 0; a < N; ++a) din[a] = 0.f;
    affine_scan<N, true>(A, b, din, sm.tot, warp, lane);
    matvec<N>(A, din, x);
#pragma unroll
    for (int a = 0; a < N; ++a) x[a] = xg[a] + (b[a] + x[a]);
    // each mean once more from its neighbour's, in the innovation form
#pragma unroll
    for (int a = 0; a < N; ++a) sm.lam[k * N + a] = x[a];
    __syncthreads();
    if (k > 0) {
        float e[M], z[M];
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = sm.lam[(k - 1) * N + a];
        mean_step<N, M>(pl.F, pl.u, pl.H, pl.d, K, yk, x, e);
#pragma unroll
        for (int q = 0; q < M; ++q) {
            float s = 0.f;
#pragma unroll
            for (int r = 0; r < M; ++r) s = fmaf(Si[q][r], e[r], s);
            z[q] = s;
        }
#pragma unroll
        for (int q = 0; q < M; ++q) e[q] = z[q];
#pragma unroll
        for (int q = 0; q < M; ++q) z[q] = on ? e[q] : 0.f;
        float h[N], o[N];
#pragma unroll
        for (int a = 0; a < N; ++a) {
            float s = 0.f;
#pragma unroll
            for (int q = 0; q < M; ++q) s = fmaf(pl.H[q * N + a], z[q], s);
            h[a] = s;
        }
        matvec_t<N>(pl.F, h, o);
#pragma unroll
        for (int a = 0; a < N; ++a) sm.hd[kStHead * N * M + k * N + a] = o[a];
#pragma unroll
        for (int i = 0; i < N * M; ++i) sm.hd[k * N * M + i] = K[i];
    }
    if (k == kStHead - 1) {
#pragma unroll
        for (int a = 0; a < N; ++a) sm.mlast[a] = x[a];
    }
    if (on) {
        if (!all_finite<N>(x)) bad |= FL_BAD;
#pragma unroll
        for (int a = 0; a < N; ++a) fm[(int64_t)k * N + a] = x[a];
    }
    __syncthreads();
}

// The head's smoothed means: thread j's map takes l_j to l_{j-1} =
// Phi_j^T l_j + b_j, scanned from the last row on; row k is m_k + P_k l_k.
// sm.lin: l_127 (zero where the sequence ends in the head).
template <int N, int M>
KS_DEV void head_reverse(SteadySmem<N, M>& sm, int len, const float* fm, const float* fc, float* __restrict__ smo,
                         Flags& bad) {
    const SteadyCore<N, M>& pl = sm.pl;
    const int k = threadIdx.x, warp = k >> 5, lane = k & 31;
    float A[N * N], b[N], in[N], l[N];
#pragma unroll
    for (int a = 0; a < N; ++a) { b[a] = 0.f; in[a] = sm.lin[a]; }
    if (k > 0 && k < len) {
        float K[N * M], Ph[N * N];
#pragma unroll
        for (int i = 0; i < N * M; ++i) K[i] = sm.hd[k * N * M + i];
        phi_of<N, M>(pl, K, Ph);
#pragma unroll
        for (int a = 0; a < N; ++a) {
            b[a] = sm.hd[kStHead * N * M + k * N + a];
#pragma unroll
            for (int c = 0; c < N; ++c) A[a * N + c] = Ph[c * N + a];
        }
    } else {
#pragma unroll
        for (int i = 0; i < N * N; ++i) A[i] = i / N == i % N ? 1.f : 0.f;
    }
    affine_scan<N, false>(A, b, in, sm.tot, warp, lane);
    matvec<N>(A, in, l);
#pragma unroll
    for (int a = 0; a < N; ++a)
        if (k > 0) sm.lam[(k - 1) * N + a] = l[a] + b[a];
    __syncthreads();
    if (k < len) {
        float P[N * N], e[N];
#pragma unroll
        for (int a = 0; a < N; ++a) l[a] = k == kStHead - 1 ? sm.lin[a] : sm.lam[k * N + a];
#pragma unroll
        for (int i = 0; i < N * N; ++i) P[i] = fc[(int64_t)k * N * N + i];
        matvec<N>(P, l, e);
        if (!all_finite<N>(e)) bad |= FL_BAD;
#pragma unroll
        for (int a = 0; a < N; ++a) smo[(int64_t)k * N + a] = fm[(int64_t)k * N + a] + e[a];
    }
}

// Work of block `slot` of a launch (see steady_blocks).  Reads the offsets and
// the measurements before it waits for the plan's kernel: they are the
// caller's, complete before that kernel began.
template <int N, int M>
KS_DEV void steady_block(char* dsm, const SteadyArgs<N, M>& g, int64_t slot) {
    using SM = SteadySmem<N, M>;
    constexpr int NN = N * N, SY = SM::SY, MP = SM::MP, YP = SM::YP, PR = SM::PR;
    SM& sm = *reinterpret_cast<SM*>(dsm);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // ---- which sequence: the last one whose first slot is <= slot (32 probes at a time)
    int64_t a0 = 0, a1 = g.T, first = 0;
    int b = 0;
    if (g.off != nullptr) {
        if (warp == 0) {
            int lo = 0, hi = g.B;
            while (hi - lo > 1) {
                const int step = (hi - lo + 31) / 32, at = lo + lane * step;
                const bool le = at < hi && g.off[at] / kStOut + at <= slot;
                const int n = max(1, __popc(__ballot_sync(0xffffffffu, le)));
                lo += (n - 1) * step;
                hi = min(hi, lo + step);
            }
            if (lane == 0) sm.seq = lo;
        }
        __syncthreads();
        b = sm.seq;
        a0 = g.off[b];
        a1 = g.off[b + 1];
        first = a0 / kStOut + b;
    }
    // no block leaves before the wait: what follows this launch must find the plan done
    if (!(a0 >= 0 && a0 < a1 && a1 <= g.T) || slot < first) {   // an inconsistent table (reported by the plan)
        pdl_wait();
        return;
    }
    const int64_t j = slot - first;
    const int len = (int)(a1 - a0);
    if (j >= steady_windows(len)) {
        pdl_wait();
        return;
    }
    const StWindow win = steady_window(len, (int)j);
    const bool head = win.head, last = win.last;
    const int o0 = win.o0, o1 = win.o1, w0 = win.w0, rows = win.rows;
    const float* y = g.y + a0 * M;
    float *fm = g.fm + a0 * N, *fc = g.fc + a0 * NN;
    float* so = g.sm ? g.sm + a0 * N : nullptr;
    float* sc = g.sc ? g.sc + a0 * NN : nullptr;
    {   // the measurements on their way, one thread's 16 steps side by side, before the plan is there
        const float* src = y + (int64_t)w0 * M;
        const int n = rows * M;
        for (int i = tid; i < n; i += kStNT) {
            const int w = i / M;
            cp_async4(sm.ys + (w / kStCH) * YP + (w % kStCH) * M + i % M, src + i);
        }
    }
    pdl_wait();
    if (g.plan[b].ok == 0) {
        if (j == 0 && tid == 0) atomicOr(g.status + HDR_GENERAL, 1u);
        cp_async_wait_all();
        return;
    }
    pdl_trigger();   // not before: what follows is to know whether the plans passed (gate_closed)
    {   // the plan (the head's part too for a head)
        using Core = SteadyCore<N, M>;
        const int n = (int)((head || last ? sizeof(Core) : offsetof(Core, W)) / 16);
        const float4* src = reinterpret_cast<const float4*>(g.plan + b);
        float4* dst = reinterpret_cast<float4*>(&sm.pl);
        for (int i = tid; i < n; i += kStNT) dst[i] = src[i];
    }
    __syncthreads();
    const SteadyCore<N, M>& pl = sm.pl;
    Flags bad = 0u;
    // ---- constant covariance rows: bulk copies of a pattern, in flight while the means are computed
    const int s1 = last ? max(o0, len - kStHead) : o1;         // smoothed rows that are settled: [o0, s1)
    const bool fillf = g.keep != 0 && o1 > o0, fills = sc != nullptr && s1 > o0;
    for (int i = tid; i < PR * NN; i += kStNT) {
        sm.pat[0][i] = pl.Pf[i % NN];
        sm.pat[1][i] = pl.Ps[i % NN];
    }
    fence_proxy_async();
    __syncthreads();
    // Issued in kFill slices between the passes, each copy by another warp: the
    // copies go out no faster than the memory takes them, and a warp that
    // issues them all at once keeps the block waiting at its next barrier.
    constexpr int kFill = 6;
    const int nf = fillf ? (o1 - o0 + PR - 1) / PR : 0, ns = fills ? (s1 - o0 + PR - 1) / PR : 0;
    auto fill = [&](int slice) {
        const int lo = (nf + ns) * slice / kFill, hi = (nf + ns) * (slice + 1) / kFill;
        for (int i = lo + lane * 4 + warp; i < hi; i += kStNT) {
            const bool f = i < nf;
            const int r = o0 + (f ? i : i - nf) * PR, end = f ? o1 : s1;
            bulk_store((f ? fc : sc) + (int64_t)r * NN, sm.pat[f ? 0 : 1], 4u * NN * (uint32_t)min(PR, end - r));
        }
    };
    fill(0);
    if (head || (last && sc != nullptr)) head_covs<N, M>(sm, g.plan + b, head, last, len, o0, fc, sc, bad);
    if (head) head_forward<N, M>(sm, y, len, fm, bad);
    else if (last) __syncthreads();   // the tables are read, the window may take their place
    if (rows > 0) {
        cp_async_wait_all();
        __syncthreads();
        const int c0 = tid * kStCH, cnt = steady_chunk(rows, c0);   // the thread's chunk
        float* yc = sm.ys + tid * YP;
        float* mc = sm.ms + tid * MP;
        float xg[N], x[N], v[N];
        float K[N * M];
#pragma unroll
        for (int i = 0; i < N * M; ++i) K[i] = pl.K[i];
        auto load_y = [&](const float* p, float (&o)[M]) {
#pragma unroll
            for (int q = 0; q < M; ++q) o[q] = p[q];
        };
        // the step's constants in registers (the loops store to shared memory, so
        // the compiler cannot keep them there itself)
        float F[NN], H[M * N], u[N], d[M];
#pragma unroll
        for (int i = 0; i < NN; ++i) F[i] = pl.F[i];
#pragma unroll
        for (int i = 0; i < M * N; ++i) H[i] = pl.H[i];
#pragma unroll
        for (int i = 0; i < N; ++i) u[i] = pl.u[i];
#pragma unroll
        for (int i = 0; i < M; ++i) d[i] = pl.d[i];
        // ---- pass 1: each chunk from its guess; what it misses the next chunk's guess by
        {
            float yv[M], e[M];
            load_y(yc, yv);
            lift<N, M>(pl.Lf, pl.d, yv, xg);
#pragma unroll
            for (int a = 0; a < N; ++a) x[a] = xg[a];
#pragma unroll(N <= 4 ? 2 : 1)
            for (int i = 0; i < cnt; ++i) {
                load_y(yc + i * M, yv);
                mean_step<N, M>(F, u, H, d, K, yv, x, e);
            }
            if (c0 + kStCH < rows) {
                float xn[N];
                load_y(yc + YP, yv);
                lift<N, M>(pl.Lf, pl.d, yv, xn);
#pragma unroll
                for (int a = 0; a < N; ++a) x[a] -= xn[a];
            } else {
#pragma unroll
                for (int a = 0; a < N; ++a) x[a] = 0.f;
            }
        }
        fill(1);
        // ---- scan of the differences d_{c+1} = Phi^16 d_c + (miss of chunk c); Phi^512 = 0
        if (lane == 31) {
#pragma unroll
            for (int a = 0; a < N; ++a) sm.wd[0][warp * N + a] = x[a];
        }
        __syncthreads();
#pragma unroll
        for (int a = 0; a < N; ++a) {
            const float up = __shfl_up_sync(0xffffffffu, x[a], 1);
            const float in = warp > 0 ? sm.wd[0][(warp - 1) * N + a] : (head ? sm.mlast[a] - xg[a] : 0.f);
            v[a] = lane > 0 ? up : in;
        }
#pragma unroll
        for (int i = 0; i < kStPow; ++i) {
            float o[N], t[N];
#pragma unroll
            for (int a = 0; a < N; ++a) o[a] = __shfl_up_sync(0xffffffffu, v[a], 1 << i);
            matvec<N>(pl.FP[i], o, t);
#pragma unroll
            for (int a = 0; a < N; ++a) v[a] += lane >= (1 << i) ? t[a] : 0.f;
        }
        if (lane == 31) {
#pragma unroll
            for (int a = 0; a < N; ++a) sm.wd[1][warp * N + a] = v[a];
        }
        __syncthreads();
        if (warp > 0 && lane < 31) {
            float z[N];
#pragma unroll
            for (int a = 0; a < N; ++a) z[a] = sm.wd[1][(warp - 1) * N + a];
#pragma unroll
            for (int i = 0; i < kStPow; ++i)
                if ((lane + 1) >> i & 1) {
                    float t[N];
                    matvec<N>(pl.FP[i], z, t);
#pragma unroll
                    for (int a = 0; a < N; ++a) z[a] = t[a];
                }
#pragma unroll
            for (int a = 0; a < N; ++a) v[a] += z[a];
        }
        // a neighbour leaves out what lies beyond its halo, which only this window sees (the
        // first and the last one too, although their own outer ends are exact)
        const bool alone = head && last;
        if (cnt > 0 && !alone && !(pl.nphi * in_sd<N>(v, pl.rsd) <= kStMeanTol)) bad |= FL_NEED;
        // ---- pass 2: the means, and the innovations in the measurements' place
#pragma unroll
        for (int a = 0; a < N; ++a) x[a] = xg[a] + v[a];
#pragma unroll(N <= 4 ? 2 : 1)
        for (int i = 0; i < cnt; ++i) {
            float yv[M], e[M];
            load_y(yc + i * M, yv);
            mean_step<N, M>(F, u, H, d, K, yv, x, e);
#pragma unroll
            for (int q = 0; q < M; ++q) yc[i * M + q] = e[q];
#pragma unroll
            for (int a = 0; a < N; ++a) mc[i * N + a] = x[a];
        }
        if (cnt > 0 && !all_finite<N>(x)) bad |= FL_BAD;
        fill(2);
        __syncthreads();
        if (g.keep) copy_rows<N>(sm.ms, w0, o0, o1, fm, tid);
        fill(3);
        if (so != nullptr) {
            float Ph[NN], Bm[N * M], P[SY];
#pragma unroll
            for (int i = 0; i < NN; ++i) Ph[i] = pl.Ph[i];
#pragma unroll
            for (int i = 0; i < N * M; ++i) Bm[i] = pl.B[i];
#pragma unroll
            for (int a = 0; a < N; ++a)
#pragma unroll
                for (int c = 0; c <= a; ++c) P[sidx(a, c)] = pl.Pf[a * N + c];
            // l <- Phi^T l + B (innovation of the next row)
            auto back = [&](const float* ep, float (&l)[N]) {
                float t[N];
                matvec_t<N>(Ph, l, t);
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    float s = t[a];
#pragma unroll
                    for (int q = 0; q < M; ++q) s = fmaf(Bm[a * M + q], ep[q], s);
                    l[a] = s;
                }
            };
            const int top = c0 + cnt == rows ? cnt - 2 : cnt - 1;    // the window's last row keeps l = 0
#pragma unroll
            for (int a = 0; a < N; ++a) x[a] = 0.f;
#pragma unroll(N <= 4 ? 2 : 1)
            for (int i = top; i >= 0; --i) back(i + 1 < kStCH ? yc + (i + 1) * M : yc + YP, x);
            fill(4);
            if (lane == 0) {
#pragma unroll
                for (int a = 0; a < N; ++a) sm.wd[0][warp * N + a] = x[a];
            }
            __syncthreads();
#pragma unroll
            for (int a = 0; a < N; ++a) {
                const float dn = __shfl_down_sync(0xffffffffu, x[a], 1);
                v[a] = lane < 31 ? dn : (warp < 3 ? sm.wd[0][(warp + 1) * N + a] : 0.f);
            }
#pragma unroll
            for (int i = 0; i < kStPow; ++i) {
                float o[N], t[N];
#pragma unroll
                for (int a = 0; a < N; ++a) o[a] = __shfl_down_sync(0xffffffffu, v[a], 1 << i);
                matvec_t<N>(pl.FP[i], o, t);
#pragma unroll
                for (int a = 0; a < N; ++a) v[a] += lane + (1 << i) < 32 ? t[a] : 0.f;
            }
            if (lane == 0) {
#pragma unroll
                for (int a = 0; a < N; ++a) sm.wd[1][warp * N + a] = v[a];
            }
            __syncthreads();
            if (warp < 3 && lane > 0) {
                float z[N];
#pragma unroll
                for (int a = 0; a < N; ++a) z[a] = sm.wd[1][(warp + 1) * N + a];
#pragma unroll
                for (int i = 0; i < kStPow; ++i)
                    if ((32 - lane) >> i & 1) {
                        float t[N];
                        matvec_t<N>(pl.FP[i], z, t);
#pragma unroll
                        for (int a = 0; a < N; ++a) z[a] = t[a];
                    }
#pragma unroll
                for (int a = 0; a < N; ++a) v[a] += z[a];
            }
            if (cnt > 0 && !alone && !(pl.ndual * in_sd<N>(v, pl.sd) <= kStMeanTol)) bad |= FL_NEED;
            if (c0 + cnt == rows) {                                // the row after the window does not count
#pragma unroll
                for (int a = 0; a < N; ++a) v[a] = 0.f;
            }
#pragma unroll(N <= 4 ? 2 : 1)
            for (int i = top; i >= 0; --i) {
                back(i + 1 < kStCH ? yc + (i + 1) * M : yc + YP, v);
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    float s = 0.f;
#pragma unroll
                    for (int c = 0; c < N; ++c) s = fmaf(P[sidx(a, c)], v[c], s);
                    mc[i * N + a] += s;
                }
            }
            if (cnt > 0 && !all_finite<N>(v)) bad |= FL_BAD;
            if (tid == 0) {                                        // l_127 from row 128, for the head
                back(yc, v);
#pragma unroll
                for (int a = 0; a < N; ++a) sm.lin[a] = v[a];
            }
            fill(5);
            __syncthreads();
            copy_rows<N>(sm.ms, w0, o0, o1, so, tid);
        } else {
            fill(4);
            fill(5);
        }
    }
    if (head && so != nullptr) {
        if (len <= kStHead && tid < N) sm.lin[tid] = 0.f;
        __syncthreads();
        head_reverse<N, M>(sm, len, fm, fc, so, bad);
    }
    if (__any_sync(0xffffffffu, bad != 0u) && lane == 0) atomicOr(g.status + HDR_GENERAL, 1u);
    bulk_commit();
    bulk_wait_read_all();
}

template <int N>
constexpr int kSteadyMinBlocks = N <= 2 ? 4 : N <= 4 ? 3 : N <= 6 ? 2 : 1;

template <int N, int M>
__global__ void __launch_bounds__(kStNT, kSteadyMinBlocks<N>) steady_kernel(SteadyArgs<N, M> g) {
    extern __shared__ __align__(16) char dsm[];
    steady_block<N, M>(dsm, g, (int64_t)blockIdx.x);
}

// ---------------------------------------------------------------- host
template <int N, int M>
int launch_plan_kernel(const PlanArgs<N, M>& g, cudaStream_t st) {
    constexpr int smem = (int)plan_dyn_smem<N, M>();
    static_assert(smem <= 48 * 1024, "no opt-in needed");
    if constexpr (N <= 6) {
        if (g.coef != nullptr) {
            plan_kernel<N, M, true><<<g.B, kPlanThreads, smem, st>>>(g);
            return launch_status();
        }
    }
    plan_kernel<N, M, false><<<g.B, kPlanThreads, smem, st>>>(g);
    return launch_status();
}

template <int N, int M>
int launch_steady_kernel(const SteadyArgs<N, M>& g, cudaStream_t st) {
    constexpr int smem = (int)sizeof(SteadySmem<N, M>);
    auto k = steady_kernel<N, M>;
    static const bool ok =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess;
    if (!ok) return KS_ECUDA;
    return launch_pdl(k, (int)steady_blocks(g.T, g.B), kStNT, smem, st, g);
}

}  // namespace ks
