// The settled path at nx = 32, ny = 8 (ks_steady32.cuh).
#include "ks_steady32.cuh"

#include <cstddef>

#include "ks_steady_kernels.cuh"
#include "ks_tc.cuh"

namespace ks {
namespace {

constexpr int N = 32, M = 8, P = 36;                 // P: row pitch of a matrix in shared memory
constexpr int MATF = 33 * P;                         // floats of one (gj_inverse's buffers have a spare row)
constexpr unsigned kAll = 0xffffffffu;

// Rows [w R, w R + R) of D = sa op(A) op(B) (+ add), by one warp, lane = column.
// Row operands are read by broadcast (16 bytes at a time), so a product costs
// about 400 shared-memory cycles however many warps share it.
template <int R, bool TA, bool TB>
KS_DEV void mprod(const float* A, const float* B, float* D, int w, int lane, const float* add = nullptr,
                  float sa = 1.f) {
    static_assert(R % 4 == 0 || !TA, "transposed rows come four at a time");
    float acc[R];
    const int r0 = w * R;
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.f;
#pragma unroll 2
    for (int k = 0; k < N; k += 4) {
        float b[4];
        if constexpr (TB) {
            const float4 t = *reinterpret_cast<const float4*>(B + lane * P + k);
            b[0] = t.x; b[1] = t.y; b[2] = t.z; b[3] = t.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) b[i] = B[(k + i) * P + lane];
        }
        if constexpr (TA) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int r = 0; r < R; r += 4) {
                    const float4 t = *reinterpret_cast<const float4*>(A + (k + i) * P + r0 + r);
                    acc[r] = fmaf(t.x, b[i], acc[r]);
                    acc[r + 1] = fmaf(t.y, b[i], acc[r + 1]);
                    acc[r + 2] = fmaf(t.z, b[i], acc[r + 2]);
                    acc[r + 3] = fmaf(t.w, b[i], acc[r + 3]);
                }
        } else {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 t = *reinterpret_cast<const float4*>(A + (r0 + r) * P + k);
                acc[r] = fmaf(t.x, b[0], acc[r]);
                acc[r] = fmaf(t.y, b[1], acc[r]);
                acc[r] = fmaf(t.z, b[2], acc[r]);
                acc[r] = fmaf(t.w, b[3], acc[r]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const float v = sa * acc[r];
        D[(r0 + r) * P + lane] = add ? add[(r0 + r) * P + lane] + v : v;
    }
}

KS_DEV void add_identity(float* X, int t) {
    if (t < N) X[t * P + t] += 1.f;
}
// X <- (X + X^T) / 2 by nt threads.
KS_DEV void symmetrise(float* X, int t, int nt) {
    for (int e = t; e < N * N; e += nt) {
        const int a = e / N, b = e % N;
        if (b < a) {
            const float v = 0.5f * (X[a * P + b] + X[b * P + a]);
            X[a * P + b] = v;
            X[b * P + a] = v;
        }
    }
}
KS_DEV void load32(float* X, const float* __restrict__ g, int t, int nt) {
    for (int e = t; e < 256; e += nt)
        *reinterpret_cast<float4*>(X + (e / 8) * P + (e % 8) * 4) = reinterpret_cast<const float4*>(g)[e];
}
KS_DEV void store32(float* __restrict__ g, const float* X, int t, int nt) {
    for (int e = t; e < 256; e += nt)
        reinterpret_cast<float4*>(g)[e] = *reinterpret_cast<const float4*>(X + (e / 8) * P + (e % 8) * 4);
}
KS_DEV void store32_t(float* __restrict__ g, const float* X, int t, int nt) {
    for (int e = t; e < 1024; e += nt) g[e] = X[(e % N) * P + e / N];
}

// S^{-1} of the innovation covariance S = HP H^T + R (HP [8][P], one warp), the
// gain K = HP^T S^{-1} and B = HF^T S^{-1}, [32][8] each.
KS_DEV bool gains(const float* HP, const float* H, const float* HF, const float* R, float* S, float* Si,
                  float* __restrict__ Ko, float* __restrict__ Bo, float* Ks, int lane) {
    for (int e = lane; e < M * M; e += 32) {
        const int a = e / M, b = e % M;
        float s = R[e];
        for (int c = 0; c < N; ++c) s = fmaf(HP[a * P + c], H[b * P + c], s);
        S[e] = s;
    }
    __syncwarp();
    float cond;
    const bool ok = warp_inverse<M>(S, Si, lane, cond) && cond <= kRefineCond;
    __syncwarp();
#pragma unroll
    for (int q = 0; q < M; ++q) {
        float k = 0.f, b = 0.f;
#pragma unroll
        for (int r = 0; r < M; ++r) {
            k = fmaf(HP[r * P + lane], Si[r * M + q], k);
            b = fmaf(HF[r * P + lane], Si[r * M + q], b);
        }
        Ko[lane * M + q] = k;
        Bo[lane * M + q] = b;
        if (Ks) { Ks[lane * M + q] = k; Ks[256 + lane * M + q] = b; }
    }
    return __all_sync(kAll, ok);
}

// ---------------------------------------------------------------- plan
constexpr int kPlanNT = 512;
struct PlanSmem32 {
    float A[2][MATF], C[2][MATF], J[2][MATF], Mx[MATF], Mi[MATF], X[MATF], W[MATF], V[MATF], Y[MATF], Z[MATF];
    float H[M * P], HF[M * P], HP[M * P], S[64], Si[64], R[64], KB[512], sd[N], vs[tc::VS<N>::FLOATS];
    int ok;
};
__host__ __device__ constexpr size_t plan32_off() {
    return (((sizeof(PrepSmem<N, M>) + 15) / 16) * 16 + sizeof(ModelConst<N, M>) + 31) / 16 * 16;
}

KS_DEV float scaled_norm32(const float* X, const float* sd, int lane, bool col) {
    float s = 0.f;
    for (int b = 0; b < N; ++b)
        s = col ? fmaf(fabsf(X[b * P + lane]), 1.f / sd[b], s) : fmaf(fabsf(X[lane * P + b]), sd[b], s);
    s = col ? s * sd[lane] : s / sd[lane];
    if (!(s < 1e18f)) s = 1e18f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = fmaxf(s, __shfl_xor_sync(kAll, s, o));
    return s;
}

__global__ void __launch_bounds__(kPlanNT) plan32_kernel(Args32 g) {
    extern __shared__ __align__(128) char dsm32[];
    PrepSmem<N, M>& p = *reinterpret_cast<PrepSmem<N, M>*>(dsm32);
    ModelConst<N, M>& mc = *reinterpret_cast<ModelConst<N, M>*>(dsm32 + ((sizeof(PrepSmem<N, M>) + 15) / 16) * 16);
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    Plan32& out = *g.s.plan;
    pdl_trigger();
    if (blockIdx.x == 0 && t == 0) g.status[HDR_GENERAL] = 0u;
    prep_inputs<N, M>(p, 0, 1, g.F, g.u, g.Q, g.H, g.d, g.R, g.m0, g.P0, g.y, g.status, g.zero,
                      blockIdx.x == 0 ? g.nzero : 0, nullptr, g.T, nullptr);
    if (blockIdx.x == 1) {   // the k = 1 element in FP64, and beside it the scans' own constants
        if (t < kFirstThreads) first_element_fp64<N, M>(p, mc, t);
        else if (w == 4) prep_consts<N, M>(p, mc, lane);
        __syncthreads();
        prep_store<N, M>(p, mc, g.mconst, g.status);
        for (int e = t; e < N; e += kPlanNT) out.b1[e] = mc.b1[e];
        for (int e = t; e < N * N; e += kPlanNT) out.C1[e] = mc.C1[sidx(e / N, e % N)];
        if (t == 0) out.ok1 = p.ok0 && p.ok1;
        return;
    }
    PlanSmem32& s = *reinterpret_cast<PlanSmem32*>(dsm32 + plan32_off());
    const tc::VS<N> vs{s.vs};
    if (t == 0) s.ok = 1;
    // Lemma 3's constants with S^-1 in place of its factor: HQ, HF; S; K = (H Q)^T S^-1, V = S^-1 H F;
    // A = F - K H F, C = Q - K H Q, J = (H F)^T V
    float *HQ = s.X, *V8 = s.W;
    {
        const int q = (t & 255) / N, a = t % N;
        float v = 0.f;
        if (t < 256) {
#pragma unroll 8
            for (int c = 0; c < N; ++c) v = fmaf(p.H[q][c], 0.5f * (p.Q[c][a] + p.Q[a][c]), v);
            HQ[q * P + a] = v;
        } else {
#pragma unroll 8
            for (int c = 0; c < N; ++c) v = fmaf(p.H[q][c], p.F[c][a], v);
            s.HF[q * P + a] = v;
            out.HF[q * N + a] = v;
            s.H[q * P + a] = p.H[q][a];
            out.H[q * N + a] = p.H[q][a];
        }
    }
    __syncthreads();
    if (t < 64) {
        const int a = t / M, b = t % M;
        const float r = 0.5f * (p.R[a][b] + p.R[b][a]);
        s.R[t] = r;
        out.R[t] = r;
        float v = r;
#pragma unroll 8
        for (int c = 0; c < N; ++c) v = fmaf(HQ[a * P + c], p.H[b][c], v);
        s.S[t] = v;
    }
    __syncthreads();
    if (w == 0) {
        float cond;
        const bool ok = warp_inverse<M>(s.S, s.Si, lane, cond) && cond <= kRefineCond;
        if (!__all_sync(kAll, ok) && lane == 0) s.ok = 0;
    }
    __syncthreads();
    {
        const int q = (t & 255) / N, a = t % N;
        float v = 0.f;
#pragma unroll
        for (int r = 0; r < M; ++r) v = fmaf(s.Si[q * M + r], t < 256 ? HQ[r * P + a] : s.HF[r * P + a], v);
        if (t < 256) s.KB[a * M + q] = v;
        else V8[q * P + a] = v;
    }
    __syncthreads();
    for (int e = t; e < N * N; e += kPlanNT) {
        const int a = e / N, b = e % N;
        const float qs = 0.5f * (p.Q[a][b] + p.Q[b][a]);
        float va = p.F[a][b], vc = qs, vj = 0.f;
#pragma unroll
        for (int q = 0; q < M; ++q) {
            va = fmaf(-s.KB[a * M + q], s.HF[q * P + b], va);
            vc = fmaf(-s.KB[a * M + q], HQ[q * P + b], vc);
            vj = fmaf(s.HF[q * P + a], V8[q * P + b], vj);
        }
        s.A[0][a * P + b] = va;
        s.C[0][a * P + b] = vc;
        s.J[0][a * P + b] = vj;
        out.F[e] = p.F[a][b];
        out.Q[e] = qs;
    }
    if (t < N) out.u[t] = p.u[t];
    if (t < M) out.d[t] = p.d[t];
    __syncthreads();
    symmetrise(s.C[0], t, kPlanNT);
    symmetrise(s.J[0], t, kPlanNT);
    __syncthreads();
    // ---- doubling: 16 warps, four to a product
    int cur = 0;
    const int grp = w >> 2, gw = w & 3;
#pragma unroll 1
    for (int lev = 0; lev < 7; ++lev, cur ^= 1) {
        const float *A = s.A[cur], *C = s.C[cur], *J = s.J[cur];
        float *A2 = s.A[cur ^ 1], *C2 = s.C[cur ^ 1], *J2 = s.J[cur ^ 1];
        mprod<2, false, false>(C, J, s.Mx, w, lane);
        __syncthreads();
        add_identity(s.Mx, t);
        __syncthreads();
        if (w == 0) {
            bool ok = true;
            const float cond = tc::gj_inverse<N>(s.Mx, s.Mi, vs, ok);
            if (!(__all_sync(kAll, ok) && cond <= kRefineCond) && lane == 0) s.ok = 0;
        } else {   // the powers, beside it
            store32(out.EA[lev], A, t - 32, kPlanNT - 32);
            store32(out.EC[lev], C, t - 32, kPlanNT - 32);
            store32(out.EJ[lev], J, t - 32, kPlanNT - 32);
        }
        __syncthreads();
        if (grp == 0) mprod<8, false, false>(A, s.Mi, s.X, gw, lane);
        else if (grp == 1) mprod<8, false, false>(s.Mi, C, s.W, gw, lane);
        else if (grp == 2) mprod<8, true, false>(s.Mi, J, s.V, gw, lane);
        __syncthreads();
        if (grp == 0) mprod<8, false, false>(s.X, A, A2, gw, lane);
        else if (grp == 1) mprod<8, false, false>(A, s.W, s.Y, gw, lane);
        else if (grp == 2) mprod<8, false, false>(s.V, A, s.Z, gw, lane);
        __syncthreads();
        if (grp == 0) mprod<8, false, true>(s.Y, A, C2, gw, lane, C);
        else if (grp == 1) mprod<8, true, false>(A, s.Z, J2, gw, lane, J);
        __syncthreads();
        symmetrise(C2, t, kPlanNT);
        symmetrise(J2, t, kPlanNT);
        __syncthreads();
    }
    // ---- settled covariances, gains, Phi
    const float *A = s.A[cur], *Pf = s.C[cur], *J = s.J[cur];
    float* Fs = s.V;
    for (int e = t; e < N * N; e += kPlanNT) Fs[(e / N) * P + e % N] = p.F[e / N][e % N];
    __syncthreads();
    if (grp == 0) mprod<8, false, false>(Fs, Pf, s.X, gw, lane);          // F P
    else if (grp == 1) mprod<8, false, false>(Pf, J, s.Mx, gw, lane);     // P J
    store32(out.Pf, Pf, t, kPlanNT);
    if (w == 15) {
        s.sd[lane] = sqrtf(Pf[lane * P + lane]);
        out.sd[lane] = s.sd[lane];
        out.rsd[lane] = 1.f / s.sd[lane];
    }
    __syncthreads();
    add_identity(s.Mx, t);
    if (grp == 1) mprod<8, false, true>(s.X, Fs, s.Y, gw, lane);          // F P F^T
    __syncthreads();
    for (int e = t; e < N * N; e += kPlanNT) {
        const int a = e / N, b = e % N;
        if (b <= a) {
            const float v = 0.5f * (s.Y[a * P + b] + s.Y[b * P + a]) + 0.5f * (p.Q[a][b] + p.Q[b][a]);
            s.Z[a * P + b] = v;                                           // P-
            s.Z[b * P + a] = v;
        }
    }
    __syncthreads();
    if (w == 0) {
        bool ok = true;
        const float cond = tc::gj_inverse<N>(s.Mx, s.Mi, vs, ok);         // (I + P J)^-1
        if (!(__all_sync(kAll, ok) && cond <= kRefineCond) && lane == 0) s.ok = 0;
    } else if (w == 1) {
        for (int q = 0; q < M; ++q) {
            float v = 0.f;
            for (int c = 0; c < N; ++c) v = fmaf(s.H[q * P + c], s.Z[c * P + lane], v);
            s.HP[q * P + lane] = v;
        }
        __syncwarp();
        const bool ok = gains(s.HP, s.H, s.HF, s.R, s.S, s.Si, out.K, out.B, s.KB, lane);
        if (!ok && lane == 0) s.ok = 0;
        // the lift H^T (H H^T)^-1, zero where that is singular (S, Si are free again)
        __syncwarp();
        for (int e = lane; e < M * M; e += 32) {
            float v = 0.f;
            for (int c = 0; c < N; ++c) v = fmaf(s.H[(e / M) * P + c], s.H[(e % M) * P + c], v);
            s.S[e] = v;
        }
        __syncwarp();
        float cond;
        const bool lok = __all_sync(kAll, warp_inverse<M>(s.S, s.Si, lane, cond) && cond <= kRefineCond);
        __syncwarp();
        for (int q = 0; q < M; ++q) {
            float v = 0.f;
            for (int r = 0; r < M; ++r) v = fmaf(s.H[r * P + lane], s.Si[r * M + q], v);
            out.Lf[lane * M + q] = lok ? v : 0.f;
        }
    } else if (w == 2) {
        const float n = scaled_norm32(A, s.sd, lane, false);
        if (lane == 0) out.nA = n;
    }
    __syncthreads();
    float *f0 = s.A[cur ^ 1], *f1 = s.X, *o0 = s.C[cur ^ 1], *o1 = s.Y;
    for (int e = t; e < N * N; e += kPlanNT) {
        const int a = e / N, b = e % N;
        float v = Fs[a * P + b], o = 0.f;
        for (int q = 0; q < M; ++q) {
            v = fmaf(-s.KB[a * M + q], s.HF[q * P + b], v);
            o = fmaf(s.KB[256 + a * M + q], s.HF[q * P + b], o);
        }
        f0[a * P + b] = v;                                                // Phi = F - K H F
        o0[a * P + b] = o;                                                // O_1 = F^T H^T S^-1 H F
    }
    if (grp == 3) mprod<8, false, false>(s.Mi, Pf, s.W, gw, lane);        // Ps = (I + P J)^-1 P
    __syncthreads();
    symmetrise(s.W, t, kPlanNT);
    symmetrise(o0, t, kPlanNT);
    __syncthreads();
    store32(out.Ps, s.W, t, kPlanNT);
    store32(out.Ph, f0, t, kPlanNT);
    store32_t(out.PhT, f0, t, kPlanNT);
    // ---- powers
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
        if (i < 7) store32(out.PW[i], f0, t, kPlanNT);
        store32(out.OW[i], o0, t, kPlanNT);
        if (i == 5) { store32(out.P32, f0, t, kPlanNT); store32_t(out.P32T, f0, t, kPlanNT); }
        if (grp < 2) mprod<4, false, false>(f0, f0, f1, w, lane);
        else if (i < 7) mprod<4, false, false>(o0, f0, s.Z, w - 8, lane);
        __syncthreads();
        if (i < 7) {
            if (grp < 2) mprod<4, true, false>(f0, s.Z, o1, w, lane, o0); // O_2h = O_h + Phi^hT O_h Phi^h
            __syncthreads();
            symmetrise(o1, t, kPlanNT);
            __syncthreads();
            float* x = o0; o0 = o1; o1 = x;
        }
        float* x = f0; f0 = f1; f1 = x;
    }
    if (w == 0) {
        const float nf = scaled_norm32(f0, s.sd, lane, false), nd = scaled_norm32(f0, s.sd, lane, true);
        if (lane == 0) {
            out.nphi = nf;
            out.ndual = nd;
            // wait settings of the look-back are a test's: it wants the scans
            out.ok = (s.ok != 0 && nf <= kStPowTol && nd <= kStPowTol && g.status[HDR_WAIT] == 0u &&
                      g.status[HDR_FIRST_TILE] == 0u) ? 1 : 0;
        }
    }
}

// ---------------------------------------------------------------- vector recursions, one warp each
struct WarpBuf {
    float x[N], z[N];
};

KS_DEV void load_row(const float* __restrict__ g, int lane, float (&r)[N]) {
#pragma unroll
    for (int c = 0; c < N; c += 4) {
        const float4 t = *reinterpret_cast<const float4*>(g + lane * N + c);
        r[c] = t.x; r[c + 1] = t.y; r[c + 2] = t.z; r[c + 3] = t.w;
    }
}
KS_DEV void load_row8(const float* __restrict__ g, int lane, float (&r)[M]) {
#pragma unroll
    for (int c = 0; c < M; c += 4) {
        const float4 t = *reinterpret_cast<const float4*>(g + lane * M + c);
        r[c] = t.x; r[c + 1] = t.y; r[c + 2] = t.z; r[c + 3] = t.w;
    }
}
// X v with lane a holding row a of X; v through the warp's buffer.
KS_DEV float mv(const float (&X)[N], float v, float* buf, int lane) {
    __syncwarp();
    buf[lane] = v;
    __syncwarp();
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int c = 0; c < N; c += 4) {
        const float4 t = *reinterpret_cast<const float4*>(buf + c);
        a0 = fmaf(X[c], t.x, a0);
        a1 = fmaf(X[c + 1], t.y, a1);
        a2 = fmaf(X[c + 2], t.z, a2);
        a3 = fmaf(X[c + 3], t.w, a3);
    }
    return (a0 + a1) + (a2 + a3);
}
// sum_q r[q] e_q with e_q on lanes 4 q .. 4 q + 3.
KS_DEV float mv8(const float (&r)[M], float e) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < M; ++q) s = fmaf(r[q], __shfl_sync(kAll, e, 4 * q), s);
    return s;
}

// Constants of the filter step in registers: row a of F, an eighth of a row of
// H (lane 4 q + i: H[q][8 i .. 8 i + 7]).
struct Step32 {
    float F[N], Hq[8], u, d;
    KS_DEV void load(const Plan32& p, int lane) {
        load_row(p.F, lane, F);
#pragma unroll
        for (int c = 0; c < 8; ++c) Hq[c] = p.H[lane * 8 + c];
        u = p.u[lane];
        d = p.d[lane >> 2];
    }
    // x <- F x + u + K e; returns e_q on lanes 4 q..4 q + 3, yq: y[q] there.
    KS_DEV float step(float& x, const float (&K)[M], float yq, WarpBuf& b, int lane) const {
        const float mp = u + mv(F, x, b.x, lane);
        b.z[lane] = mp;
        __syncwarp();
        float s = 0.f;
#pragma unroll
        for (int c = 0; c < 8; c += 4) {
            const float4 t = *reinterpret_cast<const float4*>(b.z + (lane & 3) * 8 + c);
            s = fmaf(Hq[c], t.x, s);
            s = fmaf(Hq[c + 1], t.y, s);
            s = fmaf(Hq[c + 2], t.z, s);
            s = fmaf(Hq[c + 3], t.w, s);
        }
        s += __shfl_xor_sync(kAll, s, 1);
        s += __shfl_xor_sync(kAll, s, 2);
        const float e = (yq - d) - s;
        x = mp + mv8(K, e);
        return e;
    }
};

// The start guess of a chunk: the lift of its first measurement.
KS_DEV float lift32(const Plan32& p, const float* __restrict__ y, int lane) {
    float r[M];
    load_row8(p.Lf, lane, r);
    return mv8(r, y[lane >> 2] - p.d[lane >> 2]);
}

// ---------------------------------------------------------------- rows, and the chunks' first pass
constexpr int kRowNT = 256;
struct RowSmem32 {
    float Ph[2][MATF], O[2][MATF], X[MATF], Y[MATF], Mx[MATF], Mi[MATF], D[MATF], Pk[MATF], Pf[MATF];
    float H[M * P], HF[M * P], HP[M * P], R[64], S[64], Si[64], vs[tc::VS<N>::FLOATS];
    WarpBuf wb[8];
    float yb[8][(kS32Chunk + 1) * M];
    alignas(128) float pat[1024];
};

// n floats of a warp's measurements into its buffer (all in flight at once; a
// step is shorter than a load).
KS_DEV void stage(float* __restrict__ dst, const float* __restrict__ src, int n, int lane) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 9; ++i)
        if (lane + 32 * i < n) cp_async4(dst + lane + 32 * i, src + lane + 32 * i);
    cp_async_wait_all();
    __syncwarp();
}

// A chunk's constant covariance rows go out as bulk copies of a shared-memory
// row, one beside each step of the chunk's recursion: the memory takes them no
// faster than it writes, and a step is longer than its share of that.
KS_DEV void fill_row(float* __restrict__ dst, const float* pat, int64_t r, int64_t end, int lane) {
    if (lane == 0 && r < end) bulk_store(dst + r * 1024, pat, 4096u);
}

__global__ void __launch_bounds__(kRowNT) rows32_kernel(Args32 g) {
    extern __shared__ __align__(128) char dsm32[];
    RowSmem32& s = *reinterpret_cast<RowSmem32*>(dsm32);
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const Plan32& p = *g.s.plan;
    pdl_wait();
    bool okp, narrow;
    {   // the chain's checks, and the transient of P_1 (relative to P) after 128 steps
        float f = p.C1[lane * 33] * p.rsd[lane] * p.rsd[lane];
        narrow = __any_sync(kAll, !(f >= kStNarrow));
        if (!(f < 1e18f)) f = 1e18f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) f = fmaxf(f, __shfl_xor_sync(kAll, f, o));
        okp = p.ok != 0 && p.ok1 != 0 && fmaxf(f, 1.f) * p.nA * p.nA <= kStCovTol;
    }
    if (!okp) {
        if (blockIdx.x == 0 && t == 0) atomicOr(g.status + HDR_GENERAL, 1u);
        return;
    }
    pdl_trigger();   // not before: what follows is to know whether the plan passed (gate_closed)
    const int64_t T = g.T;
    if (blockIdx.x >= kS32Head) {
        // ---- eight chunks: one pass from the guess, what it misses the next chunk's guess by
        const int64_t c = (blockIdx.x - kS32Head) * 8 + w, r0 = kS32Head + c * kS32Chunk;
        const int64_t fend = g.keep ? T : 0;          // constant filtered rows: all of them
        for (int e = t; e < 1024; e += kRowNT) s.pat[e] = p.Pf[e];
        fence_proxy_async();
        __syncthreads();
        if (r0 + kS32Chunk < T) {
            Step32 st;
            st.load(p, lane);
            float K[M];
            load_row8(p.K, lane, K);
            float* y = s.yb[w];
            stage(y, g.y + r0 * M, (kS32Chunk + 1) * M, lane);
            float x = lift32(p, y, lane);
#pragma unroll 1
            for (int i = 0; i < kS32Chunk; ++i) {
                st.step(x, K, y[i * M + (lane >> 2)], s.wb[w], lane);
                fill_row(g.fc, s.pat, r0 + i, fend, lane);
            }
            g.s.miss[c * 32 + lane] = x - lift32(p, y + kS32Chunk * M, lane);
        } else {                                      // the last chunk's miss is not needed
            for (int i = 0; i < kS32Chunk; ++i) fill_row(g.fc, s.pat, r0 + i, fend, lane);
        }
        bulk_commit();
        bulk_wait_read_all();
        return;
    }
    // ---- head row k and the k-th row from the end
    const int k = blockIdx.x;
    bool bad = false;
    const tc::VS<N> vs{s.vs};
    load32(s.Pf, p.Pf, t, kRowNT);
    for (int e = t; e < M * N; e += kRowNT) {
        s.H[(e / N) * P + e % N] = p.H[e];
        s.HF[(e / N) * P + e % N] = p.HF[e];
    }
    if (t < 64) s.R[t] = p.R[t];
    int cur = 0;
    bool have = false;
#pragma unroll 1
    for (int i = 0; i < 7; ++i) {                     // Phi^k, O_k from the bits of k
        if (!(k >> i & 1)) continue;
        if (!have) {
            load32(s.Ph[0], p.PW[i], t, kRowNT);
            load32(s.O[0], p.OW[i], t, kRowNT);
            __syncthreads();
            have = true;
            continue;
        }
        load32(s.X, p.PW[i], t, kRowNT);
        load32(s.Y, p.OW[i], t, kRowNT);
        __syncthreads();
        if (w < 4) mprod<8, false, false>(s.Ph[cur], s.X, s.Ph[cur ^ 1], w, lane);
        else mprod<8, false, false>(s.O[cur], s.X, s.Mx, w - 4, lane);
        __syncthreads();
        mprod<4, true, false>(s.X, s.Mx, s.O[cur ^ 1], w, lane, s.Y);
        __syncthreads();
        cur ^= 1;
        symmetrise(s.O[cur], t, kRowNT);
        __syncthreads();
    }
    const float *Phk = s.Ph[cur], *Ok = s.O[cur];
    // (I + L R)^-1 of two symmetric matrices into Mi, its Skeel condition tested
    // (see inverse_ixj)
    auto inverse_of = [&](const float* L, const float* R) {
        mprod<4, false, false>(L, R, s.Mx, w, lane);
        __syncthreads();
        add_identity(s.Mx, t);
        __syncthreads();
        if (w == 0) {
            bool ok = true;
            tc::gj_inverse<N>(s.Mx, s.Mi, vs, ok);
            float e = 0.f, c = 0.f;
#pragma unroll
            for (int q = 0; q < N; q += 4) {
                const float4 v = *reinterpret_cast<const float4*>(s.Mx + lane * P + q);
                e += (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
            }
#pragma unroll
            for (int q = 0; q < N; q += 4) {
                const float4 v = *reinterpret_cast<const float4*>(s.Mi + lane * P + q);
                c = fmaf(fabsf(v.x), __shfl_sync(kAll, e, q), c);
                c = fmaf(fabsf(v.y), __shfl_sync(kAll, e, q + 1), c);
                c = fmaf(fabsf(v.z), __shfl_sync(kAll, e, q + 2), c);
                c = fmaf(fabsf(v.w), __shfl_sync(kAll, e, q + 3), c);
            }
            if (!__all_sync(kAll, ok && c <= kHeadCond)) bad = true;
        }
        __syncthreads();
    };
    if (narrow) {   // P_1 through the element powers of the bits of k
        load32(s.Pk, p.C1, t, kRowNT);
#pragma unroll 1
        for (int i = 0; i < 7; ++i) {
            if (!(k >> i & 1)) continue;
            load32(s.X, p.EJ[i], t, kRowNT);
            load32(s.Y, p.EA[i], t, kRowNT);
            load32(s.D, p.EC[i], t, kRowNT);
            __syncthreads();
            inverse_of(s.Pk, s.X);
            mprod<4, false, false>(s.Mi, s.Pk, s.X, w, lane);
            __syncthreads();
            mprod<4, false, false>(s.Y, s.X, s.Mx, w, lane);
            __syncthreads();
            mprod<4, false, true>(s.Mx, s.Y, s.Pk, w, lane, s.D);
            __syncthreads();
            symmetrise(s.Pk, t, kRowNT);
            __syncthreads();
        }
        __syncthreads();
    }
    for (int e = t; e < N * N; e += kRowNT) {
        const int i = (e / N) * P + e % N;
        s.D[i] = (narrow ? s.Pk[i] : p.C1[e]) - s.Pf[i];
    }
    __syncthreads();
    if (!narrow) {
        if (k > 0) {
            inverse_of(s.D, Ok);
            mprod<4, false, false>(s.Mi, s.D, s.X, w, lane);
            __syncthreads();
            mprod<4, false, false>(Phk, s.X, s.Y, w, lane);
            __syncthreads();
            mprod<4, false, true>(s.Y, Phk, s.D, w, lane);
            __syncthreads();
            symmetrise(s.D, t, kRowNT);
            __syncthreads();
        }
        for (int e = t; e < N * N; e += kRowNT) {
            const int i = (e / N) * P + e % N;
            s.Pk[i] = k == 0 ? p.C1[e] : s.Pf[i] + s.D[i];
        }
        __syncthreads();
    }
    store32(g.fc + (int64_t)k * 1024, s.Pk, t, kRowNT);
    // the next row's gain
    if (k + 1 < kS32Head) {
        load32(s.X, p.F, t, kRowNT);
        __syncthreads();
        mprod<4, false, false>(s.X, s.Pk, s.Y, w, lane);
        __syncthreads();
        mprod<4, false, true>(s.Y, s.X, s.Mx, w, lane);
        __syncthreads();
        for (int e = t; e < N * N; e += kRowNT) {
            const int a = e / N, b = e % N;
            s.Mi[a * P + b] = 0.5f * (s.Mx[a * P + b] + s.Mx[b * P + a]) + p.Q[e];
        }
        __syncthreads();
        {   // H P-: warp q its row
            float v = 0.f;
            for (int c = 0; c < N; ++c) v = fmaf(s.H[w * P + c], s.Mi[c * P + lane], v);
            s.HP[w * P + lane] = v;
        }
        __syncthreads();
        if (w == 0) {
            const int64_t o = (int64_t)(k + 1) * 256;
            if (!gains(s.HP, s.H, s.HF, s.R, s.S, s.Si, g.s.Kr + o, g.s.Br + o, nullptr, lane)) bad = true;
        }
        __syncthreads();
    }
    // the transition of rows k+1..k+16 for the head's chunks
    if (k % 16 == 0 && k > 0 && k < 112) {
        load32(s.X, p.OW[4], t, kRowNT);
        load32(s.Y, p.PW[4], t, kRowNT);
        __syncthreads();
        inverse_of(s.D, s.X);
        mprod<4, false, false>(s.Y, s.Mi, s.X, w, lane);
        __syncthreads();
        store32(g.s.Psi + (k / 16) * 1024, s.X, t, kRowNT);
        __syncthreads();
    }
    if (g.sc != nullptr) {
        // smoothed head row: (I - P O_128) (I + D_k O_128)^-1 P_k
        load32(s.X, p.OW[7], t, kRowNT);
        __syncthreads();
        inverse_of(s.D, s.X);
        mprod<4, false, false>(s.Mi, s.Pk, s.Y, w, lane);
        __syncthreads();
        mprod<4, false, false>(s.X, s.Y, s.Mx, w, lane);
        __syncthreads();
        mprod<4, false, false>(s.Pf, s.Mx, s.Mi, w, lane, s.Y, -1.f);
        __syncthreads();
        symmetrise(s.Mi, t, kRowNT);
        __syncthreads();
        store32(g.sc + (int64_t)k * 1024, s.Mi, t, kRowNT);
        // the k-th row from the end: P - P O_k P
        if (k > 0) {
            mprod<4, false, false>(s.Pf, Ok, s.X, w, lane);
            __syncthreads();
            mprod<4, false, false>(s.X, s.Pf, s.Y, w, lane, s.Pf, -1.f);
            __syncthreads();
            symmetrise(s.Y, t, kRowNT);
            __syncthreads();
        }
        store32(g.sc + (T - 1 - k) * 1024, k > 0 ? s.Y : s.Pf, t, kRowNT);
    }
    if (bad && lane == 0) atomicOr(g.status + HDR_GENERAL, 1u);
}

// ---------------------------------------------------------------- forward
constexpr int kFwdNT = 256;
constexpr int kS32Fwd = 18;         // rows of a chunk whose smoothed covariance the forward kernel fills
struct FwdSmem32 {
    WarpBuf wb[8];
    float guess[9][N], miss[8][N], d[8][N], xlast[N];
    float eps[8][kS32Chunk * M];
    alignas(128) float pat[1024];
};

// Whether the scans are wanted already (one answer for the whole block: other
// blocks of the same launch may ask for them meanwhile).
KS_DEV bool general_set(const uint32_t* status) {
    __shared__ int stop;
    if (threadIdx.x == 0) stop = *(const volatile uint32_t*)(status + HDR_GENERAL) != 0u;
    __syncthreads();
    return stop != 0;
}

__global__ void __launch_bounds__(kFwdNT) forward32_kernel(Args32 g) {
    extern __shared__ __align__(128) char dsm32[];
    FwdSmem32& s = *reinterpret_cast<FwdSmem32*>(dsm32);
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const Plan32& p = *g.s.plan;
    if (!general_wanted(g.status)) pdl_trigger();
    pdl_wait();
    if (general_set(g.status)) return;
    const int64_t T = g.T, nch = (T - kS32Head + kS32Chunk - 1) / kS32Chunk;
    const int64_t c = (int64_t)blockIdx.x * 8 + w, r0 = kS32Head + c * kS32Chunk;
    const bool head = blockIdx.x == 0;
    bool bad = false;
    // constant smoothed rows, all but the last 128 (the first kS32Fwd of each
    // chunk here, the others in the reverse kernel)
    const int64_t fend = g.sc != nullptr ? T - kS32Head : 0;
    for (int e = t; e < 1024; e += kFwdNT) s.pat[e] = p.Ps[e];
    fence_proxy_async();
    __syncthreads();
    Step32 st;
    st.load(p, lane);
    float P32[N];
    load_row(p.P32, lane, P32);
    float d = 0.f;
    if (head) {
        // head chunk w: rows 16 w + 1 .. 16 w + 16 (the last: .. 127), its own gains
        const int a = 16 * w, cnt = w < 7 ? 16 : 15;
        float* y = s.eps[w];
        stage(y, g.y + (int64_t)(a + 1) * M, cnt * M, lane);
        const float guess = w == 0 ? p.b1[lane] : lift32(p, g.y + (int64_t)a * M, lane);
        s.guess[w][lane] = guess;
        auto pass = [&](float x, bool write) {
            float K[M];
            load_row8(g.s.Kr + (int64_t)(a + 1) * 256, lane, K);
#pragma unroll 1
            for (int i = 0; i < cnt; ++i) {
                float Kn[M];
                load_row8(g.s.Kr + (int64_t)(a + 1 + (i + 1 < cnt ? i + 1 : i)) * 256, lane, Kn);
                const float e = st.step(x, K, y[i * M + (lane >> 2)], s.wb[w], lane);
                if (write) {
                    g.fm[(int64_t)(a + 1 + i) * N + lane] = x;
                    if ((lane & 3) == 0) g.s.eps[(int64_t)(a + 1 + i) * M + (lane >> 2)] = e;
                }
#pragma unroll
                for (int q = 0; q < M; ++q) K[q] = Kn[q];
            }
            return x;
        };
        if (w < 7) s.miss[w][lane] = pass(guess, false);
        __syncthreads();
        if (w == 0) {                                  // d_{h+1} = Psi_h d_h + (miss of chunk h)
            float dd = s.miss[0][lane] - s.guess[1][lane];
            s.d[0][lane] = 0.f;
            s.d[1][lane] = dd;
#pragma unroll 1
            for (int h = 1; h < 7; ++h) {
                float X[N];
                load_row(g.s.Psi + h * 1024, lane, X);
                dd = mv(X, dd, s.wb[0].x, lane) + (s.miss[h][lane] - s.guess[h + 1][lane]);
                s.d[h + 1][lane] = dd;
            }
            g.fm[lane] = p.b1[lane];
        }
        __syncthreads();
        const float x = pass(guess + s.d[w][lane], true);
        if (w == 7) s.xlast[lane] = x;
        bad = !(fabsf(x) < 1e30f);
        __syncthreads();
        // the first eight chunks after the head start exactly
        if (w == 0) {
            float dd = s.xlast[lane] - lift32(p, g.y + (int64_t)kS32Head * M, lane);
#pragma unroll 1
            for (int h = 0; h < 8; ++h) {
                s.d[h][lane] = dd;
                dd = mv(P32, dd, s.wb[0].x, lane) + (h + 1 < nch ? g.s.miss[h * 32 + lane] : 0.f);
            }
        }
        __syncthreads();
        d = s.d[w][lane];
        // chunk c + 8 leaves out what lies before chunk c, which only this block sees
        if (c + kS32Back < nch && !(p.nphi * fabsf(d) * p.rsd[lane] <= kStMeanTol)) bad = true;
    } else if (c < nch) {
        float m[kS32Back];
#pragma unroll
        for (int i = 0; i < kS32Back; ++i) m[i] = g.s.miss[(c - 1 - i) * 32 + lane];
#pragma unroll
        for (int i = kS32Back - 1; i >= 0; --i) d = mv(P32, d, s.wb[w].x, lane) + m[i];
        if (!(p.nphi * fabsf(d) * p.rsd[lane] <= kStMeanTol)) bad = true;
    }
    if (c < nch) {
        const int cnt = (int)min((int64_t)kS32Chunk, T - r0);
        float* ep = s.eps[w];                         // measurements, then innovations
        stage(ep, g.y + r0 * M, cnt * M, lane);
        float K[M];
        load_row8(p.K, lane, K);
        float x = lift32(p, ep, lane) + d;
#pragma unroll 1
        for (int i = 0; i < cnt; ++i) {
            const float e = st.step(x, K, ep[i * M + (lane >> 2)], s.wb[w], lane);
            g.fm[(r0 + i) * N + lane] = x;
            if ((lane & 3) == 0) ep[i * M + (lane >> 2)] = e;
            if (i < kS32Fwd) fill_row(g.sc, s.pat, r0 + i, fend, lane);
        }
        if (!(fabsf(x) < 1e30f)) bad = true;
        __syncwarp();
        if (g.sm != nullptr) {
            // innovations for the reverse pass; the chunk's adjoint from zero
            for (int i = lane; i < cnt * M; i += 32) g.s.eps[r0 * M + i] = ep[i];
            float PhT[N], B[M];
            load_row(p.PhT, lane, PhT);
            load_row8(p.B, lane, B);
            float l = 0.f;
#pragma unroll 1
            for (int i = cnt - 1; i >= 0; --i) l = mv(PhT, l, s.wb[w].x, lane) + mv8(B, ep[i * M + (lane >> 2)]);
            g.s.mu[c * 32 + lane] = l;
        }
    }
    bulk_commit();
    if (__any_sync(kAll, bad) && lane == 0) atomicOr(g.status + HDR_GENERAL, 1u);
    bulk_wait_read_all();
}

// ---------------------------------------------------------------- reverse
struct RevSmem32 {
    WarpBuf wb[8];
    float nu[8][N], l[9][N];
    float eps[8][kS32Chunk * M];
    alignas(128) float pat[1024];
};

__global__ void __launch_bounds__(256, 2) reverse32_kernel(Args32 g) {
    __shared__ RevSmem32 s;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    const Plan32& p = *g.s.plan;
    if (!general_wanted(g.status)) pdl_trigger();
    pdl_wait();
    if (general_set(g.status)) return;
    const int64_t T = g.T, nch = (T - kS32Head + kS32Chunk - 1) / kS32Chunk;
    float P32T[N];
    load_row(p.P32T, lane, P32T);
    // the adjoint that enters chunk c from the eight chunks after it
    auto enter = [&](int64_t c) {
        float l = 0.f, m[kS32Back];
#pragma unroll
        for (int i = 0; i < kS32Back; ++i) m[i] = c + 1 + i < nch ? g.s.mu[(c + 1 + i) * 32 + lane] : 0.f;
#pragma unroll
        for (int i = kS32Back - 1; i >= 0; --i) l = mv(P32T, l, s.wb[w].x, lane) + m[i];
        return l;
    };
    bool bad = false;
    if (blockIdx.x == 0) {   // the head
        // chunk w: rows 16 w + 16 (the last: 127) down to 16 w + 1, from the adjoint at its top row
        const int a = 16 * w, cnt = w < 7 ? 16 : 15;
        float FT[N], H[M];
#pragma unroll
        for (int c = 0; c < N; ++c) FT[c] = p.F[c * N + lane];
#pragma unroll
        for (int q = 0; q < M; ++q) H[q] = p.H[q * N + lane];
        // l_{j-1} = Phi_j^T l_j + B_j e_j, Phi_j^T l = F^T (l - H^T K_j^T l)
        auto back = [&](int j, float l) {
            const float* K = g.s.Kr + (int64_t)j * 256;
            __syncwarp();
            s.wb[w].z[lane] = l;
            __syncwarp();
            float k = 0.f;                              // lane 4 q + i: a quarter of (K^T l)_q
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int r = (lane & 3) * 8 + c;
                k = fmaf(K[r * M + (lane >> 2)], s.wb[w].z[r], k);
            }
            k += __shfl_xor_sync(kAll, k, 1);
            k += __shfl_xor_sync(kAll, k, 2);
            const float v = l - mv8(H, k);
            float B[M];
            load_row8(g.s.Br + (int64_t)j * 256, lane, B);
            return mv(FT, v, s.wb[w].x, lane) + mv8(B, g.s.eps[(int64_t)j * M + (lane >> 2)]);
        };
        if (w == 7) {
            float l = enter(-1);
            if (!(p.ndual * fabsf(l) * p.sd[lane] <= kStMeanTol)) bad = true;
            s.l[8][lane] = l;
            for (int i = cnt; i >= 1; --i) l = back(a + i, l);
            s.l[7][lane] = l;                           // at row 112
        } else if (w > 0) {
            float l = 0.f;
            for (int i = cnt; i >= 1; --i) l = back(a + i, l);
            s.nu[w][lane] = l;
        }
        __syncthreads();
        if (w == 0) {
            float l = s.l[7][lane];
#pragma unroll 1
            for (int h = 6; h >= 1; --h) {              // l at row 16 h = Psi_h^T (l at row 16 h + 16) + nu_h
                float X[N];
#pragma unroll
                for (int c = 0; c < N; ++c) X[c] = g.s.Psi[h * 1024 + c * N + lane];
                l = mv(X, l, s.wb[0].x, lane) + s.nu[h][lane];
                s.l[h][lane] = l;
            }
        }
        __syncthreads();
        float l = s.l[w + 1][lane];
        auto smooth_row = [&](int j, float lj) {
            float X[N];
#pragma unroll
            for (int c = 0; c < N; ++c) X[c] = g.fc[(int64_t)j * 1024 + c * N + lane];
            const float v = g.fm[(int64_t)j * N + lane] + mv(X, lj, s.wb[w].x, lane);
            g.sm[(int64_t)j * N + lane] = v;
            if (!(fabsf(v) < 1e30f)) bad = true;
        };
        for (int i = cnt; i >= 1; --i) {
            smooth_row(a + i, l);
            l = back(a + i, l);
        }
        if (w == 0) smooth_row(0, l);
    } else {
        const int64_t c = (int64_t)(blockIdx.x - 1) * 8 + w, r0 = kS32Head + c * kS32Chunk;
        for (int e = t; e < 1024; e += 256) s.pat[e] = p.Ps[e];
        fence_proxy_async();
        __syncthreads();
        if (c < nch) {
            const int cnt = (int)min((int64_t)kS32Chunk, T - r0);
            float PhT[N], Pr[N], B[M];
            load_row(p.PhT, lane, PhT);
            load_row(p.Pf, lane, Pr);
            load_row8(p.B, lane, B);
            stage(s.eps[w], g.s.eps + r0 * M, cnt * M, lane);
            const int64_t fend = T - kS32Head;
            float l = enter(c);
            // chunk c - 8 (the head before chunk 7) leaves out what enters here
            if (nch > kS32Back && !(p.ndual * fabsf(l) * p.sd[lane] <= kStMeanTol)) bad = true;
            constexpr int AH = 4;                       // filtered means loaded ahead
            float mn[AH];
#pragma unroll
            for (int j = 0; j < AH; ++j) mn[j] = g.fm[(r0 + max(cnt - 1 - j, 0)) * N + lane];
            const float* ep = s.eps[w];
#pragma unroll 1
            for (int i0 = cnt - 1; i0 >= 0; i0 -= AH) {
                float m[AH];
#pragma unroll
                for (int j = 0; j < AH; ++j) {
                    m[j] = mn[j];
                    mn[j] = g.fm[(r0 + max(i0 - AH - j, 0)) * N + lane];
                }
#pragma unroll
                for (int j = 0; j < AH; ++j) {
                    const int i = i0 - j;
                    if (i < 0) break;
                    if (i >= kS32Fwd) fill_row(g.sc, s.pat, r0 + i, fend, lane);
                    g.sm[(r0 + i) * N + lane] = m[j] + mv(Pr, l, s.wb[w].x, lane);
                    // the same buffer holds l: Phi^T l needs no second broadcast
                    float a0 = 0.f, a1 = 0.f;
#pragma unroll
                    for (int q = 0; q < N; q += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(s.wb[w].x + q);
                        a0 = fmaf(PhT[q], v.x, a0);
                        a1 = fmaf(PhT[q + 1], v.y, a1);
                        a0 = fmaf(PhT[q + 2], v.z, a0);
                        a1 = fmaf(PhT[q + 3], v.w, a1);
                    }
                    l = (a0 + a1) + mv8(B, ep[i * M + (lane >> 2)]);
                }
            }
            if (!(fabsf(l) < 1e30f)) bad = true;
        }
    }
    if (__any_sync(kAll, bad) && lane == 0) atomicOr(g.status + HDR_GENERAL, 1u);
    bulk_commit();
    bulk_wait_read_all();
}

template <class K>
bool opt_in(K kernel, size_t bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
}

}  // namespace

int launch_steady32_plan(const Args32& g, cudaStream_t st) {
    constexpr size_t smem = plan32_off() + sizeof(PlanSmem32);
    static const bool ok = opt_in(plan32_kernel, smem);
    if (!ok) return KS_ECUDA;
    plan32_kernel<<<2, kPlanNT, smem, st>>>(g);
    return launch_status();
}

int launch_steady32(const Args32& g, cudaStream_t st) {
    static const bool ok = opt_in(rows32_kernel, sizeof(RowSmem32)) && opt_in(forward32_kernel, sizeof(FwdSmem32));
    if (!ok) return KS_ECUDA;
    const int nb = (int)((s32_chunks(g.T) + 7) / 8);
    int rc = launch_pdl(rows32_kernel, kS32Head + nb, kRowNT, sizeof(RowSmem32), st, g);
    if (rc) return rc;
    if ((rc = launch_pdl(forward32_kernel, nb, kFwdNT, sizeof(FwdSmem32), st, g))) return rc;
    if (g.sm == nullptr) return KS_OK;
    return launch_pdl(reverse32_kernel, 1 + nb, 256, 0, st, g);
}

}  // namespace ks
