// ks_hmmw.cuh -- the discrete-state (HMM) filter and smoother for K = 16 and
// 32 states: one K-lane group of a warp per chain of steps, lane z holding
// row z of each K x K element (Section III's Definitions 1 and 2 with sums,
// as in ks_hmm.cuh).
//
// A chain's elements are too large for one thread's registers at this K, so
// every scan runs as reduce / spine / apply launches (as the nx = 8 and
// nx = 32 Gaussian paths do):
//  * forward reduce: each warp folds its chain's step elements into one
//    Definition 1 element; warp 0 combines the block's chains in order,
//    storing each chain's exclusive in-tile prefix and the tile aggregate;
//  * spine: Kogge-Stone over the tile aggregates (one launch per level);
//  * forward apply: each chain starts from its prefix (all rows equal:
//    p(x | y_1:k) and log p(y_1:k)) and steps through its measurements writing
//    filt and loglik;
//  * reverse: smoothing as filt . beta / sum with beta(z) = p(what follows | z).
//    A spine over the same tile aggregates in reversed order, then an apply:
//    beta enters a chain through the elements of the tile's later chains, one
//    matrix-vector product each, and walks the chain backwards.  (Definition 2
//    elements folded beside the forward apply cost another K^2 products per
//    lane and step, half of the forward scan.)
// Likelihood rows are scaled to a maximum near 1 and g is kept as log g, so
// that p(y_1:k) survives long prefixes in FP32.
#pragma once

#include "ks_scan.cuh"

namespace ks {
namespace hmmw {

// Shared-memory pitches: Pi rows are read by all lanes of a chain at once
// (broadcast), so pitch K with float4 rows; element slots are written a row per
// lane with float4 stores and read by broadcast, so pitch Q (a multiple of 4,
// rows in distinct banks per quarter-warp).
template <int K>
struct Dims {
    static constexpr int Q = K + 4;
    static constexpr int SLOT = K * Q + K;       // rows, then log g
    static constexpr int FREC = K * K + K;       // global filtering record: rows, then log g
};

// A chain is K lanes of one warp (lane z = row z); 32 / K chains per warp.
template <int K>
KS_DEV unsigned gmask() {
    if constexpr (K == 32) return 0xffffffffu;
    else return ((1u << K) - 1u) << (threadIdx.x & (32 - K));
}

template <int K>
KS_DEV int glane() { return threadIdx.x & (K - 1); }

template <int K>
struct Const {
    float Pi[K * K];
    float q1[K];   // p(x_1) = pi Pi
};

// One warp's share of a filtering element: lane z holds row z and lg[z].
template <int K>
struct FRow {
    float f[K];
    float lg;
};

template <int K>
KS_DEV float group_sum(float v) {
#pragma unroll
    for (int o = K / 2; o > 0; o >>= 1) v += __shfl_xor_sync(gmask<K>(), v, o, K);
    return v;
}

template <int K>
KS_DEV float group_max(float v) {
#pragma unroll
    for (int o = K / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(gmask<K>(), v, o, K));
    return v;
}

template <int K>
KS_DEV int group_max_i(int v) {
#pragma unroll
    for (int o = K / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(gmask<K>(), v, o, K));
    return v;
}

// log g relative to its largest, all that beta needs: over a long suffix the
// sum itself would leave no bits for the differences between states.
template <int K>
KS_DEV void relative_lg(FRow<K>& r) { r.lg -= group_max<K>(r.lg); }

// Pi (pitch K) into shared memory.
template <int K>
KS_DEV void load_pi(const Const<K>* __restrict__ cg, float* __restrict__ Pi, float* q1) {
    for (int e = threadIdx.x; e < K * K; e += blockDim.x) Pi[e] = __ldg(cg->Pi + e);
    for (int e = threadIdx.x; e < K; e += blockDim.x) q1[e] = __ldg(cg->q1 + e);
}

template <int K>
KS_DEV void load_frow(const float* __restrict__ src, FRow<K>& r) {
    const int z = glane<K>();
    const float4* p = reinterpret_cast<const float4*>(src + z * K);
#pragma unroll
    for (int i = 0; i < K / 4; ++i) {
        const float4 q = __ldcg(p + i);
        r.f[4 * i] = q.x;
        r.f[4 * i + 1] = q.y;
        r.f[4 * i + 2] = q.z;
        r.f[4 * i + 3] = q.w;
    }
    r.lg = __ldcg(src + K * K + z);
}

template <int K>
KS_DEV void store_frow(float* __restrict__ dst, const FRow<K>& r) {
    const int z = glane<K>();
    float4* p = reinterpret_cast<float4*>(dst + z * K);
#pragma unroll
    for (int i = 0; i < K / 4; ++i) p[i] = make_float4(r.f[4 * i], r.f[4 * i + 1], r.f[4 * i + 2], r.f[4 * i + 3]);
    dst[K * K + z] = r.lg;
}

// A chain's element in a shared-memory slot (pitch Q rows, then lg).
template <int K>
KS_DEV void put_srow(float* __restrict__ buf, const float (&a)[K]) {
    float4* p = reinterpret_cast<float4*>(buf + glane<K>() * Dims<K>::Q);
#pragma unroll
    for (int i = 0; i < K / 4; ++i) p[i] = make_float4(a[4 * i], a[4 * i + 1], a[4 * i + 2], a[4 * i + 3]);
}

template <int K>
KS_DEV void put_frow(float* __restrict__ buf, const FRow<K>& r) {
    put_srow(buf, r.f);
    buf[K * Dims<K>::Q + glane<K>()] = r.lg;
}

// Row y of a K x K shared-memory matrix with a 16-byte-aligned pitch, as float4s.
template <int PITCH, int K>
KS_DEV void smem_row(const float* __restrict__ M, int y, float (&v)[K]) {
    const float4* p = reinterpret_cast<const float4*>(M + y * PITCH);
#pragma unroll
    for (int i = 0; i < K / 4; ++i) {
        const float4 q = p[i];
        v[4 * i] = q.x;
        v[4 * i + 1] = q.y;
        v[4 * i + 2] = q.z;
        v[4 * i + 3] = q.w;
    }
}

// 2^-e and e for the exponent e of a positive finite r.
KS_DEV float pow2_of(float r, int& e) {
    e = (int)(__float_as_uint(r) >> 23) - 127;
    return __uint_as_float((uint32_t)(127 - e) << 23);
}

// Likelihood row of step k (the same for every lane) scaled by a power of two
// to a maximum in [1, 2); returns the exponent taken out.
template <int K>
KS_DEV int lik_row2(const float* __restrict__ lik, int64_t k, float (&l)[K], Flags& bad) {
    const float4* p = reinterpret_cast<const float4*>(lik + k * K);
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < K / 4; ++i) {
        const float4 q = __ldg(p + i);
        l[4 * i] = q.x;
        l[4 * i + 1] = q.y;
        l[4 * i + 2] = q.z;
        l[4 * i + 3] = q.w;
    }
#pragma unroll
    for (int x = 0; x < K; ++x) m = fmaxf(m, l[x]);
    const bool ok = m > 0.f && m <= 3.0e38f;
    bad |= !ok;
    int e;
    const float s = pow2_of(ok ? m : 1.f, e);
#pragma unroll
    for (int x = 0; x < K; ++x) l[x] *= s;
    return e;
}

// Fold of a step element into row z: (f Pi)[z] . l, kept at a sum in [1, 2) by
// a power of two (exponents added up in ex: no division, no logarithm).
template <int K>
KS_DEV void fold_row(FRow<K>& r, int& ex, const float* __restrict__ Pi, const float (&l)[K], int le, Flags& bad) {
    float o[K];
#pragma unroll
    for (int x = 0; x < K; ++x) o[x] = 0.f;
#pragma unroll
    for (int y = 0; y < K; ++y) {
        float pr[K];
        smem_row<K>(Pi, y, pr);
#pragma unroll
        for (int x = 0; x < K; ++x) o[x] = fmaf(r.f[y], pr[x], o[x]);
    }
    float s = 0.f;
#pragma unroll
    for (int x = 0; x < K; ++x) {
        o[x] *= l[x];
        s += o[x];
    }
    bad |= !(s > 0.f);
    int e;
    const float rs = pow2_of(s, e);
#pragma unroll
    for (int x = 0; x < K; ++x) r.f[x] = o[x] * rs;
    ex += e + le;
}

// End of a fold: row of sum one, log g from the exponents and the last sum.
template <int K>
KS_DEV void fold_end(FRow<K>& r, int ex, Flags& bad) {
    float s = 0.f;
#pragma unroll
    for (int x = 0; x < K; ++x) s += r.f[x];
    bad |= !(s > 0.f);
    const float rs = 1.f / s;
#pragma unroll
    for (int x = 0; x < K; ++x) r.f[x] *= rs;
    r.lg = fmaf((float)ex, 0.693147180559945f, logf(s));
}

// Definition 1, (row z of a_i, in registers) (x) a_j (in shared memory).
template <int K>
KS_DEV void combine_row(FRow<K>& r, const float* __restrict__ ej, Flags& bad) {
    float mx = ej[K * Dims<K>::Q];
#pragma unroll
    for (int y = 1; y < K; ++y) mx = fmaxf(mx, ej[K * Dims<K>::Q + y]);
    float o[K], d = 0.f;
#pragma unroll
    for (int x = 0; x < K; ++x) o[x] = 0.f;
#pragma unroll
    for (int y = 0; y < K; ++y) {
        const float fw = r.f[y] * __expf(ej[K * Dims<K>::Q + y] - mx);
        d += fw;
        float er[K];
        smem_row<Dims<K>::Q>(ej, y, er);
#pragma unroll
        for (int x = 0; x < K; ++x) o[x] = fmaf(fw, er[x], o[x]);
    }
    bad |= !(d > 0.f);
    const float rd = 1.f / d;
#pragma unroll
    for (int x = 0; x < K; ++x) r.f[x] = o[x] * rd;
    r.lg += mx + __logf(d);
}

// The prefix (all rows equal) as a state: lane x takes p(x) from row 0.
template <int K>
KS_DEV void row0_state(const FRow<K>& r, float& p, float& L) {
    const int lane = glane<K>();
    p = 0.f;
#pragma unroll
    for (int x = 0; x < K; ++x) {
        const float v = __shfl_sync(gmask<K>(), r.f[x], 0, K);
        if (lane == x) p = v;
    }
    L = __shfl_sync(gmask<K>(), r.lg, 0, K);
}

// sum_x m[x] v(x) for a vector with v(x) on lane x, through the group's buffer
// (K floats of shared memory): one store and K / 4 broadcast loads in place of K
// shuffles.
template <int K>
KS_DEV float row_dot(const float (&m)[K], float v, float* __restrict__ buf) {
    __syncwarp(gmask<K>());
    buf[glane<K>()] = v;
    __syncwarp(gmask<K>());
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int x = 0; x < K; x += 4) {
        const float4 t = *reinterpret_cast<const float4*>(buf + x);
        a0 = fmaf(m[x], t.x, a0);
        a1 = fmaf(m[x + 1], t.y, a1);
        a2 = fmaf(m[x + 2], t.z, a2);
        a3 = fmaf(m[x + 3], t.w, a3);
    }
    return (a0 + a1) + (a2 + a3);
}

// Filtering state (lane x: p(x)) (x) step: p'(x) = (p Pi)(x) l(x) / c, with the
// lane's column of Pi in registers.
template <int K>
KS_DEV void advance_step(float& p, float& L, float& comp, const float (&col)[K], float lx, float lm, float* buf,
                         Flags& bad) {
    const float v = row_dot<K>(col, p, buf) * lx;
    const float c = group_sum<K>(v);
    bad |= !(c > 0.f);
    p = v / c;
    const float t = (lm + __logf(c)) - comp;   // Kahan-compensated running log-likelihood
    const float Ln = L + t;
    comp = (Ln - L) - t;
    L = Ln;
}

// beta(z) of an element with log weights lg followed by v(z) = (f beta')(z):
// exp(lg - max) v, rescaled by a power of two to a maximum in [1, 2).
template <int K>
KS_DEV float beta_of(float v, float lg) {
    v *= __expf(lg - group_max<K>(lg));
    int e;
    return v * pow2_of(group_max<K>(v), e);
}

// ---------------------------------------------------------------- kernels
struct Bufs {
    float* fexcl;     // [nchains][FREC] exclusive in-tile prefixes of the forward scan
    float* fspine0;   // [ntiles][FREC]
    float* fspine1;
    float* chain;     // [nchains][FREC] chain elements, for the reverse scan (null: not wanted)
    float* sspine0;   // [ntiles][FREC] tile aggregates again, for the reversed spine
    float* sspine1;
};

// NG = NW * 32 / K chains per block (one K-lane group each).
template <int K, int NW>
struct alignas(16) Smem {
    static constexpr int NG = NW * 32 / K;
    float Pi[K * K];
    float q1[K];
    int top[(NG + 3) / 4 * 4];
    float slot[NG][Dims<K>::SLOT];   // one element per chain (pitch Q rows + lg)
};

template <int K, int NW, int CH>
__global__ void __launch_bounds__(NW * 32) filter_reduce_kernel(const Const<K>* __restrict__ cg,
                                                                const float* __restrict__ lik, int64_t T, Bufs b,
                                                                uint32_t* status) {
    __shared__ Smem<K, NW> sm;
    constexpr int NG = Smem<K, NW>::NG;
    load_pi(cg, sm.Pi, sm.q1);
    __syncthreads();
    const int w = threadIdx.x / K;
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t c = (int64_t)blockIdx.x * NG + w;
    const int64_t left = nch - (int64_t)blockIdx.x * NG;
    const int nvalid = left < NG ? (int)left : NG;
    Flags bad = 0u;
    if (w < nvalid) {
        const int64_t k0 = c * CH, k1 = (k0 + CH < T) ? k0 + CH : T;
        FRow<K> r;
        float l[K];
        int ex = lik_row2(lik, k0, l, bad);
        const float* first = k0 == 0 ? sm.q1 : sm.Pi + glane<K>() * K;   // k = 1: every row p(x_1, y_1)
#pragma unroll
        for (int x = 0; x < K; ++x) r.f[x] = first[x] * l[x];
#pragma unroll 1
        for (int64_t k = k0 + 1; k < k1; ++k) {
            const int le = lik_row2(lik, k, l, bad);
            fold_row(r, ex, sm.Pi, l, le, bad);
        }
        // log g relative to the chain's largest exponent, which is kept beside it
        const int top = group_max_i<K>(ex);
        fold_end(r, ex - top, bad);
        put_frow(sm.slot[w], r);
        if (glane<K>() == 0) sm.top[w] = top;
        if (b.chain != nullptr) store_frow(b.chain + c * Dims<K>::FREC, r);
    }
    __syncthreads();
    if (w == 0) {   // in-tile combine, chain order
        FRow<K> acc;
        smem_row<Dims<K>::Q>(sm.slot[0], glane<K>(), acc.f);
        acc.lg = sm.slot[0][K * Dims<K>::Q + glane<K>()];
        int top = sm.top[0];
        auto absolute = [&](float* dst) {   // log g itself, for the prefixes
            FRow<K> q = acc;
            q.lg = fmaf((float)top, 0.693147180559945f, q.lg);
            store_frow(dst, q);
        };
#pragma unroll 1
        for (int t = 1; t < nvalid; ++t) {
            absolute(b.fexcl + ((int64_t)blockIdx.x * NG + t) * Dims<K>::FREC);
            combine_row(acc, sm.slot[t], bad);
            top += sm.top[t];
        }
        absolute(b.fspine0 + (int64_t)blockIdx.x * Dims<K>::FREC);
        if (b.chain != nullptr) {
            relative_lg<K>(acc);
            store_frow(b.sspine0 + (int64_t)blockIdx.x * Dims<K>::FREC, acc);
        }
    }
    report_flags(status, bad, kFull, (threadIdx.x & 31) == 0);
}

// Kogge-Stone level s over tile aggregates: dst[t] = src[t - s] (x) src[t]
// (prefixes), or src[t] (x) src[t + s] (suffixes).
template <bool PREFIX, int K, int NW>
__global__ void __launch_bounds__(NW * 32) spine_kernel(const float* __restrict__ src, float* __restrict__ dst,
                                                        int ntiles, int s, uint32_t* status) {
    constexpr int NG = NW * 32 / K;
    __shared__ __align__(16) float slot[NG][Dims<K>::SLOT];
    constexpr int REC = Dims<K>::FREC;
    const int w = threadIdx.x / K;
    const int t = blockIdx.x * NG + w;
    Flags bad = 0u;
    if (t < ntiles) {
        const int left = PREFIX ? t - s : t, right = PREFIX ? t : t + s;
        if (left >= 0 && right < ntiles) {
            FRow<K> r;
            load_frow(src + (int64_t)right * REC, r);
            put_frow(slot[w], r);
            __syncwarp(gmask<K>());
            load_frow(src + (int64_t)left * REC, r);
            combine_row(r, slot[w], bad);
            if constexpr (!PREFIX) relative_lg<K>(r);
            store_frow(dst + (int64_t)t * REC, r);
        } else {
            const float4* p = reinterpret_cast<const float4*>(src + (int64_t)t * REC);
            float4* q = reinterpret_cast<float4*>(dst + (int64_t)t * REC);
            for (int i = glane<K>(); i < REC / 4; i += K) q[i] = __ldcg(p + i);
        }
    }
    report_flags(status, bad, kFull, (threadIdx.x & 31) == 0);
}

// Forward apply: filt [T][K], loglik [T] (may be null); `pre` holds the
// inclusive tile prefixes from the spine.
template <int K, int NW, int CH>
__global__ void __launch_bounds__(NW * 32) filter_apply_kernel(const Const<K>* __restrict__ cg,
                                                               const float* __restrict__ lik, int64_t T,
                                                               float* __restrict__ filt, float* __restrict__ loglik,
                                                               Bufs b, const float* __restrict__ pre,
                                                               uint32_t* status) {
    __shared__ Smem<K, NW> sm;
    constexpr int NG = Smem<K, NW>::NG;
    load_pi(cg, sm.Pi, sm.q1);
    __syncthreads();
    const int w = threadIdx.x / K, lane = glane<K>();
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t c = (int64_t)blockIdx.x * NG + w;
    Flags bad = 0u;
    if (c < nch) {
        const int64_t k0 = c * CH, k1 = (k0 + CH < T) ? k0 + CH : T;
        // incoming prefix: tile prefix (x) the chain's exclusive in-tile prefix
        const bool has_tile = blockIdx.x > 0, has_in = w > 0;
        float p = 0.f, L = 0.f;
        bool has = has_tile || has_in;
        if (has) {
            FRow<K> r;
            if (has_tile) {
                load_frow(pre + ((int64_t)blockIdx.x - 1) * Dims<K>::FREC, r);
                if (has_in) {
                    FRow<K> e;
                    load_frow(b.fexcl + c * Dims<K>::FREC, e);
                    put_frow(sm.slot[w], e);
                    __syncwarp(gmask<K>());
                    combine_row(r, sm.slot[w], bad);
                }
            } else {
                load_frow(b.fexcl + c * Dims<K>::FREC, r);
            }
            row0_state(r, p, L);
        }
        float comp = 0.f;
        float col[K];   // this lane's column of Pi
#pragma unroll
        for (int y = 0; y < K; ++y) col[y] = sm.Pi[y * K + lane];
        float* buf = sm.slot[w];
        float ln = __ldg(lik + k0 * K + lane);
#pragma unroll 1
        for (int64_t k = k0; k < k1; ++k) {
            float lx = ln;
            if (k + 1 < k1) ln = __ldg(lik + (k + 1) * K + lane);
            const float m = group_max<K>(lx);
            bad |= !(m > 0.f) || !(m <= 3.0e38f) || !(lx <= 3.0e38f);
            lx *= 1.f / m;
            const float lm = __logf(m);
            if (!has) {   // step 1
                float v = sm.q1[lane] * lx;
                const float s = group_sum<K>(v);
                bad |= !(s > 0.f);
                p = v / s;
                L = lm + __logf(s);
                has = true;
            } else {
                advance_step<K>(p, L, comp, col, lx, lm, buf, bad);
            }
            filt[k * K + lane] = p;
            if (loglik && lane == 0) loglik[k] = L;
        }
        bad |= !isfinite(p) || !isfinite(L);
    }
    report_flags(status, bad, kFull, (threadIdx.x & 31) == 0);
}

// Reverse apply: smooth [T][K] = filt . beta / sum; `suf` holds the inclusive
// tile suffixes (rows of sum one, so that beta before a tile is its g).
template <int K, int NW, int CH>
__global__ void __launch_bounds__(NW * 32) smoother_apply_kernel(const Const<K>* __restrict__ cg,
                                                                 const float* __restrict__ lik,
                                                                 const float* __restrict__ filt, int64_t T,
                                                                 float* __restrict__ smooth, Bufs b,
                                                                 const float* __restrict__ suf, int ntiles,
                                                                 uint32_t* status) {
    constexpr int NG = NW * 32 / K;
    __shared__ __align__(16) float vec[NG][K];
    const int w = threadIdx.x / K, lane = glane<K>();
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t c = (int64_t)blockIdx.x * NG + w;
    Flags bad = 0u;
    if (c < nch) {
        const int64_t k0 = c * CH, k1 = (k0 + CH < T) ? k0 + CH : T;
        float be = 1.f;   // lane z: beta(z) after the chain
        float* buf = vec[w];
        if ((int)blockIdx.x + 1 < ntiles) {
            const float lg = __ldcg(suf + ((int64_t)blockIdx.x + 1) * Dims<K>::FREC + K * K + lane);
            be = beta_of<K>(1.f, lg);
        }
        const int64_t ctop = min(nch, ((int64_t)blockIdx.x + 1) * NG);
#pragma unroll 1
        for (int64_t j = ctop - 1; j > c; --j) {   // the tile's later chains
            FRow<K> r;
            load_frow(b.chain + j * Dims<K>::FREC, r);
            be = beta_of<K>(row_dot<K>(r.f, be, buf), r.lg);
        }
        float row[K];   // this lane's row of Pi
#pragma unroll
        for (int x = 0; x < K; ++x) row[x] = __ldg(cg->Pi + lane * K + x);
        constexpr float kUp = 1.152921504606847e18f;   // 2^60: see hmm::smoothed
        float pn = __ldg(filt + (k1 - 1) * K + lane), ln = __ldg(lik + (k1 - 1) * K + lane);
        float s = 0.f;
#pragma unroll 1
        for (int64_t k = k1 - 1; k >= k0; --k) {
            const float p = pn, lx = ln;
            if (k > k0) {
                pn = __ldg(filt + (k - 1) * K + lane);
                ln = __ldg(lik + (k - 1) * K + lane);
            }
            s = (p * kUp) * (be * kUp);
            const float t = group_sum<K>(s), m = group_max<K>(lx);
            bad |= !(t > 0.f) || !(m > 0.f);
            s = s / t;
            smooth[k * K + lane] = s;
            // beta_{k-1} = Pi (l_k . beta_k), both factors rescaled by powers of two
            int e;
            const float v = row_dot<K>(row, lx * pow2_of(m, e) * be, buf);
            be = v * pow2_of(group_max<K>(v), e);
        }
        bad |= !isfinite(s);
    }
    report_flags(status, bad, kFull, (threadIdx.x & 31) == 0);
}

template <int K>
__global__ void __launch_bounds__(64) prep_kernel(const float* __restrict__ pi, const float* __restrict__ Pi,
                                                  Const<K>* __restrict__ out, uint32_t* __restrict__ status) {
    const int t = threadIdx.x;
    Flags bad = 0u;
    for (int e = t; e < K * K; e += blockDim.x) {
        const float v = Pi[e];
        bad |= !(v >= 0.f) || !(v <= 3.0e38f);
        out->Pi[e] = v;
    }
    for (int x = t; x < K; x += blockDim.x) {
        float s = 0.f;
        for (int y = 0; y < K; ++y) s = fmaf(pi[y], Pi[y * K + x], s);
        bad |= !(s >= 0.f) || !(s <= 3.0e38f);
        out->q1[x] = s;
    }
    report_flags(status, bad, kFull, (t & 31) == 0);
}

}  // namespace hmmw
}  // namespace ks
