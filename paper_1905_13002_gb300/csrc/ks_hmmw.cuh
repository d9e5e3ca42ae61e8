// ks_hmmw.cuh -- the discrete-state (HMM) filter and smoother for K = 8, 16 and
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
    static constexpr int OFF = K * K + K;        // global filtering record: rows, log g relative to
    static constexpr int FREC = OFF + 4;         // an offset, the offset in FP64 (16 bytes kept for it)
};

// A chain is K lanes of one warp (lane z = row z); 32 / K chains per warp.  The
// chains of a warp step together (a shorter or absent one repeats its last step
// with the results dropped), so that every exchange is among all lanes.
template <int K>
KS_DEV int glane() { return threadIdx.x & (K - 1); }

template <int K>
struct Const {
    float Pi[K * K];
    float q1[K];   // p(x_1) = pi Pi
};

// One warp's share of a filtering element: lane z holds row z and log g(z) as
// lg + off, lg relative to the element's largest and off common to its rows.
// Kept as one FP32 number, a long prefix's log g (-1e5 and beyond) would leave no
// bits for the differences between states, which weigh its rows (K = 8, 2^20 steps
// of a nearly static chain: marginals 1e-3 off).
template <int K>
struct FRow {
    float f[K];
    float lg;
    double off;
};

template <int K>
KS_DEV float group_sum(float v) {
#pragma unroll
    for (int o = K / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o, K);
    return v;
}

template <int K>
KS_DEV float group_max(float v) {
#pragma unroll
    for (int o = K / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o, K));
    return v;
}

template <int K>
KS_DEV int group_max_i(int v) {
#pragma unroll
    for (int o = K / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o, K));
    return v;
}

// The largest of lg into the offset.
template <int K>
KS_DEV void relative_lg(FRow<K>& r) {
    const float m = group_max<K>(r.lg);
    r.lg -= m;
    r.off += (double)m;
}

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
    r.off = __ldcg(reinterpret_cast<const double*>(src + Dims<K>::OFF));
}

template <int K>
KS_DEV void store_frow(float* __restrict__ dst, const FRow<K>& r) {
    const int z = glane<K>();
    float4* p = reinterpret_cast<float4*>(dst + z * K);
#pragma unroll
    for (int i = 0; i < K / 4; ++i) p[i] = make_float4(r.f[4 * i], r.f[4 * i + 1], r.f[4 * i + 2], r.f[4 * i + 3]);
    dst[K * K + z] = r.lg;
    if (z == 0) *reinterpret_cast<double*>(dst + Dims<K>::OFF) = r.off;
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

// 2^-e and e for the exponent e of a positive r < 2^127 (2^-127 is no normal number).
KS_DEV float pow2_of(float r, int& e) {
    e = (int)(__float_as_uint(r) >> 23) - 127;
    return __uint_as_float((uint32_t)(127 - e) << 23);
}

// Two FP32 multiply-adds in one instruction (each rounded as fmaf).
KS_DEV void ffma2(uint64_t& d, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
KS_DEV uint64_t dup2(float v) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
    return r;
}
KS_DEV void unpack2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }

// o[r][x] = sum_y f[r][y] M[y][x] for a shared-memory M whose rows (pitch PITCH
// floats) all lanes of the chain read together: pairs of columns in packed
// multiply-adds (half the instructions of the scalar form), each loaded row
// used for R rows (the loads bound the K = 32 fold with R = 1).
template <int PITCH, int K, int R>
KS_DEV void rows_times(const float* const (&f)[R], const float* __restrict__ M, uint64_t (&acc)[R][K / 2]) {
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int i = 0; i < K / 2; ++i) acc[r][i] = 0ull;
#pragma unroll
    for (int y = 0; y < K; ++y) {
        const ulonglong2* p = reinterpret_cast<const ulonglong2*>(M + y * PITCH);
        uint64_t fy[R];
#pragma unroll
        for (int r = 0; r < R; ++r) fy[r] = dup2(f[r][y]);
#pragma unroll
        for (int i = 0; i < K / 4; ++i) {
            const ulonglong2 q = p[i];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                ffma2(acc[r][2 * i], fy[r], q.x);
                ffma2(acc[r][2 * i + 1], fy[r], q.y);
            }
        }
    }
}

// Fold of a step element into row z of R chains: (f Pi)[z] . l, kept at a sum in
// [1, 2) by a power of two (exponents added up in ex: no division, no
// logarithm).  l[r]: the chain's scaled likelihood row in shared memory, le its
// exponent; on[r] false: nothing happens to chain r.
template <int K, int R>
KS_DEV void fold_rows(FRow<K> (&fr)[R], int (&ex)[R], const float* __restrict__ Pi, const float* const (&l)[R],
                      const int (&le)[R], const bool (&on)[R], Flags (&bad)[R]) {
    uint64_t acc[R][K / 2];
    const float* f[R];
#pragma unroll
    for (int r = 0; r < R; ++r) f[r] = fr[r].f;
    rows_times<K, K, R>(f, Pi, acc);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        float o[K], s = 0.f;
#pragma unroll
        for (int i = 0; i < K / 2; ++i) unpack2(acc[r][i], o[2 * i], o[2 * i + 1]);
#pragma unroll
        for (int x = 0; x < K; x += 4) {
            const float4 q = *reinterpret_cast<const float4*>(l[r] + x);
            o[x] *= q.x;
            o[x + 1] *= q.y;
            o[x + 2] *= q.z;
            o[x + 3] *= q.w;
            s += (o[x] + o[x + 1]) + (o[x + 2] + o[x + 3]);
        }
        int e;
        const float rs = pow2_of(s, e);
        if (on[r]) {
            bad[r] |= !(s > 0.f);
#pragma unroll
            for (int x = 0; x < K; ++x) fr[r].f[x] = o[x] * rs;
            ex[r] += e + le[r];
        }
    }
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

// Definition 1, (row z of a_i, in registers) (x) a_j (in shared memory, its
// offset offj).
template <int K>
KS_DEV void combine_row(FRow<K>& r, const float* __restrict__ ej, double offj, Flags& bad) {
    float mx = ej[K * Dims<K>::Q];
#pragma unroll
    for (int y = 1; y < K; ++y) mx = fmaxf(mx, ej[K * Dims<K>::Q + y]);
    float o[K], fw[K], d = 0.f;
#pragma unroll
    for (int y = 0; y < K; ++y) {
        fw[y] = r.f[y] * __expf(ej[K * Dims<K>::Q + y] - mx);
        d += fw[y];
    }
    {
        uint64_t acc[1][K / 2];
        const float* const f[1] = {fw};
        rows_times<Dims<K>::Q, K, 1>(f, ej, acc);
#pragma unroll
        for (int i = 0; i < K / 2; ++i) unpack2(acc[0][i], o[2 * i], o[2 * i + 1]);
    }
    bad |= !(d > 0.f);
    const float rd = 1.f / d;
#pragma unroll
    for (int x = 0; x < K; ++x) r.f[x] = o[x] * rd;
    r.lg += mx + __logf(d);
    r.off += offj;
    relative_lg<K>(r);
}

// The prefix (all rows equal) as a state: lane x takes p(x) from row 0.
template <int K>
KS_DEV void row0_state(const FRow<K>& r, float& p, float& L) {
    const int lane = glane<K>();
    p = 0.f;
#pragma unroll
    for (int x = 0; x < K; ++x) {
        const float v = __shfl_sync(kFull, r.f[x], 0, K);
        if (lane == x) p = v;
    }
    L = (float)(r.off + (double)__shfl_sync(kFull, r.lg, 0, K));
}

// sum_x m[x] v(x) for a vector with v(x) on lane x, through the group's buffer
// (K floats of shared memory): one store and K / 4 broadcast loads in place of K
// shuffles.
template <int K>
KS_DEV float row_dot(const float (&m)[K], float v, float* __restrict__ buf) {
    __syncwarp(kFull);
    buf[glane<K>()] = v;
    __syncwarp(kFull);
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

constexpr int kAhead = 4;   // steps a chain loads ahead: a step is much shorter than a load from memory

// NG = NW * 32 / K * R chains per block: one K-lane group each R chains in the
// reduce, one chain in the applies.
template <int K, int NG>
struct alignas(16) Smem {
    float Pi[K * K];
    float q1[K];
    int top[(NG + 3) / 4 * 4];
    float slot[NG][Dims<K>::SLOT];   // one element per chain (pitch Q rows + lg)
};

// One chain's column of a [T][K] array (this lane's state), kAhead steps at a
// time and a group ahead: step i sits at base + i stride.
template <int K>
struct Ahead {
    const float* base;
    int n, stride;
    float next[kAhead];
    KS_DEV void fetch(int i0) {
#pragma unroll
        for (int j = 0; j < kAhead; ++j) next[j] = __ldg(base + min(i0 + j, n - 1) * stride);
    }
    KS_DEV void init(const float* b, int steps, int st) {
        base = b;
        n = steps;
        stride = st;
        fetch(0);
    }
    KS_DEV void take(int i0, float (&v)[kAhead]) {
#pragma unroll
        for (int j = 0; j < kAhead; ++j) v[j] = next[j];
        fetch(i0 + kAhead);
    }
};

// Likelihood entries scaled by a power of two to a row maximum in [1, 2), the
// topmost (2^127 and above) to [2, 4); le:
// the exponents taken out.
template <int K>
KS_DEV void scale_rows(float (&lx)[kAhead], int (&le)[kAhead], Flags& bad) {
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
        const float m = group_max<K>(lx[j]);
        const bool ok = m > 0.f && m <= 3.0e38f && lx[j] <= 3.0e38f;
        bad |= !ok;
        lx[j] *= pow2_of(ok ? fminf(m, 1.7e38f) : 1.f, le[j]);
    }
}

template <int K, int NW, int CH, int R>
__global__ void __launch_bounds__(NW * 32) filter_reduce_kernel(const Const<K>* __restrict__ cg,
                                                                const float* __restrict__ lik, int64_t T, Bufs b,
                                                                uint32_t* status) {
    constexpr int NG = NW * 32 / K * R;
    __shared__ Smem<K, NG> sm;
    pdl_trigger();
    pdl_wait();
    load_pi(cg, sm.Pi, sm.q1);
    __syncthreads();
    const int w = threadIdx.x / K, lane = glane<K>();
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t c0 = (int64_t)blockIdx.x * NG;
    const int nvalid = nch - c0 < NG ? (int)(nch - c0) : NG;
    Flags bad = 0u;
    {
        FRow<K> fr[R];
        int ex[R], n[R], nmax = 0;
        Ahead<K> lk[R];
        float* buf[R];
        const float* cbuf[R];
        Flags fbad[R];   // an absent chain folds the last one's steps from another row: its flags do not count
#pragma unroll
        for (int r = 0; r < R; ++r) {
            fbad[r] = 0u;
            const int64_t k0 = min(c0 + w * R + r, nch - 1) * CH;
            n[r] = (int)((k0 + CH < T ? k0 + CH : T) - k0);
            nmax = max(nmax, n[r]);
            lk[r].init(lik + k0 * K + lane, n[r], K);
            cbuf[r] = buf[r] = sm.slot[w * R + r];   // the chain's scaled likelihood row
            ex[r] = 0;
        }
        nmax = (int)__reduce_max_sync(kFull, (unsigned)nmax);
#pragma unroll 1
        for (int i0 = 0; i0 < nmax; i0 += kAhead) {
            float lx[R][kAhead];
            int le[R][kAhead];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                lk[r].take(i0, lx[r]);
                scale_rows<K>(lx[r], le[r], fbad[r]);
            }
#pragma unroll
            for (int j = 0; j < kAhead; ++j) {
                __syncwarp();
#pragma unroll
                for (int r = 0; r < R; ++r) buf[r][lane] = lx[r][j];
                __syncwarp();
                if (i0 + j == 0) {   // the chain's first element; k = 1: every row p(x_1, y_1)
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float* first = c0 + w * R + r == 0 ? sm.q1 : sm.Pi + lane * K;
#pragma unroll
                        for (int x = 0; x < K; ++x) fr[r].f[x] = first[x] * buf[r][x];
                        ex[r] = le[r][j];
                    }
                } else {
                    int lej[R];
                    bool on[R];
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        lej[r] = le[r][j];
                        on[r] = i0 + j < n[r];
                    }
                    fold_rows<K, R>(fr, ex, sm.Pi, cbuf, lej, on, fbad);
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int t = w * R + r;
            // log g relative to the chain's largest exponent, which is kept beside it
            const int top = group_max_i<K>(ex[r]);
            fold_end(fr[r], ex[r] - top, fbad[r]);
            if (t < nvalid) bad |= fbad[r];
            fr[r].off = 0.0;   // beta needs no offset
            put_frow(sm.slot[t], fr[r]);
            if (lane == 0) sm.top[t] = top;
            if (b.chain != nullptr && t < nvalid) store_frow(b.chain + (c0 + t) * Dims<K>::FREC, fr[r]);
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {   // in-tile combine, chain order (every chain group of the warp does the same)
        FRow<K> acc;
        smem_row<Dims<K>::Q>(sm.slot[0], lane, acc.f);
        acc.lg = sm.slot[0][K * Dims<K>::Q + lane];
        constexpr double kLn2 = 0.69314718055994531;
        acc.off = sm.top[0] * kLn2;
        const bool mine = w == 0;
#pragma unroll 1
        for (int t = 1; t < nvalid; ++t) {
            if (mine) store_frow(b.fexcl + (c0 + t) * Dims<K>::FREC, acc);
            combine_row(acc, sm.slot[t], sm.top[t] * kLn2, bad);
        }
        if (mine) store_frow(b.fspine0 + (int64_t)blockIdx.x * Dims<K>::FREC, acc);
        if (b.chain != nullptr && mine) store_frow(b.sspine0 + (int64_t)blockIdx.x * Dims<K>::FREC, acc);
    }
    report_flags(status, bad, kFull, (threadIdx.x & 31) == 0);
}

// Kogge-Stone level s over tile aggregates: dst[t] = src[t - s] (x) src[t]
// (prefixes, blockIdx.y = 0), and in the same launch src[t] (x) src[t + s]
// (suffixes, blockIdx.y = 1).
template <int K, int NW>
__global__ void __launch_bounds__(NW * 32) spine_kernel(const float* __restrict__ psrc, float* __restrict__ pdst,
                                                        const float* __restrict__ ssrc, float* __restrict__ sdst,
                                                        int ntiles, int s, uint32_t* status) {
    constexpr int NG = NW * 32 / K;
    __shared__ __align__(16) float slot[NG][Dims<K>::SLOT];
    constexpr int REC = Dims<K>::FREC;
    pdl_trigger();
    pdl_wait();
    const bool prefix = blockIdx.y == 0;
    const float* src = prefix ? psrc : ssrc;
    float* dst = prefix ? pdst : sdst;
    const int w = threadIdx.x / K;
    const int t = blockIdx.x * NG + w;
    Flags bad = 0u, none = 0u;
    const int left = prefix ? t - s : t, right = prefix ? t : t + s;
    const bool in = t < ntiles, comb = in && left >= 0 && right < ntiles;
    FRow<K> r;   // every group combines; one without a partner copies instead
    load_frow(src + (int64_t)(comb ? right : 0) * REC, r);
    put_frow(slot[w], r);
    const double offj = r.off;
    __syncwarp();
    load_frow(src + (int64_t)(comb ? left : 0) * REC, r);
    combine_row(r, slot[w], offj, comb ? bad : none);
    if (comb) {
        store_frow(dst + (int64_t)t * REC, r);
    } else if (in) {
        const float4* p = reinterpret_cast<const float4*>(src + (int64_t)t * REC);
        float4* q = reinterpret_cast<float4*>(dst + (int64_t)t * REC);
        for (int i = glane<K>(); i < REC / 4; i += K) q[i] = __ldcg(p + i);
    }
    report_flags(status, bad, kFull, (threadIdx.x & 31) == 0);
}

// Forward apply: filt [T][K], loglik [T] (may be null); `pre` holds the
// inclusive tile prefixes from the spine.
// TC: chains per tile (of the reduce).
template <int K, int NW, int CH, int TC>
__global__ void __launch_bounds__(NW * 32) filter_apply_kernel(const Const<K>* __restrict__ cg,
                                                               const float* __restrict__ lik, int64_t T,
                                                               float* __restrict__ filt, float* __restrict__ loglik,
                                                               Bufs b, const float* __restrict__ pre,
                                                               uint32_t* status) {
    constexpr int NG = NW * 32 / K;
    __shared__ __align__(16) float slot[NG][Dims<K>::SLOT];
    pdl_trigger();
    pdl_wait();
    const int w = threadIdx.x / K, lane = glane<K>();
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t cr = (int64_t)blockIdx.x * NG + w, c = min(cr, nch - 1);
    const bool own = cr < nch;
    const int64_t k0 = c * CH;
    const int n = (int)((k0 + CH < T ? k0 + CH : T) - k0);
    Flags bad = 0u, none = 0u;
    // incoming prefix: tile prefix (x) the chain's exclusive in-tile prefix (absent: not used)
    const int64_t tile = c / TC;
    const bool has_tile = tile > 0, has_in = c % TC > 0;
    float p, L;
    {
        FRow<K> r, e;
        load_frow(has_tile ? pre + (tile - 1) * Dims<K>::FREC : b.fspine0, r);
        load_frow(has_in ? b.fexcl + c * Dims<K>::FREC : b.fspine0, e);
        put_frow(slot[w], e);
        __syncwarp();
        FRow<K> both = r;
        combine_row(both, slot[w], e.off, has_tile && has_in ? bad : none);
        float p1, L1, p2, L2;
        row0_state(has_tile ? r : e, p1, L1);
        row0_state(both, p2, L2);
        p = has_tile && has_in ? p2 : p1;
        L = has_tile && has_in ? L2 : L1;
    }
    const bool start = !has_tile && !has_in;   // the chain of step 1
    float col[K], comp = 0.f;                  // this lane's column of Pi
#pragma unroll
    for (int y = 0; y < K; ++y) col[y] = __ldg(cg->Pi + y * K + lane);
    const float q1 = __ldg(cg->q1 + lane);
    if (start) L = 0.f;
    float* buf = slot[w];
    float* fo = filt + k0 * K + lane;
    float* lo = loglik ? loglik + k0 : nullptr;
    Ahead<K> lk;
    lk.init(lik + k0 * K + lane, n, K);
    const int nmax = (int)__reduce_max_sync(kFull, (unsigned)n);
#pragma unroll 1
    for (int i0 = 0; i0 < nmax; i0 += kAhead) {
        float lx[kAhead];
        int le[kAhead];
        lk.take(i0, lx);
        scale_rows<K>(lx, le, bad);
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            // p'(x) = (p Pi)(x) l(x) / c, L' = L + log c (Kahan-compensated)
            float v = row_dot<K>(col, p, buf);
            if (start && i0 + j == 0) v = q1;
            v *= lx[j];
            const float s = group_sum<K>(v);
            if (i0 + j < n) {
                bad |= !(s > 0.f);
                p = v * (1.f / s);
                const float t = fmaf((float)le[j], 0.693147180559945f, __logf(s)) - comp;
                const float Ln = L + t;
                comp = (Ln - L) - t;
                L = Ln;
                if (own) {
                    fo[(i0 + j) * K] = p;
                    if (lo != nullptr && lane == 0) lo[i0 + j] = L;
                }
            }
        }
    }
    bad |= !isfinite(p) || !isfinite(L);
    report_flags(status, own ? bad : 0u, kFull, (threadIdx.x & 31) == 0);
}

// Reverse apply: smooth [T][K] = filt . beta / sum; `suf` holds the inclusive
// tile suffixes (rows of sum one, so that beta before a tile is its g).
template <int K, int NW, int CH, int TC>
__global__ void __launch_bounds__(NW * 32) smoother_apply_kernel(const Const<K>* __restrict__ cg,
                                                                 const float* __restrict__ lik,
                                                                 const float* __restrict__ filt, int64_t T,
                                                                 float* __restrict__ smooth, Bufs b,
                                                                 const float* __restrict__ suf, int ntiles,
                                                                 uint32_t* status) {
    constexpr int NG = NW * 32 / K;
    __shared__ __align__(16) float vec[NG][K];
    pdl_trigger();
    pdl_wait();
    const int w = threadIdx.x / K, lane = glane<K>();
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t cr = (int64_t)blockIdx.x * NG + w, c = min(cr, nch - 1);
    const bool own = cr < nch;
    const int64_t k0 = c * CH;
    const int n = (int)((k0 + CH < T ? k0 + CH : T) - k0);
    Flags bad = 0u;
    const int64_t tile = c / TC;
    float* buf = vec[w];
    float be = 1.f;   // lane z: beta(z) after the chain
    {
        const bool more = (int)tile + 1 < ntiles;
        const float b1 = beta_of<K>(1.f, __ldcg(suf + (more ? tile + 1 : tile) * Dims<K>::FREC + K * K + lane));
        be = more ? b1 : 1.f;
        const int64_t ctop = min(nch, (tile + 1) * TC);
        const int later = (int)(ctop - 1 - c);   // the tile's later chains, a record ahead
        const int lmax = (int)__reduce_max_sync(kFull, (unsigned)later);
        FRow<K> nx;
        load_frow(b.chain + (ctop - 1) * Dims<K>::FREC, nx);
#pragma unroll 1
        for (int j = 0; j < lmax; ++j) {
            const FRow<K> r = nx;
            load_frow(b.chain + max(ctop - 2 - j, c) * Dims<K>::FREC, nx);
            const float v = beta_of<K>(row_dot<K>(r.f, be, buf), r.lg);
            if (j < later) be = v;
        }
    }
    float row[K];   // this lane's row of Pi
#pragma unroll
    for (int x = 0; x < K; ++x) row[x] = __ldg(cg->Pi + lane * K + x);
    constexpr float kUp = 1.152921504606847e18f;   // 2^60: see hmm::smoothed
    Ahead<K> pf, lk;
    pf.init(filt + (k0 + n - 1) * K + lane, n, -K);
    lk.init(lik + (k0 + n - 1) * K + lane, n, -K);
    float* so = smooth + (k0 + n - 1) * K + lane;
    float s = 0.f;
    const int nmax = (int)__reduce_max_sync(kFull, (unsigned)n);
#pragma unroll 1
    for (int i0 = 0; i0 < nmax; i0 += kAhead) {
        float p[kAhead], lx[kAhead];
        int le[kAhead];
        pf.take(i0, p);
        lk.take(i0, lx);
        scale_rows<K>(lx, le, bad);
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            // beta_{k-1} = Pi (l_k . beta_k), rescaled by a power of two, beside the row's own sum
            const float v = row_dot<K>(row, lx[j] * be, buf);
            s = (p[j] * kUp) * (be * kUp);
            const float t = group_sum<K>(s), m = group_max<K>(v);
            if (i0 + j < n) {
                bad |= !(t > 0.f);
                s *= 1.f / t;
                if (own) so[-(i0 + j) * K] = s;
                int e;
                be = v * pow2_of(m, e);
            }
        }
    }
    bad |= !isfinite(be);
    report_flags(status, own ? bad : 0u, kFull, (threadIdx.x & 31) == 0);
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
