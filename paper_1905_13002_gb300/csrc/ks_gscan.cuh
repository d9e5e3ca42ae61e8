// ks_gscan.cuh -- forward and reverse scans for larger state sizes, one lane
// group per chain of CH consecutive steps (elements in shared-memory slots,
// see ks_group.cuh: 8 lanes per chain for nx <= 8, a warp otherwise).  Each
// scan runs as three kinds of launch (the paper's block-level elements,
// Section III-C, one block per tile of NG chains):
//   reduce   each group folds its chain into one block element; group 0 then
//            combines the tile's chain totals in order, storing each chain's
//            exclusive in-tile prefix, and writes the tile aggregate;
//   spine    one Kogge-Stone level over the tile aggregates per launch
//            (log2 tiles launches, one group per tile, no waiting on other
//            blocks); a left operand that is already a complete prefix is
//            applied in its prefix-state form;
//   apply    each group starts from the prefix entering its chain and applies
//            its elements one by one, writing one posterior per step.
// With a full nx x nx combine (a pivoted inverse) per step of a cross-tile
// walk, a decoupled look-back kept most of each block waiting; the spine
// takes one combine per level instead.  Segmented batches need nothing in
// the spine: a sequence's first filtering element has A = 0 and its last
// smoothing element E = 0, so combines across a sequence start or end drop
// the other sequence exactly (the builders in reduce/apply know the segments).
#pragma once

#include "ks_group.cuh"
#include "ks_scan.cuh"

namespace ks {
namespace grp {

// Global scratch of one scan: per chain its total and its exclusive in-tile
// prefix (slot layout each), two spine buffers of one slot per tile, and (the
// reverse scan) every step's smoothing element, built once in reduce.
struct GBuf {
    float* chains;   // nchains x 2 x slot
    float* spine0;   // ntiles x slot
    float* spine1;   // ntiles x slot
    float* elems;    // T smoothing slots (reverse scan only)
};

// Copy an element slot (n floats) between two locations, by the lanes of the
// calling chain's group (LANES = 32: by the whole warp): kCopy loads of each
// lane in flight before the first is stored (one load at a time, a 234-float
// element took ~30 trips to L2, longer than its combine).  CG: data written
// by other blocks or launches (L2 loads).
constexpr int kCopy = 16;
template <int N, bool CG, int LANES>
KS_DEV void copy_slot(float* dst, const float* src, int n) {
    for (int i0 = threadIdx.x & (LANES - 1); i0 < n; i0 += LANES * kCopy) {
        float v[kCopy];
#pragma unroll
        for (int u = 0; u < kCopy; ++u) {
            const int i = i0 + u * LANES;
            v[u] = i < n ? (CG ? __ldcg(src + i) : src[i]) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < kCopy; ++u) {
            const int i = i0 + u * LANES;
            if (i < n) dst[i] = v[u];
        }
    }
    if constexpr (LANES == 32) __syncwarp();
    else gsync<N>();
}
template <int N, int LANES = Grp<N>::GS>
KS_DEV void copy_floats(float* dst, const float* src, int n) { copy_slot<N, false, LANES>(dst, src, n); }
template <int N, int LANES = Grp<N>::GS>
KS_DEV void copy_floats_cg(float* dst, const float* src, int n) { copy_slot<N, true, LANES>(dst, src, n); }

template <int N, int M>
KS_DEV void load_const_all(const ModelConst<N, M>* __restrict__ g, ModelConst<N, M>& s) {
    const float* src = reinterpret_cast<const float*>(g);
    float* dst = reinterpret_cast<float*>(&s);
    for (int i = threadIdx.x; i < (int)(sizeof(ModelConst<N, M>) / 4); i += blockDim.x) dst[i] = __ldg(src + i);
}

// Per-chain buffer: three element slots and the scratch.  With 8-lane groups
// the stride is padded to 8 (mod 32) words, so the four groups of a warp
// reading their own row r (word 9 r + j + 8 g) or one broadcast row hit
// distinct banks.
template <int N>
struct GChain {
    static constexpr int FS = Dim<N>::FSLOT, SS = Dim<N>::SSLOT;
    static constexpr int SLOT = FS > SS ? FS : SS;
    static constexpr int RAW = 3 * SLOT + Scratch<N>::FLOATS;
    static constexpr int STRIDE = Grp<N>::GS == 32 ? RAW : RAW + ((8 - RAW % 32) + 32) % 32;
};

// Steps of a time-varying model read ahead by a chain's group (kStaged): two
// buffers of one step's inputs, filled by asynchronous copies while the step
// before is combined.  Read where they are used, the constants cost a chain of
// L2 round trips in every step (nx = 8, 8 steps a chain and too few chains to
// cover it: reduce 58 -> 33 us, apply 54 -> 39 us at 20 Ki steps).  8-lane groups only: at larger nx the element slots
// leave no room.
template <int N, int M>
struct Stage {
    using MC = ModelConst<N, M>;
    static constexpr bool on = Grp<N>::GS == 8 && sizeof(MC) % 16 == 0;
    static constexpr int MCF = (int)sizeof(MC) / 4;
    static constexpr int PRED = N * N + N + sym_size(N);              // F, u, Q lead a ModelConst
    static constexpr int POST = (PRED + 3) / 4 * 4;                   // reverse scan: the filtered rows behind them
    static constexpr int FLOATS = (MCF + M + 3) / 4 * 4;
    static_assert(!on || POST + Dim<N>::MAT + Dim<N>::NP <= FLOATS, "reverse inputs fit");

    static KS_DEV void copy16(float* dst, const float* src, int nf, int r) {   // whole 16-byte words covering nf floats
        for (int c = r; c < (nf + 3) / 4; c += Grp<N>::GS) cp_async16(dst + 4 * c, src + 4 * c);
    }
    // Step k of the forward scan: its constants and its measurement.
    static KS_DEV void forward(int r, float* buf, const MC* mc, const float* yk) {
        copy16(buf, reinterpret_cast<const float*>(mc), MCF, r);
        for (int q = r; q < M; q += Grp<N>::GS) cp_async4(buf + MCF + q, yk + q);
    }
    // Step k of the reverse scan: the transition after it and its filtered row.
    static KS_DEV void reverse(int r, float* buf, const MC* mc, const float* fm, const float* fc) {
        copy16(buf, reinterpret_cast<const float*>(mc), PRED, r);
        for (int e = r; e < N * N; e += Grp<N>::GS) cp_async4(buf + POST + (e / N) * Dim<N>::NP + e % N, fc + e);
        for (int e = r; e < N; e += Grp<N>::GS) cp_async4(buf + POST + Dim<N>::MAT + e, fm + e);
    }
};

// Shared memory of a scan launch: the model constants, NW warps' chains and,
// staged, two step buffers per chain.
template <int N, int M, int NW, bool STAGED = false>
struct GSmem {
    static constexpr int SLOT = GChain<N>::SLOT;
    static constexpr int NG = NW * 32 / Grp<N>::GS;                  // chains per block
    static constexpr int CONST = ((int)sizeof(ModelConst<N, M>) + 15) / 16 * 16;
    static constexpr int CHAINS = (NG * GChain<N>::STRIDE * 4 + 15) / 16 * 16;
    static constexpr int BYTES = CONST + CHAINS + (STAGED ? NG * 2 * Stage<N, M>::FLOATS * 4 : 0);
    static KS_DEV ModelConst<N, M>& mc(char* base) { return *reinterpret_cast<ModelConst<N, M>*>(base); }
    static KS_DEV float* chain(char* base, int g) {
        return reinterpret_cast<float*>(base + CONST) + g * GChain<N>::STRIDE;
    }
    static KS_DEV float* stage(char* base, int g, int i) {
        return reinterpret_cast<float*>(base + CONST + CHAINS) + (2 * g + (i & 1)) * Stage<N, M>::FLOATS;
    }
};

// Shared memory of a spine launch (no model constants): NWS warps, one tile each.
template <int N, int NWS>
struct GSpineSmem {
    static constexpr int NG = NWS;
    static constexpr int BYTES = NWS * GChain<N>::STRIDE * 4;
    static KS_DEV float* chain(char* base, int g) { return reinterpret_cast<float*>(base) + g * GChain<N>::STRIDE; }
};
// Warps per spine block: up to 4, within 200 KB of shared memory.
template <int N>
constexpr int gspine_warps() {
    constexpr int per = GChain<N>::STRIDE * 4;
    return per * 4 <= 200 * 1024 ? 4 : (200 * 1024 / per > 0 ? 200 * 1024 / per : 1);
}

// ---------------------------------------------------------------- forward
template <int N, int M, int NW, int CH, bool SEG, bool TV = false>
__global__ void __launch_bounds__(NW * 32) gfilter_reduce_kernel(const ModelConst<N, M>* __restrict__ mcg,
                                                                 const float* __restrict__ y, int64_t T, GBuf gb,
                                                                 uint32_t* status, Segs<N, M> segs, const uint32_t* gate) {
    if (gate_closed(gate)) return;
    constexpr bool kStaged = TV && Stage<N, M>::on;
    using SM = GSmem<N, M, NW, kStaged>;
    constexpr int FS = Dim<N>::FSLOT, NG = SM::NG;
    extern __shared__ __align__(16) char gsm[];
    ModelConst<N, M>& mc = SM::mc(gsm);
    load_const_all<N, M>(mcg, mc);
    __syncthreads();
    const int tile = blockIdx.x;
    const int w = threadIdx.x / Grp<N>::GS, r = threadIdx.x & (Grp<N>::GS - 1);
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t c = (int64_t)tile * NG + w;
    const int64_t left = nch - (int64_t)tile * NG;
    const int nvalid = left < NG ? (int)left : NG;
    const bool valid = w < nvalid;
    const int64_t k0 = c * CH;
    float* wb = SM::chain(gsm, w);
    FSlot<N> X[3] = {FSlot<N>{wb}, FSlot<N>{wb + SM::SLOT}, FSlot<N>{wb + 2 * SM::SLOT}};
    Scratch<N> s{wb + 3 * SM::SLOT};
    Flags bad = 0u;
    Cursor<N, M, SEG, TV> cur;

    // ---- chain fold
    if (valid) {
        cur.seek(segs, &mc, k0, T);
        int a = 0;
        const auto stage = [&](int i) {                       // the constants and the measurement of step i + 1 on their way
            if constexpr (kStaged) {
                const int64_t k = k0 + i + 1;
                if (i + 1 < CH && k < T) Stage<N, M>::forward(r, SM::stage(gsm, w, i + 1), segs.mcg + k, y + k * M);
                cp_async_commit();
            }
        };
        const auto staged = [&](int i) {                      // those of step i have arrived
            cp_async_wait<1>();
            gsync<N>();
            return SM::stage(gsm, w, i);
        };
        const ModelConst<N, M>* mk = cur.mc;
        const float* yk = y + k0 * M;
        stage(-1);
        stage(0);
        if constexpr (kStaged) {
            const float* b = staged(0);
            mk = reinterpret_cast<const ModelConst<N, M>*>(b);
            yk = b + Stage<N, M>::MCF;
        }
        if (cur.first(k0)) {
            first_elem<N, M>(r, *mk, X[0]);
        } else {
            float wv[M];
            const float b = meas<N, M>(r, *mk, yk, wv);
            expand_meas<N, M>(r, *mk, b, wv, X[0]);
        }
        gsync<N>();
#pragma unroll 1
        for (int i = 1; i < CH; ++i) {
            const int64_t k = k0 + i;
            if (k >= T) break;
            cur.forward(segs, k);
            mk = cur.mc;
            yk = y + k * M;
            stage(i);
            if constexpr (kStaged) {
                const float* b = staged(i);
                mk = reinterpret_cast<const ModelConst<N, M>*>(b);
                yk = b + Stage<N, M>::MCF;
            }
            if (cur.first(k)) {
                reset_first<N, M>(r, *mk, X[a]);
                gsync<N>();
            } else {
                float wv[M];
                const float b = meas<N, M>(r, *mk, yk, wv);
                fcombine_meas<N, M, false>(r, X[a], *mk, b, wv, X[a ^ 1], s, bad);
                a ^= 1;
            }
        }
        if (a != 0) copy_floats<N>(X[0].p, X[a].p, FS);       // the chain's total, where warp 0 looks for it
    }
    __syncthreads();

    // ---- in-tile combine (warp 0): E_t = T_0 (x) ... (x) T_{t-1}
    if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        float* cb = SM::chain(gsm, 0);
        const FSlot<N> Y[3] = {FSlot<N>{cb}, FSlot<N>{cb + SM::SLOT}, FSlot<N>{cb + 2 * SM::SLOT}};
        const Scratch<N> sc{cb + 3 * SM::SLOT};
        int a = 0;
#pragma unroll 1
        for (int t = 1; t < nvalid; ++t) {
            copy_floats<N, 32>(gb.chains + (((size_t)tile * NG + t) * 2 + 1) * FS, Y[a].p, FS);
            const int b = a == 1 ? 2 : 1;
            warp_fcombine<N>(l, Y[a], FSlot<N>{SM::chain(gsm, t)}, Y[b], sc, bad, false);
            a = b;
        }
        copy_floats<N, 32>(gb.spine0 + (size_t)tile * FS, Y[a].p, FS);
    }
    report_flags(status, bad, gmask<N>(), r == 0);
}

// dst[t] = src[t - s] (x) src[t] for t >= s, else src[t].  src[t - s] covers
// tiles from 0 when t - s < s: then it is a prefix state (A = 0) and only b
// and C of the result are formed.
template <int N, int NWS>
__global__ void __launch_bounds__(NWS * 32) gspine_filter_kernel(const float* __restrict__ src, float* __restrict__ dst,
                                                                 int ntiles, int s, uint32_t* status, const uint32_t* gate) {
    if (gate_closed<false>(gate)) return;
    using SM = GSpineSmem<N, NWS>;
    constexpr int FS = Dim<N>::FSLOT;
    constexpr int SLOT = GChain<N>::SLOT;
    extern __shared__ __align__(16) char gsm[];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int t = blockIdx.x * SM::NG + w;
    if (t >= ntiles) return;                              // whole warps; no block barrier below
    float* o = dst + (size_t)t * FS;
    if (t < s) {
        copy_floats_cg<N, 32>(o, src + (size_t)t * FS, FS);
        return;
    }
    float* wb = SM::chain(gsm, w);
    FSlot<N> X[3] = {FSlot<N>{wb}, FSlot<N>{wb + SLOT}, FSlot<N>{wb + 2 * SLOT}};
    Scratch<N> sc{wb + 3 * SLOT};
    Flags bad = 0u;
    copy_floats_cg<N, 32>(X[0].p, src + (size_t)(t - s) * FS, FS);
    copy_floats_cg<N, 32>(X[1].p, src + (size_t)t * FS, FS);
    warp_fcombine<N>(l, X[0], X[1], X[2], sc, bad, t - s < s);
    copy_floats<N, 32>(o, X[2].p, FS);
    report_flags(status, bad, kFullMask, l == 0);
}

// `pre`: the spine's inclusive prefixes (slot t covers tiles 0..t).
template <int N, int M, int NW, int CH, bool SEG, bool TV = false>
__global__ void __launch_bounds__(NW * 32) gfilter_apply_kernel(const ModelConst<N, M>* __restrict__ mcg,
                                                                const float* __restrict__ y, int64_t T,
                                                                float* __restrict__ fmean, float* __restrict__ fcov,
                                                                GBuf gb, const float* __restrict__ pre,
                                                                uint32_t* status, Segs<N, M> segs, const uint32_t* gate) {
    if (gate_closed(gate)) return;
    constexpr bool kStaged = TV && Stage<N, M>::on;
    using SM = GSmem<N, M, NW, kStaged>;
    constexpr int FS = Dim<N>::FSLOT, NG = SM::NG;
    extern __shared__ __align__(16) char gsm[];
    ModelConst<N, M>& mc = SM::mc(gsm);
    load_const_all<N, M>(mcg, mc);
    __syncthreads();
    const int tile = blockIdx.x;
    const int w = threadIdx.x / Grp<N>::GS, r = threadIdx.x & (Grp<N>::GS - 1);
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t c = (int64_t)tile * NG + w;
    if (c >= nch) return;                                 // whole warps; no block barrier below
    const int64_t k0 = c * CH;
    const float* chE = gb.chains + (size_t)c * 2 * FS + FS;
    float* wb = SM::chain(gsm, w);
    FSlot<N> X[3] = {FSlot<N>{wb}, FSlot<N>{wb + SM::SLOT}, FSlot<N>{wb + 2 * SM::SLOT}};
    Scratch<N> s{wb + 3 * SM::SLOT};
    Flags bad = 0u;
    Cursor<N, M, SEG, TV> cur;
    int a = 0;
    bool has = false;
    const auto stage = [&](int i) {
        if constexpr (kStaged) {
            const int64_t k = k0 + i + 1;
            if (i + 1 < CH && k < T) Stage<N, M>::forward(r, SM::stage(gsm, w, i + 1), segs.mcg + k, y + k * M);
            cp_async_commit();
        }
    };
    stage(-1);
    if (tile != 0) {
        const float* tex = pre + (size_t)(tile - 1) * FS;
        if (w >= 1) {
            copy_floats_cg<N>(X[2].p, tex, FS);
            copy_floats_cg<N>(X[1].p, chE, FS);
            fadvance<N>(r, X[2], X[1], X[0], s, bad);
        } else {
            copy_floats_cg<N>(X[0].p, tex, FS);
        }
        has = true;
    } else if (w >= 1) {
        copy_floats_cg<N>(X[0].p, chE, FS);                 // E_w has A = 0 (it starts with the first element)
        has = true;
    }
    cur.seek(segs, &mc, k0, T);
    float probe = 0.f;
#pragma unroll 1
    for (int i = 0; i < CH; ++i) {
        const int64_t k = k0 + i;
        if (k >= T) break;
        cur.forward(segs, k);
        const ModelConst<N, M>* mk = cur.mc;
        const float* yk = y + k * M;
        stage(i);
        if constexpr (kStaged) {
            cp_async_wait<1>();
            gsync<N>();
            const float* b = SM::stage(gsm, w, i);
            mk = reinterpret_cast<const ModelConst<N, M>*>(b);
            yk = b + Stage<N, M>::MCF;
        }
        if (cur.first(k) || !has) {
            first_state<N, M>(r, *mk, X[a]);
            has = true;
        } else {
            float wv[M];
            const float b = meas<N, M>(r, *mk, yk, wv);
            fcombine_meas<N, M, true>(r, X[a], *mk, b, wv, X[a ^ 1], s, bad);
            a ^= 1;
        }
        if (r < N) {
            const float bm = X[a].b()[r];
            fmean[k * N + r] = bm;
            float* crow = fcov + (k * N + r) * N;
            const float* src = X[a].C() + r * Dim<N>::NP;
#pragma unroll Unroll<N>::K
            for (int q = 0; q < N; ++q) crow[q] = src[q];
            probe += bm + src[r];
        }
    }
    bad |= !isfinite(probe);
    report_flags(status, bad, gmask<N>(), r == 0);
}

// ---------------------------------------------------------------- reverse
// Chains are the forward blocks of CH steps, visited last first; in time
// order the operator takes the earlier step on the left (Lemma 6).
template <int N, int M, int NW, int CH, bool SEG, bool TV = false>
__global__ void __launch_bounds__(NW * 32) gsmoother_reduce_kernel(const ModelConst<N, M>* __restrict__ mcg,
                                                                   const float* __restrict__ fmean,
                                                                   const float* __restrict__ fcov, int64_t T, GBuf gb,
                                                                   uint32_t* status, Segs<N, M> segs, const uint32_t* gate) {
    if (gate_closed(gate)) return;
    constexpr bool kStaged = TV && Stage<N, M>::on;
    using SM = GSmem<N, M, NW, kStaged>;
    constexpr int SS = Dim<N>::SSLOT, NG = SM::NG;
    extern __shared__ __align__(16) char gsm[];
    ModelConst<N, M>& mc = SM::mc(gsm);
    load_const_all<N, M>(mcg, mc);
    __syncthreads();
    const int tile = blockIdx.x;
    const int w = threadIdx.x / Grp<N>::GS, r = threadIdx.x & (Grp<N>::GS - 1);
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t u = (int64_t)tile * NG + w;            // scan-order chain index
    const int64_t left = nch - (int64_t)tile * NG;
    const int nvalid = left < NG ? (int)left : NG;
    const bool valid = w < nvalid;
    const int64_t cblk = nch - 1 - u;                     // forward block
    const int64_t klo = cblk * CH;
    const int64_t khi = valid ? ((klo + CH < T ? klo + CH : T) - 1) : -1;
    float* wb = SM::chain(gsm, w);
    SSlot<N> X[3] = {SSlot<N>{wb}, SSlot<N>{wb + SM::SLOT}, SSlot<N>{wb + 2 * SM::SLOT}};
    Scratch<N> s{wb + 3 * SM::SLOT};
    Flags bad = 0u;
    Cursor<N, M, SEG, TV> cur;

    // ---- chain fold: a_{klo} (x) ... (x) a_{khi}, from the latest step back
    if (valid) {
        cur.seek(segs, &mc, khi, T);
        // What step k needs: the filtered row in P, xb and the transition mk.
        const ModelConst<N, M>* mk = &mc;
        const float *P = s.S(3), *xb = s.V(5);
        const auto stage = [&](int64_t k) {                   // step k's inputs on their way (buffer by its place in the chain)
            if constexpr (kStaged) {
                if (k >= klo) Stage<N, M>::reverse(r, SM::stage(gsm, w, (int)(k - klo)), cur.trans(k), fmean + k * N, fcov + k * N * N);
                cp_async_commit();
            }
        };
        const auto load = [&](int64_t k) {
            if constexpr (kStaged) {
                cp_async_wait<1>();
                const float* b = SM::stage(gsm, w, (int)(k - klo));
                mk = reinterpret_cast<const ModelConst<N, M>*>(b);
                P = b + Stage<N, M>::POST;
                xb = P + Dim<N>::MAT;
            } else {
                mk = cur.trans(k);
                if (r < N) {
                    const float* src = fcov + (k * N + r) * N;
                    float* dst = s.S(3) + r * Dim<N>::NP;
#pragma unroll Unroll<N>::K
                    for (int q = 0; q < N; ++q) dst[q] = __ldg(src + q);
                    s.V(5)[r] = __ldg(fmean + k * N + r);
                }
            }
            gsync<N>();
        };
        int a = 0;
        stage(khi);
        stage(khi - 1);
        load(khi);
        selem<N, M>(r, *mk, P, xb, cur.last(khi), X[0], s, bad);
        copy_floats<N>(gb.elems + (size_t)khi * SS, X[0].p, SS);
#pragma unroll 1
        for (int64_t k = khi - 1; k >= klo; --k) {
            cur.backward(segs, k);
            stage(k - 1);
            load(k);
            selem<N, M>(r, *mk, P, xb, cur.last(k), X[2], s, bad);
            copy_floats<N>(gb.elems + (size_t)k * SS, X[2].p, SS);
            scombine<N, false>(r, X[2], X[a], X[a ^ 1], s);
            a ^= 1;
        }
        if (a != 0) copy_floats<N>(X[0].p, X[a].p, SS);
    }
    __syncthreads();

    // ---- in-tile combine (warp 0): E_t = T_{t-1} (x) ... (x) T_0 in time order
    if (threadIdx.x < 32) {
        const int l = threadIdx.x;
        float* cb = SM::chain(gsm, 0);
        const SSlot<N> Y[3] = {SSlot<N>{cb}, SSlot<N>{cb + SM::SLOT}, SSlot<N>{cb + 2 * SM::SLOT}};
        const Scratch<N> sc{cb + 3 * SM::SLOT};
        int a = 0;
#pragma unroll 1
        for (int t = 1; t < nvalid; ++t) {
            copy_floats<N, 32>(gb.chains + (((size_t)tile * NG + t) * 2 + 1) * SS, Y[a].p, SS);
            const int b = a == 1 ? 2 : 1;
            warp_scombine<N>(l, SSlot<N>{SM::chain(gsm, t)}, Y[a], Y[b], sc, false);
            a = b;
        }
        copy_floats<N, 32>(gb.spine0 + (size_t)tile * SS, Y[a].p, SS);
    }
    report_flags(status, bad, gmask<N>(), r == 0);
}

// Scan order (tile 0 = latest time): dst[u] = src[u] (x) src[u - s] in time
// order for u >= s, else src[u].  src[u - s] reaches the sequence's end when
// u - s < s: then it is a suffix state (E = 0) and only g and L are formed.
template <int N, int NWS>
__global__ void __launch_bounds__(NWS * 32) gspine_smoother_kernel(const float* __restrict__ src,
                                                                   float* __restrict__ dst, int ntiles, int s,
                                                                   uint32_t* status, const uint32_t* gate) {
    if (gate_closed<false>(gate)) return;
    using SM = GSpineSmem<N, NWS>;
    constexpr int SS = Dim<N>::SSLOT;
    constexpr int SLOT = GChain<N>::SLOT;
    extern __shared__ __align__(16) char gsm[];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    const int u = blockIdx.x * SM::NG + w;
    if (u >= ntiles) return;                              // whole warps; no block barrier below
    float* o = dst + (size_t)u * SS;
    if (u < s) {
        copy_floats_cg<N, 32>(o, src + (size_t)u * SS, SS);
        return;
    }
    float* wb = SM::chain(gsm, w);
    SSlot<N> X[3] = {SSlot<N>{wb}, SSlot<N>{wb + SLOT}, SSlot<N>{wb + 2 * SLOT}};
    Scratch<N> sc{wb + 3 * SLOT};
    copy_floats_cg<N, 32>(X[0].p, src + (size_t)u * SS, SS);
    copy_floats_cg<N, 32>(X[1].p, src + (size_t)(u - s) * SS, SS);
    warp_scombine<N>(l, X[0], X[1], X[2], sc, u - s < s);
    copy_floats<N, 32>(o, X[2].p, SS);
    (void)status;
}

// `pre`: the spine's inclusive suffixes (slot u covers scan tiles 0..u).
// The smoothing elements come from the reduce launch (gb.elems).
template <int N, int M, int NW, int CH>
__global__ void __launch_bounds__(NW * 32) gsmoother_apply_kernel(int64_t T, float* __restrict__ smean,
                                                                  float* __restrict__ scov, GBuf gb,
                                                                  const float* __restrict__ pre, uint32_t* status, const uint32_t* gate) {
    if (gate_closed(gate)) return;
    using SM = GSmem<N, M, NW>;
    constexpr int SS = Dim<N>::SSLOT, NG = SM::NG;
    extern __shared__ __align__(16) char gsm[];
    const int tile = blockIdx.x;
    const int w = threadIdx.x / Grp<N>::GS, r = threadIdx.x & (Grp<N>::GS - 1);
    const int64_t nch = (T + CH - 1) / CH;
    const int64_t u = (int64_t)tile * NG + w;
    if (u >= nch) return;                                 // whole warps; no block barrier in this kernel
    const int64_t cblk = nch - 1 - u;
    const int64_t klo = cblk * CH;
    const int64_t khi = (klo + CH < T ? klo + CH : T) - 1;
    const float* chE = gb.chains + (size_t)u * 2 * SS + SS;
    float* wb = SM::chain(gsm, w);
    SSlot<N> X[3] = {SSlot<N>{wb}, SSlot<N>{wb + SM::SLOT}, SSlot<N>{wb + 2 * SM::SLOT}};
    Scratch<N> s{wb + 3 * SM::SLOT};
    Flags bad = 0u;
    int a = 0;
    bool has = false;
    if (tile != 0) {
        const float* tex = pre + (size_t)(tile - 1) * SS;
        if (w >= 1) {
            copy_floats_cg<N>(X[2].p, tex, SS);
            copy_floats_cg<N>(X[1].p, chE, SS);
            scombine<N, true>(r, X[1], X[2], X[0], s);
        } else {
            copy_floats_cg<N>(X[0].p, tex, SS);
        }
        has = true;
    } else if (w >= 1) {
        copy_floats_cg<N>(X[0].p, chE, SS);                 // E = 0: it ends with the sequence's last element
        has = true;
    }
    float probe = 0.f;
#pragma unroll 1
    for (int64_t k = khi; k >= klo; --k) {
        copy_floats_cg<N>(X[2].p, gb.elems + (size_t)k * SS, SS);
        if (!has) {
            copy_floats<N>(X[a].p, X[2].p, SS);
            has = true;
        } else {
            scombine<N, true>(r, X[2], X[a], X[a ^ 1], s);
            a ^= 1;
        }
        if (r < N) {
            const float g = X[a].g()[r];
            smean[k * N + r] = g;
            float* lrow = scov + (k * N + r) * N;
            const float* src = X[a].L() + r * Dim<N>::NP;
#pragma unroll Unroll<N>::K
            for (int q = 0; q < N; ++q) lrow[q] = src[q];
            probe += g + src[r];
        }
    }
    bad |= !isfinite(probe);
    report_flags(status, bad, gmask<N>(), r == 0);
}

// ---------------------------------------------------------------- time-varying models
// Lemma 3's constants of every step k >= 1 (Q and R symmetrised), by one lane
// group per step, entries spread over its lanes.  One thread per step, its
// matrices in local memory and its accesses a whole model apart, took 64 us
// at nx = 8, 20 Ki steps; this takes 19 us, behind step 0's preparation.
template <int N>
constexpr int kTvThreads = Grp<N>::GS == 8 ? 128 : 64;
template <int N, int M>
__global__ void __launch_bounds__(kTvThreads<N>) tv_const_kernel(TVArgs tv, int64_t T, ModelConst<N, M>* __restrict__ out,
                                                                 uint32_t* __restrict__ status) {
    pdl_trigger();
    constexpr int GS = Grp<N>::GS, NG = kTvThreads<N> / GS;
    struct Sm {
        float F[N * N], Q[N * N], H[M * N], R[M * M], u[N], d[M];
        float HQ[M * N], HF[M * N], tmp[M * N], K[N * M], Ls[M * M], Lsi[M * M];
    };
    __shared__ Sm all[NG];
    const int g = threadIdx.x / GS, r = threadIdx.x & (GS - 1);
    static_assert(M <= GS, "one lane per measurement row");
    Sm& p = all[g];
    Flags bad = 0u;
    for (int64_t k = 1 + (int64_t)blockIdx.x * NG + g; k < T; k += (int64_t)gridDim.x * NG) {
        ModelConst<N, M>& mc = out[k];
        for (int e = r; e < N * N; e += GS) {
            const int a = e / N, c = e % N;
            p.F[e] = __ldg(tv.F + k * N * N + e);
            p.Q[e] = 0.5f * (__ldg(tv.Q + k * N * N + e) + __ldg(tv.Q + k * N * N + c * N + a));
        }
        for (int e = r; e < M * N; e += GS) p.H[e] = __ldg(tv.H + k * M * N + e);
        for (int e = r; e < M * M; e += GS)
            p.R[e] = 0.5f * (__ldg(tv.R + k * M * M + e) + __ldg(tv.R + k * M * M + (e % M) * M + e / M));
        for (int e = r; e < N; e += GS) p.u[e] = tv.u ? __ldg(tv.u + k * N + e) : 0.f;
        if (r < M) p.d[r] = tv.d ? __ldg(tv.d + k * M + r) : 0.f;
        gsync<N>();
        for (int e = r; e < M * N; e += GS) {
            const int q = e / N, a = e % N;
            float sq = 0.f, sf = 0.f;
#pragma unroll 8
            for (int c = 0; c < N; ++c) {
                sq = fmaf(p.H[q * N + c], p.Q[c * N + a], sq);
                sf = fmaf(p.H[q * N + c], p.F[c * N + a], sf);
            }
            p.HQ[e] = sq;
            p.HF[e] = sf;
        }
        gsync<N>();
        for (int e = r; e < M * M; e += GS) {                 // S = R + H Q H^T
            const int i = e / M, j = e % M;
            float t = p.R[e];
#pragma unroll 8
            for (int c = 0; c < N; ++c) t = fmaf(p.HQ[i * N + c], p.H[j * N + c], t);
            p.Ls[e] = t;
        }
        gsync<N>();
        for (int j = 0; j < M; ++j) {                         // Cholesky, row i on lane i
            float t = 0.f;
            if (r >= j && r < M) {
                t = p.Ls[r * M + j];
                for (int l = 0; l < j; ++l) t = fmaf(-p.Ls[r * M + l], p.Ls[j * M + l], t);
            }
            const float sj = __shfl_sync(gmask<N>(), t, j, GS);
            bad |= !(sj > 0.f);
            const float rj = rsqrtf(fmaxf(sj, 1e-37f));
            gsync<N>();
            if (r >= j && r < M) p.Ls[r * M + j] = t * rj;
            gsync<N>();
        }
        if (r < M) {                                          // L_S^{-1}, column r
            for (int i = 0; i < M; ++i) {
                float t = (i == r) ? 1.f : 0.f;
                if (i < r) {
                    p.Lsi[i * M + r] = 0.f;
                    continue;
                }
                for (int l = r; l < i; ++l) t = fmaf(-p.Ls[i * M + l], p.Lsi[l * M + r], t);
                p.Lsi[i * M + r] = t / p.Ls[i * M + i];
            }
            float hu = p.d[r];
            for (int c = 0; c < N; ++c) hu = fmaf(p.H[r * N + c], p.u[c], hu);
            mc.hud[r] = hu;
        }
        gsync<N>();
        for (int e = r; e < M * N; e += GS) {
            const int q = e / N, a = e % N;
            float st = 0.f, sv = 0.f;
            for (int l = 0; l <= q; ++l) {
                st = fmaf(p.Lsi[q * M + l], p.HQ[l * N + a], st);
                sv = fmaf(p.Lsi[q * M + l], p.HF[l * N + a], sv);
            }
            p.tmp[e] = st;
            mc.U[e] = sv;
        }
        for (int e = r; e < M * M; e += GS) mc.Lsi[e] = p.Lsi[e];
        gsync<N>();
        for (int e = r; e < N * M; e += GS) {
            const int a = e / M, q = e % M;
            float sk = 0.f;
            for (int l = q; l < M; ++l) sk = fmaf(p.tmp[l * N + a], p.Lsi[l * M + q], sk);
            p.K[e] = sk;
            mc.K[e] = sk;
        }
        gsync<N>();
        for (int e = r; e < N * N; e += GS) {
            const int a = e / N, b = e % N;
            float sa = p.F[e];
#pragma unroll 4
            for (int q = 0; q < M; ++q) sa = fmaf(-p.K[a * M + q], p.HF[q * N + b], sa);
            mc.A[e] = sa;
            mc.F[e] = p.F[e];
            if (b <= a) {
                float c = p.Q[e];
#pragma unroll 4
                for (int q = 0; q < M; ++q) c = fmaf(-p.tmp[q * N + a], p.tmp[q * N + b], c);
                mc.C[sidx(a, b)] = c;
                mc.Q[sidx(a, b)] = p.Q[e];
            }
        }
        for (int e = r; e < N; e += GS) {
            mc.u[e] = p.u[e];
            mc.b1[e] = 0.f;
        }
        for (int e = r; e < sym_size(N); e += GS) mc.C1[e] = 0.f;
        for (int e = r; e < 4; e += GS) mc.pad[e] = 0.f;
        gsync<N>();
    }
    // not before the end: the steps need nothing of step 0's preparation, but when
    // this kernel is done the chained launches behind it take that one for done too
    pdl_wait();
    report_flags(status, bad, gmask<N>(), r == 0);
}

}  // namespace grp
}  // namespace ks
