// ks_window.h -- the settled path's rows: which window of a sequence computes
// which of its rows (plain C++, so that it compiles without CUDA too).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define KS_HD __host__ __device__ __forceinline__
#else
#define KS_HD inline
#endif

namespace ks {

constexpr int kStNT = 128;                        // threads of a block = rows of the head
constexpr int kStHead = 128;
constexpr int kStCH = 16;                         // steps per thread of a window
constexpr int kStWin = kStNT * kStCH;             // 2048 rows
constexpr int kStHalo = 256;                      // rows before and after a window's own rows
constexpr int kStOut = kStWin - 2 * kStHalo;      // rows of an inner window: 1536
constexpr int kStFirst = kStWin - kStHalo;        // rows of a first window (it starts exactly): 1792

// Windows of a sequence of len steps (at least one: the first has the head).
KS_HD int steady_windows(int len) {
    return len <= kStHead + kStWin ? 1 : 1 + (len - kStHead - kStWin + kStOut - 1) / kStOut;
}

// Window j of a sequence: it computes `rows` rows from w0 on (0 when the
// sequence ends in the head), of which [o0, o1) are its own.  Rows inside the
// window are counted from w0: w0 + kStWin can lie beyond 2^31.
struct StWindow {
    bool head, last;
    int o0, o1, w0, rows;
};
KS_HD StWindow steady_window(int len, int j) {
    StWindow w;
    w.head = j == 0;
    w.last = j == steady_windows(len) - 1;
    w.o0 = w.head ? kStHead : kStHead + kStFirst + (j - 1) * kStOut;
    w.w0 = w.head ? kStHead : w.o0 - kStHalo;
    w.o1 = w.last ? len : (w.head ? kStHead + kStFirst : w.o0 + kStOut);
    const int left = len - w.w0;
    w.rows = left < 0 ? 0 : (left < kStWin ? left : kStWin);
    return w;
}

// Rows of the chunk that starts at row c0 of a window.
KS_HD int steady_chunk(int rows, int c0) {
    const int n = rows - c0;
    return n < 0 ? 0 : (n < kStCH ? n : kStCH);
}

}  // namespace ks
