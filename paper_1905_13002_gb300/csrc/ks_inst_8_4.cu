// Instantiation nx = 8, ny = 4: one 8-lane group per chain, four chains (one
// warp) per tile of 4 chains of 8, 16 or 32 steps.
#include "ks_gimpl.cuh"

namespace ks {
extern const GVariant kG_8_4_8, kG_8_4_16;   // ks_inst_8_4_8.cu, ks_inst_8_4_16.cu

namespace {
using G32 = GImpl<8, 4, 1, 32>;
constexpr GVariant kG_8_4_32 = gvariant<G32>();
const GVariant* const kG[3] = {&kG_8_4_8, &kG_8_4_16, &kG_8_4_32};

const GVariant& pick(int64_t T) { return *kG[T < 48 * 1024 ? 0 : T < 160 * 1024 ? 1 : 2]; }

Layout layout(int64_t T, int B) {
    Layout L = G32::layout(T, B);
    for (const GVariant* v : kG) {
        const Layout Lv = v->layout(T, B);
        L.bytes_smooth = std::max(L.bytes_smooth, Lv.bytes_smooth);
        L.bytes_elements = std::max(L.bytes_elements, Lv.bytes_elements);
    }
    return L;
}
size_t tv_bytes(int64_t T) { return std::max({kG[0]->tv_bytes(T), kG[1]->tv_bytes(T), kG[2]->tv_bytes(T)}); }

int smooth_scan(const ks_model* m, int64_t T, const float* fm, const float* fc, void* ws, size_t ws_bytes, float* sm,
                float* sc, cudaStream_t st) {
    if (T < 1 || T > 0x7fffffffLL || ws_bytes < layout(T, 1).bytes_smooth)
        return G32::smooth_scan(m, T, fm, fc, ws, 0, sm, sc, st);   // its argument checks
    return pick(T).smooth_scan(m, T, fm, fc, ws, ws_bytes, sm, sc, st);
}
int smooth(const ks_model* m, const float* y, int64_t T, void* ws, size_t ws_bytes, float* fm, float* fc, float* sm,
           float* sc, cudaStream_t st, void* const* ev) {
    return pick(T).smooth(m, y, T, ws, ws_bytes, fm, fc, sm, sc, st, ev);
}
int smooth_batch(const ks_model_batch* mb, const float* y, int64_t T, void* ws, size_t ws_bytes, float* fm, float* fc,
                 float* sm, float* sc, cudaStream_t st) {
    return pick(T).smooth_batch(mb, y, T, ws, ws_bytes, fm, fc, sm, sc, st);
}

constexpr VTable vtable() {
    VTable t = G32::vtable();
    t.layout = &layout;
    t.smooth_scan = &smooth_scan;
    t.smooth = &smooth;
    t.smooth_batch = &smooth_batch;
    t.tv_bytes = &tv_bytes;
    return t;
}
}  // namespace

extern const VTable kImpl_8_4 = vtable();
}
