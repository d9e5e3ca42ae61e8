// nx = 8 scans with chains of 16 steps (ks_inst_8_4.cu picks by length).
#include "ks_gimpl.cuh"

namespace ks {
extern const GVariant kG_8_4_16 = gvariant<GImpl<8, 4, 1, 16>>();
}
