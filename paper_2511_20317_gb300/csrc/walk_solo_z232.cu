// Thread-per-walker variants: Z_2, terms of at most 32 coefficients.
#include "walk_thread.cuh"

#ifndef TFG_SLICED_Z2_BLOCK
#define TFG_SLICED_Z2_BLOCK 128   // threads per block of the bit-sliced kernel (register slices)
#endif

namespace tfg {
const WalkVariant *walk_variants_solo_z232(int *n) {
    static const WalkVariant v[] = {
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint32_t, 32, 12, 32),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint32_t, 32, 16, 32),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint32_t, 32, 24, 32),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint32_t, 32, 32, 32),
        TFG_THREAD_VARIANT_AUTO(TFG_MODE_Z2, uint32_t, 32, 64, 32),
        TFG_SOLO_SLICED_VARIANT(TFG_MODE_Z2, uint32_t, 32, 32, TFG_SLICED_Z2_BLOCK, 9, false),
        TFG_SOLO_SLICED_VARIANT(TFG_MODE_Z2, uint32_t, 32, 32, TFG_SLICED_Z2_BLOCK, 9, true),
    };
    *n = (int)(sizeof(v) / sizeof(v[0]));
    return v;
}
}  // namespace tfg
