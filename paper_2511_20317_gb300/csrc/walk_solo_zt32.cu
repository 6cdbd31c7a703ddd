// Thread-per-walker variants: Z_T, terms of at most 32 coefficients.
#include "walk_thread.cuh"

#ifndef TFG_SLICED_ZT_BLOCK
#define TFG_SLICED_ZT_BLOCK 64   // threads per block of the bit-sliced kernel (shared-memory slices)
#endif

namespace tfg {
const WalkVariant *walk_variants_solo_zt32(int *n) {
    static const WalkVariant v[] = {
        TFG_THREAD_VARIANT(TFG_MODE_ZT, uint32_t, 32, 12, 32),
        TFG_THREAD_VARIANT(TFG_MODE_ZT, uint32_t, 32, 16, 32),
        TFG_THREAD_VARIANT(TFG_MODE_ZT, uint32_t, 32, 24, 32),
        TFG_THREAD_VARIANT(TFG_MODE_ZT, uint32_t, 32, 32, 32),
        TFG_THREAD_VARIANT_AUTO(TFG_MODE_ZT, uint32_t, 32, 64, 32),
        TFG_SLICED_ZT_VARIANT(uint32_t, 32, TFG_SLICED_ZT_BLOCK, 9, false),
        TFG_SLICED_ZT_VARIANT(uint32_t, 32, TFG_SLICED_ZT_BLOCK, 9, true),
    };
    *n = (int)(sizeof(v) / sizeof(v[0]));
    return v;
}
}  // namespace tfg
