// Thread-per-walker variants: Z_2, terms of 33 to 64 coefficients.  The first of a
// capacity is its default; the others are walkers-per-block choices of the
// same kernel.
#include "walk_thread.cuh"

namespace tfg {
const WalkVariant *walk_variants_solo_z264(int *n) {
    static const WalkVariant v[] = {
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 16, 64),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 32, 64),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 48, 64),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 64, 64),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 72, 64),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 88, 64),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 16, 128),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 32, 128),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 48, 128),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 64, 128),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 72, 128),
        TFG_THREAD_VARIANT(TFG_MODE_Z2, uint64_t, 64, 88, 128),
    };
    *n = (int)(sizeof(v) / sizeof(v[0]));
    return v;
}
}  // namespace tfg
