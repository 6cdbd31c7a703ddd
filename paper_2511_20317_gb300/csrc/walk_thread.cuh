// Variants of the thread-per-walker mapping: the walker with kept factor classes
// (walk_link.cuh), and the one that tests every slot in every step (walk_solo.cuh) where
// that is still the faster.
#pragma once
#include <algorithm>

#include "walk_link.cuh"
#include "walk_solo.cuh"

namespace tfg {

// Lanes a warp would get if the population kept classes: few for a small one.
inline int class_lanes(const SegDesc &d) { return walk_lanes(d, (int64_t)8 * sm_count()); }
// At most a full warp a scheduler: a step's latency counts, not its instructions.
inline bool one_warp_each(const SegDesc &d) { return d.population <= (int64_t)128 * sm_count(); }

// Keeping the classes pays when most steps only read them, and when the rank is large.
// It does not when nearly every step changes the scheme and nothing else in the step
// needs the search: walk policy 2 (no reduction test after a flip) on few slots or over
// Z_2 (9 of 10 flips are accepted), and walk policy 1 on the smallest ranks, where
// expansions and reductions alternate.  Small populations keep classes all the same: their
// short dependent loops are what few lanes a warp save most on.  Measured, 300 steps, ms
// testing every slot / keeping classes (both in few lanes where that is faster):
//   policy 1: Z_T (2,2,2) 11 slots, 7500 walkers 2.61 / 2.61, 10000 3.17 / 2.83, 14000 3.17 / 3.26, 30000 4.18 /
//     4.35; 14 slots, 14000 4.65 / 4.34, 65536 12.4 / 8.1
//     Z_2 (2,2,2) 11 slots, 2500 1.00 / 0.69, 5000 0.97 / 0.95, 7500 0.97 / 1.33, 65536 2.53 / 3.73; (2,2,3) 15
//     slots, 2500 1.05 / 0.69, 5000 1.07 / 0.93, 7500 1.28 / 1.34, 30000 1.81 / 2.69
//     Z_2 (2,2,3) 18 slots, 10000 1.75 / 1.48, 14000 1.71 / 2.04; (2,3,3) 21 slots, 10000 1.68 / 1.23, 14000 1.71 /
//     1.61, 18000 1.60 / 1.69; 24 slots, 10000 1.70 / 1.41, 14000 1.69 / 1.89; (2,2,5) 26 slots, 14000 1.85 / 1.59
//   policy 2: Z_T (2,2,3) 1200 0.31 / 0.26, 5000 0.35 / 0.43; (2,3,4) 1200 0.39 / 0.26, 5000 0.43 /
//     0.42, 18000 0.45 / 0.51, 30000 0.62 / 0.56; Z_2 (2,3,4) 1200 0.33 / 0.34, 18000 0.35 / 0.58;
//     (4,4,5) 1200 0.67 / 0.50, 5000 0.68 / 0.73, 30000 1.05 / 1.43
template <int MODE, class Wd>
inline bool every_slot_faster(const SegDesc &d) {
    constexpr bool z2 = MODE == TFG_MODE_Z2, small = sizeof(Wd) == 4;
    const int lanes = class_lanes(d);
    if (d.walk_policy == 2) {
        if (z2) return small || lanes > 1;
        return small && (d.R <= 20 ? lanes > 2 : lanes > 4 && one_warp_each(d));
    }
    if (d.walk_policy == 1) {   // by walkers an SM
        const int64_t walkers = std::max(d.beside, d.population);
        return small && d.R <= (z2 ? 24 : 12) && walkers > (int64_t)(z2 && d.R <= 16 ? 40 : 80) * sm_count();
    }
    return false;
}

// Capacities at which the every-slot walker is compiled (its loops are unrolled to the capacity)
template <int MODE, class Wd, int CAP>
constexpr bool has_every_slot() {
    return (sizeof(Wd) == 4 && CAP <= 32) || MODE == TFG_MODE_Z2;
}

template <int MODE, class Wd, int CAP>
void prepare_walk_thread() {
    prepare_walk_link<MODE, Wd, (CAP + 31) / 32>();
    if constexpr (has_every_slot<MODE, Wd, CAP>()) prepare_walk_solo<MODE, Wd, CAP, 128>();
}

template <int MODE, class Wd, int CAP>
LaunchShape thread_shape(const SegDesc &d, int block) {
    if constexpr (has_every_slot<MODE, Wd, CAP>())
        if (every_slot_faster<MODE, Wd>(d)) return solo_shape<MODE, Wd, CAP, 128>(d, block);
    return link_launch_shape<MODE, Wd, (CAP + 31) / 32>(d, block);
}
template <int MODE, class Wd, int CAP>
void launch_walk_thread(const SegDesc &d, int32_t steps, int grid, int block, cudaStream_t st) {
    if constexpr (has_every_slot<MODE, Wd, CAP>()) {
        if (every_slot_faster<MODE, Wd>(d)) {
            launch_walk_solo<MODE, Wd, CAP, 128>(d, steps, grid, block, st);
            return;
        }
    }
    launch_walk_link<MODE, Wd, (CAP + 31) / 32>(d, steps, grid, block, st);
}

// Bit-sliced kernels of Z_T (walk_solo.cuh): 971 instructions a warp-step at 64% of the issue
// rate, against 600 to 800 with kept classes.  The plateau policy keeps classes beyond a warp a
// scheduler, and so does every policy in a small population.  Measured, (3,3,3), slices /
// classes, ms: 300 steps, 1200 walkers 0.35 / 0.24, 5000 0.43 / 0.41, 10000 0.44 / 0.47; policy
// 1, 2500 0.65 / 0.59; policy 2, 2500 0.365 / 0.34, 5000 0.38 / 0.43; 1000 steps, 14000 1.39 / 1.46,
// 20000 1.77 / 1.57, 40000 2.29 / 1.74, 65536 2.88 / 2.43, 131072 5.2 / 4.66; policy 1, 20000 2.35 /
// 2.71, 65536 4.11 / 4.01.  Over Z_2 (643 instructions, half the slices, in registers)
// the slices are the faster or as fast: 300 walkers 0.30 / 0.29, 5000 0.32 / 0.48, 65536 2.05 / 2.50.
inline bool slices_faster(const SegDesc &d) {
    const int lanes = class_lanes(d);
    return d.walk_policy == 0 ? lanes > 4 && one_warp_each(d) : lanes > 2;
}
template <class Wd, int BT, int FL, bool SQ>
void prepare_walk_sliced_zt() {
    prepare_walk_solo<TFG_MODE_ZT, Wd, 32, BT, FL, SQ>();
    prepare_walk_link<TFG_MODE_ZT, Wd, 1>();
}
inline int sliced_class_block(const SegDesc &d, int block) { return d.own_block ? block : 32; }
template <class Wd, int BT, int FL, bool SQ>
LaunchShape sliced_zt_shape(const SegDesc &d, int block) {
    if (slices_faster(d)) return solo_shape<TFG_MODE_ZT, Wd, 32, BT, FL, SQ>(d, block);
    return link_launch_shape<TFG_MODE_ZT, Wd, 1>(d, sliced_class_block(d, block));
}
template <class Wd, int BT, int FL, bool SQ>
void launch_walk_sliced_zt(const SegDesc &d, int32_t steps, int grid, int block, cudaStream_t st) {
    if (slices_faster(d))
        launch_walk_solo<TFG_MODE_ZT, Wd, 32, BT, FL, SQ>(d, steps, grid, block, st);
    else
        launch_walk_link<TFG_MODE_ZT, Wd, 1>(d, steps, grid, sliced_class_block(d, block), st);
}

}  // namespace tfg

// capacity CAP, BLOCK walkers per block
#define TFG_THREAD_VARIANT(MODE, WD, BITS, CAP, BLOCK) \
    WalkVariant{MODE, BITS, 1, 1, CAP, BLOCK, &launch_walk_thread<MODE, WD, CAP>, \
                reinterpret_cast<const void *>(&dev::walk_link_kernel<MODE, WD, (CAP + 31) / 32, BITS == 64, false>), \
                &prepare_walk_thread<MODE, WD, CAP>, &thread_shape<MODE, WD, CAP>}
// 32-bit terms beyond 32 slots: not selectable by tfg_params.mapping, and by default for large
// populations (default_variant)
#define TFG_THREAD_VARIANT_AUTO(MODE, WD, BITS, CAP, BLOCK) \
    WalkVariant{MODE, BITS, 1, 1, CAP, BLOCK, &launch_walk_link<MODE, WD, (CAP + 31) / 32>, \
                reinterpret_cast<const void *>(&dev::walk_link_kernel<MODE, WD, (CAP + 31) / 32, BITS == 64, false>), \
                &prepare_walk_link<MODE, WD, (CAP + 31) / 32>, &link_launch_shape<MODE, WD, (CAP + 31) / 32>, 0, 0, 0, true}
// Z_T bit-sliced, 32 slots: factors of at most FL coefficients (SQ: exactly FL each)
#define TFG_SLICED_ZT_VARIANT(WD, BITS, BT, FL, SQ) \
    WalkVariant{TFG_MODE_ZT, BITS, 1, 1, 32, BT, &launch_walk_sliced_zt<WD, BT, FL, SQ>, \
                reinterpret_cast<const void *>(dev::solo_kernel<TFG_MODE_ZT, WD, 32, BT, FL, SQ>()), \
                &prepare_walk_sliced_zt<WD, BT, FL, SQ>, &sliced_zt_shape<WD, BT, FL, SQ>, 0, FL, SQ ? 1 : 0}
