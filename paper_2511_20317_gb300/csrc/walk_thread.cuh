// Variants of the thread-per-walker mapping: the walker with kept factor classes
// (walk_link.cuh), and the one that tests every slot in every step (walk_solo.cuh) where
// that is still the faster.
#pragma once
#include "walk_link.cuh"
#include "walk_solo.cuh"

namespace tfg {

// Keeping the classes pays when most steps only read them, and when the rank is large.
// It does not when nearly every step changes the scheme and nothing else in the step
// needs the search: walk policy 2 (no reduction test after a flip) on few slots or over
// Z_2 (9 of 10 flips are accepted), and walk policy 1 on the smallest ranks, where
// expansions and reductions alternate.  A small population is bound by the latency
// of one step, where the classes' short dependent loops cost most.  Measured, 300 steps,
// ms testing every slot / keeping classes:
//   policy 1: (2,2,2) Z_T 1000 walkers 3.25 / 4.18, (2,2,3) Z_T 3.05 / 2.69, 30000 walkers 5.08 / 3.28;
//     Z_2 (2,3,3) 30000 2.31 / 2.47, (2,3,4) 1000 1.70 / 2.00, 30000 3.00 / 2.20, (2,4,5) 1000 3.35 / 1.71
//   policy 2: Z_T (2,3,3) 1000 0.40 / 0.48, 30000 0.53 / 0.53, (2,3,4) 30000 0.62 / 0.56, (2,4,5) 1000 0.70 / 0.63;
//     Z_2 (2,3,4) 30000 0.45 / 0.63, (4,4,5) 30000 1.04 / 1.42
template <int MODE, class Wd>
inline bool every_slot_faster(const SegDesc &d) {
    constexpr bool z2 = MODE == TFG_MODE_Z2;
    constexpr int64_t small = 16384;
    if (d.walk_policy == 2) return z2 || (sizeof(Wd) == 4 && (d.R <= 20 || d.n_walkers < small));
    if (d.walk_policy == 1) return sizeof(Wd) == 4 && (z2 ? d.R <= 24 || d.n_walkers < small : d.R <= 12);
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
void launch_walk_thread(const SegDesc &d, int32_t steps, int grid, int block, cudaStream_t st) {
    if constexpr (has_every_slot<MODE, Wd, CAP>()) {
        if (every_slot_faster<MODE, Wd>(d)) {
            launch_walk_solo<MODE, Wd, CAP, 128>(d, steps, (int)((d.n_walkers + 127) / 128), 128, st);
            return;
        }
    }
    launch_walk_link<MODE, Wd, (CAP + 31) / 32>(d, steps, grid, block, st);
}

// Bit-sliced kernels of Z_T (walk_solo.cuh): 971 instructions a warp-step at 64% of the issue
// rate, against about 600 with kept classes.  The plateau policy keeps classes from more
// than a warp a scheduler on; below, a step's latency counts, and there the slices are the
// faster.  Measured, (3,3,3), ms per 1000 steps, slices / classes: 1024 walkers 1.36 / 1.44,
// 14000 1.39 / 1.46, 20000 1.77 / 1.57, 40000 2.29 / 1.74, 65536 2.88 / 2.43, 131072 5.2 /
// 4.66; policy 1, 20000 walkers 2.35 / 2.71, 65536 4.11 / 4.01.  Over Z_2 (643
// instructions, half the slices, in registers) slices are always the faster: 65536 walkers
// 2.05 / 2.50.
constexpr int64_t kSlicedMax = 152 * 128;
template <class Wd, int BT, int FL, bool SQ>
void prepare_walk_sliced_zt() {
    prepare_walk_solo<TFG_MODE_ZT, Wd, 32, BT, FL, SQ>();
    prepare_walk_link<TFG_MODE_ZT, Wd, 1>();
}
template <class Wd, int BT, int FL, bool SQ>
void launch_walk_sliced_zt(const SegDesc &d, int32_t steps, int grid, int block, cudaStream_t st) {
    if (d.walk_policy == 0 && d.n_walkers > kSlicedMax)
        launch_walk_link<TFG_MODE_ZT, Wd, 1>(d, steps, (int)((d.n_walkers + 31) / 32), 32, st);
    else
        launch_walk_solo<TFG_MODE_ZT, Wd, 32, BT, FL, SQ>(d, steps, grid, block, st);
}

}  // namespace tfg

// capacity CAP, BLOCK walkers per block
#define TFG_THREAD_VARIANT(MODE, WD, BITS, CAP, BLOCK) \
    WalkVariant{MODE, BITS, 1, 1, CAP, BLOCK, &launch_walk_thread<MODE, WD, CAP>, \
                reinterpret_cast<const void *>(&dev::walk_link_kernel<MODE, WD, (CAP + 31) / 32, BITS == 64, false>), \
                &prepare_walk_thread<MODE, WD, CAP>}
// 32-bit terms beyond 32 slots: not selectable by tfg_params.mapping, and by default for large
// populations (default_variant)
#define TFG_THREAD_VARIANT_AUTO(MODE, WD, BITS, CAP, BLOCK) \
    WalkVariant{MODE, BITS, 1, 1, CAP, BLOCK, &launch_walk_link<MODE, WD, (CAP + 31) / 32>, \
                reinterpret_cast<const void *>(&dev::walk_link_kernel<MODE, WD, (CAP + 31) / 32, BITS == 64, false>), \
                &prepare_walk_link<MODE, WD, (CAP + 31) / 32>, 0, 0, 0, true}
// Z_T bit-sliced, 32 slots: factors of at most FL coefficients (SQ: exactly FL each)
#define TFG_SLICED_ZT_VARIANT(WD, BITS, BT, FL, SQ) \
    WalkVariant{TFG_MODE_ZT, BITS, 1, 1, 32, BT, &launch_walk_sliced_zt<WD, BT, FL, SQ>, \
                reinterpret_cast<const void *>(dev::solo_kernel<TFG_MODE_ZT, WD, 32, BT, FL, SQ>()), \
                &prepare_walk_sliced_zt<WD, BT, FL, SQ>, 0, FL, SQ ? 1 : 0}
