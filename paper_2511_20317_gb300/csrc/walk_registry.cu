// Registry of the compiled walk-kernel variants, and the launch shape of small populations.
#include <algorithm>
#include <atomic>
#include <vector>

#include <cuda_runtime.h>

#include "tfg_internal.h"

namespace tfg {
const WalkVariant *walk_variants_group_zt32(int *n);
const WalkVariant *walk_variants_group_z232(int *n);
const WalkVariant *walk_variants_group_64(int *n);
const WalkVariant *walk_variants_wide(int *n);
const WalkVariant *walk_variants_solo_zt32(int *n);
const WalkVariant *walk_variants_solo_z232(int *n);
const WalkVariant *walk_variants_solo_zt64(int *n);
const WalkVariant *walk_variants_solo_z264(int *n);

const WalkVariant *walk_variants(int *count) {
    static std::vector<WalkVariant> all = [] {
        std::vector<WalkVariant> v;
        const WalkVariant *(*parts[])(int *) = {
            walk_variants_group_zt32,
            walk_variants_group_z232,
            walk_variants_group_64,
            walk_variants_wide,
            walk_variants_solo_zt32,
            walk_variants_solo_z232,
            walk_variants_solo_zt64,
            walk_variants_solo_z264,
        };
        for (auto part : parts) {
            int n = 0;
            const WalkVariant *p = part(&n);
            v.insert(v.end(), p, p + n);
        }
        return v;
    }();
    *count = (int)all.size();
    return all.data();
}

int sm_count() {
    static std::atomic<int> known[64];   // by device; 0: not asked yet
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    const bool keep = dev >= 0 && dev < 64;
    if (keep && (sms = known[dev].load(std::memory_order_relaxed)) > 0) return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    if (keep) known[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

int walk_lanes(const SegDesc &d, int64_t warps) {
    if (d.own_block) return 32;
    const int64_t n = std::max(d.beside, d.population);
    int lanes = 32;
    while (lanes > 1 && (n + lanes / 2 - 1) / (lanes / 2) <= warps) lanes /= 2;
    return lanes;
}
}  // namespace tfg
