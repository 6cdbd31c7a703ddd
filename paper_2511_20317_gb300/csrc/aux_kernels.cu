// Auxiliary kernels around the walk: population set-up, exact verification of
// best schemes (Eq. (1)), best-walker selection and population statistics.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <type_traits>

#include "tfg_internal.h"
#include "pterm.cuh"

namespace tfg {
namespace {

// ---- population set-up: every walker starts from the prepared start scheme
template <class Wd>
__global__ void replicate_kernel(const SegDesc d, const Wd *__restrict__ start, int32_t r0,
                                 uint32_t id_base, int32_t fidx, uint32_t start_nnz) {
    const int64_t w = blockIdx.x;
    if (w >= d.n_walkers) return;
    const size_t per = (size_t)d.R * d.nws;
    Wd *s = reinterpret_cast<Wd *>(d.slots) + per * w;
    Wd *b = reinterpret_cast<Wd *>(d.best) + per * w;
    for (size_t e = threadIdx.x; e < per; e += blockDim.x) {
        const Wd v = (e < (size_t)r0 * d.nws) ? start[e] : Wd(0);
        s[e] = v;
        b[e] = v;
    }
    if (threadIdx.x == 0) {
        tfg_walker_info h;
        h.r = r0; h.best_r = r0; h.r_max = d.R; h.format = fidx;
        h.t = 0; h.plateau = 0; h.best_t = 0;
        h.walker_id = id_base + (uint32_t)w;
        h.digest = 0xCBF29CE484222325ull ^ (uint64_t)h.walker_id;
        h.accepted = h.rejected = h.nocand = h.drops = h.merges = h.plus = h.reductions = 0;
        h.best_nnz = start_nnz;
        d.hdr[w] = h;
    }
}

// ---- re-seeding: walker `first`'s live slots hold the new packed scheme;
// copy them to the live slots of walkers first+1 .. first+count-1 and to the
// best slots of all of them, and restart their records at rank r.
template <class Wd>
__global__ void reseed_kernel(const SegDesc d, int64_t first, int32_t r, uint32_t nnz) {
    const int64_t w = first + blockIdx.x;
    const size_t per = (size_t)d.R * d.nws;
    const Wd *src = reinterpret_cast<const Wd *>(d.slots) + per * first;
    Wd *s = reinterpret_cast<Wd *>(d.slots) + per * w;
    Wd *b = reinterpret_cast<Wd *>(d.best) + per * w;
    for (size_t e = threadIdx.x; e < per; e += blockDim.x) {
        const Wd v = src[e];
        if (w != first) s[e] = v;
        b[e] = v;
    }
    if (threadIdx.x == 0) {
        tfg_walker_info &h = d.hdr[w];
        h.r = r;
        h.best_r = r;
        h.plateau = 0;
        h.best_t = h.t;
        h.best_nnz = nnz;
    }
}

// ---- Eq. (1) on every walker's best scheme, by sparse accumulation with a count
// of the non-zero entries.  A team (a warp, or a block when the tensor is large)
// owns one accumulator per entry of the difference D = sum_l u_l (x) v_l (x) w_l -
// (matrix-multiplication tensor), and adds only the products of non-zero
// coefficients and the tensor's mnp ones.  Every addition is a returning
// shared-memory atomic, so the thread sees the entry leave or reach zero and
// counts +1 or -1: the sum of the counts is the number of non-zero entries of D,
// and Eq. (1) holds iff it is zero.  No pass over the entries is needed, neither
// to compare them (there are up to 2^18 per walker against a few thousand
// products) nor to clear them: after a scheme that passes they are all zero
// again, and the team takes its next walker.
// Entries are FB-bit fields: Z_T holds the sum plus a bias of 2^(FB-1), Z_2 one
// bit, changed by XOR.  |D| <= rank + 1 fits 8 bits up to rank 126; above, 8 bits
// nearly always do, since an entry is covered by few terms: an addition that
// would leave them is seen by its old value, and the walker is done again with
// 16 bits (ranks are at most 1023).  Tensors beyond the team's shared memory
// are done in slabs of u-indices.
// The products of a term are spread over a warp's lanes, by lists of the positions of
// its non-zero coefficients: terms have 1 to 300 products, and loops over the
// set bits in every lane run the longest lane's nesting (45 ms on the large
// formats, 8.0 ms on the five formats below).
// Measured on 32768 walkers each of (4,5,12), (5,6,10), (6,7,9): 65.3 ms with a dense
// compare of every entry (index divisions for each), now 10.9 ms; five formats up
// to (4,4,5), 262144 walkers: 9.9 ms, now 3.8 ms; (3,3,3) 65536 Z_T + 65536 Z_2
// walkers: 1.53 ms, now 0.58 ms.
constexpr int kVerifyWarpBlock = 128;    // threads per block of warp teams
constexpr int kVerifyTeam = 1024;        // threads of a block team (256: 16.7 ms, 512: 12.0, 1024: 10.9 on the large formats)

// Change of the number of non-zero entries by one addition, from the old word.
template <int FB>
struct Tally {
    static constexpr uint32_t FM = FB == 32 ? ~0u : (1u << FB) - 1u, BIAS = 1u << (FB - 1);
    int nz = 0;
    bool over = false;   // the field would have left its range
    __device__ __forceinline__ static uint32_t add(uint32_t *acc, int e, bool minus) {
        if constexpr (FB == 1) {
            return (atomicXor(&acc[e >> 5], 1u << (e & 31)) >> (e & 31)) & 1u;
        } else {
            constexpr int PER = 32 / FB;
            const int sh = (e % PER) * FB;
            return (atomicAdd(&acc[e / PER], minus ? 0u - (1u << sh) : (1u << sh)) >> sh) & FM;
        }
    }
    __device__ __forceinline__ void see(uint32_t old, bool minus) {
        if constexpr (FB == 1) {
            nz += old ? -1 : 1;
        } else {
            const uint32_t now = minus ? old - 1u : old + 1u;
            nz += (int)(old == BIAS) - (int)(now == BIAS);
            over |= (minus ? old : now) == (minus ? 0u : FM + 1u);
        }
    }
};

// D's non-zero entries of u-indices [a0, a1), added up in acc by the warp: one term
// after another (first, first + step, ...), the positions of its non-zero
// coefficients (at most 127, bit 7 the sign) in the warp's lists, then its
// products over the lanes.  inv[n] = ceil(2^32 / n), n < 129.
template <class Wd, int FB>
__device__ __forceinline__ void add_terms(const SegDesc &d, const Wd *b, int r, int a0, int a1, uint32_t *acc,
                                          uint8_t (*list)[128], const uint32_t *inv, int first, int step, int lane,
                                          Tally<FB> &tl) {
    constexpr int WB = (int)sizeof(Wd) * 8;
    const int LU = d.m * d.n, LV = d.n * d.p, LW = d.p * d.m;
    // lane q holds word q of the term (at most 12), fetched one term ahead
    Wd ahead = (first < r && lane < d.nws) ? b[(size_t)first * d.nws + lane] : Wd(0);
    for (int l = first; l < r; l += step) {
        const Wd words = ahead;
        if (l + step < r && lane < d.nws) ahead = b[(size_t)(l + step) * d.nws + lane];
        int cnt[3];
        if (d.tw == 1 && a1 - a0 == LU) {
            // the whole term in one word per sign: lane e takes bits e and e + 32
            const Wd pw = __shfl_sync(0xffffffffu, words, 0);
            const Wd nw = FB == 1 ? Wd(0) : __shfl_sync(0xffffffffu, words, 1), nz = pw | nw;
            const int ln = LU + LV, lt = ln + LW;
#pragma unroll
            for (int h = 0; h < WB; h += 32) {
                const int bit = h + lane;
                if ((nz >> bit) & 1) {
                    const int f = bit < LU ? 0 : (bit < ln ? 1 : 2);
                    const Wd below = nz & ((Wd(1) << bit) - 1) & (Wd)(f == 0 ? d.fmask[0][0] : (f == 1 ? d.fmask[1][0] : d.fmask[2][0]));
                    const int rank = sizeof(Wd) == 8 ? __popcll(below) : __popc((uint32_t)below);
                    list[f][rank] = (uint8_t)((bit - (f == 0 ? 0 : (f == 1 ? LU : ln))) | ((int)((nw >> bit) & 1) << 7));
                }
                if (h + 32 >= lt) break;
            }
#pragma unroll
            for (int f = 0; f < 3; ++f)
                cnt[f] = sizeof(Wd) == 8 ? __popcll(nz & d.fmask[f][0]) : __popc((uint32_t)(nz & d.fmask[f][0]));
        } else {
            const int lo[3] = {d.fbase[0] + a0, d.fbase[1], d.fbase[2]};
            const int len[3] = {a1 - a0, LV, LW};
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                cnt[f] = 0;
                for (int e0 = 0; e0 < len[f]; e0 += 32) {
                    const int e = e0 + lane, bit = lo[f] + min(e, len[f] - 1);
                    bool pv = (__shfl_sync(0xffffffffu, words, bit / WB) >> (bit % WB)) & 1, nv = false;
                    if (FB != 1) nv = (__shfl_sync(0xffffffffu, words, d.tw + bit / WB) >> (bit % WB)) & 1;
                    pv = pv && e < len[f];
                    nv = nv && e < len[f];
                    const unsigned m = __ballot_sync(0xffffffffu, pv || nv);
                    if (pv || nv) list[f][cnt[f] + __popc(m & ((1u << lane) - 1u))] = (uint8_t)(e | (nv ? 128 : 0));
                    cnt[f] += __popc(m);
                }
            }
        }
        __syncwarp();
        const int nvw = cnt[1] * cnt[2], total = cnt[0] * nvw;
        for (int q = lane; q < total; q += 32) {
            int iu = 0, rem = q;
            if (cnt[0] > 1) {
                iu = nvw == 1 ? q : (nvw < 129 ? (int)__umulhi((uint32_t)q, inv[nvw]) : q / nvw);
                rem = q - iu * nvw;
            }
            const int iv = cnt[2] == 1 ? rem : (int)__umulhi((uint32_t)rem, inv[cnt[2]]);
            const int u = list[0][iu], v = list[1][iv], w = list[2][rem - iv * cnt[2]];
            const bool minus = ((u ^ v ^ w) & 128) != 0;
            tl.see(Tally<FB>::add(acc, ((u & 127) * LV + (v & 127)) * LW + (w & 127), minus), minus);
        }
        __syncwarp();
    }
}

// WIDE: 8-bit fields whose range a rank of R could leave
template <class Wd, bool BLOCK, int FB, bool WIDE>
__global__ void __launch_bounds__(BLOCK ? kVerifyTeam : kVerifyWarpBlock)
    verify_best_kernel(const SegDesc d, int64_t first, int64_t count, int slab_rows, int slab_words,
                       unsigned long long *failures) {
    extern __shared__ __align__(16) uint32_t vsm[];
    __shared__ int sh_nz;
    __shared__ uint8_t lists[(BLOCK ? kVerifyTeam : kVerifyWarpBlock) / 32][3][128];
    __shared__ uint32_t inv[129];
    constexpr int TEAM = BLOCK ? kVerifyTeam : 32;
    const int teams = BLOCK ? 1 : kVerifyWarpBlock / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tid = BLOCK ? threadIdx.x : lane, team = BLOCK ? 0 : warp;
    uint32_t *acc = vsm + (size_t)team * slab_words;
    const int n = d.n, p = d.p, LU = d.m * n, LV = n * p, LW = p * d.m;
    auto sync = [&] { if constexpr (BLOCK) __syncthreads(); else __syncwarp(); };
    auto clear = [&](uint32_t zero) {
        sync();
        for (int e = tid; e < slab_words; e += TEAM) acc[e] = zero;
        sync();
    };
    // one walker: the number of non-zero entries of D, or -1 when a field left its range
    auto difference = [&](auto field, const Wd *b, int r, int rows) -> int {
        constexpr int F = decltype(field)::value;
        for (int a0 = 0; a0 < LU; a0 += rows) {
            const int a1 = min(LU, a0 + rows);
            Tally<F> tl;
            // the tensor's ones: a = (i,k), b = (k,j), c = (j,i)
            for (int e = tid; e < (a1 - a0) * p; e += TEAM) {
                const int ra = e / p, j = e - ra * p, a = a0 + ra, i = a / n, k = a - i * n;
                tl.see(Tally<F>::add(acc, (ra * LV + k * p + j) * LW + j * d.m + i, true), true);
            }
            add_terms<Wd, F>(d, b, r, a0, a1, acc, lists[warp], inv, BLOCK ? warp : 0, BLOCK ? TEAM / 32 : 1, lane, tl);
            int nz = __reduce_add_sync(0xffffffffu, tl.nz);
            bool over = __any_sync(0xffffffffu, tl.over);
            if constexpr (BLOCK) {
                if (threadIdx.x == 0) sh_nz = 0;
                over = __syncthreads_or(over);
                if (lane == 0 && nz) atomicAdd(&sh_nz, nz);
                __syncthreads();
                nz = sh_nz;
                __syncthreads();
            }
            if (over) return -1;
            if (nz != 0) return nz;
        }
        return 0;
    };
    constexpr uint32_t kZero = FB == 1 ? 0u : (FB == 8 ? 0x80808080u : 0x80008000u);
    for (int e = threadIdx.x; e < 129; e += blockDim.x) inv[e] = e < 2 ? 0u : 0xffffffffu / (uint32_t)e + 1u;
    __syncthreads();
    clear(kZero);
    for (int64_t w = (int64_t)blockIdx.x * teams + team; w < count; w += (int64_t)gridDim.x * teams) {
        const int r = d.hdr[first + w].best_r;
        const Wd *b = reinterpret_cast<const Wd *>(d.best) + (size_t)d.R * d.nws * (first + w);
        bool bad = r < 0 || r > d.R;
        if (!bad) {
            int nz = difference(std::integral_constant<int, FB>{}, b, r, slab_rows);
            if (nz) clear(kZero);
            if constexpr (WIDE) {
                if (nz < 0) {
                    clear(0x80008000u);
                    nz = difference(std::integral_constant<int, 16>{}, b, r, max(1, (int)(2 * (int64_t)slab_words / ((int64_t)LV * LW))));
                    clear(kZero);
                }
            }
            bad = nz != 0;
        }
        if (bad && tid == 0) atomicAdd(failures, 1ull);
    }
}

__global__ void argmin_kernel(const SegDesc d, unsigned long long *key) {
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long k = ~0ull;
    if (w < d.n_walkers) k = ((unsigned long long)(uint32_t)d.hdr[w].best_r << 32) | (unsigned long long)(uint32_t)w;
    // warp minimum, then one atomic per warp
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, k, o);
        k = y < k ? y : k;
    }
    if ((threadIdx.x & 31) == 0 && k != ~0ull) atomicMin(key, k);
}

// Counters, extremes and histogram of a population.  A block sums its walkers'
// records in registers, then across its warps, and adds one value per counter to
// the totals (every walker adding to the same eleven words by itself serialised
// on them: 0.34 ms for 65536 walkers, now 5 us).
constexpr int kStatSums = 9;
__global__ void __launch_bounds__(256) stats_kernel(const SegDesc d, unsigned long long *sums, int *minmax,
                                                    unsigned long long *hist, int hist_len) {
    extern __shared__ int sh_hist[];   // [hist_len]
    __shared__ unsigned long long sh_sum[kStatSums];
    __shared__ int sh_min, sh_max;
    for (int e = threadIdx.x; e < hist_len; e += blockDim.x) sh_hist[e] = 0;
    if (threadIdx.x < kStatSums) sh_sum[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        sh_min = INT_MAX;
        sh_max = INT_MIN;
    }
    __syncthreads();
    unsigned long long v[kStatSums] = {};
    int lo = INT_MAX, hi = INT_MIN;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < d.n_walkers; w += (int64_t)gridDim.x * blockDim.x) {
        const tfg_walker_info &h = d.hdr[w];
        v[0] += 1;
        v[1] += (unsigned long long)h.t;
        v[2] += (unsigned long long)h.accepted;
        v[3] += (unsigned long long)h.rejected;
        v[4] += (unsigned long long)h.nocand;
        v[5] += (unsigned long long)h.drops;
        v[6] += (unsigned long long)h.merges;
        v[7] += (unsigned long long)h.plus;
        v[8] += (unsigned long long)h.reductions;
        lo = min(lo, h.best_r);
        hi = max(hi, h.best_r);
        if (h.best_r >= 0 && h.best_r < hist_len) atomicAdd(&sh_hist[h.best_r], 1);
    }
#pragma unroll
    for (int k = 0; k < kStatSums; ++k) {
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&sh_sum[k], v[k]);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&sh_min, lo);
        atomicMax(&sh_max, hi);
    }
    __syncthreads();
    if (threadIdx.x < kStatSums) atomicAdd(&sums[threadIdx.x], sh_sum[threadIdx.x]);
    if (threadIdx.x == 0) {
        atomicMin(&minmax[0], sh_min);
        atomicMax(&minmax[1], sh_max);
    }
    for (int e = threadIdx.x; e < hist_len; e += blockDim.x)
        if (sh_hist[e]) atomicAdd(&hist[e], (unsigned long long)sh_hist[e]);
}

__global__ void philox_kernel(const uint32_t *ctr, int n, uint32_t k0, uint32_t k1, uint32_t *out) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const dev::U4 x = dev::philox10(ctr[4 * e], ctr[4 * e + 1], ctr[4 * e + 2], ctr[4 * e + 3], k0, k1);
    out[4 * e] = x.x; out[4 * e + 1] = x.y; out[4 * e + 2] = x.z; out[4 * e + 3] = x.w;
}

}  // namespace

void launch_replicate(const SegDesc &d, const void *start_words, int32_t r0, uint32_t id_base,
                      int32_t format_idx, uint32_t start_nnz, cudaStream_t st) {
    if (d.n_walkers <= 0) return;
    if (d.word_bits == 32)
        replicate_kernel<uint32_t><<<(unsigned)d.n_walkers, 128, 0, st>>>(
            d, reinterpret_cast<const uint32_t *>(start_words), r0, id_base, format_idx, start_nnz);
    else
        replicate_kernel<uint64_t><<<(unsigned)d.n_walkers, 128, 0, st>>>(
            d, reinterpret_cast<const uint64_t *>(start_words), r0, id_base, format_idx, start_nnz);
}

namespace {

constexpr int64_t kWarpWords = 3072, kSlabWords = 40960;   // accumulators of a warp's tensor / a block's slab
template <class Wd, bool BLOCK, int FB, bool WIDE>
void verify_variant(const SegDesc &d, int64_t first, int64_t count, int slab_rows, int slab_words, int sms,
                    unsigned long long *fail, cudaStream_t st) {
    const int teams = BLOCK ? 1 : kVerifyWarpBlock / 32;
    const int threads = BLOCK ? kVerifyTeam : kVerifyWarpBlock;
    const size_t smem = (size_t)teams * slab_words * 4;
    auto kernel = verify_best_kernel<Wd, BLOCK, FB, WIDE>;
    // the most of any launch: another thread may be about to launch the same kernel with more
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSlabWords * 4);
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    const int64_t blocks = std::min<int64_t>((count + teams - 1) / teams, (int64_t)sms * std::max(per_sm, 1));
    kernel<<<(unsigned)blocks, threads, smem, st>>>(d, first, count, slab_rows, slab_words, fail);
}

template <class Wd, int FB>
void verify_teams(const SegDesc &d, int64_t first, int64_t count, unsigned long long *fail, cudaStream_t st) {
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    constexpr int PER = 32 / FB;
    const int lu = d.m * d.n, lvw = (d.n * d.p) * (d.p * d.m);
    const int64_t words = ((int64_t)lu * lvw + PER - 1) / PER;
    const bool wide = FB == 8 && d.R + 1 > 127;
    // A warp per walker while the whole tensor fits in kWarpWords (four warps' accumulators
    // then leave room for several blocks on an SM); a block per walker beyond, in one
    // slab up to kSlabWords, else in even ones.  A slab of one u-index has at most 128 x
    // 128 entries.
    // Few walkers (a collected best scheme): a block each, whose warps share the terms.
    if (words <= kWarpWords && !wide && count > 2 * sms) {
        verify_variant<Wd, false, FB, false>(d, first, count, lu, (int)words, sms, fail, st);
        return;
    }
    const int64_t fit = std::max<int64_t>(1, kSlabWords * PER / lvw);
    const int slabs = (int)((lu + fit - 1) / fit), rows = (lu + slabs - 1) / slabs;
    const int64_t slab = std::max(((int64_t)rows * lvw + PER - 1) / PER, wide ? (int64_t)(lvw + 1) / 2 : (int64_t)1);
    if (FB == 8 && wide) verify_variant<Wd, true, FB, FB == 8>(d, first, count, rows, (int)slab, sms, fail, st);
    else verify_variant<Wd, true, FB, false>(d, first, count, rows, (int)slab, sms, fail, st);
}

}  // namespace

void launch_verify_best(const SegDesc &d, int64_t first, int64_t count, int mode, int64_t *d_failures,
                        cudaStream_t st) {
    count = std::min(count, d.n_walkers - first);
    if (count <= 0) return;
    auto *fail = reinterpret_cast<unsigned long long *>(d_failures);
    if (d.word_bits == 32) {
        if (mode != TFG_MODE_ZT) verify_teams<uint32_t, 1>(d, first, count, fail, st);
        else verify_teams<uint32_t, 8>(d, first, count, fail, st);
    } else {
        if (mode != TFG_MODE_ZT) verify_teams<uint64_t, 1>(d, first, count, fail, st);
        else verify_teams<uint64_t, 8>(d, first, count, fail, st);
    }
}

void launch_reseed(const SegDesc &d, int64_t first, int64_t count, int32_t r, uint32_t nnz, cudaStream_t st) {
    if (count <= 0) return;
    if (d.word_bits == 32) reseed_kernel<uint32_t><<<(unsigned)count, 128, 0, st>>>(d, first, r, nnz);
    else reseed_kernel<uint64_t><<<(unsigned)count, 128, 0, st>>>(d, first, r, nnz);
}

void launch_argmin_best(const SegDesc &d, unsigned long long *d_key, cudaStream_t st) {
    const int64_t blocks = (d.n_walkers + 255) / 256;
    if (blocks > 0) argmin_kernel<<<(unsigned)blocks, 256, 0, st>>>(d, d_key);
}

void launch_stats(const SegDesc &d, int64_t *d_sums, int *d_minmax, int64_t *d_hist, int hist_len,
                  cudaStream_t st) {
    // at most 256 blocks, so that a block's additions to the totals are shared by many walkers
    const int64_t blocks = std::min<int64_t>((d.n_walkers + 255) / 256, 256);
    if (blocks > 0)
        stats_kernel<<<(unsigned)blocks, 256, (size_t)hist_len * sizeof(int), st>>>(
            d, reinterpret_cast<unsigned long long *>(d_sums), d_minmax, reinterpret_cast<unsigned long long *>(d_hist),
            hist_len);
}

void launch_philox(const uint32_t *d_ctr, int n, uint32_t k0, uint32_t k1, uint32_t *d_out, cudaStream_t st) {
    if (n > 0) philox_kernel<<<(n + 127) / 128, 128, 0, st>>>(d_ctr, n, k0, k1, d_out);
}

}  // namespace tfg
