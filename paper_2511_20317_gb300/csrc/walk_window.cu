// Window-mode walk step (learned flip proposal, Z_T): instead of the
// candidates of one sampled term, each step considers a window of up to
// kWin candidates: starting at term i0 = mulhi(x0, r), terms i0, i0+1, ...
// (mod r) append their try_flip candidates in (factor, slot, rho) order until
// the window is full.  Per step:
//   1. window_kernel  (one warp per walker): the window as candidate
//      descriptors (8 bytes per row; features only when asked for);
//   2. learned policy: window_score_kernel, the tensor-core MLP (mlp_pipe.cuh)
//      whose producer computes each row's 32 features from the descriptor and
//      the walker's slots straight into the shared-memory A tile, so no
//      feature row goes through device memory; it writes one score per row;
//   3. window_apply_kernel (one thread per walker, working on its slots in
//      place in device memory): policy choice (uniform over the window via
//      x1, or epsilon-greedy argmax of the scores with epsilon decided by
//      x3), then the flip, reductions and bookkeeping of
//      the uniform walker; optional logging of the chosen candidate's features
//      (computed from the state before the flip) with the label "the step
//      lowered the rank" for training.
#include <cstdint>
#include <type_traits>
#include <cuda_bf16.h>

#include "mlp_pipe.cuh"
#include "walk_link.cuh"
#include "walk_solo.cuh"

namespace tfg {
namespace dev {

constexpr int kWin = 256;         // window capacity: up to 256 candidate pairs per step (two tensor-core tiles of rows)
constexpr int kFeat = 32;

// candidate descriptor: i (10 bits) | X (2) | j (10) | sign (1) | rho (1)
__device__ __forceinline__ uint32_t pack_cand(int i, int X, int j, int sneg, int rho) {
    return (uint32_t)i | ((uint32_t)X << 10) | ((uint32_t)j << 12) | ((uint32_t)sneg << 22) | ((uint32_t)rho << 23);
}

template <class Wd>
__device__ __forceinline__ int popc_w(Wd v) {
    if constexpr (sizeof(Wd) == 4) return __popc(v);
    else return __popcll(v);
}

// Byte counts of one factor (mask M) of terms a and b: non-zeros of a, of b, in both, in both with
// the same sign (each at most 64).
template <class Wd>
__device__ __forceinline__ uint32_t factor_counts(const PTerm<Wd, 1, true> &a, const PTerm<Wd, 1, true> &b, Wd M) {
    const Wd ad = (a.p[0] | a.n[0]) & M, bd = (b.p[0] | b.n[0]) & M;
    const Wd same = ((a.p[0] & b.p[0]) | (a.n[0] & b.n[0])) & M;
    return (uint32_t)popc_w<Wd>(ad) | (uint32_t)popc_w<Wd>(bd) << 8 | (uint32_t)popc_w<Wd>(ad & bd) << 16 |
           (uint32_t)popc_w<Wd>(same) << 24;
}

// Two integers below 128 as a packed bf16x2 word, from the bytes of v that sel names (4: zero): as
// 128 + k, whose BF16 bits are 0x4300 + k, less 128.
__device__ __forceinline__ uint32_t bytes_bf16x2(uint32_t v, uint32_t sel) {
    const uint32_t biased = __byte_perm(v, 0x00004300u, 0x5050u | (sel & 0xfu) | (sel & 0xf0u) << 4);
    const uint32_t base = 0x43004300u;
    __nv_bfloat162 x, c;
    memcpy(&x, &biased, 4);
    memcpy(&c, &base, 4);
    const __nv_bfloat162 y = __hsub2(x, c);
    uint32_t r;
    memcpy(&r, &y, 4);
    return r;
}

// Features of candidate dc (X, j, sign, rho) of term a = slot i (b = slot j) as 16 packed
// bf16x2 words (small integers: exact):
//   0-2 one-hot X, 3 rho, 4 sign, then with Y, Z the other two factors in rho's order
//   5 |X_i|, 6 |Y_i|, 7 |Y_j|, 8 |Y_i + Y_j|, 9 the sum stays in {-1, 0, 1}, 10 |Z_i|, 11 |Z_j|,
//   12 |Z_j - s Z_i|, 13 the difference stays in it, 14 |Y_i and Y_j|, 15 |Z_i and Z_j|,
//   16 valid and zero sum, 17 valid and zero difference (8, 12: zero where not valid),
//   18 k_i, 19 r - best r, 20 r, 21-23 m, n, p, 24 q, 31 one, the rest zero.
// A valid sum or difference has no position with equal (opposite) signs, so its
// non-zeros are |Y_i| + |Y_j| - 2 |both|: a byte dot product.  All three factors are
// counted before rho and X choose among them (four bytes a factor: the choice moves
// one word, not masks), and integers become BF16 two at a time without the
// conversion unit.  These rows share the scoring kernel's issue slots
// with its epilogues: with the masks chosen first and each feature a float, 2.63 ms a step for
// 262144 walkers of (3,4,5) with full windows, now 2.51 (with 16-byte loads of the slots).
template <class Wd>
__device__ __forceinline__ void cand_features_bf16(const PTerm<Wd, 1, true> &a, const PTerm<Wd, 1, true> &b,
                                                   const Masks<Wd, 1> &mk, uint32_t dc, uint32_t info, int r,
                                                   int best_r, int m, int n, int p, uint32_t (&h)[kFeat / 2]) {
    const uint32_t X = (dc >> 10) & 3u;
    const bool sneg = (dc >> 22) & 1u, rho = (dc >> 23) & 1u;
    const uint32_t cu = factor_counts<Wd>(a, b, mk.m[0][0]), cv = factor_counts<Wd>(a, b, mk.m[1][0]),
                   cw = factor_counts<Wd>(a, b, mk.m[2][0]);
    const uint32_t cx = X == 0 ? cu : (X == 1 ? cv : cw);
    const uint32_t c1 = X == 0 ? cv : (X == 1 ? cw : cu), c2 = X == 0 ? cw : (X == 1 ? cu : cv);
    const uint32_t cy = rho ? c2 : c1, cz = rho ? c1 : c2;
    const bool vy = cy < (1u << 24);                                               // no equal signs
    const bool vz = sneg ? cz < (1u << 24) : (cz >> 24) == ((cz >> 16) & 255u);    // no equal, or only equal ones
    const uint32_t ny = (uint32_t)__dp4a((int)cy, 0x00FE0101, 0), nz = (uint32_t)__dp4a((int)cz, 0x00FE0101, 0);
    const uint32_t one_lo = 0x00003F80u, one_hi = 0x3F800000u;
    h[0] = X == 0 ? one_lo : (X == 1 ? one_hi : 0u);
    h[1] = (X == 2 ? one_lo : 0u) | (rho ? one_hi : 0u);
    h[2] = (sneg ? one_lo : 0u) | bytes_bf16x2(cx, 0x04);
    h[3] = bytes_bf16x2(cy, 0x10);
    h[4] = vy ? bytes_bf16x2(ny | 0x100u, 0x10) : 0u;
    h[5] = bytes_bf16x2(cz, 0x10);
    h[6] = vz ? bytes_bf16x2(nz | 0x100u, 0x10) : 0u;
    h[7] = bytes_bf16x2(__byte_perm(cy, cz, 0x6262), 0x10);
    h[8] = (vy && ny == 0 ? one_lo : 0u) | (vz && nz == 0 ? one_hi : 0u);
    h[9] = mlp::pack_bf16x2((float)min((int)(info & 255u), 64), (float)(r - best_r));
    h[10] = mlp::pack_bf16x2((float)r, (float)m);
    h[11] = mlp::pack_bf16x2((float)n, (float)p);
    h[12] = bytes_bf16x2(min(info >> 8, 64u), 0x40);
    h[13] = h[14] = 0u;
    h[15] = one_hi;
}

// One warp per walker; lane l holds slots l, l + 32, ... (NCH of them, r <= 32 NCH).
// Matches of all terms at once: the slots' 16-bit factor hashes are transposed by
// ballots into words over the slots, and a lane compares each of its slots' hash
// with all slots by one word operation per bit, chunk and factor.  The hash classes
// are the factor classes when every slot equals the lowest slot of its hash class
// on the full words (one comparison per slot and factor); a walker with a collision
// (about 3% at 64 slots) drops the false members one by one.  Then the counts' prefix
// sums in slot order, rotated to start at term i0, give every term's first window
// row, the lanes write their terms' rows to shared memory (the two rows of a match
// in one 16-byte store), and the warp copies the rows out.  With `feat` it also
// writes their feature rows (coalesced 64-byte rows; rows past the window are zero).
// Bound by integer issue.  The kernel it replaces compared eight terms a round with all
// slots, a quarter of the slots per lane, until the window was full, which in a
// long walk takes every term (about 3.5 candidates each): (3,4,5) 262144 walkers
// 1.77 ms, (4,4,4) 2.04 ms; now 0.56 and 0.6 ms.
constexpr int kWinHash = 16;
template <class Wd>
struct alignas(2 * sizeof(Wd)) WinSlot {
    Wd p, n;
};
template <class Wd, int NCH>
__device__ __forceinline__ void window_of(const SegDesc &d, int64_t w, int lane, WinSlot<Wd> *st, uint2 *srow,
                                          __nv_bfloat16 *feat, uint2 *desc, int *kwin) {
    using T = PTerm<Wd, 1, true>;
    using LW = LinkWalker<TFG_MODE_ZT, Wd, NCH, false, false>;   // hash and comparison of factors
    using Slot = WinSlot<Wd>;
    constexpr unsigned full = 0xffffffffu;
    Masks<Wd, 1> mk;
    mk.load(d);
    const tfg_walker_info &H = d.hdr[w];
    const int r = H.r, best_r = H.best_r;
    const U4 x = philox10((uint32_t)H.t, (uint32_t)(H.t >> 32), H.walker_id, 0u, d.key0, d.key1);
    const int i0 = (int)__umulhi(x.x, (uint32_t)r);
    const Slot *src = reinterpret_cast<const Slot *>(d.slots) + (size_t)w * d.R;
    T own[NCH];
    uint32_t live[NCH];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int k = 32 * c + lane;
        Slot v{Wd(0), Wd(0)};
        if (k < r) v = src[k];
        own[c].p[0] = v.p;
        own[c].n[0] = v.n;
        st[k] = v;
        const int lo = r - 32 * c;
        live[c] = lo >= 32 ? full : (lo > 0 ? (1u << lo) - 1u : 0u);
    }
    __syncwarp();
    // ---- m[f][c][e]: members of chunk e in the class of factor f of slot 32 c + lane (without it)
    uint32_t m[3][NCH][NCH];
    bool exact = true;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        uint32_t h[NCH];
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            h[c] = LW::factor_hash16(own[c], mk.m[f][0]);
#pragma unroll
            for (int e = 0; e < NCH; ++e) m[f][c][e] = 0u;
        }
        // one top bit of every byte a round (rolled: the code is read once per walker)
#pragma unroll 1
        for (int round = 0; round < kWinHash / 4; ++round) {
            auto bit = [&](auto byte) {
                constexpr int B = decltype(byte)::value;
                uint32_t word[NCH];
#pragma unroll
                for (int e = 0; e < NCH; ++e) word[e] = __ballot_sync(full, (h[e] >> (8 * B + 7)) & 1u);
#pragma unroll
                for (int c = 0; c < NCH; ++c) {
                    const uint32_t sp = sign_spread<B>(h[c]);
#pragma unroll
                    for (int e = 0; e < NCH; ++e) m[f][c][e] |= word[e] ^ sp;
                }
            };
            bit(std::integral_constant<int, 0>{});
            bit(std::integral_constant<int, 1>{});
            bit(std::integral_constant<int, 2>{});
            bit(std::integral_constant<int, 3>{});
#pragma unroll
            for (int c = 0; c < NCH; ++c) h[c] <<= 1;
        }
#pragma unroll
        for (int c = 0; c < NCH; ++c) {
            int first = 0;   // lowest live slot of the hash class
#pragma unroll
            for (int e = NCH - 1; e >= 0; --e) {
                m[f][c][e] = ~m[f][c][e] & live[e];
                first = m[f][c][e] ? 32 * e + __ffs(m[f][c][e]) - 1 : first;
            }
            const Slot v = st[first];
            T t;
            t.p[0] = v.p;
            t.n[0] = v.n;
            exact = exact && (LW::same(t, own[c], mk.m[f][0]) || 32 * c + lane >= r);
            m[f][c][c] &= ~(1u << lane);
        }
    }
    if (!__all_sync(full, exact)) {
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int c = 0; c < NCH; ++c)
#pragma unroll
                for (int e = 0; e < NCH; ++e) {
                    uint32_t left = m[f][c][e];
#pragma unroll 1
                    while (left) {
                        const uint32_t low = left & (0u - left);
                        left ^= low;
                        const Slot v = st[32 * e + __ffs(low) - 1];
                        T t;
                        t.p[0] = v.p;
                        t.n[0] = v.n;
                        if (!LW::same(t, own[c], mk.m[f][0])) m[f][c][e] ^= low;
                    }
                }
    }
    // ---- window offsets: candidates (two per match) of the terms before, from i0 on
    int ki[NCH], pre[NCH], total = 0;
    uint32_t wneg[NCH];   // slots whose w starts with -1
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        int n = 0;
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int e = 0; e < NCH; ++e) n += __popc(m[f][c][e]);
        ki[c] = 32 * c + lane < r ? 2 * n : 0;
        int incl = ki[c];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(full, incl, o);
            if (lane >= o) incl += y;
        }
        pre[c] = total + incl - ki[c];
        total += __shfl_sync(full, incl, 31);
        const Wd dw = (own[c].p[0] | own[c].n[0]) & mk.m[2][0];
        wneg[c] = __ballot_sync(full, (own[c].n[0] & dw & (Wd(0) - dw)) != Wd(0));
    }
    int start = 0;   // candidates of the slots before i0
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int y = __shfl_sync(full, pre[c], i0 & 31);
        start = (i0 >> 5) == c ? y : start;
    }
    const int K = total < kWin ? total : kWin;
    // ---- rows: term, then factor, then slot, then rho
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const int i = 32 * c + lane;
        int pos = pre[c] - start + (i < i0 ? total : 0);
        const int q = i >= i0 ? i - i0 : i - i0 + r;
        const uint32_t info = (uint32_t)(ki[c] < 64 ? ki[c] : 64) | ((uint32_t)(q < 64 ? q : 64) << 8);
        const uint32_t mine = (wneg[c] >> lane) & 1u;
        if (i >= r) pos = kWin;
#pragma unroll
        for (int f = 0; f < 3; ++f)
#pragma unroll
            for (int e = 0; e < NCH; ++e) {
                uint32_t left = m[f][c][e];
#pragma unroll 1
                while (left && pos < kWin) {   // pos is even, and so is kWin
                    const int o = __ffs(left) - 1;
                    left &= left - 1u;
                    const uint32_t sneg = f == 2 ? ((wneg[e] >> o) & 1u) ^ mine : 0u;
                    const uint32_t dc = pack_cand(i, f, 32 * e + o, (int)sneg, 0);
                    reinterpret_cast<uint4 *>(srow)[pos >> 1] = make_uint4(dc, info, dc | (1u << 23), info);
                    pos += 2;
                }
            }
    }
    __syncwarp();
    uint2 *dw = desc + (size_t)w * kWin;
    if (((uintptr_t)desc & 15u) == 0) {   // the scratch is; a dump's array may start at any 8 bytes
        const uint4 *sw = reinterpret_cast<const uint4 *>(srow);
        for (int row = lane; row < K / 2; row += 32) reinterpret_cast<uint4 *>(dw)[row] = sw[row];
    } else {
        for (int row = lane; row < K; row += 32) dw[row] = srow[row];
    }
    if (feat) {
        __nv_bfloat16 *fw = feat + (size_t)w * kWin * kFeat;
        for (int row = lane; row < kWin; row += 32) {
            uint4 *dst = reinterpret_cast<uint4 *>(fw + (size_t)row * kFeat);
            if (row < K) {
                const uint32_t dc = srow[row].x, in = srow[row].y;
                const Slot vi = st[dc & 1023u], vj = st[(dc >> 12) & 1023u];
                T ti, tj;
                ti.p[0] = vi.p;
                ti.n[0] = vi.n;
                tj.p[0] = vj.p;
                tj.n[0] = vj.n;
                uint32_t h[kFeat / 2];
                cand_features_bf16<Wd>(ti, tj, mk, dc, in, r, best_r, d.m, d.n, d.p, h);
#pragma unroll
                for (int k = 0; k < kFeat / 8; ++k) dst[k] = make_uint4(h[4 * k], h[4 * k + 1], h[4 * k + 2], h[4 * k + 3]);
            } else {
#pragma unroll
                for (int k = 0; k < kFeat / 8; ++k) dst[k] = make_uint4(0, 0, 0, 0);
            }
        }
    }
    if (lane == 0) kwin[w] = K;
}

// NCH: chunks of the slot capacity; a walker runs at the chunks of its rank.
template <class Wd, int NCH>
__global__ void __launch_bounds__(128) window_kernel(const SegDesc d, __nv_bfloat16 *__restrict__ feat,
                                                     uint2 *__restrict__ desc, int *__restrict__ kwin) {
    __shared__ WinSlot<Wd> st[4][32 * NCH];
    __shared__ __align__(16) uint2 srow[4][kWin];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t w = (int64_t)blockIdx.x * 4 + warp;
    if (w >= d.n_walkers) return;
    const int r = d.hdr[w].r;
    if (NCH > 2 && r > 64) window_of<Wd, NCH>(d, w, lane, st[warp], srow[warp], feat, desc, kwin);
    else if (NCH > 1 && r > 32) window_of<Wd, NCH < 2 ? 1 : 2>(d, w, lane, st[warp], srow[warp], feat, desc, kwin);
    else window_of<Wd, 1>(d, w, lane, st[warp], srow[warp], feat, desc, kwin);
}

// Producer of the fused scoring kernel.  A warpgroup takes a contiguous share of the half
// windows (unit 2 w + half: rows 0-127 or 128-255 of walker w) and lays their rows end to
// end in groups of 32, the last group of a window ragged: warp j of its tile k takes
// group 4 k + j.  (A tile for every half window left the rows past it empty: 3000 walkers
// of (4,4,5), two learned steps, 246 us with it and 215 so.)
// A lane holds the window size of one unit of 32 and the running count of their
// groups; the next 32 sizes are loaded a chunk ahead.  A thread computes the features of
// its row from the row's descriptor and the walker's two slots, straight into the A
// tile; rows past the window get zero features and no score.  Loads in two
// phases, so that none waits on another while the previous tile runs: begin() the row's
// descriptor and the walker's rank (every row's descriptor word is read; a row past
// the window holds a stale or undefined one, so its slot indices are clamped), mid()
// the two slots the descriptor names.
template <class Wd>
struct WindowProducer {
    static constexpr bool kFold = true;   // the producer writes features 29, 30 = 1: biases in the MMAs
    const Wd *slots;
    const tfg_walker_info *hdr;
    int R, m, n, p;
    const uint2 *desc;
    const int *kwin;
    float *score;
    Masks<Wd, 1> mk;
    // the warpgroup's units: those of this chunk of 32 start at base, the next one's at next
    int64_t base, next, end;
    int size, size_next, upto, total;   // this lane's unit: window size, groups up to and with it; all groups
    int first;                          // the next tile's first group, counted from the chunk's
    // loaded by begin() / mid()
    int64_t w;
    int row, K, r, best_r;
    uint2 dci;
    PTerm<Wd, 1, true> ti, tj;
    __device__ __forceinline__ int groups(int64_t u, int k) const {   // of unit u, window size k
        const int left = k - (int)(u & 1) * (kWin / 2);
        return left <= 0 ? 0 : min((left + 31) / 32, kWin / 64);
    }
    __device__ __forceinline__ int size_at(int64_t u) const { return u < end ? kwin[u >> 1] : 0; }
    __device__ __forceinline__ void share(int64_t units, int64_t part, int64_t parts) {
        base = next = units * part / parts;
        end = units * (part + 1) / parts;
        size_next = size_at(next + (threadIdx.x & 31));
        total = first = 0;
    }
    // the next chunk of units
    __device__ __forceinline__ void advance(int lane) {
        first -= total;
        base = next;
        next += 32;
        size = size_next;
        size_next = size_at(next + lane);
        upto = groups(base + lane, size);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int below = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += below;
        }
        total = __shfl_sync(0xffffffffu, upto, 31);
    }
    __device__ __forceinline__ bool begin(int q) {
        const int lane = q & 31;
        while (first >= total && next < end) advance(lane);
        if (first >= total) return false;
        while (first + (q >> 5) >= total && next < end) advance(lane);   // this warp's group
        const int mine = first + (q >> 5);
        first += 4;
        // the unit that holds it (none: past the last one)
        const int src = min(__popc(__ballot_sync(0xffffffffu, upto <= mine)), 31);
        const int64_t u = base + src;
        K = mine < total ? __shfl_sync(0xffffffffu, size, src) : 0;
        row = (int)(u & 1) * (kWin / 2) + 32 * (mine - __shfl_sync(0xffffffffu, upto, src) + groups(u, K)) + lane;
        if (mine >= total) {
            row = 0;
            w = base >> 1;
        } else {
            w = u >> 1;
        }
        dci = desc[(size_t)w * kWin + row];
        r = hdr[w].r;
        best_r = hdr[w].best_r;
        return true;
    }
    __device__ __forceinline__ void mid(int) {
        const int i = min((int)(dci.x & 1023u), R - 1), j = min((int)((dci.x >> 12) & 1023u), R - 1);
        const WinSlot<Wd> *src = reinterpret_cast<const WinSlot<Wd> *>(slots) + (size_t)w * R;
        const WinSlot<Wd> vi = src[i], vj = src[j];
        ti.p[0] = vi.p;
        ti.n[0] = vi.n;
        tj.p[0] = vj.p;
        tj.n[0] = vj.n;
    }
    __device__ __forceinline__ int64_t fill(uint8_t *sX, int q) {
        uint32_t h[kFeat / 2];
        if (row < K) {
            cand_features_bf16<Wd>(ti, tj, mk, dci.x, dci.y, r, best_r, m, n, p, h);
            h[14] |= 0x3F800000u;   // feature 29 = 1 (bf16), the bias inputs of the folded MMA
            h[15] |= 0x00003F80u;   // feature 30 = 1 (feature 31 is 1 already)
        } else {
#pragma unroll
            for (int k = 0; k < kFeat / 2; ++k) h[k] = 0u;
        }
#pragma unroll
        for (int c = 0; c < kFeat / 8; ++c)
            mlp::st_row8(sX, q, 8 * c, mlp::kIn, make_uint4(h[4 * c], h[4 * c + 1], h[4 * c + 2], h[4 * c + 3]));
        return row < K ? w * kWin + row : -1;
    }
    __device__ __forceinline__ void emit(float y, int64_t o) {
        if (o >= 0) score[o] = y;
    }
};

constexpr int kScoreWG = 4;

template <class Wd>
__global__ void __launch_bounds__(kScoreWG * 128, 1)
    window_score_kernel(const SegDesc d, const uint8_t *__restrict__ params, const uint2 *__restrict__ desc,
                        const int *__restrict__ kwin, float *__restrict__ score, int *__restrict__ err,
                        uint32_t first_limit) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t mbar[kScoreWG];
    __shared__ uint32_t tslot;
    __shared__ int tflag;
    WindowProducer<Wd> pr;
    pr.slots = reinterpret_cast<const Wd *>(d.slots);
    pr.hdr = d.hdr;
    pr.R = d.R;
    pr.m = d.m;
    pr.n = d.n;
    pr.p = d.p;
    pr.desc = desc;
    pr.kwin = kwin;
    pr.score = score;
    pr.mk.load(d);
    pr.share(d.n_walkers * 2, (int64_t)blockIdx.x * kScoreWG + (threadIdx.x >> 7), (int64_t)gridDim.x * kScoreWG);
    mlp::run_tiles<kScoreWG>(params, pr, err, first_limit, smem, mbar, &tslot, &tflag);
}

// Log entry `slot` := (features, label, walker id, step).
__device__ __forceinline__ void write_log_entry(const WindowLog &log, unsigned long long slot,
                                                const uint32_t (&f)[kFeat / 2], float label, uint32_t wid,
                                                uint32_t step) {
    WindowLogEntry *e = reinterpret_cast<WindowLogEntry *>(log.d_entries) + slot;
#pragma unroll
    for (int k = 0; k < kFeat / 8; ++k)
        reinterpret_cast<uint4 *>(e->feat)[k] = make_uint4(f[4 * k], f[4 * k + 1], f[4 * k + 2], f[4 * k + 3]);
    e->label = label;
    e->walker_id = wid;
    e->step = step;
    e->pad = 0;
}

// Logs a step's chosen candidate: features lf (of the state before the flip), positive:
// the step's reductions lowered the rank.
__device__ __forceinline__ void log_step(const WindowLog &log, int64_t w, const uint32_t (&lf)[kFeat / 2], bool positive,
                                         int64_t t_step, uint32_t wid, uint32_t key0, uint32_t key1) {
    const int H = log.horizon > 1 ? log.horizon : 1;
    bool keep0 = false;
    if (!positive && log.neg_thresh) {
        const U4 y = philox10((uint32_t)t_step, (uint32_t)(t_step >> 32), wid, 0x100u, key0, key1);
        keep0 = y.x < log.neg_thresh;
    }
    if (H > 1) {
        // this step's features into ring slot t mod H; a rank-lowering step appends the
        // entries of steps t-H+1 .. t still in the ring (step order) and empties it
        uint4 *ring = reinterpret_cast<uint4 *>(log.d_ring) + (size_t)w * H * (kFeat / 8);
        uint32_t *rs = log.d_ring_step + (size_t)w * H;
        const int kt = (int)(t_step % H);
#pragma unroll
        for (int k = 0; k < kFeat / 8; ++k)
            ring[kt * (kFeat / 8) + k] = make_uint4(lf[4 * k], lf[4 * k + 1], lf[4 * k + 2], lf[4 * k + 3]);
        rs[kt] = (uint32_t)t_step;
        if (positive) {
            int n = 0;
            for (int dd = 0; dd < H && dd <= t_step; ++dd)
                n += rs[(int)((t_step - dd) % H)] == (uint32_t)(t_step - dd);
            unsigned long long slot = atomicAdd(reinterpret_cast<unsigned long long *>(log.d_count),
                                                (unsigned long long)n);
            for (int dd = H - 1; dd >= 0; --dd) {
                if (dd > t_step) continue;
                const int k = (int)((t_step - dd) % H);
                if (rs[k] != (uint32_t)(t_step - dd)) continue;
                if (slot < (unsigned long long)log.capacity) {
                    uint32_t e16[kFeat / 2];
#pragma unroll
                    for (int q = 0; q < kFeat / 8; ++q) {
                        const uint4 v = ring[k * (kFeat / 8) + q];
                        e16[4 * q] = v.x; e16[4 * q + 1] = v.y; e16[4 * q + 2] = v.z; e16[4 * q + 3] = v.w;
                    }
                    write_log_entry(log, slot, e16, 1.f, wid, (uint32_t)(t_step - dd));
                }
                ++slot;
            }
            for (int k = 0; k < H; ++k) rs[k] = 0xFFFFFFFFu;
        }
    }
    const bool keep = (H == 1 && positive) || keep0;
    if (keep) {
        const unsigned long long slot = atomicAdd(reinterpret_cast<unsigned long long *>(log.d_count), 1ull);
        if (slot < (unsigned long long)log.capacity) write_log_entry(log, slot, lf, positive ? 1.f : 0.f, wid,
                                                                     (uint32_t)t_step);
    }
}

// Steps of uniform window walks, many per launch, one walker per thread, on the walker with
// kept factor classes (walk_link.cuh).  Uniform choice needs of the window only its
// size and the chosen row: with every slot's number of matches n_k kept
// beside the classes, K = min(256, 2 sum n_k), and row c belongs to the first term
// after i0 whose running sum of 2 n_k exceeds c.
// Bound by the latency of a step, most of it the walk over the counts (two slots a
// word, 15 to 33 words a step on (4,4,4)).  Measured on (4,4,4), 262144 walkers: 2.17 ms a
// step with a window kernel that lists all 256 rows and an apply kernel per step,
// now 0.1 ms (20 steps, the last one by those kernels: 43.6, now 2.55 ms);
// 4096 logged walkers (the training data), 500 steps: 28.4 ms, now 2.6 with 32 walkers a
// warp (the whole collection 5.2 ms; 4.6 with 4 walkers a warp).
template <class Wd, int NW, bool GM>
__global__ void __launch_bounds__(64, 7) window_walk_kernel(const SegDesc d, int32_t steps, int32_t *__restrict__ choices,
                                                            int64_t choice_stride, WindowLog log) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned wmask = walker_lanes(d, w);
    if (w >= d.n_walkers) return;   // no block-wide barrier is used
    using LW = LinkWalker<TFG_MODE_ZT, Wd, NW, GM, false, true>;
    using T = typename LW::T;
    LW wk;
    link_rows<LW, Wd>(wk, d, w, GM, smem_raw);
    wk.load(d, w);
    Wd *bestp = reinterpret_cast<Wd *>(d.best) + (size_t)w * d.R * 2;
    __syncwarp(wmask);
    const int lane = threadIdx.x & 31;
    const int nl = __popc(wmask);
    U4 x = philox10((uint32_t)wk.t, (uint32_t)(wk.t >> 32), wk.wid, 0u, wk.key0, wk.key1);
#pragma unroll 1
    for (int32_t step = 0; step < steps; ++step) {
        const int64_t t_step = wk.t, tn = wk.t + 1;
        const U4 xn = philox10((uint32_t)tn, (uint32_t)(tn >> 32), wk.wid, 0u, wk.key0, wk.key1);
        const int r = wk.r, i0 = (int)__umulhi(x.x, (uint32_t)r);
        typename LW::Step did{kNoCand, i0, 0, 0, 0, 0};
        const int K = min(2 * wk.matches, kWin);
        int c = -1;
        uint32_t lf[kFeat / 2];   // logged features of the chosen candidate (state before the flip)
        if (K > 0) {
            c = (int)__umulhi(x.y, (uint32_t)K);
            // the term of row c: skip c / 2 matches from i0 on (around the last slot)
            const int nw = (r + 1) >> 1;
            int left = c >> 1, wi = i0 >> 1;
            uint32_t v = wk.cn[wi * kLane] & ((i0 & 1) ? 0xffff0000u : ~0u);
#pragma unroll 1
            for (int n = 0; n < nw; ++n) {
                const int sum = (int)(v & 0xffffu) + (int)(v >> 16);
                if (left < sum) break;
                left -= sum;
                wi = wi + 1 == nw ? 0 : wi + 1;
                v = wk.cn[wi * kLane];
            }
            const int lo = (int)(v & 0xffffu), odd = (int)(left >= lo);
            left -= odd ? lo : 0;
            const int n_i = odd ? (int)(v >> 16) : lo;
            typename LW::Sample s;
            s.i = 2 * wi + odd;
            s.ti = wk.ld(s.i);
            s.l[0] = wk.ix[s.i * kLane];
            did.i = s.i;
            did.rho = c & 1;
            typename LW::Cand cd;
            wk.candidates(s, cd);
            const int n01 = cd.n0 + cd.n1;
            did.X = (int)(left >= cd.n0) + (int)(left >= n01);
            did.j = wk.member(s, did.X, left - (did.X == 0 ? 0 : (did.X == 1 ? cd.n0 : n01)), cd);
            const T tj = wk.ld(did.j);
            if (log.d_entries) {
                const int sneg = did.X == 2 ? (int)(((s.ti.p[0] ^ tj.p[0]) & wk.mk.m[2][0]) != Wd(0)) : 0;
                const int q = s.i >= i0 ? s.i - i0 : s.i - i0 + r;
                const uint32_t info = (uint32_t)min(2 * n_i, 64) | ((uint32_t)min(q, 64) << 8);
                cand_features_bf16<Wd>(s.ti, tj, wk.mk, pack_cand(s.i, did.X, did.j, sneg, did.rho), info, r, wk.best_r, d.m,
                                       d.n, d.p, lf);
            }
            wk.flip(s.ti, tj, 0, did);
        }
        wk.c_acc += did.action == kAccept;
        wk.c_rej += did.action == kReject;
        wk.cascade_all(wmask);
        const bool lowered = wk.r < r;
        wk.c_red += lowered;
        if (choices) choices[(int64_t)step * choice_stride + w] = c;
        if (log.d_entries && c >= 0) log_step(log, w, lf, lowered, t_step, wk.wid, wk.key0, wk.key1);
        wk.finish(d, wmask, lane, nl, bestp, 0, x.z, x.w, did);
        x = xn;
        wk.t = tn;
    }
    wk.store(d, w, (uint32_t)steps);
}

// Row of highest score (first on ties) of every lane's walker that asks for one: in a full
// warp four walkers at a time, eight lanes each, whose loads (16 bytes a lane) cover
// consecutive rows.  (A thread reading its own walker's 256 scores touches 32 lines a
// load: 0.34 ms for 262144 walkers of (3,4,5) with the rest of the step, now 0.22.)  As a scan
// from row 0 that moves on a greater score does, a NaN is never chosen over another
// row, and one in row 0 stays chosen.
__device__ __forceinline__ int best_row(unsigned wmask, int lane, int nl, bool ask, int K, const float *mine) {
    if (nl < 32 || __reduce_max_sync(wmask, ask ? K : 0) <= 32) {
        // also for short windows, whose rows are a line or less: one round of loads, not eight
        int c = 0;
        if (ask) {
            float best = mine[0];
#pragma unroll 8
            for (int k = 1; k < K; ++k)
                if (mine[k] > best) { best = mine[k]; c = k; }
        }
        return c;
    }
    // order-preserving integers of scores (-0 as +0); 0: no score
    auto key = [](float f) -> uint32_t {
        const uint32_t u = __float_as_uint(f + 0.f);
        return f != f ? 1u : (u & 0x80000000u ? ~u : u | 0x80000000u);
    };
    int c = 0;
    const unsigned pend = __ballot_sync(wmask, ask);
#pragma unroll 1
    for (int r = 0; r < 8; ++r) {
        if (((pend >> (4 * r)) & 15u) == 0u) continue;
        const int a = 4 * r + (lane >> 3);   // the walker of these eight lanes
        const int Ka = __shfl_sync(wmask, ask ? K : 0, a);
        const float4 *row = reinterpret_cast<const float4 *>(
            __shfl_sync(wmask, reinterpret_cast<unsigned long long>(mine), a));
        uint32_t top = 0u;
        int at = 0;
#pragma unroll 4
        for (int k0 = 4 * (lane & 7); k0 < Ka; k0 += 32) {
            const float4 v = row[k0 >> 2];
            const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t u = key(f[q]);
                if (k0 + q == 0 && u == 1u) u = 0xffffffffu;
                u = k0 + q < Ka ? u : 0u;
                at = u > top ? k0 + q : at;
                top = max(u, top);
            }
        }
        __syncwarp(wmask);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            const uint32_t t2 = __shfl_xor_sync(wmask, top, o);
            const int a2 = __shfl_xor_sync(wmask, at, o);
            if (t2 > top || (t2 == top && a2 < at)) {
                top = t2;
                at = a2;
            }
        }
        const int got = __shfl_sync(wmask, at, (lane & 3) * 8);   // lane 4 r + g: group g's row
        if ((lane >> 2) == r) c = got;
    }
    return c;
}

// One window-mode step per thread (walker), on the solo walker's state machine.
template <class Wd, int RMAX, int BT>
__global__ void __launch_bounds__(BT) window_apply_kernel(const SegDesc d, const uint2 *__restrict__ desc,
                                                          const int *__restrict__ kwin,
                                                          const float *__restrict__ score, int policy,
                                                          uint32_t eps_thresh, int32_t *__restrict__ choices,
                                                          WindowLog log) {
    const int64_t w = (int64_t)blockIdx.x * BT + threadIdx.x;
    if (w >= d.n_walkers) return;
    // one step per launch: the walker works on its slots in place in device memory
    // (staging them through shared memory cost more than the step: 255 registers,
    // 3.5 warps per SM)
    using SW = SoloWalker<TFG_MODE_ZT, Wd, RMAX, BT, 0, false, true>;
    using T = typename SW::T;
    SW wk;
    wk.sm = reinterpret_cast<Wd *>(d.slots) + (size_t)w * d.R * 2;
    wk.load(d, w);
    Wd *bestp = reinterpret_cast<Wd *>(d.best) + (size_t)w * d.R * 2;
    const unsigned wmask = __activemask();
    const int lane = threadIdx.x & 31;
    const int nl = __popc(wmask);
    const int64_t t_step = wk.t;
    const U4 x = philox10((uint32_t)wk.t, (uint32_t)(wk.t >> 32), wk.wid, 0u, wk.key0, wk.key1);
    const int r_before = wk.r;
    const int K = kwin[w];
    int action = kNoCand, X = 0, j = 0, rho = 0, sneg = 0, c = -1;
    int i = (int)__umulhi(x.x, (uint32_t)wk.r);
    bool need_check = false;
    uint32_t lf[kFeat / 2];   // logged features of the chosen candidate (state before the flip)
    T ti2, tj2;
    ti2.p[0] = tj2.p[0] = 0;
    ti2.n[0] = tj2.n[0] = 0;
    const bool greedy = K > 0 && policy != 0 && x.w >= eps_thresh;
    const int top = policy != 0 ? best_row(wmask, lane, nl, greedy, K, score + (size_t)w * kWin) : 0;
    if (K > 0) {
        c = greedy ? top : (int)__umulhi(x.y, (uint32_t)K);
        const uint2 dci = desc[(size_t)w * kWin + c];
        const uint32_t dc = dci.x;
        i = (int)(dc & 1023u);
        X = (int)((dc >> 10) & 3u);
        j = (int)((dc >> 12) & 1023u);
        sneg = (int)((dc >> 22) & 1u);
        rho = (int)((dc >> 23) & 1u);
        const T ti = wk.ld(i);
        if (log.d_entries) cand_features_bf16<Wd>(ti, wk.ld(j), wk.mk, dc, dci.y, wk.r, wk.best_r, d.m, d.n, d.p, lf);
        wk.apply_candidate(ti, i, X, j, sneg, rho, action, need_check, ti2, tj2);
    } else {
        wk.c_noc += 1;
    }
    wk.finish_step(d, wmask, lane, nl, bestp, x.z, x.w, r_before, action, X, rho, sneg, i, j, need_check, ti2, tj2);
    if (choices) choices[w] = c;
    if (log.d_entries && c >= 0) log_step(log, w, lf, wk.c_red > 0, t_step, wk.wid, wk.key0, wk.key1);
    wk.store(d, w);
}

}  // namespace dev

int window_cap() { return dev::kWin; }

void launch_window(const SegDesc &d, void *feat, uint2 *desc, int *kwin, cudaStream_t st) {
    const unsigned blocks = (unsigned)((d.n_walkers + 3) / 4);
    if (d.n_walkers <= 0) return;
    auto *fb = reinterpret_cast<__nv_bfloat16 *>(feat);
    if (d.word_bits == 32) dev::window_kernel<uint32_t, 1><<<blocks, 128, 0, st>>>(d, fb, desc, kwin);
    else if (d.R <= 32) dev::window_kernel<uint64_t, 1><<<blocks, 128, 0, st>>>(d, fb, desc, kwin);
    else if (d.R <= 64) dev::window_kernel<uint64_t, 2><<<blocks, 128, 0, st>>>(d, fb, desc, kwin);
    else dev::window_kernel<uint64_t, 3><<<blocks, 128, 0, st>>>(d, fb, desc, kwin);
}

template <class Wd>
static void score_variant(const SegDesc &d, const void *params, const uint2 *desc, const int *kwin, float *score,
                          int *err, cudaStream_t st) {
    constexpr uint32_t smem = mlp::Layout<true>::bytes(dev::kScoreWG);
    static bool attr = [] {
        cudaFuncSetAttribute(dev::window_score_kernel<Wd>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return true;
    }();
    (void)attr;
    const int grid = score_grid(d.n_walkers * 2, dev::kScoreWG);
    dev::window_score_kernel<Wd><<<grid, dev::kScoreWG * 128, smem, st>>>(
        d, reinterpret_cast<const uint8_t *>(params), desc, kwin, score, err, first_wait_limit());
}

void launch_window_score(const SegDesc &d, const void *params, const uint2 *desc, const int *kwin, float *score,
                         int *err, cudaStream_t st) {
    if (d.n_walkers <= 0) return;
    if (d.word_bits == 32) score_variant<uint32_t>(d, params, desc, kwin, score, err, st);
    else score_variant<uint64_t>(d, params, desc, kwin, score, err, st);
}

template <class Wd, int RMAX>
static void apply_variant(const SegDesc &d, const uint2 *desc, const int *kwin, const float *score, int policy,
                          uint32_t eps, int32_t *choices, const WindowLog &log, cudaStream_t st) {
    constexpr int BT = 128;
    const int64_t blocks = (d.n_walkers + BT - 1) / BT;
    dev::window_apply_kernel<Wd, RMAX, BT><<<(unsigned)blocks, BT, 0, st>>>(d, desc, kwin, score, policy, eps,
                                                                           choices, log);
}

// Capacity of the apply kernel chosen for a population (0: not supported).
int window_apply_capacity(int word_bits, int R) {
    if (word_bits == 32) {
        for (int c : {12, 16, 32}) if (R <= c) return c;
    } else {
        for (int c : {48, 64, 72, 88}) if (R <= c) return c;
    }
    return 0;
}

int launch_window_apply(const SegDesc &d, const uint2 *desc, const int *kwin, const float *score, int policy,
                        uint32_t eps, int32_t *choices, const WindowLog &log, cudaStream_t st) {
    if (d.n_walkers <= 0) return 0;
    const int cap = window_apply_capacity(d.word_bits, d.R);
    if (d.word_bits == 32) {
        if (cap == 12) apply_variant<uint32_t, 12>(d, desc, kwin, score, policy, eps, choices, log, st);
        else if (cap == 16) apply_variant<uint32_t, 16>(d, desc, kwin, score, policy, eps, choices, log, st);
        else if (cap == 32) apply_variant<uint32_t, 32>(d, desc, kwin, score, policy, eps, choices, log, st);
        else return -1;
    } else {
        if (cap == 48) apply_variant<uint64_t, 48>(d, desc, kwin, score, policy, eps, choices, log, st);
        else if (cap == 64) apply_variant<uint64_t, 64>(d, desc, kwin, score, policy, eps, choices, log, st);
        else if (cap == 72) apply_variant<uint64_t, 72>(d, desc, kwin, score, policy, eps, choices, log, st);
        else if (cap == 88) apply_variant<uint64_t, 88>(d, desc, kwin, score, policy, eps, choices, log, st);
        else return -1;
    }
    return 0;
}

template <class Wd, int NW>
static void window_walk_variant(const SegDesc &d, int32_t steps, int32_t *choices, int64_t stride, const WindowLog &log,
                                cudaStream_t st) {
    using Shared = dev::LinkWalker<TFG_MODE_ZT, Wd, NW, false, false, true>;
    using Device = dev::LinkWalker<TFG_MODE_ZT, Wd, NW, true, false, true>;
    constexpr int kBlock = 64;
    static bool attr = [] {
        cudaFuncSetAttribute(dev::window_walk_kernel<Wd, NW, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinkSmem);
        if constexpr (sizeof(Wd) == 8)
            cudaFuncSetAttribute(dev::window_walk_kernel<Wd, NW, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinkSmem);
        return true;
    }();
    (void)attr;
    SegDesc free = d;
    free.own_block = 0;   // the walkers per block of tfg_walk
    const LinkShape k = link_shape(free, kBlock, Shared::thread_bytes(d.R),
                                   sizeof(Wd) == 8 ? Device::thread_bytes(d.R) : (size_t)0);
    if (k.shared) {
        dev::window_walk_kernel<Wd, NW, false><<<k.grid, k.block, k.smem, st>>>(d, steps, choices, stride, log);
    } else if constexpr (sizeof(Wd) == 8) {
        dev::window_walk_kernel<Wd, NW, true><<<k.grid, k.block, k.smem, st>>>(d, steps, choices, stride, log);
    }
}

// `steps` uniform window steps of a population that window_apply_capacity accepts.
// choices (may be null): the first step's row of the population's walkers, `stride` apart.
void launch_window_walk(const SegDesc &d, int32_t steps, int32_t *choices, int64_t stride, const WindowLog &log,
                        cudaStream_t st) {
    if (d.n_walkers <= 0 || steps <= 0) return;
    if (d.word_bits == 32) window_walk_variant<uint32_t, 1>(d, steps, choices, stride, log, st);
    else if (d.R <= 64) window_walk_variant<uint64_t, 2>(d, steps, choices, stride, log, st);
    else window_walk_variant<uint64_t, 3>(d, steps, choices, stride, log, st);
}

}  // namespace tfg
