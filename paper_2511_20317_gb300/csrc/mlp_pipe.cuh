// Tile pipeline of the proposal MLP 32 -> 128 -> 128 -> 1 on the tcgen05
// tensor cores, shared by the row-scoring kernel (features read from device
// memory) and the fused window-scoring kernel (features computed in place).
//
// A CTA holds the weights once (W1 and W2 as MN-major BF16 operands, w3 in
// FP32) and runs NWG independent warpgroups.  Warpgroup g owns
// TMEM columns [128 g, 128 g + 128) (its accumulator), an A tile X (128 rows
// x 32 features) and an A tile H1 (128 rows x 128 hidden inputs) in shared
// memory, one mbarrier and one named barrier; its thread q owns tile row q,
// which is TMEM lane 32 (warp % 4) + lane, so every tcgen05.ld of a thread
// reads its own row.  Per tile:
//   producer: row q -> X                      (the Prod object, prefetched a tile ahead)
//   MMA1  acc = X W1        (2 x K=16, one elected thread, commit -> mbarrier)
//   epi1  H1 = bf16(relu(acc + b1))            (cvt.rn.relu.bf16x2: ReLU and rounding in one)
//   MMA2  acc = H1 W2 + b2  (9 x K=16)
//   epi2  y = b3 + sum_o w3[o] relu(acc[o])
// The warpgroups of a CTA interleave on the tensor pipe: while one waits for
// its products, the others run their epilogues; a warpgroup itself writes
// the next tile's X while its MMA2 runs (X's only reader, MMA1, is done), so
// the next MMA1 follows epi2 at once.  TMEM loads are issued one 16-column
// chunk ahead of the arithmetic on the previous chunk.
//
// MMA2 adds its bias, as one more K=16 step: its A operand, shared by all warpgroups,
// holds three ones in every row, its B operand b2 as three BF16 pieces (hi + mid + lo to
// FP32 precision), the rest is zero.  Where the producer controls the feature rows
// (Prod::kFold) MMA1 adds its own too: the constant-one input f31 is joined by f29 =
// f30 = 1 on every real row, and W1's rows 29, 30, 31 hold the pieces of W1[31] + b1.
// Features f29 and f30 are zero by definition, so their W1 rows never contribute
// otherwise; rows past a window (all features zero) get no bias, and their
// scores are not used.  For arbitrary rows epi1 adds b1 in FP32, as ever: its sum is
// rounded to BF16, and another order of the sum rounds some of them the other way.
// It reads the accumulator in the 16x256b shape, where 16 pairs of biases a lane serve
// all its rows, and stay in registers.
//
// Bounds: a round trip of a product (barrier, issue, commit, wait) takes 375 cycles
// beside the product's 64 a K=16 step, and a warpgroup makes two a tile; four
// warpgroups, as many as tensor memory has accumulators for, do not hide it all
// (1048576 rows: 32 us with the epilogues left out, 45 with either).  A 16-byte
// shared load that all lanes share costs four wavefronts; b1, b2 and w3 read so were half
// of the shared-memory traffic: 66.5 us, w3 alone 53.6.
//
// Every mbarrier wait is bounded; a warpgroup whose wait gives up records
// the timeout, stops taking tiles, waits (bounded again) for its products in
// flight and sets *err before the CTA releases its tensor memory.
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

#include "tc_common.cuh"

namespace tfg {
namespace mlp {

constexpr int kIn = 32, kHid = 128, kTile = 128;
// parameter blob (bytes): W1 bf16 [32][128], W2 bf16 [128][128], b1, b2, w3 f32 [128], b3 f32, pad
constexpr uint32_t kParamW1 = 0;
constexpr uint32_t kParamW2 = kParamW1 + kIn * kHid * 2;
constexpr uint32_t kParamB1 = kParamW2 + kHid * kHid * 2;
constexpr uint32_t kParamB2 = kParamB1 + kHid * 4;
constexpr uint32_t kParamW3 = kParamB2 + kHid * 4;
constexpr uint32_t kParamB3 = kParamW3 + kHid * 4;
constexpr uint32_t kParamBytes = kParamB3 + 16;
constexpr uint32_t kWRow = (kHid / 8) * 128;   // shared bytes of eight rows of a weight matrix

// Shared-memory layout (dynamic part): W1, W2 (each with its bias rows), the bias steps' A
// operand, w3, then per warpgroup X and H1.
template <bool FOLD>
struct Layout {
    static constexpr int W2Rows = kHid + 16;
    static constexpr uint32_t W1 = 0;                             // B of MMA1: 32 (input) x 128 (hidden)
    static constexpr uint32_t W2 = W1 + kIn * kHid * 2;        // B of MMA2: W2Rows x 128 (out)
    static constexpr uint32_t Ones = W2 + W2Rows * kHid * 2;      // 128 x 16: 1 1 1 0 ... in every row
    static constexpr uint32_t Vec = Ones + kTile * 16 * 2;        // w3
    static constexpr uint32_t WG = Vec + kHid * 4;                // first warpgroup area
    static constexpr uint32_t X = 0;                              // per warpgroup: X 128 x 32
    static constexpr uint32_t H1 = kTile * kIn * 2;               //                H1 128 x 128
    static constexpr uint32_t WGBytes = H1 + kTile * kHid * 2;
    static constexpr uint32_t bytes(int nwg) { return WG + nwg * WGBytes; }
};
template <int NWG>
constexpr uint32_t tmem_cols() { return NWG <= 1 ? 128u : (NWG <= 2 ? 256u : 512u); }

__device__ __forceinline__ uint32_t pack_relu_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// named barrier of warpgroup g (ids 1..NWG; 0 is __syncthreads)
__device__ __forceinline__ void wg_sync(int g) {
    asm volatile("bar.sync %0, 128;" ::"r"(g + 1) : "memory");
}
// named barrier with an OR reduction of a predicate over the warpgroup
__device__ __forceinline__ bool wg_any(int g, bool p) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred pi, po;\n\t"
        "setp.ne.u32 pi, %2, 0;\n\t"
        "bar.red.or.pred po, %1, 128, pi;\n\t"
        "selp.u32 %0, 1, 0, po;\n\t}\n"
        : "=r"(r)
        : "r"(g + 1), "r"((uint32_t)p)
        : "memory");
    return r != 0;
}

// 16 consecutive FP32 accumulator columns of this thread's TMEM lane, without
// waiting: the registers are valid after the next tmem_wait().
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// Wait for this thread's TMEM loads; the empty asm afterwards redefines the
// registers of the chunk that is read next, so no use of them moves above the wait.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                   "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
                   "+r"(r[14]), "+r"(r[15]));
}

__device__ __forceinline__ __nv_bfloat16 bf(float v) { return __float2bfloat16_rn(v); }

// Weights, bias pieces and w3 of the parameter blob into the CTA's shared memory.  W1 and
// W2 stay row-major (row = input unit), 16 bytes at a time into 8 x 16-byte core
// matrices: the products read them as MN-major B operands.
template <bool FOLD>
__device__ __forceinline__ void load_weights(const uint8_t *__restrict__ params, uint8_t *smem, int tid, int nthr) {
    using LY = Layout<FOLD>;
    const float *b1 = reinterpret_cast<const float *>(params + kParamB1);
    const float *b2 = reinterpret_cast<const float *>(params + kParamB2);
    // consecutive lanes take the eight rows of a core matrix
    for (int e = tid; e < (kIn + LY::W2Rows) * (kHid / 8); e += nthr) {
        const int row = ((e >> 7) << 3) | (e & 7), kg = (e >> 3) & 15;   // rows of W1, then of W2
        const bool first = row < kIn;
        const int k = first ? row : row - kIn;   // row of its matrix
        const int piece = first ? kIn - 1 - k : k - kHid;   // of the bias
        uint4 v;
        if (first ? FOLD && piece < 3 : piece >= 0) {
            uint32_t h[4] = {0u, 0u, 0u, 0u};
            if (piece < 3) {
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int c = 8 * kg + u;
                    float f = first ? b1[c] : b2[c];
                    if (first) f += __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(params)[31 * kHid + c]);
                    float hi = __bfloat162float(bf(f));
                    if (isinf(hi)) hi = __bfloat162float(__float2bfloat16_rz(f));   // finite, unless f is not
                    const float rest = isinf(hi) ? 0.f : f - hi, mid = __bfloat162float(bf(rest));
                    f = piece == 0 ? hi : (piece == 1 ? mid : rest - mid);
                    h[u >> 1] |= (uint32_t)__bfloat16_as_ushort(bf(f)) << (16 * (u & 1));
                }
            }
            v = make_uint4(h[0], h[1], h[2], h[3]);
        } else {
            v = *reinterpret_cast<const uint4 *>(params + (first ? kParamW1 : kParamW2) + ((size_t)k * kHid + kg * 8) * 2);
        }
        *reinterpret_cast<uint4 *>(smem + LY::W1 + (row >> 3) * kWRow + kg * 128 + (row & 7) * 16) = v;
    }
    for (int e = tid; e < kTile * 2; e += nthr) {   // row e / 2: 1 1 1 0 0 0 0 0, then zeros
        const bool ones = (e & 8) == 0;
        *reinterpret_cast<uint4 *>(smem + LY::Ones + e * 16) =
            make_uint4(ones ? 0x3F803F80u : 0u, ones ? 0x00003F80u : 0u, 0u, 0u);
    }
    float *vec = reinterpret_cast<float *>(smem + LY::Vec);
    for (int e = tid; e < kHid; e += nthr) {
        vec[e] = reinterpret_cast<const float *>(params + kParamW3)[e];
    }
}

// Store 8 consecutive features (as 4 packed bf16x2 words) of row q into an A tile.
__device__ __forceinline__ void st_row8(uint8_t *tile, int q, int col0, int K, uint4 v) {
    *reinterpret_cast<uint4 *>(tile + tc::kmajor_offset(q, col0, K)) = v;
}

// The pipeline.  Prod (one object per thread; static bool kFold) provides
//   bool begin(int q)                 start loading the warpgroup's next tile's input for row q;
//                                     false: no tile is left (the same answer for the 128 rows)
//   void mid(int q)                   second load phase of the tile begun last (may be empty)
//   int64_t fill(uint8_t *sX, int q)  write row q of the tile loaded last into X (kFold:
//                                     features 29 and 30 one on every real row); returns
//                                     the row's output index (-1: no output)
//   void emit(float y, int64_t o)     the score y of the row whose fill returned o
template <int NWG, class Prod>
__device__ __forceinline__ void run_tiles(const uint8_t *__restrict__ params, Prod &prod, int *__restrict__ err,
                                          uint32_t first_limit, uint8_t *smem,
                                          uint64_t *mbar, uint32_t *tslot, int *timeout_flag) {
    constexpr bool FOLD = Prod::kFold;
    using LY = Layout<FOLD>;
    const int tid = threadIdx.x, g = tid >> 7, q = tid & 127, warp = tid >> 5, lane = tid & 31;
    load_weights<FOLD>(params, smem, tid, NWG * 128);
    uint8_t *sX = smem + LY::WG + g * LY::WGBytes + LY::X;
    uint8_t *sH1 = smem + LY::WG + g * LY::WGBytes + LY::H1;
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(tslot), tmem_cols<NWG>());
    if (q == 0) tc::mbar_init(tc::smem_u32(&mbar[g]), 1);
    if (tid == 0) *timeout_flag = 0;
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();

    const uint32_t tacc = *tslot + (uint32_t)(g * 128);
    const uint32_t tlane = tacc + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t mb = tc::smem_u32(&mbar[g]);
    const uint32_t aX = tc::smem_u32(sX), aH1 = tc::smem_u32(sH1);
    const uint32_t aW1 = tc::smem_u32(smem + LY::W1), aW2 = tc::smem_u32(smem + LY::W2);
    const uint64_t ones = tc::make_desc(tc::smem_u32(smem + LY::Ones), 128, 256);
    const float *w3 = reinterpret_cast<const float *>(smem + LY::Vec);
    const float b3 = *reinterpret_cast<const float *>(params + kParamB3);
    constexpr uint32_t idesc = tc::idesc_bf16_f32(kTile, kHid) | tc::kMnMajorB;
    uint32_t phase = 0;
    bool timed_out = false, first_wait = true;
    float2 b1[FOLD ? 1 : 16];   // not folded: of this lane's columns, 8 k + 2 (lane % 4) + {0, 1}
    if constexpr (!FOLD) {
#pragma unroll
        for (int k = 0; k < 16; ++k) b1[k] = reinterpret_cast<const float2 *>(params + kParamB1)[4 * k + (lane & 3)];
    }

    // the first tile, its features in X
    bool has = prod.begin(q);
    if (has) prod.mid(q);
    int64_t out_cur = has ? prod.fill(sX, q) : -1;
    while (has) {
        const bool more = prod.begin(q);   // first load phase of the next tile
        tc::fence_async_smem();
        tc::fence_before_sync();
        wg_sync(g);
        tc::fence_after_sync();
        if (q == 0) {
#pragma unroll
            for (int kc = 0; kc < kIn / 16; ++kc)
                tc::mma_bf16(tacc, tc::make_desc(aX + kc * 256, 128, (kIn / 8) * 128),
                             tc::make_desc(aW1 + kc * 2 * kWRow, kWRow, 128), idesc, kc > 0);
            tc::mma_commit(mb);
        }
        bool ok = tc::mbar_wait(mb, phase, first_wait ? first_limit : tc::kWaitLimit);
        first_wait = false;
        if (wg_any(g, !ok)) { timed_out = true; break; }
        phase ^= 1;
        tc::fence_after_sync();
        // ---- epi1: h1 = bf16(relu(z1)) -> H1
        if constexpr (FOLD) {   // row q, TMEM chunks of 16 columns one ahead
            uint32_t ra[16], rb[16];
            tmem_ld16_nowait(tlane, ra);
            tmem_wait(ra);
#pragma unroll
            for (int c = 0; c < kHid / 16; ++c) {
                uint32_t(&cur)[16] = (c & 1) ? rb : ra;
                uint32_t(&nxt)[16] = (c & 1) ? ra : rb;
                if (c + 1 < kHid / 16) tmem_ld16_nowait(tlane + 16 * (c + 1), nxt);
#pragma unroll
                for (int u = 0; u < 16; u += 8) {
                    float f[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) f[k] = __uint_as_float(cur[u + k]);
                    st_row8(sH1, q, 16 * c + u, kHid,
                            make_uint4(pack_relu_bf16x2(f[0], f[1]), pack_relu_bf16x2(f[2], f[3]),
                                       pack_relu_bf16x2(f[4], f[5]), pack_relu_bf16x2(f[6], f[7])));
                }
                if (c + 1 < kHid / 16) tmem_wait(nxt);
            }
        } else {
            // blocks of 16 rows x 32 columns: a lane's biases stay in registers
            tc::for_blocks(tlane, [&](int c, int h, uint32_t(&r)[16]) {
                float v[16];
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int e = 4 * j; e < 4 * j + 4; e += 2) {
                        const float2 z = __fadd2_rn(
                            make_float2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), b1[4 * c + j]);
                        v[e] = z.x;
                        v[e + 1] = z.y;
                    }
                tc::st_block<true>(aH1, lane, (q & 96) + 16 * h, c, v);
            });
        }
        if (more) prod.mid(q);   // second load phase of the next tile
        tc::fence_async_smem();
        tc::fence_before_sync();
        wg_sync(g);
        tc::fence_after_sync();
        if (q == 0) {
#pragma unroll
            for (int kc = 0; kc < kHid / 16; ++kc)
                tc::mma_bf16(tacc, tc::make_desc(aH1 + kc * 256, 128, kWRow),
                             tc::make_desc(aW2 + kc * 2 * kWRow, kWRow, 128), idesc, kc > 0);
            tc::mma_bf16(tacc, ones, tc::make_desc(aW2 + (kHid / 8) * kWRow, kWRow, 128), idesc, true);
            tc::mma_commit(mb);
        }
        // while MMA2 runs: the next tile's features into X (MMA1, its only reader, is done)
        const int64_t out_next = more ? prod.fill(sX, q) : -1;
        ok = tc::mbar_wait(mb, phase);
        if (wg_any(g, !ok)) { timed_out = true; break; }
        phase ^= 1;
        tc::fence_after_sync();
        // ---- epi2: y = b3 + w3 . relu(z2)
        float2 y2 = make_float2(b3, 0.f);
        {
            uint32_t ra[16], rb[16];
            tmem_ld16_nowait(tlane, ra);
            tmem_wait(ra);
#pragma unroll
            for (int c = 0; c < kHid / 16; ++c) {
                uint32_t(&cur)[16] = (c & 1) ? rb : ra;
                uint32_t(&nxt)[16] = (c & 1) ? ra : rb;
                if (c + 1 < kHid / 16) tmem_ld16_nowait(tlane + 16 * (c + 1), nxt);
#pragma unroll
                for (int u = 0; u < 16; u += 4) {
                    const float4 w = *reinterpret_cast<const float4 *>(w3 + 16 * c + u);
                    const float z0 = __uint_as_float(cur[u]), z1 = __uint_as_float(cur[u + 1]);
                    const float z2 = __uint_as_float(cur[u + 2]), z3 = __uint_as_float(cur[u + 3]);
                    y2 = __ffma2_rn(make_float2(fmaxf(z0, 0.f), fmaxf(z1, 0.f)), make_float2(w.x, w.y), y2);
                    y2 = __ffma2_rn(make_float2(fmaxf(z2, 0.f), fmaxf(z3, 0.f)), make_float2(w.z, w.w), y2);
                }
                if (c + 1 < kHid / 16) tmem_wait(nxt);
            }
        }
        prod.emit(y2.x + y2.y, out_cur);
        // the next MMA1 overwrites the accumulator: order this thread's loads before it
        tc::fence_before_sync();
        out_cur = out_next;
        has = more;
    }
    if (timed_out) {
        // the awaited products may still be in flight: one more bounded wait before release
        tc::mbar_wait(mb, phase);
        if (q == 0) {
            *timeout_flag = 1;
            atomicExch(err, 1);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(*tslot, tmem_cols<NWG>());
}

}  // namespace mlp
}  // namespace tfg
