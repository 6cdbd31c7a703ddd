// Training of the proposal MLP on the tensor cores: one fused kernel computes,
// per 128-sample tile, the forward pass, the weighted logistic loss and the
// backward pass, and accumulates the weight gradients of the CTA's tiles in
// tensor memory; an Adam kernel then adds up the CTAs' gradients, updates FP32
// master weights and rewrites the BF16 parameter blob.
//
// Products (all BF16 x BF16 -> FP32, K = 16 per tcgen05.mma):
//   Z1  = X  W1            M = sample, N = hidden, K = input
//   Z2  = H1 W2            M = sample, N = hidden, K = hidden
//   dH1 = dZ2 W2^T         M = sample, N = hidden, K = hidden
//   dW2^T += dZ2^T H1      M = hidden, N = hidden, K = sample
//   dW1^T += dZ1^T X       M = hidden, N = input,  K = sample
// Every matrix is kept once, as 8 x 16-byte core matrices of a row-major tile; a
// product that wants its transpose reads the same tile as an MN-major operand.
// (Second, transposed copies written two bytes at a time, four lanes to a bank,
// were the larger part of the earlier kernel's 174 us for 262144 samples.)
//
// Epilogues read their accumulator in the 16x256b shape: a lane holds two adjacent
// columns of a row, so that packed BF16 pairs go out by stmatrix as whole core
// matrices, and it holds the same 32 columns in every tile, so that the sums over
// samples (b1, b2, w3) are additions into registers; only the output y is summed
// across lanes (four to a row).  Sums over the lanes and warps are taken once, at
// the end, in a fixed order.
//
// Two warpgroups, a tile each, hide one another's epilogues and products; a
// ninth warp issues all products, in a fixed order (the warpgroups share the
// weight gradients' accumulators: same sums on every run).  Per tile and
// warpgroup: wait Z1, write H1; wait Z2, write dZ2; wait dH1 and dW2, write
// dZ1 over dZ2; then dW1 and the next tile's Z1 go out together (its X was copied
// meanwhile into the other of two buffers).
#include <cstdint>
#include <cuda_bf16.h>

#include "tc_common.cuh"
#include "tfg_internal.h"

namespace tfg {
namespace {

constexpr int kIn = 32, kHid = 128, kTile = 128;
constexpr int kNumParams = kIn * kHid + kHid * kHid + 3 * kHid + 1;
// parameter blob offsets (bytes), shared with the scoring kernel
constexpr uint32_t kPB1 = (kIn + kHid) * kHid * 2, kPB3 = kPB1 + 3 * kHid * 4;   // after W1, W2; after b1, b2, w3
// FP32 parameter vector offsets (elements): W1 [32][128], W2 [128][128], b1, b2, w3, b3
constexpr int kVW1 = 0, kVW2 = kIn * kHid, kVB1 = kVW2 + kHid * kHid, kVB2 = kVB1 + kHid, kVW3 = kVB2 + kHid,
              kVB3 = kVW3 + kHid;

// shared memory regions (bytes); row-major tiles of core matrices
constexpr int kGradPartialRows = 256;          // CTAs of a deterministic (partial-row) gradient launch, at most
constexpr int kWGs = 2;                        // warpgroups, a tile each
constexpr int kGradThreads = kWGs * 128 + 32;  // and the warp that issues the products
constexpr uint32_t kSW1 = 0;                            // (i, h)
constexpr uint32_t kSW2 = kSW1 + kIn * kHid * 2;        // (h, o)
constexpr uint32_t kSD = kSW2 + kHid * kHid * 2;        // per warpgroup (s, o) = dZ2, then (s, h) = dZ1
constexpr uint32_t kSH = kSD + kWGs * kTile * kHid * 2; // per warpgroup (s, h) = H1
constexpr uint32_t kSX = kSH + kWGs * kTile * kHid * 2; // per warpgroup two of (s, i) = X
constexpr uint32_t kSVec = kSX + kWGs * 2 * kTile * kIn * 2;   // 0 - b1, b2, w3
constexpr uint32_t kTrainSmem = kSVec + 3 * kHid * 4;
constexpr uint32_t kHidRow = tc::kBlockRow;      // bytes of eight rows of a tile 128 columns wide
constexpr uint32_t kInRow = (kIn / 8) * 128;     // of one 32 columns wide

// tensor memory: the warpgroups' accumulators at 0 and 128, dW2^T, dW1^T
constexpr uint32_t kTmemCols = 512, kTmemDW2 = kWGs * 128, kTmemDW1 = kTmemDW2 + 128;

__device__ __forceinline__ void mbar_arrive(uint32_t mbar_saddr) {
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];\n\t}\n" ::"r"(mbar_saddr) : "memory");
}

// Eight BF16 weights; the blob may start at any 4-byte boundary.
__device__ __forceinline__ uint4 load_weights8(const uint8_t *p, bool aligned) {
    if (aligned) return *reinterpret_cast<const uint4 *>(p);
    const uint32_t *q = reinterpret_cast<const uint32_t *>(p);
    return make_uint4(q[0], q[1], q[2], q[3]);
}

// Gradient sums: every lane keeps its columns' sums, added over lanes and warps in
// a fixed order at the end; the CTA's totals go to grad by atomics
// (tfg_mlp_grad), or, with `partial`, to the CTA's own row
// partial[blockIdx.x][P + 1], which adam_kernel adds up in a fixed order: the
// training step's gradient is then the same bits on every run.
__global__ void __launch_bounds__(kGradThreads, 1) mlp_grad_kernel(
    const uint8_t *__restrict__ params, const __nv_bfloat16 *__restrict__ x, const float *__restrict__ label,
    const float *__restrict__ weight, int64_t n, float *__restrict__ grad, float *__restrict__ partial,
    int *__restrict__ err) {
    extern __shared__ __align__(1024) uint8_t smem[];
    __shared__ __align__(8) uint64_t s_ready[kWGs], s_done[kWGs], s_drain;
    __shared__ uint32_t tslot;
    __shared__ int timeout;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sm = tc::smem_u32(smem);
    float *vec = reinterpret_cast<float *>(smem + kSVec);

    {   // weights, 16 bytes at a time; eight lanes fill a core matrix
        const bool aligned = ((uintptr_t)params & 15u) == 0;
        for (int e = tid; e < (kIn + kHid) * 16; e += kGradThreads) {
            const int row = ((e >> 7) << 3) | (e & 7), kg = (e >> 3) & 15;   // rows of W1, then of W2
            *reinterpret_cast<uint4 *>(smem + (row >> 3) * kHidRow + kg * 128 + (row & 7) * 16) =
                load_weights8(params + ((size_t)row * kHid + kg * 8) * 2, aligned);
        }
        const float *v = reinterpret_cast<const float *>(params + kPB1);
        for (int e = tid; e < 3 * kHid; e += kGradThreads) vec[e] = e < kHid ? 0.f - v[e] : v[e];
    }
    if (warp == 0) tc::tmem_alloc(tc::smem_u32(&tslot), kTmemCols);
    if (tid == 0) {
        for (int g = 0; g < kWGs; ++g) {
            tc::mbar_init(tc::smem_u32(&s_ready[g]), 4);
            tc::mbar_init(tc::smem_u32(&s_done[g]), 1);
        }
        tc::mbar_init(tc::smem_u32(&s_drain), 1);
        timeout = 0;
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = tslot;

    // tile k of warpgroup g: blockIdx.x + gridDim.x (g + kWGs k)
    const int64_t ntiles = (n + kTile - 1) / kTile, round = (int64_t)gridDim.x * kWGs;
    auto tiles_of = [&](int g) {
        const int64_t t0 = blockIdx.x + (int64_t)gridDim.x * g;
        return t0 < ntiles ? (ntiles - t0 + round - 1) / round : (int64_t)0;
    };
    float gb1[32], gm2[32], gw3[32];   // column sums of dZ1, of dy where z2 > 0, of dy h2
#pragma unroll
    for (int k = 0; k < 32; ++k) gb1[k] = gm2[k] = gw3[k] = 0.f;
    float my_gb3 = 0.f, my_loss = 0.f;

    if (warp == kWGs * 4) {
        if (lane == 0) {
            constexpr uint32_t id_z = tc::idesc_bf16_f32(128, 128) | tc::kMnMajorB, id_h = tc::idesc_bf16_f32(128, 128),
                               id_w2 = tc::idesc_bf16_f32(128, 128) | tc::kMnMajorA | tc::kMnMajorB,
                               id_w1 = tc::idesc_bf16_f32(128, 32) | tc::kMnMajorA | tc::kMnMajorB;
            uint32_t phase = 0;   // bit g: parity of the next readiness of warpgroup g
            bool ok = true, first_w2 = true, first_w1 = true;
            auto ready = [&](int g) {
                ok = tc::mbar_wait(tc::smem_u32(&s_ready[g]), (phase >> g) & 1u);
                phase ^= 1u << g;
                tc::fence_after_sync();
                return ok;
            };
            auto layer1 = [&](int g, int64_t k) {
                const uint32_t X = sm + kSX + (uint32_t)(2 * g + (int)(k & 1)) * (kTile * kIn * 2);
#pragma unroll
                for (int kc = 0; kc < kIn / 16; ++kc)
                    tc::mma_bf16(tmem + 128 * g, tc::make_desc(X + kc * 256, 128, kInRow),
                                 tc::make_desc(sm + kSW1 + kc * 2 * kHidRow, kHidRow, 128), id_z, kc > 0);
            };
            for (int g = 0; g < kWGs; ++g)
                if (tiles_of(g) > 0 && ok && ready(g)) {
                    layer1(g, 0);
                    tc::mma_commit(tc::smem_u32(&s_done[g]));
                }
            const int64_t count[kWGs] = {tiles_of(0), tiles_of(1)};
            for (int64_t k = 0; k < count[0] && ok; ++k)
                for (int stage = 0; stage < 3 && ok; ++stage)
                    for (int g = 0; g < kWGs; ++g) {
                        const int64_t own = g == 0 ? count[0] : count[1];
                        if (k >= own || !ok || !ready(g)) continue;
                        const uint32_t acc = tmem + 128 * g, H = sm + kSH + g * (kTile * kHid * 2),
                                       D = sm + kSD + g * (kTile * kHid * 2);
                        if (stage == 0) {
#pragma unroll
                            for (int kc = 0; kc < kHid / 16; ++kc)
                                tc::mma_bf16(acc, tc::make_desc(H + kc * 256, 128, kHidRow),
                                             tc::make_desc(sm + kSW2 + kc * 2 * kHidRow, kHidRow, 128), id_z, kc > 0);
                        } else if (stage == 1) {
#pragma unroll
                            for (int kc = 0; kc < kHid / 16; ++kc)   // dH1 = dZ2 W2^T (K = output unit)
                                tc::mma_bf16(acc, tc::make_desc(D + kc * 256, 128, kHidRow),
                                             tc::make_desc(sm + kSW2 + kc * 256, 128, kHidRow), id_h, kc > 0);
#pragma unroll
                            for (int kc = 0; kc < kTile / 16; ++kc)  // dW2^T += dZ2^T H1 (K = sample)
                                tc::mma_bf16(tmem + kTmemDW2, tc::make_desc(D + kc * 2 * kHidRow, kHidRow, 128),
                                             tc::make_desc(H + kc * 2 * kHidRow, kHidRow, 128), id_w2,
                                             !first_w2 || kc > 0);
                            first_w2 = false;
                        } else {
                            const uint32_t X = sm + kSX + (uint32_t)(2 * g + (int)(k & 1)) * (kTile * kIn * 2);
#pragma unroll
                            for (int kc = 0; kc < kTile / 16; ++kc)  // dW1^T += dZ1^T X (K = sample)
                                tc::mma_bf16(tmem + kTmemDW1, tc::make_desc(D + kc * 2 * kHidRow, kHidRow, 128),
                                             tc::make_desc(X + kc * 2 * kInRow, kInRow, 128), id_w1,
                                             !first_w1 || kc > 0);
                            first_w1 = false;
                            if (k + 1 < own) layer1(g, k + 1);
                        }
                        tc::mma_commit(tc::smem_u32(&s_done[g]));
                    }
            if (!ok) timeout = 1;
            // all products done before the accumulators are read or given back
            tc::mma_commit(tc::smem_u32(&s_drain));
            if (!tc::mbar_wait(tc::smem_u32(&s_drain), 0)) timeout = 1;
        }
        __syncwarp();
    } else {
        const int g = warp >> 2, wq = warp & 3;
        const uint32_t tacc = tmem + 128 * g + ((uint32_t)(wq * 32) << 16);
        const uint32_t H = sm + kSH + g * (kTile * kHid * 2), D = sm + kSD + g * (kTile * kHid * 2);
        const uint32_t ready = tc::smem_u32(&s_ready[g]), done = tc::smem_u32(&s_done[g]);
        const float2 *nB1 = reinterpret_cast<const float2 *>(vec) + (lane & 3), *B2 = nB1 + kHid / 2, *W3 = B2 + kHid / 2;
        const float b3 = *reinterpret_cast<const float *>(params + kPB3);
        const int64_t own = tiles_of(g);
        uint32_t phase = 0;
        auto publish = [&] {   // this warp's part of an operand is written, its accumulator rows are read
            tc::fence_async_smem();
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(ready);
        };
        auto wait = [&] {
            const bool ok = tc::mbar_wait(done, phase);
            phase ^= 1;
            tc::fence_after_sync();
            return __all_sync(0xffffffffu, ok) != 0;
        };
        auto load_x = [&](int64_t k) {   // tile k's rows (zero past n), eight lanes to a core matrix
            const int64_t row0 = (blockIdx.x + (int64_t)gridDim.x * (g + kWGs * k)) * kTile;
            const uint32_t X = sm + kSX + (uint32_t)(2 * g + (int)(k & 1)) * (kTile * kIn * 2);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int rg = wq * 4 + i;
                const int64_t row = row0 + rg * 8 + (lane & 7);
                const bool in = row < n;
                tc::cp_async16(X + rg * kInRow + lane * 16, x + (in ? row * kIn + (lane >> 3) * 8 : 0), in);
            }
        };
        bool ok = true;
        if (own > 0) {
            load_x(0);
            tc::cp_async_wait();
            publish();
        }
        for (int64_t k = 0; k < own; ++k) {
            // this lane's sample for the loss: row lane / 4 + 8 (lane % 4) of the warp's 32
            const int64_t row = (blockIdx.x + (int64_t)gridDim.x * (g + kWGs * k)) * kTile + wq * 32 + (lane >> 2) +
                                8 * (lane & 3);
            const float lab = row < n ? label[row] : 0.f;
            const float wt = row < n ? weight[row] : 0.f;
            if (!(ok = wait())) break;
            if (k + 1 < own) load_x(k + 1);   // dW1 of tile k - 1, the buffer's last reader, is done
            // ---- layer 1: h1 = relu(z1 + b1) as BF16; bits of z1 > 0.  As -z: its minimum with +0
            // has the sign bit exactly where z > 0.
            uint32_t mask[4] = {0u, 0u, 0u, 0u};
            float2 b[4], w[4];   // a chunk's biases and weights, kept for the lower rows
            tc::for_blocks(tacc, [&](int c, int h, uint32_t(&r)[16]) {
                float v[16];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (h == 0) b[j] = nB1[16 * c + 4 * j];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float t = fminf(((e & 1) ? b[j].y : b[j].x) - __uint_as_float(r[4 * j + e]), 0.f);
                        mask[c] = __funnelshift_l(__float_as_uint(t), mask[c], 1);
                        v[4 * j + e] = -t;
                    }
                }
                tc::st_block<false>(H, lane, wq * 32 + h * 16, c, v);
            });
            publish();
            if (!(ok = wait())) break;
            // ---- layer 2 and output: y of four rows, summed over the four lanes of a row
            float2 ys[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) ys[q] = make_float2(0.f, 0.f);
            tc::for_blocks(tacc, [&](int c, int h, uint32_t(&r)[16]) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (h == 0) b[j] = B2[16 * c + 4 * j], w[j] = W3[16 * c + 4 * j];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float2 z = __fadd2_rn(
                            make_float2(__uint_as_float(r[4 * j + 2 * q]), __uint_as_float(r[4 * j + 2 * q + 1])), b[j]);
                        ys[2 * h + q] = __ffma2_rn(make_float2(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f)), w[j], ys[2 * h + q]);
                    }
                }
            });
            float y = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float s = ys[q].x + ys[q].y;
                s += __shfl_xor_sync(0xffffffffu, s, 1);
                s += __shfl_xor_sync(0xffffffffu, s, 2);
                y = (lane & 3) == q ? s : y;
            }
            y += b3;
            const float mrg = -(2.f * lab - 1.f) * y;
            my_loss += wt * (fmaxf(mrg, 0.f) + log1pf(expf(-fabsf(mrg))));
            const float dy1 = wt * (1.f / (1.f + expf(-y)) - lab);
            my_gb3 += dy1;
            float dy[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) dy[q] = __shfl_sync(0xffffffffu, dy1, (lane & 28) | q);
            // dz2 = dy w3 relu'(z2); sums for w3 and b2
            tc::for_blocks(tacc, [&](int c, int h, uint32_t(&r)[16]) {
                float v[16];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (h == 0) b[j] = B2[16 * c + 4 * j], w[j] = W3[16 * c + 4 * j];
                    const int a = 8 * c + 2 * j;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float2 z = __fadd2_rn(
                            make_float2(__uint_as_float(r[4 * j + 2 * q]), __uint_as_float(r[4 * j + 2 * q + 1])), b[j]);
                        const float d = dy[2 * h + q];
                        const float2 on = make_float2(z.x > 0.f ? d : 0.f, z.y > 0.f ? d : 0.f);
                        const float2 gw = __ffma2_rn(make_float2(d, d), make_float2(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f)),
                                                     make_float2(gw3[a], gw3[a + 1]));
                        const float2 gm = __fadd2_rn(make_float2(gm2[a], gm2[a + 1]), on);
                        gw3[a] = gw.x; gw3[a + 1] = gw.y;
                        gm2[a] = gm.x; gm2[a + 1] = gm.y;
                        v[4 * j + 2 * q] = on.x * w[j].x;
                        v[4 * j + 2 * q + 1] = on.y * w[j].y;
                    }
                }
                tc::st_block<false>(D, lane, wq * 32 + h * 16, c, v);
            });
            publish();
            if (!(ok = wait())) break;
            // ---- dz1 = dH1 relu'(z1) over dZ2; sums for b1
            tc::for_blocks(tacc, [&](int c, int h, uint32_t(&r)[16]) {
                float v[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) {   // bit 31 - (16 h + e) of mask[c]
                    v[e] = (mask[c] >> (31 - 16 * h - e)) & 1u ? __uint_as_float(r[e]) : 0.f;
                    const int a = 8 * c + 2 * (e >> 2) + (e & 1);
                    gb1[a] += v[e];
                }
                tc::st_block<false>(D, lane, wq * 32 + h * 16, c, v);
            });
            tc::cp_async_wait();   // the next tile's rows
            publish();
        }
        tc::cp_async_wait();
        if (!ok) timeout = 1;
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (timeout) {
        if (tid == 0) atomicExch(err, 1);
    } else {
        // ---- flush: dW2[h][o] (TMEM lane o, column h), dW1[i][h] (lane h, column i), vectors
        float *pp = partial ? partial + (size_t)blockIdx.x * (kNumParams + 1) : nullptr;
        auto put = [&](int e, float v) {
            if (pp) pp[e] = v;
            else atomicAdd(&grad[e], v);
        };
        float *sums = reinterpret_cast<float *>(smem + kSD);    // [3][8][128], over the operands
        float *scal = sums + 3 * 4 * kWGs * kHid;               // [8][2]
        if (warp < 4 * kWGs) {
            const int g = warp >> 2, unit = tid & 127;
            const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
#pragma unroll
            for (int c0 = 0; c0 < kHid / kWGs; c0 += 32) {
                float v[32];
                const int h0 = g * (kHid / kWGs) + c0;
                tc::tmem_ld32(tmem + kTmemDW2 + lanes + h0, v);
#pragma unroll
                for (int q = 0; q < 32; ++q) put(kVW2 + (h0 + q) * kHid + unit, v[q]);
            }
            if (g == kWGs - 1) {
                float v[32];
                tc::tmem_ld32(tmem + kTmemDW1 + lanes, v);
#pragma unroll
                for (int q = 0; q < 32; ++q) put(kVW1 + q * kHid + unit, v[q]);
            }
            // the eight lanes of a column pair, then (below) the eight warps
            auto column = [&](int which, float (&s)[32]) {
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    float t = s[k];
                    t += __shfl_xor_sync(0xffffffffu, t, 4);
                    t += __shfl_xor_sync(0xffffffffu, t, 8);
                    t += __shfl_xor_sync(0xffffffffu, t, 16);
                    if (lane < 4) sums[(which * 4 * kWGs + warp) * kHid + 8 * (k >> 1) + 2 * lane + (k & 1)] = t;
                }
            };
            column(0, gb1);
            column(1, gm2);
            column(2, gw3);
            for (int o = 16; o > 0; o >>= 1) {
                my_gb3 += __shfl_xor_sync(0xffffffffu, my_gb3, o);
                my_loss += __shfl_xor_sync(0xffffffffu, my_loss, o);
            }
            if (lane == 0) {
                scal[2 * warp] = my_gb3;
                scal[2 * warp + 1] = my_loss;
            }
        }
        __syncthreads();
        for (int e = tid; e < 3 * kHid; e += kGradThreads) {   // b1, b2, w3
            const float *s = sums + (e / kHid) * 4 * kWGs * kHid + e % kHid;
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < 4 * kWGs; ++w) v += s[w * kHid];
            // b2: dz2 = w3 dy where z2 > 0, w3 the same for every sample
            if (e / kHid == 1 && v != 0.f) v *= vec[2 * kHid + e % kHid];
            put(kVB1 + e, v);
        }
        if (tid < 2) {   // b3, then the loss after the gradient vector
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < 4 * kWGs; ++w) v += scal[2 * w + tid];
            put(tid == 0 ? kVB3 : kNumParams, v);
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, kTmemCols);
}

// Adam on FP32 master weights; the BF16 / FP32 parameter blob is rewritten.
// The gradient is first added up from `parts` rows of partial[][P + 1], by eight
// threads an element in a fixed order (one thread an element, over 64 rows, was a
// launch of its own of 3.3 us beside Adam's 2.5), and kept in grad with the loss.
// omb1 = 1 - beta1, omb2 = 1 - beta2 and the bias corrections bc1 = 1 - beta1^t,
// bc2 = 1 - beta2^t come from the host, formed in double precision (1 - beta
// formed from an FP32 beta would be off by up to 2^-24 / (1 - beta) relative).
constexpr int kAdamSplit = 8;
__global__ void __launch_bounds__(32 * kAdamSplit) adam_kernel(
    float *master, float *m1, float *m2, float *grad, const float *__restrict__ partial, int parts, uint8_t *blob,
    float lr, float beta1, float omb1, float beta2, float omb2, float eps, float bc1, float bc2) {
    __shared__ float part[kAdamSplit][32];
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (e <= kNumParams) {
        const int b0 = (int)((int64_t)parts * q / kAdamSplit), b1 = (int)((int64_t)parts * (q + 1) / kAdamSplit);
#pragma unroll 8
        for (int b = b0; b < b1; ++b) s += partial[(size_t)b * (kNumParams + 1) + e];
    }
    part[q][lane] = s;
    __syncthreads();
    if (q != 0 || e > kNumParams) return;
    float g = part[0][lane];
#pragma unroll
    for (int k = 1; k < kAdamSplit; ++k) g += part[k][lane];
    grad[e] = g;
    if (e == kNumParams) return;   // the loss
    const float a = beta1 * m1[e] + omb1 * g;
    const float b = beta2 * m2[e] + omb2 * g * g;
    m1[e] = a;
    m2[e] = b;
    const float p = master[e] - lr * (a / bc1) / (sqrtf(b / bc2) + eps);
    master[e] = p;
    if (e < kVB1) {
        *reinterpret_cast<__nv_bfloat16 *>(blob + (size_t)e * 2) = __float2bfloat16_rn(p);
    } else {
        reinterpret_cast<float *>(blob + kPB1)[e - kVB1] = p;
    }
}

__global__ void master_from_blob_kernel(const uint8_t *blob, float *master, float *m1, float *m2) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= kNumParams) return;
    master[e] = e < kVB1 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(blob)[e])
                         : reinterpret_cast<const float *>(blob + kPB1)[e - kVB1];
    m1[e] = 0.f;
    m2[e] = 0.f;
}

}  // namespace

int mlp_num_params() { return kNumParams; }

int grad_partial_rows() { return kGradPartialRows; }

int launch_mlp_grad(const void *params, const void *x, const float *label, const float *weight, int64_t n,
                    float *grad, int *err, cudaStream_t st, float *partial) {
    if (n <= 0) return 0;
    static bool attr = [] {
        cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTrainSmem);
        return true;
    }();
    (void)attr;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t tiles = (n + kTile - 1) / kTile;
    int grid = (int)(tiles < sms ? tiles : sms);
    if (partial && grid > kGradPartialRows) grid = kGradPartialRows;
    mlp_grad_kernel<<<grid, kGradThreads, kTrainSmem, st>>>(
        reinterpret_cast<const uint8_t *>(params), reinterpret_cast<const __nv_bfloat16 *>(x), label, weight, n, grad,
        partial, err);
    return grid;
}

void launch_adam(float *master, float *m1, float *m2, float *grad, const float *partial, int parts, void *blob,
                 float lr, int step, cudaStream_t st) {
    const double beta1 = 0.9, beta2 = 0.999, eps = 1e-8;
    double p1 = 1.0, p2 = 1.0;
    for (int k = 0; k < step; ++k) { p1 *= beta1; p2 *= beta2; }
    adam_kernel<<<(kNumParams + 1 + 31) / 32, 32 * kAdamSplit, 0, st>>>(
        master, m1, m2, grad, partial, parts, reinterpret_cast<uint8_t *>(blob), lr, (float)beta1,
        (float)(1.0 - beta1), (float)beta2, (float)(1.0 - beta2), (float)eps, (float)(1.0 - p1), (float)(1.0 - p2));
}

void launch_master_from_blob(const void *blob, float *master, float *m1, float *m2, cudaStream_t st) {
    master_from_blob_kernel<<<(kNumParams + 255) / 256, 256, 0, st>>>(reinterpret_cast<const uint8_t *>(blob),
                                                                      master, m1, m2);
}

}  // namespace tfg
