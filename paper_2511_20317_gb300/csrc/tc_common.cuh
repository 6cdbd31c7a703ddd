// tcgen05 building blocks for the proposal MLP (sm_103a): tensor-memory
// allocation, shared-memory matrix descriptors, BF16 MMA with FP32
// accumulation, commit to an mbarrier with a bounded wait, and TMEM loads.
//
// Operand layout in shared memory: K-major, no swizzle.  A matrix of R rows
// by K bf16 columns is stored as "core matrices" of 8 rows x 16 bytes
// (8 x 8 elements); core matrix (rg, kg) sits at byte (rg * K/8 + kg) * 128
// and its row q at +16q.  For one MMA of K = 16 the descriptor's leading
// byte offset is the distance between the two K-adjacent core matrices
// (128 B) and the stride byte offset the distance between 8-row groups
// (K/8 * 128 B).
#pragma once
#include <cstdint>
#include <cuda_bf16.h>

namespace tfg {
namespace tc {

constexpr uint32_t kWaitLimit = 1u << 22;   // bounded mbarrier polling

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// byte offset of element (row, col) of an R x K bf16 operand (K-major, no swizzle)
__device__ __forceinline__ uint32_t kmajor_offset(int row, int col, int K) {
    return (uint32_t)(((row >> 3) * (K >> 3) + (col >> 3)) * 128 + (row & 7) * 16 + (col & 7) * 2);
}

// Shared-memory matrix descriptor: start address, leading / stride byte
// offsets (16-byte units), descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// An operand read MN-major takes the same core matrices of a row-major tile whose rows run
// along K: its leading byte offset is the distance between 8-row groups, its stride byte
// offset that between 8-column groups (128 B).
constexpr uint32_t kMnMajorA = 1u << 15, kMnMajorB = 1u << 16;   // bits of the instruction descriptor
// Instruction descriptor of kind::f16: D = F32, A = B = BF16, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot_saddr, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_saddr), "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// make generic-proxy shared-memory writes visible to the tensor core (async proxy)
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, bool accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"((uint32_t)accumulate));
}

__device__ __forceinline__ void mma_commit(uint32_t mbar_saddr) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar_saddr)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar_saddr, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar_saddr), "r"(count));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Bounded wait for the mbarrier phase `parity` to complete: at most `limit`
// polls; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar_saddr, uint32_t parity, uint32_t limit = kWaitLimit) {
    for (uint32_t it = 0; it < limit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(mbar_saddr), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int c = 0; c < 32; ++c) v[c] = __uint_as_float(r[c]);
}

// 16 bytes from global to shared memory (zeros unless full), and the wait for all of a thread's.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool full) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(full ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 32 columns x 16 rows of an accumulator: registers 4 j + {0, 1} hold columns 8 j + 2 (lane % 4)
// + {0, 1} of row lane / 4, registers 4 j + {2, 3} those of row lane / 4 + 8.  (Measured, 16
// warps an SM: such a load every 32 cycles and scheduler; one of 16 columns of a lane's own
// row, the 32x32b shape, every 9.)
__device__ __forceinline__ void tmem_ld_block(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    asm volatile(""
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                   "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
                   "+r"(r[14]), "+r"(r[15]));
}

// f(c, h, r) for the eight blocks of a warp's 32 rows (half h) x 128 columns (32 c), each block's
// load issued before the work on the one before it.
template <class F>
__device__ __forceinline__ void for_blocks(uint32_t tacc, F &&f) {
    uint32_t ra[16], rb[16];
    tmem_ld_block(tacc, ra);
    tmem_ld_wait(ra);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
        uint32_t(&cur)[16] = (b & 1) ? rb : ra;
        uint32_t(&nxt)[16] = (b & 1) ? ra : rb;
        if (b < 7) tmem_ld_block(tacc + ((uint32_t)(((b + 1) & 1) * 16) << 16) + 32 * ((b + 1) >> 1), nxt);
        f(b >> 1, b & 1, cur);
        if (b < 7) tmem_ld_wait(nxt);
    }
}

template <bool RELU>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    uint32_t r;
    if (RELU) asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    else asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// A block (as tmem_ld_block's, values v; RELU: negative ones as zero) as BF16 into rows row0 .. row0 + 15 (a multiple of 8),
// columns 32 c .. 32 c + 31 of a 128-column tile: eight core matrices.
constexpr uint32_t kBlockRow = 16 * 128;   // bytes of eight rows of the tile
template <bool RELU>
__device__ __forceinline__ void st_block(uint32_t tile, int lane, int row0, int c, const float (&v)[16]) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t at = tile + (uint32_t)(row0 / 8 + k) * kBlockRow + (uint32_t)c * 512 + (uint32_t)lane * 16;
        asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(at),
                     "r"(pack2<RELU>(v[2 * k], v[2 * k + 1])), "r"(pack2<RELU>(v[4 + 2 * k], v[5 + 2 * k])),
                     "r"(pack2<RELU>(v[8 + 2 * k], v[9 + 2 * k])), "r"(pack2<RELU>(v[12 + 2 * k], v[13 + 2 * k]))
                     : "memory");
    }
}

}  // namespace tc
}  // namespace tfg
