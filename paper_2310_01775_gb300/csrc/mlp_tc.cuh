// tcgen05 / TMA pieces of the BF16 MLP kernels (mlp.cu, surrogate_mlp.cu):
// tensor memory, descriptors, the K-major tile layout described in mlp.cu, and
// the activations.  Internal linkage: each translation unit gets its own copy.
#pragma once

#include <cstdint>

#include "async_copy.cuh"
#include "mlp.cuh"

namespace stamp {
namespace mlp {
namespace {

using async::fence_async_shared;
using async::kWaitLimit;
using async::mbar_expect_tx;
using async::mbar_init;
using async::mbar_try_wait;
using async::smem_u32;
using async::tma_load_1d;

// ---------------- tcgen05 ---------------------------------------------------
__device__ __forceinline__ void tmem_alloc(unsigned* slot, unsigned ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(unsigned taddr, unsigned ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// Shared-memory matrix descriptor: start address, LBO, SBO (all >> 4), the
// descriptor version bits (0b01 at bit 46), no swizzle.
__device__ __forceinline__ uint64_t smem_desc(const void* p, unsigned lbo, unsigned sbo) {
    const uint64_t a = (smem_u32(p) & 0x3FFFFu) >> 4;
    return a | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) | ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) |
           (1ull << 46);
}
// Instruction descriptor, kind::f16: D = F32 (bits 4-5 = 1), A = B = BF16
// (bits 7-9 and 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(unsigned tmem_d, uint64_t adesc, uint64_t bdesc,
                                        uint32_t idesc, unsigned accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar))
                 : "memory");
}
// 32 consecutive FP32 columns of this warp's 32 TMEM lanes (one lane per thread).
__device__ __forceinline__ void tmem_ld32(unsigned taddr, float (&v)[32]) {
    unsigned r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld16(unsigned taddr, float (&v)[16]) {
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld8(unsigned taddr, float (&v)[8]) {
    unsigned r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                   "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ unsigned pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const unsigned*>(&h);
}
// z sigmoid(z) with the fast reciprocal (its error, a few float ulps, is far
// below the bfloat16 rounding of the result)
__device__ __forceinline__ float silu(float z) { return __fdividef(z, 1.f + __expf(-z)); }

// Byte offset of element (row, col) in a K-major core-matrix tile of K columns.
__host__ __device__ __forceinline__ unsigned tile_off(int row, int col, int K) {
    return (unsigned)((row >> 3) * (K / 8) * 128 + (col >> 3) * 128 + (row & 7) * 16 + (col & 7) * 2);
}

constexpr int kRows = 128;                        // rows per tile (MMA M)

// D (128 x N) = A (128 x K) . B (N x K)^T, K-major operands; K is 16, 32 or 256.
// A slice of 16 columns is 256 bytes on in both: 16 in a descriptor's address.
__device__ __forceinline__ void mma_tile(unsigned tmem, const unsigned char* A, const unsigned char* B,
                                         int K, int N) {
    const uint32_t idesc = idesc_bf16(kRows, N);
    const uint64_t da = smem_desc(A, 128, (K / 8) * 128), db = smem_desc(B, 128, (K / 8) * 128);
    mma_bf16(tmem, da, db, idesc, 0u);
    if (K >= 32) mma_bf16(tmem, da + 16, db + 16, idesc, 1u);
    if (K >= 256)
#pragma unroll
        for (int kk = 2; kk < 16; ++kk) mma_bf16(tmem, da + 16 * kk, db + 16 * kk, idesc, 1u);
}
// 16 warps: warp w reads TMEM lane quarter w % 4 (rows 32 (w % 4) ...) and
// takes part w / 4 of the four column parts in the epilogues
constexpr int kThreads = 512;
constexpr int kParts = kThreads / 128;
constexpr unsigned kTmemCols = 256;
constexpr unsigned kActBytes = kRows * kHidden * 2;            // 64 KB
constexpr unsigned kWBytes = kHidden * kHidden * 2;            // 128 KB
constexpr unsigned kInBytes = kRows * kIn * 2;                 // 8 KB per input tile

struct FwdSmem {
    alignas(128) unsigned char act[kActBytes];
    alignas(128) unsigned char w[kWBytes];
    uint64_t tma_bar, mma_bar;
    unsigned tmem_slot;
};

// Layer l: K (inputs), N (outputs), packed forward weight bytes.
__host__ __device__ constexpr int layer_k(int l) { return l == 0 ? kIn : kHidden; }
__host__ __device__ constexpr int layer_n(int l) { return l == 3 ? kOut : kHidden; }

__device__ __forceinline__ float silu_grad(float z) {
    const float sg = __fdividef(1.f, 1.f + __expf(-z));
    return sg * (1.f + z * (1.f - sg));
}
__device__ __forceinline__ float bf_lo(unsigned w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(unsigned w) { return __uint_as_float(w & 0xFFFF0000u); }

}  // namespace
}  // namespace mlp
}  // namespace stamp
