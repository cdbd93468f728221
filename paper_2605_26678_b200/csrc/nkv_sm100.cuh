// sm_100a building blocks shared by the tensor-core key pass: mbarriers with bounded waits, tiled TMA
// loads, tcgen05 (UMMA) descriptors and issue, tensor-memory allocation and loads, packed fp32 pairs.
#pragma once

#include <cuda.h>

#include "nkv_common.cuh"

namespace nkv {

// Tensor map of bf16 or fp16 keys [G][H][N][d] for boxes of 64 columns x box_rows rows, 128-byte swizzle (host).
cudaError_t encode_key_map(const TensorView& K, int dtype, int G, int box_rows, CUtensorMap* out);

namespace sm100 {

constexpr uint32_t kSpinLimit = 1u << 22;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// ---------------------------------------------------------------------------- mbarriers
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bounded wait: false (after recording where) if the phase never completes.  The polling loop is one
// out-of-line function: the roles of a kernel run side by side and share the instruction cache, and a
// wait that finds its phase complete at the first look costs one instruction.
static __device__ __noinline__ bool mbar_wait_poll(uint64_t* bar, uint32_t parity, int* status, int where,
                                                  uint32_t limit = kSpinLimit) {
    for (uint32_t spin = 0; spin < limit; ++spin) {
        if (mbar_try_wait(bar, parity)) return true;
        if (spin >= 4) __nanosleep(64);   // leave the issue slots to the warps that have work
    }
    set_status(status, NKV_ERR_TIMEOUT, where);
    return false;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* status, int where) {
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_poll(bar, parity, status, where);
}

// A whole warp waits; false for all of its lanes when any of them gave up.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, int* status, int where) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, status, where));
}

// The same for two barriers, whose first looks overlap (a wait that finds its phase complete takes 150 cycles beside busy warps).
__device__ __forceinline__ bool warp_wait2(uint64_t* a, uint32_t parity_a, uint64_t* b, uint32_t parity_b, int* status, int where) {
    const bool oa = mbar_try_wait(a, parity_a), ob = mbar_try_wait(b, parity_b);
    if (__all_sync(0xffffffffu, oa && ob)) return true;
    return warp_wait(a, parity_a, status, where) && warp_wait(b, parity_b, status, where + 1);
}

// Named barrier over `count` threads that also ORs a predicate over them.
__device__ __forceinline__ bool bar_or(int id, int count, bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.or.pred p, %2, %3, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred), "r"(id), "r"(count)
        : "memory");
    return r != 0;
}

// ---------------------------------------------------------------------------- TMA
__device__ __forceinline__ uint64_t l2_evict_normal_policy() {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}
// Keys are read once per pass and are far larger than L2: marking their lines "evict first" leaves L2 to what is read again
// (anchors, weights, the scores written for the next kernel).
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t policy;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    return policy;
}
// One box of a 4-d tiled tensor map into shared memory, with an L2 cache policy; c0 is the innermost coordinate (c0 * element
// size must be a multiple of 16 bytes).  Rows outside the tensor arrive as zeros.
__device__ __forceinline__ void tma_load_4d(void* dst_smem, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, "
        "%4, %5}], [%6], %7;" ::"r"(smem_addr(dst_smem)),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_addr(bar)), "l"(policy)
        : "memory");
}

// ---------------------------------------------------------------------------- tensor memory
__device__ __forceinline__ void tmem_alloc(uint32_t* slot_smem, uint32_t cols) {   // whole warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot_smem)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {      // whole warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive fp32 columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// kCount groups of 8 consecutive fp32 columns of this warp's 32 lanes, kApart columns apart, and the wait for them.
template <int kCount, int kApart>
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (*v)[8]) {
    static_assert(kCount == 2 || kCount == 4, "two or four groups");
    uint32_t r[4][8];
#pragma unroll
    for (int k = 0; k < kCount; ++k)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[k][0]), "=r"(r[k][1]), "=r"(r[k][2]), "=r"(r[k][3]), "=r"(r[k][4]), "=r"(r[k][5]), "=r"(r[k][6]), "=r"(r[k][7])
                     : "r"(taddr + (uint32_t)(k * kApart))
                     : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < kCount; ++k) {   // no use is scheduled above the wait
        asm volatile("" : "+r"(r[k][0]), "+r"(r[k][1]), "+r"(r[k][2]), "+r"(r[k][3]), "+r"(r[k][4]), "+r"(r[k][5]), "+r"(r[k][6]), "+r"(r[k][7]));
#pragma unroll
        for (int i = 0; i < 8; ++i) v[k][i] = __uint_as_float(r[k][i]);
    }
}

// Wait for the tensor-memory loads issued so far; a and b (16 values each) are the registers the loads
// fill, named here so that no use of them is scheduled above the wait.
__device__ __forceinline__ void tmem_wait_ld(float* a, float* b) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]), "+f"(a[8]), "+f"(a[9]), "+f"(a[10]), "+f"(a[11]), "+f"(a[12]), "+f"(a[13]), "+f"(a[14]), "+f"(a[15]), "+f"(b[0]), "+f"(b[1]), "+f"(b[2]), "+f"(b[3]), "+f"(b[4]), "+f"(b[5]), "+f"(b[6]), "+f"(b[7]), "+f"(b[8]), "+f"(b[9]), "+f"(b[10]), "+f"(b[11]), "+f"(b[12]), "+f"(b[13]), "+f"(b[14]), "+f"(b[15])
                 :
                 : "memory");
}

__device__ __forceinline__ void tmem_wait_ld(float* a) {   // the same for one group of 16 values
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]), "+f"(a[4]), "+f"(a[5]), "+f"(a[6]), "+f"(a[7]), "+f"(a[8]), "+f"(a[9]), "+f"(a[10]), "+f"(a[11]), "+f"(a[12]), "+f"(a[13]), "+f"(a[14]), "+f"(a[15])
                 :
                 : "memory");
}

// 16 lanes x 32 fp32 columns in the accumulator-fragment layout: lane base = the lane field of taddr (a multiple
// of 16 inside the warp's quarter); thread t receives in v[4 k + 2 j + e] the element of row t / 4 + 8 j and column
// 8 k + 2 (t % 4) + e, so four threads share a row and a thread sees the same eight columns of four rows in two loads.
__device__ __forceinline__ void tmem_ld_frag32(uint32_t taddr, float* v) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// ---------------------------------------------------------------------------- UMMA (tcgen05.mma)
// Shared-memory operand descriptor for a K-major tile of 16-bit numbers stored as 8-row x 128-byte swizzle atoms
// (the layout a 128B-swizzled TMA box of 64 such columns produces): consecutive 8-row groups are
// 1024 bytes apart.  `addr` is the shared address of the first row at the wanted K offset (a
// multiple of 32 bytes inside the 128-byte atom row); the tile base must be 1024-byte aligned.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3ffffu) >> 4);   // start address
    d |= (uint64_t)1 << 16;                     // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                     // descriptor version of sm_100
    d |= (uint64_t)2 << 61;                     // 128-byte swizzle
    return d;
}
// The same for an operand that lies in memory with its rows along K, 64 columns (M or N) per atom: `addr` is the first atom
// of the wanted K offset (16 rows per K step, so a multiple of 2048 bytes), the next 64 columns are `next64` bytes on.
__device__ __forceinline__ uint64_t umma_desc_sw128_mn(uint32_t addr, uint32_t next64) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3ffffu) >> 4);    // start address
    d |= (uint64_t)(next64 >> 4) << 16;         // leading byte offset: between atoms along M or N
    d |= (uint64_t)(1024 >> 4) << 32;           // stride byte offset: between 8-row groups along K
    d |= (uint64_t)1 << 46;                     // descriptor version of sm_100
    d |= (uint64_t)2 << 61;                     // 128-byte swizzle
    return d;
}
constexpr uint32_t kTransposeA = 1u << 15;      // instruction descriptor: A lies that way
// Instruction descriptor: bf16 x bf16 or fp16 x fp16 -> fp32, both operands K-major, tile M x N.
template <typename T> constexpr uint32_t kOperandType = 1u;            // bf16
template <> inline constexpr uint32_t kOperandType<__half> = 0u;
template <typename T>
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N) {
    return (1u << 4) | (kOperandType<T> << 7) | (kOperandType<T> << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// D[tmem] (+)= A[smem] * B[smem]^T.  Products and commits are issued by a whole warp in step, of which one elected lane
// (always the same) counts: the operands then stay in uniform registers.  From a thread that has left its warp behind a
// product took 61 cycles to issue, on an idle SM, and up to 270 beside busy warps; so it takes 6 for a batch of eight, and
// the tensor core sets the pace (97 cycles for M = 128, N = 192, K = 16; 33 for N = 16).
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          bool accumulate) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %4, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"((uint32_t)accumulate)
        : "memory");
}
// The barrier gets one arrival once every MMA issued so far by this warp has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile(
        "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_addr(bar))
        : "memory");
}
// Products already issued keep reading shared memory and writing tensor memory: a warp that gives up waits (bounded)
// for them before the CTA frees both.
static __device__ __noinline__ void umma_drain(uint64_t* bar) {
    __syncwarp();
    umma_commit(bar);
    for (uint32_t spin = 0; spin < (1u << 16) && !mbar_try_wait(bar, 0); ++spin) __nanosleep(256);
    __syncwarp();
}

// ---------------------------------------------------------------------------- packed fp32 pairs
struct F2 {
    unsigned long long v;
};
__device__ __forceinline__ F2 pack2(float a, float b) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(F2 x, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ float hsum2(F2 x) {
    float a, b;
    unpack2(x, a, b);
    return a + b;
}
// eight 16-bit values of a 16-byte chunk as four fp32 pairs
template <typename T> __device__ __forceinline__ void unpack8(const uint4& q, F2* p);
template <> __device__ __forceinline__ void unpack8<__nv_bfloat16>(const uint4& q, F2* p) {
    p[0] = pack2(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u));
    p[1] = pack2(__uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
    p[2] = pack2(__uint_as_float(q.z << 16), __uint_as_float(q.z & 0xffff0000u));
    p[3] = pack2(__uint_as_float(q.w << 16), __uint_as_float(q.w & 0xffff0000u));
}
template <> __device__ __forceinline__ void unpack8<__half>(const uint4& q, F2* p) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
        p[j] = pack2(f.x, f.y);
    }
}

}  // namespace sm100
}  // namespace nkv
