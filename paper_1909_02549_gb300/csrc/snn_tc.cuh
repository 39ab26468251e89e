// Blackwell (sm_103a) building blocks of the tensor-core kernels: mbarriers,
// TMA tile loads, shared-memory matrix descriptors, tcgen05 instruction
// descriptors and tensor-memory loads, and the host encoder of TMA tensor maps.
// Shared by the recurrent network's dense form and the main network's tensor
// form.
//
// Operand convention: every operand is a row-major [rows][K] bfloat16 matrix
// ("K-major": K contiguous), loaded in tiles of 64 K-elements (128 bytes) x
// box_rows rows with the 128-byte swizzle, so one tile row is one swizzled
// 128-byte line and eight rows form a 1024-byte swizzle atom.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace snn {
namespace tc {

constexpr int KB = 64;                                    // K-elements per tile (128 bytes of bf16)

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(su32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(su32(b)) : "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(su32(b)), "r"(parity) : "memory");
    return ok != 0;
}
// Waits for the phase with the given parity to complete; false once limit_ns
// of %globaltimer have passed (the caller then reports an error and leaves).
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, unsigned long long limit_ns) {
    if (mbar_try(b, parity)) return true;
    const unsigned long long t0 = now_ns();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try(b, parity)) return true;
        if (now_ns() - t0 > limit_ns) return false;
    }
}
// The same with 64 tries before the timer is first read, which costs far more
// than a try: for waits that are short (the recurrent gather's ring).  Where the
// wait is long and other warps work meanwhile, as in the products' epilogues, the
// plain one is faster (784->626, B = 626 in the tensor form: 2.4 % over a run).
__device__ __forceinline__ bool mbar_wait_short(uint64_t* b, uint32_t parity, unsigned long long limit_ns) {
    for (int i = 0; i < 64; ++i)
        if (mbar_try(b, parity)) return true;
    return mbar_wait(b, parity, limit_ns);
}
// True in one lane of a converged warp, always the same one.  Under a branch on it
// the compiler knows that a single lane runs, so the operands of copies and products
// go to the uniform registers these instructions take with no work per lane.  With a
// branch on lane == 0 the issue of a stage's four products and their commit took 400
// cycles, more than the products themselves below 192 columns: with this one
// 1024->4096, B = 64 went from 38.6 to 28.4 us a step (recurrent), B = 4096 from 146
// to 140, 784->6400, B = 1024 from 176 to 151 (learning, tensor form, T = 250).
__device__ __forceinline__ bool elect_one() {
    uint32_t one;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(one));
    return one != 0u;
}
// One 2D tile of a tensor map into shared memory; completion is counted in
// bytes on the mbarrier.  c0 is the K coordinate (a multiple of 64 here, so
// 128-byte aligned), c1 the row.
__device__ __forceinline__ void tma_2d(void* dst, const CUtensorMap* tm, int c0, int c1, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3}], [%4];"
                 :: "r"(su32(dst)), "l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(su32(bar)) : "memory");
}
// The same for a pair of CTAs (cta_group::2): into this CTA's shared memory, the
// bytes counted on the mbarrier at cluster address `bar`, which may be the peer's.
__device__ __forceinline__ void tma_2d_pair(void* dst, const CUtensorMap* tm, int c0, int c1, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%2, %3}], [%4];"
                 :: "r"(su32(dst)), "l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(bar) : "memory");
}
// An arrival on the mbarrier at a cluster address.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(bar) : "memory");
}
// The pair's products issued before have finished: an arrival on this mbarrier in
// both CTAs.
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 :: "r"(su32(bar)), "h"((uint16_t)3) : "memory");
}
// 16-byte asynchronous copies (through L2 only); cp_async_arrive makes the
// mbarrier's current phase wait for the calling thread's copies so far (one
// arrival of its expected count).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(src));
}
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" :: "r"(su32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// Shared-memory matrix descriptor of a K-major tile with 128-byte rows and the
// 128-byte swizzle: groups of 8 rows 1024 bytes apart (SBO), version 1,
// swizzle mode 2.  Advancing K by 16 elements adds 32 bytes (2 in the address
// field) inside the swizzled row.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
// Instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator, bfloat16
// A and B, both K-major, M = 128, N = n (a multiple of 16, 16..256).
__host__ __device__ constexpr uint32_t idesc_bf16(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
// D (tensor memory) [+]= A * B^T for one K = 16 slice; acc = 0 overwrites D.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 :: "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
// The mbarrier completes once every MMA this thread issued before has finished.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :: "r"(su32(bar)) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Allocates ncols tensor-memory columns (a power of two >= 32) for the CTA;
// one whole warp calls it, and the address lands in *slot (shared memory).
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 :: "r"(su32(slot)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(taddr), "r"(ncols) : "memory");
}
// 16 consecutive 32-bit accumulator columns of the warp's 32 lanes (lane =
// row); the wait is in the same statement, so no register is read early.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}

// In a launch with programmatic serialization: waits until the launch before has
// finished and its writes are visible, then lets the launch after begin (its blocks
// take their places as this one's leave, and wait in turn).
__device__ __forceinline__ void after_previous_launch() {
    asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
}

// Thread-block clusters: every thread of every CTA of the cluster arrives and
// waits (release / acquire: shared-memory writes before the barrier are seen
// by other CTAs' reads after it).  Without .aligned, so a warp need not be
// converged.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// The address in CTA `rank`'s shared memory of this CTA's shared address.
__device__ __forceinline__ uint32_t cluster_map(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

// Host: a [rows][K] bfloat16 matrix (row pitch K elements, K a multiple of 8)
// as a tensor map of 64 x box_rows tiles with the 128-byte swizzle; rows and K
// past the end read as zero.  False if the driver's encoder is unavailable or
// refuses the map.
bool encode_bf16_map(CUtensorMap* m, const void* base, int rows, int K, int box_rows);

}  // namespace tc
}  // namespace snn
