// PTX wrappers shared by the tcgen05 kernels: mbarriers with bounded waits, TMA tile loads, shared-memory and
// instruction descriptors for tcgen05.mma (kind::f16, K-major operands, 128-byte swizzle), TMEM loads.
#pragma once

#include <cuda.h>

#include <memory>

#include "rkv_common.cuh"

namespace rkv {
namespace sm100 {

constexpr long long kWaitCycles = 4000000000ll;   // default limit of a wait, about two seconds: far beyond any legitimate wait

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// The dynamic shared memory from its first 1024-byte boundary on, by pointer arithmetic: an address that has been through an
// integer is a generic one to the compiler, and every access through it is resolved at run time.
__device__ __forceinline__ uint8_t *align_smem(uint8_t *raw) { return raw + ((1024u - (smem_u32(raw) & 1023u)) & 1023u); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// The same, the thread asleep for up to about 20 us while the phase is not complete: warps that poll take issue slots from
// those that work.
__device__ __forceinline__ bool mbar_try_wait_asleep(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}

// Bounded wait.  Returns false if the block is aborting (this wait ran out of time, or another one did).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, const ErrSink &sink)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long start = clock64();
    while (true) {
        if (mbar_try_wait_asleep(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - start > sink.wait_cycles) break;
    }
    *abort_flag = 1;
    report_timeout(sink);
    return false;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// The tensor map is on its way to where the copies look for it, while the kernel waits for the one before it.
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows 128 bytes apart, 8-row groups
// 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);          // start address
    d |= (uint64_t)1 << 16;                           // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024 >> 4) << 32;                 // stride byte offset between 8-row groups
    d |= (uint64_t)1 << 46;                           // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                           // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: bf16 x bf16 -> fp32, both operands K-major, M x N tile.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accum)
        : "memory");
}
// One 128 x N x 128 product: the eight K = 16 steps of two K-major, 128-byte swizzled bf16 operand tiles (each two
// 16 KB boxes of 64 columns, 1024-byte aligned) into the accumulator at d_tmem, overwriting it.  Everything is in
// one statement so that the issuing thread spends a handful of instructions per step: the descriptors differ
// only in their start-address field (16-byte units; +2 per step, +1024 for the second box).
__device__ __forceinline__ void umma_tile_k128(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc)
{
    const uint32_t a_lo = ((a_addr & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t b_lo = ((b_addr & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);      // stride 1024 B, descriptor version, 128-byte swizzle
    asm volatile(
        "{\n\t.reg .pred p0, p1;\n\t.reg .b64 da, db;\n\t.reg .b32 ta, tb;\n\t"
        "setp.ne.u32 p0, %3, %3;\n\tsetp.eq.u32 p1, %3, %3;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p0;\n\t"
        "add.u32 ta, %1, 2;\n\tadd.u32 tb, %2, 2;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 4;\n\tadd.u32 tb, %2, 4;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 6;\n\tadd.u32 tb, %2, 6;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 1024;\n\tadd.u32 tb, %2, 1024;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 1026;\n\tadd.u32 tb, %2, 1026;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 1028;\n\tadd.u32 tb, %2, 1028;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 1030;\n\tadd.u32 tb, %2, 1030;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc)
        : "memory");
}
// The same product with the second 64-column half of each operand at its own distance from the first (a_half,
// b_half bytes; multiples of 1024): for operand blocks with fewer than 128 rows packed back to back.
__device__ __forceinline__ void umma_tile_k128_halves(uint32_t d_tmem, uint32_t a_addr, uint32_t a_half, uint32_t b_addr,
                                                      uint32_t b_half, uint32_t idesc)
{
    const uint32_t a0 = ((a_addr & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t b0 = ((b_addr & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t a1 = (((a_addr + a_half) & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t b1 = (((b_addr + b_half) & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);      // stride 1024 B, descriptor version, 128-byte swizzle
    asm volatile(
        "{\n\t.reg .pred p0, p1;\n\t.reg .b64 da, db;\n\t.reg .b32 ta, tb;\n\t"
        "setp.ne.u32 p0, %3, %3;\n\tsetp.eq.u32 p1, %3, %3;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p0;\n\t"
        "add.u32 ta, %1, 2;\n\tadd.u32 tb, %2, 2;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 4;\n\tadd.u32 tb, %2, 4;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %1, 6;\n\tadd.u32 tb, %2, 6;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "mov.b64 da, {%5, %3};\n\tmov.b64 db, {%6, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %5, 2;\n\tadd.u32 tb, %6, 2;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %5, 4;\n\tadd.u32 tb, %6, 4;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "add.u32 ta, %5, 6;\n\tadd.u32 tb, %6, 6;\n\tmov.b64 da, {ta, %3};\n\tmov.b64 db, {tb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "}"
        ::"r"(d_tmem), "r"(a0), "r"(b0), "r"(hi), "r"(idesc), "r"(a1), "r"(b1)
        : "memory");
}
// The product of 64-dimensional keys: the four K = 16 steps of one 64-column box of each operand.
__device__ __forceinline__ void umma_tile_k64(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc)
{
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) umma(d_tmem, smem_desc(a_addr + 32 * ks), smem_desc(b_addr + 32 * ks), idesc, ks > 0 ? 1u : 0u);
}
// Instruction descriptor of kind::f8f6f4: E4M3 x E4M3 -> fp32, both operands K-major, M x N tile.
__host__ __device__ constexpr uint32_t instr_desc_codes(int M, int N) { return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24); }
// The product of keys whose rows are 128 bytes: 64 dimensions in bf16, or 128 E4M3 codes (four K = 32 steps of the 8-bit kind; products
// of codes are exact, the accumulator is the same fp32 one that bf16 steps add to).
template <bool kCodes>
__device__ __forceinline__ void umma_tile_row128(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc)
{
    if (!kCodes) {
        umma_tile_k64(d_tmem, a_addr, b_addr, idesc);
        return;
    }
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(smem_desc(a_addr + 32 * ks)), "l"(smem_desc(b_addr + 32 * ks)), "r"(idesc), "r"(ks)
            : "memory");
}
// One more K = 16 step onto the accumulator at d_tmem: both operands are 128 rows x 16 bf16 (32-byte rows, 32-byte
// swizzle, 8-row groups 256 bytes apart, 256-byte aligned).
__device__ __forceinline__ void umma_k16_sw32(uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t idesc)
{
    const uint32_t a_lo = ((a_addr & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t b_lo = ((b_addr & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t hi = (256u >> 4) | (1u << 14) | (6u << 29);       // stride 256 B, descriptor version, 32-byte swizzle
    asm volatile(
        "{\n\t.reg .pred p1;\n\t.reg .b64 da, db;\n\t"
        "setp.eq.u32 p1, %3, %3;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p1;\n\t"
        "}"
        ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_wait4(uint32_t (&r)[4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]) :: "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld1(uint32_t taddr, uint32_t &r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
}
// Wait for the thread's TMEM loads; the loaded registers pass through the statement so that nothing that uses
// them can be scheduled ahead of it.
__device__ __forceinline__ void tmem_wait8(uint32_t (&r)[8])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
                 :: "memory");
}
__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]),
                   "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :: "memory");
}

// Entry `at` of 32 registers, by a select tree
__device__ __forceinline__ float pick32(const uint32_t (&g)[32], int at)
{
    uint32_t t16[16], t8[8], t4[4];
#pragma unroll
    for (int c = 0; c < 16; ++c) t16[c] = (at & 16) ? g[16 + c] : g[c];
#pragma unroll
    for (int c = 0; c < 8; ++c) t8[c] = (at & 8) ? t16[8 + c] : t16[c];
#pragma unroll
    for (int c = 0; c < 4; ++c) t4[c] = (at & 4) ? t8[4 + c] : t8[c];
    const uint32_t u0 = (at & 2) ? t4[2] : t4[0], u1 = (at & 2) ? t4[3] : t4[1];
    return __uint_as_float((at & 1) ? u1 : u0);
}
// max(a, b, c), NaN operands ignored
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}



// ---- host side: tensor maps -------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) != cudaSuccess ||
            qres != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(sym);
    }();
    return fn;
}

// A tensor map is a function of what is described here, and a decode loop asks for the same few hundred over and over
// (three per attention call): the thread's last ones are kept.  Encoding takes 0.3 us.
struct MapKey {
    const void *base;
    uint64_t rows;
    uint32_t type, dim, row_bytes, box_x, box_y, swizzle;
    bool operator==(const MapKey &o) const
    {
        return base == o.base && rows == o.rows && type == o.type && dim == o.dim && row_bytes == o.row_bytes && box_x == o.box_x &&
               box_y == o.box_y && swizzle == o.swizzle;
    }
};
inline bool encode_map(CUtensorMap *map, const MapKey &k)
{
    constexpr int kKept = 512;
    struct Kept {
        MapKey key;
        CUtensorMap map;
    };
    static thread_local std::unique_ptr<Kept[]> kept;
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    if (!kept) kept.reset(new Kept[kKept]());
    uint64_t h = (reinterpret_cast<uintptr_t>(k.base) >> 8) * 0x9E3779B97F4A7C15ull + k.rows * 0xC2B2AE3D27D4EB4Full + k.box_y * 31u + k.box_x;
    Kept &slot = kept[(h >> 40) % kKept];
    if (!(slot.key == k)) {
        const cuuint64_t dims[2] = {(cuuint64_t)k.dim, (cuuint64_t)k.rows};
        const cuuint64_t strides[1] = {(cuuint64_t)k.row_bytes};
        const cuuint32_t box[2] = {k.box_x, k.box_y};
        const cuuint32_t estr[2] = {1u, 1u};
        slot.key.base = nullptr;
        if (fn(&slot.map, (CUtensorMapDataType)k.type, 2, const_cast<void *>(k.base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, (CUtensorMapSwizzle)k.swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return false;
        slot.key = k;
    }
    *map = slot.map;
    return true;
}

// Rows of the 2-D view of k_cache: all heads' rows, or all pages of a paged pool.
inline uint64_t key_rows_total(const Params &p)
{
    return p.block_table ? (uint64_t)p.pool_pages * kTile : (uint64_t)p.batch * p.hkv * p.cap;
}

// 2-D bf16 view [rows][dim] of a contiguous tensor (dim a multiple of 64), boxes of box_rows x 64 elements, 128-byte
// swizzle, out-of-range rows read as zero.
inline bool make_map_rows(CUtensorMap *map, const void *base, uint64_t rows, int dim, uint32_t box_rows)
{
    return encode_map(map, MapKey{base, rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (uint32_t)dim, (uint32_t)dim * 2, 64u, box_rows,
                                  CU_TENSOR_MAP_SWIZZLE_128B});
}
inline bool make_map(CUtensorMap *map, const void *base, uint64_t rows, uint32_t box_rows)
{
    return make_map_rows(map, base, rows, kHeadDim, box_rows);
}

// 2-D view [rows][128 bytes] of a cache whose rows are 128 bytes long -- E4M3 codes of 128 dimensions, or bf16 keys of 64
// dimensions --, boxes of 128 rows, 128-byte swizzle, out-of-range rows read as zero.
inline bool make_map_row128(CUtensorMap *map, const void *base, uint64_t rows, bool codes)
{
    const uint32_t dim = codes ? 128u : 64u;
    return encode_map(map, MapKey{base, rows, (uint32_t)(codes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16), dim, 128u,
                                  dim, (uint32_t)kTile, CU_TENSOR_MAP_SWIZZLE_128B});
}

// The K = 16 slices of key rows: stored as [rows][8] bf16 (16 bytes), read as boxes of 128 rows x 16 elements whose second
// half, beyond the view, comes as zeros; 32-byte swizzle.
constexpr int kSliceElems = 8;
inline bool make_map_k16(CUtensorMap *map, const void *base, uint64_t rows)
{
    return encode_map(map, MapKey{base, rows, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (uint32_t)kSliceElems, kSliceElems * 2u, 16u, (uint32_t)kTile,
                                  CU_TENSOR_MAP_SWIZZLE_32B});
}

}  // namespace sm100

// The key sum of a head as the first scoring pass reads it beside 8-bit keys: 16 rows of 128 codes, the first kSumParts of which are
// s 2^e in parts that are a 16th of the one before each; then 2^-e.  (The rows take the first half of the head's room for bf16 rows.)
constexpr int kSumParts = 7, kSumHeadBytes = 16 * kHeadDim * 2, kSumScaleAt = 16 * kHeadDim;

// first scoring pass of the two-pass tensor-core route (its own file); the maps are built by the caller
cudaError_t launch_scores_pass1_sm100(const Params &p, cudaStream_t s, const CUtensorMap &map_k, const CUtensorMap &map_hs,
                                      const CUtensorMap &map_ns, const CUtensorMap &map_ts);

// symmetric route of the second pass (its own file)
cudaError_t launch_scores_dense_sm100(const Params &p, cudaStream_t s, const CUtensorMap &map_k, const CUtensorMap &map_ns);
cudaError_t launch_dense_finish(const Params &p, cudaStream_t s);

}  // namespace rkv
