// What the tcgen05 kernels (ffn_rows.cuh, ffn_q4.cuh, layer_tc.cuh) have in common: the group table's
// entry, unit arithmetic, PTX helpers for TMA tensor copies, mbarriers and the 5th-generation tensor
// cores, and the set of tensor maps of the split-K kernels.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "ffn_stream.cuh"

namespace s2moe {

constexpr int kTcKT = 4;                       // k-tiles (of 64) per unit of the split-K kernels
constexpr int kTcWTile = 128 * 128;            // bytes of one bf16 weight k-tile in shared memory
constexpr int kTcQ4KG = 4;                     // int4: k-tiles per ring stage (a whole unit)
static_assert(kTcQ4KG == kTcKT, "an int4 stage is a whole unit");
constexpr int kTcQ4Packed = 128 * 32;          // bytes of one packed weight k-tile (128 rows x 64 nibbles)
constexpr int kTcQ4Scales = 128 * 16;          // 8 binary16 scales per row: the 256 columns of the unit
constexpr int kTcQ4ACol = 256;                 // int4: TMEM columns 256.. hold the A operand (32 per k-tile), 0..255 the accumulators
#ifndef S2MOE_MAX_STAGES
#define S2MOE_MAX_STAGES 10
#endif
constexpr int kTcMaxStages = S2MOE_MAX_STAGES;
constexpr int kTcMaxSmem = 232448 - 9216;      // dynamic shared memory; the rest is static (unit table, barriers)
constexpr unsigned kTcSpinLimit = 1u << 22;
// Share of the experts in wave 0 of the split-K kernels (by units of the first projection).  The second
// projection of wave 0 is what hides the hand-over of wave 1, the first projection of wave 1 what hides
// that of wave 0.
#ifndef S2MOE_SPLIT_NUM
#define S2MOE_SPLIT_NUM 7
#define S2MOE_SPLIT_DEN 16
#endif
constexpr int kTcSplitNum = S2MOE_SPLIT_NUM, kTcSplitDen = S2MOE_SPLIT_DEN;
constexpr int kTcReady = 512;                  // ws.sync[kTcReady - 8 + w], [kTcReady - 4 + w]: the two counters of wave w

// one active group in shared memory: 32 bytes, so that an entry is two aligned 16-byte reads
// (wider entries were measured: 48 bytes cost 0.7 us per layer)
struct TcGroup {
    unsigned long long mask;   // tokens of the batch bucketed to this group
    int group, T, off, f;      // group id (offloaded experts: device slot), tokens, first slot, inner dim
    int p1, p2;                // first phase-1 / phase-2 unit of the group
};
static_assert(sizeof(TcGroup) == 32, "layout");

// units of a group: phase 1 = 2 matrices x row blocks x k-pieces, phase 2 = row blocks x k-pieces
__host__ __device__ __forceinline__ int tc_kpieces(int K) { return ((K + 63) / 64 + kTcKT - 1) / kTcKT; }
__host__ __device__ __forceinline__ int tc_units1(int f_g, int d) { return 2 * ((f_g + 127) / 128) * tc_kpieces(d); }
__host__ __device__ __forceinline__ int tc_units2(int f_g, int d) { return ((d + 127) / 128) * tc_kpieces(f_g); }

// ---- PTX helpers (tcgen05, TMA tensor copies) ------------------------------------------

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}
// Weight tiles are read once: mark their L2 lines evict-first, so that the stream does not push
// out what is reused across layers (kernel code, bucketing arrays, activations).
__device__ __forceinline__ uint64_t l2_evict_first_policy()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void tma_load_2d_stream(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar,
                                                   uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int x, int y, int z, int w, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}
// (x & mask) | bits in one logic instruction
__device__ __forceinline__ void tc_nibble_pair(uint32_t &out, uint32_t x, uint32_t mask, uint32_t bits)
{
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(out) : "r"(x), "r"(mask), "r"(bits));
}
// non-blocking test of a phase (a thread that serves two rings polls both)
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// one thread of a converged warp: a role that runs in a thread chosen this way issues a tcgen05
// instruction in 39 cycles, in lane 0 behind a comparison it took 55
__device__ __forceinline__ bool tc_elect()
{
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred P;\n\t"
        "elect.sync _|P, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, P;\n\t}"
        : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// A and B in shared memory, the two descriptors given as their 32-bit halves: the shared-memory address sits in
// the low 14 bits of the low word (in units of 16 bytes), so stepping from tile to tile is one
// 32-bit add.  The issuing thread shares its scheduler with busy warps, and every instruction it
// needs per MMA delays the MMA.
__device__ __forceinline__ void tc_mma_bf16_parts(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                                  uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        ".reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, {%7, %7, %7, %7}, p;\n\t"
        "}\n" ::"r"(d_tmem),
        "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(0u)
        : "memory");
}
// A operand in tensor memory (row i of the 128 x 16 tile in lane i, two bf16 per 32-bit column)
__device__ __forceinline__ void tc_mma_bf16_tmem_a(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi,
                                                   uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        ".reg .b64 db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, {%6, %6, %6, %6}, p;\n\t"
        "}\n" ::"r"(d_tmem),
        "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate), "r"(0u)
        : "memory");
}
// 16 consecutive 32-bit columns of this thread's lane
__device__ __forceinline__ void tc_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
          "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tc_ld8(uint32_t taddr, float (&v)[8])
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// the sums of 16 columns and 16 others
__device__ __forceinline__ void tc_ld16_sum(uint32_t taddr, uint32_t taddr2, float (&v)[16])
{
    uint32_t r[16], q[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]), "=r"(q[8]), "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15])
        : "r"(taddr), "r"(taddr2)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]) + __uint_as_float(q[i]);
}
// K-major, 128-byte swizzle: rows 128 bytes apart, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t tc_smem_desc(const void *p)
{
    const uint64_t addr = (uint64_t)((smem_u32(p) >> 4) & 0x3FFFu);
    return addr | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// the same with 8-row groups `sbo` bytes apart
__device__ __forceinline__ uint64_t tc_smem_desc_sbo(const void *p, uint32_t sbo)
{
    const uint64_t addr = (uint64_t)((smem_u32(p) >> 4) & 0x3FFFu);
    return addr | (1ull << 16) | ((uint64_t)(sbo >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ uint32_t tc_idesc(int n)
{
    // D = F32, A = B = BF16, both K-major, N = n, M = 128
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}
__device__ __forceinline__ uint32_t tc_idesc_f16(int n)
{
    // the same with A = B = binary16 (int4 path: the dequantised weights and, because the two
    // operands of an instruction must have one format, the token tiles as well)
    return (1u << 4) | (0u << 7) | (0u << 10) | ((uint32_t)(n >> 3) << 17) | ((128u >> 4) << 24);
}

// Barrier among the four epilogue warps on an mbarrier (count 4), so that the wait is bounded.
__device__ __forceinline__ bool tc_bar(uint64_t *bar, uint32_t &phase, int lane)
{
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
    const bool ok = mbar_wait(bar, phase);
    phase ^= 1u;
    return ok;
}

// counter += 1 with release semantics at GPU scope (one instruction instead of fence + atomic)
__device__ __forceinline__ void tc_red_release(int32_t *counter)
{
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(counter) : "memory");
}

// next slot of the ring; the parity flips on wrap-around
__device__ __forceinline__ void tc_ring_next(int &s, uint32_t &parity, int S)
{
    if (++s == S) { s = 0; parity ^= 1u; }
}

// tensor maps: 0 gate, 1 up, 2 down, 3 sh_gate, 4 sh_up, 5 sh_down, 6 hidden, 7 activations of the
// routed slots, 8 of the shared slots: 3-D {k, slot, hi|lo}, so that one copy of box {64, 16, 2}
// lands the hi tile and, right behind it, the lo tile of 16 slots
// block-int4 weights: 0..5 are the packed matrices (bytes, boxes of four k-tiles), 9..14 their scales
// (binary16), 6 is the (column-permuted) hidden states as {k in tile, row, k-tile} with a box of all rows x kg
// k-tiles, 7 and 8 the activations as {k in tile, slot, k-tile, hi|lo} with a box {64, 8, kg, 2}:
// one copy per stage (per 8 slots) instead of one per k-tile
struct TcMaps {
    CUtensorMap m[15];
};

}  // namespace s2moe
