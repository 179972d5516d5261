// tcgen05 expert kernel for bf16 weights (kernel plan 3): the first projection is cut by ROWS of the
// inner dimension, so that no partial sum of it ever leaves a CTA.
//
// Bound: HBM (T flop per weight byte).  Per layer the kernel moves U * 3 * d * f * 2 bytes once;
// everything below serves one goal, a weight stream that never stops.
//
//   first projection   a task is up to 64 consecutive rows of the inner dimension of one group (expert),
//                      over the WHOLE contraction: rows of W_gate and of W_up arrive interleaved in
//                      groups of eight (one 5-D tensor map over both matrices), so that one MMA of
//                      128 weight rows holds 64 gate and 64 up rows and lane l of the accumulator has
//                      its partner in lane l ^ 8 of the same warp.  The epilogue forms silu(g) * u in
//                      registers and stores it once, as bf16 hi + lo parts.
//   second projection  a task is a run of k-tiles of one 128-row block of W_down; partial sums of a
//                      row block cut by a CTA boundary meet in y (red.add).
//
// Against cutting both projections along the contraction (units of 128 rows x 256 columns, partial
// pre-activations reduced to memory, converted between the projections by a second grid-wide round)
// this saves the pre-activation traffic, its clearing, the conversion and one of two grid-wide rounds
// per wave.  The boxes are chosen by a streaming probe without any arithmetic (16 experts of 2048 x
// 1024, us per layer): contiguous bulk copies 33.0, this split 32.7, boxes of 8 or 16 rows of one
// matrix and two k-tiles 43 to 51, W_down cut by columns (which would need no hand-over) 38 to 40.
//
// The groups are cut into waves; the order of a CTA's work is the first projection of all waves, then
// the second projection of all waves, every part one contiguous share, so that the hand-over of a
// wave hides behind the work in between.  The hand-over is one counter per wave: the epilogue warps of
// a CTA arrive (release) when their activations of the wave are stored, a watcher warp polls it and
// opens the wave's token tiles to the producer.
//
// Early start: see route.cuh.  The kernel is resident while the routing kernel still runs (its blocks
// are small enough to share the SMs), even before the layer in front has ended.  It streams the weights
// of the shared experts' first projection at once; as soon as the router's logits are there, and beside
// the gating, the first projection of the top_k experts (RwPlan::n_early) of largest aggregated importance g_e (Eq. 4),
// which are nearly always selected: over the shapes of the workloads, 1 to 64 tokens, noise 0.1 to 1, with
// and without the bias, at most 0.1 of them is not.  An expert that is not has been read for nothing: it
// gets no tokens and no second projection.  The first projection of all others follows when the
// selection is known, the second projection when warps 6..9 have built the tables from the finished
// gating.  Early results wait in tensor memory (two or four tasks) for the token lists.  Nothing but
// weights is read before the routing kernel says that its own inputs are there, and no weights either in
// the first layer of a call: what is in front of that in the stream is the caller's and may be writing them.
// (In a later layer the library's own kernels are in front, and those of the first layer have waited.)
//
// Warp roles (352 threads): 0 TMA producer, 1 MMA issuer (owns the TMEM allocation), 2..5 and 6..9 two
// epilogue sets that take alternate tasks (6..9 build the tables first), 10 watcher (early experts,
// selection and the tasks of the first projection, then the wave counters).  The single-thread roles run
// in a thread chosen by elect.sync: measured on B200, an MMA of 128 x 16 x 16 then issues every 39 cycles
// against 55 from a `lane == 0` branch (the tensor core itself needs 32 to read the 4 KiB of
// weights), which is why one issuer is enough.
// Measured on one GPU, us per layer, split-K kernel / this one when it replaced it: OLMoE shape 1 token 41.1 / 35.5,
// 8 tokens 50.9 / 46.7, Qwen1.5-MoE shape 16 tokens 54.9 / 46.7, DeepSeek-V2-Lite shape 16 tokens 59.5 / 54.5,
// 64 tokens 131.5 / 130.5, 128 wide experts 8 tokens 89.7 / 75.4.
// The tensor core truncates when it adds to an accumulator, so the k-tiles of a task go in turn to several
// accumulators (chains) that the epilogue adds: eight in the first projection up to 16 tokens, four above, and as
// many as their columns hold in the second one.  Relative 2-norm of the error against float64, two / four /
// eight chains in the first projection: OLMoE shape 1 token 3.2e-6 / 2.6e-6 / 2.4e-6, 8 tokens 3.4e-6 / 2.7e-6 /
// 2.5e-6, 64 tokens 3.8e-6 / 2.8e-6 / -, 128 narrow experts 13 tokens 3.5e-6 / 2.7e-6 / 2.5e-6, 128 wide ones
// 8 tokens 4.5e-6 / 3.0e-6 / 2.6e-6 (one chain, OLMoE shape 8 tokens: 5.3e-6); the split-K kernel had 2.5e-6,
// 2.8e-6, 3.1e-6, 2.7e-6 and 4.0e-6.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "tc_common.cuh"

namespace s2moe {

constexpr int kRwThreads = 352;
constexpr int kRwMaxStages = 8;
constexpr int kRwMaxAcc = 4;
constexpr int kRwWBytes = 32768;               // weight bytes of a stage: 8 row pairs x 2 k-tiles, or a 128-row block x 2 k-tiles
constexpr int kRwStaticSmem = 2048;            // static shared memory at most (barriers, lots, ids)
constexpr int kRwMaxSmem = 232448 - kRwStaticSmem;
constexpr int kRwSets = 2;                     // epilogue sets
constexpr int kRwMaxWaves = 2;
constexpr int kRwLots2 = kRwMaxWaves + 1;      // lots of the second projection: wave 0, shared experts, wave 1
constexpr int kRwLevels = 3;                   // task lists: shared experts, early list, all experts, second projection

// Division of 0 <= n < 2^31 by a launch constant d: with L = ceil(log2 d) and m = floor(2^(31 + L) / d) + 1, which
// has 32 bits, n / d is n * m >> (31 + L): m * d exceeds 2^(31 + L) by at most 2^L, which n times is less than 2^(31 + L).
struct RwDiv {
    unsigned d, m;
    int s;               // L - 1
};
inline RwDiv rw_div_make(unsigned d)
{
    int L = 0;
    while (L < 31 && (1u << L) < d) ++L;
    return d <= 1 ? RwDiv{d, 0u, 0} : RwDiv{d, (unsigned)((1ull << (31 + L)) / d + 1), L - 1};
}
__device__ __forceinline__ int rw_div(int n, const RwDiv &v) { return v.d <= 1 ? n : (int)(__umulhi((unsigned)n, v.m) >> v.s); }

struct RwPlan {
    int feasible;
    int n_cta;
    int stages, stage_bytes;
    int n1;              // N of the first projection's MMAs: tokens padded to 16
    int xr;              // rows of a resident hidden-state tile (8 up to 8 tokens: the MMA's other 8 columns are not read)
    int x_bytes;         // > 0: the hidden states stay resident in shared memory
    int c1;              // chains of a first-projection task
    int acc_cols, n_acc, tmem_cols;
    int max_tasks;
    int tab_bytes;
    int smem_bytes;
    int early, n_early;           // early start; its experts
    int one_rows;                 // second-projection tasks of that many slots take one k-tile per stage (0: none)
    int split16;         // where wave 1 begins, in 16ths of the first projection
    RwDiv gf, gs, tf, ts, kr, ks, rb, p;   // row groups and tasks of a routed / shared expert, P2 units of their row blocks, row blocks, CTAs
};

struct RwArgs {
    Shape sh;
    Workspace ws;
    RwPlan plan;
    float *y;
    __nv_bfloat16 *act_hi, *act_lo;
    int B;
    int first;           // first layer of a call: the kernel in front in the stream may be the caller's and write weights
    int mode;            // bit 0 / 1: in the gate|up maps of the routed / shared experts W_up comes first;
                         // bit 2 / 3: the two matrices are too far apart for one map (make_gateup_maps)
};

// tensor maps: 0..2 gate|up of the routed experts with 1, 2, 4 row pairs per box, 3..5 of the shared
// experts (or, RwArgs::mode bit 2 / 3, gate and up by themselves with 8 rows per box); 6 / 7 W_down
// routed / shared (64 x 128), 8 / 9 the same with 64 rows (last block of a ragged d); 10 hidden
// states; 11..14 activations of the routed slots (8, 16, 32, 64 rows, hi and lo), 15..18 shared
struct RwMaps {
    CUtensorMap m[19];
};

// one task in shared memory, read as two 16-byte words
struct RwTask {
    int flags;           // bit 0: second projection, 1: shared, 2..3: wave, 4: half row block; >> 8: row pairs or token rows
    int x0;              // P1: first row group in the gate|up map; P2: first row of W_down
    int k;               // P2: first k-tile | end << 16
    int srow;            // P2: row of the activation map
    int a;               // group slot
    int pos;             // P1: first row of the inner dimension; P2: first output row
    int pad[2];
};
static_assert(sizeof(RwTask) == 32, "layout");

// chains of a second-projection task of `rows` slots: 2 * rows columns each (hi and lo parts)
__device__ __forceinline__ int rw_chains2(int acc_cols, int rows)
{
    return 16 * rows <= acc_cols ? 8 : 8 * rows <= acc_cols ? 4 : 2;
}

// rows of the activation box that holds T tokens
__host__ __device__ __forceinline__ int rw_tok_rows(int T) { return T <= 8 ? 8 : (T <= 16 ? 16 : (T <= 32 ? 32 : 64)); }

// route_smem: shared memory of a routing block that is to share an SM with a CTA of this kernel (0: none does)
inline RwPlan rw_make_plan(const Shape &sh, int B, int n_sm, bool early, int route_smem)
{
    RwPlan p{};
    if (sh.weight_dtype != DT_BF16 || sh.act_dtype != DT_BF16 || sh.d % 64 || sh.f % 32 || (sh.n_sh && sh.f_sh % 32) || B > kMaxTokens)
        return p;
    const int G = sh.E + sh.n_sh, n_slots = B * sh.k + sh.n_sh * B;
    p.early = early && n_sm > 1;
    // experts whose first projection starts before the gating (see the header comment)
    // One or two tokens select little more than top_k, and wave 1 begins behind the early experts: a quarter is
    // left for it.  Measured, us per layer, three quarters / all of top_k: OLMoE shape (top 8) 1 token 30.4 / 32.9,
    // 2 tokens 35.3 / 37.1, 128 narrow experts (top 8) 1 token 30.4 / 29.6, Qwen1.5-MoE shape (top 4) 35.7 / 34.9.
    p.n_early = p.early ? (B <= 2 ? (3 * sh.k + 2) / 4 : sh.k) : 0;
    p.n1 = (B + 15) & ~15;
    const int trows = rw_tok_rows(B);
    // Tasks of the second projection whose token tiles would make every stage larger (32 slots where the batch
    // has up to 32 tokens, 64 above) take one k-tile per stage: few groups are that large, and a stage of 40
    // or 48 instead of 48 or 64 KiB gives the ring a stage more.  Measured, us per layer, two k-tiles / one:
    // DeepSeek-V2-Lite shape 20 tokens 61.8 / 58.1, 32 tokens 69.3 / 65.6, 64 tokens 117.7 / 113.7, OLMoE shape
    // 24 tokens 57.2 / 53.7, Qwen1.5-MoE shape 32 tokens 53.1 / 50.8.  At 16 slots it loses: 51.9 / 53.6 (the
    // shared experts' tasks are a larger part there, and the ring does not get a stage more beside the
    // resident tiles and a routing block).
    p.one_rows = trows >= 32 ? trows : 0;
    const int tok2 = (p.one_rows ? 1 : 2) * 2 * trows * 128, tok1 = 2 * p.n1 * 128;
    p.c1 = p.n1 == 16 ? 8 : 4;
    p.acc_cols = p.c1 * p.n1 > 4 * trows ? p.c1 * p.n1 : 4 * trows;       // (128, 256: a power of two)
    while (p.acc_cols & (p.acc_cols - 1)) p.acc_cols += 32;
    p.n_acc = 512 / p.acc_cols;
    if (p.n_acc > kRwMaxAcc) p.n_acc = kRwMaxAcc;
    p.tmem_cols = p.acc_cols * p.n_acc;
    p.gf = rw_div_make(sh.f / 8);
    p.gs = rw_div_make(sh.n_sh ? sh.f_sh / 8 : 1);
    p.tf = rw_div_make((p.gf.d + 7) / 8);
    p.ts = rw_div_make((p.gs.d + 7) / 8);
    p.kr = rw_div_make((sh.f + 127) / 128);
    p.ks = rw_div_make(sh.n_sh ? (sh.f_sh + 127) / 128 : 1);
    p.rb = rw_div_make((sh.d + 127) / 128);
    // tasks of a CTA at most: a share of n units in groups of g, m units per task, meets n / g + 2 groups,
    // and every group adds at most one ragged task to n / m whole ones (44: four per lot, and room for
    // the tables' first pass)
    const long long P = n_sm - 1 > 0 ? n_sm - 1 : 1, U = sh.E < (long long)B * sh.k + p.n_early ? sh.E : (long long)B * sh.k + p.n_early;
    const long long n1r = U * p.gf.d, n1s = sh.n_sh ? (long long)sh.n_sh * p.gs.d : 0;
    const long long n2r = U * p.rb.d * p.kr.d, n2s = sh.n_sh ? (long long)sh.n_sh * p.rb.d * p.ks.d : 0;
    const long long tasks = n1r / P / 8 + n1r / P / p.gf.d + n1s / P / 8 + n1s / P / p.gs.d + n2r / P / p.kr.d + n2s / P / p.ks.d +
                            44;
    // (unit numbers are 31-bit, those of the first projection also 8 times over; k-tiles are kept in 15 bits)
    if (8 * (n1r + n1s) + 64 * P >= 1ll << 31 || n1r + n1s + n2r + n2s + 128 * P >= 1ll << 31 ||
        p.kr.d >= 1u << 14 || p.ks.d >= 1u << 14)
        return p;
    // (as many as there are: a table that leaves no room for two stages makes the plan infeasible)
    p.max_tasks = (int)tasks;
    const int nk = sh.d / 64;
    p.tab_bytes = ((int)sizeof(TcGroup) * (G + 1 + sh.n_sh) + 8 * n_slots + (int)sizeof(RwTask) * p.max_tasks + 1023) & ~1023;
    // Early start: a routing block shares every SM with a CTA of this kernel if that leaves room for three
    // stages (two blocks on an SM share 228 KiB, 1 KiB of it reserved for each).  If not, one CTA less than
    // SMs: the SM that runs the gating is taken until the routing kernel ends, and its CTA would start
    // last with a full share.  Up to 16 tokens only: with more the stage that the routing block costs is worth
    // more (us per layer beside / not: OLMoE shape 8 tokens 41.6 / 43.3, 24 tokens 54.0 / 53.6, 128 experts
    // at 32 tokens 61.3 / 55.7).
    const int full = kRwMaxSmem - p.tab_bytes - 1024, shared = 228 * 1024 - 2048 - kRwStaticSmem - route_smem - p.tab_bytes - 1024;
    const int x_res = ((nk + 7) & ~7) * (B <= 8 ? 8 : p.n1) * 128 + 1024, st_res = kRwWBytes + ((tok2 + 1023) & ~1023);
    const int st_tok = kRwWBytes + (((tok1 > tok2 ? tok1 : tok2) + 1023) & ~1023);
    const bool beside = p.early && route_smem > 0 && p.n1 == 16 &&
                        ((shared - x_res) / st_res >= 3 || ((full - x_res) / st_res < 3 && shared / st_tok >= 4));
    const int budget = beside ? shared : full;
    p.n_cta = p.early && !beside ? n_sm - 1 : n_sm;
    p.p = rw_div_make(p.n_cta);
    // Hidden states resident where at least three stages fit beside them; else their tiles travel
    // with the stages, one copy more and at most one chunk of two k-tiles per stage.  Measured, us per
    // layer, three stages with resident tiles / five without: DeepSeek-V2-Lite shape at 16 tokens 54.5 /
    // 57.5, Qwen1.5-MoE shape 46.7 / 50.1, 128 experts at 13 tokens 48.7 / 51.3.  (MMAs of a task with
    // few rows read past the rows it has, up to 60 KiB from the start of a stage: room for that behind
    // the last stage.)
    for (int res = 1; res >= 0; --res) {
        p.xr = res && B <= 8 ? 8 : p.n1;
        p.x_bytes = res ? ((nk + 7) & ~7) * p.xr * 128 + 1024 : 0;
        const int tok = res ? tok2 : (tok1 > tok2 ? tok1 : tok2);
        p.stage_bytes = kRwWBytes + ((tok + 1023) & ~1023);
        int slack = 61440 - p.stage_bytes - p.x_bytes;
        if (slack < 0) slack = 0;
        p.stages = (budget - p.x_bytes - slack) / p.stage_bytes;
        if (p.stages > kRwMaxStages) p.stages = kRwMaxStages;
        p.smem_bytes = p.tab_bytes + 1024 + p.stages * p.stage_bytes + p.x_bytes + slack;
        if (p.stages >= (res ? 3 : 2)) { p.feasible = 1; break; }
    }
    if (!p.feasible) return p;
    // Two waves, cut in the middle.  Measured, us per layer, with a third one from 13/16 on: OLMoE shape at 8
    // tokens 40.9 / 41.0, one token 32.1 / 32.4, DeepSeek-V2-Lite shape at 16 tokens 51.7 / 52.4, at 64
    // 126.5 / 127.9, Qwen1.5-MoE shape 42.3 / 43.1, 128 narrow experts at 13 tokens 38.3 / 38.2, 128 wide ones
    // at 8 75.4 / 76.2.
    p.split16 = 8;
    return p;
}

__device__ __forceinline__ void rw_tma_gateup(uint32_t dst, const CUtensorMap *map, int kt, int grp, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %3, %4, %3, %5}], [%2], %6;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(0), "r"(kt), "r"(grp), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void rw_tma_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar, uint64_t policy)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%3, %4}], [%2], %5;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "l"(policy)
        : "memory");
}
__device__ __forceinline__ void rw_tma_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}
__device__ __forceinline__ void rw_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void rw_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
        "}\n" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc)
        : "memory");
}
// sums of eight columns at t, t + step, .. (n pieces, four loaded at a time)
__device__ __forceinline__ void rw_ld8_sums(uint32_t t, uint32_t step, int n, float (&v)[8])
{
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = 0.0f;
#pragma unroll 1
    for (; n >= 4; n -= 4, t += 4 * step) {
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                         : "=r"(r[8 * i]), "=r"(r[8 * i + 1]), "=r"(r[8 * i + 2]), "=r"(r[8 * i + 3]), "=r"(r[8 * i + 4]),
                           "=r"(r[8 * i + 5]), "=r"(r[8 * i + 6]), "=r"(r[8 * i + 7])
                         : "r"(t + step * i));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int j = 0; j < 8; ++j)
            v[j] += (__uint_as_float(r[j]) + __uint_as_float(r[8 + j])) + (__uint_as_float(r[16 + j]) + __uint_as_float(r[24 + j]));
    }
#pragma unroll 1
    for (; n > 0; --n, t += step) {
        float w[8];
        tc_ld8(t, w);
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += w[j];
    }
}

// A lot: units in groups of g.d, dealt to the CTAs in contiguous shares.  Of this CTA's share: first
// unit, and its tasks, which never cross a group and have at most 1 << m units each.
struct RwSeg {
    int start, head, t_head, full, tail, n;      // t_head tasks in the first group's `head` units, `full` whole groups, `tail` units
};
__device__ __forceinline__ RwSeg rw_seg(int start, int cnt, const RwDiv &g, int m, int tasks_per_group)
{
    RwSeg s{start, 0, 0, 0, 0, 0};
    if (cnt <= 0) return s;
    const int round = (1 << m) - 1;
    s.head = min(cnt, (int)g.d - (start - rw_div(start, g) * (int)g.d));
    s.t_head = (s.head + round) >> m;
    s.full = rw_div(cnt - s.head, g);
    s.tail = cnt - s.head - s.full * (int)g.d;
    s.n = s.t_head + s.full * tasks_per_group + ((s.tail + round) >> m);
    return s;
}
// task j of a share: first unit and length
__device__ __forceinline__ void rw_seg_task(const RwSeg &s, const RwDiv &g, int m, const RwDiv &tasks_per_group, int j, int &unit, int &len)
{
    int base = 0, have = s.head, q = j;
    if (j >= s.t_head) {
        j -= s.t_head;
        const int grp = min(rw_div(j, tasks_per_group), s.full);
        q = j - grp * (int)tasks_per_group.d;
        base = s.head + grp * (int)g.d;
        have = grp < s.full ? (int)g.d : s.tail;
    }
    unit = s.start + base + (q << m);
    len = min(1 << m, have - (q << m));
}

// (bound of 1024 threads: at most 64 registers, so that a routing block of 512 threads x 80 registers fits beside it)
__global__ void __launch_bounds__(1024, 1)
ffn_rows_kernel(const __grid_constant__ RwMaps maps, const __grid_constant__ RwArgs p)
{
    extern __shared__ __align__(1024) uint8_t rw_smem[];
    __shared__ __align__(8) uint64_t full_bar[kRwMaxStages], empty_bar[kRwMaxStages];
    __shared__ __align__(8) uint64_t acc_full[kRwMaxAcc], acc_empty[kRwMaxAcc], x_bar, in_bar, lvl_bar[kRwLevels], ep_bar[kRwSets];
    __shared__ uint32_t s_tmem;
    __shared__ int s_lim[kRwLevels + 1];           // tasks known at each level (kRwLevels)
    __shared__ int s_n_bad, s_U, s_waves;          // early experts without tokens; experts in s_id; waves
    __shared__ uint16_t s_id[kMaxExperts];         // routed experts in this kernel's order: the early ones, then the others, ascending
    __shared__ uint8_t s_sel[kMaxExperts];         // the early ones that have tokens
    __shared__ volatile int s_ready[kRwMaxWaves];  // wave w's activations are written (set by the watcher)
    __shared__ RwSeg s_lot[kRwMaxWaves], s_lot2[kRwLots2];
    __shared__ int s_first[kRwMaxWaves + 1], s_first2[kRwLots2 + 1], s_bound[kRwMaxWaves + 1];   // first task of a lot; first routed group of a wave

    const Shape &sh = p.sh;
    const Workspace &ws = p.ws;
    const RwPlan &pl = p.plan;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = sh.E + sh.n_sh, GP = G + 1;      // GP: provisional groups of the shared experts
    const int n_routed = p.B * sh.k, n_slots = n_routed + sh.n_sh * p.B;
    const bool EARLY = pl.early != 0;
    const int P = (int)pl.p.d, cta = (int)blockIdx.x;
    const int Gf = (int)pl.gf.d, Gs = sh.n_sh ? (int)pl.gs.d : 0;

    TcGroup *groups = reinterpret_cast<TcGroup *>(rw_smem);
    RwTask *tasks = reinterpret_cast<RwTask *>(rw_smem + sizeof(TcGroup) * (G + 1 + sh.n_sh));
    int *s_slot_token = reinterpret_cast<int *>(tasks + pl.max_tasks);
    float *s_slot_w = reinterpret_cast<float *>(s_slot_token + n_slots);
    uint8_t *ring = rw_smem + pl.tab_bytes;
    ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(ring) + 1023) & ~(uintptr_t)1023);
    uint8_t *xres = ring + (size_t)pl.stages * pl.stage_bytes;
    const int S = pl.stages, nk = sh.d / 64;

    // This CTA's share of a lot of n units of which `before` units have been dealt already: the CTAs that
    // get one unit more than others rotate, so that all totals differ by one unit at most.
    auto share = [&](int n, int before, int &start, int &cnt) {
        const int q = rw_div(n, pl.p), r = n - q * P;
        int c = cta - (before - rw_div(before, pl.p) * P);
        if (c < 0) c += P;
        start = c * q + min(c, r);
        cnt = q + (c < r ? 1 : 0);
    };
    // where a routed expert's weights lie (offloaded experts: a device slot)
    auto weights_of = [&](int id) -> int { return ws.slot_of ? __ldg(&ws.slot_of[id]) : id; };
    auto make_p1 = [&](RwTask *t, int a, int expert, int in, int len, int shared, int wave) {
        t->flags = (shared << 1) | (wave << 2) | (len << 8);
        t->x0 = expert * (shared ? Gs : Gf) + in;
        t->a = a;
        t->pos = in * 8;
    };

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"((uint32_t)pl.tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else if (warp == 2) {
        if (lane < S) {
            mbar_init(&full_bar[lane], 1);
            mbar_init(&empty_bar[lane], 1);
        }
        if (lane < pl.n_acc) {
            mbar_init(&acc_full[lane], 1);
            mbar_init(&acc_empty[lane], 4);
        }
        if (lane < kRwMaxWaves) s_ready[lane] = 0;
        if (lane == 0) {
            mbar_init(&x_bar, 1);
            mbar_init(&in_bar, 1);
            for (int l = 0; l < kRwLevels; ++l) mbar_init(&lvl_bar[l], 1);
            mbar_init(&ep_bar[0], 4);
            mbar_init(&ep_bar[1], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (warp == 3) {
        // lot S: the shared experts' first projection, known before any routing
        int start, cnt;
        share(sh.n_sh * Gs, 0, start, cnt);
        const RwSeg sg = rw_seg(start, sh.n_sh ? cnt : 0, pl.gs, 3, (int)pl.ts.d);
        for (int j = lane; j < sg.n; j += 32) {
            int u, len;
            rw_seg_task(sg, pl.gs, 3, pl.ts, j, u, len);
            const int g = rw_div(u, pl.gs);
            make_p1(&tasks[j], GP + g, g, u - g * Gs, len, 1, 0);
        }
        const unsigned long long all = p.B >= 64 ? ~0ull : ((1ull << p.B) - 1ull);
        if (lane < sh.n_sh) {
            TcGroup gr;
            gr.mask = all; gr.group = sh.E + lane; gr.T = p.B; gr.off = n_routed + lane * p.B; gr.f = sh.f_sh;
            gr.p1 = 0; gr.p2 = 0;
            groups[GP + lane] = gr;
        }
        if (lane == 0) s_lim[0] = sg.n;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem;
    const int lim0 = s_lim[0];
    // the hidden states may be read (see warp 3); by the one thread that issues their copies
    auto inputs_wait = [&]() -> bool {
        if (!mbar_wait(&in_bar, 0)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); return false; }
        asm volatile("fence.proxy.async.global;" ::: "memory");
        return true;
    };

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (tc_elect()) {
            const uint64_t wpolicy = l2_evict_first_policy();
            const uint32_t ring_a = smem_u32(ring), full_a = smem_u32(full_bar);
            int s = 0, lim = lim0, level = 0, ready_w = 0;
            uint32_t par = 1;
            bool alive = (pl.x_bytes != 0 && !p.first) || inputs_wait();
            // second-projection stages whose weights are in flight but whose token tiles wait for the
            // activations of wave pend_w: pend_n stages from ring slot pend_s, task pend_t, k-tile pend_k on
            int pend_n = 0, pend_s = 0, pend_t = 0, pend_k = 0, pend_w = 0;

            auto load_tokens = [&](const RwTask &t, int slot, int kt) {
                const int rows = t.flags >> 8, mi = (t.flags & 2 ? 15 : 11) + (rows == 8 ? 0 : (rows == 16 ? 1 : (rows == 32 ? 2 : 3)));
                const uint32_t dst = ring_a + (uint32_t)(slot * pl.stage_bytes + kRwWBytes), bar = full_a + 8u * slot;
                rw_tma_3d(dst, &maps.m[mi], kt * 64, t.srow, 0, bar);
                if (rows != pl.one_rows && kt + 1 < (t.k >> 16)) rw_tma_3d(dst + rows * 256u, &maps.m[mi], kt * 64 + 64, t.srow, 0, bar);
            };
            auto flush = [&]() {
                // the wave's activations are written: order them before the copies below
                __threadfence_block();
                asm volatile("fence.proxy.async.global;" ::: "memory");
                ready_w = pend_w + 1;
                RwTask t = tasks[pend_t];
                for (; pend_n > 0; --pend_n) {
                    if (pend_k >= (t.k >> 16)) { t = tasks[++pend_t]; pend_k = t.k & 0xffff; }
                    load_tokens(t, pend_s, pend_k);
                    pend_k += (t.flags >> 8) == pl.one_rows ? 1 : 2;
                    if (++pend_s == S) pend_s = 0;
                }
            };
            // a free slot: while token tiles are outstanding, the readiness of their wave is polled beside it
            auto slot_wait = [&]() -> bool {
                if (pend_n == 0) {
                    if (mbar_wait(&empty_bar[s], par)) return true;
                    atomicExch(ws.status, ST_MBAR_TIMEOUT);
                    return false;
                }
                for (unsigned i = 0; i < kTcSpinLimit; ++i) {
                    if (pend_n > 0 && s_ready[pend_w]) flush();
                    if (mbar_test(&empty_bar[s], par)) return true;
                    __nanosleep(20);
                }
                atomicExch(ws.status, ST_DEP_TIMEOUT);
                return false;
            };
            auto ready_wait = [&]() -> bool {
                for (unsigned i = 0; i < kTcSpinLimit; ++i) {
                    if (s_ready[pend_w]) { flush(); return true; }
                    __nanosleep(20);
                }
                atomicExch(ws.status, ST_DEP_TIMEOUT);
                return false;
            };

            for (int i = 0; alive; ++i) {
                while (i >= lim && level < kRwLevels) {
                    if (!mbar_wait(&lvl_bar[level], 0)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); alive = false; break; }
                    lim = s_lim[++level];
                }
                if (!alive || i >= lim) break;
                const RwTask t = tasks[i];
                if (!(t.flags & 1)) {
                    const int np = t.flags >> 8, shd = (t.flags >> 1) & 1;
                    const CUtensorMap *gm = &maps.m[3 * shd];
                    const bool apart = ((p.mode >> (2 + shd)) & 1) != 0;
                    const int cps = pl.x_bytes ? 8 / np : 1;        // chunks of two k-tiles per stage
                    for (int kt = 0; kt < nk; kt += 2 * cps) {
                        if (!slot_wait()) { alive = false; break; }
                        const int nc = min(cps, (nk - kt + 1) >> 1);
                        const uint32_t bar = full_a + 8u * s;
                        uint32_t dst = ring_a + (uint32_t)(s * pl.stage_bytes);
                        rw_expect(bar, (uint32_t)(nc * np * 4096 + (pl.x_bytes ? 0 : 2 * pl.n1 * 128)));
                        if (!pl.x_bytes) rw_tma_3d(dst + kRwWBytes, &maps.m[10], 0, 0, kt, bar);
                        for (int c = 0; c < nc; ++c) {
                            const int k0 = kt + 2 * c;
                            int g = t.x0;
                            if (apart) {
                                for (int q = 0; q < np; ++q, ++g, dst += 4096) {
                                    rw_tma_3d(dst, gm, 0, g * 8, k0, bar);
                                    rw_tma_3d(dst + 2048, gm + 1, 0, g * 8, k0, bar);
                                }
                                continue;
                            }
                            if (np & 8) { rw_tma_gateup(dst, gm + 2, k0, g, bar, wpolicy); dst += 16384; g += 4; }
                            if (np & 12) { rw_tma_gateup(dst, gm + 2, k0, g, bar, wpolicy); dst += 16384; g += 4; }
                            if (np & 2) { rw_tma_gateup(dst, gm + 1, k0, g, bar, wpolicy); dst += 8192; g += 2; }
                            if (np & 1) { rw_tma_gateup(dst, gm, k0, g, bar, wpolicy); dst += 4096; }
                        }
                        if (++s == S) { s = 0; par ^= 1u; }
                    }
                } else {
                    const int k1 = t.k >> 16, wv = (t.flags >> 2) & 3, rows = t.flags >> 8, half = (t.flags >> 4) & 1;
                    const CUtensorMap *dm = &maps.m[(t.flags & 2 ? 7 : 6) + 2 * half];
                    const uint32_t wb = half ? 8192u : 16384u;
                    if (pend_n > 0 && wv != pend_w) { if (!ready_wait()) { alive = false; break; } }
                    if (pend_n == 0 && wv >= ready_w && s_ready[wv]) { pend_w = wv; pend_t = i; flush(); }
                    const int step = rows == pl.one_rows ? 1 : 2;
                    for (int kt = t.k & 0xffff; kt < k1; kt += step) {
                        // (every slot waits for its tokens: nothing can become free before they are there)
                        if (pend_n == S) { if (!ready_wait()) { alive = false; break; } }
                        if (!slot_wait()) { alive = false; break; }
                        const int two = min(step, k1 - kt);
                        const uint32_t bar = full_a + 8u * s, dst = ring_a + (uint32_t)(s * pl.stage_bytes);
                        rw_expect(bar, (uint32_t)two * (wb + (uint32_t)rows * 256u));
                        rw_tma_2d(dst, dm, kt * 64, t.x0, bar, wpolicy);
                        if (two == 2) rw_tma_2d(dst + 16384, dm, kt * 64 + 64, t.x0, bar, wpolicy);
                        if (wv < ready_w) {
                            load_tokens(t, s, kt);
                        } else {
                            if (pend_n == 0) { pend_s = s; pend_t = i; pend_k = kt; pend_w = wv; }
                            ++pend_n;
                        }
                        if (++s == S) { s = 0; par ^= 1u; }
                    }
                }
            }
            if (alive && pend_n > 0) ready_wait();
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (tc_elect()) {
            bool alive = true, x_there = pl.x_bytes == 0, x_copied = false;
            if (pl.x_bytes && (alive = inputs_wait())) {
                // the hidden states' tiles, eight k-tiles per copy (past the end: zeros)
                const uint32_t xb = smem_u32(&x_bar), xd = smem_u32(xres);
                rw_expect(xb, (uint32_t)(((nk + 7) & ~7) * pl.xr * 128));
                for (int kt = 0; kt < nk; kt += 8) rw_tma_3d(xd + (uint32_t)(kt * pl.xr * 128), &maps.m[10], 0, 0, kt, xb);
                x_copied = true;
            }
            int s = 0, lim = lim0, level = 0;
            uint32_t par = 0, run = 0;
            const uint32_t nbm = (uint32_t)pl.n_acc - 1u, nbs = (uint32_t)__ffs(pl.n_acc) - 1u;
            const uint64_t ring_d = tc_smem_desc(ring), ring_d2 = tc_smem_desc_sbo(ring, 2048u), xres_d = tc_smem_desc(xres);
            const uint32_t idesc1 = tc_idesc(pl.n1), x_step = (uint32_t)pl.xr * 8u;     // (descriptor units of 16 bytes)
            for (int i = 0; alive; ++i) {
                while (i >= lim && level < kRwLevels) {
                    if (!mbar_wait(&lvl_bar[level], 0)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); alive = false; break; }
                    lim = s_lim[++level];
                }
                if (!alive || i >= lim) break;
                const int flags = tasks[i].flags, tk = tasks[i].k;
                const uint32_t buf = run & nbm;
                if (!mbar_wait(&acc_empty[buf], ((run >> nbs) & 1u) ^ 1u)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
                if (!x_there) {
                    if (!mbar_wait(&x_bar, 0)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
                    x_there = true;
                }
                const uint32_t d_tmem = tmem_base + buf * (uint32_t)pl.acc_cols;
                if (!(flags & 1)) {
                    const int np = flags >> 8, cps = pl.x_bytes ? 8 / np : 1, last = pl.c1 - 1;
                    for (int kt = 0; kt < nk; kt += 2 * cps) {
                        if (!mbar_wait(&full_bar[s], par)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); alive = false; break; }
                        tc_fence_after();
                        const uint64_t st_a = (uint64_t)((uint32_t)(s * pl.stage_bytes) >> 4);
                        uint64_t ad = ring_d2 + st_a;
                        uint64_t bd = pl.x_bytes ? xres_d + (uint64_t)((uint32_t)kt * x_step) : ring_d + st_a + (kRwWBytes >> 4);
                        const int ke = min(nk, kt + 2 * cps);
                        for (int k = kt; k < ke; k += 2) {
#pragma unroll
                            for (int q = 0; q < 2; ++q) {
                                if (k + q < ke) {
#pragma unroll
                                    for (int h = 0; h < 4; ++h)
                                        rw_mma(d_tmem + (uint32_t)((q + (k & last)) * pl.n1), ad + (uint64_t)(64 * q + 2 * h),
                                               bd + (uint64_t)(x_step * q + 2 * h), idesc1, h > 0 || k + q > last ? 1u : 0u);
                                }
                            }
                            ad += (uint64_t)(np * 256);
                            bd += (uint64_t)(2 * x_step);
                        }
                        tc_commit(&empty_bar[s]);
                        if (++s == S) { s = 0; par ^= 1u; }
                    }
                } else {
                    const int k1 = tk >> 16, k0 = tk & 0xffff, rows = flags >> 8;
                    const uint32_t idesc = tc_idesc(2 * rows);
                    const int last = rw_chains2(pl.acc_cols, rows) - 1;
                    const int step = rows == pl.one_rows ? 1 : 2;
                    for (int kt = k0; kt < k1; kt += step) {
                        if (!mbar_wait(&full_bar[s], par)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); alive = false; break; }
                        tc_fence_after();
                        const uint64_t ad = ring_d + (uint64_t)((uint32_t)(s * pl.stage_bytes) >> 4), bd = ad + (kRwWBytes >> 4);
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            if (q < step && kt + q < k1) {
#pragma unroll
                                for (int h = 0; h < 4; ++h)
                                    rw_mma(d_tmem + (uint32_t)(2 * rows * ((kt + q - k0) & last)), ad + (uint64_t)(1024 * q + 2 * h),
                                           bd + (uint64_t)(rows * 16 * q + 2 * h), idesc, h > 0 || kt + q - k0 > last ? 1u : 0u);
                            }
                        }
                        tc_commit(&empty_bar[s]);
                        if (++s == S) { s = 0; par ^= 1u; }
                    }
                }
                if (!alive) break;
                tc_commit(&acc_full[buf]);
                ++run;
            }
            // (a CTA without tasks: the copies of the hidden states must have landed before it ends)
            if (x_copied && !x_there && !mbar_wait(&x_bar, 0)) atomicExch(ws.status, ST_MBAR_TIMEOUT);
        }
    } else if (warp == 10) {
        // ------------------------------------------------------------------ early experts, first projection's tasks; then watcher
        // Bounded wait for words of the routing kernel, each polled by a lane of its own until its tag is
        // there.  (They are cleared before this grid is scheduled.)
        const int nwords = (sh.E + 31) >> 5;
        auto poll = [&](const unsigned long long *words, int n) -> unsigned {
            unsigned long long v = 0ull;
            for (unsigned i = 0; i < (1u << 21); ++i) {
                if (lane < n)
                    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(words + lane) : "memory");
                if (__all_sync(0xffffffffu, lane >= n || (v >> 32) == 1ull)) return lane < n ? (unsigned)v : 0u;
                __nanosleep(20);
            }
            if (lane == 0) atomicExch(ws.status, ST_DEP_TIMEOUT);
            return 0u;
        };
        // experts of a set (lane q: word q) to s_id[n ..], ascending; returns the new n
        auto expand = [&](unsigned w, int n) -> int {
#pragma unroll 1
            for (int q = 0; q < nwords; ++q) {
                const unsigned wq = __shfl_sync(0xffffffffu, w, q);
                if ((wq >> lane) & 1u) s_id[n + __popc(wq & ((1u << lane) - 1u))] = (uint16_t)(32 * q + lane);
                n += __popc(wq);
            }
            __syncwarp();
            return n;
        };
        auto open = [&](int level, int tasks_known) {
            __syncwarp();
            if (lane == 0) {
                s_lim[level] = min(tasks_known, pl.max_tasks);
                mbar_arrive(&lvl_bar[level - 1]);
            }
        };
        // Two passes over the same code.  The first, with made-up inputs while there is nothing to wait for yet,
        // brings the code into the instruction caches: it runs once per launch, and fetched cold with the
        // weight stream on the memory system it took 3 us between the selection and the tasks.
#pragma unroll 1
        for (int real = EARLY ? 0 : 1; real < 2; ++real) {
            int n_early = 0, n_bad = 0, U = 0, nt = lim0, start, cnt;
            const int n_sh_units = sh.n_sh * Gs;
            if (EARLY) {
                if (real) {
                    // all blocks of the routing kernel have arrived: logits and importances are there, what it
                    // clears is cleared
                    const unsigned target = __shfl_sync(0xffffffffu, poll(ws.early + kEarlyWords, 1), 0);
                    bool there = false;
                    for (unsigned i = 0; i < (1u << 21); ++i) {
                        unsigned v;
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ws.ticket) : "memory");
                        if (__all_sync(0xffffffffu, (int)(v - target) >= 0)) { there = true; break; }
                        __nanosleep(20);
                    }
                    if (!there && lane == 0) atomicExch(ws.status, ST_TICKET_TIMEOUT);
                }
                // The n_early experts of largest importance: lane owns experts lane, lane + 32, .., as integer
                // keys in the order of the floats whose last bits name the expert, so that no two are equal
                // (24 bits of the importance decide, which is plenty for a guess).
                unsigned key[kEarlyWords], won = 0u;
#pragma unroll
                for (int q = 0; q < kEarlyWords; ++q) {
                    const int e = lane + 32 * q;
                    key[q] = 0u;
                    if (e < sh.E) {
                        const unsigned f = real ? __float_as_uint(__ldcg(&ws.gsum[e])) : 0u;
                        key[q] = ((f & 0x80000000u ? ~f : f | 0x80000000u) & 0xffffff00u) | (255u - (unsigned)e);
                    }
                }
                auto take = [&](auto words) {
#pragma unroll 1
                    for (int r = 0; r < pl.n_early; ++r) {
                        unsigned m = key[0];
#pragma unroll
                        for (int q = 1; q < words(); ++q) m = max(m, key[q]);
                        m = __reduce_max_sync(0xffffffffu, m);
#pragma unroll
                        for (int q = 0; q < words(); ++q) {
                            won |= key[q] == m ? 1u << q : 0u;
                            key[q] = key[q] == m ? 0u : key[q];
                        }
                    }
                };
                if (nwords <= 2) take([] { return 2; });
                else take([] { return kEarlyWords; });
                // (the set as words, lane q: word q, and its experts in ascending order)
                unsigned w = 0u;
#pragma unroll 1
                for (int q = 0; q < nwords; ++q) {
                    const unsigned word = __ballot_sync(0xffffffffu, (won >> q) & 1u);
                    if ((word >> lane) & 1u) s_id[n_early + __popc(word & ((1u << lane) - 1u))] = (uint16_t)(32 * q + lane);
                    if (lane == q) w = word;
                    n_early += __popc(word);
                }
                __syncwarp();
                // lot E: their first projection
                share(n_early * Gf, n_sh_units, start, cnt);
                const RwSeg sg = rw_seg(start, cnt, pl.gf, 3, (int)pl.tf.d);
                for (int j = lane; j < sg.n; j += 32) {
                    int u, len;
                    rw_seg_task(sg, pl.gf, 3, pl.tf, j, u, len);
                    const int g = rw_div(u, pl.gf);
                    if (nt + j < pl.max_tasks) make_p1(&tasks[nt + j], g, s_id[g], u - g * Gf, len, 0, 0);
                }
                nt += sg.n;
                if (real) open(1, nt);
                // all others, as soon as the selection is known
                const unsigned all = real ? poll(ws.early, nwords) : w ^ (lane < nwords ? 1u : 0u);
                U = expand(all & ~w, n_early);
                int a = 0, ns = 0;
#pragma unroll 1
                for (int q = 0; q < nwords; ++q) {
                    const unsigned wq = __shfl_sync(0xffffffffu, w, q), sq = wq & __shfl_sync(0xffffffffu, all, q), below = (1u << lane) - 1u;
                    if ((sq >> lane) & 1u) s_sel[ns + __popc(sq & below)] = (uint8_t)(a + __popc(wq & below));
                    a += __popc(wq);
                    ns += __popc(sq);
                }
                n_bad = n_early - ns;
            } else {
                open(1, nt);
                asm volatile("griddepcontrol.wait;" ::: "memory");
                U = ws.header[2];
                for (int a = lane; a < U; a += 32) s_id[a] = (uint16_t)ws.active[a];
                __syncwarp();
            }
            // lane w: wave w begins at the first routed group whose first projection lies past split16 / 16
            // of all of it (the early and the shared experts are in wave 0); lane kRwMaxWaves: the end
            int bnd = 0;
            if (lane > 0 && lane < kRwMaxWaves) {
                const int want = ((U * Gf + n_sh_units) * pl.split16 >> 4) - n_sh_units;
                bnd = min(U, max(rw_div(max(want, 0) + Gf - 1, pl.gf), max(n_early, sh.n_sh ? 0 : 1)));
            } else if (lane >= kRwMaxWaves) {
                bnd = U;
            }
            if (lane <= kRwMaxWaves) s_bound[lane] = bnd;
            const unsigned some = __ballot_sync(0xffffffffu, lane > 0 && lane < kRwMaxWaves && bnd < U);
            // lane w: first projection of wave w without the early experts
            const int lo = max(bnd, n_early), hi = __shfl_down_sync(0xffffffffu, bnd, 1);
            const int n = lane < kRwMaxWaves ? max(0, hi - lo) * Gf : 0;
            share(n, n_sh_units + lo * Gf, start, cnt);
            const RwSeg sg = rw_seg(start, n > 0 ? cnt : 0, pl.gf, 3, (int)pl.tf.d);
            int first = sg.n;
#pragma unroll
            for (int o = 1; o < kRwMaxWaves; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, first, o);
                if (lane >= o) first += t;
            }
            if (lane < kRwMaxWaves) {
                s_lot[lane] = sg;
                s_first[lane] = nt + first - sg.n;
                if (lane == kRwMaxWaves - 1) s_first[kRwMaxWaves] = nt + first;
            }
            if (lane == 0) {
                s_waves = 1 + __popc(some);
                s_n_bad = n_bad;
                s_U = U;
            }
            __syncwarp();
            const int end = s_first[kRwMaxWaves];
            for (int i = nt + lane; i < end && i < pl.max_tasks; i += 32) {
                int w = 0;
#pragma unroll
                for (int l = 1; l < kRwMaxWaves; ++l) w += i >= s_first[l] ? 1 : 0;
                int u, len;
                rw_seg_task(s_lot[w], pl.gf, 3, pl.tf, i - s_first[w], u, len);
                const int gq = rw_div(u, pl.gf), a = gq + max(s_bound[w], n_early);
                make_p1(&tasks[i], a, weights_of(s_id[a]), u - gq * Gf, len, 0, w);
            }
            __syncwarp();
            if (real) {
                if (lane == 0 && end > pl.max_tasks) atomicExch(ws.status, ST_BAD_PLAN);
                open(2, end);
            }
        }
        if (lane == 0) {
            // the waves' counters (the activations of all CTAs are stored), published in shared memory, so
            // that the producer never waits on global memory
            if (mbar_wait(&lvl_bar[kRwLevels - 1], 0)) {
                const int nw = s_waves;
                for (int w = 0; w < nw; ++w) {
                    bool there = false;
                    for (unsigned i = 0; i < (1u << 21); ++i) {
                        if (ld_acquire(&ws.sync[kTcReady - 8 + w]) >= kRwSets * P) { there = true; break; }
                        __nanosleep(20);
                    }
                    if (!there) { atomicExch(ws.status, ST_DEP_TIMEOUT); break; }
                    __threadfence_block();
                    s_ready[w] = 1;
                    // (every CTA has read the importances: back to zero for the next layer)
                    if (w == 0 && EARLY && cta == 0)
                        for (int e = 0; e < sh.E; ++e) ws.gsum[e] = 0.0f;
                }
            } else {
                atomicExch(ws.status, ST_MBAR_TIMEOUT);
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue sets
        const int set = warp >= 6 ? 1 : 0;
        if (warp == 3) {
            // the inputs may be read: the routing kernel has passed its own grid dependency (and says so), or ended
            if (EARLY) {
                bool there = false;
                for (unsigned i = 0; i < (1u << 21); ++i) {
                    unsigned long long v;
                    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ws.early + kEarlyWords) : "memory");
                    if (__all_sync(0xffffffffu, v != 0ull)) { there = true; break; }
                    __nanosleep(20);
                }
                if (!there && lane == 0) atomicExch(ws.status, ST_DEP_TIMEOUT);
            } else {
                asm volatile("griddepcontrol.wait;" ::: "memory");
            }
            if (lane == 0) mbar_arrive(&in_bar);
        }
        if (set == 1) {
            // the tables and the second projection's tasks, by warps 6..9 (128 threads on hardware barrier 1).
            // The next kernel in the stream may come up once this CTA has read the words of the early start:
            // the next layer's routing kernel clears them before anything else.
            // Two passes over the same code, as for warp 10: the first one makes tasks of one expert at the very
            // end of the table, where no real one of the first projection can be.
            const int tt = tid - 192;
            bool el_ok = true;
#pragma unroll 1
            for (int real = EARLY ? 0 : 1; real < 2; ++real) {
                if (real) {
                    el_ok = mbar_wait(&lvl_bar[1], 0) && mbar_wait(&in_bar, 0);
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
                }
                const int U = real ? s_U : 1, n_bad = real ? s_n_bad : 0, b0 = real ? s_lim[2] : pl.max_tasks - 8;
                // the groups in their final form and the slot arrays
                for (int a = tt; a < U; a += 128) {
                    const int id = real ? (int)s_id[a] : 0;
                    TcGroup gr;
                    gr.T = __ldcg(&ws.counts[id]);       // (past L1: the first pass may be ahead of the routing kernel)
                    gr.off = __ldcg(&ws.offsets[id]);
                    gr.mask = __ldcg(&ws.tokmask[id]);
                    gr.group = weights_of(id);
                    gr.f = sh.f;
                    gr.p1 = 0; gr.p2 = 0;
                    groups[a] = gr;
                }
                for (int i = tt; i < (real ? n_slots : 0); i += 128) {
                    s_slot_token[i] = ws.slot_token[i];
                    s_slot_w[i] = ws.slot_w[i];
                }
                const int RB = (int)pl.rb.d, u2r = RB * (int)pl.kr.d, u2s = sh.n_sh ? RB * (int)pl.ks.d : 0;
                if (warp == 6) {
                    // lane l: lot l of the second projection: wave 0, shared experts, waves 1 ..
                    const bool sx = lane == 1;
                    const int w = lane < 2 ? 0 : min(lane - 1, kRwMaxWaves - 1);
                    int n = sx ? sh.n_sh * u2s : (real ? s_bound[w + 1] - s_bound[w] - (w == 0 ? n_bad : 0) : w < 2) * u2r;
                    if (lane >= kRwLots2) n = 0;
                    // units dealt before this lot (a CTA that got a unit more of the first projection gets its full share
                    // of the second one all the same: taking d / 1024 units from it cost 0.9 % at 8 tokens of
                    // the OLMoE shape and 2.5 % at 64 of the DeepSeek-V2-Lite shape)
                    int before = n;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        const int t = __shfl_up_sync(0xffffffffu, before, o);
                        if (lane >= o) before += t;
                    }
                    int start, cnt;
                    share(n, before - n + sh.n_sh * Gs + U * Gf, start, cnt);
                    const RwSeg sg = rw_seg(start, n > 0 ? cnt : 0, sx ? pl.ks : pl.kr, 24, 1);
                    int first = sg.n;
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) {
                        const int t = __shfl_up_sync(0xffffffffu, first, o);
                        if (lane >= o) first += t;
                    }
                    if (lane < kRwLots2) {
                        s_lot2[lane] = sg;
                        s_first2[lane] = b0 + first - sg.n;
                        if (lane == kRwLots2 - 1) s_first2[kRwLots2] = b0 + first;
                    }
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");          // the group table and the lots are complete
                const int b1 = s_first2[kRwLots2];
                for (int i = b0 + tt; i < b1 && i < pl.max_tasks; i += 128) {
                    int l = 0;
#pragma unroll
                    for (int j = 1; j < kRwLots2; ++j) l += i >= s_first2[j] ? 1 : 0;
                    const bool sx = l == 1;
                    const int w = l < 2 ? 0 : l - 1;
                    const RwDiv kd = sx ? pl.ks : pl.kr;
                    RwTask *t = &tasks[i];
                    int u, len;
                    rw_seg_task(s_lot2[l], kd, 24, RwDiv{1u, 0u, 0}, i - s_first2[l], u, len);
                    const int gq = rw_div(u, kd), in = u - gq * (int)kd.d, eq = rw_div(gq, pl.rb), rbk = gq - eq * RB;
                    // (wave 0: the early experts that have tokens, then the others)
                    const int a = sx ? GP + eq : (w > 0 || n_bad == 0 ? eq + (real ? s_bound[w] : 0) : (eq < pl.n_early - n_bad ? (int)s_sel[eq] : eq + n_bad));
                    const TcGroup &g = groups[a];
                    const int kts = ((sx ? sh.f_sh : sh.f) + 63) >> 6;
                    t->flags = 1 | (sx ? 2 : 0) | (w << 2) | (sh.d - rbk * 128 <= 64 ? 16 : 0) | (rw_tok_rows(g.T) << 8);
                    t->x0 = (sx ? eq : g.group) * sh.d + rbk * 128;
                    t->k = (2 * in) | (min(kts, 2 * (in + len)) << 16);
                    t->srow = sx ? g.off - n_routed : g.off;
                    t->a = a;
                    t->pos = rbk * 128;
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (tt == 0 && real) {
                    if (!el_ok) atomicExch(ws.status, ST_MBAR_TIMEOUT);
                    if (b1 > pl.max_tasks) atomicExch(ws.status, ST_BAD_PLAN);
                    s_lim[kRwLevels] = min(b1, pl.max_tasks);
                    mbar_arrive(&lvl_bar[kRwLevels - 1]);               // (release: the tables are written)
                }
            }
        }
        const int q = warp & 3;                                     // TMEM lane quarter this warp may read
        const uint32_t nbm = (uint32_t)pl.n_acc - 1u, nbs = (uint32_t)__ffs(pl.n_acc) - 1u;
        int lim = lim0, level = 0, arrived = 0, waves = kRwMaxWaves;
        uint32_t ep_phase = 0;
        bool alive = true;
        auto wait_level = [&](int to) -> bool {
            while (level < to) {
                if (!mbar_wait(&lvl_bar[level], 0)) { if (lane == 0) atomicExch(ws.status, ST_MBAR_TIMEOUT); return false; }
                lim = s_lim[++level];
                if (level == kRwLevels) waves = s_waves;
            }
            return true;
        };
        // this set's activations of every wave below `upto` are stored: arrive on the waves' counters
        auto service = [&](int upto) -> bool {
            if (arrived >= min(upto, waves)) return true;
            if (!wait_level(kRwLevels)) return false;                // (the counters are clear once the routing kernel has ended)
            upto = min(upto, waves);
            if (arrived >= upto) return true;
            asm volatile("fence.proxy.async.global;" ::: "memory");  // the activations are read by TMA copies of other CTAs
            if (!tc_bar(&ep_bar[set], ep_phase, lane)) return false;
            for (; arrived < upto; ++arrived)
                if ((warp == 2 || warp == 6) && lane == 0) tc_red_release(&ws.sync[kTcReady - 8 + arrived]);
            return true;
        };
        for (int i = set; alive; i += kRwSets) {
            while (i >= lim && level < kRwLevels) { if (!wait_level(level + 1)) { alive = false; break; } }
            if (!alive || i >= lim) break;
            const RwTask t = tasks[i];
            const uint32_t buf = (uint32_t)i & nbm;
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + buf * (uint32_t)pl.acc_cols;
            // (a task of the second projection, or of a later wave: this set's part of the waves before is done)
            if (!service((t.flags & 1) ? kRwMaxWaves : (t.flags >> 2) & 3)) { alive = false; break; }
            // a routed expert: its tokens and slots come with the tables
            if (!(t.flags & 3) && level < kRwLevels) { if (!wait_level(kRwLevels)) { alive = false; break; } }
            if (!mbar_wait(&acc_full[buf], ((uint32_t)i >> nbs) & 1u)) {
                if (lane == 0) atomicExch(ws.status, ST_MBAR_TIMEOUT);
                alive = false;
                break;
            }
            tc_fence_after();
            const TcGroup g = groups[t.a];
            if (!(t.flags & 1)) {
                // lane l: row pair l / 16, gate (l & 8 == 0) or up; partner in lane l ^ 8.  Of two
                // neighbouring tokens the gate lane finishes the first, the up lane the second.
                const int shd = (t.flags >> 1) & 1, L = q * 32 + lane, pair = L >> 4, up = ((L >> 3) ^ (p.mode >> shd)) & 1;
                const bool row_ok = pair < (t.flags >> 8);
                const int fr = t.pos + pair * 8 + (L & 7);
                const size_t base = shd ? (size_t)n_routed * sh.f + (size_t)(g.off - n_routed) * sh.f_sh + fr : (size_t)g.off * sh.f + fr;
                const size_t stride = shd ? (size_t)sh.f_sh : (size_t)sh.f;
                for (int c = 0; c < p.B; c += 8) {
                    const unsigned m8 = (unsigned)((g.mask >> c) & 0xffull);
                    if (m8 == 0u) continue;
                    float v[8];
                    rw_ld8_sums(taddr + c, (uint32_t)pl.n1, min(pl.c1, nk), v);      // (a chain without a k-tile is not read)
                    int rank = __popcll(g.mask & ((1ull << c) - 1ull));
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        const unsigned mm = (m8 >> j) & 3u;
                        if (mm) {
                            const float other = __shfl_xor_sync(0xffffffffu, up ? v[j] : v[j + 1], 8);
                            const float a = up ? silu_mul(other, v[j + 1]) : silu_mul(v[j], other);
                            if (row_ok && ((mm >> up) & 1u)) {
                                const size_t o = base + (size_t)(rank + (up ? (int)(mm & 1u) : 0)) * stride;
                                const __nv_bfloat16 hi = __float2bfloat16_rn(a);
                                p.act_hi[o] = hi;
                                p.act_lo[o] = __float2bfloat16_rn(a - __bfloat162float(hi));
                            }
                            rank += __popc(mm);
                        }
                    }
                }
            } else {
                const int row = t.pos + q * 32 + lane, rows = t.flags >> 8;
                const bool row_ok = row < sh.d;
                const int pieces = 2 * min(rw_chains2(pl.acc_cols, rows), (t.k >> 16) - (t.k & 0xffff));   // hi and lo of every chain
                for (int c = 0; c < g.T; c += 8) {
                    float v[8];
                    rw_ld8_sums(taddr + c, (uint32_t)rows, pieces, v);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        if (c + j < g.T && row_ok) {
                            const int slot = g.off + c + j;
                            atomicAdd(&p.y[(size_t)s_slot_token[slot] * sh.d + row], s_slot_w[slot] * v[j]);
                        }
                    }
                }
            }
            // the accumulator may be overwritten
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[buf]);
        }
        if (alive && wait_level(kRwLevels)) service(kRwMaxWaves);
    }
    // every path ends here (all waits above are bounded), so the TMEM is always returned
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)pl.tmem_cols)
                     : "memory");
    }
}

}  // namespace s2moe
