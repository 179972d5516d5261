// tcgen05 expert kernel for block-int4 weights (kernel plan 3).
//
// Both projections are cut into split-K units of equal cost, 128 rows x 256 columns of one matrix:
//   phase 1: W_gate or W_up of one expert against the hidden states of all B tokens
//            -> red.add into pre[gate|up][slot][row]   (only the expert's tokens)
//   phase 2: W_down of one expert against its slots' activations (binary16 hi + lo parts)
//            -> y[token][row] += p * D                 (red.add, fp32)
// The experts are split into two waves.  When a CTA has finished its phase-1 units of a wave its epilogue
// hands the wave over to the CTA's converter warps, which arrive on the wave's grid-wide counter, wait
// (bounded) until all CTAs have arrived, turn their slice of the wave's pre into a = silu(g) * u and
// arrive on the wave's second counter, which the phase-2 token tiles of that wave wait for.  So the
// hand-over between the projections of one wave hides behind the other wave's work.  One persistent CTA
// per SM; of each of the four segments (phase 1 / 2 of wave 0 / 1) a CTA takes one contiguous run of
// units, so that consecutive k-pieces of a row block are summed up in registers and reduced to memory once.
//
// What a unit passes through: TMA brings its packed rows and scales into a stage of the ring; a group of
// dequantising warps turns it into binary16 values q * scale in tensor memory, the A operand of the MMAs,
// whose accumulators stay there over a run of units.  The token tiles of a unit are fetched into a buffer
// that belongs to the A operand's slot, so a stage is free as soon as it has been dequantised.
//
// What bounds it: instruction issue and latency.  At 6.5 TB/s an SM gets 42 weights per cycle; a weight
// costs 13 / 8 thread instructions to dequantise and nearly as much again for everything around it.  The MMAs
// themselves are cheap (A in tensor memory, N = 16: 22 cycles each from one thread, 16 a unit; N = 32: 26, N = 64: 37),
// but every instruction of a single thread's role waits for its turn behind the busy warps of its scheduler.  So
//   - the groups (three, each with a slot of its own, where the accumulators leave room for three, that is up to 32
//     tokens; else two) take the units in turn: a unit is some 800 cycles of issue, then its group waits 700 to 750 for the
//     issuer to notice, the MMAs and their completion, and the other groups work meanwhile.  With one group the schedulers
//     idled that long in every unit, with two the groups fell into step and idled together;
//   - weights and token tiles have a producer each: one thread for both needed 600 cycles per copy under that load, so
//     weights arrived just as they were asked for although the ring had stages to spare;
//   - a unit's entry in shared memory holds what the roles need (16 bytes and the row of the map), and what only some
//     units need is a function of its own (inlined everywhere it pushes the loops out of the instruction cache).
// A slot, and a stage of the ring (whose length is a multiple of the groups), belong to one group, so that whoever waits for
// their barriers sees every phase: a barrier tells only odd phases from even ones.
// Measured at the Mixtral shape, us per layer, with one group and one producer / now: 1 token 66.4 / 58.8, 8 tokens
// 120.7 / 97.3, 16 132.6 / 107.0, 32 138.7 / 119.1, 64 159.4 / 151.7 (the weights alone: 31 at 1 token, 62 at 8 at the
// measured copy rate).  Layers of a few units per CTA pay 0.5 to 1.3 us for it (more warps to start, a unit takes its group of
// four longer): 8 experts of 2048 x 1536, 8 tokens 28.5 / 29.0, 48 tokens 34.6 / 35.9; 128 of 2048 x 768, 8 tokens 38.7 / 38.5.
//
// Tried instead: the nibbles as binary16 subnormals n - 8 (9 instructions per 8 weights, exact), one
// accumulator per block of 32 columns and the scales applied in fp32 behind the MMAs: eight accumulators a unit
// instead of one a run have to be read back, 163 us at 8 tokens and 376 at 32 (147 and 183 for the kernel of the time).
// Units ordered so that a set of token tiles serves eight row blocks: eight times the reductions at the ends of
// runs, 128 at 8 tokens against 121.  Two issuers, unit by unit, with two groups: 111 and 133 at 8 and 32 tokens.
//
// Early start: the grid does not wait for the routing kernel as a whole.  The selected experts, known
// before the mixing weights and the buckets, are enough for every unit but the epilogue's targets, so
// the first projection streams while the gating ends.
//
// Warp roles (Q4Plan::threads): 0 weight producer; 1 MMA issuer; 2..5 epilogue; 6 none; 7..9 converters; 10 watcher (polls
// the waves' second counters and publishes them in shared memory); 11 token producer; from 12 on dequantising.  Warps
// 7..10 build the tables first.
#pragma once

#include "tc_common.cuh"

namespace s2moe {

constexpr int kQ4FirstDeq = 12;                // first dequantising warp (a multiple of 4)
constexpr int kQ4MaxThreads = 32 * (kQ4FirstDeq + 16);
constexpr int kQ4MaxGroups = 3;                // dequantising groups, unit by unit in turn
constexpr int kQ4MaxUnits = 384;               // units of one CTA decoded once into shared memory
constexpr int kQ4MaxWaves = 2, kQ4Segs = 2 * kQ4MaxWaves;

struct Q4Plan {
    int feasible;
    int n_cta;
    int stages;
    int n1;            // tokens padded to 16 (phase-1 N)
    int tab_bytes;
    int smem_bytes;
    int tokb;          // bytes of the token tiles of one k-tile
    int groups;        // dequantising groups; each has a slot of the A operand, 128 columns at the end of tensor memory
    int deq_warps;     // warps of a group: 4 (a row per thread) or 8 (half a row)
    int threads;
    int acc_cols;      // columns of an accumulator
    int early;         // the first projection starts when the selection is known
};

struct Q4Args {
    Shape sh;
    Workspace ws;
    Q4Plan plan;
    float *y;
    float *pre;                       // [gate|up][slot][f_g] fp32 pre-activations (zeroed by the routing kernel)
    __nv_bfloat16 *act_hi, *act_lo;   // [slot][f_g], binary16 parts, columns permuted inside groups of 8
    int B;
};

constexpr int kQ4StageBytes = kTcQ4KG * kTcQ4Packed + kTcQ4Scales;
static_assert(kQ4StageBytes % 1024 == 0, "stages are aligned for the 128-byte swizzle");

inline Q4Plan q4_make_plan(const Shape &sh, int B, int n_sm, bool early)
{
    Q4Plan p{};
    const int G = sh.E + sh.n_sh, n_slots = B * sh.k + sh.n_sh * B;
    p.n1 = (B + 15) & ~15;
    p.tokb = 2048 * ((B + 7) / 8);             // phase 2: per 8 slots their hi and lo rows; phase 1: n1 rows
    p.tab_bytes = ((int)sizeof(TcGroup) * G + 8 * n_slots + 1023) & ~1023;
    // Tensor memory: two accumulators of 64 columns (of 128 above 32 tokens) and the slots of the A operand.  The K-steps of a
    // run go to two chains in turn, since the tensor core truncates when it adds: both in one accumulator where twice a
    // unit's N columns fit it, else, up to 32 tokens, one in each of the two (an expert with 17 and more tokens; the next run
    // waits for the epilogue then).  Measured for those experts, all tokens on four of them, relative error of the second
    // projection's sums at d_ff 1536 / 3072 / 6144: two chains 1.9 / 3.1 / 6.5e-7, one chain cut after 12 k-pieces 3.5 /
    // 6.6 / 12.5e-7.  Time against that, us per layer: Mixtral shape 24 tokens 113.9 / 112.9, 32 tokens 121.0 / 119.2, d_ff
    // 4096 32 tokens 41.9 / 40.8.  Chains cut after half of every run, so that the accumulators stay two: 44.5 there.
    // Above 32 tokens an accumulator of 128 columns holds two chains of up to 64, or one of more (33 and more tokens).
    // Three groups of four warps up to 32 tokens, two of eight above (three slots do not fit).  Measured, us per layer at the
    // Mixtral shape, three / two (with the chains cut, on one box): 8 tokens 96 / 111, 16 tokens 105 / 120, 32 tokens 117 /
    // 133; four-warp groups with a row's eight chunks loaded together 99 / - at 8, and two of them 172 against 164 at 64.
    p.acc_cols = B <= 32 ? 64 : 128;
    p.groups = (512 - 2 * p.acc_cols) / 128;
    p.deq_warps = p.groups == 3 ? 4 : 8;
    p.threads = 32 * (kQ4FirstDeq + p.groups * p.deq_warps);
    // The token tiles lie beside the ring, one set per slot of the A operand: a stage is free as soon as its
    // weights and scales have been read, and not only when the MMAs have completed.
    p.stages = (kTcMaxSmem - p.tab_bytes - 1024 - p.groups * kTcQ4KG * p.tokb) / kQ4StageBytes;
    if (p.stages > kTcMaxStages) p.stages = kTcMaxStages;
    // (a stage is always the same group's: nine stages at most for three groups; where 8 or 7 become 6, at 17 to 32 tokens, the
    // groups gain more, and with the largest tables, where 7 become 3, 256 experts of 1024 x 512, top 16, beside 4 shared ones
    // take 77 us at 32 tokens as with one group and seven stages; at 64 tokens two stages for three cost 2 %, 117.2 / 115.0)
    p.stages -= p.stages % p.groups;
    p.smem_bytes = p.tab_bytes + p.stages * kQ4StageBytes + p.groups * kTcQ4KG * p.tokb + 1024;
    // (the SM that runs the gating is taken until the routing kernel ends: its CTA would start last with a
    // full share)
    p.early = early && n_sm > 1 ? 1 : 0;
    p.n_cta = n_sm - p.early;
    // (two stages at the limits: 60 and more tokens of 14 and more of 256 experts beside 4 shared ones; never less)
    p.feasible = p.stages >= p.groups && B <= kMaxTokens && sh.weight_dtype == DT_Q4B32 && sh.act_dtype == DT_BF16 && sh.d % 256 == 0 &&
                 sh.f % 256 == 0 && (sh.n_sh == 0 || sh.f_sh % 256 == 0);
    return p;
}

// What a unit needs, in one 16-byte entry: meta = first | last << 1 | (phase 2) << 2 | N << 8 (N of a phase-2
// unit is filled in with the buckets), group entry | map << 16 | segment << 20, first row of the matrix, first k-tile;
// beside it the first row of the map
struct Q4Segments {
    int start[kQ4Segs], cnt[kQ4Segs];  // this CTA's run of units of every segment
    int total1, U;                     // units of the first projection, routed experts
};
// unit i of this CTA (out of line: it runs once per unit while the tables are built, and only for units
// past the table afterwards; inlined at every use it pushes the roles' loops out of the instruction cache)
__device__ __noinline__ uint4 q4_unit_make(const Q4Segments &sg, const TcGroup *groups, const Shape &sh, int n1, int i)
{
    int seg = 0, j = i;
    while (seg < kQ4Segs - 1 && j >= sg.cnt[seg]) { j -= sg.cnt[seg]; ++seg; }
    const int total1 = sg.total1, U = sg.U, u = sg.start[seg] + j, last = sg.cnt[seg] - 1;
    const int kp1 = sh.d >> 8, rb2 = sh.d >> 7;
    int a, mat, rb, piece, kp;
    if (u < total1) {
        const int ur = 2 * (sh.f >> 7) * kp1, us = 2 * (sh.f_sh >> 7) * kp1;
        const bool sx = u >= U * ur;
        const int v = sx ? u - U * ur : u, per = sx ? us : ur, q = v / per, local = v - q * per, rest = local / kp1;
        const int rbs = (sx ? sh.f_sh : sh.f) >> 7;
        a = sx ? U + q : q;
        kp = kp1;
        piece = local - rest * kp1;
        mat = rest / rbs;
        rb = rest - mat * rbs;
    } else {
        const int ur = rb2 * (sh.f >> 8), us = rb2 * (sh.f_sh >> 8), w = u - total1;
        const bool sx = w >= U * ur;
        const int v = sx ? w - U * ur : w, per = sx ? us : ur, q = v / per, local = v - q * per;
        kp = (sx ? sh.f_sh : sh.f) >> 8;
        a = sx ? U + q : q;
        rb = local / kp;
        piece = local - rb * kp;
        mat = 2;
    }
    const uint32_t first = j == 0 || piece == 0, end = j == last || piece == kp - 1;
    // (N of a phase-2 unit: 0 before the buckets are known)
    const uint32_t n = mat < 2 ? (uint32_t)n1 : 16u * (((uint32_t)groups[a].T + 7u) >> 3);
    return make_uint4(first | (end << 1) | (mat == 2 ? 4u : 0u) | (n << 8), (uint32_t)a | ((uint32_t)(a >= U ? mat + 3 : mat) << 16) | ((uint32_t)seg << 20),
                      (uint32_t)rb * 128u, (uint32_t)(4 * piece));
}

__global__ void __launch_bounds__(kQ4MaxThreads, 1)
ffn_q4_kernel(const __grid_constant__ TcMaps maps, const __grid_constant__ Q4Args p)
{
    extern __shared__ __align__(1024) uint8_t q4_smem[];
    __shared__ __align__(8) uint64_t full_bar[kTcMaxStages], empty_bar[kTcMaxStages], a_full[kQ4MaxGroups], a_empty[kQ4MaxGroups];
    __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], conv_go[kQ4MaxWaves], tab_bar[2], cv_bar, tok_go;
    __shared__ uint32_t s_tmem;
    __shared__ int s_flag, s_n_units, s_split, s_n_active;
    __shared__ Q4Segments s_seg;
    __shared__ uint4 s_units[kQ4MaxUnits];
    __shared__ int s_row[kQ4MaxUnits];
    __shared__ uint16_t s_id[kMaxExperts];
    __shared__ volatile int s_ready[kQ4MaxWaves];  // wave w's activations are written (set by the watcher warp)

    const Shape &sh = p.sh;
    const Workspace &ws = p.ws;
    const Q4Plan &pl = p.plan;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int S = pl.stages, P = (int)gridDim.x, NG = pl.groups, ACC = pl.acc_cols;
    const uint32_t a_col = 512u - 128u * (uint32_t)NG;      // first column of the A operand's slots
    const bool EARLY = pl.early != 0;
    const int n_routed = p.B * sh.k, n_slots = n_routed + sh.n_sh * p.B;
    const int kp1 = sh.d >> 8, rb2 = sh.d >> 7;
    const int u1r = 2 * (sh.f >> 7) * kp1, u2r = rb2 * (sh.f >> 8);
    const int u1s = 2 * (sh.f_sh >> 7) * kp1, u2s = rb2 * (sh.f_sh >> 8);

    TcGroup *groups = reinterpret_cast<TcGroup *>(q4_smem);
    int *s_slot_token = reinterpret_cast<int *>(q4_smem + sizeof(TcGroup) * (sh.E + sh.n_sh));
    float *s_slot_w = reinterpret_cast<float *>(s_slot_token + n_slots);
    uint8_t *ring = q4_smem + pl.tab_bytes;
    ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(ring) + 1023) & ~(uintptr_t)1023);
    uint8_t *tokring = ring + (size_t)S * kQ4StageBytes;           // token tiles, one set per slot of the A operand

    if (warp == 2) {
        if (lane < S) {
            mbar_init(&full_bar[lane], 1);
            mbar_init(&empty_bar[lane], pl.deq_warps);
        }
        if (lane < 2) {
            mbar_init(&acc_full[lane], 1);
            mbar_init(&acc_empty[lane], 4);
        }
        if (lane < kQ4MaxGroups) {
            mbar_init(&a_full[lane], pl.deq_warps + 1);             // the dequantising warps and the token producer's arrival with the token bytes
            mbar_init(&a_empty[lane], 1);
        }
        if (lane < 2) mbar_init(&tab_bar[lane], 1);
        if (lane < kQ4MaxWaves) {
            mbar_init(&conv_go[lane], 4);
            s_ready[lane] = 0;
        }
        if (lane == 0) {
            mbar_init(&cv_bar, 3);
            mbar_init(&tok_go, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = s_tmem;

    auto unit_at = [&](int i) -> uint4 { return i < kQ4MaxUnits ? s_units[i] : q4_unit_make(s_seg, groups, sh, pl.n1, i); };
    auto umeta_at = [&](int i) -> uint32_t { return i < kQ4MaxUnits ? s_units[i].x : q4_unit_make(s_seg, groups, sh, pl.n1, i).x; };
    auto map_row = [&](const uint4 &un) -> int {
        const TcGroup &g = groups[un.y & 0xffffu];
        const int mi = (int)(un.y >> 16) & 15;
        return (mi >= 3 ? g.group - sh.E : g.group) * (mi == 2 || mi == 5 ? sh.d : g.f) + (int)un.z;
    };
    // level 0: every unit; level 1: tokens and slots of the routed experts (and everything the routing
    // kernel clears is clear)
    auto tab_wait = [&](int level) -> bool {
        if (mbar_wait(&tab_bar[level], 0)) return true;
        atomicExch(ws.status, ST_MBAR_TIMEOUT);
        return false;
    };

    if (warp >= 7 && warp <= 10) {
        // ------------------------------------------------------------------ tables
        const int tt = tid - 224, nwords = (sh.E + 31) >> 5;
        if (warp == 7) {
            int U = 0;
            if (EARLY) {
                // bounded wait for words of the routing kernel, each polled by a lane of its own until its tag is
                // there (they are cleared before this grid is scheduled)
                auto poll = [&](const unsigned long long *words, int n) -> unsigned {
                    unsigned long long v = 0ull;
                    for (unsigned i = 0; i < (1u << 21); ++i) {
                        if (lane < n) asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(words + lane) : "memory");
                        if (__all_sync(0xffffffffu, lane >= n || (v >> 32) == 1ull)) return lane < n ? (unsigned)v : 0u;
                        __nanosleep(20);
                    }
                    if (lane == 0) atomicExch(ws.status, ST_DEP_TIMEOUT);
                    return 0u;
                };
                // all blocks of the routing kernel have arrived: the permuted hidden states are there
                const unsigned target = __shfl_sync(0xffffffffu, poll(ws.early + kEarlyWords, 1), 0);
                bool there = false;
                for (unsigned i = 0; i < (1u << 21) && !there; ++i) {
                    unsigned v;
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ws.ticket) : "memory");
                    there = __all_sync(0xffffffffu, (int)(v - target) >= 0);
                    if (!there) __nanosleep(20);
                }
                if (!there && lane == 0) atomicExch(ws.status, ST_TICKET_TIMEOUT);
                // the selection: one word per 32 experts
                const unsigned w = poll(ws.early, nwords);
                for (int q = 0; q < nwords; ++q) {
                    const unsigned wq = __shfl_sync(0xffffffffu, w, q);
                    if ((wq >> lane) & 1u) s_id[U + __popc(wq & ((1u << lane) - 1u))] = (uint16_t)(32 * q + lane);
                    U += __popc(wq);
                }
            } else {
                asm volatile("griddepcontrol.wait;" ::: "memory");
                U = ws.header[2];
                for (int a = lane; a < U; a += 32) s_id[a] = (uint16_t)ws.active[a];
            }
            if (lane == 0) s_seg.U = U;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const int U = s_seg.U, n_active = U + sh.n_sh;
        const int total1 = U * u1r + sh.n_sh * u1s, total2 = U * u2r + sh.n_sh * u2s;
        for (int a = tt; a < n_active; a += 128) {
            TcGroup gr;
            const bool sx = a >= U;
            const int s = a - U;
            // (offloaded experts: the device slot a routed expert's weights lie in)
            gr.group = sx ? sh.E + s : (ws.slot_of ? __ldg(&ws.slot_of[s_id[a]]) : (int)s_id[a]);
            gr.T = sx ? p.B : 0;
            gr.off = sx ? n_routed + s * p.B : 0;
            gr.f = sx ? sh.f_sh : sh.f;
            gr.mask = sx ? (p.B >= 64 ? ~0ull : ((1ull << p.B) - 1ull)) : 0ull;
            gr.p1 = sx ? U * u1r + s * u1s : a * u1r;
            gr.p2 = sx ? U * u2r + s * u2s : a * u2r;
            groups[a] = gr;
        }
        // wave 1 starts at the first group whose first-projection units begin at or after its share of all of them
        int split;
        {
            const int want = (total1 * kTcSplitNum + kTcSplitDen - 1) / kTcSplitDen;
            split = (want + u1r - 1) / u1r;
            if (split > U) split = sh.n_sh ? U + max(0, (want - U * u1r + u1s - 1) / u1s) : U;
            split = min(max(split, 1), n_active);
            if (split >= n_active && n_active > 1) split = n_active - 1;
        }
        const int s1 = split < U ? split * u1r : U * u1r + (split - U) * u1s, s2 = split < U ? split * u2r : U * u2r + (split - U) * u2s;
        // every CTA takes one contiguous run of units of each segment (sizes differ by at most one; the CTAs
        // that get the extra unit rotate from segment to segment, so the totals differ by at most one as well)
        int n_units = 0;
        {
            const int begin[kQ4Segs] = {0, s1, total1, total1 + s2}, n[kQ4Segs] = {s1, total1 - s1, s2, total2 - s2};
            int rot = 0;
#pragma unroll
            for (int g = 0; g < kQ4Segs; ++g) {
                const int q = n[g] / P, r = n[g] - q * P;
                int c = (int)blockIdx.x - rot;
                if (c < 0) c += P;
                if (tt == 0) { s_seg.start[g] = begin[g] + c * q + min(c, r); s_seg.cnt[g] = q + (c < r ? 1 : 0); }
                n_units += q + (c < r ? 1 : 0);
                rot += r;
                if (rot >= P) rot -= P;
            }
        }
        if (tt == 0) {
            s_n_units = n_units;
            s_seg.total1 = total1;
            s_split = split;
            s_n_active = n_active;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        for (int i = tt; i < n_units && i < kQ4MaxUnits; i += 128) {
            const uint4 un = q4_unit_make(s_seg, groups, sh, pl.n1, i);
            s_units[i] = un;
            s_row[i] = map_row(un);
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (tt == 0) mbar_arrive(&tab_bar[0]);                     // (release: the tables are written)
        // The next kernel in the stream may come up once this CTA has read the words of the early start: the next
        // layer's routing kernel clears them before anything else.
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        for (int a = tt; a < U; a += 128) {
            const int id = s_id[a];
            groups[a].T = __ldcg(&ws.counts[id]);
            groups[a].off = __ldcg(&ws.offsets[id]);
            groups[a].mask = __ldcg(&ws.tokmask[id]);
        }
        for (int i = tt; i < n_slots; i += 128) {
            s_slot_token[i] = __ldcg(&ws.slot_token[i]);
            s_slot_w[i] = __ldcg(&ws.slot_w[i]);
        }
        if (EARLY && blockIdx.x == 0)
            for (int e = tt; e < sh.E; e += 128) ws.gsum[e] = 0.0f;   // (nobody reads it here; back to zero for the next layer)
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const int n_p1 = s_seg.cnt[0] + s_seg.cnt[1];
        for (int i = n_p1 + tt; i < n_units && i < kQ4MaxUnits; i += 128)
            s_units[i].x = (s_units[i].x & 0xffu) | ((16u * (((uint32_t)groups[s_units[i].y & 0xffffu].T + 7u) >> 3)) << 8);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (tt == 0) mbar_arrive(&tab_bar[1]);
    }

    if (warp == 0) {
        // ------------------------------------------------------------------ weight producer
        // packed k-tiles (128 bytes of every row) and the 8 scales per row of these 256 columns into the ring
        if (tc_elect() && tab_wait(0)) {
            const uint64_t wpolicy = l2_evict_first_policy();
            const int n_units = s_n_units;
            int s = 0;
            uint32_t ring_par = 1;
            for (int i = 0; i < n_units; ++i) {
                uint4 un;
                int row;
                if (i < kQ4MaxUnits) {
                    un = s_units[i];
                    row = s_row[i];
                } else {
                    un = q4_unit_make(s_seg, groups, sh, pl.n1, i);
                    row = map_row(un);
                }
                const CUtensorMap *map = &maps.m[(un.y >> 16) & 15u];
                uint8_t *stage = ring + (size_t)s * kQ4StageBytes;
                if (!mbar_wait(&empty_bar[s], ring_par)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
                mbar_expect_tx(&full_bar[s], kQ4StageBytes);
                tma_load_2d_stream(stage, map, (int)un.w * 32, row, &full_bar[s], wpolicy);
                tma_load_2d(stage + kTcQ4KG * kTcQ4Packed, map + 9, (int)un.w * 2, row, &full_bar[s]);
                if (i == 0) mbar_arrive(&tok_go);
                tc_ring_next(s, ring_par, S);
            }
            if (n_units == 0) mbar_arrive(&tok_go);
        }
    } else if (warp == 11) {
        // ------------------------------------------------------------------ token producer
        // The token tiles go into the set of the A operand's slot they are used with (free once the MMAs that read
        // it have completed; their bytes are counted by the barrier the dequantising warps arrive on, so that an MMA
        // issuer waits once), in the second projection only when their wave's activations are written.  The first ones go out
        // behind the first weights, which take longer to be of use (0.3 to 0.5 us of a layer of a few units per CTA: 8 experts of
        // 4096 x 1024, 8 tokens 30.9 -> 30.7 us, of 2048 x 768 27.4 -> 26.9; Mixtral shape +-0.1 %).
        if (tc_elect() && mbar_wait(&tok_go, 0)) {             // (the tables are written: the weight producer has waited for them)
            const int n_units = s_n_units, split = s_split;
            int ta = 0, ready_w = 0;
            uint32_t t_par = 1;
            // (the permuted hidden states are written by the routing kernel with generic stores)
            asm volatile("fence.proxy.async.global;" ::: "memory");
            for (int i = 0; i < n_units; ++i) {
                uint4 un = unit_at(i);
                const bool p2 = (un.x & 4u) != 0;
                if (p2) {
                    const int wv = (int)(un.y & 0xffffu) >= split ? 1 : 0;
                    if (wv >= ready_w) {
                        bool ok = false;
                        for (unsigned t = 0; t < kTcSpinLimit && !ok; ++t) {
                            ok = s_ready[wv] != 0;
                            if (!ok) __nanosleep(100);
                        }
                        // the activations of this wave are written: order them before the copies below
                        __threadfence_block();
                        asm volatile("fence.proxy.async.global;" ::: "memory");
                        if (!ok || !tab_wait(1)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
                        un = unit_at(i);
                        ready_w = wv + 1;
                    }
                }
                uint8_t *op = tokring + (size_t)ta * kTcQ4KG * pl.tokb;
                if (!mbar_wait(&a_empty[ta], t_par)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
                if (!p2) {
                    // the hidden-state tiles of all four k-tiles in one copy: [k-tile][tokb / 128 rows]
                    mbar_expect_tx(&a_full[ta], (uint32_t)(kTcQ4KG * pl.tokb));
                    tma_load_3d(op, &maps.m[6], 0, 0, (int)un.w, &a_full[ta]);
                } else {
                    // one copy per 8 slots for all four k-tiles: [hi | lo][k-tile][8 rows]
                    const TcGroup &g = groups[un.y & 0xffffu];
                    const bool shared = g.group >= sh.E;
                    const int srow = shared ? g.off - n_routed : g.off, n = (int)(un.x >> 8);
                    mbar_expect_tx(&a_full[ta], (uint32_t)(kTcQ4KG * n * 128));
                    for (int r = 0; r < n / 2; r += 8)
                        tma_load_4d(op + r * 256 * kTcQ4KG, &maps.m[shared ? 8 : 7], 0, srow + r, (int)un.w, 0, &a_full[ta]);
                }
                tc_ring_next(ta, t_par, NG);
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (tc_elect() && tab_wait(0)) {
            const int n_units = s_n_units;
            const uint32_t hi1 = (uint32_t)(tc_smem_desc(tokring) >> 32), hi2 = (uint32_t)(tc_smem_desc_sbo(tokring, (uint32_t)kTcQ4KG * 1024u) >> 32);
            const uint32_t tok_lo = (uint32_t)tc_smem_desc(tokring), a_tmem0 = tmem_base + a_col;
            const uint32_t tok_slot = (uint32_t)kTcQ4KG * ((uint32_t)pl.tokb >> 4), step1 = (uint32_t)pl.tokb >> 4;
            uint32_t buf = 0, run_par = 1, a_par = 0, um = n_units > 0 ? umeta_at(0) : 0u;
            int ta = 0;
            bool tabs = false;
            // (an instruction between two MMAs costs as much as the MMA: the K-steps are straight-line code, and a
            // unit's entry is read before the wait for the unit in front of it)
            for (int ui = 0; ui < n_units; ++ui) {
                if ((um & 4u) && !tabs) {
                    tabs = true;
                    if (!tab_wait(1)) break;
                    um = umeta_at(ui);
                }
                const uint32_t m = um;
                const bool p2 = (m & 4u) != 0, first = (m & 1u) != 0;
                // slot ta's k-tiles (32 columns each) and their token tiles: phase 1 [k-tile][rows], phase 2
                // [8 slots][hi | lo][k-tile][8 rows] (8-row groups 4 KiB apart)
                const uint32_t N = m >> 8, idesc = tc_idesc_f16((int)N), d_tmem = tmem_base + buf * (uint32_t)ACC;
                // where the odd K-steps add up: behind the even ones, in the other accumulator, or with them
                const bool both = ACC == 64 && 2u * N > 64u;
                const uint32_t odd = 2u * N <= (uint32_t)ACC ? N : !both ? 0u : buf ? 0u - 64u : 64u;
                const uint32_t a_tm = a_tmem0 + (uint32_t)ta * (kTcQ4KG * 32u), b_lo = tok_lo + (uint32_t)ta * tok_slot;
                const uint32_t b_step = p2 ? 64u : step1, b_hi = p2 ? hi2 : hi1;
                if (first && (!mbar_wait(&acc_empty[buf], run_par) || (both && !mbar_wait(&acc_empty[buf ^ 1u], run_par ^ buf)))) {
                    atomicExch(ws.status, ST_MBAR_TIMEOUT);
                    break;
                }
                if (ui + 1 < n_units) um = umeta_at(ui + 1);
                // the unit in tensor memory, written by the dequantising warps, and its token tiles
                if (!mbar_wait(&a_full[ta], a_par)) { atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
                tc_fence_after();
#pragma unroll
                for (uint32_t g = 0; g < kTcQ4KG; ++g)
#pragma unroll
                    for (uint32_t k = 0; k < 4; ++k)
                        tc_mma_bf16_tmem_a(d_tmem + (k & 1u ? odd : 0u), a_tm + 32u * g + 8u * k, b_lo + g * b_step + 2u * k, b_hi, idesc,
                                           g > 0 || k > 1 || (k == 1 && odd == 0u) || !first ? 1u : 0u);
                tc_commit(&a_empty[ta]);               // frees the A operand and the token tiles
                if (m & 2u) {
                    tc_commit(&acc_full[buf]);
                    if (both) tc_commit(&acc_full[buf ^ 1u]);      // (and the accumulator in turn is the same one)
                    else buf ^= 1u;
                    if (both || buf == 0) run_par ^= 1u;
                }
                tc_ring_next(ta, a_par, NG);
            }
        }
        __syncwarp();
    } else if (warp >= kQ4FirstDeq) {
        // ------------------------------------------------------------------ dequantising warps
        // Every row of a packed k-tile (64 nibbles, stored q + 8) becomes 64 binary16 values q * scale (row =
        // lane, two values per 32-bit column): per 32-bit word eight nibbles -> 1024 + n or 1024 + 16 n as
        // binary16 by an OR into the mantissa, then n - 8 (exact), times the block's scale (binary16 as stored,
        // so the product is the only rounding: 2^-12 relative).
        // A stage holds 256 columns: per row eight chunks of 16 packed bytes (32 weights, one scale each).  A warp
        // reaches the 32 lanes of its quarter (warp index mod 4) only, so thread (r, h) takes row
        // r = 32 * (warp mod 4) + lane and, in a group of four warps, all its chunks, in a group of eight chunks 4 h ..
        // 4 h + 3, h = 0 for the first four warps, 1 for the others.
        // While a group waits for the MMAs of its unit before, the others have the schedulers: groups that take
        // their units in step (two of them, measured) leave them idle for a third of the time.
        const int r = 32 * (warp & 3) + lane, dw = warp - kQ4FirstDeq, grp = dw / pl.deq_warps;
        const int h0 = (dw - grp * pl.deq_warps) >> 2, h1 = pl.deq_warps == 4 ? 2 : h0 + 1;
        int s = grp;
        uint32_t ring_par = 0, a_par = 1;
        const uint32_t a_slot = tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + a_col + (uint32_t)grp * 128u;
        const __half2 minus1032 = __floats2half2_rn(-1032.0f, -1032.0f), sixteenth = __floats2half2_rn(0.0625f, 0.0625f),
                      minus72 = __floats2half2_rn(-72.0f, -72.0f);
        const int n_units = tab_wait(0) ? s_n_units : 0;
        for (int ui = grp; ui < n_units; ui += NG) {
            const bool ok_full = mbar_wait(&full_bar[s], ring_par);
            if (!ok_full || !mbar_wait(&a_empty[grp], a_par)) { if (lane == 0) atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
            tc_fence_after();                                      // the MMAs that read this slot have completed
            const uint8_t *stage = ring + (size_t)s * kQ4StageBytes, *prow = stage + (size_t)r * 128;
#pragma unroll 1
            for (int h = h0; h < h1; ++h) {
                const uint2 sc2w = *reinterpret_cast<const uint2 *>(stage + kTcQ4KG * kTcQ4Packed + r * 16 + h * 8);   // four scales
                const uint32_t sc[2] = {sc2w.x, sc2w.y};
                // all packed chunks first: the stores to tensor memory below order
                // memory accesses, so a load behind one of them would wait for it
                uint4 pks[4];
#pragma unroll
                for (int qi = 0; qi < 4; ++qi) {
                    // (the packed rows are swizzled over their 128 bytes by the TMA copy)
                    pks[qi] = *reinterpret_cast<const uint4 *>(prow + (((h * 4 + qi) ^ (r & 7)) * 16));
                }
#pragma unroll
                for (int qi = 0; qi < 4; ++qi) {
                    const int q = h * 4 + qi;                     // chunk of 32 weights inside the stage
                    const uint4 pk = pks[qi];
                    // the block's scale is binary16 already: both halves of a register
                    const uint32_t sc2u = __byte_perm(sc[qi >> 1], 0u, (qi & 1) ? 0x3232u : 0x1010u);
                    const __half2 sc2 = *reinterpret_cast<const __half2 *>(&sc2u);
                    const uint32_t w[4] = {pk.x, pk.y, pk.z, pk.w};
                    uint32_t o[16];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        // A nibble n OR-ed into the mantissa of binary16 1024 is 1024 + n exactly; one
                        // that sits four bits higher gives 1024 + 16 n, which one fused multiply-add
                        // (x / 16 - 72) turns into the same n - 8 without a shift.  So a 32-bit word
                        // costs one shift and four logic instructions, and the pairs come out as
                        // (n0, n4), (n1, n5), (n2, n6), (n3, n7): the token tiles carry the same
                        // permutation of every 8 columns, so no instruction is spent on reordering.
                        // n - 8 is exact; the product with the scale rounds once (2^-12 relative).
                        const uint32_t mlo = 0x000F000Fu, mhi = 0x00F000F0u, k1024 = 0x64006400u;
                        const uint32_t w8 = w[c] >> 8;
                        uint32_t e[4];
                        tc_nibble_pair(e[0], w[c], mlo, k1024);
                        tc_nibble_pair(e[1], w[c], mhi, k1024);
                        tc_nibble_pair(e[2], w8, mlo, k1024);
                        tc_nibble_pair(e[3], w8, mhi, k1024);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const __half2 x = *reinterpret_cast<const __half2 *>(&e[j]);
                            const __half2 qv = (j & 1) ? __hfma2(x, sixteenth, minus72) : __hadd2(x, minus1032);
                            const __half2 v = __hmul2(qv, sc2);
                            o[4 * c + j] = *reinterpret_cast<const uint32_t *>(&v);
                        }
                    }
                    tc_st16(a_slot + (uint32_t)q * 16u, o);      // k-tile q / 2, its columns 16 * (q % 2) ..
                }
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&a_full[grp]);
                mbar_arrive(&empty_bar[s]);                        // the packed tiles have been read
            }
            s += NG;                                               // (the ring's length is a multiple of the groups)
            if (s >= S) { s -= S; ring_par ^= 1u; }
            a_par ^= 1u;
        }
    } else if (warp == 10) {
        // ------------------------------------------------------------------ watcher
        // polls the waves' second counters (all CTAs have written their slice of the activations) and publishes
        // them in shared memory, so that the producer never waits on global memory
        if (lane == 0) {
            const int W = 1 + (s_split < s_n_active ? 1 : 0);
            for (int w = 0; w < W; ++w) {
                bool ok = false;
                for (unsigned i = 0; i < (1u << 21); ++i) {
                    if (ld_acquire(&ws.sync[kTcReady - 4 + w]) >= P) { ok = true; break; }
                    __nanosleep(32);
                }
                if (!ok) { atomicExch(ws.status, ST_DEP_TIMEOUT); break; }
                __threadfence_block();
                s_ready[w] = 1;
            }
        }
    } else if (warp >= 7 && warp <= 9) {
        // ------------------------------------------------------------------ converter warps
        // per wave: wait for this CTA's hand-over, arrive on the wave's grid-wide counter, wait (bounded) for
        // all CTAs, convert this CTA's slice of the wave, arrive on the second counter
        const int et = tid - 224;                      // 0..95 among the converter threads
        uint32_t cv_phase = 0;
        const long long n_el = (long long)n_routed * sh.f + (long long)sh.n_sh * p.B * sh.f_sh;
        const int split = s_split, n_active = s_n_active, W = 1 + (split < n_active ? 1 : 0);
        const long long el_split = split < n_active ? (long long)act_offset(groups[split].off, n_routed, sh.f, sh.f_sh) : n_el;
        for (int w = 0; w < W; ++w) {
            // the hand-over may come late in the kernel: a long but bounded wait
            bool ok = false;
            for (unsigned i = 0; i < (1u << 22); ++i) {
                if (mbar_try_wait(&conv_go[w], 0)) { ok = true; break; }
                __nanosleep(24);
            }
            if (!ok) { if (lane == 0) atomicExch(ws.status, ST_MBAR_TIMEOUT); break; }
            if (et == 0) {
                tc_red_release(&ws.sync[kTcReady - 8 + w]);        // orders the CTA's reductions, observed through conv_go
                ok = false;
                for (unsigned i = 0; i < (kTcSpinLimit >> 2); ++i) {
                    if (ld_acquire(&ws.sync[kTcReady - 8 + w]) >= P) { ok = true; break; }
                    __nanosleep(16);
                }
                if (!ok) atomicExch(ws.status, ST_DEP_TIMEOUT);
                s_flag = ok;
            }
            if (!tc_bar(&cv_bar, cv_phase, lane) || !s_flag) break;
            __threadfence_block();                 // the counter was read with acquire by one thread of this barrier

            // pre holds a gate plane and an up plane, both indexed exactly like the activations (act_offset(slot)
            // + row): this CTA converts a contiguous slice of the wave's range, four elements per thread and step
            const long long w_lo = w ? el_split : 0, w_hi = w == W - 1 ? n_el : el_split;
            const long long n4 = (w_hi - w_lo) >> 2;
            const long long lo4 = n4 * blockIdx.x / P, hi4 = n4 * (blockIdx.x + 1) / P;
            // eight loads in flight per thread
            for (long long q0 = lo4 + et; q0 < hi4; q0 += 96 * 4) {
                float4 gv[4], uv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const long long q = q0 + 96 * u, i = w_lo + 4 * q;
                    if (q < hi4) {
                        gv[u] = __ldcg(reinterpret_cast<const float4 *>(p.pre + i));
                        uv[u] = __ldcg(reinterpret_cast<const float4 *>(p.pre + n_el + i));
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const long long q = q0 + 96 * u, i = w_lo + 4 * q;
                    if (q >= hi4) continue;
                    const float a0 = silu_mul(gv[u].x, uv[u].x), a1 = silu_mul(gv[u].y, uv[u].y), a2 = silu_mul(gv[u].z, uv[u].z),
                                a3 = silu_mul(gv[u].w, uv[u].w);
                    // binary16 hi + lo parts.  Columns i .. i + 3 of their group of 8 go to positions 0, 2, 4, 6 (first
                    // half of the group) or 1, 3, 5, 7 (second half): the order the dequantised weights are in
                    const __half2 h01 = __floats2half2_rn(a0, a1), h23 = __floats2half2_rn(a2, a3);
                    const __half2 l01 = __floats2half2_rn(a0 - __low2float(h01), a1 - __high2float(h01));
                    const __half2 l23 = __floats2half2_rn(a2 - __low2float(h23), a3 - __high2float(h23));
                    const long long o = (i & ~7ll) + ((i >> 2) & 1);
                    __half *ph = reinterpret_cast<__half *>(p.act_hi) + o, *pq = reinterpret_cast<__half *>(p.act_lo) + o;
                    ph[0] = __low2half(h01); ph[2] = __high2half(h01); ph[4] = __low2half(h23); ph[6] = __high2half(h23);
                    pq[0] = __low2half(l01); pq[2] = __high2half(l01); pq[4] = __low2half(l23); pq[6] = __high2half(l23);
                }
            }
            // the activations are read by TMA copies of other CTAs: proxy fence over global memory by every
            // writer, then one release at GPU scope behind the barrier of the converter warps
            asm volatile("fence.proxy.async.global;" ::: "memory");
            if (!tc_bar(&cv_bar, cv_phase, lane)) break;
            if (et == 0) tc_red_release(&ws.sync[kTcReady - 4 + w]);
        }
    } else if (warp >= 2 && warp <= 5) {
        // ------------------------------------------------------------------ epilogue warps
        const int q = warp & 3;                        // TMEM lane quarter this warp may read
        const long long n_el = (long long)n_routed * sh.f + (long long)sh.n_sh * p.B * sh.f_sh;
        uint32_t run = 0;
        int handed = 0, n_units = 0, W = 0;
        bool alive = tab_wait(0), tabs = false;
        if (alive) {
            n_units = s_n_units;
            W = 1 + (s_split < s_n_active ? 1 : 0);
        }
        // hand a wave over once this CTA's phase-1 units of it are all done (segment w is phase 1 of wave w)
        auto service = [&](int seg) {
            while (handed < W && seg > handed) {
                __syncwarp();
                if (lane == 0) mbar_arrive(&conv_go[handed]);
                ++handed;
            }
        };
        for (int ui = 0; ui < n_units && alive; ++ui) {
            uint4 un = unit_at(ui);
            service((int)(un.y >> 20));
            if (!(un.x & 6u)) continue;                // the run's accumulator is read after its last unit
            if (!tabs) {
                tabs = true;
                if (!tab_wait(1)) break;
                un = unit_at(ui);
            }
            if (!(un.x & 2u)) continue;
            const TcGroup &g = groups[un.y & 0xffffu];
            const int n = (int)(un.x >> 8), row = (int)un.z + q * 32 + lane;
            const uint32_t buf = run & 1u;
            const bool both = ACC == 64 && 2 * n > 64;                  // the run's two chains took both accumulators
            if (!mbar_wait(&acc_full[buf], (run >> 1) & 1u) || (both && !mbar_wait(&acc_full[buf ^ 1u], ((run + 1u) >> 1) & 1u))) {
                if (lane == 0) atomicExch(ws.status, ST_MBAR_TIMEOUT);
                alive = false;
                break;
            }
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + buf * (uint32_t)ACC;
            const bool p2 = (un.x & 4u) != 0;
            // slot of the expert's i-th token = g.off + i; walk its tokens in ascending order
            const int mi = (int)(un.y >> 16) & 15;
            float *dst = p.pre + (size_t)(mi >= 3 ? mi - 3 : mi) * n_el + act_offset(g.off, n_routed, sh.f, sh.f_sh) + row;
            const size_t f = (size_t)g.f;
            const uint32_t odd = both ? (buf ? 0u - 64u : 64u) : (uint32_t)n;   // columns from a chain to the odd K-steps' one
            for (int c = 0; c < n; c += 16) {
                float v[16];                           // phase 2: 8 hi, 8 lo of slots c / 2 .. c / 2 + 7
                if (both || 2 * n <= ACC) tc_ld16_sum(taddr + c, taddr + odd + c, v);
                else tc_ld16(taddr + c, v);
                if (c + 16 >= n) {                     // the accumulator may be overwritten
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive(&acc_empty[buf]);
                        if (both) mbar_arrive(&acc_empty[buf ^ 1u]);
                    }
                }
                if (!p2) {
                    const unsigned m16 = (unsigned)((g.mask >> c) & 0xffffull);
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if ((m16 >> i) & 1u) {
                            atomicAdd(dst, v[i]);
                            dst += f;
                        }
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int ti = (c >> 1) + i;
                        if (ti < g.T)
                            atomicAdd(&p.y[(size_t)s_slot_token[g.off + ti] * sh.d + row], s_slot_w[g.off + ti] * (v[i] + v[i + 8]));
                    }
                }
            }
            run += both ? 2u : 1u;
        }
        service(kQ4Segs);
    }
    // every path ends here (all waits above are bounded), so the TMEM is always returned
    tc_fence_before();
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

}  // namespace s2moe
