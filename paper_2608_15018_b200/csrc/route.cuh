// Router logits and reuse-aware expert gating (Sec. 4.2) for one draft batch.
//
//   route_kernel : l_{b,e} = h_b . W_r[e] (and the shared-expert gate logit) in float64, so
//                  that the discrete choices below do not depend on the summation order;
//                  block 0 then runs gating_block once every row has arrived:
//   gating_block : Eq. 4 aggregation, TopCap, lambda_b, biased top-k, mixing weights,
//                  union / unique count (gating.cuh), token->expert bucketing, stage tables.
#pragma once

#include "common.cuh"
#include "ffn_stream.cuh"
#include "gating.cuh"

namespace s2moe {


// What the expert kernels read of a finished gating (see gating_group for gm): the bucketing
// arrays in the workspace, tokens ascending inside an expert, the shared experts' groups behind
// the routed ones, and the stage tables of the streaming kernel.
__device__ __forceinline__ void gating_writeout(const Shape &sh, int B, const Workspace &ws, const GateMem &gm, int has_gate,
                                                int32_t *__restrict__ n_unique, const GateGroup gg)
{
    const int tid = gg.t, nt = gg.n;
    const int E = sh.E, k = sh.k;
    const int U = *gm.U, n_routed = B * k;
#pragma unroll 1
    for (int e = tid; e < E; e += nt) {
        ws.counts[e] = gm.cnt[e];
        ws.offsets[e] = gm.off[e];
        ws.tokmask[e] = gm.mask[e];
        if (gm.cnt[e] > 0) ws.active[gm.pos[e]] = e;
    }
    // bucket the (token, choice) pairs: tokens ascending inside an expert
#pragma unroll 1
    for (int i = tid; i < n_routed; i += nt) {
        const int b = i / k;
        const int e = gm.sel[i];
        const int pos = gm.off[e] + __popcll(gm.mask[e] & ((1ull << b) - 1ull));
        ws.slot_token[pos] = b;
        ws.slot_w[pos] = gm.pw[i];
    }
    // shared experts: every token, weight c_b
    const unsigned long long all = B >= 64 ? ~0ull : ((1ull << B) - 1ull);
#pragma unroll 1
    for (int i = tid; i < sh.n_sh * B; i += nt) {
        const int s = i / B, b = i - s * B;
        float c = 1.0f;
        if (has_gate) c = (float)(1.0 / (1.0 + exp_once(-__ldcg(&ws.gate_logit[b]))));
        ws.slot_token[n_routed + i] = b;
        ws.slot_w[n_routed + i] = c;
        if (b == 0) {
            ws.counts[E + s] = B;
            ws.offsets[E + s] = n_routed + s * B;
            ws.active[U + s] = E + s;
            ws.tokmask[E + s] = all;
        }
    }
    if (sh.plan == 2) {
        // stage tables of the streaming kernel: per active group, its first phase-1 stage
        // (4 gate + 4 up rows each) and first phase-2 stage (8 down rows x one K-slice)
        gate_sync(gg);
#pragma unroll 1
        for (int e = tid; e < E; e += nt)
            gm.cnt[e] = gm.cnt[e] > 0 ? st_nks(sh.f, gm.cnt[e], sh.op_cap, sh.d) * (sh.d / 8) : 0;   // phase-2 stages
        gate_sync(gg);
#pragma unroll 1
        for (int e = tid; e < E; e += nt) {
            if (gm.mask[e]) {
                int pre = 0;
#pragma unroll 1
                for (int o = 0; o < e; ++o) pre += gm.cnt[o];
                const int a = gm.pos[e];
                ws.upfx1[a] = a * (sh.f / 4);
                ws.upfx2[a] = pre;
                ws.sync[a] = 0;
                if (a == U - 1) gm.off[0] = pre + gm.cnt[e];   // all routed phase-2 stages
            }
        }
        gate_sync(gg);
        if (tid == 0) {
            int t1 = U * (sh.f / 4), t2 = gm.off[0];
#pragma unroll 1
            for (int s = 0; s <= sh.n_sh; ++s) {
                ws.upfx1[U + s] = t1;
                ws.upfx2[U + s] = t2;
                ws.sync[U + s] = 0;
                if (s < sh.n_sh) {
                    t1 += sh.f_sh / 4;
                    t2 += st_nks(sh.f_sh, B, sh.op_cap, sh.d) * (sh.d / 8);
                }
            }
            ws.header[4] = t1;
            ws.header[5] = t2;
        }
    }
    if (tid == 0) {
        ws.offsets[E + sh.n_sh] = n_routed + sh.n_sh * B;
        ws.header[0] = U + sh.n_sh;
        ws.header[1] = n_routed + sh.n_sh * B;
        ws.header[2] = U;
        ws.header[3] = B;
        *n_unique = U;
    }
}

// Gating of one batch by a whole thread block (kRouteThreads threads) on the logits in the workspace.
// s_l: shared memory for B * E + B doubles (the logits and the confidences are staged there) and, behind
// them, gate_mem_bytes(E, B, k).
// repair(): called by the block if `nonfinite`, with the logits staged (repair_logits).
template <int JE, class Repair>
__device__ __forceinline__ void gating_block(const Shape &sh, int B, const Workspace &ws, const float *__restrict__ conf,
                                             int has_gate, int32_t *__restrict__ sel_idx, float *__restrict__ sel_w,
                                             int32_t *__restrict__ n_unique, double *s_l, int ksplit, const double *__restrict__ lpart,
                                             int early, bool nonfinite, Repair repair)
{
    // (sized by this batch and not for the largest one: a routing block shares its SM with the expert kernel)
    const GateMem gm = gate_mem_carve(s_l + ((B * sh.E + B + 1) & ~1), sh.E, B, sh.k);
    const GateGroup gg{(int)threadIdx.x, (int)blockDim.x, 0};
    double *s_w = s_l + B * sh.E;
    if (ksplit > 0) {
        // the pieces of a row added in ascending order (all loads first); the sums go back to the
        // workspace, where the write-out (gate logits) and debug reads find them
        const int n_rows = sh.E + has_gate;
#pragma unroll 1
        for (int i = gg.t; i < B * n_rows; i += gg.n) {
            const int b = i / n_rows, r = i - b * n_rows;
            double v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = q < ksplit ? __ldcg(&lpart[((size_t)q * B + b) * n_rows + r]) : 0.0;
            double acc = v[0];
#pragma unroll
            for (int q = 1; q < 8; ++q) acc += v[q];
            if (r < sh.E) { s_l[b * sh.E + r] = acc; ws.logits[b * sh.E + r] = acc; }
            else ws.gate_logit[b] = acc;
        }
    } else {
#pragma unroll 1
        for (int i = gg.t; i < B * sh.E; i += gg.n) s_l[i] = __ldcg(&ws.logits[i]);
    }
#pragma unroll 1
    for (int b = gg.t; b < B; b += gg.n) s_w[b] = conf ? (double)conf[b] : 1.0;
    __syncthreads();                                      // the logits are staged
    if (nonfinite) repair();
    gating_part1<JE>(sh, B, s_l, s_w, gg, gm);
    gating_part2<JE>(sh, B, s_l, gg, gm, sel_idx, sel_w, early ? ws.early : nullptr);
    gating_writeout(sh, B, ws, gm, has_gate, n_unique, gg);
}

constexpr int kRouteThreads = 512;
constexpr int kRouteThreadsBig = 1024;
constexpr int kRouteTok = 16;   // most tokens accumulated per pass

// Buffers that the layer's later kernels accumulate into and that must start at zero; the
// routing blocks clear them (16-byte units) so that no separate fill precedes the layer.
// 4 consecutive elements of a plain (f32 / bf16) row starting at column c (c % 4 == 0)
template <int DT>
__device__ __forceinline__ void load4_plain(const void *row, int c, float (&v)[4])
{
    if (DT == DT_F32) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(row) + c));
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    } else {
        const uint2 a = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(row) + c));
        v[0] = bf16_lo(a.x); v[1] = bf16_hi(a.x); v[2] = bf16_lo(a.y); v[3] = bf16_hi(a.y);
    }
}

// two bf16 values -> two binary16 values (round to nearest; exact for magnitudes in [2^-14, 65504])
__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t u)
{
    const __half2 h = __floats2half2_rn(bf16_lo(u), bf16_hi(u));
    return *reinterpret_cast<const uint32_t *>(&h);
}

struct ZeroList {
    void *ptr[3];
    unsigned long long n16[3];
    // int4 tensor-core path: a binary16 copy of the bf16 hidden states whose columns are permuted
    // inside every group of 8 (position p holds column [0,4,1,5,2,6,3,7][p]), the order in which
    // the dequantising warps of the expert kernel get the nibbles of a 32-bit word for free
    const uint4 *perm_src;
    uint4 *perm_dst;
    unsigned long long perm_n16;
    // logit pass: the tokens of a batch are split into this many groups, each with its own set of
    // row blocks (0 and 1: every row block takes all tokens)
    int groups;
    // logit pass by warp tasks (larger batches): ksplit > 0 pieces of the contraction per router row,
    // partial sums in lpart [piece][token][row] (see route_logit_tasks); 0: by row blocks
    int ksplit;
    double *lpart;
    // 1: the expert kernel behind this launch starts before the gating has ended, on the experts of largest
    // aggregated importance (see gsum); it reads what Workspace::early holds
    int early;
};

// Sums over the warp of NT values per lane in log2(32) steps for all of them together (halving the
// number of values a lane holds while that is more than one): lane l ends up with the sum of value
// l / (32 / NT).  16 values take 16 + 1 shuffles instead of 80.
template <int NT>
__device__ __forceinline__ double warp_sums(double (&a)[NT], int lane)
{
    int o = 16;
#pragma unroll
    for (int n = NT / 2; n > 0; n >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int t = 0; t < n; ++t) {
            const double send = up ? a[t] : a[t + n], keep = up ? a[t + n] : a[t];
            a[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    return a[0];
}

// x * 2^-896 exactly for every finite x, subnormal numbers included, by moving the bits of the binary32
// number into place (a conversion instruction has a quarter of the rate of the fused multiply-add it
// feeds); the other factor carries the 2^896.  An infinity or a NaN comes out as some finite number: a batch
// that holds one is found by nonfinite_scan, and its tokens get their logits from repair_logits.
__device__ __forceinline__ double scaled_double(float x, bool bf16)
{
    const uint32_t u = __float_as_uint(x);
    return __hiloint2double((int)(((u >> 3) & 0x0fffffffu) | (u & 0x80000000u)), bf16 ? 0 : (int)(u << 29));
}

// Whether the thread's share of n16 16-byte units (thread t of n) holds an infinity or a NaN: an exponent field
// of all ones carries into the sign's place.  Block 0, which has no logits to form, looks through the batch while
// it waits for the others, eight loads in flight per thread (256 KB, 64 tokens of 2048, in some 3 us).
// Measured against the alternatives in the logit pass itself (0 * x summed beside it) and in slices
// beside it (marks in memory that block 0 collects): those cost 0.6 to 1.1 us per layer at 13 and 64 tokens, and at 1.
template <int ACT>
__device__ __forceinline__ bool nonfinite_scan(const void *__restrict__ hidden, int n16, int t, int n)
{
    const uint32_t keep = ACT == DT_F32 ? 0x7fffffffu : 0x7fff7fffu, one = ACT == DT_F32 ? 0x00800000u : 0x00800080u;
    uint32_t bad = 0u;
#pragma unroll 1
    for (int i = t; i < n16; i += 8 * n) {
        uint4 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            v[j] = i + j * n < n16 ? __ldg(reinterpret_cast<const uint4 *>(hidden) + i + j * n) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            bad |= ((v[j].x & keep) + one) | ((v[j].y & keep) + one) | ((v[j].z & keep) + one) | ((v[j].w & keep) + one);
    }
    return (bad & ~keep) != 0u;
}

// The logits of the tokens with an infinity or a NaN by plain float64 arithmetic on the stored values (a warp per
// token and row), by a whole block; s_l [B][E] and the workspace get them.  Out of line: it runs for no other batch.
template <int ACT, int RT>
__device__ __noinline__ void repair_logits(int B, int d, int E, int n_rows, const void *hidden, const void *router, const void *sh_scale,
                                           double *s_l, double *logits, double *gate_logit)
{
    __shared__ unsigned long long s_marks;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const size_t row = (size_t)d * (ACT == DT_F32 ? 4 : 2);
    if (threadIdx.x == 0) s_marks = 0ull;
    __syncthreads();
    for (int b = warp; b < B; b += nw)
        if (nonfinite_scan<ACT>(reinterpret_cast<const uint8_t *>(hidden) + (size_t)b * row, (int)(row / 16), lane, 32))
            atomicOr(&s_marks, 1ull << b);
    __syncthreads();
    for (unsigned long long marks = s_marks; marks; marks &= marks - 1ull) {
        const int b = __ffsll((long long)marks) - 1;
        for (int r = warp; r < n_rows; r += nw) {
            const uint8_t *w = r < E ? reinterpret_cast<const uint8_t *>(router) + (size_t)r * d * (RT == DT_F32 ? 4 : 2)
                                     : reinterpret_cast<const uint8_t *>(sh_scale);
            double v = 0.0;
            for (int c = lane * 4; c < d; c += 128) {
                float a[4], h[4];
                load4_plain<RT>(w, c, a);
                load4_plain<ACT>(reinterpret_cast<const uint8_t *>(hidden) + (size_t)b * row, c, h);
#pragma unroll
                for (int i = 0; i < 4; ++i) v = fma((double)a[i], (double)h[i], v);
            }
            v = warp_sum(v);
            if (lane == 0) {
                if (r < E) s_l[b * E + r] = logits[b * E + r] = v;
                else gate_logit[b] = v;
            }
        }
    }
    __syncthreads();
}

// Router logits by the warps of the whole grid: a task is one router row (row E: the shared
// experts' gate vector) x 8 tokens x one piece of the contraction, float64 accumulation; its
// partial sums go to lpart[piece][token][row], which the gating adds up in a fixed order.
// EXACT: by conversion instructions, for a caller that does not look for infinities and NaN (see scaled_double).
template <int ACT, int RT, bool EXACT>
__device__ __forceinline__ void route_logit_tasks(const Shape &sh, int B, const void *__restrict__ hidden,
                                                  const void *__restrict__ router, const void *__restrict__ sh_scale,
                                                  double *__restrict__ lpart, int ksplit, const float *__restrict__ conf,
                                                  float *__restrict__ gsum, int gwarp, int n_gwarps, int lane)
{
    const int d = sh.d, n_rows = sh.E + (sh_scale ? 1 : 0), n_tg = (B + 7) >> 3;
    const int len = ((d + 4 * ksplit - 1) / (4 * ksplit)) * 4;              // columns of a piece, a multiple of 4
    const int n_tasks = n_rows * n_tg * ksplit;
    const size_t rb = RT == DT_F32 ? 4 : 2, ab = ACT == DT_F32 ? 4 : 2;
#pragma unroll 1
    for (int task = gwarp; task < n_tasks; task += n_gwarps) {
        const int row = task % n_rows, rest = task / n_rows, tg = rest % n_tg, piece = rest / n_tg;
        const int c0 = piece * len, c1 = min(d, c0 + len), b0 = tg * 8;
        const uint8_t *wrow = row < sh.E ? reinterpret_cast<const uint8_t *>(router) + (size_t)row * d * rb
                                         : reinterpret_cast<const uint8_t *>(sh_scale);
        double acc[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) acc[t] = 0.0;
#pragma unroll 2
        for (int c = c0 + lane * 4; c < c1; c += 128) {
            float w[4], x[8][4];
            load4_plain<RT>(wrow, c, w);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                const int bt = min(b0 + t, B - 1);           // past the batch: the last token again (not stored)
                load4_plain<ACT>(reinterpret_cast<const uint8_t *>(hidden) + (size_t)bt * d * ab, c, x[t]);
            }
            double wd[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) wd[i] = EXACT ? (double)w[i] : (double)w[i] * 0x1p896;
#pragma unroll
            for (int t = 0; t < 8; ++t)
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    acc[t] = fma(wd[i], EXACT ? (double)x[t][i] : scaled_double(x[t][i], ACT == DT_BF16), acc[t]);
        }
        const double v = warp_sums<8>(acc, lane);             // token lane / 4
        const int bt = b0 + (lane >> 2);
        float g = 0.0f;
        if ((lane & 3) == 0 && bt < B) {
            lpart[((size_t)piece * B + bt) * n_rows + row] = v;
            g = (gsum && conf ? conf[bt] : 1.0f) * (float)v;
        }
        if (gsum && row < sh.E) {
#pragma unroll
            for (int o = 16; o > 2; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
            if (lane == 0) atomicAdd(&gsum[row], g);
        }
    }
}

// One pass of a router row over NT tokens b0 .. b0 + NT - 1 (indices past B - 1 repeat token
// B - 1, so that every load is unconditional and issued before the first use).
template <int ACT, int RT, int NT>
__device__ __forceinline__ void route_pass(const Shape &sh, int B, int b0, const Workspace &ws, int row, const uint8_t *wrow,
                                           const void *__restrict__ hidden, const float *__restrict__ conf, float *__restrict__ gsum,
                                           double *s_part)
{
    static_assert(kRouteThreads == 32 * 16 && NT <= 16, "16 partial sums per token");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, d = sh.d;
    const size_t ab = ACT == DT_F32 ? 4 : 2;
    const int tok = tid >> 4;                             // token whose partial sums this thread adds up at the end
    const bool mine = tok < NT && b0 + tok < B;
    const float wb = (gsum && conf && mine) ? conf[b0 + tok] : 1.0f;
    double acc[NT];
#pragma unroll
    for (int t = 0; t < NT; ++t) acc[t] = 0.0;
    for (int c = tid * 4; c < d; c += kRouteThreads * 4) {
        float w[4], x[NT][4];
        load4_plain<RT>(wrow, c, w);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
            const int bt = min(b0 + t, B - 1);
            load4_plain<ACT>(reinterpret_cast<const uint8_t *>(hidden) + (size_t)bt * d * ab, c, x[t]);
        }
        double wd[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) wd[i] = (double)w[i] * 0x1p896;
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[t] = fma(wd[i], scaled_double(x[t][i], ACT == DT_BF16), acc[t]);
    }
    const double v = warp_sums<NT>(acc, lane);
    if ((lane & (32 / NT - 1)) == 0) s_part[warp * kRouteTok + lane / (32 / NT)] = v;
    __syncthreads();
    if (tid < 16 * NT) {                                  // (whole warps: two tokens each)
        double s = s_part[(tid & 15) * kRouteTok + tok];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        float g = mine ? wb * (float)s : 0.0f;
        if ((tid & 15) == 0 && mine) {
            if (row < sh.E) ws.logits[(size_t)(b0 + tok) * sh.E + row] = s;
            else ws.gate_logit[b0 + tok] = s;
        }
        if (gsum && row < sh.E) {
            g += __shfl_xor_sync(0xffffffffu, g, 16);
            if (lane == 0) atomicAdd(&gsum[row], g);
        }
    }
    __syncthreads();
}

// Router logits and gating in one launch.  A block computes one row of the router (row E is the
// shared-expert gate vector) against one group of the batch's tokens in float64; block 0, which has no
// row, runs the gating for the whole batch once every block has arrived (atomic ticket).
// Dynamic shared memory: B * E + B doubles and gate_mem_bytes(E, B, k), at least 16 * kRouteTok doubles.
// JE: experts per lane in the gating (2, 4 or 8 for up to 64, 128, 256 experts): a kernel of its own
// for each, so that the gating code of a launch is one straight piece
// THREADS: kRouteThreads, or kRouteThreadsBig for the kernel of the larger batches (warp tasks only)
template <int ACT, int RT, int JE, int THREADS>
__device__ __forceinline__ void route_body(const Shape &sh, int B, const Workspace &ws, const void *__restrict__ hidden,
                                           const void *__restrict__ router, const void *__restrict__ sh_scale,
                                           const float *__restrict__ conf, int32_t *__restrict__ sel_idx,
                                           float *__restrict__ sel_w, int32_t *__restrict__ n_unique, const ZeroList &zl)
{
    extern __shared__ __align__(16) double s_dyn[];       // (the gating reads parts of it 16 bytes at a time)
    __shared__ int s_last;
    const int tid = threadIdx.x;
    // Programmatic dependent launch: everything this kernel writes is read by the kernels of the layer in
    // front, so it waits for them before it does; only the lists that the expert kernel of this layer
    // polls are cleared before (the expert kernel in front lets this grid start once it has read
    // them).  The expert kernel of this layer may come up once every block has passed
    // launch_dependents, that is, while the layer in front still runs: it sets itself up and
    // streams weights that do not depend on any routing.  (Both instructions do nothing in a plain launch.)
    if (zl.early && blockIdx.x == 0) {
        if (tid <= kEarlyWords) {
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(ws.early + tid), "l"(0ull) : "memory");
            __threadfence();
        }
        __syncthreads();
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // what this block will read first, into L2 while it waits: its router row (the hidden states come from
    // the kernel in front and are there already, or from the caller's memory: a prefetch changes nothing)
    if (zl.ksplit == 0 && blockIdx.x > 0) {
        const int row_p = ((int)blockIdx.x - 1) % (sh.E + (sh_scale ? 1 : 0));
        const size_t rbytes = (size_t)sh.d * (RT == DT_F32 ? 4 : 2), hbytes = (size_t)B * sh.d * (ACT == DT_F32 ? 4 : 2);
        const uint8_t *wr = row_p < sh.E ? reinterpret_cast<const uint8_t *>(router) + (size_t)row_p * rbytes
                                         : reinterpret_cast<const uint8_t *>(sh_scale);
        const size_t o = (size_t)tid * 128;
        if (o < rbytes) asm volatile("prefetch.global.L2 [%0];" ::"l"(wr + o));
        const size_t ho = ((size_t)(blockIdx.x - 1) * THREADS + tid) * 128;
        if (ho < hbytes) asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const uint8_t *>(hidden) + ho));
    }
    const int n_rows = sh.E + (sh_scale ? 1 : 0), n_grp = zl.groups > 1 ? zl.groups : 1;
    const int n_arrive = zl.ksplit > 0 ? (int)gridDim.x - 1 : n_rows * n_grp;   // blocks 1 .. n_arrive; those past that only clear
    const int rblk = (int)blockIdx.x - 1;
    const size_t rb = RT == DT_F32 ? 4 : 2;
    // block 0: where the arrival counter stood when the launch before had ended (that launch is over: a
    // kernel lets this one start only when its own routing kernel has ended); see below
    unsigned ticket_target = 0u;
    if (blockIdx.x == 0 && tid == 0) {
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(ticket_target) : "l"(ws.ticket + 1) : "memory");
        ticket_target += (unsigned)n_arrive;
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (zl.early && blockIdx.x == 0 && tid == 0)
        asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(ws.early + kEarlyWords), "l"((1ull << 32) | (unsigned long long)ticket_target)
                     : "memory");
    // (before the logit pass, whose end and arrival release it: the expert kernel copies it with TMA as soon as
    // all blocks have arrived)
    if (zl.perm_n16 && rblk >= 0 && rblk < n_arrive) {
        for (unsigned long long i = (unsigned long long)rblk * THREADS + tid; i < zl.perm_n16; i += (unsigned long long)n_arrive * THREADS) {
            const uint4 v = zl.perm_src[i];             // halves h0..h7 (bf16)
            zl.perm_dst[i] = make_uint4(bf16x2_to_f16x2(__byte_perm(v.x, v.z, 0x5410)), bf16x2_to_f16x2(__byte_perm(v.x, v.z, 0x7632)),
                                        bf16x2_to_f16x2(__byte_perm(v.y, v.w, 0x5410)), bf16x2_to_f16x2(__byte_perm(v.y, v.w, 0x7632)));
        }
        asm volatile("fence.proxy.async.global;" ::: "memory");
    }
    // A row block takes one router row and one group of tokens: a larger batch is split over
    // several sets of row blocks (as many as fit on the SMs beside each other), because a block
    // takes 16 tokens per pass and its passes run one after the other (B = 64: 22 us in one set).
    if (zl.ksplit > 0) {
        // larger batches: the logit pass as warp tasks over all blocks but the first
        if (rblk >= 0)
            route_logit_tasks<ACT, RT, false>(sh, B, hidden, router, sh_scale, zl.lpart, zl.ksplit, conf, zl.early ? ws.gsum : nullptr, (tid >> 5) * n_arrive + rblk,
                                       (THREADS / 32) * n_arrive, tid & 31);
        __syncthreads();
    } else if constexpr (THREADS == kRouteThreads) {
        if (rblk >= 0 && rblk < n_arrive) {
            const int row = rblk % n_rows, grp = rblk / n_rows;
            const int tg = 4 * ((B + 4 * n_grp - 1) / (4 * n_grp));            // tokens per group, a multiple of 4
            const int b_lo = min(B, grp * tg), b_hi = min(B, b_lo + tg);
            const uint8_t *wrow = row < sh.E ? reinterpret_cast<const uint8_t *>(router) + (size_t)row * sh.d * rb
                                             : reinterpret_cast<const uint8_t *>(sh_scale);
            float *const gsum = zl.early ? ws.gsum : nullptr;
            for (int b0 = b_lo; b0 < b_hi;) {
                const int left = b_hi - b0;
                if (left > 8) { route_pass<ACT, RT, 16>(sh, B, b0, ws, row, wrow, hidden, conf, gsum, s_dyn); b0 += 16; }
                else if (left > 4) { route_pass<ACT, RT, 8>(sh, B, b0, ws, row, wrow, hidden, conf, gsum, s_dyn); b0 += 8; }
                else { route_pass<ACT, RT, 4>(sh, B, b0, ws, row, wrow, hidden, conf, gsum, s_dyn); b0 += 4; }
            }
        }
    }
    // Block 0 runs the gating once every row has arrived (its SM tends to be the same from layer
    // to layer, so part of the gating code is still in its instruction cache: measured 0.6 % of
    // a layer against letting the last block to arrive do it).  Every row block adds one arrival, released
    // by one thread, to a counter that is never reset; block 0
    // polls it, bounded, for the value it has when all blocks of THIS launch have arrived: the
    // value it will end on was left in the word behind the counter by the launch before (launches of
    // a context follow each other in stream order), and block 0 leaves the next one there, whether
    // its wait succeeded or not, since the late blocks still arrive.  So a wait that ran out poisons
    // nothing, and the waiting path is one reduction and one polled load, as short as it can be.  The
    // barriers on both sides extend the ordering to the block's other threads; the other blocks
    // wait for nothing.
    // The arrival is one thread's and covers the whole block only behind a barrier.  A logit pass ends with one,
    // but a row block whose group of tokens is empty (12 rows, 64 tokens: 12 groups of 8 tokens, 4 of them empty)
    // makes no pass and has written its part of the binary16 copy all the same.
    if (zl.perm_n16) __syncthreads();
    if (tid == 0 && rblk >= 0 && rblk < n_arrive)
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ws.ticket) : "memory");
    if (blockIdx.x == 0 && tid == 0) {
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(ws.ticket + 1), "r"(ticket_target) : "memory");
        int ok = 0;
        for (unsigned i = 0; i < (1u << 22) && !ok; ++i) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ws.ticket) : "memory");
            if ((int)(v - ticket_target) >= 0) ok = 1;
            else __nanosleep(20);
        }
        if (!ok) atomicExch(ws.status, ST_TICKET_TIMEOUT);
        s_last = ok;
    }
    bool bad = false;
    if (blockIdx.x == 0 && tid >= 32) bad = nonfinite_scan<ACT>(hidden, B * sh.d / (ACT == DT_F32 ? 4 : 8), tid - 32, THREADS - 32);
    // What the kernels behind accumulate into is cleared after the arrival (they touch it once this grid
    // has ended), by all blocks but the one that runs the gating.
    if (blockIdx.x > 0) {
        const unsigned first = blockIdx.x - 1u, blocks = gridDim.x - 1u;
#pragma unroll
        for (int z = 0; z < 3; ++z) {
            uint4 *p = reinterpret_cast<uint4 *>(zl.ptr[z]);
            for (unsigned long long i = (unsigned long long)first * THREADS + tid; i < zl.n16[z]; i += (unsigned long long)blocks * THREADS)
                p[i] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
    if (blockIdx.x > 0) return;
    bad = __syncthreads_or(bad) != 0;
    if (!s_last) return;
    gating_block<JE>(sh, B, ws, conf, sh_scale ? 1 : 0, sel_idx, sel_w, n_unique, s_dyn, zl.ksplit, zl.lpart, zl.early, bad,
                     [&]() { repair_logits<ACT, RT>(B, sh.d, sh.E, n_rows, hidden, router, sh_scale, s_dyn, ws.logits, ws.gate_logit); });
}

// (bound of 768 threads instead of 512: at most 80 registers, so that a block fits beside a CTA of the
// expert kernel, 352 threads x 64 registers)
template <int ACT, int RT, int JE>
__global__ void __launch_bounds__(768, 1)
route_kernel(Shape sh, int B, Workspace ws, const void *__restrict__ hidden, const void *__restrict__ router,
             const void *__restrict__ sh_scale, const float *__restrict__ conf, int32_t *__restrict__ sel_idx,
             float *__restrict__ sel_w, int32_t *__restrict__ n_unique, ZeroList zl)
{
    route_body<ACT, RT, JE, kRouteThreads>(sh, B, ws, hidden, router, sh_scale, conf, sel_idx, sel_w, n_unique, zl);
}

// The same with twice the warps, for the larger batches (logit pass by warp tasks only): the gating
// takes one warp per token, and at 64 tokens four passes of 16 warps were most of the kernel.
template <int ACT, int RT, int JE>
__global__ void __launch_bounds__(kRouteThreadsBig)
route_kernel_big(Shape sh, int B, Workspace ws, const void *__restrict__ hidden, const void *__restrict__ router,
                 const void *__restrict__ sh_scale, const float *__restrict__ conf, int32_t *__restrict__ sel_idx,
                 float *__restrict__ sel_w, int32_t *__restrict__ n_unique, ZeroList zl)
{
    route_body<ACT, RT, JE, kRouteThreadsBig>(sh, B, ws, hidden, router, sh_scale, conf, sel_idx, sel_w, n_unique, zl);
}

}  // namespace s2moe
