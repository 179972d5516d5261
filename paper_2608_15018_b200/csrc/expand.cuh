// Routing-aware adaptive speculative expansion (Sec. 4.1): predicted expert sets as bit
// masks, marginal verification cost (Eq. 2), utility (Eq. 3) and the greedy admission loop.
// The step that chooses the draft batch which the verification layer then runs on.
#pragma once

#include <cstdint>

#include "gating.cuh"

namespace s2moe {

constexpr int kExpandMaxCand = 256;     // candidates per call (one thread each)
constexpr int kExpandMaxWords = 512;    // n_layers * ceil(n_experts / 64)
constexpr int kExpandThreads = 512;
constexpr int kExpandMaxSmem = 200 * 1024;   // rows of all candidates in shared memory up to this size

// masks[t * stride + w]: bit (e % 64) of word (e / 64) set for every expert e in sel_idx[t][*]
__global__ void expert_masks_kernel(const int32_t *__restrict__ sel_idx, int n_tokens, int k, int words,
                                    unsigned long long *__restrict__ masks, int stride)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tokens) return;
    for (int w = 0; w < words; ++w) {
        unsigned long long m = 0ull;
        for (int j = 0; j < k; ++j) {
            const int e = sel_idx[t * k + j];
            if ((e >> 6) == w) m |= 1ull << (e & 63);
        }
        masks[(size_t)t * stride + w] = m;
    }
}

// Prefix confidence p_i = p_parent * p_{i,j} into s_p, block of 32 candidates by block: parents precede their
// children, so a block needs earlier blocks (shared memory) and itself (shuffles).  A parent index that
// does not precede is not followed: the candidate gets confidence 0, is never eligible (nor are its
// descendants) and the call reports it.  Thread i of the block takes candidate i.
__device__ __forceinline__ bool expand_prefix(int n, const int32_t *__restrict__ parent, const float *__restrict__ p_tok, double *s_p)
{
    const int i = threadIdx.x, lane = i & 31, warp = i >> 5, nw = (n + 31) >> 5;
    const int par_in = i < n ? parent[i] : -1;
    const bool malformed = i < n && par_in >= i;
    const int par = malformed ? -1 : par_in;
    const float pt = i < n ? p_tok[i] : 0.0f;
    for (int b = 0; b < nw; ++b) {
        if (warp == b) {
            double v = malformed ? 0.0 : (double)pt;
            bool done = i >= n || par < 0;
            const bool inside = !done && par >= 32 * b;
            if (!done && !inside) { v = __dmul_rn(s_p[par], v); done = true; }
            while (!__all_sync(0xffffffffu, done)) {
                const int src = inside ? par & 31 : lane;
                const double pv = __shfl_sync(0xffffffffu, v, src);
                const int there = __shfl_sync(0xffffffffu, (int)done, src);
                if (!done && there) { v = __dmul_rn(pv, v); done = true; }
            }
            if (i < n) s_p[i] = v;
        }
        __syncthreads();
    }
    return malformed;
}

// Utility of a candidate (Eq. 2 and Eq. 3) as an order-preserving key, 0 where it is not a number; float64 with
// every operation rounded on its own (no fused multiply-add), so that the decisions are those of the plain definition.
__device__ __forceinline__ unsigned long long expand_key(double benefit, int fresh, double t_exp, double c_draft)
{
    const double cost = __dadd_rn(__dmul_rn((double)fresh, t_exp), c_draft);                              // Eq. 2
    const double u = cost == 0.0 ? __longlong_as_double(0x7ff0000000000000ll) : __ddiv_rn(benefit, cost);   // Eq. 3
    return u == u ? dkey(u) : 0ull;
}

// One block.  Thread i < n owns candidate i: its utility, and its place in the search for the largest one.
// The sets are what costs: after every admission the experts it brought are new to nobody any more.  So
// the kernel keeps, per word and candidate, only the bits NOT yet in the union (s_rem, candidates side by
// side, so that a warp reads neighbouring banks) and their number per candidate (s_fresh).  An
// admission of b makes a list of the words in which b brings anything, and only those are visited: by
// all threads, thread t at candidate t mod np, several threads sharing a candidate's words.  All arithmetic
// that decides an admission is float64 with every operation rounded on its own (no fused
// multiply-add), so that the decisions are those of the plain definition.
// Bound by latency: three block barriers and one float64 division (some 400 cycles) per admission.
// Measured, us per call, where s2moe_adaptive_expand uses it: 96 candidates x 24 words 109, 128 x 64 175, 256 x 16 277, 160 x 96
// 262 (770 with every candidate counting all its words again for every admission).
// SMEM: the rows fit shared memory; else they are read from global memory.
template <bool SMEM>
__global__ void __launch_bounds__(kExpandThreads)
adaptive_expand_kernel(int n, int lw, const int32_t *__restrict__ parent, const float *__restrict__ p_tok,
                       const unsigned long long *__restrict__ masks, const float *__restrict__ c_draft, float t_ar,
                       float t_exp, int32_t *__restrict__ admitted, int32_t *__restrict__ order,
                       int32_t *__restrict__ n_admitted, unsigned long long *__restrict__ union_out)
{
    extern __shared__ unsigned long long s_rem[];                       // [lw][n | 1]
    __shared__ double s_p[kExpandMaxCand];
    __shared__ int s_adm[kExpandMaxCand], s_fresh[kExpandMaxCand];
    __shared__ unsigned long long s_union[kExpandMaxWords], s_new[kExpandMaxWords];   // s_new, s_word: the list of an admission
    __shared__ int s_word[kExpandMaxWords];
    __shared__ unsigned long long s_wk[kExpandMaxCand / 32];
    __shared__ int s_wi[kExpandMaxCand / 32], s_best, s_words;

    const int i = threadIdx.x, lane = i & 31, warp = i >> 5, nw = (n + 31) >> 5;
    const int np = nw * 32, pitch = n | 1, c_mine = i % np, part = i / np, parts = (int)blockDim.x / np;
    const int par = i < n ? parent[i] : -1;
    const double cd = (i < n && c_draft) ? (double)c_draft[i] : 0.0;
    if (i < n) { s_adm[i] = 0; s_fresh[i] = 0; }
    for (int w = i; w < lw; w += blockDim.x) s_union[w] = 0ull;
    if (SMEM)
        for (int c = warp; c < n; c += (int)blockDim.x >> 5)
            for (int w = lane; w < lw; w += 32) s_rem[w * pitch + c] = masks[(size_t)c * lw + w];
    const bool malformed = expand_prefix(n, parent, p_tok, s_p);
    const int bad = __syncthreads_or(malformed ? 1 : 0);
    const double benefit = i < n ? __dmul_rn(s_p[i], (double)t_ar) : 0.0;
    if (part < parts && c_mine < n) {
        int cnt = 0;
        for (int w = part; w < lw; w += parts) cnt += __popcll(SMEM ? s_rem[w * pitch + c_mine] : masks[(size_t)c_mine * lw + w]);
        if (cnt) atomicAdd(&s_fresh[c_mine], cnt);
    }
    __syncthreads();

    int count = 0;
    for (int step = 0; step < n; ++step) {
        if (warp < nw) {
            unsigned long long key = 0ull;                               // 0: not eligible (or not a number)
            if (i < n && !malformed && !s_adm[i] && (par < 0 || s_adm[par])) key = expand_key(benefit, s_fresh[i], (double)t_exp, cd);
            // largest utility, lowest index on ties
            const int wl = __ffs(warp_max_holders(key, true)) - 1;
            if (lane == wl) { s_wk[warp] = key; s_wi[warp] = i; }
        }
        __syncthreads();
        if (warp == 0) {
            const unsigned long long k = lane < nw ? s_wk[lane] : 0ull;
            const int wl = __ffs(warp_max_holders(k, true)) - 1;
            const int b = s_wi[wl];
            const unsigned long long bk = shfl_key(k, wl);
            const bool go = bk != 0ull && dkey_value(bk) >= 1.0;
            if (go) {
                int words = 0;
                for (int w0 = 0; w0 < lw; w0 += 32) {
                    const int w = w0 + lane;
                    unsigned long long nb = 0ull;
                    if (w < lw) nb = SMEM ? s_rem[w * pitch + b] : masks[(size_t)b * lw + w] & ~s_union[w];
                    const unsigned some = __ballot_sync(0xffffffffu, nb != 0ull);
                    if (nb != 0ull) {
                        const int at = words + __popc(some & ((1u << lane) - 1u));
                        s_new[at] = nb;
                        s_word[at] = w;
                        s_union[w] |= nb;
                    }
                    words += __popc(some);
                }
                if (lane == 0) {
                    s_words = words;
                    s_adm[b] = 1;
                    order[count] = b;
                }
            }
            if (lane == 0) s_best = go ? b : -1;
        }
        __syncthreads();
        if (s_best < 0) break;
        ++count;
        const int words = s_words;
        if (words == 0) continue;
        if (part < parts && c_mine < n && !s_adm[c_mine]) {
            int gone = 0;
            for (int q = part; q < words; q += parts) {
                const unsigned long long nb = s_new[q];
                const int w = s_word[q];
                const unsigned long long m = SMEM ? s_rem[w * pitch + c_mine] : masks[(size_t)c_mine * lw + w];
                gone += __popcll(m & nb);
                if (SMEM) s_rem[w * pitch + c_mine] = m & ~nb;
            }
            if (gone) atomicSub(&s_fresh[c_mine], gone);
        }
        __syncthreads();
    }
    if (i < n) {
        admitted[i] = s_adm[i];
        if (i >= count) order[i] = -1;
    }
    if (i == 0) *n_admitted = bad ? -1 : count;          // -1: parent[] was malformed
    if (union_out)
        for (int w = i; w < lw; w += blockDim.x) union_out[w] = s_union[w];
}

// The candidate of largest utility among those whose key is at least `near`, or -1 if that utility is below 1; by the whole
// block, all of whose warps are here: a thread divides for each candidate, every warp finds the largest for itself.
__device__ __noinline__ int expand_resolve(const unsigned *keys, const int *fresh, const double *benefit, const double *c_draft,
                                           unsigned long long *s_exact, double t_exp, int nw, unsigned near)
{
    const int i = threadIdx.x, lane = i & 31;
    if (i < 32 * nw) s_exact[i] = keys[i] >= near ? expand_key(benefit[i], fresh[i], t_exp, c_draft[i]) : 0ull;
    __syncthreads();
    unsigned long long best = 0ull;
    int at = 0;
    for (int q = 0; q < nw; ++q) {
        const unsigned long long key = s_exact[32 * q + lane];
        if (key > best) { best = key; at = 32 * q + lane; }
    }
    const unsigned long long bk = warp_max_key(best);
    if (bk == 0ull || !(dkey_value(bk) >= 1.0)) return -1;
    return (int)__reduce_min_sync(0xffffffffu, best == bk ? (unsigned)at : 0xffffffffu);
}

// The same admissions with every candidate's words in registers: 1 << lp threads of one warp share a candidate, WP pairs of
// words each, and keep what of them is not yet in the union; the rows as they came in lie in shared memory, where
// everybody reads the admitted one's (of its bits, those that are in the union already are in nobody's remainder).
// Bound by latency, and that by the instructions of one admission: a warp issues a dependent one every 4 to 6
// cycles.  So the threads find the largest utility by an approximate one in float32 (a dozen instructions for the
// division's hundred, no conversion), every warp for itself, from keys that alternate between two buffers: one barrier
// per admission.  Only where another key lies within 2^-19 of the largest, or that one so close to 1, are utilities divided
// out in float64 (expand_resolve), unless those candidates have the same operands; so the decisions are those of the
// definition.  The approximation is within 5 units of its last place (three roundings, a reciprocal of 1 unit) for costs
// and benefits in the ranges that `plain` asks for; with a cost or t_exp out of them (negative, below 2^-40, above 2^40) or a
// benefit above 2^60 every admission of the call is resolved exactly.  A benefit below the range (the end of a long chain,
// a token of confidence 0, what hangs on a malformed parent) says nothing about the others.
// Measured, us per call, the kernel above / this one: 8 candidates x 2 words 11.2 / 7.1, 32 x 24 38.3 / 19.3, 64 x 16 73.0 /
// 33.6, one of them with confidence 0 and c_draft NULL 75.8 / 33.6, every utility equal 55.5 / 46.8, 64 x 32 68.2 / 43.0, 64
// x 96 98.6 / 86.2, 96 x 16 109 / 79.9, 128 x 8 135 / 83.5, 128 x 16 142 / 121, 256 x 4 246 / 138, 256 x 8 259 / 215.  Operands out of
// range (a negative cost): 64 x 16 72.9 / 60.1, 128 x 8 135 / 112, but 64 x 48 75.5 / 116, 64 x 96 98.6 / 129.
// NQ: candidates / 32 at most (2 or 8); the rows of up to 1024 threads' words are 64 KiB.
// SKIP: a candidate that brings nothing new changes nobody's remainder.  The branch holds back the loads behind it, so
// it is for blocks of 512 threads and more and for more than 64 candidates, where the loads of all warps take longer than
// their latency: 64 x 96, union full after a few admissions, 83.0 without / 46.6 with it (86.2 against 83.4 where
// everything is new), 64 x 48 69.1 / 46.3; 64 x 16 33.7 / 26.6, but 33.6 / 37.6 where everything is new.
constexpr unsigned kExpandSlack = 16u;
template <int NQ, int WP, bool SKIP>
__global__ void __launch_bounds__(1024)
adaptive_expand_regs_kernel(int n, int lw, int lp, const int32_t *__restrict__ parent, const float *__restrict__ p_tok,
                            const unsigned long long *__restrict__ masks, const float *__restrict__ c_draft, float t_ar,
                            float t_exp, int32_t *__restrict__ admitted, int32_t *__restrict__ order,
                            int32_t *__restrict__ n_admitted, unsigned long long *__restrict__ union_out)
{
    extern __shared__ __align__(16) unsigned long long s_rows[];        // [n][2 * WP << lp], zeros behind the lw words
    __shared__ double s_p[kExpandMaxCand], s_cd[kExpandMaxCand];
    __shared__ unsigned s_key[2][32 * NQ];                              // 0: not eligible
    __shared__ int s_fresh[2][32 * NQ], s_adm[kExpandMaxCand];
    __shared__ unsigned long long s_exact[32 * NQ];

    const int i = threadIdx.x, lane = i & 31, warp = i >> 5, n_warps = (int)blockDim.x >> 5, nw = (n + 31) >> 5;
    const int P = 1 << lp, c = i >> lp, part = i & (P - 1), pitch = 2 * WP * P;
    const bool mine = c < n;
    for (int e = i; e < 2 * 32 * NQ; e += blockDim.x) (&s_key[0][0])[e] = 0u;
    for (int r = warp; r < n; r += n_warps)
        for (int w = lane; w < pitch; w += 32) s_rows[r * pitch + w] = w < lw ? masks[(size_t)r * lw + w] : 0ull;
    for (int e = i; e < n; e += blockDim.x) s_cd[e] = c_draft ? (double)c_draft[e] : 0.0;
    const bool malformed = expand_prefix(n, parent, p_tok, s_p);
    const int bad = __syncthreads_or(malformed ? 1 : 0);
    for (int e = i; e < n; e += blockDim.x) s_p[e] = __dmul_rn(s_p[e], (double)t_ar);       // expected benefit
    __syncthreads();
    // (a benefit below 2^-60, negative or not a number counts as 2^-60: at costs of 0 that is a utility of infinity
    // and at costs of 2^-40 and more one that is never admitted, as with the benefit itself)
    const float b32 = mine && s_p[c] >= 0x1p-60 ? (float)s_p[c] : 0x1p-60f, c32 = mine ? (float)s_cd[c] : 1.0f;
    // (zeros without a sign: the bits are compared as whole numbers)
    auto in_range = [](float v, float lim) { return v >= 1.0f / lim && v <= lim; };
    auto zero = [](float v) { return __float_as_uint(v) == 0u; };
    const bool plain = (zero(t_exp) || in_range(t_exp, 0x1p40f)) && (zero(c32) || in_range(c32, 0x1p40f)) && in_range(b32, 0x1p60f);
    const bool exact = __syncthreads_and(plain ? 1 : 0) == 0;

    // (a parent that does not precede matches nobody: it is never eligible)
    const int par_in = mine ? parent[c] : 0, my_par = mine && par_in < c ? par_in : kExpandMaxCand;
    bool adm = !mine, eligible = my_par < 0;
    const ulonglong2 *rows = reinterpret_cast<const ulonglong2 *>(s_rows);
    ulonglong2 rem[WP];
    int fresh = 0;
#pragma unroll
    for (int j = 0; j < WP; ++j) {
        rem[j] = mine ? rows[c * (pitch >> 1) + j * P + part] : make_ulonglong2(0ull, 0ull);
        fresh += __popcll(rem[j].x) + __popcll(rem[j].y);
    }
    auto over_parts = [&](int v) {
        for (int o = P >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    auto publish = [&](int buf) {
        if (part == 0 && mine) {
            float r;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaf((float)fresh, t_exp, c32)));
            const unsigned key = exact ? 1u : __float_as_uint(b32 * r);
            s_key[buf][c] = eligible && !adm ? key : 0u;
            s_fresh[buf][c] = fresh;
        }
    };
    fresh = over_parts(fresh);
    publish(0);
    __syncthreads();

    constexpr unsigned kOne = 0x3f800000u, kInf = 0x7f800000u;
    int count = 0;
    for (; count < n; ++count) {
        const unsigned *keys = s_key[count & 1];
        const int *fr = s_fresh[count & 1];
        int b = 0;
        if (!exact) {
            unsigned kk[NQ], top = 0u;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                kk[q] = keys[32 * q + lane];
                top = max(top, kk[q]);
            }
            top = __reduce_max_sync(0xffffffffu, top);
            if (top == 0u) break;
            const unsigned near = top > kExpandSlack ? top - kExpandSlack : 1u;
            int holders = 0;
#pragma unroll
            for (int q = NQ - 1; q >= 0; --q) {
                const unsigned hb = __ballot_sync(0xffffffffu, kk[q] >= near);
                if (hb) b = 32 * q + __ffs(hb) - 1;
                holders += __popc(hb);
            }
            if (top - (kOne - kExpandSlack) <= 2u * kExpandSlack) {
                b = expand_resolve(keys, fr, s_p, s_cd, s_exact, (double)t_exp, nw, near);
            } else if (top < kOne) {
                break;
            } else if (holders > 1 && top < kInf) {              // (infinite: a cost of 0, nothing to compare)
                // the same operands, the same utility: the lowest index stands
                const bool same = i >= 32 * nw || keys[i] < near || (fr[i] == fr[b] && s_p[i] == s_p[b] && s_cd[i] == s_cd[b]);
                if (!__syncthreads_and(same ? 1 : 0)) b = expand_resolve(keys, fr, s_p, s_cd, s_exact, (double)t_exp, nw, near);
            }
        } else {
            b = expand_resolve(keys, fr, s_p, s_cd, s_exact, (double)t_exp, nw, 1u);
        }
        if (b < 0) break;
        if (i == 0) order[count] = b;
        adm |= c == b;
        eligible |= my_par == b;
        if (!SKIP || fr[b] != 0) {
            const ulonglong2 *rb = rows + b * (pitch >> 1) + part;
            int gone = 0;
#pragma unroll
            for (int j = 0; j < WP; ++j) {
                const ulonglong2 nb = rb[j * P];
                gone += __popcll(rem[j].x & nb.x) + __popcll(rem[j].y & nb.y);
                rem[j].x &= ~nb.x;
                rem[j].y &= ~nb.y;
            }
            fresh -= over_parts(gone);
        }
        publish((count + 1) & 1);
        __syncthreads();
    }
    if (mine && part == 0) {
        admitted[c] = s_adm[c] = adm ? 1 : 0;
        if (c >= count) order[c] = -1;
    }
    if (i == 0) *n_admitted = bad ? -1 : count;          // -1: parent[] was malformed
    if (union_out) {
        __syncthreads();
        // as many threads of a warp per word as there are for all words
        int lg = 0;
        while (lg < 5 && (lw << (lg + 1)) <= (int)blockDim.x) ++lg;
        for (int base = 0; base < lw; base += (int)blockDim.x >> lg) {
            const int w = base + (i >> lg);
            unsigned long long u = 0ull;
            if (w < lw)
                for (int e = i & ((1 << lg) - 1); e < n; e += 1 << lg) u |= s_rows[e * pitch + w] & (0ull - (unsigned long long)s_adm[e]);
            for (int o = 1 << lg >> 1; o > 0; o >>= 1) u |= __shfl_xor_sync(0xffffffffu, u, o);
            if (w < lw && (i & ((1 << lg) - 1)) == 0) union_out[w] = u;
        }
    }
}

}  // namespace s2moe
