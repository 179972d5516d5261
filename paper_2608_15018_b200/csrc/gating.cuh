// Reuse-aware expert gating (Sec. 4.2) of one draft batch on given float64 router logits,
// written for a GROUP of warps of a thread block (the whole block of the routing kernel, or the
// warps of the fused layer kernel that have nothing else to do while the layer starts):
//
//   Eq. 4 aggregation g_e = sum_b w_b l_{b,e}, TopCap (E* = the cap experts of largest g),
//   lambda_b = alpha (l_(1) - l_(k+1)), biased top-k in the order (l' descending, l descending,
//   id ascending), mixing weights, union / unique count.
//
// Everything that decides an index is an exact comparison of float64 values through
// order-preserving 64-bit integer keys.  One warp per token; a selection is k rounds of a
// warp-wide maximum over the lanes' best remaining experts (every lane keeps its few experts sorted).
// The rounds compare the upper halves of the keys, without branches: about 45 cycles each, where
// rounds that handle equal keys on the spot took 190 (order statistics) and 340 (selection).  Where
// two lanes meet with equal upper halves (2^-20 relative) the token is done again by those.
// (Measured against it on the same GPU: sorting every token's experts with a
// bitonic network and merging the two lists that the bias leaves in order is data-independent
// and has no long chain, but needs about three times the instructions per token, and with several
// tokens' warps on one scheduler that made the gating 1 us slower at 8 tokens.)
// The path to the selection is kept free of everything that only the mixing weights need: a float64
// exponential or division is a dependent chain of 150 cycles, so they come after the selection has
// been published.  What an SM sees once per launch costs by its number of instructions (straight-line
// code runs at the rate it is fetched, some 4 cycles per instruction, on a warm cache as well, and a turn
// of a loop costs some 60), so loops are unrolled a little or not at all and nothing divides.
#pragma once

#include "common.cuh"

namespace s2moe {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// One copy of the double-precision exponential for code that runs once per layer.
__device__ __noinline__ double exp_once(double x) { return exp(x); }

// Monotone map from doubles (no NaN) to unsigned integers: a < b  <=>  dkey(a) < dkey(b), and
// equal doubles (-0 included) have equal keys.  Keys of finite values are never 0.
__device__ __forceinline__ unsigned long long dkey(double x)
{
    const long long b = __double_as_longlong(x + 0.0);
    return (unsigned long long)(b ^ ((b >> 63) | (long long)0x8000000000000000ull));
}
__device__ __forceinline__ double dkey_value(unsigned long long k)
{
    const long long b = (long long)k;
    return __longlong_as_double(b < 0 ? (b ^ (long long)0x8000000000000000ull) : ~b);
}
// maximum of a 64-bit key over the warp: two 32-bit warp reductions
__device__ __forceinline__ unsigned long long warp_max_key(unsigned long long k)
{
    const unsigned hi = (unsigned)(k >> 32);
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)k : 0u);
    return ((unsigned long long)mh << 32) | ml;
}
// lanes (as a ballot) that hold the largest key among the lanes with `has`; the common case
// (one lane has the largest upper half) takes one warp reduction and one ballot
__device__ __forceinline__ unsigned warp_max_holders(unsigned long long k, bool has)
{
    const unsigned hi = has ? (unsigned)(k >> 32) : 0u;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    bool hold = has && hi == mh;
    unsigned hb = __ballot_sync(0xffffffffu, hold);
    if (__popc(hb) > 1) {
        const unsigned ml = __reduce_max_sync(0xffffffffu, hold ? (unsigned)k : 0u);
        hold = hold && (unsigned)k == ml;
        hb = __ballot_sync(0xffffffffu, hold);
    }
    return hb;
}
__device__ __forceinline__ unsigned long long shfl_key(unsigned long long k, int src)
{
    const unsigned lo = __shfl_sync(0xffffffffu, (unsigned)k, src);
    const unsigned hi = __shfl_sync(0xffffffffu, (unsigned)(k >> 32), src);
    return ((unsigned long long)hi << 32) | lo;
}

// a group of warps of one block and the two named barriers that belong to it
struct GateGroup {
    int t, n, bar;      // thread index inside the group, threads of the group (a multiple of 32, at least 64),
                        // first of two consecutive hardware barriers
};
__device__ __forceinline__ void gate_sync(const GateGroup &g)
{
    asm volatile("bar.sync %0, %1;" ::"r"(g.bar), "r"(g.n) : "memory");
}

// shared memory of the gating; the results stay here for whoever called it
struct GateMem {
    unsigned long long *mask;   // [E] bit b: token b selected the expert
    unsigned long long *gk;     // [E] keys of the aggregated importance g_e
    double *lam;                // [B] lambda_b
    unsigned *gh;               // [E + 4] upper halves of gk
    int *sel;                   // [B * k] selected experts in selection order
    float *pw;                  // [B * k] their mixing weights
    int *cnt, *off, *pos;       // [E] tokens per expert, [E + 1] first slot, [E] index in the active list
    int *U;                     // [1] distinct selected experts
    unsigned *star32;           // [8] E* as bit words (bit i of word j: expert i + 32 j)
    unsigned *topk;             // [B][J] every token's first k experts by original logit, same bit layout (bias on only)
    unsigned char *star;        // [E] member of E*
};
__host__ __device__ __forceinline__ size_t gate_mem_bytes(int E, int B, int k)
{
    return 20 * (size_t)E + 40 + 8 * (size_t)B + 8 * (size_t)B * k + 4 * (size_t)(3 * E + 1) + 4 + 32 + 4 * (size_t)B * 8 +
           (((size_t)E + 15) & ~(size_t)15) + 16;
}
// base: 16-byte aligned shared memory (only pointer arithmetic here, so that the compiler still knows it
// is shared memory and not any)
__device__ __forceinline__ GateMem gate_mem_carve(double *base, int E, int B, int k)
{
    GateMem m;
    uint8_t *p = reinterpret_cast<uint8_t *>(base);
    m.gh = reinterpret_cast<unsigned *>(p); p += (4 * (size_t)E + 31) & ~(size_t)15;    // (first: 16-byte loads)
    m.mask = reinterpret_cast<unsigned long long *>(p); p += 8 * (size_t)E;
    m.gk = reinterpret_cast<unsigned long long *>(p); p += 8 * (size_t)E;
    m.lam = reinterpret_cast<double *>(p); p += 8 * (size_t)B;
    m.sel = reinterpret_cast<int *>(p); p += 4 * (size_t)B * k;
    m.pw = reinterpret_cast<float *>(p); p += 4 * (size_t)B * k;
    m.cnt = reinterpret_cast<int *>(p); p += 4 * (size_t)E;
    m.off = reinterpret_cast<int *>(p); p += 4 * (size_t)(E + 1);
    m.pos = reinterpret_cast<int *>(p); p += 4 * (size_t)E;
    m.U = reinterpret_cast<int *>(p); p += 4;
    m.star32 = reinterpret_cast<unsigned *>(p); p += 32;
    m.topk = reinterpret_cast<unsigned *>(p); p += 4 * (size_t)B * 8;
    m.star = p;
    return m;
}

// The lane's J keys in descending order; equal ones stay in the order of their ids (ascending) unless
// `less` tells them apart.
template <int J, class Less>
__device__ __forceinline__ void lane_sort(unsigned long long (&key)[J], int (&id)[J], Less less)
{
#pragma unroll
    for (int i = J - 1; i > 0; --i)
#pragma unroll
        for (int j = 0; j < i; ++j) {
            if (key[j] < key[j + 1] || (key[j] == key[j + 1] && key[j] != 0ull && less(id[j], id[j + 1]))) {
                const unsigned long long t = key[j];
                key[j] = key[j + 1];
                key[j + 1] = t;
                const int u = id[j];
                id[j] = id[j + 1];
                id[j + 1] = u;
            }
        }
}
template <int J>
__device__ __forceinline__ void lane_pop(unsigned long long (&key)[J], int (&id)[J])
{
#pragma unroll
    for (int j = 0; j + 1 < J; ++j) { key[j] = key[j + 1]; id[j] = id[j + 1]; }
    key[J - 1] = 0ull;
}

// Order statistics of one token's original logits, one warp per token (lane owns experts lane,
// lane + 32, ...), with the bias on: lambda_b = alpha (l_(1) - l_(k+1)) by k + 1 rounds of a warp-wide
// maximum, winners in the exact order (logit descending, id ascending); with TRACK the token's first k
// experts in that order as bit words (word j, bit i: expert i + 32 j; s_topk).  Only TRACK has to tell
// equal logits apart: the order statistics are the same whichever of two wins a round.
template <int J, bool TRACK>
__device__ __forceinline__ void gate_stats(const Shape &sh, int b, const double *s_l, double *s_lam, unsigned *s_topk, int lane)
{
    const unsigned full = 0xffffffffu;
    const int E = sh.E, k = sh.k;
    unsigned long long key[J];
    int id[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        id[j] = lane + 32 * j;
        key[j] = id[j] < E ? dkey(s_l[b * E + id[j]]) : 0ull;
    }
    lane_sort<J>(key, id, [](int, int) { return false; });
    if (!TRACK) {
        // (the order statistics themselves are the same whichever of two equal logits wins a round)
        unsigned h[J], cnt = 0;
        bool first = false;
#pragma unroll
        for (int j = 0; j < J; ++j) h[j] = (unsigned)(key[j] >> 32);
#pragma unroll 1
        for (int r = 0; r < k; ++r) {
            const unsigned m = __reduce_max_sync(full, h[0]);
            const bool win = h[0] == m;
            if (r == 0) first = win;
            cnt += win ? 1u : 0u;
#pragma unroll
            for (int j = 0; j < J; ++j) h[j] = win ? (j + 1 < J ? h[j + 1] : 0u) : h[j];
        }
        const unsigned m = __reduce_max_sync(full, h[0]), hb = __ballot_sync(full, h[0] == m), fb = __ballot_sync(full, first);
        // (two winners in a round: equal upper halves)
        if (__reduce_add_sync(full, cnt) == (unsigned)k && (hb & (hb - 1u)) == 0u) {
            unsigned long long mine = key[0];
#pragma unroll
            for (int j = 1; j < J; ++j) mine = cnt == (unsigned)j ? key[j] : mine;
            const unsigned long long top = shfl_key(key[0], __ffs(fb) - 1), kth = shfl_key(mine, __ffs(hb) - 1);
            if (lane == 0) s_lam[b] = sh.alpha * (dkey_value(top) - dkey_value(kth));
            return;
        }
    }
    unsigned long long top1 = 0ull, kth = 0ull;
    unsigned won = 0;                                    // bit j: expert lane + 32 j is among the first k
#pragma unroll 1
    for (int r = 0; r <= k; ++r) {
        unsigned hb = warp_max_holders(key[0], key[0] != 0ull);
        if (TRACK && __popc(hb) > 1) {                   // equal logits: lower expert id first
            const bool hold = (hb >> lane) & 1u;
            const unsigned me = __reduce_min_sync(full, hold ? (unsigned)id[0] : 0xffffffffu);
            hb = __ballot_sync(full, hold && (unsigned)id[0] == me);
        }
        const int wl = __ffs(hb) - 1;
        if (r == 0) top1 = shfl_key(key[0], wl);
        if (r == k) kth = shfl_key(key[0], wl);
        if (lane == wl) {                                // drop the winner
            if (TRACK && r < k) won |= 1u << (id[0] >> 5);
            lane_pop<J>(key, id);
        }
    }
    if (TRACK) {
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const unsigned word = __ballot_sync(full, (won >> j) & 1u);
            if (lane == 0) s_topk[b * J + j] = word;
        }
    }
    if (lane == 0) s_lam[b] = sh.alpha * (dkey_value(top1) - dkey_value(kth));
}

// Biased top-k of one token in the order (l' descending, l descending, id ascending), one
// winner per round.
template <int J>
__device__ __forceinline__ void gate_select(const Shape &sh, int b, const double *s_l, const unsigned char *s_star,
                                            const double *s_lam, int *s_sel, unsigned long long *s_mask, int lane)
{
    const int E = sh.E, k = sh.k;
    const double lam = s_lam[b], *row = s_l + b * E;
    unsigned long long key[J];
    int id[J];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        id[j] = lane + 32 * j;
        key[j] = 0ull;
        if (id[j] < E) {
            const double l = row[id[j]] + 0.0;
            key[j] = dkey(s_star[id[j]] ? l + lam : l);
        }
    }
    // (equal biased logits: larger original logit first)
    lane_sort<J>(key, id, [&](int i, int j) { return dkey(row[i]) < dkey(row[j]); });
    // the token's bit in an expert's 64-bit mask: a native 32-bit shared-memory atomic on the half that
    // holds it (a 64-bit atomicOr would be a compare-and-swap loop)
    auto select = [&](int r, int e) {
        s_sel[b * k + r] = e;
        atomicOr(reinterpret_cast<unsigned *>(&s_mask[e]) + (b >> 5), 1u << (b & 31));
    };
    unsigned h[J], ranks = 0, cnt = 0;                   // the lane's winners: their ranks, 4 bits each, and their number
#pragma unroll
    for (int j = 0; j < J; ++j) h[j] = (unsigned)(key[j] >> 32);
#pragma unroll 1
    for (int r = 0; r < k; ++r) {
        const unsigned m = __reduce_max_sync(0xffffffffu, h[0]);
        const bool win = h[0] == m;
        ranks |= win ? (unsigned)r << (4u * cnt) : 0u;
        cnt += win ? 1u : 0u;
#pragma unroll
        for (int j = 0; j < J; ++j) h[j] = win ? (j + 1 < J ? h[j + 1] : 0u) : h[j];
    }
    if (__reduce_add_sync(0xffffffffu, cnt) == (unsigned)k) {     // (two winners in a round: equal upper halves)
#pragma unroll
        for (int j = 0; j < J; ++j)
            if ((unsigned)j < cnt) select((int)((ranks >> (4 * j)) & 15u), id[j]);
        return;
    }
#pragma unroll 1
    for (int r = 0; r < k; ++r) {
        unsigned hb = warp_max_holders(key[0], key[0] != 0ull);
        if (__popc(hb) > 1) {                            // equal biased logits: larger original logit first
            const bool in = (hb >> lane) & 1u;
            hb = warp_max_holders(in ? dkey(row[id[0]]) : 0ull, in);
            if (__popc(hb) > 1) {                        // still equal: lower expert id first
                const bool hold = (hb >> lane) & 1u;
                const unsigned me = __reduce_min_sync(0xffffffffu, hold ? (unsigned)id[0] : 0xffffffffu);
                hb = __ballot_sync(0xffffffffu, hold && (unsigned)id[0] == me);
            }
        }
        if (lane == __ffs(hb) - 1) {
            select(r, id[0]);
            lane_pop<J>(key, id);
        }
    }
}

// Mixing weights of one token's selected experts: softmax over all experts of l (weight_mode 0) or l'
// (weight_mode 1), gathered; with renorm the sum over the selected ones takes the place of the sum over
// all.  The lane that owns an expert computes its exponential once.
template <int J>
__device__ __forceinline__ void gate_weights(const Shape &sh, int b, const double *s_l, const unsigned char *s_star, const double *s_lam,
                                             const int *s_sel, float *s_pw, int32_t *__restrict__ sel_idx, float *__restrict__ sel_w,
                                             int lane)
{
    const int E = sh.E, k = sh.k;
    const double lam = sh.weight_mode ? s_lam[b] : 0.0;
    double z[J];
    unsigned long long zk = 0ull;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int e = lane + 32 * j;
        z[j] = 0.0;
        if (e < E) {
            z[j] = (s_l[b * E + e] + 0.0) + (sh.weight_mode && s_star[e] ? lam : 0.0);
            const unsigned long long kk = dkey(z[j]);
            if (kk > zk) zk = kk;
        }
    }
    const double zmax = dkey_value(warp_max_key(zk));
    double den = 0.0;
#pragma unroll
    for (int j = 0; j < J; j += 2) {                      // (two chains at a time)
        z[j] = lane + 32 * j < E ? exp(z[j] - zmax) : 0.0;
        if (j + 1 < J) z[j + 1] = lane + 32 * (j + 1) < E ? exp(z[j + 1] - zmax) : 0.0;
        den += j + 1 < J ? z[j] + z[j + 1] : z[j];
    }
    const int my_sel = lane < k ? s_sel[b * k + lane] : 0;
    double p = 0.0;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const double v = __shfl_sync(0xffffffffu, z[j], my_sel & 31);
        if ((my_sel >> 5) == j) p = v;
    }
    den = warp_sum(sh.renorm ? (lane < k ? p : 0.0) : den);
    if (lane < k) {
        const float w = (float)(p / den);
        s_pw[b * k + lane] = w;
        if (sel_idx) {
            sel_idx[b * k + lane] = my_sel;
            sel_w[b * k + lane] = w;
        }
    }
}

// Steps O2..O5 for B tokens on `s_l` [B][E] (logits) and `s_w` [B] (confidences), both in SHARED
// memory and visible to the group (every row is read several times and E* needs all of them, so a
// caller stages them once: one memory round trip for the whole gating), by the warps of `gg`, in
// two parts.  After gating_part1 (the group is synchronised) gm holds E* (star, star32), lambda_b and
// (want_topk) every token's first k experts by original logit (topk: with the bias on these are the
// experts that the token keeps whenever they are in E*, see the fused kernel); after gating_part2 sel / pw
// in selection order, the per-expert token masks and counts, the exclusive scan `off`, the index
// `pos` of every active expert in the ascending list of active experts, and U.  sel_idx / sel_w
// (global, or NULL) receive the selection and the weights.
// J: experts per lane (2, 4, 8 for up to 64, 128, 256 experts).
// lanes (a power of two, at most 8) that share an expert among cn threads
__device__ __forceinline__ int gate_share_log2(int E, int cn)
{
    int ql = 3;
    while (ql > 0 && (E << ql) > cn) --ql;
    return ql;
}

// Eq. 4 by cn threads (thread ct of them; a multiple of 32): keys of g_e to gm.gk, their upper halves to
// gm.gh as well.  Neighbouring lanes share an expert's tokens.
__device__ __forceinline__ void gating_importance(const Shape &sh, int B, const double *__restrict__ s_l,
                                                  const double *__restrict__ s_w, const GateMem &gm, int ct, int cn)
{
    const int E = sh.E, ql = gate_share_log2(E, cn), step = 1 << ql;
#pragma unroll 1
    for (int i = ct; i < (((E << ql) + 31) & ~31); i += cn) {
        const int e = i >> ql;
        double g = 0.0;
        if (e < E) {
#pragma unroll 2
            for (int b = i & (step - 1); b < B; b += step) g = fma(s_w[b], s_l[b * E + e], g);
        }
#pragma unroll 1
        for (int o = 1; o < step; o <<= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if (e < E && (i & (step - 1)) == 0) {
            const unsigned long long k = dkey(g);
            gm.gk[e] = k;
            gm.gh[e] = (unsigned)(k >> 32);
        }
    }
}

// TopCap by rank in the order (g descending, id ascending), by cn threads (a multiple of 32).
// Neighbouring lanes share an expert's comparisons, which are of the keys' upper halves (four per load)
// and do not tell equal ones apart: that matters when more than cap experts come out, and then
// gating_topcap_exact is needed.  gm.star and gm.star32 must have been cleared, gm.gh padded with 0.
__device__ __forceinline__ void gating_topcap(const Shape &sh, const GateMem &gm, int ct, int cn)
{
    const int E = sh.E, ql = gate_share_log2(E, cn), step = 1 << ql, chunk = (((E + step - 1) >> ql) + 3) & ~3;
#pragma unroll 1
    for (int i = ct; i < (((E << ql) + 31) & ~31); i += cn) {
        const int e = i >> ql;
        int rank = 0;
        if (e < E) {
            const unsigned he = gm.gh[e];
            const int o0 = (i & (step - 1)) * chunk, o1 = min(E, o0 + chunk);
            int r1 = 0, r2 = 0, r3 = 0;                   // (independent counts: a dependent add is 6 cycles)
#pragma unroll 2
            for (int o = o0; o < o1; o += 4) {
                const uint4 v = *reinterpret_cast<const uint4 *>(gm.gh + o);
                rank += v.x > he ? 1 : 0;
                r1 += v.y > he ? 1 : 0;
                r2 += v.z > he ? 1 : 0;
                r3 += v.w > he ? 1 : 0;
            }
            rank += r1 + r2 + r3;
        }
#pragma unroll 1
        for (int o = 1; o < step; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        if (e < E && (i & (step - 1)) == 0 && rank < sh.cap) {
            gm.star[e] = 1;
            atomicOr(&gm.star32[e >> 5], 1u << (e & 31));
        }
    }
}
__device__ __forceinline__ bool gating_topcap_ok(const Shape &sh, const GateMem &gm)
{
    int n = 0;
#pragma unroll 1
    for (int q = 0; 32 * q < sh.E; ++q) n += __popc(gm.star32[q]);
    return n == sh.cap;
}
// (by cn threads, between two barriers of them)
__device__ __noinline__ void gating_topcap_exact(int E, int cap, const unsigned long long *gk, unsigned char *star, unsigned *star32, int ct, int cn)
{
    for (int e = ct; e < E; e += cn) {
        const unsigned long long ge = gk[e];
        int rank = 0;
        for (int o = 0; o < E; ++o) rank += gk[o] > ge || (gk[o] == ge && o < e) ? 1 : 0;
        star[e] = rank < cap;
        if (rank >= cap) atomicAnd(&star32[e >> 5], ~(1u << (e & 31)));
    }
}

// E* by cn threads (thread ct of them; a multiple of 32) that meet on hardware barrier `bar`.
__device__ __forceinline__ void gating_estar(const Shape &sh, int B, const double *__restrict__ s_l,
                                             const double *__restrict__ s_w, const GateMem &gm, int ct, int cn, int bar)
{
    gating_importance(sh, B, s_l, s_w, gm, ct, cn);
    for (int e = sh.E + ct; e < ((sh.E + 3) & ~3); e += cn) gm.gh[e] = 0u;
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(cn) : "memory");
    gating_topcap(sh, gm, ct, cn);
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(cn) : "memory");
    if (!gating_topcap_ok(sh, gm)) {
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(cn) : "memory");
        gating_topcap_exact(sh.E, sh.cap, gm.gk, gm.star, gm.star32, ct, cn);
    }
}

template <int J>
__device__ __forceinline__ void gating_part1(const Shape &sh, int B, const double *__restrict__ s_l,
                                             const double *__restrict__ s_w, const GateGroup gg, const GateMem gm,
                                             bool star_done = false, bool want_topk = false)
{
    const int tid = gg.t, nt = gg.n, warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    const int E = sh.E, k = sh.k, cap = sh.cap;
    const bool bias_on = sh.alpha > 0.0 && cap < E && k < E;
#pragma unroll 1
    for (int e = tid; e < E; e += nt) {
        if (!star_done) gm.star[e] = 0;
        gm.mask[e] = 0ull;
    }
    if (tid < 8 && !star_done) gm.star32[tid] = 0u;
    if (!bias_on)
        for (int b = tid; b < B; b += nt) gm.lam[b] = 0.0;
    gate_sync(gg);
    if (!bias_on) return;

    // E* (unless the caller has it already) on one half of the warps beside the tokens' order statistics on
    // the other half where that leaves every token a warp; else by all warps one after the other
    const int cw = star_done || 2 * B > nw ? 0 : nw / 2, c0 = nw - cw;
    const bool all = cw == 0 && !star_done;
    if (all) {
        gating_importance(sh, B, s_l, s_w, gm, tid, nt);
        if (tid < 4) gm.gh[E + tid] = 0u;
    }
    if (warp >= c0) gating_estar(sh, B, s_l, s_w, gm, tid - c0 * 32, cw * 32, gg.bar + 1);
    else if (want_topk) {
#pragma unroll 1
        for (int b = warp; b < B; b += c0) gate_stats<J, true>(sh, b, s_l, gm.lam, gm.topk, lane);
    } else {
#pragma unroll 1
        for (int b = warp; b < B; b += c0) gate_stats<J, false>(sh, b, s_l, gm.lam, nullptr, lane);
    }
    gate_sync(gg);
    if (all) {
        gating_topcap(sh, gm, tid, nt);
        gate_sync(gg);
        if (!gating_topcap_ok(sh, gm)) {
            gate_sync(gg);
            gating_topcap_exact(E, cap, gm.gk, gm.star, gm.star32, tid, nt);
            gate_sync(gg);
        }
    }
}

// list (or NULL): global words that receive the set of selected experts as soon as it is known, {1 << 32 |
// bits of 32 experts} each.  Nothing else is read on the strength of these words, so they are plain
// stores: a release would wait for the selections that have just been stored (1.5 us with the expert
// kernel's traffic on the memory system).
template <int J>
__device__ __forceinline__ void gating_part2(const Shape &sh, int B, const double *__restrict__ s_l, const GateGroup gg,
                                             const GateMem gm, int32_t *__restrict__ sel_idx, float *__restrict__ sel_w,
                                             unsigned long long *list = nullptr)
{
    const int tid = gg.t, nt = gg.n, warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    const int E = sh.E;
#pragma unroll 1
    for (int b = warp; b < B; b += nw) gate_select<J>(sh, b, s_l, gm.star, gm.lam, gm.sel, gm.mask, lane);
    gate_sync(gg);

    if (list && warp == nw - 2) {
#pragma unroll 1
        for (int q = 0; 32 * q < E; ++q) {
            const int e = 32 * q + lane;
            const unsigned bits = __ballot_sync(0xffffffffu, e < E && gm.mask[e] != 0ull);
            if (lane == 0)
                asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(list + q), "l"((1ull << 32) | (unsigned long long)bits) : "memory");
        }
    }
    // union, unique count, exclusive scan, list of active experts: the last warp, lane owns a run of experts
    if (warp == nw - 1) {
        const int C = (E + 31) >> 5, e0 = lane * C;
        int sum = 0, act = 0;
#pragma unroll 1
        for (int i = 0; i < C; ++i) {
            const int e = e0 + i;
            if (e < E) {
                const int c = __popcll(gm.mask[e]);
                gm.cnt[e] = c;
                sum += c;
                act += c > 0;
            }
        }
        int xs = sum, xa = act;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, xs, o), u = __shfl_up_sync(0xffffffffu, xa, o);
            if (lane >= o) { xs += t; xa += u; }
        }
        int off = xs - sum, pos = xa - act;
#pragma unroll 1
        for (int i = 0; i < C; ++i) {
            const int e = e0 + i;
            if (e < E) {
                const int c = gm.cnt[e];
                gm.off[e] = off; gm.pos[e] = pos;
                off += c; pos += c > 0;
            }
        }
        if (lane == 31) { gm.off[E] = xs; *gm.U = xa; }
    }
#pragma unroll 1
    for (int b = warp; b < B; b += nw) gate_weights<J>(sh, b, s_l, gm.star, gm.lam, gm.sel, gm.pw, sel_idx, sel_w, lane);
    gate_sync(gg);
}

}  // namespace s2moe
