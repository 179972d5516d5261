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

// One block.  Thread i < n owns candidate i: its utility, and its place in the search for the largest one.
// The sets are what costs: after every admission the experts it brought are new to nobody any more.  So
// the kernel keeps, per word and candidate, only the bits NOT yet in the union (s_rem, candidates side by
// side, so that a warp reads neighbouring banks) and their number per candidate (s_fresh).  An
// admission of b makes a list of the words in which b brings anything, and only those are visited: by
// all threads, thread t at candidate t mod np, several threads sharing a candidate's words.  All arithmetic
// that decides an admission is float64 with every operation rounded on its own (no fused
// multiply-add), so that the decisions are those of the plain definition.
// Bound by latency: three block barriers and one float64 division (some 400 cycles) per admission.
// Measured against every candidate counting all its words again for every admission: 64 candidates x
// 16 words (all admitted) 98 -> 74 us, 160 x 96 770 -> 262 us.
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
    const int par_in = i < n ? parent[i] : -1;
    const bool malformed = i < n && par_in >= i;
    const int par = malformed ? -1 : par_in;
    const float pt = i < n ? p_tok[i] : 0.0f;
    const double cd = (i < n && c_draft) ? (double)c_draft[i] : 0.0;
    if (i < n) { s_adm[i] = 0; s_fresh[i] = 0; }
    for (int w = i; w < lw; w += blockDim.x) s_union[w] = 0ull;
    if (SMEM)
        for (int c = warp; c < n; c += (int)blockDim.x >> 5)
            for (int w = lane; w < lw; w += 32) s_rem[w * pitch + c] = masks[(size_t)c * lw + w];
    // Prefix confidence p_i = p_parent * p_{i,j}, block of 32 candidates by block: parents precede their
    // children, so a block needs earlier blocks (shared memory) and itself (shuffles).  A parent index that
    // does not precede is not followed: the candidate gets confidence 0, is never eligible (nor are its
    // descendants) and the call reports it.
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
    const int bad = __syncthreads_or(malformed ? 1 : 0);
    const double benefit = i < n ? __dmul_rn(s_p[i], (double)t_ar) : 0.0;
    const double pos_inf = __longlong_as_double(0x7ff0000000000000ll);
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
            if (i < n && !malformed && !s_adm[i] && (par < 0 || s_adm[par])) {
                const double cost = __dadd_rn(__dmul_rn((double)s_fresh[i], (double)t_exp), cd);   // Eq. 2
                const double u = cost == 0.0 ? pos_inf : __ddiv_rn(benefit, cost);                  // Eq. 3
                if (u == u) key = dkey(u);
            }
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

}  // namespace s2moe
