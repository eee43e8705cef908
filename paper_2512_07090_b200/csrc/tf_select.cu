// Step a4: keep/prune selection and compaction, one CTA per sequence.
//
// RATIO mode prunes exactly P = min(E, floor(ratio*S)) eligible tokens: those that come first
// when eligible tokens are ordered by (score descending, index descending).  The P-th key is
// found with a 4-pass, 8-bit MSB-first radix select over order-preserving 32-bit keys; tokens
// whose key equals it are then taken from the highest index down.  THRESHOLD mode prunes the
// eligible tokens whose score is strictly above threshold[b] (Alg. 1, "skip if s_KV > tau").
// The retained positions are compacted in ascending order with warp ballots and a block-wide
// prefix sum.  For sequences of up to 16384 tokens every thread keeps its scores in registers
// (token i*1024 + tid in slot i), so the passes run out of registers and shared memory; longer
// sequences stage the scores in shared memory (up to 51200 tokens) or re-read them from global memory
// on each pass.  (Producing the scores inside this
// kernel as well was measured: one CTA per sequence reads the per-head similarities far too slowly.)  Sequences of
// up to 240 tokens have a kernel of their own, select_small_kernel, which also makes the scores.
#include <algorithm>
#include <math_constants.h>

#include "tf_common.cuh"

namespace tf {

constexpr int kSelThreads = 1024;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kMaxTableChunks = 64;   // longer sequences (> 65536 tokens) fall back to two block scans per 1024 tokens

struct SelectParams {
    const float* score;        // [B,S]
    const uint8_t* eligible;   // [B,S] or null
    const float* threshold;    // [B] (threshold mode)
    int S, warmup, mode;
    long long p_target;        // floor(ratio*S), computed on the host in double
    int stage;                 // re-reading form only: 1 = the launch has S floats of dynamic shared memory for the scores
    uint8_t* keep_mask; int32_t* kept_idx; int32_t* n_kept; float* theta;
};

// block-wide exclusive prefix over one flag per thread; returns this thread's exclusive rank
// and the block total (s_warp must hold kSelWarps ints; two barriers inside)
__device__ __forceinline__ int block_rank(bool flag, int* s_warp, int& total) {
    const unsigned int bal = __ballot_sync(0xffffffffu, flag);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) s_warp[wid] = __popc(bal);
    __syncthreads();
    int before = 0, tot = 0;
#pragma unroll
    for (int w2 = 0; w2 < kSelWarps; ++w2) {
        const int c = s_warp[w2];
        before += (w2 < wid) ? c : 0;
        tot += c;
    }
    __syncthreads();
    total = tot;
    return before + __popc(bal & ((1u << lane) - 1u));
}

// KPT = scores per thread held in registers (0: read them from global memory each time)
template <int KPT>
__global__ void __launch_bounds__(kSelThreads, 1) select_kernel(const SelectParams p) {
    __shared__ int hist[256];
    __shared__ int s_warp[kSelWarps];
    __shared__ unsigned int s_prefix;
    __shared__ int s_rank, s_count, s_few_eq, s_total;
    __shared__ int s_tab[KPT > 0 ? KPT : kMaxTableChunks][kSelWarps];   // [chunk][warp] ballot counts of the final sweep
    __shared__ unsigned int s_few[32];

    grid_dependency_wait();
    // One CTA per sequence: the attention grid may take the other SMs and set up meanwhile.  After the wait, so that whatever
    // was queued before this kernel is complete when that grid starts and it may read the inputs ahead of its own wait.
    grid_launch_dependents();
    const int b = blockIdx.x, tid = threadIdx.x, S = p.S;
    const float* sc = p.score + (size_t)b * S;
    if (KPT == 0 && p.stage) {   // too many scores for registers: the passes below read them from shared memory
        extern __shared__ float s_scores[];
        for (int t = tid; t < S; t += kSelThreads) s_scores[t] = sc[t];
        __syncthreads();
        sc = s_scores;
    }
    const uint8_t* el = p.eligible ? p.eligible + (size_t)b * S : nullptr;
    constexpr int NR = KPT > 0 ? KPT : 1;
    float sreg[NR];
    if (KPT > 0) {
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int t = i * kSelThreads + tid;
            float s = 0.f;
            if (t < S) {
                s = sc[t];
            }
            sreg[i] = s;
        }
    }
    // score of token t = i*1024 + tid (i is a compile-time index wherever KPT > 0)
    auto score_at = [&](int i, int t) -> float { return KPT > 0 ? sreg[KPT > 0 ? i : 0] : sc[t]; };
    constexpr int kChunks = KPT;   // register form: exactly KPT chunks of 1024 tokens
    auto candidate = [&](int t, float s) -> bool {
        return t >= p.warmup && (el == nullptr || el[t] != 0) && s == s;   // NaN never pruned
    };

    unsigned int key_thr = 0;   // ratio mode: key of the P-th candidate
    int take_eq = 0;            // ratio mode: how many tokens with key == key_thr go (highest index first)
    int n_eq = 0;               // ratio mode: how many candidates have key == key_thr
    float tau = 0.f;
    bool nothing = false;       // nothing to prune

    if (p.mode == TF_SELECT_THRESHOLD) {
        tau = p.threshold[b];
    } else {
        if (p.p_target <= 0) {
            nothing = true;
        } else {
            // radix select: rank r (1-based from the top) among candidates matching the prefix so far.  The number
            // of candidates E, which caps the number to prune (P = min(E, target)), is the total of the first pass's
            // histogram.
            unsigned int prefix = 0, mask = 0;
            int r = 0;
            for (int shift = 24; shift >= 0; shift -= 8) {
                for (int i = tid; i < 256; i += kSelThreads) hist[i] = 0;
                __syncthreads();
#pragma unroll
                for (int i = 0; i < (KPT > 0 ? kChunks : 1 << 30); ++i) {
                    const int t0 = i * kSelThreads;
                    if (KPT == 0 && t0 >= S) break;
                    const int t = t0 + tid;
                    int bin = 256;   // sentinel: this lane adds nothing
                    if (t < S) {
                        const float s = score_at(i, t);
                        if (candidate(t, s)) {
                            const unsigned int k = score_key(s);
                            if ((k & mask) == prefix) bin = (int)((k >> shift) & 255u);
                        }
                    }
                    // scores crowd into a few bins: one shared-memory atomic per distinct bin per warp
                    const unsigned int same = __match_any_sync(0xffffffffu, bin);
                    if (bin < 256 && (tid & 31) == __ffs(same) - 1) atomicAdd(&hist[bin], __popc(same));
                }
                __syncthreads();
                // descending inclusive scan of the histogram: the bin where the count reaches r
                int hval = 0, incl = 0;
                if (tid < 256) {
                    hval = hist[255 - tid];
                    incl = hval;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int n = __shfl_up_sync(0xffffffffu, incl, o);
                        if ((tid & 31) >= o) incl += n;
                    }
                    if ((tid & 31) == 31) s_warp[tid >> 5] = incl;
                }
                __syncthreads();
                if (shift == 24) {                       // first pass: E is known now (uniform over the CTA)
                    int E = 0;
#pragma unroll
                    for (int w2 = 0; w2 < 8; ++w2) E += s_warp[w2];
                    r = (int)(p.p_target < (long long)E ? p.p_target : (long long)E);
                    if (r <= 0) { nothing = true; break; }
                }
                if (tid < 256) {
                    int off = 0;
                    for (int w2 = 0; w2 < (tid >> 5); ++w2) off += s_warp[w2];
                    incl += off;
                    const int excl = incl - hval;
                    if (excl < r && incl >= r) {
                        s_prefix = prefix | ((unsigned int)(255 - tid) << shift);
                        s_rank = r - excl;
                        s_count = hval;
                    }
                }
                __syncthreads();
                prefix = s_prefix;
                r = s_rank;
                n_eq = s_count;
                mask |= 255u << shift;
                // (no barrier here: the next pass writes s_prefix, s_rank and s_count only after two more barriers)
                // Few candidates left under this prefix (typical after two passes: scores share their exponent): one
                // warp ranks them directly instead of two more histogram passes.  Same result: the key of rank r among
                // them, how many candidates carry it, and the rank within those.
                if (shift > 0 && n_eq <= 32) {
                    __syncthreads();                          // everybody has read s_count
                    if (tid == 0) s_count = 0;
                    __syncthreads();
#pragma unroll
                    for (int i = 0; i < (KPT > 0 ? kChunks : 1 << 30); ++i) {
                        const int t0 = i * kSelThreads;
                        if (KPT == 0 && t0 >= S) break;
                        const int t = t0 + tid;
                        if (t < S) {
                            const float sv = score_at(i, t);
                            if (candidate(t, sv)) {
                                const unsigned int k = score_key(sv);
                                if ((k & mask) == prefix) s_few[atomicAdd(&s_count, 1)] = k;
                            }
                        }
                    }
                    __syncthreads();
                    if (tid < 32) {
                        const unsigned int key = tid < n_eq ? s_few[tid] : 0u;
                        int greater = 0, equal = 0;
                        for (int o = 0; o < n_eq; ++o) {
                            const unsigned int ko = __shfl_sync(0xffffffffu, key, o);
                            greater += ko > key ? 1 : 0;
                            equal += ko == key ? 1 : 0;
                        }
                        if (tid < n_eq && greater < r && r <= greater + equal) {   // every lane holding that key writes the same
                            s_prefix = key;
                            s_rank = r - greater;
                            s_few_eq = equal;
                        }
                    }
                    __syncthreads();
                    prefix = s_prefix;
                    r = s_rank;
                    n_eq = s_few_eq;
                    break;
                }
            }
            key_thr = prefix;
            take_eq = r;   // 1 <= r <= n_eq
        }
    }

    // ---- sweep in index order: decide, count equals, compact ---------------------------------------
    int kept_base = 0, eq_base = 0;
    float th_min = CUDART_INF_F;
    if constexpr (KPT > 0) {
        // Register form: ranks in index order (token = chunk * 1024 + thread) come from ONE block-wide scan of a
        // [chunk][warp] table of ballot counts per question (rank among the equal keys, position among the kept
        // tokens), instead of two block scans per chunk of 1024 tokens.
        int* tab = &s_tab[0][0];
        const int lane = tid & 31, wid = tid >> 5;
        const unsigned int lt = (1u << lane) - 1u;
        auto scan_table = [&]() {          // exclusive prefix over tab[0 .. KPT*32), in place; s_total = the sum
            __syncthreads();
            if (wid == 0) {
                int v[NR], sum = 0;
#pragma unroll
                for (int e = 0; e < NR; ++e) { v[e] = tab[lane * NR + e]; sum += v[e]; }
                int incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int n = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += n;
                }
                int run = incl - sum;
#pragma unroll
                for (int e = 0; e < NR; ++e) { tab[lane * NR + e] = run; run += v[e]; }
                if (lane == 31) s_total = incl;
            }
            __syncthreads();
        };
        unsigned int eq_bits = 0, prune_bits = 0;
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int t = i * kSelThreads + tid;
            const float sv = sreg[i];
            const bool cand = t < S && candidate(t, sv);
            if (p.mode == TF_SELECT_THRESHOLD) {
                if (cand && sv > tau) prune_bits |= 1u << i;
            } else if (!nothing && cand) {
                const unsigned int k = score_key(sv);
                if (k > key_thr) prune_bits |= 1u << i;
                if (k == key_thr) eq_bits |= 1u << i;
            }
        }
        if (p.mode != TF_SELECT_THRESHOLD && !nothing) {      // CTA-uniform
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const unsigned int bal = __ballot_sync(0xffffffffu, (eq_bits >> i) & 1u);
                if (lane == 0) tab[i * kSelWarps + wid] = __popc(bal);
            }
            scan_table();
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const bool eq = (eq_bits >> i) & 1u;
                const unsigned int bal = __ballot_sync(0xffffffffu, eq);
                const int eq_rank = tab[i * kSelWarps + wid] + __popc(bal & lt);     // 0-based among equals, index order
                // the take_eq equals with the highest index: ranks n_eq-take_eq .. n_eq-1
                if (eq && eq_rank >= n_eq - take_eq) prune_bits |= 1u << i;
            }
            __syncthreads();                                   // the table is reused below
        }
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int t = i * kSelThreads + tid;
            const bool keep = t < S && !((prune_bits >> i) & 1u);
            const unsigned int bal = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) tab[i * kSelWarps + wid] = __popc(bal);
        }
        scan_table();
#pragma unroll
        for (int i = 0; i < NR; ++i) {
            const int t = i * kSelThreads + tid;
            const bool in = t < S, prune = (prune_bits >> i) & 1u;
            const bool keep = in && !prune;
            const unsigned int bal = __ballot_sync(0xffffffffu, keep);
            const int pos = tab[i * kSelWarps + wid] + __popc(bal & lt);
            if (prune) th_min = fminf(th_min, sreg[i]);
            if (in) {
                p.keep_mask[(size_t)b * S + t] = keep ? 1 : 0;
                if (keep) p.kept_idx[(size_t)b * S + pos] = t;
            }
        }
        kept_base = s_total;
    } else if ((S + kSelThreads - 1) / kSelThreads <= kMaxTableChunks) {
        // The same one-scan-per-question sweep with a run-time number of chunks: the per-chunk decisions are kept as bits
        // of two 64-bit words per thread, the scores are read again (shared or global memory) where they are needed.
        const int n_chunks = (S + kSelThreads - 1) / kSelThreads;
        int* tab = &s_tab[0][0];
        const int lane = tid & 31, wid = tid >> 5;
        const unsigned int lt = (1u << lane) - 1u;
        auto scan_table = [&]() {          // exclusive prefix over tab[0 .. n_chunks*32), in place; s_total = the sum
            __syncthreads();
            if (wid == 0) {
                int sum = 0;
                for (int e = 0; e < n_chunks; ++e) sum += tab[lane * n_chunks + e];
                int incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int n = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += n;
                }
                int run = incl - sum;
                for (int e = 0; e < n_chunks; ++e) { const int v = tab[lane * n_chunks + e]; tab[lane * n_chunks + e] = run; run += v; }
                if (lane == 31) s_total = incl;
            }
            __syncthreads();
        };
        unsigned long long eq_bits = 0ull, prune_bits = 0ull;
        for (int i = 0; i < n_chunks; ++i) {
            const int t = i * kSelThreads + tid;
            const float sv = t < S ? sc[t] : 0.f;
            const bool cand = t < S && candidate(t, sv);
            if (p.mode == TF_SELECT_THRESHOLD) {
                if (cand && sv > tau) prune_bits |= 1ull << i;
            } else if (!nothing && cand) {
                const unsigned int k = score_key(sv);
                if (k > key_thr) prune_bits |= 1ull << i;
                if (k == key_thr) eq_bits |= 1ull << i;
            }
        }
        if (p.mode != TF_SELECT_THRESHOLD && !nothing) {      // CTA-uniform
            for (int i = 0; i < n_chunks; ++i) {
                const unsigned int bal = __ballot_sync(0xffffffffu, (eq_bits >> i) & 1ull);
                if (lane == 0) tab[i * kSelWarps + wid] = __popc(bal);
            }
            scan_table();
            for (int i = 0; i < n_chunks; ++i) {
                const bool eq = (eq_bits >> i) & 1ull;
                const unsigned int bal = __ballot_sync(0xffffffffu, eq);
                const int eq_rank = tab[i * kSelWarps + wid] + __popc(bal & lt);     // 0-based among equals, index order
                if (eq && eq_rank >= n_eq - take_eq) prune_bits |= 1ull << i;        // the take_eq equals with the highest index
            }
            __syncthreads();                                   // the table is reused below
        }
        for (int i = 0; i < n_chunks; ++i) {
            const int t = i * kSelThreads + tid;
            const bool keep = t < S && !((prune_bits >> i) & 1ull);
            const unsigned int bal = __ballot_sync(0xffffffffu, keep);
            if (lane == 0) tab[i * kSelWarps + wid] = __popc(bal);
        }
        scan_table();
        for (int i = 0; i < n_chunks; ++i) {
            const int t = i * kSelThreads + tid;
            const bool in = t < S, prune = (prune_bits >> i) & 1ull;
            const bool keep = in && !prune;
            const unsigned int bal = __ballot_sync(0xffffffffu, keep);
            const int pos = tab[i * kSelWarps + wid] + __popc(bal & lt);
            if (prune) th_min = fminf(th_min, sc[t]);
            if (in) {
                p.keep_mask[(size_t)b * S + t] = keep ? 1 : 0;
                if (keep) p.kept_idx[(size_t)b * S + pos] = t;
            }
        }
        kept_base = s_total;
    } else {
    #pragma unroll
        for (int i = 0; i < (KPT > 0 ? kChunks : 1 << 30); ++i) {
            const int t0 = i * kSelThreads;
            if (t0 >= S) break;
            const int t = t0 + tid;
            const bool in = t < S;
            const float s = in ? score_at(i, t) : 0.f;
            const bool cand = in && candidate(t, s);
            bool prune = false;
            if (p.mode == TF_SELECT_THRESHOLD) {
                prune = cand && (s > tau);
            } else if (!nothing) {
                const unsigned int k = cand ? score_key(s) : 0u;
                const bool eq = cand && (k == key_thr);
                int eq_tot;
                const int eq_rank = block_rank(eq, s_warp, eq_tot) + eq_base;   // 0-based among equals
                eq_base += eq_tot;
                // the take_eq equals with the highest index: ranks n_eq-take_eq .. n_eq-1
                prune = cand && ((k > key_thr) || (eq && eq_rank >= n_eq - take_eq));
            }
            if (prune) th_min = fminf(th_min, s);
            const bool keep = in && !prune;
            int kept_tot;
            const int pos = block_rank(keep, s_warp, kept_tot) + kept_base;
            kept_base += kept_tot;
            if (in) {
                p.keep_mask[(size_t)b * S + t] = keep ? 1 : 0;
                if (keep) p.kept_idx[(size_t)b * S + pos] = t;
            }
        }
    }
    for (int i = kept_base + tid; i < S; i += kSelThreads) p.kept_idx[(size_t)b * S + i] = -1;
    if (tid == 0) p.n_kept[b] = kept_base;
    if (p.theta) {
        // lowest pruned score
        th_min = -warp_max(-th_min);
        if ((tid & 31) == 0) s_warp[tid >> 5] = __float_as_int(th_min);
        __syncthreads();
        if (tid == 0) {
            float m = CUDART_INF_F;
            for (int w2 = 0; w2 < kSelWarps; ++w2) m = fminf(m, __int_as_float(s_warp[w2]));
            p.theta[b] = m;
        }
    }
}

// ---------------------------------------------------------------------------------------------------------
// Short sequences (up to 240 tokens): step a3 and step a4 in one launch, one CTA per sequence, without radix passes: the rank of
// every token among all candidates is counted outright.  A chain of latencies, so what counts is how few there are: one round trip to
// memory for all similarities, one for the outputs, five block barriers.  us per pass, two launches / this one: fp32 1 x 33 x 8 heads 15.4
// / 12.9, 1 x 128 x 32 19.7 / 18.1, 2 x 192 x 40 44.2 / 43.5; bf16 4 x 33 x 8 20.8 / 17.6, 4 x 128 x 8 21.6 / 18.4, 1 x 192 x 32 22.8 / 21.9.  The
// line: the comparisons grow with the square of the length, and one SM reads all similarities: 240 x 32 heads 24.4 / 24.4, 256 x 32
// 24.7 / 25.1, 256 x 8 23.8 / 23.2.  The scores have the bits of score_fuse_kernel<G>: the same order of additions, every rounding
// spelled out.
// ---------------------------------------------------------------------------------------------------------
struct SmallParams {
    SelectParams sel;
    const float* sim_k; const float* sim_v;   // [B,S,H]; null: the scores are read
    float* score_out;                         // [B,S]: written when sim_k is given
    int H, fuse_mode;
    int vec4;                                 // the similarities can be read as float4 (H a multiple of 4, 16-byte aligned)
    float eps;
    DevStatus* status;
};
constexpr int kSmallTokens = 256, kSmallHeads = 64;     // room of the kernel
constexpr int kSmallSeq = 240;                          // ... and the line to the other forms

template <int G>
__global__ void __launch_bounds__(kSelThreads, 1) select_small_kernel(const SmallParams sp) {
    __shared__ float s_score[kSmallTokens];
    __shared__ __align__(16) unsigned int s_key[kSmallTokens];     // 0: not a candidate
    __shared__ unsigned char s_prune[kSmallTokens];
    __shared__ int s_cnt[kSmallTokens / 32];
    __shared__ float s_low[kSmallTokens / 32];
    const SelectParams& p = sp.sel;
    grid_dependency_wait();
    grid_launch_dependents();   // (after the wait: see select_kernel)
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, S = p.S, H = sp.H;
    if (sp.sim_k) {
        // Rows to shared memory as they lie, 4 words apart (a warp then reads 8 tokens x 4 heads without conflicts).  Four threads
        // fuse a token: thread q has the lanes q, q + 4, .. of score_fuse_kernel<G>'s group, so all but the last two steps of its sums
        // are a thread's own (a group of lanes per token spends 20 shuffles on one: 128 tokens x 32 heads 20.8 us per pass instead of 18.1).
        extern __shared__ __align__(16) float s_sim[];                // [2][S][H + 4]
        const int stride = H + 4, n = S * H;
        float* const ks = s_sim;
        float* const vs = s_sim + S * stride;
        const float* gk = sp.sim_k + (size_t)b * n;
        const float* gv = sp.sim_v + (size_t)b * n;
        if (sp.vec4) {
            for (int i = tid * 4; i < n; i += 4 * blockDim.x) {
                const float4 k = __ldg(reinterpret_cast<const float4*>(gk + i)), v = __ldg(reinterpret_cast<const float4*>(gv + i));
                const int at = i + (i / H) * 4;
                *reinterpret_cast<float4*>(ks + at) = k;
                *reinterpret_cast<float4*>(vs + at) = v;
            }
        } else {
            for (int i = tid; i < n; i += blockDim.x) {
                const float k = __ldg(gk + i), v = __ldg(gv + i);
                const int at = i + (i / H) * 4;
                ks[at] = k; vs[at] = v;
            }
        }
        __syncthreads();
        const int t = tid >> 2, q = tid & 3;
        const float* xk = ks + t * stride;
        const float* xv = vs + t * stride;
        constexpr int kOwn = G / 4;
        auto total = [](float (&v)[kOwn]) {
#pragma unroll
            for (int o = kOwn / 2; o > 0; o >>= 1)
#pragma unroll
                for (int e = 0; e < o; ++e) v[e] = __fadd_rn(v[e], v[e + o]);
            v[0] = __fadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], 2));
            return __fadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], 1));
        };
        const float inv = 1.f / (float)H;
        float a[kOwn][2], c[kOwn][2], pk[kOwn], pv[kOwn];
#pragma unroll
        for (int e = 0; e < kOwn; ++e) {
            const int l = q + 4 * e;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const bool in = t < S && l + u * G < H;
                a[e][u] = in ? xk[l + u * G] : 0.f;
                c[e][u] = in ? xv[l + u * G] : 0.f;
            }
            pk[e] = __fadd_rn(0.f, a[e][0]); pv[e] = __fadd_rn(0.f, c[e][0]);
            if (l + G < H) { pk[e] = __fadd_rn(pk[e], a[e][1]); pv[e] = __fadd_rn(pv[e], c[e][1]); }
        }
        const float sk = __fmul_rn(total(pk), inv), sv = __fmul_rn(total(pv), inv);
#pragma unroll
        for (int e = 0; e < kOwn; ++e) {
            pk[e] = pv[e] = 0.f;
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (q + 4 * e + u * G < H) {
                    const float dk = __fsub_rn(a[e][u], sk), dv = __fsub_rn(c[e][u], sv);
                    pk[e] = __fmaf_rn(dk, dk, pk[e]);
                    pv[e] = __fmaf_rn(dv, dv, pv[e]);
                }
        }
        const float vk = __fmul_rn(total(pk), inv), vv = __fmul_rn(total(pv), inv);
        if (q == 0 && t < S) {
            const float s = fuse_score(sp.fuse_mode, sk, vk, sv, vv, sp.eps);
            s_score[t] = s;
            sp.score_out[(size_t)b * S + t] = s;
            note_nan_score(sp.status, s, (unsigned long long)b * S + t);
        }
    } else if (tid < S) {
        s_score[tid] = p.score[(size_t)b * S + tid];
    }
    __syncthreads();
    const uint8_t* el = p.eligible ? p.eligible + (size_t)b * S : nullptr;
    bool cand = false;
    if (tid < kSmallTokens) {
        const float s = tid < S ? s_score[tid] : 0.f;
        cand = tid < S && tid >= p.warmup && (el == nullptr || el[tid] != 0) && s == s;    // NaN never pruned
        s_key[tid] = cand ? score_key(s) : 0u;                                              // (no score's key is 0)
    }
    const int E = __syncthreads_count(cand ? 1 : 0);
    {   // token t, a quarter of the others per thread: higher keys, and equal ones with a higher index, go first
        const int t = tid >> 2, part = tid & 3;
        bool prune = false;
        if (p.mode == TF_SELECT_THRESHOLD) {
            prune = t < S && s_key[t] != 0u && s_score[t] > p.threshold[b];
        } else {
            const int P = (int)(p.p_target < (long long)E ? p.p_target : (long long)E);
            const unsigned int key = s_key[t];
            int rank = 0;
            if (t < S)
                for (int o = part * 4; o < S; o += 16) {              // (keys from S on are 0)
                    const uint4 k = *reinterpret_cast<const uint4*>(&s_key[o]);
                    rank += (k.x > key || (k.x == key && o > t)) ? 1 : 0;
                    rank += (k.y > key || (k.y == key && o + 1 > t)) ? 1 : 0;
                    rank += (k.z > key || (k.z == key && o + 2 > t)) ? 1 : 0;
                    rank += (k.w > key || (k.w == key && o + 3 > t)) ? 1 : 0;
                }
            rank += __shfl_xor_sync(0xffffffffu, rank, 1);
            rank += __shfl_xor_sync(0xffffffffu, rank, 2);
            prune = t < S && key != 0u && rank < P;
        }
        if (part == 0) s_prune[t] = prune ? 1 : 0;
    }
    __syncthreads();
    unsigned int bal = 0;
    bool keep = false;
    if (tid < kSmallTokens) {
        const bool prune = tid < S && s_prune[tid] != 0;
        keep = tid < S && !prune;
        bal = __ballot_sync(0xffffffffu, keep);
        const float low = -warp_max(prune ? -s_score[tid] : -CUDART_INF_F);
        if (lane == 0) { s_cnt[wid] = __popc(bal); s_low[wid] = low; }
    }
    __syncthreads();
    if (tid >= S) return;
    int before = 0, kept = 0;
    float low = CUDART_INF_F;
#pragma unroll
    for (int w = 0; w < kSmallTokens / 32; ++w) {
        before += w < wid ? s_cnt[w] : 0;
        kept += s_cnt[w];
        low = fminf(low, s_low[w]);
    }
    p.keep_mask[(size_t)b * S + tid] = keep ? 1 : 0;
    if (keep) p.kept_idx[(size_t)b * S + before + __popc(bal & ((1u << lane) - 1u))] = tid;
    if (tid >= kept) p.kept_idx[(size_t)b * S + tid] = -1;
    if (tid == 0) {
        p.n_kept[b] = kept;
        if (p.theta) p.theta[b] = low;
    }
}

namespace {
// both steps, or step a4 alone (sim_k null)
bool select_small_takes(const tf_ctx* ctx, const tf_shape& s, bool fuses) {
    return ctx->select_form == 0 && s.seq <= kSmallSeq && (!fuses || s.n_kv_heads <= kSmallHeads);
}
cudaError_t launch_select_small(tf_ctx* ctx, const tf_shape& s, const SelectParams& sel, const tf_filter_params& p, const float* sim_k, const float* sim_v,
                                float* score_out, cudaStream_t st) {
    if (s.seq == 0) return cudaErrorInvalidValue;
    SmallParams sp{};
    sp.sel = sel; sp.sim_k = sim_k; sp.sim_v = sim_v; sp.score_out = score_out;
    sp.H = s.n_kv_heads; sp.fuse_mode = p.fuse_mode; sp.eps = p.var_eps > 0.f ? p.var_eps : 1e-8f;
    sp.status = ctx->dev_status;
    sp.vec4 = (s.n_kv_heads % 4 == 0 && ((reinterpret_cast<uintptr_t>(sim_k) | reinterpret_cast<uintptr_t>(sim_v)) & 15) == 0) ? 1 : 0;
    static bool attr_set_dev[kDeviceFlagSlots] = {};      // function attributes are per device
    bool& attr_set = attr_set_dev[ctx->device >= 0 && ctx->device < kDeviceFlagSlots ? ctx->device : 0];
    if (!attr_set) {
        constexpr int most = 2 * kSmallTokens * (kSmallHeads + 4) * (int)sizeof(float);
        cudaError_t e = cudaFuncSetAttribute(select_small_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(select_small_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(select_small_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const size_t smem = sim_k ? 2 * (size_t)s.seq * (s.n_kv_heads + 4) * sizeof(float) : 0;
    auto kernel = s.n_kv_heads <= 8 ? select_small_kernel<8> : s.n_kv_heads <= 16 ? select_small_kernel<16> : select_small_kernel<32>;
    const cudaError_t e = launch_dependent(kernel, dim3((unsigned)s.batch), dim3((unsigned)std::max(kSmallTokens, (4 * s.seq + 31) / 32 * 32)), smem, st, sp);     // four threads a token
    ctx->launches += 1;
    return e;
}
SelectParams select_params(const tf_shape& s, const tf_filter_params& p, const float* score, uint8_t* keep_mask, int32_t* kept_idx, int32_t* n_kept, float* theta) {
    SelectParams sp{};
    sp.score = score; sp.eligible = p.eligible; sp.threshold = p.threshold;
    sp.S = s.seq; sp.warmup = p.warmup_tokens; sp.mode = p.select_mode;
    sp.p_target = (long long)floor(p.prune_ratio * (double)s.seq);
    sp.keep_mask = keep_mask; sp.kept_idx = kept_idx; sp.n_kept = n_kept; sp.theta = theta;
    return sp;
}

cudaError_t launch_select_form(const SelectParams& sp, int batch, cudaStream_t st) {
    const dim3 grid(batch), block(kSelThreads);
    const int S = sp.S;
    if (S <= 2 * kSelThreads) return launch_dependent(select_kernel<2>, grid, block, 0, st, sp);
    if (S <= 4 * kSelThreads) return launch_dependent(select_kernel<4>, grid, block, 0, st, sp);
    if (S <= 8 * kSelThreads) return launch_dependent(select_kernel<8>, grid, block, 0, st, sp);
    if (S <= 16 * kSelThreads) return launch_dependent(select_kernel<16>, grid, block, 0, st, sp);
    // longer sequences: the scores go to shared memory once (up to 200 KiB = 51200 tokens), else every pass re-reads them
    constexpr size_t kStageMax = 200 << 10;
    SelectParams sp2 = sp;
    const size_t need = (size_t)S * sizeof(float);
    sp2.stage = need <= kStageMax ? 1 : 0;
    if (sp2.stage) {
        static bool attr_set_dev[kDeviceFlagSlots] = {};
        int dev = 0;
        cudaGetDevice(&dev);
        bool& attr_set = attr_set_dev[dev >= 0 && dev < kDeviceFlagSlots ? dev : 0];
        if (!attr_set) {
            cudaError_t e = cudaFuncSetAttribute(select_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStageMax);
            if (e != cudaSuccess) return e;
            attr_set = true;
        }
    }
    return launch_dependent(select_kernel<0>, grid, block, sp2.stage ? need : 0, st, sp2);
}
}  // namespace

cudaError_t launch_select(tf_ctx* ctx, const tf_shape& s, const tf_filter_params& p,
                          const float* score, uint8_t* keep_mask, int32_t* kept_idx,
                          int32_t* n_kept, float* theta, cudaStream_t st) {
    if (s.batch == 0) return cudaSuccess;
    // sequences of 1025 to 32768 tokens are shared by the CTAs of a cluster
    if (ctx->select_form == 2 || (ctx->select_form == 0 && select_cluster_preferred(s)))
        return launch_select_cluster(ctx, s, p, nullptr, nullptr, const_cast<float*>(score), keep_mask, kept_idx, n_kept, theta, st);
    const SelectParams sp = select_params(s, p, score, keep_mask, kept_idx, n_kept, theta);
    if (s.seq > 0 && select_small_takes(ctx, s, false)) return launch_select_small(ctx, s, sp, p, nullptr, nullptr, nullptr, st);
    cudaError_t e = launch_select_form(sp, s.batch, st);
    ctx->launches += 1;
    return e;
}

cudaError_t launch_score_select(tf_ctx* ctx, const tf_shape& s, const tf_filter_params& p, const float* sim_k,
                                const float* sim_v, float* score, uint8_t* keep_mask, int32_t* kept_idx,
                                int32_t* n_kept, float* theta, cudaStream_t st) {
    if ((ctx->select_form == 2 && select_cluster_usable(s) && select_cluster_fuses(s)) ||
        (ctx->select_form == 0 && select_cluster_preferred(s) && select_cluster_fuses(s)))
        return launch_select_cluster(ctx, s, p, sim_k, sim_v, score, keep_mask, kept_idx, n_kept, theta, st);
    if (s.batch > 0 && s.seq > 0 && select_small_takes(ctx, s, true))
        return launch_select_small(ctx, s, select_params(s, p, score, keep_mask, kept_idx, n_kept, theta), p, sim_k, sim_v, score, st);
    cudaError_t e = launch_score_fuse(ctx, s, p, sim_k, sim_v, score, st);
    if (e == cudaSuccess) e = launch_select(ctx, s, p, score, keep_mask, kept_idx, n_kept, theta, st);
    return e;
}

}  // namespace tf
