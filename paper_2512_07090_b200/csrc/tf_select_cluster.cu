// Steps a3 + a4 in one launch, a thread-block cluster per sequence.
//
// The selection of tf_select.cu runs one CTA per sequence, so a batch of 8 sequences of 16384 tokens keeps 8 of
// the GPU's SMs busy for its whole duration, and the fused scores it reads come from a launch of their own.  Here
// a cluster of 4 or 8 CTAs shares a sequence, CTA r of the cluster owning the contiguous token range
// [r L, (r + 1) L), L = 512 KPT:
//   * step a3 (optional, up to 8 KV heads: a row of similarities is then one or two 16-byte loads and a warp reads
//     a contiguous stretch; with more heads a thread per token reads 32 scattered lines per instruction and step a3
//     stays a launch of its own): every thread computes the fused score of its own tokens from the per-head
//     similarities (mean and population variance over heads, Eq. 2 weight, Eq. 3 score) in exactly the order of
//     additions the 8-lanes-per-token kernel of tf_scan.cu uses, so both give the same bits; the scores are written
//     out (they are an output of the layer step) and stay in registers for step a4;
//   * step a4, RATIO mode: the same 4-pass, 8-bit MSB-first radix select over order-preserving keys as the
//     one-CTA kernel.  Each CTA histograms its own candidates and stores the histogram into every CTA's shared
//     memory; every CTA adds them up and takes the same decision; once at most 32 candidates share the prefix every CTA
//     is told all of them and ranks them instead of further passes;
//   * ranks in index order (which of the tokens that tie with the P-th key go, and where a retained token lands in
//     kept_idx) are a CTA-local scan plus the totals of the CTAs before it in the cluster, told the same way.
// Same results as select_kernel, bit for bit: same keys, same tie rule (equal scores go from the highest index
// down), same outputs.
#include <cooperative_groups.h>
#include <math_constants.h>

#include "tf_ptx.cuh"

namespace cg = cooperative_groups;

namespace tf {
namespace {

constexpr int kCsThreads = 512;
constexpr int kCsWarps = kCsThreads / 32;
constexpr int kCsRanks = 8;                   // CTAs of a cluster, at most
constexpr unsigned int kFewMax = 32;          // candidates that are ranked one by one
constexpr int kFewWords = 36;                 // {count, keys}, in whole 16 bytes

struct ClusterSelectParams {
    const float* sim_k; const float* sim_v;   // [B,S,H]; null: the scores are read from `score`
    float* score;                             // [B,S]: written when sim_k is given, read otherwise
    const uint8_t* eligible;                  // [B,S] or null
    const float* threshold;                   // [B] (threshold mode)
    int S, H, warmup, mode, fuse_mode;
    float eps;
    int vec4;                                 // the similarities can be read as float4 (H a multiple of 4, 16-byte aligned)
    long long p_target;                       // floor(ratio*S), computed on the host in double
    uint8_t* keep_mask; int32_t* kept_idx; int32_t* n_kept; float* theta;
    DevStatus* status;
    long long wait_cycles;                    // budget of one mbarrier wait
};

// Step a3 for one token by one thread from the token's similarities in registers (up to 8 KV heads; xk[h], xv[h] are
// read for h < H only), in the order of operations of score_fuse_kernel<8>: "lane" l holds head l (0 + x, as the
// kernel's accumulator starts at zero), the 8 partial values are folded in halves (l with l + 4, then + 2, then + 1).
__device__ __forceinline__ float fuse_token8(const float (&xk)[8], const float (&xv)[8], int H, int mode, float eps) {
    auto fold = [](float (&v)[8]) {
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
#pragma unroll
            for (int l = 0; l < o; ++l) v[l] = __fadd_rn(v[l], v[l + o]);
        return v[0];
    };
    float pk[8], pv[8];
#pragma unroll
    for (int l = 0; l < 8; ++l) {
        pk[l] = l < H ? __fadd_rn(0.f, xk[l]) : 0.f;
        pv[l] = l < H ? __fadd_rn(0.f, xv[l]) : 0.f;
    }
    const float inv = 1.f / (float)H;
    const float sk = __fmul_rn(fold(pk), inv), sv = __fmul_rn(fold(pv), inv);
#pragma unroll
    for (int l = 0; l < 8; ++l) {
        const float a = __fsub_rn(xk[l], sk), b = __fsub_rn(xv[l], sv);
        pk[l] = l < H ? __fmaf_rn(a, a, 0.f) : 0.f;
        pv[l] = l < H ? __fmaf_rn(b, b, 0.f) : 0.f;
    }
    const float vk = __fmul_rn(fold(pk), inv), vv = __fmul_rn(fold(pv), inv);
    return fuse_score(mode, sk, vk, sv, vv, eps);
}

constexpr int kFuseLanes = 8;   // the lane count score_fuse_kernel uses for up to 8 KV heads

template <int KPT>
__global__ void __launch_bounds__(kCsThreads, 1) select_cluster_kernel(const ClusterSelectParams p) {
    // What the CTAs tell one another is stored straight into every CTA's shared memory (its own included), where an mbarrier counts the
    // bytes: nobody waits for more than the numbers themselves.  (A cluster barrier before reading the others' numbers took 1,000 to
    // 1,350 cycles, five times a selection, and the reads as much again: selection of 1 x 2048 tokens 6.3 -> 4.9 us, 1 x 4096 6.7 -> 5.4,
    // 2 x 8192 8.2 -> 7.0, with the scans by one warp.)  Every exchange has its own barrier, used once; the histograms take two buffers
    // in turn: a CTA that sends the pass after next has had everybody's next one, which follows their reading of this one.
    __shared__ __align__(16) unsigned int rx_hist[2][kCsRanks][256];
    __shared__ __align__(16) unsigned int rx_few[kCsRanks][kFewWords];     // {count, keys}
    __shared__ __align__(16) unsigned int rx_eq[kCsRanks][4];              // {equal keys}
    __shared__ __align__(16) unsigned int rx_pub[kCsRanks][4];             // {retained, lowest pruned score}
    __shared__ __align__(8) unsigned long long s_bars[7];                  // passes 0-3, few, equal, published
    __shared__ __align__(16) unsigned int hist[256];
    __shared__ __align__(16) unsigned int s_few[kFewWords];
    __shared__ int s_abort;
    __shared__ int s_warp[kCsWarps];
    __shared__ float s_min;
    __shared__ unsigned int s_prefix;
    __shared__ int s_rank, s_count, s_total;
    __shared__ int s_tab[KPT * kCsWarps];     // [chunk][warp] ballot counts of the final sweep

    cg::cluster_group cluster = cg::this_cluster();
    const int n_ranks = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int b = (int)blockIdx.x / n_ranks, tid = threadIdx.x, S = p.S;
    const int lane = tid & 31, wid = tid >> 5;
    const uint32_t bars = smem_u32(s_bars);
    volatile int* abort_flag = &s_abort;
    if (tid == 0) {
        s_abort = 0;
        for (int i = 0; i < 7; ++i) mbar_init(bars + 8 * i, 1);
        mbar_fence_init();
        for (int i = 0; i < 7; ++i)
            mbar_expect_tx(bars + 8 * i, (uint32_t)n_ranks * (i < 4 ? 1024u : i == 4 ? 4u * kFewWords : 16u));
    }
    if (tid < kFewWords) s_few[tid] = 0;
    cluster.barrier_arrive();    // (waited for before the first store into another CTA: its barriers are set up then)
    // thread (q, k): 16 bytes k of src to place k of this CTA's row in CTA q
    auto tell = [&](const unsigned int* src, unsigned int* row, int words, int bar) {
        const int per = words / 4, q = tid / per, k = tid - q * per;
        if (q < n_ranks)
            st_async16(cluster_addr(smem_u32(row + 4 * k), q), *reinterpret_cast<const uint4*>(src + 4 * k), cluster_addr(bars + 8 * bar, q));
    };
    auto heard = [&](int bar) { mbar_wait_cluster(bars + 8 * bar, 0, abort_flag, p.wait_cycles, p.status, 700 + bar); };
    grid_dependency_wait();
    grid_launch_dependents();   // few CTAs: the attention grid may take the other SMs and set up meanwhile (see select_kernel)
    const int t_base = rank * (KPT * kCsThreads);
    const uint8_t* el = p.eligible ? p.eligible + (size_t)b * S : nullptr;
    float* sc = p.score + (size_t)b * S;

    // token of slot i: t_base + i*512 + tid (ascending in (i, tid))
    float sreg[KPT];
    if (p.sim_k) {
        // the similarities of up to four tokens per thread are requested together (one round trip to memory, not one
        // per token and pass), then fused from registers
        constexpr int kBatch = KPT < 4 ? KPT : 4;
#pragma unroll
        for (int i0 = 0; i0 < KPT; i0 += kBatch) {
            float xk[kBatch][8], xv[kBatch][8];
#pragma unroll
            for (int u = 0; u < kBatch; ++u) {
                const int t = t_base + (i0 + u) * kCsThreads + tid;
                const size_t row = ((size_t)b * S + (t < S ? t : 0)) * p.H;
                if (p.vec4) {
#pragma unroll
                    for (int h4 = 0; h4 < 2; ++h4) {
                        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), c = a;
                        if (t < S && h4 * 4 < p.H) {
                            a = __ldg(reinterpret_cast<const float4*>(p.sim_k + row) + h4);
                            c = __ldg(reinterpret_cast<const float4*>(p.sim_v + row) + h4);
                        }
                        xk[u][4 * h4] = a.x; xk[u][4 * h4 + 1] = a.y; xk[u][4 * h4 + 2] = a.z; xk[u][4 * h4 + 3] = a.w;
                        xv[u][4 * h4] = c.x; xv[u][4 * h4 + 1] = c.y; xv[u][4 * h4 + 2] = c.z; xv[u][4 * h4 + 3] = c.w;
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 8; ++h) {
                        xk[u][h] = (t < S && h < p.H) ? __ldg(p.sim_k + row + h) : 0.f;
                        xv[u][h] = (t < S && h < p.H) ? __ldg(p.sim_v + row + h) : 0.f;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kBatch; ++u) sreg[i0 + u] = fuse_token8(xk[u], xv[u], p.H, p.fuse_mode, p.eps);
        }
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const int t = t_base + i * kCsThreads + tid;
            if (t < S) {
                sc[t] = sreg[i];
                note_nan_score(p.status, sreg[i], (unsigned long long)b * S + t);
            } else {
                sreg[i] = 0.f;
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const int t = t_base + i * kCsThreads + tid;
            sreg[i] = t < S ? sc[t] : 0.f;
        }
    }
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
    } else if (p.p_target <= 0) {
        nothing = true;
    } else {
        unsigned int prefix = 0, mask = 0;
        int r = 0, pass = 0;
        for (int shift = 24; shift >= 0; shift -= 8, ++pass) {
            if (tid < 256) hist[tid] = 0;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const int t = t_base + i * kCsThreads + tid;
                int bin = 256;   // sentinel: this lane adds nothing
                if (t < S && candidate(t, sreg[i])) {
                    const unsigned int k = score_key(sreg[i]);
                    if ((k & mask) == prefix) bin = (int)((k >> shift) & 255u);
                }
                if (pass == 0) {     // (most scores share a few exponents; under a prefix they spread out)
                    const unsigned int same = __match_any_sync(0xffffffffu, bin);
                    if (bin < 256 && lane == __ffs(same) - 1) atomicAdd(&hist[bin], (unsigned int)__popc(same));
                } else if (bin < 256) {
                    atomicAdd(&hist[bin], 1u);
                }
            }
            __syncthreads();
            if (pass == 0) cluster.barrier_wait();
            tell(hist, rx_hist[pass & 1][rank], 256, pass);
            // descending inclusive scan of the cluster's histogram: the bin where the count reaches r.  One warp, eight bins a lane
            if (wid == 0) {
                heard(pass);
                int v[8], sum = 0;      // bins 255 - 8 lane, 254 - 8 lane, ..
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = 0;
                for (int q = 0; q < n_ranks; ++q) {
                    const uint4* src = reinterpret_cast<const uint4*>(&rx_hist[pass & 1][q][248 - 8 * lane]);
                    const uint4 lo = src[0], hi = src[1];
                    v[0] += (int)hi.w; v[1] += (int)hi.z; v[2] += (int)hi.y; v[3] += (int)hi.x;
                    v[4] += (int)lo.w; v[5] += (int)lo.z; v[6] += (int)lo.y; v[7] += (int)lo.x;
                }
#pragma unroll
                for (int e = 0; e < 8; ++e) sum += v[e];
                int incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int n = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += n;
                }
                // first pass: the number of candidates E caps the number to prune (same in every CTA)
                const int E = __shfl_sync(0xffffffffu, incl, 31);
                const int want = pass == 0 ? (int)(p.p_target < (long long)E ? p.p_target : (long long)E) : r;
                if (lane == 0 && want <= 0) s_rank = 0;
                int excl = incl - sum;
                if (excl < want && incl >= want) {
                    int e = 0;
#pragma unroll
                    for (int k = 0; k < 7; ++k)
                        if (e == k && excl + v[k] < want) { excl += v[k]; e = k + 1; }
                    int count = v[7];
#pragma unroll
                    for (int k = 0; k < 7; ++k) count = e == k ? v[k] : count;
                    s_prefix = prefix | ((unsigned int)(255 - 8 * lane - e) << shift);
                    s_rank = want - excl;
                    s_count = count;
                }
            }
            __syncthreads();
            r = s_rank;
            if (r <= 0) { nothing = true; break; }           // (first pass only)
            prefix = s_prefix;
            n_eq = s_count;
            mask |= 255u << shift;
            __syncthreads();     // s_prefix, s_rank and s_count are written again below
            // Few candidates left under this prefix (typical after two or three passes): every CTA is told all of them and ranks
            // them instead of further histogram passes.  Same result: the key of rank r among them, how many candidates carry it,
            // and the rank within those.  (n_eq is the same in every CTA.)
            if (shift > 0 && n_eq <= (int)kFewMax) {
#pragma unroll
                for (int i = 0; i < KPT; ++i) {
                    const int t = t_base + i * kCsThreads + tid;
                    if (t < S && candidate(t, sreg[i])) {
                        const unsigned int k = score_key(sreg[i]);
                        if ((k & mask) == prefix) s_few[1 + min(atomicAdd(&s_few[0], 1u), kFewMax - 1u)] = k;     // n_eq in all CTAs
                    }
                }
                __syncthreads();
                tell(s_few, rx_few[rank], kFewWords, 4);
                if (tid < 32) {
                    heard(4);
                    unsigned int key = 0u;
                    int at = tid;
                    for (int q = 0; q < n_ranks; ++q) {
                        const int c = min((int)rx_few[q][0], (int)kFewMax);
                        if (at >= 0 && at < c) key = rx_few[q][1 + at];
                        at -= c;
                    }
                    int greater = 0, equal = 0;
#pragma unroll
                    for (int o = 0; o < (int)kFewMax; ++o) {         // (a lane without a candidate has key 0, below all of them)
                        const unsigned int ko = __shfl_sync(0xffffffffu, key, o);
                        greater += ko > key ? 1 : 0;
                        equal += ko == key ? 1 : 0;
                    }
                    if (tid < n_eq && greater < r && r <= greater + equal) {   // every lane holding that key writes the same
                        s_prefix = key;
                        s_rank = r - greater;
                        s_count = equal;
                    }
                }
                __syncthreads();
                prefix = s_prefix;
                r = s_rank;
                n_eq = s_count;
                break;
            }
        }
        key_thr = prefix;
        take_eq = r;             // 1 <= r <= n_eq
    }

    // ---- sweep in index order: decide, rank the equal keys, compact ---------------------------------------
    const unsigned int lt = (1u << lane) - 1u;
    auto scan_table = [&]() {    // exclusive prefix over s_tab[0 .. KPT*16), in place; s_total = the sum
        __syncthreads();
        if (wid == 0) {
            constexpr int kEnt = KPT * kCsWarps, kPer = (kEnt + 31) / 32;
            int v[kPer], sum = 0;
#pragma unroll
            for (int e = 0; e < kPer; ++e) { v[e] = lane * kPer + e < kEnt ? s_tab[lane * kPer + e] : 0; sum += v[e]; }
            int incl = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int n = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += n;
            }
            int run = incl - sum;
#pragma unroll
            for (int e = 0; e < kPer; ++e) { if (lane * kPer + e < kEnt) s_tab[lane * kPer + e] = run; run += v[e]; }
            if (lane == 31) s_total = incl;
        } else if (wid == 1) {                                // (the last time: the lowest pruned score)
            const float m = -warp_max(lane < kCsWarps ? -__int_as_float(s_warp[lane]) : -CUDART_INF_F);
            if (lane == 0) s_min = m;
        }
        __syncthreads();
    };
    unsigned int eq_bits = 0, prune_bits = 0;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const int t = t_base + i * kCsThreads + tid;
        const bool cand = t < S && candidate(t, sreg[i]);
        if (p.mode == TF_SELECT_THRESHOLD) {
            if (cand && sreg[i] > tau) prune_bits |= 1u << i;
        } else if (!nothing && cand) {
            const unsigned int k = score_key(sreg[i]);
            if (k > key_thr) prune_bits |= 1u << i;
            if (k == key_thr) eq_bits |= 1u << i;
        }
    }
    if (p.mode != TF_SELECT_THRESHOLD && !nothing) {          // cluster-uniform
        if (take_eq == n_eq) {
            prune_bits |= eq_bits;                            // every token that ties with the P-th key goes
        } else {
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const unsigned int bal = __ballot_sync(0xffffffffu, (eq_bits >> i) & 1u);
                if (lane == 0) s_tab[i * kCsWarps + wid] = __popc(bal);
            }
            scan_table();
            if (tid < n_ranks) st_async16(cluster_addr(smem_u32(rx_eq[rank]), tid), make_uint4((unsigned int)s_total, 0u, 0u, 0u), cluster_addr(bars + 8 * 5, tid));
            heard(5);
            int eq_before = 0;                                // equal keys in the CTAs before this one
            for (int q = 0; q < rank; ++q) eq_before += (int)rx_eq[q][0];
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const bool eq = (eq_bits >> i) & 1u;
                const unsigned int bal = __ballot_sync(0xffffffffu, eq);
                const int eq_rank = eq_before + s_tab[i * kCsWarps + wid] + __popc(bal & lt);   // 0-based among equals, index order
                // the take_eq equals with the highest index: ranks n_eq-take_eq .. n_eq-1
                if (eq && eq_rank >= n_eq - take_eq) prune_bits |= 1u << i;
            }
            __syncthreads();                                  // the table is reused below
        }
    }
    float th_min = CUDART_INF_F;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const int t = t_base + i * kCsThreads + tid;
        const bool keep = t < S && !((prune_bits >> i) & 1u);
        const unsigned int bal = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) s_tab[i * kCsWarps + wid] = __popc(bal);
        if ((prune_bits >> i) & 1u) th_min = fminf(th_min, sreg[i]);
    }
    th_min = -warp_max(-th_min);
    if (lane == 0) s_warp[wid] = __float_as_int(th_min);
    scan_table();
    if (p.mode == TF_SELECT_THRESHOLD || p.p_target <= 0) cluster.barrier_wait();     // (there was no histogram pass)
    if (tid < n_ranks)
        st_async16(cluster_addr(smem_u32(rx_pub[rank]), tid), make_uint4((unsigned int)s_total, __float_as_uint(s_min), 0u, 0u), cluster_addr(bars + 8 * 6, tid));
    heard(6);
    if (__syncthreads_or(*abort_flag)) {         // a wait gave up: everybody is told
        if (tid < n_ranks) *cluster.map_shared_rank(&s_abort, tid) = 1;
        __threadfence();
        __syncwarp();
    }
    // nobody leaves before everybody has come this far: nothing is stored into another CTA after it (relaxed: there is nothing else to order)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    int kept_before = 0, kept_all = 0;
    for (int q = 0; q < n_ranks; ++q) {
        const int n = (int)rx_pub[q][0];
        kept_before += q < rank ? n : 0;
        kept_all += n;
    }
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const int t = t_base + i * kCsThreads + tid;
        const bool in = t < S, keep = in && !((prune_bits >> i) & 1u);
        const unsigned int bal = __ballot_sync(0xffffffffu, keep);
        const int pos = kept_before + s_tab[i * kCsWarps + wid] + __popc(bal & lt);
        if (in) {
            p.keep_mask[(size_t)b * S + t] = keep ? 1 : 0;
            if (keep && (unsigned int)pos < (unsigned int)S) p.kept_idx[(size_t)b * S + pos] = t;   // (outside only after a wait that gave up)
            if (t >= kept_all) p.kept_idx[(size_t)b * S + t] = -1;   // the list's tail: positions kept_all .. S-1 (pos <= t, so never a slot just filled)
        }
    }
    if (rank == 0 && tid == 0) {
        p.n_kept[b] = kept_all;
        if (p.theta) {
            float m = CUDART_INF_F;
            for (int q = 0; q < n_ranks; ++q) m = fminf(m, __uint_as_float(rx_pub[q][1]));
            p.theta[b] = m;
        }
    }
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    if (*abort_flag) {           // in all CTAs or none: nothing kept is better than a list with holes, which the attention would follow
        cluster.sync();
        for (int i = 0; i < KPT; ++i) {
            const int t = t_base + i * kCsThreads + tid;
            if (t < S) { p.kept_idx[(size_t)b * S + t] = -1; p.keep_mask[(size_t)b * S + t] = 0; }
        }
        if (rank == 0 && tid == 0) {
            p.n_kept[b] = 0;
            if (p.theta) p.theta[b] = CUDART_INF_F;
        }
        const long long t0 = clock64();          // stores still under way land before the shared memory goes away
        while (clock64() - t0 < 2000000ll) { }
    }
}

template <int KPT>
cudaError_t launch_form(const ClusterSelectParams& cp, int batch, int n_ranks, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(batch * n_ranks));
    cfg.blockDim = dim3(kCsThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)n_ranks;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, select_cluster_kernel<KPT>, cp);
}

}  // namespace

// Sequence lengths the cluster form takes, and is chosen for: more than 1024 tokens and at most 8 CTAs x 512 threads x 8 scores per
// thread.  Up to 1024 one CTA per sequence selects in the same time (us a launch, one CTA / cluster: 4 x 256 tokens 3.8 / 3.8, 4 x 512 3.9 / 4.4,
// 4 x 768 4.1 / 4.1, 1 x 1000 4.2 / 4.1, 4 x 1024 4.4 / 4.1); with up to 8 KV heads the cluster would also save the fusion's launch (both
// steps, two launches / cluster: 4 x 256 5.1 / 4.4, 4 x 512 5.5 / 5.1, 4 x 768 5.5 / 4.9, 4 x 1024 5.6 / 4.8), with more it does not fuse.
bool select_cluster_usable(const tf_shape& s) { return s.seq > 1024 && s.seq <= 8 * kCsThreads * 8; }
bool select_cluster_preferred(const tf_shape& s) { return select_cluster_usable(s); }
bool select_cluster_fuses(const tf_shape& s) { return s.n_kv_heads <= kFuseLanes; }

// sim_k == nullptr: selection only, the scores are read from `score`
cudaError_t launch_select_cluster(tf_ctx* ctx, const tf_shape& s, const tf_filter_params& p, const float* sim_k,
                                  const float* sim_v, float* score, uint8_t* keep_mask, int32_t* kept_idx,
                                  int32_t* n_kept, float* theta, cudaStream_t st) {
    if (!select_cluster_usable(s) || (sim_k && !select_cluster_fuses(s))) return cudaErrorNotSupported;
    if (s.batch == 0) return cudaSuccess;
    ClusterSelectParams cp{};
    cp.sim_k = sim_k; cp.sim_v = sim_v; cp.score = score;
    cp.eligible = p.eligible; cp.threshold = p.threshold;
    cp.S = s.seq; cp.H = s.n_kv_heads; cp.warmup = p.warmup_tokens; cp.mode = p.select_mode; cp.fuse_mode = p.fuse_mode;
    cp.eps = p.var_eps > 0.f ? p.var_eps : 1e-8f;
    cp.vec4 = (sim_k && s.n_kv_heads % 4 == 0 && ((reinterpret_cast<uintptr_t>(sim_k) | reinterpret_cast<uintptr_t>(sim_v)) & 15) == 0) ? 1 : 0;
    cp.p_target = (long long)floor(p.prune_ratio * (double)s.seq);
    cp.keep_mask = keep_mask; cp.kept_idx = kept_idx; cp.n_kept = n_kept; cp.theta = theta;
    cp.status = ctx->dev_status;
    cp.wait_cycles = ctx_wait_cycles(ctx);
    const int n_ranks = s.seq > 2048 ? 8 : 4;
    const int per_rank = (s.seq + n_ranks - 1) / n_ranks;
    int kpt = 1;
    while (kpt * kCsThreads < per_rank) kpt *= 2;
    cudaError_t e = kpt == 1 ? launch_form<1>(cp, s.batch, n_ranks, st) : kpt == 2 ? launch_form<2>(cp, s.batch, n_ranks, st)
                  : kpt == 4 ? launch_form<4>(cp, s.batch, n_ranks, st) : launch_form<8>(cp, s.batch, n_ranks, st);
    ctx->launches += 1;
    return e;
}

}  // namespace tf
