// Online decode step: Algorithm 1 for ONE new token per sequence, with the threshold feedback of
// Section 3.3 (T_l <- T_l + eta (P_current - P_tail)) and the attention it gates.
//
// decode_decide_kernel (one CTA per sequence, a warp per KV head, beyond 8 heads per two):
//   per head: cosine of the current token's key / value to the anchor carried in the state (sum of
//   past tokens, or the EMA of Eq. 1); then one warp: mean / variance over heads, weight alpha
//   (Eq. 2), score s_KV (Eq. 3), threshold adaptation, skip decision; then the anchor takes the
//   token in and the counters advance.  Order as in Algorithm 1: compare first, update after
//   (the inclusive reading updates first).
// decode_attention_stream_kernel, decode_attention_split_kernel (bf16 with 1, 2, 4 or 8 query heads per KV head): below.
// decode_attention_kernel (fp32 and other group sizes; one CTA per (query head, sequence)): standard single-query
//   attention over cache positions <= pos (optionally windowed) unless the token is skipped, in which case its output row
//   is zero (Section 3.2).  The 8 warps take interleaved blocks of 32 keys, each with its own online softmax; the
//   partial results are merged through shared memory.
#include <algorithm>
#include <atomic>
#include <cooperative_groups.h>

#include "tf_ptx.cuh"

namespace tf {

constexpr int kDecWarps = 8;

struct DecideParams {
    const void* K; const void* V;       // cache [B,S,Hkv,128]
    Strides3 ks, vs;
    const int32_t* pos;                 // [B] position of the current token
    int Hkv, anchor_mode, fuse_mode, warmup;
    float gamma, var_eps, eta;
    double target;                      // the target skip ratio, as the caller gave it
    int alg1_sign;
    float* sum_k; float* sum_v; long long* count;      // state
    int sums16;                         // the sums are 16-byte aligned
    int early;                          // the kernel after this one may start now (it waits before it reads what this one writes)
    float* tau; long long* steps; long long* skips;
    float* score_out; uint8_t* skip_out;
    unsigned int* next_piece;           // the streaming kernel's work list, set to its start here (null: there is none)
    DevStatus* status;
};

template <typename T> __device__ __forceinline__ float dec_to_f(T v);
template <> __device__ __forceinline__ float dec_to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float dec_to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T dec_from_f(float v);
template <> __device__ __forceinline__ float dec_from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 dec_from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// four consecutive elements of a cache row (the rows are 16-byte aligned)
__device__ __forceinline__ void dec_load4(const float* p, float (&f)[4]) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
__device__ __forceinline__ void dec_load4(const __nv_bfloat16* p, float (&f)[4]) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xffff0000u);
    f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xffff0000u);
}

// One chain of dependent loads (position, then rows), so what counts is how much of it is in flight at once: a warp per
// KV head, beyond 8 heads per two as far as 32 warps reach, every load a full vector (where the state is aligned).  Once everything before the
// step is complete the attention kernel may start and fetch its first tiles under this kernel.
constexpr int kDecideWarps = 32;

template <typename T, int kHeadsPerWarp>
__global__ void __launch_bounds__(kDecideWarps * 32) decode_decide_kernel(const DecideParams p) {
    extern __shared__ float cos_s[];        // [2][Hkv]
    grid_dependency_wait();                 // launched early; the step before this one on the stream must be complete
    if (p.early) grid_launch_dependents();
    const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    const int t = p.pos[b];
    const long long n0 = p.count[b];
    const bool ema = p.anchor_mode == TF_ANCHOR_EMA, incl = p.anchor_mode == TF_ANCHOR_INCL_MEAN;
    const float a = ema ? p.gamma : 1.f, w = ema ? 1.f - p.gamma : 1.f;
    const long long n_cmp = n0 + (incl ? 1 : 0);            // tokens the anchor covers when it is compared
    // The controller's state is read now, under the row loads below, not after the block barrier.  (The threshold is adapted after it:
    // a 64-bit division ahead of it holds up warp 0, for which all wait: 16 x 250 keys x 32 heads 18.5 -> 19.0 us, 1 x 420 x 8 5.9 either way.)
    long long steps = 0, skips = 0;
    float tau_old = 0.f;
    if (threadIdx.x == 0) { steps = p.steps[b]; skips = p.skips[b]; tau_old = p.tau[b]; }
    if (p.next_piece && b == 0 && threadIdx.x == 0) *p.next_piece = 0u;   // (drawn from after that kernel's wait for this one)

    for (int h0 = warp; h0 < p.Hkv; h0 += kHeadsPerWarp * n_warps) {    // two heads at a time: all of their loads go out together
        float xk4[kHeadsPerWarp][4], xv4[kHeadsPerWarp][4], ak4[kHeadsPerWarp][4], av4[kHeadsPerWarp][4];
#pragma unroll
        for (int u = 0; u < kHeadsPerWarp; ++u) {
            const int h = min(h0 + u * n_warps, p.Hkv - 1);
            dec_load4(reinterpret_cast<const T*>(p.K) + (long long)b * p.ks.b + (long long)t * p.ks.t + (long long)h * p.ks.h + lane * 4, xk4[u]);
            dec_load4(reinterpret_cast<const T*>(p.V) + (long long)b * p.vs.b + (long long)t * p.vs.t + (long long)h * p.vs.h + lane * 4, xv4[u]);
            const size_t off = ((size_t)b * p.Hkv + h) * kHeadDim + lane * 4;
            if (p.sums16) {
                const float4 sk4 = *reinterpret_cast<const float4*>(p.sum_k + off), sv4 = *reinterpret_cast<const float4*>(p.sum_v + off);
                ak4[u][0] = sk4.x; ak4[u][1] = sk4.y; ak4[u][2] = sk4.z; ak4[u][3] = sk4.w;
                av4[u][0] = sv4.x; av4[u][1] = sv4.y; av4[u][2] = sv4.z; av4[u][3] = sv4.w;
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) { ak4[u][i] = p.sum_k[off + i]; av4[u][i] = p.sum_v[off + i]; }
            }
        }
#pragma unroll
        for (int u = 0; u < kHeadsPerWarp; ++u) {
            const int h = h0 + u * n_warps;
            if (h >= p.Hkv) break;
            float dk = 0.f, kk = 0.f, pk = 0.f, dv = 0.f, vv = 0.f, pv = 0.f;
            float nk4[4], nv4[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float xk = xk4[u][i], xv = xv4[u][i];
                float ak = ak4[u][i], av = av4[u][i];
                const float uk = fmaf(a, ak, w * xk), uv = fmaf(a, av, w * xv);    // anchor after the token is taken in
                if (incl) { ak = uk; av = uv; }
                dk = fmaf(xk, ak, dk); kk = fmaf(xk, xk, kk); pk = fmaf(ak, ak, pk);
                dv = fmaf(xv, av, dv); vv = fmaf(xv, xv, vv); pv = fmaf(av, av, pv);
                nk4[i] = uk; nv4[i] = uv;
            }
            dk = warp_sum(dk); kk = warp_sum(kk); pk = warp_sum(pk);
            dv = warp_sum(dv); vv = warp_sum(vv); pv = warp_sum(pv);
            if (lane == 0) {
                float ck = 0.f, cv = 0.f;
                if (n_cmp > 0) {
                    const float s = ema ? 1.f : 1.f / (float)n_cmp;     // anchor = sum * s
                    ck = (dk * s) / (fmaxf(sqrtf(kk), kNormEps) * fmaxf(sqrtf(pk) * s, kNormEps));
                    cv = (dv * s) / (fmaxf(sqrtf(vv), kNormEps) * fmaxf(sqrtf(pv) * s, kNormEps));
                }
                cos_s[h] = ck; cos_s[p.Hkv + h] = cv;
            }
            const size_t off = ((size_t)b * p.Hkv + h) * kHeadDim + lane * 4;
            if (p.sums16) {
                *reinterpret_cast<float4*>(p.sum_k + off) = make_float4(nk4[0], nk4[1], nk4[2], nk4[3]);
                *reinterpret_cast<float4*>(p.sum_v + off) = make_float4(nv4[0], nv4[1], nv4[2], nv4[3]);
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) { p.sum_k[off + i] = nk4[i]; p.sum_v[off + i] = nv4[i]; }
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        const int H = p.Hkv;
        float mk = 0.f, mv = 0.f;
        for (int h = lane; h < H; h += 32) { mk += cos_s[h]; mv += cos_s[H + h]; }
        const float inv = 1.f / (float)H;
        mk = warp_sum(mk) * inv; mv = warp_sum(mv) * inv;
        float vk = 0.f, vvv = 0.f;
        for (int h = lane; h < H; h += 32) {
            const float x = cos_s[h] - mk, y = cos_s[H + h] - mv;
            vk = fmaf(x, x, vk); vvv = fmaf(y, y, vvv);
        }
        vk = warp_sum(vk) * inv; vvv = warp_sum(vvv) * inv;
        if (lane == 0) {
            const float eps = p.var_eps;
            float alpha;
            switch (p.fuse_mode) {
                case TF_FUSE_EQ2_LITERAL: alpha = (vk + eps) / (vk + vvv + 2.f * eps); break;
                case TF_FUSE_KEY_ONLY: alpha = 1.f; break;
                case TF_FUSE_VALUE_ONLY: alpha = 0.f; break;
                case TF_FUSE_MEAN: alpha = 0.5f; break;
                default: alpha = (vvv + eps) / (vk + vvv + 2.f * eps); break;
            }
            float s = alpha * mk + (1.f - alpha) * mv;
            s += 0.f;
            // ratio and step in double, the threshold itself is an fp32 state word
            const double rho = steps > 0 ? (double)skips / (double)steps : 0.0;
            const double delta = (double)p.eta * (p.alg1_sign ? (p.target - rho) : (rho - p.target));
            const float tau = tau_old + (float)delta;
            const bool decide = s > tau;              // false for NaN
            const bool skip = decide && t >= p.warmup;
            p.tau[b] = tau;
            p.steps[b] = steps + 1;
            p.skips[b] = skips + (decide ? 1 : 0);
            p.count[b] = n0 + 1;
            if (p.score_out) p.score_out[b] = s;
            p.skip_out[b] = skip ? 1 : 0;
            if (s != s && p.status) {
                atomicAdd(&p.status->nan_count, 1ull);
                report_error(p.status, TF_ERR_NAN_SCORE, (unsigned long long)b);
            }
        }
    }
}

struct DecAttnParams {
    const void* Q; const void* K; const void* V; void* O;
    long long q_b, q_h, o_b, o_h;       // element strides of the [B,Hq,128] query / output
    Strides3 ks, vs;
    const int32_t* pos; const uint8_t* skip;
    int Hq, Hkv, window;
    float scale_log2;
};

template <typename T>
__global__ void __launch_bounds__(kDecWarps * 32) decode_attention_kernel(const DecAttnParams p) {
    constexpr int EPV = Elem<T>::kPerVec, NVEC = kHeadDim / EPV;
    __shared__ __align__(16) float q_s[kHeadDim];
    __shared__ float m_s[kDecWarps], l_s[kDecWarps];
    __shared__ float acc_s[kDecWarps][kHeadDim];

    grid_dependency_wait();
    const int qh = blockIdx.x, b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    T* orow = reinterpret_cast<T*>(p.O) + (long long)b * p.o_b + (long long)qh * p.o_h;
    if (p.skip[b]) {
        if (threadIdx.x < kHeadDim) orow[threadIdx.x] = dec_from_f<T>(0.f);
        return;
    }
    const int t = p.pos[b];
    const int kh = qh / (p.Hq / p.Hkv);
    const T* qrow = reinterpret_cast<const T*>(p.Q) + (long long)b * p.q_b + (long long)qh * p.q_h;
    if (threadIdx.x < kHeadDim) q_s[threadIdx.x] = dec_to_f<T>(qrow[threadIdx.x]) * p.scale_log2;
    __syncthreads();
    const T* Kb = reinterpret_cast<const T*>(p.K) + (long long)b * p.ks.b + (long long)kh * p.ks.h;
    const T* Vb = reinterpret_cast<const T*>(p.V) + (long long)b * p.vs.b + (long long)kh * p.vs.h;
    const int j_lo = (p.window > 0) ? max(0, t - p.window + 1) : 0;

    float m = -1e30f, lsum = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
    for (int j0 = j_lo + warp * 32; j0 <= t; j0 += kDecWarps * 32) {
        const int j = j0 + lane;
        float s = -1e30f;
        if (j <= t) {
            const T* krow = Kb + (long long)j * p.ks.t;
            float d0 = 0.f, d1 = 0.f;
#pragma unroll 4
            for (int v = 0; v < NVEC; ++v) {
                float f[EPV];
                Elem<T>::unpack(ldg16(krow + v * EPV), f);
                const float* qq = &q_s[v * EPV];
#pragma unroll
                for (int e = 0; e < EPV; e += 2) { d0 = fmaf(f[e], qq[e], d0); d1 = fmaf(f[e + 1], qq[e + 1], d1); }
            }
            s = d0 + d1;
        }
        const float m_new = fmaxf(m, warp_max(s));
        const float corr = exp2f(m - m_new);
        const float pj = (j <= t) ? exp2f(s - m_new) : 0.f;
        lsum = lsum * corr + warp_sum(pj);
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] *= corr;
        const int n_here = min(32, t - j0 + 1);
        for (int jj = 0; jj < n_here; ++jj) {
            const float pw = __shfl_sync(0xffffffffu, pj, jj);
            const T* vrow = Vb + (long long)(j0 + jj) * p.vs.t + lane * 4;
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] = fmaf(pw, dec_to_f<T>(vrow[i]), acc[i]);
        }
        m = m_new;
    }
    if (lane == 0) { m_s[warp] = m; l_s[warp] = lsum; }
#pragma unroll
    for (int i = 0; i < 4; ++i) acc_s[warp][lane * 4 + i] = acc[i];
    __syncthreads();
    if (threadIdx.x < kHeadDim) {
        float mm = -1e30f;
#pragma unroll
        for (int w2 = 0; w2 < kDecWarps; ++w2) mm = fmaxf(mm, m_s[w2]);
        float l = 0.f, o = 0.f;
#pragma unroll
        for (int w2 = 0; w2 < kDecWarps; ++w2) {
            const float c = exp2f(m_s[w2] - mm);       // a warp that saw no key has l = 0 and acc = 0
            l = fmaf(l_s[w2], c, l);
            o = fmaf(acc_s[w2][threadIdx.x], c, o);
        }
        orow[threadIdx.x] = dec_from_f<T>(o / l);
    }
}

// ---------------------------------------------------------------------------------------------------
// bf16 decode attention for ungrouped heads, streaming form: one persistent CTA per SM.  The path is a stream of K / V rows: what bounds it is HBM bandwidth, and what it takes to reach it is that every SM has loads in flight from its
// first to its last cycle.
//   work    the visible keys of every unskipped (sequence, KV head) -- a work item -- are cut into tiles of 64 keys, and the list
//           of all tiles into pieces: 5/8 of it into one piece per CTA, the rest into small pieces that are drawn from a
//           counter, so that CTAs that started late or run on slower SMs take fewer (equal shares alone: the first CTA done
//           14 % before the last).  A work item that lies in several pieces leaves partial results (unnormalised output,
//           maximum, sum) in scratch, and decode_combine_kernel merges them (merging by whichever CTA arrives last was slower:
//           4 x 4096 keys x 40 heads 61.2 against 60.5 us).  Where there are many
//           short work items a piece is a work item, and nothing is merged; so it is without scratch.
//   warp 8  producer: K and V tiles (and the query rows) by TMA into a ring of slots, 192 KB in flight per SM,
//           running ahead across work items.  It starts while the decision kernel still runs, as if no token were skipped; if
//           one is, what it fetched is thrown away.
//   warps 0-3 / 4-7 consume the even / odd tiles, 16 keys per warp, on m16n8k16 products:
//           S^T[16 keys x 8 columns] = K Q^T (A by ldmatrix; column 0 is the head, the others are zero: the products are not what
//           bounds this), online softmax on the accumulator layout (lane holds keys g, g + 8 for columns 2t, 2t + 1), P^T
//           through two 8x8 register transposes, O^T[128 dims x 8] += V^T P^T (A by ldmatrix.trans) with what rounding P to
//           bf16 leaves in column 1: the result is as exact as its own rounding.
//   warps 9-12 merge: at the end of a segment (a work item, or the part of one in this piece) the consumers leave their
//           states in shared memory and go on with the next segment at once; these warps merge the eight states and write the result.
// Every wait is bounded, those of the warps for one another too (mbarriers, no named barriers): on expiry the CTA records
// TF_ERR_TIMEOUT, stops waiting, lets copies in flight land and exits.
//   Against the split kernel: 128 sequences x 400 keys x 40 heads (half of them skipped) 112 -> 96 us, 4 x 4096 keys x 40
// heads 75.5 -> 59 us.
// ---------------------------------------------------------------------------------------------------
constexpr int kPartialFloats = kHeadDim + 2;
constexpr int kStreamKeys = 64;                            // keys per tile
constexpr int kStreamHalf = kStreamKeys * 128;             // one [64 keys][128 B] swizzled block
constexpr int kStreamStage = 4 * kStreamHalf;              // K dims 0-63, 64-127, V dims 0-63, 64-127
constexpr int kStreamThreads = 416;
constexpr int kStreamSegs = 4;                             // segment descriptors in flight
constexpr int kStreamMaxBatch = 512;                       // sequences per launch
constexpr int kStreamDrawn = 1;                            // drawn pieces per CTA on average (4: 8 x 4096 keys x 8 heads 39 instead of 32 us)
constexpr size_t kStreamScratch = (size_t)1 << 20;         // partial results: room for more pieces than there are
// an EVEN number of ring slots: a slot then always belongs to the same half of the consumers, which so waits for every
// phase of its barrier (a half that skipped phases could mistake an earlier one's completion for its own)
constexpr unsigned int kStages = 6;
constexpr int kStreamQ = kHeadDim * 2;                     // the query row of a work item
constexpr int kStreamOffQ = kStages * kStreamStage;
constexpr int kStreamOffPart = kStreamOffQ + kStages * kStreamQ;
constexpr int kStreamSmem = kStreamOffPart + 8 * kPartialFloats * 4 + 1024;   // + alignment slack

struct DecStreamParams {
    const __nv_bfloat16* Q; __nv_bfloat16* O;
    long long q_b, q_h, o_b, o_h;
    const int32_t* pos; const uint8_t* skip;
    int B, Hq, Hkv, window;
    float scale_log2;
    uint4* begun;                     // for decode_combine_kernel: [piece] {sequence or ~0, KV head, last piece} of the work item that begins in the
                                      // piece and ends in a later one; in front of it {pieces, next piece to be drawn}: all of a step's state
                                      // is in its workspace, so that steps on different workspaces do not share any
    float* partial;                   // [slot][130]; null: a work item is never split
    unsigned int max_slots;
    DevStatus* status;
    long long wait_cycles;
};

__device__ __forceinline__ void mma_bf16_16816(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t transpose8x8_b16(uint32_t a) {
    uint32_t d;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(d) : "r"(a));
    return d;
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

// Maps of K and V by the tile's length in blocks of 16 keys: the last tile of a work item is fetched as far as it is visible, not as
// far as it could reach (401 of 525 keys, 128 sequences x 40 heads, half of them skipped: 96.0 -> 91.0 us, none 171 -> 161; 416 rows an item instead of 448).  Four
// copies a tile either way; a box of 16 keys at a time costs one lane up to 16 small ones.  A map whose address is computed costs the
// ring time, though, where a CTA has one long work item and nothing but the ring bounds it: whole tiles then (kBoxes false; no
// workspace, boxes / whole tiles: 2 x 20000 keys x 40 heads 156 / 150 us, 1 x 3000 x 100 34.1 / 33.8; several items a CTA, 400 keys of 525:
// 128 x 40 heads 164 / 183, 128 x 10 heads of 650 keys 71 / 76).
constexpr int kStreamBoxes = kStreamKeys / 16;
struct StreamMaps { CUtensorMap k[kStreamBoxes], v[kStreamBoxes]; };

// The cut of the list of tiles: tiles below `cut` in pieces of `share` tiles, the rest in pieces of `piece`.
struct StreamCut {
    unsigned int cut, share, piece;
    __device__ __forceinline__ unsigned int piece_of(unsigned int y) const { return y < cut ? y / share : cut / share + (y - cut) / piece; }
};
// A piece leaves at most two partial results: slot 2 x for the item it finds begun, 2 x + 1 for the one it begins and does not end.

// a segment: the tiles of one work item in one piece
struct StreamSeg {
    int b, kh, j;                     // sequence, KV head, first tile of the work item
    int count;                        // tiles; 0: no more work
    int slot;                         // where the result goes in the scratch; -1: it is the whole work item
    unsigned int p_last;              // the last piece the work item lies in
    int ends_piece;                   // 1: the piece's last segment ...
    unsigned int piece;               // ... and that piece
};

template <bool kBoxes>
__global__ void __launch_bounds__(kStreamThreads, 1)
decode_attention_stream_kernel(const DecStreamParams p, const __grid_constant__ StreamMaps maps) {
    extern __shared__ uint8_t stream_raw[];
    __shared__ unsigned int pre[kStreamMaxBatch + 1];      // tiles per KV head of the sequences before b
    __shared__ int s_pos[kStreamMaxBatch];
    __shared__ unsigned short active[kStreamMaxBatch];     // the sequences that have tiles
    __shared__ StreamSeg segs[kStreamSegs];
    __shared__ __align__(8) unsigned long long bars[2 * kStages + 2 * kStreamSegs + 2];
    __shared__ unsigned int s_tiles, s_segs;
    __shared__ int s_abort;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(stream_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, cta = blockIdx.x;
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * kStages, bar_seg = bar_empty + 8 * kStages,
                   bar_seg_free = bar_seg + 8 * kStreamSegs, bar_part = bar_seg_free + 8 * kStreamSegs, bar_part_free = bar_part + 8;
    volatile int* abort_flag = &s_abort;
    if (tid == 256) {                                       // the thread that uses the barriers before the first block-wide one
        prefetch_map(&maps.k[kStreamBoxes - 1]); prefetch_map(&maps.v[kStreamBoxes - 1]);
        for (unsigned int i = 0; i < kStages; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 4); }
        for (int i = 0; i < kStreamSegs; ++i) { mbar_init(bar_seg + 8 * i, 1); mbar_init(bar_seg_free + 8 * i, 12); }
        mbar_init(bar_part, 8); mbar_init(bar_part_free, 4);
        s_abort = 0;
        mbar_fence_init();
    }

    // ---- the list of tiles, made by warp 8 -----------------------------------------------------------------------------
    // The positions (like K, V and Q) are not written by the decision kernel, and this grid starts only when every CTA of that
    // kernel has seen all work before it complete: they can be read before the wait (past L1, which may hold older data).
    auto first_key = [&](int t_pos) { return p.window > 0 ? max(0, t_pos - p.window + 1) : 0; };
    unsigned int n_seqs = 0, longest = 0;                   // sequences with work, most tiles of one work item
    auto make_list = [&](bool decided) {
        unsigned int run = 0;
        n_seqs = 0; longest = 0;
        for (int b0 = 0; b0 < p.B; b0 += 32) {
            const int b = b0 + lane;
            unsigned int n = 0;
            if (b < p.B) {
                const int t_pos = decided ? s_pos[b] : __ldcg(p.pos + b);
                if (!decided) s_pos[b] = t_pos;
                if (!decided || !p.skip[b]) n = (unsigned int)(t_pos - first_key(t_pos) + kStreamKeys) / kStreamKeys;
            }
            unsigned int in = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned int v = __shfl_up_sync(0xffffffffu, in, o);
                if (lane >= o) in += v;
            }
            if (b < p.B) pre[b] = run + in - n;
            run += __shfl_sync(0xffffffffu, in, 31);
            const unsigned int with = __ballot_sync(0xffffffffu, n > 0);
            if (n > 0) active[n_seqs + __popc(with & ((1u << lane) - 1u))] = (unsigned short)b;
            n_seqs += __popc(with);
            longest = max(longest, __reduce_max_sync(0xffffffffu, n));
        }
        if (lane == 0) pre[p.B] = run;
        __syncwarp();
    };
    unsigned int total = 0, n_pieces = 0;
    bool whole = false;
    StreamCut cut{};
    auto make_cut = [&]() {                                 // reads pre[]
        total = pre[p.B] * (unsigned int)p.Hkv;
        const unsigned int n_cta = min(gridDim.x, max(total, 1u)), items = n_seqs * (unsigned int)p.Hkv;
        // whole: a piece is a work item, so nothing has to be merged: without scratch, and when there are many short work
        // items anyway
        whole = !p.partial || (items >= 8 * n_cta && longest <= total / (4 * n_cta));
        if (whole) {
            n_pieces = items;
        } else {
            cut.share = max(1u, (total / 8 * 5 + n_cta - 1) / n_cta);
            cut.cut = min(total / cut.share, n_cta) * cut.share;
            const unsigned int rest = total - cut.cut, most = max(1u, min(kStreamDrawn * n_cta, p.max_slots / 2 - n_cta - 1));
            cut.piece = max(1u, (rest + most - 1) / most);
            n_pieces = cut.cut / cut.share + (rest + cut.piece - 1) / cut.piece;
        }
    };
    // producer state (warp 8, lane 0): the current segment, the next tile of it, and where the piece ends
    StreamSeg pt{};
    int pk_lo = 0, p_done = 0, p_vis = 0;                   // first visible key, tiles requested, visible keys from the segment's first on
    unsigned int n_segs = 0;
    int walk = 0;                                           // a sequence at or before the next piece
    unsigned int py = 0, py_end = 0, p_now = 0, pn = 0;     // tile number, end of the piece, its number; tiles of the work item
    auto open_segment = [&]() {                             // from tile py of work item (pt.b, pt.kh, pt.j) on
        pk_lo = first_key(s_pos[pt.b]);
        p_vis = s_pos[pt.b] - pk_lo + 1 - pt.j * kStreamKeys;
        pt.count = (int)min(pn - pt.j, py_end - py);
        p_done = 0;
        pt.p_last = whole ? p_now : cut.piece_of(py - pt.j + pn - 1);
        pt.ends_piece = py + (unsigned int)pt.count == py_end ? 1 : 0;
        pt.piece = p_now;
        pt.slot = (unsigned int)pt.count == pn ? -1 : (int)(2 * p_now + (pt.j == 0 ? 1 : 0));
    };
    auto next_item = [&]() {                                // there is one
        pt.j = 0;
        if (++pt.kh == p.Hkv) {
            pt.kh = 0;
            do { ++pt.b; pn = pre[pt.b + 1] - pre[pt.b]; } while (pn == 0);
        }
    };
    auto open_piece = [&](unsigned int x) {                 // x < n_pieces
        // (on the path of the loads: one division here, and a walk over the sequences instead of a search -- pieces only go up)
        p_now = x;
        if (whole) {
            const unsigned int i = x / (unsigned int)p.Hkv;
            pt.b = active[i]; pt.kh = (int)(x - i * (unsigned int)p.Hkv); pt.j = 0;
            pn = pre[pt.b + 1] - pre[pt.b];
            py = 0; py_end = pn;
        } else {
            const unsigned int n_static = cut.cut / cut.share;
            py = x < n_static ? x * cut.share : cut.cut + (x - n_static) * cut.piece;
            py_end = min(total, x < n_static ? py + cut.share : py + cut.piece);
            while (pre[walk + 1] * (unsigned int)p.Hkv <= py) ++walk;
            pt.b = walk;
            pn = pre[walk + 1] - pre[walk];
            const unsigned int rem = py - pre[walk] * (unsigned int)p.Hkv;
            pt.kh = (int)(rem / pn); pt.j = (int)(rem - (unsigned int)pt.kh * pn);
        }
        open_segment();
    };
    auto announce = [&]() {                                 // the segment's descriptor (its ring slot is free)
        segs[n_segs % kStreamSegs] = pt;
        mbar_arrive(bar_seg + 8 * (n_segs % kStreamSegs));
        ++n_segs;
    };
    auto produce = [&](unsigned int it) {
        const unsigned int st = it % kStages;
        const uint32_t dst = sbase + st * kStreamStage, bar = bar_full + 8 * st;
        const int key = pk_lo + (pt.j + p_done) * kStreamKeys;
        const bool with_q = p_done < 2;                    // either half of the consumers finds the query rows with its first tile
        const int box = kBoxes ? min((p_vis - p_done * kStreamKeys + 15) / 16, kStreamBoxes) - 1 : kStreamBoxes - 1;
        const CUtensorMap *mk = &maps.k[box], *mv = &maps.v[box];
        mbar_expect_tx(bar, (box + 1) * (4 * 16 * 128) + (with_q ? kStreamQ : 0));
        tma_load_4d(dst, mk, bar, 0, pt.kh, key, pt.b);
        tma_load_4d(dst + kStreamHalf, mk, bar, 64, pt.kh, key, pt.b);
        tma_load_4d(dst + 2 * kStreamHalf, mv, bar, 0, pt.kh, key, pt.b);
        tma_load_4d(dst + 3 * kStreamHalf, mv, bar, 64, pt.kh, key, pt.b);
        if (with_q) bulk_load(sbase + kStreamOffQ + st * kStreamQ, p.Q + (long long)pt.b * p.q_b + (long long)pt.kh * p.q_h, kStreamQ, bar);
        ++p_done; ++py;
        if (p_done == pt.count && py < py_end) { next_item(); open_segment(); }
    };
    if (warp == 8) {
        make_list(false);
        if (lane == 0) {
            unsigned int n = 0;
            make_cut();
            if ((unsigned int)cta < n_pieces) {
                open_piece(cta);
                for (; n < kStages && py < py_end && (p_done > 0 || n_segs < kStreamSegs); ++n) {
                    if (p_done == 0) announce();
                    produce(n);
                }
            }
            s_tiles = n;                                    // tiles fetched and segments announced before the decisions are known
            s_segs = n_segs;
        }
    }
    __syncwarp();
    grid_dependency_wait();
    int any_skip = 0;
    for (int b = tid; b < p.B; b += kStreamThreads) any_skip |= p.skip[b];
    any_skip = __syncthreads_or(any_skip);
    const unsigned int ahead = s_tiles;
    const unsigned int wasted = any_skip ? ahead : 0u, wasted_segs = any_skip ? s_segs : 0u;   // in vain: everybody lets them pass
    if (warp == 8) {
        // ================================ producer ============================================================
        if (any_skip) { make_list(true); walk = 0; }
        if (lane == 0) make_cut();
        if (cta == 0 && lane == 0 && p.begun) p.begun[-1].x = whole ? 0u : n_pieces;
        if (lane == 0) {
            unsigned int x = cta, it = ahead;
            bool ok = true, open = !any_skip && ahead > 0;   // the piece opened above goes on
            auto slot_free = [&]() {
                return it < kStages || mbar_wait_bounded(bar_empty + 8 * (it % kStages), ((it / kStages) - 1) & 1u, abort_flag, p.wait_cycles, p.status, 601);
            };
            auto seg_free = [&]() {
                return n_segs < kStreamSegs ||
                       mbar_wait_bounded(bar_seg_free + 8 * (n_segs % kStreamSegs), ((n_segs / kStreamSegs) - 1) & 1u, abort_flag, p.wait_cycles, p.status, 606);
            };
            while (ok && x < n_pieces) {
                if (!open) open_piece(x);
                unsigned int x_next = x + gridDim.x;
                bool drawn = !p.partial;
                while (ok && py < py_end) {
                    if (!drawn && py + 3 >= py_end) {       // as late as the answer is still there in time
                        x_next = gridDim.x + atomicAdd(&p.begun[-1].y, 1u);
                        drawn = true;
                    }
                    if (p_done == 0) {
                        ok = seg_free();
                        if (ok) announce();
                    }
                    ok = ok && slot_free();
                    if (ok) { produce(it); ++it; }
                }
                if (!drawn) x_next = gridDim.x + atomicAdd(&p.begun[-1].y, 1u);
                open = false;
                x = x_next;
            }
            if (ok && seg_free()) {                         // no more work
                pt.count = 0;
                announce();
            }
        }
    } else if (warp < 8) {
        // ================================ consumers ===========================================================
        grid_launch_dependents();
        float* part_s = reinterpret_cast<float*>(smem + kStreamOffPart);
        const int half = warp >> 2, kb = (warp & 3) * 16;   // this warp's 16 keys of every second tile
        const int g = lane >> 2, t = lane & 3;
        // ldmatrix row of this lane: K as A (rows = keys), V as transposed A (rows = keys of the stored tile)
        const int rk = kb + (lane & 7) + ((lane >> 3) & 1) * 8, ck = lane >> 4;
        const int rv = kb + (lane & 7) + (lane >> 4) * 8, cv = (lane >> 3) & 1;
        unsigned int it = 0;
        bool ok = true;
        for (; it < wasted; ++it) {
            if ((int)(it & 1) != half) continue;
            ok = __all_sync(0xffffffffu, ok && mbar_wait_bounded(bar_full + 8 * (it % kStages), 0, abort_flag, p.wait_cycles, p.status, 603));
            if (ok && lane == 0) mbar_arrive(bar_empty + 8 * (it % kStages));
        }
        for (unsigned int sg = 0; ok; ++sg) {
            const unsigned int ss = sg % kStreamSegs;
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_seg + 8 * ss, (sg / kStreamSegs) & 1u, abort_flag, p.wait_cycles, p.status, 607));
            if (!ok) break;
            const StreamSeg seg = segs[ss];
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_seg_free + 8 * ss);
            if (sg < wasted_segs) continue;
            if (seg.count == 0) break;
            const int t_pos = s_pos[seg.b], n_vis = t_pos - first_key(t_pos) + 1 - seg.j * kStreamKeys;      // visible keys from the segment's first on
            float m = -1e30f, l = 0.f;                          // of column 2t (m is the same in all lanes of equal t; l is the lane's share)
            float o[8][4];                                      // O^T: dims 16 mt + g and 16 mt + 8 + g, columns 2t, 2t + 1
            uint32_t qb[8][2];
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) { o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f; }
            const int i0 = ((int)(it & 1) == half) ? 0 : 1;      // this half's first tile
            for (int i = i0; i < seg.count; i += 2) {
                const unsigned int st = (it + i) % kStages;
                ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_full + 8 * st, ((it + i) / kStages) & 1u, abort_flag, p.wait_cycles, p.status, 602));
                if (!ok) break;
                if (i < 2) {                                     // Q^T as the B operand
                    const uint8_t* q = smem + kStreamOffQ + st * kStreamQ + t * 4;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        qb[kk][0] = g == 0 ? *reinterpret_cast<const uint32_t*>(q + kk * 32) : 0u;
                        qb[kk][1] = g == 0 ? *reinterpret_cast<const uint32_t*>(q + kk * 32 + 16) : 0u;
                    }
                }
                const uint32_t ka = sbase + st * kStreamStage, va = ka + 2 * kStreamHalf;
                const int left = n_vis - i * kStreamKeys - kb;   // visible keys of this warp's 16
                if (left > 0) {
                    float s[4] = {0.f, 0.f, 0.f, 0.f}, s2[4] = {0.f, 0.f, 0.f, 0.f};   // two accumulation chains
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        uint32_t a[4];
                        const int ch = kk * 2 + ck;
                        ldmatrix4(ka + (ch >> 3) * kStreamHalf + rk * 128 + (((ch & 7) ^ (rk & 7)) << 4), a);
                        mma_bf16_16816(kk & 1 ? s2 : s, a[0], a[1], a[2], a[3], qb[kk][0], qb[kk][1]);
                    }
                    if (left < 16) {   // rows past the last visible key hold whatever the cache holds: their values must not reach the sum
                        for (int z = lane; z < (16 - left) * 16; z += 32) {
                            const int row = kb + left + (z >> 4);
                            *reinterpret_cast<uint4*>(smem + st * kStreamStage + (2 + ((z >> 3) & 1)) * kStreamHalf + row * 128 + ((z & 7) << 4)) = make_uint4(0, 0, 0, 0);
                        }
                        __syncwarp();
                    }
                    const bool v0 = g < left, v1 = g + 8 < left;
                    const float sa = v0 ? (s[0] + s2[0]) * p.scale_log2 : -1e30f, sb = v1 ? (s[2] + s2[2]) * p.scale_log2 : -1e30f;
                    float mx = fmaxf(sa, sb);
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
                    const float mn = fmaxf(m, mx), corr = ex2_approx(m - mn);
                    m = mn;
                    const float pa = v0 ? ex2_approx(sa - mn) : 0.f, pb = v1 ? ex2_approx(sb - mn) : 0.f;
                    l = fmaf(l, corr, pa + pb);
                    // P^T (keys x columns) -> the B operand wants column g with keys 2t, 2t+1 / 2t+8, 2t+9: two 8x8 transposes.
                    // The odd columns have no head of their own: they take what rounding a probability to bf16 leaves, so
                    // that it is not lost (4 x 4095 keys x 40 heads, error against 64 bits: without it 1.82e-3).
                    const float ha = __bfloat162float(__float2bfloat16_rn(pa)), hb = __bfloat162float(__float2bfloat16_rn(pb));
                    const uint32_t pb0 = transpose8x8_b16(pack_bf16x2(ha, pa - ha));
                    const uint32_t pb1 = transpose8x8_b16(pack_bf16x2(hb, pb - hb));
                    if (__any_sync(0xffffffffu, corr != 1.f)) {
#pragma unroll
                        for (int mt = 0; mt < 8; ++mt) { o[mt][0] *= corr; o[mt][1] *= corr; o[mt][2] *= corr; o[mt][3] *= corr; }
                    }
#pragma unroll
                    for (int mt = 0; mt < 8; ++mt) {
                        uint32_t a[4];
                        const int ch = mt * 2 + cv;
                        ldmatrix4_trans(va + (ch >> 3) * kStreamHalf + rv * 128 + (((ch & 7) ^ (rv & 7)) << 4), a);
                        mma_bf16_16816(o[mt], a[0], a[1], a[2], a[3], pb0, pb1);
                    }
                }
                if (left < 16) fence_proxy_async();              // zeros written above, before TMA writes the slot again
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_empty + 8 * st);
            }
            if (!ok) break;
            it += seg.count;
            // ---- the warp's state to the merging warps ---------------------------------------------------------------
            l += __shfl_xor_sync(0xffffffffu, l, 4);
            l += __shfl_xor_sync(0xffffffffu, l, 8);
            l += __shfl_xor_sync(0xffffffffu, l, 16);
            const unsigned int k_seg = sg - wasted_segs;         // (the first wait passes: nothing has been left there yet)
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(bar_part_free, (k_seg & 1u) ^ 1u, abort_flag, p.wait_cycles, p.status, 605));
            if (!ok) break;
            if (t == 0) {                                        // columns 0 and 1 are the head
                // (ordered by the tiles, not by the half that the ring happened to give them to: the merge then adds in one
                // order whichever pieces this CTA drew before, and the result has the same bits every time)
                float* dst = part_s + (i0 * 4 + (warp & 3)) * kPartialFloats;
#pragma unroll
                for (int mt = 0; mt < 8; ++mt) { dst[16 * mt + g] = o[mt][0] + o[mt][1]; dst[16 * mt + 8 + g] = o[mt][2] + o[mt][3]; }
                if (g == 0) { dst[kHeadDim] = m; dst[kHeadDim + 1] = l; }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_part);
        }
    } else {
        // ================================ merging warps =======================================================
        const float* part_s = reinterpret_cast<const float*>(smem + kStreamOffPart);
        const int mt = tid - 288;                           // 0 .. 127: output dim
        for (int b = cta; b < p.B; b += (int)gridDim.x)     // skipped tokens' output rows
            if (p.skip[b])
                for (int i = mt; i < p.Hq * (kHeadDim / 8); i += 128)
                    *reinterpret_cast<uint4*>(p.O + (long long)b * p.o_b + (long long)(i >> 4) * p.o_h + (i & 15) * 8) = make_uint4(0, 0, 0, 0);
        for (unsigned int sg = 0;; ++sg) {
            const unsigned int ss = sg % kStreamSegs;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar_seg + 8 * ss, (sg / kStreamSegs) & 1u, abort_flag, p.wait_cycles, p.status, 608))) break;
            const StreamSeg seg = segs[ss];
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_seg_free + 8 * ss);
            if (sg < wasted_segs) continue;
            if (seg.count == 0) break;
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar_part, (sg - wasted_segs) & 1u, abort_flag, p.wait_cycles, p.status, 609))) break;
            float M = -1e30f, L = 0.f, acc = 0.f;
#pragma unroll
            for (int w2 = 0; w2 < 8; ++w2) M = fmaxf(M, part_s[w2 * kPartialFloats + kHeadDim]);
#pragma unroll
            for (int w2 = 0; w2 < 8; ++w2) {
                const float* src = part_s + w2 * kPartialFloats;
                const float e = ex2_approx(src[kHeadDim] - M);
                L = fmaf(src[kHeadDim + 1], e, L);
                acc = fmaf(src[mt], e, acc);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_part_free);
            if (seg.slot < 0) {
                p.O[(long long)seg.b * p.o_b + (long long)seg.kh * p.o_h + mt] = __float2bfloat16_rn(acc / L);
            } else {
                float* dst = p.partial + (size_t)seg.slot * kPartialFloats;
                dst[mt] = acc;
                if (mt == 0) { dst[kHeadDim] = M; dst[kHeadDim + 1] = L; }
            }
            if (p.begun && seg.ends_piece && mt == 0 && seg.piece < gridDim.x * (1 + kStreamDrawn))
                p.begun[seg.piece] = seg.slot == (int)(2 * seg.piece + 1) ? make_uint4((unsigned int)seg.b, (unsigned int)seg.kh, seg.p_last, 0u)
                                                                          : make_uint4(0xffffffffu, 0u, 0u, 0u);
        }
    }
    __syncwarp();
    __syncthreads();
    if (*abort_flag) {   // a wait gave up: let copies in flight land before the shared memory goes away
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) { }
    }
}

// merges the work items that lie in several pieces: CTA x the one that begins in piece x, a thread per dim
__global__ void __launch_bounds__(kHeadDim) decode_combine_kernel(const DecStreamParams p) {
    grid_dependency_wait();
    const unsigned int x = blockIdx.x, n_pieces = p.begun[-1].x;
    if (x == 0 && threadIdx.x == 0) p.begun[-1].y = 0u;     // for the next sequences of the same step, if there are more
    // Beyond the last piece, and in the pieces of a CTA that gave up waiting, stands whatever the workspace held: an entry
    // that does not name a work item is passed over, not followed.
    const uint4 it = p.begun[x];
    if (x >= n_pieces || it.x >= (unsigned int)p.B || it.y >= (unsigned int)p.Hkv || it.z < x || it.z >= n_pieces) return;
    const int n = (int)(it.z - x) + 1, d = threadIdx.x;
    const float* base = p.partial + (size_t)(2 * x) * kPartialFloats;
    float M = -1e30f, L = 0.f, acc = 0.f;
    for (int q0 = 0; q0 < n; q0 += 8) {                     // eight parts requested together: one round trip, not one per part
        float m[8], l[8], v[8], mx = M;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = min(q0 + u, n - 1);
            const float* src = base + (size_t)(2 * q + (q == 0 ? 1 : 0)) * kPartialFloats;
            m[u] = src[kHeadDim]; l[u] = src[kHeadDim + 1]; v[u] = src[d];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = fmaxf(mx, m[u]);
        const float e0 = exp2f(M - mx);
        L *= e0; acc *= e0; M = mx;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float e = q0 + u < n ? exp2f(m[u] - M) : 0.f;
            L = fmaf(l[u], e, L);
            acc = fmaf(v[u], e, acc);
        }
    }
    p.O[(long long)it.x * p.o_b + (long long)it.y * p.o_h + d] = __float2bfloat16_rn(acc / L);
}

// what decode_combine_kernel reads, in front of the slots
static size_t stream_table_bytes(int grid) { return (1 + (size_t)grid * (1 + kStreamDrawn)) * sizeof(uint4); }

size_t decode_scratch_bytes(const tf_shape& s) { return s.dtype == TF_BF16 ? kStreamScratch + stream_table_bytes(sm_count()) + 256 : 0; }   // (+ alignment)

static cudaError_t launch_stream(const DecStreamParams& sp, int grid, int device, const StreamMaps& maps, cudaStream_t st) {
    static bool attr_set_dev[kDeviceFlagSlots] = {};      // function attributes are per device
    bool& attr_set = attr_set_dev[device >= 0 && device < kDeviceFlagSlots ? device : 0];
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(decode_attention_stream_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStreamSmem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(decode_attention_stream_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStreamSmem);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const bool boxes = sp.begun || (long long)sp.B * sp.Hkv > grid;      // (one whole item a CTA at most: see StreamMaps)
    const cudaError_t e = launch_dependent(boxes ? decode_attention_stream_kernel<true> : decode_attention_stream_kernel<false>, dim3((unsigned)grid),
                                           dim3(kStreamThreads), kStreamSmem, st, sp, maps);
    if (e != cudaSuccess || !sp.begun) return e;
    return launch_dependent(decode_combine_kernel, dim3((unsigned)(grid * (1 + kStreamDrawn))), dim3(kHeadDim), 0, st, sp);
}

// ---------------------------------------------------------------------------------------------------
// Grouped heads, and ungrouped ones in a short step: one CTA per (split of the visible keys, KV head, sequence), two CTAs per SM.
// No list of work to make, and the head start of this form outweighs the equal shares of the streaming kernel: always for grouped
// heads (whose cache is a G-th of the bytes; us a step, this / streaming with four heads a tile: 1 x 8192 14.6 / 23.3, 8 x 4096
// 28.6 / 30.3, 64 x 1000 48.6 / 52.7, 128 x 4000 327 / 323), for ungrouped ones as far as launch_decode_step says.  Operands come
// straight from global memory, no shared memory: a dot product does not care in which order the dims are visited, so lane (g, t)
// loads 16-byte pieces t, t+4, t+8, t+12 of its two key rows (g, g+8) and of the query head of column g; of its four value rows (2t,
// 2t+1, 2t+8, 2t+9) it loads 16 dims, and the pairs "same dim, two consecutive keys" the A operand wants are byte permutes.
// The 8 warps take key blocks 8 apart and are merged through shared memory.  The splits of a short step are a thread-block cluster
// (kAsCluster): they are merged through distributed shared memory, without scratch and without a third launch; otherwise the CTA
// leaves (max, sum, unnormalised output) per head in scratch and decode_merge_splits_kernel merges the splits.
//   The kernel starts while the decision is made: keys, values, queries and positions are not written by the decision kernel, which
// lets this one start once all work before it is complete.  A CTA waits for the decision with its first keys in flight (kEarly), one
// of a cluster with its third 128 keys in flight, or when its products are done: one stream of 420 keys 8.0 -> 5.8 us, 8 x 4096 keys
// 30.1 -> 28.0.  What it loads for a skipped sequence is lost, so a cluster does not go further ahead (us a step, keys from HBM, waiting
// only when the products are done / with the third / the second / the first 128 keys in flight; none skipped: 8 x 420 8.8 / 8.5 / 8.4 /
// 9.2, 4 x 1500 11.1 / 10.4 / 10.4 / 11.5, 8 x 1000 13.3 / 12.1 / 12.1 / 13.2, 1 x 1500 x 40 ungrouped 12.2 / 11.3 / 12.7; half of them
// skipped: 4 x 1500 11.1 / 10.3 / 10.3 / 10.9, 8 x 1000 13.2 / 12.0 / 11.9 / 12.5; all: 9.6 / 8.4 / 6.8 / 5.0, 11.6 / 8.6 / 6.9 / 4.8).
// Letting the kernel after this one start as early made every step slower (1 x 8192 14.7 -> 16.5).
// ---------------------------------------------------------------------------------------------------
struct DecGqaParams {
    const __nv_bfloat16* Q; const __nv_bfloat16* K; const __nv_bfloat16* V; __nv_bfloat16* O;
    long long q_b, q_h, o_b, o_h;
    Strides3 ks, vs;
    const int32_t* pos; const uint8_t* skip;
    int Hq, Hkv, window, n_splits;
    int n_early;                      // the CTAs that start while the decision kernel runs
    float scale_log2;
    float* partial;                   // [B][Hq][n_splits][130] when n_splits > 1
};

// loads ahead of the wait go past L1, which may hold what a row held before the kernels that are complete by now
template <bool kPastL1> __device__ __forceinline__ uint4 load16(const void* p) {
    return kPastL1 ? __ldcg(reinterpret_cast<const uint4*>(p)) : ldg16(p);
}
__device__ __forceinline__ uint32_t word_of(const uint4& r, int w) { return w == 0 ? r.x : w == 1 ? r.y : w == 2 ? r.z : r.w; }

// When a CTA waits for the decision: before its first loads, with its first keys' loads in flight, or as a cluster does
enum SplitForm { kAfterDecision, kEarly, kAsCluster };

constexpr int kClusterAhead = 2 * 8 * 16;        // keys a CTA of a cluster goes through before it waits: two blocks of 16 per warp

template <int G, int kForm>
__global__ void __launch_bounds__(256, kForm == kAsCluster ? 1 : 2) decode_attention_split_kernel(const DecGqaParams p) {
    constexpr bool kCluster = kForm == kAsCluster;
    // column 2h of the products is head h, column 2h + 1 what rounding its probabilities to bf16 leaves (as in the streaming kernel); or
    // column h is head h: eight heads fill them, and with two CTAs per SM grouped heads have no registers left for the remainder (G = 4:
    // 20 bytes spilled, 32 x 5000 keys x 8 heads 110.8 instead of 103.4 us)
    constexpr bool kRest = G == 1 || (G <= 4 && kCluster);
    constexpr int kCols = kRest ? 1 : 2;             // heads of a lane: t, or 2t and 2t + 1
    // dims of a lane's value rows: 16g .. 16g + 15, or 8g .. and 64 + 8g .., where a load instruction takes whole lines (128 x 256 keys x 8
    // heads 35.6 -> 34.0 us, 4 x 700 as clusters 6.64 -> 6.46; but ungrouped clusters 1 x 1500 x 40 9.9 -> 10.4, and with the decision
    // waited for under the loads 16 x 4096 48.5 -> 49.3)
    constexpr bool kLines = kForm == kAfterDecision || (kCluster && G > 1);
    constexpr int kDim0 = kLines ? 8 : 16, kDim8 = kLines ? 64 : 8;   // dim of piece 0 / of piece 1 beyond it, per g
    __shared__ float part_s[8][G][kPartialFloats];
    __shared__ float merge_s[kCluster ? 8 : 1][kCluster ? G : 1][kPartialFloats];   // the splits' results, in the first CTA of a cluster
    const int split = blockIdx.x, kh = blockIdx.y, b = blockIdx.z;
    if constexpr (kCluster) cooperative_groups::this_cluster().barrier_arrive();   // this CTA's shared memory may be written from now on
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int t_pos = __ldcg(p.pos + b);
    const int j_lo = (p.window > 0) ? max(0, t_pos - p.window + 1) : 0;
    const int n_vis = t_pos - j_lo + 1;
    const int per = ((n_vis + p.n_splits - 1) / p.n_splits + 15) / 16 * 16;     // keys per split, a multiple of 16
    const int k_lo = j_lo + split * per, k_hi = min(t_pos + 1, k_lo + per);       // [k_lo, k_hi)
    const uint4 zero4 = make_uint4(0, 0, 0, 0);

    // Q^T as the B operand of the 8 score products: column g, pieces t + 4i; product 2i + u takes words 2u, 2u + 1
    uint32_t qb[8][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool head = kRest ? (g & 1) == 0 && g < 2 * G : g < G;
        const uint4 r = head ? load16<kForm != kAfterDecision>(p.Q + (long long)b * p.q_b + (long long)(kh * G + (kRest ? g >> 1 : g)) * p.q_h + 8 * (t + 4 * i)) : zero4;
        qb[2 * i][0] = r.x; qb[2 * i][1] = r.y; qb[2 * i + 1][0] = r.z; qb[2 * i + 1][1] = r.w;
    }
    const __nv_bfloat16* Kb = p.K + (long long)b * p.ks.b + (long long)kh * p.ks.h;
    const __nv_bfloat16* Vb = p.V + (long long)b * p.vs.b + (long long)kh * p.vs.h + kDim0 * g;

    // this lane's part of the state (m is the same in all lanes of equal t; l is the lane's share)
    float m[kCols], l[kCols];
#pragma unroll
    for (int c = 0; c < kCols; ++c) { m[c] = -1e30f; l[c] = 0.f; }
    float o[8][4];                                   // O^T: product mt, rows (dims) kDim0 g + mt and kDim8 beyond, columns 2t, 2t + 1
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) { o[mt][0] = o[mt][1] = o[mt][2] = o[mt][3] = 0.f; }

    bool decided = false, skipped = false;
    auto decision = [&]() {
        grid_dependency_wait();
        decided = true;
        skipped = __ldcg(p.skip + b) != 0;
    };
    // (the CTAs of a later wave start after the decision: theirs costs nothing to know, and may save them their loads)
    if (kForm == kAfterDecision || (kForm == kEarly && split + p.n_splits * (kh + p.Hkv * b) >= p.n_early)) decision();
    for (int kb = k_lo + 16 * warp; kb < k_hi && !skipped; kb += 16 * 8) {       // warp-uniform bounds: the shuffles below name all lanes
        uint4 kr[2][4], vr[4][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = kb + g + 8 * h;
#pragma unroll
            for (int i = 0; i < 4; ++i) kr[h][i] = (j < k_hi) ? load16<kForm != kAfterDecision>(Kb + (long long)j * p.ks.t + 8 * (t + 4 * i)) : zero4;
        }
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
            const int j = kb + 2 * t + (q4 & 1) + 8 * (q4 >> 1);
#pragma unroll
            for (int i = 0; i < 2; ++i) vr[q4][i] = (j < k_hi) ? load16<kForm != kAfterDecision>(Vb + (long long)j * p.vs.t + kDim8 * i) : zero4;
        }
        if (!decided && (kForm == kEarly || (kForm == kAsCluster && kb >= k_lo + kClusterAhead))) {
            decision();
            if (skipped) break;
        }
        // ---- scores: rows = keys g, g + 8; columns = heads 2t, 2t + 1 -----------------------------------------
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mma_bf16_16816(s, kr[0][i].x, kr[1][i].x, kr[0][i].y, kr[1][i].y, qb[2 * i][0], qb[2 * i][1]);
            mma_bf16_16816(s, kr[0][i].z, kr[1][i].z, kr[0][i].w, kr[1][i].w, qb[2 * i + 1][0], qb[2 * i + 1][1]);
        }
        const bool v0 = kb + g < k_hi, v1 = kb + g + 8 < k_hi;
        float corr[kCols], pr[2 * kCols];
#pragma unroll
        for (int c = 0; c < kCols; ++c) {
            const float sa = v0 ? s[c] * p.scale_log2 : -1e30f, sb = v1 ? s[c + 2] * p.scale_log2 : -1e30f;
            float mx = fmaxf(sa, sb);
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
            const float mn = fmaxf(m[c], mx);
            corr[c] = ex2_approx(m[c] - mn);
            m[c] = mn;
            pr[c] = v0 ? ex2_approx(sa - mn) : 0.f;
            pr[c + kCols] = v1 ? ex2_approx(sb - mn) : 0.f;
            l[c] = fmaf(l[c], corr[c], pr[c] + pr[c + kCols]);
        }
        // P^T (keys x columns) -> the B operand wants column g with keys 2t, 2t+1 / 2t+8, 2t+9: two 8x8 transposes
        uint32_t pb0, pb1;
        if constexpr (kRest) {
            const float ha = __bfloat162float(__float2bfloat16_rn(pr[0])), hb = __bfloat162float(__float2bfloat16_rn(pr[1]));
            pb0 = transpose8x8_b16(pack_bf16x2(ha, pr[0] - ha));
            pb1 = transpose8x8_b16(pack_bf16x2(hb, pr[1] - hb));
        } else {
            pb0 = transpose8x8_b16(pack_bf16x2(pr[0], pr[1]));
            pb1 = transpose8x8_b16(pack_bf16x2(pr[2], pr[3]));
        }
#pragma unroll
        for (int mt = 0; mt < 8; ++mt) {
            o[mt][0] *= corr[0]; o[mt][1] *= corr[kCols - 1]; o[mt][2] *= corr[0]; o[mt][3] *= corr[kCols - 1];
            const int w = mt >> 1;
            const uint32_t sel = (mt & 1) ? 0x7632u : 0x5410u;     // the high / low halves of two rows' words
            const uint32_t a0 = __byte_perm(word_of(vr[0][0], w), word_of(vr[1][0], w), sel);   // the first dim,  keys 2t, 2t+1
            const uint32_t a1 = __byte_perm(word_of(vr[0][1], w), word_of(vr[1][1], w), sel);   // the second dim, keys 2t, 2t+1
            const uint32_t a2 = __byte_perm(word_of(vr[2][0], w), word_of(vr[3][0], w), sel);   // the first dim,  keys 2t+8, 2t+9
            const uint32_t a3 = __byte_perm(word_of(vr[2][1], w), word_of(vr[3][1], w), sel);
            mma_bf16_16816(o[mt], a0, a1, a2, a3, pb0, pb1);
        }
    }
    if (!decided) decision();
    if (skipped) {                                   // the whole cluster (it has one sequence)
        if (split == 0 && (kCluster || p.n_splits == 1))
            for (int i = threadIdx.x; i < G * kHeadDim; i += 256)
                p.O[(long long)b * p.o_b + (long long)(kh * G + i / kHeadDim) * p.o_h + (i % kHeadDim)] = __float2bfloat16_rn(0.f);
        if constexpr (kCluster) cooperative_groups::this_cluster().barrier_wait();
        return;
    }
    // ---- the lane's share of l -> the sum over the 8 lanes of equal t; then everything into shared memory ---------
#pragma unroll
    for (int c = 0; c < kCols; ++c) {
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 4);
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 8);
        l[c] += __shfl_xor_sync(0xffffffffu, l[c], 16);
    }
#pragma unroll
    for (int c = 0; c < kCols; ++c) {
        const int h = kCols * t + c;
        if (h < G) {
#pragma unroll
            for (int mt = 0; mt < 8; ++mt) {
                part_s[warp][h][kDim0 * g + mt] = kRest ? o[mt][0] + o[mt][1] : o[mt][c];
                part_s[warp][h][kDim0 * g + kDim8 + mt] = kRest ? o[mt][2] + o[mt][3] : o[mt][c + 2];
            }
            if (g == 0) { part_s[warp][h][kHeadDim] = m[c]; part_s[warp][h][kHeadDim + 1] = l[c]; }
        }
    }
    __syncthreads();
    if constexpr (kCluster) cooperative_groups::this_cluster().barrier_wait();
    for (int i = threadIdx.x; i < G * kHeadDim; i += 256) {
        const int h = i / kHeadDim, d = i % kHeadDim;
        float M = -1e30f;
#pragma unroll
        for (int w2 = 0; w2 < 8; ++w2) M = fmaxf(M, part_s[w2][h][kHeadDim]);
        float L = 0.f, acc = 0.f;
#pragma unroll
        for (int w2 = 0; w2 < 8; ++w2) {
            const float c = exp2f(part_s[w2][h][kHeadDim] - M);
            L = fmaf(part_s[w2][h][kHeadDim + 1], c, L);
            acc = fmaf(part_s[w2][h][d], c, acc);
        }
        const int qh = kh * G + h;
        if constexpr (kCluster) {       // to the first split of the cluster, which merges them
            float* dst = cooperative_groups::this_cluster().map_shared_rank(&merge_s[0][0][0], 0) + (split * G + h) * kPartialFloats;
            dst[d] = acc;
            if (d == 0) { dst[kHeadDim] = M; dst[kHeadDim + 1] = L; }
        } else if (p.n_splits == 1) {
            p.O[(long long)b * p.o_b + (long long)qh * p.o_h + d] = __float2bfloat16_rn(acc / L);
        } else {
            float* dst = p.partial + (((size_t)b * p.Hq + qh) * p.n_splits + split) * kPartialFloats;
            dst[d] = acc;
            if (d == 0) { dst[kHeadDim] = M; dst[kHeadDim + 1] = L; }
        }
    }
    if constexpr (kCluster) {
        cooperative_groups::this_cluster().sync();
        if (split != 0) return;
        for (int i = threadIdx.x; i < G * kHeadDim; i += 256) {
            const int h = i / kHeadDim, d = i % kHeadDim;
            float M = -1e30f, L = 0.f, acc = 0.f;
            for (int q = 0; q < p.n_splits; ++q) M = fmaxf(M, merge_s[q][h][kHeadDim]);
            for (int q = 0; q < p.n_splits; ++q) {
                const float c = exp2f(merge_s[q][h][kHeadDim] - M);
                L = fmaf(merge_s[q][h][kHeadDim + 1], c, L);
                acc = fmaf(merge_s[q][h][d], c, acc);
            }
            p.O[(long long)b * p.o_b + (long long)(kh * G + h) * p.o_h + d] = __float2bfloat16_rn(acc / L);
        }
    }
}

// merges the splits of one (query head, sequence); a skipped token gets its zero row here
__global__ void __launch_bounds__(kHeadDim) decode_merge_splits_kernel(const DecGqaParams p) {
    grid_dependency_wait();
    const int qh = blockIdx.x, b = blockIdx.y, d = threadIdx.x;
    __nv_bfloat16* out = p.O + (long long)b * p.o_b + (long long)qh * p.o_h + d;
    const bool skip = p.skip[b] != 0;
    const float* base = p.partial + ((size_t)b * p.Hq + qh) * p.n_splits * kPartialFloats;
    float M = -1e30f, L = 0.f, acc = 0.f;
    for (int q0 = 0; q0 < p.n_splits; q0 += 8) {            // eight splits requested together (a skipped token's are stale, and not used)
        float m[8], l[8], v[8], mx = M;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float* src = base + (size_t)min(q0 + u, p.n_splits - 1) * kPartialFloats;
            m[u] = src[kHeadDim]; l[u] = src[kHeadDim + 1]; v[u] = src[d];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) mx = fmaxf(mx, m[u]);
        const float e0 = exp2f(M - mx);
        L *= e0; acc *= e0; M = mx;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float e = q0 + u < p.n_splits ? exp2f(m[u] - M) : 0.f;
            L = fmaf(l[u], e, L);
            acc = fmaf(v[u], e, acc);
        }
    }
    *out = skip ? __float2bfloat16_rn(0.f) : __float2bfloat16_rn(acc / L);
}

// the launch of a grid of clusters of grid.x CTAs (attr: two entries that outlive the call)
static cudaLaunchConfig_t cluster_config(dim3 grid, cudaStream_t st, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = 0; cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = grid.x; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 2;
    return cfg;
}
template <int G>
static cudaError_t launch_split(const DecGqaParams& gp, dim3 grid, bool cluster, bool early, cudaStream_t st) {
    if (G > 4 || !cluster) return launch_dependent(early ? decode_attention_split_kernel<G, kEarly> : decode_attention_split_kernel<G, kAfterDecision>, grid, dim3(256), 0, st, gp);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(grid, st, attr);
    return cudaLaunchKernelEx(&cfg, decode_attention_split_kernel<(G > 4 ? 4 : G), kAsCluster>, gp);
}
// how many clusters of n CTAs (2 .. 8) the device runs at once: a property of the device and the kernel, asked for once
static int max_clusters(int device, int G, int n) {
    static std::atomic<int> known[kDeviceFlagSlots][3][9] = {};      // + 1; 0: not asked yet
    std::atomic<int>& k = known[device >= 0 && device < kDeviceFlagSlots ? device : 0][G >> 1][n];
    int v = k.load(std::memory_order_relaxed);
    if (v == 0) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = cluster_config(dim3((unsigned)n), nullptr, attr);
        cfg.numAttrs = 1;
        int most = 0;
        const cudaError_t e = G == 1 ? cudaOccupancyMaxActiveClusters(&most, decode_attention_split_kernel<1, kAsCluster>, &cfg)
                            : G == 2 ? cudaOccupancyMaxActiveClusters(&most, decode_attention_split_kernel<2, kAsCluster>, &cfg)
                                     : cudaOccupancyMaxActiveClusters(&most, decode_attention_split_kernel<4, kAsCluster>, &cfg);
        if (e != cudaSuccess) { (void)cudaGetLastError(); most = 0; }
        v = most + 1;
        k.store(v, std::memory_order_relaxed);
    }
    return v - 1;
}

// The scratch of a step lies at the END of the bound workspace, the records that a scan keeps from call to call at the front: a
// workspace of tf_workspace_bytes holds both.  (At the front the records had to be cleared before the next scan, which the host
// only knows of a step that it launches itself, not of one that is replayed from a CUDA graph.)  In a smaller workspace, where
// they overlap, the next scan clears its region first.
static char* step_scratch(tf_ctx* ctx, size_t bytes) {
    const size_t at = (ctx->workspace_bytes - bytes) & ~(size_t)255;
    if (at < (ctx->scan_user.bytes & ~(size_t)1)) ctx->scan_user.needs_clear = true;      // (the low bit is not part of the extent)
    return static_cast<char*>(ctx->workspace) + at;
}

// How the split kernel divides the visible keys of a (sequence, KV head), at least 256 keys each.  Through scratch: two CTAs fit an
// SM, a wave of CTAs costs (a fixed part worth ~192 keys + its keys), and a partly filled wave costs as much as a full one; the
// cheapest estimate.  As a cluster, of as many splits (8 at most, as short as 64 keys) as let the clusters of all groups run at
// once: no third launch, which is worth ~400 keys of a CTA (us a step, keys from HBM, cluster / scratch, 8 KV heads x 4: 1 x 2048 keys
// 8.3 / 10.1, 1 x 4096 11.0 / 11.3, 4 x 1500 10.4 / 13.6, 4 x 2500 13.5 / 15.2, 8 x 1400 14.9 / 14.9, 8 x 1700 16.6 / 16.9; the difference of
// keys above 400: 4 x 4096 20.5 / 18.5, 1 x 8192 19.3 / 15.4).  Clusters that wait for one another's SMs lose: 2 x 420 keys in 6 splits 6.9, in
// 7 9.9.  Without room for partial results a cluster is always the better one: 1 x 8192 19.4, as 8 whole items 88.9; 1 x 4000 x 40 ungrouped
// 24.4 / 49.3.
struct SplitPlan { int n; bool cluster; };
static size_t split_bytes(const tf_shape& s) { return (size_t)s.batch * s.n_q_heads * kPartialFloats * sizeof(float); }     // of one split
static SplitPlan split_plan(const tf_ctx* ctx, const tf_shape& s, int G, int max_keys, int sms) {
    const long long groups = (long long)s.batch * s.n_kv_heads, slots = 2ll * sms;
    SplitPlan plan{1, false};
    long long best = -1, keys_at_once = 0;                  // (of a CTA of every wave)
    for (int n = 1; n <= std::max(1, max_keys / 256); ++n) {
        if (n > 1 && (!ctx->workspace || ctx->workspace_bytes < split_bytes(s) * n)) break;
        const long long waves = (groups * n + slots - 1) / slots, keys = (max_keys + n - 1) / n, cost = waves * (192 + keys);
        if (best < 0 || cost < best) { best = cost; plan.n = n; keys_at_once = waves * keys; }
    }
    int n = G <= 4 ? (int)std::min<long long>(std::min(8, max_keys / 64), sms / groups) : 1;
    while (n > 1 && groups > max_clusters(ctx->device, G, n)) --n;
    if (n > 1 && (max_keys + n - 1) / n <= keys_at_once + (plan.n > 1 ? 400 : 0)) plan = {n, true};
    return plan;
}

cudaError_t launch_decode_step(tf_ctx* ctx, const tf_shape& s, const tf_filter_params& p, const tf_decode_args& a,
                               cudaStream_t st) {
    if (s.batch == 0) return cudaSuccess;
    DecideParams dp{};
    dp.K = a.K_cache; dp.V = a.V_cache;
    dp.ks = {s.k_stride[0], s.k_stride[1], s.k_stride[2]};
    dp.vs = {s.v_stride[0], s.v_stride[1], s.v_stride[2]};
    dp.pos = a.pos; dp.Hkv = s.n_kv_heads; dp.anchor_mode = p.anchor_mode; dp.fuse_mode = p.fuse_mode;
    dp.warmup = p.warmup_tokens; dp.gamma = p.gamma; dp.var_eps = p.var_eps > 0.f ? p.var_eps : 1e-8f;
    dp.eta = a.eta; dp.target = p.prune_ratio; dp.alg1_sign = a.alg1_sign;
    dp.sum_k = a.state->sum_k; dp.sum_v = a.state->sum_v; dp.count = reinterpret_cast<long long*>(a.state->count);
    dp.sums16 = ((reinterpret_cast<uintptr_t>(dp.sum_k) | reinterpret_cast<uintptr_t>(dp.sum_v)) & 15u) == 0;
    // bf16 with 1, 2, 4 or 8 query heads per KV head and 16-byte aligned query rows: the streaming kernel for ungrouped heads, the split
    // kernel otherwise (both sides' times stand at the split kernel) ...
    const int G = s.n_q_heads / s.n_kv_heads;
    const int sms = sm_count();
    const int max_keys = s.window > 0 ? std::min(s.window, s.seq) : s.seq;     // pos is device data: size for the worst case
    const long long tiles_max = (long long)s.batch * s.n_kv_heads * ((max_keys + kStreamKeys - 1) / kStreamKeys);
    const bool grouped = s.dtype == TF_BF16 && (G == 1 || G == 2 || G == 4 || G == 8) && ((s.q_stride[0] | s.q_stride[2]) % 8) == 0 &&
                         (reinterpret_cast<uintptr_t>(a.q_new) & 15u) == 0;
    StreamMaps maps;
    auto make_maps = [&](int b0, int n) {
        const __nv_bfloat16* K = static_cast<const __nv_bfloat16*>(a.K_cache) + (long long)b0 * s.k_stride[0];
        const __nv_bfloat16* V = static_cast<const __nv_bfloat16*>(a.V_cache) + (long long)b0 * s.v_stride[0];
        bool ok = true;
        for (int x = 0; x < kStreamBoxes; ++x)
            ok = ok && make_bshd_map(&maps.k[x], K, s.k_stride, n, s.seq, s.n_kv_heads, 2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 64, 16 * (x + 1), CU_TENSOR_MAP_SWIZZLE_128B)
                    && make_bshd_map(&maps.v[x], V, s.v_stride, n, s.seq, s.n_kv_heads, 2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 64, 16 * (x + 1), CU_TENSOR_MAP_SWIZZLE_128B);
        return ok;
    };
    // ... but not for short steps, where the streaming kernel's list and hand-overs are not paid back: up to 18 tiles of 64 keys per SM,
    // 34 where the split kernel's CTAs fill one wave or two well, 48 where these are two of whole items; beyond it shares drawn by whoever
    // is free outweigh them once sequences are skipped.  us a step of full caches from HBM, streaming / split, none skipped and half of them:
    //   no full waves: 1 x 1000 x 40 heads 14.4 / 8.0; 40 x 500 x 8 (17 tiles) 23.8 / 22.4, 22.5 / 14.9; 24 x 250 x 32 (21) 27.1 / 29.7, 23.7 / 20.8;
    //     12 x 600 x 32 (26) 32.0 / 37.1; 24 x 400 x 32 (36) 35.0 / 42.0, 28.1 / 28.8
    //   one: 8 x 1024 x 32 (28) 30.6 / 26.4, 23.7 / 22.1; 1 x 8000 x 40 (34) 34.5 / 32.4; 7 x 1500 x 40 (45) 42.3 / 38.3, 26.4 / 29.6;
    //     20 x 2000 x 12 (52) 47.7 / 42.7, 31.3 / 36.1
    //   two of whole items: 16 x 600 x 32 (35) 33.7 / 31.5, 26.5 / 21.2; 16 x 850 x 32 (48) 43.1 / 41.1, 30.3 / 26.0; 15 x 1000 x 32 (52) 46.9 / 44.9,
    //     a fifth skipped 41.0 / 43.3; 18 x 2500 x 32 (156) 120 / 116, a fifth 99.8 / 100.2
    // (5 tiles where more than two waves of whole items stream without a merge launch: 19 x 47 x 32 (4) 15.0 / 15.5, a third skipped 14.1 / 13.0;
    // 28 x 47 x 32 (6) 17.1 / 18.7, 16.0 / 16.1; 18 x 130 x 40 (15) 18.8 / 23.3, 18.2 / 18.8.)
    // Nor with one or two tiles in several launches (600 x 64 x 8 69.0 / 64.3).  Where work items are whole for want of room, an SM has one at most and they are longer than 4 tiles, the ring of the
    // streaming kernel is the faster way through them, and a cluster faster than both (no workspace, streaming / whole items of the
    // split kernel, 90 items: 192 keys 9.9 / 8.8, 384 10.6 / 11.3, 2000 22.9 / 30.0; 148 items: 10.9 / 10.1, 12.3 / 14.0, 28.8 / 37.2; 160 items:
    // 13.4 / 10.0, 16.5 / 13.9, 44.2 / 37.7; streaming / clusters: 74 items of 4000 37.6 / 32.4, 40 of 16384 130 / 66, 8 of 30000 222 / 44).
    const long long items = (long long)s.batch * s.n_kv_heads;
    const SplitPlan plan = grouped ? split_plan(ctx, s, G, max_keys, sms) : SplitPlan{1, false};
    const long long split_ctas = items * plan.n, waves = (split_ctas + 2 * sms - 1) / (2 * sms);
    const bool filled = waves <= 2 && 5 * split_ctas >= 4 * waves * 2 * sms;
    auto stream_grid = [&](int n) { return (int)std::min<long long>(sms, (long long)n * s.n_kv_heads * ((max_keys + kStreamKeys - 1) / kStreamKeys)); };
    const int first_grid = stream_grid(std::min<int>(s.batch, kStreamMaxBatch));      // (none after it is larger)
    // scratch of the streaming kernel: the table of begun work items, then slots: two per piece, and there have to be more
    // pieces than CTAs
    const size_t table = stream_table_bytes(first_grid), slot = kPartialFloats * sizeof(float);
    const bool pieces = ctx->workspace && ctx->workspace_bytes >= table + (3 * (size_t)first_grid + 2) * slot;
    const bool few_short = tiles_max <= (!filled ? (waves > 2 && !pieces ? 5ll : 18ll) : waves == 2 && plan.n == 1 ? 48ll : 34ll) * sms || (s.batch > kStreamMaxBatch && max_keys <= 2 * kStreamKeys);
    const bool split = plan.n == 1 && items <= sms && !pieces ? max_keys <= 4 * kStreamKeys : few_short || (plan.cluster && !pieces);
    const bool stream = grouped && G == 1 && !split && tiles_max < (1ll << 31) &&              // (tile numbers are 32 bits)
                        ((s.o_stride[0] | s.o_stride[2]) % 8) == 0 && (reinterpret_cast<uintptr_t>(a.O_new) & 15u) == 0 &&
                        (s.batch == 1 || (s.k_stride[0] > 0 && s.v_stride[0] > 0)) && make_maps(0, std::min<int>(s.batch, kStreamMaxBatch));
    DecStreamParams sp{};
    if (stream && pieces) {
        const size_t scratch = std::min(ctx->workspace_bytes, table + kStreamScratch);
        char* at = step_scratch(ctx, scratch);
        sp.begun = reinterpret_cast<uint4*>(at) + 1;
        sp.partial = reinterpret_cast<float*>(at + table);
        sp.max_slots = (unsigned int)((scratch - table) / slot);
        dp.next_piece = &sp.begun[-1].y;
    }
    dp.tau = a.state->tau; dp.steps = reinterpret_cast<long long*>(a.state->steps);
    dp.skips = reinterpret_cast<long long*>(a.state->skips);
    dp.score_out = a.score_out; dp.skip_out = a.skip_out; dp.status = ctx->dev_status;
    // The attention starts while the decisions are made where that is worth it: what it loads for skipped tokens is lost, and with
    // many waves little is gained (128 x 1024 keys x 8 heads, half of them skipped, 54.8 instead of 51.1 us).  In two waves of two or
    // four heads a group the loss outweighs it (us a step, early / after the decision, none, a fifth and half of them skipped: 22 x 1024 of 15739
    // keys x 8 x 4 24.6 / 25.8, 23.6 / 24.6, 18.6 / 16.4; 70 x 300 23.1 / 23.6, 21.7 / 22.3, 18.5 / 16.7; a caller's launches cover most of what the early
    // start gains, 25.8 / 26.1 and 23.7 / 23.7); ungrouped heads spill registers in the other form (16 x 850 x 32 41.1 / 50.4, 26.1 / 30.0).
    dp.early = stream || (grouped && waves <= (G == 2 || G == 4 ? 1 : 2)) ? 1 : 0;
    const size_t smem = 2 * (size_t)s.n_kv_heads * sizeof(float);
    cudaError_t e;
    // up to 8 heads a warp has one, beyond it two (two for 8: 1 x 100 keys x 8 heads fp32 15.3 us a step)
    const bool two = s.n_kv_heads > 8;
    const dim3 decide_block(32u * std::min(kDecideWarps, two ? (s.n_kv_heads + 1) / 2 : std::max(s.n_kv_heads, 4)));
    auto decide = s.dtype == TF_BF16 ? (two ? decode_decide_kernel<__nv_bfloat16, 2> : decode_decide_kernel<__nv_bfloat16, 1>)
                                     : (two ? decode_decide_kernel<float, 2> : decode_decide_kernel<float, 1>);
    e = launch_dependent(decide, dim3((unsigned)s.batch), decide_block, smem, st, dp);
    ctx->launches += 1;
    if (e != cudaSuccess) return e;

    DecAttnParams ap{};
    ap.Q = a.q_new; ap.K = a.K_cache; ap.V = a.V_cache; ap.O = a.O_new;
    ap.q_b = s.q_stride[0]; ap.q_h = s.q_stride[2]; ap.o_b = s.o_stride[0]; ap.o_h = s.o_stride[2];
    ap.ks = dp.ks; ap.vs = dp.vs; ap.pos = a.pos; ap.skip = a.skip_out;
    ap.Hq = s.n_q_heads; ap.Hkv = s.n_kv_heads; ap.window = s.window;
    const float scale = s.softmax_scale != 0.f ? s.softmax_scale : 1.f / sqrtf((float)s.head_dim);
    ap.scale_log2 = scale * 1.4426950408889634f;
    if (grouped && !stream) {
        DecGqaParams gp{};
        gp.Q = static_cast<const __nv_bfloat16*>(a.q_new); gp.K = static_cast<const __nv_bfloat16*>(a.K_cache);
        gp.V = static_cast<const __nv_bfloat16*>(a.V_cache); gp.O = static_cast<__nv_bfloat16*>(a.O_new);
        gp.q_b = ap.q_b; gp.q_h = ap.q_h; gp.o_b = ap.o_b; gp.o_h = ap.o_h;
        gp.ks = ap.ks; gp.vs = ap.vs; gp.pos = a.pos; gp.skip = a.skip_out;
        gp.Hq = s.n_q_heads; gp.Hkv = s.n_kv_heads; gp.window = s.window; gp.scale_log2 = ap.scale_log2;
        gp.n_splits = plan.n;
        gp.n_early = 2 * sms;
        const bool scratch = plan.n > 1 && !plan.cluster;
        gp.partial = scratch ? reinterpret_cast<float*>(step_scratch(ctx, split_bytes(s) * plan.n)) : nullptr;
        const dim3 grid((unsigned)plan.n, (unsigned)s.n_kv_heads, (unsigned)s.batch);
        switch (G) {
            case 1: e = launch_split<1>(gp, grid, plan.cluster, dp.early != 0, st); break;
            case 2: e = launch_split<2>(gp, grid, plan.cluster, dp.early != 0, st); break;
            case 4: e = launch_split<4>(gp, grid, plan.cluster, dp.early != 0, st); break;
            default: e = launch_split<8>(gp, grid, false, dp.early != 0, st); break;
        }
        ctx->launches += 1;
        if (e == cudaSuccess && scratch) {
            e = launch_dependent(decode_merge_splits_kernel, dim3((unsigned)s.n_q_heads, (unsigned)s.batch), dim3(kHeadDim), 0, st, gp);
            ctx->launches += 1;
        }
        return e;
    }
    if (stream) {
        sp.q_b = ap.q_b; sp.q_h = ap.q_h; sp.o_b = ap.o_b; sp.o_h = ap.o_h;
        sp.Hq = s.n_q_heads; sp.Hkv = s.n_kv_heads; sp.window = s.window; sp.scale_log2 = ap.scale_log2;
        sp.status = ctx->dev_status; sp.wait_cycles = ctx_wait_cycles(ctx);
        for (int b0 = 0; b0 < s.batch; b0 += kStreamMaxBatch) {
            const int n = std::min(s.batch - b0, kStreamMaxBatch);
            if (b0 > 0 && !make_maps(b0, n)) return cudaErrorInvalidValue;
            sp.B = n;
            sp.Q = static_cast<const __nv_bfloat16*>(a.q_new) + (long long)b0 * ap.q_b;
            sp.O = static_cast<__nv_bfloat16*>(a.O_new) + (long long)b0 * ap.o_b;
            sp.pos = a.pos + b0; sp.skip = a.skip_out + b0;
            e = launch_stream(sp, stream_grid(n), ctx->device, maps, st);
            ctx->launches += sp.begun ? 2 : 1;
            if (e != cudaSuccess) return e;
        }
        return e;
    }
    const dim3 grid((unsigned)s.n_q_heads, (unsigned)s.batch);
    if (s.dtype == TF_BF16) e = launch_dependent(decode_attention_kernel<__nv_bfloat16>, grid, dim3(kDecWarps * 32), 0, st, ap);
    else                    e = launch_dependent(decode_attention_kernel<float>, grid, dim3(kDecWarps * 32), 0, st, ap);
    ctx->launches += 1;
    return e;
}

}  // namespace tf
