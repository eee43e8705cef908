// Step a5 on CUDA cores: causal (optionally windowed) attention for retained tokens, any dtype.
//
// This is the path fp32 tensors take (fp32 accuracy rules out the 16-bit tensor-core path) and the A/B reference for the
// tensor-core kernel.  A CTA of 8 warps owns 16 or 32 consecutive entries of a sequence's retained list for one query
// head; keys and values go through shared memory in chunks of 64.  A warp owns 4 rows of the tile: lane l scores keys l and
// l + 32 of a chunk for all of them (keys from shared memory, queries by broadcast), the warp runs the online softmax,
// and each lane accumulates 4 output dims of its 4 rows over the chunk.  Scores, probabilities and sums are fp32 throughout.
//   kSplit = 1 (32 rows): all warps work on the same chunk, two CTAs per SM.
//   kSplit = 2 (16 rows): the two halves of the CTA take alternate chunks of the same rows and are merged at the end: twice
//                         as many CTAs with half the serial length, for problems that would leave SMs idle.
// The next chunk's keys are fetched (cp.async) under the P V part, its values under the next Q K part.  Shared-memory reads
// bound it: per 4 dims 16 wavefronts (a 16-byte broadcast is two) for 8 cycles of multiply-adds in Q K^T, 24 for 16 in P V.
// The CTA also zeroes the output rows of the pruned tokens before its rows (Section 3.2: a skipped token's attention output is
// zero), all warps and before the chunks, so the whole of O is written with no separate clearing pass.  Under a window it
// passes over chunks that none of its rows sees.
//   One warp per row, a key at a time per lane straight from global memory, took 48 us at 1 x 128 tokens x 32 heads (half of them
// retained); this kernel takes 11.8, 32 at 300 tokens and 405 at 2 x 1024 x 40 heads (71 % of the shared-memory wavefronts).
// CTAs with rows start before those expected to have none, over all heads (a quarter to a half of the grid was empty CTAs
// between the others), and inside a layer step the first chunk is fetched while the selection runs: per pass 1 x 300 x 32
// heads 63.5 -> 52.4 us, 1 x 700 143 -> 119, 2 x 1000 571 -> 506.
#include <algorithm>
#include <type_traits>

#include "tf_common.cuh"

namespace tf {

constexpr int kSimtChunk = 64;         // keys per chunk
constexpr int kSimtWarps = 8;
constexpr int kSimtThreads = kSimtWarps * 32;
constexpr int kSimtRows = 4;           // rows per warp

struct AttnParams {
    const void* Q; const void* K; const void* V; void* O;
    Strides3 qs, ks, vs, os;
    int S, Hq, Hkv, window;
    float scale_log2;          // softmax scale * log2(e)
    const int32_t* kept_idx;   // [B,S]
    const int32_t* n_kept;     // [B]
    int n_blocks, blocks_est;  // row blocks per head / those expected to hold retained rows (they start first)
    int early;                 // 1: the selection kernel is the one before this on the stream and the first chunk is known
    int retained_only;         // 1: a retained query sees retained tokens' keys / values only
};

template <int kSplit> struct SimtCfg {                                   // kSplit: parts of the CTA with chunks of their own
    static constexpr int kPartThreads = kSimtThreads / kSplit;
    static constexpr int kRows = kSimtWarps / kSplit * kSimtRows;
    static constexpr int kChunkFloats = kSimtChunk * kHeadDim;
    static constexpr int kOffQ = 2 * kSplit * kChunkFloats;              // [part][K, V] chunks first
    static constexpr int kOffP = kOffQ + kRows * kHeadDim;               // [warp][row][64]
    static constexpr int kSmemBytes = (kOffP + kSimtWarps * kSimtRows * kSimtChunk) * 4;
};

__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) { *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d); }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float a, float b, float c, float d) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
}
// four consecutive elements (16 bytes of fp32, 8 bytes of bf16; the caller's offset is a multiple of four elements)
__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}
// four elements from global to shared memory (zeros unless live); fp32: asynchronously
__device__ __forceinline__ void fetch4(float* dst, const float* src, bool live) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" :: "r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void fetch4(float* dst, const __nv_bfloat16* src, bool live) {
    *reinterpret_cast<float4*>(dst) = live ? load4(src) : make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void fetch_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void fetch_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void fetch_wait_all_but_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// a += w * v where `yes`, without a branch
__device__ __forceinline__ void fma4_if(float (&a)[4], float w, const float4& v, bool yes) {
    asm("{\n.reg .pred p;\nsetp.ne.u32 p, %9, 0;\n@p fma.rn.f32 %0, %4, %5, %0;\n@p fma.rn.f32 %1, %4, %6, %1;\n"
        "@p fma.rn.f32 %2, %4, %7, %2;\n@p fma.rn.f32 %3, %4, %8, %3;\n}"
        : "+f"(a[0]), "+f"(a[1]), "+f"(a[2]), "+f"(a[3]) : "f"(w), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((unsigned int)yes));
}

template <typename T>
__device__ __forceinline__ void zero_rows(T* Ob, const Strides3& os, int t_lo, int t_hi, int lane) {
    for (int t = t_lo; t < t_hi; ++t) store4(Ob + (long long)t * os.t + lane * 4, 0.f, 0.f, 0.f, 0.f);
}

template <typename T, int kSplit>
__global__ void __launch_bounds__(kSimtThreads, kSplit == 2 ? 1 : 2) attention_simt_kernel(const AttnParams p) {
    using C = SimtCfg<kSplit>;
    constexpr int R = kSimtRows;
    extern __shared__ __align__(16) float simt_smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int part = warp / (kSimtWarps / kSplit), ptid = tid & (C::kPartThreads - 1);
    const int rgroup = warp & (kSimtWarps / kSplit - 1);
    const int qh = (int)blockIdx.x % p.Hq, b = blockIdx.z, rb = (int)blockIdx.x / p.Hq;
    const int blk = p.blocks_est - 1 - rb + (rb < p.blocks_est ? 0 : p.n_blocks);     // the longest rows first, empty blocks last
    const int slot0 = blk * C::kRows;
    const int32_t* kept = p.kept_idx + (size_t)b * p.S;
    T* Ob = reinterpret_cast<T*>(p.O) + (long long)b * p.os.b + (long long)qh * p.os.h;
    float* const sK = simt_smem + part * 2 * C::kChunkFloats;
    float* const sV = sK + C::kChunkFloats;
    float* const sQ = simt_smem + C::kOffQ;
    float* const sP = simt_smem + C::kOffP + warp * R * kSimtChunk;
    const int kh = qh / (p.Hq / p.Hkv);
    const T* Kb = reinterpret_cast<const T*>(p.K) + (long long)b * p.ks.b + (long long)kh * p.ks.h;
    const T* Vb = reinterpret_cast<const T*>(p.V) + (long long)b * p.vs.b + (long long)kh * p.vs.h;
    // one 16-byte piece per thread and step; the pieces of a key row are rotated (XOR) by the row so that lanes reading the
    // same piece of 8 consecutive rows hit different banks
    auto fetch = [&](float* dst, const T* base, long long stride, int ch, int last, bool swizzle) {
#pragma unroll 4
        for (int i = ptid; i < kSimtChunk * 32; i += C::kPartThreads) {
            const int row = i >> 5, piece = i & 31, j = ch * kSimtChunk + row;
            const bool live = j <= last;
            const long long tok = live ? (p.retained_only ? kept[j] : j) : 0;
            fetch4(dst + row * kHeadDim + ((swizzle ? piece ^ (row & 7) : piece) << 2), base + tok * stride + piece * 4, live);
        }
        fetch_commit();
    };
    // the first chunk of keys and values does not depend on the selection: it is fetched while that still runs
    const bool early = p.early && blk < p.blocks_est && part * kSimtChunk < p.S;
    if (early) { fetch(sK, Kb, p.ks.t, part, p.S - 1, true); fetch(sV, Vb, p.vs.t, part, p.S - 1, false); }
    grid_dependency_wait();
    const int nk = p.n_kept[b];
    if (slot0 >= nk) {
        if (nk == 0 && slot0 == 0)
            for (int t = warp; t < p.S; t += kSimtWarps) zero_rows(Ob, p.os, t, t + 1, lane);
        fetch_wait_all();
        return;
    }

    // keys are visited by index: token positions, or positions in the retained list (retained_only), where entry c stands
    // for token kept[c] and the query itself is its own entry.  Lane l of every warp looks up row l of the CTA.
    const int slot_l = slot0 + lane, last_row = min(C::kRows, nk - slot0) - 1;
    const int t_l = lane <= last_row ? kept[slot_l] : -1, t_before = slot0 > 0 ? kept[slot0 - 1] : -1;
    int lo_l = 0, hi_l = -1;                                                // visible keys of the row (hi < lo: no such row)
    if (lane <= last_row) {
        const int t_min = p.window > 0 ? max(0, t_l - p.window + 1) : 0;
        lo_l = p.retained_only ? (t_min > 0 ? first_kept_at_or_after(kept, slot_l + 1, t_min) : 0) : t_min;
        hi_l = p.retained_only ? slot_l : t_l;
    }
    __syncwarp();
    const int c_hi = __shfl_sync(0xffffffffu, hi_l, last_row);             // the CTA's last visible key
    const int ch1 = c_hi / kSimtChunk + 1;
    // the first chunk from c on that some row sees: rows of a sparse list with a short window leave chunks between them
    auto seen_from = [&](int c) {
        if (p.window == 0) return c;
        const int mine = hi_l / kSimtChunk >= c && hi_l >= 0 ? max(c, lo_l / kSimtChunk) : ch1;
        return (int)__reduce_min_sync(0xffffffffu, (unsigned int)mine);
    };
    auto advance = [&](int c) {
        if (p.window == 0) return c + kSplit;
#pragma unroll
        for (int i = 0; i < kSplit; ++i) c = seen_from(c + 1);
        return c;
    };

    auto part_sync = [&]() {
        if (kSplit == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" :: "r"(1 + part), "n"(C::kPartThreads) : "memory");
    };
    int ch = seen_from(0);
    if (part) ch = seen_from(ch + 1);
    if (!early && ch < ch1) { fetch(sK, Kb, p.ks.t, ch, c_hi, true); fetch(sV, Vb, p.vs.t, ch, c_hi, false); }
    for (int i = tid; i < C::kRows * 32; i += kSimtThreads) {
        const int row = i >> 5, piece = i & 31, slot = slot0 + row;
        float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
        if (slot < nk)
            q = load4(reinterpret_cast<const T*>(p.Q) + (long long)b * p.qs.b + (long long)kept[slot] * p.qs.t + (long long)qh * p.qs.h + piece * 4);
        *reinterpret_cast<float4*>(sQ + row * kHeadDim + piece * 4) = make_float4(q.x * p.scale_log2, q.y * p.scale_log2, q.z * p.scale_log2, q.w * p.scale_log2);
    }
    const int row0 = rgroup * R;
    int lo[R], hi[R], w_lo = 0x7fffffff, w_hi = -1;                     // visible keys of each row of the warp
    int all_lo = 0, all_hi = 0x7fffffff;                                // keys that every row of the warp sees
#pragma unroll
    for (int r = 0; r < R; ++r) {
        lo[r] = __shfl_sync(0xffffffffu, lo_l, row0 + r);
        hi[r] = __shfl_sync(0xffffffffu, hi_l, row0 + r);
        if (row0 + r <= last_row) {
            w_lo = min(w_lo, lo[r]); w_hi = max(w_hi, hi[r]);
            all_lo = max(all_lo, lo[r]); all_hi = min(all_hi, hi[r]);
        }
    }
    // the rows of pruned tokens before each retained one (and behind the last of all) are zero; the stores run under the chunks
#pragma unroll
    for (int i = 0; i < C::kRows / kSimtWarps; ++i) {
        const int row = warp * (C::kRows / kSimtWarps) + i;
        const int t = __shfl_sync(0xffffffffu, t_l, row), before = __shfl_sync(0xffffffffu, t_l, max(row - 1, 0));
        if (row > last_row) break;
        zero_rows(Ob, p.os, (row == 0 ? t_before : before) + 1, t, lane);
        if (slot0 + row == nk - 1) zero_rows(Ob, p.os, t + 1, p.S, lane);
    }
    __syncthreads();

    float m[R], l[R], acc[R][4];                                          // l: this lane's share of the row's sum
#pragma unroll
    for (int r = 0; r < R; ++r) { m[r] = -1e30f; l[r] = 0.f; acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0.f; }
    auto weigh = [&](int jj, int j0, auto edge) {                         // four keys' values into the rows' sums
        float4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = reinterpret_cast<const float4*>(sV)[(jj + u) * 32 + lane];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float4 w = *reinterpret_cast<const float4*>(sP + r * kSimtChunk + jj);
            const float wu[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if constexpr (decltype(edge)::value) {
                    fma4_if(acc[r], wu[u], v[u], j0 + jj + u >= lo[r] && j0 + jj + u <= hi[r]);
                } else {
                    acc[r][0] = fmaf(wu[u], v[u].x, acc[r][0]); acc[r][1] = fmaf(wu[u], v[u].y, acc[r][1]);
                    acc[r][2] = fmaf(wu[u], v[u].z, acc[r][2]); acc[r][3] = fmaf(wu[u], v[u].w, acc[r][3]);
                }
            }
        }
    };
    for (int ch_next; ch < ch1; ch = ch_next) {
        const int j0 = ch * kSimtChunk;
        ch_next = advance(ch);
        const bool mine = w_hi >= j0 && w_lo < j0 + kSimtChunk;            // some row of this warp sees this chunk
        fetch_wait_all_but_one();
        part_sync();                                                       // K(ch) is there
        float s[R][2];
        if (mine) {
            // the even and the odd dims of a score are summed apart, two products per instruction.  One chain of 128 left an
            // error of 5.9e-7 (2-norm over 2-norm, 1 x 700 tokens, against 64 bits), two chains of 64 leave 3.8e-7.
            uint64_t s2[R][2];
#pragma unroll
            for (int r = 0; r < R; ++r) s2[r][0] = s2[r][1] = 0ull;
            const ulonglong2* k4 = reinterpret_cast<const ulonglong2*>(sK) + lane * 32;
            const ulonglong2* q4 = reinterpret_cast<const ulonglong2*>(sQ) + row0 * 32;
#pragma unroll 4
            for (int d = 0; d < 32; ++d) {
                const ulonglong2 ka = k4[d ^ (lane & 7)], kb = k4[32 * 32 + (d ^ (lane & 7))];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const ulonglong2 q = q4[r * 32 + d];
                    s2[r][0] = fma2(q.x, ka.x, s2[r][0]); s2[r][1] = fma2(q.x, kb.x, s2[r][1]);
                    s2[r][0] = fma2(q.y, ka.y, s2[r][0]); s2[r][1] = fma2(q.y, kb.y, s2[r][1]);
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    float even, odd;
                    unpack2(s2[r][c], even, odd);
                    s[r][c] = even + odd;
                }
        }
        part_sync();                                                       // K(ch) has been read
        if (ch_next < ch1) fetch(sK, Kb, p.ks.t, ch_next, c_hi, true); else fetch_commit();
        if (mine) {
            const int ja = j0 + lane, jb = ja + 32;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const bool va = ja >= lo[r] && ja <= hi[r], vb = jb >= lo[r] && jb <= hi[r];
                const float sa = va ? s[r][0] : -1e30f, sb = vb ? s[r][1] : -1e30f;
                const float m_new = fmaxf(m[r], warp_max(fmaxf(sa, sb)));
                const float corr = exp2f(m[r] - m_new);
                const float pa = va ? exp2f(sa - m_new) : 0.f, pb = vb ? exp2f(sb - m_new) : 0.f;
                m[r] = m_new;
                l[r] = fmaf(l[r], corr, pa + pb);
                acc[r][0] *= corr; acc[r][1] *= corr; acc[r][2] *= corr; acc[r][3] *= corr;
                sP[r * kSimtChunk + lane] = pa;
                sP[r * kSimtChunk + 32 + lane] = pb;
            }
            __syncwarp();
        }
        fetch_wait_all_but_one();
        part_sync();                                                       // V(ch) is there
        if (mine) {
            // A probability of 0 does not keep a value out of a row that may not see it (0 * Inf and 0 * NaN are NaN): groups of
            // keys that not every row of the warp sees make the products of the rows that do.
            const int jj0 = max(0, w_lo - j0) & ~3, jj1 = min(kSimtChunk, w_hi - j0 + 1);
            const int in0 = min(max(all_lo - j0 + 3, jj0) & ~3, jj1), in1 = min(max((all_hi + 1 - j0) & ~3, in0), jj1);
            for (int jj = jj0; jj < in0; jj += 4) weigh(jj, j0, std::true_type());
            for (int jj = in0; jj < in1; jj += 4) weigh(jj, j0, std::false_type());
            for (int jj = in1; jj < jj1; jj += 4) weigh(jj, j0, std::true_type());
            __syncwarp();                                                  // sP is written again in the next chunk
        }
        part_sync();                                                       // V(ch) has been read
        if (ch_next < ch1) fetch(sV, Vb, p.vs.t, ch_next, c_hi, false); else fetch_commit();
    }
#pragma unroll
    for (int r = 0; r < R; ++r) l[r] = warp_sum(l[r]);
    fetch_wait_all();
    if (kSplit == 2) {      // the second half of the CTA hands its part of every row to the first
        float* const other = simt_smem + row0 * (kHeadDim + 4);
        __syncthreads();
        if (part == 1) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                *reinterpret_cast<float4*>(other + r * (kHeadDim + 4) + lane * 4) = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
                if (lane == 0) { other[r * (kHeadDim + 4) + kHeadDim] = m[r]; other[r * (kHeadDim + 4) + kHeadDim + 1] = l[r]; }
            }
        }
        __syncthreads();
        if (part == 1) return;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float* o = other + r * (kHeadDim + 4);
            const float4 a2 = *reinterpret_cast<const float4*>(o + lane * 4);
            const float m2 = o[kHeadDim], l2 = o[kHeadDim + 1], mm = fmaxf(m[r], m2), e1 = exp2f(m[r] - mm), e2 = exp2f(m2 - mm);
            l[r] = fmaf(l[r], e1, l2 * e2);
            acc[r][0] = fmaf(acc[r][0], e1, a2.x * e2); acc[r][1] = fmaf(acc[r][1], e1, a2.y * e2);
            acc[r][2] = fmaf(acc[r][2], e1, a2.z * e2); acc[r][3] = fmaf(acc[r][3], e1, a2.w * e2);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (row0 + r > last_row) break;
        const int t = __shfl_sync(0xffffffffu, t_l, row0 + r);
        const float inv = 1.f / l[r];
        store4(Ob + (long long)t * p.os.t + lane * 4, acc[r][0] * inv, acc[r][1] * inv, acc[r][2] * inv, acc[r][3] * inv);
    }
}

template <typename T, int kSplit>
static cudaError_t launch_simt_form(AttnParams ap, double kept, int batch, int device, cudaStream_t st) {
    using C = SimtCfg<kSplit>;
    static bool attr_set_dev[kDeviceFlagSlots] = {};      // function attributes are per device
    bool& attr_set = attr_set_dev[device >= 0 && device < kDeviceFlagSlots ? device : 0];
    if (!attr_set) {
        const cudaError_t e = cudaFuncSetAttribute(attention_simt_kernel<T, kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    ap.n_blocks = (ap.S + C::kRows - 1) / C::kRows;
    ap.blocks_est = std::min(std::max((int)ceil(kept / C::kRows), 1), ap.n_blocks);
    if ((long long)ap.n_blocks * ap.Hq > 0x7fffffffll) return cudaErrorInvalidValue;
    return launch_dependent(attention_simt_kernel<T, kSplit>, dim3((unsigned)ap.n_blocks * (unsigned)ap.Hq, 1, (unsigned)batch),
                            dim3(kSimtThreads), C::kSmemBytes, st, ap);
}

cudaError_t launch_attention_simt(tf_ctx* ctx, const tf_shape& s, const tf_filter_params& p,
                                  const void* Q, const void* K, const void* V,
                                  const int32_t* kept_idx, const int32_t* n_kept, void* O,
                                  bool after_selection, cudaStream_t st) {
    if (s.batch == 0 || s.seq == 0) return cudaSuccess;
    AttnParams ap{};
    ap.retained_only = (p.kv_visibility == TF_KV_RETAINED);
    ap.Q = Q; ap.K = K; ap.V = V; ap.O = O;
    ap.qs = {s.q_stride[0], s.q_stride[1], s.q_stride[2]};
    ap.ks = {s.k_stride[0], s.k_stride[1], s.k_stride[2]};
    ap.vs = {s.v_stride[0], s.v_stride[1], s.v_stride[2]};
    ap.os = {s.o_stride[0], s.o_stride[1], s.o_stride[2]};
    ap.S = s.seq; ap.Hq = s.n_q_heads; ap.Hkv = s.n_kv_heads; ap.window = s.window;
    const float scale = s.softmax_scale != 0.f ? s.softmax_scale : 1.f / sqrtf((float)s.head_dim);
    ap.scale_log2 = scale * 1.4426950408889634f;
    ap.kept_idx = kept_idx; ap.n_kept = n_kept;
    ap.early = after_selection && s.window == 0 && !ap.retained_only;
    // Up to two 16-row CTAs per SM the split form wins (us at 1 x 128 x 32 heads, 1 x 256 x 32, 2 x 256 x 32: 11 / 33 / 52
    // split, 16 / 44 / 45 unsplit), beyond that its second set of chunks costs more than it hides (1 x 768 x 40: 196 / 177).
    // The number of retained rows is only known on the device: the ratio gives the expected count.
    const double kept_frac = (p.select_mode == TF_SELECT_RATIO) ? 1.0 - p.prune_ratio : 1.0;
    const bool split = (double)s.batch * s.n_q_heads * ceil(s.seq * kept_frac / 16.0) <= 2.0 * sm_count();
    cudaError_t e;
    const double kept = ceil(s.seq * kept_frac);
    if (s.dtype == TF_BF16) e = split ? launch_simt_form<__nv_bfloat16, 2>(ap, kept, s.batch, ctx->device, st) : launch_simt_form<__nv_bfloat16, 1>(ap, kept, s.batch, ctx->device, st);
    else                    e = split ? launch_simt_form<float, 2>(ap, kept, s.batch, ctx->device, st) : launch_simt_form<float, 1>(ap, kept, s.batch, ctx->device, st);
    ctx->launches += 1;
    ctx->last_attention_kernel = TF_KERNEL_ATTN_SIMT;
    return e;
}

}  // namespace tf
