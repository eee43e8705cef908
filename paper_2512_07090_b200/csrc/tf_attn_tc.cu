// Step a5 on the 5th-generation tensor cores: bf16 causal (optionally windowed) attention for
// retained tokens only, head_dim 128.
//
// A work item is 256 consecutive entries of a sequence's retained list for one query head, as two
// 128-row Q tiles that share every K/V tile -- or, on grouped-query shapes, the same 128 or 64 entries for
// two or four query heads of one KV group (then both tiles need the same K/V tiles with the same masks).
// Warp roles:
//   warps 0-3 / 4-7  softmax group of Q tile 0 / 1 (thread r owns row r of its tile)
//   warp 8           issues every tcgen05.mma (the whole warp runs the loop, one elected lane issues)
//   warp 9           TMA producer: K and V tiles of 128 keys into a 4-slot ring (one lane)
//   warps 10-11      fetch the next work item and its Q rows, zero the output rows of pruned tokens
// The query rows are gathered (they are scattered in the sequence) into shared memory in the
// 128-byte-swizzled K-major operand layout.  Per K/V tile j and Q tile i:
//     S_i = Q_i K_j^T      A, B from shared memory (K-major)            -> TMEM, 128 columns
//     O_i += P_i V_j       A = P_i from TMEM (bf16, written over S_i),  B = V as it lies in
//                          memory (MN-major)                            -> TMEM, 128 columns
// issued in the order PV_0(j), QK_0(j+1), PV_1(j), QK_1(j+1): the tensor pipe works on one Q tile
// while the other tile's softmax group runs its exponentials.  The pipe executes in issue order,
// so S_i(j+1) is never produced before PV_i(j) has consumed P_i(j), and once a softmax group sees
// S_i(j) it may rescale O_i (PV_i(j-1) is complete).
// Softmax (fp32): row r applies ITS OWN causal / window limits (a tile of retained rows spans
// about 128/(1-ratio) positions), keeps a running reference maximum that is only moved (and O_i
// only rescaled) when the tile maximum exceeds it by more than 2^8, and writes P as bf16 pairs
// straight back into TMEM.  A Q tile skips K/V tiles none of its rows can see.  The epilogue
// normalises, converts to bf16 and scatters rows to their token positions; rows of pruned tokens
// are zeroed with the retained row that follows them (Section 3.2: a skipped token's attention
// output is zero).
//
// Every mbarrier wait is bounded by a cycle budget; on expiry the CTA records TF_ERR_TIMEOUT,
// stops waiting, lets copies in flight land, releases its TMEM and exits.
#include <algorithm>

#include "tf_ptx.cuh"

namespace tf {
namespace {

constexpr int kTileM = 128;           // rows per Q tile
constexpr int kQTiles = 2;            // Q tiles per CTA
constexpr int kTileN = 128;           // keys per K/V tile
constexpr int kHalfBytes = 128 * 128; // one [128 rows][128 B] swizzled block (64 bf16 per row)
constexpr int kTileBytes = 2 * kHalfBytes;
constexpr int kSoftmaxThreads = kQTiles * kTileM;
constexpr int kThreads = kSoftmaxThreads + 128;   // third warpgroup: MMA warp, TMA warp, two that fetch items and Q rows (split form: only zero rows)
constexpr int kMmaWarp = kSoftmaxThreads / 32, kTmaWarp = kMmaWarp + 1;
constexpr uint32_t kTmemCols = 512;   // S0 | S1 | O0 | O1, 128 fp32 columns each
constexpr float kRescaleThreshold = 8.f;         // log2 units

struct TcParams {
    const __nv_bfloat16* Q; __nv_bfloat16* O;
    Strides3 qs, os;
    int S, Hq, Hkv, window;
    float scale_log2;
    const int32_t* kept_idx; const int32_t* n_kept;
    DevStatus* status;
    int compact;          // 1: K / V hold the retained tokens only, entry c = token kept_idx[c] (TF_KV_RETAINED)
    int n_row_blocks;     // row blocks per (batch, query head)
    int n_blocks_est;     // ... that are expected to hold retained rows (a host-side estimate; any value in 1 .. n_row_blocks is right)
    int n_items;          // work items per (batch, query head): the expected row blocks, then as many others
    int bh_group;         // CTA order: (batch, head) pairs are taken in groups of this many; within a group all of the
                          // heaviest row block first.  1 = all row blocks of a head together, n_bh = heaviest first over all heads
    int first_pair;       // n_blocks_est - 1: the row block the first CTA of a head takes
    long long wait_cycles;   // budget of one mbarrier wait
};

// shared-memory map of the split form (dynamic, base aligned to 1024 B): one Q tile, a ring filled in the order K(j), V(j),
// K(j+1), V(j+1), ..., barriers
struct SplitCfg {
    static constexpr int kStages = 6;
    static constexpr int kOffQ = 0;
    static constexpr int kOffRing = kOffQ + kTileBytes;
    static constexpr int kOffBar = kOffRing + kStages * kTileBytes;
    static constexpr int kSmemBytes = kOffBar + 256 + 1024;   // barriers + alignment slack
};

// Work items are handed out in index order.  Row blocks of a head differ in length by the causal triangle, so the heaviest
// should go first, over as many heads as possible (the grid then ends with short items from many heads, which fill the SMs
// evenly); but the CTAs that run at the same time should find K and V in L2, which the row blocks of one head do (they
// read nearly the same keys) and those of different heads do not.  So the (batch, head) pairs are taken in groups whose
// K and V fit the L2 budget, and inside a group the order is: heaviest row block of every head, next row block, ...
__device__ __forceinline__ void work_item(const TcParams& p, unsigned int item, int n_blocks, int& rb, int& bh) {
    const int n_bh = (int)(gridDim.x / (unsigned)n_blocks);
    const int per_group = p.bh_group * n_blocks;
    const int g = (int)item / per_group, within = (int)item - g * per_group;
    const int g_size = min(p.bh_group, n_bh - g * p.bh_group);     // the last group may be smaller
    rb = within / g_size;
    bh = g * p.bh_group + within % g_size;
}

// The key that the first K/V tile of an item starts at, k_first being the first that any of its rows sees.  Under a window tiles
// start there, not at a multiple of their length: a window of 4096 and rows up to 128 positions apart then take 33 tiles instead of 33 or
// 34, one of them cut by the window's start instead of two (per pass: 8 x 16384 grouped 3917 -> 3862 us, 1 x 20000 x 32 heads 3 %
// with the masks).  Compacted keys are only defined up to a multiple of the tile.
__device__ __forceinline__ int first_tile_key(const TcParams& p, int k_first) {
    return p.window <= 0 ? 0 : p.compact ? k_first / kTileN * kTileN : k_first;
}

// bounded wait; after the first expiry in this CTA nobody waits any more
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, long long budget_cycles,
                                          DevStatus* status, unsigned long long where) {
    mbar_wait_bounded(bar, parity, abort_flag, budget_cycles, status, where);
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// the 3-input maximum
__device__ __forceinline__ float max3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// instruction descriptors: M=128, N=128; the P V product takes V as it lies in memory (MN-major)
constexpr uint32_t kIdescQK = idesc_bf16(128, false, false);
constexpr uint32_t kIdescPV = idesc_bf16(128, false, true);

// byte offset of 16-byte chunk cc (0..15) of row r inside a two-block [128][64]+[128][64] operand
__device__ __forceinline__ uint32_t swz(int r, int cc) {
    return (uint32_t)((cc >> 3) * kHalfBytes + r * 128 + (((cc & 7) ^ (r & 7)) << 4));
}


// One thread's share (a row of 128 scores) of one K/V tile of 128 keys starting at key j0: S from TMEM, masking by the
// row's own visible range lo .. hi, running reference maximum, exponentials, P as bf16 pairs back into TMEM over the first
// 64 columns of S, running sum.  O (when it exists already) is rescaled when the reference maximum moves.
__device__ __forceinline__ void softmax_tile(uint32_t tm_s, uint32_t tm_o, int lo, int hi, int j0, float scale_log2,
                                             bool have_o, float& m_ref, float& l_run) {
    uint32_t sreg[128];
#pragma unroll
    for (int c = 0; c < 4; ++c) tmem_ld32(tm_s + c * 32, sreg + c * 32);
    tmem_wait_ld();
    const bool full = (j0 >= lo) && (j0 + kTileN - 1 <= hi);
    if (!full) {   // columns below c_lo or above c_hi are invisible to this row: -inf
        // One bit per column, both bounds at once: a select on a bit of a word is one instruction beside the moves of bits to
        // predicates, and rows cut at either end take the same path (three variants with two compares a column before: 2048 tokens
        // 61.2 -> 60.1 us per pass, 4 x 4096 x 40 heads 521 -> 513, 2 x 8192 grouped 578 -> 573, 8 x 16384 windowed 3939 -> 3917)
        const int c_lo = lo - j0, c_hi = hi - j0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int up = min(max(c_hi - 32 * w + 1, 0), 32), dn = min(max(c_lo - 32 * w, 0), 32);
            const uint32_t vis = (uint32_t)((1ull << up) - 1ull) & ~(uint32_t)((1ull << dn) - 1ull);
#pragma unroll
            for (int e = 0; e < 32; ++e) sreg[32 * w + e] = (vis & (1u << e)) ? sreg[32 * w + e] : 0xff800000u;
        }
    }
    float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};   // four chains, not one of 128
#pragma unroll
    for (int c = 0; c < 128; c += 8) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
            mx4[u] = max3(mx4[u], __uint_as_float(sreg[c + 2 * u]), __uint_as_float(sreg[c + 2 * u + 1]));
    }
    const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
    __syncwarp();   // rows take different masking branches; the TMEM accesses below are warp-wide
    // move the reference maximum only when the tile maximum exceeds it by 2^8 or more
    const float m_tile = mx * scale_log2;
    const bool move = m_tile > m_ref + kRescaleThreshold;   // also true on the first visible key (m_ref = -inf)
    const float m_new = move ? m_tile : m_ref;
    const float corr = move ? ex2(m_ref - m_new) : 1.f;
    if (have_o && __any_sync(0xffffffffu, move)) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t o[32];
            tmem_ld32(tm_o + c * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * corr);
            tmem_st32(tm_o + c * 32, o);
        }
    }
    m_ref = m_new;
    const float m_safe = (m_ref == -INFINITY) ? 0.f : m_ref;
    const uint64_t sc2 = pack2(scale_log2, scale_log2), nm2 = pack2(-m_safe, -m_safe);
    uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t pk[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            float x0, x1;
            unpack2(fma2(pack2(__uint_as_float(sreg[h * 64 + 2 * c]), __uint_as_float(sreg[h * 64 + 2 * c + 1])), sc2, nm2), x0, x1);
            const float p0 = ex2(x0), p1 = ex2(x1);
            acc[c & 3] = add2(acc[c & 3], pack2(p0, p1));
            pk[c] = pack_bf16(p0, p1);
        }
        tmem_st32(tm_s + h * 32, pk);   // P_i over the first 64 columns of S_i
    }
    float a0, a1, a2, a3;
    unpack2(add2(acc[0], acc[1]), a0, a1);
    unpack2(add2(acc[2], acc[3]), a2, a3);
    const float psum = (a0 + a1) + (a2 + a3);
    l_run = fmaf(l_run, corr, psum);
}

// ---------------------------------------------------------------------------------------------------------
// Shared and head forms: persistent CTAs, one per SM, that take work items (row block, head) from the hardware's own
// launch queue (cluster launch control: a running CTA cancels the launch of a waiting one and does its work).
//   kHpt = 0: an item is 256 consecutive retained rows of one head, two Q tiles of 128.
//   kHpt = 1, 2 (grouped-query shapes): a Q tile holds the same 128 / kHpt retained rows of kHpt query heads of one KV
//     group (row r of the tile is head r / (128 / kHpt), entry r % (128 / kHpt)), the item's second tile the next kHpt
//     heads of that group: both tiles have the same K/V tiles and masks, no tile is ever worked on by one group alone.
// A CTA per item spends some 15,000 cycles around its tiles (3,300 each): launch, TMEM, three dependent global round
// trips, 64 KB of scattered Q rows, the first Q K^T and the last P V with nothing beside them, the epilogue.  Here the
// next item's set-up runs under the tiles of the current one:
//   warps 10-11 claim the next item when all but the last kClaimLead K/V tiles of this one have been requested (late enough
//     for the queue to hand items to the SMs that run out first), read its indices, gather its Q rows (cp.async) and publish a
//     descriptor; then they zero the output rows of pruned tokens.
//   warp 9 goes on with the next item's K/V tiles in the same ring, warp 8 with its products: Q K^T of the next item's
//     first tile is issued right behind the last P V of this one.
//   Q tiles take turns in three slots of shared memory.  Tile 0 of the next item goes into the third slot at any time,
//     tile 1 into the slot of this item's tile 0, which its last Q K^T gives back about one tile time before it is
//     needed (kHpt > 0) or group 0's epilogue does (kHpt = 0, where group 0 finishes first).
//   The epilogue stages its rows in the slot of tile 1 (kHpt > 0) or of the group's own tile (kHpt = 0).
// One layer's pass, one CTA per item -> persistent: 8 x 16384 windowed 4276 -> 3932 us, 2 x 8192 grouped heads 609 -> 568 us,
// 4 x 4096 x 40 heads 555 -> 506 us, 3 x 1531 87.7 -> 82.8 us, 2 x 3001 retained keys 139 -> 127 us; the last two with rows of
// pruned tokens zeroed by bulk copies 76 and 118 us.
// ---------------------------------------------------------------------------------------------------------
constexpr int kGatherWarp = kTmaWarp + 1;              // and the one after it
constexpr int kGatherThreads = 64;
constexpr int kPStages = 4;                            // K/V ring slots
constexpr int kPQSlots = 3;
constexpr int kPOffQ = 0, kPOffRing = kPQSlots * kTileBytes, kPOffRows = kPOffRing + kPStages * kTileBytes;
constexpr int kPOffMisc = kPOffRows + 2 * kSoftmaxThreads * 4;      // two sets of token positions of an item's rows
constexpr int kPOffZero = kPOffMisc + 512, kZeroBytes = 512;        // zeros: what rows of pruned tokens are filled with
constexpr int kPSmemBytes = kPOffZero + kZeroBytes;    // the dynamic segment must start 1024-byte aligned (checked)
static_assert(kPSmemBytes <= 227 * 1024, "shared memory of one CTA");

// the claim goes out when the K/V ring has taken all but this many of the item's tiles, four or five tile times before the
// item ends.  0, 1, 2, 3: 76.8, 77.1, 76.2, 76.1 us (3 x 1531), 92.6, 92.2, 92.1, 91.9 us (4096 tokens), the larger cases +-0.3 %
constexpr int kClaimLead = 2;

struct TcItem {
    int valid;            // 0: there is no further item
    int b, qh, slot0, nk;
    int k0;               // K/V tile j holds keys k0 + 128 j ..
    int jb[2], je[2];     // K/V tiles jb .. je - 1 of each Q tile
};

// 64 threads (warps 10-11) agree: true if any of them says so
__device__ __forceinline__ bool gather_any(bool x) {
    uint32_t r;
    asm volatile("{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbarrier.cta.red.or.pred q, 1, 64, p;\nselp.u32 %0, 1, 0, q;\n}"
                 : "=r"(r) : "r"((uint32_t)x) : "memory");
    return r != 0;
}

template <int kHpt>
__global__ void __launch_bounds__(kThreads, 1)
attention_tc_kernel(const TcParams p, const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV) {
    static_assert(kHpt == 0 || kHpt == 1 || kHpt == 2, "one, two or four query heads per CTA");
    constexpr bool kHeads = kHpt > 0;
    constexpr int kTileRows = kHeads ? kTileM / kHpt : kTileM;   // retained-list entries per Q tile
    constexpr int kRows = kHeads ? kTileRows : 2 * kTileM;       // ... per item
    constexpr int kHeadsPerCta = kHeads ? 2 * kHpt : 1;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = smem_u32(smem);
    if (sbase & 1023u) {   // the swizzled operand layout needs it; nothing has been started yet
        if (tid == 0) report_error(p.status, TF_ERR_CUDA, 398);
        return;
    }
    const uint32_t bars = sbase + kPOffMisc;
    const uint32_t bar_full = bars, bar_empty = bar_full + 8 * kPStages;   // [kPStages] ring slot filled / read by its products
    const uint32_t bar_s = bar_empty + 8 * kPStages;     // [2] S_i ready
    const uint32_t bar_p = bar_s + 16;                   // [2] P_i written (and O_i rescaled)
    const uint32_t bar_o = bar_p + 16;                   // [2] the item's last P_i V done
    // what is filled or given back ahead of its reader has one barrier per parity of the item, so that no phase can be missed
    const uint32_t bar_qf0 = bar_o + 16, bar_qf1 = bar_qf0 + 16;   // [2], [1] Q tile 0 / 1 gathered
    const uint32_t bar_q0 = bar_qf1 + 8;                 // Q slot of tile 0 given back
    const uint32_t bar_q1 = bar_q0 + 8;                  // [2] Q slot of tile 1, the item's rows and descriptor given back
    const uint32_t bar_item = bar_q1 + 16;               // [2] item descriptor written
    const uint32_t bar_claim = bar_item + 16;            // answer of the launch queue
    const uint32_t bar_asked = bar_claim + 8;            // [2] all but the last kClaimLead K/V tiles of the item requested
    const uint32_t claim = bars + 208;                   // 16 bytes
    TcItem* const items = reinterpret_cast<TcItem*>(smem + kPOffMisc + 224);          // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kPOffMisc + 320);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kPOffMisc + 328);
    int* const rows = reinterpret_cast<int*>(smem + kPOffRows);                       // [2][256] token position, -1: no row
    static_assert(sizeof(TcItem) <= 48 && (2 * kPStages + 17) * 8 <= 208, "layout of the last 512 bytes");
    if (tid == 0) {
        for (int i = 0; i < kPStages; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar_s + 8 * i, 1); mbar_init(bar_p + 8 * i, kTileM); mbar_init(bar_o + 8 * i, 1);
            mbar_init(bar_qf0 + 8 * i, kGatherThreads); mbar_init(bar_item + 8 * i, kGatherThreads); mbar_init(bar_asked + 8 * i, 1);
            mbar_init(bar_q1 + 8 * i, kSoftmaxThreads / 32);
        }
        mbar_init(bar_qf1, kGatherThreads);
        mbar_init(bar_q0, kHeads ? 1 : kTileM / 32);
        mbar_init(bar_claim, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (tid < kZeroBytes / 16) *reinterpret_cast<uint4*>(smem + kPOffZero + tid * 16) = make_uint4(0, 0, 0, 0);
    fence_proxy_async();
    __syncwarp();
    if (warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_dependency_wait();   // kept_idx / n_kept come from the kernel before this one
    auto q_slot = [&](int n, int i) { return sbase + kPOffQ + (uint32_t)((2 * n + i) % kPQSlots) * kTileBytes; };
    // waits for the descriptor of the CTA's item n; false (for the whole warp): there is none, or a wait has given up
    auto get_item = [&](int n, TcItem& it) {
        mbar_wait(bar_item + 8 * (n & 1), (n >> 1) & 1, abort_flag, p.wait_cycles, p.status, 12);
        if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
        it = items[n & 1];
        return it.valid != 0;
    };

    // registers move from the third warpgroup (which needs few) to the two softmax groups
    // (each setmaxnreg sits at the top of the branch it governs, so no later code sees both)
    if (warp >= kMmaWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp >= kGatherWarp) {
        // ================================ items, Q rows, zero rows ====================================
        const int w = warp - kGatherWarp, sub = lane >> 4, l16 = lane & 15;
        const bool dense_heads = p.os.h == kHeadDim;
        unsigned int item = blockIdx.x;
        int n = 0, claims = 0;
        for (;;) {
            int rb, bh;
            work_item(p, item, p.n_items, rb, bh);
            const int qh = (bh % (p.Hq / kHeadsPerCta)) * kHeadsPerCta, b = bh / (p.Hq / kHeadsPerCta);   // first (or only) head
            const int nk = p.n_kept[b];
            const int32_t* kept = p.kept_idx + (size_t)b * p.S;
            __nv_bfloat16* Ob = p.O + (long long)b * p.os.b + (long long)qh * p.os.h;
            // zeroes token t's output rows of n_heads (1 or 2) heads from head hh on: bulk copies, one instruction of one lane each
            auto zero_token = [&](int t, int hh, int n_heads) {
                __nv_bfloat16* dst = Ob + (long long)hh * p.os.h + (long long)t * p.os.t;
                bulk_store(dst, sbase + kPOffZero, dense_heads ? n_heads * kHeadDim * 2 : kHeadDim * 2);
                if (n_heads == 2 && !dense_heads) bulk_store(dst + p.os.h, sbase + kPOffZero, kHeadDim * 2);
            };
            const __nv_bfloat16* Qb = p.Q + (long long)b * p.qs.b + (long long)qh * p.qs.h + l16 * 8;
            bool produced = false;
            const int blk0 = p.n_blocks_est - 1 - rb + (rb < p.n_blocks_est ? 0 : p.n_items);   // heaviest expected row block first
            if (nk <= 0 && blk0 == 0) {                       // nothing retained at all: the whole head is zero
                for (int t = w * 32 + lane; t < p.S; t += kGatherThreads)
                    for (int hh = 0; hh < kHeadsPerCta; hh += 2) zero_token(t, hh, min(kHeadsPerCta, 2));
            }
            // row blocks beyond the items (normally empty) go to the same items
            for (int blk = blk0; blk < p.n_row_blocks && blk * kRows < nk; blk += p.n_items) {
                if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
                const int slot0 = blk * kRows;
                // this warp's half of each Q tile: rows 64 w .. 64 w + 63, two per lane
                int k0[2], k1[2];
                const int e0 = slot0 + ((w * 64) & (kTileRows - 1));
                k0[0] = e0 + lane < nk ? kept[e0 + lane] : -1;
                k0[1] = e0 + 32 + lane < nk ? kept[e0 + 32 + lane] : -1;
                if (kHeads) { k1[0] = k0[0]; k1[1] = k0[1]; }
                else {
                    k1[0] = e0 + kTileM + lane < nk ? kept[e0 + kTileM + lane] : -1;
                    k1[1] = e0 + kTileM + 32 + lane < nk ? kept[e0 + kTileM + 32 + lane] : -1;
                }
                TcItem d;
                d.valid = 1; d.b = b; d.qh = qh; d.slot0 = slot0; d.nk = nk; d.k0 = 0;
#pragma unroll
                for (int i = 0; i < 2; ++i) {     // which K/V tiles each Q tile needs
                    const int s_lo = slot0 + (kHeads ? 0 : i * kTileM);
                    d.jb[i] = d.je[i] = 0;
                    if (s_lo < nk) {
                        const int s_last = min(s_lo + kTileRows, nk) - 1;
                        const int t_first = kept[s_lo], t_last = kept[s_last];
                        int k_first = p.window > 0 ? max(0, t_first - p.window + 1) : 0;   // first key the tile's first row sees
                        int k_last = t_last;                                                // last key its last row sees
                        if (p.compact) {   // keys are entries of the retained list
                            k_first = p.window > 0 ? first_kept_at_or_after(kept, s_lo + 1, k_first) : 0;
                            k_last = s_last;
                        }
                        if (i == 0) d.k0 = first_tile_key(p, k_first);
                        d.jb[i] = (k_first - d.k0) / kTileN;
                        d.je[i] = (k_last - d.k0) / kTileN + 1;
                    }
                }
                // the slot of tile 0, the descriptor and the row positions are those of item n - 2
                if (n >= 2) mbar_wait(bar_q1 + 8 * (n & 1), ((n >> 1) - 1) & 1, abort_flag, p.wait_cycles, p.status, 13);
                __syncwarp();
                int* rw = rows + (n & 1) * kSoftmaxThreads + ((w * 64) & (kTileRows - 1));
                rw[lane] = k0[0];
                rw[32 + lane] = k0[1];
                if (!kHeads) { rw[kTileM + lane] = k1[0]; rw[kTileM + 32 + lane] = k1[1]; }
                if (tid == kGatherWarp * 32) items[n & 1] = d;
                mbar_arrive(bar_item + 8 * (n & 1));
                // 16 lanes copy a 256-byte row; rows that do not exist become zero
                auto gather = [&](int i, const int (&kk)[2]) {
                    const uint32_t dst = q_slot(n, i) + (uint32_t)((l16 >> 3) * kHalfBytes);
                    const __nv_bfloat16* src = Qb + (long long)(kHeads ? i * kHpt + (kHpt == 2 ? w : 0) : 0) * p.qs.h;
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll 8
                        for (int e = 0; e < 16; ++e) {
                            const int t = __shfl_sync(0xffffffffu, kk[h], 2 * e + sub), r = w * 64 + h * 32 + 2 * e + sub;
                            cp_async16(dst + (uint32_t)(r * 128 + (((l16 & 7) ^ (r & 7)) << 4)),
                                       src + (long long)max(t, 0) * p.qs.t, t >= 0 ? 16u : 0u);
                        }
                    asm volatile("cp.async.commit_group;" ::: "memory");
                };
                gather(0, k0);
                if (n == 0) {
                    gather(1, k1);
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                    fence_proxy_async();
                    mbar_arrive(bar_qf0);
                } else {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    fence_proxy_async();
                    mbar_arrive(bar_qf0 + 8 * (n & 1));
                    mbar_wait(bar_q0, (n - 1) & 1, abort_flag, p.wait_cycles, p.status, 14);
                    __syncwarp();
                    gather(1, k1);
                }
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                fence_proxy_async();
                mbar_arrive(bar_qf1);
                // rows of pruned tokens that precede a retained row of this warp (and follow the last one of all) are zero:
                // each lane fills the gaps before its own two entries.  (Sixteen lanes storing a row took 20,000 to 26,000
                // cycles per item, longer than a short item's tiles; this takes a tenth.)
                auto zero_rows = [&](const int (&kk)[2], int first, int hh, int n_heads) {
                    int before = (first > 0 && first < nk) ? kept[first - 1] : -1;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        int prev = __shfl_up_sync(0xffffffffu, kk[h], 1);
                        if (lane == 0) prev = before;
                        before = __shfl_sync(0xffffffffu, kk[h], 31);
                        for (int t = prev + 1; t < kk[h]; ++t) zero_token(t, hh, n_heads);     // (kk[h] = -1: no entry)
                        __syncwarp();
                        const int end = nk - 1 - (first + h * 32);                             // the lane that has the last entry of all
                        if (end >= 0 && end < 32)
                            for (int t = __shfl_sync(0xffffffffu, kk[h], end) + 1 + lane; t < p.S; t += 32) zero_token(t, hh, n_heads);
                        __syncwarp();
                    }
                };
                if (kHpt == 2) zero_rows(k0, e0, 2 * w, 2);
                else zero_rows(k0, e0, 0, kHeadsPerCta);
                if (!kHeads) zero_rows(k1, e0 + kTileM, 0, 1);
                bulk_commit();
                ++n;
                produced = true;
            }
            // the next item
            __syncwarp();
            if (produced) mbar_wait(bar_asked + 8 * ((n - 1) & 1), ((n - 1) >> 1) & 1, abort_flag, p.wait_cycles, p.status, 15);
            __syncwarp();
            fence_proxy_async();                               // the last answer has been read
            if (gather_any(*abort_flag != 0)) break;
            if (tid == kGatherWarp * 32) {
                mbar_expect_tx(bar_claim, 16);
                launch_queue_claim(claim, bar_claim);
            }
            __syncwarp();
            const bool answered = mbar_wait_bounded(bar_claim, claims & 1, abort_flag, p.wait_cycles, p.status, 16);
            ++claims;
            if (gather_any(!answered)) break;
            if (!launch_queue_item(claim, item) || item >= gridDim.x) {
                if (n >= 2) mbar_wait(bar_q1 + 8 * (n & 1), ((n >> 1) - 1) & 1, abort_flag, p.wait_cycles, p.status, 17);
                if (tid == kGatherWarp * 32) items[n & 1].valid = 0;
                mbar_arrive(bar_item + 8 * (n & 1));
                break;
            }
        }
        __syncwarp();
        bulk_commit();
        bulk_wait_all();       // the zeros have been read and written
    } else if (warp == kTmaWarp) {
        // ================================ TMA producer ================================================
        TcItem it;
        int q = 0;       // ring slots filled so far
        for (int n = 0; get_item(n, it); ++n) {
            if (lane == 0) {
                const int kh = it.qh / (p.Hq / p.Hkv), J1 = max(it.je[0], it.je[1]);
                for (int j = it.jb[0]; j < J1 && !*abort_flag; ++j) {      // rows ascend, so tile 0 starts first
                    for (int kv = 0; kv < 2; ++kv, ++q) {
                        const int st = q % kPStages;
                        // the CTA's first K and V tiles go out at once; the rest of the ring is filled once the Q rows of tile 0 are
                        // in shared memory (nothing can consume it earlier, and the copies would slow each other down)
                        if (n == 0 && q == 2) mbar_wait(bar_qf0, 0, abort_flag, p.wait_cycles, p.status, 11);
                        if (q >= kPStages) mbar_wait(bar_empty + 8 * st, ((q / kPStages) - 1) & 1, abort_flag, p.wait_cycles, p.status, 10);
                        const uint32_t dst = sbase + kPOffRing + st * kTileBytes;
                        const CUtensorMap* map = kv ? &mapV : &mapK;
                        mbar_expect_tx(bar_full + 8 * st, kTileBytes);
                        tma_load_4d(dst, map, bar_full + 8 * st, 0, kh, it.k0 + j * kTileN, it.b);
                        tma_load_4d(dst + kHalfBytes, map, bar_full + 8 * st, 64, kh, it.k0 + j * kTileN, it.b);
                    }
                    if (j == max(J1 - 1 - kClaimLead, it.jb[0])) mbar_arrive(bar_asked + 8 * (n & 1));
                }
            }
            __syncwarp();
        }
    } else {
        // ================================ MMA issuer ==================================================
        const uint32_t lead = elect_one();
        TcItem cur;
        int n = 0, q0 = 0;             // the CTA's item, ring slots used by the items before it
        int done[2] = {0, 0};          // tiles of each group so far
        auto ring = [&](int q) { return sbase + kPOffRing + (q % kPStages) * kTileBytes; };
        auto wait_full = [&](int q, int where) {
            mbar_wait(bar_full + 8 * (q % kPStages), (q / kPStages) & 1, abort_flag, p.wait_cycles, p.status, where);
        };
        auto release = [&](int q) { mma_commit(bar_empty + 8 * (q % kPStages), lead); };
        auto issue_qk = [&](int i, uint32_t qaddr, uint32_t kaddr) {   // S_i = Q_i K_j^T : 8 steps of 16 dims
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const uint32_t off = (kk >> 2) * kHalfBytes + (kk & 3) * 32;
                mma_ss(tmem + i * 128, desc_kmajor(qaddr + off), desc_kmajor(kaddr + off), kIdescQK, kk > 0, lead);
            }
            mma_commit(bar_s + 8 * i, lead);
        };
        auto issue_pv = [&](int i, uint32_t vaddr, bool first) {       // O_i (+)= P_i V_j : 8 steps of 16 keys
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
                mma_ts(tmem + 256 + i * 128, tmem + i * 128 + kk * 8, desc_mnmajor(vaddr + kk * 16 * 128, kHalfBytes), kIdescPV,
                       (!first || kk > 0) ? 1u : 0u, lead);
        };
        bool more = get_item(0, cur), ahead = false;      // ahead: Q_0 K^T of the item's first tile is issued already
        while (more) {
            const int J0 = cur.jb[0], J1 = max(cur.je[0], cur.je[1]);
            const uint32_t qa[2] = {q_slot(n, 0), q_slot(n, 1)};
            auto active = [&](int i, int j) { return j >= cur.jb[i] && j < cur.je[i]; };
            // the first tile's Q K^T
            if (!ahead) {
                wait_full(q0, 21);
                mbar_wait(bar_qf0 + 8 * (n & 1), (n >> 1) & 1, abort_flag, p.wait_cycles, p.status, 20);
                tc_fence_after();
                issue_qk(0, qa[0], ring(q0));
            }
            mbar_wait(bar_qf1, n & 1, abort_flag, p.wait_cycles, p.status, 19);
            tc_fence_after();
            if (active(1, J0)) issue_qk(1, qa[1], ring(q0));
            release(q0);
            if (kHeads && J1 == J0 + 1) mma_commit(bar_q0, lead);
            ahead = false;
            for (int j = J0; j < J1; ++j) {
                const int qv = q0 + 2 * (j - J0) + 1;
                const bool last = j + 1 == J1;
                wait_full(qv, 22);
                if (!last) wait_full(qv + 1, 23);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (active(i, j)) {
                        mbar_wait(bar_p + 8 * i, done[i] & 1, abort_flag, p.wait_cycles, p.status, 24 + i);
                        tc_fence_after();
                        issue_pv(i, ring(qv), j == cur.jb[i]);
                        ++done[i];
                        if (j + 1 == cur.je[i]) mma_commit(bar_o + 8 * i, lead);
                    }
                    if (i == 1) release(qv);
                    if (!last) {
                        if (active(i, j + 1)) issue_qk(i, qa[i], ring(qv + 1));
                    } else if (i == 0) {
                        // the next item's first Q_0 K^T, if everything it needs has arrived
                        bool ready = mbar_test(bar_item + 8 * ((n + 1) & 1), ((n + 1) >> 1) & 1);
                        if (__all_sync(0xffffffffu, ready)) {
                            ready = items[(n + 1) & 1].valid != 0 && mbar_test(bar_qf0 + 8 * ((n + 1) & 1), ((n + 1) >> 1) & 1) &&
                                    mbar_test(bar_full + 8 * ((qv + 1) % kPStages), ((qv + 1) / kPStages) & 1);
                            ahead = __all_sync(0xffffffffu, ready);
                            if (ahead) {
                                tc_fence_after();
                                issue_qk(0, q_slot(n + 1, 0), ring(qv + 1));
                            }
                        }
                    }
                }
                if (!last) {
                    release(qv + 1);
                    if (kHeads && j + 2 == J1) mma_commit(bar_q0, lead);      // this item's last Q K^T
                }
            }
            q0 += 2 * (J1 - J0);
            ++n;
            more = get_item(n, cur);
        }
    }
    } else {
        // ================================ softmax groups ===============================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const int i = warp >> 2;                 // group: its Q tile
        const int r = tid & (kTileM - 1);        // row within the tile
        const uint32_t tm_s = tmem + ((uint32_t)((warp & 3) * 32) << 16) + i * 128;   // this warp's lanes, S_i / P_i
        const uint32_t tm_o = tm_s + 256;                                               // O_i
        TcItem it;
        int tiles = 0, ends = 0;                 // of this group so far
        for (int n = 0; get_item(n, it); ++n) {
            const int32_t* kept = p.kept_idx + (size_t)it.b * p.S;
            const int e_row = (kHeads ? 0 : i * kTileM) + (r & (kTileRows - 1));
            const int slot = it.slot0 + e_row;
            const int t_row = rows[(n & 1) * kSoftmaxThreads + e_row];                // the row's token position, -1 if none
            const bool valid = t_row >= 0;
            int hi = t_row;                                                           // visible keys: lo .. hi
            int lo = (valid && p.window > 0) ? max(0, t_row - p.window + 1) : 0;
            if (p.compact && valid) {
                lo = p.window > 0 ? first_kept_at_or_after(kept, slot + 1, lo) : 0;
                hi = slot;
            }
            // From here on positions in the item's tiles.  A row that does not exist (its query is zero, its output goes nowhere) sees
            // everything, so that it does not send its warp through the masks in every tile (2,250 cycles instead of 1,750): it is in
            // the last row block, which starts first.  1 x 3000 grouped 73.5 -> 68.9 us per pass, 2 x 3001 retained 116.9 -> 114.6
            lo = valid ? lo - it.k0 : 0;
            hi = valid ? hi - it.k0 : 0x7fffffff;
            __syncwarp();
            const int jb = i == 0 ? it.jb[0] : it.jb[1], je = i == 0 ? it.je[0] : it.je[1];
            float m_ref = -INFINITY, l_run = 0.f;
            for (int j = jb; j < je; ++j, ++tiles) {
                mbar_wait(bar_s + 8 * i, tiles & 1, abort_flag, p.wait_cycles, p.status, 30 + i);
                __syncwarp();
                tc_fence_after();
                softmax_tile(tm_s, tm_o, lo, hi, j * kTileN, p.scale_log2, j > jb, m_ref, l_run);
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(bar_p + 8 * i);
            }
            // ---- epilogue: O / l -> bf16 -> the row's token position --------------------------------------
            // A thread owns a row, and rows of retained tokens lie far apart in O: storing from the registers would
            // touch 32 different lines per warp instruction.  Each warp therefore stages its 32 rows, 64 columns at a
            // time, in 4 KiB of a Q slot whose products are done (16-byte chunks XOR-swizzled by the row) and writes
            // them out with 8 lanes per 128 bytes.
            if (je > jb) {
                mbar_wait(bar_o + 8 * i, ends & 1, abort_flag, p.wait_cycles, p.status, 40);
                ++ends;
                __syncwarp();
                tc_fence_after();
                const float inv = 1.f / l_run;
                __nv_bfloat16* Ow = p.O + (long long)it.b * p.os.b +
                                    (long long)(it.qh + (kHeads ? i * kHpt + ((warp & 3) * 32) / kTileRows : 0)) * p.os.h;   // a warp's rows are of one head
                uint8_t* stage = smem + (q_slot(n, kHeads ? 1 : i) - sbase) + (kHeads ? warp : (warp & 3)) * 4096;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t o[64];
                    tmem_ld32(tm_o + c * 64, o);
                    tmem_ld32(tm_o + c * 64 + 32, o + 32);
                    tmem_wait_ld();
#pragma unroll
                    for (int v = 0; v < 8; ++v) {
                        uint4 x;
                        x.x = pack_bf16(__uint_as_float(o[8 * v + 0]) * inv, __uint_as_float(o[8 * v + 1]) * inv);
                        x.y = pack_bf16(__uint_as_float(o[8 * v + 2]) * inv, __uint_as_float(o[8 * v + 3]) * inv);
                        x.z = pack_bf16(__uint_as_float(o[8 * v + 4]) * inv, __uint_as_float(o[8 * v + 5]) * inv);
                        x.w = pack_bf16(__uint_as_float(o[8 * v + 6]) * inv, __uint_as_float(o[8 * v + 7]) * inv);
                        *reinterpret_cast<uint4*>(stage + lane * 128 + ((v ^ (lane & 7)) << 4)) = x;
                    }
                    __syncwarp();
#pragma unroll
                    for (int pass = 0; pass < 8; ++pass) {
                        const int R = pass * 4 + (lane >> 3), t_out = __shfl_sync(0xffffffffu, t_row, R);
                        const uint4 x = *reinterpret_cast<const uint4*>(stage + R * 128 + (((lane & 7) ^ (R & 7)) << 4));
                        if (t_out >= 0) *reinterpret_cast<uint4*>(Ow + (long long)t_out * p.os.t + c * 64 + (lane & 7) * 8) = x;
                    }
                    __syncwarp();
                }
                tc_fence_before();      // the next item's products write over O_i and S_i
            }
            // this warp is done with the item's slots, rows and descriptor
            if (lane == 0) {
                if (!kHeads && i == 0) mbar_arrive(bar_q0);
                mbar_arrive(bar_q1 + 8 * (n & 1));
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {   // a wait gave up: give copies and MMAs still in flight time to land before leaving
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) { }
        __syncthreads();
    }
    if (warp == kMmaWarp) tmem_dealloc(tmem, kTmemCols);
}

// Split form: ONE 128-row Q tile; the softmax groups take alternate K/V tiles and their partial results (O, maximum, sum)
// are merged at the end.  Twice as many, half as long CTAs: used when the shared form would leave SMs idle.
__global__ void __launch_bounds__(kThreads, 1)
attention_tc_split_kernel(const TcParams p, const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV) {
    constexpr int kRows = kTileM;         // retained-list entries one CTA covers
    constexpr int kStep = 2;              // K/V tile stride of one softmax group
    constexpr int kStages = SplitCfg::kStages, kOffQ = SplitCfg::kOffQ, kOffRing = SplitCfg::kOffRing, kOffBar = SplitCfg::kOffBar;
    extern __shared__ uint8_t smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar_q = sbase + kOffBar;              // Q tiles written
    const uint32_t bar_full = bar_q + 8;                 // [kStages] ring slot filled by TMA
    const uint32_t bar_empty = bar_full + 8 * kStages;   // [kStages] ring slot consumed by the MMAs
    const uint32_t bar_s = bar_empty + 8 * kStages;      // [2] S_i ready
    const uint32_t bar_p = bar_s + 16;                   // [2] P_i written (and O_i rescaled)
    const uint32_t bar_o = bar_p + 16;                   // all MMAs done
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBar + 160);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffBar + 168);
    // Barriers and TMEM need nothing from global memory: they are set up before the wait for the previous kernel,
    // which (the selection, one CTA per sequence) lets this grid become resident while it still runs.  Every way
    // out of the kernel from here on gives the TMEM columns back.
    if (tid == 0) {
        mbar_init(bar_q, kSoftmaxThreads);
        for (int i = 0; i < kStages; ++i) { mbar_init(bar_full + 8 * i, 1); mbar_init(bar_empty + 8 * i, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(bar_s + 8 * i, 1); mbar_init(bar_p + 8 * i, kTileM); }
        mbar_init(bar_o, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    __syncwarp();
    if (warp == kMmaWarp) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    grid_dependency_wait();   // kept_idx / n_kept come from the kernel before this one
    int rb, bh;
    work_item(p, blockIdx.x, p.n_row_blocks, rb, bh);
    // Row blocks are taken from the heaviest expected one (the last with retained rows, a host-side estimate) down to
    // block 0, then the blocks above the estimate, which are normally empty: CTAs with nothing to do start last
    // instead of delaying the first wave of real work.  Any estimate gives a one-to-one assignment.
    int pair = p.first_pair - rb;
    if (pair < 0) pair += p.n_row_blocks;
    const int qh = bh % p.Hq, b = bh / p.Hq;
    const int nk = p.n_kept[b];
    const int slot0 = pair * kRows;
    const int32_t* kept = p.kept_idx + (size_t)b * p.S;
    __nv_bfloat16* Ob = p.O + (long long)b * p.os.b + (long long)qh * p.os.h;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    if (slot0 >= max(nk, 1) || nk == 0) {   // no retained row in this block (CTA-uniform)
        if (slot0 < max(nk, 1)) {           // nothing retained at all: the whole head is zero
            for (int i = tid; i < p.S * 16; i += kThreads)
                *reinterpret_cast<uint4*>(Ob + (long long)(i >> 4) * p.os.t + (i & 15) * 8) = zero4;
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (warp == kMmaWarp) tmem_dealloc(*tmem_slot, kTmemCols);
        return;
    }

    // The softmax threads read the retained indices of the Q rows they will gather (16 lanes per 256-byte row, the
    // 8 warps take 16 rows per round) and of their own row now, next to the loads the set-up below waits for anyway:
    // one global round trip less between the set-up and the first Q K^T.
    constexpr int kRounds = kTileM / 16;   // 16 rows per round
    int tq[kRounds];
    int t_row = -1;
    if (warp < kMmaWarp) {
#pragma unroll
        for (int it = 0; it < kRounds; ++it) {
            const int s_q = slot0 + it * 16 + warp * 2 + (lane >> 4);
            tq[it] = s_q < nk ? kept[s_q] : -1;
        }
        const int slot_pre = slot0 + (tid & (kTileM - 1));
        if (slot_pre < nk) t_row = kept[slot_pre];
    }

    // ---- which K/V tiles the Q tile needs (CTA-uniform): group i works on tiles jb[i], jb[i] + 2, ... < J1 ------------
    const int s_last = min(slot0 + kTileM, nk) - 1;
    const int t_first = kept[slot0], t_last = kept[s_last];
    int k_first = p.window > 0 ? max(0, t_first - p.window + 1) : 0;   // first key the tile's first row sees
    int k_last = t_last;                                                // last key its last row sees
    if (p.compact) {   // keys are entries of the retained list
        k_first = p.window > 0 ? first_kept_at_or_after(kept, slot0 + 1, k_first) : 0;
        k_last = s_last;
    }
    const int k0 = first_tile_key(p, k_first);
    const int J0 = (k_first - k0) / kTileN, J1 = (k_last - k0) / kTileN + 1;
    const int jb[2] = {J0, J0 + 1};
    const int kh = qh / (p.Hq / p.Hkv);

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // registers move from the third warpgroup (which needs few) to the two softmax groups
    // (each setmaxnreg sits at the top of the branch it governs, so no later code sees both)
    if (warp >= kMmaWarp) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp > kTmaWarp) {
        // ================================ zero fill (the two spare warps) ================================
        // rows of pruned tokens that precede a retained row of this CTA (and follow the last retained
        // one) are zero; 16 lanes write one row
        const int g4 = (tid - (kTmaWarp + 1) * 32) >> 4, l16 = tid & 15;
        const int s_end = min(slot0 + kRows, nk);
        for (int s_z = slot0 + g4; s_z < s_end; s_z += 4) {
            const int prev = s_z == 0 ? -1 : kept[s_z - 1], cur = kept[s_z];
            for (int t = prev + 1; t < cur; ++t) *reinterpret_cast<uint4*>(Ob + (long long)t * p.os.t + l16 * 8) = zero4;
            if (s_z == nk - 1)
                for (int t = cur + 1; t < p.S; ++t) *reinterpret_cast<uint4*>(Ob + (long long)t * p.os.t + l16 * 8) = zero4;
        }
    } else if (warp == kTmaWarp) {
        // ================================ TMA producer ================================================
        if (lane == 0) {
            int q = 0;
            for (int j = J0; j < J1; ++j) {
                for (int kv = 0; kv < 2; ++kv, ++q) {
                    const int st = q % kStages;
                    // the first K and V tiles go out at once; the rest of the ring is filled once the Q rows are in shared
                    // memory (nothing can consume it earlier, and a ring's worth of arriving tiles keeps the gather's
                    // shared-memory stores waiting)
                    if (q == 2) mbar_wait(bar_q, 0, abort_flag, p.wait_cycles, p.status, 11);
                    if (q >= kStages) mbar_wait(bar_empty + 8 * st, ((q / kStages) - 1) & 1, abort_flag, p.wait_cycles, p.status, 10);
                    const uint32_t dst = sbase + kOffRing + st * kTileBytes;
                    const CUtensorMap* map = kv ? &mapV : &mapK;
                    mbar_expect_tx(bar_full + 8 * st, kTileBytes);
                    tma_load_4d(dst, map, bar_full + 8 * st, 0, kh, k0 + j * kTileN, b);
                    tma_load_4d(dst + kHalfBytes, map, bar_full + 8 * st, 64, kh, k0 + j * kTileN, b);
                }
            }
        }
    } else if (warp == kMmaWarp) {
        // ================================ MMA issuer ==================================================
        {
            const uint32_t lead = elect_one();
            auto slot_of = [&](int j, int kv) { return (2 * (j - J0) + kv) % kStages; };
            auto par_of = [&](int j, int kv) { return ((2 * (j - J0) + kv) / kStages) & 1; };
            auto issue_qk = [&](int i, int j) {   // S_i = Q_i K_j^T : 8 steps of 16 dims
                const uint32_t kaddr = sbase + kOffRing + slot_of(j, 0) * kTileBytes;
                const uint32_t qaddr = sbase + kOffQ;   // both groups share the Q tile
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const uint32_t off = (kk >> 2) * kHalfBytes + (kk & 3) * 32;
                    mma_ss(tmem + i * 128, desc_kmajor(qaddr + off), desc_kmajor(kaddr + off), kIdescQK, kk > 0, lead);
                }
                mma_commit(bar_s + 8 * i, lead);
            };
            auto issue_pv = [&](int i, int j, bool first) {   // O_i (+)= P_i V_j : 8 steps of 16 keys
                const uint32_t vaddr = sbase + kOffRing + slot_of(j, 1) * kTileBytes;
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                    mma_ts(tmem + 256 + i * 128, tmem + i * 128 + kk * 8, desc_mnmajor(vaddr + kk * 16 * 128, kHalfBytes), kIdescPV,
                           (!first || kk > 0) ? 1u : 0u, lead);
            };
            mbar_wait(bar_q, 0, abort_flag, p.wait_cycles, p.status, 20);
            int done[kQTiles] = {0, 0};
            {
                // tile j belongs to group (j - J0) & 1; order: QK_0(J0), QK_1(J0+1), then per tile PV(j), QK(j+2)
                for (int j = J0; j < min(J0 + 2, J1); ++j) {
                    mbar_wait(bar_full + 8 * slot_of(j, 0), par_of(j, 0), abort_flag, p.wait_cycles, p.status, 21);
                    tc_fence_after();
                    issue_qk(j - J0, j);
                    mma_commit(bar_empty + 8 * slot_of(j, 0), lead);
                }
                for (int j = J0; j < J1; ++j) {
                    const int i = (j - J0) & 1;
                    mbar_wait(bar_full + 8 * slot_of(j, 1), par_of(j, 1), abort_flag, p.wait_cycles, p.status, 22);
                    mbar_wait(bar_p + 8 * i, done[i] & 1, abort_flag, p.wait_cycles, p.status, 24 + i);
                    tc_fence_after();
                    issue_pv(i, j, done[i] == 0);
                    ++done[i];
                    mma_commit(bar_empty + 8 * slot_of(j, 1), lead);
                    if (j + 2 < J1) {
                        mbar_wait(bar_full + 8 * slot_of(j + 2, 0), par_of(j + 2, 0), abort_flag, p.wait_cycles, p.status, 23);
                        issue_qk(i, j + 2);
                        mma_commit(bar_empty + 8 * slot_of(j + 2, 0), lead);
                    }
                }
            }
            mma_commit(bar_o, lead);
        }
    }
    } else {
        // ================================ softmax groups ===============================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const int i = warp >> 2;                 // group: its half of the K/V tiles
        const int r = tid & (kTileM - 1);        // row within the tile
        const int slot = slot0 + r;
        const bool valid = slot < nk;               // t_row (fetched above) is the row's token position, -1 if none
        int hi = t_row;                                                           // visible keys: lo .. hi
        int lo = (valid && p.window > 0) ? max(0, t_row - p.window + 1) : 0;
        if (p.compact && valid) {
            lo = p.window > 0 ? first_kept_at_or_after(kept, slot + 1, lo) : 0;
            hi = slot;
        }
        lo = valid ? lo - k0 : 0;                   // (a row that does not exist sees everything: no masks on its account)
        hi = valid ? hi - k0 : 0x7fffffff;
        {
            // gather the Q rows into the swizzled K-major operand layout
            const int sub = lane >> 4, cc = lane & 15, w8 = tid >> 5;
            uint4 qv[kRounds];
            const __nv_bfloat16* qbase = p.Q + (long long)b * p.qs.b + (long long)qh * p.qs.h + cc * 8;
#pragma unroll
            for (int it = 0; it < kRounds; ++it) qv[it] = tq[it] >= 0 ? ldg16(qbase + (long long)tq[it] * p.qs.t) : zero4;
#pragma unroll
            for (int it = 0; it < kRounds; ++it)
                *reinterpret_cast<uint4*>(smem + kOffQ + swz(it * 16 + w8 * 2 + sub, cc)) = qv[it];
            fence_proxy_async();
            mbar_arrive(bar_q);
        }
        __syncwarp();
        const uint32_t tm_s = tmem + ((uint32_t)((warp & 3) * 32) << 16) + i * 128;   // this warp's lanes, S_i / P_i
        const uint32_t tm_o = tm_s + 256;                                               // O_i
        float m_ref = -INFINITY, l_run = 0.f;
        for (int j = jb[i]; j < J1; j += kStep) {
            const int c_it = (j - jb[i]) / kStep;
            const int j0 = j * kTileN;
            mbar_wait(bar_s + 8 * i, c_it & 1, abort_flag, p.wait_cycles, p.status, 30 + i);
            __syncwarp();
            tc_fence_after();
            softmax_tile(tm_s, tm_o, lo, hi, j0, p.scale_log2, c_it > 0, m_ref, l_run);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar_p + 8 * i);
        }
        // ---- epilogue: O / l -> bf16 -> the row's token position --------------------------------------
        // A thread owns a row, and rows of retained tokens lie far apart in O: storing from the registers would
        // touch 32 different lines per warp instruction.  The rows are therefore staged in the shared memory of the
        // Q tile (nobody reads it once every MMA has completed; 16-byte chunks XOR-swizzled by the row) and written
        // out with 16 lanes per 256-byte row.  (maximum, sum) of the split form and the rows' token positions
        // travel through the first K/V ring slot, equally idle by now.
        {
            // merge the two groups' partial results: both accumulators sit in the TMEM lanes of this row,
            // so each group finishes 64 of the 128 output columns
            mbar_wait(bar_o, 0, abort_flag, p.wait_cycles, p.status, 40);
            __syncwarp();
            tc_fence_after();
            float2* ml = reinterpret_cast<float2*>(smem + kOffRing);
            int* trow_s = reinterpret_cast<int*>(smem + kOffRing + 4096);
            ml[i * kTileM + r] = make_float2(m_ref, l_run);
            if (i == 0) trow_s[r] = t_row;                        // -1: no such row
            asm volatile("bar.sync 1, %0;" :: "n"(kSoftmaxThreads) : "memory");
            const float2 other = ml[(i ^ 1) * kTileM + r];
            const bool both = J1 > jb[1];                       // group 1 had tiles (CTA-uniform)
            const float m0 = i == 0 ? m_ref : other.x, l0 = i == 0 ? l_run : other.y;   // group 0 always has a tile
            const float m1 = i == 0 ? other.x : m_ref, l1 = i == 0 ? other.y : l_run;
            const float m_all = both ? fmaxf(m0, m1) : m0;
            const float e0 = ex2(m0 - m_all), e1 = both ? ex2(m1 - m_all) : 0.f;
            const float inv = 1.f / (l0 * e0 + l1 * e1);
            const float w0 = e0 * inv, w1 = e1 * inv;
            const uint32_t tm_row = tmem + ((uint32_t)((warp & 3) * 32) << 16);
            uint8_t* stage = smem + kOffQ + r * 256;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t o0[32], o1[32];
                tmem_ld32(tm_row + 256 + i * 64 + c * 32, o0);
                if (both) tmem_ld32(tm_row + 384 + i * 64 + c * 32, o1);
                tmem_wait_ld();
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    float f[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        f[e] = __uint_as_float(o0[8 * v + e]) * w0;
                        if (both) f[e] = fmaf(__uint_as_float(o1[8 * v + e]), w1, f[e]);
                    }
                    uint4 w;
                    w.x = pack_bf16(f[0], f[1]); w.y = pack_bf16(f[2], f[3]);
                    w.z = pack_bf16(f[4], f[5]); w.w = pack_bf16(f[6], f[7]);
                    *reinterpret_cast<uint4*>(stage + (((i * 8 + c * 4 + v) ^ (r & 15)) << 4)) = w;
                }
            }
            asm volatile("bar.sync 1, %0;" :: "n"(kSoftmaxThreads) : "memory");
            const int sub = tid >> 4, l16 = tid & 15;              // 256 threads: 16 rows per pass
#pragma unroll
            for (int pass = 0; pass < kTileM / 16; ++pass) {
                const int R = pass * 16 + sub, t_out = trow_s[R];
                if (t_out >= 0)
                    *reinterpret_cast<uint4*>(Ob + (long long)t_out * p.os.t + l16 * 8) =
                        *reinterpret_cast<const uint4*>(smem + kOffQ + R * 256 + ((l16 ^ (R & 15)) << 4));
            }
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {   // a wait gave up: give copies and MMAs still in flight time to land before leaving
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) { }
        __syncthreads();
    }
    if (warp == kMmaWarp) tmem_dealloc(tmem, kTmemCols);
}

// ---------------------------------------------------------------------------------------------------------
// Single form: ONE 128-row Q tile and ONE softmax group per CTA -- 256 threads, 256 TMEM columns (S | O) and 96 KiB
// of shared memory (the Q tile, one K slot, one V slot), so that TWO CTAs share an SM.  What the two softmax groups
// of the other forms do for each other inside a CTA (one exponentiates while the tensor pipe works for the other),
// two independent CTAs do here, and in addition the set-up, Q gather and epilogue of one CTA run under the steady
// state of its neighbour: the fixed cost per CTA, a third of all SM time on small problems, is no longer idle time.
// Every Q tile streams its own K/V tiles (as in the split form), so this form suits problems whose K/V traffic the
// L2 can feed twice over.  Warp roles: warps 0-3 softmax (thread r owns row r), warp 4 issues the products, warp 5
// the TMA loads, warps 6-7 zero the output rows of pruned tokens.
//   K(j+1) is requested as soon as Q K_j^T has read K(j), V(j+1) as soon as P V_j has read V(j): with one slot each
//   the loads run under the softmax of tile j and the products of the neighbouring CTA.
// ---------------------------------------------------------------------------------------------------------
constexpr int kThreads1 = 256;
constexpr int kMmaWarp1 = 4, kTmaWarp1 = 5;
constexpr uint32_t kTmemCols1 = 256;
constexpr int kOffQ1 = 0, kOffK1 = kTileBytes, kOffV1 = 2 * kTileBytes, kOffBar1 = 3 * kTileBytes;
constexpr int kSmemBytes1 = kOffBar1 + 256;      // the dynamic segment must start 1024-byte aligned (checked)
constexpr int kRegs1 = 128;                      // registers per thread at launch: 256 x 128 = 128 x 200 + 128 x 56

__global__ void __launch_bounds__(kThreads1, 2)
attention_tc_single_kernel(const TcParams p, const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapV) {
    extern __shared__ __align__(1024) uint8_t smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = smem_u32(smem);
    if (sbase & 1023u) {   // the swizzled operand layout needs it; nothing has been started yet
        if (tid == 0) report_error(p.status, TF_ERR_CUDA, 399);
        return;
    }
    const uint32_t bar_q = sbase + kOffBar1;              // Q tile written
    const uint32_t bar_fk = bar_q + 8, bar_fv = bar_q + 16;   // K / V slot filled by TMA
    const uint32_t bar_ek = bar_q + 24, bar_ev = bar_q + 32;  // K / V slot consumed by the products
    const uint32_t bar_s = bar_q + 40, bar_p = bar_q + 48, bar_o = bar_q + 56;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBar1 + 64);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffBar1 + 72);
    if (tid == 0) {
        mbar_init(bar_q, kTileM);
        mbar_init(bar_fk, 1); mbar_init(bar_fv, 1); mbar_init(bar_ek, 1); mbar_init(bar_ev, 1);
        mbar_init(bar_s, 1); mbar_init(bar_p, kTileM); mbar_init(bar_o, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    __syncwarp();
    if (warp == kMmaWarp1) tmem_alloc(smem_u32(tmem_slot), kTmemCols1);
    grid_dependency_wait();   // kept_idx / n_kept come from the kernel before this one
    int rb, bh;
    work_item(p, blockIdx.x, p.n_row_blocks, rb, bh);
    int blk = p.first_pair - rb;          // heaviest expected row block first, blocks expected to be empty last
    if (blk < 0) blk += p.n_row_blocks;
    const int qh = bh % p.Hq, b = bh / p.Hq;
    const int nk = p.n_kept[b];
    const int slot0 = blk * kTileM;
    const int32_t* kept = p.kept_idx + (size_t)b * p.S;
    __nv_bfloat16* Ob = p.O + (long long)b * p.os.b + (long long)qh * p.os.h;
    const uint4 zero4 = make_uint4(0, 0, 0, 0);
    if (slot0 >= max(nk, 1) || nk == 0) {   // no retained row in this block (CTA-uniform)
        if (slot0 < max(nk, 1)) {           // nothing retained at all: the whole head is zero
            for (int i = tid; i < p.S * 16; i += kThreads1)
                *reinterpret_cast<uint4*>(Ob + (long long)(i >> 4) * p.os.t + (i & 15) * 8) = zero4;
        }
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        if (warp == kMmaWarp1) tmem_dealloc(*tmem_slot, kTmemCols1);
        return;
    }
    // retained indices of the Q rows this thread gathers (16 lanes per 256-byte row, the 4 softmax warps take 8 rows per
    // round) and of its own row
    constexpr int kRounds = kTileM / 8;
    int tq[kRounds];
    int t_row = -1;
    if (warp < kMmaWarp1) {
#pragma unroll
        for (int it = 0; it < kRounds; ++it) {
            const int s_q = slot0 + it * 8 + warp * 2 + (lane >> 4);
            tq[it] = s_q < nk ? kept[s_q] : -1;
        }
        if (slot0 + tid < nk) t_row = kept[slot0 + tid];
    }
    // which K/V tiles the Q tile needs (CTA-uniform): J0 .. J1 - 1
    int J0, J1;
    {
        const int s_last = min(slot0 + kTileM, nk) - 1;
        const int t_first = kept[slot0], t_last = kept[s_last];
        int k_first = p.window > 0 ? max(0, t_first - p.window + 1) : 0;
        int k_last = t_last;
        if (p.compact) {   // keys are entries of the retained list
            k_first = p.window > 0 ? first_kept_at_or_after(kept, slot0 + 1, k_first) : 0;
            k_last = s_last;
        }
        J0 = k_first / kTileN;
        J1 = k_last / kTileN + 1;
    }
    const int kh = qh / (p.Hq / p.Hkv);

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp >= kMmaWarp1) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
        if (warp > kTmaWarp1) {
            // ================================ zero fill ====================================================
            const int g4 = (tid - (kTmaWarp1 + 1) * 32) >> 4, l16 = tid & 15;
            const int s_end = min(slot0 + kTileM, nk);
            for (int s_z = slot0 + g4; s_z < s_end; s_z += 4) {
                const int prev = s_z == 0 ? -1 : kept[s_z - 1], cur = kept[s_z];
                for (int t = prev + 1; t < cur; ++t) *reinterpret_cast<uint4*>(Ob + (long long)t * p.os.t + l16 * 8) = zero4;
                if (s_z == nk - 1)
                    for (int t = cur + 1; t < p.S; ++t) *reinterpret_cast<uint4*>(Ob + (long long)t * p.os.t + l16 * 8) = zero4;
            }
        } else if (warp == kTmaWarp1) {
            // ================================ TMA producer ================================================
            if (lane == 0) {
                for (int j = J0; j < J1; ++j) {
                    const int n = j - J0;
                    if (n > 0) mbar_wait(bar_ek, (n - 1) & 1, abort_flag, p.wait_cycles, p.status, 10);
                    mbar_expect_tx(bar_fk, kTileBytes);
                    tma_load_4d(sbase + kOffK1, &mapK, bar_fk, 0, kh, j * kTileN, b);
                    tma_load_4d(sbase + kOffK1 + kHalfBytes, &mapK, bar_fk, 64, kh, j * kTileN, b);
                    if (n > 0) mbar_wait(bar_ev, (n - 1) & 1, abort_flag, p.wait_cycles, p.status, 11);
                    mbar_expect_tx(bar_fv, kTileBytes);
                    tma_load_4d(sbase + kOffV1, &mapV, bar_fv, 0, kh, j * kTileN, b);
                    tma_load_4d(sbase + kOffV1 + kHalfBytes, &mapV, bar_fv, 64, kh, j * kTileN, b);
                }
            }
        } else {
            // ================================ MMA issuer ==================================================
            {
                const uint32_t lead = elect_one();
                auto issue_qk = [&]() {           // S = Q K_j^T : 8 steps of 16 dims
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        const uint32_t off = (kk >> 2) * kHalfBytes + (kk & 3) * 32;
                        mma_ss(tmem, desc_kmajor(sbase + kOffQ1 + off), desc_kmajor(sbase + kOffK1 + off), kIdescQK, kk > 0, lead);
                    }
                    mma_commit(bar_s, lead);
                    mma_commit(bar_ek, lead);
                };
                mbar_wait(bar_q, 0, abort_flag, p.wait_cycles, p.status, 20);
                mbar_wait(bar_fk, 0, abort_flag, p.wait_cycles, p.status, 21);
                tc_fence_after();
                issue_qk();
                for (int j = J0; j < J1; ++j) {
                    const int n = j - J0;
                    mbar_wait(bar_fv, n & 1, abort_flag, p.wait_cycles, p.status, 22);
                    mbar_wait(bar_p, n & 1, abort_flag, p.wait_cycles, p.status, 24);
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk)    // O (+)= P V_j : 8 steps of 16 keys
                        mma_ts(tmem + 128, tmem + kk * 8, desc_mnmajor(sbase + kOffV1 + kk * 16 * 128, kHalfBytes), kIdescPV,
                               (n > 0 || kk > 0) ? 1u : 0u, lead);
                    mma_commit(bar_ev, lead);
                    if (j + 1 < J1) {
                        mbar_wait(bar_fk, (n + 1) & 1, abort_flag, p.wait_cycles, p.status, 23);
                        tc_fence_after();
                        issue_qk();
                    }
                }
                mma_commit(bar_o, lead);
            }
        }
    } else {
        // ================================ softmax group ================================================
        asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
        const int r = tid;                        // row within the tile
        const int slot = slot0 + r;
        const bool valid = slot < nk;
        int hi = t_row;                                                           // visible keys: lo .. hi
        int lo = (valid && p.window > 0) ? max(0, t_row - p.window + 1) : 0;
        if (p.compact && valid) {
            lo = p.window > 0 ? first_kept_at_or_after(kept, slot + 1, lo) : 0;
            hi = slot;
        }
        {   // gather the Q rows into the swizzled K-major operand layout
            const int sub = lane >> 4, cc = lane & 15;
            uint4 qv[kRounds];
            const __nv_bfloat16* qbase = p.Q + (long long)b * p.qs.b + (long long)qh * p.qs.h + cc * 8;
#pragma unroll
            for (int it = 0; it < kRounds; ++it) qv[it] = tq[it] >= 0 ? ldg16(qbase + (long long)tq[it] * p.qs.t) : zero4;
#pragma unroll
            for (int it = 0; it < kRounds; ++it)
                *reinterpret_cast<uint4*>(smem + kOffQ1 + swz(it * 8 + warp * 2 + sub, cc)) = qv[it];
            fence_proxy_async();
            mbar_arrive(bar_q);
        }
        __syncwarp();
        const uint32_t tm_s = tmem + ((uint32_t)(warp * 32) << 16);   // this warp's lanes: S / P
        const uint32_t tm_o = tm_s + 128;                             // O
        float m_ref = -INFINITY, l_run = 0.f;
        for (int j = J0; j < J1; ++j) {
            const int n = j - J0;
            mbar_wait(bar_s, n & 1, abort_flag, p.wait_cycles, p.status, 30);
            __syncwarp();
            tc_fence_after();
            softmax_tile(tm_s, tm_o, lo, hi, j * kTileN, p.scale_log2, n > 0, m_ref, l_run);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(bar_p);
        }
        // ---- epilogue: O / l -> bf16 -> staged in the Q tile's shared memory -> the rows' token positions ----------
        mbar_wait(bar_o, 0, abort_flag, p.wait_cycles, p.status, 40);
        __syncwarp();
        tc_fence_after();
        const float inv = 1.f / l_run;
        int* trow_s = reinterpret_cast<int*>(smem + kOffK1);          // the K slot is idle by now
        trow_s[r] = t_row;
        uint8_t* stage = smem + kOffQ1 + r * 256;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t o[32];
            tmem_ld32(tm_o + c * 32, o);
            tmem_wait_ld();
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                uint4 w;
                w.x = pack_bf16(__uint_as_float(o[8 * v + 0]) * inv, __uint_as_float(o[8 * v + 1]) * inv);
                w.y = pack_bf16(__uint_as_float(o[8 * v + 2]) * inv, __uint_as_float(o[8 * v + 3]) * inv);
                w.z = pack_bf16(__uint_as_float(o[8 * v + 4]) * inv, __uint_as_float(o[8 * v + 5]) * inv);
                w.w = pack_bf16(__uint_as_float(o[8 * v + 6]) * inv, __uint_as_float(o[8 * v + 7]) * inv);
                *reinterpret_cast<uint4*>(stage + (((c * 4 + v) ^ (r & 15)) << 4)) = w;
            }
        }
        asm volatile("bar.sync 1, %0;" :: "n"(kTileM) : "memory");      // the 128 softmax threads
        const int sub = r >> 4, l16 = r & 15;                           // 8 rows per pass
#pragma unroll
        for (int pass = 0; pass < kTileM / 8; ++pass) {
            const int R = pass * 8 + sub, t_out = trow_s[R];
            if (t_out >= 0)
                *reinterpret_cast<uint4*>(Ob + (long long)t_out * p.os.t + l16 * 8) =
                    *reinterpret_cast<const uint4*>(smem + kOffQ1 + R * 256 + ((l16 ^ (R & 15)) << 4));
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {   // a wait gave up: give copies and products still in flight time to land before leaving
        const long long t0 = clock64();
        while (clock64() - t0 < 2000000ll) { }
        __syncthreads();
    }
    if (warp == kMmaWarp1) tmem_dealloc(tmem, kTmemCols1);
}

// ---- host side: tensor maps over the caller's K / V (two 64-column boxes of kTileN keys per tile) ---------
bool make_kv_map(CUtensorMap* map, const void* base, const int64_t st[3], int B, int S, int H) {
    return make_bshd_map(map, base, st, B, S, H, 2, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 64, kTileN, CU_TENSOR_MAP_SWIZZLE_128B);
}

// TF_KV_RETAINED: copy the retained tokens' K and V rows (all KV heads) to dense [B,S,Hkv,128] buffers,
// entry c of a sequence = token kept_idx[c]; entries from n_kept up to the next multiple of the key tile
// are zeroed (they are masked, but a tile may not contain NaN bit patterns: 0 * NaN would reach O).
__global__ void __launch_bounds__(256) compact_kv_kernel(const __nv_bfloat16* __restrict__ K, const __nv_bfloat16* __restrict__ V,
                                                         Strides3 ks, Strides3 vs, int S, int Hkv,
                                                         const int32_t* __restrict__ kept_idx, const int32_t* __restrict__ n_kept,
                                                         __nv_bfloat16* __restrict__ Kc, __nv_bfloat16* __restrict__ Vc) {
    grid_dependency_wait();
    grid_launch_dependents();      // the attention's CTAs set themselves up as these drain
    const int b = blockIdx.y, nk = n_kept[b];
    const int c_end = min(S, (nk + kTileN - 1) / kTileN * kTileN);
    const int chunks = Hkv * 16;                               // 16-byte chunks per row of one tensor
    const int32_t* kept = kept_idx + (size_t)b * S;
    for (int c = blockIdx.x * 8 + (threadIdx.x >> 5); c < c_end; c += gridDim.x * 8) {
        const bool live = c < nk;
        const long long t = live ? kept[c] : 0;
        for (int q = threadIdx.x & 31; q < chunks; q += 32) {
            const int h = q >> 4, off = (q & 15) * 8;
            uint4 kv = make_uint4(0, 0, 0, 0), vv = kv;
            if (live) {
                kv = ldg16(K + (long long)b * ks.b + t * ks.t + (long long)h * ks.h + off);
                vv = ldg16(V + (long long)b * vs.b + t * vs.t + (long long)h * vs.h + off);
            }
            const size_t dst = (((size_t)b * S + c) * Hkv + h) * kHeadDim + off;
            *reinterpret_cast<uint4*>(Kc + dst) = kv;
            *reinterpret_cast<uint4*>(Vc + dst) = vv;
        }
    }
}

}  // namespace

size_t kv_compact_bytes(const tf_shape& s) {
    return 2 * ((size_t)s.batch * s.seq * s.n_kv_heads * kHeadDim * sizeof(__nv_bfloat16) + 255) / 256 * 256;
}

cudaError_t launch_attention_tc(tf_ctx* ctx, const tf_shape& s, const tf_filter_params& p,
                                const void* Q, const void* K, const void* V,
                                const int32_t* kept_idx, const int32_t* n_kept, void* O,
                                void* kv_compact, cudaStream_t st) {
    if (s.dtype != TF_BF16 || s.head_dim != kHeadDim) return cudaErrorNotSupported;
    if (s.batch == 0 || s.seq == 0) return cudaSuccess;
    const bool compact = (p.kv_visibility == TF_KV_RETAINED);
    CUtensorMap mapK, mapV;
    if (compact) {
        if (!kv_compact) return cudaErrorNotSupported;
        __nv_bfloat16* Kc = static_cast<__nv_bfloat16*>(kv_compact);
        __nv_bfloat16* Vc = reinterpret_cast<__nv_bfloat16*>(static_cast<char*>(kv_compact) + kv_compact_bytes(s) / 2);
        const int64_t dense[3] = {(int64_t)s.seq * s.n_kv_heads * kHeadDim, (int64_t)s.n_kv_heads * kHeadDim, kHeadDim};
        if (!make_kv_map(&mapK, Kc, dense, s.batch, s.seq, s.n_kv_heads) ||
            !make_kv_map(&mapV, Vc, dense, s.batch, s.seq, s.n_kv_heads))
            return cudaErrorNotSupported;
        const Strides3 ks = {s.k_stride[0], s.k_stride[1], s.k_stride[2]}, vs = {s.v_stride[0], s.v_stride[1], s.v_stride[2]};
        const unsigned gx = (unsigned)std::min<long long>(((long long)s.seq + 7) / 8, 4096);
        cudaError_t e = launch_dependent(compact_kv_kernel, dim3(gx, (unsigned)s.batch), dim3(256), 0, st,
                                         static_cast<const __nv_bfloat16*>(K), static_cast<const __nv_bfloat16*>(V), ks, vs,
                                         s.seq, s.n_kv_heads, kept_idx, n_kept, Kc, Vc);
        ctx->launches += 1;
        if (e != cudaSuccess) return e;
    } else if (!make_kv_map(&mapK, K, s.k_stride, s.batch, s.seq, s.n_kv_heads) ||
               !make_kv_map(&mapV, V, s.v_stride, s.batch, s.seq, s.n_kv_heads))
        return cudaErrorNotSupported;
    static bool attr_set_dev[kDeviceFlagSlots] = {};      // function attributes are per device
    bool& attr_set = attr_set_dev[ctx->device >= 0 && ctx->device < kDeviceFlagSlots ? ctx->device : 0];
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(attention_tc_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attention_tc_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPSmemBytes);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(attention_tc_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPSmemBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(attention_tc_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SplitCfg::kSmemBytes);
        if (e != cudaSuccess) return e;
        // The kernel moves registers from its third warpgroup to the softmax warpgroups (setmaxnreg: 168 -> 72
        // releases 128 x 96, 168 -> 216 takes 256 x 48).  An inc only receives what a dec of the same CTA
        // released and waits for it without limit, so the trade must balance: refuse to launch a build that
        // does not start at 168 registers per thread.
        // That is a defect of the build, not a property of the call: it is reported as an error of its own and
        // never answered by running another kernel.
        cudaFuncAttributes fa{};
        if (cudaFuncGetAttributes(&fa, attention_tc_kernel<0>) != cudaSuccess || fa.numRegs != 168 ||
            cudaFuncGetAttributes(&fa, attention_tc_kernel<1>) != cudaSuccess || fa.numRegs != 168 ||
            cudaFuncGetAttributes(&fa, attention_tc_kernel<2>) != cudaSuccess || fa.numRegs != 168 ||
            cudaFuncGetAttributes(&fa, attention_tc_split_kernel) != cudaSuccess || fa.numRegs != 168)
            return cudaErrorInvalidDeviceFunction;
        // the single form: 256 threads at 128 registers, traded 128 x 200 + 128 x 56
        e = cudaFuncSetAttribute(attention_tc_single_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes1);
        if (e != cudaSuccess) return e;
        if (cudaFuncGetAttributes(&fa, attention_tc_single_kernel) != cudaSuccess || fa.numRegs != kRegs1)
            return cudaErrorInvalidDeviceFunction;
        attr_set = true;
    }
    TcParams tp{};
    tp.Q = static_cast<const __nv_bfloat16*>(Q);
    tp.O = static_cast<__nv_bfloat16*>(O);
    tp.qs = {s.q_stride[0], s.q_stride[1], s.q_stride[2]};
    tp.os = {s.o_stride[0], s.o_stride[1], s.o_stride[2]};
    tp.S = s.seq; tp.Hq = s.n_q_heads; tp.Hkv = s.n_kv_heads; tp.window = s.window;
    const float scale = s.softmax_scale != 0.f ? s.softmax_scale : 1.f / sqrtf((float)s.head_dim);
    tp.scale_log2 = scale * 1.4426950408889634f;
    tp.kept_idx = kept_idx; tp.n_kept = n_kept;
    tp.status = ctx->dev_status;
    tp.compact = compact ? 1 : 0;
    tp.wait_cycles = ctx_wait_cycles(ctx);
    // The shared form needs enough CTAs to fill and balance the SMs (CTAs of one head differ in length by
    // the causal triangle); below that the split form, with twice as many CTAs of half the length, wins.
    // The number of retained rows is only known on the device: the ratio gives the expected count.
    const double kept_frac = (p.select_mode == TF_SELECT_RATIO) ? 1.0 - p.prune_ratio : 1.0;
    const double ctas_shared = (double)s.batch * s.n_q_heads * ceil(s.seq * kept_frac / (kQTiles * kTileM));
    const int sms = sm_count();
    const bool single = ctx->attention_form == 3;
    // ... when all its CTAs run at once, or when a row's keys are many: with few tiles per CTA the second wave of CTAs costs more
    // than the halved length saves (us, split / shared: 4 x 512 tokens x 32 heads, 4 tiles, 23.0 / 16.7, 2 x 768, 6 tiles, 22.7 /
    // 18.3, 2 x 1024, 8 tiles, 26.2 / 23.6, 1 x 1280, 10 tiles, 22.2 / 24.8, 1 x 1536, 12 tiles, 24.2 / 28.9, 1 x 2048, 16 tiles,
    // 34.4 / 37.7; grouped heads 2 x 1024 26.2 / 21.3).  The crossing is between 8 and 10 tiles; the line stays below it, where all
    // head groups of a call through host memory take the form that the whole call takes, and so have its bits.
    double keys = compact ? s.seq * kept_frac : (double)s.seq;
    if (s.window > 0) keys = std::min(keys, (double)s.window + kTileM / std::max(kept_frac, 1e-3));
    const bool split = ctx->attention_form == 2 ||
                       (ctx->attention_form == 0 && ctas_shared < 1.0 * sms && (2.0 * ctas_shared <= sms || keys > 7.0 * kTileN));
    // Grouped-query attention with an even number of query heads per KV head: the two Q tiles of a shared-form CTA are
    // the same 128 retained rows of two query heads of one group instead of 256 rows of one head; with a multiple of
    // four, the same 64 rows of four heads (two per tile): the shorter the span of positions a CTA's rows cover, the
    // fewer K/V tiles it has to visit beyond the window (or the causal triangle) itself.
    const int q_per_kv = (s.n_kv_heads > 0 && s.n_q_heads % s.n_kv_heads == 0) ? s.n_q_heads / s.n_kv_heads : 1;
    if ((ctx->attention_form == 4 && q_per_kv % 2) || (ctx->attention_form == 5 && q_per_kv % 4)) return cudaErrorNotSupported;
    const int hpt = ctx->attention_form == 4 ? 1 : ctx->attention_form == 5 ? 2     // heads per Q tile, 0 = one head per CTA
                  : (ctx->attention_form == 0 && !split) ? (q_per_kv % 4 == 0 ? 2 : q_per_kv % 2 == 0 ? 1 : 0) : 0;
    const bool heads = hpt > 0;
    const int rows_per_cta = heads ? kTileM / hpt : (split || single) ? kTileM : kQTiles * kTileM;
    tp.n_row_blocks = (s.seq + rows_per_cta - 1) / rows_per_cta;
    {
        const long long prunable = std::max<long long>((long long)s.seq - p.warmup_tokens, 0);
        const long long kept_est = (p.select_mode == TF_SELECT_RATIO) ? (long long)s.seq - std::min((long long)floor(p.prune_ratio * (double)s.seq), prunable)
                                                                      : (long long)s.seq;
        const long long blocks = (std::max<long long>(kept_est, 1) + rows_per_cta - 1) / rows_per_cta;
        tp.first_pair = (int)std::min<long long>(std::max<long long>(blocks - 1, 0), tp.n_row_blocks - 1);
        tp.n_blocks_est = tp.first_pair + 1;
        // Where the caller restricts what may be pruned the list can be of any length up to all tokens: every row block is an
        // item then.  (With items for the expected blocks only, 1 x 16384 tokens x 32 heads at ratio 0.9 with 5 % eligible: 224
        // items of nine or ten blocks on 148 SMs, 2513 us instead of 2307 with a CTA per block.)
        tp.n_items = p.eligible ? tp.n_row_blocks : tp.n_blocks_est;
    }
    const long long n_bh = (long long)(heads ? s.n_q_heads / (2 * hpt) : s.n_q_heads) * s.batch;
    const long long n_ctas = (long long)(split || single ? tp.n_row_blocks : tp.n_items) * n_bh;
    {
        // Groups of (batch, head) pairs.  Heaviest-first over ALL heads balances best and costs nothing while all of K
        // and V stays in L2 (c4: 555 -> 526 us).  Once the K and V of the heads that run together exceed L2, every CTA
        // streams its keys from HBM (3.9 KB per MFLOP of tile products): in short loops the balance still wins
        // (c3: 405 -> 372 us), under the power cap of a long run the HBM traffic lowers the clock and loses
        // (425 -> 445 us).  So a group is as many pairs as keep their K and V within kL2Budget, in equal groups
        // (c3: 5 groups of 32 heads, 438 -> 422 us in long loops, 430 -> 397 in short ones).  A window makes the row
        // blocks equally long, so there is nothing to balance and the row blocks of a pair stay together (c5: every
        // larger group measured 2-12 % slower).  A grid of a few CTAs per SM is balanced over all heads whatever the size.
        constexpr double kL2Budget = 72e6;
        const double kv_all = 2.0 * s.batch * (double)s.seq * s.n_kv_heads * kHeadDim * sizeof(__nv_bfloat16);
        const double kv_per_bh = kv_all / (double)std::max<long long>(n_bh, 1);
        const bool windowed = s.window > 0 && (long long)s.window + 1024 < s.seq;
        long long g = windowed ? 1 : std::max<long long>((long long)(kL2Budget / kv_per_bh), 1);
        if (kv_all <= kL2Budget || ctas_shared < 6.0 * sms) g = n_bh;
        g = std::min<long long>(g, std::max<long long>(n_bh, 1));
        const long long n_groups = (std::max<long long>(n_bh, 1) + g - 1) / g;      // equal groups, not a small last one
        g = (std::max<long long>(n_bh, 1) + n_groups - 1) / n_groups;
        tp.bh_group = (int)std::min<long long>(std::max<long long>(g, 1), std::max<long long>(n_bh, 1));
    }
    if (n_ctas > 0x7fffffffll) return cudaErrorInvalidValue;
    cudaError_t e;
    if (single) e = launch_dependent(attention_tc_single_kernel, dim3((unsigned)n_ctas), dim3(kThreads1), kSmemBytes1, st, tp, mapK, mapV);
    else if (split) e = launch_dependent(attention_tc_split_kernel, dim3((unsigned)n_ctas), dim3(kThreads), SplitCfg::kSmemBytes, st, tp, mapK, mapV);
    else if (hpt == 2) e = launch_dependent(attention_tc_kernel<2>, dim3((unsigned)n_ctas), dim3(kThreads), kPSmemBytes, st, tp, mapK, mapV);
    else if (hpt == 1) e = launch_dependent(attention_tc_kernel<1>, dim3((unsigned)n_ctas), dim3(kThreads), kPSmemBytes, st, tp, mapK, mapV);
    else       e = launch_dependent(attention_tc_kernel<0>, dim3((unsigned)n_ctas), dim3(kThreads), kPSmemBytes, st, tp, mapK, mapV);
    ctx->launches += 1;
    ctx->last_attention_kernel = single ? TF_KERNEL_ATTN_TC_SINGLE : hpt == 2 ? TF_KERNEL_ATTN_TC_HEAD_QUAD : hpt == 1 ? TF_KERNEL_ATTN_TC_HEAD_PAIR
                                        : split ? TF_KERNEL_ATTN_TC_SPLIT : TF_KERNEL_ATTN_TC_SHARED;
    return e;
}

}  // namespace tf
