// scl_kernel.cuh -- CRC-aided successive cancellation list decoding (Sec. II-A of the paper).
//
// One warp decodes one frame; a persistent grid takes frames from a device work counter (the
// CRC-failed frames compacted by the BP kernel, or all frames).  SC tree: level k holds 2^k LLRs
// per path (level n is the channel, level 0 the bit LLR).  For bit i > 0 with t = ctz(i) the
// path recomputes level t by g from level t+1 and the partial sums C_t of the left sibling, then
// levels t-1..0 by f; bit 0 runs f from the channel down.  f(a, b) = sign(a) sign(b) min(|a|,|b|),
// g(a, b, v) = b + (1 - 2v) a.
//
// List step at an information bit (lane = candidate): candidate c = 2p + b of path p gets metric
// m + |lambda| [b != HD(lambda)]; its rank is the number of candidates before it in
// (metric, index) order -- the paper's pruned pseudo sort d = sum H(m_c - m_j) made a total order
// by the index tie-break -- and the rank < L candidates survive, renumbered in ascending index.
//
// Leaf blocks: the tree below level 6 is a 32-bit leaf block.  Lane p holds path p's LLR arrays of
// levels 4..1 (30 values) and its partial sums of levels 0..4 (one word each) in registers; level 5
// stays in shared memory, one row per path.  Aligned nodes of 32, 16, 8 and 4 bits that are all
// frozen or all information are taken whole where that gives the bit-by-bit result exactly
// (leaf_frozen, leaf_all_hard); the rest goes bit by bit.  When a list step duplicates paths, a
// survivor copies from its parent's lane (shuffles) only the leaf levels that a later bit of the
// block reads before rewriting: level k after bit r iff bit k-1 of r is clear, the partial sum of
// level k iff bit k of r is set.
//
// Upper levels (LLR 6..n-1, partial sums 5..n) are touched once per block.  They use lazy copies:
// every upper level keeps L physical arrays and a path holds one 5-bit pointer per level, packed in
// two registers per table.  A survivor copies only its parent's pointer words; a path about to
// rewrite a level it shares takes a free array of that level (the lowest-numbered sharer keeps the
// old one), so no upper-level data is ever copied.  The small upper levels live in the warp's
// shared memory, the large ones in its slot of the global workspace (L2-resident).
//
// Partial sums: after deciding bit i, the completed subtree re-encodes bottom-up,
// v_{k+1} = (C_k xor v_k) || v_k, until the first level k where the completed node is a left
// child (k = number of trailing ones of i); v_k is stored there.  After the last bit the level-n
// array holds the path's codeword x, and u = x G (G is an involution) gives the decided bits for
// the CRC check and the output.
#pragma once

#include <algorithm>
#include <type_traits>

#include "polar_common.cuh"

namespace polar {

struct SCLArgs {
    const float* llr;
    int B;
    int L;
    uint8_t* bits;
    uint8_t* status;
    const DevCode* code;
    const int* list;   // frame indices to decode (null: 0..B-1)
    const int* count;  // device count of `list` (null: B)
    int* next;         // work counter, zero before the launch
    float* scratch;    // per-warp slots of the global levels (null: all levels in shared memory)
    int row_bytes;
    int KS, KC;        // last LLR / partial-sum level kept in shared memory (single code)
    int KSm, KCm;      // the same when a CTA decodes one frame at a time, with all its shared memory
    int warp_words;    // shared-memory words per warp
    int list_words;    // shared-memory words per list (two lists per warp when L <= 8)
    long long slot_words;  // global words per list
    // several codes in one batch: code_of[frame] selects codes[], llr_off[frame] the LLR row
    const int* code_of;
    const long long* llr_off;
    const DevCode* codes[32];
};

__host__ __device__ inline int scl_cw(int k) { return k < 5 ? 1 : 1 << (k - 5); }  // words of a level-k C array
// Per-path stride of the level-k C arrays: one pad word beyond a single word makes the stride
// odd, so the same word of different paths falls in different banks.
__host__ __device__ inline int scl_cs(int k) { return scl_cw(k) > 1 ? scl_cw(k) + 1 : 1; }
__host__ __device__ inline int scl_cssum(int k) { return k <= 5 ? k : (1 << (k - 5)) + k - 2; }  // sum of cs(q), q < k

__host__ __device__ inline int log2_host(int v)
{
    int n = 0;
    while ((1 << n) < v) ++n;
    return n;
}

// Host plan of the shared/global split of the upper levels for (N, L): LLR levels 6..KS and
// partial-sum levels 5..KC in shared memory, the rest in the warp's global slot.
struct SCLPlan {
    int KS, KC;
    int warp_words, list_words;
    long long slot_words;
};
// Level 5 of a path is computed by its lane from the path's level-6 array, which is always in shared
// memory, and kept in a staging row of 32 words.  Both are read and written by 32 lanes at a time, each
// in its own row, 16 bytes per access: the 16-byte chunk index is XORed with the row number modulo 8,
// which spreads eight rows over all banks.
constexpr int kSclStage = 32;
__host__ __device__ inline int scl_chunk(int row, int chunk) { return (chunk ^ (row & 7)) << 2; }  // word offset
// per warp: 16 words of list-step scratch, then the packed path pointers of a level and the path count
constexpr int kSclScratch = 16, kSclPtrs = 40, kSclWarpWords = kSclScratch + kSclPtrs;
__host__ __device__ inline long long scl_smem_llr_words(int KS, int L) { return KS >= 6 ? (long long)L * ((2 << KS) - 64) : 0; }
__host__ __device__ inline long long scl_smem_c_words(int KC, int L) { return KC >= 5 ? (long long)L * (scl_cssum(KC + 1) - 5) : 0; }
// `lists` = frames per warp (1, or 2 with half-warp lists): the shared-memory budget of a frame
// is divided by it.
__host__ __device__ inline SCLPlan scl_plan(int N, int L, bool all_smem, int lists = 1)
{
    const int n = log2_host(N);
    SCLPlan p{};
    if (all_smem) {
        p.KS = n - 1;
        p.KC = n;
    } else {
        p.KS = 6;
        // up to 6 KB of LLR levels per frame, at least level 6
        while (p.KS + 1 <= n - 1 && 4 * scl_smem_llr_words(p.KS + 1, L) * lists <= 6144) ++p.KS;
        p.KC = 4;
        while (p.KC + 1 <= n && 4 * scl_smem_c_words(p.KC + 1, L) * lists <= 2048) ++p.KC;
    }
    // per list: [LLR levels 6..KS][level-5 staging, L rows of 32 words][C levels 5..KC]; per warp:
    // the lists, then kSclWarpWords words of scratch
    p.list_words = (int)(scl_smem_llr_words(p.KS, L) + scl_smem_c_words(p.KC, L)) + L * kSclStage;
    p.list_words = (p.list_words + 3) & ~3;
    p.warp_words = lists * p.list_words + kSclWarpWords;
    p.slot_words = (long long)L * (N - (2 << p.KS)) + (long long)L * (scl_cssum(n + 1) - scl_cssum(p.KC + 1));
    return p;
}
// The levels in shared memory of a list that has `words` of it to itself (and fits there with the split
// of scl_plan): as many LLR levels as leave room for the partial sums up to level 8, then the partial
// sums.  With the per-warp split the partial sums of long codes and all but one or two LLR levels came
// from L2, and a frame alone on its SM waits for every access (N = 4096, L = 32, 138 frames: 5.20 -> 5.15 ms with the exact-g BP).
inline void scl_plan_cta(int N, int L, long long words, int* KS, int* KC)
{
    const int n = log2_host(N);
    const auto fits = [&](int ks, int kc) {
        return scl_smem_llr_words(ks, L) + L * kSclStage + scl_smem_c_words(kc, L) <= words;
    };
    int ks = 6, kc = 5;
    while (ks + 1 <= n - 1 && fits(ks + 1, std::min(n, 8))) ++ks;
    while (kc + 1 <= n && fits(ks, kc + 1)) ++kc;
    if (ks < *KS || kc < *KC) return;
    *KS = ks;
    *KC = kc;
}
inline bool scl_fits_smem(int N, int L) { return 4LL * scl_plan(N, L, true).warp_words <= 80 * 1024; }
constexpr int kSclWarpsPerSM = 32;
constexpr int kSclWarpsPerCTA = 4;
inline int scl_sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms > 0 ? sms : 1;
}
// List width of a CA-SCL launch, mixed batches included: two frames per warp (half-warp lists) for
// L <= 8 in the global layout.
inline bool scl_two_lists(int L, bool all_smem) { return L <= 8 && !all_smem; }
// global workspace of the SCL list arrays (one slot per resident list: up to kSclWarpsPerSM lists
// per SM)
inline size_t scl_scratch_bytes(int N, int L)
{
    const long long w = std::max(scl_plan(N, L, false).slot_words, scl_plan(N, L, false, 2).slot_words);
    return (size_t)scl_sm_count() * kSclWarpsPerSM * (size_t)w * 4;
}

// 5-bit pointer of upper level k (5 <= k <= 12) in a path's two pointer words: levels 1..6 in word
// 0, levels 7..12 in word 1
__device__ __forceinline__ uint32_t fld(const uint32_t (&w)[2], int k)
{
    return (k <= 6 ? w[0] >> (5 * (k - 1)) : w[1] >> (5 * (k - 7))) & 31u;
}
__device__ __forceinline__ void set_fld(uint32_t (&w)[2], int k, uint32_t v)
{
    const int s = 5 * (k <= 6 ? k - 1 : k - 7);
    if (k <= 6)
        w[0] = (w[0] & ~(31u << s)) | (v << s);
    else
        w[1] = (w[1] & ~(31u << s)) | (v << s);
}
static_assert(kMaxN <= 4096, "upper-level pointers of levels up to 12");

// Lanes of one list: the whole warp (W = 32, one frame per warp) or one half of it (W = 16, two
// frames per warp, lists of at most 8 paths).  Path p of the list sits in lane base + p.  Every
// collective below is executed by all 32 lanes; with W = 16 the two halves compute their own
// results (shuffle offsets below 16 stay within a half).
template <int W>
struct Lanes {
    int lane, pl, base;
    __device__ __forceinline__ Lanes() : lane(threadIdx.x & 31), pl(lane & (W - 1)), base(lane & ~(W - 1)) {}
    __device__ __forceinline__ uint32_t ballot(bool p) const
    {
        const uint32_t b = __ballot_sync(0xffffffffu, p);
        return W == 32 ? b : (b >> base) & 0xffffu;
    }
    template <class V>
    __device__ __forceinline__ V shfl(V v, int p) const { return __shfl_sync(0xffffffffu, v, base + p); }
    // Reductions over the list: one redux.sync for a whole-warp list; for half-warp lists one per
    // half, each lane feeding the other half's reduction the identity, and keeping its own half's.
    __device__ __forceinline__ uint32_t red_or(uint32_t v) const
    {
        if constexpr (W == 32) {
            return __reduce_or_sync(0xffffffffu, v);
        } else {
            const uint32_t lo = __reduce_or_sync(0xffffffffu, base ? 0u : v);
            const uint32_t hi = __reduce_or_sync(0xffffffffu, base ? v : 0u);
            return base ? hi : lo;
        }
    }
    __device__ __forceinline__ uint32_t red_xor(uint32_t v) const
    {
        if constexpr (W == 32) {
            return __reduce_xor_sync(0xffffffffu, v);
        } else {
            const uint32_t lo = __reduce_xor_sync(0xffffffffu, base ? 0u : v);
            const uint32_t hi = __reduce_xor_sync(0xffffffffu, base ? v : 0u);
            return base ? hi : lo;
        }
    }
    __device__ __forceinline__ uint32_t red_max(uint32_t v) const
    {
        if constexpr (W == 32) {
            return __reduce_max_sync(0xffffffffu, v);
        } else {
            const uint32_t lo = __reduce_max_sync(0xffffffffu, base ? 0u : v);
            const uint32_t hi = __reduce_max_sync(0xffffffffu, base ? v : 0u);
            return base ? hi : lo;
        }
    }
    __device__ __forceinline__ uint32_t red_min(uint32_t v) const
    {
        if constexpr (W == 32) {
            return __reduce_min_sync(0xffffffffu, v);
        } else {
            const uint32_t lo = __reduce_min_sync(0xffffffffu, base ? 0xffffffffu : v);
            const uint32_t hi = __reduce_min_sync(0xffffffffu, base ? v : 0xffffffffu);
            return base ? hi : lo;
        }
    }
    __device__ __forceinline__ uint32_t match_any(uint32_t v) const
    {
        const uint32_t m = __match_any_sync(0xffffffffu, W == 32 ? v : v | ((uint32_t)base << 8));
        return W == 32 ? m : (m >> base) & 0xffffu;
    }
    // the larger of the two lists' values (W = 16), for loop bounds every lane must share
    __device__ __forceinline__ int both_max(int v) const
    {
        return W == 32 ? v : max(v, __shfl_xor_sync(0xffffffffu, v, 16));
    }
};

// A path about to rewrite level k that it shares takes a free array of that level (lane = path;
// `act` active paths; the lowest lane of each group of sharers keeps its array).  A list without
// sharing is left unchanged, so the call is safe for a list that does not need it.
template <int W>
__device__ __forceinline__ void scl_own(uint32_t (&w)[2], int k, int act, int L)
{
    const Lanes<W> sg;
    const bool on = sg.pl < act;
    const uint32_t mine = on ? fld(w, k) : 64u + sg.pl;
    const uint32_t same = sg.match_any(mine);
    const uint32_t below = (1u << sg.pl) - 1u;
    const bool need = on && (same & below) != 0u;
    const uint32_t used = sg.red_or(on ? (1u << mine) : 0u);
    uint32_t freem = ~used & (L >= 32 ? 0xffffffffu : ((1u << L) - 1u));
    const int r = __popc(sg.ballot(need) & below);
    if (need) {
#pragma unroll 1
        for (int q = 0; q < r; ++q) freem &= freem - 1u;  // drop the r lowest free arrays
        set_fld(w, k, (uint32_t)(__ffs(freem) - 1));
    }
}

// g = b + (1 - 2v) a with v = bit j of c: a's sign flipped by the bit (b - a and b + (-a) are the same)
__device__ __forceinline__ float scl_g(float a, float b, uint32_t c, int j)
{
    return __fadd_rn(b, __uint_as_float(__float_as_uint(a) ^ ((c << (31 - j)) & 0x80000000u)));
}

struct SCLWarp {
    float* stage;  // shared level-5 staging rows [L][kSclStage]
    float* sA;     // shared LLR levels 6..KS
    uint32_t* sC;  // shared partial-sum levels 5..KC
    float* gA;     // global LLR levels KS+1..n-1
    uint32_t* gC;  // global partial-sum levels KC+1..n
    int L, KS, KC;
    __device__ __forceinline__ float* A(int k) const  // k >= 6
    {
        return k <= KS ? sA + L * ((1 << k) - 64) : gA + L * ((1 << k) - (2 << KS));
    }
    __device__ __forceinline__ uint32_t* Cl(int k) const  // k >= 5
    {
        return k <= KC ? sC + L * (scl_cssum(k) - 5) : gC + L * (scl_cssum(k) - scl_cssum(KC + 1));
    }
};

// ------------------------------------------------------------------ leaf block
// A 32-bit leaf block is walked as a tree over the path's registers: level 5 stays in the shared
// staging rows (a path keeps the number of its row), levels 4..1 live in registers.
template <int LEN>
__device__ __forceinline__ void leaf_f(const float (&src)[2 * LEN], float (&dst)[LEN])
{
#pragma unroll
    for (int j = 0; j < LEN; ++j) dst[j] = xmin(src[j], src[j + LEN]);
}
template <int LEN>
__device__ __forceinline__ void leaf_g(const float (&src)[2 * LEN], float (&dst)[LEN], uint32_t c)
{
#pragma unroll
    for (int j = 0; j < LEN; ++j) dst[j] = scl_g(src[j], src[j + LEN], c, j);
}
template <int LEN>
__device__ __forceinline__ void leaf_copy(float (&a)[LEN], int parent)
{
#pragma unroll
    for (int j = 0; j < LEN; ++j) a[j] = __shfl_sync(0xffffffffu, a[j], parent);
}

struct Leaf {
    float l4[16], l3[8], l2[4], l1[2];
    uint32_t c[5];  // partial sums of the left siblings at levels 0..4
    int row;        // staging row of this path's level 5
};

// Metric of a node whose 2^K leaves are all frozen, from the node's LLRs: every leaf LLR (partial
// sums 0, so g is a plain addition) in order, each penalty added in order -- the same operations
// as bit by bit, without the bit loop.  m - min(lambda, 0) = m + |lambda| [lambda < 0].
template <int LEN>
__device__ __forceinline__ void leaf_frozen(const float (&a)[LEN], float& pm)
{
    if constexpr (LEN == 1) {
        pm = __fsub_rn(pm, fminf(a[0], 0.0f));
    } else {
        constexpr int H = LEN / 2;
        float b[H];
#pragma unroll
        for (int j = 0; j < H; ++j) b[j] = xmin(a[j], a[j + H]);
        leaf_frozen<H>(b, pm);
#pragma unroll
        for (int j = 0; j < H; ++j) b[j] = __fadd_rn(a[j + H], a[j]);
        leaf_frozen<H>(b, pm);
    }
}

// A node of 2^K information bits, decided at once.  Let every path take its hard decisions inside
// the node: f keeps the smaller magnitude and g then adds magnitudes of equal signs, so the first
// leaf's |lambda| is m = min |a_j| and no later leaf's is smaller (also after rounding, which is
// monotone).  So if the full list's largest metric is below every path's metric plus m, the list
// step's shortcut holds at the first bit and, metrics unchanged, at every later one: the survivors
// are the paths themselves with the sign bits of a as the node's codeword.  If the condition
// fails, the first bit's shortcut fails as well.  (A zero LLR makes m = 0 and fails it, so the
// signs are those of nonzero values.)
template <int W, int LEN>
__device__ __forceinline__ bool leaf_all_hard(const Lanes<W>& sg, const float (&a)[LEN], float pm, int act, int L,
                                              uint32_t& v)
{
    if constexpr (W == 32) {
        if (act != L) return false;
    } else {
        if (!__all_sync(0xffffffffu, act == L || act == 0)) return false;
    }
    float m[LEN >= 4 ? 4 : LEN];
    v = 0u;
#pragma unroll
    for (int j = LEN - 1; j >= 0; --j) {
        const float x = a[j];
        v = __funnelshift_l(__float_as_uint(x), v, 1);
        constexpr int Q = LEN >= 4 ? 4 : LEN;
        m[j % Q] = j + Q >= LEN ? fabsf(x) : fminf(m[j % Q], fabsf(x));
    }
    float mm = m[0];
#pragma unroll
    for (int q = 1; q < (LEN >= 4 ? 4 : LEN); ++q) mm = fminf(mm, m[q]);
    const bool on = sg.pl < act;
    const uint32_t hd_max = sg.red_max(on ? __float_as_uint(pm) : 0u);
    const uint32_t pen_min = sg.red_min(on ? __float_as_uint(__fadd_rn(pm, mm)) : 0xffffffffu);
    if constexpr (W == 32)
        return hd_max < pen_min;
    else
        return __all_sync(0xffffffffu, hd_max < pen_min || act == 0);
}

// Launches the persistent CA-SCL grid (defined in scl_launch.cu).  `a.scratch` null selects the
// all-shared-memory layout; list_words_max / slot_words_max widen the per-warp storage for mixed
// batches.
cudaError_t scl_launch(SCLArgs a, int N, int L, cudaStream_t st, int list_words_max = 0,
                       long long slot_words_max = 0);

#ifdef POLAR_SCL_KERNELS
// One list step at an information bit: candidates, ranks, survivors.  Lane = path in and out;
// returns the survivor's parent lane and decided bit, updates pm/act, reports duplication and
// whether any survivor sits in another lane than its parent (`moved`, warp-uniform).  `ranked`: the
// full-list shortcut is known to fail at this bit.
template <bool TWO>
__device__ __forceinline__ int scl_list_step(float lam, float& pm, int& act, int L, uint8_t* selc, bool ranked,
                                             uint32_t& bitv, bool& dup, bool& moved)
{
    const int lane = threadIdx.x & 31;
    if (act == L && !ranked) {
        // Full list: when every path's hard-decision child (metric pm) comes before every
        // penalised child (pm + |lambda|), the L survivors are exactly the hard-decision children,
        // in path order -- the same result as the ranking below, without it.  Metrics are >= +0,
        // so their bit patterns order like their values.
        const bool on = lane < act;
        const uint32_t hd_max = __reduce_max_sync(0xffffffffu, on ? __float_as_uint(pm) : 0u);
        const uint32_t pen_min =
            __reduce_min_sync(0xffffffffu, on ? __float_as_uint(__fadd_rn(pm, fabsf(lam))) : 0xffffffffu);
        if (hd_max < pen_min) {
            bitv = lam < 0.0f ? 1u : 0u;
            dup = false;
            moved = false;
            return lane;
        }
    }
    const int nc = 2 * act;
    float cm0, cm1 = 0.0f;
    {
        const float lp = __shfl_sync(0xffffffffu, lam, (lane >> 1) & 31);
        const float pp = __shfl_sync(0xffffffffu, pm, (lane >> 1) & 31);
        cm0 = ((uint32_t)(lane & 1) != (uint32_t)(lp < 0.0f)) ? __fadd_rn(pp, fabsf(lp)) : pp;
    }
    if constexpr (TWO) {
        const float lp = __shfl_sync(0xffffffffu, lam, 16 + (lane >> 1));
        const float pp = __shfl_sync(0xffffffffu, pm, 16 + (lane >> 1));
        cm1 = ((uint32_t)(lane & 1) != (uint32_t)(lp < 0.0f)) ? __fadd_rn(pp, fabsf(lp)) : pp;
    }
    const uint32_t below = (1u << lane) - 1u;
    uint32_t km0, km1 = 0u;
    if (nc <= L) {
        // every candidate survives
        km0 = __ballot_sync(0xffffffffu, lane < nc);
        if constexpr (TWO) km1 = __ballot_sync(0xffffffffu, lane + 32 < nc);
    } else if (TWO || nc > 16) {
        // Threshold selection.  tau = the L-th smallest metric: with two candidates per lane, a
        // bitonic sort of the first 32 ascending and of the second 32 descending, whose
        // element-wise minimum holds the 32 smallest (the half-cleaner of a bitonic merge); with
        // one per lane, the sorted value of lane L - 1.  The survivors are every candidate below
        // tau and the lowest-index candidates equal to tau -- the L smallest in (metric, index)
        // order, the same set as ranking every candidate.
        const float inf = __int_as_float(0x7f800000);
        float x0 = lane < nc ? cm0 : inf;
        float x1 = (TWO && lane + 32 < nc) ? cm1 : inf;
#pragma unroll
        for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
            for (int j = k >> 1; j > 0; j >>= 1) {
                const float o0 = __shfl_xor_sync(0xffffffffu, x0, j);
                const bool take_min = ((lane & j) == 0) == ((lane & k) == 0);
                if constexpr (TWO) {
                    const float o1 = __shfl_xor_sync(0xffffffffu, x1, j);
                    x0 = take_min ? fminf(x0, o0) : fmaxf(x0, o0);
                    x1 = take_min ? fmaxf(x1, o1) : fminf(x1, o1);  // descending
                } else {
                    x0 = take_min ? fminf(x0, o0) : fmaxf(x0, o0);
                }
            }
        }
        float tau;
        if constexpr (TWO)
            tau = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fminf(x0, x1))));  // L = 32
        else
            tau = __shfl_sync(0xffffffffu, x0, L - 1);
        const bool v0 = lane < nc, v1 = TWO && lane + 32 < nc;
        const uint32_t lt0 = __ballot_sync(0xffffffffu, v0 && cm0 < tau);
        const uint32_t lt1 = TWO ? __ballot_sync(0xffffffffu, v1 && cm1 < tau) : 0u;
        const uint32_t eq0 = __ballot_sync(0xffffffffu, v0 && cm0 == tau);
        const uint32_t eq1 = TWO ? __ballot_sync(0xffffffffu, v1 && cm1 == tau) : 0u;
        const int need = L - __popc(lt0) - __popc(lt1);
        km0 = lt0 | __ballot_sync(0xffffffffu, ((eq0 >> lane) & 1u) && __popc(eq0 & below) < need);
        if constexpr (TWO)
            km1 = lt1 | __ballot_sync(0xffffffffu, ((eq1 >> lane) & 1u) && __popc(eq0) + __popc(eq1 & below) < need);
    } else {
        // few candidates (at most 16, one per lane): rank by counting
        int rank0 = 0;
#pragma unroll 8
        for (int c2 = 0; c2 < nc; ++c2) {
            const float o = __shfl_sync(0xffffffffu, cm0, c2);
            rank0 += (o < cm0) || (o == cm0 && c2 < lane);
        }
        km0 = __ballot_sync(0xffffffffu, lane < nc && rank0 < L);
    }
    if (km0 & (1u << lane)) selc[__popc(km0 & below)] = (uint8_t)lane;
    if (TWO && (km1 & (1u << lane))) selc[__popc(km0) + __popc(km1 & below)] = (uint8_t)(lane + 32);
    dup = ((km0 & (km0 >> 1) & 0x55555555u) | (km1 & (km1 >> 1) & 0x55555555u)) != 0u;
    const int nact = __popc(km0) + __popc(km1);
    __syncwarp();
    const int cq = lane < nact ? selc[lane] : 0;
    __syncwarp();
    const float m0 = __shfl_sync(0xffffffffu, cm0, cq & 31);
    const float m1 = TWO ? __shfl_sync(0xffffffffu, cm1, cq & 31) : 0.0f;
    bitv = (uint32_t)(cq & 1);
    pm = lane < nact ? (cq < 32 ? m0 : m1) : 0.0f;
    act = nact;
    moved = __any_sync(0xffffffffu, lane < nact && (cq >> 1) != lane);
    return cq >> 1;
}

// List step of a half-warp list (W = 16, L <= 8, at most 16 candidates, one per lane): the same
// survivors as scl_list_step, computed with loop bounds shared by both halves -- the fast path is
// taken only when both lists qualify, and the ranks count over all 2L candidate slots with the
// unused ones at +inf.  Returns the survivor's parent path (within the list).
__device__ __forceinline__ int scl_list_step_half(float lam, float& pm, int& act, int L, uint8_t* selc, bool ranked,
                                                  uint32_t& bitv, bool& dup, bool& moved)
{
    const Lanes<16> sg;
    const int pl = sg.pl;
    if (!ranked) {
        const bool on = pl < act;
        const uint32_t hd_max = sg.red_max(on ? __float_as_uint(pm) : 0u);
        const uint32_t pen_min = sg.red_min(on ? __float_as_uint(__fadd_rn(pm, fabsf(lam))) : 0xffffffffu);
        const bool fast = act == L && hd_max < pen_min;
        if (__all_sync(0xffffffffu, fast || act == 0)) {
            bitv = lam < 0.0f ? 1u : 0u;
            dup = false;
            moved = false;
            return pl;
        }
    }
    const int nc = 2 * act;
    const float inf = __int_as_float(0x7f800000);
    float cm0;
    {
        const float lp = sg.shfl(lam, (pl >> 1) & 15);
        const float pp = sg.shfl(pm, (pl >> 1) & 15);
        cm0 = ((uint32_t)(pl & 1) != (uint32_t)(lp < 0.0f)) ? __fadd_rn(pp, fabsf(lp)) : pp;
        if (pl >= nc) cm0 = inf;
    }
    int rank0 = 0;
    for (int c2 = 0; c2 < 2 * L; ++c2) {
        const float o = sg.shfl(cm0, c2);
        rank0 += (o < cm0) || (o == cm0 && c2 < pl);
    }
    const uint32_t below = (1u << pl) - 1u;
    const uint32_t km0 = sg.ballot(pl < nc && (nc <= L || rank0 < L));
    uint8_t* sel = selc + sg.base;
    if (km0 & (1u << pl)) sel[__popc(km0 & below)] = (uint8_t)pl;
    dup = (km0 & (km0 >> 1) & 0x55555555u) != 0u;
    const int nact = __popc(km0);
    __syncwarp();
    const int cq = pl < nact ? sel[pl] : 0;
    __syncwarp();
    const float m0 = sg.shfl(cm0, cq & 15);
    bitv = (uint32_t)(cq & 1);
    pm = pl < nact ? m0 : 0.0f;
    act = nact;
    moved = __any_sync(0xffffffffu, pl < nact && (cq >> 1) != pl);
    return cq >> 1;
}

// Decode one frame per list: the warp's frame (W = 32), or each half-warp's frame (W = 16; a
// half without a frame passes frame < 0 and decodes nothing).  TWO: L = 32, two candidates per
// lane.  mw (W = 32): every warp of the CTA calls with the same frame; warp 0 holds the list and runs
// the bit loop, and all warps share the element-parallel upper-level updates, with CTA barriers
// around each level.  W = 32 passes the path pointers of a level through `ptab` (kSclPtrs words; mw:
// warp 0's), W = 16 by shuffles.  (mw is a run-time flag and everything done once per frame is a loop:
// the body is long, and with 16 warps at different places of it instruction fetch is a top stall.)
template <bool TWO, int W>
__device__ void scl_decode_frame(const SCLArgs& a, const DevCode& C, int frame, const SCLWarp& S, uint8_t* selc,
                                 uint32_t* ptab, const bool mw)
{
    static_assert(W == 32 || !TWO, "half-warp lists hold at most 8 paths");
    const bool lead = !mw || threadIdx.x < 32;
    auto level_sync = [&]() {
        if (W == 32 && mw)
            __syncthreads();
        else
            __syncwarp();
    };
    const Lanes<W> sg;
    const int lane = sg.pl;  // path of this lane within its list
    const int N = C.N, n = C.n, L = a.L;
    const float* y = a.llr + (frame < 0 ? 0 : (a.llr_off ? a.llr_off[frame] : (long long)frame * N));
    const bool y16 = (reinterpret_cast<uintptr_t>(y) & 15u) == 0;
    uint32_t pA[2] = {0u, 0u}, pC[2] = {0u, 0u};  // upper-level pointer rows of path `lane`
    float pm = 0.0f;
    int act = frame < 0 ? 0 : 1;
    uint32_t shA = 0u, shC = 0u;  // upper levels that may be shared since the last duplication
    Leaf lf;
#pragma unroll
    for (int k = 0; k < 5; ++k) lf.c[k] = 0u;
    const int nblocks = N >> 5;
    for (int blk = 0; blk < nblocks; ++blk) {
        // ------------------------------------------------ upper levels on entering the block
        const int t = blk == 0 ? n : 5 + __ffs(blk) - 1;
        const int act_both = sg.both_max(act);
        // element stride of a round: the list's lanes, or every thread of the CTA
        const int TW = W == 32 && mw ? (int)blockDim.x : W, tix = W == 32 && mw ? (int)threadIdx.x : lane;
        // Two levels per pass: a lane's two units of level k are partners, so level k - 1 comes from
        // them in registers instead of being read back (level 6 alone takes a pass when it is left).
#pragma unroll 1
        for (int k = min(t, n - 1); k >= 6;) {
            const bool two = k > 6;
            if (lead) {
                const uint32_t both = two ? 3u << (k - 1) : 1u << k;
                const uint32_t own = __reduce_or_sync(0xffffffffu, shA & both);
#pragma unroll 1
                for (int q = k; q >= k - (two ? 1 : 0); --q)
                    if ((own >> q) & 1u) scl_own<W>(pA, q, act, L);
                shA &= ~both;
            }
            const bool use_g = blk != 0 && k == t;
            const bool from_ch = k + 1 == n;
            const int len = 1 << k, sh = two ? k - 3 : k - 2;
            float* dst = S.A(k);
            float* dst2 = S.A(two ? k - 1 : k);
            const float* srcb = from_ch ? y : S.A(k + 1);
            const uint32_t* cbk = S.Cl(k);
            // a path's arrays of levels k (written), k + 1 (read), of the partial sums of level k, and
            // of level k - 1 (written)
            const uint32_t mine = fld(pA, k) | (from_ch ? 0u : fld(pA, k + 1) << 8) | fld(pC, k) << 16 |
                                  fld(pA, two ? k - 1 : k) << 24;
            int nact = act, nact_both = act_both;
            if constexpr (W == 32) {
                if (lead) {
                    ptab[lane] = mine;
                    if (lane == 0) ptab[32] = (uint32_t)act;
                }
                level_sync();
                nact = nact_both = (int)ptab[32];
            }
            const int cwk = scl_cs(k), tot = nact << sh, tmax = nact_both << sh;
            // level 6 is stored with permuted chunks
            const int swz = k == 6 ? 7 : 0, swz2 = k == 7 ? 7 : 0;
            // Units of four consecutive elements of one path (a level has at least 64): one 16-byte
            // load per operand and one set of pointers per unit, two units per lane and round.  All
            // loads of a round are issued before any store, so the L2 latency of the upper levels
            // (global for long lists) is paid once per round.  The loads are unconditional (a unit
            // past the list's end reads a valid slot: its path index is below L and its offset below
            // len), so nothing but the stores is predicated and the units' chains interleave.
            // The channel row is staged as CA-SCL reads it; the caller's row may start at any float,
            // so its 16-byte loads need `y16`.
            auto rounds = [&](auto USE_G) {
                constexpr bool G = decltype(USE_G)::value;
#pragma unroll 1
                for (int e0 = 0; e0 < tmax; e0 += two ? TW : 2 * TW) {
                    float4 va[2], vb[2], r[2];
                    uint32_t vw[2], ptr[2];
                    int u[2];
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int e = e0 + tix + (two ? 0 : TW * q);
                        const int p = (e >> sh) & (W - 1);
                        u[q] = (e & ((1 << sh) - 1)) + (two ? q << sh : 0);
                        ptr[q] = W == 32 ? ptab[p] : sg.shfl(mine, p);
                        const float* src = srcb + ((((ptr[q] >> 8) & 31u) << (k + 1)) + 4 * u[q]);
                        if (from_ch && !y16) {
                            va[q] = make_float4(src[0], src[1], src[2], src[3]);
                            vb[q] = make_float4(src[len], src[len + 1], src[len + 2], src[len + 3]);
                        } else {
                            va[q] = *reinterpret_cast<const float4*>(src);
                            vb[q] = *reinterpret_cast<const float4*>(src + len);
                        }
                        if constexpr (G)
                            vw[q] = cbk[((ptr[q] >> 16) & 31u) * cwk + (u[q] >> 3)] >> (4 * (u[q] & 7));
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int d = ptr[q] & 31u;
                        float4 x = va[q], y4 = vb[q];
                        if (from_ch) {
                            x = make_float4(scl_stage(x.x), scl_stage(x.y), scl_stage(x.z), scl_stage(x.w));
                            y4 = make_float4(scl_stage(y4.x), scl_stage(y4.y), scl_stage(y4.z), scl_stage(y4.w));
                        }
                        if constexpr (G)
                            r[q] = make_float4(scl_g(x.x, y4.x, vw[q], 0), scl_g(x.y, y4.y, vw[q], 1),
                                               scl_g(x.z, y4.z, vw[q], 2), scl_g(x.w, y4.w, vw[q], 3));
                        else
                            r[q] = make_float4(xmin(x.x, y4.x), xmin(x.y, y4.y), xmin(x.z, y4.z), xmin(x.w, y4.w));
                        if (e0 + tix + (two ? 0 : TW * q) < tot)
                            *reinterpret_cast<float4*>(dst + (d << k) + 4 * (u[q] ^ (d & swz))) = r[q];
                    }
                    if (two && e0 + tix < tot) {
                        const int d = ptr[0] >> 24;
                        *reinterpret_cast<float4*>(dst2 + (d << (k - 1)) + 4 * (u[0] ^ (d & swz2))) =
                            make_float4(xmin(r[0].x, r[1].x), xmin(r[0].y, r[1].y), xmin(r[0].z, r[1].z),
                                        xmin(r[0].w, r[1].w));
                    }
                }
            };
            if (use_g)
                rounds(std::true_type{});
            else
                rounds(std::false_type{});
            level_sync();
            k -= two ? 2 : 1;
        }
        if (!lead) continue;  // the helper warps only share the upper levels
        // ------------------------------------------------ the 32 bits of the block
        // A runtime walk of the block's tree, four bits at a time; one copy of the list step serves
        // all bits (unrolling it per bit overflowed the instruction cache).  Lanes past the list
        // work on its first array and row and compute values nobody reads.
        const uint32_t fw = C.frozen_bits[blk], dw = C.decided_bits[blk];
        uint32_t v5 = 0u;
        lf.row = lane < L ? lane : 0;
        int r = 0, failed = -1;  // failed: bit at which the full-list shortcut is known to fail
        {
            // level 5 of this lane's path, from its level-6 array
            float l5[32];
            const int m6 = lane < L ? (int)fld(pA, 6) : 0;
            const float* row6 = S.sA + m6 * 64;
            const uint32_t c5 = S.Cl(5)[fld(pC, 5)];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float4 x = *reinterpret_cast<const float4*>(row6 + scl_chunk(m6, c));
                const float4 z = *reinterpret_cast<const float4*>(row6 + scl_chunk(m6, c + 8));
                if (t == 5) {
                    l5[4 * c] = scl_g(x.x, z.x, c5, 4 * c);
                    l5[4 * c + 1] = scl_g(x.y, z.y, c5, 4 * c + 1);
                    l5[4 * c + 2] = scl_g(x.z, z.z, c5, 4 * c + 2);
                    l5[4 * c + 3] = scl_g(x.w, z.w, c5, 4 * c + 3);
                } else {
                    l5[4 * c] = xmin(x.x, z.x);
                    l5[4 * c + 1] = xmin(x.y, z.y);
                    l5[4 * c + 2] = xmin(x.z, z.z);
                    l5[4 * c + 3] = xmin(x.w, z.w);
                }
            }
            if (fw == 0u) {
                if (leaf_all_hard(sg, l5, pm, act, L, v5))
                    r = 32;
                else
                    failed = 0;
            }
            if (r == 0) {
                if (lane < L) {
                    float* row = S.stage + lane * kSclStage;
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *reinterpret_cast<float4*>(row + scl_chunk(lane, c)) =
                            make_float4(l5[4 * c], l5[4 * c + 1], l5[4 * c + 2], l5[4 * c + 3]);
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) lf.l4[j] = xmin(l5[j], l5[j + 16]);
                __syncwarp();
            }
        }
#pragma unroll 1
        while (r < 32) {
            uint32_t v = 0u;
            int k = 5;  // level of the node decided by this step; 5: none yet
            if ((r & 15) == 0) {
                if (r != 0) {
                    const float* row = S.stage + lf.row * kSclStage;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const float4 x = *reinterpret_cast<const float4*>(row + scl_chunk(lf.row, c));
                        const float4 z = *reinterpret_cast<const float4*>(row + scl_chunk(lf.row, c + 4));
                        lf.l4[4 * c] = scl_g(x.x, z.x, lf.c[4], 4 * c);
                        lf.l4[4 * c + 1] = scl_g(x.y, z.y, lf.c[4], 4 * c + 1);
                        lf.l4[4 * c + 2] = scl_g(x.z, z.z, lf.c[4], 4 * c + 2);
                        lf.l4[4 * c + 3] = scl_g(x.w, z.w, lf.c[4], 4 * c + 3);
                    }
                }
                const uint32_t f = (fw >> r) & 0xffffu;
                if (f == 0xffffu) {
                    leaf_frozen(lf.l4, pm);
                    k = 4;
                } else if (f == 0u && failed != r) {
                    if (leaf_all_hard(sg, lf.l4, pm, act, L, v)) k = 4;
                    else failed = r;
                }
            }
            if (k == 5 && (r & 7) == 0) {
                if (r & 8)
                    leaf_g<8>(lf.l4, lf.l3, lf.c[3]);
                else
                    leaf_f<8>(lf.l4, lf.l3);
                const uint32_t f = (fw >> r) & 0xffu;
                if (f == 0xffu) {
                    leaf_frozen(lf.l3, pm);
                    k = 3;
                } else if (f == 0u && failed != r) {
                    if (leaf_all_hard(sg, lf.l3, pm, act, L, v)) k = 3;
                    else failed = r;
                }
            }
            if (k == 5) {
                if (r & 4)
                    leaf_g<4>(lf.l3, lf.l2, lf.c[2]);
                else
                    leaf_f<4>(lf.l3, lf.l2);
                const uint32_t f = (fw >> r) & 0xfu;
                k = 2;
                bool whole = false;
                if (f == 0xfu) {
                    leaf_frozen(lf.l2, pm);
                    whole = true;
                } else if (f == 0u && failed != r) {
                    whole = leaf_all_hard(sg, lf.l2, pm, act, L, v);
                    if (!whole) failed = r;
                }
                if (!whole) {
                    int q = r;
                    if ((f & 3u) == 3u) {
                        // two or three frozen bits first: their metrics in one run
                        leaf_f<2>(lf.l2, lf.l1);
                        pm = __fsub_rn(pm, fminf(xmin(lf.l1[0], lf.l1[1]), 0.0f));
                        pm = __fsub_rn(pm, fminf(__fadd_rn(lf.l1[1], lf.l1[0]), 0.0f));
                        lf.c[0] = lf.c[1] = 0u;
                        q = r + 2;
                        if (f & 4u) {
                            lf.l1[0] = __fadd_rn(lf.l2[2], lf.l2[0]);
                            lf.l1[1] = __fadd_rn(lf.l2[3], lf.l2[1]);
                            pm = __fsub_rn(pm, fminf(xmin(lf.l1[0], lf.l1[1]), 0.0f));
                            q = r + 3;
                        }
                    }
                    // bit by bit
#pragma unroll 1
                    for (; q < r + 4; ++q) {
                        float lam;
                        if (q & 1) {
                            lam = scl_g(lf.l1[0], lf.l1[1], lf.c[0], 0);
                        } else {
                            if (q & 2)
                                leaf_g<2>(lf.l2, lf.l1, lf.c[1]);
                            else
                                leaf_f<2>(lf.l2, lf.l1);
                            lam = xmin(lf.l1[0], lf.l1[1]);
                        }
                        uint32_t bitv = 0u;
                        if ((fw >> q) & 1u) {
                            pm = __fsub_rn(pm, fminf(lam, 0.0f));
                        } else if ((dw >> q) & 1u) {
                            // decision aiding: each path takes its hard decision, no branching, no metric
                            bitv = lam < 0.0f ? 1u : 0u;
                        } else {
                            bool dup = false, moved = false;
                            int parent;
                            if constexpr (W == 32)
                                parent = scl_list_step<TWO>(lam, pm, act, L, selc, failed == q, bitv, dup, moved);
                            else
                                parent = scl_list_step_half(lam, pm, act, L, selc, failed == q, bitv, dup, moved);
                            if (moved) {
                                const int src = sg.base + parent;
                                if (!(q & 8)) leaf_copy<16>(lf.l4, src);
                                if (!(q & 4)) leaf_copy<8>(lf.l3, src);
                                if (!(q & 2)) leaf_copy<4>(lf.l2, src);
                                if (!(q & 1)) leaf_copy<2>(lf.l1, src);
#pragma unroll
                                for (int i = 0; i < 5; ++i)
                                    if (q & (1 << i)) lf.c[i] = __shfl_sync(0xffffffffu, lf.c[i], src);
                                lf.row = __shfl_sync(0xffffffffu, lf.row, src);
                                pA[0] = __shfl_sync(0xffffffffu, pA[0], src);
                                pA[1] = __shfl_sync(0xffffffffu, pA[1], src);
                                pC[0] = __shfl_sync(0xffffffffu, pC[0], src);
                                pC[1] = __shfl_sync(0xffffffffu, pC[1], src);
                            }
                            if (dup) shA = shC = 0xffffffffu;
                        }
                        // partial sums of levels 0..1; the last bit completes the node's codeword
                        if (!(q & 1)) {
                            lf.c[0] = bitv;
                        } else {
                            const uint32_t v1 = (bitv ^ lf.c[0]) | (bitv << 1);
                            if (q & 2)
                                v = (v1 ^ lf.c[1]) | (v1 << 2);
                            else
                                lf.c[1] = v1;
                        }
                    }
                }
            }
            // the node of 2^k bits at r has codeword v: fold it into its ancestors
            const int r0 = r;
            r += 1 << k;
            if (k == 2) {
                if (r0 & 4) {
                    v = (v ^ lf.c[2]) | (v << 4);
                    k = 3;
                } else {
                    lf.c[2] = v;
                }
            }
            if (k == 3) {
                if (r0 & 8) {
                    v = (v ^ lf.c[3]) | (v << 8);
                    k = 4;
                } else {
                    lf.c[3] = v;
                }
            }
            if (k == 4) {
                if (r0 & 16)
                    v5 = (v ^ lf.c[4]) | (v << 16);
                else
                    lf.c[4] = v;
            }
        }
        // ------------------------------------------------ block complete: partial sums upward
        {
            const int i_last = blk * 32 + 31;
            const int kc = __ffs(~i_last) - 1;  // >= 5; n after the last block
            if (__any_sync(0xffffffffu, (shC >> kc) & 1u)) {
                scl_own<W>(pC, kc, act, L);
                shC &= ~(1u << kc);
            }
            uint32_t* dstl = S.Cl(kc);
            const int cwk = scl_cs(kc);
            if (lane < act) dstl[fld(pC, kc) * cwk] = v5;
            __syncwarp();
            const uint32_t my_dst = fld(pC, kc);
            const int act_both2 = sg.both_max(act);
            for (int k = 5; k < kc; ++k) {
                const int Wk = 1 << (k - 5), total = act * Wk, tmax = act_both2 * Wk;
                const uint32_t* ckb = S.Cl(k);
                const uint32_t my_k = fld(pC, k);
                if constexpr (W == 32) {
                    // four elements per lane and round, loads first and unconditional (an element
                    // past the list reads a word of a valid array), stores predicated
                    constexpr int UC = 4;
                    for (int e0 = 0; e0 < tmax; e0 += UC * W) {
                        uint32_t xv[UC], cv[UC], pdv[UC];
#pragma unroll
                        for (int q = 0; q < UC; ++q) {
                            const int e = e0 + W * q + lane;
                            const int p = (e >> (k - 5)) & (W - 1);
                            const int w = e & (Wk - 1);
                            pdv[q] = sg.shfl(my_dst, p);
                            xv[q] = dstl[pdv[q] * cwk + w];
                            cv[q] = ckb[sg.shfl(my_k, p) * scl_cs(k) + w];
                        }
#pragma unroll
                        for (int q = 0; q < UC; ++q) {
                            const int e = e0 + W * q + lane;
                            if (e < total) {
                                uint32_t* dst = dstl + pdv[q] * cwk;
                                const int w = e & (Wk - 1);
                                dst[Wk + w] = xv[q];
                                dst[w] = xv[q] ^ cv[q];
                            }
                        }
                    }
                } else {
                    // half-warp lists: one element per lane (the unrolled form measured slower
                    // with 2^16 frames, the two lists' registers)
                    for (int e0 = 0; e0 < tmax; e0 += W) {
                        const int e = e0 + lane;
                        const int p = (e >> (k - 5)) & (W - 1);
                        const uint32_t pd = sg.shfl(my_dst, p);
                        const uint32_t pk = sg.shfl(my_k, p);
                        if (e < total) {
                            const int w = e & (Wk - 1);
                            uint32_t* dst = dstl + pd * cwk;
                            const uint32_t x = dst[w];
                            dst[Wk + w] = x;
                            dst[w] = x ^ ckb[pk * scl_cs(k) + w];
                        }
                    }
                }
                __syncwarp();
            }
        }
    }
    if (!lead) return;
    // ------------------------------------------------------------------ CRC selection
    // The paths in (metric, index) order: the CRC syndrome of a path is the XOR of the syndrome columns
    // of the bits of its codeword x (its level-n array) that are 1, four columns per lane and load.  The
    // first path whose syndrome is zero is output, the best one if none is; only its codeword is turned
    // into u = x G.  On most frames that is one path's work, against a column load and XOR per path and
    // bit, and a shuffle per list step, for syndromes kept along the way.  But a frame that fails tries
    // every path, and a launch of few frames waits for it: with a transform per path and a shuffle
    // search for the best, list of 32, 1200 frames: N = 128 74.4 -> 63.1 us, 256 115 -> 99, 512 224 -> 207.
    const int words = N >> 5;
    uint32_t* xl = S.Cl(n);
    const uint32_t my_x = fld(pC, n);
    uint32_t* uw = nullptr;  // u of the output path
    bool avail = lane < act, done = act == 0, any_ok = false;
    __syncwarp();
#pragma unroll 1
    while (__any_sync(0xffffffffu, !done)) {
        const uint32_t key = avail ? __float_as_uint(pm) : 0xffffffffu;  // metrics are >= 0: ordered as integers
        const int who = __ffs(sg.ballot(key == sg.red_min(key))) - 1;
        uint32_t* xw = xl + sg.shfl(my_x, who) * scl_cs(n);
        uint32_t syn = 0u;
        const bool on = !done;
        if (on) {
#pragma unroll 4
            for (int i = lane; i < N >> 2; i += W) {
                const uint4 col = *reinterpret_cast<const uint4*>(C.xsyn + 4 * i);
                const uint32_t x = xw[i >> 3] >> (4 * (i & 7));
                syn ^= ((x & 1u) ? col.x : 0u) ^ ((x & 2u) ? col.y : 0u) ^ ((x & 4u) ? col.z : 0u) ^
                       ((x & 8u) ? col.w : 0u);
            }
        }
        syn = sg.red_xor(syn);
        if (on) {
            any_ok = syn == 0u;
            if (!uw || any_ok) uw = xw;
            if (lane == who) avail = false;
        }
        const bool none_left = sg.ballot(avail) == 0u;
        done = done || any_ok || none_left;
    }
    if (uw) {
        const uint32_t m[5] = {0x55555555u, 0x33333333u, 0x0F0F0F0Fu, 0x00FF00FFu, 0x0000FFFFu};
#pragma unroll 1
        for (int i = lane; i < words; i += W) {
            uint32_t x = uw[i];
#pragma unroll
            for (int e = 0; e < 5; ++e) x ^= (x >> (1 << e)) & m[e];
            uw[i] = x;
        }
    }
#pragma unroll 1
    for (int D = 1; D < words; D <<= 1) {
        __syncwarp();
        if (uw) {
#pragma unroll 1
            for (int i = lane; i < words >> 1; i += W) {  // word pair (j, j + D), bit log2 D of j clear
                const int j = ((i & ~(D - 1)) << 1) | (i & (D - 1));
                uw[j] ^= uw[j + D];
            }
        }
    }
    __syncwarp();
    if (frame >= 0) {
        uint8_t* out = a.bits + (size_t)frame * a.row_bytes;
        for (int by = lane; by < a.row_bytes; by += W) {
            uint32_t v = 0u;
            for (int r = 0; r < 8; ++r) {
                const int p = by * 8 + r;
                if (p >= C.P) break;
                const int j = C.info_idx[p];
                v |= ((uw[j >> 5] >> (j & 31)) & 1u) << r;
            }
            out[by] = (uint8_t)v;
        }
        if (lane == 0) a.status[frame] = any_ok ? POLAR_FRAME_SCL_OK : POLAR_FRAME_SCL_CRC_FAIL;
    }
    __syncwarp();
}

// Decode `frame` (frame < 0: nothing, on this lane's list) by the calling warp with code `code_id`
// of a mixed batch (-1: the batch's single code): plan of the code, the list's shared words `ws`
// and global slot `slot` (null: every level in shared memory).  A list without a frame still walks
// the code's structure with no path, so both lists of a warp must be given the same code.
template <bool TWO, int W>
__device__ __forceinline__ void scl_warp_frame(const SCLArgs& a, int frame, int code_id, uint32_t* ws, float* slot,
                                               uint8_t* selc, uint32_t* ptab, bool mw)
{
    constexpr int LISTS = 32 / W;
    const int L = a.L;
    const DevCode& C = code_id >= 0 ? *a.codes[code_id] : *a.code;
    SCLWarp S;
    S.L = L;
    if (a.code_of) {
        const SCLPlan p = scl_plan(C.N, L, slot == nullptr, LISTS);
        S.KS = p.KS;
        S.KC = p.KC;
    } else {
        S.KS = mw ? a.KSm : a.KS;
        S.KC = mw ? a.KCm : a.KC;
    }
    // the LLR levels first: their 16-byte accesses need the list's 16-byte aligned start
    S.sA = reinterpret_cast<float*>(ws);
    S.stage = S.sA + scl_smem_llr_words(S.KS, L);
    S.sC = reinterpret_cast<uint32_t*>(S.stage + L * kSclStage);
    S.gA = slot;
    S.gC = slot ? reinterpret_cast<uint32_t*>(slot + (size_t)L * (C.N - (2 << S.KS))) : nullptr;
    scl_decode_frame<TWO, W>(a, C, frame, S, selc, ptab, mw);
}

// The frames of a launch.  W = 32: one frame per warp (mw: per CTA); W = 16: two (one per half-warp
// list), claimed together.  In a mixed batch (frames sorted by code) the two frames of a pair normally
// share their code; a pair whose codes differ is decoded one list after the other.
template <bool TWO, int W>
__device__ __forceinline__ void scl_run(const SCLArgs& a, int count, const bool mw, uint32_t* smem)
{
    constexpr int LISTS = 32 / W;
    const int lane = threadIdx.x & 31, li = lane / W;  // this lane's list
    const int wid = mw ? 0 : threadIdx.x >> 5;
    uint32_t* wsw = smem + (size_t)wid * a.warp_words;
    uint32_t* ws = wsw + li * a.list_words;
    uint32_t* scratch = wsw + (mw ? (blockDim.x >> 5) : 1) * a.warp_words - kSclWarpWords;
    uint8_t* selc = reinterpret_cast<uint8_t*>(scratch);
    uint32_t* ptab = scratch + kSclScratch;
    float* slot = a.scratch
        ? a.scratch + (((size_t)blockIdx.x * (blockDim.x >> 5) + wid) * LISTS + li) * (size_t)a.slot_words
        : nullptr;
#pragma unroll 1
    for (;;) {
        int idx = 0;
        if (mw) {
            if (threadIdx.x == 0) ptab[33] = (uint32_t)atomicAdd(a.next, 1);
            __syncthreads();
            idx = (int)ptab[33];
            __syncthreads();
        } else {
            if (lane == 0) idx = atomicAdd(a.next, LISTS);
            idx = __shfl_sync(0xffffffffu, idx, 0);
        }
        if (idx >= count) break;  // uniform over the warp (mw: the CTA)
        const int k = idx + li;
        const int frame = k < count ? (a.list ? a.list[k] : k) : -1;
        // one call site: every inlined copy of the decoder would be scheduled and allocated apart
        int code = a.code_of && frame >= 0 ? a.code_of[frame] : -1, passes = 1;
        int other = -1;
        if constexpr (LISTS == 2) {
            if (a.code_of) {
                const int c0 = __shfl_sync(0xffffffffu, code, 0), c1 = __shfl_sync(0xffffffffu, code, 16);
                passes = c0 >= 0 && c1 >= 0 && c0 != c1 ? 2 : 1;
                code = c0 >= 0 ? c0 : c1;
                other = c1;
            }
        }
#pragma unroll 1
        for (int q = 0; q < passes; ++q)
            scl_warp_frame<TWO, W>(a, passes == 1 || li == q ? frame : -1, q ? other : code, ws, slot, selc, ptab, mw);
        if (mw) __syncthreads();
    }
}

// Few frames (at most one per CTA, single code): each CTA takes one frame at a time and all its warps
// share the frame's upper-level updates, which shortens the frame's decoding latency: warp 0's list
// words, scratch and global slot serve the CTA's frame.  Short lists leave their half-warp form for it:
// a frame alone also takes the list step's shortcuts whenever its own list allows them, not only when a
// neighbour's does (37 frames of N = 1024, L = 8, of which 23 reach CA-SCL: 411 -> 353 us with BP).  More frames than CTAs fill the warps by themselves.
template <bool TWO, int W>
__global__ void __launch_bounds__(kSclWarpsPerCTA * 32, 4) scl_kernel(const SCLArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int count = a.count ? *a.count : a.B;
    const bool mw = !a.code_of && count <= (int)gridDim.x && blockDim.x >= 64;
    if constexpr (W == 16) {
        if (mw) {
            scl_run<TWO, 32>(a, count, true, smem);
            return;
        }
    }
    scl_run<TWO, W>(a, count, W == 32 && mw, smem);
}

// Persistent launch: as many CTAs as fit on the device (bounded by the global slots and, when it
// is known on the host, by the work); returns cudaSuccess or the launch error.
cudaError_t scl_launch(SCLArgs a, int N, int L, cudaStream_t st, int list_words_max, long long slot_words_max)
{
    const bool all_smem = a.scratch == nullptr;
    const int lists = scl_two_lists(L, all_smem) ? 2 : 1;
    const SCLPlan p = scl_plan(N, L, all_smem, lists);
    a.KS = p.KS;
    a.KC = p.KC;
    a.list_words = std::max(p.list_words, list_words_max);
    a.warp_words = lists * a.list_words + kSclWarpWords;
    // slots hold 16-byte vectors: each starts on a 16-byte boundary, wherever the caller's workspace
    // starts, so the same scratch bytes may give a few slots less than it was sized for
    const long long slot_words = std::max(p.slot_words, slot_words_max);
    a.slot_words = (slot_words + 3) / 4 * 4;
    long long slots = (long long)scl_sm_count() * kSclWarpsPerSM;
    if (!all_smem && slot_words > 0) {
        const long long skip = (long long)((16 - (reinterpret_cast<uintptr_t>(a.scratch) & 15)) & 15) / 4;
        a.scratch += skip;
        slots = (slots * slot_words - skip) / a.slot_words;
    }
    int W = kSclWarpsPerCTA;
    const size_t wb = (size_t)a.warp_words * 4;
    while (W > 1 && (size_t)W * wb > 200 * 1024) W >>= 1;
    const size_t smem = (size_t)W * wb;
    a.KSm = a.KS;
    a.KCm = a.KC;
    if (!all_smem) scl_plan_cta(N, L, (long long)W * a.warp_words - kSclWarpWords, &a.KSm, &a.KCm);
    const bool two = L > 16;
    const void* fn = lists == 2 ? (const void*)scl_kernel<false, 16>
                                : (two ? (const void*)scl_kernel<true, 32> : (const void*)scl_kernel<false, 32>);
    cudaError_t e = raise_smem_limit(fn, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, W * 32, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int sms = scl_sm_count();
    long long grid = (long long)sms * per_sm;
    if (!all_smem) grid = std::min<long long>(grid, slots / (W * lists));
    if (!a.list) {
        // known work: at most one frame per CTA of the full grid gets a CTA per frame (its warps then
        // share each frame's upper levels), otherwise no idle CTAs
        const long long need = (a.B + W * lists - 1) / (W * lists);
        grid = (W > 1 && !a.code_of && a.B <= grid) ? std::max(a.B, 1) : std::min(grid, need);
    }
    if (grid < 1) grid = 1;
    if (lists == 2)
        scl_kernel<false, 16><<<(unsigned)grid, W * 32, smem, st>>>(a);
    else if (two)
        scl_kernel<true, 32><<<(unsigned)grid, W * 32, smem, st>>>(a);
    else
        scl_kernel<false, 32><<<(unsigned)grid, W * 32, smem, st>>>(a);
    return cudaGetLastError();
}

#endif  // POLAR_SCL_KERNELS

}  // namespace polar
