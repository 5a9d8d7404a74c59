// Steps K4 and K5: byte-level BPE per piece, token counts and scatter of the IDs.
//
// Paper Sec. 4.2: every piece is encoded independently; merge ranks and vocabulary entries live in
// GPU hash tables; a round's minimum rank identifies one pair value, merging all its leftmost
// non-overlapping occurrences equals iterated single merges, and only pairs next to a completed
// merge need to be probed again.  Work is dispatched by piece length and difficulty:
//   * the first kernel (k_pretok, fused) has looked every piece up as a whole vocabulary entry (one sector, at times two) and
//     left the others in its tile's queue region by length class;
//   * k_merge (a request) / k_closing + k_merge_bulk (bulk text): a warp per piece (<= 32 bytes: tokens in registers,
//     candidates as ballot masks; <= 256 bytes: several tokens per lane, compaction through shared memory), or, where
//     the call has many pieces of <= 32 bytes, up to 32 of them at once, a thread per piece (lane_merge); a longer piece is
//     merged as runs of bytes if it has few, else cut into windows of 256 bytes, a warp each, that are joined at
//     shared tokens (see "long pieces"); where windows do not meet, the piece is merged whole by a CTA of 768 threads
//     (cta_merge_long: state in shared memory, or in global scratch while it still has more than 14,336 tokens).
// Token ids inside the kernels are "internal": byte b -> b, result of the merge of rank r -> 256 + r;
// the caller's ids are looked up when the tokens are staged.
//
// Rounds merge more than the minimum rank.  The sequential algorithm (always the leftmost pair of the lowest
// rank) performs a fixed set of merges on a piece; a round may perform any of them early, because the set, not
// the order, fixes the result.  A pair (t[i], t[i+1]) of rank r is certain to be in that set when neither token
// can be taken by another merge before rank r comes up:
//   * t[i] can only be taken from the left by a merge (X, t[i]) whose left operand X ends with the present
//     token t[i-1] (X is t[i-1] itself or was built on top of it).  cl(u, t) is the lowest rank of any
//     vocabulary merge (X, t) with u on the right spine of X's merge tree; the left guard is r < cl(t[i-1], t[i]);
//   * t[i+1] can only be taken from the right by a merge (t[i+1], Y) whose right operand begins with t[i+2].
//     cr(t, w) is the lowest rank of any merge (t, Y) with w on the left spine of Y; the right guard is
//     r <= cr(t[i+1], t[i+2]) (at equal rank the pair on the left comes first).
// Both guards are static properties of the vocabulary and are stored with the pair's rank, so one probe
// returns (rank, cl, cr) for a pair of adjacent tokens.  The pairs of the round's minimum rank need no guard
// (nothing can come before them).  In a run of identical pairs (t t t t ...) every other pair from a selected
// first one is selected, as in the sequential left-to-right order.  Everything selected in a round is merged
// at once; the result is the sequential one.
#pragma once
#include "tt_common.cuh"

// ---- pair table: (left, right) -> (rank, cl, cr) ----------------------------------------------------------
// Two-choice (cuckoo) hashing over buckets of two 16-byte slots (one 32-byte sector): a key is in one of its
// two buckets or nowhere, so a probe is two independent sector loads and no chain to walk, hit or miss.
// slot = { (left << 38) | (right << 20) | rank20, cl, cr } with rank20 = 0xFFFFF for a pair that is no merge
// itself (it is in the table for its guards).  A free slot is all ones.  The top bit of a bucket's first slot's second word is zero
// where no key with this first bucket had to go to its second one: who can wait for the first bucket need not look there.
struct PairInfo { u32 r, cl, cr; };                   // TT_RANK_INF where there is none
struct PairTable {
    const uint4* slots;   // 2 * (mask + 1) slots
    const u64* bytepair;  // (byte a, byte b) at [a << 8 | b]: rank20 | cl20 << 20 | cr20 << 40 (0xFFFFF = none): a piece's first probes
    u32 mask;             // number of buckets - 1 (power of two, >= 256)
    u32 shift;            // 32 - log2(number of buckets)
};
constexpr u32 TT_F20 = 0xFFFFFu;                      // 20-bit field: none
TT_HD u32 f20_decode(u32 f) { return f == TT_F20 ? TT_RANK_INF : f; }
TT_HD u32 f20_encode(u32 r) { return r < TT_F20 ? r : TT_F20; }
TT_HD u32 pair_bucket(u64 key, u32 shift) {
    const u32 x = ((u32)key ^ ((u32)(key >> 32) * 0x9E3779B1u)) * 0x85EBCA6Bu;
    return (x ^ (x >> 15)) * 0xC2B2AE35u >> shift;
}
TT_HD u32 pair_bucket_alt(u64 key, u32 shift, u32 first) {      // the key's other bucket, never the first one
    u32 x = ((u32)(key >> TT_ID_BITS) * 0xCC9E2D51u) ^ ((u32)key * 0x1B873593u);
    x ^= x >> 16; x *= 0x7FEB352Du; x ^= x >> 15;
    const u32 h = (x * 0x846CA68Bu) >> shift;
    return h == first ? (first ^ 1u) : h;
}

__device__ __forceinline__ PairInfo pair_none() { PairInfo p; p.r = p.cl = p.cr = TT_RANK_INF; return p; }
constexpr u32 PAIR_HI = 0x00FFFFFFu, PAIR_OVERFLOW = 0x80000000u;      // second word of a slot: the key's upper 24 bits; of a bucket's first slot: see above
// A slot's first word holds the key's low 12 bits over the rank: where key and slot agree, their difference is the rank.  (A free slot
// reads as the pair of the two highest ids, which is no merge and has no guards.)
__device__ __forceinline__ bool pair_match(const uint4 s, u32 hi, u32 lo, PairInfo& out) {
    const u32 r = s.x ^ lo;
    if (((s.y ^ hi) & PAIR_HI) != 0 || r > TT_F20) return false;
    out.r = f20_decode(r); out.cl = s.z; out.cr = s.w;
    return true;
}

__device__ __forceinline__ PairInfo pair_probe(const PairTable& t, u32 a, u32 b) {
    const u64 key = ((u64)a << TT_ID_BITS) | b;
    const u32 h0 = pair_bucket(key, t.shift), h1 = pair_bucket_alt(key, t.shift, h0);
    const uint4* b0 = t.slots + 2 * (size_t)h0;
    const uint4* b1 = t.slots + 2 * (size_t)h1;
    uint4 x0, y0, x1, y1;
    ldg_sector(b0, x0, y0); ldg_sector(b1, x1, y1);
    PairInfo out = pair_none();
    const u32 hi = (u32)(key >> 12), lo = (u32)key << 20;
    if (!pair_match(x0, hi, lo, out) && !pair_match(y0, hi, lo, out) && !pair_match(x1, hi, lo, out)) pair_match(y1, hi, lo, out);
    return out;
}
__device__ __forceinline__ PairInfo bytepair_info(const PairTable& t, u32 a, u32 b) {
    const u64 x = __ldg(t.bytepair + ((a << 8) | b));
    PairInfo p;
    p.r = f20_decode((u32)x & TT_F20); p.cl = f20_decode((u32)(x >> 20) & TT_F20); p.cr = f20_decode((u32)(x >> 40) & TT_F20);
    return p;
}

// Asks for [p, p + bytes) to be brought into L2, spread over the whole grid (no result, nothing waits for it).
// Used by a kernel while it waits for its predecessor: the tables it is about to probe at random are fetched
// with idle bandwidth, so that after a cold start its dependent loads find them in L2.  A grid that would have to issue
// more than two lines per thread leaves it: so small a text probes a few hundred slots of a table of tens of thousands
// of lines, and walking the table took longer than the whole call (2 KB of text with a 16 MB table: 75 us of 90).
__device__ __forceinline__ void grid_prefetch_l2(const void* p, size_t bytes) {
    const char* c = reinterpret_cast<const char*>(p);
    const size_t lines = (bytes + 127) / 128, stride = (size_t)gridDim.x * blockDim.x;
    if (lines > 2 * stride) return;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < lines; i += stride)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(c + i * 128));
}

// ---- whole-piece table: byte string of a vocabulary entry -> its id ------------------------------------
// Holds the single bytes and every token of at most TT_TOKTAB_MAXLEN bytes whose own byte string encodes to exactly that
// token (checked at load time by running the merge kernel below on every token string), so a hit
// returns what the merge loop would return.  Two tables, both two-choice (cuckoo) hashed over 32-byte buckets (one
// sector): entries of 1..8 bytes -- most pieces of ordinary text -- two 16-byte slots (length, the caller's id, two key words,
// little endian, zero padded) to a bucket; entries of 9..24 bytes one slot with six key words.  A key is in its first
// bucket, or, where that bucket's overflow bit is set, perhaps in its second one, so a look-up is one sector load and at
// times another.  (Linear probing in one table of 32-byte slots: a miss walked to the next empty slot, the longest walk of
// a warp's 32 was 5 to 8 dependent loads, and the first kernel spent 2 to 7 us of a request's 12 to 16 there.)
constexpr int TT_TOKTAB_MAXLEN = 24;
constexpr u32 TT_TOKTAB_SHORT = 8;
constexpr u32 TOK_OVERFLOW = 0x80000000u, TOK_LEN = 0xFFu;        // word 0 of a bucket's first slot
struct TokSlot { u32 len; int32_t id; u32 k[6]; };
static_assert(sizeof(TokSlot) == 32, "slot layout");
struct TokTable {
    const uint4* shorts;      // 2 << (32 - short_shift) slots, then the longer entries; nullptr: no table
    const TokSlot* slots;     // 1 << (32 - shift) of them
    u32 short_shift, shift;
    u32 mul[6];               // multipliers of the key words (odd)
    size_t bytes;             // of both, from `shorts` on
};

// Key words beyond the piece are zero, so they add nothing: a piece of at most 8 bytes is hashed from two words.
// The multipliers belong to the table: entries that collide under some (equal sums share both buckets) part under others.
TT_HD u32 toktab_hash_short(const TokTable& tab, u32 k0, u32 k1, u32 n) { return n * 0x9E3779B1u + k0 * tab.mul[0] + k1 * tab.mul[1]; }
TT_HD u32 toktab_hash_rest(const TokTable& tab, u32 h, u32 k2, u32 k3, u32 k4, u32 k5) { return h + k2 * tab.mul[2] + k3 * tab.mul[3] + k4 * tab.mul[4] + k5 * tab.mul[5]; }
TT_HD u32 toktab_hash_final(u32 h) { h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; return h ^ (h >> 15); }
TT_HD u32 toktab_bucket(u32 h, u32 shift) { return h >> shift; }
TT_HD u32 toktab_bucket_alt(u32 h, u32 shift) {                   // the key's other bucket, never the first one
    const u32 b = (h * 0x9E3779B1u) >> shift, a = h >> shift;
    return b == a ? (a ^ 1u) : b;
}
TT_HD u32 toktab_mask_word(u32 w, u32 n, u32 j) {      // key word j of a piece of n bytes: bytes beyond the piece are zero
    const u32 have = n > 4 * j ? n - 4 * j : 0u;
#if defined(__CUDA_ARCH__)
    u32 m;
    asm("bmsk.clamp.b32 %0, 0, %1;" : "=r"(m) : "r"(8 * have));       // the low 8 * have bits, at most all 32
    return w & m;
#endif
    return have >= 4 ? w : have == 0 ? 0u : w & ((1u << (8 * have)) - 1u);
}

#if defined(__CUDACC__)
// Key words 0 and 1 of the piece of n >= 1 bytes at text + a, from the aligned words x0, x1, x2 that hold it
// (x1 / x2 only where the piece reaches them).
__device__ __forceinline__ void toktab_key01(u32 x0, u32 x1, u32 x2, u32 sb, u32 n, u32& k0, u32& k1) {
    const u32 sh = sb * 8;
    k0 = toktab_mask_word(__funnelshift_r(x0, x1, sh), n, 0);
    k1 = toktab_mask_word(__funnelshift_r(x1, x2, sh), n, 1);
}
// A piece of 1..8 bytes, the two slots of its first bucket at hand; h: its hash.
__device__ __forceinline__ bool toktab_short_match(const uint4 s, u32 n, u32 k0, u32 k1, u32& val) {
    if ((((s.x ^ n) & TOK_LEN) | (s.z ^ k0) | (s.w ^ k1)) != 0) return false;
    val = s.y;
    return true;
}
__device__ __forceinline__ bool toktab_short(const TokTable& tab, const uint4 e0, const uint4 e1, u32 h, u32 n, u32 k0, u32 k1, u32& val) {
    if (toktab_short_match(e0, n, k0, k1, val) || toktab_short_match(e1, n, k0, k1, val)) return true;
    if (!(e0.x & TOK_OVERFLOW)) return false;
    const uint4* const b = tab.shorts + 2 * (size_t)toktab_bucket_alt(h, tab.short_shift);
    uint4 f0, f1;
    ldg_sector(b, f0, f1);
    return toktab_short_match(f0, n, k0, k1, val) || toktab_short_match(f1, n, k0, k1, val);
}
// Looks a piece of 1..24 bytes up; returns true and the id on a hit.  (The first kernel has its own copy of the
// first steps for pieces of at most 8 bytes, four pieces in flight per thread.)
__device__ __forceinline__ bool toktab_lookup(const TokTable& tab, const u8* __restrict__ text, u32 a, u32 n, int32_t& id) {
    const uintptr_t addr = (uintptr_t)(text + a);
    const u32* w = reinterpret_cast<const u32*>(addr & ~(uintptr_t)3);
    const u32 sb = (u32)(addr & 3), sh = sb * 8, used = sb + n;           // bytes of the aligned window that hold the piece
    u32 x[7];
#pragma unroll
    for (int j = 0; j < 7; j++) x[j] = used > 4u * j ? w[j] : 0u;          // only words that hold a piece byte (plain loads: the first kernel may have written the text itself)
    u32 k[6];
#pragma unroll
    for (int j = 0; j < 6; j++) k[j] = toktab_mask_word(__funnelshift_r(x[j], x[j + 1], sh), n, j);
    const u32 s = toktab_hash_short(tab, k[0], k[1], n);
    if (n <= TT_TOKTAB_SHORT) {
        const u32 h = toktab_hash_final(s);
        const uint4* const b = tab.shorts + 2 * (size_t)toktab_bucket(h, tab.short_shift);
        u32 val = 0;
        uint4 e0, e1;
        ldg_sector(b, e0, e1);
        const bool hit = toktab_short(tab, e0, e1, h, n, k[0], k[1], val);
        id = (int32_t)val;
        return hit;
    }
    const u32 h = toktab_hash_final(toktab_hash_rest(tab, s, k[2], k[3], k[4], k[5]));
    u32 at = toktab_bucket(h, tab.shift);
#pragma unroll 1
    for (int probe = 0; probe < 2; probe++) {
        uint4 lo, hi;
        ldg_sector(reinterpret_cast<const uint4*>(tab.slots + at), lo, hi);
        if ((((lo.x ^ n) & TOK_LEN) | (lo.z ^ k[0]) | (lo.w ^ k[1]) | (hi.x ^ k[2]) | (hi.y ^ k[3]) | (hi.z ^ k[4]) | (hi.w ^ k[5])) == 0) { id = (int32_t)lo.y; return true; }
        if (!(lo.x & TOK_OVERFLOW)) return false;
        at = toktab_bucket_alt(h, tab.shift);
    }
    return false;
}
#endif

// ---- long-entry table (ignore_merges only): vocabulary entries of more than TT_TOKTAB_MAXLEN bytes --------
// Slot = (64-bit hash of the bytes, offset into a byte blob, length, id); open addressing, load <= 0.5.  A hit
// needs equal hash, equal length and equal bytes.
struct LongSlot { u64 hash; u32 off; u32 len; int32_t id; u32 pad; };
static_assert(sizeof(LongSlot) == 24, "slot layout");
struct LongTable { const LongSlot* slots; const u8* blob; u32 mask; u32 maxlen; };   // slots == nullptr: none

TT_HD u64 longtab_hash(const u8* p, u32 n) {
    u64 h = 0xCBF29CE484222325ull ^ n;
    for (u32 i = 0; i < n; i++) { h ^= p[i]; h *= 0x100000001B3ull; }
    h ^= h >> 32;
    return h * 0x9E3779B97F4A7C15ull;
}
__device__ __forceinline__ bool longtab_lookup(const LongTable& tab, const u8* __restrict__ text, u32 a, u32 n, int32_t& id) {
    const u64 h = longtab_hash(text + a, n);
    u32 s = (u32)(h >> 32) & tab.mask;
    for (u32 probe = 0; probe <= tab.mask; probe++) {             // bounded by the capacity
        const LongSlot e = tab.slots[s];
        if (e.len == 0) return false;
        if (e.hash == h && e.len == n) {
            u32 k = 0;
            while (k < n && tab.blob[e.off + k] == text[a + k]) k++;
            if (k == n) { id = e.id; return true; }
        }
        s = (s + 1) & tab.mask;
    }
    return false;
}

// Internal token -> the caller's id.  Where the ids are the internal ones plus a constant (bytes in order first, results in order of
// rank) no table is read: 1M chars of Thai-like text 84.0 us, with the table 85.6; 1M of transcripts 32.9 and 33.1.  Vocabularies
// that permute the bytes, as GPT-2's do, take the table.  (The constant for the results and the table for the bytes only: no
// faster than the table for those, and 1 to 3 % slower for the others.)
struct ExtMap {
    const int32_t* id; int32_t delta; bool plain;
    __device__ __forceinline__ int32_t operator[](u32 t) const { return plain ? (int32_t)t + delta : id[t]; }
};
constexpr u32 RK_STALE = 0xFFFFFFFEu;                 // rank must be probed again
constexpr int BPE_WARPS = 8;                          // warps per CTA of the piece kernels
constexpr int BPE_THREADS = BPE_WARPS * 32;           // = pieces per CTA iteration
constexpr int WCH = TT_WARP_PIECE_MAX / 32;           // 32-token chunks per piece

// ---- warp merge rounds with at most 32 tokens: one token per lane, no shared memory -----------------------
// t = token of position `lane`, p = (rank, cl, cr) of the pair (lane, lane + 1) or none, m = token count.
// The tokens stay in their lanes: a mask says which lanes still hold one, and neighbours are found by bit searches.  (Moving
// the survivors together after every round -- a bit selection and four shuffles between the selection and the next
// probe -- made a round 1,200 cycles, two thirds of them the probe's.)
// Runs rounds to the fixpoint, hands token j of the result to out(j, token) and returns their count.
// A round: Q marks a pair identical to the pair on its left (t t t); a pair that is not Q heads a run; a head
// may go if its left guard holds or it has the round's minimum rank; a pair goes if its run's head may go, it
// lies an even number of places behind the head and its right guard holds (or it has the minimum rank).
template <class Out>
__device__ __forceinline__ u32 warp_merge_reg_rounds(u32 t, PairInfo p, u32 m, const PairTable& tab, int lane, Out out) {
    const u32 FULL = 0xFFFFFFFFu, lt = (1u << lane) - 1, le = lt | (1u << lane), gt = ~le;
    u32 r = p.r, cl = p.cl, cr = p.cr;
    u32 al = m >= 32 ? FULL : (1u << m) - 1;                // lanes that hold a token; lane 0 always does
    u32 up = al & gt, dn = al & lt;                         // ... of them above and below this one
    int nx = __ffs(up) - 1, pv = 31 - __clz(dn);            // neighbours (-1: none)
    u32 tl = __shfl_sync(FULL, t, pv & 31), tn = __shfl_sync(FULL, t, nx & 31);
    if (!up || !((al >> lane) & 1)) r = cl = cr = TT_RANK_INF;      // the last token has no pair
    const u32 max_rounds = m;                               // every round merges at least one pair
    for (u32 round = 0; round < max_rounds; round++) {
        const u32 mn = __reduce_min_sync(FULL, r);
        if (mn == TT_RANK_INF) break;
        u32 cll = __shfl_sync(FULL, cl, pv & 31), crr = __shfl_sync(FULL, cr, nx & 31);
        if (!dn) cll = TT_RANK_INF;
        if (!up) crr = TT_RANK_INF;
        const bool R = r != TT_RANK_INF, Mn = r == mn;
        const bool Q = R && dn && tl == t && t == tn;
        const u32 qm = __ballot_sync(FULL, Q), hm = __ballot_sync(FULL, !Q && R && (r < cll || Mn));
        const u32 h = 31u - (u32)__clz(~qm & al & le);      // the head of the run (lane 0 is never Q)
        const u32 sel = __ballot_sync(FULL, R && ((hm >> h) & 1) && (__popc(al & le & (FULL << h)) & 1) && (r <= crr || Mn));
        const bool me = (sel >> lane) & 1;
        // a merge gives its lane the new token; the lane of its right token is empty from here on
        const u32 gone = __ballot_sync(FULL, dn && ((al & sel) >> (pv & 31)) & 1);
        al &= ~gone;
        up = al & gt; dn = al & lt;
        nx = __ffs(up) - 1; pv = 31 - __clz(dn);
        if (me) t = 256u + r;
        tl = __shfl_sync(FULL, t, pv & 31); tn = __shfl_sync(FULL, t, nx & 31);
        const bool have = ((al >> lane) & 1) && up;
        if (!have) r = cl = cr = TT_RANK_INF;
        else if (me || ((sel >> (nx & 31)) & 1)) { const PairInfo q = pair_probe(tab, t, tn); r = q.r; cl = q.cl; cr = q.cr; }
    }
    if ((al >> lane) & 1) out((u32)__popc(al & lt), t);
    return (u32)__popc(al);
}

// A piece of up to 32 bytes.
template <class Out>
__device__ __forceinline__ u32 warp_merge_reg(const u8* __restrict__ text, u32 a, u32 n, const PairTable& tab, int lane, Out out) {
    const u32 t = (u32)lane < n ? text[a + lane] : 0;
    const u32 tn = __shfl_down_sync(0xFFFFFFFFu, t, 1);
    const PairInfo p = ((u32)lane + 1 < n) ? bytepair_info(tab, t, tn) : pair_none();
    return warp_merge_reg_rounds(t, p, n, tab, lane, out);
}

// ---- warp merge, 33..32 E bytes: E tokens per lane, compaction through shared memory ------------------------
// Position k lives in lane k % 32, register k / 32.  Shared memory holds two copies of four arrays of 32 E
// words (token, rank, cl, cr by position).  Each round the survivors are written to their new positions in
// the other copy and read back (one warp barrier); ranks next to a merge are marked stale and probed again,
// the probed guards go to the current copy, from which the next round reads its neighbours' values.
template <int E, class Out>
__device__ __forceinline__ u32 warp_merge_perm(u32* buf /* 2 * 4 * 32 E words of this warp */, const u8* __restrict__ text,
                                               u32 a, u32 n, const PairTable& tab, int lane, Out out) {
    constexpr u32 N = 32 * E;
    const u32 FULL = 0xFFFFFFFFu, lt = (1u << lane) - 1, le = lt | (1u << lane);
    u32 t[E], r[E];
    u32 m = n;
    u32* cb = buf;                                      // current copy: tokens [0, N), ranks [N, 2N), cl [2N, 3N), cr [3N, 4N)
    u32* ob = buf + 4 * N;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < E; j++) {
        const u32 k = j * 32 + lane;
        t[j] = k < n ? text[a + k] : 0;
        cb[k] = t[j];
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < E; j++) {
        const u32 k = j * 32 + lane;
        const PairInfo p = (k + 1 < n) ? bytepair_info(tab, t[j], cb[k + 1]) : pair_none();
        r[j] = p.r; cb[2 * N + k] = p.cl; cb[3 * N + k] = p.cr;
    }
    for (u32 round = 0; round < n; round++) {          // at most n - 1 merges, at least one per round
        u32 mn = r[0];
#pragma unroll
        for (int j = 1; j < E; j++) mn = min(mn, r[j]);
        mn = __reduce_min_sync(FULL, mn);
        if (mn == TT_RANK_INF) break;
        __syncwarp();                                   // the guards written after the probes are visible
        if (m <= 32) {                                  // cheaper rounds from here on
            PairInfo p; p.r = r[0]; p.cl = cb[2 * N + lane]; p.cr = cb[3 * N + lane];
            return warp_merge_reg_rounds(t[0], p, m, tab, lane, out);
        }
        const int nch = (int)((m + 31) >> 5);
        u32 sel[E];
        u32 carry_hok = 0, carry_par = 0;               // head of the run that reaches into the word: may it go / parity of its position
#pragma unroll
        for (int j = 0; j < E; j++) {
            sel[j] = 0;
            if (j < nch) {
                const u32 k = j * 32 + lane;
                const bool R = r[j] != TT_RANK_INF, Mn = r[j] == mn;          // R implies k + 1 < m
                const u32 tl = k ? cb[k - 1] : 0xFFFFFFFFu, tn = R ? cb[k + 1] : 0xFFFFFFFEu;
                const u32 cll = k ? cb[2 * N + k - 1] : TT_RANK_INF;
                const u32 crr = (k + 2 < m) ? cb[3 * N + k + 1] : TT_RANK_INF;
                const bool Q = R && tl == t[j] && t[j] == tn;
                const u32 qm = __ballot_sync(FULL, Q), hm = __ballot_sync(FULL, !Q && R && (r[j] < cll || Mn));
                const u32 z = ~qm & le;
                u32 hok, par;
                if (z) { const u32 ph = 31u - (u32)__clz(z); hok = (hm >> ph) & 1; par = ((u32)lane - ph) & 1; }
                else { hok = carry_hok; par = ((u32)lane & 1) ^ carry_par; }
                sel[j] = __ballot_sync(FULL, R && hok && !par && (r[j] <= crr || Mn));
                if (~qm) { const u32 ph = 31u - (u32)__clz(~qm); carry_par = ph & 1; carry_hok = (hm >> ph) & 1; }
            }
        }
        u32 removed = 0;
#pragma unroll
        for (int j = 0; j < E; j++) {
            if (j < nch) {
                const u32 k = j * 32 + lane;
                const u32 s = sel[j];
                const bool me = (s >> lane) & 1;
                const bool gone = lane ? ((s >> (lane - 1)) & 1) : (j ? (sel[j > 0 ? j - 1 : 0] >> 31) & 1 : 0);
                const bool next_sel = lane < 31 ? ((s >> (lane + 1)) & 1) : ((j + 1 < E) ? (sel[j + 1 < E ? j + 1 : j] & 1) : 0);
                if (k < m && !gone) {
                    const u32 np = k - removed - __popc(s & lt);
                    ob[np] = me ? 256u + r[j] : t[j];
                    ob[N + np] = (me || next_sel) ? RK_STALE : r[j];
                    ob[2 * N + np] = cb[2 * N + k];
                    ob[3 * N + np] = cb[3 * N + k];
                }
                removed += __popc(s);
            }
        }
        m -= removed;
        { u32* x = cb; cb = ob; ob = x; }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < E; j++) {
            const u32 k = j * 32 + lane;
            r[j] = TT_RANK_INF;
            if (k < m) {
                t[j] = cb[k];
                r[j] = cb[N + k];
                if (k + 1 >= m) r[j] = TT_RANK_INF;
                else if (r[j] == RK_STALE) {
                    const PairInfo p = pair_probe(tab, t[j], cb[k + 1]);
                    r[j] = p.r; cb[2 * N + k] = p.cl; cb[3 * N + k] = p.cr;
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < E; j++) {
        const u32 k = j * 32 + lane;
        if (k < m) out(k, t[j]);
    }
    return m;
}

// ---- a thread per piece, <= 32 bytes: tokens and pair ranks in shared memory ------------------------------
// Paper Sec. 4.2 gives the shortest length class to single threads.  A warp per piece takes fewer rounds (it merges more than one pair
// a round), a thread per piece keeps 32 independent chains per warp in flight and issues an order of magnitude fewer
// instructions per piece.  A round is one merge: the leftmost pair of the lowest rank, as the definition has it.  What bounds a
// batch is the chain of a round -- minimum, neighbours, two probes side by side -- times the merges of its slowest
// piece, so the minimum is found without a dependent step per position: a pair's rank and position are one word, the words of
// four positions one 16-byte load, and places without a pair hold all ones (walking the live positions one after the other
// and merging all occurrences of the rank at once, a batch of 32 pieces took 50 to 110 us; 132 MB batch 851 -> 804, 3M chars of long
// runs 1.1 to 1.2 times as fast by text, 1,000 messages 68.5 -> 61).
constexpr int LANE_SLOTS = 32;                        // pieces a warp merges at once
constexpr int LANE_MAX = 32;                          // bytes per piece on this path
constexpr u32 LANE_NONE = 0xFFFFFFFFu;                // no pair begins here
// Two independent probes, ranks only (TT_F20 or more: none).  A slot's first word holds the key's low 12 bits over the rank: where key and
// slot agree, their difference is the rank.  ALL: all four buckets at once, the shorter chain, for a request; else a key's second
// bucket only where the first has not got it and says that it overflowed, for bulk text, whose warps saturate the way to L2 (132 MB batch:
// all at once 773 us a call, the second afterwards 740, only of those that overflowed 731; 64 documents of 100,000 characters with
// 4,096 merges 241, 225, 213.  15,000 pieces of 1,000 messages: the second bucket afterwards 60 us, all at once 55.6).
__device__ __forceinline__ u32 pair_rank_of(const uint4 s, u32 hi, u32 lo) { return ((s.y ^ hi) & PAIR_HI) == 0 ? s.x ^ lo : TT_RANK_INF; }
template <bool ALL>
__device__ __forceinline__ void pair_probe2(const PairTable& t, u64 key0, u64 key1, u32& r0, u32& r1) {
    const u32 h00 = pair_bucket(key0, t.shift), h10 = pair_bucket(key1, t.shift);
    const uint4* const p01 = t.slots + 2 * (size_t)pair_bucket_alt(key0, t.shift, h00);
    const uint4* const p11 = t.slots + 2 * (size_t)pair_bucket_alt(key1, t.shift, h10);
    const u32 hi0 = (u32)(key0 >> 12), lo0 = (u32)key0 << 20, hi1 = (u32)(key1 >> 12), lo1 = (u32)key1 << 20;
    uint4 a00, a01, a02, a03, a10, a11, a12, a13;
    ldg_sector(t.slots + 2 * (size_t)h00, a00, a01); ldg_sector(t.slots + 2 * (size_t)h10, a10, a11);
    if (ALL) { ldg_sector(p01, a02, a03); ldg_sector(p11, a12, a13); }
    r0 = min(pair_rank_of(a00, hi0, lo0), pair_rank_of(a01, hi0, lo0));
    r1 = min(pair_rank_of(a10, hi1, lo1), pair_rank_of(a11, hi1, lo1));
    if (!ALL) {
        a02 = a03 = make_uint4(~lo0, hi0, 0, 0); a12 = a13 = make_uint4(~lo1, hi1, 0, 0);             // (not this key's)
        if (r0 > TT_F20 && (a00.y & PAIR_OVERFLOW)) ldg_sector(p01, a02, a03);
        if (r1 > TT_F20 && (a10.y & PAIR_OVERFLOW)) ldg_sector(p11, a12, a13);
    }
    r0 = min(r0, min(pair_rank_of(a02, hi0, lo0), pair_rank_of(a03, hi0, lo0)));
    r1 = min(r1, min(pair_rank_of(a12, hi1, lo1), pair_rank_of(a13, hi1, lo1)));
}

// Tokens stay at the byte position where they began; `al` has a bit per position that still holds a token, and the word of a
// pair is kept at its left position, so a merge moves nothing.  tok[LANE_MAX][LANE_SLOTS], a column per thread; the
// words of positions 4j .. 4j + 3 are rk[j][thread]: any two threads of the warp find their tokens, and any eight
// neighbouring threads their four words, in different banks.
__device__ __forceinline__ u32 lane_word(u32 r20, u32 k) { return r20 >= TT_F20 ? LANE_NONE : (r20 << 5) | k; }
template <bool ALL>
__device__ __forceinline__ u32 lane_merge(u32* __restrict__ tok, int s, const u8* __restrict__ text, u32 a, u32 n,
                                          const PairTable& tab, const ExtMap& ext_id, int32_t* __restrict__ stage) {
    u32* const rk = tok + LANE_MAX * LANE_SLOTS;
#define TK(k) tok[(k) * LANE_SLOTS + s]
#define RK(k) rk[(((k) >> 2) * LANE_SLOTS + s) * 4 + ((k) & 3)]
    uint4* const rk4 = reinterpret_cast<uint4*>(rk) + s;
    const bool wide = n > 16;
    {
        const uintptr_t addr = (uintptr_t)(text + a);
        const u32* const w = reinterpret_cast<const u32*>(addr & ~(uintptr_t)3);
        const u32 sh = (u32)(addr & 3) * 8, used = (u32)(addr & 3) + n;       // bytes of the aligned words that hold the piece
        const u32* const bp = reinterpret_cast<const u32*>(tab.bytepair);     // (the rank is in the low half of an entry)
        u32 x[9];
#pragma unroll
        for (int j = 0; j < 9; j++) x[j] = used > 4u * j ? w[j] : 0u;          // only words that hold a piece byte
#pragma unroll
        for (int j = 0; j < 8; j++) {
            if (j >= 4 && !wide) break;
            const u32 v = __funnelshift_r(x[j], x[j + 1], sh), vn = j < 7 ? __funnelshift_r(x[j + 1], x[j + 2 < 9 ? j + 2 : 8], sh) : 0u;
            const u32 t0 = v & 0xFFu, t1 = (v >> 8) & 0xFFu, t2 = (v >> 16) & 0xFFu, t3 = v >> 24, t4 = vn & 0xFFu;
            const u32 k = 4 * j;
            uint4 r = make_uint4(TT_F20, TT_F20, TT_F20, TT_F20);
            if (k + 1 < n) r.x = __ldg(bp + 2 * ((t0 << 8) | t1)) & TT_F20;
            if (k + 2 < n) r.y = __ldg(bp + 2 * ((t1 << 8) | t2)) & TT_F20;
            if (k + 3 < n) r.z = __ldg(bp + 2 * ((t2 << 8) | t3)) & TT_F20;
            if (k + 4 < n) r.w = __ldg(bp + 2 * ((t3 << 8) | t4)) & TT_F20;
            rk4[j * LANE_SLOTS] = make_uint4(lane_word(r.x, k), lane_word(r.y, k + 1), lane_word(r.z, k + 2), lane_word(r.w, k + 3));
            TK(k) = t0; TK(k + 1) = t1; TK(k + 2) = t2; TK(k + 3) = t3;
        }
    }
    u32 al = 0xFFFFFFFFu >> (32 - n);
    for (u32 round = 1; round < n; round++) {             // at most n - 1 merges
        const auto min8 = [&](int j) {
            const uint4 x = rk4[j * LANE_SLOTS], y = rk4[(j + 1) * LANE_SLOTS];
            return __vimin3_u32(__vimin3_u32(x.x, x.y, x.z), __vimin3_u32(x.w, y.x, y.y), min(y.z, y.w));
        };
        u32 mn = min(min8(0), min8(2));
        if (wide) mn = __vimin3_u32(mn, min8(4), min8(6));
        if (mn == LANE_NONE) break;
        const u32 k = mn & 31u, t = 256u + (mn >> 5);
        u32 up = al & (0xFFFFFFFEu << k);                 // the tokens above; the first of them goes into the merge
        const u32 p = __ffs(up) - 1;
        up &= up - 1; al &= ~(1u << p);
        const u32 q = __ffs(up) - 1, dn = al & ((1u << k) - 1), l = 31 - __clz(dn);
        TK(k) = t;
        RK(p) = LANE_NONE;
        const u64 right = ((u64)t << TT_ID_BITS) | (up ? TK(q) : 0u), left = dn ? ((u64)TK(l) << TT_ID_BITS) | t : right;
        u32 rl, rr;
        pair_probe2<ALL>(tab, left, right, rl, rr);
        if (dn) RK(l) = lane_word(rl, l);
        RK(k) = up ? lane_word(rr, k) : LANE_NONE;
    }
    u32 m = 0;
    for (u32 x = al; x; x &= x - 1) stage[a + m++] = ext_id[TK(__ffs(x) - 1)];
#undef TK
#undef RK
    return m;
}

// ---- CTA-wide helpers ------------------------------------------------------------------------------------
__device__ __forceinline__ u32 cta_excl_sum_scan(u32 v, u32* scratch /* >= 33 */, u32* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    u32 x = v;
    for (int o = 1; o < 32; o <<= 1) { u32 t = __shfl_up_sync(0xFFFFFFFFu, x, o); if (lane >= o) x += t; }
    __syncthreads();
    if (lane == 31) scratch[wid] = x;
    __syncthreads();
    if (wid == 0) {
        u32 s = lane < nw ? scratch[lane] : 0, y = s;
        for (int o = 1; o < 32; o <<= 1) { u32 t = __shfl_up_sync(0xFFFFFFFFu, y, o); if (lane >= o) y += t; }
        if (lane < nw) scratch[lane] = y - s;
        if (lane == nw - 1) scratch[32] = y;
    }
    __syncthreads();
    *total = scratch[32];
    return scratch[wid] + x - v;
}
// Sums of two values over the CTA, returned to every thread (scratch >= 66 entries; two barriers).
__device__ __forceinline__ void cta_sum2_u64(unsigned long long& x, unsigned long long& y, unsigned long long* scratch) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    for (int o = 16; o; o >>= 1) { x += __shfl_xor_sync(0xFFFFFFFFu, x, o); y += __shfl_xor_sync(0xFFFFFFFFu, y, o); }
    __syncthreads();
    if (lane == 0) { scratch[2 * wid] = x; scratch[2 * wid + 1] = y; }
    __syncthreads();
    x = 0; y = 0;
    for (int w = 0; w < nw; w++) { x += scratch[2 * w]; y += scratch[2 * w + 1]; }
}

__device__ __forceinline__ u32 cta_min_u32(u32 v, u32* scratch /* >= 33 */) {
    v = __reduce_min_sync(0xFFFFFFFFu, v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    u32 r = scratch[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); w++) r = min(r, scratch[w]);
    return r;
}

// ---- CTA merge for long pieces -----------------------------------------------------------------------------
// arr[i] = token | rank20 << 18 | cl20 << 38 and crr[i] = cr20 for position i (rank and guards of the pair
// (i, i + 1); 20-bit fields, 0xFFFFF = none), in global scratch or shared memory.  One round: the minimum rank
// is found, every thread takes LK consecutive positions and decides which of its pairs are merged (same rule
// as in the warp rounds; the state of a run of identical pairs that crosses slices -- may its head go, parity
// of the distance to it -- is carried from thread to thread with one ballot-based scan; LK is even, so a
// slice that lies inside one run passes the state on unchanged), and the survivors are written to their new
// positions in place, chunk after chunk (every thread of a chunk has its positions in registers before
// anything is written, and writes never pass the read front).  Ranks next to a merge are marked stale and
// probed again in a second sweep, which also yields the next round's minimum.
#ifndef TT_LK
#define TT_LK 6        // measured with 768 threads: 64 KB of random letters 94 ms at 16, 59 at 8, 45 at 6, 51 at 4, 59 at 2
#endif
constexpr int LK = TT_LK;                               // positions per thread and chunk (even)
// words of the CTA's scratch array: [0, 33) block scans and per-warp run states, then per-warp "last position merged" flags,
// the carried token / guard of a chunk's last position, and two words for broadcasts
constexpr int SCR_LASTM = 40, SCR_CARRY_TOK = 72, SCR_CARRY_CL = 73, SCR_FLAG = 74, SCR_VALUE = 75, SCR_WORDS = 80;
constexpr u32 F20_STALE = 0xFFFFEu;
TT_HD u64 lp_pack(u32 t, u32 r20, u32 cl20) { return (u64)t | ((u64)r20 << TT_ID_BITS) | ((u64)cl20 << (TT_ID_BITS + 20)); }
TT_HD u32 lp_tok(u64 v) { return (u32)v & (TT_MAX_INTERNAL - 1); }
TT_HD u32 lp_rank(u64 v) { return (u32)(v >> TT_ID_BITS) & TT_F20; }
TT_HD u32 lp_cl(u64 v) { return (u32)(v >> (TT_ID_BITS + 20)) & TT_F20; }

// padshift: 4 for arrays in shared memory (index i lives at i + i / 16: the slices of LK consecutive positions that the
// threads of a warp read then spread over more banks), 31 for arrays in global scratch (no padding).
#define AX(i) ((i) + ((i) >> padshift))
__device__ __noinline__ u32 cta_merge_rounds(u64* arr, u32* crr, u32 m, const PairTable& tab, u32* s_scr /* SCR_WORDS */, u32 stop_at, bool& finished, u32 padshift,
                                           u64* stg_a = nullptr, u32* stg_c = nullptr) {
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = T >> 5;
    const u32 FULL = 0xFFFFFFFFu, inmask = (1u << LK) - 1;
    finished = false;
    // minimum rank of the current array
    u32 lmin = TT_F20;
    for (u32 i0 = tid; i0 < m; i0 += (u32)T * 8) {
        u64 xs[8];
#pragma unroll
        for (int u = 0; u < 8; u++) { const u32 i = i0 + (u32)u * T; xs[u] = i < m ? arr[AX(i)] : lp_pack(0, TT_F20, TT_F20); }
#pragma unroll
        for (int u = 0; u < 8; u++) lmin = min(lmin, lp_rank(xs[u]));
    }
    for (;;) {
        const u32 mn = cta_min_u32(lmin, s_scr);
        if (mn >= F20_STALE) { finished = true; return m; }
        if (m <= stop_at) return m;
        u32 carry_hok = 0, carry_par = 0, carry_last = 0, out = 0;    // run state and last selection before the chunk; survivors so far
        for (u32 base = 0; base < m; base += (u32)T * LK) {
            const u32 i0 = base + (u32)tid * LK;
            u64 v[LK + 3];                                  // positions i0 - 1 .. i0 + LK + 1
            u32 c[LK + 3];
#pragma unroll
            for (int k = 0; k < LK + 3; k++) {
                const u32 i = i0 + k - 1;                   // wraps for position -1 of the piece: not below m
                v[k] = lp_pack(0, TT_F20, TT_F20); c[k] = TT_F20;
                if (k == 0 && tid == 0) { if (base) v[k] = lp_pack(s_scr[SCR_CARRY_TOK], TT_F20, s_scr[SCR_CARRY_CL]); }   // overwritten by the chunk before: carried
                else if (i < m) { v[k] = arr[AX(i)]; c[k] = crr[AX(i)]; }
            }
            const u32 nval = i0 < m ? min((u32)LK, m - i0) : 0;
            u32 Qm = 0, Hm = 0, Gm = 0;                     // bit k: position i0 + k, k = 0 .. LK
#pragma unroll
            for (int k = 0; k <= LK; k++) {
                const u32 rr = lp_rank(v[k + 1]), tk = lp_tok(v[k + 1]);
                const bool R = rr < F20_STALE, Mn = rr == mn;
                const bool Q = R && (i0 + k >= 1) && lp_tok(v[k]) == tk && tk == lp_tok(v[k + 2]);
                Qm |= (u32)Q << k;
                Hm |= (u32)(!Q && R && (rr < lp_cl(v[k]) || Mn)) << k;
                Gm |= (u32)(R && (rr <= c[k + 2] || Mn)) << k;
            }
            // state handed to the next slice: from my highest pair that heads a run
            const u32 nq = ~Qm & inmask;
            const bool all = nq == 0;
            u32 out_hok = 0, out_par = 0;
            if (nq) { const u32 ph = 31u - (u32)__clz(nq); out_hok = (Hm >> ph) & 1; out_par = ((u32)LK - ph) & 1; }
            const u32 allm = __ballot_sync(FULL, all), hokm = __ballot_sync(FULL, out_hok), parm = __ballot_sync(FULL, out_par);
            const u32 lower = ~allm & ((1u << lane) - 1);
            __syncthreads();
            if (lane == 31) {
                const u32 na = ~allm;
                u32 e = 0;
                if (na) { const u32 src = 31u - (u32)__clz(na); e = 4u | (((hokm >> src) & 1) << 1) | ((parm >> src) & 1); }
                s_scr[wid] = e;                              // 0 = all lanes pass through
            }
            __syncthreads();
            u32 in_hok, in_par;
            if (lower) { const u32 src = 31u - (u32)__clz(lower); in_hok = (hokm >> src) & 1; in_par = (parm >> src) & 1; }
            else {
                in_hok = carry_hok; in_par = carry_par;
                for (int w = wid - 1; w >= 0; w--) { const u32 e = s_scr[w]; if (e) { in_hok = (e >> 1) & 1; in_par = e & 1; break; } }
            }
            u32 next_hok = carry_hok, next_par = carry_par;
            for (int w = nw - 1; w >= 0; w--) { const u32 e = s_scr[w]; if (e) { next_hok = (e >> 1) & 1; next_par = e & 1; break; } }
            // selection inside the slice (positions 0..LK; position LK only to know whether it is merged)
            u32 sel = 0;
            {
                u32 hok = in_hok, par = in_par;
#pragma unroll
                for (int k = 0; k <= LK; k++) {
                    if (!((Qm >> k) & 1)) { hok = (Hm >> k) & 1; par = 0; }
                    sel |= (((Gm >> k) & 1) & hok & (par ^ 1u)) << k;
                    par ^= 1u;
                }
            }
            // was the position before my slice merged with my first one?
            const u32 lastm = __ballot_sync(FULL, (sel >> (LK - 1)) & 1);
            if (lane == 31) s_scr[SCR_LASTM + wid] = lastm >> 31;
            if (tid == T - 1) { s_scr[SCR_CARRY_TOK] = lp_tok(v[LK]); s_scr[SCR_CARRY_CL] = lp_cl(v[LK]); }     // position i0 + LK - 1 as it is now
            __syncthreads();
            const u32 gone0 = lane ? (lastm >> (lane - 1)) & 1 : (wid ? s_scr[SCR_LASTM + wid - 1] : carry_last);
            const u32 next_last = s_scr[SCR_LASTM + nw - 1];
            const u32 gone = ((sel << 1) | gone0) & inmask;
            const u32 valid = nval >= LK ? inmask : ((1u << nval) - 1);
            const u32 surv = valid & ~gone;
            u32 tot;
            const u32 ex = cta_excl_sum_scan(__popc(surv), s_scr, &tot);         // all loads of the chunk are done: barrier inside
            // Arrays in global scratch: the chunk's survivors are collected in shared memory and written out with
            // coalesced stores (a thread storing its own run of positions touches a line per store and lane, which
            // is what a chunk spent most of its time on).
            u64* const wa = stg_a ? stg_a : arr;
            u32* const wc = stg_a ? stg_c : crr;
            u32 o = stg_a ? ex : out + ex;
#pragma unroll
            for (int k = 0; k < LK; k++) {
                if ((surv >> k) & 1) {
                    const bool me = (sel >> k) & 1;
                    const bool nxt = me ? false : ((sel >> (k + 1)) & 1);
                    const u64 x = v[k + 1];
                    const u32 oi = stg_a ? o : AX(o);
                    wa[oi] = lp_pack(me ? 256u + lp_rank(x) : lp_tok(x), (me || nxt) ? F20_STALE : lp_rank(x), lp_cl(x));
                    wc[oi] = c[k + 1];
                    o++;
                }
            }
            if (stg_a) {
                __syncthreads();
                for (u32 e = tid; e < tot; e += T) { arr[out + e] = stg_a[e]; crr[out + e] = stg_c[e]; }
            }
            out += tot;
            carry_hok = next_hok; carry_par = next_par; carry_last = next_last;
            __syncthreads();
        }
        m = out;
        __syncthreads();
        // probe the stale ranks again; collect the minimum for the next round
        // (eight loads in flight per thread: in global scratch every one of them is an L2 round trip)
        lmin = TT_F20;
        for (u32 i0 = tid; i0 < m; i0 += (u32)T * 8) {
            u64 xs[8];
#pragma unroll
            for (int u = 0; u < 8; u++) { const u32 i = i0 + (u32)u * T; xs[u] = i < m ? arr[AX(i)] : lp_pack(0, TT_F20, TT_F20); }
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const u32 i = i0 + (u32)u * T;
                const u64 x = xs[u];
                u32 r = lp_rank(x);
                if (i < m) {
                    if (i + 1 >= m) { r = TT_F20; arr[AX(i)] = lp_pack(lp_tok(x), TT_F20, TT_F20); crr[AX(i)] = TT_F20; }
                    else if (r == F20_STALE) {
                        const PairInfo p = pair_probe(tab, lp_tok(x), lp_tok(arr[AX(i + 1)]));
                        r = f20_encode(p.r);
                        arr[AX(i)] = lp_pack(lp_tok(x), r, f20_encode(p.cl)); crr[AX(i)] = f20_encode(p.cr);
                    }
                }
                lmin = min(lmin, r);
            }
        }
        __syncthreads();
    }
}

#ifndef TT_LONG_SMEM_TOKENS
#define TT_LONG_SMEM_TOKENS 14336
#endif
constexpr int LONG_SMEM_TOKENS = TT_LONG_SMEM_TOKENS;   // long pieces move into shared memory below this many tokens
constexpr int LONG_SMEM_SLOTS = LONG_SMEM_TOKENS + LONG_SMEM_TOKENS / 16 + 8;   // with the padding of the shared-memory layout; also holds a chunk's survivors


// Encodes one piece of n > TT_WARP_PIECE_MAX bytes with the whole CTA.  gbuf: n entries of global scratch; the
// piece's own n words of the staging array serve as the second global array until the ids are staged there.
// sbuf: LONG_SMEM_SLOTS u64 followed by LONG_SMEM_SLOTS u32.
__device__ u32 cta_merge_long(const u8* __restrict__ text, u32 a, u32 n, const PairTable& tab, const ExtMap& ext_id,
                              int32_t* __restrict__ stage, u64* gbuf, u64* sbuf, u32* s_scr) {
    const int tid = threadIdx.x, T = blockDim.x;
    u32* const scr = reinterpret_cast<u32*>(sbuf + LONG_SMEM_SLOTS);
    u32* const gcr = reinterpret_cast<u32*>(stage + a);
    u64* arr = n <= LONG_SMEM_TOKENS ? sbuf : gbuf;
    u32* crr = n <= LONG_SMEM_TOKENS ? scr : gcr;
    u32 padshift = n <= LONG_SMEM_TOKENS ? 4u : 31u;
    __syncthreads();
    for (u32 i = tid; i < n; i += T) {
        const u32 t0 = text[a + i];
        const PairInfo p = (i + 1 < n) ? bytepair_info(tab, t0, text[a + i + 1]) : pair_none();
        arr[AX(i)] = lp_pack(t0, f20_encode(p.r), f20_encode(p.cl));
        crr[AX(i)] = f20_encode(p.cr);
    }
    __syncthreads();
    bool finished;
    u32 m = cta_merge_rounds(arr, crr, n, tab, s_scr, arr == gbuf ? LONG_SMEM_TOKENS : 0, finished, padshift,
                             arr == gbuf ? sbuf : nullptr, arr == gbuf ? scr : nullptr);       // the shared buffer stages the stores meanwhile
    if (!finished && arr == gbuf) {
        __syncthreads();
        padshift = 4u;
        for (u32 i = tid; i < m; i += T) { sbuf[AX(i)] = gbuf[i]; scr[AX(i)] = gcr[i]; }
        __syncthreads();
        arr = sbuf;
        m = cta_merge_rounds(arr, scr, m, tab, s_scr, 0, finished, padshift);
    }
    __syncthreads();
    for (u32 i = tid; i < m; i += T) stage[a + i] = ext_id[lp_tok(arr[AX(i)])];
    __syncthreads();
    return m;
}
#undef AX

// ---- what the first kernel (tag + piece starts + whole-piece lookups) leaves per tile -----------------------
// See TTWorkspace.  A queue entry of a tile names one unsettled piece of at most 256 bytes that lies inside the
// tile: offset in the tile | index among the tile's pieces << 11 | (bytes - 1) << 22.  The tile's LAST piece is
// never settled by the first kernel (its end is the next piece start, which another CTA finds): k_merge
// settles it, looking the end up in tile_first of the following tiles.
__device__ __forceinline__ u32 tile_queue_entry(u32 off, u32 idx, u32 n) { return off | (idx << 11) | ((n - 1) << 22); }
constexpr u32 TQ_MAY_LONG = 0x80000000u;              // tile_q: the tile allows for a piece of more than 256 bytes (see k_pretok)
constexpr u32 TQ_HAS_DOC = 0x40000000u;               // tile_q, bulk text: a document starts in the tile
constexpr u32 TQ_NS_MASK = 0x7FFu, TQ_NW_SHIFT = 11, TQ_NW_MASK = 0x7Fu, TQ_NL_SHIFT = 18, TQ_NL_MASK = 0xFu;

struct PieceParams {
    const u8* base;            // aligned frame origin (text = base + shift)
    long long shift, hi;       // text occupies [shift, hi)
    int ntiles;
    const u32* tile_cnt;
    const u32* tile_first;
    const u32* tile_last;
    const u32* tile_q;
    const u16* tile_long;
    const u16* piece_off16;
    const u32* q;
    TTHeader* hdr;
    unsigned long long epoch;
    PairTable tab;
    TokTable toktab;           // shorts == nullptr: no whole-piece table (while the table itself is being built)
    const u32* litstart;       // literal pass: a piece that begins at such a bit is an added token whose id is staged, or null
    LongTable longtab;         // ignore_merges: entries longer than the whole-piece table holds (else slots == nullptr)
    ExtMap ext_id;
    u32* piece_cnt;
    int32_t* stage;            // ids staged at the text offset of their piece
    u64* pairbuf;              // global scratch of the long-piece path, indexed like the text
    u32* tile_tok;
    u32* grp_tok;              // bulk text: tokens per group of TT_GROUP_TILES tiles (written by the last CTA), else null
    u64* wq;                   // bulk text: the warp-class pieces of all tiles (tile << 32 | queue entry), else null
    u64* gq;                   // bulk text: the short pieces of all tiles, gathered by k_closing (tile << 32 | queue entry),
    u64* gq_x[3];              // one list per length class (tt_short_class_max); gq is the first
    uint4* lq;                 // long pieces (text offset, bytes, piece slot, state): of all tiles, listed by k_closing (bulk text), or those
                               // that k_merge hands to the whole grid (a request)
    const u16* tok_len;        // bytes of every internal token (65,535 = that many or more)
};

// ---- K4, second half: the merges ------------------------------------------------------------------------------
// Work of this kernel: the unsettled pieces the first kernel queued per tile, and the last piece of every tile.
// A request (k_merge): every CTA scans the tiles' counts once (merge_index), so that a warp finds any queued piece by bisection
// and nothing is handed out through a list.  Then
//   - pieces of more than 256 bytes, where a tile allows for one (cta_find_long): those of every gridDim.x-th tile by a CTA, or,
//     if one is too long for that, by tickets, its windows later by the whole grid (long_phase);
//   - everything else by warps, without a barrier: job j is warp j's, in the order warp-class pieces (the longest chains),
//     closing pieces of the tiles, short pieces; by tickets where CTAs had long pieces first.  With many short pieces these go in
//     batches, a thread each (merge_short_batches).
// Bulk text (k_merge_bulk): k_closing has gathered global lists.  Long pieces by tickets of a CTA, warp-class pieces a warp each
// by index, short pieces by tickets of up to 32 of one length class, a thread each, the longest class first.
#ifndef TT_MERGE_WARPS
#define TT_MERGE_WARPS 24
#endif
constexpr int MERGE_WARPS = TT_MERGE_WARPS;           // one CTA per SM: a long piece gets all its 768 threads and 192 KiB
constexpr int MERGE_THREADS = MERGE_WARPS * 32;
constexpr int WARP_SMEM_WORDS = 1024;                 // u64 per warp: two lane-path arrays of 32 x 32 u32, or two copies of four 256-word merge arrays
static_assert(MERGE_WARPS * WARP_SMEM_WORDS * sizeof(u64) >= LONG_SMEM_SLOTS * (sizeof(u64) + sizeof(u32)), "the CTA's buffer must hold a long piece");
static_assert(LONG_SMEM_TOKENS >= MERGE_WARPS * 32 * LK, "the survivors of a chunk (threads x LK positions) must fit the shared buffer");
constexpr size_t MERGE_SMEM_BYTES = (size_t)MERGE_WARPS * WARP_SMEM_WORDS * sizeof(u64);   // dynamic shared memory of k_merge_bulk (192 KiB)
static_assert(WARP_SMEM_WORDS * sizeof(u64) >= 2 * LANE_SLOTS * LANE_MAX * sizeof(u32) && WARP_SMEM_WORDS * sizeof(u64) >= 2 * 4 * TT_WARP_PIECE_MAX * sizeof(u32), "per-warp buffer");
// Pieces of a batch of lane_merge: as few as give BATCH_WARPS of a CTA's warps one each, up to 32.  More warps with fewer pieces each
// only issue the same instructions more often (1,000 messages: all 24 warps 60.4 us, 12 warps 55.6, 8 56.4, 5 57.0; 3M chars of long
// runs 197, 190, 200, 204).
constexpr u32 BATCH_WARPS = 12;
__device__ __forceinline__ u32 short_batch(u32 pieces) { const u32 warps = gridDim.x * BATCH_WARPS; return min((u32)LANE_SLOTS, max(1u, (pieces + warps - 1) / warps)); }
constexpr int MERGE_SR_MAX_TILES = 2048;              // the per-warp job search covers at most 32 lanes x 64 tiles

#ifndef TT_MERGE_CTAS_PER_SM
#define TT_MERGE_CTAS_PER_SM 1
#endif
constexpr int MERGE_CTAS_PER_SM = TT_MERGE_CTAS_PER_SM;   // resident CTAs per SM (registers and the 192 KiB of shared memory each)

// End (aligned frame) of the piece that starts last in `tile`: the first piece start of a later tile, or the text end.
__device__ __forceinline__ u32 closing_piece_end(const PieceParams& P, int tile) {
    for (int t = tile + 1; t < P.ntiles; t++) {                   // bounded by the number of tiles
        const u32 f = P.tile_first[t];
        if (f != TT_NONE) return (u32)t * TT_TILE_BYTES + f;
    }
    return (u32)P.hi;
}

// Bulk text: what k_scatter_bulk needs of a merged piece in one word -- bit 31, its number of ids (20 bits), its offset in the tile -- so that
// the pieces' offsets are neither written nor read (2 bytes a piece, both ways; see k_scatter_bulk).  PIECE_MANY: at least as many ids;
// such a piece covers the whole tile behind the one it starts in, and the first word of that one's pieces holds the number.
constexpr u32 PIECE_STAGED = 0x80000000u, PIECE_MANY = 0xFFFFFu;
static_assert(PIECE_MANY >= 2 * TT_TILE_BYTES, "a piece of so many bytes covers the tile behind its own");
TT_HD u32 piece_staged_word(u32 off, u32 m) { return PIECE_STAGED | (m << 11) | off; }

// A piece that needs no merging: an extracted literal (its id is staged already), a single byte, or a whole
// vocabulary entry.  Returns true and the value for piece_cnt.  One thread.
__device__ __forceinline__ bool piece_settled_without_merge(const PieceParams& P, const u8* __restrict__ text, u32 a, u32 n, u32& value) {
    if (P.litstart != nullptr) {
        const long long g = (long long)a + P.shift;
        if ((P.litstart[g >> 5] >> (g & 31)) & 1) { value = P.gq != nullptr ? piece_staged_word((u32)(g % TT_TILE_BYTES), 1u) : 0u - 1u; return true; }
    }
    int32_t id;
    if (n == 1) { value = (u32)P.ext_id[text[a]]; return true; }
    if (n <= TT_TOKTAB_MAXLEN) {
        if (P.toktab.shorts != nullptr && toktab_lookup(P.toktab, text, a, n, id)) { value = (u32)id; return true; }
    } else if (P.longtab.slots != nullptr && n <= P.longtab.maxlen && longtab_lookup(P.longtab, text, a, n, id)) { value = (u32)id; return true; }
    return false;
}

__device__ __forceinline__ void piece_done(const PieceParams& P, u32 a, u32 slot, u32 m) {
    if (P.gq != nullptr) {
        P.piece_cnt[slot] = piece_staged_word((u32)(a + P.shift) % TT_TILE_BYTES, min(m, PIECE_MANY));
        if (m >= PIECE_MANY) P.piece_cnt[(slot / TT_TILE_BYTES + 1) * TT_TILE_BYTES] = m;
    } else P.piece_cnt[slot] = 0u - m;
    atomicAdd(&P.tile_tok[slot / TT_TILE_BYTES], m);
}

// One piece of 2..256 bytes, the whole warp.
__device__ __forceinline__ bool piece_in_range(const PieceParams& P, u32 a, u32 n, u32 slot, u32 site) {
    const bool ok = n >= 1 && (long long)a + n <= P.hi - P.shift && slot < (u32)P.ntiles * TT_TILE_BYTES;
    if (!ok) hdr_selfcheck_failed(P.hdr, P.epoch, site, a, n, slot, 0u);
    return ok;
}
__device__ __forceinline__ void warp_merge_piece(const PieceParams& P, const u8* __restrict__ text, u32 a, u32 n, u32 slot, u64* wbuf, int lane) {
    if (!piece_in_range(P, a, n, slot, 1u) || n < 2 || n > (u32)TT_WARP_PIECE_MAX) { if (n < 2 || n > (u32)TT_WARP_PIECE_MAX) hdr_selfcheck_failed(P.hdr, P.epoch, 2u, a, n, slot, 0u); return; }
    u32* const pbuf = reinterpret_cast<u32*>(wbuf);
    const auto out = [&](u32 j, u32 t) { P.stage[a + j] = P.ext_id[t]; };
    const u32 m = n <= LANE_MAX ? warp_merge_reg(text, a, n, P.tab, lane, out)
                : n <= 64 ? warp_merge_perm<2>(pbuf, text, a, n, P.tab, lane, out)
                : n <= 128 ? warp_merge_perm<4>(pbuf, text, a, n, P.tab, lane, out)
                           : warp_merge_perm<WCH>(pbuf, text, a, n, P.tab, lane, out);
    if (lane == 0) piece_done(P, a, slot, m);
}

// ---- bulk text only: the closing pieces, and one list per length class for the whole text ---------------------
// A thread per tile settles the tile's closing piece where no merging is needed and gathers what is left of the
// 32 tiles of its warp -- queued short pieces, a short closing piece -- into one global list (one reservation
// per warp), so that k_merge's warps take 32 short pieces at a time whatever tile they come from; warp-class
// closing pieces join the first kernel's list, long pieces get a list of their own.  The counters were cleared
// by the memset in front of the chain.
constexpr int CLOSING_THREADS = 64;
// Length class of a short piece (2..32 bytes).
__device__ __forceinline__ int short_class(u32 n) {
    return n <= (u32)tt_short_class_max(0) ? 0 : n <= (u32)tt_short_class_max(1) ? 1 : n <= (u32)tt_short_class_max(2) ? 2 : 3;
}

__global__ void __launch_bounds__(CLOSING_THREADS)
k_closing(const __grid_constant__ PieceParams P) {
    const int lane = threadIdx.x & 31;
    const u32 FULL = 0xFFFFFFFFu;
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();                         // the first kernel's per-tile records are complete from here on
    if (hdr_status(P.hdr, P.epoch) != 0) return;
    const u8* text = P.base + P.shift;
    const int t = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    u32 ns = 0, nl = 0, np = 0, centry = 0;                  // centry != 0: a short closing piece to be queued
    if (t < P.ntiles) {
        const u32 q = P.tile_q[t];
        ns = q & TQ_NS_MASK; nl = (q >> TQ_NL_SHIFT) & TQ_NL_MASK; np = P.tile_cnt[t];
    }
    // the tile's first queue entries, on their way while the closing piece is looked up (one at a time in the two loops below, the
    // kernel took 19 us whatever the text's length)
    constexpr u32 AHEAD = 8;
    u32 ahead[AHEAD];
#pragma unroll
    for (u32 e = 0; e < AHEAD; e++) ahead[e] = e < ns ? P.q[(size_t)t * TT_TILE_QCAP + e] : 0u;
    u32 cn = 0, ca = 0, cslot = 0, clast = 0;
    if (np) {
        clast = P.tile_last[t];
        const u32 st = (u32)t * TT_TILE_BYTES + clast;
        cn = closing_piece_end(P, t) - st;
        ca = (u32)((long long)st - P.shift); cslot = (u32)t * TT_TILE_BYTES + np - 1;
        u32 v;
        if (piece_settled_without_merge(P, text, ca, cn, v)) { P.piece_cnt[cslot] = v; P.tile_tok[t] += 1u; cn = 0; }   // this thread is the tile's only writer here
        else if (cn <= (u32)LANE_MAX) { centry = tile_queue_entry(clast, np - 1, cn); }
        else if (cn <= (u32)TT_WARP_PIECE_MAX) P.wq[atomicAdd(&P.hdr->nwq, 1u)] = ((u64)(u32)t << 32) | tile_queue_entry(clast, np - 1, cn);
    }
    // long pieces: those inside the tile (listed by the first kernel) and a long closing piece
    const u32 nlong = nl + (cn > (u32)TT_WARP_PIECE_MAX ? 1u : 0u);
    if (nlong) {
        u32 b = atomicAdd(&P.hdr->nq_long, nlong);
        for (u32 j = 0; j < nl && j < (u32)TT_TILE_LONGCAP; j++) {
            const u32 idx = P.tile_long[(size_t)t * TT_TILE_LONGCAP + j];
            const u32 o = P.piece_off16[(size_t)t * TT_TILE_BYTES + idx], o2 = P.piece_off16[(size_t)t * TT_TILE_BYTES + idx + 1];
            P.lq[b++] = make_uint4((u32)((long long)t * TT_TILE_BYTES + o - P.shift), o2 - o, (u32)t * TT_TILE_BYTES + idx, 0u);
        }
        if (cn > (u32)TT_WARP_PIECE_MAX) P.lq[b] = make_uint4(ca, cn, cslot, 0u);
    }
    // short pieces: four lists by length (a warp later merges up to 32 pieces of one list at a time, a thread each, and
    // waits for the longest), one reservation per warp and list
    u64 mine = 0;                                             // four counts of 16 bits (a warp's 32 tiles hold fewer than 2^16 pieces)
#pragma unroll
    for (u32 e = 0; e < AHEAD; e++) if (e < ns) mine += 1ull << (16 * short_class((ahead[e] >> 22) + 1));
    for (u32 e = AHEAD; e < ns; e++) mine += 1ull << (16 * short_class((P.q[(size_t)t * TT_TILE_QCAP + e] >> 22) + 1));
    if (centry) mine += 1ull << (16 * short_class(cn));
    u64 pre = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const u64 v = __shfl_up_sync(FULL, pre, o); if (lane >= o) pre += v; }
    const u64 tot = __shfl_sync(FULL, pre, 31);
    u32 base[TT_SHORT_CLASSES];
#pragma unroll
    for (int c = 0; c < TT_SHORT_CLASSES; c++) {
        const u32 n = (u32)(tot >> (16 * c)) & 0xFFFFu;
        base[c] = 0;
        if (lane == 31 && n) base[c] = atomicAdd(c ? &P.hdr->nq_short_x[c - 1] : &P.hdr->nq_short, n);
    }
    pre -= mine;
#pragma unroll
    for (int c = 0; c < TT_SHORT_CLASSES; c++) base[c] = __shfl_sync(FULL, base[c], 31) + ((u32)(pre >> (16 * c)) & 0xFFFFu);
    const auto list = [&](u32 entry) {
        const int c = short_class((entry >> 22) + 1);
        const u64 x = ((u64)(u32)t << 32) | entry;
        if (c == 0) P.gq[base[0]++] = x;
        else if (c == 1) P.gq_x[0][base[1]++] = x;
        else if (c == 2) P.gq_x[1][base[2]++] = x;
        else P.gq_x[2][base[3]++] = x;
    };
#pragma unroll
    for (u32 e = 0; e < AHEAD; e++) if (e < ns) list(ahead[e]);
    for (u32 e = AHEAD; e < ns; e++) list(P.q[(size_t)t * TT_TILE_QCAP + e]);
    if (centry) list(centry);
}

// ---- long pieces --------------------------------------------------------------------------------------------------
// A piece of more than 256 bytes used to be merged by one CTA, round after round over the whole piece: 0.8 ms for the 64 KB
// blank runs of the 3M-char case, 45 ms for 64 KB of letters, with the rest of the GPU idle.  Now it is cut into windows.
//
// Why that is exact.  Call two tokens compatible if the byte string of the two together encodes to exactly these two.  A
// token sequence is the encoding of its byte string if and only if all its neighbours are compatible:
//   * If they are, look at the first merge of the sequential run on the whole string that crosses a boundary between two
//     of the tokens u, v.  Until then every merge lay inside a token, so the merges inside u and v were those of the run
//     on "u v" alone, in the same order (the lowest rank, leftmost, of the whole string is also that of the part it lies
//     in).  The run on "u v" alone would therefore make the crossing merge too, and u, v would not be compatible.
//   * Conversely the final run never crossed u | v, so the run on "u v" alone makes the same merges and ends with u, v.
// A window's encoding is a run of compatible neighbours.  Where the encodings of two overlapping windows share one token
// (same bytes, same place), the first one up to and including it, followed by the second one behind it, is again a run
// of compatible neighbours, whatever either window made of the rest.  So the windows are encoded independently, each by
// a warp, and joined at a shared token of every overlap; only if some overlap has none (a run of one character whose
// tokens stand at different phases in the two windows) the piece is merged as a whole by one CTA.
constexpr u32 LWIN = 256, LSTEP = 192;                 // bytes of a window (what a warp merges) and distance of their starts
constexpr u32 LQ_WINDOWS = 1, LQ_DONE = 2, LQ_FALLBACK = 3;       // states of an entry of lq
constexpr int LQ_CHUNK = 256;
constexpr int TT_RUNS = 32;                            // runs of one token that a warp keeps, one per lane
struct LongShared {
    uint4 q[LQ_CHUNK]; u32 pre[LQ_CHUNK + 1];          // a stretch of lq and the windows before each of its pieces
    u32 ticket;
    u32 nruns, rpos[TT_RUNS], rtok[2 * TT_RUNS], rcnt[2 * TT_RUNS];   // a piece of few byte runs (cta_run_piece)
};
__device__ __forceinline__ u32 long_windows(u32 n) { return n <= LWIN ? 1u : (n - LWIN + LSTEP - 1) / LSTEP + 1u; }

// The grid works through the steps below by tickets: a step's tasks are taken one by one by whichever CTA or warp comes,
// and a CTA waits before the next step until every task that was taken has been done.  So a CTA only ever waits for CTAs
// that are running: one that starts late, or never gets its place while others run, is not needed and finds nothing left
// to do.  Every wait is bounded.  step: 0 pieces found, 1 windows, 2 counts, 3 places, 4 ids.
__device__ __forceinline__ u32 warp_take(u32* counter, int lane) {
    u32 t = 0;
    if (lane == 0) t = atomicAdd(counter, 1u);
    return __shfl_sync(0xFFFFFFFFu, t, 0);
}
__device__ __forceinline__ u32 cta_take(u32* counter, u32* s_word) {
    __syncthreads();
    if (threadIdx.x == 0) *s_word = atomicAdd(counter, 1u);
    __syncthreads();
    return *s_word;
}
__device__ __noinline__ bool long_wait(const PieceParams& P, int step, u32 tasks) {          // all `tasks` tasks of the step are done
    bool ok = true;
    if (threadIdx.x == 0) {
        u32 seen = 0, tries = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&P.hdr->long_done[step]) : "memory");
            if (seen >= tasks) break;
            if ((++tries & 1023u) == 0 && hdr_status(P.hdr, P.epoch) != 0) { ok = false; break; }     // (a CTA that found an error does not come)
            if (tries > 10000000u) { ok = false; hdr_selfcheck_failed(P.hdr, P.epoch, 8u, seen, tasks, (u32)step, blockIdx.x); break; }
            __nanosleep(64);
        }
    }
    return __syncthreads_and(ok);
}
__device__ __forceinline__ void long_did(const PieceParams& P, int step, u32 tasks) {         // one thread, after its group's last write
    __threadfence();
    atomicAdd(&P.hdr->long_done[step], tasks);
}

// A piece that is a few runs of one byte each -- 64 KB of blanks, a ruler of equals signs -- is merged as runs: (token, how often),
// a lane each.  The round of the lowest rank (x, y) turns every run of x (if x = y) into half as many new tokens, with the
// odd one left at the end, or takes one token from the end of a run of x and one from the start of the run of y behind
// it.  A run of 2^k bytes takes k rounds whatever its tokens' lengths are, where rounds over its positions took 0.4 ms
// for 50 KB and windows would see tokens of thousands of bytes only in part.  Returns false if the piece has (or
// comes to have) more than 32 runs; then nothing is done.  Called by the whole CTA.
__device__ __noinline__ bool cta_run_piece(const PieceParams& P, const u8* __restrict__ text, u32 a, u32 n, u32 slot, LongShared& LS) {
    const u32 tid = threadIdx.x, T = blockDim.x, FULL = 0xFFFFFFFFu;
    const u8* const p = text + a;
    volatile u32* const nruns = &LS.nruns;
    __syncthreads();
    if (tid == 0) *nruns = 0;
    __syncthreads();
    // where the byte changes
    const auto change = [&](u32 pos) { if (*nruns < 2u * TT_RUNS) { const u32 k = atomicAdd(&LS.nruns, 1u); if (k < (u32)TT_RUNS) LS.rpos[k] = pos; } };
    const u32 skew = (u32)(4 - ((uintptr_t)p & 3)) & 3, nw = (n - skew) / 4;
    const u32* const w = reinterpret_cast<const u32*>(p + skew);
    if (tid >= 1 && tid < skew && p[tid] != p[tid - 1]) change(tid);
    if (tid < (n - skew) % 4) { const u32 q = skew + 4 * nw + tid; if (p[q] != p[q - 1]) change(q); }
    for (u32 i0 = tid; i0 < nw && *nruns < 2u * TT_RUNS; i0 += 8 * T) {
        u32 x[8], y[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const u32 i = i0 + u * T;
            x[u] = i < nw ? w[i] : 0u;
            y[u] = i < nw ? (i ? w[i - 1] >> 24 : skew ? (u32)p[skew - 1] : x[u] & 0xFFu) : 0u;      // the byte before the word
        }
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const u32 d = x[u] ^ ((x[u] << 8) | y[u]);
            if (d) for (u32 k = 0; k < 4; k++) if ((d >> (8 * k)) & 0xFFu) change(skew + 4 * (i0 + u * T) + k);
        }
    }
    __syncthreads();
    const u32 changes = *nruns;
    __syncthreads();
    if (changes >= (u32)TT_RUNS) return false;
    if (tid < 32) {
        const u32 lane = tid;
        u32 m = changes + 1;
        // runs in order
        const u32 mine = lane < changes ? LS.rpos[lane] : 0xFFFFFFFFu;
        u32 before = 0;
        for (int i = 0; i < 32; i++) { const u32 o = __shfl_sync(FULL, mine, i); before += o < mine; }
        __syncwarp();
        if (lane < changes) LS.rcnt[before + 1] = mine;              // start of run `before` + 1
        if (lane == 0) LS.rcnt[0] = 0;
        __syncwarp();
        u32 cnt = 0, tok = 0;
        if (lane < m) { const u32 s = LS.rcnt[lane]; cnt = (lane + 1 < m ? LS.rcnt[lane + 1] : n) - s; tok = p[s]; }
        __syncwarp();
        bool ok = true;
        for (u32 round = 0;; round++) {
            if (round > 4096) { ok = false; break; }
            // ranks of the pair inside the run and of the pair with the next run
            const u32 tn = __shfl_down_sync(FULL, tok, 1);
            u32 rs = TT_RANK_INF, rb = TT_RANK_INF;
            if (lane < m && cnt >= 2) rs = pair_probe(P.tab, tok, tok).r;
            if (lane + 1 < m) rb = pair_probe(P.tab, tok, tn).r;
            const u32 mn = __reduce_min_sync(FULL, min(rs, rb));
            if (mn == TT_RANK_INF) break;
            const bool self = rs == mn, cut = rb == mn;
            const u32 prev = __shfl_up_sync(FULL, (u32)cut, 1);
            const u32 k = lane < m ? cnt - ((lane > 0 && prev) ? 1u : 0u) - (cut ? 1u : 0u) : 0u;     // (self and cut exclude each other: a rank is one pair)
            // what becomes of the run, in order: (t0, k0), (t1, k1)
            u32 t0 = tok, k0 = k, t1 = 256u + mn, k1 = cut ? 1u : 0u;
            if (self) { t0 = 256u + mn; k0 = cnt >> 1; t1 = tok; k1 = cnt & 1; }
            const u32 c = (k0 ? 1u : 0u) + (k1 ? 1u : 0u);
            u32 at = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const u32 v = __shfl_up_sync(FULL, at, o); if (lane >= (u32)o) at += v; }
            const u32 total = __shfl_sync(FULL, at, 31);
            at -= c;
            if (k0) { LS.rtok[at] = t0; LS.rcnt[at] = k0; at++; }
            if (k1) { LS.rtok[at] = t1; LS.rcnt[at] = k1; }
            __syncwarp();
            // neighbours of one token become one run: a lane looks at elements 2 lane and 2 lane + 1
            const u32 e0 = 2 * lane, e1 = e0 + 1;
            const u32 a0 = e0 < total ? LS.rtok[e0] : 0xFFFFFFFFu, a1 = e1 < total ? LS.rtok[e1] : 0xFFFFFFFFu;
            const u32 n0 = e0 < total ? LS.rcnt[e0] : 0u, n1 = e1 < total ? LS.rcnt[e1] : 0u;
            u32 ap = __shfl_up_sync(FULL, a1, 1);
            if (lane == 0) ap = 0xFFFFFFFEu;
            const bool h0 = e0 < total && a0 != ap, h1 = e1 < total && a1 != a0;
            u32 hd = (h0 ? 1u : 0u) + (h1 ? 1u : 0u);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const u32 v = __shfl_up_sync(FULL, hd, o); if (lane >= (u32)o) hd += v; }
            m = __shfl_sync(FULL, hd, 31);
            if (m > 32) { ok = false; break; }
            __syncwarp();
            LS.rcnt[lane] = 0;
            __syncwarp();
            const u32 i1 = hd - 1, i0 = i1 - (h1 ? 1u : 0u);          // runs of the two elements
            if (e0 < total) { if (h0) LS.rtok[i0] = a0; atomicAdd(&LS.rcnt[i0], n0); }
            if (e1 < total) { if (h1) LS.rtok[i1] = a1; atomicAdd(&LS.rcnt[i1], n1); }
            __syncwarp();
            tok = lane < m ? LS.rtok[lane] : 0u; cnt = lane < m ? LS.rcnt[lane] : 0u;
            __syncwarp();
        }
        if (ok) {
            u32 end = lane < m ? cnt : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const u32 v = __shfl_up_sync(FULL, end, o); if (lane >= (u32)o) end += v; }
            LS.rtok[lane] = tok; LS.rcnt[lane] = end;                  // (lanes beyond the runs: no token, the same end)
        }
        if (lane == 0) *nruns = ok ? m : 0u;
    }
    __syncthreads();
    const u32 m = *nruns;
    if (m == 0) return false;
    const u32 total = LS.rcnt[m - 1];
    for (u32 r = 0; r < m; r++) {
        const int32_t id = P.ext_id[LS.rtok[r]];
        for (u32 j = (r ? LS.rcnt[r - 1] : 0u) + tid; j < LS.rcnt[r]; j += T) P.stage[a + j] = id;
    }
    if (tid == 0) piece_done(P, a, slot, total);
    __syncthreads();
    return true;
}

// The part of lq that starts at c0, with the number of windows before each of its pieces; returns how many there are.
__device__ u32 long_chunk(const PieceParams& P, u32 c0, u32 nl, LongShared& LS, u32* sc) {
    const u32 tid = threadIdx.x;
    __syncthreads();
    uint4 q = make_uint4(0, 0, 0, 0);
    if (tid < (u32)LQ_CHUNK && c0 + tid < nl) q = __ldcg(&P.lq[c0 + tid]);
    u32 total;
    const u32 ex = cta_excl_sum_scan(q.w == LQ_WINDOWS ? long_windows(q.y) : 0u, sc, &total);
    if (tid < (u32)LQ_CHUNK) { LS.q[tid] = q; LS.pre[tid] = ex; }
    __syncthreads();
    return total;
}
__device__ __forceinline__ uint4 long_find(const LongShared& LS, u32 w, u32& k) {      // piece and number of window w of the chunk
    u32 lo = 0, hi = LQ_CHUNK;                           // the last piece with at most w windows before it
    while (hi - lo > 1) { const u32 mid = (lo + hi) >> 1; if (LS.pre[mid] <= w) lo = mid; else hi = mid; }
    k = w - LS.pre[lo];
    return LS.q[lo];
}

// The windows' results stand at the byte positions of their tokens, two words per position: even windows in the first, odd
// ones in the second (a window overlaps its neighbours only).  Entry = token + 1 where a token begins, else 0.
__device__ __forceinline__ u32* long_at(const PieceParams& P, u32 a, u32 pos, u32 k) { return reinterpret_cast<u32*>(P.pairbuf + a + pos) + (k & 1); }
// A word per window that no window's result uses: 64 bytes into window k, in the words of the other windows.
__device__ __forceinline__ u32* long_word(const PieceParams& P, u32 a, u32 k) { return long_at(P, a, k * LSTEP + 64, k + 1); }

__device__ __noinline__ void long_window(const PieceParams& P, const u8* __restrict__ text, uint4 q, u32 k, u64* wbuf, int lane) {
    u32* const buf = reinterpret_cast<u32*>(wbuf);
    const u32 s = k * LSTEP, size = min(LWIN, q.y - s);
    if (k == 0 && lane == 0) P.piece_cnt[q.z] = 0u;      // (set to 1 where two windows do not meet)
    const u32 m = warp_merge_perm<WCH>(buf, text, q.x + s, size, P.tab, lane, [&](u32 j, u32 t) { buf[j] = t; });
    __syncwarp();
    u32 t[8], len[8], sum = 0;                           // eight neighbouring tokens per lane
#pragma unroll
    for (int j = 0; j < 8; j++) { const u32 i = lane * 8 + j; t[j] = i < m ? buf[i] : 0u; len[j] = i < m ? (u32)P.tok_len[t[j]] : 0u; sum += len[j]; }
    u32 pos = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const u32 x = __shfl_up_sync(0xFFFFFFFFu, pos, o); if (lane >= o) pos += x; }
    pos -= sum;
    u32* const arr = buf + 512;
#pragma unroll
    for (int j = 0; j < 8; j++) arr[j * 32 + lane] = 0u;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 8; j++) { if (lane * 8 + j < m && pos < LWIN) arr[pos] = t[j] + 1u; pos += len[j]; }
    __syncwarp();
    for (u32 p = lane; p < size; p += 32) *long_at(P, q.x, s + p, k) = arr[p];
    __syncwarp();
}
// Where windows k and k + 1 share a token (offset in the piece), 0xFFFFFFFF: nowhere.
__device__ __forceinline__ u32 long_seam(const PieceParams& P, uint4 q, u32 k, int lane) {
    const u32 from = (k + 1) * LSTEP, to = min(k * LSTEP + LWIN, q.y);
    u32 hit[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const u32 p = from + h * 32 + lane;
        u32 x = 0, y = 1;
        if (p < to) { x = __ldcg(long_at(P, q.x, p, k)); y = __ldcg(long_at(P, q.x, p, k + 1)); }
        hit[h] = __ballot_sync(0xFFFFFFFFu, x != 0 && x == y);
    }
    return hit[0] ? from + (u32)__ffs(hit[0]) - 1 : hit[1] ? from + 32 + (u32)__ffs(hit[1]) - 1 : 0xFFFFFFFFu;
}
__device__ __forceinline__ void long_span(const PieceParams& P, uint4 q, u32 k, int lane, u32& left, u32& right) {     // window k decides [left, right)
    left = k ? long_seam(P, q, k - 1, lane) : 0u;
    right = k + 1 < long_windows(q.y) ? long_seam(P, q, k, lane) : q.y;
}

__device__ __forceinline__ u32 long_count(const PieceParams& P, uint4 q, u32 k, u32 left, u32 right, int lane) {       // tokens of window k in [left, right)
    u32 cnt = 0;
    for (u32 p0 = left; p0 < right; p0 += 32) cnt += __popc(__ballot_sync(0xFFFFFFFFu, p0 + lane < right && __ldcg(long_at(P, q.x, p0 + lane, k)) != 0));
    return cnt;
}
__device__ __forceinline__ void long_write(const PieceParams& P, uint4 q, u32 k, u32 left, u32 right, u32 at, int lane) {   // ... to the piece's places from `at` on
    for (u32 p0 = left; p0 < right; p0 += 32) {
        const u32 v = p0 + lane < right ? __ldcg(long_at(P, q.x, p0 + lane, k)) : 0u;
        const u32 b = __ballot_sync(0xFFFFFFFFu, v != 0);
        if (v && at < q.y) P.stage[q.x + at + __popc(b & ((1u << lane) - 1))] = P.ext_id[v - 1];
        at += __popc(b);
    }
}

// A piece of at most as many windows as the CTA has warps is the CTA's own: nobody waits for it.
constexpr u32 LONG_CTA_MAX = (MERGE_WARPS - 1) * LSTEP + LWIN;
constexpr u32 LONG_MANY = 8;
__device__ __noinline__ void cta_window_piece(const PieceParams& P, const u8* __restrict__ text, uint4 q, u64* s_buf, u32* sc) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const u32 nw = long_windows(q.y), k = (u32)wid;
    __syncthreads();
    if (k < nw) long_window(P, text, q, k, s_buf + wid * WARP_SMEM_WORDS, lane);
    __syncthreads();
    u32 left = 0, right = 0, cnt = 0;
    if (k < nw) long_span(P, q, k, lane, left, right);
    const bool meet = left != 0xFFFFFFFFu && right != 0xFFFFFFFFu;
    if (meet) cnt = long_count(P, q, k, left, right, lane);
    if (lane == 0) sc[wid] = cnt;
    u32 total = 0;
    if (__syncthreads_and(meet)) {
        u32 at = 0;
        for (int w = 0; w < MERGE_WARPS; w++) { const u32 c = sc[w]; total += c; if (w < wid) at += c; }
        long_write(P, q, k, left, right, at, lane);
    } else total = cta_merge_long(text, q.x, q.y, P.tab, P.ext_id, P.stage, P.pairbuf + q.x, s_buf, sc);
    if (threadIdx.x == 0) piece_done(P, q.x, q.z, total);
    __syncthreads();
}
// What a CTA does with a long piece that it comes upon; false: the piece is for the whole grid.  many: so are all but runs of bytes.
__device__ __forceinline__ bool cta_long_piece(const PieceParams& P, const u8* __restrict__ text, uint4 q, u64* s_buf, u32* sc, LongShared& LS, bool many = false) {
    if (cta_run_piece(P, text, q.x, q.y, q.z, LS)) return true;
    if (many || q.y > LONG_CTA_MAX) return false;
    cta_window_piece(P, text, q, s_buf, sc);
    return true;
}

// The pieces of lq in state LQ_WINDOWS, once the `found` tasks that look for long pieces are done.  Called by every CTA.
__device__ __noinline__ void long_phase(const PieceParams& P, const u8* __restrict__ text, u32 found, u64* s_buf, u32* sc, LongShared& LS) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (!long_wait(P, 0, found)) return;
    const u32 nl = *reinterpret_cast<volatile u32*>(&P.hdr->nq_long);
    if (nl == 0) return;
    u64* const wbuf = s_buf + wid * WARP_SMEM_WORDS;
    // f(piece, window) for the windows of the list, by tickets of step `step`; returns the number of windows
    auto each_window = [&](int step, auto f) {
        u32 base = 0, mine = 0, t = warp_take(&P.hdr->long_take[step], lane);
        for (u32 c0 = 0; c0 < nl; c0 += LQ_CHUNK) {
            const u32 total = long_chunk(P, c0, nl, LS, sc);
            while (t - base < total) { u32 k; const uint4 q = long_find(LS, t - base, k); f(q, k); mine++; t = warp_take(&P.hdr->long_take[step], lane); }
            base += total;
        }
        __syncwarp();
        if (lane == 0 && mine) long_did(P, step, mine);
        return base;
    };
    const u32 nwin = each_window(1, [&](const uint4& q, u32 k) { long_window(P, text, q, k, wbuf, lane); });
    if (!long_wait(P, 1, nwin)) return;
    // how many tokens each window contributes
    each_window(2, [&](const uint4& q, u32 k) {
        u32 left, right;
        long_span(P, q, k, lane, left, right);
        if (left == 0xFFFFFFFFu || right == 0xFFFFFFFFu) { if (lane == 0) P.piece_cnt[q.z] = 1u; return; }
        const u32 cnt = long_count(P, q, k, left, right, lane);
        if (lane == 0) *long_word(P, q.x, k) = cnt;
    });
    if (!long_wait(P, 2, nwin)) return;
    // a CTA per piece: the places of the windows' tokens
    {
        u32 mine = 0;
        for (u32 e; (e = cta_take(&P.hdr->long_take[3], &LS.ticket)) < nl;) {     // block-uniform
            mine++;
            const uint4 q = __ldcg(&P.lq[e]);
            if (q.w != LQ_WINDOWS) continue;
            const u32 bad = __ldcg(&P.piece_cnt[q.z]);
            __syncthreads();
            if (bad) { if (tid == 0) P.lq[e].w = LQ_FALLBACK; continue; }
            const u32 nw = long_windows(q.y);
            u32 carry = 0;
            for (u32 k0 = 0; k0 < nw; k0 += blockDim.x) {
                const u32 k = k0 + tid;
                u32 total;
                const u32 ex = cta_excl_sum_scan(k < nw ? __ldcg(long_word(P, q.x, k)) : 0u, sc, &total);
                if (k < nw) *long_word(P, q.x, k) = carry + ex;
                carry += total;
                __syncthreads();
            }
            if (tid == 0) piece_done(P, q.x, q.z, carry);
        }
        __syncthreads();
        if (tid == 0 && mine) long_did(P, 3, mine);
    }
    if (!long_wait(P, 3, nl)) return;
    // the ids
    each_window(4, [&](const uint4& q, u32 k) {
        u32 left, right;
        long_span(P, q, k, lane, left, right);
        long_write(P, q, k, left, right, __ldcg(long_word(P, q.x, k)), lane);
    });
    // windows that do not meet: the piece as a whole (nobody waits any more)
    for (u32 e; (e = cta_take(&P.hdr->long_take[5], &LS.ticket)) < nl;) {         // block-uniform
        const uint4 q = __ldcg(&P.lq[e]);
        if (q.w != LQ_FALLBACK) continue;
        const u32 m = cta_merge_long(text, q.x, q.y, P.tab, P.ext_id, P.stage, P.pairbuf + q.x, s_buf, sc);
        if (tid == 0) piece_done(P, q.x, q.z, m);
    }
    __syncthreads();
}

// A request: the long pieces of one tile, by one thread; f(piece) for each.
template <class F>
__device__ __forceinline__ void tile_long_pieces(const PieceParams& P, int t, u32 tq, u32 np, u32 last, u32 next, F f) {
    const u32 nl = (tq >> TQ_NL_SHIFT) & TQ_NL_MASK;
    for (u32 j = 0; j < nl && j < (u32)TT_TILE_LONGCAP; j++) {
        const u32 idx = P.tile_long[(size_t)t * TT_TILE_LONGCAP + j];
        const u32 o = P.piece_off16[(size_t)t * TT_TILE_BYTES + idx], o2 = P.piece_off16[(size_t)t * TT_TILE_BYTES + idx + 1];
        f(make_uint4((u32)((long long)t * TT_TILE_BYTES + o - P.shift), o2 - o, (u32)t * TT_TILE_BYTES + idx, 0u));
    }
    if (np) {
        const u32 st = (u32)t * TT_TILE_BYTES + last, n = (next != TT_NONE ? (u32)(t + 1) * TT_TILE_BYTES + next : closing_piece_end(P, t)) - st;
        if (n > (u32)TT_WARP_PIECE_MAX) f(make_uint4((u32)((long long)st - P.shift), n, (u32)t * TT_TILE_BYTES + np - 1, 0u));
    }
}
// The long pieces of the list LS.q[0 .. cnt), by the whole CTA.
__device__ __noinline__ void cta_long_list(const PieceParams& P, const u8* __restrict__ text, u32 cnt, u64* s_buf, u32* sc, LongShared& LS) {
    const int tid = threadIdx.x;
    for (u32 e = 0; e < cnt; e++) {                                   // block-uniform
        const uint4 q = LS.q[e];
        __syncthreads();
        if (!piece_in_range(P, q.x, q.y, q.z, 3u)) continue;
        if (tid == 0) { u32 v = 0; sc[SCR_FLAG] = piece_settled_without_merge(P, text, q.x, q.y, v) ? 1u : 0u; sc[SCR_VALUE] = v; }
        __syncthreads();
        if (sc[SCR_FLAG]) { if (tid == 0) { P.piece_cnt[q.z] = sc[SCR_VALUE]; atomicAdd(&P.tile_tok[q.z / TT_TILE_BYTES], 1u); } continue; }
        const bool done = cta_long_piece(P, text, q, s_buf, sc, LS);
        if (tid == 0 && !done) P.lq[atomicAdd(&P.hdr->nq_long, 1u)] = make_uint4(q.x, q.y, q.z, LQ_WINDOWS);
    }
    __syncthreads();
}
// A request: looks for its long pieces.  Without one for the whole grid, the CTA merges those of every gridDim.x-th tile and
// nobody waits for it; with one, the tiles go by tickets, LONG_FIND each, so that all of them are looked at by the CTAs
// that run.  Returns whether there are long pieces (1) and some for the grid (2); every CTA comes to the same answer.
constexpr int LONG_FIND = 8;
__device__ __forceinline__ u32 long_find_tasks(const PieceParams& P) { return (u32)(P.ntiles + LONG_FIND - 1) / LONG_FIND; }
__device__ __noinline__ u32 cta_find_long(const PieceParams& P, const u8* __restrict__ text, u64* s_buf, u32* sc, LongShared& LS) {
    const int tid = threadIdx.x;
    if (tid == 0) LS.pre[0] = 0;
    __syncthreads();
    bool any = false, grid = false;
    for (int t = tid; t < P.ntiles; t += MERGE_THREADS) {
        const u32 next = t + 1 < P.ntiles ? P.tile_first[t + 1] : TT_NONE;
        tile_long_pieces(P, t, P.tile_q[t], P.tile_cnt[t], P.tile_last[t], next, [&](uint4 q) {
            any = true; grid |= q.y > LONG_CTA_MAX;
            if (t % (int)gridDim.x == (int)blockIdx.x) { const u32 k = atomicAdd(&LS.pre[0], 1u); if (k < (u32)LQ_CHUNK) LS.q[k] = q; }
        });
    }
    // (a share of more than 256 long pieces: by tickets too)
    grid |= P.ntiles > (int)gridDim.x * (LQ_CHUNK / (TT_TILE_LONGCAP + 1));
    if (!__syncthreads_or(any)) return 0;
    if (!__syncthreads_or(grid)) { cta_long_list(P, text, LS.pre[0], s_buf, sc, LS); return 1; }
    const u32 tasks = long_find_tasks(P);
    u32 mine = 0;
    for (u32 task; (task = cta_take(&P.hdr->long_take[0], &LS.ticket)) < tasks;) {
        mine++;
        if (tid == 0) LS.pre[0] = 0;
        __syncthreads();
        const int t = (int)task * LONG_FIND + tid;
        static_assert(LONG_FIND * (TT_TILE_LONGCAP + 1) <= LQ_CHUNK, "the long pieces of a task");
        if (tid < LONG_FIND && t < P.ntiles)
            tile_long_pieces(P, t, P.tile_q[t], P.tile_cnt[t], P.tile_last[t], t + 1 < P.ntiles ? P.tile_first[t + 1] : TT_NONE, [&](uint4 q) { LS.q[atomicAdd(&LS.pre[0], 1u)] = q; });
        __syncthreads();
        cta_long_list(P, text, LS.pre[0], s_buf, sc, LS);
    }
    __syncthreads();
    if (tid == 0 && mine) long_did(P, 0, mine);
    return 2;
}

// Bulk text: the last CTA of k_merge_bulk to finish sums the token counts of every group of 256 tiles for k_scatter_bulk (a
// counter cleared before the chain tells which CTA that is; nobody waits for anybody), a warp a group.  (One warp for all the
// groups took 100 us behind the merges of a 132 MB batch.)
__device__ __forceinline__ void merge_group_totals(const PieceParams& P, u32* s_last) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const u32 FULL = 0xFFFFFFFFu;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) *s_last = atomicAdd(&P.hdr->merge_done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!*s_last) return;
    __threadfence();
    const int ngroups = (P.ntiles + TT_GROUP_TILES - 1) / TT_GROUP_TILES;
    for (int g = wid; g < ngroups; g += MERGE_WARPS) {                // eight loads per lane and group
        u32 sum = 0;
#pragma unroll
        for (int u = 0; u < TT_GROUP_TILES / 32; u++) { const int t = g * TT_GROUP_TILES + u * 32 + lane; if (t < P.ntiles) sum += __ldcg(&P.tile_tok[t]); }
        sum = __reduce_add_sync(FULL, sum);
        if (lane == 0) P.grp_tok[g] = sum;
    }
}

// Bulk text (k_closing has gathered the lists): long pieces a CTA each where that is quick, else window by window with the
// whole grid, warp-class pieces a warp each by index, short pieces in batches of one length class by ticket, a thread each.
__device__ void merge_bulk_lists(const PieceParams& P, const u8* __restrict__ text, u64* s_buf, u32* sc, LongShared& LS, u32* s_last) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const u32 FULL = 0xFFFFFFFFu;
    const u32 nl = P.hdr->nq_long, nw = P.hdr->nwq, ns = P.hdr->nq_short;
    // With more long pieces than LONG_MANY per CTA their windows go to the warps of the whole grid: a CTA that takes a piece of 300 bytes
    // has work for two of its 24 warps (6 MB of words of 300 letters, 20,000 pieces, 4,096 merges: 6.3 ms a call so, now 4.3; with one CTA for a whole piece 5.6).
    const bool many = nl > LONG_MANY * gridDim.x;
    if (nl) {
        u32 mine = 0;
        for (u32 e; (e = cta_take(&P.hdr->long_take[0], &LS.ticket)) < nl;) {     // block-uniform
            mine++;
            const uint4 q = P.lq[e];
            u32 state = LQ_DONE;
            if (piece_in_range(P, q.x, q.y, q.z, 3u) && !cta_long_piece(P, text, q, s_buf, sc, LS, many)) state = LQ_WINDOWS;
            if (tid == 0) P.lq[e].w = state;
        }
        __syncthreads();
        if (tid == 0 && mine) long_did(P, 0, mine);
    }
    u64* wbuf = s_buf + wid * WARP_SMEM_WORDS;
    const u32 W = gridDim.x * MERGE_WARPS, gw = (u32)wid * gridDim.x + blockIdx.x;
    for (u32 j = gw; j < nw; j += W) {                                // bounded by the list length
        const u64 x = P.wq[j];
        const u32 t = (u32)(x >> 32), e = (u32)x;
        warp_merge_piece(P, text, (u32)((long long)t * TT_TILE_BYTES + (e & 2047u) - P.shift), (e >> 22) + 1, t * TT_TILE_BYTES + ((e >> 11) & 2047u), wbuf, lane);
    }
    u32* const tok = reinterpret_cast<u32*>(wbuf);
    // tickets: a batch of one list each, the list of the longest pieces first
    u32 cnts[TT_SHORT_CLASSES], nb[TT_SHORT_CLASSES], nball = 0;
#pragma unroll
    for (int c = 0; c < TT_SHORT_CLASSES; c++) { cnts[c] = c ? P.hdr->nq_short_x[c - 1] : ns; nball += cnts[c]; }
    const u32 per = short_batch(nball);
    nball = 0;
#pragma unroll
    for (int c = 0; c < TT_SHORT_CLASSES; c++) { nb[c] = (cnts[c] + per - 1) / per; nball += nb[c]; }
    for (;;) {                                                        // bounded by the number of tickets
        u32 tk = 0;
        if (lane == 0) tk = atomicAdd(&P.hdr->t_short, 1u);
        tk = __shfl_sync(FULL, tk, 0);
        if (tk >= nball) break;
        const u64* list = P.gq; u32 cnt = 0, e0 = 0;
        {
            u32 r = tk;
            bool found = false;
#pragma unroll
            for (int c = TT_SHORT_CLASSES - 1; c >= 0; c--) {
                if (!found && r < nb[c]) { list = c ? P.gq_x[c - 1] : P.gq; cnt = cnts[c]; e0 = r * per; found = true; }
                if (!found) r -= nb[c];
            }
        }
        if ((u32)lane < per && e0 + lane < cnt) {
            const u64 x = list[e0 + lane];
            const u32 t = (u32)(x >> 32), e = (u32)x;
            const u32 a = (u32)((long long)t * TT_TILE_BYTES + (e & 2047u) - P.shift), n = (e >> 22) + 1, slot = t * TT_TILE_BYTES + ((e >> 11) & 2047u);
            if (!piece_in_range(P, a, n, slot, 4u) || n < 2 || n > (u32)LANE_MAX) hdr_selfcheck_failed(P.hdr, P.epoch, 5u, a, n, slot, e0);
            else {
                const u32 m = lane_merge<false>(tok, lane, text, a, n, P.tab, P.ext_id, P.stage);
                piece_done(P, a, slot, m);
            }
        }
        __syncwarp();
    }
    if (nl) long_phase(P, text, nl, s_buf, sc, LS);
    merge_group_totals(P, s_last);
}

// The merge kernel of bulk text (more tiles than a request's job search covers): works off the lists k_closing built.
__global__ void __launch_bounds__(MERGE_THREADS, MERGE_CTAS_PER_SM)
k_merge_bulk(const __grid_constant__ PieceParams P) {
    extern __shared__ __align__(16) u64 s_buf[];              // MERGE_SMEM_BYTES
    __shared__ u32 sc[SCR_WORDS];
    __shared__ u32 s_last;
    __shared__ LongShared LS;
    cudaTriggerProgrammaticLaunchCompletion();               // k_scatter may be placed; it waits for this grid's memory itself
    grid_prefetch_l2(P.tab.slots, ((size_t)P.tab.mask + 1) * 2 * sizeof(uint4));
    grid_prefetch_l2(P.tab.bytepair, 65536 * sizeof(u64));
    cudaGridDependencySynchronize();                         // k_closing's lists are complete from here on
    if (hdr_status(P.hdr, P.epoch) != 0) return;
    merge_bulk_lists(P, P.base + P.shift, s_buf, sc, LS, &s_last);
}

// Where a request's unsettled pieces stand, for the job search of k_merge: exclusive prefixes of the tiles' counts of short
// and of warp-class pieces, in shared memory behind the warps' buffers (an entry is one tile up to 2,048 tiles).  The CTA
// scans them once with one 16-byte load per thread; every warp then finds its jobs by bisection.  (Each warp summing the
// counts of all tiles for itself took 1.6 us at 489 tiles, 13 at 1,400 and 24 at 1,900.)
constexpr int MERGE_ENTRIES = MERGE_SR_MAX_TILES;
struct MergeIndex { u32 pre_s[MERGE_ENTRIES + 1], pre_w[MERGE_ENTRIES + 1]; u64 wtot[MERGE_WARPS]; };
constexpr size_t MERGE_SMEM_REQUEST = MERGE_SMEM_BYTES + sizeof(MergeIndex);
static_assert(4 * MERGE_THREADS >= MERGE_ENTRIES, "four entries per thread");

// Returns whether any tile allows for a piece of more than 256 bytes.
__device__ __forceinline__ bool merge_index(const PieceParams& P, int unit, int entries, MergeIndex& X) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    u32 c[4] = {0, 0, 0, 0}, flags = 0;                           // per entry: short pieces (low half), warp-class pieces
    u64 mine = 0;
    if (4 * tid < entries) {
        if (unit == 1) {
            const uint4 v = *reinterpret_cast<const uint4*>(P.tile_q + 4 * tid);
            c[0] = v.x; c[1] = v.y; c[2] = v.z; c[3] = v.w;
        }
#pragma unroll
        for (int h = 0; h < 4; h++) {
            u32 s = 0, w = 0;
            for (int u = 0; u < unit; u++) {
                const int t = (4 * tid + h) * unit + u;
                if (t < P.ntiles) { const u32 q = unit == 1 ? c[h] : P.tile_q[t]; s += q & TQ_NS_MASK; w += (q >> TQ_NW_SHIFT) & TQ_NW_MASK; flags |= q; }
            }
            c[h] = s | (w << 16);
            mine += (u64)s | ((u64)w << 32);
        }
    }
    u64 x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const u64 t = __shfl_up_sync(0xFFFFFFFFu, x, o); if (lane >= o) x += t; }
    if (lane == 31) X.wtot[wid] = x;
    __syncthreads();
    const u64 wt = lane < wid ? X.wtot[lane] : 0ull;             // (a warp's counts fit 32 bits each)
    const u64 before = x - mine + __reduce_add_sync(0xFFFFFFFFu, (u32)wt) + ((u64)__reduce_add_sync(0xFFFFFFFFu, (u32)(wt >> 32)) << 32);
    if (4 * tid < entries) {
        u32 s = (u32)before, w = (u32)(before >> 32);
#pragma unroll
        for (int h = 0; h < 4; h++) if (4 * tid + h <= entries) { X.pre_s[4 * tid + h] = s; X.pre_w[4 * tid + h] = w; s += c[h] & 0xFFFFu; w += c[h] >> 16; }
        if (4 * tid + 4 >= entries) { X.pre_s[entries] = s; X.pre_w[entries] = w; }       // (entries behind the last one count nothing)
    }
    return __syncthreads_or(flags >> 31);
}
// The last entry with at most k pieces before it.
__device__ __forceinline__ u32 merge_find(const u32* pre, u32 entries, u32 k) {
    u32 lo = 0, hi = entries;
    while (hi - lo > 1) { const u32 mid = (lo + hi) >> 1; if (pre[mid] <= k) lo = mid; else hi = mid; }
    return lo;
}

constexpr u32 SHORT_PER_WARP = 5;                    // more short pieces than that per warp of the grid: see k_merge
// The k-th queued piece of its class (warp-class or short).
__device__ __forceinline__ void merge_queued(const PieceParams& P, const MergeIndex& X, int unit, int entries, bool wclass, u32 k, u32& a, u32& n, u32& slot) {
    const u32* const pre = wclass ? X.pre_w : X.pre_s;
    const u32 en = merge_find(pre, (u32)entries, k);
    u32 r = k - pre[en], t = en * (u32)unit;
    for (int u = 0; u + 1 < unit; u++) {
        const u32 q = P.tile_q[t], c = wclass ? (q >> TQ_NW_SHIFT) & TQ_NW_MASK : q & TQ_NS_MASK;
        if (r < c) break;
        r -= c; t++;
    }
    const u32 e = P.q[(size_t)t * TT_TILE_QCAP + (wclass ? (u32)TT_TILE_QCAP - 1 - r : r)];
    n = (e >> 22) + 1;
    a = (u32)((long long)t * TT_TILE_BYTES + (e & 2047u) - P.shift); slot = t * TT_TILE_BYTES + ((e >> 11) & 2047u);
}
// The closing piece of tile t, where it has at most 256 bytes and needs merging (every lane computes the same).
__device__ __forceinline__ bool merge_closing(const PieceParams& P, const u8* __restrict__ text, u32 t, int lane, u32& a, u32& n, u32& slot) {
    const u32 np = P.tile_cnt[t], last = P.tile_last[t], next = t + 1 < (u32)P.ntiles ? P.tile_first[t + 1] : TT_NONE;
    if (np == 0) return false;
    const u32 st = t * TT_TILE_BYTES + last;
    n = (next != TT_NONE ? (t + 1) * TT_TILE_BYTES + next : closing_piece_end(P, (int)t)) - st;
    if (n > (u32)TT_WARP_PIECE_MAX) return false;                    // a long piece
    a = (u32)((long long)st - P.shift); slot = t * TT_TILE_BYTES + np - 1;
    u32 v;
    if (!piece_settled_without_merge(P, text, a, n, v)) return true;
    if (lane == 0) { P.piece_cnt[slot] = v; atomicAdd(&P.tile_tok[t], 1u); }
    return false;
}
// The queued short pieces in batches, in their order, whatever tiles they stand in, a thread each; the batches are spread over the
// grid, by tickets where some CTAs first had a long piece.  (With a ticket per tile 147 warps took the 150,000 two-byte pieces of
// 300 KB, most of them on the few SMs that came first: 78 to 118 us, now 54 to 66.)  Out of line: when a call of 4,000 characters,
// which does none of this, took 33 us, it took 0.3 us more with the batches in line.  Now it takes 20.3 either way, 1,000 messages 55.8
// and in line 54.4, 3M chars of long runs 189.8 and 186.3.
__device__ __noinline__ void merge_short_batches(const PieceParams& P, const u8* __restrict__ text, const MergeIndex& X, int unit, int entries, bool by_ticket, u32* buf) {
    const u32 lane = threadIdx.x & 31, W = gridDim.x * MERGE_WARPS, NS = X.pre_s[entries], per = short_batch(NS), nb = (NS + per - 1) / per;
    u32 b = by_ticket ? warp_take(&P.hdr->t_tiles, (int)lane) : (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    while (b < nb) {
        const u32 k = per * b + lane;
        if (lane < per && k < NS) {
            u32 a, n, slot;
            merge_queued(P, X, unit, entries, false, k, a, n, slot);
            if (!piece_in_range(P, a, n, slot, 4u) || n < 2 || n > (u32)LANE_MAX) hdr_selfcheck_failed(P.hdr, P.epoch, 5u, a, n, slot, k);
            else piece_done(P, a, slot, lane_merge<true>(buf, (int)lane, text, a, n, P.tab, P.ext_id, P.stage));
        }
        __syncwarp();
        b = by_ticket ? warp_take(&P.hdr->t_tiles, (int)lane) : b + W;
    }
}

// The kernel's work once the first kernel's records are complete.  s_buf: MERGE_SMEM_REQUEST bytes.
__device__ __forceinline__ void merge_request(const PieceParams& P, u64* s_buf, u32* sc, LongShared& LS) {
    MergeIndex& X = *reinterpret_cast<MergeIndex*>(s_buf + MERGE_WARPS * WARP_SMEM_WORDS);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int status = hdr_status(P.hdr, P.epoch);
    const int unit = (P.ntiles + MERGE_ENTRIES - 1) / MERGE_ENTRIES, entries = (P.ntiles + unit - 1) / unit;   // tiles per entry: 1 for a request
    const bool may_long = merge_index(P, unit, entries, X);
    if (status != 0) return;
    const u8* text = P.base + P.shift;
    const u32 longs = may_long ? cta_find_long(P, text, s_buf, sc, LS) : 0u;
    u64* wbuf = s_buf + wid * WARP_SMEM_WORDS;
    const u32 W = gridDim.x * MERGE_WARPS, gw = (u32)wid * gridDim.x + blockIdx.x;   // numbered across the CTAs first
    const u32 NS = X.pre_s[entries], NW = X.pre_w[entries], NT = (u32)P.ntiles;
    // A warp per piece, or a thread per piece?  A warp takes its pieces one after the other, 4 to 6 us each; a batch takes as long as its
    // slowest piece, 20 to 25 us, however few pieces there are.  Measured, short pieces and tiles per warp of the grid -> us a call with
    // a warp / a thread per piece: Unicode-heavy prose 2.5 -> 41.8 / 44.6, 5.0 -> 68.5 / 55.6, 8 -> 75.8 / 61.4; prose with 4,096
    // merges 4 -> 41.0 / 47.6, 6 -> 50.4 / 46.0, 7.5 -> 56.1 / 48.8; transcripts 2.5 -> 57.0 / 66.
    const bool many = NS + NT > SHORT_PER_WARP * W;
    const u32 J = many ? NW : NW + NT + NS;                          // jobs of a warp: all pieces, or the warp-class ones
    // Job by job in order (warp-class pieces, closing pieces, short pieces); where some CTAs first had a long piece to merge, by
    // tickets of `step` jobs, the next one drawn in advance.
    const u32 step = longs ? max(1u, J / (2 * W)) : 1u;
    u32 jt = gw, jn = gw + W;
    if (longs) { jt = warp_take(&P.hdr->t_short, lane); jn = warp_take(&P.hdr->t_short, lane); }
    for (u32 j = jt * step, left = step; j < J;) {                   // bounded by the number of jobs
        const u32 job = j;
        if (--left) j++;
        else { j = jn * step; left = step; jn = longs ? (j < J ? warp_take(&P.hdr->t_short, lane) : jn) : jn + W; }
        u32 a, n, slot;
        if (job >= NW && job < NW + NT) {                            // the closing piece of tile job - NW
            if (!merge_closing(P, text, job - NW, lane, a, n, slot)) continue;
        } else merge_queued(P, X, unit, entries, job < NW, job < NW ? job : job - NW - NT, a, n, slot);
        warp_merge_piece(P, text, a, n, slot, wbuf, lane);
    }
    if (many) {
        // (a place of their own for the closing pieces: with the merges in one place for both ways, the way without batches took 3 %
        // longer on transcripts and long runs)
        for (u32 t = gw; t < NT; t += W) {
            u32 a, n, slot;
            if (merge_closing(P, text, t, lane, a, n, slot)) warp_merge_piece(P, text, a, n, slot, wbuf, lane);
        }
        merge_short_batches(P, text, X, unit, entries, longs != 0, reinterpret_cast<u32*>(wbuf));
    }
    if (longs == 2) long_phase(P, text, long_find_tasks(P), s_buf, sc, LS);
}
__global__ void __launch_bounds__(MERGE_THREADS, MERGE_CTAS_PER_SM)
k_merge(const __grid_constant__ PieceParams P) {
    extern __shared__ __align__(16) u64 s_buf[];              // MERGE_SMEM_REQUEST
    __shared__ u32 sc[SCR_WORDS];
    __shared__ LongShared LS;
    cudaTriggerProgrammaticLaunchCompletion();               // k_scatter may be placed; it waits for this grid's memory itself
    grid_prefetch_l2(P.tab.slots, ((size_t)P.tab.mask + 1) * 2 * sizeof(uint4));
    grid_prefetch_l2(P.tab.bytepair, 65536 * sizeof(u64));
    cudaGridDependencySynchronize();                         // the first kernel's per-tile records are complete from here on
    merge_request(P, s_buf, sc, LS);
}

// ---- K5: coalesced scatter of the staged ids, one text tile per CTA iteration ---------------------------------
// Also writes the token offset of every document that starts in the tile (batch calls).
struct ScatterParams {
    long long shift, hi;
    int ntiles;
    const u32* tile_cnt;
    const u32* tile_tok;       // tokens per tile
    const u32* grp_tok;        // bulk text: tokens per group of TT_GROUP_TILES tiles, else null
    const u16* piece_off16;
    const u32* tile_q;         // bulk text: says where a document starts in the tile
    unsigned long long ids_cap;
    const u32* piece_cnt;
    const int32_t* stage;
    TTHeader* hdr;
    unsigned long long epoch;
    int32_t* ids_out;
    long long* count_out;
    int32_t* status_out;
    const u32* docmask;        // batch: bit per byte of document starts, else null
    const long long* doc_off;  // batch: n_docs + 1 offsets
    int n_docs;
    long long* ids_off_out;    // batch: n_docs + 1 token offsets
};

constexpr int SCATTER_STAGE_IDS = 2048;                   // ids of one work item that are put together in shared memory
// CTAs per SM the kernel is compiled for.  A text of at most 4 tiles per SM gets all 64 registers, its loads are what counts; with
// more tiles than that five CTAs of 48 registers (Thai-like text of 2.9 MB 97 -> 89 us per call; eight of 32 registers
// spill: 1M chars 32 -> 37 us).
constexpr int SCATTER_CTAS = 4, SCATTER_CTAS_MANY = 5;
constexpr u32 SCATTER_WARP_MAX = 512;                     // tokens of a piece that one warp copies; longer ones the whole CTA
// Work items: (tile, block of 512 of its pieces), two neighbouring pieces per thread.  (A piece of more than eight ids has at least nine
// bytes: a tile has at most 228 of them, which is what `big` holds.)  A request has a tile per CTA and most
// tiles one item, so what counts is the chain of dependent steps: everything that does not depend on anything else -- the
// tiles' token counts, the first item's values and offsets, read before its length is known -- is asked for at once, the sums
// over the tiles and the scan over the item's pieces share one barrier, and a staged piece's ids are fetched side by
// side.  (Step by step, with a barrier after each, the kernel took 7.5 us behind k_merge on a 1M-char request.)
struct ScatterShared {
    u32 scan[2][BPE_WARPS], before[BPE_WARPS], total[BPE_WARPS];
    u32 big[TT_TILE_BYTES / 8][3];
    u32 nbig;
    int32_t out[SCATTER_STAGE_IDS];                          // the ids of one item on their way out
};
// The kernel's work once the merges are complete.  (A function of its own with its shared memory in one structure: written out in the kernel, the
// five-CTA instance took 20.5 us instead of 18.4 for 2.9 MB of Thai-like text.)
__device__ __forceinline__ void scatter_tiles(const ScatterParams& P, ScatterShared& SH) {
    auto& s_scan = SH.scan; auto& s_before = SH.before; auto& s_total = SH.total; auto& s_big = SH.big; auto& s_out = SH.out;
    u32& s_nbig = SH.nbig;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const u32 FULL = 0xFFFFFFFFu;
    // Each CTA takes a contiguous range of tiles and sums the token counts before it, and all of them (the count, and the
    // capacity check, which every CTA makes for itself).
    const int per = (P.ntiles + (int)gridDim.x - 1) / (int)gridDim.x;
    const int tile_lo = (int)blockIdx.x * per, tile_hi = min(P.ntiles, tile_lo + per);
    if (tile_lo >= tile_hi) return;                           // (the first CTA always has a tile)
    if (tid == 0) s_nbig = 0;
    int tile = tile_lo;
    u32 b = 0, np = P.tile_cnt[tile];
    uint2 v = *reinterpret_cast<const uint2*>(P.piece_cnt + (size_t)tile * TT_TILE_BYTES + 2 * tid);
    u32 o2 = *reinterpret_cast<const u32*>(P.piece_off16 + (size_t)tile * TT_TILE_BYTES + 2 * tid);
    int status = hdr_status(P.hdr, P.epoch);
    u32 before = 0, total = 0;                                // (a text has fewer than 2^31 bytes)
    for (int t0 = 0; t0 < P.ntiles; t0 += BPE_THREADS * 4) {
        u32 x[4];
#pragma unroll
        for (int u = 0; u < 4; u++) { const int t = t0 + u * BPE_THREADS + tid; x[u] = t < P.ntiles ? P.tile_tok[t] : 0u; }
#pragma unroll
        for (int u = 0; u < 4; u++) { total += x[u]; if (t0 + u * BPE_THREADS + tid < tile_lo) before += x[u]; }
    }
    before = __reduce_add_sync(FULL, before); total = __reduce_add_sync(FULL, total);
    if (lane == 0) { s_before[wid] = before; s_total[wid] = total; }
    u32 carry = 0;
    for (int item = 0;; item++) {                             // block-uniform
        // the item after this one
        int tile2 = tile;
        u32 b2 = b + 2 * BPE_THREADS, np2 = np;
        if (b2 >= np) { b2 = 0; tile2++; np2 = tile2 < tile_hi ? P.tile_cnt[tile2] : 0u; }
        uint2 vn = make_uint2(0, 0);
        u32 on = 0;
        if (tile2 < tile_hi) {
            const size_t q0 = (size_t)tile2 * TT_TILE_BYTES + b2 + 2 * (u32)tid;
            if (b2 + 2 * (u32)tid < (u32)TT_TILE_BYTES) { vn = *reinterpret_cast<const uint2*>(P.piece_cnt + q0); on = *reinterpret_cast<const u32*>(P.piece_off16 + q0); }
        }
        // this item
        const u32 i0 = b + 2 * (u32)tid;
        const long long t0 = (long long)tile * TT_TILE_BYTES - P.shift;      // text offset of the tile start
        const int32_t x[2] = {i0 < np ? (int32_t)v.x : 0, i0 + 1 < np ? (int32_t)v.y : 0};     // an id, or minus the staged count
        const u32 c[2] = {i0 < np ? (x[0] >= 0 ? 1u : (u32)(-x[0])) : 0u, i0 + 1 < np ? (x[1] >= 0 ? 1u : (u32)(-x[1])) : 0u};
        u32 inc = c[0] + c[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const u32 y = __shfl_up_sync(FULL, inc, o); if (lane >= o) inc += y; }
        if (lane == 31) s_scan[item & 1][wid] = inc;
        const bool some_big = __syncthreads_or(c[0] > 8 || c[1] > 8);
        if (item == 0) {
            total = 0;
#pragma unroll
            for (int w = 0; w < BPE_WARPS; w++) { carry += s_before[w]; total += s_total[w]; }
            if (status == 0 && total > P.ids_cap) status = 5;         // TT_ERR_CAPACITY
            if (blockIdx.x == 0 && tid == 0) {
                if (P.status_out) *P.status_out = status;
                if (P.count_out) *P.count_out = status ? 0 : (long long)total;
            }
            if (status != 0) {
                // (by the CTAs that are here: those without a tile have left)
                const long long step = (long long)((P.ntiles + per - 1) / per) * blockDim.x;
                if (P.ids_off_out) for (long long d = (long long)blockIdx.x * blockDim.x + tid; d <= P.n_docs; d += step) P.ids_off_out[d] = 0;
                return;
            }
            if (P.ids_off_out && blockIdx.x == 0) {
                // documents that start at the very end of the text (empty trailing documents) and the total
                const long long len = P.hi - P.shift;
                for (int d = P.n_docs - tid; d >= 0 && P.doc_off[d] >= len; d -= blockDim.x) P.ids_off_out[d] = (long long)total;
            }
        }
        u32 d0 = carry + inc - c[0] - c[1], tot = 0;
#pragma unroll
        for (int w = 0; w < BPE_WARPS; w++) { const u32 y = s_scan[item & 1][w]; tot += y; if (w < wid) d0 += y; }
        // An item of at most SCATTER_STAGE_IDS tokens (nearly all) is put together in shared memory and leaves in whole lines, every
        // thread writing consecutive words: the output may be mapped host memory, where a warp that writes every other word
        // costs a bus transaction per word (100 KB of Unicode-heavy text, written piece by piece: 27 us instead of 9).
        const bool staged = tot <= (u32)SCATTER_STAGE_IDS;
        int32_t* const out = staged ? s_out - carry : P.ids_out;             // same index either way
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const u32 i = i0 + h, dst = h ? d0 + c[0] : d0, off = h ? o2 >> 16 : o2 & 0xFFFFu;
            if (i >= np) continue;
            if (dst + c[h] > total || (x[h] < 0 && t0 + off + c[h] > P.hi - P.shift)) { hdr_selfcheck_failed(P.hdr, P.epoch, 6u, (u32)tile, i, (u32)x[h], dst); continue; }
            const u32 src = (u32)(t0 + off);
            if (x[h] >= 0) out[dst] = x[h];
            else if (c[h] <= 8) {
                int32_t id[8];
#pragma unroll
                for (int kk = 0; kk < 8; kk++) id[kk] = (u32)kk < c[h] ? P.stage[src + kk] : 0;
#pragma unroll
                for (int kk = 0; kk < 8; kk++) if ((u32)kk < c[h]) out[dst + kk] = id[kk];
            } else {
                const u32 slot = atomicAdd(&s_nbig, 1u);
                if (slot < TT_TILE_BYTES / 8) { s_big[slot][0] = src; s_big[slot][1] = dst; s_big[slot][2] = c[h]; }
            }
            if (P.docmask) {
                const long long g = (long long)tile * TT_TILE_BYTES + off;
                if ((P.docmask[g >> 5] >> (g & 31)) & 1) {
                    // every document that starts at this byte (empty ones included) gets this token offset
                    const long long want = g - P.shift;
                    int lo = 0, hi2 = P.n_docs;
                    while (lo < hi2) { int mid = (lo + hi2) >> 1; if (P.doc_off[mid] < want) lo = mid + 1; else hi2 = mid; }
                    for (int d = lo; d <= P.n_docs && P.doc_off[d] == want; d++) P.ids_off_out[d] = dst;
                }
            }
        }
        if (staged || some_big) __syncthreads();                  // (both block-uniform)
        if (some_big) {                                           // pieces of more than 8 tokens
            // a warp each, four loads in flight per lane (one after the other by the whole CTA they took 45 us where most pieces
            // of 3 MB of text have 50 to 100 tokens); the few very long ones by the whole CTA
            const u32 nbig = min(s_nbig, (u32)(TT_TILE_BYTES / 8));
            for (u32 e = 0; e < nbig; e++) {
                const u32 cc = s_big[e][2];
                const bool whole = cc > SCATTER_WARP_MAX;         // block-uniform
                if (!whole && (int)(e % BPE_WARPS) != wid) continue;
                const u32 src = s_big[e][0], d2 = s_big[e][1], step = whole ? (u32)BPE_THREADS : 32u;
                for (u32 k0 = whole ? (u32)tid : (u32)lane; k0 < cc; k0 += 4 * step) {
                    int32_t id[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) id[u] = k0 + u * step < cc ? P.stage[src + k0 + u * step] : 0;
#pragma unroll
                    for (int u = 0; u < 4; u++) if (k0 + u * step < cc) out[d2 + k0 + u * step] = id[u];
                }
            }
            __syncthreads();
            if (tid == 0) s_nbig = 0;                             // (the next item's barrier comes before anyone adds)
        }
        // (not beyond the total that was checked against the capacity, whatever the pieces of the item add up to)
        const u32 leave = carry < total ? min(tot, total - carry) : 0u;
        if (staged) for (u32 kk = tid; kk < leave; kk += BPE_THREADS) P.ids_out[carry + kk] = s_out[kk];
        carry += tot;
        if (tile2 >= tile_hi) break;
        tile = tile2; b = b2; np = np2; v = vn; o2 = on;
    }
}
template <int MINB>
__global__ void __launch_bounds__(BPE_THREADS, MINB)
k_scatter(const __grid_constant__ ScatterParams P) {
    __shared__ ScatterShared SH;
    cudaGridDependencySynchronize();                         // k_merge's (and with it the first kernel's) results are complete from here on
    // The next call's first kernel may be placed from here on; it waits for this grid itself.  (Allowed earlier, while this grid still waits
    // for k_merge, its CTAs -- and those of the call's other kernels -- gathered on the SMs whose k_merge CTA was through first:
    // 150,000 pieces of two bytes, call after call, 177 us instead of 108, 300 KB of short accented words 815 instead of 651;
    // 300 KB of Unicode-heavy text 38.8 instead of 35.5.)
    cudaTriggerProgrammaticLaunchCompletion();
    scatter_tiles(P, SH);
}

// ---- K5 for bulk text: a warp per tile, no barrier after the prologue -----------------------------------------
// Each CTA takes a contiguous range of tiles, its warps every eighth tile of it.  A warp knows where its tile's ids
// go from the token counts of the tiles before it (group totals, then tile counts) and takes the tile's pieces 32 by 32, one per
// lane, the loads of SCATTER_AHEAD such groups in flight: loads and stores are whole lines, a group without merged pieces (two
// thirds of the transcripts' groups) needs no scan, and merged pieces are listed and copied many at a time.  What bounds it is
// instruction issue.  (Four neighbouring pieces per lane, scanned in any case, with their offsets: 132 MB batch 897 us a call, so
// 838; the loop kept short on purpose: unrolled eight times it waited for instructions, 871.)
// SCATTER_BULK_CTAS CTAs per SM: as many as are resident, so that the ranges are one wave (132 MB batch: 5 CTAs 806 us, 6 796, 8 with
// 32 registers 864).
constexpr int SCATTER_BULK_CTAS = 6, SCATTER_AHEAD = 4, SCATTER_LIST = 64, SCATTER_NEXT = 14;
__global__ void __launch_bounds__(BPE_THREADS, SCATTER_BULK_CTAS)
k_scatter_bulk(const __grid_constant__ ScatterParams P) {
    __shared__ unsigned long long s_sum[66];
    __shared__ uint3 s_list[BPE_WARPS][SCATTER_LIST];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const u32 FULL = 0xFFFFFFFFu;
    cudaGridDependencySynchronize();                         // k_merge_bulk's (and with it the kernels' before it) results are complete
    cudaTriggerProgrammaticLaunchCompletion();               // the next call's first kernel may be placed (see k_scatter)
    const int per = (P.ntiles + (int)gridDim.x - 1) / (int)gridDim.x;
    const int tile_lo = (int)blockIdx.x * per, tile_hi = min(P.ntiles, tile_lo + per);
    unsigned long long before = 0, total = 0;
    {
        const int ngroups = (P.ntiles + TT_GROUP_TILES - 1) / TT_GROUP_TILES, g_lo = tile_lo / TT_GROUP_TILES;
        for (int g = tid; g < ngroups; g += BPE_THREADS) { const u32 x = P.grp_tok[g]; total += x; if (g < g_lo) before += x; }
        for (int t = g_lo * TT_GROUP_TILES + tid; t < tile_lo; t += BPE_THREADS) before += P.tile_tok[t];
    }
    cta_sum2_u64(before, total, s_sum);
    int status = hdr_status(P.hdr, P.epoch);
    if (status == 0 && total > P.ids_cap) status = 5;          // TT_ERR_CAPACITY
    if (blockIdx.x == 0 && tid == 0) {
        if (P.status_out) *P.status_out = status;
        if (P.count_out) *P.count_out = status ? 0 : (long long)total;
    }
    if (status != 0) {
        if (P.ids_off_out)
            for (long long d = (long long)blockIdx.x * blockDim.x + tid; d <= P.n_docs; d += (long long)gridDim.x * blockDim.x) P.ids_off_out[d] = 0;
        return;
    }
    if (P.ids_off_out && blockIdx.x == 0) {
        for (int d = P.n_docs - tid; d >= 0 && P.doc_off[d] >= P.hi - P.shift; d -= blockDim.x) P.ids_off_out[d] = (long long)total;
    }
    // tokens of the tiles of this CTA's range before the warp's first tile
    u32 carry = (u32)before;
    {
        const u32 x = (lane < wid && tile_lo + lane < tile_hi) ? P.tile_tok[tile_lo + lane] : 0u;
        carry += __reduce_add_sync(FULL, x);
    }
    const long long len = P.hi - P.shift;
    const u32 total32 = (u32)total;                          // (a text has fewer than 2^31 bytes)
    uint3* const list = s_list[wid];                         // merged pieces that are still to be copied: source, destination, ids
    u32 listed = 0;
    // a lane each, all loads side by side; pieces of more than eight ids by the whole warp, four loads in flight per lane
    const auto copy_listed = [&]() {
        __syncwarp();
#pragma unroll 1
        for (u32 e0 = 0; e0 < listed; e0 += 32) {
            uint3 e = make_uint3(0, 0, 0);
            if (e0 + lane < listed) e = list[e0 + lane];
            const u32 few = e.z <= 8 ? e.z : 0u;
            int32_t id[8];
#pragma unroll
            for (int k = 0; k < 8; k++) id[k] = (u32)k < few ? P.stage[e.x + k] : 0;
#pragma unroll
            for (int k = 0; k < 8; k++) if ((u32)k < few) P.ids_out[e.y + k] = id[k];
#pragma unroll 1
            for (u32 m = __ballot_sync(FULL, e.z > 8); m; m &= m - 1) {                   // warp-uniform
                const int l = __ffs(m) - 1;
                const u32 s2 = __shfl_sync(FULL, e.x, l), d2 = __shfl_sync(FULL, e.y, l), c2 = __shfl_sync(FULL, e.z, l);
#pragma unroll 1
                for (u32 k0 = lane; k0 < c2; k0 += 128) {
                    int32_t x[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) x[u] = k0 + 32 * u < c2 ? P.stage[s2 + k0 + 32 * u] : 0;
#pragma unroll
                    for (int u = 0; u < 4; u++) if (k0 + 32 * u < c2) P.ids_out[d2 + k0 + 32 * u] = x[u];
                }
            }
        }
        listed = 0;
        __syncwarp();
    };
#pragma unroll 1
    for (int tile = tile_lo + wid; tile < tile_hi; tile += BPE_WARPS) {   // warp-uniform
        const u32* const pc = P.piece_cnt + (size_t)tile * TT_TILE_BYTES;
        // the tile's first pieces, asked for before their number is known (the array has a place for every byte)
        u32 v[SCATTER_AHEAD];
#pragma unroll
        for (int g = 0; g < SCATTER_AHEAD; g++) v[g] = pc[32 * g + lane];
        // ... and those of the warp's next tile brought into L2
        if (lane < SCATTER_NEXT && tile + BPE_WARPS < tile_hi) asm volatile("prefetch.global.L2 [%0];" ::"l"(pc + BPE_WARPS * TT_TILE_BYTES + 32 * lane));
        const u32 np = P.tile_cnt[tile];
        // does any document start in this tile?  (few tiles: the pieces of the others need not look)
        const bool tile_has_doc = P.docmask != nullptr && (P.tile_q[tile] & TQ_HAS_DOC) != 0;
        // the seven tiles between this one and the warp's next
        u32 skip = (lane >= 1 && lane < BPE_WARPS && tile + lane < tile_hi) ? P.tile_tok[tile + lane] : 0u;
        const long long t0 = (long long)tile * TT_TILE_BYTES - P.shift;      // text offset of the tile start
        u32 run = carry;
#pragma unroll 1
        for (u32 b = 0; b < np; b += 32) {                                // warp-uniform
            const u32 i = b + lane, x = v[0];
#pragma unroll
            for (int g = 0; g + 1 < SCATTER_AHEAD; g++) v[g] = v[g + 1];
            if (i + 32 * SCATTER_AHEAD < np) v[SCATTER_AHEAD - 1] = pc[i + 32 * SCATTER_AHEAD];
            const bool in = i < np, staged = in && (int32_t)x < 0;
            const u32 m = __ballot_sync(FULL, staged);
            u32 dst = run + lane;
            run += min(32u, np - b);
            if (m) {
                u32 c = in ? 1u : 0u;
                if (staged) { c = (x >> 11) & PIECE_MANY; if (c == PIECE_MANY) c = pc[TT_TILE_BYTES]; }
                u32 inc = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const u32 y = __shfl_up_sync(FULL, inc, o); if (lane >= o) inc += y; }
                dst += inc - c - lane; run = dst - (inc - c) + __shfl_sync(FULL, inc, 31);
                if (staged) {
                    const u32 src = (u32)(t0 + (x & (TT_TILE_BYTES - 1)));
                    const bool fits = c <= total32 && dst <= total32 - c && (long long)src + c <= len;
                    if (!fits) hdr_selfcheck_failed(P.hdr, P.epoch, 7u, (u32)tile, i, x, dst);
                    list[listed + __popc(m & ((1u << lane) - 1))] = make_uint3(src, dst, fits ? c : 0u);
                }
                listed += __popc(m);
                if (listed > SCATTER_LIST - 32) copy_listed();
            }
            if (in && !staged) {
                if (dst < total32) P.ids_out[dst] = (int32_t)x;
                else hdr_selfcheck_failed(P.hdr, P.epoch, 7u, (u32)tile, i, x, dst);
            }
            if (tile_has_doc && in) {
                const long long gpos = (long long)tile * TT_TILE_BYTES + P.piece_off16[(size_t)tile * TT_TILE_BYTES + i];
                if ((P.docmask[gpos >> 5] >> (gpos & 31)) & 1) {
                    // every document that starts at this byte (empty ones included) gets this token offset
                    const long long want = gpos - P.shift;
                    int lo = 0, hi2 = P.n_docs;
                    while (lo < hi2) { int mid = (lo + hi2) >> 1; if (P.doc_off[mid] < want) lo = mid + 1; else hi2 = mid; }
                    for (int d = lo; d <= P.n_docs && P.doc_off[d] == want; d++) P.ids_off_out[d] = dst;
                }
            }
        }
        if (listed > SCATTER_LIST / 4) copy_listed();
        carry = run + __reduce_add_sync(FULL, skip);
    }
    if (listed) copy_listed();
}
