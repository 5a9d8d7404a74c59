// Added-token literal pass (paper Sec. 4.3 / 4.4): added and special tokens are literal strings that map to one
// reserved id each; a leftmost-longest pass extracts them before the tokenizer family handles the segments in
// between.  Two kernels prepare what the ordinary chain then consumes:
//   k_lit_scan    for every byte the longest literal that matches there (its length goes to
//                 cand[], its id to stage[] at the byte's text offset);
//   k_lit_select  leftmost-longest selection.  A candidate that no other candidate overlaps from the left is
//                 selected on its own; a chain of overlapping candidates is walked by the thread of its first
//                 member (each selected literal suppresses the candidates it covers, the next candidate behind
//                 it is selected in turn).  A selected literal becomes a document of its own in the boundary
//                 mask (so the segments around it are tokenized as independent texts), its first byte is
//                 marked in litstart and its other bytes in litin.
// Where no match can overlap another -- no literal holds, behind its first byte, a byte that any of them begins with, as with
// "<|user|>" and its like -- every match is selected, and one kernel writes the masks at once (k_lit_mark).
// k_pretok then forces exactly one piece per literal (start bit at its first byte, none inside) and, in its look-up
// half, takes the staged id for a piece that begins at a litstart bit.
#pragma once
#include "tt_classify.cuh"

struct LitEntry { u32 first4, next4, off_len; int32_t id; };         // the first eight bytes (zero behind the end), offset in the blob << 8 | length
TT_HD u32 lit_len(const LitEntry& e) { return e.off_len & 0xFFu; }
struct LitTable {
    const LitEntry* entries;     // sorted by length, longest first
    const u8* blob;              // the literals' bytes
    u32 n;
    u32 maxlen;
    u32 first_byte[8];           // bit b set: some literal begins with byte b
    u32 second_byte[8];          // bit b set: some literal has b as its second byte, or only one byte
    bool apart;                  // no literal holds a byte with which one begins behind its first: matches never overlap
};

struct LitParams {
    const u8* base;              // aligned frame origin (text = base + lo)
    long long lo, hi;
    LitTable tab;
    u8* cand;                    // [hi + 1] aligned frame: length of the longest literal starting at the byte, 0 = none
    int32_t* stage;              // text offsets: id of that literal
    u32* docmask; u32* litstart; u32* litin;     // bit per byte, aligned frame (written whole by k_lit_mark, else cleared by k_lit_scan)
};

// A thread takes 16 bytes: nearly none of them begins a literal, so what counts is one load and one store for all of them.  (A
// thread per byte took 8.9 us for 300 KB, and clearing the three masks three memsets more in front of it.)
constexpr int LIT_THREADS = 128;
constexpr u32 LIT_AHEAD = 8;
static_assert(sizeof(LitEntry) == 16, "read as one vector");
// Length and id of the longest literal that begins at byte g, whose byte begins one; 0: none.
__device__ __forceinline__ u32 lit_longest(const LitParams& P, const u32* s_second, long long g, int32_t& id) {
    const u32 avail = (u32)min((long long)P.tab.maxlen, P.hi - g);
    u32 w = P.base[g], w2 = 0;
    for (u32 k = 1; k < 4 && k < avail; k++) w |= (u32)P.base[g + k] << (8 * k);
    if (P.tab.n < LIT_AHEAD) {                       // few literals: one by one, first four bytes first
        for (u32 e = 0; e < P.tab.n; e++) {
            const LitEntry L = P.tab.entries[e];
            const u32 len = lit_len(L), off = L.off_len >> 8;
            if (len > avail) continue;
            const u32 m = len >= 4 ? 0xFFFFFFFFu : (1u << (8 * len)) - 1;
            if ((w & m) != L.first4) continue;
            u32 k = 4;
            while (k < len && P.tab.blob[off + k] == P.base[g + k]) k++;
            if (k >= len) { id = L.id; return len; }
        }
        return 0;
    }
    const u32 b1 = (w >> 8) & 0xFFu;
    if (!((s_second[b1 >> 5] >> (b1 & 31)) & 1u)) return 0;
    if (avail > 4) for (u32 k = 4; k < 8 && k < avail; k++) w2 |= (u32)P.base[g + k] << (8 * (k - 4));
    const auto begins = [&](const LitEntry& L) {     // the first eight bytes agree
        const u32 len = lit_len(L);
        return len <= avail && (((w ^ L.first4) & (len >= 4 ? 0xFFFFFFFFu : (1u << (8 * len)) - 1)) |
                                ((w2 ^ L.next4) & (len >= 8 ? 0xFFFFFFFFu : len > 4 ? (1u << (8 * (len - 4))) - 1 : 0u))) == 0;
    };
    u32 found = 0;
    const auto take = [&](const LitEntry& L) {       // ... and the others: the literal stands here
        const u32 len = lit_len(L), off = L.off_len >> 8;
        u32 k = 8;
        while (k < len && P.tab.blob[off + k] == P.base[g + k]) k++;
        if (k < len) return false;
        id = L.id; found = len;
        return true;
    };
    // Longest first: the first match is the longest.  LIT_AHEAD entries at once: what a byte costs is the chain of its look-ups (300
    // KB of transcripts with 2,000 literals, entry by entry 556 us, so 175; 2,000 that all begin the text, 1,240 and 420).
    u32 e = 0;
    for (; e + LIT_AHEAD <= P.tab.n && !found; e += LIT_AHEAD) {
        uint4 x[LIT_AHEAD];
#pragma unroll
        for (u32 u = 0; u < LIT_AHEAD; u++) x[u] = __ldg(reinterpret_cast<const uint4*>(P.tab.entries) + e + u);
        u32 maybe = 0;
#pragma unroll
        for (u32 u = 0; u < LIT_AHEAD; u++) maybe |= (begins(LitEntry{x[u].x, x[u].y, x[u].z, (int32_t)x[u].w}) ? 1u : 0u) << u;
        for (; maybe && !found; maybe &= maybe - 1) take(P.tab.entries[e + (u32)__ffs(maybe) - 1]);
    }
    for (; e < P.tab.n && !found; e++) { const LitEntry L = P.tab.entries[e]; if (begins(L)) take(L); }
    return found;
}
// Which of the 16 bytes of a chunk may begin a literal.
__device__ __forceinline__ u32 lit_hits(const LitParams& P, const u32* s_first, long long g0) {
    const uint4 v = *reinterpret_cast<const uint4*>(P.base + g0);
    const u32 x[4] = {v.x, v.y, v.z, v.w};
    u32 hits = 0;
#pragma unroll
    for (int i = 0; i < TT_CHUNK; i++) { const u32 b = (x[i >> 2] >> (8 * (i & 3))) & 0xFFu; hits |= ((s_first[b >> 5] >> (b & 31)) & 1u) << i; }
    return hits & tt_valid_bytes(g0, P.lo, P.hi);
}

__global__ void __launch_bounds__(LIT_THREADS)
k_lit_scan(const __grid_constant__ LitParams P) {
    __shared__ u32 s_first[8], s_second[8];
    cudaTriggerProgrammaticLaunchCompletion();
    if (threadIdx.x < 8) { s_first[threadIdx.x] = P.tab.first_byte[threadIdx.x]; s_second[threadIdx.x] = P.tab.second_byte[threadIdx.x]; }
    __syncthreads();
    cudaGridDependencySynchronize();                         // the work before this call: its text, its use of the masks
    const long long nchunks = (P.hi + TT_CHUNK - 1) / TT_CHUNK, nwords = P.hi / 32 + 4;
    const long long step = (long long)gridDim.x * LIT_THREADS, first = (long long)blockIdx.x * LIT_THREADS + threadIdx.x;
    for (long long w = first; w < nwords; w += step) { P.docmask[w] = 0; P.litstart[w] = 0; P.litin[w] = 0; }
    for (long long c = first; c < nchunks; c += step) {
        const long long g0 = c * TT_CHUNK;
        u32 hits = lit_hits(P, s_first, g0);                 // bytes that may begin a literal
        *reinterpret_cast<uint4*>(P.cand + g0) = make_uint4(0, 0, 0, 0);
        for (; hits; hits &= hits - 1) {
            const long long g = g0 + __ffs(hits) - 1;
            int32_t id = 0;
            const u32 len = lit_longest(P, s_second, g, id);
            if (len) { P.cand[g] = (u8)len; P.stage[g - P.lo] = id; }
        }
    }
}

__device__ __forceinline__ void lit_set_bits(u32* mask, long long from, long long to) {      // bits [from, to)
    while (from < to) {
        const long long wend = ((from >> 5) + 1) << 5, e = to < wend ? to : wend;
        const u32 bits = (e - from >= 32) ? 0xFFFFFFFFu : (((1u << (int)(e - from)) - 1) << (from & 31));
        atomicOr(&mask[from >> 5], bits);
        from = e;
    }
}

// Is some candidate q in (g - maxlen, g) long enough to cover byte g?
__device__ __forceinline__ bool lit_covered(const LitParams& P, long long g) {
    const long long lo = g - (long long)P.tab.maxlen + 1 > P.lo ? g - (long long)P.tab.maxlen + 1 : P.lo;
    for (long long q = g - 1; q >= lo; q--) {
        const u32 l = P.cand[q];
        if (l && q + l > g) return true;
    }
    return false;
}

// The text's literals one by one, by the thread of their chunk.
__global__ void __launch_bounds__(LIT_THREADS)
k_lit_select(const __grid_constant__ LitParams P) {
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();                         // the candidates are complete from here on
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&P.docmask[P.lo >> 5], 1u << (P.lo & 31));      // the text itself starts a document
    const long long nchunks = (P.hi + TT_CHUNK - 1) / TT_CHUNK;
    for (long long c = (long long)blockIdx.x * LIT_THREADS + threadIdx.x; c < nchunks; c += (long long)gridDim.x * LIT_THREADS) {
      const uint4 v = *reinterpret_cast<const uint4*>(P.cand + c * TT_CHUNK);
      if ((v.x | v.y | v.z | v.w) == 0) continue;
      for (int i = 0; i < TT_CHUNK; i++) {
        const long long g0 = c * TT_CHUNK + i;
        if (g0 < P.lo || g0 >= P.hi || !P.cand[g0] || lit_covered(P, g0)) continue;           // only the first member of a chain works
        long long g = g0;
        for (;;) {                                                 // bounded by the text length: g strictly grows
            const long long end = g + P.cand[g];
            lit_set_bits(P.litstart, g, g + 1);
            lit_set_bits(P.litin, g + 1, end);
            lit_set_bits(P.docmask, g, g + 1);
            if (end < P.hi) lit_set_bits(P.docmask, end, end + 1);
            // the next candidate at or behind `end`, if it belongs to this chain (something before it covers it)
            long long r = end;
            const long long stop = end + (long long)P.tab.maxlen < P.hi ? end + (long long)P.tab.maxlen : P.hi;
            while (r < stop && !P.cand[r]) r++;
            if (r >= stop || !lit_covered(P, r)) break;            // none near, or it heads a chain of its own
            g = r;
        }
      }
    }
}

// Both at once where matches never overlap: a CTA writes the masks of 2 KB of text whole, from the matches that begin there and those
// that reach in from the bytes before (at most maxlen of them, looked at again), so that nothing is cleared in front and no
// candidates pass through memory: one dependent launch where there were two (300 KB of transcripts with five markers 43.2 -> 36.6 us).
constexpr int LIT_TILE_CHUNKS = 128, LIT_TILE_WORDS = LIT_TILE_CHUNKS / 2, LIT_HALO = 256 / TT_CHUNK;
constexpr int LIT_MARK_THREADS = LIT_TILE_CHUNKS + 32;       // a chunk each, those before the stretch by the last warp
static_assert(LIT_HALO <= 32, "a lane each");
__global__ void __launch_bounds__(LIT_MARK_THREADS)
k_lit_mark(const __grid_constant__ LitParams P) {
    __shared__ u32 s_first[8], s_second[8], s_doc[LIT_TILE_WORDS], s_start[LIT_TILE_WORDS], s_in[LIT_TILE_WORDS];
    const int tid = threadIdx.x;
    cudaTriggerProgrammaticLaunchCompletion();
    if (tid < 8) { s_first[tid] = P.tab.first_byte[tid]; s_second[tid] = P.tab.second_byte[tid]; }
    cudaGridDependencySynchronize();                         // the work before this call: its text, its use of the masks
    const long long nchunks = (P.hi + TT_CHUNK - 1) / TT_CHUNK, nwords = P.hi / 32 + 4;
    const long long reach = (long long)P.tab.maxlen;         // (a literal's end marks the byte behind it, too)
    for (long long w0 = (long long)blockIdx.x * LIT_TILE_WORDS; w0 < nwords; w0 += (long long)gridDim.x * LIT_TILE_WORDS) {
        const long long t0 = w0 * 32;                         // the stretch's first byte, aligned frame
        if (tid < LIT_TILE_WORDS) { s_doc[tid] = w0 + tid == (P.lo >> 5) ? 1u << (P.lo & 31) : 0u; s_start[tid] = 0; s_in[tid] = 0; }      // the text itself starts a document
        __syncthreads();
        const int k = tid < LIT_TILE_CHUNKS ? tid : tid - LIT_TILE_CHUNKS - 32;
        const long long c = t0 / TT_CHUNK + k, g0 = c * TT_CHUNK;
        if (c >= 0 && c < nchunks && g0 + TT_CHUNK + reach > t0) {
            for (u32 hits = lit_hits(P, s_first, g0); hits; hits &= hits - 1) {
                const long long g = g0 + __ffs(hits) - 1;
                if (g + reach < t0) continue;
                int32_t id = 0;
                const u32 len = lit_longest(P, s_second, g, id);
                if (len == 0) continue;
                const int at = (int)(g - t0), end = at + (int)len;            // (at < 0: it begins before the stretch)
                if (at >= 0) {
                    P.stage[g - P.lo] = id;
                    atomicOr(&s_start[at >> 5], 1u << (at & 31)); atomicOr(&s_doc[at >> 5], 1u << (at & 31));
                }
                for (int b = max(at + 1, 0); b < min(end, 32 * LIT_TILE_WORDS);) {
                    const int n = min(32 - (b & 31), min(end, 32 * LIT_TILE_WORDS) - b);
                    atomicOr(&s_in[b >> 5], (n == 32 ? 0xFFFFFFFFu : (1u << n) - 1u) << (b & 31));
                    b += n;
                }
                if (end >= 0 && end < 32 * LIT_TILE_WORDS && t0 + end < P.hi) atomicOr(&s_doc[end >> 5], 1u << (end & 31));
            }
        }
        __syncthreads();
        if (tid < LIT_TILE_WORDS && w0 + tid < nwords) { P.docmask[w0 + tid] = s_doc[tid]; P.litstart[w0 + tid] = s_start[tid]; P.litin[w0 + tid] = s_in[tid]; }
        __syncthreads();
    }
}
