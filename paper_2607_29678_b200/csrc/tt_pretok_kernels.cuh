// Kernels of the pre-tokenization half: document mask, tag + piece-start flags (K1 + K2) with the
// per-tile piece counts and their prefix, and compaction into piece offsets (K3).
#pragma once
#include "tt_pretok.cuh"
#include "tt_pretok_p1.cuh"
#include "tt_bpe.cuh"

// ---- CTA-wide reductions over 256 threads (results broadcast to every thread) ---------------
__device__ __forceinline__ long long cta_max_ll(long long v, long long* scratch /* >= 9 */) {
    for (int o = 16; o; o >>= 1) { long long t = __shfl_xor_sync(0xFFFFFFFFu, v, o); v = t > v ? t : v; }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    long long r = scratch[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); w++) r = scratch[w] > r ? scratch[w] : r;
    return r;
}
__device__ __forceinline__ u32 cta_sum_u32(u32 v, long long* scratch) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    u32 r = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) r += (u32)scratch[w];
    return r;
}
// exclusive prefix of v over the CTA; *total receives the CTA sum
__device__ __forceinline__ u32 cta_exscan_u32(u32 v, u32* scratch /* >= 33 */, u32* total) {
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
    if (total) *total = scratch[32];
    return scratch[wid] + x - v;
}

// ---- document mask ---------------------------------------------------------------------------
// Writes the mask with the bit of every document's first byte (aligned frame), and checks the offsets: they must be ascending,
// start at 0 and end at the total length; a violation is reported as TT_ERR_ARG in the status word.  A CTA writes a stretch of
// DOCMASK_WORDS words: it finds the first document of its stretch by a search in 32 steps at a time.  (Clearing the mask and
// setting bits in it with atomics were two launches, and two gaps, in front of the chain.)  Documents of a few bytes each, of
// which a stretch holds thousands, get shorter stretches (docmask_stretch) and DOCMASK_AHEAD offsets in flight per thread, and
// all CTAs share the check: 400 KB in documents of one byte 207 us a call, so 64.
constexpr int DOCMASK_WORDS = 2048, DOCMASK_WORDS_DENSE = 256, DOCMASK_THREADS = 256, DOCMASK_AHEAD = 8;
// More documents than one round of the loop takes per stretch?
inline int docmask_stretch(long long mask_words, long long n_docs) {
    return n_docs > (long long)DOCMASK_THREADS * DOCMASK_AHEAD * ((mask_words + DOCMASK_WORDS - 1) / DOCMASK_WORDS) ? DOCMASK_WORDS_DENSE : DOCMASK_WORDS;
}
__global__ void __launch_bounds__(DOCMASK_THREADS)
k_docmask(const long long* __restrict__ doc_off, int n_docs, long long shift, long long len, long long nwords, int stretch,
          u32* __restrict__ docmask, TTHeader* hdr, unsigned long long epoch) {
    __shared__ __align__(16) u32 s_mask[DOCMASK_WORDS];
    __shared__ int s_first;
    const int tid = threadIdx.x, lane = tid & 31;
    const u32 FULL = 0xFFFFFFFFu;
    // (No early trigger: bulk text fills every place of the GPU with CTAs that stay, and what was placed beside this grid stayed
    // unevenly spread: 535 -> 558 us for 12 MB.)
    cudaGridDependencySynchronize();                         // the work before this call reads the mask, or writes the offsets
    const long long w0 = (long long)blockIdx.x * stretch;
    const int words = (int)max(0ll, min((long long)stretch, nwords - w0));        // (0: a CTA that only helps to check)
    if (words > 0) {
        for (int i = tid; i < words; i += DOCMASK_THREADS) s_mask[i] = 0;
        const long long from = w0 * 32 - shift, to = min((w0 + words) * 32 - shift, len);          // text bytes of the stretch
        if (tid < 32) {                                       // first document that starts at `from` or behind it
            int lo = 0, hi = n_docs;                          // (the answer is in [lo, hi])
            while (hi > lo) {
                const int step = (hi - lo + 31) / 32, at = lo + lane * step;
                const bool less = at < hi && doc_off[at] < from;
                const int c = __popc(__ballot_sync(FULL, less));                                   // ascending: the first c probes are below
                if (c == 0) hi = lo;
                else { const int l2 = lo + (c - 1) * step + 1; hi = min(hi, lo + c * step); lo = l2; }
            }
            if (lane == 0) s_first = lo;
        }
        __syncthreads();
        for (long long d0 = s_first + tid;; d0 += DOCMASK_THREADS * DOCMASK_AHEAD) {               // by whole warps
            long long o[DOCMASK_AHEAD];
#pragma unroll
            for (int u = 0; u < DOCMASK_AHEAD; u++) { const long long d = d0 + u * DOCMASK_THREADS; o[u] = d < n_docs ? doc_off[d] : to; }
#pragma unroll
            for (int u = 0; u < DOCMASK_AHEAD; u++) {
                const bool in = o[u] >= from && o[u] >= 0 && o[u] < to;
                if (!__any_sync(FULL, in)) continue;
                const int g = in ? (int)(o[u] + shift - w0 * 32) : -1;                             // bit of the stretch
                const u32 bit = in ? 1u << (g & 31) : 0u;
                const int word = g >> 5, before = __shfl_up_sync(FULL, word, 1);
                // neighbouring documents in one word: one lane sets the bits of all
                if (__any_sync(FULL, in && lane > 0 && before == word)) {
                    const u32 peers = __match_any_sync(FULL, word), bits = __reduce_or_sync(peers, bit);
                    if (in && lane == __ffs(peers) - 1) atomicOr(&s_mask[word], bits);
                } else if (in) atomicOr(&s_mask[word], bit);
            }
            if (__any_sync(FULL, o[DOCMASK_AHEAD - 1] >= to)) break;       // ascending: nothing behind it starts in the stretch
        }
    }
    // the check, shared by all CTAs
    for (long long d0 = (long long)blockIdx.x * DOCMASK_THREADS * DOCMASK_AHEAD + tid; d0 <= n_docs; d0 += (long long)gridDim.x * DOCMASK_THREADS * DOCMASK_AHEAD) {
        long long o[DOCMASK_AHEAD], before[DOCMASK_AHEAD];
#pragma unroll
        for (int u = 0; u < DOCMASK_AHEAD; u++) {
            const long long d = d0 + u * DOCMASK_THREADS;
            o[u] = d <= n_docs ? doc_off[d] : 0; before[u] = d > 0 && d <= n_docs ? doc_off[d - 1] : 0;
        }
        bool ok = true;
#pragma unroll
        for (int u = 0; u < DOCMASK_AHEAD; u++) {
            const long long d = d0 + u * DOCMASK_THREADS;
            if (d <= n_docs) ok = ok && o[u] >= before[u] && o[u] <= len && (d > 0 || o[u] == 0) && (d < n_docs || o[u] == len);
        }
        if (!ok) hdr_set_status(hdr, epoch, 1 /* TT_ERR_ARG */);
    }
    __syncthreads();
    for (int i = tid; i < words; i += DOCMASK_THREADS) docmask[w0 + i] = s_mask[i];
}

__device__ __forceinline__ u32 doc_bits(const PretokParams& P, long long word) {
    if (word < 0 || word >= P.nwords) return 0;
    if (P.docmask) return P.docmask[word];
    return word == 0 ? (1u << P.lo) : 0u;                            // (0 <= lo < 16)
}
// Eight words of text of the mask word `word` (zero outside the text).
__device__ __forceinline__ uint4 load_chunk_raw(const PretokParams& P, const u8* rd, long long chunk) {
    return chunk < 0 || chunk >= P.nchunks ? make_uint4(0, 0, 0, 0) : *reinterpret_cast<const uint4*>(rd + chunk * TT_CHUNK);
}
__device__ __forceinline__ uint4 text_of_chunk(const PretokParams& P, uint4 v, long long chunk) {
    if (chunk == 0 || chunk == P.nchunks - 1) {                      // the ends of the text
        const u32 valid = tt_valid_bytes((chunk >> 1) * TT_WORD, P.lo, P.hi);
        v = tt_zero_invalid(v, (chunk & 1) ? valid >> 16 : valid & 0xFFFFu);
    }
    return v;
}
__device__ __forceinline__ uint4 load_chunk(const PretokParams& P, const u8* rd, long long chunk) { return text_of_chunk(P, load_chunk_raw(P, rd, chunk), chunk); }

// ---- bounded CTA-cooperative walks over the text (runs that leave the shared-memory window) ----
// Every loop below advances by a word per thread and iteration and stops at the ends of the text.  All
// positions are in the aligned frame; `gend` is exclusive.

enum { RUN_NUM = 0, RUN_NL = 1, RUN_SL = 2 };
// The walks are rarely executed, so their instructions come from L2 or beyond, a cache line at a time: what a walk
// costs is mostly the size of the code it runs through.  They share one copy of the classifier.
TT_D_COLD WordMasks coop_classify(const PretokParams& P, const ClassTables& T, long long word) {
    const u8* const rd = P.src ? P.src : P.base;
    u32 buf[10];                                                     // the word with four bytes on either side
    const uint4 a = load_chunk(P, rd, 2 * word), b = load_chunk(P, rd, 2 * word + 1);
    const u32 x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int j = 0; j < 8; j++) buf[j + 1] = x[j];
    buf[0] = load_chunk(P, rd, 2 * word - 1).w; buf[9] = load_chunk(P, rd, 2 * word + 2).x;
    return tt_classify_word(x, reinterpret_cast<const u8*>(buf + 1), tt_valid_bytes(word * TT_WORD, P.lo, P.hi), T);
}
constexpr long long COOP_NONE = -(1ll << 60);

__device__ __forceinline__ u32 run_mask(const WordMasks& m, int kind) {
    return kind == RUN_NUM ? m.num : kind == RUN_NL ? m.nl : m.sl;
}
__device__ __forceinline__ u32 below_end(long long word, long long gend) {      // bytes of the word below gend
    return word * TT_WORD + TT_WORD <= gend ? 0xFFFFFFFFu : gend > word * TT_WORD ? (0xFFFFFFFFu >> (int)(word * TT_WORD + TT_WORD - gend)) : 0u;
}

// Most steps of a long walk lie inside the run, and there nothing has to be classified: is the word made of nothing but bytes of one
// plain kind, with no document start in it or right behind it?  (Bytes outside the text are zero.)
enum { PLAIN_NUM = RUN_NUM, PLAIN_NL = RUN_NL, PLAIN_SL = RUN_SL, PLAIN_BLANK = 3 /* not CR/LF */, PLAIN_SAME = 4 /* every byte the one in `same` */ };
__device__ __forceinline__ bool plain_u32(u32 x, int kind, u32 same) {
    if (kind == PLAIN_SAME) return x == same;
    const u32 y = kind == PLAIN_NUM ? tt_swar_range(x, '0', '9') : kind == PLAIN_SL ? tt_swar_range(x, '/', '/')
                : kind == PLAIN_NL ? tt_swar_range(x, '\n', '\n') | tt_swar_range(x, '\r', '\r')
                                   : tt_swar_range(x, '\t', '\t') | tt_swar_range(x, 0x0B, 0x0C) | tt_swar_range(x, ' ', ' ');
    return (x & 0x80808080u) == 0 && y == 0x80808080u;
}
__device__ __forceinline__ bool plain_word(const PretokParams& P, long long word, int kind, u32 same = 0) {
    if (word < 0 || word >= P.nwords) return false;
    const u8* const rd = P.src ? P.src : P.base;
    const uint4 a = load_chunk(P, rd, 2 * word), b = load_chunk(P, rd, 2 * word + 1);
    return plain_u32(a.x, kind, same) && plain_u32(a.y, kind, same) && plain_u32(a.z, kind, same) && plain_u32(a.w, kind, same) &&
           plain_u32(b.x, kind, same) && plain_u32(b.y, kind, same) && plain_u32(b.z, kind, same) && plain_u32(b.w, kind, same) &&
           doc_bits(P, word) == 0 && (doc_bits(P, word + 1) & 1) == 0;
}

// Walks down from gend-1 through bytes of the run class `kind` (cut at document starts).  Returns the
// position of the first byte that is not part of the run, with flags in the low four bits:
// 1 = the run was cut by a document start, 2 = that byte is "other" (4 = a mark), 8 = it is CR/LF.
// *leads receives the number of code-point leads inside the run (RUN_NUM only).
TT_D_COLD long long coop_back_run(const PretokParams& P, const ClassTables& T, long long gend, int kind,
                                   long long* scratch, u32* leads) {
    u32 total = 0;
    long long found = COOP_NONE;
    const long long wtop = (gend + TT_WORD - 1) / TT_WORD;            // words below wtop are examined
    for (long long wb = wtop - (int)blockDim.x;; wb -= (int)blockDim.x) {
        const long long word = wb + threadIdx.x;
        if (wb + (int)blockDim.x < wtop && __syncthreads_and(plain_word(P, word, kind))) { total += blockDim.x * TT_WORD; continue; }    // (a character a byte)
        const WordMasks m = coop_classify(P, T, word);
        const u32 d = doc_bits(P, word), dn = doc_bits(P, word + 1);
        const u32 live = below_end(word, gend);
        // a document start at gend itself does not cut the run (the caller has checked that byte)
        u32 dc = (d >> 1) | (dn << 31);
        if (gend - 1 >= word * TT_WORD && gend - 1 < word * TT_WORD + TT_WORD) dc &= ~(1u << (int)(gend - 1 - word * TT_WORD));
        u32 cut = (~run_mask(m, kind) | dc) & live;
        if (word < 0) cut = live;
        long long pos = COOP_NONE;
        if (cut) {
            const int b = tt_hibit(cut);
            const u32 flags = ((dc >> b) & 1) | (((m.oth >> b) & 1) << 1) | (((m.mark >> b) & 1) << 2) | (((m.nl >> b) & 1) << 3);
            pos = ((word * TT_WORD + b) << 4) | flags;
        }
        const long long top = cta_max_ll(pos, scratch);
        const long long top_pos = top == COOP_NONE ? COOP_NONE : (top >> 4);
        if (leads) {
            u32 mine = 0;
            if (word >= 0 && word * TT_WORD + TT_WORD - 1 > top_pos) {
                u32 keep = live;
                if (top_pos >= word * TT_WORD) keep &= tt_bits_above((int)(top_pos - word * TT_WORD));
                mine = tt_popc(m.lead & run_mask(m, kind) & keep);
            }
            total += cta_sum_u32(mine, scratch);
        }
        if (top != COOP_NONE) { found = top; break; }
        if (wb <= 0) { found = ((long long)-1 << 4) | 1; break; }
    }
    if (leads) *leads = total;
    return found;
}

// Number leads (mod 3) of the number run that ends right before gend.
TT_D_COLD u32 coop_back_num(const PretokParams& P, const ClassTables& T, long long gend, long long* scratch) {
    u32 leads = 0;
    coop_back_run(P, T, gend, RUN_NUM, scratch, &leads);
    return leads % 3;
}
// Is the byte before gend an "other" character, or a CR/LF run glued to one?  (marks count as
// "other" only for pattern 0)
TT_D_COLD u32 coop_back_nl(const PretokParams& P, const ClassTables& T, long long gend, long long* scratch) {
    const long long r = coop_back_run(P, T, gend, RUN_NL, scratch, nullptr);
    if (r & 1) return 0;
    return ((r >> 1) & 1) | (P.pattern != 1 ? ((r >> 2) & 1) : 0);
}
// Pattern 1: is the byte before gend a '/' run (or CR/LF run) that belongs to a punctuation tail?
TT_D_COLD u32 coop_back_slash(const PretokParams& P, const ClassTables& T, long long gend, long long* scratch) {
    const long long r = coop_back_run(P, T, gend, RUN_SL, scratch, nullptr);
    if ((r & 1) || !((r >> 3) & 1)) return 0;                 // cut by a document, or not preceded by CR/LF
    return coop_back_nl(P, T, (r >> 4) + 1, scratch);
}

// Does the whitespace run that continues at word w0 (its first byte) still contain a CR/LF?
TT_D_COLD u32 coop_fwd_nl(const PretokParams& P, const ClassTables& T, long long w0, long long* scratch) {
    for (long long wb = w0;; wb += (int)blockDim.x) {
        const long long word = wb + threadIdx.x;
        if (wb > w0 && __syncthreads_and(plain_word(P, word, PLAIN_BLANK))) continue;
        const WordMasks m = coop_classify(P, T, word);
        const u32 d = doc_bits(P, word);
        const u32 ev = ~m.spc | d | m.nl;                    // bytes past the end are not whitespace
        long long neg = COOP_NONE;
        if (ev) {
            const int j = tt_lobit(ev);
            const u32 is_nl = ((m.nl & m.spc & ~d) >> j) & 1;
            // smallest position wins: negate, keep the answer in the low bit
            neg = -(((word * TT_WORD + j) << 1) | (is_nl ^ 1));
        }
        const long long best = cta_max_ll(neg, scratch);
        if (best != COOP_NONE) return (u32)(((-best) & 1) ^ 1);
        if (wb + (int)blockDim.x >= P.nwords) return 0;
    }
}

// Pattern 1: nearest sure piece start (sure_only) or nearest sure-start / unresolved-construct event
// below gend.  Returns (position << 1) | is_unresolved; the text start is always a sure start.
TT_D_COLD long long coop_back_event(const PretokParams& P, const ClassTables& T, long long gend, bool sure_only,
                                     long long* scratch) {
    // A warp classifies 32 neighbouring words, a lane each, and examines the inner 30, which find their neighbours' masks in the lanes
    // beside them (each thread classifying three words for itself took 18 us a step on Thai-like text).
    const int lane = threadIdx.x & 31, step = 30 * (int)(blockDim.x >> 5);
    const long long wtop0 = (gend + TT_WORD - 1) / TT_WORD;
    for (long long wtop = wtop0;; wtop -= step) {
        const long long wb = wtop - step, word = wb + 30 * (int)(threadIdx.x >> 5) - 1 + lane;
        if (wtop < wtop0) {
            // What a word holds follows from it and its two neighbours.  The step before found nothing: where its lowest words and
            // all of these are one byte over and over, there is nothing here either.
            const u32 c = load_chunk(P, P.src ? P.src : P.base, 2 * wtop).x;
            if (__syncthreads_and(c != 0 && (c & 0x80u) == 0 && (c & 0xFFu) * 0x01010101u == c && plain_word(P, word, PLAIN_SAME, c) &&
                                  (threadIdx.x > 1 || plain_word(P, wtop + 1 + threadIdx.x, PLAIN_SAME, c)))) continue;
        }
        long long pos = COOP_NONE;
        {
            WordDoc p, c, n;
            c.m = coop_classify(P, T, word); c.doc = doc_bits(P, word);
#define NEIGHBOURS(f) p.f = __shfl_up_sync(0xFFFFFFFFu, c.f, 1); n.f = __shfl_down_sync(0xFFFFFFFFu, c.f, 1);
            NEIGHBOURS(doc) NEIGHBOURS(m.lead) NEIGHBOURS(m.oth) NEIGHBOURS(m.mark) NEIGHBOURS(m.spc) NEIGHBOURS(m.num) NEIGHBOURS(m.low) NEIGHBOURS(m.upp)
            NEIGHBOURS(m.cless) NEIGHBOURS(m.nl) NEIGHBOURS(m.sp) NEIGHBOURS(m.ap) NEIGHBOURS(m.sl)
#undef NEIGHBOURS
            p.m.bad = 0; n.m.bad = 0;
            if (word >= 0 && lane >= 1 && lane <= 30) {
                tt_marks_inside_words_cm(p, c, n);
                u32 sure, hard, upcl, apch;
                tt_sure_hard_cm(p, c, n, sure, hard, upcl, apch);
                const u32 ev = (sure | (sure_only ? 0u : hard)) & below_end(word, gend);
                if (ev) { const int b = tt_hibit(ev); pos = ((word * TT_WORD + b) << 1) | (sure_only ? 0u : ((hard >> b) & 1)); }
            }
        }
        const long long top = cta_max_ll(pos, scratch);
        if (top != COOP_NONE) return top;
        if (wb <= 0) return (P.lo << 1);
    }
}

// ---- K1 + K2 -----------------------------------------------------------------------------------
template <int PAT>
__device__ __forceinline__ void store_slot(u32 (*sm)[TT_SLOTS], int s, const WordMasks& m, u32 d) {
    sm[F_LEAD][s] = m.lead; sm[F_SPC][s] = m.spc; sm[F_NUM][s] = m.num; sm[F_NL][s] = m.nl; sm[F_SP][s] = m.sp; sm[F_AP][s] = m.ap; sm[F_DOC][s] = d;
    if (PAT == TT_PATTERN_CUTS) sm[F_CLESS0][s] = m.cless;
    else if (PAT != 1) { sm[F_OTH][s] = m.oth | m.mark; sm[F_LET][s] = m.low | m.upp | m.cless; }
    else { sm[F_OTH][s] = m.oth; sm[F_MARK][s] = m.mark; sm[F_LOW][s] = m.low; sm[F_UPP][s] = m.upp; sm[F_CLESS][s] = m.cless; sm[F_SL][s] = m.sl; }
}

// What the fused kernel needs beyond the piece-start predicate: the per-tile records it leaves (see TTWorkspace)
// and the tables of the whole-piece lookups.
struct FrontParams {
    u32* tile_last; u32* tile_tok; u32* tile_q; u16* tile_long; u16* piece_off16; u32* piece_cnt; u32* q;
    u64* wq;                   // bulk text (more tiles than a request's job search covers): the warp-class pieces of all tiles go
                               // to this one list, appended tile by tile (hdr->nwq, cleared before the chain); else null
    TokTable toktab;           // shorts == nullptr: none
    LongTable longtab;         // ignore_merges: entries longer than the whole-piece table holds (else slots == nullptr)
    const int32_t* ext_id;
};

// A piece on the general path of the fused kernel: a single byte, a vocabulary entry of up to 24 bytes, or
// (ignore_merges) a longer entry.  Returns true and the value for piece_cnt if it needs no merging.
// tb + o: its n bytes in shared memory.
__device__ __forceinline__ bool front_piece_general(const FrontParams& F, const u8* tb, u32 o, u32 n, u32& val) {
    int32_t id;
    if (n == 1) { val = (u32)F.ext_id[tb[o]]; return true; }
    if (n <= (u32)TT_TOKTAB_MAXLEN) {
        if (F.toktab.shorts != nullptr && toktab_lookup(F.toktab, tb, o, n, id)) { val = (u32)id; return true; }
    } else if (F.longtab.slots != nullptr && n <= F.longtab.maxlen && longtab_lookup(F.longtab, tb, o, n, id)) { val = (u32)id; return true; }
    return false;
}
// An unsettled piece (offset o in the tile, index i, n bytes) goes to the tile's queue of its length class.
__device__ __forceinline__ void front_piece_queue(const FrontParams& F, int tile, u32 o, u32 i, u32 n, u32* s_ns, u32* s_nw, u32* s_nl, u16* s_wlist) {
    if (n > (u32)TT_WARP_PIECE_MAX) {
        F.tile_long[(size_t)tile * TT_TILE_LONGCAP + atomicAdd(s_nl, 1u)] = (u16)i;
        if (F.wq != nullptr) { u16* const at = F.piece_off16 + (size_t)tile * TT_TILE_BYTES + i; at[0] = (u16)o; at[1] = (u16)(o + n); }   // (see k_pretok)
    }
    else if (n > (u32)LANE_MAX) {
        const u32 k = atomicAdd(s_nw, 1u);
        if (F.wq != nullptr) s_wlist[k] = (u16)i;
        else F.q[(size_t)tile * TT_TILE_QCAP + (u32)TT_TILE_QCAP - 1 - k] = tile_queue_entry(o, i, n);
    }
    else F.q[(size_t)tile * TT_TILE_QCAP + atomicAdd(s_ns, 1u)] = tile_queue_entry(o, i, n);
}

// FUSED = false: the start flags go to P.startmask, with the pieces per tile (tt_pretokenize and the cut pass of the
// three-splitter composition).
// FUSED = true (the encode chain's first kernel): the tile's flags stay in shared memory and become its list of
// piece offsets (K3); every piece but the tile's last one -- whose end another tile knows -- is settled here if it
// is a single byte, an extracted literal or a whole vocabulary entry (one 32-byte probe), and queued for k_merge
// otherwise.  Everything a tile leaves behind has this CTA as its only writer: no atomics on global memory, no
// counter that would have to be cleared before the call.
// NT = threads per CTA, MINB = CTAs per SM the kernel is compiled for.  A request (at most a few tiles per CTA) is a latency
// chain: 128 threads, so that classification (72 words with the halo) is one step and the look-ups are short, and
// four table look-ups in flight per thread.  Bulk text is bound by instruction issue: 64 threads, as many as a tile has
// words, so that no warp waits idle for the predicate, and one look-up at a time per thread; 18 CTAs per SM leave 56 registers
// (132 MB batch: 16 CTAs 791 us a call, 17 765, 18 763, 19 794, 20 with 48 registers 788; two look-ups in flight 808 to 815).
// PAT = the pattern the kernel is compiled for (P.pattern says the same): each pattern's rules are a lot of code, and a
// kernel that carries all of them keeps missing the instruction caches on its way through the one it runs.
constexpr int PRETOK_THREADS_REQUEST = 128, PRETOK_CTAS_REQUEST = 6, PRETOK_THREADS_BULK = 64, PRETOK_CTAS_BULK = 18, PRETOK_RUN = 8;
template <int PAT> struct PretokSmem {
    static constexpr int ROWS = PAT == 1 ? F_COUNT : F_P0_COUNT;
    // the piece offsets take the place of the masks once the predicate has been evaluated
    static constexpr size_t MASK_BYTES = (size_t)ROWS * TT_SLOTS * sizeof(u32), OFF_BYTES = (TT_TILE_BYTES + 2) * sizeof(u16);
    static constexpr size_t BYTES = ((MASK_BYTES > OFF_BYTES ? MASK_BYTES : OFF_BYTES) + 15) / 16 * 16;
};
// Bulk text: a CTA takes runs of P.run neighbouring tiles and keeps the masks of the last eight slots (the next tile's low halo and
// first word) and the text of the very last, so that 64 threads load and classify 64 words; with the halo taken in anew, one
// warp went through both a second time for eight words while the other waited (132 MB batch 823 -> 809 us).  (Pattern 1 rewrites
// the masks of its window afterwards, and host text is copied tile by tile: P.run is 1 there.)
template <bool FUSED, int NT, int PAT> struct PretokShared {
    static constexpr bool BULK = FUSED && NT == PRETOK_THREADS_BULK, CARRY = BULK && PAT != 1;
    static constexpr int CARRY_ROWS = F_P0_COUNT;
    alignas(16) u8 raw[PretokSmem<PAT>::BYTES];              // class masks of the tile and its halo; later: piece offsets of the tile
    alignas(16) u32 text[4 + TT_SLOTS * 8 + 4];              // the text of the slots, four bytes more on either side
    long long scratch[40];
    u32 need, first, islast, wtot[TT_TILE_WORDS / 32], ns, nw, nl, total, wbase, nslow;
    u16 wlist[TT_TILE_BYTES / (LANE_MAX + 1) + 2];           // bulk text: the tile's warp-class pieces
    u16 slow[TT_TILE_BYTES / 9 + 4];                         // pieces of more than 8 bytes (looked up together)
    u32 carry[CARRY ? CARRY_ROWS * (TT_LOW_HALO + 1) : 1];
};
// The kernel's work once what it reads is complete.
template <bool FUSED, int NT, int PAT>
__device__ __forceinline__ void pretok_tiles(const PretokParams& P, const FrontParams& F, PretokShared<FUSED, NT, PAT>& SH) {
    static_assert(NT >= TT_TILE_WORDS && NT % 32 == 0 && TT_TILE_WORDS % 32 == 0, "a thread per word of the tile, whole warps of them (tt_eval_word_p1 asks the warp)");
    constexpr bool BULK = SH.BULK, CARRY = SH.CARRY;
    constexpr int CARRY_ROWS = SH.CARRY_ROWS;
    static_assert(!CARRY || NT == TT_TILE_WORDS, "the words of a run's later tiles, one per thread");
    u32 (*const sm)[TT_SLOTS] = reinterpret_cast<u32 (*)[TT_SLOTS]>(SH.raw);
    u16* const s_off = reinterpret_cast<u16*>(SH.raw);
    u32 (&s_text)[4 + TT_SLOTS * 8 + 4] = SH.text;
    long long (&scratch)[40] = SH.scratch;
    u32 &s_need = SH.need, &s_first = SH.first, &s_islast = SH.islast, &s_ns = SH.ns, &s_nw = SH.nw, &s_nl = SH.nl, &s_total = SH.total, &s_wbase = SH.wbase, &s_nslow = SH.nslow;
    auto& s_wtot = SH.wtot; auto& s_wlist = SH.wlist; auto& s_slow = SH.slow; auto& s_carry = SH.carry;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (FUSED) {
        if (blockIdx.x == 0 && tid == 0) {                    // k_merge's counters (k_merge touches them only after this grid)
            P.hdr->t_tiles = 0; P.hdr->merge_done = 0;
            for (int s = 0; s < 6; s++) { P.hdr->long_take[s] = 0; P.hdr->long_done[s] = 0; }
            if (F.wq == nullptr) { P.hdr->t_short = 0; P.hdr->nq_long = 0; }
        }
    }
    // The class tables stay in global memory (21 KB, read through L1): ASCII characters -- nearly all of a
    // transcript -- are classified without any table, so shared memory is left to the masks and more CTAs fit an SM.
    ClassTables T;
    T.stage1 = P.cls_tables; T.stage2 = P.cls_tables + 0x1100; T.ascii = P.cls_tables + P.cls_bytes - 128;
    SeqCtx SC;
    // Where the text is read from: the device buffer, or (host calls with pinned text) the caller's host memory.  In
    // the second case the CTA also writes its tile to the device copy, which later kernels (and rare walks) read.
    const u8* const rd = P.src ? P.src : P.base;
    SC.base = rd; SC.lo = P.lo; SC.hi = P.hi; SC.docmask = P.docmask; SC.T = T;
    u32 any_bad = 0;
    u8* const stx = reinterpret_cast<u8*>(s_text + 4);                // byte 0 of slot 0
    const u8* const tb = stx + TT_LOW_HALO * TT_WORD;                 // byte 0 of the tile

    const int run = CARRY ? P.run : 1;
    int left = run;                                               // tiles of the run from this one on
    for (int tile = (int)blockIdx.x * run; tile < P.ntiles; tile += CARRY && --left ? 1 : (left = run, ((int)gridDim.x - 1) * run + 1)) {
        __syncthreads();
        const bool carried = CARRY && left != run;        // the tile before was this CTA's: block-uniform
        if (tid == 0) { s_need = 0; s_first = 0xFFFFFFFFu; s_ns = 0; s_nw = 0; s_nl = 0; s_total = 0; s_nslow = 0; }
        const long long w_first = (long long)tile * TT_TILE_WORDS;    // mask word of the tile's first byte
        // phase A: the text of the tile and its halo into shared memory, a vector load per thread and step
        {
            const long long c0 = 2 * (w_first - TT_LOW_HALO);
            if (carried) {
                // (the threads that are about to replace the text of the high halo and of the word before it keep the one as the tile's
                // first word and the other's last bytes, which a contraction may begin in)
                if (tid == NT - 3) s_text[4 + 8 * TT_LOW_HALO - 1] = s_text[4 + 8 * (TT_SLOTS - 1) - 1];
                if (tid >= NT - 2) *reinterpret_cast<uint4*>(s_text + 4 + 4 * (2 * TT_LOW_HALO + tid - (NT - 2))) = *reinterpret_cast<const uint4*>(s_text + 4 + 4 * (2 * (TT_SLOTS - 1) + tid - (NT - 2)));
                for (int e = tid; e < CARRY_ROWS * (TT_LOW_HALO + 1); e += NT) sm[e / (TT_LOW_HALO + 1)][e % (TT_LOW_HALO + 1)] = s_carry[e];
            }
            for (int c = tid + (carried ? 2 * (TT_LOW_HALO + 1) : 0); c < 2 * TT_SLOTS; c += NT) {
                const uint4 v = load_chunk_raw(P, rd, c0 + c);
                *reinterpret_cast<uint4*>(s_text + 4 + 4 * c) = text_of_chunk(P, v, c0 + c);
                if (P.src && c >= 2 * TT_LOW_HALO && c < 2 * (TT_LOW_HALO + TT_TILE_WORDS) && c0 + c < P.nchunks) *reinterpret_cast<uint4*>(P.copy + (c0 + c) * TT_CHUNK) = v;
            }
            if (tid == NT - 1 && !carried) s_text[3] = load_chunk(P, rd, c0 - 1).w;
            if (tid == NT - 2) s_text[4 + TT_SLOTS * 8] = load_chunk(P, rd, c0 + 2 * TT_SLOTS).x;
        }
        __syncthreads();
        // phase B: classify, a word per thread and step
        for (int s = tid + (carried ? TT_LOW_HALO + 1 : 0); s < TT_SLOTS; s += NT) {
            const long long word = w_first - TT_LOW_HALO + s;
            const uint4 a = *reinterpret_cast<const uint4*>(s_text + 4 + 8 * s), b = *reinterpret_cast<const uint4*>(s_text + 8 + 8 * s);
            const u32 x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            const u32 valid = tt_valid_bytes(word * TT_WORD, P.lo, P.hi);
            const WordMasks m = tt_classify_word(x, stx + s * TT_WORD, valid, T);
            const u32 d = doc_bits(P, word);
            store_slot<PAT>(sm, s, m, d);
            if (s >= TT_LOW_HALO && (CARRY || s < TT_LOW_HALO + TT_TILE_WORDS)) any_bad |= m.bad | (d & ~m.lead & valid & ~m.bad);
        }
        __syncthreads();
        if (PAT == 1) {                                          // marks inside words count as caseless letters from here on
            constexpr int STEPS = (TT_SLOTS + NT - 1) / NT;
            u32 in[STEPS];
#pragma unroll
            for (int k = 0; k < STEPS; k++) { const int s = tid + k * NT; in[k] = s < TT_SLOTS ? tt_marks_inside_words(sm, s) : 0u; }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < STEPS; k++) { const int s = tid + k * NT; if (in[k]) { sm[F_MARK][s] &= ~in[k]; sm[F_CLESS][s] |= in[k]; } }
            __syncthreads();
            // sure starts / unresolved constructs per slot
            const long long gs0 = (w_first - TT_LOW_HALO) * TT_WORD;        // byte 0 of slot 0
            for (int s = tid; s < TT_SLOTS - 1; s += NT) {
                if (s == 0) continue;
                u32 su, ha;
                tt_sure_hard(sm, s, su, ha, rd, gs0, P.hi);
                sm[F_SURE][s] = su; sm[F_HARD][s] = ha;
            }
            __syncthreads();
        }
        // phase C: evaluate the piece-start predicate, a thread per word of the tile
        TileCarry tc;
        tc.n_before = 0; tc.nl_absorbed_before = 0; tc.nl_later_after = 0; tc.slash_absorbed_before = 0;
        tc.dirty_before = 0; tc.sure_before = P.lo;
        const int slot = tid + TT_LOW_HALO;
        const bool has_word = NT == TT_TILE_WORDS || tid < TT_TILE_WORDS;
        const long long g0 = (w_first + tid) * TT_WORD;
        const u8* const tx = tb + tid * TT_WORD;
        u32 need = 0, S = 0;
        for (int pass = 0; pass < 2; pass++) {                        // the second one only where an aggregate leaves the window
            if (has_word)
                S = PAT == TT_PATTERN_CUTS ? tt_eval_word_cuts(sm, slot, tc, pass != 0, need)
                  : PAT != 1 ? tt_eval_word_p0(sm, slot, tx, rd, g0, P.hi, tc, pass != 0, need, PAT == 2, P.docmask)
                             : tt_eval_word_p1(sm, slot, tx, SC, g0, tc, pass != 0, need);
            if (pass) break;
            if (need) atomicOr(&s_need, need);
            __syncthreads();
            const u32 need_all = s_need;
            if (!need_all) break;                                     // block-uniform
            const long long below = (w_first - TT_LOW_HALO) * TT_WORD;     // first byte of the low halo
            if (need_all & NEED_N) tc.n_before = coop_back_num(P, T, below, scratch);
            if (need_all & NEED_A) tc.nl_absorbed_before = coop_back_nl(P, T, below, scratch);
            if (PAT == 1 && (need_all & NEED_S)) tc.slash_absorbed_before = coop_back_slash(P, T, below, scratch);
            if (need_all & NEED_F) tc.nl_later_after = coop_fwd_nl(P, T, w_first + TT_TILE_WORDS + 1, scratch);
            if (PAT == 1 && (need_all & (NEED_H | NEED_C))) {
                // events of slot 0 (first halo word) are not examined by the walks in shared memory
                const long long gend = below + TT_WORD;
                const long long ev = coop_back_event(P, T, gend, false, scratch);
                tc.dirty_before = (u32)(ev & 1);
                tc.sure_before = (ev & 1) ? (coop_back_event(P, T, (ev >> 1) + 1, true, scratch) >> 1) : (ev >> 1);
            }
            need = 0;
        }
        if (P.litstart && has_word && w_first + tid < P.nwords)       // an extracted literal is one piece whatever the pattern says
            S = (S & ~P.litin[w_first + tid]) | P.litstart[w_first + tid];
        if (!FUSED) {
            if (has_word && w_first + tid < P.nwords) P.startmask[w_first + tid] = S;
            if (S) atomicMin(&s_first, (u32)(tid * TT_WORD + tt_lobit(S)));
            u32 total = cta_sum_u32(tt_popc(S), scratch);
            if (tid == 0) { P.tile_cnt[tile] = total; P.tile_first[tile] = s_first; }
            continue;
        }
        // ---- K3 in shared memory: the tile's piece offsets ------------------------------------------------------
        const u32 cnt = tt_popc(S);
        u32 x = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const u32 t = __shfl_up_sync(0xFFFFFFFFu, x, o); if (lane >= o) x += t; }
        if (has_word && lane == 31) s_wtot[wid] = x;
        bool has_doc = false;                                         // bulk text: a document starts in the tile
        if (CARRY) for (int e = tid; e < CARRY_ROWS * (TT_LOW_HALO + 1); e += NT) s_carry[e] = sm[e / (TT_LOW_HALO + 1)][TT_TILE_WORDS + e % (TT_LOW_HALO + 1)];
        if (BULK) has_doc = __syncthreads_or(sm[F_DOC][slot] != 0);
        else __syncthreads();                                         // (the masks have been read: their place is free)
        u32 np = 0, r = x - cnt;
#pragma unroll
        for (int w = 0; w < TT_TILE_WORDS / 32; w++) { const u32 v = s_wtot[w]; np += v; if (w < wid) r += v; }
        for (u32 m = S; m; m &= m - 1) s_off[r++] = (u16)(tid * TT_WORD + tt_lobit(m));
        __syncthreads();
        const size_t p0 = (size_t)tile * TT_TILE_BYTES;              // pieces are indexed per tile
        u32 may_long = 0;
        // (bulk text: the offsets of a tile are asked for only where a document starts in it, and those of long pieces)
        if (!BULK || has_doc) for (u32 i = tid; i < np; i += NT) F.piece_off16[p0 + i] = s_off[i];
        if (tid == 0) {
            P.tile_cnt[tile] = np;
            P.tile_first[tile] = np ? (u32)s_off[0] : TT_NONE;
            F.tile_last[tile] = np ? (u32)s_off[np - 1] : TT_NONE;
            // a piece of more than 256 bytes that crosses a tile boundary leaves 129 bytes before it or 128 behind it
            const u32 used = (u32)min((long long)TT_TILE_BYTES, P.hi - w_first * TT_WORD);
            may_long = np == 0 || s_off[0] >= 128 || used - s_off[np - 1] > 128 ? TQ_MAY_LONG : 0u;
        }
        // ---- K4, first half: whole-piece lookups, a thread per piece, LW pieces per thread and step, their buckets
        // fetched side by side.  Pieces of at most 8 bytes -- most of them -- take a path of their own: two key words, a
        // table of 16-byte slots.  The text comes from shared memory.  The tile's last piece is left to k_merge.
        const long long gt = w_first * TT_WORD;                       // the tile's first byte, aligned frame
        const u32 nlook = np ? np - 1 : 0;
        const bool quick = F.toktab.shorts != nullptr;               // block-uniform
        const u32* const tw = reinterpret_cast<const u32*>(tb);
        u32 wsum = 0;
        constexpr int LW = NT == PRETOK_THREADS_REQUEST ? 4 : 1;        // look-ups in flight per thread
        for (u32 ib = tid; ib < nlook; ib += LW * NT) {
            u32 o[LW], n[LW], k0[LW], k1[LW], h[LW];
            uint4 sl[LW], sm2[LW];
            bool lit[LW];
#pragma unroll
            for (int j = 0; j < LW; j++) {
                const u32 i = ib + j * NT;
                o[j] = 0; n[j] = 0;
                if (i < nlook) { o[j] = s_off[i]; n[j] = (u32)s_off[i + 1] - o[j]; }
                k0[j] = 0; k1[j] = 0; h[j] = 0; sl[j] = make_uint4(0, 0, 0, 0); sm2[j] = sl[j]; lit[j] = false;
                if (P.litstart != nullptr && n[j] != 0) lit[j] = (P.litstart[(gt + o[j]) >> 5] >> ((gt + o[j]) & 31)) & 1;
                if (quick && n[j] != 0 && n[j] <= TT_TOKTAB_SHORT) {
                    const u32* const w = tw + (o[j] >> 2);
                    toktab_key01(w[0], w[1], w[2], o[j] & 3, n[j], k0[j], k1[j]);
                    h[j] = toktab_hash_final(toktab_hash_short(F.toktab, k0[j], k1[j], n[j]));
                    ldg_sector(F.toktab.shorts + 2 * (size_t)toktab_bucket(h[j], F.toktab.short_shift), sl[j], sm2[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < LW; j++) {
                const u32 i = ib + j * NT;
                if (n[j] == 0) continue;
                bool settled = false;
                u32 val = 0;
                if (lit[j]) { val = BULK ? piece_staged_word(o[j], 1u) : 0u - 1u; settled = true; }         // one staged id (written by the literal pass)
                else if (quick && n[j] <= TT_TOKTAB_SHORT) settled = toktab_short(F.toktab, sl[j], sm2[j], h[j], n[j], k0[j], k1[j], val);
                else if (quick) { s_slow[atomicAdd(&s_nslow, 1u)] = (u16)i; continue; }     // longer pieces: together, below
                else settled = front_piece_general(F, tb, o[j], n[j], val);
                if (settled) { F.piece_cnt[p0 + i] = val; wsum++; }
                else front_piece_queue(F, tile, o[j], i, n[j], &s_ns, &s_nw, &s_nl, s_wlist);
            }
        }
        if (quick) {                                                  // block-uniform: the pieces of more than 8 bytes, a thread each
            __syncthreads();
            const u32 nslow = s_nslow;
            for (u32 e = tid; e < nslow; e += NT) {
                const u32 i = s_slow[e], o = s_off[i], n = (u32)s_off[i + 1] - o;
                u32 val = 0;
                if (front_piece_general(F, tb, o, n, val)) { F.piece_cnt[p0 + i] = val; wsum++; }
                else front_piece_queue(F, tile, o, i, n, &s_ns, &s_nw, &s_nl, s_wlist);
            }
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) wsum += __shfl_xor_sync(0xFFFFFFFFu, wsum, o);
        if (lane == 0 && wsum) atomicAdd(&s_total, wsum);
        __syncthreads();
        if (tid == 0) {
            F.tile_tok[tile] = s_total;
            F.tile_q[tile] = may_long | (BULK && has_doc ? TQ_HAS_DOC : 0u) | (s_nl ? TQ_MAY_LONG : 0u) | s_ns | ((F.wq != nullptr ? 0u : s_nw) << TQ_NW_SHIFT) | (s_nl << TQ_NL_SHIFT);
            if (F.wq != nullptr && s_nw) s_wbase = atomicAdd(&P.hdr->nwq, s_nw);
        }
        if (F.wq != nullptr && s_nw) {                                // block-uniform
            __syncthreads();
            for (u32 k = tid; k < s_nw; k += NT) {
                const u32 i = s_wlist[k];
                F.wq[s_wbase + k] = ((u64)(u32)tile << 32) | tile_queue_entry(s_off[i], i, (u32)s_off[i + 1] - s_off[i]);
            }
        }
    }
    if (any_bad) hdr_set_status(P.hdr, P.epoch, 4 /* TT_ERR_INVALID_UTF8 */);

    // the last CTA to finish turns the tile counts into their exclusive prefix (only where the piece list is
    // materialised: the encode chain indexes its pieces per tile and needs no prefix)
    if (FUSED || !P.want_prefix) return;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_islast = (atomicAdd(&P.hdr->pretok_done, 1u) == gridDim.x - 1);
    __syncthreads();
    if (s_islast) {
        __threadfence();
        u32* sc = reinterpret_cast<u32*>(scratch);
        u32 carry = 0;
        for (int b0 = 0; b0 < P.ntiles; b0 += blockDim.x) {
            int i = b0 + tid;
            u32 v = i < P.ntiles ? P.tile_cnt[i] : 0, tot;
            u32 ex = cta_exscan_u32(v, sc, &tot);
            if (i < P.ntiles) P.tile_cnt[i] = carry + ex;
            carry += tot;
            __syncthreads();
        }
        if (tid == 0) { P.tile_cnt[P.ntiles] = carry; P.hdr->n_pieces = carry; }
    }
}
template <bool FUSED, int NT, int MINB, int PAT>
__global__ void __launch_bounds__(NT, MINB)
k_pretok(const __grid_constant__ PretokParams P, const __grid_constant__ FrontParams F) {
    __shared__ PretokShared<FUSED, NT, PAT> SH;
    cudaTriggerProgrammaticLaunchCompletion();               // the next kernel may be placed; it waits for this grid's memory itself
    // the whole-piece table is probed at random a few microseconds from now: ask for it to be brought into L2
    if (FUSED && F.toktab.shorts != nullptr) grid_prefetch_l2(F.toktab.shorts, F.toktab.bytes);
    cudaGridDependencySynchronize();                         // what was enqueued before this call is complete: its text, its use of the workspace
    pretok_tiles<FUSED, NT, PAT>(P, F, SH);
}

// ---- K3: compaction of the start flags into piece offsets (tt_pretokenize) --------------------------
// piece_off[i] = byte offset (relative to the text) of piece i; piece_off[n_pieces] = len.  The encode
// chain does the same per tile in shared memory (the fused half of k_pretok) and keeps the offsets per tile.
__global__ void __launch_bounds__(TT_TILE_WORDS)
k_compact(const u32* __restrict__ startmask, const u32* __restrict__ tile_base, long long nwords, int ntiles,
          long long shift, long long len, u32* __restrict__ piece_off, TTHeader* hdr, unsigned long long epoch) {
    __shared__ u32 sc[40];
    if (hdr_status(hdr, epoch) != 0) return;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long word = (long long)tile * TT_TILE_WORDS + threadIdx.x;
        u32 m = word < nwords ? startmask[word] : 0;
        u32 r = tile_base[tile] + cta_exscan_u32(tt_popc(m), sc, nullptr);
        const long long g0 = word * TT_WORD - shift;
        while (m) { int i = tt_lobit(m); m &= m - 1; piece_off[r++] = (u32)(g0 + i); }
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) piece_off[tile_base[ntiles]] = (u32)len;
}
