// Steps K2 and K3: run-local piece-start rules and stream compaction.
//
// Paper Sec. 4.1: whether a character begins a piece depends only on its offset within its
// maximal same-class run, a few characters of look-back across the run boundary, and per-run
// aggregates of whitespace runs (run start, first non-CR/LF position, last CR/LF position); the
// test is an independent per-character predicate.  Here one thread evaluates the predicate for the
// 32 bytes of its word as bit-parallel operations on class masks (bit i <-> byte i), with the bits that
// enter from the words before and after it funnelled in.  Aggregates that reach further (offset mod 3 inside a number
// run, CR/LF runs glued to preceding punctuation, "is there a CR/LF later in this whitespace run")
// are resolved by walking the words' masks in shared memory and, beyond the tile, by a bounded
// CTA-cooperative walk over the text itself -- no CTA ever waits for another CTA.
#pragma once
#include "tt_classify.cuh"

// Rows of masks in shared memory, a word per slot.
enum { F_LEAD = 0, F_OTH, F_SPC, F_NUM, F_NL, F_SP, F_AP, F_DOC,
       F_LET, F_P0_COUNT,                                // patterns 0 and 2: all letters (F_OTH includes the marks there)
       F_CLESS0 = F_LET,                                 // the cut pass of pattern 3: caseless letters
       F_LOW = F_LET, F_UPP, F_CLESS, F_MARK, F_SL,      // pattern 1
       F_SURE, F_HARD,                                   // pattern 1: sure piece starts / unresolved constructs, filled after classification
       F_COUNT };
constexpr int TT_LOW_HALO = 7;                          // words below the tile (look-back context, 224 bytes)
constexpr int TT_SLOTS = TT_TILE_WORDS + TT_LOW_HALO + 1;    // low halo, tile, one high halo word
typedef const u32 (*MaskRows)[TT_SLOTS];

enum { NEED_N = 1, NEED_A = 2, NEED_F = 4, NEED_S = 8, NEED_H = 16, NEED_C = 32 };

struct PretokParams {
    const u8* base;          // 16-byte aligned address at or below the text
    const u8* src;           // null, or the same frame in pinned host memory that the device can read: the kernel then takes the
    u8* copy;                // text from there and leaves a copy of every 16-byte chunk, whole, at `copy` (= base) for all that reads the text later
    long long lo, hi;        // the text occupies [lo, hi) in the aligned frame
    long long nchunks;       // ceil(hi / 16): vector loads
    long long nwords;        // ceil(hi / 32): mask words
    int ntiles;
    int run;                 // neighbouring tiles that a CTA takes one after the other (see CARRY in k_pretok)
    int pattern;
    const u32* docmask;      // bit per byte (aligned frame) marking document starts, or null (one document)
    const u32* litstart;     // literal pass: first bytes of extracted literals (each becomes exactly one piece), or null
    const u32* litin;        //               their other bytes (start nothing)
    u32* startmask;          // out (flags-only kernel): one u32 per word
    u32* tile_cnt;           // out: pieces per tile; flags-only kernel with want_prefix: replaced by the exclusive prefix (ntiles + 1)
    u32* tile_first;         // out: offset inside the tile of its first piece start, or ~0 if it has none
    int want_prefix;         // turn tile_cnt into its exclusive prefix and count the pieces (tt_pretokenize only)
    TTHeader* hdr;
    unsigned long long epoch; // of this call (see TTHeader)
    const u8* cls_tables;    // stage1 | stage2 | ascii, contiguous in global memory
    int cls_bytes;
};

struct TileCarry {           // aggregates of runs that enter or leave the shared-memory window
    u32 n_before;            // number leads (mod 3) of the number run ending right before the low halo
    u32 nl_absorbed_before;  // the CR/LF run ending right before the low halo is glued to punctuation
    u32 nl_later_after;      // the whitespace run leaving the high halo word still contains a CR/LF
    u32 slash_absorbed_before;   // pattern 1: the '/' run ending right before the low halo is part of a punctuation tail
    u32 dirty_before;        // pattern 1: an unresolved construct lies between the last sure piece start and the low halo
    long long sure_before;   // pattern 1: position (aligned frame) of the last sure piece start before the low halo
};

TT_HD int tt_hibit(u32 x) {   // position of the highest set bit, x != 0
#if defined(__CUDA_ARCH__)
    return 31 - __clz(x);
#else
    return 31 - __builtin_clz(x);
#endif
}
TT_HD int tt_lobit(u32 x) {   // position of the lowest set bit, x != 0
#if defined(__CUDA_ARCH__)
    return __ffs(x) - 1;
#else
    return __builtin_ctz(x);
#endif
}
TT_HD int tt_popc(u32 x) {
#if defined(__CUDA_ARCH__)
    return __popc(x);
#else
    return __builtin_popcount(x);
#endif
}
TT_HD u32 tt_brev(u32 x) {
#if defined(__CUDA_ARCH__)
    return __brev(x);
#else
    u32 r = 0;
    for (int i = 0; i < 32; i++) r |= ((x >> i) & 1u) << (31 - i);
    return r;
#endif
}
// Mask of a word moved up by k places (bit i <- bit i - k), the top bits of the word before it entering; 1 <= k <= 31.
TT_HD u32 tt_up(u32 before, u32 x, int k) {
#if defined(__CUDA_ARCH__)
    return __funnelshift_l(before, x, k);
#else
    return (x << k) | (before >> (32 - k));
#endif
}
// Moved down by k places (bit i <- bit i + k), the low bits of the word after it entering.
TT_HD u32 tt_down(u32 x, u32 after, int k) {
#if defined(__CUDA_ARCH__)
    return __funnelshift_r(x, after, k);
#else
    return (x >> k) | (after << (32 - k));
#endif
}
TT_HD u32 tt_bits_above(int b) { return b >= 31 ? 0u : 0xFFFFFFFFu << (b + 1); }      // bits b + 1 .. 31

// Number leads in the number run that ends at the last byte of slot `s` (walking down).
// Returns the count; sets `open` when the run continues below slot 0.
TT_HD u32 tt_walk_back_num(MaskRows sm, int s, bool& open) {
    u32 cnt = 0;
    open = false;
    for (; s >= 0; s--) {
        const u32 n = sm[F_NUM][s], d = sm[F_DOC][s], ld = sm[F_LEAD][s];
        const u32 cut = ~n | (d >> 1);              // byte j ends the walk if it is not a number byte or j+1 starts a document
        if (cut) return cnt + tt_popc(ld & n & tt_bits_above(tt_hibit(cut)));
        cnt += tt_popc(ld & n);
        if (d & 1) return cnt;                      // run starts at a document start
    }
    open = true;
    return cnt;
}

// Is the CR/LF run that ends at bit `top` of slot `s` glued to a preceding punctuation char?
// (0 / 1; `open` when the run continues below slot 0.)
TT_HD u32 tt_walk_back_nl(MaskRows sm, int s, bool& open, int top = 31) {
    open = false;
    u32 keep = 0xFFFFFFFFu >> (31 - top);
    for (; s >= 0; s--, keep = 0xFFFFFFFFu) {
        const u32 nl = sm[F_NL][s], d = sm[F_DOC][s];
        const u32 cut = (~nl | (d >> 1)) & keep;
        if (cut) {
            const int b = tt_hibit(cut);
            if (((d >> 1) >> b) & 1) return 0;      // the run starts at a document start
            return (sm[F_OTH][s] >> b) & 1;
        }
        if (d & 1) return 0;
    }
    open = true;
    return 0;
}

// The whitespace run that continues at the first byte of slot `s`: does it still contain a CR/LF?
TT_HD u32 tt_walk_fwd_nl(MaskRows sm, int s, bool& open) {
    open = false;
    for (; s < TT_SLOTS; s++) {
        const u32 w = sm[F_SPC][s], nl = sm[F_NL][s], d = sm[F_DOC][s];
        const u32 ev = ~w | d | nl;
        if (ev) return ((nl & w & ~d) >> tt_lobit(ev)) & 1;
    }
    open = true;
    return 0;
}

// For a word of four bytes below 0x80, tt_swar_ge(y, c) has the top bit of a byte set exactly where that byte is
// >= c (1 <= c <= 0x80): the byte-wise sums stay below 0x100, so nothing carries from byte to byte.  A range is
// ge(lo) & ~ge(hi + 1).
TT_HD u32 tt_swar_ge(u32 y, u32 c) { return y + (0x80u - c) * 0x01010101u; }
TT_HD u32 tt_swar_range(u32 y, u32 lo, u32 hi) { return tt_swar_ge(y, lo) & ~tt_swar_ge(y, hi + 1) & 0x80808080u; }

// The same question asked of the raw text from byte g on (the run has left the shared-memory window):
// 1 / 0 = answered from ASCII bytes alone, -1 = undecided (a non-ASCII byte, which may be whitespace, or more
// than `limit` bytes of blanks).  A document start cuts the run.  One thread, plain loads.
TT_HD int tt_raw_fwd_nl(const u8* base, long long g, long long hi, const u32* docmask, int limit = 256) {
    int k = 0;
    // sixteen bytes at a time while they are all blanks other than CR/LF and no document starts among them (g is a
    // multiple of 16 for every caller; `base` is 16-byte aligned)
    if ((g & 15) == 0) {
        for (; k + 16 <= limit && g + 16 <= hi; k += 16, g += 16) {
            const uint4 v = *reinterpret_cast<const uint4*>(base + g);
            const u32 w[4] = {v.x, v.y, v.z, v.w};
            bool plain = ((v.x | v.y | v.z | v.w) & 0x80808080u) == 0;
            if (docmask) plain = plain && reinterpret_cast<const u16*>(docmask)[g >> 4] == 0;
#pragma unroll
            for (int j = 0; j < 4; j++)
                plain = plain && (tt_swar_range(w[j], 0x09, 0x09) | tt_swar_range(w[j], 0x0B, 0x0C) | tt_swar_range(w[j], ' ', ' ')) == 0x80808080u;
            if (!plain) break;
        }
    }
    for (; k < limit; k++, g++) {
        if (g >= hi) return 0;
        if (docmask && ((docmask[g >> 5] >> (g & 31)) & 1)) return 0;        // the run is cut by a document start
        const u32 b = base[g];
        if (b == '\n' || b == '\r') return 1;
        if (b >= 0x80) return -1;
        if (!(b == ' ' || (b >= 0x09 && b <= 0x0C))) return 0;
    }
    return -1;
}

// Contraction suffix length at the apostrophe whose two following bytes are b1, b2 (0 = none).
TT_HD int tt_contraction_len(u32 b1, u32 b2) {
    const u32 a = b1 | 0x20, b = b2 | 0x20;       // ASCII case fold; no other byte maps onto these letters
    if (a == 's' || a == 't' || a == 'm' || a == 'd') return 2;
    if ((a == 'r' && b == 'e') || (a == 'v' && b == 'e') || (a == 'l' && b == 'l')) return 3;
    return 0;
}

// Number runs of the word in `slot`: every third number lead counted from the start of its run.  pN = the bytes whose
// predecessor in the same document is a number byte.
TT_HD u32 tt_number_starts(MaskRows sm, int slot, u32 N, u32 lead, u32 pN, const TileCarry& tc, bool have_tc, u32& need) {
    u32 m = N & lead;
    if (!m) return 0;
    const u32 nstart = N & ~pN, R = N & pN;          // run starts / bytes that continue a run
    u32 cnt = 0;
    if (R & 1) {                                     // a run enters from the word before
        bool open;
        cnt = tt_walk_back_num(sm, slot - 1, open);
        if (open) { if (have_tc) cnt += tc.n_before; else need |= NEED_N; }
        cnt %= 3;
    }
    if (m == N) {
        // every number a single byte: the starts spread upwards in steps of 3, 6, 12 and 24 as long as nothing but
        // continuing bytes lie in between
        u32 s = nstart;
        if (R & 1) {
            const u32 k = cnt ? 3u - cnt : 0u, through = (2u << k) - 1u;
            if ((R & through) == through) s |= 1u << k;
        }
        u32 J = R & (R << 1) & (R << 2);
        s |= (s << 3) & J;  J &= J << 3;
        s |= (s << 6) & J;  J &= J << 6;
        s |= (s << 12) & J; J &= J << 12;
        s |= (s << 24) & J;
        return s;
    }
    u32 S = 0;
    while (m) {
        const int i = tt_lobit(m); m &= m - 1;
        if ((nstart >> i) & 1) cnt = 0;
        if (cnt == 0) S |= 1u << i;
        cnt = cnt == 2 ? 0 : cnt + 1;
    }
    return S;
}

// Characters right behind a CR/LF of a whitespace run (cand) that no later CR/LF of the same run follows: they begin a piece.
// W, NL, D = masks of the word; base: the text, g0: position of the word's first byte.
TT_HD u32 tt_after_last_newline(MaskRows sm, int slot, u32 cand, u32 W, u32 NL, u32 D, const u8* base, long long g0, long long hi,
                                const u32* docmask, const TileCarry& tc, bool have_tc, u32& need) {
    const u32 U = W & ~D, g = U & NL;                // U: bytes that continue the run of the byte before them
    const u32 r = tt_brev(U), s = tt_brev(g);
    const u32 Z = tt_brev((r & ~(r + s)) | s);       // bytes of U that have a CR/LF at or above them (the carry runs down from it)
    const u32 later = Z >> 1;
    const u32 nU = ~U;
    const u32 top = nU ? 0xFFFFFFFFu << tt_hibit(nU) : 0xFFFFFFFFu;     // bytes whose run goes on through bit 31
    u32 S = cand & ~later & ~top;
    const u32 open_bits = cand & ~later & top;
    if (open_bits) {
        bool open;
        u32 more = tt_walk_fwd_nl(sm, slot + 1, open);
        if (open) {
            const int raw = tt_raw_fwd_nl(base, g0 + (long long)(TT_SLOTS - slot) * TT_WORD, hi, docmask);
            if (raw >= 0) more = (u32)raw;
            else if (have_tc) more = tc.nl_later_after;
            else { need |= NEED_F; more = 1; }
        }
        if (!more) S |= open_bits;
    }
    return S;
}

// First two stages of the three-splitter composition (paper Sec. 4.1: three splitters applied in sequence
// fold into the same per-character predicate, provided each splitter re-splits every piece of the stage
// before it and unmatched spans survive as pieces): number groups of up to three digits and runs of
// caseless letters are isolated.  Returns the cut bits of the word in `slot`: a bit where a span of
// these two stages begins.  The third stage (pattern 0) then runs with the cuts as document boundaries,
// i.e. on every span as a text of its own.
constexpr int TT_PATTERN_CUTS = 100;              // internal pattern id of this pass
#define OWN(f) sm[f][slot]
#define BEF(f) sm[f][slot - 1]
#define AFT(f) sm[f][slot + 1]
TT_HD u32 tt_eval_word_cuts(MaskRows sm, int slot, const TileCarry& tc, bool have_tc, u32& need) {
    const u32 lead = OWN(F_LEAD), N = OWN(F_NUM), C = OWN(F_CLESS0), D = OWN(F_DOC), nD = ~D;
    const u32 pN = tt_up(BEF(F_NUM), N, 1) & nD, pC = tt_up(BEF(F_CLESS0), C, 1) & nD;
    u32 S = D;
    S |= lead & ~N & pN;                             // first character after a number run
    S |= C & lead & ~pC;                             // a run of caseless letters begins
    S |= lead & ~C & pC;                             // first character after such a run
    S |= tt_number_starts(sm, slot, N, lead, pN, tc, have_tc, need);
    return S & lead;
}

// Pattern 0 (cl100k-style).  Returns the start bits of the word in `slot`; `need` receives the
// NEED_* flags of aggregates that leave the shared-memory window (then `tc` must be filled and the
// function called again).  tx: the word's bytes (readable two bytes beyond it), base / g0: the text and the position of
// the word's first byte in it.
TT_HD u32 tt_eval_word_p0(MaskRows sm, int slot, const u8* tx, const u8* base, long long g0, long long hi,
                          const TileCarry& tc, bool have_tc, u32& need, bool single_digits = false,
                          const u32* docmask = nullptr) {
    const u32 lead = OWN(F_LEAD), L = OWN(F_LET), N = OWN(F_NUM), W = OWN(F_SPC), O = OWN(F_OTH), NL = OWN(F_NL), D = OWN(F_DOC);
    const u32 nD = ~D;
    const u32 Lb = BEF(F_LET), Nb = BEF(F_NUM), Wb = BEF(F_SPC), Ob = BEF(F_OTH), SPb = BEF(F_SP), NLb = BEF(F_NL), Db = BEF(F_DOC), leadb = BEF(F_LEAD);
    const u32 V = L | N | W | O;                       // bytes that exist and are valid
    const u32 cont = V & ~lead, contb = (Lb | Nb | Wb | Ob) & ~leadb;
    const u32 pO = tt_up(Ob, O, 1) & nD, pNL = tt_up(NLb, NL, 1) & nD;
    // punctuation runs: start of the run, unless a blank precedes it (the blank starts the piece); Gb: the same for the last
    // bytes of the word before (its bit 0 is not needed)
    const u32 G = O & lead & ~pO & ~(tt_up(SPb, OWN(F_SP), 1) & nD);
    const u32 Gb = Ob & leadb & ~(((Ob | SPb) << 1) & ~Db);
    u32 S = G;
    // letter runs: the run start, unless non-CR/LF whitespace or a single match-start punctuation char precedes it
    u32 pfx = tt_up(Gb, G, 1);
    if (cont | contb) {
        const u32 c1 = tt_up(contb, cont, 1), c2 = tt_up(contb, cont, 2), c3 = tt_up(contb, cont, 3);
        pfx |= (tt_up(Gb, G, 2) & c1) | (tt_up(Gb, G, 3) & c2 & c1) | (tt_up(Gb, G, 4) & c3 & c2 & c1);
    }
    S |= L & lead & ~((tt_up(Lb, L, 1) | (tt_up(Wb, W, 1) & ~pNL) | pfx) & nD);
    // contractions: apostrophe that is a match start, then s/t/m/d or re/ve/ll; the letter after the suffix starts a piece
    u32 ga = G & OWN(F_AP) & 0x3FFFFFFFu, gb = Gb & BEF(F_AP) & 0xE0000000u;       // bytes -3 .. 29 can put a start into this word
    while (ga | gb) {
        int p;
        if (gb) { p = tt_lobit(gb) - 32; gb &= gb - 1; } else { p = tt_lobit(ga); ga &= ga - 1; }
        const u32 d = p < 0 ? tt_up(Db, D, -p) : D >> p;                           // bit k: a document starts k bytes behind the apostrophe
        const u32 b1 = (d >> 1) & 1 ? 0u : tx[p + 1], b2 = (d >> 2) & 1 ? 0u : tx[p + 2];     // (bytes outside the text are zero)
        const int cl = tt_contraction_len(b1, b2);
        if (cl && (u32)(p + cl) < 32u && ((d >> 1) & ((1u << cl) - 1)) == 0) S |= (1u << (p + cl)) & L & lead;
    }
    // number runs: every third number lead counted from the run start (single-digit variant: every lead)
    if (single_digits) S |= N & lead;
    else S |= tt_number_starts(sm, slot, N, lead, tt_up(Nb, N, 1) & nD, tc, have_tc, need);
    // whitespace runs
    if (W) {
        const u32 Wa = AFT(F_SPC), Da = AFT(F_DOC), Va = AFT(F_LET) | AFT(F_NUM) | Wa | AFT(F_OTH);
        // (a) run start, unless it is a CR/LF glued to preceding punctuation
        S |= W & lead & ~(tt_up(Wb, W, 1) & nD) & ~(pO & NL);
        // (b) CR/LF absorbed by preceding punctuation: CR/LF runs that begin right after punctuation
        u32 prev_absorbed = 0;                             // byte before the word is an absorbed CR/LF
        if ((NLb >> 31) && !(D & 1)) {
            bool open;
            prev_absorbed = tt_walk_back_nl(sm, slot - 1, open);
            if (open) { if (have_tc) prev_absorbed = tc.nl_absorbed_before; else need |= NEED_A; }
        }
        const u32 nlq = NL & nD;
        const u32 sel = (NL & ~pNL & pO) | (nlq & prev_absorbed);          // (prev_absorbed is 0 or 1: bit 0)
        const u32 absorbed = nlq & ~(nlq + sel);
        S |= W & lead & ~NL & ((absorbed << 1) | prev_absorbed) & nD;
        // (c) last character of the run when something follows in the same document (and it is not CR/LF)
        const u32 nDn = ~tt_down(D, Da, 1);
        const u32 wend = W & nDn & tt_down(V & ~W, Va & ~Wa, 1);
        u32 last = wend;
        const u32 ca = Va & ~AFT(F_LEAD);
        if ((W & ~lead) | (Wa & ca & 7u)) {                // multi-byte blanks: their lead byte
            const u32 wenda = Wa & ~(Da >> 1) & ((Va & ~Wa) >> 1);        // (exact in the bits that are used)
            const u32 k1 = tt_down(cont, ca, 1), k2 = tt_down(cont, ca, 2), k3 = tt_down(cont, ca, 3);
            last |= (tt_down(wend, wenda, 1) & k1) | (tt_down(wend, wenda, 2) & k1 & k2) | (tt_down(wend, wenda, 3) & k1 & k2 & k3);
        }
        S |= lead & W & ~NL & last;
        // (d) first character after the last CR/LF of the run
        const u32 cand = W & lead & ~NL & pNL;
        if (cand) S |= tt_after_last_newline(sm, slot, cand, W, NL, D, base, g0, hi, docmask, tc, have_tc, need);
    }
    return S & lead;
}
#undef OWN
#undef BEF
#undef AFT
