// Step K1: vector loads of UTF-8 text, strict validation, per-code-point class tagging.
//
// One call classifies one aligned 32-byte word of the text and returns, for its 32 bytes, one bit per byte in each of
// the masks below.  Continuation bytes carry the class of their lead byte, so that a maximal run of one class is
// contiguous in byte space (paper Sec. 4.1: character classes and maximal same-class runs; Sec. 4.2: on-device UTF-8
// decoding and character classification).
//
// The 32 bytes are first transposed into eight bit planes (plane k = bit k of every byte), after which a class of ASCII
// characters is a handful of three-input logic operations on whole planes: about 110 instructions for 32 bytes, where
// byte-wise range tests on 32-bit words with the bits gathered afterwards took about 300 for 16.  Only the lead bytes of
// multi-byte characters are visited one by one.
#pragma once
#include "tt_common.cuh"

struct ClassTables {          // pointers into global memory (read through L1)
    const u8* stage1;         // [0x1100]  code point >> 8 -> block
    const u8* stage2;         // [nblocks * 128] two 4-bit class codes per byte
    const u8* ascii;          // [128] class code | (flag << 3); flag: 1 CR/LF, 2 blank, 3 apostrophe, 4 slash
};

struct WordMasks {
    u32 lead;                 // byte starts a code point
    u32 oth, mark, spc, num, low, upp, cless;   // class of the code point the byte belongs to
    u32 nl, sp, ap, sl;       // CR/LF, U+0020, apostrophe, slash (ASCII, single byte)
    u32 bad;                  // byte takes part in a UTF-8 violation
};

// Stage 1 names a block of stage 2, or (from CLS_UNIFORM on) the one class of all 256 code points: CJK and Hangul take one load.
constexpr u32 CLS_UNIFORM = 0xF8;
TT_HD u32 tt_class_of(u32 cp, const ClassTables& T) {
    const u32 blk = T.stage1[cp >> 8];
    if (blk >= CLS_UNIFORM) return blk & 7u;
    const u32 v = T.stage2[blk * 128 + ((cp & 0xFF) >> 1)];
    return (cp & 1) ? (v >> 4) : (v & 15);
}

// Fills the 128-entry ASCII table (used on the host when the vocab is loaded).
inline void tt_fill_ascii_table(u8* t) {
    for (int b = 0; b < 128; b++) {
        u32 code = CC_OTHER;
        if (b >= '0' && b <= '9') code = CC_NUMBER;
        else if (b >= 'a' && b <= 'z') code = CC_LOWER;
        else if (b >= 'A' && b <= 'Z') code = CC_UPPER;
        else if ((b >= 9 && b <= 13) || b == 32) code = CC_SPACE;
        u32 flag = (b == 10 || b == 13) ? 1 : b == 32 ? 2 : b == 39 ? 3 : b == 47 ? 4 : 0;
        t[b] = (u8)(code | (flag << 3));
    }
}

// ---- bit planes ---------------------------------------------------------------------------------------------
TT_HD u32 tt_perm(u32 x, u32 y, u32 sel) {                              // bytes of {x, y} picked by four selector nibbles
#if defined(__CUDA_ARCH__)
    return __byte_perm(x, y, sel);
#else
    const u64 v = ((u64)y << 32) | x;
    u32 r = 0;
    for (int i = 0; i < 4; i++) r |= (u32)((v >> (8 * ((sel >> (4 * i)) & 7))) & 0xFF) << (8 * i);
    return r;
#endif
}
// x = the 32 bytes as eight little-endian words; p[k] bit i <- bit k of byte i.
TT_HD void tt_bit_planes(const u32 (&x)[8], u32 (&p)[8]) {
    // bytes first: word m takes bytes m, 8 + m, 16 + m, 24 + m
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const u32 a = tt_perm(x[h], x[2 + h], 0x5140u), b = tt_perm(x[4 + h], x[6 + h], 0x5140u);
        const u32 c = tt_perm(x[h], x[2 + h], 0x7362u), d = tt_perm(x[4 + h], x[6 + h], 0x7362u);
        p[4 * h] = tt_perm(a, b, 0x5410u); p[4 * h + 1] = tt_perm(a, b, 0x7632u);
        p[4 * h + 2] = tt_perm(c, d, 0x5410u); p[4 * h + 3] = tt_perm(c, d, 0x7632u);
    }
    // then an 8 x 8 bit transposition in every byte lane: blocks of 4, 2 and 1 bits change places
#define TT_SWAP_BLOCKS(i, j, s, M) { const u32 a = p[i], b = p[j]; p[i] = (a & M) | ((b << s) & ~M); p[j] = ((a >> s) & M) | (b & ~M); }
#pragma unroll
    for (int i = 0; i < 4; i++) TT_SWAP_BLOCKS(i, i + 4, 4, 0x0F0F0F0Fu)
#pragma unroll
    for (int i = 0; i < 8; i += 4) { TT_SWAP_BLOCKS(i, i + 2, 2, 0x33333333u) TT_SWAP_BLOCKS(i + 1, i + 3, 2, 0x33333333u) }
#pragma unroll
    for (int i = 0; i < 8; i += 2) TT_SWAP_BLOCKS(i, i + 1, 1, 0x55555555u)
#undef TT_SWAP_BLOCKS
}

// Bytes of the word at global position g0 (aligned frame) that exist, i.e. lie inside [lo, hi).
TT_HD u32 tt_valid_bytes(long long g0, long long lo, long long hi) {
    const long long vlo = lo - g0, vhi = hi - g0;
    if (vlo >= 32 || vhi <= 0) return 0u;
    u32 v = 0xFFFFFFFFu;
    if (vhi < 32) v = (1u << vhi) - 1u;
    if (vlo > 0) v &= ~((1u << vlo) - 1u);
    return v;
}
// The 16 bytes of one vector load with the bytes outside `valid` (16 bits) set to zero.
TT_HD uint4 tt_zero_invalid(uint4 v, u32 valid) {
#define TT_NIB(k) (((((valid >> (k)) & 0xFu) * 0x00204081u) & 0x01010101u) * 0xFFu)
    v.x &= TT_NIB(0); v.y &= TT_NIB(4); v.z &= TT_NIB(8); v.w &= TT_NIB(12);
#undef TT_NIB
    return v;
}

// x: the 32 bytes (those outside the text zero); tx: the same bytes in memory, readable from tx - 4 to tx + 35 and 4-byte
// aligned; valid: the bytes that exist.
TT_HD WordMasks tt_classify_word(const u32 (&x)[8], const u8* tx, u32 valid, const ClassTables& T) {
    u32 p[8];
    tt_bit_planes(x, p);
    const u32 A = ~p[7];                                                // ASCII bytes
    const u32 col2 = A & ~p[6] & p[5] & ~p[4];                          // 0x20 .. 0x2F
    const u32 low3 = p[2] | p[1] | p[0], low4 = p[3] | low3;
    WordMasks m;
    m.sp = col2 & ~low4 & valid;
    m.num = A & ~p[6] & p[5] & p[4] & ~(p[3] & (p[2] | p[1])) & valid;                                  // 0x30 .. 0x39
    const u32 let = A & p[6] & (p[4] | low4) & ~(p[4] & p[3] & (p[2] | (p[1] & p[0]))) & valid;         // 1 .. 26 of columns 4-5, 6-7
    m.low = let & p[5]; m.upp = let & ~p[5];
    const u32 ctl = A & ~(p[6] | p[5] | p[4]) & p[3] & low3 & ~(p[2] & p[1]) & valid;                   // 9 .. 13
    m.spc = ctl | m.sp;
    m.nl = ctl & (p[2] ^ p[1]) & (p[1] ^ p[0]);                                                          // 10 and 13 of them
    const u32 p210 = p[2] & p[1] & p[0] & col2 & valid;
    m.ap = p210 & ~p[3]; m.sl = p210 & p[3];                                                             // 0x27, 0x2F
    m.oth = A & ~(let | m.num | m.spc) & valid;
    m.lead = (A | p[6]) & valid;                                        // all but continuation bytes
    m.mark = 0; m.cless = 0; m.bad = 0;
    // multi-byte characters: their lead bytes in this word and in the three bytes before it
    const u32 before = *reinterpret_cast<const u32*>(tx - 4);
    const u32 lb = (before & (before << 1) & 0x80808000u);             // bytes -3 .. -1 whose top two bits are set
    if ((p[7] & valid) | lb) {
        u32 c0 = 0, c1 = 0, c2 = 0, cov = 0, bad = 0;                   // class code of every covered byte, as three planes
        u64 todo = ((u64)(p[7] & p[6] & valid) << 3) | ((lb >> 15) & 1u) | ((lb >> 22) & 2u) | ((lb >> 29) & 4u);
        while (todo) {
#if defined(__CUDA_ARCH__)
            const int j = __ffsll((long long)todo) - 4;
#else
            const int j = __builtin_ctzll(todo) - 3;
#endif
            todo &= todo - 1;
            const u32* const w = reinterpret_cast<const u32*>(tx) + (j >> 2);
            const u32 sh = (u32)(j & 3) * 8, x0 = w[0], x1 = w[1];
            const u32 v = sh ? (x0 >> sh) | (x1 << (32 - sh)) : x0;     // the lead byte and the three bytes behind it
            const u32 b = v & 0xFFu;
            const int n = b >= 0xF0 ? 4 : b >= 0xE0 ? 3 : 2;
            if (j + n <= 0) continue;                                   // ends before this word
            const u32 b1 = (v >> 8) & 0xFFu, b2 = (v >> 16) & 0xFFu, b3 = v >> 24;
            bool ok = (b >= 0xC2) && (b <= 0xF4) && ((b1 & 0xC0) == 0x80);
            u32 cp = ((b & (0x7Fu >> n)) << 6) | (b1 & 0x3F);
            if (n >= 3) { ok = ok && ((b2 & 0xC0) == 0x80); cp = (cp << 6) | (b2 & 0x3F); }
            if (n >= 4) { ok = ok && ((b3 & 0xC0) == 0x80); cp = (cp << 6) | (b3 & 0x3F); }
            if (n == 3) ok = ok && cp >= 0x800 && !(cp >= 0xD800 && cp <= 0xDFFF);
            if (n == 4) ok = ok && cp >= 0x10000 && cp <= 0x10FFFF;
            const u32 span = (u32)(((u64)((1u << n) - 1u) << (j + 3)) >> 3);   // bytes of this character inside the word
            if (!ok) { bad |= span; continue; }
            const u32 c = tt_class_of(cp, T);
            c0 |= (c & 1) ? span : 0u; c1 |= (c & 2) ? span : 0u; c2 |= (c & 4) ? span : 0u;
            cov |= span;
        }
        cov &= valid;
        static_assert(CC_OTHER == 0 && CC_MARK == 1 && CC_SPACE == 2 && CC_NUMBER == 3 && CC_LOWER == 4 && CC_UPPER == 5 && CC_CASELESS == 6, "planes of the class code");
        m.oth |= cov & ~c2 & ~c1 & ~c0; m.mark = cov & ~c2 & ~c1 & c0; m.spc |= cov & ~c2 & c1 & ~c0; m.num |= cov & ~c2 & c1 & c0;
        m.low |= cov & c2 & ~c1 & ~c0;  m.upp |= cov & c2 & ~c1 & c0;  m.cless = cov & c2 & c1;
        m.bad = (bad | (p[7] & ~p[6] & ~cov)) & valid;                  // (a continuation byte without a lead is bad too)
    }
    return m;
}
