// Span export: byte and character spans of the tokens of an encoded text.
//
// Paper App. E.3: the IDs gather per-token byte lengths, a cumulative sum yields byte offsets, and a
// second cumulative sum over the non-continuation text bytes lifts them to character offsets.  The
// tokens of a text concatenate to exactly its bytes, so the number of non-continuation bytes inside a
// token is a property of the token itself; both sums therefore run over per-token table values and the
// text is never read (its length only checks that the IDs belong to it).
#pragma once
#include "tt_common.cuh"
#include "tt_bpe.cuh"

// A block of SPAN_BLOCK tokens is a CTA's, four neighbouring tokens a thread's, so that four table entries are on their way at
// once.  Pass 1 leaves the sums of every block (SPAN_BAD where an id is unknown); in pass 2 every CTA adds up what lies before
// its blocks, and all of it for the check of the length.  Nothing has to be cleared and nobody waits for a last CTA (a
// memset, a scan by the last CTA and two scans per block made the pair 15.5 us behind a 1M-char request: now 10).
constexpr int SPAN_THREADS = 256, SPAN_PER_THREAD = 4, SPAN_BLOCK = SPAN_THREADS * SPAN_PER_THREAD;
constexpr u32 SPAN_BAD = 0xFFFFFFFFu;          // as a block's bytes (no text is that long)

struct SpanParams {
    const int32_t* ids;
    const long long* count;    // DEVICE: number of ids
    unsigned long long ids_cap;
    unsigned long long text_len;
    const uint2* meta;         // per caller id: (byte length, non-continuation bytes); length 0 = unknown id
    u32 meta_n;
    uint2* blk;                // per block of SPAN_BLOCK tokens: (bytes, chars)
    int32_t* byte_off;         // out [count + 1]
    int32_t* char_off;         // out [count + 1]
    int32_t* status_out;
};

__device__ __forceinline__ uint2 span_meta_of(const uint2* meta, u32 meta_n, int32_t id, bool& bad) {
    uint2 m = make_uint2(0, 0);
    if (id >= 0 && (u32)id < meta_n) m = meta[id];
    if (m.x == 0) bad = true;
    return m;
}
// The four tokens from i0 on: their lengths, zero behind the last one.
__device__ __forceinline__ void span_load(const SpanParams& P, unsigned long long i0, unsigned long long n, uint2 (&m)[SPAN_PER_THREAD], bool& bad) {
    int32_t id[SPAN_PER_THREAD];
    if (i0 + SPAN_PER_THREAD <= n && ((uintptr_t)P.ids & 15) == 0) {
        const int4 v = __ldcg(reinterpret_cast<const int4*>(P.ids + i0));
        id[0] = v.x; id[1] = v.y; id[2] = v.z; id[3] = v.w;
    } else {
#pragma unroll
        for (int u = 0; u < SPAN_PER_THREAD; u++) id[u] = i0 + u < n ? __ldcg(P.ids + i0 + u) : 0;
    }
#pragma unroll
    for (int u = 0; u < SPAN_PER_THREAD; u++) { m[u] = make_uint2(0, 0); if (i0 + u < n) m[u] = span_meta_of(P.meta, P.meta_n, id[u], bad); }
}
__device__ __forceinline__ u64 span_pack(uint2 m) { return (u64)m.x | ((u64)m.y << 32); }

// Pass 1: (bytes, chars) per block of tokens.
__global__ void __launch_bounds__(SPAN_THREADS)
k_span_sums(const __grid_constant__ SpanParams P) {
    __shared__ u64 s_sum[SPAN_THREADS / 32];
    cudaGridDependencySynchronize();                         // the ids and their count
    cudaTriggerProgrammaticLaunchCompletion();               // (not earlier: k_span_write reads them before it waits)
    const long long cnt = __ldcg(P.count);
    const unsigned long long n = cnt < 0 || (unsigned long long)cnt > P.ids_cap ? 0 : (unsigned long long)cnt;
    const unsigned long long nblk = (n + SPAN_BLOCK - 1) / SPAN_BLOCK;
    for (unsigned long long b = blockIdx.x; b < nblk; b += gridDim.x) {
        uint2 m[SPAN_PER_THREAD];
        bool bad = false;
        span_load(P, b * SPAN_BLOCK + SPAN_PER_THREAD * threadIdx.x, n, m, bad);
        u64 x = 0;
#pragma unroll
        for (int u = 0; u < SPAN_PER_THREAD; u++) x += span_pack(m[u]);
#pragma unroll
        for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
        if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = x;
        const bool any_bad = __syncthreads_or(bad);
        if (threadIdx.x == 0) {
            x = 0;
#pragma unroll
            for (int w = 0; w < SPAN_THREADS / 32; w++) x += s_sum[w];
            P.blk[b] = make_uint2(any_bad ? SPAN_BAD : (u32)x, (u32)(x >> 32));
        }
        __syncthreads();
    }
}

// Pass 2: offsets of every token.
__global__ void __launch_bounds__(SPAN_THREADS)
k_span_write(const __grid_constant__ SpanParams P) {
    __shared__ unsigned long long s_part[3 * (SPAN_THREADS / 32)];
    __shared__ u64 s_sum[2][SPAN_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    cudaTriggerProgrammaticLaunchCompletion();
    // The ids and their count are complete: every CTA of k_span_sums has waited for them before this grid was let in.  So the lengths
    // of the first block's tokens are fetched while k_span_sums runs (past L1, which may hold what these buffers held before;
    // a request of 1M chars with its spans 42.0 -> 40.4 us).
    const long long cnt = __ldcg(P.count);
    const bool bad_count = cnt < 0 || (unsigned long long)cnt > P.ids_cap;
    const unsigned long long n = bad_count ? 0 : (unsigned long long)cnt;
    const unsigned long long nblk = (n + SPAN_BLOCK - 1) / SPAN_BLOCK, per = (nblk + gridDim.x - 1) / gridDim.x;
    const unsigned long long b_lo = per * blockIdx.x, b_hi = min(nblk, b_lo + per);
    unsigned long long before_b = 0, before_c = 0, total = 0;
    bool bad = bad_count;
    uint2 m[SPAN_PER_THREAD];
    bool unknown = false;                                    // (k_span_sums has told)
    span_load(P, b_lo * SPAN_BLOCK + SPAN_PER_THREAD * tid, b_lo < b_hi ? n : 0, m, unknown);
    cudaGridDependencySynchronize();                         // the blocks' sums
    for (unsigned long long b = tid; b < nblk; b += SPAN_THREADS) {
        const uint2 x = P.blk[b];
        bad |= x.x == SPAN_BAD;
        total += x.x;
        if (b < b_lo) { before_b += x.x; before_c += x.y; }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) { total += __shfl_xor_sync(0xFFFFFFFFu, total, o); before_b += __shfl_xor_sync(0xFFFFFFFFu, before_b, o); before_c += __shfl_xor_sync(0xFFFFFFFFu, before_c, o); }
    if (lane == 0) { s_part[3 * wid] = total; s_part[3 * wid + 1] = before_b; s_part[3 * wid + 2] = before_c; }
    bad = __syncthreads_or(bad);
    total = before_b = before_c = 0;
#pragma unroll
    for (int w = 0; w < SPAN_THREADS / 32; w++) { total += s_part[3 * w]; before_b += s_part[3 * w + 1]; before_c += s_part[3 * w + 2]; }
    const int status = bad || total != P.text_len ? 8 /* TT_ERR_BAD_IDS */ : 0;      // (the ids have to spell a text of this length)
    if (blockIdx.x == 0 && tid == 0) {
        *P.status_out = status;
        if (status != 0 || n == 0) { P.byte_off[0] = 0; P.char_off[0] = 0; }
    }
    if (status != 0) return;
    u64 carry = before_b | (before_c << 32);
    const bool wide = (((uintptr_t)P.byte_off | (uintptr_t)P.char_off) & 15) == 0;
    for (unsigned long long b = b_lo; b < b_hi; b++) {
        const unsigned long long i0 = b * SPAN_BLOCK + SPAN_PER_THREAD * tid;
        if (b != b_lo) span_load(P, i0, n, m, unknown);
        u64 mine = 0;
#pragma unroll
        for (int u = 0; u < SPAN_PER_THREAD; u++) mine += span_pack(m[u]);
        u64 x = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const u64 t = __shfl_up_sync(0xFFFFFFFFu, x, o); if (lane >= o) x += t; }
        if (lane == 31) s_sum[b & 1][wid] = x;
        __syncthreads();
        u64 at = carry + x - mine;
#pragma unroll
        for (int w = 0; w < SPAN_THREADS / 32; w++) { const u64 t = s_sum[b & 1][w]; carry += t; if (w < wid) at += t; }
        int32_t bo[SPAN_PER_THREAD], co[SPAN_PER_THREAD];
#pragma unroll
        for (int u = 0; u < SPAN_PER_THREAD; u++) { bo[u] = (int32_t)(u32)at; co[u] = (int32_t)(u32)(at >> 32); at += span_pack(m[u]); }
        if (wide && i0 + SPAN_PER_THREAD <= n) {
            *reinterpret_cast<int4*>(P.byte_off + i0) = make_int4(bo[0], bo[1], bo[2], bo[3]);
            *reinterpret_cast<int4*>(P.char_off + i0) = make_int4(co[0], co[1], co[2], co[3]);
        } else {
#pragma unroll
            for (int u = 0; u < SPAN_PER_THREAD; u++) if (i0 + u < n) { P.byte_off[i0 + u] = bo[u]; P.char_off[i0 + u] = co[u]; }
        }
        if (i0 < n && i0 + SPAN_PER_THREAD >= n) { P.byte_off[n] = (int32_t)(u32)at; P.char_off[n] = (int32_t)(u32)(at >> 32); }     // the end of the last token
    }
}
