// Batched streaming Gaussian elimination over GF(2) (Sec. 2.2) on sm_103a.
//
// A call runs two passes over each context's rows (stream order = CSR order):
//
//  Pass 1 (dedup): the first occurrence of every distinct observation (x, y)
//  of a context is its representative; later equal rows are its duplicates.
//  A duplicate needs no elimination: its row equals an earlier row, so it
//  lies in the span when it arrives and is classified exactly as that earlier
//  row was -- redundant if the representative was consistent, a
//  contradiction if the representative was one (T never changes on the span).
//  Equality is decided by comparing the full rows (hash tables in shared
//  memory only propose the candidates), so the pass is exact.
//
//  Pass 2 (elimination) streams the representatives of each context, in
//  order, through a reduced basis B[k] = (r_k, z_k) held in shared memory:
//   1. open: an empty basis is filled from the first rows, a few a lane, each
//      pivot applied to the group's rows at once, so that they stay reduced
//      among themselves and no stored row is read (rows of more than 17 words:
//      1,024 rows, a thread each, elim_open_kernel);
//   2. reduce: each lane reduces its row against the basis as it stood at
//      the start of the round (the snapshot).  The basis is reduced (RREF,
//      the paper's step (5)), so the rows to XOR are exactly the pivots set
//      in the row itself: the warp walks the union of those pivots and every
//      lane XORs the broadcast row under its own bit, or, where it fits and
//      pays, looks four columns at a time up in a table of the basis that is
//      kept while the rows inserted since are few;
//   3. classify: a zero feature residual means the row lies in the span of
//      the snapshot, and the map T fixed by the snapshot never changes
//      afterwards (contradicting rows are not inserted, insertions only
//      extend it), so the classification equals the one-row-at-a-time one:
//      zero word residual -> redundant, else contradiction (steps (2)-(3)).
//      A contradicting representative counts once for itself and once per
//      duplicate; its index is the first of them;
//   4. insert: the remaining rows (candidates) are eliminated among
//      themselves in stream order inside the warp (step (4)), then merged:
//      new rows go to their pivot slots and every older row is cleared at
//      the new pivot columns (step (5)).  The basis, including every z_k, is
//      the sequential algorithm's.
//
// Both passes give one warp to small contexts (many per CTA) and a whole CTA
// to large ones.  Contexts of few rows go to the elimination without the first
// pass.  The elimination is in elim.cuh, instantiated by width in
// elim_small.cu (d <= 96), elim_narrow.cu (d <= 288) and elim_wide.cu (up to
// d = 1025); the full-rank check on the tensor cores in verify_tc.cu.  Plan
// kernels validate the CSR batch and order the work longest-first.
#include <string.h>

#include <mutex>

#include "full.cuh"

using namespace f2;

namespace {

// ---------------------------------------------------------------------------
// Check of a handed-off context (Sec. 2.2 steps (1)-(3) with the basis
// fixed).  Until a representative falls outside the span, the sequential
// algorithm leaves the basis as it is, so it classifies every such
// representative against this basis, and in any order: CTAs claim chunks
// of CHECK_CHUNK representatives, hold the basis in shared memory (a slot
// per pivot column) and reduce each representative by the pivot rows its
// own bits select (the warp walks the pivots set in any of its lanes).  A
// representative outside the span would extend the basis: the chunk
// records the first such one, and only representatives before the
// context's first are counted.  The last chunk of a context commits its
// counts; if some representative was outside the span, the context is
// listed for a second launch of the elimination from that one on.
//
// 10,000 contexts of 128..512 bits of parsed values, 13.4M rows: 443 us while
// every CTA claimed its way through the whole list of contexts, an atomic each,
// a row's words were loaded one by one and every basis row was XOR-ed whole;
// 190 without that, 228 now that it is handed every long context that walks its
// pivots (41..48% of the issue slots; warps wait at the barriers of a chunk and
// for its rows).  Two rows a lane made no difference, nor fewer barriers a chunk.
// ---------------------------------------------------------------------------
struct CheckArgs {
    const int64_t* row_off;
    const int64_t* x_off;
    const uint32_t* x;
    const uint4* y;
    const int32_t* rep_list;  // NULL: every row is its own representative
    const int32_t* rep_dup;
    const int32_t* rep_count;
    const int* snap_count;
    const int32_t* snap_list;
    const int32_t* snap_start;
    int* ctr;                 // [C] chunks claimed, [C] chunks done
    uint4* rec;               // two uint4 per chunk: (first outside, count lo, count hi, -), (first contradiction)
    int* resume_count;
    int32_t* resume_list;
    int32_t* resume_from;
};

struct DedupArgs {
    const int64_t* row_off;
    const int64_t* x_off;
    const uint32_t* x;
    const uint4* y;
    int32_t* rep_list;
    int32_t* rep_dup;
    int32_t* rep_count;
    const int32_t* queue;
    int* counters;
    unsigned long long* timing;  // per-context timestamps (F2_OPT_TIMING), NULL = off
    int32_t* shard_reps;         // [DD_MAX_SHARDS * C]: representatives of each shard of a split context
    int32_t* shard_done;         // [C]: shards of a split context finished (the last one compacts)
};

constexpr int FULL_THREADS = 1024;  // verify_full_kernel: one table shared by 32 warps

// Pass 1: 16 warps per CTA, two CTAs per SM (64 registers a thread: the pass
// is bound by dependent per-row chains, so warps hide latency better than
// rows held in flight by one warp).  A warp-owned context (at most
// DD_WARP_MAX_ROWS rows) gets a table of next_pow2(2T) entries in a 6 KB
// region; a CTA-owned context a table of up to DD_CTA_E entries.  Entry =
// (fingerprint, row index) plus a duplicate counter: 12 bytes.
constexpr int DD_THREADS = 512;
constexpr int DD_WARPS = DD_THREADS / 32;
constexpr int DD_CTAS_PER_SM = 2;
constexpr int DD_WARP_MAX_ROWS = 256;           // warp-owned up to this many rows
constexpr int DD_QUAD_MAX_ROWS = 4096;          // 4-warp-owned up to this many rows
constexpr int DD_WARP_E = 512;
constexpr int DD_WARP_REGION = 3 * DD_WARP_E;   // words
constexpr int DD_QUAD_E = 4 * DD_WARP_E;
constexpr int DD_CTA_E = 8192;
constexpr int DD_SMEM = 4 * 3 * DD_CTA_E;       // bytes (also 16 warp regions)
constexpr int DD_SEG_ROWS = 16384;              // rows a CTA takes at a time (10..16-word rows)
constexpr int DD_QUAD_REPS = 1024;              // most distinct rows numbered by a quad, by a CTA (as above)
constexpr int DD_CTA_REPS = 4096;
constexpr int DD_AHEAD_XW = 5;                  // widest rows whose next round is loaded ahead
constexpr int DD_XW = NARROW_WD;                // widest feature row (words) of dedup_kernel<false>
constexpr int DD_XW_WIDE = 16;                  // widest of dedup_kernel<true> (one row in flight)
constexpr int DEDUP_PROBES = 8;                 // linear-probe limit
// A CTA-owned context with much more than its share of the call's rows is
// split into up to DD_MAX_SHARDS consecutive row ranges deduplicated by
// different CTAs (a queue item = context | shard << 24 | (shards - 1) << 28).
constexpr int DD_MAX_SHARDS = 8;
constexpr int SHARD_CTX_LIMIT = 1 << 24;
// Shards of at most this many rows (a shard's table of DD_CTA_E entries
// stays at most half full when half its rows repeat earlier ones).
#ifndef F2_DD_SHARD_ROWS
#define F2_DD_SHARD_ROWS 16384
#endif
constexpr int DD_SHARD_ROWS = F2_DD_SHARD_ROWS;
// A context of the 4-warp class with more than 1/DD_QUAD_SHARE of a shard
// share goes to a whole CTA (4 warps would finish it long after the SMs'
// median).
#ifndef F2_DD_QUAD_PROMOTE
#define F2_DD_QUAD_PROMOTE 1
#endif
constexpr int DD_QUAD_SHARE = 4;
// Neither applies below these sizes, where a CTA's fixed costs (its table,
// its barriers, the shards' compaction) outweigh what the split saves.
constexpr int DD_PROMOTE_MIN_ROWS = 1024;
constexpr int DD_SHARD_MIN_ROWS = 2048;
// Contexts of at most this many rows in a call skip the duplicate pass: a
// warp opens a basis with 128 rows at once, repeats or not, and a CTA takes
// 256 rows a round, so their repeats cost less than finding them.  A call
// without longer contexts leaves the duplicate pass and the second plan with
// nothing to do: eight batches of 32 rows for each of 4,096 contexts went from
// 625 to 444 us.
constexpr int DEDUP_MIN_WARP = 128;
constexpr int DEDUP_MIN_CTA = 1024;
static_assert(DD_WARPS * DD_WARP_REGION * 4 <= DD_SMEM, "warp regions exceed the dedup shared memory");

// Dispatch on a feature-row width to a template instantiation.
#define F2_XWIDE_SWITCH(wd, CALL)    \
    switch (wd) {                    \
    case 10: CALL(10); break;        \
    case 11: CALL(11); break;        \
    case 12: CALL(12); break;        \
    case 13: CALL(13); break;        \
    case 14: CALL(14); break;        \
    case 15: CALL(15); break;        \
    case 16: CALL(16); break;        \
    default: break;                  \
    }

#define F2_NARROW_SWITCH(wd, CALL)   \
    switch (wd) {                    \
    case 1: CALL(1); break;          \
    case 2: CALL(2); break;          \
    case 3: CALL(3); break;          \
    case 4: CALL(4); break;          \
    case 5: CALL(5); break;          \
    case 6: CALL(6); break;          \
    case 7: CALL(7); break;          \
    case 8: CALL(8); break;          \
    case 9: CALL(9); break;          \
    default: break;                  \
    }


// ------------------------------------------------------------------ pass 1

__device__ __forceinline__ uint32_t last_mask(int n) { return (n & 31) ? ((1u << (n & 31)) - 1u) : 0xffffffffu; }

// Full comparison of rows i and j of a context (feature bits < n and word).
__device__ __forceinline__ bool rows_equal(const uint32_t* xc, const uint4* yc, int xw, int n,
                                           int64_t i, const uint4& yi, int64_t j)
{
    const uint4 yj = ld(yc + j);
    if (yj.x != yi.x || yj.y != yi.y || yj.z != yi.z || yj.w != yi.w) return false;
    const uint32_t lm = last_mask(n);
    for (int v = 0; v < xw; ++v) {
        const uint32_t m = (v == xw - 1) ? lm : 0xffffffffu;
        if (((ld(xc + i * xw + v) ^ ld(xc + j * xw + v)) & m) != 0u) return false;
    }
    return true;
}

// Find the entry of row i's content starting at slot `slot`, inserting it
// if absent.  Returns the slot (whose index field ends as the smallest row
// index of that content), or -1 when the probe budget runs out (the row then
// counts as its own representative, which is always exact).
__device__ __noinline__ int dd_find_insert(uint2* tab, int E, uint32_t h, int64_t i, const uint4& yi,
                                           const uint32_t* xc, const uint4* yc, int xw,
                                           int n, uint32_t slot, int budget)
{
    const uint32_t fp = h | 1u;
    for (int p = 0; p < budget; ++p, slot = (slot + 1) & (uint32_t)(E - 1)) {
        uint2 e = tab[slot];
        if (e.x == 0u) {
            const unsigned long long want = ((unsigned long long)(uint32_t)i << 32) | fp;
            const unsigned long long old = atomicCAS(reinterpret_cast<unsigned long long*>(tab + slot), 0ull, want);
            if (old == 0ull) return (int)slot;
            e.x = (uint32_t)old;
            e.y = (uint32_t)(old >> 32);
        }
        if (e.x == fp && rows_equal(xc, yc, xw, n, i, yi, (int64_t)e.y)) {
            if ((uint32_t)i < e.y) atomicMin(&tab[slot].y, (uint32_t)i);
            return (int)slot;
        }
    }
    return -1;
}

// Feature words of a row: the widest loads that every row of the context
// allows (`al`: log2 of the words its rows are aligned to).
template <int XW>
__device__ __forceinline__ void load_words(const uint32_t* p, int al, uint32_t (&x)[XW])
{
    if (XW % 4 == 0 && al >= 2) {
#pragma unroll
        for (int v = 0; v + 3 < XW; v += 4) {
            const uint4 t = ld(reinterpret_cast<const uint4*>(p + v));
            x[v] = t.x;
            x[v + 1] = t.y;
            x[v + 2] = t.z;
            x[v + 3] = t.w;
        }
    } else if (XW % 2 == 0 && al >= 1) {
#pragma unroll
        for (int v = 0; v + 1 < XW; v += 2) {
            const uint2 t = ld(reinterpret_cast<const uint2*>(p + v));
            x[v] = t.x;
            x[v + 1] = t.y;
        }
    } else {
#pragma unroll
        for (int v = 0; v < XW; ++v) x[v] = ld(p + v);
    }
}

// Hash of an observation: a sum of the words times odd constants, mixed.  It
// only proposes candidates; every match is confirmed by comparing the rows.
template <int XW>
__device__ __forceinline__ uint32_t dd_hash(const uint32_t (&x)[XW], const uint4& y)
{
    uint32_t h = y.x * 0x9E3779B1u + y.y * 0x85EBCA77u + y.z * 0xC2B2AE3Du + y.w * 0x27D4EB2Fu;
    uint32_t k = 0x165667B1u;
#pragma unroll
    for (int v = 0; v < XW; ++v) {
        h += x[v] * k;
        k = k * 0x01000193u + 0x3C6EF372u;  // constants at compile time
        k |= 1u;
    }
    h ^= h >> 16;
    h *= 0x7FEB352Du;
    h ^= h >> 15;
    return h;
}

// Group synchronisation for pass 1: a warp, a quad of 4 warps (named
// barrier 1 + quad index, 128 threads) or the whole CTA.
template <int G>
__device__ __forceinline__ void dd_sync()
{
    if (G == 1) __syncwarp();
    else if (G == DD_WARPS) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x >> 5) / G), "r"(32 * G) : "memory");
}

// The queue item of the context a dedup CTA is on (context, shard, shard
// count); a CTA-owned pass reads it here, before and again after its rows, so
// that no register holds it through them.
__shared__ uint32_t dd_cta_item;

// Closes a context's (or a shard's) pass: publishes its count and, in the last
// shard of a split context to finish, moves the shards' lists together.
// Returns whether the context is done.
template <int G>
__device__ bool dd_finish(const DedupArgs& a, int c, int nrep, int t)
{
    constexpr int NT = 32 * G;
    int shard = 0, nsh = 1;
    if constexpr (G == DD_WARPS) {
        const uint32_t qi = *reinterpret_cast<const volatile uint32_t*>(&dd_cta_item);
        shard = (int)((qi >> 24) & 7u);
        nsh = (int)(qi >> 28) + 1;
    }
    if (nsh == 1) {
        if (t == 0) a.rep_count[c] = nrep;
        dd_sync<G>();
        return true;
    }
    // a split context: publish this shard's count; the last shard to finish
    // moves the lists of shards 1.. down behind shard 0's (never upward: a
    // shard's list starts at or after its destination), chunk by chunk
    // through registers, renumbering their rows from the context's first
    __shared__ int s_last;
    __threadfence();  // this thread's list entries, before the count that publishes them
    dd_sync<G>();
    if (t == 0) {
        a.shard_reps[(size_t)DD_MAX_SHARDS * c + shard] = nrep;
        __threadfence();
        s_last = (atomicAdd(a.shard_done + c, 1) == nsh - 1);
    }
    dd_sync<G>();
    if (!s_last) return false;
    __threadfence();
    const int64_t cbase = a.row_off[c];
    const int Tall = (int)(a.row_off[c + 1] - cbase);
    int dst = 0;
    for (int k = 0; k < nsh; ++k) {
        const int src = (int)(((long long)Tall * k) / nsh);
        const int cnt = __ldcg(a.shard_reps + (size_t)DD_MAX_SHARDS * c + k);
        if (k > 0) {
            for (int b0 = 0; b0 < cnt; b0 += NT) {
                const int j = b0 + t;
                int32_t rl = 0, rd = 0;
                if (j < cnt) {
                    rl = __ldcg(a.rep_list + cbase + src + j) + src;
                    rd = __ldcg(a.rep_dup + cbase + src + j);
                }
                dd_sync<G>();
                if (j < cnt) {
                    a.rep_list[cbase + dst + j] = rl;
                    a.rep_dup[cbase + dst + j] = rd;
                }
                dd_sync<G>();
            }
        }
        dst += cnt;
    }
    if (t == 0) a.rep_count[c] = dst;
    dd_sync<G>();
    return true;
}

// One group of G warps finds the representatives of context c and writes
// them, in stream order, to rep_list[row_off[c] + k] with their duplicate
// counts in rep_dup; rep_count[c] = number of representatives.  Each thread
// takes a row a round.  Table slot: (fingerprint, smallest row index
// of that content) plus a duplicate counter; a full row comparison decides
// every match, so a row is a duplicate only if it equals an earlier row.
//
// Shard k of nsh takes the context's rows [lo, hi) = [T*k/nsh, T*(k+1)/nsh)
// and writes its representatives, numbered from lo, at
// rep_list[row_off[c] + lo + ...]; a row
// equal to a row of an earlier shard becomes its own representative there,
// which the elimination classifies exactly all the same (it lies in the span
// when it arrives).  The last shard to finish moves the shards' lists
// together, in stream order, and sets rep_count[c].  Returns whether the
// context is done (false in the shards that did not finish last).
//
template <int G, int XW>
__device__ bool dedup_ctx(const StoreDev& s, const DedupArgs& a, int c, uint32_t* region, int E, int* wcnt)
{
    int shard = 0, nsh = 1;
    if constexpr (G == DD_WARPS) {
        const uint32_t qi = dd_cta_item;
        shard = (int)((qi >> 24) & 7u);
        nsh = (int)(qi >> 28) + 1;
    }
    constexpr int NT = 32 * G;
    const int lane = threadIdx.x & 31;
    const int gw = (G == 1) ? 0 : (int)((threadIdx.x >> 5) % G);  // warp within the group
    const int t = 32 * gw + lane;
    uint2* tab = reinterpret_cast<uint2*>(region);
    int* D = reinterpret_cast<int*>(region + 2 * E);
    const CtxDesc cd = s.desc[c];
    const int n = cd.n;
    const int Tc = (int)(a.row_off[c + 1] - a.row_off[c]);
    const int lo = (int)(((long long)Tc * shard) / nsh);
    const int64_t r0 = a.row_off[c] + lo;  // this shard's rows, and its part of rep_list / rep_dup
    const int T = (int)(((long long)Tc * (shard + 1)) / nsh) - lo;
    const uint32_t Tu = (uint32_t)T;  // (rows past the last are counted unsigned: T may be 2^31 - 1)
    const uint32_t* xc = a.x + a.x_off[c] + (int64_t)lo * XW;
    const uint4* yc = a.y + r0;
    const uint32_t lm = last_mask(n);
    const int al = ((uintptr_t)xc & 15) == 0 ? 2 : (((uintptr_t)xc & 7) == 0 ? 1 : 0);
    const uint32_t emask = (uint32_t)(E - 1);
    for (int e = t; e < E; e += NT) {
        tab[e] = make_uint2(0u, 0u);
        D[e] = 0;
    }
    dd_sync<G>();
    int nrep = 0;
    // Rows of up to DD_AHEAD_XW words are loaded a round ahead: the pass waits on
    // memory, and the 64 registers hold two rows a thread either way (two at
    // once instead: 77,926 contexts 2,607 against 2,505 us, 4,096 contexts 284
    // against 275).
    constexpr bool AHEAD = XW <= DD_AHEAD_XW;
    uint4 yn;
    uint32_t xn[XW];
    auto load_round = [&](uint32_t base) {
        const uint32_t i = base + (uint32_t)t;
        const int ic = i < Tu ? (int)i : T - 1;  // (a row read twice, not counted)
        yn = ld(yc + ic);
        load_words<XW>(xc + (int64_t)ic * XW, al, xn);
    };
    if (AHEAD) load_round(0);
    for (uint32_t base = 0; base < Tu; base += NT) {
        if (!AHEAD) load_round(base);
        const uint32_t i = base + (uint32_t)t;
        const bool valid = i < Tu;
        const uint4 yv = yn;
        uint32_t xv[XW];
#pragma unroll
        for (int v = 0; v < XW; ++v) xv[v] = (v == XW - 1) ? xn[v] & lm : xn[v];
        if (AHEAD) load_round(base + NT);
        const uint32_t h = dd_hash<XW>(xv, yv);
        // probe by fingerprint only (shared memory): the first slot holding
        // this fingerprint, or an empty slot that the row then claims
        int mine = valid ? -2 : -1;  // -2 = unresolved
        uint2 ent = make_uint2(0u, 0u);
        uint32_t cs = 0u;
        if (valid) {
            const uint32_t fp = h | 1u;
            uint32_t slot = (h >> 7) & emask;
            int p = 0;
            for (; p < DEDUP_PROBES; ++p, slot = (slot + 1) & emask) {
                uint2 e = tab[slot];
                if (e.x == 0u) {
                    const unsigned long long want = ((unsigned long long)i << 32) | fp;
                    const unsigned long long old =
                        atomicCAS(reinterpret_cast<unsigned long long*>(tab + slot), 0ull, want);
                    if (old == 0ull) {
                        mine = (int)slot;
                        break;
                    }
                    e.x = (uint32_t)old;
                    e.y = (uint32_t)(old >> 32);
                }
                if (e.x == fp) {
                    ent = e;
                    cs = slot;
                    break;
                }
            }
            if (p == DEDUP_PROBES) mine = -1;  // table region full: own representative
        }
        // full comparison with the row of that fingerprint
        const bool need = mine == -2;
        uint4 yo = make_uint4(0, 0, 0, 0);
        uint32_t xo[XW];
#pragma unroll
        for (int v = 0; v < XW; ++v) xo[v] = 0u;
        if (need) {
            yo = ld(yc + ent.y);
            load_words<XW>(xc + (int64_t)ent.y * XW, al, xo);
        }
        if (need) {
            bool e = yo.x == yv.x && yo.y == yv.y && yo.z == yv.z && yo.w == yv.w;
#pragma unroll
            for (int v = 0; v < XW; ++v) {
                const uint32_t w = (v == XW - 1) ? (xo[v] & lm) : xo[v];
                e = e && (w == xv[v]);
            }
            if (e) {
                if (i < ent.y) atomicMin(&tab[cs].y, i);
                mine = (int)cs;
            } else {  // a different row with the same fingerprint: keep probing
                mine = dd_find_insert(tab, E, h, i, yv, xc, yc, XW, n, (cs + 1) & emask, DEDUP_PROBES - 1);
            }
        }
        dd_sync<G>();
        const uint32_t rep = (valid && mine >= 0) ? tab[mine].y : i;
        const bool isrep = valid && rep == i;
        if (valid && !isrep) atomicAdd(D + mine, 1);
        const uint32_t bal = __ballot_sync(FULL, isrep);
        int before = 0, total = __popc(bal);
        if (G > 1) {
            if (lane == 0) wcnt[gw] = total;
            dd_sync<G>();
            const int v = lane < G ? wcnt[lane] : 0;
            total = __reduce_add_sync(FULL, v);
            before = __reduce_add_sync(FULL, lane < gw ? v : 0);
        }
        if (isrep) {
            const int pos = nrep + before + __popc(bal & ((1u << lane) - 1u));
            a.rep_list[r0 + pos] = (int32_t)i;  // within the shard
            a.rep_dup[r0 + pos] = mine;
        }
        nrep += total;
        // (the next round's first barrier comes before it writes wcnt again)
    }
    dd_sync<G>();
    for (uint32_t k = t; k < (uint32_t)nrep; k += NT) {
        const int slot = a.rep_dup[r0 + k];
        a.rep_dup[r0 + k] = (slot >= 0) ? D[slot] : 0;
    }
    if (t == 0) {
        // the call's work, for the elimination plan's thresholds
        atomicAdd(reinterpret_cast<unsigned long long*>(a.counters + CNT_WORK),
                  (unsigned long long)nrep * (unsigned long long)cd.d);
        atomicAdd(reinterpret_cast<unsigned long long*>(a.counters + CNT_REPS), (unsigned long long)nrep);
    }
    return dd_finish<G>(a, c, nrep, t);
}

__device__ __forceinline__ int pow2_at_least(int v)
{
    int e = 64;
    while (e < v) e <<= 1;
    return e;
}

// ---------------------------------------------------------------------------
// Pass 1 for feature rows of 10..16 words.  Confirming a repeat from global
// memory costs such a row 14 to 20 scattered loads, so copies of the distinct
// rows are kept in shared memory, and a warp never waits for the others between
// rows.  10,000 contexts of parsed values went from 1,471 to 1,403 us; with
// rows of up to nine words the form above is as fast or faster (77,926
// contexts 2,609 us and 2,598 with this one, 4,096 contexts 282 and 287):
// there the extra instructions cost what the loads save.
// ---------------------------------------------------------------------------
// A group's shared memory while it looks for the distinct rows among at most
// DD_SEG_ROWS consecutive rows of a context.  The distinct rows found so far
// are numbered; number r has its smallest row index idx[r], its repeats
// dup[r], and for r < cap a copy of the row itself (ys, xs), so that a repeat
// is confirmed from shared memory: 32 random rows in global memory cost the
// L1 a tag lookup each, which bound the pass.  A slot of the hash table holds
// (16 bits of the hash, r + 1), a bucket four slots that one load fetches: with
// single slots nearly every round had some lane on its third or fourth probe.
// Rows that find no room (nrep numbers, the probe limit, a distinct row with
// their fingerprint in the bucket) are marked in `ovf` and stand for
// themselves, which is exact.
// (Word offsets into the CTA's dynamic shared memory.)
struct DdSmem {
    int tab, idx, dup;
    int bm;   // rows that are the first of their content
    int ovf;  // rows that found no room
    int pre;  // first rows in the bitmap words before
    int cnt;  // numbers given out; rows without room (0 or 1)
    int ys, xs;
    uint32_t emask;
    int nrep, cap, words;
};
__device__ __forceinline__ uint32_t* dd_smem()
{
    extern __shared__ __align__(16) uint32_t smem[];
    return smem;
}
__device__ __forceinline__ uint4 dd_load4(int word)  // volatile: other warps fill it
{
    uint4 v;
    asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(smem_addr(dd_smem() + word))
                 : "memory");
    return v;
}
__device__ __forceinline__ uint4* dd_smem4(int word) { return reinterpret_cast<uint4*>(dd_smem() + word); }

template <int XW>
__device__ __forceinline__ DdSmem dd_layout(int region, int region_words, int T, int most)
{
    DdSmem m;
    m.words = (T + 31) >> 5;
    // three quarters of the rows: beyond that most rows have no repeat to find
    const int want = (((3 * T) >> 2) + 31) & ~31;
    m.nrep = want < most ? (want < 32 ? 32 : want) : most;
    const int E = pow2_at_least(m.nrep + m.nrep / 3);
    m.emask = (uint32_t)(E / 4 - 1);  // buckets of four slots
    m.tab = region;
    m.idx = m.tab + E;
    m.dup = m.idx + m.nrep;
    m.bm = m.dup + m.nrep;
    m.ovf = m.bm + m.words;
    m.pre = m.ovf + m.words;
    m.cnt = m.pre + m.words;
    const int used = (E + 2 * m.nrep + 3 * m.words + 2 + 3) & ~3;
    const int cap = (region_words - used) / (4 + XW);
    m.cap = cap < m.nrep ? cap : m.nrep;
    m.ys = region + used;
    m.xs = region + used + 4 * m.cap;
    return m;
}

// Row (x, y) equals the row numbered r, whose smallest index so far is i0.
template <int XW>
__device__ __forceinline__ bool dd_same(const DdSmem& m, int r, const uint32_t (&x)[XW], const uint4& y,
                                        const uint32_t* xc, const uint4* yc, uint32_t lm)
{
    uint4 o;
    uint32_t diff = 0;
    if (r < m.cap) {
        o = *dd_smem4(m.ys + 4 * r);
#pragma unroll
        for (int v = 0; v < XW; ++v) diff |= dd_smem()[m.xs + r * XW + v] ^ x[v];
    } else {
        const int64_t j = (int64_t)*reinterpret_cast<const volatile uint32_t*>(dd_smem() + m.idx + r);
        o = ld(yc + j);
#pragma unroll
        for (int v = 0; v < XW; ++v) {
            const uint32_t w = ld(xc + j * XW + v);
            diff |= (v == XW - 1 ? w & lm : w) ^ x[v];
        }
    }
    return (diff | (o.x ^ y.x) | (o.y ^ y.y) | (o.z ^ y.z) | (o.w ^ y.w)) == 0u;
}

// The distinct rows among T <= DD_SEG_ROWS rows, by a group of G warps: their
// indices (plus `off`), in stream order, and repeats go to rep / dups; returns
// their number.  Each thread takes a row a round and no round waits for
// another, so the warps hide each other's latencies; the first rows are put in
// order at the end, through a bitmap.
template <int G, int XW>
__device__ int dedup_rows(const uint32_t* xc, const uint4* yc, int T, int off, uint32_t lm,
                          int al, const DdSmem& m, int32_t* __restrict__ rep, int32_t* __restrict__ dups, int* wcnt)
{
    constexpr int NT = 32 * G;
    const int lane = threadIdx.x & 31;
    const int gw = (G == 1) ? 0 : (int)((threadIdx.x >> 5) % G);  // warp within the group
    const int t = 32 * gw + lane;
    for (int e = m.tab + t; e < m.idx; e += NT) dd_smem()[e] = 0u;
    for (int e = t; e < 2 * m.words; e += NT) dd_smem()[m.bm + (e)] = 0u;  // bm and ovf
    if (t < 2) dd_smem()[m.cnt + (t)] = 0u;
    dd_sync<G>();
    for (int base = 0; base < T; base += NT) {
        const int i = base + t;
        const int ic = i < T ? i : T - 1;  // (a row read twice, not counted)
        const uint4 y = ld(yc + ic);
        uint32_t x[XW];
        load_words<XW>(xc + (int64_t)ic * XW, al, x);
        x[XW - 1] &= lm;
        const uint32_t h = dd_hash<XW>(x, y);
        const uint32_t fp = (h & 0xFFFF0000u) | 0x80000000u;  // never an empty slot's
        int bucket = m.tab + 4 * (int)(h & m.emask);
        int mine = -1;                // a number allocated for this row
        int same = -1;                // the number of the row it repeats
        bool pending = i < T, alone = false;
        for (int p = 0; p < DEDUP_PROBES; ++p) {
            uint4 e = make_uint4(~0u, ~0u, ~0u, ~0u);
            if (pending) e = dd_load4(bucket);
            // the bucket's slot with this fingerprint, its first free slot
            uint32_t v = 0;
            if ((e.w ^ fp) < 0x10000u) v = e.w;
            if ((e.z ^ fp) < 0x10000u) v = e.z;
            if ((e.y ^ fp) < 0x10000u) v = e.y;
            if ((e.x ^ fp) < 0x10000u) v = e.x;
            const int free = e.x == 0u ? 0 : (e.y == 0u ? 1 : (e.z == 0u ? 2 : (e.w == 0u ? 3 : 4)));
            const bool claim = pending && v == 0u && free < 4;
            // numbers for the rows that found a free slot, one atomic a warp
            const uint32_t want = __ballot_sync(FULL, claim && mine == -1);
            if (want) {
                uint32_t r0 = 0;
                if (lane == __ffs(want) - 1) r0 = atomicAdd(dd_smem() + m.cnt, (uint32_t)__popc(want));
                r0 = __shfl_sync(FULL, r0, __ffs(want) - 1);
                if ((want >> lane) & 1u) {
                    mine = (int)r0 + __popc(want & ((1u << lane) - 1u));
                    if (mine >= m.nrep) {  // no room
                        mine = -2;
                        pending = false;
                        alone = true;
                    } else {
                        // the row before the slot that publishes it
                        if (mine < m.cap) {
                            *dd_smem4(m.ys + 4 * mine) = y;
#pragma unroll
                            for (int u = 0; u < XW; ++u) dd_smem()[m.xs + mine * XW + u] = x[u];
                        }
                        dd_smem()[m.idx + mine] = (uint32_t)i;
                        dd_smem()[m.dup + mine] = 0u;
                    }
                }
                __threadfence_block();
            }
            if (claim && mine >= 0) {
                // (a slot that another row took first: look at the bucket again)
                if (atomicCAS(dd_smem() + bucket + free, 0u, fp | (uint32_t)(mine + 1)) == 0u) pending = false;
            } else if (pending && v != 0u) {
                const int r = (int)(v & 0xFFFFu) - 1;
                pending = false;
                if (dd_same<XW>(m, r, x, y, xc, yc, lm)) same = r;
                else alone = true;  // another row with this fingerprint
            } else if (pending) {  // a full bucket: the next one
                bucket += 4;
                if (bucket == m.idx) bucket = m.tab;
            }
            if (!__any_sync(FULL, pending)) break;
        }
        if (same >= 0) {
            if ((uint32_t)i < *reinterpret_cast<const volatile uint32_t*>(dd_smem() + m.idx + same)) atomicMin(dd_smem() + m.idx + same, (uint32_t)i);
            atomicAdd(dd_smem() + m.dup + same, 1u);
            if (mine >= 0) dd_smem()[m.idx + (mine)] = ~0u;  // a number given out in vain
        } else if (pending || alone) {
            if (mine >= 0) dd_smem()[m.idx + (mine)] = ~0u;
            atomicOr(dd_smem() + m.ovf + (i >> 5), 1u << (i & 31));
            dd_smem()[m.cnt + (1)] = 1u;
        }
    }
    dd_sync<G>();
    const int n = (int)(dd_smem()[m.cnt + (0)] < (uint32_t)m.nrep ? dd_smem()[m.cnt + (0)] : (uint32_t)m.nrep);
    const bool over = dd_smem()[m.cnt + (1)] != 0u;
    for (int k = t; k < n; k += NT) {
        const uint32_t i = dd_smem()[m.idx + (k)];
        if (i != ~0u) atomicOr(dd_smem() + m.bm + (i >> 5), 1u << (i & 31));
    }
    dd_sync<G>();
    // first rows before each bitmap word (at most one word a thread)
    uint32_t w = 0;
    if (t < m.words) {
        w = dd_smem()[m.bm + (t)] | dd_smem()[m.ovf + (t)];
        dd_smem()[m.bm + (t)] = w;
    }
    int inc = __popc(w);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += u;
    }
    int before = 0, total = __shfl_sync(FULL, inc, 31);
    if (G > 1) {
        if (lane == 31) wcnt[gw] = inc;
        dd_sync<G>();
        total = 0;
#pragma unroll
        for (int ww = 0; ww < G; ++ww) {
            const int c = wcnt[ww];
            if (ww < gw) before += c;
            total += c;
        }
    }
    if (t < m.words) dd_smem()[m.pre + (t)] = (uint32_t)(before + inc - __popc(w));
    dd_sync<G>();
    for (int k = t; k < n; k += NT) {
        const uint32_t i = dd_smem()[m.idx + (k)];
        if (i == ~0u) continue;
        const int pos = (int)dd_smem()[m.pre + (i >> 5)] + __popc(dd_smem()[m.bm + (i >> 5)] & ((1u << (i & 31)) - 1u));
        rep[pos] = (int)i + off;
        dups[pos] = (int)dd_smem()[m.dup + (k)];
    }
    if (over) {
        for (int i = t; i < T; i += NT) {
            if (!((dd_smem()[m.ovf + (i >> 5)] >> (i & 31)) & 1u)) continue;
            const int pos = (int)dd_smem()[m.pre + (i >> 5)] + __popc(dd_smem()[m.bm + (i >> 5)] & ((1u << (i & 31)) - 1u));
            rep[pos] = i + off;
            dups[pos] = 0;
        }
    }
    dd_sync<G>();
    return total;
}

// As dedup_ctx; a range longer than DD_SEG_ROWS is taken in pieces, whose
// repeats of earlier pieces stay, as with shards.
template <int G, int XW>
__device__ bool dedup_wide_ctx(const StoreDev& s, const DedupArgs& a, int c, int region, int* wcnt)
{
    int shard = 0, nsh = 1;
    if constexpr (G == DD_WARPS) {
        const uint32_t qi = dd_cta_item;
        shard = (int)((qi >> 24) & 7u);
        nsh = (int)(qi >> 28) + 1;
    }
    constexpr int NT = 32 * G;
    constexpr int SEG = (G == 1) ? DD_WARP_MAX_ROWS : (G == 4 ? DD_QUAD_MAX_ROWS : DD_SEG_ROWS);
    constexpr int MOST = (G == 1) ? DD_WARP_MAX_ROWS : (G == 4 ? DD_QUAD_REPS : DD_CTA_REPS);
    static_assert(SEG <= 32 * NT, "a bitmap word a thread");
    const int t = (G == 1) ? (int)(threadIdx.x & 31) : (int)(threadIdx.x % NT);
    const int Tc = (int)(a.row_off[c + 1] - a.row_off[c]);
    const int lo = (int)(((long long)Tc * shard) / nsh);
    const int64_t r0 = a.row_off[c] + lo;  // this shard's rows, and its part of rep_list / rep_dup
    const int T = (int)(((long long)Tc * (shard + 1)) / nsh) - lo;
    const uint32_t* xc = a.x + a.x_off[c] + (int64_t)lo * XW;
    const uint32_t lm = last_mask(s.desc[c].n);
    const int al = ((uintptr_t)xc & 15) == 0 ? 2 : (((uintptr_t)xc & 7) == 0 ? 1 : 0);
    int nrep = 0;
    for (int s0 = 0, s1; s0 < T; s0 = s1) {
        s1 = step_to(s0, SEG, T);
        const int n = s1 - s0;
        const DdSmem m = dd_layout<XW>(region, G * DD_WARP_REGION, n, MOST);
        // (a piece starts at a multiple of SEG rows, so its rows keep the alignment)
        nrep += dedup_rows<G, XW>(xc + (int64_t)s0 * XW, a.y + r0 + s0, n, s0, lm, al, m, a.rep_list + r0 + nrep,
                                  a.rep_dup + r0 + nrep, wcnt);
    }
    if (t == 0) {
        // the call's work, for the elimination plan's thresholds
        atomicAdd(reinterpret_cast<unsigned long long*>(a.counters + CNT_WORK),
                  (unsigned long long)nrep * (unsigned long long)s.desc[c].d);
        atomicAdd(reinterpret_cast<unsigned long long*>(a.counters + CNT_REPS), (unsigned long long)nrep);
    }
    return dd_finish<G>(a, c, nrep, t);
}

// Pass 1 kernel: CTA-owned contexts first, then quads, then warps.
template <bool WX>
__global__ void __launch_bounds__(DD_THREADS, DD_CTAS_PER_SM) dedup_kernel(StoreDev s, DedupArgs a)
{
    pdl_wait();
    // WX: the contexts whose feature rows have DD_XW + 1 .. DD_XW_WIDE words
    constexpr int C_CTA = WX ? CLS_DDW_CTA : CLS_DD_CTA;
    constexpr int C_QUAD = WX ? CLS_DDW_QUAD : CLS_DD_QUAD;
    constexpr int C_WARP = WX ? CLS_DDW_WARP : CLS_DD_WARP;
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int s_item[DD_WARPS];
    __shared__ int wcnt[DD_WARPS];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (a.counters[CNT_DEDUPED] == 0) return;
    {
        const int n = a.counters[CNT_COUNT + C_CTA];
        const int b = a.counters[CNT_BEGIN + C_CTA];
        for (;;) {
            __syncthreads();
            if (threadIdx.x == 0) {
                const int it = atomicAdd(a.counters + CNT_HEAD + C_CTA, 1);
                s_item[0] = it;
                if (it < n) dd_cta_item = (uint32_t)a.queue[b + it];
            }
            __syncthreads();
            const int item = s_item[0];
            if (item >= n) break;
            const uint32_t qi = dd_cta_item;
            const int c = (int)(qi & (SHARD_CTX_LIMIT - 1));
            const int nsh = (int)(qi >> 28) + 1;
            const int T = (int)(a.row_off[c + 1] - a.row_off[c]);
            const int E = table_entries((int)(((int64_t)T + nsh - 1) / nsh), DD_CTA_E);
            // a split context's pass: from its first shard's start to the end of the last one
            if (threadIdx.x == 0 && ((qi >> 24) & 7u) == 0) time_mark(a.timing, c, 0);
            bool done = true;
#define F2_DD_CTA(W) done = dedup_ctx<DD_WARPS, W>(s, a, c, smem, E, wcnt)
#define F2_DDW_CTA(W) done = dedup_wide_ctx<DD_WARPS, W>(s, a, c, 0, wcnt)
            if constexpr (WX) {
                F2_XWIDE_SWITCH(s.desc[c].xw, F2_DDW_CTA)
            } else {
                F2_NARROW_SWITCH(s.desc[c].xw, F2_DD_CTA)
            }
#undef F2_DD_CTA
#undef F2_DDW_CTA
            if (threadIdx.x == 0 && done) time_mark(a.timing, c, 1);
        }
    }
    {
        const int q = warp / 4;
        const int n = a.counters[CNT_COUNT + C_QUAD];
        const int b = a.counters[CNT_BEGIN + C_QUAD];
        uint32_t* region = smem + q * 4 * DD_WARP_REGION;
        for (;;) {
            dd_sync<4>();
            if ((warp & 3) == 0 && lane == 0) s_item[q] = atomicAdd(a.counters + CNT_HEAD + C_QUAD, 1);
            dd_sync<4>();
            const int item = s_item[q];
            if (item >= n) break;
            const int c = a.queue[b + item];
            const int T = (int)(a.row_off[c + 1] - a.row_off[c]);
            const int E = table_entries(T, DD_QUAD_E);
            if ((warp & 3) == 0 && lane == 0) time_mark(a.timing, c, 0);
#define F2_DD_QUAD(W) dedup_ctx<4, W>(s, a, c, region, E, wcnt + q * 4)
#define F2_DDW_QUAD(W) dedup_wide_ctx<4, W>(s, a, c, q * 4 * DD_WARP_REGION, wcnt + q * 4)
            if constexpr (WX) {
                F2_XWIDE_SWITCH(s.desc[c].xw, F2_DDW_QUAD)
            } else {
                F2_NARROW_SWITCH(s.desc[c].xw, F2_DD_QUAD)
            }
#undef F2_DD_QUAD
#undef F2_DDW_QUAD
            if ((warp & 3) == 0 && lane == 0) time_mark(a.timing, c, 1);
        }
    }
    {
        const int n = a.counters[CNT_COUNT + C_WARP];
        const int b = a.counters[CNT_BEGIN + C_WARP];
        uint32_t* region = smem + warp * DD_WARP_REGION;
        for (;;) {
            int item = 0;
            if (lane == 0) item = atomicAdd(a.counters + CNT_HEAD + C_WARP, 1);
            item = __shfl_sync(FULL, item, 0);
            if (item >= n) break;
            const int c = a.queue[b + item];
            const int T = (int)(a.row_off[c + 1] - a.row_off[c]);
            const int E = table_entries(T, DD_WARP_E);
            if (lane == 0) time_mark(a.timing, c, 0);
#define F2_DD_WARP(W) dedup_ctx<1, W>(s, a, c, region, E, nullptr)
#define F2_DDW_WARP(W) dedup_wide_ctx<1, W>(s, a, c, warp * DD_WARP_REGION, nullptr)
            if constexpr (WX) {
                F2_XWIDE_SWITCH(s.desc[c].xw, F2_DDW_WARP)
            } else {
                F2_NARROW_SWITCH(s.desc[c].xw, F2_DD_WARP)
            }
#undef F2_DD_WARP
#undef F2_DDW_WARP
            if (lane == 0) time_mark(a.timing, c, 1);
        }
    }
}

__device__ __forceinline__ int64_t check_slot(const CheckArgs& a, int c)
{
    return a.row_off[c] / CHECK_CHUNK + c;  // the context's first chunk record (chunks never overlap)
}

// Feature words of a row of up to WD words (bits >= n cleared), by the widest
// loads that every row of the context allows (`al` as in load_words).
template <int WD>
__device__ __forceinline__ void load_row_words(const uint32_t* p, int al, bool valid, int n, int xw,
                                               uint32_t (&x)[WD])
{
#pragma unroll
    for (int v = 0; v < WD; ++v) x[v] = 0;
    if (valid) {
        if (WD >= 4 && al >= 2) {
#pragma unroll
            for (int v = 0; v + 3 < WD; v += 4)
                if (v < xw) {
                    const uint4 t = ld(reinterpret_cast<const uint4*>(p + v));
                    x[v] = t.x;
                    x[v + 1] = t.y;
                    x[v + 2] = t.z;
                    x[v + 3] = t.w;
                }
        } else if (WD >= 2 && al >= 1) {
#pragma unroll
            for (int v = 0; v + 1 < WD; v += 2)
                if (v < xw) {
                    const uint2 t = ld(reinterpret_cast<const uint2*>(p + v));
                    x[v] = t.x;
                    x[v + 1] = t.y;
                }
        } else {
#pragma unroll
            for (int v = 0; v < WD; ++v)
                if (v < xw) x[v] = ld(p + v);
        }
    }
    const uint32_t last = (n & 31) ? (1u << (n & 31)) - 1u : FULL;
#pragma unroll
    for (int v = 0; v < WD; ++v) x[v] &= (v == xw - 1) ? last : FULL;
}

// Reduces q and y by the basis rows of pivot words W and up.  A basis row has no
// bit above its pivot.
template <int WD, int W>
__device__ __forceinline__ void check_words(uint32_t (&q)[WD], uint4& y, const uint32_t* S, const uint32_t* Ps,
                                            const uint32_t* Ds)
{
    constexpr int RS = row_stride(WD);
    const uint32_t sel = q[W];
    uint32_t uw = __reduce_or_sync(FULL, sel & Ps[W]);
    uint32_t dw = uw & Ds[W];
    uw &= ~dw;
    while (uw) {  // two a step, their loads issued together
        const int b0 = __ffs(uw) - 1;
        uw &= uw - 1;
        const bool two = uw != 0u;
        const int b1 = two ? __ffs(uw) - 1 : b0;
        uw &= uw - 1;
        const uint4 z0 = *reinterpret_cast<const uint4*>(S + (32 * W + b0) * RS);
        const uint4 z1 = *reinterpret_cast<const uint4*>(S + (32 * W + b1) * RS);
        const uint32_t m0 = 0u - ((sel >> b0) & 1u);
        const uint32_t m1 = two ? 0u - ((sel >> b1) & 1u) : 0u;
        y.x ^= (z0.x & m0) ^ (z1.x & m1);
        y.y ^= (z0.y & m0) ^ (z1.y & m1);
        y.z ^= (z0.z & m0) ^ (z1.z & m1);
        y.w ^= (z0.w & m0) ^ (z1.w & m1);
    }
    while (dw) {
        const int b = __ffs(dw) - 1;
        dw &= dw - 1;
        const uint32_t* row = S + (32 * W + b) * RS;
        const uint4 z = *reinterpret_cast<const uint4*>(row);
        const uint32_t m = 0u - ((sel >> b) & 1u);
        y.x ^= z.x & m;
        y.y ^= z.y & m;
        y.z ^= z.z & m;
        y.w ^= z.w & m;
#pragma unroll
        for (int v4 = 0; v4 <= W / 4; ++v4) {
            const uint4 e = *reinterpret_cast<const uint4*>(row + 4 + 4 * v4);
            const uint32_t ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (4 * v4 + j <= W && 4 * v4 + j < WD) q[4 * v4 + j] ^= ev[j] & m;
        }
    }
    if constexpr (W + 1 < WD) check_words<WD, W + 1>(q, y, S, Ps, Ds);
}

// Classes of the representatives kb .. ke-1 of a context under its basis S of
// pivots Ps: 2 outside the span, 1 a contradiction, 0 redundant.  The basis is
// reduced, so a row's pivot bits select its basis rows whatever their order;
// and where a basis row is its pivot alone (not in Ds: with values that differ
// in single bits, nearly every row) only its 128-bit word counts.
template <int WD>
__device__ void check_chunk(const StoreDev& s, const CheckArgs& a, int c, int kb, int ke, const uint32_t* S,
                            const uint32_t* Ps, const uint32_t* Ds, uint8_t* flags)
{
    const CtxDesc cd = s.desc[c];
    const int64_t r0 = a.row_off[c];
    const int32_t* reps = a.rep_list ? a.rep_list + r0 : nullptr;
    const uint32_t* xc = a.x + a.x_off[c];
    const uint4* yc = a.y + r0;
    const uintptr_t bits = (uintptr_t)xc | (uintptr_t)(4 * cd.xw);
    const int al = (bits & 15) == 0 ? 2 : ((bits & 7) == 0 ? 1 : 0);
    const int n = ke - kb;
    auto row_of = [&](int j) { return j < n ? (reps ? ld(reps + kb + j) : kb + j) : 0; };
    int next = row_of(threadIdx.x);
    // every lane of a warp in each round: the pivot walk is warp-uniform
    for (int base = 0; base < n; base += blockDim.x) {
        const int j = base + (int)threadIdx.x;
        const bool valid = j < n;
        const int i = next;
        next = row_of(j + (int)blockDim.x);
        uint32_t xin[WD], q[WD];
        uint4 y = valid ? ld(yc + i) : make_uint4(0, 0, 0, 0);
        load_row_words<WD>(xc + (int64_t)i * cd.xw, al, valid, cd.n, cd.xw, xin);
        make_q<WD>(xin, valid, s.raw, q);
        check_words<WD, 0>(q, y, S, Ps, Ds);
        uint32_t resid = 0;
#pragma unroll
        for (int w = 0; w < WD; ++w) resid |= q[w] & ~Ps[w];
        if (valid) flags[j] = resid ? 2 : (nonzero4(y) ? 1 : 0);
    }
}

// Shared memory of the check: the basis (a slot of row_stride words per
// column), the chunk's classes (CHECK_CHUNK bytes), then CHECK_CTL_WORDS of
// control (the pivot words, those whose rows have other columns too, the
// claimed chunk, the chunk's sums, the pivots).
constexpr int CHECK_CTL_WORDS = 64 + 16 * WIDE_M_WD;
constexpr int CHECK_SMEM_BYTES = 4 * CHECK_BASIS_WORDS + CHECK_CHUNK + 4 * CHECK_CTL_WORDS;

__global__ void __launch_bounds__(256, 3) check_snap_kernel(StoreDev s, CheckArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) uint32_t smem[];
    uint32_t* const S = smem;
    uint8_t* const flags = reinterpret_cast<uint8_t*>(smem + CHECK_BASIS_WORDS);
    uint32_t* const ctl = smem + CHECK_BASIS_WORDS + CHECK_CHUNK / 4;
    uint32_t* const Ps = ctl;       // 24 pivot words (WIDE_M_WD at most)
    uint32_t* const Ds = ctl + 24;  // 24 words
    uint16_t* const list = reinterpret_cast<uint16_t*>(ctl + 64);  // 32 * WIDE_M_WD columns at most
    int* const s_c = reinterpret_cast<int*>(ctl + 48);
    int* const s_k = s_c + 1;
    int* const s_first_out = s_c + 2;
    unsigned long long* const s_cnt = reinterpret_cast<unsigned long long*>(ctl + 52);
    long long* const s_first = reinterpret_cast<long long*>(ctl + 54);
    const int t = threadIdx.x;
    // CTAs start at different contexts and go round; a CTA stays with a context
    // while it has chunks left.  A warp looks at 32 contexts at a time.
    const int nq = *a.snap_count;
    const int q0 = nq > 0 ? (int)((int64_t)blockIdx.x * nq / gridDim.x) : 0;
    int tried = 0, built = -1;
    auto reps_of = [&](int c) {
        return a.rep_list ? a.rep_count[c] : (int)(a.row_off[c + 1] - a.row_off[c]);
    };
    for (;;) {
        if (t < 32) {
            int c = -1, k = 0;
            if (built >= 0) {
                if (t == 0) k = atomicAdd(a.ctr + built, 1);
                k = __shfl_sync(FULL, k, 0);
                if (chunk_exists(a.snap_start[built], k, CHECK_CHUNK, reps_of(built))) c = built;
            }
            while (c < 0 && tried < nq) {
                int cq = -1;
                if (tried + t < nq) {
                    const int at = q0 + tried + t;
                    cq = a.snap_list[at < nq ? at : at - nq];
                    if (!chunk_exists(a.snap_start[cq], __ldcg(a.ctr + cq), CHECK_CHUNK, reps_of(cq))) cq = -1;
                }
                const uint32_t left = __ballot_sync(FULL, cq >= 0);
                if (!left) {
                    tried += 32;
                    continue;
                }
                cq = __shfl_sync(FULL, cq, __ffs(left) - 1);
                if (t == 0) k = atomicAdd(a.ctr + cq, 1);
                k = __shfl_sync(FULL, k, 0);
                if (chunk_exists(a.snap_start[cq], k, CHECK_CHUNK, reps_of(cq))) c = cq;
            }
            if (t == 0) {
                *s_c = c;
                *s_k = k;
                *s_first_out = INT_MAX;
                *s_cnt = 0ull;
                *s_first = LLONG_MAX;
            }
        }
        __syncthreads();
        const int c = *s_c;
        const int ck = *s_k;
        if (c < 0) break;
        const CtxDesc cd = s.desc[c];
        const int R = reps_of(c);
        const int st0 = a.snap_start[c];
        const int kb = st0 + ck * CHECK_CHUNK;
        const int ke = step_to(kb, CHECK_CHUNK, R);
        if (built != c) {  // the basis into shared memory (pivot rows only)
            if (t < 24) {
                Ps[t] = (t < cd.wd) ? s.pivot[cd.pw_off + t] : 0u;
                Ds[t] = 0u;
            }
            __syncthreads();
            // the stride of the instance that checks it (rows of 10..17 words: the 17-word one)
            const int rs = row_stride(cd.wd <= NARROW_WD ? cd.wd : WIDE_M_WD);
            int np = 0;  // the pivots in a list, then a thread a word of their rows
            for (int v = 0; v < cd.wd; ++v) {
                const uint32_t P = Ps[v];
                const int b = t - (32 * v & 255);
                if (b >= 0 && b < 32 && ((P >> b) & 1u)) list[np + __popc(P & ((1u << b) - 1u))] = (uint16_t)(32 * v + b);
                np += __popc(P);
            }
            __syncthreads();
            for (int r = t; r < np; r += blockDim.x)
                *reinterpret_cast<uint4*>(S + list[r] * rs) = s.bz[cd.slot_off + list[r]];
            const int per = rs - 4, all = np * per;
#pragma unroll 4
            for (int j = t; j < all; j += 256) {
                const int r = j / per, v = j - r * per, kk = list[r];
                const uint32_t e = v < cd.wd ? s.bx[cd.xw_off + (int64_t)kk * cd.wd + v] : 0u;
                S[kk * rs + 4 + v] = e;
                if (v < cd.wd && (e & ~Ps[v])) atomicOr(Ds + (kk >> 5), 1u << (kk & 31));
            }
            built = c;
            __syncthreads();
        }
#define F2_CHECK(W) check_chunk<W>(s, a, c, kb, ke, S, Ps, Ds, flags)
        switch (cd.wd) {
        case 1: F2_CHECK(1); break;
        case 2: F2_CHECK(2); break;
        case 3: F2_CHECK(3); break;
        case 4: F2_CHECK(4); break;
        case 5: F2_CHECK(5); break;
        case 6: F2_CHECK(6); break;
        case 7: F2_CHECK(7); break;
        case 8: F2_CHECK(8); break;
        case 9: F2_CHECK(9); break;
        default: F2_CHECK(WIDE_M_WD); break;
        }
#undef F2_CHECK
        __syncthreads();
        // the first representative outside the span, then the contradictions
        // before it (weights: the representative and its repeats)
        for (int j = t; j < ke - kb; j += blockDim.x)
            if (flags[j] == 2) atomicMin(s_first_out, kb + j);
        __syncthreads();
        const int fo = *s_first_out;
        unsigned long long cnt = 0;
        long long first = LLONG_MAX;
        for (int j = t; j < ke - kb && kb + j < fo; j += blockDim.x) {
            if (flags[j] != 1) continue;
            const int k = kb + j;
            const int i = a.rep_list ? ld(a.rep_list + a.row_off[c] + k) : k;
            cnt += 1u + (a.rep_dup ? (uint32_t)ld(a.rep_dup + a.row_off[c] + k) : 0u);
            first = min(first, (long long)i);
        }
        if (cnt) {
            atomicAdd(s_cnt, cnt);
            atomicMin(s_first, first);
        }
        __syncthreads();
        if (t == 0) {
            const int64_t slot = check_slot(a, c) + ck;
            const unsigned long long sc = *s_cnt;
            const long long sf = *s_first;
            a.rec[2 * slot] = make_uint4((uint32_t)fo, (uint32_t)sc, (uint32_t)(sc >> 32), 0u);
            a.rec[2 * slot + 1] = make_uint4((uint32_t)sf, (uint32_t)((unsigned long long)sf >> 32), 0u, 0u);
            __threadfence();
            const int nch = chunk_count(st0, CHECK_CHUNK, R);
            if (atomicAdd(a.ctr + s.num_ctx + c, 1) == nch - 1) {  // the context's last chunk
                __threadfence();
                const int64_t s0 = check_slot(a, c);
                int f = INT_MAX;
                for (int k = 0; k < nch; ++k) f = min(f, (int)__ldcg(a.rec + 2 * (s0 + k)).x);
                unsigned long long tot = 0;
                long long fi = LLONG_MAX;
                for (int k = 0; k < nch; ++k) {
                    if (st0 + k * CHECK_CHUNK >= f) break;  // chunks past the first outside
                    const uint4 r = __ldcg(a.rec + 2 * (s0 + k));
                    const uint4 r2 = __ldcg(a.rec + 2 * (s0 + k) + 1);
                    tot += (unsigned long long)r.y | ((unsigned long long)r.z << 32);
                    fi = min(fi, (long long)((unsigned long long)r2.x | ((unsigned long long)r2.y << 32)));
                }
                const long long seen = s.rows_seen[c];
                if (tot) {
                    s.n_contra[c] += tot;
                    s.contra[c] = 1;
                    if (s.first_contra[c] < 0) s.first_contra[c] = seen + fi;
                }
                if (f == INT_MAX) {
                    s.rows_seen[c] = seen + (a.row_off[c + 1] - a.row_off[c]);
                } else {  // the rest from the first representative outside the span
                    a.resume_from[c] = f;
                    a.resume_list[atomicAdd(a.resume_count, 1)] = c;
                }
            }
        }
        __syncthreads();
    }
}

// Validate the batch and order the work longest-first, in three kernels:
// per-context keys and a histogram (grid), the bucket offsets (one block),
// and the scatter into the queue (grid).  A key is (class, work bucket,
// width); within a class, buckets run from the most work to the least and,
// inside a bucket, widths in increasing order (so few template variants run
// at once).
//   mode 0 (dedup plan): every valid non-empty context of more than dedup_min
//     rows and at most DD_XW_WIDE feature words goes to the warp, quad or CTA
//     dedup queue by its row count, the others straight to an elimination
//     queue; rep_count[c] becomes 0 (filled by the dedup pass), -1 (invalid,
//     skipped) or all_rows(T) (every row is its own representative);
//   mode 1 (elimination plan): contexts with rows to eliminate go to the
//     warp, CTA or wide elimination queue.  After a mode-0 plan that sent no
//     context to the duplicate pass it has nothing to do and returns.
constexpr int PLAN_SUB = PLAN_BUCKETS * NARROW_WD;  // (bucket, width) keys per class
constexpr int PLAN_KEYS = NUM_CLASSES * PLAN_SUB;
static_assert(PLAN_KEYS <= PLAN_HIST_WORDS, "the plan histogram holds every key");

// Scratch that a learn call counts in, cleared by the first plan of the call
// where one block plans (plan_small_kernel), else by a fill before it.
struct PlanZero {
    int* work;                    // CNT_WORK .. CNT_WORDS of the counters; NULL: cleared already
    int32_t* shard_done;          // [C]
    int* full_ctr;                // [2C], and the late count at [4C]
    unsigned long long* full_cnt; // [C]
    unsigned long long* full_first;  // [C], all ones
    int* hand;                    // two counts, and [2C] from 2 + 4C; NULL: not used in this call
};

struct PlanArgs {
    PlanZero zero;
    const int64_t* row_off;
    const int64_t* x_off;
    int64_t total_rows;
    int64_t total_xw;
    int32_t* rep_count;
    int mode;
    int warp_region_words;
    int64_t heavy_rows;
    int64_t warp_work;
    int dedup_min; // mode 0: contexts of at most this many rows are not deduplicated
    int after;     // mode 1: a mode-0 plan ran before
    int scale;     // mode 1: scale heavy_rows / warp_work to the totals of the duplicate pass
    int num_sms;
    long long shard_work;  // mode 0: rows x (xw + 4) of one shard share; 0 = no splitting
    int max_shards;        // mode 0: most shards of one context
    int shard_cap;         // mode 0: queue slots for shard items beyond one per context
    int32_t* queue;
    int32_t* keybuf;
    int* hist;     // PLAN_KEYS counts (zeroed before plan_key_kernel), then cursors
    int hist_zeroed;  // hist is zero already (else launch_plan clears it)
    int* counters;
};

// Ownership thresholds of the elimination plan, scaled to the call's work
// when the duplicate pass has measured it: a warp-owned context must not run
// (dependent round after round) much longer than the whole call.
struct PlanLimits {
    long long heavy_rows, warp_work;
};
__device__ __forceinline__ PlanLimits plan_limits(const PlanArgs& p)
{
    PlanLimits L{p.heavy_rows, p.warp_work};
    if (p.mode == 1 && p.scale) {
        const unsigned long long tw = *reinterpret_cast<const unsigned long long*>(p.counters + CNT_WORK);
        const unsigned long long tr = *reinterpret_cast<const unsigned long long*>(p.counters + CNT_REPS);
        const long long hr = (long long)(tr / ((unsigned long long)p.num_sms * HEAVY_REPS_DIV));
        const long long ww = (long long)(tw / ((unsigned long long)p.num_sms * WARP_WORK_DIV));
        L.heavy_rows = hr < HEAVY_ROWS_MIN ? HEAVY_ROWS_MIN : (hr > L.heavy_rows ? L.heavy_rows : hr);
        L.warp_work = ww < WARP_WORK_MIN ? WARP_WORK_MIN : (ww > L.warp_work ? L.warp_work : ww);
    }
    return L;
}

// What a plan reads of context c, all loads independent.
struct PlanRow {
    CtxDesc cd;
    int64_t a0, a1, x0;
    int rank, reps;
};
__device__ __forceinline__ PlanRow plan_load(const StoreDev& s, const PlanArgs& p, int c)
{
    PlanRow r{};
    r.cd = s.desc[c];
    r.rank = s.rank[c];
    if (p.mode == 1 && p.rep_count) {
        r.reps = p.rep_count[c];
    } else {
        r.a0 = p.row_off[c];
        r.a1 = p.row_off[c + 1];
        r.x0 = p.x_off[c];
    }
    return r;
}

// Validates context c's part of the batch and returns its key (bits 0..15:
// class, work bucket and width; bits 16..18: shards - 1), or -1 when it has
// no work; nsh_out = its queue items.
__device__ __forceinline__ int plan_key_of(const StoreDev& s, const PlanArgs& p, const PlanLimits& L, int c,
                                           const PlanRow& r, int& nsh_out)
{
    nsh_out = 0;
    const CtxDesc& cd = r.cd;
    int64_t R;
    bool direct = p.mode == 1;  // to an elimination queue
    if (p.mode == 1 && p.rep_count) {
        R = r.reps;
        if (R <= -2) R = rows_of((int32_t)R);
    } else {
        const int64_t a0 = r.a0, a1 = r.a1;
        const int64_t rows = a1 - a0;
        const int64_t x0 = r.x0;
        const bool ok = a0 >= 0 && rows >= 0 && rows < (1ll << 31) && a1 <= p.total_rows && x0 >= 0 &&
                        rows <= p.total_xw && x0 + rows * cd.xw <= p.total_xw;
        if (!ok) record_status(s.status, F2_ERR_ROWS);
        R = ok ? rows : -1;
        if (p.mode == 0 && p.rep_count) {
            // wide rows and short contexts are not deduplicated; rows of a
            // full-rank context are checked one by one (verify_full_kernel)
            if (R > 0 && (cd.xw > DD_XW_WIDE || R <= p.dedup_min || r.rank == cd.d)) {
                p.rep_count[c] = all_rows(R);
                direct = true;
            } else {
                p.rep_count[c] = (R > 0) ? 0 : (int32_t)R;
            }
        }
    }
    int key = -1;
    if (R > 0) {
        int cls;
        unsigned long long work;
        if (!direct) {
            cls = (R <= DD_WARP_MAX_ROWS) ? CLS_DD_WARP : (R <= DD_QUAD_MAX_ROWS ? CLS_DD_QUAD : CLS_DD_CTA);
            if (cd.xw > DD_XW) cls += CLS_DDW_CTA - CLS_DD_CTA;  // the 10..16-word instance
            work = (unsigned long long)R * (unsigned long long)(cd.xw + 4);
        } else {
            const bool heavy = elim_words(cd.d, cd.wd) > p.warp_region_words || R >= L.heavy_rows ||
                               R * cd.d > L.warp_work;
            if (r.rank == cd.d) cls = CLS_FULL;
            else if (cd.wd > NARROW_WD) cls = (cd.wd <= WIDE_M_WD) ? CLS_WIDE_M : CLS_WIDE;
            else if (cd.wd <= SMALL_WD) cls = heavy ? CLS_CTA_S : CLS_WARP_S;
            else cls = heavy ? CLS_CTA : CLS_WARP;
            work = (unsigned long long)R * (unsigned long long)(cd.wd + 4) * (unsigned long long)cd.d;
        }
        int nsh = 1;
        if (!direct && p.shard_work > 0) {
            if (F2_DD_QUAD_PROMOTE && (cls == CLS_DD_QUAD || cls == CLS_DDW_QUAD) && R >= DD_PROMOTE_MIN_ROWS &&
                (long long)work * DD_QUAD_SHARE > p.shard_work)
                cls += CLS_DD_CTA - CLS_DD_QUAD;
            if (cls == CLS_DD_CTA || cls == CLS_DDW_CTA) {
                long long k = (long long)work / p.shard_work;
                if (DD_SHARD_ROWS > 0 && (R + DD_SHARD_ROWS - 1) / DD_SHARD_ROWS > k)
                    k = (R + DD_SHARD_ROWS - 1) / DD_SHARD_ROWS;
                if (k > R / DD_SHARD_MIN_ROWS) k = R / DD_SHARD_MIN_ROWS;
                nsh = k < 1 ? 1 : (k > p.max_shards ? p.max_shards : (int)k);
                // the queue holds shard_cap extra items; past that, contexts stay whole
                if (nsh > 1 && atomicAdd(p.counters + CNT_SHARDS, nsh - 1) + (nsh - 1) > p.shard_cap) nsh = 1;
                work /= (unsigned long long)nsh;
            }
        }
        int bucket = 63 - __clzll(work);
        if (bucket >= PLAN_BUCKETS) bucket = PLAN_BUCKETS - 1;
        const int width = direct ? cd.wd : cd.xw;
        const int sub = (PLAN_BUCKETS - 1 - bucket) * NARROW_WD + (width > NARROW_WD ? NARROW_WD : width) - 1;
        key = cls * PLAN_SUB + sub;
        key |= (nsh - 1) << 16;
        nsh_out = nsh;
    }
    return key;
}

// The second plan of a call whose first one left nothing to the duplicate pass.
__device__ __forceinline__ bool plan_done(const PlanArgs& p) { return p.after && p.counters[CNT_DEDUPED] == 0; }

__global__ void __launch_bounds__(256) plan_key_kernel(StoreDev s, PlanArgs p)
{
    pdl_wait();
    if (plan_done(p)) return;
    __shared__ int hist[PLAN_KEYS];
    for (int i = threadIdx.x; i < PLAN_KEYS; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    const PlanLimits L = plan_limits(p);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < s.num_ctx; c += gridDim.x * blockDim.x) {
        int nsh;
        const int kv = plan_key_of(s, p, L, c, plan_load(s, p, c), nsh);
        if (kv >= 0) atomicAdd(&hist[kv & 0xFFFF], nsh);
        p.keybuf[c] = kv;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < PLAN_KEYS; i += blockDim.x)
        if (hist[i]) atomicAdd(p.hist + i, hist[i]);
}

// Exclusive scan of the key counts `hist` (global or shared) in key order by
// one block of 1024 threads; hist becomes the cursors and the class blocks of
// `counters` (first item, count, head) are set.
__device__ void plan_scan_block(int* hist, int* counters, int mode)
{
    constexpr int PER = (PLAN_KEYS + 1023) / 1024;
    __shared__ int wsum[32];
    __shared__ int s_total;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int v[PER];
    int tot = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int k = t * PER + j;
        v[j] = (k < PLAN_KEYS) ? hist[k] : 0;
        tot += v[j];
    }
    int inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = wsum[lane];
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(FULL, wi, o);
            if (lane >= o) wi += u;
        }
        wsum[lane] = wi - w;
        if (lane == 31) s_total = wi;
    }
    __syncthreads();
    int run = wsum[warp] + inc - tot;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int k = t * PER + j;
        if (k < PLAN_KEYS) hist[k] = run;  // becomes the cursor of key k
        run += v[j];
    }
    __syncthreads();
    // a class's items run from the cursor of its first key to that of the next class
    if (t < NUM_CLASSES) {
        const int b = hist[t * PLAN_SUB];
        const int e = (t + 1 < NUM_CLASSES) ? hist[(t + 1) * PLAN_SUB] : s_total;
        counters[CNT_BEGIN + t] = b;
        counters[CNT_HEAD + t] = 0;
        counters[CNT_COUNT + t] = e - b;
    }
    if (mode == 0 && t == 0)  // items of the duplicate pass (its classes are consecutive keys)
        counters[CNT_DEDUPED] = (hist[(CLS_DD_WARP + 1) * PLAN_SUB] - hist[CLS_DD_CTA * PLAN_SUB]) +
                                (hist[(CLS_DDW_WARP + 1) * PLAN_SUB] - hist[CLS_DDW_CTA * PLAN_SUB]);
}

__global__ void __launch_bounds__(1024) plan_scan_kernel(PlanArgs p)
{
    pdl_wait();
    if (plan_done(p)) return;
    plan_scan_block(p.hist, p.counters, p.mode);
}

// Queue item(s) of context c with key kv at the cursor of its key.
__device__ __forceinline__ void plan_place(const PlanArgs& p, int* cursor, int c, int kv)
{
    const int key = kv & 0xFFFF, nsh = (kv >> 16) + 1;
    if (nsh == 1) {
        p.queue[atomicAdd(cursor + key, 1)] = c;
    } else {  // one item per shard
        const int q0 = atomicAdd(cursor + key, nsh);
        for (int k = 0; k < nsh; ++k)
            p.queue[q0 + k] = (int32_t)((uint32_t)c | ((uint32_t)k << 24) | ((uint32_t)(nsh - 1) << 28));
    }
}

__global__ void __launch_bounds__(256) plan_scatter_kernel(StoreDev s, PlanArgs p)
{
    pdl_wait();
    if (plan_done(p)) return;
    // the lanes of a warp with the same key take their slots with one atomic
    const int lane = threadIdx.x & 31;
    for (int b = blockIdx.x * blockDim.x; b < s.num_ctx; b += gridDim.x * blockDim.x) {
        const int c = b + (int)threadIdx.x;
        const int kv = (c < s.num_ctx) ? p.keybuf[c] : -1;
        const bool single = kv >= 0 && (kv >> 16) == 0;
        const int key = single ? kv : -1 - lane;  // a lane of its own unless a single item
        const unsigned peers = __match_any_sync(FULL, key);
        if (single) {
            const int leader = __ffs(peers) - 1;
            int q0 = 0;
            if (lane == leader) q0 = atomicAdd(p.hist + key, __popc(peers));
            q0 = __shfl_sync(peers, q0, leader);
            p.queue[q0 + __popc(peers & ((1u << lane) - 1u))] = c;
        } else if (kv >= 0) {
            plan_place(p, p.hist, c, kv);
        }
    }
}

// The three steps in one block, the histogram in shared memory, for stores
// of at most PLAN_SMALL_MAX contexts (one launch instead of a memset and
// three kernels: what a small batch waits for).
constexpr int PLAN_SMALL_MAX = 8192;
__global__ void __launch_bounds__(1024) plan_small_kernel(StoreDev s, PlanArgs p)
{
    pdl_wait();
    __shared__ int hist[PLAN_KEYS];
    if (plan_done(p)) return;
    for (int i = threadIdx.x; i < PLAN_KEYS; i += blockDim.x) hist[i] = 0;
    if (p.zero.work) {
        const PlanZero& z = p.zero;
        const int C = s.num_ctx;
        if (threadIdx.x < CNT_WORDS - CNT_WORK) z.work[threadIdx.x] = 0;
        if (threadIdx.x == 0) z.full_ctr[4 * C] = 0;
        if (threadIdx.x < 2 && z.hand) z.hand[threadIdx.x] = 0;
        for (int c = threadIdx.x; c < C; c += blockDim.x) {
            z.shard_done[c] = 0;
            z.full_ctr[c] = z.full_ctr[C + c] = 0;
            z.full_cnt[c] = 0ull;
            z.full_first[c] = ~0ull;
            if (z.hand) z.hand[2 + 4 * C + c] = z.hand[2 + 5 * C + c] = 0;
        }
    }
    __syncthreads();
    const PlanLimits L = plan_limits(p);
    constexpr int PER = PLAN_SMALL_MAX / 1024;
    const int lane = threadIdx.x & 31;
    int kv[PER];
    bool same[PER];
    PlanRow row{}, next{};
    if ((int)threadIdx.x < s.num_ctx) next = plan_load(s, p, threadIdx.x);
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int c = j * 1024 + (int)threadIdx.x;
        kv[j] = -1;
        same[j] = false;
        if (j * 1024 >= s.num_ctx) continue;
        row = next;
        if (c + 1024 < s.num_ctx) next = plan_load(s, p, c + 1024);
        int nsh = 0;
        if (c < s.num_ctx) kv[j] = plan_key_of(s, p, L, c, row, nsh);
        // The contexts of a store are often alike: one atomic for a warp whose
        // lanes all have the same key (sorting other keys out took longer than
        // an atomic each: 17.5 and 11.0 us for the plans of 4,096 contexts of
        // many widths and lengths, 19.1 and 14.3 with __match_any_sync).
        int alike;
        __match_all_sync(FULL, nsh == 1 ? kv[j] : -1 - lane, &alike);
        same[j] = alike;
        if (alike) {
            if (lane == 0) atomicAdd(&hist[kv[j]], 32);
        } else if (kv[j] >= 0) {
            atomicAdd(&hist[kv[j] & 0xFFFF], nsh);
        }
    }
    __syncthreads();
    plan_scan_block(hist, p.counters, p.mode);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int c = j * 1024 + (int)threadIdx.x;
        if (same[j]) {
            int q0 = 0;
            if (lane == 0) q0 = atomicAdd(hist + kv[j], 32);
            p.queue[__shfl_sync(FULL, q0, 0) + lane] = c;
        } else if (kv[j] >= 0) {
            plan_place(p, hist, c, kv[j]);
        }
    }
}

int launch_plan(const StoreDev& sd, const PlanArgs& pa, int num_sms, cudaStream_t cs)
{
    if (sd.num_ctx <= PLAN_SMALL_MAX) {
        f2_launch(plan_small_kernel, 1, 1024, 0, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, pa);
        return f2_cuda_status(cudaGetLastError());
    }
    if (!pa.hist_zeroed) {
        const cudaError_t e = cudaMemsetAsync(pa.hist, 0, sizeof(int) * PLAN_KEYS, cs);
        if (e != cudaSuccess) return f2_cuda_status(e);
    }
    int blocks = (sd.num_ctx + 255) / 256;
    if (blocks > num_sms * 2) blocks = num_sms * 2;
    if (blocks < 1) blocks = 1;
    f2_launch(plan_key_kernel, blocks, 256, 0, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, pa);
    f2_launch(plan_scan_kernel, 1, 1024, 0, cs, sd.num_ctx <= EARLY_MAX_CTX, pa);
    f2_launch(plan_scatter_kernel, blocks, 256, 0, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, pa);
    return f2_cuda_status(cudaGetLastError());
}

inline bool is_aligned(const void* p, size_t al) { return ((uintptr_t)p % al) == 0; }

// ---------------------------------------------------------------------------
// Full-rank contexts.  When rank = d at the start of a call the reduced basis
// is the identity (every coordinate is a pivot and a reduced row has no other
// pivot bit), so every row lies in the span and T(q) = XOR of z_k over the set
// coordinates k of q.  A row is redundant if its word equals T(phi(x)) and a
// contradiction otherwise (Sec. 2.2 steps (2)-(3)); nothing is inserted, so
// the rows are independent.  CTAs claim chunks of FULL_CHUNK rows of a
// context, look T up in a 4-bit table of the z_k in shared memory (built when
// a CTA moves to a context: entry 16p + v = XOR of z_{4p+b} over the bits b
// of v), and the last chunk of a context commits the contradiction count,
// the first contradicting row and rows_seen.
// ---------------------------------------------------------------------------
constexpr int FULL_STAGE = FULL_THREADS;  // rows staged in shared memory at a time (one per thread)
// The table: low and high halves of the 16 entries of each group of four
// coordinates in two planes of 8-byte entries (a warp's lookups at one group
// fall in distinct banks), groups padded with zero entries to a multiple of
// eight (one 32-bit word of q = eight lookups, no bounds test), the high
// plane at a fixed distance from the low one and the base 1024-byte aligned,
// so that an entry's address is the word's base OR the nibble times eight,
// with the group and the plane in the loads' immediate offsets.
constexpr int FULL_NP_MAX = 8 * ((MAX_D + 31) / 32);      // 264 groups
constexpr int FULL_ZH_BYTES = FULL_NP_MAX * 16 * 8;        // 33,792: low plane, then the high plane
constexpr int FULL_TABLE_WORDS = 2 * FULL_ZH_BYTES / 4 + 256;  // both planes + alignment slack

__global__ void __launch_bounds__(FULL_THREADS) verify_full_kernel(StoreDev s, FullArgs a)
{
    pdl_wait();
    extern __shared__ uint4 full_smem[];
    // the table at the first 1024-byte boundary of the dynamic shared memory
    const uint32_t pad = ((1024u - (smem_addr(full_smem) & 1023u)) & 1023u) / 4u;
    uint32_t* const tabw = reinterpret_cast<uint32_t*>(full_smem) + pad;
    uint32_t* const stage = reinterpret_cast<uint32_t*>(full_smem) + a.table_words;
    __shared__ int s_q, s_k;
    __shared__ unsigned long long s_cnt, s_first;
    const int t = threadIdx.x, lane = t & 31;
    const FullList list(a);
    const int q0 = (int)((long long)blockIdx.x * list.n / gridDim.x);
    int q = -1, tried = 0, built = -1;
    for (;;) {
        if (t < 32) {
            int k;
            const int qn = full_claim(s, a, list, false, q0, q, tried, lane, k);
            if (t == 0) {
                s_q = qn;
                s_k = k;
                s_cnt = 0ull;
                s_first = ~0ull;
            }
        }
        __syncthreads();
        q = s_q;
        if (q < 0) break;
        const int k = s_k;
        const int c = list.ctx(a, q);
        const int64_t i_first = list.start(a, q, c);
        const CtxDesc cd = s.desc[c];
        const int np = (cd.d + 3) >> 2;
        const int nw = (np + 7) >> 3;  // words of q, eight groups each
        uint2* Zl = reinterpret_cast<uint2*>(tabw);
        uint2* Zh = Zl + FULL_ZH_BYTES / 8;
        if (built != c) {
            for (int j = t; j < 4 * np; j += FULL_THREADS) {
                const uint4 z = (j < cd.d) ? ld(s.bz + cd.slot_off + j) : make_uint4(0, 0, 0, 0);
                const int e = (j >> 2) * 16 + (1 << (j & 3));
                Zl[e] = make_uint2(z.x, z.y);
                Zh[e] = make_uint2(z.z, z.w);
                if ((j & 3) == 0) {
                    Zl[e - 1] = make_uint2(0, 0);
                    Zh[e - 1] = make_uint2(0, 0);
                }
            }
            __syncthreads();
            for (int f = t; f < 16 * np; f += FULL_THREADS) {
                const int v = f & 15;
                if (__popc(v) < 2) continue;
                const int eb = f & ~15;
                uint2 lo = make_uint2(0, 0), hi = make_uint2(0, 0);
#pragma unroll
                for (int bb = 0; bb < 4; ++bb) {
                    if ((v >> bb) & 1) {
                        const uint2 l = Zl[eb + (1 << bb)], h = Zh[eb + (1 << bb)];
                        lo.x ^= l.x;
                        lo.y ^= l.y;
                        hi.x ^= h.x;
                        hi.y ^= h.y;
                    }
                }
                Zl[f] = lo;
                Zh[f] = hi;
            }
            for (int f = 16 * np + t; f < 128 * nw; f += FULL_THREADS) {  // padding groups
                Zl[f] = make_uint2(0, 0);
                Zh[f] = make_uint2(0, 0);
            }
            built = c;
        }
        const int64_t r0 = a.row_off[c];
        const int64_t T = a.row_off[c + 1] - r0;
        const int64_t i0 = i_first + (int64_t)k * FULL_CHUNK;
        const int64_t i1 = (i0 + FULL_CHUNK < T) ? i0 + FULL_CHUNK : T;
        const uint32_t* xc = a.x + a.x_off[c];
        const int xw = cd.xw;
        const int sst = xw | 1;  // odd staging stride: a row per lane reads distinct banks
        const uint32_t lm = (cd.n & 31) ? (1u << (cd.n & 31)) - 1u : 0xFFFFFFFFu;
        unsigned long long cnt = 0ull, first = ~0ull;
        for (int64_t b0 = i0; b0 < i1; b0 += FULL_STAGE) {
            const int nb = (int)((i1 - b0) < FULL_STAGE ? (i1 - b0) : FULL_STAGE);
            __syncthreads();  // the table is complete / the previous rows are consumed
            const uint32_t* src = xc + b0 * xw;  // the rows are contiguous
            {
                // word w = r * xw + v of the block, stepped by FULL_THREADS
                // without a division per word
                int r = t / xw, v = t - (t / xw) * xw;
                const int dr = FULL_THREADS / xw, dv = FULL_THREADS - dr * xw;
                for (int w = t; w < nb * xw; w += FULL_THREADS) {
                    stage[r * sst + v] = ld(src + w);
                    r += dr;
                    v += dv;
                    if (v >= xw) {
                        v -= xw;
                        ++r;
                    }
                }
            }
            __syncthreads();
            if (t < nb) {
                const int64_t i = b0 + t;
                const uint4 yi = ld(a.y + r0 + i);
                const uint32_t* xr = stage + t * sst;
                uint32_t a0 = 0, a1 = 0, a2 = 0, a3 = 0, prev = 0;
                const char* const zt = reinterpret_cast<const char*>(tabw);
                for (int w = 0; w < nw; ++w) {
                    uint32_t xv = (w < xw) ? xr[w] : 0u;
                    if (w == xw - 1) xv &= lm;
                    uint32_t qw;
                    if (s.raw) {
                        qw = xv;
                    } else {  // phi(x) = [1 || x]: the constant at index 0, x bit j at 1 + j
                        qw = (xv << 1) | (prev >> 31) | (w == 0 ? 1u : 0u);
                        prev = xv;
                    }
                    const char* const zb = zt + w * 1024;
                    // two lookups a step: entry byte offset = nibble * 8
#pragma unroll
                    for (int h = 0; h < 8; h += 2) {
                        const uint32_t oa = (h == 0) ? ((qw << 3) & 0x78u) : ((qw >> (4 * h - 3)) & 0x78u);
                        const uint32_t ob = (qw >> (4 * h + 1)) & 0x78u;
                        const uint2 la = *reinterpret_cast<const uint2*>(zb + oa + 128 * h);
                        const uint2 ha = *reinterpret_cast<const uint2*>(zb + oa + FULL_ZH_BYTES + 128 * h);
                        const uint2 lb = *reinterpret_cast<const uint2*>(zb + ob + 128 * (h + 1));
                        const uint2 hb = *reinterpret_cast<const uint2*>(zb + ob + FULL_ZH_BYTES + 128 * (h + 1));
                        a0 ^= la.x ^ lb.x;
                        a1 ^= la.y ^ lb.y;
                        a2 ^= ha.x ^ hb.x;
                        a3 ^= ha.y ^ hb.y;
                    }
                }
                if (a0 != yi.x || a1 != yi.y || a2 != yi.z || a3 != yi.w) {
                    ++cnt;
                    if ((unsigned long long)i < first) first = (unsigned long long)i;
                }
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cnt += __shfl_xor_sync(FULL, cnt, o);
            const unsigned long long f2 = __shfl_xor_sync(FULL, first, o);
            first = f2 < first ? f2 : first;
        }
        if (lane == 0 && cnt) {
            atomicAdd(&s_cnt, cnt);
            atomicMin(&s_first, first);
        }
        __syncthreads();
        if (t == 0) full_commit(s, a, c, i_first, T, s_cnt, s_first, false);
        __syncthreads();
    }
}

// The default hand-off (see f2_learn_batched): calls of at least this many
// rows on stores with rows of 10..17 words, contexts with at least this many
// representatives left that walk their pivots.  On 10,000 contexts of parsed
// values (13.4M rows) the learn call takes 1,054 us; 1,060 from 1,024
// representatives on, 1,066 where a context must also hold a sixteenth of an
// SM's share of the call's work (1,102 with chunks of 512, where an eighth took
// 1,162).  Contexts that run against a lookup table stay: the check walks the
// pivots, which costs a context of high rank more than its table, and one context
// of 10..17 words would turn that on for a whole store.  With one such context,
// without the hand-off / with it / with it for contexts with a table too:
// 10,000 contexts of 100..256 features (16.3M rows) 2,343 / 2,362 / 2,642 us,
// 4,096 of 32..128 (2.5M) 308 / 321 / 350, 77,926 (80M) 2,459 / 2,482 / 2,534,
// 5,000 of parsed values of 128..256 bits (6.7M) 800 / 466 / 466; where a few long
// contexts with tables bound the call it would gain: 1,000 contexts (8.2M rows)
// 1,507 / 1,528 / 1,363, 5,000 of one parsed value 491 / 513 / 290.
constexpr int64_t HANDOFF_AUTO_ROWS = int64_t(1) << 20;
constexpr int HANDOFF_AUTO_REPS = 2048;

// A second stream for kernels that work on disjoint contexts: the first
// such kernel goes to `aux` (forked from the caller's stream), the others to
// the caller's stream, and join() makes the caller's stream wait for `aux`.
struct Fork {
    cudaStream_t cs, aux;
    cudaEvent_t ev_fork, ev_join;
    bool forked = false;
    cudaError_t e = cudaSuccess;
    cudaStream_t next(int kernels_left)
    {
        if (!aux || forked || kernels_left < 2) return cs;
        e = cudaEventRecord(ev_fork, cs);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(aux, ev_fork, 0);
        if (e != cudaSuccess) return cs;
        forked = true;
        return aux;
    }
    cudaError_t join()
    {
        if (!forked || e != cudaSuccess) return e;
        forked = false;
        e = cudaEventRecord(ev_join, aux);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(cs, ev_join, 0);
        return e;
    }
};

// Enqueue pass 2 (plan + kernels) for one batch.
int launch_elimination(const StoreDev& sd, const LearnArgs& la, const int64_t* row_off, const int64_t* x_off,
                       int64_t total_rows, int64_t total_xw, int32_t* rep_count, int64_t heavy_rows,
                       int64_t warp_work, int32_t* queue, int32_t* keybuf, int* hist, int num_sms,
                       const Widths& wv, int* full_ctr, unsigned long long* full_cnt,
                       unsigned long long* full_first, cudaStream_t cs, Fork* fk = nullptr, int scale = 0,
                       bool prezeroed = false, int64_t long_rows = DEFAULT_LONG_CALL_ROWS, const CheckArgs* check = nullptr,
                       const PlanZero& zero = PlanZero{}, int fail_wait = 0)
{
    // prezeroed: the caller has cleared full_ctr's first 2C words and late
    // count, full_cnt, full_first (to -1) and hist
    // full_ctr: chunks claimed [C], chunks done [C], late start [C], late list [C], late count,
    // rows taken by elim_open_kernel [C]
    const int C = sd.num_ctx;
    LearnArgs lx = la;
    lx.late_start = full_ctr + 2 * C;
    lx.late_list = full_ctr + 3 * C;
    lx.late_count = full_ctr + 4 * C;
    lx.open_from = full_ctr + 4 * C + 1;
    if (!prezeroed) {
        cudaError_t e0 = cudaMemsetAsync(full_ctr, 0, sizeof(int) * 2 * (size_t)C, cs);
        if (e0 == cudaSuccess) e0 = cudaMemsetAsync(lx.late_count, 0, sizeof(int), cs);
        if (e0 == cudaSuccess) e0 = cudaMemsetAsync(full_cnt, 0, sizeof(unsigned long long) * (size_t)C, cs);
        if (e0 == cudaSuccess) e0 = cudaMemsetAsync(full_first, 0xff, sizeof(unsigned long long) * (size_t)C, cs);
        if (e0 != cudaSuccess) return f2_cuda_status(e0);
    }
    PlanArgs pa;
    pa.zero = zero;
    pa.row_off = row_off;
    pa.x_off = x_off;
    pa.total_rows = total_rows;
    pa.total_xw = total_xw;
    pa.rep_count = rep_count;
    pa.mode = 1;
    pa.warp_region_words = la.warp_region_words;
    pa.heavy_rows = heavy_rows;
    pa.warp_work = warp_work;
    pa.dedup_min = 0;
    pa.after = rep_count != nullptr;
    pa.scale = scale;
    pa.num_sms = num_sms;
    pa.shard_work = 0;
    pa.max_shards = 1;
    pa.shard_cap = 0;
    pa.queue = queue;
    pa.keybuf = keybuf;
    pa.hist = hist;
    pa.hist_zeroed = prezeroed;
    pa.counters = la.counters;
    int rc = launch_plan(sd, pa, num_sms, cs);
    if (rc != F2_OK) return rc;
    // the width classes hold disjoint contexts: with a second stream their
    // kernels overlap (each fills the others' tails)
    Fork solo{cs, nullptr, nullptr, nullptr};
    Fork& f = fk ? *fk : solo;
    int left = (int)wv.has_narrow + (int)wv.has_wide + (int)wv.has_wide_m + (int)wv.has_small;
    auto eliminate = [&](const LearnArgs& lk) -> cudaError_t {
        cudaError_t er = cudaSuccess;
        auto stream = [&]() { return lk.resume_from ? cs : f.next(left--); };
        const bool resume = lk.resume_from != nullptr;
        if (er == cudaSuccess && wv.has_wide && !resume)  // wider contexts hand nothing off
            er = elim_launch_wide(sd, lk, wv.max_wide_d, false, num_sms, stream());
        if (er == cudaSuccess && wv.has_wide_m)
            er = elim_launch_wide(sd, lk, wv.max_wide_m_d, true, num_sms, stream());
        if (er == cudaSuccess && wv.has_narrow)
            er = elim_launch_narrow(sd, lk, wv.max_narrow_words, total_rows >= long_rows && !resume ? 4 : LEARN_WARPS,
                                    num_sms, stream());
        if (er == cudaSuccess && wv.has_small) er = elim_launch_small(sd, lk, wv.max_small_words, num_sms, stream());
        return er == cudaSuccess ? f.e : er;
    };
    cudaError_t e = eliminate(lx);
    if (e != cudaSuccess) return f2_cuda_status(e);
    e = f.join();
    if (e != cudaSuccess) return f2_cuda_status(e);
    if (check && la.handoff_min > 0) {
        // the handed-off contexts: their remaining representatives checked
        // in parallel, then any that met a representative outside the
        // span eliminated from there on
        const size_t csmem = CHECK_SMEM_BYTES;
        e = cudaFuncSetAttribute(check_snap_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csmem);
        if (e != cudaSuccess) return f2_cuda_status(e);
        f2_launch(check_snap_kernel, num_sms * 3, 256, csmem, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, *check);
        e = cudaGetLastError();
        if (e != cudaSuccess) return f2_cuda_status(e);
        LearnArgs lr = lx;
        lr.handoff_min = 0;
        lr.resume_from = check->resume_from;
        lr.resume_list = check->resume_list;
        lr.resume_count = check->resume_count;
        e = eliminate(lr);
        if (e != cudaSuccess) return f2_cuda_status(e);
    }
    {  // full-rank contexts: at the start of the call (the plan decides on the
       // device which, if any) or reached during it (listed by the kernels above)
        FullArgs fa;
        fa.row_off = row_off;
        fa.x_off = x_off;
        fa.x = la.x;
        fa.y = la.y;
        fa.queue = queue;
        fa.counters = la.counters;
        fa.ctr = full_ctr;
        fa.late_count = lx.late_count;
        fa.late_list = lx.late_list;
        fa.late_start = lx.late_start;
        fa.cnt = full_cnt;
        fa.first = full_first;
        fa.table_words = FULL_TABLE_WORDS;
        fa.fail_wait = fail_wait;
        fa.tensor = wv.has_tensor && total_rows >= TC_MIN_ROWS;
        if (fa.tensor) {
            e = verify_launch_tc(sd, fa, num_sms, cs);
            if (e != cudaSuccess) return f2_cuda_status(e);
        }
        const size_t smem = 4 * ((size_t)fa.table_words + (size_t)FULL_STAGE * (size_t)(wv.max_xw | 1));
        e = cudaFuncSetAttribute(verify_full_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return f2_cuda_status(e);
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, verify_full_kernel, FULL_THREADS, smem);
        if (e != cudaSuccess) return f2_cuda_status(e);
        if (per_sm < 1) per_sm = 1;
        f2_launch(verify_full_kernel, num_sms * per_sm, FULL_THREADS, smem, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, fa);
        e = cudaGetLastError();
        if (e != cudaSuccess) return f2_cuda_status(e);
    }
    return F2_OK;
}

Widths width_summary(const int32_t* n_bits, int32_t num_ctx, bool raw)
{
    Widths w;
    for (int32_t c = 0; c < num_ctx; ++c) {
        const int d = raw ? n_bits[c] : n_bits[c] + 1;
        const int wd = (d + 31) / 32;
        const int words = elim_words(d, wd);
        if (d > w.max_d) w.max_d = d;
        if (tensor_features(n_bits[c])) w.has_tensor = true;
        if ((n_bits[c] + 31) / 32 > w.max_xw) w.max_xw = (n_bits[c] + 31) / 32;
        if (wd <= SMALL_WD) {
            w.has_small = true;
            if (words > w.max_small_words) w.max_small_words = words;
        } else if (wd <= NARROW_WD) {
            w.has_narrow = true;
            if (words > w.max_narrow_words) w.max_narrow_words = words;
        } else if (wd <= WIDE_M_WD) {
            w.has_wide_m = true;
            if (d > w.max_wide_m_d) w.max_wide_m_d = d;
        } else {
            w.has_wide = true;
            if (d > w.max_wide_d) w.max_wide_d = d;
        }
    }
    return w;
}

}  // namespace

extern "C" int f2_learn_batched(f2_store* st, const int64_t* row_off, const uint32_t* x, const int64_t* x_off,
                                const uint32_t* y, int64_t total_rows, int64_t total_x_words,
                                f2_stream_t stream)
{
    F2_NVTX_RANGE("f2_learn_batched");
    if (!st || total_rows < 0 || total_x_words < 0) return F2_ERR_INVALID_ARG;
    if (st->num_ctx == 0) return F2_OK;
    if (!row_off || !x_off || (!x && total_x_words) || (!y && total_rows)) return F2_ERR_INVALID_ARG;
    if (!is_aligned(row_off, 8) || !is_aligned(x_off, 8) || !is_aligned(x, 4) || !is_aligned(y, 16))
        return F2_ERR_ALIGN;
    cudaStream_t cs = (cudaStream_t)stream;
    cudaError_t e;
    const bool dedup = st->dedup && total_rows > 0;
    if (dedup && total_rows > st->rep_capacity) {  // per-row scratch of pass 1, grown stream-ordered
        if (st->rep_list) cudaFreeAsync(st->rep_list, cs);
        if (st->rep_dup) cudaFreeAsync(st->rep_dup, cs);
        st->rep_list = st->rep_dup = nullptr;
        st->rep_capacity = 0;
        e = f2_dev_alloc(st, (void**)&st->rep_list, sizeof(int32_t) * (size_t)total_rows, cs, true);
        if (e == cudaSuccess) e = f2_dev_alloc(st, (void**)&st->rep_dup, sizeof(int32_t) * (size_t)total_rows, cs, true);
        if (e != cudaSuccess) return F2_ERR_OOM;
        st->rep_capacity = total_rows;
    }
    if (!st->widths_ready) {  // fixed by the widths: computed once per store
        st->widths = width_summary(st->n_bits.data(), st->num_ctx, (st->flags & F2_FLAG_RAW_FEATURES) != 0);
        st->widths_ready = true;
    }
    const Widths& wv = st->widths;
    // Hand-off of saturated contexts, in calls long enough to have some.  By
    // default only in calls with contexts of 10..17 words, whose rows cost most.
    const bool auto_hand = st->handoff_min < 0 && dedup && wv.has_wide_m && total_rows >= HANDOFF_AUTO_ROWS;
    int hand_min = auto_hand ? HANDOFF_AUTO_REPS
                         : (st->handoff_min > 0 && total_rows >= HANDOFF_CALL_FACTOR * st->handoff_min)
                             ? (int)st->handoff_min
                             : 0;
    // every scratch counter of the call, zeroed by one launch
    const size_t C = (size_t)st->num_ctx;
    if (hand_min > 0) {  // the check's chunk records, grown stream-ordered
        const int64_t slots = total_rows / CHECK_CHUNK + (int64_t)C + 1;
        if (slots > st->check_rec_cap) {
            if (st->check_rec) cudaFreeAsync(st->check_rec, cs);
            st->check_rec = nullptr;
            st->check_rec_cap = 0;
            if (f2_dev_alloc(st, (void**)&st->check_rec, 2 * sizeof(uint4) * (size_t)slots, cs, true) == cudaSuccess) {
                st->check_rec_cap = slots;
            } else {
                st->check_rec = nullptr;
                if (!auto_hand) return F2_ERR_OOM;
                hand_min = 0;  // not asked for: the call goes without
                (void)cudaGetLastError();
            }
        }
    }
    F2FillList zl;
    if (st->timing_on) {  // diagnostics: per-context timestamps of this call
        const size_t bytes = sizeof(unsigned long long) * TIME_WORDS * C;
        if (!st->timing && f2_dev_alloc(st, (void**)&st->timing, bytes, cs, true) != cudaSuccess) return F2_ERR_OOM;
        zl.add(st->timing, bytes);
    }
    PlanZero zero{};
    if (st->num_ctx <= PLAN_SMALL_MAX) {  // by the call's first plan
        zero = {st->counters + CNT_WORK, st->shard_done, st->full_ctr, st->full_cnt, st->full_first,
                hand_min > 0 ? st->hand : nullptr};
    } else {
        if (hand_min > 0) {  // hand-off: the two list counts and the chunk counters
            zl.add(st->hand, sizeof(int) * 2);
            zl.add(st->hand + 2 + 4 * C, sizeof(int) * 2 * C);
        }
        if (dedup) {  // the work totals and the shard items of the duplicate pass
            zl.add(st->counters + CNT_WORK, (CNT_WORDS - CNT_WORK) * sizeof(int));
            zl.add(st->shard_done, sizeof(int32_t) * C);
        }
        zl.add(st->full_ctr, sizeof(int) * 2 * C);        // full-rank chunks claimed and done
        zl.add(st->full_ctr + 4 * C, sizeof(int));        // late count
        zl.add(st->full_cnt, sizeof(unsigned long long) * C);
        zl.add(st->full_first, sizeof(unsigned long long) * C, 0xff);
        zl.add(st->plan_hist, sizeof(int) * 2 * PLAN_HIST_WORDS);  // the histograms of the two plans
    }
    e = f2_fill(zl, cs);
    if (e != cudaSuccess) return f2_cuda_status(e);
    const StoreDev sd = st->dev();
    {
        const int rc = f2_ensure_aux(st);
        if (rc != F2_OK) return rc;
    }
    Fork fk{cs, st->aux, st->ev_fork, st->ev_join};
    // Rows from which a context gets a whole CTA: unless set explicitly, it
    // scales with the batch -- in a short call a warp-owned context of a few
    // thousand rows, dependent round after round, would outlast everything
    // else, while in a long one warps keep the SMs fuller
    // else, and in a store of at most ALL_CTA_PER_SM contexts per SM, every
    // context gets one: none waits for a CTA, and a CTA takes eight warps'
    // rows per dependent round
    int64_t heavy = st->heavy_rows;
    const bool all_cta = !st->heavy_rows_set && st->num_ctx <= (int64_t)ALL_CTA_PER_SM * st->num_sms;
    if (all_cta) {
        heavy = 1;
    } else if (!st->heavy_rows_set && !dedup) {
        heavy = total_rows / HEAVY_ROWS_BATCH_DIV;
        if (heavy < HEAVY_ROWS_MIN) heavy = HEAVY_ROWS_MIN;
        if (heavy > st->heavy_rows) heavy = st->heavy_rows;
    }
    if (dedup) {
        PlanArgs pa;
        pa.zero = zero;
        zero = PlanZero{};  // (the second plan finds it cleared)
        pa.row_off = row_off;
        pa.x_off = x_off;
        pa.total_rows = total_rows;
        pa.total_xw = total_x_words;
        pa.rep_count = st->rep_count;
        pa.mode = 0;
        pa.warp_region_words = (int)(st->warp_basis_bytes / 4);
        pa.heavy_rows = heavy;
        pa.warp_work = st->warp_work;
        pa.dedup_min = st->handoff_min > 0 ? 0 : (all_cta ? DEDUP_MIN_CTA : DEDUP_MIN_WARP);
        pa.after = 0;
        pa.scale = 0;
        pa.num_sms = st->num_sms;
        // a shard share: the call's rows x (feature words + 4) over four per SM
        pa.max_shards = st->dd_shards;
        pa.shard_cap = f2_shard_queue_extra(st->num_sms);
        pa.shard_work = (st->num_ctx < SHARD_CTX_LIMIT && st->dd_shards > 1)
                            ? (total_x_words + 4 * total_rows) / (4 * (long long)st->num_sms) + 1
                            : 0;
        pa.queue = st->queue;
        pa.keybuf = st->keybuf;
        pa.hist = st->plan_hist;
        pa.hist_zeroed = 1;
        pa.counters = st->counters;
        int rc = launch_plan(sd, pa, st->num_sms, cs);
        if (rc != F2_OK) return rc;
        DedupArgs da;
        da.row_off = row_off;
        da.x_off = x_off;
        da.x = x;
        da.y = reinterpret_cast<const uint4*>(y);
        da.rep_list = st->rep_list;
        da.rep_dup = st->rep_dup;
        da.rep_count = st->rep_count;
        da.queue = st->queue;
        da.counters = st->counters;
        da.timing = st->timing_on ? st->timing : nullptr;
        da.shard_reps = st->shard_reps;
        da.shard_done = st->shard_done;
        // the two instances hold disjoint contexts: side by side when both run
        const bool wide_rows = st->max_xw > DD_XW;  // some context has feature rows of 10..16 words
        e = cudaFuncSetAttribute(dedup_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, DD_SMEM);
        if (e != cudaSuccess) return f2_cuda_status(e);
        cudaStream_t ks = fk.next(wide_rows ? 2 : 1);
        if (fk.e != cudaSuccess) return f2_cuda_status(fk.e);
        f2_launch(dedup_kernel<false>, DD_CTAS_PER_SM * st->num_sms, DD_THREADS, DD_SMEM, ks,
                  sd.num_ctx <= EARLY_MAX_CTX, sd, da);
        e = cudaGetLastError();
        if (e != cudaSuccess) return f2_cuda_status(e);
        if (wide_rows) {
            e = cudaFuncSetAttribute(dedup_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, DD_SMEM);
            if (e != cudaSuccess) return f2_cuda_status(e);
            f2_launch(dedup_kernel<true>, DD_CTAS_PER_SM * st->num_sms, DD_THREADS, DD_SMEM, fk.next(1),
                      sd.num_ctx <= EARLY_MAX_CTX, sd, da);
            e = cudaGetLastError();
            if (e != cudaSuccess) return f2_cuda_status(e);
        }
        e = fk.join();
        if (e != cudaSuccess) return f2_cuda_status(e);
    }
    LearnArgs la;
    la.row_off = row_off;
    la.x_off = x_off;
    la.x = x;
    la.y = reinterpret_cast<const uint4*>(y);
    la.rep_list = dedup ? st->rep_list : nullptr;
    la.rep_dup = dedup ? st->rep_dup : nullptr;
    la.rep_count = dedup ? st->rep_count : nullptr;
    la.queue = st->queue;
    la.counters = st->counters;
    la.timing = st->timing_on ? st->timing : nullptr;
    la.warp_region_words = (int)(st->warp_basis_bytes / 4);
    la.tables = st->elim_tables;
    la.small_region_words = (int)(st->small_basis_bytes / 4);
    la.cta_region_words = 0;  // set per launch
    la.handoff_min = hand_min;
    la.handoff_tables = !auto_hand;
    la.snap_count = st->hand;
    la.snap_list = st->hand + 2;
    la.snap_start = st->hand + 2 + C;
    la.resume_from = nullptr;
    la.resume_list = nullptr;
    la.resume_count = nullptr;
    const int scale = dedup && !all_cta && !st->heavy_rows_set && !st->warp_work_set;
    CheckArgs ca;
    ca.row_off = row_off;
    ca.x_off = x_off;
    ca.x = x;
    ca.y = reinterpret_cast<const uint4*>(y);
    ca.rep_list = la.rep_list;
    ca.rep_dup = la.rep_dup;
    ca.rep_count = la.rep_count;
    ca.snap_count = la.snap_count;
    ca.snap_list = la.snap_list;
    ca.snap_start = la.snap_start;
    ca.resume_count = st->hand + 1;
    ca.resume_list = st->hand + 2 + 2 * C;
    ca.resume_from = st->hand + 2 + 3 * C;
    ca.ctr = st->hand + 2 + 4 * C;
    ca.rec = st->check_rec;
    return launch_elimination(sd, la, row_off, x_off, total_rows, total_x_words, dedup ? st->rep_count : nullptr,
                              heavy, st->warp_work, st->queue, st->keybuf, st->plan_hist + PLAN_HIST_WORDS,
                              st->num_sms, wv, st->full_ctr, st->full_cnt, st->full_first, cs, &fk, scale, true,
                              all_cta ? INT64_MAX : st->long_call_rows, &ca, zero, st->fail_wait);
}

extern "C" int f2_learn_timing(const f2_store* st, uint64_t* out_host, f2_stream_t stream)
{
    if (!st || !out_host) return F2_ERR_INVALID_ARG;
    if (!st->timing) return F2_ERR_INVALID_ARG;  // no learn call since F2_OPT_TIMING was set
    cudaStream_t cs = (cudaStream_t)stream;
    cudaError_t e = cudaMemcpyAsync(out_host, st->timing, sizeof(uint64_t) * TIME_WORDS * (size_t)st->num_ctx,
                                    cudaMemcpyDeviceToHost, cs);
    if (e == cudaSuccess) e = cudaStreamSynchronize(cs);
    return f2_cuda_status(e);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of f2_learn_batched (no counterpart in the paper;
// see f2_learn_batched_noalloc in f2gpu.h).  The scheduling scratch that a
// store would own lives in one file-scope device array of fixed capacity.

#include <mutex>

namespace {

struct NoallocScratch {
    CtxDesc desc[F2_NOALLOC_MAX_CTX];
    int32_t n_bits[F2_NOALLOC_MAX_CTX];
    int32_t queue[F2_NOALLOC_MAX_CTX];
    int32_t keybuf[F2_NOALLOC_MAX_CTX];
    int counters[CNT_WORDS];
    int plan_hist[PLAN_KEYS];
    int full_ctr[5 * F2_NOALLOC_MAX_CTX + 1];
    unsigned long long full_cnt[F2_NOALLOC_MAX_CTX];
    unsigned long long full_first[F2_NOALLOC_MAX_CTX];
};

// Device storage for the scratch; in host code this name is only a symbol
// handle, its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoallocScratch)];

constexpr int NOALLOC_MAX_DEVICES = 64;
constexpr int NOALLOC_HEAVY_ROWS = DEFAULT_HEAVY_ROWS;
constexpr int NOALLOC_WARP_REGION_WORDS = DEFAULT_WARP_REGION_BYTES / 4;

struct NoallocDevice {
    NoallocScratch* scratch;
    int num_sms;
    bool ready;
};
NoallocDevice g_noalloc_dev[NOALLOC_MAX_DEVICES];
std::mutex g_noalloc_mu;

// Context descriptors and canonical offsets (exclusive prefix sums of d,
// d*wd and wd) for up to F2_NOALLOC_MAX_CTX contexts, one block.
__global__ void __launch_bounds__(1024) noalloc_desc_kernel(const int32_t* n_bits, int C, uint32_t raw,
                                                            CtxDesc* desc)
{
    pdl_wait();
    constexpr int PER = (F2_NOALLOC_MAX_CTX + 1023) / 1024;
    __shared__ long long wsum[3][32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    long long a = 0, b = 0, c = 0;
    for (int i = 0; i < PER; ++i) {
        const int k = t * PER + i;
        if (k < C) {
            const int n = n_bits[k];
            const int d = raw ? n : n + 1;
            const int wd = (d + 31) / 32;
            a += d;
            b += (long long)d * wd;
            c += wd;
        }
    }
    long long ia = a, ib = b, ic = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long va = __shfl_up_sync(FULL, ia, o), vb = __shfl_up_sync(FULL, ib, o),
                        vc = __shfl_up_sync(FULL, ic, o);
        if (lane >= o) {
            ia += va;
            ib += vb;
            ic += vc;
        }
    }
    if (lane == 31) {
        wsum[0][warp] = ia;
        wsum[1][warp] = ib;
        wsum[2][warp] = ic;
    }
    __syncthreads();
    if (warp == 0) {
        long long sa = wsum[0][lane], sb = wsum[1][lane], sc = wsum[2][lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long va = __shfl_up_sync(FULL, sa, o), vb = __shfl_up_sync(FULL, sb, o),
                            vc = __shfl_up_sync(FULL, sc, o);
            if (lane >= o) {
                sa += va;
                sb += vb;
                sc += vc;
            }
        }
        wsum[0][lane] = sa - wsum[0][lane];
        wsum[1][lane] = sb - wsum[1][lane];
        wsum[2][lane] = sc - wsum[2][lane];
    }
    __syncthreads();
    long long ea = wsum[0][warp] + ia - a, eb = wsum[1][warp] + ib - b, ec = wsum[2][warp] + ic - c;
    for (int i = 0; i < PER; ++i) {
        const int k = t * PER + i;
        if (k < C) {
            CtxDesc cd;
            cd.n = n_bits[k];
            cd.d = raw ? cd.n : cd.n + 1;
            cd.wd = (cd.d + 31) / 32;
            cd.xw = (cd.n + 31) / 32;
            cd.slot_off = ea;
            cd.xw_off = eb;
            cd.pw_off = ec;
            cd.pad = 0;
            desc[k] = cd;
            ea += cd.d;
            eb += (long long)cd.d * cd.wd;
            ec += cd.wd;
        }
    }
}

// Host copy of the caller's widths: the device copy is made from here, so the
// caller's array is free again when the call returns (a copy from pageable
// memory is staged before cudaMemcpyAsync returns).  Guarded by g_noalloc_mu.
int32_t g_noalloc_nbits[F2_NOALLOC_MAX_CTX];

// Every kernel the allocation-free path can launch.  Loading a kernel's code
// (on its first launch, under lazy module loading) may allocate device
// memory, so the first call on a device loads all of them.
cudaError_t noalloc_load_kernels()
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, noalloc_desc_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, plan_key_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, plan_scan_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, plan_scatter_kernel);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, plan_small_kernel);
    if (e == cudaSuccess) e = elim_load_small();
    if (e == cudaSuccess) e = elim_load_narrow();
    if (e == cudaSuccess) e = elim_load_wide();
    if (e == cudaSuccess) e = verify_load_tc();
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, verify_full_kernel);
    return e;
}

// Once per device (with that device current): resolve the scratch address
// and load the kernels.
int noalloc_setup(NoallocDevice** out)
{
    int device = -1;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return f2_cuda_status(e);
    if (device < 0 || device >= NOALLOC_MAX_DEVICES) return F2_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoallocDevice& d = g_noalloc_dev[device];
    if (!d.ready) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || p == nullptr) return e != cudaSuccess ? f2_cuda_status(e) : F2_ERR_CUDA;
        int sms = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        if (e == cudaSuccess) e = noalloc_load_kernels();
        if (e != cudaSuccess) return f2_cuda_status(e);
        d.scratch = static_cast<NoallocScratch*>(p);
        d.num_sms = sms;
        d.ready = true;
    }
    *out = &d;
    return F2_OK;
}

}  // namespace

extern "C" int f2_learn_batched_noalloc(int32_t num_ctx, const int32_t* n_bits_host, uint32_t flags,
                                        int32_t* rank_dev, uint32_t* pivot_mask_dev, uint32_t* basis_x_dev,
                                        uint32_t* basis_z_dev, uint8_t* contra_dev, int64_t* first_contra_dev,
                                        uint64_t* n_contra_dev, int64_t* rows_seen_dev, int32_t* status_dev,
                                        const int64_t* row_off_dev, const uint32_t* x_dev, const int64_t* x_off_dev,
                                        const uint32_t* y_dev, int64_t total_rows, int64_t total_x_words,
                                        f2_stream_t stream)
{
    F2_NVTX_RANGE("f2_learn_batched_noalloc");
    if (num_ctx < 0 || num_ctx > F2_NOALLOC_MAX_CTX || (flags & ~F2_FLAG_RAW_FEATURES) || total_rows < 0 ||
        total_x_words < 0 || !status_dev)
        return F2_ERR_INVALID_ARG;
    if (num_ctx == 0)  // nothing to learn: only the status word is written
        return f2_cuda_status(cudaMemsetAsync(status_dev, 0, sizeof(int32_t), (cudaStream_t)stream));
    if (!n_bits_host || !rank_dev || !pivot_mask_dev || !basis_x_dev || !basis_z_dev || !contra_dev ||
        !first_contra_dev || !n_contra_dev || !rows_seen_dev || !row_off_dev || !x_off_dev ||
        (!x_dev && total_x_words) || (!y_dev && total_rows))
        return F2_ERR_INVALID_ARG;
    if (!is_aligned(row_off_dev, 8) || !is_aligned(x_off_dev, 8) || !is_aligned(x_dev, 4) || !is_aligned(y_dev, 16) ||
        !is_aligned(basis_z_dev, 16) || !is_aligned(first_contra_dev, 8) || !is_aligned(n_contra_dev, 8) ||
        !is_aligned(rows_seen_dev, 8) || !is_aligned(rank_dev, 4) || !is_aligned(pivot_mask_dev, 4) ||
        !is_aligned(basis_x_dev, 4) || !is_aligned(status_dev, 4))
        return F2_ERR_ALIGN;
    const bool raw = (flags & F2_FLAG_RAW_FEATURES) != 0;
    for (int32_t c = 0; c < num_ctx; ++c)
        if (n_bits_host[c] < 1 || n_bits_host[c] > MAX_N) return F2_ERR_NBITS;
    NoallocDevice* nd = nullptr;
    int rc = noalloc_setup(&nd);
    if (rc != F2_OK) return rc;
    NoallocScratch* sc = nd->scratch;
    cudaStream_t cs = (cudaStream_t)stream;

    cudaError_t e = cudaMemsetAsync(status_dev, 0, sizeof(int32_t), cs);
    if (e == cudaSuccess) {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        memcpy(g_noalloc_nbits, n_bits_host, sizeof(int32_t) * (size_t)num_ctx);
        e = cudaMemcpyAsync(sc->n_bits, g_noalloc_nbits, sizeof(int32_t) * (size_t)num_ctx, cudaMemcpyHostToDevice,
                            cs);
    }
    if (e != cudaSuccess) return f2_cuda_status(e);
    f2_launch(noalloc_desc_kernel, 1, 1024, 0, cs, num_ctx <= EARLY_MAX_CTX, sc->n_bits, num_ctx, raw ? 1u : 0u,
              sc->desc);

    StoreDev sd;
    sd.desc = sc->desc;
    sd.rank = rank_dev;
    sd.contra = contra_dev;
    sd.first_contra = reinterpret_cast<long long*>(first_contra_dev);
    sd.n_contra = reinterpret_cast<unsigned long long*>(n_contra_dev);
    sd.rows_seen = reinterpret_cast<long long*>(rows_seen_dev);
    sd.pivot = pivot_mask_dev;
    sd.bx = basis_x_dev;
    sd.bz = reinterpret_cast<uint4*>(basis_z_dev);
    sd.status = status_dev;
    sd.num_ctx = num_ctx;
    sd.raw = raw ? 1u : 0u;
    LearnArgs la;
    la.row_off = row_off_dev;
    la.x_off = x_off_dev;
    la.x = x_dev;
    la.y = reinterpret_cast<const uint4*>(y_dev);
    la.rep_list = nullptr;  // every row is its own representative: no per-row scratch
    la.rep_dup = nullptr;
    la.rep_count = nullptr;
    la.queue = sc->queue;
    la.counters = sc->counters;
    la.timing = nullptr;
    la.tables = 1;
    la.small_region_words = DEFAULT_SMALL_REGION_BYTES / 4;
    la.cta_region_words = 0;
    la.handoff_min = 0;
    la.handoff_tables = 0;
    la.snap_count = nullptr;
    la.snap_list = nullptr;
    la.snap_start = nullptr;
    la.resume_from = nullptr;
    la.resume_list = nullptr;
    la.resume_count = nullptr;
    la.warp_region_words = NOALLOC_WARP_REGION_WORDS;
    const Widths wv = width_summary(n_bits_host, num_ctx, raw);
    return launch_elimination(sd, la, row_off_dev, x_off_dev, total_rows, total_x_words, nullptr, NOALLOC_HEAVY_ROWS,
                              DEFAULT_WARP_WORK, sc->queue, sc->keybuf, sc->plan_hist, nd->num_sms, wv, sc->full_ctr,
                              sc->full_cnt, sc->full_first, cs);
}
