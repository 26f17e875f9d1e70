// Elimination of the representatives (pass 2 of a learn call): device code
// shared by the translation units of the width classes (elim_small.cu,
// elim_narrow.cu, elim_wide.cu) and by the check of handed-off contexts
// (learn.cu).  The algorithm is described at the top of learn.cu.
#pragma once

#include <limits.h>

#include <type_traits>

#include "f2_internal.cuh"

namespace f2 {

struct LearnArgs {
    const int64_t* row_off;
    const int64_t* x_off;
    const uint32_t* x;
    const uint4* y;
    const int32_t* rep_list;   // representatives (row indices, per-context at row_off[c]); NULL = every row
    const int32_t* rep_dup;    // duplicates of each representative (NULL = none)
    const int32_t* rep_count;  // representatives per context (NULL = all rows)
    const int32_t* queue;
    int* counters;
    int warp_region_words;
    // contexts that reach full rank with rows left (not deduplicated): listed
    // here, the rest of their rows checked by verify_full_kernel
    int* late_count;
    int32_t* late_list;
    int32_t* late_start;
    unsigned long long* timing;  // per-context timestamps (F2_OPT_TIMING), NULL = off
    int tables;                  // reduce against a lookup table of the snapshot where it pays
    int small_region_words;      // shared memory of a warp-owned context of the small-width kernel
    int cta_region_words;        // shared memory of a CTA-owned context (the launch's dynamic size)
    // a CTA-owned context whose rank has not grown for HANDOFF_QUIET rounds,
    // with at least handoff_min representatives left, stops and is listed
    // here: check_snap_kernel checks the rest against its basis in parallel
    int handoff_min;             // 0 = never
    int handoff_tables;          // also contexts that run against a lookup table
    int* snap_count;
    int32_t* snap_list;
    int32_t* snap_start;         // its first representative left
    // a launch that takes up contexts the check sent back: each listed
    // context's first representative, the list and its length (NULL: a
    // normal launch)
    const int32_t* resume_from;
    const int32_t* resume_list;
    const int* resume_count;
    // rows of each context of more than 17 words that elim_open_kernel has
    // taken already
    int32_t* open_from;
};

// The elimination kernels' launches, one function per translation unit (each
// with the widest dynamic shared memory its contexts need), and the loading of
// their code ahead of a first launch.
cudaError_t elim_launch_small(const StoreDev& sd, LearnArgs la, int max_words, int num_sms, cudaStream_t cs);
cudaError_t elim_launch_narrow(const StoreDev& sd, LearnArgs la, int max_words, int warps, int num_sms,
                               cudaStream_t cs);
// (for rows of more than 17 words: elim_open_kernel, then the streaming kernel)
cudaError_t elim_launch_wide(const StoreDev& sd, LearnArgs la, int max_d, bool medium, int num_sms, cudaStream_t cs);
cudaError_t elim_load_small();
cudaError_t elim_load_narrow();
cudaError_t elim_load_wide();

// Shared-memory control area of a CTA-owned context (32-bit words).
constexpr int CTL_NPR = 0;     // pivots a warp has just added, 48 words
constexpr int CTL_CAND = 48;   // per-warp candidate ballots, two buffers of 16 words
constexpr int CTL_CNT = 80;    // contradiction count (uint64, 8-byte aligned)
constexpr int CTL_FIRST = 82;  // first contradiction index (int64)
constexpr int CTL_WORDS = 84;  // size of the control area (16-byte multiple)

constexpr int FULL_CHUNK = 2048;   // rows of a full-rank context claimed at a time
constexpr int FULL_LATE_MIN = 64;  // rows left for a context that reaches full rank mid-call to be checked that way

__host__ __device__ __forceinline__ int elim_words(int d, int wd) { return CTL_WORDS + d * row_stride(wd); }

// Per-context timestamps of a learn call (diagnostics, F2_OPT_TIMING):
// TIME_WORDS words per context -- %globaltimer at the start and end of its
// duplicate pass and of its elimination, then the SM ids that ran them.
constexpr int TIME_WORDS = 6;
__device__ __forceinline__ unsigned smid()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void time_mark(unsigned long long* timing, int c, int slot)
{
    if (timing) {
        timing[(size_t)TIME_WORDS * c + slot] = global_ns();
        timing[(size_t)TIME_WORDS * c + 4 + (slot >> 1)] = smid();
    }
}

__device__ __forceinline__ bool nonzero4(const uint4& v) { return (v.x | v.y | v.z | v.w) != 0u; }

__device__ __forceinline__ void xor4(uint4& a, const uint4& b)
{
    a.x ^= b.x;
    a.y ^= b.y;
    a.z ^= b.z;
    a.w ^= b.w;
}

// Bit v set iff feature word v (< wd) still has a non-pivot column.  Words
// made only of pivot columns are never XOR-ed: the residual is zero there.
template <int WD>
__device__ __forceinline__ uint64_t mixed_words(const uint32_t (&P)[WD], int d, int wd)
{
    uint64_t m = 0;
#pragma unroll
    for (int v = 0; v < WD; ++v) {
        if (v < wd) {
            const uint32_t valid = (v < wd - 1 || (d & 31) == 0) ? 0xffffffffu : ((1u << (d & 31)) - 1u);
            if (P[v] != valid) m |= 1ull << v;
        }
    }
    return m;
}

// Feature words exactly as supplied (bits >= n cleared), and the word.
template <int WD>
__device__ __forceinline__ void load_raw(const uint32_t* xrow, const uint4* yrow,
                                         bool valid, int n, int xw, uint32_t (&xin)[WD], uint4& y)
{
#pragma unroll
    for (int v = 0; v < WD; ++v) {
        uint32_t t = 0;
        if (valid && v < xw) t = ld(xrow + v);
        if (v == xw - 1 && (n & 31)) t &= (1u << (n & 31)) - 1u;
        xin[v] = t;
    }
    y = valid ? ld(yrow) : make_uint4(0, 0, 0, 0);
}

// q = [1 || x] (index 0 = constant) or x itself for raw feature rows.
template <int WD>
__device__ __forceinline__ void make_q(const uint32_t (&xin)[WD], bool valid, uint32_t raw, uint32_t (&q)[WD])
{
    if (raw) {
#pragma unroll
        for (int v = 0; v < WD; ++v) q[v] = xin[v];
    } else {
        q[0] = (xin[0] << 1) | (valid ? 1u : 0u);
#pragma unroll
        for (int v = 1; v < WD; ++v) q[v] = (xin[v] << 1) | (xin[v - 1] >> 31);
    }
}

template <bool CTA>
__device__ __forceinline__ void group_sync()
{
    if (CTA) __syncthreads();
    else __syncwarp();
}

// ------------------------------------------------------------------ pass 2
//
// One group (a warp, or a whole CTA) streams the representatives of a context
// through a basis in shared memory: slot k holds [z_k (4 words) | r_k], padded
// to row_stride(WD) words.  Rows live in registers, one a lane (the opening: four).

// The rows that a group streams, and one of them as loaded.
struct RowStream {
    const int32_t* reps;  // row of each representative; NULL: every row
    const int32_t* dups;  // its later duplicates; NULL: none
    const uint32_t* xc;
    const uint4* yc;
    int R;                // representatives
    int n, xw;
    uint32_t raw;
    long long seen;       // rows of the context before this call
};
template <int WD>
struct Row {
    uint32_t x[WD];
    uint4 y;
    int i;
    uint32_t weight;
    bool valid;
};

template <int WD>
__device__ __forceinline__ void fetch_row(const RowStream& rs, int base, int j, Row<WD>& r)
{
    const int k = (int)((uint32_t)base + (uint32_t)j);
    r.valid = item_in(base, j, rs.R);
    r.i = r.valid ? (rs.reps ? ld(rs.reps + k) : k) : 0;
    r.weight = 1u + ((r.valid && rs.dups) ? (uint32_t)ld(rs.dups + k) : 0u);
    load_raw<WD>(rs.xc + (int64_t)r.i * rs.xw, rs.yc + r.i, r.valid, rs.n, rs.xw, r.x, r.y);
}

// Step (1): XOR into each lane's row the stored rows of the pivots M that the
// row has set.  A stored row never changes another pivot bit of M, so the bit
// that selects row b is the row's own bit b however the rows are ordered: the
// warp walks the union of its rows' pivots, two per step with their loads issued
// together, every lane under its own bits.  Words that only pivots fill (not in
// `mixed`) are never XOR-ed: the caller clears the pivot columns.
template <int WD>
__device__ __forceinline__ void reduce_rows(uint32_t (&xr)[WD], uint4& yr, const uint32_t* __restrict__ S,
                                            const uint32_t (&M)[WD], uint64_t mixed)
{
    constexpr int RS = row_stride(WD);
#pragma unroll
    for (int w = 0; w < WD; ++w) {
        const uint32_t sel = xr[w];
        uint32_t uw = __reduce_or_sync(FULL, sel & M[w]);
        const bool xwork = (mixed & ((2ull << w) - 1ull)) != 0;
        while (uw) {
            const int b0 = __ffs(uw) - 1;
            uw &= uw - 1;
            const bool two = uw != 0u;
            const int b1 = two ? __ffs(uw) - 1 : b0;
            uw &= uw - 1;
            const uint32_t* row0 = S + (32 * w + b0) * RS;
            const uint32_t* row1 = S + (32 * w + b1) * RS;
            const uint4 z0 = *reinterpret_cast<const uint4*>(row0);
            const uint4 z1 = *reinterpret_cast<const uint4*>(row1);
            const uint32_t m0 = 0u - ((sel >> b0) & 1u);
            const uint32_t m1 = two ? 0u - ((sel >> b1) & 1u) : 0u;
            yr.x ^= (z0.x & m0) ^ (z1.x & m1);
            yr.y ^= (z0.y & m0) ^ (z1.y & m1);
            yr.z ^= (z0.z & m0) ^ (z1.z & m1);
            yr.w ^= (z0.w & m0) ^ (z1.w & m1);
            if (xwork) {
#pragma unroll
                for (int v4 = 0; v4 <= w / 4; ++v4) {
                    const uint4 xa = *reinterpret_cast<const uint4*>(row0 + 4 + 4 * v4);
                    const uint4 xb = *reinterpret_cast<const uint4*>(row1 + 4 + 4 * v4);
                    const uint32_t ea[4] = {xa.x, xa.y, xa.z, xa.w};
                    const uint32_t eb[4] = {xb.x, xb.y, xb.z, xb.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int v = 4 * v4 + j;
                        if (v <= w && v < WD)
                            if ((mixed >> v) & 1ull) xr[v] ^= (ea[j] & m0) ^ (eb[j] & m1);
                    }
                }
            }
        }
    }
}

// The address of the basis slot of coordinate k: coordinate k itself, or
// (rows held by compressed residual) the k-th free coordinate of the table.
template <int RS>
__device__ __forceinline__ uint32_t* slot_row(uint32_t* S, const uint16_t* FL, int k)
{
    return S + (FL ? (int)FL[k] : k) * RS;
}

template <int WD>
__device__ __forceinline__ bool nonzero_row(const uint32_t (&x)[WD])
{
    uint32_t any = 0;
#pragma unroll
    for (int v = 0; v < WD; ++v) any |= x[v];
    return any != 0u;
}

// One insertion of step (4): the row b | z (its words above W are zero) takes
// the pivot of its highest set bit, and every row of the warp with that bit
// set is XOR-ed with it, so the warp's rows stay reduced among themselves.
// Returns the pivot, or -1 if the row is zero.  `own`: this lane's slot 0 holds
// the row; slots outside `live` hold none.
template <int W, int WD, int K>
__device__ __forceinline__ int pivot_step(uint32_t (&xr)[K][WD], uint4 (&yr)[K], const uint32_t (&b)[WD],
                                          const uint4& z, bool own, uint32_t live, uint32_t (&NP)[WD])
{
    if (b[W]) {  // uniform: b is a broadcast
        const int kb = 31 - __clz(b[W]);
        const uint32_t m = 1u << kb;
        NP[W] |= m;
#pragma unroll
        for (int t = 0; t < K; ++t) {
            if (K > 1 && !((live >> t) & 1u)) continue;
            if ((xr[t][W] & m) != 0u && !(t == 0 && own)) {
#pragma unroll
                for (int v = 0; v <= W; ++v) xr[t][v] ^= b[v];
                xor4(yr[t], z);
            }
        }
        return 32 * W + kb;
    }
    if constexpr (W > 0) return pivot_step<W - 1, WD, K>(xr, yr, b, z, own, live, NP);
    return -1;
}

// Row k of the basis (z | x) to its slot.
template <int WD>
__device__ __forceinline__ void store_row(uint32_t* __restrict__ slot, const uint32_t (&xr)[WD], const uint4& yr)
{
    uint4* row = reinterpret_cast<uint4*>(slot);
    row[0] = yr;
#pragma unroll
    for (int v4 = 0; 4 * v4 < WD; ++v4) {
        uint32_t e[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) e[j] = 4 * v4 + j < WD ? xr[4 * v4 + j < WD ? 4 * v4 + j : 0] : 0u;
        row[1 + v4] = make_uint4(e[0], e[1], e[2], e[3]);
    }
}

template <int WD>
__device__ __forceinline__ void broadcast_row(const uint32_t (&xr)[WD], const uint4& yr, int i, uint32_t (&b)[WD],
                                              uint4& z)
{
#pragma unroll
    for (int v = 0; v < WD; ++v) b[v] = __shfl_sync(FULL, xr[v], i);
    z.x = __shfl_sync(FULL, yr.x, i);
    z.y = __shfl_sync(FULL, yr.y, i);
    z.z = __shfl_sync(FULL, yr.z, i);
    z.w = __shfl_sync(FULL, yr.w, i);
}

// Step (4) for the candidate rows of one warp, in stream (lane) order: the new
// rows go to their basis slots (row stride RS), NP receives their pivots.  A
// candidate that rows inserted before it reduce to zero is classified (its
// word residual decides).  Returns the number of rows inserted.
template <int WD, int RS>
__device__ int insert_rows(uint32_t (&xr)[1][WD], uint4 (&yr)[1], uint32_t cand, uint32_t* __restrict__ S,
                           const uint16_t* __restrict__ FL, int lane, long long idx, uint32_t weight,
                           long long& first, unsigned long long& cnt, uint32_t (&NP)[WD])
{
    int pk = -1, added = 0;
#pragma unroll
    for (int v = 0; v < WD; ++v) NP[v] = 0;
    const bool mine = (cand >> lane) & 1u;
    while (cand) {
        const int i = __ffs(cand) - 1;
        uint32_t b[WD];
        uint4 z;
        broadcast_row<WD>(xr[0], yr[0], i, b, z);
        const int k = pivot_step<WD - 1, WD, 1>(xr, yr, b, z, lane == i, 1u, NP);
        ++added;
        if (lane == i) pk = k;
        // the rows after it that are not zero yet
        cand &= (0xfffffffeu << i) & __ballot_sync(FULL, nonzero_row<WD>(xr[0]));
    }
    if (mine && pk < 0 && nonzero4(yr[0])) {  // reduced to zero on the way
        cnt += weight;
        first = min(first, idx);
    }
    if (added) {
        if (pk >= 0) store_row<WD>(slot_row<RS>(S, FL, pk), xr[0], yr[0]);
        __syncwarp();
    }
    return added;
}

// Step (5) for one stored row rj: clear the new pivot columns NP.
template <int WD, int RS>
__device__ __forceinline__ void back_clear_row(uint32_t* __restrict__ rj, const uint32_t* __restrict__ S,
                                               const uint16_t* __restrict__ FL, const uint32_t (&NP)[WD])
{
    uint32_t xj[WD];
    uint32_t hits = 0;
#pragma unroll
    for (int v4 = 0; 4 * v4 < WD; ++v4) {
        const uint4 t4 = *reinterpret_cast<const uint4*>(rj + 4 + 4 * v4);
        const uint32_t e[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * v4 + j < WD) xj[4 * v4 + j] = e[j];
    }
#pragma unroll
    for (int v = 0; v < WD; ++v) hits |= xj[v] & NP[v];
    if (!hits) return;
    uint4 zj = *reinterpret_cast<const uint4*>(rj);
#pragma unroll
    for (int v = 0; v < WD; ++v) {
        uint32_t m = xj[v] & NP[v];
        while (m) {
            const int b = __ffs(m) - 1;
            m &= m - 1;
            const uint32_t* rk = slot_row<RS>(const_cast<uint32_t*>(S), FL, 32 * v + b);
            xor4(zj, *reinterpret_cast<const uint4*>(rk));
#pragma unroll
            for (int v4 = 0; 4 * v4 <= v; ++v4) {
                const uint4 t4 = *reinterpret_cast<const uint4*>(rk + 4 + 4 * v4);
                const uint32_t e[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (4 * v4 + j <= v) xj[4 * v4 + j] ^= e[j];
            }
        }
    }
    *reinterpret_cast<uint4*>(rj) = zj;
#pragma unroll
    for (int v = 0; v < WD; ++v) rj[4 + v] = xj[v];
}

// Step (5): clear the new pivot columns NP from the stored rows of the pivots
// P (warp `warp` of `nw` takes every nw-th word of coordinates, a row a lane).
template <int WD, int RS>
__device__ __forceinline__ void back_clear(uint32_t* __restrict__ S, const uint16_t* __restrict__ FL,
                                           const uint32_t (&P)[WD], const uint32_t (&NP)[WD], int lane, int warp,
                                           int nw)
{
#pragma unroll 1
    for (int w0 = warp; w0 < WD; w0 += nw) {
        uint32_t pw = 0;
#pragma unroll
        for (int v = 0; v < WD; ++v)
            if (v == w0) pw = P[v];
        if ((pw >> lane) & 1u) back_clear_row<WD, RS>(slot_row<RS>(S, FL, 32 * w0 + lane), S, FL, NP);
    }
}

// The stored basis moves between global and shared memory by its pivot rows
// only: an empty slot is zero in the store and never read in shared memory
// (every read of S selects a pivot), and a slot that became a pivot stays one.
template <int WD>
__device__ void basis_to_smem(const StoreDev& s, const CtxDesc& cd, uint32_t* S, const uint32_t (&P)[WD], int lane,
                              int warp, int nw)
{
    constexpr int RS = row_stride(WD);
#pragma unroll 1
    for (int w0 = warp; w0 < WD; w0 += nw) {
        uint32_t pw = 0;
#pragma unroll
        for (int v = 0; v < WD; ++v)
            if (v == w0) pw = P[v];
        if (!((pw >> lane) & 1u)) continue;
        const int k = 32 * w0 + lane;
        uint32_t* row = S + k * RS;
        *reinterpret_cast<uint4*>(row) = s.bz[cd.slot_off + k];
        const uint32_t* src = s.bx + cd.xw_off + (int64_t)k * cd.wd;
        for (int v = 0; v < RS - 4; ++v) row[4 + v] = (v < cd.wd) ? src[v] : 0u;
    }
}

template <int WD>
__device__ void basis_from_smem(const StoreDev& s, const CtxDesc& cd, const uint32_t* S, const uint32_t (&P)[WD],
                                int lane, int warp, int nw)
{
    constexpr int RS = row_stride(WD);
#pragma unroll 1
    for (int w0 = warp; w0 < WD; w0 += nw) {
        uint32_t pw = 0;
#pragma unroll
        for (int v = 0; v < WD; ++v)
            if (v == w0) pw = P[v];
        if (!((pw >> lane) & 1u)) continue;
        const int k = 32 * w0 + lane;
        const uint32_t* row = S + k * RS;
        s.bz[cd.slot_off + k] = *reinterpret_cast<const uint4*>(row);
        uint32_t* dst = s.bx + cd.xw_off + (int64_t)k * cd.wd;
        for (int v = 0; v < cd.wd; ++v) dst[v] = row[4 + v];
    }
}

__device__ __forceinline__ void warp_stats(long long& first, unsigned long long& cnt)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        first = min(first, __shfl_xor_sync(FULL, first, o));
        cnt += __shfl_xor_sync(FULL, cnt, o);
    }
}

__device__ __forceinline__ void commit_stats(const StoreDev& s, int c, long long first, unsigned long long cnt)
{
    if (cnt) {
        s.n_contra[c] += cnt;
        s.contra[c] = 1;
        if (s.first_contra[c] < 0) s.first_contra[c] = first;
    }
}

// Set compressed residual bit tt (< 32 * RW).
template <int RW>
__device__ __forceinline__ void set_rbit(uint32_t (&er)[RW], int tt)
{
#pragma unroll
    for (int u = 0; u < RW; ++u)
        if ((tt >> 5) == u) er[u] |= 1u << (tt & 31);
}

constexpr int FL_WORDS = 64;  // free-coordinate list of a table: 128 uint16 entries
constexpr int WARP_TABLE_RW = 1;  // most residual words of a warp-owned context's table

// The lookup table (layout in f2_internal.cuh) of the basis held in shared
// memory: pivot rows S (row stride row_stride(WD)), pivot mask P, with RW residual
// planes (at least the words that the free coordinates need); FL receives the non-pivot coordinates in increasing order (the meaning of the
// compressed residual bits).  All nt threads of the group take part.
template <int WD, int RW, bool CTA>
__device__ __forceinline__ void build_table_smem(const uint32_t* __restrict__ S, const uint32_t (&P)[WD], int d, int wd,
                                                 uint32_t* __restrict__ TB, uint16_t* __restrict__ FL, int t, int nt)
{
    constexpr int RS = row_stride(WD);
    const int np = (d + 3) >> 2;
    uint32_t f[WD];  // non-pivot coordinates of each word
    int pre[WD];     // non-pivot coordinates in the words before
    {
        int acc = 0;
#pragma unroll
        for (int w = 0; w < WD; ++w) {
            const uint32_t valid = (w < wd) ? ((w == wd - 1 && (d & 31)) ? ((1u << (d & 31)) - 1u) : 0xffffffffu) : 0u;
            f[w] = ~P[w] & valid;
            pre[w] = acc;
            acc += __popc(f[w]);
        }
    }
    uint2* const Zl = reinterpret_cast<uint2*>(TB);
    uint2* const Zh = Zl + 16 * np;
    uint32_t* const R = TB + 64 * np;
    for (int j = t; j < 4 * np; j += nt) {
        uint4 z = make_uint4(0, 0, 0, 0);
        uint32_t er[RW];
#pragma unroll
        for (int u = 0; u < RW; ++u) er[u] = 0u;
        if (j < d) {
            const int w = j >> 5, b = j & 31;
            uint32_t fw = 0;
            int pw = 0;
#pragma unroll
            for (int u = 0; u < WD; ++u)
                if (u == w) {
                    fw = f[u];
                    pw = pre[u];
                }
            if ((fw >> b) & 1u) {  // a non-pivot coordinate: its unit vector
                const int tt = pw + __popc(fw & ((1u << b) - 1u));
                set_rbit(er, tt);
                FL[tt] = (uint16_t)j;
            } else {  // a pivot: z_j and r_j on the non-pivot coordinates
                const uint32_t* row = S + j * RS;
                z = *reinterpret_cast<const uint4*>(row);
#pragma unroll
                for (int u = 0; u < WD; ++u) {
                    if (u <= w) {
                        uint32_t bits = row[4 + u] & f[u];
                        while (bits) {
                            const int bb = __ffs(bits) - 1;
                            bits &= bits - 1u;
                            set_rbit(er, pre[u] + __popc(f[u] & ((1u << bb) - 1u)));
                        }
                    }
                }
            }
        }
        const int e = 16 * (j >> 2) + (1 << (j & 3));
        Zl[e] = make_uint2(z.x, z.y);
        Zh[e] = make_uint2(z.z, z.w);
#pragma unroll
        for (int u = 0; u < RW; ++u) R[u * 16 * np + e] = er[u];
        if ((j & 3) == 0) {
            const int e0 = 16 * (j >> 2);
            Zl[e0] = make_uint2(0, 0);
            Zh[e0] = make_uint2(0, 0);
#pragma unroll
            for (int u = 0; u < RW; ++u) R[u * 16 * np + e0] = 0u;
        }
    }
    group_sync<CTA>();
    // entries of two or more coordinates: XOR of their single entries
    for (int k = t; k < 16 * np; k += nt) {
        const int v = k & 15;
        if (__popc(v) < 2) continue;
        const int eb = k & ~15;
        uint2 lo = make_uint2(0, 0), hi = make_uint2(0, 0);
        uint32_t rr[RW];
#pragma unroll
        for (int u = 0; u < RW; ++u) rr[u] = 0u;
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) {
            if ((v >> bb) & 1) {
                const int es = eb + (1 << bb);
                const uint2 l = Zl[es], h = Zh[es];
                lo.x ^= l.x;
                lo.y ^= l.y;
                hi.x ^= h.x;
                hi.y ^= h.y;
#pragma unroll
                for (int u = 0; u < RW; ++u) rr[u] ^= R[u * 16 * np + es];
            }
        }
        Zl[k] = lo;
        Zh[k] = hi;
#pragma unroll
        for (int u = 0; u < RW; ++u) R[u * 16 * np + k] = rr[u];
    }
    group_sync<CTA>();
}

// The full residual (feature words, zero at the pivots) from its compressed
// form: bit t is the non-pivot coordinate FL[t].
template <int WD, int RW>
__device__ __forceinline__ void decompress_residual(const uint32_t (&cr)[RW], const uint16_t* __restrict__ FL,
                                                    uint32_t (&xr)[WD])
{
#pragma unroll
    for (int v = 0; v < WD; ++v) xr[v] = 0u;
#pragma unroll
    for (int u = 0; u < RW; ++u) {
        uint32_t bits = cr[u];
        while (bits) {
            const int bb = __ffs(bits) - 1;
            bits &= bits - 1u;
            const int coord = FL[32 * u + bb];
#pragma unroll
            for (int v = 0; v < WD; ++v)
                if ((coord >> 5) == v) xr[v] |= 1u << (coord & 31);
        }
    }
}

// Hand-off of saturated contexts (see LearnArgs): the quiet rounds before
// it, the widest basis the check can hold (shared memory words, a slot per
// coordinate) and its chunks of representatives; the row widths of the two
// instances of the wide kernel (the 10..17-word one takes part).
constexpr int HANDOFF_QUIET = 2;
constexpr int CHECK_BASIS_WORDS = 14336;  // 56 KB
constexpr int CHECK_CHUNK = 1024;
constexpr int HANDOFF_CALL_FACTOR = 16;  // calls of fewer rows than this many hand-off minimums hand off none
constexpr int WIDE_WD = 33;    // widest row (d <= 1056)
constexpr int WIDE_M_WD = 17;  // rows of 10..17 words (d <= 544): half the registers, two CTAs per SM

// The fewest representatives left for a context to hand off.  The
// check needs the representatives' list, which a context that skipped the
// duplicate pass of this call has not.
__device__ __forceinline__ int handoff_least(const LearnArgs& a, bool deduped)
{
    if (a.handoff_min <= 0 || a.resume_from || deduped != (a.rep_count != nullptr)) return INT_MAX;
    return a.handoff_min;
}

// What a group knows of its context while it streams the rows.
template <int WD>
struct ElimState {
    uint32_t P[WD];   // pivots of the basis in shared memory
    int rank;
    int base;         // next representative
    int quiet;        // rounds in a row that inserted nothing (CTA)
    int hand_min;     // representatives left from which a saturated context hands off (CTA)
    int parity;       // ballot buffer of the next barrier (CTA)
    long long first;  // this lane's contradictions
    unsigned long long cnt;
};

// The candidates of every warp of a CTA: publishes this warp's, returns the
// warps that have some.  Two ballot buffers alternate: each use ends with the
// buffer being read after the barrier, and the next use writes the other.
__device__ __forceinline__ uint32_t publish_candidates(uint32_t cand, uint32_t* wc, int& parity, int warp, int lane,
                                                       int G)
{
    uint32_t* const wcp = wc + 16 * parity;
    parity ^= 1;
    if (lane == 0) wcp[warp] = cand;
    __syncthreads();
    uint32_t wmask = 0;
    for (int ww = 0; ww < G; ++ww)
        if (wcp[ww]) wmask |= 1u << ww;
    return wmask;
}

// Rounds against a lookup table of the basis (f2_internal.cuh), from st.base
// on.  The table is not rebuilt when rows are inserted: it stays the linear
// map of the basis it was built from, a row's residual after it lives on that
// basis's non-pivot coordinates, compressed to RW words, and the rows inserted
// since (N, pivots NP, kept reduced among themselves and held compressed in
// the slots of their coordinates) are walked after it.  Returns when the rows
// are done, when the walks over N have cost what a new table costs, or (CTA)
// when the context hands off (returns its representative, else -1); N is then
// merged into the basis: decompressed, and its columns cleared from the older
// rows (step (5)).
template <int WD, int RW, bool CTA>
__device__ int table_rounds(const LearnArgs& a, const RowStream& rs, ElimState<WD>& st, uint32_t* __restrict__ S,
                            const uint32_t* __restrict__ TB, const uint16_t* __restrict__ FL, int d, uint32_t* wc,
                            uint32_t* NPR)
{
    constexpr int RS = row_stride(WD);
    const int lane = threadIdx.x & 31;
    const int warp = CTA ? (int)(threadIdx.x >> 5) : 0;
    const int G = CTA ? (int)(blockDim.x >> 5) : 1;
    const int nt = 32 * G;
    const int np = (d + 3) >> 2;
    uint32_t NP[RW];
#pragma unroll
    for (int u = 0; u < RW; ++u) NP[u] = 0u;
    int n_new = 0, spent = 0, snap_at = -1;
    Row<WD> nx;
    fetch_row<WD>(rs, st.base, 32 * warp + lane, nx);
    while (st.base < rs.R) {
        const bool valid = nx.valid;
        uint32_t q[WD], cr[RW];
        uint4 yr[1] = {nx.y}, acc;
        const long long idx = rs.seen + nx.i;
        const uint32_t weight = nx.weight;
        make_q<WD>(nx.x, valid, rs.raw, q);
        fetch_row<WD>(rs, st.base, nt + 32 * warp + lane, nx);  // the next round's row, in flight
        table_reduce<RW, WD>(TB, np, q, acc, cr);
        xor4(yr[0], acc);
        if (n_new) {
#pragma unroll
            for (int u = 0; u < RW; ++u) {
                const uint32_t sel = cr[u];
                uint32_t uw = __reduce_or_sync(FULL, sel & NP[u]);
                while (uw) {
                    const int b = __ffs(uw) - 1;
                    uw &= uw - 1;
                    const uint32_t* row = S + (int)FL[32 * u + b] * RS;
                    if ((sel >> b) & 1u) {
                        xor4(yr[0], *reinterpret_cast<const uint4*>(row));
#pragma unroll
                        for (int v = 0; v <= u; ++v) cr[v] ^= row[4 + v];
                    }
                }
            }
        }
        uint32_t nz = 0;
#pragma unroll
        for (int u = 0; u < RW; ++u) nz |= cr[u];
        if (valid && !nz && nonzero4(yr[0])) {
            st.cnt += weight;
            st.first = min(st.first, idx);
        }
        bool inserted = false;
        uint32_t c1 = __ballot_sync(FULL, valid && nz != 0u);
        uint32_t xr[1][RW], N1[RW];
#pragma unroll
        for (int u = 0; u < RW; ++u) xr[0][u] = cr[u];
        if constexpr (CTA) {
            uint32_t wmask = publish_candidates(c1, wc, st.parity, warp, lane, G);
            inserted = wmask != 0u;
            while (wmask) {
                const int fw = __ffs(wmask) - 1;
                if (warp == fw) {
                    (void)insert_rows<RW, RS>(xr, yr, c1, S, FL, lane, idx, weight, st.first, st.cnt, N1);
                    if (lane < RW) {
                        uint32_t t = 0;
#pragma unroll
                        for (int u = 0; u < RW; ++u)
                            if (u == lane) t = N1[u];
                        NPR[lane] = t;
                    }
                    c1 = 0u;
                }
                __syncthreads();
#pragma unroll
                for (int u = 0; u < RW; ++u) {
                    N1[u] = NPR[u];
                    n_new += __popc(N1[u]);
                }
                back_clear<RW, RS>(S, FL, NP, N1, lane, warp, G);
                if (warp > fw && c1) {
#pragma unroll
                    for (int u = 0; u < RW; ++u) {
                        const uint32_t sel = xr[0][u];
                        uint32_t uw = __reduce_or_sync(FULL, sel & N1[u]);
                        while (uw) {
                            const int b = __ffs(uw) - 1;
                            uw &= uw - 1;
                            const uint32_t* row = S + (int)FL[32 * u + b] * RS;
                            if ((sel >> b) & 1u) {
                                xor4(yr[0], *reinterpret_cast<const uint4*>(row));
#pragma unroll
                                for (int v = 0; v <= u; ++v) xr[0][v] ^= row[4 + v];
                            }
                        }
                    }
                    uint32_t left = 0;
#pragma unroll
                    for (int u = 0; u < RW; ++u) left |= xr[0][u];
                    if (((c1 >> lane) & 1u) && !left && nonzero4(yr[0])) {
                        st.cnt += weight;
                        st.first = min(st.first, idx);
                    }
                    c1 = __ballot_sync(FULL, left != 0u);
                }
#pragma unroll
                for (int u = 0; u < RW; ++u) NP[u] |= N1[u];
                wmask = publish_candidates(c1, wc, st.parity, warp, lane, G);
            }
        } else if (c1) {
            inserted = true;
            n_new += insert_rows<RW, RS>(xr, yr, c1, S, FL, lane, idx, weight, st.first, st.cnt, N1);
            back_clear<RW, RS>(S, FL, NP, N1, lane, 0, 1);
            __syncwarp();
#pragma unroll
            for (int u = 0; u < RW; ++u) NP[u] |= N1[u];
        }
        st.base = step_to(st.base, nt, rs.R);
        if constexpr (CTA) {
            st.quiet = inserted ? 0 : st.quiet + 1;
            if (a.handoff_tables && st.quiet >= HANDOFF_QUIET && rs.R - st.base >= st.hand_min && st.rank + n_new < d &&
                d * RS <= CHECK_BASIS_WORDS) {
                snap_at = st.base;
                break;
            }
        }
        spent += n_new;
        if (n_new && spent > (CTA ? 64 : 4 * np)) break;  // a new table pays
    }
    if (n_new) {
        // N into the basis: full residuals, then step (5) on the older rows
        uint32_t NF[WD];
#pragma unroll
        for (int v = 0; v < WD; ++v) NF[v] = 0u;
#pragma unroll
        for (int u = 0; u < RW; ++u) {
            const bool mine = (NP[u] >> lane) & 1u;
            const int coord = mine ? (int)FL[32 * u + lane] : 0;
            if (mine && (!CTA || u % G == warp)) {
                uint32_t* row = S + coord * RS;
                uint32_t c[RW], xf[WD];
#pragma unroll
                for (int v = 0; v < RW; ++v) c[v] = row[4 + v];
                decompress_residual<WD, RW>(c, FL, xf);
#pragma unroll
                for (int v = 0; v < WD; ++v) row[4 + v] = xf[v];
            }
#pragma unroll
            for (int v = 0; v < WD; ++v)
                NF[v] |= __reduce_or_sync(FULL, (mine && (coord >> 5) == v) ? 1u << (coord & 31) : 0u);
        }
        group_sync<CTA>();
        back_clear<WD, RS>(S, nullptr, st.P, NF, lane, warp, G);
        group_sync<CTA>();
#pragma unroll
        for (int v = 0; v < WD; ++v) st.P[v] |= NF[v];
        st.rank += n_new;
    }
    return snap_at;
}

// The residual planes of a table of a basis of m free coordinates: few
// instances of the rounds, so 0 and 3 words take the next one up.
__device__ __forceinline__ int table_planes(int m)
{
    const int rw = (m + 31) >> 5;
    return rw == 0 ? 1 : (rw == 3 ? 4 : rw);
}

__device__ __forceinline__ int table_room(int d, int rw) { return 16 * ((d + 3) >> 2) * (4 + rw); }

// Builds the table of the basis and runs rounds against it.
template <int WD, int RW, bool CTA>
__device__ __forceinline__ int table_phase(const LearnArgs& a, const RowStream& rs, ElimState<WD>& st, uint32_t* S,
                                           uint32_t* TB, uint16_t* FL, int d, int wd, uint32_t* wc, uint32_t* NPR)
{
    build_table_smem<WD, RW, CTA>(S, st.P, d, wd, TB, FL, CTA ? (int)threadIdx.x : (int)(threadIdx.x & 31),
                                  CTA ? (int)blockDim.x : 32);
    return table_rounds<WD, RW, CTA>(a, rs, st, S, TB, FL, d, wc, NPR);
}

// The first rows of an empty basis, up to OPEN_K a lane, by one warp: there is
// nothing to reduce them by, so they are eliminated among themselves, in
// stream order, and what remains of them is the reduced basis.  Each insertion
// serves all of them: with 128 rows at a time most contexts (median 75
// distinct rows) never walk their basis at all, which costs about 17
// instructions per pivot and 32 rows against 8 or so here.  The code takes the
// rows of slot 0 and rotates the slots, so it stands once: unrolled over the
// slots, the kernel waited for instructions three times as long.
constexpr int OPEN_K = 4;

template <int WD>
__device__ __forceinline__ void open_basis(const RowStream& rs, ElimState<WD>& st, uint32_t* S, int lane)
{
    constexpr int K = OPEN_K, RS = row_stride(WD);
    uint32_t xr[K][WD];
    uint4 yr[K];
    int pk[K];
    const int n_live = rs.R > 32 * (K - 1) ? K : (rs.R + 31) >> 5;
    uint32_t live = (1u << n_live) - 1u;
#pragma unroll
    for (int t = 0; t < K; ++t) {
        Row<WD> r;
        fetch_row<WD>(rs, 0, 32 * t + lane, r);
        make_q<WD>(r.x, r.valid, rs.raw, xr[t]);
        yr[t] = r.y;
        pk[t] = -1;
    }
#pragma unroll 1
    for (int t = 0; t < n_live; ++t) {
        uint32_t cand = __ballot_sync(FULL, nonzero_row<WD>(xr[0]));
#pragma unroll 1
        while (cand) {
            const int i = __ffs(cand) - 1;
            uint32_t b[WD];
            uint4 z;
            broadcast_row<WD>(xr[0], yr[0], i, b, z);
            const int k = pivot_step<WD - 1, WD, K>(xr, yr, b, z, lane == i, live, st.P);
            ++st.rank;
            if (lane == i) pk[0] = k;
            // the rows after it that are not zero yet
            cand = (0xfffffffeu << i) & __ballot_sync(FULL, nonzero_row<WD>(xr[0]));
        }
        const int kr = 32 * t + lane;
        if (kr < rs.R && pk[0] < 0 && nonzero4(yr[0])) {  // in the span of the rows before it
            st.cnt += 1u + (rs.dups ? (uint32_t)ld(rs.dups + kr) : 0u);
            st.first = min(st.first, rs.seen + (rs.reps ? ld(rs.reps + kr) : kr));
        }
        // slot 1 becomes slot 0, slot 0 the last
        uint32_t x0[WD];
        const uint4 y0 = yr[0];
        const int p0 = pk[0];
#pragma unroll
        for (int v = 0; v < WD; ++v) x0[v] = xr[0][v];
#pragma unroll
        for (int u = 0; u + 1 < K; ++u) {
#pragma unroll
            for (int v = 0; v < WD; ++v) xr[u][v] = xr[u + 1][v];
            yr[u] = yr[u + 1];
            pk[u] = pk[u + 1];
        }
#pragma unroll
        for (int v = 0; v < WD; ++v) xr[K - 1][v] = x0[v];
        yr[K - 1] = y0;
        pk[K - 1] = p0;
        live = (live >> 1) | ((live & 1u) << (K - 1));
    }
#pragma unroll
    for (int t = 0; t < K; ++t)
        if (pk[t] >= 0) store_row<WD>(S + pk[t] * RS, xr[t], yr[t]);
    __syncwarp();
    st.base = step_to(0, 32 * n_live, rs.R);
}

// A round of 32 rows by one warp against the basis itself: walk, insert the
// candidates, clear their columns from the older rows.
template <int WD>
__device__ __forceinline__ void walk_round(const RowStream& rs, ElimState<WD>& st, uint32_t* S, int d, int wd, int lane)
{
    constexpr int RS = row_stride(WD);
    uint32_t xr[1][WD];
    Row<WD> r;
    fetch_row<WD>(rs, st.base, lane, r);
    uint4 yr[1] = {r.y};
    const long long idx = rs.seen + r.i;
    make_q<WD>(r.x, r.valid, rs.raw, xr[0]);
    if (st.rank) reduce_rows<WD>(xr[0], yr[0], S, st.P, mixed_words<WD>(st.P, d, wd));
    uint32_t nz = 0;
#pragma unroll
    for (int v = 0; v < WD; ++v) {
        xr[0][v] &= ~st.P[v];
        nz |= xr[0][v];
    }
    if (r.valid && !nz && nonzero4(yr[0])) {
        st.cnt += r.weight;
        st.first = min(st.first, idx);
    }
    const uint32_t cand = __ballot_sync(FULL, r.valid && nz != 0u);
    if (cand) {
        uint32_t NP[WD];
        st.rank += insert_rows<WD, RS>(xr, yr, cand, S, nullptr, lane, idx, r.weight, st.first, st.cnt, NP);
        back_clear<WD, RS>(S, nullptr, st.P, NP, lane, 0, 1);
        __syncwarp();
#pragma unroll
        for (int v = 0; v < WD; ++v) st.P[v] |= NP[v];
    }
    st.base = step_to(st.base, 32, rs.R);
}

__device__ __forceinline__ RowStream row_stream(const StoreDev& s, const LearnArgs& a, const CtxDesc& cd, int c,
                                                bool& deduped)
{
    RowStream rs;
    const int64_t r0 = a.row_off[c];
    const int T = (int)(a.row_off[c + 1] - r0);
    const int rc = a.rep_count ? a.rep_count[c] : all_rows(T);
    deduped = rc >= 0;
    rs.R = deduped ? rc : rows_of(rc);
    rs.reps = deduped ? a.rep_list + r0 : nullptr;
    rs.dups = deduped ? a.rep_dup + r0 : nullptr;
    rs.xc = a.x + a.x_off[c];
    rs.yc = a.y + r0;
    rs.n = cd.n;
    rs.xw = cd.xw;
    rs.raw = s.raw;
    rs.seen = s.rows_seen[c];
    return rs;
}

// A warp streams the representatives of context c through its basis.
template <int WD>
__device__ void elim_warp(const StoreDev& s, const LearnArgs& a, int c, uint32_t* region, int region_words)
{
    constexpr int RS = row_stride(WD);
    const int lane = threadIdx.x & 31;
    const CtxDesc cd = s.desc[c];
    const int rank0 = s.rank[c];
    bool deduped;
    const RowStream rs = row_stream(s, a, cd, c, deduped);
    uint32_t* const S = region;
    ElimState<WD> st;
#pragma unroll
    for (int v = 0; v < WD; ++v) st.P[v] = (rank0 && v < cd.wd) ? s.pivot[cd.pw_off + v] : 0u;
    st.rank = rank0;
    st.base = 0;
    st.quiet = st.parity = 0;
    st.first = LLONG_MAX;
    st.cnt = 0;
    if (rank0) {
        basis_to_smem<WD>(s, cd, S, st.P, lane, 0, 1);
        __syncwarp();
    } else {
        open_basis<WD>(rs, st, S, lane);
    }
    // the table's room: after the basis, the free-coordinate list at the region's end
    uint32_t* const TB = S + cd.d * RS;
    uint16_t* const FL = reinterpret_cast<uint16_t*>(region + region_words - FL_WORDS);
    const int tab_cap = region_words - FL_WORDS - cd.d * RS;
    const int np = (cd.d + 3) >> 2;
    while (st.base < rs.R) {
        const int left = rs.R - st.base;
        // A table costs about 40 np warp-instructions to build and 8 np a
        // round to use, a walk about 14 per pivot and round: the table pays
        // from the rounds left where the saving covers the build.
        const int rw = table_planes(cd.d - st.rank);
        if (a.tables && rw <= WARP_TABLE_RW && table_room(cd.d, rw) <= tab_cap &&
            (((int64_t)left + 31) >> 5) * (14 * st.rank - 8 * np) > 40 * np) {
            (void)table_phase<WD, 1, false>(a, rs, st, S, TB, FL, cd.d, cd.wd, nullptr, nullptr);
        } else {
            walk_round<WD>(rs, st, S, cd.d, cd.wd, lane);
        }
    }
    warp_stats(st.first, st.cnt);
    if (st.rank != rank0) {
        if (lane < cd.wd) {
            uint32_t t = 0;
#pragma unroll
            for (int v = 0; v < WD; ++v)
                if (v == lane) t = st.P[v];
            s.pivot[cd.pw_off + lane] = t;
        }
        basis_from_smem<WD>(s, cd, S, st.P, lane, 0, 1);
    }
    if (lane == 0) {
        s.rank[c] = st.rank;
        commit_stats(s, c, st.first, st.cnt);
        s.rows_seen[c] = rs.seen + (a.row_off[c + 1] - a.row_off[c]);
    }
    __syncwarp();
}

// A CTA streams the representatives of context c through its basis.
template <int WD>
__device__ void elim_cta(const StoreDev& s, const LearnArgs& a, int c, uint32_t* region, int region_words)
{
    constexpr int RS = row_stride(WD);
    const int G = (int)(blockDim.x >> 5);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = threadIdx.x, nt = blockDim.x;
    const CtxDesc cd = s.desc[c];
    uint32_t* const NPR = region + CTL_NPR;
    uint32_t* const wc = region + CTL_CAND;
    unsigned long long* cnt_s = reinterpret_cast<unsigned long long*>(region + CTL_CNT);
    long long* first_s = reinterpret_cast<long long*>(region + CTL_FIRST);
    uint32_t* const S = region + CTL_WORDS;
    const int rank0 = s.rank[c];
    bool deduped;
    const RowStream rs = row_stream(s, a, cd, c, deduped);
    ElimState<WD> st;
#pragma unroll
    for (int v = 0; v < WD; ++v) st.P[v] = (rank0 && v < cd.wd) ? s.pivot[cd.pw_off + v] : 0u;
    st.rank = rank0;
    st.base = a.resume_from ? a.resume_from[c] : 0;  // the first representative of this launch
    if constexpr (WD > WIDE_M_WD) st.base = a.open_from[c];
    st.quiet = st.parity = 0;
    st.hand_min = handoff_least(a, deduped);
    st.first = LLONG_MAX;
    st.cnt = 0;
    if (t == 0) {
        *cnt_s = 0ull;
        *first_s = LLONG_MAX;
    }
    int stop_at = -1;
    if constexpr (WD > NARROW_WD) {  // full rank: the rows left are checks only (below)
        if (!deduped && a.late_list && rank0 == cd.d && rs.R - st.base >= FULL_LATE_MIN) stop_at = st.base;
    }
    if (rank0 && stop_at < 0 && st.base < rs.R) basis_to_smem<WD>(s, cd, S, st.P, lane, warp, G);
    __syncthreads();
    uint64_t mixed = mixed_words<WD>(st.P, cd.d, cd.wd);
    uint32_t* const TB = S + cd.d * RS;
    uint16_t* const FL = reinterpret_cast<uint16_t*>(region + region_words - FL_WORDS);
    const int tab_cap = region_words - FL_WORDS - CTL_WORDS - cd.d * RS;
    const int np = (cd.d + 3) >> 2;
    Row<WD> nx;
    fetch_row<WD>(rs, st.base, t, nx);
    int snap_at = -1;  // handed off from this representative on
    while (st.base < rs.R && stop_at < 0) {
        if constexpr (WD <= TABLE_MAX_WD) {
            // by lookup table where it fits and costs fewer instructions than
            // the walk (about d/4 lookups a row against rank/2 two-pivot steps)
            const int rw = table_planes(cd.d - st.rank);
            if (a.tables && rw <= TABLE_MAX_RW && table_room(cd.d, rw) <= tab_cap && 4 * st.rank >= 5 * np) {
                if (rw == 1) snap_at = table_phase<WD, 1, true>(a, rs, st, S, TB, FL, cd.d, cd.wd, wc, NPR);
                else if (rw == 2) snap_at = table_phase<WD, 2, true>(a, rs, st, S, TB, FL, cd.d, cd.wd, wc, NPR);
                else snap_at = table_phase<WD, 4, true>(a, rs, st, S, TB, FL, cd.d, cd.wd, wc, NPR);
                if (snap_at >= 0) break;
                mixed = mixed_words<WD>(st.P, cd.d, cd.wd);
                fetch_row<WD>(rs, st.base, t, nx);
                continue;
            }
        }
        const bool valid = nx.valid;
        uint32_t xr[1][WD];
        uint4 yr[1] = {nx.y};
        const long long idx = rs.seen + nx.i;
        const uint32_t weight = nx.weight;
        make_q<WD>(nx.x, valid, rs.raw, xr[0]);
        fetch_row<WD>(rs, st.base, nt + t, nx);
        if (st.rank) reduce_rows<WD>(xr[0], yr[0], S, st.P, mixed);
        uint32_t nz = 0;
#pragma unroll
        for (int v = 0; v < WD; ++v) {
            xr[0][v] &= ~st.P[v];
            nz |= xr[0][v];
        }
        if (valid && !nz && nonzero4(yr[0])) {
            st.cnt += weight;
            st.first = min(st.first, idx);
        }
        uint32_t cand = __ballot_sync(FULL, valid && nz != 0u);
        uint32_t wmask = publish_candidates(cand, wc, st.parity, warp, lane, G);
        st.base = step_to(st.base, nt, rs.R);
        st.quiet = wmask ? 0 : st.quiet + 1;
        // the first warp with candidates inserts them; then every warp clears
        // its share of the older rows (step (5)) and reduces its own
        // candidates by the new rows, so that what is left for the later
        // warps to insert, one after another, is only what is new
        while (wmask) {
            const int fw = __ffs(wmask) - 1;
            uint32_t NP[WD];
            if (warp == fw) {
                (void)insert_rows<WD, RS>(xr, yr, cand, S, nullptr, lane, idx, weight, st.first, st.cnt, NP);
                if (lane == 0) {
#pragma unroll
                    for (int v = 0; v < WD; ++v) NPR[v] = NP[v];
                }
                cand = 0u;
            }
            __syncthreads();
#pragma unroll
            for (int v = 0; v < WD; ++v) {
                NP[v] = NPR[v];
                st.rank += __popc(NP[v]);
            }
            back_clear<WD, RS>(S, nullptr, st.P, NP, lane, warp, G);
            if (warp > fw && cand) {
                reduce_rows<WD>(xr[0], yr[0], S, NP, ~0ull);
                uint32_t left = 0;
#pragma unroll
                for (int v = 0; v < WD; ++v) left |= xr[0][v];
                if (((cand >> lane) & 1u) && !left && nonzero4(yr[0])) {
                    st.cnt += weight;
                    st.first = min(st.first, idx);
                }
                cand = __ballot_sync(FULL, left != 0u);
            }
#pragma unroll
            for (int v = 0; v < WD; ++v) st.P[v] |= NP[v];
            wmask = publish_candidates(cand, wc, st.parity, warp, lane, G);
            if (!wmask) mixed = mixed_words<WD>(st.P, cd.d, cd.wd);
        }
        // (wide contexts) full rank with rows left: every later row is a check
        // only (the rows are their own representatives)
        if constexpr (WD > NARROW_WD) {
            if (!deduped && a.late_list && st.quiet == 0 && rs.R - st.base >= FULL_LATE_MIN && st.rank == cd.d) {
                stop_at = st.base;
                break;
            }
        }
        if constexpr (WD <= NARROW_WD || WD == WIDE_M_WD) {
            // a saturated context with many representatives left hands the
            // rest off to the parallel check (block-uniform)
            if (st.quiet >= HANDOFF_QUIET && rs.R - st.base >= st.hand_min && st.rank < cd.d &&
                cd.d * RS <= CHECK_BASIS_WORDS) {
                snap_at = st.base;
                break;
            }
        }
    }
    warp_stats(st.first, st.cnt);
    if (lane == 0 && st.cnt) {
        atomicAdd(cnt_s, st.cnt);
        atomicMin(first_s, st.first);
    }
    if (st.rank != rank0) {
        if (warp == 0) {
            for (int w0 = lane; w0 < cd.wd; w0 += 32) {
                uint32_t p = 0;
#pragma unroll
                for (int v = 0; v < WD; ++v)
                    if (v == w0) p = st.P[v];
                s.pivot[cd.pw_off + w0] = p;
            }
        }
        basis_from_smem<WD>(s, cd, S, st.P, lane, warp, G);
    }
    __syncthreads();
    if (t == 0) {
        s.rank[c] = st.rank;
        commit_stats(s, c, *first_s, *cnt_s);
        if (snap_at >= 0) {  // rows_seen is advanced by check_snap_kernel (or the launch that resumes it)
            a.snap_start[c] = snap_at;
            a.snap_list[atomicAdd(a.snap_count, 1)] = c;
        } else if (stop_at < 0) {
            s.rows_seen[c] = rs.seen + (a.row_off[c + 1] - a.row_off[c]);
        } else {  // rows_seen is advanced by verify_full_kernel
            a.late_start[c] = stop_at;
            a.late_list[atomicAdd(a.late_count, 1)] = c;
        }
    }
    __syncthreads();
}

// ------------------------------------------------------------------ queues

// The contexts of class CLS that this launch takes, each by the whole CTA.  A
// launch that takes up contexts sent back by the check walks their list and
// keeps those of its class.
__device__ __forceinline__ int width_class(int wd)
{
    return wd <= SMALL_WD ? CLS_CTA_S : (wd <= NARROW_WD ? CLS_CTA : (wd <= WIDE_M_WD ? CLS_WIDE_M : CLS_WIDE));
}

template <int CLS, int RESUME, typename F>
__device__ __forceinline__ void elim_cta_queue(const StoreDev& s, const LearnArgs& a, F&& run)
{
    __shared__ int s_item;
    const bool resume = a.resume_from != nullptr;
    const int n = resume ? *a.resume_count : a.counters[CNT_COUNT + CLS];
    const int32_t* const list = resume ? a.resume_list : a.queue + a.counters[CNT_BEGIN + CLS];
    int* const head = a.counters + CNT_HEAD + (resume ? RESUME : CLS);
    if (n == 0) return;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = atomicAdd(head, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= n) break;
        const int c = list[item];
        if (resume && width_class(s.desc[c].wd) != CLS) continue;
        // (elim_open_kernel marks the start of the widest ones)
        if (threadIdx.x == 0 && !resume && CLS != CLS_WIDE) time_mark(a.timing, c, 2);
        run(c);
        if (threadIdx.x == 0) time_mark(a.timing, c, 3);
    }
}

// CTA-owned contexts, then warp-owned ones (a region of shared memory a warp).
template <int C_CTA, int C_WARP, int RESUME, typename F>
__device__ __forceinline__ void elim_queues(const StoreDev& s, const LearnArgs& a, uint32_t* smem, int region_words,
                                            F&& run)
{
    elim_cta_queue<C_CTA, RESUME>(s, a, [&](int c) { run(c, std::true_type{}, smem, a.cta_region_words); });
    if (a.resume_from) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_w = a.counters[CNT_COUNT + C_WARP];
    const int b_w = a.counters[CNT_BEGIN + C_WARP];
    uint32_t* region = smem + warp * region_words;
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(a.counters + CNT_HEAD + C_WARP, 1);
        item = __shfl_sync(FULL, item, 0);
        if (item >= n_w) break;
        const int c = a.queue[b_w + item];
        if (lane == 0) time_mark(a.timing, c, 2);
        run(c, std::false_type{}, region, region_words);
        if (lane == 0) time_mark(a.timing, c, 3);
    }
}

template <int WD, bool CTA>
__device__ __forceinline__ void elim_one(const StoreDev& s, const LearnArgs& a, int c, uint32_t* region, int words)
{
    if constexpr (CTA) elim_cta<WD>(s, a, c, region, words);
    else elim_warp<WD>(s, a, c, region, words);
}

// CTAs of a kernel with `smem` bytes of dynamic shared memory that fit an SM
// (228 KB, 1 KB of it taken by each CTA), at most `most` by its registers.
inline int resident_ctas(size_t smem, int most)
{
    const int fit = (int)((size_t)(228 * 1024) / (smem + 1024 + 64));
    return fit < 1 ? 1 : (fit < most ? fit : most);
}

template <typename K>
cudaError_t launch_queues(K kernel, const StoreDev& sd, LearnArgs la, int max_words, int region_words, int warps,
                          int per_sm, int num_sms, cudaStream_t cs)
{
    const size_t regions = (size_t)warps * (size_t)region_words;
    const size_t smem = 4 * (regions > (size_t)max_words ? regions : (size_t)max_words);
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    la.cta_region_words = (int)(smem / 4);
    f2_launch(kernel, num_sms * resident_ctas(smem, per_sm), warps * 32, smem, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, la);
    return cudaGetLastError();
}

}  // namespace f2
