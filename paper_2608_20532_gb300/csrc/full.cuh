// The full-rank check: what its two kernels (learn.cu: lookup tables in shared
// memory; verify_tc.cu: tensor cores) share.
#pragma once

#include "elim.cuh"

namespace f2 {

struct FullArgs {
    const int64_t* row_off;
    const int64_t* x_off;
    const uint32_t* x;
    const uint4* y;
    const int32_t* queue;
    const int* counters;
    int* ctr;                         // [2C]: chunks claimed, chunks done
    const int* late_count;            // contexts listed by the elimination kernels
    const int32_t* late_list;
    const int32_t* late_start;        // their first row left
    unsigned long long* cnt;          // [C] contradicting rows of the call
    unsigned long long* first;        // [C] first contradicting row of the call (all ones: none)
    int table_words;                  // FULL_TABLE_WORDS
    int tensor;                       // contexts of full_by_tensor are left to verify_tc_kernel
    int fail_wait;                    // test hook: verify_tc_kernel's waits for sums give up
};

// Which check a context with n features and T rows takes.  By rows of 300
// contexts with 16,384 each, the table check (n/4 lookups of 16 bytes a row)
// takes 125 + 0.67 n us and the tensor check 255 + 85 for each chunk of 256
// features, begun or whole, and 65 more where a feature row is not a multiple of
// 16 bytes (one word a load instead of four).  Table / tensor: 256 features
// 288 / 339 us, 384 379 / 423, 512 466 / 437, 544 492 / 581, 640 549 / 514,
// 736 629 / 583, 768 632 / 516, 800 666 / 636, 1,000 793 / 598.  Its map (128 bytes a
// feature, spread over a CTA's shared memory) wants rows, too: 600 contexts with
// 4,096 rows of 512 features 269 / 270, of 1,024 443 / 360, with 2,048 rows 159 / 172
// and 250 / 224; but where it runs at all, its CTAs' look through a list of 600
// contexts that are not its own costs 20 us, so the line is not drawn above 2,048.
constexpr int TC_CHUNK = 256;  // features of a chunk
constexpr int TC_MIN_ROWS = 2048;
__host__ __device__ __forceinline__ bool tensor_features(int n)
{
    const int chunks = (n + TC_CHUNK - 1) / TC_CHUNK;
    const int odd = (((n + 31) / 32) & 3) ? 195 : 0;
    return 2 * n > 400 + 255 * chunks + odd;
}
__host__ __device__ __forceinline__ bool full_by_tensor(int n, int64_t T)
{
    return T >= TC_MIN_ROWS && tensor_features(n);
}

cudaError_t verify_launch_tc(const StoreDev& sd, const FullArgs& fa, int num_sms, cudaStream_t cs);
cudaError_t verify_load_tc();

// The contexts to check: full at the start of the call, then full mid-call.
struct FullList {
    int nfull, begin, n;
    __device__ __forceinline__ FullList(const FullArgs& a)
        : nfull(a.counters[CNT_COUNT + CLS_FULL]), begin(a.counters[CNT_BEGIN + CLS_FULL]), n(nfull + *a.late_count)
    {
    }
    __device__ __forceinline__ int ctx(const FullArgs& a, int q) const
    {
        return q < nfull ? a.queue[begin + q] : a.late_list[q - nfull];
    }
    __device__ __forceinline__ int64_t start(const FullArgs& a, int q, int c) const
    {
        return q < nfull ? 0 : (int64_t)a.late_start[c];
    }
};

// A warp claims the next chunk k of a listed context: of the one at `stay` while
// it has any, else of the first with chunks left, 32 looked at together, from
// q0 round the list (`tried` of it are used up).  Returns its place in the list,
// or -1.  (One thread that went from context to context, an atomic on each, took
// most of the 29.6 us of the table kernel on 64 contexts that are all the other
// kernel's, now 5.1, and 28 of the 513 us of that one on 4.2M rows.)
__device__ __forceinline__ int full_claim(const StoreDev& s, const FullArgs& a, const FullList& l, bool tensor, int q0,
                                          int stay, int& tried, int lane, int& k)
{
    auto rows_left = [&](int q, int& c) {
        c = l.ctx(a, q);
        return a.row_off[c + 1] - a.row_off[c] - l.start(a, q, c);
    };
    auto take = [&](int q) {
        int c;
        const int64_t T = rows_left(q, c);
        if (lane == 0) k = atomicAdd(a.ctr + c, 1);
        k = __shfl_sync(FULL, k, 0);
        return (int64_t)k * FULL_CHUNK < T;
    };
    k = 0;
    if (stay >= 0 && take(stay)) return stay;
    while (tried < l.n) {
        int at = -1;
        if (tried + lane < l.n) {
            at = q0 + tried + lane;
            if (at >= l.n) at -= l.n;
            int c;
            const int64_t T = rows_left(at, c);
            if ((a.tensor && full_by_tensor(s.desc[c].n, T)) != tensor || (int64_t)__ldcg(a.ctr + c) * FULL_CHUNK >= T)
                at = -1;
        }
        const uint32_t left = __ballot_sync(FULL, at >= 0);
        if (!left) {
            tried += 32;
            continue;
        }
        at = __shfl_sync(FULL, at, __ffs(left) - 1);
        if (take(at)) return at;
    }
    return -1;
}

// A chunk of context c's rows is checked (one thread): cnt contradictions, the
// first at `first`; the last chunk of the context commits its counts and
// advances rows_seen.  Where a chunk's check failed (a wait gave up) its counts
// are unknown, so nothing of the context is committed: the mark is a bit that
// no count reaches.
constexpr unsigned long long FULL_FAILED = 1ull << 63;

__device__ __forceinline__ void full_commit(const StoreDev& s, const FullArgs& a, int c, int64_t i_first, int64_t T,
                                            unsigned long long cnt, unsigned long long first, bool failed)
{
    if (failed) {
        atomicOr(a.cnt + c, FULL_FAILED);
    } else if (cnt) {
        atomicAdd(a.cnt + c, cnt);
        atomicMin(a.first + c, first);
    }
    __threadfence();
    const int nch = (int)((T - i_first + FULL_CHUNK - 1) / FULL_CHUNK);
    if (atomicAdd(a.ctr + s.num_ctx + c, 1) != nch - 1) return;
    __threadfence();
    const unsigned long long tot = atomicAdd(a.cnt + c, 0ull);
    if (tot & FULL_FAILED) return;
    const unsigned long long fi = atomicMin(a.first + c, ~0ull);
    const long long seen = s.rows_seen[c];
    if (tot) {
        s.n_contra[c] += tot;
        s.contra[c] = 1;
        if (s.first_contra[c] < 0) s.first_contra[c] = seen + (long long)fi;
    }
    s.rows_seen[c] = seen + T;
}

}  // namespace f2
