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
};

// A context with n features and T rows to check goes to the tensor cores: the
// table check costs d/4 lookups of 16 bytes a row, 0.71 ms for 4.2M rows of
// 1,024 features, the tensor cores 0.54 ms; spreading the map over a CTA's
// shared memory (128 bytes a feature) wants a few thousand rows to pay.
constexpr int TC_MIN_N = 192;
constexpr int TC_MIN_ROWS = 2048;
__host__ __device__ __forceinline__ bool full_by_tensor(int n, int64_t T) { return n >= TC_MIN_N && T >= TC_MIN_ROWS; }

cudaError_t verify_launch_tc(const StoreDev& sd, const FullArgs& fa, int num_sms, cudaStream_t cs);
cudaError_t verify_load_tc();

// A chunk of context c's rows is checked (one thread): cnt contradictions, the
// first at `first`; the last chunk of the context commits its counts and
// advances rows_seen.
__device__ __forceinline__ void full_commit(const StoreDev& s, const FullArgs& a, int c, int64_t i_first, int64_t T,
                                            unsigned long long cnt, unsigned long long first)
{
    if (cnt) {
        atomicAdd(a.cnt + c, cnt);
        atomicMin(a.first + c, first);
    }
    __threadfence();
    const int nch = (int)((T - i_first + FULL_CHUNK - 1) / FULL_CHUNK);
    if (atomicAdd(a.ctr + s.num_ctx + c, 1) != nch - 1) return;
    __threadfence();
    const unsigned long long tot = atomicAdd(a.cnt + c, 0ull);
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
