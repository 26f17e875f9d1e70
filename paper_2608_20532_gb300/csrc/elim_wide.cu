// Elimination of the contexts of more than NARROW_WD words, a CTA each.
#include "elim.cuh"

namespace f2 {
namespace {

template <int WDT, int CLS, int RESUME>
__global__ void __launch_bounds__(WIDE_WARPS * 32, WDT <= WIDE_M_WD ? 2 : 1) elim_wide_kernel(StoreDev s, LearnArgs a)
{
    pdl_wait();
    extern __shared__ __align__(16) uint32_t smem[];
    elim_cta_queue<CLS, RESUME>(s, a, [&](int c) { elim_cta<WDT>(s, a, c, smem, a.cta_region_words); });
}

// ---------------------------------------------------------------------------
// The first OPEN_THREADS rows of an empty basis of up to WIDE_WD words, a row
// a thread, in registers.  The rows go in stream order, OPEN_GROUP at a time:
// their warp puts one after another into shared memory, finds its highest set
// bit and applies it to its own rows at once; after one barrier every thread
// of the other warps whose row has such a bit XORs the row from there
// (broadcast loads, only the words up to the pivot's).  The rows stay reduced
// among themselves, so what remains is the reduced basis.  (One row a barrier
// took 1,475 cycles a pivot, four take 1,310, of which the XORs alone 610: 38
// integer instructions a warp at half rate; groups of 8, 16 and 32 rows were
// no faster.)  Streaming 256 rows at a time against a basis in shared memory,
// the 1,025 pivots of a dense 1,024-bit context took 3,000 cycles each, most of
// it in reading older rows a lane each.  Two batches of 65,536 rows for 64 such
// contexts went from 3,012 to 2,256 us, and to 2,180 with four rows a barrier.
// Dense rows are a few pivots short of full rank after d rows: up to OPEN_EXTRA
// further rows are reduced one at a time by all threads (a XOR reduction of the
// rows their bits select).  (Rows this wide are never deduplicated: each stands
// for itself.)
// ---------------------------------------------------------------------------
constexpr int OPEN_THREADS = 1024;
constexpr int OPEN_GROUP = 4;
constexpr int OPEN_EXTRA = 32;
constexpr int OPEN_Z = 9;  // uint4 index of the word in a shared row; the features before it

struct OpenSmem {
    uint4 row[2][OPEN_GROUP][OPEN_Z + 1];
    uint32_t q[WIDE_WD + 3];  // a further row's own bits
    uint32_t mask[WIDE_WD + 3];
    int head[2][OPEN_GROUP];
    int holder;
    unsigned long long cnt;
    long long first;
};

template <int W>
__device__ __forceinline__ void open_xor(uint32_t (&x)[WIDE_WD], uint4& y, const uint4* __restrict__ row, uint32_t m,
                                         bool own)
{
    if ((x[W] & m) != 0u && !own) {
        xor4(y, row[OPEN_Z]);
#pragma unroll
        for (int c = 0; 4 * c <= W; ++c) {
            const uint4 t = row[c];
            const uint32_t e[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (4 * c + j <= W) x[4 * c + j] ^= e[j];
        }
    }
}

// XOR the row with pivot k into this thread's row if that has bit k set.
__device__ __forceinline__ void open_step(int k, uint32_t (&x)[WIDE_WD], uint4& y, const uint4* __restrict__ row,
                                          bool own)
{
    const uint32_t m = 1u << (k & 31);
#define F2_OPEN(W) case W: open_xor<W>(x, y, row, m, own); break;
    switch (k >> 5) {
        F2_OPEN(0) F2_OPEN(1) F2_OPEN(2) F2_OPEN(3) F2_OPEN(4) F2_OPEN(5) F2_OPEN(6) F2_OPEN(7) F2_OPEN(8)
        F2_OPEN(9) F2_OPEN(10) F2_OPEN(11) F2_OPEN(12) F2_OPEN(13) F2_OPEN(14) F2_OPEN(15) F2_OPEN(16)
        F2_OPEN(17) F2_OPEN(18) F2_OPEN(19) F2_OPEN(20) F2_OPEN(21) F2_OPEN(22) F2_OPEN(23) F2_OPEN(24)
        F2_OPEN(25) F2_OPEN(26) F2_OPEN(27) F2_OPEN(28) F2_OPEN(29) F2_OPEN(30) F2_OPEN(31) F2_OPEN(32)
    default: break;
    }
#undef F2_OPEN
}

// Highest set bit of a row in shared memory, by a warp; -1 if it is zero.
__device__ __forceinline__ int open_top(const uint4* row, int lane)
{
    static_assert(WIDE_WD == 33, "one word past the lanes");
    const uint32_t* w = reinterpret_cast<const uint32_t*>(row);
    const uint32_t v = w[lane], last = w[32];
    const uint32_t b = __ballot_sync(FULL, v != 0u);
    const int tw = b ? 31 - __clz(b) : 0;
    const uint32_t t = __shfl_sync(FULL, v, tw);
    if (last) return 1024 + 31 - __clz(last);
    return b ? 32 * tw + 31 - __clz(t) : -1;
}

__global__ void __launch_bounds__(OPEN_THREADS, 1) elim_open_kernel(StoreDev s, LearnArgs a)
{
    pdl_wait();
    __shared__ OpenSmem sm;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n_items = a.counters[CNT_COUNT + CLS_WIDE];
    const int32_t* const list = a.queue + a.counters[CNT_BEGIN + CLS_WIDE];
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int c = list[item];
        if (t == 0) time_mark(a.timing, c, 2);
        if (s.rank[c] != 0) {
            if (t == 0) a.open_from[c] = 0;
            continue;
        }
        const CtxDesc cd = s.desc[c];
        bool deduped;
        const RowStream rs = row_stream(s, a, cd, c, deduped);
        const int n = rs.R < OPEN_THREADS ? rs.R : OPEN_THREADS;
        Row<WIDE_WD> r;
        fetch_row<WIDE_WD>(rs, 0, t, r);
        uint32_t x[WIDE_WD];
        make_q<WIDE_WD>(r.x, r.valid, rs.raw, x);
        uint4 y = r.y;
        int pk = -1, rank = 0;
        __syncthreads();  // the last context's shared memory is done with
        if (t < WIDE_WD) sm.mask[t] = 0u;
        if (t == 0) {
            sm.cnt = 0ull;
            sm.first = LLONG_MAX;
        }
        for (int i0 = 0, buf = 0; i0 < n && rank < cd.d; i0 += OPEN_GROUP, buf ^= 1) {
            const bool owner = warp == (i0 >> 5);
            if (owner) {
#pragma unroll 1
                for (int j = 0; j < OPEN_GROUP; ++j) {
                    uint4* const row = sm.row[buf][j];
                    const bool own = t == i0 + j;
                    if (own) {
#pragma unroll
                        for (int v4 = 0; v4 < OPEN_Z; ++v4) {
                            uint32_t e[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                e[u] = 4 * v4 + u < WIDE_WD ? x[4 * v4 + u < WIDE_WD ? 4 * v4 + u : 0] : 0u;
                            row[v4] = make_uint4(e[0], e[1], e[2], e[3]);
                        }
                        row[OPEN_Z] = y;
                    }
                    __syncwarp();
                    const int k = open_top(row, lane);
                    if (own) {
                        sm.head[buf][j] = k;
                        pk = k;
                    }
                    if (k >= 0) open_step(k, x, y, row, own);
                }
            }
            __syncthreads();
#pragma unroll 1
            for (int j = 0; j < OPEN_GROUP; ++j) {
                const int k = sm.head[buf][j];
                if (k < 0) continue;
                ++rank;
                if (!owner) open_step(k, x, y, sm.row[buf][j], false);
            }
        }
        // rows without a pivot lie in the span of the rows before them
        if (t < n && pk < 0 && nonzero4(y)) {
            atomicAdd(&sm.cnt, 1ull);
            atomicMin(&sm.first, rs.seen + t);
        }
        int base = n;
        for (int extra = 0; rank < cd.d && base < rs.R && extra < OPEN_EXTRA; ++extra, ++base) {
            __syncthreads();
            uint4* const arow = sm.row[0][0];
            uint32_t* const acc = reinterpret_cast<uint32_t*>(arow);
            if (warp == 0) {
                const uint32_t* xr = rs.xc + (int64_t)base * rs.xw;
                for (int w = lane; w < WIDE_WD + 3; w += 32) {
                    auto word = [&](int v) {
                        if (v < 0 || v >= rs.xw) return 0u;
                        uint32_t u = ld(xr + v);
                        if (v == rs.xw - 1 && (rs.n & 31)) u &= (1u << (rs.n & 31)) - 1u;
                        return u;
                    };
                    uint32_t q = 0;
                    if (w < WIDE_WD) q = rs.raw ? word(w) : (word(w) << 1) | (w ? word(w - 1) >> 31 : 1u);
                    acc[w] = q;
                    sm.q[w] = q;
                }
                if (lane == 0) {
                    arow[OPEN_Z] = ld(rs.yc + base);
                    sm.holder = OPEN_THREADS;
                }
            }
            __syncthreads();
            const bool sel = pk >= 0 && ((sm.q[pk >= 0 ? pk >> 5 : 0] >> (pk & 31)) & 1u);
            if (__any_sync(FULL, sel)) {
#pragma unroll
                for (int v = 0; v < WIDE_WD; ++v) {
                    const uint32_t g = __reduce_xor_sync(FULL, sel ? x[v] : 0u);
                    if (lane == 0 && g) atomicXor(acc + v, g);
                }
                const uint32_t z[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const uint32_t g = __reduce_xor_sync(FULL, sel ? z[v] : 0u);
                    if (lane == 0 && g) atomicXor(acc + 4 * OPEN_Z + v, g);
                }
            }
            if (pk < 0) atomicMin(&sm.holder, t);
            __syncthreads();
            const int k = open_top(arow, lane);
            const uint4 z = arow[OPEN_Z];
            if (k < 0) {
                if (t == 0 && nonzero4(z)) {
                    ++sm.cnt;
                    if (rs.seen + base < sm.first) sm.first = rs.seen + base;
                }
                continue;
            }
            ++rank;
            open_step(k, x, y, arow, false);
            if (t == sm.holder) {
#pragma unroll
                for (int v = 0; v < WIDE_WD; ++v) x[v] = acc[v];
                y = z;
                pk = k;
            } else if (sm.holder == OPEN_THREADS && t == 0) {
                // every thread holds a pivot: this is the last one (d <= 1,025)
                s.bz[cd.slot_off + k] = z;
                for (int v = 0; v < cd.wd; ++v) s.bx[cd.xw_off + (int64_t)k * cd.wd + v] = acc[v];
                atomicOr(sm.mask + (k >> 5), 1u << (k & 31));
            }
        }
        if (pk >= 0) {
            s.bz[cd.slot_off + pk] = y;
            uint32_t* dst = s.bx + cd.xw_off + (int64_t)pk * cd.wd;
#pragma unroll
            for (int v = 0; v < WIDE_WD; ++v)
                if (v < cd.wd) dst[v] = x[v];
            atomicOr(sm.mask + (pk >> 5), 1u << (pk & 31));
        }
        __syncthreads();
        if (t < cd.wd) s.pivot[cd.pw_off + t] = sm.mask[t];
        if (t == 0) {
            s.rank[c] = rank;
            a.open_from[c] = base;
            commit_stats(s, c, sm.first, sm.cnt);
        }
    }
}

template <typename K>
cudaError_t launch(K kernel, const StoreDev& sd, LearnArgs la, int max_d, int wdt, int per_sm, int num_sms,
                   cudaStream_t cs)
{
    la.cta_region_words = elim_words(max_d, wdt);
    const size_t smem = 4 * (size_t)la.cta_region_words;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    f2_launch(kernel, num_sms * resident_ctas(smem, per_sm), WIDE_WARPS * 32, smem, cs, sd.num_ctx <= EARLY_MAX_CTX, sd,
              la);
    return cudaGetLastError();
}

}  // namespace

cudaError_t elim_launch_wide(const StoreDev& sd, LearnArgs la, int max_d, bool medium, int num_sms, cudaStream_t cs)
{
    if (medium)
        return launch(elim_wide_kernel<WIDE_M_WD, CLS_WIDE_M, CLS_RESUME_W>, sd, la, max_d, WIDE_M_WD, 2, num_sms, cs);
    f2_launch(elim_open_kernel, num_sms, OPEN_THREADS, 0, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, la);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch(elim_wide_kernel<WIDE_WD, CLS_WIDE, CLS_RESUME_W>, sd, la, max_d, WIDE_WD, 1, num_sms, cs);
}

cudaError_t elim_load_wide()
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, elim_wide_kernel<WIDE_M_WD, CLS_WIDE_M, CLS_RESUME_W>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, elim_open_kernel);
    return e != cudaSuccess ? e : cudaFuncGetAttributes(&fa, elim_wide_kernel<WIDE_WD, CLS_WIDE, CLS_RESUME_W>);
}

}  // namespace f2
