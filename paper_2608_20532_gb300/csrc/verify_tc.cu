// The full-rank check (learn.cu) on the tensor cores.
//
// A context of full rank accepts a row iff y = T(phi(x)) = b XOR A x: over the
// integers, bit j of A x is the parity of a dot product of two 0/1 vectors of
// n <= 1024 entries, which the tensor cores' fp8 products and fp32 sums give
// exactly (sums of at most 1024 ones).  A CTA keeps the context's A (128 x n,
// one byte an entry) in shared memory and takes 128 rows at a time: two threads
// a row spread its feature bits to bytes in registers and store them to tensor
// memory, from where tcgen05.mma reads the rows; the 128 sums of a row come
// back to its threads, which pack their parities and compare them with y.  Two
// groups of eight warps work on alternate tiles, so one spreads bits while the
// other's products run; in a group two buffers of 256 features alternate.
//
// 4.2M rows of 1,024 features (0.60 GB): 0.71 ms by lookup tables, which the
// shared memory binds; here 0.66 ms with one thread a row (ten instructions to
// spread four bits and pack a parity, two warps a scheduler), 0.62 with two,
// 0.54 with one mask a word and parities taken from sign bits.  The products
// take 64 cycles each, 0.22 ms in all (tensor pipe 45% active).  Rows read by
// their own threads, four words at a time 4 * xw bytes apart, cost two batches
// of 65,536 rows a context 1,864 us; read a tile ahead, coalesced, and staged in
// shared memory, 1,830.  The kernel now takes 0.49 ms.
#include "elim.cuh"
#include "full.cuh"

namespace f2 {
namespace {

constexpr int TC_THREADS = 512;
constexpr int TC_TILE = 128;       // rows of a tile: two threads of a group each
constexpr int TC_KC = TC_CHUNK;    // features of a chunk (bytes of A, 64 columns of tensor memory)
constexpr int TC_KW = TC_KC / 64;  // its words for each of a row's two threads
constexpr int TC_N = 128;          // bits of y
// The order of the features along K is free, so the byte at 32 v + 4 w + j of a
// row is feature 32 v + 8 j + w: word w of the eight that hold a feature word's
// bits is that word, shifted for all w alike or not, under one mask.  Its
// bytes are single bits at tc_bit(w), e4m3 powers of two, and A's bytes there
// the inverse powers: a product of two ones is 1.
__host__ __device__ constexpr int tc_bit(int w) { return w < 3 ? w + 3 : (w < 7 ? w : 3); }
__host__ __device__ constexpr uint32_t tc_inverse(int w)
{
    // 2^-6, 2^-5, 2^-3, 2^1 at bits 3..6; bit 3 + ... of the exponent field
    return tc_bit(w) == 3 ? 0x68u : (tc_bit(w) == 4 ? 0x60u : (tc_bit(w) == 5 ? 0x50u : 0x30u));
}
// A in shared memory, K-major without swizzle: core matrices of 8 rows x 16
// bytes, the 16 row groups of one 16-byte column side by side.
constexpr int TC_LBO = TC_N * 16;  // bytes between 16-byte columns
constexpr int TC_SBO = 128;        // bytes between groups of 8 rows
constexpr int TC_A_BYTES = MAX_N * TC_N;
constexpr uint32_t TC_IDESC = (1u << 4) |                          // fp32 sums
                              ((uint32_t)(TC_N >> 3) << 17) |      // N; A and B e4m3, both K-major
                              ((uint32_t)(TC_TILE >> 4) << 24);    // M
constexpr int TC_STAGE_WORDS = TC_TILE * (MAX_N / 32 + 4);  // a group's rows
constexpr int TC_ST = TC_TILE * (MAX_N / 32) / 256;         // words of them that a thread loads
constexpr int TC_SMEM_BYTES = TC_A_BYTES + 2 * 4 * TC_STAGE_WORDS;
constexpr int TC_COLS = 512;       // tensor memory columns: two groups of 128 sums and 2 x 64 of rows
constexpr int TC_GROUP_COLS = 256;

struct TcSmem {
    unsigned long long bar[2][2];  // [group][buffer]: the products of a buffer are done
    uint32_t tmem;
    int q, k;
    uint32_t bad[2][4];            // [group][quarter]: rows that the second threads found contradicting
    unsigned long long cnt, first;
};

__device__ __forceinline__ uint64_t tc_desc(uint32_t addr)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(TC_LBO >> 4) << 16) | ((uint64_t)(TC_SBO >> 4) << 32) |
           (1ull << 46);  // descriptor version of this architecture, no swizzle
}

__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint64_t b, bool add)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a), "l"(b), "r"(TC_IDESC), "r"((uint32_t)add)
        : "memory");
}

__device__ __forceinline__ void tc_commit(unsigned long long* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

// Waits, with a limit, for the products that complete the phase of `bar`;
// false if they did not.  The lanes leave the wait at different times and the
// tensor-memory instructions after it take a whole warp, so they vote first;
// the fence orders those instructions after the products.
__device__ __forceinline__ bool tc_wait(unsigned long long* bar, uint32_t parity)
{
    const bool ok = __all_sync(FULL, mbar_wait_bounded(bar, parity)) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return ok;
}

__device__ __forceinline__ void tc_store32(uint32_t addr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(addr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]),
        "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]),
        "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

__device__ __forceinline__ void tc_load32(uint32_t addr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(addr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Barrier of a group (named barrier 1 + g): whether any of its threads says so.
__device__ __forceinline__ bool tc_any(int g, bool p)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, %2, 256, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(1 + g)
        : "memory");
    return r != 0u;
}

// A (column j of the map = the word of feature j) as bytes; features from n to
// kp are zero.
__device__ void tc_build(const StoreDev& s, const CtxDesc& cd, uint8_t* A, int kp, int t)
{
    const int first = s.raw ? 0 : 1;  // slot 0 holds the constant's word
    for (int k = 4 * t; k < kp; k += 4 * TC_THREADS) {
        const int w8 = (k >> 2) & 7;
        const uint32_t one = tc_inverse(w8);
        uint4 z[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int f = (k & ~31) + 8 * j + w8;
            z[j] = f < cd.n ? ld(s.bz + cd.slot_off + first + f) : make_uint4(0, 0, 0, 0);
        }
        uint8_t* const col = A + (k >> 4) * TC_LBO + (k & 15);
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint32_t v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = w == 0 ? z[j].x : (w == 1 ? z[j].y : (w == 2 ? z[j].z : z[j].w));
#pragma unroll 8
            for (int b = 0; b < 32; ++b) {
                const uint32_t bits = ((v[0] >> b) & 1u) | (((v[1] >> b) & 1u) << 8) | (((v[2] >> b) & 1u) << 16) |
                                      (((v[3] >> b) & 1u) << 24);
                const int row = 32 * w + b;
                *reinterpret_cast<uint32_t*>(col + (row >> 3) * TC_SBO + (row & 7) * 16) = bits * one;
            }
        }
    }
}

__global__ void __launch_bounds__(TC_THREADS, 1) verify_tc_kernel(StoreDev s, FullArgs a)
{
    pdl_wait();
    extern __shared__ __align__(128) uint8_t tc_smem[];
    __shared__ TcSmem sm;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // group, the half of each row's features and sums that is this thread's, and
    // the quarter of the rows (a warp reaches 32 lanes of tensor memory)
    const int g = warp >> 3, half = (warp >> 2) & 1, wg = warp & 3;
    const FullList list(a);
    if (list.n == 0) return;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&sm.tmem)),
                     "r"(TC_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (t == 0) {
        for (int i = 0; i < 4; ++i) mbar_init(&sm.bar[i >> 1][i & 1], 1);
        mbar_init_fence();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t base = sm.tmem + (uint32_t)(g * TC_GROUP_COLS);
    const uint32_t lanes = (uint32_t)(32 * wg) << 16;
    const uint32_t a_addr = smem_addr(tc_smem);
    // CTAs start at different contexts and go round, so that each builds few maps
    const int q0 = (int)((long long)blockIdx.x * list.n / gridDim.x);
    int q = -1, tried = 0, built = -1;
    uint32_t uses = 0;  // chunks this group has issued
    for (;;) {
        if (t < 32) {
            int k;
            const int qn = full_claim(s, a, list, true, q0, q, tried, lane, k);
            if (t == 0) {
                sm.q = qn;
                sm.k = k;
                sm.cnt = 0ull;
                sm.first = ~0ull;
            }
        }
        __syncthreads();
        q = sm.q;
        if (q < 0) break;
        const int c = list.ctx(a, q);
        const int64_t i_first = list.start(a, q, c);
        const CtxDesc cd = s.desc[c];
        const int nch = (cd.n + TC_KC - 1) / TC_KC;
        if (built != c) {  // (every product of the last context is done: its sums were read)
            tc_build(s, cd, tc_smem, nch * TC_KC, t);
            fence_proxy_async_smem();  // written by threads, read by the tensor cores
            built = c;
            __syncthreads();
        }
        const int64_t r0 = a.row_off[c];
        const int64_t T = a.row_off[c + 1] - r0;
        const int64_t i0 = i_first + (int64_t)sm.k * FULL_CHUNK;
        const int64_t i1 = (i0 + FULL_CHUNK < T) ? i0 + FULL_CHUNK : T;
        const uint32_t* const xc = a.x + a.x_off[c];
        const int xw = cd.xw;
        const bool vec = ((uintptr_t)xc & 15) == 0 && (xw & 3) == 0;
        const uint4 b = s.raw ? make_uint4(0, 0, 0, 0) : ld(s.bz + cd.slot_off);
        unsigned long long cnt = 0ull, first = ~0ull;
        // A tile's rows are contiguous: the group loads the next one into
        // registers, coalesced, while it works on this one from shared memory.
        // (Bits past the last feature meet zeros in the map.)
        const int tg = t & 255;
        const int rw = 4 * ((xw + 3) / 4) + 4;  // words of a staged row: 16-byte pieces, rows apart in the banks
        uint32_t* const stage = reinterpret_cast<uint32_t*>(tc_smem + TC_A_BYTES) + g * TC_STAGE_WORDS;
        uint32_t st[TC_ST];
        auto fetch = [&](int64_t tile) {
            const int rows = (int)(i1 - tile < TC_TILE ? i1 - tile : TC_TILE);
            const uint32_t* const src = xc + tile * xw;
            if (vec) {
#pragma unroll
                for (int u = 0; u < TC_ST / 4; ++u) {
                    const int k = tg + 256 * u;
                    if (4 * k < rows * xw) {
                        const uint4 v = ld(reinterpret_cast<const uint4*>(src) + k);
                        st[4 * u] = v.x;
                        st[4 * u + 1] = v.y;
                        st[4 * u + 2] = v.z;
                        st[4 * u + 3] = v.w;
                    }
                }
            } else {
#pragma unroll
                for (int u = 0; u < TC_ST; ++u) {
                    const int k = tg + 256 * u;
                    if (k < rows * xw) st[u] = ld(src + k);
                }
            }
        };
        auto put = [&]() {
            if (vec) {
                const int per = xw / 4;
#pragma unroll
                for (int u = 0; u < TC_ST / 4; ++u) {
                    const int k = tg + 256 * u, r = k / per;
                    if (r < TC_TILE)
                        *reinterpret_cast<uint4*>(stage + r * rw + 4 * (k - r * per)) =
                            make_uint4(st[4 * u], st[4 * u + 1], st[4 * u + 2], st[4 * u + 3]);
                }
            } else {
#pragma unroll
                for (int u = 0; u < TC_ST; ++u) {
                    const int k = tg + 256 * u, r = k / xw;
                    if (r < TC_TILE) stage[r * rw + k - r * xw] = st[u];
                }
            }
        };
        int64_t tile = i0 + (int64_t)g * TC_TILE;
        if (tile < i1) fetch(tile);
        // A wait that gives up ends the group's work: the tile's sums are then
        // unknown and not counted.  The group agrees on it at the tile's last
        // barrier only (a barrier with a result for each chunk took 35 us more for 4.2M rows);
        // what is still done for the tile until then is done in vain.
        bool gone = false;
        for (; tile < i1 && !gone; tile += 2 * TC_TILE) {
            const int64_t i = tile + 32 * wg + lane;
            const bool valid = i < i1;
            // (the group is done with the last tile's rows: its sums were compared)
            put();
            asm volatile("bar.sync %0, 256;" ::"r"(1 + g) : "memory");
            if (tile + 2 * TC_TILE < i1) fetch(tile + 2 * TC_TILE);
            const uint4 y = ld(a.y + r0 + (valid ? i : tile));
            const uint32_t* const xr = stage + (32 * wg + lane) * rw;
            bool ok = true;  // this warp's waits for the tile
            for (int ch = 0; ch < nch; ++ch, ++uses) {
                const int w0 = (2 * ch + half) * TC_KW;
                const uint4 xv = w0 < xw ? *reinterpret_cast<const uint4*>(xr + w0) : make_uint4(0, 0, 0, 0);
                const uint32_t x[TC_KW] = {xv.x, xv.y, xv.z, xv.w};
                const int buf = (int)(uses & 1u);
                const uint32_t use = uses >> 1;
                if (use > 0 && ok) ok = tc_wait(&sm.bar[g][buf], (use - 1) & 1u);
                const uint32_t at = base + TC_N + (uint32_t)(buf * (TC_KC / 4));
                uint32_t e[32];
#pragma unroll
                for (int v = 0; v < TC_KW; ++v) {
                    const uint32_t up = x[v] << 3, down = x[v] >> 4;
#pragma unroll
                    for (int w = 0; w < 8; ++w)
                        e[8 * v + w] = (w < 3 ? up : (w < 7 ? x[v] : down)) & (0x01010101u << tc_bit(w));
                }
                tc_store32(at + lanes + (uint32_t)(32 * half), e);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                asm volatile("bar.sync %0, 256;" ::"r"(1 + g) : "memory");
                if ((warp & 7) == 0 && lane == 0) {
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < TC_KC / 32; ++j)
                        tc_mma(base, at + (uint32_t)(8 * j),
                               tc_desc(a_addr + (uint32_t)((ch * (TC_KC / 16) + 2 * j) * TC_LBO)), ch > 0 || j > 0);
                    tc_commit(&sm.bar[g][buf]);
                }
                __syncwarp();
            }
            // the tile's sums
            const uint32_t last = uses - 1;
            if (ok) ok = !a.fail_wait && tc_wait(&sm.bar[g][last & 1u], (last >> 1) & 1u);
            uint32_t bad = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t v[32];
                tc_load32(base + lanes + (uint32_t)(64 * half + 32 * h), v);
                uint32_t word = 0;
#pragma unroll
                for (int j = 31; j >= 0; --j)  // 2^23 + an integer below 2^23: its lowest bit is the parity
                    word = __funnelshift_l(__float_as_uint(__uint_as_float(v[j]) + 8388608.0f) * 0x80000000u, word, 1);
                bad |= word ^ (h == 0 ? (half ? y.z ^ b.z : y.x ^ b.x) : (half ? y.w ^ b.w : y.y ^ b.y));
            }
            if (half) {
                const uint32_t m = __ballot_sync(FULL, bad != 0u);
                if (lane == 0) sm.bad[g][wg] = m;
            }
            gone = tc_any(g, !ok);
            if (!half && !gone && valid && (bad || ((sm.bad[g][wg] >> lane) & 1u))) {
                ++cnt;
                if ((unsigned long long)i < first) first = (unsigned long long)i;
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");  // before the next tile's products
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cnt += __shfl_xor_sync(FULL, cnt, o);
            const unsigned long long f = __shfl_xor_sync(FULL, first, o);
            first = f < first ? f : first;
        }
        if (lane == 0 && cnt) {
            atomicAdd(&sm.cnt, cnt);
            atomicMin(&sm.first, first);
        }
        const bool failed = __syncthreads_or(gone) != 0;
        if (t == 0) {
            if (failed) record_status(s.status, F2_ERR_TIMEOUT);
            full_commit(s, a, c, i_first, T, sm.cnt, sm.first, failed);
        }
        __syncthreads();
        if (failed) break;  // other CTAs take what is left
    }
    // the products still in flight (none, unless a wait gave up)
    for (uint32_t u = uses < 2 ? 0 : uses - 2; u < uses; ++u)
        (void)tc_wait(&sm.bar[g][u & 1u], (u >> 1) & 1u);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(TC_COLS) : "memory");
}

}  // namespace

cudaError_t verify_launch_tc(const StoreDev& sd, const FullArgs& fa, int num_sms, cudaStream_t cs)
{
    const cudaError_t e =
        cudaFuncSetAttribute(verify_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_BYTES);
    if (e != cudaSuccess) return e;
    f2_launch(verify_tc_kernel, num_sms, TC_THREADS, TC_SMEM_BYTES, cs, sd.num_ctx <= EARLY_MAX_CTX, sd, fa);
    return cudaGetLastError();
}

cudaError_t verify_load_tc()
{
    cudaFuncAttributes fa;
    return cudaFuncGetAttributes(&fa, verify_tc_kernel);
}

}  // namespace f2
