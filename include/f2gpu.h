/*
 * f2gpu.h -- C ABI of libf2gpu.so: batched streaming Gaussian elimination over
 * GF(2), affine-map extraction and batched encoding with a span check, on one
 * NVIDIA GB300 (sm_103a).
 *
 * The method is the exact bit-linear encoder learner of "Learning Exact
 * NVIDIA SASS Encoders with F2 Linear Algebra" (F2Asm):
 *   - an encoding context receives observations (x, y), x in F2^n (feature
 *     bits), y in F2^128 (instruction word); the feature vector is
 *     phi(x) = [1 || x] with the affine constant at index 0 and feature bit j
 *     at index 1+j (Sec. 2.1, parsed-value feature map), d = n + 1;
 *   - each augmented row [phi(x) | y] is reduced against the context's
 *     reduced basis B[k] = (r_k, z_k); zero/zero residuals are discarded, a
 *     zero feature residual with a nonzero word residual is a contradiction,
 *     anything else is inserted with pivot k = highest set feature index after
 *     clearing bit k from the stored rows (Sec. 2.2, steps (1)-(5));
 *   - the learned map is T(r_k) = z_k on S = rowspan(Phi) (Sec. 2.3);
 *     f2_solve_affine extends it by zero on non-pivot coordinates;
 *   - encoding reduces q = phi(x) against the basis while XOR-ing the z_k of
 *     every row used; a zero residual proves q in S and yields T(q), otherwise
 *     the query is rejected (Sec. 2.3, Appendix B).
 *
 * Conventions for every entry point:
 *   - Pointers named *_dev are device pointers (or managed/mapped memory the
 *     device can read); pointers named *_host are host pointers.  The caller
 *     owns all of them; the library never frees caller memory.
 *   - Feature words: uint32, bit j of x = bit j%32 of word j/32; a row of
 *     context c occupies W_c = ceil(n_c/32) words; bits at positions >= n_c
 *     are ignored.  128-bit words: four uint32 (bit i = bit i%32 of word
 *     i/32, the little-endian numbering of Appendix C), 16-byte aligned.
 *   - Every call is asynchronous on the caller's stream and ordered with the
 *     caller's other work on that stream; results are valid once the stream
 *     has been synchronized.  Calls on one store must not overlap on
 *     different streams.  The device that the store was created on is the
 *     current one, and `stream` a stream of it, in every call on the store
 *     (f2_get_basis, f2_device_status, f2_learn_timing, f2_store_export and
 *     f2_store_import copy only and take any current device).
 *   - Return value: F2_OK or an F2_ERR_* code for errors detected on the host
 *     before anything is enqueued (nothing is enqueued on error).  Errors that
 *     only the device can detect (bad CSR offsets, out-of-range context ids)
 *     are recorded in the store's device status word; read it with
 *     f2_device_status.  Contradictions and rejected queries are results,
 *     not errors.
 */
#ifndef F2GPU_H
#define F2GPU_H

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

/* Same type as cudaStream_t; NULL is the legacy default stream. */
typedef struct CUstream_st* f2_stream_t;

typedef struct f2_store f2_store;

enum f2_status {
    F2_OK = 0,
    F2_ERR_INVALID_ARG = 1, /* null pointer, negative size, bad flags, mismatched import */
    F2_ERR_NBITS = 2,       /* a feature width outside [1, 1024] */
    F2_ERR_CTX_RANGE = 3,   /* (device) an encode query named a context id outside [0, num_ctx) */
    F2_ERR_ALIGN = 4,       /* a pointer misses its required alignment */
    F2_ERR_OOM = 5,         /* device or host allocation failed */
    F2_ERR_CUDA = 6,        /* a CUDA runtime call failed */
    F2_ERR_TIMEOUT = 7,     /* (device) a bounded device-side wait gave up: the queries it was for are
                               not written; a full-rank context whose rows it was for keeps its
                               contradiction records and its row count as they were */
    F2_ERR_ROWS = 8,        /* (device) CSR offsets of a context are decreasing or out of bounds;
                               that context's rows were skipped */
    F2_ERR_STRIDE = 9       /* (device) a query's context needs more words than x_stride_words */
};

/* Rows are complete feature vectors: no implicit constant, d = n, feature
   bit j is index j.  Without this flag d = n + 1 and phi(x) = [1 || x]. */
#define F2_FLAG_RAW_FEATURES 1u

/* Text for a status code (static storage). */
const char* f2_status_string(int status);

/*
 * Create a store of num_ctx contexts on the current CUDA device.
 * n_bits_host[c] in [1, 1024] is context c's feature width n_c.  Allocates
 * the basis (slot k of context c for k < d_c), pivot masks, ranks and
 * contradiction records, all zeroed on `stream`.  On success *out receives
 * the handle; on failure *out is NULL.
 * Errors: F2_ERR_INVALID_ARG (out or n_bits_host NULL, num_ctx < 0, unknown
 * flags), F2_ERR_NBITS, F2_ERR_OOM, F2_ERR_CUDA.
 */
int f2_create(f2_store** out, int32_t num_ctx, const int32_t* n_bits_host, uint32_t flags,
              f2_stream_t stream);

/* Release the store's device memory (synchronizes the device). NULL is a no-op. */
void f2_destroy(f2_store* store);

/* Forget everything learned (bases, ranks, contradiction records, row counts). */
int f2_reset(f2_store* store, f2_stream_t stream);

/*
 * Host copies of the canonical layout offsets, each an array of num_ctx+1
 * int64 (any may be NULL):
 *   slot_off[c] = sum_{c'<c} d_c'              (128-bit slots: basis z, solve output)
 *   xw_off[c]   = sum_{c'<c} d_c' * Wd_c'      (basis feature words, Wd = ceil(d/32))
 *   pw_off[c]   = sum_{c'<c} Wd_c'             (pivot-mask words)
 */
int f2_layout(const f2_store* store, int64_t* slot_off, int64_t* xw_off, int64_t* pw_off);

/* Number of contexts, and the total sizes of the canonical arrays. */
int f2_sizes(const f2_store* store, int32_t* num_ctx, int64_t* slots, int64_t* basis_words,
             int64_t* pivot_words);

/*
 * Learn one batch of observations (Sec. 2.2).  May be called repeatedly: each
 * call continues every context's stream where the previous call stopped.
 *   row_off_dev[num_ctx+1] (int64): rows of context c are the 128-bit words
 *       y_dev[row_off[c] .. row_off[c+1]) in stream order (row_off[0] need
 *       not be 0);
 *   x_off_dev[num_ctx] (int64): row i of context c has its W_c feature words
 *       at x_dev[x_off[c] + i*W_c];
 *   y_dev: 4 uint32 per row, 16-byte aligned;
 *   total_rows / total_x_words: sizes of y_dev (rows) and x_dev (words); a
 *       context whose rows or words fall outside them is skipped and
 *       F2_ERR_ROWS is recorded on the device.
 * Per context: rank, reduced basis, pivot mask, contradiction flag (sticky),
 * index of the first contradicting row (counted over the context's whole
 * stream, across calls, from 0) and the number of contradicting rows.
 * Contradicting rows are not inserted; learning continues after them.
 * At most 2^31 - 1 rows per context per call (larger contexts: F2_ERR_ROWS).
 * Scratch: the scheduling queues allocated by f2_create and 8 bytes per row
 * of y_dev (grown stream-ordered with cudaMallocAsync when total_rows exceeds
 * the previous capacity); calls on one store must not overlap.
 * Errors: F2_ERR_INVALID_ARG (NULL pointer or negative size), F2_ERR_ALIGN
 * (y_dev not 16-byte aligned, offsets not 8-byte aligned), F2_ERR_CUDA.
 */
int f2_learn_batched(f2_store* store, const int64_t* row_off_dev, const uint32_t* x_dev,
                     const int64_t* x_off_dev, const uint32_t* y_dev, int64_t total_rows,
                     int64_t total_x_words, f2_stream_t stream);

/*
 * Copy the learned state into caller device buffers (any may be NULL):
 *   rank_dev[num_ctx] int32; pivot_mask_dev[pivot_words] uint32 (bit k of
 *   context c at word pw_off[c] + k/32); basis_x_dev[basis_words] uint32
 *   (row k of context c at xw_off[c] + k*Wd_c: r_k, bit j = feature index
 *   j); basis_z_dev[4*slots] uint32 (z_k at slot slot_off[c] + k);
 *   contra_dev[num_ctx] uint8 (0/1); first_contra_dev[num_ctx] int64 (-1 if
 *   none); n_contra_dev[num_ctx] uint64; rows_seen_dev[num_ctx] int64.
 * Empty slots are zero.  The basis is in reduced echelon form: r_k has its
 * highest set bit at k and is zero at every other pivot (Appendix B).
 */
int f2_get_basis(const f2_store* store, int32_t* rank_dev, uint32_t* pivot_mask_dev,
                 uint32_t* basis_x_dev, uint32_t* basis_z_dev, uint8_t* contra_dev,
                 int64_t* first_contra_dev, uint64_t* n_contra_dev, int64_t* rows_seen_dev,
                 f2_stream_t stream);

/*
 * Affine solve (Sec. 2.3): W_dev[4*slots] receives, for context c and index
 * j < d_c, the 128-bit row W[c][j] at slot slot_off[c] + j: z_j if j is a
 * pivot, zero otherwise (free coordinates set to zero; W is unique only on
 * the span).  Without F2_FLAG_RAW_FEATURES, b = W[c][0] and column j of A is
 * W[c][1+j], so y = A x XOR b for every x whose phi(x) lies in the span.
 * Errors: F2_ERR_INVALID_ARG, F2_ERR_ALIGN (W_dev not 16-byte aligned).
 */
int f2_solve_affine(const f2_store* store, uint32_t* W_dev, f2_stream_t stream);

/*
 * Encode Q queries (Sec. 2.3, Appendix B).  Query q names context
 * ctx_id_dev[q]; its feature words are x_dev[q*x_stride_words ...].
 * y_out_dev[4*q ..] receives T(phi(x)) when phi(x) is in the context's span
 * and zero otherwise; in_span_dev[q] receives 1 (supported), 0 (rejected) or
 * 0xFF (context id out of range -- F2_ERR_CTX_RANGE is recorded -- or the
 * context needs more than x_stride_words words -- F2_ERR_STRIDE).
 * The queries are grouped by context on the device first, and every context
 * with at least F2_OPT_ENCODE_TABLE_MIN queries in a pass gets a lookup table
 * of its basis (16*ceil(d/4)*(4 + ceil((d - rank)/32)) words, for d <= 288 and
 * d - rank <= 128).  The store keeps that scratch: 20 bytes per query (at most
 * 2^25 queries per pass), about 8*(1 + chunks) bytes per context, and a table
 * pool with room for the table of every context that can have one (at most
 * 1 GiB; a context whose table does not fit is encoded without one), all
 * allocated stream-ordered with cudaMallocAsync on first need.
 * Errors: F2_ERR_INVALID_ARG (Q < 0, NULL pointers, x_stride_words < 1),
 * F2_ERR_ALIGN (y_out_dev not 16-byte aligned), F2_ERR_OOM (scratch).
 */
int f2_encode_batched(const f2_store* store, int64_t Q, const int32_t* ctx_id_dev,
                      const uint32_t* x_dev, int32_t x_stride_words, uint32_t* y_out_dev,
                      uint8_t* in_span_dev, f2_stream_t stream);

/*
 * Learning from host memory (Sec. 2.2, as f2_learn_batched): the same CSR
 * batch, but row_off_host, x_host, x_off_host and y_host are host arrays
 * (page-locked memory lets the copies overlap the kernels; pageable memory
 * works, with the copies serialised).  The batch is validated on the host
 * (F2_ERR_INVALID_ARG for decreasing offsets, offsets outside the arrays)
 * and cut into chunks of whole contexts of about F2_OPT_HOST_CHUNK_BYTES of
 * rows; a private copy stream moves chunk j + 1 into a device double buffer
 * while `stream` learns chunk j.  The resulting state equals one
 * f2_learn_batched call on the same batch (contexts are independent).  The
 * host arrays are read asynchronously: keep them unchanged until `stream`
 * has passed the call.  Device scratch: two chunk buffers and the rebased
 * offsets (16 bytes per context), grown on demand (the call then
 * synchronizes `stream`); kept by the store until f2_destroy.  Errors:
 * F2_ERR_INVALID_ARG (NULL pointers, negative sizes, the host checks above;
 * nothing is enqueued), F2_ERR_OOM, F2_ERR_CUDA, and those of
 * f2_learn_batched for each chunk (device-detected ones in the status word).
 */
int f2_learn_host(f2_store* store, const int64_t* row_off_host, const uint32_t* x_host,
                  const int64_t* x_off_host, const uint32_t* y_host, int64_t total_rows,
                  int64_t total_x_words, f2_stream_t stream);

/*
 * Encoding from and to host memory (Sec. 2.3, as f2_encode_batched):
 * ctx_id_host int32[Q], x_host uint32[Q * x_stride_words], y_out_host
 * uint32[4 * Q], in_span_host uint8[Q] are host arrays (page-locked for
 * overlap).  Queries go in chunks of at most F2_OPT_HOST_CHUNK_BYTES (and at
 * least four chunks of at least 65,536 queries when Q allows): chunk
 * j + 1 is copied in on a private stream while `stream` encodes chunk j and
 * a second private stream copies the words of chunk j - 1 out.  Results are
 * those of f2_encode_batched; device errors are recorded in the store's
 * status word as there.  The outputs are written asynchronously: they are on
 * the host once `stream` has passed the call.  Errors: F2_ERR_INVALID_ARG
 * (Q < 0, NULL pointers, x_stride_words < 1), F2_ERR_OOM, F2_ERR_CUDA.
 */
int f2_encode_host(const f2_store* store, int64_t Q, const int32_t* ctx_id_host, const uint32_t* x_host,
                   int32_t x_stride_words, uint32_t* y_out_host, uint8_t* in_span_host, f2_stream_t stream);

/*
 * Map pooling (Sec. 3: the bases of an (f, m) group are combined and
 * eliminated together; one shared map if the equations are consistent and
 * the output masks match, else separate maps).  group_of_host[c] in
 * [0, num_groups) puts source context c in a group (-1: left out); every
 * group needs at least one member and all members of a group the same d.
 * *out receives a new store with F2_FLAG_RAW_FEATURES and one context per
 * group of width d (its feature rows are phi-space vectors, index 0 = the
 * constant): the members' basis rows, members in context order and pivots in
 * increasing order, learned as one stream.  Its basis is the reduced echelon
 * form of the union of the members' spans; its contradiction flag marks
 * inconsistent equations (first_contra / n_contra count merged rows).
 * out_mask_host (uint32[4*num_ctx], the learned output bits of each context;
 * NULL: all equal) and mask_ok_host (uint8[num_groups], may be NULL): 1 where
 * all members' masks are equal.  A group shares one map iff mask_ok and not
 * contra.  The call synchronizes `stream`; destroy *out with f2_destroy.
 * Errors: F2_ERR_INVALID_ARG, F2_ERR_CTX_RANGE (group id out of range),
 * F2_ERR_NBITS (members of different widths), F2_ERR_OOM, F2_ERR_CUDA.
 */
int f2_merge_bases(const f2_store* src, int32_t num_groups, const int32_t* group_of_host,
                   const uint32_t* out_mask_host, f2_store** out, uint8_t* mask_ok_host, f2_stream_t stream);

/*
 * Encode epilogue (Appendix C, Eq. hmma-full-word; Appendix D): turns the
 * learned words of accepted queries into full instruction words, in place.
 * Scheduler control is kept outside the learned bits and merged at bits
 * 105..121; bits a context's opaque mask excludes from learning (App. D:
 * 122 and 124 of DEPBAR_SB_II) are restored from state the caller recorded.
 * For every q with in_span_dev[q] == 1 and c = ctx_id_dev[q]:
 *   y = ((y XOR (sc_dev[q] << 105)) AND NOT M_c) OR (state_dev[q] AND M_c)
 * with sc_dev[q] the 17 scheduler-control bits (higher bits ignored),
 * state_dev[4*q ..] the recorded 128-bit word (only its M_c bits are used)
 * and M_c = opaque_mask_dev[4*c ..] (128-bit, same numbering as y).
 * sc_dev NULL: no merge; state_dev or opaque_mask_dev NULL: no restore.
 * Rejected queries (in_span != 1) keep their zero word.  y_dev is
 * y_out_dev of f2_encode_batched (uint32[4*Q], 16-byte aligned).
 * Errors: F2_ERR_INVALID_ARG (Q < 0, NULL y, in_span or ctx_id),
 * F2_ERR_ALIGN (y_dev, state_dev or opaque_mask_dev not 16-byte aligned).
 */
int f2_encode_epilogue(const f2_store* store, int64_t Q, const int32_t* ctx_id_dev,
                       const uint8_t* in_span_dev, const uint32_t* sc_dev, const uint32_t* state_dev,
                       const uint32_t* opaque_mask_dev, uint32_t* y_dev, f2_stream_t stream);

/*
 * Synchronize `stream`, then read and clear the store's device status word:
 * *status receives F2_OK or the first device-detected F2_ERR_* code since the
 * last read.
 */
int f2_device_status(f2_store* store, int* status, f2_stream_t stream);

/*
 * Checkpoint: serialize the whole learned state into host memory.  With
 * host_buf NULL, *size receives the number of bytes needed.  Otherwise
 * *size must be at least that; the call synchronizes `stream`.
 */
int f2_store_export(const f2_store* store, void* host_buf, size_t* size, f2_stream_t stream);

/* Restore a checkpoint written by f2_store_export from a store with the same
   context count, widths and flags (F2_ERR_INVALID_ARG otherwise). */
int f2_store_import(f2_store* store, const void* host_buf, size_t size, f2_stream_t stream);

/* Scheduling knobs of f2_learn_batched (performance only, never results). */
enum f2_option {
    F2_OPT_HEAVY_ROWS = 1,   /* contexts with at least this many rows in a call get a whole CTA; unless
                                this or F2_OPT_WARP_WORK is set, the call scales both to its own work
                                (representatives / (20 SMs), within [1024, 4096]; with the duplicate
                                pass off, rows / 20000). Unless this is set, a store of at most two
                                contexts per SM gives every context a whole CTA */
    F2_OPT_WARP_BASIS_BYTES = 2, /* shared memory (bytes) of one warp-owned context */
    F2_OPT_WARP_WORK = 3,        /* largest rows x d (per call) of a warp-owned context; default 131072,
                                    scaled like F2_OPT_HEAVY_ROWS (sum of rows x d / (45 SMs), at least
                                    32768) */
    F2_OPT_DEDUP = 4,            /* 1 (default): eliminate only the first occurrence of each distinct
                                    row and classify its repeats with it; 0: eliminate every row */
    F2_OPT_ENCODE_TABLE_MIN = 5, /* fewest queries of one context (in a pass of f2_encode_batched)
                                    for which a lookup table of its basis is built; default 64, at
                                    least 1; a value above the pass size disables the tables */
    F2_OPT_HOST_CHUNK_BYTES = 6, /* bytes of rows (f2_learn_host) or of queries (f2_encode_host) per
                                    copied chunk; default 512 MiB, at least 64 KiB */
    F2_OPT_ENCODE_CHUNK_SHIFT = 7, /* log2 of the consecutive queries whose table-encoded results are
                                    written together (L2 locality of f2_encode_batched's output);
                                    default 20, in [11, 25]; raised so a pass has at most 64 chunks */
    F2_OPT_ENCODE_CHUNK_MIN = 8, /* fewest queries of one context (in a pass) for which its queries are
                                    laid out chunk by chunk (the others keep one run); default 512 */
    F2_OPT_FAIL_ALLOC = 9,       /* test hook: the device allocation made after `value` more successful
                                    ones by calls on this store fails as if out of memory (the call
                                    returns F2_ERR_OOM and the store stays usable; where it was for a
                                    hand-off that the call makes by default, the call goes without);
                                    -1 (default) = off */
    F2_OPT_TIMING = 10,          /* 1: f2_learn_batched records per-context timestamps (f2_learn_timing);
                                    0 (default): off */
    F2_OPT_ELIM_TABLES = 11,     /* 1 (default): step (1) against the basis uses a 4-bit lookup table of it
                                    where it fits and pays; 0: always walk the pivots */
    F2_OPT_SMALL_BASIS_BYTES = 12, /* shared memory (bytes) of one warp-owned context of width d <= 96;
                                    default 9472, in [4096, 24576] */
    F2_OPT_DEDUP_SHARDS = 13,    /* most CTAs that the duplicate pass of one context is split over
                                    (consecutive row ranges of at least 2048 rows: one per 1/(4 x SMs)
                                    of the call's rows x (feature words + 4) the context holds, and
                                    at least one per 16384 rows); default 4, in [1, 8]; 1 = never
                                    split (and no 4-warp context promoted to a whole CTA) */
    F2_OPT_ENCODE_DIRECT_MAX = 14, /* f2_encode_batched calls of at most this many queries encode each
                                    query on its own from the stored basis, with no grouping and no
                                    tables (one kernel launch); default 65536, 0 = never */
    F2_OPT_LONG_CALL_ROWS = 15,  /* f2_learn_batched calls of at least this many rows eliminate the contexts
                                    of 4..9 words in CTAs of four warps instead of eight (more contexts
                                    side by side; the longest contexts take longer); default 2^25. A store
                                    small enough for a CTA per context keeps eight */
    F2_OPT_HANDOFF_REPS = 16,    /* a context owned by a whole CTA whose rank has stopped growing hands
                                    the rest of its call off to a parallel check when at least this many
                                    of its representatives are left (a representative outside the basis
                                    sends the rest back to elimination from there); only in calls of at
                                    least 16x this many rows; 0 = never. -1 (default): calls of at
                                    least 2^20 rows on a store with contexts of 10..17 words hand off
                                    the contexts with at least 2048 representatives left that do not
                                    run against a lookup table */
    F2_OPT_FAIL_WAIT = 17,       /* test hook: 1: the waits of f2_learn_batched's tensor-core full-rank check
                                    (contexts of many features) act as if they had given up
                                    (F2_ERR_TIMEOUT); 0 (default): off */
};
int f2_set_option(f2_store* store, int option, int64_t value);

/*
 * Per-context timestamps of the last f2_learn_batched call on a store with
 * F2_OPT_TIMING = 1 (a diagnostic with no counterpart in the paper: it shows
 * how the contexts' work spreads over the SMs and how long the last context
 * runs past the others).  out_host: host uint64[6*num_ctx]; for context c,
 * words 6c..6c+3 are the device's %globaltimer (ns) at the start and end of
 * the context's duplicate pass and of its elimination, words 6c+4 and 6c+5
 * the ids of the SMs that ran them; zero where the context had no such work
 * in that call.  Synchronizes `stream`.  Errors: F2_ERR_INVALID_ARG (NULL
 * pointers, or no learn call with timing on), F2_ERR_CUDA.
 */
int f2_learn_timing(const f2_store* store, uint64_t* out_host, f2_stream_t stream);

/*
 * Allocation-free learning (the paper has no counterpart; this is a
 * deployment aid).  Some callers cannot call cudaMalloc: processes whose
 * device memory is entirely pre-reserved by a pooling allocator (a
 * framework's caching allocator, an inference server's arena), where an
 * extra cudaMalloc fails or breaks the memory budget, and latency-critical
 * code that must not pay the implicit device synchronization that
 * cudaMalloc and cudaFree can cause.  f2_learn_batched_noalloc performs one
 * call of f2_learn_batched without any allocation: no store, no cudaMalloc,
 * cudaFree or allocating library routine.  The caller owns every buffer;
 * the scheduling scratch (context descriptors, work queues, counters) lives
 * in one fixed, file-scope device array of the library, sized for
 * F2_NOALLOC_MAX_CTX contexts (about 1.6 MB), that every GPU which loads the
 * library holds until the process exits.
 *
 *   num_ctx        in [0, F2_NOALLOC_MAX_CTX]; larger values are rejected
 *                  with F2_ERR_INVALID_ARG before anything is enqueued.
 *                  With num_ctx == 0 the call only sets *status_dev to F2_OK.
 *   n_bits_host    host int32[num_ctx], each in [1, 1024] (F2_ERR_NBITS);
 *                  copied during the call (through a library-owned host
 *                  array), so it may be reused as soon as the call returns.
 *   flags          0 or F2_FLAG_RAW_FEATURES, as for f2_create.
 *   state (device, caller-owned, in/out, canonical layout of f2_get_basis;
 *          sizes from d_c = n_c + 1 (n_c for raw rows), Wd_c = ceil(d_c/32)):
 *     rank_dev int32[num_ctx], pivot_mask_dev uint32[sum Wd_c],
 *     basis_x_dev uint32[sum d_c*Wd_c], basis_z_dev uint32[4*sum d_c]
 *     (16-byte aligned), contra_dev uint8[num_ctx], first_contra_dev
 *     int64[num_ctx], n_contra_dev uint64[num_ctx], rows_seen_dev
 *     int64[num_ctx].  Before the first call every array must be zero except
 *     first_contra_dev, which must be -1 everywhere; each call then continues
 *     the streams exactly as f2_learn_batched continues a store's.
 *   status_dev     device int32: set to F2_OK by the call, then receives the
 *                  first device-detected error (F2_ERR_ROWS).
 *   row_off_dev, x_dev, x_off_dev, y_dev, total_rows, total_x_words: one
 *                  CSR batch, exactly as for f2_learn_batched.
 * The first call on a device (per process) does a one-time set-up: it looks
 * up the device address of the scratch array with cudaGetSymbolAddress and
 * loads every kernel this entry point can launch (loading a kernel's code
 * may itself allocate device memory, so only this first call may allocate);
 * make that first call before any stream capture.  Every call shares the
 * one scratch array and rewrites what it uses, so calls that overlap on the
 * GPU (different streams, or different host threads) race: serialize them.
 * Results are bit-identical to f2_learn_batched on the same inputs.
 * Errors: F2_ERR_INVALID_ARG, F2_ERR_NBITS, F2_ERR_ALIGN, F2_ERR_CUDA.
 */
#define F2_NOALLOC_MAX_CTX 16384
int f2_learn_batched_noalloc(int32_t num_ctx, const int32_t* n_bits_host, uint32_t flags,
                             int32_t* rank_dev, uint32_t* pivot_mask_dev, uint32_t* basis_x_dev,
                             uint32_t* basis_z_dev, uint8_t* contra_dev, int64_t* first_contra_dev,
                             uint64_t* n_contra_dev, int64_t* rows_seen_dev, int32_t* status_dev,
                             const int64_t* row_off_dev, const uint32_t* x_dev, const int64_t* x_off_dev,
                             const uint32_t* y_dev, int64_t total_rows, int64_t total_x_words,
                             f2_stream_t stream);

#ifdef __cplusplus
}
#endif

#endif /* F2GPU_H */
