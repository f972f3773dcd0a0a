/*
 * tahq.h -- C ABI of the B200 (sm_100a) TAH-Quant boundary codec.
 *
 * The library compresses the activation (or activation-gradient) tensor that
 * crosses a pipeline-stage boundary and restores it on the other side
 * (TAH-Quant, Sec. 3.1-3.4; Algorithm 1 lines 4-5).  All work runs in CUDA
 * kernels on the caller's stream; there is no CPU fallback.
 *
 * Conventions for every entry point
 *   - Pointers named d_* are DEVICE pointers, 16-byte aligned, owned by the
 *     caller.  The library never allocates, frees or synchronises, and never
 *     touches a stream other than the one passed in.
 *   - Calls are asynchronous and stream-ordered.  Host-detectable errors
 *     (every code but TAHQ_ERR_CUDA) are returned before anything is enqueued.
 *   - d_ws is scratch memory of at least tahq_workspace_bound() bytes.  Its
 *     first 4 bytes are a device status word (0 = ok, see TAHQ_DEV_*) that the
 *     caller may read after synchronising the stream.  Two calls that overlap
 *     on the GPU must not share a workspace.
 *   - Inputs must be finite.  Non-finite inputs give unspecified values but
 *     never touch memory outside the buffers.
 *   - Same inputs, same bytes: every byte of [0, tahq_packed_bound()) is
 *     written, padding included.
 */
#ifndef TAHQ_H
#define TAHQ_H

#include <stddef.h>
#include <stdint.h>

#ifdef __cplusplus
extern "C" {
#endif

/* Opaque stand-in for cudaStream_t so that this header needs no CUDA include. */
typedef struct CUstream_st *tahq_stream;

typedef enum {
  TAHQ_OK = 0,
  TAHQ_ERR_INVALID_ARG = 1,      /* null pointer, bad struct_size, bad shape/tile/budget        */
  TAHQ_ERR_UNSUPPORTED = 2,      /* valid in the format but not built (see alloc_tile)          */
  TAHQ_ERR_BUFFER_TOO_SMALL = 3, /* packed_cap / packed_bytes / ws_cap below the bound          */
  TAHQ_ERR_MISALIGNED = 4,       /* a device pointer is not 16-byte aligned                     */
  TAHQ_ERR_CUDA = 5,             /* a CUDA runtime call (launch, memset) failed                 */
  TAHQ_ERR_TOO_LARGE = 6         /* tahq_encode_noalloc: needs more scratch than is built in    */
} tahq_status;

typedef enum { TAHQ_F32 = 0, TAHQ_BF16 = 1 } tahq_dtype;

/* Bits of the device status word at d_ws[0..4). */
enum {
  TAHQ_DEV_OK = 0,
  TAHQ_DEV_BAD_HEADER = 1,       /* decode: the buffer's header does not match the parameters   */
  TAHQ_DEV_BAD_BITMAP = 2,       /* decode: bit map population does not match the payload size  */
  TAHQ_DEV_TIMEOUT = 4,          /* a bounded device-side wait ran out                          */
  TAHQ_DEV_INTERNAL = 8          /* encode: a screening bound of the tile selection was violated */
};

/*
 * One boundary tensor.  Names follow the paper: a tile is a quantisation group
 * of G contiguous channels of one token (Sec. 3.1); allocation tiles equal
 * quantisation tiles (A = G, the default of Sec. 3.2); a ranking group is one
 * sample of S = group_tokens consecutive tokens (Sec. 3.2, top-p% selection).
 */
typedef struct {
  uint32_t struct_size;      /* = sizeof(tahq_params)                                            */
  uint32_t dtype;            /* tahq_dtype of the dense row-major [tokens x hidden] tensor       */
  uint64_t tokens;           /* T = B*S                                                          */
  uint32_t hidden;           /* C, a multiple of tile                                            */
  uint32_t group_tokens;     /* S; 0 = the whole tensor is one ranking group; must divide T      */
  uint32_t tile;             /* G in {8, 16, 32, 64, 128} (8 and 16: the small groups of the paper's
                                ablation; their metadata costs 5.1 / 2.6 bits per element)          */
  uint32_t budget_millibits; /* payload bits per element x 1000, in [2000, 8000].  lo = b/1000
                                bits for every tile, and the floor(n_g*(b%1000)/1000) highest-
                                entropy tiles of each ranking group get lo+1.  3800 is the
                                paper's 80% INT4 + 20% INT3.                                     */
  float tau;                 /* outlier threshold of Eq. 3 (paper: 2.0; 0 = always transform,
                                +inf = never)                                                    */
  float eps_l1;              /* epsilon  of Eq. 1 (1e-8f)                                        */
  float eps_log;             /* varsigma of Eq. 2 (1e-8f); a positive normal binary32 number     */
  float eps_ratio;           /* varrho   of Eq. 3 (1e-8f)                                        */
  uint32_t rounding;         /* 0 = round-half-even (the default; the paper names no mode);
                                1 = stochastic: q = min(floor(clamp(y, 0, 2^b-1) + u), 2^b-1) on the
                                binary32 product y = (v - z) * (1/s), u = top 24 bits of word (i mod 4)
                                of Philox4x32-10(key = seed, counter = i / 4) times 2^-24, i = the
                                element's index in the tensor: codes are a function of (input, seed)  */
  uint64_t seed;             /* used only when rounding == 1                                     */
  uint32_t alloc_tile;       /* A of Sec. 3.2: allocation-tile width, a multiple of tile that divides
                                hidden and is at most 8192; 0 = tile (the paper's default).  The entropy
                                is taken over A channels, the top-p% of the S*hidden/A allocation tiles of
                                a ranking group get the higher width, and every quantisation tile inside
                                shares it; A = hidden is token-level allocation.  A above 8192 is
                                TAHQ_ERR_UNSUPPORTED.                                                */
} tahq_params;

/* Byte offsets of the sections of the packed buffer (all multiples of 128). */
typedef struct {
  uint64_t n_tiles, n_groups, tiles_per_group, k_hi;
  uint32_t lo_bits, hi_bits;
  uint64_t off_bitmap, off_scale_zero, off_pivot, off_payload;
  uint64_t payload_bytes, total_bytes;
} tahq_layout;

/*
 * Exact size in bytes of the packed buffer (Sec. 3.4: a fixed-shape uint8
 * stream; the size depends on the parameters only, never on the data).
 * Returns 0 when the parameters are invalid or unsupported.  Host-only.
 */
size_t tahq_packed_bound(const tahq_params *p);

/* Section offsets of the packed buffer; TAHQ_OK or an error.  Host-only. */
tahq_status tahq_packed_layout(const tahq_params *p, tahq_layout *out);

/*
 * Bytes of scratch that tahq_encode / tahq_decode need for these parameters
 * (tile scores, offset prefixes, the flags of a decode's offset look-back, status
 * word).  Returns 0 when the parameters are invalid.  Host-only.
 */
size_t tahq_workspace_bound(const tahq_params *p);

/*
 * Encode (Sec. 3.1-3.4): d_in [tokens x hidden] (dtype) -> d_packed.
 *   Per tile: entropy score on the raw tile (Eq. 1-2); per ranking group the
 *   top-p% scores get the higher width (Sec. 3.2); outlier test (Eq. 3), pivot
 *   swap + Hadamard on flagged tiles (Eq. 4); min-max asymmetric quantisation
 *   with binary16 scale and zero-point (Sec. 3.3); variable-width little-endian
 *   bit packing plus bit map, scale/zero and pivot sections (Sec. 3.4).
 * d_in is read only; d_packed[0, packed_bound) is fully overwritten.
 * Errors: INVALID_ARG, UNSUPPORTED, BUFFER_TOO_SMALL (packed_cap or ws_cap),
 * MISALIGNED, CUDA.  Nothing is enqueued when one of the host-detectable errors (all but CUDA) is returned.
 */
tahq_status tahq_encode(const tahq_params *p, const void *d_in, void *d_packed, size_t packed_cap,
                        void *d_ws, size_t ws_cap, tahq_stream stream);

/*
 * Decode (Sec. 3.3, Algorithm 1 line 5): d_packed -> d_out [tokens x hidden]
 * (dtype): bit map -> widths and offsets, unpack, z + q*s, inverse Hadamard
 * and un-swap on flagged tiles, store (round-to-nearest-even for bf16).
 * The header inside d_packed must describe the same parameters; a mismatch is
 * reported through the device status word (TAHQ_DEV_BAD_HEADER) and the output
 * is left untouched.  A bit map whose population does not match the payload
 * size is reported as TAHQ_DEV_BAD_BITMAP; the output is then unspecified, and
 * no byte outside the two buffers is read or written.
 * Errors as for tahq_encode (packed_bytes must be >= tahq_packed_bound()).
 */
tahq_status tahq_decode(const tahq_params *p, const void *d_packed, size_t packed_bytes, void *d_out,
                        void *d_ws, size_t ws_cap, tahq_stream stream);

/*
 * Encode without a caller-provided workspace (the paper has no counterpart; this is a convenience of
 * the library).  Same operation, same bytes in d_packed as tahq_encode, but the scratch memory lives
 * in a fixed buffer (TAHQ_NOALLOC_SCRATCH_BYTES and 8 MiB of prefixes) that is part of the library image
 * on every GPU that loads it, so the call neither needs a workspace pointer nor allocates or frees anything.
 *
 * Who needs this: code that is handed device pointers but owns no allocator and may not call
 * cudaMalloc -- a communication plug-in working on buffers registered by its host framework, a
 * process whose device memory was carved up in advance by a pool it cannot ask, or a step that runs
 * where an allocation would force a device-wide synchronisation.
 *
 * Limits and rules
 *   - Accepts every configuration with tahq_workspace_bound(p) <= TAHQ_NOALLOC_SCRATCH_BYTES (8192 x 4096
 *     elements at tile 64 need 2.3 MB).  Where ranking groups share words of the bit map, the offset
 *     prefixes (4 bytes per 32 tiles) do not count towards that: the library has room for them.
 *     Anything larger returns TAHQ_ERR_TOO_LARGE and enqueues nothing.
 *   - The first call on each device looks up the device address of the built-in buffer (a host-side
 *     set-up step, done once per device with that device current).  Make that first call before any
 *     stream capture begins.
 *   - All calls on one device share the one buffer.  It keeps the previous call's contents, of which no
 *     call reads any.  Two calls that may overlap on the GPU (different streams without an ordering
 *     between them) race on it: order them, or use tahq_encode with separate workspaces.
 *   - The device status word of the call cannot be read back by the caller; use tahq_encode when that
 *     is needed.
 * Errors: as tahq_encode, plus TAHQ_ERR_TOO_LARGE.
 */
#define TAHQ_NOALLOC_SCRATCH_BYTES (8u << 20)
tahq_status tahq_encode_noalloc(const tahq_params *p, const void *d_in, void *d_packed, size_t packed_cap,
                                tahq_stream stream);

/*
 * Fixed-point gradient compressor Q_Naive (Algorithm 1 lines 6-7, Sec. 3.5; pre-scale of the appendix,
 * g_hat = Q(c g) / c).  The paper names it and gives no formula; this library's reading:
 *   y = c * g (binary32);  per token (row) or per tensor: s = max|y| / L, L = 2^(b-1) - 1, kept as binary32;
 *   q = clamp(round(y * (1/s)), -L, L), product rounded once, ties to even; code = q + L in b bits;
 *   g_hat = (q * s) / c (binary32 product, then binary32 division).
 * Packed buffer: 128-byte header, binary32 scales, then one row of codes per token (little-endian bit
 * stream, element k at bits [k b, (k+1) b)), rows padded to 16 bytes, sections to 128; size depends on
 * the parameters only; every byte is written.
 * d_in / d_out: dense row-major [tokens x hidden] (dtype), device, 16-byte aligned.  d_ws: at least
 * tahq_qnaive_workspace_bound() bytes; its first 4 bytes are the device status word (TAHQ_DEV_BAD_HEADER
 * when decode is handed a buffer whose header does not match; the output is then untouched).
 * Errors as for tahq_encode / tahq_decode.
 */
typedef struct {
  uint32_t struct_size;      /* = sizeof(tahq_qnaive_params)                     */
  uint32_t dtype;            /* tahq_dtype                                       */
  uint64_t tokens;
  uint32_t hidden;           /* a multiple of 8                                  */
  uint32_t bits;             /* b in [2, 16] (the paper uses 6, 8 and 10)        */
  uint32_t per_tensor;       /* 0: one scale per token; 1: one for the tensor    */
  float prescale;            /* c > 0, finite (1.0f = none)                      */
} tahq_qnaive_params;

size_t tahq_qnaive_packed_bound(const tahq_qnaive_params *p);      /* 0 if the parameters are invalid */
size_t tahq_qnaive_workspace_bound(const tahq_qnaive_params *p);
tahq_status tahq_qnaive_encode(const tahq_qnaive_params *p, const void *d_in, void *d_packed, size_t packed_cap,
                               void *d_ws, size_t ws_cap, tahq_stream stream);
tahq_status tahq_qnaive_decode(const tahq_qnaive_params *p, const void *d_packed, size_t packed_bytes, void *d_out,
                               void *d_ws, size_t ws_cap, tahq_stream stream);

/* Static string for a status code. */
const char *tahq_status_string(tahq_status s);

#ifdef __cplusplus
}
#endif
#endif /* TAHQ_H */
